"""Tensor-core products of vectors that hold an Inf or a NaN."""
import numpy as np
import pytest

from paper_2103_16841_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("level,slabs", [(1, 3), (0, 14), (0, 43), (0, 64)])
@pytest.mark.parametrize("dtype", ["tf32", "bf16"])
@pytest.mark.parametrize("bad", [np.inf, -np.inf, np.nan, 1e300])
def test_only_rows_with_a_value_see_it(level, slabs, dtype, bad):
    """One or many columns per tile, one tile or two: the rows without an entry at
    the panel keep the bits or an FP32 sum of the same rounded terms, the others
    get the entry's sign times Inf, or NaN; other right-hand sides keep their bits."""
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import paper_2103_16841_gb300 as stb
    ctx = stb.Context(0)
    m = inputs.sphere_mesh(level, slabs, 2.0, 0.2, seed=8)
    op = stb.Operator(ctx, stb.Mesh.from_spacetime(ctx, m), "mixed")
    A = op.export_dense()
    j = int(np.argmax(((A == 0) & (np.abs(A).sum(axis=1) > 0)[:, None]).sum(axis=0) * (A != 0).any(axis=0)))
    x = np.random.default_rng(1).normal(size=(17, m.n_tet))
    x[3, j] = 0.0
    clean = op.matvec(torch.tensor(x, device="cuda"), dtype=dtype).cpu().numpy()
    x[3, j] = bad
    y = op.matvec(torch.tensor(x, device="cuda"), dtype=dtype).cpu().numpy()
    assert np.array_equal(np.delete(y, 3, 0), np.delete(clean, 3, 0))
    sees = A[:, j] != 0
    assert sees.any() and not sees.all()
    with np.errstate(over="ignore"):
        want = np.sign(A[sees, j]) * np.float32(bad)
    assert np.array_equal(y[3, sees], want, equal_nan=True)
    x[3, j] = 0.0
    u = {"tf32": 2.0 ** -11, "bf16": 2.0 ** -8}[dtype]
    bound = (2 * u + 2 * u * u + ((A != 0).sum(axis=1) + 2) * 2.0 ** -24) * (np.abs(x[3]) @ np.abs(A).T) + 1e-300
    assert (np.abs(y[3] - x[3] @ A.T) / bound)[~sees].max() <= 1.0
