"""Device memory short while a context keeps its quadrature scratch."""
import gc

import numpy as np
import pytest

from paper_2103_16841_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("call", ["solve", "tf32", "matrix_free"])
def test_idle_scratch_is_given_back(call):
    """An assembly of 14,400 panels leaves 1 GiB of scratch with its context. With
    less than that free elsewhere, a solve whose basis takes 0.7 GB (32 right-hand
    sides, 200 steps), a TF32 product with its tables and slots (0.2 GB) and another
    operator all find room."""
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import paper_2103_16841_gb300 as stb
    gc.collect()
    ctx = stb.Context(0)
    mesh = stb.Mesh.from_spacetime(ctx, inputs.sphere_mesh(2, 15, 4.0, 0.2, seed=1))
    op = stb.Operator(ctx, mesh, "mixed")
    b = np.random.default_rng(0).normal(size=(mesh.n_tet, 32))
    x = torch.tensor(np.ascontiguousarray(b.T), device="cuda")

    def solve(restart):
        return op.solve(b, tol=1e-14, restart=restart, maxit=2, inner="fp64", allow_unconverged=True)[0]

    small = solve(2)                       # (kernels and small buffers are there)
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    left = {"solve": 500, "tf32": 64, "matrix_free": 32}[call] << 20
    hold = torch.empty(torch.cuda.mem_get_info()[0] - left, dtype=torch.uint8, device="cuda")
    try:
        if call == "solve":
            assert np.isfinite(solve(200)).all()
        elif call == "tf32":
            y = torch.empty_like(x[:1])
            op.matvec(x[:1].contiguous(), y, dtype="tf32")
            torch.cuda.synchronize()
            assert bool(torch.isfinite(y).all())
        else:
            stb.Operator(ctx, mesh, "mixed", matrix_free=True).close()
    finally:
        del hold
        torch.cuda.empty_cache()
    assert np.isfinite(small).all()


def test_right_hand_sides_in_a_small_workspace():
    """220,000 right-hand sides of 60 panels with 400 MB free: 0.22 GB for them in
    both panel orders and their parameters, and no workspace of 0.28 GB beside
    that. The same bits as in pieces."""
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import paper_2103_16841_gb300 as stb
    ctx = stb.Context(0)
    op = stb.Operator(ctx, stb.Mesh.from_spacetime(ctx, inputs.sphere_mesh(0, 1, 0.5, 0.2, seed=2)), "mixed")
    prm = inputs.pulse_params(220000, seed=3, width=4.0)
    pieces = [op.rhs(stb.DATA_PULSE, prm[i:i + 40000]) for i in range(0, len(prm), 40000)]
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    hold = torch.empty(torch.cuda.mem_get_info()[0] - (400 << 20), dtype=torch.uint8, device="cuda")
    try:
        b = op.rhs(stb.DATA_PULSE, prm)
    finally:
        del hold
        torch.cuda.empty_cache()
    assert np.array_equal(b, np.concatenate(pieces, axis=1))


def test_calls_after_one_that_found_no_memory():
    """A refused call leaves nothing behind that a later launch would report."""
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import paper_2103_16841_gb300 as stb
    ctx = stb.Context(0)
    mesh = stb.Mesh.from_spacetime(ctx, inputs.sphere_mesh(2, 15, 4.0, 0.2, seed=1))
    op = stb.Operator(ctx, stb.Mesh.from_spacetime(ctx, inputs.sphere_mesh(0, 1, 0.5, 0.2, seed=2)), "mixed")
    prm = inputs.pulse_params(3, seed=3)
    want = op.rhs(stb.DATA_PULSE, prm)
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    hold = torch.empty(torch.cuda.mem_get_info()[0] - (64 << 20), dtype=torch.uint8, device="cuda")
    try:
        with pytest.raises(stb._lib.BemError):
            stb.Operator(ctx, mesh, "mixed")
        assert np.array_equal(op.rhs(stb.DATA_PULSE, prm), want)
    finally:
        del hold
        torch.cuda.empty_cache()
