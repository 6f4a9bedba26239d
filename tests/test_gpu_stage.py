"""The staged quadrature and the pattern pass at the edges of their ranges:
the smallest column, the largest (192 panels, 193 faces: U of the FP64
operator leaves shared memory), word edges of the pattern bits, every m_Q,
coplanar columns, and several test columns per work item of the pattern pass."""
import os

import numpy as np
import pytest

import oracle
from paper_2103_16841_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import paper_2103_16841_gb300 as stb
    return stb.Context(0)


def _square(m):
    """[0, 1]^2 in the plane z = 0, m x m squares of two triangles."""
    v = np.array([[i / m, j / m, 0.0] for i in range(m + 1) for j in range(m + 1)])
    f = []
    for i in range(m):
        for j in range(m):
            a, b, c, d = i * (m + 1) + j, (i + 1) * (m + 1) + j, (i + 1) * (m + 1) + j + 1, i * (m + 1) + j + 1
            f += [(a, b, c), (a, c, d)]
    return v, np.array(f, dtype=np.int32)


@pytest.mark.parametrize("surface,level,slabs,T,mq", [
    ("sphere", 0, 1, 0.5, 3), ("sphere", 0, 64, 4.0, 3), ("sphere", 0, 21, 2.0, 4), ("sphere", 0, 11, 2.0, 1),
    ("square", 1, 11, 2.0, 2), ("square", 10, 1, 0.3, 3)])
def test_entries_and_pattern(ctx, surface, level, slabs, T, mq):
    """Pattern bit-exact; FP64 entries within 1e-11 of the oracle's, relative
    to the largest (the error of the parity tests); mixed entries within 1e-5
    of the FP64 ones (FP32 face geometry, about 1e-6, with a margin of 10)."""
    import paper_2103_16841_gb300 as stb
    v, f = inputs.icosphere(level) if surface == "sphere" else _square(level)
    m = inputs.prism_mesh(v, f, slabs, T, 0.2, seed=7)
    om = oracle.Mesh.from_spacetime(m)
    mesh = stb.Mesh.from_spacetime(ctx, m)
    rng = np.random.default_rng(1)
    rows = np.sort(rng.choice(m.n_tet, min(24, m.n_tet), replace=False)).astype(np.int32)
    want = om.pattern_rows(rows, mq=mq)
    ops = {p: stb.Operator(ctx, mesh, p, m_q=mq) for p in ("fp64", "mixed")}
    for op in ops.values():
        for a, b in zip(op.pattern_rows(rows), want):
            assert np.array_equal(a, b)
    ij = np.array([(r, c) for r, cols in zip(rows, want) for c in rng.choice(cols, min(40, len(cols)), replace=False)])
    out = np.array([(r, c) for r, cols in zip(rows, want) for c in np.setdiff1d(np.arange(m.n_tet), cols)[:20]])
    ref = om.entries(ij, mq=mq, nthreads=os.cpu_count())
    scale = np.abs(ref).max()
    assert np.abs(ops["fp64"].entries(ij) - ref).max() <= 1e-11 * scale
    assert np.abs(ops["mixed"].entries(ij) - ref).max() <= 1e-5 * scale
    for op in ops.values():
        assert out.size == 0 or np.all(op.entries(out) == 0.0)
        assert op.check()[0] == 0


@pytest.mark.parametrize("level,slabs,T,width", [(0, 1, 0.2, 4.0), (0, 3, 2.0, 0.25), (1, 5, 3.0, 0.05), (1, 2, 1.0, 0.5)])
def test_rhs_over_the_refinement_levels(ctx, level, slabs, T, width):
    """Right-hand sides from one level (no split of the triangles) to the
    deepest (4), with pulses far outside the time window (results that
    underflow) among them, against the oracle: 1e-12 of the largest (the bound
    of the parity test)."""
    import paper_2103_16841_gb300 as stb
    m = inputs.sphere_mesh(level, slabs, T, 0.2, seed=4)
    op = stb.Operator(ctx, stb.Mesh.from_spacetime(ctx, m), "fp64")
    prm = inputs.pulse_params(5, seed=3, width=width)
    prm[3, 3] = 60.0
    g = op.rhs(stb.DATA_PULSE, prm)
    r = oracle.Mesh.from_spacetime(m).rhs(stb.DATA_PULSE, prm)
    assert np.abs(g - r).max() <= 1e-12 * np.abs(r).max()
    assert np.array_equal(op.rhs(stb.DATA_PULSE, prm), g)


@pytest.mark.parametrize("level,slabs", [(0, 1), (0, 2), (0, 3), (1, 4), (0, 64), (1, 21)])
@pytest.mark.parametrize("precision", ["fp64", "mixed"])
def test_products_over_the_column_sizes(ctx, level, slabs, precision):
    """Products for column sizes of every divisor (rows per thread 1, 2, 4), one
    slot to many, a cluster of CTAs per column, and ragged groups of right-hand
    sides, against the exported matrix: FP64 accumulation within n 2^-53, FP32
    within (n + 2) 2^-24 of |A| |x| (n the row's entries; the classical bound of a
    sum in any order)."""
    import paper_2103_16841_gb300 as stb
    m = inputs.sphere_mesh(level, slabs, 2.0, 0.2, seed=5)
    op = stb.Operator(ctx, stb.Mesh.from_spacetime(ctx, m), precision)
    A = op.export_dense()
    row = (A != 0).sum(axis=1)
    for nrhs in (1, 3, 4, 5, 9):
        x = np.random.default_rng(nrhs).normal(size=(nrhs, m.n_tet))
        ref, mag = x @ A.T, np.abs(x) @ np.abs(A).T
        for dtype, u in (("fp64", 2.0 ** -53), ("fp32", 2.0 ** -24)):
            y = op.matvec(torch.tensor(x, device="cuda"), dtype=dtype).cpu().numpy()
            assert np.all(np.abs(y - ref) <= (2 * row + 4) * u * mag + 1e-300), (nrhs, dtype)


@pytest.mark.parametrize("level,slabs", [(0, 1), (0, 14), (0, 42), (0, 43), (0, 64), (1, 3), (1, 16), (2, 2)])
@pytest.mark.parametrize("dtype", ["tf32", "bf16"])
def test_tensor_core_products_over_the_row_groups(ctx, level, slabs, dtype):
    """Tensor-core products with one to many columns per 128-row tile, tiles
    that are full, nearly full and exceeded (129 rows: two tiles), and groups
    split over several CTAs, row by row within the rounding of the operands and
    of an FP32 sum: (2 u + 2 u^2 + (n + 2) 2^-24) |A| |x|."""
    import paper_2103_16841_gb300 as stb
    m = inputs.sphere_mesh(level, slabs, 2.0, 0.2, seed=8)
    op = stb.Operator(ctx, stb.Mesh.from_spacetime(ctx, m), "mixed")
    A = op.export_dense()
    u = {"tf32": 2.0 ** -11, "bf16": 2.0 ** -8}[dtype]
    for nrhs in (1, 17, 64):
        x = np.random.default_rng(nrhs).normal(size=(nrhs, m.n_tet))
        y = op.matvec(torch.tensor(x, device="cuda"), dtype=dtype).cpu().numpy()
        bound = (2 * u + 2 * u * u + ((A != 0).sum(axis=1) + 2) * 2.0 ** -24) * (np.abs(x) @ np.abs(A).T) + 1e-300
        assert (np.abs(y - x @ A.T) / bound).max() <= 1.0, nrhs
    assert op.check()[0] == 0
