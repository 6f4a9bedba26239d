"""Matrix-free operators: what they hold, and their products with either scratch."""
import numpy as np
import pytest

from paper_2103_16841_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import paper_2103_16841_gb300 as stb
    return stb.Context(0)


def test_memory_of_matrix_free_operators(ctx):
    """An operator whose values would take 200 MB holds 64 MiB of scratch and its
    sparsity structure (outer points of 46 faces on 320 triangles, 9 points of 48
    bytes each; 28 bytes for each of 320^2 blocks: 10 MB), in granules of 2 MiB an
    array; products use the context's scratch and leave nothing behind."""
    import paper_2103_16841_gb300 as stb
    mesh = stb.Mesh.from_spacetime(ctx, inputs.sphere_mesh(2, 15, 4.0, 0.2, seed=1))
    x = torch.randn(mesh.n_tet, dtype=torch.float64, device="cuda")
    first = stb.Operator(ctx, mesh, "mixed", matrix_free=True)
    y = first.matvec(x)
    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info()[0]
    ops = [stb.Operator(ctx, mesh, "mixed", matrix_free=True) for _ in range(3)]
    for op in ops:
        op.matvec(x, y)
    torch.cuda.synchronize()
    assert free - torch.cuda.mem_get_info()[0] <= 3 * (96 << 20)


@pytest.mark.parametrize("precision", ["mixed", "fp64"])
def test_products_with_either_scratch(ctx, precision):
    """With the context's scratch, with the operator's own (the allocation-free
    entry point, and a product beside unfinished work of another stream on the
    context's), and several at once on one context: the assembled matrix's entries
    summed in FP64 in some order, within (2 n + 4) 2^-53 of |A| |x|."""
    import paper_2103_16841_gb300 as stb
    mesh = stb.Mesh.from_spacetime(ctx, inputs.sphere_mesh(1, 9, 4.0, 0.2, seed=3))
    A = stb.Operator(ctx, mesh, precision).export_dense()
    ops = [stb.Operator(ctx, mesh, precision, matrix_free=True) for _ in range(3)]
    x = torch.randn((2, mesh.n_tet), dtype=torch.float64, device="cuda")
    torch.cuda.synchronize()
    xs = x.cpu().numpy()
    ref, bound = xs @ A.T, (2 * (A != 0).sum(axis=1) + 4) * 2.0 ** -53 * (np.abs(xs) @ np.abs(A).T) + 1e-300
    streams = [torch.cuda.Stream() for _ in ops]
    ys = []
    for _ in range(3):
        for op, s in zip(ops, streams):          # side by side, an operator on one stream
            ys.append(torch.empty_like(x))
            op.matvec(x, ys[-1], stream=s)
    torch.cuda.synchronize()
    for op in ops:
        ys.append(torch.empty_like(x))
        op.matvec_noalloc(x, ys[-1])
        torch.cuda.synchronize()
    for y in ys:
        assert (np.abs(y.cpu().numpy() - ref) <= bound).all()
