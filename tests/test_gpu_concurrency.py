"""Calls of several threads and streams on one context."""
import threading

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


def test_async_matrix_free_solve_beside_assemblies(ctx):
    """A solve captures its matrix-free products into a graph on its own stream
    while this thread assembles on the same context: the solve reaches its
    tolerance (residual formed with the assembled operator, whose entries are the
    same numbers) and every assembly has the bits of one made alone."""
    import paper_2103_16841_gb300 as stb
    mesh = stb.Mesh.from_spacetime(ctx, inputs.sphere_mesh(1, 6, 2.0, 0.2, seed=5))
    ops = {p: stb.Operator(ctx, mesh, p) for p in ("fp64", "mixed")}
    alone = {p: op.export_dense() for p, op in ops.items()}
    free = stb.Operator(ctx, mesh, "fp64", matrix_free=True)
    b = torch.tensor(ops["fp64"].rhs(stb.DATA_PULSE, inputs.pulse_params(2, seed=3)).T.copy(), device="cuda")
    for _ in range(3):
        w, tol = torch.zeros_like(b), 1e-9
        torch.cuda.synchronize()
        req = free.solve_async(b, w, tol=tol, restart=60, stream=torch.cuda.Stream())
        n, out = 0, None
        while out is None:
            for p in alone:
                op = stb.Operator(ctx, mesh, p)
                assert np.array_equal(op.export_dense(), alone[p]), p
                op.close()
                n += 1
            out = req.wait(0.0)
        req.close()
        assert n >= 2 and out[0] == 0 and all(i["converged"] for i in out[1])
        r = (b - ops["fp64"].matvec(w)).norm(dim=1) / b.norm(dim=1)
        assert float(r.max()) <= 2 * tol


def test_assemblies_of_several_threads(ctx):
    """One assembly has the context's scratch and second stream, the others a
    block of their own: the same bits as alone."""
    import paper_2103_16841_gb300 as stb
    mesh = stb.Mesh.from_spacetime(ctx, inputs.sphere_mesh(1, 7, 3.0, 0.2, seed=6))
    kinds = [("mixed", 3), ("fp64", 2), ("mixed", 4)]

    def make(k):
        op = stb.Operator(ctx, mesh, kinds[k][0], m_q=kinds[k][1])
        A = op.export_dense()
        op.close()
        return A

    alone = [make(k) for k in range(len(kinds))]
    bad = []

    def work(k):
        try:
            for _ in range(4):
                if not np.array_equal(make(k), alone[k]):
                    bad.append((k, "other bits"))
        except Exception as e:
            bad.append((k, repr(e)))

    ts = [threading.Thread(target=work, args=(k,)) for k in range(len(kinds))]
    for t in ts:
        t.start()
    for t in ts:
        t.join()
    assert not bad, bad


def test_matrix_free_product_beside_a_capture():
    """Another thread's product, for which the context's scratch (given back
    meanwhile) is allocated again, while this one captures (global mode): the
    capture stays valid and the product is the assembled matrix's, within
    (2 n + 4) 2^-53 of |A| |x|."""
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import paper_2103_16841_gb300 as stb
    ctx = stb.Context(0)
    mesh = stb.Mesh.from_spacetime(ctx, inputs.sphere_mesh(1, 9, 4.0, 0.2, seed=7))
    large = stb.Mesh.from_spacetime(ctx, inputs.sphere_mesh(3, 8, 4.0, 0.2, seed=1))
    free = stb.Operator(ctx, mesh, "mixed", matrix_free=True)
    x = torch.randn(mesh.n_tet, dtype=torch.float64, device="cuda")
    out, y = torch.empty_like(x), torch.zeros_like(x)
    mine, other = torch.cuda.Stream(), torch.cuda.Stream()
    free.matvec(x, y, stream=other)        # (its kernels and vectors are there)
    torch.mul(x, 2.0, out=out)
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    hold = torch.empty(torch.cuda.mem_get_info()[0] - (64 << 20), dtype=torch.uint8, device="cuda")
    with pytest.raises(stb._lib.BemError):
        stb.Operator(ctx, large, "mixed")
    del hold
    torch.cuda.empty_cache()
    y.zero_()
    torch.cuda.synchronize()
    bad = []

    def work():
        try:
            free.matvec(x, y, stream=other)
        except Exception as e:
            bad.append(repr(e))

    g = torch.cuda.CUDAGraph()
    with torch.cuda.stream(mine):
        g.capture_begin()
        torch.mul(x, 3.0, out=out)
        t = threading.Thread(target=work)
        t.start()
        t.join()
        g.capture_end()
    g.replay()
    torch.cuda.synchronize()
    assert not bad, bad
    assert torch.equal(out, 3.0 * x)
    A, xs = stb.Operator(ctx, mesh, "mixed").export_dense(), x.cpu().numpy()
    bound = (2 * (A != 0).sum(axis=1) + 4) * 2.0 ** -53 * (np.abs(A) @ np.abs(xs)) + 1e-300
    assert (np.abs(y.cpu().numpy() - A @ xs) <= bound).all()
