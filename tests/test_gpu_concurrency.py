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
