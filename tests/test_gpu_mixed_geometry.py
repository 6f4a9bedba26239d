"""Mixed operators form an apex's relative position, height, foot point and
corner distances in FP64; the FP32 face integrals start from their roundings."""
import os

import numpy as np
import pytest

from paper_2103_16841_gb300 import inputs

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
HERE = os.path.dirname(os.path.abspath(__file__))


def _cube(m):
    """Unit cube centred at the origin, each face m x m squares of two triangles."""
    ids, verts, tri = {}, [], []

    def vid(p):
        if p not in ids:
            ids[p] = len(verts)
            verts.append([q / m - 0.5 for q in p])
        return ids[p]

    for ax in range(3):
        for side in (0, m):
            for i in range(m):
                for j in range(m):
                    c = []
                    for u, v in ((i, j), (i + 1, j), (i + 1, j + 1), (i, j + 1)):
                        p = [0, 0, 0]
                        p[ax], p[(ax + 1) % 3], p[(ax + 2) % 3] = side, u, v
                        c.append(vid(tuple(p)))
                    if side == 0:
                        c = c[::-1]
                    tri += [(c[0], c[1], c[2]), (c[0], c[2], c[3])]
    return np.array(verts, dtype=np.float64), np.array(tri, dtype=np.int32)


def test_mixed_entries_follow_from_fp64_geometry():
    """Entries whose faces lie next to a decision of the FP32 integrals (near
    field or far, series or closed form, a root in or out) have the bits that
    FP64 geometry gives them."""
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import paper_2103_16841_gb300 as stb
    ij, want = [], []
    for line in open(os.path.join(HERE, "golden", "mixed_entries.txt")):
        if not line.startswith("#"):
            i, j, v = line.split()
            ij.append((int(i), int(j)))
            want.append(float.fromhex(v))
    v, f = _cube(3)
    ctx = stb.Context(0)
    op = stb.Operator(ctx, stb.Mesh.from_spacetime(ctx, inputs.prism_mesh(v, f, 7, 3.1, 0.2, seed=3)), "mixed", m_q=4)
    assert np.array_equal(op.entries(ij), np.array(want))
