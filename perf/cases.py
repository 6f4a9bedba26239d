"""The work that programs built on this library have it do, as measurable cases.

A program meshes the lateral boundary of a scatterer, assembles the retarded
single layer operator, forms right-hand sides, and solves; between these it
multiplies with the operator (residuals, inner iterations, several right-hand
sides at once) and it does the same for many small scatterers together. Each
case is one such call on one mesh:

  assemble  Operator(...) and one product with it (what the new operator says)
  product   y = A x with an operator at hand, in one of the product arithmetics
  rhs       the right-hand sides of a set of plane pulses
  solve     the densities of one operator for some right-hand sides
  batch     Batch(...) of small scatterers and the densities of all of them

Meshes: icospheres ("sphere", 20 * 4^level triangles) and boxes ("cube",
12 * level^2 triangles, with many coplanar panel pairs) times `slabs` time
slabs of [0, T] with jittered interior time nodes.

Products in FP32, TF32 and BF16 are FP32 sums widened to the FP64 vectors of
the call, so they are returned as the FP32 numbers they are; mixed operators
have single precision values, and the densities computed with them are kept
in single precision.
"""
import math

import numpy as np
import torch

import paper_2103_16841_gb300 as stb
from paper_2103_16841_gb300 import inputs

_ctx = None


def _context():
    global _ctx
    if _ctx is None:
        _ctx = stb.Context(0)
    return _ctx


def listed():
    return [
        # the FP64 operator of the smallest benchmark workload: validation runs
        {"name": "assemble_fp64_sphere1x4", "call": "assemble", "surface": "sphere", "level": 1, "slabs": 4, "T": 2.0,
         "precision": "fp64", "m_q": 3},
        # one small scatterer of a serving mix, an odd number of slabs: latency counts
        {"name": "assemble_mixed_sphere1x9", "call": "assemble", "surface": "sphere", "level": 1, "slabs": 9, "T": 4.0,
         "precision": "mixed", "m_q": 3},
        # a box: one sixth of the panel pairs are coplanar
        {"name": "assemble_mixed_cube5x10", "call": "assemble", "surface": "cube", "level": 5, "slabs": 10, "T": 2.5,
         "precision": "mixed", "m_q": 3},
        # the benchmark's column height (32 slabs) on a coarser sphere
        {"name": "assemble_mixed_sphere2x32", "call": "assemble", "surface": "sphere", "level": 2, "slabs": 32, "T": 4.0,
         "precision": "mixed", "m_q": 3},
        # the benchmark's surface (level 3, 1280 triangles) with fewer slabs
        {"name": "assemble_mixed_sphere3x8", "call": "assemble", "surface": "sphere", "level": 3, "slabs": 8, "T": 4.0,
         "precision": "mixed", "m_q": 3},
        # the inner iterations of a solve for one right-hand side
        {"name": "product_fp32_sphere3x8_1", "call": "product", "surface": "sphere", "level": 3, "slabs": 8, "T": 4.0,
         "precision": "mixed", "dtype": "fp32", "nrhs": 1},
        # the FP64 residuals of a refined solve, a ragged number of right-hand sides
        {"name": "product_fp64_sphere2x15_5", "call": "product", "surface": "sphere", "level": 2, "slabs": 15, "T": 4.0,
         "precision": "mixed", "dtype": "fp64", "nrhs": 5},
        # many pulses at once on the tensor cores, the benchmark's 64 and a ragged 13
        {"name": "product_tf32_sphere2x32_64", "call": "product", "surface": "sphere", "level": 2, "slabs": 32, "T": 4.0,
         "precision": "mixed", "dtype": "tf32", "nrhs": 64},
        {"name": "product_bf16_sphere3x8_13", "call": "product", "surface": "sphere", "level": 3, "slabs": 8, "T": 4.0,
         "precision": "mixed", "dtype": "bf16", "nrhs": 13},
        # the right-hand sides of the benchmark's 64 pulses
        {"name": "rhs_sphere2x32_64", "call": "rhs", "surface": "sphere", "level": 2, "slabs": 32, "T": 4.0,
         "precision": "mixed", "nrhs": 64},
        # a solve as the benchmark does it: FP32 inner iterations, FP64 refinement
        {"name": "solve_mixed_sphere2x6_4", "call": "solve", "surface": "sphere", "level": 2, "slabs": 6, "T": 3.0,
         "precision": "mixed", "inner": "fp32", "nrhs": 4, "tol": 1e-8},
        # small ellipsoid scatterers assembled and solved together
        {"name": "batch_mixed_8", "call": "batch", "surface": "sphere", "level": 1, "slabs": 8, "T": 4.0,
         "precision": "mixed", "inner": "fp32", "count": 8, "tol": 1e-8},
    ]


def _log_int(rng, lo, hi):
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    most = {"assemble": _inner(listed()[4]), "product": _inner(listed()[4]), "rhs": _inner(listed()[3]),
            "solve": _inner(listed()[10]), "batch": 1.3 * _inner({"surface": "sphere", "level": 1, "slabs": 16, "T": 4.0}),
            "fp64": 4e7}
    while True:
        call = rng.choice(["assemble", "assemble", "assemble", "product", "product", "rhs", "solve", "batch"])
        c = {"call": call, "surface": rng.choice(["sphere", "sphere", "cube"])}
        # about 12 ... 1280 triangles
        target = math.exp(rng.uniform(math.log(12.0), math.log(1300.0)))
        if c["surface"] == "sphere":
            c["level"] = min(3, max(0, int(round(math.log(target / 20.0, 4.0)))))
        else:
            c["level"] = min(8, max(1, int(round(math.sqrt(target / 12.0)))))
        c["slabs"] = _log_int(rng, 2, 32)
        c["T"] = round(rng.uniform(1.5, 4.0), 2)
        c["precision"] = "fp64" if rng.random() < 0.2 else "mixed"
        limit = most[call]
        if call == "assemble":
            c["m_q"] = rng.choice([3, 3, 3, 2, 4])
        elif call == "product":
            c["dtype"] = rng.choice(["fp64", "fp32", "tf32", "bf16"])
            c["nrhs"] = _log_int(rng, 1, 64)
        elif call == "rhs":
            c["nrhs"] = _log_int(rng, 1, 64)
        elif call == "solve":
            c["surface"], c["level"] = "sphere", min(2, max(1, c["level"] // 2 + 1))
            c["slabs"] = min(16, c["slabs"] + 2)
            c["inner"] = rng.choice(["fp64", "fp32"])
            c["nrhs"] = _log_int(rng, 1, 5)
            c["tol"] = 1e-10 if c["precision"] == "fp64" else 1e-8
        else:
            c["surface"], c["level"] = "sphere", rng.choice([0, 1, 1])
            c["slabs"] = rng.randint(5, 10)
            c["precision"], c["inner"], c["tol"] = "mixed", "fp32", 1e-8
            c["count"] = rng.randint(2, 8)
        if c["precision"] == "fp64":
            limit = min(limit, most["fp64"])
        if c["surface"] == "cube" and c["precision"] == "mixed":
            limit = min(limit, _inner(listed()[2]))
        if _inner(c) <= limit:
            return c


# ---------------------------------------------------------------------------
# meshes
# ---------------------------------------------------------------------------

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


def _surface(case):
    return inputs.icosphere(case["level"]) if case["surface"] == "sphere" else _cube(case["level"])


def _mesh(case, seed):
    v, f = _surface(case)
    return inputs.prism_mesh(v, f, case["slabs"], case["T"], 0.2, seed=seed + 1)


def _scatterers(case, seed):
    """Ellipsoids with seeded semi-axes in [0.5, 1.5]: (mesh, pulses) each."""
    out = []
    for k in range(case["count"]):
        axes = 0.5 + inputs.uniform(1000 + seed, 3, 3 * k)
        v, f = inputs.ellipsoid(case["level"], axes)
        m = inputs.prism_mesh(v, f, case["slabs"] + k % 3, case["T"], 0.2, seed=seed * 131 + k + 1)
        out.append((m, inputs.pulse_params(1 + k % 4, seed=seed * 137 + k + 2)))
    return out


def _sizes(case):
    """(triangles, panels, faces with nu_t != 0)"""
    n_tri = 20 * 4 ** case["level"] if case["surface"] == "sphere" else 12 * case["level"] ** 2
    return n_tri, 3 * n_tri * case["slabs"], n_tri * (3 * case["slabs"] + 1)


def _inner(case):
    """Estimate of the (outer point, panel) integrals of one assembly."""
    n_tri, n_tet, n_surf = _sizes(case)
    area = 12.57 if case["surface"] == "sphere" else 6.0
    h, dt = math.sqrt(2.3 * area / n_tri), case["T"] / case["slabs"]
    per = min(3.0 * case["slabs"], 3.0 * (1.0 + 2.2 * h / dt))
    return 0.7 * n_surf * n_tri * case.get("m_q", 3) ** 2 * per


def _x(n, nrhs, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    shape = (n,) if nrhs == 1 else (nrhs, n)
    return torch.randn(shape, dtype=torch.float64, device="cuda", generator=g)


# ---------------------------------------------------------------------------
# a case's state, one pass, and its necessary work
# ---------------------------------------------------------------------------

def prepare(case, seed):
    ctx, call = _context(), case["call"]
    s = {"case": case, "ctx": ctx}
    if call == "batch":
        members = _scatterers(case, seed)
        s["meshes"] = [stb.Mesh.from_spacetime(ctx, m) for m, _ in members]
        s["params"] = [p for _, p in members]
        return s
    m = _mesh(case, seed)
    s["mesh"] = stb.Mesh.from_spacetime(ctx, m)
    if call == "assemble":
        s["x"] = _x(m.n_tet, 1, seed)
        return s
    s["op"] = stb.Operator(ctx, s["mesh"], case["precision"])
    if call == "product":
        s["x"] = _x(m.n_tet, case["nrhs"], seed)
    else:
        s["params"] = inputs.pulse_params(case["nrhs"], seed=seed + 2)
        if call == "solve":
            s["b"] = s["op"].rhs(stb.DATA_PULSE, s["params"])
    return s


def run(state):
    c = state["case"]
    call, mixed = c["call"], c["precision"] == "mixed"
    if call == "assemble":
        op = stb.Operator(state["ctx"], state["mesh"], c["precision"], m_q=c["m_q"])
        return op.matvec(state["x"], dtype="fp32").float() if mixed else op.matvec(state["x"])
    if call == "product":
        y = state["op"].matvec(state["x"], dtype=c["dtype"])
        return y if c["dtype"] == "fp64" else y.float()
    if call == "rhs":
        return state["op"].rhs(stb.DATA_PULSE, state["params"])
    kept = np.float32 if mixed else np.float64
    if call == "solve":
        w, _ = state["op"].solve(state["b"], tol=c["tol"], inner=c["inner"])
        return w.astype(kept)
    batch = stb.Batch(state["ctx"], state["meshes"], c["precision"])
    ws, _ = batch.solve(state["params"], tol=c["tol"], inner=c["inner"])
    return [w.astype(kept) for w in ws]


# one (outer point, panel) integral: about 1.3 conic arcs or clipped edges of
# four nodes each at some 40 operations, and the crossings they start from
_FLOPS_PER_INNER = 250


def work(case):
    call = case["call"]
    if call == "batch":
        per = [work(dict(case, call="solve", slabs=case["slabs"] + k % 3, nrhs=1 + k % 4)) for k in range(case["count"])]
        asm = [work(dict(case, call="assemble", slabs=case["slabs"] + k % 3)) for k in range(case["count"])]
        return {k: sum(p[k] for p in per + asm) for k in ("bytes", "flops")}
    n_tri, n_tet, n_surf = _sizes(case)
    nnz = _inner(case) / case.get("m_q", 3) ** 2   # about one entry per (face, panel)
    item = 8 if case["precision"] == "fp64" else 4
    mesh = 150 * n_tet
    if call == "assemble":
        return {"bytes": 2 * nnz * item + mesh + 16 * n_tet, "flops": _inner(case) * _FLOPS_PER_INNER + 2 * nnz}
    if call == "product":
        item = {"fp64": item, "fp32": 4, "tf32": 4, "bf16": 2}[case["dtype"]]
        return {"bytes": nnz * item + 16 * n_tet * case["nrhs"], "flops": 2 * nnz * case["nrhs"]}
    if call == "rhs":   # 64 nodes of some 30 operations per face and pulse
        return {"bytes": 8 * n_tet * case["nrhs"] + mesh, "flops": 64 * 30 * n_surf * case["nrhs"]}
    # about 60 products and Gram-Schmidt steps of 30 basis vectors each
    return {"bytes": 60 * (nnz * item + 30 * 8 * n_tet * case["nrhs"]),
            "flops": 60 * case["nrhs"] * (2 * nnz + 30 * 8 * n_tet)}


# ---------------------------------------------------------------------------
# the same in 64 bits, from the definition: the potential of a face's
# half-infinite column in polar coordinates around the apex's foot point,
#   W(x) = int dphi int_{lit rho} rho / r drho = int dphi (r(b) - r(a)),
# Gauss-Legendre in phi between the angles where the lit radii change course
# ---------------------------------------------------------------------------

_COMBOS = 4.5e8    # largest number of (outer point, face) pairs looked at


def _rule(mq):
    p = []
    for off, last in ((1.0 / 3.0, mq), (2.0 / 3.0, mq - 1)):
        for i in range(mq):
            for j in range(last - i):
                p.append(((i + off) / mq, (j + off) / mq))
    return torch.tensor(p, dtype=torch.float64, device="cuda")


def _nodes(n):
    x, w = np.polynomial.legendre.leggauss(n)
    s, w = 0.5 * (x + 1.0), 0.5 * w
    # phi = a + (b - a) (3 s^2 - 2 s^3): square roots at the ends become smooth
    return (torch.tensor(3 * s ** 2 - 2 * s ** 3, device="cuda"), torch.tensor(w * 6 * s * (1 - s), device="cuda"))


def _potentials(q, d, g, c, nodes):
    """int dphi (r(b) - r(a)) for corners q [n, 3, 2] relative to the foot
    point, heights d, face gradients g [n, 2] and c = t - P(foot)."""
    two_pi = 2.0 * math.pi
    e = torch.roll(q, -1, 1) - q                     # edges k: q_k -> q_k+1
    ang = [torch.atan2(q[..., 1], q[..., 0])]
    # the conic |y|^2 + d^2 = (c - <g, y>)^2 on the edges
    gq, ge = (q * g[:, None]).sum(-1), (e * g[:, None]).sum(-1)
    lin0 = c[:, None] - gq
    a2 = (e * e).sum(-1) - ge ** 2
    b2 = (q * e).sum(-1) + lin0 * ge
    c2 = (q * q).sum(-1) + (d ** 2)[:, None] - lin0 ** 2
    root = torch.sqrt(torch.clamp(b2 ** 2 - a2 * c2, min=0.0))
    for sgn in (-1.0, 1.0):
        lam = torch.clamp(torch.nan_to_num((-b2 + sgn * root) / a2, nan=0.0, posinf=1.0, neginf=0.0), 0.0, 1.0)
        y = q + lam[..., None] * e
        ang.append(torch.atan2(y[..., 1], y[..., 0]))
    # tangents to the conic (<g, n>^2 = 1 - c^2 / d^2) and asymptotes (<g, n> = +-1)
    gn, pg = torch.sqrt((g * g).sum(-1)), torch.atan2(g[:, 1], g[:, 0])
    tang = torch.sqrt(torch.clamp(1.0 - (c / torch.where(d == 0, torch.ones_like(d), d)) ** 2, min=0.0))
    for level in (tang, torch.ones_like(tang)):
        for sgn in (-1.0, 1.0):
            ac = torch.acos(torch.clamp(sgn * level / torch.clamp(gn, min=1e-300), -1.0, 1.0))
            ang.append(torch.stack((pg + ac, pg - ac), 1))
    ang = torch.sort(torch.remainder(torch.cat(ang, 1), two_pi), 1)[0]
    ang = torch.cat((ang, ang[:, :1] + two_pi), 1)
    area2 = e[:, 0, 0] * e[:, 1, 1] - e[:, 0, 1] * e[:, 1, 0]
    nrm = torch.stack((e[..., 1], -e[..., 0]), -1) * torch.sign(area2)[:, None, None]   # outer normals
    off = (nrm * q).sum(-1)                          # <nrm, y> <= off inside
    X, Wt = nodes
    span = torch.diff(ang, dim=1)
    phi = ang[:, :-1, None] + span[..., None] * X    # [n, interval, node]
    co, si = torch.cos(phi), torch.sin(phi)
    nrm, off, g, c, d2 = (t[..., None, None] for t in (nrm, off, g, c, d ** 2))
    lo, hi = torch.zeros_like(phi), torch.full_like(phi, 1e30)
    for m in range(3):                               # the triangle on the ray
        v = nrm[:, m, 0] * co + nrm[:, m, 1] * si
        r = off[:, m] / v
        hi = torch.where(v > 0, torch.minimum(hi, r), hi)
        lo = torch.where(v < 0, torch.maximum(lo, r), lo)
        lo = torch.where((v == 0) & (off[:, m] < 0), 1e30, lo)
    gp = g[:, 0] * co + g[:, 1] * si
    A, B = 1.0 - gp ** 2, c * gp
    disc = c ** 2 - d2 * A
    sq = torch.sqrt(torch.clamp(disc, min=0.0))
    r1, r2 = (-B - sq) / A, (-B + sq) / A
    ra, rb = torch.minimum(r1, r2), torch.maximum(r1, r2)
    ell = A > 0
    dark = ell & ((disc <= 0) | (c - 0.5 * (ra + rb) * gp <= 0))
    lo = torch.where(ell, torch.maximum(lo, ra), torch.where(gp < 0, torch.maximum(lo, rb), lo))
    hi = torch.where(ell, torch.minimum(hi, rb), torch.where(gp > 0, torch.minimum(hi, ra), hi))
    ok = (hi > lo) & ~dark
    lo, hi = torch.where(ok, lo, 0.0), torch.where(ok, hi, 0.0)
    f = (hi - lo) * (hi + lo) / (torch.sqrt(hi ** 2 + d2) + torch.sqrt(lo ** 2 + d2) + 1e-300)
    return ((f * Wt).sum(2) * span).sum(1)


def _exact_matrix(m, mq):
    """Dense Galerkin matrix of a space-time prism mesh in 64 bits."""
    dev = "cuda"
    f8 = dict(dtype=torch.float64, device=dev)
    tri = torch.tensor(np.sort(m.tri, axis=1).astype(np.int64), device=dev)
    X = torch.tensor(m.svert, **f8)[tri]                                 # [K, 3, 3]
    tn = torch.tensor(m.tnodes, **f8)
    ns, K = m.n_slabs, tri.shape[0]
    # faces of a column: after n slabs with the first s corners lifted, s = 0, 1, 2
    P = []
    for n in range(ns):
        for s in range(3):
            P.append(torch.stack([tn[tri[:, k], n + (1 if k < s else 0)] for k in range(3)], 1))
    P.append(torch.stack([tn[tri[:, k], ns] for k in range(3)], 1))
    P = torch.stack(P, 1)                                                # [K, F, 3]
    F = P.shape[1]
    e1, e2 = X[:, 1] - X[:, 0], X[:, 2] - X[:, 0]
    nv = torch.linalg.cross(e1, e2)
    area = 0.5 * nv.norm(dim=1)
    nv = nv / nv.norm(dim=1, keepdim=True)
    u = e1 / e1.norm(dim=1, keepdim=True)
    v = torch.linalg.cross(nv, u)
    Q = torch.stack((torch.zeros(K, 2, **f8), torch.stack(((e1 * u).sum(1), torch.zeros(K, **f8)), 1),
                     torch.stack(((e2 * u).sum(1), (e2 * v).sum(1)), 1)), 1)    # [K, 3, 2]
    g0 = (P[..., 1] - P[..., 0]) / Q[:, None, 1, 0]
    g1 = (P[..., 2] - P[..., 0] - g0 * Q[:, None, 2, 0]) / Q[:, None, 2, 1]
    G = torch.stack((g0, g1), -1)                                        # [K, F, 2]
    xi = _rule(mq)
    Xq = X[:, None, 0] + xi[None, :, :1] * e1[:, None] + xi[None, :, 1:] * e2[:, None]      # [K, q, 3]
    Tq = P[..., None, 0] + xi[:, 0] * (P[..., None, 1] - P[..., None, 0]) + xi[:, 1] * (P[..., None, 2] - P[..., None, 0])
    nq = xi.shape[0]
    U = torch.zeros(K, F, K, F, **f8)                                    # sum over q of W: [I, f, J, s]
    nodes = _nodes(14)

    def potentials(*a):
        return torch.cat([_potentials(*(t[i:i + 50000] for t in a), nodes) for i in range(0, a[1].shape[0], 50000)])

    for I in range(K):
        rel = Xq[I][:, None] - X[None, :, 0]                             # [q, K, 3]
        d = (rel * nv).sum(-1)
        d = torch.where(d.abs() < 1e-13, 0.0, d)
        foot = torch.stack(((rel * u).sum(-1), (rel * v).sum(-1)), -1)
        q = Q[None] - foot[:, :, None]                                   # [q, K, 3, 2]
        r = torch.sqrt((q * q).sum(-1) + (d * d)[..., None])             # [q, K, 3]
        # every triangle fully lit
        zero = torch.zeros(nq * K, **f8)
        full = potentials(q.reshape(-1, 3, 2), d.reshape(-1), torch.zeros(nq * K, 2, **f8), zero + 1e6).reshape(nq, K)
        e = torch.roll(q, -1, 2) - q
        s = torch.sign(e[..., 0, 0] * e[..., 1, 1] - e[..., 0, 1] * e[..., 1, 0])[..., None]
        out = s * (e[..., 1] * q[..., 0] - e[..., 0] * q[..., 1]) / e.norm(dim=-1)
        far = torch.clamp(-out, min=0.0).amax(-1)                        # distance to the nearest edge line outside
        rmin = torch.sqrt(d * d + far * far)
        t = Tq[I][:, :, None, None]                                      # [F, q, 1, 1]
        cone = P[None, None] + r[None, :, :, None] - t[..., None]        # [F, q, K, F, 3]
        lit = (cone < 0).all(-1)
        cut = ~lit & (P.amin(-1)[None, None] + rmin[None, ..., None] < t)
        W = torch.where(lit, full[None, ..., None], 0.0)
        f, iq, j, k = cut.nonzero(as_tuple=True)
        if f.numel():
            c = Tq[I, f, iq] - (P[j, k, 0] + (G[j, k] * foot[iq, j]).sum(-1))
            W[f, iq, j, k] = potentials(q[iq, j], d[iq, j], G[j, k], c)
        U[I] = W.sum(1)
    D = U[:, :, :, :-1] - U[:, :, :, 1:]                                 # panel = between two faces
    D = D[:, :-1] - D[:, 1:]
    A = D * (area / (4.0 * math.pi * nq))[:, None, None, None]
    return A.reshape(K * (F - 1), K * (F - 1))


def _exact_rhs(m, params):
    """Right-hand sides of plane pulses: composite 12 x 12 Gauss rules per face."""
    tri, ns = np.sort(m.tri, axis=1), m.n_slabs
    X = torch.tensor(m.svert, device="cuda")[torch.tensor(tri.astype(np.int64), device="cuda")]
    tn = torch.tensor(m.tnodes, device="cuda")
    tr = torch.tensor(tri.astype(np.int64), device="cuda")
    area2 = torch.linalg.cross(X[:, 1] - X[:, 0], X[:, 2] - X[:, 0]).norm(dim=1)
    x, w = np.polynomial.legendre.leggauss(12)
    x, w = 0.5 * (x + 1.0), 0.5 * w
    pts, wts, sub = [], [], 4
    for p in range(sub):
        for q in range(sub - p):
            for c in ([(p, q), (p + 1, q), (p, q + 1)], [(p + 1, q), (p + 1, q + 1), (p, q + 1)])[:1 if p + q == sub - 1 else 2]:
                for a in range(12):
                    for b in range(12):
                        l0, l1, l2 = 1 - x[a], x[a] * (1 - x[b]), x[a] * x[b]
                        z = [(l0 * c[0][k] + l1 * c[1][k] + l2 * c[2][k]) / sub for k in (0, 1)]
                        pts.append((1 - z[0] - z[1], z[0], z[1]))
                        wts.append(w[a] * w[b] * x[a] / sub ** 2)
    bary, wts = torch.tensor(pts, device="cuda"), torch.tensor(wts, device="cuda")
    Y = torch.einsum("pk,tkc->tpc", bary, X)
    prm = torch.tensor(params, device="cuda")
    S = []
    for f in range(3 * ns + 1):
        n, s = divmod(f, 3)
        P = torch.stack([tn[tr[:, k], n + (1 if k < s else 0)] for k in range(3)], 1)
        t = P @ bary.T                                                   # [tri, points]
        S.append(torch.stack([(torch.exp(-((t - Y @ p[:3] - p[3]) / p[4]) ** 2) @ wts) * area2 for p in prm], 1))
    S = torch.stack(S, 1)                                                # [tri, faces, rhs]
    return (S[:, :-1] - S[:, 1:]).reshape(-1, prm.shape[0])


def exact(case, seed):
    call, mq = case["call"], case.get("m_q", 3)
    if call == "rhs":
        return _exact_rhs(_mesh(case, seed), inputs.pulse_params(case["nrhs"], seed=seed + 2)).cpu().numpy()
    members = case.get("count", 1)
    _, _, n_surf = _sizes(dict(case, slabs=case["slabs"] + (2 if members > 2 else 0)))
    if members * n_surf ** 2 * mq ** 2 > _COMBOS:
        return None
    if call == "batch":
        out = []
        for m, prm in _scatterers(case, seed):
            out.append(torch.linalg.solve(_exact_matrix(m, mq), _exact_rhs(m, prm)).cpu().numpy())
        return out
    m = _mesh(case, seed)
    A = _exact_matrix(m, mq)
    if call == "solve":
        b = _exact_rhs(m, inputs.pulse_params(case["nrhs"], seed=seed + 2))
        return torch.linalg.solve(A, b).cpu().numpy()
    x = _x(m.n_tet, case.get("nrhs", 1), seed)
    return x @ A.T
