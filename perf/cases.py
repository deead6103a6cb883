"""The cases this framework's speed is measured on.

Each case is one call (or one step) that a user's program makes through the
public entry points of paper_1608_04607_gb300.dfm, on the jittered Kuhn meshes
of paper_1608_04607_gb300.inputs: assembly of the operator, its application
inside a user's own iteration (one vector, many, several damping moments, the
high orders of the cuboid verification), the interior density of every tet, a
differentiable solve, a whole step of a many-source job, and a small stationary
solve.  The solves run the low-precision preconditioner, the Krylov vectors and
the adjoint contraction as a user's program reaches them.  `exact` restates
every path in plain torch in 64 bits (where its FP64 assembly takes seconds).

    listed()            the cases
    draw(rng)           another case of the same ranges
    prepare(case, seed) mesh, operator, vectors: what a program holds before the call
    run(state)          one pass
    work(case)          bytes and operations a pass cannot do without
    exact(case, seed)   the outputs in 64 bits, or None
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1608_04607_gb300 import dfm
from paper_1608_04607_gb300 import inputs

REFL = 0.95   # boundary reflection of every cube workload
MU = 0.05     # uniform damping of the cube workloads, and the median of the log-normal field
MU_FIT = 0.5  # median damping of the gradient steps, between the cubes' 0.05 .. 0.2 and the cuboid's 0.4 pi
MU_C = 0.1    # expansion point of the damping moments
CUBOID_MU = 0.4 * math.pi  # the cuboid verification's damping (its walls reflect fully)

_STORE = {"f32": dfm.F32, "bf16": dfm.BF16, "f64": dfm.F64}


def listed():
    return [
        # a coarse mesh re-assembled with a new damping field, as in a parameter study
        dict(name="assemble-np4-1296", kind="assemble", mesh="cube", n=6, Np=4, store="f32", mu="field"),
        # the 48,000-tet workload's assembly: part of every one of its solves
        dict(name="assemble-np4-48000", kind="assemble", mesh="cube", n=20, Np=4, store="f32", mu="uniform"),
        # 45 functions with BF16 blocks, the storage of the many-source workload
        dict(name="assemble-np8-24576-bf16", kind="assemble", mesh="cube", n=16, Np=8, store="bf16", mu="uniform"),
        # one high order of the cuboid verification (153 functions)
        dict(name="assemble-np16-768", kind="assemble", mesh="cuboid", n=4, Np=16, store="f32", mu="uniform"),
        # one operator application of a user's own Krylov iteration
        dict(name="apply-np4-48000", kind="apply", mesh="cube", n=20, Np=4, R=1, trans=False, x0=True),
        # the same for a block of 16 sources with 45 functions
        dict(name="apply-np8-24576-r16", kind="apply", mesh="cube", n=16, Np=8, R=16, trans=False, x0=True),
        # sources with a damping of their own: three damping moments applied together
        dict(name="combo-np4-48000-r16", kind="combo", mesh="cube", n=20, Np=4, R=16, K=3),
        # the application that the cuboid verification's solve repeats some 300 times
        dict(name="apply-np16-768", kind="apply", mesh="cuboid", n=4, Np=16, R=1, trans=False, x0=True),
        # the density's coefficients at every tet's centroid (the read-out of a solve)
        dict(name="density-np4-6000", kind="density", mesh="cube", n=10, Np=4),
        # one gradient step on per-tet damping through torch.autograd: assembly, solve, adjoint, contraction
        dict(name="gradient-np4-48000", kind="gradient", mesh="cube", n=20, Np=4),
        # one step of a many-source job: assembly, block solve of 16 sources, adjoint, every source's gradient
        dict(name="job-np8-3072-r16", kind="job", mesh="cube", n=8, Np=8, R=16),
        # the smallest use: the unit cube of six tets, Neumann series in FP64
        dict(name="neumann-np2-6", kind="solve64", mesh="cube", n=1, Np=2, method="neumann", tol=1e-10),
    ]


# what a drawn case may cost at most: bytes moved, or 50 operations in the place of a byte
_MOST = 1.4e11


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    while True:
        kind = rng.choice(["assemble", "assemble", "wide", "wide", "apply", "apply", "combo", "density", "gradient",
                           "gradient", "job", "solve64"])
        if kind == "assemble":
            c = dict(kind="assemble", mesh="cube", n=_log_int(rng, 2, 20), Np=rng.randint(1, 8),
                     store=rng.choice(["f32", "f32", "bf16"]), mu=rng.choice(["field", "uniform"]))
        elif kind == "wide":
            c = dict(kind=rng.choice(["assemble", "apply"]), mesh="cuboid", n=_log_int(rng, 2, 5),
                     Np=rng.randint(9, 20))
            c |= dict(store="f32", mu="uniform") if c["kind"] == "assemble" else \
                dict(R=rng.randint(1, 2), trans=False, x0=True)
        elif kind == "apply":
            c = dict(kind="apply", mesh="cube", n=_log_int(rng, 3, 24), Np=rng.randint(2, 8), R=_log_int(rng, 1, 16),
                     trans=rng.random() < 0.4, x0=rng.random() < 0.7)
        elif kind == "combo":
            c = dict(kind="combo", mesh="cube", n=_log_int(rng, 3, 20), Np=rng.randint(2, 6), R=_log_int(rng, 1, 16),
                     K=rng.randint(2, 3))
        elif kind == "density":
            c = dict(kind="density", mesh="cube", n=_log_int(rng, 2, 12), Np=rng.randint(2, 8))
        elif kind == "gradient":
            c = dict(kind="gradient", mesh="cube", n=_log_int(rng, 3, 20), Np=rng.randint(2, 6))
        elif kind == "job":
            c = dict(kind="job", mesh="cube", n=_log_int(rng, 3, 9), Np=rng.randint(3, 8), R=rng.randint(4, 16))
        else:
            c = dict(kind="solve64", mesh="cube", n=_log_int(rng, 1, 6), Np=rng.randint(1, 4),
                     method=rng.choice(["neumann", "gmres"]))
            c["tol"] = rng.choice([1e-10, 1e-12]) if c["method"] == "neumann" else 1e-12
        w = work(c)
        if max(w["bytes"], w["flops"] / 50) <= _MOST:
            return c


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
def _mesh(case, seed):
    if case["mesh"] == "cuboid":
        return inputs.kuhn_cuboid_mesh(case["n"], seed=seed), 1.0
    if case["n"] == 1:  # no interior vertex to move: the six tets are scaled instead
        m = inputs.kuhn_cube_mesh(1, jitter=0.0)
        s = 1.0 + 0.2 * np.random.Generator(np.random.PCG64(seed)).uniform(-1, 1, size=3)
        return inputs.KuhnMesh(verts=m.verts * s, tets=m.tets, n=1, h=1.0), 0.9
    return inputs.kuhn_cube_mesh(case["n"], jitter=0.2, seed=seed), REFL


def _field(m, seed, median=MU):
    """Log-normal damping per tet, in the FP32 of a parameter that is fitted."""
    return torch.from_numpy(inputs.lognormal_mu(m, median=median, seed=seed + 1).astype(np.float32)).cuda()


def _taylor(case, seed):
    """Weights (mu_r - mu_c)^k / k! of the damping moments, mu_r ~ U[0.01, 0.2]."""
    mu = np.random.Generator(np.random.PCG64(seed + 3)).uniform(0.01, 0.2, size=case["R"])
    return np.stack([(mu - MU_C) ** k / math.factorial(k) for k in range(case["K"])], 1)


def _vectors(shape, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    return torch.randn(shape, generator=g, device="cuda", dtype=torch.float32)


def _uniform_mu(case):
    return CUBOID_MU if case["mesh"] == "cuboid" else (0.1 if case["n"] == 1 else MU)


def _receiver(m):
    c = m.n // 2
    return inputs.cell_tets(m, max(0, c - 1), c + 1)


def _sources(m, count, seed):
    return inputs.random_boundary_rows(m, count, seed=seed + 2)


def prepare(case, seed):
    m, refl = _mesh(case, seed)
    mesh = dfm.Mesh(m.verts, m.tets, refl=refl)
    kind, Np, nb = case["kind"], case["Np"], dfm.nbasis(case["Np"])
    s = dict(kind=kind, case=case, mesh=mesh)
    if kind == "assemble":
        s["mu"] = _field(m, seed) if case["mu"] == "field" else _uniform_mu(case)
        s["op"] = dfm.Operator(mesh, Np, mu=_uniform_mu(case), precision=_STORE[case["store"]])
    elif kind in ("apply", "combo"):
        if kind == "apply":
            s["op"] = dfm.Operator(mesh, Np, mu=_uniform_mu(case))
        else:
            s["ops"] = [dfm.Operator(mesh, Np, mu=MU_C, moment=k) for k in range(case["K"])]
            s["coef"] = _taylor(case, seed)
        s["x"] = _vectors((case["R"], mesh.n_rows, nb), seed)
        s["x0"] = _vectors((case["R"], mesh.n_rows, nb), seed + 1) if case.get("x0", True) else None
        s["out"] = torch.empty_like(s["x"])
    elif kind == "density":
        s["mu"] = _field(m, seed).double()
        s["tets"] = np.arange(m.n_tets)
    elif kind in ("gradient", "job"):
        rec = _receiver(m)
        s["mu"] = _field(m, seed, MU_FIT)
        s["rho0"] = dfm.source(mesh, Np, _sources(m, case.get("R", 1), seed))
        s["g"], s["dg"] = dfm.interior_density(mesh, Np, rec, weights=1.0 / len(rec), mu=s["mu"])
        if kind == "job":
            s["op"] = dfm.Operator(mesh, Np, mu=MU_FIT)
        else:
            s["mu"].requires_grad_(True)
    else:
        s["op"] = dfm.Operator(mesh, Np, mu=_uniform_mu(case), precision=dfm.F64)
        s["rho0"] = dfm.source(mesh, Np, _sources(m, 1, seed))
    return s


def run(s):
    kind, c = s["kind"], s["case"]
    if kind == "assemble":
        s["op"].reassemble(s["mu"])
        return s["op"].blocks()
    if kind == "apply":
        return s["op"].apply(s["x"], x0=s["x0"], trans=c["trans"], out=s["out"])
    if kind == "combo":
        return dfm.apply_combo(s["ops"], s["coef"], s["x"], x0=s["x0"], out=s["out"])
    if kind == "density":
        return dfm.interior_density(s["mesh"], c["Np"], s["tets"], mu=s["mu"])
    if kind == "gradient":
        mu = s["mu"]
        mu.grad = None
        rho = dfm.DFMSolve.apply(s["mesh"], c["Np"], mu, s["rho0"], 1e-8, precond_precision=dfm.FP8E4M3)
        (s["g"] * rho[0]).sum().backward()
        return mu.grad
    if kind == "job":
        op, kw = s["op"], dict(tol=1e-8, restart=24, poly_degree=64, precond_precision=dfm.FP8E4M3)
        op.reassemble(s["mu"])
        rho, _ = op.solve(s["rho0"], batch=c["R"], block=1, **kw)
        _, dj, _ = op.adjoint(rho, s["g"], s["dg"], **kw)
        return dj.to(s["mu"].dtype)  # a gradient has its parameter's type
    if c["method"] == "neumann":
        return s["op"].solve(s["rho0"], method=dfm.NEUMANN, tol=c["tol"])[0]
    return s["op"].solve(s["rho0"], method=dfm.GMRES, tol=c["tol"], poly_degree=32, restart=256)[0]


# ---------------------------------------------------------------------------
# work
# ---------------------------------------------------------------------------
def _tets(case):
    return (12 if case["mesh"] == "cuboid" else 6) * case["n"] ** 3


def _assembly_work(case, eb):
    """Blocks written once; per quadrature node the rank-1 update, the two
    Zernike vectors and the node's geometry (about 14 patches per face pair)."""
    nt, Np = _tets(case), case["Np"]
    nb = dfm.nbasis(Np)
    nodes = 12 * nt * 14 * (Np + 6) ** 2
    return nt * (12 * nb * nb * eb + 160.0), nodes * (2.0 * nb * nb + 2 * (6 * Np + 4 * nb) + 130)


def _apply_bytes(case, eb, R, vectors, vb):
    rows, nb = 4 * _tets(case), dfm.nbasis(case["Np"])
    return rows * (3.0 * nb * nb * eb + 4 + vectors * R * nb * vb)


def work(case):
    kind, Np, nt = case["kind"], case["Np"], _tets(case)
    nb = dfm.nbasis(Np)
    eb = {"f32": 4, "bf16": 2, "f64": 8}.get(case.get("store"), 4)
    mac = 2.0 * 3 * nb * nb * 4 * nt  # one operator application to one vector
    if kind == "assemble":
        b, f = _assembly_work(case, eb)
    elif kind == "apply":
        b, f = _apply_bytes(case, 4, case["R"], 3 if case["x0"] else 2, 4), mac * case["R"]
    elif kind == "combo":
        b, f = _apply_bytes(case, 4 * case["K"], case["R"], 3, 4), mac * case["R"] * case["K"]
    elif kind == "density":  # 3,456 nodes per face
        b, f = nt * (8.0 * 8 * nb + 4 * 128 + 32), 4.0 * nt * 3456 * (4 * nb + 40)
    elif kind in ("gradient", "job"):  # assembly, contraction, some 400 hops on an 8-bit copy each way
        b, f = _assembly_work(case, 4)
        R = case.get("R", 1)
        b += 400 * (_apply_bytes(case, 1, R, 3, 2) + _apply_bytes(case, 1, 1, 3, 2))
        f = 1.2 * f + 400 * mac * (R + 1)
    else:  # about 150 applications
        b, f = 150 * _apply_bytes(case, 8, 1, 3, 8), 150 * mac
    return {"bytes": b, "flops": f}


# ---------------------------------------------------------------------------
# the same in 64 bits, in plain torch
# ---------------------------------------------------------------------------
# operations of an FP64 assembly that stay within about ten seconds
_EXACT_FLOPS = 6.0e12


def _topology(tets):
    """recv[4t + f]: the row across face f of tet t, or 4t + f itself on the boundary."""
    nt = tets.shape[0]
    faces = np.sort(np.stack([tets[:, [(f + 1) % 4, (f + 2) % 4, (f + 3) % 4]] for f in range(4)], 1).reshape(-1, 3), 1)
    order = np.lexsort(faces.T[::-1])
    s = faces[order]
    same = np.nonzero(np.all(s[1:] == s[:-1], axis=1))[0]
    recv = np.arange(4 * nt)
    recv[order[same]], recv[order[same + 1]] = order[same + 1], order[same]
    return recv


def _unit(v):
    return v / v.norm(dim=-1, keepdim=True)


def _frames(V, T):
    """Per row: first face vertex, e1, e2, inward normal, area."""
    P = torch.stack([torch.stack([V[T[:, (f + 1 + k) % 4]] for k in range(3)], 1) for f in range(4)], 1)  # nt,4,3,3
    e1 = _unit(P[:, :, 1] - P[:, :, 0])
    cr = torch.linalg.cross(P[:, :, 1] - P[:, :, 0], P[:, :, 2] - P[:, :, 0])
    area = 0.5 * cr.norm(dim=-1)
    n = _unit(cr)
    inward = ((V[T] - P[:, :, 0]) * n).sum(-1, keepdim=True)
    n = torch.where(inward < 0, -n, n)
    return P, e1, torch.linalg.cross(n, e1), n, area


def _zernike(Np, x, y):
    """Z_n^m (m = -n, -n + 2, .., n) at points of the disc: [..., nb]."""
    r2 = x * x + y * y
    c, s = [torch.ones_like(x)], [torch.zeros_like(x)]
    for _ in range(Np):
        c, s = c + [c[-1] * x - s[-1] * y], s + [c[-1] * y + s[-1] * x]
    Q, out = {}, []
    for n in range(Np + 1):
        for m in range(n & 1, n + 1, 2):
            if m == n:
                Q[n, m] = torch.ones_like(x)
            elif m == 0:
                Q[n, m] = 2 * r2 * Q[n - 1, 1] - Q[n - 2, 0]
            else:
                Q[n, m] = Q[n - 1, m - 1] + r2 * Q[n - 1, m + 1] - Q[n - 2, m]
        out += [Q[n, abs(m)] * (c[m] if m >= 0 else s[-m]) for m in range(-n, n + 1, 2)]
    return torch.stack(out, -1)


def _invnorm(Np, dev):
    v = [(2 * n + 2) / ((2 if m == 0 else 1) * math.pi) for n in range(Np + 1) for m in range(-n, n + 1, 2)]
    return torch.tensor(v, dtype=torch.float64, device=dev)


def _phi2(k, x):
    """k-th derivative of phi2(x) = (x - 1 + e^-x) / x^2 by its series (x is below 4 here)."""
    s = torch.zeros_like(x)
    for j in range(45, -1, -1):
        c = math.factorial(j + k) / (math.factorial(j) * math.factorial(j + k + 2))
        s = s * x + (-1) ** (j + k) * c
    return s


def _split(P):
    """The four children of spherical polygons [N, nv, 3] by edge midpoints."""
    nv = P.shape[1]
    mid = [_unit(P[:, k] + P[:, (k + 1) % nv]) for k in range(nv)]
    if nv == 3:
        kids = [(P[:, 0], mid[0], mid[2]), (mid[0], P[:, 1], mid[1]), (mid[2], mid[1], P[:, 2]), tuple(mid)]
    else:
        c = _unit(P.sum(1))
        kids = [(P[:, 0], mid[0], c, mid[3]), (mid[0], P[:, 1], mid[1], c), (c, mid[1], P[:, 2], mid[2]),
                (mid[3], c, mid[2], P[:, 3])]
    return torch.cat([torch.stack(k, 1) for k in kids])


def _assemble64(m, refl, Np, mu, orders=(0,)):
    """(recv, [d^k B / dmu^k for k in orders]), each [rows, 3, nb, nb]: row R's
    three blocks, in the order of the source faces of tet recv[R] / 4 (its exit
    face left out).  The rule is the framework's: Gauss order Np + 6 on
    patches of at most 60 degrees (five levels)."""
    dev = "cuda"
    V = torch.as_tensor(m.verts, dtype=torch.float64, device=dev)
    T = torch.as_tensor(m.tets, dtype=torch.int64, device=dev)
    recv = torch.as_tensor(_topology(m.tets), device=dev)
    nt, nb = T.shape[0], dfm.nbasis(Np)
    P, e1, e2, n, area = _frames(V, T)
    mu = torch.as_tensor(mu, dtype=torch.float64, device=dev).expand(nt)
    t = torch.arange(nt, device=dev).repeat_interleave(12)
    f = torch.arange(4, device=dev).repeat_interleave(3).repeat(nt)
    k = torch.arange(3, device=dev).repeat(4 * nt)
    fp = k + (k >= f)
    R = recv[4 * t + fp]
    axes = torch.stack([e1[t, f], e2[t, f], n[t, f]], 1)  # source frame
    loc = torch.einsum("pvc,pac->pva", V[T[t]] - P[t, f, 0][:, None], axes)
    pick = torch.arange(t.shape[0], device=dev)
    others = [(f + j) % 4 for j in (1, 2, 3)]
    b = torch.where(others[0] != fp, others[0], others[1])
    c = torch.where(others[2] != fp, others[2], others[1])
    A, B, C, D = loc[pick, fp], loc[pick, b], loc[pick, c], loc[pick, f]

    def form(X, Y, Z):  # s_X(d) = m_X . d
        zy = Z - Y
        den = zy[:, 0] * (X - Y)[:, 1] - zy[:, 1] * (X - Y)[:, 0]
        beta = (zy[:, 0] * (D - Y)[:, 1] - zy[:, 1] * (D - Y)[:, 0]) / den
        return torch.stack([D[:, 2] * zy[:, 1] / den, -D[:, 2] * zy[:, 0] / den, beta], 1)

    forms = torch.stack([form(A, B, C), form(B, C, A), form(C, A, B)], 1)
    rec = torch.stack([e1.reshape(-1, 3)[R], e2.reshape(-1, 3)[R]], 1)
    rec = torch.einsum("pkc,pac->pka", rec, axes)
    boundary = R == 4 * t + fp
    scale = torch.where(boundary, refl, 1.0) / torch.sqrt(area[t, f] * area[t, fp])
    tri = torch.cat([torch.stack([D - A, D - B, D - C], 1), torch.stack([D - A, B - A, C - A], 1)])
    quad = torch.cat([torch.stack([D - A, D - B, C - B, C - A], 1), torch.stack([D - A, D - C, B - C, B - A], 1)])
    patches, owner = [], []
    for polys in (_unit(tri), _unit(quad)):
        own = pick.repeat(2)
        for depth in range(5):
            edge = (polys * polys.roll(-1, 1)).sum(-1).amin(1)
            cut = (edge < math.cos(math.pi / 3)) & (depth < 4)
            four = polys if polys.shape[1] == 4 else torch.cat([polys, polys[:, :1]], 1)
            patches.append(four[~cut])
            owner.append(own[~cut])
            polys, own = _split(polys[cut]), own[cut].repeat(4)
    patches, owner = torch.cat(patches), torch.cat(owner)
    q = Np + 6
    gx, gw = (torch.as_tensor(v, device=dev) for v in np.polynomial.legendre.leggauss(q))
    xi, eta = gx[:, None].expand(q, q).reshape(-1, 1), gx[None].expand(q, q).reshape(-1, 1)
    w2 = (gw[:, None] * gw[None]).reshape(-1)
    out = [torch.zeros((t.shape[0], nb, nb), dtype=torch.float64, device=dev) for _ in orders]
    chunk = max(1, int(1.5e8 / (q * q * nb)))
    for i in range(0, patches.shape[0], chunk):
        v, o = patches[i:i + chunk], owner[i:i + chunk]
        v1, v2, v3, v4 = (v[:, j, None] for j in range(4))
        ca, cb, cc, cd = 0.25 * (v1 + v2 + v3 + v4), 0.25 * (v2 - v1 + v3 - v4), 0.25 * (v3 + v4 - v1 - v2), \
            0.25 * (v3 - v4 + v1 - v2)
        F = ca + cb * xi + cc * eta + cd * xi * eta
        det = (F * torch.linalg.cross(cb + cd * eta, cc + cd * xi)).sum(-1)
        r = F.norm(dim=-1)
        jac = (F[..., 2] * det).abs() / r ** 4
        d = F / r[..., None]
        sA, sB, sC = torch.einsum("pnc,pkc->kpn", d, forms[o])
        ok = sA > 0
        den = torch.where(ok, sA + sB.clamp(min=0) + sC.clamp(min=0), 1.0)
        LO = D[o, 2, None] / den
        w = torch.where(ok, w2 * jac * 2 * area[t, f][o, None] * sA / den, 0.0)
        x = mu[t][o, None] * LO
        Zp = _zernike(Np, d[..., 0], d[..., 1])
        p = torch.einsum("pnc,pkc->kpn", d, rec[o])
        Zq = _zernike(Np, p[0], p[1]).transpose(1, 2)
        for k, res in zip(orders, out):
            res.index_add_(0, o, torch.bmm(Zq * (w * LO ** k * _phi2(k, x))[:, None], Zp))
    slot = f - (f > fp).long()
    blocks = []
    for blk in out:
        full = torch.zeros((4 * nt, 3, nb, nb), dtype=torch.float64, device=dev)
        full[R, slot] = blk * scale[:, None, None] * _invnorm(Np, dev)[:, None]
        blocks.append(full)
    return recv, blocks


def _source_rows(recv):
    """[rows, 3]: the rows whose coefficients row R reads."""
    e = recv % 4
    k = torch.arange(3, device=recv.device)
    return 4 * (recv // 4)[:, None] + k + (k >= e[:, None]).long()


def _apply64(B, src, x, trans=False):
    """B x or B^T x for x [R, rows, nb]."""
    R, rows, nb = x.shape
    if not trans:
        full = B.permute(0, 2, 1, 3).reshape(rows, nb, 3 * nb)
        return torch.bmm(full, x[:, src].reshape(R, rows, 3 * nb).permute(1, 2, 0)).permute(2, 0, 1)
    z = torch.bmm(B.permute(0, 1, 3, 2).reshape(rows, 3 * nb, nb), x.permute(1, 2, 0)).reshape(rows * 3, nb, R)
    y = torch.zeros((rows, nb, R), dtype=x.dtype, device=x.device).index_add_(0, src.reshape(-1), z)
    return y.permute(2, 0, 1)


def _solve64(B, src, b, trans=False):
    """(I - B)^{-1} b by the Neumann series, to an increment of 1e-14."""
    x = b.clone()
    for it in range(200000):
        y = b + _apply64(B, src, x, trans)
        if it % 50 == 0 and (y - x).norm() <= 1e-14 * y.norm():
            return y
        x = y
    return x


def _density64(m, Np, mu, tets):
    """Coefficients of the density at the centroids and their mu-derivatives:
    the split polar rule with 24 points per direction, [rows, nb] each."""
    dev, n = "cuda", 24
    V = torch.as_tensor(m.verts, dtype=torch.float64, device=dev)
    T = torch.as_tensor(m.tets, dtype=torch.int64, device=dev)
    nt, nb = T.shape[0], dfm.nbasis(Np)
    P, e1, e2, nrm, area = _frames(V, T)
    gx, gw = (torch.as_tensor(v, device=dev) for v in np.polynomial.legendre.leggauss(n))
    xa, wa = 0.5 * (gx + 1), 0.5 * gw
    g = torch.zeros((nt, 4, nb), dtype=torch.float64, device=dev)
    dg = torch.zeros_like(g)
    sel = torch.as_tensor(tets, device=dev)
    for lo in range(0, sel.shape[0], max(1, int(2e7 / (n * n * nb)))):
        e = sel[lo:lo + max(1, int(2e7 / (n * n * nb)))]
        r = V[T[e]].mean(1)
        for f in range(4):
            h = ((r - P[e, f, 0]) * nrm[e, f]).sum(-1)
            F = r - h[:, None] * nrm[e, f]
            on = (torch.linalg.cross(P[e, f, 1] - P[e, f, 0], P[e, f, 2] - P[e, f, 0]) * nrm[e, f]).sum(-1)
            XY = torch.stack([((P[e, f] - F[:, None]) * a[e, f][:, None]).sum(-1) for a in (e1, e2)], -1)
            for edge in range(3):
                a, b = XY[:, edge], XY[:, (edge + 1) % 3]
                t = _unit(b - a)
                d = (a[:, 0] * t[:, 1] - a[:, 1] * t[:, 0]).abs()
                sgn = torch.sign(a[:, 0] * b[:, 1] - a[:, 1] * b[:, 0]) * torch.where(on >= 0, 1.0, -1.0)
                uA, uB = (a * t).sum(-1), (b * t).sum(-1)
                M = a - uA[:, None] * t
                cc = torch.sqrt(h * h + d * d)
                sA, sB = torch.atan2(uA, cc), torch.atan2(uB, cc)
                cut = torch.where((sA < 0) & (sB > 0), 0.0, 0.5 * (sA + sB))
                for s0, s1 in ((sA, cut), (cut, sB)):
                    s = s0[:, None] + (s1 - s0)[:, None] * xa
                    u = cc[:, None] * torch.tan(s)
                    ell = torch.sqrt(d[:, None] ** 2 + u * u)
                    ex = (M[:, None] + u[..., None] * t[:, None]) / ell[..., None]
                    jac = (s1 - s0)[:, None] * wa * (cc * d)[:, None] / (torch.cos(s) ** 2 * ell ** 2)
                    Phi = torch.atan2(ell, h[:, None])
                    phi = Phi[..., None] * xa
                    w = (sgn[:, None] * jac * Phi)[..., None] * wa * torch.sin(phi)
                    w = torch.where((d > 1e-15 * (b - a).norm(dim=-1))[:, None, None], w, 0.0)
                    dist = h[:, None, None] / torch.cos(phi)
                    ker = w * torch.exp(-mu[e][:, None, None] * dist)
                    Z = _zernike(Np, -torch.sin(phi) * ex[..., 0, None], -torch.sin(phi) * ex[..., 1, None])
                    g[e, f] += torch.einsum("eab,eabz->ez", ker, Z)
                    dg[e, f] -= torch.einsum("eab,eabz->ez", ker * dist, Z)
    s = 1 / torch.sqrt(area)[..., None]
    return (g * s).reshape(-1, nb), (dg * s).reshape(-1, nb)


def exact(case, seed):
    kind, Np = case["kind"], case["Np"]
    m, refl = _mesh(case, seed)
    nb, rows = dfm.nbasis(Np), 4 * m.n_tets
    if kind == "density":
        if 4.0 * m.n_tets * 3456 * nb > 3e9:
            return None
        g, dg = _density64(m, Np, _field(m, seed).double(), np.arange(m.n_tets))
        return [g, dg]
    if _assembly_work(case, 8)[1] * (2 if kind in ("gradient", "job") else case.get("K", 1)) > _EXACT_FLOPS:
        return None
    if kind == "assemble":
        mu = _field(m, seed) if case["mu"] == "field" else _uniform_mu(case)
        return _assemble64(m, refl, Np, mu)[1][0]
    if kind == "apply":
        recv, (B,) = _assemble64(m, refl, Np, _uniform_mu(case))
        shape = (case["R"], rows, nb)
        y = _apply64(B, _source_rows(recv), _vectors(shape, seed).double(), case["trans"])
        return y + _vectors(shape, seed + 1).double() if case["x0"] else y
    if kind == "combo":
        recv, Bs = _assemble64(m, refl, Np, MU_C, range(case["K"]))
        src, shape = _source_rows(recv), (case["R"], rows, nb)
        x, coef = _vectors(shape, seed).double(), torch.as_tensor(_taylor(case, seed), device="cuda")
        return _vectors(shape, seed + 1).double() + sum(
            _apply64(B, src, x) * coef[:, k, None, None] for k, B in enumerate(Bs))
    if kind == "solve64":
        recv, (B,) = _assemble64(m, refl, Np, _uniform_mu(case))
        _, _, _, _, area = _frames(torch.as_tensor(m.verts, device="cuda"),
                                   torch.as_tensor(m.tets, dtype=torch.int64, device="cuda"))
        row = int(_sources(m, 1, seed)[0])
        b = torch.zeros((1, rows, nb), dtype=torch.float64, device="cuda")
        b[0, row, 0] = torch.sqrt(area.reshape(-1)[row])
        return _solve64(B, _source_rows(recv), b)
    # gradient, job: dJ/dmu_t = lambda . dB/dmu_t rho (+ dg . rho of the tet for a job)
    mu = _field(m, seed, MU_FIT).double()
    recv, (B, dB) = _assemble64(m, refl, Np, mu, (0, 1))
    src = _source_rows(recv)
    _, _, _, _, area = _frames(torch.as_tensor(m.verts, device="cuda"),
                               torch.as_tensor(m.tets, dtype=torch.int64, device="cuda"))
    rec = _receiver(m)
    g, dg = (v / len(rec) for v in _density64(m, Np, mu, rec))
    at = torch.as_tensor(_sources(m, case.get("R", 1), seed), device="cuda")
    b = torch.zeros((at.shape[0], rows, nb), dtype=torch.float64, device="cuda")
    b[torch.arange(at.shape[0], device="cuda"), at, 0] = torch.sqrt(area.reshape(-1)[at])
    rho = _solve64(B, src, b)
    lam = _solve64(B, src, g[None], trans=True)[0]
    per_row = (_apply64(dB, src, rho) * lam).sum(-1)  # [R, rows], belonging to tet recv / 4
    grad = torch.zeros((at.shape[0], m.n_tets), dtype=torch.float64, device="cuda").index_add_(1, recv // 4, per_row)
    if kind == "job":
        return grad + (dg * rho).sum(-1).reshape(at.shape[0], m.n_tets, 4).sum(-1)
    return grad[0]
