"""Performance cases of the library: the calls its users make, from one element layer of the path
(operator, residual, smoother, transfers, V-cycle) to whole solves and batches.

Kinds of case (all through the C ABI binding):

  operator   y = M QQ^T A_L M u               (se_ax), the Krylov method's matrix product
  residual   r = M (b - QQ^T A_L u)           (se_residual), the V-cycle's residual
  smooth     s = S r                          (se_pmg_smooth), a Schwarz smoother
  transfer   rc = P^T rf and ef = P ec        (se_pmg_restrict, se_pmg_prolong)
  vcycle     z = M^-1 r                       (se_pmg_apply), one preconditioner application
  solve      A x = b                          (se_solve), FPCG or FGMRES, V-cycle in FP64, FP32 or
                                              double-float arithmetic
  batch      many problems, one graph launch  (se_batch_run)

Meshes are boxes of nx x ny x nz deformed elements (interior lattice vertices moved by up to 5% of
the element width, then the smooth sine map), as in the synthetic workloads of this repository.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2110_07663_gb300 import se

AMP = 0.05        # smooth map of the meshes
PERTURB = 0.05    # perturbation of interior vertices, fraction of the element width
SMOOTHERS = {"ras": se.SE_SMOOTH_RAS, "asm": se.SE_SMOOTH_ASM, "jacobi": se.SE_SMOOTH_JACOBI}
PRECISIONS = {"fp64": se.SE_FP64, "fp32": se.SE_FP32, "df64": se.SE_DF64}
# orders of the levels below the finest: the paper's Table 5 schedules (p, about p/2, 1) for the
# Schwarz smoothers and steps of two for Jacobi; even orders likewise
SCHWARZ_MID = {2: (), 3: (), 4: (2,), 5: (3,), 6: (3,), 7: (3,), 8: (4,), 9: (5,), 10: (5,)}
JACOBI_MID = {2: (), 3: (), 4: (2,), 5: (3,), 6: (4, 2), 7: (5, 3), 8: (6, 4, 2), 9: (7, 5, 3),
              10: (8, 6, 4, 2)}


# ------------------------------------------------------------------------------- the cases
def listed():
    return [
        # the smallest solve of the workloads (64 elements): launches and latency, no arithmetic
        dict(name="solve_box4_p7_ras", kind="solve", nx=4, ny=4, nz=4, p=7, bc="DDDDDD",
             smoother="ras", order=2, mid="3", precision="fp64", method="fpcg", graph=True, tol=1e-8),
        # the benchmark solve: 32768 elements, the preconditioner its run-time search picks
        dict(name="solve_box32_p7_jacobi", kind="solve", nx=32, ny=32, nz=32, p=7, bc="DDDDDD",
             smoother="jacobi", order=1, mid="5,3", precision="fp64", method="fpcg", graph=True,
             tol=1e-8),
        # the paper's default preconditioner with FP32 V-cycle, the order of its larger cases
        dict(name="solve_box16_p9_ras_fp32", kind="solve", nx=16, ny=17, nz=15, p=9, bc="DDDDDD",
             smoother="ras", order=2, mid="5", precision="fp32", method="fpcg", graph=True, tol=1e-8),
        # host-driven flexible GMRES(20) with additive Schwarz, the paper's outer method
        dict(name="solve_box12_p7_asm_gmres", kind="solve", nx=13, ny=12, nz=11, p=7, bc="DDDDDD",
             smoother="asm", order=2, mid="3", precision="fp64", method="fgmres", graph=False,
             tol=1e-8),
        # a batch of uneven problems in one graph launch (mixed precision)
        dict(name="batch12_mixed", kind="batch", count=12, mix=1, emin=8, emax=16, orders="3,5,7,9",
             precision="fp32", tol=1e-8),
        # the outer operator at the benchmark's size
        dict(name="operator_box32_p7", kind="operator", nx=32, ny=32, nz=32, p=7, bc="DDDDDD"),
        # a small operator call: launch-bound
        dict(name="operator_box6_p5", kind="operator", nx=6, ny=5, nz=7, p=5, bc="DDDDDD"),
        # odd point count per line (even order), ragged mesh, Neumann faces
        dict(name="residual_box19_p8_mixedbc", kind="residual", nx=19, ny=17, nz=18, p=8, bc="DNNDDN"),
        # the Schwarz smoothers of Table 5: restrictive at p = 7, additive at p = 9
        dict(name="smooth_ras_box24_p7", kind="smooth", nx=24, ny=24, nz=24, p=7, bc="DDDDDD",
             smoother="ras"),
        dict(name="smooth_asm_box11_p9", kind="smooth", nx=11, ny=13, nz=12, p=9, bc="DDDDDD",
             smoother="asm"),
        # one application of the FP64 preconditioner
        dict(name="vcycle_box20_p7_ras", kind="vcycle", nx=20, ny=20, nz=20, p=7, bc="DDDDDD",
             smoother="ras", order=2, mid="5,3", precision="fp64"),
        # both transfers between the two finest levels of a p = 9 hierarchy
        dict(name="transfer_box20_p9_p5", kind="transfer", nx=20, ny=19, nz=21, p=9, bc="DDDDDD", pc=5),
    ]


def _box(rng, points, p):
    """Elements per direction of a ragged box of about `points` local points."""
    e = max(8.0, points / (p + 1) ** 3)
    c = e ** (1.0 / 3.0)
    n = [max(2, round(c * rng.uniform(0.75, 1.3))) for _ in range(2)]
    n.append(max(2, round(e / (n[0] * n[1]))))
    rng.shuffle(n)
    return n


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    kind = rng.choice(["solve"] * 4 + ["operator"] * 2 + ["residual", "smooth", "smooth", "vcycle",
                                                          "transfer", "batch"])
    if kind == "batch":
        return dict(kind=kind, count=rng.randint(4, 16), mix=rng.randint(1, 1000), emin=rng.randint(4, 8),
                    emax=rng.randint(9, 16), orders="3,5,7,9",
                    precision=rng.choice(["fp32", "fp32", "fp64"]), tol=1e-8)
    p = rng.randint(3, 10) if kind != "solve" else rng.choice([3, 5, 6, 7, 7, 8, 9, 10])
    bc = rng.choice(["DDDDDD", "DDDDDD", "DNDDND", "NDDNDD", "DDNNDD"])
    if kind in ("operator", "residual"):
        n = _box(rng, _log(rng, 2.0e4, 1.6e7), p)
        return dict(kind=kind, nx=n[0], ny=n[1], nz=n[2], p=p, bc=bc)
    if kind == "smooth":
        n = _box(rng, _log(rng, 2.0e4, 6.0e6), p)
        return dict(kind=kind, nx=n[0], ny=n[1], nz=n[2], p=p, bc=bc, smoother=rng.choice(["ras", "asm"]))
    if kind == "transfer":
        n = _box(rng, _log(rng, 2.0e4, 1.2e7), p)
        return dict(kind=kind, nx=n[0], ny=n[1], nz=n[2], p=p, bc=bc,
                    pc=rng.choice([p - 2, (p + 1) // 2]) if p > 3 else 1)
    smoother = rng.choice(["ras", "ras", "jacobi", "asm"])
    mid = ",".join(str(q) for q in (JACOBI_MID if smoother == "jacobi" else SCHWARZ_MID)[p])
    order = rng.randint(1, 3)
    if kind == "vcycle":
        n = _box(rng, _log(rng, 2.0e4, 5.0e6), p)
        return dict(kind=kind, nx=n[0], ny=n[1], nz=n[2], p=p, bc=bc, smoother=smoother, order=order,
                    mid=mid, precision=rng.choice(["fp64", "df64"]))
    n = _box(rng, _log(rng, 3.0e4, 2.5e6), p)
    method = rng.choice(["fpcg", "fpcg", "fgmres"])
    return dict(kind=kind, nx=n[0], ny=n[1], nz=n[2], p=p, bc=bc, smoother=smoother, order=order,
                mid=mid, precision=rng.choice(["fp64", "fp64", "fp32", "df64"]), method=method,
                graph=method == "fpcg" and rng.random() < 0.7, tol=1e-8)


# ------------------------------------------------------------------------------- inputs
def _vertices(nel, seed):
    """Vertex lattice (nz+1, ny+1, nx+1, 3) of the unit box with perturbed interior vertices."""
    nx, ny, nz = nel
    c, b, a = np.meshgrid(np.arange(nz + 1) / nz, np.arange(ny + 1) / ny, np.arange(nx + 1) / nx,
                          indexing="ij")
    V = np.stack([a, b, c], axis=-1)
    move = np.random.default_rng(seed).uniform(-1.0, 1.0, V.shape) * PERTURB / np.array([nx, ny, nz])
    V[1:-1, 1:-1, 1:-1] += move[1:-1, 1:-1, 1:-1]
    return V


def _gid(nel, p, dev):
    """Global node id of every local point (L) and the lattice extents."""
    nx, ny, nz = nel
    e = torch.arange(nx * ny * nz, device=dev)
    r = torch.arange(p + 1, device=dev)
    I = ((e % nx) * p)[:, None] + r
    J = ((e // nx % ny) * p)[:, None] + r
    K = ((e // (nx * ny)) * p)[:, None] + r
    NX, NY = nx * p + 1, ny * p + 1
    g = I[:, None, None, :] + NX * (J[:, None, :, None] + NY * K[:, :, None, None])
    return g.reshape(-1), (NX, NY, nz * p + 1)


def _mask_global(ext, bc, dev):
    """1 on free lattice nodes, 0 on the Dirichlet faces (z, y, x order)."""
    NX, NY, NZ = ext
    m = torch.ones((NZ, NY, NX), dtype=torch.float64, device=dev)
    for f, sl in enumerate([(2, 0), (2, NX - 1), (1, 0), (1, NY - 1), (0, 0), (0, NZ - 1)]):
        if bc[f] == "D":
            m.select(sl[0], sl[1]).zero_()
    return m.reshape(-1)


def _continuous(nel, p, bc, seed, dev, masked=True):
    """Random continuous L-vector (one normal value per global node), zero on Dirichlet nodes:
    residuals and Krylov vectors hold every scale of the mesh."""
    gid, ext = _gid(nel, p, dev)
    g = torch.Generator(device=dev)
    g.manual_seed(seed)
    v = torch.randn(ext[0] * ext[1] * ext[2], dtype=torch.float64, device=dev, generator=g)
    if masked:
        v = v * _mask_global(ext, bc, dev)
    return v[gid]


def _nel(case):
    return case["nx"], case["ny"], case["nz"]


class _Handles:
    """Library handles of one state, destroyed with it (latest first)."""

    def __init__(self):
        self.items = []

    def add(self, h, destroy):
        self.items.append((h, destroy))
        return h

    def __del__(self):
        while self.items:
            h, destroy = self.items.pop()
            destroy(h)


def _mesh(keep, nel, p, bc, seed):
    return keep.add(se.se_mesh_create(nel, p, vertex_xyz=_vertices(nel, seed), deform_amp=AMP,
                                      bc=[0 if c == "D" else 1 for c in bc]), se.se_mesh_destroy)


def _pmg(keep, m, case, schedule):
    d = se.pmg_desc(schedule, SMOOTHERS[case["smoother"]], case.get("order", 2),
                    precision=PRECISIONS[case.get("precision", "fp64")])
    return keep.add(se.se_pmg_setup(m, d), se.se_pmg_destroy)


def _schedule(case):
    return (case["p"],) + tuple(int(q) for q in case["mid"].split(",") if q) + (1,)


def _modes(seed):
    """Eight sine modes of a smooth random forcing: wave numbers 1..4, amplitudes."""
    rng = np.random.default_rng(seed + 1)
    return rng.integers(1, 5, size=(8, 3)), rng.uniform(-1.0, 1.0, size=8) + 0.25


def _forcing(xyz, seed):
    k, a = _modes(seed)
    f = torch.zeros_like(xyz[0])
    for (kx, ky, kz), am in zip(k, a):
        f += (am * math.pi ** 2 * float(kx * kx + ky * ky + kz * kz)) * torch.sin(math.pi * int(kx) * xyz[0]) \
            * torch.sin(math.pi * int(ky) * xyz[1]) * torch.sin(math.pi * int(kz) * xyz[2])
    return f


def _rhs(m, seed, dev):
    L = se.se_mesh_get_info(m).L
    xyz = torch.empty(3 * L, dtype=torch.float64, device=dev)
    se.se_mesh_nodes(m, xyz)
    f = _forcing(xyz.view(3, -1), seed)
    b = torch.empty_like(f)
    se.se_mesh_rhs(m, f, b)
    return b


def _batch_problems(case, seed):
    """Sizes and orders are the case's (stream `mix`); meshes and forcings are the seed's."""
    rng = np.random.default_rng(case["mix"])
    orders = [int(q) for q in case["orders"].split(",")]
    return [dict(n=int(rng.integers(case["emin"], case["emax"] + 1)), p=int(rng.choice(orders)),
                 seed=seed + 100 * i) for i in range(case["count"])]


def prepare(case, seed):
    dev = torch.device("cuda:0")
    keep = _Handles()
    st = dict(case=case, keep=keep)
    if case["kind"] == "batch":
        probs = []
        for q in _batch_problems(case, seed):
            nel = (q["n"],) * 3
            m = _mesh(keep, nel, q["p"], "DDDDDD", q["seed"])
            P = _pmg(keep, m, dict(smoother="ras", order=2, precision=case["precision"]),
                     (q["p"],) + SCHWARZ_MID[q["p"]] + (1,))
            b = _rhs(m, q["seed"], dev)
            probs.append((m, P, b, torch.zeros_like(b)))
        st["x"] = [q[3] for q in probs]
        st["b"] = [q[2] for q in probs]
        st["batch"] = keep.add(se.se_batch_create(probs, tol=case["tol"]), se.se_batch_destroy)
        return st
    nel, p, bc = _nel(case), case["p"], case["bc"]
    st["m"] = m = _mesh(keep, nel, p, bc, seed)
    if case["kind"] == "solve":
        st["P"] = _pmg(keep, m, case, _schedule(case))
        st["b"] = _rhs(m, seed, dev)
        st["x"] = torch.zeros_like(st["b"])
        return st
    if case["kind"] == "transfer":
        st["P"] = _pmg(keep, m, dict(smoother="jacobi"), (p, case["pc"]) + ((1,) if case["pc"] > 1 else ()))
        st["u"] = _continuous(nel, p, bc, seed, dev)
        st["uc"] = _continuous(nel, case["pc"], bc, seed + 1, dev)
        st["y"], st["yc"] = torch.empty_like(st["u"]), torch.empty_like(st["uc"])
        return st
    st["u"] = _continuous(nel, p, bc, seed, dev)
    st["y"] = torch.empty_like(st["u"])
    if case["kind"] == "residual":
        st["b"] = _continuous(nel, p, bc, seed + 1, dev)
    elif case["kind"] == "smooth":
        st["P"] = _pmg(keep, m, case, (p,) + SCHWARZ_MID[p] + (1,))
    elif case["kind"] == "vcycle":
        st["P"] = _pmg(keep, m, case, _schedule(case))
    return st


def run(st):
    case = st["case"]
    kind = case["kind"]
    if kind == "operator":
        se.se_ax(st["m"], st["u"], st["y"], se.SE_AX_ASSEMBLE | se.SE_AX_MASK)
        return st["y"]
    if kind == "residual":
        se.se_residual(st["m"], st["b"], st["u"], st["y"])
        return st["y"]
    if kind == "smooth":
        se.se_pmg_smooth(st["P"], 0, st["u"], st["y"])
        return st["y"]
    if kind == "transfer":
        se.se_pmg_restrict(st["P"], 0, st["u"], st["yc"])
        se.se_pmg_prolong(st["P"], 0, st["uc"], st["y"])
        return {"restricted": st["yc"], "prolonged": st["y"]}
    if kind == "vcycle":
        se.se_pmg_apply(st["P"], st["u"], st["y"])
        return st["y"]
    if kind == "batch":
        for x in st["x"]:
            x.zero_()
        se.se_batch_run(st["batch"])
        return list(st["x"])
    st["x"].zero_()
    se.se_solve(st["m"], st["P"], st["b"], st["x"],
                method=se.SE_FGMRES if case["method"] == "fgmres" else se.SE_FPCG, tol=case["tol"],
                graph_capture=1 if case["graph"] else 0,
                operator_df64=1 if case["precision"] == "df64" else 0)
    return st["x"]


# ------------------------------------------------------------------------------- what a pass needs
def _elements(case):
    return case["nx"] * case["ny"] * case["nz"]


def _ax_flops(E, p):
    return E * (12.0 * (p + 1) ** 4 + 15.0 * (p + 1) ** 3)


def _smooth_flops(E, p, smoother):
    pb, n = p + 3.0, (p + 1.0 if smoother == "ras" else p + 3.0)
    if smoother == "jacobi":
        return E * (p + 1.0) ** 3
    return E * (6 * pb ** 4 + pb ** 3 + 2 * (pb ** 3 * n + pb ** 2 * n ** 2 + pb * n ** 3))


def _transfer_flops(E, pf, pc):
    f, c = pf + 1.0, pc + 1.0
    return 2 * E * (f ** 3 * c + f ** 2 * c ** 2 + f * c ** 3)


def _vcycle_flops(E, sched, smoother, order):
    fl = 0.0
    for l, p in enumerate(sched[:-1]):  # pre- and post-smoothing, two residuals, both transfers
        fl += (2 * order + 2) * _ax_flops(E, p) + 2 * (order + 1) * _smooth_flops(E, p, smoother)
        fl += 2 * _transfer_flops(E, p, sched[l + 1])
    return fl


def _factor_bytes(E, p, smoother):
    """Operator data of one level: geometric factors, and S and Lambda or the diagonal."""
    n3 = (p + 1) ** 3
    return 8.0 * E * (6 * n3 + (n3 if smoother == "jacobi" else 3 * (p + 3) ** 2 + 3 * (p + 3)))


def _solve_work(E, sched, smoother, order, iterations, iterate_bytes):
    p = sched[0]
    fl = iterations * (_vcycle_flops(E, sched, smoother, order) + _ax_flops(E, p))
    by = sum(_factor_bytes(E, q, smoother) for q in sched[:-1]) + iterate_bytes
    return by, fl


def work(case):
    """Bytes: each input, factor and output once.  Flops: the sum factorisation's; a solve counts
    the iterations such problems take (Jacobi smoothing about 10, Schwarz about 6)."""
    kind = case["kind"]
    if kind == "batch":
        by = fl = 0.0
        for q in _batch_problems(case, 0):
            E, sched = q["n"] ** 3, (q["p"],) + SCHWARZ_MID[q["p"]] + (1,)
            b, f = _solve_work(E, sched, "ras", 2, 6, 16.0 * E * (q["p"] + 1) ** 3)
            by, fl = by + b, fl + f
        return {"bytes": by, "flops": fl}
    E, p = _elements(case), case["p"]
    L = E * (p + 1) ** 3
    if kind == "operator":
        return {"bytes": 8.0 * 8 * L, "flops": _ax_flops(E, p)}
    if kind == "residual":
        return {"bytes": 8.0 * 9 * L, "flops": _ax_flops(E, p)}
    if kind == "smooth":
        return {"bytes": 16.0 * L + 8.0 * E * (3 * (p + 3) ** 2 + 3 * (p + 3)),
                "flops": _smooth_flops(E, p, case["smoother"])}
    if kind == "transfer":
        return {"bytes": 16.0 * (L + E * (case["pc"] + 1) ** 3),
                "flops": 2 * _transfer_flops(E, p, case["pc"])}
    sched = _schedule(case)
    its = 1 if kind == "vcycle" else (10 if case["smoother"] == "jacobi" else 6)
    by, fl = _solve_work(E, sched, case["smoother"], case["order"], its, 16.0 * L)
    return {"bytes": by, "flops": fl}


# ------------------------------------------------------------------------------- 64-bit reference
def _gll(p):
    """GLL points and weights: the roots of P_p' polished by Newton's method."""
    leg = np.polynomial.legendre.Legendre.basis(p)
    x = np.concatenate([[-1.0], np.sort(leg.deriv().roots().real), [1.0]]) if p > 1 else np.array([-1.0, 1.0])
    for _ in range(3):
        x[1:-1] -= leg.deriv()(x[1:-1]) / leg.deriv(2)(x[1:-1])
    x = 0.5 * (x - x[::-1])
    return x, 2.0 / (p * (p + 1) * leg(x) ** 2)


def _deriv(x):
    n = len(x)
    lam = np.array([1.0 / np.prod([x[j] - x[m] for m in range(n) if m != j]) for j in range(n)])
    D = np.array([[0.0 if i == j else lam[j] / lam[i] / (x[i] - x[j]) for j in range(n)] for i in range(n)])
    return D - np.diag(D.sum(axis=1))


def _interp(pf, pc):
    xf, xc = _gll(pf)[0], _gll(pc)[0]
    return np.array([[np.prod([(x - xc[m]) / (xc[j] - xc[m]) for m in range(pc + 1) if m != j])
                      for j in range(pc + 1)] for x in xf])


def _lines(A, u):
    """A applied along r, s and t of u [E, k, j, i] in turn."""
    return _along(A, _along(A, _along(A, u, 3), 2), 1)


def _along(A, u, dim):
    return torch.movedim(torch.movedim(u, dim, -1) @ A.T, -1, dim)


class _Ref:
    """The discrete problem on one order: operator, QQ^T, mask (torch, 64 bits)."""

    def __init__(self, nel, p, bc, V, dev):
        self.nel, self.p, self.N, self.dev = nel, p, p + 1, dev
        E = nel[0] * nel[1] * nel[2]
        self.shape = (E, p + 1, p + 1, p + 1)
        xi, w = _gll(p)
        self.D = torch.tensor(_deriv(xi), device=dev)
        self.gid, self.ext = _gid(nel, p, dev)
        ng = self.ext[0] * self.ext[1] * self.ext[2]
        self.ng = ng
        self.mask = _mask_global(self.ext, bc, dev)[self.gid].view(self.shape)
        self.mult = torch.bincount(self.gid, minlength=ng).to(torch.float64)[self.gid].view(self.shape)
        nx, ny, nz = nel
        C = np.stack([V[c:c + nz, b:b + ny, a:a + nx].reshape(E, 3) for c in (0, 1) for b in (0, 1)
                      for a in (0, 1)], axis=1).reshape(E, 2, 2, 2, 3)
        self.corners = C
        C = torch.tensor(C, device=dev)
        phi = torch.tensor(np.stack([(1.0 - xi) / 2.0, (1.0 + xi) / 2.0]), device=dev)
        X = torch.einsum("ezyxc,zk,yj,xi->cekji", C, phi, phi, phi)
        X = X + AMP * (torch.sin(2 * math.pi * X[0]) * torch.sin(2 * math.pi * X[1])
                       * torch.sin(2 * math.pi * X[2]))
        self.X = X
        J = [[_along(self.D, X[c], d) for d in (3, 2, 1)] for c in range(3)]  # dx_c / dr_a
        # grad r_a = (cofactors of J) / det J
        cof = [[J[(c + 1) % 3][(a + 1) % 3] * J[(c + 2) % 3][(a + 2) % 3]
                - J[(c + 1) % 3][(a + 2) % 3] * J[(c + 2) % 3][(a + 1) % 3] for c in range(3)] for a in range(3)]
        det = sum(J[c][0] * cof[0][c] for c in range(3))
        wt = torch.tensor(w, device=dev)
        self.W = wt[:, None, None] * wt[None, :, None] * wt[None, None, :]
        self.B = self.W * det
        self.G = {(a, b): self.W * sum(cof[a][c] * cof[b][c] for c in range(3)) / det
                  for a in range(3) for b in range(a, 3)}

    def qqt(self, u):
        return torch.zeros(self.ng, dtype=torch.float64, device=self.dev).index_add_(
            0, self.gid, u.reshape(-1))[self.gid].view(self.shape)

    def local(self, u):
        g = [_along(self.D, u, d) for d in (3, 2, 1)]
        y = 0.0
        for a, d in enumerate((3, 2, 1)):
            y = y + _along(self.D.T, sum(self.G[min(a, b), max(a, b)] * g[b] for b in range(3)), d)
        return y

    def ax(self, u):
        return self.mask * self.qqt(self.local(self.mask * u.view(self.shape)))

    def diagonal(self):
        D, G = self.D, self.G
        d = _along((D * D).T, G[0, 0], 3) + _along((D * D).T, G[1, 1], 2) + _along((D * D).T, G[2, 2], 1)
        g = torch.diagonal(D)
        d = d + 2 * (g[None, None, :] * g[None, :, None] * G[0, 1] + g[None, None, :] * g[:, None, None] * G[0, 2]
                     + g[None, :, None] * g[:, None, None] * G[1, 2])
        return self.qqt(d)


def _box_lengths(ref):
    """Mean corner-to-corner edge length of every mapped element along each direction."""
    C = ref.corners
    s = np.prod(np.sin(2 * math.pi * C), axis=-1, keepdims=True)
    C = C + AMP * s
    return np.stack([np.linalg.norm(np.take(C, 1, axis=ax) - np.take(C, 0, axis=ax), axis=-1).mean(axis=(1, 2))
                     for ax in (3, 2, 1)], axis=1)


def _schwarz_factors(ref, bc):
    """S and Lambda of the extended one-dimensional problems, per element and direction."""
    p, (nx, ny, nz) = ref.p, ref.nel
    E, N, pb = nx * ny * nz, p + 1, p + 3
    xi, w = _gll(p)
    D = _deriv(xi)
    Ke = D.T @ np.diag(w) @ D
    lens = _box_lengths(ref)
    e = np.arange(E)
    place = np.stack([e % nx, e // nx % ny, e // (nx * ny)], axis=1)
    S, lam = np.zeros((3, E, pb, pb)), np.ones((3, E, pb))
    window = np.array([p - 1] + list(range(p, 2 * p + 1)) + [2 * p + 1])
    for d in range(3):
        step = (1, nx, nx * ny)[d]
        for left in (False, True):
            for right in (False, True):
                at = np.nonzero(((place[:, d] > 0) == left) & ((place[:, d] < ref.nel[d] - 1) == right))[0]
                if not len(at):
                    continue
                A, B = np.zeros((len(at), 3 * p + 1, 3 * p + 1)), np.zeros((len(at), 3 * p + 1))
                for s in range(3):
                    if (s == 0 and not left) or (s == 2 and not right):
                        continue
                    l = lens[at + (s - 1) * step, d]
                    A[:, s * p:s * p + N, s * p:s * p + N] += (2.0 / l)[:, None, None] * Ke
                    B[:, s * p:s * p + N] += (l / 2.0)[:, None] * w
                act = [q for q in range(pb)
                       if not (q == 0 and not left) and not (q == pb - 1 and not right)
                       and not (q == 1 and not left and bc[2 * d] == "D")
                       and not (q == pb - 2 and not right and bc[2 * d + 1] == "D")]
                i = window[act]
                bi = 1.0 / np.sqrt(B[:, i])
                v, Q = np.linalg.eigh(bi[:, :, None] * A[:, i[:, None], i[None, :]] * bi[:, None, :])
                Sa = np.zeros((len(at), pb, pb))
                Sa[:, act, :len(act)] = bi[:, :, None] * Q
                S[d][at] = Sa
                lam[d][at, :len(act)] = v
    return [torch.tensor(S[d], device=ref.dev) for d in range(3)], [torch.tensor(lam[d], device=ref.dev) for d in range(3)]


def _schwarz(ref, bc, r, kind):
    p, (nx, ny, nz), pb = ref.p, ref.nel, ref.p + 3
    NX, NY, NZ = ref.ext
    S, lam = _schwarz_factors(ref, bc)
    g = torch.zeros(ref.ng, dtype=torch.float64, device=ref.dev)
    g[ref.gid] = r.reshape(-1)
    pad = torch.zeros((NZ + 2, NY + 2, NX + 2), dtype=torch.float64, device=ref.dev)
    pad[1:-1, 1:-1, 1:-1] = g.view(NZ, NY, NX)
    e = torch.arange(nx * ny * nz, device=ref.dev)
    o = torch.arange(pb, device=ref.dev)
    ix = ((e % nx) * p)[:, None] + o
    iy = ((e // nx % ny) * p)[:, None] + o
    iz = ((e // (nx * ny)) * p)[:, None] + o
    at = ix[:, None, None, :] + (NX + 2) * (iy[:, None, :, None] + (NY + 2) * iz[:, :, None, None])
    t = pad.reshape(-1)[at]
    t = torch.einsum("eia,ekji->ekja", S[0], t)
    t = torch.einsum("ejb,ekji->ekbi", S[1], t)
    t = torch.einsum("ekc,ekji->ecji", S[2], t)
    t = t / (lam[2][:, :, None, None] + lam[1][:, None, :, None] + lam[0][:, None, None, :])
    t = torch.einsum("eai,ekji->ekja", S[0], t)
    t = torch.einsum("ebj,ekji->ekbi", S[1], t)
    t = torch.einsum("eck,ekji->ecji", S[2], t)
    if kind == "ras":
        return ref.mask * ref.qqt(t[:, 1:-1, 1:-1, 1:-1] / ref.mult)
    acc = torch.zeros(pad.numel(), dtype=torch.float64, device=ref.dev).index_add_(0, at.reshape(-1), t.reshape(-1))
    cnt = torch.bincount(at.reshape(-1), minlength=pad.numel())
    s = (acc / cnt).view(pad.shape)[1:-1, 1:-1, 1:-1].reshape(-1)
    return ref.mask * s[ref.gid].view(ref.shape)


def _solution(ref, f, tol=1e-13, most=2000):
    """x of A x = M QQ^T B f by Jacobi-preconditioned conjugate gradients."""
    b = ref.mask * ref.qqt(ref.B * f)
    di = ref.mask / ref.diagonal()
    wt = 1.0 / ref.mult
    x, r = torch.zeros_like(b), b.clone()
    z = di * r
    q, rz = z.clone(), (r * z * wt).sum()
    stop = tol * (b * b * wt).sum().sqrt()
    for k in range(most):
        if k % 10 == 0 and (r * r * wt).sum().sqrt() <= stop:
            break
        w = ref.ax(q)
        a = rz / (q * w * wt).sum()
        x += a * q
        r -= a * w
        z = di * r
        new = (r * z * wt).sum()
        q = z + (new / rz) * q
        rz = new
    return x


def exact(case, seed):
    """The outputs in 64 bits by plain torch: operator, residual, smoothers and transfers in
    closed form, small solves by conjugate gradients on the same discrete problem.  None for a
    V-cycle, whose coarse solve is an iteration stopped early, and for the larger solves."""
    kind = case["kind"]
    if kind in ("vcycle", "batch"):
        return None
    nel, p, bc = _nel(case), case["p"], case["bc"]
    if kind == "solve" and _elements(case) * (p + 1) ** 3 > 400000:
        return None
    dev = torch.device("cuda:0")
    V = _vertices(nel, seed)
    if kind == "transfer":
        J = torch.tensor(_interp(p, case["pc"]), device=dev)
        gf, gc = _gid(nel, p, dev), _gid(nel, case["pc"], dev)
        u = _continuous(nel, p, bc, seed, dev)
        uc = _continuous(nel, case["pc"], bc, seed + 1, dev)
        mult = torch.bincount(gf[0]).to(torch.float64)[gf[0]]
        N, Nc = p + 1, case["pc"] + 1
        t = _lines(J.T, (u / mult).view(-1, N, N, N)).reshape(-1)
        n = gc[1][0] * gc[1][1] * gc[1][2]
        rc = torch.zeros(n, dtype=torch.float64, device=dev).index_add_(0, gc[0], t)
        rc = (rc * _mask_global(gc[1], bc, dev))[gc[0]]
        return {"restricted": rc, "prolonged": _lines(J, uc.view(-1, Nc, Nc, Nc)).reshape(-1)}
    ref = _Ref(nel, p, bc, V, dev)
    if kind == "solve":
        return _solution(ref, _forcing(ref.X, seed)).reshape(-1)
    u = _continuous(nel, p, bc, seed, dev).view(ref.shape)
    if kind == "operator":
        return ref.ax(u).reshape(-1)
    if kind == "residual":
        b = _continuous(nel, p, bc, seed + 1, dev).view(ref.shape)
        return (ref.mask * (b - ref.qqt(ref.local(u)))).reshape(-1)
    return _schwarz(ref, bc, u, case["smoother"]).reshape(-1)
