"""The work a user of the library has it do, as measurable cases.

Every case is one call (or the short run of calls a program makes together) of a
public entry point: the operator alone, whole solves, set-up of a mesh, the
learned preconditioner's inference and its training gradient.  Meshes are boxes
of hexahedra with perturbed vertices; sizes, orders and options are those of the
repository's own configurations, tests and benchmark, plus odd and ragged ones.
`exact` gives the same outputs from plain torch in 64 bits.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2011_04981_gb300 import inputs, nekax
from paper_2011_04981_gb300.problem import DeviceBatch, DeviceProblem

DEV = "cuda"
NPARAM_SHAPES = ((16, 2), (16, 16), (1, 16))  # the network's three convolutions: (out, in) channels, 27 taps each


# ------------------------------------------------------------------ the cases
def listed():
    return [
        # The operator alone on the benchmark's mesh size and order: what the headline is made of.
        dict(name="ax_ff_32x32x32_nx10", kind="ax_ff", ex=32, ey=32, ez=32, nx=10, perturb=0.1),
        # The operator on a small mesh of an odd order and ragged sizes (a coarse level, a test problem).
        dict(name="ax_ff_11x9x5_nx7", kind="ax_ff", ex=11, ey=9, ez=5, nx=7, perturb=0.1),
        # The paper's own order, 16 points a direction, 4096 elements.
        dict(name="ax_ff_16x16x16_nx16", kind="ax_ff", ex=16, ey=16, ez=16, nx=16, perturb=0.1),
        # The native FP64 operator, the default of a solve that asks for nothing else.
        dict(name="ax_fp64_20x20x20_nx8", kind="ax_fp64", ex=20, ey=20, ez=20, nx=8, perturb=0.1),
        # The benchmark's solve: Jacobi-PCG at a fixed iteration count with the FP64-accurate operator.
        dict(name="cg_ff_24x24x24_nx10", kind="cg", impl="ff", ex=24, ey=24, ez=24, nx=10, perturb=0.1, tol=0.0,
             iters=20),
        # The smallest configuration, solved to 1e-8 with the call's defaults (native FP64, residual read every
        # iteration): latency and launches.
        dict(name="cg_4x4x4_nx8", kind="cg", impl="fp64", ex=4, ey=4, ez=4, nx=8, perturb=0.05, tol=1e-8, iters=500),
        # FP64 defect correction with the FP16 inner solve, to full accuracy.
        dict(name="mixed_f16_16x16x16_nx10", kind="mixed", prec="f16", ex=16, ey=16, ez=16, nx=10, perturb=0.1,
             tol=1e-12),
        # Many uneven problems of orders 6, 8, 10 and 12 in one batched solve.
        dict(name="batch_24_problems", kind="batch", nprob=24, specs=4, iters=30),
        # One application of the learned preconditioner's network on the evaluation mesh's elements.
        dict(name="net_apply_bf16_13824", kind="net", nelt=24 ** 3),
        # One training gradient (element energy norm) at the training loop's batch.
        dict(name="train_energy_256", kind="train", batch=256),
        # Flexible CG with the network as preconditioner, window of 8 directions.
        dict(name="fcg_16x16x16", kind="fcg", ex=16, ey=16, ez=16, nx=8, perturb=0.15, iters=10),
        # A program whose mesh moves: geometric factors, their float-pair split and the Jacobi diagonal anew.
        dict(name="setup_24x24x24_nx10", kind="setup", ex=24, ey=24, ez=24, nx=10, perturb=0.1),
    ]


def _box(rng, lo, hi, nx, most):
    """Element counts of a box: log-uniform total in [lo, hi] elements, any aspect, at most `most` points."""
    total = min(math.exp(rng.uniform(math.log(lo), math.log(hi))), most / nx ** 3)
    a = max(1, round(total ** (1 / 3) * math.exp(rng.uniform(-0.5, 0.5))))
    b = max(1, round(math.sqrt(total / a) * math.exp(rng.uniform(-0.4, 0.4))))
    c = max(1, int(total / (a * b)))
    return dict(ex=a, ey=b, ez=c, nx=nx, perturb=0.1)


def draw(rng):
    kind = rng.choice(["ax_ff", "ax_ff", "ax_fp64", "cg", "cg", "mixed", "batch", "net", "train", "fcg", "setup"])
    if kind == "ax_ff":
        return dict(kind=kind, **_box(rng, 64, 32768, rng.randint(2, 16), 3.2e7))
    if kind == "ax_fp64":
        return dict(kind=kind, **_box(rng, 64, 8000, rng.randint(2, 16), 4e6))
    if kind == "cg":
        impl = rng.choice(["ff", "ff", "fp64", "oz"])
        nx = rng.choice([4, 6, 8, 10]) if impl == "oz" else rng.randint(3, 14)
        return dict(kind=kind, impl=impl, **_box(rng, 64, 13824, nx, 1.2e7 if impl != "fp64" else 2e6), tol=0.0,
                    iters=rng.randint(5, 20))
    if kind == "mixed":
        return dict(kind=kind, prec=rng.choice(["f32", "bf16", "f16"]),
                    **_box(rng, 64, 1500, rng.choice([6, 7, 8, 10, 12]), 2e6), tol=1e-12)
    if kind == "batch":
        return dict(kind=kind, nprob=rng.randint(2, 24), specs=rng.randint(10, 10 ** 6), iters=rng.randint(5, 20))
    if kind == "net":
        return dict(kind=kind, nelt=round(math.exp(rng.uniform(math.log(64), math.log(13824)))))
    if kind == "train":
        return dict(kind=kind, batch=rng.randint(16, 256))
    if kind == "fcg":
        return dict(kind=kind, **_box(rng, 64, 4096, 8, 2e6), iters=rng.randint(2, 10))
    return dict(kind=kind, **_box(rng, 64, 13824, rng.randint(4, 16), 1.2e7))


# ------------------------------------------------------------------ inputs
def _gen(seed, stream):
    g = torch.Generator(device=DEV)
    g.manual_seed(1_000_003 * int(seed) + stream)
    return g


def _uniform(seed, stream, *shape, dtype=torch.float64):
    return torch.rand(*shape, generator=_gen(seed, stream), device=DEV, dtype=dtype) * 2 - 1


def _corners(case, seed):
    """[nelt, 8, 3] vertices of the perturbed unit box."""
    V = inputs.vertex_lattice(case["ex"], case["ey"], case["ez"], case["perturb"], seed=seed)
    return np.ascontiguousarray(inputs.element_corners(V))


def _mesh(case, seed):
    return inputs.box_mesh(case["ex"], case["ey"], case["ez"], case["nx"], perturb=case["perturb"], seed=seed)


def _field(case, seed):
    """One value per global node, copied to its local copies."""
    n = case["nx"] - 1
    g = _uniform(seed, 2, (case["ex"] * n + 1) * (case["ey"] * n + 1) * (case["ez"] * n + 1))
    return g[_glo(case)]


def _glo(case):
    """Lexicographic lattice node of every local point, [nelt, nx^3]."""
    ex, ey, ez, nx = case["ex"], case["ey"], case["ez"], case["nx"]
    n = nx - 1
    ar = lambda m: torch.arange(m, device=DEV)
    X = (ar(ex)[:, None] * n + ar(nx)[None, :]).view(1, 1, ex, 1, 1, nx)
    Y = (ar(ey)[:, None] * n + ar(nx)[None, :]).view(1, ey, 1, 1, nx, 1)
    Z = (ar(ez)[:, None] * n + ar(nx)[None, :]).view(ez, 1, 1, nx, 1, 1)
    return (X + (ex * n + 1) * (Y + (ey * n + 1) * Z)).reshape(ex * ey * ez, nx ** 3)


def _theta(seed):
    """Weights scaled by 1/sqrt(fan-in) and small biases, FP32, in the library's parameter order."""
    rng = np.random.default_rng([seed, 7])
    parts = []
    for co, ci in NPARAM_SHAPES:
        parts.append(rng.normal(scale=1.0 / math.sqrt(27 * ci), size=co * ci * 27))
        parts.append(rng.normal(scale=0.05, size=co))
    return torch.from_numpy(np.concatenate(parts).astype(np.float32)).to(DEV)


def _net_inputs(n, seed):
    """Two channels of unit RMS an element, as the solver's residual and its Jacobi-scaled form are."""
    x = _uniform(seed, 11, n, 2, 512)
    x[:, 1] = 0.6 * x[:, 0] + 0.4 * x[:, 1]
    x = x / x.pow(2).mean(-1, keepdim=True).sqrt()
    return x.float()


def _train_inputs(case, seed):
    n = case["batch"]
    xin = _net_inputs(n, seed)
    target = (0.3 * xin[:, 1] + 0.5 * _uniform(seed, 12, n, 512, dtype=torch.float32)).contiguous()
    # FP32 geometric factors of stretched elements, scaled per element by a power of two
    mesh = dict(ex=8, ey=8, ez=8, perturb=0.15)
    corners = torch.from_numpy(_corners(mesh, seed)).to(DEV)[:n]
    s = torch.exp(math.log(8.0) * (_uniform(seed, 13, 3) * 0.5 + 0.5))
    G = _geom64(corners * s, 8)
    gscale = torch.exp2(torch.ceil(torch.log2(G.abs().amax(dim=(1, 2)))))
    Glp = (G / gscale[:, None, None]).float().contiguous()
    return xin, target, Glp, gscale.float().contiguous()


def _net_scale_c(n, seed):
    scale = torch.exp(2.0 * _uniform(seed, 14, n)).float()
    i = torch.arange(8, device=DEV)
    edge = ((i == 0) | (i == 7)).double() + 1.0
    c = (1.0 / (edge[:, None, None] * edge[None, :, None] * edge[None, None, :])).reshape(1, 512)
    return scale, c.expand(n, 512).contiguous()


def _batch_meshes(case, seed):
    specs = inputs.batch_problem_specs(case["nprob"], seed=case["specs"], nelt_range=(8, 1024))
    return [inputs.box_mesh(s["ex"], s["ey"], s["ez"], s["nx"], perturb=0.1, seed=s["seed"] + seed) for s in specs]


def _batch_fields(meshes, seed):
    return [inputs.random_global_field(m, seed=seed * 1009 + q) for q, m in enumerate(meshes)]


class _State:
    pass


def _ax_state(case, seed, pairs):
    """Plan and input of the operator alone: D, G (or its float-pair split) and a discontinuous field."""
    S = _State()
    S.kind, S.nelt, S.nx = case["kind"], case["ex"] * case["ey"] * case["ez"], case["nx"]
    S.D = torch.from_numpy(nekax.gll(S.nx)[2]).to(DEV)
    n3 = S.nx ** 3
    S.G = torch.empty((S.nelt, n3, 6), dtype=torch.float64, device=DEV)
    nekax.geom(S.nelt, S.nx, torch.from_numpy(_corners(case, seed)).to(DEV), S.G)
    if pairs:
        G, S.G = S.G, torch.empty((S.nelt, n3, 12), dtype=torch.float32, device=DEV)
        nekax.geom_ff(S.nelt, S.nx, G, S.G)
    S.u = _uniform(seed, 1, S.nelt, n3)
    S.w = torch.empty_like(S.u)
    torch.cuda.synchronize()  # the temporaries above are free to go
    return S


def prepare(case, seed):
    kind = case["kind"]
    if kind in ("ax_ff", "ax_fp64"):
        return _ax_state(case, seed, kind == "ax_ff")
    S = _State()
    S.kind = kind
    if kind in ("cg", "mixed", "fcg"):
        S.P = DeviceProblem(_mesh(case, seed), DEV)
        S.f = _field(case, seed)
        S.x = torch.empty_like(S.f)
        S.iters = case.get("iters")
    if kind == "cg":
        S.impl = {"ff": nekax.AX_FF, "fp64": nekax.AX_FP64, "oz": nekax.AX_OZ}[case["impl"]]
        if case["impl"] == "ff":
            S.P.prepare_ff()
        elif case["impl"] == "oz":
            S.P.prepare_oz()
        S.tol = case["tol"]
        S.ws = torch.empty(nekax.cg_workspace_bytes(S.P.nelt, S.P.nx, False) // 8 + 64, dtype=torch.float64,
                           device=DEV)
    elif kind == "mixed":
        S.P.prepare_ff()
        S.prec = {"f32": nekax.PREC_F32, "bf16": nekax.PREC_BF16, "f16": nekax.PREC_F16}[case["prec"]]
        dt = {"f32": torch.float32, "bf16": torch.bfloat16, "f16": torch.float16}[case["prec"]]
        S.Glp = torch.empty((S.P.nelt, S.P.nx ** 3, 6), dtype=dt, device=DEV)
        S.gscale = torch.empty(S.P.nelt, dtype=torch.float32, device=DEV)
        nekax.geom_lowp(S.P.nelt, S.P.nx, S.prec, S.P.G, S.Glp, S.gscale)
        S.tol = case["tol"]
    elif kind == "fcg":
        S.P.prepare_ff()
        S.theta = _theta(seed)
    elif kind == "batch":
        meshes = _batch_meshes(case, seed)
        S.B = DeviceBatch(meshes, _batch_fields(meshes, seed), DEV)
        S.x = torch.empty(S.B.npts, dtype=torch.float64, device=DEV)
        S.ws = torch.empty(S.B.plan.workspace_bytes(False) // 8 + 64, dtype=torch.float64, device=DEV)
        S.iters = case["iters"]
    elif kind == "net":
        S.n = case["nelt"]
        S.theta = _theta(seed)
        S.xin = _net_inputs(S.n, seed)
        S.scale, S.c = _net_scale_c(S.n, seed)
        S.z = torch.empty((S.n, 512), dtype=torch.float64, device=DEV)
    elif kind == "train":
        S.n = case["batch"]
        S.theta = _theta(seed)
        S.xin, S.target, S.Glp, S.gscale = _train_inputs(case, seed)
        S.D = torch.from_numpy(nekax.gll(8)[2]).to(DEV)
        S.grad = torch.empty_like(S.theta)
        S.loss = torch.zeros(1, dtype=torch.float32, device=DEV)
        S.ws = torch.empty(nekax.net_train_workspace_bytes(S.n) // 4 + 64, dtype=torch.float32, device=DEV)
    elif kind == "setup":
        S.nelt, S.nx = case["ex"] * case["ey"] * case["ez"], case["nx"]
        m = _mesh(case, seed)
        S.gs = nekax.GsPlan(S.nelt, S.nx, m.glo_num)
        S.mask = torch.from_numpy(m.mask).to(DEV)
        S.D = torch.from_numpy(nekax.gll(S.nx)[2]).to(DEV)
        S.corners = torch.from_numpy(_corners(case, seed)).to(DEV)
        n3 = S.nx ** 3
        S.G = torch.empty((S.nelt, n3, 6), dtype=torch.float64, device=DEV)
        S.Gff = torch.empty((S.nelt, n3, 12), dtype=torch.float32, device=DEV)
        S.minv = torch.empty((S.nelt, n3), dtype=torch.float64, device=DEV)
    torch.cuda.synchronize()
    return S


def run(S):
    if S.kind == "ax_ff":
        nekax.ax_ff(S.nelt, S.nx, S.D, S.G, S.u, S.w)
        return S.w
    if S.kind == "ax_fp64":
        nekax.ax(S.nelt, S.nx, S.D, S.G, S.u, S.w)
        return S.w
    if S.kind == "cg":
        r = S.P.cg(S.f, S.x, tol=S.tol, max_iter=S.iters, workspace=S.ws, ax_impl=S.impl)
        return {"x": S.x, "relres": r["relres"], "status": r["status"], "iters": r["iters"]}
    if S.kind == "mixed":
        P = S.P
        r = nekax.cg_solve_mixed(P.gs, P.nelt, P.nx, P.D, P.G, P.Gff, S.prec, S.Glp, S.gscale, P.mask, P.minv, S.f,
                                 S.x, tol=S.tol)
        return {"x": S.x, "status": r["status"]}
    if S.kind == "fcg":
        P = S.P
        r = nekax.fcg_solve(P.gs, P.nelt, P.nx, P.D, P.G, P.Gff, P.mask, P.minv, S.theta, S.f, S.x, tol=1e-14,
                            max_iter=S.iters, stag_window=200, stag_factor=0.8, truncation=8)
        return {"x": S.x, "relres": r["relres"], "status": r["status"], "iters": r["iters"]}
    if S.kind == "batch":
        r = S.B.solve(S.x, tol=0.0, max_iter=S.iters, workspace=S.ws)
        return {"x": S.x, "relres": r["relres"], "status": r["status"], "iters": r["iters"]}
    if S.kind == "net":
        nekax.net_apply_bf16(S.n, 8, S.theta, S.xin, S.scale, S.c, S.z)
        return S.z
    if S.kind == "train":
        nekax.net_train_grad_energy(S.n, S.theta, S.xin, S.target, S.D, S.Glp, S.gscale, S.grad, S.loss, S.ws)
        return {"grad": S.grad, "loss": S.loss}
    nekax.geom(S.nelt, S.nx, S.corners, S.G)
    nekax.geom_ff(S.nelt, S.nx, S.G, S.Gff)
    nekax.jacobi_minv(S.gs, S.nelt, S.nx, S.D, S.G, S.mask, S.minv)
    return {"G": S.G, "Gff": S.Gff, "minv": S.minv}


# ------------------------------------------------------------------ what a pass cannot do without
def _pts(case):
    return case["ex"] * case["ey"] * case["ez"] * case["nx"] ** 3


def _iteration(pts, nx):
    """One Jacobi-PCG iteration: G; x, r, p read and written; the inverse diagonal; w out of the operator and into
    the r update (the sum over shared nodes stands between them); operator and vector operations."""
    return pts * (48 + 3 * 16 + 8 + 16), pts * (12 * nx + 11 + 12)


def work(case):
    kind = case["kind"]
    if kind in ("ax_ff", "ax_fp64"):
        return {"bytes": _pts(case) * 64, "flops": _pts(case) * (12 * case["nx"] + 11)}
    conv = 2 * 27 * 512 * sum(co * ci for co, ci in NPARAM_SHAPES)  # one forward pass of one element
    if kind in ("cg", "mixed"):
        its = case["iters"] if kind == "cg" and case["tol"] == 0.0 else 80 if kind == "cg" else 600
        b, f = _iteration(_pts(case), case["nx"])
        if kind == "mixed":  # FP32 vectors and 16-bit factors (24 bytes of them with FP32)
            b = _pts(case) * (36 + (24 if case["prec"] == "f32" else 12))
        return {"bytes": its * b, "flops": its * f}
    if kind == "fcg":  # a plain iteration, the network, and the window's directions and images once each
        b, f = _iteration(_pts(case), 8)
        win = sum(min(k, 8) for k in range(case["iters"]))
        return {"bytes": case["iters"] * (b + _pts(case) * 16) + win * _pts(case) * 16,
                "flops": case["iters"] * (f + _pts(case) // 512 * conv) + win * _pts(case) * 4}
    if kind == "batch":
        tot_b = tot_f = 0
        for s in inputs.batch_problem_specs(case["nprob"], seed=case["specs"], nelt_range=(8, 1024)):
            b, f = _iteration(_pts(s), s["nx"])
            tot_b, tot_f = tot_b + b, tot_f + f
        return {"bytes": case["iters"] * tot_b, "flops": case["iters"] * tot_f}
    if kind == "net":
        return {"bytes": case["nelt"] * 512 * (8 + 16), "flops": case["nelt"] * conv}
    if kind == "train":
        return {"bytes": case["batch"] * 512 * (8 + 4 + 24), "flops": 3 * case["batch"] * conv}
    pts = _pts(case)
    return {"bytes": pts * (48 + 48 + 8), "flops": pts * (60 + 9 * case["nx"])}


# ------------------------------------------------------------------ the same in plain 64-bit torch
def _gll64(nx):
    """Gauss-Lobatto-Legendre nodes, weights and derivative matrix (numpy)."""
    N = nx - 1
    P = np.polynomial.legendre.Legendre.basis(N)
    x = np.concatenate([[-1.0], np.sort(P.deriv().roots().real), [1.0]])
    for _ in range(3):  # Newton on (1 - x^2) P_N'(x) from its roots
        if N > 1:
            d1, d2 = P.deriv()(x[1:-1]), P.deriv(2)(x[1:-1])
            x[1:-1] -= d1 / d2
    x = 0.5 * (x - x[::-1])
    L = P(x)
    D = np.zeros((nx, nx))
    for i in range(nx):
        for l in range(nx):
            if i != l:
                D[i, l] = L[i] / L[l] / (x[i] - x[l])
    D[0, 0], D[N, N] = -N * (N + 1) / 4.0, N * (N + 1) / 4.0
    return x, 2.0 / (N * (N + 1) * L * L), D


def _geom64(corners, nx):
    """[nelt, nx^3, 6] geometric factors rr, rs, rt, ss, st, tt of trilinear elements."""
    x, rho, _ = _gll64(nx)
    x, rho = torch.from_numpy(x).to(DEV), torch.from_numpy(rho).to(DEV)
    lo, hi = (1 - x) / 2, (1 + x) / 2
    val, der = torch.stack([lo, hi], -1), torch.stack([-0.5 * torch.ones_like(x), 0.5 * torch.ones_like(x)], -1)
    c = corners.reshape(-1, 2, 2, 2, 3)  # [e][dk][dj][di][xyz]
    f = lambda R, Sx, T: torch.einsum("ezyxc,kz,jy,ix->ekjic", c, T, Sx, R)
    a, b, g = f(der, val, val), f(val, der, val), f(val, val, der)  # columns of the Jacobian
    ca, cb, cg = torch.linalg.cross(b, g), torch.linalg.cross(g, a), torch.linalg.cross(a, b)
    J = (a * ca).sum(-1)
    wq = (rho[:, None, None] * rho[None, :, None] * rho[None, None, :]) / J
    dot = lambda p, q: (p * q).sum(-1) * wq
    G = torch.stack([dot(ca, ca), dot(ca, cb), dot(ca, cg), dot(cb, cb), dot(cb, cg), dot(cg, cg)], -1)
    return G.reshape(G.shape[0], nx ** 3, 6)


def _ax64(u, G, D):
    n = D.shape[0]
    u = u.reshape(-1, n, n, n)
    G = G.reshape(-1, n, n, n, 6)
    ur, us, ut = u @ D.T, D @ u, torch.einsum("kl,elji->ekji", D, u)
    wr = G[..., 0] * ur + G[..., 1] * us + G[..., 2] * ut
    ws = G[..., 1] * ur + G[..., 3] * us + G[..., 4] * ut
    wt = G[..., 2] * ur + G[..., 4] * us + G[..., 5] * ut
    return (wr @ D + D.T @ ws + torch.einsum("lk,elji->ekji", D, wt)).reshape(u.shape[0], n ** 3)


class _Problem64:
    """Assembled operator of one box in plain torch."""

    def __init__(self, case, corners):
        nx = case["nx"]
        self.D = torch.from_numpy(_gll64(nx)[2]).to(DEV)
        self.G = _geom64(torch.from_numpy(corners).to(DEV), nx)
        self.glo = _glo(case)
        n = nx - 1
        gx, gy, gz = case["ex"] * n + 1, case["ey"] * n + 1, case["ez"] * n + 1
        self.nglob = gx * gy * gz
        X, r = self.glo % gx, self.glo // gx
        Y, Z = r % gy, r // gy
        self.mask = ((X > 0) & (X < gx - 1) & (Y > 0) & (Y < gy - 1) & (Z > 0) & (Z < gz - 1)).double()
        self.c = 1.0 / self.dssum(torch.ones_like(self.mask))
        d = self._diag()
        self.minv = self.mask / self.dssum(d)

    def dssum(self, v):
        g = torch.zeros(self.nglob, dtype=torch.float64, device=DEV)
        return g.index_add_(0, self.glo.reshape(-1), v.reshape(-1))[self.glo]

    def _diag(self):
        n = self.D.shape[0]
        G = self.G.reshape(-1, n, n, n, 6)
        D2, dd = self.D * self.D, torch.diagonal(self.D)
        d = (G[..., 0] @ D2 + D2.T @ G[..., 3] + torch.einsum("lk,elji->ekji", D2, G[..., 5]))
        i, j, k = dd.view(1, 1, n), dd.view(1, n, 1), dd.view(n, 1, 1)
        d = d + 2 * (G[..., 1] * i * j + G[..., 2] * i * k + G[..., 4] * j * k)
        return d.reshape(-1, n ** 3)

    def ax(self, p):
        return self.mask * self.dssum(_ax64(p, self.G, self.D))

    def dot(self, a, b):
        return float((self.c * a * b).sum())

    def pcg(self, f, tol, iters):
        r = self.mask * f
        x, z = torch.zeros_like(r), self.minv * r
        p, rz, b, it = z, self.dot(r, z), math.sqrt(self.dot(r, r)), 0
        rel = 1.0
        while it < iters:
            w = self.ax(p)
            a = rz / self.dot(p, w)
            x, r, it = x + a * p, r - a * w, it + 1
            rel = math.sqrt(self.dot(r, r)) / b
            if tol > 0 and rel <= tol:
                break
            z = self.minv * r
            new = self.dot(r, z)
            p, rz = z + new / rz * p, new
        return x, rel, it


def _net64(theta, x):
    """Output [n, 512] of the network with BF16 weights, everything else in 64 bits."""
    o, h = 0, x.double().reshape(-1, 2, 8, 8, 8)
    for l, (co, ci) in enumerate(NPARAM_SHAPES):
        W = theta[o:o + co * ci * 27].bfloat16().double().view(co, ci, 3, 3, 3)
        b = theta[o + co * ci * 27:o + co * ci * 27 + co].bfloat16().double()
        o += co * ci * 27 + co
        h = torch.cat([torch.nn.functional.conv3d(q, W, b, padding=1) for q in h.split(512)])
        if l < 2:
            h = torch.nn.functional.gelu(h)
    return h.reshape(-1, 512)


def _round_weights(theta):
    """BF16 rounding of the weights that a gradient passes through unchanged."""
    return theta + (theta.detach().bfloat16().double() - theta.detach())


def _train64(case, seed):
    xin, target, Glp, gscale = _train_inputs(case, seed)
    D = torch.from_numpy(_gll64(8)[2]).to(DEV)
    G = Glp.double() * gscale.double()[:, None, None]
    theta = _theta(seed).double().requires_grad_(True)
    tq, o, h = _round_weights(theta), 0, xin.double().reshape(-1, 2, 8, 8, 8)
    for l, (co, ci) in enumerate(NPARAM_SHAPES):
        W, b = tq[o:o + co * ci * 27].view(co, ci, 3, 3, 3), tq[o + co * ci * 27:o + co * ci * 27 + co]
        o += co * ci * 27 + co
        h = torch.nn.functional.conv3d(h, W, b, padding=1)
        if l < 2:
            h = torch.nn.functional.gelu(h)
    t = target.double()
    d = h.reshape(-1, 512) - t
    loss = ((d * _ax64(d, G, D)).sum(-1) / (t * _ax64(t, G, D)).sum(-1)).mean()
    loss.backward()
    return {"grad": theta.grad, "loss": loss.detach().reshape(1)}


def _fcg64(case, seed):
    P = _Problem64(case, _corners(case, seed))
    theta, f = _theta(seed), _field(case, seed)
    r = P.mask * f
    x, b, win, rel = torch.zeros_like(r), math.sqrt(P.dot(r, r)), [], 1.0
    rms = lambda v: v.pow(2).mean(-1, keepdim=True).sqrt().clamp_min(1e-300)
    for _ in range(case["iters"]):
        j = P.minv * r
        s = rms(j)
        z = P.mask * P.dssum(_net64(theta, torch.stack([r / rms(r), j / s], 1)) * s * P.c)
        p = z
        for q, wq, pwq in win:
            p = p - P.dot(z, wq) / pwq * q
        w = P.ax(p)
        pw = P.dot(p, w)
        a = P.dot(p, r) / pw
        x, r = x + a * p, r - a * w
        rel = math.sqrt(P.dot(r, r)) / b
        win = [(p, w, pw)] + win[:7]
    return {"x": x, "relres": rel, "status": None, "iters": case["iters"]}


@torch.no_grad()
def _exact(case, seed):
    kind = case["kind"]
    if kind in ("ax_ff", "ax_fp64"):
        nx, u = case["nx"], _uniform(seed, 1, case["ex"] * case["ey"] * case["ez"], case["nx"] ** 3)
        D = torch.from_numpy(_gll64(nx)[2]).to(DEV)
        c = torch.from_numpy(_corners(case, seed)).to(DEV)
        step = max(1, 4_000_000 // nx ** 3)
        return torch.cat([_ax64(u[q:q + step], _geom64(c[q:q + step], nx), D) for q in range(0, u.shape[0], step)])
    if kind == "cg":
        x, rel, it = _Problem64(case, _corners(case, seed)).pcg(_field(case, seed), case["tol"], case["iters"])
        return {"x": x, "relres": rel, "status": None, "iters": None}
    if kind == "mixed":
        x, _, _ = _Problem64(case, _corners(case, seed)).pcg(_field(case, seed), 1e-15, 3000)
        return {"x": x, "status": None}
    if kind == "fcg":
        return _fcg64(case, seed)
    if kind == "batch":
        meshes = _batch_meshes(case, seed)
        fields = _batch_fields(meshes, seed)
        order = sorted(range(len(meshes)), key=lambda q: (meshes[q].nx, meshes[q].nelt, q))
        xs, rels = [], []
        for q in order:
            m = meshes[q]
            P = _Problem64(dict(ex=m.ex, ey=m.ey, ez=m.ez, nx=m.nx), m.corners)
            x, rel, _ = P.pcg(torch.from_numpy(fields[q]).to(DEV), 0.0, case["iters"])
            xs.append(x.reshape(-1))
            rels.append(rel)
        return {"x": torch.cat(xs), "relres": np.array(rels), "status": None, "iters": None}
    if kind == "net":
        scale, c = _net_scale_c(case["nelt"], seed)
        return _net64(_theta(seed), _net_inputs(case["nelt"], seed)) * scale.double()[:, None] * c
    m = _Problem64(case, _corners(case, seed))
    return {"G": m.G, "Gff": None, "minv": m.minv}


def exact(case, seed):
    return _train64(case, seed) if case["kind"] == "train" else _exact(case, seed)
