"""Performance cases: the work that users of the framework have it do.

Every case calls the public entry points (paper_1607_00693_gb300.api) on
seeded synthetic inputs, at the sizes of this repository's workloads
(workloads.py) and at odd sizes of the same ranges:

  step     sample the coefficient, upscale every cell, solve the coarse
           systems: one small Monte Carlo batch by direct calls
  plan     the same step through a plan's captured graph, with moments
  upscale  the local upscaling alone (coefficient in hand): FP64, FP32 and
           FP32 + FP64 refinement; Galerkin or Petrov-Galerkin; bilinear or
           oscillatory cell data; with and without oversampling
  coarse   the coarse solves of a batch and its moments (K_e in hand)
  sample   coefficient sampling alone
  fine     fine-grid FEM solves of the two-level Monte Carlo estimator
  pod      online reduced-basis upscaling
  ri       online random interpolation
"""
import math

import numpy as np
import torch

from paper_1607_00693_gb300 import api

EXP, SIGMOID = api.FIELD_EXP, api.FIELD_EXP_SIGMOID
DEV = "cuda"
F64 = torch.float64

# ------------------------------------------------------------------ the cases

_BUMPS_64 = dict(kind=EXP, nbx=4, nby=4, width=0.1, scale=1.0, clog=0.0, gain=1.0)
_BUMPS_1024 = dict(kind=EXP, nbx=16, nby=16, width=2.0 / 32, scale=math.log(100.0) / (2 * math.pi), clog=0.0, gain=1.0)
_BUMPS_2048 = dict(kind=SIGMOID, nbx=32, nby=32, width=1.5 / 64, scale=1.0, clog=math.log(1e4), gain=8.0)


def _upscale(nf, nc, S, precision, max_o=0, pg=0, osc=0, field=_BUMPS_1024):
    return dict(path="upscale", nf=nf, nc=nc, S=S, precision=precision, max_o=max_o, pg=pg, osc=osc, **field)


def listed():
    return [
        # the smallest batch a user steps through: 64 samples of the 64^2 / 8^2
        # grid by direct calls, where launches and latency count
        dict(name="step_64_fp64", path="step", nf=64, nc=8, S=64, precision=api.FP64, max_o=0, **_BUMPS_64),
        # the Monte Carlo step in production: H/h = 32 with oversampling,
        # FP32, one captured graph, running moments
        dict(name="plan_1024_fp32", path="plan", nf=1024, nc=32, S=64, precision=api.FP32, max_o=4, **_BUMPS_1024),
        # its dominant part through the direct call (default launch choices)
        dict(name="upscale_1024_fp32", **_upscale(1024, 32, 32, api.FP32, 4)),
        # the plain FP64 form, the paper's own arithmetic
        dict(name="upscale_1024_fp64", **_upscale(1024, 32, 4, api.FP64, 4)),
        # FP32 factor with FP64 refinement (the default two sweeps)
        dict(name="upscale_1024_fp32r", **_upscale(1024, 32, 8, api.FP32_REFINED, 4)),
        # high-contrast channel medium, no oversampling, H/h = 32
        dict(name="upscale_2048_fp32", **_upscale(2048, 64, 4, api.FP32, 0, field=_BUMPS_2048)),
        # odd sizes, Petrov-Galerkin with the oscillatory cell data (the
        # options of the short-correlation example), an odd sample count
        dict(name="upscale_345_pg_osc_fp32", **_upscale(345, 15, 37, api.FP32, 3, 1, 1, dict(_BUMPS_1024, nbx=7, nby=9, width=0.1))),
        # the coarse systems of one large batch, with moments
        dict(name="coarse_32", path="coarse", nc=32, S=512),
        # FP64 coefficient sampling of one batch
        dict(name="sample_1024_fp64", path="sample", nf=1024, S=32, **_BUMPS_1024),
        # level-1 solves of the two-level estimator
        dict(name="fine_1024", path="fine", nf=1024, S=8, **_BUMPS_1024),
        # online reduced basis on 10^4 samples
        dict(name="pod_64", path="pod", nf=64, nc=8, S=10000, train=60, **_BUMPS_64),
        # online random interpolation on 10^5 samples
        dict(name="ri_64", path="ri", nf=64, nc=8, S=100000, eps=1e-3, nu_max=8, **_BUMPS_64),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _draw_field(rng, nf):
    if rng.random() < 0.7:
        n = rng.randint(2, 16)
        return dict(kind=EXP, nbx=n, nby=rng.randint(2, 16), width=rng.uniform(0.7, 2.0) / n,
                    scale=rng.uniform(0.4, 1.0), clog=0.0, gain=1.0)
    n = rng.randint(8, 32)
    return dict(kind=SIGMOID, nbx=n, nby=rng.randint(8, 32), width=rng.uniform(0.7, 1.0) / n,
                scale=1.0, clog=math.log(_log_int(rng, 100, 10000)), gain=8.0)


def draw(rng):
    path = rng.choice(["step", "plan", "upscale", "upscale", "upscale", "coarse", "sample", "fine", "pod", "ri"])
    if path in ("step", "plan", "upscale"):
        rho = rng.randint(3, 32)
        nc = _log_int(rng, 3, min(64, 1500 // rho))
        prec = rng.choice([api.FP64, api.FP32, api.FP32_REFINED])
        nf = nc * rho
        max_o = 0 if rng.random() < 0.3 else rng.randint(1, 4)
        pg = osc = 0
        if path == "upscale":
            pg, osc = int(rng.random() < 0.3), int(rng.random() < 0.3)
        # unit costs about rho^4; the listed FP64 and FP32 calls bound the work
        units = 4096 if prec == api.FP64 else 8192 if prec == api.FP32_REFINED else 32768
        most = max(1, int(units * 0.7 * (32.0 / (rho + 6)) ** 3.5 / (nc * nc)))
        S = _log_int(rng, 1, min(512, most, 30000000 // (nf * nf) + 1))
        case = dict(path=path, nf=nf, nc=nc, S=S, precision=prec, max_o=max_o, **_draw_field(rng, nf))
        if path == "upscale":
            case.update(pg=pg, osc=osc)
        return case
    if path == "coarse":
        nc = rng.randint(4, 64)
        return dict(path=path, nc=nc, S=_log_int(rng, 1, max(2, min(1024, int(400 * (32.0 / nc) ** 4)))))
    if path == "sample":
        nf = _log_int(rng, 32, 2048)
        return dict(path=path, nf=nf, S=_log_int(rng, 1, max(2, min(4096, 16000000 // (nf * nf)))), **_draw_field(rng, nf))
    if path == "fine":
        nf = rng.randint(9, 16) * 2 ** rng.randint(1, 6)
        S = _log_int(rng, 1, max(2, min(256, 5000000 // (nf * nf) if nf > 64 else 256)))
        return dict(path=path, nf=nf, S=S, **_draw_field(rng, nf))
    if path == "pod":
        return dict(path=path, nf=64, nc=8, S=_log_int(rng, 1, 8000), train=60, **_BUMPS_64)
    return dict(path="ri", nf=64, nc=8, S=_log_int(rng, 1, 80000), eps=rng.choice([1e-3, 1e-2]), nu_max=8, **_BUMPS_64)


# ------------------------------------------------------- inputs from the seed

def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed) + 1607)
    return g


def _draw_xi(case, S, gen):
    """xi ~ U[-1, 1], or N(0, 1) for the high-contrast sigmoid media."""
    K = case["nbx"] * case["nby"]
    if case["kind"] == SIGMOID:
        return torch.randn((S, K), dtype=F64, device=DEV, generator=gen)
    return torch.rand((S, K), dtype=F64, device=DEV, generator=gen) * 2.0 - 1.0


def _bump_axis(case, coords, n):
    c = (torch.arange(n, dtype=F64, device=DEV) + 0.5) / n
    return torch.exp(-((coords[:, None] - c[None, :]) / case["width"]) ** 2)  # [coords][n]


def _coefficient(case, xi, xs, ys):
    """a [S][len(ys)][len(xs)] at the given centroid coordinates."""
    S = xi.shape[0]
    gx, gy = _bump_axis(case, xs, case["nbx"]), _bump_axis(case, ys, case["nby"])
    z = torch.matmul(torch.matmul(gy, xi.view(S, case["nby"], case["nbx"])), gx.t())
    if case["kind"] == SIGMOID:
        return torch.exp(case["clog"] / (1.0 + torch.exp(-case["gain"] * z))).contiguous()
    return torch.exp(case["scale"] * z).contiguous()


def _centroids(nf):
    return (torch.arange(nf, dtype=F64, device=DEV) + 0.5) / nf


def _field_of(case):
    return api.field(case["kind"], case["nbx"], case["nby"], case["width"], case["scale"], case["clog"], case["gain"])


def _oversample(case, gen):
    if not case["max_o"]:
        return None
    return torch.randint(0, case["max_o"] + 1, (case["nc"] ** 2,), device=DEV, generator=gen).to(torch.int8)


def _coarse_matrices(case, gen):
    """K_e [S][cells][10], b_e [S][cells][4] of effective tensors (kx, ky, kxy):
    SPD element matrices with zero row sums, as the upscaling gives."""
    S, nc = case["S"], case["nc"]
    shape = (S, nc * nc, 1)
    kx = torch.exp(0.8 * torch.randn(shape, dtype=F64, device=DEV, generator=gen))
    ky = torch.exp(0.8 * torch.randn(shape, dtype=F64, device=DEV, generator=gen))
    kxy = 0.4 * torch.sqrt(kx * ky) * (2.0 * torch.rand(shape, dtype=F64, device=DEV, generator=gen) - 1.0)
    X = np.array([[2, -2, -1, 1], [-2, 2, 1, -1], [-1, 1, 2, -2], [1, -1, -2, 2]]) / 6.0
    Y = np.array([[2, 1, -1, -2], [1, 2, -2, -1], [-1, -2, 2, 1], [-2, -1, 1, 2]]) / 6.0
    XY = np.array([[1, 0, -1, 0], [0, -1, 0, 1], [-1, 0, 1, 0], [0, 1, 0, -1]]) / 2.0
    up = np.triu_indices(4)
    dev = lambda m: torch.from_numpy(m[up]).to(DEV)
    Ke = kx * dev(X) + ky * dev(Y) + kxy * dev(XY)
    be = (0.25 + 0.02 * torch.randn((S, nc * nc, 4), dtype=F64, device=DEV, generator=gen)) / nc ** 2
    return Ke.contiguous(), be.contiguous()


def _empty(*shape, dtype=F64):
    return torch.zeros(shape, dtype=dtype, device=DEV)


def _inputs(case, seed):
    """The random inputs alone (shared by prepare and exact)."""
    gen = _gen(seed)
    path = case["path"]
    if path == "coarse":
        Ke, be = _coarse_matrices(case, gen)
        return dict(Ke=Ke, be=be)
    out = dict(xi=_draw_xi(case, case["S"], gen))
    if path in ("step", "plan", "upscale"):
        out["oversample"] = _oversample(case, gen)
    if path in ("upscale", "fine", "pod"):
        c = _centroids(case["nf"])
        out["a"] = _coefficient(case, out["xi"], c, c)
    return out


def prepare(case, seed):
    st = dict(case=case, **_inputs(case, seed))
    path, S = case["path"], case["S"]
    nf, nc = case.get("nf"), case.get("nc", 1)
    g = st["g"] = api.grid(nf or nc, nc)
    cells, nodes = nc * nc, (nc + 1) ** 2
    if path in ("step", "plan", "sample"):
        st["field"] = _field_of(case)
    if path in ("step", "sample"):
        st["a"] = _empty(S, nf, nf)
    if path in ("step", "upscale", "pod", "ri"):
        st["Ke"] = _empty(S, cells, 16 if case.get("pg") else 10)
        st["be"] = _empty(S, cells, 4)
    if path in ("step", "upscale"):
        _, ws = api.stomsfem_upscale_workspace_size(g, case["max_o"], case["precision"])
        st["ws"] = _empty(ws, dtype=torch.uint8)
    if path in ("step", "plan", "coarse"):
        st["u"] = _empty(S, nodes)
    if path in ("step", "coarse"):
        st["cws"] = _empty(api.stomsfem_coarse_workspace_size(g, S), dtype=torch.uint8)
    if path in ("plan", "coarse"):
        st["mean"], st["m2"], st["count"] = _empty(nodes), _empty(nodes), _empty(1)
    if path == "plan":
        st["plan"] = api.stomsfem_plan_create(g, st["field"], S, case["precision"], st["oversample"], case["max_o"])
        # the choice that plan_tune makes on these workloads, set directly so
        # that every preparation runs the same one
        api.stomsfem_plan_set_choice(st["plan"], 0, 1, api.ENGINE_AUTO, api.ORDER_PATCH)
        st["stream"] = torch.cuda.Stream()
    if path == "fine":
        st["u"] = _empty(S, (nf + 1) ** 2)
        st["ws"] = _empty(api.stomsfem_fine_fem_workspace_size(g, S), dtype=torch.uint8)
    if path == "pod":
        # the basis from training samples of their own
        gen = _gen(987654321)
        c = _centroids(nf)
        at = _coefficient(case, _draw_xi(case, case["train"], gen), c, c)
        phi = _cells_64bit(dict(case, S=case["train"], max_o=0), at, None, with_phi=True)[2]
        st["handle"], _ = api.stomsfem_pod_build(g, phi, at, tol=1e-6, max_rank=27)
        st["ws"] = _empty(api.stomsfem_pod_workspace_size(st["handle"], S), dtype=torch.uint8)
        st["status"] = _empty(S, cells, dtype=torch.int32)
    if path == "ri":
        st["handle"], _ = api.stomsfem_ri_build(g, _field_of(case), case["eps"], case["nu_max"], api.RI_LEGENDRE)
        st["ws"] = _empty(api.stomsfem_ri_workspace_size(st["handle"], S), dtype=torch.uint8)
        st["fell"] = _empty(S, cells, dtype=torch.uint8)
    torch.cuda.synchronize()
    return _State(st)


class _State(dict):
    """The prepared objects; library handles end with them."""

    def __del__(self):
        end = {"plan": ("plan", api.stomsfem_plan_destroy), "pod": ("handle", api.stomsfem_pod_destroy),
               "ri": ("handle", api.stomsfem_ri_destroy)}.get(self["case"]["path"])
        if end and end[0] in self:
            torch.cuda.synchronize()
            end[1](self.pop(end[0]))


# -------------------------------------------------------------------- one pass

def run(st):
    case, g = st["case"], st["g"]
    path = case["path"]
    if path == "step":
        api.stomsfem_sample_coef(g, st["field"], st["xi"], st["a"])
        api.stomsfem_upscale(g, st["a"], st["Ke"], st["be"], oversample=st["oversample"], max_oversample=case["max_o"],
                             precision=case["precision"], workspace=st["ws"])
        api.stomsfem_coarse_solve(g, st["Ke"], st["be"], st["u"], workspace=st["cws"])
        return dict(a=st["a"], Ke=st["Ke"], be=st["be"], u=st["u"])
    if path == "plan":
        # a new estimate's moments, then one step, on the caller's own stream
        cur = torch.cuda.current_stream()
        st["stream"].wait_stream(cur)
        with torch.cuda.stream(st["stream"]):
            st["mean"].zero_(), st["m2"].zero_(), st["count"].zero_()
            api.stomsfem_plan_step(st["plan"], st["xi"], st["u"], st["mean"], st["m2"], st["count"])
        cur.wait_stream(st["stream"])
        return dict(u=st["u"], mean=st["mean"], m2=st["m2"], count=st["count"])
    if path == "upscale":
        args = (g, st["a"], st["Ke"], st["be"])
        opts = dict(oversample=st["oversample"], max_oversample=case["max_o"], precision=case["precision"],
                    workspace=st["ws"])
        if case["osc"]:
            api.stomsfem_upscale_bc(g, case["pg"], api.BC_OSCILLATORY, *args[1:], **opts)
        elif case["pg"]:
            api.stomsfem_upscale_pg(*args, **opts)
        else:
            api.stomsfem_upscale(*args, **opts)
        return dict(Ke=st["Ke"], be=st["be"])
    if path == "coarse":
        st["mean"].zero_(), st["m2"].zero_(), st["count"].zero_()
        api.stomsfem_coarse_solve(g, st["Ke"], st["be"], st["u"], st["mean"], st["m2"], st["count"], workspace=st["cws"])
        return dict(u=st["u"], mean=st["mean"], m2=st["m2"], count=st["count"])
    if path == "sample":
        api.stomsfem_sample_coef(g, st["field"], st["xi"], st["a"])
        return dict(a=st["a"])
    if path == "fine":
        api.stomsfem_fine_fem(g, st["a"], st["u"], workspace=st["ws"])
        return dict(u=st["u"])
    if path == "pod":
        api.stomsfem_pod_upscale(st["handle"], g, st["a"], st["Ke"], st["be"], unit_status=st["status"],
                                 workspace=st["ws"])
        return dict(Ke=st["Ke"], be=st["be"], status=st["status"])
    api.stomsfem_ri_upscale(st["handle"], g, st["xi"], None, st["Ke"], st["be"], st["fell"], workspace=st["ws"])
    return dict(Ke=st["Ke"], be=st["be"], fell=st["fell"])


# ------------------------------------------------------------------------ work

def _cell_flops(rho, max_o):
    """Banded Cholesky, three right-hand sides and K_e of one cell, at the mean oversampling."""
    m = rho + max_o - 1  # 2 * (max_o / 2) added elements
    n, b = m * m, m + 1
    return n * b * (b + 1) + 12 * n * b + 70 * rho * rho


def work(case):
    path, S = case["path"], case["S"]
    nf, nc = case.get("nf"), case.get("nc", 1)
    cells, nodes = nc * nc, (nc + 1) ** 2
    K = case["nbx"] * case["nby"] if "nbx" in case else 0
    fine = S * nf * nf if nf else 0
    ke = S * cells * 8 * ((16 if case.get("pg") else 10) + 4)
    solve = S * ((nc - 1) ** 2 * nc * (nc + 1) + 4 * (nc - 1) ** 2 * nc)
    sampling = 2.0 * fine * case.get("nbx", 0) + 2.0 * S * (nf or 0) * K
    up = S * cells * _cell_flops(nf // nc, case.get("max_o", 0)) if path in ("step", "plan", "upscale") else 0
    if path == "step":
        return {"bytes": 8 * S * K + 8 * fine + ke + 8 * S * nodes, "flops": sampling + up + solve}
    if path == "plan":
        return {"bytes": 8 * S * K + 8 * S * nodes, "flops": sampling + up + solve}
    if path == "upscale":
        return {"bytes": 8 * fine + ke, "flops": up}
    if path == "coarse":
        return {"bytes": ke + 8 * S * nodes, "flops": solve}
    if path == "sample":
        return {"bytes": 8 * S * K + 8 * fine, "flops": sampling}
    if path == "fine":
        # about ten multigrid-preconditioned CG iterations of ~150 operations a node
        return {"bytes": 16 * fine, "flops": 1500.0 * fine}
    if path == "pod":
        return {"bytes": 8 * fine + ke, "flops": S * cells * 2.0 * (nf // nc) ** 2 * 496}
    return {"bytes": 8 * S * K + ke + S * cells, "flops": S * cells * 28.0 * 160}


# ------------------------------------------- the same quantities in 64 bits

def _band_solve(E, rhs, mx):
    """Solves the 9-point-stencil SPD systems of a batch: E [U][n][5] the
    couplings of node r to r, r-1, r-mx+1, r-mx, r-mx-1, rhs [U][n][R];
    elementwise banded LDL^T."""
    U, n, _ = E.shape
    b = mx + 1
    W = torch.zeros((U, b + 1, b + 1), dtype=F64, device=DEV)
    offs = (0, 1, mx - 1, mx, mx + 1)

    def put(r, at):
        if r >= n:
            return
        for k, d in enumerate(offs):
            j = at - d
            if j < 0 or (k and d == 0):
                continue
            W[:, at, j] += E[:, r, k]
            if d:
                W[:, j, at] += E[:, r, k]

    for r in range(b + 1):
        put(r, r)
    y = rhs.clone()
    Lc = torch.zeros((n, U, b), dtype=F64, device=DEV)
    D = torch.zeros((n, U), dtype=F64, device=DEV)
    for k in range(n):
        d, c = W[:, 0, 0].clone(), W[:, 1:, 0].clone()
        l = c / d[:, None]
        D[k], Lc[k] = d, l
        nxt = torch.zeros_like(W)
        torch.addcmul(W[:, 1:, 1:], l[:, :, None], c[:, None, :], value=-1.0, out=nxt[:, :b, :b])
        W = nxt
        put(k + 1 + b, b)
        m = min(b, n - 1 - k)
        if m:
            y[:, k + 1:k + 1 + m] -= l[:, :m, None] * y[:, k:k + 1]
    for k in range(n - 1, -1, -1):
        m = min(b, n - 1 - k)
        y[:, k] /= D[k][:, None]
        if m:
            y[:, k] -= (Lc[k][:, :m, None] * y[:, k + 1:k + 1 + m]).sum(1)
    return y


_KREF = np.array([[4, -1, -2, -1], [-1, 4, -1, -2], [-2, -1, 4, -1], [-1, -2, -1, 4]]) / 6.0


def _patch_psi(a, osc):
    """psi [U][4][Ny+1][Nx+1] of patches with coefficient a [U][Ny][Nx]."""
    U, Ny, Nx = a.shape
    psi = torch.zeros((U, 4, Ny + 1, Nx + 1), dtype=F64, device=DEV)

    def coord(ae):  # [U][N] along an edge -> [U][N+1]
        N = ae.shape[1]
        if not osc:
            return (torch.arange(N + 1, dtype=F64, device=DEV) / N).expand(U, N + 1)
        c = torch.zeros((U, N + 1), dtype=F64, device=DEV)
        c[:, 1:] = torch.cumsum(1.0 / ae, 1)
        return c / c[:, -1:]

    bot, top, lef, rig = coord(a[:, 0]), coord(a[:, -1]), coord(a[:, :, 0]), coord(a[:, :, -1])
    psi[:, 0, 0], psi[:, 1, 0] = 1 - bot, bot
    psi[:, 3, -1], psi[:, 2, -1] = 1 - top, top
    psi[:, 0, :, 0], psi[:, 3, :, 0] = 1 - lef, lef
    psi[:, 1, :, -1], psi[:, 2, :, -1] = 1 - rig, rig
    if Nx < 2 or Ny < 2:
        return psi
    sw, se, ne, nw = a[:, :-1, :-1], a[:, :-1, 1:], a[:, 1:, 1:], a[:, 1:, :-1]
    mx, my = Nx - 1, Ny - 1
    E = torch.zeros((U, my, mx, 5), dtype=F64, device=DEV)
    E[..., 0] = (sw + se + ne + nw) * (2.0 / 3.0)
    E[:, :, 1:, 1] = -((sw + nw) / 6.0)[:, :, 1:]
    E[:, 1:, :-1, 2] = -(se / 3.0)[:, 1:, :-1]
    E[:, 1:, :, 3] = -((sw + se) / 6.0)[:, 1:]
    E[:, 1:, 1:, 4] = -(sw / 3.0)[:, 1:, 1:]
    # -(A g)_I with g the boundary values (zero inside)
    p = psi[:, :3]
    q = lambda dj, di: p[:, :, 1 + dj:1 + dj + my, 1 + di:1 + di + mx]
    rhs = ((sw + nw)[:, None] * q(0, -1) + (se + ne)[:, None] * q(0, 1) + (sw + se)[:, None] * q(-1, 0)
           + (nw + ne)[:, None] * q(1, 0)) / 6.0 + (sw[:, None] * q(-1, -1) + se[:, None] * q(-1, 1)
                                                    + nw[:, None] * q(1, -1) + ne[:, None] * q(1, 1)) / 3.0
    x = _band_solve(E.reshape(U, my * mx, 5), rhs.permute(0, 2, 3, 1).reshape(U, my * mx, 3), mx)
    x = x.reshape(U, my, mx, 3).permute(0, 3, 1, 2)
    psi[:, :3, 1:-1, 1:-1] = x
    psi[:, 3, 1:-1, 1:-1] = 1.0 - x.sum(1)
    return psi


def _cells_64bit(case, a, oversample, with_phi=False):
    """K_e, b_e (and phi) of every cell of the samples a [S][nf][nf]."""
    S, nf, nc = a.shape[0], case["nf"], case["nc"]
    rho, pg, osc = nf // nc, case.get("pg", 0), case.get("osc", 0)
    over = [0] * (nc * nc) if oversample is None else oversample.tolist()
    groups = {}
    for cell in range(nc * nc):
        cx, cy, o = cell % nc, cell // nc, over[cell]
        x0, x1 = max(0, cx * rho - o), min(nf, (cx + 1) * rho + o)
        y0, y1 = max(0, cy * rho - o), min(nf, (cy + 1) * rho + o)
        groups.setdefault((x1 - x0, y1 - y0, cx * rho - x0, cy * rho - y0), []).append((cell, x0, y0))
    Ke = torch.zeros((S, nc * nc, 16 if pg else 10), dtype=F64, device=DEV)
    be = torch.zeros((S, nc * nc, 4), dtype=F64, device=DEV)
    phi = torch.zeros((S, nc * nc, 4, (rho + 1) ** 2), dtype=F64, device=DEV) if with_phi else None
    up = np.triu_indices(4)
    up = (torch.from_numpy(up[0]).to(DEV), torch.from_numpy(up[1]).to(DEV))
    t = torch.arange(rho + 1, dtype=F64, device=DEV) / rho
    qx, qy = t[None, :], t[:, None]
    Q = torch.stack([(1 - qx) * (1 - qy), qx * (1 - qy), qx * qy, (1 - qx) * qy])[None]

    def energy(p, q, ac):  # [U][4][4] a_cell(p_j, q_k)
        c = lambda v: (v[:, :, :-1, :-1], v[:, :, :-1, 1:], v[:, :, 1:, 1:], v[:, :, 1:, :-1])
        P, R = c(p), c(q)
        M = torch.zeros((p.shape[0], 4, 4), dtype=F64, device=DEV)
        for i in range(4):
            for k in range(4):
                v = sum(float(_KREF[r, s]) * P[r][:, i] * R[s][:, k] for r in range(4) for s in range(4))
                M[:, i, k] = (ac * v).sum((1, 2))
        return M

    step = max(1, 12000 // S)
    for (Nx, Ny, ox, oy), cells in groups.items():
        for at in range(0, len(cells), step):
            part = cells[at:at + step]
            ap = torch.stack([a[:, y0:y0 + Ny, x0:x0 + Nx] for _, x0, y0 in part], 1).reshape(-1, Ny, Nx)
            psi = _patch_psi(ap, osc)[:, :, oy:oy + rho + 1, ox:ox + rho + 1]
            ac = ap[:, oy:oy + rho, ox:ox + rho]
            C = torch.stack([psi[:, :, 0, 0], psi[:, :, 0, -1], psi[:, :, -1, -1], psi[:, :, -1, 0]], 2)
            f = torch.einsum("ujk,ukyx->ujyx", torch.linalg.inv(C), psi) if (Nx, Ny) != (rho, rho) else psi
            idx = torch.tensor([c for c, _, _ in part], device=DEV)
            sh = (S, len(part), -1)
            if pg:
                Ke[:, idx] = energy(f, Q.expand(f.shape), ac).reshape(sh)
                be[:, idx] = 0.25 / nc ** 2
            else:
                Ke[:, idx] = energy(f, f, ac)[:, up[0], up[1]].reshape(sh)
                s = (f[..., :-1, :-1] + f[..., :-1, 1:] + f[..., 1:, 1:] + f[..., 1:, :-1]).sum((2, 3))
                be[:, idx] = (s / (4.0 * nf * nf)).reshape(sh)
            if with_phi:
                phi[:, idx] = f.reshape(S, len(part), 4, -1)
    return Ke, be, phi


def _coarse_64bit(nc, Ke, be):
    S, m = Ke.shape[0], nc - 1
    K = torch.zeros((S, nc, nc, 4, 4), dtype=F64, device=DEV)
    i, j = np.triu_indices(4)
    for q, (r, c) in enumerate(zip(i, j)):
        K[..., r, c] = K[..., c, r] = Ke[:, :, q].reshape(S, nc, nc)
    B = be.reshape(S, nc, nc, 4)
    u = torch.zeros((S, nc + 1, nc + 1), dtype=F64, device=DEV)
    if m > 0:
        sw, se, ne, nw = K[:, :-1, :-1], K[:, :-1, 1:], K[:, 1:, 1:], K[:, 1:, :-1]
        E = torch.zeros((S, m, m, 5), dtype=F64, device=DEV)
        E[..., 0] = sw[..., 2, 2] + se[..., 3, 3] + ne[..., 0, 0] + nw[..., 1, 1]
        E[:, :, 1:, 1] = (sw[..., 2, 3] + nw[..., 1, 0])[:, :, 1:]
        E[:, 1:, :-1, 2] = se[..., 3, 1][:, 1:, :-1]
        E[:, 1:, :, 3] = (sw[..., 2, 1] + se[..., 3, 0])[:, 1:]
        E[:, 1:, 1:, 4] = sw[..., 2, 0][:, 1:, 1:]
        r = B[:, :-1, :-1, 2] + B[:, :-1, 1:, 3] + B[:, 1:, 1:, 0] + B[:, 1:, :-1, 1]
        u[:, 1:-1, 1:-1] = _band_solve(E.reshape(S, m * m, 5), r.reshape(S, m * m, 1), m).reshape(S, m, m)
    return u.reshape(S, -1)


def _moments(u):
    mean = u.mean(0)
    return mean, ((u - mean) ** 2).sum(0), torch.full((1,), float(u.shape[0]), dtype=F64, device=DEV)


def _fine_64bit(nf, a):
    """Q1 FEM by CG preconditioned with the constant-coefficient inverse (sine
    transform); None where it does not converge quickly."""
    S, m = a.shape[0], nf - 1
    t = torch.cos(math.pi * torch.arange(1, nf, dtype=F64, device=DEV) / nf)
    lam = 8.0 / 3.0 - (2.0 / 3.0) * (t[:, None] + t[None, :]) - (4.0 / 3.0) * t[:, None] * t[None, :]
    scale = torch.sqrt(a.amax((1, 2)) * a.amin((1, 2)))[:, None, None]

    def dst(v):
        for dim in (1, 2):
            z = torch.zeros([v.shape[0]] + [2 * nf if d == dim else v.shape[d] for d in (1, 2)], dtype=F64, device=DEV)
            z.narrow(dim, 1, m).copy_(v)
            z.narrow(dim, nf + 1, m).copy_(-v.flip(dim))
            v = -torch.fft.rfft(z, dim=dim).imag.narrow(dim, 1, m)
        return v

    sw, se, ne, nw = a[:, :-1, :-1], a[:, :-1, 1:], a[:, 1:, 1:], a[:, 1:, :-1]

    def mul(v):
        z = torch.nn.functional.pad(v, (1, 1, 1, 1))
        q = lambda dj, di: z[:, 1 + dj:1 + dj + m, 1 + di:1 + di + m]
        return ((2.0 / 3.0) * (sw + se + ne + nw) * v
                - ((sw + nw) * q(0, -1) + (se + ne) * q(0, 1) + (sw + se) * q(-1, 0) + (nw + ne) * q(1, 0)) / 6.0
                - (sw * q(-1, -1) + se * q(-1, 1) + nw * q(1, -1) + ne * q(1, 1)) / 3.0)

    dot = lambda p, q: (p * q).sum((1, 2), keepdim=True)
    b = torch.full((S, m, m), 1.0 / nf ** 2, dtype=F64, device=DEV)
    x, r = torch.zeros_like(b), b.clone()
    z = dst(dst(r) / lam) / (nf * nf) / scale
    p, rz = z.clone(), dot(r, z)
    for it in range(400):
        q = mul(p)
        al = rz / dot(p, q)
        x += al * p
        r -= al * q
        if it % 10 == 9 and float((dot(r, r) / dot(b, b)).max()) < 1e-28:
            u = torch.zeros((S, nf + 1, nf + 1), dtype=F64, device=DEV)
            u[:, 1:-1, 1:-1] = x
            return u.reshape(S, -1)
        z = dst(dst(r) / lam) / (nf * nf) / scale
        new = dot(r, z)
        p = z + (new / rz) * p
        rz = new
    return None


def _ri_64bit(case, xi):
    """The tensor Lagrange interpolant in the local parameters, cell by cell."""
    nf, nc, S = case["nf"], case["nc"], case["S"]
    rho, H = nf // nc, 1.0 / nc
    Ke = torch.zeros((S, nc * nc, 10), dtype=F64, device=DEV)
    be = torch.zeros((S, nc * nc, 4), dtype=F64, device=DEV)
    for cell in range(nc * nc):
        cx, cy = cell % nc, cell // nc
        dims = []
        for by in range(case["nby"]):
            for bx in range(case["nbx"]):
                px, py = (bx + 0.5) / case["nbx"], (by + 0.5) / case["nby"]
                dx = max(cx * H - px, 0.0, px - (cx + 1) * H)
                dy = max(cy * H - py, 0.0, py - (cy + 1) * H)
                g = abs(case["scale"]) * math.exp(-(dx * dx + dy * dy) / case["width"] ** 2)
                nu, term = 0, g
                while nu < case["nu_max"] and term > case["eps"]:
                    nu += 1
                    term *= 0.5 * g / (nu + 1)
                if nu:
                    dims.append((by * case["nbx"] + bx, np.polynomial.legendre.leggauss(nu + 1)[0]))
        pts = np.array(np.meshgrid(*[n for _, n in dims], indexing="ij")).reshape(len(dims), -1).T if dims else np.zeros((1, 0))
        xp = torch.zeros((len(pts), xi.shape[1]), dtype=F64, device=DEV)
        wts = torch.ones((S, 1), dtype=F64, device=DEV)
        for k, (i, nodes) in enumerate(dims):
            xp[:, i] = torch.from_numpy(pts[:, k].copy()).to(DEV)
            t = xi[:, i]
            l = torch.stack([math.prod([1.0] + [1.0 / (nodes[j] - nodes[q]) for q in range(len(nodes)) if q != j])
                             * torch.stack([t - nodes[q] for q in range(len(nodes)) if q != j]).prod(0)
                             for j in range(len(nodes))], 1)
            wts = (wts[:, :, None] * l[:, None, :]).reshape(S, -1)
        xs = (torch.arange(cx * rho, (cx + 1) * rho, dtype=F64, device=DEV) + 0.5) / nf
        ys = (torch.arange(cy * rho, (cy + 1) * rho, dtype=F64, device=DEV) + 0.5) / nf
        K, b, _ = _cells_64bit(dict(nf=rho, nc=1), _coefficient(case, xp, xs, ys), None)
        Ke[:, cell] = wts @ K[:, 0]
        be[:, cell] = wts @ b[:, 0] * H * H
    return Ke, be


def exact(case, seed):
    path = case["path"]
    if path == "pod":
        return None  # depends on the trained basis
    inp = _inputs(case, seed)
    if path == "coarse":
        u = _coarse_64bit(case["nc"], inp["Ke"], inp["be"])
        mean, m2, count = _moments(u)
        return dict(u=u, mean=mean, m2=m2, count=count)
    if path == "ri":
        Ke, be = _ri_64bit(case, inp["xi"])
        return dict(Ke=Ke, be=be, fell=None)
    nf = case["nf"]
    c = _centroids(nf)
    a = inp.get("a") if inp.get("a") is not None else _coefficient(case, inp["xi"], c, c)
    if path == "sample":
        return dict(a=a)
    if path == "fine":
        u = _fine_64bit(nf, a)
        return None if u is None else dict(u=u)
    Ke, be, _ = _cells_64bit(case, a, inp["oversample"])
    if path == "upscale":
        return dict(Ke=Ke, be=be)
    u = _coarse_64bit(case["nc"], Ke, be)
    if path == "step":
        return dict(a=a, Ke=Ke, be=be, u=u)
    mean, m2, count = _moments(u)
    return dict(u=u, mean=mean, m2=m2, count=count)
