"""The tiled kernels at the sizes where their rules turn, against the FP64
oracle: the FP32 trailing update's 8-row tiles (half bandwidths around 24, 32
and 40, and pitches that are not multiples of 8), the FP64 forms with four and
two units per warp, the unit order by patch size with flagged cells and
oversampling clipped to a small grid, the CTA-wide banded solves, the
multigrid's level counts, the reduced solves at every tile remainder of the
rank and the sampling's bump groups.

Tolerances as in the parity tests: FP64 1e-11 (relative Frobenius of a unit's
K_e and b_e), refinement 1e-10, FP32 1e-5; coarse solutions 1e-9 and the
multigrid solutions 1e-10 in relative L2; a sampled coefficient within the
rounding of its exponent, 4 (g sum psi 8 eps + 4 eps)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

from paper_1607_00693_gb300 import api

DEV = "cuda:0"
TOL = {api.FP64: 1e-11, api.FP32_REFINED: 1e-10, api.FP32: 1e-5}


@pytest.fixture(scope="module")
def orc():
    from paper_1607_00693_gb300.build import build_library
    import oracle
    build_library()
    oracle.build()
    return oracle


def _t(x, dtype=None):
    return torch.from_numpy(np.ascontiguousarray(x, dtype=dtype)).to(DEV)


def _rel(x, y):
    return float(np.max(np.linalg.norm(x - y, axis=-1) / np.linalg.norm(y, axis=-1)))


def _coef(S, nf, seed, s=1.0):
    return np.exp(np.random.default_rng(seed).uniform(-s, s, size=(S, nf, nf)))


def _upscale(nf, nc, a, ov, mo, precision, slots=None):
    g = api.grid(nf, nc)
    S, cells = a.shape[0], nc * nc
    Ke = torch.zeros((S, cells, 10), dtype=torch.float64, device=DEV)
    be = torch.zeros((S, cells, 4), dtype=torch.float64, device=DEV)
    st = torch.full((S, cells), 99, dtype=torch.int32, device=DEV)
    ws = None
    if slots:
        ws = torch.zeros(api.stomsfem_upscale_workspace_size(g, mo, precision)[0] * slots, dtype=torch.uint8, device=DEV)
    api.stomsfem_upscale(g, _t(a), Ke, be, oversample=None if ov is None else _t(ov, np.int8), max_oversample=mo,
                         precision=precision, unit_status=st, workspace=ws)
    torch.cuda.synchronize()
    return Ke.cpu().numpy(), be.cpu().numpy(), st.cpu().numpy()


# half bandwidth = rho + 2 o inside the domain: 17 .. 41 with mixed patches
@pytest.mark.parametrize("rho,mo", [(17, 0), (21, 2), (24, 0), (25, 0), (24, 4), (29, 0), (32, 0), (33, 0), (30, 3),
                                    (32, 4), (36, 0), (37, 1), (40, 0), (41, 0)])
@pytest.mark.parametrize("precision", [api.FP32, api.FP32_REFINED])
def test_fp32_tiles_at_the_band_edges(orc, rho, mo, precision):
    nc, S = 2 + (mo > 0), 3
    nf = nc * rho
    a = _coef(S, nf, 100 + rho)
    ov = np.random.default_rng(rho).integers(0, mo + 1, size=nc * nc).astype(np.int8) if mo else None
    Ko, bo = orc.upscale(nf, nc, 1.0, a, ov)
    Kg, bg, st = _upscale(nf, nc, a, ov, mo, precision)
    assert not st.any()
    assert _rel(Kg, Ko) <= TOL[precision] and _rel(bg, bo) <= TOL[precision]


# four units per warp up to b = 12 from three samples on; two below, beyond,
# or with a workspace of less than a block of eight slots
@pytest.mark.parametrize("rho,mo", [(1, 0), (2, 0), (3, 0), (4, 0), (5, 1), (8, 0), (8, 2), (12, 0), (13, 0)])
@pytest.mark.parametrize("S,slots", [(1, None), (3, None), (5, None), (9, 8), (5, 4)])
def test_fp64_units_per_warp(orc, rho, mo, S, slots):
    nc = 5
    nf = nc * rho
    a = _coef(S, nf, 200 + rho)
    ov = np.random.default_rng(rho).integers(0, mo + 1, size=nc * nc).astype(np.int8) if mo else None
    Ko, bo = orc.upscale(nf, nc, 1.0, a, ov)
    Kg, bg, st = _upscale(nf, nc, a, ov, mo, api.FP64, slots)
    assert not st.any()
    assert _rel(Kg, Ko) <= 1e-11 and _rel(bg, bo) <= 1e-11


# four units per warp need a full chip (about 1000 pairs of units): every
# remainder of the samples by four, with and without oversampling
@pytest.mark.parametrize("rho,mo", [(1, 1), (2, 0), (3, 0), (4, 0), (4, 1), (5, 0), (8, 0), (6, 3), (12, 0)])
@pytest.mark.parametrize("S", [8, 9, 10, 11])
def test_fp64_four_units_per_warp(orc, rho, mo, S):
    nc = 16
    nf = nc * rho
    a = _coef(S, nf, 300 + rho)
    ov = np.random.default_rng(rho).integers(0, mo + 1, size=nc * nc).astype(np.int8) if mo else None
    Ko, bo = orc.upscale(nf, nc, 1.0, a, ov)
    Kg, bg, st = _upscale(nf, nc, a, ov, mo, api.FP64)
    assert not st.any()
    assert _rel(Kg, Ko) <= 1e-11 and _rel(bg, bo) <= 1e-11


@pytest.mark.parametrize("nf,nc,mo", [(48, 8, 3), (8, 4, 100), (70, 35, 2)])
@pytest.mark.parametrize("precision", [api.FP64, api.FP32])
def test_order_by_patch_size_with_flagged_cells(orc, nf, nc, mo, precision):
    """More cells than a pass of the list kernel (35^2), cells outside [0, mo]
    and an oversampling far beyond the grid."""
    a = _coef(2, nf, nf)
    ov = np.random.default_rng(nf).integers(0, min(mo, 4) + 1, size=nc * nc).astype(np.int8)
    if mo == 100:
        ov[1::3] = 100
    ok = np.ones(nc * nc, dtype=bool)
    bad = ov.copy()
    bad[2::5] = -1
    bad[3::7] = 127
    ok[2::5] = ok[3::7] = False
    Ko, bo = orc.upscale(nf, nc, 1.0, a, ov)
    Kg, bg, st = _upscale(nf, nc, a, bad, mo, precision)
    assert not st[:, ok].any() and (st[:, ~ok] == -1).all() and np.isnan(Kg[:, ~ok]).all()
    assert _rel(Kg[:, ok], Ko[:, ok]) <= TOL[precision] and _rel(bg[:, ok], bo[:, ok]) <= TOL[precision]


# (small calls keep the cell order unless told otherwise; the default takes
# the patch order once there is more than one block an SM)
@pytest.mark.parametrize("nf,nc,mo,S", [(48, 8, 3, 3), (8, 4, 100, 2), (16, 16, 1, 5), (16, 16, 1, 3), (70, 35, 2, 1)])
@pytest.mark.parametrize("precision", [api.FP64, api.FP32_REFINED, api.FP32])
def test_unit_order_does_not_change_the_results(nf, nc, mo, S, precision):
    a = _t(_coef(S, nf, nf))
    ov = np.random.default_rng(nf).integers(0, min(mo, 4) + 1, size=nc * nc).astype(np.int8)
    ov[2::5] = -1
    if mo == 100:
        ov[1::3] = 100
    g, out = api.grid(nf, nc), []
    for order in (None, api.ORDER_CELL, api.ORDER_PATCH):
        Ke = torch.full((S, nc * nc, 10), 7.0, dtype=torch.float64, device=DEV)
        be = torch.full((S, nc * nc, 4), 7.0, dtype=torch.float64, device=DEV)
        api.stomsfem_upscale(g, a, Ke, be, oversample=_t(ov), max_oversample=mo, precision=precision, order=order)
        out.append((Ke.cpu().numpy(), be.cpu().numpy()))
    for K, b in out[1:]:
        assert np.array_equal(K, out[0][0], equal_nan=True) and np.array_equal(b, out[0][1], equal_nan=True)
    assert np.isfinite(out[0][0][:, ov >= 0]).all()


@pytest.mark.parametrize("nc", [1, 2, 3, 4, 9, 16, 31, 32, 33, 47, 63])
def test_coarse_solve_sizes(orc, nc):
    """Last blocks of every remainder, one and two rows per lane, S above and
    below the workspace's slots, an indefinite sample beside sound ones."""
    S = 5
    a = _coef(S, 2 * nc, nc)
    K, b = orc.upscale(2 * nc, nc, 1.0, a)
    uo = orc.coarse_solve(nc, K, b)
    g = api.grid(2 * nc, nc)
    for slots in (None, 2):
        ws = None if slots is None else torch.zeros(
            api.stomsfem_coarse_workspace_size(g, 2), dtype=torch.uint8, device=DEV)
        u = torch.zeros((S, (nc + 1) ** 2), dtype=torch.float64, device=DEV)
        mean, m2 = (torch.zeros((nc + 1) ** 2, dtype=torch.float64, device=DEV) for _ in range(2))
        cnt = torch.zeros(1, dtype=torch.float64, device=DEV)
        api.stomsfem_coarse_solve(g, _t(K), _t(b), u, mean, m2, cnt, workspace=ws)
        ug = u.cpu().numpy()
        assert np.linalg.norm(ug - uo) <= 1e-9 * max(np.linalg.norm(uo), 1e-300)
        mo, vo = uo.mean(0), ((uo - uo.mean(0)) ** 2).sum(0)
        assert np.allclose(mean.cpu().numpy(), mo, rtol=1e-9, atol=1e-12)
        assert np.allclose(m2.cpu().numpy(), vo, rtol=1e-8, atol=1e-14) and float(cnt[0]) == S
    if nc > 2:
        K[2] = -K[2]
        api.stomsfem_coarse_solve(g, _t(K), _t(b), u)
        ug = u.cpu().numpy()
        inner = uo[2] != 0
        assert np.isnan(ug[2][inner]).all()
        keep = [0, 1, 3, 4]
        assert np.linalg.norm(ug[keep] - uo[keep]) <= 1e-9 * np.linalg.norm(uo[keep])


# 16 lanes per system up to 16 unknowns (nc = 5, 4^2 interior nodes; nc = 3 with all
# nodes unknown), a CTA beyond; ragged groups of eight systems
@pytest.mark.parametrize("nc", [1, 2, 3, 4, 5, 6])
@pytest.mark.parametrize("S", [2, 7, 8, 37])
def test_small_systems(orc, nc, S):
    a = _coef(S, 2 * nc, 10 * nc + S)
    K, b = orc.upscale(2 * nc, nc, 1.0, a)
    g, nn = api.grid(2 * nc, nc), (nc + 1) ** 2
    bad = S // 2  # an indefinite sample among sound ones
    keep = np.arange(S) != bad
    Kb = K.copy()
    Kb[bad] = -Kb[bad]
    u = torch.full((S, nn), 7.0, dtype=torch.float64, device=DEV)
    api.stomsfem_coarse_solve(g, _t(Kb), _t(b), u)
    ug, uo = u.cpu().numpy(), orc.coarse_solve(nc, K, b)
    assert np.linalg.norm((ug - uo)[keep]) <= 1e-9 * np.linalg.norm(uo[keep]) and (ug[keep][uo[keep] == 0] == 0).all()
    inner = np.zeros((nc + 1, nc + 1), bool)
    inner[1:-1, 1:-1] = True
    assert np.isnan(ug[bad][inner.ravel()]).all() and (ug[bad][~inner.ravel()] == 0).all()
    # mixed data: prescribed left and right, every node an unknown
    dm = np.zeros((nc + 1, nc + 1), np.uint8)
    dm[:, 0] = dm[:, -1] = 1
    gv = np.where(dm, np.arange(nc + 1)[None, :] + 0.5, 0.0)
    api.stomsfem_coarse_solve_bc(g, 0, _t(Kb), _t(b), _t(dm.ravel()), _t(gv.ravel()), u)
    ug, uo = u.cpu().numpy(), orc.coarse_solve_bc(nc, K, b, dm.ravel(), gv.ravel())
    assert np.linalg.norm((ug - uo)[keep]) <= 1e-9 * np.linalg.norm(uo[keep])
    if nc > 1:
        assert np.isnan(ug[bad]).all()
    # the fine grid's own system
    af = _coef(S, nc, nc + S)
    uf = torch.full((S, nn), 7.0, dtype=torch.float64, device=DEV)
    api.stomsfem_fine_fem(api.grid(nc, 1), _t(af), uf)
    for s in range(S):
        ref = orc.fine_fem(nc, 1.0, af[s]).reshape(-1) if nc > 1 else np.zeros(nn)
        assert np.linalg.norm(uf[s].cpu().numpy() - ref) <= 1e-10 * np.linalg.norm(ref) + 1e-300


@pytest.mark.parametrize("r,place", [(2, "corner"), (2, "edge")] +
                         [(r, p) for r in (4, 8, 16) for p in ("corner", "edge", "centre")])
def test_fine_solver_just_below_the_contrast_rule(orc, r, place):
    """Inclusions of contrast 999, mirrored so that a bilinear level's elements of r^2
    fine cells are all alike (largest eigenvalues of D^-1 A up to 2.354 on some
    level): the bilinear cycle has to converge.  The residual is 1e-13 of the load's
    and the load is smooth, so the solution's error is of that order; the direct
    reference's rounding (about its condition number, 1e7, times 1e-16 at most) sets
    the bound."""
    nf = 128
    a = np.ones((1, nf, nf))
    x = np.arange(nf) % (2 * r)
    m = np.minimum(x, 2 * r - 1 - x)  # 0 .. r - 1 from one mirror line to the other
    side = max(1, r // 4)
    low, mid = m < side, np.abs(m - (r - 1) / 2) < max(side, 1) / 2 + 0.25
    hot = {"corner": low[:, None] & low[None, :], "edge": low[:, None] & mid[None, :],
           "centre": mid[:, None] & mid[None, :]}[place]
    a[0][hot] = 999.0
    u = torch.zeros((1, (nf + 1) ** 2), dtype=torch.float64, device=DEV)
    api.stomsfem_fine_fem(api.grid(nf, 1), _t(a), u)
    uo = orc.fine_fem(nf, 1.0, a[0]).reshape(-1)
    assert np.linalg.norm(u[0].cpu().numpy() - uo) <= 1e-9 * np.linalg.norm(uo)


@pytest.mark.parametrize("contrast", [1.0, 2e3])
@pytest.mark.parametrize("unit", [2.0 ** 125, 2.0 ** -132, 1e-150, 1e150])
def test_fine_solver_coefficient_units(orc, contrast, unit):
    """A coefficient whose FP32 value or its reciprocal leaves the type's range; a load
    of the same side keeps the solution's magnitude ordinary or the residual in
    range."""
    nf, S = 96, 2
    a = np.exp(np.random.default_rng(nf).uniform(-1.0, 1.0, size=(S, nf, nf)))
    a[:, 30:32, :] *= contrast
    u = torch.zeros((S, (nf + 1) ** 2), dtype=torch.float64, device=DEV)
    f = min(max(unit, 1e-20), 1e20)  # (the FP32 residual's range is the load's)
    api.stomsfem_fine_fem(api.grid(nf, 1, f), _t(a * unit), u)
    for s in range(S):
        uo = orc.fine_fem(nf, 1.0, a[s]).reshape(-1)
        assert np.linalg.norm(u[s].cpu().numpy() * (unit / f) - uo) <= 1e-10 * np.linalg.norm(uo)


@pytest.mark.parametrize("contrast", [1.0, 2e3])
@pytest.mark.parametrize("shift", [0, 4, 8, 12])
def test_fine_solver_workspace_alignment(orc, contrast, shift):
    """A workspace of exactly the reported size at any place: the solver's 16-byte
    accesses start at a boundary of their own."""
    nf, S = 80, 3
    a = np.exp(np.random.default_rng(nf).uniform(-1.0, 1.0, size=(S, nf, nf)))
    a[:, 30:32, :] *= contrast
    g = api.grid(nf, 1)
    need = api.stomsfem_fine_fem_workspace_size(g, S)
    buf = torch.full((need + 64,), 0xFF, dtype=torch.uint8, device=DEV)
    assert buf.data_ptr() % 16 == 0
    u = torch.zeros((S, (nf + 1) ** 2), dtype=torch.float64, device=DEV)
    api.stomsfem_fine_fem(g, _t(a), u, workspace=buf[shift:shift + need])
    assert bool((buf[shift + need:] == 0xFF).all()) and bool((buf[:shift] == 0xFF).all())
    for s in range(S):
        uo = orc.fine_fem(nf, 1.0, a[s]).reshape(-1)
        assert np.linalg.norm(u[s].cpu().numpy() - uo) <= 1e-10 * np.linalg.norm(uo)


# one and 32 threads per node; the rule turns at 48 samples, and one more for each
# 56 nodes past 2400
@pytest.mark.parametrize("n", [9, 1089, 9409, 40001])
@pytest.mark.parametrize("S", [1, 3, 48, 49, 65, 66, 173, 174])
def test_moments_threads_per_node(n, S):
    """Two batches against NumPy; values in [0, 1): sums of S terms carry at most S
    roundings, the squared deviations at most 12 S of their sum."""
    u = np.random.default_rng(n + S).uniform(size=(2, S, n))
    mean, m2 = (torch.zeros(n, dtype=torch.float64, device=DEV) for _ in range(2))
    cnt = torch.zeros(1, dtype=torch.float64, device=DEV)
    for b in range(2):
        api.stomsfem_mc_moments(_t(u[b]), mean, m2, cnt)
    v = u.reshape(2 * S, n)
    tol = 32 * 2 * S * np.finfo(float).eps
    assert float(cnt[0]) == 2 * S
    assert np.allclose(mean.cpu().numpy(), v.mean(0), rtol=tol, atol=tol)
    assert np.allclose(m2.cpu().numpy(), ((v - v.mean(0)) ** 2).sum(0), rtol=tol, atol=tol * S)


# levels 66, 33 is odd: not offered; one to four levels below the finest
@pytest.mark.parametrize("nf", [2, 9, 33, 64, 72, 80, 96, 112, 128, 240])
@pytest.mark.parametrize("contrast", [False, True])
def test_fine_solver_levels(orc, nf, contrast):
    r = np.random.default_rng(nf)
    a = np.exp(r.uniform(-1.0, 1.0, size=(2, nf, nf)))
    if contrast:
        a[:, nf // 3: nf // 3 + 2, :] = 2e3
    g = api.grid(nf, 1)
    u = torch.zeros((2, (nf + 1) ** 2), dtype=torch.float64, device=DEV)
    api.stomsfem_fine_fem(g, _t(a), u)
    for s in range(2):
        uo = orc.fine_fem(nf, 1.0, a[s]).reshape(-1)
        assert np.linalg.norm(u[s].cpu().numpy() - uo) <= 1e-10 * np.linalg.norm(uo)


@pytest.mark.parametrize("rank", [1, 2, 3, 4, 5, 7, 8, 26, 27])
def test_reduced_solves_at_every_remainder(orc, rank):
    """Rank remainders of the 4 x 4 tiles and ragged sample counts against the
    FP64-refined online stage, within the unrefined stage's 5e-3."""
    nf, nc, Ns, S = 16, 2, 12, 131
    a_tr, a = _coef(Ns, nf, 1, 0.3), _coef(S, nf, 2, 0.3)
    g = api.grid(nf, nc)
    phi = _t(orc.upscale(nf, nc, 1.0, a_tr, want_phi=True)[2])
    h, rk = api.stomsfem_pod_build(g, phi, _t(a_tr), ranks=[rank, max(1, rank - 1), rank, 1])
    try:
        out = []
        for refine in (0, 4):
            Ke = torch.zeros((S, nc * nc, 10), dtype=torch.float64, device=DEV)
            be = torch.zeros((S, nc * nc, 4), dtype=torch.float64, device=DEV)
            st = torch.full((S, nc * nc), 9, dtype=torch.int32, device=DEV)
            api.stomsfem_pod_upscale(h, g, _t(a), Ke, be, refine_iters=refine, unit_status=st)
            assert not st.cpu().numpy().any()
            out.append((Ke.cpu().numpy(), be.cpu().numpy()))
        assert _rel(out[0][0], out[1][0]) <= 5e-3 and _rel(out[0][1], out[1][1]) <= 5e-3
        for n in (1, 31, 32, 33):  # a sample's result does not depend on the batch
            Ke = torch.zeros((n, nc * nc, 10), dtype=torch.float64, device=DEV)
            be = torch.zeros((n, nc * nc, 4), dtype=torch.float64, device=DEV)
            api.stomsfem_pod_upscale(h, g, _t(a[:n]), Ke, be)
            assert np.array_equal(Ke.cpu().numpy(), out[0][0][:n]) and np.array_equal(be.cpu().numpy(), out[0][1][:n])
    finally:
        api.stomsfem_pod_destroy(h)


# one unit per thread (more than 2048 units) at every remainder of the rank, with one K
# step (the streaming product: 1500 samples of 64 cells are 768 tiles, five a CTA with
# a change of cell among them; one half of the accumulator or two) and several (H/h =
# 16), against batches of 32, which take a warp per unit and the other product
@pytest.mark.parametrize("rho,nc,rank,S", [(8, 8, 27, 1500), (8, 8, 12, 1500)] +
                         [(8, 8, r, 131) for r in (1, 2, 3, 4, 5, 7, 8, 26, 27)] + [(16, 4, 5, 200), (16, 4, 27, 200)])
@pytest.mark.parametrize("split", [1, 0])
def test_reduced_units_do_not_depend_on_the_batch(rho, nc, rank, S, split):
    nf, cells, Ns = rho * nc, nc * nc, 12
    g = api.grid(nf, nc)
    a_tr, a = _t(_coef(Ns, nf, 1, 0.3)), _t(_coef(S, nf, 2, 0.3))
    phi = torch.zeros((Ns, cells, 4, (rho + 1) ** 2), dtype=torch.float64, device=DEV)
    K0, b0 = (torch.zeros((Ns, cells, k), dtype=torch.float64, device=DEV) for k in (10, 4))
    api.stomsfem_upscale(g, a_tr, K0, b0, phi=phi)
    h, _ = api.stomsfem_pod_build(g, phi, a_tr, ranks=[max(1, rank - c % 3) for c in range(cells)])

    def online(lo, hi, refine=0):
        n = hi - lo
        Ke = torch.full((n, cells, 10), 7.0, dtype=torch.float64, device=DEV)
        be = torch.full((n, cells, 4), 7.0, dtype=torch.float64, device=DEV)
        st = torch.full((n, cells), 9, dtype=torch.int32, device=DEV)
        api.stomsfem_pod_upscale(h, g, a[lo:hi].contiguous(), Ke, be, refine_iters=refine, unit_status=st)
        assert not st.cpu().numpy().any()
        return Ke.cpu().numpy(), be.cpu().numpy()

    try:
        api.stomsfem_pod_set_gemm_split(h, split)
        Ke, be = online(0, S)
        for lo in list(range(0, S - 32, 32 if S < 300 else 96)) + [S - 32]:
            K, b = online(lo, lo + 32)
            assert np.array_equal(K, Ke[lo:lo + 32]) and np.array_equal(b, be[lo:lo + 32])
        if rho <= 8:
            # split: the dropped products are below 2^-16 of the sums, three of
            # them per entry of K_e, amplified by the solves at most tenfold
            tol = 5e-4 if split else 5e-3
            K, b = online(S - 40, S, 4)
            assert _rel(Ke[S - 40:], K) <= tol and _rel(be[S - 40:], b) <= tol
    finally:
        api.stomsfem_pod_destroy(h)


@pytest.mark.parametrize("nf,nbx,nby,width,S", [(1, 1, 1, 0.3, 3), (7, 3, 5, 0.02, 2), (33, 4, 4, 0.1, 40),
                                                (64, 17, 2, 0.01, 3), (257, 33, 9, 0.02, 2), (300, 5, 64, 0.004, 2),
                                                (520, 64, 3, 0.5, 1)])
@pytest.mark.parametrize("kind", [api.FIELD_EXP, api.FIELD_EXP_SIGMOID])
def test_sampling_bump_groups(orc, nf, nbx, nby, width, S, kind):
    fld = dict(kind=kind, nbx=nbx, nby=nby, width=width, scale=0.7, contrast_log=np.log(1e3), gain=2.0)
    xi = np.random.default_rng(nf).uniform(-1, 1, size=(S, nbx * nby))
    ref = orc.sample_coef(nf, fld, xi)
    a = torch.zeros((S, nf, nf), dtype=torch.float64, device=DEV)
    api.stomsfem_sample_coef(api.grid(nf, 1), api.field_from_dict(fld), _t(xi), a)
    x = (np.arange(nf) + 0.5) / nf
    psi = [np.exp(-((x[:, None] - (np.arange(n) + 0.5) / n) / width) ** 2).sum(1).max() for n in (nbx, nby)]
    gain = 0.7 if kind == api.FIELD_EXP else np.log(1e3) * 2.0 / 4
    eps = np.finfo(float).eps
    bound = 4 * (gain * psi[0] * psi[1] * 8 * eps + 4 * eps) + (0 if kind == api.FIELD_EXP else 8 * np.log(1e3) * eps)
    assert np.max(np.abs(a.cpu().numpy() / ref - 1)) <= bound


def test_sampling_large_and_non_finite_amplitudes():
    """Far bumps are left out only below the amplitude bound: a large one is
    summed everywhere, and a NaN reaches every element of its sample."""
    nf, n, width = 64, 16, 0.01
    fld = api.field(api.FIELD_AFFINE, n, n, width, 1.0, 0.0, 2.0)
    xi = torch.zeros((3, n * n), dtype=torch.float64, device=DEV)
    xi[1, 0] = 1e200
    xi[2, 5] = float("nan")
    a = torch.zeros((3, nf, nf), dtype=torch.float64, device=DEV)
    api.stomsfem_sample_coef(api.grid(nf, 1), fld, xi, a)
    got = a.cpu().numpy()
    x = (np.arange(nf) + 0.5) / nf
    b = np.exp(-((x - 0.5 / n) / width) ** 2)
    want = 2.0 + 1e200 * b[:, None] * b[None, :]
    assert np.array_equal(got[0], np.full((nf, nf), 2.0))
    near = want < 1e300
    assert np.allclose(got[1][near], want[near], rtol=1e-10)
    assert np.isnan(got[2]).all()


@pytest.mark.parametrize("nf,nbx,nby,width,S", [(33, 3, 4, 0.2, 300), (77, 16, 5, 0.06, 60), (97, 4, 3, 0.3, 150),
                                                (130, 20, 8, 0.03, 40), (225, 2, 9, 0.4, 30)])
def test_sampling_row_groups_and_strips(orc, nf, nbx, nby, width, S):
    """Column groups of 1..8 warps with shared bump values, strips of uneven
    rest and blocks that take several (place, sample) pairs; distant narrow
    bumps whose values are zero."""
    fld = dict(kind=api.FIELD_EXP, nbx=nbx, nby=nby, width=width, scale=0.7, contrast_log=0.0, gain=1.0)
    xi = np.random.default_rng(nf).uniform(-1, 1, size=(S, nbx * nby))
    ref = orc.sample_coef(nf, fld, xi)
    a = torch.zeros((S, nf, nf), dtype=torch.float64, device=DEV)
    api.stomsfem_sample_coef(api.grid(nf, 1), api.field_from_dict(fld), _t(xi), a)
    x = (np.arange(nf) + 0.5) / nf
    psi = [np.exp(-((x[:, None] - (np.arange(n) + 0.5) / n) / width) ** 2).sum(1).max() for n in (nbx, nby)]
    eps = np.finfo(float).eps
    assert np.max(np.abs(a.cpu().numpy() / ref - 1)) <= 4 * (0.7 * psi[0] * psi[1] * 8 * eps + 4 * eps)


# dynamic shared memory of exactly 48 KB: the bump values of 64-row strips
# alone (47 + 48 bumps), and with the shared column values (the others)
@pytest.mark.parametrize("nf,nbx,nby,S", [(1024, 47, 48, 20), (1024, 48, 47, 20), (128, 21, 32, 1000),
                                          (128, 16, 47, 700), (110, 20, 44, 700)])
def test_sampling_at_the_shared_memory_limit(orc, nf, nbx, nby, S):
    width = 0.02
    fld = dict(kind=api.FIELD_EXP, nbx=nbx, nby=nby, width=width, scale=0.7, contrast_log=0.0, gain=1.0)
    xi = np.random.default_rng(nf).uniform(-1, 1, size=(S, nbx * nby))
    a = torch.zeros((S, nf, nf), dtype=torch.float64, device=DEV)
    api.stomsfem_sample_coef(api.grid(nf, 1), api.field_from_dict(fld), _t(xi), a)
    some = [0, S // 2, S - 1]
    ref = orc.sample_coef(nf, fld, xi[some])
    x = (np.arange(nf) + 0.5) / nf
    psi = [np.exp(-((x[:, None] - (np.arange(n) + 0.5) / n) / width) ** 2).sum(1).max() for n in (nbx, nby)]
    eps = np.finfo(float).eps
    assert np.max(np.abs(a[some].cpu().numpy() / ref - 1)) <= 4 * (0.7 * psi[0] * psi[1] * 8 * eps + 4 * eps)


def test_sampling_affine_field_without_mean():
    """With no mean level beside them the far bumps are the field: every
    element relative to its own value.  Places, widths and products of the
    reference differ from the kernel's by roundings of the exponent (at most
    2 (0.125 / 0.01)^2 = 313): 8 eps each, and of the sums."""
    nf, n, width, S = 1024, 4, 0.01, 3
    fld = api.field(api.FIELD_AFFINE, n, n, width, 1.0, 0.0, 0.0)
    xi = np.random.default_rng(5).uniform(0.5, 1.0, size=(S, n * n))
    a = torch.zeros((S, nf, nf), dtype=torch.float64, device=DEV)
    api.stomsfem_sample_coef(api.grid(nf, 1), fld, _t(xi), a)
    x = (np.arange(nf) + 0.5) / nf
    t = -((x[:, None] - (np.arange(n) + 0.5) / n) ** 2) / width ** 2
    b = np.exp(t)
    want = np.einsum("yj,sji,xi->syx", b, xi.reshape(S, n, n), b)
    assert want.min() < 1e-100
    assert np.max(np.abs(a.cpu().numpy() / want - 1)) <= (8 * 313 + 64) * np.finfo(float).eps


@pytest.mark.parametrize("eps", [1e-3, 1e-2])
def test_interpolation_units_per_thread(eps):
    """A sample's interpolant does not depend on the batch: one and two units
    a thread, ragged tiles, a parameter outside the box."""
    from paper_1607_00693_gb300 import workloads as W
    w = W.workload("msfem_64")
    g = api.grid(w["nf"], w["nc"], w["f"])
    h, _ = api.stomsfem_ri_build(g, api.field_from_dict(w["field"]), eps, 8, api.RI_LEGENDRE)
    try:
        S, cells = 5003, w["nc"] ** 2
        xi = _t(W.draw_xi(w["field"], S, 3))
        xi[0, 2] = 1.5
        ref = None
        for n in (S, 1, 2, 33, 130, 700):
            Ke = torch.full((n, cells, 10), 7.0, dtype=torch.float64, device=DEV)
            be = torch.full((n, cells, 4), 7.0, dtype=torch.float64, device=DEV)
            fb = torch.full((n, cells), 9, dtype=torch.uint8, device=DEV)
            api.stomsfem_ri_upscale(h, g, xi[:n].contiguous(), None, Ke, be, fb)
            out = [t.cpu().numpy() for t in (Ke, be, fb)]
            if ref is None:
                ref = out
                assert set(np.unique(out[2])) == {0, 2} and not out[2][1:].any()
            for x, y in zip(out, ref):
                assert np.array_equal(x, y[:n], equal_nan=x.dtype.kind == "f")
    finally:
        api.stomsfem_ri_destroy(h)
