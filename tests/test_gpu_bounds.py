"""The harmonic sum by bounds (csrc/harmonic_bound.cu) against the plain one.

fdas_threshold on a plan that sums by bounds must return exactly the crossings
of the sums that fdas_harmonic_sums writes out for the same plane (another
kernel, which sums every cell): the same cells, bit-identical powers.  The
statistics given set the thresholds: a mean of 1 on unit-mean planes is the
search's case (few boxes summed exactly), smaller ones send more boxes to the
exact sums, and the smallest more than their list holds (the plain kernel takes
over).
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def capi():
    import paper_2211_13517_gb300 as pkg
    pkg.build()
    from paper_2211_13517_gb300 import capi as c
    c.lib()
    return c


def _plane(plan, seed, interbin=False):
    """Exponential cells (unit mean) with bright ones, among them the edges."""
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    shape = (plan.info.n_z, plan.info.plane_cols)
    p = -torch.log1p(-torch.rand(shape, generator=g, device="cuda"))
    r = np.random.RandomState(seed)
    for _ in range(12):
        p[r.randint(shape[0]), r.randint(shape[1])] = float(r.uniform(20.0, 300.0))
    p[0, 0] = p[-1, -1] = p[0, -1] = p[-1, 0] = 60.0
    p[:, 4:12] = 0.0
    if plan.info.precision == 2:
        p = p / 16.0
    return p.to(plan.spec_dtype)


def _check(capi, plan, plane, mean):
    info = plan.info
    stats = torch.tensor([mean, mean], dtype=torch.float64, device="cuda")
    st, c, nf = plan.threshold(plane, stats, capacity=1 << 23)
    assert st == capi.FDAS_OK and nf == len(c)
    sums = plan.harmonic_sums(plane)
    at = 0   # records come ordered by (harm, iz, ir)
    for s in range(info.n_stages):
        thr = np.float32(mean * info.stage_factor[s])
        z, r = torch.nonzero(sums[s] > float(thr), as_tuple=True)
        mine = c[at:at + len(z)]
        at += len(z)
        assert np.all(mine["harm"] == 1 << s)
        assert np.array_equal(mine["iz"], z.cpu().numpy())
        assert np.array_equal(mine["ir"], r.cpu().numpy())
        assert np.array_equal(mine["power"], sums[s][z, r].cpu().numpy())
    assert at == nf
    return nf


@pytest.mark.parametrize("prec", [0, 1, 2])
@pytest.mark.parametrize("harm", [1, 2, 4, 8, 16])
@pytest.mark.parametrize("n_log2,z_max,z_step", [(12, 0.0, 1.0), (12, 2.0, 1.0), (13, 5.0, 0.5),
                                                 (15, 96.0, 1.0)])
def test_threshold_is_the_plain_sums(capi, prec, harm, n_log2, z_max, z_step):
    plan = capi.Plan(1 << n_log2, 64e-6, z_max, z_step, 2048, harm, precision=prec,
                     max_candidates=1 << 23)
    plane = _plane(plan, 10 * n_log2 + harm)
    found = [_check(capi, plan, plane, mean) for mean in (1.0, 0.6, 0.25)]
    assert 0 < found[0] <= found[1] <= found[2]
    # far from unit mean: every box is summed exactly
    _check(capi, plan, plane * 0.0, 1.0)
    plan.close()


@pytest.mark.parametrize("prec", [0, 1, 2])
def test_threshold_on_the_half_bin_plane(capi, prec):
    plan = capi.Plan(1 << 13, 64e-6, 20.0, 1.0, 2048, 8, precision=prec, interbin=True)
    plane = _plane(plan, 5)
    assert plane.shape[1] == 1 << 13
    for mean in (1.0, 0.5):
        assert _check(capi, plan, plane, mean) > 0
    plan.close()


@pytest.mark.parametrize("corr", [1, 2])
def test_a_search_with_many_crossings_and_a_short_series(capi, corr):
    """Bright series of both lengths on one plan: the same records as a plan
    whose threshold rule keeps the plain kernel, at equal thresholds."""
    import synthetic as S
    n = 1 << 15
    xs = []
    for m in (n, n // 2, n // 8):
        x = S.inject_sinusoid(S.white_noise(m, 3), 0.11 * m + 0.2, 3.0, 0.3)
        xs.append(torch.from_numpy(x).cuda())
    plan = capi.Plan(n, 64e-6, 24.0, 1.0, 2048, 16, precision=1, correlator=corr)
    st, c, nf = plan.search(xs, capacity=1 << 18)
    assert st == capi.FDAS_OK and nf == len(c) > 100
    # each series alone, through the stages
    for t, x in enumerate(xs):
        sub = capi.Plan(x.numel(), 64e-6, 24.0, 1.0, 2048, 16, precision=1, correlator=corr)
        plane, stats = sub.power_plane(sub.spectrum(x))
        st1, c1, n1 = sub.threshold(plane, stats, capacity=1 << 18)
        mine = c[c["trial_id"] == t]
        assert st1 == capi.FDAS_OK and n1 == len(mine)
        for k in ("harm", "iz", "ir", "power"):
            assert np.array_equal(mine[k], c1[k]), k
        mean = float(stats[0])
        assert _check(capi, sub, plane, mean) == n1
        sub.close()
    plan.close()


@pytest.mark.parametrize("prec", [0, 1, 2])
@pytest.mark.parametrize("harm", [2, 8, 16])
@pytest.mark.parametrize("z_max", [4.0, 96.0])   # 9 rows: the plain kernel; 193: by bounds
def test_cells_beside_nan_and_inf(capi, prec, harm, z_max):
    """NaN and +inf cells of a caller's plane beside bright ones: the sums that
    read them are not crossings or are infinite, those beside them (in the same
    boxes of 2 bins x 4 rows, and through the harmonics) keep their crossings."""
    plan = capi.Plan(1 << 14, 64e-6, z_max, 1.0, 2048, harm, precision=prec, max_candidates=1 << 22)
    plane = _plane(plan, 70 + harm)
    n_z, cols = plane.shape
    r = np.random.RandomState(harm)
    scale = 1.0 / 16.0 if prec == 2 else 1.0
    for k in range(60):
        z, c = r.randint(1, n_z - 1), r.randint(2, cols - 2)
        dz, dc = r.randint(-1, 2), r.randint(-1, 2)
        plane[z, c] = float(r.uniform(60.0, 300.0)) * scale
        if (dz, dc) != (0, 0):
            plane[z + dz, c + dc] = float("nan") if k % 4 else float("inf")
    assert torch.isnan(plane).any() and torch.isinf(plane).any()
    for mean in (1.0, 0.5):
        assert _check(capi, plan, plane, mean) > 60
    plan.close()


def _by_bounds(capi, plan):
    """Whether a search on the plan sums by bounds: by its launches of the harmonic
    group (2 plain, statistics included)."""
    plan.profile(False)
    plan.search([torch.randn(plan.info.n_samples, device="cuda")], capacity=1 << 16)
    return plan.profile()["harmonic"][0] > 2


@pytest.mark.parametrize("harm,z_step,sigma,by_bounds", [
    (16, 1.0, 5.3, False), (16, 1.0, 5.4, True), (16, 0.5, 5.4, True),
    (16, 2.0, 5.9, False), (16, 2.0, 6.0, True),
    (16, 4.0, 6.0, False), (16, 4.0, 6.5, False), (16, 4.0, 6.6, True),
    (16, 8.0, 7.1, False), (16, 8.0, 7.2, True), (16, 9.0, 8.0, False),
    (8, 1.0, 4.9, False), (8, 1.0, 5.0, True), (8, 2.0, 5.1, False), (8, 2.0, 5.125, True),
    (8, 8.0, 5.3, False), (8, 8.0, 5.375, True),
    (4, 8.0, 4.9, False), (4, 8.0, 5.0, True), (2, 4.0, 5.0, True), (1, 1.0, 6.0, False),
])
def test_thresholds_that_go_by_bounds(capi, harm, z_step, sigma, by_bounds):
    """Where noise alone would overflow the list of boxes the plain kernel is kept."""
    plan = capi.Plan(1 << 14, 64e-6, 16 * z_step, z_step, 2048, harm, threshold_sigma=sigma)
    assert _by_bounds(capi, plan) == by_bounds
    plan.close()


@pytest.mark.parametrize("prec,corr", [(0, 1), (1, 2), (2, 2)])
@pytest.mark.parametrize("z_step,sigma", [(0.5, 5.4), (1.0, 5.4), (2.0, 6.0), (4.0, 6.6), (8.0, 7.2)])
def test_coarse_and_fine_drift_steps_at_their_lowest_threshold(capi, prec, corr, z_step, sigma):
    """The plane of a pulse train, 16 harmonics: the crossings by bounds are the plain sums'."""
    n = 1 << 17
    plan = capi.Plan(n, 64e-6, 24 * z_step, z_step, 4096, 16, precision=prec, correlator=corr,
                     threshold_sigma=sigma)
    assert _by_bounds(capi, plan)
    u = np.arange(n) / n
    ph = 1700.3 * u + 2.0 * z_step * (u - 0.5) ** 2
    x = np.random.RandomState(4).randn(n) + 1.2 * ((ph - np.floor(ph)) < 0.05)
    plane, stats = plan.power_plane(plan.spectrum(torch.from_numpy(x.astype(np.float32)).cuda()))
    assert _check(capi, plan, plane, float(stats[0])) > 20
    plan.close()


@pytest.mark.parametrize("prec,harm,n_log2,rows,by_bounds", [
    (0, 16, 14, 13, False), (0, 16, 14, 15, True), (0, 16, 21, 13, True), (0, 8, 21, 13, False),
    (0, 8, 22, 13, True), (0, 2, 22, 13, False), (0, 2, 14, 15, True), (0, 16, 11, 27, False),
    (0, 16, 12, 27, True), (0, 16, 22, 11, False),
    (1, 16, 14, 13, False), (1, 16, 14, 15, True), (1, 8, 14, 15, False), (1, 8, 14, 17, True),
    (1, 8, 20, 23, False), (1, 8, 20, 25, True), (1, 8, 23, 17, True), (1, 4, 20, 95, False),
    (1, 4, 20, 97, True), (2, 2, 18, 193, False), (2, 2, 23, 23, False),
])
def test_sizes_that_go_by_bounds(capi, prec, harm, n_log2, rows, by_bounds):
    plan = capi.Plan(1 << n_log2, 64e-6, float(rows // 2), 1.0, 2048 if n_log2 > 11 else 1024, harm,
                     precision=prec)
    assert plan.info.n_z == rows
    assert _by_bounds(capi, plan) == by_bounds
    plan.close()


@pytest.mark.parametrize("prec", [1, 2])
@pytest.mark.parametrize("harm", [2, 4])
def test_few_harmonics_of_a_large_plane(capi, prec, harm):
    plan = capi.Plan(1 << 20, 64e-6, 48.0, 1.0, 2048, harm, precision=prec, threshold_sigma=5.0)
    assert _by_bounds(capi, plan)
    u = np.arange(1 << 20) / (1 << 20)
    ph = 17000.3 * u + 2.0 * (u - 0.5) ** 2
    x = np.random.RandomState(4).randn(1 << 20) + 0.4 * ((ph - np.floor(ph)) < 0.05)
    plane, stats = plan.power_plane(plan.spectrum(torch.from_numpy(x.astype(np.float32)).cuda()))
    assert _check(capi, plan, plane, float(stats[0])) > 20
    plan.close()


def _sparse_plane(plan, seed):
    """Cells below 0.5, whose sums cross nothing and list no box, and 8 bright ones,
    among them the corners: less than 300 boxes read one, so the list (4096 boxes at
    least) never overflows."""
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    shape = (plan.info.n_z, plan.info.plane_cols)
    p = 0.5 * torch.rand(shape, generator=g, device="cuda")
    r = np.random.RandomState(seed)
    for _ in range(4):
        p[r.randint(shape[0]), r.randint(shape[1])] = float(r.uniform(60.0, 300.0))
    p[0, 0] = p[-1, -1] = p[0, -1] = p[-1, 0] = 60.0
    return (p / 16.0 if plan.info.precision == 2 else p).to(plan.spec_dtype)


@pytest.mark.parametrize("prec", [0, 1, 2])
@pytest.mark.parametrize("harm", [8, 16])
@pytest.mark.parametrize("n_log2,rows,by_bounds", [(11, 27, False), (12, 25, True), (12, 27, True),
                                                   (13, 29, True), (14, 193, True)])
def test_a_few_bright_cells(capi, prec, harm, n_log2, rows, by_bounds):
    """By bounds and the exact sums alone, at the shortest rows (1024 columns are too
    few) and where the last block of rows and the last step of 8 blocks are partial;
    with every threshold out of FP16's range; and with every cell a crossing, which
    overflows the list of any plane of more than 4096 boxes."""
    plan = capi.Plan(1 << n_log2, 64e-6, float(rows // 2), 1.0, 2048 if n_log2 > 11 else 1024, harm,
                     precision=prec, max_candidates=1 << 23)
    assert plan.info.n_z == rows and _by_bounds(capi, plan) == by_bounds
    plane = _sparse_plane(plan, rows + harm)
    assert _check(capi, plan, plane, 1.0) >= 8
    for scale in (1e-3, 1e4):
        assert _check(capi, plan, plane * scale, scale) >= 8
    if n_log2 <= 13:
        full = torch.full_like(plane, 40.0 / (16.0 if prec == 2 else 1.0))
        assert _check(capi, plan, full, 1.0) == full.numel() * plan.info.n_stages
    plan.close()


@pytest.mark.parametrize("prec,corr,interbin", [(1, 2, False), (2, 2, False), (0, 3, False),
                                                (1, 2, True), (2, 2, True), (0, 1, True)])
def test_pooled_planes_of_the_correlation_and_of_the_plane(capi, prec, corr, interbin):
    """A search, whose pooled plane the tensor-core epilogue writes (with half bins the
    fix-up kernel too), against fdas_threshold on the same plane, which pools it by a
    kernel, and against the plain sums; a series of the plan's length and a half of it."""
    import synthetic as S
    n = 1 << 15
    make = lambda m: capi.Plan(m, 64e-6, 30.0, 1.0, 2048, 16, precision=prec, correlator=corr,
                               interbin=interbin)
    plan = make(n)
    assert _by_bounds(capi, plan)
    for m in (n, n // 2):
        # a tone half-way between two bins, the last one of its warp
        x = S.inject_sinusoid(S.white_noise(m, 7), 255.5 + 512 * (m // 2048), 2.0, 0.5)
        x = torch.from_numpy(x).cuda()
        st, found, nf = plan.search([x], capacity=1 << 18)
        assert st == capi.FDAS_OK and nf == len(found) > 100
        sub = make(m)
        plane, stats = sub.power_plane(sub.spectrum(x))
        st, staged, _ = sub.threshold(plane, stats, capacity=1 << 18)
        # (not sigma: the fix-up kernel sums the half bins' statistics by row blocks in a
        # search, by rows in a stage call, and their means differ by FP32 rounding)
        assert st == capi.FDAS_OK and len(found) == len(staged)
        for k in ("harm", "iz", "ir", "power"):
            assert np.array_equal(found[k], staged[k]), k
        assert _check(capi, sub, plane, float(stats[0])) == nf
        sub.close()
    plan.close()
