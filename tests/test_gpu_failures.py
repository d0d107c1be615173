"""Calls that fail, what they leave behind, and data that has no minimum."""
import time

import numpy as np
import pytest

import paper_2002_07858_gb300 as fc
import workloads

pytestmark = pytest.mark.gpu

PRECISIONS = [fc.FC_PREC_FP64, fc.FC_PREC_MIXED]


@pytest.fixture()
def ctx():
    fc.load()
    c = fc.fc_create(0)
    yield c
    fc.fc_destroy(c)


@pytest.fixture(scope="module")
def grid():
    S, F, _ = workloads.osc_2d(20, 20, 40, seed=4)
    return S, F


def _indefinite(F):
    """Symmetric and finite, but diag(s) F diag(s) (+ diag(s)) has a negative diagonal entry for s > 1."""
    bad = F.copy()
    bad[7, 7] = -1.0
    return bad


def _not_spd(call):
    with pytest.raises(fc.FCError) as e:
        call()
    assert e.value.status == fc.FC_ERR_NOT_SPD


# ---- covariances that are not positive definite ---------------------------------------------

CALLS = {
    "scan": lambda c, g, d, prec: fc.fc_scan(c, g, d, np.arange(len(d)), prec, 8),
    "data": lambda c, g, d, prec: fc.fc_data_dchi2(c, g, d[0], np.array([3, 9]), opts=dict(precision=prec)),
    "data_fixed": lambda c, g, d, prec: fc.fc_data_dchi2(c, g, d[0], np.array([3]), opts=dict(precision=prec,
                                                                                           cov=fc.FC_COV_FIXED)),
    "points": lambda c, g, d, prec: fc.fc_run_points(c, g, np.array([5, 300]), 1, 30, opts=dict(precision=prec)),
    "points_identity": lambda c, g, d, prec: fc.fc_run_points(c, g, np.array([5, 300]), 1, 30, opts=dict(
        precision=prec, cov=fc.FC_COV_IDENTITY)),
    "points_gauss_identity": lambda c, g, d, prec: fc.fc_run_points(c, g, np.array([5]), 1, 30, opts=dict(
        precision=prec, cov=fc.FC_COV_IDENTITY, fluct=fc.FC_FLUCT_GAUSS)),
}


@pytest.mark.parametrize("prec", PRECISIONS)
@pytest.mark.parametrize("name", list(CALLS))
def test_not_spd_is_reported_and_the_context_goes_on(ctx, grid, name, prec):
    S, F = grid
    d = np.random.default_rng(0).poisson(S[:24]).astype(np.float32)
    gid = fc.fc_load_grid(ctx, S)
    fc.fc_set_frac_cov(ctx, gid, F)
    ref = CALLS[name](ctx, gid, d, prec)
    fc.fc_set_frac_cov(ctx, gid, _indefinite(F))
    _not_spd(lambda: CALLS[name](ctx, gid, d, prec))
    fc.fc_set_frac_cov(ctx, gid, F)
    for a, b in zip(CALLS[name](ctx, gid, d, prec), ref):
        assert np.array_equal(a, b)


def test_not_spd_covariance_and_factor(ctx, grid):
    S, F = grid
    gid = fc.fc_load_grid(ctx, S)
    fc.fc_set_frac_cov(ctx, gid, _indefinite(F))
    _not_spd(lambda: fc.fc_covariance(ctx, gid, 5, 40, 40, want_L=False))
    _not_spd(lambda: fc.fc_covariance(ctx, gid, 5, 40, 40, want_A=False))
    _not_spd(lambda: fc.fc_fake_data(ctx, gid, np.array([5]), 1, 3, 40))


# ---- data without a minimum -----------------------------------------------------------------

@pytest.mark.parametrize("prec", PRECISIONS)
@pytest.mark.parametrize("G", [1, 400, 3 * 256 + 1])
def test_universe_without_a_minimum(ctx, prec, G):
    """NaN data: best -1 and chi2 NaN for that universe alone, the others as without it."""
    S, F, _ = workloads.osc_2d(28, 28, 40, seed=4)
    S = np.ascontiguousarray(S[:G])
    gid = fc.fc_load_grid(ctx, S)
    fc.fc_set_frac_cov(ctx, gid, F)
    d = np.random.default_rng(1).poisson(S[np.arange(70) % G]).astype(np.float32)
    q = np.arange(70) % G
    best, chi2 = fc.fc_scan(ctx, gid, d, q, prec, 8)
    bad = d.copy()
    bad[[0, 33], [2, 39]] = np.nan
    b, c = fc.fc_scan(ctx, gid, bad, q, prec, 8)
    none = np.zeros(70, bool)
    none[[0, 33]] = True
    assert np.array_equal(b[~none], best[~none]) and np.array_equal(c[~none], chi2[~none])
    assert (b[none] == -1).all() and np.isnan(c[none]).all()


# ---- a screen whose waits run out ------------------------------------------------------------

@pytest.mark.parametrize("stop_after", [0, 1, 3])
@pytest.mark.parametrize("G,n,P,U", [(400, 40, 1, 24576),      # tiles for every SM: one thread per residual
                                     (400, 16, 200, 128),      # the same with a covariance per tile
                                     (256 * 40, 20, 2, 33)])   # few tiles: the grid split over the SMs
def test_screen_timeout_leaves_no_items(ctx, G, n, P, U, stop_after):
    """After an aborted screen nothing is rescored from what an earlier launch left behind, and the context goes on."""
    side = int(np.ceil(np.sqrt(G)))
    S, F, _ = workloads.osc_2d(side, side, n, seed=6)
    gid = fc.fc_load_grid(ctx, S[:G])
    fc.fc_set_frac_cov(ctx, gid, F)
    ps = np.linspace(0, G - 1, P).astype(np.int64)
    ref = fc.fc_run_points(ctx, gid, ps, 2, U)
    fc.fc_set_wait_test(ctx, 150_000_000, stop_after)
    with pytest.raises(fc.FCError) as e:
        fc.fc_run_points(ctx, gid, ps, 3, U)
    assert e.value.status == fc.FC_ERR_TIMEOUT
    fc.fc_set_wait_test(ctx, 0, -1)
    for a, b in zip(fc.fc_run_points(ctx, gid, ps, 2, U), ref):
        assert np.array_equal(a, b)


# ---- a failed covariance is not kept ---------------------------------------------------------

@pytest.mark.parametrize("prec", PRECISIONS)
@pytest.mark.parametrize("slots", [0, 4])
def test_failed_covariance_fails_again(ctx, grid, prec, slots):
    """One spectrum with an empty bin: its covariance fails on every call, and the others keep their results."""
    S, F = grid
    S = S.copy()
    S[17, 3] = 0.0
    gid = fc.fc_load_grid(ctx, S)
    fc.fc_set_frac_cov(ctx, gid, F)
    fc.fc_set_tuning(ctx, gid, cache_slots=slots)
    d = np.random.default_rng(2).poisson(S[:12] + 1.0).astype(np.float32)
    good, bad = np.array([0, 1, 2] * 4), np.array([0, 1, 17] * 4)
    ref = fc.fc_scan(ctx, gid, d, good, prec, 8)
    A, _ = fc.fc_covariance(ctx, gid, 2, 40, 40, want_L=False)
    for _ in range(3):
        _not_spd(lambda: fc.fc_scan(ctx, gid, d, bad, prec, 8))
        _not_spd(lambda: fc.fc_covariance(ctx, gid, 17, 40, 40, want_L=False))
        for a, b in zip(fc.fc_scan(ctx, gid, d, good, prec, 8), ref):
            assert np.array_equal(a, b)
        assert np.array_equal(fc.fc_covariance(ctx, gid, 2, 40, 40, want_L=False)[0], A)


def test_served_job_fails_alone(ctx, grid):
    """A job that starts at such a spectrum fails; the jobs around it on another grid give their results."""
    S, F = grid
    bad = S.copy()
    bad[17, 3] = 0.0
    g1, g2 = fc.fc_load_grid(ctx, S), fc.fc_load_grid(ctx, bad)
    for g in (g1, g2):
        fc.fc_set_frac_cov(ctx, g, F)
    ref = fc.fc_run_points(ctx, g1, np.array([5, 6]), 3, 50)
    jobs = [fc.fc_submit(ctx, g, np.array([p, 6]), 3, 50, want_bestfit=True, want_nscans=True)
            for g, p in ((g1, 5), (g2, 17), (g1, 5))]
    status = {}
    end = time.time() + 60
    while len(status) < 3 and time.time() < end:
        for t, _ in jobs:
            if t in status:
                continue
            try:
                st, _ = fc.fc_poll(ctx, t)
            except fc.FCError as e:
                st = e.status
            if st != fc.FC_PENDING:
                status[t] = st
        time.sleep(0.001)
    assert [status[t] for t, _ in jobs] == [fc.FC_OK, fc.FC_ERR_NOT_SPD, fc.FC_OK]
    for k in (0, 2):
        for a, b in zip(jobs[k][1], ref):
            assert np.array_equal(np.asarray(a).ravel(), np.asarray(b).ravel())


# ---- tight budgets ---------------------------------------------------------------------------

@pytest.mark.parametrize("side,n,P,U,prec,budget", [
    (100, 20, 2, 64, fc.FC_PREC_MIXED, 18_800_000),      # no room for the split screen's lists
    (100, 20, 2, 20000, fc.FC_PREC_MIXED, 45_500_000),   # nor for the small chunks of a list round
    (60, 45, 40, 500, fc.FC_PREC_MIXED, 46_600_000),
    (60, 45, 40, 500, fc.FC_PREC_FP64, 17_800_000),
    (30, 100, 10, 2000, fc.FC_PREC_MIXED, 51_200_000),
])
def test_storage_that_only_saves_time_gives_way(side, n, P, U, prec, budget):
    """Budgets that these fits, the first of a context, have always fitted in: what they take beyond the least is
    given up, with the same results."""
    fc.load()
    S, F, _ = workloads.osc_2d(side, side, n, seed=1)
    ps = np.linspace(0, len(S) - 1, P).astype(np.int64)
    out = []
    for b in (0, budget):
        c = fc.fc_create(0, b)
        try:
            gid = fc.fc_load_grid(c, S)
            fc.fc_set_frac_cov(c, gid, F)
            out.append(fc.fc_run_points(c, gid, ps, 4, U, opts=dict(precision=prec)))
            assert not b or fc.fc_get_stats(c)["device_bytes"] <= b
        finally:
            fc.fc_destroy(c)
    assert all(np.array_equal(x, y) for x, y in zip(*out))


@pytest.mark.parametrize("n", [40, 170])
@pytest.mark.parametrize("P", [1, 100, 400])
def test_not_spd_factor_in_every_form(ctx, n, P):
    S, F, _ = workloads.osc_2d(20, 20, n, seed=4)
    gid = fc.fc_load_grid(ctx, S)
    fc.fc_set_frac_cov(ctx, gid, _indefinite(F))
    _not_spd(lambda: fc.fc_fake_data(ctx, gid, np.arange(P), 1, 2, n))
