"""Edges of single kernels: sizes at which a split, a tile or a remainder can go wrong."""
import numpy as np
import pytest

import paper_2002_07858_gb300 as fc
import workloads

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    fc.load()
    c = fc.fc_create(0)
    yield c
    fc.fc_destroy(c)


def _grid(G, n, seed):
    """G spectra of n bins, an oscillation grid cut to length, and their fractional covariance."""
    side = int(np.ceil(np.sqrt(G)))
    S, F, _ = workloads.osc_2d(side, side, n, seed=seed)
    return np.ascontiguousarray(S[:G]), F


def _data(S, pts, U, seed):
    rng = np.random.default_rng(seed)
    return np.concatenate([rng.poisson(S[p], (U, S.shape[1])) for p in pts]).astype(np.float32), np.repeat(pts, U)


def _same_scan(ctx, gid, d, q, top_k):
    """The screened scan against the plain binary64 one: same minimum, chi2 to 1e-9 relative."""
    best, chi2 = fc.fc_scan(ctx, gid, d, q, fc.FC_PREC_MIXED, top_k)
    b64, c64 = fc.fc_scan(ctx, gid, d, q, fc.FC_PREC_FP64, top_k)
    assert np.array_equal(best, b64)
    np.testing.assert_allclose(chi2, c64, rtol=1e-9, atol=0)
    return best, chi2


# ---- screen split over the grid: few universe tiles, ranges of grid tiles --------------------

@pytest.mark.parametrize("top_k", [4, 8, 16])
@pytest.mark.parametrize("G,n,n_pts,U", [(257, 20, 1, 1), (256 * 7 + 1, 45, 1, 40), (256 * 40, 45, 3, 33),
                                         (256 * 131 + 5, 29, 40, 2), (256 * 30 + 255, 61, 2, 65),
                                         (256 * 30 + 1, 110, 5, 7)])
def test_split_screen(ctx, G, n, n_pts, U, top_k):
    S, F = _grid(G, n, 11)
    gid = fc.fc_load_grid(ctx, S)
    fc.fc_set_frac_cov(ctx, gid, F)
    pts = np.linspace(0, G - 1, n_pts).astype(np.int64)
    d, q = _data(S, pts, U, 5)
    for rnd in (fc.FC_ROUND_LIST, fc.FC_ROUND_TOPK):
        fc.fc_set_tuning(ctx, gid, first_round=rnd)
        _same_scan(ctx, gid, d, q, top_k)
    fc.fc_unload_grid(ctx, gid)


def test_split_screen_ties_take_the_lowest_index(ctx):
    """The grid repeated three times: every minimum is tied across ranges, and the first copy's index wins."""
    S, F = _grid(256 * 9 + 3, 33, 3)
    gid = fc.fc_load_grid(ctx, np.concatenate([S, S, S]))
    fc.fc_set_frac_cov(ctx, gid, F)
    pts = np.array([0, 1000, len(S) - 1])
    d, q = _data(S, pts, 20, 9)
    best, _ = _same_scan(ctx, gid, d, q + len(S), 16)
    assert best.max() < len(S)
    fc.fc_unload_grid(ctx, gid)


@pytest.mark.parametrize("n", [3, 15, 16, 17, 32, 45, 48, 50, 64, 67])
def test_one_point_matches_the_batch(ctx, n):
    """A universe's result has the same bits alone (a split screen, residuals spread over warps) and in a batch
    large enough to run unsplit with one thread per residual (N <= 64)."""
    S, F = _grid(256 * 20, n, 1)
    gid = fc.fc_load_grid(ctx, S)
    fc.fc_set_frac_cov(ctx, gid, F)
    ps = np.arange(0, len(S), 3, dtype=np.int64)
    d, b, ns = fc.fc_run_points(ctx, gid, ps, 7, 96)
    for k in (0, 500, len(ps) - 1):
        d1, b1, n1 = fc.fc_run_points(ctx, gid, ps[k:k + 1], 7, 96)
        assert np.array_equal(d[k], d1[0]) and np.array_equal(b[k], b1[0]) and np.array_equal(ns[k], n1[0])
    fc.fc_unload_grid(ctx, gid)


# ---- quantiles: selection, and the sort behind it --------------------------------------------

def _quantile_rows(kind, rows, n, rng):
    if kind == "chi2":
        x = rng.chisquare(2, (rows, n))
        return np.where(x < 0.2, 0.0, x)
    if kind == "normal":
        return rng.standard_normal((rows, n))
    if kind == "ties":  # few distinct values: crowded buckets
        return rng.integers(0, 3, (rows, n)).astype(np.float64)
    if kind == "equal":
        return np.full((rows, n), 1.25)
    if kind == "outlier":  # everything but one value in one bucket
        x = rng.random((rows, n))
        x[:, n // 2] = 1e30
        return x
    if kind == "huge":  # beyond binary32
        return rng.standard_normal((rows, n)) * 1e300
    x = rng.chisquare(2, (rows, n))
    x[:, ::7] = np.inf
    x[0, 0] = -np.inf
    return x


@pytest.mark.parametrize("kind", ["chi2", "normal", "ties", "equal", "outlier", "huge", "inf"])
@pytest.mark.parametrize("n", [1, 2, 31, 129, 1000, 2048, 2049, 16384])
@pytest.mark.parametrize("nq", [1, 3, 8, 9])
def test_quantiles(ctx, kind, n, nq):
    import torch

    x = _quantile_rows(kind, 3, n, np.random.default_rng(n * 10 + nq))
    probs = np.linspace(0.0, 1.0, nq) if nq > 1 else np.array([0.9])
    with np.errstate(invalid="ignore"):
        s = np.sort(x, axis=1)
        h = (n - 1) * probs
        lo = np.floor(h).astype(int)
        a, b = s[:, lo], s[:, np.minimum(lo + 1, n - 1)]
        want = a + (h - lo) * (b - a)  # the rule itself: numpy's own function rounds its blend differently
    # a blend of two values: a few roundings of the larger one
    np.testing.assert_allclose(fc.fc_quantiles(ctx, x, probs), want, rtol=0, atol=4e-16 * np.max(np.abs(
        np.where(np.isfinite(x), x, 0.0))))
    dev = torch.from_numpy(x).cuda()
    torch.cuda.synchronize()
    assert np.array_equal(fc.fc_quantiles(ctx, dev, probs), fc.fc_quantiles(ctx, x, probs), equal_nan=True)


def test_quantiles_with_nan_sorts_it_last(ctx):
    x = np.random.default_rng(0).random((2, 100))
    x[1, 5] = np.nan
    q = fc.fc_quantiles(ctx, x, np.array([0.0, 0.5, 1.0]))
    assert np.isfinite(q[0]).all() and np.isfinite(q[1, :2]).all() and np.isnan(q[1, 2])


# ---- tensor-core q-vectors: triangular steps, slots interleaved in 16-row blocks -------------

@pytest.mark.parametrize("n", [5, 13, 14, 29, 45, 61, 77, 93, 109, 125, 141, 157, 173, 189, 200])
@pytest.mark.parametrize("n_pts", [1, 2, 7])
def test_qvec_groups(ctx, n, n_pts):
    """Every K, with whole and partial slot groups: the scan equals the plain one, and needs no fallback."""
    S, F = _grid(700, n, 2)
    gid = fc.fc_load_grid(ctx, S)
    fc.fc_set_frac_cov(ctx, gid, F)
    pts = np.linspace(3, 690, n_pts).astype(np.int64)
    d, q = _data(S, pts, 12, n)
    _same_scan(ctx, gid, d, q, 8)
    tc = fc.fc_run_points(ctx, gid, pts, 3, 20)
    assert fc.fc_get_stats(ctx)["fallback"] == 0
    fc.fc_set_tuning(ctx, gid, qvec=fc.FC_QVEC_SIMT)
    simt = fc.fc_run_points(ctx, gid, pts, 3, 20)
    assert all(np.array_equal(a, b) for a, b in zip(tc, simt))
    fc.fc_unload_grid(ctx, gid)


# ---- fake data: blocks of 64 universes, 8 rows of L, queued draws -----------------------------

@pytest.mark.parametrize("nf,collapse", [(1, False), (3, True), (7, False), (8, False), (9, True), (33, True),
                                         (90, True), (200, False)])
@pytest.mark.parametrize("U", [1, 63, 64, 65, 130])
def test_fake_data_blocks(ctx, nf, collapse, U):
    """Bit for bit against the oracle, with bins from nearly empty (inversion) to crowded (rejection)."""
    import oracle

    S, F = _grid(12, nf, nf)
    S = S * np.logspace(-2.5, 0.5, nf)[None, ::-1]
    coll = workloads.pair_collapse(nf) if collapse else None
    n_fit = (nf + 1) // 2 if collapse else nf
    ps = np.array([0, 11, 5], np.int64)
    gid = fc.fc_load_grid(ctx, S, coll, n_fit)
    fc.fc_set_frac_cov(ctx, gid, F)
    for fluct in (fc.FC_FLUCT_POISSON_SYS, fc.FC_FLUCT_GAUSS):
        got = fc.fc_fake_data(ctx, gid, ps, 17, U, n_fit, fluct)
        want = oracle.fake_data(S, F, ps, 17, U, coll, n_fit, fluct)
        assert np.array_equal(got, want)
    fc.fc_unload_grid(ctx, gid)


# ---- systematic factor: panels of 8 columns, one CTA or a cluster of 8 a point ----------------

@pytest.mark.parametrize("nf", [1, 7, 8, 9, 16, 17, 24, 63, 90, 155, 156, 200])
def test_systematic_factor(ctx, nf):
    """Bit for bit the oracle's, for a lone point (a cluster) and through the fake data of many (a CTA each)."""
    import oracle

    S, F = _grid(40, nf, nf + 3)
    gid = fc.fc_load_grid(ctx, S)
    fc.fc_set_frac_cov(ctx, gid, F)
    for q in (0, 39):
        assert np.array_equal(fc.fc_covariance(ctx, gid, q, nf, nf, want_A=False)[1], oracle.chol_sys(S[q], F))
    ps = np.arange(40, dtype=np.int64)
    many = fc.fc_fake_data(ctx, gid, ps, 5, 3, nf)
    for k in (0, 20, 39):
        assert np.array_equal(fc.fc_fake_data(ctx, gid, ps[k:k + 1], 5, 3, nf)[0], many[k])
    assert np.array_equal(many, oracle.fake_data(S, F, ps, 5, 3))
    fc.fc_unload_grid(ctx, gid)


# ---- list rounds: long lists ------------------------------------------------------------------

@pytest.mark.parametrize("n", [7, 33, 62, 77, 120, 199])
def test_crowded_lists(ctx, n):
    """Thousands of nearly equal spectra along one direction: long lists, the plain path's minimum, and ties
    (every spectrum twice) to the lowest index."""
    rng = np.random.default_rng(n)
    b, f = rng.uniform(50.0, 500.0, n), rng.uniform(5.0, 50.0, n)
    amp = np.concatenate([np.logspace(-5, 0, 3000), np.linspace(0.0, 1.0, 2001)])
    S = b + amp[:, None] * np.sin(np.linspace(0.1, 9.0, n))[None, :] ** 2 * f
    S = np.repeat(S, 2, axis=0)
    _, F = _grid(4, n, n)
    gid = fc.fc_load_grid(ctx, S)
    fc.fc_set_frac_cov(ctx, gid, F)
    pts = np.array([0, 5000, 9000], np.int64)
    d, q = _data(S, pts, 30, 1)
    chi2 = {}
    for prec in (fc.FC_PREC_MIXED, fc.FC_PREC_FP64):
        chi2[prec] = fc.fc_scan(ctx, gid, d, q, prec, 8)
    best, c = chi2[fc.FC_PREC_MIXED]
    b64, c64 = chi2[fc.FC_PREC_FP64]
    np.testing.assert_allclose(c, c64, rtol=1e-9)
    assert (best % 2 == 0).all()
    # neighbours closer than the two paths' own rounding may change places
    differ = best != b64
    assert np.all(np.abs(best - b64)[differ] <= 4) and differ.mean() < 0.2
    fc.fc_unload_grid(ctx, gid)


# ---- host lists on their way to the device ----------------------------------------------------

def test_long_host_lists(ctx):
    """A list longer than the staging block, and lists that fill it up between two waits: every point of a grid
    as a true point, against the same points alone."""
    S, F = _grid(192 * 192, 2, 8)
    gid = fc.fc_load_grid(ctx, S)
    fc.fc_set_frac_cov(ctx, gid, F)
    opts = dict(precision=fc.FC_PREC_FP64, cov=fc.FC_COV_FIXED)
    ps = np.arange(len(S), dtype=np.int64)[::-1].copy()
    d, b, ns = fc.fc_run_points(ctx, gid, ps, 3, 1, opts=opts)
    for k in (0, 1, 20000, len(ps) - 1):
        d1, b1, n1 = fc.fc_run_points(ctx, gid, ps[k:k + 1], 3, 1, opts=opts)
        assert np.array_equal(d[k], d1[0]) and np.array_equal(b[k], b1[0]) and np.array_equal(ns[k], n1[0])
    fc.fc_unload_grid(ctx, gid)


# ---- several threads on one device ------------------------------------------------------------

def test_threads_of_different_sizes():
    """Contexts of two threads whose launches need different shared memory: neither's limit cuts the other's."""
    import threading

    S1, F1 = _grid(30, 200, 1)
    S2, F2 = _grid(30, 90, 2)
    errors, out = [], {}

    def work(key, S, F, reps):
        try:
            n = S.shape[1]
            c = fc.fc_create(0)
            gid = fc.fc_load_grid(c, S)
            fc.fc_set_frac_cov(c, gid, F)
            ps = np.arange(20, dtype=np.int64)  # a CTA a point
            x = np.random.default_rng(n).random((4, 16384 if n == 200 else 5000))
            got = []
            for _ in range(reps):
                A, L = fc.fc_covariance(c, gid, 3, n, n)
                fc.fc_set_frac_cov(c, gid, F)  # the next covariance is built again
                got.append((A, L, fc.fc_fake_data(c, gid, ps, 5, 3, n), *fc.fc_run_points(c, gid, ps[:2], 5, 9),
                            fc.fc_quantiles(c, x, np.array([0.1, 0.9]))))
            out[key] = got
            fc.fc_destroy(c)
        except Exception as e:  # the launch that finds the limit too low is an error of the call
            errors.append(e)

    threads = [threading.Thread(target=work, args=a) for a in ((200, S1, F1, 150), (90, S2, F2, 300))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors[0]
    for got in out.values():
        for g in got[1:]:
            assert all(np.array_equal(a, b) for a, b in zip(g, got[0]))


@pytest.mark.parametrize("n", [5, 100, 3000])
@pytest.mark.parametrize("nq", [3, 9])
def test_quantiles_sort_every_nan_last(ctx, n, nq):
    """NaN of both signs behind the row's numbers and infinities, as numpy sorts them."""
    x = np.random.default_rng(n).standard_normal((4, n))
    x[1, 0], x[2, n - 1], x[3, 0], x[3, 3] = -np.nan, np.nan, -np.nan, np.nan
    assert np.signbit(x[1, 0]) and not np.signbit(x[2, n - 1])
    x[3, 1], x[3, 2] = -np.inf, np.inf
    probs = np.linspace(0.0, 1.0, nq)
    s, h = np.sort(x, axis=1), (n - 1) * probs
    lo = np.floor(h).astype(int)
    with np.errstate(invalid="ignore"):
        a, b = s[:, lo], s[:, np.minimum(lo + 1, n - 1)]
        want = a + (h - lo) * (b - a)
    # two orders of the blend's three roundings differ by at most 10 half-ulps of the row's largest number
    np.testing.assert_allclose(fc.fc_quantiles(ctx, x, probs), want, rtol=0,
                               atol=1.2e-15 * np.max(np.abs(x), where=np.isfinite(x), initial=0.0))


# ---- systematic factor: the form for many points, and the lines between the three -------------

@pytest.mark.parametrize("nf", [1, 20, 39, 40, 63, 64, 90, 155, 156, 200])
@pytest.mark.parametrize("P", [28, 29, 152, 153, 330])
def test_systematic_factor_forms(ctx, nf, P):
    """Bit for bit the oracle's fake data on both sides of every line, in both fluctuation modes."""
    import oracle

    S, F = _grid(330, nf, nf + 1)
    gid = fc.fc_load_grid(ctx, S)
    fc.fc_set_frac_cov(ctx, gid, F)
    ps = np.arange(P, dtype=np.int64)[::-1].copy()
    for fluct in (fc.FC_FLUCT_POISSON_SYS, fc.FC_FLUCT_GAUSS):
        got = fc.fc_fake_data(ctx, gid, ps, 5, 2, nf, fluct)
        assert np.array_equal(got, oracle.fake_data(S, F, ps, 5, 2, None, nf, fluct))
    fc.fc_unload_grid(ctx, gid)


# ---- covariances: 256 and 512 threads ---------------------------------------------------------

@pytest.mark.parametrize("n", [1, 2, 40, 112, 113])
def test_covariance_thread_counts(ctx, n):
    """A covariance has the same bits alone (512 threads) and among many (256 up to N = 112)."""
    S, F = _grid(1000, n, n)
    gid = fc.fc_load_grid(ctx, S)
    ps = np.arange(len(S), dtype=np.int64)
    many, alone = [], []
    fc.fc_set_frac_cov(ctx, gid, F)
    fc.fc_run_points(ctx, gid, ps, 1, 1, opts=dict(cov=fc.FC_COV_FIXED))
    for q in (0, 500, 999):
        many.append(fc.fc_covariance(ctx, gid, q, n, n, want_L=False)[0])
    fc.fc_set_frac_cov(ctx, gid, F)
    for q in (0, 500, 999):
        alone.append(fc.fc_covariance(ctx, gid, q, n, n, want_L=False)[0])
    for q, a, b in zip((0, 500, 999), many, alone):
        assert np.array_equal(a, b)
        M = S[q][:, None] * F * S[q][None, :] + np.diag(S[q])
        # n multiply-adds a factor, inverse and product element, scaled by the condition number
        tol = 3 * n * 2.0 ** -52 * np.linalg.cond(M) * np.abs(np.linalg.inv(M)).max()
        np.testing.assert_allclose(a, np.linalg.inv(M), rtol=0, atol=tol)
    fc.fc_unload_grid(ctx, gid)


@pytest.mark.parametrize("kind", ["chi2", "ties", "equal", "outlier", "inf"])
@pytest.mark.parametrize("n", [1, 2, 33, 100, 129, 1000, 2048])
@pytest.mark.parametrize("nq", [1, 8])
def test_quantiles_of_many_rows(ctx, kind, n, nq):
    """More rows than SMs (the small CTA): every row as alone (the wide one)."""
    x = _quantile_rows(kind, 200, n, np.random.default_rng(n + nq))
    probs = np.linspace(0.03, 1.0, nq)
    got = fc.fc_quantiles(ctx, x, probs)
    for r in (0, 1, 77, 199):
        assert np.array_equal(got[r:r + 1], fc.fc_quantiles(ctx, x[r:r + 1], probs), equal_nan=True)
    with np.errstate(invalid="ignore"):
        s, h = np.sort(x, axis=1), (n - 1) * probs
        lo = np.floor(h).astype(int)
        a, b = s[:, lo], s[:, np.minimum(lo + 1, n - 1)]
        want = a + (h - lo) * (b - a)
    np.testing.assert_allclose(got, want, rtol=0, atol=1.2e-15 * np.max(np.abs(x), where=np.isfinite(x), initial=0.0))


# ---- fake data: a thread, or a CTA of 128 or 256 threads, per 64 universes --------------------

@pytest.mark.parametrize("nf", [1, 2, 3, 4, 7, 8, 9, 16, 31, 52, 53])
@pytest.mark.parametrize("P,U", [(3, 1), (3, 33), (700, 2), (1300, 1), (1300, 65), (20, 4000)])
def test_fake_data_forms(ctx, nf, P, U):
    """Both sides of every line, with and without a collapse, in both modes: the oracle's bits for some of the
    points, and the same bits for a point alone."""
    import oracle

    S, F = _grid(1300, nf, nf + 2)
    S = S * np.logspace(-2.5, 0.5, nf)[None, ::-1]
    coll = workloads.pair_collapse(nf)
    ps = np.arange(P, dtype=np.int64)
    some = [0, P // 2, P - 1]
    for c, n_fit in ((None, nf), (coll, (nf + 1) // 2)):
        gid = fc.fc_load_grid(ctx, S, c, n_fit)
        fc.fc_set_frac_cov(ctx, gid, F)
        for fluct in (fc.FC_FLUCT_POISSON_SYS, fc.FC_FLUCT_GAUSS):
            got = fc.fc_fake_data(ctx, gid, ps, 23, U, n_fit, fluct)
            assert np.array_equal(got[some], oracle.fake_data(S, F, ps[some], 23, U, c, n_fit, fluct))
            assert np.array_equal(got[P - 1:], fc.fc_fake_data(ctx, gid, ps[P - 1:], 23, U, n_fit, fluct))
        fc.fc_unload_grid(ctx, gid)
