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
