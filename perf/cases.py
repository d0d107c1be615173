"""Performance cases of the Feldman-Cousins library: what users call, over the sizes they call it at.

Inputs follow the shape models of the repository's workloads (sizes, parameter ranges, number of bins, universes per
point), with every random number taken from the case's seed.  Grids are built on the GPU; handles, loaded grids and
output buffers are what a program keeps between calls.
"""
import math
import time

import numpy as np
import torch

import paper_2002_07858_gb300 as fc

BUDGET = 80 << 30  # device-memory budget of every context: the serving configuration's
DEV = "cuda"


def listed():
    return [
        # one true point on the 25x25 grid: the smallest fit, where launches and waits count
        {"name": "point_25x25", "kind": "fit", "model": "osc2", "n": 25, "bins": 40, "pairs": False, "P": 1, "U": 1000,
         "new_F": False, "precision": 1, "top_k": 8},
        # the same point on the plain binary64 path
        {"name": "point_25x25_fp64", "kind": "fit", "model": "osc2", "n": 25, "bins": 40, "pairs": False, "P": 1,
         "U": 1000, "new_F": False, "precision": 0, "top_k": 8},
        # the full Feldman-Cousins job of the 100x100 grid, every point a true point, bins collapsed in pairs, with a
        # new fractional covariance each time (the job is run once per covariance)
        {"name": "full_100x100", "kind": "fit", "model": "osc2", "n": 100, "bins": 90, "pairs": True, "P": 10000,
         "U": 1000, "new_F": True, "precision": 1, "top_k": 8},
        # some true points of the three-parameter 64^3 grid: nearly every universe refits its own covariance
        {"name": "points_64cubed", "kind": "fit", "model": "app3", "n": 64, "bins": 120, "pairs": False, "P": 128,
         "U": 500, "new_F": True, "precision": 1, "top_k": 8},
        # a six-parameter grid of 16.7 million points kept as its shape model, top-16
        {"name": "points_16pow6", "kind": "fit", "model": "terms6", "n": 16, "bins": 64, "pairs": False, "P": 4, "U": 16,
         "new_F": True, "precision": 1, "top_k": 16},
        # the widest spectra the library takes (200 bins)
        {"name": "points_n200", "kind": "fit", "model": "app3", "n": 27, "bins": 200, "pairs": False, "P": 4, "U": 500,
         "new_F": True, "precision": 1, "top_k": 8},
        # one scan of a user's own pseudo-data under given covariances
        {"name": "scan_141x141", "kind": "scan", "model": "osc2", "n": 141, "bins": 90, "pairs": True, "P": 64,
         "U": 64, "precision": 1, "top_k": 8},
        # the observed data's statistic at every grid point (its covariances stay resident)
        {"name": "data_100x100", "kind": "data", "model": "osc2", "n": 100, "bins": 90, "pairs": True, "P": 10000,
         "precision": 1, "top_k": 8},
        # fake data alone
        {"name": "fake_500x1000", "kind": "fake", "model": "osc2", "n": 100, "bins": 90, "pairs": True, "P": 500,
         "U": 1000},
        # critical values of the full job
        {"name": "quantiles_10000x1000", "kind": "quantiles", "rows": 10000, "n": 1000},
        # a handful of jobs of different grids, bins and universes in flight at once
        {"name": "serve_12_jobs", "kind": "serve", "n2": 50, "bins2": 64, "n3": 20, "bins3": 90, "n4": 12, "bins4": 150,
         "jobs": 12},
        # a new grid from host memory: load it, set the covariance, look at one, scan a few data sets, unload
        {"name": "new_grid_71x71", "kind": "load", "model": "osc2", "n": 71, "bins": 90, "pairs": True, "P": 8, "U": 16},
    ]


def _logint(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["fit2", "fit2", "fit3", "fit6", "fp64", "scan", "data", "fake", "quantiles", "serve", "load"])
    if kind == "quantiles":
        n = _logint(rng, 100, 16384)
        return {"kind": "quantiles", "rows": _logint(rng, 100, min(20000, 20_000_000 // n)), "n": n}
    if kind == "serve":
        return {"kind": "serve", "n2": rng.randint(25, 70), "bins2": rng.randint(40, 90), "n3": rng.randint(10, 24),
                "bins3": rng.randint(60, 120), "n4": rng.randint(6, 12), "bins4": rng.randint(100, 180),
                "jobs": rng.randint(4, 14)}
    if kind == "fit3":
        while True:
            c = {"kind": "fit", "model": "app3", "n": rng.randint(10, 64), "bins": rng.randint(60, 200), "pairs": False,
                 "P": _logint(rng, 2, 128), "U": _logint(rng, 50, 500), "new_F": True, "precision": 1,
                 "top_k": rng.choice([8, 16])}
            if c["P"] * c["U"] * c["n"] ** 3 * c["bins"] ** 2 <= 64 * 500 * 64 ** 3 * 120 ** 2:
                return c
    if kind == "fit6":
        return {"kind": "fit", "model": "terms6", "n": rng.randint(6, 14), "bins": rng.randint(41, 72), "pairs": False,
                "P": rng.randint(1, 5), "U": rng.randint(8, 16), "new_F": True, "precision": 1, "top_k": 16}
    bins = rng.randint(40, 120)
    c = {"kind": "fit", "model": "osc2", "n": rng.randint(25, 100), "bins": bins, "pairs": rng.random() < 0.5}
    if kind == "fit2":
        c.update(P=_logint(rng, 1, 600), U=_logint(rng, 100, 1500), new_F=rng.random() < 0.5, precision=1,
                 top_k=rng.choice([4, 8, 16]))
        c["P"] = min(c["P"], c["n"] ** 2)
    elif kind == "fp64":
        c.update(P=rng.randint(1, 3), U=_logint(rng, 100, 1000), new_F=rng.random() < 0.5, precision=0, top_k=8)
    elif kind == "scan":
        c.update(kind="scan", n=rng.randint(25, 180), P=rng.randint(1, 100), U=_logint(rng, 4, 100),
                 precision=1, top_k=rng.choice([4, 8, 16]))
    elif kind == "data":
        c.update(kind="data", precision=1, top_k=8)
        c["P"] = c["n"] ** 2
    elif kind == "fake":
        c.update(kind="fake", P=_logint(rng, 1, 500), U=_logint(rng, 100, 1000))
        c["P"] = min(c["P"], c["n"] ** 2)
    else:
        c.update(kind="load", P=rng.randint(1, 16), U=rng.randint(4, 32))
    return c


# ---------------------------------------------------------------- inputs --

class Model:
    """Spectra of one grid and their fractional covariance, from a seed."""

    def __init__(self, model, n, bins, pairs, seed):
        rng = np.random.default_rng(seed)
        self.model, self.n, self.bins = model, n, bins
        b = rng.uniform(50.0, 500.0, bins)
        T = {"osc2": 1, "app3": 1, "terms4": 2, "terms6": 3}[model]
        f = rng.uniform(5.0, 50.0, (T, bins))
        L = rng.choice(np.array([110.0, 470.0, 600.0]), bins)
        E = np.linspace(0.2, 3.0, bins)
        sig = rng.uniform(0.05, 0.2, bins)
        W = rng.standard_normal((bins, 5))
        W /= np.linalg.norm(W, axis=1, keepdims=True)
        F = sig[:, None] * (W @ W.T + 0.2 * np.eye(bins)) * sig[None, :]
        self.F = np.ascontiguousarray(0.5 * (F + F.T))
        self.collapse = (np.arange(bins) // 2).astype(np.int32) if pairs else None
        self.n_fit = (bins + 1) // 2 if pairs else bins
        dm2 = np.logspace(-2, 2, n)
        if model == "osc2":
            self.axes, self.terms = [dm2, np.logspace(-4, 0, n)], [(1, 0)]
        elif model == "app3":
            self.axes = [dm2, np.logspace(-4, math.log10(0.5), n), np.logspace(-4, math.log10(0.45), n)]
            if bins % 2:
                E = np.concatenate([np.linspace(0.2, 3.0, bins // 2), np.linspace(0.2, 3.0, bins - bins // 2)])
        else:
            self.axes = [np.linspace(0.0, 0.1, n), dm2] * T
            self.terms = [(2 * t, 2 * t + 1) for t in range(T)]
        self.b, self.f, self.L, self.E = b, f, L, E
        self.G = n ** len(self.axes)

    def rows(self, idx):
        """Full-bin spectra [len(idx)][bins] of the grid indices idx, float64 on the GPU."""
        t = lambda x: torch.as_tensor(x, dtype=torch.float64, device=DEV)  # noqa: E731
        idx = torch.as_tensor(idx, device=DEV)
        d = len(self.axes)
        at = [(idx // self.n ** (d - 1 - a)) % self.n for a in range(d)]
        ax = [t(a) for a in self.axes]
        arg = 1.27 * ax[1 if self.model.startswith("terms") else 0][:, None] * t(self.L) / t(self.E)
        osc = torch.sin(arg) ** 2                                   # [n][bins], one row per dm2 value
        b, f = t(self.b), t(self.f)
        if self.model == "app3":
            h = self.bins // 2
            o, ue, um = osc[at[0]], ax[1][at[1]][:, None], ax[2][at[2]][:, None]
            app = b[:h] + 4.0 * ue * um * o[:, :h] * f[0, :h]
            dis = b[h:] * (1.0 - 4.0 * um * (1.0 - um) * o[:, h:])
            return torch.cat([app, dis], 1).contiguous()
        s = b.expand(len(idx), -1)
        for k, (amp, dm) in enumerate(self.terms):
            s = s + ax[amp][at[amp]][:, None] * osc[at[dm]] * f[k]
        return s.contiguous()

    def spectra(self):
        return self.rows(torch.arange(self.G, device=DEV))

    def fit_space(self, S):
        if self.collapse is None:
            return S
        out = torch.zeros(S.shape[0], self.n_fit, dtype=S.dtype, device=S.device)
        return out.index_add_(1, torch.as_tensor(self.collapse, device=S.device).long(), S)

    def cov(self, s):
        """Fit-space covariances [k][n_fit][n_fit] of full-bin spectra s [k][bins]."""
        F = torch.as_tensor(self.F, device=DEV)
        M = s[:, :, None] * F * s[:, None, :] + torch.diag_embed(s)
        if self.collapse is None:
            return M
        k = M.shape[0]
        half = self.fit_space(M.reshape(-1, self.bins)).reshape(k, self.bins, self.n_fit)
        return self.fit_space(half.transpose(1, 2).reshape(-1, self.bins)).reshape(k, self.n_fit, self.n_fit)

    def load(self, ctx):
        if self.model == "terms6":  # too large to keep as spectra: the shape model itself
            gid = fc.fc_load_grid_osc(ctx, self.axes, self.terms, self.b, self.f, self.L, self.E, recompute=True)
        else:
            S = self.spectra()
            torch.cuda.synchronize()  # the context works on a stream of its own
            gid = fc.fc_load_grid(ctx, S, self.collapse, self.n_fit)
        fc.fc_set_frac_cov(ctx, gid, self.F)
        return gid

    def pseudo_data(self, points, U, gen):
        """U pseudo-experiments [len(points) * U][n_fit] float32 of each grid point: systematic shift, then Poisson."""
        s = self.rows(points)
        F = torch.as_tensor(self.F, device=DEV)
        Lc = torch.linalg.cholesky(s[:, :, None] * F * s[:, None, :])
        z = torch.randn(len(s), U, self.bins, dtype=torch.float64, device=DEV, generator=gen)
        lam = (s[:, None, :] + z @ Lc.transpose(1, 2)).clamp_(min=0.0)
        d = torch.poisson(lam.reshape(-1, self.bins), generator=gen)
        return self.fit_space(d).float().contiguous()


def _points(G, P, seed):
    if P >= G:
        return np.arange(G, dtype=np.int64)
    rng = np.random.default_rng([seed, 1])
    if G < 1 << 20:
        return np.sort(rng.choice(G, P, replace=False)).astype(np.int64)
    return np.unique(rng.integers(0, G, 4 * P))[:P].astype(np.int64)


def _gen(seed):
    return torch.Generator(device=DEV).manual_seed(int(seed))


def _model(case, seed):
    return Model(case["model"], case["n"], case["bins"], case["pairs"], seed)


def _given_data(case, m, seed):
    """Points, pseudo-data and covariance indices of a scan: U data sets at each of P points."""
    pts = _points(m.G, case["P"], seed)
    d = m.pseudo_data(pts, case["U"], _gen(seed))
    return pts, d, np.repeat(pts, case["U"])


def _observed(case, m, seed):
    """One observed data vector: a pseudo-experiment of a point of the grid's upper half."""
    p = np.array([m.G // 2 + seed % (m.G // 2)])
    return m.pseudo_data(p, 1, _gen(seed))[0]


def _quantile_input(case, seed):
    """Statistics of rows x n universes: two degrees of freedom, a share of them exactly zero (the best fit is the
    true point), as a full job leaves them on the device."""
    g = _gen(seed)
    x = -2.0 * torch.log(torch.rand(case["rows"], case["n"], dtype=torch.float64, device=DEV, generator=g).clamp_(1e-12))
    return torch.where(x < 0.1, torch.zeros_like(x), x)


PROBS = np.array([0.68, 0.90, 0.95])


class State:
    """A context with what the program keeps in it; the context goes when the state goes."""

    def __init__(self, kind):
        self.kind, self.ctx = kind, None
        self.ctx = fc.fc_create(0, BUDGET)

    def __del__(self):
        if self.ctx is not None:
            fc.fc_destroy(self.ctx)
            self.ctx = None


def prepare(case, seed):
    kind = case["kind"]
    st = State(kind)
    st.seed = seed
    if kind == "quantiles":
        st.x = _quantile_input(case, seed)
        torch.cuda.synchronize()
        return st
    if kind == "serve":
        rng = np.random.default_rng([seed, 2])
        grids = [Model("osc2", case["n2"], case["bins2"], False, seed), Model("app3", case["n3"], case["bins3"], False, seed + 1),
                 Model("terms4", case["n4"], case["bins4"], False, seed + 2)]
        gids = [m.load(st.ctx) for m in grids]
        st.jobs = []
        for k in range(case["jobs"]):
            m, U = grids[k % 3], int(round(100.0 * 100.0 ** ((0.5 + 0.618034 * k) % 1.0)))  # log-uniform in [100, 10000]
            st.jobs.append((gids[k % 3], np.array([rng.integers(0, m.G)]), int(rng.integers(0, 2 ** 62)),
                            [np.empty((1, U)), np.empty((1, U), np.int64), np.empty((1, U), np.int8)]))
        return st
    m = st.m = _model(case, seed)
    if kind == "load":
        st.S = m.spectra().cpu().numpy()
        st.ps, d, st.q = _given_data(case, m, seed)
        st.d = d.cpu().numpy()
        return st
    st.gid = m.load(st.ctx)
    st.opts = fc.fc_default_opts(precision=case.get("precision", 1), top_k=case.get("top_k", 8))
    st.top_k, st.precision, st.U, st.new_F = case.get("top_k", 8), case.get("precision", 1), case.get("U", 1), case.get("new_F")
    if kind == "scan":
        st.ps, st.d, st.q = _given_data(case, m, seed)
    else:
        st.ps = _points(m.G, case["P"], seed)
        if kind == "data":
            st.d = _observed(case, m, seed).cpu().numpy()
        elif kind == "fake":
            st.out = torch.empty(len(st.ps), st.U, m.n_fit, dtype=torch.float32, device=DEV)
        else:
            shape = (len(st.ps), st.U)
            st.out = [torch.empty(shape, dtype=t, device=DEV) for t in (torch.float64, torch.int64, torch.int8)]
    torch.cuda.synchronize()
    return st


# ---------------------------------------------------------------- one pass --

def run(st):
    if st.kind == "fit":
        if st.new_F:
            fc.fc_set_frac_cov(st.ctx, st.gid, st.m.F)
        fc.fc_run_points(st.ctx, st.gid, st.ps, st.seed, st.U, st.opts, *st.out)
        return {"dchi2": st.out[0], "bestfit": st.out[1], "nscans": st.out[2]}
    if st.kind == "scan":
        best, chi2 = fc.fc_scan(st.ctx, st.gid, st.d, st.q, st.precision, st.top_k)
        return {"best": best, "chi2_min": chi2}
    if st.kind == "data":
        dchi2, best, ns = fc.fc_data_dchi2(st.ctx, st.gid, st.d, st.ps, st.opts)
        return {"dchi2": dchi2, "bestfit": best, "nscans": ns}
    if st.kind == "fake":
        return fc.fc_fake_data(st.ctx, st.gid, st.ps, st.seed, st.U, st.m.n_fit, out=st.out)
    if st.kind == "quantiles":
        return fc.fc_quantiles(st.ctx, st.x, PROBS)
    if st.kind == "serve":
        left = [fc.fc_submit(st.ctx, gid, p, seed, out[0].shape[1], None, *out)[0] for gid, p, seed, out in st.jobs]
        while left:
            left = [t for t in left if fc.fc_poll(st.ctx, t)[0] == fc.FC_PENDING]
            if left:
                time.sleep(1e-4)
        return [out for _, _, _, out in st.jobs]
    m = st.m
    gid = fc.fc_load_grid(st.ctx, st.S, m.collapse, m.n_fit)
    fc.fc_set_frac_cov(st.ctx, gid, m.F)
    A, L = fc.fc_covariance(st.ctx, gid, int(st.ps[0]), m.n_fit, m.bins)
    best, chi2 = fc.fc_scan(st.ctx, gid, st.d, st.q)
    fc.fc_unload_grid(st.ctx, gid)
    return {"A": A, "L": L, "best": best, "chi2_min": chi2}


def work(case):
    """What a pass cannot do without: the grid (and data) read once and the results written once; two scans of every
    universe (the second one finds the minimum repeated) as one multiply-add per bin and grid point."""
    kind = case["kind"]
    if kind == "quantiles":
        n = case["rows"] * case["n"]
        return {"bytes": 8 * n + 24 * case["rows"], "flops": n * math.log2(case["n"])}
    if kind == "serve":
        fits = case["jobs"] / 3 * 2150  # mean of U log-uniform in [100, 10000]
        size = [(case["n2"] ** 2, case["bins2"]), (case["n3"] ** 3, case["bins3"]), (case["n4"] ** 4, case["bins4"])]
        return {"bytes": sum(4 * G * N for G, N in size) + 51 * fits, "flops": sum(2 * 2 * G * N * fits for G, N in size)}
    d = {"osc2": 2, "app3": 3, "terms6": 6}[case["model"]]
    G, N = case["n"] ** d, (case["bins"] + 1) // 2 if case["pairs"] else case["bins"]
    U = case["P"] * case.get("U", 1)
    if kind == "fake":  # the triangular product and about ten operations a bin; the counts written
        return {"bytes": 4 * U * N + 4 * case["P"] * case["bins"] ** 2, "flops": U * case["bins"] * (case["bins"] + 10)}
    scans = 1 if kind in ("scan", "load") else 2
    image = 4 * G * N if kind != "load" else 8 * G * case["bins"]
    return {"bytes": image + U * (17 + (4 * N if kind in ("scan", "load") else 0)), "flops": scans * 2 * U * G * N}


# ---------------------------------------------------------------- in 64 bits --

def _whiten(m, q):
    """W [k][N][N] with W^T W = M(q)^-1 for the grid indices q."""
    Lc = torch.linalg.cholesky(m.cov(m.rows(q)))
    eye = torch.eye(m.n_fit, dtype=torch.float64, device=DEV).expand_as(Lc)
    return torch.linalg.solve_triangular(Lc, eye, upper=False)


def _exact_scan(m, pts, d, per):
    """Minimum over the grid of |W (s_g - d)|^2, `per` data sets under the covariance of each point."""
    S = m.fit_space(m.spectra())
    d = d.double().reshape(len(pts), per, -1)
    best, chi2 = [], []
    for k in range(len(pts)):
        W = _whiten(m, pts[k:k + 1])[0]
        TS = S @ W.T
        for u in range(per):
            c = ((TS - W @ d[k, u]) ** 2).sum(1)
            v, i = c.min(0)
            best.append(i)
            chi2.append(v)
    return torch.stack(best).cpu().numpy(), torch.stack(chi2).cpu().numpy()


def exact(case, seed):
    """The results in binary64 for the cases whose inputs are numbers.  The fits draw their universes from the
    library's own random streams (as does the fake data, whole counts), so they have no value from outside it."""
    kind = case["kind"]
    if kind == "quantiles":
        x = _quantile_input(case, seed).sort(1).values
        h = (case["n"] - 1) * torch.as_tensor(PROBS, device=DEV)
        lo = h.floor().long()
        a, b = x[:, lo], x[:, (lo + 1).clamp(max=case["n"] - 1)]
        return (a + (h - lo) * (b - a)).cpu().numpy()
    if kind == "scan":
        m = _model(case, seed)
        pts, d, _ = _given_data(case, m, seed)
        best, chi2 = _exact_scan(m, pts, d, case["U"])
        return {"best": best, "chi2_min": chi2}
    if kind == "load":
        m = _model(case, seed)
        pts, d, _ = _given_data(case, m, seed)
        best, chi2 = _exact_scan(m, pts, d, case["U"])
        s = m.rows(pts[:1])
        Lc = torch.linalg.cholesky(s[:, :, None] * torch.as_tensor(m.F, device=DEV) * s[:, None, :])[0]
        W = _whiten(m, pts[:1])[0]
        return {"A": (W.T @ W).cpu().numpy(), "L": Lc.cpu().numpy(), "best": best, "chi2_min": chi2}
    if kind == "data":
        m = _model(case, seed)
        d = _observed(case, m, seed).double()
        R = (m.fit_space(m.spectra()) - d).T
        pts = torch.as_tensor(_points(m.G, case["P"], seed), device=DEV)
        cur, ns = pts.clone(), torch.zeros(len(pts), dtype=torch.int8)
        best, dchi2 = torch.zeros(len(pts), dtype=torch.int64), torch.zeros(len(pts), dtype=torch.float64)
        open_ = torch.arange(len(pts))
        for it in range(1, 6):
            qs = torch.unique(cur[open_.to(DEV)])
            for q0 in range(0, len(qs), 64):
                part = qs[q0:q0 + 64]
                c = ((_whiten(m, part) @ R) ** 2).sum(1)  # [covariances][G]
                v, i = c.min(1)
                mine = open_[torch.isin(cur[open_.to(DEV)], part).cpu()]
                kk = torch.searchsorted(part, cur[mine.to(DEV)])
                best[mine] = i[kk].cpu()
                dchi2[mine] = (c[kk, pts[mine.to(DEV)]] - v[kk]).cpu()
            ns[open_] = it
            going = best[open_] != cur[open_.to(DEV)].cpu()
            open_ = open_[going]
            if not len(open_):
                break
            if it < 5:
                cur[open_.to(DEV)] = best[open_].to(DEV)
        return {"dchi2": dchi2.numpy(), "bestfit": best.numpy(), "nscans": ns.numpy()}
    return None
