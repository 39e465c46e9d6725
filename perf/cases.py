"""Performance cases: the calls that a covariance study makes, over the sizes it makes them at.

Every case goes through the public Python entry points of the package on one
context, as a program does: it holds the catalogues (or the correlation
functions), the binning and the context, and calls.  Four kinds of case:

  count     binned pair counts of several mocks (tpcf_count): periodic boxes
            with s or (s, mu) bins, cut-sky shells with the midpoint line of
            sight, logarithmic s bins, the fine 200 x 100 binning of a slab,
            many random subsets per mock, catalogues on the device (float64
            or pre-quantised) or in pinned host memory
  study     a whole small study: counts, the split Landy-Szalay estimates
            over R1, R2 and both, and the linear-construction covariance
  cov       the linear-construction or the sample covariance of given
            correlation functions, in each precision
  after     what follows the counts of a large study: projection onto
            multipoles, covariance, its accuracy and its eigenvalues
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_2205_11852_gb300 as tp

DEV = "cuda"
PREC = {"fp64": tp.TPCF_FP64, "tf32x3": tp.TPCF_TF32X3, "bf16x3": tp.TPCF_BF16X3}
M_FINAL = 50.0

_ctx = None


def _context():
    """The one context that a program keeps."""
    global _ctx
    if _ctx is None:
        _ctx = tp.Context(0)
    return _ctx


# ---------------------------------------------------------------------------
# the cases
# ---------------------------------------------------------------------------

def listed():
    return [
        # a quick study of a small simulation: the smallest calls, where launches and host work count
        {"name": "study_small", "kind": "study", "geom": "box", "n_mock": 16, "n_d": 4000, "L": 500.0, "M": 2,
         "s_max": 100.0, "n_s": 20, "n_mu": 1, "bins": "linear", "input": "f64", "prec": "fp64"},
        # an ordinary simulation box in (s, mu)
        {"name": "count_mid", "kind": "count", "geom": "box", "n_mock": 8, "n_d": 100_000, "L": 1000.0, "M": 2,
         "s_max": 200.0, "n_s": 40, "n_mu": 10, "bins": "linear", "input": "f64"},
        # a few of the largest mocks: the bulk of a production run
        {"name": "count_scale", "kind": "count", "geom": "box", "n_mock": 3, "n_d": 1_000_000, "L": 2000.0, "M": 2,
         "s_max": 200.0, "n_s": 40, "n_mu": 10, "bins": "linear", "input": "f64"},
        # light-cone mocks: an octant shell, uneven catalogue sizes, the line of sight to the pair's midpoint
        {"name": "count_cutsky", "kind": "count", "geom": "shell", "n_mock": 12, "n_d": 50_000, "n_d_hi": 400_000,
         "L": 2400.0, "M": 2, "s_max": 200.0, "n_s": 40, "n_mu": 5, "bins": "linear", "input": "f64"},
        # the brute-force comparison: one mock against 50 random subsets, pre-quantised once
        {"name": "count_subsets", "kind": "count", "geom": "box", "n_mock": 1, "n_d": 50_021, "L": 1000.0, "M": 50,
         "s_max": 200.0, "n_s": 40, "n_mu": 10, "bins": "linear", "input": "u32"},
        # the paper's own slab and binning, 1 Mpc/h x 0.01 in mu, later merged into wider bins
        {"name": "count_fine", "kind": "count", "geom": "slab", "n_mock": 1, "n_d": 155_250, "L": 1500.0, "M": 2,
         "s_max": 200.0, "n_s": 200, "n_mu": 100, "bins": "linear", "input": "f64"},
        # logarithmic separation bins, no mu: the one-dimensional function from small to large scales
        {"name": "count_log", "kind": "count", "geom": "box", "n_mock": 3, "n_d": 100_000, "L": 1000.0, "M": 2,
         "s_max": 150.0, "n_s": 24, "n_mu": 1, "bins": "log", "input": "f64"},
        # catalogues as a reader leaves them: pinned host memory
        {"name": "count_host", "kind": "count", "geom": "box", "n_mock": 8, "n_d": 60_000, "L": 1000.0, "M": 2,
         "s_max": 150.0, "n_s": 30, "n_mu": 6, "bins": "linear", "input": "host"},
        # the covariance of a full set of mocks in float64 (the default precision)
        {"name": "cov_fp64", "kind": "cov", "which": "lc", "n_mock": 3500, "nbin": 200, "prec": "fp64"},
        # the split precisions, at the full set's shape and at a ragged one
        {"name": "cov_tf32", "kind": "cov", "which": "lc", "n_mock": 3500, "nbin": 200, "prec": "tf32x3"},
        {"name": "cov_bf16_ragged", "kind": "cov", "which": "sample", "n_mock": 1201, "nbin": 333, "prec": "bf16x3"},
        # after the counts: multipoles of all mocks, their covariance, its accuracy, its eigenvalues
        {"name": "after_multipoles", "kind": "after", "n_mock": 3500, "n_s": 40, "n_mu": 5},
    ]


def _log_between(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def _pairs(c):
    """Binned pairs to expect: DD, DR_i and RR_i of uniform catalogues."""
    v = 4.0 / 3.0 * math.pi * c["s_max"] ** 3
    vol = {"box": c["L"] ** 3, "slab": c["L"] ** 2 * 300.0,
           "shell": math.pi / 6.0 * (1.0 - 0.125) * c["L"] ** 3}[c["geom"]]
    total = 0.0
    for n in _sizes(c):
        total += n * n * min(1.0, v / vol) * (0.5 + 1.5 * c["M"])
    return total


def draw(rng):
    what = rng.choice(["box", "box", "box", "shell", "log", "fine", "subsets", "host", "study", "cov", "cov",
                       "after"])
    if what == "cov":
        n_mock = int(_log_between(rng, 40, 5000))
        nbin = int(_log_between(rng, 20, 420))
        return {"kind": "cov", "which": rng.choice(["lc", "lc", "sample"]), "n_mock": n_mock, "nbin": nbin,
                "prec": rng.choice(["fp64", "fp64", "tf32x3", "bf16x3"])}
    if what == "after":
        return {"kind": "after", "n_mock": int(_log_between(rng, 200, 4000)), "n_s": rng.randrange(11, 61),
                "n_mu": rng.randrange(4, 9)}
    if what == "study":
        return {"kind": "study", "geom": "box", "n_mock": rng.randrange(5, 33), "n_d": int(_log_between(rng, 2000, 8000)),
                "L": 500.0, "M": 2, "s_max": rng.choice([80.0, 100.0, 120.0]), "n_s": rng.randrange(10, 31),
                "n_mu": rng.choice([1, 1, 4]), "bins": "linear", "input": "f64",
                "prec": rng.choice(["fp64", "tf32x3"])}
    s_max = rng.choice([120.0, 150.0, 160.0, 200.0])
    c = {"kind": "count", "geom": "box", "n_mock": 1, "n_d": 0, "L": 0.0, "M": 2, "s_max": s_max,
         "n_s": rng.randrange(12, 41), "n_mu": rng.choice([1, 4, 5, 8, 10]), "bins": "linear", "input": "f64"}
    most = 4.0e10
    if what == "shell":
        c.update(geom="shell", L=2400.0, n_d=int(_log_between(rng, 20_000, 100_000)), n_mu=rng.choice([4, 5, 8, 10]))
        c["n_d_hi"] = int(c["n_d"] * rng.uniform(1.5, 6.0))
        most = 1.2e10
    elif what == "fine":
        c.update(geom="slab", L=1500.0, n_d=int(_log_between(rng, 40_000, 160_000)), s_max=200.0, n_s=200, n_mu=100)
        most = 6.0e9
    else:
        c["n_d"] = int(_log_between(rng, 20_000, 1_000_000 if what == "box" else 120_000))
        # between a sparse halo sample and a dense one
        c["L"] = round((c["n_d"] / _log_between(rng, 4.0e-5, 1.5e-4)) ** (1.0 / 3.0), 1)
        c["L"] = max(c["L"], 3.0 * s_max + 1.0)
        if what == "log":
            c.update(bins="log", n_mu=rng.choice([1, 1, 5]))
            most = 6.0e9
        elif what == "subsets":
            c.update(M=rng.randrange(10, 51), input="u32")
        elif what == "host":
            c["input"] = "host"
    one = _pairs(c)
    while one > most and c["n_d"] > 10_000:
        c["n_d"] = int(c["n_d"] * 0.8)
        if "n_d_hi" in c:
            c["n_d_hi"] = int(c["n_d_hi"] * 0.8)
        one = _pairs(c)
    if what != "subsets":
        c["n_mock"] = max(1, min(rng.randrange(1, 17), int(most / one)))
    return c


def work(c):
    if c["kind"] == "cov":
        v = 3 if c["which"] == "lc" else 1
        n, b = c["n_mock"], c["nbin"]
        return {"bytes": 8 * (v * n * b + (5 if v == 3 else 1) * b * b), "flops": v * n * b * (b + 1)}
    if c["kind"] == "after":
        n, b, o = c["n_mock"], c["n_s"] * c["n_mu"], 3 * c["n_s"]
        return {"bytes": 8 * (3 * n * b + 3 * n * o + o * b + 6 * o * o),
                "flops": 3 * 2 * n * o * b + 3 * n * o * (o + 1) + 4 * o ** 3 // 3}
    pts = sum(_sizes(c)) * (1 + c["M"])
    out = 8 * c["n_mock"] * (1 + 2 * c["M"]) * c["n_s"] * c["n_mu"]
    # a pair cannot do without its squared distance (7), and a binned one without its bin and its add (8)
    return {"bytes": pts * (12 if c["input"] == "u32" else 24) + out, "flops": int(15 * _pairs(c))}


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------

def _sizes(c):
    """Data points of each mock (the random subsets have as many each)."""
    lo, hi = c["n_d"], c.get("n_d_hi", c["n_d"])
    return [int(lo + (hi - lo) * ((0.5 + 0.6180339887 * i) % 1.0)) for i in range(c["n_mock"])]


def _wrap(x, top):
    x = torch.remainder(x, top)
    return torch.where(x >= top, torch.zeros_like(x), x)


def _clustered(g, n, L, n_parent, sigma):
    """Children of uniform parents with a Gaussian scatter in a periodic cube."""
    n_p = max(1, round(n_parent * L ** 3))
    parents = torch.rand(n_p, 3, generator=g, device=DEV, dtype=torch.float64) * L
    which = torch.randint(n_p, (n,), generator=g, device=DEV)
    return _wrap(parents[which] + sigma * torch.randn(n, 3, generator=g, device=DEV, dtype=torch.float64), L)


def _shell_clustered(g, n, L):
    """Clustered points in the octant shell L/2 <= r < L."""
    got, have = [], 0
    while have < n:
        x = _clustered(g, int((n - have) / 0.458 * 1.15) + 1024, L, 1.0e-5, 3.0)
        r2 = (x * x).sum(1)
        got.append(x[(r2 >= 0.25 * L * L) & (r2 < L * L)])
        have += len(got[-1])
    return torch.cat(got)[:n].contiguous()


def _shell_uniform(g, n, L):
    u = torch.rand(n, generator=g, device=DEV, dtype=torch.float64)
    r = (u * (1.0 - 0.125) + 0.125) ** (1.0 / 3.0) * (L * (1.0 - 1e-12))
    d = torch.randn(n, 3, generator=g, device=DEV, dtype=torch.float64).abs()
    return d / d.norm(dim=1, keepdim=True) * r[:, None]


def _catalogues(c, seed):
    """[(data, randoms of all M subsets)] of every mock, float64 on the device."""
    g = torch.Generator(device=DEV).manual_seed(1_000_003 * int(seed) + 17)
    out = []
    for n in _sizes(c):
        nr = n * c["M"]
        if c["geom"] == "shell":
            out.append((_shell_clustered(g, n, c["L"]), _shell_uniform(g, nr, c["L"])))
        elif c["geom"] == "slab":
            dims = torch.tensor([c["L"], c["L"], 300.0], device=DEV, dtype=torch.float64)
            d = _clustered(g, n, c["L"], 1.0e-5, 3.0)
            d[:, 2] *= 300.0 / c["L"]
            out.append((d, torch.rand(nr, 3, generator=g, device=DEV, dtype=torch.float64) * dims))
        else:
            out.append((_clustered(g, n, c["L"], 1.0e-5 if c["L"] < 1500.0 else 2.0e-6, 3.0),
                        _wrap(torch.rand(nr, 3, generator=g, device=DEV, dtype=torch.float64) * c["L"], c["L"])))
    return out


def _grid(x, L):
    """Grid coordinates of a periodic box, [3][n] 32-bit."""
    t = x / L
    v = torch.floor((t - torch.floor(t)) * 4294967296.0)
    v = torch.where(v >= 4294967296.0, v - 4294967296.0, v).to(torch.int64)
    return torch.where(v >= 2 ** 31, v - 2 ** 32, v).to(torch.int32).T.contiguous()


def _edges(c):
    if c["bins"] == "log":
        return np.geomspace(c["s_max"] / 200.0, c["s_max"], c["n_s"] + 1)
    return np.linspace(0.0, c["s_max"], c["n_s"] + 1)


def _binning(c):
    if c["geom"] == "box":
        return tp.make_binning(_edges(c), c["n_mu"], tp.TPCF_PERIODIC, c["L"])
    if c["geom"] == "slab":
        return tp.make_binning(_edges(c), c["n_mu"], tp.TPCF_OPEN, c["L"], los=tp.TPCF_LOS_X)
    return tp.make_binning(_edges(c), c["n_mu"], tp.TPCF_OPEN, c["L"], los=tp.TPCF_LOS_MIDPOINT,
                           observer=(0.0, 0.0, 0.0))


def _mocks(c, seed):
    mocks = []
    for d, r in _catalogues(c, seed):
        offs = [len(d) * i for i in range(c["M"] + 1)]
        if c["input"] == "u32":
            mocks.append({"data_u32": _grid(d, c["L"]), "randoms_u32": _grid(r, c["L"]), "offsets": offs})
        elif c["input"] == "host":
            mocks.append({"data": d.cpu().pin_memory(), "randoms": r.cpu().pin_memory(), "offsets": offs})
        else:
            mocks.append({"data": d, "randoms": r, "offsets": offs})
    return mocks


def _variants(n_mock, nbin, seed):
    """Correlation functions of n_mock mocks against R1, R2 and R1 u R2: a smooth mean, a few correlated
    modes, and noise of its own from each random subset."""
    g = torch.Generator(device=DEV).manual_seed(1_000_003 * int(seed) + 29)

    def normal(*shape):
        return torch.randn(*shape, generator=g, device=DEV, dtype=torch.float64)

    k = torch.arange(nbin, device=DEV, dtype=torch.float64)
    modes = torch.stack([torch.cos(math.pi * (j + 0.5) * k / nbin) for j in range(8)])
    amp = normal(n_mock, 8) * (0.02 / (1.0 + torch.arange(8, device=DEV, dtype=torch.float64)))
    data = 0.5 * torch.exp(-k / (0.2 * nbin)) + amp @ modes + 0.003 * normal(n_mock, nbin)
    e1, e2 = 0.004 * normal(n_mock, nbin), 0.004 * normal(n_mock, nbin)
    return data + e1, data + e2, data + 0.5 * (e1 + e2)


def prepare(case, seed):
    c = dict(case)
    s = {"case": c, "ctx": _context()}
    if c["kind"] == "cov":
        xs = _variants(c["n_mock"], c["nbin"], seed)
        s["xi"] = xs if c["which"] == "lc" else xs[2:]
    elif c["kind"] == "after":
        s["xi"] = _variants(c["n_mock"], c["n_s"] * c["n_mu"], seed)
        s["P"] = torch.from_numpy(tp.tpcf_multipole_matrix(c["n_s"], c["n_mu"], (0, 2, 4))).to(DEV)
    else:
        s["mocks"] = _mocks(c, seed)
        s["binning"] = _binning(c)
        s["n_d"] = _sizes(c)
        s["n_r"] = [[n] * c["M"] for n in s["n_d"]]
    return s


# ---------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------

def run(s):
    c, ctx = s["case"], s["ctx"]
    if c["kind"] == "count":
        return ctx.tpcf_count(s["mocks"], s["binning"])
    if c["kind"] == "study":
        n = ctx.tpcf_count(s["mocks"], s["binning"])
        xi = [ctx.tpcf_ls(n["dd"], n["dr"], n["rr"], s["n_d"], s["n_r"], sel) for sel in ([0], [1], [0, 1])]
        return {"counts": n, "xi": xi, "cov": ctx.tpcf_lc_cov(*xi, 1, M_FINAL, PREC[c["prec"]])}
    if c["kind"] == "cov":
        if c["which"] == "sample":
            return ctx.tpcf_sample_cov(s["xi"][0], PREC[c["prec"]])
        return ctx.tpcf_lc_cov(*s["xi"], 1, M_FINAL, PREC[c["prec"]])
    y = [ctx.tpcf_project(s["P"], x) for x in s["xi"]]
    cov = ctx.tpcf_lc_cov(*y, 1, M_FINAL, tp.TPCF_FP64)
    return {"y": y, "cov": cov,
            "var": ctx.tpcf_covcov_var(cov["A"], cov["B"], c["n_mock"], 1, M_FINAL),
            "chi2": ctx.tpcf_chi2_predict(cov["A"], cov["B"], cov["C_lc"], 1, M_FINAL),
            "eig": ctx.tpcf_eigvalsh(cov["C_lc"])}


# ---------------------------------------------------------------------------
# the same in 64 bits, in plain torch
# ---------------------------------------------------------------------------

def _exact_sample(x):
    y = x - x.mean(0, keepdim=True)
    y = y - y.mean(0, keepdim=True)
    return (y.T @ y) / (x.shape[0] - 1)


def _exact_lc(xs):
    c1, c2, cb = (_exact_sample(x) for x in xs)
    ca = 0.5 * (c1 + c2)
    a, b = 2.0 * cb - ca, 2.0 * (ca - cb)
    return {"C_lc": a + b / M_FINAL, "Ca": ca, "Cb": cb, "A": a, "B": b}


def _exact_pairs(a, b, L, edges, n_mu):
    """Histogram of the ordered pairs of two periodic catalogues, brute force."""
    n_s = len(edges) - 1
    h = torch.zeros(n_s * n_mu, device=DEV, dtype=torch.int64)
    e = torch.from_numpy(edges).to(DEV)
    for i in range(0, len(a), 500):
        d = a[i:i + 500, None, :] - b[None, :, :]
        d = d - L * torch.round(d / L)
        s = d.square().sum(2).sqrt()
        k = torch.bucketize(s, e, right=True) - 1
        ok = (k >= 0) & (k < n_s) & (s > 0.0)
        j = (n_mu * d[..., 0].abs() / s.clamp(min=1e-300)).to(torch.int64).clamp(max=n_mu - 1)
        h += torch.bincount((k * n_mu + j)[ok], minlength=n_s * n_mu)
    return h.to(torch.float64)


def _multipoles(n_s, n_mu):
    """(2l+1) times the integral of P_l over each |mu| bin, l = 0, 2, 4."""
    m = np.linspace(0.0, 1.0, n_mu + 1)
    prim = [m, 2.5 * (m ** 3 - m), 9.0 / 8.0 * (7.0 * m ** 5 - 10.0 * m ** 3 + 3.0 * m)]
    rows = [np.kron(np.eye(n_s), np.diff(p)[None, :]) for p in prim]
    return torch.from_numpy(np.concatenate(rows)).to(DEV)


def exact(case, seed):
    c = dict(case)
    if c["kind"] == "cov":
        xs = _variants(c["n_mock"], c["nbin"], seed)
        return _exact_lc(xs) if c["which"] == "lc" else _exact_sample(xs[2])
    if c["kind"] == "after":
        P = _multipoles(c["n_s"], c["n_mu"])
        y = [x @ P.T for x in _variants(c["n_mock"], c["n_s"] * c["n_mu"], seed)]
        cov = _exact_lc(y)
        A, B, C, w = cov["A"], cov["B"], cov["C_lc"], 0.5 - 1.0 / M_FINAL
        D = A + 0.5 * B

        def fluct(m):
            return torch.outer(m.diagonal(), m.diagonal()) + m * m

        var = (fluct(D) + w * w * fluct(B)) / (c["n_mock"] - 1)
        chi2 = ((c["n_mock"] - 1) * var / torch.outer(C.diagonal(), C.diagonal())).mean()
        return {"y": y, "cov": cov, "var": var, "chi2": chi2, "eig": torch.linalg.eigvalsh(C)}
    if c["kind"] == "study":
        if sum(n * n for n in _sizes(c)) * (1 + 2 * c["M"]) > 8e9:
            return None
        xi, edges = [[], [], []], _edges(c)
        for d, r in _catalogues(c, seed):
            n = len(d)
            rs = [r[i * n:(i + 1) * n] for i in range(c["M"])]
            ddn = _exact_pairs(d, d, c["L"], edges, c["n_mu"]) / 2.0 / (n * (n - 1) / 2.0)
            drn = [_exact_pairs(d, x, c["L"], edges, c["n_mu"]) / (float(n) * n) for x in rs]
            rrn = [_exact_pairs(x, x, c["L"], edges, c["n_mu"]) / 2.0 / (n * (n - 1) / 2.0) for x in rs]
            for v, sel in enumerate(([0], [1], [0, 1])):
                q = sum(drn[i] for i in sel) / len(sel)
                p = sum(rrn[i] for i in sel) / len(sel)
                xi[v].append((ddn - 2.0 * q) / p + 1.0)
        xi = [torch.stack(x) for x in xi]
        return {"counts": None, "xi": xi, "cov": _exact_lc(xi)}
    return None  # counts are whole numbers
