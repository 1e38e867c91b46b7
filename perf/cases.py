"""The cases that this library's speed is measured on.

Every case is one pass of a user's program through the public entry points
(``Items``, ``overlap_align``): all pairs of a point-cloud set, their adjoint
or a batch of registrations, all pairs or a list of pairs of a vector set, all
pairs of a sparse set.  Item sets are kept in handles, as programs keep them;
vector sets are loaded anew in every pass (``Items.update``), because that is
how a program feeds a stream of new vectors to one handle.

``exact`` restates each result in 64 bits with plain torch.  The tolerances
are about four times the distance from those restatements, rounded up.

Paths whose time is the host link's (vectors in pinned host memory, in and out
of core) are left to ``bench.py``: a link's rate differs from box to box by
more than a kernel could change.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2009_04755_gb300 import (AP_FN_BHATTACHARYYA, AP_FN_COSINE, AP_FN_GMM_L2,
                                    AP_FN_OVERLAP, AP_FN_PEARSON, AP_PREC_FP32,
                                    AP_PREC_SPLIT_BF16, Items)
from paper_2009_04755_gb300.autograd import overlap_align

FN = {"overlap": AP_FN_OVERLAP, "gmm_l2": AP_FN_GMM_L2, "bhattacharyya": AP_FN_BHATTACHARYYA}
LN2 = math.log(2.0)
ETA, FMIN = 1e-3, 1e-30
COMMON_SHARE, COMMON_BOOST = 1.0 / 16.0, 8.0      # of a sparse set's codes


def listed():
    return [
        # a handful of small particles compared while someone waits: launches
        # and latency are all there is
        dict(name="overlap2d_small", family="clouds", fn="overlap", dim=2, n=48, sizes="uniform",
             lo=20, hi=60, smin=0.02, smax=0.05, weights=False, transforms=False),
        # the plain method's standard set: 256 clouds of 64-128 points
        dict(name="overlap2d_n256", family="clouds", fn="overlap", dim=2, n=256, sizes="uniform",
             lo=64, hi=128, smin=0.02, smax=0.05, weights=False, transforms=False),
        # uneven 3-D clouds of 50-5000 points (the batching workload's sizes)
        dict(name="overlap3d_lognormal", family="clouds", fn="overlap", dim=3, n=1000,
             sizes="lognormal", lo=50, hi=5000, smin=0.01, smax=0.05, weights=False,
             transforms=False),
        # localisation-microscopy particles, scored by the GMM L2 distance
        dict(name="gmm_l2_particles", family="clouds", fn="gmm_l2", dim=2, n=256, sizes="uniform",
             lo=1000, hi=2000, smin=0.01, smax=0.03, weights=False, transforms=False),
        # one step of a user's own optimiser: the overlap of every pair under
        # its transform, and the gradient, through autograd
        dict(name="align2d", family="align", n=301, lo=100, hi=400),
        # all-to-all registration: 20 ascent steps for every pair
        dict(name="ascent2d", family="ascent", n=400, lo=100, hi=400, steps=20, pairs=0),
        # a few short noise vectors: launches and latency again
        dict(name="pearson_small", family="pearson", precision="split", n=100, dim=1000),
        # an ordinary correlation of ragged size
        dict(name="pearson_mid", family="pearson", precision="split", n=1000, dim=50_000),
        # long noise patterns, the headline workload's vector length
        dict(name="pearson_large", family="pearson", precision="split", n=4096, dim=1 << 20),
        # the plain FP32 precision, chosen by those who do not want the split
        dict(name="pearson_fp32", family="pearson", precision="fp32", n=1024, dim=65_536),
        # chosen pairs of a resident set
        dict(name="pearson_list", family="pearson_list", precision="split", n=1024, dim=1 << 18,
             pairs=3000),
        # composition vectors over 20^6 codes, 1e5 to 1.8e6 entries each
        dict(name="cosine_sparse", family="cosine", n=256, codes=20 ** 6, lo=100_000,
             hi=1_800_000),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    family = rng.choice(["clouds", "clouds", "score", "align", "ascent", "pearson", "pearson",
                         "pearson_list", "cosine"])
    if family in ("clouds", "score"):
        dim = rng.choice([2, 3])
        fn = "overlap" if family == "clouds" else rng.choice(["gmm_l2", "bhattacharyya"])
        sizes = rng.choice(["uniform", "lognormal"])
        lo = _log_int(rng, 50, 500)
        hi = min(5000, lo * 10) if sizes == "lognormal" else 2 * lo
        mean = (lo + hi) / 2 if sizes == "uniform" else 3 * lo
        most = int(min(2000.0, math.sqrt(2 * 5e10) / mean))      # point pairs of one pass
        return dict(family="clouds", fn=fn, dim=dim, n=_log_int(rng, 4, most), sizes=sizes, lo=lo,
                    hi=hi, smin=rng.choice([0.01, 0.02]), smax=rng.choice([0.03, 0.05]),
                    weights=rng.random() < 0.4, transforms=dim == 2 and rng.random() < 0.4)
    if family == "align":
        return dict(family="align", n=_log_int(rng, 4, 500), lo=rng.randint(20, 100),
                    hi=rng.randint(100, 400))
    if family == "ascent":
        n = _log_int(rng, 4, 400)
        return dict(family="ascent", n=n, lo=rng.randint(20, 100), hi=rng.randint(100, 400),
                    steps=rng.randint(1, 20),
                    pairs=_log_int(rng, 1, n * (n - 1) // 2) if rng.random() < 0.5 else 0)
    if family == "pearson":
        precision = rng.choice(["split", "split", "fp32"])
        dim = _log_int(rng, 64, 1 << 19)
        n = _log_int(rng, 8, min(3000, (1 << 30) // dim))
        if precision == "fp32":
            n = max(8, min(n, int(math.sqrt(2e11 / dim))))
        return dict(family="pearson", precision=precision, n=n, dim=dim)
    if family == "pearson_list":
        dim = _log_int(rng, 64, 1 << 18)
        n = _log_int(rng, 8, min(2000, (1 << 28) // dim))
        return dict(family="pearson_list", precision=rng.choice(["split", "fp32"]), n=n, dim=dim,
                    pairs=_log_int(rng, 16, 5000))
    codes = 20 ** rng.randint(3, 6)
    hi = max(8, int(codes * rng.uniform(0.002, 0.03)))
    return dict(family="cosine", n=_log_int(rng, 8, 256), codes=codes, lo=max(4, hi // 18), hi=hi)


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
def _gen(seed, device="cuda"):
    return torch.Generator(device=device).manual_seed(int(seed))


def _uniform(g, count, lo, hi):
    return torch.rand(count, generator=g, device="cuda") * (hi - lo) + lo


def _cloud_inputs(c, seed):
    """Points uniform in the box [-1, 1]^dim, per-point sigma uniform."""
    h = np.random.default_rng([int(seed), 1])
    if c["sizes"] == "lognormal":
        s = np.exp(math.log(math.sqrt(c["lo"] * c["hi"]) * 0.6) + h.standard_normal(c["n"]))
        s = np.clip(np.rint(s), c["lo"], c["hi"]).astype(np.int64)
    else:
        s = h.integers(c["lo"], c["hi"] + 1, size=c["n"])
    off = np.concatenate([[0], np.cumsum(s)]).astype(np.int64)
    g, m = _gen(seed), int(off[-1])
    return {"dim": c["dim"], "offsets": off, "x": _uniform(g, m, -1, 1), "y": _uniform(g, m, -1, 1),
            "z": _uniform(g, m, -1, 1) if c["dim"] == 3 else None,
            "sigma": _uniform(g, m, c["smin"], c["smax"]),
            "weight": _uniform(g, m, 0.25, 1.75) if c["weights"] else None}


def _template_inputs(c, seed):
    """Clouds that are random poses of 8 templates of 400 points, with jitter."""
    h = np.random.default_rng([int(seed), 2])
    n = c["n"]
    s = h.integers(c["lo"], c["hi"] + 1, size=n)
    off = np.concatenate([[0], np.cumsum(s)]).astype(np.int64)
    templ = h.uniform(-0.5, 0.5, size=(8, 400, 2))
    theta, t = h.uniform(-math.pi, math.pi, n), h.uniform(-0.5, 0.5, (n, 2))
    xy = np.empty((int(off[-1]), 2))
    for i in range(n):
        p = templ[i % 8, h.permutation(400)[:s[i]]]
        co, si = math.cos(theta[i]), math.sin(theta[i])
        xy[off[i]:off[i + 1]] = p @ np.array([[co, si], [-si, co]]) + t[i]
    xy += 0.01 * h.standard_normal(xy.shape)
    xy = torch.from_numpy(xy.astype(np.float32)).cuda()
    return {"dim": 2, "offsets": off, "x": xy[:, 0].contiguous(), "y": xy[:, 1].contiguous(),
            "z": None, "sigma": _uniform(_gen(seed), int(off[-1]), 0.02, 0.05), "weight": None}


def _params(n_pairs, seed):
    """Transforms (theta, tx, ty) near the identity, as an optimiser visits them."""
    return torch.randn(n_pairs, 3, generator=_gen(seed + 1), device="cuda") * 0.1


def _vector_inputs(c, seed):
    """Unit noise plus a component of weight 0.05 shared by groups of 16 rows."""
    g = _gen(seed)
    X = torch.randn(c["n"], c["dim"], generator=g, device="cuda")
    shared = torch.randn((c["n"] + 15) // 16, c["dim"], generator=g, device="cuda")
    group = torch.from_numpy(np.random.default_rng([int(seed), 3]).permutation(c["n"]) // 16).cuda()
    for r in range(0, c["n"], 256):
        X[r:r + 256].add_(shared[group[r:r + 256]], alpha=0.05)
    return X


def _sparse_inputs(c, seed):
    """Codes 8 times as frequent in the first sixteenth of the index space,
    values that share a global component, so rows correlate where they meet."""
    g = _gen(seed)
    codes = c["codes"]
    common = max(1, int(codes * COMMON_SHARE))
    share = _common_share()
    sizes = np.random.default_rng([int(seed), 4]).integers(c["lo"], c["hi"] + 1, size=c["n"])
    field = torch.randn(codes, generator=g, device="cuda")
    idx, val, off = [], [], [0]
    for m in sizes:
        m = int(m)
        k = int(round(m * share))
        a = torch.randint(0, common, (k,), generator=g, device="cuda", dtype=torch.int32)
        b = torch.randint(common, codes, (m - k,), generator=g, device="cuda", dtype=torch.int32)
        ids = torch.unique(torch.cat([a, b]))
        idx.append(ids)
        val.append(0.6 * field[ids.long()] + torch.randn(len(ids), generator=g, device="cuda"))
        off.append(off[-1] + len(ids))
    return np.array(off, np.int64), torch.cat(idx), torch.cat(val)


def _common_share():
    return COMMON_SHARE * COMMON_BOOST / (COMMON_SHARE * COMMON_BOOST + 0.5)


def _list(c, seed):
    h = np.random.default_rng([int(seed), 5])
    a = h.integers(0, c["n"], size=c["pairs"])
    b = (a + h.integers(1, c["n"], size=c["pairs"])) % c["n"]
    return a.astype(np.int32), b.astype(np.int32)


def _inputs(c, seed):
    """Everything a pass reads, as the caller has it."""
    f = c["family"]
    if f == "clouds":
        d = {"clouds": _cloud_inputs(c, seed)}
        d["params"] = _params(c["n"] * (c["n"] - 1) // 2, seed) if c["transforms"] else None
        return d
    if f == "align":
        p = c["n"] * (c["n"] - 1) // 2
        return {"clouds": _template_inputs(c, seed), "params": _params(p, seed),
                "grad": torch.rand(p, generator=_gen(seed + 2), device="cuda") + 0.5}
    if f == "ascent":
        p = c["pairs"] or c["n"] * (c["n"] - 1) // 2
        return {"clouds": _template_inputs(c, seed), "pairs": _list(c, seed) if c["pairs"] else None,
                "params": _params(p, seed) * 0.1}
    if f == "pearson":
        return {"X": _vector_inputs(c, seed)}
    if f == "pearson_list":
        return {"X": _vector_inputs(c, seed), "pairs": _list(c, seed)}
    return {"csr": _sparse_inputs(c, seed)}


def _precision(c):
    return AP_PREC_FP32 if c["precision"] == "fp32" else AP_PREC_SPLIT_BF16


def prepare(case, seed):
    s = _inputs(case, seed)
    s["case"] = case
    if "clouds" in s:
        s["items"] = Items.from_clouds(s.pop("clouds"))
    elif "X" in s:
        s["items"] = Items.from_vectors(s["X"], precisions=(_precision(case),))
        if case["family"] == "pearson_list":
            torch.cuda.synchronize()
            del s["X"]
    else:
        s["items"] = Items.from_sparse(*s.pop("csr"), dim=case["codes"])
    return s


# ---------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------
def run(s):
    c, items = s["case"], s["items"]
    f = c["family"]
    if f == "clouds":
        return items.run_pairs(FN[c["fn"]], params=s["params"])
    if f == "align":
        params = s["params"].detach().requires_grad_()
        cost = overlap_align(items, params)
        cost.backward(s["grad"])
        return {"f": cost.detach(), "grad": params.grad}
    if f == "ascent":
        start = s["params"].clone()
        if s["pairs"] is None:
            params, cost, flags = items.ascent(start, c["steps"], ETA, FMIN)
        else:
            params, cost, flags = items.ascent_list(*s["pairs"], start, c["steps"], ETA, FMIN)
        return {"params": params, "f": cost, "flags": flags}
    if f == "pearson":
        items.update(s["X"])
        return items.run_pairs(AP_FN_PEARSON, precision=_precision(c))
    if f == "pearson_list":
        return items.run_pairs_list(*s["pairs"], AP_FN_PEARSON, precision=_precision(c))
    return items.run_pairs(AP_FN_COSINE)


def _point_pairs(c):
    if c["family"] == "clouds" and c["sizes"] == "lognormal":
        mid = math.log(math.sqrt(c["lo"] * c["hi"]) * 0.6)
        z = np.linspace(-4, 4, 2001)
        w = np.exp(-z * z / 2)
        mean = float((np.clip(np.exp(mid + z), c["lo"], c["hi"]) * w).sum() / w.sum())
    else:
        mean = (c["lo"] + c["hi"]) / 2
    return mean, (c.get("pairs") or c["n"] * (c["n"] - 1) // 2) * mean * mean


def work(case):
    """Points, rows or entries read once and results written once; the
    arithmetic of each term, an exponential or a reciprocal counted as one."""
    c, f = case, case["family"]
    if f in ("clouds", "align", "ascent"):
        mean, terms = _point_pairs(c)
        pairs = c.get("pairs") or c["n"] * (c["n"] - 1) // 2
        points = c["n"] * mean * 16
        dim = c.get("dim", 2)
        per = 3 * dim + 4 + (1 if c.get("fn", "overlap") != "overlap" else 0)
        if f == "clouds":
            return {"bytes": points + pairs * (16 if c["transforms"] else 4), "flops": per * terms}
        per += 5
        if f == "align":
            return {"bytes": points + pairs * 32, "flops": per * terms}
        return {"bytes": points + pairs * 32, "flops": per * terms * c["steps"]}
    if f == "pearson":
        pairs = c["n"] * (c["n"] - 1) // 2
        return {"bytes": 4.0 * c["n"] * c["dim"] + 8.0 * pairs,
                "flops": (6.0 if c["precision"] == "split" else 2.0) * c["dim"] * pairs}
    if f == "pearson_list":
        # rows that the list names at all
        rows = c["n"] * (1 - (1 - 1 / c["n"]) ** (2 * c["pairs"]))
        return {"bytes": 4.0 * rows * c["dim"] + 16.0 * c["pairs"],
                "flops": (6.0 if c["precision"] == "split" else 2.0) * c["dim"] * c["pairs"]}
    m, share = (c["lo"] + c["hi"]) / 2, _common_share()
    pairs = c["n"] * (c["n"] - 1) // 2
    common = c["codes"] * COMMON_SHARE
    meets = (m * share) ** 2 / common + (m * (1 - share)) ** 2 / (c["codes"] - common)
    return {"bytes": 8.0 * c["n"] * m + 8.0 * pairs, "flops": 2.0 * meets * pairs}


def tolerance(case):
    """Measured against ``exact``: 3e-8 to 8e-8 for costs (FP32 terms), 1.5e-7
    for gradients, 4.5e-6 for the split-BF16 Gram (c = hi + lo leaves 2^-17 of
    every factor, the correlations being 1/sqrt(dim) in size), 4.7e-6 for FP32
    sums over 65,536 columns (a random walk, so it goes with the square root),
    3e-8 for the sparse cosine."""
    f = case["family"]
    if f == "clouds":
        return {"rel": 4e-7, "max": 4e-6}
    if f == "align":
        return {"rel": 8e-7, "max": 2e-5}
    if f == "ascent":
        return {"rel": 1e-6, "max": 1e-4, "differ": 1e-3}
    if f in ("pearson", "pearson_list"):
        if case["precision"] == "split":
            return {"rel": 2e-5, "max": 2e-4}
        rel = max(4e-6, 8e-8 * math.sqrt(case["dim"]))
        return {"rel": rel, "max": 20 * rel}
    return {"rel": 2e-7, "max": 4e-6}


# ---------------------------------------------------------------------------
# the same results in 64 bits
# ---------------------------------------------------------------------------
def _terms(fn, dim, d2, s2, ww, sa, sb):
    if fn == "overlap":
        return ww * torch.exp(-d2 / (2 * s2))
    if fn == "gmm_l2":
        return ww * (2 * math.pi * s2) ** (-dim / 2) * torch.exp(-d2 / (2 * s2))
    return ww.sqrt() * (2 * sa * sb / s2) ** (dim / 2) * torch.exp(-d2 / (4 * s2))


def _exact_clouds(c, d):
    cl, fn, dim, n = d["clouds"], c["fn"], c["dim"], c["n"]
    off = cl["offsets"]
    X = torch.stack([cl[k].double() for k in ("x", "y", "z")[:dim]])
    S = cl["sigma"].double()
    W = cl["weight"].double() if cl["weight"] is not None else torch.ones_like(S)
    size = torch.from_numpy(np.diff(off)).cuda()
    item = torch.repeat_interleave(torch.arange(n, device="cuda"), size)
    P = d["params"].double() if d["params"] is not None else None
    step = 1 << 27

    def sums(i, b0, b1, Y):
        """Per point b in [b0, b1) (at Y), its terms with cloud i summed."""
        a0, a1 = int(off[i]), int(off[i + 1])
        out = torch.zeros(b1 - b0, dtype=torch.float64, device="cuda")
        for q0 in range(b0, b1, max(1, step // max(1, a1 - a0))):
            q1 = min(b1, q0 + max(1, step // max(1, a1 - a0)))
            d2 = 0
            for k in range(dim):
                d2 = d2 + (X[k, a0:a1, None] - Y[k, None, q0 - b0:q1 - b0]) ** 2
            s2 = S[a0:a1, None] ** 2 + S[None, q0:q1] ** 2
            out[q0 - b0:q1 - b0] = _terms(fn, dim, d2, s2, W[a0:a1, None] * W[None, q0:q1],
                                          S[a0:a1, None], S[None, q0:q1]).sum(0)
        return out

    rows = []
    own = torch.zeros(n, dtype=torch.float64, device="cuda")
    for i in range(n):
        b0, b1 = int(off[i + 1]), int(off[n])
        if fn == "gmm_l2":
            own[i] = sums(i, int(off[i]), b0, X[:, int(off[i]):b0]).sum()
        if i == n - 1:
            break
        Y = X[:, b0:b1]
        if P is not None:
            p0 = i * n - i * (i + 1) // 2
            p = P[p0:p0 + n - 1 - i][item[b0:b1] - i - 1]
            co, si = torch.cos(p[:, 0]), torch.sin(p[:, 0])
            Y = torch.stack([co * Y[0] - si * Y[1] + p[:, 1], si * Y[0] + co * Y[1] + p[:, 2]])
        row = torch.zeros(n - 1 - i, dtype=torch.float64, device="cuda")
        rows.append(row.index_add_(0, item[b0:b1] - i - 1, sums(i, b0, b1, Y)))
    f = torch.cat(rows)
    if fn == "gmm_l2":
        pi, pj = torch.triu_indices(n, n, 1, device="cuda")
        f = own[pi] + own[pj] - 2 * f
    return f


def _cost_and_gradient(cl, pi, pj, P):
    """f and df/d(theta, tx, ty) of the listed pairs, pj moved; 64 bits."""
    off = cl["offsets"]
    x, y, s = cl["x"].double(), cl["y"].double(), cl["sigma"].double()
    size = np.diff(off)
    f = torch.empty(len(pi), dtype=torch.float64, device="cuda")
    g = torch.empty(len(pi), 3, dtype=torch.float64, device="cuda")
    order = np.argsort(pi, kind="stable")
    cut = np.flatnonzero(np.diff(pi[order])) + 1
    for group in np.split(order, cut):
        i = int(pi[group[0]])
        js = pj[group]
        a = slice(int(off[i]), int(off[i + 1]))
        at = np.concatenate([np.arange(off[j], off[j + 1]) for j in js])
        seg = torch.from_numpy(np.repeat(np.arange(len(js)), size[js])).cuda()
        b, k = torch.from_numpy(at).cuda(), torch.from_numpy(group).cuda()
        p = P[k][seg]
        co, si = torch.cos(p[:, 0]), torch.sin(p[:, 0])
        rx, ry = co * x[b] - si * y[b], si * x[b] + co * y[b]
        dx, dy = x[a, None] - (rx + p[:, 1])[None], y[a, None] - (ry + p[:, 2])[None]
        s2 = s[a, None] ** 2 + s[b][None] ** 2
        e = torch.exp(-(dx * dx + dy * dy) / (2 * s2))
        es = e / s2
        gx, gy = (es * dx).sum(0), (es * dy).sum(0)
        m = torch.zeros(len(js), 4, dtype=torch.float64, device="cuda")
        m.index_add_(0, seg, torch.stack([e.sum(0), gy * rx - gx * ry, gx, gy], 1))
        f[k], g[k] = m[:, 0], m[:, 1:]
    return f, g


def _exact_pearson(c, X, pairs):
    n, dim = X.shape
    mu = torch.cat([X[r:r + 64].double().mean(1) for r in range(0, n, 64)])
    if pairs is not None:
        pi, pj = (torch.from_numpy(v).long().cuda() for v in pairs)
        out = []
        m = max(1, (1 << 28) // dim)
        for k in range(0, len(pi), m):
            a = X[pi[k:k + m]].double() - mu[pi[k:k + m], None]
            b = X[pj[k:k + m]].double() - mu[pj[k:k + m], None]
            out.append((a * b).sum(1) / ((a * a).sum(1) * (b * b).sum(1)).sqrt())
        return torch.cat(out)
    G = torch.zeros(n, n, dtype=torch.float64, device="cuda")
    rows = max(64, (n + 7) // 8)
    for k in range(0, dim, 1 << 16):
        C = X[:, k:k + (1 << 16)].double() - mu[:, None]
        for r in range(0, n, rows):
            G[r:r + rows, r:] += C[r:r + rows] @ C[r:].T
    pi, pj = torch.triu_indices(n, n, 1, device="cuda")
    ss = G.diagonal()
    return G[pi, pj] / (ss[pi] * ss[pj]).sqrt()


def _exact_cosine(c, csr):
    off, idx, val = csr
    n, codes = c["n"], c["codes"]
    row = torch.repeat_interleave(torch.arange(n, device="cuda"),
                                  torch.from_numpy(np.diff(off)).cuda())
    G = torch.zeros(n, n, dtype=torch.float64, device="cuda")
    step = 1 << 21
    for k in range(0, codes, step):
        m = (idx >= k) & (idx < k + step)
        A = torch.zeros(n, min(step, codes - k), dtype=torch.float64, device="cuda")
        A[row[m], idx[m].long() - k] = val[m].double()
        G += A @ A.T
    pi, pj = torch.triu_indices(n, n, 1, device="cuda")
    ss = G.diagonal()
    return G[pi, pj] / (ss[pi] * ss[pj]).sqrt()


def exact(case, seed):
    c, f = case, case["family"]
    d = _inputs(c, seed)
    if f == "clouds":
        return _exact_clouds(c, d)
    if f == "pearson":
        return _exact_pearson(c, d["X"], None)
    if f == "pearson_list":
        return _exact_pearson(c, d["X"], d["pairs"])
    if f == "cosine":
        return _exact_cosine(c, d["csr"])
    cl = d["clouds"]
    pi, pj = d.get("pairs") or np.triu_indices(c["n"], 1)
    P = d["params"].double()
    if f == "align":
        cost, g = _cost_and_gradient(cl, pi, pj, P)
        return {"f": cost, "grad": g * d["grad"].double()[:, None]}
    flags = torch.zeros(len(pi), dtype=torch.int32, device="cuda")
    for _ in range(c["steps"]):
        cost, g = _cost_and_gradient(cl, pi, pj, P)
        up = cost >= FMIN
        P = torch.where(up[:, None], P + ETA * g / cost.clamp_min(FMIN)[:, None], P)
        flags |= (~up).to(torch.int32)
    return {"params": P, "f": cost, "flags": flags}
