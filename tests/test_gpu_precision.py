"""How far the cloud costs are from 64 bits: the sums keep what a plain FP32
evaluation in the order of the points gives, whichever way a set is swept."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def ap():
    import paper_2009_04755_gb300 as ap
    ap.lib()
    return ap


def _clouds(sizes, dim, seed, box, sigma, weights=False):
    rng = np.random.default_rng(seed)
    off = np.concatenate([[0], np.cumsum(sizes)]).astype(np.int64)
    m = int(off[-1])

    def u(lo, hi):
        return rng.uniform(lo, hi, m).astype(np.float32)

    return {"dim": dim, "offsets": off, "x": u(-box, box), "y": u(-box, box),
            "z": u(-box, box) if dim == 3 else None, "sigma": u(*sigma),
            "weight": u(0.25, 1.75) if weights else None}


@pytest.mark.parametrize("dim", [2, 3])
@pytest.mark.parametrize("weights", [False, True])
def test_few_points_take_a_reciprocal_each(ap, dim, weights):
    """Against partners of up to 8 points no two terms share a reciprocal: the
    bits of a set with a far point in it, where none do."""
    sizes = np.array([1, 2, 3, 7, 8, 9, 40, 200] * 6)
    c = _clouds(sizes, dim, 1, 0.08, (0.02, 0.05), weights)
    far = {k: v if v is None or k in ("dim", "offsets") else
           np.concatenate([v, np.float32([0.5 if k == "sigma" else 1.0])])
           for k, v in c.items()}
    far["offsets"] = np.concatenate([c["offsets"], c["offsets"][-1:] + 1])
    far["x"][-1] = 1e16
    n = len(sizes)
    pi, pj = np.triu_indices(n, 1)
    with ap.Items.from_clouds(c) as a, ap.Items.from_clouds(far) as b:
        f, g = a.run_pairs_list(pi, pj), b.run_pairs_list(pi, pj)
    few = torch.from_numpy((sizes[pi] <= 8) & (sizes[pj] <= 8)).cuda()
    many = torch.from_numpy((sizes[pi] > 8) & (sizes[pj] > 8)).cuda()
    assert torch.equal(f[few], g[few]) and not torch.equal(f[many], g[many])


def _pairs64(c, fn):
    """The cost of every pair (no transforms) in 64 bits, plain torch."""
    off, dim = c["offsets"], c["dim"]
    n = len(off) - 1
    x = torch.stack([torch.from_numpy(c[k]).cuda().double() for k in "xyz"[:dim]], 1)
    s = torch.from_numpy(c["sigma"]).cuda().double()
    w = torch.ones_like(s) if c["weight"] is None else torch.from_numpy(c["weight"]).cuda().double()
    item = torch.repeat_interleave(torch.arange(n, device="cuda"),
                                   torch.from_numpy(np.diff(off)).cuda())
    out = torch.zeros(n, n, dtype=torch.float64, device="cuda")
    for i in range(n - 1):
        a = slice(int(off[i]), int(off[i + 1]))
        for b0 in range(int(off[i + 1]), len(s), 1 << 16):
            b = slice(b0, min(len(s), b0 + (1 << 16)))
            s2 = s[a, None] ** 2 + s[b][None] ** 2
            d2 = sum((x[a, k][:, None] - x[b, k][None]) ** 2 for k in range(dim))
            if fn == "overlap":
                t = torch.exp(-d2 / (2 * s2)) * w[a, None] * w[b][None]
            else:
                t = ((2 * s[a, None] * s[b][None] / s2) ** (dim / 2) * torch.exp(-d2 / (4 * s2))
                     * (w[a, None] * w[b][None]).sqrt())
            out[i].index_add_(0, item[b], t.sum(0))
    pi, pj = torch.triu_indices(n, n, 1, device="cuda")
    return out[pi, pj]


def _off(f, ref):
    f = f.double()
    return (float((f - ref).norm() / ref.norm()),                 # in the 2-norm
            float(((f - ref) / ref).pow(2).mean().sqrt()))        # relative, rms


@pytest.mark.parametrize("dim", [2, 3])
@pytest.mark.parametrize("weights", [False, True])
def test_bhattacharyya_log_weights_are_rounded_once(ap, dim, weights):
    """A term's two log-weights carry one rounding each of an ulp of theirs
    (uniform: 12^-0.5 of it rms), times ln 2, beside the terms' own 1e-7."""
    c = _clouds(np.full(60, 100), dim, 2, 0.1, (0.02, 0.05), weights)
    with ap.Items.from_clouds(c) as it:
        f = it.run_pairs(ap.AP_FN_BHATTACHARYYA)
    l = 0.25 * dim * np.log2(c["sigma"].astype(np.float64) ** 2)
    ulp = 2.0 ** (np.floor(np.log2(np.abs(l).max())) - 23)
    bound = np.log(2) * np.sqrt(2.0) * ulp / np.sqrt(12.0) + 1e-7
    assert _off(f, _pairs64(c, "bhattacharyya"))[1] < bound


def _pose64(c, params):
    """f and df/d(theta, tx, ty) of every pair under its transform, 64 bits."""
    off, P = c["offsets"], params.double()
    n = len(off) - 1
    x, y, s = (torch.from_numpy(c[k]).cuda().double() for k in ("x", "y", "sigma"))
    f, g = [], []
    for p, (i, j) in enumerate(zip(*np.triu_indices(n, 1))):
        a, b = slice(int(off[i]), int(off[i + 1])), slice(int(off[j]), int(off[j + 1]))
        co, si = torch.cos(P[p, 0]), torch.sin(P[p, 0])
        rx, ry = co * x[b] - si * y[b], si * x[b] + co * y[b]
        dx, dy = x[a, None] - (rx + P[p, 1])[None], y[a, None] - (ry + P[p, 2])[None]
        s2 = s[a, None] ** 2 + s[b][None] ** 2
        e = torch.exp(-(dx * dx + dy * dy) / (2 * s2))
        gx, gy = (e / s2 * dx).sum(0), (e / s2 * dy).sum(0)
        f.append(e.sum())
        g.append(torch.stack([(gy * rx - gx * ry).sum(), gx.sum(), gy.sum()]))
    return torch.stack(f), torch.stack(g)


def test_adjoint_cost_is_as_close_as_the_cost(ap):
    """The adjoint's f sums 32 points in FP32 (five roundings, each of its
    level's share: 0.6 of a last one's 2^-24 / 3^0.5, beside the 5.6e-8 of the
    terms and of the result) and what follows in two floats."""
    c = _clouds(np.full(48, 150), 2, 3, 0.5, (0.02, 0.05))
    params = torch.randn(48 * 47 // 2, 3, generator=torch.Generator("cuda").manual_seed(3),
                         device="cuda") * 0.1
    with ap.Items.from_clouds(c) as it:
        f = it.run_pairs(params=params)
        _, fb = it.backward(params=params)
    ref, _ = _pose64(c, params)
    assert _off(fb, ref)[1] < np.hypot(_off(f, ref)[1], 0.6 * 2.0 ** -24 / np.sqrt(3.0))


@pytest.mark.parametrize("points", [1000, 1500])
def test_gradient_of_large_clouds_is_summed_by_blocks(ap, points):
    """Stored neighbour by neighbour, large clouds give a point terms of one
    sign in a row: their sum goes no further off than with the points as given
    (1.7e-7 in the 2-norm, FP32 sums over 1000 to 1500 terms that cancel)."""
    c = _clouds(np.full(24, points), 2, points, 0.5, (0.02, 0.05))
    params = torch.randn(24 * 23 // 2, 3, generator=torch.Generator("cuda").manual_seed(points),
                         device="cuda") * 0.1
    with ap.Items.from_clouds(c) as it:
        g, _ = it.backward(params=params)
    _, ref = _pose64(c, params)
    assert float((g.double() - ref).norm() / ref.norm()) < 1.7e-7


@pytest.mark.parametrize("dim,seed,bound", [(3, 20, 5.45e-8),   # points as given: 5.37e-8
                                            (3, 16, 5.6e-8),    # 5.43e-8
                                            (2, 12, 4.9e-8)])   # 4.82e-8
def test_cost_of_large_clouds_is_summed_two_by_two(ap, dim, seed, bound):
    """Stored neighbour by neighbour, the terms of large clouds are no further
    off than with the points as given (the 2-norm weighs the largest pairs, so
    a set differs from the next by a few per cent: sets and bounds as measured,
    where single sums gave 5.97e-8, 5.84e-8 and 4.95e-8)."""
    rng = np.random.default_rng(seed)
    sizes = np.exp(np.log(np.sqrt(50 * 5000) * 0.6) + rng.standard_normal(150))
    c = _clouds(np.clip(np.rint(sizes), 50, 5000).astype(np.int64), dim, seed, 1.0, (0.01, 0.05))
    with ap.Items.from_clouds(c) as it:
        assert _off(it.run_pairs(), _pairs64(c, "overlap"))[0] < bound


@pytest.mark.parametrize("dim", [2, 3])
@pytest.mark.parametrize("weights", [False, True])
def test_boxed_items_of_every_remainder(ap, dim, weights):
    """The last pairs of an item: remainders of 4 points, of blocks of 16 and 32
    and of the staging windows, with padding points among them."""
    sizes = np.array([1601, 1602, 1603, 1604, 1615, 1616, 1617, 1633, 1634, 2050, 2063, 4098, 6, 161])
    c = _clouds(sizes, dim, 7, 0.5, (0.05, 0.1), weights)
    ref = _pairs64(c, "overlap")
    with ap.Items.from_clouds(c) as it:
        f = it.run_pairs()
        assert it.last_device_error() == 0
    assert float(((f.double() - ref) / ref).abs().max()) < 1e-6
