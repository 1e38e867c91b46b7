"""GPU parity of the Gaussian overlap cost (2-D and 3-D point clouds) against
the FP64 oracle, through the C ABI."""
import numpy as np
import pytest

import synth
from gpu_util import check_overlap

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def ap():
    import paper_2009_04755_gb300 as ap
    ap.lib()
    return ap


def _gpu_overlap(ap, c, params=None):
    with ap.Items.from_clouds(c) as it:
        prm = None if params is None else torch.as_tensor(params, dtype=torch.float32).cuda()
        f = it.run_pairs(ap.AP_FN_OVERLAP, params=prm).cpu().numpy()
        assert it.last_device_error() == 0
    return f


def test_overlap_2d_n256_all_pairs(ap, oracle_lib):
    """256 2-D clouds of 64-128 points, every one of the 32,640 pairs."""
    c = synth.clouds_uniform(n=256, dim=2, size=(64, 128), seed=0)
    pi, pj = oracle_lib.all_pairs(256)
    ref, kappa, bound = oracle_lib.overlap(c, pi, pj, with_cond=True)
    f = _gpu_overlap(ap, c)
    assert f.shape == ref.shape
    check_overlap(f, ref, kappa, bound, "2d n256")


def test_overlap_3d_lognormal_sorted(ap, oracle_lib):
    # uneven sizes take the size-sorted plan; includes items far above one chunk
    c = synth.clouds_lognormal(n=160, dim=3, median=300, clip=(50, 3000), seed=5)
    pi, pj = oracle_lib.all_pairs(160)
    ref, kappa, bound = oracle_lib.overlap(c, pi, pj, with_cond=True)
    check_overlap(_gpu_overlap(ap, c), ref, kappa, bound, "3d lognormal")


@pytest.mark.parametrize("dim", [2, 3])
def test_overlap_weights_and_ragged(ap, oracle_lib, dim):
    rng = np.random.default_rng(dim)
    sizes = np.array([0, 1, 3, 4, 5, 33, 64, 65, 127, 128, 129, 200, 0, 7, 300, 2])
    c = synth.clouds_uniform(n=len(sizes), dim=dim, size=(1, 2), seed=dim)
    off = np.concatenate([[0], np.cumsum(sizes)]).astype(np.int64)
    tot = int(off[-1])
    pts = rng.uniform(-0.3, 0.3, (tot, 3)).astype(np.float32)
    c = {"dim": dim, "offsets": off, "x": pts[:, 0].copy(), "y": pts[:, 1].copy(),
         "z": pts[:, 2].copy() if dim == 3 else None,
         "sigma": rng.uniform(0.02, 0.08, tot).astype(np.float32),
         "weight": rng.uniform(0.0, 2.0, tot).astype(np.float32)}
    c["weight"][::7] = 0.0
    n = len(sizes)
    pi, pj = oracle_lib.all_pairs(n)
    ref, kappa, bound = oracle_lib.overlap(c, pi, pj, with_cond=True)
    f = _gpu_overlap(ap, c)
    # empty items give exactly 0
    empty = (sizes[pi] == 0) | (sizes[pj] == 0)
    assert np.all(f[empty] == 0.0)
    check_overlap(f[~empty], ref[~empty], kappa[~empty], bound[~empty], f"ragged {dim}d")


def test_overlap_with_transform(ap, oracle_lib):
    c = synth.clouds_templates(n=40, seed=4)
    pi, pj = oracle_lib.all_pairs(40)
    rng = np.random.default_rng(1)
    params = np.stack([rng.uniform(-np.pi, np.pi, len(pi)), rng.uniform(-0.3, 0.3, len(pi)),
                       rng.uniform(-0.3, 0.3, len(pi))], 1).astype(np.float32)
    ref, kappa, bound = oracle_lib.overlap(c, pi, pj, params=params.astype(np.float64),
                                           with_cond=True)
    check_overlap(_gpu_overlap(ap, c, params), ref, kappa, bound, "transform")


@pytest.mark.parametrize("dim,n", [(2, 256), (3, 500), (2, 3)])
def test_overlap_coverage_every_pair_once(ap, dim, n):
    c = (synth.clouds_lognormal(n=n, dim=3, clip=(50, 2000), seed=1) if dim == 3
         else synth.clouds_uniform(n=n, dim=2, seed=1))
    with ap.Items.from_clouds(c) as it:
        cnt = it.run_pairs(ap.AP_FN_COVERAGE).cpu().numpy()
    assert cnt.shape == (n * (n - 1) // 2,)
    assert np.all(cnt == 1)


def test_overlap_small_n(ap):
    for n in (0, 1):
        c = synth.clouds_uniform(n=max(n, 1), dim=2, seed=0)
        c["offsets"] = c["offsets"][:n + 1]
        with ap.Items.from_clouds(c) as it:
            assert it.run_pairs().numel() == 0


def test_overlap_symmetric_at_identity(ap):
    # f(i, j) computed with the roles swapped (reverse the item order)
    c = synth.clouds_uniform(n=30, dim=2, seed=3)
    f = _gpu_overlap(ap, c)
    n = 30
    off = c["offsets"]
    order = np.arange(n)[::-1]
    sizes = np.diff(off)[order]
    roff = np.concatenate([[0], np.cumsum(sizes)]).astype(np.int64)
    idx = np.concatenate([np.arange(off[k], off[k + 1]) for k in order])
    rc = {"dim": 2, "offsets": roff, "x": c["x"][idx], "y": c["y"][idx], "z": None,
          "sigma": c["sigma"][idx], "weight": c["weight"][idx]}
    g = _gpu_overlap(ap, rc)
    for i, j in [(0, 1), (3, 17), (28, 29), (0, 29)]:
        p = ap.pair_index(i, j, n)
        q = ap.pair_index(n - 1 - j, n - 1 - i, n)
        assert abs(f[p] - g[q]) <= 1e-5 * abs(f[p])


def test_clouds_created_on_a_side_stream_from_pinned_host(ap, oracle_lib):
    # creation copies and packs on the caller's stream: the pairs run on the
    # same stream with no host synchronisation in between
    c = synth.clouds_uniform(n=40, dim=2, size=(20, 60), seed=12)
    pi, pj = oracle_lib.all_pairs(40)
    ref, kappa, bound = oracle_lib.overlap(c, pi, pj, with_cond=True)
    s = torch.cuda.Stream()
    it = ap.Items.from_clouds(c, device="cpu", stream=s, sync=False)
    out = it.run_pairs(stream=s)
    s.synchronize()
    check_overlap(out.cpu().numpy(), ref, kappa, bound, "side stream")
    it.close()


def _edge_clouds(dim, scale=1.0, weights=False, sizes=None):
    """Sizes at the edges of a group of 4 points, a piece of 8 groups, a full
    warp of 4 points per lane and (the last) of the staging windows."""
    sizes = np.array(sizes or [1, 31, 32, 33, 36, 64, 65, 96, 127, 128, 129, 160, 161, 255, 257,
                               2047, 2049, 4101])
    off = np.concatenate([[0], np.cumsum(sizes)]).astype(np.int64)
    rng = np.random.default_rng(int(off[-1]) + dim)
    pts = rng.uniform(-0.3, 0.3, (int(off[-1]), 3)) * scale
    sig = rng.uniform(0.03, 0.08, int(off[-1])) * scale
    w = rng.uniform(0.5, 1.5, int(off[-1])) if weights else None
    f32 = np.float32
    return {"dim": dim, "offsets": off, "x": pts[:, 0].astype(f32), "y": pts[:, 1].astype(f32),
            "z": pts[:, 2].astype(f32) if dim == 3 else None, "sigma": sig.astype(f32),
            "weight": None if w is None else w.astype(f32)}


@pytest.mark.parametrize("dim", [2, 3])
@pytest.mark.parametrize("plan", [None, (4, 256, 2), (32, 8192, 4)])
@pytest.mark.parametrize("kind", ["unit", "weighted", "tiny", "huge"])
def test_overlap_fragment_and_window_edges(ap, oracle_lib, dim, plan, kind):
    """Unit weights and weights take their own loops; lengths of 1e-12 (whose
    s2k products leave the FP32 range) and coordinates of 1e16 the general
    one.  The cost does not depend on the unit of length, so the oracle sees
    the same set."""
    scale = {"tiny": 1e-12, "huge": 1e16}.get(kind, 1.0)
    c = _edge_clouds(dim, scale, kind == "weighted")
    n = len(c["offsets"]) - 1
    pi, pj = oracle_lib.all_pairs(n)
    ref, kappa, bound = oracle_lib.overlap(c, pi, pj, with_cond=True)
    with ap.Items.from_clouds(c) as it:
        if plan:
            it.set_plan(*plan)
        f = it.run_pairs().cpu().numpy()
        one = it.run_pairs_list(pi, pj).cpu().numpy()
        cnt = it.run_pairs(ap.AP_FN_COVERAGE).cpu().numpy()
        assert it.last_device_error() == 0
    check_overlap(f, ref, kappa, bound, f"{kind} {dim}d {plan}")
    assert np.all(cnt == 1)
    if dim == 2:
        # stored in item order: a listed pair sums the same fragments in the same order
        np.testing.assert_array_equal(one, f)
    else:
        check_overlap(one, ref, kappa, bound, f"listed {kind} {dim}d {plan}")


def _spread_clouds(dim, weights):
    """Items whose points reach a small part of their extent, around the sizes
    at which blocks of 32 points are passed over, with a coarse point in some."""
    sizes = np.array([1, 160, 161, 192, 900, 0, 1001, 2049, 2051, 4101])
    off = np.concatenate([[0], np.cumsum(sizes)]).astype(np.int64)
    rng = np.random.default_rng(50 + dim)
    tot = int(off[-1])
    pts = rng.uniform(-1, 1, (tot, 3)).astype(np.float32)
    pts[off[4]:off[5], 0] = 0.25                 # no extent along one axis
    sig = rng.uniform(0.01, 0.02, tot)
    sig[off[6]::97] = 0.3
    w = rng.uniform(0.0, 2.0, tot).astype(np.float32)
    w[::7] = 0.0
    return {"dim": dim, "offsets": off, "x": pts[:, 0].copy(), "y": pts[:, 1].copy(),
            "z": pts[:, 2].copy() if dim == 3 else None, "sigma": sig.astype(np.float32),
            "weight": w if weights else None}


@pytest.mark.parametrize("dim", [2, 3])
@pytest.mark.parametrize("weights", [False, True])
def test_overlap_passes_over_far_blocks(ap, oracle_lib, dim, weights):
    c = _spread_clouds(dim, weights)
    n = len(c["offsets"]) - 1
    pi, pj = oracle_lib.all_pairs(n)
    ref, kappa, bound = oracle_lib.overlap(c, pi, pj, with_cond=True)
    with ap.Items.from_clouds(c) as it:
        f = it.run_pairs().cpu().numpy()
        one = it.run_pairs_list(pi, pj).cpu().numpy()
        it.set_plan(4, 256, 2)                   # sweeps every block
        every = it.run_pairs().cpu().numpy()
        assert it.last_device_error() == 0
    check_overlap(f, ref, kappa, bound, f"blocks {dim}d")
    # a block passed over adds exactly nothing; pieces of another length are
    # summed in another order, in two floats, and rounded once
    np.testing.assert_array_max_ulp(every, f, maxulp=1)
    if dim == 2:
        np.testing.assert_array_equal(one, f)
    else:
        check_overlap(one, ref, kappa, bound, f"listed blocks {dim}d")


def test_far_blocks_under_transforms(ap, oracle_lib):
    """Transforms that keep the clouds together, part them for good, or are no
    numbers: the last give NaN for their own pair alone."""
    c = _spread_clouds(2, True)
    n = len(c["offsets"]) - 1
    pi, pj = oracle_lib.all_pairs(n)
    rng = np.random.default_rng(9)
    prm = rng.uniform(-0.5, 0.5, (len(pi), 3)).astype(np.float32)
    far = np.arange(len(pi)) % 5 == 1
    prm[far, 1] = 1e6
    ref, kappa, bound = oracle_lib.overlap(c, pi, pj, params=prm.astype(np.float64),
                                           with_cond=True)
    sizes = np.diff(c["offsets"])
    nan = (np.arange(len(pi)) % 5 == 2) & (sizes[pi] > 0) & (sizes[pj] > 0)
    prm[nan, 2] = np.nan
    with ap.Items.from_clouds(c) as it:
        p = torch.from_numpy(prm).cuda()
        f = it.run_pairs(params=p).cpu().numpy()
        g = it.backward(params=p)[0].cpu().numpy()
        it.set_plan(4, 256, 2)
        f2 = it.run_pairs(params=p).cpu().numpy()
        g2 = it.backward(params=p)[0].cpu().numpy()
        assert it.last_device_error() == 0
    ok = ~nan
    near = ok & ~far
    check_overlap(f[near], ref[near], kappa[near], bound[near], "blocks, transforms")
    assert np.all(f[far & ok] == 0) and np.isnan(f[nan]).all()
    np.testing.assert_array_max_ulp(f2[ok], f[ok], maxulp=1)
    # the sums are the same but for their order over a warp's lanes
    scale = np.abs(g2[ok]).max()
    np.testing.assert_allclose(g[ok], g2[ok], rtol=1e-4, atol=1e-6 * scale)


@pytest.mark.parametrize("plan", [None, (4, 256, 2)])     # with boxes and without
def test_clouds_moved_onto_the_padding(ap, plan):
    """Unit weights, odd sizes: a pair parked far away by its transform has no
    term with the points that fill its partner's storage up (x = 1e18, with
    whose x these translations coincide), whichever call asks."""
    sizes = np.array([1, 3, 5, 33, 129, 161, 1001, 2049])
    off = np.concatenate([[0], np.cumsum(sizes)]).astype(np.int64)
    rng = np.random.default_rng(3)
    pts = rng.uniform(-0.3, 0.3, (2, int(off[-1]))).astype(np.float32)
    c = {"dim": 2, "offsets": off, "x": pts[0], "y": pts[1], "z": None, "weight": None,
         "sigma": rng.uniform(0.2, 0.4, int(off[-1])).astype(np.float32)}
    n = len(sizes)
    pi, pj = np.triu_indices(n, 1)
    away = torch.zeros(len(pi), 3, device="cuda")
    away[:, 1] = 1e18                            # moved points at x = -1e18: nothing there
    onto = torch.zeros(len(pi), 3, device="cuda")
    onto[:, 1] = -torch.linspace(0.4e18, 1.6e18, len(pi), device="cuda")
    onto[::2, 1] = -1e18
    with ap.Items.from_clouds(c) as it:
        if plan:
            it.set_plan(*plan)
        assert torch.all(it.run_pairs(params=onto) == 0)
        assert torch.all(it.run_pairs_list(pi, pj, params=onto) == 0)
        assert torch.equal(it.run_pairs(ap.AP_FN_GMM_L2, params=onto),
                           it.run_pairs(ap.AP_FN_GMM_L2, params=away))
        assert torch.all(it.run_pairs(ap.AP_FN_BHATTACHARYYA, params=onto) == 0)
        for g, f in (it.backward(params=onto), it.backward_list(pi, pj, params=onto)):
            assert torch.all(f == 0) and torch.all(g == 0)
        p, f, flags = it.ascent(onto.clone(), 3, 1e-2)
        assert torch.all(f == 0) and torch.all(flags == 1) and torch.equal(p, onto)
        assert it.last_device_error() == 0


@pytest.mark.parametrize("n,items,tiles", [(700, 8, 8000), (1200, 16, 12_000), (5000, 32, 32_000)])
def test_tiles_of_many_small_clouds(ap, n, items, tiles):
    """Blocks take more items as sets of small clouds grow, so that the list
    of tiles grows with the pairs' work and not with the square of the eighths."""
    c = synth.clouds_uniform(n=n, dim=2, size=(2, 6), seed=n)
    with ap.Items.from_clouds(c) as it:
        assert it.plan()["block_items"] == items and it.stats()["tiles"] < tiles
        assert torch.all(it.run_pairs(ap.AP_FN_COVERAGE) == 1)
        f = it.run_pairs()
        it.set_plan(8, 384, 4)
        assert torch.equal(it.run_pairs(), f)


@pytest.mark.parametrize("dim", [2, 3])
def test_sums_beyond_the_fp32_range_are_infinite(ap, dim):
    """Weights whose products leave the range: infinity for the pairs that hold
    two of them, whatever way the sums go, and numbers for the others."""
    sizes = np.array([1, 2, 30, 200, 1500, 3, 40, 160])
    off = np.concatenate([[0], np.cumsum(sizes)]).astype(np.int64)
    rng = np.random.default_rng(8)
    pts = rng.uniform(-0.01, 0.01, (3, int(off[-1]))).astype(np.float32)
    w = np.ones(int(off[-1]), np.float32)
    heavy = [0, 2, 3, 4]
    w[off[heavy]] = 1e30
    c = {"dim": dim, "offsets": off, "x": pts[0], "y": pts[1], "z": pts[2] if dim == 3 else None,
         "sigma": np.full(int(off[-1]), 0.5, np.float32), "weight": w}
    pi, pj = np.triu_indices(len(sizes), 1)
    both = torch.from_numpy(np.isin(pi, heavy) & np.isin(pj, heavy)).cuda()
    with ap.Items.from_clouds(c) as it:
        fs = [it.run_pairs(), it.run_pairs_list(pi, pj)]
        if dim == 2:
            zero = torch.zeros(len(pi), 3, device="cuda")
            fs += [it.run_pairs(params=zero), it.backward(zero)[1]]
        it.set_plan(4, 256, 2)
        fs.append(it.run_pairs())
        for f in fs:
            assert torch.all(torch.isposinf(f[both])) and torch.all(torch.isfinite(f[~both]))
