"""GPU checks of the tile-plan autotuner and of the ascent's CUDA graph: any
plan the tuner can pick gives results within tolerance of the oracle, replays
and repeated launches are bit-identical, and explicit plans round-trip."""
import numpy as np
import pytest

import synth
from gpu_util import check_grad, check_overlap, cloud_wsum

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def ap():
    import paper_2009_04755_gb300 as ap
    ap.lib()
    return ap


def test_tune_then_parity_2d(ap, oracle_lib):
    c = synth.clouds_uniform(n=256, dim=2, size=(64, 128), seed=0)
    pi, pj = oracle_lib.all_pairs(256)
    ref, kappa, bound = oracle_lib.overlap(c, pi, pj, with_cond=True)
    with ap.Items.from_clouds(c) as it:
        plan = it.tune(0)
        assert plan["rate"] > 0
        assert plan["block_items"] in (2, 4, 8, 16, 32)
        assert plan["block_pts"] in (2048, 4096, 8192)
        assert plan["reg_r"] in (2, 4)
        assert it.plan()["block_items"] == plan["block_items"]
        f1 = it.run_pairs().cpu().numpy()
        f2 = it.run_pairs().cpu().numpy()
    check_overlap(f1, ref, kappa, bound, "tuned 2d")
    assert np.array_equal(f1, f2)


@pytest.mark.parametrize("bi,bp,rr", [(2, 2048, 2), (32, 8192, 4), (5, 100, 2), (1, 64, 4)])
def test_every_plan_is_correct_3d(ap, oracle_lib, bi, bp, rr):
    c = synth.clouds_lognormal(n=120, dim=3, median=200, clip=(50, 1500), seed=9)
    pi, pj = oracle_lib.all_pairs(120)
    ref, kappa, bound = oracle_lib.overlap(c, pi, pj, with_cond=True)
    with ap.Items.from_clouds(c) as it:
        it.set_plan(bi, bp, rr)
        f = it.run_pairs().cpu().numpy()
        cnt = it.run_pairs(ap.AP_FN_COVERAGE).cpu().numpy()
    check_overlap(f, ref, kappa, bound, f"plan {bi}/{bp}/{rr}")
    assert np.all(cnt == 1)


def test_set_plan_rejects(ap):
    c = synth.clouds_uniform(n=20, dim=2, seed=1)
    with ap.Items.from_clouds(c) as it:
        for bad in [(0, 4096, 2), (33, 4096, 2), (4, 32, 2), (4, 9000, 2), (4, 4096, 3), (4, 4096, 1)]:
            with pytest.raises(ap.APError):
                it.set_plan(*bad)


def test_tune_adjoint_then_ascent(ap, oracle_lib):
    n = 40
    c = synth.clouds_templates(n=n, seed=21)
    pi, pj = oracle_lib.all_pairs(n)
    with ap.Items.from_clouds(c) as it:
        plan = it.tune(1)
        assert plan["rate"] > 0
        g, f = it.backward(params=None)
        p = torch.zeros(len(pi), 3, device="cuda")
        p1, f1, _ = it.ascent(p.clone(), 4, 1e-3)
        p2, f2, _ = it.ascent(p.clone(), 4, 1e-3)   # second call replays the graph
        assert torch.equal(p1, p2) and torch.equal(f1, f2)
    f_ref, g_ref = oracle_lib.overlap_grad(c, pi, pj, None)
    check_grad(g.cpu().numpy(), g_ref, cloud_wsum(c, pi, pj))


def test_graph_replay_respects_new_buffers(ap):
    c = synth.clouds_uniform(n=64, dim=2, seed=2)
    with ap.Items.from_clouds(c) as it:
        a = it.run_pairs().clone()
        out = torch.zeros_like(a)
        it.run_pairs(out=out)                     # a new output buffer
        assert torch.equal(a, out)
        first, second = (torch.zeros(len(a), 3, device="cuda") for _ in range(2))
        p1, f1, _ = it.ascent(first, 3, 1e-3)     # captured for these buffers
        p2, f2, _ = it.ascent(second, 3, 1e-3)    # other parameters: another graph
        assert torch.equal(p1, p2) and torch.equal(f1, f2) and p1 is first and p2 is second
        assert bool((first != 0).any())
        it.set_plan(4, 2048, 2)                   # a new plan invalidates the graphs
        b = it.run_pairs()
        assert torch.allclose(a, b, rtol=1e-5, atol=0)
        p3, f3, _ = it.ascent(first.zero_(), 3, 1e-3)
        torch.testing.assert_close(p3, p2, rtol=1e-4, atol=1e-6)
        torch.testing.assert_close(f3, f2, rtol=1e-5, atol=0)


def test_handles_of_one_kernel_keep_their_launch_shapes(ap):
    """Two sets run by the same kernel with different amounts of shared
    memory, in turn: neither run changes what the other may use."""
    big = synth.clouds_uniform(n=12, dim=2, size=(900, 2000), seed=1)
    small = synth.clouds_uniform(n=12, dim=2, size=(5, 9), seed=2)
    with ap.Items.from_clouds(big) as a, ap.Items.from_clouds(small) as b:
        fa, fb = a.run_pairs().clone(), b.run_pairs().clone()
        for _ in range(2):
            assert torch.equal(a.run_pairs(), fa) and torch.equal(b.run_pairs(), fb)
            assert a.run_pairs_list([0, 3], [1, 5]).shape == (2,)


def test_new_plans_are_there_for_every_stream(ap):
    """A run on a side stream straight after set_plan, tune or a list's first
    call, with nothing that waits in between: plans of megabytes, whose copies
    take longer than the launch."""
    rng = np.random.default_rng(4)
    sizes = rng.integers(3, 12, 2500)
    off = np.concatenate([[0], np.cumsum(sizes)]).astype(np.int64)
    pts = rng.uniform(-1, 1, (2, int(off[-1]))).astype(np.float32)
    c = {"dim": 2, "offsets": off, "x": pts[0], "y": pts[1], "z": None, "weight": None,
         "sigma": rng.uniform(0.1, 0.2, int(off[-1])).astype(np.float32)}
    side = torch.cuda.Stream()
    pi, pj = np.triu_indices(400, 1)
    with ap.Items.from_clouds(c) as it:
        ref = it.run_pairs()
        one = it.run_pairs_list(pi, pj)
        out, few = torch.zeros_like(ref), torch.zeros_like(one)
        torch.cuda.synchronize()
        for plan in [(8, 384, 4), (2, 64, 4), (32, 2048, 4), (3, 8192, 4)] * 3:
            it.set_plan(*plan)
            it.run_pairs(out=out, stream=side)
            side.synchronize()
            assert torch.equal(out, ref), plan
            it.set_plan(plan[0], plan[1], 2)      # other one-item blocks
            it.run_pairs_list(pi[::2], pj[::2], out=few[:len(pi[::2])], stream=side)
            it.run_pairs_list(pi, pj, out=few, stream=side)
            side.synchronize()
            torch.testing.assert_close(few, one, rtol=1e-6, atol=0)
        it.tune(0, stream=side)
        it.run_pairs(out=out)
        torch.testing.assert_close(out, ref, rtol=1e-6, atol=0)
        assert it.last_device_error() == 0


def test_runs_that_overlap_spoil_no_later_run(ap):
    """Runs of one handle on two streams at once, of unequal numbers of tiles
    (which programs should not do: the header says so): later runs are whole,
    more of them than there are queue heads, and so is a replayed capture."""
    c = synth.clouds_uniform(n=150, dim=2, size=(5, 60), seed=6)
    pi, pj = np.triu_indices(150, 1)
    a, b = torch.cuda.Stream(), torch.cuda.Stream()
    with ap.Items.from_clouds(c) as it:
        ref = it.run_pairs()
        one, x, y = torch.empty_like(ref), torch.empty_like(ref), torch.zeros_like(ref)
        torch.cuda.synchronize()
        for _ in range(40):
            it.run_pairs(out=x, stream=a)
            it.run_pairs(out=y, stream=b)
            it.run_pairs_list(pi[:777], pj[:777], out=one, stream=b)
            it.run_pairs(out=x, stream=a)
        torch.cuda.synchronize()
        for _ in range(150):
            x.zero_()
            it.run_pairs(out=x)
            assert torch.equal(x, ref)
        p0 = torch.zeros(len(pi), 3, device="cuda")
        p1, f1, _ = it.ascent(p0.clone(), 5, 1e-3)
        p2, f2 = p0.clone(), None
        for _ in range(5):                       # odd numbers of steps: the heads alternate
            p2, f2, _ = it.ascent(p2, 1, 1e-3)
        assert torch.equal(p1, p2) and torch.equal(f1, f2)
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g):
            it.run_pairs(out=x)
            it.run_pairs(out=y)
        for _ in range(3):
            x.zero_(), y.zero_()
            g.replay()
            assert torch.equal(x, ref) and torch.equal(y, ref)
        assert it.last_device_error() == 0
