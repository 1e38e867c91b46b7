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
