"""The order in which the pair loops add up, bit for bit.

A training run feeds its own results back: a pair whose Q lies within rounding
of k^2 enters or leaves with a weight of e^(-k^2/2), so another order of the
same sum - a last bit of a mean - can move single gradients of the next step by
a hundredth. The order is therefore part of what the library returns. Here
every pair has the weight 1 (hit points at the means: Q = 0), so the sums are
plain float32 sums that numpy takes in the stated order."""

import math

import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def gpf():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2512_12459_gb300 as g
    return g


def _points(x):
    m = len(x)
    up = np.tile(np.array([[0.0], [0.0], [1.0]]), (1, m)).astype(np.float32)
    return synth.Queries(x=np.ascontiguousarray(np.asarray(x, np.float32).T), n=up, wo=up.copy(),
                         valid=np.ones(m, np.uint8))


def _field(mean, scale, channels, seed):
    n = len(mean)
    rng = np.random.default_rng(seed)
    f, _ = synth.config1_random(seed=seed, n=n, m=1, channels=channels)
    f.mean = np.ascontiguousarray(np.asarray(mean, np.float32).T)
    f.logscale = np.broadcast_to(np.log(np.asarray(scale, np.float64)), (3, n)).astype(
        np.float32).copy()
    f.spectrum = rng.standard_normal((channels, n)).astype(np.float32)
    return f


def _in_turn(v):
    """The float32 sum of the columns of v, one after the other."""
    return np.add.accumulate(v, axis=1, dtype=np.float32)[:, -1]


def _over_lanes(v):
    """Column i to lane i mod 32, each lane in turn; then the lanes' sums by
    halving exchanges."""
    lanes = np.zeros((v.shape[0], 32), np.float32)
    for i in range(0, v.shape[1], 32):
        part = v[:, i:i + 32]
        lanes[:, :part.shape[1]] += part
    for o in (16, 8, 4, 2, 1):
        lanes = lanes + lanes[:, np.arange(32) ^ o]
    return lanes[:, 0]


CENTRES = np.array([[0.25, 0.25, 0.25], [0.75, 0.25, 0.25], [0.25, 0.75, 0.25],
                    [0.5, 0.5, 0.75], [0.75, 0.75, 0.75]])
COUNTS = [1, 2, 33, 301, 1000]


@pytest.mark.parametrize("channels", [1, 3, 4, 8])
@pytest.mark.parametrize("r", [math.inf, 0.02])
def test_a_small_gaussians_sums_take_its_hit_points_in_turn(gpf, channels, r):
    """A Gaussian within 2 x 2 x 2 query-level cells: one lane, hit points in
    sorted order, whatever their number."""
    import torch
    from paper_2512_12459_gb300.setup_index import make_index
    rng = np.random.default_rng(channels)
    at = rng.permutation(np.repeat(np.arange(5), COUNTS))
    fnp = _field(CENTRES, 1e-3, channels, 3)
    field, queries = gpf.Field.from_numpy(fnp), gpf.Queries.from_numpy(_points(CENTRES[at]))
    idx = make_index(field, queries, query_cell=0.1)
    idx.build(field, queries)
    assert idx.stats()["n_small"] == 5
    G = rng.standard_normal((channels, len(at))).astype(np.float32)
    g = gpf.gpf_radiance_bwd(idx, field, queries, torch.from_numpy(G).cuda(), mode=gpf.GPF_SUM,
                             r_max=r)
    for c in range(5):
        np.testing.assert_array_equal(g.spectrum[:, c].cpu().numpy(), _in_turn(G[:, at == c]))


@pytest.mark.parametrize("channels", [1, 3, 4, 8])
@pytest.mark.parametrize("count", COUNTS)
@pytest.mark.parametrize("cell", [0.1, 0.02])
def test_a_large_gaussians_sums_take_its_hit_points_over_the_lanes(gpf, channels, count, cell):
    """A Gaussian over more cells: a warp, hit point i of a block of 32 rows to
    lane i mod 32; on the fine grid its rows are split into parts."""
    import torch
    from paper_2512_12459_gb300.setup_index import make_index
    rng = np.random.default_rng(count)
    x = np.full((count, 3), 0.5)
    corners = np.array([[0.0] * 3, [1.0] * 3])     # they set the grid's extent only
    fnp = _field(np.concatenate([x[:1], corners]), [0.1, 1e-3, 1e-3], channels, 3)
    field, queries = gpf.Field.from_numpy(fnp), gpf.Queries.from_numpy(_points(x))
    idx = make_index(field, queries, query_cell=cell)
    idx.build(field, queries)
    assert idx.stats()["n_live"] == 1 and idx.stats()["n_small"] == 0
    G = rng.standard_normal((channels, count)).astype(np.float32)
    g = gpf.gpf_radiance_bwd(idx, field, queries, torch.from_numpy(G).cuda(), mode=gpf.GPF_SUM)
    np.testing.assert_array_equal(g.spectrum[:, 0].cpu().numpy(), _over_lanes(G))

