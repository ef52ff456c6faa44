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



# more hit points than the calls whose lists a team of warps shares (152 * 32
# tiles of 32); all but a few are not valid
MANY = 32 * 152 * 32 + 7


def _forward(gpf, fnp, x, split, r, **grid):
    """(out, z) at the points x, the only valid ones of MANY."""
    from paper_2512_12459_gb300.setup_index import make_index
    qnp = _points(np.concatenate([x, np.full((MANY - len(x), 3), 0.5)]))
    qnp.valid[len(x):] = 0
    field, queries = gpf.Field.from_numpy(fnp), gpf.Queries.from_numpy(qnp)
    g = gpf.grid_for_bounds([0.0] * 3, [1.0] * 3, 1.0 / 1024, fnp.channels, fnp.n, MANY, 100_000,
                            **grid)
    idx = make_index(field, queries, grid=g, split_items=split)
    idx.build(field, queries)
    assert idx.stats()["flags"] == 0
    out, z = gpf.gpf_radiance_fwd(idx, field, queries, gpf.GPF_SUM, r_max=r)
    assert not out[:, len(x):].any()
    return out[:, :len(x)].cpu().numpy(), z[:len(x)].cpu().numpy()


def _parts(items, split):
    return min(64, -(-items // split)) if split and items > split else 1


def _walked(lists, parts):
    """The sum over lists of columns, each level's one list: a part takes every
    parts-th chunk of 32 of every list, in list order."""
    total = np.zeros(lists[0].shape[0], np.float32)
    for p in range(parts):
        s, chunk = np.zeros_like(total), 0
        for v in lists:
            for i in range(0, v.shape[1], 32):
                if chunk % parts == p:
                    for k in range(i, min(i + 32, v.shape[1])):
                        s = s + v[:, k]
                chunk += 1
        total = total + s
    return total


def _pooled(levels, parts, channels):
    """[channels, 32]: the sums over each hit point's own lists. A level's lists
    are laid end to end and taken 32 items at a time, one per lane; a lane hands
    its sum over when its item's hit point or the level changes."""
    total = np.zeros((channels, 32), np.float32)
    for p in range(parts):
        acc, chunk = np.zeros((channels, 32), np.float32), 0
        for lists in levels:
            own = np.repeat(np.arange(32), [v.shape[1] for v in lists])
            val = np.concatenate(lists, axis=1)
            cur, pc = np.full(32, -1), np.zeros((channels, 32), np.float32)

            def flush(f):
                key = np.where(f, cur, 64 + np.arange(32))
                t = np.where(f, pc, np.float32(0))
                for d in (1, 2, 4, 8, 16):
                    same = np.zeros(32, bool)
                    same[d:] = key[d:] == key[:-d]
                    u = np.zeros_like(t)
                    u[:, d:] = t[:, :-d]
                    t = np.where(same, t + u, t)
                for lane in range(32):
                    if f[lane] and (lane == 31 or key[lane + 1] != key[lane]):
                        acc[:, key[lane]] += t[:, lane]
                pc[:, f] = 0

            for i in range(0, len(own), 32):
                if chunk % parts == p:
                    o = np.full(32, 32)
                    o[:len(own[i:i + 32])] = own[i:i + 32]
                    if (o != cur).any():
                        flush((o != cur) & (cur >= 0) & (cur < 32))
                        cur = o
                    for lane in np.flatnonzero(o < 32):
                        pc[:, lane] += val[:, i + lane]
                chunk += 1
            flush((cur >= 0) & (cur < 32))
        total = total + acc
    return total


SMALL, MIDDLE = 1e-4, 1.5e-3        # scales whose levels hold nothing else


@pytest.mark.parametrize("channels", [1, 3, 8])
@pytest.mark.parametrize("n", [1, 31, 33, 1000])
@pytest.mark.parametrize("split", [0, 64, 4096])
def test_walked_lists_are_summed_in_list_order(gpf, channels, n, split):
    rng = np.random.default_rng(n)
    at = np.array([[0.5 + 0.5 / 1024] * 3])
    kind = rng.integers(0, 2, n)
    fnp = _field(np.repeat(at, n, axis=0), np.where(kind, SMALL, MIDDLE), channels, n)
    lists = [fnp.spectrum[:, kind == 1], fnp.spectrum[:, kind == 0]]
    parts = _parts(8 * n, split)
    out, z = _forward(gpf, fnp, np.repeat(at, 41, axis=0), split, math.inf, levels=6,
                      query_level=3)
    assert (z == n).all()
    ref = _walked(lists, parts)
    for k in range(out.shape[1]):
        np.testing.assert_array_equal(out[:, k], ref)


@pytest.mark.parametrize("channels", [1, 3, 8])
@pytest.mark.parametrize("most", [3, 70])
@pytest.mark.parametrize("split", [0, 64, 4096])
@pytest.mark.parametrize("r", [math.inf, 0.02])
def test_pooled_lists_are_summed_over_the_lanes(gpf, channels, most, split, r):
    rng = np.random.default_rng(most)
    x = np.full((32, 3), 0.5 + 0.5 / 1024)
    x[:, 0] = (32 * np.arange(32) + 0.5) / 1024
    counts = rng.integers(0, most, (2, 32))
    at = np.repeat(np.tile(np.arange(32), 2), counts.ravel())
    kind = np.repeat(np.repeat([1, 0], 32), counts.ravel())
    order = rng.permutation(len(at))
    at, kind = at[order], kind[order]
    fnp = _field(x[at], np.where(kind, SMALL, MIDDLE), channels, most)
    levels = [[fnp.spectrum[:, (at == o) & (kind == k)] for o in range(32)] for k in (1, 0)]
    parts = _parts(4 * int(counts[:, ::4].sum()), split)
    out, z = _forward(gpf, fnp, x, split, r, levels=6, query_level=3, hash_bits=24)
    assert (z == counts.sum(0)).all()
    np.testing.assert_array_equal(out, _pooled(levels, parts, channels))
