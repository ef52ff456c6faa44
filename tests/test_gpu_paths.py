"""The branches that a size, a box or a value selects inside the build and the
pair loops, each against the brute-force path or the float64 build of the same
library: teams of warps per tile, boxes of more cells than the occupancy mask
holds, fields on either side of the small-group limit, hit points that fill a
cell with odd counts between empty ones, tiles longer than their samples say,
upstream gradients that are not finite, and a centre grid too large for its
fine occupancy bits."""

import math

import numpy as np
import pytest

import oracle
import synth
from gpu_helpers import GRAD_TOL

pytestmark = pytest.mark.gpu

# two float32 sums of the same positive terms, at most 2000 of them, in
# different orders: below 2000 * 2^-24 apart relative to the sum
SUM_RTOL = 1.2e-4
KEYS = ("mean", "quat", "logscale", "spectrum")


@pytest.fixture(scope="module")
def gpf():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2512_12459_gb300 as g
    return g


def _both(gpf, fnp, qnp, mode, r, **kw):
    """(out, z, counts) on a grid and by brute force."""
    from paper_2512_12459_gb300.setup_index import make_index
    field, queries = gpf.Field.from_numpy(fnp), gpf.Queries.from_numpy(qnp)
    res = []
    for k in (kw, {"brute_force": True}):
        idx = make_index(field, queries, cutoff_sigma=3.0, **k)
        idx.build(field, queries)
        out, z = gpf.gpf_radiance_fwd(idx, field, queries, mode, r_max=r)
        res.append((out.cpu().numpy(), z.cpu().numpy(),
                    gpf.gpf_count_pairs(idx, field, queries)["included"], idx))
    return field, queries, res


@pytest.mark.parametrize("m", [1, 33, 32 * 152 * 8, 32 * 152 * 8 + 1, 32 * 152 * 32 + 65])
@pytest.mark.parametrize("split", [0, 64])
def test_teams_of_warps_sum_the_same_pairs(gpf, m, split):
    fnp, qnp = synth.config1_random(seed=m % 1000, n=150, m=m, albedo=True)
    _, _, ((o, z, c, _), (ob, zb, cb, _)) = _both(gpf, fnp, qnp, gpf.GPF_SUM, 0.1,
                                                  query_cell=0.1, split_items=split)
    assert c == cb
    np.testing.assert_allclose(z, zb, rtol=SUM_RTOL, atol=1e-30)
    np.testing.assert_allclose(o, ob, rtol=SUM_RTOL, atol=1e-30)


@pytest.mark.parametrize("n", [2**17, 2**19 - 1, 2**19, 2**19 + 1])
def test_sort_on_either_side_of_the_small_tiles(gpf, n):
    import torch
    k = np.random.default_rng(n).integers(0, 1 << 20, n, dtype=np.uint64).astype(np.uint32)
    ok, ov = gpf.gpf_sort_pairs(torch.from_numpy(k.view(np.int32)).cuda(),
                                torch.arange(n, dtype=torch.int32, device="cuda"), 20)
    order = np.argsort(k, kind="stable")
    assert np.array_equal(ok.cpu().numpy().view(np.uint32), k[order])
    assert np.array_equal(ov.cpu().numpy(), order.astype(np.int32))


@pytest.mark.parametrize("n", [63, 64, 65, 65536, 65537])
@pytest.mark.parametrize("span", [4, 5, 9])
def test_group_edges_and_boxes_of_many_cells(gpf, n, span):
    """Lists of boxes of up to 27, 64 and 512 cells, and every Gaussian of the
    last, partly filled group."""
    fnp, qnp = synth.config1_random(seed=n + span, n=n, m=2000)
    fnp.logscale = (fnp.logscale - 0.33 * math.log(n / 64.0)).astype(np.float32)
    _, _, ((o, z, c, idx), (ob, zb, cb, _)) = _both(gpf, fnp, qnp, gpf.GPF_SUM, math.inf,
                                                    max_span=span)
    assert c == cb and idx.stats()["flags"] == 0
    np.testing.assert_allclose(z, zb, rtol=SUM_RTOL, atol=1e-30)


@pytest.mark.parametrize("per", [1535, 1537, 4000])
def test_tiles_whose_samples_miss_a_dense_cell(gpf, per):
    """One hit point in a hundred stands in a dense cell of its own, so most of
    those tiles cost more than their sampled points say; just below and above
    the length at which such a tile is put off, and far above it."""
    rng = np.random.default_rng(per)
    m, dense = 1600, 16
    x = rng.uniform(0.0, 1.0, (m, 3))
    n = per * dense
    fnp, qnp = synth.config1_random(seed=per, n=n, m=m)
    fnp.mean = np.repeat(x[::m // dense], per, axis=0).T.astype(np.float32).copy()
    fnp.logscale = np.full_like(fnp.logscale, math.log(3e-3))
    qnp.x = np.ascontiguousarray(x.T.astype(np.float32))
    qnp.valid = np.ones_like(qnp.valid)
    _, _, ((o, z, c, idx), (ob, zb, cb, _)) = _both(gpf, fnp, qnp, gpf.GPF_SUM, 0.02,
                                                    query_cell=0.02, split_items=64)
    assert c == cb and idx.stats()["flags"] == 0
    tol = 4000 * 2.0 ** -24                       # at most 4000 positive terms
    np.testing.assert_allclose(z, zb, rtol=tol, atol=1e-30)
    np.testing.assert_allclose(o, ob, rtol=tol, atol=1e-30)


def _clusters(seed, per, n_clusters=60):
    """Hit points in tight clusters (per each, an odd number) far apart on a
    line of cells, so that sorted neighbours lie cells apart."""
    rng = np.random.default_rng(seed)
    c = rng.uniform(0.05, 0.95, (n_clusters, 3))
    x = np.repeat(c, per, axis=0) + rng.normal(0, 2e-3, (n_clusters * per, 3))
    x = x[: len(x) - (len(x) + 1) % 2]            # an odd number of hit points
    m = len(x)
    up = np.tile(np.array([[0.0], [0.0], [1.0]]), (1, m)).astype(np.float32)
    return synth.Queries(x=np.ascontiguousarray(x.T.astype(np.float32)), n=up, wo=up.copy(),
                         valid=np.ones(m, np.uint8))


@pytest.mark.parametrize("per", [1, 7, 65, 333])
@pytest.mark.parametrize("channels", [1, 3, 4, 8])
def test_backward_row_ends_and_full_cells(gpf, per, channels):
    import torch
    from paper_2512_12459_gb300.setup_index import make_index
    qnp = _clusters(per, per)
    fnp, _ = synth.config1_random(seed=5 + per, n=900, m=8, channels=channels)
    field, queries = gpf.Field.from_numpy(fnp), gpf.Queries.from_numpy(qnp)
    rng = np.random.default_rng(per)
    G = torch.as_tensor(rng.standard_normal((channels, qnp.m)).astype(np.float32), device="cuda")
    for cell in (0.02, 0.3):
        idx = make_index(field, queries, query_cell=cell)
        idx.build(field, queries)
        for mode in (gpf.GPF_SUM, gpf.GPF_NORMALIZED):
            o, z = gpf.gpf_radiance_fwd(idx, field, queries, mode, r_max=0.2)
            g, g64 = (gpf.gpf_radiance_bwd(idx, field, queries, G, o, z, mode, r_max=0.2,
                                           f64_sums=f) for f in (False, True))
            for k in KEYS:
                a, b = getattr(g, k).double(), getattr(g64, k).double()
                assert float((a - b).norm()) <= GRAD_TOL * float(b.norm()), (k, cell, mode)


@pytest.mark.parametrize("most", [95, 97, 500, 3000])
def test_small_gaussians_over_uneven_cells(gpf, most):
    """Gaussians of a few cells whose cells hold one hit point or many, side by
    side in a warp: those with many may leave their lanes for the whole warp."""
    import torch
    from paper_2512_12459_gb300.setup_index import make_index
    rng = np.random.default_rng(most)
    c = rng.uniform(0.05, 0.95, (40, 3))
    x = np.repeat(c, np.where(np.arange(40) % 5, 1, most), axis=0)
    x = x + rng.normal(0, 2e-3, x.shape)
    m = len(x)
    up = np.tile(np.array([[0.0], [0.0], [1.0]]), (1, m)).astype(np.float32)
    queries = gpf.Queries.from_numpy(synth.Queries(
        x=np.ascontiguousarray(x.T.astype(np.float32)), n=up, wo=up.copy(),
        valid=np.ones(m, np.uint8)))
    fnp, _ = synth.config1_random(seed=most, n=960, m=8)
    fnp.mean = (np.tile(c, (24, 1)) + rng.normal(0, 2e-3, (960, 3))).T.astype(np.float32).copy()
    fnp.logscale = rng.normal(math.log(4e-3), 0.3, (3, 960)).astype(np.float32)
    field = gpf.Field.from_numpy(fnp)
    G = torch.as_tensor(rng.standard_normal((3, m)).astype(np.float32), device="cuda")
    idx = make_index(field, queries, query_cell=0.05)
    idx.build(field, queries)
    assert idx.stats()["n_small"] > 0
    o, z = gpf.gpf_radiance_fwd(idx, field, queries, gpf.GPF_SUM, r_max=0.2)
    g, g64 = (gpf.gpf_radiance_bwd(idx, field, queries, G, o, z, gpf.GPF_SUM, r_max=0.2,
                                   f64_sums=f) for f in (False, True))
    for k in KEYS:
        a, b = getattr(g, k).double(), getattr(g64, k).double()
        assert float((a - b).norm()) <= GRAD_TOL * float(b.norm()), k


@pytest.mark.parametrize("value", [math.nan, math.inf])
def test_a_wild_upstream_value_reaches_its_own_gaussians_only(gpf, value):
    import torch
    from paper_2512_12459_gb300.setup_index import make_index
    fnp, qnp = synth.config1_random(seed=77, n=1500, m=3001)
    field, queries = gpf.Field.from_numpy(fnp), gpf.Queries.from_numpy(qnp)
    act = np.flatnonzero(np.sum(qnp.n.astype(np.float64) * qnp.wo, axis=0) > 0)
    p = int(act[len(act) // 2])
    ref = oracle.radiance_fwd(fnp.mean, fnp.quat, fnp.logscale, fnp.spectrum, qnp.x[:, [p]],
                              qnp.n[:, [p]], qnp.wo[:, [p]], mode=oracle.GPF_SUM, r_max=math.inf,
                              cutoff_sigma=3.0)
    assert not ref["near_cutoff"][0]
    G = torch.randn((3, qnp.m), generator=torch.Generator("cuda").manual_seed(3), device="cuda")
    idx = make_index(field, queries, query_cell=0.08)
    idx.build(field, queries)
    grads = []
    for v in (0.0, value):
        H = G.clone()
        H[:, p] = v
        grads.append(gpf.gpf_radiance_bwd(idx, field, queries, H, mode=gpf.GPF_SUM))
    bad = ~torch.isfinite(grads[1].spectrum[0])
    d = qnp.x[:, [p]].astype(np.float64) - fnp.mean
    assert 0 < int(bad.sum()) <= int((np.linalg.norm(d, axis=0)
                                      <= 3.0 * np.exp(fnp.logscale.max(axis=0)) * 1.001).sum())
    for a, b in zip(grads[0].tensors(), grads[1].tensors()):
        assert torch.equal(a[:, ~bad], b[:, ~bad])


@pytest.mark.parametrize("k_min", [1, 3, 8])
def test_knn_without_fine_occupancy_bits(gpf, k_min):
    """A centre grid of more than 2^29 cells keeps only the coarse bits."""
    from paper_2512_12459_gb300.setup_index import make_index
    fnp, qnp = synth.config1_random(seed=9, n=400, m=700)
    # in a tenth of the grid, so that the nearest means lie within its rings
    fnp.mean, qnp.x = (np.float32(0.45) + np.float32(0.1) * v for v in (fnp.mean, qnp.x))
    fnp.logscale = fnp.logscale - np.float32(math.log(10.0))
    field, queries = gpf.Field.from_numpy(fnp), gpf.Queries.from_numpy(qnp)
    sparse = gpf.grid_for_bounds([0.0] * 3, [1.0] * 3, 1.0 / 1600, 3, 400, 700, 400_000,
                                 levels=8, query_level=4, hash_bits=16)
    outs = []
    for grid in (None, sparse):
        kw = {"query_cell": 0.1} if grid is None else {"grid": grid}
        idx = make_index(field, queries, ball_radius=1.0 / 2000, **kw)
        idx.build(field, queries)
        assert idx.stats()["flags"] == 0
        o, _ = gpf.gpf_radiance_fwd(idx, field, queries, gpf.GPF_NORMALIZED, r_max=math.inf,
                                    neighbourhood=gpf.GPF_NB_BALL_KNN, ball_r=1.0 / 2000,
                                    k_min=k_min)
        outs.append(o.cpu().numpy())
    np.testing.assert_array_equal(outs[0], outs[1])


def test_disk_gather_on_one_fine_level(gpf):
    """The disk kernel on a grid finer than the disk (boxes over many cells)."""
    fnp, qnp = synth.config1_random(seed=19, n=500, m=4000)
    fnp.logscale[:] = math.log(0.1 / 3.0)
    _, _, ((o, z, _, _), (ob, zb, _, _)) = _both(gpf, fnp, qnp, gpf.GPF_DISK_KDE, 0.1,
                                                 max_span=12, query_cell=0.05, coop_cells=8)
    np.testing.assert_array_equal(z, zb)
    np.testing.assert_allclose(o, ob, rtol=SUM_RTOL, atol=1e-30)
