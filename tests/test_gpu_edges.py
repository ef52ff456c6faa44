"""Values and sizes at which a branch of the build or of the pair loops changes
its mind, beside those of test_gpu_paths.py."""

import math

import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def gpf():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2512_12459_gb300 as g
    return g


@pytest.mark.parametrize("channels", [3, 4, 8])
@pytest.mark.parametrize("cell", [0.02, 0.3])
def test_products_that_overflow_reach_their_own_gaussians_only(gpf, channels, cell):
    """A finite upstream value whose product with a spectrum is infinite: the
    Gaussians that include that hit point get it, the others nothing of it."""
    import torch
    from paper_2512_12459_gb300.setup_index import make_index
    fnp, qnp = synth.config1_random(seed=78, n=1500, m=3001, channels=channels)
    fnp.spectrum = (fnp.spectrum + 10.0).astype(np.float32)
    field, queries = gpf.Field.from_numpy(fnp), gpf.Queries.from_numpy(qnp)
    act = np.flatnonzero(np.sum(qnp.n.astype(np.float64) * qnp.wo, axis=0) > 0)
    p = int(act[len(act) // 2])
    ref = oracle.radiance_fwd(fnp.mean, fnp.quat, fnp.logscale, fnp.spectrum, qnp.x[:, [p]],
                              qnp.n[:, [p]], qnp.wo[:, [p]], mode=oracle.GPF_SUM, r_max=math.inf,
                              cutoff_sigma=3.0)
    assert not ref["near_cutoff"][0]
    G = torch.randn((channels, qnp.m), generator=torch.Generator("cuda").manual_seed(4),
                    device="cuda")
    idx = make_index(field, queries, query_cell=cell)
    idx.build(field, queries)
    grads = []
    for v in (0.0, 2e38):
        H = G.clone()
        H[:, p] = v
        grads.append(gpf.gpf_radiance_bwd(idx, field, queries, H, mode=gpf.GPF_SUM))
    bad = ~torch.isfinite(grads[1].logscale[0])
    d = qnp.x[:, [p]].astype(np.float64) - fnp.mean
    assert 0 < int(bad.sum()) <= int((np.linalg.norm(d, axis=0)
                                      <= 3.0 * np.exp(fnp.logscale.max(axis=0)) * 1.001).sum())
    # (a Gaussian may include the point with a finite term: those that change at all)
    near = torch.from_numpy(np.linalg.norm(d, axis=0)
                            <= 3.0 * np.exp(fnp.logscale.max(axis=0)) * 1.001).cuda()
    for a, b in zip(grads[0].tensors(), grads[1].tensors()):
        assert torch.equal(a[:, ~near], b[:, ~near])


def test_two_threads_with_indexes_of_different_levels(gpf):
    """Small queries through one kernel from two host threads, each on a stream
    and an index of its own, whose warps need different shared memory."""
    import threading

    import torch
    from paper_2512_12459_gb300.setup_index import make_index
    fnp, qnp = synth.config1_random(seed=5, n=300, m=640)
    field, queries = gpf.Field.from_numpy(fnp), gpf.Queries.from_numpy(qnp)
    work = []
    for levels, coop in ((16, 8), (6, 8), (10, 8)):
        grid = gpf.grid_for_bounds([0.0] * 3, [1.0] * 3, 0.01, 3, 300, 640, 200_000,
                                   levels=levels, query_level=2, hash_bits=14)
        grid.coop_cells = coop
        idx = make_index(field, queries, grid=grid)
        idx.build(field, queries)
        out, _ = gpf.gpf_radiance_fwd(idx, field, queries, gpf.GPF_SUM)
        work.append((idx, out, torch.cuda.Stream()))
    torch.cuda.synchronize()
    errors = []

    def run(idx, out, stream):
        try:
            with torch.cuda.stream(stream):
                for _ in range(2000):
                    o, _ = gpf.gpf_radiance_fwd(idx, field, queries, gpf.GPF_SUM)
                stream.synchronize()
                assert torch.equal(o, out)
        except Exception as e:              # noqa: BLE001 (reported by the main thread)
            errors.append(repr(e))

    threads = [threading.Thread(target=run, args=w) for w in work]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors[0]


@pytest.mark.parametrize("n", [40, 400, 4000])
@pytest.mark.parametrize("height", [0.0, 0.05, 0.7])
def test_nearest_means_of_a_field_a_few_cells_high(gpf, n, height):
    """Means and hit points on a floor (and up to a height above it): rings of
    many coarse cells in one or a few layers. The nearest means are summed by
    distance, so cells of another size give the same sums bit for bit."""
    from paper_2512_12459_gb300.setup_index import make_index
    rng = np.random.default_rng(n)
    fnp, qnp = synth.config1_random(seed=n, n=n, m=1500)
    fnp.mean = np.concatenate([rng.uniform(0, 2, (2, n)), rng.uniform(0, 1, (1, n)) * height]
                              ).astype(np.float32)
    qnp.x = np.concatenate([rng.uniform(0, 2, (2, 1500)), rng.uniform(0, 1, (1, 1500)) * height]
                           ).astype(np.float32)
    field, queries = gpf.Field.from_numpy(fnp), gpf.Queries.from_numpy(qnp)
    outs = []
    for ball in (0.02, 0.05, 0.4):
        idx = make_index(field, queries, query_cell=0.05, ball_radius=ball)
        idx.build(field, queries)
        assert idx.stats()["flags"] == 0
        outs.append(gpf.gpf_radiance_fwd(idx, field, queries, gpf.GPF_SUM, r_max=0.5,
                                         neighbourhood=gpf.GPF_NB_BALL_KNN, ball_r=0.0,
                                         k_min=4)[0].cpu().numpy())
    assert outs[0].any()
    for o in outs[1:]:
        np.testing.assert_array_equal(o, outs[0])



# two float32 sums of the same positive terms, at most 2000 of them, in
# different orders: below 2000 * 2^-24 apart relative to the sum
SUM_RTOL = 1.2e-4


def _on_and_by_brute_force(gpf, fnp, qnp, mode, r, **kw):
    """(out, z) on a grid, twice, and by brute force; the pairs agree."""
    from paper_2512_12459_gb300.setup_index import make_index
    field, queries = gpf.Field.from_numpy(fnp), gpf.Queries.from_numpy(qnp)
    res, counts = [], []
    for k in (kw, {"brute_force": True}):
        idx = make_index(field, queries, cutoff_sigma=3.0, **k)
        idx.build(field, queries)
        assert idx.stats()["flags"] == 0
        for _ in range(1 if "brute_force" in k else 2):
            out, z = gpf.gpf_radiance_fwd(idx, field, queries, mode, r_max=r)
            res.append((out.cpu().numpy(), z.cpu().numpy()))
        counts.append(gpf.gpf_count_pairs(idx, field, queries)["included"])
    assert counts[0] == counts[1]
    return res


@pytest.mark.parametrize("tiles,every", [(1000, 1), (3000, 1), (6000, 3), (5000, 1)])
def test_density_estimate_whose_samples_miss_a_dense_cell(gpf, tiles, every):
    """A photon gather in which one unsampled point of (every third of) the tiles
    stands in a dense cell of 1,600 photons, so that these tiles are put off to the
    second launch: with teams of 16 and of 4 warps, one warp, and more tiles than
    the second launch has room to split."""
    m, per, r = 32 * tiles, 1600, 0.02
    a = np.array([1.1, 1.1, 1.1])
    x = np.tile(a + 0.12, (m, 1))                 # (one query-level cell: index order)
    x[1::32 * every] = a
    mean = np.concatenate([np.tile(a, (per, 1)), np.tile(a + 0.12, (5, 1)), [[0.0] * 3, [4.0] * 3]])
    fnp, qnp = synth.config1_random(seed=tiles, n=len(mean), m=m)
    fnp.mean = np.ascontiguousarray(mean.T.astype(np.float32))
    fnp.logscale[:] = math.log(r / 3.0)
    qnp.x = np.ascontiguousarray(x.T.astype(np.float32))
    qnp.n[:], qnp.valid = qnp.wo, np.ones_like(qnp.valid)
    (o, z), (o2, z2), (ob, zb) = _on_and_by_brute_force(gpf, fnp, qnp, gpf.GPF_DISK_KDE, r,
                                                        query_cell=0.85, split_items=64)
    np.testing.assert_array_equal(z, np.where(np.arange(m) % (32 * every) == 1, per, 5))
    np.testing.assert_array_equal(z, zb)
    np.testing.assert_array_equal(o, o2)
    np.testing.assert_array_equal(z, z2)
    np.testing.assert_allclose(o, ob, rtol=SUM_RTOL, atol=1e-30)


@pytest.mark.parametrize("m", [32, 32 * 152 * 32 + 32])
@pytest.mark.parametrize("split", [0, 64])
def test_tiles_of_more_than_32_walked_lists(gpf, m, split):
    """Hit points in eight cells on each of six levels: 48 lists a tile."""
    rng = np.random.default_rng(m)
    at = 0.1 + 0.25 * np.stack(np.meshgrid(range(4), range(4), [0], indexing="ij"), -1).reshape(-1, 3)[:8]
    x = at[np.arange(m) % 8] + 1e-4 * rng.standard_normal((m, 3))
    k = np.repeat(np.arange(8), 6 * 40)
    fnp, qnp = synth.config1_random(seed=m % 1000, n=len(k), m=m)
    fnp.mean = (at[k] + 1e-4 * rng.standard_normal((len(k), 3))).T.astype(np.float32).copy()
    fnp.logscale = np.tile(np.log(3e-4 * 2.0 ** (np.arange(len(k)) % 6)), (3, 1)).astype(np.float32)
    qnp.x = np.ascontiguousarray(x.T.astype(np.float32))
    qnp.n[:], qnp.valid = qnp.wo, np.ones_like(qnp.valid)
    grid = gpf.grid_for_bounds([0.0] * 3, [1.0] * 3, 8e-4, 3, len(k), m, 100_000, levels=6,
                               query_level=10, hash_bits=16)
    grid.coop_cells = 8
    (o, z), (o2, _), (ob, zb) = _on_and_by_brute_force(gpf, fnp, qnp, gpf.GPF_SUM, math.inf,
                                                       grid=grid, split_items=split)
    np.testing.assert_array_equal(o, o2)
    np.testing.assert_allclose(z, zb, rtol=SUM_RTOL, atol=1e-30)
    np.testing.assert_allclose(o, ob, rtol=SUM_RTOL, atol=1e-30)


@pytest.mark.parametrize("n", [255, 256, 257, 16383, 16384, 16385])
@pytest.mark.parametrize("span", [3, 9])
def test_edges_of_the_groups_that_list_their_entries(gpf, n, span):
    """Every Gaussian of the last, partly filled group of 256 and super-group of
    64 groups."""
    fnp, qnp = synth.config1_random(seed=n, n=n, m=2000)
    fnp.logscale = (fnp.logscale - 0.33 * math.log(n / 64.0)).astype(np.float32)
    (_, z), _, (_, zb) = _on_and_by_brute_force(gpf, fnp, qnp, gpf.GPF_SUM, math.inf,
                                                max_span=span)
    np.testing.assert_allclose(z, zb, rtol=SUM_RTOL, atol=1e-30)
