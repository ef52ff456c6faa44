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

