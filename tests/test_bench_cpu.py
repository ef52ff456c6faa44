"""bench.py's captured DRAM bytes belong to one grid and one set of sources."""

import pytest

import bench


class _Grid:
    cell_size, query_level, max_span, coop_cells, split_items = 0.01, 2, 3, 8, 4096


@pytest.fixture
def captured(monkeypatch):
    monkeypatch.setattr(bench, "_sha256", lambda p: "hash of " + p)
    monkeypatch.setattr(bench, "PROFILED_TRAFFIC", [
        {"kernel": "fwd_kernel", "grid": (0.04, 3, 8, 4096), "bytes": 7,
         "sources": {"a.cu": "hash of a.cu"}},
        {"kernel": "bwd_grid_kernel", "grid": (0.04, 3, 8, 4096), "bytes": 9,
         "sources": {"a.cu": "another hash"}}])


def test_traffic_is_reported_for_the_grid_it_was_captured_on(captured):
    key = bench.grid_key(_Grid())
    assert key == (0.04, 3, 8, 4096)
    assert bench.profiled_traffic("fwd_kernel", key) == 7
    assert bench.profiled_traffic("fwd_kernel", (0.04 * (1 + 1e-5),) + key[1:]) == 7


@pytest.mark.parametrize("key", [(0.02, 3, 8, 4096), (0.04, 4, 8, 4096), (0.04, 3, 4, 4096),
                                 (0.04, 3, 8, 0)])
def test_traffic_of_another_grid_is_not_reported(captured, key):
    assert bench.profiled_traffic("fwd_kernel", key) is None


def test_traffic_of_other_sources_or_kernels_is_not_reported(captured):
    assert bench.profiled_traffic("bwd_grid_kernel", (0.04, 3, 8, 4096)) is None
    assert bench.profiled_traffic("loss_kernel", (0.04, 3, 8, 4096)) is None


def test_the_captures_name_kernels_that_are_timed():
    assert all(r["kernel"] in ("fwd_kernel", "bwd_grid_kernel") and len(r["grid"]) == 4
               and r["bytes"] > 0 for r in bench.PROFILED_TRAFFIC)
