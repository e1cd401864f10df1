"""The default launch shapes of single solves and of plain batches (no GPU), at
sizes where another shape took longer."""
import ctypes
import shutil

import pytest

from paper_2508_05773_gb300 import scenarios as sc

pytestmark = pytest.mark.skipif(shutil.which("nvcc") is None, reason="nvcc not available")
MOVING = dict(flags=sc.FLAG_OBS8)
THIRD = dict(flags=sc.FLAG_OBS8 | sc.FLAG_THIRD_ORDER)
DISCS = dict(flags=sc.FLAG_OBS8, **sc.FIVE_DISCS)


def _single(S, n_obs, terms):
    from tests import plan_probe
    c = plan_probe.HostContext(sc.params(S=S, H=30, **terms), max_obstacles=n_obs, max_path_pts=388)
    try:
        return plan_probe.single(c, n_obs, 388)
    finally:
        c.close()


@pytest.mark.parametrize("terms,n_obs,S,width", [(DISCS, 24, 64, 32), (DISCS, 16, 1000, 32), (DISCS, 24, 2000, 16),
                                                 (THIRD, 100, 256, 32), (MOVING, 124, 512, 32), ({}, 64, 512, 32),
                                                 ({}, 60, 512, 16), ({}, 100, 2000, 16)])
def test_more_than_sixteen_blocks_take_32_lanes_for_few_samples(terms, n_obs, S, width):
    p = _single(S, n_obs, terms)
    assert p["tps"] == width and p["tiles"] * (p["threads"] // p["tps"]) >= S


@pytest.mark.parametrize("n_obs,S,width", [(1, 9000, 2), (1, 10000, 1), (4, 12000, 1), (4, 17000, 1), (8, 16000, 2),
                                           (1, 4096, 2)])
def test_batches_of_few_rows_past_one_block_an_sm_take_one_lane(n_obs, S, width):
    import paper_2508_05773_gb300 as pkg
    from tests import plan_probe
    c = plan_probe.HostContext(sc.params(S=S, H=50), max_obstacles=n_obs, max_path_pts=388, max_batch=1)
    try:
        assert pkg.brmppi_get_batch_launch(ctypes.c_void_p(c.ctx))["threads_per_sample"] == width
    finally:
        c.close()


@pytest.mark.parametrize("n_obs,S,threads,ns", [(100, 10000, 192, 1), (100, 12000, 256, 2), (124, 11000, 256, 2),
                                                (124, 8500, 224, 1), (64, 25000, 256, 2), (64, 20000, 192, 1)])
def test_pairs_before_three_even_blocks_an_sm(n_obs, S, threads, ns):
    p = _single(S, n_obs, {})
    assert (p["threads"], p["ns"]) == (threads, ns), p


@pytest.mark.parametrize("rows,threads", [(388, 256), (2401, 384)])
def test_large_solves_share_long_tables_over_more_samples(rows, threads):
    from tests import plan_probe
    c = plan_probe.HostContext(sc.params(S=65536, H=100), max_obstacles=64, max_path_pts=rows)
    try:
        p = plan_probe.single(c, 64, rows)
        assert (p["threads"], p["ns"]) == (threads, 2), p
    finally:
        c.close()


@pytest.mark.parametrize("n_obs,threads", [(64, 128), (70, 128), (124, 128)])
def test_batches_of_many_ellipses_keep_small_tiles(n_obs, threads):
    import paper_2508_05773_gb300 as pkg
    from tests import plan_probe
    c = plan_probe.HostContext(sc.params(S=4096, H=50), max_obstacles=n_obs, max_path_pts=388, max_batch=64)
    try:
        assert pkg.brmppi_get_batch_launch(ctypes.c_void_p(c.ctx))["block_threads"] == threads
    finally:
        c.close()


@pytest.mark.parametrize("rows", [8100, 8140, 8180])
def test_few_samples_stay_unpaired_when_a_block_fills_shared_memory(rows):
    """One block an SM, whatever its tables: three tiles are no reason for two
    samples a lane, up to the last kilobyte of shared memory."""
    from tests import plan_probe
    c = plan_probe.HostContext(sc.params(S=1000, H=140), max_obstacles=28, max_path_pts=rows, threads_per_sample=1,
                               block_threads=384)
    try:
        p = plan_probe.single(c, 28, rows)
        assert p["tiles"] == 3 and p["smem"] > 228000 and (p["ns"], p["local"]) == (1, 0), p
    finally:
        c.close()
