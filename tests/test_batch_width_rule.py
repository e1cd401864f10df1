"""The default team width of batches with the optional terms (no GPU): a large
context's batches, which may hold one solve or two, keep teams of at most two
Philox blocks a lane where one lane a sample takes longer for those."""
import ctypes
import shutil

import pytest

from paper_2508_05773_gb300 import scenarios as sc

pytestmark = pytest.mark.skipif(shutil.which("nvcc") is None, reason="nvcc not available")
MOVING = dict(flags=sc.FLAG_OBS8)
THIRD = dict(flags=sc.FLAG_OBS8 | sc.FLAG_THIRD_ORDER | sc.FLAG_JERK)
DISCS = dict(flags=sc.FLAG_OBS8, **sc.FIVE_DISCS)
BUFFER = dict(flags=sc.FLAG_OBS8 | sc.FLAG_ALPHA_BUFFER)
COLLISION = dict(flags=sc.FLAG_PROJ_NONE | sc.FLAG_COLLISION_COST)


@pytest.mark.parametrize("terms,n_obs,solves,width", [
    ({}, 8, 1, 4), ({}, 8, 200, 1),
    (MOVING, 3, 200, 1), (MOVING, 8, 16, 2), (MOVING, 8, 200, 1), (MOVING, 20, 200, 4), (MOVING, 40, 200, 8),
    (THIRD, 3, 16, 2), (THIRD, 8, 16, 2), (THIRD, 8, 200, 2), (THIRD, 16, 200, 4), (THIRD, 100, 200, 16),
    (BUFFER, 11, 16, 2), (BUFFER, 11, 200, 1),
    (DISCS, 1, 200, 2), (DISCS, 2, 200, 2), (DISCS, 4, 200, 4), (DISCS, 8, 200, 8),
    (COLLISION, 8, 200, 1), (COLLISION, 16, 200, 2), (COLLISION, 16, 1, 4), (COLLISION, 28, 200, 2),
])
def test_width_of_a_context(terms, n_obs, solves, width):
    import paper_2508_05773_gb300 as pkg
    from tests import plan_probe
    c = plan_probe.HostContext(sc.params(S=4096, H=50, **terms), max_obstacles=n_obs, max_path_pts=388,
                               max_batch=solves)
    try:
        assert pkg.brmppi_get_batch_launch(ctypes.c_void_p(c.ctx))["threads_per_sample"] == width
    finally:
        c.close()
