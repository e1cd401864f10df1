"""The default team width of batches: one rule for the served and the caller's
batches of a serving context."""
import time

import numpy as np
import pytest

from paper_2508_05773_gb300 import scenarios as sc
from tests.served import served_costs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pkg():
    from paper_2508_05773_gb300 import build as native_build
    native_build.build()
    import paper_2508_05773_gb300
    paper_2508_05773_gb300.load()
    return paper_2508_05773_gb300


@pytest.mark.parametrize("flags", [0, sc.FLAG_OBS8, sc.FLAG_OBS8 | sc.FLAG_THIRD_ORDER])
@pytest.mark.parametrize("max_batch", [1, 128])
def test_served_solve_equals_a_batch_of_one(pkg, flags, max_batch):
    """Whatever the batch capacity of the serving context and its optional
    terms (served_costs asserts the equality of the bits)."""
    c = sc.small_random(77, S=512, H=10, n_obs=5)
    if flags:
        c = sc.with_moving(c, 4)
    c["params"] = dict(c["params"], flags=flags)
    s = pkg.Solver(c["params"], max_obstacles=6, max_path_pts=c["path"].shape[0], max_vehicles=1, max_batch=max_batch)
    try:
        s.register(0, c["path"], c["ds"], c["U_nom"], c["seed"])
        U0, seed, counter = s.vehicle_export(0)
        st, ticket = s.submit(0, c["x0"], c["obs"])
        assert st == 0
        st, end = -3, time.time() + 30.0
        while st == -3 and time.time() < end:  # EAGAIN
            st, U, _, _ = s.poll(ticket, True)
        assert st == 0
        served_costs(s, c, U0, seed, counter, U)
    finally:
        s.close()
