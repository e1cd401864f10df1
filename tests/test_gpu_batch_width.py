"""The default team width of batches: one rule for the served and the caller's
batches of a serving context, and the widths of contexts with few samples."""
import time

import numpy as np
import pytest

import oracle
from paper_2508_05773_gb300 import scenarios as sc
from tests.gpu_solve import device_tensors, host_outputs
from tests.parity import assert_solve_matches
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


@pytest.mark.parametrize("n_obs,S,threads,width", [(8, 1000, 0, 4), (0, 500, 0, 2), (20, 333, 0, 8), (20, 333, 64, 4),
                                                   (8, 16000, 0, 2), (8, 18000, 0, 1)])
def test_small_contexts_take_wider_teams(pkg, n_obs, S, threads, width):
    """A context of few samples takes a team about a Philox block a lane wide,
    as far as a block size that the caller sets leaves 16 teams a block; the
    solves match the oracle, and alone and in a batch of two are the same bits."""
    import torch
    dev = torch.device("cuda:0")
    c = sc.small_random(500 + n_obs, S=S, H=6, n_obs=n_obs)
    s = pkg.Solver(c["params"], max_obstacles=max(1, n_obs), max_path_pts=c["path"].shape[0], max_batch=1 + (S < 8000),
                   batch_block_threads=threads)
    try:
        assert s.batch_launch()["threads_per_sample"] == width
        one, two = ([dict(device_tensors(c, dev), U_next=torch.empty((6, 3), device=dev)) for _ in range(n)]
                    for n in (1, 1 + (S < 8000)))
        s.solve_batch(one)
        s.solve_batch(two)
        torch.cuda.synchronize()
        a, b = host_outputs(one[0]), host_outputs(two[-1])
        for key in ("U", "traj", "J", "J_lo", "u_hist", "U_next"):
            assert np.array_equal(a[key], b[key]), key
        p = sc.as_float32(c["params"])
        ref = oracle.solve(p, c["x0"], c["U_nom"], c["obs"], c["path"], c["ds"], c["seed"], c["counter"],
                           want_uhist=True)
        assert_solve_matches(a, ref, p, f"width {width}")
    finally:
        s.close()
