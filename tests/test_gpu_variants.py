"""Instantiations that only some sizes reach, each asserted to be the one that
runs: rows' state in local memory with a steer-rate column (one float4 a row),
teams that draw their noise themselves, and packed pairs of the optional terms.
A variant's solve gives the same bits as the same shape with the rows in shared
memory, or with one sample a team, and matches the FP64 oracle."""
import numpy as np
import pytest

import oracle
from paper_2508_05773_gb300 import scenarios as sc
from tests import plan_probe
from tests.gpu_solve import device_solve, device_tensors, host_outputs
from tests.parity import assert_solve_matches

pytestmark = pytest.mark.gpu
KEYS = ("U", "traj", "J", "J_lo", "u_hist")


@pytest.fixture(scope="module")
def pkg():
    from paper_2508_05773_gb300 import build as native_build
    native_build.build()
    import paper_2508_05773_gb300
    paper_2508_05773_gb300.load()
    return paper_2508_05773_gb300


def _terms(c, family):
    """The scenario with the terms of a family of instantiations."""
    if family == "moving":
        return sc.with_moving(c, 3)
    if family == "point":
        c = sc.jerk_model(sc.with_moving(c, 3), a0=0.2, seed=3)
        return dict(c, params=dict(c["params"], flags=c["params"]["flags"] | sc.FLAG_THIRD_ORDER))
    if family == "discs":
        return dict(c, params=dict(c["params"], **sc.FIVE_DISCS))
    return c


def _check(out, c, label):
    p = sc.as_float32(c["params"])
    ref = oracle.solve(p, c["x0"], c["U_nom"], c["obs"], c["path"], c["ds"], c["seed"], c["counter"], want_uhist=True)
    ref["traj"] = ref["traj"][:, :7]
    assert_solve_matches(out, ref, p, label)


@pytest.mark.parametrize("family,tps,threads,n_obs", [("point", 1, 512, 28), ("discs", 1, 512, 5), ("point", 2, 480, 32),
                                                      ("discs", 4, 480, 12)])
def test_rows_with_a_steer_rate_column_in_local_memory(pkg, family, tps, threads, n_obs):
    c = sc.small_random(461 + tps, S=300, H=6, n_obs=n_obs)
    c = _terms(dict(c, path=sc.path_table([("S", 60.0), ("A", 12.0, 1.2)], 0.01, True)[:7000].copy(), ds=0.01), family)
    out = {}
    for local, rows in ((1, 7000), (0, 1500)):  # the rollouts stay within the first metre
        s = pkg.Solver(c["params"], max_obstacles=n_obs, max_path_pts=7000, threads_per_sample=tps,
                       block_threads=threads if local else 128)
        try:
            plan = plan_probe.single(s, n_obs, rows)
            assert (plan["family"], plan["tps"], plan["local"], plan["ns"]) == (family, tps, local, 1), plan
            out[local] = device_solve(s, dict(c, path=c["path"][:rows]))
        finally:
            s.close()
    for key in ("J", "J_lo", "u_hist"):  # (the block's size orders the sums of U)
        assert np.array_equal(out[0][key], out[1][key]), key
    _check(out[1], c, f"local rows {family} tps={tps}")


@pytest.mark.parametrize("family", ["plain", "moving", "point"])
@pytest.mark.parametrize("tps,n_obs", [(2, 25), (4, 40), (8, 70)])
def test_teams_that_draw_three_blocks_a_lane(pkg, family, tps, n_obs):
    c = _terms(sc.small_random(471 + tps, S=150, H=6, n_obs=n_obs), family)
    s = pkg.Solver(c["params"], max_obstacles=n_obs, max_path_pts=c["path"].shape[0], threads_per_sample=tps,
                   block_threads=128)
    try:
        plan = plan_probe.single(s, n_obs, c["path"].shape[0])
        assert (plan["family"], plan["bpt"], plan["local"], plan["ns"]) == (family, 3, 0, 1), plan
        _check(device_solve(s, c), c, f"three blocks a lane {family} tps={tps}")
    finally:
        s.close()


@pytest.mark.parametrize("family,n_obs", [("plain", 61), ("moving", 124), ("point", 70), ("discs", 24)])
def test_few_samples_of_many_rows_take_32_lanes(pkg, family, n_obs):
    c = _terms(sc.small_random(477, S=150, H=6, n_obs=n_obs), family)
    s = pkg.Solver(c["params"], max_obstacles=n_obs, max_path_pts=c["path"].shape[0])
    try:
        plan = plan_probe.single(s, n_obs, c["path"].shape[0])
        assert (plan["family"], plan["tps"]) == (family, 32), plan
        _check(device_solve(s, c), c, f"32 lanes {family}")
    finally:
        s.close()


@pytest.mark.parametrize("family,tps,most", [("moving", 2, 25), ("moving", 4, 40), ("moving", 8, 70), ("discs", 1, 5),
                                             ("point", 1, 11)])
def test_pairs_of_the_optional_terms_equal_one_sample(pkg, family, tps, most):
    import torch
    dev = torch.device("cuda:0")
    threads = 128
    spb = threads // tps
    base = _terms(sc.small_random(481 + tps, S=20 * spb + 1, H=5, n_obs=most), family)
    cases = [dict(base, obs=base["obs"][:n], seed=800 + n) for n in (1, most // 2, most)]
    n_fill = 14 * 152 // 21
    s = pkg.Solver(base["params"], max_obstacles=most, max_path_pts=base["path"].shape[0],
                   max_batch=n_fill + len(cases), batch_threads_per_sample=tps, batch_block_threads=threads)
    instance = lambda c: dict(device_tensors(c, dev), U_next=torch.empty((5, 3), device=dev))  # noqa: E731
    try:
        mix = [instance(c) for c in cases]
        fill = [dict(instance(cases[0]), seed=7000 + i) for i in range(n_fill)]
        plan = plan_probe.batch(s, mix + fill)
        assert (plan["family"], plan["tps"], plan["ns"]) == (family, tps, 2), plan
        s.solve_batch(mix + fill)
        torch.cuda.synchronize()
        for c, d in zip(cases, mix):
            one = instance(c)
            assert plan_probe.batch(s, [one])["ns"] == 1
            s.solve_batch([one])
            torch.cuda.synchronize()
            a, b = host_outputs(d), host_outputs(one)
            for key in KEYS + ("U_next",):
                assert np.array_equal(a[key], b[key]), (len(c["obs"]), key)
            _check(a, c, f"pairs {family} tps={tps} n_obs={len(c['obs'])}")
    finally:
        s.close()
