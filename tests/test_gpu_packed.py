"""The variants that draw their noise in registers (one or two samples a
team, rows' state in shared or local memory) and the contouring cost with
unequal weights, where they can go wrong: against the FP64 oracle at the
parity tolerances, and against one another bit for bit."""
import numpy as np
import pytest

import oracle
from paper_2508_05773_gb300 import scenarios as sc
from tests.gpu_solve import device_solve, device_tensors, host_outputs
from tests.parity import assert_solve_matches

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pkg():
    from paper_2508_05773_gb300 import build as native_build
    native_build.build()
    import paper_2508_05773_gb300
    paper_2508_05773_gb300.load()
    return paper_2508_05773_gb300


def _oracle(c):
    p = sc.as_float32(c["params"])
    return p, oracle.solve(p, c["x0"], c["U_nom"], c["obs"], c["path"], c["ds"], c["seed"], c["counter"],
                           want_uhist=True)


def _instance(c, dev):
    import torch
    d = device_tensors(c, dev)
    d["U_next"] = torch.empty((int(c["params"]["H"]), 3), device=dev)
    return d


@pytest.mark.parametrize("tps,threads,most", [(1, 128, 28), (1, 256, 28), (1, 512, 28), (2, 128, 28), (4, 256, 40), (8, 256, 70)])
def test_two_samples_a_team_equal_one(pkg, tps, threads, most):
    """A batch with enough tiles runs two samples a team in packed
    registers, the same solve alone one sample a team: every output is the
    same bits.  S odd leaves a pair with one real sample; 0, 1, 4, 13 and the
    most obstacles leave empty, partial and full passes over the Philox blocks."""
    import torch
    dev = torch.device("cuda:0")
    spb = threads // tps
    rng = np.random.default_rng(tps)
    base = sc.small_random(400 + tps, S=20 * spb + 1, H=5, n_obs=most)
    cases = [dict(base, obs=base["obs"][:n], seed=int(rng.integers(2**62))) for n in (0, 1, 4, 13, most)]
    # filler so that the tiles are several waves of packed CTAs
    n_fill = 14 * 152 // 21
    s = pkg.Solver(base["params"], max_obstacles=most, max_path_pts=base["path"].shape[0],
                   max_batch=n_fill + len(cases), batch_threads_per_sample=tps, batch_block_threads=threads)
    try:
        mix = [_instance(c, dev) for c in cases]
        fill = [dict(_instance(dict(base, obs=base["obs"][:2]), dev), seed=7000 + i) for i in range(n_fill)]
        s.solve_batch(mix + fill)
        torch.cuda.synchronize()
        for c, d in zip(cases, mix):
            one = _instance(c, dev)
            s.solve_batch([one])
            torch.cuda.synchronize()
            a, b = host_outputs(d), host_outputs(one)
            assert a["status"] == 0 and b["status"] == 0
            for key in ("U", "traj", "J", "J_lo", "u_hist", "U_next"):
                assert np.array_equal(a[key], b[key]), (len(c["obs"]), key)
            p, ref = _oracle(c)
            assert_solve_matches(a, ref, p, f"packed tps={tps} n_obs={len(c['obs'])}")
    finally:
        s.close()


@pytest.mark.parametrize("moving", [False, True])
def test_rows_in_local_memory(pkg, moving):
    """512-thread CTAs of one lane a sample with a long path and 28 rows a
    lane: the rows' state does not fit in shared memory beside the path."""
    c = sc.small_random(431, S=700, H=6, n_obs=28)
    c["path"] = sc.path_table([("S", 60.0), ("A", 12.0, 1.2)], 0.01, True)[:7000].copy()
    c["ds"] = 0.01
    if moving:
        c = sc.with_moving(c, 3)
    p, ref = _oracle(c)
    s = pkg.Solver(c["params"], max_obstacles=28, max_path_pts=7000, threads_per_sample=1, block_threads=512)
    try:
        assert_solve_matches(device_solve(s, c), ref, p, f"local rows moving={moving}")
    finally:
        s.close()


@pytest.mark.parametrize("tps", [1, 2, 4, 8])
def test_unequal_contour_and_lag_weights(pkg, tps):
    """Qc != Ql: the stage cost needs the path's direction."""
    c = sc.small_random(441, S=300, H=14, n_obs=9)
    c["params"] = dict(c["params"], Qc=7.0, Ql=12.5)
    p, ref = _oracle(c)
    s = pkg.Solver(c["params"], max_obstacles=9, max_path_pts=c["path"].shape[0], threads_per_sample=tps,
                   block_threads=64)
    try:
        assert_solve_matches(device_solve(s, c), ref, p, f"weights tps={tps}")
    finally:
        s.close()


@pytest.mark.parametrize("flags", [sc.FLAG_OBS8, sc.FLAG_OBS8 | sc.FLAG_COLLISION_COST | sc.FLAG_ALPHA_BUFFER])
def test_two_samples_a_lane_equal_one_with_optional_terms(pkg, flags):
    """The same for the family with the optional terms (one lane a sample in
    contexts whose capacity fills the GPU): 1, 3 and 11 moving rows."""
    import torch
    dev = torch.device("cuda:0")
    base = sc.with_moving(sc.small_random(451, S=20 * 128 + 1, H=5, n_obs=11), 4)
    base["params"] = dict(base["params"], flags=flags)
    cases = [dict(base, obs=base["obs"][:n], seed=900 + n) for n in (1, 3, 11)]
    n_fill = 14 * 152 // 21
    s = pkg.Solver(base["params"], max_obstacles=11, max_path_pts=base["path"].shape[0], max_batch=n_fill + len(cases))
    try:
        assert s.batch_launch()["threads_per_sample"] == 1
        mix = [_instance(c, dev) for c in cases]
        fill = [dict(_instance(cases[1], dev), seed=7000 + i) for i in range(n_fill)]
        s.solve_batch(mix + fill)
        torch.cuda.synchronize()
        for c, d in zip(cases, mix):
            one = _instance(c, dev)
            s.solve_batch([one])
            torch.cuda.synchronize()
            a, b = host_outputs(d), host_outputs(one)
            for key in ("U", "traj", "J", "J_lo", "u_hist", "U_next"):
                assert np.array_equal(a[key], b[key]), (len(c["obs"]), key)
            p, ref = _oracle(c)
            extra = None
            if flags & sc.FLAG_ALPHA_BUFFER:
                from tests.parity import buffer_conditioning
                extra = buffer_conditioning(p, c)
            assert_solve_matches(a, ref, p, f"packed optional terms n_obs={len(c['obs'])}", j_extra=extra)
    finally:
        s.close()
