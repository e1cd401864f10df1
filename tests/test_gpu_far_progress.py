"""A solve that begins millions of path cells before the path and reaches it
within the horizon: the stage cost reads the rows of the cells it reaches.

Tolerance.  The sampled progress rate carries up to four binary32 roundings (the
two constants of its map, the map, the sample), so the progress psi - psi0 is
known to 4 2^-24 of itself: delta = 4 2^-24 |psi0| / ds cells where the path is
reached.  A cell turns the reference heading by 1e-4 rad (two angle errors, at
most pi each) and moves the reference by 1e-5 m (5 m away at most), and at most
two steps are on the path: |dJ| <= 2 delta (2 Qth 2 pi 1e-4 + 2 Ql 5 1e-5).  A
solve that reads the first row instead is off by up to a tenth of J."""
import numpy as np
import pytest

import oracle
from paper_2508_05773_gb300 import scenarios as sc
from tests.gpu_solve import device_solve
from tests.parity import assert_solve_matches

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("psi0", [-30.0, -17.0, -0.02])
@pytest.mark.parametrize("tps", [1, 4])
def test_progress_from_far_before_the_path(psi0, tps):
    from paper_2508_05773_gb300 import build as native_build
    native_build.build()
    import paper_2508_05773_gb300 as pkg
    c = sc.small_random(611, S=300, H=12, n_obs=2)
    rate = np.float32(-psi0 + 0.02) / np.float32(12 * 0.05)  # the middle of the path at the last step
    n = 4000
    row = np.arange(n)
    path = np.stack([-1e-5 * row, 0.0 * row, np.pi + 1e-4 * row], 1).astype(np.float32)
    params = dict(c["params"], nu_bar=float(rate), R=(0.1, 0.1, 0.0),
                  z_hi=tuple(c["params"]["z_hi"][:2]) + (float(rate) + 20.0,))
    U = c["U_nom"].copy()
    U[:, 2] = rate + params["rho"] * (rate - 0.5 * params["z_hi"][2])  # (the projection pulls the rate to mid-range)
    x0 = c["x0"].copy()
    x0[6] = psi0
    c = dict(c, params=params, path=path, ds=1e-5, U_nom=U, x0=x0)
    p = sc.as_float32(params)
    ref = oracle.solve(p, c["x0"], c["U_nom"], c["obs"], c["path"], c["ds"], c["seed"], c["counter"], want_uhist=True)
    s = pkg.Solver(params, max_obstacles=2, max_path_pts=n, threads_per_sample=tps)
    try:
        delta = 4 * 2.0**-24 * abs(psi0) / 1e-5
        extra = 2 * delta * (2 * p["Qth"] * 2 * np.pi * 1e-4 + 2 * p["Ql"] * 5 * 1e-5)
        assert_solve_matches(device_solve(s, c), ref, p, f"psi0={psi0} tps={tps}", j_extra=np.full(300, extra))
    finally:
        s.close()
