"""Solves whose launch overlaps the stream's previous kernel: what that kernel
writes is what the solve reads, and what the next one overwrites has been
read, in a captured chain of warm starts and between other kernels."""
import pytest

from paper_2508_05773_gb300 import scenarios as sc
from tests.gpu_solve import device_tensors

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pkg():
    from paper_2508_05773_gb300 import build as native_build
    native_build.build()
    import paper_2508_05773_gb300
    paper_2508_05773_gb300.load()
    return paper_2508_05773_gb300


@pytest.mark.parametrize("S,H", [(1, 1), (257, 12), (4096, 20)])
def test_chained_solves_read_their_predecessors_results(pkg, S, H):
    import torch
    dev = torch.device("cuda:0")
    c = sc.small_random(31, S=S, H=H, n_obs=5)
    d = device_tensors(c, dev)
    s = pkg.Solver(c["params"], max_obstacles=5, max_path_pts=c["path"].shape[0])
    n = 4
    warm = [d["U_nom"].clone()] + [torch.empty_like(d["U_nom"]) for _ in range(n)]
    U = [torch.zeros_like(d["U_nom"]) for _ in range(n)]

    def solve(i, u_nom, u_next):
        assert s.solve_device(d["x0"], u_nom, d["obs"], d["path"], c["ds"], c["seed"], i, U[i], None, None, u_next,
                              None) == 0

    try:
        for i in range(n):  # one at a time
            solve(i, warm[i], warm[i + 1])
            torch.cuda.synchronize()
        ref = [u.clone() for u in U]
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g):
            for i in range(n):
                solve(i, warm[i], warm[i + 1])
        for _ in range(3):
            for u in U:
                u.zero_()
            g.replay()
        torch.cuda.synchronize()
        assert all(torch.equal(a, b) for a, b in zip(ref, U))
        for _ in range(10):  # between kernels that write what a solve reads, before and after it
            x = warm[0] * 1.0
            solve(0, x, warm[1].fill_(7.0))
            y = warm[1].clone()
            x.zero_()
            solve(1, y, warm[2])
            y.fill_(3.0)
            torch.cuda.synchronize()
            assert torch.equal(U[0], ref[0]) and torch.equal(U[1], ref[1])
    finally:
        s.close()
