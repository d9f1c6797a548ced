"""Rows of hundreds and thousands of entries among short ones in the iterative
coarsest solve, where they go beyond what eight lanes take (256). Cycle and
solutions against the oracle at the tolerances of the other parity tests. A hub
is a chain of dependent loads that the whole grid waits for, so its time is
compared with that of another path over the same row, with a fifth for the noise
and for what else differs."""
import numpy as np
import pytest

from gpu_util import assert_same_solution, dev, setup, solve, vcycle
from paper_2006_16147_gb300 import workloads as W

pytestmark = pytest.mark.gpu
COARSE_CG = dict(max_levels=2, max_dense=100, krylov=1)


@pytest.mark.parametrize("sizes", [[9, 33, 40], [250, 256, 257, 300], [64, 2500, 600, 6000]])
def test_coarsest_cg(orc, sizes):
    from paper_2006_16147_gb300 import amg
    A = W.with_hubs(W.poisson3d(30), sizes, 3)
    H = orc.Hierarchy(A, max_levels=2, max_dense=100)
    h = setup(A, **COARSE_CG)
    assert amg.amg_hierarchy_info(h)["coarse_solver"] == 1
    r = np.random.default_rng(1).standard_normal(A.n)
    zo = H.vcycle(r)
    assert np.linalg.norm(vcycle(h, r) - zo) <= 1e-10 * np.linalg.norm(zo)
    xo, io = H.pcg(r, flexible=True)
    xg, ig = solve(h, r)
    assert_same_solution(H, r, xg, ig, xo, io, flexible=True)
    h.close()


def test_time_of_a_hub_in_the_coarsest_solve():
    # 22K rows, a hub of thousands: the solve for one column beside the block solve's for one column
    import torch
    from paper_2006_16147_gb300 import amg
    A = W.with_hubs(W.poisson3d(60, 54, 50), [40, 200, 5000], 7)
    h = setup(A, profile=1, **COARSE_CG)
    b = dev(np.random.default_rng(1).standard_normal(A.n))
    ms = []
    for call in (lambda x: amg.amg_solve(h, b, x), lambda x: amg.amg_solve_batch(h, b.view(-1, 1), x.view(-1, 1))):
        call(torch.zeros_like(b))
        amg.amg_kernel_stats_reset(h)
        call(torch.zeros_like(b))
        torch.cuda.synchronize()
        n, t, _ = amg.amg_kernel_stats(h)["coarse_solve"]
        ms.append(t / n)
    h.close()
    assert ms[0] <= 1.2 * ms[1]
