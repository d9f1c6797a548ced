"""Rows of hundreds and thousands of entries among short ones: the iterative
coarsest solve, whose long rows go beyond what eight lanes take (256 entries),
and the outer product of FP32 block solves in slices wider than 64. Cycle and
solutions against the oracle at the tolerances of the other parity tests. A hub
is a chain of dependent loads that the whole grid waits for, so its time is
compared with that of another path over the same row, with a fifth for the noise
and for what else differs."""
import time

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


@pytest.mark.parametrize("sizes", [[58, 60, 70], [64, 65, 66, 67], [1500, 90]])
@pytest.mark.parametrize("k", [1, 3, 8, 33])
def test_fp32_block(orc, sizes, k):
    import torch
    from paper_2006_16147_gb300 import amg
    A = W.with_hubs(W.poisson3d(14), sizes, 5)
    B = W.rhs_normal(A.n, 6, k)
    X = {}
    for p in (0, 1):
        h = setup(A, precision=p, krylov=1)
        x = torch.zeros(B.shape, dtype=torch.float64, device="cuda:0")
        infos = amg.amg_solve_batch(h, dev(B), x, rtol=1e-10)
        h.close()
        X[p] = x.cpu().numpy()
        assert max(i["true_relres"] for i in infos) <= 1e-10
    # both solve to 1e-10: apart by at most cond(A) times that, cond below 1e3 for the diagonally dominant hubs
    assert np.linalg.norm(X[1] - X[0]) <= 2e-7 * np.linalg.norm(X[0])


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


def test_time_of_a_hub_in_the_fp32_product():
    # a block solve with the FP32 V-cycle beside the FP64 one, in the same number of iterations: every kernel's
    # entries are half as long or the same
    import torch
    from paper_2006_16147_gb300 import amg
    A = W.with_hubs(W.poisson3d(40, 44, 30), [40, 200, 5000], 7)
    B = dev(W.rhs_normal(A.n, 3, 1))
    t, its = [], []
    for p in (0, 1):
        h = setup(A, precision=p, **COARSE_CG)
        runs = []
        for _ in range(6):
            X = torch.zeros_like(B)
            torch.cuda.synchronize()
            a = time.perf_counter()
            its.append(amg.amg_solve_batch(h, B, X)[0]["iterations"])
            torch.cuda.synchronize()
            runs.append(time.perf_counter() - a)
        h.close()
        t.append(np.median(runs[1:]))
    assert max(its) == min(its)
    assert t[1] <= 1.2 * t[0]
