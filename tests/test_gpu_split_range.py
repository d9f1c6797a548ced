"""Block solves with the FP32 V-cycle at the ends of the range in which the outer
product takes FP32 pieces: a system scaled by a power of two has the same
iterations and the scaled solution (up to what the last bits of the two product
paths do to CG, 1e-8 as in the other test of the pieces), and a small right-hand
side costs the time of an ordinary one: the same kernels in the same number, so
15% for the noise of two medians, where a row that needs pieces and FP64 chain
made the solve 1.4 times as long."""
import time

import numpy as np
import pytest

from gpu_util import dev
from paper_2006_16147_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def setup(A, scale=1.0):
    from paper_2006_16147_gb300 import amg
    return amg.amg_setup(dev(A.row_ptr), dev(A.col), dev(A.val * scale), dev(np.ones(A.n)), precision=1, krylov=1)


@pytest.mark.parametrize("op", ["poisson", "varcoef"])
@pytest.mark.parametrize("scale_a,scale_b", [(1.0, 2.0 ** -70), (1.0, 2.0 ** -88), (1.0, 2.0 ** 100), (2.0 ** -85, 2.0 ** -30),
                                             (2.0 ** -99, 2.0 ** -40), (2.0 ** 104, 2.0 ** 20)])
def test_scaled_systems(op, scale_a, scale_b):
    import torch
    from paper_2006_16147_gb300 import amg
    A = W.poisson3d(17, 16, 15) if op == "poisson" else W.varcoef3d(16, 4)
    B = W.rhs_normal(A.n, 5, 4)
    X, its = [], []
    for sa, sb in ((1.0, 1.0), (scale_a, scale_b)):
        h = setup(A, sa)
        x = torch.zeros(B.shape, dtype=torch.float64, device="cuda:0")
        infos = amg.amg_solve_batch(h, dev(B * sb), x)
        h.close()
        assert max(i["true_relres"] for i in infos) <= 1e-6
        X.append(x.cpu().numpy() * (sa / sb))
        its.append([i["iterations"] for i in infos])
    assert its[0] == its[1]
    assert np.linalg.norm(X[1] - X[0]) <= 1e-8 * np.linalg.norm(X[0])


def test_time_of_a_small_right_hand_side():
    import torch
    from paper_2006_16147_gb300 import amg
    A = W.poisson3d(64)
    h = setup(A)
    B = [dev(W.rhs_normal(A.n, 6, 64) * s) for s in (1.0, 2.0 ** -70)]
    X = torch.zeros_like(B[0])
    t = [[], []]
    for rep in range(8):
        for i in range(2):
            X.zero_()
            torch.cuda.synchronize()
            a = time.perf_counter()
            amg.amg_solve_batch(h, B[i], X)
            torch.cuda.synchronize()
            if rep:
                t[i].append(time.perf_counter() - a)
    h.close()
    assert np.median(t[1]) <= 1.15 * np.median(t[0])
