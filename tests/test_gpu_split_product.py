"""Block solves with the FP32 V-cycle, whose outer product takes the FP32 z in
FP32 pieces where every product is in range and the FP64 chain elsewhere:
matrices and right-hand sides scaled by powers of two through both, with
coefficients that are and are not floats, odd column counts, and a column of
zeros. A power of two changes no rounding, so the solution scales with it, up to
what the two product paths' last bits do to CG (1e-16 in FP64, passed through
the V-cycle's FP32 roundings: 1e-8 allowed)."""
import numpy as np
import pytest

from gpu_util import dev
from paper_2006_16147_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def run(A, B, scale_a, scale_b):
    import torch
    from paper_2006_16147_gb300 import amg
    h = amg.amg_setup(dev(A.row_ptr), dev(A.col), dev(A.val * scale_a), dev(np.ones(A.n)), precision=1, krylov=1)
    X = torch.zeros(B.shape, dtype=torch.float64, device="cuda:0")
    infos = amg.amg_solve_batch(h, dev(B * scale_b), X)
    h.close()
    return X.cpu().numpy() * (scale_a / scale_b), [i["iterations"] for i in infos], max(i["true_relres"] for i in infos)


@pytest.mark.parametrize("op", ["poisson", "varcoef"])
@pytest.mark.parametrize("k", [1, 3, 8])
@pytest.mark.parametrize("scale_a,scale_b", [(1.0, 2.0 ** -50), (1.0, 2.0 ** 50), (2.0 ** -90, 2.0 ** -60),
                                             (2.0 ** 60, 2.0 ** 90)])
def test_scaled_systems(op, k, scale_a, scale_b):
    A = W.poisson3d(17, 16, 15) if op == "poisson" else W.varcoef3d(16, 4)
    B = W.rhs_normal(A.n, 9, k)
    if k == 3:
        B[:, 1] = 0.0
    X1, it1, res1 = run(A, B, 1.0, 1.0)
    X2, it2, res2 = run(A, B, scale_a, scale_b)
    assert res1 <= 1e-6 and res2 <= 1e-6 and it1 == it2
    assert np.linalg.norm(X2 - X1) <= 1e-8 * np.linalg.norm(X1)
    R = B - np.stack([W.csr_matvec(A, X1[:, j]) for j in range(k)], 1)
    assert np.linalg.norm(R) <= 1.1e-6 * np.linalg.norm(B)
