"""Level-0 matrices of the FP32 V-cycle whose slices are lined up by col - row
(more than 32 slices per SM): a stencil with lines that do and do not end with a
slice, a last partial slice, and matrices that line up only in places (random
columns, a few long rows), which keep their columns. The FP32 cycle is compared
with the oracle's FP64 cycle at the tolerance of the other mixed-precision tests
(FP32 rounding through a V-cycle), the solution at its residual."""
import numpy as np
import pytest

from gpu_util import setup, solve, vcycle
from paper_2006_16147_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def matrix(kind):
    if kind == "lines_of_64":
        return W.poisson3d(64, 64, 40)
    if kind == "odd_box":
        return W.poisson3d(61, 53, 49)
    if kind == "plane":
        return W.poisson2d_aniso(397, 403)
    if kind == "random":
        return W.random_spd_sparse(157000, 3, 5)
    return W.with_hubs(W.poisson3d(60, 54, 50), [40, 200], 7)


@pytest.mark.parametrize("kind", ["lines_of_64", "odd_box", "plane", "random", "hubs"])
def test_fp32_cycle(orc, kind):
    A = matrix(kind)
    assert A.n > 32 * 152 * 32
    r = np.random.default_rng(2).standard_normal(A.n)
    H = orc.Hierarchy(A)
    h = setup(A, precision=1, krylov=1)
    zo = H.vcycle(r)
    assert np.linalg.norm(vcycle(h, r) - zo) <= 2e-5 * np.linalg.norm(zo)
    x, info = solve(h, r)
    res = np.linalg.norm(r - W.csr_matvec(A, x)) / np.linalg.norm(r)
    assert info["status"] == 0 and res <= 1.01e-6
    h.close()
