"""Solves around the size where the row products change their batch (eight
entries at a time with overlapping launches, four with all warps resident): the
same problem just below and above it, rows of one entry, of exactly eight, nine
and sixteen, and repeated solves on one hierarchy while its kernels overlap.
Against the oracle at the tolerance of the other parity tests (1e-10)."""
import numpy as np
import pytest

from gpu_util import assert_same_solution, setup, solve, vcycle
from paper_2006_16147_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("nx", [154, 158])       # 154^2 * 6 rows: below 152 * 4 * 8 slices; 158^2 * 6: above
def test_batch_boundary(orc, nx, precision):
    A = W.poisson3d(nx, nx, 6 + (nx > 154))
    b, _ = W.rhs_uniform(A, 3)
    H = orc.Hierarchy(A)
    h = setup(A, precision=precision)
    xo, io = H.pcg(b)
    xg, ig = solve(h, b)
    assert abs(ig["iterations"] - io["iterations"]) <= 1 and ig["true_relres"] <= 1e-6
    if precision == 0:
        assert_same_solution(H, b, xg, ig, xo, io)
    again, _ = solve(h, b)
    assert np.array_equal(xg, again)
    h.close()


@pytest.mark.parametrize("n,k", [(300, 0), (300, 8), (5000, 2), (5000, 4), (5000, 8)])
def test_row_lengths(orc, n, k):
    A = W.random_spd_sparse(n, k, 17 + k) if k else W.Csr(np.arange(n + 1), np.arange(n), np.linspace(1.0, 2.0, n))
    r = np.random.default_rng(n + k).standard_normal(n)
    H = orc.Hierarchy(A, max_coarse=40)
    h = setup(A, max_coarse=40)
    zo = H.vcycle(r)
    assert np.linalg.norm(vcycle(h, r) - zo) <= 1e-10 * np.linalg.norm(zo)
    xo, io = H.pcg(r)
    xg, ig = solve(h, r)
    assert_same_solution(H, r, xg, ig, xo, io)
    h.close()
