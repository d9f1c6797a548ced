"""Level-0 matrices of the FP64 V-cycle above 32 slices per SM, whose rows take
their columns place by place from the differences that a slice shares: matrices
where all slices line up, where some places leave the matrix, and where few line
up, with a last partial slice. The cycle and the solution against the oracle at
the tolerance of the other parity tests (1e-10)."""
import numpy as np
import pytest

from gpu_util import assert_same_solution, setup, solve, vcycle
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
    if kind == "part_random":                    # a box and rows without a pattern: most slices shared, some not
        return W.block_diagonal([W.poisson3d(64, 64, 36), W.random_spd_sparse(12345, 3, 6)])[0]
    return W.with_hubs(W.poisson3d(60, 54, 50), [40, 200], 7)


@pytest.mark.parametrize("kind", ["lines_of_64", "odd_box", "plane", "random", "part_random", "hubs"])
def test_fp64_cycle(orc, kind):
    import torch
    A = matrix(kind)
    assert A.n > 32 * 32 * torch.cuda.get_device_properties(0).multi_processor_count
    r = np.random.default_rng(2).standard_normal(A.n)
    H = orc.Hierarchy(A)
    h = setup(A)
    zo = H.vcycle(r)
    assert np.linalg.norm(vcycle(h, r) - zo) <= 1e-10 * np.linalg.norm(zo)
    xo, io = H.pcg(r)
    xg, ig = solve(h, r)
    assert ig["status"] == 0
    assert_same_solution(H, r, xg, ig, xo, io)
    h.close()
