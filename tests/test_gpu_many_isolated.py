"""Batches above the size at which level 0's slices are lined up (32 slices per
SM): a system with a right-hand side of zeros, which takes no step, or with one
that holds a NaN changes no bit of the others, whatever an earlier solve left in
the kept vectors. The reference is the same batch with finite right-hand sides
in every system."""
import numpy as np
import pytest

from gpu_util import dev
from paper_2006_16147_gb300 import workloads as W

pytestmark = pytest.mark.gpu
ODD = 12                                     # the system with zeros or a NaN


def batch(kind):
    if kind == "boxes":                      # the last and first lines of neighbours share slices
        mats = [W.poisson3d(17)] * 38
    else:                                    # rows of very different lengths at the boundaries
        mats = [W.poisson3d(30), W.poisson2d_aniso(131, 57), W.random_spd_sparse(9000, 3, 4)] * 6
    return mats, np.concatenate([[0], np.cumsum([A.n for A in mats])])


def overflow(h, offs):
    """A solve of the union that breaks down: the odd system's part of the kept CG vectors is not finite after it."""
    import torch
    from paper_2006_16147_gb300 import amg
    b = np.zeros(offs[-1])
    b[offs[ODD]:offs[ODD + 1]] = 1e308
    with pytest.raises(amg.AmgError):
        amg.amg_solve(h, dev(b), torch.zeros(len(b), dtype=torch.float64, device="cuda:0"))


def setup(mats, precision):
    import torch
    from paper_2006_16147_gb300 import amg
    assert sum(A.n for A in mats) > 32 * 32 * torch.cuda.get_device_properties(0).multi_processor_count
    return amg.amg_setup_many([(dev(A.row_ptr), dev(A.col), dev(A.val), dev(np.ones(A.n))) for A in mats],
                              precision=precision)


def solve(h, b, m):
    """x and the iterations of every system, also where the call reports a failed one."""
    import torch
    from paper_2006_16147_gb300 import amg
    x, bd = torch.zeros(len(b), dtype=torch.float64, device="cuda:0"), dev(b)
    infos = (amg.amg_solve_info * m)()
    st = amg.lib().amg_solve_many(h.handle, bd.data_ptr(), x.data_ptr(), 1e-6, 200, infos)
    return st, x.cpu().numpy(), [i.iterations for i in infos]


def same_elsewhere(offs, got, ref):
    out = np.ones(offs[-1], bool)
    out[offs[ODD]:offs[ODD + 1]] = False
    return np.array_equal(got[out], ref[out])


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("kind", ["boxes", "mixed"])
def test_zero_right_hand_side(kind, precision):
    mats, offs = batch(kind)
    m = len(mats)
    b = W.rhs_normal(offs[-1], 3)
    h = setup(mats, precision)
    st, x0, it0 = solve(h, b, m)
    assert st == 0
    overflow(h, offs)
    b[offs[ODD]:offs[ODD + 1]] = 0.0
    st, x1, it1 = solve(h, b, m)
    h.close()
    assert st == 0 and it1[ODD] == 0 and not x1[offs[ODD]:offs[ODD + 1]].any()
    assert it0[:ODD] + it0[ODD + 1:] == it1[:ODD] + it1[ODD + 1:]
    assert same_elsewhere(offs, x1, x0)


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("kind", ["boxes", "mixed"])
@pytest.mark.parametrize("row", [0, -1])
def test_right_hand_side_with_nan(kind, precision, row):
    import torch
    from paper_2006_16147_gb300 import amg
    mats, offs = batch(kind)
    m = len(mats)
    b = W.rhs_normal(offs[-1], 4)
    h = setup(mats, precision)
    st, x0, it0 = solve(h, b, m)
    assert st == 0
    z = [torch.empty(len(b), dtype=torch.float64, device="cuda:0") for _ in range(2)]
    amg.amg_vcycle(h, dev(b), z[0])
    b[offs[ODD] if row == 0 else offs[ODD + 1] - 1] = np.nan
    amg.amg_vcycle(h, dev(b), z[1])
    assert same_elsewhere(offs, z[1].cpu().numpy(), z[0].cpu().numpy())
    st, x1, it1 = solve(h, b, m)
    h.close()
    assert st == amg.AMG_ERR_BREAKDOWN                       # of that system alone
    assert it0[:ODD] + it0[ODD + 1:] == it1[:ODD] + it1[ODD + 1:]
    assert same_elsewhere(offs, x1, x0)
