"""Block solves whose B and X start 8 bytes off a 16-byte boundary, as a
contiguous view into a larger tensor may: the same bits as from tensors of their
own, for column counts that take vector loads and that do not."""
import numpy as np
import pytest

from gpu_util import dev, setup
from paper_2006_16147_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("k", [1, 2, 3, 8, 64])
@pytest.mark.parametrize("off", [(1, 0), (0, 1), (1, 1)])
def test_offset_blocks(k, precision, off):
    import torch
    from paper_2006_16147_gb300 import amg
    A = W.poisson3d(17, 16, 15)
    h = setup(A, precision=precision)
    B = dev(W.rhs_normal(A.n, 2, k))
    X = torch.zeros_like(B)
    ref = amg.amg_solve_batch(h, B, X)
    room = [torch.zeros(A.n * k + 2, dtype=torch.float64, device="cuda:0") for _ in range(2)]
    Bo, Xo = (r[o:o + A.n * k].view(A.n, k) for r, o in zip(room, off))
    assert Bo.data_ptr() % 16 == 8 * off[0] and Xo.data_ptr() % 16 == 8 * off[1]
    Bo.copy_(B)
    got = amg.amg_solve_batch(h, Bo, Xo)
    h.close()
    assert torch.equal(Xo, X)
    assert [i["iterations"] for i in got] == [i["iterations"] for i in ref]
    assert room[1][off[1] + A.n * k:].eq(0).all() and room[1][:off[1]].eq(0).all()
