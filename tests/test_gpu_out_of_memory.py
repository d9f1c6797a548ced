"""Calls that find too little device memory report it and leave nothing behind:
the next call does not report it again, and the same one succeeds once there is
room."""
import ctypes

import numpy as np
import pytest

from gpu_util import dev, setup
from paper_2006_16147_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def leave(room):
    """Takes the device's free memory but for `room` bytes."""
    import torch
    torch.cuda.synchronize()
    rt = ctypes.CDLL("libcudart.so." + torch.version.cuda.split(".")[0])
    pool = ctypes.c_void_p()
    assert rt.cudaDeviceGetDefaultMemPool(ctypes.byref(pool), 0) == 0
    assert rt.cudaMemPoolTrimTo(pool, ctypes.c_size_t(0)) == 0
    torch.cuda.empty_cache()
    return torch.empty(torch.cuda.mem_get_info()[0] - room, dtype=torch.uint8, device="cuda:0")


def test_setup_after_a_failed_one():
    import torch
    from paper_2006_16147_gb300 import amg
    A, S = W.poisson3d(128), W.poisson3d(8)        # the large one needs some 800 MB
    c = [dev(v) for v in (A.row_ptr, A.col, A.val, np.ones(A.n))]
    hog = leave(256 << 20)
    with pytest.raises(amg.AmgError) as e:
        amg.amg_setup(*c)
    assert e.value.status == amg.AMG_ERR_OOM
    setup(S).close()
    del hog
    torch.cuda.empty_cache()
    h = amg.amg_setup(*c)
    assert amg.amg_hierarchy_info(h)["n"][0] == A.n
    h.close()


def test_block_solve_after_a_failed_one():
    import torch
    from paper_2006_16147_gb300 import amg
    A = W.poisson3d(64)
    k = 192                                        # some 4 GB of work arrays
    h = setup(A)
    B = dev(W.rhs_normal(A.n, 2, k))
    X = torch.zeros_like(B)
    hog = leave(1 << 30)
    with pytest.raises(amg.AmgError) as e:
        amg.amg_solve_batch(h, B, X)
    assert e.value.status == amg.AMG_ERR_OOM
    few = torch.zeros((A.n, 2), dtype=torch.float64, device="cuda:0")
    assert amg.amg_solve_batch(h, B[:, :2].contiguous(), few)[0]["status"] == 0
    del hog
    torch.cuda.empty_cache()
    infos = amg.amg_solve_batch(h, B, X)
    assert infos[0]["status"] == 0 and max(i["true_relres"] for i in infos) <= 1e-6
    r = B[:, 0].cpu().numpy() - W.csr_matvec(A, X[:, 0].cpu().numpy())
    assert np.linalg.norm(r) <= 1.01e-6 * np.linalg.norm(B[:, 0].cpu().numpy())
    h.close()
