"""The dense inverse of a coarsest level that one launch factors over many
blocks: sizes at the edges of its 32-column panels and 8-row tiles, as a
single-level hierarchy (its V-cycle is the product with the inverse) and as
blocks of a batch above 256 rows. The factor has the oracle's bits; the product
is compared with numpy's solve within 8 n eps cond(A), the size of the forward
error bound of a Cholesky inverse (Higham, Accuracy and Stability of Numerical
Algorithms, ch. 14)."""
import numpy as np
import pytest

from gpu_util import dev, setup, vcycle
from paper_2006_16147_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def check(A, b, z):
    D = A.to_dense()
    x = np.linalg.solve(D, b)
    assert np.linalg.norm(z - x) <= 8 * A.n * np.finfo(float).eps * np.linalg.cond(D) * np.linalg.norm(x)


@pytest.mark.parametrize("n", [1, 2, 7, 8, 9, 31, 32, 33, 63, 64, 65, 97, 185, 257, 600])
def test_inverse_of_a_single_block(orc, n):
    from paper_2006_16147_gb300 import amg
    A = W.random_spd(n, 0.2, 11 + n)
    h = setup(A, max_coarse=n)
    assert amg.amg_hierarchy_info(h)["n"] == [n]
    assert np.array_equal(orc.Hierarchy(A, max_coarse=n).coarse_factor(), amg.amg_coarse_factor(h))
    b = np.random.default_rng(n).standard_normal(n)
    check(A, b, vcycle(h, b))
    h.close()


def test_indefinite_block_is_refused():
    from paper_2006_16147_gb300 import amg
    A = W.random_spd(150, 0.5, 5)
    val = A.val.copy()
    val[np.repeat(np.arange(A.n), np.diff(A.row_ptr)) == A.col] *= 1e-3
    A = W.Csr(A.row_ptr, A.col, val)
    with pytest.raises(amg.AmgError):
        setup(A, max_coarse=200)


@pytest.mark.parametrize("sizes", [(300, 40, 1), (33, 257)])
def test_batch_with_a_large_block(sizes):
    import torch
    from paper_2006_16147_gb300 import amg
    mats = [W.random_spd(n, 0.2, 70 + n) for n in sizes]
    h = amg.amg_setup_many([(dev(A.row_ptr), dev(A.col), dev(A.val), dev(np.ones(A.n))) for A in mats],
                           max_coarse=1000)
    b = np.random.default_rng(3).standard_normal(sum(sizes))
    z = torch.empty(len(b), dtype=torch.float64, device="cuda:0")
    amg.amg_vcycle(h, dev(b), z)
    z = z.cpu().numpy()
    at = 0
    for A in mats:
        check(A, b[at:at + A.n], z[at:at + A.n])
        at += A.n
    h.close()
