"""FP64 factor solves: a column's result does not depend on the block it is solved in -- blocks are worked off 16
columns at a time, rows in groups of 16 with the groups beyond a supernode's edge left out.  (The accuracy of the
solves is compared with the oracle's in test_gpu_steps.py.)"""
import numpy as np
import pytest

from paper_1308_2445_gb300 import pufe_inputs as pi

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def dev(a):
    t = torch.zeros(a.shape[0], (a.shape[1] + 3) // 4 * 4, dtype=torch.float64, device="cuda")[:, :a.shape[1]]
    t.copy_(torch.from_numpy(a))
    return t


@pytest.mark.parametrize("k", [2, 15, 16, 17, 31, 33, 48, 65])
def test_columns_of_any_block(k):
    from paper_1308_2445_gb300 import hbsd
    p = pi.small_case()
    s = hbsd.Session.from_problem(p, precond=hbsd.PRECOND_GLOBAL)
    R = pi.seed_normal_block(11, p.n, k)
    P = dev(0 * R)
    s.precond_apply(dev(R), P)
    P = P.cpu().numpy()
    one = dev(np.zeros((p.n, 1)))
    for j in sorted({0, 1, k // 2, k - 1}):
        s.precond_apply(dev(R[:, j:j + 1]), one)
        assert np.array_equal(one.cpu().numpy()[:, 0], P[:, j])
    s.close()
