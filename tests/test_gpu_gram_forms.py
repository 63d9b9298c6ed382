"""The double-float Gram at the edges of its tiles, stages and chunks, against FP64 products.

Bound: each entry within 2^-44 of |Z|^T |ZH|: pairs carry 48 bits and keep sums of 64 rows between FP64
flushes.
"""
import numpy as np
import pytest

from paper_1308_2445_gb300 import pufe_inputs as pi

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def blocks(q, n, seed):
    """Z, ZH, ZS with rows over many decades (inversely in Z and in ZH, ZS) and columns of different sizes."""
    Z, ZH, ZS = (pi.seed_normal_block(seed + i, n, q) for i in range(3))
    d = 10.0 ** (8.0 * pi.uniform(seed, 9, n))[:, None]
    c = np.logspace(-4, 2, q)
    ZH = ZH + 3.0 * Z
    ZS = ZS + 0.5 * Z
    return Z * d * c, ZH * c / d, ZS * c / d


def gram(Z, ZH, ZS, ld=None):
    from paper_1308_2445_gb300 import hbsd
    n, q = Z.shape
    bufs = []
    for a in (Z, ZH, ZS):
        t = torch.zeros(n, ld or q + (q & 1), dtype=torch.float64, device="cuda")[:, :q]
        t.copy_(torch.from_numpy(a))
        bufs.append(t)
    HR = torch.zeros(q, q, dtype=torch.float64, device="cuda")
    SR = torch.zeros(q, q, dtype=torch.float64, device="cuda")
    hbsd.gram_df64(*bufs, HR, SR)
    torch.cuda.synchronize()
    return HR.cpu().numpy(), SR.cpu().numpy()


def check(Z, ZH, ZS, **kw):
    HR, SR = gram(Z, ZH, ZS, **kw)
    iu = np.triu_indices(Z.shape[1])
    for out, B in ((HR, ZH), (SR, ZS)):
        assert np.array_equal(out, out.T)
        bound = 2.0 ** -44 * (np.abs(Z).T @ np.abs(B)) + 1e-300
        assert np.all(np.abs(out - Z.T @ B)[iu] <= bound[iu])


@pytest.mark.parametrize("q,n", [(1, 1), (4, 3), (31, 63), (32, 64), (33, 65), (64, 129), (97, 5003)])
def test_gram_df64_tile_edges(q, n):
    check(*blocks(q, n, 100 + q))
