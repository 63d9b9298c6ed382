"""The two forms of the double-float Gram -- float pairs on the FP32 pipes, digit slices on the tensor
cores from n q^2 = 8e7 on -- at the edges of their tiles, stages and chunks, against FP64 products.

Bound: each entry within 2^-44 of |Z|^T |ZH|.  Pairs carry 48 bits and keep sums of 64 rows between FP64
flushes; the slices' truncation is held to the same level by the guard and the fix-up of the entries that
fail it.
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


@pytest.mark.parametrize("q,n", [(538, 300), (129, 5003), (161, 3200), (97, 8705), (71, 17001), (33, 80001)])
def test_gram_tensor_core_tile_edges(q, n):
    check(*blocks(q, n, 300 + q))


def test_gram_tensor_core_entries_below_the_guard():
    """Columns whose large entries lie in disjoint rows: the sum of |z||h| is then far below the product of
    the maxima, so these entries have to come from the fix-up (a few pairs) or the double-float tiles."""
    q, n = 130, 6000
    Z, ZH, ZS = blocks(q, n, 900)
    half = np.arange(n) < n // 2
    Z[half, 3] *= 1e-7          # one column against its counterparts in ZH, ZS
    ZH[~half, 40] *= 1e-8
    ZS[~half, 40] *= 1e-8
    check(Z, ZH, ZS)
    Z[half, :64] *= 1e-8        # half of the columns: whole tiles
    ZH[~half, 64:] *= 1e-8
    ZS[~half, 64:] *= 1e-8
    check(Z, ZH, ZS)


def test_gram_tensor_core_wild_magnitudes():
    """Entries over 24 decades without any row or column structure, and zero rows and columns."""
    q, n = 100, 9000
    Z, ZH, ZS = (pi.seed_normal_block(70 + i, n, q) * 10.0 ** (24.0 * pi.uniform(80 + i, 9, n * q).reshape(n, q) - 12.0)
                 for i in range(3))
    Z[100:140] = 0.0
    ZH[130:150] = 0.0
    Z[:, 7] = 0.0
    ZS[:, 8] = 0.0
    check(Z, ZH, ZS)


@pytest.mark.parametrize("bad", [np.inf, np.nan])
def test_gram_tensor_core_non_finite(bad):
    """A non-finite entry reaches the entries of its column and leaves the others as they are."""
    q, n = 130, 6000
    Z, ZH, ZS = blocks(q, n, 950)
    Z[4321, 50] = bad
    HR, SR = gram(Z, ZH, ZS)
    iu = np.triu_indices(q)
    hit = (iu[0] == 50)
    ok = Z.copy()
    ok[4321, 50] = 0.0
    for out, B in ((HR, ZH), (SR, ZS)):
        assert not np.isfinite(out[iu][hit]).any()
        bound = 2.0 ** -44 * (np.abs(ok).T @ np.abs(B)) + 1e-300
        assert np.all((np.abs(out - ok.T @ B) <= bound)[iu][~hit])


@pytest.mark.parametrize("n", [1, 31, 33, 646, 5003])
@pytest.mark.parametrize("q", [1, 23, 24, 25, 33, 48, 71, 73, 97])
def test_gram_fp64_tiles_and_chunks(q, n):
    """24 x 24 and 32 x 32 tiles, chunks of 32 rows and more: symmetric, and each entry within the rounding of its n
    products summed in any order (and of the mean with its mirror image)."""
    from paper_1308_2445_gb300 import hbsd
    Z, ZH, ZS = blocks(q, n, 1000 + q)
    bufs = []
    for a in (Z, ZH, ZS):
        t = torch.zeros(n, q + (q & 1), dtype=torch.float64, device="cuda")[:, :q]
        t.copy_(torch.from_numpy(a))
        bufs.append(t)
    HR, SR = (torch.zeros(q, q, dtype=torch.float64, device="cuda") for _ in range(2))
    hbsd.gram(*bufs, HR, SR)
    for out, B in ((HR.cpu().numpy(), ZH), (SR.cpu().numpy(), ZS)):
        assert np.array_equal(out, out.T)
        exact, mag = Z.T @ B, np.abs(Z).T @ np.abs(B)
        assert np.all(np.abs(out - 0.5 * (exact + exact.T)) <= 2.0 ** -53 * (n + 4) * (mag + mag.T))
