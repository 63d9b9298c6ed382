"""The two forms of the double-float update -- float pairs on the FP32 pipes, digit slices on the tensor cores
from n >= 6144, k >= 56, n q k >= 2e8 on -- at the edges of their tiles, phases and slabs, against FP64 products.

Bound: each entry within 2^-44 of |Z| |W|.  Pairs carry 48 bits, renormalised every 8 terms; the slices'
truncation is held to the same level by the guard, whose failing entries are computed in FP64.
"""
import numpy as np
import pytest

from paper_1308_2445_gb300 import pufe_inputs as pi

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def blocks(n, q, k, seed):
    """Columns of Z of different sizes, rows over eight decades; W's rows and columns over a few."""
    Z = pi.seed_normal_block(seed, n, q) * 10.0 ** (8.0 * pi.uniform(seed, 9, n))[:, None] * np.logspace(-4, 2, q)
    W = pi.seed_normal_block(seed + 1, q, k) * np.logspace(3, -3, q)[:, None] * np.logspace(0, 2, k)
    return Z, W


def update(Z, W, ld=None, off=0):
    """Z(:, :k) := Z W on the device, Z at an offset of off doubles with leading dimension ld."""
    from paper_1308_2445_gb300 import hbsd
    n, q = Z.shape
    ld = ld or q + (q & 1)
    buf = torch.zeros(n * ld + off, dtype=torch.float64, device="cuda")
    t = buf[off:].view(n, ld)[:, :q]
    t.copy_(torch.from_numpy(Z))
    hbsd.update_df64(t, torch.from_numpy(W).cuda(), W.shape[1])
    torch.cuda.synchronize()
    return t.cpu().numpy()


def check(Z, W, **kw):
    k = W.shape[1]
    out = update(Z, W, **kw)
    assert np.array_equal(out[:, k:], Z[:, k:])
    assert np.all(np.abs(out[:, :k] - Z @ W) <= 2.0 ** -44 * (np.abs(Z) @ np.abs(W)) + 1e-300)


# one and more column tiles, phases of 16 steps with and without a remainder, an odd number of steps, two slabs,
# the largest k
@pytest.mark.parametrize("n,q,k", [(38913, 100, 56), (40011, 97, 57), (32769, 96, 64), (20001, 160, 65), (12161, 256, 128),
                                   (6145, 257, 129), (65537, 113, 64), (25001, 539, 282), (6144, 514, 512)])
def test_update_tensor_core_tile_edges(n, q, k):
    check(*blocks(n, q, k, 500 + q))


@pytest.mark.parametrize("kw", [dict(ld=161), dict(off=1), dict(ld=170), dict(off=2, ld=164)])
def test_update_strides_and_alignment(kw):
    """Odd strides and 8-byte alignment stay with the pairs; even ones with a gap take the tensor cores."""
    check(*blocks(9001, 160, 140, 600), **kw)


@pytest.mark.parametrize("n,q,k", [(6144, 513, 513), (6143, 257, 129), (60001, 97, 55)])
def test_update_just_outside_the_rule(n, q, k):
    check(*blocks(n, q, k, 650))


def test_update_entries_below_the_guard():
    """Rows of Z whose large entries meet small entries of W: a few rows, then half of the entries."""
    n, q, k = 12001, 170, 100
    Z, W = blocks(n, q, k, 700)
    Z[5:90, :80] *= 1e-9
    W[80:, 30] *= 1e-9
    check(Z, W)
    Z[: n // 2, :80] *= 1e-9
    W[80:, :64] *= 1e-9
    check(Z, W)


def test_update_wild_magnitudes():
    """Entries over 24 decades without structure, and zero rows and columns in both factors."""
    n, q, k = 12001, 170, 100
    wild = [10.0 ** (24.0 * pi.uniform(800 + i, 9, m).reshape(-1, c) - 12.0) for i, m, c in ((0, n * q, q), (1, q * k, k))]
    Z, W = pi.seed_normal_block(801, n, q) * wild[0], pi.seed_normal_block(802, q, k) * wild[1]
    Z[100:140] = 0.0
    Z[:, 7] = 0.0
    W[20] = 0.0
    W[:, 9] = 0.0
    check(Z, W)


@pytest.mark.parametrize("bad", [np.inf, np.nan])
def test_update_non_finite(bad):
    """A non-finite entry of Z reaches its row, one of W its column, and nothing else."""
    n, q, k = 12001, 170, 100
    Z, W = blocks(n, q, k, 900)
    exact, bound = Z @ W, 2.0 ** -44 * (np.abs(Z) @ np.abs(W)) + 1e-300
    hit = np.zeros((n, k), bool)
    Z[4321, 50] = bad
    W[60, 11] = bad
    hit[4321] = True
    hit[:, 11] = True
    out = update(Z, W)[:, :k]
    assert not np.isfinite(out[hit]).any()
    assert np.all((np.abs(out - exact) <= bound)[~hit])


@pytest.mark.parametrize("n,q,k", [(1, 1, 1), (15, 3, 3), (17, 40, 16), (33, 70, 63), (16, 90, 64), (47, 66, 65), (100, 140, 130)])
def test_update_fp64_columns(n, q, k):
    """The FP64 form's items (four rows, a column) at the edges of warps, CTAs and rows: the rounding of q products."""
    from paper_1308_2445_gb300 import hbsd
    Z, W = blocks(n, q, k, 1100 + q)
    t = torch.zeros(n, q + (q & 1), dtype=torch.float64, device="cuda")[:, :q]
    t.copy_(torch.from_numpy(Z))
    hbsd.update(t, torch.from_numpy(W).cuda(), k)
    out = t.cpu().numpy()
    assert np.array_equal(out[:, k:], Z[:, k:])
    assert np.all(np.abs(out[:, :k] - Z @ W) <= 2.0 ** -53 * 2 * (q + 2) * (np.abs(Z) @ np.abs(W)))


@pytest.mark.parametrize("n,q,k,most", [(12288, 170, 100, 7.2), (6144, 538, 282, 7.6)])
def test_update_entries_just_above_the_guard(n, q, k, most):
    """sum |z||w| from 2^2 down to the guard's line, sqrt(q) 2^-11 of the product P of the row's and the column's leading
    powers of two: one entry of about 1 in each row of Z and each column of W, at indices that do not meet, the
    others smaller by up to 2^most, half of the rows and columns of one sign.  Bound 2^-46 of |Z| |W|: the sums of the
    lowest levels are rounded to 2^-56 P once per 256 terms and the operands to 2^-62 of their maxima, 2^-49 of the
    line, and the largest of a million entries may be 8 times the usual one."""
    rng = np.random.default_rng(q)
    m, w = np.exp2(-np.linspace(1.0, most, n)), np.exp2(-np.linspace(1.0, most, k))
    Z = m[:, None] * rng.uniform(0.5, 1.5, (n, q)) * np.where(np.arange(n) % 2, 1.0, rng.choice([-1.0, 1.0], (q, n))).T
    W = w * rng.uniform(0.5, 1.5, (q, k)) * np.where(np.arange(k) % 2, 1.0, rng.choice([-1.0, 1.0], (q, k)))
    Z[:, 0], Z[:, 1] = 1.3, 0.0
    W[0], W[1] = 0.0, 1.7
    W[:, 0] = 1.0     # the same scale for every row of W
    out = update(Z, W)[:, 1:k]
    exact, mag = (Z @ W)[:, 1:], (np.abs(Z) @ np.abs(W))[:, 1:]
    rel = (np.abs(out - exact) / mag).max()
    assert rel <= 2.0 ** -46, np.log2(rel)


# q k below and from 7,200 on, waves of row tiles filled and not, n q k below and from 3e8 on: pairs, slices, pairs, slices,
# pairs, slices; then column tiles of one column, q one more and one less than whole steps of 16
@pytest.mark.parametrize("n,q,k", [(37001, 100, 71), (37001, 100, 72), (40001, 100, 72), (44003, 100, 90), (23003, 128, 90),
                                   (28003, 128, 90), (38913, 129, 90), (40003, 175, 57), (40013, 113, 90), (12289, 257, 65),
                                   (37005, 111, 65)])
def test_update_around_the_rule_of_narrow_blocks(n, q, k):
    check(*blocks(n, q, k, 1300 + q))


def test_update_captured_after_fewer_rows():
    """A captured call allocates nothing after a call of fewer rows, of either form, and an uncaptured call of more rows
    leaves the graph's scratch where it is.  Bound as above."""
    import threading
    from paper_1308_2445_gb300 import hbsd
    errors = []

    def work():   # a thread of its own: the scratch of these calls is kept per thread
        try:
            side = torch.cuda.Stream()
            with torch.cuda.stream(side):
                for q, k, n0, n1, n2 in ((160, 140, 100, 9000, 30000), (160, 140, 9000, 9500, 40000)):
                    W = torch.randn(q, k, dtype=torch.float64, device="cuda")
                    small, Z, large = (torch.randn(n, q, dtype=torch.float64, device="cuda") for n in (n0, n1, n2))
                    Z0, L0 = Z.clone(), large.clone()
                    hbsd.update_df64(small, W, k, stream=side.cuda_stream)
                    side.synchronize()
                    g = torch.cuda.CUDAGraph()
                    with torch.cuda.graph(g, stream=side):
                        hbsd.update_df64(Z, W, k, stream=side.cuda_stream)
                    hbsd.update_df64(large, W, k, stream=side.cuda_stream)
                    g.replay()
                    side.synchronize()
                    for A, B in ((Z0, Z), (L0, large)):
                        assert ((B[:, :k] - A @ W).abs() <= 2.0 ** -44 * (A.abs() @ W.abs())).all()
        except Exception as e:   # noqa: BLE001 - handed to the test
            errors.append(e)

    t = threading.Thread(target=work)
    t.start()
    t.join()
    assert not errors, errors[0]
