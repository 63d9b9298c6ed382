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


def rows_at_the_line(n, q, most, tail, seed):
    """Columns with one entry of about 1 in every block of 256 rows, in another row for Z than for ZH and ZS, and entries
    of 2^-1 .. 2^-most in one row in 16, where alone Z and ZH, ZS meet: sum |z||h| then goes down to the guard's line,
    sqrt(rows) 2^-11 of the product of the maxima.  The last columns fix the rows' scales and make these rows those that
    the guard looks at.  Half of the columns have one sign.  tail: the other rows hold large entries of Z against
    2^-50 ones of ZH, ZS, whose rounding to 62 bits all go the same way if they are cut."""
    rng = np.random.default_rng(seed)
    i = np.arange(n)
    heavy = i % 16 == 3
    mag = np.exp2(-np.linspace(1.0, most, q))
    out = []
    for m in range(3):
        A = np.zeros((n, q))
        if tail:
            A[:] = 1.9 if m == 0 else 2.0 ** -50 * rng.uniform(0.5, 1.0, (n, q))
        A[heavy] = mag * rng.uniform(0.5, 1.5, (int(heavy.sum()), q))
        A[heavy] *= np.where(np.arange(q) % 2, 1.0, rng.choice([-1.0, 1.0], (int(heavy.sum()), q)))
        A[i % 256 == (0 if m == 0 else 1)] = 1.3 if m == 0 else 1.7
        A[i % 256 == (1 if m == 0 else 0)] = 0.0
        A[:, -1] = 1.9 if m == 0 else np.where(heavy, 64.0, 1.0)
        out.append(A)
    return out


# most: where 16 of 256 rows (128 of 2,048) leave sum |z||h| at about the line for the smallest pair of columns
@pytest.mark.parametrize("n,most,tail", [(6000, 5.4, False), (48000, 6.2, False), (48000, 6.2, True)])
def test_gram_tensor_core_entries_just_above_the_guard(n, most, tail):
    """Entries that the guard accepts at its line.  Bound 2^-46 of |Z|^T |ZH|: with P the product of the columns' leading
    powers of two and R rows, the sums of the lowest levels are rounded to 2^-56 P once per 256 rows, and rounding
    the operands to 2^-62 of their maxima leaves sqrt(R) 2^-60 P; against the line that is 2^-49, and the largest of
    some ten thousand entries may be 6 times the usual one.  Pairs stay within 2^-47 on such columns."""
    q = 130
    Z, ZH, ZS = rows_at_the_line(n, q, most, tail, 77)
    HR, SR = gram(Z, ZH, ZS)
    iu = np.triu_indices(q - 1)
    for out, B in ((HR, ZH), (SR, ZS)):
        mag = np.abs(Z).T @ np.abs(B)
        rel = (np.abs(out - Z.T @ B) / mag)[iu]
        assert rel.max() <= 2.0 ** -46, np.log2(rel.max())


@pytest.mark.parametrize("q,n", [(47, 40001), (48, 34721), (48, 34817), (49, 33537), (64, 20225), (65, 19201)])
def test_gram_on_both_sides_of_the_width_rule(q, n):
    """Pairs below 48 columns whatever the rows, and below n q^2 = 8e7; digit slices above, with nearly empty second
    tiles of 32 and of 128 columns."""
    check(*blocks(q, n, 400 + q))


def test_gram_scratch_covers_every_row_count():
    """hbsd_gram's scratch depends on the width alone: after one call of a few rows, calls of any height at
    widths of as many 32-column tiles can be captured (nothing is allocated)."""
    import threading
    from paper_1308_2445_gb300 import hbsd
    errors = []

    def work():   # a thread of its own: the scratch of these calls is kept per thread
        try:
            side = torch.cuda.Stream()
            with torch.cuda.stream(side):
                for q in (24, 72, 144, 358):
                    dev = lambda n: torch.randn(n, q, dtype=torch.float64, device="cuda")
                    HR, SR = (torch.zeros(q, q, dtype=torch.float64, device="cuda") for _ in range(2))
                    small, Z = dev(64), dev(90000 if q < 300 else 20000)
                    hbsd.gram(small, small, small, HR, SR, stream=side.cuda_stream)
                    side.synchronize()
                    g = torch.cuda.CUDAGraph()
                    with torch.cuda.graph(g, stream=side):
                        hbsd.gram(Z, Z, Z, HR, SR, stream=side.cuda_stream)
                    g.replay()
                    side.synchronize()
                    exact = Z.T @ Z
                    assert (HR - exact).abs().max() <= 1e-12 * exact.abs().max()
        except Exception as e:   # noqa: BLE001 - handed to the test
            errors.append(e)

    t = threading.Thread(target=work)
    t.start()
    t.join()
    assert not errors, errors[0]


def test_gram_df64_captured_after_fewer_rows():
    """A captured call allocates nothing after a call of fewer rows -- of either form, with as many rows as give every
    SM its CTAs --, and an uncaptured call of more rows leaves the graph's scratch where it is.  Bound as above."""
    import threading
    from paper_1308_2445_gb300 import hbsd
    errors = []

    def work():   # a thread of its own: the scratch of these calls is kept per thread
        try:
            side = torch.cuda.Stream()
            with torch.cuda.stream(side):
                for q, n0, n1, n2 in ((149, 25000, 47620, 90000), (40, 104000, 120000, 160000), (149, 3000, 2900, 30000)):
                    dev = lambda n: torch.randn(n, q, dtype=torch.float64, device="cuda")
                    HR, SR, H2, S2 = (torch.zeros(q, q, dtype=torch.float64, device="cuda") for _ in range(4))
                    small, Z, large = dev(n0), dev(n1), dev(n2)
                    hbsd.gram_df64(small, small, small, HR, SR, stream=side.cuda_stream)
                    side.synchronize()
                    g = torch.cuda.CUDAGraph()
                    with torch.cuda.graph(g, stream=side):
                        hbsd.gram_df64(Z, Z, Z, HR, SR, stream=side.cuda_stream)
                    hbsd.gram_df64(large, large, large, H2, S2, stream=side.cuda_stream)
                    g.replay()
                    side.synchronize()
                    for A, B, C in ((Z, HR, SR), (large, H2, S2)):
                        exact, bound = A.T @ A, 2.0 ** -44 * (A.abs().T @ A.abs())
                        assert ((B - exact).abs() <= bound).all() and ((C - exact).abs() <= bound).all()
        except Exception as e:   # noqa: BLE001 - handed to the test
            errors.append(e)

    t = threading.Thread(target=work)
    t.start()
    t.join()
    assert not errors, errors[0]
