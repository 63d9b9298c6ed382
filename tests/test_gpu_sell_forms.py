"""The stored pencil, filled on the device, and its products at the edges of their splits, against CSR products:
rows of 0 to 60 entries with and without a diagonal, slices that are not full, rows split over 8, 4, 2 and 1 groups of
lanes, one and several passes of columns, new H values on the pattern.

Bounds, per entry: FP64 (len + 4) 2^-53 |A| |X|; FP32 (len + 4) 2^-24 |DAD| |X|; double-float 2^-44 |A| |X|.
"""
import numpy as np
import pytest

from paper_1308_2445_gb300 import pufe_inputs as pi

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
sp = pytest.importorskip("scipy.sparse")

SIGMA = -0.37


def pattern(n, seed):
    """Row lengths 0 to 60, sorted columns; every third row without its diagonal entry."""
    u = pi.uniform(seed, 1, n)
    rows = []
    for i in range(n):
        c = np.unique((pi.uniform(seed + 7 * i + 1, 2, int(60 * u[i] ** 3)) * n).astype(np.int64))
        c = c[c != i] if i % 3 == 0 else np.union1d(c, [i])
        rows.append(c[c < n])
    rp = np.concatenate([[0], np.cumsum([len(c) for c in rows])]).astype(np.int64)
    return rp, np.concatenate(rows).astype(np.int32)


def make(n, seed):
    from paper_1308_2445_gb300 import hbsd
    rp, ci = pattern(n, seed)
    rows = np.repeat(np.arange(n), np.diff(rp))
    h, h2, s = (pi.seed_normal_block(seed + i, max(ci.size, 1), 1)[:ci.size, 0] for i in range(3))
    s[rows == ci] = np.abs(s[rows == ci]) + 0.1
    nodes = (np.arange(n) % 8).astype(np.int32)
    ses = hbsd.Session(n, rp, ci, h, s, nodes, (2, 2, 2), SIGMA, precond=hbsd.PRECOND_LOCAL, precision=hbsd.PRECISION_MIXED)
    # h - sigma s rounded once: two roundings would be off by 2^-53 (|h| + |sigma s|), which cancellation can make many
    # times 2^-53 of the difference
    once = [(v.astype(np.longdouble) - np.longdouble(SIGMA) * s).astype(np.float64) for v in (h, h2)]
    csr = [sp.csr_matrix((v, ci, rp), shape=(n, n)) for v in (*once, s)]
    d = np.ones(n)
    d[rows[rows == ci]] = 1.0 / np.sqrt(s[rows == ci])
    return ses, h2, csr, d, np.diff(rp)[:, None]


def dev(a, dtype=torch.float64):
    t = torch.zeros(a.shape[0], (a.shape[1] + 3) // 4 * 4, dtype=dtype, device="cuda")[:, :a.shape[1]]
    t.copy_(torch.from_numpy(a))
    return t


def check(ses, H, S, d, length, X, e):
    Xd, Y, Z = dev(X), dev(0 * X), dev(0 * X)
    ses.spmm_pair(Xd, Y, Z)
    for out, A in ((Y, H), (Z, S)):
        assert np.all(np.abs(out.cpu().numpy() - A @ X) <= (length + 4) * 2.0 ** -53 * (abs(A) @ np.abs(X)) * 2)
    ses.spmm_shifted(Xd, torch.from_numpy(e).cuda(), Y)
    mag = abs(H) @ np.abs(X) + np.abs(e) * (abs(S) @ np.abs(X))
    assert np.all(np.abs(Y.cpu().numpy() - (H @ X - e * (S @ X))) <= (length + 4) * 2.0 ** -53 * mag * 2)
    ses.spmm_pair_df64(Xd, Y, Z)
    for out, A in ((Y, H), (Z, S)):
        assert np.all(np.abs(out.cpu().numpy() - A @ X) <= 2.0 ** -44 * (abs(A) @ np.abs(X)))
    X32 = X.astype(np.float32).astype(np.float64)
    Xf, Yf, Zf = (dev(a, torch.float32) for a in (X32, 0 * X, 0 * X))
    ses.spmm_pair_f32(Xf, Yf, Zf)
    D = sp.diags(d)
    for out, A in ((Yf, D @ H @ D), (Zf, D @ S @ D)):
        assert np.all(np.abs(out.cpu().numpy() - A @ X32) <= (length + 4) * 2.0 ** -24 * (abs(A) @ np.abs(X32)) * 2)


@pytest.mark.parametrize("n,ks", [(1, (1, 3)), (7, (2, 9)), (33, (1, 5)), (1024, (4, 8, 17, 33)), (1025, (9, 85)), (2049, (3, 25)),
                                  (4097, (1, 19, 64)), (19449, (1, 2, 7, 23, 43, 85, 149))])
def test_products_at_the_edges_of_the_splits(n, ks):
    ses, h2, (H, H2, S), d, length = make(n, 40 + n)
    assert np.allclose(ses.dscale(), d, rtol=4e-16, atol=0)
    for k in ks:
        check(ses, H, S, d, length, pi.seed_normal_block(k, n, k), pi.uniform(k, 3, k))
    ses.update_H(h2)
    check(ses, H2, S, d, length, pi.seed_normal_block(77, n, ks[-1]), pi.uniform(78, 3, ks[-1]))
    ses.close()
