"""Rayleigh-Ritz over the whole GPU (from 20 columns on) at the edges of its 32-column blocks, 16 rows per
cluster round and 16 x 16 tiles, against the oracle.

Tolerances as for the other sizes: eigenvalues to 1e-11 of the largest (the solver's own bar is 1e-9),
W^T S_R W = I and W^T H_R W = diag(theta) to 1e-10, which FP64 reaches with room on pencils whose scaled S_R
has a condition number of up to 1e6 (1e-16 * 1e6).
"""
import numpy as np
import pytest

from oracle import labpsd as L

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def run(HR, SR, k):
    from paper_1308_2445_gb300 import hbsd
    dev = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()
    th = torch.zeros(k, dtype=torch.float64, device="cuda")
    W = torch.zeros(HR.shape[0], k, dtype=torch.float64, device="cuda")
    info = torch.zeros(2, dtype=torch.int32, device="cuda")
    hbsd.rayleigh_ritz(dev(HR), dev(SR), k, th, W, info)
    torch.cuda.synchronize()
    return th.cpu().numpy(), W.cpu().numpy(), info.cpu().numpy()


def pencil(q, cond, seed):
    """Spectrum of shells of up to 8 equal eigenvalues, S_R of the given condition, columns of many sizes."""
    rng = np.random.default_rng(seed)
    lam = np.repeat(np.cumsum(0.5 + rng.random(q)), rng.integers(1, 9, q))[:q]
    U, V = (np.linalg.qr(rng.standard_normal((q, q)))[0] for _ in range(2))
    G = (U * np.sqrt(np.logspace(0, -np.log10(cond), q))) @ V
    G *= 10.0 ** rng.uniform(-3, 2, q)
    HR, SR = G.T @ (lam[:, None] * G), G.T @ G
    return 0.5 * (HR + HR.T), 0.5 * (SR + SR.T)


@pytest.mark.parametrize("q,k", [(20, 1), (21, 21), (31, 7), (32, 32), (33, 20), (48, 47), (63, 33), (64, 16), (65, 65),
                                 (97, 96), (129, 40), (161, 161), (260, 31)])
def test_block_edges(q, k):
    HR, SR = pencil(q, 1e3, q)
    th, W, info = run(HR, SR, k)
    g, _, fb = L.rayleigh_ritz(HR, SR, k)
    assert info[0] == 0 and info[1] == q and not fb
    scale = np.abs(g).max()
    assert np.abs(th - g).max() <= 1e-11 * scale and np.all(np.diff(th) >= 0)
    assert np.abs(W.T @ SR @ W - np.eye(k)).max() <= 1e-10
    assert np.abs(W.T @ HR @ W - np.diag(th)).max() <= 1e-10 * scale


def test_ill_conditioned_and_one_shell():
    HR, SR = pencil(150, 1e6, 5)
    th, W, info = run(HR, SR, 85)
    g, _, _ = L.rayleigh_ritz(HR, SR, 85)
    assert info[0] == 0 and np.abs(th - g).max() <= 1e-9 * np.abs(g).max()
    assert np.abs(W.T @ SR @ W - np.eye(85)).max() <= 1e-8
    # every eigenvalue the same: T is diagonal, the vectors are anything orthonormal
    q = 70
    th, W, _ = run(3.0 * np.eye(q), np.eye(q), 40)
    assert np.abs(th - 3.0).max() <= 1e-13
    assert np.abs(W.T @ W - np.eye(40)).max() <= 1e-12


@pytest.mark.parametrize("q,k,ndep", [(64, 30, 2), (150, 85, 5)])
def test_dependent_columns_reach_the_rank_revealing_branch(q, k, ndep):
    HR, SR = pencil(q, 10.0, 3 * q)
    C = np.eye(q)
    for t in range(ndep):
        C[:, q - 1 - t] = C[:, t] - 0.5 * C[:, t + 1]
    HR, SR = C.T @ HR @ C, C.T @ SR @ C
    HR, SR = 0.5 * (HR + HR.T), 0.5 * (SR + SR.T)
    th, _, info = run(HR, SR, k)
    g, _, fb = L.rayleigh_ritz(HR, SR, k)
    assert fb and info[0] == 1 and info[1] == q - ndep
    assert np.abs(th - g).max() <= 1e-8 * np.abs(g).max()


@pytest.mark.parametrize("q,first,later", [(260, 5, 120), (150, 31, 40), (400, 1, 399)])
def test_dependent_columns_in_an_early_panel(q, first, later):
    """The first failing pivot lies in a panel that many CTAs factor at once: all of them leave it, and the rank-revealing
    branch takes over."""
    HR, SR = pencil(q, 10.0, 7 * q)
    C = np.eye(q)
    C[:, first] = C[:, 0] if first == 1 else C[:, 2] - 0.5 * C[:, 3]
    C[:, later] = C[:, 8] + C[:, 9]
    HR, SR = C.T @ HR @ C, C.T @ SR @ C
    HR, SR = 0.5 * (HR + HR.T), 0.5 * (SR + SR.T)
    k = 20
    th, _, info = run(HR, SR, k)
    g, _, fb = L.rayleigh_ritz(HR, SR, k)
    assert fb and info[0] == 1 and info[1] == q - 2
    assert np.abs(th - g).max() <= 1e-8 * np.abs(g).max()


@pytest.mark.parametrize("q,small,dep", [(12, 5e-9, 0), (20, 3e-9, 0), (40, 1e-9, 0), (150, 5e-10, 0), (40, 1e-10, 1)])
def test_nearly_tridiagonal(q, small, dep):
    """A nearly tridiagonal pencil: what lies outside the three diagonals is below 1e-8 of a row's largest entry, and has
    to be eliminated, not dropped.  The vectors diagonalise H_R and S_R to the rounding of a few hundred FP64
    operations (1e-12 of the largest entry).  S_R = I; dep: nearly tridiagonal as well, with one column twice, which the
    rank-revealing kernel reduces first."""
    rng = np.random.default_rng(q)

    def matrix(off, diag):
        A = np.triu(small * rng.uniform(0.5, 1.0, (q, q)), 2) + np.diag(np.full(q - 1, off), 1)
        return A + A.T + np.diag(diag)

    H, S, C = matrix(1.0, np.arange(q) / 4.0), np.eye(q), np.eye(q)
    if dep:
        S, C = matrix(0.3, np.ones(q)), np.hstack([C, C[:, -1:]])
    k = q // 2
    th, W, info = run(C.T @ H @ C, C.T @ S @ C, k)
    scale = np.abs(np.linalg.eigvalsh(H)).max()
    assert info[0] == dep and info[1] == q
    Li = np.linalg.inv(np.linalg.cholesky(S))
    g = np.linalg.eigvalsh(Li @ H @ Li.T)[:k]
    V = C @ W
    assert np.abs(th - g).max() <= 1e-12 * scale
    assert np.abs(V.T @ S @ V - np.eye(k)).max() <= 1e-12
    assert np.abs(V.T @ H @ V - np.diag(th)).max() <= 1e-12 * scale
    assert np.abs(H @ V - S @ V * th).max() <= 1e-12 * scale


def test_entries_too_small_to_square():
    """Rows whose remaining entries have squares below the normal range, and a NaN among them: zeros to the first, and the
    second is not lost (the call must not return finite pairs)."""
    q = 40
    H = np.diag(np.arange(q) / 4.0) + np.diag(np.ones(q - 1), 1) + np.diag(np.ones(q - 1), -1)
    tiny = np.triu(np.full((q, q), 1e-160), 2)
    th, W, _ = run(H + tiny + tiny.T, np.eye(q), 10)
    assert np.abs(th - np.linalg.eigvalsh(H)[:10]).max() <= 1e-12 * 11
    assert np.abs(W.T @ W - np.eye(10)).max() <= 1e-12
    th, W, _ = run(np.diag(np.arange(q) / 4.0) + tiny + tiny.T, np.eye(q), 10)   # x0 = 0 as well
    assert np.abs(th - np.arange(10) / 4.0).max() <= 1e-12 * 11
    H[20, 30] = H[30, 20] = np.nan
    from paper_1308_2445_gb300 import hbsd
    try:
        th, W, _ = run(H, np.eye(q), 10)
    except hbsd.HbsdError:
        return
    assert not (np.isfinite(th).all() and np.isfinite(W).all())


def test_trace_output():
    """HBSD_TRACE prints the phases of a call and HBSD_RRDBG=2 a line per vector, whichever kernels ran."""
    import os
    import subprocess
    import sys
    code = ("import numpy as np, torch\nfrom paper_1308_2445_gb300 import hbsd\n"
            "for q in (12, 64):\n"
            "    H = torch.diag(torch.arange(q, dtype=torch.float64)).cuda() + 0.01\n"
            "    S = torch.eye(q, dtype=torch.float64, device='cuda')\n"
            "    th, W = (torch.zeros(s, dtype=torch.float64, device='cuda') for s in ((9,), (q, 9)))\n"
            "    hbsd.rayleigh_ritz(H, S, 9, th, W, torch.zeros(2, dtype=torch.int32, device='cuda'))\n")
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    r = subprocess.run([sys.executable, "-c", code], cwd=root, env=dict(os.environ, HBSD_TRACE="1", HBSD_RRDBG="2"),
                       capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stderr
    assert r.stderr.count("RR vec") == 2 * 9
    for q in (12, 64):
        line = [x for x in r.stderr.splitlines() if f"RR q {q} k 9" in x]
        assert len(line) == 1
        for phase in ("chol", "C", "tridiag", "eig", "rqi", "cholqr", "back"):
            assert f" {phase} " in line[0]


@pytest.mark.parametrize("q,k", [(640, 40), (2200, 24)])
def test_rows_and_iterates_in_global_memory(q, k):
    """From 625 columns on the rows of the tridiagonalisation leave shared memory, from 2,134 on the inverse iteration's
    scratch does.  S_R diagonal, so that the reference is one standard eigenproblem; tolerances as above."""
    rng = np.random.default_rng(q)
    B = rng.standard_normal((q, q))
    B = np.diag(np.arange(q) * 1.0) + (B + B.T) / np.sqrt(q)
    d = 10.0 ** rng.uniform(-2, 2, q)
    HR, SR = d[:, None] * B * d, np.diag(d * d)
    HR = 0.5 * (HR + HR.T)
    th, W, info = run(HR, SR, k)
    g = np.linalg.eigvalsh(B)
    scale = np.abs(g).max()
    assert info[0] == 0 and info[1] == q
    assert np.abs(th - g[:k]).max() <= 1e-11 * scale
    assert np.abs(W.T @ SR @ W - np.eye(k)).max() <= 1e-10
    assert np.abs(W.T @ HR @ W - np.diag(th)).max() <= 1e-10 * scale
