"""The scratch that a mixed solve reserves before its loop covers the double-float Gram and update of every width that
the loop reaches, in either form, so that nothing is reallocated in it.  Sizes from the host code, no GPU."""
import ctypes as C

import pytest

from paper_1308_2445_gb300 import hbsd


def size(symbol, *args):
    f = getattr(hbsd.lib(), symbol)
    f.restype = C.c_size_t
    return f(*args)


# rows and eigenpairs of the 8^3, 16^3, 32^3 and 64^3 problems, and of a large one with few columns
@pytest.mark.parametrize("n,m", [(646, 16), (4797, 64), (47620, 64), (47620, 17), (334272, 256), (3000000, 30)])
def test_reserved_scratch_covers_the_loop(n, m):
    n_ = C.c_int64(n)
    w = m + max(3, (m + 9) // 10)
    have = size("_ZN4hbsd18df64_solve_doublesEliii", n_, w, w + m, w)
    need = [size("_ZN4hbsd17gram_df64_doublesEli", n_, w + p) for p in range(m + 1)]
    need += [size("_ZN4hbsd19update_df64_doublesEliii", n_, w, p, w) for p in range(m + 1)]
    assert have == max(need)
    # the sums of a product alone: two matrices of one chunk of rows
    assert min(need[:m + 1]) >= 2 * w * w
