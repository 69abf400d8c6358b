"""The forms of the pivot blocks' explicit inverse -- 32, 16 or 8 columns of it per task in
shared memory, or 8 in global memory, which pivot blocks of more than 1536, 3072 and 6144
unknowns take -- on small fronts at the edges of their blocks.  The hook fills the inverse's
storage with NaNs first.  A column's sums have the same terms in the same order in every form, so
the bits are those of the 32-column form, which is checked against an FP64 elimination (the
bound of test_gpu_front_tiles: at most p rank-1 updates of 2^-24 relative)."""
import numpy as np
import pytest

from tests.test_gpu_front_factor import _errors, indefinite

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,p", [(1, 1), (9, 9), (31, 17), (33, 33), (65, 64), (97, 65), (130, 104), (200, 129),
                                 (321, 225), (420, 400)])
def test_inverse_forms(n, p):
    from paper_2106_05306_gb300 import front_factor
    A = indefinite(n, 5 * n + p)
    F, X = front_factor(A, p, threads=512)
    e_piv, e_tr, e_inv, upper_zero = _errors(A, p, F, X)
    tol = (p + 8) * 2.0 ** -22
    assert upper_zero and e_piv <= tol and e_tr <= tol and e_inv <= tol, (e_piv, e_tr, e_inv, tol)
    for kw in (dict(threads=256), dict(threads=128), dict(use_gscr=True)):
        F2, X2 = front_factor(A, p, **kw)
        assert np.array_equal(F, F2) and np.array_equal(X, X2), kw
