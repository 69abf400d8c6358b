"""The front factorisation at the edges of its tiles: 32-column panels, 96 rows per
panel CTA, 64 x 64 and (tensor cores) 128 x 64 update tiles, pivot blocks whose inverse
takes 32 or 16 columns per CTA, and their remainders, against an FP64 elimination.

Tolerance: every entry is the result of at most p rank-1 updates, each rounded to
2^-24 of terms no larger than the front's largest entry times a small growth
factor on these diagonally dominant fronts, so (p + 8) 2^-22 of the largest
entry bounds it with a factor of four to spare."""
import numpy as np
import pytest

from tests.test_gpu_front_factor import _errors, indefinite

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("tc", [False, True])
@pytest.mark.parametrize("n,p", [(1, 1), (2, 1), (31, 31), (32, 32), (33, 32), (33, 33), (65, 64), (96, 96), (97, 65),
                                 (128, 32), (129, 32), (160, 64), (161, 97), (192, 192), (193, 129), (256, 1),
                                 (321, 225), (900, 300),
                                 (1700, 1600)])
def test_front_tiles(n, p, tc):
    from paper_2106_05306_gb300 import front_factor
    A = indefinite(n, 7 * n + p)
    F, Linv = front_factor(A, p, use_tc=tc, use_gscr=n > 1000)
    tol = (p + 8) * 2.0 ** -22
    e_piv, e_tr, e_inv, upper_zero = _errors(A, p, F, Linv)
    assert upper_zero
    assert e_piv <= tol and e_tr <= tol and e_inv <= tol, (e_piv, e_tr, e_inv, tol)
