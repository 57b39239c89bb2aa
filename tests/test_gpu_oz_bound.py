"""The digit-sliced product's stated bound on the data that come closest to it."""
from fractions import Fraction

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("k", [1, 16, 700, 5000])
def test_worst_digits(k):
    """Entries x (1 -+ i), x the number just above one half whose seven base-128
    digits are 64, 63, ..., 63 (all the dropped digit products as large and of
    one sign): 2^-45.1 k max|A| max|B|, within the bound of 1.25 x 2^-45 in each
    component and beyond the 2^-48 of random data."""
    import paper_1404_1768_gb300 as fg
    x = 0.5038754921259841
    A, B = np.full((2, k), x * (1 - 1j)), np.full((k, 3), x * (1 + 1j))
    C = fg.zgemm_oz(A, B)
    exact = 2 * k * Fraction(x) ** 2
    for c in C.ravel():
        re, im = abs(Fraction(float(c.real)) - exact), abs(Fraction(float(c.imag)))
        assert max(re, im) <= Fraction(5, 4) / 2 ** 45 * k * Fraction(x) ** 2
        assert re >= k * Fraction(x) ** 2 / 2 ** 46
