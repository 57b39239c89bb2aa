"""The test basis U2 R2 = B U1 (Cholesky QR whose first factorisation is FP32
from 33 columns on) over the conditions of B U1 that this first factorisation
takes: U2 must be orthonormal to the accuracy of the FP64 form whatever
the first pass leaves to be corrected."""
import numpy as np
import pytest

from paper_1404_1768_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,m0", [(128, 33), (128, 64), (256, 120), (512, 250)])
@pytest.mark.parametrize("logcond", [0.3, 2.0, 3.2, 3.6, 4.0, 4.6])
def test_orthonormal(n, m0, logcond):
    """The last Gram matrix measured carries 2^-48 n of digit slicing times the
    square of the columns' largest entry (about (4 / sqrt(n))^2): 2^-44, twice for
    the correction made from it and the final rounding."""
    import paper_1404_1768_gb300 as fg
    rng = np.random.default_rng(n + m0)
    U = np.linalg.qr(inputs.complex_normal(rng, (n, n)))[0]
    B = (U * np.logspace(0, -logcond, n)) @ np.linalg.qr(inputs.complex_normal(rng, (n, n)))[0]
    U1 = np.linalg.qr(inputs.complex_normal(rng, (n, m0)))[0]
    g = fg.Feast(B, B, U1.copy(), prec=fg.FEAST_C64_REFINE, q=8, center=0j, a=1.0)
    g.set_subspace(U1)
    U2, R2 = g.get("U2"), g.get("R2")
    g.close()
    assert np.abs(U2.conj().T @ U2 - np.eye(m0)).max() <= 2.0 ** -43
    # n roundings of the digit-sliced products on B's norm of 1
    assert np.abs(U2 @ R2 - B @ U1).max() <= n * 2.0 ** -48
