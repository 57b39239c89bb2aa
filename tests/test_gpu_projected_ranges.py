"""The projected eigensolve (feast_zqz_batched, and line 6 of a solve) away from
entries of order one: pencils scaled by powers of two, spectra that are narrow
against their distance from the origin, weakly coupled and ill-conditioned
eigenvectors."""
import numpy as np
import pytest

from paper_1404_1768_gb300 import inputs
from test_gpu_projected import _check, _pencil

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("m", [66, 234])
@pytest.mark.parametrize("ea,eb", [(-36, 24), (24, -36), (-60, 0), (60, 0), (0, 60), (-60, -60), (90, -60), (400, 400)])
def test_scaled(m, ea, eb):
    """Powers of two change neither the eigenvectors nor, but for their exponent,
    the eigenvalues: the bounds of the unscaled pencil."""
    rng = np.random.default_rng(m)
    lam = 2 * np.sqrt(rng.random(m)) * np.exp(2j * np.pi * rng.random(m))
    A, B = _pencil(rng, m, lam)
    _check(A * 2.0 ** ea, B * 2.0 ** eb, lam * 2.0 ** (ea - eb), 32 * m * 2.0 ** -53)
