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


def _chain(rng, m, p):
    """Well separated eigenvalues with a few large couplings (eigenvector condition up to ~1e4 at p = 4.5)."""
    lam = (np.arange(1, m + 1) + 0.3j * rng.random(m)) / m
    B = np.eye(m) + 0.1 * np.triu(inputs.complex_normal(rng, (m, m))) / np.sqrt(m)
    W = np.linalg.qr(inputs.complex_normal(rng, (m, m)))[0]
    T = np.diag(lam) + 10 ** (p / 2) * np.triu(inputs.complex_normal(rng, (m, m)), 1) * (rng.random((m, m)) < 1.5 / m) / m
    return B @ W @ T @ W.conj().T, B


@pytest.mark.parametrize("m,p,nb", [(3, 4.5, 400), (6, 3.5, 300), (10, 3.0, 200), (24, 3.5, 100), (66, 3.5, 4), (100, 3.0, 3)])
def test_slow_contraction(m, p, nb):
    """Left vectors that FP32 only has to a few per cent, so that the Newton
    steps gain little each: the backward error is still that of an FP64 QZ (4 m
    roundings; above 64 rows the double-single QR's 2^-44 of C for what is left
    to it, on top of B's condition of 2)."""
    import paper_1404_1768_gb300 as fg
    P = [_chain(np.random.default_rng([1, m, int(10 * p), s]), m, p) for s in range(nb)]
    al, be, V, fail = fg.zqz_batched([a for a, _ in P], [b for _, b in P])
    assert fail == 0
    for (A, B), a, b, v in zip(P, al, be, V):
        B = np.triu(B)
        r = np.linalg.norm(A @ (v * b) - B @ (v * a), axis=0)
        scale = np.abs(b) * np.linalg.norm(A) + np.abs(a) * np.linalg.norm(B)
        assert np.max(r / scale) <= 4 * m * (2.0 ** -53 if m <= 64 else 2.0 ** -47)


@pytest.mark.parametrize("m", [3, 8, 33, 64])
def test_diagonal(m):
    """Nothing couples the pairs, so the first step already finds nothing to
    correct but the eigenvalues: all 53 bits of them must come back (one rounding
    of the sum, one of the scale)."""
    import paper_1404_1768_gb300 as fg
    rng = np.random.default_rng(m)
    lam = 2 * np.sqrt(rng.random(m)) * np.exp(2j * np.pi * rng.random(m))
    for d in (lam, lam.real + 0j):
        al, be, V, fail = fg.zqz_batched([np.diag(d)], [np.eye(m, dtype=complex)])
        assert fail == 0
        got = al[0] / be[0]
        err = np.abs(got[:, None] - d[None, :]).min(1)
        assert np.max(err / np.abs(got)) <= 2 * np.sqrt(2) * 2.0 ** -53
