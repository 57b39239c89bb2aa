"""The projected eigensolve (feast_zqz_batched): an FP32 Schur form made exact
by a Newton iteration with an FP64 residual, or QZ (up to 64 rows) where that
does not fit.  Sizes at the edges of the 16-row tiles, of the warp, of the
one-CTA forms (64 rows for the whole solve, 232 for the QR), and spectra on both
sides of the iteration's own branches: separated eigenvalues, pairs that
FP32 cannot tell apart, exact multiplicity, a singular B, a Jordan block."""
import numpy as np
import pytest

from paper_1404_1768_gb300 import inputs

pytestmark = pytest.mark.gpu


def _pencil(rng, m, lam):
    W = np.linalg.qr(inputs.complex_normal(rng, (m, m)))[0]
    X = W @ (np.eye(m) + 0.1 * inputs.complex_normal(rng, (m, m)) / np.sqrt(m))
    B = np.eye(m) + 0.1 * np.triu(inputs.complex_normal(rng, (m, m))) / np.sqrt(m)
    return B @ (X * lam) @ np.linalg.inv(X), B


def _check(A, B, lam, tol):
    import paper_1404_1768_gb300 as fg
    al, be, V, fail = fg.zqz_batched([A, A], [B, B])
    assert fail == 0
    m = A.shape[0]
    for b in range(2):
        got = al[b] / be[b]
        d = np.abs(got[:, None] - np.asarray(lam)[None, :])
        assert max(d.min(0).max(), d.min(1).max()) <= tol * np.abs(lam).max()
        r = np.linalg.norm(A @ (V[b] * be[b]) - B @ (V[b] * al[b]), axis=0)
        scale = np.abs(be[b]) * np.linalg.norm(A) + np.abs(al[b]) * np.linalg.norm(B)
        # FP64 backward error: m roundings of entries of the size of the norms
        assert np.max(r / scale) <= 4 * m * 2.0 ** -53
        assert np.max(np.abs(np.linalg.norm(V[b], axis=0) - 1)) <= 4 * m * 2.0 ** -53


@pytest.mark.parametrize("m", [3, 4, 15, 16, 17, 31, 32, 33, 63, 64, 65, 97, 232, 233])
def test_separated(m):
    rng = np.random.default_rng(m)
    lam = 2 * np.sqrt(rng.random(m)) * np.exp(2j * np.pi * rng.random(m))
    A, B = _pencil(rng, m, lam)
    _check(A, B, lam, 32 * m * 2.0 ** -53)   # (eigenvalue condition <= 2, B's <= 2)


@pytest.mark.parametrize("m", [5, 18, 33, 64, 66, 234])
@pytest.mark.parametrize("gap", [1e-4, 1e-6, 1e-8, 1e-10, 0.0])
def test_close_pairs(m, gap):
    rng = np.random.default_rng(100 + m)
    lam = np.arange(1, m + 1).astype(complex)
    lam[1::2] = lam[0:m - 1:2] + gap
    A, B = _pencil(rng, m, lam)
    _check(A, B, lam, 32 * m * 2.0 ** -53)


def test_triple_and_scaled():
    rng = np.random.default_rng(7)
    lam = np.arange(1, 21).astype(complex)
    lam[3:6] = [4.0, 4.0 + 1e-9, 4.0 - 1e-9j]
    A, B = _pencil(rng, 20, lam)
    _check(A, B, lam, 32 * 20 * 2.0 ** -53)
    _check(A * 2.0 ** 90, B * 2.0 ** -60, lam * 2.0 ** 150, 32 * 20 * 2.0 ** -53)


def test_forms_left_to_qz():
    import paper_1404_1768_gb300 as fg
    rng = np.random.default_rng(8)
    m = 12
    J = np.eye(m, dtype=complex) + np.diag(np.ones(m - 1), 1)
    al, be, _, fail = fg.zqz_batched([J], [np.eye(m, dtype=complex)])
    assert fail == 0 and np.max(np.abs(al[0] / be[0] - 1)) < 1e-12
    A, B = inputs.complex_normal(rng, (m, m)), np.triu(np.eye(m) + 0.1 * inputs.complex_normal(rng, (m, m)))
    B[4, 4] = 0.0   # one infinite eigenvalue
    al, be, V, fail = fg.zqz_batched([A], [B])
    assert fail == 0
    assert np.sum(np.abs(be[0]) < 1e-13 * np.abs(al[0])) == 1
    r = np.linalg.norm(A @ (V[0] * be[0]) - B @ (V[0] * al[0]), axis=0)
    assert np.max(r / (np.abs(be[0]) * np.linalg.norm(A) + np.abs(al[0]) * np.linalg.norm(B))) < 4 * m * 2.0 ** -53 * 8
