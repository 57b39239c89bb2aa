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


@pytest.mark.parametrize("m", [3, 24, 64, 100, 300])
@pytest.mark.parametrize("ratio", [3e-2, 1e-3, 1e-4, 1e-5, 1e-6])
@pytest.mark.parametrize("ea", [0, 70])
def test_narrow_spectrum(m, ratio, ea):
    """Eigenvalues in a disk of that radius around 1: the bounds of the general
    pencil, relative to |lambda|."""
    rng = np.random.default_rng(m)
    lam = 1 + ratio * 2 * np.sqrt(rng.random(m)) * np.exp(2j * np.pi * rng.random(m))
    A, B = _pencil(rng, m, lam)
    _check(A * 2.0 ** ea, B, lam * 2.0 ** ea, 32 * m * 2.0 ** -53)


def test_narrow_spectrum_left_to_qz():
    """A shifted pencil that goes on to QZ: three equal eigenvalues, one of them defective."""
    import paper_1404_1768_gb300 as fg
    rng = np.random.default_rng(2)
    m = 12
    T = np.diag(1 + 1e-5 * np.concatenate([[0.5, 0.5, 0.5], np.arange(1, m - 2)])).astype(complex)
    T[0, 1] = 1e-5
    W = np.linalg.qr(inputs.complex_normal(rng, (m, m)))[0]
    B = np.eye(m) + 0.1 * np.triu(inputs.complex_normal(rng, (m, m))) / np.sqrt(m)
    A = B @ W @ T @ W.conj().T
    al, be, V, fail = fg.zqz_batched([A], [B])
    assert fail == 0
    r = np.linalg.norm(A @ (V[0] * be[0]) - B @ (V[0] * al[0]), axis=0)
    assert np.max(r / (np.abs(be[0]) * np.linalg.norm(A) + np.abs(al[0]) * np.linalg.norm(B))) <= 4 * m * 2.0 ** -53
    got = al[0] / be[0]
    # (the defective pair splits by the square root of the backward error over its coupling)
    assert np.abs(np.sort(got.real) - np.sort(np.diag(T).real)).max() <= 1e-5 * np.sqrt(32 * m * 2.0 ** -53 / 1e-5)


def _narrow_pencil(rng, n, nin, ratio, far):
    lin = 1 + ratio * 0.95 * np.sqrt(rng.random(nin)) * np.exp(2j * np.pi * rng.random(nin))
    if far:
        lout = 4 + np.sqrt(rng.random(n - nin)) * np.exp(2j * np.pi * rng.random(n - nin))
    else:
        rad = 1.05 * np.sqrt(1 + (n - nin) / nin * rng.random(n - nin))
        lout = 1 + ratio * rad * np.exp(2j * np.pi * rng.random(n - nin))
    P, Q = (np.eye(n) + 0.1 * inputs.complex_normal(rng, (n, n)) / np.sqrt(n) for _ in range(2))
    return (P * np.concatenate([lin, lout])) @ Q, P @ Q, lin


@pytest.mark.parametrize("ratio", [1e-3, 1e-4, 1e-5])
@pytest.mark.parametrize("prec", [0, 1])
def test_narrow_contour_warm(ratio, prec):
    """A contour that is narrow against its centre, in a spectrum of the same
    density around it: every pass is solved by the FP32 Schur form and its
    iteration, and warm once columns have converged."""
    import paper_1404_1768_gb300 as fg
    rng = np.random.default_rng(11)
    A, B, _ = _narrow_pencil(rng, 600, 80, ratio, False)
    g = fg.Feast(A, B, inputs.complex_normal(rng, (600, 112)), center=1 + 0j, a=ratio, q=16, prec=prec, eps=1e-12, max_iter=7)
    infos = g.run()
    g.close()
    assert all(i["qz_cold_fp32"] >= 0 for i in infos)
    assert infos[-1]["qz_warm"] == 1


@pytest.mark.parametrize("m0", [56, 112])
@pytest.mark.parametrize("ratio", [1e-2, 1e-4])
@pytest.mark.parametrize("prec", [0, 1])
def test_narrow_contour_eigenvalues(m0, ratio, prec):
    """The same with the rest of the spectrum far away: residuals below eps bound
    the eigenvalues' errors by eps (|A| + |lambda| |B|) times the pairs' condition (< 3)."""
    import paper_1404_1768_gb300 as fg
    rng = np.random.default_rng(12)
    A, B, lin = _narrow_pencil(rng, 400, int(m0 / 1.4), ratio, True)
    eps = 1e-11
    g = fg.Feast(A, B, inputs.complex_normal(rng, (400, m0)), center=1 + 0j, a=ratio, q=16, prec=prec, eps=eps, max_iter=12)
    infos = g.run()
    lam = np.asarray(g.eigs(False)["lam"])
    g.close()
    assert infos[-1]["flag"] == 1 and lam.size == lin.size
    d = np.abs(lam[:, None] - lin[None, :])
    assert max(d.min(0).max(), d.min(1).max()) <= 3 * eps * (np.linalg.norm(A, 2) + np.linalg.norm(B, 2))


def _pass_launches(A, B, Y, passes, **kw):
    import paper_1404_1768_gb300 as fg
    g = fg.Feast(A, B, Y, max_iter=passes + 2, **kw)
    out = []
    for _ in range(passes):
        n0 = fg.kernel_launches()
        info = g.iterate()
        out.append((fg.kernel_launches() - n0, info))
        if info["flag"] != 2:
            break
    g.close()
    return out


def test_refused_small_pencil_is_tried_once():
    """A cluster of three that goes to QZ: one launch more than the pass of an easy
    pencil of the same sizes (k_qz), not a second attempt before it."""
    rng = np.random.default_rng(21)
    n, m0 = 64, 16
    P, Q = (np.eye(n) + 0.1 * inputs.complex_normal(rng, (n, n)) / np.sqrt(n) for _ in range(2))
    Y = inputs.complex_normal(rng, (n, m0))
    lam = np.concatenate([0.9 * (np.arange(1, 13) / 13) * np.exp(1j * np.arange(12)), 3 + np.arange(n - 12) / n])
    hard = lam.copy()
    hard[1:3] = hard[0]
    kw = dict(center=0j, a=1.0, q=16, prec=0, eps=1e-13)
    easy_n = _pass_launches((P * lam) @ Q, P @ Q, Y, 1, **kw)[0][0]
    hard_n = _pass_launches((P * hard) @ Q, P @ Q, Y, 1, **kw)[0][0]
    assert hard_n == easy_n + 1


def _clustered(gaps, passes, m0=104):
    """72 eigenvalues inside, the first three those gaps apart, the others far outside."""
    rng = np.random.default_rng(22)
    n, nin = 300, 72
    P, Q = (np.eye(n) + 0.1 * inputs.complex_normal(rng, (n, n)) / np.sqrt(n) for _ in range(2))
    lam = np.concatenate([0.9 * np.sqrt(rng.random(nin)) * np.exp(2j * np.pi * rng.random(nin)), 4 + rng.random(n - nin)])
    lam[1:3] = lam[0] + np.array(gaps)
    return _pass_launches((P * lam) @ Q, P @ Q, inputs.complex_normal(rng, (n, m0)), passes, center=0j, a=1.0, q=16, prec=0,
                          eps=1e-30, converged_only=True)


@pytest.mark.parametrize("gaps", [(2e-7, 3.5e-7j), (1e-5, 2e-5j), (0.1, 0.2j)])
def test_warm_after_convergence(gaps):
    """Passes after the pairs inside have converged stay warm, whatever the extra
    directions of the subspace look like: their columns pass for converged
    before their couplings are below their gaps."""
    out = _clustered(gaps, 5)
    assert [i["qz_warm"] for _, i in out[2:]] == [1] * (len(out) - 2)
