"""Both sides of the size lines between two forms of one step: the CGS2 panel on a
cluster or on the grid (n = 3328, and the cluster's size below), the FP64 LU panel
on one CTA or a cluster (3096 rows), and the right operand of the digit-sliced
product sliced in one launch or two (2048 rows)."""
import numpy as np
import pytest

from paper_1404_1768_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [41, 64, 65, 256, 257, 3327, 3328, 3329])
def test_cgs2_panel(n):
    """U2 R2 = B U1 of a tridiagonal B (norm below 3): errors of n roundings."""
    import paper_1404_1768_gb300 as fg
    rng = np.random.default_rng(n)
    m0 = 40
    ab = 0.3 * inputs.complex_normal(rng, (3, n))   # rows: super-, main and subdiagonal
    ab[1] += 1.5
    U1 = np.linalg.qr(inputs.complex_normal(rng, (n, m0)))[0]
    g = fg.Feast(ab, ab, U1.copy(), kind=1, kl=1, ku=1, prec=0, q=2, center=10 + 0j, a=1.0)
    g.set_subspace(U1)
    U2, R2 = g.get("U2"), g.get("R2")
    g.close()
    BU = ab[1][:, None] * U1
    BU[:-1] += ab[0][1:, None] * U1[1:]
    BU[1:] += ab[2][:-1, None] * U1[:-1]
    assert np.abs(U2.conj().T @ U2 - np.eye(m0)).max() <= n * 2.0 ** -53
    assert np.abs(U2 @ R2 - BU).max() <= 3 * n * 2.0 ** -53


def test_lu_panel():
    """A factorisation whose first panel is beyond the cluster's rows and whose
    others are not: backward error of n roundings."""
    import paper_1404_1768_gb300 as fg
    n = 3128
    rng = np.random.default_rng(n)
    M = inputs.complex_normal(rng, (n, n)) + 3 * np.sqrt(n) * np.eye(n)
    R = inputs.complex_normal(rng, (n, 3))
    F, piv, info = fg.zgetrf_batched([M])
    assert info == 0
    X = fg.zgetrs_batched(F, piv, [R])[0]
    assert np.linalg.norm(M @ X - R) <= 4 * n * 2.0 ** -53 * np.linalg.norm(M) * np.linalg.norm(X)


@pytest.mark.parametrize("n", [1, 8, 70])
def test_sliced_columns(n):
    """A zero row more takes the operand to the other form; the product stays the same to the bit."""
    import paper_1404_1768_gb300 as fg
    rng = np.random.default_rng(n)
    A, B = inputs.complex_normal(rng, (33, 2048)), inputs.complex_normal(rng, (2048, n))
    one = fg.zgemm_oz(A, B)
    two = fg.zgemm_oz(np.hstack([A, np.zeros((33, 1))]), np.vstack([B, np.zeros((1, n))]))
    assert np.array_equal(one, two)
    ref = A @ B
    bound = 2.0 ** -44 * 2048 * np.abs(A).max(1)[:, None] * np.abs(B).max(0)[None, :]
    assert np.all(np.abs(one - ref) <= bound)


@pytest.mark.parametrize("batch", [8, 9, 32, 33, 64, 65])
@pytest.mark.parametrize("n", [40, 140, 420])
def test_lu_batches(n, batch):
    """8, 4, 2 and 1 CTAs a matrix by the batch's size (more where the panel's rows need them)."""
    import paper_1404_1768_gb300 as fg
    rng = np.random.default_rng(n + batch)
    M = [inputs.complex_normal(rng, (n, n)) + 3 * np.sqrt(n) * np.eye(n) for _ in range(batch)]
    R = [inputs.complex_normal(rng, (n, 2)) for _ in range(batch)]
    F, piv, info = fg.zgetrf_batched(M)
    assert info == 0
    for m, r, x in zip(M, R, fg.zgetrs_batched(F, piv, R)):
        assert np.linalg.norm(m @ x - r) <= 4 * n * 2.0 ** -53 * np.linalg.norm(m) * np.linalg.norm(x)


@pytest.mark.parametrize("q", [32, 33])
@pytest.mark.parametrize("n", [70, 330])
def test_complex64_lu_batches(n, q):
    """The node-batched complex64 LU with 8 CTAs a matrix and with one, through the
    filter of the precision form refined to FP64."""
    import oracle
    import paper_1404_1768_gb300 as fg
    p = inputs.prescribed_pencil(n, n // 4, seed=n)
    Y = inputs.complex_normal(np.random.default_rng(q), (n, 5))
    kw = dict(contour_kind=0, rule=0, q=q, center=0j, a=1.0)
    g = fg.Feast(p.A, p.B, Y, prec=fg.FEAST_C64_REFINE, refine_tol=1e-14, max_refine=6, **kw)
    o = oracle.Feast(p.A, p.B, Y, **kw)
    Ug, Uo = g.filter(Y), o.filter(Y)
    g.close(); o.close()
    assert np.abs(Ug - Uo).max() <= 1e-10 * np.abs(Uo).max()
