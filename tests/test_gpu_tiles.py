"""The FP64 and complex64 kernels behind the batched LU and solves, at the
edges of their tiles: panels of 32 columns, GEMM tiles of 16 / 32 / 64, one warp
or one thread per right-hand side (the line is 9728 columns in all), against
numpy.  Random matrices shifted by 3 sqrt(n) I: condition below 10, no growth."""
import numpy as np
import pytest

from paper_1404_1768_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,batch,nrhs", [(1, 1, 1), (31, 3, 2), (32, 2, 9), (33, 2, 8), (64, 1, 1), (65, 2, 17),
                                          (100, 1, 100), (129, 9, 33), (160, 64, 160), (257, 2, 40)])
def test_lu_solve_edges(n, batch, nrhs):
    import paper_1404_1768_gb300 as fg
    rng = np.random.default_rng(n + batch)
    M = [inputs.complex_normal(rng, (n, n)) + 3 * np.sqrt(n) * np.eye(n) for _ in range(batch)]
    R = [inputs.complex_normal(rng, (n, nrhs)) for _ in range(batch)]
    F, piv, info = fg.zgetrf_batched(M)
    assert info == 0
    X = fg.zgetrs_batched(F, piv, R)
    for b in (0, batch - 1):
        L, U = np.tril(F[b], -1) + np.eye(n), np.triu(F[b])
        P = M[b].copy()
        for k in range(n):
            P[[k, piv[b][k]]] = P[[piv[b][k], k]]
        # backward errors of n roundings per entry
        assert np.linalg.norm(L @ U - P) <= 2 * n * 2.0 ** -53 * np.linalg.norm(L) * np.linalg.norm(U)
        res = np.linalg.norm(M[b] @ X[b] - R[b]) / (np.linalg.norm(M[b]) * np.linalg.norm(X[b]))
        assert res <= 4 * n * 2.0 ** -53


@pytest.mark.parametrize("m,n,k", [(1, 1, 1), (63, 64, 16), (64, 65, 255), (65, 63, 257), (31, 33, 31), (130, 70, 1025),
                                   (700, 600, 128), (33, 257, 3000)])
@pytest.mark.parametrize("update", [False, True])
def test_digit_sliced_gemm_edges(m, n, k, update):
    """Tiles of 64 x 64, K-blocks of 16, chunks of 256 and the K splits of 1 to
    8 CTAs a tile: 2^-48 k max|A_i.| max|B_.j| an entry (the entry point's
    bound), the alpha A B + beta C rounding on top."""
    import paper_1404_1768_gb300 as fg
    rng = np.random.default_rng(m + n + k)
    A, B = inputs.complex_normal(rng, (m, k)), inputs.complex_normal(rng, (k, n))
    C0 = inputs.complex_normal(rng, (m, n))
    out = fg.zgemm_oz(A, B, C0, alpha=-1.0, beta=1.0) if update else fg.zgemm_oz(A, B)
    ref = C0 - A @ B if update else A @ B
    ra = np.max(np.maximum(np.abs(A.real), np.abs(A.imag)), axis=1)
    cb = np.max(np.maximum(np.abs(B.real), np.abs(B.imag)), axis=0)
    bound = 2 * (2.0 ** -48 * k * np.outer(ra, cb) + 4 * 2.0 ** -53 * (np.abs(C0) + np.abs(ref)))
    assert np.all(np.abs(out - ref) <= bound)


@pytest.mark.parametrize("m,n,k,batch", [(1, 1, 1, 1), (31, 33, 17, 2), (32, 256, 16, 3), (129, 257, 255, 1),
                                         (200, 8, 300, 2)])
def test_tf32_split_gemm_edges(m, n, k, batch):
    """The operand transposes of the complex64 GEMM at the edges of their 32 x
    32 tiles and 256-row columns: FP32-like error, 2^-20 sqrt(k) of the norms."""
    import paper_1404_1768_gb300 as fg
    rng = np.random.default_rng(m * n + k)
    A = [inputs.complex_normal(rng, (m, k)).astype(np.complex64) for _ in range(batch)]
    X = [inputs.complex_normal(rng, (k, n)).astype(np.complex64) for _ in range(batch)]
    for a, x, c in zip(A, X, fg.cgemm_tc(A, X)):
        ref = a.astype(np.complex128) @ x.astype(np.complex128)
        assert np.linalg.norm(c - ref) <= 2.0 ** -20 * np.sqrt(k) * max(np.linalg.norm(ref), 1e-30)


@pytest.mark.parametrize("m0", [1, 2, 5, 31, 32, 33, 48, 63, 65, 97])
def test_cholesky_blocks(m0):
    """U2 R2 = B U1 at the edges of the 32-column Cholesky blocks and of the
    halves their inverses are built from (FP64 up to 32 columns, the first
    factorisation in FP32 from 33), U1 orthonormal: errors of m0 roundings of
    B's norm, on top of 2^-48 n of the digit-sliced products."""
    import paper_1404_1768_gb300 as fg
    n = 128
    rng = np.random.default_rng(m0)
    B = np.eye(n) + 0.1 * inputs.complex_normal(rng, (n, n)) / np.sqrt(n)
    U1 = np.linalg.qr(inputs.complex_normal(rng, (n, m0)))[0]
    g = fg.Feast(B, B, U1.copy(), prec=fg.FEAST_C64_REFINE, q=8, center=0j, a=1.0)
    g.set_subspace(U1)
    U2, R2 = g.get("U2"), g.get("R2")
    g.close()
    tol = 4 * n * 2.0 ** -48 * np.linalg.norm(B, 2)
    assert np.allclose(np.tril(R2, -1), 0) and np.all(np.diag(R2).real > 0)
    assert np.abs(U2.conj().T @ U2 - np.eye(m0)).max() < tol
    assert np.abs(U2 @ R2 - B @ U1).max() < tol
