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
