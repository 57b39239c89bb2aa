// Projected pencils (A~, B~) of GFEAST line 6 with up to 64 rows, one CTA per
// pencil: an FP32 Schur form made exact by a Newton iteration with an FP64
// residual (k_eig_refined, below), and, for what that leaves, complex QZ in FP64.
//
// B~ = U2^H B U1 is upper triangular by construction (U2 R2 = B U1, so
// B~ = R2 up to rounding), so the usual initial QR of B is skipped and its
// strictly lower part is treated as zero.  QZ: Hessenberg-triangular
// reduction by Givens rotations, single-shift complex QZ sweeps with
// deflation (Moler-Stewart), and right eigenvectors by back-substitution on
// the generalized Schur form (beta S - alpha P) y = 0 mapped back by Z.
//
// The sweep is a chain of dependent 2x2 rotations, each applied to a row or
// column pair; the CTA's four warps share each rotation's updates of H, T
// and Z (one merged index range, so every SM partition's FP64 units work)
// and meet at a barrier between rotations.  The three m x m arrays live in
// shared memory (m <= 64).  Larger projected problems go to k_warm.cu.
#include "chase32.cuh"
#include "common.cuh"

namespace feast {

namespace {

__device__ __forceinline__ zd zsqrt_d(zd z)
{
    double r = hypot(z.x, z.y);
    if (r == 0.0) return zmake(0.0, 0.0);
    if (z.x >= 0.0) {
        double t = sqrt(0.5 * (r + z.x));
        return zmake(t, z.y / (2.0 * t));
    }
    double t = sqrt(0.5 * (r - z.x));
    return zmake(fabs(z.y) / (2.0 * t), copysign(t, z.y));
}

// Left rotation G = [c s; -conj(s) c], G [x; y] = [r; 0].
__device__ __forceinline__ void giv_left(zd x, zd y, double &c, zd &s)
{
    double ax = zabs(x), ay = zabs(y);
    if (ay == 0.0) { c = 1.0; s = zmake(0.0, 0.0); return; }
    if (ax == 0.0) { c = 0.0; s = zmake(1.0, 0.0); return; }
    double r = hypot(ax, ay);
    c = ax / r;
    s = zscale(zmul(zscale(x, 1.0 / ax), zconj(y)), 1.0 / r);
}
// Right rotation R = [c -conj(s); s c] on a column pair, [t0 t1] R = [0 r].
__device__ __forceinline__ void giv_right(zd t0, zd t1, double &c, zd &s)
{
    double a0 = zabs(t0), a1 = zabs(t1);
    if (a0 == 0.0) { c = 1.0; s = zmake(0.0, 0.0); return; }
    if (a1 == 0.0) { c = 0.0; s = zmake(1.0, 0.0); return; }
    double r = hypot(a0, a1);
    c = a1 / r;
    zd t = zscale(zmul(t0, zconj(t1)), -1.0 / (a1 * r));
    s = t;
}

struct Mat {
    zd *p;
    int ld;
    __device__ __forceinline__ zd &operator()(int i, int j) const { return p[i + (int64_t)j * ld]; }
};

template <int NT>
struct Team {
    __device__ __forceinline__ static void bar()
    {
        if (NT == 32) __syncwarp(); else __syncthreads();
    }
};

// rows (i, j) of M over columns [c0, c1]; optionally force M(j, zc) = 0
template <int NT>
__device__ __forceinline__ void rot_rows(Mat M, int i, int j, int c0, int c1, double c, zd s,
                                         int zc)
{
    for (int col = c0 + (int)threadIdx.x; col <= c1; col += NT) {
        zd a = M(i, col), b = M(j, col);
        zd ni = zadd(zscale(a, c), zmul(s, b));
        zd nj = zadd(zscale(zmul(zconj(s), a), -1.0), zscale(b, c));
        M(i, col) = ni;
        M(j, col) = (col == zc) ? zmake(0.0, 0.0) : nj;
    }
}
// columns (i, j) of M over rows [r0, r1]; optionally force M(zr, i) = 0
template <int NT>
__device__ __forceinline__ void rot_cols(Mat M, int i, int j, int r0, int r1, double c, zd s,
                                         int zr)
{
    for (int row = r0 + (int)threadIdx.x; row <= r1; row += NT) {
        zd a = M(row, i), b = M(row, j);
        zd ni = zadd(zscale(a, c), zmul(b, s));
        zd nj = zadd(zscale(zmul(a, zconj(s)), -1.0), zscale(b, c));
        M(row, i) = (row == zr) ? zmake(0.0, 0.0) : ni;
        M(row, j) = nj;
    }
}

// Left rotation on rows (i, j) of two matrices at once: M1 over columns
// [a0, a1] (optionally zeroing M1(j, z1)), M2 over [b0, b1]; the threads
// share the concatenated index range so all warps stay busy.
template <int NT>
__device__ __forceinline__ void rot_rows2(Mat M1, int a0, int a1, int z1, Mat M2, int b0, int b1,
                                          int i, int j, double c, zd s)
{
    const int na = a1 - a0 + 1, nb = b1 - b0 + 1;
    for (int t = (int)threadIdx.x; t < na + nb; t += NT) {
        Mat M = (t < na) ? M1 : M2;
        const int col = (t < na) ? a0 + t : b0 + (t - na);
        zd a = M(i, col), b = M(j, col);
        zd ni = zadd(zscale(a, c), zmul(s, b));
        zd nj = zadd(zscale(zmul(zconj(s), a), -1.0), zscale(b, c));
        M(i, col) = ni;
        M(j, col) = (t < na && col == z1) ? zmake(0.0, 0.0) : nj;
    }
}
// Right rotation on columns (i, j) of three matrices at once: M1 rows
// [0, r1], M2 rows [0, r2] (optionally zeroing M2(z2, i)), M3 rows [0, r3].
template <int NT>
__device__ __forceinline__ void rot_cols3(Mat M1, int r1, Mat M2, int r2, int z2, Mat M3, int r3,
                                          int i, int j, double c, zd s)
{
    const int n1 = r1 + 1, n2 = r2 + 1, n3 = r3 + 1;
    for (int t = (int)threadIdx.x; t < n1 + n2 + n3; t += NT) {
        Mat M;
        int row;
        bool zero_ok = false;
        if (t < n1) { M = M1; row = t; }
        else if (t < n1 + n2) { M = M2; row = t - n1; zero_ok = true; }
        else { M = M3; row = t - n1 - n2; }
        zd a = M(row, i), b = M(row, j);
        zd ni = zadd(zscale(a, c), zmul(b, s));
        zd nj = zadd(zscale(zmul(a, zconj(s)), -1.0), zscale(b, c));
        M(row, i) = (zero_ok && row == z2) ? zmake(0.0, 0.0) : ni;
        M(row, j) = nj;
    }
}

template <int NT>
__device__ double block_max(double v, double *red)
{
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) v = fmax(v, __shfl_xor_sync(0xffffffffu, v, off));
    if (NT == 32) return v;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    if (lane == 0) red[wid] = v;
    __syncthreads();
    double r = red[0];
    for (int w = 1; w < NT / 32; ++w) r = fmax(r, red[w]);
    __syncthreads();
    return r;
}

template <int NT>
__global__ void __launch_bounds__(NT) k_qz(int m, zd *A, int64_t lda, int64_t sA, zd *B,
                                           int64_t ldb, int64_t sB, zd *alpha, zd *beta, zd *V,
                                           int64_t ldv, int64_t sV, zd *work, int use_smem,
                                           int *fail, int only_redo)
{
    extern __shared__ zd smem[];
    __shared__ double red[32];
    const int b = blockIdx.x;
    A += (int64_t)b * sA;
    B += (int64_t)b * sB;
    V += (int64_t)b * sV;
    alpha += (int64_t)b * m;
    beta += (int64_t)b * m;
    zd *Wk = work + (int64_t)b * m * m;
    const int tid = threadIdx.x;
    zd sigma = zmake(0.0, 0.0);
    if (only_redo) {
        if (*(volatile int *)Wk == 0) return;        // k_eig_refined has solved this pencil
        sigma = zmake(((volatile double *)Wk)[2], ((volatile double *)Wk)[3]);
        Team<NT>::bar();
    }
    const double eps = 2.220446049250313e-16;

    Mat H, T, Z, Yh;
    if (use_smem) {
        H = Mat{smem, m};
        T = Mat{smem + m * m, m};
        Z = Mat{smem + 2 * m * m, m};
    } else {
        H = Mat{A, (int)lda};
        T = Mat{B, (int)ldb};
        Z = Mat{Wk, m};
    }
    Yh = Mat{use_smem ? Wk : V, use_smem ? m : (int)ldv};
    // load / initialise
    for (int e = tid; e < m * m; e += NT) {
        int r = e % m, c = e / m;
        if (use_smem) {
            H(r, c) = A[r + c * lda];
            T(r, c) = (r <= c) ? B[r + c * ldb] : zmake(0.0, 0.0);
        } else if (r > c) {
            T(r, c) = zmake(0.0, 0.0);
        }
        Z(r, c) = zmake(r == c ? 1.0 : 0.0, 0.0);
    }
    Team<NT>::bar();
    double c;
    zd s;
    // Hessenberg-triangular reduction
    for (int j = 0; j + 2 < m; ++j)
        for (int i = m - 1; i >= j + 2; --i) {
            giv_left(H(i - 1, j), H(i, j), c, s);
            Team<NT>::bar();
            rot_rows2<NT>(H, j, m - 1, j, T, i - 1, m - 1, i - 1, i, c, s);
            Team<NT>::bar();
            giv_right(T(i, i - 1), T(i, i), c, s);
            Team<NT>::bar();
            rot_cols3<NT>(H, m - 1, T, i, i, Z, m - 1, i - 1, i, c, s);
            Team<NT>::bar();
        }
    // norms for the deflation tests
    double hn = 0.0, tn = 0.0;
    for (int e = tid; e < m * m; e += NT) {
        hn = fmax(hn, zabs(H(e % m, e / m)));
        tn = fmax(tn, zabs(T(e % m, e / m)));
    }
    hn = block_max<NT>(hn, red);
    tn = block_max<NT>(tn, red);
    const double htol = eps * fmax(hn, 1e-300);
    // QZ sweeps
    int ihi = m - 1, iter = 0, total = 0, failed = 0;
    while (ihi > 0) {
        int l = ihi;
        bool found = false;
        while (l > 0) {
            double sub = zabs(H(l, l - 1));
            double loc = zabs(H(l - 1, l - 1)) + zabs(H(l, l));
            if (sub <= eps * loc || sub <= htol) { found = true; break; }
            --l;
        }
        Team<NT>::bar();
        if (found) {
            if (tid == 0) H(l, l - 1) = zmake(0.0, 0.0);
            Team<NT>::bar();
        }
        if (l == ihi) { --ihi; iter = 0; continue; }
        if (++total > 60 * m) { failed = 1; break; }
        ++iter;
        zd sigma;
        zd h00 = H(ihi - 1, ihi - 1), h01 = H(ihi - 1, ihi), h10 = H(ihi, ihi - 1), h11 = H(ihi, ihi);
        zd t00 = T(ihi - 1, ihi - 1), t01 = T(ihi - 1, ihi), t11 = T(ihi, ihi);
        if (iter % 11 == 10) {
            zd den = (t11.x != 0.0 || t11.y != 0.0) ? t11 : zmake(1.0, 0.0);
            double a = zabs(h10);
            sigma = zadd(zdiv(h11, den), zmake(a, 0.5 * a));
        } else if (zabs(t00) > eps * tn && zabs(t11) > eps * tn) {
            zd qa = zmul(t00, t11);
            zd qb = zscale(zsub(zadd(zmul(h00, t11), zmul(h11, t00)), zmul(t01, h10)), -1.0);
            zd qc = zsub(zmul(h00, h11), zmul(h01, h10));
            zd disc = zsqrt_d(zsub(zmul(qb, qb), zscale(zmul(qa, qc), 4.0)));
            zd twoa = zscale(qa, 2.0);
            zd r1 = zdiv(zadd(zscale(qb, -1.0), disc), twoa);
            zd r2 = zdiv(zsub(zscale(qb, -1.0), disc), twoa);
            zd ref = zdiv(h11, t11);
            sigma = (zabs(zsub(r1, ref)) < zabs(zsub(r2, ref))) ? r1 : r2;
        } else {
            sigma = zmake(0.0, 0.0);
        }
        for (int k = l; k < ihi; ++k) {
            zd x, y;
            if (k == l) { x = zsub(H(l, l), zmul(sigma, T(l, l))); y = H(l + 1, l); }
            else        { x = H(k, k - 1); y = H(k + 1, k - 1); }
            giv_left(x, y, c, s);
            Team<NT>::bar();
            rot_rows2<NT>(H, (k > l) ? k - 1 : l, m - 1, (k > l) ? k - 1 : -1, T, k, m - 1, k, k + 1, c, s);
            Team<NT>::bar();
            giv_right(T(k + 1, k), T(k + 1, k + 1), c, s);
            Team<NT>::bar();
            int rl = (k + 2 < ihi) ? k + 2 : ihi;
            rot_cols3<NT>(H, rl, T, k + 1, k + 1, Z, m - 1, k, k + 1, c, s);
            Team<NT>::bar();
        }
    }
    if (failed && tid == 0 && fail) atomicAdd(fail, 1);
    // eigenvalues
    for (int k = tid; k < m; k += NT) {
        alpha[k] = only_redo ? zadd(H(k, k), zmul(sigma, T(k, k))) : H(k, k);   // (A was shifted by sigma B)
        beta[k] = T(k, k);
    }
    // y_hat_k by back-substitution, one thread per eigenvector
    for (int k = tid; k < m; k += NT) {
        const zd al = H(k, k), be = T(k, k);
        const double g = eps * (hn * zabs(be) + tn * zabs(al));   // rounding level of be S - al P, whatever their scales
        for (int i = k + 1; i < m; ++i) Yh(i, k) = zmake(0.0, 0.0);
        Yh(k, k) = zmake(1.0, 0.0);
        for (int i = k - 1; i >= 0; --i) {
            zd sum = zmake(0.0, 0.0);
            for (int p = i + 1; p <= k; ++p)
                zfma(sum, zsub(zmul(be, H(i, p)), zmul(al, T(i, p))), Yh(p, k));
            zd d = zsub(zmul(be, H(i, i)), zmul(al, T(i, i)));
            if (zabs(d) < g) d = zmake(g, 0.0);
            if (d.x == 0.0 && d.y == 0.0) d = zmake(1e-300, 0.0);
            zd q = zdiv(sum, d);
            Yh(i, k) = zmake(-q.x, -q.y);
        }
    }
    Team<NT>::bar();
    // V = Z * Y_hat with unit columns.  The product column k needs Y_hat(:, k)
    // only, and is written to a buffer that holds neither Z nor Y_hat: V
    // itself in the shared-memory layout (Y_hat is in work), H's storage in
    // the global layout (Y_hat is in V; H is no longer needed).
    Mat P = use_smem ? Mat{V, (int)ldv} : H;
    for (int k = tid; k < m; k += NT) {
        double nrm = 0.0;
        for (int r = 0; r < m; ++r) {
            zd acc = zmake(0.0, 0.0);
            for (int p = 0; p <= k; ++p) zfma(acc, Z(r, p), Yh(p, k));
            P(r, k) = acc;
            nrm += zabs2(acc);
        }
        nrm = sqrt(nrm);
        const double inv = nrm > 0.0 ? 1.0 / nrm : 1.0;
        for (int r = 0; r < m; ++r) P(r, k) = zscale(P(r, k), inv);
    }
    Team<NT>::bar();
    if (use_smem) {
        for (int e = tid; e < m * m; e += NT) {
            int r = e % m, cc = e / m;
            A[r + cc * lda] = H(r, cc);
            B[r + cc * ldb] = T(r, cc);
        }
    } else {
        for (int e = tid; e < m * m; e += NT) {
            int r = e % m, cc = e / m;
            V[r + cc * ldv] = H(r, cc);
        }
    }
}

// ---------------------------------------------------------------- refined
// Eigenpairs of (A, B), B upper triangular, from an FP32 Schur form made
// exact by an FP64 Newton iteration on the pencil itself; one CTA per pencil.
//
// GB300 issues one warp-wide FP64 instruction per 64 clocks on each SM
// quarter, whatever the number of active lanes, and a QZ rotation is a chain
// of ~80 of them (three hypot, two divisions): k_qz spent ~10 us per rotation
// pair, 70 ms at m = 64.  In FP32 the same chain is ~0.2 us, and what FP32
// leaves is small enough for Newton's iteration to remove: with approximate
// eigenvectors V and L^H = (B V)^{-1},
//     R = A V - B V Lambda  (FP64),  W = L^H R,  lambda_j += W_jj,
//     G_ij = W_ij / (lambda_j - lambda_i),  V += V G,
// where only R carries FP64 products (8 m^3 DFMA on the tile grid); L, W, G
// and V G multiply something small, so FP32 is enough for them and sets the
// rate of convergence, not the limit.  The error left by a step is about
// |G| (m |G| + delta), delta = ||I - L^H B V||_F measured at the start and
// bounded from then on; the iteration ends when that, or the contraction
// seen from step to step, leaves less than EZ_DONE.  B is only inverted in
// FP32, so the limit is the residual's FP64 rounding, as for QZ.
// Two eigenvalues closer than FP32 resolves (|W_ij| > EZ_PAIR |lambda_j - lambda_i|)
// are separated by the eigenvectors of their own 2 x 2 block of Lambda + W,
// which the FP64 residual determines, before the iteration goes on.
// Pencils it does not fit (B singular or cond(B) beyond FP32's reach, three
// or more eigenvalues that close, non-finite entries) raise *redo; the caller
// then takes the QZ (k_qz) or the double-single QR.  Measured on GB300, see
// zqz_batched.
constexpr int EZ_T = 256;            // threads per CTA
constexpr int EZ_Q = 192;            // of them in the QR iteration
constexpr int EZ_MIN_M = 3;          // smallest pencil
constexpr int EZ_STEPS = 10;         // most Newton steps
constexpr float EZ_PAIR = 1.f / 16;  // largest G_ij of a Newton step
constexpr float EZ_NARROW = 1.f / 16;   // |A - sigma B| / |A| from which A is shifted
constexpr double EZ_DONE = 4e-15;    // error bound at which the iteration ends
constexpr float EZ_BERR = 0x1p-52f;  // residual column at rounding level: <= EZ_BERR m (1 + |lambda'|)

__device__ __forceinline__ void ez_bar() { asm volatile("bar.sync 1, %0;" ::"n"(EZ_Q) : "memory"); }

// Sum over the CTA of one float per thread, in a fixed order.
__device__ __forceinline__ float ez_sum(float v, float *red)
{
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
    __syncthreads();
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
    __syncthreads();
    float r = 0.f;
    for (int w = 0; w < EZ_T / 32; ++w) r += red[w];
    return r;
}
__device__ __forceinline__ float ez_max(float v, float *red)
{
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, off));
    __syncthreads();
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
    __syncthreads();
    float r = red[0];
    for (int w = 1; w < EZ_T / 32; ++w) r = fmaxf(r, red[w]);
    return r;
}

// C <- op(X) op(Y) (m x m in shared memory, row-major, ld), 4 x 4 entries per
// thread with interleaved rows and columns; HY: Y^H.  C is neither X nor Y.
template <bool HY>
__device__ void ez_mul(int m, int ld, const cf *X, const cf *Y, cf *C)
{
    const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
    cf acc[4][4];
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j] = cmakef(0.f, 0.f);
    for (int p = 0; p < m; ++p) {
        cf x[4], y[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) x[i] = (ty + 16 * i < m) ? X[(ty + 16 * i) * ld + p] : cmakef(0.f, 0.f);
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const int c = tx + 16 * j;
            y[j] = (c < m) ? (HY ? cconj(Y[c * ld + p]) : Y[p * ld + c]) : cmakef(0.f, 0.f);
        }
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int j = 0; j < 4; ++j) cfma(acc[i][j], x[i], y[j]);
    }
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j)
            if (ty + 16 * i < m && tx + 16 * j < m) C[(ty + 16 * i) * ld + tx + 16 * j] = acc[i][j];
    __syncthreads();
}

// Rows of X (and X2, when given) <- U^{-1} X by back-substitution, U upper
// triangular (UNIT: unit diagonal); row-major, ld.
template <bool UNIT>
__device__ void ez_back_solve(int m, int ld, const cf *U, cf *X, cf *X2)
{
    // thread: column t mod 128 of [X | X2] (m <= 64 each), every other row
    const int c = threadIdx.x & 127, half = threadIdx.x >> 7;
    cf *x = c < 64 ? X + c : X2 + (c - 64);
    const bool on = c < 64 ? c < m : (X2 != nullptr && c - 64 < m);
    for (int i = m - 1; i >= 0; --i) {
        cf xi = on ? x[i * ld] : cmakef(0.f, 0.f);
        if (!UNIT) {
            xi = cdiv(xi, U[i * ld + i]);
            __syncthreads();
            if (on && half == 0) x[i * ld] = xi;
        }
        const cf nx = cneg(xi);
        if (on)
            for (int r = half; r < i; r += 2) {
                cf v = x[r * ld];
                cfma(v, nx, U[r * ld + i]);
                x[r * ld] = v;
            }
        __syncthreads();
    }
}

// Hessenberg form of H by Householder reflectors, Z <- product (both m x m
// row-major, ld); hv: m entries.
__device__ void ez_hess(int m, int ld, cf *H, cf *Z, cf *hv)
{
    const int t = threadIdx.x, lane = t & 31;
    for (int e = t; e < m * m; e += EZ_T) Z[(e / m) * ld + e % m] = cmakef(e / m == e % m ? 1.f : 0.f, 0.f);
    __syncthreads();
    for (int j = 0; j + 2 < m; ++j) {
        const int len = m - j - 1;
        // every warp forms the same reflector
        float s = 0.f;
        for (int i = lane; i < len; i += 32) s += cabs2(H[(j + 1 + i) * ld + j]);
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) s += __shfl_xor_sync(0xffffffffu, s, off);
        const cf x0 = H[(j + 1) * ld + j];
        const float nrm = sqrtf(s), a0 = abs32(x0);
        const cf ph = a0 > 0.f ? cmakef(x0.x / a0, x0.y / a0) : cmakef(1.f, 0.f);
        const float vv = 2.f * nrm * (nrm + a0), tau = vv > 0.f ? 2.f / vv : 0.f;
        for (int i = t; i < len; i += EZ_T)
            hv[i] = (i == 0) ? cmakef(x0.x + ph.x * nrm, x0.y + ph.y * nrm) : H[(j + 1 + i) * ld + j];
        __syncthreads();
        // left: four threads per column j+1 .. m-1
        {
            const int c = j + 1 + (t >> 2), part = t & 3;
            cf acc = cmakef(0.f, 0.f);
            if (c < m)
                for (int i = part; i < len; i += 4) cfma(acc, cconj(hv[i]), H[(j + 1 + i) * ld + c]);
            acc.x += __shfl_xor_sync(0xffffffffu, acc.x, 1);
            acc.y += __shfl_xor_sync(0xffffffffu, acc.y, 1);
            acc.x += __shfl_xor_sync(0xffffffffu, acc.x, 2);
            acc.y += __shfl_xor_sync(0xffffffffu, acc.y, 2);
            const cf f = cmakef(-tau * acc.x, -tau * acc.y);
            if (c < m)
                for (int i = part; i < len; i += 4) cfma(H[(j + 1 + i) * ld + c], hv[i], f);
        }
        if (t < len) H[(j + 1 + t) * ld + j] = (t == 0) ? cmakef(-ph.x * nrm, -ph.y * nrm) : cmakef(0.f, 0.f);
        __syncthreads();
        // right: two threads per row of H and of Z
        {
            const int r = t >> 1, part = t & 1;
            cf *row = (r < m) ? H + r * ld : Z + (r - m) * ld;
            const bool on = r < 2 * m;
            cf acc = cmakef(0.f, 0.f);
            if (on)
                for (int i = part; i < len; i += 2) cfma(acc, row[j + 1 + i], hv[i]);
            acc.x += __shfl_xor_sync(0xffffffffu, acc.x, 1);
            acc.y += __shfl_xor_sync(0xffffffffu, acc.y, 1);
            const cf f = cmakef(-tau * acc.x, -tau * acc.y);
            if (on)
                for (int i = part; i < len; i += 2) cfma(row[j + 1 + i], f, cconj(hv[i]));
        }
        __syncthreads();
    }
}

// Single-shift QR of the Hessenberg H to triangular form, Z <- Z Q (row-major,
// ld), by the first EZ_Q threads: warp 0 scans for deflation and runs the
// sweep's chain of rotations (chase32.cuh), 32 at a time; then warp 1 applies
// them to the columns of H beyond the chunk, threads 64 .. 127 to the rows of
// H and threads 128 .. 191 to those of Z.  rot: CHASE_N rotations; ctl: two
// ints, sg: the shift.  false: budget spent.
__device__ bool ez_qr(int m, int ld, cf *H, cf *Z, float tol_abs, RotF *rot, int *ctl, cf *sg)
{
    const int t = threadIdx.x, lane = t & 31;
    const float tol_rel = 2.4e-7f;
    int hi = m - 1, it = 0, tot = 0;
    for (;;) {
        if (t < 32) {
            int lo = 0;
            while (hi > 0) {
                lo = 0;
                for (int base = hi; base >= 1 && lo == 0; base -= 32) {
                    const int p = base - lane;
                    bool neg = false;
                    if (p >= 1) {
                        const float sub = abs32(H[p * ld + p - 1]);
                        const float loc = abs32(H[(p - 1) * ld + p - 1]) + abs32(H[p * ld + p]);
                        neg = !(sub > tol_rel * loc) || !(sub > tol_abs);
                    }
                    const unsigned b = __ballot_sync(0xffffffffu, neg);
                    if (b) lo = base - (__ffs(b) - 1);
                }
                if (lo < hi) break;
                --hi;
                it = 0;
            }
            if (hi > 0 && ++tot > 40 * m) hi = -1;
            if (hi > 0) {
                ++it;
                const cf h00 = H[(hi - 1) * ld + hi - 1], h01 = H[(hi - 1) * ld + hi];
                const cf h10 = H[hi * ld + hi - 1], h11 = H[hi * ld + hi];
                cf sigma = shift32(h00, h01, h10, h11);
                if (it % 11 == 10) {
                    const float a = abs32(h10);
                    sigma = cmakef(h11.x + a, h11.y + 0.5f * a);
                }
                if (lane == 0) *sg = sigma;
            }
            if (lane == 0) {
                ctl[0] = lo;
                ctl[1] = hi;
            }
        }
        ez_bar();
        const int lo = ctl[0], h = ctl[1];
        if (h <= 0) return h == 0;
        const RowsLd R{H, ld};
        for (int k0 = lo; k0 < h; k0 += CHASE_N) {
            const int k1 = (k0 + CHASE_N < h) ? k0 + CHASE_N : h;
            if (t < 32) chase_left(R, m, lo, h, k0, k1, *sg, rot);
            ez_bar();
            if (t < 64) {
                const int c = k0 + 1 + t;               // (warp 1: columns k0 + 33 ..)
                if (t >= 32 && c < m) far_left(R, c, k0, k1, rot);
            } else if (t < 128) {
                const int r = t - 64;
                if (r < k1) chase_right(H + r * ld, k0, r > k0 ? r : k0, k1, rot);
            } else if (t - 128 < m) {
                chase_right(Z + (t - 128) * ld, k0, k0, k1, rot);
            }
            ez_bar();
        }
    }
}

// Eigenvector columns of the upper triangle of T into Y (upper triangular,
// unit diagonal), one warp per eigenvector; row-major, ld.  An entry whose
// eigenvalue is within small of the column's is left at zero: FP32 cannot
// tell the two apart, the quotient would make the columns parallel, and the
// pair's own block settles it in the iteration.
__device__ void ez_vectors(int m, int ld, const cf *T, cf *Y, float small)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (int e = threadIdx.x; e < m * m; e += EZ_T) Y[(e / m) * ld + e % m] = cmakef(0.f, 0.f);
    __syncthreads();
    for (int k = warp; k < m; k += EZ_T / 32) {
        const cf lam = T[k * ld + k];
        // lane l holds entries l and l + 32 of the vector
        cf y0 = cmakef(lane == k ? 1.f : 0.f, 0.f), y1 = cmakef(lane + 32 == k ? 1.f : 0.f, 0.f);
        for (int i = k - 1; i >= 0; --i) {
            cf acc = cmakef(0.f, 0.f);
            if (lane > i && lane <= k) cfma(acc, T[i * ld + lane], y0);
            if (lane + 32 > i && lane + 32 <= k) cfma(acc, T[i * ld + lane + 32], y1);
#pragma unroll
            for (int off = 16; off > 0; off >>= 1) {
                acc.x += __shfl_xor_sync(0xffffffffu, acc.x, off);
                acc.y += __shfl_xor_sync(0xffffffffu, acc.y, off);
            }
            cf d = T[i * ld + i];
            d = cmakef(lam.x - d.x, lam.y - d.y);
            const cf q = cabs2(d) < small * small ? cmakef(0.f, 0.f) : cdiv(acc, d);
            if (lane == i) y0 = q;
            if (lane + 32 == i) y1 = q;
        }
        if (lane <= k) Y[lane * ld + k] = y0;
        if (lane + 32 <= k) Y[(lane + 32) * ld + k] = y1;
    }
    __syncthreads();
}

// a += x v: a and x unevaluated sums of two floats (~2^-46 relative), v a float
// (error-free product by FMA).
struct f2 {
    float h, l;
};
__device__ __forceinline__ void f2_fma(f2 &a, float xh, float xl, float v)
{
    const float p = __fmul_rn(xh, v);
    const float e = __fmaf_rn(xl, v, __fmaf_rn(xh, v, -p));
    const float s = __fadd_rn(a.h, p);
    const float b = __fsub_rn(s, a.h);
    const float t = __fadd_rn(__fadd_rn(__fsub_rn(a.h, __fsub_rn(s, b)), __fsub_rn(p, b)), __fadd_rn(a.l, e));
    a.h = __fadd_rn(s, t);
    a.l = __fsub_rn(t, __fsub_rn(a.h, s));
}
__device__ __forceinline__ float f2_sub_mul(f2 a, f2 br, float lr, f2 bi, float li)   // a - br lr - bi li
{
    f2_fma(a, br.h, br.l, -lr);
    f2_fma(a, bi.h, bi.l, -li);
    return a.h + a.l;
}

// R' = A' V - B' V Lambda' of the first step, where V (= V32) and Lambda (=
// diag, FP32) are FP32 exactly: the products in double-single on the FP32 pipe,
// a sixth of the FP64 form's time.  As: m x m float4 of scratch, Bh: m ld
// scratch; W: scratch, then R'.
__device__ void ez_resid_first(int m, int ld, const zd *A, int64_t lda, double fa, const zd *B, int64_t ldb, double fb,
                               const cf *V32, const float *lf, float4 *As, cf *Bh, cf *W)
{
    const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
    for (int e = threadIdx.x; e < m * m; e += EZ_T) {
        const int r = e % m, c = e / m;
        const double x = A[r + c * lda].x * fa, y = A[r + c * lda].y * fa;
        const float xh = (float)x, yh = (float)y;
        As[e] = make_float4(xh, (float)(x - (double)xh), yh, (float)(y - (double)yh));
        cf h = cmakef(0.f, 0.f), l = h;
        if (r <= c) {
            const double u = B[r + c * ldb].x * fb, v = B[r + c * ldb].y * fb;
            h = cmakef((float)u, (float)v);
            l = cmakef((float)(u - (double)h.x), (float)(v - (double)h.y));
        }
        Bh[r * ld + c] = h;
        W[r * ld + c] = l;
    }
    __syncthreads();
    cf out[4][4];
#pragma unroll
    for (int i2 = 0; i2 < 4; i2 += 2) {
        f2 ar[2][4], ai[2][4], br[2][4], bi[2][4];
#pragma unroll
        for (int i = 0; i < 2; ++i)
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                ar[i][j].h = ar[i][j].l = ai[i][j].h = ai[i][j].l = 0.f;
                br[i][j].h = br[i][j].l = bi[i][j].h = bi[i][j].l = 0.f;
                out[i2 + i][j] = cmakef(0.f, 0.f);
            }
        if (16 * i2 < m) {
            for (int p = 0; p < m; ++p) {
#pragma unroll
                for (int i = 0; i < 2; ++i) {
                    const int r = ty + 16 * (i2 + i);
                    if (r >= m) continue;
                    const float4 x = As[r + p * m];
                    const cf h = Bh[r * ld + p], l = W[r * ld + p];
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        const int c = tx + 16 * j;
                        if (c >= m) continue;
                        const cf v = V32[p * ld + c];
                        f2_fma(ar[i][j], x.x, x.y, v.x);
                        f2_fma(ar[i][j], x.z, x.w, -v.y);
                        f2_fma(ai[i][j], x.x, x.y, v.y);
                        f2_fma(ai[i][j], x.z, x.w, v.x);
                        if (r <= p) {
                            f2_fma(br[i][j], h.x, l.x, v.x);
                            f2_fma(br[i][j], h.y, l.y, -v.y);
                            f2_fma(bi[i][j], h.x, l.x, v.y);
                            f2_fma(bi[i][j], h.y, l.y, v.x);
                        }
                    }
                }
            }
#pragma unroll
            for (int i = 0; i < 2; ++i)
#pragma unroll
                for (int j = 0; j < 4; ++j) {
                    const int c = tx + 16 * j;
                    if (c >= m) continue;
                    const float lr = lf[4 * c], li = lf[4 * c + 2];
                    out[i2 + i][j] = cmakef(f2_sub_mul(ar[i][j], br[i][j], lr, bi[i][j], -li),
                                            f2_sub_mul(ai[i][j], br[i][j], li, bi[i][j], lr));
                }
        }
    }
    __syncthreads();
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j)
            if (ty + 16 * i < m && tx + 16 * j < m) W[(ty + 16 * i) * ld + tx + 16 * j] = out[i][j];
}

// exponent bits of the largest |component| (0x7ff: a non-finite entry)
__device__ __forceinline__ unsigned ez_hi(zd v)
{
    const unsigned a = (unsigned)__double2hiint(v.x) & 0x7fffffffu, b = (unsigned)__double2hiint(v.y) & 0x7fffffffu;
    return a > b ? a : b;
}
__device__ __forceinline__ double ez_pow2(int e) { return __longlong_as_double((long long)(e + 1023) << 52); }

__host__ __device__ inline int ez_ld(int m) { return m | 1; }   // odd: rows fall on different banks
__host__ inline size_t ez_smem_bytes(int m)
{
    return sizeof(zd) * (size_t)m * m + 4 * sizeof(cf) * (size_t)m * ez_ld(m) + sizeof(cf) * (size_t)m +
           sizeof(zd) * (size_t)m + 4 * sizeof(float) * (size_t)m + 2 * sizeof(zd) * (size_t)m + 2 * sizeof(int) * (size_t)m;
}

__global__ void __launch_bounds__(EZ_T) k_eig_refined(int m, zd *A, int64_t lda, int64_t sA,
                                                      const zd *__restrict__ B, int64_t ldb, int64_t sB,
                                                      zd *__restrict__ alpha, zd *__restrict__ beta,
                                                      zd *__restrict__ V, int64_t ldv, int64_t sV, zd *work)
{
    extern __shared__ zd smem[];
    __shared__ float red[EZ_T / 32];
    __shared__ unsigned s_ea, s_eb;
    __shared__ int s_bad, s_ctl[2];
    __shared__ cf s_sg;
    const int b = blockIdx.x, t = threadIdx.x, ld = ez_ld(m);
    A += (int64_t)b * sA;
    B += (int64_t)b * sB;
    V += (int64_t)b * sV;
    alpha += (int64_t)b * m;
    beta += (int64_t)b * m;
    int *redo = (int *)(work + (int64_t)b * m * m);
    zd *Vd = smem;                                  // V, column-major, ld m
    zd *lam = Vd + (size_t)m * m;
    zd *pu = lam + m;                               // pair (i, j): U = [1 pu_i; pu_j 1], and det U
    zd *pd = pu + m;
    cf *H = (cf *)(pd + m), *Z = H + m * ld, *W = Z + m * ld, *L = W + m * ld, *hv = L + m * ld;
    float *lf = (float *)(hv + m);                  // lambda as double-single pairs: 4 floats each
    int *part = (int *)(lf + 4 * m);                // the index this one is too close to, or -1
    int *near = part + m;                           // the same where the coupling is at rounding level
    const cf zero = cmakef(0.f, 0.f);
    zd *shift = work + (int64_t)b * m * m + 1;      // (beside the flag: m >= 3)
    if (t == 0) { s_ea = 0; s_eb = 0; s_bad = 0; *redo = 1; *shift = zmake(0.0, 0.0); }
    __syncthreads();
    {
        unsigned ha = 0, hb = 0;
        for (int e = t; e < m * m; e += EZ_T) {
            const int r = e % m, c = e / m;
            ha = max(ha, ez_hi(A[r + c * lda]));
            if (r <= c) hb = max(hb, ez_hi(B[r + c * ldb]));
        }
        atomicMax(&s_ea, ha);
        atomicMax(&s_eb, hb);
    }
    __syncthreads();
    // A' = 2^-ea A, B' = 2^-eb B have entries below 1; lambda' = 2^(eb - ea) lambda
    int xa = (int)(s_ea >> 20);
    const int xb = (int)(s_eb >> 20);
    if (xa < 523 || xa > 1523 || xb < 523 || xb > 1523) return;   // zero, non-finite or far out of range: QZ
    double fa = ez_pow2(1022 - xa), fl = ez_pow2(xa - xb);
    const double fb = ez_pow2(1022 - xb);
    for (int e = t; e < m * m; e += EZ_T) {
        const int r = e % m, c = e / m;
        const zd a = A[r + c * lda];
        H[r * ld + c] = cmakef((float)(a.x * fa), (float)(a.y * fa));
        cf v = zero;
        if (r <= c) {
            const zd w = B[r + c * ldb];
            v = cmakef((float)(w.x * fb), (float)(w.y * fb));
        }
        W[r * ld + c] = v;
        if (r == c && !(cabs2(v) > 1e-14f)) s_bad = 1;            // |B_ii| <= 1e-7 max|B|
        L[r * ld + c] = cmakef(r == c ? 1.f : 0.f, 0.f);
    }
    __syncthreads();
    if (s_bad) return;
    // A spectrum that is narrow against its distance from the origin (A nearly
    // sigma B, sigma the projection of A on B): A <- A - sigma B, or FP32 would
    // round away the gaps (refused from a 1e-5 of the distance on at 24 and 64
    // rows; 0.7 and 2.9 ms as against 10 and 68 for k_qz)
    zd sigma = zmake(0.0, 0.0);
    {
        cf ab = zero;
        float aa = 0.f, bb = 0.f;
        for (int e = t; e < m * m; e += EZ_T) {
            const cf a = H[(e % m) * ld + e / m], v = W[(e % m) * ld + e / m];
            cfma(ab, cconj(v), a);
            aa += cabs2(a);
            bb += cabs2(v);
        }
        ab.x = ez_sum(ab.x, red);
        ab.y = ez_sum(ab.y, red);
        aa = ez_sum(aa, red);
        bb = ez_sum(bb, red);
        if (aa * bb - cabs2(ab) <= EZ_NARROW * EZ_NARROW * aa * bb) {
            sigma = zmake((double)(ab.x / bb) * fl, (double)(ab.y / bb) * fl);
            unsigned ha = 0;
            for (int e = t; e < m * m; e += EZ_T) {
                const int r = e % m, c = e / m;
                zd &a = A[r + c * lda];
                if (r <= c) a = zsub(a, zmul(sigma, B[r + c * ldb]));
                ha = max(ha, ez_hi(a));
            }
            if (t == 0) { s_ea = 0; *shift = sigma; }
            __syncthreads();
            atomicMax(&s_ea, ha);
            __syncthreads();
            xa = (int)(s_ea >> 20);
            if (xa < 523 || xa > 1523) return;
            fa = ez_pow2(1022 - xa);
            fl = ez_pow2(xa - xb);
            for (int e = t; e < m * m; e += EZ_T) {
                const int r = e % m, c = e / m;
                const zd a = A[r + c * lda];
                H[r * ld + c] = cmakef((float)(a.x * fa), (float)(a.y * fa));
            }
            __syncthreads();
        }
    }
    // H = C = B'^{-1} A', L = B'^{-1}
    ez_back_solve<false>(m, ld, W, H, L);
    float cn = 0.f;
    for (int e = t; e < m * m; e += EZ_T) {
        const float a = cabs2(H[(e / m) * ld + e % m]);
        cn = fmaxf(cn, a == a ? a : __int_as_float(0x7f800000));   // (fmaxf drops a NaN)
    }
    cn = sqrtf(ez_max(cn, red));
    if (!(cn > 0.f && cn < 1e15f)) return;
    ez_hess(m, ld, H, Z, hv);
    if (t < EZ_Q && !ez_qr(m, ld, H, Z, 6e-8f * cn, (RotF *)Vd, s_ctl, &s_sg) && t == 0) s_bad = 1;
    __syncthreads();
    if (s_bad) return;
    // Y into W; V = Z Y with unit columns; L^H = (B' V)^{-1} = D Y^{-1} Z^H B'^{-1}
    ez_vectors(m, ld, H, W, 1e-5f * cn);
    for (int j = t; j < m; j += EZ_T) lam[j] = zmake((double)H[j * ld + j].x, (double)H[j * ld + j].y);
    __syncthreads();
    for (int e = t; e < m * m; e += EZ_T) H[(e / m) * ld + e % m] = cmakef(e / m == e % m ? 1.f : 0.f, 0.f);
    __syncthreads();
    ez_back_solve<true>(m, ld, W, H, nullptr);      // H = Y^{-1}
    {
        cf *T1 = (cf *)Vd;                          // (V is not there yet)
        ez_mul<true>(m, ld, H, Z, T1);              // needs m ld entries: ld <= 2 m
        ez_mul<false>(m, ld, T1, L, H);             // H = Y^{-1} Z^H B'^{-1}
        ez_mul<false>(m, ld, Z, W, L);              // L = Z Y
    }
    for (int j = t; j < m; j += EZ_T) {
        float s = 0.f;
        for (int r = 0; r < m; ++r) s += cabs2(L[r * ld + j]);
        lf[j] = sqrtf(s);
    }
    __syncthreads();
    for (int e = t; e < m * m; e += EZ_T) {
        const int r = e % m, c = e / m;
        const float d = lf[c], di = 1.f / d;
        cf v = L[r * ld + c];
        v = cmakef(v.x * di, v.y * di);
        L[r * ld + c] = v;                          // V (FP32 so far)
    }
    for (int e = t; e < m * m; e += EZ_T) {
        const int r = e / m, c = e % m;
        cf v = H[r * ld + c];
        H[r * ld + c] = cmakef(v.x * lf[r], v.y * lf[r]);
    }
    // delta = || I - L^H B' V ||_F (B' again into W, B' V into Z, the product into W)
    for (int e = t; e < m * m; e += EZ_T) {
        const int r = e % m, c = e / m;
        cf v = zero;
        if (r <= c) {
            const zd w = B[r + c * ldb];
            v = cmakef((float)(w.x * fb), (float)(w.y * fb));
        }
        W[r * ld + c] = v;
    }
    __syncthreads();
    ez_mul<false>(m, ld, W, L, Z);
    ez_mul<false>(m, ld, H, Z, W);
    float dl = 0.f;
    for (int e = t; e < m * m; e += EZ_T) {
        const int r = e / m, c = e % m;
        cf v = W[r * ld + c];
        if (r == c) v.x -= 1.f;
        dl += cabs2(v);
    }
    dl = sqrtf(ez_sum(dl, red));
    if (!(dl < 0.05f)) return;
    bool done = false, ever = false;
    float gprev = 0.f, wprev = 0.f;
    for (int step = 0; step < EZ_STEPS && !done; ++step) {
        for (int j = t; j < m; j += EZ_T) {
            const zd l = lam[j];
            const float hx = (float)l.x, hy = (float)l.y;
            lf[4 * j] = hx;
            lf[4 * j + 1] = (float)(l.x - (double)hx);
            lf[4 * j + 2] = hy;
            lf[4 * j + 3] = (float)(l.y - (double)hy);
            part[j] = near[j] = -1;
        }
        // R' = 2^-ea (A V - B V Lambda), a 4 x 4 tile per thread, into W (FP32):
        // in double-single for the first step (whose V and Lambda are FP32), in
        // FP64 from then on
        if (step == 0) {
            __syncthreads();
            ez_resid_first(m, ld, A, lda, fa, B, ldb, fb, L, lf, (float4 *)Vd, Z, W);
            __syncthreads();
            for (int e = t; e < m * m; e += EZ_T) {
                const cf v = L[(e % m) * ld + e / m];
                Vd[e] = zmake((double)v.x, (double)v.y);
            }
        } else {
            const int tx = t & 15, ty = t >> 4;
            zd ra[4][4], rb[4][4];
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int j = 0; j < 4; ++j) ra[i][j] = rb[i][j] = zmake(0.0, 0.0);
            const int ilo = ty;   // B's rows ty, ty + 16, ...: nothing left of column ty
            for (int p = 0; p < m; ++p) {
                zd a[4], v[4];
#pragma unroll
                for (int i = 0; i < 4; ++i) a[i] = (ty + 16 * i < m) ? A[ty + 16 * i + p * lda] : zmake(0.0, 0.0);
#pragma unroll
                for (int j = 0; j < 4; ++j) v[j] = (tx + 16 * j < m) ? Vd[p + (tx + 16 * j) * m] : zmake(0.0, 0.0);
#pragma unroll
                for (int i = 0; i < 4; ++i)
                    if (16 * i < m)
#pragma unroll
                        for (int j = 0; j < 4; ++j)
                            if (16 * j < m) zfma(ra[i][j], a[i], v[j]);
                if (p < ilo) continue;
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    // (uniform over a warp's two rows but for the diagonal's neighbour, where B is zero)
                    if (16 * i < m && p >= 16 * i) {
                        const zd w = (ty + 16 * i <= p) ? B[ty + 16 * i + p * ldb] : zmake(0.0, 0.0);
#pragma unroll
                        for (int j = 0; j < 4; ++j)
                            if (16 * j < m) zfma(rb[i][j], w, v[j]);
                    }
                }
            }
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const int c = tx + 16 * j;
                if (c >= m) continue;
                const zd l = zscale(lam[c], fl);
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const int r = ty + 16 * i;
                    if (r >= m) continue;
                    const zd d = zscale(zsub(ra[i][j], zmul(l, rb[i][j])), fa);
                    W[r * ld + c] = cmakef((float)d.x, (float)d.y);
                }
            }
        }
        __syncthreads();
        // where the iteration may be standing still: is R' at rounding level?
        bool rough = true;
        if (gprev > 0.f && gprev <= 1e-7f) {
            const int c = t >> 2;                   // four threads per column
            float s = 0.f;
            if (c < m)
                for (int r = t & 3; r < m; r += 4) s += cabs2(W[r * ld + c]);
            s += __shfl_xor_sync(0xffffffffu, s, 1);
            s += __shfl_xor_sync(0xffffffffu, s, 2);
            const float d = c < m ? EZ_BERR * (float)m * (1.f + hypotf(lf[4 * c], lf[4 * c + 2])) : 0.f;
            rough = __syncthreads_or(!(s <= d * d));
        }
        ez_mul<false>(m, ld, H, W, Z);              // Z = L^H R'
        float gm = 0.f, wm = 0.f;
        bool paired = false;
        for (int e = t; e < m * m; e += EZ_T) {
            const int i = e / m, j = e % m;
            if (i == j) continue;
            const cf w = Z[i * ld + j];
            const cf d = cmakef((lf[4 * j] - lf[4 * i]) + (lf[4 * j + 1] - lf[4 * i + 1]),
                                (lf[4 * j + 2] - lf[4 * i + 2]) + (lf[4 * j + 3] - lf[4 * i + 3]));
            const float w2 = cabs2(w), d2 = cabs2(d);
            wm = fmaxf(wm, w2);
            cf gg = zero;
            if (sqrtf(w2) <= 1e-14f * cn) {
                // coupling at rounding level: converged.  (For a close pair G
                // may still be large, and V G in FP32 would put FP32 errors
                // back into V: only a small one is applied that way, a larger one
                // as the pair's block, in FP64.)
                const bool small = w2 <= 1e-16f * d2 && d2 > 1e-30f;
                W[i * ld + j] = small ? cdiv(w, d) : zero;
                if (!small && w2 <= EZ_PAIR * EZ_PAIR * d2 && d2 > 1e-30f) {
                    atomicMax(near + i, j);
                    atomicMax(near + j, i);
                }
                continue;
            } else if (w2 <= EZ_PAIR * EZ_PAIR * d2 && d2 > 1e-30f) {
                gg = cdiv(w, d);
            } else {
                const int pi = atomicCAS(part + i, -1, j), pj = atomicCAS(part + j, -1, i);
                if ((pi != -1 && pi != j) || (pj != -1 && pj != i)) s_bad = 1;
                paired = true;
            }
            gm = fmaxf(gm, cabs2(gg));
            W[i * ld + j] = gg;
        }
        gm = sqrtf(ez_max(gm, red));                // (a barrier: s_bad, the pairs and G are out)
        wm = sqrtf(ez_max(wm, red));
        paired = __syncthreads_or(paired);
        if (s_bad) return;
        int mate = -1;
        if (t < m) {
            mate = part[t];
            const int k = near[t];
            if (mate < 0 && k >= 0 && near[k] == t && part[k] < 0) mate = k;
        }
        __syncthreads();
        if (t < m) {
            const int i = t, j = mate;
            part[i] = j;
            const cf w = Z[i * ld + i];
            const zd li = zmake(lam[i].x + (double)w.x, lam[i].y + (double)w.y);
            if (j > i) {
                // the block [a b; c d] of Lambda + W: eigenvectors (1, c / g) and (-b / g, 1),
                // g = h + s, h = (a - d) / 2, s = sqrt(h^2 + b c) on the side of h
                const cf wj = Z[j * ld + j], wb = Z[i * ld + j], wc = Z[j * ld + i];
                const zd lj = zmake(lam[j].x + (double)wj.x, lam[j].y + (double)wj.y);
                const zd bb = zmake((double)wb.x, (double)wb.y), cc = zmake((double)wc.x, (double)wc.y);
                const zd h = zscale(zsub(li, lj), 0.5);
                zd r = zsqrt_d(zadd(zmul(h, h), zmul(bb, cc)));
                if (r.x * h.x + r.y * h.y < 0.0) r = zscale(r, -1.0);
                const zd g = zadd(h, r), mid = zscale(zadd(li, lj), 0.5);
                if (g.x == 0.0 && g.y == 0.0) {
                    s_bad = 1;
                } else {
                    pu[i] = zscale(zdiv(bb, g), -1.0);
                    pu[j] = zdiv(cc, g);
                    const zd det = zsub(zmake(1.0, 0.0), zmul(pu[i], pu[j]));
                    if (!(zabs2(det) > 2.5e-3)) s_bad = 1;   // nearly parallel: not for this iteration
                    pd[i] = pd[j] = det;
                }
                lam[i] = zadd(mid, r);
                lam[j] = zsub(mid, r);
                W[i * ld + j] = W[j * ld + i] = zero;
            } else if (j < 0) {
                lam[i] = li;
            }
            W[i * ld + i] = zero;
        }
        __syncthreads();
        if (s_bad) return;
        ez_mul<false>(m, ld, L, W, Z);              // V G
        for (int e = t; e < m * m; e += EZ_T) {
            const int r = e % m, c = e / m;
            const cf g = Z[r * ld + c];
            Vd[e] = zmake(Vd[e].x + (double)g.x, Vd[e].y + (double)g.y);
        }
        __syncthreads();
        if (paired || gm > 1e-6f) {
            // L^H <- (I - G) L^H (to be (B V)^{-1} of the new V up to |G|^2)
            ez_mul<false>(m, ld, W, H, Z);
            for (int e = t; e < m * m; e += EZ_T) {
                const int o = (e / m) * ld + e % m;
                H[o] = cmakef(H[o].x - Z[o].x, H[o].y - Z[o].y);
            }
            __syncthreads();
            dl += (float)m * gm * gm;
        } else {
            dl += (float)m * gm;
        }
        // V[:, (i j)] <- V[:, (i j)] U, rows (i j) of L^H <- U^{-1} L^H
        for (int e = t; e < m * m; e += EZ_T) {
            const int r = e % m, i = e / m, j = part[i];
            if (j <= i) continue;
            zd vi = Vd[r + i * m], vj = Vd[r + j * m];
            Vd[r + i * m] = zadd(vi, zmul(vj, pu[j]));
            Vd[r + j * m] = zadd(vj, zmul(vi, pu[i]));
            const zd di = zdiv(zmake(1.0, 0.0), pd[i]);
            const cf hi = H[i * ld + r], hj = H[j * ld + r];
            const zd xi = zmake((double)hi.x, (double)hi.y), xj = zmake((double)hj.x, (double)hj.y);
            const zd yi = zmul(di, zsub(xi, zmul(pu[i], xj))), yj = zmul(di, zsub(xj, zmul(pu[j], xi)));
            H[i * ld + r] = cmakef((float)yi.x, (float)yi.y);
            H[j * ld + r] = cmakef((float)yj.x, (float)yj.y);
        }
        __syncthreads();
        for (int e = t; e < m * m; e += EZ_T) {
            const int r = e % m, c = e / m;
            const zd v = Vd[e];
            L[r * ld + c] = cmakef((float)v.x, (float)v.y);
        }
        __syncthreads();
        // what this step leaves, by the bound on delta or by the contraction
        // seen (|G| over the step before's, at least delta); a pair's block is
        // followed by another step
        const double seen = 8.0 * fmax((double)gm, (double)gm / (double)gprev), bnd = (double)m * (double)gm + (double)dl;
        // (|G| that no longer falls, nor |W|: a close pair's G can stand still while
        // the others still converge, is the residual's rounding when the
        // residual this step began with shows it; otherwise a slow contraction)
        // (the first step's residual has 46 bits: a later one in FP64 always follows)
        const bool still = !rough && gm <= 1e-8f && gprev > 0.f && gm > 0.1f * gprev && wm > 0.1f * wprev;
        done = !paired && step > 0 && (still || (double)gm * fmin(seen, bnd) <= (ever ? 0.25 : 1.0) * EZ_DONE);
        // (after a pair's block neither size says how the iteration contracts)
        gprev = paired ? 0.f : gm;
        wprev = wm;
        ever = ever || paired;
    }
    if (!done) return;
    // unit columns, the eigenvalues on their own scale
    {
        const int j = t >> 2;                       // four threads per column
        double s = 0.0;
        if (j < m)
            for (int r = t & 3; r < m; r += 4) s += zabs2(Vd[r + j * m]);
        s += __shfl_xor_sync(0xffffffffu, s, 1);
        s += __shfl_xor_sync(0xffffffffu, s, 2);
        const double inv = 1.0 / sqrt(s);
        if (j < m)
            for (int r = t & 3; r < m; r += 4) V[r + j * ldv] = zscale(Vd[r + j * m], inv);
        if (j < m && (t & 3) == 0) {
            alpha[j] = zadd(zscale(lam[j], fl), sigma);
            beta[j] = zmake(1.0, 0.0);
        }
    }
    if (t == 0) *redo = 0;
}
}  // namespace

size_t zqz_work_bytes(int m)
{
    size_t small = (size_t)m * m * sizeof(zd);
    if (m <= 64) return small;
    const size_t big = zeig_large_work_bytes(m), ref = zeig_refined_large_work_bytes(m);
    return ((big > ref ? big : ref) + 255) & ~(size_t)255;
}

int zeig_refined(cudaStream_t s, int m, int batch, zd *A, int64_t lda, int64_t sA, const zd *B, int64_t ldb,
                 int64_t sB, zd *alpha, zd *beta, zd *V, int64_t ldv, int64_t sV, void *work)
{
    if (m < EZ_MIN_M || m > 64 || batch <= 0) return FEAST_EINVAL;
    FEAST_CUDA_TRY(ensure_dyn_smem(k_eig_refined, ez_smem_bytes(m)));
    k_eig_refined<<<batch, EZ_T, ez_smem_bytes(m), s>>>(m, A, lda, sA, B, ldb, sB, alpha, beta, V, ldv, sV, (zd *)work);
    FEAST_LAUNCH_CHECK();
    return FEAST_OK;
}

int zqz_left(cudaStream_t s, int m, int batch, zd *A, int64_t lda, int64_t sA, zd *B, int64_t ldb, int64_t sB, zd *alpha,
             zd *beta, zd *V, int64_t ldv, int64_t sV, void *work, int *fail, int refined)
{
    const size_t sm = 3 * (size_t)m * m * sizeof(zd);
    FEAST_CUDA_TRY(ensure_dyn_smem(k_qz<128>, sm));
    k_qz<128><<<batch, 128, sm, s>>>(m, A, lda, sA, B, ldb, sB, alpha, beta, V, ldv, sV, (zd *)work, 1, fail, refined);
    FEAST_LAUNCH_CHECK();
    return FEAST_OK;
}

int zqz_batched(cudaStream_t s, int m, int batch, zd *A, int64_t lda, int64_t sA, zd *B,
                int64_t ldb, int64_t sB, zd *alpha, zd *beta, zd *V, int64_t ldv, int64_t sV,
                void *work, int *fail, int *timeout, int *stats, double defl)
{
    if (m <= 0 || batch <= 0) return FEAST_OK;
    if (m <= 64) {
        // refined FP32 Schur form first (GB300, one pencil per SM: 0.41 ms at
        // m = 24 and 2.5 ms at m = 64, against 10.5 and 67 ms for k_qz, whose
        // every rotation is a chain of FP64 instructions); k_qz then solves
        // the pencils that it left (its CTAs return at once on the others).
        // Up to two rows there is nothing to iterate: k_qz alone.
        const int refined = m >= EZ_MIN_M;
        int e;
        if (refined && (e = zeig_refined(s, m, batch, A, lda, sA, B, ldb, sB, alpha, beta, V, ldv, sV, work))) return e;
        return zqz_left(s, m, batch, A, lda, sA, B, ldb, sB, alpha, beta, V, ldv, sV, work, fail, refined);
    }
    if (lda != m || ldb != m || ldv != m) return FEAST_EINVAL;
    const size_t wb = zqz_work_bytes(m);
    // refined FP32 Schur form first, the double-single QR for what it leaves
    // (GB300, one pencil of 300 rows: 33 ms against 231 ms for the latter)
    for (int b = 0; b < batch; ++b) {
        RefineResult rr;
        zd *Ab = A + (int64_t)b * sA, *Bb = B + (int64_t)b * sB, *al = alpha + (int64_t)b * m, *be = beta + (int64_t)b * m;
        zd *Vb = V + (int64_t)b * sV, sigma = zmake(0.0, 0.0);
        char *wk = (char *)work + b * wb;
        RefineParams prm{0, EZ_DONE, 0.f, 1};
        int e = zeig_refined_large(s, m, Ab, Bb, al, be, Vb, wk, prm, &rr, timeout, stats);
        if (e) return e;
        if (rr.narrow) {
            sigma = rr.sigma;
            prm.find = 0;
            if ((e = shift_pencil(s, m, Ab, Bb, sigma))) return e;
            if ((e = zeig_refined_large(s, m, Ab, Bb, al, be, Vb, wk, prm, &rr, timeout, stats))) return e;
        }
        if (!rr.accepted && (e = zeig_large(s, m, Ab, Bb, al, be, Vb, wk, fail, timeout, stats, defl))) return e;
        if ((sigma.x != 0.0 || sigma.y != 0.0) && (e = shift_values(s, m, al, be, sigma))) return e;
    }
    return FEAST_OK;
}

}  // namespace feast
