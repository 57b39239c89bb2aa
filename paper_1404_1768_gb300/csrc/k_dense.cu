// Complex dense kernels (FP64 for the plain path, FP32 for the low-precision
// factors of the precision form): batched GEMM, formation
// of the shifted matrices z_j B - A (eq. 4.2), blocked right-looking LU with
// partial pivoting, blocked triangular solves with many right-hand sides,
// and the quadrature node-sum U = sum_j w_j X_j (eq. 4.1).
//
// GB300 runs FP64 at ~2 DFMA per clock per SM (1.05 TFLOP/s measured for
// the whole GPU), so these kernels are bound by the FP64 pipe, not by
// memory: a modest register tile (4 x 4 complex per thread) already keeps
// the pipe busy, and the work is spread over all 152 SMs through the batch
// (node) dimension and the tile grid.
#include "common.cuh"

namespace feast {

// ------------------------------------------------------------------ GEMM
namespace {
constexpr int GB_K = 8, GB_T = 256;

constexpr int GB_SMAX = 8;     // most K-slices of a tile summed in one (portable) cluster

__device__ __forceinline__ void atomic_cadd(double2 *p, double2 v)
{
    atomicAdd(&p->x, v.x);
    atomicAdd(&p->y, v.y);
}
__device__ __forceinline__ void atomic_cadd(float2 *p, float2 v)
{
    atomicAdd(&p->x, v.x);
    atomicAdd(&p->y, v.y);
}

// splits > 1: blockIdx.z = batch * splits + s takes the s-th slice of K.
// Up to GB_SMAX slices the launch groups a tile's slices into one cluster
// (s = the CTA's rank in it) and CTA 0 sums the slices' tiles in rank order
// through distributed shared memory before it writes C, so the result does
// not depend on which slice finishes first; beyond that (long, skinny
// products) the slices add alpha * partial into C atomically, C pre-scaled
// by beta on the host side of the launch.
// A CTA of 16 x 16 threads computes a 16 TM x 16 TM tile, TM x TM entries per
// thread.
template <typename T, int TM>
__global__ void __launch_bounds__(GB_T) k_gemm(int conj_a, int64_t m, int64_t n, int64_t k,
                                               T alpha, const T *__restrict__ A, int64_t lda,
                                               int64_t sA, const T *__restrict__ B,
                                               int64_t ldb, int64_t sB, T beta,
                                               T *__restrict__ C, int64_t ldc, int64_t sC,
                                               int splits, int64_t kchunk, int tri)
{
    constexpr int GB_M = 16 * TM, GB_N = 16 * TM;
    __shared__ T As[GB_K][GB_M + 1];
    __shared__ T Bs[GB_K][GB_N + 1];
    extern __shared__ __align__(16) unsigned char gb_red_raw[];   // splits > 1: this slice's tile
    const int b = blockIdx.z / splits, sp = blockIdx.z % splits;
    const int64_t i0 = (int64_t)blockIdx.x * GB_M, j0 = (int64_t)blockIdx.y * GB_N;
    if (tri == 3 && i0 >= j0 + GB_N) return;  // tile below the diagonal (uniform per CTA)
    int64_t kbeg = (int64_t)sp * kchunk;
    int64_t kend = (kbeg + kchunk < k) ? kbeg + kchunk : k;
    if (tri == 1 && kbeg < i0) kbeg = i0;            // op(A)(i, k) = 0 for k < i
    if (tri == 2 && kend > j0 + GB_N) kend = j0 + GB_N;  // B(k, j) = 0 for k > j
    A += (int64_t)b * sA;
    B += (int64_t)b * sB;
    C += (int64_t)b * sC;
    const int tx = threadIdx.x % 16, ty = threadIdx.x / 16;
    T acc[TM][TM];
#pragma unroll
    for (int a = 0; a < TM; ++a)
#pragma unroll
        for (int c = 0; c < TM; ++c) acc[a][c] = cx<T>(0, 0);

    for (int64_t k0 = kbeg; k0 < kend; k0 += GB_K) {
        // A tile: op(A)(i0 + r, k0 + kk)
        for (int e = threadIdx.x; e < GB_M * GB_K; e += GB_T) {
            int r, kk;
            if (!conj_a) { r = e % GB_M; kk = e / GB_M; }
            else         { kk = e % GB_K; r = e / GB_K; }
            int64_t gi = i0 + r, gk = k0 + kk;
            T v = cx<T>(0, 0);
            if (gi < m && gk < kend) v = conj_a ? cconj(A[gk + gi * lda]) : A[gi + gk * lda];
            As[kk][r] = v;
        }
        for (int e = threadIdx.x; e < GB_N * GB_K; e += GB_T) {
            int kk = e % GB_K, c = e / GB_K;
            int64_t gj = j0 + c, gk = k0 + kk;
            Bs[kk][c] = (gj < n && gk < kend) ? B[gk + gj * ldb] : cx<T>(0, 0);
        }
        __syncthreads();
#pragma unroll
        for (int kk = 0; kk < GB_K; ++kk) {
            T av[TM], bv[TM];
#pragma unroll
            for (int a = 0; a < TM; ++a) av[a] = As[kk][ty + 16 * a];
#pragma unroll
            for (int c = 0; c < TM; ++c) bv[c] = Bs[kk][tx + 16 * c];
#pragma unroll
            for (int a = 0; a < TM; ++a)
#pragma unroll
                for (int c = 0; c < TM; ++c) cfma(acc[a][c], av[a], bv[c]);
        }
        __syncthreads();
    }
    if (splits > GB_SMAX) {
#pragma unroll
        for (int a = 0; a < TM; ++a)
#pragma unroll
            for (int c = 0; c < TM; ++c) {
                int64_t gi = i0 + ty + 16 * a, gj = j0 + tx + 16 * c;
                if (gi < m && gj < n) atomic_cadd(&C[gi + gj * ldc], cmul(alpha, acc[a][c]));
            }
        return;
    }
    if (splits > 1) {
        // every slice's tile into its own shared memory; CTA 0 adds the
        // others' in rank order (distributed shared memory), then all wait
        // until it has read them
        T *red = reinterpret_cast<T *>(gb_red_raw);
        const unsigned rank = cluster_rank_id();
#pragma unroll
        for (int a = 0; a < TM; ++a)
#pragma unroll
            for (int c = 0; c < TM; ++c) red[(a * TM + c) * GB_T + threadIdx.x] = acc[a][c];
        cluster_barrier();
        if (rank == 0)
            for (int r = 1; r < splits; ++r)
#pragma unroll
                for (int a = 0; a < TM; ++a)
#pragma unroll
                    for (int c = 0; c < TM; ++c)
                        acc[a][c] = cadd(acc[a][c], peer_load(red + (a * TM + c) * GB_T + threadIdx.x, r));
        cluster_barrier();
        if (rank != 0) return;
    }
    const bool beta0 = cis_zero(beta);
#pragma unroll
    for (int a = 0; a < TM; ++a)
#pragma unroll
        for (int c = 0; c < TM; ++c) {
            int64_t gi = i0 + ty + 16 * a, gj = j0 + tx + 16 * c;
            if (gi < m && gj < n) {
                T v = cmul(alpha, acc[a][c]);
                if (!beta0) v = cadd(v, cmul(beta, C[gi + gj * ldc]));
                C[gi + gj * ldc] = v;
            }
        }
}
// C <- beta C (beta = 0 writes zeros, so stale NaNs do not survive)
template <typename T>
__global__ void k_scale(int64_t m, int64_t n, T beta, T *C, int64_t ldc, int64_t sC)
{
    T *Cb = C + (int64_t)blockIdx.y * sC;
    const bool zero = cis_zero(beta);
    for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < m * n;
         e += (int64_t)gridDim.x * blockDim.x) {
        int64_t r = e % m, c = e / m;
        T &x = Cb[r + c * ldc];
        x = zero ? cx<T>(0, 0) : cmul(beta, x);
    }
}
}  // namespace

// gemm_batched with a given tile.
template <typename T, int TM>
static int gemm_tiled(cudaStream_t s, int conj_a, int64_t m, int64_t n, int64_t k, T alpha, const T *A, int64_t lda,
                      int64_t sA, const T *B, int64_t ldb, int64_t sB, T beta, T *C, int64_t ldc, int64_t sC, int batch,
                      int tri)
{
    constexpr int GB_M = 16 * TM, GB_N = 16 * TM;
    const unsigned tiles = cdiv(m, GB_M) * cdiv(n, GB_N) * (unsigned)batch;
    // split K when the output tiles cannot fill the GPU twice over, in slices
    // of at least 32 (complex64: 128); up to GB_SMAX slices are summed in a
    // fixed order (one cluster per tile), more of them atomically (products
    // with a long K and only a tile or two of output)
    const bool fp64 = sizeof(T) == sizeof(zd);
    const int64_t kmin = fp64 ? 32 : 128;
    int splits = 1;
    if (tiles < 2 * 152 && k >= (fp64 ? 2 * kmin : 4 * kmin)) {
        const int64_t want = (2 * 152 + tiles - 1) / tiles;
        const int64_t many = k >= 512 ? (want < k / 128 ? want : k / 128) : 0;   // slices of >= 128
        int64_t few = want < k / kmin ? want : k / kmin;                         // slices of >= kmin
        if (few > GB_SMAX) few = GB_SMAX;
        splits = (int)(many > GB_SMAX ? many : few);
        if (splits * batch > 65535) splits = 65535 / batch;
        if (splits < 1) splits = 1;
    }
    int64_t kchunk = (k + splits - 1) / splits;
    kchunk = ((kchunk + GB_K - 1) / GB_K) * GB_K;
    dim3 grid(cdiv(m, GB_M), cdiv(n, GB_N), batch * splits);
    if (grid.y > 65535) return FEAST_EINVAL;
    if (splits == 1) {
        k_gemm<T, TM><<<grid, GB_T, 0, s>>>(conj_a, m, n, k, alpha, A, lda, sA, B, ldb, sB, beta, C, ldc, sC, 1, kchunk,
                                            tri);
        FEAST_LAUNCH_CHECK();
        return FEAST_OK;
    }
    if (splits > GB_SMAX) {
        // C <- beta C first; the slices then add alpha * partial atomically
        if (!(beta.x == 1 && beta.y == 0)) {
            unsigned gx = cdiv((size_t)m * n, 256);
            k_scale<T><<<dim3(gx > 4096 ? 4096 : gx, batch), 256, 0, s>>>(m, n, beta, C, ldc, sC);
            FEAST_LAUNCH_CHECK();
        }
        k_gemm<T, TM><<<grid, GB_T, 0, s>>>(conj_a, m, n, k, alpha, A, lda, sA, B, ldb, sB, beta, C, ldc, sC, splits,
                                            kchunk, tri);
        FEAST_LAUNCH_CHECK();
        return FEAST_OK;
    }
    const size_t red = sizeof(T) * TM * TM * GB_T;
    FEAST_CUDA_TRY(ensure_dyn_smem(k_gemm<T, TM>, red));
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = 1;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = (unsigned)splits;
    cfg.gridDim = grid;
    cfg.blockDim = dim3(GB_T);
    cfg.dynamicSmemBytes = red;
    cfg.stream = s;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    FEAST_CUDA_TRY(cudaLaunchKernelEx(&cfg, k_gemm<T, TM>, conj_a, m, n, k, alpha, A, lda, sA, B, ldb, sB, beta, C, ldc,
                                      sC, splits, kchunk, tri));
    FEAST_LAUNCH_CHECK();
    return FEAST_OK;
}

template <typename T>
int gemm_batched(cudaStream_t s, int conj_a, int64_t m, int64_t n, int64_t k, T alpha,
                 const T *A, int64_t lda, int64_t sA, const T *B, int64_t ldb, int64_t sB,
                 T beta, T *C, int64_t ldc, int64_t sC, int batch, int tri)
{
    if (m <= 0 || n <= 0 || batch <= 0) return FEAST_OK;
    if (batch > 65535) return FEAST_EINVAL;
    if (tri < 0 || tri > 3 || (conj_a && (tri == 1 || tri == 2))) return FEAST_EINVAL;
    // Tile: a 64 x 64 x 32 product keeps one SM's FP64 pipe busy for 137 us
    // (2 DFMA a clock), so a few large tiles leave the other SMs idle, and a
    // smaller tile costs that pipe nothing: 64 x 64 only from eight waves of
    // them on (a last wave then costs at most an eighth), 32 x 32 down to two
    // waves, 16 x 16 below (a rank-32 update of 16 nodes of 200 x 64: 150 ->
    // 30 us).  In FP32 the large tile's reuse pays as soon as it fills the GPU.
    const bool fp64 = sizeof(T) == sizeof(zd);
    auto tiles_of = [&](int tm) { return (long long)cdiv(m, 16 * tm) * cdiv(n, 16 * tm) * batch; };
    const int tm = tiles_of(4) >= (fp64 ? 8 * 152 : 152) ? 4 : (tiles_of(2) >= 2 * 152 || !fp64) ? 2 : 1;
    if (tm == 4) return gemm_tiled<T, 4>(s, conj_a, m, n, k, alpha, A, lda, sA, B, ldb, sB, beta, C, ldc, sC, batch, tri);
    if (tm == 2) return gemm_tiled<T, 2>(s, conj_a, m, n, k, alpha, A, lda, sA, B, ldb, sB, beta, C, ldc, sC, batch, tri);
    return gemm_tiled<T, 1>(s, conj_a, m, n, k, alpha, A, lda, sA, B, ldb, sB, beta, C, ldc, sC, batch, tri);
}
template int gemm_batched<double2>(cudaStream_t, int, int64_t, int64_t, int64_t, double2, const double2 *,
                                   int64_t, int64_t, const double2 *, int64_t, int64_t, double2, double2 *,
                                   int64_t, int64_t, int, int);
template int gemm_batched<float2>(cudaStream_t, int, int64_t, int64_t, int64_t, float2, const float2 *,
                                  int64_t, int64_t, const float2 *, int64_t, int64_t, float2, float2 *,
                                  int64_t, int64_t, int, int);

int zgemm_batched(cudaStream_t s, int conj_a, int64_t m, int64_t n, int64_t k, zd alpha,
                  const zd *A, int64_t lda, int64_t sA, const zd *B, int64_t ldb, int64_t sB,
                  zd beta, zd *C, int64_t ldc, int64_t sC, int batch, int tri)
{
    return gemm_batched<zd>(s, conj_a, m, n, k, alpha, A, lda, sA, B, ldb, sB, beta, C, ldc, sC, batch, tri);
}

// ------------------------------------------------------------------ z_j B - A
namespace {
__global__ void k_form_shifted(int64_t n, const zd *__restrict__ A, const zd *__restrict__ B,
                               int64_t ld, const zd *__restrict__ z, zd *__restrict__ F,
                               int64_t ldf, int64_t sF)
{
    const int j = blockIdx.y;
    const zd zj = z[j];
    const int64_t total = n * n;
    for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < total;
         e += (int64_t)gridDim.x * blockDim.x) {
        int64_t r = e % n, c = e / n;
        zd bij = B ? B[r + c * ld] : zmake(r == c ? 1.0 : 0.0, 0.0);
        F[(int64_t)j * sF + r + c * ldf] = zsub(zmul(zj, bij), A[r + c * ld]);
    }
}
}  // namespace

int zform_shifted(cudaStream_t s, int64_t n, int q, const zd *A, const zd *B, int64_t ld,
                  const zd *z, zd *F, int64_t ldf, int64_t sF)
{
    unsigned gx = cdiv(n * n, 256);
    if (gx > 1024) gx = 1024;
    k_form_shifted<<<dim3(gx, q), 256, 0, s>>>(n, A, B, ld, z, F, ldf, sF);
    FEAST_LAUNCH_CHECK();
    return FEAST_OK;
}

// ------------------------------------------------------------------ diagonal solves
namespace {
constexpr int SV_NB = 32;

// X rows [k0, k0+nb) <- T^{-1} X rows [k0, k0+nb) for the diagonal block T of
// the factor (lower = unit lower L, else upper U).  One thread per column.
template <typename C>
__global__ void k_trsv_diag(int64_t nrhs, int64_t k0, int nb, int lower,
                            const C *F, int64_t ldf, int64_t sF, C *X, int64_t ldx, int64_t sX)
{
    const int b = blockIdx.y;
    const C *Am = F + (int64_t)b * sF;
    C *Xb = X + (int64_t)b * sX;
    __shared__ C T[SV_NB][SV_NB + 1];
    for (int e = threadIdx.x; e < nb * nb; e += blockDim.x) {
        int r = e % nb, c = e / nb;
        T[r][c] = Am[(k0 + r) + (k0 + c) * ldf];
    }
    __syncthreads();
    const int64_t c = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= nrhs) return;
    C x[SV_NB];
#pragma unroll
    for (int r = 0; r < SV_NB; ++r)
        if (r < nb) x[r] = Xb[(k0 + r) + c * ldx];
    if (lower) {
#pragma unroll
        for (int i = 0; i < SV_NB; ++i) {
            if (i >= nb) break;
#pragma unroll
            for (int r = i + 1; r < SV_NB; ++r)
                if (r < nb) cfma(x[r], cneg(T[r][i]), x[i]);
        }
    } else {
#pragma unroll
        for (int i = SV_NB - 1; i >= 0; --i) {
            if (i >= nb) continue;
            x[i] = cdiv(x[i], T[i][i]);
#pragma unroll
            for (int r = 0; r < SV_NB; ++r)
                if (r < i) cfma(x[r], cneg(T[r][i]), x[i]);
        }
    }
#pragma unroll
    for (int r = 0; r < SV_NB; ++r)
        if (r < nb) Xb[(k0 + r) + c * ldx] = x[r];
}


// The same with a warp per column, lane r holding row r: the rows of T and of
// X are divided by the diagonal once (upper), and each step passes one solved
// entry by shuffles.  32 dependent steps instead of 496 multiply-adds per
// thread.
constexpr int SW_W = 8;    // columns (warps) per CTA
template <typename C>
__global__ void __launch_bounds__(32 * SW_W) k_trsv_warp(int64_t nrhs, int64_t k0, int nb, int lower, const C *F,
                                                         int64_t ldf, int64_t sF, C *X, int64_t ldx, int64_t sX)
{
    const int b = blockIdx.y;
    const C *Am = F + (int64_t)b * sF;
    C *Xb = X + (int64_t)b * sX;
    __shared__ C T[SV_NB][SV_NB + 1];
    __shared__ C dinv[SV_NB];
    const int lane = threadIdx.x & 31;
    for (int e = threadIdx.x; e < nb * nb; e += 32 * SW_W) {
        const int r = e % nb, c = e / nb;
        T[r][c] = Am[(k0 + r) + (k0 + c) * ldf];
    }
    __syncthreads();
    if (!lower) {
        if (threadIdx.x < nb) dinv[threadIdx.x] = cdiv(cx<C>(1, 0), T[threadIdx.x][threadIdx.x]);
        __syncthreads();
        for (int e = threadIdx.x; e < nb * nb; e += 32 * SW_W) {
            const int r = e % nb, c = e / nb;
            if (c > r) T[r][c] = cmul(T[r][c], dinv[r]);
        }
        __syncthreads();
    }
    const int64_t c = (int64_t)blockIdx.x * SW_W + (threadIdx.x >> 5);
    if (c >= nrhs) return;
    const bool on = lane < nb;
    C x = on ? Xb[(k0 + lane) + c * ldx] : cx<C>(0, 0);
    if (lower) {
        for (int i = 0; i + 1 < nb; ++i) {
            C xi;
            xi.x = __shfl_sync(0xffffffffu, x.x, i);
            xi.y = __shfl_sync(0xffffffffu, x.y, i);
            if (lane > i && on) cfma(x, cneg(T[lane][i]), xi);
        }
    } else {
        if (on) x = cmul(x, dinv[lane]);
        for (int i = nb - 1; i > 0; --i) {
            C xi;
            xi.x = __shfl_sync(0xffffffffu, x.x, i);
            xi.y = __shfl_sync(0xffffffffu, x.y, i);
            if (lane < i) cfma(x, cneg(T[lane][i]), xi);
        }
    }
    if (on) Xb[(k0 + lane) + c * ldx] = x;
}

// X rows [k0, k0 + nb) <- T^{-1} X rows (see the kernels).  A warp per column
// takes 32 dependent steps, a thread per column 496; in FP64 a warp-wide
// instruction holds its SM quarter's pipe for 64 clocks whatever the lanes, so
// the warp form costs ~8 k clocks per column and quarter (608 quarters)
// against ~127 k per 32 columns: it wins up to 16 columns a quarter (8 nodes x
// 150 columns: 98 -> ~20 us).  In FP32 the warp form always wins (32 nodes x
// 640 columns: 27 -> ~8 us).
template <typename C>
int trsv_diag(cudaStream_t s, int64_t nrhs, int batch, int64_t k0, int nb, int lower, const C *F, int64_t ldf,
              int64_t sF, C *X, int64_t ldx, int64_t sX)
{
    if (sizeof(C) == sizeof(cf) || nrhs * batch <= 16 * 608)
        k_trsv_warp<C><<<dim3(cdiv(nrhs, SW_W), batch), 32 * SW_W, 0, s>>>(nrhs, k0, nb, lower, F, ldf, sF, X, ldx, sX);
    else
        k_trsv_diag<C><<<dim3(cdiv(nrhs, 64), batch), 64, 0, s>>>(nrhs, k0, nb, lower, F, ldf, sF, X, ldx, sX);
    FEAST_LAUNCH_CHECK();
    return FEAST_OK;
}
}  // namespace

// ------------------------------------------------------------------ LU
namespace {
constexpr int LU_NB = 32;     // panel width
constexpr int LU_PT = 512;    // panel threads
constexpr int LU_NBO = 256;   // outer block of the tensor-core LU

// Factor the panel [k0, k0 + nb) x [k0, n) of every batch member: pivot by
// largest modulus (ties -> smallest row), swap within the panel columns,
// scale, rank-1 update of the remaining panel columns.
template <typename T>
__global__ void __launch_bounds__(LU_PT) k_lu_panel(int64_t n, int64_t k0, int nb, T *F,
                                                   int64_t ldf, int64_t sF, int *piv, int64_t pstride,
                                                   int *info, int *row)
{
    typedef typename CxReal<T>::type R;
    const int b = blockIdx.x;
    T *Am = F + (int64_t)b * sF;
    __shared__ R s_val[LU_PT / 32];
    __shared__ int64_t s_idx[LU_PT / 32];
    __shared__ int64_t s_p;
    __shared__ T s_row[LU_NB];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    for (int j = 0; j < nb; ++j) {
        const int64_t col = k0 + j;
        R best = -1;
        int64_t bi = col;
        for (int64_t i = col + threadIdx.x; i < n; i += LU_PT) {
            R v = cabs2(Am[i + col * ldf]);
            if (v > best) { best = v; bi = i; }
        }
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) {
            R ov = __shfl_down_sync(0xffffffffu, best, off);
            int64_t oi = __shfl_down_sync(0xffffffffu, bi, off);
            if (ov > best || (ov == best && oi < bi)) { best = ov; bi = oi; }
        }
        if (lane == 0) { s_val[wid] = best; s_idx[wid] = bi; }
        __syncthreads();
        if (threadIdx.x == 0) {
            R bv = s_val[0];
            int64_t bx = s_idx[0];
            for (int w = 1; w < LU_PT / 32; ++w)
                if (s_val[w] > bv || (s_val[w] == bv && s_idx[w] < bx)) { bv = s_val[w]; bx = s_idx[w]; }
            s_p = bx;
            piv[(int64_t)b * pstride + col] = (int)bx;
            if (bv == 0 && info) {
                // record the first failing block (1-based) and column
                if (atomicCAS(info, 0, b + 1) == 0 && row) *row = (int)col + 1;
            }
        }
        __syncthreads();
        const int64_t p = s_p;
        if (p != col && threadIdx.x < nb) {
            int64_t c = k0 + threadIdx.x;
            T t = Am[col + c * ldf];
            Am[col + c * ldf] = Am[p + c * ldf];
            Am[p + c * ldf] = t;
        }
        __syncthreads();
        if (threadIdx.x < nb) s_row[threadIdx.x] = Am[col + (k0 + threadIdx.x) * ldf];
        __syncthreads();
        const T d = s_row[j];
        if (!cis_zero(d)) {
            for (int64_t i = col + 1 + threadIdx.x; i < n; i += LU_PT) {
                T l = cdiv(Am[i + col * ldf], d);
                Am[i + col * ldf] = l;
                const T nl = cneg(l);
                for (int c = j + 1; c < nb; ++c) {
                    T &a = Am[i + (k0 + c) * ldf];
                    T v = a;
                    cfma(v, nl, s_row[c]);
                    a = v;
                }
            }
        }
        __syncthreads();
    }
}

// Magnitude key of v for the pivot search: non-negative numbers order like
// their bits; 0 for a NaN, 1 for zero.
__device__ __forceinline__ unsigned long long mag_key(double2 v)
{
    const double m = cabs2(v);
    const unsigned long long b = (unsigned long long)__double_as_longlong(m);
    return b > 0x7ff0000000000000ull ? 0ull : b + 1ull;
}
__device__ __forceinline__ unsigned long long mag_key(float2 v)
{
    const unsigned b = __float_as_uint(cabs2(v));
    return b > 0x7f800000u ? 0ull : (unsigned long long)b + 1ull;
}
__device__ __forceinline__ void key_max(unsigned long long &k, int &r, unsigned long long ok, int orow)
{
    if (ok > k || (ok == k && orow < r)) { k = ok; r = orow; }
}

// The same panel by a cluster of C CTAs, each keeping its rows of the panel in
// shared memory: per column every CTA publishes its best candidate (key, row
// index, the row itself) and the owner of the diagonal row publishes that row;
// after one cluster barrier all of them know the pivot, take its row through
// distributed shared memory and update their own rows (two buffers, used
// alternately: a buffer is rewritten only after the barrier that follows its
// last read).  The multipliers come from one reciprocal.  The one-CTA form runs
// on one SM per matrix, and at n = 1000 in FP64 its rank-1 updates and
// divisions keep that SM's FP64 pipe busy for ~600 us a panel (8 nodes: 8 of
// 152 SMs); this one takes ~100 us, and ~60 us instead of 287 us for 32
// complex64 panels of 2048 rows.  Pivots as in the one-CTA form (largest
// modulus, ties to the smallest row).
constexpr int LC_T = 256;
constexpr int LC_MAX = 8;                // CTAs per matrix at most
template <typename T>
struct LuCand {
    T row[LU_NB], cur[LU_NB];
    unsigned long long key, idx;
};
template <typename T>
__global__ void __launch_bounds__(LC_T) k_lu_panel_cl(int64_t n, int64_t k0, int nb, T *F, int64_t ldf, int64_t sF,
                                                      int *piv, int64_t pstride, int *info, int *row, int C, int rp)
{
    extern __shared__ __align__(16) unsigned char lc_raw[];
    T *slab = reinterpret_cast<T *>(lc_raw);
    constexpr int P = LU_NB + 1;
    __shared__ LuCand<T> cand[2];
    __shared__ unsigned long long s_key[LC_T / 32];
    __shared__ int s_idx[LC_T / 32];
    __shared__ T s_row[LU_NB];
    const int t = threadIdx.x, lane = t & 31, wid = t >> 5;
    const int rank = C > 1 ? (int)cluster_rank_id() : 0;
    const int b = blockIdx.x / C;
    T *Am = F + (int64_t)b * sF + k0 + k0 * ldf;
    const int total = (int)(n - k0), r0 = rank * rp;
    const int rows = total - r0 < rp ? (total - r0 > 0 ? total - r0 : 0) : rp;
    for (int c = wid; c < nb; c += LC_T / 32)
        for (int r = lane; r < rows; r += 32) slab[r * P + c] = Am[r0 + r + (int64_t)c * ldf];
    __syncthreads();
    // threads per row of the update: a power of two, all of a row in one warp
    int tpr = 1;
    while (tpr < 32 && 2 * tpr * rows <= LC_T) tpr *= 2;
    const int part = t % tpr, rbeg = t / tpr, rstep = LC_T / tpr;
    const int none = 0x7fffffff;
    unsigned long long key = 0;
    int idx = none;
    for (int r = t; r < rows; r += LC_T) {
        const unsigned long long k = mag_key(slab[r * P]);
        if (idx == none || k > key) { key = k; idx = r0 + r; }
    }
    for (int j = 0; j < nb; ++j) {
        // this CTA's candidate
#pragma unroll
        for (int off = 16; off > 0; off >>= 1)
            key_max(key, idx, __shfl_xor_sync(0xffffffffu, key, off), __shfl_xor_sync(0xffffffffu, idx, off));
        if (lane == 0) { s_key[wid] = key; s_idx[wid] = idx; }
        __syncthreads();
        LuCand<T> &cd = cand[j & 1];
        if (wid == 0) {
            key = lane < LC_T / 32 ? s_key[lane] : 0ull;
            idx = lane < LC_T / 32 ? s_idx[lane] : none;
#pragma unroll
            for (int off = 4; off > 0; off >>= 1)
                key_max(key, idx, __shfl_xor_sync(0xffffffffu, key, off), __shfl_xor_sync(0xffffffffu, idx, off));
            key = __shfl_sync(0xffffffffu, key, 0);
            idx = __shfl_sync(0xffffffffu, idx, 0);
            if (idx != none && lane < nb) cd.row[lane] = slab[(idx - r0) * P + lane];
            if (lane == 0) { cd.key = key; cd.idx = (unsigned long long)idx; }
        } else if (wid == 1 && j >= r0 && j < r0 + rows && lane < nb) {
            cd.cur[lane] = slab[(j - r0) * P + lane];
        }
        if (C > 1) cluster_barrier();
        else __syncthreads();
        // the pivot: the best of the C candidates (every warp finds it)
        unsigned long long bk = 0;
        int bi = none;
        if (lane < C) {
            bk = C > 1 ? peer_load(&cd.key, (unsigned)lane) : cd.key;
            bi = (int)(C > 1 ? peer_load(&cd.idx, (unsigned)lane) : cd.idx);
        }
#pragma unroll
        for (int off = 4; off > 0; off >>= 1)
            key_max(bk, bi, __shfl_xor_sync(0xffffffffu, bk, off), __shfl_xor_sync(0xffffffffu, bi, off));
        bk = __shfl_sync(0xffffffffu, bk, 0);
        bi = __shfl_sync(0xffffffffu, bi, 0);
        const int p = bi;
        const bool own_j = j >= r0 && j < r0 + rows, own_p = p >= r0 && p < r0 + rows;
        if (wid == 0 && lane < nb) {
            const T v = C > 1 ? peer_load(&cd.row[lane], (unsigned)(p / rp)) : cd.row[lane];
            s_row[lane] = v;
            if (own_j) slab[(j - r0) * P + lane] = v;
        } else if (wid == 1 && lane < nb && own_p && p != j) {
            slab[(p - r0) * P + lane] = C > 1 ? peer_load(&cd.cur[lane], (unsigned)(j / rp)) : cd.cur[lane];
        }
        if (rank == 0 && t == 64) {
            piv[(int64_t)b * pstride + k0 + j] = (int)(k0 + p);
            if (bk == 1ull && info) {
                // record the first failing block (1-based) and column
                if (atomicCAS(info, 0, b + 1) == 0 && row) *row = (int)(k0 + j) + 1;
            }
        }
        __syncthreads();
        const T d = s_row[j];
        const bool live = !cis_zero(d);
        const T inv = live ? crecip(d) : cx<T>(0, 0);
        key = 0;
        idx = none;
        T lkeep = cx<T>(0, 0);                               // several threads a row: one row each, its multiplier
        int rkeep = -1;                                      // stored once all of them have read a[j]
        for (int r = rbeg; r < rows; r += rstep) {
            if (r0 + r <= j) continue;
            T *a = slab + r * P;
            if (live) {
                const T l = cmul(a[j], inv), nl = cneg(l);
                for (int c = j + 1 + part; c < nb; c += tpr) {
                    T v = a[c];
                    cfma(v, nl, s_row[c]);
                    a[c] = v;
                }
                if (tpr == 1) a[j] = l;
                else if (part == 0) { lkeep = l; rkeep = r; }
            }
            if (part == 0 && j + 1 < nb) {                   // (part 0 has updated column j + 1 itself)
                const unsigned long long k = mag_key(a[j + 1]);
                if (idx == none || k > key) { key = k; idx = r0 + r; }
            }
        }
        __syncthreads();
        if (rkeep >= 0) slab[rkeep * P + j] = lkeep;
    }
    __syncthreads();
    for (int c = wid; c < nb; c += LC_T / 32)
        for (int r = lane; r < rows; r += 32) Am[r0 + r + (int64_t)c * ldf] = slab[r * P + c];
    if (C > 1) cluster_barrier();                            // no CTA leaves while a peer reads its candidate
}

// The panel [k0, k0 + nb) of every batch member: the cluster form while its
// CTAs' rows fit shared memory (200 KB: n - k0 <= 3096 in FP64, 6200 in
// complex64), the one-CTA form on global memory beyond.  At least 16 rows a CTA:
// below that the barrier costs more than the rows.  A larger batch fills the SMs
// by itself, and then the columns' barriers and repeated searches cost more than
// the split gives.  FP64: 8 CTAs a matrix up to 8 matrices, 4 up to 32, 2 up
// to 64, 1 beyond (whole LU of 200 rows with 1 / 2 / 4 / 8, us: 8 matrices 1245 /
// 1142 / 1049 / 1021, 16 1446 / 1344 / 1252 / 1379, 48 2265 / 2163 / 2360 / 2445,
// 96 3446 / 3747 / 3868 / 4426, 256 8625 / 9272 / 10044 / 11311, and 10475 by the
// one-CTA form on global memory).  complex64: 8 up to 32 matrices, 1 beyond (LU
// of 200 rows with 1 / 8, us: 128 matrices 997 / 1405, 256 1317 / 2162, 1670 by
// the form on global memory; 48 of 800 rows 6547 / 6790, 32 5413 / 5469).
template <typename T>
int lu_panel(cudaStream_t s, int64_t n, int64_t k0, int nb, int batch, T *F, int64_t ldf, int64_t sF, int *piv,
             int64_t pstride, int *info, int *row)
{
    const int64_t total = n - k0;
    const int most = sizeof(T) == sizeof(cf) ? (batch <= 32 ? LC_MAX : 1)
                     : batch <= 8 ? LC_MAX : batch <= 32 ? 4 : batch <= 64 ? 2 : 1;
    auto rows_of = [&](int c) { return (total + c - 1) / c; };
    auto smem_of = [&](int c) { return (size_t)rows_of(c) * (LU_NB + 1) * sizeof(T); };
    int C = 1;
    while (C < LC_MAX && 32 * C <= total && (C < most || smem_of(C) > 200 * 1024)) C *= 2;
    const int64_t rp = rows_of(C);
    const size_t sm = smem_of(C);
    if (sm > 200 * 1024 || (int64_t)batch * C > 0x7fffffff) {
        k_lu_panel<T><<<batch, LU_PT, 0, s>>>(n, k0, nb, F, ldf, sF, piv, pstride, info, row);
        FEAST_LAUNCH_CHECK();
        return FEAST_OK;
    }
    FEAST_CUDA_TRY(ensure_dyn_smem(k_lu_panel_cl<T>, sm));
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = (unsigned)C;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    cfg.gridDim = dim3((unsigned)(batch * C));
    cfg.blockDim = dim3(LC_T);
    cfg.dynamicSmemBytes = sm;
    cfg.stream = s;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    FEAST_CUDA_TRY(cudaLaunchKernelEx(&cfg, k_lu_panel_cl<T>, n, k0, nb, F, ldf, sF, piv, pstride, info, row, C, (int)rp));
    FEAST_LAUNCH_CHECK();
    return FEAST_OK;
}

// Apply the panel's row interchanges to the columns outside the panel.
template <typename T>
__global__ void k_laswp_outside(int64_t n, int64_t k0, int nb, T *F, int64_t ldf, int64_t sF,
                                const int *piv)
{
    const int b = blockIdx.y;
    T *Am = F + (int64_t)b * sF;
    const int *pv = piv + (int64_t)b * n;
    for (int64_t c = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; c < n;
         c += (int64_t)gridDim.x * blockDim.x) {
        if (c >= k0 && c < k0 + nb) continue;
        for (int j = 0; j < nb; ++j) {
            int64_t r = k0 + j, p = pv[r];
            if (p != r) {
                T t = Am[r + c * ldf];
                Am[r + c * ldf] = Am[p + c * ldf];
                Am[p + c * ldf] = t;
            }
        }
    }
}

}  // namespace

template <typename T>
int getrf_batched(cudaStream_t s, int64_t n, int batch, T *F, int64_t ldf, int64_t sF, int *piv,
                  int *info, int *row)
{
    if (n <= 0 || batch <= 0) return FEAST_OK;
    for (int64_t k0 = 0; k0 < n; k0 += LU_NB) {
        int nb = (int)((n - k0) < LU_NB ? (n - k0) : LU_NB);
        int e = lu_panel<T>(s, n, k0, nb, batch, F, ldf, sF, piv, n, info, row);
        if (e) return e;
        unsigned gx = cdiv(n, 128);
        k_laswp_outside<T><<<dim3(gx, batch), 128, 0, s>>>(n, k0, nb, F, ldf, sF, piv);
        FEAST_LAUNCH_CHECK();
        int64_t rest = n - k0 - nb;
        if (rest > 0) {
            e = trsv_diag<T>(s, rest, batch, k0, nb, 1, F, ldf, sF, F + (k0 + nb) * ldf, ldf, sF);
            if (e) return e;
            e = gemm_batched<T>(s, 0, rest, rest, nb, cx<T>(-1, 0), F + k0 + nb + k0 * ldf,
                                    ldf, sF, F + k0 + (k0 + nb) * ldf, ldf, sF, cx<T>(1, 0),
                                    F + (k0 + nb) + (k0 + nb) * ldf, ldf, sF, batch);
            if (e) return e;
        }
    }
    return FEAST_OK;
}
template int getrf_batched<double2>(cudaStream_t, int64_t, int, double2 *, int64_t, int64_t, int *, int *, int *);

// complex64 LU with the bulk of its flops on the tensor cores.  Two-level
// right-looking blocking: an outer block of LU_NBO columns is factored with
// the LU_NB-wide panel kernel as above, except that each inner rank-LU_NB
// update is confined to the outer block's columns (all rows below) and to
// the outer block's rows (columns beyond it); the trailing matrix then takes
// one rank-LU_NBO update A22 -= L21 U12 through the tcgen05 GEMM.  The
// factors and pivots are those of the one-level routine up to rounding.
size_t getrf_tc_scratch_floats(int64_t n, int batch)
{
    return tc_scratch_floats(n, LU_NBO, n, batch);
}

int getrf_batched_tc(cudaStream_t s, int64_t n, int batch, cf *F, int64_t ldf, int64_t sF, int *piv,
                     int *info, int *row, float *scratch, int *tc_err, TcTimer *tt)
{
    if (n <= 0 || batch <= 0) return FEAST_OK;
    const cf mone = cx<cf>(-1, 0), one = cx<cf>(1, 0);
    int e;
    for (int64_t k0 = 0; k0 < n; k0 += LU_NBO) {
        const int64_t nbo = (n - k0) < LU_NBO ? (n - k0) : LU_NBO;
        const int64_t kend = k0 + nbo;                  // first column after the outer block
        for (int64_t kk = k0; kk < kend; kk += LU_NB) {
            const int nb = (int)((kend - kk) < LU_NB ? (kend - kk) : LU_NB);
            if ((e = lu_panel<cf>(s, n, kk, nb, batch, F, ldf, sF, piv, n, info, row))) return e;
            k_laswp_outside<cf><<<dim3(cdiv(n, 128), batch), 128, 0, s>>>(n, kk, nb, F, ldf, sF, piv);
            FEAST_LAUNCH_CHECK();
            const int64_t c1 = kk + nb;                 // first column right of the panel
            if (kend > c1) {
                // inside the outer block only: columns beyond it keep their
                // original values (row swaps included) until the block is done
                if ((e = trsv_diag<cf>(s, kend - c1, batch, kk, nb, 1, F, ldf, sF, F + c1 * ldf, ldf, sF))) return e;
                if ((e = gemm_batched<cf>(s, 0, n - c1, kend - c1, nb, mone, F + c1 + kk * ldf, ldf, sF,
                                          F + kk + c1 * ldf, ldf, sF, one, F + c1 + c1 * ldf, ldf, sF, batch)))
                    return e;
            }
        }
        const int64_t rest = n - kend;
        if (rest <= 0) break;
        // U12 = L11^{-1} A12 for the columns beyond the block, LU_NB rows at a time
        for (int64_t kk = k0; kk < kend; kk += LU_NB) {
            const int nb = (int)((kend - kk) < LU_NB ? (kend - kk) : LU_NB);
            if ((e = trsv_diag<cf>(s, rest, batch, kk, nb, 1, F, ldf, sF, F + kend * ldf, ldf, sF))) return e;
            const int64_t r1 = kk + nb;
            if (r1 < kend) {
                if ((e = gemm_batched<cf>(s, 0, kend - r1, rest, nb, mone, F + r1 + kk * ldf, ldf, sF,
                                          F + kk + kend * ldf, ldf, sF, one, F + r1 + kend * ldf, ldf, sF,
                                          batch)))
                    return e;
            }
        }
        // A22 -= L21 U12   (rest x rest, inner dimension nbo)
        if ((e = tc_cgemm(s, rest, rest, nbo, mone, F + kend + k0 * ldf, ldf, sF, F + k0 + kend * ldf, ldf, sF,
                          one, F + kend + kend * ldf, ldf, sF, batch, scratch, tc_err, tt)))
            return e;
    }
    return FEAST_OK;
}

// Factor only the leading panel (columns 0..nb-1, all rows) of each batch
// member; pivots at piv[b * pstride + k].
template <typename T>
int getrf_panel(cudaStream_t s, int64_t rows, int nb, int batch, T *F, int64_t ldf, int64_t sF,
                int *piv, int64_t pstride, int *info, int *row)
{
    if (rows <= 0 || nb <= 0 || batch <= 0) return FEAST_OK;
    return lu_panel<T>(s, rows, 0, nb, batch, F, ldf, sF, piv, pstride, info, row);
}
template int getrf_panel<double2>(cudaStream_t, int64_t, int, int, double2 *, int64_t, int64_t, int *,
                                  int64_t, int *, int *);
template int getrf_panel<float2>(cudaStream_t, int64_t, int, int, float2 *, int64_t, int64_t, int *,
                                 int64_t, int *, int *);
template int getrf_batched<float2>(cudaStream_t, int64_t, int, float2 *, int64_t, int64_t, int *, int *, int *);

int zgetrf_batched(cudaStream_t s, int64_t n, int batch, zd *F, int64_t ldf, int64_t sF,
                   int *piv, int *info, int *row)
{
    return getrf_batched<zd>(s, n, batch, F, ldf, sF, piv, info, row);
}

// ------------------------------------------------------------------ solves
namespace {
// Apply the interchanges piv[0..n) to each column of X in sequence.
template <typename T>
__global__ void k_laswp_rhs(int64_t n, int64_t nrhs, const int *piv, T *X, int64_t ldx,
                            int64_t sX)
{
    const int b = blockIdx.y;
    T *Xb = X + (int64_t)b * sX;
    const int *pv = piv + (int64_t)b * n;
    const int64_t c = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= nrhs) return;
    for (int64_t k = 0; k < n; ++k) {
        int64_t p = pv[k];
        if (p != k) {
            T t = Xb[k + c * ldx];
            Xb[k + c * ldx] = Xb[p + c * ldx];
            Xb[p + c * ldx] = t;
        }
    }
}

// Composition of the interchanges: perm[i] = original row that ends at i.
__global__ void k_piv_to_perm(int64_t n, const int *piv, int *perm)
{
    const int b = blockIdx.x;
    const int *pv = piv + (int64_t)b * n;
    int *pm = perm + (int64_t)b * n;
    for (int64_t i = threadIdx.x; i < n; i += blockDim.x) pm[i] = (int)i;
    __syncthreads();
    if (threadIdx.x == 0)
        for (int64_t k = 0; k < n; ++k) {
            int64_t p = pv[k];
            if (p != k) { int t = pm[k]; pm[k] = pm[p]; pm[p] = t; }
        }
}

template <typename T>
__global__ void k_gather_rows(int64_t n, int64_t nrhs, const int *perm, const T *R, int64_t ldr,
                              int64_t sR, T *X, int64_t ldx, int64_t sX)
{
    const int b = blockIdx.y;
    const int *pm = perm + (int64_t)b * n;
    const T *Rb = R + (int64_t)b * sR;
    T *Xb = X + (int64_t)b * sX;
    const int64_t total = n * nrhs;
    for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < total;
         e += (int64_t)gridDim.x * blockDim.x) {
        int64_t r = e % n, c = e / n;
        Xb[r + c * ldx] = Rb[pm[r] + c * ldr];
    }
}
}  // namespace

// Complex64 L U solve of already-permuted right-hand sides with the bulk of
// the flops on the tensor cores: outer blocks of LU_NBO rows, solved inside
// with the SV_NB-wide diagonal kernel and SIMT updates confined to the
// block, and one rank-LU_NBO tensor-core update (tc_cgemm) of the rows
// beyond the block per outer step.  scratch: tc_scratch_floats(n, LU_NBO,
// nrhs, batch) floats.
// The off-block panels of the factors as tensor-core left operands, in the
// order trsm_lu_tc uses them: forward (L) panels F[kend:, k0:kend] for
// k0 = 0, LU_NBO, ...; then backward (U) panels F[0:k0, k0:kend] for k0
// from the last block down.
size_t trsm_tc_cache_floats(int64_t n, int batch)
{
    size_t tot = 0;
    for (int64_t k0 = 0; k0 < n; k0 += LU_NBO) {
        const int64_t kend = (k0 + LU_NBO < n) ? k0 + LU_NBO : n;
        if (kend < n) tot += tc_prepA_floats(n - kend, kend - k0, batch);
        if (k0 > 0) tot += tc_prepA_floats(k0, kend - k0, batch);
    }
    return tot;
}

int trsm_tc_cache_fill(cudaStream_t s, int64_t n, int batch, const cf *F, int64_t ldf, int64_t sF, float *cache)
{
    int e;
    size_t off = 0;
    for (int64_t k0 = 0; k0 < n; k0 += LU_NBO) {
        const int64_t kend = (k0 + LU_NBO < n) ? k0 + LU_NBO : n;
        if (kend < n) {
            if ((e = tc_prepare_A(s, n - kend, kend - k0, F + kend + k0 * ldf, ldf, sF, batch, cache + off))) return e;
            off += tc_prepA_floats(n - kend, kend - k0, batch);
        }
    }
    const int64_t last = ((n - 1) / LU_NBO) * LU_NBO;
    for (int64_t k0 = last; k0 >= 0; k0 -= LU_NBO) {
        const int64_t kend = (k0 + LU_NBO < n) ? k0 + LU_NBO : n;
        if (k0 > 0) {
            if ((e = tc_prepare_A(s, k0, kend - k0, F + k0 * ldf, ldf, sF, batch, cache + off))) return e;
            off += tc_prepA_floats(k0, kend - k0, batch);
        }
    }
    return FEAST_OK;
}

int trsm_lu_tc(cudaStream_t s, int64_t n, int64_t nrhs, int batch, const cf *F, int64_t ldf, int64_t sF, cf *X,
               int64_t ldx, int64_t sX, float *scratch, int *tc_err, const float *cache, TcTimer *tt)
{
    if (n <= 0 || nrhs <= 0 || batch <= 0) return FEAST_OK;
    size_t coff = 0;
    const cf mone = cx<cf>(-1, 0), one = cx<cf>(1, 0);
    int e;
    // forward: unit lower L
    for (int64_t k0 = 0; k0 < n; k0 += LU_NBO) {
        const int64_t kend = (k0 + LU_NBO < n) ? k0 + LU_NBO : n;
        for (int64_t kk = k0; kk < kend; kk += SV_NB) {
            const int nb = (int)((kend - kk) < SV_NB ? (kend - kk) : SV_NB);
            if ((e = trsv_diag<cf>(s, nrhs, batch, kk, nb, 1, F, ldf, sF, X, ldx, sX))) return e;
            const int64_t r1 = kk + nb;
            if (r1 < kend &&
                (e = gemm_batched<cf>(s, 0, kend - r1, nrhs, nb, mone, F + r1 + kk * ldf, ldf, sF, X + kk, ldx, sX,
                                      one, X + r1, ldx, sX, batch)))
                return e;
        }
        if (kend < n) {
            if (cache) {
                e = tc_cgemm_prepA(s, n - kend, nrhs, kend - k0, mone, cache + coff, X + k0, ldx, sX, one, X + kend,
                                   ldx, sX, batch, scratch, tc_err, tt);
                coff += tc_prepA_floats(n - kend, kend - k0, batch);
            } else {
                e = tc_cgemm(s, n - kend, nrhs, kend - k0, mone, F + kend + k0 * ldf, ldf, sF, X + k0, ldx, sX, one,
                             X + kend, ldx, sX, batch, scratch, tc_err, tt);
            }
            if (e) return e;
        }
    }
    // backward: upper U
    const int64_t last = ((n - 1) / LU_NBO) * LU_NBO;
    for (int64_t k0 = last; k0 >= 0; k0 -= LU_NBO) {
        const int64_t kend = (k0 + LU_NBO < n) ? k0 + LU_NBO : n;
        const int64_t ilast = k0 + ((kend - k0 - 1) / SV_NB) * SV_NB;
        for (int64_t kk = ilast; kk >= k0; kk -= SV_NB) {
            const int nb = (int)((kend - kk) < SV_NB ? (kend - kk) : SV_NB);
            if ((e = trsv_diag<cf>(s, nrhs, batch, kk, nb, 0, F, ldf, sF, X, ldx, sX))) return e;
            if (kk > k0 &&
                (e = gemm_batched<cf>(s, 0, kk - k0, nrhs, nb, mone, F + k0 + kk * ldf, ldf, sF, X + kk, ldx, sX,
                                      one, X + k0, ldx, sX, batch)))
                return e;
        }
        if (k0 > 0) {
            if (cache) {
                e = tc_cgemm_prepA(s, k0, nrhs, kend - k0, mone, cache + coff, X + k0, ldx, sX, one, X, ldx, sX,
                                   batch, scratch, tc_err, tt);
                coff += tc_prepA_floats(k0, kend - k0, batch);
            } else {
                e = tc_cgemm(s, k0, nrhs, kend - k0, mone, F + k0 * ldf, ldf, sF, X + k0, ldx, sX, one, X, ldx, sX,
                             batch, scratch, tc_err, tt);
            }
            if (e) return e;
        }
    }
    return FEAST_OK;
}

int zpiv_to_perm(cudaStream_t s, int64_t n, int batch, const int *piv, int *perm)
{
    k_piv_to_perm<<<batch, 256, 0, s>>>(n, piv, perm);
    FEAST_LAUNCH_CHECK();
    return FEAST_OK;
}

template <typename T>
int gather_rows(cudaStream_t s, int64_t n, int64_t nrhs, int batch, const int *perm, const T *R,
                int64_t ldr, int64_t sR, T *X, int64_t ldx, int64_t sX)
{
    unsigned gx = cdiv(n * nrhs, 256);
    if (gx > 2048) gx = 2048;
    k_gather_rows<T><<<dim3(gx, batch), 256, 0, s>>>(n, nrhs, perm, R, ldr, sR, X, ldx, sX);
    FEAST_LAUNCH_CHECK();
    return FEAST_OK;
}
template int gather_rows<double2>(cudaStream_t, int64_t, int64_t, int, const int *, const double2 *,
                                  int64_t, int64_t, double2 *, int64_t, int64_t);
template int gather_rows<float2>(cudaStream_t, int64_t, int64_t, int, const int *, const float2 *,
                                 int64_t, int64_t, float2 *, int64_t, int64_t);

int zgather_rows(cudaStream_t s, int64_t n, int64_t nrhs, int batch, const int *perm,
                 const zd *R, int64_t ldr, zd *X, int64_t ldx, int64_t sX)
{
    return gather_rows<zd>(s, n, nrhs, batch, perm, R, ldr, 0, X, ldx, sX);
}

// Forward substitution with the unit-lower factor (in place).
template <typename T>
int trsm_lower_batched(cudaStream_t s, int64_t n, int64_t nrhs, int batch, const T *F, int64_t ldf,
                       int64_t sF, T *X, int64_t ldx, int64_t sX)
{
    if (n <= 0 || nrhs <= 0 || batch <= 0) return FEAST_OK;
    for (int64_t k0 = 0; k0 < n; k0 += SV_NB) {
        int nb = (int)((n - k0) < SV_NB ? (n - k0) : SV_NB);
        int e = trsv_diag<T>(s, nrhs, batch, k0, nb, 1, F, ldf, sF, X, ldx, sX);
        if (e) return e;
        int64_t rest = n - k0 - nb;
        if (rest > 0) {
            e = gemm_batched<T>(s, 0, rest, nrhs, nb, cx<T>(-1, 0), F + (k0 + nb) + k0 * ldf,
                                    ldf, sF, X + k0, ldx, sX, cx<T>(1, 0), X + k0 + nb, ldx, sX,
                                    batch);
            if (e) return e;
        }
    }
    return FEAST_OK;
}

// Back substitution with the upper factor (in place).
template <typename T>
int trsm_upper_batched(cudaStream_t s, int64_t n, int64_t nrhs, int batch, const T *F, int64_t ldf,
                       int64_t sF, T *X, int64_t ldx, int64_t sX)
{
    if (n <= 0 || nrhs <= 0 || batch <= 0) return FEAST_OK;
    int64_t last = ((n - 1) / SV_NB) * SV_NB;
    for (int64_t k0 = last; k0 >= 0; k0 -= SV_NB) {
        int nb = (int)((n - k0) < SV_NB ? (n - k0) : SV_NB);
        int e = trsv_diag<T>(s, nrhs, batch, k0, nb, 0, F, ldf, sF, X, ldx, sX);
        if (e) return e;
        if (k0 > 0) {
            e = gemm_batched<T>(s, 0, k0, nrhs, nb, cx<T>(-1, 0), F + k0 * ldf, ldf, sF,
                                    X + k0, ldx, sX, cx<T>(1, 0), X, ldx, sX, batch);
            if (e) return e;
        }
    }
    return FEAST_OK;
}

// L U solve of already-permuted right-hand sides.
template <typename T>
int trsm_lu_batched(cudaStream_t s, int64_t n, int64_t nrhs, int batch, const T *F, int64_t ldf,
                    int64_t sF, T *X, int64_t ldx, int64_t sX)
{
    int e = trsm_lower_batched<T>(s, n, nrhs, batch, F, ldf, sF, X, ldx, sX);
    if (e) return e;
    return trsm_upper_batched<T>(s, n, nrhs, batch, F, ldf, sF, X, ldx, sX);
}
template int trsm_upper_batched<double2>(cudaStream_t, int64_t, int64_t, int, const double2 *, int64_t,
                                         int64_t, double2 *, int64_t, int64_t);
template int trsm_upper_batched<float2>(cudaStream_t, int64_t, int64_t, int, const float2 *, int64_t,
                                        int64_t, float2 *, int64_t, int64_t);
template int trsm_lu_batched<double2>(cudaStream_t, int64_t, int64_t, int, const double2 *, int64_t,
                                      int64_t, double2 *, int64_t, int64_t);
template int trsm_lu_batched<float2>(cudaStream_t, int64_t, int64_t, int, const float2 *, int64_t,
                                     int64_t, float2 *, int64_t, int64_t);

int ztrsm_lu_batched(cudaStream_t s, int64_t n, int64_t nrhs, int batch, const zd *F,
                     int64_t ldf, int64_t sF, zd *X, int64_t ldx, int64_t sX)
{
    return trsm_lu_batched<zd>(s, n, nrhs, batch, F, ldf, sF, X, ldx, sX);
}

int zgetrs_batched(cudaStream_t s, int64_t n, int64_t nrhs, int batch, const zd *F,
                   int64_t ldf, int64_t sF, const int *piv, zd *X, int64_t ldx, int64_t sX)
{
    if (n <= 0 || nrhs <= 0 || batch <= 0) return FEAST_OK;
    k_laswp_rhs<zd><<<dim3(cdiv(nrhs, 64), batch), 64, 0, s>>>(n, nrhs, piv, X, ldx, sX);
    FEAST_LAUNCH_CHECK();
    return ztrsm_lu_batched(s, n, nrhs, batch, F, ldf, sF, X, ldx, sX);
}

// ------------------------------------------------------------------ node sum
namespace {
__global__ void k_node_sum(int64_t n, int64_t m, int q, const zd *__restrict__ w,
                           const zd *__restrict__ X, int64_t ldx, int64_t sX, zd *__restrict__ U,
                           int64_t ldu)
{
    const int64_t total = n * m;
    for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < total;
         e += (int64_t)gridDim.x * blockDim.x) {
        int64_t r = e % n, c = e / n;
        zd acc = zmake(0.0, 0.0);
        for (int j = 0; j < q; ++j) zfma(acc, w[j], X[(int64_t)j * sX + r + c * ldx]);
        U[r + c * ldu] = acc;
    }
}
}  // namespace

int znode_sum(cudaStream_t s, int64_t n, int64_t m, int q, const zd *w, const zd *X,
              int64_t ldx, int64_t sX, zd *U, int64_t ldu)
{
    unsigned gx = cdiv(n * m, 256);
    if (gx > 152 * 16) gx = 152 * 16;
    k_node_sum<<<gx, 256, 0, s>>>(n, m, q, w, X, ldx, sX, U, ldu);
    FEAST_LAUNCH_CHECK();
    return FEAST_OK;
}

}  // namespace feast
