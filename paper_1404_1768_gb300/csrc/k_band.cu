// Banded pencils (e.g. the 5-point convection-diffusion operator, half
// bandwidth = grid width): formation of z_j B - A in LAPACK general-band
// storage, node-batched blocked band LU with partial pivoting, band solves
// with many right-hand sides, band products and the refinement residual.
//
// Factor storage per node: ldab = 2 kl + ku + 1 rows, kv = kl + ku; entry
// (i, c) lives at F[kv + i - c + c * ldab] for c - kv <= i <= c + kl.  The
// multipliers follow the unblocked convention (each column's multipliers
// are stored as they were when that column was eliminated; later row
// interchanges are not applied to them), so L stays inside kl subdiagonals
// and the solve interleaves interchanges and eliminations column by column.
//
// The LU is blocked by panels of NB columns.  A panel (NB + kl rows) is
// copied to a dense scratch, factored there with the dense panel kernel,
// its interchanges are applied to the columns right of it, U12 = L11^{-1}
// A12 and the trailing update A22 -= L21 U12 (kl x kv, band-masked) follow,
// and the panel is written back with its multipliers converted to the
// unblocked convention.  The solves are sequential along the band (one
// column per step) but parallel over nodes and over chunks of right-hand
// sides; each CTA keeps a sliding window of kl + 1 (forward) or kv + 1
// (backward) rows of its right-hand sides in shared memory.
#include "common.cuh"

namespace feast {

namespace {
constexpr int GB_NB = 32;     // panel width
constexpr int GB_CW = 8;      // right-hand sides per solve CTA (at most; fewer for wide bands)
constexpr int GB_ST = 256;    // solve threads (>= kl and >= kv handled by striding)
constexpr int GB_JC = 32;     // solve steps per staged chunk (at most: one warp's lanes)

__host__ __device__ __forceinline__ int64_t bidx(int64_t kv, int64_t ldab, int64_t i, int64_t c)
{
    return kv + i - c + c * ldab;
}

__device__ __forceinline__ float2 shfl_cx(float2 v, int src)
{
    return make_float2(__shfl_sync(0xffffffffu, v.x, src), __shfl_sync(0xffffffffu, v.y, src));
}
__device__ __forceinline__ double2 shfl_cx(double2 v, int src)
{
    return make_double2(__shfl_sync(0xffffffffu, v.x, src), __shfl_sync(0xffffffffu, v.y, src));
}

// F_j = z_j B - A in factor storage; rows 0..kl-1 of each column (fill) = 0.
template <typename T>
__global__ void k_gb_form(int64_t n, int64_t kl, int64_t ku, const zd *A, const zd *B, int64_t ldin,
                          const zd *z, T *F, int64_t ldab, int64_t sF)
{
    typedef typename CxReal<T>::type R;
    const int j = blockIdx.y;
    const zd zj = z[j];
    const int64_t kv = kl + ku, total = ldab * n;
    for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < total;
         e += (int64_t)gridDim.x * blockDim.x) {
        const int64_t r = e % ldab, c = e / ldab;
        const int64_t i = r - kv + c;  // matrix row of this slot
        zd v = zmake(0.0, 0.0);
        if (r >= kl && i >= 0 && i < n) {
            const int64_t s = ku + i - c + c * ldin;  // compact storage slot
            zd bij = B ? B[s] : zmake(i == c ? 1.0 : 0.0, 0.0);
            v = zsub(zmul(zj, bij), A[s]);
        }
        F[(int64_t)j * sF + e] = cx<T>((R)v.x, (R)v.y);
    }
}

// Dense scratch of the panel: D(r, cc) = F(k0 + r, k0 + cc), zero outside
// the band or the matrix.  D: rows x NB per node (leading dim ldd).
template <typename T>
__global__ void k_gb_gather(int64_t n, int64_t kl, int64_t ku, int64_t k0, int rows, int nb,
                            const T *F, int64_t ldab, int64_t sF, T *D, int ldd, int64_t sD)
{
    const int b = blockIdx.y;
    const T *Fb = F + (int64_t)b * sF;
    T *Db = D + (int64_t)b * sD;
    const int64_t kv = kl + ku;
    for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < ldd * GB_NB; e += gridDim.x * blockDim.x) {
        const int r = e % ldd, cc = e / ldd;
        const int64_t i = k0 + r, c = k0 + cc;
        T v = cx<T>(0, 0);
        if (r < rows && cc < nb && i - c <= kl && c - i <= kv) v = Fb[bidx(kv, ldab, i, c)];
        Db[r + (int64_t)cc * ldd] = v;
    }
}

// Apply the panel's interchanges to the columns right of it (band-limited).
template <typename T>
__global__ void k_gb_swap_right(int64_t n, int64_t kl, int64_t ku, int64_t k0, int nb, T *F,
                                int64_t ldab, int64_t sF, const int *pivl, int ldp)
{
    const int b = blockIdx.y;
    T *Fb = F + (int64_t)b * sF;
    const int *pv = pivl + (int64_t)b * ldp;
    const int64_t kv = kl + ku;
    const int64_t c = k0 + nb + (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= n || c >= k0 + nb + kv) return;
    for (int j = 0; j < nb; ++j) {
        const int64_t r = k0 + j, p = k0 + pv[j];
        if (p != r && c - r <= kv) {
            T t = Fb[bidx(kv, ldab, r, c)];
            Fb[bidx(kv, ldab, r, c)] = Fb[bidx(kv, ldab, p, c)];
            Fb[bidx(kv, ldab, p, c)] = t;
        }
    }
}

// U12 = L11^{-1} A12 (L11 unit lower from the factored scratch D); U12 is
// written to the band storage and to a dense scratch (nb x kv, ld GB_NB).
template <typename T>
__global__ void k_gb_u12(int64_t n, int64_t kl, int64_t ku, int64_t k0, int nb, T *F, int64_t ldab,
                         int64_t sF, const T *D, int ldd, int64_t sD, T *U, int64_t sU)
{
    const int b = blockIdx.y;
    T *Fb = F + (int64_t)b * sF;
    const T *Db = D + (int64_t)b * sD;
    T *Ub = U + (int64_t)b * sU;
    __shared__ T L[GB_NB][GB_NB + 1];
    for (int e = threadIdx.x; e < nb * nb; e += blockDim.x) L[e % nb][e / nb] = Db[(e % nb) + (e / nb) * ldd];
    __syncthreads();
    const int64_t kv = kl + ku;
    const int cc = blockIdx.x * blockDim.x + threadIdx.x;   // 0 .. kv-1
    const int64_t c = k0 + nb + cc;
    if (cc >= kv) return;
    T x[GB_NB];
#pragma unroll
    for (int r = 0; r < GB_NB; ++r) {
        x[r] = cx<T>(0, 0);
        const int64_t i = k0 + r;
        if (r < nb && c < n && c - i <= kv) x[r] = Fb[bidx(kv, ldab, i, c)];
    }
#pragma unroll
    for (int i = 0; i < GB_NB; ++i) {
        if (i >= nb) break;
#pragma unroll
        for (int r = i + 1; r < GB_NB; ++r)
            if (r < nb) cfma(x[r], cneg(L[r][i]), x[i]);
    }
#pragma unroll
    for (int r = 0; r < GB_NB; ++r) {
        Ub[r + (int64_t)cc * GB_NB] = (r < nb && c < n) ? x[r] : cx<T>(0, 0);
        const int64_t i = k0 + r;
        if (r < nb && c < n && c - i <= kv) Fb[bidx(kv, ldab, i, c)] = x[r];
    }
}

// A22 -= L21 U12 on the band: rows k0+nb .. k0+nb+kl-1, columns
// k0+nb .. k0+nb+kv-1, in-band entries only.  L21 = D rows nb.., U12 scratch.
template <typename T>
__global__ void k_gb_update(int64_t n, int64_t kl, int64_t ku, int64_t k0, int nb, int rows, T *F,
                            int64_t ldab, int64_t sF, const T *D, int ldd, int64_t sD, const T *U,
                            int64_t sU)
{
    const int b = blockIdx.z;
    T *Fb = F + (int64_t)b * sF;
    const T *Lb = D + (int64_t)b * sD + nb;      // row nb of D
    const T *Ub = U + (int64_t)b * sU;
    const int64_t kv = kl + ku;
    __shared__ T Ls[GB_NB][32 + 1];
    __shared__ T Us[GB_NB][32 + 1];
    const int r0 = blockIdx.x * 32, c0 = blockIdx.y * 32;
    const int tx = threadIdx.x % 32, ty = threadIdx.x / 32;   // 32 x 8
    const int lrows = rows - nb;                              // rows of L21
    for (int e = threadIdx.x; e < 32 * GB_NB; e += blockDim.x) {
        int r = e % 32, k = e / 32;
        Ls[k][r] = (r0 + r < lrows && k < nb) ? Lb[(r0 + r) + (int64_t)k * ldd] : cx<T>(0, 0);
        int c = e % 32;
        Us[k][c] = (c0 + c < kv && k < nb) ? Ub[k + (int64_t)(c0 + c) * GB_NB] : cx<T>(0, 0);
    }
    __syncthreads();
    for (int rr = ty; rr < 32; rr += 8) {
        const int lr = r0 + rr;
        const int64_t i = k0 + nb + lr, c = k0 + nb + c0 + tx;
        if (lr >= lrows || c0 + tx >= kv || c >= n || i >= n) continue;
        if (i - c > kl || c - i > kv) continue;
        T acc = cx<T>(0, 0);
#pragma unroll 8
        for (int k = 0; k < GB_NB; ++k) cfma(acc, Ls[k][rr], Us[k][tx]);
        T &dst = Fb[bidx(kv, ldab, i, c)];
        dst = cadd(dst, cneg(acc));
    }
}

// Write the factored panel back: U part as is, multipliers converted to the
// unblocked convention (undo the later interchanges of the panel), global
// pivots recorded.
template <typename T>
__global__ void k_gb_writeback(int64_t n, int64_t kl, int64_t ku, int64_t k0, int nb, int rows, T *F,
                               int64_t ldab, int64_t sF, const T *D, int ldd, int64_t sD,
                               const int *pivl, int ldp, int *piv)
{
    const int b = blockIdx.x;
    T *Fb = F + (int64_t)b * sF;
    const T *Db = D + (int64_t)b * sD;
    const int *pv = pivl + (int64_t)b * ldp;
    const int64_t kv = kl + ku;
    extern __shared__ unsigned char sm_raw[];
    T *col = reinterpret_cast<T *>(sm_raw);   // rows entries
    for (int j = 0; j < nb; ++j) {
        const int64_t c = k0 + j;
        for (int r = threadIdx.x; r < rows; r += blockDim.x) col[r] = Db[r + (int64_t)j * ldd];
        __syncthreads();
        if (threadIdx.x == 0) {
            for (int t = nb - 1; t > j; --t) {
                const int p = pv[t];
                if (p != t) { T tmp = col[t]; col[t] = col[p]; col[p] = tmp; }
            }
            piv[(int64_t)b * n + c] = (int)(k0 + pv[j]);
        }
        __syncthreads();
        for (int r = threadIdx.x; r < rows; r += blockDim.x) {
            const int64_t i = k0 + r;
            if (i - c <= kl && c - i <= kv) Fb[bidx(kv, ldab, i, c)] = col[r];
        }
        __syncthreads();
    }
}

// Asynchronous global -> shared copies of B bytes (B = 4, 8 or 16); an
// invalid source writes zeros instead (nothing is read).  The staging of
// the next chunk's factor columns runs under the current chunk's solves.
template <int B>
__device__ __forceinline__ void cp_async(void *dst, const void *src, bool valid)
{
    const uint32_t d = (uint32_t)__cvta_generic_to_shared(dst);
    asm volatile("cp.async.ca.shared.global [%0], [%1], %2, %3;" ::"r"(d), "l"(src), "n"(B), "r"(valid ? B : 0)
                 : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_group 0;" ::: "memory"); }

// Division by b in Smith's form (cdiv) with the divisor's part done once -- 32
// divisions in turn are the solve's chain; each quotient n / d is the correctly
// rounded one, by Markstein's correction of n * (1 / d).  FUSED false rounds the
// products of d and of the numerators by themselves, as cdiv compiles: the LU's
// multipliers are cdiv's bit for bit.  FP64: by the reciprocal.
template <typename T, bool FUSED>
struct GbDiv;
template <bool FUSED>
struct GbDiv<cf, FUSED> {
    float r, d, y;
    bool h;
    static __device__ __forceinline__ float mad(float a, float b, float c)
    {
        return FUSED ? fmaf(a, b, c) : __fadd_rn(c, __fmul_rn(a, b));
    }
    __device__ __forceinline__ explicit GbDiv(cf b)
    {
        h = fabsf(b.x) >= fabsf(b.y);
        const float p = h ? b.x : b.y, q = h ? b.y : b.x;
        r = q / p;
        d = mad(q, r, p);
        y = 1.f / d;
    }
    __device__ __forceinline__ float quot(float n) const
    {
        const float q = n * y;
        return fmaf(fmaf(-q, d, n), y, q);
    }
    __device__ __forceinline__ cf operator()(cf a) const
    {
        const float u = h ? a.x : a.y, v = h ? a.y : a.x;
        const float im = mad(-u, r, v);
        return cmakef(quot(mad(v, r, u)), quot(h ? im : -im));
    }
};
template <bool FUSED>
struct GbDiv<zd, FUSED> {
    zd inv;
    __device__ __forceinline__ explicit GbDiv(zd b) : inv(crecip(b)) {}
    __device__ __forceinline__ zd operator()(zd a) const { return zmul(a, inv); }
};

template <int N>
struct GbInt {
    static constexpr int value = N;
};

// C consecutive entries of a row of the window (shared memory), in 16-byte loads
// where they divide it.
template <int C, typename T>
__device__ __forceinline__ void gb_row(T (&v)[C], const T *p)
{
    if constexpr (sizeof(T) < 16 && C * sizeof(T) % 16 == 0) {
        union {
            float4 f[C * sizeof(T) / 16];
            T t[C];
        } u;
#pragma unroll
        for (int i = 0; i < (int)(C * sizeof(T) / 16); ++i) u.f[i] = reinterpret_cast<const float4 *>(p)[i];
#pragma unroll
        for (int i = 0; i < C; ++i) v[i] = u.t[i];
    } else {
#pragma unroll
        for (int i = 0; i < C; ++i) v[i] = p[i];
    }
}
// acc[c] -= f_jj x_jj[c], jj = jj0 .. jc - 1: the factor's entries f[jj * fs], the
// solved rows of the window from slot s on in steps of STEP (+-1, mod WL).
template <int C, int STEP, int CW, typename T>
__device__ __forceinline__ void gb_rank_update(T (&acc)[C], const T *f, int64_t fs, const T *W, int WL, int s, int jj0,
                                               int jc)
{
    int sj = s + STEP * jj0;
    if (sj >= WL) sj -= WL;
    if (sj < 0) sj += WL;
#pragma unroll 4
    for (int jj = jj0; jj < jc; ++jj) {
        const T u = cneg(f[jj * fs]);
        T x[C];
        gb_row<C>(x, W + (size_t)sj * CW);
#pragma unroll
        for (int c = 0; c < C; ++c) cfma(acc[c], u, x[c]);
        sj += STEP;
        if (STEP > 0 && sj == WL) sj = 0;
        if (STEP < 0 && sj < 0) sj = WL - 1;
    }
}

// Forward pass of the solve (unblocked convention: for j = 0..n-1, swap
// rows j and piv[j], then rows j+1 .. j+kl -= l_j x_j), taken jc steps at a
// time.  Within a chunk the interchanges commute to the front: the chunk is
// x <- L'_{jc-1} .. L'_0 P_{jc-1} .. P_0 x with L'_i's column = the later
// interchanges of the chunk applied to l_i (they touch only rows below
// i).  So a chunk is (1) its interchanges on the right-hand sides, (2) a
// unit lower triangular solve on its jc rows (one warp per right-hand
// side, a lane per row, the solved value passed by shuffles), (3) one
// rank-jc update of the kl rows below it.  CTA = (chunk of cw <= GB_CW
// right-hand sides, node); the right-hand sides live in a circular window
// of WL = kl + 1 + jcm rows of cw entries in shared memory, the chunk's
// multipliers (jcm + kl rows x jcm columns, column-major) and pivots beside it,
// in nbuf = 2 buffers when they fit (the next chunk's copied in meanwhile).
//
// Bound by the chain of chunks (512 of them at n = 16384): the solve's shuffles
// and the update's FP32 rate on one SM.  The window keeps the right-hand sides
// of a row together, so an update step reads its cw solved values in cw / 2
// loads; the copies run a warp per column without a division; only the
// interchanges that move a row are walked; up to kl = 128 the two halves of the
// CTA share the right-hand sides of a row.  n = 16384, kl = ku = 128, 16 nodes
// x 64 right-hand sides: before, forward 3.82 ms and backward 7.01 ms.
template <typename T, int CW>
__global__ void __launch_bounds__(GB_ST) k_gb_fwd(int64_t n, int64_t kl, int64_t ku, int64_t nrhs,
                                                  const T *F, int64_t ldab, int64_t sF, const int *piv, T *X,
                                                  int64_t ldx, int64_t sX, int jcm, int nbuf)
{
    constexpr int cw = CW, NW = GB_ST / 32;
    extern __shared__ __align__(16) unsigned char sm_raw[];
    const int WL = (int)(kl + 1 + jcm), LR = (int)(jcm + kl), kv = (int)(kl + ku);
    T *W = reinterpret_cast<T *>(sm_raw);      // WL slots of cw entries: row r of column cc at W[(r % WL) * cw + cc]
    T *const Lb0 = W + (size_t)WL * cw;         // LR x jcm: Lb[jj * LR + rho] = L'(j0 + rho, j0 + jj)
    T *const Lb1 = Lb0 + (size_t)(nbuf - 1) * LR * jcm;
    int *const pb0 = reinterpret_cast<int *>(Lb0 + (size_t)nbuf * LR * jcm);   // the chunk's pivots (global rows)
    int *const pb1 = pb0 + (nbuf - 1) * jcm;
    const int b = blockIdx.y;
    const T *Fb = F + (int64_t)b * sF;
    const int *pv = piv + (int64_t)b * n;
    T *Xb = X + (int64_t)b * sX;
    const int64_t c0 = (int64_t)blockIdx.x * cw;
    const int ncol = (int)((nrhs - c0) < cw ? (nrhs - c0) : cw);
    const int wid = threadIdx.x >> 5, lane = threadIdx.x & 31;
    auto stage = [&](int64_t js, T *Lb, int *ps) {
        const int jcs = (int)((n - js) < jcm ? (n - js) : jcm);
        for (int jj = wid; jj < jcs; jj += NW) {
            const T *col = Fb + bidx(kv, ldab, js, js + jj);
            for (int rho = lane; rho < LR; rho += 32) {
                const bool in = rho > jj && rho <= jj + kl && js + rho < n;
                cp_async<sizeof(T)>(Lb + jj * LR + rho, in ? (const void *)(col + rho) : (const void *)Fb, in);
            }
        }
        if (threadIdx.x < jcs) cp_async<4>(ps + threadIdx.x, pv + js + threadIdx.x, true);
    };
    for (int cc = wid; cc < cw; cc += NW)
        for (int r = lane; r < WL; r += 32) {
            const bool in = r < n && cc < ncol;
            cp_async<sizeof(T)>(W + r * cw + cc, in ? (const void *)(Xb + r + (c0 + cc) * ldx) : (const void *)Xb, in);
        }
    stage(0, Lb0, pb0);
    cp_async_commit();
    int k = 0;
    for (int64_t j0 = 0; j0 < n; j0 += jcm, ++k) {
        const int jc = (int)((n - j0) < jcm ? (n - j0) : jcm);
        const int s0 = (int)(j0 % WL);
        T *Lb = (k & 1) ? Lb1 : Lb0;
        const int *ps = (k & 1) ? pb1 : pb0;
        cp_async_wait_all();
        __syncthreads();
        if (wid < 2) {
            const int pl = lane < jc ? (int)(ps[lane] - j0) : lane;
            unsigned moves = __ballot_sync(0xffffffffu, pl != lane);
            while (moves) {
                const int jp = __ffs(moves) - 1, p = __shfl_sync(0xffffffffu, pl, jp);
                moves &= moves - 1;
                if (wid == 0 && lane < cw) {
                    // (1) the chunk's interchanges, in order, on the right-hand sides
                    int sa = s0 + jp, sb = s0 + p;
                    if (sa >= WL) sa -= WL;
                    if (sb >= WL) sb -= WL;
                    const T t = W[sa * cw + lane];
                    W[sa * cw + lane] = W[sb * cw + lane];
                    W[sb * cw + lane] = t;
                }
                if (wid == 1 && lane < jp) {
                    // L'_jj: the later interchanges of the chunk on column jj
                    T *col = Lb + lane * LR;
                    const T t = col[jp];
                    col[jp] = col[p];
                    col[p] = t;
                }
            }
        }
        __syncthreads();
        const bool more = j0 + jcm < n;
        if (nbuf == 2 && more) {
            stage(j0 + jcm, (k & 1) ? Lb0 : Lb1, (k & 1) ? pb0 : pb1);
            cp_async_commit();
        }
        // (2) unit lower triangular solve on the chunk's rows
        if (wid < cw) {
            int sl = s0 + lane;
            if (sl >= WL) sl -= WL;
            T x = (lane < jc) ? W[sl * cw + wid] : cx<T>(0, 0);
#pragma unroll 8
            for (int jj = 0; jj < jc - 1; ++jj) {
                const T l = cneg(Lb[jj * LR + (lane < jc ? lane : 0)]);
                const T xj = shfl_cx(x, jj);
                if (lane > jj && lane < jc) cfma(x, l, xj);
            }
            if (lane < jc) {
                W[sl * cw + wid] = x;
                if (wid < ncol) Xb[j0 + lane + (c0 + wid) * ldx] = x;
            }
        }
        __syncthreads();
        // (3) rows j0 + jc .. j0 + jc + kl - 1 -= L'(those rows, chunk) x(chunk):
        // a thread per row and all cw right-hand sides, or half of them (one
        // multiplier load per cw products; the x values are broadcast)
        auto update = [&](auto cn, int t0, int step, int cc) {
            constexpr int C = decltype(cn)::value;
            for (int t = t0; t < kl; t += step) {
                if (j0 + jc + t >= n) break;
                int sr = s0 + jc + t;
                while (sr >= WL) sr -= WL;
                T acc[C];
                gb_row<C>(acc, W + sr * cw + cc);
                gb_rank_update<C, 1, CW>(acc, Lb + jc + t, LR, W + cc, WL, s0, 0, jc);
#pragma unroll
                for (int c = 0; c < C; ++c) W[sr * cw + cc + c] = acc[c];
            }
        };
        if (CW >= 4 && kl <= GB_ST / 2)
            update(GbInt<(CW >= 4 ? CW / 2 : CW)>(), threadIdx.x % (GB_ST / 2), GB_ST / 2,
                   (threadIdx.x / (GB_ST / 2)) * (CW / 2));
        else
            update(GbInt<CW>(), threadIdx.x, GB_ST, 0);
        __syncthreads();
        // rows j0 .. j0+jc-1 are final; their slots take rows j0+WL ..
        for (int cc = wid; cc < cw; cc += NW)
            if (lane < jc) {
                const int64_t r = j0 + lane + WL;
                int sl = s0 + lane;
                if (sl >= WL) sl -= WL;
                const bool in = r < n && cc < ncol;
                cp_async<sizeof(T)>(W + sl * cw + cc, in ? (const void *)(Xb + r + (c0 + cc) * ldx) : (const void *)Xb,
                                    in);
            }
        if (nbuf == 1 && more) stage(j0 + jcm, Lb0, pb0);   // (its buffer is free only now)
        cp_async_commit();
    }
    cp_async_wait_all();
}

// Backward pass: for j = n-1..0: x_j /= U(j,j); rows j-kv .. j-1 -= U(:, j) x_j,
// taken jc columns at a time: an upper triangular solve on the chunk's rows
// (a warp per right-hand side; the divisions prepared first, all at once),
// then one rank-jc update of the kv rows above it.  Window of WL = kv + 1 + jcm
// rows; the chunk's columns of U (diagonal included) staged column-major,
// Us[jj * (kv + 1) + t] = U(j - t, j) with j = j1 - jj, in nbuf buffers as in the
// forward pass.
template <typename T, int CW>
__global__ void __launch_bounds__(GB_ST) k_gb_bwd(int64_t n, int64_t kl, int64_t ku, int64_t nrhs,
                                                  const T *F, int64_t ldab, int64_t sF, T *X,
                                                  int64_t ldx, int64_t sX, int jcm, int nbuf)
{
    constexpr int cw = CW, NW = GB_ST / 32;
    extern __shared__ __align__(16) unsigned char sm_raw[];
    const int kv = (int)(kl + ku), WL = kv + 1 + jcm, UL = kv + 1;
    T *W = reinterpret_cast<T *>(sm_raw);      // WL slots of cw entries: row r of column cc at W[(r % WL) * cw + cc]
    T *const Ub0 = W + (size_t)WL * cw;
    T *const Ub1 = Ub0 + (size_t)(nbuf - 1) * jcm * UL;
    const int b = blockIdx.y;
    const T *Fb = F + (int64_t)b * sF;
    T *Xb = X + (int64_t)b * sX;
    const int64_t c0 = (int64_t)blockIdx.x * cw;
    const int ncol = (int)((nrhs - c0) < cw ? (nrhs - c0) : cw);
    const int wid = threadIdx.x >> 5, lane = threadIdx.x & 31;
    auto stage = [&](int64_t js, T *Us) {
        const int jcs = (int)((js + 1) < jcm ? (js + 1) : jcm);
        for (int jj = wid; jj < jcs; jj += NW) {
            const int64_t c = js - jj;
            const T *col = Fb + bidx(kv, ldab, c, c);
            for (int t = lane; t < UL; t += 32) {
                const bool in = c - t >= 0;
                cp_async<sizeof(T)>(Us + jj * UL + t, in ? (const void *)(col - t) : (const void *)Fb, in);
            }
        }
    };
    for (int cc = wid; cc < cw; cc += NW)
        for (int t = lane; t < WL; t += 32) {
            const int64_t r = n - 1 - t;
            if (r < 0) break;
            const bool in = cc < ncol;
            cp_async<sizeof(T)>(W + (int)(r % WL) * cw + cc, in ? (const void *)(Xb + r + (c0 + cc) * ldx)
                                                                : (const void *)Xb, in);
        }
    stage(n - 1, Ub0);
    cp_async_commit();
    int k = 0;
    for (int64_t j1 = n - 1; j1 >= 0; j1 -= jcm, ++k) {
        const int jc = (int)((j1 + 1) < jcm ? (j1 + 1) : jcm);
        const int s1 = (int)(j1 % WL);        // slot of row j1; row j1 - d at s1 - d (mod WL)
        const T *Us = (k & 1) ? Ub1 : Ub0;
        const bool more = j1 - jcm >= 0;
        cp_async_wait_all();
        __syncthreads();
        if (nbuf == 2 && more) {
            stage(j1 - jcm, (k & 1) ? Ub0 : Ub1);
            cp_async_commit();
        }
        // upper triangular solve on rows j1 - jc + 1 .. j1 (lane d: row j1 - d)
        if (wid < cw) {
            int sl = s1 - lane;
            if (sl < 0) sl += WL;
            T x = (lane < jc) ? W[sl * cw + wid] : cx<T>(0, 0);
            const GbDiv<T, true> div((lane < jc) ? Us[lane * UL] : cx<T>(1, 0));
#pragma unroll 8
            for (int jj = 0; jj < jc; ++jj) {
                const int t = lane - jj;
                const bool on = t > 0 && t <= kv && lane < jc;
                const T u = cneg(Us[jj * UL + (on ? t : 0)]);
                const T y = div(x);
                const T xj = shfl_cx(y, jj);
                if (t == 0) x = y;
                if (on) cfma(x, u, xj);
            }
            if (lane < jc) {
                W[sl * cw + wid] = x;
                if (wid < ncol) Xb[j1 - lane + (c0 + wid) * ldx] = x;
            }
        }
        __syncthreads();
        // rows above the chunk: r = j1 - jc - tt, tt = 0 .. kv-1, a thread
        // per row and all cw right-hand sides (column jj reaches it from
        // jj = jc + tt - kv on)
        for (int tt = threadIdx.x; tt < kv; tt += GB_ST) {
            if (j1 - jc - tt < 0) break;
            int sr = s1 - jc - tt;
            while (sr < 0) sr += WL;
            T acc[CW];
            gb_row<CW>(acc, W + sr * cw);
            const int jj0 = jc + tt > kv ? jc + tt - kv : 0;
            gb_rank_update<CW, -1, CW>(acc, Us + jc + tt, (int64_t)UL - 1, W, WL, s1, jj0, jc);
#pragma unroll
            for (int c = 0; c < CW; ++c) W[sr * cw + c] = acc[c];
        }
        __syncthreads();
        // rows j1-jc+1 .. j1 are final; their slots take rows j - WL
        for (int cc = wid; cc < cw; cc += NW)
            if (lane < jc) {
                const int64_t r = j1 - lane - WL;
                int sl = s1 - lane;
                if (sl < 0) sl += WL;
                const bool in = cc < ncol;
                if (r >= 0)
                    cp_async<sizeof(T)>(W + sl * cw + cc, in ? (const void *)(Xb + r + (c0 + cc) * ldx)
                                                             : (const void *)Xb, in);
            }
        if (nbuf == 1 && more) stage(j1 - jcm, Ub0);
        cp_async_commit();
    }
    cp_async_wait_all();
}

// Y = op X with op = A (which 0) or z_j B - A style combinations done by the
// caller; plain band product Y[:, c] = M X[:, c], M in compact storage.
__global__ void k_gb_matmul(int64_t n, int64_t kl, int64_t ku, const zd *M, int64_t ldin,
                            int64_t m, const zd *X, int64_t ldx, zd *Y, int64_t ldy)
{
    const int64_t total = n * m;
    for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < total;
         e += (int64_t)gridDim.x * blockDim.x) {
        const int64_t i = e % n, c = e / n;
        const int64_t j0 = i - kl > 0 ? i - kl : 0, j1 = i + ku < n - 1 ? i + ku : n - 1;
        zd acc = zmake(0.0, 0.0);
        for (int64_t j = j0; j <= j1; ++j) zfma(acc, M[ku + i - j + j * ldin], X[j + c * ldx]);
        Y[i + c * ldy] = acc;
    }
}

// The whole band LU of one node in one cluster of GL_C CTAs (complex64;
// one launch for all nodes), GL_NB columns at a time.  Every CTA of the cluster
// factors the panel's nb + kl rows with partial pivoting (pivot: largest |.|^2,
// the first on ties) -- the same arithmetic in the same order in every CTA, so
// their panels agree bit for bit and nothing is exchanged -- and takes its own
// slice of the kv columns right of the panel: U12 = L11^{-1} A12, then
// A22 -= L21 U12.  A cluster barrier closes each panel; the clusters (nodes)
// never wait for one another.
//
// Bound by the chain of pivots, 32 a panel: a thread keeps its row (RPT rows
// from 256 up) in registers for the whole panel and only its position moves, so
// an interchange costs nothing; each warp offers its best row in shared memory
// and one barrier a column settles the pivot.  The multipliers go back in the
// unblocked convention as they arise (column j by CTA j mod GL_C, at the
// positions of step j).  The slice right of the panel is copied to shared memory
// under the panel and read there through the final positions.  Before, each
// column took four barriers and a pass over the panel in shared memory, and the
// interchanges right of it were a chain of loads and stores in L2: 49.5 ms
// for 16 nodes of n = 16384, kl = ku = 128.
constexpr int GL_T = 256;
constexpr int GL_C = 8;          // CTAs per node (a portable cluster)
constexpr int GL_NB = 32;
// Order of the pivot search: 0 no candidate, 1 a NaN on the diagonal (taken
// when there is nothing else), 2 zero, then by magnitude.
__device__ __forceinline__ unsigned gl_key(cf v, bool diag)
{
    const unsigned b = __float_as_uint(cabs2(v));
    return b > 0x7f800000u ? (diag ? 1u : 0u) : b + 2u;
}
template <int RPT>
__global__ void __launch_bounds__(GL_T) k_gb_lu_fused(int64_t n, int kl, int ku, cf *F, int64_t ldab, int64_t sF,
                                                     int *piv, int tc, int *info, int *row)
{
    constexpr int NB = GL_NB, NW = GL_T / 32;
    extern __shared__ __align__(16) unsigned char sm_raw[];
    __shared__ __align__(16) cf s_row[2][NW][NB];
    __shared__ unsigned s_key[2][NW];
    __shared__ int s_pos[2][NW];
    __shared__ int s_piv[NB];
    const int kv = kl + ku, ldd = NB + kl, ldu = tc + 2;
    const int rank = (int)cluster_rank_id(), kvs = (kv + GL_C - 1) / GL_C;
    const int cb = rank * kvs, ce = (cb + kvs < kv) ? cb + kvs : kv;   // this CTA's columns [cb, ce) right of a panel
    cf *D = reinterpret_cast<cf *>(sm_raw);          // the factored panel by final position, column-major
    cf *U = D + (size_t)ldd * NB;                     // NB x tc slice of U12, row-major
    cf *Tr = U + (size_t)NB * ldu;                    // the rows of tc columns right of the panel, column-major
    int *prow = reinterpret_cast<int *>(Tr + (size_t)tc * ldd);   // row of the panel that ends at a position
    const int b = blockIdx.x / GL_C;
    cf *Fb = F + (int64_t)b * sF;
    int *pvb = piv + (int64_t)b * n;
    const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    const cf zero = cmakef(0.f, 0.f);
    for (int64_t k0 = 0; k0 < n; k0 += NB) {
        const int nb = (int)((n - k0) < NB ? (n - k0) : NB);
        const int rows = (int)((n - k0) < ldd ? (n - k0) : ldd);
        auto gather = [&](int x0) {
            const int w = (ce - x0) < tc ? (ce - x0) : tc;
            for (int cl = wid; cl < w; cl += NW) {
                const int64_t c = k0 + nb + x0 + cl;
                for (int r = lane; r < rows; r += 32) {
                    const bool in = c < n && c - (k0 + r) <= kv;
                    cp_async<sizeof(cf)>(Tr + cl * ldd + r, in ? (const void *)(Fb + bidx(kv, ldab, k0 + r, c)) : (const void *)Fb,
                                         in);
                }
            }
            cp_async_commit();
        };
        // the panel, a row per thread (a warp's loads run along the columns)
        cf a[RPT][NB];
        int pos[RPT];
#pragma unroll
        for (int q = 0; q < RPT; ++q) {
            const int r = tid + q * GL_T;
            pos[q] = r;
#pragma unroll
            for (int cc = 0; cc < NB; ++cc) {
                const bool in = r < rows && cc < nb && r - cc <= kl && cc - r <= kv;
                a[q][cc] = in ? Fb[bidx(kv, ldab, k0 + r, k0 + cc)] : zero;
            }
        }
        if (cb < ce) gather(cb);
        // every CTA holds the panel before any of it is written back
        cluster_barrier();
#pragma unroll
        for (int j = 0; j < NB; ++j) {
            if (j >= nb) break;
            const int pb = j & 1;
            unsigned key[RPT], km = 0;
#pragma unroll
            for (int q = 0; q < RPT; ++q) {
                key[q] = (pos[q] >= j && pos[q] < rows) ? gl_key(a[q][j], pos[q] == j) : 0u;
                km = key[q] > km ? key[q] : km;
            }
            km = __reduce_max_sync(0xffffffffu, km);
            int pm = 0x7fffffff;
#pragma unroll
            for (int q = 0; q < RPT; ++q)
                if (key[q] == km && pos[q] < pm) pm = pos[q];
            pm = __reduce_min_sync(0xffffffffu, pm);
#pragma unroll
            for (int q = 0; q < RPT; ++q)
                if (pos[q] == pm && km > 0) {
#pragma unroll
                    for (int cc = 0; cc < NB; ++cc)
                        if (cc >= j) s_row[pb][wid][cc] = a[q][cc];
                }
            if (lane == 0) {
                s_key[pb][wid] = km;
                s_pos[pb][wid] = pm;
            }
            __syncthreads();
            const unsigned kk = lane < NW ? s_key[pb][lane] : 0u;
            const int pp = lane < NW ? s_pos[pb][lane] : 0x7fffffff;
            const unsigned kbest = __reduce_max_sync(0xffffffffu, kk);
            const int p = __reduce_min_sync(0xffffffffu, (lane < NW && kk == kbest) ? pp : 0x7fffffff);
            const int src = __ffs(__ballot_sync(0xffffffffu, lane < NW && kk == kbest && pp == p)) - 1;
            const cf *pr = s_row[pb][src];
            if (tid == 0) {
                s_piv[j] = p;
                if (kbest == 2u && rank == 0 && info && atomicCAS(info, 0, b + 1) == 0 && row) *row = (int)(k0 + j) + 1;
            }
            const cf d = pr[j];
            const bool live = !cis_zero(d);
            const GbDiv<cf, false> div(live ? d : cmakef(1.f, 0.f));
            const bool store = rank == j % GL_C;
#pragma unroll
            for (int q = 0; q < RPT; ++q) {
                const int o = pos[q];
                if (o == p) pos[q] = j;
                else if (o == j) pos[q] = p;
                if (pos[q] <= j || pos[q] >= rows) continue;
                if (live) {
                    const cf l = div(a[q][j]), nl = cneg(l);
                    a[q][j] = l;
#pragma unroll
                    for (int c2 = 0; c2 < NB; c2 += 2) {
                        if (c2 + 1 <= j) continue;
                        const float4 v = *reinterpret_cast<const float4 *>(pr + c2);
                        if (c2 > j) cfma(a[q][c2], nl, cmakef(v.x, v.y));
                        cfma(a[q][c2 + 1], nl, cmakef(v.z, v.w));
                    }
                }
                if (store && pos[q] - j <= kl) Fb[bidx(kv, ldab, k0 + pos[q], k0 + j)] = a[q][j];
            }
        }
#pragma unroll
        for (int q = 0; q < RPT; ++q) {
            const int o = pos[q];
            if (o >= rows) continue;
            prow[o] = tid + q * GL_T;
#pragma unroll
            for (int cc = 0; cc < NB; ++cc) {
                D[cc * ldd + o] = a[q][cc];
                if (cc % GL_C == rank && o <= cc && cc < nb && cc - o <= kv) Fb[bidx(kv, ldab, k0 + o, k0 + cc)] = a[q][cc];
            }
        }
        __syncthreads();
        if (rank == 0 && tid < nb) pvb[k0 + tid] = (int)(k0 + s_piv[tid]);
        const int R2 = rows - nb, rt = (R2 + 31) / 32;
        for (int x0 = cb; x0 < ce; x0 += tc) {
            const int w = (ce - x0) < tc ? (ce - x0) : tc;
            if (x0 > cb) gather(x0);
            cp_async_wait_all();
            __syncthreads();
            // U12: four columns per warp, a lane per row, the solved values by shuffles
            for (int g = wid * 4; g < w; g += NW * 4) {
                cf x[4];
#pragma unroll
                for (int u = 0; u < 4; ++u) x[u] = (lane < nb && g + u < w) ? Tr[(g + u) * ldd + prow[lane]] : zero;
                for (int i = 0; i + 1 < nb; ++i) {
                    const cf l = cneg(D[i * ldd + lane]);
#pragma unroll
                    for (int u = 0; u < 4; ++u) {
                        const cf xi = shfl_cx(x[u], i);
                        if (lane > i && lane < nb) cfma(x[u], l, xi);
                    }
                }
                if (lane < nb)
#pragma unroll
                    for (int u = 0; u < 4; ++u) {
                        const int64_t c = k0 + nb + x0 + g + u;
                        U[lane * ldu + g + u] = x[u];
                        if (g + u < w && c < n && c - (k0 + lane) <= kv) Fb[bidx(kv, ldab, k0 + lane, c)] = x[u];
                    }
            }
            __syncthreads();
            // A22 -= L21 U12: rows k0 + nb + t (t < R2 <= kl), all inside the
            // band; a warp per 32 rows x 8 columns
            for (int task = wid; task < rt * ((w + 7) / 8); task += NW) {
                const int t = (task % rt) * 32 + lane, c8 = (task / rt) * 8;
                if (t >= R2) continue;
                cf acc[8];
#pragma unroll
                for (int u = 0; u < 8; ++u) acc[u] = zero;
                for (int k = 0; k < nb; ++k) {
                    const cf l = D[k * ldd + nb + t];
                    const float4 *uk = reinterpret_cast<const float4 *>(U + k * ldu + c8);
#pragma unroll
                    for (int u = 0; u < 4; ++u) {
                        const float4 v = uk[u];
                        cfma(acc[2 * u], l, cmakef(v.x, v.y));
                        cfma(acc[2 * u + 1], l, cmakef(v.z, v.w));
                    }
                }
                const int pt = prow[nb + t];
#pragma unroll
                for (int u = 0; u < 8; ++u) {
                    const int64_t c = k0 + nb + x0 + c8 + u;
                    if (c8 + u < w && c < n)
                        Fb[bidx(kv, ldab, k0 + nb + t, c)] = cadd(Tr[(c8 + u) * ldd + pt], cneg(acc[u]));
                }
            }
            __syncthreads();   // (the next columns, or the next panel, come into the same buffers)
        }
        // every CTA's updates (and the panel) are in memory before any
        // CTA reads the next panel
        cluster_barrier();
    }
}

// R_j = RHS - (z_j B - A) X_j for every node (FP64).  B null -> identity.
__global__ void k_gb_residual(int64_t n, int64_t kl, int64_t ku, const zd *A, const zd *B,
                              int64_t ldin, const zd *z, int64_t m, const zd *RHS, const zd *X,
                              zd *R, double *nrm2)
{
    __shared__ double red[32];
    const int jn = blockIdx.y;
    const zd zj = z[jn];
    const zd *Xj = X + (int64_t)jn * n * m;
    zd *Rj = R + (int64_t)jn * n * m;
    const int64_t total = n * m;
    double part = 0.0;
    for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < total;
         e += (int64_t)gridDim.x * blockDim.x) {
        const int64_t i = e % n, c = e / n;
        const int64_t j0 = i - kl > 0 ? i - kl : 0, j1 = i + ku < n - 1 ? i + ku : n - 1;
        zd acc = RHS[i + c * n];
        for (int64_t j = j0; j <= j1; ++j) {
            const int64_t s = ku + i - j + j * ldin;
            zd bij = B ? B[s] : zmake(i == j ? 1.0 : 0.0, 0.0);
            zd mij = zsub(zmul(zj, bij), A[s]);
            zfma(acc, zmake(-mij.x, -mij.y), Xj[j + c * n]);
        }
        Rj[i + c * n] = acc;
        part += zabs2(acc);
    }
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) part += __shfl_xor_sync(0xffffffffu, part, off);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = part;
    __syncthreads();
    if (threadIdx.x == 0) {
        double s = 0.0;
        for (int w = 0; w < (int)(blockDim.x / 32); ++w) s += red[w];
        atomicAdd(nrm2 + jn, s);
    }
}

// ---------------------------------------------- double-single band residual
// Unevaluated float pairs (hi, lo) with error-free products (FMA) and sums;
// the explicit _rn intrinsics keep the compiler from contracting the error
// terms away.  ~48 significant bits.
struct BDS {
    float h, l;
};
__device__ __forceinline__ void bds_mac(BDS &acc, float ah, float al, float xh, float xl)
{
    float p = __fmul_rn(ah, xh);
    float e = __fmaf_rn(ah, xh, -p);
    e = __fmaf_rn(ah, xl, e);
    e = __fmaf_rn(al, xh, e);
    float s = __fadd_rn(acc.h, p);
    float bb = __fsub_rn(s, acc.h);
    float err = __fadd_rn(__fsub_rn(acc.h, __fsub_rn(s, bb)), __fsub_rn(p, bb));
    float t = __fadd_rn(acc.l, __fadd_rn(err, e));
    float h = __fadd_rn(s, t);
    acc.l = __fsub_rn(t, __fsub_rn(h, s));
    acc.h = h;
}

// Complex FP64 values as double-single pairs, packed (hi.re, hi.im, lo.re,
// lo.im): the band of A once at set-up, the solutions X_j before each
// residual.
__global__ void k_z2ds(int64_t count, const zd *__restrict__ x, float4 *__restrict__ y)
{
    for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < count;
         e += (int64_t)gridDim.x * blockDim.x) {
        const zd v = x[e];
        const float hr = (float)v.x, hm = (float)v.y;
        y[e] = make_float4(hr, hm, (float)(v.x - (double)hr), (float)(v.y - (double)hm));
    }
}

// R_j = RHS - z_j X_j + A X_j for B = I (M_j = z_j I - A), the band product
// A X_j in double-single arithmetic on the FP32 pipe (the FP64 pipe is 64x
// slower); nrm2[j] += ||R_j||_F^2.  Thread per (row, column) of one node:
// a warp's A loads are one column of the band (coalesced), its X loads one
// broadcast element.
__global__ void k_gb_residual_ds(int64_t n, int64_t kl, int64_t ku, const float4 *__restrict__ Ads, int64_t ldin,
                                 const zd *__restrict__ z, int64_t m, const zd *__restrict__ RHS,
                                 const zd *__restrict__ X, const float4 *__restrict__ Xds, zd *__restrict__ R,
                                 double *__restrict__ nrm2)
{
    __shared__ double red[32];
    const int jn = blockIdx.y;
    const zd zj = z[jn];
    const zd *Xj = X + (int64_t)jn * n * m;
    const float4 *Dj = Xds + (int64_t)jn * n * m;
    zd *Rj = R + (int64_t)jn * n * m;
    const int64_t total = n * m;
    double part = 0.0;
    for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < total;
         e += (int64_t)gridDim.x * blockDim.x) {
        const int64_t i = e % n, c = e / n;
        const int64_t j0 = i - kl > 0 ? i - kl : 0, j1 = i + ku < n - 1 ? i + ku : n - 1;
        BDS re{0.f, 0.f}, im{0.f, 0.f};
        const float4 *xc = Dj + c * n;
        for (int64_t j = j0; j <= j1; ++j) {
            const float4 a = Ads[ku + i - j + j * ldin];
            const float4 x = xc[j];
            // (a.re + i a.im)(x.re + i x.im), each part hi + lo
            bds_mac(re, a.x, a.z, x.x, x.z);
            bds_mac(re, -a.y, -a.w, x.y, x.w);
            bds_mac(im, a.x, a.z, x.y, x.w);
            bds_mac(im, a.y, a.w, x.x, x.z);
        }
        const zd x = Xj[i + c * n];
        const zd rhs = RHS[i + c * n];
        const zd zx = zmul(zj, x);
        const zd acc = zmake(rhs.x - zx.x + ((double)re.h + (double)re.l),
                             rhs.y - zx.y + ((double)im.h + (double)im.l));
        Rj[i + c * n] = acc;
        part += zabs2(acc);
    }
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) part += __shfl_xor_sync(0xffffffffu, part, off);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = part;
    __syncthreads();
    if (threadIdx.x == 0) {
        double s = 0.0;
        for (int w = 0; w < (int)(blockDim.x / 32); ++w) s += red[w];
        atomicAdd(nrm2 + jn, s);
    }
}
}  // namespace

size_t gb_scratch_elems(int64_t kl, int64_t ku, int q)
{
    // dense panel (NB + kl) x NB and U12 NB x kv per node
    return (size_t)q * ((size_t)(GB_NB + kl) * GB_NB + (size_t)GB_NB * (kl + ku));
}
size_t gb_piv_scratch(int64_t kl, int q) { return (size_t)q * (GB_NB + kl); }

template <typename T>
int gb_form(cudaStream_t s, int64_t n, int64_t kl, int64_t ku, const zd *A, const zd *B,
            int64_t ldin, int q, const zd *z, T *F)
{
    const int64_t ldab = 2 * kl + ku + 1;
    unsigned gx = cdiv(ldab * n, 256);
    if (gx > 2048) gx = 2048;
    k_gb_form<T><<<dim3(gx, q), 256, 0, s>>>(n, kl, ku, A, B, ldin, z, F, ldab, ldab * n);
    FEAST_LAUNCH_CHECK();
    return FEAST_OK;
}

// Shared memory of the one-launch band LU (per CTA) with tc columns right of the
// panel at a time.
static size_t gb_lu_fused_smem(int64_t kl, int tc)
{
    const size_t ldd = (size_t)(GL_NB + kl);
    return (ldd * GL_NB + (size_t)GL_NB * (tc + 2) + (size_t)tc * ldd) * sizeof(cf) + ldd * sizeof(int);
}

template <typename T>
int gb_getrf(cudaStream_t s, int64_t n, int64_t kl, int64_t ku, int q, T *F, int *piv, void *scratch,
             int *pivl, int *info, int *row)
{
    const int64_t ldab = 2 * kl + ku + 1, kv = kl + ku, sF = ldab * n;
    if constexpr (sizeof(T) == sizeof(cf)) {
        // complex64: the whole LU of each node in one cluster when the band is
        // narrow enough that the cluster's share of the trailing updates
        // (kl x kv x nb per panel) stays near the panel's own latency; wider
        // bands spread their updates over the whole GPU below.  The widest
        // slice of trailing columns whose shared memory fits (8 always do).
        if (kv <= 512) {
            int tc = (int)((kv + GL_C - 1) / GL_C + 7) & ~7;
            if (tc < 8) tc = 8;
            while (tc > 8 && gb_lu_fused_smem(kl, tc) + 8192 > kSmemOptinMax) tc -= 8;
            const int rpt = (int)((GL_NB + kl + GL_T - 1) / GL_T);
            auto kern = rpt == 1 ? k_gb_lu_fused<1> : rpt == 2 ? k_gb_lu_fused<2> : k_gb_lu_fused<3>;
            const size_t sm = gb_lu_fused_smem(kl, tc);
            FEAST_CUDA_TRY(ensure_dyn_smem(kern, sm));
            cudaLaunchConfig_t cfg = {};
            cudaLaunchAttribute at[1];
            at[0].id = cudaLaunchAttributeClusterDimension;
            at[0].val.clusterDim.x = GL_C;
            at[0].val.clusterDim.y = 1;
            at[0].val.clusterDim.z = 1;
            cfg.gridDim = dim3((unsigned)(q * GL_C));
            cfg.blockDim = dim3(GL_T);
            cfg.dynamicSmemBytes = sm;
            cfg.stream = s;
            cfg.attrs = at;
            cfg.numAttrs = 1;
            FEAST_CUDA_TRY(cudaLaunchKernelEx(&cfg, kern, n, (int)kl, (int)ku, F, ldab, sF, piv, tc, info, row));
            FEAST_LAUNCH_CHECK();
            return FEAST_OK;
        }
    }
    const int ldd = (int)(GB_NB + kl);
    T *D = (T *)scratch;
    const int64_t sD = (int64_t)ldd * GB_NB;
    T *U = D + (size_t)q * sD;
    const int64_t sU = (int64_t)GB_NB * kv;
    for (int64_t k0 = 0; k0 < n; k0 += GB_NB) {
        const int nb = (int)((n - k0) < GB_NB ? (n - k0) : GB_NB);
        const int rows = (int)((n - k0) < ldd ? (n - k0) : ldd);
        k_gb_gather<T><<<dim3(cdiv((size_t)ldd * GB_NB, 256), q), 256, 0, s>>>(n, kl, ku, k0, rows, nb, F, ldab, sF,
                                                                             D, ldd, sD);
        FEAST_LAUNCH_CHECK();
        // dense panel factorization of the scratch (rows x nb, pivots local)
        int e = getrf_panel<T>(s, rows, nb, q, D, ldd, sD, pivl, ldd, info, row);
        if (e) return e;
        if (kv > 0) {
            k_gb_swap_right<T><<<dim3(cdiv(kv, 128), q), 128, 0, s>>>(n, kl, ku, k0, nb, F, ldab, sF, pivl, ldd);
            FEAST_LAUNCH_CHECK();
            k_gb_u12<T><<<dim3(cdiv(kv, 64), q), 64, 0, s>>>(n, kl, ku, k0, nb, F, ldab, sF, D, ldd, sD, U, sU);
            FEAST_LAUNCH_CHECK();
            if (rows > nb) {
                dim3 g(cdiv(rows - nb, 32), cdiv(kv, 32), q);
                k_gb_update<T><<<g, 256, 0, s>>>(n, kl, ku, k0, nb, rows, F, ldab, sF, D, ldd, sD, U, sU);
                FEAST_LAUNCH_CHECK();
            }
        }
        FEAST_CUDA_TRY(ensure_dyn_smem(k_gb_writeback<T>, (size_t)rows * sizeof(T)));
        k_gb_writeback<T><<<q, 256, (size_t)rows * sizeof(T), s>>>(n, kl, ku, k0, nb, rows, F, ldab, sF, D,
                                                                  ldd, sD, pivl, ldd, piv);
        FEAST_LAUNCH_CHECK();
    }
    return FEAST_OK;
}

// Dynamic shared memory of the band solves (forward, backward) for elements
// of es bytes: the staged factor columns and right-hand-side chunks.
static size_t gb_fwd_smem(int64_t kl, size_t es, int cw, int jcm, int nbuf)
{
    return ((size_t)(kl + 1 + jcm) * cw + (size_t)nbuf * jcm * (jcm + kl)) * es + (size_t)nbuf * jcm * sizeof(int) + 16;
}
static size_t gb_bwd_smem(int64_t kl, int64_t ku, size_t es, int cw, int jcm, int nbuf)
{
    const int64_t kv = kl + ku;
    return ((size_t)(kv + 1 + jcm) * cw + (size_t)nbuf * jcm * (kv + 1)) * es;
}

// Staging of the band solves: the most right-hand sides per CTA (cw), then
// the deepest factor staging (jcm) whose shared memory fits, with the next
// chunk's factor columns double-buffered (nbuf = 2) while a chunk of at
// least 8 steps fits that way.  Wide bands trade all three for the band
// itself: cw = jcm = nbuf = 1 holds a window of kv + 2 rows and one factor
// column.
struct GbPlan {
    int cw, jcm, nbuf;
    size_t smf, smb;
};
static GbPlan gb_plan(int64_t kl, int64_t ku, size_t es)
{
    const size_t lim = kSmemOptinMax - 1024;
    for (int nbuf = 2; nbuf >= 1; --nbuf)
        for (int cw = GB_CW; cw >= 1; cw /= 2)
            for (int jcm = GB_JC; jcm >= (nbuf == 2 ? 8 : 1); jcm /= 2) {
                const size_t f = gb_fwd_smem(kl, es, cw, jcm, nbuf), b = gb_bwd_smem(kl, ku, es, cw, jcm, nbuf);
                if (f <= lim && b <= lim) return GbPlan{cw, jcm, nbuf, f, b};
            }
    // (does not fit: the caller refuses the band)
    return GbPlan{1, 1, 1, gb_fwd_smem(kl, es, 1, 1, 1), gb_bwd_smem(kl, ku, es, 1, 1, 1)};
}

size_t gb_solve_smem_bytes(int64_t kl, int64_t ku, size_t es)
{
    const GbPlan p = gb_plan(kl, ku, es);
    return p.smf > p.smb ? p.smf : p.smb;
}

template <typename T, int CW>
static int gb_solve_cw(cudaStream_t s, int64_t n, int64_t kl, int64_t ku, int q, const T *F, const int *piv,
                       int64_t nrhs, T *X, int64_t ldx, int64_t sX, const GbPlan &pl)
{
    const int64_t ldab = 2 * kl + ku + 1, sF = ldab * n;
    dim3 g(cdiv(nrhs, CW), q);
    FEAST_CUDA_TRY(ensure_dyn_smem(k_gb_fwd<T, CW>, pl.smf));
    FEAST_CUDA_TRY(ensure_dyn_smem(k_gb_bwd<T, CW>, pl.smb));
    k_gb_fwd<T, CW><<<g, GB_ST, pl.smf, s>>>(n, kl, ku, nrhs, F, ldab, sF, piv, X, ldx, sX, pl.jcm, pl.nbuf);
    FEAST_LAUNCH_CHECK();
    k_gb_bwd<T, CW><<<g, GB_ST, pl.smb, s>>>(n, kl, ku, nrhs, F, ldab, sF, X, ldx, sX, pl.jcm, pl.nbuf);
    FEAST_LAUNCH_CHECK();
    return FEAST_OK;
}

template <typename T>
int gb_solve(cudaStream_t s, int64_t n, int64_t kl, int64_t ku, int q, const T *F, const int *piv,
             int64_t nrhs, T *X, int64_t ldx, int64_t sX)
{
    const GbPlan pl = gb_plan(kl, ku, sizeof(T));
    if (pl.smf > kSmemOptinMax - 1024 || pl.smb > kSmemOptinMax - 1024) return FEAST_EINVAL;
    switch (pl.cw) {
    case 8: return gb_solve_cw<T, 8>(s, n, kl, ku, q, F, piv, nrhs, X, ldx, sX, pl);
    case 4: return gb_solve_cw<T, 4>(s, n, kl, ku, q, F, piv, nrhs, X, ldx, sX, pl);
    case 2: return gb_solve_cw<T, 2>(s, n, kl, ku, q, F, piv, nrhs, X, ldx, sX, pl);
    default: return gb_solve_cw<T, 1>(s, n, kl, ku, q, F, piv, nrhs, X, ldx, sX, pl);
    }
}

int gb_matmul(cudaStream_t s, int64_t n, int64_t kl, int64_t ku, const zd *M, int64_t ldin, int64_t m,
              const zd *X, zd *Y)
{
    unsigned gx = cdiv(n * m, 256);
    if (gx > 4096) gx = 4096;
    k_gb_matmul<<<gx, 256, 0, s>>>(n, kl, ku, M, ldin, m, X, n, Y, n);
    FEAST_LAUNCH_CHECK();
    return FEAST_OK;
}

int gb_residual(cudaStream_t s, int64_t n, int64_t kl, int64_t ku, const zd *A, const zd *B,
                int64_t ldin, int q, const zd *z, int64_t m, const zd *RHS, const zd *X, zd *R,
                double *nrm2)
{
    FEAST_CUDA_TRY(cudaMemsetAsync(nrm2, 0, sizeof(double) * q, s));
    unsigned gx = cdiv(n * m, 256);
    if (gx > 1024) gx = 1024;
    k_gb_residual<<<dim3(gx, q), 256, 0, s>>>(n, kl, ku, A, B, ldin, z, m, RHS, X, R, nrm2);
    FEAST_LAUNCH_CHECK();
    return FEAST_OK;
}

template int gb_form<double2>(cudaStream_t, int64_t, int64_t, int64_t, const zd *, const zd *, int64_t, int,
                              const zd *, double2 *);
template int gb_form<float2>(cudaStream_t, int64_t, int64_t, int64_t, const zd *, const zd *, int64_t, int,
                             const zd *, float2 *);
template int gb_getrf<double2>(cudaStream_t, int64_t, int64_t, int64_t, int, double2 *, int *, void *, int *,
                               int *, int *);
template int gb_getrf<float2>(cudaStream_t, int64_t, int64_t, int64_t, int, float2 *, int *, void *, int *,
                              int *, int *);
template int gb_solve<double2>(cudaStream_t, int64_t, int64_t, int64_t, int, const double2 *, const int *,
                               int64_t, double2 *, int64_t, int64_t);
template int gb_solve<float2>(cudaStream_t, int64_t, int64_t, int64_t, int, const float2 *, const int *,
                              int64_t, float2 *, int64_t, int64_t);

int z2ds(cudaStream_t s, int64_t count, const zd *x, float4 *y)
{
    unsigned g = cdiv(count, 256);
    if (g > 4096) g = 4096;
    k_z2ds<<<g, 256, 0, s>>>(count, x, y);
    FEAST_LAUNCH_CHECK();
    return FEAST_OK;
}

int gb_residual_ds(cudaStream_t s, int64_t n, int64_t kl, int64_t ku, const float4 *Ads, int64_t ldin, int q,
                   const zd *z, int64_t m, const zd *RHS, const zd *X, float4 *Xds, zd *R, double *nrm2)
{
    int e;
    if ((e = z2ds(s, (int64_t)q * n * m, X, Xds))) return e;
    FEAST_CUDA_TRY(cudaMemsetAsync(nrm2, 0, sizeof(double) * q, s));
    unsigned gx = cdiv(n * m, 256);
    if (gx > 1024) gx = 1024;
    k_gb_residual_ds<<<dim3(gx, q), 256, 0, s>>>(n, kl, ku, Ads, ldin, z, m, RHS, X, Xds, R, nrm2);
    FEAST_LAUNCH_CHECK();
    return FEAST_OK;
}

}  // namespace feast
