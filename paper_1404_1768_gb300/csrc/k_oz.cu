// FP64-accurate complex GEMM on the bf16 tensor cores (tcgen05, kind::f16)
// by exact integer slicing, for the refinement residual of the precision
// form (and any FP64 product that tolerates 2^-44 K relative to max|A| max|B|).
//
//   C = beta C + alpha_c A B       A: M x K, B: K x N complex128, column-major
//
// Complex as real: A' (2M x 2K) has rows 2i = [Re a_ik, -Im a_ik]_k and
// 2i+1 = [Im a_ik, Re a_ik]_k; B' (2K x N) is B's columns read as
// interleaved reals.  Every row of A' is scaled by a power of two 2^-e_i so
// its entries lie in (-1, 1) and written in base 128 with OZ_S signed digits
// (digit 1 in [-128, 128], later digits in [-64, 64]):
//     A' = diag(2^e) sum_s 128^-s A_s ,   likewise B' = (sum_t 128^-t B_t) diag(2^f).
// Digits are small integers, exact in bf16, and a digit product is exact in
// the FP32 accumulator; so is any sum of products of one weight class
// g = s + t over a K-chunk of OZ_KC terms while it stays below 2^24 (all but
// the last class always do; it can pass it only by a factor 1.13 at worst, and
// rounds then at a weight below 2^-60).  The kernel keeps one tensor-memory
// accumulator per class g = 2..8 (all products with s + t <= OZ_S + 1), reads the classes out after each K-chunk and adds them
// on the integer pipe into two exact int64 sums per entry,
//     hi = sum_(g<=5) 128^(5-g) S_g ,   lo = sum_(g>=6) 128^(8-g) S_g ;
// FP64 enters once per entry, at the end: C gets alpha_c 2^(e_i + f_j - 14)
// 2^-21 (hi + 2^-21 lo).  Integer sums do not depend on their order, so K is
// split over the CTAs of a cluster where the tiles do not fill the GPU evenly,
// with the same result.
// Error, in units of 2^(e_i + f_j) per real product: 2^-50 for each operand's
// digits beyond the seventh and 6 x 64 x 64 x 128^-9 = 1.5 x 2^-49 for class 9,
// 2.5 x 2^-49 in all.  A complex entry sums 2 K of them, and a maximum may be
// just above half of its power of two (a factor 4): at most 1.25 x 2^-45 K
// max_k|A'_ik| max_k|B'_kj| in each component, below 2^-44 K in modulus; random
// data stay near 2^-49 sqrt(K).
//
// Seven base-128 digits are 28 slice products; the eight base-64 digits before
// them were 36 products and left 2.2 times the error, with an FP64 sum per chunk
// that the shorter chunks (512 instead of 2048 terms) would have made a third
// of the time: an FP64 instruction takes 64 clocks of an SM quarter here.
//
// Per CTA: one 128 x 64 tile of A'B' over its share of K.  Warp 8 (one lane)
// streams K-stages of 32 bf16 (64-byte swizzle rows) of all OZ_S slices of both
// operands with TMA into a two-deep ring; warp 9 (one lane) issues the 28 slice
// products per K-step of 16 into the seven accumulators (7 x 64 TMEM columns)
// and commits each stage and each K-chunk; warps 0-7 read the chunks out (TMEM
// lane quarter = warp % 4, columns 0-31 or 32-63) and write the result.  What
// bounds it: the A slices are read from shared memory for every product (4 KB
// per 128 x 64 x 16, 48 clocks for 32 of MMA), which accounts for 0.35 of the
// 0.65 ms that 2048 x 640 x 2048 takes; the rest is not separated yet (the ring
// holds two stages, the read-out of a chunk overlaps nothing).  All waits are bounded; on expiry the CTA
// raises *err and finishes.
#include "tcgen05.cuh"

namespace feast {

namespace {
using namespace tc;

constexpr int OZ_S = 7;                      // digits per operand entry
constexpr int OZ_BITS = 7;                   // base 128
constexpr int OZ_NG = OZ_S;                  // weight classes g = 2 .. OZ_S + 1
constexpr int OZ_BM = 128;                   // rows of A' per tile
constexpr int OZ_BN = 64;                    // columns per tile
constexpr int OZ_BK = 32;                    // bf16 per stage row (64 bytes)
constexpr int OZ_STAGES = 2;
constexpr int OZ_KC = 512;                   // K per exact chunk (real K)
constexpr int OZ_GM = 8;                     // row tiles per raster group
constexpr int OZ_READ = 256;                 // read-out threads
constexpr int OZ_THREADS = OZ_READ + 64;
constexpr int OZ_SMAX = 8;                   // most CTAs that share a tile's K
// most complex K of one launch: its int64 sums gain up to 2^44.1 per chunk (2^18.9 chunks)
constexpr int64_t OZ_KMAX = 1 << 26;
constexpr int OZ_COL1_MAX = 2048;            // longest column of a one-launch right operand
constexpr int OZ_A_TILE = OZ_BM * OZ_BK * 2; // 8 KiB per slice
constexpr int OZ_B_TILE = OZ_BN * OZ_BK * 2; // 4 KiB per slice
constexpr int OZ_STAGE = OZ_S * (OZ_A_TILE + OZ_B_TILE);
static_assert(OZ_STAGES * OZ_STAGE >= OZ_BM * OZ_BN * 16, "the int64 sums of a tile reuse the ring");

__device__ __forceinline__ uint32_t pack_bf16x2(float lo, float hi)
{
    // exact: |digit| <= 128
    const uint32_t a = __float_as_uint(lo) >> 16, b = __float_as_uint(hi) >> 16;
    return a | (b << 16);
}

// A row or column with an Inf or NaN entry: its products are NaN (its
// digits are zero, and the epilogue writes NaN).
constexpr int OZ_NONFINITE = -0x40000000;

// The larger of |Re v|, |Im v| as IEEE bits (non-negative doubles order like
// their bits), folded into mx; bad is set for a non-finite entry.
__device__ __forceinline__ void fold_mag(zd v, unsigned long long &mx, bool &bad)
{
    const unsigned long long a = (unsigned long long)__double_as_longlong(v.x) & 0x7fffffffffffffffull;
    const unsigned long long b = (unsigned long long)__double_as_longlong(v.y) & 0x7fffffffffffffffull;
    const unsigned long long m = a > b ? a : b;
    bad = bad || m >= 0x7ff0000000000000ull;
    mx = m > mx ? m : mx;
}

// The exponent e with |x| < 2^e for the magnitude bits of x (0 for zero).
__device__ __forceinline__ int exponent_of(unsigned long long mx)
{
    if (mx == 0) return 0;
    const int bexp = (int)(mx >> 52);
    return bexp ? bexp - 1022 : 64 - __clzll((long long)mx) - 1074;   // (subnormal)
}

// Warp-wide: the exponent e with max < 2^e (frexp's; 0 for zero), or
// OZ_NONFINITE, in every lane.
__device__ __forceinline__ int warp_exponent(unsigned long long mx, bool bad)
{
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
        const unsigned long long o = __shfl_xor_sync(0xffffffffu, mx, off);
        mx = o > mx ? o : mx;
    }
    if (__any_sync(0xffffffffu, bad)) return OZ_NONFINITE;
    return exponent_of(mx);
}

// e_i with max_k max(|Re a_ik|, |Im a_ik|) < 2^e_i (0 for a zero row).  32 rows
// per CTA, lane = row, the warps share K: reads run along the stored columns.
constexpr int RE_W = 16;
__global__ void __launch_bounds__(32 * RE_W) k_oz_rowexp(int64_t M, int64_t K, const zd *__restrict__ A, int64_t lda,
                                                         int *__restrict__ e)
{
    __shared__ unsigned long long smx[RE_W][32];
    __shared__ int sbad[RE_W][32];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int64_t i = (int64_t)blockIdx.x * 32 + lane;
    unsigned long long mx = 0;
    bool bad = false;
    if (i < M)
        for (int64_t k = w; k < K; k += RE_W) fold_mag(A[i + k * lda], mx, bad);
    smx[w][lane] = mx;
    sbad[w][lane] = bad;
    __syncthreads();
    if (w != 0 || i >= M) return;
    for (int x = 1; x < RE_W; ++x) {
        mx = smx[x][lane] > mx ? smx[x][lane] : mx;
        bad = bad || sbad[x][lane];
    }
    e[i] = bad ? OZ_NONFINITE : exponent_of(mx);
}

// f_j for column j of B (one warp per column); also e_j of a conjugate-
// transposed left operand, whose rows are stored columns.
__global__ void k_oz_colexp(int64_t K, int64_t N, const zd *__restrict__ B, int64_t ldb, int *__restrict__ f)
{
    const int64_t j = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int lane = threadIdx.x & 31;
    if (j >= N) return;
    unsigned long long mx = 0;
    bool bad = false;
    for (int64_t k = lane; k < K; k += 32) fold_mag(B[k + j * ldb], mx, bad);
    const int ex = warp_exponent(mx, bad);
    if (lane == 0) f[j] = ex;
}

// Digits of one real value v (IEEE bits b) scaled by 2^-e into (-1, 1):
// with N_s = rint(128^s v 2^-e) (round half to even), digit s is
// N_s - 128 N_(s-1) -- the same digits as the recursion t = 128 r, d = rint(t),
// r = t - d, whose steps are all exact (a subtracted multiple of 128 is even,
// so it commutes with the rounding).  Each N_s comes from the 53-bit
// significand by an integer shift with round-half-even, so the slicing runs
// on the integer pipe, not the FP64 one (1/64 of the FP32 rate on this part),
// and is exact for subnormal rows too.  (v is finite: rows and columns with
// an Inf or NaN are not sliced.)
__device__ __forceinline__ void digits(unsigned long long b, int e, float (&d)[OZ_S])
{
    const int ex = (int)(b >> 52) & 0x7ff;
    const unsigned long long mant = (b & 0xfffffffffffffull) | (ex ? (1ull << 52) : 0ull);
    const int base = (ex ? ex : 1) - 1075 - e;   // |v| 2^-e = mant 2^base < 1
    const bool neg = (b >> 63) != 0;
    long long prev = 0;
#pragma unroll
    for (int s = 1; s <= OZ_S; ++s) {
        const int rs = -(base + OZ_BITS * s);
        unsigned long long q;
        if (rs <= 0) {
            q = mant << (-rs);                       // (a subnormal row: no bits below the point)
        } else if (rs >= 64) {
            q = 0;                                   // below 2^-11
        } else {
            q = mant >> rs;
            const unsigned long long rem = mant & ((1ull << rs) - 1), half = 1ull << (rs - 1);
            q += (rem > half || (rem == half && (q & 1))) ? 1ull : 0ull;
        }
        const long long N = neg ? -(long long)q : (long long)q;
        d[s - 1] = (float)(int)(N - (prev << OZ_BITS));   // |digit| <= 128: exact
        prev = N;
    }
}

// A' digit planes: plane s is (2M x kp) bf16, row-major, columns K .. kp/2 - 1
// zero padding.  A CTA takes 32 rows x 32 complex columns of A through shared
// memory, read along the stored columns and written along the rows; an entry's
// digits serve both of its rows (those of -x are the negatives).  HBM-bound:
// 16 bytes read and 56 written per entry (at 2048 x 2048 the thread-per-row
// form, whose reads strode through A, took 184 us).
__global__ void __launch_bounds__(256) k_oz_slice_rows(int64_t M, int64_t K, const zd *__restrict__ A, int64_t lda,
                                                       int ct, const int *__restrict__ e,
                                                       uint32_t *__restrict__ planes, int64_t kp)
{
    __shared__ zd tile[32][33];
    const int64_t half = kp / 2, plane = M * kp;   // in 32-bit words
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int64_t i0 = (int64_t)blockIdx.x * 32;
    for (int64_t k0 = (int64_t)blockIdx.y * 32; k0 < half; k0 += (int64_t)gridDim.y * 32) {   // (once up to half = 32 x 65535)
        if (k0 != (int64_t)blockIdx.y * 32) __syncthreads();
        for (int r = w; r < 32; r += 8) {
            const int64_t a = ct ? k0 + lane : i0 + lane, b = ct ? i0 + r : k0 + r;   // stored row, column
            const bool in = ct ? (a < K && b < M) : (a < M && b < K);
            zd v = in ? A[a + b * lda] : zmake(0.0, 0.0);
            if (ct) tile[r][lane] = zconj(v);
            else tile[lane][r] = v;
        }
        __syncthreads();
        const int64_t kc = k0 + lane;
        if (kc >= half) continue;
        for (int r = w; r < 32; r += 8) {
            const int64_t i = i0 + r;
            if (i >= M) break;
            const int ei = e[i];
            float dr[OZ_S], di[OZ_S];
            if (kc < K && ei != OZ_NONFINITE) {
                const zd v = tile[r][lane];
                digits((unsigned long long)__double_as_longlong(v.x), ei, dr);
                digits((unsigned long long)__double_as_longlong(v.y), ei, di);
            } else {
#pragma unroll
                for (int s = 0; s < OZ_S; ++s) { dr[s] = 0.f; di[s] = 0.f; }
            }
            const int64_t o = 2 * i * half + kc;
#pragma unroll
            for (int s = 0; s < OZ_S; ++s) {
                planes[(int64_t)s * plane + o] = pack_bf16x2(dr[s], -di[s]);
                planes[(int64_t)s * plane + o + half] = pack_bf16x2(di[s], dr[s]);
            }
        }
    }
}

// B' digit planes: plane s is (N x kp) bf16, row j = column j of B as
// interleaved reals; a warp per column.
__device__ __forceinline__ void slice_col(int64_t K, int64_t half, int64_t plane, int64_t j, const zd *__restrict__ col,
                                          int fj, int64_t k0, int64_t k1, int step, uint32_t *__restrict__ planes)
{
    for (int64_t kc = k0; kc < k1; kc += step) {
        float d0[OZ_S], d1[OZ_S];
        if (kc < K && fj != OZ_NONFINITE) {
            const zd v = col[kc];
            digits((unsigned long long)__double_as_longlong(v.x), fj, d0);
            digits((unsigned long long)__double_as_longlong(v.y), fj, d1);
        } else {
#pragma unroll
            for (int s = 0; s < OZ_S; ++s) { d0[s] = 0.f; d1[s] = 0.f; }
        }
#pragma unroll
        for (int s = 0; s < OZ_S; ++s) planes[(int64_t)s * plane + j * half + kc] = pack_bf16x2(d0[s], d1[s]);
    }
}
__global__ void __launch_bounds__(256) k_oz_slice_cols(int64_t K, int64_t N, const zd *__restrict__ B, int64_t ldb,
                                                       const int *__restrict__ f, uint32_t *__restrict__ planes,
                                                       int64_t kp)
{
    const int64_t half = kp / 2;
    const int lane = threadIdx.x & 31;
    const int64_t j = (int64_t)blockIdx.x * 8 + (threadIdx.x >> 5);
    if (j >= N) return;
    for (int64_t k0 = (int64_t)blockIdx.y * 256; k0 < half; k0 += (int64_t)gridDim.y * 256)   // (once up to 256 x 65535 rows)
        slice_col(K, half, N * half, j, B + j * ldb, f[j], k0 + lane, k0 + 256 < half ? k0 + 256 : half, 32, planes);
}

// The columns' exponents and digits in one launch (K <= OZ_COL1_MAX): w warps
// (1, 2, 4 or 8) per column, which is read a second time from L1.  A small product
// is bound by its launches, and a column's digits waited for all columns' exponents
// (2048 x 640: one launch of 38 us for two of 20 and 34; the whole product 831 -> 813 us).
__global__ void __launch_bounds__(256) k_oz_cols(int64_t K, int64_t N, int w, const zd *__restrict__ B, int64_t ldb,
                                                 int *__restrict__ f, uint32_t *__restrict__ planes, int64_t kp)
{
    __shared__ unsigned long long smx[8];
    __shared__ int sbad[8];
    const int wid = threadIdx.x >> 5, lane = threadIdx.x & 31, sub = wid % w, g0 = wid - sub;
    const int64_t j = (int64_t)blockIdx.x * (8 / w) + wid / w;
    const zd *col = B + j * ldb;
    unsigned long long mx = 0;
    bool bad = false;
    if (j < N)
        for (int64_t k = sub * 32 + lane; k < K; k += 32 * w) fold_mag(col[k], mx, bad);
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
        const unsigned long long o = __shfl_xor_sync(0xffffffffu, mx, off);
        mx = o > mx ? o : mx;
    }
    const int any = __any_sync(0xffffffffu, bad);
    if (lane == 0) {
        smx[wid] = mx;
        sbad[wid] = any;
    }
    __syncthreads();
    if (j >= N) return;
    bad = false;
    for (int x = g0; x < g0 + w; ++x) {
        mx = smx[x] > mx ? smx[x] : mx;
        bad = bad || sbad[x];
    }
    const int fj = bad ? OZ_NONFINITE : exponent_of(mx);
    if (sub == 0 && lane == 0) f[j] = fj;
    const int64_t half = kp / 2;
    slice_col(K, half, N * half, j, col, fj, sub * 32 + lane, half, 32 * w, planes);
}

struct OzOut {
    zd *C;
    int64_t ldc;
    zd alpha;
    const zd *zcol;     // optional per-column-block factor (alpha_c = alpha * zcol[c / cblk])
    int64_t cblk;
    zd beta;
};

// K-blocks from kfirst on, of kr real terms.  splits CTAs (a cluster, 1 to
// OZ_SMAX) share a tile: CTA r takes K-blocks [r kbs, (r + 1) kbs) of them, then
// finishes 64 / splits of the tile's columns from all of their sums.
__global__ void __launch_bounds__(OZ_THREADS, 1)
    k_oz_gemm(const __grid_constant__ CUtensorMap tA, const __grid_constant__ CUtensorMap tB, int mr, int n,
              int kfirst, int kr, int splits, int kbs, const int *__restrict__ ea, const int *__restrict__ fb, OzOut out,
              int *err)
{
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    unsigned char *base = (unsigned char *)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    __shared__ __align__(8) uint64_t full[OZ_STAGES], empty[OZ_STAGES], chunk_full, tmem_empty;
    __shared__ uint32_t tmem_base;
    __shared__ int s_fail;

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int rank = splits > 1 ? (int)(blockIdx.x % splits) : 0;
    // raster: OZ_GM row tiles side by side share each column tile's operands in L2
    const int Mt = (mr + OZ_BM - 1) / OZ_BM, Nt = (n + OZ_BN - 1) / OZ_BN;
    const int L = blockIdx.x / splits;
    const int grp = L / (OZ_GM * Nt);
    const int gbase = grp * OZ_GM;
    const int gsz = (Mt - gbase) < OZ_GM ? (Mt - gbase) : OZ_GM;
    const int rem = L - grp * OZ_GM * Nt;
    const int rt = gbase + rem % gsz, ct = rem / gsz;
    const int row0 = rt * OZ_BM, col0 = ct * OZ_BN;
    const int kb_all = (kr + OZ_BK - 1) / OZ_BK, kb0 = rank * kbs;
    int kb_n = kb_all - kb0 < kbs ? kb_all - kb0 : kbs;    // this CTA's K-blocks (maybe none)
    if (kb_n < 0) kb_n = 0;
    constexpr int KB_CHUNK = OZ_KC / OZ_BK;
    const int nchunk = (kb_n + KB_CHUNK - 1) / KB_CHUNK;

    if (threadIdx.x == 0) {
        for (int s = 0; s < OZ_STAGES; ++s) {
            mbar_init(&full[s], 1);
            mbar_init(&empty[s], 1);
        }
        mbar_init(&chunk_full, 1);
        mbar_init(&tmem_empty, OZ_READ);
        s_fail = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_base)),
                     "r"(512));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    asm volatile("tcgen05.fence::before_thread_sync;");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;");
    const uint32_t tmem = tmem_base;
    // the read-out threads' exact sums: 32 columns each
    long long hi[32], lo[32];

    if (warp == OZ_READ / 32) {
        if (lane == 0) {
            // producer
            int issued = 0;
            for (int kb = 0; kb < kb_n; ++kb) {
                const int s = kb % OZ_STAGES;
                const uint32_t ph = (uint32_t)((kb / OZ_STAGES) & 1);
                if (!mbar_wait(&empty[s], ph ^ 1u) || *(volatile int *)&s_fail) { s_fail = 1; break; }
                unsigned char *st = base + s * OZ_STAGE;
                mbar_expect_tx(&full[s], OZ_STAGE);
                const int kx = (kfirst + kb0 + kb) * OZ_BK;
#pragma unroll 1
                for (int sl = 0; sl < OZ_S; ++sl) {
                    tma_load_3d(st + sl * OZ_A_TILE, &tA, &full[s], kx, row0, sl);
                    tma_load_3d(st + OZ_S * OZ_A_TILE + sl * OZ_B_TILE, &tB, &full[s], kx, col0, sl);
                }
                issued = kb + 1;
            }
            // on failure, let the copies already issued land before the CTA exits
            if (s_fail)
                for (int kb = (issued > OZ_STAGES ? issued - OZ_STAGES : 0); kb < issued; ++kb)
                    mbar_wait(&full[kb % OZ_STAGES], (uint32_t)((kb / OZ_STAGES) & 1));
        }
    } else if (warp == OZ_READ / 32 + 1) {
        if (lane == 0) {
            constexpr uint32_t idesc = idesc_f32acc(1u, OZ_BM, OZ_BN);
            bool ok = true;
            for (int kb = 0; kb < kb_n && ok; ++kb) {
                const int s = kb % OZ_STAGES;
                const uint32_t ph = (uint32_t)((kb / OZ_STAGES) & 1);
                const int chunk = kb / KB_CHUNK;
                const bool first = (kb % KB_CHUNK) == 0;
                if (first && chunk > 0) {
                    // the read-out of the previous chunk must be done
                    if (!mbar_wait(&tmem_empty, (uint32_t)((chunk - 1) & 1))) { ok = false; break; }
                    asm volatile("tcgen05.fence::after_thread_sync;");
                }
                if (!mbar_wait(&full[s], ph) || *(volatile int *)&s_fail) { ok = false; break; }
                asm volatile("tcgen05.fence::after_thread_sync;");
                unsigned char *st = base + s * OZ_STAGE;
                const uint64_t adesc = sdesc<64>(st), bdesc = sdesc<64>(st + OZ_S * OZ_A_TILE);
#pragma unroll
                for (int kk = 0; kk < OZ_BK / 16; ++kk) {
#pragma unroll
                    for (int sa = 0; sa < OZ_S; ++sa) {
#pragma unroll
                        for (int sb = 0; sb < OZ_S - sa; ++sb) {
                            const int g = sa + sb;
                            const uint64_t ad = adesc + (uint64_t)((sa * OZ_A_TILE + kk * 32) >> 4);
                            const uint64_t bd = bdesc + (uint64_t)((sb * OZ_B_TILE + kk * 32) >> 4);
                            const uint32_t acc = (first && kk == 0 && sa == 0) ? 0u : 1u;
                            mma_f16(tmem + (uint32_t)(g * OZ_BN), ad, bd, idesc, acc);
                        }
                    }
                }
                mma_commit(&empty[s]);
                if ((kb % KB_CHUNK) == KB_CHUNK - 1 || kb == kb_n - 1) mma_commit(&chunk_full);
            }
            if (!ok) s_fail = 1;
        }
    } else {
        // read-out: TMEM lanes 32 (warp % 4) .., columns 32 (warp / 4) ..
#pragma unroll
        for (int j = 0; j < 32; ++j) hi[j] = lo[j] = 0;
        const uint32_t tw = tmem + ((uint32_t)((warp & 3) * 32) << 16) + (uint32_t)((warp >> 2) * 32);
        static_assert(OZ_NG == 7, "the read-out takes seven weight classes");
        for (int c = 0; c < nchunk; ++c) {
            if (!mbar_wait(&chunk_full, (uint32_t)(c & 1)) || *(volatile int *)&s_fail) {
                if (lane == 0) s_fail = 1;
                break;
            }
            asm volatile("tcgen05.fence::after_thread_sync;");
#pragma unroll
            for (int cg = 0; cg < 4; ++cg) {
                uint32_t va[8], vb[8];
                int p01[8], p23[8], p45[8];
                // p = 128 S_g + S_(g+1) fits 32 bits for the first four classes
                // (|S| <= 1.5 2^23, and 1.25 2^23 for the one scaled up)
                tmem_ld8x2(tw + (uint32_t)(0 * OZ_BN + cg * 8), tw + (uint32_t)(1 * OZ_BN + cg * 8), va, vb);
#pragma unroll
                for (int j = 0; j < 8; ++j)
                    p01[j] = __float2int_rn(__uint_as_float(va[j])) * 128 + __float2int_rn(__uint_as_float(vb[j]));
                tmem_ld8x2(tw + (uint32_t)(2 * OZ_BN + cg * 8), tw + (uint32_t)(3 * OZ_BN + cg * 8), va, vb);
#pragma unroll
                for (int j = 0; j < 8; ++j) {
                    p23[j] = __float2int_rn(__uint_as_float(va[j])) * 128 + __float2int_rn(__uint_as_float(vb[j]));
                    hi[cg * 8 + j] += (long long)p01[j] * 16384 + p23[j];
                }
                tmem_ld8x2(tw + (uint32_t)(4 * OZ_BN + cg * 8), tw + (uint32_t)(5 * OZ_BN + cg * 8), va, vb);
#pragma unroll
                for (int j = 0; j < 8; ++j) {
                    lo[cg * 8 + j] += (long long)__float2int_rn(__uint_as_float(va[j])) * 16384;
                    p45[j] = __float2int_rn(__uint_as_float(vb[j]));
                }
                tmem_ld8x2(tw + (uint32_t)(6 * OZ_BN + cg * 8), tw + (uint32_t)(6 * OZ_BN + cg * 8), va, vb);
#pragma unroll
                for (int j = 0; j < 8; ++j)
                    lo[cg * 8 + j] += (long long)p45[j] * 128 + __float2int_rn(__uint_as_float(va[j]));
            }
            asm volatile("tcgen05.fence::before_thread_sync;");
            mbar_arrive(&tmem_empty);
        }
    }
    asm volatile("tcgen05.fence::before_thread_sync;");
    __syncthreads();   // every copy has landed and every MMA is done: the ring is free
    // sums[(2 column + {hi, lo}) * 128 + row]
    long long *sums = (long long *)base;
    const int quarter = warp & 3, half = warp >> 2;
    if (threadIdx.x < OZ_READ) {
#pragma unroll
        for (int j = 0; j < 32; ++j) {
            long long *q = sums + (size_t)(2 * (half * 32 + j)) * OZ_BM + quarter * 32 + lane;
            q[0] = hi[j];
            q[OZ_BM] = lo[j];
        }
    }
    if (splits > 1) cluster_barrier();
    else __syncthreads();
    if (threadIdx.x < OZ_READ && !s_fail) {
        const int r = row0 + quarter * 32 + lane;            // real row
        const bool im_row = (r & 1) != 0;
        const int64_t ci = r >> 1;
        const int er = (r < mr) ? ea[ci] : 0;
        const int cw = OZ_BN / splits;                       // columns of this CTA
        const bool rd = (out.beta.x != 0.0 || out.beta.y != 0.0);
        // (a real alpha and a unit beta, the common cases, skip the complex products)
        const bool real_alpha = out.zcol == nullptr && out.alpha.y == 0.0;
        const bool unit_beta = out.beta.x == 1.0 && out.beta.y == 0.0;
        // two columns at a time: neighbouring lanes hold the Re and Im rows of
        // one complex row; the even lane finishes the first column, the odd the
        // second
        for (int c2 = rank * cw + half * (cw / 2); c2 < rank * cw + half * (cw / 2) + cw / 2; c2 += 2) {
            double v[2];
#pragma unroll
            for (int t = 0; t < 2; ++t) {
                const long long *q = sums + (size_t)(2 * (c2 + t)) * OZ_BM + quarter * 32 + lane;
                long long h = q[0], l = q[OZ_BM];
                for (int x = 1; x < splits; ++x) {
                    const int pr = (rank + x) % splits;
                    h += peer_load(q, pr);
                    l += peer_load(q + OZ_BM, pr);
                }
                v[t] = fma((double)l, 0x1p-21, (double)h);
            }
            const double o0 = __shfl_xor_sync(0xffffffffu, v[0], 1);
            const double o1 = __shfl_xor_sync(0xffffffffu, v[1], 1);
            const zd d = im_row ? zmake(o1, v[1]) : zmake(v[0], o0);
            const int col = col0 + c2 + (im_row ? 1 : 0);
            if (r >= mr || col >= n) continue;
            zd &C = out.C[ci + (int64_t)col * out.ldc];
            const int fc = fb[col];
            if (er == OZ_NONFINITE || fc == OZ_NONFINITE) {
                C = zmake(__longlong_as_double(0x7ff8000000000000LL), __longlong_as_double(0x7ff8000000000000LL));
                continue;
            }
            // d 2^(e_i + f_j - 35): a power of two built from its bits, or (a
            // result near the ends of the range) ldexp, one rounding
            const int ex = er + fc - 35;
            zd res = (ex >= -1022 && ex <= 1023)
                         ? zscale(d, __longlong_as_double((long long)(ex + 1023) << 52))
                         : zmake(ldexp(d.x, ex), ldexp(d.y, ex));
            if (real_alpha) {
                if (out.alpha.x != 1.0) res = zscale(res, out.alpha.x);
            } else {
                zd al = out.alpha;
                if (out.zcol) al = zmul(al, out.zcol[col / out.cblk]);
                res = zmul(al, res);
            }
            if (rd) res = zadd(res, unit_beta ? C : zmul(out.beta, C));
            C = res;
        }
    }
    __syncthreads();
    if (splits > 1) cluster_barrier();   // no CTA leaves while a peer reads its sums
    if (threadIdx.x == 0 && s_fail) atomicOr(err, TO_OZ);
    if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512));
}

int64_t oz_kp(int64_t K) { return ((2 * K + 63) / 64) * 64; }
}  // namespace

size_t oz_rows_bytes(int64_t M, int64_t K) { return (size_t)OZ_S * 2 * M * oz_kp(K) * 2 + 256 + 4 * (size_t)M; }
size_t oz_cols_bytes(int64_t K, int64_t N) { return (size_t)OZ_S * N * oz_kp(K) * 2 + 256 + 4 * (size_t)N; }

// Digit planes of the left operand (M x K): A itself, or with ct the
// conjugate transpose of the stored K x M matrix A; at `work`,
// oz_rows_bytes(M, K).
int oz_prepare_rows(cudaStream_t s, int64_t M, int64_t K, const zd *A, int64_t lda, void *work, int ct)
{
    if (M <= 0 || K <= 0) return FEAST_OK;
    const int64_t kp = oz_kp(K);
    uint32_t *planes = (uint32_t *)work;
    int *e = (int *)((char *)work + (size_t)OZ_S * 2 * M * kp * 2 + 256);
    if (ct) k_oz_colexp<<<cdiv((size_t)M * 32, 256), 256, 0, s>>>(K, M, A, lda, e);
    else k_oz_rowexp<<<cdiv((size_t)M, 32), 32 * RE_W, 0, s>>>(M, K, A, lda, e);
    FEAST_LAUNCH_CHECK();
    const unsigned gk = cdiv((size_t)kp / 2, 32);
    k_oz_slice_rows<<<dim3(cdiv((size_t)M, 32), gk > 65535 ? 65535 : gk), 256, 0, s>>>(M, K, A, lda, ct, e, planes, kp);
    FEAST_LAUNCH_CHECK();
    return FEAST_OK;
}

// Digit planes of the right operand B (K x N): at `work`, oz_cols_bytes(K, N).
int oz_prepare_cols(cudaStream_t s, int64_t K, int64_t N, const zd *B, int64_t ldb, void *work)
{
    if (N <= 0 || K <= 0) return FEAST_OK;
    const int64_t kp = oz_kp(K);
    uint32_t *planes = (uint32_t *)work;
    int *f = (int *)((char *)work + (size_t)OZ_S * N * kp * 2 + 256);
    // one launch while a column is a few loads a thread; longer columns spread
    // their slicing over more CTAs than there are columns.  Whole products with
    // one / two launches, us: K = 2048, N = 16 84 / 91, N = 640 147 / 166; K =
    // 16384, N = 16 641 / 684, N = 640 1081 / 1132 (128 rows); two win only where
    // columns are few and long (N = 1, K = 16384 431 / 404, 32768 840 / 768; 16
    // rows), so the line could lie higher
    if (K <= OZ_COL1_MAX) {
        int w = 1;
        while (w < 8 && w * 64 < K) w *= 2;
        k_oz_cols<<<cdiv((size_t)N * w, 8), 256, 0, s>>>(K, N, w, B, ldb, f, planes, kp);
        FEAST_LAUNCH_CHECK();
        return FEAST_OK;
    }
    k_oz_colexp<<<cdiv((size_t)N * 32, 256), 256, 0, s>>>(K, N, B, ldb, f);
    FEAST_LAUNCH_CHECK();
    const unsigned gk = cdiv((size_t)kp / 2, 256);
    k_oz_slice_cols<<<dim3(cdiv((size_t)N, 8), gk > 65535 ? 65535 : gk), 256, 0, s>>>(K, N, B, ldb, f, planes, kp);
    FEAST_LAUNCH_CHECK();
    return FEAST_OK;
}

// C = beta C + alpha_c A B from prepared digit planes (A: M x K rows work,
// B: K x N cols work).  alpha_c = alpha * zcol[c / cblk] when zcol is set.
int oz_gemm(cudaStream_t s, int64_t M, int64_t N, int64_t K, const void *Arows, const void *Bcols, zd alpha,
            const zd *zcol, int64_t cblk, zd beta, zd *C, int64_t ldc, int *err)
{
    if (M <= 0 || N <= 0 || K <= 0) return FEAST_OK;
    const int64_t kp = oz_kp(K);
    const int64_t mr = 2 * M;
    const int *ea = (const int *)((const char *)Arows + (size_t)OZ_S * mr * kp * 2 + 256);
    const int *fb = (const int *)((const char *)Bcols + (size_t)OZ_S * N * kp * 2 + 256);
    CUtensorMap mA, mB;
    int e;
    if ((e = make_map_3d(&mA, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, Arows, kp, mr, OZ_S, kp * 2, mr * kp * 2, OZ_BK,
                         OZ_BM, CU_TENSOR_MAP_SWIZZLE_64B)))
        return e;
    if ((e = make_map_3d(&mB, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, Bcols, kp, N, OZ_S, kp * 2, N * kp * 2, OZ_BK,
                         OZ_BN, CU_TENSOR_MAP_SWIZZLE_64B)))
        return e;
    const size_t smem = (size_t)OZ_STAGES * OZ_STAGE + 1024;
    FEAST_CUDA_TRY(allow_dyn_smem(k_oz_gemm));
    const int64_t tiles = ((mr + OZ_BM - 1) / OZ_BM) * ((N + OZ_BN - 1) / OZ_BN);
    if (tiles > 0x7fffffff) return FEAST_EINVAL;
    // K split over a cluster: the split with the least waves x (its K-blocks at
    // 2 x 28 x 48 clocks + the fixed cost of a CTA: pipeline fill, read-out,
    // result, and the exchange when it shares its tile)
    const int64_t kpiece = K < OZ_KMAX ? K : OZ_KMAX;
    const int kb = (int)((2 * kpiece + OZ_BK - 1) / OZ_BK);
    int splits = 1;
    double best = 0.0;
    for (int x = 1; x <= OZ_SMAX; x *= 2) {
        if (x > 1 && kb / x < 4) break;
        const double waves = (double)((tiles * x + 151) / 152);
        const double cost = waves * (((kb + x - 1) / x) * 2688.0 + (x > 1 ? 14000.0 : 10000.0));
        if (x == 1 || cost < best) {
            best = cost;
            splits = x;
        }
    }
    if (tiles * splits > 0x7fffffff) return FEAST_EINVAL;
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = (unsigned)splits;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    cfg.gridDim = dim3((unsigned)(tiles * splits));
    cfg.blockDim = dim3(OZ_THREADS);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    for (int64_t k0 = 0; k0 < K; k0 += kpiece) {
        OzOut o{C, ldc, alpha, zcol, cblk > 0 ? cblk : 1, k0 ? zmake(1.0, 0.0) : beta};
        const int64_t kn = K - k0 < kpiece ? K - k0 : kpiece;
        FEAST_CUDA_TRY(cudaLaunchKernelEx(&cfg, k_oz_gemm, mA, mB, (int)mr, (int)N, (int)(2 * k0 / OZ_BK), (int)(2 * kn),
                                          splits, (kb + splits - 1) / splits, ea, fb, o, err));
        FEAST_LAUNCH_CHECK();
    }
    return FEAST_OK;
}

}  // namespace feast
