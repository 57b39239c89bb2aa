// Projected eigensolve of more than 64 rows (GFEAST line 6): an FP32 Schur
// form made exact by a Newton iteration whose residual alone is FP64.
//
// The pencil (A, B), B upper triangular, is reduced in FP32: C = B^{-1} A,
// C = Q T Q^H (k_zeig32.cu), T Y = Y Lambda, V = Q Y, L^H = (B V)^{-1} =
// Y^{-1} Q^H B^{-1}.  Then, until what a step leaves is below the caller's
// target,
//
//     R = A V - B V Lambda  (FP64),  W = L^H R,  lambda_j += W_jj,
//     G_ij = W_ij / (lambda_j - lambda_i),  V += V G,  L^H -= G L^H,
//
// as in k_eig_refined (k_zqz.cu), whose file comment has the reasoning: only R
// carries FP64 products, everything else multiplies something small.  Two
// eigenvalues closer than FP32 resolves are separated by the eigenvectors of
// their own 2 x 2 block of Lambda + W.  R's two products are FP64 GEMMs, or
// digit-sliced tensor-core GEMMs (48-bit per row and column) while the
// iteration is still above their resolution.  It replaces a double-single QR
// of the whole matrix (226 ms at 300 rows) and, in the precision form, an
// FP32 QR whose polish took seven digit-sliced products, two FP64 triangular
// inverses and an FP64 back-substitution.
//
// Warm start.  When the filter of line 16 is applied to the Ritz vectors of
// the previous pass, ordered by their expected residual after filtering (r_i /
// |rho(lambda_i)|, rho the filter function of eq. 4.1, so the most converged
// pairs come first), the QR factorisation of line 17 keeps the order, and
// every leading group of converged Ritz vectors spans an (almost) invariant
// subspace: C is block upper triangular up to a small remainder,
//
//     C = [ T11 + E11   C12 ]      T11 upper triangular (k x k),
//         [ E21         C22 ]      E11 strictly lower, E11 and E21 small.
//
// k comes from the norms of the strictly lower parts of C's columns; the
// Schur form is that of the trailing block alone (C22 = Z T22 Z^H, Q =
// diag(I, Z), T = [T11 C12 Z; 0 T22]), and the iteration removes the
// remainder along with FP32's error.  The subspace of every pass is the
// paper's (span of the filtered Ritz vectors = span of the filtered U1); only
// the way the projected problem is solved changes.
#include "common.cuh"

namespace feast {
namespace {

constexpr double RF_NARROW = 1.0 / 16;  // |A - sigma B| / |A| from which A is shifted (prm.find)
constexpr float RF_PAIR = 1.f / 16;   // largest G_ij of a step (beyond: the pair's own block)
constexpr int RF_STEPS = 10;          // most steps
// converged column: strictly lower part <= RF_TAU max|C|.  The iteration
// removes the remainder as it removes FP32's error (a step squares it over a
// gap), so the line is where its first step still contracts: at n = 2048, m0 =
// 640 passes 3 on are warm with 1e-3 and 1e-2 alike (5-9 ms against ~130 ms
// cold), from pass 5 with 3e-6.  A start that does not contract is tried again
// from the columns below RF_TIGHT (pairs outside the contour can pass the first
// line while they are still further off than their gaps: n = 300, 72 pairs
// inside, m0 = 104: 1.1 ms where the cold solve takes 4.6, and 22 if a cluster
// sends that one to the double-single QR), then cold.
constexpr float RF_TAU = 3e-3f, RF_TIGHT = 1e-5f;
constexpr double RF_BERR = 0x1p-52;   // residual column at rounding level: <= RF_BERR m (1 + |lambda'|) (entries of
                                      // A', B' below 1; it measures 6 x 2^-53 at m = 300)
constexpr int RF_PART = 64;           // partial sums of the defect norm

struct RefineStat {
    unsigned gm;                      // bits of max |G|^2 (non-negative floats order like their bits)
    int bad, paired;
    unsigned wm;                      // the same of max |W_ij|^2, i != j
    int tiny;                         // a close pair's coupling at rounding level was seen
    unsigned rm;                      // bits of max_j (|R_j| / (1 + |lambda'_j|))^2
    int pad[2];
};

// Sizes: the iteration runs on A' = 2^-ea A and B' = 2^-eb B, whose largest
// components lie in [1/2, 1), with lambda' = 2^(eb - ea) lambda, since its FP32
// parts square what they compare (couplings of 1e-14 max|C|, gaps): all scales
// are powers of two, so nothing is rounded.  ext[0], ext[1]: high words of
// the largest |component| of A and of the upper triangle of B.
__device__ __forceinline__ unsigned rf_high(zd v)
{
    const unsigned a = (unsigned)__double2hiint(v.x) & 0x7fffffffu, b = (unsigned)__double2hiint(v.y) & 0x7fffffffu;
    return a > b ? a : b;
}
constexpr int RF_EXP = 500;           // largest |exponent| taken
__host__ __device__ inline bool rf_exp_ok(unsigned ext)   // (0x7ff: an Inf or a NaN)
{
    const int x = (int)(ext >> 20) - 1023;
    return x >= -RF_EXP && x <= RF_EXP;
}
__global__ void k_rf_extent(int m, const zd *__restrict__ A, const zd *__restrict__ Bt, unsigned *__restrict__ ext)
{
    const int64_t total = (int64_t)m * m;
    unsigned ma = 0, mb = 0;
    for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < total;
         e += (int64_t)gridDim.x * blockDim.x) {
        const int i = (int)(e % m), j = (int)(e / m);
        const unsigned a = rf_high(A[e]), b = (i <= j) ? rf_high(Bt[e]) : 0u;
        ma = a > ma ? a : ma;
        mb = b > mb ? b : mb;
    }
    ma = __reduce_max_sync(0xffffffffu, ma);
    mb = __reduce_max_sync(0xffffffffu, mb);
    if ((threadIdx.x & 31) == 0) {
        atomicMax(ext, ma);
        atomicMax(ext + 1, mb);
    }
}
__device__ __forceinline__ double rf_scale(unsigned ext)   // 2^-e (1 where the size is out of range: the caller leaves)
{
    const int x = rf_exp_ok(ext) ? (int)(ext >> 20) : 1022;
    return __longlong_as_double((long long)(2045 - x) << 52);
}

// X = [C | I], both m x m: C = A' and the identity in FP32; B32 = the upper
// triangle of B', Bu the same in FP64.  mom (may be null): per block (at most
// RF_MOM of 256 threads) the sums of conj(b) a, |a|^2 and |b|^2.
constexpr int RF_MOM = 256;
__global__ void __launch_bounds__(256) k_rf_cast(int m, const zd *__restrict__ A, const zd *__restrict__ Bt,
                                                 cf *__restrict__ X, cf *__restrict__ B32, zd *__restrict__ Bu,
                                                 const unsigned *__restrict__ ext, float4 *__restrict__ mom)
{
    float4 q = make_float4(0.f, 0.f, 0.f, 0.f);
    const int64_t total = (int64_t)m * m;
    const double fa = rf_scale(ext[0]), fb = rf_scale(ext[1]);
    for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < total;
         e += (int64_t)gridDim.x * blockDim.x) {
        const int i = (int)(e % m), j = (int)(e / m);
        const zd a = A[e], b = (i <= j) ? zscale(Bt[e], fb) : zmake(0.0, 0.0);
        const cf af = cmakef((float)(a.x * fa), (float)(a.y * fa)), bf = cmakef((float)b.x, (float)b.y);
        X[e] = af;
        X[total + e] = cmakef(i == j ? 1.f : 0.f, 0.f);
        B32[e] = bf;
        Bu[e] = b;
        q.x += bf.x * af.x + bf.y * af.y;
        q.y += bf.x * af.y - bf.y * af.x;
        q.z += cabs2(af);
        q.w += cabs2(bf);
    }
    if (!mom) return;
    __shared__ float4 red[8];
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
        q.x += __shfl_xor_sync(0xffffffffu, q.x, off);
        q.y += __shfl_xor_sync(0xffffffffu, q.y, off);
        q.z += __shfl_xor_sync(0xffffffffu, q.z, off);
        q.w += __shfl_xor_sync(0xffffffffu, q.w, off);
    }
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = q;
    __syncthreads();
    if (threadIdx.x != 0) return;
    for (int w = 1; w < 8; ++w) {
        q.x += red[w].x;
        q.y += red[w].y;
        q.z += red[w].z;
        q.w += red[w].w;
    }
    mom[blockIdx.x] = q;
}

__global__ void k_shift_pencil(int m, zd *__restrict__ A, const zd *__restrict__ Bt, zd sigma)
{
    const int64_t total = (int64_t)m * m;
    for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < total;
         e += (int64_t)gridDim.x * blockDim.x)
        if (e % m <= e / m) A[e] = zsub(A[e], zmul(sigma, Bt[e]));
}
__global__ void k_shift_values(int m, zd *__restrict__ alpha, const zd *__restrict__ beta, zd sigma)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < m) alpha[i] = zadd(alpha[i], zmul(sigma, beta[i]));
}

// Per column j of C: ||C[j+1:m, j]||_2 and max_i |C_ij| (Inf for a NaN).  Warp per column.
__global__ void k_col_stats32(int m, const cf *__restrict__ C, float *__restrict__ lower, float *__restrict__ cmax)
{
    const int j = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
    if (j >= m) return;
    const cf *c = C + (int64_t)j * m;
    float s = 0.f, mx = 0.f;
    for (int i = lane; i < m; i += 32) {
        const float a2 = cabs2(c[i]);
        if (i > j) s += a2;
        mx = (a2 <= mx) ? mx : (a2 == a2 ? a2 : __int_as_float(0x7f800000));
    }
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
        s += __shfl_xor_sync(0xffffffffu, s, off);
        mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, off));
    }
    if (lane == 0) {
        lower[j] = sqrtf(s);
        cmax[j] = sqrtf(mx);
    }
}

// Out = In^T, complex64 m x m.
__global__ void k_transpose32(int m, const cf *__restrict__ In, cf *__restrict__ Out)
{
    __shared__ cf tile[32][33];
    const int bx = blockIdx.x * 32, by = blockIdx.y * 32, tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
    for (int r = ty; r < 32; r += 8)
        if (bx + tx < m && by + r < m) tile[r][tx] = In[bx + tx + (int64_t)(by + r) * m];
    __syncthreads();
    for (int r = ty; r < 32; r += 8)
        if (by + tx < m && bx + r < m) Out[by + tx + (int64_t)(bx + r) * m] = tile[tx][r];
}

// The eigenvectors of the upper triangle of T, one warp each: warps 0 .. m-1
// the right ones (columns of Y, unit upper triangular, by back-substitution
// along rows of T: Tt is T^T), warps m .. 2m-1 the left ones (rows of U =
// Y^{-1}, by forward substitution along columns of T; U's conjugate transpose
// is stored).  An entry whose eigenvalue is within small of the vector's own is
// left at zero (the pair's block settles it in the iteration).  Bound by the
// chain of m dot products; the warps of a CTA take vectors a grid apart, so
// that long and short chains mix.
__global__ void k_tri_vectors32(int m, const cf *__restrict__ T, const cf *__restrict__ Tt, cf *__restrict__ Y,
                                cf *__restrict__ Uh, float small)
{
    extern __shared__ cf vec[];
    const int lane = threadIdx.x & 31;
    const int id = blockIdx.x + (int)gridDim.x * (threadIdx.x >> 5);
    if (id >= 2 * m) return;
    cf *y = vec + (size_t)(threadIdx.x >> 5) * m;
    const bool right = id < m;
    const int k = right ? id : id - m;
    const cf lam = T[k + (int64_t)k * m];
    const int cnt = right ? k : m - 1 - k;                 // entries to solve for
    if (lane == 0) y[k] = cmakef(1.f, 0.f);
    __syncwarp();
    for (int st = 0; st < cnt; ++st) {
        const int i = right ? k - 1 - st : k + 1 + st;
        const cf *line = (right ? Tt : T) + (int64_t)i * m; // T[i, :] or T[:, i]
        const int p0 = right ? i + 1 : k, p1 = right ? k : i - 1;
        cf acc = cmakef(0.f, 0.f), ac2 = acc;
        int p = p0 + lane;
        for (; p + 32 <= p1; p += 64) {
            cfma(acc, line[p], y[p]);
            cfma(ac2, line[p + 32], y[p + 32]);
        }
        if (p <= p1) cfma(acc, line[p], y[p]);
        acc = cadd(acc, ac2);
#pragma unroll
        for (int off = 16; off > 0; off >>= 1) {
            acc.x += __shfl_xor_sync(0xffffffffu, acc.x, off);
            acc.y += __shfl_xor_sync(0xffffffffu, acc.y, off);
        }
        if (lane == 0) {
            cf d = line[i];
            d = cmakef(lam.x - d.x, lam.y - d.y);
            y[i] = cabs2(d) < small * small ? cmakef(0.f, 0.f) : cdiv(acc, d);
        }
        __syncwarp();
    }
    cf *out = (right ? Y : Uh) + (int64_t)k * m;
    for (int i = lane; i < m; i += 32) {
        const bool on = right ? i <= k : i >= k;
        const cf v = on ? y[i] : cmakef(0.f, 0.f);
        out[i] = right ? v : cconj(v);
    }
}

// Unit columns: V32 scaled, V its FP64 copy, nv the norms.  Warp per column.
__global__ void k_rf_scale(int m, cf *__restrict__ V32, zd *__restrict__ V, float *__restrict__ nv)
{
    const int j = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
    if (j >= m) return;
    cf *v = V32 + (int64_t)j * m;
    float s = 0.f;
    for (int i = lane; i < m; i += 32) s += cabs2(v[i]);
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) s += __shfl_xor_sync(0xffffffffu, s, off);
    const float nrm = sqrtf(s), inv = 1.f / nrm;
    if (lane == 0) nv[j] = nrm;
    for (int i = lane; i < m; i += 32) {
        const cf x = cmakef(v[i].x * inv, v[i].y * inv);
        v[i] = x;
        V[i + (int64_t)j * m] = zmake((double)x.x, (double)x.y);
    }
}

__global__ void k_rf_scale_rows(int m, cf *__restrict__ L, const float *__restrict__ nv)
{
    const int64_t total = (int64_t)m * m;
    for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < total;
         e += (int64_t)gridDim.x * blockDim.x) {
        const float f = nv[e % m];
        L[e] = cmakef(L[e].x * f, L[e].y * f);
    }
}

// part[b] = block b's share of || E - I ||_F^2 (RF_PART blocks of 256).
__global__ void k_rf_defect(int m, const cf *__restrict__ E, float *__restrict__ part)
{
    __shared__ float red[8];
    const int64_t total = (int64_t)m * m;
    float s = 0.f;
    for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < total;
         e += (int64_t)gridDim.x * blockDim.x) {
        cf v = E[e];
        if (e % m == e / m) v.x -= 1.f;
        s += cabs2(v);
    }
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) s += __shfl_xor_sync(0xffffffffu, s, off);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = s;
    __syncthreads();
    if (threadIdx.x == 0) {
        float r = 0.f;
        for (int w = 0; w < 8; ++w) r += red[w];
        part[blockIdx.x] = r;
    }
}

__global__ void k_rf_lam(int m, const cf *__restrict__ T, zd *__restrict__ lam)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < m) lam[i] = zmake((double)T[i + (int64_t)i * m].x, (double)T[i + (int64_t)i * m].y);
}

// R32 = A' V - (B' V) Lambda', rounded to FP32 (fa: A' = fa A), and its largest
// column against the column's own scale; part and near (the m after it) = -1.
// Warp per column.
__global__ void k_rf_resid(int m, const zd *__restrict__ AV, double fa, const zd *__restrict__ BV,
                           const zd *__restrict__ lam, cf *__restrict__ R32, int *__restrict__ part,
                           RefineStat *__restrict__ st)
{
    const int j = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
    if (j >= m) return;
    const zd l = lam[j];
    float s = 0.f;
    for (int i = lane; i < m; i += 32) {
        const int64_t e = i + (int64_t)j * m;
        const zd r = zsub(zscale(AV[e], fa), zmul(l, BV[e]));
        const cf rf = cmakef((float)r.x, (float)r.y);
        R32[e] = rf;
        s += cabs2(rf);
    }
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) s += __shfl_xor_sync(0xffffffffu, s, off);
    if (lane != 0) return;
    part[j] = part[m + j] = -1;
    const float d = 1.f + hypotf((float)l.x, (float)l.y), q = s / (d * d);
    atomicMax(&st->rm, __float_as_uint(q == q ? q : __int_as_float(0x7f800000)));
}

// G from W (off the diagonal): see the file comment.  tiny: couplings at
// rounding level are converged (only a small G is applied for them: V G in
// FP32 would put FP32 errors back into V for a close pair; near[] names such
// pairs, whose blocks are then settled in FP64).
__global__ void k_rf_g(int m, const cf *__restrict__ W, const zd *__restrict__ lam, float tiny, cf *__restrict__ G,
                       int *__restrict__ part, int *__restrict__ near, RefineStat *__restrict__ st)
{
    const int64_t total = (int64_t)m * m;
    float gm = 0.f, wm = 0.f;
    for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < total;
         e += (int64_t)gridDim.x * blockDim.x) {
        const int i = (int)(e % m), j = (int)(e / m);
        cf g = cmakef(0.f, 0.f);
        if (i != j) {
            const cf w = W[e];
            const zd dd = zsub(lam[j], lam[i]);
            const cf d = cmakef((float)dd.x, (float)dd.y);
            const float w2 = cabs2(w), d2 = cabs2(d);
            wm = fmaxf(wm, w2);
            if (sqrtf(w2) <= tiny) {
                if (w2 <= 1e-16f * d2 && d2 > 1e-30f) {
                    g = cdiv(w, d);
                } else if (w2 <= RF_PAIR * RF_PAIR * d2 && d2 > 1e-30f) {
                    atomicMax(near + i, j);
                    atomicMax(near + j, i);
                    st->tiny = 1;
                }
            } else if (w2 <= RF_PAIR * RF_PAIR * d2 && d2 > 1e-30f) {
                g = cdiv(w, d);
                gm = fmaxf(gm, cabs2(g));
            } else {
                const int pi = atomicCAS(part + i, -1, j), pj = atomicCAS(part + j, -1, i);
                if ((pi != -1 && pi != j) || (pj != -1 && pj != i)) st->bad = 1;   // three or more that close
                st->paired = 1;
            }
        }
        G[e] = g;
    }
    if (gm > 0.f) atomicMax(&st->gm, __float_as_uint(gm));
    if (wm > 0.f) atomicMax(&st->wm, __float_as_uint(wm));
}

__device__ __forceinline__ zd rf_sqrt(zd z)
{
    const double r = hypot(z.x, z.y);
    if (r == 0.0) return zmake(0.0, 0.0);
    if (z.x >= 0.0) {
        const double t = sqrt(0.5 * (r + z.x));
        return zmake(t, z.y / (2.0 * t));
    }
    const double t = sqrt(0.5 * (r - z.x));
    return zmake(fabs(z.y) / (2.0 * t), copysign(t, z.y));
}

// lambda += diag(W); for a pair (i, j) the eigenvalues of its 2 x 2 block of
// Lambda + W and the eigenvectors U = [1 pu_i; pu_j 1] (pd = det U), its
// entries of G cleared.  lam_out is another array than lam.
__global__ void k_rf_lambda(int m, const cf *__restrict__ W, const zd *__restrict__ lam, zd *__restrict__ lam_out,
                            const int *__restrict__ part, const int *__restrict__ near, int *__restrict__ eff,
                            cf *__restrict__ G, zd *__restrict__ pu, zd *__restrict__ pd, RefineStat *__restrict__ st)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= m) return;
    const cf w = W[i + (int64_t)i * m];
    const zd li = zmake(lam[i].x + (double)w.x, lam[i].y + (double)w.y);
    int j = part[i];
    if (j < 0) {
        const int k = near[i];
        if (k >= 0 && near[k] == i && part[k] < 0) j = k;
    }
    eff[i] = j;
    if (j < 0) lam_out[i] = li;
    if (j <= i) return;
    // block [a b; c d]: eigenvectors (1, c / g) and (-b / g, 1), g = h + s,
    // h = (a - d) / 2, s = sqrt(h^2 + b c) on the side of h
    const cf wj = W[j + (int64_t)j * m], wb = W[i + (int64_t)j * m], wc = W[j + (int64_t)i * m];
    const zd lj = zmake(lam[j].x + (double)wj.x, lam[j].y + (double)wj.y);
    const zd b = zmake((double)wb.x, (double)wb.y), c = zmake((double)wc.x, (double)wc.y);
    const zd h = zscale(zsub(li, lj), 0.5);
    zd s = rf_sqrt(zadd(zmul(h, h), zmul(b, c)));
    if (s.x * h.x + s.y * h.y < 0.0) s = zscale(s, -1.0);
    const zd g = zadd(h, s), mid = zscale(zadd(li, lj), 0.5);
    zd u = zmake(0.0, 0.0), v = u;
    if (g.x != 0.0 || g.y != 0.0) {
        u = zscale(zdiv(b, g), -1.0);
        v = zdiv(c, g);
    } else {
        st->bad = 1;
    }
    const zd det = zsub(zmake(1.0, 0.0), zmul(u, v));
    if (!(zabs2(det) > 2.5e-3)) st->bad = 1;   // nearly parallel: not for this iteration
    pu[i] = u;
    pu[j] = v;
    pd[i] = pd[j] = det;
    lam_out[i] = zadd(mid, s);
    lam_out[j] = zsub(mid, s);
    G[i + (int64_t)j * m] = G[j + (int64_t)i * m] = cmakef(0.f, 0.f);
}

// V += VG; then, with pairs, V[:, (i j)] <- V[:, (i j)] U; V32 its FP32 copy.
__global__ void k_rf_update(int m, const cf *__restrict__ VG, const int *__restrict__ part,
                            const zd *__restrict__ pu, int paired, zd *__restrict__ V, cf *__restrict__ V32)
{
    const int64_t total = (int64_t)m * m;
    for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < total;
         e += (int64_t)gridDim.x * blockDim.x) {
        const int r = (int)(e % m), i = (int)(e / m), j = paired ? part[i] : -1;
        if (j >= 0 && j < i) continue;               // (its partner's thread writes both)
        zd v = zmake(V[e].x + (double)VG[e].x, V[e].y + (double)VG[e].y);
        if (j > i) {
            const int64_t f = r + (int64_t)j * m;
            const zd x = zmake(V[f].x + (double)VG[f].x, V[f].y + (double)VG[f].y);
            const zd y = zadd(x, zmul(v, pu[i]));
            v = zadd(v, zmul(x, pu[j]));
            V[f] = y;
            V32[f] = cmakef((float)y.x, (float)y.y);
        }
        V[e] = v;
        V32[e] = cmakef((float)v.x, (float)v.y);
    }
}

// Rows (i j) of L <- U^{-1} L for every pair.
__global__ void k_rf_rows(int m, const int *__restrict__ part, const zd *__restrict__ pu, const zd *__restrict__ pd,
                          cf *__restrict__ L)
{
    const int64_t total = (int64_t)m * m;
    for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < total;
         e += (int64_t)gridDim.x * blockDim.x) {
        const int i = (int)(e % m), j = part[i];
        if (j <= i) continue;
        const int64_t f = e - i + j;
        const zd di = zdiv(zmake(1.0, 0.0), pd[i]);
        const zd xi = zmake((double)L[e].x, (double)L[e].y), xj = zmake((double)L[f].x, (double)L[f].y);
        const zd yi = zmul(di, zsub(xi, zmul(pu[i], xj))), yj = zmul(di, zsub(xj, zmul(pu[j], xi)));
        L[e] = cmakef((float)yi.x, (float)yi.y);
        L[f] = cmakef((float)yj.x, (float)yj.y);
    }
}

// alpha = lambda = fl lambda', beta = 1.
__global__ void k_rf_out(int m, const zd *__restrict__ lam, double fl, zd *__restrict__ alpha, zd *__restrict__ beta)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= m) return;
    alpha[i] = zscale(lam[i], fl);
    beta[i] = zmake(1.0, 0.0);
}

// Column gather: Vout[:, i] = Vin[:, perm[i]] (rows x m, leading dim rows).
__global__ void k_permute_cols(int64_t rows, int m, const int *__restrict__ perm, const zd *__restrict__ Vin,
                               zd *__restrict__ Vout)
{
    const int64_t total = rows * m;
    for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < total;
         e += (int64_t)gridDim.x * blockDim.x) {
        const int64_t i = e % rows;
        const int j = (int)(e / rows);
        Vout[e] = Vin[i + (int64_t)perm[j] * rows];
    }
}

struct RefineCarve {
    cf *X, *T, *Q, *B32, *Y, *Uh, *V32, *L, *W, *G;   // X: [C | B^{-1}], 2 m^2 entries
    zd *AV, *BV, *Bu, *lam, *lam2, *pu, *pd;
    float *lower, *cmax, *nv, *part;
    int *pair, *near, *eff, *fail;
    unsigned *ext;
    float4 *mom;
    RefineStat *st;
    void *schur;
    size_t bytes;
};

RefineCarve refine_carve(void *work, int m)
{
    RefineCarve w;
    const size_t mm = (size_t)m * m;
    char *p = (char *)work;
    size_t off = 0;
    auto take = [&](size_t b) {
        off = (off + 255) & ~(size_t)255;
        char *q = p + off;
        off += b;
        return q;
    };
    w.X = (cf *)take(2 * mm * sizeof(cf));
    cf **c32[] = {&w.T, &w.Q, &w.B32, &w.Y, &w.Uh, &w.V32, &w.L, &w.W, &w.G};
    for (cf **c : c32) *c = (cf *)take(mm * sizeof(cf));
    w.AV = (zd *)take(mm * sizeof(zd));
    w.BV = (zd *)take(mm * sizeof(zd));
    w.Bu = (zd *)take(mm * sizeof(zd));
    zd **c64[] = {&w.lam, &w.lam2, &w.pu, &w.pd};
    for (zd **c : c64) *c = (zd *)take((size_t)m * sizeof(zd));
    w.lower = (float *)take(2 * (size_t)m * sizeof(float));
    w.cmax = w.lower + m;
    w.nv = (float *)take((size_t)m * sizeof(float));
    w.part = (float *)take(RF_PART * sizeof(float));
    w.pair = (int *)take(3 * (size_t)m * sizeof(int));
    w.near = w.pair + m;
    w.eff = w.near + m;
    w.fail = (int *)take(sizeof(int));
    w.ext = (unsigned *)take(8);
    w.mom = (float4 *)take(RF_MOM * sizeof(float4));
    w.st = (RefineStat *)take(sizeof(RefineStat));
    w.schur = take(schur32_work_bytes(m));
    w.bytes = off;
    return w;
}

unsigned grid_for(size_t count)
{
    const unsigned g = cdiv(count, 256);
    return g > 4096 ? 4096 : g;
}

}  // namespace

size_t zeig_refined_large_work_bytes(int m) { return refine_carve(nullptr, m).bytes + 256; }

int shift_pencil(cudaStream_t s, int m, zd *A, const zd *Bt, zd sigma)
{
    k_shift_pencil<<<grid_for((size_t)m * m), 256, 0, s>>>(m, A, Bt, sigma);
    FEAST_LAUNCH_CHECK();
    return FEAST_OK;
}

int shift_values(cudaStream_t s, int m, zd *alpha, const zd *beta, zd sigma)
{
    k_shift_values<<<cdiv(m, 128), 128, 0, s>>>(m, alpha, beta, sigma);
    FEAST_LAUNCH_CHECK();
    return FEAST_OK;
}

int permute_cols(cudaStream_t s, int64_t rows, int m, const int *perm, const zd *Vin, zd *Vout)
{
    k_permute_cols<<<grid_for((size_t)rows * m), 256, 0, s>>>(rows, m, perm, Vin, Vout);
    FEAST_LAUNCH_CHECK();
    return FEAST_OK;
}


static int refined_attempt(cudaStream_t s, int m, const zd *A, const zd *Bt, zd *alpha, zd *beta, zd *V, void *work,
                           const RefineParams &prm, RefineResult *res, int *timeout, int *stats, GemmTimer *gt,
                           const OzScratch *oz)
{
    *res = RefineResult{};
    if (m < 3) return FEAST_OK;
    const RefineCarve w = refine_carve((void *)(((uintptr_t)work + 255) & ~(uintptr_t)255), m);
    const size_t mm = (size_t)m * m;
    const zd one = zmake(1.0, 0.0), zero = zmake(0.0, 0.0);
    const cf fone = cmakef(1.f, 0.f), fzero = cmakef(0.f, 0.f), fmone = cmakef(-1.f, 0.f);
    int e;
    auto mul32 = [&](int conj_a, int64_t M, int64_t N, int64_t K, cf al, const cf *Am, int64_t lda, const cf *Bm,
                     int64_t ldb, cf be, cf *Cm, int64_t ldc) {
        return gemm_batched<cf>(s, conj_a, M, N, K, al, Am, lda, 0, Bm, ldb, 0, be, Cm, ldc, 0, 1);
    };
    // C = B'^{-1} A' and B'^{-1}, FP32
    FEAST_CUDA_TRY(cudaMemsetAsync(w.ext, 0, 8, s));
    k_rf_extent<<<grid_for(mm), 256, 0, s>>>(m, A, Bt, w.ext);
    FEAST_LAUNCH_CHECK();
    const unsigned gc = prm.find && grid_for(mm) > RF_MOM ? RF_MOM : grid_for(mm);
    k_rf_cast<<<gc, 256, 0, s>>>(m, A, Bt, w.X, w.B32, w.Bu, w.ext, prm.find ? w.mom : nullptr);
    FEAST_LAUNCH_CHECK();
    if ((e = trsm_upper_batched<cf>(s, m, 2 * m, 1, w.B32, m, 0, w.X, m, 0))) return e;
    cf *C = w.X, *Bi = w.X + mm;
    k_col_stats32<<<cdiv((size_t)m * 32, 256), 256, 0, s>>>(m, C, w.lower, w.cmax);
    FEAST_LAUNCH_CHECK();
    unsigned ext[2] = {0, 0};
    float4 mom[RF_MOM];
    if (prm.find) FEAST_CUDA_TRY(cudaMemcpyAsync(mom, w.mom, gc * sizeof(float4), cudaMemcpyDeviceToHost, s));
    float *h = (float *)malloc(sizeof(float) * 2 * (size_t)m);
    if (!h) return FEAST_ENOMEM;
    if (cudaMemcpyAsync(h, w.lower, sizeof(float) * 2 * (size_t)m, cudaMemcpyDeviceToHost, s) != cudaSuccess ||
        cudaMemcpyAsync(ext, w.ext, 8, cudaMemcpyDeviceToHost, s) != cudaSuccess ||
        cudaStreamSynchronize(s) != cudaSuccess) {
        free(h);
        return FEAST_ECUDA;
    }
    float cn = 0.f;
    for (int j = 0; j < m; ++j) cn = h[m + j] > cn ? h[m + j] : cn;
    const int xa = (int)(ext[0] >> 20) - 1022, xb = (int)(ext[1] >> 20) - 1022;
    const float tau = prm.tau > 0.f ? prm.tau : RF_TAU;
    int k = 0;
    while (k < m && h[k] <= tau * cn) ++k;
    res->k = k;
    while (res->k_tight < m && h[res->k_tight] <= RF_TIGHT * cn) ++res->k_tight;
    free(h);
    // (zero, non-finite or far out of range; B singular shows as a non-finite C)
    if (!rf_exp_ok(ext[0]) || !rf_exp_ok(ext[1]) || !(cn > 0.f && cn < 1e14f)) return FEAST_OK;
    const double fa = ldexp(1.0, -xa), fl = ldexp(1.0, xa - xb);
    if (prm.find) {
        double x = 0.0, y = 0.0, aa = 0.0, bb = 0.0;
        for (unsigned i = 0; i < gc; ++i) {
            x += mom[i].x;
            y += mom[i].y;
            aa += mom[i].z;
            bb += mom[i].w;
        }
        if (aa * bb - (x * x + y * y) <= RF_NARROW * RF_NARROW * aa * bb) {
            res->narrow = 1;
            res->sigma = zmake(x / bb * fl, y / bb * fl);
            return FEAST_OK;
        }
    }
    if (k > m - 8) k = m - 8;
    if (!prm.warm || k < m / 4) k = 0;               // too little has converged: the whole matrix
    const int mb = m - k;
    res->tail = mb;
    // Schur form of the trailing block: T = [C11 C12 Z; 0 T22], Z in w.Q (mb x mb)
    FEAST_CUDA_TRY(cudaMemcpy2DAsync(w.G, sizeof(cf) * mb, C + k + (int64_t)k * m, sizeof(cf) * m, sizeof(cf) * mb, mb,
                                     cudaMemcpyDeviceToDevice, s));
    FEAST_CUDA_TRY(cudaMemsetAsync(w.fail, 0, sizeof(int), s));
    if ((e = schur32(s, mb, w.G, w.Q, cn, w.schur, w.fail, timeout, stats))) return e;
    if (k > 0) {
        FEAST_CUDA_TRY(cudaMemcpyAsync(w.T, C, sizeof(cf) * (size_t)m * k, cudaMemcpyDeviceToDevice, s));
        if ((e = mul32(0, k, mb, mb, fone, C + (int64_t)k * m, m, w.Q, mb, fzero, w.T + (int64_t)k * m, m))) return e;
    }
    FEAST_CUDA_TRY(cudaMemcpy2DAsync(w.T + k + (int64_t)k * m, sizeof(cf) * m, w.G, sizeof(cf) * mb, sizeof(cf) * mb, mb,
                                     cudaMemcpyDeviceToDevice, s));
    // eigenvectors of T: Y, and U = Y^{-1} (its conjugate transpose)
    k_transpose32<<<dim3(cdiv(m, 32), cdiv(m, 32)), 256, 0, s>>>(m, w.T, w.W);
    FEAST_LAUNCH_CHECK();
    {
        int dev = 0, sms = 0;
        FEAST_CUDA_TRY(cudaGetDevice(&dev));
        FEAST_CUDA_TRY(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
        int wpc = (2 * m + sms - 1) / sms;           // warps per CTA, one CTA per SM
        const int most = (int)(200 * 1024 / (sizeof(cf) * (size_t)m));
        if (wpc > 16) wpc = 16;
        if (wpc > most) wpc = most;
        if (wpc < 1) wpc = 1;
        const size_t sm = sizeof(cf) * (size_t)m * wpc;
        FEAST_CUDA_TRY(ensure_dyn_smem(k_tri_vectors32, sm));
        k_tri_vectors32<<<cdiv((size_t)2 * m, wpc), 32 * wpc, sm, s>>>(m, w.T, w.W, w.Y, w.Uh, 1e-5f * cn);
        FEAST_LAUNCH_CHECK();
    }
    k_rf_lam<<<cdiv(m, 128), 128, 0, s>>>(m, w.T, w.lam);
    FEAST_LAUNCH_CHECK();
    // V = diag(I, Z) Y;  L^H = U diag(I, Z)^H B^{-1}
    if (k > 0) {
        FEAST_CUDA_TRY(cudaMemcpy2DAsync(w.V32, sizeof(cf) * m, w.Y, sizeof(cf) * m, sizeof(cf) * k, m,
                                         cudaMemcpyDeviceToDevice, s));
        FEAST_CUDA_TRY(cudaMemcpy2DAsync(w.W, sizeof(cf) * m, Bi, sizeof(cf) * m, sizeof(cf) * k, m,
                                         cudaMemcpyDeviceToDevice, s));
    }
    if ((e = mul32(0, mb, m, mb, fone, w.Q, mb, w.Y + k, m, fzero, w.V32 + k, m))) return e;
    if ((e = mul32(1, mb, m, mb, fone, w.Q, mb, Bi + k, m, fzero, w.W + k, m))) return e;
    if ((e = mul32(1, m, m, m, fone, w.Uh, m, w.W, m, fzero, w.L, m))) return e;
    k_rf_scale<<<cdiv((size_t)m * 32, 256), 256, 0, s>>>(m, w.V32, V, w.nv);
    FEAST_LAUNCH_CHECK();
    k_rf_scale_rows<<<grid_for(mm), 256, 0, s>>>(m, w.L, w.nv);
    FEAST_LAUNCH_CHECK();
    // delta = || I - L^H B V ||_F
    if ((e = mul32(0, m, m, m, fone, w.B32, m, w.V32, m, fzero, w.W, m))) return e;
    if ((e = mul32(0, m, m, m, fone, w.L, m, w.W, m, fzero, w.G, m))) return e;
    k_rf_defect<<<RF_PART, 256, 0, s>>>(m, w.G, w.part);
    FEAST_LAUNCH_CHECK();
    float hp[RF_PART];
    int qfail = 0;
    FEAST_CUDA_TRY(cudaMemcpyAsync(hp, w.part, sizeof(hp), cudaMemcpyDeviceToHost, s));
    FEAST_CUDA_TRY(cudaMemcpyAsync(&qfail, w.fail, sizeof(int), cudaMemcpyDeviceToHost, s));
    FEAST_CUDA_TRY(cudaStreamSynchronize(s));
    double dl = 0.0;
    for (float x : hp) dl += (double)x;
    dl = sqrt(dl);
    if (qfail || !(dl < 0.1)) return FEAST_OK;
    double gprev = 0.0, wprev = 0.0;
    bool last64 = false, only64 = false, ever = false;
    zd *lam = w.lam, *lam2 = w.lam2;
    for (int step = 0; step < RF_STEPS; ++step) {
        // the digit-sliced products while what they leave (about 1e-13 of
        // max|C| over a gap) is not yet what limits the result
        const bool use_oz = oz && !only64 &&
                            (prm.target > 1e-10 || (!last64 && (step == 0 || gprev == 0.0 || gprev > 1e-6)));
        last64 = !use_oz;
        const bool timed = gt && !use_oz && gt->used + 2 <= GemmTimer::kMax;
        if (timed) FEAST_CUDA_TRY(cudaEventRecord(gt->ev[gt->used++], s));
        if (use_oz) {
            if ((e = oz_prepare_cols(s, m, m, V, m, oz->cols))) return e;
            if ((e = oz_prepare_rows(s, m, m, A, m, oz->rows))) return e;
            if ((e = oz_gemm(s, m, m, m, oz->rows, oz->cols, one, nullptr, 0, zero, w.AV, m, oz->err))) return e;
            if ((e = oz_prepare_rows(s, m, m, w.Bu, m, oz->rows))) return e;
            if ((e = oz_gemm(s, m, m, m, oz->rows, oz->cols, one, nullptr, 0, zero, w.BV, m, oz->err))) return e;
        } else {
            if ((e = zgemm_batched(s, 0, m, m, m, one, A, m, 0, V, m, 0, zero, w.AV, m, 0, 1))) return e;
            if ((e = zgemm_batched(s, 0, m, m, m, one, w.Bu, m, 0, V, m, 0, zero, w.BV, m, 0, 1, 1))) return e;
        }
        if (timed) {
            FEAST_CUDA_TRY(cudaEventRecord(gt->ev[gt->used++], s));
            gt->flops += 12.0 * (double)m * m * m;
        }
        FEAST_CUDA_TRY(cudaMemsetAsync(w.st, 0, sizeof(RefineStat), s));
        k_rf_resid<<<cdiv((size_t)m * 32, 256), 256, 0, s>>>(m, w.AV, fa, w.BV, lam, w.G, w.pair, w.st);
        FEAST_LAUNCH_CHECK();
        if ((e = mul32(0, m, m, m, fone, w.L, m, w.G, m, fzero, w.W, m))) return e;
        k_rf_g<<<grid_for(mm), 256, 0, s>>>(m, w.W, lam, (use_oz ? 1e-12f : 1e-14f) * cn, w.G, w.pair, w.near, w.st);
        FEAST_LAUNCH_CHECK();
        k_rf_lambda<<<cdiv(m, 128), 128, 0, s>>>(m, w.W, lam, lam2, w.pair, w.near, w.eff, w.G, w.pu, w.pd, w.st);
        FEAST_LAUNCH_CHECK();
        if ((e = mul32(0, m, m, m, fone, w.V32, m, w.G, m, fzero, w.Y, m))) return e;
        RefineStat hs;
        FEAST_CUDA_TRY(cudaMemcpyAsync(&hs, w.st, sizeof(hs), cudaMemcpyDeviceToHost, s));
        FEAST_CUDA_TRY(cudaStreamSynchronize(s));
        if (hs.bad) return FEAST_OK;
        float g2, w2, r2;
        memcpy(&g2, &hs.gm, sizeof(float));
        memcpy(&w2, &hs.wm, sizeof(float));
        memcpy(&r2, &hs.rm, sizeof(float));
        const double gm = sqrt((double)g2), wm = sqrt((double)w2);
        k_rf_update<<<grid_for(mm), 256, 0, s>>>(m, w.Y, w.eff, w.pu, hs.paired || hs.tiny, V, w.V32);
        FEAST_LAUNCH_CHECK();
        zd *t = lam;
        lam = lam2;
        lam2 = t;
        // what the step leaves: by the bound on delta, or by the contraction
        // seen (|G| over the step before's, at least delta); a pair's block is
        // followed by another step.  |G| that no longer falls (nor |W|: a close
        // pair's G can stand still while the others still converge) is either
        // the residual's rounding or a slow contraction (delta is let in up to
        // 0.1), and the residual that the step began with tells them apart: the
        // pairs are accepted when its backward error is that of an FP64 QZ
        const double ratio = gprev > 0.0 ? gm / gprev : 1e300;
        const double left = gm * fmin(8.0 * fmax(gm, ratio), (double)m * gm + dl);
        const bool still = gm <= 1e-8 && step > 0 && ratio > 0.1 && ratio < 1e200 && wm > 0.1 * wprev;
        const bool exact = still && sqrt((double)r2) <= RF_BERR * (double)m;
        only64 = only64 || (still && !exact);
        res->steps = step + 1;
        res->resid = exact ? gm : left;
        if (!hs.paired && (exact || left <= (ever ? 0.25 : 1.0) * prm.target) &&
            (!oz || prm.target > 1e-10 || last64)) {
            if ((e = normalise_cols(s, m, V))) return e;
            k_rf_out<<<cdiv(m, 128), 128, 0, s>>>(m, lam, fl, alpha, beta);
            FEAST_LAUNCH_CHECK();
            res->accepted = 1;
            return FEAST_OK;
        }
        if (hs.paired || gm > 1e-6) {
            // L^H to (B V)^{-1} of the new V, up to |G|^2
            FEAST_CUDA_TRY(cudaMemcpyAsync(w.Y, w.L, sizeof(cf) * mm, cudaMemcpyDeviceToDevice, s));
            if ((e = mul32(0, m, m, m, fmone, w.G, m, w.Y, m, fone, w.L, m))) return e;
            dl += (double)m * gm * gm;
        } else {
            dl += (double)m * gm;
        }
        if (hs.paired || hs.tiny) {
            k_rf_rows<<<grid_for(mm), 256, 0, s>>>(m, w.eff, w.pu, w.pd, w.L);
            FEAST_LAUNCH_CHECK();
        }
        // (after a pair's block neither size says how the iteration contracts)
        gprev = hs.paired ? 0.0 : gm > 0.0 ? gm : 1e-30;
        wprev = wm;
        ever = ever || hs.paired;
    }
    return FEAST_OK;
}

int zeig_refined_large(cudaStream_t s, int m, const zd *A, const zd *Bt, zd *alpha, zd *beta, zd *V, void *work,
                       const RefineParams &prm, RefineResult *res, int *timeout, int *stats, GemmTimer *gt,
                       const OzScratch *oz)
{
    int e = refined_attempt(s, m, A, Bt, alpha, beta, V, work, prm, res, timeout, stats, gt, oz);
    if (e || res->accepted || res->narrow || res->tail == m || !prm.warm) return e;
    const int k = res->k;
    RefineParams next = prm;
    if (res->k_tight >= m / 4 && res->k_tight < m - res->tail) {   // (m - tail: the columns that it started from)
        next.tau = RF_TIGHT;
        e = refined_attempt(s, m, A, Bt, alpha, beta, V, work, next, res, timeout, stats, gt, oz);
        res->k = k;
        if (e || res->accepted) return e;
    }
    next.warm = 0;   // the warm start does not contract: the whole matrix
    e = refined_attempt(s, m, A, Bt, alpha, beta, V, work, next, res, timeout, stats, gt, oz);
    res->k = k;
    return e;
}

}  // namespace feast
