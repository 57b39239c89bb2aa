// Schur form of a complex64 matrix in plain FP32: schur32.  It starts the
// Newton iteration of k_warm.cu, whose residual alone is FP64.
//
//   up to SC_MAX rows: the Hessenberg matrix fits the shared memory of one
//     CTA (packed by rows), whose warp 0 holds the QR iteration's chain of
//     rotations in registers (chase32.cuh) while the other warps apply each
//     chunk of 32 to the far columns and the rows above; the rotations are
//     logged, and k_apply_rot32 turns the log into Schur vectors, a thread
//     per row;
//   beyond: the cooperative multishift QR of k_zeig.cu built in FP32.
#define FEAST_QR_FP32 1
#include "k_zeig.cu"

#include "chase32.cuh"

namespace feast {
namespace {

constexpr int SC_MAX = 232;      // packed_elems(232) complex64 entries: 220 KB
constexpr int SC_T = 512;
constexpr int SC_LOG = 2;        // rotation log: SC_LOG m^2 entries (a run takes ~1.4 m^2)

// status[0]: 0 done, 1 iteration budget spent, 2 log full; status[1]:
// rotations logged; status[2]: sweeps.  H (m x m, column-major, ld m; Hessenberg) becomes
// the triangular factor when status[0] = 0 and keeps its value otherwise.
// A log entry is (c, Re s, Im s, k).
__global__ void __launch_bounds__(SC_T, 1) k_schur_cta(int m, cf *__restrict__ H, float4 *__restrict__ log,
                                                       int max_log, int *__restrict__ status)
{
    extern __shared__ cf sc[];
    __shared__ RotF rot[CHASE_N];
    __shared__ float red[SC_T / 32];
    __shared__ int ctl[2];
    __shared__ cf s_sigma;
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    const RowsPacked R{sc, m};
    float mx = 0.f;
    for (int c = warp; c < m; c += SC_T / 32)
        for (int r = lane; r < m && r <= c + 2; r += 32) {
            const cf v = (r <= c + 1) ? H[r + (int64_t)c * m] : cmakef(0.f, 0.f);
            R.row(r)[c] = v;
            mx = fmaxf(mx, fmaxf(fabsf(v.x), fabsf(v.y)));
        }
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, off));
    if (lane == 0) red[warp] = mx;
    __syncthreads();
    mx = red[0];
    for (int w = 1; w < SC_T / 32; ++w) mx = fmaxf(mx, red[w]);
    // a subdiagonal entry is negligible at FP32 rounding of its neighbours or of the matrix
    const float tol_rel = 2.4e-7f, tol_abs = 6e-8f * mx;
    int hi = m - 1, it = 0, tot = 0, nr = 0, st = 0;
    for (;;) {
        if (warp == 0) {
            int lo = 0;
            while (hi > 0) {
                lo = 0;
                for (int base = hi; base >= 1 && lo == 0; base -= 32) {
                    const int p = base - lane;
                    bool neg = false;
                    if (p >= 1) {
                        const cf *rp = R.row(p), *rq = R.row(p - 1);
                        const float sub = abs32(rp[p - 1]), loc = abs32(rq[p - 1]) + abs32(rp[p]);
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
                const cf *rh = R.row(hi), *rg = R.row(hi - 1);
                const cf h11 = rh[hi], h10 = rh[hi - 1];
                cf sigma = shift32(rg[hi - 1], rg[hi], h10, h11);
                if (it % 11 == 10) {
                    const float a = abs32(h10);
                    sigma = cmakef(h11.x + a, h11.y + 0.5f * a);
                }
                if (lane == 0) s_sigma = sigma;
            }
            if (lane == 0) {
                ctl[0] = lo;
                ctl[1] = hi;
            }
        }
        __syncthreads();
        const int lo = ctl[0], h = ctl[1];
        if (h <= 0) {
            st = h == 0 ? 0 : 1;
            break;
        }
        if (nr + (h - lo) > max_log) {
            st = 2;
            break;
        }
        for (int k0 = lo; k0 < h; k0 += CHASE_N) {
            const int k1 = (k0 + CHASE_N < h) ? k0 + CHASE_N : h;
            if (warp == 0) chase_left(R, m, lo, h, k0, k1, s_sigma, rot);
            __syncthreads();
            if (t < 256) {
                if (t < k1) chase_right(R.row(t), k0, t > k0 ? t : k0, k1, rot);
            } else {
                const int c = k0 + CHASE_N + 1 + (t - 256);
                if (c < m) far_left(R, c, k0, k1, rot);
                if (t >= SC_T - CHASE_N && t - (SC_T - CHASE_N) < k1 - k0) {
                    const int i = t - (SC_T - CHASE_N);
                    const RotF g = rot[i];
                    log[nr + i] = make_float4(g.c, g.s.x, g.s.y, __int_as_float(k0 + i));
                }
            }
            nr += k1 - k0;
            __syncthreads();
        }
    }
    if (t == 0) {
        status[0] = st;
        status[1] = nr;
        status[2] = tot;
    }
    if (st) return;
    for (int c = warp; c < m; c += SC_T / 32)
        for (int r = lane; r < m; r += 32) H[r + (int64_t)c * m] = (r <= c) ? R.row(r)[c] : cmakef(0.f, 0.f);
}

// Q <- Q G_1^H G_2^H ... (the logged rotations, in order): a thread per row of
// Q (m x m column-major), AZ rows per CTA in shared memory; the two entries
// that a rotation touches are carried in registers along a sweep.  Nothing
// when the Schur form was not reached.
constexpr int AZ = 32, AZ_LOG = 256;
__global__ void __launch_bounds__(AZ) k_apply_rot32(int m, cf *__restrict__ Q, const float4 *__restrict__ log,
                                                   const int *__restrict__ status)
{
    extern __shared__ cf zsm[];                  // AZ rows, odd leading dimension
    __shared__ float4 chunk[AZ_LOG];
    if (status[0] != 0) return;
    const int t = threadIdx.x, ld = m | 1;
    const int r0 = blockIdx.x * AZ, r = r0 + t;
    const int nr = status[1];
    cf *zr = zsm + (size_t)t * ld;
    for (int c = 0; c < m; ++c)
        if (r < m) zr[c] = Q[r + (int64_t)c * m];
    int cur = -2;
    cf a = cmakef(0.f, 0.f), b = a;
    for (int e0 = 0; e0 < nr; e0 += AZ_LOG) {
        const int cnt = (nr - e0) < AZ_LOG ? (nr - e0) : AZ_LOG;
        __syncwarp();
        for (int e = t; e < cnt; e += AZ) chunk[e] = log[e0 + e];
        __syncwarp();
        if (r >= m) continue;
        for (int e = 0; e < cnt; ++e) {
            const float4 L = chunk[e];
            const int k = __float_as_int(L.w);
            if (k == cur + 1) {
                zr[cur] = a;
                a = b;
                b = zr[k + 1];
            } else {
                if (cur >= 0) {
                    zr[cur] = a;
                    zr[cur + 1] = b;
                }
                a = zr[k];
                b = zr[k + 1];
            }
            cur = k;
            RotF g;
            g.c = L.x;
            g.s = cmakef(L.y, -L.z);
            rot32_pair(g, a, b);
        }
    }
    if (r >= m) return;
    if (cur >= 0) {
        zr[cur] = a;
        zr[cur + 1] = b;
    }
    for (int c = 0; c < m; ++c) Q[r + (int64_t)c * m] = zr[c];
}

__global__ void k_schur_report(const int *__restrict__ status, int *fail, int *stats)
{
    if (status[0]) atomicAdd(fail, 1);
    if (stats) stats[0] += status[2];
}

__global__ void k_c2ds(int64_t count, const cf *__restrict__ x, float4 *__restrict__ y)
{
    for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < count; e += (int64_t)gridDim.x * blockDim.x)
        y[e] = make_float4(x[e].x, 0.f, x[e].y, 0.f);
}
__global__ void k_ds2c(int64_t count, const float4 *__restrict__ x, cf *__restrict__ y)
{
    for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < count; e += (int64_t)gridDim.x * blockDim.x)
        y[e] = make_float2(x[e].x, x[e].z);
}

unsigned grid_s(size_t count)
{
    const unsigned g = cdiv(count, 256);
    return g > 4096 ? 4096 : g;
}

}  // namespace

size_t schur32_work_bytes(int m)
{
    // barrier words, status, the window's transfer buffers, then the rotation
    // log or the multishift QR's copies of H and Q (32 m^2 bytes either way;
    // monotone in m, so a trailing block fits its matrix's work)
    return 1024 + sizeof(RotDS) * NSH * CH + sizeof(float2) * NSH + sizeof(float4) * NW * NW +
           2 * sizeof(float4) * (size_t)m * m;
}

int schur32(cudaStream_t s, int m, cf *C, cf *Q, float cmax, void *work, int *fail, int *timeout, int *stats)
{
    if (m <= 0) return FEAST_OK;
    char *p = (char *)work;
    unsigned *hbar = (unsigned *)p, *bar = hbar + 16;
    int *ctl = (int *)(hbar + 32), *sst = ctl + 4;
    p += 512;
    RotDS *rots = (RotDS *)p;
    float2 *shifts = (float2 *)(rots + NSH * CH);
    float4 *vwin = (float4 *)(((uintptr_t)(shifts + NSH) + 15) & ~(uintptr_t)15);
    float4 *big = (float4 *)(((uintptr_t)(vwin + NW * NW) + 255) & ~(uintptr_t)255);
    const size_t mm = (size_t)m * m;
    k_eye_c<<<grid_s(mm), 256, 0, s>>>(m, Q);
    FEAST_LAUNCH_CHECK();
    int dev = 0, sms = 0, per = 0;
    FEAST_CUDA_TRY(cudaGetDevice(&dev));
    FEAST_CUDA_TRY(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
    FEAST_CUDA_TRY(cudaMemsetAsync(hbar, 0, 512, s));
    int mi = m, ldm = m;
    if (m >= 3) {
        const size_t hsm = sizeof(cf) * (size_t)m;
        FEAST_CUDA_TRY(ensure_dyn_smem(k_hess_grid<cf>, hsm));
        FEAST_CUDA_TRY(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, k_hess_grid<cf>, HG_T, hsm));
        if (per < 1) return FEAST_ECUDA;
        const int need = (2 * m + HG_R - 1) / HG_R;     // right-update slabs
        GridSync hg{hbar, hbar + 1, timeout, TO_HESS};
        void *hargs[] = {&mi, &C, &Q, &ldm, &hg};
        FEAST_CUDA_TRY(cudaLaunchCooperativeKernel((void *)k_hess_grid<cf>, dim3(sms < need ? sms : need), dim3(HG_T),
                                                   hargs, hsm, s));
        FEAST_LAUNCH_CHECK();
    }
    if (m <= SC_MAX) {
        FEAST_CUDA_TRY(allow_dyn_smem(k_schur_cta));
        k_schur_cta<<<1, SC_T, sizeof(cf) * (size_t)packed_elems(m), s>>>(m, C, big, SC_LOG * (int)mm, sst);
        FEAST_LAUNCH_CHECK();
        FEAST_CUDA_TRY(ensure_dyn_smem(k_apply_rot32, sizeof(cf) * AZ * (size_t)(m | 1)));
        k_apply_rot32<<<cdiv(m, AZ), AZ, sizeof(cf) * AZ * (size_t)(m | 1), s>>>(m, Q, big, sst);
        FEAST_LAUNCH_CHECK();
        // (budget or log spent: reported as a failed iteration)
        k_schur_report<<<1, 1, 0, s>>>(sst, fail, stats);
        FEAST_LAUNCH_CHECK();
        return FEAST_OK;
    }
    const size_t dyn = sizeof(AedShared);
    FEAST_CUDA_TRY(allow_dyn_smem(k_hqr));
    FEAST_CUDA_TRY(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, k_hqr, QT, dyn));
    if (per < 1) return FEAST_ECUDA;
    // at most one CTA per SM; the far-part passes have ~3 m independent lines
    // and a sweep at most NSH bulges, so a smaller problem takes a
    // proportionally small grid (and leaves the rest of the GPU to others)
    int grid = m / 8;
    if (grid < NSH) grid = NSH;
    if (grid > sms) grid = sms;
    float4 *Hds = big, *Qds = big + mm;
    k_c2ds<<<grid_s(mm), 256, 0, s>>>((int64_t)mm, C, Hds);
    FEAST_LAUNCH_CHECK();
    k_c2ds<<<grid_s(mm), 256, 0, s>>>((int64_t)mm, Q, Qds);
    FEAST_LAUNCH_CHECK();
    float tol_rel = 1e-6f, tol_abs = 1e-6f * cmax;   // a few FP32 units
    GridSync gs{bar, bar + 1, timeout, TO_HQR};
    void *args[] = {&mi, &Hds, &Qds, &ldm, &rots, &shifts, &vwin, &ctl, &gs, &fail, &tol_rel, &tol_abs, &stats};
    FEAST_CUDA_TRY(cudaLaunchCooperativeKernel((void *)k_hqr, dim3(grid), dim3(QT), args, dyn, s));
    FEAST_LAUNCH_CHECK();
    k_ds2c<<<grid_s(mm), 256, 0, s>>>((int64_t)mm, Hds, C);
    FEAST_LAUNCH_CHECK();
    k_ds2c<<<grid_s(mm), 256, 0, s>>>((int64_t)mm, Qds, Q);
    FEAST_LAUNCH_CHECK();
    return FEAST_OK;
}

}  // namespace feast
