// Schur form of a complex64 matrix in plain FP32: schur32.  It starts the
// Newton iteration of k_warm.cu, whose residual alone is FP64.
//
//   up to SC_MAX rows: the Hessenberg matrix fits the shared memory of one
//     CTA (packed by rows), whose warp 0 holds the QR iteration's chain of
//     rotations in registers (chase32.cuh) while the other warps apply each
//     chunk of 32 to the far columns and the rows above; the rotations are
//     logged, and k_apply_rot32 turns the log into Schur vectors, a thread
//     per row;
//   beyond: the cooperative multishift QR of k_zeig.cu built in FP32, which
//     finishes active blocks below MS_MIN rows the same way.
#define FEAST_QR_FP32 1
#include "k_zeig.cu"

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
    __shared__ float red[SC_T / 32];
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
    int nr = 0, tot = 0;
    const int st = schur_cta_core<SC_T>(R, m, 2.4e-7f, 6e-8f * mx, log, max_log, &nr, &tot);
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
// Q (m x m column-major), AZ rows per CTA.  Nothing when the Schur form was
// not reached.
constexpr int AZ = 32;
__global__ void __launch_bounds__(AZ) k_apply_rot32(int m, cf *__restrict__ Q, const float4 *__restrict__ log,
                                                   const int *__restrict__ status)
{
    extern __shared__ cf zsm[];                  // AZ rows, odd leading dimension
    __shared__ float4 chunk[256];
    if (status[0] != 0) return;
    const int r = blockIdx.x * AZ + threadIdx.x;
    apply_log(m, r < m ? Q + r : nullptr, m, false, log, status[1], zsm + (size_t)threadIdx.x * (m | 1), chunk);
}

__global__ void k_schur_report(const int *__restrict__ status, int *fail, int *stats)
{
    if (status[0]) atomicAdd(fail, 1);
    if (stats) stats[0] += status[2];
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
    // log (monotone in m, so a trailing block fits its matrix's work)
    const size_t ml = (size_t)(m < SC_MAX ? m : SC_MAX);
    return 1024 + sizeof(RotDS) * NSH * CH + sizeof(float2) * NSH + sizeof(cf) * NW * NW +
           SC_LOG * sizeof(float4) * ml * ml;
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
    cf *vwin = (cf *)(((uintptr_t)(shifts + NSH) + 15) & ~(uintptr_t)15);
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
    // the window's arrays, or a block that is finished in one CTA
    const size_t fin = sizeof(cf) * (size_t)packed_elems(MS_MIN - 1);
    const size_t dyn = sizeof(AedShared) > fin ? sizeof(AedShared) : fin;
    FEAST_CUDA_TRY(allow_dyn_smem(k_hqr));
    FEAST_CUDA_TRY(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, k_hqr, QT, dyn));
    if (per < 1) return FEAST_ECUDA;
    // at most one CTA per SM; the far-part passes have ~3 m independent lines
    // and a sweep at most NSH bulges, so a smaller problem takes a
    // proportionally small grid (and leaves the rest of the GPU to others)
    int grid = m / 8;
    if (grid < NSH) grid = NSH;
    if (grid > sms) grid = sms;
    float tol_rel = 1e-6f, tol_abs = 1e-6f * cmax;   // a few FP32 units
    GridSync gs{bar, bar + 1, timeout, TO_HQR};
    int max_log = SC_LOG * MS_MIN * MS_MIN;
    void *args[] = {&mi, &C,    &Q,       &ldm,     &rots,  &shifts, &vwin,    &ctl,
                    &gs, &fail, &tol_rel, &tol_abs, &stats, &big,    &max_log};
    FEAST_CUDA_TRY(cudaLaunchCooperativeKernel((void *)k_hqr, dim3(grid), dim3(QT), args, dyn, s));
    FEAST_LAUNCH_CHECK();
    return FEAST_OK;
}

}  // namespace feast
