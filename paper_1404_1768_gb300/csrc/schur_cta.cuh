// The FP32 QR iteration of an upper Hessenberg matrix held in the shared memory
// of one CTA (chase32.cuh), and the application of its rotations elsewhere.
#pragma once

#include "chase32.cuh"

namespace feast {
namespace {

// Triangular form of the m x m Hessenberg matrix R (packed, shared memory; m <=
// 232) by the whole CTA of NT >= 512 threads, single-shift sweeps: warp 0
// scans for deflation (a subdiagonal entry below tol_rel of its neighbours or
// below tol_abs) and holds the chain of rotations, 32 at a time; then threads
// 0 .. 255 apply them to the rows passed and the others to the columns beyond.
// Every rotation is logged as (c, Re s, Im s, k).  Returns 0 done, 1 iteration
// budget spent, 2 log full; *nr rotations, *sweeps sweeps.
template <int NT>
__device__ int schur_cta_core(RowsPacked R, int m, float tol_rel, float tol_abs, float4 *log, int max_log, int *nr,
                              int *sweeps)
{
    static_assert(NT >= 512, "256 row threads and 224 column threads");
    __shared__ RotF rot[CHASE_N];
    __shared__ int ctl[2];
    __shared__ cf s_sigma;
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    int hi = m - 1, it = 0, tot = 0, n = 0, st = 0;
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
        if (n + (h - lo) > max_log) {
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
                if (t >= NT - CHASE_N && t - (NT - CHASE_N) < k1 - k0) {
                    const int i = t - (NT - CHASE_N);
                    const RotF g = rot[i];
                    log[n + i] = make_float4(g.c, g.s.x, g.s.y, __int_as_float(k0 + i));
                }
            }
            n += k1 - k0;
            __syncthreads();
        }
    }
    *nr = n;
    *sweeps = tot;   // (counted by warp 0)
    __syncthreads();
    return st;
}

// The logged rotations on 32 lines of L entries each: line x of this warp is
// base[i * stride], i < L, for lanes with base != null; left: G is applied to
// adjacent entries (columns of H), otherwise G^H from the right (rows).  The
// lines are staged in shared memory (zr: this lane's L entries), the two
// entries that a rotation touches are carried in registers along a sweep.
// chunk: 256 entries of this warp's.
__device__ __forceinline__ void apply_log(int L, cf *base, int64_t stride, bool left, const float4 *log, int nr,
                                          cf *zr, float4 *chunk)
{
    constexpr int N = 256;
    const int lane = threadIdx.x & 31;
    if (base)
        for (int i = 0; i < L; ++i) zr[i] = __ldcg(base + i * stride);
    int cur = -2;
    cf a = cmakef(0.f, 0.f), b = a;
    for (int e0 = 0; e0 < nr; e0 += N) {
        const int cnt = (nr - e0) < N ? (nr - e0) : N;
        __syncwarp();
        for (int e = lane; e < cnt; e += 32) chunk[e] = __ldcg(log + e0 + e);
        __syncwarp();
        if (!base) continue;
        for (int e = 0; e < cnt; ++e) {
            const float4 q = chunk[e];
            const int k = __float_as_int(q.w);
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
            g.c = q.x;
            g.s = cmakef(q.y, left ? q.z : -q.z);
            rot32_pair(g, a, b);
        }
    }
    if (!base) return;
    if (cur >= 0) {
        zr[cur] = a;
        zr[cur + 1] = b;
    }
    for (int i = 0; i < L; ++i) __stcg(base + i * stride, zr[i]);
}

// Grid-wide: the rotations of the diagonal block of L rows at l on the rest of
// H (m x m column-major) and on Z: columns l .. of the rows above and of all
// rows of Z, rows l .. of the columns to the right.  One warp per CTA, 32
// lines at a time (the chain through the log is the bound, not the lines).
__device__ void apply_log_lines(int m, cf *H, cf *Z, int ld, int l, int L, const float4 *log, int nr, cf *sp)
{
    __shared__ float4 chunk[256];
    if (threadIdx.x < 32) {
        const int right = m - (l + L), lines = l + m + right;
        cf *zr = sp + (size_t)threadIdx.x * (L | 1);
        for (int x0 = blockIdx.x * 32; x0 < lines; x0 += gridDim.x * 32) {
            const int x = x0 + (int)threadIdx.x;
            cf *base = nullptr;
            int64_t stride = ld;
            if (x < l) base = H + x + (int64_t)l * ld;
            else if (x < l + m) base = Z + (x - l) + (int64_t)l * ld;
            else if (x < lines) { base = H + l + (int64_t)(l + L + (x - l - m)) * ld; stride = 1; }
            apply_log(L, base, stride, x >= l + m, log, nr, zr, chunk);
        }
    }
    __syncthreads();
}

}  // namespace
}  // namespace feast
