// FP32 bulge chase of the single-shift complex QR iteration on a block in
// shared memory, as a chain held by one warp.
//
// What bounds a QR sweep is the chain of its rotations: rotation k needs two
// entries that rotation k - 1 has just produced.  With every rotation applied
// to whole rows and columns before the next is formed, a link cost two or
// three barriers and as many trips through shared memory (~0.27 us in the
// warp form, ~0.5 us in the CTA form).  Here the link is registers only:
//   * every lane keeps the two entries to be annihilated and the two of the
//     next column, and forms the rotation and the 3 x 2 corner that the next
//     one needs redundantly;
//   * a lane owns one of the next 32 columns and carries its entry down the
//     chunk (the left rotations); the one entry that the corner needs of the
//     next column comes by a shuffle, in the shadow of the rotation's
//     reciprocal square roots;
//   * the columns beyond and the right rotations of the rows already passed
//     follow a chunk of up to 32 rotations at a time (far_left, chase_right: a
//     thread per column or row).
#pragma once

#include "common.cuh"

namespace feast {

struct RotF {
    float c;
    cf s;
};

// 1 / sqrt(x) with one Newton step: rsqrtf alone is off by up to 2^-22.9
// with a bias, which thousands of rotations would add up
__device__ __forceinline__ float rsqrt_nr(float x)
{
    const float y = rsqrtf(x);
    return y * fmaf(-0.5f * x * y, y, 1.5f);
}

// G = [c s; -conj(s) c] with G [x; y] = [r; 0], whatever the sizes of x and y:
// the larger entry is brought into [1, 2) first, so that squares neither
// overflow nor vanish.
static __device__ __noinline__ RotF rot32_scaled(cf x, cf y)
{
    RotF g;
    const float mx = fmaxf(fmaxf(fabsf(x.x), fabsf(x.y)), fmaxf(fabsf(y.x), fabsf(y.y)));
    int ex = (int)(__float_as_uint(mx) >> 23);
    ex = ex < 1 ? 1 : (ex > 253 ? 253 : ex);
    const float f = __uint_as_float((unsigned)(254 - ex) << 23);
    x = cmakef(x.x * f, x.y * f);
    y = cmakef(y.x * f, y.y * f);
    const float ax2 = cabs2(x), ay2 = cabs2(y);
    if (ay2 == 0.f) { g.c = 1.f; g.s = cmakef(0.f, 0.f); return g; }
    if (ax2 < 1e-36f) {
        g.c = 0.f;
        const float ia = rsqrt_nr(ay2);
        g.s = cmakef(y.x * ia, -y.y * ia);
        return g;
    }
    const float k = rsqrt_nr(ax2) * rsqrt_nr(ax2 + ay2);
    g.c = ax2 * k;
    g.s = cmakef((x.x * y.x + x.y * y.y) * k, (x.y * y.x - x.x * y.y) * k);   // x conj(y) k
    return g;
}
// The same; the reciprocal roots are under way before the sizes are looked at
// (the test ahead of them cost 50 of 134 clocks).
__device__ __forceinline__ RotF rot32(cf x, cf y)
{
    RotF g;
    const float ax2 = cabs2(x), s2 = ax2 + cabs2(y);
    float ia, ir;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(ia) : "f"(ax2));
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(ir) : "f"(s2));
    const float px = fmaf(x.x, y.x, x.y * y.y), py = fmaf(x.y, y.x, -x.x * y.y);
    if (__builtin_expect(!(ax2 > 1e-30f && s2 > 1e-24f && s2 < 1e30f), 0)) return rot32_scaled(x, y);
    ia *= fmaf(-0.5f * ax2 * ia, ia, 1.5f);
    ir *= fmaf(-0.5f * s2 * ir, ir, 1.5f);
    const float k = ia * ir;
    g.c = ax2 * k;
    g.s = cmakef(px * k, py * k);
    return g;
}
__device__ __forceinline__ void rot32_pair(const RotF &g, cf &a, cf &b)          // G [a; b]
{
    const cf s = g.s;
    const cf na = cmakef(fmaf(g.c, a.x, fmaf(s.x, b.x, -s.y * b.y)), fmaf(g.c, a.y, fmaf(s.x, b.y, s.y * b.x)));
    b = cmakef(fmaf(g.c, b.x, -fmaf(s.x, a.x, s.y * a.y)), fmaf(g.c, b.y, -fmaf(s.x, a.y, -s.y * a.x)));
    a = na;
}
__device__ __forceinline__ RotF rot32_h(const RotF &g)   // [a b] G^H is rot32_pair with conj(s)
{
    RotF h;
    h.c = g.c;
    h.s = cmakef(g.s.x, -g.s.y);
    return h;
}

__device__ __forceinline__ float abs32(cf a) { return sqrtf(cabs2(a)); }

// Wilkinson shift of the trailing 2 x 2 block [h00 h01; h10 h11]: h11 plus the
// smaller root of z^2 - 2 d z - h01 h10, d = (h00 - h11) / 2.
__device__ __forceinline__ cf shift32(cf h00, cf h01, cf h10, cf h11)
{
    const cf d = cmakef(0.5f * (h00.x - h11.x), 0.5f * (h00.y - h11.y));
    const cf bc = cmul(h01, h10);
    const cf w = cadd(cmul(d, d), bc);
    // principal square root of w, on the side of d
    float re = sqrtf(0.5f * (abs32(w) + fabsf(w.x))), im = re > 0.f ? 0.5f * w.y / re : 0.f;
    if (w.x < 0.f) { const float q = re; re = fabsf(im); im = copysignf(q, w.y); }
    if (re * d.x + im * d.y < 0.f) { re = -re; im = -im; }
    const cf den = cmakef(d.x + re, d.y + im);
    const cf corr = cis_zero(den) ? cmakef(0.f, 0.f) : cdiv(bc, den);
    return cmakef(h11.x - corr.x, h11.y - corr.y);
}

// Row k of a block in shared memory as a pointer p with entry c at p[c]:
// row-major with a leading dimension, or packed (rows keep columns >= k - 2,
// the Hessenberg part and the bulge; base(k + 1) - base(k) = m for k < 2,
// m + 1 - k from there on).
struct RowsLd {
    cf *p;
    int ld;
    __device__ __forceinline__ cf *row(int k) const { return p + k * ld; }
    // shared-memory byte address of row k, and of row k + 1 from it
    __device__ __forceinline__ uint32_t addr(int k) const { return (uint32_t)__cvta_generic_to_shared(p) + 8u * (uint32_t)(k * ld); }
    __device__ __forceinline__ uint32_t next(uint32_t a, int) const { return a + 8u * (uint32_t)ld; }
};
__host__ __device__ __forceinline__ int packed_base(int m, int k)
{
    return k <= 2 ? k * m : 2 * m + (k - 2) * (m + 1) - (k * (k - 1) / 2 - 1);
}
__host__ __device__ inline int packed_elems(int m) { return packed_base(m, m - 1) + m; }
struct RowsPacked {
    cf *p;
    int m;
    __device__ __forceinline__ cf *row(int k) const { return p + packed_base(m, k); }
    __device__ __forceinline__ uint32_t addr(int k) const
    {
        return (uint32_t)__cvta_generic_to_shared(p) + 8u * (uint32_t)packed_base(m, k);
    }
    __device__ __forceinline__ uint32_t next(uint32_t a, int k) const { return a + 8u * (uint32_t)(k < 2 ? m : m + 1 - k); }
};
__device__ __forceinline__ cf lds32(uint32_t a)
{
    cf v;
    asm volatile("ld.shared.v2.f32 {%0, %1}, [%2];" : "=f"(v.x), "=f"(v.y) : "r"(a) : "memory");
    return v;
}
__device__ __forceinline__ void sts32(uint32_t a, cf v)
{
    asm volatile("st.shared.v2.f32 [%0], {%1, %2};" ::"r"(a), "f"(v.x), "f"(v.y) : "memory");
}

// Most rotations of one chase_left() call.
constexpr int CHASE_N = 32;

// One warp: rotations k0 .. k1 - 1 (at most CHASE_N) of a sweep with shift
// sigma over the active rows [lo, hi] of the w x w upper Hessenberg block H;
// k1 <= hi.  k0 == lo starts the sweep; otherwise the bulge stands at
// H[k0 + 1][k0 - 1].  Rotation k goes to rot[k - k0].  Columns k0 + 1 ..
// k0 + 32 are updated (left rotations); those beyond wait for far_left(), the
// rows above k1 for chase_right().  On return the bulge stands at
// H[k1 + 1][k1 - 1] (k1 < hi).  Ends with __syncwarp().
//
// Nothing but the column's own store is written inside the chain: lane k - k0
// keeps what rotation k was made of and of column k, and finishes column k - 1
// and the diagonal entry after the chunk (a store by single lanes inside the
// loop cost 100 clocks per rotation and more).  ~214 clocks per rotation on 64 rows (366 before;
// 241 without the unrolling, whose two copies need no register moves).
template <typename Rows>
__device__ __forceinline__ void chase_left(Rows H, int w, int lo, int hi, int k0, int k1, cf sigma, RotF *rot)
{
    const int lane = threadIdx.x & 31;
    const cf zero = cmakef(0.f, 0.f);
    const int c = k0 + 1 + lane;
    const bool in = c < w;
    const uint32_t oc = 8u * (uint32_t)(in ? c : w - 1);       // (a lane without a column reads the last one)
    uint32_t r0 = H.addr(k0), r1 = H.next(r0, k0);
    cf d0 = lds32(r0 + 8 * k0), d1 = lds32(r1 + 8 * k0), x, y;
    if (k0 == lo) {
        x = cmakef(d0.x - sigma.x, d0.y - sigma.y);
        y = d1;
    } else {
        x = lds32(r0 + 8 * (k0 - 1));
        y = lds32(r1 + 8 * (k0 - 1));
    }
    // this lane's column: the carried entry of row k, and row k + 1's
    cf a = lds32(r0 + oc), n = lds32(r1 + oc);
    cf v = lds32(r1 + 8 * (k0 + 1));
    uint32_t r2 = (k0 + 2 <= hi) ? H.next(r1, k0 + 1) : r1;
    cf e = (k0 + 2 <= hi) ? lds32(r2 + 8 * (k0 + 1)) : zero;
    cf kx = zero, ky = zero, kd0 = zero, kd1 = zero;           // lane k - k0: rotation k's
    RotF kg;
    kg.c = 1.f;
    kg.s = zero;
#pragma unroll 2
    for (int k = k0; k < k1; ++k) {
        // the next column's entry of row k, and the next step's entries
        const cf u = cmakef(__shfl_sync(0xffffffffu, a.x, k - k0), __shfl_sync(0xffffffffu, a.y, k - k0));
        const cf nn = lds32(r2 + oc);                           // (row k + 2; past the end: row hi again, unused)
        const cf vn = lds32(r2 + 8 * (k + 2 <= hi ? k + 2 : hi));
        const bool third = k + 3 <= hi && k + 1 < k1;          // (a block may end at row k1 + 1)
        const uint32_t r3 = third ? H.next(r2, k + 2) : r2;
        const cf el = lds32(r3 + 8 * (third ? k + 2 : k));
        const cf en = third ? el : zero;
        const RotF g = rot32(x, y);
        const bool mine = lane == k - k0;
        kx = mine ? x : kx;
        ky = mine ? y : ky;
        kd0 = mine ? d0 : kd0;
        kd1 = mine ? d1 : kd1;
        kg.c = mine ? g.c : kg.c;
        kg.s = mine ? g.s : kg.s;
        // the corner: row k + 1 of columns k, k + 1 (left), then rows k + 1, k + 2 (right)
        const RotF gh = rot32_h(g);
        cf p1 = cmakef(fmaf(g.c, d1.x, -fmaf(g.s.x, d0.x, g.s.y * d0.y)), fmaf(g.c, d1.y, -fmaf(g.s.x, d0.y, -g.s.y * d0.x)));
        cf q1 = cmakef(fmaf(g.c, v.x, -fmaf(g.s.x, u.x, g.s.y * u.y)), fmaf(g.c, v.y, -fmaf(g.s.x, u.y, -g.s.y * u.x)));
        rot32_pair(gh, p1, q1);
        x = p1;
        d0 = q1;
        y = cmul(e, gh.s);
        d1 = cmakef(g.c * e.x, g.c * e.y);
        // this lane's column (from k + 1 on)
        rot32_pair(g, a, n);
        if (c > k && in) sts32(r0 + oc, a);
        a = n;
        n = nn;
        v = vn;
        e = en;
        r0 = r1;
        r1 = r2;
        r2 = r3;
    }
    // row k1 and the bulge (r0 = row k1, r1 = row k1 + 1 when k1 < hi)
    if (c > k1 && in) sts32(r0 + oc, a);
    if (lane == 0) {
        sts32(r0 + 8 * k1, d0);
        sts32(r0 + 8 * (k1 - 1), x);
        if (k1 < hi) {
            sts32(r1 + 8 * k1, d1);
            sts32(r1 + 8 * (k1 - 1), y);
        }
    }
    // rotation k = k0 + lane: columns k - 1, (r, 0), and k, the entry of row k
    const int k = k0 + lane;
    if (k < k1) {
        const uint32_t rk = H.addr(k);
        rot32_pair(kg, kd0, kd1);
        sts32(rk + 8 * k, kd0);
        if (k > lo) {
            rot32_pair(kg, kx, ky);
            sts32(rk + 8 * (k - 1), kx);
            sts32(H.next(rk, k) + 8 * (k - 1), zero);
        }
        rot[lane] = kg;
    }
    __syncwarp();
}

// The left rotations k0 .. k1 - 1 on column c (> k0 + 32) of the block.  A
// thread per column.
template <typename Rows>
__device__ __forceinline__ void far_left(Rows H, int c, int k0, int k1, const RotF *rot)
{
    cf *r = H.row(k0);
    cf a = r[c];
    cf *rn = H.row(k0 + 1);
    cf b = rn[c];
    for (int k = k0; k < k1; ++k) {
        cf *rnn = (k + 2 <= k1) ? H.row(k + 2) : rn;
        const cf bn = rnn[c];
        rot32_pair(rot[k - k0], a, b);
        r[c] = a;
        a = b;
        b = bn;
        r = rn;
        rn = rnn;
    }
    r[c] = a;
}

// The right rotations kb .. k1 - 1 of one row (row[c], stride 1), rot[k - k0];
// kb >= k0.  A thread per row.
__device__ __forceinline__ void chase_right(cf *row, int k0, int kb, int k1, const RotF *rot)
{
    if (kb >= k1) return;
    cf a = row[kb], b = row[kb + 1];
    for (int k = kb; k < k1; ++k) {
        const cf bn = (k + 2 <= k1) ? row[k + 2] : cmakef(0.f, 0.f);
        rot32_pair(rot32_h(rot[k - k0]), a, b);
        row[k] = a;
        a = b;
        b = bn;
    }
    row[k1] = a;
}

}  // namespace feast
