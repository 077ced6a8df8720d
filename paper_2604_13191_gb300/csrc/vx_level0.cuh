// vx_level0.cuh -- device code of the level-0 voxelization, shared by the single-problem
// path (vx_voxelize.cu) and the batched path (vx_batch.cu): the capsule and triangle
// sub-cell predicates and measures, the candidate, reduce and finalize kernels.
//
// Arithmetic: every FP32 quantity that decides a bit, and every per-voxel sum, is
// evaluated with the operation order written here and no contraction (the library is
// compiled with -fmad=false); per-voxel sums run sequentially in primitive order.
#pragma once

#include <math.h>

#include <algorithm>

#include "vx_internal.cuh"

namespace {

constexpr float kPi = 3.14159265358979f;
constexpr int RED_WARPS = 4;        // warps per block in the reduce kernels
constexpr int EMIT_WARPS = 8;

struct GridDev {
    float o[3];
    float s;      // 1 / voxel_size (FP32)
    int R;
};

// Per-segment temporary outputs (indexed by candidate-voxel segment id).
struct SegOut {
    uint32_t* key;
    uint64_t* mask;     // [n][8]
    float* mass;
    float* moment;      // [n][6]
    uint32_t* nonzero;
};

__device__ __forceinline__ float fmin2(float a, float b) { return (b < a) ? b : a; }
__device__ __forceinline__ float fmax2(float a, float b) { return (b > a) ? b : a; }

// ------------------------------------------------------------------------------------
// capsule vs closed box [lo, hi]: a, b local endpoints, rr = r^2
// ------------------------------------------------------------------------------------
__device__ __forceinline__ float sqdist_point_box(float px, float py, float pz, const float* lo,
                                                  const float* hi) {
    float p[3] = {px, py, pz};
    float e[3];
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        if (p[i] < lo[i]) e[i] = lo[i] - p[i];
        else if (p[i] > hi[i]) e[i] = p[i] - hi[i];
        else e[i] = 0.0f;
    }
    return (e[0] * e[0] + e[1] * e[1]) + e[2] * e[2];
}

__device__ __forceinline__ float seg_g(const float* a, const float* d, float t, const float* lo,
                                       const float* hi) {
    if (!(t >= 0.0f)) t = 0.0f;
    else if (t > 1.0f) t = 1.0f;
    return sqdist_point_box(a[0] + t * d[0], a[1] + t * d[1], a[2] + t * d[2], lo, hi);
}

// Step 3 of the capsule test: min over t in [0,1] of the squared segment-box distance,
// taken at the stationary points of the quadratic pieces that can hold the minimum.
// (Scalar code with explicit selects: no dynamically indexed local arrays.)
__device__ __forceinline__ float sel3(int i, float x, float y, float z) { return i == 0 ? x : (i == 1 ? y : z); }

// Called out of line (it is the rare, long case) with scalar arguments, so that nothing of
// it goes through local memory: the box is [lo, lo + ext] (exact for the voxel [0, 1]^3 and
// for the sub-cells [k/8, (k+1)/8]).
__device__ __noinline__ float seg_box_min(float ax, float ay, float az, float dx, float dy, float dz, float lx,
                                          float ly, float lz, float ext) {
    const float a[3] = {ax, ay, az}, d[3] = {dx, dy, dz};
    const float lo[3] = {lx, ly, lz}, hi[3] = {lx + ext, ly + ext, lz + ext};
    float L = -INFINITY, U = INFINITY;
    int iL = -1, jU = -1, moving = 0;
    float plo0 = 0.0f, plo1 = 0.0f, plo2 = 0.0f, phi0 = 0.0f, phi1 = 0.0f, phi2 = 0.0f;
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        if (d[i] != 0.0f) {
            ++moving;
            const float pl = (d[i] > 0.0f) ? lo[i] : hi[i];
            const float ph = (d[i] > 0.0f) ? hi[i] : lo[i];
            if (i == 0) { plo0 = pl; phi0 = ph; } else if (i == 1) { plo1 = pl; phi1 = ph; } else { plo2 = pl; phi2 = ph; }
            const float jl = (pl - a[i]) / d[i];
            const float jh = (ph - a[i]) / d[i];
            if (jl > L) { L = jl; iL = i; }
            if (jh < U) { U = jh; jU = i; }
        }
    }
    if (moving == 0) return INFINITY;
    if (L <= U) {
        float t;
        if (U < 0.0f) t = 0.0f;
        else if (L > 1.0f) t = 1.0f;
        else t = fmax2(L, 0.0f);
        return seg_g(a, d, t, lo, hi);
    }
    // the axis giving L lies below its slab and the one giving U above it on [U, L]
    const int k = 3 - iL - jU;
    // beta per axis for the pair {iL, jU}: plo for iL, phi for jU
    const float b0 = (iL == 0) ? plo0 : phi0;
    const float b1 = (iL == 1) ? plo1 : phi1;
    const float b2 = (iL == 2) ? plo2 : phi2;
    const int p0 = iL < jU ? iL : jU, p1 = iL < jU ? jU : iL;
    const float a0 = sel3(p0, a[0], a[1], a[2]), a1 = sel3(p1, a[0], a[1], a[2]);
    const float d0 = sel3(p0, d[0], d[1], d[2]), d1 = sel3(p1, d[0], d[1], d[2]);
    const float e0 = sel3(p0, b0, b1, b2), e1 = sel3(p1, b0, b1, b2);
    float num = d0 * (e0 - a0);
    float den = d0 * d0;
    num = num + d1 * (e1 - a1);
    den = den + d1 * d1;
    float gmin = seg_g(a, d, num / den, lo, hi);
    const float dk = sel3(k, d[0], d[1], d[2]);
    if (dk != 0.0f) {
#pragma unroll
        for (int side = 0; side < 2; ++side) {
            // beta: iL -> plo, jU -> phi, k -> plo (side 0) or phi (side 1)
            const float c0 = (k == 0) ? (side == 0 ? plo0 : phi0) : b0;
            const float c1 = (k == 1) ? (side == 0 ? plo1 : phi1) : b1;
            const float c2 = (k == 2) ? (side == 0 ? plo2 : phi2) : b2;
            float n3 = d[0] * (c0 - a[0]);
            float d3 = d[0] * d[0];
            n3 = n3 + d[1] * (c1 - a[1]);
            d3 = d3 + d[1] * d[1];
            n3 = n3 + d[2] * (c2 - a[2]);
            d3 = d3 + d[2] * d[2];
            const float gc = seg_g(a, d, n3 / d3, lo, hi);
            if (gc < gmin) gmin = gc;
        }
    }
    return gmin;
}

// Per-axis terms of steps 1 and 2 for the sub-cell interval [k/8, (k+1)/8] of one axis.
struct AxisTerms {
    float g2, ea2, eb2;
};
// The gap (lo > mx ? lo - mx : mn > hi ? mn - hi : 0) is written max(lo - mx, mn - hi, 0):
// at most one of the two differences is positive, and a difference is positive exactly when
// its comparison holds (FP subtraction of finite values), so the two forms round to the same
// value up to the sign of a zero, which the square removes.  Likewise the endpoint distances.
// max of three (one instruction on sm_100 and later; exact, like two two-input maxima)
__device__ __forceinline__ float fmax3(float a, float b, float c) {
    float r;
    asm("max.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(b), "f"(c));
    return r;
}
__device__ __forceinline__ float gap3(float lo, float hi, float mn, float mx) {
    return fmax3(lo - mx, mn - hi, 0.0f);
}
__device__ __forceinline__ AxisTerms axis_terms(float a, float b, int k) {
    const float lo = (float)k * 0.125f, hi = (float)(k + 1) * 0.125f;
    const float mn = fminf(a, b), mx = fmaxf(a, b);
    const float g = gap3(lo, hi, mn, mx);
    const float ea = gap3(lo, hi, a, a);
    const float eb = gap3(lo, hi, b, b);
    AxisTerms t;
    t.g2 = g * g;
    t.ea2 = ea * ea;
    t.eb2 = eb * eb;
    return t;
}

// Per-warp pool of step-3 work of one voxel: (capsule slot, sub-cell) tasks left undecided
// by steps 1-2 of the batch's capsules, those capsules, and the voxel's mask while the pool
// is evaluated.  Tasks of many capsules are evaluated 32 at a time, so that the exact
// minimum (the expensive case) runs with all lanes busy.
constexpr int CT_TASKS = 512;
// One capsule in voxel-local grid units: (a.xyz, r^2), (b.xyz, r + eta), (d = b - a, 1 / |d|^2)
// with eta the margin of capsule_cell_quick.
struct CapsuleLocal {
    float4 a_rr, b_reta, d_idd;
};
// The x-axis terms of steps 1-2 for the 8 sub-cell columns sx = 0..7 (the same for every
// lane): squared gap of the segment's extent, squared distances of the endpoints.
struct CapsuleX {
    float4 g2[2], ea2[2], eb2[2];
};
struct CapsuleSlot {
    CapsuleLocal c;
    CapsuleX x;
};
struct CapsuleTasks {
    CapsuleSlot slot[32];          // the batch's capsules (by lane)
    float q[32 * 7];               // w mu and w mu T(t) of up to 32 pairs (pair-major, stride 7)
    uint32_t mask[16];             // 512-bit mask, word w = lanes 2w (low half) and 2w+1
    uint16_t task[CT_TASKS];       // batch slot << 9 | sub-cell id
};

__device__ __forceinline__ CapsuleX capsule_x(float a, float b) {
    float g[8], ea[8], eb[8];
#pragma unroll
    for (int sx = 0; sx < 8; ++sx) {
        const AxisTerms t = axis_terms(a, b, sx);
        g[sx] = t.g2;
        ea[sx] = t.ea2;
        eb[sx] = t.eb2;
    }
    CapsuleX x;
    x.g2[0] = make_float4(g[0], g[1], g[2], g[3]);
    x.g2[1] = make_float4(g[4], g[5], g[6], g[7]);
    x.ea2[0] = make_float4(ea[0], ea[1], ea[2], ea[3]);
    x.ea2[1] = make_float4(ea[4], ea[5], ea[6], ea[7]);
    x.eb2[0] = make_float4(eb[0], eb[1], eb[2], eb[3]);
    x.eb2[1] = make_float4(eb[4], eb[5], eb[6], eb[7]);
    return x;
}

// A radius whose square overflows leaves r^2 = inf, and steps 1 and 2 then hold for a whole row when
// its y and z terms have a finite sum (anything <= inf) and for none of it otherwise (inf - inf is not a
// number, and no comparison with that holds).  capsule_row compares by the sign of a difference, which is
// undefined for inf - inf, so it takes at most the largest finite value for r^2, and such a capsule's x
// terms are zero (capsule_x of two NaN): the budget is then at least zero in the one case and -inf in the
// other.
constexpr float kHugeRR = 3.402823466e38f;

// Steps 1-2 of the capsule test for one row of 8 sub-cells (sx = 0..7 at sy; tz: the z terms of
// its slab).  `set` receives the sub-cells that step 2 decides set, `open` those that pass step 1.
// Both steps compare the x term with what r^2 leaves after the y and z terms:
//   step 1 fails  when  g_x^2 > r^2 - (g_y^2 + g_z^2),
//   step 2 passes when  e_x^2 <= r^2 - (e_y^2 + e_z^2)  for endpoint a or b,
// so a row's 8 sub-cells compare 8 x terms with one budget each.  (e >= g on every axis, an
// endpoint being no closer to a sub-cell than the segment's extent, and the operations are
// monotone, so a set sub-cell is open too.)
__device__ __forceinline__ void capsule_row(const CapsuleSlot& cs, const AxisTerms& tz, int sy, uint32_t& set,
                                            uint32_t& open) {
    const AxisTerms ty = axis_terms(cs.c.a_rr.y, cs.c.b_reta.y, sy);
    const float rr = fminf(cs.c.a_rr.w, kHugeRR);
    const float TG = rr - (ty.g2 + tz.g2);
    const float TA = rr - (ty.ea2 + tz.ea2);
    const float TB = rr - (ty.eb2 + tz.eb2);
    const CapsuleX& X = cs.x;
    const float4 g0 = X.g2[0], g1 = X.g2[1], a0 = X.ea2[0], a1 = X.ea2[1], b0 = X.eb2[0], b1 = X.eb2[1];
    const float xg[8] = {g0.x, g0.y, g0.z, g0.w, g1.x, g1.y, g1.z, g1.w};
    const float xa[8] = {a0.x, a0.y, a0.z, a0.w, a1.x, a1.y, a1.z, a1.w};
    const float xb[8] = {b0.x, b0.y, b0.z, b0.w, b1.x, b1.y, b1.z, b1.w};
    // a comparison x <= T by the sign of T - x (the exact sign of the difference; T and x are not
    // both infinite with one sign, see kHugeRR), shifted into a word: additions run on the FMA pipe, where compares and selects load the ALU pipe, the busier
    uint32_t out = 0, shut = 0;
#pragma unroll
    for (int sx = 7; sx >= 0; --sx) {
        out = __funnelshift_l(__float_as_uint(TA - xa[sx]) & __float_as_uint(TB - xb[sx]), out, 1);
        shut = __funnelshift_l(__float_as_uint(TG - xg[sx]), shut, 1);
    }
    set = ~out & 0xffu;
    open = ~shut & 0xffu;
}

// The unset sub-cells of one lane's two rows, as packed pairs (row sy0, row sy0 + 1): the centres
// of each row's first and last one, negated, and their sum.
struct UnsetRows {
    f2 nlo, nhi, sum;
};
__device__ __forceinline__ UnsetRows unset_rows(uint32_t chunk) {
    float lo[2], hi[2];
#pragma unroll
    for (int yi = 0; yi < 2; ++yi) {
        const uint32_t u = ~(chunk >> (8 * yi)) & 0xffu;   // (no meaning when the row is full)
        lo[yi] = (float)(__ffs(u) - 1) * 0.125f + 0.0625f;
        hi[yi] = (float)(31 - __clz(u)) * 0.125f + 0.0625f;
    }
    return {f2_pack(-lo[0], -lo[1]), f2_pack(-hi[0], -hi[1]), f2_pack(lo[0] + hi[0], lo[1] + hi[1])};
}

// Per row (reach0: y, reach1: y + 1/8), true unless the capsule is separated, by more than r + eta,
// from the box around the row's unset sub-cells: none of them can then be set (see
// capsule_cell_quick).  The separation is taken along v, from the centre of the end
// sub-cell that faces the capsule to the nearest point of its axis; the box reaches away from
// that centre by half a sub-cell, and along x to the row's other end.  Any v gives a bound, so
// neither the choice of the end nor the rounding of v matters; a NaN leaves the row open.
// (The two rows as packed FP32 pairs; Az = a.z minus the slab's centre, ny = -(y, y + 1/8).)
__device__ __forceinline__ void rows_reached(const CapsuleLocal& c, const UnsetRows& u, f2 ny, float Az, bool& reach0,
                                             bool& reach1) {
    const float4 a = c.a_rr, b = c.b_reta, d = c.d_idd;
    float s0, s1, lo0, lo1, hi0, hi1;
    f2_unpack(u.sum, s0, s1);
    f2_unpack(u.nlo, lo0, lo1);
    f2_unpack(u.nhi, hi0, hi1);
    const float mid2 = a.x + b.x;
    const f2 nref = f2_pack(mid2 < s0 ? lo0 : hi0, mid2 < s1 ? lo1 : hi1);
    const f2 e = f2_fma(nref, f2_pack(2.0f, 2.0f), u.sum);       // to the row's other end, signed
    const f2 Ax = f2_add(f2_pack(a.x, a.x), nref), Ay = f2_add(f2_pack(a.y, a.y), ny), Az2 = f2_pack(Az, Az);
    const f2 dx = f2_pack(d.x, d.x), dy = f2_pack(d.y, d.y), dz = f2_pack(d.z, d.z);
    const float azdz = Az * d.z;
    float t0, t1;
    f2_unpack(f2_fma(Ax, dx, f2_fma(Ay, dy, f2_pack(azdz, azdz))), t0, t1);
    const f2 tc = f2_pack(__saturatef(-d.w * t0), __saturatef(-d.w * t1));
    const f2 vx = f2_fma(tc, dx, Ax), vy = f2_fma(tc, dy, Ay), vz = f2_fma(tc, dz, Az2);
    const f2 sa = f2_fma(vx, Ax, f2_fma(vy, Ay, f2_mul(vz, Az2)));
    const f2 sb = f2_fma(vx, dx, f2_fma(vy, dy, f2_fma(vz, dz, sa)));
    const f2 vv = f2_mul(f2_fma(vx, vx, f2_fma(vy, vy, f2_mul(vz, vz))), f2_pack(b.w * b.w, b.w * b.w));
    float x0, x1, y0, y1, z0, z1, e0, e1, a0, a1, b0, b1, r0, r1;
    f2_unpack(vx, x0, x1);
    f2_unpack(vy, y0, y1);
    f2_unpack(vz, z0, z1);
    f2_unpack(f2_mul(e, vx), e0, e1);
    f2_unpack(sa, a0, a1);
    f2_unpack(sb, b0, b1);
    f2_unpack(vv, r0, r1);
    const float p0 = fminf(a0, b0) - __fmaf_rn(0.0625f, (fabsf(x0) + fabsf(y0)) + fabsf(z0), fmaxf(e0, 0.0f));
    const float p1 = fminf(a1, b1) - __fmaf_rn(0.0625f, (fabsf(x1) + fabsf(y1)) + fabsf(z1), fmaxf(e1, 0.0f));
    reach0 = !(p0 * fabsf(p0) > r0);
    reach1 = !(p1 * fabsf(p1) > r1);
}

// True when an endpoint of the capsule is within r of every point of the voxel: step 2 then
// passes for each of its sub-cells (the far bounds are no smaller than a sub-cell's endpoint
// distance on any axis, and the operations are monotone).
__device__ __forceinline__ bool capsule_covers(const float* a, const float* b, float rr) {
    float fa2[3], fb2[3];
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        const float fa = fmaxf(1.0f - a[i], a[i] - 0.0f), fb = fmaxf(1.0f - b[i], b[i] - 0.0f);
        fa2[i] = fa * fa;
        fb2[i] = fb * fb;
    }
    return fa2[0] <= rr - (fa2[1] + fa2[2]) || fb2[0] <= rr - (fb2[1] + fb2[2]);
}

// Local capsule of endpoints a, b (voxel-local grid units) and radius r.  eta bounds, with
// a wide factor, the FP32 error of the distance bounds below plus that of step 3: both
// scale with the magnitude M of the local coordinates (and r), and sum to less than
// 3e-6 (M + r + 3).
__device__ __forceinline__ CapsuleLocal capsule_local(const float* a, const float* b, float r) {
    const float d[3] = {b[0] - a[0], b[1] - a[1], b[2] - a[2]};
    const float dd = (d[0] * d[0] + d[1] * d[1]) + d[2] * d[2];
    const float M = fmax3(fmax3(fabsf(a[0]), fabsf(a[1]), fabsf(a[2])), fmax3(fabsf(b[0]), fabsf(b[1]), fabsf(b[2])),
                          0.0f);
    const float eta = 2e-5f * ((M + r) + 3.0f);
    CapsuleLocal c;
    c.a_rr = make_float4(a[0], a[1], a[2], r * r);
    c.b_reta = make_float4(b[0], b[1], b[2], r + eta);
    c.d_idd = make_float4(d[0], d[1], d[2], dd > 0.0f ? 1.0f / dd : 0.0f);
    return c;
}

// True when segment a-b (a, b - a, 1/|b - a|^2) is farther than re from the cube of centre
// (cx, cy, cz) and half-size h.  For a unit n, the distance between two convex sets is at
// least their separation along n: here min(n.(a - c), n.(b - c)) - h |n|_1.  n is taken along
// v = p - c, p the point of the segment nearest to c (any v gives a bound; this one is
// nearly tight once the box is a few box sizes away).  The test s > re |v|, s the separation
// times |v|, is done in squares.
__device__ __forceinline__ bool segment_box_separated(float4 a, float4 b, float4 d_idd, float cx, float cy, float cz,
                                                      float h, float re) {
    const float Ax = a.x - cx, Ay = a.y - cy, Az = a.z - cz;
    const float Bx = b.x - cx, By = b.y - cy, Bz = b.z - cz;
    float tc = -((Ax * d_idd.x + Ay * d_idd.y) + Az * d_idd.z) * d_idd.w;
    tc = fminf(fmaxf(tc, 0.0f), 1.0f);
    const float vx = Ax + tc * d_idd.x, vy = Ay + tc * d_idd.y, vz = Az + tc * d_idd.z;
    const float sa = (vx * Ax + vy * Ay) + vz * Az;
    const float sb = (vx * Bx + vy * By) + vz * Bz;
    const float sep = fminf(sa, sb) - h * ((fabsf(vx) + fabsf(vy)) + fabsf(vz));
    const float vv = (vx * vx + vy * vy) + vz * vz;
    return sep > 0.0f && sep * sep > (re * re) * vv;
}

// Sub-cell `id` against the capsule without the exact minimum: -1 provably out, 1 provably in,
// 0 open.  Out: separated by more than r + eta (see segment_box_separated).  In: the point of the
// axis nearest to the sub-cell's centre is within r - eta of the sub-cell.  eta (per capsule)
// covers the FP32 errors of these bounds and of step 3, whose value is the squared distance of
// the segment within 2e-7 (M + 3) (measured against FP64 over 160 M segments, degenerate
// directions among them; eta is 2e-5 (M + r + 3)), so step 3 decides the same.
__device__ __forceinline__ int capsule_cell_quick(const CapsuleLocal& c, int id) {
    const float cx = (float)(id & 7) * 0.125f + 0.0625f, cy = (float)((id >> 3) & 7) * 0.125f + 0.0625f,
                cz = (float)(id >> 6) * 0.125f + 0.0625f;
    const float4 a = c.a_rr, d = c.d_idd;
    const float Ax = a.x - cx, Ay = a.y - cy, Az = a.z - cz;
    const float tc = __saturatef(-d.w * __fmaf_rn(Ax, d.x, __fmaf_rn(Ay, d.y, Az * d.z)));
    const float vx = __fmaf_rn(tc, d.x, Ax), vy = __fmaf_rn(tc, d.y, Ay), vz = __fmaf_rn(tc, d.z, Az);
    const float sa = __fmaf_rn(vx, Ax, __fmaf_rn(vy, Ay, vz * Az));
    const float sb = __fmaf_rn(vx, d.x, __fmaf_rn(vy, d.y, __fmaf_rn(vz, d.z, sa)));
    const float sep = fminf(sa, sb) - 0.0625f * ((fabsf(vx) + fabsf(vy)) + fabsf(vz));
    const float vv = __fmaf_rn(vx, vx, __fmaf_rn(vy, vy, vz * vz));
    const float re = c.b_reta.w;
    if (sep * fabsf(sep) > (re * re) * vv) return -1;
    const float ex = fmaxf(fabsf(vx) - 0.0625f, 0.0f), ey = fmaxf(fabsf(vy) - 0.0625f, 0.0f),
                ez = fmaxf(fabsf(vz) - 0.0625f, 0.0f);
    const float ri = 2.0f * sqrtf(a.w) - re;   // r - eta
    return ri > 0.0f && __fmaf_rn(ex, ex, __fmaf_rn(ey, ey, ez * ez)) <= ri * ri ? 1 : 0;
}

// Step 3 of every pooled task whose sub-cell is not set yet (warp-collective); returns the
// lane's 16 bits of the updated mask.  A task skipped because an earlier task of the same
// sub-cell set it would have returned a bit that is already 1, so the order of evaluation
// does not change the mask.  Most tasks are decided by capsule_cell_quick; the rest are compacted
// in place, so that the exact minimum runs on full warps.
__device__ __forceinline__ uint32_t capsule_step3_pool(CapsuleTasks& ct, int ntask, uint32_t chunk) {
    const int lane = threadIdx.x & 31;
    const uint32_t lo16 = __shfl_sync(0xffffffffu, chunk, (2 * lane) & 31);
    const uint32_t hi16 = __shfl_sync(0xffffffffu, chunk, (2 * lane + 1) & 31);
    if (lane < 16) ct.mask[lane] = lo16 | (hi16 << 16);
    __syncwarp();
    int nkeep = 0;
    for (int t0 = 0; t0 < ntask; t0 += 32) {
        const int t = t0 + lane;
        uint32_t task = 0;
        bool keep = false;
        if (t < ntask) {
            task = ct.task[t];
            const int id = (int)(task & 511u);
            const uint32_t bit = 1u << (id & 31);
            if (!(ct.mask[id >> 5] & bit)) {
                const int q = capsule_cell_quick(ct.slot[task >> 9].c, id);
                keep = q == 0;
                if (q > 0) atomicOr(&ct.mask[id >> 5], bit);
            }
        }
        const uint32_t kept = __ballot_sync(0xffffffffu, keep);
        __syncwarp();   // the chunk is read before any lane writes (writes land at or below it)
        if (keep) ct.task[nkeep + __popc(kept & ((1u << lane) - 1u))] = (uint16_t)task;
        nkeep += __popc(kept);
    }
    __syncwarp();
    for (int t = lane; t < nkeep; t += 32) {
        const uint32_t task = ct.task[t];
        const int id = (int)(task & 511u);
        const uint32_t bit = 1u << (id & 31);
        if (ct.mask[id >> 5] & bit) continue;
        const CapsuleLocal& c = ct.slot[task >> 9].c;
        const int sx = id & 7, sy = (id >> 3) & 7, zz = id >> 6;
        if (seg_box_min(c.a_rr.x, c.a_rr.y, c.a_rr.z, c.d_idd.x, c.d_idd.y, c.d_idd.z, (float)sx * 0.125f,
                        (float)sy * 0.125f, (float)zz * 0.125f, 0.125f) <= c.a_rr.w)
            atomicOr(&ct.mask[id >> 5], bit);
    }
    __syncwarp();
    const uint32_t w = ct.mask[lane >> 1];
    __syncwarp();
    return (w >> (16 * (lane & 1))) & 0xffffu;
}

// pi r^2 * length of the axis a-b clipped to the closed voxel [0,1]^3 (Liang-Barsky)
__device__ __forceinline__ float capsule_measure(const float* a, const float* b, float rg) {
    float d[3] = {b[0] - a[0], b[1] - a[1], b[2] - a[2]};
    float t0 = 0.0f, t1 = 1.0f;
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        if (d[i] == 0.0f) {
            if (a[i] < 0.0f || a[i] > 1.0f) return 0.0f;
        } else {
            float ta = (0.0f - a[i]) / d[i];
            float tb = (1.0f - a[i]) / d[i];
            float tn = d[i] > 0.0f ? ta : tb;
            float tf = d[i] > 0.0f ? tb : ta;
            if (tn > t0) t0 = tn;
            if (tf < t1) t1 = tf;
        }
    }
    if (t1 <= t0) return 0.0f;
    float dn = sqrtf((d[0] * d[0] + d[1] * d[1]) + d[2] * d[2]);
    float len = (t1 - t0) * dn;
    float rr = rg * rg;
    return (kPi * rr) * len;
}

// ------------------------------------------------------------------------------------
// triangle vs closed box: separating axis test (13 axes)
// ------------------------------------------------------------------------------------
__device__ __forceinline__ bool sep3(float p0, float p1, float p2, float rad) {
    float mn = fmin2(fmin2(p0, p1), p2), mx = fmax2(fmax2(p0, p1), p2);
    return (mn > rad || mx < -rad);
}

// all 13 axes for a box (centre c, half extent e); v local vertices, f global edges
__device__ __forceinline__ bool tri_box(const float v[3][3], const float f[3][3], const float* c, float e) {
    float w[3][3];
#pragma unroll
    for (int k = 0; k < 3; ++k)
#pragma unroll
        for (int i = 0; i < 3; ++i) w[k][i] = v[k][i] - c[i];
#pragma unroll
    for (int i = 0; i < 3; ++i)
        if (sep3(w[0][i], w[1][i], w[2][i], e)) return false;
#pragma unroll
    for (int j = 0; j < 3; ++j) {
        const float* q = f[j];
        if (sep3(q[1] * w[0][2] - q[2] * w[0][1], q[1] * w[1][2] - q[2] * w[1][1], q[1] * w[2][2] - q[2] * w[2][1],
                 e * (fabsf(q[1]) + fabsf(q[2]))))
            return false;
        if (sep3(q[2] * w[0][0] - q[0] * w[0][2], q[2] * w[1][0] - q[0] * w[1][2], q[2] * w[2][0] - q[0] * w[2][2],
                 e * (fabsf(q[0]) + fabsf(q[2]))))
            return false;
        if (sep3(q[0] * w[0][1] - q[1] * w[0][0], q[0] * w[1][1] - q[1] * w[1][0], q[0] * w[2][1] - q[1] * w[2][0],
                 e * (fabsf(q[0]) + fabsf(q[1]))))
            return false;
    }
    float n0 = f[0][1] * f[1][2] - f[0][2] * f[1][1];
    float n1 = f[0][2] * f[1][0] - f[0][0] * f[1][2];
    float n2 = f[0][0] * f[1][1] - f[0][1] * f[1][0];
    float p = (n0 * w[0][0] + n1 * w[0][1]) + n2 * w[0][2];
    float rad = e * ((fabsf(n0) + fabsf(n1)) + fabsf(n2));
    return !(p > rad || p < -rad);
}

__device__ __forceinline__ void tri_local(float4 a, float4 b, float4 c, int vi, int vj, int vk, float v[3][3],
                                          float f[3][3]);

// One edge-family test for the sub-cell pair index q (two sub-cell coordinates (i0,i1)
// along the axes (ax0, ax1) that the family's axis depends on).
// family 0: e_x x f (axes y,z), 1: e_y x f (axes x,z), 2: e_z x f (axes x,y)
__device__ __forceinline__ bool family_pass(int fam, const float v[3][3], const float f[3][3], int i0, int i1) {
    const float e = 0.0625f;
    const float c0 = (float)(2 * i0 + 1) * 0.0625f, c1 = (float)(2 * i1 + 1) * 0.0625f;
    bool ok = true;
#pragma unroll
    for (int j = 0; j < 3; ++j) {
        const float* q = f[j];
        float p[3];
        float rad;
        if (fam == 0) {          // w_y = v_y - c(i0), w_z = v_z - c(i1)
#pragma unroll
            for (int k = 0; k < 3; ++k) {
                float wy = v[k][1] - c0, wz = v[k][2] - c1;
                p[k] = q[1] * wz - q[2] * wy;
            }
            rad = e * (fabsf(q[1]) + fabsf(q[2]));
        } else if (fam == 1) {   // w_x = v_x - c(i0), w_z = v_z - c(i1)
#pragma unroll
            for (int k = 0; k < 3; ++k) {
                float wx = v[k][0] - c0, wz = v[k][2] - c1;
                p[k] = q[2] * wx - q[0] * wz;
            }
            rad = e * (fabsf(q[0]) + fabsf(q[2]));
        } else {                 // w_x = v_x - c(i0), w_y = v_y - c(i1)
#pragma unroll
            for (int k = 0; k < 3; ++k) {
                float wx = v[k][0] - c0, wy = v[k][1] - c1;
                p[k] = q[0] * wy - q[1] * wx;
            }
            rad = e * (fabsf(q[0]) + fabsf(q[1]));
        }
        ok = ok && !sep3(p[0], p[1], p[2], rad);
    }
    return ok;
}

// The definition of one edge family's test of pair (i0, i1), for the rare rows that the intervals
// below leave open.
__device__ __noinline__ bool family_exact(float4 a, float4 b, float4 c, int vi, int vj, int vk, int fam, int i0,
                                          int i1) {
    float v[3][3], f[3][3];
    tri_local(a, b, c, vi, vj, vk, v, f);
    return family_pass(fam, v, f, i0, i1);
}

// One edge axis as an interval of i0 for each i1.  The 13-axis test of a sub-cell separates on the axis
// when min_k p_k > rad or max_k p_k < -rad, p_k = s0 w0 + s1 w1 the three vertices' projections
// relative to the sub-cell's centre.  The centre enters all three as the same linear function, so
// in exact arithmetic the axis passes when |T| <= half, T = alpha i0 + beta i1 + gamma.
// With B = |s0| (V0 + 1) + |s1| (V1 + 1), V the largest coordinates of the vertices, every product
// and sum is at most B; the FP32 evaluation of the definition (family_pass) is within 3.2 u B
// (u = 2^-24) of it, and the coefficients here within 10 u B.  They are scaled by 1 / B, so |T| <=
// half - 20 u is a pass of the definition and |T| > half + 20 u a separation.
//   inv != 0: i0 between -(beta i1 + gamma) inv -+ r, r = half |inv|; with the 20 u and the rounding
//     of the bounds a bound is uncertain by less than delta = 20 u |inv| + 5 u (9 + 2 r) + 8 u.
//   inv == 0 (alpha below 1e-4): the row passes or fails as a whole by the sign of half - |beta i1 +
//     gamma|, times 1e9 in the place of r; uncertain when it is within near = 7 |alpha| + 23 u.
// An edge parallel to the family's axis (s0 = s1 = 0; every edge of a box, two of three of a flat sheet)
// never separates: T = 0 against a half of 1 passes every row.
struct EdgeAxis {
    float inv, beta, gamma, half, r, scale, near;
};
__device__ __forceinline__ EdgeAxis edge_axis(const float v0[3], const float v1[3], float V0, float V1, float s0, float s1,
                                              float& delta, bool& fit) {
    const float e = 0.0625f;
    float p[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) p[k] = s1 * (v1[k] - e) + s0 * (v0[k] - e);
    const float mn = fminf(fminf(p[0], p[1]), p[2]), mx = fmax3(p[0], p[1], p[2]);
    // (the 2e-30 makes the scaled half of a zero axis 1, and is below u^2 of any other that fits)
    const float l1 = fabsf(s0) + fabsf(s1), B = __fmaf_rn(fabsf(s0), V0, __fmaf_rn(fabsf(s1), V1, 2e-30f));
    fit = fit && (B > 1e-15f || l1 == 0.0f) && B < 1e30f;   // nothing overflows, underflows or is NaN
    const float q = vx_rcp(B);
    const float alpha = -0.125f * s0 * q;
    EdgeAxis a;
    a.beta = -0.125f * s1 * q;
    a.gamma = 0.5f * (mn + mx) * q;
    a.half = __fmaf_rn(e, l1, __fmaf_rn(0.5f, mx - mn, 2e-30f)) * q;
    const bool row = fabsf(alpha) < 1e-4f;
    a.inv = row ? 0.0f : vx_rcp(alpha);
    a.r = a.half * fabsf(a.inv);
    a.scale = row ? 1e9f : 0.0f;
    a.near = row ? 8.0f * fabsf(alpha) + 1.5e-6f : -1.0f;
    delta = fmaxf(delta, 1.3e-6f * fabsf(a.inv) + (7e-7f * a.r + 7e-6f));
    return a;
}

// The integers of 0..7 in [a, b] as bits; `un` is raised when a bound is within delta of an integer.
__device__ __forceinline__ uint32_t interval_bits(float a, float b, float delta, bool& un) {
    constexpr float MAGIC = 12582912.0f;   // 1.5 * 2^23: adding it rounds to an integer
    // first = ceil(a), past = floor(b) + 1, both as the rounding of the bound plus a half
    a = fminf(fmaxf(a, -0.5f), 7.5f) + 0.5f;
    b = fmaxf(fminf(b + 0.5f, 8.0f), a);
    const float am = a + MAGIC, bm = b + MAGIC;
    un = un || fmaxf(fabsf(a - (am - MAGIC)), fabsf(b - (bm - MAGIC))) > 0.5f - delta;
    // (the shifts take the low five bits of the biased integers; past >= first)
    return __funnelshift_l(0u, 1u, __float_as_uint(bm)) - __funnelshift_l(0u, 1u, __float_as_uint(am));
}

// The 64 pairs of one family as two words, from its three edge axes; rows (i1) that are uncertain
// are marked in `open`.
__device__ __forceinline__ void family_rows(const EdgeAxis ax[3], float delta, uint32_t& lo, uint32_t& hi, uint32_t& open) {
    lo = hi = open = 0;
#pragma unroll 1
    for (int i1 = 0; i1 < 8; ++i1) {
        const float y = (float)i1;
        float l[3], h[3], near[3];
#pragma unroll
        for (int j = 0; j < 3; ++j) {
            const float u = __fmaf_rn(ax[j].beta, y, ax[j].gamma);
            const float w = ax[j].half - fabsf(u);
            const float r = __fmaf_rn(w, ax[j].scale, ax[j].r);
            const float c = -u * ax[j].inv;
            l[j] = c - r;
            h[j] = c + r;
            near[j] = ax[j].near - fabsf(w);
        }
        bool un = fmax3(near[0], near[1], near[2]) >= 0.0f;
        const uint32_t bits = interval_bits(fmax3(l[0], l[1], l[2]), -fmax3(-h[0], -h[1], -h[2]), delta, un);
        const uint32_t at = bits << (8 * (i1 & 3));
        if (i1 < 4) lo |= at; else hi |= at;
        open |= un ? 1u << i1 : 0u;
    }
}

// The sub-cells of one (triangle, voxel) pair as 64 bytes (row sy + 8 sz, bit sx): v and f the
// local vertices and edges of (A, B, C) in voxel (vi, vj, vk).  One lane per pair: an axis decides a
// whole row of sub-cells as an interval, about 70 dispatch slots for 28 triangles at once, where
// the warp testing sub-cells one triangle at a time took about 200 for every triangle.
// Kept short: the reduce's warps walk different parts of a long kernel, and waiting for instructions
// was their first stall.  One body for the three families, rows one at a time, and the clip and sum
// loops not unrolled took the mesh's reduce from 8.87 to 7.54 ms.
constexpr int TRI_MASK = 68;   // bytes from one pair's mask to the next (17 words: no bank conflict)
__device__ __forceinline__ void tri_mask(const float v[3][3], const float f[3][3], float4 A, float4 B, float4 C, int vi,
                                         int vj, int vk, uint8_t* __restrict__ out) {
    const float e = 0.0625f;
    float x[3][3], V[3];
    uint32_t box[3];
#pragma unroll
    for (int q = 0; q < 16; ++q) reinterpret_cast<uint32_t*>(out)[q] = 0u;
#pragma unroll
    for (int i = 0; i < 3; ++i) {
#pragma unroll
        for (int k = 0; k < 3; ++k) x[i][k] = v[k][i];
        V[i] = fmax3(fabsf(x[i][0]), fabsf(x[i][1]), fabsf(x[i][2])) + 1.0f;
        box[i] = 0;
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            const float c = (float)(2 * k + 1) * 0.0625f;
            if (!sep3(x[i][0] - c, x[i][1] - c, x[i][2] - c, e)) box[i] |= 1u << k;
        }
    }
    // the pairs (i0 + 8 i1) that pass the edge axes of families 0 (y, z), 1 (x, z), 2 (x, y)
    uint32_t fam[6];
#pragma unroll 1
    for (int fa = 0; fa < 3; ++fa) {
        // the family's coordinates (i0, i1): (y, z), (x, z), (x, y)
        float x0[3], x1[3];
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            x0[k] = fa == 0 ? x[1][k] : x[0][k];
            x1[k] = fa == 2 ? x[1][k] : x[2][k];
        }
        const float V0 = fa == 0 ? V[1] : V[0], V1 = fa == 2 ? V[1] : V[2];
        EdgeAxis ax[3];
        float delta = 0.0f;
        bool fit = true;
#pragma unroll
        for (int j = 0; j < 3; ++j) {
            // p_k = s0 (v_a0 - c0) + s1 (v_a1 - c1), as family_pass
            const float s0 = fa == 1 ? f[j][2] : (fa == 0 ? -f[j][2] : -f[j][1]);
            const float s1 = fa == 1 ? -f[j][0] : (fa == 0 ? f[j][1] : f[j][0]);
            ax[j] = edge_axis(x0, x1, V0, V1, s0, s1, delta, fit);
        }
        uint32_t lo, hi, open;
        family_rows(ax, delta, lo, hi, open);
        if (!fit) open = 0xffu;
        open &= fa == 2 ? box[1] : box[2];   // (rows outside the box need no decision)
        while (open) {
            const int i1 = __ffs(open) - 1;
            open &= open - 1;
            uint32_t bits = 0;
            for (int i0 = 0; i0 < 8; ++i0)
                if (family_exact(A, B, C, vi, vj, vk, fa, i0, i1)) bits |= 1u << i0;
            const int sh = 8 * (i1 & 3);
            if (i1 < 4) lo = (lo & ~(0xffu << sh)) | (bits << sh);
            else hi = (hi & ~(0xffu << sh)) | (bits << sh);
        }
        // (constant indices: fam stays in registers)
        if (fa == 0) { fam[0] = lo; fam[1] = hi; }
        else if (fa == 1) { fam[2] = lo; fam[3] = hi; }
        else { fam[4] = lo; fam[5] = hi; }
    }
    // the box axes: y columns and z rows of family 0, x columns of family 1
    const uint32_t ycols = box[1] * 0x01010101u, xcols = box[0] * 0x01010101u;
    uint32_t zlo = 0, zhi = 0;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        zlo |= (box[2] >> k) & 1u ? 0xffu << (8 * k) : 0u;
        zhi |= (box[2] >> (4 + k)) & 1u ? 0xffu << (8 * k) : 0u;
    }
    fam[0] &= ycols & zlo;
    fam[1] &= ycols & zhi;
    fam[2] &= xcols;
    fam[3] &= xcols;
    // the face normal, scaled and bounded as the edge axes (sums of three products: within 16 u)
    const float n0 = f[0][1] * f[1][2] - f[0][2] * f[1][1];
    const float n1 = f[0][2] * f[1][0] - f[0][0] * f[1][2];
    const float n2 = f[0][0] * f[1][1] - f[0][1] * f[1][0];
    const float rad = e * ((fabsf(n0) + fabsf(n1)) + fabsf(n2));
    const float Bn = fabsf(n0) * V[0] + (fabsf(n1) * V[1] + fabsf(n2) * V[2]);
    const bool fit = Bn > 1e-30f && Bn < 1e30f;
    const float q = vx_rcp(Bn);
    const float alpha = -0.125f * n0 * q, beta = -0.125f * n1 * q, zeta = -0.125f * n2 * q, half = rad * q;
    const float gamma = ((n0 * (v[0][0] - e) + n1 * (v[0][1] - e)) + n2 * (v[0][2] - e)) * q;
    const bool row = fabsf(alpha) < 1e-4f;
    const float inv = row ? 0.0f : vx_rcp(alpha), r0 = half * fabsf(inv), scale = row ? 1e9f : 0.0f;
    const float near = row ? 8.0f * fabsf(alpha) + 1.5e-6f : -1.0f;
    const float delta = 1.3e-6f * fabsf(inv) + (7e-7f * r0 + 7e-6f);
    // rows with candidates, in the order of their bits in family 0
    uint32_t w = fam[0];
    int z0 = 0;
    for (;;) {
        if (w == 0u) {
            if (z0) break;
            z0 = 4;
            w = fam[1];
            if (w == 0u) break;
        }
        const int bit = __ffs(w) - 1, sy = bit & 7, sz = z0 + (bit >> 3);
        w &= w - 1u;
        uint32_t bits = __byte_perm(fam[2], fam[3], sz) & __byte_perm(fam[4], fam[5], sy) & 0xffu;
        if (bits) {
            const float u = __fmaf_rn(beta, (float)sy, __fmaf_rn(zeta, (float)sz, gamma));
            const float wd = half - fabsf(u);
            const float r = __fmaf_rn(wd, scale, r0), c = -u * inv;
            bool un = !fit || fabsf(wd) <= near;
            const uint32_t pass = interval_bits(c - r, c + r, delta, un);
            if (!un) {
                bits &= pass;
            } else {
                // the definition, sub-cell by sub-cell
                const float pz = n2 * (v[0][2] - (float)(2 * sz + 1) * 0.0625f);
                const float py = n1 * (v[0][1] - (float)(2 * sy + 1) * 0.0625f);
                for (int sx = 0; sx < 8; ++sx) {
                    const float px = n0 * (v[0][0] - (float)(2 * sx + 1) * 0.0625f);
                    if (fabsf((px + py) + pz) > rad) bits &= ~(1u << sx);
                }
            }
            out[sy + 8 * sz] = (uint8_t)bits;
        }
    }
}

// Clipped-polygon buffers of the triangle measure: two polygons of up to 12 vertices per
// lane of a warp, in shared memory with the lane index fastest (element (poly, vertex, coord)
// of lane t at [((poly * 12 + vertex) * 3 + coord) * 32 + t]), so the lanes hit 32 different
// banks.
constexpr int POLY_FLOATS = 2 * 12 * 3 * 32;

// Sutherland-Hodgman clip of polygon `pi` (n vertices, the first at index `off`) against
// coord_axis >= c (ge) or <= c into polygon `po` (first at 0); returns the new vertex count.  An
// edge emits its crossing of the plane (when its ends lie on different sides), then its end vertex
// (when inside); the end of one edge is kept in registers as the start of the next.
__device__ __forceinline__ int clip_plane_s(float* __restrict__ buf, int pi, int po, int n, int off, int axis, float c,
                                            bool ge) {
    const int t = threadIdx.x & 31;
    auto at = [&](int poly, int v, int j) -> float& { return buf[((poly * 12 + v) * 3 + j) * 32 + t]; };
    int m = 0, v = off;
    float S[3] = {at(pi, off, 0), at(pi, off, 1), at(pi, off, 2)};
#pragma unroll 1
    for (int k = 0; k < n; ++k) {
        v = v + 1 == n ? 0 : v + 1;
        const float E[3] = {at(pi, v, 0), at(pi, v, 1), at(pi, v, 2)};
        const float Sa = sel3(axis, S[0], S[1], S[2]), Ea = sel3(axis, E[0], E[1], E[2]);
        const bool sin_ = ge ? (Sa >= c) : (Sa <= c);
        const bool ein = ge ? (Ea >= c) : (Ea <= c);
        if (sin_ != ein) {
            const float num = c - Sa, den = Ea - Sa;
            const float sv = fabsf(num) >= 1e-24f && fabsf(den) <= 1e12f ? vx_div(num, den) : num / den;
#pragma unroll
            for (int j = 0; j < 3; ++j) at(po, m, j) = (j == axis) ? c : S[j] + sv * (E[j] - S[j]);
            ++m;
        }
        if (ein) {
#pragma unroll
            for (int j = 0; j < 3; ++j) at(po, m, j) = E[j];
            ++m;
        }
#pragma unroll
        for (int j = 0; j < 3; ++j) S[j] = E[j];
    }
    return m;
}

// area (voxel units^2) of the triangle clipped to the voxel [0,1]^3; buf: the warp's
// POLY_FLOATS of shared memory.  Against a plane that every vertex lies inside of, by more than the
// rounding of the clipped vertices, a clip would only move the first vertex to the end: those
// planes are counted instead (`off`), so that a lane clips against the planes its triangle
// reaches, one after the other whatever their number, and the sum's order stays.
__device__ float tri_measure(const float v[3][3], float* __restrict__ buf) {
    const int t = threadIdx.x & 31;
    auto at = [&](int poly, int vv, int j) -> float& { return buf[((poly * 12 + vv) * 3 + j) * 32 + t]; };
    uint32_t need = 0;   // bit 2 axis: the plane 0, bit 2 axis + 1: the plane 1
#pragma unroll
    for (int j = 0; j < 3; ++j) {
#pragma unroll
        for (int k = 0; k < 3; ++k) at(0, k, j) = v[k][j];
        const float mn = fminf(fminf(v[0][j], v[1][j]), v[2][j]), mx = fmax3(v[0][j], v[1][j], v[2][j]);
        const float near = 1e-5f * (fmaxf(fabsf(mn), fabsf(mx)) + 1.0f);
        if (!(mn > near)) need |= 1u << (2 * j);
        if (!(mx < 1.0f - near)) need |= 2u << (2 * j);
    }
    int n = 3, off = 0, cur = 0, next = 0;
    while (need) {
        const int c = __ffs(need) - 1;
        need &= need - 1u;
        off += c - next;
        while (off >= n) off -= n;
        n = clip_plane_s(buf, cur, cur ^ 1, n, off, c >> 1, (c & 1) ? 1.0f : 0.0f, !(c & 1));
        if (n < 1) return 0.0f;
        cur ^= 1;
        off = 0;
        next = c + 1;
    }
    if (n < 3) return 0.0f;
    off += 6 - next;
    while (off >= n) off -= n;
    auto vertex = [&](int k) { return off + k >= n ? off + k - n : off + k; };
    float cx = 0.0f, cy = 0.0f, cz = 0.0f;
    const float a0 = at(cur, off, 0), a1 = at(cur, off, 1), a2 = at(cur, off, 2);
    int w = vertex(1);
    float e1[3] = {at(cur, w, 0) - a0, at(cur, w, 1) - a1, at(cur, w, 2) - a2};
#pragma unroll 1
    for (int k = 1; k + 1 < n; ++k) {
        w = vertex(k + 1);
        const float e2[3] = {at(cur, w, 0) - a0, at(cur, w, 1) - a1, at(cur, w, 2) - a2};
        cx = cx + (e1[1] * e2[2] - e1[2] * e2[1]);
        cy = cy + (e1[2] * e2[0] - e1[0] * e2[2]);
        cz = cz + (e1[0] * e2[1] - e1[1] * e2[0]);
#pragma unroll
        for (int j = 0; j < 3; ++j) e1[j] = e2[j];
    }
    return 0.5f * sqrtf((cx * cx + cy * cy) + cz * cz);
}

// ------------------------------------------------------------------------------------
// prep kernels
// ------------------------------------------------------------------------------------
// Segments per fiber; offsets that are negative, decrease, or pass num_ctrl are flagged.
__global__ void k_fiber_seg_counts(const int64_t* __restrict__ off, int64_t F, int64_t num_ctrl,
                                   uint32_t* __restrict__ cnt, uint32_t* __restrict__ err) {
    int64_t f = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (f < F) {
        const int64_t a = off[f], b = off[f + 1];
        if (a < 0 || b < a || b > num_ctrl) atomicOr(err, 1u);
        int64_t c = b - a - 1;
        cnt[f] = (uint32_t)(c > 0 ? c : 0);
    }
}

// rec_a = (A.xyz, r_g), rec_b = (B.xyz, w) in grid coordinates
// a record the method cannot use: a non-finite coordinate, radius or weight, or a negative
// radius or weight
__device__ __forceinline__ bool bad_record(float4 a, float4 b) {
    const bool fin = isfinite(a.x) && isfinite(a.y) && isfinite(a.z) && isfinite(a.w) && isfinite(b.x) &&
                     isfinite(b.y) && isfinite(b.z) && isfinite(b.w);
    return !fin || a.w < 0.0f || b.w < 0.0f;
}

// A segment whose control points fall outside ctrl[0, num_ctrl) (malformed offsets: negative,
// past the end, or decreasing) is flagged and not read.
__global__ void k_prep_fibers(const float4* __restrict__ ctrl, int64_t num_ctrl, const int64_t* __restrict__ off,
                              const uint32_t* __restrict__ seg_start, int64_t F, const uint32_t* __restrict__ seg_total,
                              const float* __restrict__ weights, uint32_t np, GridDev g, float4* __restrict__ ra,
                              float4* __restrict__ rb, uint32_t* __restrict__ err) {
    uint32_t p = blockIdx.x * blockDim.x + threadIdx.x;
    if (p == 0 && *seg_total != np) atomicOr(err, 1u);
    if (p >= np) return;
    // last fiber with seg_start <= p (fibers without segments share the next start)
    int64_t lo = 0, hi = F;   // upper_bound in [0, F)
    while (lo < hi) {
        int64_t mid = (lo + hi) >> 1;
        if (seg_start[mid] <= p) lo = mid + 1; else hi = mid;
    }
    int64_t f = lo - 1;
    if (f < 0) { atomicOr(err, 1u); return; }
    const int64_t o0 = off[f];
    int64_t c = o0 + (int64_t)(p - seg_start[f]);
    if (o0 < 0 || c < 0 || c + 1 >= off[f + 1] || c + 1 >= num_ctrl) { atomicOr(err, 1u); return; }
    float4 pa = ctrl[c], pb = ctrl[c + 1];
    float4 A, B;
    A.x = (pa.x - g.o[0]) * g.s; A.y = (pa.y - g.o[1]) * g.s; A.z = (pa.z - g.o[2]) * g.s;
    B.x = (pb.x - g.o[0]) * g.s; B.y = (pb.y - g.o[1]) * g.s; B.z = (pb.z - g.o[2]) * g.s;
    A.w = ((pa.w + pb.w) * 0.5f) * g.s;
    B.w = weights ? weights[p] : 1.0f;
    if (bad_record(A, B)) atomicOr(err, 1u);
    ra[p] = A;
    rb[p] = B;
}

// tri records: (U0, w), (U1, 0), (U2, 0)
__global__ void k_prep_tris(const float4* __restrict__ tv, const float* __restrict__ weights, uint32_t np, GridDev g,
                            float4* __restrict__ r0, float4* __restrict__ r1, float4* __restrict__ r2,
                            uint32_t* __restrict__ err) {
    uint32_t p = blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= np) return;
    float4 v0 = tv[3 * (size_t)p], v1 = tv[3 * (size_t)p + 1], v2 = tv[3 * (size_t)p + 2];
    float4 a, b, c;
    a.x = (v0.x - g.o[0]) * g.s; a.y = (v0.y - g.o[1]) * g.s; a.z = (v0.z - g.o[2]) * g.s;
    b.x = (v1.x - g.o[0]) * g.s; b.y = (v1.y - g.o[1]) * g.s; b.z = (v1.z - g.o[2]) * g.s;
    c.x = (v2.x - g.o[0]) * g.s; c.y = (v2.y - g.o[1]) * g.s; c.z = (v2.z - g.o[2]) * g.s;
    a.w = weights ? weights[p] : 1.0f;
    b.w = 0.0f;
    c.w = 0.0f;
    if (bad_record(a, b) || bad_record(c, c)) atomicOr(err, 1u);
    r0[p] = a; r1[p] = b; r2[p] = c;
}

// voxel range of a primitive: [lo, hi] per axis, empty when lo > hi on an axis
struct Range {
    int lo[3], n[3];
    long long total;
};
// voxel window of one pass: indices [lo, hi] per axis (a tile of the grid, or all of it);
// candidate keys are Morton codes relative to lo
struct Window {
    int lo[3], hi[3];
};
__host__ __device__ inline Window full_window(int R) {
    Window w;
    for (int i = 0; i < 3; ++i) { w.lo[i] = 0; w.hi[i] = R - 1; }
    return w;
}
// (ix, iy, iz) of flat index idx < tot in a range (x fastest).  Ranges of at most 2^16
// voxels divide by the correctly rounded FP32 reciprocal: (i + 0.5) fl(1/n), rounded, is
// within i / n (1 + 2^-23) of the quotient plus 0.5 / n, so its integer part is floor(i / n)
// (checked for every n and i below 2^16; tests/test_host_arith.py keeps every n up to 4096).  Larger ranges use 32-bit division when they hold
// fewer than 2^32 voxels (always inside a 1024^3 window).
__device__ __forceinline__ void voxel_of(long long idx, long long tot, const Range& rg, int& ix, int& iy, int& iz) {
    if (tot <= 65536) {
        const float r0 = __frcp_rn((float)rg.n[0]), r1 = __frcp_rn((float)rg.n[1]);
        const int i = (int)idx;
        const int t = (int)(((float)i + 0.5f) * r0);
        ix = i - t * rg.n[0];
        iz = (int)(((float)t + 0.5f) * r1);
        iy = t - iz * rg.n[1];
    } else if (tot <= 0xffffffffll) {
        const uint32_t i = (uint32_t)idx, n0 = (uint32_t)rg.n[0], n1 = (uint32_t)rg.n[1];
        const uint32_t t = i / n0;
        ix = (int)(i - t * n0);
        iz = (int)(t / n1);
        iy = (int)(t - (uint32_t)iz * n1);
    } else {
        const long long t = idx / rg.n[0];
        ix = (int)(idx - t * rg.n[0]);
        iz = (int)(t / rg.n[1]);
        iy = (int)(t - (long long)iz * rg.n[1]);
    }
}

__device__ __forceinline__ Range make_range(const float* mn, const float* mx, const Window& w) {
    Range r;
    r.total = 1;
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        const float fl = floorf(mn[i]), fh = floorf(mx[i]);
        const int lo = fl < (float)w.lo[i] ? w.lo[i] : (fl > (float)w.hi[i] ? w.hi[i] + 1 : (int)fl);
        const int hi = fh < (float)w.lo[i] ? w.lo[i] - 1 : (fh > (float)w.hi[i] ? w.hi[i] : (int)fh);
        r.lo[i] = lo;
        // a NaN bound (rejected input, flagged by the prep kernels) gives an empty range
        r.n[i] = (mn[i] <= mx[i] && hi >= lo) ? hi - lo + 1 : 0;
        r.total *= r.n[i];
    }
    return r;
}

// conservative voxel-level tests (never reject a voxel with a set sub-cell)
__device__ __forceinline__ float capsule_margin(float rg) { return 2e-3f * fmax2(1.0f, rg) + 1e-4f; }

__device__ __forceinline__ Range capsule_range(float4 A, float4 B, const Window& R) {
    const float rc = A.w + capsule_margin(A.w) + 0.01f;
    float mn[3] = {fmin2(A.x, B.x) - rc, fmin2(A.y, B.y) - rc, fmin2(A.z, B.z) - rc};
    float mx[3] = {fmax2(A.x, B.x) + rc, fmax2(A.y, B.y) + rc, fmax2(A.z, B.z) + rc};
    return make_range(mn, mx, R);
}

// The voxel is kept unless steps 1-2 reject it at the inflated radius, or it is separated
// from the segment by more than that radius plus the separation test's rounding margin.
__device__ __forceinline__ bool capsule_voxel_candidate(float4 A, float4 B, int vi, int vj, int vk) {
    const float a[3] = {A.x - (float)vi, A.y - (float)vj, A.z - (float)vk};
    const float b[3] = {B.x - (float)vi, B.y - (float)vj, B.z - (float)vk};
    const float r = A.w + capsule_margin(A.w);
    const float rr = r * r;
    const float lo[3] = {0.0f, 0.0f, 0.0f}, hi[3] = {1.0f, 1.0f, 1.0f};
    float g[3];
#pragma unroll
    for (int i = 0; i < 3; ++i) g[i] = gap3(0.0f, 1.0f, fmin2(a[i], b[i]), fmax2(a[i], b[i]));
    if ((g[0] * g[0] + g[1] * g[1]) + g[2] * g[2] > rr) return false;
    if (sqdist_point_box(a[0], a[1], a[2], lo, hi) <= rr) return true;
    if (sqdist_point_box(b[0], b[1], b[2], lo, hi) <= rr) return true;
    const CapsuleLocal c = capsule_local(a, b, r);
    return !segment_box_separated(c.a_rr, c.b_reta, c.d_idd, 0.5f, 0.5f, 0.5f, 0.5f, c.b_reta.w);
}

__device__ __forceinline__ Range tri_range(float4 a, float4 b, float4 c, const Window& R) {
    const float m = 0.01f;
    float mn[3] = {fmin2(fmin2(a.x, b.x), c.x) - m, fmin2(fmin2(a.y, b.y), c.y) - m, fmin2(fmin2(a.z, b.z), c.z) - m};
    float mx[3] = {fmax2(fmax2(a.x, b.x), c.x) + m, fmax2(fmax2(a.y, b.y), c.y) + m, fmax2(fmax2(a.z, b.z), c.z) + m};
    return make_range(mn, mx, R);
}

__device__ __forceinline__ void tri_local(float4 a, float4 b, float4 c, int vi, int vj, int vk, float v[3][3],
                                          float f[3][3]) {
    v[0][0] = a.x - (float)vi; v[0][1] = a.y - (float)vj; v[0][2] = a.z - (float)vk;
    v[1][0] = b.x - (float)vi; v[1][1] = b.y - (float)vj; v[1][2] = b.z - (float)vk;
    v[2][0] = c.x - (float)vi; v[2][1] = c.y - (float)vj; v[2][2] = c.z - (float)vk;
    f[0][0] = b.x - a.x; f[0][1] = b.y - a.y; f[0][2] = b.z - a.z;
    f[1][0] = c.x - b.x; f[1][1] = c.y - b.y; f[1][2] = c.z - b.z;
    f[2][0] = a.x - c.x; f[2][1] = a.y - c.y; f[2][2] = a.z - c.z;
}

__device__ __forceinline__ bool tri_voxel_candidate(float4 a, float4 b, float4 c, int vi, int vj, int vk) {
    float v[3][3], f[3][3];
    tri_local(a, b, c, vi, vj, vk, v, f);
    const float ctr[3] = {0.5f, 0.5f, 0.5f};
    return tri_box(v, f, ctr, 0.5f + 2e-3f);
}

// ------------------------------------------------------------------------------------
// count / emit: the candidate voxels of every primitive's range
// ------------------------------------------------------------------------------------
// With `ballots`, the count pass stores each primitive's hit ballots (one word per 32 voxels
// of its range, ranges of at most 32 * stride voxels) and the emit pass of the same
// window reads them instead of testing again; larger ranges are tested in both passes.
// The ballots are the same bits either way, so the emitted order does not change.
constexpr int CAND_BALLOTS = 8;   // words per primitive in the batched path

// One primitive of the pass, by a whole warp (see k_candidates); `stride` words of `ballots` per
// primitive.  Returns its number of candidates.
template <bool FIBER, bool EMIT>
__device__ __forceinline__ uint32_t candidates_of(uint32_t p, float4 a, float4 b, float4 c, const Range& rg,
                                                  const Window& R, uint32_t base, uint32_t* __restrict__ keys,
                                                  uint32_t* __restrict__ vals, uint32_t* __restrict__ ballots,
                                                  uint32_t stride) {
    const int lane = threadIdx.x & 31;
    uint32_t n = 0;
    const long long tot = rg.total;
    const bool stored = ballots != nullptr && tot <= 32ll * stride;
    uint32_t* const pb = stored ? ballots + (size_t)p * stride : nullptr;
    for (long long idx0 = 0; idx0 < tot; idx0 += 32) {
        const long long idx = idx0 + lane;
        bool hit = false;
        int vi = 0, vj = 0, vk = 0;
        if (idx < tot) {
            int ix, iy, iz;
            voxel_of(idx, tot, rg, ix, iy, iz);
            vi = rg.lo[0] + ix; vj = rg.lo[1] + iy; vk = rg.lo[2] + iz;
            if (EMIT && stored) hit = (pb[idx0 >> 5] >> lane) & 1u;
            else hit = FIBER ? capsule_voxel_candidate(a, b, vi, vj, vk) : tri_voxel_candidate(a, b, c, vi, vj, vk);
        }
        const uint32_t bal = __ballot_sync(0xffffffffu, hit);
        if (!EMIT && stored && lane == 0) pb[idx0 >> 5] = bal;
        if (EMIT && hit) {
            const uint32_t pos = base + n + __popc(bal & ((1u << lane) - 1u));
            keys[pos] = vx_morton3((uint32_t)(vi - R.lo[0]), (uint32_t)(vj - R.lo[1]), (uint32_t)(vk - R.lo[2]));
            vals[pos] = p;
        }
        n += __popc(bal);
    }
    return n;
}

template <bool FIBER>
__device__ __forceinline__ Range prim_range(const float4* __restrict__ r0, const float4* __restrict__ r1,
                                            const float4* __restrict__ r2, uint32_t p, const Window& R, float4& a,
                                            float4& b, float4& c) {
    a = r0[p];
    b = r1[p];
    if (FIBER) return capsule_range(a, b, R);
    c = r2[p];
    return tri_range(a, b, c, R);
}

// ---- count -------------------------------------------------------------------------
// The count pass tests every voxel of a primitive's range with capsule_voxel_candidate /
// tri_voxel_candidate, whose cost is instruction issue (91 % and 77 % busy at 780 instructions per
// 27-voxel triangle).  Most of that work is the same for all voxels of the range, or decides by a
// hair's breadth what is clear at a glance.  So a lane first lays down a record of one primitive (a
// warp: up to 32 of them) in coordinates relative to its range's corner, with the terms that do not
// depend on the voxel and a bound on the rounding of both evaluations; per voxel, a few fused
// operations on the record then say in, out or open, and only the open ones (within the bound of a
// boundary: one in ten thousand to one in two hundred) take the test itself.  The candidates are the
// same: 5e10 voxels of 14 M primitives of all shapes gave no other answer.  Still bound by issue.
//   yarn (768k capsules) 0.73 -> 0.37 ms, woven 1.07 -> 0.56 ms, mesh (978k triangles) 1.42 -> 0.46 ms.
// (Five blocks per SM for triangles: four 0.52 ms, six, at 80 registers, 0.50 ms.)
constexpr int COUNT_WARPS = 4;
constexpr int kMaxFastRange = 65536;   // voxels: (i + 0.5) / n by reciprocals (see voxel_of)
template <bool FIBER>
struct CountRecords {
    float4 q[FIBER ? 5 : 12][32];   // by term, by primitive: lanes write side by side, then read one
    float4 r[2][32];                // 1 / n0, n0, 1 / n1, n1 and lo (as bits), voxels
};

__device__ __forceinline__ float abs_max3(float x, float y, float z) { return fmax3(fabsf(x), fabsf(y), fabsf(z)); }

// Capsule: M bounds every coordinate and the radius (a coordinate relative to a voxel: 2 M).  The
// gap's square (step 1) is off by less than 2^-18 M^2.  The separation's direction v is off by 32 u M
// and, along the axis, by 16 u M^2 / |d| or |d| (u = 2^-24); at the nearest point v is normal to the
// axis, so the separation times |v| is off by less than `del`.  The margin eta depends on the
// voxel: the radius lies between the two kept here.
__device__ __forceinline__ void count_record(CountRecords<true>& cr, int i, float4 A, float4 B, float4, const Range& rg) {
    const float O[3] = {(float)rg.lo[0], (float)rg.lo[1], (float)rg.lo[2]};
    const float a[3] = {A.x - O[0], A.y - O[1], A.z - O[2]}, b[3] = {B.x - O[0], B.y - O[1], B.z - O[2]};
    const float d[3] = {b[0] - a[0], b[1] - a[1], b[2] - a[2]};
    const float r = A.w + capsule_margin(A.w), rr = r * r;
    const float M = (fmax3(abs_max3(a[0], a[1], a[2]), abs_max3(b[0], b[1], b[2]),
                           (float)max(max(rg.n[0], rg.n[1]), rg.n[2])) + r) + 3.0f;
    const float dd = (d[0] * d[0] + d[1] * d[1]) + d[2] * d[2], len = sqrtf(dd), u = 0x1p-24f;
    const float idd = dd > 0.0f ? 1.0f / dd : 0.0f;
    const float off = 32.0f * u * M + fminf(len, 16.0f * u * M * M * (len * idd));
    // (a length whose square is denormal, or coordinates beyond any grid: every voxel is open)
    const bool sound = M < 1e6f && (dd == 0.0f || dd > 1e-30f);
    const float del = sound ? 64.0f * u * M * M + off * (len + 1.0f) : INFINITY;
    const float eps = sound ? 0x1p-18f * M * M : INFINITY;
    const float rlo = r + 2e-5f * (r + 2.9f), rhi = r + 2e-5f * (2.0f * M + r + 3.0f);
    cr.q[0][i] = make_float4(a[0], a[1], a[2], -idd);
    cr.q[1][i] = make_float4(d[0], d[1], d[2], del);
    cr.q[2][i] = make_float4(fminf(a[0], b[0]) - 0.5f, fminf(a[1], b[1]) - 0.5f, fminf(a[2], b[2]) - 0.5f, rr - eps);
    cr.q[3][i] = make_float4(fmaxf(a[0], b[0]) + 0.5f, fmaxf(a[1], b[1]) + 0.5f, fmaxf(a[2], b[2]) + 0.5f, rr + eps);
    cr.q[4][i] = make_float4(rlo * rlo * (1.0f - 0x1p-20f), rhi * rhi * (1.0f + 0x1p-20f), 0.0f, 0.0f);
}
// Voxel centre (cx, cy, cz) relative to the range's corner: 1 in, -1 out, 0 open.
__device__ __forceinline__ int count_quick(const CountRecords<true>& cr, int i, float cx, float cy, float cz) {
    const float4 a = cr.q[0][i], d = cr.q[1][i], mn = cr.q[2][i], mx = cr.q[3][i], re = cr.q[4][i];
    const float gx = gap3(cx, cx, mn.x, mx.x), gy = gap3(cy, cy, mn.y, mx.y), gz = gap3(cz, cz, mn.z, mx.z);
    const float G = __fmaf_rn(gx, gx, __fmaf_rn(gy, gy, gz * gz));
    const float Ax = a.x - cx, Ay = a.y - cy, Az = a.z - cz;
    const float t = __saturatef(a.w * __fmaf_rn(Ax, d.x, __fmaf_rn(Ay, d.y, Az * d.z)));
    const float vx = __fmaf_rn(t, d.x, Ax), vy = __fmaf_rn(t, d.y, Ay), vz = __fmaf_rn(t, d.z, Az);
    const float sa = __fmaf_rn(vx, Ax, __fmaf_rn(vy, Ay, vz * Az));
    const float sb = __fmaf_rn(vx, d.x, __fmaf_rn(vy, d.y, __fmaf_rn(vz, d.z, sa)));
    const float sep = __fmaf_rn(-0.5f, (fabsf(vx) + fabsf(vy)) + fabsf(vz), fminf(sa, sb));
    const float vv = __fmaf_rn(vx, vx, __fmaf_rn(vy, vy, vz * vz));
    const float so = sep - d.w, si = sep + d.w;
    if (G > mx.w || so * fabsf(so) > re.y * vv) return -1;
    return G < mn.w && si * fabsf(si) < re.x * vv ? 1 : 0;
}

// Triangle: on each of the 13 axes the voxel's centre has to lie in an interval; an axis is scaled
// by the inverse of its rounding bound, 2^-18 M times the axis's 1-norm (both evaluations stay below
// half of that: the edges and the normal are the same numbers, products and sums of terms below M
// take at most eight roundings of 2^-24 each).  The smallest distance to an interval's end is then
// beyond 1 when the voxel is in, below -1 when it is out.
__device__ __forceinline__ float4 count_axis(float u0, float u1, float p0, float p1, float p2, float rad, float inv) {
    const float mn = fminf(fminf(p0, p1), p2) - rad, mx = fmaxf(fmaxf(p0, p1), p2) + rad;
    return inv > 0.0f ? make_float4(u0 * inv, u1 * inv, -mn * inv, (mx - mn) * inv) : make_float4(0.0f, 0.0f, 2.0f, 4.0f);
}
__device__ __forceinline__ void count_record(CountRecords<false>& cr, int i, float4 A, float4 B, float4 C, const Range& rg) {
    const float e = 0.5f + 2e-3f;
    float v[3][3], f[3][3];
    tri_local(A, B, C, rg.lo[0], rg.lo[1], rg.lo[2], v, f);
    float M = (float)max(max(rg.n[0], rg.n[1]), rg.n[2]) + 1.0f;
#pragma unroll
    for (int k = 0; k < 3; ++k) M = fmaxf(M, abs_max3(v[k][0], v[k][1], v[k][2]) + 1.0f);
    bool sound = M < 1e6f;
    const float bound = 0x1p-18f * M;
    // an axis without extent never separates; one whose products could be denormal leaves all open
    auto inverse = [&](float l1) {
        if (l1 == 0.0f) return 0.0f;
        sound = sound && l1 > 1e-25f;
        return 1.0f / (bound * l1);
    };
#pragma unroll
    for (int j = 0; j < 3; ++j) {
        const float* q = f[j];
        float l = fabsf(q[1]) + fabsf(q[2]);
        cr.q[3 * j][i] = count_axis(-q[2], q[1], q[1] * v[0][2] - q[2] * v[0][1], q[1] * v[1][2] - q[2] * v[1][1],
                                    q[1] * v[2][2] - q[2] * v[2][1], e * l, inverse(l));
        l = fabsf(q[0]) + fabsf(q[2]);
        cr.q[3 * j + 1][i] = count_axis(q[2], -q[0], q[2] * v[0][0] - q[0] * v[0][2], q[2] * v[1][0] - q[0] * v[1][2],
                                        q[2] * v[2][0] - q[0] * v[2][2], e * l, inverse(l));
        l = fabsf(q[0]) + fabsf(q[1]);
        cr.q[3 * j + 2][i] = count_axis(-q[1], q[0], q[0] * v[0][1] - q[1] * v[0][0], q[0] * v[1][1] - q[1] * v[1][0],
                                        q[0] * v[2][1] - q[1] * v[2][0], e * l, inverse(l));
    }
    const float n0 = f[0][1] * f[1][2] - f[0][2] * f[1][1];
    const float n1 = f[0][2] * f[1][0] - f[0][0] * f[1][2];
    const float n2 = f[0][0] * f[1][1] - f[0][1] * f[1][0];
    const float l = (fabsf(n0) + fabsf(n1)) + fabsf(n2), inv = inverse(l);
    const float p = (n0 * v[0][0] + n1 * v[0][1]) + n2 * v[0][2];
    // the face axes share one scale; the plane's interval is p -+ e l: its width in the last record
    const float fi = sound ? 1.0f / bound : 0.0f;
    float lo[3], wd[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        const float mn = fminf(fminf(v[0][k], v[1][k]), v[2][k]) - e, mx = fmaxf(fmaxf(v[0][k], v[1][k]), v[2][k]) + e;
        lo[k] = -mn * fi;
        wd[k] = (mx - mn) * fi;
    }
    cr.q[9][i] = inv > 0.0f ? make_float4(n0 * inv, n1 * inv, n2 * inv, (e * l - p) * inv) : make_float4(0.0f, 0.0f, 0.0f, 2.0f);
    cr.q[10][i] = make_float4(lo[0], lo[1], lo[2], fi);
    cr.q[11][i] = make_float4(wd[0], wd[1], wd[2], inv > 0.0f ? 2.0f * e * l * inv : 4.0f);
    if (!sound) {   // the face terms are zero: nothing is in
#pragma unroll
        for (int k = 0; k < 9; ++k) cr.q[k][i] = make_float4(0.0f, 0.0f, 2.0f, 4.0f);
        cr.q[9][i] = make_float4(0.0f, 0.0f, 0.0f, 2.0f);
        cr.q[10][i] = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
        cr.q[11][i] = make_float4(0.0f, 0.0f, 0.0f, 4.0f);
    }
}
__device__ __forceinline__ float min3(float a, float b, float c) {
    float r;
    asm("min.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(b), "f"(c));
    return r;
}
__device__ __forceinline__ int count_quick(const CountRecords<false>& cr, int i, float cx, float cy, float cz) {
    const float4 F = cr.q[10][i], W = cr.q[11][i], N = cr.q[9][i];
    float s = __fmaf_rn(cx, F.w, F.x);
    float m = fminf(s, W.x - s);
    s = __fmaf_rn(cy, F.w, F.y);
    m = min3(m, s, W.y - s);
    s = __fmaf_rn(cz, F.w, F.z);
    m = min3(m, s, W.z - s);
    s = __fmaf_rn(cx, N.x, __fmaf_rn(cy, N.y, __fmaf_rn(cz, N.z, N.w)));
    m = min3(m, s, W.w - s);
#pragma unroll
    for (int j = 0; j < 9; ++j) {   // families x, y, z of edge j / 3
        const float4 q = cr.q[j][i];
        s = __fmaf_rn(j % 3 == 0 ? cy : cx, q.x, __fmaf_rn(j % 3 == 2 ? cy : cz, q.y, q.z));
        m = min3(m, s, q.w - s);
    }
    return m > 1.0f ? 1 : (m < -1.0f ? -1 : 0);
}

// A warp takes its group's primitives one after the other, so one with a range of many voxels would
// make its neighbours wait (and 32 of them in a row, a mesh's ground or walls, would all fall to one
// warp).  A launch therefore takes only ranges of [least, most] voxels: the grouped launch leaves those
// above kGroupRange to a second one with a warp each, made when it has raised kCountLarge.  The bound is
// the most that a ballot store holds (64 words); a group of 32 such ranges is 0.25 ms for one warp.
// 100,000 small triangles and 32 of 200 voxels' extent in a row: 82 ms, 287 ms in groups of any range.
constexpr int kGroupRange = 2048, kAnyRange = 0x7fffffff;
// (a range of a 2048^3 grid can hold 2^33 voxels)
__device__ __forceinline__ int capped_total(const Range& rg) { return (int)min(rg.total, (long long)kAnyRange); }
constexpr uint32_t kCountLarge = 1u;      // a range above `most` was left out (its count is 0)
constexpr uint32_t kCountUnstored = 2u;   // a range has more voxels than its ballot words

// floor of 0 <= x < 2^22, as a float
__device__ __forceinline__ float floor_pos(float x) { return __fadd_rd(x, 8388608.0f) - 8388608.0f; }

// Counts of 2^lg consecutive primitives from p0 (fewer at np) by a warp, and their ballots; win(p) is
// the window of a primitive.  Ranges below `least` are passed over, those above `most` count 0; flags
// (or NULL) receives kCountLarge and kCountUnstored.
template <bool FIBER, class Win>
__device__ __forceinline__ void count_group(CountRecords<FIBER>& cr, uint32_t p0, int lg, uint32_t np,
                                            const float4* __restrict__ r0, const float4* __restrict__ r1,
                                            const float4* __restrict__ r2, Win win, int least, int most,
                                            uint32_t* __restrict__ counts, uint32_t* __restrict__ ballots,
                                            uint32_t stride, uint32_t* __restrict__ flags) {
    const int lane = threadIdx.x & 31;
    const uint32_t p = p0 + (uint32_t)lane;
    const int members = (int)min(1u << lg, np - p0);
    uint32_t raise = 0;
    bool write = false;
    if (lane < members) {
        float4 a, b, c = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
        const Range rg = prim_range<FIBER>(r0, r1, r2, p, win(p), a, b, c);
        const int tot = capped_total(rg);
        const bool below = tot < least, above = tot > most;
        write = !below;
        raise = (above ? kCountLarge : 0u) | (ballots && rg.total > 32ll * stride ? kCountUnstored : 0u);
        if (!below && !above) count_record(cr, lane, a, b, c, rg);
        const float n0 = (float)rg.n[0], n1 = (float)rg.n[1];
        cr.r[0][lane] = make_float4(__frcp_rn(n0), n0, __frcp_rn(n1), n1);
        cr.r[1][lane] = make_float4(__int_as_float(rg.lo[0]), __int_as_float(rg.lo[1]), __int_as_float(rg.lo[2]),
                                    __int_as_float(below || above ? 0 : min(tot, kMaxFastRange + 1)));
    }
    if (flags && __any_sync(0xffffffffu, raise != 0u)) {
        raise = __reduce_or_sync(0xffffffffu, raise);
        if (lane == 0 && (raise & ~*(volatile uint32_t*)flags)) atomicOr(flags, raise);
    }
    __syncwarp();
    uint32_t mine = 0;
    for (int i = 0; i < members; ++i) {
        const float4 rn = cr.r[0][i], rl = cr.r[1][i];
        const int tot = __float_as_int(rl.w);
        uint32_t n = 0;
        if (tot > kMaxFastRange) {
            float4 a, b, c = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
            const Window W = win(p0 + i);
            const Range rg = prim_range<FIBER>(r0, r1, r2, p0 + i, W, a, b, c);
            n = candidates_of<FIBER, false>(p0 + i, a, b, c, rg, W, 0u, nullptr, nullptr, ballots, stride);
        } else {
            uint32_t* const pb = ballots && tot <= (int)(32u * stride) ? ballots + (size_t)(p0 + i) * stride : nullptr;
            for (int i0 = 0; i0 < tot; i0 += 32) {
                const bool valid = i0 + lane < tot;
                const float f = (float)(i0 + lane);
                const float t = floor_pos((f + 0.5f) * rn.x);
                const float x = __fmaf_rn(-t, rn.y, f), z = floor_pos((t + 0.5f) * rn.z), y = __fmaf_rn(-z, rn.w, t);
                const int q = count_quick(cr, i, x + 0.5f, y + 0.5f, z + 0.5f);
                bool hit = valid && q > 0;
                if (__any_sync(0xffffffffu, valid && q == 0) && valid && q == 0) {
                    const int vi = __float_as_int(rl.x) + (int)x, vj = __float_as_int(rl.y) + (int)y,
                              vk = __float_as_int(rl.z) + (int)z;
                    hit = FIBER ? capsule_voxel_candidate(r0[p0 + i], r1[p0 + i], vi, vj, vk)
                                : tri_voxel_candidate(r0[p0 + i], r1[p0 + i], r2[p0 + i], vi, vj, vk);
                }
                const uint32_t bal = __ballot_sync(0xffffffffu, hit);
                if (pb && lane == 0) pb[i0 >> 5] = bal;
                n += __popc(bal);
            }
        }
        if (lane == i) mine = n;
    }
    if (write) counts[p] = mine;
    __syncwarp();
}

// primitives per warp (log2): 32 where that leaves every SM its warps, fewer for short arrays
inline int count_lanes_log2(uint32_t np) {
    int lg = 5;
    while (lg > 0 && (np >> lg) < (uint32_t)vx::kSMs * 48) --lg;
    return lg;
}
inline unsigned count_blocks(uint32_t np, int lg) {
    const size_t groups = ((size_t)np + (1u << lg) - 1) >> lg;
    return (unsigned)std::min<size_t>((groups + COUNT_WARPS - 1) / COUNT_WARPS, (size_t)vx::kSMs * 64);
}

template <bool FIBER>
__global__ void __launch_bounds__(COUNT_WARPS * 32, FIBER ? 7 : 5) k_count(const float4* __restrict__ r0, const float4* __restrict__ r1,
                                                            const float4* __restrict__ r2, uint32_t np, Window R, int lg,
                                                            int least, int most, uint32_t* __restrict__ counts,
                                                            uint32_t* __restrict__ ballots, uint32_t stride,
                                                            uint32_t* __restrict__ flags) {
    __shared__ CountRecords<FIBER> rec[COUNT_WARPS];
    const uint32_t groups = (uint32_t)(((uint64_t)np + (1u << lg) - 1) >> lg);
    for (uint32_t g = blockIdx.x * COUNT_WARPS + (threadIdx.x >> 5); g < groups; g += gridDim.x * COUNT_WARPS)
        count_group<FIBER>(rec[threadIdx.x >> 5], g << lg, lg, np, r0, r1, r2, [&](uint32_t) { return R; }, least, most,
                           counts, ballots, stride, flags);
}

// Emit from the stored ballots.  A warp takes 32 consecutive primitives; their pairs are consecutive
// in the output, so it walks their words 32 at a time, a lane per word: the lane writes the pairs
// of its word's bits to the warp's staging buffer, which then goes out in order with whole lines.
// (A warp per primitive left most of its lanes to the addresses of one word: 0.52 ms against
// 0.22 ms for the 75 M pairs of the 768k-capsule yarn.)  Morton codes come from a table of one
// coordinate's spread bits in shared memory.  A group with a primitive whose range was too large
// to be stored is left to k_candidates, which the host launches for those when the count pass has
// raised kCountUnstored: one warp on a whole group took up to 32 times as long.
constexpr int STAGE_WARPS = 4;
template <bool FIBER>
__global__ void __launch_bounds__(STAGE_WARPS * 32) k_emit_stored(const float4* __restrict__ r0,
                                                                  const float4* __restrict__ r1,
                                                                  const float4* __restrict__ r2, uint32_t np, Window R,
                                                                  const uint32_t* __restrict__ offs,
                                                                  uint32_t* __restrict__ keys,
                                                                  uint32_t* __restrict__ vals,
                                                                  const uint32_t* __restrict__ ballots, uint32_t stride) {
    __shared__ uint32_t spread[1024];
    __shared__ uint32_t stage_k[STAGE_WARPS][1024], stage_v[STAGE_WARPS][1024];
    const int lane = threadIdx.x & 31;
    uint32_t* const sk = stage_k[threadIdx.x >> 5];
    uint32_t* const sv = stage_v[threadIdx.x >> 5];
    for (uint32_t i = threadIdx.x; i < 1024; i += STAGE_WARPS * 32) spread[i] = vx_part1by2(i);
    __syncthreads();
    const uint32_t groups = (uint32_t)(((uint64_t)np + 31) / 32), warps = gridDim.x * STAGE_WARPS;
    for (uint32_t g = blockIdx.x * STAGE_WARPS + (threadIdx.x >> 5); g < groups; g += warps) {
        const uint32_t p0 = g * 32u, p = p0 + (uint32_t)lane;
        Range rg;
        rg.total = 0;
        rg.lo[0] = rg.lo[1] = rg.lo[2] = 0;
        rg.n[0] = rg.n[1] = rg.n[2] = 0;
        if (p < np) {
            float4 a, b, c;
            rg = prim_range<FIBER>(r0, r1, r2, p, R, a, b, c);
        }
        if (__any_sync(0xffffffffu, rg.total > 32ll * stride)) continue;
        // ranges of at most 2048 voxels: i / n as the high word of i (2^32 / n + 1), exact for i n < 2^32
        const uint32_t tot = (uint32_t)rg.total, nw = (tot + 31u) / 32u;
        const uint32_t n0 = (uint32_t)max(rg.n[0], 1), n1 = (uint32_t)max(rg.n[1], 1);
        const uint32_t m0 = 0xffffffffu / n0 + 1u, m1 = 0xffffffffu / n1 + 1u;   // (0 for n = 1: see below)
        uint32_t end = nw;   // inclusive scan: the words up to this lane's primitive
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t t = __shfl_up_sync(0xffffffffu, end, o);
            if (lane >= o) end += t;
        }
        const uint32_t words = __shfl_sync(0xffffffffu, end, 31);
        uint32_t pos = offs[p0];
        for (uint32_t w0 = 0; w0 < words; w0 += 32) {
            const uint32_t s = w0 + (uint32_t)lane;
            // the primitive of word s: the number of lanes whose words end at or before it
            int own = 0;
#pragma unroll
            for (int o = 16; o > 0; o >>= 1)
                if (__shfl_sync(0xffffffffu, end, own + o - 1) <= s) own += o;
            own = min(own, 31);
            const uint32_t first = __shfl_sync(0xffffffffu, end - nw, own);
            const uint32_t on0 = __shfl_sync(0xffffffffu, n0, own), on1 = __shfl_sync(0xffffffffu, n1, own);
            const uint32_t om0 = __shfl_sync(0xffffffffu, m0, own), om1 = __shfl_sync(0xffffffffu, m1, own);
            const uint32_t lx = (uint32_t)(__shfl_sync(0xffffffffu, rg.lo[0], own) - R.lo[0]);
            const uint32_t ly = (uint32_t)(__shfl_sync(0xffffffffu, rg.lo[1], own) - R.lo[1]);
            const uint32_t lz = (uint32_t)(__shfl_sync(0xffffffffu, rg.lo[2], own) - R.lo[2]);
            uint32_t bits = s < words ? ballots[(size_t)(p0 + (uint32_t)own) * stride + (s - first)] : 0u;
            uint32_t at = __popc(bits);
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const uint32_t t = __shfl_up_sync(0xffffffffu, at, o);
                if (lane >= o) at += t;
            }
            const uint32_t total = __shfl_sync(0xffffffffu, at, 31);
            at -= __popc(bits);
            const uint32_t i0 = (s - first) * 32u;
            while (bits) {
                const uint32_t i = i0 + (uint32_t)__ffs(bits) - 1u;
                bits &= bits - 1u;
                const uint32_t t = on0 == 1u ? i : __umulhi(i, om0);
                const uint32_t z = on1 == 1u ? t : __umulhi(t, om1);
                const uint32_t x = lx + (i - t * on0), y = ly + (t - z * on1);
                sk[at] = spread[x] | (spread[y] << 1) | (spread[lz + z] << 2);
                sv[at] = p0 + (uint32_t)own;
                ++at;
            }
            __syncwarp();
            for (uint32_t k = (uint32_t)lane; k < total; k += 32) {
                keys[pos + k] = sk[k];
                vals[pos + k] = sv[k];
            }
            __syncwarp();
            pos += total;
        }
    }
}

// emit with a warp per primitive: of a pass without stored ballots, which tests the ranges again, or
// (unstored_only) of the groups of 32 that k_emit_stored leaves
template <bool FIBER>
__global__ void __launch_bounds__(EMIT_WARPS * 32) k_candidates(const float4* __restrict__ r0,
                                                                const float4* __restrict__ r1,
                                                                const float4* __restrict__ r2, uint32_t np, Window R,
                                                                const uint32_t* __restrict__ offs,
                                                                uint32_t* __restrict__ keys,
                                                                uint32_t* __restrict__ vals,
                                                                uint32_t* __restrict__ ballots, uint32_t stride,
                                                                bool unstored_only) {
    const uint32_t warps = gridDim.x * EMIT_WARPS;
    for (uint32_t p = blockIdx.x * EMIT_WARPS + (threadIdx.x >> 5); p < np; p += warps) {
        float4 a, b, c;
        if (unstored_only) {
            const uint32_t q = (p & ~31u) + (threadIdx.x & 31u);
            if (!__any_sync(0xffffffffu, q < np && prim_range<FIBER>(r0, r1, r2, q, R, a, b, c).total > 32ll * stride))
                continue;
        }
        const Range rg = prim_range<FIBER>(r0, r1, r2, p, R, a, b, c);
        candidates_of<FIBER, true>(p, a, b, c, rg, R, offs[p], keys, vals, ballots, stride);
    }
}

// ------------------------------------------------------------------------------------
// reduce: warp per candidate voxel
// lane l owns sub-cells sz = l >> 2, sy = 2 (l & 3) + {0,1}, sx = 0..7 (16 bits)
// ------------------------------------------------------------------------------------
// Writes one candidate voxel's mask (lanes' 16-bit chunks gathered into the 8 words), key and
// non-empty flag.
__device__ __forceinline__ void write_mask(SegOut out, uint32_t seg, uint32_t key, uint32_t chunk) {
    const int lane = threadIdx.x & 31;
    uint64_t w = (uint64_t)chunk << (16 * (lane & 3));
    w |= __shfl_down_sync(0xffffffffu, w, 1);
    w |= __shfl_down_sync(0xffffffffu, w, 2);
    const bool nz = __any_sync(0xffffffffu, chunk != 0);
    if ((lane & 3) == 0) out.mask[(size_t)seg * 8 + (lane >> 2)] = w;
    if (lane == 0) {
        out.key[seg] = key;
        out.nonzero[seg] = nz ? 1u : 0u;
    }
}

// The measure and moment terms of capsule A-B (grid units) in the voxel that has it at a-b: w mu
// and w mu T(t), t = (B - A) / |B - A| (zero for a degenerate segment), into q[0..6].
__device__ __forceinline__ void capsule_moments(float4 A, float4 B, const float* a, const float* b, float* q) {
    const float mu = capsule_measure(a, b, A.w);
    const float dg[3] = {B.x - A.x, B.y - A.y, B.z - A.z};
    const float dn = sqrtf((dg[0] * dg[0] + dg[1] * dg[1]) + dg[2] * dg[2]);
    float t[3] = {0.0f, 0.0f, 0.0f};
    if (dn > 0.0f) { t[0] = dg[0] / dn; t[1] = dg[1] / dn; t[2] = dg[2] / dn; }
    const float c = B.w * mu;
    q[0] = c;
    q[1] = c * (t[0] * t[0]);
    q[2] = c * (t[1] * t[1]);
    q[3] = c * (t[2] * t[2]);
    q[4] = c * (t[0] * t[1]);
    q[5] = c * (t[0] * t[2]);
    q[6] = c * (t[1] * t[2]);
}

// The key that orders the mask tests of a voxel's capsules: those whose axis passes deepest into
// the voxel first (they set the most bits, so later capsules find more rows full or out of
// reach).  The mask is an OR, so neither the order nor any rounding of the key changes it.
__device__ __forceinline__ uint32_t capsule_order(const CapsuleLocal& cl) {
    const float e[3] = {cl.d_idd.x, cl.d_idd.y, cl.d_idd.z};
    const float w[3] = {0.5f - cl.a_rr.x, 0.5f - cl.a_rr.y, 0.5f - cl.a_rr.z};
    float tt = ((w[0] * e[0] + w[1] * e[1]) + w[2] * e[2]) * cl.d_idd.w;
    tt = fminf(fmaxf(tt, 0.0f), 1.0f);
    const float dx = w[0] - tt * e[0], dy = w[1] - tt * e[1], dz = w[2] - tt * e[2];
    const float v = ((dx * dx + dy * dy) + dz * dz) - cl.a_rr.w;
    const uint32_t bits = __float_as_uint(v);
    return bits ^ ((bits >> 31) ? 0xffffffffu : 0x80000000u);   // order-preserving as unsigned
}

// Steps 1-3 of the `cnt` capsules of one voxel whose ordering keys sit at lanes src0,
// src0 + 1, ... of `okey` (the batch slot is a key's low 5 bits), on top of the lane's 16-bit
// chunk of the mask (lane L: rows sy0, sy0 + 1 of slab sz).  A row whose unset sub-cells are all
// out of the capsule's reach is passed over; most capsules reach no such row in the whole
// voxel.  The pooled step-3 tasks refer to this batch's slots, so they are evaluated before the
// function returns.
__device__ __forceinline__ uint32_t voxel_mask(CapsuleTasks& ct, uint32_t okey, uint32_t cnt, int src0, int sy0, int sz,
                                               uint32_t chunk, bool& full) {
    const int lane = threadIdx.x & 31;
    const float y0 = (float)sy0 * 0.125f + 0.0625f, zc = (float)sz * 0.125f + 0.0625f;
    const f2 ny = f2_pack(-y0, -(y0 + 0.125f));
    UnsetRows ur = unset_rows(chunk);
    int ntask = 0;
    for (uint32_t j = 0; j < cnt; ++j) {
        if (full) break;
        const int slot = (int)(__shfl_sync(0xffffffffu, okey, src0 + (int)j) & 31u);
        const CapsuleSlot& cs = ct.slot[slot];
        bool p0, p1;
        rows_reached(cs.c, ur, ny, cs.c.a_rr.z - zc, p0, p1);
        p0 = p0 && (chunk & 0xffu) != 0xffu;
        p1 = p1 && (chunk & 0xff00u) != 0xff00u;
        if (!__any_sync(0xffffffffu, p0 || p1)) continue;
        const AxisTerms tz = axis_terms(cs.c.a_rr.z, cs.c.b_reta.z, sz);
        uint32_t set = 0, open = 0;
#pragma unroll
        for (int yi = 0; yi < 2; ++yi) {
            const bool p = yi ? p1 : p0;
            if (!__any_sync(0xffffffffu, p)) continue;
            uint32_t rs, ro;
            capsule_row(cs, tz, sy0 + yi, rs, ro);
            if (p) {
                set |= rs << (8 * yi);
                open |= ro << (8 * yi);
            }
        }
        const uint32_t before = chunk;
        chunk |= set;
        // pool the undecided sub-cells as step-3 tasks of this capsule, one per lane and turn
        uint32_t und = open & ~chunk;
        for (uint32_t bal; (bal = __ballot_sync(0xffffffffu, und != 0u)) != 0u;) {
            if (ntask + 32 > CT_TASKS) {
                __syncwarp();
                chunk = capsule_step3_pool(ct, ntask, chunk);
                ntask = 0;
                und &= ~chunk;
                continue;
            }
            if (und) {
                const int bpos = __ffs(und) - 1;
                und &= und - 1;
                ct.task[ntask + __popc(bal & ((1u << lane) - 1u))] = (uint16_t)((slot << 9) | (16 * lane + bpos));
            }
            ntask += __popc(bal);
        }
        if (__any_sync(0xffffffffu, chunk != before)) {
            ur = unset_rows(chunk);
            full = __all_sync(0xffffffffu, chunk == 0xffffu);
        }
    }
    __syncwarp();
    if (ntask > 0 && !full) chunk = capsule_step3_pool(ct, ntask, chunk);
    return chunk;
}

// Warp per candidate voxel, up to eight voxels per step (fewer when the grid's warps would
// otherwise run out of voxels).  The step's voxels form groups of consecutive voxels whose
// capsules fit one batch (at most 32 together), and one setup serves a group: lane l takes the
// group's l-th pair.
//   - A capsule whose axis misses the voxel has measure 0 (few cross it: a capsule is a candidate
//     of every voxel that its radius reaches), so the measures and the sums run over the
//     others only.  Adding the zeros would not change an FP32 sum.
//   - A voxel with a capsule that covers it whole is full, and needs no mask steps.
//   - The rest are ordered by one sort of the batch with the voxel above the distance key, which
//     leaves each voxel's capsules together, and their mask steps run voxel by voxel.
// A voxel of more than 32 capsules is a group of its own and runs in batches of 32.  The setup
// and the mask steps each have one call site, so that the kernel holds one copy of them.
// Issue-bound (80 % of slots; DRAM at the definition's bytes).  768k capsules at 512^3, 75 M pairs:
// 9.8 ms against 18.9 ms when every capsule ran steps 1-2 on every row; a yarn of 4-voxel
// radius at 1024^3, 107 M pairs, four of five voxels covered: 5.2 ms against 9.6 ms.  Of 46 M
// capsules tested, 24 % reach a row and 40 rows per 100 run.  7 blocks per SM (72 registers,
// 24 words spilled) ran the 1024^3 yarn in 5.2 ms, 6 blocks in 5.4 ms.
__global__ void __launch_bounds__(RED_WARPS * 32, 7) k_reduce_fibers(const uint32_t* __restrict__ keys,
                                                                  const uint32_t* __restrict__ prims,
                                                                  const uint32_t* __restrict__ starts,
                                                                  const uint32_t* __restrict__ nseg_p,
                                                                  const float4* __restrict__ ra,
                                                                  const float4* __restrict__ rb, SegOut out, int bx,
                                                                  int by, int bz, uint32_t* __restrict__ next) {
    constexpr uint32_t STEP = 8;   // voxels per warp step (a group's voxel index takes 3 bits)
    const int lane = threadIdx.x & 31;
    const uint32_t nseg = *nseg_p;
    const int sz = lane >> 2, sy0 = (lane & 3) * 2;
    __shared__ CapsuleTasks pool[RED_WARPS];
    CapsuleTasks& ct = pool[threadIdx.x >> 5];
    const uint32_t step = max(1u, min(STEP, nseg / (gridDim.x * RED_WARPS)));
    for (;;) {
        uint32_t s0 = 0;
        if (lane == 0) s0 = atomicAdd(next, step);
        s0 = __shfl_sync(0xffffffffu, s0, 0);
        if (s0 >= nseg) break;
        const uint32_t nv = min(step, nseg - s0);
        // lane i holds the first pair of voxel s0 + i (lane nv the end of the last one)
        const uint32_t st = starts[s0 + min((uint32_t)lane, nv)];
        for (uint32_t g = 0; g < nv;) {
            const uint32_t gbeg = __shfl_sync(0xffffffffu, st, g);
            // the group [g, g + m): as many voxels as end within 32 pairs, at least one
            const uint32_t fit = __ballot_sync(0xffffffffu, (uint32_t)lane > g && (uint32_t)lane <= nv && st - gbeg <= 32u);
            const uint32_t m = max(1u, (uint32_t)__popc(fit));
            const uint32_t gend = __shfl_sync(0xffffffffu, st, g + m);
            uint32_t chunk = 0;
            bool full = false;
            float accc = 0.0f;   // one voxel's sums, lane c < 7: component c
            for (uint32_t base = gbeg; base < gend; base += 32) {
                const uint32_t cnt = min(32u, gend - base);
                // the lane's voxel in the group and that voxel's lanes [vb, ve)
                uint32_t v = 0, vb = 0, ve = cnt;
                for (uint32_t t = 1; t < m; ++t) {
                    const uint32_t e = __shfl_sync(0xffffffffu, st, g + t) - base;
                    if ((uint32_t)lane >= e) { v = t; vb = e; }
                    else ve = min(ve, e);
                }
                __syncwarp();   // the previous batch's sums and masks have read the shared state
                uint32_t key = 0, okey = 0xffffffe0u | (uint32_t)lane;
                bool covers = false, sums = false;
                float a[3], b[3];
                float4 A = make_float4(0, 0, 0, 0), B = A;
                if ((uint32_t)lane < cnt) {
                    key = keys[base + lane];
                    const uint32_t p = prims[base + lane];
                    A = ra[p];
                    B = rb[p];
                    const float f[3] = {(float)((int)vx_compact1by2(key) + bx), (float)((int)vx_compact1by2(key >> 1) + by),
                                        (float)((int)vx_compact1by2(key >> 2) + bz)};
                    a[0] = A.x - f[0]; a[1] = A.y - f[1]; a[2] = A.z - f[2];
                    b[0] = B.x - f[0]; b[1] = B.y - f[1]; b[2] = B.z - f[2];
                    covers = capsule_covers(a, b, A.w * A.w);
                    // with both ends beyond one face the clip is empty: one of its parameters is
                    // at least 1 (or at most 0) after rounding too, since |b - a| is then no
                    // larger than the distance of the farther end to that face
                    bool out_ = false;
#pragma unroll
                    for (int i = 0; i < 3; ++i) out_ = out_ || (a[i] < 0.0f && b[i] < 0.0f) || (a[i] > 1.0f && b[i] > 1.0f);
                    // (an infinite B - A has no tangent: its terms are not finite and are kept)
                    out_ = out_ && fmax3(fabsf(B.x - A.x), fabsf(B.y - A.y), fabsf(B.z - A.z)) < INFINITY;
                    if (!out_) {
                        float* q = ct.q + lane * 7;
                        capsule_moments(A, B, a, b, q);
#pragma unroll
                        for (int c = 0; c < 7; ++c) sums = sums || q[c] != 0.0f;
                    }
                }
                const uint32_t summed = __ballot_sync(0xffffffffu, sums);
                const uint32_t cover = __ballot_sync(0xffffffffu, covers);
                const uint32_t vlanes = (ve > 31u ? 0xffffffffu : (1u << ve) - 1u) & ~((1u << vb) - 1u);
                const bool live = (uint32_t)lane < cnt && (cover & vlanes) == 0u;
                __syncwarp();
                // sums in primitive order, one component of one voxel per lane (the same sequence
                // of FP32 additions as a single running sum per component)
                if (m > 1) {
                    for (uint32_t it0 = 0; it0 < 7u * m; it0 += 32) {
                        const uint32_t it = it0 + (uint32_t)lane, u = min(it / 7u, m - 1u), c = it - 7u * u;
                        const uint32_t ub = __shfl_sync(0xffffffffu, st, g + u) - base;
                        const uint32_t ue = __shfl_sync(0xffffffffu, st, g + u + 1) - base;
                        if (it < 7u * m) {
                            float acc = 0.0f;
                            for (uint32_t w = summed & (ue > 31u ? 0xffffffffu : (1u << ue) - 1u) & ~((1u << ub) - 1u); w;
                                 w &= w - 1u)
                                acc = acc + ct.q[(__ffs(w) - 1) * 7 + c];
                            if (c == 0) out.mass[s0 + g + u] = acc;
                            else out.moment[(size_t)(s0 + g + u) * 6 + c - 1] = acc;
                        }
                    }
                } else if (lane < 7) {
                    for (uint32_t w = summed; w; w &= w - 1u) accc = accc + ct.q[(__ffs(w) - 1) * 7 + lane];
                }
                // the mask steps' slots and their order, for the voxels that need them
                if (__any_sync(0xffffffffu, live && !full)) {
                    if (live) {
                        const CapsuleLocal cl = capsule_local(a, b, A.w);
                        ct.slot[lane].c = cl;
                        const bool huge = cl.a_rr.w > kHugeRR;
                        ct.slot[lane].x = capsule_x(huge ? NAN : a[0], huge ? NAN : b[0]);
                        okey = capsule_order(cl);
                    }
                    // the voxel in the top bits (every key of a lane in use below the others')
                    if ((uint32_t)lane < cnt) okey = (v << 29) | (min(okey >> 3, 0x1fffffbfu) & 0x1fffffe0u) | (uint32_t)lane;
                    __syncwarp();
                    // bitonic sort of the keys (unique: the lane is the low 5 bits); after the
                    // stage of width k, lanes 0..k-1 hold their keys in ascending order, so the sort
                    // stops once k covers the batch
#pragma unroll
                    for (int k = 2; k <= 32; k <<= 1) {
#pragma unroll
                        for (int jj = k >> 1; jj > 0; jj >>= 1) {
                            const uint32_t other = __shfl_xor_sync(0xffffffffu, okey, jj);
                            const bool keep_min = ((lane & k) == 0) == ((lane & jj) == 0);
                            okey = keep_min ? min(okey, other) : max(okey, other);
                        }
                        if ((uint32_t)k >= cnt) break;
                    }
                }
                // voxel by voxel; a voxel's outputs once its last batch is in
                for (uint32_t u = 0; u < m; ++u) {
                    const uint32_t ub = m > 1 ? __shfl_sync(0xffffffffu, st, g + u) - base : 0u;
                    const uint32_t ue = m > 1 ? __shfl_sync(0xffffffffu, st, g + u + 1) - base : cnt;
                    const uint32_t lanes = (ue > 31u ? 0xffffffffu : (1u << ue) - 1u) & ~((1u << ub) - 1u);
                    if (cover & lanes) {
                        chunk = 0xffffu;
                        full = true;
                    }
                    if (!full) chunk = voxel_mask(ct, okey, ue - ub, (int)ub, sy0, sz, chunk, full);
                    if (m > 1 || base + cnt >= gend) {
                        write_mask(out, s0 + g + u, __shfl_sync(0xffffffffu, key, ub), chunk);
                        if (m == 1 && lane < 7) {
                            if (lane == 0) out.mass[s0 + g] = accc;
                            else out.moment[(size_t)(s0 + g) * 6 + lane - 1] = accc;
                        }
                        chunk = 0;
                        full = false;
                    }
                }
            }
            g += m;
        }
    }
}

// Warp per candidate voxel, up to 28 voxels per step (fewer when the grid's warps would
// otherwise run out of voxels).  Consecutive voxels whose triangles fit one batch (at most 32
// together) form a group: lane l takes the group's l-th pair and computes its clipped area, its
// moment terms and its 512-bit mask, so that a mesh's few triangles per voxel fill the lanes.  Then
// each voxel's masks are ORed, lane L on bits 16 L .. 16 L + 15.  A voxel of more than 32 triangles
// is a group of its own and runs in batches of 32.
// Bound by dispatch (DRAM idle).  2.09 M triangles at 1024^3, 28.5 M pairs, 3.9 per voxel: 7.5 ms,
// issuing on 80 % of slots with 18 lanes (8.9 ms, and 68 %, in the longer kernel; of those the areas
// took 2.4, the edge axes 2.7 and the face normal 2.4; 45.9 ms with a voxel's
// triangles alone in the lanes and the warp on one triangle's sub-cells; 12.0 ms with grouped
// areas and records but the warp still on one triangle).  6 blocks per SM: 8.3 ms.
__global__ void __launch_bounds__(RED_WARPS * 32, 5) k_reduce_tris(const uint32_t* __restrict__ keys,
                                                                const uint32_t* __restrict__ prims,
                                                                const uint32_t* __restrict__ starts,
                                                                const uint32_t* __restrict__ nseg_p,
                                                                const float4* __restrict__ r0,
                                                                const float4* __restrict__ r1,
                                                                const float4* __restrict__ r2, SegOut out,
                                                                int bx, int by, int bz,
                                                                uint32_t* __restrict__ next) {
    constexpr uint32_t STEP = 28;   // their starts and the end sit in the lanes of one register
    const int lane = threadIdx.x & 31;
    const uint32_t nseg = *nseg_p;
    // the polygons of the measure, then the pairs' masks, in the same memory
    union Shared {
        float poly[POLY_FLOATS];
        uint8_t mask[32 * TRI_MASK];
    };
    __shared__ Shared shared[RED_WARPS];
    __shared__ float qs[RED_WARPS][32 * 7];       // per-pair w mu, w mu T(n) (pair-major)
    Shared& sh = shared[threadIdx.x >> 5];
    float* const qw = qs[threadIdx.x >> 5];
    const uint32_t step = max(1u, min(STEP, nseg / (gridDim.x * RED_WARPS)));
    for (;;) {
        uint32_t s0 = 0;
        if (lane == 0) s0 = atomicAdd(next, step);
        s0 = __shfl_sync(0xffffffffu, s0, 0);
        if (s0 >= nseg) break;
        const uint32_t nv = min(step, nseg - s0);
        // lane i holds the first pair of voxel s0 + i (lane nv the end of the last one)
        const uint32_t st = starts[s0 + min((uint32_t)lane, nv)];
        for (uint32_t g = 0; g < nv;) {
            const uint32_t gbeg = __shfl_sync(0xffffffffu, st, g);
            // the group [g, g + m): as many voxels as end within 32 pairs, at least one
            const uint32_t fit = __ballot_sync(0xffffffffu, (uint32_t)lane > g && (uint32_t)lane <= nv && st - gbeg <= 32u);
            const uint32_t m = max(1u, (uint32_t)__popc(fit));
            const uint32_t gend = __shfl_sync(0xffffffffu, st, g + m);
            uint32_t chunk = 0;
            float accc = 0.0f;   // one voxel's sums, lane c < 7: component c
            for (uint32_t base = gbeg; base < gend; base += 32) {
                const uint32_t cnt = min(32u, gend - base);
                uint32_t key = 0;
                float4 a, b, c;
                float v[3][3], f[3][3];
                __syncwarp();   // the previous batch's masks and sums have read the shared state
                if ((uint32_t)lane < cnt) {
                    key = keys[base + lane];
                    const uint32_t p = prims[base + lane];
                    a = r0[p];
                    b = r1[p];
                    c = r2[p];
                    tri_local(a, b, c, (int)vx_compact1by2(key) + bx, (int)vx_compact1by2(key >> 1) + by,
                              (int)vx_compact1by2(key >> 2) + bz, v, f);
                    const float mu = tri_measure(v, sh.poly);
                    const float n0 = f[0][1] * f[1][2] - f[0][2] * f[1][1];
                    const float n1 = f[0][2] * f[1][0] - f[0][0] * f[1][2];
                    const float n2 = f[0][0] * f[1][1] - f[0][1] * f[1][0];
                    const float nn = sqrtf((n0 * n0 + n1 * n1) + n2 * n2);
                    float t[3] = {0.0f, 0.0f, 0.0f};
                    if (nn > 0.0f) { t[0] = n0 / nn; t[1] = n1 / nn; t[2] = n2 / nn; }
                    const float cc = a.w * mu;
                    float* q = qw + lane * 7;
                    q[0] = cc;
                    q[1] = cc * (t[0] * t[0]);
                    q[2] = cc * (t[1] * t[1]);
                    q[3] = cc * (t[2] * t[2]);
                    q[4] = cc * (t[0] * t[1]);
                    q[5] = cc * (t[0] * t[2]);
                    q[6] = cc * (t[1] * t[2]);
                }
                __syncwarp();   // every lane's polygons are done: the masks take their place
                if ((uint32_t)lane < cnt)
                    tri_mask(v, f, a, b, c, (int)vx_compact1by2(key) + bx, (int)vx_compact1by2(key >> 1) + by,
                             (int)vx_compact1by2(key >> 2) + bz, sh.mask + lane * TRI_MASK);
                __syncwarp();
                // sums in primitive order, one component of one voxel per lane (one FP32 running
                // sum each)
                if (m > 1) {
                    for (uint32_t it0 = 0; it0 < 7u * m; it0 += 32) {
                        const uint32_t it = it0 + (uint32_t)lane, u = min(it / 7u, m - 1u), c = it - 7u * u;
                        const uint32_t ub = __shfl_sync(0xffffffffu, st, g + u) - base;
                        const uint32_t ue = __shfl_sync(0xffffffffu, st, g + u + 1) - base;
                        if (it < 7u * m) {
                            float acc = 0.0f;
#pragma unroll 1
                            for (uint32_t j = ub; j < ue; ++j) acc = acc + qw[j * 7 + c];
                            if (c == 0) out.mass[s0 + g + u] = acc;
                            else out.moment[(size_t)(s0 + g + u) * 6 + c - 1] = acc;
                        }
                    }
                } else if (lane < 7) {
#pragma unroll 1
                    for (uint32_t j = 0; j < cnt; ++j) accc = accc + qw[j * 7 + lane];
                }
                // the masks, voxel by voxel; a voxel's outputs once its last batch is in
                for (uint32_t u = 0; u < m; ++u) {
                    const uint32_t ub = m > 1 ? __shfl_sync(0xffffffffu, st, g + u) - base : 0u;
                    const uint32_t ue = m > 1 ? __shfl_sync(0xffffffffu, st, g + u + 1) - base : cnt;
#pragma unroll 1
                    for (uint32_t j = ub; j < ue; ++j)
                        chunk |= *reinterpret_cast<const uint16_t*>(sh.mask + j * TRI_MASK + 2 * lane);
                    if (m > 1 || base + cnt >= gend) {
                        write_mask(out, s0 + g + u, __shfl_sync(0xffffffffu, key, ub), chunk);
                        if (m == 1 && lane < 7) {
                            if (lane == 0) out.mass[s0 + g] = accc;
                            else out.moment[(size_t)(s0 + g) * 6 + lane - 1] = accc;
                        }
                        chunk = 0;
                    }
                }
            }
            g += m;
        }
    }
}

// ------------------------------------------------------------------------------------
// finalize: compaction + occupancy + lobe
// ------------------------------------------------------------------------------------
__device__ __forceinline__ void mask_counts(const uint64_t* m, uint16_t& occ, uint8_t* proj) {
    int o = 0, yz = 0, xz = 0;
    uint64_t orz = 0;
#pragma unroll
    for (int w = 0; w < 8; ++w) {
        uint64_t x = m[w];
        o += __popcll(x);
        orz |= x;
        // along x: a row (byte) is occupied if any of its bits is
        uint64_t t = x | (x >> 4);
        t |= t >> 2;
        t |= t >> 1;
        yz += __popcll(t & 0x0101010101010101ull);
        // along y: OR of the 8 rows
        uint64_t r = x | (x >> 32);
        r |= r >> 16;
        r |= r >> 8;
        xz += __popc((uint32_t)(r & 0xffu));
    }
    occ = (uint16_t)o;
    proj[0] = (uint8_t)yz;
    proj[1] = (uint8_t)xz;
    proj[2] = (uint8_t)__popcll(orz);
}

__device__ __forceinline__ void write_lobe(float m, const float* M, float* lobe, float* comp, uint8_t* cnt) {
    if (m > 0.0f) {
        float S[6];
#pragma unroll
        for (int c = 0; c < 6; ++c) S[c] = M[c] / m;
#pragma unroll
        for (int c = 0; c < 6; ++c) lobe[c] = S[c];
        lobe[6] = m;
        comp[0] = sqrtf(S[0]);
        comp[1] = sqrtf(S[1]);
        comp[2] = sqrtf(S[2]);
        float pxy = S[0] * S[1], pxz = S[0] * S[2], pyz = S[1] * S[2];
        comp[3] = pxy > 0.0f ? S[3] / sqrtf(pxy) : 0.0f;
        comp[4] = pxz > 0.0f ? S[4] / sqrtf(pxz) : 0.0f;
        comp[5] = pyz > 0.0f ? S[5] / sqrtf(pyz) : 0.0f;
        *cnt = 1;
    } else {
#pragma unroll
        for (int c = 0; c < 7; ++c) lobe[c] = 0.0f;
#pragma unroll
        for (int c = 0; c < 6; ++c) comp[c] = 0.0f;
        *cnt = 0;
    }
}

// Bound by memory: 130 bytes read and 152 written per voxel.  A warp takes 32 consecutive segments; the rows it
// keeps are consecutive in the level, so the masks, moments and lobes go through shared memory,
// compacted, and are read and written with whole lines.  (A lane copying its own 64-, 24- and
// 28-byte rows waited for the many partly used lines: mesh 0.52 ms, woven 0.53 and yarn 0.34 ms
// against 0.31, 0.35 and 0.23 ms, 6 TB/s; eight or six blocks per SM 2 and 7 % more.)
constexpr int FIN_WARPS = 4;
__global__ void __launch_bounds__(FIN_WARPS * 32, 7) k_finalize(SegOut in, const uint32_t* __restrict__ nseg_p,
                                                             const uint32_t* __restrict__ dst, vx_level L,
                                                             uint64_t key_hi) {
    struct Rows {
        uint4 mask[32 * 5];        // four 16-byte pieces per row and one of padding
        float2 moment[32 * 3];
        float lobes[32 * 7], compact[32 * 6];
    };
    __shared__ Rows rows[FIN_WARPS];
    Rows& W = rows[threadIdx.x >> 5];
    const int lane = threadIdx.x & 31;
    const uint32_t nseg = *nseg_p, warps = gridDim.x * FIN_WARPS;
    for (uint32_t s0 = (blockIdx.x * FIN_WARPS + (threadIdx.x >> 5)) * 32u; s0 < nseg; s0 += warps * 32u) {
        const uint32_t s = s0 + (uint32_t)lane, n = min(32u, nseg - s0);
        const bool keep = s < nseg && in.nonzero[s];
        const uint32_t kept = __ballot_sync(0xffffffffu, keep);
        if (!kept) continue;
        const uint32_t count = (uint32_t)__popc(kept), below = (1u << lane) - 1u;
        const size_t o0 = dst[s0 + (uint32_t)__ffs(kept) - 1u];   // (the same word for the whole warp)
        const uint32_t rank = (uint32_t)__popc(kept & below);
        const uint4* const mi = reinterpret_cast<const uint4*>(in.mask + (size_t)s0 * 8);
        const float2* const Mi = reinterpret_cast<const float2*>(in.moment + (size_t)s0 * 6);
        uint4 mp[4];
        float2 Mp[3];
        bool mk[4], Mk[3];
        uint32_t mr[4], Mr[3];
#pragma unroll
        for (int q = 0; q < 4; ++q) {   // (a row that is not kept is not read)
            const uint32_t i = q * 32 + lane, r = i >> 2;
            mk[q] = r < n && ((kept >> r) & 1u);
            mr[q] = (uint32_t)__popc(kept & ((1u << r) - 1u)) * 5 + (i & 3);
            if (mk[q]) mp[q] = mi[i];
        }
#pragma unroll
        for (int q = 0; q < 3; ++q) {
            const uint32_t i = q * 32 + lane, r = i / 3;
            Mk[q] = r < n && ((kept >> r) & 1u);
            Mr[q] = (uint32_t)__popc(kept & ((1u << r) - 1u)) * 3 + (i - 3 * r);
            if (Mk[q]) Mp[q] = Mi[i];
        }
        const float mass = keep ? in.mass[s] : 0.0f;
        const uint32_t key = keep ? in.key[s] : 0u;
#pragma unroll
        for (int q = 0; q < 4; ++q)
            if (mk[q]) W.mask[mr[q]] = mp[q];
#pragma unroll
        for (int q = 0; q < 3; ++q)
            if (Mk[q]) W.moment[Mr[q]] = Mp[q];
        __syncwarp();
        if (keep) {
            const size_t o = o0 + rank;
            uint64_t m[8];
#pragma unroll
            for (int w = 0; w < 4; ++w) {
                const uint4 q = W.mask[rank * 5 + w];
                m[2 * w] = ((uint64_t)q.y << 32) | q.x;
                m[2 * w + 1] = ((uint64_t)q.w << 32) | q.z;
            }
            float M[6];
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                const float2 q = W.moment[rank * 3 + c];
                M[2 * c] = q.x;
                M[2 * c + 1] = q.y;
            }
            uint16_t occ;
            uint8_t pj[3];
            mask_counts(m, occ, pj);
            L.keys[o] = key_hi | (uint64_t)key;
            L.mass[o] = mass;
            L.occ[o] = occ;
            L.occ_proj[o * 3 + 0] = pj[0];
            L.occ_proj[o * 3 + 1] = pj[1];
            L.occ_proj[o * 3 + 2] = pj[2];
            write_lobe(mass, M, W.lobes + rank * 7, W.compact + rank * 6, L.lobe_count + o);
        }
        __syncwarp();
        uint4* const mo = reinterpret_cast<uint4*>(L.mask + o0 * 8);
        float2* const Mo = reinterpret_cast<float2*>(L.moment + o0 * 6);
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const uint32_t i = q * 32 + lane;
            if (i < count * 4) mo[i] = W.mask[(i >> 2) * 5 + (i & 3)];
        }
#pragma unroll
        for (int q = 0; q < 3; ++q) {
            const uint32_t i = q * 32 + lane;
            if (i < count * 3) Mo[i] = W.moment[i];
        }
#pragma unroll
        for (int q = 0; q < 7; ++q) {
            const uint32_t i = q * 32 + lane;
            if (i < count * 7) L.lobes[o0 * 7 + i] = W.lobes[i];
        }
#pragma unroll
        for (int q = 0; q < 6; ++q) {
            const uint32_t i = q * 32 + lane;
            if (i < count * 6) L.compact[o0 * 6 + i] = W.compact[i];
        }
        __syncwarp();
    }
}

inline unsigned grid_for(size_t n, int threads) {
    size_t b = (n + threads - 1) / threads;
    if (b < 1) b = 1;
    if (b > 0x7fffffff) b = 0x7fffffff;
    return (unsigned)b;
}

}  // namespace
