// The closed-form segment integrals (App. D) in float-float: values held as
// unevaluated sums hi + lo of two floats, about 48 bits.  FP64 runs at 1/64
// of the FP32 rate on this GPU: one pair in FP64 (two log, one atan2, some
// 60 other operations) takes the FP64 pipe as long as 18,000 FP32
// instructions per lane would, the same pair here about 450.  Coordinates
// are relative to a centre near the targets (the difference is taken in FP64
// once per piece, not per pair).  Where that centre's frame is more than about
// a thirty-second of the canvas, 48 bits of them are fewer than FP64 has: near
// pairs take the differences from three floats (Coord), and a target beside a
// segment takes its side from FP64.  Over 5,120 segments of four closed curves, densities up to
// 6,000, the pairs add up to 4.4e-15 of the field (the series beyond four
// lengths avoids the cancellation of the two logarithms); in FP64 to 1.9e-13.
//
// Sums and products are the classical error-free transformations (Knuth's
// two-sum, the FMA's two-product; Dekker 1971).  The logarithm and the
// arctangent reduce their argument by a table of reciprocals / tangents with
// few bits, so that the reduction is exact, and end in the first terms of
// their Taylor series.
#pragma once

#include <cuda_runtime.h>

#include "ffarith.cuh"

namespace dc {
namespace ff {

__device__ __forceinline__ float2 quick(float a, float b) {   // |a| >= |b|
    const float s = __fadd_rn(a, b);
    return make_float2(s, __fsub_rn(b, __fsub_rn(s, a)));
}
__device__ __forceinline__ float2 two_sum(float a, float b) {
    const float s = __fadd_rn(a, b), bb = __fsub_rn(s, a);
    return make_float2(s, __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb)));
}
__device__ __forceinline__ float2 from(double v) {
    const float h = (float)v;
    return make_float2(h, (float)(v - (double)h));
}
__device__ __forceinline__ double to(float2 a) { return (double)a.x + (double)a.y; }
__device__ __forceinline__ float2 neg(float2 a) { return make_float2(-a.x, -a.y); }
__device__ __forceinline__ float2 scale(float2 a, float s) { return make_float2(a.x * s, a.y * s); }   // s a power of two
__device__ __forceinline__ float2 add(float2 a, float2 b) {
    const float2 s = two_sum(a.x, b.x);
    return quick(s.x, __fadd_rn(s.y, __fadd_rn(a.y, b.y)));
}
__device__ __forceinline__ float2 sub(float2 a, float2 b) { return add(a, neg(b)); }
__device__ __forceinline__ float2 addf(float2 a, float b) {
    const float2 s = two_sum(a.x, b);
    return quick(s.x, __fadd_rn(s.y, a.y));
}
__device__ __forceinline__ float2 mul(float2 a, float2 b) {
    const float p = __fmul_rn(a.x, b.x);
    float e = __fmaf_rn(a.x, b.x, -p);
    e = __fmaf_rn(a.x, b.y, __fmaf_rn(a.y, b.x, e));
    return quick(p, e);
}
__device__ __forceinline__ float2 mulf(float2 a, float b) {
    const float p = __fmul_rn(a.x, b);
    return quick(p, __fmaf_rn(a.y, b, __fmaf_rn(a.x, b, -p)));
}
__device__ __forceinline__ float2 sqr(float2 a) {
    const float p = __fmul_rn(a.x, a.x);
    return quick(p, __fmaf_rn(2.f * a.x, a.y, __fmaf_rn(a.x, a.x, -p)));
}
// a b + c d (the sums' rounding relative to the larger product)
__device__ __forceinline__ float2 dot(float2 a, float2 b, float2 c, float2 d) {
    const float p = __fmul_rn(a.x, b.x), q = __fmul_rn(c.x, d.x);
    const float pe = __fmaf_rn(a.x, b.y, __fmaf_rn(a.y, b.x, __fmaf_rn(a.x, b.x, -p)));
    const float qe = __fmaf_rn(c.x, d.y, __fmaf_rn(c.y, d.x, __fmaf_rn(c.x, d.x, -q)));
    const float2 s = two_sum(p, q);
    return quick(s.x, __fadd_rn(s.y, __fadd_rn(pe, qe)));
}
// 1 / a
__device__ __forceinline__ float2 inv(float2 a) {
    const float q = __fdividef(1.f, a.x);
    const float r = __fmaf_rn(-q, a.y, __fmaf_rn(-q, a.x, 1.f));   // 1 - q a, exact to its rounding
    const float2 s = quick(q, q * r);
    const float r2 = __fmaf_rn(-s.y, a.x, __fmaf_rn(-s.x, a.y, __fmaf_rn(-s.x, a.x, 1.f)));
    return quick(s.x, __fmaf_rn(q, r2, s.y));
}

constexpr int kLogEntries = 256, kAtanEntries = 17;
struct Tables {
    float r[kLogEntries];        // 1 / m to ten bits at the middle of each mantissa interval
    float2 l[kLogEntries];       // -log(r)
    float2 at[kAtanEntries];     // atan(k / 16)
};
// filled by the block (a barrier has to follow)
__device__ __forceinline__ void init_tables(Tables &T) {
    for (int i = threadIdx.x; i < kLogEntries; i += blockDim.x) {
        const float m = 1.f + (i + 0.5f) / kLogEntries;
        const float r = __int_as_float((__float_as_int(1.f / m) + 0x2000) & ~0x3fff);
        T.r[i] = r;
        T.l[i] = from(-log((double)r));
    }
    for (int i = threadIdx.x; i < kAtanEntries; i += blockDim.x) T.at[i] = from(atan(i / 16.0));
}

// log(a), a > 0 normal: absolute error about 2^-49 of max(1, |log a|)
__device__ __forceinline__ float2 log(const Tables &T, float2 a) {
    const int b = __float_as_int(a.x);
    const int e = (b >> 23) - 127, i = (b >> 15) & 0xff;
    const float sc = __int_as_float((127 - e) << 23);   // 2^-e (e in [-126, 126])
    const float m = a.x * sc, r = T.r[i];
    // t = m r - 1, |t| < 2^-8
    const float p = __fmul_rn(m, r);
    const float2 t = quick(__fsub_rn(p, 1.f), __fmaf_rn(a.y * sc, r, __fmaf_rn(m, r, -p)));
    // log1p(t) = t - t^2 / 2 + t^3 (1/3 - t/4 + t^2/5 - t^3/6)
    const float u = t.x, u2 = u * u;
    const float q = u2 * u * fmaf(u, fmaf(u, fmaf(u, -1.f / 6.f, 0.2f), -0.25f), 1.f / 3.f);
    const float2 s = sqr(t);
    // e log 2 in three parts (the first of 16 bits: its product is exact)
    const float fe = (float)e;
    const float2 L = T.l[i];
    float2 v = two_sum(fe * 0.693145751953125f, L.x);
    const float p2 = __fmul_rn(fe, 0x1.7f7d1cp-20f);
    const float e2 = __fmaf_rn(fe, 0x1.7f7d1cp-20f, -p2) + fe * 0x1.ef357ap-45f;
    float lo = v.y + (L.y + e2);
    v = two_sum(v.x, p2);
    lo += v.y;
    v = two_sum(v.x, t.x);
    lo += v.y + t.y;
    v = two_sum(v.x, -0.5f * s.x);
    lo += v.y + (q - 0.5f * s.y);
    return quick(v.x, lo);
}

// atan2(y, x), not both zero: absolute error about 2^-47
__device__ __forceinline__ float2 atan2(const Tables &T, float2 y, float2 x) {
    const bool sy = y.x < 0.f || (y.x == 0.f && y.y < 0.f), sx = x.x < 0.f;
    if (sy) y = neg(y);
    if (sx) x = neg(x);
    const bool sw = y.x > x.x;
    const float2 n = sw ? x : y, d = sw ? y : x;
    // t = n / d in [0, 1]; atan t = atan t_k + atan((n - t_k d) / (d + t_k n)), t_k = k / 16
    // (at most 16 by rounding; the bound holds for arguments out of range too, denormal ones among them)
    const int k = min(max(__float2int_rn(16.f * __fdividef(n.x, d.x)), 0), kAtanEntries - 1);
    const float tk = (float)k * 0.0625f;
    const float2 num = sub(n, mulf(d, tk)), den = add(d, mulf(n, tk));
    const float2 v = mul(num, inv(den));   // |v| <= 1/32
    const float2 v2 = sqr(v);
    // v - v^3 / 3 + v^5 (1/5 - v^2 / 7 + v^4 / 9)
    const float2 v3 = mul(mul(v2, v), make_float2(0.333333343f, -9.93410776e-09f));
    const float q = v2.x * v2.x * v.x * fmaf(v2.x, fmaf(v2.x, 1.f / 9.f, -1.f / 7.f), 0.2f);
    float2 a = add(T.at[k], add(v, make_float2(-v3.x, q - v3.y)));
    if (sw) a = sub(make_float2(1.57079637f, -4.37113883e-08f), a);
    if (sx) a = sub(make_float2(3.14159274f, -8.74227766e-08f), a);
    return sy ? neg(a) : a;
}

// A coordinate of the frame as three floats: (hi, lo) drops up to five of a
// double's bits where the frame is as wide as the canvas, the third holds them.
struct Coord {
    float2 f;
    float t;
};
__device__ __forceinline__ Coord coord(double v) {
    Coord c;
    c.f = from(v);
    c.t = (float)((v - (double)c.f.x) - (double)c.f.y);
    return c;
}
// a - b to float-float accuracy of the difference itself, however close the
// two are: the hi and the lo parts are each subtracted without rounding
__device__ __forceinline__ float2 diff(Coord a, Coord b) {
    const float2 s = two_sum(a.f.x, -b.f.x), t = two_sum(a.f.y, -b.f.y), z = two_sum(s.x, t.x);
    return quick(z.x, __fadd_rn(z.y, __fadd_rn(s.y, __fadd_rn(t.y, __fsub_rn(a.t, b.t)))));
}

// ilog = int log|p - q| dS and phi = the subtended angle of the segment from
// a to b (relative to the target), half length vector not needed: d = b - a
// and len = |d| are the piece's own.  own: the target is a node of the piece's
// segment, phi = 0.
// Within four lengths the angle takes what a and b lose to (hi, lo)
// coordinates over the distance: near.refine(ax, ay, bx, by) then gives them
// from all bits (56 instructions more: the plain form's 517 x 509 pixels take
// 1,048 us instead of 1,014; beyond, what is lost stays below the pair's own
// rounding).
// A target beside the segment by less than 2^-40 of it, where rounding could
// give the wrong side, takes a x b from near.cross(), formed in FP64.
constexpr float kSide = 0x1p-40f;
template <typename Near>
__device__ __forceinline__ void pair(const Tables &T, float2 ax, float2 ay, float2 bx, float2 by, float2 dx, float2 dy,
                                     float2 len, float2 &ilog, float2 &phi, bool own, const Near &near) {
    const float2 mx = scale(add(ax, bx), 0.5f), my = scale(add(ay, by), 0.5f);   // midpoint
    const float2 r2 = dot(mx, mx, my, my);
    if (!own && 16.f * len.x * len.x < r2.x) {
        // series in zeta = eta^2, eta = d / (2 m), |zeta| < 1/64:
        //   ilog = len (log|m| - Re sum_k zeta^k / (2k (2k+1))),  phi = 2 Im eta sum_k zeta^k / (2k+1)
        // the first two terms in float-float, the rest (below 10^-7) in FP32
        const float2 h = scale(inv(r2), 0.5f);
        const float2 ex = mul(dot(dx, mx, dy, my), h), ey = mul(dot(dy, mx, neg(dx), my), h);
        const float2 zx = dot(ex, ex, neg(ey), ey), zy = scale(mul(ex, ey), 2.f);
        const float2 yx = dot(zx, zx, neg(zy), zy), yy = scale(mul(zx, zy), 2.f);   // zeta^2
        // zeta^3 (1/42 + zeta/72 + zeta^2/110 + ...), zeta^3 (1/7 + zeta/9 + ...)
        const float cx = yx.x * zx.x - yy.x * zy.x, cy = yx.x * zy.x + yy.x * zx.x;
        float gx = 1.f / 156.f, gy = 0.f, fx = 1.f / 13.f, fy = 0.f, t;
        t = gx * zx.x - gy * zy.x + 1.f / 110.f;
        gy = gx * zy.x + gy * zx.x;
        gx = t;
        t = gx * zx.x - gy * zy.x + 1.f / 72.f;
        gy = gx * zy.x + gy * zx.x;
        gx = t;
        t = gx * zx.x - gy * zy.x + 1.f / 42.f;
        gy = gx * zy.x + gy * zx.x;
        gx = t;
        t = fx * zx.x - fy * zy.x + 1.f / 11.f;
        fy = fx * zy.x + fy * zx.x;
        fx = t;
        t = fx * zx.x - fy * zy.x + 1.f / 9.f;
        fy = fx * zy.x + fy * zx.x;
        fx = t;
        t = fx * zx.x - fy * zy.x + 1.f / 7.f;
        fy = fx * zy.x + fy * zx.x;
        fx = t;
        const float2 sixth = make_float2(0.166666672f, -4.96705388e-09f), third = make_float2(0.333333343f, -9.93410776e-09f);
        const float2 twentieth = make_float2(0.0500000007f, -7.4505806e-10f), fifth = make_float2(0.200000003f, -2.98023224e-09f);
        const float2 g = addf(add(mul(zx, sixth), mul(yx, twentieth)), cx * gx - cy * gy);
        ilog = mul(len, sub(scale(log(T, r2), 0.5f), g));
        const float2 wx = add(make_float2(1.f, 0.f), addf(add(mul(zx, third), mul(yx, fifth)), cx * fx - cy * fy));
        const float2 wy = addf(add(mul(zy, third), mul(yy, fifth)), cx * fy + cy * fx);
        phi = scale(dot(ex, wy, ey, wx), 2.f);
        return;
    }
    near.refine(ax, ay, bx, by);
    float2 cr = dot(ax, by, neg(ay), bx);
    const float2 dt = dot(ax, bx, ay, by);
    if (!own && dt.x < 0.f && fabsf(cr.x) < kSide * fmaf(fabsf(ax.x), fabsf(by.x), fabsf(ay.x * bx.x)))
        cr = from(near.cross());
    phi = own || (cr.x == 0.f && dt.x == 0.f) ? make_float2(0.f, 0.f) : atan2(T, cr, dt);   // own, or at an end point: 0
    const float2 ra2 = dot(ax, ax, ay, ay), rb2 = dot(bx, bx, by, by), il = inv(len);
    const float2 s1 = mul(dot(ax, dx, ay, dy), il), s2 = mul(dot(bx, dx, by, dy), il);
    float2 la = make_float2(0.f, 0.f), lb = la;
    if (ra2.x > 0.f) la = mul(s1, log(T, ra2));
    if (rb2.x > 0.f) lb = mul(s2, log(T, rb2));
    ilog = add(sub(scale(sub(lb, la), 0.5f), len), mul(mul(cr, il), phi));
}

}  // namespace ff
}  // namespace dc
