// Targets evaluated in float-float (ffmath.cuh): the pixels of the FP64 FMM
// form and of the dense form.  Segments are staged in shared memory in a
// frame around the targets, differences taken in FP64 (once per segment and
// block), then held as (hi, lo) floats.
#pragma once

#include <cuda_runtime.h>

#include "ffmath.cuh"

namespace dc {
namespace evalff {

constexpr int kStage = 64;   // segments staged per round

struct Stage {
    // x1 y1 | x2 y2 | dx dy, each (hi, lo); len and the weights of the three
    // channels: -w sigma / 2 pi and -w mu / 2 pi; p3: third floats of x1 y1 x2 y2
    float4 p1[kStage], p2[kStage], p3[kStage], d[kStage];
    float2 len[kStage], sg[kStage][3], mg[kStage][3];
};

// Entry i of the stage: the segment q (x1 y1 x2 y2) relative to (cx, cy),
// times iw (a power of two that brings the frame to about one: squares of
// distances have to stay normal floats); ks, km: what multiplies sb and mb.
__device__ __forceinline__ void stage_segment(Stage &t, int i, const double *__restrict__ q, double cx, double cy,
                                              double iw, double len, double ks, double km,
                                              const double *__restrict__ sb, const double *__restrict__ mb) {
    const ff::Coord x1 = ff::coord((q[0] - cx) * iw), y1 = ff::coord((q[1] - cy) * iw);
    const ff::Coord x2 = ff::coord((q[2] - cx) * iw), y2 = ff::coord((q[3] - cy) * iw);
    const float2 dx = ff::from((q[2] - q[0]) * iw), dy = ff::from((q[3] - q[1]) * iw);
    t.p1[i] = make_float4(x1.f.x, x1.f.y, y1.f.x, y1.f.y);
    t.p2[i] = make_float4(x2.f.x, x2.f.y, y2.f.x, y2.f.y);
    t.p3[i] = make_float4(x1.t, y1.t, x2.t, y2.t);
    t.d[i] = make_float4(dx.x, dx.y, dy.x, dy.y);
    t.len[i] = ff::from(len * iw);
    for (int c = 0; c < 3; ++c) {
        t.sg[i][c] = ff::from(ks * sb[c]);
        t.mg[i][c] = ff::from(km * mb[c]);
    }
}

// A sum of three channels: a short run in float-float (hi, lo), flushed into
// FP64 round by round.  The lo parts of a long run would lose what they hold:
// 5,120 large, cancelling terms summed without a flush were 1e-11 off, the
// pairs themselves 4e-15.
struct Sum3 {
    float h[3], l[3];
    double v[3];
    __device__ __forceinline__ void zero() {
        for (int c = 0; c < 3; ++c) {
            h[c] = l[c] = 0.f;
            v[c] = 0.0;
        }
    }
    __device__ __forceinline__ void flush() {
        for (int c = 0; c < 3; ++c) {
            v[c] += (double)h[c] + l[c];
            h[c] = l[c] = 0.f;
        }
    }
};
// a x b of the segment P (x1 y1 x2 y2) at the target (qx, qy), in FP64
static __device__ __noinline__ double cross64(const double *__restrict__ P, double qx, double qy) {
    return (P[0] - qx) * (P[3] - qy) - (P[1] - qy) * (P[2] - qx);
}
// what ff::pair asks of a pair's coordinates, from two lambdas
template <typename R, typename C>
struct NearPair {
    R refine;
    C cross;
};
template <typename R, typename C>
__device__ __forceinline__ NearPair<R, C> near_pair(R refine, C cross) {
    return {refine, cross};
}
// u += entry i's single and double layer at the target (x, y) of the frame;
// cross(): the entry's a x b at the target in FP64, in the frame's unit
template <typename Cross>
__device__ __forceinline__ void add_segment(const ff::Tables &T, const Stage &t, int i, ff::Coord x, ff::Coord y, Sum3 &u,
                                            const Cross &cross) {
    const float4 p1 = t.p1[i], p2 = t.p2[i], d = t.d[i];
    float2 il, ph;
    const auto near = near_pair(
        [&](float2 &ax, float2 &ay, float2 &bx, float2 &by) {
            const float4 p3 = t.p3[i];
            ax = ff::diff({make_float2(p1.x, p1.y), p3.x}, x);
            ay = ff::diff({make_float2(p1.z, p1.w), p3.y}, y);
            bx = ff::diff({make_float2(p2.x, p2.y), p3.z}, x);
            by = ff::diff({make_float2(p2.z, p2.w), p3.w}, y);
        },
        cross);
    ff::pair(T, ff::sub(make_float2(p1.x, p1.y), x.f), ff::sub(make_float2(p1.z, p1.w), y.f),
             ff::sub(make_float2(p2.x, p2.y), x.f), ff::sub(make_float2(p2.z, p2.w), y.f), make_float2(d.x, d.y),
             make_float2(d.z, d.w), t.len[i], il, ph, false, near);
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        dot2ff(u.h[c], u.l[c], il, t.sg[i][c]);
        dot2ff(u.h[c], u.l[c], ph, t.mg[i][c]);
    }
}

// u += Re sum_k C[c][k] p^k, k = 0 .. n - 1, for complex (px, py) and
// coefficients (re hi, re lo, im hi, im lo); the powers are shared by the
// three channels
__device__ __forceinline__ void add_powers(const float4 *__restrict__ C, int stride, int n, float2 px, float2 py, Sum3 &u) {
    float2 wx = make_float2(1.f, 0.f), wy = make_float2(0.f, 0.f);
    for (int k = 0; k < n; ++k) {
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            const float4 v = C[c * stride + k];
            dot2ff(u.h[c], u.l[c], make_float2(v.x, v.y), wx);
            dot2ff(u.h[c], u.l[c], make_float2(-v.z, -v.w), wy);
        }
        const float2 t = ff::dot(wx, px, ff::neg(wy), py);
        wy = ff::dot(wx, py, wy, px);
        wx = t;
    }
}

}  // namespace evalff
}  // namespace dc
