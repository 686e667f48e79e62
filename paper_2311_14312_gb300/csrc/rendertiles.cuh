// Pixel evaluation of the FP32 form's render (Alg. 4): L2P + list-3 M2P +
// list-1 P2P of a rectangle of pixels that lies in one leaf.
//
// Everything far from the rectangle is harmonic around it, so it is not
// evaluated pixel by pixel.  With c the rectangle's centre and R its
// half-diagonal, a source is far when all of it is at least kSep R from c;
// the field of the far sources and of the leaf's local expansion is taken
// at kSamples points of the circle |z - c| = R, and a discrete Fourier
// transform of those values gives the coefficients of
//     u(z) = Re sum_{k < kCoefs} c_k ((z - c) / R)^k
// inside the circle.  A source at distance kSep R contributes (1 / kSep)^k /
// k to c_k, so the first term left out (k = 16, and what the samples alias
// onto lower ones) is 2.7e-8 of the source's strength at the closest
// distance, below the FP32 rounding of the sums.  The near sources' closed
// forms are still evaluated at every pixel.  On the 200-curve drawing at
// 2048^2 a pixel has 79 list-1 pieces and 8 list-3 cells; sampled at 32
// points for 256 pixels instead, they cost an eighth, and with the four
// pixels +-x +-y of a rectangle sharing the powers of z the polynomial takes
// 2.5 instructions per term and pixel.  Bound by instruction issue; on one
// GB300 the evaluation went from 3.00 to 1.05 ms there (27.6 to about 8 G lane
// instructions of pair, expansion and polynomial work), and 24 viewports up to
// zoom 10^6 of the 2000-curve drawing (87 Mpixels) from 27 to 8.4 ms.  Against
// 64-bit direct sums an image is off by 8e-8 (rms of the field; 1e-7 when every
// pixel was evaluated directly), 2% of the time being for sums that keep what
// large parts cancel (add_parts) and for a cut by channel.
//
// A block of four warps takes a rectangle: the warps share the sources of the
// samples (lanes = samples), then the pixels (lanes = pixels; in a rectangle
// with fewer than 128 the lanes left over share the sources).  One warp per
// rectangle was slower: the longest rectangles set the time (a warp alone
// takes milliseconds for 64 x 64 pixels with a hundred near pieces), and warps
// in different loops evict each other's instructions.
#pragma once

namespace rtiles {

constexpr int kSamples = 32;       // points on the circle, one per lane
constexpr int kCoefs = 16;         // coefficients k = 0 .. 15
constexpr float kSep = 2.5f;       // far: at least this many radii from the centre
// pieces and cells whose strength is large (the FP64 ones: heavy, hL, hM) are
// sampled in FP64 and from twice the distance, where the first term left out
// is 0.2^16 / 16 = 4e-13
constexpr float kSepBig = 5.f;
constexpr float kMaxRadius = 0.36f, kMaxRadiusBig = 0.18f;   // R in leaf widths (local expansion)
// distance from a piece, times the largest coordinate of the canvas, below which
// its side is decided in FP64: the (hi, lo) pairs hold 48 bits (3.6e-15 of the
// coordinate; 17 times that covers the differences and products of cross_ff)
constexpr float kSideBound = 6e-14f;
constexpr int kMinSampled = 48;    // rectangles of fewer pixels are evaluated directly
// and so are those with a radius, in leaf widths, whose square is not a normal
// float: 1 / R has to be one (such pixels are the same point to FP64 except
// beside the origin)
constexpr float kMinRadius = 1e-18f;
constexpr int kStaged = 64;        // near pieces staged per warp
constexpr int kWarps = 4;          // warps per block
constexpr int kBlocksPerSM = 4;    // 128 registers; 3 and 5 blocks measured 3-9% slower

// cos(2 pi j / 32) in FP64 (j = 0 .. 8); the rest by symmetry
__device__ __forceinline__ double cos32(int j) {
    j &= 31;
    if (j > 16) j = 32 - j;
    const bool neg = j > 8;
    if (neg) j = 16 - j;
    const double c = cospi((double)j * 0.0625);
    return neg ? -c : c;
}

struct BlockMem {
    // near pieces: x1h y1h x2h y2h | x1l y1l x2l y2l | len sg012 | mg012 id |
    // (pad: lanes that read different pieces hit different banks)
    float4 pc[kWarps * kStaged][5];
    float4 far[kWarps][32][3];    // far pieces being sampled: x1 y1 x2 y2 | len sg012 | mg012
    float4 cf[kCoefs][2];         // a0 b0 a1 b1 | a2 b2 - -
    float4 d[kWarps][32];         // the samples less their mean (a copy per warp)
    float2 v[kWarps][32][3];      // the warps' shares of the samples, (hi, lo)
    // rectangles with large far sources: the shares' FP64 terms, the samples
    // less their mean, and the coefficients, in FP64
    double h[kWarps][32][3], dv[32][3], cd[kCoefs][6];
    float pv[kWarps][12][32];     // the polynomial at the four pixels of each quad
    float2 tw[32];                // e^{2 pi i j / 32}
    int cnt[kWarps], flags[kWarps], next;
};

// a + b exactly: the sum and its rounding error (Knuth)
__device__ __forceinline__ float2 two_sum(float a, float b) {
    const float s = __fadd_rn(a, b), bb = __fsub_rn(s, a);
    return make_float2(s, __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb)));
}

// u + e / 2 pi as a float and its rest: what expansions give is added to what
// pieces give without rounding, since the two may cancel
__device__ __forceinline__ float2 add_expansion(float u, float e) {
    constexpr float kLo = (float)(kInv2Pi - (double)kInv2PiF);
    const float p = __fmul_rn(e, kInv2PiF);
    const float2 z = two_sum(u, p);
    return make_float2(z.x, z.y + fmaf(e, kLo, __fmaf_rn(e, kInv2PiF, -p)));
}
// mean + u + e / 2 pi + small, rounded once (but for the small part)
__device__ __forceinline__ float add_parts(float mean, float u, float e, float small) {
    const float2 z = add_expansion(u, e), y = two_sum(mean, z.x);
    return y.x + (y.y + (z.y + small));
}

// ilog = int log|p - q| and phi = the subtended angle of the segment from a
// to b (relative to the target q) in closed form (App. D), FP32.  A call,
// like the FP64 form: the loops that use them would not fit the instruction
// cache with every copy inlined (the kernel then waited for instructions 14
// cycles per instruction issued).
// cr = a x b: by the caller, who has it more exactly beside a segment.
__device__ __noinline__ float2 pair_closed(float ax, float ay, float bx, float by, float len, float cr) {
    const float dt = ax * bx + ay * by;
    const float dx = bx - ax, dy = by - ay;
    const float ilen = 1.f / len;
    // beside the segment the angle is +-pi less a small one, whose own error is small
    const float phi = (dt < 0.f && fabsf(cr) < -0.01f * dt) ? copysignf(3.14159265358979f, cr) + atanf(cr / dt)
                                                            : atan2f(cr, dt);
    const float ra2 = ax * ax + ay * ay, rb2 = bx * bx + by * by;
    const float s1 = (ax * dx + ay * dy) * ilen, s2 = s1 + len;
    // s2 log rb2 - s1 log ra2, through log1p when rb2 ~ ra2
    const float delta = (dx * (ax + bx) + dy * (ay + by)) / ra2;
    float lg;
    if (fabsf(delta) < 0.5f) {
        lg = s2 * log1pf(delta) + len * __logf(ra2);
    } else {
        const float la = ra2 > 0.f ? s1 * __logf(ra2) : 0.f;
        const float lb = rb2 > 0.f ? s2 * __logf(rb2) : 0.f;
        lg = lb - la;
    }
    return make_float2(0.5f * lg - len + cr * ilen * phi, phi);
}
// a x b from (hi, lo) end points and target: the products and differences in
// float-float, so that its sign tells the side of the curve to about 2^-46 of
// the coordinates
__device__ __noinline__ float cross_ff(float4 H, float4 L, float xh, float xl, float yh, float yl) {
    float axh, axl, ayh, ayl, bxh, bxl, byh, byl;
    diff2(H.x, L.x, xh, xl, axh, axl);
    diff2(H.y, L.y, yh, yl, ayh, ayl);
    diff2(H.z, L.z, xh, xl, bxh, bxl);
    diff2(H.w, L.w, yh, yl, byh, byl);
    const float p = __fmul_rn(axh, byh), q = __fmul_rn(ayh, bxh);
    const float pe = __fmaf_rn(axh, byh, -p), qe = __fmaf_rn(ayh, bxh, -q);
    float d, e;
    diff2(p, pe, q, qe, d, e);
    return d + (e + ((axh * byl + axl * byh) - (ayh * bxl + ayl * bxh)));
}
// the same in FP64, from the piece's end points and the target
__device__ __noinline__ float2 pair64(const double *__restrict__ P, double qx, double qy) {
    double il, ph;
    seg_ilog_phi_f64(qx, qy, P[0], P[1], P[2], P[3], false, il, ph);
    return make_float2((float)il, (float)ph);
}
// By the series in eta = (p2 - p1) / (2 (m - q)), m the midpoint, when the
// target is at least four lengths from m.  false: it is not.
__device__ __forceinline__ bool pair_series(float ax, float ay, float bx, float by, float len, float &ilog, float &phi) {
    const float mx = 0.5f * (ax + bx), my = 0.5f * (ay + by), r2 = mx * mx + my * my;
    const float dx = bx - ax, dy = by - ay, l2 = len * len;
    if (!(16.f * l2 < r2)) return false;
    const float h = __fdividef(0.5f, r2);
    const float ex = (dx * mx + dy * my) * h, ey = (dy * mx - dx * my) * h;
    const float zx = ex * ex - ey * ey, zy = 2.f * ex * ey;
    // s = zeta (1/6 + zeta (1/20 + zeta / 42)); atanh = eta (1 + zeta (1/3 + zeta (1/5 + zeta / 7)))
    float ux = 1.f / 6.f, uy = 0.f, vx = 1.f / 3.f, vy = 0.f;
    if (1600.f * l2 > r2) {   // else the terms of order zeta^2 are below 1e-8
        float tx = 1.f / 20.f + zx * (1.f / 42.f), ty = zy * (1.f / 42.f);
        ux += zx * tx - zy * ty;
        uy = zx * ty + zy * tx;
        tx = 1.f / 5.f + zx * (1.f / 7.f);
        ty = zy * (1.f / 7.f);
        vx += zx * tx - zy * ty;
        vy = zx * ty + zy * tx;
    }
    ilog = len * (0.5f * __logf(r2) - (zx * ux - zy * uy));
    const float wx = 1.f + (zx * vx - zy * vy), wy = zx * vy + zy * vx;
    phi = 2.f * (ex * wy + ey * wx);
    return true;
}
// whether the target is so close to the segment's interior that the sign of
// the FP32 cross product is not its side
__device__ __forceinline__ bool pair_beside(float ax, float ay, float bx, float by, float len, float cr) {
    return ax * bx + ay * by < 0.f && fabsf(cr) < kNearFallback * len * len;
}

// One complex expansion of three channels at z, Re sum_k C[k] z^k, k = lo .. P1 - 1
__device__ __forceinline__ void horner3(const float2 *__restrict__ C, int P1, int lo, float2 z, float2 &s0, float2 &s1,
                                        float2 &s2) {
    s0 = C[P1 - 1];
    s1 = C[2 * P1 - 1];
    s2 = C[3 * P1 - 1];
    for (int k = P1 - 2; k >= lo; --k) {
        s0 = fadd(fmul(s0, z), C[k]);
        s1 = fadd(fmul(s1, z), C[P1 + k]);
        s2 = fadd(fmul(s2, z), C[2 * P1 + k]);
    }
}

// The FP64 terms (few rectangles have any) are calls, so that they take no
// registers from the FP32 loops.
struct D3 {
    double v[3];
};
// The leaf's local expansion at (qx, qy) in FP64 (a leaf with large coefficients)
__device__ __noinline__ D3 l2p64(const EvalArgs32 &a, int leaf, double qx, double qy) {
    D3 h;
    const double iw = 1.0 / a.t64.cw[leaf];
    const double zx = (qx - a.t64.cc[2 * leaf]) * iw, zy = (qy - a.t64.cc[2 * leaf + 1]) * iw;
    const float4 *Lc = a.L64 + (size_t)leaf * 3 * a.P1;
    for (int ch = 0; ch < 3; ++ch) {
        double sx = 0.0, sy = 0.0;
        for (int k = a.P1 - 1; k >= 0; --k) {
            const double2 l = ff_value(Lc[ch * a.P1 + k]);
            const double nx = sx * zx - sy * zy + l.x;
            sy = sx * zy + sy * zx + l.y;
            sx = nx;
        }
        h.v[ch] = sx * kInv2Pi;
    }
    return h;
}

// The multipole expansion of cell src at (qx, qy) in FP64
__device__ __noinline__ D3 m2p64(const EvalArgs32 &a, int src, double qx, double qy) {
    D3 h;
    const int P1 = a.P1;
    const double iws = 1.0 / a.t64.cw[src];
    const double zx = (qx - a.t64.cc[2 * src]) * iws, zy = (qy - a.t64.cc[2 * src + 1]) * iws;
    const double d = 1.0 / (zx * zx + zy * zy);
    const double izx = zx * d, izy = -zy * d;
    const double lz = 0.5 * log(zx * zx + zy * zy) + log(a.t64.cw[src]);
    for (int ch = 0; ch < 3; ++ch) {
        const float4 *m = a.M64 + ((size_t)src * 3 + ch) * P1;
        double sx = 0.0, sy = 0.0;
        for (int k = P1 - 1; k >= 1; --k) {
            const double2 v = ff_value(m[k]);
            const double nx = sx * izx - sy * izy + v.x / k;
            sy = sx * izy + sy * izx + v.y / k;
            sx = nx;
        }
        h.v[ch] = ((sx * izx - sy * izy) - lz * ff_value(m[0]).x) * kInv2Pi;
    }
    return h;
}

// Piece i (a heavy one) at (qx, qy) in FP64
__device__ __noinline__ D3 p2p64(const EvalArgs32 &a, int i, double qx, double qy) {
    D3 h;
    const double *P = a.t64.pc + 4 * (size_t)i;
    const size_t s3 = 3 * (size_t)a.t64.pseg[i];
    double il, ph;
    seg_ilog_phi_f64(qx, qy, P[0], P[1], P[2], P[3], false, il, ph);
    const double wg = -a.t64.pw[i] * kInv2Pi;
    for (int ch = 0; ch < 3; ++ch) h.v[ch] = wg * (il * a.sb64[s3 + ch] + ph * a.mb64[s3 + ch]);
    return h;
}
__device__ __forceinline__ void add3(double h[3], const D3 &d) {
    for (int ch = 0; ch < 3; ++ch) h[ch] += d.v[ch];
}

// The rectangle's frame: its leaf's width scaled to one (the logarithms of
// the near field are then log(r / rho); near_centre_kernel has put the
// constant rest into L_0), its centre at the origin.
struct Frame {
    float iw, rho;                   // 1 / leaf width, leaf width (powers of two)
    float cxh, cxl, cyh, cyl;        // the centre, (hi, lo)
    float tx, ty;                    // the centre relative to the leaf's, in leaf widths
    float dxh, dxl, dyh, dyl;        // pixel size in leaf widths, (hi, lo)
    float hx, hy, R;                 // half extents in pixels, radius in leaf widths
};

// Piece f of the leaf's list: (hi, lo) end points in the frame and weights.
struct Piece {
    float x1h, y1h, x2h, y2h, x1l, y1l, x2l, y2l, len, sg[3], mg[3];
    int i;
    bool heavy;
};
// (hi, lo) of (a - b) iw, normalised: world coordinates' hi parts are rounded
// at 2^-24 of the canvas, so after their difference the lo part can be the
// larger one
__device__ __forceinline__ void frame_diff(float ah, float al, float bh, float bl, float iw, float &hi, float &lo) {
    float h, l;
    diff2(ah, al, bh, bl, h, l);
    const float s = __fadd_rn(h, l);
    hi = __fmul_rn(s, iw);
    lo = __fmul_rn(__fsub_rn(l, __fsub_rn(s, h)), iw);
}
__device__ __forceinline__ Piece load_piece(const EvalArgs32 &a, const Frame &F, int f) {
    Piece p;
    const DevTree32 &t = a.t;
    const int i = t.uf_idx[f];
    const float4 ph = t.pch[i], pl = t.pcl[i];
    frame_diff(ph.x, pl.x, F.cxh, F.cxl, F.iw, p.x1h, p.x1l);
    frame_diff(ph.y, pl.y, F.cyh, F.cyl, F.iw, p.y1h, p.y1l);
    frame_diff(ph.z, pl.z, F.cxh, F.cxl, F.iw, p.x2h, p.x2l);
    frame_diff(ph.w, pl.w, F.cyh, F.cyl, F.iw, p.y2h, p.y2l);
    p.len = __fmul_rn(t.plen[i], F.iw);
    const size_t s3 = 3 * (size_t)t.pseg[i];
    const float wgt = -t.pw[i] * kInv2PiF;
    for (int ch = 0; ch < 3; ++ch) {
        p.sg[ch] = (wgt * a.sb[s3 + ch]) * F.rho;
        p.mg[ch] = wgt * a.mb[s3 + ch];
    }
    p.i = i;
    p.heavy = a.heavy[i] != 0;
    return p;
}
// Whether a source is far is decided again wherever it is needed (the
// samples, the pieces of a list too long to stay staged, the FP64 terms) and
// has to come out the same each time, or a source at the threshold would be
// taken twice or not at all: every operation's rounding is written out, since
// the compiler may fuse a product and a sum in one place and not in another.
//
// whether all of the piece is at least the separation away from the centre
__device__ __forceinline__ bool piece_far(const Piece &p, const Frame &F) {
    const float dx = __fsub_rn(p.x2h, p.x1h), dy = __fsub_rn(p.y2h, p.y1h);
    const float s = -__fmaf_rn(p.x1h, dx, __fmul_rn(p.y1h, dy));   // foot of the centre, times the length
    const float l2 = __fmaf_rn(dx, dx, __fmul_rn(dy, dy));
    const float k = l2 > 0.f ? fminf(fmaxf(__fdiv_rn(s, l2), 0.f), 1.f) : 0.f;
    const float x = __fmaf_rn(k, dx, p.x1h), y = __fmaf_rn(k, dy, p.y1h);
    const float r = __fmaf_rn(1e-6f, p.len, __fmul_rn(p.heavy ? kSepBig : kSep, F.R));
    return __fmaf_rn(x, x, __fmul_rn(y, y)) >= __fmul_rn(r, r);
}
// whether cell src (list-3 entry e of the leaf) is far: its bounding circle
// at the separation, and the sampled circle outside 1.5 of its widths, where
// its multipole expansion converges as it does for list 3 itself
__device__ __forceinline__ bool cell_far(const EvalArgs32 &a, const Frame &F, int e, int src, bool big) {
    const float2 off = a.t.w_off[e];
    // centre to centre, in leaf widths
    const float dx = __fsub_rn(F.tx, __fmul_rn(off.x, F.iw)), dy = __fsub_rn(F.ty, __fmul_rn(off.y, F.iw));
    const float ws = __fdiv_rn(F.iw, a.t.iw[src]);
    const float d = __fsqrt_rn(__fmaf_rn(dx, dx, __fmul_rn(dy, dy)));
    return __fmaf_rn(-0.7072f, ws, d) >= __fmul_rn(big ? kSepBig : kSep, F.R) && d >= __fmaf_rn(1.5f, ws, F.R);
}

// A sampled rectangle's pixels come in quads +-x +-y around its centre, one
// of each in its upper right quarter: row and column of slot i (++, --, +-,
// -+) of quad q.  false where it is no pixel of its own (on the middle row or
// column and another slot's).
__device__ __forceinline__ bool quad_pixel(const RTile &tl, int q, int i, int &r, int &c) {
    const int nx2 = (tl.nc + 1) / 2, qr = q / nx2, qc = q - qr * nx2;
    const bool px = !(i & 1), py = i == 0 || i == 3;
    c = px ? tl.nc - 1 - qc : qc;
    r = py ? tl.nr - 1 - qr : qr;
    return (px || 2 * qc != tl.nc - 1) && (py || 2 * qr != tl.nr - 1);
}

// 2 pi times the multipole expansion of list-3 entry e (cell src) at (x, y) of the frame
__device__ __forceinline__ float3 m2p32(const EvalArgs32 &a, const Frame &F, int e, int src, float x, float y) {
    const float2 off = a.t.w_off[e];
    const float iws = a.t.iw[src];
    const float2 zz = make_float2(((x + F.tx) * F.rho - off.x) * iws, ((y + F.ty) * F.rho - off.y) * iws);
    const float2 iz = finv(zz);
    const float lz = 0.5f * __logf(zz.x * zz.x + zz.y * zz.y) + a.t.logw[src];
    const int P1 = a.P1;
    const float2 *Ms = a.M + (size_t)src * 3 * P1;
    float2 s0, s1, s2;
    horner3(Ms, P1, 1, iz, s0, s1, s2);
    return make_float3((s0.x * iz.x - s0.y * iz.y) - lz * Ms[0].x, (s1.x * iz.x - s1.y * iz.y) - lz * Ms[P1].x,
                       (s2.x * iz.x - s2.y * iz.y) - lz * Ms[2 * P1].x);
}

__device__ __forceinline__ void item(const EvalArgs32 &a, int it, BlockMem &B) {
    const unsigned full = 0xffffffffu;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const DevTree32 &t = a.t;
    const RTile tl = a.rects[it];
    const VpDev &vp = a.vps[tl.vp];   // read where it is needed (registers)
    const int leaf = tl.leaf, P1 = a.P1, npx = tl.nr * tl.nc;
    Frame F;
    F.iw = t.iw[leaf];
    F.rho = 1.f / F.iw;
    F.cxh = tl.cxh;
    F.cxl = tl.cxl;
    F.cyh = tl.cyh;
    F.cyl = tl.cyl;
    F.tx = tl.tx * F.iw;
    F.ty = tl.ty * F.iw;
    F.dxh = vp.dxh * F.iw;
    F.dxl = vp.dxl * F.iw;
    F.dyh = vp.dyh * F.iw;
    F.dyl = vp.dyl * F.iw;
    F.hx = 0.5f * (tl.nc - 1);
    F.hy = 0.5f * (tl.nr - 1);
    F.R = sqrtf(F.hx * F.hx * F.dxh * F.dxh + F.hy * F.hy * F.dyh * F.dyh);
    const bool hL = a.hL[leaf] != 0;
    const bool samp = npx >= kMinSampled && F.R >= kMinRadius && F.R <= (hL ? kMaxRadiusBig : kMaxRadius);
    const int f0 = t.uf_ptr[leaf], f1 = t.uf_ptr[leaf + 1], w0 = t.w_ptr[leaf], w1 = t.w_ptr[leaf + 1];
    constexpr int kChunk = kWarps * kStaged;
    const bool one = f1 - f0 <= kChunk;   // the near pieces are staged once
    const unsigned below = (1u << lane) - 1u;

    // ---- pieces: the near ones staged, the far ones sampled at this lane's
    // point of the circle; expansions sampled
    const float2 e = B.tw[lane];
    const float qx = F.R * e.x, qy = F.R * e.y;
    float u0 = 0.f, u1 = 0.f, u2 = 0.f;      // pieces
    float e0 = 0.f, e1 = 0.f, e2 = 0.f;      // expansions, times 2 pi
    double h[3] = {0.0, 0.0, 0.0};           // FP64 terms
    // flags: 1 FP64 terms among the samples, 2 FP64 terms at the pixels, 4 near pieces, 8 near list-3 cells
    int flags = samp ? (hL ? 1 : 0) : (hL ? 2 : 0) | 4 | (w1 > w0 ? 8 : 0);
    auto px64 = [&]() { return ((double)F.cxh + F.cxl) + (double)qx * F.rho; };   // the point in world units, FP64
    auto py64 = [&]() { return ((double)F.cyh + F.cyl) + (double)qy * F.rho; };
    int cnt = 0;
    for (int c0 = f0; c0 < f1; c0 += kChunk)
        for (int f = c0 + kStaged * warp; f < min(f1, c0 + kStaged * (warp + 1)); f += 32) {
            Piece p;
            bool far = false, near = false;
            p.heavy = false;
            if (f + lane < f1) {
                p = load_piece(a, F, f + lane);
                far = samp && piece_far(p, F);
                near = !far;
            }
            const unsigned mnear = __ballot_sync(full, near && !p.heavy), mfar = __ballot_sync(full, far && !p.heavy);
            unsigned mheavy = __ballot_sync(full, far && p.heavy);
            if (__any_sync(full, near && p.heavy)) flags |= 2 | 4;
            if (mnear) flags |= 4;
            if (one && near && !p.heavy) {
                float4 *o = B.pc[kStaged * warp + cnt + __popc(mnear & below)];
                o[0] = make_float4(p.x1h, p.y1h, p.x2h, p.y2h);
                o[1] = make_float4(p.x1l, p.y1l, p.x2l, p.y2l);
                o[2] = make_float4(p.len, p.sg[0], p.sg[1], p.sg[2]);
                o[3] = make_float4(p.mg[0], p.mg[1], p.mg[2], __int_as_float(p.i));
            }
            cnt += __popc(mnear);
            if (far && !p.heavy) {
                float4 *o = B.far[warp][__popc(mfar & below)];
                o[0] = make_float4(p.x1h, p.y1h, p.x2h, p.y2h);
                o[1] = make_float4(p.len, p.sg[0], p.sg[1], p.sg[2]);
                o[2] = make_float4(p.mg[0], p.mg[1], p.mg[2], 0.f);
            }
            __syncwarp();
            const int nf = __popc(mfar);
            for (int s = 0; s < nf; ++s) {
                const float4 g = B.far[warp][s][0], c = B.far[warp][s][1], d = B.far[warp][s][2];
                const float ax = g.x - qx, ay = g.y - qy, bx = g.z - qx, by = g.w - qy;
                float ilog, phi;
                if (!pair_series(ax, ay, bx, by, c.x, ilog, phi)) {
                    // a far piece is 1e-6 of its length away at least: the
                    // product's own rounding is all that can matter
                    const float p2 = __fmul_rn(ay, bx);
                    const float2 w = pair_closed(ax, ay, bx, by, c.x, __fmaf_rn(ax, by, -p2) + __fmaf_rn(-ay, bx, p2));
                    ilog = w.x;
                    phi = w.y;
                }
                u0 = fmaf(ilog, c.y, fmaf(phi, d.x, u0));
                u1 = fmaf(ilog, c.z, fmaf(phi, d.y, u1));
                u2 = fmaf(ilog, c.w, fmaf(phi, d.z, u2));
            }
            while (mheavy) {
                const int src = __ffs(mheavy) - 1;
                mheavy &= mheavy - 1;
                add3(h, p2p64(a, __shfl_sync(full, p.i, src), px64(), py64()));
                flags |= 1;
            }
            __syncwarp();
        }
    if (samp) {
        if (warp == 0) {   // L2P (Eq. 64)
            if (hL) {
                add3(h, l2p64(a, leaf, px64(), py64()));
            } else {
                float2 s0, s1, s2;
                horner3(a.L + (size_t)leaf * 3 * P1, P1, 0, make_float2(qx + F.tx, qy + F.ty), s0, s1, s2);
                e0 = s0.x;
                e1 = s1.x;
                e2 = s2.x;
            }
        }
        // M2P of the far list-3 cells (Eq. 61), from the last warp on (the first has the L2P)
        for (int k = w0 + kWarps - 1 - warp; k < w1; k += kWarps) {
            const int src = t.w_idx[k];
            const bool hM = a.hM[src] != 0;
            if (!cell_far(a, F, k, src, hM)) {
                flags |= hM ? 2 | 8 : 8;
                continue;
            }
            if (hM) {
                add3(h, m2p64(a, src, px64(), py64()));
                flags |= 1;
                continue;
            }
            const float3 w = m2p32(a, F, k, src, qx, qy);
            e0 += w.x;
            e1 += w.y;
            e2 += w.z;
        }
        float2 *v = B.v[warp][lane];
        v[0] = add_expansion(u0, e0);
        v[1] = add_expansion(u1, e1);
        v[2] = add_expansion(u2, e2);
        if (flags & 1)
            for (int ch = 0; ch < 3; ++ch) B.h[warp][lane][ch] = h[ch];
    } else if (w1 > w0) {
        for (int k = w0 + lane; k < w1; k += 32)
            if (a.hM[t.w_idx[k]]) flags |= 2;
        flags = __reduce_or_sync(full, flags);
    }
    if (lane == 0) {
        B.cnt[warp] = one ? cnt : 0;
        B.flags[warp] = flags;
    }
    __syncthreads();
    const int big4 = (B.flags[0] & 1) | (B.flags[1] & 1) << 1 | (B.flags[2] & 1) << 2 | (B.flags[3] & 1) << 3;
    flags = B.flags[0] | B.flags[1] | B.flags[2] | B.flags[3];
    const bool big = samp && (flags & 1), flag64 = flags & 2, any_near = flags & 4, any_w = flags & 8;

    // ---- coefficients, four per warp: each warp adds up the samples, takes a
    // value near their mean off in (hi, lo) and transforms the differences
    float mean[3] = {0.f, 0.f, 0.f}, rest[3] = {0.f, 0.f, 0.f};   // c_0, (hi, lo)
    int kmax = 1;
    if (samp) {
        float4 d;
        {
            float dd[3];
            double h2[3] = {0.0, 0.0, 0.0};
            for (int ch = 0; ch < 3; ++ch) {
                float2 v = B.v[0][lane][ch];
                for (int wi = 1; wi < kWarps; ++wi) {
                    const float2 w = B.v[wi][lane][ch], z = two_sum(v.x, w.x);
                    v = make_float2(z.x, z.y + (v.y + w.y));
                }
                if (big) {
                    h2[ch] = (double)v.x + v.y;
                    for (int wi = 0; wi < kWarps; ++wi)
                        if (big4 >> wi & 1) h2[ch] += B.h[wi][lane][ch];
                    split2(h2[ch], v.x, v.y);
                }
                float s = v.x;
                for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(full, s, o);
                mean[ch] = s * (1.f / kSamples);
                const float2 z = two_sum(v.x, -mean[ch]);
                dd[ch] = z.x + (z.y + v.y);
                if (big && warp == 0) B.dv[lane][ch] = h2[ch] - (double)mean[ch];
                s = dd[ch];
                for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(full, s, o);
                rest[ch] = s * (1.f / kSamples);
            }
            d = make_float4(dd[0], dd[1], dd[2], 0.f);
        }
        B.d[warp][lane] = d;
        __syncwarp();
        // lane = (coefficient k of the warp's four, eighth of the samples)
        const int k = 4 * warp + (lane & 3);
        float ca[3] = {0.f, 0.f, 0.f}, cb[3] = {0.f, 0.f, 0.f};
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const int j = (lane >> 2) + 8 * i;
            const float2 w = B.tw[(k * j) & 31];
            const float4 g = B.d[warp][j];
            ca[0] = fmaf(g.x, w.x, ca[0]);
            ca[1] = fmaf(g.y, w.x, ca[1]);
            ca[2] = fmaf(g.z, w.x, ca[2]);
            cb[0] = fmaf(g.x, w.y, cb[0]);
            cb[1] = fmaf(g.y, w.y, cb[1]);
            cb[2] = fmaf(g.z, w.y, cb[2]);
        }
        for (int ch = 0; ch < 3; ++ch) {
            for (int o = 4; o < 32; o <<= 1) {
                ca[ch] += __shfl_xor_sync(full, ca[ch], o);
                cb[ch] += __shfl_xor_sync(full, cb[ch], o);
            }
            ca[ch] *= 2.f / kSamples;
            cb[ch] *= 2.f / kSamples;
        }
        if (lane < 4) {
            B.cf[k][0] = make_float4(ca[0], cb[0], ca[1], cb[1]);
            B.cf[k][1] = make_float4(ca[2], cb[2], 0.f, 0.f);
        }
        if (big && warp == 0) {   // FP64 coefficients
            const int k = lane & 15, j0 = lane & 16;
            double da[3] = {0.0, 0.0, 0.0}, db[3] = {0.0, 0.0, 0.0};
            for (int j = j0; j < j0 + 16; ++j) {
                const double wx = cos32(k * j), wy = cos32(k * j + 24);   // cos(x - pi / 2) = sin x
                for (int ch = 0; ch < 3; ++ch) {
                    da[ch] += B.dv[j][ch] * wx;
                    db[ch] += B.dv[j][ch] * wy;
                }
            }
            for (int ch = 0; ch < 3; ++ch) {
                const double sc = k == 0 ? 1.0 / kSamples : 2.0 / kSamples;
                da[ch] = (da[ch] + __shfl_xor_sync(full, da[ch], 16)) * sc;
                db[ch] = (db[ch] + __shfl_xor_sync(full, db[ch], 16)) * sc;
                if (lane < 16) {
                    B.cd[k][2 * ch] = da[ch];
                    B.cd[k][2 * ch + 1] = db[ch];
                }
            }
        }
        __syncthreads();
        // Terms whose sum is below a sixteenth of the FP32 rounding of the
        // value are left out; every channel has its own value, which may be
        // far smaller than another's.
        bool need = false;
        {
            const float4 c0 = B.cf[lane & 15][0], c1 = B.cf[lane & 15][1];
            const bool is0 = (lane & 15) == 0;
            const float mag[3] = {fabsf(c0.x) + fabsf(c0.y), fabsf(c0.z) + fabsf(c0.w), fabsf(c1.x) + fabsf(c1.y)};
#pragma unroll
            for (int ch = 0; ch < 3; ++ch) {
                float tail = is0 ? 0.f : mag[ch];   // sum over k' >= k
                for (int o = 1; o < 16; o <<= 1) {
                    const float x = __shfl_down_sync(full, tail, o, 16);
                    if ((lane & 15) + o < 16) tail += x;
                }
                need |= tail > 4e-9f * (__shfl_sync(full, tail, 0) + fabsf(mean[ch]));
            }
        }
        const unsigned keep = __ballot_sync(full, (lane & 15) > 0 && need) & 0xffffu;
        kmax = keep ? 32 - __clz(keep) : 1;
    }

    // ---- the pixels, one per lane (more would not fit the instruction cache:
    // the loop over the near pieces is a few dozen instructions).  Each warp
    // takes a quarter of the rectangle; with fewer than 32 pixels in it, ng
    // lanes take the pixels and 32 / ng such sets every (32 / ng)th source
    // each, summed at the end.
    const int nall = samp ? ((tl.nc + 1) / 2) * ((tl.nr + 1) / 2) : npx;   // quads or pixels
    const int share = (nall + kWarps - 1) / kWarps, first = warp * share, mine = min(share, nall - first);
    const int per = samp ? 4 * share : share;   // pixels of a warp
    const int ng = per > 16 ? 32 : per > 8 ? 16 : per > 4 ? 8 : per > 2 ? 4 : per;   // 1 and 2 as they are
    const int nsub = 32 / ng, sub = lane / ng;
    for (int q0 = 0; q0 < share; q0 += (samp ? 32 : share)) {
        const int G = samp ? max(1, min(32, mine - q0)) : max(1, mine), nP = samp ? 4 * min(32, share - q0) : share;
        const bool some = mine - q0 > 0;
        if (samp && !big && some) {
            // Re sum c_k z^k for z, -z, conj z, -conj z at once: even and odd
            // terms, and the real and imaginary parts' terms, apart
            int r, c;
            quad_pixel(tl, first + q0 + min(lane, G - 1), 0, r, c);
            const float iR = 1.f / F.R, zx = ((float)c - F.hx) * F.dxh * iR, zy = ((float)r - F.hy) * F.dyh * iR;
            float px = zx, py = zy;
            float Ae[3] = {0, 0, 0}, Ao[3] = {0, 0, 0}, Be[3] = {0, 0, 0}, Bo[3] = {0, 0, 0};
            for (int k = 1; k < kmax; k += 2) {
                float4 cc = B.cf[k][0];
                float2 d = *reinterpret_cast<const float2 *>(&B.cf[k][1]);
                Ao[0] = fmaf(cc.x, px, Ao[0]);
                Bo[0] = fmaf(cc.y, py, Bo[0]);
                Ao[1] = fmaf(cc.z, px, Ao[1]);
                Bo[1] = fmaf(cc.w, py, Bo[1]);
                Ao[2] = fmaf(d.x, px, Ao[2]);
                Bo[2] = fmaf(d.y, py, Bo[2]);
                float nx = fmaf(px, zx, -py * zy);
                py = fmaf(px, zy, py * zx);
                px = nx;
                if (k + 1 >= kmax) break;
                cc = B.cf[k + 1][0];
                d = *reinterpret_cast<const float2 *>(&B.cf[k + 1][1]);
                Ae[0] = fmaf(cc.x, px, Ae[0]);
                Be[0] = fmaf(cc.y, py, Be[0]);
                Ae[1] = fmaf(cc.z, px, Ae[1]);
                Be[1] = fmaf(cc.w, py, Be[1]);
                Ae[2] = fmaf(d.x, px, Ae[2]);
                Be[2] = fmaf(d.y, py, Be[2]);
                nx = fmaf(px, zx, -py * zy);
                py = fmaf(px, zy, py * zx);
                px = nx;
            }
#pragma unroll
            for (int ch = 0; ch < 3; ++ch) {
                const float p = Ae[ch] + Ao[ch], n = Ae[ch] - Ao[ch], s = Be[ch] + Bo[ch], u = Be[ch] - Bo[ch];
                B.pv[warp][ch][lane] = p + s;
                B.pv[warp][3 + ch][lane] = n + u;
                B.pv[warp][6 + ch][lane] = p - s;
                B.pv[warp][9 + ch][lane] = n - u;
            }
        }
        __syncwarp();
        // nP and share are the same for all warps: the loop's barriers match
        for (int p0 = 0; p0 < nP; p0 += ng) {
            int pi = p0 + lane % ng, r, c, slot = 0, quad = 0;
            bool on = some && pi < (samp ? 4 * G : G);
            pi = min(pi, (samp ? 4 * G : G) - 1);
            const int base = some ? first + (samp ? q0 : 0) : 0;
            if (samp) {
                slot = pi / G;
                quad = pi - slot * G;
                on = quad_pixel(tl, base + quad, slot, r, c) && on;
            } else {
                r = (base + pi) / tl.nc;
                c = base + pi - r * tl.nc;
            }
            float xh, xl, yh, yl;
            u0 = u1 = u2 = 0.f;
            {
                const float ox = (float)c - F.hx, oy = (float)r - F.hy;   // exact (half integers)
                xh = ox * F.dxh;
                xl = fmaf(ox, F.dxl, fmaf(ox, F.dxh, -xh));
                yh = oy * F.dyh;
                yl = fmaf(oy, F.dyl, fmaf(oy, F.dyh, -yh));
            }
            r += tl.r0;
            c += tl.c0;
            // P2P of the near pieces
            if (any_near)
                for (int c0 = f0; c0 < f1; c0 += kChunk) {
                    if (!one) {   // too many pieces to stay staged: again, chunk by chunk
                        __syncthreads();
                        int n = 0;
                        for (int f = c0 + kStaged * warp; f < min(f1, c0 + kStaged * (warp + 1)); f += 32) {
                            Piece p;
                            bool take = false;
                            if (f + lane < f1) {
                                p = load_piece(a, F, f + lane);
                                take = !p.heavy && !(samp && piece_far(p, F));
                            }
                            const unsigned mk = __ballot_sync(full, take);
                            if (take) {
                                float4 *o = B.pc[kStaged * warp + n + __popc(mk & below)];
                                o[0] = make_float4(p.x1h, p.y1h, p.x2h, p.y2h);
                                o[1] = make_float4(p.x1l, p.y1l, p.x2l, p.y2l);
                                o[2] = make_float4(p.len, p.sg[0], p.sg[1], p.sg[2]);
                                o[3] = make_float4(p.mg[0], p.mg[1], p.mg[2], __int_as_float(p.i));
                            }
                            n += __popc(mk);
                        }
                        if (lane == 0) B.cnt[warp] = n;
                        __syncthreads();
                    }
                    for (int wi = 0; wi < kWarps; ++wi) {
                        const int n = some ? B.cnt[wi] : 0;
                        for (int s = sub; s < n; s += nsub) {
                            const float4 *o = B.pc[kStaged * wi + s];
                            const float4 A = o[0], Bl = o[1], C = o[2], D = o[3];
                            const float ax = (A.x - xh) + (Bl.x - xl), ay = (A.y - yh) + (Bl.y - yl);
                            const float bx = (A.z - xh) + (Bl.z - xl), by = (A.w - yh) + (Bl.w - yl);
                            float ilog, phi;
                            if (!pair_series(ax, ay, bx, by, C.x, ilog, phi)) {
                                float2 w;
                                float cr = ax * by - ay * bx;
                                bool exact = false;
                                if (pair_beside(ax, ay, bx, by, C.x, cr)) {
                                    cr = cross_ff(A, Bl, xh, xl, yh, yl);
                                    exact = fabsf(cr) < a.side * F.iw * C.x;
                                }
                                if (exact) {   // closer than the (hi, lo) coordinates resolve
                                    w = pair64(a.t64.pc + 4 * (size_t)__float_as_int(D.w), vp.x0 + (c + 0.5) * vp.dx,
                                               vp.y0 + (r + 0.5) * vp.dy);
                                    // world units to the scaled frame: il / rho - len' log(rho)
                                    w.x = w.x * F.iw + C.x * __logf(F.iw);
                                } else {
                                    w = pair_closed(ax, ay, bx, by, C.x, cr);
                                }
                                ilog = w.x;
                                phi = w.y;
                            }
                            u0 = fmaf(ilog, C.y, fmaf(phi, D.x, u0));
                            u1 = fmaf(ilog, C.z, fmaf(phi, D.y, u1));
                            u2 = fmaf(ilog, C.w, fmaf(phi, D.z, u2));
                        }
                    }
                    if (one) break;
                }
            __syncwarp();
            // expansions at the pixels: the near list-3 cells, and without
            // samples the local one.  They have a sum of their own (times
            // 2 pi), added to the pieces' at the end: the two may cancel.
            e0 = e1 = e2 = 0.f;
            if (any_w)
                for (int k = w0 + sub; k < w1; k += nsub) {
                    const int src = t.w_idx[k];
                    if (a.hM[src] || (samp && cell_far(a, F, k, src, false))) continue;
                    const float3 w = m2p32(a, F, k, src, xh, yh);
                    e0 += w.x;
                    e1 += w.y;
                    e2 += w.z;
                }
            __syncwarp();
            if (!samp && !hL && sub == nsub - 1) {
                float2 s0, s1, s2;
                horner3(a.L + (size_t)leaf * 3 * P1, P1, 0, make_float2(xh + F.tx, yh + F.ty), s0, s1, s2);
                e0 += s0.x;
                e1 += s1.x;
                e2 += s2.x;
            }
            __syncwarp();
            for (int o = ng; o < 32; o <<= 1) {
                u0 += __shfl_xor_sync(full, u0, o);
                u1 += __shfl_xor_sync(full, u1, o);
                u2 += __shfl_xor_sync(full, u2, o);
                e0 += __shfl_xor_sync(full, e0, o);
                e1 += __shfl_xor_sync(full, e1, o);
                e2 += __shfl_xor_sync(full, e2, o);
            }
            float pv0 = 0.f, pv1 = 0.f, pv2 = 0.f;   // the polynomial less the mean
            if (samp && !big) {
                const float *pv = &B.pv[warp][3 * slot][quad];
                pv0 = rest[0] + pv[0];
                pv1 = rest[1] + pv[32];
                pv2 = rest[2] + pv[64];
            }
            // FP64 terms
            if (flag64 || big) {
                h[0] = h[1] = h[2] = 0.0;
                const double qx64 = vp.x0 + (c + 0.5) * vp.dx, qy64 = vp.y0 + (r + 0.5) * vp.dy;
                if (big) {
                    const double sc = (double)F.iw / F.R;
                    const double zx = ((double)(c - tl.c0) - F.hx) * vp.dx * sc, zy = ((double)(r - tl.r0) - F.hy) * vp.dy * sc;
                    double wx = 1.0, wy = 0.0;
                    for (int k = 0; k < kCoefs; ++k) {
                        for (int ch = 0; ch < 3; ++ch) h[ch] += B.cd[k][2 * ch] * wx + B.cd[k][2 * ch + 1] * wy;
                        const double nx = wx * zx - wy * zy;
                        wy = wx * zy + wy * zx;
                        wx = nx;
                    }
                }
                if (!samp && hL) add3(h, l2p64(a, leaf, qx64, qy64));
                if (flag64 && any_w)
                    for (int k = w0; k < w1; ++k) {
                        const int src = t.w_idx[k];
                        if (!a.hM[src] || (samp && cell_far(a, F, k, src, true))) continue;
                        add3(h, m2p64(a, src, qx64, qy64));
                    }
                if (flag64 && any_near)
                    for (int f = f0; f < f1; f += 32) {
                        bool take = false;
                        int idx = 0;
                        if (f + lane < f1) {
                            idx = t.uf_idx[f + lane];
                            take = a.heavy[idx] != 0;
                            if (take && samp) take = !piece_far(load_piece(a, F, f + lane), F);
                        }
                        unsigned mk = __ballot_sync(full, take);
                        while (mk) {
                            const int src = __ffs(mk) - 1;
                            mk &= mk - 1;
                            add3(h, p2p64(a, __shfl_sync(full, idx, src), qx64, qy64));
                        }
                    }
                u0 = (float)(((double)u0 + (double)e0 * kInv2Pi) + (h[0] + ((double)mean[0] + pv0)));
                u1 = (float)(((double)u1 + (double)e1 * kInv2Pi) + (h[1] + ((double)mean[1] + pv1)));
                u2 = (float)(((double)u2 + (double)e2 * kInv2Pi) + (h[2] + ((double)mean[2] + pv2)));
            } else {   // without samples the mean is zero
                u0 = add_parts(mean[0], u0, e0, pv0);
                u1 = add_parts(mean[1], u1, e1, pv1);
                u2 = add_parts(mean[2], u2, e2, pv2);
            }
            if (on && sub == 0) {
                const size_t o = 3 * ((size_t)vp.offset + (size_t)r * vp.width + c);
                if (a.rgb) {
                    if (a.rgb_dtype == DC_F64) {
                        double *d = static_cast<double *>(a.rgb) + o;
                        d[0] = u0;
                        d[1] = u1;
                        d[2] = u2;
                    } else {
                        float *d = static_cast<float *>(a.rgb) + o;
                        d[0] = u0;
                        d[1] = u1;
                        d[2] = u2;
                    }
                }
                if (a.rgb8) {
                    a.rgb8[o] = quant8(u0);
                    a.rgb8[o + 1] = quant8(u1);
                    a.rgb8[o + 2] = quant8(u2);
                }
            }
        }
        __syncwarp();
    }
}

// Persistent: blocks take rectangles from the counter in list order (listed by
// decreasing estimated cost).
__global__ void __launch_bounds__(32 * kWarps, kBlocksPerSM) render32_kernel(const __grid_constant__ EvalArgs32 a) {
    __shared__ BlockMem B;
    if (threadIdx.x < 32) {
        float s, c;
        sincospif((float)threadIdx.x * 0.0625f, &s, &c);
        B.tw[threadIdx.x] = make_float2(c, s);
    }
    if (threadIdx.x == 0) B.next = atomicAdd(a.queue, 1);
    __syncthreads();
    while (true) {
        const int it = B.next;
        if (it >= a.n_items) break;
        __syncthreads();   // the last rectangle's shared memory and B.next have been read
        if (threadIdx.x == 0) B.next = atomicAdd(a.queue, 1);
        item(a, it, B);
        __syncthreads();
    }
}

}  // namespace rtiles
