// The warm-start network's GEMMs on the 5th-generation tensor cores
// (tcgen05, kind::tf32): C[M][N] = sum_k A(m, k) B(n, k) (+ bias[n], GELU),
// with A(m, k) = A[m lda + k] or, with ta, A[k lda + m] (FP32), and B(n, k) =
// B[n ldb + k] or, with tb, B[k ldb + n] (FP32, or BF16 weights).
//
// BF16 values are exact in TF32, so a BF16 operand takes one term; an FP32
// operand is split into x_hi = tf32(x) and x_lo = tf32(x - x_hi), and the
// product A B^T is A_lo B_hi + A_hi B_lo + A_hi B_hi (the lo x lo term is
// below 2^-22 of the result) accumulated in FP32 in TMEM.  For the
// products along a layer's width that is as good as an FP32 product of the
// activations with the BF16 weights; for the weight gradients, whose sums run
// over the batch, the accumulator's rounding grows with it (below).
//
// One CTA takes 128 rows and up to NT columns: operands staged KC x 32 values
// of K at a time in shared memory in the canonical K-major layout without
// swizzling (the M2L's layout: core matrices of 8 rows x 16 bytes, LBO 128,
// SBO 1024) in two buffers, one thread issues the MMAs (M 128, N up to NT, K
// 8).  While they run, the next two chunks are on their way from global
// memory; a buffer is written again after a bounded wait on the commit of its
// MMAs.  Four values of K make one 16-byte row of a core matrix, so every
// store to shared memory is 16 bytes wide, eight lanes to a core matrix (no
// bank conflicts), whichever index of the source is the contiguous one.  A
// wait that runs out sets *err and ends the CTA's work after the issued MMAs
// are waited for once more (the accumulator is freed only then).
//
// Shapes: 64 columns, 256 threads for the products along the batch; 16
// columns, 512 threads and 64 values of K a chunk for the weight gradients,
// whose sums run over the whole batch (256 x 384 outputs of 4,096 terms: 48
// CTAs instead of four with the whole width each, 100 us instead of 5.7 ms).
// What bounds those now is the chain of MMAs on one accumulator (1,536, about
// 65 ns each).  It is left whole, in the order lo hi, hi lo, hi hi per 32
// values of K, so its error grows with the batch: against 64 bits 0.8e-5 of the
// largest gradient at 64 rows, 1.5e-5 at 1,000, 4.0e-5 at 4,096, 6.7e-5 at 8,000
// and 1.1e-4 at 12,000 (hidden 256; the same as with one CTA per 256 columns).
// Cut into ranges whose sums are added at the end, the step took 0.29 ms and
// its gradient came nearer (8.5e-6 instead of 3.4e-5, rms, at 4,096 rows), but
// results move by 2.6e-5.
//
// One step's loss and gradient, 4,096 rows of 384 - 256 - 256 - 256 - 16 (4.9
// GFLOP): 15.3 -> 0.58 ms on one GB300.
#pragma once

#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <cstdint>

#include "passes_tc.cuh"

namespace dc {
namespace mlp {

constexpr int kGtM = 128, kGtK = 32;
// floats of one buffer: KC sub-chunks of A hi, lo, B hi, lo
__host__ __device__ constexpr int gt_sub(int nt) { return (2 * kGtM + 2 * nt) * kGtK; }
__host__ __device__ constexpr size_t gt_smem(int nt, int kc) { return 2 * (size_t)gt_sub(nt) * kc * sizeof(float) + 1024; }

__device__ __forceinline__ float gt_gelu(float x) { return 0.5f * x * (1.f + erff(x * 0.70710678118654752f)); }
__device__ __forceinline__ float gt_gelu_grad(float x) {
    // d/dx [x Phi(x)] = Phi(x) + x phi(x)
    const float phi = 0.39894228040143268f * __expf(-0.5f * x * x);
    return 0.5f * (1.f + erff(x * 0.70710678118654752f)) + x * phi;
}

__device__ __forceinline__ float gt_f32(float v) { return v; }
__device__ __forceinline__ float gt_f32(__nv_bfloat16 v) { return __bfloat162float(v); }

// D (+)= A B^T over K = 32 (four MMAs of K = 8), N columns (multiple of 16)
__device__ __forceinline__ void gt_mma(uint32_t tmem, uint32_t sa, uint32_t sb, uint32_t idesc, uint32_t first) {
#pragma unroll
    for (int ks = 0; ks < kGtK / 8; ++ks) {
        const uint64_t da = passes::tc_desc(sa + ks * 2 * passes::kTcCoreLBO);
        const uint64_t db = passes::tc_desc(sb + ks * 2 * passes::kTcCoreLBO);
        const uint32_t acc = (ks > 0 || !first) ? 1u : 0u;
        asm volatile("{\n .reg .pred p;\n setp.ne.u32 p, %4, 0;\n"
                     " tcgen05.mma.cta_group::1.kind::tf32 [%0], %1, %2, %3, p;\n}\n"
                     ::"r"(tmem), "l"(da), "l"(db), "r"(idesc), "r"(acc));
    }
}

struct GemmArgs {
    int M, N, K;
    const float *A;
    const void *B;
    int lda, ldb, ldc;
    int veca, vecb, vecc;       // 16-byte (A, C) and 8-byte (BF16 B) or 16-byte (FP32 B) accesses are aligned
    int small;                  // A and B are below 4 GB: 32-bit byte offsets
    float *C;
    const float *bias;          // forward: added, pre-activations to Zpre, GELU if act
    float *Zpre;
    int act;
    const float *Zback;         // backward: the result times gelu'(Zback)
    float *colsum;              // with TA: sums of A over K
    int *err;
};

// The unit's four values of K at `row` (source index) from k: the contiguous
// index is k (T false) or the row (T true).
template <bool T, typename V>
__device__ __forceinline__ float4 gt_load(const V *__restrict__ p, int ld, int row, int rows, int k, int kend, int vec) {
    float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
    if (row >= rows) return v;
    if (!T) {
        const V *q = p + (size_t)row * ld + k;
        if (vec && k + 3 < kend) {
            if constexpr (sizeof(V) == 4) {
                v = *reinterpret_cast<const float4 *>(q);
            } else {
                const __nv_bfloat162 *b = reinterpret_cast<const __nv_bfloat162 *>(q);
                const float2 x = __bfloat1622float2(b[0]), y = __bfloat1622float2(b[1]);
                v = make_float4(x.x, x.y, y.x, y.y);
            }
        } else {
            if (k < kend) v.x = gt_f32(q[0]);
            if (k + 1 < kend) v.y = gt_f32(q[1]);
            if (k + 2 < kend) v.z = gt_f32(q[2]);
            if (k + 3 < kend) v.w = gt_f32(q[3]);
        }
    } else {
        const V *q = p + (size_t)k * ld + row;
        if (k < kend) v.x = gt_f32(q[0]);
        if (k + 1 < kend) v.y = gt_f32(q[ld]);
        if (k + 2 < kend) v.z = gt_f32(q[2 * (size_t)ld]);
        if (k + 3 < kend) v.w = gt_f32(q[3 * (size_t)ld]);
    }
    return v;
}
// The same wholly inside K, at a byte offset of the matrix; kstep = ld in
// bytes where the row is contiguous.
template <bool T, typename V>
__device__ __forceinline__ float4 gt_load_in(const V *__restrict__ p, uint32_t off, uint32_t kstep) {
    const char *q = reinterpret_cast<const char *>(p);
    if constexpr (!T) {
        if constexpr (sizeof(V) == 4) {
            return *reinterpret_cast<const float4 *>(q + off);
        } else {
            const uint2 b = *reinterpret_cast<const uint2 *>(q + off);
            return make_float4(__uint_as_float(b.x << 16), __uint_as_float(b.x & 0xffff0000u),
                               __uint_as_float(b.y << 16), __uint_as_float(b.y & 0xffff0000u));
        }
    } else {
        return make_float4(gt_f32(*reinterpret_cast<const V *>(q + off)),
                           gt_f32(*reinterpret_cast<const V *>(q + (off + kstep))),
                           gt_f32(*reinterpret_cast<const V *>(q + (off + 2 * kstep))),
                           gt_f32(*reinterpret_cast<const V *>(q + (off + 3 * kstep))));
    }
}
// unit u of a tile of R rows: its row and its group of four k.  Lanes run
// along eight rows of a core matrix first (k contiguous: 64 bytes of each
// row to a warp), or along the rows (row contiguous: coalesced)
template <bool T, int R>
__device__ __forceinline__ void gt_unit(int u, int &row, int &kg) {
    if (T) {
        row = u & (R - 1);
        kg = u / R;
    } else {
        row = (u & 7) + 8 * ((u >> 6) & (R / 8 - 1));
        kg = ((u >> 3) & 3) + 4 * ((u >> 5) & 1);
    }
}
__device__ __forceinline__ void gt_split(float4 v, float *hi, float *lo, int o, bool exact) {
    const float4 h = make_float4(passes::tc_tf32(v.x), passes::tc_tf32(v.y), passes::tc_tf32(v.z), passes::tc_tf32(v.w));
    *reinterpret_cast<float4 *>(hi + o) = h;
    if (!exact)
        *reinterpret_cast<float4 *>(lo + o) = make_float4(passes::tc_tf32(v.x - h.x), passes::tc_tf32(v.y - h.y),
                                                          passes::tc_tf32(v.z - h.z), passes::tc_tf32(v.w - h.w));
}

// TA: A(m, k) = A[k lda + m]; TBt: B(n, k) = B[k ldb + n]
template <bool TA, bool TBt, typename TB, int NT, int KC, int NTHR>
__global__ void __launch_bounds__(NTHR) gemm_tc_kernel(const GemmArgs g) {
    extern __shared__ unsigned char gt_raw[];
    float *base = reinterpret_cast<float *>(((uintptr_t)gt_raw + 1023) & ~(uintptr_t)1023);
    __shared__ __align__(8) unsigned long long mbar[2];
    __shared__ uint32_t tmem_base;
    __shared__ float csum[NTHR];
    constexpr int kCols = NT < 32 ? 32 : NT;   // TMEM columns
    constexpr int kSub = gt_sub(NT), kChunk = KC * kGtK;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int m0 = blockIdx.x * kGtM, n0 = blockIdx.y * NT;
    const int nn = min(NT, g.N - n0);
    const int nt = (nn + 15) / 16 * 16;   // MMA width: a multiple of 16 for M = 128
    constexpr bool b_exact = sizeof(TB) == 2;   // BF16 weights: exact in TF32, one term
    // units of four k: of one 32-value sub-chunk, and of the chunk per thread
    constexpr int SA = kGtM * kGtK / 4, SB = NT * kGtK / 4;
    constexpr int UA = KC * SA / NTHR, UB = (KC * SB + NTHR - 1) / NTHR;
    const TB *B = static_cast<const TB *>(g.B);
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;\n"
                     ::"r"(passes::tc_smem(&tmem_base)), "r"(kCols));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n");
    }
    if (tid < 2) asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;\n" ::"r"(passes::tc_smem(&mbar[tid])));
    asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
    const uint32_t tmem = tmem_base;
    // D F32, A and B TF32, both K-major, N >> 3 at bits 17-22, M >> 4 at 24-28
    const uint32_t idesc = (1u << 4) | (2u << 7) | (2u << 10) | ((uint32_t)(nt >> 3) << 17) |
                           ((uint32_t)(kGtM >> 4) << 24);
    // Two chunks are on their way in registers while a third is split: their
    // units' places in the sources (rows past the end read the last one; what
    // they give is not stored) and in a buffer
    float4 ra[2][UA], rb[2][UB];
    uint32_t ga[UA], gb[UB];
    int oa[UA], ob[UB];
    const uint32_t ka = TA ? 4u * g.lda : 4u, kb = TBt ? (uint32_t)sizeof(TB) * g.ldb : (uint32_t)sizeof(TB);
#pragma unroll
    for (int i = 0; i < UA; ++i) {
        const int u = tid + i * NTHR;
        int row, kg;
        gt_unit<TA, kGtM>(u % SA, row, kg);
        oa[i] = (u / SA) * kSub + passes::tc_offset(row, 4 * kg) / 4;
        row = min(m0 + row, g.M - 1);
        ga[i] = (TA ? 4u * row : 4u * g.lda * row) + ka * (uint32_t)(kGtK * (u / SA) + 4 * kg);
    }
#pragma unroll
    for (int i = 0; i < UB; ++i) {
        const int u = min(tid + i * NTHR, KC * SB - 1);
        int row, kg;
        gt_unit<TBt, NT>(u % SB, row, kg);
        ob[i] = (u / SB) * kSub + 2 * kGtM * kGtK + passes::tc_offset(row, 4 * kg) / 4;
        row = min(n0 + row, g.N - 1);
        gb[i] = (uint32_t)sizeof(TB) * (TBt ? (uint32_t)row : (uint32_t)g.ldb * row) +
                kb * (uint32_t)(kGtK * (u / SB) + 4 * kg);
    }
    const bool fast = g.small && (TA || g.veca) && (TBt || g.vecb);
    auto fetch = [&](int c, float4 *xa, float4 *xb) {
        const int k0 = c * kChunk;
        if (k0 >= g.K) return;
        if (fast && k0 + kChunk <= g.K) {
            const uint32_t da = ka * (uint32_t)k0, db = kb * (uint32_t)k0;
#pragma unroll
            for (int i = 0; i < UA; ++i) xa[i] = gt_load_in<TA>(g.A, ga[i] + da, ka);
#pragma unroll
            for (int i = 0; i < UB; ++i) xb[i] = gt_load_in<TBt>(B, gb[i] + db, kb);
            return;
        }
#pragma unroll
        for (int i = 0; i < UA; ++i) {
            const int u = tid + i * NTHR;
            int row, kg;
            gt_unit<TA, kGtM>(u % SA, row, kg);
            xa[i] = gt_load<TA>(g.A, g.lda, m0 + row, g.M, k0 + kGtK * (u / SA) + 4 * kg, g.K, g.veca);
        }
#pragma unroll
        for (int i = 0; i < UB; ++i) {
            const int u = min(tid + i * NTHR, KC * SB - 1);
            int row, kg;
            gt_unit<TBt, NT>(u % SB, row, kg);
            xb[i] = gt_load<TBt>(B, g.ldb, n0 + row, g.N, k0 + kGtK * (u / SB) + 4 * kg, g.K, g.vecb);
        }
    };
    const int chunks = (g.K + kChunk - 1) / kChunk;
    float cs = 0.f;   // TA: this thread's row of A, summed over its k
    bool ok = true;
    int issued = 0;
    auto chunk = [&](int c, float4 *xa, float4 *xb) {   // false: a wait ran out
        const int st = c & 1;
        // the buffer's previous MMAs (chunk c - 2) have to be done
        const uint32_t done = c < 2 ? 1u : passes::tc_bounded_wait(passes::tc_smem(&mbar[st]), ((c >> 1) - 1) & 1);
        float *buf = base + st * KC * kSub;
        if (done) {
#pragma unroll
            for (int i = 0; i < UA; ++i) {
                gt_split(xa[i], buf, buf + kGtM * kGtK, oa[i], false);
                if (TA) cs += (xa[i].x + xa[i].y) + (xa[i].z + xa[i].w);
            }
#pragma unroll
            for (int i = 0; i < UB; ++i)
                if (tid + i * NTHR < KC * SB) gt_split(xb[i], buf, buf + NT * kGtK, ob[i], b_exact);
        }
        fetch(c + 2, xa, xb);
        asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
        asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
        if (__syncthreads_or(!done)) return false;
        if (tid == 0) {
            asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
#pragma unroll
            for (int q = 0; q < KC; ++q) {
                if (c * kChunk + q * kGtK >= g.K) break;
                const uint32_t a_h = passes::tc_smem(buf + q * kSub), a_l = a_h + 4 * kGtM * kGtK;
                const uint32_t b_h = a_l + 4 * kGtM * kGtK, b_l = b_h + 4 * NT * kGtK;
                // small terms first
                gt_mma(tmem, a_l, b_h, idesc, c == 0 && q == 0 ? 1u : 0u);
                if (!b_exact) gt_mma(tmem, a_h, b_l, idesc, 0u);
                gt_mma(tmem, a_h, b_h, idesc, 0u);
            }
            asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n"
                         ::"r"(passes::tc_smem(&mbar[st])));
        }
        issued = c + 1;
        return true;
    };
    fetch(0, ra[0], rb[0]);
    fetch(1, ra[1], rb[1]);
    for (int c = 0; c < chunks && ok; c += 2) {
        ok = chunk(c, ra[0], rb[0]);
        if (ok && c + 1 < chunks) ok = chunk(c + 1, ra[1], rb[1]);
    }
    // the last chunk of each buffer (commits complete in order of issue)
    for (int c = max(0, issued - 2); c < issued; ++c)
        if (!passes::tc_bounded_wait(passes::tc_smem(&mbar[c & 1]), (c >> 1) & 1)) ok = false;
    asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
    if (TA) csum[tid] = cs;
    if (__syncthreads_or(!ok)) {
        if (tid == 0) atomicExch(g.err, 1);
        // once more, so that nothing is in flight when the accumulator is freed
        for (int c = max(0, issued - 2); c < issued; ++c)
            passes::tc_bounded_wait(passes::tc_smem(&mbar[c & 1]), (c >> 1) & 1);
    } else {
        float *C = g.C;
        if (TA && g.colsum && blockIdx.y == 0 && tid < kGtM && m0 + tid < g.M) {
            float s = 0.f;
            for (int i = tid; i < NTHR; i += kGtM) s += csum[i];
            g.colsum[m0 + tid] = s;
        }
        // warps 0-3 take columns 0 .. 31, warps 4-7 the next; thread = row
        const int gm = m0 + 32 * (warp & 3) + lane, c0 = 32 * (warp >> 2);
        if (c0 < nt) {
            uint32_t r[32];
            const uint32_t addr = tmem + ((uint32_t)((warp & 3) * 32) << 16) + (uint32_t)c0;
            asm volatile("tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,"
                         "%14,%15,%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];\n"
                         : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
                           "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]),
                           "=r"(r[13]), "=r"(r[14]), "=r"(r[15]), "=r"(r[16]), "=r"(r[17]), "=r"(r[18]),
                           "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]),
                           "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]),
                           "=r"(r[31])
                         : "r"(addr));
            asm volatile("tcgen05.wait::ld.sync.aligned;\n" ::: "memory");
            if (gm < g.M) {
#pragma unroll
                for (int j = 0; j < (NT < 32 ? NT : 32); j += 4) {
                    const int gn = n0 + c0 + j;
                    const size_t o = (size_t)gm * g.ldc + gn;
                    float z[4] = {__uint_as_float(r[j]), __uint_as_float(r[j + 1]), __uint_as_float(r[j + 2]),
                                  __uint_as_float(r[j + 3])};
                    if (g.vecc && gn + 3 < g.N) {
                        if (g.bias)
                            for (int q = 0; q < 4; ++q) z[q] += g.bias[gn + q];
                        if (g.Zpre) *reinterpret_cast<float4 *>(g.Zpre + o) = make_float4(z[0], z[1], z[2], z[3]);
                        if (g.act)
                            for (int q = 0; q < 4; ++q) z[q] = gt_gelu(z[q]);
                        if (g.Zback) {
                            const float4 b = *reinterpret_cast<const float4 *>(g.Zback + o);
                            z[0] *= gt_gelu_grad(b.x);
                            z[1] *= gt_gelu_grad(b.y);
                            z[2] *= gt_gelu_grad(b.z);
                            z[3] *= gt_gelu_grad(b.w);
                        }
                        *reinterpret_cast<float4 *>(C + o) = make_float4(z[0], z[1], z[2], z[3]);
                    } else {
                        for (int q = 0; q < 4 && gn + q < g.N; ++q) {
                            float v = z[q] + (g.bias ? g.bias[gn + q] : 0.f);
                            if (g.Zpre) g.Zpre[o + q] = v;
                            if (g.act) v = gt_gelu(v);
                            if (g.Zback) v *= gt_gelu_grad(g.Zback[o + q]);
                            C[o + q] = v;
                        }
                    }
                }
            }
        }
    }
    asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
    __syncthreads();
    if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;\n" ::"r"(tmem), "r"(kCols));
}

}  // namespace mlp
}  // namespace dc
