// laq_decode.cu -- the decoder operations around the quantized projections of one decode step
// of a Qwen3-style model (the models whose decoding speed Sec. 5.2 reports): RMSNorm with the
// residual add, per-head q/k RMSNorm with rotary position embedding and the KV-cache append,
// grouped-query attention of the new token over its cache (the tokens split over the warps of a
// cluster of CTAs, combined in a fixed order), SiLU(gate) * up, the embedding gather and the greedy
// argmax.  The paper defines none of them; they follow the standard decoder definitions, with
// fp32 arithmetic and one fp16 rounding per stored tensor.
//
// Every kernel lets its successor launch at once (griddepcontrol.launch_dependents) and waits
// for its predecessor (griddepcontrol.wait) before reading or writing what its results depend on
// (attention prefetches cache rows into L2 before), so inside a CUDA graph of
// programmatically dependent launches each one's launch and set-up overlap the previous one.
#include <cooperative_groups.h>
#include <cuda_fp16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <atomic>

#include "laq.h"
#include "laq_device.cuh"
#include "laq_internal.cuh"

namespace cg = cooperative_groups;

namespace laq {
namespace {

constexpr int kHeadDim = 128;    // D: the only head size the attention kernels are built for
constexpr int kMaxGroup = 8;     // most q heads per kv head
constexpr int kChunk = 64;       // tokens per partial that the workspace has room for
constexpr int kPartial = kHeadDim + 2;  // floats per partial: acc[D], max, sum

__device__ __forceinline__ float warp_sum(float v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

__device__ __forceinline__ void unpack8(const uint4 u, float (&f)[8]) {
    const uint32_t w[4] = {u.x, u.y, u.z, u.w};
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const float2 t = __half22float2(*reinterpret_cast<const __half2*>(&w[i]));
        f[2 * i] = t.x;
        f[2 * i + 1] = t.y;
    }
}

__device__ __forceinline__ uint4 pack8(const float (&f)[8]) {
    uint32_t w[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const __half2 h = __floats2half2_rn(f[2 * i], f[2 * i + 1]);
        w[i] = *reinterpret_cast<const uint32_t*>(&h);
    }
    return make_uint4(w[0], w[1], w[2], w[3]);
}


// RMSNorm over a head (lane l holds elements 4l .. 4l+3 of the warp's head), times the norm
// weights, then the rotate-half rotation at position p; every lane of the warp takes part.
// The rotation angles of lane l's elements 4l .. 4l+3 at position p: cos and sin of
// p * theta^(-2i/D), i = the element's index mod D/2 (the same for every head).
__device__ __forceinline__ void rope_angles(int lane, int64_t p, float log2_theta,
                                            float (&cs)[4], float (&sn)[4]) {
#pragma unroll
    for (int e = 0; e < 4; ++e) {
        const int i = (4 * lane + e) & (kHeadDim / 2 - 1);  // frequency index
        const float inv_freq = exp2f(-(2.f * (float)i / (float)kHeadDim) * log2_theta);
        sincosf((float)p * inv_freq, &sn[e], &cs[e]);
    }
}

__device__ __forceinline__ void norm_rope4(const float (&x)[4], const __half* __restrict__ wn,
                                           int lane, const float (&cs)[4], const float (&sn)[4],
                                           float eps, float (&o)[4]) {
    float ss = 0.f;
#pragma unroll
    for (int e = 0; e < 4; ++e) ss = fmaf(x[e], x[e], ss);
    ss = warp_sum(ss);
    const float inv = rsqrtf(ss / (float)kHeadDim + eps);
    float y[4];
#pragma unroll
    for (int e = 0; e < 4; ++e) y[e] = x[e] * inv * __half2float(wn[4 * lane + e]);
#pragma unroll
    for (int e = 0; e < 4; ++e) {
        const float partner = __shfl_xor_sync(0xffffffffu, y[e], 16);
        o[e] = lane < 16 ? y[e] * cs[e] - partner * sn[e] : y[e] * cs[e] + partner * sn[e];
    }
}

__device__ __forceinline__ void load4(const __half* src, float (&x)[4]) {
    const uint2 raw = *reinterpret_cast<const uint2*>(src);
    const float2 a = __half22float2(*reinterpret_cast<const __half2*>(&raw.x));
    const float2 b = __half22float2(*reinterpret_cast<const __half2*>(&raw.y));
    x[0] = a.x; x[1] = a.y; x[2] = b.x; x[3] = b.y;
}

__device__ __forceinline__ uint2 round4(const float (&o)[4]) {
    const __half2 lo = __floats2half2_rn(o[0], o[1]), hi = __floats2half2_rn(o[2], o[3]);
    uint2 w;
    w.x = *reinterpret_cast<const uint32_t*>(&lo);
    w.y = *reinterpret_cast<const uint32_t*>(&hi);
    return w;
}

// ---- RMSNorm with the residual add ----
// Row m: h = X + R (rounded to fp16; h = X without R), R_out = h, Y = h / sqrt(mean(h^2) + eps)
// * w.  One CTA per row; each thread keeps up to kRmsChunks 8-element chunks in registers.
constexpr int kRmsThreads = 256;
constexpr int kRmsChunks = 4;  // H <= 8 * 256 * 4 = 8192

__global__ void __launch_bounds__(kRmsThreads) rmsnorm_kernel(const __half* __restrict__ X,
                                                              const __half* __restrict__ R,
                                                              __half* R_out,
                                                              const __half* __restrict__ w,
                                                              int H, float eps, __half* Y) {
    pdl_launch_dependents();
    prefetch_l2(w, (size_t)H * 2);
    pdl_wait();
    __shared__ float red[kRmsThreads / 32];
    const size_t row = (size_t)blockIdx.x * H;
    float h[kRmsChunks][8];
    float ss = 0.f;
#pragma unroll
    for (int c = 0; c < kRmsChunks; ++c) {
        const int i = (int)threadIdx.x + c * kRmsThreads;  // chunk index
        if (8 * i < H) {
            unpack8(*reinterpret_cast<const uint4*>(X + row + 8 * i), h[c]);
            if (R) {
                float r[8];
                unpack8(*reinterpret_cast<const uint4*>(R + row + 8 * i), r);
#pragma unroll
                for (int e = 0; e < 8; ++e) h[c][e] = __half2float(__float2half_rn(h[c][e] + r[e]));
            }
#pragma unroll
            for (int e = 0; e < 8; ++e) ss = fmaf(h[c][e], h[c][e], ss);
        }
    }
    ss = warp_sum(ss);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = ss;
    __syncthreads();
    float tot = 0.f;
#pragma unroll
    for (int k = 0; k < kRmsThreads / 32; ++k) tot += red[k];  // same order in every thread
    const float inv = rsqrtf(tot / (float)H + eps);
#pragma unroll
    for (int c = 0; c < kRmsChunks; ++c) {
        const int i = (int)threadIdx.x + c * kRmsThreads;
        if (8 * i < H) {
            if (R_out) *reinterpret_cast<uint4*>(R_out + row + 8 * i) = pack8(h[c]);
            float wv[8], y[8];
            unpack8(*reinterpret_cast<const uint4*>(w + 8 * i), wv);
#pragma unroll
            for (int e = 0; e < 8; ++e) y[e] = h[c][e] * inv * wv[e];
            *reinterpret_cast<uint4*>(Y + row + 8 * i) = pack8(y);
        }
    }
}

// ---- q/k RMSNorm + rotary embedding + KV-cache append ----
// One warp per head of qkv row m (q heads, then k heads, then v heads); lane l holds elements
// 4l .. 4l+3, so element d and its rotation partner d +- D/2 sit in lanes l and l ^ 16.
// Rotation (the rotate-half form): for i < D/2, angle a_i = pos * theta^(-2i/D),
//   out[i] = x[i] cos a_i - x[i + D/2] sin a_i,   out[i + D/2] = x[i + D/2] cos a_i + x[i] sin a_i.
__global__ void __launch_bounds__(128) qk_norm_rope_kernel(
    const __half* __restrict__ qkv, const __half* __restrict__ qw,
    const __half* __restrict__ kw, const int32_t* __restrict__ pos, int Hq, int Hkv,
    float log2_theta, float eps, __half* q_out, __half* k_cache, __half* v_cache,
    int64_t L_max) {
    pdl_launch_dependents();
    prefetch_l2(qw, kHeadDim * 2);
    prefetch_l2(kw, kHeadDim * 2);
    pdl_wait();
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int head = blockIdx.x * 4 + warp, m = blockIdx.y;
    const int nh = Hq + 2 * Hkv;
    if (head >= nh) return;
    const int64_t p = pos[m];
    const bool in_cache = p >= 0 && p < L_max;  // a position outside the cache is not stored
    const __half* src = qkv + ((size_t)m * nh + head) * kHeadDim + 4 * lane;
    const uint2 raw = *reinterpret_cast<const uint2*>(src);
    if (head >= Hq + Hkv) {  // v: appended as is
        const int g = head - Hq - Hkv;
        if (in_cache)
            *reinterpret_cast<uint2*>(v_cache + (((size_t)m * Hkv + g) * L_max + p) * kHeadDim +
                                      4 * lane) = raw;
        return;
    }
    float x[4];
    {
        const float2 a = __half22float2(*reinterpret_cast<const __half2*>(&raw.x));
        const float2 b = __half22float2(*reinterpret_cast<const __half2*>(&raw.y));
        x[0] = a.x; x[1] = a.y; x[2] = b.x; x[3] = b.y;
    }
    float cs[4], sn[4], o[4];
    rope_angles(lane, p, log2_theta, cs, sn);
    norm_rope4(x, head < Hq ? qw : kw, lane, cs, sn, eps, o);
    const __half2 lo = __floats2half2_rn(o[0], o[1]), hi = __floats2half2_rn(o[2], o[3]);
    uint2 outw;
    outw.x = *reinterpret_cast<const uint32_t*>(&lo);
    outw.y = *reinterpret_cast<const uint32_t*>(&hi);
    if (head < Hq) {
        *reinterpret_cast<uint2*>(q_out + ((size_t)m * Hq + head) * kHeadDim + 4 * lane) = outw;
    } else if (in_cache) {
        const int g = head - Hq;
        *reinterpret_cast<uint2*>(k_cache + (((size_t)m * Hkv + g) * L_max + p) * kHeadDim +
                                  4 * lane) = outw;
    }
}

// ---- grouped-query attention of one decode step ----
// One cluster of C CTAs works on one (row, kv head): the row's n cached tokens are cut into steps
// of 16, dealt round robin to the cluster's warps, so the split follows the actual length.  A
// warp streams its steps' K and V rows (2 x 4 KB) through a private cp.async ring and keeps the
// online softmax of its own tokens for the G = Hq / Hkv q heads at once, on the tensor cores
// (m16n8k16, fp16 operands, fp32 accumulation):
//   scores^T = K q^T: A the 16 tokens' K rows straight from ldmatrix, B the q heads (fp16, as
//     stored; the products are exact);
//   out^T += V^T P^T: A from ldmatrix.trans, B the probabilities after a movmatrix transpose, as
//     P = hi + lo with both halves fp16: 22 to 23 significand bits of P's 24, so within one fp32 unit
//     in the last place of p (p is scaled by 2^15, which cancels against the sum of p, so that its small
//     values stay above fp16's range).  For G <= 4 the MMA's 8 columns are 4 heads' hi and 4 heads' lo
//     (q's B columns 4-7 repeat heads 0-3, so the lanes that would idle hold the same probabilities and
//     contribute their low halves); WIDE (G = 5..8) issues one MMA for each half.
// The tensor core truncates what it adds, so no sum grows inside it: the 8 MMAs of a score and the
// steps of out^T start from zero and are added in fp32.  (Kept in one accumulator, a warp's 32 steps
// of a row of 8192 tokens left 0.29 % of the outputs rounded apart from 64 bits where V has mean 1, 0.005
// % here and with fp32 FMAs throughout; the fp16 rounding is 2.08e-4 of the result in either.)
// The warps' results meet in shared memory, the CTAs' through distributed shared memory: CTA r of
// the cluster combines the head dimensions [128 r / C, 128 (r + 1) / C) in rank order and stores
// fp16, so a call needs one launch and no scratch.  (Partials in a workspace and a combine kernel,
// fp32 FMAs and a 4-shuffle score: 13.3 us a call for one row of 2048 tokens, 129 us for 16 rows of
// 2048 .. 8192; this form 6.7 and 62 us, 5.4 TB/s.)  Where the clusters of all (row, kv head)
// pairs leave most SMs idle and the rows may be long, S clusters share a pair, write fp32 partials
// (acc[D], max, sum) to the workspace, and attn_combine_kernel adds them in order.
// Bound: HBM for long batches; for one short row the latency of a dependent launch (4.6 us at 256
// tokens) plus about 1 us per step of a warp.  So the ring is one step deep and the CTA has 8
// warps: at the same shared memory 4 warps with two steps measured 1301 us for a decode step at
// 2048 tokens against 1261; 16 warps an SM overlap each other's copies and arithmetic.  K and V
// loaded straight into MMA operand registers (no ring) was slower (249 us against 167 for 24
// calls), and 131 KB rings keep a CTA from sharing an SM with the kernels before and after it.
// Swizzle: 16-byte chunk j of a 256-byte row sits at j ^ (row & 7), so the 8 rows of an ldmatrix
// phase hit different banks.
constexpr int kStep = 16;                   // tokens per warp step
constexpr int kAttnWarps = 8;
constexpr int kAttnStages = 1;              // ring depth, steps (see the comment above)
constexpr int kStepBytes = 2 * kStep * kHeadDim * 2;  // K and V rows of a step
constexpr int kMaxCluster = 16;
constexpr int kRedRow = kHeadDim + 4;       // floats per row of red (lanes of a store: 32 banks)

struct AttnSmem {
    uint8_t ring[kAttnWarps][kAttnStages][kStepBytes];  // later red[warp][G][kRedRow] fp32
    uint8_t q[kMaxGroup * kHeadDim * 2];                // fp16 q heads, swizzled rows
    float recv[kMaxGroup * kHeadDim];                   // [C][G][128 / C] partials of this slice
    float2 ml[kMaxCluster][kMaxGroup];                  // (max, sum) of every CTA of the cluster
    float2 wml[kAttnWarps][kMaxGroup];                  // (max, sum) of every warp
};

struct AttnParams {
    const __half* q;        // [M][Hq][D], or qkv [M][Hq + 2 Hkv][D] (fused form)
    const __half* qw;       // fused: q and k norm weights
    const __half* kw;
    const int32_t* len;     // cached tokens per row; fused: positions (tokens - 1)
    __half* k_cache;
    __half* v_cache;
    __half* out;
    float* part;            // S > 1: [M][Hq][S][kPartial]
    int64_t L_max;
    int Hq, Hkv, C, S;
    float log2_theta, eps, scale;
};

__device__ __forceinline__ void cp_async16_zfill(uint32_t dst, const void* src, bool ok) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n" ::"r"(dst), "l"(src),
                 "r"(ok ? 16 : 0)
                 : "memory");
}
__device__ __forceinline__ void ldsm4(uint32_t addr, uint32_t (&r)[4]) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];\n"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                 : "r"(addr)
                 : "memory");
}
__device__ __forceinline__ void ldsm4t(uint32_t addr, uint32_t (&r)[4]) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];\n"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                 : "r"(addr)
                 : "memory");
}
// transpose of an 8 x 8 matrix of 16-bit values spread over the warp (two per lane)
__device__ __forceinline__ uint32_t movmatrix(uint32_t v) {
    uint32_t r;
    asm("movmatrix.sync.aligned.m8n8.trans.b16 %0, %1;\n" : "=r"(r) : "r"(v));
    return r;
}
// byte offset of 16-byte chunk j of row r
__device__ __forceinline__ int swz(int r, int j) { return r * 256 + ((j ^ (r & 7)) << 4); }

__device__ __forceinline__ float exp2_diff(float a, float b) {  // 2^(a - b); a = -inf: 0
    return a == -INFINITY ? 0.f : exp2f(a - b);
}

// Two CTAs per SM, as attn_shape counts on (the copies' addresses below cost the WIDE form 156
// registers when the compiler is left free, 128 and no spills with the bound).
template <bool FUSED, bool WIDE>
__global__ void __launch_bounds__(kAttnWarps * 32, 2) attn_kernel(const AttnParams p) {
    pdl_launch_dependents();
    if (p.C > 1) asm volatile("barrier.cluster.arrive.relaxed.aligned;\n" ::: "memory");
    extern __shared__ __align__(128) uint8_t attn_smem[];
    AttnSmem& sm = *reinterpret_cast<AttnSmem*>(attn_smem);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, c = lane & 3, r = lane >> 2;
    const int g = blockIdx.y, m = blockIdx.z, G = p.Hq / p.Hkv;
    const int C = p.C, rank = blockIdx.x % C;
    const int wi = blockIdx.x * kAttnWarps + warp, nw = gridDim.x * kAttnWarps;
    const size_t kv0 = ((size_t)m * p.Hkv + g) * p.L_max * kHeadDim;
    // While the preceding kernel finishes: ask L2 for the K and V rows of the warp's first steps
    // and compute the rotation angles, both by the position as it is now.  A prefetch returns no
    // data (whatever the preceding kernel still writes is seen by the loads below), and the
    // position is read again after the wait and the angles redone if it has changed.
    const int32_t pos_hint = *(const volatile int32_t*)(p.len + m);
    float cs[4], sn[4];
    {
        const int64_t nh = min((int64_t)pos_hint + (FUSED ? 1 : 0), p.L_max);
#pragma unroll
        for (int i = 0; i < kAttnStages; ++i) {
            const int64_t t = (int64_t)(wi + i * nw) * kStep + (lane >> 1);
            if (t < nh) {  // half a row of 128 bytes per lane
                const size_t off = kv0 + (size_t)t * kHeadDim + 64 * (lane & 1);
                asm volatile("prefetch.global.L2 [%0];\n" ::"l"(p.k_cache + off));
                asm volatile("prefetch.global.L2 [%0];\n" ::"l"(p.v_cache + off));
            }
        }
        if (FUSED) {
            prefetch_l2(p.qw, kHeadDim * 2);
            prefetch_l2(p.kw, kHeadDim * 2);
            rope_angles(lane, pos_hint, p.log2_theta, cs, sn);
        }
    }
    pdl_wait();

    const int64_t pos = *(const volatile int32_t*)(p.len + m);  // fused: the new token's position
    constexpr int kPerWarp = kMaxGroup / kAttnWarps;  // q heads a warp prepares
    float x[kPerWarp][4];
    const __half* row = p.q + (size_t)m * (p.Hq + 2 * p.Hkv) * kHeadDim + 4 * lane;
    if constexpr (FUSED) {
#pragma unroll
        for (int u = 0; u < kPerWarp; ++u) {
            const int j = warp + kAttnWarps * u;
            if (j < G) load4(row + (size_t)(g * G + j) * kHeadDim, x[u]);
        }
    }
    // (a cache of 2^31 tokens would not fit the GPU)
    const int n = (int)min(min(max(FUSED ? pos + 1 : pos, (int64_t)0), p.L_max),
                           (int64_t)0x7fffff00);
    const int nsteps = (n + kStep - 1) / kStep;
    const int pstep = (int)(pos / kStep);  // fused: the step that holds the new token

    // 16 rows of K and V of step s into ring slot `slot` (zeros past the row's end: a probability
    // of 0 times garbage could be NaN).  Lane: chunk lane % 16 of rows lane / 16 + 2 u.
    const uint32_t ring = (uint32_t)__cvta_generic_to_shared(sm.ring[warp]);
    const __half* kl = p.k_cache + kv0;
    const __half* vl = p.v_cache + kv0;
    auto issue = [&](int s, int slot) {
        if (s < nsteps) {
            const uint32_t dst = ring + slot * kStepBytes;
            const size_t off = (size_t)s * (kStep * kHeadDim);
            const int left = n - s * kStep;
#pragma unroll
            for (int u = 0; u < kStep / 2; ++u) {
                const int rr = 2 * u + (lane >> 4);
                const bool ok = rr < left;
                const size_t o = off + attn_copy_offset(lane, u, left);
                cp_async16_zfill(dst + swz(rr, lane & 15), kl + o, ok);
                cp_async16_zfill(dst + kStepBytes / 2 + swz(rr, lane & 15), vl + o, ok);
            }
        }
        cp_async_commit();
    };
#pragma unroll
    for (int i = 0; i < kAttnStages; ++i) issue(wi + i * nw, i);

    // q heads as fp16 rows (zeros past G; rows 4-7 repeat 0-3 unless WIDE); fused: normalised and
    // rotated here, and the warp that owns the new token's step makes its k and v.
    const bool holds_new = FUSED && pos >= 0 && pos < p.L_max && pstep % nw == wi;
    uint2 knew = make_uint2(0u, 0u), vnew = make_uint2(0u, 0u);
    float xk[4];
    if (holds_new) {
        load4(row + (size_t)(p.Hq + g) * kHeadDim, xk);
        vnew = *reinterpret_cast<const uint2*>(row + (size_t)(p.Hq + p.Hkv + g) * kHeadDim);
    }
    if (FUSED && pos != pos_hint) rope_angles(lane, pos, p.log2_theta, cs, sn);
#pragma unroll
    for (int u = 0; u < kPerWarp; ++u) {
        const int j = warp + kAttnWarps * u;
        uint2 w = make_uint2(0u, 0u);
        if (j < G) {
            if constexpr (FUSED) {
                float o[4];
                norm_rope4(x[u], p.qw, lane, cs, sn, p.eps, o);
                w = round4(o);
            } else {  // (q need not be 8-byte aligned here)
                const uint16_t* src = reinterpret_cast<const uint16_t*>(p.q) +
                                      ((size_t)m * p.Hq + g * G + j) * kHeadDim + 4 * lane;
                w.x = src[0] | (uint32_t)src[1] << 16;
                w.y = src[2] | (uint32_t)src[3] << 16;
            }
        }
        if (WIDE || j < 4) *reinterpret_cast<uint2*>(sm.q + swz(j, lane >> 1) + 8 * (lane & 1)) = w;
        if (!WIDE && j < 4)
            *reinterpret_cast<uint2*>(sm.q + swz(j + 4, lane >> 1) + 8 * (lane & 1)) = w;
    }
    if (holds_new) {
        float o[4];
        norm_rope4(xk, p.kw, lane, cs, sn, p.eps, o);
        knew = round4(o);
    }
    __syncthreads();
    uint32_t qb[8][2];  // B fragments of the 8 k16 steps
    {
        const uint32_t qs = (uint32_t)__cvta_generic_to_shared(sm.q);
#pragma unroll
        for (int t = 0; t < 4; ++t) {
            uint32_t f[4];
            ldsm4(qs + swz(lane & 7, 4 * t + (lane >> 3)), f);
            qb[2 * t][0] = f[0];
            qb[2 * t][1] = f[1];
            qb[2 * t + 1][0] = f[2];
            qb[2 * t + 1][1] = f[3];
        }
    }

    const float sl = p.scale * 1.4426950408889634f;  // scores in powers of two
    // of MMA columns 2c and 2c + 1: scaled max, and this lane's share of sum p
    float mx[2] = {-INFINITY, -INFINITY}, sum[2] = {0.f, 0.f};
    // out^T: acc[t][v] is dimension 16 t + r + 8 (v / 2), column 2c + v % 2 (WIDE: acl the low
    // halves' products)
    float acc[8][4], acl[WIDE ? 8 : 1][4];
#pragma unroll
    for (int t = 0; t < 8; ++t)
#pragma unroll
        for (int v = 0; v < 4; ++v) acc[t][v] = acl[WIDE ? t : 0][v] = 0.f;

    const int krow = swz(lane & 15, lane >> 4);  // ldmatrix: tokens lane % 16, chunk lane / 16
    const int vrow = (((lane >> 4) & 1) * 8 + (lane & 7)) * 256, vj = (lane >> 3) & 1;
    int slot = 0;
    for (int s = wi; s < nsteps; s += nw) {
        cp_async_wait(kAttnStages - 1);
        __syncwarp();
        const uint32_t kb = ring + slot * kStepBytes, vb = kb + kStepBytes / 2;
        if (holds_new && s == pstep) {  // the new token replaces the staged (stale) row
            const int rr = (int)pos - s * kStep;
            uint8_t* dst = sm.ring[warp][slot] + swz(rr, lane >> 1) + 8 * (lane & 1);
            *reinterpret_cast<uint2*>(dst) = knew;
            *reinterpret_cast<uint2*>(dst + kStepBytes / 2) = vnew;
            const size_t off = kv0 + (size_t)pos * kHeadDim + 4 * lane;
            *reinterpret_cast<uint2*>(p.k_cache + off) = knew;
            *reinterpret_cast<uint2*>(p.v_cache + off) = vnew;
            __syncwarp();
        }
        // scores: sc[v] is token r + 8 (v / 2), column 2c + v % 2
        float sc[4], se[8][4];
#pragma unroll
        for (int ks = 0; ks < 8; ++ks) {
            uint32_t a[4];
            ldsm4(kb + (krow ^ (ks << 5)), a);  // chunks 2 ks and 2 ks + 1 of the 16 tokens
            se[ks][0] = se[ks][1] = se[ks][2] = se[ks][3] = 0.f;
            mma16816(se[ks], a[0], a[1], a[2], a[3], qb[ks][0], qb[ks][1]);
        }
#pragma unroll
        for (int v = 0; v < 4; ++v)
            sc[v] = ((se[0][v] + se[1][v]) + (se[2][v] + se[3][v])) +
                    ((se[4][v] + se[5][v]) + (se[6][v] + se[7][v]));
        const int left = n - s * kStep;  // (>= 16 in all but the last step)
        float nm[2];
        bool grew = false;
#pragma unroll
        for (int e = 0; e < 2; ++e) {
            sc[e] = r < left ? sc[e] : -INFINITY;
            sc[2 + e] = r + 8 < left ? sc[2 + e] : -INFINITY;
            float v = fmaxf(sc[e], sc[2 + e]);
            v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, 4));
            v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, 8));
            v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, 16)) * sl;
            nm[e] = fmaxf(mx[e], v);
            grew |= nm[e] > mx[e];
        }
        if (__any_sync(0xffffffffu, grew)) {
#pragma unroll
            for (int e = 0; e < 2; ++e) {
                const float f = exp2_diff(mx[e], nm[e]);
                mx[e] = nm[e];
                sum[e] *= f;
#pragma unroll
                for (int t = 0; t < 8; ++t) {
                    acc[t][e] *= f;
                    acc[t][2 + e] *= f;
                    if (WIDE) {
                        acl[WIDE ? t : 0][e] *= f;
                        acl[WIDE ? t : 0][2 + e] *= f;
                    }
                }
            }
        }
        uint32_t bh[2], bl[2];  // B fragments: tokens 0-7 and 8-15 of the step
#pragma unroll
        for (int t = 0; t < 2; ++t) {
            float pr[2];
#pragma unroll
            for (int e = 0; e < 2; ++e) {
                const float off = (mx[e] == -INFINITY ? 0.f : mx[e]) - 15.f;
                pr[e] = exp2f(fmaf(sc[2 * t + e], sl, -off));
                sum[e] += pr[e];
            }
            const __half2 h = __floats2half2_rn(pr[0], pr[1]);
            const float2 hf = __half22float2(h);
            const __half2 l = __floats2half2_rn(pr[0] - hf.x, pr[1] - hf.y);
            const uint32_t hw = *reinterpret_cast<const uint32_t*>(&h);
            const uint32_t lw = *reinterpret_cast<const uint32_t*>(&l);
            bh[t] = movmatrix(WIDE || c < 2 ? hw : lw);
            if (WIDE) bl[t] = movmatrix(lw);
        }
#pragma unroll
        for (int t = 0; t < 8; ++t) {
            uint32_t a[4];  // V^T: dimensions 16 t .. 16 t + 15 of the 16 tokens
            ldsm4t(vb + vrow + (((2 * t + vj) ^ (lane & 7)) << 4), a);
            float d[4] = {0.f, 0.f, 0.f, 0.f};
            mma16816(d, a[0], a[1], a[2], a[3], bh[0], bh[1]);
#pragma unroll
            for (int v = 0; v < 4; ++v) acc[t][v] += d[v];
            if (WIDE) mma16816(acl[WIDE ? t : 0], a[0], a[1], a[2], a[3], bl[0], bl[1]);
        }
        __syncwarp();  // every lane is done with the slot
        issue(s + kAttnStages * nw, slot);
        slot = slot + 1 == kAttnStages ? 0 : slot + 1;
    }
    asm volatile("cp.async.wait_all;\n" ::: "memory");

    // ---- warps -> CTA (shared memory) ----
#pragma unroll
    for (int e = 0; e < 2; ++e) {
#pragma unroll
        for (int o = 4; o < 32; o <<= 1) sum[e] += __shfl_xor_sync(0xffffffffu, sum[e], o);
        if (r == 0) sm.wml[warp][2 * c + e] = make_float2(mx[e], sum[e]);
    }
    __syncthreads();  // (also: every warp is done with its ring)
    float* red = reinterpret_cast<float*>(&sm.ring[0][0][0]);  // [warp][G][kRedRow]
#pragma unroll
    for (int e = 0; e < 2; ++e) {
        const int j = 2 * c + e;  // head
        float cm = sm.wml[0][j].x;
#pragma unroll
        for (int w = 1; w < kAttnWarps; ++w) cm = fmaxf(cm, sm.wml[w][j].x);
        const float f = exp2_diff(mx[e], cm);
#pragma unroll
        for (int t = 0; t < 8; ++t)
#pragma unroll
            for (int u = 0; u < 2; ++u) {
                const float h = acc[t][2 * u + e];
                const float l = WIDE ? acl[WIDE ? t : 0][2 * u + e]
                                     : __shfl_xor_sync(0xffffffffu, h, 2);
                // (an infinite v times a low half of 0 or of the other sign: the high half alone)
                if (j < G)
                    red[(warp * G + j) * kRedRow + 16 * t + 8 * u + r] =
                        f * (h + (isfinite(l) ? l : 0.f));
            }
    }
    __syncthreads();
    const int per = kHeadDim / C;  // dimensions of a CTA's slice
    cg::cluster_group cluster = cg::this_cluster();
    if (C > 1) asm volatile("barrier.cluster.wait.aligned;\n" ::: "memory");  // peers have started
    for (int e = threadIdx.x; e < G * kHeadDim; e += kAttnWarps * 32) {
        const int j = e / kHeadDim, d = e % kHeadDim;
        float* recv = C > 1 ? cluster.map_shared_rank(sm.recv, d / per) : sm.recv;
        float a = 0.f;
#pragma unroll
        for (int w = 0; w < kAttnWarps; ++w) a += red[(w * G + j) * kRedRow + d];
        recv[(rank * G + j) * per + d % per] = a;
    }
    for (int u = threadIdx.x; u < C * G; u += kAttnWarps * 32) {
        const int j = u % G, dst = u / G;
        float cm = sm.wml[0][j].x, cs = 0.f;
#pragma unroll
        for (int w = 1; w < kAttnWarps; ++w) cm = fmaxf(cm, sm.wml[w][j].x);
#pragma unroll
        for (int w = 0; w < kAttnWarps; ++w)
            cs += exp2_diff(sm.wml[w][j].x, cm) * sm.wml[w][j].y;
        float2* ml = C > 1 ? cluster.map_shared_rank(&sm.ml[0][0], dst) : &sm.ml[0][0];
        ml[rank * kMaxGroup + j] = make_float2(cm, cs);
    }
    // ---- CTAs -> cluster (distributed shared memory), in rank order ----
    if (C > 1)
        cluster.sync();
    else
        __syncthreads();
    for (int e = threadIdx.x; e < G * per; e += kAttnWarps * 32) {
        const int j = e / per, dd = e % per, dim = rank * per + dd;
        float M = sm.ml[0][j].x;
        for (int q = 1; q < C; ++q) M = fmaxf(M, sm.ml[q][j].x);
        float num = 0.f, den = 0.f;
        for (int q = 0; q < C; ++q) {
            const float2 ml = sm.ml[q][j];
            const float f = exp2_diff(ml.x, M);
            // (a CTA without tokens has f = 0 and partials of 0)
            num = fmaf(f, sm.recv[(q * G + j) * per + dd], num);
            den = fmaf(f, ml.y, den);
        }
        const size_t h = (size_t)m * p.Hq + g * G + j;
        if (p.S == 1) {
            p.out[h * kHeadDim + dim] = __float2half_rn(n == 0 ? 0.f : num / den);
        } else {
            float* pp = p.part + (h * p.S + blockIdx.x / C) * kPartial;
            pp[dim] = num;
            if (dim == 0) {
                pp[kHeadDim] = M;
                pp[kHeadDim + 1] = den;
            }
        }
    }
}

// Add the partials of the S clusters of each (row, head) in order (maxima in powers of two; a
// cluster without tokens has max -inf and weight 0).  A row without tokens gets zeros.
__global__ void __launch_bounds__(kHeadDim) attn_combine_kernel(const float* __restrict__ part,
                                                                const int32_t* __restrict__ len,
                                                                int len_is_pos, int Hq, int S,
                                                                __half* out) {
    pdl_launch_dependents();
    pdl_wait();
    const size_t h = (size_t)blockIdx.y * Hq + blockIdx.x;
    const float* pp = part + h * S * kPartial;
    const int d = threadIdx.x;
    float M = -INFINITY;
    for (int s = 0; s < S; ++s) M = fmaxf(M, pp[s * kPartial + kHeadDim]);
    float num = 0.f, den = 0.f;
    for (int s = 0; s < S; ++s) {
        const float f = exp2_diff(pp[s * kPartial + kHeadDim], M);
        num = fmaf(f, pp[s * kPartial + d], num);
        den = fmaf(f, pp[s * kPartial + kHeadDim + 1], den);
    }
    const bool empty = (int64_t)len[blockIdx.y] + (len_is_pos ? 1 : 0) <= 0;
    out[h * kHeadDim + d] = __float2half_rn(empty ? 0.f : num / den);
}

// ---- SiLU(gate) * up ----
__global__ void __launch_bounds__(256) silu_mul_kernel(const __half* __restrict__ gu, int64_t I,
                                                       int64_t chunks, __half* hout) {
    pdl_launch_dependents();
    pdl_wait();
    const int64_t u = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;  // 8-element chunk
    if (u >= chunks) return;
    const int64_t per_row = I / 8;
    const int64_t m = u / per_row, i = (u - m * per_row) * 8;
    float g[8], up[8], y[8];
    unpack8(*reinterpret_cast<const uint4*>(gu + m * 2 * I + i), g);
    unpack8(*reinterpret_cast<const uint4*>(gu + m * 2 * I + I + i), up);
#pragma unroll
    for (int e = 0; e < 8; ++e) y[e] = g[e] / (1.f + expf(-g[e])) * up[e];
    *reinterpret_cast<uint4*>(hout + m * I + i) = pack8(y);
}

// ---- embedding gather ----
__global__ void __launch_bounds__(256) embed_kernel(const __half* __restrict__ E,
                                                    const int32_t* __restrict__ tokens, int64_t V,
                                                    int64_t H, __half* X) {
    pdl_launch_dependents();
    pdl_wait();
    const int m = blockIdx.x;
    const int64_t t = tokens[m];
    const bool ok = t >= 0 && t < V;
    for (int64_t i = threadIdx.x; i < H / 8; i += blockDim.x) {
        const uint4 v = ok ? *reinterpret_cast<const uint4*>(E + t * H + 8 * i)
                           : make_uint4(0u, 0u, 0u, 0u);
        *reinterpret_cast<uint4*>(X + (size_t)m * H + 8 * i) = v;
    }
}

// ---- greedy argmax (ties: the smallest index; NaN never wins) ----
constexpr int kArgThreads = 1024;
// (bv, bi) starts at (-inf, none); a value must beat it strictly, ties between real candidates
// go to the smaller index, so -inf and NaN never win.
constexpr int kNone = 0x7fffffff;
__device__ __forceinline__ void better(float& bv, int& bi, float v, int i) {
    if (v > bv || (v == bv && bi != kNone && i < bi)) {
        bv = v;
        bi = i;
    }
}
// A cluster of C (1 or 8) CTAs per row: CTA r scans the r-th of C equal parts of the row (in whole 8-element
// chunks where the row allows 16-byte loads), sends its candidate to CTA 0, and CTA 0 picks the
// winner in part order.  Bound: the latency of a dependent launch; one CTA per row took 11 us for
// a 151,936-entry row (0.3 MB through one SM).  With eight, the head's GEMV + argmax: 67.4 -> 63.4
// us.
__global__ void __launch_bounds__(kArgThreads) argmax_kernel(const __half* __restrict__ logits,
                                                             int64_t V, int C, int32_t* out) {
    pdl_launch_dependents();
    if (C > 1) asm volatile("barrier.cluster.arrive.relaxed.aligned;\n" ::: "memory");
    pdl_wait();
    __shared__ float bvs[kArgThreads / 32];
    __shared__ int bis[kArgThreads / 32];
    __shared__ float cvs[8];  // candidates of the cluster's CTAs (in CTA 0)
    __shared__ int cis[8];
    const int m = blockIdx.y, rank = blockIdx.x;
    const __half* row = logits + (size_t)m * V;
    float bv = -INFINITY;
    int bi = kNone;
    if (((uintptr_t)row & 15u) == 0 && V % 8 == 0) {
        // 16-byte loads, four in flight per thread
        const int64_t all8 = V / 8, lo = all8 * rank / C, n8 = all8 * (rank + 1) / C;
        for (int64_t b = lo + threadIdx.x; b < n8; b += 4 * kArgThreads) {
            uint4 u[4];
#pragma unroll
            for (int r = 0; r < 4; ++r) {
                const int64_t i8 = b + r * kArgThreads;
                u[r] = i8 < n8 ? *reinterpret_cast<const uint4*>(row + 8 * i8)
                               : make_uint4(0xfc00fc00u, 0xfc00fc00u, 0xfc00fc00u, 0xfc00fc00u);
            }
#pragma unroll
            for (int r = 0; r < 4; ++r) {
                float f[8];
                unpack8(u[r], f);
                const int i0 = (int)(8 * (b + r * kArgThreads));
#pragma unroll
                for (int e = 0; e < 8; ++e) better(bv, bi, f[e], i0 + e);
            }
        }
    } else {
        const int64_t lo = V * rank / C, hi = V * (rank + 1) / C;
        for (int64_t i = lo + threadIdx.x; i < hi; i += kArgThreads)
            better(bv, bi, __half2float(row[i]), (int)i);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const float v = __shfl_xor_sync(0xffffffffu, bv, o);
        const int i = __shfl_xor_sync(0xffffffffu, bi, o);
        better(bv, bi, v, i);
    }
    if ((threadIdx.x & 31) == 0) {
        bvs[threadIdx.x >> 5] = bv;
        bis[threadIdx.x >> 5] = bi;
    }
    __syncthreads();
    if (threadIdx.x < 32) {
        float v = bvs[threadIdx.x];
        int i = bis[threadIdx.x];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            const float w = __shfl_xor_sync(0xffffffffu, v, o);
            const int k = __shfl_xor_sync(0xffffffffu, i, o);
            better(v, i, w, k);
        }
        bv = v;
        bi = i;
    }
    if (C > 1) {
        cg::cluster_group cluster = cg::this_cluster();
        asm volatile("barrier.cluster.wait.aligned;\n" ::: "memory");  // CTA 0 has started
        if (threadIdx.x == 0) {
            cluster.map_shared_rank(cvs, 0)[rank] = bv;
            cluster.map_shared_rank(cis, 0)[rank] = bi;
        }
        cluster.sync();
        if (rank == 0 && threadIdx.x == 0)
            for (int k = 1; k < C; ++k) better(bv, bi, cvs[k], cis[k]);
    }
    if (rank == 0 && threadIdx.x == 0) out[m] = bi == kNone ? 0 : bi;  // none above -inf: 0
}

// Launch with programmatic stream serialization (the kernel may start while its predecessor
// finishes; it waits for it with griddepcontrol.wait).
template <typename... KArgs, typename... Args>
laq_status launch_pdl(void (*fn)(KArgs...), dim3 grid, dim3 block, cudaStream_t stream,
                      Args... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.stream = stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    const cudaError_t e = cudaLaunchKernelEx(&cfg, fn, args...);
    return e == cudaSuccess ? LAQ_OK : LAQ_ERR_CUDA;
}

// Clusters of C CTAs per (row, kv head) pair, S clusters per pair.
//  * C: the most, up to 16 (8 where the device takes no more), that keeps the grid within two CTAs
//    per SM, the CTAs that are resident together; never more than give each warp one step.
//    Measured on GB300, fused form, 8 kv heads, 2048 tokens: one row 7.0 / 6.7 us a call at C = 8
//    / 16; 4 rows 10.9 / 9.9 / 20.1 at C = 4 / 8 / 16; 16 rows 25.0 / 28.7 / 36.7 at C = 2 / 4 / 8.
//  * S > 1 only where the clusters leave half the SMs idle and a CTA would walk more than 512
//    tokens: the partials then cost a second launch, less than the walk (one row, 1 kv head: 20.5
//    -> 12.3 us at 32768 tokens with S = 4, 69 -> 21 us at 131072 with 8; 4 kv heads: 18.4 ->
//    16.5 us at 16384 with 2; but 8 kv heads, 128 CTAs, 12.9 -> 19 us at 8192 with 2).
struct AttnShape {
    int C, S;
};
AttnShape attn_shape(int64_t pairs, int64_t L_max, int sms, int max_cluster) {
    int C = max_cluster;
    while (C > 1 && pairs * C > 2 * (int64_t)sms) C /= 2;
    const int64_t steps = (L_max + kStep - 1) / kStep;
    while (C > 1 && steps <= kAttnWarps * (C / 2)) C /= 2;
    int64_t S = 1;
    if (2 * pairs * C <= sms) {
        const int64_t fill = sms / (pairs * C);
        const int64_t most = L_max / (512 * (int64_t)C);
        S = fill < most ? fill : most;
        if (S < 1) S = 1;
    }
    return AttnShape{C, (int)S};
}

// Once per device and form: the shared-memory limit and the cluster size.  Returns the largest
// cluster the device schedules (16, or 8), 0 on a CUDA error.
template <bool FUSED, bool WIDE>
int attn_setup(int* sms) {
    static std::atomic<int> cluster_of[64], sms_of[64];
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return 0;
    int c = cluster_of[dev].load();
    if (c == 0) {
        int n = 0;
        const void* fn = (const void*)attn_kernel<FUSED, WIDE>;
        if (cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess ||
            cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)sizeof(AttnSmem)) != cudaSuccess ||
            cudaFuncSetAttribute(fn, cudaFuncAttributePreferredSharedMemoryCarveout,
                                 (int)cudaSharedmemCarveoutMaxShared) != cudaSuccess)
            return 0;
        c = 8;
        if (cudaFuncSetAttribute(fn, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) ==
            cudaSuccess) {
            cudaLaunchConfig_t cfg = {};
            cfg.gridDim = dim3(kMaxCluster);
            cfg.blockDim = dim3(kAttnWarps * 32);
            cfg.dynamicSmemBytes = sizeof(AttnSmem);
            cudaLaunchAttribute attr[1];
            attr[0].id = cudaLaunchAttributeClusterDimension;
            attr[0].val.clusterDim.x = kMaxCluster;
            attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
            cfg.attrs = attr;
            cfg.numAttrs = 1;
            int fit = 0;
            if (cudaOccupancyMaxActiveClusters(&fit, fn, &cfg) != cudaSuccess)
                cudaGetLastError();  // (a refused cluster size is not an error of this call)
            else if (fit > 0)
                c = kMaxCluster;
        } else {
            cudaGetLastError();
        }
        sms_of[dev].store(n);
        cluster_of[dev].store(c);
    }
    *sms = sms_of[dev].load();
    return c;
}

template <bool FUSED, bool WIDE>
laq_status run_attention(AttnParams p, int64_t M, cudaStream_t stream) {
    int sms = 0;
    const int max_cluster = attn_setup<FUSED, WIDE>(&sms);
    if (max_cluster == 0) return LAQ_ERR_CUDA;
    const AttnShape sh = attn_shape(M * p.Hkv, p.L_max, sms, max_cluster);
    p.C = sh.C;
    p.S = sh.S;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(sh.C * sh.S), (unsigned)p.Hkv, (unsigned)M);
    cfg.blockDim = dim3(kAttnWarps * 32);
    cfg.dynamicSmemBytes = sizeof(AttnSmem);
    cfg.stream = stream;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = (unsigned)sh.C;
    attr[1].val.clusterDim.y = attr[1].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = sh.C > 1 ? 2 : 1;
    if (cudaLaunchKernelEx(&cfg, attn_kernel<FUSED, WIDE>, p) != cudaSuccess) return LAQ_ERR_CUDA;
    if (sh.S == 1) return LAQ_OK;
    return launch_pdl(attn_combine_kernel, dim3((unsigned)p.Hq, (unsigned)M), dim3(kHeadDim),
                      stream, (const float*)p.part, p.len, FUSED ? 1 : 0, p.Hq, sh.S, p.out);
}

template <bool FUSED>
laq_status run_attention(const AttnParams& p, int64_t M, void* stream) {
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    return p.Hq / p.Hkv > 4 ? run_attention<FUSED, true>(p, M, s)
                            : run_attention<FUSED, false>(p, M, s);
}

bool aligned16(const void* p) { return ((uintptr_t)p & 15u) == 0; }

}  // namespace
}  // namespace laq

using namespace laq;

extern "C" {

laq_status laq_rmsnorm(const void* X, const void* R, void* R_out, const void* w, int64_t M,
                       int64_t H, float eps, void* Y, void* stream) {
    if (!X || !w || !Y) return LAQ_ERR_NULL;
    if (M < 1 || M > 65535 || H < 8 || H % 8 || H > 8 * kRmsThreads * kRmsChunks)
        return LAQ_ERR_SHAPE;
    if (!(eps >= 0.f)) return LAQ_ERR_SHAPE;
    if (!aligned16(X) || !aligned16(w) || !aligned16(Y) || (R && !aligned16(R)) ||
        (R_out && !aligned16(R_out)))
        return LAQ_ERR_ALIGN;
    return launch_pdl(rmsnorm_kernel, dim3((unsigned)M), dim3(kRmsThreads),
                      static_cast<cudaStream_t>(stream), static_cast<const __half*>(X),
                      static_cast<const __half*>(R), static_cast<__half*>(R_out),
                      static_cast<const __half*>(w), (int)H, eps, static_cast<__half*>(Y));
}

laq_status laq_qk_norm_rope(const void* qkv, const void* q_norm_w, const void* k_norm_w,
                            const int32_t* pos, int64_t M, int32_t Hq, int32_t Hkv, int32_t D,
                            float theta, float eps, void* q_out, void* k_cache, void* v_cache,
                            int64_t L_max, void* stream) {
    if (!qkv || !q_norm_w || !k_norm_w || !pos || !q_out || !k_cache || !v_cache)
        return LAQ_ERR_NULL;
    if (D != kHeadDim || M < 1 || M > 65535 || Hq < 1 || Hkv < 1 || Hq % Hkv ||
        Hq / Hkv > kMaxGroup || L_max < 1 || !(theta > 1.f) || !(eps >= 0.f))
        return LAQ_ERR_SHAPE;
    if (((uintptr_t)qkv & 7u) || ((uintptr_t)q_out & 7u) || ((uintptr_t)k_cache & 7u) ||
        ((uintptr_t)v_cache & 7u))
        return LAQ_ERR_ALIGN;
    const int nh = Hq + 2 * Hkv;
    return launch_pdl(qk_norm_rope_kernel, dim3((unsigned)((nh + 3) / 4), (unsigned)M), dim3(128),
                      static_cast<cudaStream_t>(stream), static_cast<const __half*>(qkv),
                      static_cast<const __half*>(q_norm_w), static_cast<const __half*>(k_norm_w),
                      pos, (int)Hq, (int)Hkv, log2f(theta), eps, static_cast<__half*>(q_out),
                      static_cast<__half*>(k_cache), static_cast<__half*>(v_cache), L_max);
}

size_t laq_attention_workspace_bytes(int64_t M, int32_t Hq, int64_t L_max) {
    if (M < 1 || Hq < 1 || L_max < 1) return 0;
    const int64_t nchunk = (L_max + kChunk - 1) / kChunk;
    return (size_t)M * Hq * nchunk * kPartial * sizeof(float);
}

laq_status laq_attention_decode(const void* q, const void* k_cache, const void* v_cache,
                                const int32_t* len, int64_t M, int32_t Hq, int32_t Hkv,
                                int32_t D, int64_t L_max, float scale, void* out,
                                void* workspace, size_t workspace_bytes, void* stream) {
    if (!q || !k_cache || !v_cache || !len || !out || !workspace) return LAQ_ERR_NULL;
    if (D != kHeadDim || M < 1 || M > 65535 || Hq < 1 || Hkv < 1 || Hq % Hkv ||
        Hq / Hkv > kMaxGroup || Hkv > 65535 || L_max < 1 || !(scale > 0.f))
        return LAQ_ERR_SHAPE;
    if (!aligned16(k_cache) || !aligned16(v_cache) || ((uintptr_t)q & 1u) ||
        ((uintptr_t)out & 1u) || ((uintptr_t)workspace & 3u))
        return LAQ_ERR_ALIGN;
    if (workspace_bytes < laq_attention_workspace_bytes(M, Hq, L_max)) return LAQ_ERR_WORKSPACE;
    const int64_t nchunk = (L_max + kChunk - 1) / kChunk;
    if (nchunk > 0x7fffffff) return LAQ_ERR_SHAPE;
    AttnParams p = {};
    p.q = static_cast<const __half*>(q);
    p.len = len;
    p.k_cache = const_cast<__half*>(static_cast<const __half*>(k_cache));  // only read
    p.v_cache = const_cast<__half*>(static_cast<const __half*>(v_cache));
    p.out = static_cast<__half*>(out);
    p.part = static_cast<float*>(workspace);
    p.L_max = L_max;
    p.Hq = Hq;
    p.Hkv = Hkv;
    p.scale = scale;
    return run_attention<false>(p, M, stream);
}

size_t laq_attention_qkv_workspace_bytes(int64_t M, int32_t Hq, int32_t Hkv, int64_t L_max) {
    if (M < 1 || Hq < 1 || Hkv < 1 || L_max < 1) return 0;
    return laq_attention_workspace_bytes(M, Hq, L_max);
}

laq_status laq_attention_qkv(const void* qkv, const void* q_norm_w, const void* k_norm_w,
                             const int32_t* pos, int64_t M, int32_t Hq, int32_t Hkv, int32_t D,
                             float theta, float eps, void* k_cache, void* v_cache, int64_t L_max,
                             float scale, void* out, void* workspace, size_t workspace_bytes,
                             void* stream) {
    if (!qkv || !q_norm_w || !k_norm_w || !pos || !k_cache || !v_cache || !out || !workspace)
        return LAQ_ERR_NULL;
    if (D != kHeadDim || M < 1 || M > 65535 || Hq < 1 || Hkv < 1 || Hq % Hkv ||
        Hq / Hkv > kMaxGroup || Hkv > 65535 || L_max < 1 || !(theta > 1.f) || !(eps >= 0.f) ||
        !(scale > 0.f))
        return LAQ_ERR_SHAPE;
    if (((uintptr_t)qkv & 7u) || !aligned16(k_cache) || !aligned16(v_cache) ||
        ((uintptr_t)out & 1u) || !aligned16(workspace))
        return LAQ_ERR_ALIGN;
    if (workspace_bytes < laq_attention_qkv_workspace_bytes(M, Hq, Hkv, L_max))
        return LAQ_ERR_WORKSPACE;
    const int64_t nchunk = (L_max + kChunk - 1) / kChunk;
    if (nchunk > 0x7fffffff) return LAQ_ERR_SHAPE;
    AttnParams p = {};
    p.q = static_cast<const __half*>(qkv);
    p.qw = static_cast<const __half*>(q_norm_w);
    p.kw = static_cast<const __half*>(k_norm_w);
    p.len = pos;
    p.k_cache = static_cast<__half*>(k_cache);
    p.v_cache = static_cast<__half*>(v_cache);
    p.out = static_cast<__half*>(out);
    p.part = static_cast<float*>(workspace);
    p.L_max = L_max;
    p.Hq = Hq;
    p.Hkv = Hkv;
    p.log2_theta = log2f(theta);
    p.eps = eps;
    p.scale = scale;
    return run_attention<true>(p, M, stream);
}

laq_status laq_silu_mul(const void* gate_up, int64_t M, int64_t I, void* h, void* stream) {
    if (!gate_up || !h) return LAQ_ERR_NULL;
    if (M < 1 || I < 8 || I % 8) return LAQ_ERR_SHAPE;
    if (!aligned16(gate_up) || !aligned16(h)) return LAQ_ERR_ALIGN;
    const int64_t chunks = M * I / 8;
    return launch_pdl(silu_mul_kernel, dim3((unsigned)((chunks + 255) / 256)), dim3(256),
                      static_cast<cudaStream_t>(stream), static_cast<const __half*>(gate_up), I,
                      chunks, static_cast<__half*>(h));
}

laq_status laq_embed(const void* E, const int32_t* tokens, int64_t M, int64_t V, int64_t H,
                     void* X, void* stream) {
    if (!E || !tokens || !X) return LAQ_ERR_NULL;
    if (M < 1 || M > 65535 || V < 1 || H < 8 || H % 8) return LAQ_ERR_SHAPE;
    if (!aligned16(E) || !aligned16(X)) return LAQ_ERR_ALIGN;
    return launch_pdl(embed_kernel, dim3((unsigned)M), dim3(256),
                      static_cast<cudaStream_t>(stream), static_cast<const __half*>(E), tokens, V,
                      H, static_cast<__half*>(X));
}

laq_status laq_argmax(const void* logits, int64_t M, int64_t V, int32_t* out, void* stream) {
    if (!logits || !out) return LAQ_ERR_NULL;
    if (M < 1 || M > 65535 || V < 1 || V > 0x7ffffffe) return LAQ_ERR_SHAPE;
    if ((uintptr_t)logits & 1u) return LAQ_ERR_ALIGN;
    // A cluster of 8 per row where one CTA would need more than one round of its 32,768-element loads
    // and few rows leave SMs idle.  Measured on GB300, one CTA against 8, us per call: M = 1, V =
    // 32768 3.1, 3.6; 49152 4.4, 3.6; 151936 8.1, 3.9; M = 16, V = 65536 4.6, 5.9; 98304 5.9, 6.0;
    // 151936 8.2, 5.9.
    const int C = (V > 32768 && M <= 4) || (V > 98304 && M <= 16) ? 8 : 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)C, (unsigned)M);
    cfg.blockDim = dim3(kArgThreads);
    cfg.stream = static_cast<cudaStream_t>(stream);
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = (unsigned)C;
    attr[1].val.clusterDim.y = attr[1].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = C > 1 ? 2 : 1;
    return cudaLaunchKernelEx(&cfg, argmax_kernel, static_cast<const __half*>(logits), V, C, out) ==
                   cudaSuccess
               ? LAQ_OK
               : LAQ_ERR_CUDA;
}

}  // extern "C"
