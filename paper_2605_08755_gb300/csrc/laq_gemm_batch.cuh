// laq_gemm_batch.cuh -- the dequantize-fused GEMM kernel for batches (M = 5..16, and M = 1..4 on
// wide outputs; the lines stand at batch_takes in laq_api.cu), included by the translation units
// that instantiate it (laq_gemm_batch.cu: plain X, laq_gemm_prologue.cu: X made by a fused prologue).
// Same records, extraction and group algebra as laq_gemm_kernel.cuh:
// D = sum_k (c_k + q_k) x_k on the tensor cores, y += s (D - P - z S) per group, with
// P = sum_k c_k x_k and S = sum_k x_k.
//
// What bounds a batch is instruction issue per record (16 columns x 128 rows), not HBM: 8 MMAs
// for every 8 batch rows (NB = 1 or 2), about 50 integer instructions of extraction, and the X
// fragments and group sums around them (gemm_kernel: ~380 instructions per record at M = 16, 4 KB
// of X fragments from shared memory each).  So here
//  * a warp takes TW = 2 adjacent 16-column tiles of a group: one load of the group's B fragments
//    (2 KB per 8 rows) and of its (S, P) serves two records;
//  * X sits in shared memory in fragment order -- chunk 4c + q (x[32c + 8q ..]) of batch row b of
//    group g at ((g NB + b / 8) 4 + q) 32 + (4 (b % 8) + c), xor 2q -- so a lane's fragment is 4
//    conflict-free 16-byte loads without address selection, and staging only moves 16-byte
//    chunks, four loads in flight per thread (cp.async queues behind the weight copies: 3.9 us
//    for 32 KB per CTA against 1.1, median CTA of a tracing build);
//  * S and P come from 8 NB MMAs per group against a constant A (row 0: c_k, row 1: ones), once
//    per CTA instead of once per staged chunk;
//  * D and P are two accumulator chains each (even and odd k16 steps) from zero, in the same order:
//    the tensor core truncates every sum at the magnitude of the running value (up to 1024 sum |x|),
//    so halves that stay half as long, and a P whose truncation follows D's, leave less in D - P.
//    Error against 64 bits beyond the final fp16 rounding, W4 2560 x 19456 M = 16, N(0, 1) X: 2.8e-5
//    of the result (gemm_kernel, with P by fp32 additions, 2.8e-5; one chain started at -P - z S
//    4.6e-5, one chain from zero 4.3e-5); with 1 % outliers of 50 in X 2.0e-5, 3.6e-5, 6.7e-5, 2.9e-5.
// 8 warps per CTA, two CTAs per SM: Wt tile slots x Wk = 8 / Wt teams that split the CTA's
// groups, K split further over a cluster of 1..8 CTAs (any size, so that the grid fills the SMs),
// reduced through distributed shared memory in rank order.
// Measured, us per call in a chain of calls (measure/kernel_choice.py --chain): 4096 x 24576 W3 M = 16
// gemm_kernel 42.3, this one 19.9; 2560 x 19456 W3 M = 8 10.8, 9.1, W4 M = 4 9.3, 8.0; 9728 x 2560 W4
// M = 4 6.7, 6.3; 2560 x 151936 W3 M = 1 51.2, 37.9.  Of the first about half is outside the group
// loop: launch, 45 KB of X per CTA, S and P, reduction.  S and P with conversions and branches and
// integer divisions in the reduction cost 10 us of it, cp.async for X 1.  The scales, zeros and group
// sums are loaded after the products, not held across them: at NB = TW = 2 the second accumulator
// chain otherwise spills (16 Qwen3-8B layers at M = 16 782 us, 766 so).
#pragma once
#include "laq_gemm_kernel.cuh"

namespace laq {

namespace {

struct BatchParams : Params {
    int slots;  // tile slots (warps along the tiles) per CTA
};

constexpr int kBatchWarps = 8;
constexpr int kBatchStages = 3;  // ring depth per warp, in groups (TW records each)

// 16-byte chunk of shared X: chunk j (0..15) of batch row b of phase group lg
template <int NB>
__device__ __forceinline__ int xb_slot(int lg, int b, int j) {
    const int c = j >> 2, q = j & 3;
    return ((lg * NB + (b >> 3)) * 4 + q) * 32 + ((4 * (b & 7) + c) ^ (2 * q));
}

// Which of 1024, 512, 64, 8 is row_offset<BITS>(i).
template <int BITS>
__device__ __forceinline__ constexpr int offset_index(int i) {
    return BITS == 4 ? (i & 1 ? 2 : 0) : i < 6 ? 1 : i < 12 ? 2 : i < 15 ? 3 : 2;
}

template <int BITS, int NB, int TW, bool PRO>
__global__ void __launch_bounds__(kBatchWarps * 32, 2) gemm_batch_kernel(const BatchParams p) {
    using F = RecordFmt<BITS>;
    constexpr int WPL = BITS == 4 ? 8 : 6;
    constexpr int S = kBatchStages, kSlot = TW * F::kBytes;

    pdl_launch_dependents();
    if (gridDim.y > 1) asm volatile("barrier.cluster.arrive.relaxed.aligned;\n" ::: "memory");

    extern __shared__ __align__(128) uint8_t smem[];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, c = lane & 3, R = lane >> 2;
    const int Wt = p.slots, Wk = kBatchWarps / Wt, TC = Wt * TW;
    const int slot = warp % Wt, team = warp / Wt;
    const int M = p.M, GP = p.gpp;
    const int T0 = blockIdx.x * TC, tl = slot * TW;  // the CTA's first tile, the warp's first in it
    const int C = gridDim.y, rank = blockIdx.y;
    const int g0 = (int)((long long)p.G * rank / C);
    const int g1 = (int)((long long)p.G * (rank + 1) / C);

    // shared memory: ring [8][S][TW records] (later the warps' partial sums) | X fragments
    //   [GP][NB][4][32] 16 B | (S, P) [GP][8 NB] float2 | (s, z) [GP][TC][16] half2
    //   | part [C][UL][16] fp32, UL = ceil(TC M / C) | (prologue) inv_rms [16],
    //   sums of squares by warp [8][16] and by CTA [8][16], fp32, norm weights [GP][128] fp16
    uint8_t* ring = smem;
    uint4* xs = reinterpret_cast<uint4*>(smem + kBatchWarps * S * kSlot);
    float2* ps = reinterpret_cast<float2*>(xs + (size_t)GP * NB * 128);
    uint32_t* sz = reinterpret_cast<uint32_t*>(ps + (size_t)GP * NB * 8);
    float* part = reinterpret_cast<float*>(sz + (size_t)GP * TC * 16);
    const int U = TC * M, UL = (U + C - 1) / C;  // (tile, batch row) units of 16 outputs
    // u / M and u / UL by a high multiplication (exact for u < 2^16; a divisor of 1 overflows the
    // reciprocal)
    const uint32_t inv_m = 0xffffffffu / (uint32_t)M + 1u, inv_ul = 0xffffffffu / (uint32_t)UL + 1u;
    auto tile_of = [&](int u) { return M == 1 ? u : (int)__umulhi((uint32_t)u, inv_m); };
    auto owner_of = [&](int u) { return UL == 1 ? u : (int)__umulhi((uint32_t)u, inv_ul); };
    float* inv_rms = part + (C > 1 ? C * UL * 16 : 0);

    const uint32_t ring_s =
        (uint32_t)__cvta_generic_to_shared(ring) + (uint32_t)(warp * S * kSlot);
    const uint8_t* ring_w = ring + warp * S * kSlot;

    float yacc[TW][NB][4];
#pragma unroll
    for (int t = 0; t < TW; ++t)
#pragma unroll
        for (int h = 0; h < NB; ++h)
#pragma unroll
            for (int v = 0; v < 4; ++v) yacc[t][h][v] = 0.f;

    // RMSNorm where one phase holds the CTA's whole slice of K (and every CTA has one): X and R are
    // read once, h = fp16(X + R) is staged, its sums of squares come from the staged fragments and,
    // over a cluster, from its CTAs, and the staged rows are normalised in place.  (Reading all of X
    // and R in every CTA for the sums and the slice again for staging: 120 KB per CTA at M = 8, K =
    // 2560, 4.2 us more per call than a plain GEMM; in place 3.2.)
    const bool in_place = PRO && p.pro == kProRmsNorm && p.gc <= GP && C <= p.G;
    uint4* wsm = reinterpret_cast<uint4*>(inv_rms + 16 + 2 * 8 * 16);  // w of the slice
    bool first = true;
    for (int pa = g0; pa < g1; pa += GP) {
        const int ng = min(g1, pa + GP) - pa;
        // groups of this warp: pa + team + i Wk, i < nw (none for tiles past the edge)
        const int nw = T0 + tl < p.T ? (ng - team + Wk - 1) / Wk : 0;
        // Source of the lane's next copy of each tile (a second tile past the edge repeats the
        // first; it is never stored): 16 + 16 or 16 + 8 bytes of a record.
        const uint8_t* wsrc[TW];
#pragma unroll
        for (int t = 0; t < TW; ++t)
            wsrc[t] = p.packed + lane * 16 +
                      ((size_t)(T0 + tl + (T0 + tl + t < p.T ? t : 0)) * p.G + pa + team) *
                          F::kBytes;
        const size_t wstep = (size_t)Wk * F::kBytes;
        auto issue = [&](bool more, uint32_t dst) {  // the warp's next group into a ring slot
            if (more) {
#pragma unroll
                for (int t = 0; t < TW; ++t) {
                    cp_async16(dst + t * F::kBytes + lane * 16, wsrc[t]);
                    if (F::kChunk1 == 16)
                        cp_async16(dst + t * F::kBytes + 512 + lane * 16, wsrc[t] + 512);
                    else
                        cp_async8(dst + t * F::kBytes + 512 + lane * 8, wsrc[t] + 512 - lane * 8);
                    wsrc[t] += wstep;
                }
            }
            cp_async_commit();
        };
        for (int i = 0; i < S - 1; ++i) issue(i < nw, ring_s + i * kSlot);

        if (!first) __syncthreads();  // every warp is done with the previous phase
        // (s, z) of the phase's groups and the CTA's columns as fp16 pairs (z <= 15 is exact), 4
        // columns per thread; weights, so read before the wait for the preceding kernel
        for (int u = threadIdx.x; u < ng * TC * 4; u += kBatchWarps * 32) {
            const int lg = u / (TC * 4), col = 4 * (u % (TC * 4));  // (TC is a power of two)
            if (T0 * 16 + col < p.N) {
                const size_t off = (size_t)(pa + lg) * p.N + (size_t)T0 * 16 + col;
                const uint2 sv = *reinterpret_cast<const uint2*>(p.s + off);
                const uint32_t zv = *reinterpret_cast<const uint32_t*>(p.z + off);
                uint32_t w[4];
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    const uint32_t z16 = __half_as_ushort(__ushort2half_rn((zv >> (8 * e)) & 255u));
                    w[e] = ((e < 2 ? sv.x : sv.y) >> (16 * (e & 1)) & 0xffffu) | z16 << 16;
                }
                *reinterpret_cast<uint4*>(sz + lg * TC * 16 + col) =
                    make_uint4(w[0], w[1], w[2], w[3]);
            }
        }
        if (first) {
            if (PRO && p.pro == kProRmsNorm) prefetch_l2(p.w, (size_t)p.K * 2);
            pdl_wait();  // X (and Y) belong to the preceding kernel until it completes
            if (PRO && p.pro == kProRmsNorm && !in_place) rms_rows(p, inv_rms);
            first = false;
        }
        {   // X of the phase, 16-byte chunks, several loads in flight per thread
            const int per_row = ng * 16, nu = M * per_row;  // < 2^16
            const uint32_t inv = 0xffffffffu / (uint32_t)per_row + 1u;
            constexpr int kFly = PRO ? 3 : 4;
            if (PRO && in_place)
                for (int q = threadIdx.x; q < per_row; q += kBatchWarps * 32)
                    cp_async16((uint32_t)__cvta_generic_to_shared(wsm + q),
                               p.w + (size_t)pa * 128 + q * 8);
            for (int u0 = threadIdx.x; u0 < nu; u0 += kFly * kBatchWarps * 32) {
                uint4 v[kFly], v1[PRO ? kFly : 1];
#pragma unroll
                for (int k = 0; k < kFly; ++k) {
                    const int u = u0 + k * kBatchWarps * 32;
                    if (u < nu) {
                        const int b = (int)__umulhi((uint32_t)u, inv), q = u - b * per_row;
                        const size_t col = (size_t)pa * 128 + q * 8;
                        if (PRO)
                            prologue_load(p, b, col, v[k], v1[PRO ? k : 0]);
                        else
                            v[k] = ld_cg16(p.X + (size_t)b * p.K + col);
                    }
                }
#pragma unroll
                for (int k = 0; k < kFly; ++k) {
                    const int u = u0 + k * kBatchWarps * 32;
                    if (u < nu) {
                        const int b = (int)__umulhi((uint32_t)u, inv), q = u - b * per_row;
                        const size_t col = (size_t)pa * 128 + q * 8;
                        if (PRO && in_place) {
                            v[k] = add8h(v[k], v1[PRO ? k : 0]);
                            if (p.R_out && blockIdx.x == 0)
                                *reinterpret_cast<uint4*>(p.R_out + (size_t)b * p.K + col) = v[k];
                        } else if (PRO) {
                            v[k] = prologue_math(p, col, v[k], v1[PRO ? k : 0],
                                                 p.pro == kProRmsNorm ? inv_rms[b] : 0.f);
                        }
                        xs[xb_slot<NB>(q >> 4, b, q & 15)] = v[k];
                    }
                }
            }
            asm volatile("cp.async.wait_all;\n" ::: "memory");
            __syncthreads();
        }

        // B fragments of group lg, batch rows 8h .. 8h + 7 (rows past M hold garbage; an MMA column
        // depends on its own row only, and those columns are never stored)
        auto load_b = [&](int lg, uint32_t (&B)[NB][8][2]) {
#pragma unroll
            for (int h = 0; h < NB; ++h)
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    const uint4 v = xs[((lg * NB + h) * 4 + q) * 32 + (lane ^ (2 * q))];
                    B[h][2 * q][0] = v.x;
                    B[h][2 * q][1] = v.y;
                    B[h][2 * q + 1][0] = v.z;
                    B[h][2 * q + 1][1] = v.w;
                }
        };
        if constexpr (PRO) {
            if (in_place) {
                // Sums of squares in fp32 (the tensor core truncates: on it 20 % of the rows at K =
                // 4096 had every input rounded as by 64 bits, here and in gemm_kernel 80 %).  A lane
                // of a group's fragments holds 32 of the 128 elements of row 8h + R.
                float d[NB];
#pragma unroll
                for (int h = 0; h < NB; ++h) d[h] = 0.f;
                for (int lg = warp; lg < ng; lg += kBatchWarps) {
                    uint32_t B[NB][8][2];
                    load_b(lg, B);
#pragma unroll
                    for (int h = 0; h < NB; ++h) {
                        float e0 = 0.f, e1 = 0.f;
#pragma unroll
                        for (int j = 0; j < 8; ++j)
#pragma unroll
                            for (int k = 0; k < 2; ++k) {
                                const float2 f =
                                    __half22float2(*reinterpret_cast<const __half2*>(&B[h][j][k]));
                                e0 = fmaf(f.x, f.x, e0);
                                e1 = fmaf(f.y, f.y, e1);
                            }
                        d[h] += e0 + e1;
                    }
                }
                float* wsum = inv_rms + 16;        // [8 warps][16]
                float* csum = wsum + 8 * 16;       // [C][16]
#pragma unroll
                for (int h = 0; h < NB; ++h) {
                    d[h] += __shfl_xor_sync(0xffffffffu, d[h], 1);
                    d[h] += __shfl_xor_sync(0xffffffffu, d[h], 2);
                    if (c == 0) wsum[warp * 16 + 8 * h + R] = d[h];
                }
                __syncthreads();
                if (C > 1)  // every CTA of the cluster has started
                    asm volatile("barrier.cluster.wait.aligned;\n" ::: "memory");
                for (int u = threadIdx.x; u < 16 * C; u += kBatchWarps * 32) {
                    float tot = 0.f;
#pragma unroll
                    for (int k = 0; k < kBatchWarps; ++k) tot += wsum[k * 16 + (u & 15)];
                    float* dst = C > 1 ? cg::this_cluster().map_shared_rank(csum, u >> 4) : csum;
                    dst[rank * 16 + (u & 15)] = tot;
                }
                if (C > 1)
                    cg::this_cluster().sync();
                else
                    __syncthreads();
                if (threadIdx.x < M) {  // (rows past M hold garbage)
                    float tot = 0.f;
                    for (int k = 0; k < C; ++k) tot += csum[k * 16 + threadIdx.x];
                    inv_rms[threadIdx.x] = rsqrtf(tot / (float)p.K + p.eps);
                }
                __syncthreads();
                const int per_row = ng * 16, nu = M * per_row;
                const uint32_t inv = 0xffffffffu / (uint32_t)per_row + 1u;
                for (int u = threadIdx.x; u < nu; u += kBatchWarps * 32) {
                    const int b = (int)__umulhi((uint32_t)u, inv), q = u - b * per_row;
                    uint4* x = xs + xb_slot<NB>(q >> 4, b, q & 15);
                    float h[8];
                    residual8(*x, make_uint4(0u, 0u, 0u, 0u), h);
                    *x = rms_apply(h, wsm[q], inv_rms[b]);
                }
                __syncthreads();
            }
        }
        // (S, P) of every group and row: MMA row 0 sums c_k x_k, row 1 sums x_k.  A's registers,
        // one per distinct c (bit patterns: a conversion would run at every use).
        uint32_t ca[4];
        {
            constexpr uint32_t kC[4] = {0x64006400u, 0x60006000u, 0x54005400u, 0x48004800u};
#pragma unroll
            for (int k = 0; k < 4; ++k) ca[k] = R == 0 ? kC[k] : R == 1 ? 0x3c003c00u : 0u;
        }
        for (int lg = warp; lg < ng; lg += kBatchWarps) {
            uint32_t B[NB][8][2];
            load_b(lg, B);
            float d[2][NB][4];
#pragma unroll
            for (int a = 0; a < 2; ++a)
#pragma unroll
                for (int h = 0; h < NB; ++h)
#pragma unroll
                    for (int v = 0; v < 4; ++v) d[a][h][v] = 0.f;
#pragma unroll
            for (int j = 0; j < 8; ++j) {
                const int k0 = offset_index<BITS>(2 * j), k1 = offset_index<BITS>(2 * j + 1);
#pragma unroll
                for (int h = 0; h < NB; ++h)
                    mma16816(d[j & 1][h], ca[k0], 0u, ca[k1], 0u, B[h][j][0], B[h][j][1]);
            }
            if (R < 2) {
#pragma unroll
                for (int h = 0; h < NB; ++h)
#pragma unroll
                    for (int e = 0; e < 2; ++e) {
                        float* dst = reinterpret_cast<float*>(ps + (lg * NB + h) * 8 + 2 * c + e);
                        dst[R == 0 ? 1 : 0] = d[0][h][e] + d[1][h][e];
                    }
            }
        }
        __syncthreads();

        const uint4* xq[4];  // the lane's chunk q of the group's B fragments
#pragma unroll
        for (int q = 0; q < 4; ++q) xq[q] = xs + team * NB * 128 + q * 32 + (lane ^ (2 * q));
        const float4* spp = reinterpret_cast<const float4*>(ps + team * NB * 8 + 2 * c);
        const uint32_t* szp = sz + (team * TC + tl) * 16 + R;
        int cur = 0, prev = (S - 1) * kSlot;  // ring offsets of this group and of the one before
        for (int i = 0; i < nw; ++i) {
            issue(i + S - 1 < nw, ring_s + prev);
            uint32_t B[NB][8][2];
#pragma unroll
            for (int h = 0; h < NB; ++h) {
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    const uint4 v = xq[q][h * 128];
                    B[h][2 * q][0] = v.x;
                    B[h][2 * q][1] = v.y;
                    B[h][2 * q + 1][0] = v.z;
                    B[h][2 * q + 1][1] = v.w;
                }
            }
            cp_async_wait(S - 1);
            const uint8_t* rec = ring_w + cur;
#pragma unroll
            for (int t = 0; t < TW; ++t) {
                uint32_t wd[WPL];
                const uint4 c0 = *reinterpret_cast<const uint4*>(rec + t * F::kBytes + lane * 16);
                wd[0] = c0.x; wd[1] = c0.y; wd[2] = c0.z; wd[3] = c0.w;
                if constexpr (BITS == 4) {
                    const uint4 c1 =
                        *reinterpret_cast<const uint4*>(rec + t * F::kBytes + 512 + lane * 16);
                    wd[4] = c1.x; wd[5] = c1.y; wd[6] = c1.z; wd[7] = c1.w;
                } else {
                    const uint2 c1 =
                        *reinterpret_cast<const uint2*>(rec + t * F::kBytes + 512 + lane * 8);
                    wd[4] = c1.x; wd[5] = c1.y;
                }
                float D[2][NB][4];
#pragma unroll
                for (int e = 0; e < 2; ++e)
#pragma unroll
                    for (int h = 0; h < NB; ++h)
#pragma unroll
                        for (int v = 0; v < 4; ++v) D[e][h][v] = 0.f;
                uint32_t a[8][4];
                extract<BITS>(wd, p.exps, a);
#pragma unroll
                for (int j = 0; j < 8; ++j)
#pragma unroll
                    for (int h = 0; h < NB; ++h)
                        mma16816(D[j & 1][h], a[j][0], a[j][1], a[j][2], a[j][3], B[h][j][0],
                                 B[h][j][1]);
                float2 szv[2];  // columns R and R + 8 of the tile
#pragma unroll
                for (int r = 0; r < 2; ++r) {
                    const uint32_t w = szp[16 * t + 8 * r];
                    szv[r] = __half22float2(*reinterpret_cast<const __half2*>(&w));
                }
#pragma unroll
                for (int h = 0; h < NB; ++h) {
                    const float4 sp = spp[h * 4];  // (S, P) of batch rows 8h + 2c and 8h + 2c + 1
#pragma unroll
                    for (int v = 0; v < 4; ++v) {  // y += s (D - P - z S)
                        const float d = D[0][h][v] + D[1][h][v] - (v & 1 ? sp.w : sp.y);
                        yacc[t][h][v] = fmaf(szv[v >> 1].x,
                                             fmaf(-szv[v >> 1].y, v & 1 ? sp.z : sp.x, d),
                                             yacc[t][h][v]);
                    }
                }
            }
#pragma unroll
            for (int q = 0; q < 4; ++q) xq[q] += Wk * NB * 128;
            spp += Wk * NB * 4;
            szp += Wk * TC * 16;
            prev = cur;
            cur = cur + kSlot == S * kSlot ? 0 : cur + kSlot;
        }
        asm volatile("cp.async.wait_all;\n" ::: "memory");
    }
    if (first) {  // a CTA without groups still writes Y (and CTA (0, 0) R_out) after the previous kernel
        pdl_wait();
        if (PRO && p.pro == kProRmsNorm && p.R_out) rms_rows(p, inv_rms);
    }

    // ---- reduction: teams (shared memory) -> cluster (distributed shared memory) ----
    // Partial sums [8 TW tiles][8 NB rows][16 columns], rows 20 floats apart (the lanes of a store
    // hit 32 banks); everything below moves 4 columns at a time.
    constexpr int kRow = 20;
    __syncthreads();
    float* red = reinterpret_cast<float*>(smem);
#pragma unroll
    for (int t = 0; t < TW; ++t)
#pragma unroll
        for (int h = 0; h < NB; ++h)
#pragma unroll
            for (int v = 0; v < 4; ++v)
                red[((warp * TW + t) * NB * 8 + 8 * h + 2 * c + (v & 1)) * kRow + R + 8 * (v >> 1)] =
                    yacc[t][h][v];
    __syncthreads();
    auto add4 = [](float4& a, const float4 b) {
        a.x += b.x;
        a.y += b.y;
        a.z += b.z;
        a.w += b.w;
    };
    auto store = [&](int tile, int b, int q, const float4 a) {
        if (T0 + tile < p.T) {
            const __half2 lo = __floats2half2_rn(a.x, a.y), hi = __floats2half2_rn(a.z, a.w);
            uint2 w;
            w.x = *reinterpret_cast<const uint32_t*>(&lo);
            w.y = *reinterpret_cast<const uint32_t*>(&hi);
            *reinterpret_cast<uint2*>(p.Y + (size_t)b * p.N + (size_t)(T0 + tile) * 16 + 4 * q) = w;
        }
    };
    cg::cluster_group cluster = cg::this_cluster();
    // Units [r UL, (r + 1) UL) belong to CTA r: every CTA pushes its sums over the teams there, one
    // cluster barrier, then the owner adds the C partials in rank order.
    if (C > 1 && !in_place)  // every CTA has started
        asm volatile("barrier.cluster.wait.aligned;\n" ::: "memory");
    for (int f = threadIdx.x; f < 4 * U; f += kBatchWarps * 32) {
        const int u = f >> 2, q = f & 3, tile = tile_of(u), b = u - tile * M;
        float4 a = make_float4(0.f, 0.f, 0.f, 0.f);
        for (int k = 0; k < Wk; ++k)
            add4(a, *reinterpret_cast<const float4*>(
                        red + (((size_t)k * TC + tile) * NB * 8 + b) * kRow + 4 * q));
        if (C == 1) {
            store(tile, b, q, a);
        } else {
            const int owner = owner_of(u);
            float* dst = cluster.map_shared_rank(part, owner);
            *reinterpret_cast<float4*>(dst + (rank * UL + u - owner * UL) * 16 + 4 * q) = a;
        }
    }
    if (C > 1) {
        cluster.sync();
        for (int f = threadIdx.x; f < 4 * UL; f += kBatchWarps * 32) {
            const int u = rank * UL + (f >> 2), q = f & 3;
            if (u < U) {
                float4 a = make_float4(0.f, 0.f, 0.f, 0.f);
                for (int k = 0; k < C; ++k)
                    add4(a, *reinterpret_cast<const float4*>(part + (k * UL + (f >> 2)) * 16 + 4 * q));
                const int tile = tile_of(u);
                store(tile, u - tile * M, q, a);
            }
        }
    }
}

template <int BITS, bool PRO>
const void* pick_batch(int nb, int tw) {
    if (nb == 1)
        return tw == 1 ? (const void*)gemm_batch_kernel<BITS, 1, 1, PRO>
                       : (const void*)gemm_batch_kernel<BITS, 1, 2, PRO>;
    return tw == 1 ? (const void*)gemm_batch_kernel<BITS, 2, 1, PRO>
                   : (const void*)gemm_batch_kernel<BITS, 2, 2, PRO>;
}

}  // namespace

// The plain-X instances (laq_gemm_batch.cu) and the prologue instances (laq_gemm_prologue.cu).
const void* gemm_batch_plain_kernel(int bits, int nb, int tw);
const void* gemm_batch_prologue_kernel(int bits, int nb, int tw);

}  // namespace laq
