// laq_quant.cu -- offline model-preparation kernels: the RTN group quantizer of Eq. (1) and the
// packer / unpacker of the library's record layout (both run once per weight, not per token).
//
// All of them share one work split.  A CTA of 4 warps owns 128 columns x one group of 128 rows;
// warp c owns rows 32c .. 32c+31 and its lane l columns 4l .. 4l+3, so a row of the CTA is one
// coalesced 256-byte (fp16) or 128-byte (codes) access per warp, all 32 of a lane's row loads
// are in flight together, and the rows of warp c are exactly the rows that record lanes 4r + c
// own: a column's 32 codes of the warp become its share of the words of record lane 4r + c in
// registers, one exchange with lane ^ 2 (columns r and r + 8 share words) completes the words,
// and swizzled shared memory turns them into whole 16-byte pieces of the record.
//
// Bound: HBM for pack and unpack; issue slots (about 10 instructions per weight) and HBM about
// equally for the quantizer.  The earlier forms divided in fp64 per weight, which GB300's fp64
// pipe (2 FMAs per clock and SM) held at 1190 us for 2560 x 19456, and gathered (scattered)
// single code bytes.  Quantize + pack of 2560 x 19456 at 4 bits: 1220 -> 42 us, in one kernel
// without the codes between them (laq_quantize_pack) 29 us (126 MB: 4.4 TB/s); quantize + pack +
// unpack of 12288 x 4096 at 3 bits: 1324 -> 56 us.
#include <cuda_fp16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <type_traits>

#include "laq_internal.cuh"

namespace laq {

namespace {

constexpr int kGroup = 128;
constexpr int kCols = 128;      // columns per CTA
constexpr int kThreads = 128;   // 4 warps, 32 rows each

// w / s for fp16 values with |w| <= 16 s, accurate enough that rintf() of it equals rint() of
// the exact quotient.  The residual w - q s of the first product is exact in one fma (q is
// within an ulp of w / s), so the corrected quotient is the nearest fp32 to w / s up to an ulp,
// and equals it whenever w / s has few bits: a tie k + 1/2 comes out as exactly k + 1/2.  A
// quotient that is not a tie is at least 2^-13 away from one (a multiple of the smaller ulp
// over 2 s), far more than an fp32 ulp, so it rounds to the exact quotient's side.
__device__ __forceinline__ float quotient(float w, float s, float inv) {
    const float q = w * inv;
    return fmaf(fmaf(-q, s, w), inv, q);
}

// The scale (fp16 bits) and zero of one group from its smallest and largest weight.
template <int BITS>
__device__ __forceinline__ void group_params(float lo, float hi, uint16_t* sh_out, int* z_out) {
    constexpr float qmax = (float)((1 << BITS) - 1);
    if (lo == hi) {  // constant group c: s = |c| (1 when c == 0), z = 1 for c < 0: w_hat == c
        *sh_out = lo != 0.f ? __half_as_ushort(__float2half_rn(fabsf(lo))) : (uint16_t)0x3c00u;
        *z_out = lo < 0.f ? 1 : 0;
        return;
    }
    const float l0 = fmaxf(-lo, 0.f), h0 = fmaxf(hi, 0.f);  // range widened to contain 0
    // l0 + h0 exactly: sum + err (the rounding error of adding two floats is a float)
    const float sum = l0 + h0;
    const float err = fminf(l0, h0) - (sum - fmaxf(l0, h0));
    // the smallest fp16 h with h * qmax >= l0 + h0: the product is exact in fp32 (15 bits), and
    // sum is the nearest float to l0 + h0, so comparing with sum decides unless they are equal
    auto covers = [&](uint16_t h) {
        const float p = __half2float(__ushort_as_half(h)) * qmax;
        return p > sum || (p == sum && err <= 0.f);
    };
    uint16_t h = __half_as_ushort(__float2half_rn(sum * (1.f / qmax)));  // within one fp16
    if (!covers(h)) {
        h = (uint16_t)(h + 1);
    } else if (h > 0 && covers((uint16_t)(h - 1))) {
        h = (uint16_t)(h - 1);
    }
    if (h < 0x0400u) h = 0x0400u;  // smallest normal fp16
    const float s = __half2float(__ushort_as_half(h));
    *sh_out = h;
    *z_out = (int)rintf(quotient(l0, s, 1.f / s));
}

// ---- record words of 4 columns x 32 rows (layout in laq.h) ----
// slot 0: the column is r of its record, slot 1: r + 8.  A column's share of record word w.
template <int BITS>
struct ColumnWords {
    static constexpr int kWords = BITS == 4 ? 8 : 6;
    uint32_t w[4][kWords];

    __device__ __forceinline__ void clear() {
#pragma unroll
        for (int j = 0; j < 4; ++j)
#pragma unroll
            for (int k = 0; k < kWords; ++k) w[j][k] = 0u;
    }
    // pair i of column j: codes of rows 2i (low half) and 2i + 1 (high half)
    __device__ __forceinline__ void put(int j, int i, uint32_t pair, int slot) {
        if (BITS == 4) {
            w[j][i >> 1] |= pair << (4 * (i & 1) + 8 * slot);
        } else if (i < 6) {
            w[j][i] |= pair << (1 + 9 * slot);
        } else if (i < 12) {
            w[j][i - 6] |= pair << (4 + 9 * slot);
        } else if (i < 15) {
            const uint32_t v = pair << 7;
            w[j][2 * (i - 12)] |= slot ? 0u : v;
            w[j][2 * (i - 12) + 1] |= slot ? v : 0u;
        } else {
#pragma unroll
            for (int b = 0; b < 3; ++b) {
                const uint32_t v = (pair >> b) & 0x00010001u;
                w[j][b] |= slot ? 0u : v;
                w[j][b + 3] |= slot ? v : 0u;
            }
        }
    }
    __device__ __forceinline__ uint32_t get(int j, int i, int slot) const {
        if (BITS == 4) return (w[j][i >> 1] >> (4 * (i & 1) + 8 * slot)) & 0x000f000fu;
        if (i < 6) return (w[j][i] >> (1 + 9 * slot)) & 0x00070007u;
        if (i < 12) return (w[j][i - 6] >> (4 + 9 * slot)) & 0x00070007u;
        if (i < 15)
            return ((slot ? w[j][2 * (i - 12) + 1] : w[j][2 * (i - 12)]) >> 7) & 0x00070007u;
        uint32_t v = 0;
#pragma unroll
        for (int b = 0; b < 3; ++b) v |= ((slot ? w[j][b + 3] : w[j][b]) & 0x00010001u) << b;
        return v;
    }
};

// Staging of the CTA's 8 records: piece x = 4r + c of record tile t (16 bytes; at b = 3 the
// second pieces are 8 bytes) sits at a swizzled position, so that the 8 (16) lanes of a store
// phase, which differ in r by twos and in t, hit different banks, as do consecutive pieces.
template <int BITS>
struct Stage {
    uint4 first[8 * 32];
    typename std::conditional<BITS == 4, uint4, uint2>::type second[8 * 32];
    __device__ static int p16(int t, int x) { return t * 32 + (x ^ ((x >> 3) & 3) ^ ((t & 1) << 2)); }
    __device__ static int p2(int t, int x) {
        return BITS == 4 ? p16(t, x)
                         : t * 32 + (x ^ (x >> 4) ^ ((t & 1) << 1) ^ ((t & 2) << 1));
    }
};

// Complete the words (columns r and r + 8 sit in lanes l and l ^ 2) and write the CTA's records.
template <int BITS>
__device__ __forceinline__ void store_records(ColumnWords<BITS>& cw, Stage<BITS>& st, int64_t n0,
                                              int64_t N, int64_t G, int64_t g,
                                              uint8_t* __restrict__ packed) {
    constexpr int NW = ColumnWords<BITS>::kWords;
    const int lane = threadIdx.x & 31, c = threadIdx.x >> 5, slot = (lane >> 1) & 1;
    const int tile = lane >> 2;
#pragma unroll
    for (int j = 0; j < 2; ++j) {  // slot 0 completes columns 0, 1 of its four, slot 1 2, 3
        uint32_t v[NW];
#pragma unroll
        for (int k = 0; k < NW; ++k) {
            const uint32_t give = slot ? cw.w[j][k] : cw.w[j + 2][k];
            const uint32_t mine = slot ? cw.w[j + 2][k] : cw.w[j][k];
            v[k] = mine | __shfl_xor_sync(0xffffffffu, give, 2);
        }
        const int x = 4 * (4 * (lane & 1) + j + 2 * slot) + c;
        st.first[Stage<BITS>::p16(tile, x)] = make_uint4(v[0], v[1], v[2], v[3]);
        if constexpr (BITS == 4)
            st.second[Stage<BITS>::p2(tile, x)] = make_uint4(v[4], v[5], v[6], v[7]);
        else
            st.second[Stage<BITS>::p2(tile, x)] = make_uint2(v[4], v[5]);
    }
    __syncthreads();
    const int64_t T0 = n0 >> 4, T = N >> 4;
    constexpr int64_t rec = 256 * BITS;
#pragma unroll
    for (int k = 0; k < 2; ++k) {
        const int t = (int)(threadIdx.x >> 5) + 4 * k;
        if (T0 + t < T) {
            uint8_t* dst = packed + ((T0 + t) * G + g) * rec;
            reinterpret_cast<uint4*>(dst)[lane] = st.first[Stage<BITS>::p16(t, lane)];
            if constexpr (BITS == 4)
                reinterpret_cast<uint4*>(dst + 512)[lane] = st.second[Stage<BITS>::p2(t, lane)];
            else
                reinterpret_cast<uint2*>(dst + 512)[lane] = st.second[Stage<BITS>::p2(t, lane)];
        }
    }
}

// Four fp16 weights of row `p` at columns 0 .. 3 past it (cols of them exist).
template <bool VEC>
__device__ __forceinline__ uint2 load_w4(const uint16_t* p, int cols) {
    if (VEC) return cols > 0 ? *reinterpret_cast<const uint2*>(p) : make_uint2(0u, 0u);
    uint32_t v[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) v[j] = j < cols ? p[j] : 0u;
    return make_uint2(v[0] | v[1] << 16, v[2] | v[3] << 16);
}

template <bool VEC>
__device__ __forceinline__ void store_c4(uint8_t* p, uint32_t v, int cols) {
    if (VEC) {
        if (cols > 0) *reinterpret_cast<uint32_t*>(p) = v;
    } else {
#pragma unroll
        for (int j = 0; j < 4; ++j)
            if (j < cols) p[j] = (uint8_t)(v >> (8 * j));
    }
}

template <bool VEC>
__device__ __forceinline__ uint32_t load_c4(const uint8_t* p, int cols) {
    if (VEC) return cols > 0 ? *reinterpret_cast<const uint32_t*>(p) : 0u;
    uint32_t v = 0;
#pragma unroll
    for (int j = 0; j < 4; ++j)
        if (j < cols) v |= (uint32_t)p[j] << (8 * j);
    return v;
}

__device__ __forceinline__ __half2 as_half2(uint32_t v) {
    return *reinterpret_cast<const __half2*>(&v);
}

// Quantize one group of 128 columns: codes[K][N] (PACK false) or packed records (PACK true).
// VEC: 8-byte row accesses (N % 4 == 0, W 8-byte and codes 4-byte aligned).
//
// All arithmetic is fp32 and still makes exactly the decisions of the rule in laq.h: see
// quotient() and group_params().
template <int BITS, bool VEC, bool PACK>
__global__ void __launch_bounds__(kThreads)
quantize_kernel(const uint16_t* __restrict__ W, int64_t N, int64_t G, uint8_t* __restrict__ codes,
                uint8_t* __restrict__ packed, uint16_t* __restrict__ s,
                uint8_t* __restrict__ z) {
    constexpr int qmax = (1 << BITS) - 1;
    __shared__ __align__(16) uint16_t lo_sm[4][kCols], hi_sm[4][kCols];
    __shared__ __align__(16) float s_sm[kCols], inv_sm[kCols];
    __shared__ __align__(16) int z_sm[kCols];
    const int lane = threadIdx.x & 31, c = threadIdx.x >> 5;
    const int64_t n0 = (int64_t)blockIdx.x * kCols, g = blockIdx.y, n = n0 + 4 * lane;
    const int cols = (int)min((int64_t)4, max((int64_t)0, N - n));
    const int64_t row0 = (g * kGroup + 32 * c) * N + n;

    uint2 d[32];
#pragma unroll
    for (int i = 0; i < 32; ++i) d[i] = load_w4<VEC>(W + row0 + i * N, cols);
    uint32_t lo[2] = {d[0].x, d[0].y}, hi[2] = {d[0].x, d[0].y};
#pragma unroll
    for (int i = 1; i < 32; ++i) {
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const uint32_t v = h ? d[i].y : d[i].x;
            const __half2 a = __hmin2(as_half2(lo[h]), as_half2(v));
            const __half2 b = __hmax2(as_half2(hi[h]), as_half2(v));
            lo[h] = *reinterpret_cast<const uint32_t*>(&a);
            hi[h] = *reinterpret_cast<const uint32_t*>(&b);
        }
    }
    *reinterpret_cast<uint2*>(&lo_sm[c][4 * lane]) = make_uint2(lo[0], lo[1]);
    *reinterpret_cast<uint2*>(&hi_sm[c][4 * lane]) = make_uint2(hi[0], hi[1]);
    __syncthreads();
    {   // thread t: the parameters of column t
        const int t = threadIdx.x;
        float l = __half2float(__ushort_as_half(lo_sm[0][t]));
        float h = __half2float(__ushort_as_half(hi_sm[0][t]));
#pragma unroll
        for (int k = 1; k < 4; ++k) {
            l = fminf(l, __half2float(__ushort_as_half(lo_sm[k][t])));
            h = fmaxf(h, __half2float(__ushort_as_half(hi_sm[k][t])));
        }
        uint16_t sh;
        int zz;
        group_params<BITS>(l, h, &sh, &zz);
        const float sv = __half2float(__ushort_as_half(sh));
        s_sm[t] = sv;
        inv_sm[t] = 1.f / sv;
        z_sm[t] = zz;
        if (n0 + t < N) {
            s[g * N + n0 + t] = sh;
            z[g * N + n0 + t] = (uint8_t)zz;
        }
    }
    __syncthreads();
    // rint by adding 1.5 * 2^23: the low bits of the sum's pattern are the rounded integer
    constexpr float kMagic = 12582912.f;
    constexpr int kMagicBits = 0x4b400000;
    const float4 sv4 = *reinterpret_cast<const float4*>(&s_sm[4 * lane]);
    const float4 iv4 = *reinterpret_cast<const float4*>(&inv_sm[4 * lane]);
    const int4 zv4 = *reinterpret_cast<const int4*>(&z_sm[4 * lane]);
    const float sv[4] = {sv4.x, sv4.y, sv4.z, sv4.w}, iv[4] = {iv4.x, iv4.y, iv4.z, iv4.w};
    const int zo[4] = {zv4.x - kMagicBits, zv4.y - kMagicBits, zv4.z - kMagicBits,
                       zv4.w - kMagicBits};
    const int slot = (lane >> 1) & 1;
    ColumnWords<BITS> cw;
    if (PACK) cw.clear();
#pragma unroll
    for (int i = 0; i < 16; ++i) {  // rows 2i, 2i + 1
        uint32_t q[2][4];
#pragma unroll
        for (int e = 0; e < 2; ++e) {
            const float2 a = __half22float2(as_half2(d[2 * i + e].x));
            const float2 b = __half22float2(as_half2(d[2 * i + e].y));
            const float w[4] = {a.x, a.y, b.x, b.y};
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const float m = quotient(w[j], sv[j], iv[j]) + kMagic;
                q[e][j] = (uint32_t)min(max(__float_as_int(m) + zo[j], 0), qmax);  // then add z
            }
        }
        if (PACK) {
#pragma unroll
            for (int j = 0; j < 4; ++j) cw.put(j, i, q[0][j] | q[1][j] << 16, slot);
        } else {
#pragma unroll
            for (int e = 0; e < 2; ++e)
                store_c4<VEC>(codes + row0 + (2 * i + e) * N,
                              q[e][0] | q[e][1] << 8 | q[e][2] << 16 | q[e][3] << 24, cols);
        }
    }
    if constexpr (PACK) {
        __shared__ Stage<BITS> st;
        store_records<BITS>(cw, st, n0, N, G, g, packed);
    }
}

// codes[K][N] -> records.  VEC: codes 4-byte aligned (N % 16 == 0 always).
template <int BITS, bool VEC>
__global__ void __launch_bounds__(kThreads)
pack_kernel(const uint8_t* __restrict__ codes, int64_t N, int64_t G,
            uint8_t* __restrict__ packed) {
    constexpr uint32_t mask = BITS == 4 ? 0x000f000fu : 0x00070007u;
    __shared__ Stage<BITS> st;
    const int lane = threadIdx.x & 31, c = threadIdx.x >> 5;
    const int64_t n0 = (int64_t)blockIdx.x * kCols, g = blockIdx.y, n = n0 + 4 * lane;
    const int cols = n < N ? 4 : 0;
    const uint8_t* src = codes + (g * kGroup + 32 * c) * N + n;
    uint32_t d[32];
#pragma unroll
    for (int i = 0; i < 32; ++i) d[i] = load_c4<VEC>(src + i * N, cols);
    const int slot = (lane >> 1) & 1;
    ColumnWords<BITS> cw;
    cw.clear();
#pragma unroll
    for (int i = 0; i < 16; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j)  // byte j of rows 2i and 2i + 1
            cw.put(j, i, __byte_perm(d[2 * i], d[2 * i + 1], (4 + j) << 8 | j) & mask, slot);
    store_records<BITS>(cw, st, n0, N, G, g, packed);
}

// records -> codes[K][N]
template <int BITS, bool VEC>
__global__ void __launch_bounds__(kThreads)
unpack_kernel(const uint8_t* __restrict__ packed, int64_t N, int64_t G,
              uint8_t* __restrict__ codes) {
    __shared__ Stage<BITS> st;
    const int lane = threadIdx.x & 31, c = threadIdx.x >> 5;
    const int64_t n0 = (int64_t)blockIdx.x * kCols, g = blockIdx.y, n = n0 + 4 * lane;
    const int64_t T0 = n0 >> 4, T = N >> 4;
    constexpr int64_t rec = 256 * BITS;
#pragma unroll
    for (int k = 0; k < 2; ++k) {
        const int t = c + 4 * k;
        if (T0 + t < T) {
            const uint8_t* src = packed + ((T0 + t) * G + g) * rec;
            st.first[Stage<BITS>::p16(t, lane)] = reinterpret_cast<const uint4*>(src)[lane];
            if constexpr (BITS == 4)
                st.second[Stage<BITS>::p2(t, lane)] =
                    reinterpret_cast<const uint4*>(src + 512)[lane];
            else
                st.second[Stage<BITS>::p2(t, lane)] =
                    reinterpret_cast<const uint2*>(src + 512)[lane];
        }
    }
    __syncthreads();
    if (n >= N) return;
    const int slot = (lane >> 1) & 1, tile = lane >> 2;
    ColumnWords<BITS> cw;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        const int x = 4 * (4 * (lane & 1) + j) + c;
        const uint4 a = st.first[Stage<BITS>::p16(tile, x)];
        cw.w[j][0] = a.x; cw.w[j][1] = a.y; cw.w[j][2] = a.z; cw.w[j][3] = a.w;
        if constexpr (BITS == 4) {
            const uint4 b = st.second[Stage<BITS>::p2(tile, x)];
            cw.w[j][4] = b.x; cw.w[j][5] = b.y; cw.w[j][6] = b.z; cw.w[j][7] = b.w;
        } else {
            const uint2 b = st.second[Stage<BITS>::p2(tile, x)];
            cw.w[j][4] = b.x; cw.w[j][5] = b.y;
        }
    }
    uint8_t* dst = codes + (g * kGroup + 32 * c) * N + n;
#pragma unroll
    for (int i = 0; i < 16; ++i) {
        uint32_t p[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) p[j] = cw.get(j, i, slot);
#pragma unroll
        for (int e = 0; e < 2; ++e) {  // row 2i + e: byte 2e of each pair
            const uint32_t a = __byte_perm(p[0], p[1], (4 + 2 * e) << 4 | 2 * e);
            const uint32_t b = __byte_perm(p[2], p[3], (4 + 2 * e) << 4 | 2 * e);
            store_c4<VEC>(dst + (2 * i + e) * N, __byte_perm(a, b, 0x5410), 4);
        }
    }
}

bool aligned(const void* p, uintptr_t a) { return (reinterpret_cast<uintptr_t>(p) % a) == 0; }

dim3 grid_of(int64_t K, int64_t N) {
    return dim3((unsigned)((N + kCols - 1) / kCols), (unsigned)(K / kGroup));
}

template <int BITS>
void run_quantize(const uint16_t* W, int64_t K, int64_t N, uint8_t* codes, uint8_t* packed,
                  uint16_t* s, uint8_t* z, cudaStream_t stream) {
    const int64_t G = K / kGroup;
    const dim3 grid = grid_of(K, N);
    const bool vec = N % 4 == 0 && aligned(W, 8) && aligned(codes, 4);
    if (packed) {
        if (vec)
            quantize_kernel<BITS, true, true><<<grid, kThreads, 0, stream>>>(W, N, G, codes, packed, s, z);
        else
            quantize_kernel<BITS, false, true><<<grid, kThreads, 0, stream>>>(W, N, G, codes, packed, s, z);
    } else if (vec) {
        quantize_kernel<BITS, true, false><<<grid, kThreads, 0, stream>>>(W, N, G, codes, packed, s, z);
    } else {
        quantize_kernel<BITS, false, false><<<grid, kThreads, 0, stream>>>(W, N, G, codes, packed, s, z);
    }
}

}  // namespace

cudaError_t launch_quantize(const uint16_t* W, int64_t K, int64_t N, int bits, uint8_t* codes,
                            uint8_t* packed, uint16_t* s, uint8_t* z, cudaStream_t stream) {
    if (bits == 3)
        run_quantize<3>(W, K, N, codes, packed, s, z, stream);
    else
        run_quantize<4>(W, K, N, codes, packed, s, z, stream);
    return cudaGetLastError();
}

cudaError_t launch_pack(const uint8_t* codes, int64_t K, int64_t N, int bits, uint8_t* packed,
                        cudaStream_t stream) {
    const dim3 grid = grid_of(K, N);
    const int64_t G = K / kGroup;
    const bool vec = aligned(codes, 4);
    if (bits == 3) {
        if (vec) pack_kernel<3, true><<<grid, kThreads, 0, stream>>>(codes, N, G, packed);
        else pack_kernel<3, false><<<grid, kThreads, 0, stream>>>(codes, N, G, packed);
    } else {
        if (vec) pack_kernel<4, true><<<grid, kThreads, 0, stream>>>(codes, N, G, packed);
        else pack_kernel<4, false><<<grid, kThreads, 0, stream>>>(codes, N, G, packed);
    }
    return cudaGetLastError();
}

cudaError_t launch_unpack(const uint8_t* packed, int64_t K, int64_t N, int bits, uint8_t* codes,
                          cudaStream_t stream) {
    const dim3 grid = grid_of(K, N);
    const int64_t G = K / kGroup;
    const bool vec = aligned(codes, 4);
    if (bits == 3) {
        if (vec) unpack_kernel<3, true><<<grid, kThreads, 0, stream>>>(packed, N, G, codes);
        else unpack_kernel<3, false><<<grid, kThreads, 0, stream>>>(packed, N, G, codes);
    } else {
        if (vec) unpack_kernel<4, true><<<grid, kThreads, 0, stream>>>(packed, N, G, codes);
        else unpack_kernel<4, false><<<grid, kThreads, 0, stream>>>(packed, N, G, codes);
    }
    return cudaGetLastError();
}

}  // namespace laq
