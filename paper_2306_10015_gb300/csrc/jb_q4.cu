// jb_q4.cu -- PerturbParameters on 4-bit weights (Section 3, Training Speed:
// layer weights are dequantized before the noise is added and quantized again).
//
// Code (the paper fixes none; it cites QLoRA's NormalFloat): 16 levels built
// from quantiles of N(0,1) and scaled to [-1, 1] (gen_q4_levels.py); blocks of
// 64 elements share one fp32 scale, the largest |w| of the block; a weight is
// level[code] * scale; quantizing picks the nearest level (ties to the lower).
//
// Per element: dequantize, w' = w + eps z as one fused multiply-add (as in the
// plain perturbation) with the same z as every other path (global index
// flat_offset + i), then per block scale' = max |w'| and
// code' = nearest level of w' / scale'. Codes and scales are rewritten in place.
// A lane takes 32 consecutive elements, so a 64-element block is two lanes and
// its maximum is one butterfly shuffle.
//
// Dequantizing reads two levels at once: the codes of elements 4b and 4b + 2 are
// nibbles 0 and 2 of a 16-bit group (4b + 1 and 4b + 3: nibbles 1 and 3), and a
// shared-memory table holds (level[a], level[b]) at byte offset 8 a + 2048 b, so
// one shift and one mask of the code word give the address of both.
//
// Nearest level = the number of midpoints strictly below x. Consecutive
// midpoints are more than 1/16 apart, so each bucket [j/16, (j+1)/16) of
// [-1, 1) holds at most one; with b = floor(16 x) (exact in fp32), the code is
// (midpoints below the bucket) + (x > the bucket's midpoint, if any): one
// shared-memory read and one comparison instead of a 4-step binary search.
#include <cuda_bf16.h>

#include <algorithm>
#include <atomic>
#include <cstddef>
#include <cstring>

#include "jb_internal.h"
#include "jb_rng.cuh"

namespace jb {
namespace {

// gen_q4_levels.py
constexpr float kQ4Level[16] = {
    -0x1.000000p+0f, -0x1.6311acp-1f, -0x1.0b8d60p-1f, -0x1.924c0ap-2f, -0x1.21b102p-2f,
    -0x1.7851c6p-3f, -0x1.72d976p-4f, 0x0.0p+0f,       0x1.4421acp-4f,  0x1.47c076p-3f,
    0x1.f54804p-3f,  0x1.582f80p-2f,  0x1.c1002ap-2f,  0x1.1eba52p-1f,  0x1.70ca9ap-1f,
    0x1.000000p+0f};

__constant__ float c_level[16] = {
    kQ4Level[0], kQ4Level[1], kQ4Level[2],  kQ4Level[3],  kQ4Level[4],  kQ4Level[5],
    kQ4Level[6], kQ4Level[7], kQ4Level[8],  kQ4Level[9],  kQ4Level[10], kQ4Level[11],
    kQ4Level[12], kQ4Level[13], kQ4Level[14], kQ4Level[15]};
// midpoints (L_j + L_j+1) / 2 of the fp32 levels, rounded to fp32 (gen_q4_levels.py)
constexpr float kQ4Mid[15] = {
    -0x1.b188d6p-1f, -0x1.374f86p-1f, -0x1.d4b364p-2f, -0x1.59fe86p-2f, -0x1.ddd9e4p-3f,
    -0x1.18df40p-3f, -0x1.72d976p-5f, 0x1.4421acp-5f,  0x1.e9d14cp-4f,  0x1.9e843cp-3f,
    0x1.2969c0p-2f,  0x1.8c97d4p-2f,  0x1.ff3a68p-2f,  0x1.47c276p-1f,  0x1.b8654cp-1f};

// Buckets: entry j < 32 = (the midpoint in [(j - 16)/16, (j - 15)/16) or +inf, the number
// of midpoints below (j - 16)/16 in each of the eight nibbles); entries 32 .. 63 = (+inf,
// 15), for x = 1. For x in [-1, 1], y = x 2^-12 + 1 + 2^-12 rounded toward minus infinity
// lies in [1, 1 + 2^-11], and its fraction bits 7 .. 12 are floor(16 (x + 1)): the exact
// value is 1 + 2^11 (x + 1) 2^-23, every multiple of 2^-16 there is representable, so
// rounding down never crosses one. The mask gives the byte offset of a row of 16 equal
// 8-byte entries, one for each lane of a half warp: a 64-bit read serves half a warp at a
// time, so no two lanes meet in a bank. A NaN x gets an unspecified code.
constexpr float kQ4IdxScale = 0x1p-12f, kQ4IdxBias = 0x1.001p+0f;  // 1 + 2^-12
constexpr int kBucketRow = 16;
constexpr int kQ4Epl = 32;  // elements per lane and tile

struct Bucket {
    float mid;
    uint32_t below;
};
struct Buckets {
    Bucket b[64];
};
constexpr Buckets make_buckets() {
    Buckets t{};
    for (int j = 0; j < 64; ++j) {
        const float lo = static_cast<float>(j - 16) * 0.0625f;
        uint32_t below = 0;
        t.b[j].mid = __builtin_inff();
        for (int k = 0; k < 15; ++k) {
            if (kQ4Mid[k] < lo) ++below;
            if (kQ4Mid[k] >= lo && kQ4Mid[k] < lo + 0.0625f) t.b[j].mid = kQ4Mid[k];
        }
        t.b[j].below = below * 0x11111111u;
    }
    return t;
}
__constant__ Buckets c_bucket = make_buckets();

// ow with nibble K replaced by the code of x. The count of midpoints is there in every
// nibble and x above the bucket's own midpoint adds one in nibble K (a count is at most 14
// where a midpoint can lie above), so a code costs a comparison, a predicated addition and
// one bitwise select, and no shift; shifting each code into place cost 14 instructions of
// the integer-multiply pipe per four elements, the pipe that bounds this kernel.
template <int K>
__device__ __forceinline__ uint32_t put_code(uint32_t ow, float x, float y, const float2* bucket,
                                             uint32_t lane_off) {
    uint32_t off;
    asm("lop3.b32 %0, %1, %2, %3, 0xEA;" : "=r"(off) : "r"(__float_as_uint(y)), "r"(0x1F80u), "r"(lane_off));
    const float2 e = *reinterpret_cast<const float2*>(reinterpret_cast<const char*>(bucket) + off);
    uint32_t v = __float_as_uint(e.y);
    asm("{\n\t.reg .pred p;\n\tsetp.gt.f32 p, %1, %2;\n\t@p add.u32 %0, %0, %3;\n\t}"
        : "+r"(v) : "f"(x), "f"(e.x), "n"(1u << (4 * K)));
    if constexpr (K == 0) return v;
    uint32_t r;
    asm("lop3.b32 %0, %1, %2, %3, 0xE4;" : "=r"(r) : "r"(v), "r"(ow), "r"(0xFu << (4 * K)));
    return r;
}

// max(a, b, c) in one instruction
__device__ __forceinline__ float fmax3(float a, float b, float c) {
    float r;
    asm("max.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(b), "f"(c));
    return r;
}

// (level[a], level[b]) at byte offset 8 a + 2048 b: 15 * 256 + 16 entries, 256 used
constexpr int kPairEntries = 15 * 256 + 16;

// Levels of the codes in nibbles (n, n + 2) of cw, n = 4 BB + (ODD ? 1 : 0):
// elements (4b, 4b + 2) or (4b + 1, 4b + 3) of the word's block b = BB.
template <int BB, bool ODD>
__device__ __forceinline__ float2 pair_at(const float2* pair, uint32_t cw) {
    constexpr int sh = 16 * BB + (ODD ? 4 : 0) - 3;
    const uint32_t off = (sh < 0 ? cw << (-sh) : cw >> sh) & 0x7878u;
    return *reinterpret_cast<const float2*>(reinterpret_cast<const char*>(pair) + off);
}

template <int B>
__device__ __forceinline__ void dequant_block(const float2* pair, const uint32_t* cw, float2& le, float2& lo) {
    le = pair_at<B % 2, false>(pair, cw[B / 2]);
    lo = pair_at<B % 2, true>(pair, cw[B / 2]);
}

constexpr int kThreadsQ4 = 1024;

template <typename P>
__device__ __forceinline__ const SegParamQ4& q4_seg(const P& p, uint32_t s) {
    return reinterpret_cast<const SegParamQ4*>(p.data)[s];
}

// A warp tile is 1024 consecutive elements of one tensor, 32 per lane; tiles and spans as
// in the update's kernels. Bound, like those, by operand reads and the instruction mix
// (151 instructions and 218 cycles per scheduler and four elements of a warp; FMA pipe 76%
// busy, shared-memory reads 36%). Eight warps per scheduler at 64 registers, 36 bytes of them
// spilled: 2^28 elements in 358 us (768 threads 364, 640 threads 365, 512 threads 386). With
// lanes numbered across tensors, codes shifted into place and bank conflicts on the buckets
// it took 397.
// ONE_HI: the pair's constants hold for every block of the launch; otherwise they are
// formed for the high word of each block's own index (2^28 elements 358 -> 376 us).
template <bool ONE_HI, typename P>
__global__ void __launch_bounds__(kThreadsQ4) q4_perturb_kernel(const __grid_constant__ P p) {
    constexpr int E = kQ4Epl, NB = E / 4, NW = E / 8;
    static_assert(NB == 8 && 64 == 2 * E, "two 32-element lanes per scale block");
    __shared__ float2 pair[kPairEntries];
    __shared__ float2 bucket[64 * kBucketRow];
    for (int i = threadIdx.x; i < 256; i += kThreadsQ4)
        pair[(i & 15) + 256 * (i >> 4)] = make_float2(c_level[i & 15], c_level[i >> 4]);
    for (int i = threadIdx.x; i < 64 * kBucketRow; i += kThreadsQ4) {
        const Bucket b = c_bucket.b[i / kBucketRow];
        bucket[i] = make_float2(b.mid, __uint_as_float(b.below));
    }
    __syncthreads();  // every thread reaches this before any work

    const uint32_t lane = threadIdx.x & 31u;
    const uint32_t lane_off = 8u * (lane % kBucketRow);
    SeedParam sc = seed_param(p.seed, p.block_hi, p.eps);
    const float2 eps2 = splat(p.eps);
    const uint64_t span = p.span;
    const uint64_t stride = span * (static_cast<uint64_t>(gridDim.x) * (kThreadsQ4 / 32));
    uint32_t s = 0;  // tensor cursor; only moves forward
    // all 32 lanes run every iteration (the block maximum is a warp shuffle)
    for (uint64_t t0 = span * (static_cast<uint64_t>(threadIdx.x >> 5) * gridDim.x + blockIdx.x);
         t0 < p.n_tiles; t0 += stride) {
        const uint32_t t_end = static_cast<uint32_t>(t0 + span < p.n_tiles ? t0 + span : p.n_tiles);
        for (uint32_t t = static_cast<uint32_t>(t0); t < t_end; ++t) {
            if (t >= q4_seg(p, s + 1).tile0) {
                uint32_t lo = s + 1, hi = p.n_segs;
                while (hi - lo > 1) {
                    const uint32_t m = (lo + hi) / 2;
                    if (q4_seg(p, m).tile0 <= t) lo = m;
                    else hi = m;
                }
                s = lo;
            }
            const SegParamQ4& g = q4_seg(p, s);
            const uint64_t first = static_cast<uint64_t>(t - g.tile0) * (32u * E);
            const uint64_t i0 = first + E * lane;
            const bool fast = first + 32u * E <= g.n;  // the same for every lane
            const bool any = fast || i0 < g.n;
            const bool full = fast || i0 + E <= g.n;
            uint8_t* codes = reinterpret_cast<uint8_t*>(g.codes) + i0 / 2;
            float* scale = reinterpret_cast<float*>(g.scale) + i0 / 64;

            uint32_t cw[NW];  // 32 codes, 8 per word
#pragma unroll
            for (int j = 0; j < NW; ++j) cw[j] = 0u;
            if (full) {
                if (g.wide) {
                    const uint4 v = __ldcs(reinterpret_cast<const uint4*>(codes));
                    cw[0] = v.x; cw[1] = v.y; cw[2] = v.z; cw[3] = v.w;
                } else {
#pragma unroll
                    for (int j = 0; j < NW; j += 2) {  // codes are 8-byte aligned
                        const uint2 v = *reinterpret_cast<const uint2*>(codes + 4 * j);
                        cw[j] = v.x;
                        cw[j + 1] = v.y;
                    }
                }
            } else if (any) {
#pragma unroll
                for (int b = 0; b < E / 2; ++b)
                    if (i0 + 2 * b < g.n) cw[b / 4] |= static_cast<uint32_t>(codes[b]) << (8 * (b % 4));
            }
            const float2 s2 = splat(any ? *scale : 0.0f);

            // dequantize and perturb: w = fma(cos or sin, eps r, level * scale), the
            // Philox words of block b + 1 computed while block b is transformed;
            // wv[2b] = elements (4b, 4b + 2), wv[2b + 1] = (4b + 1, 4b + 3)
            float2 wv[E / 2];
            const uint32_t blk = g.blk0 + static_cast<uint32_t>(i0 >> 2);
            const auto words = [&](int b) {
                if constexpr (!ONE_HI) {
                    const uint64_t at = ((static_cast<uint64_t>(g.blk_hi) << 32) | g.blk0) + (i0 >> 2) + b;
                    sc = seed_param(p.seed, static_cast<uint32_t>(at >> 32), p.eps);
                    return philox_block(sc, blk + b);
                }
                return philox_block(sc, block_after(block_ctr(blk + (b & ~1)), b & 1));
            };
            uint4 wcur = words(0);
#pragma unroll
            for (int b = 0; b < NB; ++b) {
                uint4 wnext;
                if (b + 1 < NB) wnext = words(b + 1);
                const Polar2 o = polar2(wcur);
                if (b + 1 < NB) wcur = wnext;
                const float2 rc = mul2(eps2, o.rr);
                float2 le, lo;
                if (b % 2 == 0) dequant_block<0>(pair, cw + b / 2, le, lo);
                else dequant_block<1>(pair, cw + b / 2, le, lo);
                wv[2 * b] = fma2(o.cm, rc, mul2(le, s2));
                wv[2 * b + 1] = fma2(o.sm, rc, mul2(lo, s2));
            }
            // elements past the end of the tensor do not count towards the maximum
            if (!full) {
#pragma unroll
                for (int b = 0; b < NB; ++b) {
                    if (i0 + 4 * b + 0 >= g.n) wv[2 * b].x = 0.0f;
                    if (i0 + 4 * b + 2 >= g.n) wv[2 * b].y = 0.0f;
                    if (i0 + 4 * b + 1 >= g.n) wv[2 * b + 1].x = 0.0f;
                    if (i0 + 4 * b + 3 >= g.n) wv[2 * b + 1].y = 0.0f;
                }
            }
            float m = 0.0f;
#pragma unroll
            for (int i = 0; i < E / 2; ++i) m = fmax3(m, fabsf(wv[i].x), fabsf(wv[i].y));
            // block maximum over the two lanes of the block (lanes 2j, 2j + 1)
            m = fmaxf(m, __shfl_xor_sync(0xFFFFFFFFu, m, 1));
            // 1/m rounded down: every |w / m| then rounds to at most 1, so x needs no clamp
            const float2 inv2 = splat(m > 0.0f ? __frcp_rd(m) : 0.0f);

            // quantize again: x = w / m, its bucket from y = RD(x 2^-12 + 1 + 2^-12)
            uint32_t ow[NW];
#pragma unroll
            for (int j = 0; j < NW; ++j) {
                float2 x[4], y[4];  // elements (0, 2), (1, 3), (4, 6), (5, 7) of the word
#pragma unroll
                for (int h = 0; h < 4; ++h) {
                    x[h] = mul2(wv[4 * j + h], inv2);
                    y[h] = __ffma2_rd(x[h], splat(kQ4IdxScale), splat(kQ4IdxBias));
                }
                uint32_t o = put_code<0>(0u, x[0].x, y[0].x, bucket, lane_off);
                o = put_code<1>(o, x[1].x, y[1].x, bucket, lane_off);
                o = put_code<2>(o, x[0].y, y[0].y, bucket, lane_off);
                o = put_code<3>(o, x[1].y, y[1].y, bucket, lane_off);
                o = put_code<4>(o, x[2].x, y[2].x, bucket, lane_off);
                o = put_code<5>(o, x[3].x, y[3].x, bucket, lane_off);
                o = put_code<6>(o, x[2].y, y[2].y, bucket, lane_off);
                ow[j] = put_code<7>(o, x[3].y, y[3].y, bucket, lane_off);
            }
            if (full) {
                if (g.wide) {
                    __stcs(reinterpret_cast<uint4*>(codes), make_uint4(ow[0], ow[1], ow[2], ow[3]));
                } else {
#pragma unroll
                    for (int j = 0; j < NW; j += 2)
                        *reinterpret_cast<uint2*>(codes + 4 * j) = make_uint2(ow[j], ow[j + 1]);
                }
            } else if (any) {
#pragma unroll
                for (int b = 0; b < E / 2; ++b) {
                    if (i0 + 2 * b >= g.n) continue;
                    const uint8_t byte = static_cast<uint8_t>(ow[b / 4] >> (8 * (b % 4)));
                    // an odd tail leaves the unused high nibble of the last byte as it was
                    codes[b] = (i0 + 2 * b + 1 < g.n) ? byte
                                                      : static_cast<uint8_t>((codes[b] & 0xF0u) | (byte & 0x0Fu));
                }
            }
            if (any && (lane & 1u) == 0u) *scale = m;
        }
    }
}

std::atomic<int> g_q4_grid[64][4];

template <bool ONE_HI, typename P>
cudaError_t launch_q4(P& p, int slot, cudaStream_t stream) {
    auto kernel = q4_perturb_kernel<ONE_HI, P>;
    int dev = 0;
    cudaError_t err = cudaGetDevice(&dev);
    if (err != cudaSuccess) return err;
    int grid = dev < 64 ? g_q4_grid[dev][slot].load(std::memory_order_relaxed) : 0;
    if (grid <= 0) {
        int sms = 0, per_sm = 0;
        err = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
        if (err != cudaSuccess) return err;
        err = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, kThreadsQ4, 0);
        if (err != cudaSuccess) return err;
        grid = sms * (per_sm > 0 ? per_sm : 1);
        if (dev < 64) g_q4_grid[dev][slot].store(grid, std::memory_order_relaxed);
    }
    // spans as in the update's launches
    const uint64_t warps = static_cast<uint64_t>(grid) * (kThreadsQ4 / 32);
    p.span = 4;
    while (p.span > 1 && p.n_tiles < 8 * warps * p.span) p.span /= 2;
    const uint32_t needed = (p.n_tiles + p.span - 1) / p.span;
    if (needed < static_cast<uint32_t>(grid)) grid = static_cast<int>(needed);
    kernel<<<grid, kThreadsQ4, 0, stream>>>(p);
    return cudaGetLastError();
}

}  // namespace

void q4_levels_host(float out[16]) {
    for (int i = 0; i < 16; ++i) out[i] = kQ4Level[i];
}

cudaError_t enqueue_q4(const SeedRaw& seed, float eps, const Q4Seg* segs, size_t n_segs, cudaStream_t stream) {
    using P = Q4Launch<kParamBytes>;
    static thread_local P p;  // ~32 KB: keep it off the stack
    p.seed = seed;
    p.eps = eps;
    constexpr size_t room = P::kBytes / sizeof(SegParamQ4) - 1;  // and the sentinel
    SegParamQ4* table = reinterpret_cast<SegParamQ4*>(p.data);
    size_t i = 0;
    uint64_t at = 0;  // elements of segs[i] already launched
    while (i < n_segs) {
        size_t count = 0;
        uint64_t tiles = 0;
        bool one_hi = true;
        p.block_hi = static_cast<uint32_t>((segs[i].fo + at) >> 34);
        while (i < n_segs && count < room && tiles < (1ull << 30)) {
            const uint64_t n = std::min<uint64_t>(segs[i].n - at, 1ull << 40);  // keeps a tile number in 32 bits
            const uint64_t fo = segs[i].fo + at;
            SegParamQ4& g = table[count++];
            g.codes = segs[i].codes + at / 2;
            g.scale = segs[i].scale + at / 64 * 4;
            g.n = n;
            g.blk0 = static_cast<uint32_t>(fo >> 2);
            g.blk_hi = static_cast<uint32_t>(fo >> 34);
            g.tile0 = static_cast<uint32_t>(tiles);
            g.wide = (g.codes & 15ull) == 0 ? 1u : 0u;
            // (a lane past the end of a tensor draws nothing that is kept)
            if ((fo >> 34) != p.block_hi || ((fo + n - 1) >> 34) != p.block_hi) one_hi = false;
            tiles += (n + 32 * kQ4Epl - 1) / (32 * kQ4Epl);
            at += n;
            if (at == segs[i].n) {
                ++i;
                at = 0;
            }
        }
        table[count].tile0 = static_cast<uint32_t>(tiles);
        p.n_segs = static_cast<uint32_t>(count);
        p.n_tiles = static_cast<uint32_t>(tiles);
        cudaError_t err;
        const size_t used = (count + 1) * sizeof(SegParamQ4);
        if (used <= kSmallParamBytes) {
            Q4Launch<kSmallParamBytes> q;
            std::memcpy(&q, &p, offsetof(P, data) + used);
            err = one_hi ? launch_q4<true>(q, 0, stream) : launch_q4<false>(q, 1, stream);
        } else {
            err = one_hi ? launch_q4<true>(p, 2, stream) : launch_q4<false>(p, 3, stream);
        }
        if (err != cudaSuccess) return err;
    }
    return cudaSuccess;
}

}  // namespace jb
