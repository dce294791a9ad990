// jb_kernels.cu -- sm_103a kernels of the seeded-perturbation hot path.
//
//   seeded_kernel<T>         the step update (Section 2; Algorithm 1):
//                            theta_e <- round_T(theta_e + sum_k c_k z_e(s_k)),
//                            the K pairs regenerated in registers, so theta is
//                            read once and written once whatever K is.
//   one_seed_kernel<T, M>    one pair: PerturbParameters(theta, eps, s) (Algorithm 1,
//                            subroutine), theta_e <- round_T(fma(s_e, eps r_e, theta_e)),
//                            and the update at K = 1, in place or from a source table.
//   general_update_kernel<T> the update read from one table and written to
//                            another, seeds in groups rounded to T after each
//                            (the backup-fused restore and the multi-step replay).
//   checksum_kernel<T>       the model checksum of ChecksumMatch (Algorithm 1).
//   debug kernels            raw Philox words, z by element, Box-Muller of given
//                            words (test hooks only).
//
// Design. Nothing here is a dense contraction, so there is no tensor-core
// work: the cost is one HBM read and write of theta (2 sizeof(T) bytes per
// element) against K Gaussians per element (a quarter Philox4x32-10 block and
// half a Box-Muller transform each). A warp tile is 32 V consecutive 16-byte
// vectors of one segment, lane l taking vectors l, l + 32, ..., so every load and
// store instruction of a warp covers 512 contiguous bytes (fully coalesced, 128-bit
// per thread). Each thread keeps V vectors in flight for instruction-level
// parallelism, in their storage form while the pairs are summed. The grid is
// persistent; a warp strides over spans of consecutive tiles.
// The K (seed, coefficient) pairs live in the kernel parameter space and are
// read with warp-uniform indices (constant-bank broadcast). Accumulation is a
// fixed-order fp32 FMA chain with no atomics: results are bitwise repeatable
// and independent of the grid and of how tensors are split.
#include <cuda_bf16.h>

#include <algorithm>
#include <atomic>
#include <cstddef>
#include <cstring>
#include <type_traits>

#include "jb_internal.h"
#include "jb_offgrid.h"
#include "jb_rng.cuh"

namespace jb {
namespace {

// The shape of a kernel: vectors per thread and warp tile, threads per CTA (one CTA per
// SM: the threads set how many registers each may use) and unrolling of the seed loop.
// What bounds these kernels is the reading of operands and the issue of the instruction
// mix (the bf16 update: 92 instructions and 154 cycles per scheduler for a warp's block and
// pair, 82% of them with the FMA pipe that multiplies integers busy), not latency or
// memory, so the shapes differ by a few percent. Measured on 2^28 elements (us):
//   update, K = 16   fp32 5 x 512: 4111 (4 x 512: 4147, 4 x 768: 4171, 6 x 512: 4156)
//                    bf16 3 x 512: 4163 (2 x 512: 4332, 2 x 768: 4171, 2 x 640: 4156)
//                    (at 128 registers a thread: bf16 3 x 512 spills 20 bytes of them, fp32
//                    5 x 512 without round keys 12)
//   replay, 10 pairs fp32 4 x 512: 2663 (4 x 768: 2871, 6 x 512: 2812)
//                    bf16 2 x 512: 2667 (2 x 768: 2794, 3 x 512: 2817)
//   one pair         fp32 4 x 1024: 318 (4 x 768: 338, 4 x 512: 329; HBM alone: 316)
//                    bf16 4 x 1024: 282 and 291 (perturbation, update; 6 x 768: 286 and 290,
//                    8 x 768: 284 and 285, but up to 14% slower at 8M to 32M elements;
//                    4 x 512: 306 and 303)
//   one pair that writes source and destination, fp32 (memory alone: 474): 16 warps per SM
//                    4 x 512: 482; more of them in flight cost bandwidth (4 x 1024: 525)
//   checksum         fp32 6 x 512: 152 (8 x 512: 153, 4 x 512: 157), bf16 80 (81, 83);
//                    1.3B bf16 364: 7.2 TB/s
// Small tables take one vector per thread in every kernel, and their launch fewer
// parameter bytes: a scheduler needs about one warp's worth of blocks to be busy, so what
// counts is that all 608 have some. The line lies where the large shape gives most of its
// 16 warps per SM a tile (us, one vector / large shape: K = 32 update fp32 512K elements
// 27 / 29, 1M 43 / 39, 2M 84 / 76; bf16 256K 14 / 25, 512K 25 / 35, 1M 43 / 47, 1.5M 62 / 61,
// 3M 111 / 104; replay of 10 pairs fp32 512K 12 / 12, 1M 18 / 16, bf16 512K 11 / 13, 1M
// 16 / 16; perturbation fp32 512K 4.8 / 6.2, 1M 4.8 / 6.3, 2M 8.2 / 6.2, bf16 1.5M 6.1 / 6.3,
// 3M 8.2 / 7.5; checksum fp32 1M 6.2 / 7.2, 2M 7.9 / 7.7, bf16 2M 6.2 / 7.3, 4M 8.2 / 8.1).
// It counts tiles, also those that short tensors leave mostly empty: 2000 tensors of 64 to
// 800 elements take 83 to 152 us in the K = 32 update.
template <int V_, int THREADS_, int UNROLL_, int CTAS_ = 0>
struct Shape {
    static constexpr int V = V_, THREADS = THREADS_, UNROLL = UNROLL_;
    static constexpr int CTAS = CTAS_;  // most CTAs per SM (0: as many as fit)
};

constexpr uint64_t kSmallTiles = 1600;  // tiles of the large shape
// Tables that cross a multiple of 2^34 elements (checksum of bf16: 2^35) take one launch
// with a set of pairs for each of two high words up to this many tiles, or twice as many for
// one pair: two launches of fewer tiles leave more warps idle at their ends and cost about
// 4 us each (two launches / one, us: fp32 perturbation 4M elements 14.2 / 8.2, 8M 18.6 /
// 14.3, 128M 170 / 168; K = 3 update 4.6M fp32 24.5 / 20.5, bf16 26.1 / 20.4, 128M 421 / 420
// and 418 / 415; bf16 perturbation 256M 290 / 287). Above it the kernels for one high word
// are up to 2 % faster, and in fp32 the round keys come with the pairs. The checksum takes
// one launch always (256M fp32 161 / 155).
constexpr uint64_t kMergeTiles = 1u << 17;

template <typename T>
struct Traits;
template <>
struct Traits<float> {
    static constexpr int E = 4;                     // elements per 16-byte vector
    static constexpr uint64_t SPLIT_TILES = 608;    // most 128-element tiles of the split update
    using Update = Shape<5, 512, 2>;
    using General = Shape<4, 512, 2>;
    using Pair = Shape<4, 1024, 1>;
    using Refresh = Shape<4, 512, 1, 1>;  // one pair that writes the source too
    using Sum = Shape<6, 512, 1>;
    using Small = Shape<1, 512, 2>;
};
template <>
struct Traits<__nv_bfloat16> {
    static constexpr int E = 8;
    static constexpr uint64_t SPLIT_TILES = 1216;
    using Update = Shape<3, 512, 2>;
    using General = Shape<2, 512, 2>;
    using Pair = Shape<4, 1024, 1>;
    using Refresh = Pair;
    using Sum = Shape<6, 512, 1>;
    using Small = Shape<1, 512, 2>;
};

__device__ __forceinline__ float bf16_lo(uint32_t w) { return __uint_as_float(w << 16); }
__device__ __forceinline__ float bf16_hi(uint32_t w) { return __uint_as_float(w & 0xFFFF0000u); }
__device__ __forceinline__ uint32_t pack_bf16(float lo, float hi) {
    const __nv_bfloat162 h = __floats2bfloat162_rn(lo, hi);  // nearest, ties to even
    return *reinterpret_cast<const uint32_t*>(&h);
}

// The elements of a vector as fp32, in the order of the accumulators: pair [b][0] holds
// elements 4b and 4b + 2 (the even ones of Philox block b), [b][1] holds 4b + 1, 4b + 3.
__device__ __forceinline__ void unpack(uint4 w, float2 (&x)[1][2]) {
    x[0][0] = make_float2(__uint_as_float(w.x), __uint_as_float(w.z));
    x[0][1] = make_float2(__uint_as_float(w.y), __uint_as_float(w.w));
}
__device__ __forceinline__ uint4 pack(const float2 (&x)[1][2]) {
    return make_uint4(__float_as_uint(x[0][0].x), __float_as_uint(x[0][1].x),
                      __float_as_uint(x[0][0].y), __float_as_uint(x[0][1].y));
}
__device__ __forceinline__ void unpack(uint4 w, float2 (&x)[2][2]) {
    x[0][0] = make_float2(bf16_lo(w.x), bf16_lo(w.y));
    x[0][1] = make_float2(bf16_hi(w.x), bf16_hi(w.y));
    x[1][0] = make_float2(bf16_lo(w.z), bf16_lo(w.w));
    x[1][1] = make_float2(bf16_hi(w.z), bf16_hi(w.w));
}
__device__ __forceinline__ uint4 pack(const float2 (&x)[2][2]) {
    return make_uint4(pack_bf16(x[0][0].x, x[0][1].x), pack_bf16(x[0][0].y, x[0][1].y),
                      pack_bf16(x[1][0].x, x[1][1].x), pack_bf16(x[1][0].y, x[1][1].y));
}

__device__ __forceinline__ uint4 load_vec(uint64_t a) { return __ldcs(reinterpret_cast<const uint4*>(a)); }
__device__ __forceinline__ void store_vec(uint64_t a, uint4 w) { __stcs(reinterpret_cast<uint4*>(a), w); }

// Memory for the vectors off the 16-byte grid of their flat offset (jb_offgrid.h). They
// take kernels of their own (OFF; in the common ones the choice costs registers). One
// perturbation of 2^28 elements, against element by element: bf16 295 us at 8 bytes, 306
// at 4, 410 at 2 (541 to 615 before; 281 on the grid), fp32 349 and 368 (427; 317). One such
// tensor takes all of its launch there: 16 tensors of 2^28 elements on the grid and one of
// 1000 off it, us, without and with that one: perturbation fp32 318 / 324, bf16 283 / 285,
// K = 2 update 561 / 570 and 563 / 568, K = 16 4106 / 4125 and 4161 / 4160.
struct Global {
    __device__ uint2 load64(uint64_t a) const { return __ldcs(reinterpret_cast<const uint2*>(a)); }
    __device__ uint32_t load32(uint64_t a) const { return __ldcs(reinterpret_cast<const uint32_t*>(a)); }
    __device__ uint16_t load16(uint64_t a) const { return *reinterpret_cast<const uint16_t*>(a); }
    __device__ void store64(uint64_t a, uint2 v) const { __stcs(reinterpret_cast<uint2*>(a), v); }
    __device__ void store32(uint64_t a, uint32_t v) const { __stcs(reinterpret_cast<uint32_t*>(a), v); }
    __device__ void store16(uint64_t a, uint16_t v) const { *reinterpret_cast<uint16_t*>(a) = v; }
};

// Elements [first, last) of the window at address a (the others read as zero bits).
template <typename T>
__device__ __forceinline__ uint4 load_part(uint64_t a, int first, int last) {
    constexpr int E = Traits<T>::E, BITS = 8 * static_cast<int>(sizeof(T));
    uint32_t ww[4] = {0u, 0u, 0u, 0u};
#pragma unroll
    for (int t = 0; t < E; ++t) {
        if (t < first || t >= last) continue;
        uint32_t bits;
        if constexpr (sizeof(T) == 2) bits = reinterpret_cast<const uint16_t*>(a)[t];
        else bits = reinterpret_cast<const uint32_t*>(a)[t];
        ww[t * BITS / 32] |= bits << ((t * BITS) % 32);
    }
    return make_uint4(ww[0], ww[1], ww[2], ww[3]);
}
template <typename T>
__device__ __forceinline__ void store_part(uint64_t a, int first, int last, uint4 w) {
    constexpr int E = Traits<T>::E, BITS = 8 * static_cast<int>(sizeof(T));
    const uint32_t ww[4] = {w.x, w.y, w.z, w.w};
#pragma unroll
    for (int t = 0; t < E; ++t) {
        if (t < first || t >= last) continue;
        const uint32_t bits = ww[t * BITS / 32] >> ((t * BITS) % 32);
        if constexpr (sizeof(T) == 2) reinterpret_cast<uint16_t*>(a)[t] = static_cast<uint16_t>(bits);
        else reinterpret_cast<uint32_t*>(a)[t] = bits;
    }
}

template <typename P>
__device__ __forceinline__ const typename P::Pair& seed_at(const P& p, uint32_t k) {
    return reinterpret_cast<const typename P::Pair*>(p.data)[k];
}
template <typename P>
__device__ __forceinline__ const typename P::Seg& seg_at(const P& p, uint32_t s) {
    return reinterpret_cast<const typename P::Seg*>(p.data + p.seg_at)[s];
}
// The segment of tile t, which is not before segment s. Most steps stay in a segment.
template <typename P>
__device__ __forceinline__ uint32_t find_seg(const P& p, uint32_t s, uint32_t t) {
    if (t < seg_at(p, s + 1).tile0) return s;
    uint32_t lo = s + 1, hi = p.n_segs;
    while (hi - lo > 1) {
        const uint32_t m = (lo + hi) / 2;
        if (seg_at(p, m).tile0 <= t) lo = m;
        else hi = m;
    }
    return lo;
}

__device__ __forceinline__ uint64_t dst_of(const SegParam& g) { return g.base; }
__device__ __forceinline__ uint64_t dst_of(const SegParamOut& g) { return g.dst; }

enum Store { kInPlace, kToDst, kNowhere };

// What a kernel's launch may hold: vectors on the 16-byte grid alone, off it too, or that
// and a second high word of the indices.
enum Tables { kOnGrid, kOffGrid, kTwoHighs };

// Runs op(x, blk, present) on each of this warp's tiles and stores the result (in place,
// to the destination table, and then also back to the source when also_src, or nowhere):
// x[j] is vector 32 j + lane of the tile in storage form, blk the low word of the first
// Philox block of x[0] (x[j] is at blk + 32 j B; stored nowhere: of the window, and B is
// 1), and present (stored nowhere only) how many vectors the segment has from x[0] on. A
// warp takes spans of p.span consecutive tiles, strided by the number of warps in the
// grid; spans that follow one another go to different SMs, so that a few tiles occupy as
// many SMs. Which warp handles a tile never changes a result: every element's value
// depends only on its own stored value, its global index and the seeds. Vectors that are
// partial (the ends of a segment) go element by element. op's last argument says whether
// the tile's indices have the launch's second high word.
template <typename T, typename S, Store TO, Tables HOLDS, typename P, typename Op>
__device__ __forceinline__ void visit_tiles(const P& p, bool also_src, Op&& op) {
    constexpr int E = Traits<T>::E, V = S::V;
    constexpr uint32_t B = TO == kNowhere ? 1 : E / 4, kTileVec = 32u * V;
    constexpr bool OFF = HOLDS != kOnGrid;
    const uint32_t lane = threadIdx.x & 31u;
    const uint64_t span = p.span;
    const uint64_t stride = span * (static_cast<uint64_t>(gridDim.x) * (S::THREADS / 32));
    uint32_t s = 0;  // segment cursor; only moves forward
    for (uint64_t t0 = span * (static_cast<uint64_t>(threadIdx.x >> 5) * gridDim.x + blockIdx.x);
         t0 < p.n_tiles; t0 += stride) {
        uint32_t t = static_cast<uint32_t>(t0);
        const uint32_t t_end = static_cast<uint32_t>(t0 + span < p.n_tiles ? t0 + span : p.n_tiles);
        s = find_seg(p, s, t);
        while (true) {
            const auto& g = seg_at(p, s);
            const uint32_t next = seg_at(p, s + 1).tile0;
            const uint32_t stop = next < t_end ? next : t_end;
            const uint32_t v_lo = g.lo, v_hi = g.full;
            const uint32_t load_align = OFF ? g.load : 16u, store_align = OFF ? g.store : 16u;
            // from lane 0, so that the compiler knows it for the same in all lanes and reads the
            // pairs with uniform indices (K = 16 update of 2^28 elements 4340 -> 4140 us)
            const bool second = HOLDS == kTwoHighs && __shfl_sync(0xFFFFFFFFu, s >= p.second_from ? 1 : 0, 0) != 0;
            uint32_t v = (t - g.tile0) * kTileVec;  // first vector of the tile
            uint64_t src = g.base + 16ull * (v + lane);
            uint64_t dst = dst_of(g) + 16ull * (v + lane);
            uint32_t blk = g.blk0 + (v + lane) * B;
#pragma unroll 1
            for (; t < stop; ++t) {
                const bool fast = v >= v_lo && v + kTileVec <= v_hi;  // the same for every lane
                uint4 x[V];
                if (fast && load_align == 16u) {
#pragma unroll
                    for (int j = 0; j < V; ++j) x[j] = load_vec(src + 512ull * j);
                } else if (fast) {
#pragma unroll
                    for (int j = 0; j < V; ++j) x[j] = load_off_grid(Global(), src + 512ull * j, load_align);
                } else {
#pragma unroll
                    for (int j = 0; j < V; ++j) {
                        const uint32_t vj = v + lane + 32u * j;
                        if (vj >= v_lo && vj < v_hi && load_align == 16u) {
                            x[j] = load_vec(src + 512ull * j);
                        } else {
                            const uint64_t e0 = static_cast<uint64_t>(vj) * E;
                            const int last = e0 >= g.end ? 0 : (g.end - e0 < E ? static_cast<int>(g.end - e0) : E);
                            x[j] = load_part<T>(src + 512ull * j, vj == 0u ? static_cast<int>(g.head) : 0, last);
                        }
                    }
                }
                if constexpr (TO == kNowhere) {
                    const uint64_t vecs = (g.end + E - 1) / E;  // a tile has at least one
                    op(x, blk, fast ? kTileVec : static_cast<uint32_t>(vecs < v + lane ? 0 : vecs - v - lane),
                       second);
                } else {
                    op(x, blk, second);
                }
                constexpr bool TO_DST = TO == kToDst;
                const uint64_t out = TO_DST ? dst : src;
                if constexpr (TO == kNowhere) {
                } else if (fast && store_align == 16u) {
#pragma unroll
                    for (int j = 0; j < V; ++j) {
                        store_vec(out + 512ull * j, x[j]);
                        if (TO_DST && also_src) {
                            if (load_align == 16u) store_vec(src + 512ull * j, x[j]);
                            else store_off_grid(Global(), src + 512ull * j, load_align, x[j]);
                        }
                    }
                } else if (fast) {
#pragma unroll
                    for (int j = 0; j < V; ++j) {
                        store_off_grid(Global(), out + 512ull * j, store_align, x[j]);
                        if (TO_DST && also_src) {
                            if (load_align == 16u) store_vec(src + 512ull * j, x[j]);
                            else store_off_grid(Global(), src + 512ull * j, load_align, x[j]);
                        }
                    }
                } else {
#pragma unroll
                    for (int j = 0; j < V; ++j) {
                        const uint32_t vj = v + lane + 32u * j;
                        if (vj >= v_lo && vj < v_hi && load_align == 16u && store_align == 16u) {
                            store_vec(out + 512ull * j, x[j]);
                            if (TO_DST && also_src) store_vec(src + 512ull * j, x[j]);
                        } else {
                            const uint64_t e0 = static_cast<uint64_t>(vj) * E;
                            const int last = e0 >= g.end ? 0 : (g.end - e0 < E ? static_cast<int>(g.end - e0) : E);
                            const int first = vj == 0u ? static_cast<int>(g.head) : 0;
                            store_part<T>(out + 512ull * j, first, last, x[j]);
                            if (TO_DST && also_src) store_part<T>(src + 512ull * j, first, last, x[j]);
                        }
                    }
                }
                v += kTileVec;
                src += 16ull * kTileVec;
                dst += 16ull * kTileVec;
                blk += kTileVec * B;
            }
            if (t == t_end) break;
            ++s;
        }
    }
}

// acc_even += c z_even, acc_odd += c z_odd for the Gaussians of one Philox block.
// The scale c is applied to the radius (rc = c r, rounded once) and each product
// c z is formed as one fused multiply-add of the signed cosine or sine with rc: one
// packed multiply fewer per block than scaling z = cos r after it is rounded.
__device__ __forceinline__ void accum_block(uint4 w, float2 c, float2& acc_even, float2& acc_odd) {
    const Polar2 o = polar2(w);
    const float2 rc = mul2(c, o.rr);
    acc_even = fma2(o.cm, rc, acc_even);
    acc_odd = fma2(o.sm, rc, acc_odd);
}

// x + acc with one fp32 rounding, stored as T.
template <int B>
__device__ __forceinline__ uint4 add_round(uint4 raw, const float2 (&acc)[B][2]) {
    float2 x[B][2];
    unpack(raw, x);
#pragma unroll
    for (int b = 0; b < B; ++b) {
        x[b][0] = add2(x[b][0], acc[b][0]);
        x[b][1] = add2(x[b][1], acc[b][1]);
    }
    return pack(x);
}

// theta += sum_k c_k z_k over the tile, accumulated in fp32 in seed order; with GROUPS,
// rounded to T after each pair that ends a group. The Philox words of pair k + 1 are
// computed while pair k is transformed and accumulated, block by block: the
// integer-multiply and the fp32 work are independent and interleave in one instruction
// stream (one block's words ahead instead of the tile's: 4% slower). The last pair is
// peeled. Philox round 1's product of the block counter is the same for every pair.
template <typename T, typename S, bool GROUPS, typename P>
__device__ __forceinline__ void update_tile(const P& p, uint4 (&x)[S::V], uint32_t blk, bool second) {
    constexpr int V = S::V, B = Traits<T>::E / 4, NB = V * B;
    const uint32_t n = p.n_seeds, first = second ? n : 0u;
    if (GROUPS && n == 0u) return;  // a copy
    float2 acc[V][B][2];
    BlockCtr bc[NB];
#pragma unroll
    for (int i = 0; i < NB; ++i) {
        acc[i / B][i % B][0] = acc[i / B][i % B][1] = make_float2(0.0f, 0.0f);
        bc[i] = block_ctr(blk + 32 * B * (i / B) + i % B);
    }
    uint4 w[NB];
#pragma unroll
    for (int i = 0; i < NB; ++i) w[i] = philox_block(seed_at(p, first), bc[i]);
    auto pair = [&](uint32_t k, auto more) {
        const auto& sd = seed_at(p, first + k);
        const float2 c = splat(sd.coef);
#pragma unroll
        for (int i = 0; i < NB; ++i) {
            uint4 wn;
            if constexpr (decltype(more)::value) wn = philox_block(seed_at(p, first + k + 1), bc[i]);
            accum_block(w[i], c, acc[i / B][i % B][0], acc[i / B][i % B][1]);
            if constexpr (decltype(more)::value) w[i] = wn;
        }
        if (GROUPS && sd.ends_group != 0u) {
#pragma unroll
            for (int j = 0; j < V; ++j) {
                x[j] = add_round(x[j], acc[j]);
#pragma unroll
                for (int b = 0; b < B; ++b) acc[j][b][0] = acc[j][b][1] = make_float2(0.0f, 0.0f);
            }
        }
    };
#pragma unroll S::UNROLL
    for (uint32_t k = 0; k + 1 < n; ++k) pair(k, std::true_type());
    pair(n - 1, std::false_type());
    if constexpr (!GROUPS) {
#pragma unroll
        for (int j = 0; j < V; ++j) x[j] = add_round(x[j], acc[j]);
    }
}

template <typename T, typename S, Tables HOLDS, typename P>
__global__ void __launch_bounds__(S::THREADS) seeded_kernel(const __grid_constant__ P p) {
    visit_tiles<T, S, kInPlace, HOLDS>(p, false, [&](uint4 (&x)[S::V], uint32_t blk, bool second) {
        update_tile<T, S, false>(p, x, blk, second);
    });
}

// One pair over the tile. PERTURB: theta <- fma(., ., theta) (one rounding of theta +
// eps z); otherwise a one-pair update, theta <- theta + (c z rounded to fp32), the
// arithmetic of seeded_kernel at K = 1. The Philox words of vector j + 1 are computed
// while vector j is transformed, so the integer-multiply and fp32 work of neighbouring
// vectors interleave (as the update does across seeds). A vector's second block takes its
// counter's product from the first one's (bf16 perturbation of 2^28 elements 288.8 -> 282.7
// us; further from the tile's first block: 282.7 too, but fp32 319 -> 325).
template <typename T, int V, bool PERTURB, typename P>
__device__ __forceinline__ void one_seed_tile(const P& p, uint4 (&x)[V], uint32_t blk, bool second) {
    constexpr int B = Traits<T>::E / 4;
    const SeedParam& sd = seed_at(p, second ? 1u : 0u);
    const float2 c = splat(sd.coef);
    uint4 wc[B], wn[B];
#pragma unroll
    for (int b = 0; b < B; ++b) wc[b] = philox_block(sd, block_after(block_ctr(blk), b));
#pragma unroll
    for (int j = 0; j < V; ++j) {
        if (j + 1 < V) {
#pragma unroll
            for (int b = 0; b < B; ++b) wn[b] = philox_block(sd, block_after(block_ctr(blk + 32 * B * (j + 1)), b));
        }
        float2 f[B][2];
        if constexpr (PERTURB) unpack(x[j], f);
#pragma unroll
        for (int b = 0; b < B; ++b) {
            if constexpr (!PERTURB) f[b][0] = f[b][1] = make_float2(0.0f, 0.0f);
            accum_block(wc[b], c, f[b][0], f[b][1]);
        }
        if constexpr (PERTURB) x[j] = pack(f);
        else x[j] = add_round(x[j], f);
        if (j + 1 < V) {
#pragma unroll
            for (int b = 0; b < B; ++b) wc[b] = wn[b];
        }
    }
}

enum OneSeed { kPerturbInPlace = 0, kAddInPlace = 1, kAddToDst = 2 };

template <typename T, typename S, int MODE, Tables HOLDS, typename P>
__global__ void __launch_bounds__(S::THREADS) one_seed_kernel(const __grid_constant__ P p) {
    constexpr bool TO_DST = MODE == kAddToDst;
    visit_tiles<T, S, TO_DST ? kToDst : kInPlace, HOLDS>(
        p, TO_DST && p.write_src != 0u, [&](uint4 (&x)[S::V], uint32_t blk, bool second) {
            one_seed_tile<T, S::V, MODE == kPerturbInPlace>(p, x, blk, second);
        });
}

// The generalised update: source -> destination (optionally also back to the
// source), seeds applied in groups with a rounding to the storage type after each
// group, exactly as successive in-place updates would round.
template <typename T, typename S, Tables HOLDS, typename P>
__global__ void __launch_bounds__(S::THREADS) general_update_kernel(const __grid_constant__ P p) {
    visit_tiles<T, S, kToDst, HOLDS>(p, p.write_src != 0u, [&](uint4 (&x)[S::V], uint32_t blk, bool second) {
        update_tile<T, S, true>(p, x, blk, second);
    });
}

// The update of a table so small that its elements cannot fill the GPU: the pairs are
// shared out too. A group of G warps takes one tile of 128 elements (a Philox block per
// lane); warp w forms the scaled radii and the signed cosines and sines of pairs w, w + G,
// ... of a chunk of 2 G pairs in shared memory, and the group's first warp adds them up in
// pair order, chunk c while the group forms chunk c + 1. The additions are those of
// update_tile, so the results are the same bit for bit. One warp alone needs about 350
// cycles per pair for a tile (the latency of the generator and the transform; 580 where a
// thread has the two blocks of a bf16 vector); shared out, an SM needs about 115, or 85 per
// tile where it has three or four (40 is what the issue of their instructions takes). K = 400
// update, us, without and with the split: fp32 1K to 19K elements 70 and 29, 65K 85 and 62,
// 78K 85 and 96; bf16 1K 117 and 31, 65K 119 and 62, 131K 150 and 112, 160K 150 and 156,
// 262K 150 and 222. So it ends at one tile per scheduler (608) in fp32 and at two in bf16.
// It is not slower for two pairs either (5.7 and 5.8 us for 1K elements, bound by the call).
constexpr int kSplitThreads = 512;
constexpr int kSplitWarps = kSplitThreads / 32;
constexpr int kSplitPairs = 2;

struct Drawn {
    float2 rc[32], cm[32], sm[32];  // of one pair, by lane
};

template <int ES>
__device__ __forceinline__ void load_block(uint64_t a, int first, int last, bool full, float (&x)[4]) {
    if constexpr (ES == 4) {
        if (full) {
            const float4 v = __ldcs(reinterpret_cast<const float4*>(a));
            x[0] = v.x; x[1] = v.y; x[2] = v.z; x[3] = v.w;
            return;
        }
#pragma unroll
        for (int i = 0; i < 4; ++i) x[i] = i >= first && i < last ? reinterpret_cast<const float*>(a)[i] : 0.0f;
    } else {
        uint32_t b[4];
        if (full) {
            const uint2 v = __ldcs(reinterpret_cast<const uint2*>(a));
            b[0] = v.x << 16; b[1] = v.x & 0xFFFF0000u; b[2] = v.y << 16; b[3] = v.y & 0xFFFF0000u;
        } else {
#pragma unroll
            for (int i = 0; i < 4; ++i)
                b[i] = i >= first && i < last ? static_cast<uint32_t>(reinterpret_cast<const uint16_t*>(a)[i]) << 16 : 0u;
        }
#pragma unroll
        for (int i = 0; i < 4; ++i) x[i] = __uint_as_float(b[i]);
    }
}

template <int ES>
__device__ __forceinline__ void store_block(uint64_t a, int first, int last, bool full, const float (&x)[4]) {
    if constexpr (ES == 4) {
        if (full) {
            __stcs(reinterpret_cast<float4*>(a), make_float4(x[0], x[1], x[2], x[3]));
            return;
        }
#pragma unroll
        for (int i = 0; i < 4; ++i)
            if (i >= first && i < last) reinterpret_cast<float*>(a)[i] = x[i];
    } else {
        const uint32_t lo = pack_bf16(x[0], x[1]), hi = pack_bf16(x[2], x[3]);
        if (full) {
            __stcs(reinterpret_cast<uint2*>(a), make_uint2(lo, hi));
            return;
        }
#pragma unroll
        for (int i = 0; i < 4; ++i)
            if (i >= first && i < last)
                reinterpret_cast<uint16_t*>(a)[i] = static_cast<uint16_t>((i < 2 ? lo : hi) >> (16 * (i % 2)));
    }
}

template <typename T, bool TO_DST, typename P>
__global__ void __launch_bounds__(kSplitThreads) split_update_kernel(const __grid_constant__ P p) {
    constexpr int ES = sizeof(T);
    __shared__ Drawn drawn[4 * kSplitWarps];
    const uint32_t lane = threadIdx.x & 31u, warp = threadIdx.x >> 5;
    const uint32_t G = p.span;  // warps of a group: 4, 8 or 16
    const uint32_t group = warp / G, w = warp % G, groups = kSplitWarps / G;
    Drawn* const buf = drawn + group * (4 * G);  // two chunks of 2 G pairs
    const uint32_t K = p.n_seeds, chunks = (K + 2 * G - 1) / (2 * G);
    uint32_t s = 0;
    // a group's warps see the same tiles: each reaches every barrier of its group
    for (uint64_t t = static_cast<uint64_t>(group) * gridDim.x + blockIdx.x; t < p.n_tiles;
         t += static_cast<uint64_t>(groups) * gridDim.x) {
        s = find_seg(p, s, static_cast<uint32_t>(t));
        const auto& g = seg_at(p, s);
        const uint32_t v = (static_cast<uint32_t>(t) - g.tile0) * 32u + lane;
        const uint32_t blk = g.blk0 + v;
        const BlockCtr bc = block_ctr(blk);
        const auto form = [&](uint32_t c) {
            Drawn* const to = buf + (c & 1u) * (2 * G);
#pragma unroll
            for (uint32_t r = 0; r < 2; ++r) {
                const uint32_t k = c * (2 * G) + r * G + w;
                if (k >= K) break;
                const SeedParam& sd = seed_at(p, k);
                const Polar2 o = polar2(philox_block(sd, bc));
                Drawn& d = to[r * G + w];
                d.rc[lane] = mul2(splat(sd.coef), o.rr);
                d.cm[lane] = o.cm;
                d.sm[lane] = o.sm;
            }
        };
        // the first warp holds theta and the sum: (elements 0, 2) and (1, 3) of the block
        const uint64_t e0 = 4ull * v;
        const int first = v == 0u ? static_cast<int>(g.head) : 0;
        const int last = e0 >= g.end ? 0 : (g.end - e0 < 4 ? static_cast<int>(g.end - e0) : 4);
        const bool full = v >= g.lo && v < g.full;
        const uint64_t src = g.base + 4ull * ES * v;
        float x[4];
        float2 even = make_float2(0.0f, 0.0f), odd = even;
        if (w == 0u) load_block<ES>(src, first, last, full, x);
        form(0);
        asm volatile("bar.sync %0, %1;" ::"r"(1 + group), "r"(32 * G) : "memory");
        for (uint32_t c = 0; c < chunks; ++c) {
            if (w == 0u) {
                const Drawn* const from = buf + (c & 1u) * (2 * G);
                const uint32_t n = K - c * (2 * G) < 2 * G ? K - c * (2 * G) : 2 * G;
#pragma unroll 8
                for (uint32_t i = 0; i < n; ++i) {
                    const float2 rc = from[i].rc[lane];
                    even = fma2(from[i].cm[lane], rc, even);
                    odd = fma2(from[i].sm[lane], rc, odd);
                    if (seed_at(p, c * (2 * G) + i).ends_group != 0u) {
                        x[0] = __fadd_rn(x[0], even.x);
                        x[2] = __fadd_rn(x[2], even.y);
                        x[1] = __fadd_rn(x[1], odd.x);
                        x[3] = __fadd_rn(x[3], odd.y);
                        if constexpr (ES == 2) {
#pragma unroll
                            for (int j = 0; j < 4; ++j) x[j] = __bfloat162float(__float2bfloat16_rn(x[j]));
                        }
                        even = odd = make_float2(0.0f, 0.0f);
                    }
                }
            }
            if (c + 1 < chunks) form(c + 1);
            asm volatile("bar.sync %0, %1;" ::"r"(1 + group), "r"(32 * G) : "memory");
        }
        if (w == 0u) {
            store_block<ES>(dst_of(g) + 4ull * ES * v, first, last, full, x);
            if (TO_DST && p.write_src != 0u) store_block<ES>(src, first, last, full, x);
        }
    }
}

// Model checksum (ChecksumMatch, Algorithm 1): the sum mod 2^64, over 16-byte
// windows of the global element space, of four Philox rounds of the window's
// storage words (elements outside the segment read as 0) keyed by the window
// index; per window (x1:x0) + (x3:x2). Integer addition is order-free, so one
// atomic add per CTA gives the same bits for any grid. Bound by HBM: one read
// of theta, one wide multiply pair per window and round. The tiles are those of the
// updates (1200 tensors of 20M elements in all: 111 -> 41 us against tiles that may cross
// tensors and a linear search for the tensor).
constexpr uint32_t kSumKey0 = 0x6A09E667u, kSumKey1 = 0xF3BCC908u;
constexpr int kSumRounds = 4;

__device__ __forceinline__ uint64_t window_hash(uint64_t win, uint4 w) {
    uint32_t x0 = w.x, x1 = w.y, x2 = w.z, x3 = w.w;
    uint32_t k0 = static_cast<uint32_t>(win) ^ kSumKey0;
    uint32_t k1 = static_cast<uint32_t>(win >> 32) ^ kSumKey1;
#pragma unroll
    for (int r = 0; r < kSumRounds; ++r) {
        if (r > 0) {
            k0 += kPhiloxW0;
            k1 += kPhiloxW1;
        }
        philox_round(x0, x1, x2, x3, k0, k1);
    }
    return ((static_cast<uint64_t>(x1) << 32) | x0) + ((static_cast<uint64_t>(x3) << 32) | x2);
}

// blk0 of the segments is the low word of the index of the first window; the high words,
// two of them, stand where other launches have their pairs. One CTA alone stores its sum,
// which saves the clearing of *out.
template <typename T, typename S, Tables HOLDS, typename P>
__global__ void __launch_bounds__(S::THREADS) checksum_kernel(const __grid_constant__ P p,
                                                             unsigned long long* out) {
    uint64_t sum = 0;
    visit_tiles<T, S, kNowhere, HOLDS>(p, false, [&](uint4 (&x)[S::V], uint32_t win, uint32_t present, bool second) {
        const uint32_t high = reinterpret_cast<const uint32_t*>(p.data)[second ? 1 : 0];
#pragma unroll
        for (int j = 0; j < S::V; ++j) {
            const uint64_t w = (static_cast<uint64_t>(high) << 32) | (win + 32u * j);
            if (32u * j < present) sum += window_hash(w, x[j]);
        }
    });
    // CTA reduction; every thread reaches the barrier
#pragma unroll
    for (int d = 16; d > 0; d >>= 1) sum += __shfl_down_sync(0xFFFFFFFFu, sum, d);
    __shared__ uint64_t part[S::THREADS / 32];
    if ((threadIdx.x & 31u) == 0u) part[threadIdx.x >> 5] = sum;
    __syncthreads();
    if (threadIdx.x == 0u) {
        uint64_t t = 0;
#pragma unroll
        for (int i = 0; i < S::THREADS / 32; ++i) t += part[i];
        if (p.write_src != 0u) *out = t;
        else atomicAdd(out, static_cast<unsigned long long>(t));
    }
}

__global__ void debug_philox_kernel(SeedRaw sr, uint64_t first, uint64_t n, uint32_t* out) {
    const uint64_t i = static_cast<uint64_t>(blockIdx.x) * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const uint64_t b = first + i;
    reinterpret_cast<uint4*>(out)[i] =
        philox_block(seed_param(sr, static_cast<uint32_t>(b >> 32), 0.0f), static_cast<uint32_t>(b));
}

// The Philox words of blocks [first, first + n), which agree in the high word of their
// index, folded by XOR into *out: the generator alone, with the hot path's block
// function, on a persistent grid (each thread keeps kFoldIlp blocks in flight). XOR is
// order-free, so the result does not depend on the grid.
constexpr int kFoldIlp = 4;

__global__ void __launch_bounds__(kThreads) debug_philox_fold_kernel(const __grid_constant__ SeedParam sd,
                                                                    uint32_t first, uint64_t n, uint32_t* out) {
    const uint64_t stride = static_cast<uint64_t>(gridDim.x) * kThreads;
    uint32_t acc = 0;
    for (uint64_t i = static_cast<uint64_t>(blockIdx.x) * kThreads + threadIdx.x; i < n;
         i += kFoldIlp * stride) {
#pragma unroll
        for (int u = 0; u < kFoldIlp; ++u) {
            const uint64_t j = i + u * stride;
            const uint4 w = philox_block(sd, first + static_cast<uint32_t>(j));
            if (j < n) acc ^= w.x ^ w.y ^ w.z ^ w.w;
        }
    }
#pragma unroll
    for (int d = 16; d > 0; d >>= 1) acc ^= __shfl_xor_sync(0xFFFFFFFFu, acc, d);
    if ((threadIdx.x & 31u) == 0) atomicXor(out, acc);
}

__global__ void debug_gaussian_kernel(SeedRaw sr, uint64_t first, uint64_t n, float* out) {
    const uint64_t i = static_cast<uint64_t>(blockIdx.x) * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const uint64_t e = first + i;
    const uint64_t b = e >> 2;
    const float4 z = block_gaussians(seed_param(sr, static_cast<uint32_t>(b >> 32), 0.0f),
                                     static_cast<uint32_t>(b));
    const unsigned w = static_cast<unsigned>(e & 3u);
    out[i] = w == 0 ? z.x : (w == 1 ? z.y : (w == 2 ? z.z : z.w));
}

__global__ void debug_box_muller_kernel(const uint32_t* words, uint64_t n, float* out) {
    // the transform runs on two word pairs at once, as in the kernels above
    const uint64_t i = 2 * (static_cast<uint64_t>(blockIdx.x) * blockDim.x + threadIdx.x);
    if (i >= n) return;
    const uint64_t i1 = i + 1 < n ? i + 1 : i;
    const GaussPair g = box_muller2(make_uint4(words[2 * i], words[2 * i + 1], words[2 * i1],
                                               words[2 * i1 + 1]));
    out[2 * i] = g.even.x;
    out[2 * i + 1] = g.odd.x;
    if (i + 1 < n) {
        out[2 * i + 2] = g.even.y;
        out[2 * i + 3] = g.odd.y;
    }
}

// Persistent grid: SM count x resident CTAs per SM (`most` at most, 0: no limit), cached
// per device and kernel.
constexpr int kMaxDevices = 64;

struct GridCache {
    std::atomic<int> ctas[kMaxDevices];
};

template <typename K>
cudaError_t persistent_grid(K kernel, int threads, int most, GridCache& cache, int* grid) {
    int dev = 0;
    cudaError_t err = cudaGetDevice(&dev);
    if (err != cudaSuccess) return err;
    if (dev < kMaxDevices) {
        const int cached = cache.ctas[dev].load(std::memory_order_relaxed);
        if (cached > 0) {
            *grid = cached;
            return cudaSuccess;
        }
    }
    int sms = 0, per_sm = 0;
    err = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (err != cudaSuccess) return err;
    err = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, threads, 0);
    if (err != cudaSuccess) return err;
    if (most > 0 && per_sm > most) per_sm = most;
    *grid = sms * (per_sm > 0 ? per_sm : 1);
    if (dev < kMaxDevices) cache.ctas[dev].store(*grid, std::memory_order_relaxed);
    return cudaSuccess;
}

// Launches `kernel` on the packed table. A warp takes spans of up to four tiles, so that
// the lookup of their segment is paid once; fewer where a warp would get less than eight
// spans, so that all warps end at about the same time.
template <typename S, typename P, typename K, typename... More>
cudaError_t launch(K kernel, GridCache& cache, P& p, int grid_ctas, cudaStream_t stream, More... more) {
    int grid = grid_ctas;
    if (grid <= 0) {
        cudaError_t err = persistent_grid(kernel, S::THREADS, S::CTAS, cache, &grid);
        if (err != cudaSuccess) return err;
    }
    const uint64_t warps = static_cast<uint64_t>(grid) * (S::THREADS / 32);
    p.span = 4;
    while (p.span > 1 && p.n_tiles < 8 * warps * p.span) p.span /= 2;
    const uint32_t needed = (p.n_tiles + p.span - 1) / p.span;
    if (grid_ctas <= 0 && needed < static_cast<uint32_t>(grid)) grid = static_cast<int>(needed);
    kernel<<<grid, S::THREADS, 0, stream>>>(p, more...);
    return cudaGetLastError();
}

// Tiles of the split update on `sms` SMs go to groups of 16, 8 or 4 warps, so that the
// CTAs, one per SM, have about one group per tile.
template <typename T, typename P>
cudaError_t launch_split(const Job& job, P& p) {
    static GridCache cache;
    auto kernel = split_update_kernel<T, std::is_same<typename P::Seg, SegParamOut>::value, P>;
    int sms = 0;
    cudaError_t err = persistent_grid(kernel, kSplitThreads, 1, cache, &sms);
    if (err != cudaSuccess) return err;
    const uint32_t ctas = static_cast<uint32_t>(job.grid_ctas > 0 ? job.grid_ctas : sms);
    p.span = p.n_tiles <= ctas ? 16u : p.n_tiles <= 2u * ctas ? 8u : 4u;
    const uint32_t groups = kSplitWarps / p.span;
    int grid = static_cast<int>(std::min(ctas, (p.n_tiles + groups - 1) / groups));
    if (job.grid_ctas > 0) grid = job.grid_ctas;
    kernel<<<grid, kSplitThreads, 0, job.stream>>>(p);
    return cudaGetLastError();
}

template <typename T, bool SMALL, Tables HOLDS, typename P>
cudaError_t launch_work(const Job& job, P& p) {
    static GridCache caches[4];
    using C = std::conditional_t<SMALL, typename Traits<T>::Small, typename Traits<T>::Sum>;
    using U = std::conditional_t<SMALL, typename Traits<T>::Small, typename Traits<T>::Update>;
    using G = std::conditional_t<SMALL, typename Traits<T>::Small, typename Traits<T>::General>;
    using S = std::conditional_t<SMALL, typename Traits<T>::Small, typename Traits<T>::Pair>;
    const int ctas = job.grid_ctas;
    if constexpr (std::is_same<typename P::Pair, KeyedParam>::value) {
        if constexpr (std::is_same<typename P::Seg, SegParamOut>::value)
            return launch<G>(general_update_kernel<T, G, HOLDS, P>, caches[0], p, ctas, job.stream);
        else
            return launch<U>(seeded_kernel<T, U, HOLDS, P>, caches[0], p, ctas, job.stream);
    } else if constexpr (std::is_same<typename P::Seg, SegParamOut>::value) {
        using R = std::conditional_t<SMALL, typename Traits<T>::Small, typename Traits<T>::Refresh>;
        static_assert(R::V == S::V, "one table for both");
        if (p.n_seeds == 1 && p.write_src != 0u)
            return launch<R>(one_seed_kernel<T, R, kAddToDst, HOLDS, P>, caches[2], p, ctas, job.stream);
        if (p.n_seeds == 1)
            return launch<S>(one_seed_kernel<T, S, kAddToDst, HOLDS, P>, caches[0], p, ctas, job.stream);
        return launch<G>(general_update_kernel<T, G, HOLDS, P>, caches[1], p, ctas, job.stream);
    } else {
        if (job.work == kChecksum)
            return launch<C>(checksum_kernel<T, C, HOLDS, P>, caches[3], p, ctas, job.stream, job.sum);
        if (job.work == kPerturb)
            return launch<S>(one_seed_kernel<T, S, kPerturbInPlace, HOLDS, P>, caches[0], p, ctas, job.stream);
        if (p.n_seeds == 1)
            return launch<S>(one_seed_kernel<T, S, kAddInPlace, HOLDS, P>, caches[1], p, ctas, job.stream);
        return launch<U>(seeded_kernel<T, U, HOLDS, P>, caches[2], p, ctas, job.stream);
    }
}

// Packs segments, cut at multiples of kPieceElems, into launches whose pieces share the
// high word of their block (checksum: window) indices or, if the table fits one launch that
// way, have one of two (kMergeTiles).
template <typename T, typename SEG, typename PAIR = SeedParam>
cudaError_t enqueue_t(const Job& job, const Seg* segs, const uint64_t* dst, size_t n_segs) {
    using P = Launch<SEG, PAIR, kParamBytes>;
    constexpr bool KEYED = std::is_same<PAIR, KeyedParam>::value;
    constexpr uint64_t E = Traits<T>::E, ES = sizeof(T);
    const uint64_t big_vec = 32ull * (job.work == kChecksum  ? Traits<T>::Sum::V
                                      : job.n_seeds == 1     ? Traits<T>::Pair::V  // = Refresh::V
                                      : job.work == kGeneral ? Traits<T>::General::V
                                                             : Traits<T>::Update::V);
    uint64_t big_tiles = 0;
    for (size_t k = 0; k < n_segs; ++k) big_tiles += (segs[k].n + E * big_vec - 1) / (E * big_vec);
    const bool small = big_tiles < kSmallTiles;
    // Pairs with their round keys are three times as long, so they are for tables that
    // still fit one launch; the keys save 16 additions per pair and tile. fp32, 2^28
    // elements: update K = 16 4128 -> 4111 us, replay 2713 -> 2663. The bf16 replay is
    // faster without keys (2667 / 2694); the bf16 update, the one-pair kernels and small
    // tables (more parameters to copy) gain nothing.
    constexpr bool MAY_KEY = std::is_same<T, float>::value;
    const uint64_t per_index = job.work == kChecksum ? E : 4;  // elements of a window or block
    const auto high = [&](uint64_t fo) { return static_cast<uint32_t>((fo / per_index) >> 32); };
    const uint32_t pair_bytes = job.work == kChecksum ? 16u : static_cast<uint32_t>(job.n_seeds * sizeof(PAIR));
    const bool may_merge = job.work == kChecksum || big_tiles <= (job.n_seeds == 1 ? 2 : 1) * kMergeTiles;
    bool merge = false;
    if (!KEYED && !small && may_merge && 2 * pair_bytes + (n_segs + 8) * sizeof(SEG) <= kParamBytes)
        for (size_t k = 0; k < n_segs && !merge; ++k)
            merge = high(segs[k].fo) != high(segs[0].fo) || high(segs[k].fo + segs[k].n - 1) != high(segs[0].fo);
    if constexpr (MAY_KEY && !KEYED) {
        if (!merge && (job.work == kUpdate || job.work == kGeneral) && job.n_seeds > 1 && !small &&
            job.n_seeds * sizeof(KeyedParam) + (n_segs + 1) * sizeof(SEG) <= kParamBytes)
            return enqueue_t<T, SEG, KeyedParam>(job, segs, dst, n_segs);
    }
    bool split = false;
    if ((job.work == kUpdate || job.work == kGeneral) && job.n_seeds >= kSplitPairs && small) {
        uint64_t tiles = 0;
        for (size_t k = 0; k < n_segs; ++k) tiles += (segs[k].n + 127) / 128;
        split = tiles <= Traits<T>::SPLIT_TILES;
    }
    const uint64_t tile_vec = small ? 32u : big_vec;
    const uint64_t win = split ? 4 : E;  // elements of a window: a vector, or a block
    static thread_local P p;  // ~32 KB: keep it off the stack
    p.n_seeds = static_cast<uint32_t>(job.n_seeds);
    p.write_src = job.write_src ? 1u : 0u;
    p.seg_at = merge && job.work != kChecksum ? 2 * pair_bytes : pair_bytes;
    const size_t room = (P::kBytes - p.seg_at) / sizeof(SEG) - 1;  // and the sentinel
    SEG* table = reinterpret_cast<SEG*>(p.data + p.seg_at);

    const uint64_t step = job.work == kChecksum ? 1 : win / 4;  // indices of a window
    size_t i = 0;
    uint64_t at = 0;  // elements of segs[i] already launched
    bool cleared = false;
    while (i < n_segs) {
        uint32_t his[2] = {high(segs[i].fo + at), 0u};
        size_t count = 0, second_from = ~static_cast<size_t>(0);
        uint64_t tiles = 0;
        bool off_grid = false;
        while (i < n_segs && count < room && tiles < (1ull << 30)) {
            const uint64_t fo = segs[i].fo + at;
            const bool second = second_from <= count;
            if (high(fo) != his[second ? 1 : 0]) {
                if (!merge || second) break;
                second_from = count;
                his[1] = high(fo);
            }
            const uint64_t n = std::min(segs[i].n - at, kPieceElems - fo % kPieceElems);
            const uint64_t src = segs[i].ptr + at * ES;
            const uint64_t to = dst != nullptr ? dst[i] + at * ES : src;
            SEG& g = table[count++];
            const uint64_t head = fo % win;
            g.head = static_cast<uint8_t>(head);
            g.base = src - head * ES;
            g.end = head + n;
            g.blk0 = static_cast<uint32_t>(fo / win * step);
            g.tile0 = static_cast<uint32_t>(tiles);
            // a vector's address is a multiple of its size iff the segment's is where its
            // flat offset is; otherwise vectors are put together from smaller accesses
            uint64_t where = g.base;
            if constexpr (std::is_same<SEG, SegParamOut>::value) {
                g.dst = to - head * ES;
                where = g.dst;
            }
            const uint64_t size = win * ES;
            const auto align = [size](uint64_t a) { return static_cast<uint8_t>(std::min(size, (a | size) & (~(a | size) + 1))); };
            g.load = align(g.base);
            g.store = align(where);
            if (g.load != size || g.store != size) off_grid = true;
            g.lo = head != 0 ? 1 : 0;
            g.full = static_cast<uint32_t>(g.end / win);
            if (split && (g.load != size || g.store != size)) g.full = 0;  // element by element
            const uint64_t vecs = (g.end + win - 1) / win;
            tiles += (vecs + tile_vec - 1) / tile_vec;
            at += n;
            if (at == segs[i].n) {
                ++i;
                at = 0;
            }
        }
        table[count].tile0 = static_cast<uint32_t>(tiles);
        p.n_segs = static_cast<uint32_t>(count);
        p.n_tiles = static_cast<uint32_t>(tiles);
        const bool two_highs = second_from < count;
        p.second_from = static_cast<uint32_t>(two_highs ? second_from : count);
        for (int h = 0; h < (two_highs ? 2 : 1); ++h) {
            PAIR* sp = reinterpret_cast<PAIR*>(p.data) + h * job.n_seeds;
            for (int k = 0; k < job.n_seeds; ++k) set_pair(sp[k], seed_param(job.seeds[k], his[h], job.coef[k]));
            for (int k = 0; k < job.n_groups; ++k) sp[job.group_end[k] - 1].ends_group = 1u;
            if (job.work == kUpdate) sp[job.n_seeds - 1].ends_group = 1u;
        }
        cudaError_t err;
        Job now = job;
        if (job.work == kChecksum) {
            std::memcpy(p.data, his, sizeof(his));
            // one CTA (two tiles per warp) instead of several and a cleared sum
            const bool alone = small && !cleared && i == n_segs && tiles <= 32 && job.grid_ctas <= 0;
            p.write_src = alone ? 1u : 0u;
            if (alone) now.grid_ctas = 1;
            if (!alone && !cleared) {
                err = cudaMemsetAsync(job.sum, 0, sizeof(*job.sum), job.stream);
                if (err != cudaSuccess) return err;
                cleared = true;
            }
        }
        const size_t used = p.seg_at + (count + 1) * sizeof(SEG);
        if constexpr (KEYED) {
            err = off_grid ? launch_work<T, false, kOffGrid>(now, p) : launch_work<T, false, kOnGrid>(now, p);
        } else if (two_highs) {
            err = launch_work<T, false, kTwoHighs>(now, p);
        } else if (split || (small && !off_grid)) {
            if (used > kSmallParamBytes) {
                err = split ? launch_split<T>(now, p) : launch_work<T, true, kOnGrid>(now, p);
            } else {
                Launch<SEG, PAIR, kSmallParamBytes> q;
                std::memcpy(&q, &p, offsetof(P, data) + used);
                err = split ? launch_split<T>(now, q) : launch_work<T, true, kOnGrid>(now, q);
            }
        } else if (small) {
            err = launch_work<T, true, kOffGrid>(now, p);
        } else {
            err = off_grid ? launch_work<T, false, kOffGrid>(now, p) : launch_work<T, false, kOnGrid>(now, p);
        }
        if (err != cudaSuccess) return err;
    }
    return cudaSuccess;
}

}  // namespace

cudaError_t enqueue(const Job& job, const Seg* segs, const uint64_t* dst, size_t n_segs) {
    if (job.work == kGeneral) {
        if (job.dtype == kF32) return enqueue_t<float, SegParamOut>(job, segs, dst, n_segs);
        return enqueue_t<__nv_bfloat16, SegParamOut>(job, segs, dst, n_segs);
    }
    if (job.dtype == kF32) return enqueue_t<float, SegParam>(job, segs, nullptr, n_segs);
    return enqueue_t<__nv_bfloat16, SegParam>(job, segs, nullptr, n_segs);
}

static unsigned blocks_for(uint64_t n) { return static_cast<unsigned>((n + 255) / 256); }

cudaError_t launch_debug_philox(SeedRaw seed, uint64_t first, uint64_t n, uint32_t* out,
                                cudaStream_t s) {
    if (n == 0) return cudaSuccess;
    debug_philox_kernel<<<blocks_for(n), 256, 0, s>>>(seed, first, n, out);
    return cudaGetLastError();
}

cudaError_t launch_debug_philox_fold(SeedRaw seed, uint64_t first, uint64_t n, uint32_t* out,
                                     cudaStream_t s) {
    static GridCache cache;
    cudaError_t err = cudaMemsetAsync(out, 0, sizeof(uint32_t), s);
    if (err != cudaSuccess || n == 0) return err;
    int full_grid = 0;
    err = persistent_grid(debug_philox_fold_kernel, kThreads, 0, cache, &full_grid);
    if (err != cudaSuccess) return err;
    while (n > 0) {  // one launch per high word of the block index
        const uint64_t m = std::min<uint64_t>(n, (1ull << 32) - (first & 0xFFFFFFFFull));
        const uint64_t needed = (m + kThreads - 1) / kThreads;
        const int grid = needed < static_cast<uint64_t>(full_grid) ? static_cast<int>(needed) : full_grid;
        debug_philox_fold_kernel<<<grid, kThreads, 0, s>>>(
            seed_param(seed, static_cast<uint32_t>(first >> 32), 0.0f), static_cast<uint32_t>(first), m, out);
        err = cudaGetLastError();
        if (err != cudaSuccess) return err;
        first += m;
        n -= m;
    }
    return cudaSuccess;
}

cudaError_t launch_debug_gaussian(SeedRaw seed, uint64_t first, uint64_t n, float* out,
                                  cudaStream_t s) {
    if (n == 0) return cudaSuccess;
    debug_gaussian_kernel<<<blocks_for(n), 256, 0, s>>>(seed, first, n, out);
    return cudaGetLastError();
}

cudaError_t launch_debug_box_muller(const uint32_t* words, uint64_t n_pairs, float* out, cudaStream_t s) {
    if (n_pairs == 0) return cudaSuccess;
    debug_box_muller_kernel<<<blocks_for((n_pairs + 1) / 2), 256, 0, s>>>(words, n_pairs, out);
    return cudaGetLastError();
}

}  // namespace jb
