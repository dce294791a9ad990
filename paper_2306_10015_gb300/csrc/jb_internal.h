// jb_internal.h -- launch descriptors shared by the C ABI (jb_capi.cpp) and
// the kernels (jb_kernels.cu, jb_q4.cu). Not part of the public interface.
//
// A launch carries its whole work description in the kernel parameter space
// (up to 32,764 bytes on sm_70 and later): the K (seed, coefficient) pairs, read
// with warp-uniform indices from the constant bank, then the segment table. The two
// share one block of bytes, so that few pairs leave room for more segments.
//
// Work is cut into 16-byte "vectors" of one segment whose elements are aligned to
// Philox blocks in global index (4 fp32 or 8 bf16 elements), and vectors into warp
// tiles of 32 V of them. A tile lies in one segment: segment s owns tiles
// tile0 .. (tile0 of the next) - 1, and a sentinel entry after the last one holds
// the number of tiles, so a tile's segment is the last entry whose tile0 is not
// above it.
//
// All global indices of a segment agree in the high word of their Philox block index: the
// host cuts segments at multiples of 2^33 elements. A launch holds segments of one high
// word, or of two with a set of pairs for each. Block counters are therefore 32-bit in the
// kernels, and the whole first round and half of the second are constants of the pair
// (jb_rng.cuh).
#pragma once
#include <cstdint>

#include <cuda_runtime.h>

namespace jb {

constexpr int kThreads = 512;  // threads per CTA of the generator alone
constexpr int kMaxSeedsPerLaunch = 512;
constexpr int kMaxGroupsPerLaunch = 512;
constexpr uint64_t kPieceElems = 1ull << 33;  // segments are cut at multiples of this index

// Philox4x32 round multipliers and key increments (Salmon et al. 2011).
constexpr uint32_t kPhiloxM0 = 0xD2511F53u;
constexpr uint32_t kPhiloxM1 = 0xCD9E8D57u;
constexpr uint32_t kPhiloxW0 = 0x9E3779B9u;
constexpr uint32_t kPhiloxW1 = 0xBB67AE85u;

// Seed s of the method: the key and the upper half of the counter.
struct SeedRaw {
    uint32_t k0, k1;        // machine id (lo, hi)
    uint32_t step, sample;  // counter words 2 and 3
};

// A pair as the kernels read it: the words of Philox4x32-10 that do not depend on the
// low word of the block index (philox_block in jb_rng.cuh), and the scale.
struct alignas(16) SeedParam {
    uint32_t c2;       // round 1: x2 = hi(M0 b_lo) ^ c2
    uint32_t c0;       // round 2: x0 = hi(M1 x2) ^ c0
    uint32_t n2, n3;   // round 2: x2 = lo(M0 b_lo) ^ n2, x3 = n3
    uint32_t k0, k1;   // keys of round 3
    float coef;        // c_k (update) or eps (perturb)
    uint32_t ends_group;  // general update: round to the storage type after this pair
};

__host__ __device__ inline SeedParam seed_param(const SeedRaw& s, uint32_t block_hi, float coef) {
    const uint64_t a = static_cast<uint64_t>(kPhiloxM1) * s.step;
    const uint32_t x0 = static_cast<uint32_t>(a >> 32) ^ block_hi ^ s.k0;  // after round 1
    const uint64_t p = static_cast<uint64_t>(kPhiloxM0) * x0;
    SeedParam r;
    r.c2 = s.sample ^ s.k1;
    r.c0 = static_cast<uint32_t>(a) ^ (s.k0 + kPhiloxW0);
    r.n2 = static_cast<uint32_t>(p >> 32) ^ (s.k1 + kPhiloxW1);
    r.n3 = static_cast<uint32_t>(p);
    r.k0 = s.k0 + 2u * kPhiloxW0;
    r.k1 = s.k1 + 2u * kPhiloxW1;
    r.coef = coef;
    r.ends_group = 0;
    return r;
}

// A pair with the round keys of rounds 3 .. 10, which the kernels otherwise add up for
// every pair and tile.
struct KeyedParam : SeedParam {
    uint32_t key[16];
};

inline void set_pair(SeedParam& to, const SeedParam& s) { to = s; }
inline void set_pair(KeyedParam& to, const SeedParam& s) {
    static_cast<SeedParam&>(to) = s;
    for (uint32_t r = 0; r < 8; ++r) {
        to.key[2 * r] = s.k0 + r * kPhiloxW0;
        to.key[2 * r + 1] = s.k1 + r * kPhiloxW1;
    }
}

struct SegParam {
    uint64_t base;   // device address of the segment's first window (its element `head` is element 0)
    uint64_t end;    // elements of the segment are [head, end) of its windows
    uint32_t blk0;   // low word of the Philox block index of the first window (checksum: its own)
    uint32_t tile0;  // first tile
    uint8_t head;    // elements of the first window before the segment (0 .. E - 1)
    uint8_t lo;      // vectors [lo, full) are read and written whole; the others go element
    uint8_t load;    //   by element. Alignment of their addresses, 2 to 16 bytes: of the
    uint8_t store;   //   source, and of where the result goes
    uint32_t full;
};

struct SegParamOut : SegParam {
    uint64_t dst;    // destination address of the first window
};

template <typename SEG, typename PAIR, int BYTES>
struct Launch {
    using Seg = SEG;
    using Pair = PAIR;
    static constexpr int kBytes = BYTES;
    uint32_t n_seeds;
    uint32_t n_segs;
    uint32_t n_tiles;
    uint32_t span;       // consecutive tiles that a warp takes at a time
    uint32_t write_src;  // write the result to the source too; checksum: one CTA, store the sum
    uint32_t second_from;  // segments from this one on have the second high word, and use
                           // the second set of pairs (checksum: the second word of `data`)
    uint32_t seg_at;     // byte offset of the segment table in `data`; the pairs are at 0
    alignas(16) unsigned char data[BYTES];
};

constexpr int kParamBytes = 32704;
// Small launches: the parameters are copied for each launch (an empty kernel: 10.8 us
// from call to end with 32 KB of them, 9.0 us with 4 KB). Small tables off the 16-byte grid
// have no kernels of their own for that and take the large ones.
constexpr int kSmallParamBytes = 4064;
static_assert(sizeof(Launch<SegParam, SeedParam, kParamBytes>) <= 32764, "launch exceeds the parameter space");

// A checked segment: element i at ptr + i sizeof(T) has global index fo + i.
struct Seg {
    uint64_t ptr, fo, n;
};

// 4-bit weights: codes (two per byte, element 2i in the low nibble) and one fp32
// scale per 64 elements.
struct SegParamQ4 {
    uint64_t codes;   // device address, 8-byte aligned
    uint64_t scale;   // device address of the fp32 scales
    uint64_t n;
    uint32_t blk0;    // Philox block index of element 0 (its global index is a multiple of 4)
    uint32_t blk_hi;
    uint32_t tile0;   // first tile (1024 elements each)
    uint32_t wide;    // the codes are 16-byte aligned
};

template <int BYTES>
struct Q4Launch {
    static constexpr int kBytes = BYTES;
    SeedRaw seed;
    float eps;
    uint32_t n_segs;
    uint32_t n_tiles;
    uint32_t span;
    uint32_t block_hi;  // high word of the block indices where they agree in it
    alignas(16) unsigned char data[BYTES];
};
static_assert(sizeof(Q4Launch<kParamBytes>) <= 32764, "4-bit launch exceeds the parameter space");

struct Q4Seg {
    uint64_t codes, scale, fo, n;
};

cudaError_t enqueue_q4(const SeedRaw& seed, float eps, const Q4Seg* segs, size_t n_segs, cudaStream_t stream);
void q4_levels_host(float out[16]);

enum DType { kF32 = 0, kBF16 = 1 };

// What a launch runs: PerturbParameters (one pair, theta + eps z as one fused
// multiply-add), the in-place update, or the general update (source to destination,
// groups). One pair in one group takes the one-pair kernel in both updates. The checksum
// has no pairs.
enum Work { kPerturb = 0, kUpdate = 1, kGeneral = 2, kChecksum = 3 };

struct Job {
    Work work;
    int dtype;
    const SeedRaw* seeds;  // in canonical order (within each group)
    const float* coef;
    int n_seeds;
    const uint16_t* group_end;  // general update: group g is the pairs up to group_end[g]
    int n_groups;
    bool write_src;
    int grid_ctas;  // <= 0: the persistent grid
    cudaStream_t stream;
    unsigned long long* sum;  // checksum: device address of the result
};

// Packs the segments into launches of the job and enqueues them. dst: the general
// update's destinations, one per segment (n_segs > 0).
cudaError_t enqueue(const Job& job, const Seg* segs, const uint64_t* dst, size_t n_segs);

cudaError_t launch_debug_philox(SeedRaw seed, uint64_t first_block, uint64_t n_blocks,
                                uint32_t* out, cudaStream_t s);
cudaError_t launch_debug_philox_fold(SeedRaw seed, uint64_t first_block, uint64_t n_blocks,
                                     uint32_t* out, cudaStream_t s);
cudaError_t launch_debug_gaussian(SeedRaw seed, uint64_t first, uint64_t n, float* out,
                                  cudaStream_t s);
cudaError_t launch_debug_box_muller(const uint32_t* words, uint64_t n_pairs, float* out,
                                    cudaStream_t s);

}  // namespace jb
