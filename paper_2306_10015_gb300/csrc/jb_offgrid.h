// jb_offgrid.h -- a whole 16-byte vector at an address that is a multiple of 8, 4 or 2
// bytes only, put together from smaller accesses. The accesses go through Mem, so that
// the same code runs on the host.
//
// Every access lies inside the vector. On an odd multiple of 2 bytes the vector's two end
// elements share their words with the vectors beside it, which other threads may be writing,
// so they are read and written by themselves: five accesses each way.
#pragma once
#include <cstdint>

#include <cuda_runtime.h>

namespace jb {

template <typename Mem>
__host__ __device__ __forceinline__ uint4 load_off_grid(const Mem& mem, uint64_t a, uint32_t align) {
    if (align == 8u) {
        const uint2 p = mem.load64(a), q = mem.load64(a + 8);
        return make_uint4(p.x, p.y, q.x, q.y);
    }
    if (align == 4u) return make_uint4(mem.load32(a), mem.load32(a + 4), mem.load32(a + 8), mem.load32(a + 12));
    const uint32_t first = mem.load16(a), p = mem.load32(a + 2), q = mem.load32(a + 6), r = mem.load32(a + 10),
                   last = mem.load16(a + 14);
    return make_uint4(first | p << 16, p >> 16 | q << 16, q >> 16 | r << 16, r >> 16 | last << 16);
}

template <typename Mem>
__host__ __device__ __forceinline__ void store_off_grid(const Mem& mem, uint64_t a, uint32_t align, uint4 w) {
    if (align == 8u) {
        mem.store64(a, make_uint2(w.x, w.y));
        mem.store64(a + 8, make_uint2(w.z, w.w));
    } else if (align == 4u) {
        mem.store32(a, w.x);
        mem.store32(a + 4, w.y);
        mem.store32(a + 8, w.z);
        mem.store32(a + 12, w.w);
    } else {
        mem.store16(a, static_cast<uint16_t>(w.x));
        mem.store32(a + 2, w.x >> 16 | w.y << 16);
        mem.store32(a + 6, w.y >> 16 | w.z << 16);
        mem.store32(a + 10, w.z >> 16 | w.w << 16);
        mem.store16(a + 14, static_cast<uint16_t>(w.w >> 16));
    }
}

}  // namespace jb
