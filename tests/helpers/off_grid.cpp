// Runs the off-grid vector accesses of jb_offgrid.h on a byte buffer whose first byte stands
// at a 16-byte boundary, and counts how often each byte of it is read and written.
#include <cstring>

#include "jb_offgrid.h"

namespace {
struct Recorded {
    unsigned char *bytes;
    int *reads, *writes;
    int* misaligned;
    template <typename V>
    V get(uint64_t a) const {
        V v;
        std::memcpy(&v, bytes + a, sizeof(V));
        for (size_t i = 0; i < sizeof(V); ++i) ++reads[a + i];
        if (a % sizeof(V) != 0) ++*misaligned;
        return v;
    }
    template <typename V>
    void put(uint64_t a, V v) const {
        std::memcpy(bytes + a, &v, sizeof(V));
        for (size_t i = 0; i < sizeof(V); ++i) ++writes[a + i];
        if (a % sizeof(V) != 0) ++*misaligned;
    }
    uint2 load64(uint64_t a) const { return get<uint2>(a); }
    uint32_t load32(uint64_t a) const { return get<uint32_t>(a); }
    uint16_t load16(uint64_t a) const { return get<uint16_t>(a); }
    void store64(uint64_t a, uint2 v) const { put(a, v); }
    void store32(uint64_t a, uint32_t v) const { put(a, v); }
    void store16(uint64_t a, uint16_t v) const { put(a, v); }
};
}  // namespace

extern "C" int off_grid_load(unsigned char* bytes, uint64_t a, uint32_t align, uint32_t* out, int* reads) {
    int misaligned = 0;
    const uint4 w = jb::load_off_grid(Recorded{bytes, reads, nullptr, &misaligned}, a, align);
    out[0] = w.x; out[1] = w.y; out[2] = w.z; out[3] = w.w;
    return misaligned;
}

extern "C" int off_grid_store(unsigned char* bytes, uint64_t a, uint32_t align, const uint32_t* in, int* writes) {
    int misaligned = 0;
    jb::store_off_grid(Recorded{bytes, nullptr, writes, &misaligned}, a, align, make_uint4(in[0], in[1], in[2], in[3]));
    return misaligned;
}
