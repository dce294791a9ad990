// jb_capi.cpp -- the C ABI of libjb (declared in include/jb.h).
//
// Host side of the hot path: argument checks, the canonical (machine id,
// step, sample id) order of the pairs (Section 2: gradients are applied in
// machine-timestamp order), the per-pair coefficients c_k = -lr deq(q_k) /
// denom (Algorithm 1: minus gradient times learning rate over the number of
// gradients), the one-byte code (Section 3, Training Speed), and the packing of
// segments and pairs into kernel launches. Every element-wise step runs in the CUDA kernels.
#include <algorithm>
#include <cmath>
#include <cstring>
#include <new>
#include <vector>

#include "jb.h"
#include "jb_internal.h"

#define JB_EXPORT extern "C" __attribute__((visibility("default")))

namespace {

constexpr uint64_t kMaxIndex = 1ull << 62;  // global element indices stay below this

using jb::Seg;

size_t elem_size(int dtype) { return dtype == JB_F32 ? 4 : 2; }

// [p, p + n * es) fits in the address space (written so that n * es cannot wrap).
bool range_fits(uint64_t p, uint64_t n, uint64_t es) { return n <= (UINT64_MAX - p) / es; }

// Runs an entry point's body; a host allocation failure (or any other C++
// exception) becomes a status instead of crossing the C interface.
template <typename F>
int guarded(F&& body) noexcept {
    try {
        return body();
    } catch (const std::bad_alloc&) {
        return JB_ERR_NO_MEMORY;
    } catch (...) {
        return JB_ERR_INVALID_ARG;
    }
}

// Checks the segment table; drops empty segments. Overlap in memory or in
// global index is an argument error.
int collect_segments(const jb_segment* segs, int n_segs, int dtype, std::vector<Seg>& out) {
    if (dtype != JB_F32 && dtype != JB_BF16) return JB_ERR_UNSUPPORTED_DTYPE;
    if (n_segs < 0 || (n_segs > 0 && segs == nullptr)) return JB_ERR_INVALID_ARG;
    const uint64_t es = elem_size(dtype);
    out.clear();
    out.reserve(static_cast<size_t>(n_segs));
    for (int i = 0; i < n_segs; ++i) {
        const jb_segment& s = segs[i];
        if (s.numel == 0) continue;
        const uint64_t p = reinterpret_cast<uint64_t>(s.ptr);
        if (p == 0) return JB_ERR_INVALID_ARG;
        if (p % es != 0) return JB_ERR_MISALIGNED;
        if (s.numel > kMaxIndex || s.flat_offset > kMaxIndex - s.numel) return JB_ERR_INVALID_ARG;
        if (!range_fits(p, s.numel, es)) return JB_ERR_INVALID_ARG;
        out.push_back({p, s.flat_offset, s.numel});
    }
    // tables are mostly in order already; only then is no sorted copy needed
    const auto by_fo = [](const Seg& a, const Seg& b) { return a.fo < b.fo; };
    const auto by_ptr = [](const Seg& a, const Seg& b) { return a.ptr < b.ptr; };
    const auto fo_overlap = [](const std::vector<Seg>& v) {
        for (size_t i = 1; i < v.size(); ++i)
            if (v[i - 1].fo + v[i - 1].n > v[i].fo) return true;
        return false;
    };
    const auto ptr_overlap = [es](const std::vector<Seg>& v) {
        for (size_t i = 1; i < v.size(); ++i)
            if (v[i - 1].ptr + v[i - 1].n * es > v[i].ptr) return true;
        return false;
    };
    const bool fo_sorted = std::is_sorted(out.begin(), out.end(), by_fo);
    const bool ptr_sorted = std::is_sorted(out.begin(), out.end(), by_ptr);
    if (fo_sorted && fo_overlap(out)) return JB_ERR_INVALID_ARG;
    if (ptr_sorted && ptr_overlap(out)) return JB_ERR_INVALID_ARG;
    if (!fo_sorted || !ptr_sorted) {
        std::vector<Seg> v(out);
        if (!fo_sorted) {
            std::sort(v.begin(), v.end(), by_fo);
            if (fo_overlap(v)) return JB_ERR_INVALID_ARG;
        }
        if (!ptr_sorted) {
            std::sort(v.begin(), v.end(), by_ptr);
            if (ptr_overlap(v)) return JB_ERR_INVALID_ARG;
        }
    }
    return JB_OK;
}

jb::SeedRaw seed_raw(const jb_seed& s) {
    return {static_cast<uint32_t>(s.machine_id), static_cast<uint32_t>(s.machine_id >> 32), s.step,
            s.sample_id};
}

// A pair as it is ordered: ascending (machine id, step, sample id).
struct Pair {
    uint64_t machine;
    uint64_t step_sample;
    int index;  // in the caller's arrays
};

// Values of the byte code's magnitudes, each computed once per call.
class Dequantizer {
public:
    explicit Dequantizer(float qscale) : scale_(qscale) {}
    double operator()(int8_t q) {
        int m = q < 0 ? -static_cast<int>(q) : static_cast<int>(q);
        if (m > 127) m = 127;
        if (!known_[m]) {
            value_[m] = std::expm1(static_cast<double>(m) / scale_);
            known_[m] = true;
        }
        return q < 0 ? -value_[m] : value_[m];
    }

private:
    double scale_;
    double value_[128];
    bool known_[128] = {};
};

// Appends pairs [first, first + K) in canonical order with their coefficients c_k.
int collect_pairs(const jb_seed* seeds, const int8_t* q, size_t first, int K, float lr, float denom,
                  Dequantizer& deq, std::vector<jb::SeedRaw>& raw, std::vector<float>& coef) {
    std::vector<Pair> order(static_cast<size_t>(K));
    for (int k = 0; k < K; ++k) {
        const jb_seed& s = seeds[first + k];
        order[k] = {s.machine_id, (static_cast<uint64_t>(s.step) << 32) | s.sample_id, k};
    }
    std::sort(order.begin(), order.end(), [](const Pair& a, const Pair& b) {
        return a.machine != b.machine ? a.machine < b.machine : a.step_sample < b.step_sample;
    });
    for (int k = 1; k < K; ++k)
        if (order[k - 1].machine == order[k].machine && order[k - 1].step_sample == order[k].step_sample)
            return JB_ERR_DUPLICATE_SEED;
    for (const Pair& o : order) {
        const size_t i = first + static_cast<size_t>(o.index);
        const double c = -static_cast<double>(lr) * deq(q[i]) / static_cast<double>(denom);
        const float cf = static_cast<float>(c);
        if (!std::isfinite(cf)) return JB_ERR_RANGE;
        raw.push_back(seed_raw(seeds[i]));
        coef.push_back(cf);
    }
    return JB_OK;
}

double dequantize(int8_t q, double qscale) {
    int m = q < 0 ? -static_cast<int>(q) : static_cast<int>(q);
    if (m > 127) m = 127;
    const double v = std::expm1(static_cast<double>(m) / qscale);
    return q < 0 ? -v : v;
}

// libjb links the CUDA runtime statically: its last-error state is its own, so the
// errors of a caller's runtime (torch's, say) are neither seen nor cleared here. A
// failed call of this library's is cleared from that state (cudaGetLastError) so that
// it cannot be reported again by a later, unrelated call.
int cuda_status(cudaError_t e) {
    if (e == cudaSuccess) return JB_OK;
    (void)cudaGetLastError();
    return JB_ERR_CUDA;
}

int perturb_impl(const jb_segment* segs, int n_segs, int dtype, jb_seed seed, float eps,
                 int grid_ctas, cudaStream_t stream) {
    std::vector<Seg> v;
    int rc = collect_segments(segs, n_segs, dtype, v);
    if (rc != JB_OK) return rc;
    if (!std::isfinite(eps)) return JB_ERR_INVALID_ARG;
    if (v.empty()) return JB_OK;
    const jb::SeedRaw raw = seed_raw(seed);
    jb::Job job{jb::kPerturb, dtype, &raw, &eps, 1, nullptr, 0, false, grid_ctas, stream, nullptr};
    return cuda_status(jb::enqueue(job, v.data(), nullptr, v.size()));
}

int update_impl(const jb_segment* segs, int n_segs, int dtype, const jb_seed* seeds,
                const int8_t* q, int K, float lr, float denom, float qscale, int grid_ctas,
                cudaStream_t stream) {
    std::vector<Seg> v;
    int rc = collect_segments(segs, n_segs, dtype, v);
    if (rc != JB_OK) return rc;
    if (K < 0 || (K > 0 && (seeds == nullptr || q == nullptr))) return JB_ERR_INVALID_ARG;
    if (!std::isfinite(lr) || !std::isfinite(denom) || denom == 0.0f || !std::isfinite(qscale) ||
        !(qscale > 0.0f))
        return JB_ERR_INVALID_ARG;
    if (K > jb::kMaxSeedsPerLaunch) return JB_ERR_TOO_MANY_SEEDS;
    if (K == 0) return JB_OK;

    std::vector<jb::SeedRaw> raw;
    std::vector<float> coef;
    raw.reserve(static_cast<size_t>(K));
    coef.reserve(static_cast<size_t>(K));
    Dequantizer deq(qscale);
    rc = collect_pairs(seeds, q, 0, K, lr, denom, deq, raw, coef);
    if (rc != JB_OK) return rc;
    if (v.empty()) return JB_OK;
    jb::Job job{jb::kUpdate, dtype, raw.data(), coef.data(), K, nullptr, 0, false, grid_ctas, stream, nullptr};
    return cuda_status(jb::enqueue(job, v.data(), nullptr, v.size()));
}

// Destination table for src: same numel and flat offsets, element-aligned; each
// destination either is its source or overlaps no source and no other destination.
int collect_destinations(const jb_segment* src, const jb_segment* dst, int n_segs, int dtype,
                         std::vector<uint64_t>& dptr) {
    if (n_segs > 0 && dst == nullptr) return JB_ERR_INVALID_ARG;
    const uint64_t es = elem_size(dtype);
    struct Iv { uint64_t a, b; int owner; bool is_dst; };
    std::vector<Iv> iv;
    dptr.clear();
    for (int i = 0; i < n_segs; ++i) {
        if (src[i].numel == 0) {
            if (dst[i].numel != 0) return JB_ERR_INVALID_ARG;
            continue;
        }
        if (dst[i].numel != src[i].numel || dst[i].flat_offset != src[i].flat_offset)
            return JB_ERR_INVALID_ARG;
        const uint64_t p = reinterpret_cast<uint64_t>(dst[i].ptr);
        if (p == 0) return JB_ERR_INVALID_ARG;
        if (p % es != 0) return JB_ERR_MISALIGNED;
        if (!range_fits(p, dst[i].numel, es)) return JB_ERR_INVALID_ARG;
        dptr.push_back(p);
        const uint64_t sp = reinterpret_cast<uint64_t>(src[i].ptr);
        iv.push_back({sp, sp + src[i].numel * es, i, false});
        if (p != sp) iv.push_back({p, p + src[i].numel * es, i, true});
    }
    std::sort(iv.begin(), iv.end(), [](const Iv& x, const Iv& y) { return x.a < y.a; });
    for (size_t i = 1; i < iv.size(); ++i)
        if (iv[i - 1].b > iv[i].a) return JB_ERR_INVALID_ARG;
    return JB_OK;
}

// Shared by jb_apply_updates_from and jb_replay_updates: groups of pairs applied in
// order, each group in canonical order with its own lr and denom, one rounding to
// the storage type per group.
int general_impl(const jb_segment* segs, const jb_segment* dsts, int n_segs, int dtype,
                 const jb_seed* seeds, const int8_t* q, const int* group_sizes, int n_groups,
                 const float* lr, const float* denom, float qscale, int write_src, int grid_ctas,
                 cudaStream_t stream) {
    std::vector<Seg> v;
    int rc = collect_segments(segs, n_segs, dtype, v);
    if (rc != JB_OK) return rc;
    std::vector<uint64_t> dptr;
    const bool out_of_place = dsts != nullptr;
    if (out_of_place) {
        rc = collect_destinations(segs, dsts, n_segs, dtype, dptr);
        if (rc != JB_OK) return rc;
    } else {
        for (const Seg& g : v) dptr.push_back(g.ptr);
    }
    if (n_groups < 0 || (n_groups > 0 && (group_sizes == nullptr || lr == nullptr || denom == nullptr)))
        return JB_ERR_INVALID_ARG;
    if (!std::isfinite(qscale) || !(qscale > 0.0f)) return JB_ERR_INVALID_ARG;
    long long total = 0;
    for (int g = 0; g < n_groups; ++g) {
        if (group_sizes[g] < 0) return JB_ERR_INVALID_ARG;
        if (group_sizes[g] > jb::kMaxSeedsPerLaunch) return JB_ERR_TOO_MANY_SEEDS;
        if (!std::isfinite(lr[g]) || !std::isfinite(denom[g]) || denom[g] == 0.0f)
            return JB_ERR_INVALID_ARG;
        total += group_sizes[g];
    }
    if (total > 0 && (seeds == nullptr || q == nullptr)) return JB_ERR_INVALID_ARG;

    // every group in canonical order, with its coefficients
    std::vector<jb::SeedRaw> raw;
    std::vector<float> coef;
    raw.reserve(static_cast<size_t>(total));
    coef.reserve(static_cast<size_t>(total));
    Dequantizer deq(qscale);
    std::vector<int> sizes;
    for (int g = 0; g < n_groups; ++g) {
        const int K = group_sizes[g];
        rc = collect_pairs(seeds, q, raw.size(), K, lr[g], denom[g], deq, raw, coef);
        if (rc != JB_OK) return rc;
        if (K > 0) sizes.push_back(K);  // an empty group changes nothing
    }
    if (v.empty()) return JB_OK;
    if (sizes.empty()) {
        if (!out_of_place) return JB_OK;
        sizes.clear();  // a pure copy: one launch with no group
    }

    // groups in launches of at most kMaxSeedsPerLaunch pairs / kMaxGroupsPerLaunch groups;
    // after the first launch the destination holds the running value
    std::vector<Seg> from(v);
    std::vector<uint16_t> ends;
    size_t g0 = 0;
    long long s0 = 0;
    do {
        size_t g1 = g0;
        long long n = 0;
        ends.clear();
        while (g1 < sizes.size() && g1 - g0 < static_cast<size_t>(jb::kMaxGroupsPerLaunch) &&
               n + sizes[g1] <= jb::kMaxSeedsPerLaunch) {
            n += sizes[g1++];
            ends.push_back(static_cast<uint16_t>(n));
        }
        const bool last = g1 >= sizes.size();
        // write_src comes with one group only (jb_apply_updates_from): one launch round
        jb::Job job{jb::kGeneral, dtype, raw.data() + s0, coef.data() + s0, static_cast<int>(n),
                    ends.data(), static_cast<int>(ends.size()), write_src && last, grid_ctas, stream, nullptr};
        rc = cuda_status(jb::enqueue(job, from.data(), dptr.data(), from.size()));
        if (rc != JB_OK) return rc;
        for (size_t i = 0; i < from.size(); ++i) from[i].ptr = dptr[i];
        s0 += n;
        g0 = g1;
    } while (g0 < sizes.size());
    return JB_OK;
}

}  // namespace

JB_EXPORT int jb_apply_updates_from(const jb_segment* src, const jb_segment* dst, int n_segs,
                                    int dtype, const jb_seed* seeds, const int8_t* q, int K,
                                    float lr, float denom, float qscale, int write_src,
                                    struct CUstream_st* stream) {
    if (dst == nullptr && n_segs > 0) return JB_ERR_INVALID_ARG;
    if (K < 0) return JB_ERR_INVALID_ARG;
    return guarded([&] {
        return general_impl(src, dst, n_segs, dtype, seeds, q, &K, 1, &lr, &denom, qscale, write_src,
                            0, stream);
    });
}

JB_EXPORT int jb_replay_updates(const jb_segment* segs, int n_segs, int dtype, const jb_seed* seeds,
                                const int8_t* q, const int* step_sizes, int n_steps,
                                const float* lr, const float* denom, float qscale,
                                struct CUstream_st* stream) {
    return guarded([&] {
        return general_impl(segs, nullptr, n_segs, dtype, seeds, q, step_sizes, n_steps, lr, denom,
                            qscale, 0, 0, stream);
    });
}

JB_EXPORT int jb_perturb(const jb_segment* segs, int n_segs, int dtype, jb_seed seed, float eps,
                         struct CUstream_st* stream) {
    return guarded([&] { return perturb_impl(segs, n_segs, dtype, seed, eps, 0, stream); });
}

JB_EXPORT int jb_perturb_with_grid(const jb_segment* segs, int n_segs, int dtype, jb_seed seed,
                                   float eps, int grid_ctas, struct CUstream_st* stream) {
    return guarded([&] { return perturb_impl(segs, n_segs, dtype, seed, eps, grid_ctas, stream); });
}

JB_EXPORT int jb_apply_updates(const jb_segment* segs, int n_segs, int dtype, const jb_seed* seeds,
                               const int8_t* q, int K, float lr, float denom, float qscale,
                               struct CUstream_st* stream) {
    return guarded([&] { return update_impl(segs, n_segs, dtype, seeds, q, K, lr, denom, qscale, 0, stream); });
}

JB_EXPORT int jb_apply_updates_with_grid(const jb_segment* segs, int n_segs, int dtype,
                                         const jb_seed* seeds, const int8_t* q, int K, float lr,
                                         float denom, float qscale, int grid_ctas,
                                         struct CUstream_st* stream) {
    return guarded(
        [&] { return update_impl(segs, n_segs, dtype, seeds, q, K, lr, denom, qscale, grid_ctas, stream); });
}

namespace {
int checksum_impl(const jb_segment* segs, int n_segs, int dtype, uint64_t* d_out, int grid_ctas,
                  cudaStream_t stream) {
    std::vector<Seg> v;
    int rc = collect_segments(segs, n_segs, dtype, v);
    if (rc != JB_OK) return rc;
    if (d_out == nullptr) return JB_ERR_INVALID_ARG;
    if (reinterpret_cast<uint64_t>(d_out) & 7ull) return JB_ERR_MISALIGNED;
    if (v.empty()) return cuda_status(cudaMemsetAsync(d_out, 0, sizeof(uint64_t), stream));
    jb::Job job{jb::kChecksum, dtype, nullptr, nullptr, 0, nullptr, 0, false, grid_ctas, stream,
                reinterpret_cast<unsigned long long*>(d_out)};
    return cuda_status(jb::enqueue(job, v.data(), nullptr, v.size()));
}
}  // namespace

JB_EXPORT int jb_checksum(const jb_segment* segs, int n_segs, int dtype, uint64_t* d_out,
                          struct CUstream_st* stream) {
    return guarded([&] { return checksum_impl(segs, n_segs, dtype, d_out, 0, stream); });
}

JB_EXPORT int jb_checksum_with_grid(const jb_segment* segs, int n_segs, int dtype, uint64_t* d_out,
                                    int grid_ctas, struct CUstream_st* stream) {
    return guarded([&] { return checksum_impl(segs, n_segs, dtype, d_out, grid_ctas, stream); });
}

namespace {
int perturb_q4_impl(const jb_q4_segment* segs, int n_segs, jb_seed seed, float eps, cudaStream_t stream) {
    if (n_segs < 0 || (n_segs > 0 && segs == nullptr)) return JB_ERR_INVALID_ARG;
    if (!std::isfinite(eps)) return JB_ERR_INVALID_ARG;
    std::vector<jb::Q4Seg> v;
    struct Iv { uint64_t a, b; };
    std::vector<Iv> mem, idx;
    for (int i = 0; i < n_segs; ++i) {
        const jb_q4_segment& g = segs[i];
        if (g.numel == 0) continue;
        const uint64_t c = reinterpret_cast<uint64_t>(g.codes), sp = reinterpret_cast<uint64_t>(g.scale);
        if (c == 0 || sp == 0) return JB_ERR_INVALID_ARG;
        if ((c & 7ull) || (sp & 3ull) || (g.flat_offset & 3ull)) return JB_ERR_MISALIGNED;
        if (g.numel > kMaxIndex || g.flat_offset > kMaxIndex - g.numel) return JB_ERR_INVALID_ARG;
        const uint64_t nb = (g.numel + 1) / 2, ns = 4 * ((g.numel + 63) / 64);
        if (c > UINT64_MAX - nb || sp > UINT64_MAX - ns) return JB_ERR_INVALID_ARG;
        v.push_back({c, sp, g.flat_offset, g.numel});
        mem.push_back({c, c + nb});
        mem.push_back({sp, sp + ns});
        idx.push_back({g.flat_offset, g.flat_offset + g.numel});
    }
    for (auto* list : {&mem, &idx}) {
        const auto before = [](const Iv& x, const Iv& y) { return x.a < y.a; };
        if (!std::is_sorted(list->begin(), list->end(), before)) std::sort(list->begin(), list->end(), before);
        for (size_t i = 1; i < list->size(); ++i)
            if ((*list)[i - 1].b > (*list)[i].a) return JB_ERR_INVALID_ARG;
    }
    if (v.empty()) return JB_OK;
    return cuda_status(jb::enqueue_q4(seed_raw(seed), eps, v.data(), v.size(), stream));
}
}  // namespace

JB_EXPORT int jb_perturb_q4(const jb_q4_segment* segs, int n_segs, jb_seed seed, float eps,
                            struct CUstream_st* stream) {
    return guarded([&] { return perturb_q4_impl(segs, n_segs, seed, eps, stream); });
}

JB_EXPORT int jb_q4_levels(float* out) {
    if (out == nullptr) return JB_ERR_INVALID_ARG;
    jb::q4_levels_host(out);
    return JB_OK;
}

JB_EXPORT int jb_quantize_grad(double g, float qscale, int8_t* out) {
    if (out == nullptr || !std::isfinite(qscale) || !(qscale > 0.0f)) return JB_ERR_INVALID_ARG;
    if (std::isnan(g)) {
        *out = 0;
        return JB_OK;
    }
    double mag = std::isinf(g) ? 127.0
                               : std::round(static_cast<double>(qscale) * std::log1p(std::fabs(g)));
    if (mag > 127.0) mag = 127.0;
    const int m = static_cast<int>(mag);
    *out = static_cast<int8_t>(g < 0 ? -m : m);
    return JB_OK;
}

JB_EXPORT int jb_dequantize_grad(int8_t q, float qscale, float* out) {
    if (out == nullptr || !std::isfinite(qscale) || !(qscale > 0.0f)) return JB_ERR_INVALID_ARG;
    *out = static_cast<float>(dequantize(q, static_cast<double>(qscale)));
    return JB_OK;
}

JB_EXPORT int jb_max_seeds_per_call(void) { return jb::kMaxSeedsPerLaunch; }

JB_EXPORT const char* jb_status_string(int status) {
    switch (status) {
        case JB_OK: return "ok";
        case JB_ERR_INVALID_ARG: return "invalid argument";
        case JB_ERR_UNSUPPORTED_DTYPE: return "unsupported dtype (use JB_F32 or JB_BF16)";
        case JB_ERR_MISALIGNED: return "segment pointer not aligned to its element size";
        case JB_ERR_DUPLICATE_SEED: return "duplicate (machine_id, step, sample_id) seed";
        case JB_ERR_CUDA: return "CUDA runtime or launch error";
        case JB_ERR_RANGE: return "update coefficient not finite in fp32";
        case JB_ERR_TOO_MANY_SEEDS: return "more seeds than one call accepts";
        case JB_ERR_NO_MEMORY: return "host memory allocation failed";
        default: return "unknown status";
    }
}

JB_EXPORT int jb_debug_philox(jb_seed seed, uint64_t first_block, uint64_t n_blocks, uint32_t* d_out,
                              struct CUstream_st* stream) {
    if (n_blocks > 0 && d_out == nullptr) return JB_ERR_INVALID_ARG;
    if (n_blocks > (1ull << 38)) return JB_ERR_INVALID_ARG;
    if (reinterpret_cast<uint64_t>(d_out) & 15ull) return JB_ERR_MISALIGNED;  // one 16-byte store per block
    return cuda_status(jb::launch_debug_philox(seed_raw(seed), first_block, n_blocks, d_out,
                                               stream));
}

JB_EXPORT int jb_debug_philox_fold(jb_seed seed, uint64_t first_block, uint64_t n_blocks,
                                   uint32_t* d_out, struct CUstream_st* stream) {
    if (d_out == nullptr) return JB_ERR_INVALID_ARG;
    if (n_blocks > (1ull << 46) || first_block > (1ull << 60)) return JB_ERR_INVALID_ARG;
    if (reinterpret_cast<uint64_t>(d_out) & 3ull) return JB_ERR_MISALIGNED;
    return cuda_status(jb::launch_debug_philox_fold(seed_raw(seed), first_block, n_blocks,
                                                    d_out, stream));
}

JB_EXPORT int jb_debug_gaussian(jb_seed seed, uint64_t first_elem, uint64_t n, float* d_out,
                                struct CUstream_st* stream) {
    if (n > 0 && d_out == nullptr) return JB_ERR_INVALID_ARG;
    if (n > (1ull << 38) || first_elem > kMaxIndex - n) return JB_ERR_INVALID_ARG;
    if (reinterpret_cast<uint64_t>(d_out) & 3ull) return JB_ERR_MISALIGNED;
    return cuda_status(jb::launch_debug_gaussian(seed_raw(seed), first_elem, n, d_out, stream));
}

JB_EXPORT int jb_debug_box_muller(const uint32_t* d_words, uint64_t n_pairs, float* d_out,
                                  struct CUstream_st* stream) {
    if (n_pairs > 0 && (d_words == nullptr || d_out == nullptr)) return JB_ERR_INVALID_ARG;
    if (n_pairs > (1ull << 38)) return JB_ERR_INVALID_ARG;
    if ((reinterpret_cast<uint64_t>(d_words) | reinterpret_cast<uint64_t>(d_out)) & 3ull)
        return JB_ERR_MISALIGNED;
    return cuda_status(jb::launch_debug_box_muller(d_words, n_pairs, d_out, stream));
}
