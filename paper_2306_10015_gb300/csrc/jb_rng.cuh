// jb_rng.cuh -- the seeded N(0,1) stream, computed in registers on sm_103a.
//
// PerturbParameters (Algorithm 1, subroutine) reseeds a generator with
// s = (machine time id, iteration, sample index) and draws z ~ N(0,1) for every
// parameter. Here z of global element e is a pure function of (s, e):
//   Philox4x32-10 (Salmon, Moraes, Dror, Shaw, SC 2011) of counter
//   (lo(b), hi(b), step, sample_id), b = e >> 2, under key (lo(mid), hi(mid));
//   Box-Muller (Box & Muller 1958) on word pairs (0,1) and (2,3):
//   r = sqrt(-2 ln u_a), u_a = ((x_a >> 9) + 1/2) 2^-23; angle 2 pi u_b,
//   u_b = ((x_b >> 8) + 1/2) 2^-24; element 4b + 2p -> r cos, 4b + 2p + 1 -> r sin.
// Nothing here is written to memory on the hot path.
//
// Arithmetic of the transform (fp32, every rounding explicit):
//   radius  u_a = 2^e f exactly, f in [1/2, 1), with sigma = 2(1 - f) exact and
//           y = sigma / (2(1 + f)) (one rcp.approx):
//           -2 ln f = 4 atanh(y) = sigma + y (sigma + w P(w)), w = y^2, P a degree-3
//           minimax polynomial. The leading term is exact, so the error of the
//           reciprocal enters only through the second term (at most 0.28 of the sum);
//           u_a near 1 has e = 0 and keeps its relative accuracy.
//           L = -2 ln f - e (2 ln 2) (2 ln 2 in fp32 is within 2.8e-9, so one product
//           is enough); r = sqrt.approx(L) (relative error below 1.1e-7 over every L).
//   angle   with t = x_b + 2^29, the angle is q pi/2 + (pi/4) x, q = t >> 30, x in
//           (-1, 1) exact from the 22 bits below; sin and cos of (pi/4) x by minimax
//           polynomials of degree 7 and 8 (relative error < 0.6 ulp for the sine, also
//           near zero; 7.2e-8 for the cosine, which stays above 0.7). Odd q swaps them
//           (and negates the sine), q >= 2 flips both: that sign goes to the radius.
// Integers become floats by placing their bits under a constant exponent (one shift,
// at most one mask, and a subtraction that the packed arithmetic does for two): an
// integer-to-float conversion costs more issue slots than those. Against f in
// [3/4, 3/2) with integer conversions, and an octant reflection with both signs applied
// to the results, one pass over 1.3B bf16 elements went from 1653 to 1524 us (one pair)
// and a K = 16 update of 125M fp32 elements from 2239 to 2123 us; it is also more
// accurate: rms |dz| 4.75e-8 -> 4.69e-8, largest over 1.3e8 draws 8.0e-7 -> 7.5e-7,
// joint worst case 8.7e-7 -> 8.2e-7.
// Coefficients: fit_poly.py (Remez exchange). The transform is checked
// against a double-precision evaluation of the same definition over all
// radius words and all angle words (|dz| <= 1e-6).
#pragma once
#include <cstdint>
#include <type_traits>

#include "jb_internal.h"

namespace jb {

// Polynomials (fit_poly.py).
constexpr float kLogP0 = 0x1.5555p+0f, kLogP1 = 0x1.99d29ep-1f, kLogP2 = 0x1.1eb3a2p-1f,
                kLogP3 = 0x1.1f0578p-1f;
constexpr float kSinHi = 0x1.921fb6p-1f;   // pi/4 = hi + lo
constexpr float kSinLo = -0x1.777a5cp-26f;
constexpr float kSinS0 = -0x1.4abbbep-4f, kSinS1 = 0x1.465facp-9f, kSinS2 = -0x1.2db5cep-15f;
constexpr float kCosC0 = -0x1.3bd3ccp-2f, kCosC1 = 0x1.03c1b0p-6f, kCosC2 = -0x1.55b2b6p-12f,
                kCosC3 = 0x1.d4f7eep-19f;
constexpr float kTwoLn2 = 0x1.62e430p+0f;

// One Philox round on (x0, x1, x2, x3) with round key (k0, k1).
__device__ __forceinline__ void philox_round(uint32_t& x0, uint32_t& x1, uint32_t& x2,
                                             uint32_t& x3, uint32_t k0, uint32_t k1) {
    const uint64_t p0 = static_cast<uint64_t>(kPhiloxM0) * x0;
    const uint64_t p1 = static_cast<uint64_t>(kPhiloxM1) * x2;
    const uint32_t y0 = static_cast<uint32_t>(p1 >> 32) ^ x1 ^ k0;
    const uint32_t y2 = static_cast<uint32_t>(p0 >> 32) ^ x3 ^ k1;
    x1 = static_cast<uint32_t>(p1);
    x3 = static_cast<uint32_t>(p0);
    x0 = y0;
    x2 = y2;
}

// The seed-independent part of round 1 for the block with low word b_lo: M0 * b_lo.
// Every seed of an update shares it.
struct BlockCtr {
    uint32_t p_hi, p_lo;
};

__device__ __forceinline__ BlockCtr block_ctr(uint32_t b_lo) {
    const uint64_t p0 = static_cast<uint64_t>(kPhiloxM0) * b_lo;
    BlockCtr c;
    c.p_hi = static_cast<uint32_t>(p0 >> 32);
    c.p_lo = static_cast<uint32_t>(p0);
    return c;
}

// The same for the block that lies `delta` (a constant) further: an addition of 64 bits
// instead of a multiplication. (Past the last block of the low word the result is not
// that of the wrapped index; no element lies there.)
__device__ __forceinline__ BlockCtr block_after(const BlockCtr& c, uint32_t delta) {
    const uint64_t p = ((static_cast<uint64_t>(c.p_hi) << 32) | c.p_lo) + static_cast<uint64_t>(kPhiloxM0) * delta;
    BlockCtr r;
    r.p_hi = static_cast<uint32_t>(p >> 32);
    r.p_lo = static_cast<uint32_t>(p);
    return r;
}

// Four words of Philox4x32-10 for block c under the pair's constants. Round 1 is the
// block's product and constants of the pair; round 2 needs one product (the other one's
// factor does not depend on the block's low word, so the host forms it, seed_param);
// rounds 3 .. 10 in full: 17 wide multiplies.
template <typename S>
__device__ __forceinline__ uint4 philox_block(const S& s, const BlockCtr& c) {
    const uint64_t p1 = static_cast<uint64_t>(kPhiloxM1) * (c.p_hi ^ s.c2);
    uint32_t x0 = static_cast<uint32_t>(p1 >> 32) ^ s.c0;
    uint32_t x1 = static_cast<uint32_t>(p1);
    uint32_t x2 = c.p_lo ^ s.n2;
    uint32_t x3 = s.n3;
    uint32_t k0 = s.k0, k1 = s.k1;
#pragma unroll
    for (int r = 2; r < 10; ++r) {
        if constexpr (std::is_same<S, KeyedParam>::value) {
            k0 = s.key[2 * (r - 2)];
            k1 = s.key[2 * (r - 2) + 1];
        }
        philox_round(x0, x1, x2, x3, k0, k1);
        k0 += kPhiloxW0;
        k1 += kPhiloxW1;
    }
    return make_uint4(x0, x1, x2, x3);
}

// Four words of the block with low word b_lo.
__device__ __forceinline__ uint4 philox_block(const SeedParam& s, uint32_t b_lo) {
    return philox_block(s, block_ctr(b_lo));
}

__device__ __forceinline__ float rcp_approx(float x) {
    float y;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

__device__ __forceinline__ float sqrt_approx(float x) {
    float y;
    asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

__device__ __forceinline__ float2 splat(float a) { return make_float2(a, a); }

// Two fp32 operations in one packed instruction, each rounded once to nearest.
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
__device__ __forceinline__ float2 mul2(float2 a, float2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ float2 add2(float2 a, float2 b) { return __fadd2_rn(a, b); }

// Box-Muller of the two word pairs of a Philox block, (w.x, w.y) and (w.z, w.w), in
// lockstep: every floating-point step is one packed fp32x2 instruction (two IEEE
// round-to-nearest operations per issue slot), integer steps stay per pair.
// Polar form: rr = the radii of pair A and pair B, with the sign of the angle's half
// turn; cm, sm = cosines and sines up to that sign, so z_even = cm rr, z_odd = sm rr.
struct Polar2 {
    float2 rr, cm, sm;
};

// The word hi : lo shifted right by n, low half: one instruction that moves bits of lo
// into the mantissa and puts an exponent above them.
__device__ __forceinline__ float shift_under(uint32_t hi, uint32_t lo, int n) {
    return __uint_as_float(__funnelshift_r(lo, hi, n));
}

// (bits & keep) | set in one instruction
__device__ __forceinline__ float masked(uint32_t bits, uint32_t keep, uint32_t set) {
    uint32_t r;
    asm("lop3.b32 %0, %1, %2, %3, 0xEA;" : "=r"(r) : "r"(bits), "r"(keep), "r"(set));
    return __uint_as_float(r);
}

__device__ __forceinline__ Polar2 polar2(uint4 w) {
    // ---- radius ----
    // 1 + (x_a >> 9) 2^-23, less 1 - 2^-24: u_a, exact
    const float2 u = add2(make_float2(shift_under(0x7Fu, w.x, 9), shift_under(0x7Fu, w.z, 9)),
                          splat(-0x1.fffffep-1f));
    const uint32_t uA = __float_as_uint(u.x), uB = __float_as_uint(u.y);
    const float2 f = make_float2(masked(uA, 0x7FFFFFu, 0x3F000000u), masked(uB, 0x7FFFFFu, 0x3F000000u));
    // 2^23 + biased exponent, less 2^23 + 126: e, exact
    const float2 e = add2(make_float2(shift_under(0x4B000000u >> 9, uA, 23),
                                      shift_under(0x4B000000u >> 9, uB, 23)), splat(-8388734.0f));
    const float2 sg = fma2(f, splat(-2.0f), splat(2.0f));             // 2(1 - f), exact
    const float2 d = fma2(f, splat(2.0f), splat(2.0f));
    const float2 y = mul2(sg, make_float2(rcp_approx(d.x), rcp_approx(d.y)));  // (1 - f) / (1 + f)
    const float2 ww = mul2(y, y);
    float2 p = fma2(ww, splat(kLogP3), splat(kLogP2));
    p = fma2(ww, p, splat(kLogP1));
    p = fma2(ww, p, splat(kLogP0));
    const float2 lf = fma2(y, fma2(ww, p, sg), sg);                   // -2 ln f
    const float2 L = fma2(e, splat(-kTwoLn2), lf);                    // -2 ln u_a

    // ---- angle ----
    const uint32_t tA = w.y + 0x20000000u, tB = w.w + 0x20000000u;
    // [1, 2) from bits 29 .. 8 and a last bit for the half: 2 (.) - 3 = x, exact. The
    // bits above become the exponent's low ones.
    const float2 x = fma2(make_float2(shift_under(0x3F800000u >> 25, tA | 0xC0000080u, 7),
                                      shift_under(0x3F800000u >> 25, tB | 0xC0000080u, 7)),
                          splat(2.0f), splat(-3.0f));
    const float2 xx = mul2(x, x);
    float2 ps = fma2(xx, splat(kSinS2), splat(kSinS1));
    ps = fma2(xx, ps, splat(kSinS0));
    ps = fma2(xx, ps, splat(kSinLo));
    const float2 S = fma2(x, splat(kSinHi), mul2(x, ps));
    float2 pc = fma2(xx, splat(kCosC3), splat(kCosC2));
    pc = fma2(xx, pc, splat(kCosC1));
    pc = fma2(xx, pc, splat(kCosC0));
    const float2 C = fma2(xx, pc, splat(1.0f));
    const bool swA = (tA & 0x40000000u) != 0u, swB = (tB & 0x40000000u) != 0u;
    Polar2 o;
    o.rr = make_float2(
        __uint_as_float(__float_as_uint(sqrt_approx(L.x)) ^ (tA & 0x80000000u)),
        __uint_as_float(__float_as_uint(sqrt_approx(L.y)) ^ (tB & 0x80000000u)));
    o.cm = make_float2(swA ? -S.x : C.x, swB ? -S.y : C.y);
    o.sm = make_float2(swA ? C.x : S.x, swB ? C.y : S.y);
    return o;
}

// even = (z of word pair A's even element, pair B's even element), odd likewise.
struct GaussPair {
    float2 even, odd;
};

__device__ __forceinline__ GaussPair box_muller2(uint4 w) {
    const Polar2 o = polar2(w);
    GaussPair g;
    g.even = mul2(o.cm, o.rr);
    g.odd = mul2(o.sm, o.rr);
    return g;
}

// The four Gaussians of the block with low word b_lo, elements 4b .. 4b + 3.
__device__ __forceinline__ float4 block_gaussians(const SeedParam& s, uint32_t b_lo) {
    const GaussPair g = box_muller2(philox_block(s, b_lo));
    return make_float4(g.even.x, g.odd.x, g.even.y, g.odd.y);
}

}  // namespace jb

