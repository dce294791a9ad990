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
//   radius  u_a = 2^e f exactly, f in [3/4, 3/2), t = f - 1 exact; with
//           q = 4t / (2 + t) (one rcp.approx), 2 ln f = q + q w R(w), w = q^2, R a
//           degree-2 minimax polynomial; 2 ln u_a = e (2 ln 2) + 2 ln f with 2 ln 2
//           split hi + lo (Cody & Waite 1980) so that e (2 ln 2)_hi is exact;
//           r = sqrt.approx(-2 ln u_a) (that instruction's relative error is below 1.1e-7;
//           r's, over all 2^23 words, is at most 1.83e-7).
//   angle   with t = x_b + 2^29, the angle is q pi/2 + (pi/4) x, q = t >> 30, x in
//           (-1, 1) exact from the 22 bits below; sin and cos of (pi/4) x by minimax
//           polynomials of degree 7 and 8 (relative error < 0.6 ulp for the sine, also
//           near zero; 7.2e-8 for the cosine, which stays above 0.7). Odd q swaps them
//           (and negates the sine), q >= 2 flips both: that sign goes to the radius.
// Integers become floats by placing their bits under a constant exponent (one shift,
// at most one mask, and a subtraction that the packed arithmetic does for two): an
// integer-to-float conversion costs more issue slots than those. e and the scale of f come
// from the exponent of (4/3) u_a, one packed product for two radii; an integer addition for
// each costs 1.2 to 1.7 % more (one pair over 1.3B bf16 elements 1401 against 1380 us, a
// K = 16 update of 125M fp32 elements 1966 against 1932). The signs of the half turn go to
// the radius. Every rounding is that of integer conversions, an octant reflection and
// signs applied to the results, so the bits of z are too; in these kernels that form takes
// 6 to 13 % more (1509 against 1424 us for the one-pair update of 1.3B bf16 elements, 2180
// against 1934 for the fp32 update). A leading term 2(1 - f) with f in [1/2, 1) would be up
// to 2 % faster still and a little more accurate, but gives other bits: a replay rounds to
// bf16 many times, and a late joiner must end with the weights of those that trained on.
// Coefficients: fit_poly.py (Remez exchange). The transform is checked
// against a double-precision evaluation of the same definition over all
// radius words and all angle words (|dz| <= 1e-6).
#pragma once
#include <cstdint>
#include <type_traits>

#include "jb_internal.h"

namespace jb {

// Polynomials (fit_poly.py).
constexpr float kLogR0 = 0x1.5555b4p-6f, kLogR1 = 0x1.992aaap-11f, kLogR2 = 0x1.36ec6ap-15f;
constexpr float kSinHi = 0x1.921fb6p-1f;   // pi/4 = hi + lo
constexpr float kSinLo = -0x1.777a5cp-26f;
constexpr float kSinS0 = -0x1.4abbbep-4f, kSinS1 = 0x1.465facp-9f, kSinS2 = -0x1.2db5cep-15f;
constexpr float kCosC0 = -0x1.3bd3ccp-2f, kCosC1 = 0x1.03c1b0p-6f, kCosC2 = -0x1.55b2b6p-12f,
                kCosC3 = 0x1.d4f7eep-19f;
constexpr float kTwoLn2Hi = 0x1.62e4p+0f;       // 2 ln 2 to 16 bits
constexpr float kTwoLn2Lo = 0x1.7f7d1cp-19f;   // 2 ln 2 - kTwoLn2Hi


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

__device__ __forceinline__ Polar2 polar2(uint4 w) {
    // ---- radius ----
    // 1/2 + (x_a >> 9) 2^-24, less 1/2 - 2^-25: u_a / 2, exact
    const float2 u = add2(make_float2(shift_under(0x7Eu, w.x, 9), shift_under(0x7Eu, w.z, 9)),
                          splat(-0x1.fffffep-2f));
    // times 4/3 (and 2): the exponent steps where f passes 3/4; fp32's 8/3 does it at the
    // right word for all 2^23 of them
    const float2 v = mul2(u, splat(0x1.555556p+1f));
    const uint32_t hA = __float_as_uint(v.x), hB = __float_as_uint(v.y);
    // 2^23 + biased exponent, less 2^23 + 127: e, exact
    const float2 e = add2(make_float2(shift_under(0x4B000000u >> 9, hA, 23),
                                      shift_under(0x4B000000u >> 9, hB, 23)), splat(-8388735.0f));
    // the exponent's complement is that of 2^(1 - e): t = f - 1, exact
    const float2 t = fma2(u, make_float2(__uint_as_float(~hA & 0x7F800000u),
                                         __uint_as_float(~hB & 0x7F800000u)), splat(-1.0f));
    const float2 d = fma2(t, splat(0.25f), splat(0.5f));                // (2 + t) / 4
    const float2 q = mul2(t, make_float2(rcp_approx(d.x), rcp_approx(d.y)));  // 4t / (2 + t)
    const float2 ww = mul2(q, q);
    float2 p = fma2(ww, splat(kLogR2), splat(kLogR1));
    p = fma2(ww, p, splat(kLogR0));
    const float2 lp = fma2(q, mul2(ww, p), q);                          // 2 ln f
    // e (2 ln 2)_hi is exact, so L is the sum of it and the rest rounded once
    const float2 L = fma2(e, splat(kTwoLn2Hi), fma2(e, splat(kTwoLn2Lo), lp));  // 2 ln u_a

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
        __uint_as_float(__float_as_uint(sqrt_approx(-L.x)) ^ (tA & 0x80000000u)),
        __uint_as_float(__float_as_uint(sqrt_approx(-L.y)) ^ (tB & 0x80000000u)));
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

