// Device building blocks of the fused bijective shuffle (sm_103a):
//   * the VariablePhilox round (Sec. 3.2) on 32-bit registers,
//   * the tile-status protocol of single-pass decoupled look-back
//     (Merrill and Garland 2016, the scan the paper fuses in Sec. 4 / Sec. 6),
//   * the in-tile scan of keep flags (Algorithm 1's exclusive scan).
#pragma once

#include <cstdint>
#include <cuda_runtime.h>

#include "bshuffle_internal.h"

namespace bsh {
namespace dev {

// Philox multiplier M0 of Listing 1 (chosen by Salmon et al.).
constexpr uint64_t kM0 = 0xD2B74407B1CE6E93ull;
constexpr uint32_t kFull = 0xffffffffu;

// Error codes written into WsHeader::error (same values as bshuffle.h).
constexpr int kErrLookbackTimeout = -8;
constexpr int kErrDeviceBounds = -9;

// ------------------------------------------------------------------ cipher

// One VariablePhilox round on the split state (left: L bits, right: R bits).
// The 64-bit product M0 * left supplies F (its high word, XORed with the
// round key and the right half into the new left half, L' = F_k(L) xor R)
// and the bijection B (its low word).  For odd k, G shifts B up one bit and
// moves the top bit b of the old right half (bit L) in underneath, so the new
// right half carries L + 1 bits.
// The right half is never masked between rounds: the next round reads only
// its low L bits (masked into the new left half) and, for odd k, exactly its
// bit L (the funnel shift below), so bits above its width are don't-care.
// The caller masks it once after the last round.
// odd_mul = 2^(31 - L) arrives as a run-time value, so the product
// right * odd_mul (which puts bit L at bit 31) stays a multiply on the FMA
// pipe instead of a shift on the busier ALU pipe (measured: odd-k rounds 17 %
// faster on GB300).
template <bool ODD>
__device__ __forceinline__ void cipher_round(uint32_t &left, uint32_t &right, uint32_t key, uint32_t odd_mul,
                                             uint32_t lmask)
{
    const uint64_t prod = kM0 * static_cast<uint64_t>(left);
    const uint32_t hi = static_cast<uint32_t>(prod >> 32);
    const uint32_t lo = static_cast<uint32_t>(prod);
    const uint32_t new_left = (hi ^ key ^ right) & lmask;
    // odd k: (lo << 1) | bit L of right
    right = ODD ? __funnelshift_l(right * odd_mul, lo, 1u) : lo;
    left = new_left;
}

// The round count of Sec. 3.2 and the library's default.  cipher_items and
// cipher_inverse_items run exactly this many rounds fully unrolled (no loop
// control, keys[r] at fixed offsets: 12 % faster index generation on GB300)
// and any other count in a loop.
constexpr uint32_t kUnrolledRounds = 24;

// ITEMS independent evaluations, rounds outer so that the ITEMS dependency
// chains interleave and each round key is loaded once per thread.
template <bool ODD, int ITEMS>
__device__ __forceinline__ void cipher_items_loop(uint32_t (&left)[ITEMS], uint32_t (&right)[ITEMS],
                                                  const uint32_t *keys, uint32_t rounds, const Geometry &g)
{
    const uint32_t odd_mul = g.odd_mul, lmask = g.lmask, rmask = g.rmask;
    for (uint32_t r = 0; r < rounds; ++r) {
        const uint32_t key = keys[r];
#pragma unroll
        for (int j = 0; j < ITEMS; ++j) cipher_round<ODD>(left[j], right[j], key, odd_mul, lmask);
    }
#pragma unroll
    for (int j = 0; j < ITEMS; ++j) right[j] &= rmask;
}

// The same with the round count fixed at compile time (fully unrolled; keys
// in kernel parameter space become constant-bank operands).
template <bool ODD, int ITEMS, int ROUNDS>
__device__ __forceinline__ void cipher_items_fixed(uint32_t (&left)[ITEMS], uint32_t (&right)[ITEMS],
                                                   const uint32_t *keys, const Geometry &g)
{
    const uint32_t odd_mul = g.odd_mul, lmask = g.lmask, rmask = g.rmask;
#pragma unroll
    for (int r = 0; r < ROUNDS; ++r) {
#pragma unroll
        for (int j = 0; j < ITEMS; ++j) cipher_round<ODD>(left[j], right[j], keys[r], odd_mul, lmask);
    }
#pragma unroll
    for (int j = 0; j < ITEMS; ++j) right[j] &= rmask;
}

// ---- domains up to 2^21: the round's products in single precision
//
// The integer round is bound by the FMA-heavy pipe, where a 32 x 32 -> 64-bit
// product takes four issue cycles of a warp and a 32-bit one two (6 cycles of
// every even-k round, 8 of an odd one), while a single-precision FMA takes
// one.  A left half of at most kFloatMaxL = 10 bits is exact in a float, so
// the left half is kept as X = 2^23 + left (its integer value is the low bits
// of the float's pattern; the OR with the exponent rides in the LOP3 that
// masks it anyway), and one FMA rounded towards minus infinity gives
//   the low word   2^23 + 659 left            (659 = M0 mod 2^10), and
//   the high word  2^23 + floor(left * 7.694...), since the high word's low
//                  L bits are floor(left * (M0 mod 2^42) / 2^32) mod 2^L and
//                  M0 mod 2^42 = 7.694... * 2^32 (24 significant bits of it
//                  give the same floor for every left < 2^10: checked for all
//                  of them, and L = 11 fails).
// Bits above L are don't-care as in the integer round.  For odd k the odd bit
// (bit L of the right half, bit L - 1 of the last low word) comes from a third
// FMA, floor(left * (M0 mod 2^L) / 2^(L-1)), bit 0, and one LOP3.
// Two items share an FMA instruction (f32x2), which halves their issue slots.
// What is left is bound by the ALU pipe (two LOP3 per even round, three per
// odd one).  Measured on GB300, 2^28 evaluations, 8 items per thread: even k
// 1.18 -> 0.80 ms, odd k 1.53 -> 1.27 ms.
constexpr uint32_t kFloatBase = 0x4B000000u;  // the pattern of 2^23
constexpr float kTwo23 = 8388608.0f;
constexpr uint32_t kM0Lo = static_cast<uint32_t>(kM0);
constexpr uint32_t kM0Hi = static_cast<uint32_t>(kM0 >> 32);
constexpr float kFloatLo = static_cast<float>(kM0Lo & ((1u << kFloatMaxL) - 1u));
constexpr float kFloatHi =
    static_cast<float>(kM0Hi & ((1u << kFloatMaxL) - 1u)) + static_cast<float>(kM0Lo >> 11) / 2097152.0f;
static_assert((kM0Hi & ((1u << kFloatMaxL) - 1u)) == 7u, "the high word's multiplier keeps 21 fraction bits");

// d[j] = floor(x[j] * mul + add) for floats kept as patterns, two per instruction.
template <int ITEMS>
__device__ __forceinline__ void floor_fma_items(uint32_t (&d)[ITEMS], const uint32_t (&x)[ITEMS], float mul, float add)
{
    const uint32_t m = __float_as_uint(mul), c = __float_as_uint(add);
#pragma unroll
    for (int j = 0; j + 1 < ITEMS; j += 2)
        asm("{\n\t.reg .b64 x, m, c;\n\t"
            "mov.b64 x, {%2, %3};\n\tmov.b64 m, {%4, %4};\n\tmov.b64 c, {%5, %5};\n\t"
            "fma.rm.f32x2 x, x, m, c;\n\t"
            "mov.b64 {%0, %1}, x;\n\t}"
            : "=r"(d[j]), "=r"(d[j + 1])
            : "r"(x[j]), "r"(x[j + 1]), "r"(m), "r"(c));
    if constexpr (ITEMS % 2 != 0)
        d[ITEMS - 1] = __float_as_uint(__fmaf_rd(__uint_as_float(x[ITEMS - 1]), mul, add));
}

// Left halves of 11 and 12 bits (domains of 2^22 to 2^25): the high word's
// multiplier (M0 mod 2^(32 + L)) / 2^32 = 1031.694... needs more than a
// float's 24 bits, so its integer part stays an integer multiply-add,
// left * 1030 + floor(left * 1.694...), whose addend is one FMA (24 bits of
// 1.694... give the same floor for every left < 2^12, and L = 13 fails; the
// FMA's addend takes off the low L bits of 2^23 * 1.694..., so that the
// pattern adds nothing below bit L).  The low word's multiplier is taken
// modulo 2^12 in its smallest form, -365.  No 64-bit product is left: four
// issue cycles of the FMA-heavy pipe per even round instead of six.  Measured
// on GB300, 2^28 evaluations: even k 1.18 -> 1.00 ms, odd k 1.53 -> 1.39 ms.
constexpr float kTwo22 = 4194304.0f;
constexpr uint32_t kMixedHi = (kM0Hi & ((1u << kMixedMaxL) - 1u)) - 1u;
constexpr float kMixedFrac = 1.0f + static_cast<float>(kM0Lo >> 9) / kTwo23;
constexpr uint32_t kMixedFracInt = (1u << 23) + (kM0Lo >> 9);  // 2^23 kMixedFrac
constexpr float kMixedLo = -365.0f;
static_assert(((kM0Lo + 365u) & ((1u << kMixedMaxL) - 1u)) == 0u, "-365 is M0 modulo 2^12");

// WIDE_HI: the left half has 11 or 12 bits (else at most 10).
template <bool ODD, bool WIDE_HI, int ITEMS, int ROUNDS>
__device__ __forceinline__ void cipher_items_float(uint32_t (&left)[ITEMS], uint32_t (&right)[ITEMS],
                                                   const uint32_t *keys, const Geometry &g)
{
    const uint32_t lmask = g.lmask;
    // odd k: G shifts the low word up one bit
    constexpr float lo_mul = (ODD ? 2.0f : 1.0f) * (WIDE_HI ? kMixedLo : kFloatLo);
    constexpr float lo_add = kTwo23 * (1.0f - lo_mul) + (WIDE_HI ? kTwo22 : 0.0f);
    const float frac_add = WIDE_HI ? -__uint2float_rn(kMixedFracInt & lmask) : 0.0f;
    // (M0 mod 2^L) / 2^(L-1), an exact float below 2
    const float odd_mul = __uint2float_rn(kM0Lo & lmask) * __uint_as_float((128u - g.L) << 23);
    const float odd_add = kTwo23 * (1.0f - odd_mul);
    uint32_t odd[ITEMS];  // bit 0: the bit that G moves underneath the next low word
#pragma unroll
    for (int j = 0; j < ITEMS; ++j) {
        left[j] |= kFloatBase;
        odd[j] = right[j] >> g.L;
    }
#pragma unroll
    for (int r = 0; r < ROUNDS; ++r) {
        const uint32_t key = keys[r];
        uint32_t hi[ITEMS], lo[ITEMS], next_odd[ITEMS];
        if constexpr (WIDE_HI) {
            floor_fma_items(hi, left, kMixedFrac, frac_add);
#pragma unroll
            for (int j = 0; j < ITEMS; ++j) hi[j] += left[j] * kMixedHi;
        } else {
            floor_fma_items(hi, left, kFloatHi, kTwo23 * (1.0f - kFloatHi));
        }
        floor_fma_items(lo, left, lo_mul, lo_add);
        if constexpr (ODD) floor_fma_items(next_odd, left, odd_mul, odd_add);
#pragma unroll
        for (int j = 0; j < ITEMS; ++j) {
            const uint32_t f = hi[j] ^ key ^ right[j];
            right[j] = ODD ? lo[j] ^ (odd[j] & 1u) : lo[j];
            if constexpr (ODD) odd[j] = next_odd[j];
            left[j] = (f & lmask) | kFloatBase;
        }
    }
#pragma unroll
    for (int j = 0; j < ITEMS; ++j) {
        left[j] &= lmask;
        right[j] &= g.rmask;
    }
}

// FORM: the form that the default round count takes (cipher_form of the left
// half's width), or Any to choose it here.  Kernels that are mostly cipher are
// instantiated per form, so that one form's registers do not set the others'
// occupancy (the staged inverse's pass 1 lost 1-2 % with all of them inside).
template <bool ODD, int ITEMS, CipherForm FORM = CipherForm::Any>
__device__ __forceinline__ void cipher_items(uint32_t (&left)[ITEMS], uint32_t (&right)[ITEMS],
                                             const uint32_t *keys, uint32_t rounds, const Geometry &g)
{
    if (rounds == kUnrolledRounds) {
        if (FORM == CipherForm::Float || (FORM == CipherForm::Any && g.L <= kFloatMaxL))
            cipher_items_float<ODD, false, ITEMS, kUnrolledRounds>(left, right, keys, g);
        else if (FORM == CipherForm::Mixed || (FORM == CipherForm::Any && g.L <= kMixedMaxL))
            cipher_items_float<ODD, true, ITEMS, kUnrolledRounds>(left, right, keys, g);
        else
            cipher_items_fixed<ODD, ITEMS, kUnrolledRounds>(left, right, keys, g);
    } else {
        cipher_items_loop<ODD, ITEMS>(left, right, keys, rounds, g);
    }
}

// i_j = first + j * STRIDE, split into halves.
template <int ITEMS, uint32_t STRIDE>
__device__ __forceinline__ void split_items(uint32_t (&left)[ITEMS], uint32_t (&right)[ITEMS], uint32_t first,
                                            const Geometry &g)
{
#pragma unroll
    for (int j = 0; j < ITEMS; ++j) {
        const uint32_t i = first + static_cast<uint32_t>(j) * STRIDE;
        left[j] = i >> g.R;
        right[j] = i & g.rmask;
    }
}

// The first round of the items i_j = first + j * STRIDE, in groups whose
// indices agree from bit L up.  A round's products depend on the left half
// alone, i >> R, which such a group shares (and so does the odd bit, bit L of
// i): they are formed once a group, and per item the new left half is left.
template <bool ODD, int ITEMS, uint32_t STRIDE, int GROUP>
__device__ __forceinline__ void shared_first_round(uint32_t (&left)[ITEMS], uint32_t (&right)[ITEMS], uint32_t first,
                                                   uint32_t key, const Geometry &g)
{
    static_assert(ITEMS % GROUP == 0, "whole groups");
#pragma unroll
    for (int q = 0; q < ITEMS; q += GROUP) {
        const uint32_t a = first + static_cast<uint32_t>(q) * STRIDE;
        uint32_t x = a >> g.R, y = a;
        // x: (high word ^ key ^ a) mod 2^L; y: the shared right half
        cipher_round<ODD>(x, y, key, g.odd_mul, g.lmask);
        x ^= a;
#pragma unroll
        for (int j = q; j < q + GROUP; ++j) {
            left[j] = (x ^ (first + static_cast<uint32_t>(j) * STRIDE)) & g.lmask;
            right[j] = y;
        }
    }
}

// cipher_items over the indices first + j * STRIDE, the first round shared
// where the left half has at least log2(GROUP * STRIDE) bits (cipher_run_form).  `first` is a
// multiple of GROUP * STRIDE plus a number below STRIDE, so that every group
// then agrees from bit L up.  Narrower left halves take the float form; the
// choice lies around all the rounds, since copies of the shared right half at
// a join after the first one cost what it saves.  Measured on GB300, without
// and with: 10,000 permutation samples of 100,000 (8 items) 3.87 -> 3.70 ms,
// indices at 2^23 + 1 (4 items) 92 -> 88 us, at 2^26 + 1 969 -> 949.
template <bool ODD, int ITEMS, uint32_t STRIDE, int GROUP = ITEMS, CipherForm FORM = CipherForm::Any>
__device__ __forceinline__ void cipher_run(uint32_t (&left)[ITEMS], uint32_t (&right)[ITEMS], uint32_t first,
                                           const uint32_t *keys, uint32_t rounds, const Geometry &g)
{
    constexpr uint32_t SPAN = GROUP * STRIDE;
    static_assert((SPAN & (SPAN - 1u)) == 0u && SPAN <= (1u << kFloatMaxL), "a power of two, of the float form");
    constexpr int REST = kUnrolledRounds - 1;
    if (rounds != kUnrolledRounds) {
        split_items<ITEMS, STRIDE>(left, right, first, g);
        cipher_items_loop<ODD, ITEMS>(left, right, keys, rounds, g);
    } else if (FORM == CipherForm::Short || (FORM == CipherForm::Any && g.lmask < SPAN - 1u)) {
        split_items<ITEMS, STRIDE>(left, right, first, g);
        cipher_items_float<ODD, false, ITEMS, kUnrolledRounds>(left, right, keys, g);
    } else if (FORM == CipherForm::Float || (FORM == CipherForm::Any && g.L <= kFloatMaxL)) {
        shared_first_round<ODD, ITEMS, STRIDE, GROUP>(left, right, first, keys[0], g);
        cipher_items_float<ODD, false, ITEMS, REST>(left, right, keys + 1, g);
    } else if (FORM == CipherForm::Mixed || (FORM == CipherForm::Any && g.L <= kMixedMaxL)) {
        shared_first_round<ODD, ITEMS, STRIDE, GROUP>(left, right, first, keys[0], g);
        cipher_items_float<ODD, true, ITEMS, REST>(left, right, keys + 1, g);
    } else {
        shared_first_round<ODD, ITEMS, STRIDE, GROUP>(left, right, first, keys[0], g);
        cipher_items_fixed<ODD, ITEMS, REST>(left, right, keys + 1, g);
    }
}

// The same for one form's launches over wider strides, any `first`: threads
// whose items agree from bit L up share the first round, the others do not.
template <bool ODD, int ITEMS, uint32_t STRIDE, CipherForm FORM>
__device__ __forceinline__ void cipher_run_wide(uint32_t (&left)[ITEMS], uint32_t (&right)[ITEMS], uint32_t first,
                                                const uint32_t *keys, uint32_t rounds, const Geometry &g)
{
    constexpr int REST = kUnrolledRounds - 1;
    const uint32_t last = first + static_cast<uint32_t>(ITEMS - 1) * STRIDE;
    if (rounds == kUnrolledRounds) {
        if (((first ^ last) >> g.L) == 0u) {
            shared_first_round<ODD, ITEMS, STRIDE, ITEMS>(left, right, first, keys[0], g);
        } else {
            split_items<ITEMS, STRIDE>(left, right, first, g);
#pragma unroll
            for (int j = 0; j < ITEMS; ++j) cipher_round<ODD>(left[j], right[j], keys[0], g.odd_mul, g.lmask);
        }
        if (FORM == CipherForm::Float || (FORM == CipherForm::Any && g.L <= kFloatMaxL))
            cipher_items_float<ODD, false, ITEMS, REST>(left, right, keys + 1, g);
        else if (FORM == CipherForm::Mixed || (FORM == CipherForm::Any && g.L <= kMixedMaxL))
            cipher_items_float<ODD, true, ITEMS, REST>(left, right, keys + 1, g);
        else
            cipher_items_fixed<ODD, ITEMS, REST>(left, right, keys + 1, g);
    } else {
        split_items<ITEMS, STRIDE>(left, right, first, g);
        cipher_items_loop<ODD, ITEMS>(left, right, keys, rounds, g);
    }
}

// Inverse of M0 modulo 2^64 (Newton's iteration; M0 is odd).
constexpr uint64_t inverse_mod_2_64(uint64_t a)
{
    uint64_t x = a;  // correct to 3 bits: a * a = 1 mod 8 for odd a
    for (int i = 0; i < 5; ++i) x *= 2 - a * x;
    return x;
}
constexpr uint32_t kM0InvLo = static_cast<uint32_t>(inverse_mod_2_64(kM0));
static_assert(static_cast<uint32_t>(kM0) * kM0InvLo == 1u, "M0 inverse");

// One inverse round, following the inversion steps of Sec. 3.2: recover
// (B_k(L), b) from the new right half (G^-1: for odd k the odd bit b sits at
// the bottom and B_k(L) above it), L = B_k^-1(B_k(L)) by multiplying with
// M0^-1 modulo 2^L, and R = F_k(L) xor L' from the recomputed high product
// word.  The left half must be exact; the right half may carry don't-care
// bits above its width (only its low L + 1 bits are read, and the product
// with M0^-1 is masked to L bits), so it is masked once after the last round.
// For odd k the round moves b to bit L with a multiply by lift_mul = 2^L, a
// run-time value, so that it runs on the FMA pipe: with a shift, the ALU pipe
// bound odd-k inverse rounds (measured on GB300: 2.22 -> 1.87 ms per 2^28
// evaluations at k = 29).
template <bool ODD>
__device__ __forceinline__ void cipher_inverse_round(uint32_t &left, uint32_t &right, uint32_t key,
                                                     uint32_t lift_mul, uint32_t lmask)
{
    const uint32_t bl = ODD ? (right >> 1) : right;
    const uint32_t old_left = (bl * kM0InvLo) & lmask;
    const uint32_t hi = __umulhi(static_cast<uint32_t>(kM0), old_left) + static_cast<uint32_t>(kM0 >> 32) * old_left;
    const uint32_t x = left ^ hi ^ key;
    // odd k: R in the low L bits and b (bit 0 of the old right half) at bit L
    right = ODD ? ((x & lmask) | ((right * lift_mul) & ~lmask)) : x;
    left = old_left;
}

// ITEMS independent inverse evaluations, rounds in reverse key order.
template <bool ODD, int ITEMS>
__device__ __forceinline__ void cipher_inverse_items_loop(uint32_t (&left)[ITEMS], uint32_t (&right)[ITEMS],
                                                          const uint32_t *keys, uint32_t rounds, const Geometry &g)
{
    const uint32_t lift_mul = g.lift_mul, lmask = g.lmask;
    for (uint32_t r = rounds; r-- > 0;) {
        const uint32_t key = keys[r];
#pragma unroll
        for (int j = 0; j < ITEMS; ++j) cipher_inverse_round<ODD>(left[j], right[j], key, lift_mul, lmask);
    }
#pragma unroll
    for (int j = 0; j < ITEMS; ++j) right[j] &= g.rmask;
}

// Default rounds: the high product word without its 32 x 32 -> 64-bit
// product (four of the even round's eight issue cycles on the FMA-heavy pipe,
// of the odd one's ten).  As in cipher_items_float the left half is kept as
// X = 2^23 + left, and the high
// word's low L bits are left * (M0hi - 1) + floor(left * 1.694...), now for
// every L up to 16: the multiplier (2^32 + M0lo) / 2^32 is split into 217 / 128
// (2^23 of it is a multiple of 2^16, so that the pattern adds nothing below bit
// L) and a negative rest of 22 bits, so both FMAs, rounded down, give the exact
// floor (the first one's value is rounded to a grid that holds the multiples of
// 2^-7 at which the second one's floor steps).  The forward round gains nothing
// from this (its product gives the low word too).  MIXED: at most 12 bits, one
// FMA.  Measured on GB300, 2^28 evaluations at k = 28: 1.35 -> 1.15 ms; the
// shuffle of 2^27 4-byte elements (odd k) 1.80 -> 1.71 ms, of 2^27 - 5 8-byte
// ones 2.38 -> 2.32.
constexpr float kFracTop = 217.0f / 128.0f;
constexpr float kFracRest = -(static_cast<float>(0xB2000000u - kM0Lo) / 4294967296.0f);
static_assert(0xB2000000u - kM0Lo < (1u << 22), "the rest of the multiplier is exact in a float");

// d[j] = floor(x[j] * mul + d[j]) for floats kept as patterns.
template <int ITEMS>
__device__ __forceinline__ void floor_fma_onto_items(uint32_t (&d)[ITEMS], const uint32_t (&x)[ITEMS], float mul)
{
    static_assert(ITEMS % 2 == 0, "two items an instruction");
    const uint32_t m = __float_as_uint(mul);
#pragma unroll
    for (int j = 0; j < ITEMS; j += 2)
        asm("{\n\t.reg .b64 x, m, c;\n\t"
            "mov.b64 x, {%2, %3};\n\tmov.b64 m, {%4, %4};\n\tmov.b64 c, {%0, %1};\n\t"
            "fma.rm.f32x2 x, x, m, c;\n\t"
            "mov.b64 {%0, %1}, x;\n\t}"
            : "+r"(d[j]), "+r"(d[j + 1])
            : "r"(x[j]), "r"(x[j + 1]), "r"(m));
}

template <bool ODD, bool MIXED, int ITEMS, int ROUNDS>
__device__ __forceinline__ void cipher_inverse_items_float(uint32_t (&left)[ITEMS], uint32_t (&right)[ITEMS],
                                                           const uint32_t *keys, const Geometry &g)
{
    const uint32_t lmask = g.lmask;
    const float frac_add = MIXED ? -__uint2float_rn(kMixedFracInt & lmask) : 0.0f;
#pragma unroll
    for (int r = ROUNDS - 1; r >= 0; --r) {
        const uint32_t key = keys[r];
        uint32_t old_left[ITEMS], hi[ITEMS];
#pragma unroll
        for (int j = 0; j < ITEMS; ++j)
            old_left[j] = (((ODD ? right[j] >> 1 : right[j]) * kM0InvLo) & lmask) | kFloatBase;
        if constexpr (MIXED) {
            floor_fma_items(hi, old_left, kMixedFrac, frac_add);
        } else {
            floor_fma_items(hi, old_left, kFracRest, -kTwo23 * kFracRest);
            floor_fma_onto_items(hi, old_left, kFracTop);
        }
#pragma unroll
        for (int j = 0; j < ITEMS; ++j) {
            const uint32_t x = left[j] ^ (old_left[j] * (kM0Hi - 1u) + hi[j]) ^ key;  // don't-care above bit L
            right[j] = ODD ? ((x & lmask) | ((right[j] * g.lift_mul) & ~lmask)) : x;
            left[j] = old_left[j];
        }
    }
#pragma unroll
    for (int j = 0; j < ITEMS; ++j) {
        left[j] &= lmask;
        right[j] &= g.rmask;
    }
}

// FORM as for cipher_items: Wide, or Mixed for left halves of at most 12 bits.
template <bool ODD, int ITEMS, CipherForm FORM = CipherForm::Wide>
__device__ __forceinline__ void cipher_inverse_items(uint32_t (&left)[ITEMS], uint32_t (&right)[ITEMS],
                                                     const uint32_t *keys, uint32_t rounds, const Geometry &g)
{
    if (rounds == kUnrolledRounds) {
        cipher_inverse_items_float<ODD, FORM == CipherForm::Mixed, ITEMS, kUnrolledRounds>(left, right, keys, g);
    } else
        cipher_inverse_items_loop<ODD, ITEMS>(left, right, keys, rounds, g);
}

// ------------------------------------------------------------------ memory helpers

__device__ __forceinline__ uint64_t ld_relaxed_gpu(const uint64_t *p)
{
    uint64_t v;
    asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
    return v;
}

__device__ __forceinline__ uint32_t ld_relaxed_gpu(const uint32_t *p)
{
    uint32_t v;
    asm volatile("ld.relaxed.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}

__device__ __forceinline__ void st_relaxed_gpu(uint64_t *p, uint64_t v)
{
    asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(p), "l"(v) : "memory");
}

__device__ __forceinline__ uint64_t global_ns()
{
    uint64_t t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

__device__ __forceinline__ uint32_t lanemask_lt()
{
    uint32_t m;
    asm("mov.u32 %0, %%lanemask_lt;" : "=r"(m));
    return m;
}

// Look-back clocks (a measurement build, off by default): with
// BSHUFFLE_LOOKBACK_CLOCKS=1 the single-pass kernels add the SM clock cycles
// their tiles wait on the look-back, and the cycles their CTAs run, to the
// workspace header, so that the share of time lost to the inter-tile chain
// is measured directly.  Otherwise these helpers compile to nothing.
#ifndef BSHUFFLE_LOOKBACK_CLOCKS
#define BSHUFFLE_LOOKBACK_CLOCKS 0
#endif
constexpr bool kLookbackClocks = BSHUFFLE_LOOKBACK_CLOCKS != 0;

__device__ __forceinline__ long long clock_mark()
{
    if constexpr (kLookbackClocks) return clock64();
    return 0;
}

__device__ __forceinline__ void clock_add(unsigned long long *acc, long long since)
{
    if constexpr (kLookbackClocks) atomicAdd(acc, static_cast<unsigned long long>(clock64() - since));
}

__device__ __forceinline__ void record_error(WsHeader *ws, int code, uint64_t info)
{
    if (atomicCAS(&ws->error, 0, code) == 0)
        atomicExch(reinterpret_cast<unsigned long long *>(&ws->error_info),
                   static_cast<unsigned long long>(info));
}

// ------------------------------------------------------------------ tile status

// A tile-status word: tag (31 bits) | inclusive flag (1 bit) | value (32 bits).
// The tag identifies the launch; a word with another tag reads as "not yet
// published".  value is the tile's aggregate (flag 0) or its inclusive
// prefix (flag 1).
__device__ __forceinline__ uint64_t status_word(uint32_t tag, bool inclusive, uint32_t value)
{
    return (static_cast<uint64_t>(tag) << 33) | (static_cast<uint64_t>(inclusive) << 32) | value;
}

__device__ __forceinline__ uint32_t next_tag(uint32_t tag)
{
    return tag >= 0x7fffffffu ? 1u : tag + 1u;
}

// Round key r of a seed: the low 32 bits of the (r + 1)-th SplitMix64 output
// started from the seed (Steele, Lea, Flood 2014), computed directly from r
// so that every lane can derive its own key.
__device__ __forceinline__ uint32_t splitmix_key(uint64_t seed, uint32_t r)
{
    uint64_t z = seed + 0x9E3779B97F4A7C15ull * (static_cast<uint64_t>(r) + 1ull);
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    return static_cast<uint32_t>(z ^ (z >> 31));
}

__device__ __forceinline__ uint64_t warp_inclusive_scan64(uint64_t v)
{
    const uint32_t lane = threadIdx.x & 31u;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const uint64_t u = __shfl_up_sync(kFull, v, d);
        if (lane >= static_cast<uint32_t>(d)) v += u;
    }
    return v;
}

__device__ __forceinline__ uint32_t warp_inclusive_scan(uint32_t v)
{
    const uint32_t lane = threadIdx.x & 31u;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const uint32_t u = __shfl_up_sync(kFull, v, d);
        if (lane >= static_cast<uint32_t>(d)) v += u;
    }
    return v;
}

// Where the tile-status words of a launch live and how they are tagged.
// Tile q's word is words[q & mask] and carries tag base_tag + (q >> shift).
// A plain launch uses one word per tile (mask = all ones, shift = 63) and the
// launch tag; the persistent batched launch reuses a ring of 2^shift words and
// tags each pass over the ring with its generation, counted on from the
// launches before it on the stream, so that neither a word left by tile
// q - 2^shift nor one of an earlier launch ever reads as tile q's.
struct StatusRing {
    uint64_t *words;
    uint64_t mask;
    uint32_t shift;
    uint32_t base_tag;
    __device__ __forceinline__ uint64_t *slot(uint64_t q) const { return words + (q & mask); }
    __device__ __forceinline__ uint32_t tag(uint64_t q) const
    {
        return base_tag + static_cast<uint32_t>(q >> shift);
    }
};

// Decoupled look-back by one warp: the exclusive prefix of tile `tile` over
// the tiles first .. tile-1.  Each pass reads the 32 nearest predecessors,
// waits until all of them are published, sums back to the nearest inclusive
// prefix and stops there, else adds all 32 aggregates and moves on.  A wait
// is bounded: after timeout_ns without progress `ok` is cleared and the
// partial sum is returned.
__device__ __forceinline__ uint32_t lookback(const StatusRing &ring, uint64_t tile, uint64_t first,
                                             uint64_t timeout_ns, bool &ok)
{
    const uint32_t lane = threadIdx.x & 31u;
    uint32_t exclusive = 0;
    int64_t pred = static_cast<int64_t>(tile) - 1;
    uint64_t wait_start = 0;
    bool waiting = false;
    uint32_t backoff = 0;
    uint32_t spins = 0;
    ok = true;
    while (true) {
        const int64_t idx = pred - static_cast<int64_t>(lane);
        bool ready = true;
        uint64_t s = status_word(0u, true, 0u);  // before the first tile: prefix 0
        if (idx >= static_cast<int64_t>(first)) {
            const uint64_t q = static_cast<uint64_t>(idx);
            s = ld_relaxed_gpu(ring.slot(q));
            ready = static_cast<uint32_t>(s >> 33) == ring.tag(q);
        }
        if (__all_sync(kFull, ready)) {
            const uint32_t incl = __ballot_sync(kFull, static_cast<uint32_t>(s >> 32) & 1u);
            uint32_t v = static_cast<uint32_t>(s);
            if (incl != 0u && static_cast<int>(lane) > __ffs(incl) - 1) v = 0u;
            exclusive += __reduce_add_sync(kFull, v);
            if (incl != 0u) break;
            pred -= 32;
            waiting = false;
            backoff = 0;
            continue;
        }
        uint64_t now = 0;
        if (lane == 0) now = global_ns();
        now = __shfl_sync(kFull, now, 0);
        if (!waiting) {
            waiting = true;
            wait_start = now;
        } else if (now - wait_start > timeout_ns || ++spins > (1u << 26)) {
            ok = false;
            break;
        }
        __nanosleep(32u << (backoff < 5u ? backoff : 5u));
        ++backoff;
    }
    return exclusive;
}

// Shared state of one tile.
template <int ENTRIES>
struct TileShared {
    uint32_t counts[ENTRIES];  // per (item, warp) keep counts, then their exclusive offsets
    uint32_t tile;             // this CTA's tile ticket
    uint32_t tag;              // launch tag
    uint32_t prefix;           // exclusive prefix of the tile over all earlier tiles
    uint32_t aggregate;        // kept elements in the tile
    uint32_t ok;               // look-back finished in time
};

// Run by one full warp after every warp has written its counts: exclusive
// scan of the ENTRIES counts in place and publication of the tile aggregate,
// which is returned.  Publishing is skipped for the tile `skip_tile` (test
// hook).
template <int ENTRIES>
__device__ __forceinline__ uint32_t tile_scan_publish(TileShared<ENTRIES> &st, const StatusRing &ring, uint64_t tile,
                                                      uint64_t first, int64_t skip_tile)
{
    constexpr int C = (ENTRIES + 31) / 32;
    const uint32_t lane = threadIdx.x & 31u;
    uint32_t local[C];
    uint32_t sum = 0;
#pragma unroll
    for (int c = 0; c < C; ++c) {
        const int e = static_cast<int>(lane) * C + c;
        local[c] = e < ENTRIES ? st.counts[e] : 0u;
        sum += local[c];
    }
    const uint32_t incl = warp_inclusive_scan(sum);
    uint32_t run = incl - sum;
#pragma unroll
    for (int c = 0; c < C; ++c) {
        const int e = static_cast<int>(lane) * C + c;
        if (e < ENTRIES) st.counts[e] = run;
        run += local[c];
    }
    const uint32_t aggregate = __shfl_sync(kFull, incl, 31);
    if (lane == 0 && static_cast<int64_t>(tile) != skip_tile)
        st_relaxed_gpu(ring.slot(tile), status_word(ring.tag(tile), tile == first, aggregate));
    return aggregate;
}

// Then, by the same warp: look-back and publication of the inclusive prefix.
template <int ENTRIES>
__device__ __forceinline__ void tile_lookback(TileShared<ENTRIES> &st, uint32_t aggregate, const StatusRing &ring,
                                              uint64_t tile, uint64_t first, uint64_t timeout_ns, int64_t skip_tile,
                                              WsHeader *ws)
{
    const uint32_t lane = threadIdx.x & 31u;
    const bool publish = static_cast<int64_t>(tile) != skip_tile;
    uint32_t exclusive = 0;
    bool ok = true;
    if (tile > first) {
        const long long c0 = clock_mark();
        exclusive = lookback(ring, tile, first, timeout_ns, ok);
        if (lane == 0) clock_add(&ws->lookback_cycles, c0);
        if (lane == 0 && publish)
            st_relaxed_gpu(ring.slot(tile), status_word(ring.tag(tile), true, exclusive + aggregate));
        if (lane == 0 && !ok) record_error(ws, kErrLookbackTimeout, tile);
    }
    if (lane == 0) {
        st.prefix = exclusive;
        st.aggregate = aggregate;
        st.ok = ok ? 1u : 0u;
    }
}

// Both steps at once.
template <int ENTRIES>
__device__ __forceinline__ void tile_scan_lookback(TileShared<ENTRIES> &st, const StatusRing &ring, uint64_t tile,
                                                   uint64_t first, uint64_t timeout_ns, int64_t skip_tile,
                                                   WsHeader *ws)
{
    const uint32_t aggregate = tile_scan_publish(st, ring, tile, first, skip_tile);
    tile_lookback(st, aggregate, ring, tile, first, timeout_ns, skip_tile, ws);
}

// Called by one thread per CTA once the CTA no longer reads the header: the
// last CTA of the launch resets the ticket and the counter and advances the
// tag, leaving the header ready for the next launch on the stream.
__device__ __forceinline__ void finish_launch(WsHeader *ws, uint32_t tag, uint32_t ctas)
{
    __threadfence();
    const uint32_t d = atomicAdd(&ws->done, 1u);
    if (d == ctas - 1u) {
        atomicExch(&ws->ticket, 0u);
        atomicExch(&ws->done, 0u);
        atomicExch(&ws->tag, next_tag(tag));
        __threadfence();
    }
}

// ------------------------------------------------------------------ async copies and mbarriers
// Helpers of the pipelined kernels: shared-memory mbarriers and cp.async copies
// global -> shared.

__device__ __forceinline__ uint32_t smem_u32(const void *p)
{
    return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

__device__ __forceinline__ void mbar_init(uint64_t *bar, uint32_t count)
{
    asm volatile("mbarrier.init.shared.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}

__device__ __forceinline__ void mbar_arrive(uint64_t *bar)
{
    asm volatile(
        "{\n\t.reg .b64 state;\n\t"
        "mbarrier.arrive.shared.b64 state, [%0];\n\t}" ::"r"(smem_u32(bar))
        : "memory");
}

__device__ __forceinline__ bool mbar_test(uint64_t *bar, uint32_t parity)
{
    uint32_t done;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(done)
        : "r"(smem_u32(bar)), "r"(parity)
        : "memory");
    return done != 0u;
}

// Waits for the completion of the barrier phase of parity `parity`; gives up
// (false) after `limit_ns` or when another role has raised `abort`.
__device__ __forceinline__ bool mbar_wait(uint64_t *bar, uint32_t parity, uint64_t limit_ns,
                                          const volatile uint32_t *abort)
{
    uint64_t start = 0;
    uint32_t spins = 0;
    while (!mbar_test(bar, parity)) {
        if (*abort != 0u) return false;
        const uint64_t now = global_ns();
        if (start == 0) {
            start = now;
        } else if (now - start > limit_ns || ++spins > (1u << 26)) {
            return false;
        }
    }
    return true;
}

// 16-byte copies bypass L1 (.cg): for random 16-byte gathers, allocating in
// L1 made the pipelined kernel 1.57x slower on GB300.  .cg takes 16 bytes
// only, so smaller copies allocate (.ca).
template <int BYTES>
__device__ __forceinline__ void cp_async(void *dst_smem, const void *src)
{
    static_assert(BYTES == 4 || BYTES == 8 || BYTES == 16, "cp.async copies 4, 8 or 16 bytes");
    if constexpr (BYTES == 16)
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_u32(dst_smem)), "l"(src) : "memory");
    else
        asm volatile("cp.async.ca.shared.global [%0], [%1], %2;" ::"r"(smem_u32(dst_smem)), "l"(src), "n"(BYTES)
                     : "memory");
}

__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_all;" ::: "memory"); }

__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }

// Waits until every copy group of this thread but the most recent one has landed.
__device__ __forceinline__ void cp_async_wait_prior() { asm volatile("cp.async.wait_group 1;" ::: "memory"); }

// Waits until every copy group of this thread but the N most recent has landed.
template <int N>
__device__ __forceinline__ void cp_async_wait_groups()
{
    asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

}  // namespace dev
}  // namespace bsh
