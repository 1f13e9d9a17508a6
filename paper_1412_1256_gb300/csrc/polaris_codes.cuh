// Data translation (Fig. 2 caption: integer codes to floats) from transposed codes.
//
// A transform's lane needs one code from each of many packed words (its column b of the rows
// n = N2 a + b), while a word holds 32/BITS consecutive samples, so decoding straight from the
// packed words costs a shared-memory load, a funnel shift and a logic operation per sample.
// Transposing SPW x SPW blocks of codes first (SPW = 32/BITS words, in one thread's registers)
// puts SPW rows of one column into one word: a lane then reads its codes with a few vector
// loads and needs no shift per sample.
#pragma once
#include <stdint.h>

#include "polaris_device.cuh"

namespace polaris {

// Codes r of words c become codes c of words r (w[i]: word i of the block; code j of a word at
// bits [j BITS, (j+1) BITS)): log2(SPW) exchange stages, the 16- and 8-bit ones two byte
// permutes per word pair, the finer ones two shifts and two three-input logic operations.
template <int BITS>
__device__ __forceinline__ void transpose_codes(uint32_t (&w)[32 / BITS]) {
  constexpr int S = 32 / BITS;
  sfor<0, ct::ilog2(S)>([&](auto st_) {
    constexpr int half = S >> (decltype(st_)::value + 1), sh = half * BITS;
    constexpr uint32_t m = sh == 16 ? 0x0000FFFFu : sh == 8 ? 0x00FF00FFu : sh == 4 ? 0x0F0F0F0Fu
                                                : sh == 2   ? 0x33333333u : 0x55555555u;
    sfor<0, S / 2>([&](auto p_) {
      constexpr int p = decltype(p_)::value;
      constexpr int i = (p / half) * 2 * half + p % half;
      const uint32_t a = w[i], b = w[i + half];
      if constexpr (sh == 16) {
        w[i] = __byte_perm(a, b, 0x5410);
        w[i + half] = __byte_perm(a, b, 0x7632);
      } else if constexpr (sh == 8) {
        w[i] = __byte_perm(a, b, 0x6240);
        w[i + half] = __byte_perm(a, b, 0x7351);
      } else {
        w[i] = (a & m) | ((b << sh) & ~m);
        w[i + half] = ((a >> sh) & m) | (b & ~m);
      }
    });
  });
}

// A transposed word as decode_codes takes it: 8-bit codes offset to unsigned (c ^ 0x80).
template <int BITS>
__device__ __forceinline__ uint32_t stored_codes(uint32_t w) {
  return BITS == 8 ? w ^ 0x80808080u : w;
}

// Code I of a word as a float whose mantissa holds it at bit position S (2^23 + c 2^S), so that
// level = value 2^(1-S) - (2^(24-S) + 2^b - 1): one multiply-add, exact.  S >= 1 keeps the odd
// constant representable; codes above the mantissa come from one shift of the word per group.
template <int BITS, int I>
struct CodeAt {
  static constexpr int FIT = (23 - 1) / BITS;            // codes of one shifted word that fit at S >= 1
  static constexpr int G = BITS == 8 ? 0 : I / FIT;      // which shifted word
  static constexpr int S = BITS == 8 ? 0 : 1 + BITS * (I % FIT);
};
template <int BITS, int I>
__device__ __forceinline__ float code_float(uint32_t w) {
  using C = CodeAt<BITS, I>;
  if constexpr (BITS == 8) {
    return __uint_as_float(__byte_perm(w, 0x4B000000u, 0x7440 | I));
  } else {
    constexpr int first = C::G * C::FIT * BITS;  // bit of the group's first code, to go to bit 1
    const uint32_t r = C::G == 0 ? w << 1 : w >> (first - 1);
    return __uint_as_float(and_or(r, ((1u << BITS) - 1u) << C::S, 0x4B000000u));
  }
}
// (level of code I of word wa, level of code I of word wb)
template <int BITS, int I>
__device__ __forceinline__ float2 code_pair(uint32_t wa, uint32_t wb) {
  using C = CodeAt<BITS, I>;
  const float2 v = make_float2(code_float<BITS, I>(wa), code_float<BITS, I>(wb));
  if constexpr (BITS == 8) {
    return __fadd2_rn(v, make_float2(-8388736.0f, -8388736.0f));  // 2^23 + (c ^ 0x80) - 2^23 - 128
  } else {
    constexpr float sc = (float)(2.0 / (double)(1u << C::S));
    constexpr float k = -((float)(1u << (24 - C::S)) + (float)((1 << BITS) - 1));
    if constexpr (C::S == 1) return __fadd2_rn(v, make_float2(k, k));
    else return __ffma2_rn(v, make_float2(sc, sc), make_float2(k, k));
  }
}

}  // namespace polaris
