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
// (level of code IA of word wa, level of code IB of word wb)
template <int BITS, int IA, int IB = IA>
__device__ __forceinline__ float2 code_pair(uint32_t wa, uint32_t wb) {
  const float2 v = make_float2(code_float<BITS, IA>(wa), code_float<BITS, IB>(wb));
  if constexpr (BITS == 8) {
    return __fadd2_rn(v, make_float2(-8388736.0f, -8388736.0f));  // 2^23 + (c ^ 0x80) - 2^23 - 128
  } else {
    constexpr int sa = CodeAt<BITS, IA>::S, sb = CodeAt<BITS, IB>::S;
    constexpr float fa = (float)(2.0 / (double)(1u << sa)), fb = (float)(2.0 / (double)(1u << sb));
    constexpr float ka = -((float)(1u << (24 - sa)) + (float)((1 << BITS) - 1));
    constexpr float kb = -((float)(1u << (24 - sb)) + (float)((1 << BITS) - 1));
    if constexpr (sa == 1 && sb == 1) return __fadd2_rn(v, make_float2(ka, kb));
    else return __ffma2_rn(v, make_float2(fa, fb), make_float2(ka, kb));
  }
}

// ------------------------------------------------------------------------------------------
// phase 1's staged tiles (Plan<LOGN>::Stage1<BITS>, WidePlan<LOGN>::Stage<BITS>): N1 rows of WPR words per IF, RP
// words apart ([IF][row][word]), transposed so that lane q1 of column col finds its rows q1 + Q1 t, t < P1, of
// both IFs in BR words: code t of IF a is code t % SPW of word t / SPW, IF b's follow IF a's.
// ------------------------------------------------------------------------------------------
// unit u of a tile: KB blocks of SPW words, from the staged words into x (transposed)
template <typename PL, typename ST, int BITS>
__device__ __forceinline__ void p1_unit_load(const uint32_t* raw, int u, uint32_t (&x)[ST::KB][32 / BITS]) {
  constexpr int SPW = ST::SPW, P = PL::P1, Q1 = PL::Q1, N1 = PL::N1, WPR = ST::WPR, RP = ST::RP, KB = ST::KB;
  const int w = u % WPR, q1 = (u / WPR) % Q1, vb = (u / (WPR * Q1)) * KB;
  // codes vb SPW .. of the lane: of one IF where P >= SPW (P codes per IF), else of both
  constexpr int BPI = P >= SPW ? P / SPW : 1;  // blocks per IF
  const uint32_t* src = raw + (P >= SPW ? (vb / BPI) * N1 * RP + (vb % BPI) * SPW * Q1 * RP : 0) + q1 * RP + w;
  sfor<0, KB>([&](auto k_) {
    constexpr int k = decltype(k_)::value;
    sfor<0, SPW>([&](auto i_) {
      constexpr int i = decltype(i_)::value, j = k * SPW + i;
      constexpr int off = P >= SPW ? j * Q1 * RP : (j / P) * N1 * RP + (j % P) * Q1 * RP;
      x[k][i] = src[off];
    });
    transpose_codes<BITS>(x[k]);
  });
}
template <typename PL, typename ST, int BITS>
__device__ __forceinline__ void p1_unit_store(uint32_t* tr, int u, const uint32_t (&x)[ST::KB][32 / BITS]) {
  constexpr int SPW = ST::SPW, Q1 = PL::Q1, WPR = ST::WPR, KB = ST::KB, VL = ST::VL;
  const int w = u % WPR, q1 = (u / WPR) % Q1, vb = (u / (WPR * Q1)) * KB;
  uint32_t* dst = tr + ((vb / VL) * Q1 * ST::SQ + q1 * ST::SQ + w * (SPW + ST::PADW)) * VL + vb % VL;
  sfor<0, SPW>([&](auto c_) {
    constexpr int c = decltype(c_)::value;
    if constexpr (KB == 4)
      *reinterpret_cast<uint4*>(dst + c * VL) =
          make_uint4(stored_codes<BITS>(x[0][c]), stored_codes<BITS>(x[1][c]), stored_codes<BITS>(x[2][c]),
                     stored_codes<BITS>(x[3][c]));
    else if constexpr (KB == 2)
      *reinterpret_cast<uint2*>(dst + c * VL) = make_uint2(stored_codes<BITS>(x[0][c]), stored_codes<BITS>(x[1][c]));
    else
      dst[c * VL] = stored_codes<BITS>(x[0][c]);
  });
}
// the codes of lane q1, column col of the tile
template <typename PL, typename ST>
__device__ __forceinline__ void p1_lane_codes(const uint32_t* tr, int q1, int col, uint32_t (&cw)[ST::BR]) {
  constexpr int VL = ST::VL;
  const uint32_t* src = tr + (q1 * ST::SQ + col + (col / ST::SPW) * ST::PADW) * VL;
  sfor<0, ST::BR / VL>([&](auto q_) {
    constexpr int q = decltype(q_)::value, o = q * PL::Q1 * ST::SQ * VL;
    if constexpr (VL == 4) {
      const uint4 x = *reinterpret_cast<const uint4*>(src + o);
      cw[4 * q] = x.x;
      cw[4 * q + 1] = x.y;
      cw[4 * q + 2] = x.z;
      cw[4 * q + 3] = x.w;
    } else if constexpr (VL == 2) {
      const uint2 x = *reinterpret_cast<const uint2*>(src + o);
      cw[2 * q] = x.x;
      cw[2 * q + 1] = x.y;
    } else {
      cw[q] = src[o];
    }
  });
}
// (level of IF a, level of IF b) of the lane's row t (HB false: no IF b, zero)
template <typename PL, typename ST, int BITS, bool HB, int T>
__device__ __forceinline__ float2 p1_level(const uint32_t (&cw)[ST::BR]) {
  constexpr int SPW = ST::SPW, P = PL::P1;
  float2 z = code_pair<BITS, T % SPW, (P + T) % SPW>(cw[T / SPW], cw[(P + T) / SPW]);
  if constexpr (!HB) z.y = 0.f;
  return z;
}

}  // namespace polaris
