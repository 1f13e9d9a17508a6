// The whole hot path of the small transforms (N = 2^10 .. 2^14) in one kernel: data translation,
// window, segment FFT, correlation and integration (Fig. 2 caption), with the pair-segment in
// registers and shared memory from its packed words to its accumulators.
//
//   k_fused  a team of W = N/1024 warps takes a range of segments of one FFT pair, one segment
//            at a time, 32 points per lane.  N = 32 B (row a, column b, n = B a + b; bin
//            k = c + 32 d): lane b runs the 32-point DFT over its column's rows, multiplies by
//            W_N^{b c} (tensor memory) and the team exchanges [c][b] through shared memory; the
//            B-point DFTs of the 32 columns c follow within warps:
//              2^10  lane c, 32 points
//              2^11  64 points over two lanes by the parity of the output index (x_i +- x_{i+32},
//                    the odd half turned by W_64^i)
//              2^12+ B = 16 P1: P1-point DFTs over b1 (b = 16 b1 + b0), W_B^{b0 d1}, an exchange
//                    among the P1/2 lanes of the column, 16-point DFTs over b0 (d = d1 + P1 d0)
//            A bin and its mirror (column 32 - c, in the same warp, conjugated and taken through
//            column c's own twiddles) meet by one shuffle per component; |X|^2, |Y|^2 and X conj(Y)
//            (as in k_phase2) accumulate in tensor memory over the range.  At the end the CTA's teams
//            are summed in shared memory and added once to the integration accumulators, which hold
//            the bins in natural order.
//            FP64 accumulators: every `flush` segments instead, the teams summed in twice FP32's
//            precision, so that the sums do not lose bits as a feed gets longer.  The lengths are those of
//            the two-kernel path's ranges (a pass of 4096 segments over its warps).  Passes of four 2-bit IFs
//            of 8 M samples with one addition at the end and so: 2^10 33.1, 38.4 us; 2^11 40.2, 41.9; 2^12
//            50.3, 52.2; 2^13 68.2, 52.2; 2^14 81.4, 61.4 (FP32 accumulators: 31.0 to 51.4): the last ones
//            from consecutive lanes adding consecutive values and from fewer FP64 instructions, which
//            bound this part (teams summed in FP64: 2^25 samples of one pair at 2^10 314 us, now 162).
//
// What bounds it: instruction issue, 47 instructions per complex point (2^14, 1024 segments of two
// pairs, set-up included) at 43 to 51% of the issue slots with 16 warps per SM (registers), against 64 of
// the two-phase path of the larger sizes, which these sizes took before and which sends every point
// through a slab in L2.  Measured against that path (GB300, four 2-bit IFs of 8 M samples, whole
// passes, Msample/s before and after): 2^10 313k, 1082k; 2^11 435k, 912k; 2^12 393k, 788k; 2^13
// 480k, 706k; 2^14 478k, 653k; 64 int8 Hann segments of 1024 points 28.7 and 13.4 us (host-bound);
// one 2^14 segment 23 and 17 us.  (2^12 with both transforms split by parity like 2^11's second one,
// 64 x 64 points, ran at 727k.)  The line: 2^15 points do not fit an SM's registers, and below 2^10
// a warp would hold several segments.
#pragma once
#include "polaris_codes.cuh"
#include "polaris_kernels.cuh"

namespace polaris {

template <int LOGN>
struct FusedPlan {
  static constexpr int N = 1 << LOGN, W = N / 1024;     // warps per team
  static constexpr int WARPS = W > 8 ? W : 8, THREADS = 32 * WARPS, T = WARPS / W;  // teams per CTA
  static constexpr int MINB = WARPS > 8 ? 1 : 2;        // CTAs per SM (16 warps either way)
  static constexpr int R = 32, B = 1 << fused_log_b(LOGN);  // rows, columns
  static constexpr int HB = B == 64 ? 2 : 1;            // lanes per column (2^10, 2^11)
  static constexpr bool THREE = B > 64;                 // the B-point DFT in two steps
  static constexpr int P1 = THREE ? B / 16 : 1;
  static constexpr int LC = THREE ? P1 / 2 : 1;         // lanes per column
  // [c][b] rows.  Two steps: an odd pitch puts consecutive c on distinct bank pairs.  Three: rows
  // also take [d1][b0] at 17 d1 + b0, and the columns of a half-warp lie an odd multiple of LC bank pairs apart
  static constexpr int PITCH = !THREE ? B + 1 : B == 128 ? 140 : B == 256 ? 280 : 544;
  static constexpr int REGION = R * PITCH;              // float2 per team
  static constexpr int TW2 = THREE ? B : 0;             // W_B^{b0 d1} at 16 d1 + b0
  static constexpr int TCOLS = (WARPS / 4) * 128;       // 64 accumulator and 64 twiddle columns per lane
  // FP64 accumulators: segments per FFT pair (14 at most) that a team sums in FP32 before it adds to them
  static constexpr int FLUSH = LOGN == 10 ? 2 : LOGN == 11 ? 4 : LOGN == 12 ? 7 : 14;
  template <int BITS>
  struct In {
    static constexpr int SPW = 32 / BITS;
    static constexpr int WPR = B * BITS / 32;           // words per row
    static constexpr int NW = N * BITS / 32;            // words per segment of one IF
    static constexpr int BR = 2 * R / SPW;              // block rows of both IFs (SPW rows each)
    static constexpr int NB = BR * WPR;                 // SPW x SPW blocks of a pair-segment
    // segments staged at once: as many as give each lane of the team a block (at most 8, for
    // shared memory; a block's transpose is 100 to 260 instructions however many lanes have one)
    static constexpr int G = (32 * W / NB < 1) ? 1 : (32 * W / NB > 8 ? 8 : 32 * W / NB);
    // A warp's lanes take WL consecutive words of consecutive block rows.  Packed words as they
    // arrive: WL words of padding per block row put those on distinct banks
    static constexpr int WL = WPR < 8 ? WPR : 8;
    static constexpr int RAWBLK = SPW * WPR + WL, RAW = BR * RAWBLK;
    // transposed words: BR words per column, VL of them side by side for one vector load, column b
    // at place b + b / PADC: the readers' eight lanes are consecutive vectors, the writers' WL
    // columns SPW apart fall on distinct ones of eight (sixteen of 8 bytes at 1 bit)
    static constexpr int VW = BR, VL = VW < 4 ? VW : 4;
    static constexpr int PADC = SPW < 8 ? 8 : SPW;
    static constexpr int SLAB = (B + B / PADC) * VL, TR = (VW / VL) * SLAB;
    static constexpr size_t TEAM = sizeof(float2) * REGION + 4 * (size_t)G * (RAW + TR);
    static constexpr size_t SMEM = T * TEAM + 16 * T + 8 * TW2 + 16;  // + extra bin per team, W_B, TMEM slot
    static_assert((G * RAW) % 4 == 0 && SLAB % VL == 0 && TR % VL == 0 && TEAM % 16 == 0, "vector loads aligned");
    static_assert(MINB * (SMEM + 1024) <= 233472, "CTAs per SM");
  };
  static_assert(REGION * sizeof(float2) % 16 == 0 && REGION * 8 >= 16 * (N / 2), "region holds the team's sums");
  static_assert(!THREE || (PITCH >= 17 * P1 && (LC == 16 || (PITCH % LC == 0 && PITCH / LC % 2 == 1))), "column rows");
};

// hi + lo += x, the rounding error of the sum (Knuth's TwoSum) kept in lo
__device__ __forceinline__ void two_sum(float& hi, float& lo, float x) {
  const float s = __fadd_rn(hi, x), b = __fsub_rn(s, hi);
  lo = __fadd_rn(lo, __fadd_rn(__fsub_rn(hi, __fsub_rn(s, b)), __fsub_rn(x, b)));
  hi = s;
}

// x in FP64, by integer operations: FP64 ones, the conversion among them, take a scheduler 64 cycles a warp
__device__ __forceinline__ double widen(float x) {
  const uint32_t b = __float_as_uint(x), e = b & 0x7F800000u;
  if (e == 0x7F800000u || (e == 0 && x != 0.f)) return (double)x;  // infinite, NaN, denormal
  const uint32_t h = (b & 0x80000000u) | (x != 0.f ? ((b & 0x7FFFFFFFu) >> 3) + 0x38000000u : 0u);
  return __hiloint2double((int)h, (int)(b << 29));
}

template <int W>
__device__ __forceinline__ void team_sync(int team) {
  if constexpr (W == 1) __syncwarp();
  else asm volatile("bar.sync %0, %1;\n" ::"r"(1 + team), "r"(32 * W) : "memory");
}

// where word j of a segment of one IF is staged
template <typename IN>
__device__ __forceinline__ uint32_t fused_raw_place(int j) {
  return (uint32_t)(j + (j / (IN::SPW * IN::WPR)) * IN::WL);
}
// codes of the cnt staged segments transposed, block by block (SPW words down a word column of one block
// row), by the TL lanes of the team
template <typename IN, int BITS, int TL>
__device__ __forceinline__ void fused_transpose(const uint32_t* raw, uint32_t* tr, int cnt, int tl) {
  constexpr int SPW = IN::SPW, WPR = IN::WPR, WL = IN::WL, VL = IN::VL;
#pragma unroll 1
  for (int k = tl; k < cnt * IN::NB; k += TL) {
    const int br = (k / WL) % IN::BR, w = k % WL + (k / (WL * IN::BR)) % (WPR / WL) * WL, g = k / IN::NB;
    const uint32_t* src = raw + g * IN::RAW + br * IN::RAWBLK + w;
    uint32_t x[SPW];
    sfor<0, SPW>([&](auto i_) { x[decltype(i_)::value] = src[decltype(i_)::value * WPR]; });
    transpose_codes<BITS>(x);
    // (columns w SPW + c, c < SPW, share one PADC group)
    uint32_t* dst = tr + g * IN::TR + (br / VL) * IN::SLAB + (w * SPW + w * SPW / IN::PADC) * VL + br % VL;
    sfor<0, SPW>([&](auto c_) { dst[decltype(c_)::value * VL] = stored_codes<BITS>(x[decltype(c_)::value]); });
  }
}
// the codes of column tl of staged segment g, and its levels in row t
template <typename IN>
__device__ __forceinline__ void fused_lane_codes(const uint32_t* tr, int g, int tl, uint32_t (&cw)[IN::VW]) {
  constexpr int VL = IN::VL;
  const uint32_t* col = tr + g * IN::TR + (tl + tl / IN::PADC) * VL;
  sfor<0, IN::VW / VL>([&](auto q_) {
    constexpr int q = decltype(q_)::value;
    if constexpr (VL == 4) {
      const uint4 x = *reinterpret_cast<const uint4*>(col + q * IN::SLAB);
      cw[4 * q] = x.x;
      cw[4 * q + 1] = x.y;
      cw[4 * q + 2] = x.z;
      cw[4 * q + 3] = x.w;
    } else {
      const uint2 x = *reinterpret_cast<const uint2*>(col + q * IN::SLAB);
      cw[2 * q] = x.x;
      cw[2 * q + 1] = x.y;
    }
  });
}
template <typename IN, int BITS, bool HB, int T>
__device__ __forceinline__ float2 fused_level(const uint32_t (&cw)[IN::VW]) {
  float2 z = code_pair<BITS, T % IN::SPW>(cw[T / IN::SPW], cw[IN::VW / 2 + T / IN::SPW]);
  if constexpr (!HB) z.y = 0.f;
  return z;
}

// FP64: the integration accumulators are doubles
template <int LOGN, int BITS, bool FP64>
__global__ void __launch_bounds__(FusedPlan<LOGN>::THREADS, FusedPlan<LOGN>::MINB) k_fused(BatchArgs a) {
  using PL = FusedPlan<LOGN>;
  using IN = typename PL::template In<BITS>;
  constexpr int W = PL::W, T = PL::T, B = PL::B, R = PL::R, HB = PL::HB, PITCH = PL::PITCH, P1 = PL::P1, LC = PL::LC;
  constexpr bool THREE = PL::THREE;
  constexpr int G = IN::G, TL = 32 * W;
  extern __shared__ __align__(16) unsigned char smf[];
  const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0), lane = tid & 31;
  const int team = warp / W, wt = warp % W, tl = wt * 32 + lane;  // team, warp and lane inside it
  unsigned char* mine = smf + team * IN::TEAM;
  float2* region = reinterpret_cast<float2*>(mine);
  uint32_t* raw = reinterpret_cast<uint32_t*>(mine + sizeof(float2) * PL::REGION);
  uint32_t* tr = raw + G * IN::RAW;
  float4* xbin = reinterpret_cast<float4*>(smf + T * IN::TEAM);
  float2* tw2 = reinterpret_cast<float2*>(xbin + T);
  uint32_t* tslot = reinterpret_cast<uint32_t*>(tw2 + PL::TW2);

  // lane roles: step A column tl.  Afterwards column cb (unit u: column u in lanes 0-15, its mirror
  // 32 - u in lanes 16-31; unit 0: columns 0 and 16), output parity hb (2^11) or lane l of the
  // column's LC (2^12 and up)
  const int mir = lane >> 4;
  const int hb = HB == 2 ? (lane >> 3) & 1 : 0, l = THREE ? lane % LC : 0;
  const int u = THREE ? (16 / LC) * wt + (lane & 15) / LC : HB == 2 ? 8 * wt + (lane & 7) : lane & 15;
  const int cb = u == 0 ? (mir ? 16 : 0) : (mir ? 32 - u : u);
  // Columns u and 32 - u, 0 < u < 16: column 32 - u goes conjugated through column u's twiddles and
  // transform, its odd b negated, so that its output d is conj Z[N - k] of bin k = u + 32 (d + B/2 mod B): a
  // lane and its `partner` hold bins and mirrors at d and d + B/2, and each two of them have had the same
  // operations.  Both columns by their own twiddles leaked the rounding of the transform's constants
  // from X into Y: cross spectra of 2^25 samples 1.5e-8 to 2.1e-8 rms off, of sqrt(A_x A_y), 4.5e-9 to
  // 6.0e-9 so; time within 2%, 2^10 4 bits 3%.
  // Columns 0 and 16 hold their own mirrors.  Two steps: output 31 - i of `partner` mirrors output
  // i; column 0's even outputs mirror onto themselves (output (32 - i) mod 32 of the lane itself).
  // Three: a lane holds d1 = l (slot 0) and P1 - 1 - l (slot 1); the mirror of (slot, d0) is the other
  // slot's 15 - d0, in column 0 in slot 1 of lane l - 1 (for slot 0) and slot 0 of lane l + 1 (for slot
  // 1), except d1 = 0 and P1/2, which mirror onto themselves
  const int partner = u != 0 ? lane ^ 16 : (THREE || HB == 1 || mir == 0) ? lane : lane ^ 8;
  const int partner0 = THREE && cb == 0 && l > 0 ? lane - 1 : partner;
  const int partner1 = THREE && cb == 0 && l < LC - 1 ? lane + 1 : partner;
  const bool conjg = mir && u != 0;
  const bool self = cb == 0 && hb == 0 && l == 0, self1 = THREE && cb == 0 && l == LC - 1;

  if constexpr (THREE) {
    for (int i = tid; i < B; i += PL::THREADS) tw2[i] = tw_small<B>((i & 15) * (i >> 4));
  }
  const uint32_t tbase = __shfl_sync(0xffffffffu, cta_tmem_begin<PL::TCOLS>(tslot, warp), 0);
  const uint32_t t_acc = tbase + ((uint32_t)(32 * (warp & 3)) << 16) + (uint32_t)((warp >> 2) * 128);
  const uint32_t t_tw = t_acc + 64;
  sfor<0, 4>([&](auto c_) {
    constexpr int cc = decltype(c_)::value;
    float z16[16], w16[16];
    sfor<0, 16>([&](auto k_) { z16[decltype(k_)::value] = 0.f; });
    tmem_st16(t_acc + 16 * cc, z16);
    sfor<0, 8>([&](auto k_) {  // W_N^{b c}, b = tl
      constexpr int k = decltype(k_)::value;
      const float2 w = __ldg(a.tw + (8 * cc + k) * B + tl);
      w16[2 * k] = w.x;
      w16[2 * k + 1] = w.y;
    });
    tmem_st16(t_tw + 16 * cc, w16);
  });
  tmem_wait_st();
  pdl_wait();  // the input and the accumulators may be touched from here on (dependent launch)

  // this team's segments of FFT pair f
  const int f = (int)(blockIdx.x % a.n_fpair), slot = (int)(blockIdx.x / a.n_fpair);
  const long long teams = (long long)(gridDim.x / a.n_fpair) * T, ti = (long long)slot * T + team;
  const int s_begin = (int)(a.nseg * ti / teams), s_end = (int)(a.nseg * (ti + 1) / teams);
  const int ia = a.fa[f], ib = a.fb[f];
  auto issue = [&](int s0) {  // the packed words of segments s0 .. s0 + G - 1 (below s_end), asynchronously
#pragma unroll 1
    for (int g = 0; g < G && s0 + g < s_end; ++g) {
      const int s = s0 + g;
      const uint32_t *pa = seg_ptr(a.in, ia, s), *pb = ib >= 0 ? seg_ptr(a.in, ib, s) : pa;
      const long long w0 = seg_word0(a.in, s), wext = s < a.in.n0 ? a.in.in_words0 : a.in.in_words1;
      const uint32_t dst = smem_addr(raw + g * IN::RAW);
      sfor<0, IN::NW / TL>([&](auto i_) {
        const int j = tl + decltype(i_)::value * TL;
        const uint32_t o = 4u * fused_raw_place<IN>(j);
        if (in_bounds(a.err, w0 + j, wext)) {
          cp_async4(dst + o, pa + j);
          cp_async4(dst + o + 4u * (uint32_t)(IN::RAW / 2), pb + j);
        }
      });
    }
    cp_async_commit();
  };

  float extra[4] = {0.f, 0.f, 0.f, 0.f};
  [[maybe_unused]] const float sgn_b = hb ? -1.f : 1.f;
  auto transpose = [&](int cnt) { fused_transpose<IN, BITS, TL>(raw, tr, cnt, tl); };
  // Segments come in groups of G.  The next group's words are copied during a group and transposed in
  // its last segment, between the two barriers of the exchange, which order those steps too: two
  // barriers per segment (with a pass of its own over each group, four per segment at 4 and 8 bits)
  if (s_begin < s_end) {
    issue(s_begin);
    cp_async_wait_all();
    team_sync<W>(team);
    transpose(min(G, s_end - s_begin));
    team_sync<W>(team);
    if (s_begin + G < s_end) issue(s_begin + G);
  }
  // rounds: one; with FP64 accumulators as many as keep a team's FP32 sums to `flush` segments
  const int flush = min(14, PL::FLUSH * a.n_fpair);
  const int rounds = FP64 ? (int)(((a.nseg + teams - 1) / teams + flush - 1) / flush) : 1;
  int g = 0, s = s_begin;
#pragma unroll 1
  for (int left = rounds; left > 0; --left) {
    const int s_stop = FP64 && left > 1 ? min(s + flush, s_end) : s_end;
#pragma unroll 1
    for (; s < s_stop; ++s) {
      const bool turn = g == G - 1 && s + 1 < s_end;  // the next segment starts a group
      // step A: decode column tl, window, 32-point DFT
      float2 v[32];
      uint32_t cw[IN::VW];
      fused_lane_codes<IN>(tr, g, tl, cw);
      auto rows = [&](auto hb_, auto tp_) {
        constexpr bool HBP = decltype(hb_)::value, TP = decltype(tp_)::value;
        [[maybe_unused]] const float4* tp = reinterpret_cast<const float4*>(a.taps) + tl;
        [[maybe_unused]] float4 w4;
        sfor<0, 32>([&](auto t_) {
          constexpr int t = decltype(t_)::value;
          float2 z = fused_level<IN, BITS, HBP, t>(cw);
          if constexpr (TP) {  // (four consecutive t per load: tap_order)
            if constexpr (t % 4 == 0) w4 = __ldg(tp + (t / 4) * B);
            const float x = t % 4 == 0 ? w4.x : t % 4 == 1 ? w4.y : t % 4 == 2 ? w4.z : w4.w;
            z = __fmul2_rn(z, make_float2(x, x));
          }
          v[ct::bitrev(t, 32)] = z;
        });
      };
      using T_ = std::true_type;
      using F_ = std::false_type;
      if (a.taps) {
        if (ib >= 0) rows(T_{}, T_{});
        else rows(F_{}, T_{});
      } else {
        if (ib >= 0) rows(T_{}, F_{});
        else rows(F_{}, F_{});
      }
      dit<32>(v);
      sfor<0, 4>([&](auto c_) {
        constexpr int cc = decltype(c_)::value;
        float w16[16];
        tmem_ld16(t_tw + 16 * cc, w16);
        tmem_wait_ld();
        sfor<0, 8>([&](auto k_) {
          constexpr int k = decltype(k_)::value, i = 8 * cc + k;
          const float2 w = make_float2(w16[2 * k], w16[2 * k + 1]);
        if constexpr (i > 16) v[i] = cmulc(v[i], w);  // conjugated: mirrors of column 32 - i
        else if constexpr (i > 0) v[i] = cmul(v[i], w);
        });
      });
      if (turn) cp_async_wait_all();
      team_sync<W>(team);  // the previous exchange and this group's codes have been read; the next group is staged
      sfor<0, 32>([&](auto i_) {
        constexpr int i = decltype(i_)::value;
        region[i * PITCH + tl] = v[i];
      });
      if (turn) transpose(min(G, s_end - s - 1));
      team_sync<W>(team);
      if (turn && s + 1 + G < s_end) issue(s + 1 + G);
      // B-point DFT of column cb
      float2* row = region + cb * PITCH;
      if constexpr (THREE) {
        sfor<0, 32 / P1>([&](auto j_) {
          constexpr int j = decltype(j_)::value;
          sfor<0, P1>([&](auto i_) {
            constexpr int i = decltype(i_)::value;
            v[j * P1 + ct::bitrev(i, P1)] = row[16 * i + l + LC * j];
          });
          dit<P1, j * P1>(v);
          sfor<1, P1>([&](auto i_) {
            constexpr int i = decltype(i_)::value;
            v[j * P1 + i] = cmul(v[j * P1 + i], tw2[16 * i + l + LC * j]);
          });
        });
        __syncwarp();  // the column's row has been read
        sfor<0, 32>([&](auto i_) {
          constexpr int i = decltype(i_)::value;
          row[17 * (i % P1) + l + LC * (i / P1)] = v[i];
        });
        __syncwarp();
        sfor<0, 2>([&](auto s_) {
          constexpr int sl = decltype(s_)::value;
          const float2* src = row + 17 * (sl ? P1 - 1 - l : l);
          sfor<0, 16>([&](auto i_) {
            constexpr int i = decltype(i_)::value;
            v[16 * sl + ct::bitrev(i, 16)] = src[i];
          });
          dit<16, 16 * sl>(v);
        });
      } else {
        sfor<0, 32>([&](auto i_) {
          constexpr int i = decltype(i_)::value;
          if constexpr (HB == 1) {
            v[ct::bitrev(i, 32)] = row[i];
          } else {
            float2 z = __ffma2_rn(row[i + 32], make_float2(sgn_b, sgn_b), row[i]);
            const float2 zt = turn64<i>(z);
            z.x = hb ? zt.x : z.x;
            z.y = hb ? zt.y : z.y;
            v[ct::bitrev(i, 32)] = z;
          }
        });
        dit<32>(v);
      }
      // correlate this lane's 16 bins below N/2, by its outputs d = HB i + hb, i < 16, or
      // d = d1 + P1 d0, d0 < 8, for the lane's two d1 (i = 8 slot + d0)
      auto correlate = [&](auto sp_) {
        constexpr bool SP = decltype(sp_)::value;  // the warp holds column 0
        sfor<0, 4>([&](auto c_) {
          constexpr int cc = decltype(c_)::value;
          float a16[16];
          tmem_ld16(t_acc + 16 * cc, a16);
          tmem_wait_ld();
          sfor<0, 4>([&](auto k_) {
            constexpr int k = decltype(k_)::value, i = 4 * cc + k;
            constexpr int sl = THREE ? i / 8 : 0, d0 = i % 8;
            constexpr int own = THREE ? 16 * sl + d0 : i, far = own + (THREE ? 8 : 16);
            const int from = !THREE ? partner : sl ? partner1 : partner0;
            float2 z = v[far];
            if constexpr (SP) {  // columns 0 and 16
              constexpr int far0 = THREE ? 16 * (sl ^ 1) + 15 - d0 : 31 - i;
              z.x = u == 0 ? v[far0].x : z.x;
              z.y = u == 0 ? -v[far0].y : z.y;
            }
            z = make_float2(__shfl_sync(0xffffffffu, z.x, from), __shfl_sync(0xffffffffu, z.y, from));
            if constexpr (SP) {  // the bins that mirror onto their own lane's outputs
              constexpr int near = THREE ? (sl ? 16 + 15 - d0 : (16 - d0) % 16) : (32 - i) % 32;
              const bool me = sl ? self1 : self;
              z.x = me ? v[near].x : z.x;
              z.y = me ? -v[near].y : z.y;
            }
            float(&q)[4] = *reinterpret_cast<float(*)[4]>(a16 + 4 * k);
            corr_acc(q, v[own], z);
          });
          tmem_st16(t_acc + 16 * cc, a16);
        });
      };
      if (W == 1 || wt == 0) correlate(std::true_type{});
      else correlate(std::false_type{});
      tmem_wait_st();
      if (self) {  // bin N/2, its own mirror
        constexpr int i = THREE ? 8 : 16;
        corr_acc(extra, v[i], make_float2(v[i].x, -v[i].y));
      }
      g = turn ? 0 : g + 1;
    }
    if (!FP64 || left == 1) pdl_trigger();
    // the CTA's teams summed in shared memory, then one add per bin (natural order; copy by CTA)
    team_sync<W>(team);
    float4* sums = reinterpret_cast<float4*>(region);
    sfor<0, 4>([&](auto c_) {
      constexpr int cc = decltype(c_)::value;
      float a16[16];
      tmem_ld16(t_acc + 16 * cc, a16);
      tmem_wait_ld();
      sfor<0, 4>([&](auto k_) {
        constexpr int k = decltype(k_)::value, i = 4 * cc + k;
        const int d = THREE ? (i / 8 ? P1 - 1 - l : l) + P1 * (i % 8) : HB * i + hb;
        // (conjugated columns: bin N/2 - u - 32 d, and X conj(Y) came out as its negative conjugate)
        sums[conjg ? PL::N / 2 - u - 32 * d : cb + 32 * d] =
            make_float4(a16[4 * k], a16[4 * k + 1], conjg ? -a16[4 * k + 2] : a16[4 * k + 2], a16[4 * k + 3]);
      });
      if (FP64 && left > 1) {
        sfor<0, 16>([&](auto i_) { a16[decltype(i_)::value] = 0.f; });
        tmem_st16(t_acc + 16 * cc, a16);
      }
    });
    if (self) xbin[team] = make_float4(extra[0], extra[1], extra[2], extra[3]);
    __syncthreads();
    const size_t base = ((size_t)(a.acc_copies > 1 ? slot % a.acc_copies : 0) * a.n_fpair + f) * (PL::N / 2 + 1);
    if constexpr (!FP64) {
      for (int k = tid; k <= PL::N / 2; k += PL::THREADS) {
        float4 t = make_float4(0.f, 0.f, 0.f, 0.f);
        for (int q = 0; q < T; ++q) {
          const float4 x = k == PL::N / 2 ? xbin[q] : reinterpret_cast<const float4*>(smf + q * IN::TEAM)[k];
          t = make_float4(t.x + x.x, t.y + x.y, t.z + x.z, t.w + x.w);
        }
        const size_t o = base + k;
        if (in_bounds(a.err, (long long)o, a.acc_slots)) atomicAdd(reinterpret_cast<float4*>(a.acc) + o, t);
      }
    } else {  // consecutive lanes take consecutive values
      double* op = reinterpret_cast<double*>(a.acc) + 4 * base;
      for (int k = tid; k < 4 * (PL::N / 2 + 1); k += PL::THREADS) {
        float hi = 0.f, lo = 0.f;  // their sum, to twice 24 bits
        for (int q = 0; q < T; ++q)
          two_sum(hi, lo, k >= 2 * PL::N ? reinterpret_cast<const float*>(xbin + q)[k - 2 * PL::N]
                                         : reinterpret_cast<const float*>(smf + q * IN::TEAM)[k]);
        const double t = T == 1 || lo != lo ? widen(hi) : widen(hi) + widen(lo);  // (lo: NaN where hi is infinite)
        if (in_bounds(a.err, (long long)base + k / 4, a.acc_slots)) atomicAdd(op + k, t);
      }
    }
    if (FP64 && left > 1) {
      for (int i = 0; i < 4; ++i) extra[i] = 0.f;
      tmem_wait_st();
      __syncthreads();  // the sums have been read: the teams' regions take the next exchange
    }
  }
  cta_tmem_end<PL::TCOLS>(tbase, warp);
}

// One launch per feed: CTAs in equal numbers per FFT pair, as many as fit and have a segment per
// team.  Either of the caller's caps holds (this kernel is both phases): with three handles and phase 1
// capped, six passes of four 2-bit IFs of 16 M samples took, uncapped and capped, 306, 295 us at 2^10,
// 368, 354 at 2^11, 404, 397 at 2^12, 465, 433 at 2^13; on one handle 339, 476; 402, 571; 439, 506; 501, 671.
template <int LOGN, int BITS, bool FP64>
static cudaError_t launch_fused_acc(const BatchArgs& a, cudaStream_t st, bool pdl) {
  using PL = FusedPlan<LOGN>;
  constexpr size_t smem = PL::template In<BITS>::SMEM;
  static int attr_dev = -1, per_sm = 1;
  int dev = 0;
  cudaGetDevice(&dev);
  if (attr_dev != dev) {
    const cudaError_t e =
        cudaFuncSetAttribute(k_fused<LOGN, BITS, FP64>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    per_sm = ctas_per_sm(k_fused<LOGN, BITS, FP64>, PL::THREADS, smem, PL::TCOLS);
    attr_dev = dev;
  }
  int eff = per_sm;
  if (a.cap1 > 0 && a.cap1 < eff) eff = a.cap1;
  if (a.cap2 > 0 && a.cap2 < eff) eff = a.cap2;
  long long slots = (long long)eff * a.num_sms / a.n_fpair;
  const long long need = ((long long)a.nseg + PL::T - 1) / PL::T;
  if (slots > need) slots = need;
  if (slots < 1) slots = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(slots * a.n_fpair));
  cfg.blockDim = dim3(PL::THREADS);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = pdl ? 1 : 0;
  return cudaLaunchKernelEx(&cfg, k_fused<LOGN, BITS, FP64>, a);
}

template <int LOGN, int BITS>
static cudaError_t launch_fused(const BatchArgs& a, cudaStream_t st, bool pdl) {
  return a.fp64 ? launch_fused_acc<LOGN, BITS, true>(a, st, pdl) : launch_fused_acc<LOGN, BITS, false>(a, st, pdl);
}

template <int LOGN>
cudaError_t run_fused(const BatchArgs& a, cudaStream_t st, bool pdl) {
  if (a.nseg <= 0) return cudaSuccess;
  switch (a.bits) {
    case 1: return launch_fused<LOGN, 1>(a, st, pdl);
    case 2: return launch_fused<LOGN, 2>(a, st, pdl);
    case 4: return launch_fused<LOGN, 4>(a, st, pdl);
    case 8: return launch_fused<LOGN, 8>(a, st, pdl);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace polaris

#define POLARIS_INSTANTIATE_FUSED(LOGN) \
  template cudaError_t polaris::run_fused<LOGN>(const polaris::BatchArgs&, cudaStream_t, bool);
