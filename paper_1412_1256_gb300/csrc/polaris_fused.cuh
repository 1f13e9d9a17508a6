// The whole hot path of the small transforms (N = 2^10 .. 2^12) in one kernel: data translation,
// window, segment FFT, correlation and integration (Fig. 2 caption), with the pair-segment in
// registers and shared memory from its packed words to its accumulators.
//
//   k_fused  a team of W = N/1024 warps takes a range of segments of one FFT pair, one segment
//            at a time, 32 points per lane.  N = R B (row a, column b, n = B a + b; bin
//            k = c + R d): lane b runs the R-point DFT over its column's rows, multiplies by
//            W_N^{b c} (tensor memory), the team exchanges [c][b] through shared memory once,
//            and lane c runs the B-point DFT.  R and B are 32 or 64: a 64-point DFT is split over
//            two lanes by the parity of the output index (x_i +- x_{i+32}, the odd half turned by
//            W_64^i), so that every lane holds 32 points throughout.
//            Lane c's bin c + R d and its mirror (in the lane of column R - c, which sits in the
//            same warp) meet by one shuffle per component; |X|^2, |Y|^2 and X conj(Y) (as in
//            k_phase2) accumulate in tensor memory over the range.  At the end the CTA's teams
//            are summed in shared memory and added once to the integration accumulators, which
//            hold the bins in natural order.
//
// What bounds it: about 40 (1024, 2048 points) and 46 (4096) instructions per complex point, against
// 64 of the two-phase path of the larger sizes, which these sizes took before and which sends
// every point through a slab in L2.  Measured against that path (GB300): 4 pairs of 1-bit IFs,
// 2441 segments of 2048 points, 41 instead of 31 + 54 us of kernel time (2.05 us per million
// complex points); 64 int8 Hann segments of 1024 points, a whole pass 14.4 (host-bound) instead of
// 28.7 us; at 4096 points 86 segments of two 4-bit pairs take 10.3 instead of 5.8 + 10.3 us.
// Sizes: 2^13 and up would split a transform over more than two lanes per output column (or keep
// more than 32 points per lane) and stay with the two phases; below 2^10 likewise.
#pragma once
#include "polaris_codes.cuh"
#include "polaris_kernels.cuh"

namespace polaris {

template <int LOGN>
struct FusedPlan {
  static constexpr int N = 1 << LOGN, W = N / 1024;     // warps per team
  static constexpr int THREADS = 256, WARPS = THREADS / 32, T = WARPS / W;  // teams per CTA
  static constexpr int B = 1 << fused_log_b(LOGN), R = N / B;
  static constexpr int HA = R / 32, HB = B / 32;        // lanes per R-point, B-point DFT
  static constexpr int PITCH = B + 1;                   // [c][b] rows: consecutive c on distinct bank pairs
  static constexpr int REGION = R * PITCH;              // float2 per team
  static constexpr int TCOLS = (WARPS / 4) * 128;       // 64 accumulator and 64 twiddle columns per lane
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
    // packed words as they arrive, WPR words of padding per block row: the lanes' (word, block
    // row) then fall on consecutive banks
    static constexpr int RAWBLK = (SPW + 1) * WPR, RAW = BR * RAWBLK;
    // transposed words: BR words per column, VL of them side by side for one vector load;
    // column b = w SPW + c at place c WPR + w, so that the writers' lanes are consecutive
    static constexpr int VW = BR, VL = VW < 4 ? VW : 4;
    static constexpr int SLAB = (B + WPR) * VL, TR = (VW / VL) * SLAB;
    static constexpr size_t TEAM = sizeof(float2) * REGION + 4 * (size_t)G * (RAW + TR);
    static constexpr size_t SMEM = T * TEAM + 16 * T + 16;  // + extra bin per team, TMEM slot
    static_assert((G * RAW) % 4 == 0 && SLAB % VL == 0 && TR % VL == 0 && TEAM % 16 == 0, "vector loads aligned");
    static_assert(2 * (SMEM + 1024) <= 233472, "two CTAs per SM");
  };
  static_assert(REGION * sizeof(float2) % 16 == 0 && REGION * 8 >= 16 * (N / 2), "region holds the team's sums");
};

template <int W>
__device__ __forceinline__ void team_sync(int team) {
  if constexpr (W == 1) __syncwarp();
  else asm volatile("bar.sync %0, %1;\n" ::"r"(1 + team), "r"(32 * W) : "memory");
}

// x e^{-2 pi i J / 64}, J compile-time (the butterflies' cosine-factored form)
template <int J>
__device__ __forceinline__ float2 turn64(float2 x) {
  constexpr ct::CS cs = ct::cossin2pi(J, 64);
  constexpr double wr = cs.c, wi = -cs.s;
  if constexpr (J == 0) return x;
  else if constexpr (J == 16) return make_float2(x.y, -x.x);
  else if constexpr (ct::dabs(wr) >= ct::dabs(wi)) {
    constexpr float r = (float)(wi / wr), sc = (float)wr;
    const float2 u = __ffma2_rn(make_float2(x.y, x.x), make_float2(-r, r), x);
    return __fmul2_rn(u, make_float2(sc, sc));
  } else {
    constexpr float r = (float)(wr / wi), sc = (float)wi;
    const float2 v = __ffma2_rn(x, make_float2(-r, r), make_float2(x.y, x.x));
    return __fmul2_rn(v, make_float2(-sc, sc));
  }
}

template <int LOGN, int BITS>
__global__ void __launch_bounds__(256, 2) k_fused(BatchArgs a) {
  using PL = FusedPlan<LOGN>;
  using IN = typename PL::template In<BITS>;
  constexpr int W = PL::W, T = PL::T, B = PL::B, R = PL::R, HA = PL::HA, HB = PL::HB, PITCH = PL::PITCH;
  constexpr int SPW = IN::SPW, WPR = IN::WPR, VL = IN::VL, G = IN::G, TL = 32 * W;
  extern __shared__ __align__(16) unsigned char smf[];
  const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0), lane = tid & 31;
  const int team = warp / W, wt = warp % W, tl = wt * 32 + lane;  // team, warp and lane inside it
  unsigned char* mine = smf + team * IN::TEAM;
  float2* region = reinterpret_cast<float2*>(mine);
  uint32_t* raw = reinterpret_cast<uint32_t*>(mine + sizeof(float2) * PL::REGION);
  uint32_t* tr = raw + G * IN::RAW;
  float4* xbin = reinterpret_cast<float4*>(smf + T * IN::TEAM);
  uint32_t* tslot = reinterpret_cast<uint32_t*>(xbin + T);

  // lane roles: step A column ba and output parity ha (the same for a whole warp); step B column
  // cb (unit u: column u, or its mirror R - u; unit 0: columns 0 and R/2) and output parity hb
  const int ba = tl % B, ha = __shfl_sync(0xffffffffu, tl / B, 0);
  const int hb = HB == 2 ? (lane >> 3) & 1 : 0, mir = lane >> 4;
  const int u = HB == 2 ? 8 * wt + (lane & 7) : lane & 15;
  const int cb = u == 0 ? (mir ? R / 2 : 0) : (mir ? R - u : u);
  // the lane whose output 31 - i is the mirror of this lane's output i; column 0's even outputs
  // mirror onto themselves (output (32 - i) mod 32 of the lane itself)
  const int partner = u == 0 ? (mir == 0 || HB == 1 ? lane : lane ^ 8) : (HB == 2 ? lane ^ 24 : lane ^ 16);
  const bool self = cb == 0 && hb == 0;

  const uint32_t tbase = __shfl_sync(0xffffffffu, cta_tmem_begin<PL::TCOLS>(tslot, warp), 0);
  const uint32_t t_acc = tbase + ((uint32_t)(32 * (warp & 3)) << 16) + (uint32_t)((warp >> 2) * 128);
  const uint32_t t_tw = t_acc + 64;
  sfor<0, 4>([&](auto c_) {
    constexpr int cc = decltype(c_)::value;
    float z16[16], w16[16];
    sfor<0, 16>([&](auto k_) { z16[decltype(k_)::value] = 0.f; });
    tmem_st16(t_acc + 16 * cc, z16);
    sfor<0, 8>([&](auto k_) {  // W_N^{ba c}, c = HA c' + ha
      constexpr int k = decltype(k_)::value;
      const float2 w = __ldg(a.tw + (HA * (8 * cc + k) + ha) * B + ba);
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
        const uint32_t o = 4u * (uint32_t)(j + (j / (SPW * WPR)) * WPR);
        if (in_bounds(a.err, w0 + j, wext)) {
          cp_async4(dst + o, pa + j);
          cp_async4(dst + o + 4u * (uint32_t)(IN::RAW / 2), pb + j);
        }
      });
    }
    cp_async_commit();
  };

  float extra[4] = {0.f, 0.f, 0.f, 0.f};
  const float sgn_b = hb ? -1.f : 1.f;
  if (s_begin < s_end) issue(s_begin);
#pragma unroll 1
  for (int s0 = s_begin; s0 < s_end; s0 += G) {
    const int cnt = min(G, s_end - s0);
    cp_async_wait_all();
    team_sync<W>(team);  // the words are staged; the last group's transposed words have been read
    // codes transposed, block by block: SPW words down a word column of one block row
#pragma unroll 1
    for (int k = tl; k < cnt * IN::NB; k += TL) {
      const int w = k % WPR, br = (k / WPR) % IN::BR, g = k / IN::NB;
      const uint32_t* src = raw + g * IN::RAW + br * IN::RAWBLK + w;
      uint32_t x[SPW];
      sfor<0, SPW>([&](auto i_) { x[decltype(i_)::value] = src[decltype(i_)::value * WPR]; });
      transpose_codes<BITS>(x);
      uint32_t* dst = tr + g * IN::TR + (br / VL) * IN::SLAB + w * VL + br % VL;
      sfor<0, SPW>([&](auto c_) { dst[decltype(c_)::value * WPR * VL] = stored_codes<BITS>(x[decltype(c_)::value]); });
    }
    team_sync<W>(team);
    if (s0 + G < s_end) issue(s0 + G);
#pragma unroll 1
    for (int g = 0; g < cnt; ++g) {
      // step A: decode column ba, window, R-point DFT
      float2 v[32];
      uint32_t cw[IN::VW];
      const uint32_t* col = tr + g * IN::TR + ((ba % SPW) * WPR + ba / SPW) * VL;
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
      auto rows = [&](auto hb_, auto tp_) {
        constexpr bool HBP = decltype(hb_)::value, TP = decltype(tp_)::value;
        const float4* tp = reinterpret_cast<const float4*>(a.taps) + ba;
        float4 w4[HA];
        auto sample = [&](auto t_, auto h_) {
          constexpr int t = decltype(t_)::value, h = decltype(h_)::value;
          float2 z = code_pair<BITS, t % SPW>(cw[t / SPW], cw[IN::VW / 2 + t / SPW]);
          if constexpr (!HBP) z.y = 0.f;
          if constexpr (TP) {
            if constexpr (t % 4 == 0) w4[h] = __ldg(tp + (t / 4) * B);
            const float x = t % 4 == 0 ? w4[h].x : t % 4 == 1 ? w4[h].y : t % 4 == 2 ? w4[h].z : w4[h].w;
            z = __fmul2_rn(z, make_float2(x, x));
          }
          return z;
        };
        sfor<0, 32>([&](auto t_) {
          constexpr int t = decltype(t_)::value;
          const float2 z = sample(t_, std::integral_constant<int, 0>{});
          if constexpr (HA == 1) {
            v[ct::bitrev(t, 32)] = z;
          } else {
            const float2 y = sample(std::integral_constant<int, t + 32>{}, std::integral_constant<int, 1>{});
            const float sg = ha ? -1.f : 1.f;
            v[ct::bitrev(t, 32)] = __ffma2_rn(y, make_float2(sg, sg), z);
          }
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
      if constexpr (HA == 2) {
        if (ha) {
          sfor<0, 32>([&](auto t_) {
            constexpr int t = decltype(t_)::value;
            v[ct::bitrev(t, 32)] = turn64<t>(v[ct::bitrev(t, 32)]);
          });
        }
      }
      dit<32>(v);
      sfor<0, 4>([&](auto c_) {
        constexpr int cc = decltype(c_)::value;
        float w16[16];
        tmem_ld16(t_tw + 16 * cc, w16);
        tmem_wait_ld();
        sfor<0, 8>([&](auto k_) {
          constexpr int k = decltype(k_)::value, i = 8 * cc + k;
          if constexpr (HA == 2 || i > 0) v[i] = cmul(v[i], make_float2(w16[2 * k], w16[2 * k + 1]));
        });
      });
      team_sync<W>(team);  // the previous segment's exchange has been read
      sfor<0, 32>([&](auto i_) {
        constexpr int i = decltype(i_)::value;
        region[(HA * i + ha) * PITCH + ba] = v[i];
      });
      team_sync<W>(team);
      // step B: B-point DFT of column cb
      const float2* src = region + cb * PITCH;
      sfor<0, 32>([&](auto i_) {
        constexpr int i = decltype(i_)::value;
        if constexpr (HB == 1) {
          v[ct::bitrev(i, 32)] = src[i];
        } else {
          float2 z = __ffma2_rn(src[i + 32], make_float2(sgn_b, sgn_b), src[i]);
          const float2 zt = turn64<i>(z);
          z.x = hb ? zt.x : z.x;
          z.y = hb ? zt.y : z.y;
          v[ct::bitrev(i, 32)] = z;
        }
      });
      dit<32>(v);
      // correlate: this lane's bins are outputs i < 16 (d = HB i + hb), k = cb + R d < N/2
      sfor<0, 4>([&](auto c_) {
        constexpr int cc = decltype(c_)::value;
        float a16[16];
        tmem_ld16(t_acc + 16 * cc, a16);
        tmem_wait_ld();
        sfor<0, 4>([&](auto k_) {
          constexpr int k = decltype(k_)::value, i = 4 * cc + k;
          const float2 own = v[(32 - i) % 32];
          float2 z = make_float2(__shfl_sync(0xffffffffu, v[31 - i].x, partner),
                                 __shfl_sync(0xffffffffu, v[31 - i].y, partner));
          z.x = self ? own.x : z.x;
          z.y = self ? own.y : z.y;
          float(&q)[4] = *reinterpret_cast<float(*)[4]>(a16 + 4 * k);
          corr_acc(q, v[i], make_float2(z.x, -z.y));
        });
        tmem_st16(t_acc + 16 * cc, a16);
      });
      tmem_wait_st();
      if (self) corr_acc(extra, v[16], make_float2(v[16].x, -v[16].y));  // bin N/2, its own mirror
    }
  }
  pdl_trigger();
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
      sums[cb + R * (HB * i + hb)] = make_float4(a16[4 * k], a16[4 * k + 1], a16[4 * k + 2], a16[4 * k + 3]);
    });
  });
  if (self) xbin[team] = make_float4(extra[0], extra[1], extra[2], extra[3]);
  __syncthreads();
  const size_t base = ((size_t)(a.acc_copies > 1 ? slot % a.acc_copies : 0) * a.n_fpair + f) * (PL::N / 2 + 1);
  for (int k = tid; k <= PL::N / 2; k += PL::THREADS) {
    float4 t = make_float4(0.f, 0.f, 0.f, 0.f);
    for (int q = 0; q < T; ++q) {
      const float4 x = k == PL::N / 2 ? xbin[q] : reinterpret_cast<const float4*>(smf + q * IN::TEAM)[k];
      t = make_float4(t.x + x.x, t.y + x.y, t.z + x.z, t.w + x.w);
    }
    const size_t o = base + k;
    if (!in_bounds(a.err, (long long)o, a.acc_slots)) continue;
    if (!a.fp64) {
      atomicAdd(reinterpret_cast<float4*>(a.acc) + o, t);
    } else {
      double* op = reinterpret_cast<double*>(a.acc) + 4 * o;
      atomicAdd(op + 0, (double)t.x);
      atomicAdd(op + 1, (double)t.y);
      atomicAdd(op + 2, (double)t.z);
      atomicAdd(op + 3, (double)t.w);
    }
  }
  cta_tmem_end<PL::TCOLS>(tbase, warp);
}

// One launch per feed: CTAs in equal numbers per FFT pair, as many as fit and have a segment per
// team.
template <int LOGN, int BITS>
static cudaError_t launch_fused(const BatchArgs& a, cudaStream_t st, bool pdl) {
  using PL = FusedPlan<LOGN>;
  constexpr size_t smem = PL::template In<BITS>::SMEM;
  static int attr_dev = -1, per_sm = 1;
  int dev = 0;
  cudaGetDevice(&dev);
  if (attr_dev != dev) {
    const cudaError_t e =
        cudaFuncSetAttribute(k_fused<LOGN, BITS>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    per_sm = ctas_per_sm(k_fused<LOGN, BITS>, PL::THREADS, smem, PL::TCOLS);
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
  return cudaLaunchKernelEx(&cfg, k_fused<LOGN, BITS>, a);
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
