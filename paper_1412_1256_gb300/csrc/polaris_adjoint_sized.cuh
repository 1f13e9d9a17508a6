// Leakage calibration: what the size-specialised segment kernels share (polaris_adjoint_sized.cu, whose
// head describes them, and polaris_adjoint_teams.cu): plan, transform passes, samples.
#pragma once

#include <cuda_runtime.h>

#include "polaris_adjoint.cuh"
#include "polaris_kernels.cuh"  // tensor-memory helpers

namespace polaris {

template <int LOGN>
struct AdjPlan {
  static constexpr int N = 1 << LOGN, PPT = LOGN >= 14 ? 32 : 16, T = N / PPT, WARPS = T / 32, NBIN = N / 2 + 1;
  static constexpr int BPT = PPT / 2 + 1;  // bins per thread: k = t + T i (i < PPT/2), and N/2 for t = 0
  static constexpr int F = LOGN / 4, REM = LOGN % 4;     // F radix-16 passes, then one of radix 2^REM
  static constexpr int NS_LAST = 1 << (4 * F);           // Ns of that last pass
  static constexpr bool FLY = REM > 0 && NS_LAST > 256;  // its twiddles formed in registers
  static constexpr int RW = (REM > 0 ? (1 << REM) : 2) - 1;  // W_N^{r t}, r = 1 .. radix - 1, per thread
  static constexpr int NTAB = FLY ? NS_LAST - 1 : N - 1; // twiddle-table entries in shared memory
  static constexpr int DATA = adj_smem_points(N);
  static constexpr int SLOTS = WARPS >= 4 ? WARPS / 4 : 1;  // warps sharing a tensor-memory lane quadrant
  // tensor-memory columns per thread: forward, BPT bins x 4 sums in groups of 16 (four bins
  // each); window pass, the PPT taps of its sample groups
  static constexpr int FCOLS = 16 * ((4 * BPT + 15) / 16), WCOLS = PPT;
  static constexpr int TCOLS_F = pow2_at_least(SLOTS * FCOLS, 32), TCOLS_W = pow2_at_least(SLOTS * WCOLS, 32);
  static constexpr size_t SMEM = (size_t)(DATA + NTAB) * sizeof(float2) + 16;
  // the forward kernel also holds a segment's words of both IFs
  static constexpr size_t smem_forward(int bits) { return SMEM + (size_t)2 * N * bits / 8 + sizeof(float2); }
  // window kernel: CTAs that may share an SM by shared memory (228 KB, 1 KB of it per CTA the
  // system's) and tensor memory, eight at most: its registers are held to that many
  static constexpr int CTAS_SMEM = (int)((228 << 10) / (SMEM + 1024)), CTAS_TMEM = 512 / TCOLS_W;
  static constexpr int CTAS_MEM = CTAS_SMEM < CTAS_TMEM ? CTAS_SMEM : CTAS_TMEM;
  static constexpr int CTAS = CTAS_MEM < 8 ? CTAS_MEM : 8;
  static_assert(T % 32 == 0 && (N / 2) / T == PPT / 2, "whole warps, PPT/2 bins per thread below N/2");
  static_assert(TCOLS_F <= 512 && TCOLS_W <= 512, "tensor memory");
};

// One Stockham pass of radix R with Ns = NS points already combined: every j < N/R reads point
// j + r N/R (r < R), multiplies by W_{NS R}^{r (j mod NS)}, takes an R-point DFT and output r is
// point (j / NS) NS R + r NS + j mod NS.  A thread takes j = t + q T, so the first pass reads, and
// the last one writes, the points t + T i (i < PPT) of thread t: those stay in its registers (u[i]),
// and only the passes between exchange through z.  All of a pass's reads of z come before any write.
// Every compile-time part of the indices below (q T, r M, r NS) is a multiple of 16, so
// apad(x + c) = apad(x) + c + c/16: one padded base per lane and j, compile-time offsets.
template <int C>
__device__ __forceinline__ constexpr int apad_c() {
  static_assert(C % 16 == 0, "offset of whole 16-point groups");
  return C + C / 16;
}
template <int LOGN, int R, int NS>
__device__ __forceinline__ void adjs_pass(float2 (&u)[AdjPlan<LOGN>::PPT], float2* z, const float2* __restrict__ tws,
                                          const float2 (&wt)[AdjPlan<LOGN>::RW], int tid) {
  using PL = AdjPlan<LOGN>;
  constexpr int T = PL::T, JPT = PL::PPT / R, M = PL::N / R;
  constexpr bool FIRST = NS == 1, LAST = NS * R == PL::N;
  float2 v[JPT][R];
  const float2* zt = z + apad(tid);
  sfor<0, JPT>([&](auto q_) {
    constexpr int q = decltype(q_)::value;
    const int j = tid + q * T;
    const int k = j & (NS - 1);
    sfor<0, R>([&](auto r_) {
      constexpr int r = decltype(r_)::value;
      float2 x;
      if constexpr (FIRST) x = u[q + r * JPT];  // point j + r M = t + T (q + r JPT)
      else x = zt[apad_c<q * T + r * M>()];
      if constexpr (NS > 1 && r > 0) {
        if constexpr (NS <= 256) {
          x = cmul(x, tws[r * NS + k - 1]);
        } else {  // the last pass: k = j, W_N^{r j} = W_N^{r t} W_PPT^{r q} (T = N/PPT)
          constexpr int e = (r * q) % PL::PPT;
          float2 w = wt[r - 1];
          if constexpr (e != 0) {
            constexpr ct::CS cs = ct::cossin2pi(e, PL::PPT);
            w = cmul(w, make_float2((float)cs.c, (float)(-cs.s)));
          }
          x = cmul(x, w);
        }
      }
      v[q][ct::bitrev(r, R)] = x;
    });
  });
  if constexpr (FIRST) sfor<0, JPT>([&](auto q_) { dit<R>(v[decltype(q_)::value]); });
  if constexpr (!LAST) __syncthreads();  // (first pass: z's readers before this transform are done)
  sfor<0, JPT>([&](auto q_) {
    constexpr int q = decltype(q_)::value;
    const int j = tid + q * T;
    if constexpr (!FIRST) dit<R>(v[q]);
    if constexpr (FIRST) {  // base = 16 j, outputs r < 16: apad(16 j + r) = 17 j + r
      sfor<0, R>([&](auto r_) {
        constexpr int r = decltype(r_)::value;
        z[17 * j + r] = v[q][r];
      });
    } else if constexpr (LAST) {  // point j + r NS = t + T (q + r JPT)
      sfor<0, R>([&](auto r_) {
        constexpr int r = decltype(r_)::value;
        u[q + r * JPT] = v[q][r];
      });
    } else {
      const int k = j & (NS - 1);
      float2* zb = z + apad((j - k) * R + k);
      sfor<0, R>([&](auto r_) {
        constexpr int r = decltype(r_)::value;
        zb[apad_c<r * NS>()] = v[q][r];  // z[apad(base + r NS)]
      });
    }
  });
  if constexpr (!LAST) __syncthreads();
}

// forward DFT of the N points u[i] = point t + T i of the CTA's threads t, in place; a barrier
// before the first write of z, none after the last read of it
template <int LOGN>
__device__ __forceinline__ void adjs_fft(float2 (&u)[AdjPlan<LOGN>::PPT], float2* z, const float2* __restrict__ tws,
                                         const float2 (&wt)[AdjPlan<LOGN>::RW], int tid) {
  using PL = AdjPlan<LOGN>;
  sfor<0, PL::F>([&](auto p_) { adjs_pass<LOGN, 16, (1 << (4 * decltype(p_)::value))>(u, z, tws, wt, tid); });
  if constexpr (PL::REM > 0) adjs_pass<LOGN, (1 << PL::REM), PL::NS_LAST>(u, z, tws, wt, tid);
}

// Points t + T i and N - (t + T i), i < PPT/2, meet in thread t: every thread puts its upper half
// (i >= PPT/2) into z, where mirror point i of thread t is zm[-apad_c<T i>()], zm = z + apad(N - t)
// (only thread 0's i = 0 is its own mirror).  Barriers before and after.
template <int LOGN>
__device__ __forceinline__ void adjs_store_upper(const float2 (&u)[AdjPlan<LOGN>::PPT], float2* z, int tid) {
  using PL = AdjPlan<LOGN>;
  float2* zt = z + apad(tid);
  __syncthreads();  // the last pass's reads of z
  sfor<PL::PPT / 2, PL::PPT>([&](auto i_) {
    constexpr int i = decltype(i_)::value;
    zt[apad_c<PL::T * i>()] = u[i];
  });
  __syncthreads();
}

// A thread's samples t + T i of one segment, from global or shared memory (seg: the segment's
// words): a warp's loads are 32 consecutive codes.  Codes below 8 bits sit at the same place of
// every word the thread reads (T is a multiple of the samples per word): the word is rotated so
// that the code starts at bit 1.  (Ordinary loads, here and of the window and the matrix: a
// read-only one could be moved up over the wait for the kernel before.)
template <int LOGN, int BITS>
struct AdjSamples {
  static constexpr int SPW = 32 / BITS;
  const uint32_t* p;
  uint32_t rot;
  __device__ __forceinline__ AdjSamples(const uint32_t* seg, int tid) {
    if constexpr (BITS == 8) p = reinterpret_cast<const uint32_t*>(reinterpret_cast<const unsigned char*>(seg) + tid);
    else p = seg + tid / SPW;
    rot = (uint32_t)(tid % SPW) * BITS - 1u;
  }
  template <int I>
  __device__ __forceinline__ float level() const {
    constexpr int off = AdjPlan<LOGN>::T * I;
    static_assert(off % SPW == 0, "whole words");
    if constexpr (BITS == 8) {  // 2^23 + (c ^ 0x80) - 2^23 - 128
      const uint32_t c = reinterpret_cast<const unsigned char*>(p)[off];
      return __uint_as_float(c ^ 0x4B000080u) - 8388736.0f;
    } else {  // (2^23 + 2c) - (2^23 + 2^b - 1)
      const uint32_t w = p[off / SPW];
      return __uint_as_float(and_or(__funnelshift_r(w, w, rot), ((1u << BITS) - 1u) << 1, 0x4B000000u)) -
             (8388608.0f + (float)((1 << BITS) - 1));
    }
  }
};

// words of a segment of one IF
template <int LOGN, int BITS>
__device__ __forceinline__ constexpr int adjs_words() { return (1 << LOGN) * BITS / 32; }

// u[i] = w[n] (x[n] + i y[n]), n = t + T i, of the segment whose words are at x and y
template <int LOGN, int BITS>
__device__ __forceinline__ void adjs_load(const float* window, const uint32_t* x, const uint32_t* y,
                                          float2 (&u)[AdjPlan<LOGN>::PPT], int tid) {
  using PL = AdjPlan<LOGN>;
  const AdjSamples<LOGN, BITS> xs(x, tid), ys(y, tid);
  const float* wp = window + tid;
  sfor<0, PL::PPT>([&](auto i_) {
    constexpr int i = decltype(i_)::value;
    const float w = wp[PL::T * i];
    u[i] = make_float2(w * xs.template level<i>(), w * ys.template level<i>());
  });
}

// both IFs' words of segment s into shared memory ([IF][words], 16-byte chunks; one copy group)
template <int LOGN, int BITS>
__device__ __forceinline__ void adjs_fetch(const AdjArgs& a, uint32_t* raw, long long s, int tid) {
  constexpr int W = adjs_words<LOGN, BITS>();
  static_assert(W % 4 == 0, "whole chunks");
  const uint32_t dst = smem_addr(raw);
  for (int c = tid; c < 2 * (W / 4); c += AdjPlan<LOGN>::T) {
    const int f = c >= W / 4;
    cp_async16(dst + 16u * (uint32_t)c, a.in[f] + s * W + 4 * (c - f * (W / 4)));
  }
  cp_async_commit();
}

}  // namespace polaris
