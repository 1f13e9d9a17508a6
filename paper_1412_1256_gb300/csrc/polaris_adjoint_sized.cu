// Leakage calibration: the segment kernels of the forward and window passes specialised per
// transform size N = 2^LOGN, kAdjSizedMin <= LOGN <= kAdjSizedMax, so that every index, pass
// and radix is a compile-time constant.  They compute what k_adj_forward and k_adj_window
// (polaris_adjoint.cu) compute (the forward pass with the same order of summation):
//   - one CTA of T = N/PPT threads per segment at a time, PPT points per thread (16; 32 at
//     N = 2^14, so that 512 threads of 128 registers hold them), radix-16 Stockham passes and
//     one pass of radix 2^(LOGN mod 4).  Thread t's points before the first and after the last
//     pass are t + T i, in registers: shared memory holds only what the passes between exchange
//     and the upper half of the spectrum (the mirror bins), 14 instead of 20 times the segment in
//     the window pass;
//   - samples and window taps are read as a warp's 32 consecutive ones; the forward kernel
//     copies the next segment's words to shared memory meanwhile (inputs and window 16-byte
//     aligned: the host routes other calls to the kernels for any N);
//   - the per-CTA partial sums over the CTA's segments (per bin in the forward pass, per tap
//     in the window pass) stay in tensor memory, used as per-thread storage, and reach global
//     memory once, at the end (instead of a read and a write per segment);
//   - the twiddles of the passes with Ns <= 256 are a shared-memory copy of the host's table
//     (exact FP64 values rounded once); the last pass of N >= 2^13 (Ns = 4096) forms
//     W_N^{r j}, j = t + q T, as W_N^{r t} (from the table, once per thread) times the
//     constant W_PPT^{r q}: one rounding of two correctly rounded factors.
// What bounds them: latency.  At 2^14 (one CTA of 16 warps per SM) a third of the shared-memory
// and a quarter of the issue slots are used, the warps wait for the window's and the samples'
// loads, the exchanges and the barriers; 256 segments on 152 SMs are two rounds, the second two
// thirds full.  Neither kernel releases its successor early: the blocks of k_adj_bins and
// k_adj_wsum would gather on the SMs that have no second segment (67.1 us a step instead of 66.0).
// Whole steps, before and after (8-bit): 256 x 2^14 94.7 -> 66.0 us, 700 x 2^13
// 112 -> 83, 5000 x 2^10 177 -> 81; 2000 x 2^12 (1 bit) 148 -> 104, 20000 x 2^9 (2 bit) 463 -> 200.
#include <cuda_runtime.h>

#include <algorithm>

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
    cp_async<16>(dst + 16u * (uint32_t)c, a.in[f] + s * W + 4 * (c - f * (W / 4)));
  }
  cp_async_commit();
}

// the set-up both kernels share: the twiddle table in shared memory, this thread's W_N^{r t}
// for a last pass formed in registers, and the CTA's tensor memory (this thread's COLS columns
// zeroed); returns the address of those columns
template <int LOGN, int TCOLS, int COLS>
__device__ __forceinline__ uint32_t adjs_setup(const AdjArgs& a, float2* tws, uint32_t* tslot,
                                               float2 (&wt)[AdjPlan<LOGN>::RW], uint32_t& tbase, int tid) {
  using PL = AdjPlan<LOGN>;
  const int warp = tid >> 5;
  for (int i = tid; i < PL::NTAB; i += PL::T) tws[i] = __ldg(a.tw + i);
  sfor<0, PL::RW>([&](auto r_) {  // W_N^{r t}: the table's entry r, k = t of the last pass
    constexpr int r = decltype(r_)::value + 1;
    wt[r - 1] = PL::FLY ? __ldg(a.tw + r * PL::NS_LAST + tid - 1) : make_float2(1.f, 0.f);
  });
  tbase = cta_tmem_begin<TCOLS>(tslot, warp);  // (its barrier also publishes the table)
  const uint32_t tacc = tbase + ((uint32_t)(32 * (warp & 3)) << 16) + (uint32_t)((warp >> 2) * COLS);
  float z16[16];
  sfor<0, 16>([&](auto i_) { z16[decltype(i_)::value] = 0.f; });
  sfor<0, COLS / 16>([&](auto c_) { tmem_st16(tacc + 16 * decltype(c_)::value, z16); });
  tmem_wait_st();
  return tacc;
}

template <int LOGN, int BITS>
__global__ void __launch_bounds__(AdjPlan<LOGN>::T) k_adjs_forward(AdjArgs a) {
  using PL = AdjPlan<LOGN>;
  constexpr int N = PL::N, T = PL::T, W = adjs_words<LOGN, BITS>();
  extern __shared__ __align__(16) float2 zs[];
  float2* z = zs;
  float2* tws = zs + PL::DATA;
  uint32_t* raw = reinterpret_cast<uint32_t*>(tws + PL::NTAB + 1);  // (NTAB is odd)
  uint32_t* tslot = raw + 2 * W;
  const int tid = threadIdx.x;
  float2 wt[PL::RW];
  uint32_t tbase;
  const uint32_t tacc = adjs_setup<LOGN, PL::TCOLS_F, PL::FCOLS>(a, tws, tslot, wt, tbase, tid);
  pdl_wait();  // (dependent launch: the inputs and the partials may be touched from here on)
  adjs_fetch<LOGN, BITS>(a, raw, blockIdx.x, tid);  // (a.grid <= a.nseg)
#pragma unroll 1
  for (long long s = blockIdx.x; s < a.nseg; s += a.grid) {
    float2 u[PL::PPT];
    cp_async_wait_all();
    __syncthreads();
    adjs_load<LOGN, BITS>(a.window, raw, raw + W, u, tid);
    adjs_fft<LOGN>(u, z, tws, wt, tid);  // (its first barrier: all have read the words)
    if (s + a.grid < a.nseg) adjs_fetch<LOGN, BITS>(a, raw, s + a.grid, tid);
    adjs_store_upper<LOGN>(u, z, tid);
    const float2* zm = z + apad(N - tid);
    // X = (Z[k] + conj Z[N-k]) / 2, Y = (Z[k] - conj Z[N-k]) / 2i; the sums of bin i of this
    // thread at columns 4 i .. 4 i + 3
    sfor<0, PL::FCOLS / 16>([&](auto c_) {
      constexpr int cc = decltype(c_)::value;
      float acc[16];
      tmem_ld16(tacc + 16 * cc, acc);
      tmem_wait_ld();
      sfor<0, 4>([&](auto i_) {
        constexpr int i = 4 * cc + decltype(i_)::value;
        if constexpr (i < PL::BPT) {
          if (i < PL::BPT - 1 || tid == 0) {  // (i = BPT - 1: bin N/2, its own mirror)
            const float2 Zk = u[i];
            float2 Zm;
            if constexpr (i == PL::BPT - 1) Zm = c_conj(Zk);
            else if constexpr (i == 0) Zm = c_conj(tid == 0 ? Zk : zm[0]);
            else Zm = c_conj(zm[-apad_c<T * i>()]);
            const float2 X = make_float2(0.5f * (Zk.x + Zm.x), 0.5f * (Zk.y + Zm.y));
            const float2 Y = make_float2(0.5f * (Zk.y - Zm.y), -0.5f * (Zk.x - Zm.x));
            constexpr int o = 4 * (i - 4 * cc);
            acc[o + 0] += fmaf(X.x, X.x, X.y * X.y);
            acc[o + 1] += fmaf(Y.x, Y.x, Y.y * Y.y);
            acc[o + 2] += fmaf(X.x, Y.x, X.y * Y.y);
            acc[o + 3] += fmaf(X.y, Y.x, -X.x * Y.y);
          }
        }
      });
      tmem_st16(tacc + 16 * cc, acc);
    });
    tmem_wait_st();
  }
  float4* part = a.part + (size_t)blockIdx.x * PL::NBIN;
  sfor<0, PL::FCOLS / 16>([&](auto c_) {
    constexpr int cc = decltype(c_)::value;
    float acc[16];
    tmem_ld16(tacc + 16 * cc, acc);
    tmem_wait_ld();
    sfor<0, 4>([&](auto i_) {
      constexpr int i = 4 * cc + decltype(i_)::value;
      if constexpr (i < PL::BPT) {
        if (i < PL::BPT - 1 || tid == 0) {
          const int k = i < PL::BPT - 1 ? tid + T * i : N / 2;
          constexpr int o = 4 * (i - 4 * cc);
          part[k] = make_float4(acc[o], acc[o + 1], acc[o + 2], acc[o + 3]);
        }
      }
    });
  });
  cta_tmem_end<PL::TCOLS_F>(tbase, tid >> 5);
}

template <int LOGN, int BITS>
__global__ void __launch_bounds__(AdjPlan<LOGN>::T, AdjPlan<LOGN>::CTAS) k_adjs_window(AdjArgs a) {
  using PL = AdjPlan<LOGN>;
  constexpr int N = PL::N, T = PL::T, W = adjs_words<LOGN, BITS>();
  extern __shared__ __align__(16) float2 zs[];
  float2* z = zs;
  float2* tws = zs + PL::DATA;
  uint32_t* tslot = reinterpret_cast<uint32_t*>(tws + PL::NTAB);
  const int tid = threadIdx.x;
  float2 wt[PL::RW];
  uint32_t tbase;
  const uint32_t tacc = adjs_setup<LOGN, PL::TCOLS_W, PL::WCOLS>(a, tws, tslot, wt, tbase, tid);
  // (dependent launch: the inputs, read before k_adj_bins started, are complete; its matrix is
  // not before the wait below)
#pragma unroll 1
  for (long long s = blockIdx.x; s < a.nseg; s += a.grid) {
    float2 u[PL::PPT];
    const uint32_t *x = a.in[0] + s * W, *y = a.in[1] + s * W;
    adjs_load<LOGN, BITS>(a.window, x, y, u, tid);
    adjs_fft<LOGN>(u, z, tws, wt, tid);
    adjs_store_upper<LOGN>(u, z, tid);
    if (s == blockIdx.x) pdl_wait();
    // G_X, G_Y per bin pair; u and z become conj of the Hermitian extension H of G_X + i G_Y
    // (the inverse transform is conj(DFT(conj H))).  Thread t owns bins k = t + T i and the slots
    // of their mirrors, so these are read and overwritten without a barrier.
    float2* zm = z + apad(N - tid);
    sfor<0, PL::PPT / 2>([&](auto i_) {
      constexpr int i = decltype(i_)::value;
      const float2 Zk = u[i];
      float2 Zm;
      if constexpr (i == 0) Zm = c_conj(tid == 0 ? Zk : zm[0]);
      else Zm = c_conj(zm[-apad_c<T * i>()]);
      float2 GX, GY;
      adj_bin_gradient(a.mat[tid + T * i], Zk, Zm, GX, GY);
      const float2 hx = make_float2(0.5f * GX.x, 0.5f * GX.y), hy = make_float2(0.5f * GY.x, 0.5f * GY.y);
      // H[k] = hx + i hy, H[N-k] = conj(hx) + i conj(hy); store their conjugates
      u[i] = make_float2(hx.x - hy.y, -(hx.y + hy.x));
      const float2 hm = make_float2(hx.x + hy.y, hx.y - hy.x);
      if constexpr (i == 0) {
        if (tid == 0) u[0] = make_float2(GX.x, -GY.x);  // H = Re G_X + i Re G_Y (likewise at N/2)
        else zm[0] = hm;
      } else {
        zm[-apad_c<T * i>()] = hm;
      }
    });
    if (tid == 0) {
      const float2 Zk = u[PL::PPT / 2];
      float2 GX, GY;
      adj_bin_gradient(a.mat[N / 2], Zk, c_conj(Zk), GX, GY);
      z[apad(N / 2)] = make_float2(GX.x, -GY.x);
    }
    __syncthreads();
    const float2* zt = z + apad(tid);
    sfor<PL::PPT / 2, PL::PPT>([&](auto i_) {
      constexpr int i = decltype(i_)::value;
      u[i] = zt[apad_c<T * i>()];
    });
    adjs_fft<LOGN>(u, z, tws, wt, tid);
    // h = conj(F): dL/dw[n] += x[n] Re h[n] + y[n] Im h[n] = x F.x - y F.y (column i: n = t + T i)
    const AdjSamples<LOGN, BITS> xs(x, tid), ys(y, tid);
    sfor<0, PL::PPT / 16>([&](auto h_) {
      constexpr int h = decltype(h_)::value;
      float acc[16];
      tmem_ld16(tacc + 16 * h, acc);
      tmem_wait_ld();
      sfor<0, 16>([&](auto j_) {
        constexpr int j = decltype(j_)::value, i = 16 * h + j;
        acc[j] += fmaf(xs.template level<i>(), u[i].x, -ys.template level<i>() * u[i].y);
      });
      tmem_st16(tacc + 16 * h, acc);
    });
    tmem_wait_st();
  }
  float* gpart = a.gpart + (size_t)blockIdx.x * N + tid;
  sfor<0, PL::PPT / 16>([&](auto h_) {
    constexpr int h = decltype(h_)::value;
    float acc[16];
    tmem_ld16(tacc + 16 * h, acc);
    tmem_wait_ld();
    sfor<0, 16>([&](auto j_) {
      constexpr int j = decltype(j_)::value;
      gpart[T * (16 * h + j)] = acc[j];
    });
  });
  cta_tmem_end<PL::TCOLS_W>(tbase, tid >> 5);
}

// ------------------------------------------------------------------------------------------
// host side
// ------------------------------------------------------------------------------------------
// Forward pass: one CTA per SM, because its grid sets the order in which a bin's segments are
// added.  (The runtime's occupancy query says one for any kernel that allocates tensor memory.)
// Window pass: as many as share an SM; at one, the sizes below 2^13 left most of it idle: 64
// threads at 1024 points.
template <int LOGN, int BITS>
static cudaError_t adjs_prepare(int* window_ctas) {
  using PL = AdjPlan<LOGN>;
  *window_ctas = PL::CTAS;
  cudaError_t e = cudaFuncSetAttribute(k_adjs_forward<LOGN, BITS>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)PL::smem_forward(BITS));
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(k_adjs_window<LOGN, BITS>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)PL::SMEM);
  return e;
}

template <int LOGN, int BITS>
static cudaError_t adjs_launch(bool window_pass, const AdjArgs& a, cudaStream_t st) {
  using PL = AdjPlan<LOGN>;
  if (window_pass) return launch_dependent(k_adjs_window<LOGN, BITS>, a.grid, PL::T, PL::SMEM, st, a);
  return launch_dependent(k_adjs_forward<LOGN, BITS>, a.grid, PL::T, PL::smem_forward(BITS), st, a);
}

template <int LOGN>
static cudaError_t adjs_dispatch(int bits, bool prepare, int* occ, bool window_pass, const AdjArgs* a,
                                 cudaStream_t st) {
  switch (bits) {
    case 1: return prepare ? adjs_prepare<LOGN, 1>(occ) : adjs_launch<LOGN, 1>(window_pass, *a, st);
    case 2: return prepare ? adjs_prepare<LOGN, 2>(occ) : adjs_launch<LOGN, 2>(window_pass, *a, st);
    case 4: return prepare ? adjs_prepare<LOGN, 4>(occ) : adjs_launch<LOGN, 4>(window_pass, *a, st);
    default: return prepare ? adjs_prepare<LOGN, 8>(occ) : adjs_launch<LOGN, 8>(window_pass, *a, st);
  }
}

static cudaError_t adjs_any(int log2n, int bits, bool prepare, int* occ, bool window_pass, const AdjArgs* a,
                            cudaStream_t st) {
  switch (log2n) {
    case 9: return adjs_dispatch<9>(bits, prepare, occ, window_pass, a, st);
    case 10: return adjs_dispatch<10>(bits, prepare, occ, window_pass, a, st);
    case 11: return adjs_dispatch<11>(bits, prepare, occ, window_pass, a, st);
    case 12: return adjs_dispatch<12>(bits, prepare, occ, window_pass, a, st);
    case 13: return adjs_dispatch<13>(bits, prepare, occ, window_pass, a, st);
    case 14: return adjs_dispatch<14>(bits, prepare, occ, window_pass, a, st);
    default: return cudaErrorInvalidValue;
  }
}

cudaError_t adj_sized_prepare(int log2n, int bits, int* window_ctas) {
  return adjs_any(log2n, bits, true, window_ctas, false, nullptr, nullptr);
}

cudaError_t adj_sized_launch(int log2n, int bits, bool window_pass, const AdjArgs& a, cudaStream_t st) {
  return adjs_any(log2n, bits, false, nullptr, window_pass, &a, st);
}

}  // namespace polaris
