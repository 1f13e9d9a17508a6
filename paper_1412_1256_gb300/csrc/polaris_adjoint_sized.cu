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
// Whole steps, before and after (8-bit, with k_adjs_teams where it runs): 256 x 2^14 94.7 -> 66.0 us,
// 700 x 2^13 112 -> 82, 5000 x 2^10 177 -> 69; 2000 x 2^12 (1 bit) 148 -> 103, 20000 x 2^9 (2 bits)
// 463 -> 119.
#include "polaris_adjoint_sized.cuh"

namespace polaris {

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
  if (e == cudaSuccess && LOGN <= kAdjTeamsMax) e = adj_teams_prepare(LOGN, BITS);
  return e;
}

template <int LOGN, int BITS>
static cudaError_t adjs_launch(bool window_pass, const AdjArgs& a, cudaStream_t st) {
  using PL = AdjPlan<LOGN>;
  if (window_pass) return launch_dependent(k_adjs_window<LOGN, BITS>, a.grid, PL::T, PL::SMEM, st, a);
  if (LOGN <= kAdjTeamsMax && a.nseg > a.grid) return adj_teams_launch(LOGN, BITS, a, st);
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
