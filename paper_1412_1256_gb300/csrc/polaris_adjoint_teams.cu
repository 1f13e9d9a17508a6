// Leakage calibration: the forward pass at 2^9 to 2^12 when there are more segments than SMs: 512 threads as teams of T,
// one segment each.  The CTA's group is the same (segments b, b + G, ..., one CTA per SM), its teams take
// consecutive segments of it, and their products, through shared memory, are added in that order, one
// chain per bin and quantity in registers: the partial sums are those of k_adjs_forward, to the bit.
// That kernel left a CTA of 32 threads alone on an SM at 512 points.  With as many segments as CTAs, or
// fewer, the teams would have nothing to do.  Whole steps, before and
// after: 20000 x 2^9 (2 bits) 200 -> 119 us, 5000 x 2^10 81 -> 69, 3000 x 2^11 (2 bits) 85 -> 77, 2000 x
// 2^12 (1 bit) 104 -> 103 (two teams).
#include "polaris_adjoint_sized.cuh"

namespace polaris {

template <int LOGN>
struct AdjTeams {
  using PL = AdjPlan<LOGN>;
  static constexpr int THREADS = 512, TEAMS = THREADS / PL::T, NC = 4 * PL::NBIN;
  static constexpr int CH = (NC + THREADS - 1) / THREADS;  // chains per thread
  static constexpr size_t smem(int bits) {
    return (size_t)(TEAMS * PL::DATA + PL::NTAB + 1) * sizeof(float2) + (size_t)TEAMS * (NC * 4 + 2 * PL::N * bits / 8);
  }
  static_assert(!PL::FLY && smem(8) <= 227 * 1024, "shared memory");
};

template <int LOGN, int BITS>
__global__ void __launch_bounds__(AdjTeams<LOGN>::THREADS, 1) k_adjs_teams(AdjArgs a) {
  using PL = AdjPlan<LOGN>;
  using TM = AdjTeams<LOGN>;
  constexpr int N = PL::N, T = PL::T, W = adjs_words<LOGN, BITS>();
  extern __shared__ __align__(16) float2 zs[];
  const int team = threadIdx.x / T, tid = threadIdx.x % T;
  float2* z = zs + team * PL::DATA;
  float2* tws = zs + TM::TEAMS * PL::DATA;
  float* prods = reinterpret_cast<float*>(tws + PL::NTAB + 1);  // (NTAB is odd)
  uint32_t* raw = reinterpret_cast<uint32_t*>(prods + TM::TEAMS * TM::NC) + team * 2 * W;
  for (int i = threadIdx.x; i < PL::NTAB; i += TM::THREADS) tws[i] = __ldg(a.tw + i);
  const float2 wt[PL::RW] = {};  // (no last pass with twiddles of its own)
  float acc[TM::CH];
  sfor<0, TM::CH>([&](auto c_) { acc[decltype(c_)::value] = 0.f; });
  auto segments = [&](long long s0) -> int {  // of the group, from s0 on, that the teams take
    const long long left = (a.nseg - 1 - s0) / a.grid + 1;
    return left < TM::TEAMS ? (int)left : TM::TEAMS;
  };
  auto fetch = [&](long long s0) {  // (idle teams: the first segment again)
    adjs_fetch<LOGN, BITS>(a, raw, s0 + (long long)(team < segments(s0) ? team : 0) * a.grid, tid);
  };
  const long long step = (long long)TM::TEAMS * a.grid;
  pdl_wait();  // (dependent launch: the inputs and the partials may be touched from here on)
  fetch(blockIdx.x);
#pragma unroll 1
  for (long long s0 = blockIdx.x; s0 < a.nseg; s0 += step) {
    float2 u[PL::PPT];
    cp_async_wait_all();
    __syncthreads();
    adjs_load<LOGN, BITS>(a.window, raw, raw + W, u, tid);
    adjs_fft<LOGN>(u, z, tws, wt, tid);  // (its first barrier: all have read the words)
    if (s0 + step < a.nseg) fetch(s0 + step);
    adjs_store_upper<LOGN>(u, z, tid);
    const float2* zm = z + apad(N - tid);
    float4* prod = reinterpret_cast<float4*>(prods + team * TM::NC);
    sfor<0, PL::BPT>([&](auto i_) {
      constexpr int i = decltype(i_)::value;
      if (i < PL::BPT - 1 || tid == 0) {  // (i = BPT - 1: bin N/2, its own mirror)
        const float2 Zk = u[i];
        float2 Zm;
        if constexpr (i == PL::BPT - 1) Zm = c_conj(Zk);
        else if constexpr (i == 0) Zm = c_conj(tid == 0 ? Zk : zm[0]);
        else Zm = c_conj(zm[-apad_c<T * i>()]);
        const float2 X = make_float2(0.5f * (Zk.x + Zm.x), 0.5f * (Zk.y + Zm.y));
        const float2 Y = make_float2(0.5f * (Zk.y - Zm.y), -0.5f * (Zk.x - Zm.x));
        prod[tid + T * i] = make_float4(fmaf(X.x, X.x, X.y * X.y), fmaf(Y.x, Y.x, Y.y * Y.y),
                                        fmaf(X.x, Y.x, X.y * Y.y), fmaf(X.y, Y.x, -X.x * Y.y));
      }
    });
    __syncthreads();
    const int n = segments(s0);
    sfor<0, TM::CH>([&](auto c_) {
      constexpr int c = decltype(c_)::value;
      const int i = threadIdx.x + c * TM::THREADS;
      if (c < TM::CH - 1 || i < TM::NC)
        for (int j = 0; j < n; ++j) acc[c] += prods[j * TM::NC + i];
    });
  }
  float* part = reinterpret_cast<float*>(a.part + (size_t)blockIdx.x * PL::NBIN);
  sfor<0, TM::CH>([&](auto c_) {
    constexpr int c = decltype(c_)::value;
    const int i = threadIdx.x + c * TM::THREADS;
    if (c < TM::CH - 1 || i < TM::NC) part[i] = acc[c];
  });
}

template <int LOGN, int BITS>
static cudaError_t teams_call(const AdjArgs* a, cudaStream_t st) {  // (null: the kernel's shared-memory limit)
  using TM = AdjTeams<LOGN>;
  if (!a)
    return cudaFuncSetAttribute(k_adjs_teams<LOGN, BITS>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)TM::smem(BITS));
  return launch_dependent(k_adjs_teams<LOGN, BITS>, a->grid, TM::THREADS, TM::smem(BITS), st, *a);
}
template <int LOGN>
static cudaError_t teams_bits(int bits, const AdjArgs* a, cudaStream_t st) {
  switch (bits) {
    case 1: return teams_call<LOGN, 1>(a, st);
    case 2: return teams_call<LOGN, 2>(a, st);
    case 4: return teams_call<LOGN, 4>(a, st);
    default: return teams_call<LOGN, 8>(a, st);
  }
}
static cudaError_t teams_any(int log2n, int bits, const AdjArgs* a, cudaStream_t st) {
  switch (log2n) {
    case 9: return teams_bits<9>(bits, a, st);
    case 10: return teams_bits<10>(bits, a, st);
    case 11: return teams_bits<11>(bits, a, st);
    case 12: return teams_bits<12>(bits, a, st);
    default: return cudaErrorInvalidValue;
  }
}

cudaError_t adj_teams_prepare(int log2n, int bits) { return teams_any(log2n, bits, nullptr, nullptr); }
cudaError_t adj_teams_launch(int log2n, int bits, const AdjArgs& a, cudaStream_t st) {
  return teams_any(log2n, bits, &a, st);
}

}  // namespace polaris
