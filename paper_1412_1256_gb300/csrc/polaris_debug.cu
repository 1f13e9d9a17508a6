// Bit-exactness check of the staged data translation (Fig. 2 caption: integer codes to
// floats).  From N = 2^13 up, the FFT kernel (k_fused at 2^13 and 2^14, k_phase1, k_phase1w from 2^18)
// stages packed words in shared memory, transposes their codes there and decodes each lane's rows
// from the transposed words (polaris_codes.cuh).  The kernels below stage in the same layout and
// transpose and decode through the same device functions, so the levels that are transformed can be
// compared with the oracle's decode bit for bit.
#include "polaris_fused.cuh"
#include "polaris_kernels.cuh"

namespace polaris {

template <int LOGN, int BITS, bool WIDE>
struct StagedPlan {
  using PL = Plan<LOGN>;
  using ST = typename PL::template Stage1<BITS>;
  static constexpr bool STAGED = ST::STAGED;
};
template <int LOGN, int BITS>
struct StagedPlan<LOGN, BITS, true> {
  using PL = WidePlan<LOGN>;
  using ST = typename PL::template Stage<BITS>;
  static constexpr bool STAGED = !(BITS == 1 && LOGN >= 19);  // (staged, but refused: what this check has always answered)
};

// One CTA per tile (segment s, first column b0): stage the tile's N1 rows of IF a (and IF b) in the
// chunks of RP words that they arrive in, transpose, then decode lane q1's rows t of column col ->
// sample n = s N + (q1 + Q1 t) N2 + b0 + col.
template <int LOGN, int BITS>
__global__ void __launch_bounds__(256) k_unpack_staged(const uint32_t* __restrict__ pa, const uint32_t* __restrict__ pb,
                                                       float* __restrict__ oa, float* __restrict__ ob) {
  using SP = StagedPlan<LOGN, BITS, (LOGN >= kWideMin)>;
  using PL = typename SP::PL;
  using ST = typename SP::ST;
  constexpr int N = PL::N, N1 = PL::N1, N2 = PL::N2, Q1 = PL::Q1, P = PL::P1, TILE = ST::TILE, RP = ST::RP;
  constexpr int SEGW = N * BITS / 32, ROWW = N2 * BITS / 32;  // words per segment, per row
  static_assert(ROWW % RP == 0 && RP % ST::WPR == 0, "whole tiles in a chunk, whole chunks in a row");
  extern __shared__ __align__(16) uint32_t stg[];
  uint32_t* tr = stg + ST::RAWW;
  constexpr int TPS = N2 / TILE;  // tiles per segment
  const int s = blockIdx.x / TPS, b0 = (blockIdx.x % TPS) * TILE, w0 = (b0 * BITS) / 32, x0 = w0 / RP * RP;
  const uint32_t* sa = pa + (size_t)s * SEGW + x0;
  const uint32_t* sbp = pb ? pb + (size_t)s * SEGW + x0 : nullptr;
  for (int k = threadIdx.x; k < N1 * RP; k += blockDim.x) {
    const int o = (k / RP) * ROWW + k % RP;
    stg[k] = sa[o];
    stg[N1 * RP + k] = sbp ? sbp[o] : sa[o];  // (IF a again without an IF b, as phase 1 stages it)
  }
  __syncthreads();
  for (int u = threadIdx.x; u < ST::UNITS; u += blockDim.x) {
    uint32_t x[ST::KB][32 / BITS];
    p1_unit_load<PL, ST, BITS>(stg + (w0 - x0), u, x);
    p1_unit_store<PL, ST, BITS>(tr, u, x);
  }
  __syncthreads();
  for (int e = threadIdx.x; e < Q1 * TILE; e += blockDim.x) {
    const int q1 = e / TILE, col = e % TILE;
    uint32_t codes[ST::BR];
    p1_lane_codes<PL, ST>(tr, q1, col, codes);
    sfor<0, P>([&](auto t_) {
      constexpr int t = decltype(t_)::value;
      const float2 z = sbp ? p1_level<PL, ST, BITS, true, t>(codes) : p1_level<PL, ST, BITS, false, t>(codes);
      const size_t n = (size_t)s * N + (size_t)(q1 + Q1 * t) * N2 + b0 + col;
      oa[n] = z.x;
      if (sbp) ob[n] = z.y;
    });
  }
}

// One CTA per segment, one team of k_fused: stage its words, transpose, then decode lane tl's rows t ->
// sample n = s N + B t + tl.
template <int LOGN, int BITS>
__global__ void __launch_bounds__(32 * FusedPlan<LOGN>::W)
    k_unpack_fused(const uint32_t* __restrict__ pa, const uint32_t* __restrict__ pb, float* __restrict__ oa,
                   float* __restrict__ ob) {
  using PL = FusedPlan<LOGN>;
  using IN = typename PL::template In<BITS>;
  constexpr int TL = 32 * PL::W;
  extern __shared__ __align__(16) uint32_t stg[];
  uint32_t* tr = stg + IN::RAW;
  const int tl = threadIdx.x;
  const size_t s = blockIdx.x;
  for (int j = tl; j < IN::NW; j += TL) {
    const uint32_t o = fused_raw_place<IN>(j);
    stg[o] = pa[s * IN::NW + j];
    stg[IN::RAW / 2 + o] = (pb ? pb : pa)[s * IN::NW + j];
  }
  __syncthreads();
  fused_transpose<IN, BITS, TL>(stg, tr, 1, tl);
  __syncthreads();
  uint32_t cw[IN::VW];
  fused_lane_codes<IN>(tr, 0, tl, cw);
  sfor<0, 32>([&](auto t_) {
    constexpr int t = decltype(t_)::value;
    const float2 z = pb ? fused_level<IN, BITS, true, t>(cw) : fused_level<IN, BITS, false, t>(cw);
    const size_t n = s * PL::N + (size_t)PL::B * t + tl;
    oa[n] = z.x;
    if (pb) ob[n] = z.y;
  });
}

template <int LOGN, int BITS>
static cudaError_t launch_unpack_staged_t(const uint32_t* pa, const uint32_t* pb, long long nseg, float* oa, float* ob,
                                          cudaStream_t st) {
  auto launch = [&](auto kernel, long long grid, int threads, size_t smem) {
    const cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    kernel<<<(unsigned)grid, threads, smem, st>>>(pa, pb, oa, ob);
    return cudaGetLastError();
  };
  if constexpr (is_fused(LOGN)) {
    using IN = typename FusedPlan<LOGN>::template In<BITS>;
    return launch(k_unpack_fused<LOGN, BITS>, nseg, 32 * FusedPlan<LOGN>::W, 4 * (size_t)(IN::RAW + IN::TR));
  } else {
    using SP = StagedPlan<LOGN, BITS, (LOGN >= kWideMin)>;
    using ST = typename SP::ST;
    if constexpr (!SP::STAGED) return cudaErrorInvalidValue;
    else
      return launch(k_unpack_staged<LOGN, BITS>, nseg * (SP::PL::N2 / ST::TILE), 256, 4 * (size_t)(ST::RAWW + ST::TRW));
  }
}

template <int LOGN>
static cudaError_t launch_unpack_staged_n(int bits, const uint32_t* pa, const uint32_t* pb, long long nseg, float* oa,
                                          float* ob, cudaStream_t st) {
  switch (bits) {
    case 1: return launch_unpack_staged_t<LOGN, 1>(pa, pb, nseg, oa, ob, st);
    case 2: return launch_unpack_staged_t<LOGN, 2>(pa, pb, nseg, oa, ob, st);
    case 4: return launch_unpack_staged_t<LOGN, 4>(pa, pb, nseg, oa, ob, st);
    case 8: return launch_unpack_staged_t<LOGN, 8>(pa, pb, nseg, oa, ob, st);
    default: return cudaErrorInvalidValue;
  }
}

template <int LOGN, int BITS>
static constexpr bool staged_t() {
  if constexpr (is_fused(LOGN)) return true;
  else return StagedPlan<LOGN, BITS, (LOGN >= kWideMin)>::STAGED;
}
template <int LOGN>
static constexpr bool staged_n(int bits) {
  return bits == 1 ? staged_t<LOGN, 1>() : bits == 2 ? staged_t<LOGN, 2>() : bits == 4 ? staged_t<LOGN, 4>()
                                                                            : staged_t<LOGN, 8>();
}

// true when this check takes the size and width
bool unpack_staged_takes(int logn, int bits) {
  switch (logn) {
#define POLARIS_ST(L) \
  case L: return staged_n<L>(bits);
    POLARIS_ST(13) POLARIS_ST(14) POLARIS_ST(15) POLARIS_ST(16) POLARIS_ST(17) POLARIS_ST(18) POLARIS_ST(19)
    POLARIS_ST(20)
#undef POLARIS_ST
    default: return false;
  }
}

// decode nseg whole segments of IF a (and IF b, may be null) through the staged decoder
cudaError_t launch_unpack_staged(int logn, int bits, const uint32_t* pa, const uint32_t* pb, long long nseg, float* oa,
                                 float* ob, cudaStream_t st) {
  switch (logn) {
#define POLARIS_US(L) \
  case L: return launch_unpack_staged_n<L>(bits, pa, pb, nseg, oa, ob, st);
    POLARIS_US(13) POLARIS_US(14) POLARIS_US(15) POLARIS_US(16) POLARIS_US(17) POLARIS_US(18) POLARIS_US(19)
    POLARIS_US(20)
#undef POLARIS_US
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace polaris
