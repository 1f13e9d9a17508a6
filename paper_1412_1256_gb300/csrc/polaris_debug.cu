// Bit-exactness check of the staged data translation (Fig. 2 caption: integer codes to
// floats).  From N = 2^13 up, phase 1 stages each tile's packed words in shared memory, transposes
// their codes there and decodes each lane's rows from the transposed words (polaris_codes.cuh).
// k_unpack_staged stages tile by tile and transposes and decodes through those same device
// functions, so the levels phase 1 transforms can be compared with the oracle's decode bit for
// bit, transposed apart (layout 0) or in place (layout 1).  (2^13 and 2^14 run in k_fused, which
// transposes and decodes through the same transpose_codes and code_pair; here they stage phase 1's tiles.)
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
  static constexpr bool STAGED = !(BITS == 1 && LOGN >= 19);  // (what this check has always answered)
};

// One CTA per tile (segment s, first column b0): stage the tile's N1 rows x WPR words of IF a
// (and IF b), transpose, then decode lane q1's rows t of column col -> sample
// n = s N + (q1 + Q1 t) N2 + b0 + col.
template <int LOGN, int BITS>
__global__ void __launch_bounds__(256) k_unpack_staged(const uint32_t* __restrict__ pa, const uint32_t* __restrict__ pb,
                                                       int in_place, float* __restrict__ oa, float* __restrict__ ob) {
  using SP = StagedPlan<LOGN, BITS, (LOGN >= kWideMin)>;
  using PL = typename SP::PL;
  using ST = typename SP::ST;
  constexpr int N = PL::N, N1 = PL::N1, N2 = PL::N2, Q1 = PL::Q1, P = PL::P1, TILE = ST::TILE, WPR = ST::WPR;
  constexpr int SEGW = N * BITS / 32, ROWW = N2 * BITS / 32;  // words per segment, per row
  constexpr int UPT = (ST::UNITS + 255) / 256;
  extern __shared__ __align__(16) uint32_t stg[];
  constexpr int TPS = N2 / TILE;  // tiles per segment
  const int s = blockIdx.x / TPS, b0 = (blockIdx.x % TPS) * TILE;
  const uint32_t* sa = pa + (size_t)s * SEGW + (b0 * BITS) / 32;
  const uint32_t* sbp = pb ? pb + (size_t)s * SEGW + (b0 * BITS) / 32 : nullptr;
  for (int k = threadIdx.x; k < N1 * WPR; k += blockDim.x) {
    const int row = k / WPR, w = k % WPR, o = row * ST::RP + w;
    stg[o] = sa[row * ROWW + w];
    stg[N1 * ST::RP + o] = sbp ? sbp[row * ROWW + w] : stg[o];  // (IF a again without an IF b, as phase 1 stages it)
  }
  __syncthreads();
  uint32_t* tr = in_place ? stg : stg + ST::RAWW;
  uint32_t x[UPT][ST::KB][32 / BITS];
#pragma unroll
  for (int i = 0; i < UPT; ++i)
    if ((int)threadIdx.x + 256 * i < ST::UNITS) p1_unit_load<PL, ST, BITS>(stg, threadIdx.x + 256 * i, x[i]);
  __syncthreads();
#pragma unroll
  for (int i = 0; i < UPT; ++i)
    if ((int)threadIdx.x + 256 * i < ST::UNITS) p1_unit_store<PL, ST, BITS>(tr, threadIdx.x + 256 * i, x[i]);
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

template <int LOGN, int BITS>
static cudaError_t launch_unpack_staged_t(const uint32_t* pa, const uint32_t* pb, long long nseg, int in_place, float* oa,
                                          float* ob, cudaStream_t st) {
  using SP = StagedPlan<LOGN, BITS, (LOGN >= kWideMin)>;
  using PL = typename SP::PL;
  using ST = typename SP::ST;
  if constexpr (!SP::STAGED) {
    return cudaErrorInvalidValue;
  } else {
    const size_t smem = 4 * (size_t)(ST::RAWW + ST::TRW);  // (in place: the larger of the two would do)
    cudaError_t e = cudaFuncSetAttribute(k_unpack_staged<LOGN, BITS>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)smem);
    if (e != cudaSuccess) return e;
    const long long grid = nseg * (PL::N2 / ST::TILE);
    k_unpack_staged<LOGN, BITS><<<(unsigned)grid, 256, smem, st>>>(pa, pb, in_place, oa, ob);
    return cudaGetLastError();
  }
}

template <int LOGN>
static cudaError_t launch_unpack_staged_n(int bits, const uint32_t* pa, const uint32_t* pb, long long nseg, int in_place,
                                          float* oa, float* ob, cudaStream_t st) {
  switch (bits) {
    case 1: return launch_unpack_staged_t<LOGN, 1>(pa, pb, nseg, in_place, oa, ob, st);
    case 2: return launch_unpack_staged_t<LOGN, 2>(pa, pb, nseg, in_place, oa, ob, st);
    case 4: return launch_unpack_staged_t<LOGN, 4>(pa, pb, nseg, in_place, oa, ob, st);
    case 8: return launch_unpack_staged_t<LOGN, 8>(pa, pb, nseg, in_place, oa, ob, st);
    default: return cudaErrorInvalidValue;
  }
}

template <int LOGN, int BITS>
static constexpr bool staged_t() {
  return StagedPlan<LOGN, BITS, (LOGN >= kWideMin)>::STAGED;
}
template <int LOGN>
static constexpr bool staged_n(int bits) {
  return bits == 1 ? staged_t<LOGN, 1>() : bits == 2 ? staged_t<LOGN, 2>() : bits == 4 ? staged_t<LOGN, 4>()
                                                                            : staged_t<LOGN, 8>();
}

// true when phase 1 stages its input (and decodes through p1_level) at this size
bool phase1_staged(int logn, int bits) {
  switch (logn) {
#define POLARIS_ST(L) \
  case L: return staged_n<L>(bits);
    POLARIS_ST(4) POLARIS_ST(5) POLARIS_ST(6) POLARIS_ST(7) POLARIS_ST(8) POLARIS_ST(9) POLARIS_ST(10)
    POLARIS_ST(11) POLARIS_ST(12) POLARIS_ST(13) POLARIS_ST(14) POLARIS_ST(15) POLARIS_ST(16) POLARIS_ST(17)
    POLARIS_ST(18) POLARIS_ST(19) POLARIS_ST(20)
#undef POLARIS_ST
    default: return false;
  }
}

// decode nseg whole segments of IF a (and IF b, may be null) through the staged decoder
cudaError_t launch_unpack_staged(int logn, int bits, const uint32_t* pa, const uint32_t* pb, long long nseg, int in_place,
                                 float* oa, float* ob, cudaStream_t st) {
  switch (logn) {
#define POLARIS_US(L) \
  case L: return launch_unpack_staged_n<L>(bits, pa, pb, nseg, in_place, oa, ob, st);
    POLARIS_US(13) POLARIS_US(14) POLARIS_US(15) POLARIS_US(16) POLARIS_US(17) POLARIS_US(18) POLARIS_US(19)
    POLARIS_US(20)
#undef POLARIS_US
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace polaris
