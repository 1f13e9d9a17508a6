// Leakage calibration (forward model and adjoint): what the segment kernels share.  The
// model, its gradients and the kernel sequence are described in polaris_adjoint.cu; the
// transforms of N = 2^9 .. 2^14 run in size-specialised kernels (polaris_adjoint_sized.cu,
// polaris_adjoint_teams.cu), those of buffers that are not 16-byte aligned in polaris_adjoint.cu's
// kernels for any N, the smaller sizes in that file's kernels of many segments per CTA.
#pragma once

#include <cuda_runtime.h>

#include <cstdint>

#include "polaris_device.cuh"
#include "polaris_launch.cuh"

namespace polaris {

struct AdjArgs {
  const uint32_t* in[2];  // the two IFs' packed words
  int N, log2n, nbin, nseg, grid, threads;
  const float2* tw;       // per-pass twiddles: tw[r Ns + k - 1] = W_{Ns R}^{r k} (N - 1 entries)
  const float* window;    // N
  float4* part;           // [grid][nbin]: (|X|^2, |Y|^2, Re X conj(Y), Im X conj(Y)) per bin
  const float4* mat;      // per bin the Hermitian matrix of the spectral gradients: (m11, m22, Re m12, Im m12)
  float* gpart;           // [grid][N] window-gradient partials
};

// shared-memory layout of the N points: one float2 of padding after every 16 keeps the
// stride-16 writes of the first pass, and every other access, free of bank conflicts
__host__ __device__ __forceinline__ int apad(int i) { return i + (i >> 4); }
__host__ __device__ constexpr int adj_smem_points(int N) { return N + N / 16; }

__device__ __forceinline__ float2 c_add(float2 a, float2 b) { return make_float2(a.x + b.x, a.y + b.y); }
__device__ __forceinline__ float2 c_conj(float2 a) { return make_float2(a.x, -a.y); }

// spectral gradients of bin k, G_X = m11 X + m12 Y, G_Y = conj(m12) X + m22 Y, with
// X = (Z[k] + Zm) / 2, Y = (Z[k] - Zm) / 2i, Zm = conj Z[N-k]
__device__ __forceinline__ void adj_bin_gradient(float4 m, float2 Zk, float2 Zm, float2& GX, float2& GY) {
  const float2 X = make_float2(0.5f * (Zk.x + Zm.x), 0.5f * (Zk.y + Zm.y));
  const float2 Y = make_float2(0.5f * (Zk.y - Zm.y), -0.5f * (Zk.x - Zm.x));
  GX = c_add(make_float2(m.x * X.x, m.x * X.y), cmul(make_float2(m.z, m.w), Y));
  GY = c_add(make_float2(m.y * Y.x, m.y * Y.y), cmul(make_float2(m.z, -m.w), X));
}

// level of sample idx of one IF (an ordinary load: a read-only one could be moved up over the wait for
// the kernel before)
template <int BITS>
__device__ __forceinline__ float adj_level(const uint32_t* in, long long idx) {
  if constexpr (BITS == 8) {
    return (float)(int)reinterpret_cast<const signed char*>(in)[idx];
  } else {
    constexpr int SPW = 32 / BITS;
    return decode_level<BITS>(in[idx / SPW], (uint32_t)(idx % SPW) * BITS);
  }
}

// Size-specialised segment kernels (polaris_adjoint_sized.cu) for log2 N in
// [kAdjSizedMin, kAdjSizedMax].  adj_sized_prepare: sets the kernels' shared-memory limits
// for this device (current) and returns how many CTAs of the window kernel may share an SM (the
// forward kernel runs one); adj_sized_launch: one segment kernel (forward or window pass) on
// a.grid CTAs.
constexpr int kAdjSizedMin = 9, kAdjSizedMax = 14;
cudaError_t adj_sized_prepare(int log2n, int bits, int* window_ctas);
cudaError_t adj_sized_launch(int log2n, int bits, bool window_pass, const AdjArgs& a, cudaStream_t st);
// the forward kernel for more segments than CTAs (polaris_adjoint_teams.cu), up to 2^kAdjTeamsMax points
// (above, two teams' points do not fit an SM)
constexpr int kAdjTeamsMax = 12;
cudaError_t adj_teams_prepare(int log2n, int bits);
cudaError_t adj_teams_launch(int log2n, int bits, const AdjArgs& a, cudaStream_t st);

}  // namespace polaris
