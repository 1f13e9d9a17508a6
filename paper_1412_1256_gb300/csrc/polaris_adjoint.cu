// Differentiable leakage calibration: forward model and hand-written adjoint.
//
// Model (ours: the paper calibrates gains offline, Sec. 2.1, and says nothing about
// polarisation leakage).  Two IFs R and L (circular feeds), segments of N samples at hop N,
// window w:
//   X_s[k] = sum_n w[n] x_s[n] e^{-2 pi i n k / N}, Y_s[k] likewise, k = 0..N/2
//   Xt = gR (X + DR[k] Y),  Yt = gL (Y + DL[k] X)
//   RR = sum_s |Xt|^2, LL = sum_s |Yt|^2, RL = sum_s Xt conj(Yt)
//   I = (RR + LL)/2, V = (RR - LL)/2, Q = Re RL, U = Im RL
//   loss = sum_k sum_S (S[k] - T_S[k])^2
//
// The mixing is linear per bin, so RR, LL and RL are quadratic forms of the plain sums
//   A = sum_s |X|^2, B = sum_s |Y|^2, C = sum_s X conj(Y):
//   P_R = sum|X + DR Y|^2 = A + |DR|^2 B + 2 Re(conj(DR) C)
//   P_L = sum|Y + DL X|^2 = B + |DL|^2 A + 2 Re(DL C)
//   Qm  = sum (X + DR Y) conj(Y + DL X) = C + conj(DL) A + DR B + DR conj(DL) conj(C)
//   RR = |gR|^2 P_R, LL = |gL|^2 P_L, RL = gR conj(gL) Qm.
// Gradients use G = dL/d re + i dL/d im for every complex parameter.  With r_S = 2 (S - T_S),
// a = (r_I + r_V)/2, b = (r_I - r_V)/2, c = r_Q + i r_U:
//   G_gR = sum_k 2a P_R gR + c gL conj(Qm)          G_gL = sum_k 2b P_L gL + conj(c) gR Qm
//   G_DR[k] = 2a |gR|^2 (B DR + C) + c conj(gR) gL (B + DL C)
//   G_DL[k] = 2b |gL|^2 (A DL + conj(C)) + conj(c) gR conj(gL) (A + DR conj(C))
// so neither needs the segments again.  The window does: per segment the spectral
// gradients are G_X = m11 X + m12 Y, G_Y = m21 X + m22 Y with a per-bin 2 x 2 matrix (from
// G_Xt = 2a Xt + c Yt, G_Yt = 2b Yt + conj(c) Xt pulled back through the mixing), and
//   dL/dw[n] = sum_s x_s[n] Re(sum_k G_X e^{+2 pi i n k/N}) + y_s[n] Re(sum_k G_Y e^{+...}),
// the real inverse transforms of the Hermitian extensions of G_X and G_Y, taken together
// as one complex inverse transform of H_X + i H_Y.  Segments are transformed again in the
// adjoint pass, not stored.
//
// Kernels (no atomics; every sum has a fixed order, so runs are bitwise reproducible):
//   k_adj_forward  (2^5 .. 2^8: k_adjm_forward and k_adjm_window, many segments per CTA)
//                  a grid of G CTAs, each over segments b, b + G, ...: decode, window, a
//                  radix-16 Stockham transform of the pair x + i y in shared memory, split
//                  into X and Y, per-CTA partial sums of |X|^2, |Y|^2, X conj(Y)
//                  (N = 2^9 .. 2^14: k_adjs_forward, the same per size at compile time,
//                  polaris_adjoint_sized.cu; likewise k_adjs_window; k_adjs_teams,
//                  polaris_adjoint_teams.cu, where there are more segments than SMs)
//   k_adj_bins     per bin: partials summed (fp32 slices, added in fp64), the model,
//                  Stokes and loss in fp64, the gain and leakage gradients and the
//                  window-adjoint matrix in fp32
//   k_adj_window   per segment again: forward transform, G_X and G_Y, inverse transform,
//                  per-CTA partials of the window gradient
//   k_adj_wsum     the window-gradient partials summed per tap, and the block partials of the
//                  loss and gain gradients in order (k_adj_finish: those alone, without gradients)
// The launches are programmatic dependent ones (but for k_adj_forward and k_adj_window): each kernel's
// set-up, and the window pass's first transform, run while the one before ends.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdint>
#include <cstdio>
#include <cstring>
#include <string>
#include <vector>

#include "../../include/polaris.h"
#include "polaris_adjoint.cuh"
#include "polaris_kernels.cuh"  // dependent launch

namespace polaris {

constexpr int kMaxCtasPerSm = 8;

// One Stockham autosort pass of radix R (Ns = product of the radices already applied), in
// place in z: every j < N/R reads z[j + r N/R] (r < R), multiplies by W_{Ns R}^{r (j mod Ns)}
// (from the pass's own table, where consecutive j read consecutive entries),
// takes an R-point DFT and writes output q to z[(j / Ns) Ns R + q Ns + j mod Ns].  All reads
// of the pass finish before any write.  The block has exactly T = N/16 threads and each
// holds 16 points: one j for R = 16, j = t, t + T, ... for smaller radices, always < N/R
// (a bounds test here would push the point arrays into local memory).
template <int R>
__device__ __forceinline__ void stockham_pass(float2* z, int N, int Ns, const float2* __restrict__ tw, int T, int t) {
  constexpr int JPT = 16 / R;
  const int m = N / R;
  float2 v[JPT][R];
#pragma unroll
  for (int q = 0; q < JPT; ++q) {
    const int j = t + q * T;
    const int k = j & (Ns - 1);
#pragma unroll
    for (int r = 0; r < R; ++r) {
      float2 a = z[apad(j + r * m)];
      if (r > 0 && Ns > 1) a = cmul(a, __ldg(tw + r * Ns + k - 1));
      v[q][ct::bitrev(r, R)] = a;
    }
  }
  __syncthreads();
#pragma unroll
  for (int q = 0; q < JPT; ++q) {
    const int j = t + q * T;
    dit<R>(v[q]);
    const int k = j & (Ns - 1);
    const int base = (j - k) * R + k;
#pragma unroll
    for (int r = 0; r < R; ++r) z[apad(base + r * Ns)] = v[q][r];
  }
  __syncthreads();
}

// forward DFT of the N points in z (natural order in and out); callers sync before
__device__ __forceinline__ void adj_fft(float2* z, int N, int log2n, const float2* __restrict__ tw, int T, int t) {
  int Ns = 1;
#pragma unroll 1
  for (int p = 0; p < (log2n >> 2); ++p, Ns <<= 4) stockham_pass<16>(z, N, Ns, tw, T, t);
  switch (log2n & 3) {
    case 1: stockham_pass<2>(z, N, Ns, tw, T, t); break;
    case 2: stockham_pass<4>(z, N, Ns, tw, T, t); break;
    case 3: stockham_pass<8>(z, N, Ns, tw, T, t); break;
    default: break;
  }
}

// z[n] = w[n] (x[n] + i y[n]) for segment s; thread t fills n = t + T e, e < 16, so that
// every load is coalesced and the stores are conflict-free
template <int BITS>
__device__ __forceinline__ void adj_load_segment(const AdjArgs& a, float2* z, long long s, int t) {
  const long long base = s * a.N;
#pragma unroll 8
  for (int e = 0; e < 16; ++e) {
    const int n = t + e * a.threads;
    const float w = a.window[n];
    z[apad(n)] = make_float2(w * adj_level<BITS>(a.in[0], base + n), w * adj_level<BITS>(a.in[1], base + n));
  }
}

// |X|^2, |Y|^2, Re and Im X conj(Y) of bin k: X = (Z[k] + conj Z[N-k]) / 2, Y = (Z[k] - conj Z[N-k]) / 2i
__device__ __forceinline__ float4 adj_products(const float2* z, int N, int k) {
  const float2 Zk = z[apad(k)], Zm = c_conj(z[apad((N - k) & (N - 1))]);
  const float2 X = make_float2(0.5f * (Zk.x + Zm.x), 0.5f * (Zk.y + Zm.y));
  const float2 Y = make_float2(0.5f * (Zk.y - Zm.y), -0.5f * (Zk.x - Zm.x));
  return make_float4(fmaf(X.x, X.x, X.y * X.y), fmaf(Y.x, Y.x, Y.y * Y.y), fmaf(X.x, Y.x, X.y * Y.y),
                     fmaf(X.y, Y.x, -X.x * Y.y));
}

// G_X and G_Y of bin k; conj of the Hermitian extension of G_X + i G_Y goes back into slots k and N - k
// (the inverse transform is conj(DFT(conj H)))
__device__ __forceinline__ void adj_pull_back(float2* z, int N, int k, float4 m) {
  const int km = (N - k) & (N - 1);
  const float2 Zk = z[apad(k)], Zm = c_conj(z[apad(km)]);
  float2 GX, GY;
  adj_bin_gradient(m, Zk, Zm, GX, GY);
  if (k == 0 || 2 * k == N) {
    z[apad(k)] = make_float2(GX.x, -GY.x);  // H = Re G_X + i Re G_Y
  } else {
    const float2 hx = make_float2(0.5f * GX.x, 0.5f * GX.y), hy = make_float2(0.5f * GY.x, 0.5f * GY.y);
    // H[k] = hx + i hy, H[N-k] = conj(hx) + i conj(hy); store their conjugates
    z[apad(k)] = make_float2(hx.x - hy.y, -(hx.y + hy.x));
    z[apad(km)] = make_float2(hx.x + hy.y, hx.y - hy.x);
  }
}

// one segment of the forward pass
template <int BITS>
__device__ __forceinline__ void adj_forward_segment(const AdjArgs& a, float2* z, long long s, bool first) {
  const int N = a.N, nbin = a.nbin;
  float4* part = a.part + (size_t)blockIdx.x * nbin;
  adj_load_segment<BITS>(a, z, s, threadIdx.x);
  __syncthreads();
  adj_fft(z, N, a.log2n, a.tw, a.threads, threadIdx.x);
#pragma unroll 1
  for (int k = threadIdx.x; k < nbin; k += a.threads) {
    const float4 v = adj_products(z, N, k);
    if (first) {
      part[k] = v;
    } else {
      const float4 o = part[k];
      part[k] = make_float4(o.x + v.x, o.y + v.y, o.z + v.z, o.w + v.w);
    }
  }
  __syncthreads();
}

template <int BITS>
__global__ void __launch_bounds__(1024) k_adj_forward(AdjArgs a) {
  extern __shared__ float2 z[];
#pragma unroll 1
  for (long long s = blockIdx.x; s < a.nseg; s += a.grid) adj_forward_segment<BITS>(a, z, s, s == blockIdx.x);
}

// one segment of the window-gradient pass
template <int BITS>
__device__ __forceinline__ void adj_window_segment(const AdjArgs& a, float2* z, long long s, bool first) {
  const int N = a.N, nbin = a.nbin;
  float* gpart = a.gpart + (size_t)blockIdx.x * N;
  adj_load_segment<BITS>(a, z, s, threadIdx.x);
  __syncthreads();
  adj_fft(z, N, a.log2n, a.tw, a.threads, threadIdx.x);
  // thread k owns slots k and N - k
#pragma unroll 1
  for (int k = threadIdx.x; k < nbin; k += a.threads) adj_pull_back(z, N, k, a.mat[k]);
  __syncthreads();
  adj_fft(z, N, a.log2n, a.tw, a.threads, threadIdx.x);
  // h = conj(F): dL/dw[n] += x[n] Re h[n] + y[n] Im h[n] = x F.x - y F.y
  const long long base = s * N;
#pragma unroll 8
  for (int e = 0; e < 16; ++e) {
    const int n = threadIdx.x + e * a.threads;
    const float2 F = z[apad(n)];
    const float g = fmaf(adj_level<BITS>(a.in[0], base + n), F.x, -adj_level<BITS>(a.in[1], base + n) * F.y);
    gpart[n] = first ? g : gpart[n] + g;
  }
  __syncthreads();
}

template <int BITS>
__global__ void __launch_bounds__(1024) k_adj_window(AdjArgs a) {
  extern __shared__ float2 z[];
#pragma unroll 1
  for (long long s = blockIdx.x; s < a.nseg; s += a.grid) adj_window_segment<BITS>(a, z, s, s == blockIdx.x);
}

// ------------------------------------------------------------------------------------------
// N = 2^5 to 2^8, where one segment's N/16 threads are a fraction of a warp: a CTA takes many segments at
// once, one per team of N/16 threads.
//   - Forward: the CTA's group is the segments b, b + G, ... that one small CTA took in turn before, its
//     teams taking consecutive ones.  The products go to shared memory and are added in that order, one
//     chain per bin and quantity, so the partial sums are the same to the bit.
//   - Window pass: every team adds its segments' taps in registers; the CTA adds its teams at the end.
// Bound by latency (loads, and barriers of two or four warps).  Whole steps of 4 M int8 samples with
// one segment per CTA at a time, eight CTAs of 4 to 16 threads per SM, and now: 2^6 517 -> 79 us, 2^7
// 301 -> 76, 2^8 (2 bits) 188 -> 85.
// ------------------------------------------------------------------------------------------
template <int LOGN, int THREADS>
struct AdjSmall {
  static constexpr int N = 1 << LOGN, T = N / 16, TEAMS = THREADS / T, NBIN = N / 2 + 1, POINTS = adj_smem_points(N);
};
constexpr int kSmallForward = 64, kSmallWindow = 128, kSmallWindowCtas = 6;  // threads; window CTAs per SM

template <int LOGN, int BITS>
__global__ void __launch_bounds__(kSmallForward) k_adjm_forward(AdjArgs a) {
  using S = AdjSmall<LOGN, kSmallForward>;
  constexpr int NC = 4 * S::NBIN, CH = (NC + kSmallForward - 1) / kSmallForward;  // chains of a bin and quantity
  __shared__ float2 zs[S::TEAMS][S::POINTS];
  __shared__ __align__(16) float prod[S::TEAMS][NC];
  const int team = threadIdx.x / S::T, t = threadIdx.x % S::T;
  float2* z = zs[team];
  float acc[CH];
#pragma unroll
  for (int c = 0; c < CH; ++c) acc[c] = 0.f;
  pdl_wait();  // (dependent launch: the inputs and the partials may be touched from here on)
#pragma unroll 1
  for (long long s0 = blockIdx.x; s0 < a.nseg; s0 += (long long)S::TEAMS * a.grid) {
    const long long left = (a.nseg - 1 - s0) / a.grid + 1;  // segments of the group from s0 on
    const int n = left < S::TEAMS ? (int)left : S::TEAMS;
    adj_load_segment<BITS>(a, z, s0 + (long long)(team < n ? team : 0) * a.grid, t);  // (idle teams: the first one again)
    __syncthreads();
    adj_fft(z, S::N, LOGN, a.tw, S::T, t);
#pragma unroll 1
    for (int k = t; k < S::NBIN; k += S::T) reinterpret_cast<float4*>(prod[team])[k] = adj_products(z, S::N, k);
    __syncthreads();
#pragma unroll
    for (int c = 0; c < CH; ++c) {
      const int i = threadIdx.x + c * kSmallForward;
      if (i < NC) {
#pragma unroll 4
        for (int j = 0; j < n; ++j) acc[c] += prod[j][i];
      }
    }
  }
  float* part = reinterpret_cast<float*>(a.part + (size_t)blockIdx.x * S::NBIN);
#pragma unroll
  for (int c = 0; c < CH; ++c) {
    const int i = threadIdx.x + c * kSmallForward;
    if (i < NC) part[i] = acc[c];
  }
}

template <int LOGN, int BITS>
__global__ void __launch_bounds__(kSmallWindow, kSmallWindowCtas) k_adjm_window(AdjArgs a) {
  using S = AdjSmall<LOGN, kSmallWindow>;
  __shared__ float2 zs[S::TEAMS][S::POINTS];
  const int team = threadIdx.x / S::T, t = threadIdx.x % S::T;
  float2* z = zs[team];
  float acc[16];
#pragma unroll
  for (int e = 0; e < 16; ++e) acc[e] = 0.f;
  pdl_wait();
#pragma unroll 1
  for (long long s0 = (long long)blockIdx.x * S::TEAMS; s0 < a.nseg; s0 += (long long)S::TEAMS * a.grid) {
    const bool mine = s0 + team < a.nseg;
    const long long s = mine ? s0 + team : s0;  // (idle teams: the CTA's first one again)
    adj_load_segment<BITS>(a, z, s, t);
    __syncthreads();
    adj_fft(z, S::N, LOGN, a.tw, S::T, t);
#pragma unroll 1
    for (int k = t; k < S::NBIN; k += S::T) adj_pull_back(z, S::N, k, a.mat[k]);
    __syncthreads();
    adj_fft(z, S::N, LOGN, a.tw, S::T, t);
    // h = conj(F): dL/dw[n] += x[n] Re h[n] + y[n] Im h[n] = x F.x - y F.y
#pragma unroll
    for (int e = 0; e < 16; ++e) {
      const int n = t + e * S::T;
      const float2 F = z[apad(n)];
      const float g = fmaf(adj_level<BITS>(a.in[0], s * S::N + n), F.x, -adj_level<BITS>(a.in[1], s * S::N + n) * F.y);
      acc[e] += mine ? g : 0.f;
    }
    __syncthreads();
  }
  // the teams' sums, in order
  float* sums = reinterpret_cast<float*>(zs[team]);
#pragma unroll
  for (int e = 0; e < 16; ++e) sums[t + e * S::T] = acc[e];
  __syncthreads();
  for (int n = threadIdx.x; n < S::N; n += kSmallWindow) {
    float g = 0.f;
#pragma unroll 4
    for (int j = 0; j < S::TEAMS; ++j) g += reinterpret_cast<const float*>(zs[j])[n];
    a.gpart[(size_t)blockIdx.x * S::N + n] = g;
  }
}

struct dc {
  double x, y;
};
__device__ __forceinline__ dc dmul(dc a, dc b) { return {a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x}; }
__device__ __forceinline__ dc dconj(dc a) { return {a.x, -a.y}; }
__device__ __forceinline__ dc dadd(dc a, dc b) { return {a.x + b.x, a.y + b.y}; }
__device__ __forceinline__ dc dscale(dc a, double s) { return {a.x * s, a.y * s}; }
__device__ __forceinline__ double dnorm(dc a) { return a.x * a.x + a.y * a.y; }
__device__ __forceinline__ float2 fscale(float2 a, float s) { return make_float2(a.x * s, a.y * s); }
__device__ __forceinline__ float fnorm(float2 a) { return fmaf(a.x, a.x, a.y * a.y); }

struct BinArgs {
  const float4* part;
  int grid, nbin;
  const float* gains;
  const float* leak;
  const float* target;
  float* stokes;
  float* grad_leak;
  float4* mat;
  double* bpart;  // [blocks][5]: loss, G_gR re/im, G_gL re/im
};

// A block covers kBinsPerBlock bins; its kSlices warps sum the per-CTA partials of the
// segment kernel (one 16-byte load per CTA and bin) over interleaved slices of CTAs in fp32, the
// slice sums are added in fp64 in slice order (one warp per quantity), then the model per bin:
// the sums, Stokes and loss in fp64, the gradients and the window-adjoint matrix in fp32.
// Bound by the latency of the loads, of which kInFlight per thread are started together (a slice
// of a grid of one CTA per SM, 152 / 8 = 19, in one round), and by the fp64 arithmetic, at 64
// cycles per warp and instruction and scheduler: four warps share it, one expression each.
constexpr int kBinsPerBlock = 32, kSlices = 8, kInFlight = 20;

__global__ void __launch_bounds__(kBinsPerBlock * kSlices, 2) k_adj_bins(BinArgs a) {
  __shared__ float red[kSlices][4][kBinsPerBlock];
  __shared__ double tot[5][kBinsPerBlock];  // A, B, C of a bin, then its loss and gain gradients
  __shared__ double mod[6][kBinsPerBlock];  // RR, LL, Qm, gR conj(gL)
  __shared__ double dif[4][kBinsPerBlock];  // Stokes minus target
  __shared__ float fmd[4][kBinsPerBlock];  // P_R, P_L, Qm
  const int nbin = a.nbin;
  const int lane = threadIdx.x & 31, sl = threadIdx.x >> 5;
  const int k = blockIdx.x * kBinsPerBlock + lane;
  float s4[4] = {0.f, 0.f, 0.f, 0.f};
  pdl_wait();  // the segment kernel's partials (dependent launch)
  if (k < nbin) {
#pragma unroll 1
    for (int g0 = sl; g0 < a.grid; g0 += kSlices * kInFlight) {
      float4 v[kInFlight];
#pragma unroll
      for (int i = 0; i < kInFlight; ++i) {
        const int g = g0 + i * kSlices;
        if (g < a.grid) v[i] = __ldcg(a.part + (size_t)g * nbin + k);
      }
#pragma unroll
      for (int i = 0; i < kInFlight; ++i)
        if (g0 + i * kSlices < a.grid) {
          s4[0] += v[i].x;
          s4[1] += v[i].y;
          s4[2] += v[i].z;
          s4[3] += v[i].w;
        }
    }
  }
  pdl_trigger();
#pragma unroll
  for (int q = 0; q < 4; ++q) red[sl][q][lane] = s4[q];
  __syncthreads();
  if (sl < 4) {
    double t = 0.0;
    for (int w = 0; w < kSlices; ++w) t += (double)red[w][sl][lane];
    tot[sl][lane] = t;
  }
  __syncthreads();
  const int kk = k < nbin ? k : 0;
  const double A = tot[0][lane], B = tot[1][lane];
  const dc C = {tot[2][lane], tot[3][lane]};
  const float2 fgR = make_float2(a.gains[0], a.gains[1]), fgL = make_float2(a.gains[2], a.gains[3]);
  const float2 fDR = make_float2(a.leak[2 * kk], a.leak[2 * kk + 1]);
  const float2 fDL = make_float2(a.leak[2 * (nbin + kk)], a.leak[2 * (nbin + kk) + 1]);
  if (sl == 0) {
    const dc gR = {fgR.x, fgR.y}, DR = {fDR.x, fDR.y};
    const double PR = A + dnorm(DR) * B + 2.0 * dmul(dconj(DR), C).x;
    mod[0][lane] = dnorm(gR) * PR;
    fmd[0][lane] = (float)PR;
  } else if (sl == 1) {
    const dc gL = {fgL.x, fgL.y}, DL = {fDL.x, fDL.y};
    const double PL = B + dnorm(DL) * A + 2.0 * dmul(DL, C).x;
    mod[1][lane] = dnorm(gL) * PL;
    fmd[1][lane] = (float)PL;
  } else if (sl == 2) {
    const dc DR = {fDR.x, fDR.y}, DL = {fDL.x, fDL.y};
    const dc Qm = dadd(dadd(C, dscale(dconj(DL), A)), dadd(dscale(DR, B), dmul(dmul(DR, dconj(DL)), dconj(C))));
    mod[2][lane] = Qm.x;
    mod[3][lane] = Qm.y;
    fmd[2][lane] = (float)Qm.x;
    fmd[3][lane] = (float)Qm.y;
  } else if (sl == 3) {
    const dc gR = {fgR.x, fgR.y}, gL = {fgL.x, fgL.y};
    const dc g = dmul(gR, dconj(gL));
    mod[4][lane] = g.x;
    mod[5][lane] = g.y;
  }
  __syncthreads();
  if (sl < 4) {  // warp q: Stokes parameter q (I, Q, U, V)
    const double RR = mod[0][lane], LL = mod[1][lane];
    const dc Qm = {mod[2][lane], mod[3][lane]}, g = {mod[4][lane], mod[5][lane]};
    double S;
    if (sl == 0) S = 0.5 * (RR + LL);
    else if (sl == 1) S = dmul(g, Qm).x;
    else if (sl == 2) S = dmul(g, Qm).y;
    else S = 0.5 * (RR - LL);
    if (k < nbin && a.stokes) a.stokes[sl * nbin + k] = (float)S;
    dif[sl][lane] = a.target ? S - (double)a.target[sl * nbin + kk] : 0.0;
  }
  __syncthreads();
  double acc[5] = {0.0, 0.0, 0.0, 0.0, 0.0};
  if (sl == 0 && k < nbin) {
    if (a.target) {
      float r[4];
      for (int q = 0; q < 4; ++q) {
        const double d = dif[q][lane];
        acc[0] += d * d;
        r[q] = (float)(2.0 * d);
      }
      if (a.mat) {
        const float ca = 0.5f * (r[0] + r[3]), cb = 0.5f * (r[0] - r[3]);
        const float2 c = make_float2(r[1], r[2]), cc = c_conj(c);
        const float2 fC = make_float2((float)C.x, (float)C.y), fQ = make_float2(fmd[2][lane], fmd[3][lane]);
        const float fA = (float)A, fB = (float)B;
        const float2 ggR = c_add(fscale(fgR, 2.f * ca * fmd[0][lane]), cmul(cmul(c, fgL), c_conj(fQ)));
        const float2 ggL = c_add(fscale(fgL, 2.f * cb * fmd[1][lane]), cmul(cmul(cc, fgR), fQ));
        acc[1] = ggR.x;
        acc[2] = ggR.y;
        acc[3] = ggL.x;
        acc[4] = ggL.y;
        const float2 gDR = c_add(fscale(c_add(fscale(fDR, fB), fC), 2.f * ca * fnorm(fgR)),
                                 cmul(cmul(c, cmulc(fgR, fgL)), c_add(make_float2(fB, 0.f), cmul(fDL, fC))));
        const float2 gDL = c_add(fscale(c_add(fscale(fDL, fA), c_conj(fC)), 2.f * cb * fnorm(fgL)),
                                 cmul(cmul(cc, cmulc(fgL, fgR)), c_add(make_float2(fA, 0.f), cmul(fDR, c_conj(fC)))));
        a.grad_leak[2 * k] = gDR.x;
        a.grad_leak[2 * k + 1] = gDR.y;
        a.grad_leak[2 * (nbin + k)] = gDL.x;
        a.grad_leak[2 * (nbin + k) + 1] = gDL.y;
        // G_Xt = al1 X + be1 Y, G_Yt = al2 X + be2 Y; G_X = conj(gR) G_Xt + conj(gL DL) G_Yt,
        // G_Y = conj(gR DR) G_Xt + conj(gL) G_Yt: a Hermitian matrix (the loss is a real function
        // of |X|^2, |Y|^2 and X conj(Y)), kept as its two real entries and m12
        const float2 gLDL = cmul(fgL, fDL), gRDR = cmul(fgR, fDR);
        const float2 al1 = c_add(fscale(fgR, 2.f * ca), cmul(c, gLDL));
        const float2 be1 = c_add(fscale(gRDR, 2.f * ca), cmul(c, fgL));
        const float2 al2 = c_add(fscale(gLDL, 2.f * cb), cmul(cc, fgR));
        const float2 be2 = c_add(fscale(fgL, 2.f * cb), cmul(cc, gRDR));
        const float2 m11 = c_add(cmulc(fgR, al1), cmulc(gLDL, al2)), m12 = c_add(cmulc(fgR, be1), cmulc(gLDL, be2));
        const float2 m22 = c_add(cmulc(gRDR, be1), cmulc(fgL, be2));
        a.mat[k] = make_float4(m11.x, m22.x, m12.x, m12.y);
      }
    }
  }
  if (a.bpart) {  // (uniform)
    __syncthreads();  // tot has been read
    if (sl == 0)
      for (int q = 0; q < 5; ++q) tot[q][lane] = acc[q];
    __syncthreads();
    if (sl < 5) {  // one warp per quantity
      double v = tot[sl][lane];
      for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
      if (lane == 0) a.bpart[5 * blockIdx.x + sl] = v;
    }
  }
}

// five warps, one per quantity: block partials summed lane-strided, then across the warp
// (the last block of k_adj_bins to finish doing this instead, elected by an atomic ticket
// after a memory fence, measured slower: 20.6 us against 13.4 + 3.7 us)
__device__ __forceinline__ void adj_finish(const double* bpart, int blocks, double* loss, float* grad_gains) {
  const int q = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (q >= 5) return;
  double t = 0.0;
#pragma unroll 4
  for (int b = lane; b < blocks; b += 32) t += bpart[5 * b + q];
  for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
  if (lane == 0) {
    if (q == 0) {
      if (loss) *loss = t;
    } else if (grad_gains) {
      grad_gains[q - 1] = (float)t;
    }
  }
}
// (without gradients; with them k_adj_wsum's last block does it)
__global__ void __launch_bounds__(160) k_adj_finish(const double* bpart, int blocks, double* loss) {
  pdl_wait();
  pdl_trigger();
  adj_finish(bpart, blocks, loss, nullptr);
}

// window-gradient partials summed per tap: 32 taps per block, kSlices warps over the CTAs,
// kInFlight loads started together (four taps per lane with one 16-byte load per CTA ran slower:
// 9.7 against 7.4 us, a quarter of the blocks); one more block sums the loss and gain gradients
__global__ void __launch_bounds__(kBinsPerBlock * kSlices) k_adj_wsum(const float* gpart, int grid, int N, float* grad_w,
                                                                      const double* bpart, int bin_blocks, double* loss,
                                                                      float* grad_gains) {
  __shared__ float red[kSlices][kBinsPerBlock];
  const int lane = threadIdx.x & 31, sl = threadIdx.x >> 5;
  const int n = blockIdx.x * kBinsPerBlock + lane;
  pdl_wait();  // the window pass's partials; k_adj_bins, which that kernel waited for, is complete too
  pdl_trigger();
  if (blockIdx.x == gridDim.x - 1) {
    adj_finish(bpart, bin_blocks, loss, grad_gains);
    return;
  }
  float t = 0.f;
  if (n < N) {
#pragma unroll 1
    for (int g0 = sl; g0 < grid; g0 += kSlices * kInFlight) {
      float v[kInFlight];
#pragma unroll
      for (int i = 0; i < kInFlight; ++i) {
        const int g = g0 + i * kSlices;
        if (g < grid) v[i] = __ldcg(gpart + (size_t)g * N + n);
      }
#pragma unroll
      for (int i = 0; i < kInFlight; ++i)
        if (g0 + i * kSlices < grid) t += v[i];
    }
  }
  red[sl][lane] = t;
  __syncthreads();
  if (sl == 0 && n < N) {
    double u = 0.0;
    for (int w = 0; w < kSlices; ++w) u += (double)red[w][lane];
    grad_w[n] = (float)u;
  }
}

}  // namespace polaris

using namespace polaris;

struct polaris_adj {
  int N = 0, log2n = 0, nbin = 0, bits = 0, device = 0, threads = 0, nsm = 0, grid_max = 0, grid_window = 0, bin_blocks = 0;
  bool sized = false;  // the size-specialised segment kernels (polaris_adjoint_sized.cu)
  size_t smem = 0;
  unsigned char* d_all = nullptr;  // the device memory of the five below
  float2* d_tw = nullptr;
  float4* d_part = nullptr;  // [grid_max][nbin]
  float* d_gpart = nullptr;  // [grid_window][N]
  float4* d_mat = nullptr;   // [nbin]
  double* d_bpart = nullptr; // [bin_blocks][5]
  std::string err;
};

static thread_local std::string g_adj_create_err;

static int adj_err(polaris_adj* h, int code, const char* msg, const char* detail = "") {
  std::string m = std::string(msg) + detail;
  if (h) h->err = m;
  else g_adj_create_err = m;
  return code;
}

template <int BITS>
static cudaError_t adj_prepare(polaris_adj* h, int* ctas_per_sm) {
  const int smem = (int)h->smem;
  cudaError_t e = cudaFuncSetAttribute(k_adj_forward<BITS>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(k_adj_window<BITS>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
  int o1 = 0, o2 = 0;
  if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&o1, k_adj_forward<BITS>, h->threads, h->smem);
  if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&o2, k_adj_window<BITS>, h->threads, h->smem);
  *ctas_per_sm = std::min(o1, o2);
  return e;
}

static void adj_free(polaris_adj* h) { cudaFree(h->d_all); }

extern "C" int polaris_adj_create(int64_t n_fft, int bits, int device, polaris_adj** out) {
  if (!out) return POLARIS_EINVAL;
  *out = nullptr;
  if (bits != 1 && bits != 2 && bits != 4 && bits != 8)
    return adj_err(nullptr, POLARIS_EINVAL, "bits must be 1, 2, 4 or 8");
  if (n_fft < 32 || n_fft > 16384 || (n_fft & (n_fft - 1)))
    return adj_err(nullptr, POLARIS_EINVAL, "n_fft must be a power of two in [32, 16384]");
  int ndev = 0;
  if (cudaGetDeviceCount(&ndev) != cudaSuccess || device < 0 || device >= ndev) {
    cudaGetLastError();
    return adj_err(nullptr, POLARIS_EINVAL, "no such CUDA device");
  }
  polaris_adj* h = new polaris_adj;
  h->N = (int)n_fft;
  while ((1 << h->log2n) < h->N) ++h->log2n;
  h->nbin = h->N / 2 + 1;
  h->bits = bits;
  h->device = device;
  h->threads = h->N / 16;
  h->sized = h->log2n >= kAdjSizedMin && h->log2n <= kAdjSizedMax;
  h->smem = (size_t)adj_smem_points(h->N) * sizeof(float2);
  h->bin_blocks = (h->nbin + kBinsPerBlock - 1) / kBinsPerBlock;
  int prev = 0;
  cudaGetDevice(&prev);
  cudaSetDevice(device);
  int &nsm = h->nsm, occ = 0;
  cudaError_t e = cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, device);
  // the kernels for any N always (they also take calls whose buffers are not 16-byte
  // aligned), the size-specialised ones where they exist; both forward kernels run on the same grid
  if (e == cudaSuccess) {
    switch (bits) {
      case 1: e = adj_prepare<1>(h, &occ); break;
      case 2: e = adj_prepare<2>(h, &occ); break;
      case 4: e = adj_prepare<4>(h, &occ); break;
      default: e = adj_prepare<8>(h, &occ); break;
    }
  }
  int window_ctas = 0;
  if (e == cudaSuccess && h->sized) {
    e = adj_sized_prepare(h->log2n, bits, &window_ctas);
    occ = std::min(occ, 1);
  }
  if (e != cudaSuccess || occ < 1) {
    cudaGetLastError();
    cudaSetDevice(prev);
    delete h;
    return adj_err(nullptr, POLARIS_ECUDA, "adjoint kernels cannot be launched: ",
                   e != cudaSuccess ? cudaGetErrorString(e) : "zero occupancy");
  }
  h->grid_max = nsm * std::min(occ, kMaxCtasPerSm);
  if (h->log2n < kAdjSizedMin) window_ctas = kSmallWindowCtas;
  h->grid_window = std::max(h->grid_max, nsm * window_ctas);
  // per-pass twiddles of the Stockham passes (radix 16, then 2, 4 or 8): pass with Ns
  // points done and radix R keeps W_{Ns R}^{r k} at r Ns + k - 1 (1 <= r < R, k < Ns); the
  // offsets Ns - 1 telescope, so the N - 1 entries tile [0, N - 1) exactly
  std::vector<float2> tw(h->N);
  for (int Ns = 1; Ns < h->N;) {
    const int R = std::min(16, h->N / Ns);
    for (int r = 1; r < R; ++r)
      for (int k = 0; k < Ns; ++k) {
        const double ang = -2.0 * M_PI * (double)r * (double)k / (double)(Ns * R);
        tw[r * Ns + k - 1] = make_float2((float)std::cos(ang), (float)std::sin(ang));
      }
    Ns *= R;
  }
  // one allocation for all of them (each costs the caller's program tens of microseconds)
  size_t total = 0;
  auto take = [&](size_t bytes) {
    const size_t at = total;
    total += (bytes + 255) & ~(size_t)255;
    return at;
  };
  const size_t at_part = take((size_t)h->grid_max * h->nbin * sizeof(float4));
  const size_t at_gpart = take((size_t)h->grid_window * h->N * sizeof(float));
  const size_t at_mat = take((size_t)h->nbin * sizeof(float4));
  const size_t at_bpart = take((size_t)h->bin_blocks * 5 * sizeof(double));
  const size_t at_tw = take(tw.size() * sizeof(float2));
  bool ok = cudaMalloc((void**)&h->d_all, total) == cudaSuccess;
  if (ok) {
    h->d_part = reinterpret_cast<float4*>(h->d_all + at_part);
    h->d_gpart = reinterpret_cast<float*>(h->d_all + at_gpart);
    h->d_mat = reinterpret_cast<float4*>(h->d_all + at_mat);
    h->d_bpart = reinterpret_cast<double*>(h->d_all + at_bpart);
    h->d_tw = reinterpret_cast<float2*>(h->d_all + at_tw);
    ok = cudaMemcpy(h->d_tw, tw.data(), tw.size() * sizeof(float2), cudaMemcpyHostToDevice) == cudaSuccess;
  }
  if (!ok) {
    cudaGetLastError();
    adj_free(h);
    cudaSetDevice(prev);
    delete h;
    return adj_err(nullptr, POLARIS_ENOMEM, "device allocation failed");
  }
  cudaSetDevice(prev);
  *out = h;
  return POLARIS_OK;
}

extern "C" void polaris_adj_destroy(polaris_adj* h) {
  if (!h) return;
  int prev = 0;
  cudaGetDevice(&prev);
  cudaSetDevice(h->device);
  adj_free(h);
  cudaSetDevice(prev);
  delete h;
}

extern "C" const char* polaris_adj_last_error(const polaris_adj* h) {
  return h ? h->err.c_str() : g_adj_create_err.c_str();
}

template <int BITS>
static cudaError_t adj_segments(const AdjArgs& a, size_t smem, bool window_pass, cudaStream_t st) {
  if (!window_pass) k_adj_forward<BITS><<<a.grid, a.threads, smem, st>>>(a);
  else k_adj_window<BITS><<<a.grid, a.threads, smem, st>>>(a);
  return cudaGetLastError();
}

template <int LOGN, int BITS>
static cudaError_t adj_small(const AdjArgs& a, bool window_pass, cudaStream_t st) {
  if (window_pass) return launch_dependent(k_adjm_window<LOGN, BITS>, a.grid, kSmallWindow, 0, st, a);
  return launch_dependent(k_adjm_forward<LOGN, BITS>, a.grid, kSmallForward, 0, st, a);
}
template <int BITS>
static cudaError_t adj_small_any(const AdjArgs& a, bool window_pass, cudaStream_t st) {
  switch (a.log2n) {
    case 5: return adj_small<5, BITS>(a, window_pass, st);
    case 6: return adj_small<6, BITS>(a, window_pass, st);
    case 7: return adj_small<7, BITS>(a, window_pass, st);
    default: return adj_small<8, BITS>(a, window_pass, st);
  }
}

static cudaError_t adj_segments_bits(int bits, const AdjArgs& a, size_t smem, bool window_pass, bool sized,
                                     cudaStream_t st) {
  if (a.log2n < kAdjSizedMin) {
    switch (bits) {
      case 1: return adj_small_any<1>(a, window_pass, st);
      case 2: return adj_small_any<2>(a, window_pass, st);
      case 4: return adj_small_any<4>(a, window_pass, st);
      default: return adj_small_any<8>(a, window_pass, st);
    }
  }
  if (sized) return adj_sized_launch(a.log2n, bits, window_pass, a, st);
  switch (bits) {
    case 1: return adj_segments<1>(a, smem, window_pass, st);
    case 2: return adj_segments<2>(a, smem, window_pass, st);
    case 4: return adj_segments<4>(a, smem, window_pass, st);
    default: return adj_segments<8>(a, smem, window_pass, st);
  }
}

extern "C" int polaris_adj_run(polaris_adj* h, const void* const* packed, int64_t n_samples, const float* window,
                               const float* gains, const float* leak, const float* target, float* stokes,
                               double* loss, float* grad_window, float* grad_gains, float* grad_leak,
                               void* cuda_stream) {
  if (!h) return POLARIS_EINVAL;
  if (!packed || !packed[0] || !packed[1] || !window || !gains || !leak)
    return adj_err(h, POLARIS_EINVAL, "null input pointer");
  if (n_samples < h->N || n_samples % h->N)
    return adj_err(h, POLARIS_EINVAL, "n_samples must be a positive multiple of n_fft (whole segments, hop = n_fft)");
  if (n_samples / h->N > 0x7fffffff) return adj_err(h, POLARIS_EINVAL, "too many segments");
  const bool grads = grad_window || grad_gains || grad_leak;
  if ((grads || loss) && !target) return adj_err(h, POLARIS_EINVAL, "loss and gradients need a target");
  if (grads && !(grad_window && grad_gains && grad_leak))
    return adj_err(h, POLARIS_EINVAL, "gradients come as a set: grad_window, grad_gains and grad_leak");
  int prev = 0;
  cudaGetDevice(&prev);
  cudaSetDevice(h->device);
  cudaStream_t st = reinterpret_cast<cudaStream_t>(cuda_stream);
  AdjArgs a;
  memset(&a, 0, sizeof a);
  a.in[0] = static_cast<const uint32_t*>(packed[0]);
  a.in[1] = static_cast<const uint32_t*>(packed[1]);
  a.N = h->N;
  a.log2n = h->log2n;
  a.nbin = h->nbin;
  a.nseg = (int)(n_samples / h->N);
  a.grid = std::min(a.nseg, h->grid_max);
  a.threads = h->threads;
  a.tw = h->d_tw;
  a.window = window;
  a.part = h->d_part;
  a.mat = h->d_mat;
  a.gpart = h->d_gpart;
  // the size-specialised kernels read the inputs and the window by 16-byte vector loads
  auto aligned16 = [](const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; };
  const bool sized = h->sized && aligned16(packed[0]) && aligned16(packed[1]) && aligned16(window);
  cudaError_t e = adj_segments_bits(h->bits, a, h->smem, false, sized, st);
  if (e == cudaSuccess) {
    BinArgs b;
    b.part = h->d_part;
    b.grid = a.grid;
    b.nbin = h->nbin;
    b.gains = gains;
    b.leak = leak;
    b.target = target;
    b.stokes = stokes;
    b.grad_leak = grads ? grad_leak : nullptr;
    b.mat = grads ? h->d_mat : nullptr;
    b.bpart = (loss || grads) ? h->d_bpart : nullptr;
    e = launch_dependent(k_adj_bins, h->bin_blocks, kBinsPerBlock * kSlices, 0, st, b);
  }
  if (e == cudaSuccess && grads) {
    if (sized) a.grid = std::min(a.nseg, h->grid_window);
    if (h->log2n < kAdjSizedMin) {  // a segment per team
      const int teams = kSmallWindow * 16 / h->N;
      a.grid = std::min((a.nseg + teams - 1) / teams, h->nsm * kSmallWindowCtas);
    }
    e = adj_segments_bits(h->bits, a, h->smem, true, sized, st);
    if (e == cudaSuccess)
      e = launch_dependent(k_adj_wsum, (h->N + kBinsPerBlock - 1) / kBinsPerBlock + 1, kBinsPerBlock * kSlices, 0, st, h->d_gpart,
                     a.grid, h->N, grad_window, h->d_bpart, h->bin_blocks, loss, grad_gains);
  } else if (e == cudaSuccess && loss) {
    e = launch_dependent(k_adj_finish, 1, 160, 0, st, h->d_bpart, h->bin_blocks, loss);
  }
  cudaSetDevice(prev);
  if (e != cudaSuccess) return adj_err(h, POLARIS_ECUDA, "CUDA: ", cudaGetErrorString(e));
  return POLARIS_OK;
}
