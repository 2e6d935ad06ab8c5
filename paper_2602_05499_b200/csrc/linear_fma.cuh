// CUDA-core linear kernel: Y = [RMSNorm](X) · Wᵀ with a fused epilogue.
//
// Used for fp32 models (the tiny configuration) and, on request, for bf16 models as
// the comparison path of the tensor-core kernel.  Weights are stored pair-major,
// W[pair][2][K] (see EpiMode in common.cuh for what a pair is).
//
// A CTA takes eight rows and 8 P pairs.  The rows are brought into shared memory once for all its warps
// (normalised there), a warp owns P pairs and sweeps K with its lanes, 128-bit loads, and the lanes' sums
// are added in the fixed xor tree.  What bounds it: at a few rows the chain of round trips from the
// previous kernel's end to this one's (the weights of the first steps are therefore asked for before
// the wait), at many rows the FMAs.  When every warp read the rows from L2 itself and re-read its weights for
// every eight rows, that traffic cost more than either: speculative decoding of 16 sequences, 6 layers d 768,
// FFN 2352, vocabulary 8192, k = 4: 147 -> 24.5 ms; of one, 4 layers d 256: 10.5 -> 7.0 ms.
// A row's result does not depend on how many rows the launch carries or on P: every (row, feature) runs
// the same additions in the same order.
#pragma once

#include "common.cuh"

namespace sdfp {

constexpr int kFmaThreads = 256;
constexpr int kFmaWarps = kFmaThreads / 32;
constexpr int kFmaRows = 8;      // rows of a CTA
constexpr int kFmaCols = 1024;   // columns staged at a time (32 KB of rows)
constexpr int kFmaAhead = 2;     // k steps (128 columns) whose weights are requested before the wait on the preceding kernel

// Sum over the warp of N values per lane, N = 2, 4, ... 32: value i ends in the lanes with (lane * N / 32) == i (returned).
// Each value is added in the xor tree of warp_sum; halving the values with the lanes takes N - 1 + log2(32 / N)
// shuffles instead of 5 N.
template <int N>
__device__ __forceinline__ float warp_sum_scatter(float (&v)[N]) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int o = 16, n = N; o > 0; o >>= 1) {
    if (n > 1) {
      n >>= 1;
      const bool up = (lane & o) != 0;  // this lane keeps the upper half of the values
#pragma unroll
      for (int i = 0; i < N / 2; ++i)
        if (i < n) {
          const float keep = up ? v[i + n] : v[i], give = up ? v[i] : v[i + n];
          v[i] = keep + __shfl_xor_sync(0xffffffffu, give, o);
        }
    } else {
      v[0] += __shfl_xor_sync(0xffffffffu, v[0], o);
    }
  }
  return v[0];
}

// Four weights as they lie in memory.  A load that is converted where it is issued is waited for there: with bf16
// weights nothing was in flight then, and a wide matrix was slower than with fp32 ones.
template <typename WT>
struct Raw4;
template <>
struct Raw4<float> {
  float4 v;
  __device__ __forceinline__ void load(const float* p, bool in) { v = in ? *reinterpret_cast<const float4*>(p) : make_float4(0.f, 0.f, 0.f, 0.f); }
  __device__ __forceinline__ float4 get() const { return v; }
};
template <>
struct Raw4<__nv_bfloat16> {
  uint2 v;
  __device__ __forceinline__ void load(const __nv_bfloat16* p, bool in) { v = in ? *reinterpret_cast<const uint2*>(p) : make_uint2(0u, 0u); }
  __device__ __forceinline__ float4 get() const {
    return make_float4(__uint_as_float(v.x << 16), __uint_as_float(v.x & 0xffff0000u), __uint_as_float(v.y << 16), __uint_as_float(v.y & 0xffff0000u));
  }
};

// P pairs per warp, 1 or 2.  Registers leave room for three CTAs on an SM with one pair and for two with two.
template <typename WT, typename KT, int P>
__global__ void __launch_bounds__(kFmaThreads, 4 - P)
linear_fma_kernel(const WT* __restrict__ W, const float* __restrict__ X, int ldx, int M, int K, int n_pairs,
                  const float* __restrict__ gain, float eps, EpiParams ep) {
  __shared__ __align__(16) float xs[kFmaRows][kFmaCols];
  __shared__ float s_inv[kFmaRows];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int m0 = blockIdx.y * kFmaRows, rows = min(kFmaRows, M - m0);
  const int p0 = (blockIdx.x * kFmaWarps + warp) * P;  // this warp's first pair
  const WT* wp[P][2];
#pragma unroll
  for (int j = 0; j < P; ++j) {  // pairs beyond the last repeat it; their sums are not used
    wp[j][0] = W + (size_t)min(p0 + j, n_pairs - 1) * 2 * K;
    wp[j][1] = wp[j][0] + K;
  }
  Raw4<WT> wq[kFmaAhead][P][2];
#pragma unroll
  for (int a = 0; a < kFmaAhead; ++a) {
    const int k = a * 128 + lane * 4;
#pragma unroll
    for (int j = 0; j < P; ++j)
#pragma unroll
      for (int h = 0; h < 2; ++h) wq[a][j][h].load(wp[j][h] + k, k < K);
  }
  pdl_wait();
  pdl_launch_dependents();
  if (gain != nullptr && K > kFmaCols) {  // rows that do not fit: their norm first
    if (warp < rows) {
      const float* x = X + (size_t)(m0 + warp) * ldx;
      float s = 0.f;
      for (int k = lane * 4; k < K; k += 128) {
        const float4 v = ld_act4(x + k);
        s = fmaf(v.x, v.x, s);
        s = fmaf(v.y, v.y, s);
        s = fmaf(v.z, v.z, s);
        s = fmaf(v.w, v.w, s);
      }
      s = warp_sum(s);
      if (lane == 0) s_inv[warp] = rsqrtf(s / (float)K + eps);
    }
  }
  float acc[kFmaRows * P * 2];  // [row][pair][half]
#pragma unroll
  for (int i = 0; i < kFmaRows * P * 2; ++i) acc[i] = 0.f;
  for (int c0 = 0; c0 < K; c0 += kFmaCols) {
    const int nc = min(kFmaCols, K - c0);
    __syncthreads();  // the previous columns are no longer read (and s_inv is written)
    // warp r stages row r, each lane the columns it will read itself
    if (warp < rows) {
      const float* x = X + (size_t)(m0 + warp) * ldx + c0;
      float s = 0.f;
#pragma unroll 4
      for (int k = lane * 4; k < nc; k += 128) {
        const float4 v = ld_act4(x + k);
        *reinterpret_cast<float4*>(&xs[warp][k]) = v;
        s = fmaf(v.x, v.x, s);
        s = fmaf(v.y, v.y, s);
        s = fmaf(v.z, v.z, s);
        s = fmaf(v.w, v.w, s);
      }
      if (gain != nullptr) {
        float r;
        if (K <= kFmaCols)
          r = rsqrtf(warp_sum(s) / (float)K + eps);
        else
          r = s_inv[warp];
        for (int k = lane * 4; k < nc; k += 128) {
          float4 v = *reinterpret_cast<const float4*>(&xs[warp][k]);
          const float4 g = load4(gain + c0 + k);
          v.x = v.x * r * g.x;
          v.y = v.y * r * g.y;
          v.z = v.z * r * g.z;
          v.w = v.w * r * g.w;
          *reinterpret_cast<float4*>(&xs[warp][k]) = v;
        }
      }
    } else {
      for (int k = lane * 4; k < nc; k += 128) *reinterpret_cast<float4*>(&xs[warp][k]) = make_float4(0.f, 0.f, 0.f, 0.f);
    }
    __syncthreads();
    for (int k = lane * 4; k < nc; k += 128) {
      const int kg = c0 + k;
      float4 w[P][2];
#pragma unroll
      for (int j = 0; j < P; ++j)
#pragma unroll
        for (int h = 0; h < 2; ++h) w[j][h] = wq[0][j][h].get();
#pragma unroll
      for (int a = 0; a + 1 < kFmaAhead; ++a)
#pragma unroll
        for (int j = 0; j < P; ++j)
#pragma unroll
          for (int h = 0; h < 2; ++h) wq[a][j][h] = wq[a + 1][j][h];
      const int kn = kg + kFmaAhead * 128;
#pragma unroll
      for (int j = 0; j < P; ++j)
#pragma unroll
        for (int h = 0; h < 2; ++h) wq[kFmaAhead - 1][j][h].load(wp[j][h] + kn, kn < K);
#pragma unroll
      for (int i = 0; i < kFmaRows; ++i) {
        if (i < rows) {
          const float4 x = *reinterpret_cast<const float4*>(&xs[i][k]);
#pragma unroll
          for (int j = 0; j < P; ++j)
#pragma unroll
            for (int h = 0; h < 2; ++h) {
              float& a = acc[(i * P + j) * 2 + h];
              a = fmaf(w[j][h].x, x.x, a);
              a = fmaf(w[j][h].y, x.y, a);
              a = fmaf(w[j][h].z, x.z, a);
              a = fmaf(w[j][h].w, x.w, a);
            }
        }
      }
    }
  }
  // lane groups end up with one (row, pair, half) each; the two halves of a pair sit next to each other
#pragma unroll
  for (int b = 0; b < kFmaRows * P * 2; b += 16) {
    float part[16];
#pragma unroll
    for (int i = 0; i < 16; ++i) part[i] = acc[b + i];
    const float mine = warp_sum_scatter<16>(part);  // value lane / 2
    const float other = __shfl_xor_sync(0xffffffffu, mine, 2);
    const int v = (b + (lane >> 1)) >> 1, row = v / P, pair = p0 + v % P;
    if ((lane & 3) == 0 && row < rows && pair < n_pairs) apply_epilogue<KT>(ep, pair, m0 + row, mine, other);
  }
}

// ---- packing: caller's row-major [out, in] matrices -> pair-major ----------------
// src row of (pair p, half r):
//   kind 0 (QKV)    three sources q, k, v of [d, d]
//   kind 1 (GATEUP) two sources gate, up of [f, d]: pair j = (gate_j, up_j)
//   kind 2 (PLAIN)  one source: rows 16*(p/8) + p%8 (+8)
struct PackSrc {
  const void* s0;
  const void* s1;
  const void* s2;
  int kind;
  int n_heads, head_dim;
};

template <typename WT>
__device__ __forceinline__ const WT* pack_src_row(const PackSrc& ps, int p, int r, int K) {
  if (ps.kind == 0) {
    const int hp = ps.head_dim >> 1;
    const int per_tensor = ps.n_heads * hp;
    const int t = p / per_tensor;
    const int rem = p - t * per_tensor;
    const int head = rem / hp;
    const int i = rem - head * hp;
    const WT* base = reinterpret_cast<const WT*>(t == 0 ? ps.s0 : (t == 1 ? ps.s1 : ps.s2));
    return base + (size_t)(head * ps.head_dim + i + r * hp) * K;
  } else if (ps.kind == 1) {
    const WT* base = reinterpret_cast<const WT*>(r == 0 ? ps.s0 : ps.s1);
    return base + (size_t)p * K;
  }
  return reinterpret_cast<const WT*>(ps.s0) + (size_t)(((p >> 3) << 4) + (p & 7) + 8 * r) * K;
}

template <typename WT>
__global__ void pack_pairs_kernel(WT* __restrict__ dst, PackSrc ps, int n_pairs, int K) {
  const size_t total = (size_t)n_pairs * 2 * K;
  for (size_t idx = (size_t)blockIdx.x * blockDim.x + threadIdx.x; idx < total;
       idx += (size_t)gridDim.x * blockDim.x) {
    const int k = (int)(idx % K);
    const size_t pr = idx / K;
    const int r = (int)(pr & 1);
    const int p = (int)(pr >> 1);
    dst[idx] = pack_src_row<WT>(ps, p, r, K)[k];
  }
}

template <typename WT>
__global__ void widen_vector_kernel(float* __restrict__ dst, const WT* __restrict__ src, int n) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) dst[i] = to_f32(src[i]);
}

}  // namespace sdfp
