// Stage A of Algorithm 1 on the GPU: the per-layer empirical-Fisher trace
//   T_l = (1/N) sum_i || grad_{theta_l} f(z_i, theta) ||^2                     (Eq. 11; Eq. 8-9)
// and the layer-wise FIT form  FIT_l = sum_{tensors t of layer l} T_t * mean(theta_t^2)   (Eq. 7,
// with the perturbation of removing the layer read as delta theta = -theta).
//
// f(z_i, theta) is the mean next-token cross-entropy of one calibration sequence: one forward pass
// that keeps the activations, one backward pass that carries the gradient with respect to the
// ACTIVATIONS only.  The gradient of a weight matrix is never formed: for y = x W^T over T rows,
// dW = dY^T X, so
//   ||dW||_F^2 = sum_{t,t'} (dY dY^T)[t,t'] * (X X^T)[t,t']
// - two T x T Gram matrices and their elementwise dot product (T is a calibration sequence's
// length, tens of tokens), instead of an [out, in] matrix per weight.  A norm gain's gradient is a
// vector and is summed directly.
//
// Everything is fp32 on CUDA cores with fp64 accumulation of the squared norms; weights are read in
// their storage type (fp32 or bf16) from the caller's row-major [out, in] matrices.  The calibration
// sequences go through the stack together, up to kFitRows rows at a time: a GEMM then reads a weight
// once for all of them, and a layer costs the same number of launches whatever the set's size.
// Every reduction runs in an order fixed by the model, the sequences' length and how many of them make a full group
// (the set's size up to kFitRows rows), so the same call gives the same bits; a sequence scored in a set of
// another size may differ in the last places.
#pragma once

#include <cooperative_groups.h>

#include <algorithm>
#include <cmath>
#include <mutex>
#include <vector>

#include "../../include/sdfp.h"
#include "common.cuh"

namespace sdfp {
namespace fit {

namespace cg = cooperative_groups;

__device__ __forceinline__ float wload(const float* p) { return *p; }
__device__ __forceinline__ float wload(const __nv_bfloat16* p) { return __bfloat162float(*p); }

// ---- fp32 GEMM on the packed FMA pipe ---------------------------------------------------------------
// Bound by FMA issue at every size met here (a bf16 weight is used for 2 R flop per 2 bytes, R rows:
// the memory would feed 100 TFLOP/s at 16 rows already), so:
//   * fma.rn.f32x2: two fp32 FMAs per instruction, the same rounding as fmaf, half the issue slots;
//   * 8 columns x BM/16 rows per thread, 16 warps on an SM, operands k-major in shared memory so that a
//     fragment is one or two 128-bit loads; the next k step's global loads are in flight during the FMAs.
//     Shared memory hands a warp 128 bytes a clock whatever its lanes share, which at 8 x 8 is as many
//     clocks as the FMAs take.  All GEMMs of 4 layers + lm-head, d 4096, FFN 11008, vocabulary 32000, 128
//     rows, 482 GFLOP: 11.6 ms (42 TFLOP/s of 74); 16 x 8 per thread needs fewer reads but leaves 8 warps
//     on an SM: 14.4 ms; A stored as (a, a) pairs to save the packing: 18.5 ms, bound by the reads; the
//     scalar 4 x 4 kernel on 64 x 64 tiles, one sequence at a time, that this replaces: about 150 ms.
//     (Two CTAs on an SM leave 128 registers a thread; with BM 128 ptxas spills 8 to 24 bytes of loop state.)
//   * a contraction is cut into S pieces run by the S CTAs of a cluster when the tiles alone would
//     leave SMs idle; the pieces are added in piece order through distributed shared memory.
// The tensor cores are not an option at this precision: tcgen05.mma cuts every addend to two bits
// below the largest one's last place and truncates the sum, so even with activations in three bf16
// parts and the accumulator drained every 64 columns a GEMM comes out 1e-7 short on average, which the
// traces (within 5e-8 of 64-bit sums here) would show.
constexpr int kGN = 128, kGK = 16, kGThreads = 256;
constexpr int kGLdW = kGN + 4;

__device__ __forceinline__ void fma2(unsigned long long& d, unsigned long long a, unsigned long long b) {
  asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(d) : "l"(a), "l"(b));
}
__device__ __forceinline__ unsigned long long pack2(float x, float y) {
  unsigned long long r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(x), "f"(y));
  return r;
}
__device__ __forceinline__ float2 unpack2(unsigned long long v) {
  float2 r;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(v));
  return r;
}

// Up to three matrices in one launch.
//   NT (forward):  C_p[R, N] = add + A[R, K] W_p[N, K]^T, one group of column tiles per matrix
//   NN (backward): C[R, K] = sum_p A_p[R, N] W_p[N, K], contractions one after the other
struct GemmArgs {
  const float* A[3];
  const void* W[3];
  float* C[3];
  const float* add;  // NT: added to the result (the residual stream), or null
  int R, N, K, parts;
};

// eight consecutive values of a row, as loaded and as floats; entries at or beyond `left` are zero
template <typename WT, bool VEC>
struct Row8;
template <>
struct Row8<float, true> {
  float4 a, b;
  __device__ __forceinline__ void load(const float* p, int left) {
    a = left > 0 ? *reinterpret_cast<const float4*>(p) : make_float4(0.f, 0.f, 0.f, 0.f);
    b = left > 4 ? *reinterpret_cast<const float4*>(p + 4) : make_float4(0.f, 0.f, 0.f, 0.f);
  }
  __device__ __forceinline__ void get(float (&v)[8]) const {
    v[0] = a.x; v[1] = a.y; v[2] = a.z; v[3] = a.w; v[4] = b.x; v[5] = b.y; v[6] = b.z; v[7] = b.w;
  }
};
template <>
struct Row8<__nv_bfloat16, true> {
  uint4 r;
  __device__ __forceinline__ void load(const __nv_bfloat16* p, int left) {
    r = left > 0 ? *reinterpret_cast<const uint4*>(p) : make_uint4(0u, 0u, 0u, 0u);
  }
  __device__ __forceinline__ void get(float (&v)[8]) const {
    const unsigned w[4] = {r.x, r.y, r.z, r.w};
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      v[2 * i] = __uint_as_float(w[i] << 16);
      v[2 * i + 1] = __uint_as_float(w[i] & 0xffff0000u);
    }
  }
};
template <typename WT>
struct Row8<WT, false> {  // any length, any alignment
  float f[8];
  __device__ __forceinline__ void load(const WT* p, int left) {
#pragma unroll
    for (int i = 0; i < 8; ++i) f[i] = i < left ? wload(p + i) : 0.f;
  }
  __device__ __forceinline__ void get(float (&v)[8]) const {
#pragma unroll
    for (int i = 0; i < 8; ++i) v[i] = f[i];
  }
};

template <int BM>
constexpr size_t gemm_smem_bytes() {  // two k steps of both operands; the split's partial tile takes their place at the end
  return (size_t)std::max(2 * kGK * ((BM + 4) + kGLdW), BM * kGN) * sizeof(float);
}

// VEC: rows of W (and, NN, of A) are whole 16-byte pieces at 16-byte addresses; A is always the library's own buffer.
template <typename WT, int BM, bool NT, bool VEC>
__global__ void __launch_bounds__(kGThreads, 2) fit_gemm_kernel(const __grid_constant__ GemmArgs g) {
  constexpr int RT = BM / 16;    // rows per thread
  constexpr int LdA = BM + 4;
  constexpr int AV = BM * kGK / 8;  // eight-value pieces of A per k step
  extern __shared__ __align__(16) float sm[];
  float* sA = sm;                    // [2][kGK][LdA]
  float* sW = sm + 2 * kGK * LdA;    // [2][kGK][kGLdW]
  const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
  const int S = gridDim.z, piece = blockIdx.z;
  const int cols = NT ? g.N : g.K;                    // columns of one output matrix
  const int inner = NT ? g.K : g.N;                   // contraction length of one part
  const int tiles = (cols + kGN - 1) / kGN;
  const int part0 = NT ? blockIdx.x / tiles : 0;
  const int c0 = (NT ? blockIdx.x - part0 * tiles : blockIdx.x) * kGN, r0 = blockIdx.y * BM;
  const int per_part = (inner + kGK - 1) / kGK;       // k steps of one part
  const int steps = NT ? per_part : per_part * g.parts;
  const int s_lo = (int)((long long)steps * piece / S), s_hi = (int)((long long)steps * (piece + 1) / S);

  Row8<float, VEC> ra;
  Row8<WT, VEC> rw;
  const int ar = tid >> 1, ak = (tid & 1) * 8;                      // A: row of the tile, k offset (threads below AV)
  const int wr = NT ? tid >> 1 : tid >> 4, wc = NT ? (tid & 1) * 8 : (tid & 15) * 8;  // W: NT (column, k) / NN (k, column)
  auto fetch = [&](int s) {
    const int part = NT ? part0 : s / per_part;
    const int k0 = (NT ? s : s - part * per_part) * kGK;
    const float* A = g.A[NT ? 0 : part];
    const WT* W = reinterpret_cast<const WT*>(g.W[part]);
    if (tid < AV) ra.load(A + (size_t)(r0 + ar) * inner + k0 + ak, r0 + ar < g.R ? inner - k0 - ak : 0);
    if (NT)
      rw.load(W + (size_t)(c0 + wr) * inner + k0 + wc, c0 + wr < cols ? inner - k0 - wc : 0);
    else
      rw.load(W + (size_t)(k0 + wr) * cols + c0 + wc, k0 + wr < inner ? cols - c0 - wc : 0);
  };
  auto stage = [&](int buf) {
    float v[8];
    if (tid < AV) {
      ra.get(v);
      float* d = sA + buf * kGK * LdA + ak * LdA + ar;
#pragma unroll
      for (int i = 0; i < 8; ++i) d[i * LdA] = v[i];
    }
    rw.get(v);
    float* d = sW + buf * kGK * kGLdW;
    if (NT) {
#pragma unroll
      for (int i = 0; i < 8; ++i) d[(wc + i) * kGLdW + wr] = v[i];
    } else {
      *reinterpret_cast<float4*>(d + wr * kGLdW + wc) = make_float4(v[0], v[1], v[2], v[3]);
      *reinterpret_cast<float4*>(d + wr * kGLdW + wc + 4) = make_float4(v[4], v[5], v[6], v[7]);
    }
  };

  // thread (ty, tx): rows ty*4.. (+64 for the second four; BM 32: ty*2, +1), columns tx*4.. and 64 + tx*4..
  unsigned long long acc[RT][4];
#pragma unroll
  for (int i = 0; i < RT; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) acc[i][j] = 0ull;
  if (s_lo < s_hi) {
    fetch(s_lo);
    stage(0);
  }
  __syncthreads();
  for (int s = s_lo; s < s_hi; ++s) {
    const int buf = (s - s_lo) & 1;
    if (s + 1 < s_hi) fetch(s + 1);
    const float* a_ = sA + buf * kGK * LdA;
    const float* w_ = sW + buf * kGK * kGLdW;
#pragma unroll
    for (int kk = 0; kk < kGK; ++kk) {
      float a[RT];
      if constexpr (RT == 2) {
        const float2 t = *reinterpret_cast<const float2*>(a_ + kk * LdA + ty * 2);
        a[0] = t.x; a[1] = t.y;
      } else {
#pragma unroll
        for (int h = 0; h < RT / 4; ++h) {
          const float4 t = *reinterpret_cast<const float4*>(a_ + kk * LdA + h * 64 + ty * 4);
          a[4 * h] = t.x; a[4 * h + 1] = t.y; a[4 * h + 2] = t.z; a[4 * h + 3] = t.w;
        }
      }
      const ulonglong2 b0 = *reinterpret_cast<const ulonglong2*>(w_ + kk * kGLdW + tx * 4);
      const ulonglong2 b1 = *reinterpret_cast<const ulonglong2*>(w_ + kk * kGLdW + 64 + tx * 4);
#pragma unroll
      for (int i = 0; i < RT; ++i) {
        const unsigned long long aa = pack2(a[i], a[i]);
        fma2(acc[i][0], aa, b0.x);
        fma2(acc[i][1], aa, b0.y);
        fma2(acc[i][2], aa, b1.x);
        fma2(acc[i][3], aa, b1.y);
      }
    }
    if (s + 1 < s_hi) stage(buf ^ 1);
    __syncthreads();
  }

  auto row_of = [&](int i) { return RT == 2 ? ty * 2 + i : (i >> 2) * 64 + ty * 4 + (i & 3); };
  auto put = [&](int r, int c, float v) {  // (row, column) of the tile
    if (r0 + r >= g.R || c0 + c >= cols) return;
    const size_t o = (size_t)(r0 + r) * cols + c0 + c;
    g.C[part0][o] = g.add != nullptr ? g.add[o] + v : v;
  };
  if (S == 1) {
#pragma unroll
    for (int i = 0; i < RT; ++i)
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const float2 v = unpack2(acc[i][j]);
        const int c = (j >> 1) * 64 + tx * 4 + (j & 1) * 2;
        put(row_of(i), c, v.x);
        put(row_of(i), c + 1, v.y);
      }
    return;
  }
  // split contraction: every CTA leaves its tile in its own shared memory, CTA z adds rows z, z + S, ...
#pragma unroll
  for (int i = 0; i < RT; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j)
      *reinterpret_cast<unsigned long long*>(sm + row_of(i) * kGN + (j >> 1) * 64 + tx * 4 + (j & 1) * 2) = acc[i][j];
  cg::cluster_group cluster = cg::this_cluster();
  cluster.sync();
  for (int e = tid; e < BM * kGN; e += kGThreads) {
    const int r = (e / kGN) * S + piece, c = e % kGN;
    if (r >= BM) break;
    float v = 0.f;
    for (int z = 0; z < S; ++z) v += cluster.map_shared_rank(sm, z)[r * kGN + c];
    put(r, c, v);
  }
  cluster.sync();  // nobody leaves while its tile is still being read
}

// fixed-order block sum (blockDim.x a multiple of 32, at most 1024); every thread gets the result
__device__ __forceinline__ double block_sum_d(double v, double* s_red) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  __syncthreads();
  if ((threadIdx.x & 31) == 0) s_red[threadIdx.x >> 5] = v;
  __syncthreads();
  double r = 0.0;
  for (int w = 0; w < (int)(blockDim.x >> 5); ++w) r += s_red[w];
  return r;
}

// h[r, :] = E[token, :], row r = token t of sequence r / T
template <typename WT>
__global__ void embed_kernel(const int* __restrict__ tok, const WT* __restrict__ E, float* __restrict__ h, int d, int T, int seq_len) {
  const int r = blockIdx.x, s = r / T, y = tok[s * seq_len + r - s * T];
  for (int k = threadIdx.x; k < d; k += blockDim.x) h[(size_t)r * d + k] = wload(E + (size_t)y * d + k);
}

// y = x * r * g with r = 1/sqrt(mean(x^2) + eps); keeps r per row
template <typename WT>
__global__ void __launch_bounds__(512) rmsnorm_fwd_kernel(const float* __restrict__ x, const WT* __restrict__ g, float* __restrict__ y,
                                                           float* __restrict__ inv, int d, float eps) {
  __shared__ double s_red[16];
  const int t = blockIdx.x;
  double s = 0.0;
  for (int k = threadIdx.x; k < d; k += blockDim.x) {
    const double v = x[(size_t)t * d + k];
    s += v * v;
  }
  const double tot = block_sum_d(s, s_red);
  const float r = (float)(1.0 / sqrt(tot / d + (double)eps));
  if (threadIdx.x == 0) inv[t] = r;
  for (int k = threadIdx.x; k < d; k += blockDim.x) y[(size_t)t * d + k] = x[(size_t)t * d + k] * r * wload(g + k);
}

// Given dy: dx = add + r z - x r^3 mean(z x) with z = g * dy (add may be null); dgain[k] = sum_t dy[t,k] x[t,k] r[t]
// is taken by gain_grad_sq_kernel below.
template <typename WT>
__global__ void __launch_bounds__(512) rmsnorm_bwd_kernel(const float* __restrict__ dy, const float* __restrict__ x,
                                                           const WT* __restrict__ g, const float* __restrict__ inv,
                                                           const float* __restrict__ add, float* __restrict__ dx, int d) {
  __shared__ double s_red[16];
  const int t = blockIdx.x;
  const float r = inv[t];
  double s = 0.0;
  for (int k = threadIdx.x; k < d; k += blockDim.x)
    s += (double)(wload(g + k) * dy[(size_t)t * d + k]) * (double)x[(size_t)t * d + k];
  const float mzx = (float)(block_sum_d(s, s_red) / d);
  for (int k = threadIdx.x; k < d; k += blockDim.x) {
    const size_t i = (size_t)t * d + k;
    const float v = r * wload(g + k) * dy[i] - x[i] * r * r * r * mzx;
    dx[i] = (add != nullptr ? add[i] : 0.f) + v;
  }
}

// || sum_t dy[t,:] * x[t,:] * r[t] ||^2, the squared norm of a gain's gradient for one sequence: block
// (32 columns, sequence), thread group g of 32 takes the rows g, g + 8, ..., adds its share to its slot
constexpr int kGainCols = 32;
__global__ void __launch_bounds__(256) gain_grad_sq_kernel(const float* __restrict__ dy, const float* __restrict__ x,
                                                            const float* __restrict__ inv, int T, int d, double* slots) {
  __shared__ double s_g[8][kGainCols];
  const int lane = threadIdx.x & 31, grp = threadIdx.x >> 5, k = blockIdx.x * kGainCols + lane;
  const size_t r0 = (size_t)blockIdx.y * T;
  double gk = 0.0;
  if (k < d) {
#pragma unroll 4
    for (int t = grp; t < T; t += 8) gk += (double)dy[(r0 + t) * d + k] * (double)x[(r0 + t) * d + k] * (double)inv[r0 + t];
  }
  s_g[grp][lane] = gk;
  __syncthreads();
  if (grp == 0) {
    double v = 0.0;
#pragma unroll
    for (int i = 0; i < 8; ++i) v += s_g[i][lane];
    v *= v;
#pragma unroll
    for (int w = 16; w > 0; w >>= 1) v += __shfl_xor_sync(0xffffffffu, v, w);
    if (lane == 0) slots[blockIdx.y * gridDim.x + blockIdx.x] += v;
  }
}

// cos and sin of the rotary angles of positions 0..T-1 in fp64, rounded to fp32: [T][hd/2]
__global__ void rope_table_kernel(float* __restrict__ cs, float* __restrict__ sn, int T, int hd, double theta) {
  const int e = blockIdx.x * blockDim.x + threadIdx.x, hp = hd >> 1;
  if (e >= T * hp) return;
  const int t = e / hp, i = e - t * hp;
  const double a = t * pow(theta, -2.0 * i / hd);
  cs[e] = (float)cos(a);
  sn[e] = (float)sin(a);
}

// Rotary embedding of q and k (blockIdx.y) in place, pairs (i, i + hd/2) of every head; dir = +1 forward, -1
// the transpose (the backward pass: the rotation is orthogonal).  cs, sn: [T][hd/2], positions 0..T-1.
__global__ void rope_kernel(float* __restrict__ xq, float* __restrict__ xk, const float* __restrict__ cs, const float* __restrict__ sn,
                            int T, int n_heads, int hd, float dir) {
  const int r = blockIdx.x, t = r % T, hp = hd >> 1;
  float* x = blockIdx.y ? xk : xq;
  for (int e = threadIdx.x; e < n_heads * hp; e += blockDim.x) {
    const int h = e / hp, i = e - h * hp;
    float* p = x + (size_t)r * n_heads * hd + h * hd;
    const float c = cs[t * hp + i], s = dir * sn[t * hp + i];
    const float a = p[i], b = p[i + hp];
    p[i] = a * c - b * s;
    p[i + hp] = b * c + a * s;
  }
}

// ---- causal attention -----------------------------------------------------------------------------------
// A block takes kAtQ consecutive queries of one head of one sequence (grid: query group, head, sequence),
// so that a key or value row is read once for all of them; sums run over the keys in order.
constexpr int kAtQ = 8, kAtThreads = 128, kAtKeys = 32, kAtDim = 64;
constexpr int kFitMaxT = 4096;  // positions of the longest sequence the entry point accepts

inline size_t attn_smem(int T) { return (size_t)(kAtQ * T + kAtQ * kAtDim + kAtKeys * (kAtDim + 1)) * sizeof(float); }

// s[i][j] = x_{t0+i} . y_j for the keys j <= t0 + i (others untouched); x, y: rows of one head, ld apart
__device__ __forceinline__ void attn_scores(const float* x, const float* y, float* s, float* sx, float* sy, int T, int t0, int nq,
                                            int hd, size_t ld) {
  const int tid = threadIdx.x, kl = tid & 31, i0 = (tid >> 5) * 2;  // key of the tile; queries i0 and i0 + 1
  for (int j0 = 0; j0 < t0 + nq; j0 += kAtKeys) {
    const int nk = min(kAtKeys, t0 + nq - j0);
    float a0 = 0.f, a1 = 0.f;
    for (int c0 = 0; c0 < hd; c0 += kAtDim) {
      const int nc = min(kAtDim, hd - c0);
      __syncthreads();
      for (int e = tid; e < nq * kAtDim; e += kAtThreads) {
        const int i = e / kAtDim, c = e % kAtDim;
        if (c < nc) sx[e] = x[(size_t)(t0 + i) * ld + c0 + c];
      }
      for (int e = tid; e < nk * kAtDim; e += kAtThreads) {
        const int j = e / kAtDim, c = e % kAtDim;
        if (c < nc) sy[j * (kAtDim + 1) + c] = y[(size_t)(j0 + j) * ld + c0 + c];
      }
      __syncthreads();
      if (kl < nk) {
#pragma unroll 8
        for (int c = 0; c < nc; ++c) {
          const float v = sy[kl * (kAtDim + 1) + c];
          a0 = fmaf(sx[i0 * kAtDim + c], v, a0);
          a1 = fmaf(sx[(i0 + 1) * kAtDim + c], v, a1);
        }
      }
    }
    const int j = j0 + kl;
    if (i0 < nq && j <= t0 + i0) s[i0 * T + j] = a0;
    if (i0 + 1 < nq && j <= t0 + i0 + 1) s[(i0 + 1) * T + j] = a1;
  }
  __syncthreads();
}

// out_{t0+i} = f * sum_{j <= t0+i} s[i][j] y_j, thread = dimension; s is zero beyond a query's own keys
__device__ __forceinline__ void attn_weighted_sum(const float* s, const float* y, float* out, int T, int t0, int nq, int hd, size_t ld, float f) {
  for (int c = threadIdx.x; c < hd; c += kAtThreads) {
    float o[kAtQ] = {};
    const int n = t0 + nq;
#pragma unroll 4
    for (int j = 0; j < n; ++j) {
      const float v = y[(size_t)j * ld + c];
#pragma unroll
      for (int i = 0; i < kAtQ; ++i) o[i] = fmaf(s[i * T + j], v, o[i]);
    }
    for (int i = 0; i < nq; ++i) out[(size_t)(t0 + i) * ld + c] = o[i] * f;
  }
}

// Forward: P[h, t, 0..t] = softmax(q_t K^T / sqrt(hd)), a[t, head] = P V.  P is kept for the backward pass.
__global__ void __launch_bounds__(kAtThreads) attn_fwd_kernel(const float* __restrict__ q, const float* __restrict__ k,
                                                               const float* __restrict__ v, float* __restrict__ P,
                                                               float* __restrict__ a, int T, int n_heads, int hd, float scale) {
  extern __shared__ float s_at[];
  float *s_p = s_at, *sx = s_at + kAtQ * T, *sy = sx + kAtQ * kAtDim;
  const int t0 = blockIdx.x * kAtQ, h = blockIdx.y, nq = min(kAtQ, T - t0), lane = threadIdx.x & 31;
  const size_t ld = (size_t)n_heads * hd, o = (size_t)blockIdx.z * T * ld + (size_t)h * hd;
  attn_scores(q + o, k + o, s_p, sx, sy, T, t0, nq, hd, ld);
  for (int i = threadIdx.x >> 5; i < kAtQ; i += kAtThreads / 32) {  // a warp per query
    float* row = s_p + i * T;
    const int t = i < nq ? t0 + i : -1;
    float mx = -INFINITY;
    for (int j = lane; j <= t; j += 32) mx = fmaxf(mx, row[j] * scale);
    mx = warp_max(mx);
    double part = 0.0;
    for (int j = lane; j <= t; j += 32) {
      const float e = expf(row[j] * scale - mx);
      row[j] = e;
      part += e;
    }
#pragma unroll
    for (int w = 16; w > 0; w >>= 1) part += __shfl_xor_sync(0xffffffffu, part, w);
    const float inv = (float)(1.0 / part);
    float* Pt = P + (((size_t)blockIdx.z * n_heads + h) * T + t0 + i) * T;
    for (int j = lane; j < T; j += 32) {
      const float pj = j <= t ? row[j] * inv : 0.f;
      row[j] = pj;
      if (i < nq) Pt[j] = pj;
    }
  }
  __syncthreads();
  attn_weighted_sum(s_p, v + o, a + o, T, t0, nq, hd, ld, 1.f);
}

// Backward, step 1: dS[h,t,j] = P (dP - sum_j P dP) with dP = da V^T, and dq[t, head] = dS K * scale.
__global__ void __launch_bounds__(kAtThreads) attn_bwd_q_kernel(const float* __restrict__ da, const float* __restrict__ k,
                                                                 const float* __restrict__ v, const float* __restrict__ P,
                                                                 float* __restrict__ dS, float* __restrict__ dq, int T, int n_heads,
                                                                 int hd, float scale) {
  extern __shared__ float s_at[];
  float *s_ds = s_at, *sx = s_at + kAtQ * T, *sy = sx + kAtQ * kAtDim;
  const int t0 = blockIdx.x * kAtQ, h = blockIdx.y, nq = min(kAtQ, T - t0), lane = threadIdx.x & 31;
  const size_t ld = (size_t)n_heads * hd, o = (size_t)blockIdx.z * T * ld + (size_t)h * hd;
  attn_scores(da + o, v + o, s_ds, sx, sy, T, t0, nq, hd, ld);
  for (int i = threadIdx.x >> 5; i < kAtQ; i += kAtThreads / 32) {
    float* row = s_ds + i * T;
    const int t = i < nq ? t0 + i : -1;
    const size_t po = (((size_t)blockIdx.z * n_heads + h) * T + t0 + i) * T;
    double part = 0.0;
    for (int j = lane; j <= t; j += 32) part += (double)P[po + j] * row[j];
#pragma unroll
    for (int w = 16; w > 0; w >>= 1) part += __shfl_xor_sync(0xffffffffu, part, w);
    const float rs = (float)part;
    for (int j = lane; j < T; j += 32) {
      const float x = j <= t ? P[po + j] * (row[j] - rs) : 0.f;
      row[j] = x;
      if (i < nq) dS[po + j] = x;
    }
  }
  __syncthreads();
  attn_weighted_sum(s_ds, k + o, dq + o, T, t0, nq, hd, ld, scale);
}

// Backward, step 2, a block takes kAtQ consecutive keys: dk[j] = sum_{t>=j} dS[t,j] q[t] * scale, dv[j] = sum_{t>=j} P[t,j] da[t]
__global__ void __launch_bounds__(kAtThreads) attn_bwd_kv_kernel(const float* __restrict__ da, const float* __restrict__ q,
                                                                  const float* __restrict__ P, const float* __restrict__ dS,
                                                                  float* __restrict__ dk, float* __restrict__ dv, int T, int n_heads,
                                                                  int hd, float scale) {
  __shared__ float s_p[kAtKeys][kAtQ], s_d[kAtKeys][kAtQ];
  const int j0 = blockIdx.x * kAtQ, h = blockIdx.y, nj = min(kAtQ, T - j0);
  const size_t ld = (size_t)n_heads * hd, o = (size_t)blockIdx.z * T * ld + (size_t)h * hd;
  const size_t po = ((size_t)blockIdx.z * n_heads + h) * T * T + j0;
  for (int c0 = 0; c0 < hd; c0 += kAtThreads) {
    const int c = c0 + threadIdx.x;
    float ak[kAtQ] = {}, av[kAtQ] = {};
    for (int t0 = j0; t0 < T; t0 += kAtKeys) {  // P and dS are zero at t < j
      const int nt = min(kAtKeys, T - t0);
      __syncthreads();
      for (int e = threadIdx.x; e < nt * kAtQ; e += kAtThreads) {
        const int t = e / kAtQ, j = e % kAtQ;
        s_p[t][j] = j < nj ? P[po + (size_t)(t0 + t) * T + j] : 0.f;
        s_d[t][j] = j < nj ? dS[po + (size_t)(t0 + t) * T + j] : 0.f;
      }
      __syncthreads();
      if (c < hd) {
#pragma unroll 4
        for (int t = 0; t < nt; ++t) {
          const float qv = q[o + (size_t)(t0 + t) * ld + c], dav = da[o + (size_t)(t0 + t) * ld + c];
#pragma unroll
          for (int j = 0; j < kAtQ; ++j) {
            ak[j] = fmaf(s_d[t][j], qv, ak[j]);
            av[j] = fmaf(s_p[t][j], dav, av[j]);
          }
        }
      }
    }
    if (c < hd)
      for (int j = 0; j < nj; ++j) {
        dk[o + (size_t)(j0 + j) * ld + c] = ak[j] * scale;
        dv[o + (size_t)(j0 + j) * ld + c] = av[j];
      }
  }
}

// u = silu(gate) * up
__global__ void swiglu_fwd_kernel(const float* __restrict__ gt, const float* __restrict__ up, float* __restrict__ u, size_t n) {
  for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x) {
    const float g = gt[i];
    u[i] = g / (1.0f + expf(-g)) * up[i];
  }
}
// dgate = du * up * silu'(gate), dup = du * silu(gate)
__global__ void swiglu_bwd_kernel(const float* __restrict__ du, const float* __restrict__ gt, const float* __restrict__ up,
                                  float* __restrict__ dgt, float* __restrict__ dup, size_t n) {
  for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x) {
    const float g = gt[i], sg = 1.0f / (1.0f + expf(-g));
    dgt[i] = du[i] * up[i] * sg * (1.0f + g * (1.0f - sg));
    dup[i] = du[i] * g * sg;
  }
}

// Mean next-token cross-entropy: dlogits[t,:] = (softmax(logits[t,:]) - onehot(target_t)) / T, in place; loss[t] kept
__global__ void __launch_bounds__(1024) ce_bwd_kernel(float* __restrict__ logits, const int* __restrict__ tok, int V, int T,
                                                       int seq_len, float* __restrict__ loss) {
  __shared__ double s_red[32];
  __shared__ float s_mx[32];
  const int t = blockIdx.x;  // row of the group; its target is the token that follows
  float* l = logits + (size_t)t * V;
  float mx = -INFINITY;
  for (int v = threadIdx.x; v < V; v += blockDim.x) mx = fmaxf(mx, l[v]);
  mx = warp_max(mx);
  if ((threadIdx.x & 31) == 0) s_mx[threadIdx.x >> 5] = mx;
  __syncthreads();
  mx = s_mx[0];
  for (int w = 1; w < 32; ++w) mx = fmaxf(mx, s_mx[w]);
  double part = 0.0;
  for (int v = threadIdx.x; v < V; v += blockDim.x) part += exp((double)l[v] - (double)mx);
  const double tot = block_sum_d(part, s_red);
  const int y = tok[(t / T) * seq_len + t % T + 1];
  if (threadIdx.x == 0) loss[t] = (float)(log(tot) + (double)mx - (double)l[y]);
  __syncthreads();
  for (int v = threadIdx.x; v < V; v += blockDim.x) {
    const double pv = exp((double)l[v] - (double)mx) / tot;
    l[v] = (float)((pv - (v == y ? 1.0 : 0.0)) / T);
  }
}

// ---- squared norms of the weight gradients -----------------------------------------------------------
// Per layer eleven Gram matrices per sequence (eight of activations or gradients d wide, three f wide)
// and seven dot products of two of them.  Bound by the fp64 FMA pipe, T^2 / 2 * (8 d + 3 f) of them a
// sequence: a CTA of two warps computes one 32 x 32 tile of one matrix over a chunk of the contraction,
// 4 x 4 outputs per thread (per contraction step 16 clocks of fp64 FMAs against 8 of shared-memory
// reads); a matrix is symmetric, so only the tiles on and below the diagonal are computed.
constexpr int kGramTile = 32, kGramThreads = 64, kGramK = 16;
constexpr int kGrams = 11, kGramsD = 8;  // the first eight are d wide
constexpr int kDots = 7;
constexpr int kFitTensors = 9;

struct GramPlan {  // how the contractions are cut: by T, d, f and the sequences of a full group
  int pairs;       // tiles on and below the diagonal
  int chunk;       // contraction length of a CTA, a multiple of kGramK
  int pd, pf;      // chunks of a d-wide and of an f-wide matrix
  int dot_blocks;
  __host__ __device__ int pieces() const { return kGramsD * pd + (kGrams - kGramsD) * pf; }
  __host__ __device__ int first(int i) const { return i < kGramsD ? i * pd : kGramsD * pd + (i - kGramsD) * pf; }
  size_t doubles(int nb) const { return (size_t)nb * pieces() * pairs * kGramTile * kGramTile; }
};
inline GramPlan gram_plan(int T, int nb, int d, int f, int n_sm) {
  GramPlan p;
  const int t = (T + kGramTile - 1) / kGramTile;
  p.pairs = t * (t + 1) / 2;
  // about twelve CTAs of two warps per SM hide the fp64 latency; chunks below 256 are mostly set-up
  const double ctas_per_column = (double)p.pairs * nb / (12.0 * n_sm);
  const double total = (double)kGramsD * d + (double)(kGrams - kGramsD) * f;
  const int longest = std::max(d, f);
  const double want = std::min(total * ctas_per_column, (double)longest);
  p.chunk = (int)(std::max(256.0, want) + kGramK - 1) / kGramK * kGramK;
  p.pd = (d + p.chunk - 1) / p.chunk;
  p.pf = (f + p.chunk - 1) / p.chunk;
  p.dot_blocks = 4 * std::min(p.pairs, 16);
  return p;
}

struct GramArgs {
  const float* A[kGrams];  // [sequences * T, d or f]
  double* G;               // [sequence][piece][tile pair][32 * 32]
  int d, f, T;
  GramPlan plan;
};

__global__ void __launch_bounds__(kGramThreads) gram_kernel(const __grid_constant__ GramArgs g) {
  constexpr int Ld = kGramTile + 2;
  __shared__ __align__(16) double sa[kGramK][Ld], sb[kGramK][Ld];
  const int tid = threadIdx.x, tx = tid & 7, ty = tid >> 3;
  int bi = 0, rest = blockIdx.x;  // tile pair (bi, bj), bj <= bi
  while (rest > bi) rest -= ++bi;
  const int bj = rest;
  const int y = blockIdx.y, nd = kGramsD * g.plan.pd;
  const int which = y < nd ? y / g.plan.pd : kGramsD + (y - nd) / g.plan.pf;
  const int piece = y - g.plan.first(which);
  const int n = which < kGramsD ? g.d : g.f;
  const float* A = g.A[which] + (size_t)blockIdx.z * g.T * n;
  const int k_lo = piece * g.plan.chunk, k_hi = min(n, k_lo + g.plan.chunk);
  const bool vec = (n & 3) == 0;
  // thread loads 8 consecutive values of one row of each tile: row tid / 2, columns (tid % 2) * 8
  const int lr = tid >> 1, lk = (tid & 1) * 8;
  const bool same = bi == bj;
  float va[8], vb[8];
  auto fetch = [&](float (&v)[8], int row, int k) {
    const float* p = A + (size_t)row * n + k;
    const int left = row < g.T ? k_hi - k : 0;
    if (vec) {
      const float4 a = left > 0 ? *reinterpret_cast<const float4*>(p) : make_float4(0.f, 0.f, 0.f, 0.f);
      const float4 b = left > 4 ? *reinterpret_cast<const float4*>(p + 4) : make_float4(0.f, 0.f, 0.f, 0.f);
      v[0] = a.x; v[1] = a.y; v[2] = a.z; v[3] = a.w; v[4] = b.x; v[5] = b.y; v[6] = b.z; v[7] = b.w;
    } else {
#pragma unroll
      for (int i = 0; i < 8; ++i) v[i] = i < left ? p[i] : 0.f;
    }
  };
  double acc[4][4] = {};
  fetch(va, bi * kGramTile + lr, k_lo + lk);
  if (!same) fetch(vb, bj * kGramTile + lr, k_lo + lk);
  for (int k0 = k_lo; k0 < k_hi; k0 += kGramK) {
#pragma unroll
    for (int i = 0; i < 8; ++i) sa[lk + i][lr] = (double)va[i];
    if (!same) {
#pragma unroll
      for (int i = 0; i < 8; ++i) sb[lk + i][lr] = (double)vb[i];
    }
    __syncthreads();
    if (k0 + kGramK < k_hi) {
      fetch(va, bi * kGramTile + lr, k0 + kGramK + lk);
      if (!same) fetch(vb, bj * kGramTile + lr, k0 + kGramK + lk);
    }
    const double(*pb)[Ld] = same ? sa : sb;
#pragma unroll
    for (int kk = 0; kk < kGramK; ++kk) {
      const double2 a0 = *reinterpret_cast<const double2*>(&sa[kk][ty * 4]), a1 = *reinterpret_cast<const double2*>(&sa[kk][ty * 4 + 2]);
      const double2 b0 = *reinterpret_cast<const double2*>(&pb[kk][tx * 2]), b1 = *reinterpret_cast<const double2*>(&pb[kk][16 + tx * 2]);
      const double av[4] = {a0.x, a0.y, a1.x, a1.y}, bv[4] = {b0.x, b0.y, b1.x, b1.y};
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j] = fma(av[i], bv[j], acc[i][j]);
    }
    __syncthreads();
  }
  double* out = g.G + (((size_t)blockIdx.z * g.plan.pieces() + y) * g.plan.pairs + blockIdx.x) * (kGramTile * kGramTile);
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    *reinterpret_cast<double2*>(out + (ty * 4 + i) * kGramTile + tx * 2) = make_double2(acc[i][0], acc[i][1]);
    *reinterpret_cast<double2*>(out + (ty * 4 + i) * kGramTile + 16 + tx * 2) = make_double2(acc[i][2], acc[i][3]);
  }
}

// One block = (share of the tile pairs and a quarter of their elements, dot product, sequence): sum over its elements of the product of
// the two matrices (chunks added in chunk order; tiles below the diagonal count twice), added to this
// block's slot of the tensor.
__global__ void __launch_bounds__(256) gram_dot_kernel(const double* __restrict__ G, GramPlan plan, double* __restrict__ slots, int n_slots) {
  __shared__ double s_red[8];
  constexpr int kE = kGramTile * kGramTile;
  // matrices in the order the host lists them: dH, x2, dHmid, a, x1, dq, dk, dv, u, dgate, dup; tensors wq, wk, wv, wo, gate, up, down
  const int left[kDots] = {4, 4, 4, 3, 1, 1, 8}, right[kDots] = {5, 6, 7, 2, 9, 10, 0};
  const int t = blockIdx.y;
  const double* base = G + (size_t)blockIdx.z * plan.pieces() * plan.pairs * kE;
  const int i1 = left[t], i2 = right[t];
  const int n1 = i1 < kGramsD ? plan.pd : plan.pf, n2 = i2 < kGramsD ? plan.pd : plan.pf;
  double s = 0.0;
  int row = 0, rest = 0;  // tile pair p = (row, rest)
  for (int p = 0; p < plan.pairs; ++p) {
    if (p % (gridDim.x / 4) == blockIdx.x / 4) {
      const double* g1 = base + ((size_t)plan.first(i1) * plan.pairs + p) * kE;
      const double* g2 = base + ((size_t)plan.first(i2) * plan.pairs + p) * kE;
      const double w = rest == row ? 1.0 : 2.0;
      {
        const int e = (blockIdx.x & 3) * 256 + threadIdx.x;
        double a = 0.0, b = 0.0;
        for (int c = 0; c < n1; ++c) a += g1[(size_t)c * plan.pairs * kE + e];
        for (int c = 0; c < n2; ++c) b += g2[(size_t)c * plan.pairs * kE + e];
        s += w * a * b;
      }
    }
    if (++rest > row) ++row, rest = 0;
  }
  const double tot = block_sum_d(s, s_red);
  if (threadIdx.x == 0) slots[(size_t)t * n_slots + blockIdx.z * gridDim.x + blockIdx.x] += tot;
}

// sum of w^2 in two fixed-order steps: per-block partial sums of every tensor of a layer, then finish_kernel
constexpr int kMsBlocks = 296;
struct SumSqArgs {
  const void* w[kFitTensors];
  size_t n[kFitTensors];
};
template <typename WT>
__global__ void __launch_bounds__(256) sum_sq_partial_kernel(const __grid_constant__ SumSqArgs a, double* __restrict__ partial) {
  __shared__ double s_red[8];
  const WT* w = reinterpret_cast<const WT*>(a.w[blockIdx.y]);
  const size_t n = a.n[blockIdx.y], stride = (size_t)gridDim.x * blockDim.x;
  constexpr int kV = 16 / sizeof(WT);
  double s = 0.0;
  size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if ((reinterpret_cast<uintptr_t>(w) & 15) == 0) {
    const size_t nv = n / kV;
    const uint4* p = reinterpret_cast<const uint4*>(w);
    auto add = [&](const uint4& r) {
      const WT* v = reinterpret_cast<const WT*>(&r);
#pragma unroll
      for (int j = 0; j < kV; ++j) {
        const double x = wload(v + j);
        s += x * x;
      }
    };
    size_t j = i;
    for (; j + 3 * stride < nv; j += 4 * stride) {  // four loads in flight
      const uint4 r0 = p[j], r1 = p[j + stride], r2 = p[j + 2 * stride], r3 = p[j + 3 * stride];
      add(r0); add(r1); add(r2); add(r3);
    }
    for (; j < nv; j += stride) add(p[j]);
    i += nv * kV;
  }
  for (; i < n; i += stride) {
    const double v = wload(w + i);
    s += v * v;
  }
  const double tot = block_sum_d(s, s_red);
  if (threadIdx.x == 0) partial[(size_t)blockIdx.y * gridDim.x + blockIdx.x] = tot;
}
// one block per (layer, tensor): out = {sum of its slots, sum of w^2}
__global__ void __launch_bounds__(256) finish_kernel(const double* __restrict__ slots, int n_slots, const double* __restrict__ ms_part,
                                                      double* __restrict__ out) {
  __shared__ double s_red[8];
  double a = 0.0, b = 0.0;
  for (int i = threadIdx.x; i < n_slots; i += 256) a += slots[(size_t)blockIdx.x * n_slots + i];
  for (int i = threadIdx.x; i < kMsBlocks; i += 256) b += ms_part[(size_t)blockIdx.x * kMsBlocks + i];
  const double ta = block_sum_d(a, s_red), tb = block_sum_d(b, s_red);
  if (threadIdx.x == 0) {
    out[2 * blockIdx.x] = ta;
    out[2 * blockIdx.x + 1] = tb;
  }
}

// ---- host side --------------------------------------------------------------------------------------
enum Tensor { T_WQ = 0, T_WK, T_WV, T_WO, T_GATE, T_UP, T_DOWN, T_ATTN_NORM, T_FFN_NORM, kTensors };
static_assert(kTensors == kFitTensors, "the kernels' tensor count");

constexpr int kFitRows = 512;  // calibration tokens that go through the stack together (at least one sequence)

// Device memory of a call, one allocation.  Up to kFitPoolKeep bytes come from a pool of the library's own, one per device:
// cudaMalloc and cudaFree take 0.7 to 1.5 ms, as much as the whole call for a small decoder (4 layers d 256, 8 x 31
// tokens: 1.07 ms from the pool, 1.82 without; 4 layers d 4096, 2 x 64 tokens, 200 MB: 12.7 and 14.3).  The pool keeps what it has
// handed out, at most kFitPoolKeep bytes, until sdfp_fit_release, until a context is destroyed or until one runs
// out of memory.  A larger working set is allocated and freed by the call itself: the call takes tens
// of milliseconds, and mapping that much through the pool costs more than cudaMalloc (0.9 GB: 17.8 and 7.7 ms a call).
constexpr unsigned long long kFitPoolKeep = 256ull << 20;
constexpr int kFitPools = 64;
struct FitPools {
  std::mutex lock;
  cudaMemPool_t pool[kFitPools] = {};
};
inline FitPools& fit_pools() {
  static FitPools p;
  return p;
}
inline cudaError_t fit_pool(int dev, cudaMemPool_t* out) {
  if (dev < 0 || dev >= kFitPools) return cudaErrorInvalidDevice;
  FitPools& f = fit_pools();
  std::lock_guard<std::mutex> g(f.lock);
  if (f.pool[dev] == nullptr) {
    cudaMemPoolProps pr = {};
    pr.allocType = cudaMemAllocationTypePinned;
    pr.location.type = cudaMemLocationTypeDevice;
    pr.location.id = dev;
    cudaMemPool_t p = nullptr;
    cudaError_t e = cudaMemPoolCreate(&p, &pr);
    if (e != cudaSuccess) return e;
    unsigned long long keep = kFitPoolKeep;
    e = cudaMemPoolSetAttribute(p, cudaMemPoolAttrReleaseThreshold, &keep);
    if (e != cudaSuccess) {
      cudaMemPoolDestroy(p);
      return e;
    }
    f.pool[dev] = p;
  }
  *out = f.pool[dev];
  return cudaSuccess;
}
inline void fit_pool_trim(int dev) {
  if (dev < 0 || dev >= kFitPools) return;
  FitPools& f = fit_pools();
  std::lock_guard<std::mutex> g(f.lock);
  if (f.pool[dev] != nullptr && cudaMemPoolTrimTo(f.pool[dev], 0) != cudaSuccess) cudaGetLastError();
}
inline cudaError_t fit_alloc(void** p, size_t bytes, int dev, cudaStream_t st) {
  if (bytes <= kFitPoolKeep) {
    cudaMemPool_t pool;
    const cudaError_t e = fit_pool(dev, &pool);
    return e != cudaSuccess ? e : cudaMallocFromPoolAsync(p, bytes, pool, st);
  }
  cudaError_t e = cudaMalloc(p, bytes);
  if (e == cudaErrorMemoryAllocation) {
    cudaGetLastError();
    fit_pool_trim(dev);
    e = cudaMalloc(p, bytes);
  }
  return e;
}
// behind whatever is still running on the buffer, and waited for: on return the results are there and the memory is the
// pool's or the device's again
inline cudaError_t fit_free(void* p, size_t bytes, cudaStream_t st) {
  const bool pooled = bytes <= kFitPoolKeep;
  const cudaError_t pe = pooled ? cudaFreeAsync(p, st) : cudaSuccess;
  const cudaError_t se = cudaStreamSynchronize(st);
  const cudaError_t fe = pooled ? pe : cudaFree(p);
  return se != cudaSuccess ? se : fe;
}

// One device allocation per call, cut into buffers: the layout runs once to learn the size and once
// more to hand the pieces out.
struct Arena {
  unsigned char* base = nullptr;
  size_t used = 0;
  template <typename T>
  T* get(size_t n) {
    T* p = base ? reinterpret_cast<T*>(base + used) : nullptr;
    used += (std::max<size_t>(n * sizeof(T), 16) + 255) & ~size_t(255);
    return p;
  }
};

struct Buffers {
  // activations kept for the backward pass, per layer
  std::vector<float*> Hs, Hmid, x1, q, k, v, P, a, x2, gt, up, u, inv1, inv2;
  float *xf, *invf, *logits, *loss, *dx, *da, *dq, *dk, *dv, *dS, *du, *dgt, *dup, *cs, *sn;
  float* dH[3];  // gradient of a layer's output, of its middle and of its input; the last is the next one's first
  double *G, *slots, *ms_part, *out;
  int* tok;
  void layout(Arena& A, int L, int d, int f, int V, int H, int hd, int T, int nb, int n_tok, size_t gram_doubles, int n_slots) {
    const size_t R = (size_t)nb * T, Rd = R * d, Rf = R * f, pp = (size_t)nb * H * T * T;
    for (auto* x : {&Hs, &Hmid, &x1, &q, &k, &v, &P, &a, &x2, &gt, &up, &u, &inv1, &inv2}) x->resize(L + 1);
    for (int l = 0; l <= L; ++l) Hs[l] = A.get<float>(Rd);
    for (int l = 0; l < L; ++l) {
      Hmid[l] = A.get<float>(Rd); x1[l] = A.get<float>(Rd); q[l] = A.get<float>(Rd); k[l] = A.get<float>(Rd); v[l] = A.get<float>(Rd);
      P[l] = A.get<float>(pp); a[l] = A.get<float>(Rd); x2[l] = A.get<float>(Rd);
      gt[l] = A.get<float>(Rf); up[l] = A.get<float>(Rf); u[l] = A.get<float>(Rf);
      inv1[l] = A.get<float>(R); inv2[l] = A.get<float>(R);
    }
    xf = A.get<float>(Rd); invf = A.get<float>(R); logits = A.get<float>(R * V); loss = A.get<float>(R);
    for (float*& x : dH) x = A.get<float>(Rd);
    dx = A.get<float>(Rd); da = A.get<float>(Rd); dq = A.get<float>(Rd); dk = A.get<float>(Rd); dv = A.get<float>(Rd);
    dS = A.get<float>(pp); du = A.get<float>(Rf); dgt = A.get<float>(Rf); dup = A.get<float>(Rf);
    cs = A.get<float>((size_t)T * (hd / 2)); sn = A.get<float>((size_t)T * (hd / 2));
    G = A.get<double>(gram_doubles);
    slots = A.get<double>((size_t)L * kTensors * n_slots);
    ms_part = A.get<double>((size_t)L * kTensors * kMsBlocks);
    out = A.get<double>((size_t)L * kTensors * 2);
    tok = A.get<int>(n_tok);
  }
};

#define FIT_OK(call)                      \
  do {                                    \
    cudaError_t e_ = (call);              \
    if (e_ != cudaSuccess) return e_;     \
  } while (0)

template <typename WT, int BM, bool NT, bool VEC>
cudaError_t fit_gemm_go(const GemmArgs& g, int tiles, int S, cudaStream_t st) {
  cudaLaunchConfig_t lc = {};
  lc.gridDim = dim3(tiles, (g.R + BM - 1) / BM, S);
  lc.blockDim = dim3(kGThreads);
  lc.dynamicSmemBytes = gemm_smem_bytes<BM>();
  lc.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = 1;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = S;
  lc.attrs = attr;
  lc.numAttrs = 1;
  return cudaLaunchKernelEx(&lc, fit_gemm_kernel<WT, BM, NT, VEC>, g);
}

struct GemmRoom {  // clusters of s CTAs with a BM = 32 << i tile that the device runs at a time
  int clusters[3][9];
};
template <typename WT, int BM>
cudaError_t gemm_prepare(int* clusters) {
  const int smem = (int)gemm_smem_bytes<BM>();
  for (const void* k : {(const void*)fit_gemm_kernel<WT, BM, true, true>, (const void*)fit_gemm_kernel<WT, BM, true, false>,
                        (const void*)fit_gemm_kernel<WT, BM, false, true>, (const void*)fit_gemm_kernel<WT, BM, false, false>})
    FIT_OK(cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, smem));
  for (int s = 1; s <= 8; ++s) {
    cudaLaunchConfig_t lc = {};
    lc.gridDim = dim3(1, 1, s);
    lc.blockDim = dim3(kGThreads);
    lc.dynamicSmemBytes = smem;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = 1;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = s;
    lc.attrs = attr;
    lc.numAttrs = 1;
    // the instantiations of a BM have the same footprint (the launch bounds), so one answers for all
    FIT_OK(cudaOccupancyMaxActiveClusters(clusters + s, fit_gemm_kernel<WT, BM, true, true>, &lc));
    clusters[s] = std::max(1, clusters[s]);
  }
  return cudaSuccess;
}

// plan_rows: the rows of a full group of sequences.  How a contraction is cut depends on them and not on g.R, so
// that a sequence's numbers do not change when it sits in a smaller group (the last one, or where memory is short).
template <typename WT, bool NT>
cudaError_t fit_gemm_launch(const GemmArgs& g, int plan_rows, const GemmRoom& room, int n_sm, cudaStream_t st) {
  const int cols = NT ? g.N : g.K, inner = NT ? g.K : g.N;
  const int tiles = (cols + kGN - 1) / kGN * (NT ? g.parts : 1);
  const int steps = (inner + kGK - 1) / kGK * (NT ? 1 : g.parts);
  // Cost of a choice, in k steps of one BM 128 tile: waves of CTAs, those of an SM sharing its FMA pipe; a
  // last wave of about one per SM leaves the pipe waiting for shared memory; narrow tiles load more
  // values per FMA.  Clusters do not fill an SM group evenly (clusters of three waste a tenth of the
  // slots), so the room for them is asked from the runtime.
  int best_bm = 128, best_s = 1;
  double best = 1e30;
  for (int i = 0; i < 3; ++i) {
    const int bm = 32 << i;
    const double per_step = bm == 128 ? 1.0 : bm == 64 ? 0.75 : 0.62;
    for (int s = 1; s <= 8; ++s) {
      if (s > 1 && steps / s < 4) break;
      const long long n = (long long)tiles * ((plan_rows + bm - 1) / bm), cap = room.clusters[i][s];
      const long long last = n % cap;
      const long long left = (last * s + n_sm - 1) / n_sm;  // CTAs of the last wave on the fullest SM
      const double waves = (double)(n / cap * cap * s) / n_sm + (left == 1 ? 1.3 : (double)left);
      const double cost = waves * per_step * ((double)((steps + s - 1) / s) + 4.0) + (s > 1 ? 6.0 : 0.0);
      if (cost < best) best = cost, best_bm = bm, best_s = s;
    }
  }
  bool vec = g.N % 8 == 0 && g.K % 8 == 0;
  for (int p = 0; p < g.parts; ++p) vec = vec && (reinterpret_cast<uintptr_t>(g.W[p]) & 15) == 0;
  if (best_bm == 128)
    return vec ? fit_gemm_go<WT, 128, NT, true>(g, tiles, best_s, st) : fit_gemm_go<WT, 128, NT, false>(g, tiles, best_s, st);
  if (best_bm == 64)
    return vec ? fit_gemm_go<WT, 64, NT, true>(g, tiles, best_s, st) : fit_gemm_go<WT, 64, NT, false>(g, tiles, best_s, st);
  return vec ? fit_gemm_go<WT, 32, NT, true>(g, tiles, best_s, st) : fit_gemm_go<WT, 32, NT, false>(g, tiles, best_s, st);
}

template <typename WT>
cudaError_t run_in(const sdfp_config& g, const sdfp_weights* w, cudaStream_t st, const int32_t* tokens, int n_seq, int seq_len,
                   std::vector<double>& sums, Buffers& B, int nb, int full, int n_sm, const GemmRoom& room, const GramPlan& gp, int n_slots) {
  const int L = g.n_layers, d = g.d_model, f = g.d_ffn, V = g.vocab, H = g.n_heads, hd = g.head_dim, T = seq_len - 1;
  const float scale = 1.0f / std::sqrt((float)hd);
  FIT_OK(cudaMemsetAsync(B.slots, 0, (size_t)L * kTensors * n_slots * sizeof(double), st));
  rope_table_kernel<<<(T * (hd / 2) + 127) / 128, 128, 0, st>>>(B.cs, B.sn, T, hd, (double)g.rope_theta);
  auto W = [&](const void* const* arr, int l) { return reinterpret_cast<const WT*>(arr[l]); };
  const int eb = 4 * n_sm;  // blocks of the elementwise kernels
  const size_t att_smem = attn_smem(T);
  cudaError_t ge = cudaSuccess;

  const int gain_blocks = (d + kGainCols - 1) / kGainCols;
  for (int s0 = 0, ns; s0 < n_seq; s0 += ns) {
    const int z0 = s0 % full;  // place of the first sequence in its full group: its slots, whatever goes through together
    ns = std::min(std::min(nb, full - z0), n_seq - s0);
    const int R = ns * T;
    const size_t Rf = (size_t)R * f;
    const int* tok = B.tok;
    FIT_OK(cudaMemcpyAsync(B.tok, tokens + (size_t)s0 * seq_len, (size_t)ns * seq_len * 4, cudaMemcpyHostToDevice, st));
    auto nt = [&](GemmArgs a, int N, int K) {
      a.R = R; a.N = N; a.K = K;
      if (ge == cudaSuccess) ge = fit_gemm_launch<WT, true>(a, full * T, room, n_sm, st);
    };
    auto nn = [&](GemmArgs a, int N, int K) {
      a.R = R; a.N = N; a.K = K;
      if (ge == cudaSuccess) ge = fit_gemm_launch<WT, false>(a, full * T, room, n_sm, st);
    };
    // ---- forward ----
    embed_kernel<WT><<<R, 256, 0, st>>>(tok, reinterpret_cast<const WT*>(w->tok_embed), B.Hs[0], d, T, seq_len);
    for (int l = 0; l < L; ++l) {
      rmsnorm_fwd_kernel<WT><<<R, 512, 0, st>>>(B.Hs[l], W(w->attn_norm, l), B.x1[l], B.inv1[l], d, g.rms_eps);
      nt({{B.x1[l]}, {w->wq[l], w->wk[l], w->wv[l]}, {B.q[l], B.k[l], B.v[l]}, nullptr, 0, 0, 0, 3}, d, d);
      rope_kernel<<<dim3(R, 2), 128, 0, st>>>(B.q[l], B.k[l], B.cs, B.sn, T, H, hd, 1.f);
      attn_fwd_kernel<<<dim3((T + kAtQ - 1) / kAtQ, H, ns), kAtThreads, att_smem, st>>>(B.q[l], B.k[l], B.v[l], B.P[l], B.a[l], T, H, hd, scale);
      nt({{B.a[l]}, {w->wo[l]}, {B.Hmid[l]}, B.Hs[l], 0, 0, 0, 1}, d, d);
      rmsnorm_fwd_kernel<WT><<<R, 512, 0, st>>>(B.Hmid[l], W(w->ffn_norm, l), B.x2[l], B.inv2[l], d, g.rms_eps);
      nt({{B.x2[l]}, {w->w_gate[l], w->w_up[l]}, {B.gt[l], B.up[l]}, nullptr, 0, 0, 0, 2}, f, d);
      swiglu_fwd_kernel<<<eb, 256, 0, st>>>(B.gt[l], B.up[l], B.u[l], Rf);
      nt({{B.u[l]}, {w->w_down[l]}, {B.Hs[l + 1]}, B.Hmid[l], 0, 0, 0, 1}, d, f);
    }
    rmsnorm_fwd_kernel<WT><<<R, 512, 0, st>>>(B.Hs[L], reinterpret_cast<const WT*>(w->final_norm), B.xf, B.invf, d, g.rms_eps);
    nt({{B.xf}, {w->lm_head}, {B.logits}, nullptr, 0, 0, 0, 1}, V, d);
    ce_bwd_kernel<<<R, 1024, 0, st>>>(B.logits, tok, V, T, seq_len, B.loss);  // logits now hold d f / d logits
    // ---- backward: gradients with respect to activations, squared norms of the weight gradients by Gram matrices ----
    nn({{B.logits}, {w->lm_head}, {B.dx}, nullptr, 0, 0, 0, 1}, V, d);
    float *dh = B.dH[0], *dmid = B.dH[1], *dnext = B.dH[2];
    rmsnorm_bwd_kernel<WT><<<R, 512, 0, st>>>(B.dx, B.Hs[L], reinterpret_cast<const WT*>(w->final_norm), B.invf, nullptr, dh, d);
    for (int l = L - 1; l >= 0; --l) {
      double* slots = B.slots + (size_t)l * kTensors * n_slots;
      // FFN block: H[l+1] = Hmid + u Wd^T
      nn({{dh}, {w->w_down[l]}, {B.du}, nullptr, 0, 0, 0, 1}, d, f);
      swiglu_bwd_kernel<<<eb, 256, 0, st>>>(B.du, B.gt[l], B.up[l], B.dgt, B.dup, Rf);
      nn({{B.dgt, B.dup}, {w->w_gate[l], w->w_up[l]}, {B.dx}, nullptr, 0, 0, 0, 2}, f, d);
      gain_grad_sq_kernel<<<dim3(gain_blocks, ns), 256, 0, st>>>(B.dx, B.Hmid[l], B.inv2[l], T, d, slots + (size_t)T_FFN_NORM * n_slots + z0 * gain_blocks);
      rmsnorm_bwd_kernel<WT><<<R, 512, 0, st>>>(B.dx, B.Hmid[l], W(w->ffn_norm, l), B.inv2[l], dh, dmid, d);  // d f / d Hmid
      // attention block: Hmid = H[l] + a Wo^T
      nn({{dmid}, {w->wo[l]}, {B.da}, nullptr, 0, 0, 0, 1}, d, d);
      attn_bwd_q_kernel<<<dim3((T + kAtQ - 1) / kAtQ, H, ns), kAtThreads, att_smem, st>>>(B.da, B.k[l], B.v[l], B.P[l], B.dS, B.dq, T, H, hd, scale);
      attn_bwd_kv_kernel<<<dim3((T + kAtQ - 1) / kAtQ, H, ns), kAtThreads, 0, st>>>(B.da, B.q[l], B.P[l], B.dS, B.dk, B.dv, T, H, hd, scale);
      rope_kernel<<<dim3(R, 2), 128, 0, st>>>(B.dq, B.dk, B.cs, B.sn, T, H, hd, -1.f);
      nn({{B.dq, B.dk, B.dv}, {w->wq[l], w->wk[l], w->wv[l]}, {B.dx}, nullptr, 0, 0, 0, 3}, d, d);
      gain_grad_sq_kernel<<<dim3(gain_blocks, ns), 256, 0, st>>>(B.dx, B.Hs[l], B.inv1[l], T, d, slots + (size_t)T_ATTN_NORM * n_slots + z0 * gain_blocks);
      rmsnorm_bwd_kernel<WT><<<R, 512, 0, st>>>(B.dx, B.Hs[l], W(w->attn_norm, l), B.inv1[l], dmid, dnext, d);  // d f / d H[l]
      // every factor of the layer's weight gradients is at hand: all its Gram matrices, then the seven dot products
      GramArgs ga{};
      const float* src[kGrams] = {dh, B.x2[l], dmid, B.a[l], B.x1[l], B.dq, B.dk, B.dv, B.u[l], B.dgt, B.dup};
      for (int i = 0; i < kGrams; ++i) ga.A[i] = src[i];
      ga.d = d; ga.f = f; ga.T = T; ga.plan = gp; ga.G = B.G;
      gram_kernel<<<dim3(gp.pairs, gp.pieces(), ns), kGramThreads, 0, st>>>(ga);
      gram_dot_kernel<<<dim3(gp.dot_blocks, kDots, ns), 256, 0, st>>>(B.G, gp, slots + z0 * gp.dot_blocks, n_slots);
      std::swap(dh, dnext);
    }
    FIT_OK(ge);
    FIT_OK(cudaGetLastError());
  }
  // mean(theta^2) per tensor
  for (int l = 0; l < L; ++l) {
    SumSqArgs sa{};
    const void* ptr[kTensors] = {w->wq[l], w->wk[l], w->wv[l], w->wo[l], w->w_gate[l], w->w_up[l], w->w_down[l], w->attn_norm[l], w->ffn_norm[l]};
    const size_t dd = (size_t)d * d, fd = (size_t)f * d;
    const size_t n[kTensors] = {dd, dd, dd, dd, fd, fd, fd, (size_t)d, (size_t)d};
    for (int t = 0; t < kTensors; ++t) sa.w[t] = ptr[t], sa.n[t] = n[t];
    sum_sq_partial_kernel<WT><<<dim3(kMsBlocks, kTensors), 256, 0, st>>>(sa, B.ms_part + (size_t)l * kTensors * kMsBlocks);
  }
  finish_kernel<<<L * kTensors, 256, 0, st>>>(B.slots, n_slots, B.ms_part, B.out);
  FIT_OK(cudaGetLastError());
  return cudaMemcpyAsync(sums.data(), B.out, sums.size() * sizeof(double), cudaMemcpyDeviceToHost, st);
}

template <typename WT>
cudaError_t run(const sdfp_config& g, const sdfp_weights* w, cudaStream_t st, const int32_t* tokens, int n_seq, int seq_len,
                double* out_trace, double* out_fit) {
  const int T = seq_len - 1;
  int dev = 0, n_sm = 0;
  FIT_OK(cudaGetDevice(&dev));
  FIT_OK(cudaDeviceGetAttribute(&n_sm, cudaDevAttrMultiProcessorCount, dev));
  GemmRoom room;
  FIT_OK((gemm_prepare<WT, 32>(room.clusters[0])));
  FIT_OK((gemm_prepare<WT, 64>(room.clusters[1])));
  FIT_OK((gemm_prepare<WT, 128>(room.clusters[2])));
  // (the limits belong to the kernels and not to this call: constants, or calls on other threads would lower them under it)
  for (const void* k : {(const void*)attn_fwd_kernel, (const void*)attn_bwd_q_kernel})
    FIT_OK(cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)attn_smem(kFitMaxT)));
  // As many sequences at a time as fill kFitRows rows; fewer if the device has no room for their activations.  How sums are
  // cut and where they are kept follows the full group either way: free memory does not show in the results.
  const int full = std::max(1, std::min(n_seq, kFitRows / T));
  const GramPlan gp = gram_plan(T, full, g.d_model, g.d_ffn, n_sm);
  const int n_slots = full * std::max((g.d_model + kGainCols - 1) / kGainCols, gp.dot_blocks);
  for (int nb = full;; nb = (nb + 1) / 2) {
    Buffers B;
    Arena A;
    auto lay = [&] {
      A.used = 0;
      B.layout(A, g.n_layers, g.d_model, g.d_ffn, g.vocab, g.n_heads, g.head_dim, T, nb, nb * seq_len, gp.doubles(nb), n_slots);
    };
    lay();
    void* p = nullptr;
    const cudaError_t me = fit_alloc(&p, A.used, dev, st);
    if (me == cudaErrorMemoryAllocation && nb > 1) {
      cudaGetLastError();
      continue;
    }
    FIT_OK(me);
    A.base = reinterpret_cast<unsigned char*>(p);
    lay();
    const int L = g.n_layers;
    std::vector<double> sums((size_t)L * kTensors * 2);  // per (layer, tensor): sum over the sequences of the squared norm, sum of theta^2
    const cudaError_t e = run_in<WT>(g, w, st, tokens, n_seq, seq_len, sums, B, nb, full, n_sm, room, gp, n_slots);
    const cudaError_t fe = fit_free(p, A.used, st);
    if (e != cudaSuccess || fe != cudaSuccess) return e != cudaSuccess ? e : fe;
    const double d = g.d_model, f = g.d_ffn;
    for (int l = 0; l < L; ++l) {
      double tr = 0.0, ft = 0.0;
      for (int t = 0; t < kTensors; ++t) {
        const double n = t < T_GATE ? d * d : t < T_ATTN_NORM ? f * d : d;
        const double Tt = sums[((size_t)l * kTensors + t) * 2] / n_seq;
        tr += Tt;
        ft += Tt * (sums[((size_t)l * kTensors + t) * 2 + 1] / n);
      }
      out_trace[l] = tr;
      if (out_fit) out_fit[l] = ft;
    }
    return cudaSuccess;
  }
}
#undef FIT_OK

}  // namespace fit
}  // namespace sdfp
