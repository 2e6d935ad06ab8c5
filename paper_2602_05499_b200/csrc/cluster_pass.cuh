// Rounds of a small decoder inside ONE thread-block cluster of sixteen CTAs: the whole greedy generation loop (Algorithm 1,
// Stage B: k draft passes, verification, accept, commit) in one launch, or one pass of a sampled round.
//
// What bounds a small decoder is not its bytes but the chain of dependent stages, five a layer: spread over 148
// SMs a stage boundary is a grid-wide exchange through L2 (about 5 us in the whole-pass kernel, about 4 us as one
// launch per operation), for a fraction of a microsecond of work.  Sixteen SMs of one cluster hand their results on
// through distributed shared memory instead:
//   * Every linear stage gives each CTA an equal share of the output features.  The finished sums are gathered in shared
//     memory; behind one barrier of the CTA a half-warp takes four pairs at a time, a lane sends the result to each of the
//     sixteen CTAs with st.async, and the bytes complete a transaction count on an mbarrier of the receiver, which starts
//     its next stage when all shares have landed.  No barrier over the cluster stands between stages, and nothing
//     goes through L2 but weights and the K/V cache.  From the last send to the last arrival 300 clocks pass.
//   * The buffers need no second copy: a CTA writes into another's buffer only when it holds the complete output of a stage
//     that the other contributed to after its last read of that buffer.  Every CTA has a share of every stage of a layer.
//   * Weights: a warp owns output pairs and walks K with its lanes; the first step is on its way before the wait for the
//     activations.
//   * The residual stream, the next norm's input and the SwiGLU output of all rows live in every CTA's shared
//     memory in fp32; products are fp32 FMAs on exact activations.
//   * K/V: the rows of the running pass are taken from shared memory, older keys from the cache in global memory,
//     which the CTA that makes an entry also writes.
// What bounds it now is instructions, 10 700 a warp and pass at 4 layers d 256, six to seven clocks each with two warps on a
// scheduler (ncu): 16 warps, weights through a ring filled by a producer warp, eight lanes on K and the others on pairs or rows, and
// mma.sync for bf16 were built and were slower at one row (58, 82, 65 and 59 us a pass against 36); four and
// sixteen warps take 10 to 30 % longer than eight.  In us a pass, 4 layers, bf16, autoregressive, this kernel
// and the whole-pass kernel: d 256 37 and 126, d 384 50 and 136, d 512 59 and 142; fp32 and one launch per operation: 42 and 101,
// 57 and 110, 97 and 114.  The line to the other paths is at cluster_wanted in engine.cu.
//
// Batch invariance: a (row, feature) sum runs over K in an order fixed by the matrix, a (row, head) softmax over
// 4- or 8-key blocks dealt to the warps by absolute key index; neither depends on the rows of the pass.
#pragma once

#include "attention.cuh"
#include "common.cuh"
#include "linear_fma.cuh"
#include "misc_kernels.cuh"
#include "pass_kernel.cuh"

namespace sdfp {

constexpr int kClCtas = 16, kClWarps = 8, kClThreads = kClWarps * 32;
constexpr int kClMaxRows = 16;
constexpr int kClUnit = 1024;  // bytes of one K step of an output pair: 512 of either feature

enum ClBar { CL_BAR_H = 0, CL_BAR_U = 1, CL_BAR_QKV = 2, CL_BAR_X = 3, CL_BAR_TOK = 4, CL_BARS = 5 };
enum ClKind { CL_QKV = 0, CL_O = 1, CL_GATE_UP = 2, CL_DOWN = 3, CL_HEAD = 4 };

template <typename WT>
struct ClElem {
  static constexpr int kLane = 16 / (int)sizeof(WT);  // columns in a lane's sixteen bytes
  static constexpr int kStep = 32 * kLane;            // columns of a K step: 256 of bf16, 128 of fp32
};
__host__ __device__ __forceinline__ int cl_steps(int K, int elem_bytes) {
  const int step = 512 / elem_bytes;
  return (K + step - 1) / step;
}
// first pair of a CTA's share: pairs are dealt in fours, so that a share is sent sixteen bytes at a time
__host__ __device__ __forceinline__ int cl_first_pair(int n_pairs, int cta) { return (n_pairs / 4) * cta / kClCtas * 4; }
__host__ __device__ __forceinline__ int cl_max_pairs(int n_pairs) { return (n_pairs / 4 + kClCtas - 1) / kClCtas * 4; }

struct ClStage {  // a linear stage of a program; the attention follows a QKV stage without an entry of its own
  const unsigned char* W;  // [pair][step][1 KB], see pack_cluster_kernel
  void *kcache, *vcache;   // CL_QKV
  int kind, n_pairs, K;
  int gain_out;            // CL_O, CL_DOWN: which norm reads the residual stream next
  int after_kv;            // the first stage behind the last CL_O
};

struct ClTab {  // the same for this CTA, in shared memory
  const unsigned char* W;  // its first pair
  void *kcache, *vcache;
  int kind, np, steps, gain_out;
  int x, K, bar, row_bytes;  // its activations: where, columns, the barrier that brings them and their bytes per row
  int norm, p0;
  int after_kv;              // the first stage behind the last attention's O-projection
};

// Shared-memory layout, worked out on the host (bytes from the start)
struct ClLayout {
  int rows, splits, heads_per_cta, resid_np, stg_floats;
  int h, y, part, xp, xml, xo, u, qkv, gain, hres, stg, rope, tok, best, tab, shared, total;
};

struct ClParams {
  const ClStage* prog_t;
  const ClStage* prog_d;
  int n_t, n_d;              // stages to run of either
  int first_gain_t, first_gain_d;
  const float* gains;        // [n_gains][d]
  int n_gains;
  int d, f, heads, vocab, max_seq;
  float eps, scale;
  const float *rope_cos, *rope_sin;
  const void* embed;
  ClLayout lay;
  // what to run: greedy rounds until everything is finished, or one pass
  int rounds;                // > 0: at most this many greedy rounds
  int first_rows;            // rows per sequence of a round's first draft pass
  PassDesc pd;               // one pass: which of a round's, for sampled decoding (its logits go to `logits`)
  int draft;                 // ... and of which model
  float* logits;             // [rows][vocab]
  GenState* gs;
  int* seq_tok;
  int* draft_tok;
  int* out_tok;
  RoundStat* stats;
  PassSync* sync;
};

struct ClMine {  // this CTA's share of a kind of matrix
  int p0, np, nq;
  unsigned magic;  // i / nq == i * magic >> 20 for the few hundred vectors of a share
};

struct ClShared {
  uint64_t bar[CL_BARS];
  ClMine mine[5];     // by ClKind
  int abort;
  unsigned long long wait_limit_ns;
  unsigned sabotage;  // bytes the next wait expects in vain (PassSync::bar_extra)
  float inv[kClMaxRows];
  int pos[kClMaxRows];
  int amax[kClMaxRows];
  // state of the sequences
  int n[kMaxBatch], n_new[kMaxBatch], done[kMaxBatch];
  int last[kMaxBatch][2];  // the last two committed tokens
  int drafts[kMaxBatch][kMaxK];
  int all_done, round, max_new, eos_id, max_rounds;
};

extern __shared__ __align__(1024) unsigned char cl_smem[];
template <typename T>
__device__ __forceinline__ T* cl_at(int off) { return reinterpret_cast<T*>(cl_smem + off); }

// ---- PTX -----------------------------------------------------------------------------------------------
__device__ __forceinline__ uint32_t cl_rank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %cluster_ctarank;" : "=r"(r));
  return r;
}
__device__ __forceinline__ uint32_t cl_map(uint32_t addr, uint32_t cta) {
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(cta));
  return r;
}
__device__ __forceinline__ void cl_send4(uint32_t dst, const float4& v, uint32_t bar) {
  asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.v4.f32 [%0], {%1, %2, %3, %4}, [%5];" ::"r"(dst), "f"(v.x),
               "f"(v.y), "f"(v.z), "f"(v.w), "r"(bar)
               : "memory");
}
__device__ __forceinline__ void cl_send2(uint32_t dst, float x, float y, uint32_t bar) {
  asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.v2.f32 [%0], {%1, %2}, [%3];" ::"r"(dst), "f"(x), "f"(y), "r"(bar)
               : "memory");
}
__device__ __forceinline__ void cl_cluster_sync() {
  asm volatile("barrier.cluster.arrive.release.aligned;\nbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ bool cl_try_wait(uint32_t bar, unsigned parity) {
  unsigned ok;
  asm volatile(
      "{\n .reg .pred p;\n mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}"
      : "=r"(ok)
      : "r"(bar), "r"(parity)
      : "memory");
  return ok != 0;
}
__device__ __forceinline__ void cl_sync() { asm volatile("bar.sync 1, %0;" ::"n"(kClThreads) : "memory"); }  // the compute warps
// ... and the same answer to "has anything failed" for all of them
__device__ __forceinline__ bool cl_agree_ok(const int* abort_flag) {
  const int seen = *reinterpret_cast<const volatile int*>(abort_flag);
  unsigned any;
  asm volatile("{\n .reg .pred p, q;\n setp.ne.s32 p, %1, 0;\n bar.red.or.pred q, 1, %2, p;\n selp.u32 %0, 1, 0, q;\n}"
               : "=r"(any)
               : "r"(seen), "n"(kClThreads)
               : "memory");
  return any == 0;
}
__device__ __forceinline__ bool cl_aborted(const ClShared* sh) { return *reinterpret_cast<const volatile int*>(&sh->abort) != 0; }

// Poll one of the CTA's barriers.  A wait that runs out records the error, and from then on the CTA only walks to its
// end: every later wait returns at once, nothing is sent any more, and what is computed is not used (whatever is derived
// from it keeps its range).
__device__ __noinline__ void cl_poll(ClShared* sh, PassSync* sync, uint32_t bar, unsigned parity) {
  const unsigned long long t0 = global_ns();
  unsigned spins = 0;
#pragma unroll 1
  while (!cl_try_wait(bar, parity)) {
    if ((++spins & 15u) == 0) {
      if (cl_aborted(sh)) break;
      if (global_ns() - t0 > sh->wait_limit_ns) {
        atomicCAS(&sync->error, 0, (int)PASS_ERR_GRID_BARRIER);
        *reinterpret_cast<volatile int*>(&sh->abort) = 1;
        break;
      }
    }
  }
}
// Wait for a buffer the other CTAs fill.  Their bytes may have been counted before the barrier is told how many to expect.
__device__ __forceinline__ void cl_wait(ClShared* sh, PassSync* sync, int which, unsigned bytes, unsigned parity) {
  if (cl_aborted(sh)) return;  // a phase that never ended must not be armed again
  if (threadIdx.x == kClThreads - 1) {
    mbar_arrive_expect_tx(&sh->bar[which], bytes + sh->sabotage);
    sh->sabotage = 0;
  }
  const uint32_t bar = smem_u32(&sh->bar[which]);
  if (!cl_try_wait(bar, parity)) cl_poll(sh, sync, bar, parity);
  __syncwarp();
}

// ---- dot products of a stage ------------------------------------------------------------------------------------
struct ClDots {
  const unsigned char* W;    // this CTA's pairs
  int np, x, K, steps;       // its pairs; activations (offset of [row][K]) and matrix
  int R;
  int bar;                   // what brings the activations (ClBar), -1: nothing to wait for
  unsigned bytes, parity;
  bool norm;                 // the rows' norms are wanted
  bool head;                 // lm-head: logits [row][vocab] or, without, the best of each (row, warp, place in the warp)
  int stg;                   // out: [half][row][np] sums
  int p0;
  float* logits;
};

// Everything that has to be there before the first product
__device__ __forceinline__ void cl_begin(const ClParams& p, const ClDots& a, ClShared* sh) {
  if (a.bar >= 0) cl_wait(sh, p.sync, a.bar, a.bytes, a.parity);
  if (a.norm) {  // the factors are needed behind the dot products only: the last warps, which have the fewest pairs, work them out
    const int lane = threadIdx.x & 31;
#pragma unroll 1
    for (int row = kClWarps - 1 - (threadIdx.x >> 5); row < a.R; row += kClWarps) {
      const float* h = cl_at<float>(p.lay.h) + row * p.d;
      float s = 0.f;
#pragma unroll 2
      for (int c = lane * 4; c < p.d; c += 128) {
        const float4 v = *reinterpret_cast<const float4*>(h + c);
        s = fmaf(v.x, v.x, s);
        s = fmaf(v.y, v.y, s);
        s = fmaf(v.z, v.z, s);
        s = fmaf(v.w, v.w, s);
      }
      s = warp_sum(s);
      if (lane == 0) sh->inv[row] = rsqrtf(s * (1.0f / (float)p.d) + p.eps);
    }
  }
  if (a.head) cl_sync();  // the logits are scaled where they are made
}

template <typename WT>
__device__ __forceinline__ void cl_fma(float& t, const uint4& w, const float4& x0, const float4& x1) {
  if (sizeof(WT) == 2) {
    t = fmaf(__uint_as_float(w.x << 16), x0.x, t);
    t = fmaf(__uint_as_float(w.x & 0xffff0000u), x0.y, t);
    t = fmaf(__uint_as_float(w.y << 16), x0.z, t);
    t = fmaf(__uint_as_float(w.y & 0xffff0000u), x0.w, t);
    t = fmaf(__uint_as_float(w.z << 16), x1.x, t);
    t = fmaf(__uint_as_float(w.z & 0xffff0000u), x1.y, t);
    t = fmaf(__uint_as_float(w.w << 16), x1.z, t);
    t = fmaf(__uint_as_float(w.w & 0xffff0000u), x1.w, t);
  } else {
    t = fmaf(__uint_as_float(w.x), x0.x, t);
    t = fmaf(__uint_as_float(w.y), x0.y, t);
    t = fmaf(__uint_as_float(w.z), x0.z, t);
    t = fmaf(__uint_as_float(w.w), x0.w, t);
  }
}
__device__ __forceinline__ int cl_feature(int pair) { return ((pair >> 3) << 4) + (pair & 7); }  // the first of a pair's features, its second is 8 further

// A warp's pairs lie behind one another in memory.  It takes P of them through RT rows at a time (more rows take another
// sweep of the weights, from L2); a K step of weights is in registers or on its way, the first before the wait for the
// activations.  (Two to four steps ahead, in as many copies of the loop's body, were slower: tiny decoders by 4 %.)  A sum is made
// in the same order whatever P and RT: K steps in order by each lane, the lanes in the xor tree.
template <typename WT, int RT, int P>
__device__ __forceinline__ void cl_dots(const ClParams& p, const ClDots& a, ClShared* sh) {
  constexpr bool BF = sizeof(WT) == 2;
  constexpr int N = RT * P * 2, CH = N < 16 ? N : 16;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int n_w = RT == 1 ? (a.np + kClWarps - 1) / kClWarps : (a.np / 2 + kClWarps - 1) / kClWarps * 2;  // pairs per warp
  const int first = warp * n_w, cnt = max(0, min(n_w, a.np - first));
  const int pair_len = a.steps * (kClUnit / 16);
#pragma unroll 1
  for (int r0 = 0; r0 < a.R; r0 += RT) {
    const int rows = RT == 1 ? 1 : min(RT, a.R - r0);
    const uint4* w = reinterpret_cast<const uint4*>(a.W) + (size_t)first * pair_len + lane;
    int ask_pairs = cnt, ask_steps = a.steps;  // pairs from the next request's on, steps left of them
    uint4 raw[P][2];
    auto ask = [&]() {
      if (ask_pairs <= 0) return;
#pragma unroll
      for (int j = 0; j < P; ++j)
        if (j < ask_pairs) {
          raw[j][0] = __ldg(w + j * pair_len);
          raw[j][1] = __ldg(w + j * pair_len + 32);
        }
      w += kClUnit / 16;
      if (--ask_steps == 0) {
        ask_steps = a.steps;
        ask_pairs -= P;
        w += (P - 1) * pair_len;
      }
    };
    ask();
    if (r0 == 0) cl_begin(p, a, sh);
    const float* const x = cl_at<float>(a.x) + r0 * a.K + lane * 4;
    const int room = a.K - lane * 4;
#pragma unroll 1
    for (int at = 0; at < cnt; at += P) {  // first pair of the running P
      float acc[N];
#pragma unroll
      for (int i = 0; i < N; ++i) acc[i] = 0.f;
#pragma unroll 1
      for (int c0 = 0; c0 < a.K; c0 += ClElem<WT>::kStep) {
        const bool in0 = c0 < room, in1 = BF && c0 + 128 < room;
#pragma unroll
        for (int i = 0; i < RT; ++i) {
          if (RT == 1 || i < rows) {
            float4 x0 = make_float4(0.f, 0.f, 0.f, 0.f), x1 = x0;
            if (in0) x0 = *reinterpret_cast<const float4*>(x + i * a.K + c0);
            if (in1) x1 = *reinterpret_cast<const float4*>(x + i * a.K + c0 + 128);
#pragma unroll
            for (int j = 0; j < P; ++j)
              if (RT > 1 || j < cnt - at) {
                cl_fma<WT>(acc[(i * P + j) * 2], raw[j][0], x0, x1);
                cl_fma<WT>(acc[(i * P + j) * 2 + 1], raw[j][1], x0, x1);
              }
          }
        }
        ask();
      }
      // lane groups end up with one (row, pair, half) each; both halves of a pair in the lane that uses them
#pragma unroll
      for (int g = 0; g < N; g += CH) {
        if (g / (2 * P) < rows) {
          float v[CH];
#pragma unroll
          for (int i = 0; i < CH; ++i) v[i] = acc[g + i];
          float v0 = warp_sum_scatter<CH>(v);
          float v1 = __shfl_xor_sync(0xffffffffu, v0, 32 / CH);
          const int pi = (g + lane / (32 / CH)) >> 1, row = r0 + pi / P, pl = first + at + pi % P;
          if (lane % (64 / CH) == 0 && row < a.R && at + pi % P < cnt) {
            if (!a.head) {
              float* o = cl_at<float>(a.stg) + row * a.np + pl;
              o[0] = v0;
              o[a.R * a.np] = v1;
            } else {
              const int f0 = cl_feature(a.p0 + pl);
              const float inv = sh->inv[row];
              v0 *= inv;
              v1 *= inv;
              if (a.logits != nullptr) {
                float* o = a.logits + (size_t)row * p.vocab + f0;
                o[0] = v0;
                o[8] = v1;
              } else {  // only this lane touches its place
                float2* best = cl_at<float2>(p.lay.best) + row * 4 * kClWarps + warp * 4 + pi % P;
                const float2 o = *best;
                const bool second = v1 > v0;
                const float bv = second ? v1 : v0;
                const int bi = second ? f0 + 8 : f0;
                if (bv > o.x || (bv == o.x && bi < __float_as_int(o.y))) *best = make_float2(bv, __int_as_float(bi));
              }
            }
          }
        }
      }
    }
  }
}

// the CTAs that hold a head: CTA c has heads c, c + 16, ...; with fewer heads than CTAs, `splits` CTAs share one
__device__ __forceinline__ int cl_heads_of(int cta, int heads, int splits) {
  if (heads >= kClCtas) return (heads - cta + kClCtas - 1) / kClCtas;
  return cta < heads * splits ? 1 : 0;
}

struct ClEnv {
  ClShared* sh;
  int warp, lane, rank;
  int R, rps;          // rows of the pass, rows per sequence; sequence b has cache slot b
  uint32_t self, dst;  // shared memory of this CTA (as an address of the cluster's), of CTA tid mod 16: what goes to all CTAs is sent by a thread each
  int stg;             // where the sums of the running stage are: two places in turn, a slow warp may still read the other
  int hres;            // residual rows of this CTA's features: likewise two places in turn
};
__device__ __forceinline__ uint32_t cl_bar_of(const ClParams& p, uint32_t cta, int which) {
  return cta + p.lay.shared + (int)offsetof(ClShared, bar) + which * 8;
}
__device__ __forceinline__ float4 cl_scale(float4 v, float s) { return make_float4(v.x * s, v.y * s, v.z * s, v.w * s); }

// ---- epilogues: four pairs of a row at a time, behind one barrier of the CTA ------------------------------------------
// Rotary embedding, cache entries, and q, k, v to the CTAs that work on the head; a thread per vector
template <typename WT, int HD>
__device__ __forceinline__ void cl_finish_qkv(const ClParams& p, const ClEnv& ev, const ClTab& t, bool send) {
  constexpr int hp = HD / 2;
  const ClMine me = ev.sh->mine[CL_QKV];
  const float4* s0 = cl_at<float4>(ev.stg);
  const float4* s1 = s0 + ev.R * me.nq;
  const int per = p.d >> 1;
#pragma unroll 1
  for (int i = kClThreads - 1 - threadIdx.x; i < ev.R * me.nq; i += kClThreads) {
    const int row = (int)((unsigned)i * me.magic >> 20), pair = me.p0 + 4 * (i - row * me.nq);
    const int which = pair >= 2 * per ? 2 : pair >= per ? 1 : 0, rem = pair - which * per, head = rem / hp, d0 = rem % hp;
    const int pos = ev.sh->pos[row];
    const float inv = ev.sh->inv[row];
    float4 a = cl_scale(s0[i], inv), b = cl_scale(s1[i], inv);
    if (which < 2) {
      const float* rp = cl_at<float>(p.lay.rope) + row * 2 * hp + d0;
      const float4 c = *reinterpret_cast<const float4*>(rp), s = *reinterpret_cast<const float4*>(rp + hp);
      const float4 r = make_float4(a.x * c.x - b.x * s.x, a.y * c.y - b.y * s.y, a.z * c.z - b.z * s.z, a.w * c.w - b.w * s.w);
      b = make_float4(b.x * c.x + a.x * s.x, b.y * c.y + a.y * s.y, b.z * c.z + a.z * s.z, b.w * c.w + a.w * s.w);
      a = r;
    }
    if (which > 0) {
      WT* dst = reinterpret_cast<WT*>(which == 1 ? t.kcache : t.vcache) + (((size_t)(row / ev.rps) * p.heads + head) * p.max_seq + pos) * HD + d0;
      if constexpr (sizeof(WT) == 2) {  // the rows of this pass see what the cache will hold
        const __nv_bfloat162 a0 = __floats2bfloat162_rn(a.x, a.y), a1 = __floats2bfloat162_rn(a.z, a.w);
        const __nv_bfloat162 b0 = __floats2bfloat162_rn(b.x, b.y), b1 = __floats2bfloat162_rn(b.z, b.w);
        if (pos >= 0) {
          *reinterpret_cast<uint2*>(dst) = make_uint2(*reinterpret_cast<const uint32_t*>(&a0), *reinterpret_cast<const uint32_t*>(&a1));
          *reinterpret_cast<uint2*>(dst + hp) = make_uint2(*reinterpret_cast<const uint32_t*>(&b0), *reinterpret_cast<const uint32_t*>(&b1));
        }
        a = make_float4(__low2float(a0), __high2float(a0), __low2float(a1), __high2float(a1));
        b = make_float4(__low2float(b0), __high2float(b0), __low2float(b1), __high2float(b1));
      } else if (pos >= 0) {
        *reinterpret_cast<float4*>(dst) = a;
        *reinterpret_cast<float4*>(dst + hp) = b;
      }
    }
    if (!send) continue;
    const int hl = p.heads >= kClCtas ? head / kClCtas : 0;
    const int off = p.lay.qkv + (((hl * 3 + which) * ev.R + row) * HD + d0) * 4;
#pragma unroll 1
    for (int s = 0, cta = p.heads >= kClCtas ? head % kClCtas : head; s < p.lay.splits; ++s, cta += p.heads) {
      const uint32_t to = cl_map(ev.self, cta), bar = cl_bar_of(p, to, CL_BAR_QKV);
      cl_send4(to + off, a, bar);
      cl_send4(to + off + hp * 4, b, bar);
    }
  }
}

// (what goes to all CTAs: a half-warp per vector, a lane per CTA)
__device__ __forceinline__ void cl_finish_gate_up(const ClParams& p, const ClEnv& ev) {
  const ClMine me = ev.sh->mine[CL_GATE_UP];
  const float4* s0 = cl_at<float4>(ev.stg);
  const float4* s1 = s0 + ev.R * me.nq;
  const uint32_t bar = cl_bar_of(p, ev.dst, CL_BAR_U);
  auto f = [](float g, float u) { return g / (1.0f + __expf(-g)) * u; };
#pragma unroll 1
  for (int i = threadIdx.x >> 4; i < ev.R * me.nq; i += kClThreads / 16) {
    const int row = (int)((unsigned)i * me.magic >> 20), j = me.p0 + 4 * (i - row * me.nq);
    const float inv = ev.sh->inv[row];
    const float4 g = cl_scale(s0[i], inv), u = cl_scale(s1[i], inv);
    cl_send4(ev.dst + p.lay.u + (row * p.f + j) * 4, make_float4(f(g.x, u.x), f(g.y, u.y), f(g.z, u.z), f(g.w, u.w)), bar);
  }
}

// new residual rows, and the same times the next norm's gain
__device__ __forceinline__ void cl_finish_resid(const ClParams& p, ClEnv& ev, const ClTab& t) {
  const ClMine me = ev.sh->mine[CL_O];
  const int half_len = p.lay.rows * p.lay.resid_np;
  const int next = p.lay.hres + (ev.hres == p.lay.hres ? half_len * 8 : 0);
  const float4* sum = cl_at<float4>(ev.stg);
  const uint32_t bar = cl_bar_of(p, ev.dst, CL_BAR_H);
  const float* gain = cl_at<float>(p.lay.gain) + t.gain_out * 2 * p.lay.resid_np;
#pragma unroll 1
  for (int i = threadIdx.x >> 4; i < 2 * ev.R * me.nq; i += kClThreads / 16) {
    const int rr = (int)((unsigned)i * me.magic >> 20), half = rr >= ev.R ? 1 : 0, row = rr - half * ev.R;
    const int pl = 4 * (i - rr * me.nq), at = half * half_len + row * p.lay.resid_np + pl;
    const float4 v = sum[i], o = *reinterpret_cast<const float4*>(cl_at<float>(ev.hres) + at);
    const float4 g = *reinterpret_cast<const float4*>(gain + half * p.lay.resid_np + pl);
    const float4 n = make_float4(o.x + v.x, o.y + v.y, o.z + v.z, o.w + v.w);
    if ((threadIdx.x & 15) == 0) *reinterpret_cast<float4*>(cl_at<float>(next) + at) = n;
    const int off = (row * p.d + cl_feature(me.p0 + pl) + half * 8) * 4;
    cl_send4(ev.dst + p.lay.y + off, make_float4(n.x * g.x, n.y * g.y, n.z * g.z, n.w * g.w), bar);
    cl_send4(ev.dst + p.lay.h + off, n, bar);
  }
  ev.hres = next;
}

// ---- attention ------------------------------------------------------------------------------------------------
// The keys of a (row, head) in blocks of KPB, dealt by absolute index over `splits` CTAs and their eight warps:
// block kb belongs to place kb mod (8 splits) = warp * splits + split.  LPK lanes hold a key, sixteen dimensions each;
// every lane group keeps its own running maximum, the groups are combined at the end.
template <typename WT, int HD>
struct ClAttn {
  static constexpr int LPK = HD / 16, KPB = 32 / LPK, V = ClElem<WT>::kLane, NV = 16 / V;
  uint4 rk[NV], rv[NV];  // a block as it lies in the cache
  __device__ __forceinline__ void load(const WT* gk, const WT* gv, int key, int dl, bool in) {
#pragma unroll
    for (int j = 0; j < NV; ++j) {
      rk[j] = rv[j] = make_uint4(0u, 0u, 0u, 0u);
      if (in) {
        rk[j] = __ldcg(reinterpret_cast<const uint4*>(gk + (size_t)key * HD + (j * LPK + dl) * V));
        rv[j] = __ldcg(reinterpret_cast<const uint4*>(gv + (size_t)key * HD + (j * LPK + dl) * V));
      }
    }
  }
  static __device__ __forceinline__ void widen(const uint4 (&r)[NV], float (&o)[16]) {
#pragma unroll
    for (int j = 0; j < NV; ++j) {
      const uint32_t w[4] = {r[j].x, r[j].y, r[j].z, r[j].w};
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        if (sizeof(WT) == 2) {
          o[j * V + 2 * e] = __uint_as_float(w[e] << 16);
          o[j * V + 2 * e + 1] = __uint_as_float(w[e] & 0xffff0000u);
        } else {
          o[j * V + e] = __uint_as_float(w[e]);
        }
      }
    }
  }
};

// row r of sequence b; `blk` holds the place's first block as far as it lies in the cache, if `loaded`
template <typename WT, int HD>
__device__ __forceinline__ void cl_attend(const ClParams& p, const ClEnv& ev, const WT* gk, const WT* gv, int hl, int b, int r, int place, int split,
                                          ClAttn<WT, HD>& blk, bool loaded) {
  using A = ClAttn<WT, HD>;
  constexpr int LPK = A::LPK, KPB = A::KPB, V = A::V, NV = A::NV;
  const int lane = ev.lane, kl = lane / LPK, dl = lane % LPK, R = ev.R, rps = ev.rps;
  const int row = b * rps + r, pos = ev.sh->pos[row];
  const int S = p.lay.splits, first = place * S + split;
  if (first * KPB > pos) return;  // also a row that carries nothing
  const int p_last = ev.sh->pos[b * rps + rps - 1], base_pos = max(0, p_last - rps + 1);
  const float* q = cl_at<float>(p.lay.qkv) + (hl * 3 * R + row) * HD;
  const float* sk = cl_at<float>(p.lay.qkv) + (hl * 3 + 1) * R * HD;
  const float* sv = sk + R * HD;
  float m = -INFINITY, l = 0.f, o[16];
#pragma unroll
  for (int e = 0; e < 16; ++e) o[e] = 0.f;
#pragma unroll 1
  for (int kb = first; kb * KPB <= pos; kb += kClWarps * S) {
    const int key = kb * KPB + kl;
    if (!loaded) blk.load(gk, gv, key, dl, key < base_pos);
    loaded = false;
    float k[16], v[16];
    A::widen(blk.rk, k);
    A::widen(blk.rv, v);
    if (key >= base_pos && key <= pos) {
      const int kr = b * rps + rps - 1 - (p_last - key);
#pragma unroll
      for (int j = 0; j < NV; ++j)
#pragma unroll
        for (int e = 0; e < V; e += 4) {
          const int dim = (j * LPK + dl) * V + e;
          const float4 x = *reinterpret_cast<const float4*>(sk + kr * HD + dim), c = *reinterpret_cast<const float4*>(sv + kr * HD + dim);
          k[j * V + e] = x.x, k[j * V + e + 1] = x.y, k[j * V + e + 2] = x.z, k[j * V + e + 3] = x.w;
          v[j * V + e] = c.x, v[j * V + e + 1] = c.y, v[j * V + e + 2] = c.z, v[j * V + e + 3] = c.w;
        }
    }
    float s4[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
    for (int j = 0; j < NV; ++j)
#pragma unroll
      for (int e = 0; e < V; e += 4) {
        const float4 x = *reinterpret_cast<const float4*>(q + (j * LPK + dl) * V + e);
        s4[0] = fmaf(x.x, k[j * V + e], s4[0]);
        s4[1] = fmaf(x.y, k[j * V + e + 1], s4[1]);
        s4[2] = fmaf(x.z, k[j * V + e + 2], s4[2]);
        s4[3] = fmaf(x.w, k[j * V + e + 3], s4[3]);
      }
    float s = (s4[0] + s4[1]) + (s4[2] + s4[3]);
#pragma unroll
    for (int w = 1; w < LPK; w <<= 1) s += __shfl_xor_sync(0xffffffffu, s, w);
    s = key <= pos ? s * p.scale : -INFINITY;
    const float mn = fmaxf(m, s), ms = mn == -INFINITY ? 0.f : mn;
    const float a = __expf(m - ms), pr = __expf(s - ms);
    m = mn;
    l = fmaf(l, a, pr);
#pragma unroll
    for (int e = 0; e < 16; ++e) o[e] = fmaf(pr, v[e], o[e] * a);
  }
  constexpr int LEFT = 16 / KPB;  // dimensions a lane ends up with
  float mx = m;
#pragma unroll
  for (int w = LPK; w < 32; w <<= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, w));
  const float fac = __expf(m - mx);  // the first block has a key the row sees: mx is finite
  l *= fac;
#pragma unroll
  for (int w = LPK; w < 32; w <<= 1) l += __shfl_xor_sync(0xffffffffu, l, w);
#pragma unroll
  for (int e = 0; e < 16; ++e) o[e] *= fac;
  int at = 0;  // first of the lane's sixteen values
#pragma unroll
  for (int w = 16, n = 8; w >= LPK; w >>= 1, n >>= 1) {
    const bool up = (lane & w) != 0;
#pragma unroll
    for (int e = 0; e < 8; ++e)
      if (e < n) {
        const float keep = up ? o[e + n] : o[e], give = up ? o[e] : o[e + n];
        o[e] = keep + __shfl_xor_sync(0xffffffffu, give, w);
      }
    at += up ? n : 0;
  }
  float* dst = cl_at<float>(p.lay.part) + ((hl * R + row) * kClWarps + place) * (HD + 4);
  const int dim = ((at / V) * LPK + dl) * V + at % V;
#pragma unroll
  for (int e = 0; e < LEFT; e += 2) *reinterpret_cast<float2*>(dst + dim + e) = make_float2(o[e], o[e + 1]);
  if (lane == 0) *reinterpret_cast<float2*>(dst + HD) = make_float2(mx, l);
}

// Attention of this CTA's heads and the sending of its outcome.  One CTA per head sends the output, several per head
// their unnormalised sums and (max, sum).
template <typename WT, int HD>
__device__ __forceinline__ void cl_attention(const ClParams& p, const ClEnv& ev, const ClTab& t, int nh, unsigned parity) {
  using A = ClAttn<WT, HD>;
  const int S = p.lay.splits, R = ev.R, rps = ev.rps;
  const bool many = p.heads >= kClCtas;
  const int split = many ? 0 : ev.rank / p.heads;
  const int head0 = many ? ev.rank : ev.rank - split * p.heads;
  auto cache_at = [&](void* base, int hl, int b) {
    return reinterpret_cast<const WT*>(base) + ((size_t)b * p.heads + head0 + hl * kClCtas) * p.max_seq * HD;
  };
  const int n_seq = R / rps;
  A blk;
  {  // the first block of this warp's first place, as far as it lies in the cache: asked for before the wait
    const int p_last = ev.sh->pos[rps - 1], key = (ev.warp * S + split) * A::KPB + ev.lane / A::LPK;
    blk.load(cache_at(t.kcache, 0, 0), cache_at(t.vcache, 0, 0), key, ev.lane % A::LPK, key < max(0, p_last - rps + 1));
  }
  cl_wait(ev.sh, p.sync, CL_BAR_QKV, (unsigned)(nh * 3 * R * HD * 4), parity);
  int turn = ev.warp;  // short contexts fill only the first places: other warps take them in every item
  bool loaded = true;
#pragma unroll 1
  for (int hl = 0; hl < nh; ++hl)
#pragma unroll 1
    for (int b = 0; b < n_seq; ++b) {
      const WT *gk = cache_at(t.kcache, hl, b), *gv = cache_at(t.vcache, hl, b);
#pragma unroll 1
      for (int r0 = 0; r0 < rps; ++r0) {
        cl_attend<WT, HD>(p, ev, gk, gv, hl, b, r0, turn & (kClWarps - 1), split, blk, loaded);
        turn += 3;
        loaded = false;
      }
    }
  cl_sync();
  // the places of every row, in order
  float* stg = cl_at<float>(ev.stg);  // [hl][row][HD], behind it [hl][row][2]
#pragma unroll 1
  for (int e = ev.warp * 32 + ev.lane; e < nh * R * HD; e += kClThreads) {
    const int hr = e / HD, dim = e % HD, row = nh == 1 ? hr : hr % R;
    const int pos = ev.sh->pos[row];
    const int blocks = pos < 0 ? 0 : pos / A::KPB + 1;  // ... that the row sees; this CTA's places among them:
    const int na = blocks > split ? min(kClWarps, (blocks - split + S - 1) / S) : 0;
    const float* q = cl_at<float>(p.lay.part) + hr * kClWarps * (HD + 4);
    float mx = -INFINITY, l = 0.f, o = 0.f;
    float2 ml[kClWarps];
    float v[kClWarps];
#pragma unroll
    for (int w = 0; w < kClWarps; ++w) {
      ml[w] = make_float2(-INFINITY, 0.f);
      v[w] = 0.f;
      if (w < na) {
        ml[w] = *reinterpret_cast<const float2*>(q + w * (HD + 4) + HD);
        v[w] = q[w * (HD + 4) + dim];
      }
    }
#pragma unroll
    for (int w = 0; w < kClWarps; ++w) mx = fmaxf(mx, ml[w].x);
#pragma unroll
    for (int w = 0; w < kClWarps; ++w)
      if (w < na) {
        const float a = __expf(ml[w].x - mx);
        l = fmaf(ml[w].y, a, l);
        o = fmaf(v[w], a, o);
      }
    if (S == 1)
      o *= l > 0.f ? 1.0f / l : 0.f;
    else if (dim == 0)
      *reinterpret_cast<float2*>(stg + nh * R * HD + hr * 2) = make_float2(mx, l);
    stg[e] = o;
  }
  cl_sync();
  if (cl_aborted(ev.sh)) return;
  const uint32_t bar = cl_bar_of(p, ev.dst, CL_BAR_X);
  const uint32_t base = ev.dst + (S == 1 ? p.lay.xo : p.lay.xp + split * R * p.d * 4);
#pragma unroll 1
  for (int i = threadIdx.x >> 4; i < nh * R * (HD / 4); i += kClThreads / 16) {
    const int hr = i / (HD / 4), dim = (i % (HD / 4)) * 4, hl = nh == 1 ? 0 : hr / R, row = hr - hl * R;
    cl_send4(base + (row * p.d + (head0 + hl * kClCtas) * HD + dim) * 4, reinterpret_cast<const float4*>(stg)[i], bar);
  }
  if (S > 1)
#pragma unroll 1
    for (int row = threadIdx.x >> 4; row < R; row += kClThreads / 16) {  // fewer heads than CTAs: one head here
      const float2 ml = *reinterpret_cast<const float2*>(stg + R * HD + row * 2);
      cl_send2(ev.dst + p.lay.xml + ((split * R + row) * p.heads + head0) * 8, ml.x, ml.y, bar);
    }
}

// splits > 1: the attention output from the CTAs' partial softmaxes, in split order
template <int HD>
__device__ __forceinline__ void cl_fold_splits(const ClParams& p, const ClEnv& ev) {
  const int S = p.lay.splits, R = ev.R;
  const float2* ml = cl_at<float2>(p.lay.xml);
  const float* xp = cl_at<float>(p.lay.xp);
  const int quads = p.d / 4;
#pragma unroll 1
  for (int e = ev.warp * 32 + ev.lane; e < R * quads; e += kClThreads) {
    const int row = R == 1 ? 0 : e / quads, col = (e - row * quads) * 4, head = col / HD;
    float mx = -INFINITY, l = 0.f;
#pragma unroll 1
    for (int s = 0; s < S; ++s) {
      const float2 v = ml[(s * R + row) * p.heads + head];
      if (v.y > 0.f) mx = fmaxf(mx, v.x);
    }
    float4 o = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll 1
    for (int s = 0; s < S; ++s) {
      const float2 v = ml[(s * R + row) * p.heads + head];
      const float a = v.y > 0.f ? __expf(v.x - mx) : 0.f;
      const float4 x = *reinterpret_cast<const float4*>(xp + (s * R + row) * p.d + col);
      l = fmaf(v.y, a, l);
      o.x = fmaf(x.x, a, o.x);
      o.y = fmaf(x.y, a, o.y);
      o.z = fmaf(x.z, a, o.z);
      o.w = fmaf(x.w, a, o.w);
    }
    *reinterpret_cast<float4*>(cl_at<float>(p.lay.xo) + row * p.d + col) = cl_scale(o, l > 0.f ? 1.0f / l : 0.f);
  }
}

// What a pass's row carries
__device__ __forceinline__ void cl_plan_row(const ClShared* sh, int kind, int step, int rps, int row, int& tok, int& pos) {
  tok = 0;
  pos = -1;
  const int b = row / rps, i = row - b * rps;
  if (sh->done[b]) return;
  const int n = sh->n[b];
  if (kind == PASS_DRAFT_FIRST) {
    pos = n - rps + i;
    tok = pos >= 0 ? sh->last[b][2 - rps + i] : 0;
  } else if (kind == PASS_DRAFT_NEXT) {
    pos = n - 1 + step;
    tok = sh->drafts[b][step - 1];
  } else {
    pos = n - 1 + i;
    tok = i == 0 ? sh->last[b][1] : sh->drafts[b][i - 1];
  }
}

// the better of (value, index) over `n` neighbouring lanes, ties to the lower index
template <int n>
__device__ __forceinline__ void cl_best_of_lanes(float& bv, int& bi) {
#pragma unroll
  for (int o = n / 2; o > 0; o >>= 1) {
    const float ov = __shfl_xor_sync(0xffffffffu, bv, o);
    const int oi = __shfl_xor_sync(0xffffffffu, bi, o);
    if (ov > bv || (ov == bv && oi < bi)) {
      bv = ov;
      bi = oi;
    }
  }
}

// accept (Eq. 2: draft token == target's argmax) and commit, one lane per sequence; every CTA keeps the state, CTA 0
// writes the results
__device__ __forceinline__ void cl_commit(const ClParams& p, ClShared* sh, int batch, int k, bool write, int b) {
  int fin = 1;
  const int round = sh->round, max_new = sh->max_new, eos_id = sh->eos_id;
  if (b < batch) {
    RoundStat st{0, 0, 0};
    const int n = sh->n[b], made = sh->n_new[b], room = max_new - made;
    int last = sh->last[b][1], before = 0;
    fin = sh->done[b];
    if (!fin) {
      const int* tgt = &sh->amax[b * (k + 1)];
      int j = 0;
#pragma unroll 1
      while (j < k && sh->drafts[b][j] == tgt[j]) ++j;
      int cnt = 0;
      bool eos = false;
#pragma unroll 1
      for (int i = 0; i <= j && cnt < room && !eos; ++i) {
        const int tok = tgt[i];  // an accepted draft token is the target's
        if (write) {
          p.seq_tok[(size_t)b * p.max_seq + n + cnt] = tok;
          p.out_tok[(size_t)b * max_new + made + cnt] = tok;
        }
        before = last;
        last = tok;
        ++cnt;
        eos = eos_id >= 0 && tok == eos_id;
      }
      sh->last[b][0] = before;
      sh->last[b][1] = last;
      sh->n[b] = n + cnt;
      sh->n_new[b] = made + cnt;
      fin = eos || made + cnt >= max_new ? 1 : 0;
      sh->done[b] = fin;
      st = RoundStat{k, j, cnt};
    }
    if (write && round < sh->max_rounds) p.stats[(size_t)round * batch + b] = st;
  }
  const bool all = __all_sync(0xffffffffu, fin);
  if (b == 0) {
    sh->round = round + 1;
    sh->all_done = all ? 1 : 0;
  }
}

template <typename WT, int HD>
__device__ __forceinline__ void cl_compute(const ClParams& p, ClShared* sh, const ClTab* tab_t, const ClTab* tab_d, int rank, bool loop, int batch, int k) {
  const int tid = threadIdx.x;
  ClEnv ev{};
  ev.sh = sh;
  ev.warp = tid >> 5;
  ev.lane = tid & 31;
  ev.rank = rank;
  ev.self = smem_u32(cl_smem);
  ev.dst = cl_map(ev.self, tid & (kClCtas - 1));
  ev.stg = p.lay.stg;
  ev.hres = p.lay.hres;
  auto other_stg = [&] { ev.stg = 2 * p.lay.stg + p.lay.stg_floats * 4 - ev.stg; };
  const int my_heads = cl_heads_of(rank, p.heads, p.lay.splits);
  unsigned phases = 0;
  auto phase = [&](int which) {
    const unsigned par = (phases >> which) & 1u;
    phases ^= 1u << which;
    return par;
  };

#pragma unroll 1
  for (int pass = 0;; pass = pass == k ? 0 : pass + 1) {  // loop mode: the number in the round, k = verification
    const bool verify = pass == k;
    const bool draft = loop ? !verify : p.draft != 0;
    const int kind = loop ? (verify ? PASS_VERIFY : pass == 0 ? PASS_DRAFT_FIRST : PASS_DRAFT_NEXT) : p.pd.kind;
    ev.rps = loop ? (verify ? k + 1 : pass == 0 ? p.first_rows : 1) : p.pd.rows_per_seq;
    ev.R = ev.rps * batch;
    const int R = ev.R;
    const ClTab* tab = draft ? tab_d : tab_t;
    const int n_stages = draft ? p.n_d : p.n_t;

    // ---- tokens, embedding, rotary factors: warp r does rows r and r + 8 ----
#pragma unroll 1
    for (int row = ev.warp; row < R; row += kClWarps) {
      int tok, pos;
      cl_plan_row(sh, kind, loop ? pass : p.pd.step, ev.rps, row, tok, pos);
      if (ev.lane == 0) sh->pos[row] = pos;
      const WT* e = reinterpret_cast<const WT*>(p.embed) + (size_t)tok * p.d;
      const float* gain = p.gains + (size_t)(draft ? p.first_gain_d : p.first_gain_t) * p.d;
      float* h = cl_at<float>(p.lay.h) + row * p.d;
      float* y = cl_at<float>(p.lay.y) + row * p.d;
      float* own = cl_at<float>(ev.hres) + row * p.lay.resid_np;
      const int q0 = sh->mine[CL_O].p0, q1 = q0 + sh->mine[CL_O].np;
      constexpr int hp = HD / 2;
      const int at = max(pos, 0) * hp;
      float cs[hp / 32], sn[hp / 32];
#pragma unroll
      for (int i = 0; i < hp / 32; ++i) {
        cs[i] = __ldg(p.rope_cos + at + i * 32 + ev.lane);
        sn[i] = __ldg(p.rope_sin + at + i * 32 + ev.lane);
      }
#pragma unroll 2
      for (int c = ev.lane * 4; c < p.d; c += 128) {
        const float4 v = pos >= 0 ? load4(e + c) : make_float4(0.f, 0.f, 0.f, 0.f);
        const float4 g = __ldg(reinterpret_cast<const float4*>(gain + c));
        *reinterpret_cast<float4*>(h + c) = v;
        *reinterpret_cast<float4*>(y + c) = make_float4(v.x * g.x, v.y * g.y, v.z * g.z, v.w * g.w);
        const int pair = (c >> 4) * 8 + (c & 7);  // of the first of these four features
        if (pair >= q0 && pair < q1) *reinterpret_cast<float4*>(own + ((c >> 3) & 1) * p.lay.rows * p.lay.resid_np + pair - q0) = v;
      }
      float* rope = cl_at<float>(p.lay.rope) + row * 2 * hp;
#pragma unroll
      for (int i = 0; i < hp / 32; ++i) {
        rope[i * 32 + ev.lane] = cs[i];
        rope[hp + i * 32 + ev.lane] = sn[i];
      }
      if (loop)
#pragma unroll
        for (int c = ev.lane; c < 4 * kClWarps; c += 32) cl_at<float2>(p.lay.best)[row * 4 * kClWarps + c] = make_float2(-INFINITY, __int_as_float(0x7fffffff));
    }
    cl_sync();

#pragma unroll 1
    for (int s = 0; s < n_stages; ++s) {
      const ClTab t = tab[s];
      ClDots a{};
      a.W = t.W;
      a.np = t.np;
      a.R = R;
      a.steps = t.steps;
      a.stg = ev.stg;
      a.x = t.x;
      a.K = t.K;
      a.bar = s > 0 ? t.bar : -1;  // the first stage's are the embedding
      a.bytes = (unsigned)(R * t.row_bytes);
      a.parity = (phases >> t.bar) & 1u;
      if (s > 0) phases ^= 1u << t.bar;
      a.norm = t.norm != 0;
      a.head = t.kind == CL_HEAD;
      a.p0 = t.p0;
      a.logits = loop ? nullptr : p.logits;
      if (p.lay.splits > 1 && t.kind == CL_O) {
        cl_wait(sh, p.sync, CL_BAR_X, a.bytes, a.parity);
        cl_fold_splits<HD>(p, ev);
        cl_sync();
        a.bar = -1;
      }
      // the pass's keys and values, before anything of the next pass is sent: their writers, long done, in a stage whose last warps have the least to do
      if (t.after_kv && tid >= kClThreads - ((R * sh->mine[CL_QKV].nq + 31) & ~31)) __threadfence();
      if (R == 1)
        cl_dots<WT, 1, 4>(p, a, sh);
      else if (R <= 4)
        cl_dots<WT, 4, 2>(p, a, sh);
      else
        cl_dots<WT, 8, 2>(p, a, sh);
      if (a.head) break;
      cl_sync();  // the sums are there
      const bool live = !cl_aborted(sh);
      if (t.kind == CL_QKV) {
        cl_finish_qkv<WT, HD>(p, ev, t, live);
        if (my_heads > 0) {
          other_stg();
          cl_attention<WT, HD>(p, ev, t, my_heads, phase(CL_BAR_QKV));
        }
      } else if (live) {
        if (t.kind == CL_GATE_UP)
          cl_finish_gate_up(p, ev);
        else
          cl_finish_resid(p, ev, t);
      }
      other_stg();
    }
    if (!loop) break;

    // ---- greedy decision: best of the CTA, then of the cluster ----
    cl_sync();
    if (!cl_aborted(sh))
#pragma unroll 1
      for (int row = ev.warp; row < R; row += kClWarps) {
        float bv = -INFINITY;
        int bi = 0x7fffffff;
#pragma unroll
        for (int e = ev.lane; e < 4 * kClWarps; e += 32) {
          const float2 c = cl_at<float2>(p.lay.best)[row * 4 * kClWarps + e];
          if (c.x > bv || (c.x == bv && __float_as_int(c.y) < bi)) {
            bv = c.x;
            bi = __float_as_int(c.y);
          }
        }
        cl_best_of_lanes<32>(bv, bi);
        if (ev.lane < kClCtas) cl_send2(ev.dst + p.lay.tok + (rank * R + row) * 8, bv, __int_as_float(bi), cl_bar_of(p, ev.dst, CL_BAR_TOK));
      }
    cl_wait(sh, p.sync, CL_BAR_TOK, (unsigned)(kClCtas * R * 8), phase(CL_BAR_TOK));
#pragma unroll 1
    for (int row = ev.warp; row < R; row += kClWarps) {
      const float2 c = cl_at<float2>(p.lay.tok)[(ev.lane & (kClCtas - 1)) * R + row];
      float bv = c.x;
      int bi = __float_as_int(c.y);
      cl_best_of_lanes<kClCtas>(bv, bi);
      if (ev.lane == 0) sh->amax[row] = min(max(bi, 0), p.vocab - 1);
    }
    cl_sync();
    if (tid < 32) {
      if (verify)
        cl_commit(p, sh, batch, k, rank == 0, tid);
      else if (tid < batch)
        sh->drafts[tid][pass] = sh->amax[tid * ev.rps + ev.rps - 1];
    }
    if (!cl_agree_ok(&sh->abort) || (verify && (sh->all_done || sh->round >= p.rounds))) break;
  }
  cl_sync();
  if (loop && rank == 0) {
    if (tid < batch) {
      p.gs->n[tid] = sh->n[tid];
      p.gs->n_new[tid] = sh->n_new[tid];
      p.gs->done[tid] = sh->done[tid];
    }
    if (tid == 0) {
      p.gs->round = sh->round;
      p.gs->all_done = sh->all_done;
      p.gs->pass_error = *reinterpret_cast<volatile int*>(&p.sync->error);
    }
  }
}

template <typename WT, int HD>
__global__ void __launch_bounds__(kClThreads, 1) cluster_pass_kernel(const __grid_constant__ ClParams p) {
  ClShared* sh = cl_at<ClShared>(p.lay.shared);
  ClTab* tab_t = cl_at<ClTab>(p.lay.tab);
  ClTab* tab_d = tab_t + p.n_t;
  const int tid = threadIdx.x, rank = (int)cl_rank();
  const bool loop = p.rounds > 0;
  const int batch = loop ? p.gs->batch : p.pd.n_seq, k = loop ? p.gs->k : 0;
  constexpr int n_threads = kClThreads;

  // ---- set-up: this CTA's shares, stage tables, the gains of its features, state ----
#pragma unroll 1
  for (int i = tid; i < p.n_t + p.n_d; i += n_threads) {
    const ClStage s = i < p.n_t ? p.prog_t[i] : p.prog_d[i - p.n_t];
    const int p0 = cl_first_pair(s.n_pairs, rank);
    ClTab& t = tab_t[i];
    t.kind = s.kind;
    t.np = cl_first_pair(s.n_pairs, rank + 1) - p0;
    t.steps = cl_steps(s.K, (int)sizeof(WT));
    t.gain_out = s.gain_out;
    t.p0 = p0;
    t.norm = s.kind == CL_QKV || s.kind == CL_GATE_UP || s.kind == CL_HEAD;
    t.x = s.kind == CL_O ? p.lay.xo : s.kind == CL_DOWN ? p.lay.u : p.lay.y;
    t.K = s.K;
    t.bar = s.kind == CL_O ? CL_BAR_X : s.kind == CL_DOWN ? CL_BAR_U : CL_BAR_H;
    t.row_bytes = s.kind == CL_O ? p.lay.splits * (p.d * 4 + (p.lay.splits > 1 ? p.heads * 8 : 0)) : s.kind == CL_DOWN ? p.f * 4 : 2 * p.d * 4;
    t.after_kv = s.after_kv;
    t.kcache = s.kcache;
    t.vcache = s.vcache;
    t.W = s.W + (size_t)p0 * t.steps * kClUnit;
  }
  if (tid >= 96 && tid < 101) {
    const int kind = tid - 96;
    const int n_pairs = kind == CL_QKV ? 3 * p.d / 2 : kind == CL_GATE_UP ? p.f : kind == CL_HEAD ? p.vocab / 2 : p.d / 2;
    ClMine& m = sh->mine[kind];
    m.p0 = cl_first_pair(n_pairs, rank);
    m.np = cl_first_pair(n_pairs, rank + 1) - m.p0;
    m.nq = m.np / 4;
    m.magic = m.nq > 0 ? (1u << 20) / m.nq + 1u : 0u;
  }
  {
    const int p0 = cl_first_pair(p.d / 2, rank), np = cl_first_pair(p.d / 2, rank + 1) - p0, ld = 2 * p.lay.resid_np;
#pragma unroll 1
    for (int i = tid; i < p.n_gains * 2 * np; i += n_threads) {
      const int g = i / (2 * np), r = i - g * 2 * np, half = r >= np ? 1 : 0, pl = r - half * np, pair = p0 + pl;
      cl_at<float>(p.lay.gain)[g * ld + half * p.lay.resid_np + pl] = __ldg(p.gains + (size_t)g * p.d + ((pair >> 3) << 4) + (pair & 7) + half * 8);
    }
  }
  if (tid < CL_BARS) mbar_init(&sh->bar[tid], 1);
  if (tid == 32) {
    // an earlier launch gave up a wait and the host has not cleared it yet: this one does nothing
    sh->abort = *reinterpret_cast<volatile int*>(&p.sync->error) != 0 ? 1 : 0;
    sh->sabotage = ld_relaxed(&p.sync->bar_extra) != 0 ? 16u : 0u;
    const unsigned long long set = ld_relaxed(&p.sync->wait_limit_ns);
    sh->wait_limit_ns = set ? set : kWaitLimitNs;
    sh->all_done = 0;
    sh->round = 0;
    if (loop) {
      sh->max_new = p.gs->max_new;
      sh->eos_id = p.gs->eos_id;
      sh->max_rounds = p.gs->max_rounds;
    }
  }
  if (tid >= 64 && tid < 64 + batch) {
    const int b = tid - 64;
    const int n = ld_act(&p.gs->n[b]);
    sh->n[b] = n;
    sh->n_new[b] = ld_act(&p.gs->n_new[b]);
    sh->done[b] = ld_act(&p.gs->done[b]);
    sh->last[b][0] = n >= 2 ? ld_act(p.seq_tok + (size_t)b * p.max_seq + n - 2) : 0;
    sh->last[b][1] = ld_act(p.seq_tok + (size_t)b * p.max_seq + n - 1);
#pragma unroll 1
    for (int s = 0; s < kMaxK; ++s) sh->drafts[b][s] = loop ? 0 : ld_act(p.draft_tok + b * kMaxK + s);
  }
  asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  cl_cluster_sync();  // barriers exist everywhere before anything is sent, and the CTA's tables are written

  cl_compute<WT, HD>(p, sh, tab_t, tab_d, rank, loop, batch, k);

  // In normal operation everything that was sent has been waited for.  After a wait that ran out something may still
  // be on its way to a CTA of the cluster: give it far longer than it takes before any CTA leaves.
  if (cl_aborted(sh)) {
    const unsigned long long t0 = global_ns();
#pragma unroll 1
    while (global_ns() - t0 < 200000ull) __nanosleep(1000);
  }
  __syncwarp();
  cl_cluster_sync();
}

// ---- packing: [pair][K step][half][512 bytes] -------------------------------------------------------------------
// A lane's sixteen bytes of a step: fp32 columns 4 lane .. +3; bf16 columns 4 lane .. +3 and 128 + 4 lane .. +3, so that
// the matching activations are two conflict-free 128-bit reads.  Columns beyond K are zero.
template <typename WT>
__global__ void pack_cluster_kernel(WT* __restrict__ dst, PackSrc ps, int n_pairs, int K) {
  constexpr int V = ClElem<WT>::kLane, STEP = ClElem<WT>::kStep;
  const int steps = cl_steps(K, (int)sizeof(WT));
  const size_t total = (size_t)n_pairs * 2 * steps * STEP;
  for (size_t e = (size_t)blockIdx.x * blockDim.x + threadIdx.x; e < total; e += (size_t)gridDim.x * blockDim.x) {
    const int in = (int)(e % STEP);
    const size_t rest = e / STEP;  // [pair][step][half]
    const int r = (int)(rest & 1), s = (int)((rest >> 1) % steps), pair = (int)((rest >> 1) / steps);
    const int lane = in / V, j = in % V;
    const int c = s * STEP + (j >> 2) * 128 + lane * 4 + (j & 3);
    dst[e] = c < K ? pack_src_row<WT>(ps, pair, r, K)[c] : WT(0.0f);
  }
}

// ---- host -------------------------------------------------------------------------------------------------------
// The layout for passes of up to `rows` rows; total = 0 when it does not fit
inline ClLayout cluster_layout(int d, int f, int heads, int hd, int n_layers, int rows, int max_seq, int max_smem) {
  ClLayout y{};
  y.rows = rows;
  const int key_block = 32 / (hd / 16);
  y.heads_per_cta = (heads + kClCtas - 1) / kClCtas;
  // CTAs per head: as many as the longest context gives a block to every warp of, one when one does
  y.splits = heads >= kClCtas ? 1 : std::max(1, std::min(kClCtas / heads, std::min(4, (max_seq + kClWarps * key_block - 1) / (kClWarps * key_block))));
  y.resid_np = cl_max_pairs(d / 2);
  int at = 0;
  auto take = [&](int& off, long long bytes) {
    off = at;
    at = (int)std::min<long long>(1 << 30, ((long long)at + bytes + 127) / 128 * 128);
  };
  take(y.h, 4LL * rows * d);
  take(y.y, 4LL * rows * d);
  // u lies over the attention's partial sums and output: it is written when every CTA has taken the O-projection's input
  // in, and read before any CTA sends attention output of the next layer
  const int u0 = at;
  take(y.part, 4LL * rows * y.heads_per_cta * kClWarps * (hd + 4));
  take(y.xp, y.splits > 1 ? 4LL * y.splits * rows * d : 0);
  take(y.xml, y.splits > 1 ? 8LL * y.splits * rows * heads : 0);
  take(y.xo, 4LL * rows * d);
  const int att_end = at;
  at = u0;
  take(y.u, 4LL * rows * f);
  at = std::max(at, att_end);
  take(y.qkv, 12LL * rows * y.heads_per_cta * hd);
  take(y.gain, 8LL * (2 * n_layers + 1) * y.resid_np);
  take(y.hres, 16LL * rows * y.resid_np);
  const int share = std::max(2 * std::max(cl_max_pairs(3 * d / 2), cl_max_pairs(f)), y.heads_per_cta * (hd + 4));  // values of a row
  y.stg_floats = rows * share;
  take(y.stg, 8LL * y.stg_floats);
  take(y.rope, 4LL * rows * hd);
  take(y.tok, 8LL * kClCtas * rows);
  take(y.best, 32LL * rows * kClWarps);
  take(y.tab, (long long)sizeof(ClTab) * 2 * (4 * n_layers + 1));
  take(y.shared, (long long)sizeof(ClShared));
  y.total = at <= max_smem ? at : 0;
  return y;
}

}  // namespace sdfp
