// Rounds of small decoders inside ONE thread-block cluster of sixteen CTAs: the whole greedy generation loop (Algorithm 1,
// Stage B: k draft passes, verification, accept, commit) in one launch, or one pass of a sampled round.
//
// What bounds a small decoder is not its bytes but the chain of dependent stages, five a layer: spread over 148
// SMs a stage boundary is a grid-wide exchange through L2 (about 5 us in the whole-pass kernel, about 4 us as one
// launch per operation), for a fraction of a microsecond of work.  Sixteen SMs of one cluster hand their results on
// through distributed shared memory instead:
//   * Every linear stage gives each CTA an equal share of the output features.  The finished values are gathered in shared
//     memory; a half-warp takes four columns at a time, a lane sends them to each of the sixteen CTAs with st.async, and
//     the bytes complete a transaction count on an mbarrier of the receiver, which starts its next stage when all
//     shares have landed.  No barrier over the cluster stands between stages, and nothing goes through L2 but
//     weights and the K/V cache.
//   * The buffers need no second copy: a CTA writes into another's buffer only when it holds the complete output of a stage
//     that the other contributed to after its last read of that buffer.  Every CTA has a share of every stage of a layer.
//   * Weights are read where the context's other kernels read them; the first ones are on their way before the wait for
//     the activations.
//   * K/V: the rows of the running pass are taken from shared memory, older keys from the cache in global memory.  The
//     CTA that reads a key in later passes is the one that appends it, so no pass waits for another CTA's cache entries.
//   * Loops are left rolled: every instruction of a pass is met once per layer.  As straight code for every shape the kernel was
//     500 KB and a pass of one row took half as long again.
// What bounds it now is dependent instructions, 18 400 a warp and pass at 4 layers d 256 bf16, six clocks each with two warps on
// a scheduler.  In us a pass of one row, 4 layers, FFN 2.7 d, vocabulary 4096, this kernel and the other path: bf16 (whole-pass
// kernel) d 256 61 and 135, d 384 74 and 135, d 512 90 and 147; fp32 (one kernel per operation) 55 and 110, 73 and 115, 119 and 123.
// The line between them is at cluster_cost in engine.cu.
//
// The results are, bit for bit, those of the path the context's other passes take (prompts, sdfp_forward_logits): the
// whole-pass kernel for bf16, one kernel per operation for fp32.  A text goes on the same whether it was decoded in one
// call or in several, and the logits a caller asks for are those that chose the tokens.  So the order of every sum is theirs:
//   * bf16: the tiles and units of pass_kernel.cuh on mma.sync, hi + lo; a warp is a k-class, and a sum is made of the classes of a
//     piece in order, then of the pieces in the order in which the whole-pass kernel's CTAs post them (StageShare).
//     Which units a warp multiplies is written down once, on the host (ClEntry).
//   * fp32: a warp owns output pairs and walks K with its lanes, as linear_fma_kernel does, on rows normalised before.
//   * Attention in chunks of 64 keys: bf16 eight splits of the chunks with a running maximum each, added in split order
//     (pass_kernel.cuh); fp32 every chunk by itself, added in chunk order (attention.cuh).
//   * Squares of the residual rows: per 128 features, then over the groups (bf16); lanes over the row (fp32).
#pragma once

#include <vector>

#include "attention.cuh"
#include "common.cuh"
#include "linear_fma.cuh"
#include "misc_kernels.cuh"
#include "pass_kernel.cuh"

namespace sdfp {

constexpr int kClCtas = 16, kClWarps = 8, kClThreads = kClWarps * 32;
static_assert(kClWarps == kClasses, "a warp is a k-class of the whole-pass kernel");
constexpr int kClMaxRows = 16;
constexpr int kClTeam = 128;     // threads that work on an attention item
constexpr int kClAttnRows = 8;   // rows of a sequence it takes together
constexpr int kClTiles = 4;      // bf16: tiles a warp multiplies together
constexpr int kClRing = 16;      // bf16: units of weights (512 bytes) a warp has on their way

enum ClBar { CL_BAR_H = 0, CL_BAR_U = 1, CL_BAR_QKV = 2, CL_BAR_PART = 3, CL_BAR_X = 4, CL_BAR_TOK = 5, CL_BARS = 6 };
enum ClKind { CL_QKV = 0, CL_O = 1, CL_GATE_UP = 2, CL_DOWN = 3, CL_HEAD = 4, CL_KINDS = 5 };

// Shares of the output features: pairs are dealt in fours, so that a share is sent sixteen bytes at a time, and in eights, the
// row tile of the MMA, where every CTA gets one (a tile cut between two CTAs is multiplied by both).
__host__ __device__ __forceinline__ int cl_deal(int n_pairs, int elem_bytes) { return elem_bytes == 2 && n_pairs >= 8 * kClCtas ? 8 : 4; }
__host__ __device__ __forceinline__ int cl_first_pair(int n_pairs, int cta, int elem_bytes) {
  const int deal = cl_deal(n_pairs, elem_bytes);
  return (int)((long long)(n_pairs / deal) * cta / kClCtas) * deal;
}
__host__ __device__ __forceinline__ int cl_max_pairs(int n_pairs, int elem_bytes) {
  const int deal = cl_deal(n_pairs, elem_bytes);
  return (n_pairs / deal + kClCtas - 1) / kClCtas * deal;
}
__host__ __device__ __forceinline__ int cl_pairs_of(int kind, int d, int f, int vocab) {
  return kind == CL_QKV ? 3 * d / 2 : kind == CL_GATE_UP ? f : kind == CL_HEAD ? vocab / 2 : d / 2;
}

// What a CTA does of the matrices of one kind: the same in every layer, made on the host
struct ClMine {
  int p0, np;             // its pairs
  int tile_width;         // bf16: tiles multiplied together, 1, 2 or 4
  int round0, n_rounds;   // its sums fit the staging buffer in one or more rounds
  int entry0, n_entries;  // bf16: list of warp w = entries entry0 + w * n_entries ...
  int pad;
};
struct ClRound {
  int quad0, n_quads;  // fours of pairs that are finished in this round
  unsigned magic;      // i / n_quads == i * magic >> 20 for the few hundred vectors of a round
  int tile0, np;       // bf16: its first tile, and the pieces a sum is made of
  int pad[3];
};
struct ClEntry {       // bf16: one k-tile of a warp, for up to kClTiles neighbouring tiles
  int w;               // the first tile's unit, in uint4 from the matrix's start
  short kt, slot;      // k-tile, -1: none; slot >= 0: the sums are complete and go to this place, a tile's np places apart
  unsigned char n_tiles, wrap, np, last;  // from tile `wrap` on they lie in the next group; last: of the round, 2: of all
  int pad2;
};
static_assert(sizeof(ClMine) == 32 && sizeof(ClRound) == 32 && sizeof(ClEntry) == 16, "copied in sixteen bytes");

struct ClStage {  // a linear stage of a program; the attention follows a QKV stage without an entry of its own
  const unsigned char* W;
  void *kcache, *vcache;  // CL_QKV
  int kind, K;
  int gain;               // fp32: the norm in front of this stage (-1: none); bf16, CL_O and CL_DOWN: the norm that reads the residual stream next
  int pad;
};

struct ClTab {  // the same for this CTA, in shared memory
  const unsigned char* W;  // bf16: the matrix, fp32: its first pair
  void *kcache, *vcache;
  const float* gain;       // fp32: of the norm in front
  int kind, K, gain_out;
  int x, bar, row_bytes;   // its activations: where, the barrier that brings them and their bytes per row
  int norm;
};

// Shared-memory layout, worked out on the host (bytes from the start)
struct ClLayout {
  int rows, splits, heads_per_cta, resid_np, part_slots;
  int h, y, part, team, team_bytes, xo, u, qkv, gain, hres, stg, red, ring, rope, tok, best, tab, plan, plan_rounds, plan_entries, plan_bytes, shared, total;
};

struct ClParams {
  const ClStage* prog_t;
  const ClStage* prog_d;
  int n_t, n_d;              // stages to run of either
  int first_gain_t, first_gain_d;
  const float* const* gains;  // [n_gains] -> [d]
  int n_gains;
  int d, f, heads, vocab, max_seq;
  float eps, scale;
  const float *rope_cos, *rope_sin;
  const void* embed;
  const unsigned char* plan;  // [CTA][plan_bytes]
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

struct ClShared {
  uint64_t bar[CL_BARS];
  int abort;
  unsigned long long wait_limit_ns;
  unsigned sabotage;  // bytes the next wait expects in vain (PassSync::bar_extra)
  float inv[kClMaxRows];
  int pos[kClMaxRows];
  int amax[kClMaxRows];
  float att_m[2][kClAttnRows], att_l[2][kClAttnRows], att_a[2][kClAttnRows];  // attention rows of a team
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
__device__ __forceinline__ void cl_send1(uint32_t dst, float v, uint32_t bar) {
  asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.b32 [%0], %1, [%2];" ::"r"(dst), "r"(__float_as_uint(v)), "r"(bar) : "memory");
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
// a barrier of the CTA that gives everybody the same answer to "has anything failed"
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
        atomicCAS(&sync->error, 0, (int)PASS_ERR_CLUSTER);
        *reinterpret_cast<volatile int*>(&sh->abort) = 1;
        break;
      }
    }
  }
}
// Wait for a buffer the other CTAs fill.  Their bytes may have been counted before the barrier is told how many to expect.
__device__ __forceinline__ void cl_wait(ClShared* sh, PassSync* sync, int which, unsigned bytes, unsigned parity) {
  if (__any_sync(0xffffffffu, cl_aborted(sh))) return;  // a phase that never ended must not be armed again; one answer for the warp
  if (threadIdx.x == kClThreads - 1) {
    mbar_arrive_expect_tx(&sh->bar[which], bytes + sh->sabotage);
    sh->sabotage = 0;
  }
  const uint32_t bar = smem_u32(&sh->bar[which]);
  if (!cl_try_wait(bar, parity)) cl_poll(sh, sync, bar, parity);
  __syncwarp();
}

// The same value in all lanes, and known to be: in a loop that could run a different number of times in the lanes of a warp, every
// shuffle first gathers the warp with a routine of a hundred clocks and more (a row's softmax took 2600 clocks instead of 600).
__device__ __forceinline__ int cl_uniform(int v) { return __shfl_sync(0xffffffffu, v, 0); }

// the better of two (value, index), ties to the lower index
__device__ __forceinline__ void cl_better(float& bv, int& bi, float v, int i) {
  if (v > bv || (v == bv && i < bi)) {
    bv = v;
    bi = i;
  }
}
template <int n>
__device__ __forceinline__ void cl_best_of_lanes(float& bv, int& bi) {  // over n neighbouring lanes
#pragma unroll
  for (int o = n / 2; o > 0; o >>= 1) cl_better(bv, bi, __shfl_xor_sync(0xffffffffu, bv, o), __shfl_xor_sync(0xffffffffu, bi, o));
}

__device__ __forceinline__ int cl_feature(int pair) { return ((pair >> 3) << 4) + (pair & 7); }  // the first of a pair's features, its second is 8 further

// Activations between the stages, sixteen bytes per four columns.  fp32: [row][K].  bf16: [eight columns][row][two columns] of
// {hi, lo}, so that a lane of the MMA reads the two halves of its fragment of sixteen columns as two 64-bit words without conflicts.
template <typename WT>
__device__ __forceinline__ int cl_x_off(int K, int R, int row, int col) {  // bytes to columns col .. col + 3
  return sizeof(WT) == 2 ? (((col >> 3) * R + row) * 4 + ((col & 7) >> 1)) * 8 : (row * K + col) * 4;
}
template <typename WT>
__device__ __forceinline__ float4 cl_x_pack(const float4& x) {
  if (sizeof(WT) == 4) return x;
  uint32_t h0, h1, l0, l1;
  split_pack(x.x, x.y, h0, l0);
  split_pack(x.z, x.w, h1, l1);
  return make_float4(__uint_as_float(h0), __uint_as_float(l0), __uint_as_float(h1), __uint_as_float(l1));
}
// (rounded products: the whole-pass kernel splits values that exist as such)
__device__ __forceinline__ float4 cl_mul(const float4& a, const float4& b) {
  return make_float4(__fmul_rn(a.x, b.x), __fmul_rn(a.y, b.y), __fmul_rn(a.z, b.z), __fmul_rn(a.w, b.w));
}

struct ClEnv {
  ClShared* sh;
  const ClMine* mine;     // by ClKind
  const ClRound* rounds;
  const ClEntry* entries;
  int tid, warp, lane, rank;
  int R, rps;          // rows of the pass, rows per sequence; sequence b has cache slot b
  uint32_t self, dst;  // shared memory of this CTA (as an address of the cluster's), of CTA tid mod 16: what goes to all CTAs is sent by a thread each
};
__device__ __forceinline__ uint32_t cl_bar_of(const ClParams& p, uint32_t cta, int which) {
  return cta + p.lay.shared + (int)offsetof(ClShared, bar) + which * 8;
}

// ---- dot products of a stage ------------------------------------------------------------------------------------
struct ClDots {
  const unsigned char* W;
  int kind, K, x;            // activations: where they are
  int bar;                   // what brings them (ClBar), -1: nothing to wait for
  unsigned bytes, parity;
  bool norm;                 // the rows' norms are wanted
  const float* gain;         // fp32: of that norm
  float* logits;             // CL_HEAD: logits [row][vocab] or, without, the best of each (row, place)
};

// fp32: the rows' norms are applied here, for this CTA's own use; gains are asked for before the wait
struct ClGain {
  float4 g[2];
  __device__ __forceinline__ void load(const float* gain, int d, int lane) {
#pragma unroll
    for (int i = 0; i < 2; ++i) {
      g[i] = make_float4(0.f, 0.f, 0.f, 0.f);
      if (i * 128 + lane * 4 < d) g[i] = __ldg(reinterpret_cast<const float4*>(gain + i * 128 + lane * 4));
    }
  }
};
__device__ __forceinline__ void cl_norm_rows(const ClParams& p, const ClEnv& ev, const float* gain, const ClGain& cg) {
#pragma unroll 1
  for (int row = ev.warp; row < ev.R; row += kClWarps) {
    const float* h = cl_at<float>(p.lay.h) + row * p.d;
    float* y = cl_at<float>(p.lay.y) + row * p.d;
    float s = 0.f;
#pragma unroll 2
    for (int c = ev.lane * 4; c < p.d; c += 128) {
      const float4 v = *reinterpret_cast<const float4*>(h + c);
      s = fmaf(v.x, v.x, s);
      s = fmaf(v.y, v.y, s);
      s = fmaf(v.z, v.z, s);
      s = fmaf(v.w, v.w, s);
    }
    const float r = rsqrtf(warp_sum(s) / (float)p.d + p.eps);
#pragma unroll 2
    for (int i = 0; i * 128 + ev.lane * 4 < p.d; ++i) {
      const int c = i * 128 + ev.lane * 4;
      const float4 g = i == 0 ? cg.g[0] : i == 1 ? cg.g[1] : __ldg(reinterpret_cast<const float4*>(gain + c));
      float4 v = *reinterpret_cast<const float4*>(h + c);
      v.x = v.x * r * g.x;
      v.y = v.y * r * g.y;
      v.z = v.z * r * g.z;
      v.w = v.w * r * g.w;
      *reinterpret_cast<float4*>(y + c) = v;
    }
  }
  __syncthreads();
}

// bf16: 1 / rms of the rows, needed behind the dot products only.  Per 128 features the squares of a pair, of the pair 32
// further, the xor tree; then the groups.
__device__ __forceinline__ void cl_row_scales(const ClParams& p, const ClEnv& ev) {
  const int pairs = p.d / 2;
#pragma unroll 1
  for (int row = kClWarps - 1 - ev.warp; row < ev.R; row += kClWarps) {
    const float* sq = cl_at<float>(p.lay.h) + row * pairs;
    float part = 0.f;
#pragma unroll 2
    for (int g = 0; g < (pairs + 63) / 64; ++g) {
      const int i = g * 64 + ev.lane;
      const float v = warp_sum((i < pairs ? sq[i] : 0.f) + (i + 32 < pairs ? sq[i + 32] : 0.f));
      if (ev.lane == (g & 31)) part += v;
    }
    const float s = warp_sum(part);
    if (ev.lane == 0) ev.sh->inv[row] = rsqrtf(s / (float)p.d + p.eps);
  }
}

// fp32.  A warp's pairs lie behind one another in memory, [pair][half][K].  It takes P of them through RT rows at a time (more
// rows take another sweep of the weights, from L2); a K step of weights is in registers or on its way, the first before the
// wait for the activations.  A sum is made in the same order whatever P and RT: K steps in order by each lane, the lanes in the xor tree.
template <int RT, int P>
__device__ __forceinline__ void cl_dots_f32(const ClParams& p, const ClEnv& ev, const ClDots& a) {
  constexpr int N = RT * P * 2, CH = N < 16 ? N : 16;
  const int warp = ev.warp, lane = ev.lane, R = ev.R;
  const ClMine& me = ev.mine[a.kind];
  const int np = cl_uniform(me.np);
  const int n_w = RT == 1 ? (np + kClWarps - 1) / kClWarps : (np / 2 + kClWarps - 1) / kClWarps * 2;  // pairs per warp
  const int first = warp * n_w, cnt = max(0, min(n_w, np - first));
  const int half_len = a.K / 4;  // in uint4
#pragma unroll 1
  for (int r0 = 0; r0 < R; r0 += RT) {
    const int rows = RT == 1 ? 1 : min(RT, R - r0);
    const uint4* w = reinterpret_cast<const uint4*>(a.W) + (size_t)first * 2 * half_len + lane;
    int ask_pairs = cnt, ask_c = lane * 4;  // pairs from the next request's on, its column
    uint4 raw[P][2];
#pragma unroll
    for (int j = 0; j < P; ++j) raw[j][0] = raw[j][1] = make_uint4(0u, 0u, 0u, 0u);
    auto ask = [&]() {
      if (ask_pairs <= 0) return;
      const bool in = ask_c < a.K;
#pragma unroll
      for (int j = 0; j < P; ++j)
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          if (!in) raw[j][h] = make_uint4(0u, 0u, 0u, 0u);
          if (in && j < ask_pairs) raw[j][h] = __ldg(w + (2 * j + h) * half_len);
        }
      w += 32;
      ask_c += 128;
      if (ask_c - lane * 4 >= a.K) {
        w += 2 * P * half_len - (ask_c / 128) * 32;
        ask_c = lane * 4;
        ask_pairs -= P;
      }
    };
    ask();
    if (r0 == 0) {
      ClGain cg;
      if (a.norm) cg.load(a.gain, p.d, lane);
      if (a.bar >= 0) cl_wait(ev.sh, p.sync, a.bar, a.bytes, a.parity);
      if (a.norm) cl_norm_rows(p, ev, a.gain, cg);
    }
    const float* const x = cl_at<float>(a.x) + r0 * a.K + lane * 4;
    const int room = a.K - lane * 4;
#pragma unroll 1
    for (int at = 0; at < cnt; at += P) {  // first pair of the running P
      float acc[N];
#pragma unroll
      for (int i = 0; i < N; ++i) acc[i] = 0.f;
#pragma unroll 1
      for (int c0 = 0; c0 < a.K; c0 += 128) {
        const bool in = c0 < room;
#pragma unroll
        for (int i = 0; i < RT; ++i) {
          if (RT == 1 || i < rows) {
            float4 xv = make_float4(0.f, 0.f, 0.f, 0.f);
            if (in) xv = *reinterpret_cast<const float4*>(x + i * a.K + c0);
#pragma unroll
            for (int j = 0; j < P; ++j)
              if (RT > 1 || j < cnt - at) {
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                  float& t = acc[(i * P + j) * 2 + h];
                  t = fmaf(__uint_as_float(raw[j][h].x), xv.x, t);
                  t = fmaf(__uint_as_float(raw[j][h].y), xv.y, t);
                  t = fmaf(__uint_as_float(raw[j][h].z), xv.z, t);
                  t = fmaf(__uint_as_float(raw[j][h].w), xv.w, t);
                }
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
          const float v0 = warp_sum_scatter<CH>(v);
          const float v1 = __shfl_xor_sync(0xffffffffu, v0, 32 / CH);
          const int pi = (g + lane / (32 / CH)) >> 1, row = r0 + pi / P, pl = first + at + pi % P;
          if (lane % (64 / CH) == 0 && row < R && at + pi % P < cnt) {
            if (a.kind != CL_HEAD) {
              float* o = cl_at<float>(p.lay.stg) + row * np + pl;
              o[0] = v0;
              o[R * np] = v1;
            } else {
              const int f0 = cl_feature(me.p0 + pl);
              if (a.logits != nullptr) {
                float* o = a.logits + (size_t)row * p.vocab + f0;
                if (!cl_aborted(ev.sh)) o[0] = v0, o[8] = v1;
              } else {  // only this lane touches its place; a NaN loses against everything, by itself
                float2* best = cl_at<float2>(p.lay.best) + row * 4 * kClWarps + warp * 4 + pi % P;
                float2 o = *best;
                if (v0 > o.x || (v0 == o.x && f0 < __float_as_int(o.y))) o = make_float2(v0, __int_as_float(f0));
                if (v1 > o.x || (v1 == o.x && f0 + 8 < __float_as_int(o.y))) o = make_float2(v1, __int_as_float(f0 + 8));
                *best = o;
              }
            }
          }
        }
      }
    }
  }
}

// bf16: the weights of a stage on their way to a warp, through a ring in shared memory.  Every lane copies what it will use
// itself, so nothing but its own wait stands between the copy and the use.  An entry of the list is a group of copies; as many are
// on their way as entries of the stage's width fill the ring.
struct ClRing {
  const uint4* W;        // the matrix, this lane's part
  const ClEntry* next;   // of this warp's list; the last one repeats itself
  int4 v;                // *next
  uint32_t buf;          // the ring
  int at, wrap_jump;     // where in it the next entry goes
  __device__ __forceinline__ void begin(const ClEntry* first) {
    next = first;
    get();
    at = 0;
  }
  template <int TW>
  __device__ __forceinline__ void fill() {
#pragma unroll 1
    for (int i = 0; i < kClRing; i += TW) ask<TW>();
  }
  template <int TW>  // the stage's width: tiles of an entry, at most
  __device__ __forceinline__ void ask() {
    if ((short)v.y >= 0) {
      const uint4* w = W + v.x;
      const int n = v.z & 255, wrap = (v.z >> 8) & 255;
#pragma unroll
      for (int t = 0; t < TW; ++t)
        if (TW == 1 || t < n)
          asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(buf + at + t * 512), "l"(w + t * 32 + (t >= wrap ? wrap_jump : 0)) : "memory");
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
    at = (at + TW * 512) & (kClRing * 512 - 1);
    if ((v.z >> 24) > 1)
      v.y = -1;  // nothing any more
    else
      ++next, get();
  }
  __device__ __forceinline__ void get() {
    v = *reinterpret_cast<const int4*>(next);
    v.y = cl_uniform(v.y);
    v.z = cl_uniform(v.z);
  }
  template <int TW>
  __device__ __forceinline__ void wait() const {  // for the oldest entry
    asm volatile("cp.async.wait_group %0;" ::"n"(kClRing / TW - 1) : "memory");
  }
};

// The entries of a round.  CG: column groups of eight rows.  Complete sums are left as [place][class][row of the tile][two rows of
// the pass] of 128 bits, as a lane holds them: {half 0 of rows 2 q and 2 q + 1, half 1 of the same}.  What an entry needs besides its
// weights is read while the one in front of it is multiplied.
template <int TW, int CG>
__device__ __forceinline__ void cl_mma_round(const ClParams& p, const ClEnv& ev, int x_at, const ClEntry*& ent, ClRing& ring) {
  const int g = ev.lane >> 2, q = ev.lane & 3, R = ev.R, Q = (R + 1) / 2;
  const uint2* const x = cl_at<uint2>(x_at) + g * 4 + q;
  float4* const red = cl_at<float4>(p.lay.red) + (ev.warp * 8 + g) * Q + q;
  float acc[TW][CG][4];
#pragma unroll
  for (int i = 0; i < TW; ++i)
#pragma unroll
    for (int c = 0; c < CG; ++c) acc[i][c][0] = acc[i][c][1] = acc[i][c][2] = acc[i][c][3] = 0.f;
  uint2 b0[CG], b1[CG];
  auto load_x = [&](int kt) {
#pragma unroll
    for (int c = 0; c < CG; ++c) {
      b0[c] = b1[c] = make_uint2(0u, 0u);
      if (kt >= 0 && c * 8 + g < R) {
        b0[c] = x[kt * 8 * R + c * 32];
        b1[c] = x[kt * 8 * R + c * 32 + 4 * R];
      }
    }
  };
  int4 v = *reinterpret_cast<const int4*>(ent);
  v.y = cl_uniform(v.y);
  v.z = cl_uniform(v.z);
  load_x((short)v.y);
  for (;;) {
    const int n = v.z & 255, slot = v.y >> 16, last = v.z >> 24;
    int4 vn = *reinterpret_cast<const int4*>(ent + (last ? 0 : 1));
    vn.y = cl_uniform(vn.y);
    vn.z = cl_uniform(vn.z);
    if ((short)v.y >= 0) {
      ring.wait<TW>();
      uint4 w[TW];
#pragma unroll
      for (int t = 0; t < TW; ++t)
        if (TW == 1 || t < n)
          asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];"
                       : "=r"(w[t].x), "=r"(w[t].y), "=r"(w[t].z), "=r"(w[t].w)
                       : "r"(ring.buf + ring.at + t * 512)
                       : "memory");
#pragma unroll
      for (int t = 0; t < TW; ++t)
        if (TW == 1 || t < n)
#pragma unroll
          for (int c = 0; c < CG; ++c) {
            mma_bf16_16816(acc[t][c], w[t], b0[c].x, b1[c].x);
            mma_bf16_16816(acc[t][c], w[t], b0[c].y, b1[c].y);
          }
    }
    ring.ask<TW>();  // into the place just read
    if (!last) load_x((short)vn.y);
    if (slot >= 0) {
      float4* o = red + slot * kClasses * 8 * Q;
      const int step = ((v.z >> 16) & 255) * kClasses * 8 * Q;
#pragma unroll
      for (int t = 0; t < TW; ++t)
#pragma unroll
        for (int c = 0; c < CG; ++c) {
          if ((TW == 1 || t < n) && c * 4 + q < Q) o[t * step + c * 4] = make_float4(acc[t][c][0], acc[t][c][1], acc[t][c][2], acc[t][c][3]);
          acc[t][c][0] = acc[t][c][1] = acc[t][c][2] = acc[t][c][3] = 0.f;
        }
    }
    ++ent;
    if (last) break;
    v = vn;
  }
}

// bf16: both halves of a pair, each the classes of a piece in order, then the pieces
__device__ __forceinline__ float2 cl_sum_pair(const ClParams& p, const ClRound& rd, int R, int row, int pair) {
  const int Q = (R + 1) / 2, step = kClasses * 32 * Q;  // words of a place
  const float* s = cl_at<float>(p.lay.red) + ((pair >> 3) - rd.tile0) * rd.np * step + ((pair & 7) * Q + (row >> 1)) * 4 + (row & 1);
  float2 v = make_float2(0.f, 0.f);
#pragma unroll 1
  for (int i = 0; i < rd.np; ++i, s += step) {
    float2 t = make_float2(0.f, 0.f);
#pragma unroll
    for (int c = 0; c < kClasses; ++c) {
      t.x += s[c * 32 * Q];
      t.y += s[c * 32 * Q + 2];
    }
    v = i == 0 ? t : make_float2(v.x + t.x, v.y + t.y);
  }
  return v;
}

// bf16 lm-head, one round: logits, or a thread's best of its row's pairs (a thread keeps to one row)
__device__ __forceinline__ void cl_head_round(const ClParams& p, const ClEnv& ev, const ClMine& me, const ClRound& rd, float* logits, int row_log, float& bv, int& bi) {
  const int row = ev.tid >> row_log;
  if (row >= ev.R || cl_aborted(ev.sh)) return;  // (what is read from the logits behind a failed wait are those of an earlier pass)
  const float inv = ev.sh->inv[row];
#pragma unroll 1
  for (int j = ev.tid & ((1 << row_log) - 1); j < 4 * rd.n_quads; j += 1 << row_log) {
    const int pair = me.p0 + 4 * rd.quad0 + j, f0 = cl_feature(pair);
    const float2 s = cl_sum_pair(p, rd, ev.R, row, pair);
    const float v0 = s.x * inv, v1 = s.y * inv;
    if (logits != nullptr) {
      float* o = logits + (size_t)row * p.vocab + f0;
      o[0] = v0;
      o[8] = v1;
    } else {  // the whole-pass kernel compares a pair's halves first: a NaN in front hides the other
      const float v = v1 > v0 ? v1 : v0;
      const int fi = v1 > v0 ? f0 + 8 : f0;
      if (v > bv || (v == bv && fi < bi)) {
        bv = v;
        bi = fi;
      }
    }
  }
}

// ---- epilogues: the values of a round, a thread per (row, pair), then behind a barrier their sending -------------------------
template <typename WT, int HD>
__device__ __forceinline__ void cl_values(const ClParams& p, const ClEnv& ev, const ClMine& me, const ClRound& rd, int kind) {
  constexpr bool BF = sizeof(WT) == 2;
  constexpr int hp = HD / 2;
#pragma unroll 1
  for (int i = ev.tid; i < 4 * ev.R * rd.n_quads; i += kClThreads) {
    const int v = i >> 2, row = (int)((unsigned)v * rd.magic >> 20), pl = 4 * (rd.quad0 + v - row * rd.n_quads) + (i & 3), pair = me.p0 + pl;
    float* o = cl_at<float>(p.lay.stg) + row * me.np + pl;
    float2 s = BF ? cl_sum_pair(p, rd, ev.R, row, pair) : make_float2(o[0], o[ev.R * me.np]);
    if (BF && (kind == CL_QKV || kind == CL_GATE_UP)) {
      const float inv = ev.sh->inv[row];
      s.x *= inv;
      s.y *= inv;
    }
    if (kind == CL_QKV) {  // rotary embedding of q and k
      if (pair < p.d) {
        const float* rp = cl_at<float>(p.lay.rope) + row * 2 * hp + pair % hp;
        const float c = rp[0], n = rp[hp];
        const float r = s.x * c - s.y * n;
        s.y = s.y * c + s.x * n;
        s.x = r;
      }
    } else if (kind == CL_GATE_UP) {
      s.x = __fmul_rn(s.x / (1.0f + __expf(-s.x)), s.y);
    } else {  // new residual rows
      float* own = cl_at<float>(p.lay.hres) + row * p.lay.resid_np + pl;
      const int half_len = p.lay.rows * p.lay.resid_np;
      s.x = own[0] + s.x;
      s.y = own[half_len] + s.y;
      own[0] = s.x;
      own[half_len] = s.y;
    }
    o[0] = s.x;
    o[ev.R * me.np] = s.y;
  }
}

// Quarters of a q row lie eight words further apart than they are long: threads that share a key read them without conflicts.
template <int HD>
struct ClQ {
  static constexpr int kLd = HD + 32;  // floats of a row
  static __device__ __forceinline__ int at(int d) { return d / (HD / 4) * (HD / 4 + 8) + d % (HD / 4); }
};

// q, k, v to the CTAs that work on the head, a thread per four columns
template <typename WT, int HD>
__device__ __forceinline__ void cl_send_qkv(const ClParams& p, const ClEnv& ev, const ClMine& me, const ClRound& rd) {
  constexpr int hp = HD / 2;
  const int per = p.d >> 1, rows_all = p.lay.heads_per_cta * ev.R, total = ev.R * rd.n_quads;
#pragma unroll 1
  for (int i = ev.tid; i < 2 * total; i += kClThreads) {
    const int half = i >= total ? 1 : 0, v = i - half * total;
    const int row = (int)((unsigned)v * rd.magic >> 20), quad = rd.quad0 + v - row * rd.n_quads, pair = me.p0 + 4 * quad;
    const int which = pair >= 2 * per ? 2 : pair >= per ? 1 : 0, rem = pair - which * per, head = rem / hp, d0 = rem % hp + half * hp;
    const float4 x = cl_at<float4>(p.lay.stg)[(half * ev.R + row) * (me.np / 4) + quad];
    const int hr = (p.heads >= kClCtas ? head / kClCtas : 0) * ev.R + row;
    const int to = which == 0 ? p.lay.qkv + (hr * ClQ<HD>::kLd + ClQ<HD>::at(d0)) * 4
                              : p.lay.qkv + rows_all * ClQ<HD>::kLd * 4 + (((which - 1) * rows_all + hr) * HD + d0) * (int)sizeof(WT);
    const __nv_bfloat162 x0 = __floats2bfloat162_rn(x.x, x.y), x1 = __floats2bfloat162_rn(x.z, x.w);  // as the cache will hold them
#pragma unroll 1
    for (int s = 0, cta = p.heads >= kClCtas ? head % kClCtas : head; s < p.lay.splits; ++s, cta += p.heads) {
      const uint32_t dst = cl_map(ev.self, cta), bar = cl_bar_of(p, dst, CL_BAR_QKV);
      if (which == 0 || sizeof(WT) == 4)
        cl_send4(dst + to, x, bar);
      else
        cl_send2(dst + to, __uint_as_float(*reinterpret_cast<const uint32_t*>(&x0)), __uint_as_float(*reinterpret_cast<const uint32_t*>(&x1)), bar);
    }
  }
}

// What goes to all CTAs: a half-warp per four columns, a lane per CTA.  SwiGLU: u.  Residual rows: fp32 as they are; bf16 times the
// next norm's gain, and the squares of the pairs.
template <typename WT>
__device__ __forceinline__ void cl_send_all(const ClParams& p, const ClEnv& ev, const ClMine& me, const ClRound& rd, int kind, int gain_out) {
  const float* gain = cl_at<float>(p.lay.gain) + gain_out * 2 * p.lay.resid_np;
  const uint32_t bar = cl_bar_of(p, ev.dst, kind == CL_GATE_UP ? CL_BAR_U : CL_BAR_H);
#pragma unroll 1
  for (int i = ev.tid >> 4; i < ev.R * rd.n_quads; i += kClThreads / 16) {
    const int row = (int)((unsigned)i * rd.magic >> 20), quad = rd.quad0 + i - row * rd.n_quads, pair = me.p0 + 4 * quad;
    const float4* s = cl_at<float4>(p.lay.stg) + row * (me.np / 4) + quad;
    const float4 a = s[0];
    if (kind == CL_GATE_UP) {
      cl_send4(ev.dst + p.lay.u + cl_x_off<WT>(p.f, ev.R, row, pair), cl_x_pack<WT>(a), bar);
      continue;
    }
    const float4 b = s[ev.R * (me.np / 4)];
    const int f0 = cl_feature(pair);
    if (sizeof(WT) == 4) {
      cl_send4(ev.dst + p.lay.h + (row * p.d + f0) * 4, a, bar);
      cl_send4(ev.dst + p.lay.h + (row * p.d + f0 + 8) * 4, b, bar);
    } else {
      const float4 ga = *reinterpret_cast<const float4*>(gain + 4 * quad), gb = *reinterpret_cast<const float4*>(gain + p.lay.resid_np + 4 * quad);
      cl_send4(ev.dst + p.lay.y + cl_x_off<WT>(p.d, ev.R, row, f0), cl_x_pack<WT>(cl_mul(a, ga)), bar);
      cl_send4(ev.dst + p.lay.y + cl_x_off<WT>(p.d, ev.R, row, f0 + 8), cl_x_pack<WT>(cl_mul(b, gb)), bar);
      cl_send4(ev.dst + p.lay.h + (row * (p.d / 2) + pair) * 4,
               make_float4(fmaf(a.x, a.x, b.x * b.x), fmaf(a.y, a.y, b.y * b.y), fmaf(a.z, a.z, b.z * b.z), fmaf(a.w, a.w, b.w * b.w)), bar);
    }
  }
}

// ---- attention ------------------------------------------------------------------------------------------------
// A head's keys in chunks of 64, dealt to places: bf16 chunk c to place c mod 8, which walks its chunks with a running maximum;
// fp32 every chunk a place.  Place j belongs to CTA j mod `splits` of the head's; a team of four warps takes one (head,
// sequence, place) at a time, up to eight rows of the sequence together.  What a row leaves in a place (sum, maximum, output)
// goes to the head's first CTA, which adds the places in order and sends the result to everybody.
template <typename WT, int HD>
struct ClAttn {
  static constexpr bool BF = sizeof(WT) == 2;
  static constexpr int C = kAttnChunk, PARTS = BF ? 4 : 2, QD = HD / PARTS;  // threads per key, dimensions of each
  static constexpr int VPR = HD * (int)sizeof(WT) / 16;                      // 16-byte vectors of a row
  static constexpr int KLD = HD + 16 / (int)sizeof(WT);                      // elements of a key row, padded
  static constexpr int OH = BF ? 2 : 1;                                      // halves of a chunk's keys summed by themselves
  static constexpr int OT = HD * OH > kClTeam ? HD * OH / kClTeam : 1;       // (dimension, half) of a thread
  static constexpr int PLD = HD + 4;                                         // floats of a row in a place: output, maximum, sum
  static __device__ __forceinline__ int places(int pos) { return pos < 0 ? 0 : BF ? min(kAttnSplits, pos / C + 1) : pos / C + 1; }
};
__host__ __device__ constexpr int cl_team_bytes(int hd, int elem_bytes) {
  return kAttnChunk * (hd * elem_bytes + 16) + kAttnChunk * hd * elem_bytes + kClAttnRows * kAttnChunk * 4;
}
static_assert(kAttnChunk * (64 * 2 + 16) >= kClAttnRows * 64 * 4, "halves are added where the keys were");
__device__ __forceinline__ void cl_team_sync(int team) { asm volatile("bar.sync %0, %1;" ::"r"(2 + team), "n"(kClTeam) : "memory"); }

template <typename WT, int HD, int RM>
__device__ __forceinline__ void cl_attend(const ClParams& p, const ClEnv& ev, const WT* gk, const WT* gv, int hl, int b, int first_row, int place, bool& waited,
                                          unsigned qkv_bytes, unsigned parity) {
  using A = ClAttn<WT, HD>;
  constexpr bool BF = A::BF;
  constexpr int C = A::C;
  const int team = ev.warp / (kClTeam / 32), w4 = ev.warp % (kClTeam / 32), tt = ev.tid % kClTeam, lane = ev.lane;
  const int R = ev.R, row0 = b * ev.rps + first_row, rps = RM == 1 ? 1 : min(RM, ev.rps - first_row), rows_all = p.lay.heads_per_cta * R;
  const int max_pos = ev.sh->pos[row0 + rps - 1];
  // positions of a sequence's rows follow one another, and with them the keys that are not in the cache
  const int new_pos = ev.sh->pos[b * ev.rps + ev.rps - 1] - ev.rps + 1, base_pos = max(0, new_pos);
  WT* sK = cl_at<WT>(p.lay.team + team * p.lay.team_bytes);
  WT* sV = sK + C * A::KLD;
  float* sS = reinterpret_cast<float*>(sV + C * HD);  // [row][C]
  float* sO = reinterpret_cast<float*>(sK);           // at the end: [row][HD]
  const float* sq = cl_at<float>(p.lay.qkv) + (hl * R + row0) * ClQ<HD>::kLd;
  const WT* nk = reinterpret_cast<const WT*>(cl_at<float>(p.lay.qkv) + rows_all * ClQ<HD>::kLd) + (hl * R + b * ev.rps) * HD;  // keys of this pass
  const WT* nv = nk + rows_all * HD;
  float* s_m = ev.sh->att_m[team];
  float* s_l = ev.sh->att_l[team];
  float* s_a = ev.sh->att_a[team];
  float o[A::OT][RM];
#pragma unroll
  for (int u = 0; u < A::OT; ++u)
#pragma unroll
    for (int i = 0; i < RM; ++i) o[u][i] = 0.f;
  if (tt < rps) {
    s_m[tt] = -INFINITY;
    s_l[tt] = 0.f;
  }
#pragma unroll 1
  for (int c = place; c * C <= max_pos; c += BF ? kAttnSplits : 1 << 24) {
    const int key0 = c * C, n_keys = min(C, max_pos + 1 - key0);  // keys any row can see
    // what lies in the cache is asked for before the rows of the pass are there
    const int n_old = min(n_keys, base_pos - key0);
#pragma unroll 2
    for (int v = tt; v < n_old * A::VPR; v += kClTeam) {
      cp_async16(sK + v / A::VPR * A::KLD + v % A::VPR * (16 / (int)sizeof(WT)), reinterpret_cast<const uint4*>(gk + (size_t)key0 * HD) + v);
      cp_async16(reinterpret_cast<uint4*>(sV) + v, reinterpret_cast<const uint4*>(gv + (size_t)key0 * HD) + v);
    }
    if (!waited) {
      cl_wait(ev.sh, p.sync, CL_BAR_QKV, qkv_bytes, parity);
      waited = true;
    }
#pragma unroll 1
    for (int v = max(0, n_old) * A::VPR + tt; v < n_keys * A::VPR; v += kClTeam) {
      const int from = (key0 - new_pos) * A::VPR + v;
      *reinterpret_cast<uint4*>(sK + v / A::VPR * A::KLD + v % A::VPR * (16 / (int)sizeof(WT))) = reinterpret_cast<const uint4*>(nk)[from];
      reinterpret_cast<uint4*>(sV)[v] = reinterpret_cast<const uint4*>(nv)[from];
    }
    cp_async_wait_all();
    cl_team_sync(team);
    // scores
#pragma unroll 1
    for (int key = tt / A::PARTS; key < C; key += kClTeam / A::PARTS) {
      const int part = tt % A::PARTS;
      const WT* kr = sK + key * A::KLD + part * A::QD;
      const float* q = sq + ClQ<HD>::at(part * A::QD);
      float acc[RM];
#pragma unroll
      for (int i = 0; i < RM; ++i) acc[i] = 0.f;
      if (key < n_keys) {
#pragma unroll(RM == 1 ? 4 : 1)
        for (int e = 0; e < A::QD; e += 4) {
          const float4 k = load4(kr + e);
          const float* qe = q + e + e / (HD / 4) * 8;
#pragma unroll
          for (int i = 0; i < RM; ++i) {  // (rows the group does not have read something of this CTA's memory, and are not used)
            const float4 qv = *reinterpret_cast<const float4*>(qe + i * ClQ<HD>::kLd);
            acc[i] = fmaf(k.x, qv.x, acc[i]);
            acc[i] = fmaf(k.y, qv.y, acc[i]);
            acc[i] = fmaf(k.z, qv.z, acc[i]);
            acc[i] = fmaf(k.w, qv.w, acc[i]);
          }
        }
      }
#pragma unroll
      for (int i = 0; i < RM; ++i)
        if (RM == 1 || i < rps) {
          float s = acc[i];
#pragma unroll
          for (int w = 1; w < A::PARTS; w <<= 1) s += __shfl_xor_sync(0xffffffffu, s, w);
          if (part == 0) sS[i * C + key] = s * p.scale;
        }
    }
    cl_team_sync(team);
    // softmax of the chunk, a warp per row
#pragma unroll 1
    for (int i = w4; i < rps; i += kClTeam / 32) {
      const int n = cl_uniform(min(C, ev.sh->pos[row0 + i] + 1 - key0));
      if (n <= 0) {  // the row sees nothing here
        if (lane == 0) s_a[i] = 1.f;
        sS[i * C + lane] = 0.f;
        sS[i * C + lane + 32] = 0.f;
        continue;
      }
      const float s0 = lane < n ? sS[i * C + lane] : -INFINITY, s1 = lane + 32 < n ? sS[i * C + lane + 32] : -INFINITY;
      const float m_old = s_m[i], m_new = fmaxf(m_old, warp_max(fmaxf(s0, s1)));
      const float p0 = lane < n ? __expf(s0 - m_new) : 0.f, p1 = lane + 32 < n ? __expf(s1 - m_new) : 0.f;
      sS[i * C + lane] = p0;
      sS[i * C + lane + 32] = p1;
      const float sum = warp_sum(p0 + p1);
      if (lane == 0) {
        const float alpha = __expf(m_old - m_new);  // 0 on the row's first chunk
        s_a[i] = alpha;
        s_m[i] = m_new;
        s_l[i] = BF ? fmaf(s_l[i], alpha, sum) : sum;
      }
    }
    cl_team_sync(team);
    // output, keys in order
#pragma unroll
    for (int u = 0; u < A::OT; ++u) {
      const int id = tt + u * kClTeam, d = id % HD, half = id / HD;
      if (half < A::OH) {
        if (BF)
#pragma unroll
          for (int i = 0; i < RM; ++i) o[u][i] *= s_a[i];
        const int lo = half * (C / A::OH), hi = min(n_keys, lo + C / A::OH);
        int k = lo;
#pragma unroll(RM == 1 ? 2 : 1)
        for (; k + 4 <= hi; k += 4) {
          float v[4];
#pragma unroll
          for (int e = 0; e < 4; ++e) v[e] = to_f32(sV[(k + e) * HD + d]);
#pragma unroll
          for (int i = 0; i < RM; ++i) {
            const float4 p4 = *reinterpret_cast<const float4*>(sS + i * C + k);
            o[u][i] = fmaf(p4.x, v[0], o[u][i]);
            o[u][i] = fmaf(p4.y, v[1], o[u][i]);
            o[u][i] = fmaf(p4.z, v[2], o[u][i]);
            o[u][i] = fmaf(p4.w, v[3], o[u][i]);
          }
        }
#pragma unroll 1
        for (; k < hi; ++k) {
          const float v = to_f32(sV[k * HD + d]);
#pragma unroll
          for (int i = 0; i < RM; ++i) o[u][i] = fmaf(sS[i * C + k], v, o[u][i]);
        }
      }
    }
    cl_team_sync(team);  // the buffers are free again
  }
  // first + second half of the keys
  if constexpr (A::OH == 2 && A::OT == 1) {
    if (tt >= HD)
#pragma unroll
      for (int i = 0; i < RM; ++i)
        if (RM == 1 || i < rps) sO[i * HD + tt - HD] = o[0][i];
    cl_team_sync(team);
    if (tt < HD)
#pragma unroll
      for (int i = 0; i < RM; ++i)
        if (RM == 1 || i < rps) o[0][i] += sO[i * HD + tt];
  } else if constexpr (A::OH == 2) {
#pragma unroll
    for (int i = 0; i < RM; ++i) o[0][i] += o[A::OT - 1][i];
  }
  // ... to the head's first CTA
  const bool here = p.lay.splits == 1 || ev.rank < p.heads, live = !cl_aborted(ev.sh);
  const uint32_t owner = cl_map(ev.self, here ? ev.rank : ev.rank % p.heads), bar = cl_bar_of(p, owner, CL_BAR_PART);
#pragma unroll
  for (int i = 0; i < RM; ++i) {
    if ((RM > 1 && i >= rps) || place >= A::places(ev.sh->pos[row0 + i])) continue;
    const int at = p.lay.part + ((hl * R + row0 + i) * p.lay.part_slots + place) * A::PLD * 4;
    if (tt < HD) {
      if (here)
        *cl_at<float>(at + tt * 4) = o[0][i];
      else if (live)
        cl_send1(owner + at + tt * 4, o[0][i], bar);
    }
    if (tt == i) {
      if (here)
        *cl_at<float2>(at + HD * 4) = make_float2(s_m[i], s_l[i]);
      else if (live)
        cl_send2(owner + at + HD * 4, s_m[i], s_l[i], bar);
    }
  }
  cl_team_sync(team);  // the rows' state is used by the next item
}

// The weights of a row's places, left where their maxima and sums were: bf16 exp(m - max) / sum, as FoldStats; fp32 exp(m - max), and 1 / sum
// beside the first
template <typename WT, int HD>
__device__ __forceinline__ void cl_weigh(float* q, int n) {
  constexpr int LD = ClAttn<WT, HD>::PLD;
  constexpr bool BF = ClAttn<WT, HD>::BF;
  float mx = -INFINITY, l = 0.f;
#pragma unroll 1
  for (int j = 0; j < n; ++j) {
    const float2 ml = *reinterpret_cast<const float2*>(q + j * LD + HD);
    if (!BF || ml.y > 0.f) mx = fmaxf(mx, ml.x);
  }
#pragma unroll 1
  for (int j = 0; j < n; ++j) {
    const float2 ml = *reinterpret_cast<const float2*>(q + j * LD + HD);
    const float w = !BF || ml.y > 0.f ? __expf(ml.x - mx) : 0.f;
    l = fmaf(ml.y, w, l);
    q[j * LD + HD] = w;
  }
  const float inv_l = !BF || l > 0.f ? 1.0f / l : 0.f;
  if (BF)
#pragma unroll 1
    for (int j = 0; j < n; ++j) q[j * LD + HD] *= inv_l;
  else
    q[HD + 1] = inv_l;
}
// The places in order, four dimensions
template <typename WT, int HD>
__device__ __forceinline__ float4 cl_fold(const float* q, int n, int dim) {
  constexpr int LD = ClAttn<WT, HD>::PLD;
  float4 o = make_float4(0.f, 0.f, 0.f, 0.f);
  if (n <= 0) return o;
#pragma unroll 1
  for (int j = 0; j < n; ++j) {
    const float w = q[j * LD + HD];
    const float4 v = *reinterpret_cast<const float4*>(q + j * LD + dim);
    o.x = fmaf(v.x, w, o.x);
    o.y = fmaf(v.y, w, o.y);
    o.z = fmaf(v.z, w, o.z);
    o.w = fmaf(v.w, w, o.w);
  }
  if (ClAttn<WT, HD>::BF) return o;
  const float inv_l = q[HD + 1];
  return make_float4(o.x * inv_l, o.y * inv_l, o.z * inv_l, o.w * inv_l);
}

// Attention of this CTA's heads, its cache entries, and the sending of the outcome
template <typename WT, int HD>
__device__ __forceinline__ void cl_attention(const ClParams& p, const ClEnv& ev, const ClTab& t, int nh, unsigned& phases) {
  using A = ClAttn<WT, HD>;
  const int S = p.lay.splits, R = ev.R, rps = ev.rps, n_seq = R / rps;
  const bool many = p.heads >= kClCtas;
  const int split = many ? 0 : ev.rank / p.heads, head0 = many ? ev.rank : ev.rank - split * p.heads;
  auto phase = [&](int which) {
    const unsigned par = (phases >> which) & 1u;
    phases ^= 1u << which;
    return par;
  };
  auto cache_at = [&](void* base, int hl, int b) {
    return reinterpret_cast<WT*>(base) + ((size_t)b * p.heads + head0 + hl * kClCtas) * p.max_seq * HD;
  };
  const unsigned qkv_bytes = (unsigned)(nh * R * (HD * 4 + 2 * HD * (int)sizeof(WT))), parity = phase(CL_BAR_QKV);
  const int team = ev.warp / (kClTeam / 32);
  bool waited = false;
  int turn = 0;
#pragma unroll 1
  for (int hl = 0; hl < nh; ++hl)
#pragma unroll 1
    for (int b = 0; b < n_seq; ++b) {
      const int n = A::places(ev.sh->pos[b * rps + rps - 1]);
#pragma unroll 1
      for (int place = split; place < n; place += S) {
        if ((turn++ & 1) != team) continue;
        const WT *gk = cache_at(t.kcache, hl, b), *gv = cache_at(t.vcache, hl, b);
        if (rps == 1)
          cl_attend<WT, HD, 1>(p, ev, gk, gv, hl, b, 0, place, waited, qkv_bytes, parity);
        else if (rps == 2)
          cl_attend<WT, HD, 2>(p, ev, gk, gv, hl, b, 0, place, waited, qkv_bytes, parity);
        else
#pragma unroll 1
          for (int r0 = 0; r0 < rps; r0 += kClAttnRows) cl_attend<WT, HD, kClAttnRows>(p, ev, gk, gv, hl, b, r0, place, waited, qkv_bytes, parity);
      }
    }
  if (!waited) cl_wait(ev.sh, p.sync, CL_BAR_QKV, qkv_bytes, parity);
  __syncthreads();
  if (split == 0) {
    if (S > 1) {  // what the head's other CTAs send
      int n = 0;
#pragma unroll 1
      for (int row = 0; row < R; ++row) {
        const int places = A::places(ev.sh->pos[row]);
        n += places - (places + S - 1) / S;
      }
      if (n > 0) cl_wait(ev.sh, p.sync, CL_BAR_PART, (unsigned)(n * (HD + 2) * 4), phase(CL_BAR_PART));
    }
    if (ev.tid < nh * R) {
      const int row = nh == 1 ? ev.tid : ev.tid % R;
      cl_weigh<WT, HD>(cl_at<float>(p.lay.part) + ev.tid * p.lay.part_slots * A::PLD, A::places(ev.sh->pos[row]));
    }
    __syncthreads();
    if (!cl_aborted(ev.sh)) {
      const uint32_t bar = cl_bar_of(p, ev.dst, CL_BAR_X);
#pragma unroll 1
      for (int i = ev.tid >> 4; i < nh * R * (HD / 4); i += kClThreads / 16) {
        const int hr = i / (HD / 4), dim = (i % (HD / 4)) * 4, hl = nh == 1 ? 0 : hr / R, row = hr - hl * R;
        const float4 o = cl_fold<WT, HD>(cl_at<float>(p.lay.part) + hr * p.lay.part_slots * A::PLD, A::places(ev.sh->pos[row]), dim);
        cl_send4(ev.dst + p.lay.xo + cl_x_off<WT>(p.d, R, row, (head0 + hl * kClCtas) * HD + dim), cl_x_pack<WT>(o), bar);
      }
    }
  }
  // the rows' keys and values into the cache, by the CTA that reads them there
  const int rows_all = p.lay.heads_per_cta * R;
  const WT* kv = reinterpret_cast<const WT*>(cl_at<float>(p.lay.qkv) + rows_all * ClQ<HD>::kLd);
#pragma unroll 1
  for (int i = ev.tid; i < 2 * nh * R * A::VPR; i += kClThreads) {
    const int hr2 = i / A::VPR, v = i % A::VPR, which = hr2 >= nh * R ? 1 : 0, hr = hr2 - which * nh * R, hl = nh == 1 ? 0 : hr / R, row = hr - hl * R;
    const int pos = ev.sh->pos[row];
    if (pos < 0) continue;
    const int chunk = pos / A::C, place = A::BF ? chunk % kAttnSplits : chunk;
    if (place % S != split) continue;
    reinterpret_cast<uint4*>(cache_at(which ? t.vcache : t.kcache, hl, row / rps) + (size_t)pos * HD)[v] =
        reinterpret_cast<const uint4*>(kv + (which * rows_all + hr) * HD)[v];
  }
}

// the CTAs that hold a head: CTA c has heads c, c + 16, ...; with fewer heads than CTAs, `splits` CTAs share one
__device__ __forceinline__ int cl_heads_of(int cta, int heads, int splits) {
  if (heads >= kClCtas) return (heads - cta + kClCtas - 1) / kClCtas;
  return cta < heads * splits ? 1 : 0;
}

// What a pass's row carries
__device__ __forceinline__ void cl_plan_row(const ClShared* sh, int kind, int step, int rps, int row, int vocab, int& tok, int& pos) {
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
  tok = min(max(tok, 0), vocab - 1);  // (no token of a round whose logits were not numbers)
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

// bf16: a linear stage, dot products to sending
template <int HD, int CG>
__device__ __forceinline__ void cl_stage_bf16(const ClParams& p, const ClEnv& ev, const ClDots& a, const ClTab& t) {
  const ClMine& me = ev.mine[a.kind];
  const bool is_head = a.kind == CL_HEAD;
  const int R = ev.R;
  const ClEntry* ent = ev.entries + me.entry0 + ev.warp * me.n_entries;
  ClRing ring;
  ring.W = reinterpret_cast<const uint4*>(a.W) + ev.lane;
  ring.buf = ev.self + p.lay.ring + ev.warp * (kClRing * 512) + ev.lane * 16;
  ring.wrap_jump = (a.K / 16 - 1) * 256;  // to the next group's unit of the same k-tile, which starts with its first tile
  const int n_rounds = cl_uniform(me.n_rounds), width = cl_uniform(me.tile_width);
  if (n_rounds > 0) {
    ring.begin(ent);
    if (width == 1)
      ring.fill<1>();
    else if (width == 2)
      ring.fill<2>();
    else
      ring.fill<4>();
  }
  if (a.bar >= 0) cl_wait(ev.sh, p.sync, a.bar, a.bytes, a.parity);
  // lm-head: 256 threads over the rows, a power of two of them each
  const int row_log = R <= 1 ? 8 : R <= 2 ? 7 : R <= 4 ? 6 : R <= 8 ? 5 : 4;
  float bv = -INFINITY;
  int bi = 0x7fffffff;
#pragma unroll 1
  for (int r = 0; r < n_rounds; ++r) {
    const ClRound& rd = ev.rounds[me.round0 + r];
    if (width == 1)
      cl_mma_round<1, CG>(p, ev, a.x, ent, ring);
    else if (width == 2)
      cl_mma_round<2, CG>(p, ev, a.x, ent, ring);
    else
      cl_mma_round<4, CG>(p, ev, a.x, ent, ring);
    if (a.norm && a.bar >= 0 && r == 0) cl_row_scales(p, ev);  // (the first stage's were made with the embedding)
    __syncthreads();  // the sums are there
    if (is_head) {
      cl_head_round(p, ev, me, rd, a.logits, row_log, bv, bi);
    } else {
      cl_values<__nv_bfloat16, HD>(p, ev, me, rd, t.kind);
      __syncthreads();
      if (cl_aborted(ev.sh)) {
      } else if (t.kind == CL_QKV) {
        cl_send_qkv<__nv_bfloat16, HD>(p, ev, me, rd);
      } else {
        cl_send_all<__nv_bfloat16>(p, ev, me, rd, t.kind, t.gain_out);
      }
    }
    if (r + 1 < n_rounds) __syncthreads();
  }
  if (is_head && a.logits == nullptr) {
    if (n_rounds == 0) __syncthreads();
#pragma unroll 1
    for (int o = min(16, 1 << (row_log - 1)); o > 0; o >>= 1) cl_better(bv, bi, __shfl_xor_sync(0xffffffffu, bv, o), __shfl_xor_sync(0xffffffffu, bi, o));
    const int lanes = min(32, 1 << row_log), in_row = ev.tid & ((1 << row_log) - 1), row = ev.tid >> row_log;
    if (row < R && in_row % lanes == 0) cl_at<float2>(p.lay.best)[row * 4 * kClWarps + in_row / lanes] = make_float2(bv, __int_as_float(bi));
  }
}

template <typename WT, int HD, int CG>
__device__ __forceinline__ void cl_compute(const ClParams& p, ClShared* sh, const ClTab* tab_t, const ClTab* tab_d, int rank, bool loop, int batch, int k) {
  constexpr bool BF = sizeof(WT) == 2;
  const int tid = threadIdx.x;
  ClEnv ev{};
  ev.sh = sh;
  ev.mine = cl_at<ClMine>(p.lay.plan);
  ev.rounds = cl_at<ClRound>(p.lay.plan_rounds);
  ev.entries = cl_at<ClEntry>(p.lay.plan_entries);
  ev.tid = tid;
  ev.warp = cl_uniform(tid >> 5);
  ev.lane = tid & 31;
  ev.rank = rank;
  ev.self = smem_u32(cl_smem);
  ev.dst = cl_map(ev.self, tid & (kClCtas - 1));
  const int my_heads = cl_heads_of(rank, p.heads, p.lay.splits);
  unsigned phases = 0;

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
    {
      const float* gain = p.gains[draft ? p.first_gain_d : p.first_gain_t];
#pragma unroll 1
      for (int row = ev.warp; row < R; row += kClWarps) {
        int tok, pos;
        cl_plan_row(sh, kind, loop ? pass : p.pd.step, ev.rps, row, p.vocab, tok, pos);
        if (ev.lane == 0) sh->pos[row] = pos;
        const WT* e = reinterpret_cast<const WT*>(p.embed) + (size_t)tok * p.d;
        float* own = cl_at<float>(p.lay.hres) + row * p.lay.resid_np;
        const int q0 = ev.mine[CL_O].p0, q1 = q0 + ev.mine[CL_O].np;
        constexpr int hp = HD / 2;
        const int at = max(pos, 0) * hp;
        float cs[hp / 32], sn[hp / 32];
#pragma unroll
        for (int i = 0; i < hp / 32; ++i) {
          cs[i] = __ldg(p.rope_cos + at + i * 32 + ev.lane);
          sn[i] = __ldg(p.rope_sin + at + i * 32 + ev.lane);
        }
        float total = 0.f;
#pragma unroll 2
        for (int c0 = 0; c0 < p.d; c0 += 128) {
          const int c = c0 + ev.lane * 4;
          float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
          if (c < p.d) {
            if (pos >= 0) v = load4(e + c);
            if (BF) {
              const float4 g = __ldg(reinterpret_cast<const float4*>(gain + c));
              *reinterpret_cast<float4*>(cl_smem + p.lay.y + cl_x_off<WT>(p.d, R, row, c)) = cl_x_pack<WT>(make_float4(v.x * g.x, v.y * g.y, v.z * g.z, v.w * g.w));
            } else {
              *reinterpret_cast<float4*>(cl_at<float>(p.lay.h) + row * p.d + c) = v;
            }
            const int pair = (c >> 4) * 8 + (c & 7);  // of the first of these four features
            if (pair >= q0 && pair < q1) *reinterpret_cast<float4*>(own + ((c >> 3) & 1) * p.lay.rows * p.lay.resid_np + pair - q0) = v;
          }
          if (BF) {  // a row's squares as the whole-pass kernel's first stage adds them: by 128 columns, the blocks in order
            float s = fmaf(v.x, v.x, 0.f);
            s = fmaf(v.y, v.y, s);
            s = fmaf(v.z, v.z, s);
            s = fmaf(v.w, v.w, s);
            total += warp_sum(s);
          }
        }
        if (BF && ev.lane == 0) sh->inv[row] = rsqrtf(total / (float)p.d + p.eps);
        float* rope = cl_at<float>(p.lay.rope) + row * 2 * hp;
#pragma unroll
        for (int i = 0; i < hp / 32; ++i) {
          rope[i * 32 + ev.lane] = cs[i];
          rope[hp + i * 32 + ev.lane] = sn[i];
        }
        if (loop) cl_at<float2>(p.lay.best)[row * 4 * kClWarps + ev.lane] = make_float2(-INFINITY, __int_as_float(0x7fffffff));
      }
    }
    __syncthreads();

#pragma unroll 1
    for (int s = 0; s < n_stages; ++s) {
      const ClTab t = tab[s];
      ClDots a{};
      a.W = t.W;
      a.kind = t.kind;
      a.x = t.x;
      a.K = t.K;
      a.bar = s > 0 ? t.bar : -1;  // the first stage's are the embedding
      a.bytes = (unsigned)(R * t.row_bytes);
      a.parity = (phases >> t.bar) & 1u;
      if (s > 0) phases ^= 1u << t.bar;
      a.norm = t.norm != 0;
      a.gain = t.gain;
      a.logits = loop ? nullptr : p.logits;
      const ClMine& me = ev.mine[t.kind];
      const bool is_head = t.kind == CL_HEAD;
      if constexpr (BF) {
        cl_stage_bf16<HD, CG>(p, ev, a, t);
      } else {
        if (R == 1)
          cl_dots_f32<1, 4>(p, ev, a);
        else if (R <= 4)
          cl_dots_f32<4, 2>(p, ev, a);
        else
          cl_dots_f32<8, 2>(p, ev, a);
        if (!is_head) {
          const ClRound& rd = ev.rounds[me.round0];
          __syncthreads();  // the sums are there
          cl_values<WT, HD>(p, ev, me, rd, t.kind);
          __syncthreads();
          if (cl_aborted(sh)) {
          } else if (t.kind == CL_QKV) {
            cl_send_qkv<WT, HD>(p, ev, me, rd);
          } else {
            cl_send_all<WT>(p, ev, me, rd, t.kind, t.gain_out);
          }
        }
      }
      if (t.kind == CL_QKV && my_heads > 0) cl_attention<WT, HD>(p, ev, t, my_heads, phases);
    }
    if (!loop) break;

    // ---- greedy decision: best of the CTA, then of the cluster ----
    __syncthreads();
    if (!cl_aborted(sh))
#pragma unroll 1
      for (int row = ev.warp; row < R; row += kClWarps) {
        const float2 c = cl_at<float2>(p.lay.best)[row * 4 * kClWarps + ev.lane];
        float bv = c.x;
        int bi = __float_as_int(c.y);
        cl_best_of_lanes<32>(bv, bi);
        if (ev.lane < kClCtas) cl_send2(ev.dst + p.lay.tok + (rank * R + row) * 8, bv, __int_as_float(bi), cl_bar_of(p, ev.dst, CL_BAR_TOK));
      }
    cl_wait(sh, p.sync, CL_BAR_TOK, (unsigned)(kClCtas * R * 8), (phases >> CL_BAR_TOK) & 1u);
    phases ^= 1u << CL_BAR_TOK;
#pragma unroll 1
    for (int row = ev.warp; row < R; row += kClWarps) {
      const float2 c = cl_at<float2>(p.lay.tok)[(ev.lane & (kClCtas - 1)) * R + row];
      float bv = c.x;
      int bi = __float_as_int(c.y);
      cl_best_of_lanes<kClCtas>(bv, bi);
      if (ev.lane == 0) sh->amax[row] = min(max(bi, 0), p.vocab - 1);
    }
    __syncthreads();
    if (tid < 32) {
      if (verify)
        cl_commit(p, sh, batch, k, rank == 0, tid);
      else if (tid < batch)
        sh->drafts[tid][pass] = sh->amax[tid * ev.rps + ev.rps - 1];
    }
    if (!cl_agree_ok(&sh->abort) || (verify && (sh->all_done || sh->round >= p.rounds))) break;
  }
  __syncthreads();
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

// CG: column groups of eight rows (bf16); all passes of a context take the same
template <typename WT, int HD, int CG>
__global__ void __launch_bounds__(kClThreads, 1) cluster_pass_kernel(const __grid_constant__ ClParams p) {
  ClShared* sh = cl_at<ClShared>(p.lay.shared);
  ClTab* tab_t = cl_at<ClTab>(p.lay.tab);
  ClTab* tab_d = tab_t + p.n_t;
  const int tid = threadIdx.x, rank = (int)cl_rank();
  const bool loop = p.rounds > 0;
  const int batch = cl_uniform(loop ? p.gs->batch : p.pd.n_seq), k = cl_uniform(loop ? p.gs->k : 0);

  // ---- set-up: this CTA's plan, stage tables, the gains of its features, state ----
#pragma unroll 1
  for (int i = tid; i < p.lay.plan_bytes / 16; i += kClThreads)
    cl_at<uint4>(p.lay.plan)[i] = __ldg(reinterpret_cast<const uint4*>(p.plan + (size_t)rank * p.lay.plan_bytes) + i);
#pragma unroll 1
  for (int i = tid; i < p.n_t + p.n_d; i += kClThreads) {
    const ClStage s = i < p.n_t ? p.prog_t[i] : p.prog_d[i - p.n_t];
    ClTab& t = tab_t[i];
    t.kind = s.kind;
    t.K = s.K;
    t.norm = s.kind == CL_QKV || s.kind == CL_GATE_UP || s.kind == CL_HEAD;
    t.gain = sizeof(WT) == 4 && t.norm ? p.gains[s.gain] : nullptr;
    t.gain_out = s.gain;
    t.x = s.kind == CL_O ? p.lay.xo : s.kind == CL_DOWN ? p.lay.u : p.lay.y;
    t.bar = s.kind == CL_O ? CL_BAR_X : s.kind == CL_DOWN ? CL_BAR_U : CL_BAR_H;
    t.row_bytes = s.kind == CL_DOWN ? p.f * 4 : s.kind == CL_O || sizeof(WT) == 4 ? p.d * 4 : p.d * 6;
    t.kcache = s.kcache;
    t.vcache = s.vcache;
    t.W = s.W + (sizeof(WT) == 4 ? (size_t)cl_first_pair(cl_pairs_of(s.kind, p.d, p.f, p.vocab), rank, 4) * 2 * s.K * 4 : 0);
  }
  if (sizeof(WT) == 2) {
    const int p0 = cl_first_pair(p.d / 2, rank, 2), np = cl_first_pair(p.d / 2, rank + 1, 2) - p0, ld = 2 * p.lay.resid_np;
#pragma unroll 1
    for (int i = tid; i < p.n_gains * 2 * np; i += kClThreads) {
      const int g = i / (2 * np), r = i - g * 2 * np, half = r >= np ? 1 : 0, pl = r - half * np, pair = p0 + pl;
      cl_at<float>(p.lay.gain)[g * ld + half * p.lay.resid_np + pl] = __ldg(p.gains[g] + cl_feature(pair) + half * 8);
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

  if (!cl_aborted(sh)) cl_compute<WT, HD, CG>(p, sh, tab_t, tab_d, rank, loop, batch, k);

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

// ---- host -------------------------------------------------------------------------------------------------------
// What every CTA does of the five kinds of matrices, [CTA][stride].  bf16: the units of a group of 128 features are cut
// as the whole-pass kernel's CTAs share them (stage_shares), and dealt to the classes from the beginning of each CTA's range.
// place_slots: places the sums of a round may take; 0: only work out what a plan needs.
struct ClPlan {
  std::vector<unsigned char> bytes;
  int rounds_at = 0, entries_at = 0, stride = 0;
  int most_places = 0;  // places the sums of a layer's stage take when it is finished in one round
  int most_cuts = 1;    // pieces of a sum
  int most_quads = 0;   // fours of pairs in a round of a layer's stage
  long long most_units = 0;  // bf16: of a matrix, in uint4
};

inline ClPlan cluster_plan(int d, int f, int vocab, int elem_bytes, int pass_grid, int place_slots) {
  struct Cut {
    int kt0, len, cls0;
    bool operator==(const Cut& o) const { return kt0 == o.kt0 && len == o.len && cls0 == o.cls0; }
  };
  struct Batch {  // up to kClTiles neighbouring tiles that are cut alike
    int tile, n, np;
  };
  struct Cta {
    ClMine mine[CL_KINDS];
    std::vector<ClRound> rounds;
    std::vector<ClEntry> entries;
  };
  std::vector<Cta> ctas(kClCtas);
  std::vector<std::vector<ClEntry>> lists(kClasses);
  std::vector<Batch> batches;
  std::vector<StageShare> shares(pass_grid);
  ClPlan out;
  for (int kind = 0; kind < CL_KINDS; ++kind) {
    const int n_pairs = cl_pairs_of(kind, d, f, vocab);
    const int K = kind == CL_DOWN ? f : d, KT = K / 16, NT = n_pairs / 8, n_groups = (NT + kUnitTiles - 1) / kUnitTiles;
    std::vector<std::vector<Cut>> cuts;
    if (elem_bytes == 2) {
      out.most_units = std::max(out.most_units, (long long)n_groups * KT * (kUnitBytes / 16));
      stage_shares(shares.data(), n_groups, KT, pass_grid);
      cuts.resize(n_groups);
      for (const StageShare& s : shares)
        for (int u = 0; u < s.n;) {
          const int grp = (s.ub + u) / KT, kt0 = (s.ub + u) % KT, len = std::min(s.n - u, KT - kt0);
          cuts[grp].push_back(Cut{kt0, len, u % kClasses});
          u += len;
        }
    }
    for (int rank = 0; rank < kClCtas; ++rank) {
      Cta& c = ctas[rank];
      ClMine& m = c.mine[kind];
      m = ClMine{};
      m.p0 = cl_first_pair(n_pairs, rank, elem_bytes);
      m.np = cl_first_pair(n_pairs, rank + 1, elem_bytes) - m.p0;
      m.round0 = (int)c.rounds.size();
      m.entry0 = (int)c.entries.size();
      m.tile_width = 1;
      auto add_round = [&](int pair0, int pair1) -> ClRound& {
        ClRound r{};
        r.quad0 = (pair0 - m.p0) / 4;
        r.n_quads = (pair1 - pair0) / 4;
        r.magic = r.n_quads > 0 ? (1u << 20) / (unsigned)r.n_quads + 1u : 0u;
        if (kind != CL_HEAD) out.most_quads = std::max(out.most_quads, r.n_quads);
        c.rounds.push_back(r);
        m.n_rounds += 1;
        return c.rounds.back();
      };
      if (elem_bytes != 2) {
        add_round(m.p0, m.p0 + m.np);
        continue;
      }
      if (m.np == 0) continue;
      batches.clear();
      const int t1 = (m.p0 + m.np + 7) / 8;
      int places = 0, width = 1;
      for (int t = m.p0 / 8; t < t1;) {
        const std::vector<Cut>& cut = cuts[t / kUnitTiles];
        const int np = (int)cut.size(), most = place_slots > 0 ? std::max(1, std::min((int)kClTiles, place_slots / np)) : kClTiles;
        int n = 1;
        while (n < most && t + n < t1 && cuts[(t + n) / kUnitTiles] == cut) ++n;
        batches.push_back(Batch{t, n, np});
        out.most_cuts = std::max(out.most_cuts, np);
        width = std::max(width, n);
        places += n * np;
        t += n;
      }
      if (kind != CL_HEAD) out.most_places = std::max(out.most_places, places);
      m.tile_width = width == 3 ? 4 : width;
      if (place_slots <= 0) continue;
      for (auto& l : lists) l.clear();
      for (size_t b = 0; b < batches.size();) {
        size_t e = b;
        int tiles = 0;  // ... of the round
        while (e < batches.size() && batches[e].np == batches[b].np && (e == b || (tiles + batches[e].n) * batches[b].np <= place_slots)) tiles += batches[e++].n;
        const int tile0 = batches[b].tile;
        ClRound& r = add_round(std::max(m.p0, tile0 * 8), std::min(m.p0 + m.np, (tile0 + tiles) * 8));
        r.tile0 = tile0;
        r.np = batches[b].np;
        for (int cls = 0; cls < kClasses; ++cls)
          for (size_t i = b; i < e; ++i) {
            const Batch& bt = batches[i];
            const int grp = bt.tile / kUnitTiles, in = bt.tile % kUnitTiles;
            for (int pc = 0; pc < bt.np; ++pc) {
              const Cut& cut = cuts[grp][pc];
              ClEntry en{};
              en.n_tiles = (unsigned char)bt.n;
              en.wrap = (unsigned char)(kUnitTiles - in);
              en.np = (unsigned char)bt.np;
              en.kt = -1;
              const int slot = (bt.tile - tile0) * bt.np + pc, first = (cls - cut.cls0 + kClasses) % kClasses;
              for (int j = first; j < cut.len; j += kClasses) {
                en.kt = (short)(cut.kt0 + j);
                en.w = (grp * KT + en.kt) * (kUnitBytes / 16) + in * 32;
                en.slot = j + kClasses < cut.len ? -1 : (short)slot;
                lists[cls].push_back(en);
              }
              if (first >= cut.len) {  // nothing to add: the place is zero
                en.slot = (short)slot;
                lists[cls].push_back(en);
              }
            }
          }
        b = e;
        for (auto& l : lists) l.back().last = b < batches.size() ? 1 : 2;
      }
      for (const auto& l : lists) m.n_entries = std::max(m.n_entries, (int)l.size());
      for (auto& l : lists) {
        l.resize(m.n_entries);
        c.entries.insert(c.entries.end(), l.begin(), l.end());
      }
    }
  }
  size_t rounds = 0, entries = 0;
  for (const Cta& c : ctas) {
    rounds = std::max(rounds, c.rounds.size());
    entries = std::max(entries, c.entries.size());
  }
  out.rounds_at = CL_KINDS * (int)sizeof(ClMine);
  out.entries_at = out.rounds_at + (int)(rounds * sizeof(ClRound));
  out.stride = out.entries_at + (int)(entries * sizeof(ClEntry));
  out.bytes.assign((size_t)out.stride * kClCtas, 0);
  for (int rank = 0; rank < kClCtas; ++rank) {
    unsigned char* at = out.bytes.data() + (size_t)rank * out.stride;
    const Cta& c = ctas[rank];
    std::copy_n(reinterpret_cast<const unsigned char*>(c.mine), sizeof c.mine, at);
    std::copy_n(reinterpret_cast<const unsigned char*>(c.rounds.data()), c.rounds.size() * sizeof(ClRound), at + out.rounds_at);
    std::copy_n(reinterpret_cast<const unsigned char*>(c.entries.data()), c.entries.size() * sizeof(ClEntry), at + out.entries_at);
  }
  return out;
}

// The layout for passes of up to `rows` rows; total = 0 when it does not fit
inline ClLayout cluster_layout(int d, int f, int heads, int hd, int n_layers, int rows, int max_seq, int elem_bytes, int place_slots, const ClPlan& plan,
                               int max_smem) {
  ClLayout y{};
  const bool bf16 = elem_bytes == 2;
  y.rows = rows;
  const int chunks = (max_seq + kAttnChunk - 1) / kAttnChunk;
  y.part_slots = bf16 ? std::min((int)kAttnSplits, chunks) : chunks;
  y.heads_per_cta = (heads + kClCtas - 1) / kClCtas;
  y.splits = heads >= kClCtas ? 1 : std::min(kClCtas / heads, y.part_slots);  // CTAs per head
  y.resid_np = cl_max_pairs(d / 2, elem_bytes);
  int at = 0;
  auto take = [&](int& off, long long bytes) {
    off = at;
    at = (int)std::min<long long>(1 << 30, ((long long)at + bytes + 127) / 128 * 128);
  };
  const long long hpr = (long long)y.heads_per_cta * rows;
  take(y.h, (bf16 ? 2LL : 4LL) * rows * d);
  take(y.y, 4LL * rows * d);
  // u lies over what the attention receives and sends: it is written when every CTA has taken the O-projection's input in, and
  // read before any CTA sends anything of the next layer's attention
  const int u0 = at;
  take(y.part, 4LL * hpr * y.part_slots * (hd + 4));
  take(y.xo, 4LL * rows * d);
  const int att_end = at;
  at = u0;
  take(y.u, 4LL * rows * f);
  at = std::max(at, att_end);
  take(y.qkv, hpr * ((hd + 32) * 4 + 2 * hd * elem_bytes));
  take(y.gain, bf16 ? 8LL * (2 * n_layers + 1) * y.resid_np : 0);
  take(y.hres, 8LL * rows * y.resid_np);
  take(y.stg, 8LL * rows * std::max(cl_max_pairs(3 * d / 2, elem_bytes), cl_max_pairs(f, elem_bytes)));
  // the attention's keys and values lie over the weights on their way and the sums: it starts behind the barrier that ends the
  // QKV stage's, and ends with one before the O-projection's begin
  const int w0 = at;
  y.team_bytes = cl_team_bytes(hd, elem_bytes);
  take(y.team, 2LL * y.team_bytes);
  const int team_end = at;
  at = w0;
  take(y.ring, bf16 ? kClWarps * (long long)kClRing * 512 : 0);
  take(y.red, bf16 ? (long long)place_slots * kClasses * 8 * ((rows + 1) / 2) * 16 : 0);
  at = std::max(at, team_end);
  take(y.rope, 4LL * rows * hd);
  take(y.tok, 8LL * kClCtas * rows);
  take(y.best, 32LL * rows * kClWarps);
  take(y.tab, (long long)sizeof(ClTab) * 2 * (4 * n_layers + 1));
  take(y.plan, plan.stride);
  y.plan_rounds = y.plan + plan.rounds_at;
  y.plan_entries = y.plan + plan.entries_at;
  y.plan_bytes = plan.stride;
  take(y.shared, (long long)sizeof(ClShared));
  // what the kernel's fields hold: the bytes of a stage on an mbarrier (20 bits), a round's vectors divided by multiplication, places, pieces
  // and k-tiles of an entry, units of a matrix; and the first norm's squares, added as sixteen warps of 128 columns do
  const long long most_bytes = std::max({6LL * rows * d, 4LL * rows * f, hpr * (4 * hd + 2 * hd * elem_bytes), hpr * y.part_slots * (hd + 2) * 4, 8LL * kClCtas * rows});
  const bool held = most_bytes < 1 << 20 && (long long)rows * plan.most_quads * plan.most_quads < 1 << 20 && place_slots < 1 << 15 && plan.most_cuts < 256 &&
                    std::max(d, f) / 16 < 1 << 15 && plan.most_units < 1LL << 31 && d <= 2048;
  y.total = held && at <= max_smem ? at : 0;
  return y;
}

}  // namespace sdfp
