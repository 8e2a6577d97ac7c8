// One pass over the logit rows of the masked positions, and the selection that follows it: the common machinery of
// dlm_unmask_select and dlm_unmask_select_scored (unmask.cu).
//
// Bound by HBM for more than a few dozen rows, by the chain of dependent round trips below that.  One block per (chunk, row):
// it reads the row's mask byte and, if that is set, streams its chunk in batches of 4096 logits, 16 per thread, one batch in
// flight during the arithmetic of the one before.  The arithmetic is about 5 instructions per logit (14 before: the
// exponential's argument, the sums and the maximum one logit at a time, indices tracked per logit; the entropy 40): packed
// pairs for subtract, multiply and add, three-input maxima, one maximum per warp instead of one per lane, and indices looked
// at only in batches that raise it.
// (A persistent variant that listed the masked rows first, dealt chunks out through a counter and streamed through a ring of
// bulk copies in shared memory was slower: 36 us against 30 at 155.7 MB; its blocks cannot start under the tail of
// the launch before, and the ring's barriers cost as much as the loads they hide.)
// All chunks of a call have the same boundaries and all trees a fixed order, so results do not depend on scheduling
// and identical rows give identical bits.
//
// A chunk's statistics (Entry) go to the workspace; the last block of a batch element to finish (a release-acquire ticket)
// merges that element's entries, eight or four lanes per row, and ranks the positions.
#pragma once

#include <math_constants.h>

#include "common.cuh"
#include "sm100_ptx.cuh"

namespace vocab {

using sm100::add2;
using sm100::fma2;
using sm100::mul2;
using sm100::pack2;
using sm100::unpack2;

constexpr int kThreads = 256;
constexpr int kWarps = kThreads / 32;
constexpr int kBlocksPerSm = 4;
constexpr int kPer = 16;                        // logits per thread and batch
constexpr int kBatch = kThreads * kPer;         // logits of a batch
constexpr int kChunkUnit = kBatch;              // workspace sizing: at most one entry per batch of a row
constexpr int kMaxBlockLen = 1024;
constexpr int kMaxRows = 65535;

// What is kept per thread, block and chunk beside the maximum m, its lowest index and s = sum exp(z - m):
enum Kind { kConfidence, kEntropy, kMargin };   // nothing; t = sum (z - m) exp(z - m); the second largest entry

struct Entry {
  float m;
  int idx;
  float s;
  float x;   // t or the second largest entry
};

struct Args {
  const float* logits;
  int rows, block_len, vocab, k;
  int chunk_len, n_chunks;   // every chunk but the last has chunk_len logits
  FastDiv by_block_len;
  uint8_t* masked;
  int32_t* tokens;
  int32_t* tok;
  float* conf;
  int32_t* sel_idx;
  int32_t* n_sel;
  // scored calls (otherwise nullptr): the ranking score, the largest logit, and what is added to ln(conf)
  float* score;
  float* zmax;
  const float* noise;
  Entry* entries;            // [rows][n_chunks]
  unsigned int* tickets;     // [batch elements] finished blocks, or nullptr: the selection is a kernel of its own
};

__device__ __forceinline__ float exp_fast(float x) { return sm100::ex2_approx(x * 1.4426950408889634f); }

__device__ __forceinline__ float max3(float a, float b, float c) {
  float r;
  asm("max.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(b), "f"(c));
  return r;
}

// ---- streaming.  VEC: every row starts on a 16-byte boundary and a thread takes 16-byte vectors; otherwise single logits 256
// apart (coalesced all the same), in every row of the call, so that a row's sums do not depend on where it lies.
template <bool VEC>
__device__ __forceinline__ int element(int base, int j) {   // index of the thread's j-th logit of the batch at `base`
  return VEC ? base + ((j >> 2) * kThreads + (int)threadIdx.x) * 4 + (j & 3) : base + j * kThreads + (int)threadIdx.x;
}

template <bool VEC>
__device__ __forceinline__ void load_batch(const float* __restrict__ z, int base, int end, float (&x)[kPer]) {
  constexpr int kLoads = VEC ? kPer / 4 : kPer, kStep = VEC ? 4 : 1;
  const float* const p = z + element<VEC>(base, 0);
  if (base + kBatch <= end) {
#pragma unroll
    for (int v = 0; v < kLoads; ++v) {
      if (VEC) {
        const float4 f = __ldcs(reinterpret_cast<const float4*>(p + v * kThreads * 4));
        x[4 * v] = f.x; x[4 * v + 1] = f.y; x[4 * v + 2] = f.z; x[4 * v + 3] = f.w;
      } else {
        x[v] = __ldcs(p + v * kThreads);
      }
    }
  } else {
#pragma unroll
    for (int v = 0; v < kLoads; ++v) {
      const bool in = element<VEC>(base, v * kStep) < end;
      if (VEC) {
        float4 f = make_float4(-CUDART_INF_F, -CUDART_INF_F, -CUDART_INF_F, -CUDART_INF_F);
        if (in) f = __ldcs(reinterpret_cast<const float4*>(p + v * kThreads * 4));
        x[4 * v] = f.x; x[4 * v + 1] = f.y; x[4 * v + 2] = f.z; x[4 * v + 3] = f.w;
      } else {
        x[v] = in ? __ldcs(p + v * kThreads) : -CUDART_INF_F;
      }
    }
  }
}

// A warp's statistics of an item so far.  The maximum is the warp's, the same in every lane (one redux per batch): batches
// that raise it become rare quickly, whereas some lane of 32 beats its own maximum in nearly every batch.  s and t are
// the lane's sums relative to it; idx is the lowest index the lane itself has found it at.
struct Running {
  float m, m2, s, t;
  int idx;
  __device__ __forceinline__ void clear() {
    m = m2 = -CUDART_INF_F;
    s = t = 0.f;
    idx = 0x7fffffff;
  }
};

__device__ __forceinline__ float warp_max(float v) {
  float r;
  asm("redux.sync.max.f32 %0, %1, 0xffffffff;" : "=f"(r) : "f"(v));
  return r;
}

// s and t of the batch relative to m
template <int KIND>
__device__ __forceinline__ void sum_batch(const float (&x)[kPer], float m, float& s, float& t) {
  const uint64_t neg_m = pack2(-m, -m), l2e = pack2(1.4426950408889634f, 1.4426950408889634f);
  uint64_t s0 = 0, s1 = 0, t0 = 0, t1 = 0;   // pairs of zeros
#pragma unroll
  for (int j = 0; j < kPer; j += 4) {
    uint64_t d0 = add2(pack2(x[j], x[j + 1]), neg_m), d1 = add2(pack2(x[j + 2], x[j + 3]), neg_m);
    float a, b;
    if (KIND == kEntropy) {   // -inf contributes 0 to both sums: far below where the exponential is 0 the difference is cut off
      unpack2(d0, a, b);
      d0 = pack2(fmaxf(a, -1e4f), fmaxf(b, -1e4f));
      unpack2(d1, a, b);
      d1 = pack2(fmaxf(a, -1e4f), fmaxf(b, -1e4f));
    }
    unpack2(mul2(d0, l2e), a, b);
    const uint64_t e0 = pack2(sm100::ex2_approx(a), sm100::ex2_approx(b));
    unpack2(mul2(d1, l2e), a, b);
    const uint64_t e1 = pack2(sm100::ex2_approx(a), sm100::ex2_approx(b));
    s0 = add2(s0, e0);
    s1 = add2(s1, e1);
    if (KIND == kEntropy) {
      t0 = fma2(d0, e0, t0);
      t1 = fma2(d1, e1, t1);
    }
  }
  float a, b;
  unpack2(add2(s0, s1), a, b);
  s = a + b;
  if (KIND == kEntropy) {
    unpack2(add2(t0, t1), a, b);
    t = a + b;
  }
}

template <int KIND, bool VEC>
__device__ __forceinline__ void take_batch(Running& r, const float (&x)[kPer], int base) {
  // the sums against the maximum so far, beside the batch's own maximum and not behind it; in the rare batch that raises
  // the maximum (and in the first) they are taken again
  float s, t = 0.f;
  sum_batch<KIND>(x, r.m, s, t);
  float b4[4];
#pragma unroll
  for (int q = 0; q < 4; ++q) b4[q] = fmaxf(max3(x[4 * q], x[4 * q + 1], x[4 * q + 2]), x[4 * q + 3]);
  const float bm = fmaxf(max3(b4[0], b4[1], b4[2]), b4[3]);
  const float wm = warp_max(bm);
  if (KIND == kMargin && wm > r.m2) {   // the batch holds one of the two largest so far
    float m1 = -CUDART_INF_F, m2 = -CUDART_INF_F;
#pragma unroll
    for (int j = 0; j < kPer; ++j) {
      m2 = fmaxf(m2, fminf(m1, x[j]));
      m1 = fmaxf(m1, x[j]);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      const float o1 = __shfl_xor_sync(0xffffffffu, m1, o), o2 = __shfl_xor_sync(0xffffffffu, m2, o);
      m2 = max3(m2, o2, fminf(m1, o1));
      m1 = fmaxf(m1, o1);
    }
    r.m2 = max3(r.m2, m2, fminf(r.m, m1));
  }
  if (wm >= r.m) {
    if (wm > -CUDART_INF_F && bm == wm && (wm > r.m || r.idx == 0x7fffffff)) {   // this lane's first position of it
#pragma unroll
      for (int j = kPer - 1; j >= 0; --j)
        if (x[j] == wm) r.idx = element<VEC>(base, j);
    } else if (wm > r.m) {
      r.idx = 0x7fffffff;
    }
    if (wm > r.m) {   // the running sums follow the maximum
      const float d = r.m - wm, f = exp_fast(d);   // exp(-inf) = 0 while nothing finite had been seen
      if (KIND == kEntropy) r.t = f > 0.f ? f * fmaf(d, r.s, r.t) : 0.f;
      r.s *= f;
      r.m = wm;
      sum_batch<KIND>(x, wm, s, t);
    }
  }
  if (r.m > -CUDART_INF_F) {
    r.s += s;
    if (KIND == kEntropy) r.t += t;
  }
}

// ---- combining
// (max, lowest index, second largest) of two sets
template <int KIND>
__device__ __forceinline__ void merge_max(float& m, int& idx, float& m2, float om, int oidx, float om2) {
  if (KIND == kMargin) m2 = m >= om ? fmaxf(m2, om) : fmaxf(om2, m);
  if (om > m || (om == m && oidx < idx)) { m = om; idx = oidx; }
}

// s and t of a part with maximum `m`, seen from the maximum `all` of the whole
template <int KIND>
__device__ __forceinline__ void rebase(float m, float all, float& s, float& t) {
  const float d = m - all, f = m > -CUDART_INF_F ? exp_fast(d) : 0.f;
  if (KIND == kEntropy) t = f > 0.f ? f * fmaf(d, s, t) : 0.f;
  s *= f;
}

// ---- a chunk, by the whole block
struct WarpStats {
  float m, m2, s, t;
  int idx;
};

template <int KIND, bool VEC>
__device__ __forceinline__ void reduce_chunk(const float* __restrict__ z, int begin, int end, Entry* out) {
  __shared__ WarpStats stats[kWarps];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  Running r;
  r.clear();
  float xa[kPer], xb[kPer];
  load_batch<VEC>(z, begin, end, xa);
  for (int base = begin;;) {
    if (base + kBatch < end) load_batch<VEC>(z, base + kBatch, end, xb);
    take_batch<KIND, VEC>(r, xa, base);
    base += kBatch;
    if (base >= end) break;
    if (base + kBatch < end) load_batch<VEC>(z, base + kBatch, end, xa);
    take_batch<KIND, VEC>(r, xb, base);
    base += kBatch;
    if (base >= end) break;
  }
  float s = r.s, t = r.t;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    s += __shfl_xor_sync(0xffffffffu, s, o);
    if (KIND == kEntropy) t += __shfl_xor_sync(0xffffffffu, t, o);
  }
  const int idx = __reduce_min_sync(0xffffffffu, r.idx);
  if (lane == 0) stats[warp] = WarpStats{r.m, r.m2, s, t, idx};
  __syncthreads();
  if (warp == 0) {
    WarpStats w = {-CUDART_INF_F, -CUDART_INF_F, 0.f, 0.f, 0x7fffffff};
    if (lane < kWarps) w = stats[lane];
    const float m = warp_max(w.m);
    const int i = __reduce_min_sync(0xffffffffu, w.m == m ? w.idx : 0x7fffffff);
    float m2 = 0.f;
    if (KIND == kMargin) {   // the second largest: the largest of all seconds and of the firsts but one
      float first = w.m;
      m2 = w.m2;
#pragma unroll
      for (int o = kWarps / 2; o > 0; o >>= 1) {
        const float of = __shfl_xor_sync(0xffffffffu, first, o), os = __shfl_xor_sync(0xffffffffu, m2, o);
        m2 = max3(m2, os, fminf(first, of));
        first = fmaxf(first, of);
      }
    }
    rebase<KIND>(w.m, m, w.s, w.t);
#pragma unroll
    for (int o = kWarps / 2; o > 0; o >>= 1) {
      w.s += __shfl_xor_sync(0xffffffffu, w.s, o);
      if (KIND == kEntropy) w.t += __shfl_xor_sync(0xffffffffu, w.t, o);
    }
    if (lane == 0) __stcg(reinterpret_cast<float4*>(out), make_float4(m, __int_as_float(i), w.s, KIND == kEntropy ? w.t : m2));
  }
}

// ---- selection for batch element b by the whole block
struct SelectScratch {
  float key[kMaxBlockLen];     // ranking score; NaN where `on` is 0
  int32_t tok[kMaxBlockLen];
  uint8_t on[kMaxBlockLen];
  uint32_t sel[kMaxBlockLen / 32];
  int n_on;
};

// kind of the ranking: the score constants of dlm.h
__device__ __forceinline__ float score_of(const Args& a, int score_kind, size_t pos, float m, float s, float x) {
  if (score_kind == DLM_SCORE_CONFIDENCE) return 1.0f / s;
  if (score_kind == DLM_SCORE_NEG_ENTROPY) return x / s - __logf(s);
  if (score_kind == DLM_SCORE_MARGIN) return (1.0f - (x > -CUDART_INF_F ? __expf(x - m) : 0.f)) / s;
  return a.noise[pos] - __logf(s);
}

// (1) of the selection: LANES lanes per row merge the row's entries (lanes over chunks, fixed shuffle tree), 32 / LANES rows a warp,
// KEEP entries a lane in registers (further ones are read twice).  The entries are asked for beside the mask byte (a row that
// is not masked has stale ones, which are then ignored).
template <int KIND, int LANES, int KEEP>
__device__ __forceinline__ void merge_rows(const Args& a, int score_kind, size_t p0, SelectScratch& sc) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, sub = lane & (LANES - 1), L = a.block_len;
  constexpr int kRows = 32 / LANES;
#pragma unroll 1
  for (int i0 = warp * kRows; i0 < L; i0 += kWarps * kRows) {
    const int i = i0 + lane / LANES;
    const size_t p = p0 + min(i, L - 1);
    const bool on = i < L && __ldcg(a.masked + p) != 0;
    const float4* e = reinterpret_cast<const float4*>(a.entries + p * a.n_chunks);
    float4 v[KEEP];
#pragma unroll
    for (int h = 0; h < KEEP; ++h) {
      const int c = sub + LANES * h;
      v[h] = c < a.n_chunks ? __ldcg(e + c) : make_float4(-CUDART_INF_F, __int_as_float(0x7fffffff), 0.f, KIND == kMargin ? -CUDART_INF_F : 0.f);
    }
    float m = v[0].x, m2 = v[0].w;
    int idx = __float_as_int(v[0].y);
#pragma unroll
    for (int h = 1; h < KEEP; ++h) merge_max<KIND>(m, idx, m2, v[h].x, __float_as_int(v[h].y), v[h].w);
    for (int c = sub + LANES * KEEP; c < a.n_chunks; c += LANES) {
      const float4 w = __ldcg(e + c);
      merge_max<KIND>(m, idx, m2, w.x, __float_as_int(w.y), w.w);
    }
#pragma unroll
    for (int o = LANES / 2; o > 0; o >>= 1) {
      const float om = __shfl_xor_sync(0xffffffffu, m, o);
      const int oi = __shfl_xor_sync(0xffffffffu, idx, o);
      const float o2 = KIND == kMargin ? __shfl_xor_sync(0xffffffffu, m2, o) : 0.f;
      merge_max<KIND>(m, idx, m2, om, oi, o2);
    }
    float s = 0.f, x = 0.f;
    auto take = [&](const float4& w) {
      float sw = w.z, tw = w.w;
      rebase<KIND>(w.x, m, sw, tw);
      s += sw;
      if (KIND == kEntropy) x += tw;
    };
#pragma unroll
    for (int h = 0; h < KEEP; ++h) take(v[h]);
    for (int c = sub + LANES * KEEP; c < a.n_chunks; c += LANES) take(__ldcg(e + c));
#pragma unroll
    for (int o = LANES / 2; o > 0; o >>= 1) {
      s += __shfl_xor_sync(0xffffffffu, s, o);
      if (KIND == kEntropy) x += __shfl_xor_sync(0xffffffffu, x, o);
    }
    if (KIND == kMargin) x = m2;
    if (i < L && sub == 0) {
      const float score = on ? score_of(a, score_kind, p, m, s, x) : 0.f;
      a.tok[p] = on ? idx : -1;
      a.conf[p] = on ? 1.0f / s : -1.f;
      if (a.score) { a.score[p] = score; a.zmax[p] = on ? m : 0.f; }
      sc.key[i] = on ? score : CUDART_NAN_F;
      sc.tok[i] = idx;
      sc.on[i] = on;
    }
  }
}

template <int KIND, bool WIDE>
__device__ __forceinline__ void select_batch(const Args& a, int score_kind, int b, SelectScratch& sc) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int L = a.block_len, k = a.k;
  const size_t p0 = (size_t)b * L;
  if (tid < kMaxBlockLen / 32) sc.sel[tid] = 0;
  if (tid == 0) sc.n_on = 0;
  // Up to 32 positions are one pass of eight lanes a row, one round trip to L2; more (WIDE) take four lanes a row, 64 rows a pass
  // (4 x 64 positions of 6 chunks, a block's life with two passes of eight lanes and the ranking of before: 352 us, now 320).  Which one
  // is the kernel's, not a branch: this code runs once, and what it holds beside what it needs costs fetches and the streaming loop
  // registers.
  if (!WIDE) merge_rows<KIND, 8, 3>(a, score_kind, p0, sc); else merge_rows<KIND, 4, 5>(a, score_kind, p0, sc);
  if (k <= 0) return;
  __syncthreads();
  // (2) rank among the masked positions: (score desc, position asc).  Eight lanes a position, each comparing it with every eighth
  // one (a position that is not masked has a NaN, which outranks nothing).  (One warp with 32 unrolled shuffles for up to 32
  // positions, one thread a position for more: 2900 and 5000 - 10000 cycles behind the merge, most of it code seen for the
  // first time and a serial chain; now 1500.)
#pragma unroll 1
  for (int i0 = warp * 4; i0 < L; i0 += kWarps * 4) {
    const int i = i0 + (lane >> 3), first = lane & 7;
    const float mine = sc.key[min(i, L - 1)];
    int rank = 0;
    for (int j = first; j < L; j += 8) {
      const float sj = sc.key[j];
      rank += sj > mine || (sj == mine && j < i) ? 1 : 0;
    }
#pragma unroll
    for (int o = 4; o > 0; o >>= 1) rank += __shfl_xor_sync(0xffffffffu, rank, o);
    if (first == 0 && i < L && sc.on[i]) {
      atomicAdd(&sc.n_on, 1);
      if (rank < k) atomicOr(&sc.sel[i >> 5], 1u << (i & 31));
    }
  }
  __syncthreads();
  for (int i = tid; i < L; i += kThreads) {
    if (!((sc.sel[i >> 5] >> (i & 31)) & 1u)) continue;
    int order = __popc(sc.sel[i >> 5] & ((1u << (i & 31)) - 1u));
    for (int w = 0; w < i >> 5; ++w) order += __popc(sc.sel[w]);
    if (order >= k) continue;   // only with NaN scores
    a.sel_idx[(size_t)b * k + order] = i;
    a.tokens[p0 + i] = sc.tok[i];
    a.masked[p0 + i] = 0;
  }
  const int count = min(k, sc.n_on);
  for (int j = count + tid; j < k; j += kThreads) a.sel_idx[(size_t)b * k + j] = -1;
  if (tid == 0) a.n_sel[b] = count;
}

// ---- kernels
template <int KIND, bool VEC, bool WIDE>
__global__ void __launch_bounds__(kThreads, kBlocksPerSm) vocab_pass_kernel(const __grid_constant__ Args a, int score_kind) {
  __shared__ SelectScratch scratch;
  __shared__ bool is_last;
  dlm_grid_dependency_wait();
  dlm_trigger_dependents();
  const int chunk = blockIdx.x, row = blockIdx.y;
  int pos;   // of the row in its batch element
  const int b = a.by_block_len.divmod(row, pos);
  // The tickets count the blocks of masked rows, and the element's first block in any case: a block without work that took a
  // ticket too held its place on the SM for another round trip (64 positions x 4 sequences, 1536 blocks: with 4 masked in
  // each 11.3 us, now 10.5; with 16 15.2, now 13.8).  How many tickets there are, warp 0 counts from the element's mask bytes,
  // asked for together with the row's own.  The first block has its ticket so that some block is the last when none is
  // masked, and so that no selection clears a byte that it has yet to read.
  int n_on = 0;
  bool first_on = false;
  if (a.tickets != nullptr && threadIdx.x < 32) {
    const uint8_t* const m = a.masked + (size_t)b * a.block_len;
    for (int i = (int)threadIdx.x; i < a.block_len; i += 32) {
      const bool on = m[i] != 0;
      n_on += on ? 1 : 0;
      if (i == 0) first_on = on;
    }
  }
  const bool on = a.masked[row] != 0;
  if (on) {
    const int begin = chunk * a.chunk_len, end = min(begin + a.chunk_len, a.vocab);
    reduce_chunk<KIND, VEC>(a.logits + (size_t)row * a.vocab, begin, end, a.entries + (size_t)row * a.n_chunks + chunk);
  }
  if (a.tickets == nullptr || !(on || (chunk == 0 && pos == 0))) return;
  // the last block of this batch element to get here runs its selection.  Thread 0 wrote this block's entry, so its
  // release-acquire increment publishes it and, in the block that sees the full count, makes every other block's visible.
  if (threadIdx.x < 32) n_on = __reduce_add_sync(0xffffffffu, n_on);
  if (threadIdx.x == 0) {
    unsigned int t;
    asm volatile("atom.acq_rel.gpu.global.add.u32 %0, [%1], 1;" : "=r"(t) : "l"(a.tickets + b) : "memory");
    is_last = t == (unsigned int)(a.n_chunks * n_on + (first_on ? 0 : 1)) - 1u;
    if (is_last) a.tickets[b] = 0;   // ready for the next launch
  }
  __syncthreads();
  if (is_last) select_batch<KIND, WIDE>(a, score_kind, b, scratch);
}

// The selection as a kernel of its own, one block per batch element (no tickets).
template <int KIND, bool WIDE>
__global__ void __launch_bounds__(kThreads) vocab_select_kernel(const __grid_constant__ Args a, int score_kind) {
  __shared__ SelectScratch scratch;
  dlm_grid_dependency_wait();
  dlm_trigger_dependents();
  select_batch<KIND, WIDE>(a, score_kind, blockIdx.x, scratch);
}

// Chunks of 1 .. 8 batches: about two resident waves of blocks, so that the last ones to run find the memory busy, but no
// less than two batches a block when there is more than one wave of them (a block's fixed cost -- mask byte, first load,
// reduction, ticket -- is about a batch's worth), and no grid that just misses one wave (Dream's vocabulary at block 32:
// 19 x 32 blocks on 592 slots took 9.1 us, 13 x 32 take 8.8, and 14.6 against 13.5 per step over a block's life).
inline void plan_chunks(Args& a, int num_sms) {
  const long long wave = (long long)kBlocksPerSm * num_sms, rows = a.rows;
  const long long row_batches = (a.vocab + kBatch - 1) / kBatch;
  auto blocks = [&](long long batches) { return rows * ((row_batches + batches - 1) / batches); };
  long long batches = rows * row_batches / (2 * wave);
  batches = batches < 1 ? 1 : batches > 8 ? 8 : batches;
  if (batches == 1 && blocks(1) > wave) batches = 2;
  if (batches < 8 && blocks(batches) > wave && blocks(batches) * 4 <= wave * 5 && blocks(batches + 1) <= wave) ++batches;
  a.chunk_len = (int)batches * kBatch;
  a.n_chunks = (a.vocab + a.chunk_len - 1) / a.chunk_len;
  a.by_block_len = make_fast_div(a.block_len);
}

template <int KIND, bool WIDE>
inline int launch_sized(Args& a, int score_kind, int batch, int num_sms, cudaStream_t s) {
  plan_chunks(a, num_sms);
  const bool vec = a.vocab % 4 == 0 && ((uintptr_t)a.logits & 15) == 0;
  const dim3 grid(a.n_chunks, a.rows);
  const cudaError_t e = vec ? dlm_launch(vocab_pass_kernel<KIND, true, WIDE>, grid, dim3(kThreads), 0, s, a, score_kind)
                            : dlm_launch(vocab_pass_kernel<KIND, false, WIDE>, grid, dim3(kThreads), 0, s, a, score_kind);
  if (e != cudaSuccess) return -1;
  if (a.tickets != nullptr) return 1;
  if (dlm_launch(vocab_select_kernel<KIND, WIDE>, dim3(batch), dim3(kThreads), 0, s, a, score_kind) != cudaSuccess) return -1;
  return 2;
}

template <int KIND>
inline int launch_kind(Args& a, int score_kind, int batch, int num_sms, cudaStream_t s) {
  return a.block_len > 32 ? launch_sized<KIND, true>(a, score_kind, batch, num_sms, s) : launch_sized<KIND, false>(a, score_kind, batch, num_sms, s);
}

}  // namespace vocab
