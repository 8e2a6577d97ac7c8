// dlm_freecache_attn_step: attention of the active window over [cache rows ; fresh rows]
// (Sec. 3.2.1 "Windowed Re-computation"; Table 1 rows QK^T and Attention Score x Value;
// bidirectional: no causal mask).
//
// One work unit is (layer, batch element, KV head, chunk of up to 256 query rows): the g = Hq/Hkv
// query heads of a KV head, q_cap rows each, are cut into chunks of 256 rows = two 128-row M
// tiles that share every K/V tile (at the block sizes of the configs, g * q_cap <= 256: one chunk,
// K/V read from HBM once per KV head; larger windows re-read them per chunk, normally from L2;
// calls with few units use chunks of 128 rows or fewer, one M tile, to have more units to spread).
// Keys are loaded in tiles of 128 rows, first the visible cache rows, then the fresh rows, and
// processed in half-steps of 64.
//
// Block = 12 warps (three warpgroups), one block per SM (persistent):
//   warps 0-3   softmax of M tile 0 (thread = query row = TMEM lane)
//   warps 4-7   softmax of M tile 1
//   warp  8     TMA producer (one lane): Q once per segment, K and V tiles through two rings
//   warp  9/10  tcgen05.mma issuer of M tile 0 / 1 (one lane each): S = Q K^T into one of two
//               64-column score buffers in TMEM, two half-steps ahead of the softmax; then
//               O += P V with P read from TMEM (it overwrites S in place as packed bf16)
//   warp  11    publisher (one lane): makes a finished partial result visible device-wide and
//               bumps its unit's counter, so the softmax warps need not wait for that
// Online softmax in fp32 with base-2 exponentials; a half-step's scores sit in registers; O stays
// in TMEM and is rescaled only when a row's scores have outgrown the maximum in use by a lot.
//
// Scheduling.  Every (unit, key tile) pair is one item of a global list; block c takes the
// contiguous share [c*T/G, (c+1)*T/G) of it.  A share covers whole units (result written
// directly) and at most two partial units (unnormalised O, running max and sum written to the
// workspace).  A block walks its share from the end to the start, so the piece at the start of a
// share (the last piece of its unit) is the last thing the block computes; that block merges the
// unit: it waits for the counter the other pieces' blocks bump after publishing their partial
// results (they have lower block indices and computed those pieces first), then folds them into
// its own O, which is still in TMEM, in block order: the result is deterministic.  When the split
// would cost more than it saves (the host estimates both) units are dealt whole, round-robin.
// Calls with few units give each unit a team: a thread-block cluster that deals the unit's key tiles among its blocks and
// exchanges the partial results through the blocks' shared memory (team_share and below), or, where no such clusters fit and a unit's
// keys are many, a team that is no cluster and exchanges through L2 (WideArgs and below).  A cluster's block with one M tile
// has a chain of warps to spare, so it splits the keys: warps 0-3 and issuer 9 take the first 64 keys of every tile, warps 4-7
// and issuer 10 the others, each half with an O, maximum and sum of its own.
#include <cuda_bf16.h>
#include <math_constants.h>

#include "common.cuh"
#include "sm100_ptx.cuh"

namespace {

using namespace sm100;

constexpr int kThreads = 384;          // 3 warpgroups: two of softmax warps, one with the producer and the MMA issuers
constexpr int kTileKeys = 128;
constexpr int kPanelBytes = 128 * 128;   // one 64-element-wide panel of a 128-row tile
constexpr int kMaxBatch = 1024;
constexpr int kTmemCols = 512;
constexpr int kRegsSoftmax = 216;     // registers per thread of the softmax warpgroups after setmaxnreg.inc
constexpr int kRegsOther = 72;        // ... of the producer / MMA warpgroup after setmaxnreg.dec
constexpr int kMaxQCap = 4096;         // active rows per call
constexpr int kTeamMax = 16;              // most blocks of a team
constexpr int kMaxGrid = 256;          // blocks of the persistent grid (one per SM)
constexpr int kMaxStages = 8;          // barrier slots reserved per ring
constexpr int kBarrierBytes = 512;     // mbarriers of a block
constexpr int kFlagBytes = 64;         // abort / never flags, TMEM slot, merge flag
constexpr int kFoldBytes = 2 * 128 * 8;   // (running max, running sum) of every row of the two key halves

template <int D>
struct Geometry {
  static constexpr int kPanels = D / 64;
  static constexpr int kTileBytes = kPanels * kPanelBytes;      // one K tile, V tile or Q M-tile
  static constexpr int kStages = (D == 128) ? 2 : 4;            // ring depth of K and of V
  static constexpr uint32_t kColO = 0;                          // O[mt] at mt * D
  static constexpr uint32_t kColS = 2 * D;                      // S[mt] at 2D + mt * 128 (P aliases it)
};

// (The decoding of units and rows stands between a block's start and its first scores, in every role: with the compiler's
// division by run-time divisors it took 1.3 us when it was in the instruction cache and 3.5 - 5.7 us when another
// kernel had run in between; hence the FastDivs.)
struct AttnParams {
  const int32_t* cache_len;
  const int32_t* q_len;
  __nv_bfloat16* out;
  float* lse;
  float* ws_o;    // [2 * grid][n_mt][D/4][128][4]  partial unnormalised O: 4 columns of a row per 16-byte vector
  float* ws_ml;   // [2 * grid][n_mt][128][2]    partial (running max in log2 units, running sum)
  int nl, layer_begin, batch, n_kv_heads, n_q_heads, group, capacity, q_cap;
  int rows_total;  // group * q_cap: query rows per (layer, batch element, KV head)
  int n_rc;        // row chunks: rows_total cut into units of up to 256 rows (each re-reads the K/V tiles)
  int rows;        // query rows per unit = min(chunk_rows, rows_total)
  int chunk_rows;  // 256 (two M tiles share every K/V tile), 128 (one M tile per unit), or 96 or 64 (less than one; teams)
  int n_mt;        // M tiles per unit (1 or 2)
  int fresh_box;   // rows per TMA box of the fresh K/V tensors = min(128, q_cap)
  int whole_units; // 1: deal whole units round-robin, no partials
  int team;        // > 1 (with whole_units): blocks [u * team, (u + 1) * team) share unit u, key tiles dealt by rank;
                   // every block then reduces its share of the unit's outputs over all the team's pieces
  int smem_bytes;           // dynamic shared memory of the launch
  FastDiv by_batch, by_rc, by_kv_heads, by_q_cap, by_team, by_live;
  int hint_len;             // cached rows to expect (only a guess)
  float scale_log2;
  int* status;
  unsigned int* tickets;   // one zero-initialised counter per unit: pieces finished
};

// Per-block scheduling tables (in the block's dynamic shared memory, sized by batch).
struct Sched {
  int* prefix;    // [batch + 1]  prefix[b] = tiles of batch elements < b; prefix[batch] = sum
  int* lc;        // [batch]      clamped cache_len
  int* lq;        // [batch]      clamped q_len
  int share, share_rem, n_cta;   // split mode: total items = share * n_cta + share_rem
  // split mode: block c owns items [lo(c), lo(c + 1)), lo(c) = floor(total * c / n_cta)
  __device__ __forceinline__ int lo(int c) const { return share * c + (share_rem * c) / n_cta; }
};
__host__ __device__ inline int sched_ints(int batch) { return 3 * (batch + 1); }

struct Segment {
  int lc_layer, b, kvh, rc;   // unit: layer within the call, batch element, KV head, row chunk
  int Lc, Lq, n_ct, T;    // lengths, cache tiles, total tiles of the unit
  int t_begin, t_end;     // tile range of this segment
  int slot;               // partial slot; -1 when the segment is the whole unit
  int merger;             // partial segment holding the unit's last tile: this block merges the unit
};

__device__ __forceinline__ int tiles_of(int Lc, int Lq, int fresh_box) {
  if (Lq <= 0) return 0;
  return (Lc + kTileKeys - 1) / kTileKeys + (Lq + fresh_box - 1) / fresh_box;
}

// Launches in which a block has one unit at most (kSingle: whole units on as many SMs, and teams): which one does not depend on
// the lengths, so it is decoded while the kernel before is still running; of the lengths a block needs those of its unit's
// batch element only, and every role reads them for itself: no tables and no barrier behind the wait for the kernel before.
// They are kernels of their own because what stands in front of the first copies is code that is not in the instruction
// cache (another kernel has run in between): with all schedules in one kernel and the tables, a one-layer call of Dream issued
// its first K copy 5360 cycles after that wait, now 2260.  Us a call, before -> now: one sequence 10.6 -> 9.3, window of 256
// rows 18.2 -> 16.8, 8 sequences 19.2 -> 17.2, an LLaDA layer (whole units) 29.5 -> 28.0, 28 layers in one call 26.1 -> 25.4 back to back.
__device__ __forceinline__ void decode_single(const AttnParams& p, Segment& g) {
  const int unit = p.team > 1 ? p.by_team.div(blockIdx.x) : (int)blockIdx.x;
  const int grp = p.by_batch.divmod(unit, g.b);
  g.lc_layer = p.by_kv_heads.divmod(p.by_rc.divmod(grp, g.rc), g.kvh);
}
__device__ __forceinline__ void set_single_lengths(const AttnParams& p, Segment& g, int Lc, int Lq) {
  g.Lc = Lc;
  g.Lq = Lq;
  g.n_ct = (Lc + kTileKeys - 1) / kTileKeys;
  g.T = tiles_of(Lc, Lq, p.fresh_box);
  g.t_begin = 0;
  g.t_end = g.T;
  if (p.team > 1) {   // this block's share of the unit's key tiles; the launch has one team per unit
    const int rank = (int)blockIdx.x - p.by_team.div(blockIdx.x) * p.team;
    g.t_begin = p.by_team.div(g.T * rank);
    g.t_end = p.by_team.div(g.T * (rank + 1));
  }
}

// Walks the segments of block `cta`.  Identical in every role, so the roles agree on the
// sequence without communicating.  Item counts fit 32 bits (the host refuses larger launches).
template <bool kSingle>
struct SegmentWalker {
  const AttnParams& p;
  const Sched& s;
  int end, range_begin;   // split mode: items [range_begin, end) are still to do
  int unit, n_units;
  __device__ __forceinline__ SegmentWalker(const AttnParams& p_, const Sched& s_, int cta) : p(p_), s(s_) {
    if (kSingle) {
      unit = end = range_begin = 0;
      n_units = 1;
      return;
    }
    n_units = p.nl * p.n_kv_heads * p.n_rc * p.batch;
    if (p.whole_units) {
      unit = cta;
      end = range_begin = 0;
    } else {
      range_begin = cta < s.n_cta ? s.lo(cta) : 0;
      end = cta < s.n_cta ? s.lo(cta + 1) : 0;
      unit = 0;
    }
  }
  __device__ __forceinline__ bool next(Segment& g, int n_cta) {
    if (kSingle) {   // g holds the block's unit already
      const bool more = unit < n_units;
      unit = n_units;
      return more;
    }
    if (p.whole_units) {
      if (unit >= n_units) return false;
      const int grp = p.by_batch.divmod(unit, g.b);
      g.lc_layer = p.by_kv_heads.divmod(p.by_rc.divmod(grp, g.rc), g.kvh);
      g.Lc = s.lc[g.b];
      g.Lq = s.lq[g.b];
      g.T = s.prefix[g.b + 1] - s.prefix[g.b];
      g.n_ct = (g.Lc + kTileKeys - 1) / kTileKeys;
      g.t_begin = 0;
      g.t_end = g.T;
      g.slot = -1;
      g.merger = 0;
      unit += n_cta;
      return true;
    }
    // split mode: from the end of the share towards its start
    if (end <= range_begin) return false;
    const int sum = s.prefix[p.batch];
    const int item = end - 1;
    // the divisor is made of lengths, so not known on the host: a float estimate, exact division where it is off
    int grp = (int)__fdividef((float)item, (float)sum);
    int rem = item - grp * sum;
    if (rem < 0 || rem >= sum) {
      grp = item / sum;
      rem = item - grp * sum;
    }
    int b = 0;
    while (s.prefix[b + 1] <= rem) ++b;   // batch is small; units with zero tiles are skipped
    const int unit_start = grp * sum + s.prefix[b];
    g.b = b;
    g.lc_layer = p.by_kv_heads.divmod(p.by_rc.divmod(grp, g.rc), g.kvh);
    g.Lc = s.lc[b];
    g.Lq = s.lq[b];
    g.T = s.prefix[b + 1] - s.prefix[b];
    g.n_ct = (g.Lc + kTileKeys - 1) / kTileKeys;
    const int seg_lo = unit_start > range_begin ? unit_start : range_begin;
    g.t_begin = seg_lo - unit_start;
    g.t_end = end - unit_start;
    const bool whole = g.t_begin == 0 && g.t_end == g.T;
    g.slot = whole ? -1 : (seg_lo == range_begin ? 2 * (int)blockIdx.x : 2 * (int)blockIdx.x + 1);
    g.merger = (!whole && g.t_end == g.T) ? 1 : 0;
    end = seg_lo;
    return true;
  }
};

// Valid keys of tile t of a unit.
__device__ __forceinline__ int tile_valid(const Segment& g, int t, int fresh_box) {
  if (t < g.n_ct) return min(kTileKeys, g.Lc - t * kTileKeys);
  return min(fresh_box, g.Lq - (t - g.n_ct) * fresh_box);
}

// The blocks whose shares overlap the unit of segment g (this block is one of them), and where
// each of them left its partial result.
struct UnitPieces {
  const Sched& s;
  int u0, u1, c_first, c_last;
  __device__ UnitPieces(const AttnParams& p, const Sched& s_, const Segment& g, int cta) : s(s_) {
    const int sum = s.prefix[p.batch];
    u0 = ((g.lc_layer * p.n_kv_heads + g.kvh) * p.n_rc + g.rc) * sum + s.prefix[g.b];
    u1 = u0 + g.T;
    c_first = c_last = cta;
    while (s.lo(c_first) > u0) --c_first;
    while (s.lo(c_last + 1) < u1) ++c_last;
  }
  // slot of the piece computed by block c (c_first <= c <= c_last): the block's first segment
  // if the piece starts where the block's share starts, else its second one
  __device__ __forceinline__ int slot_of(int c) const { return s.lo(c) >= u0 ? 2 * c : 2 * c + 1; }
};

// Waits until the counter at `addr` reaches `target` (acquire, device scope).  Bounded like the
// mbarrier waits: gives up after the same wall-time limit or when the block is aborting.
__device__ __forceinline__ bool wait_counter(const unsigned int* addr, unsigned int target, volatile int* abort_flag,
                                             uint64_t limit_ns) {
  const uint64_t t0 = global_timer_ns();
  for (uint32_t spin = 1;; ++spin) {
    unsigned int v;
    asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(addr) : "memory");
    if (v >= target) return true;
    if ((spin & 15u) == 0u) {
      if (*abort_flag) return false;
      if (global_timer_ns() - t0 > limit_ns) {
        *abort_flag = 1;
        return false;
      }
    }
  }
}

__device__ __forceinline__ uint32_t pack_bf16(float a, float b) {
  const __nv_bfloat162 h = __floats2bfloat162_rn(a, b);
  return *reinterpret_cast<const uint32_t*>(&h);
}

// 32 columns of a row's O at `t`; with the keys split, the weighted sum of both halves' (at t and t2, which
// lie D columns apart).  (A half without keys holds no O: then t2 is the other half's again and the weights are halves of its.)
template <bool kKeys>
__device__ __forceinline__ void read_o(uint32_t t, uint32_t t2, const float (&w)[2], uint32_t (&v)[32]) {
  tmem_ld32(t, v);
  if (!kKeys) {
    tmem_ld_wait();
    return;
  }
  uint32_t u[32];
  tmem_ld32(t2, u);
  tmem_ld_wait();
  const uint64_t w0 = pack2(w[0], w[0]), w1 = pack2(w[1], w[1]);
#pragma unroll
  for (int j = 0; j < 32; j += 2) {
    const uint64_t a = pack2(__uint_as_float(v[j]), __uint_as_float(v[j + 1])), b = pack2(__uint_as_float(u[j]), __uint_as_float(u[j + 1]));
    float x, y;
    unpack2(fma2(w1, b, mul2(w0, a)), x, y);
    v[j] = __float_as_uint(x);
    v[j + 1] = __float_as_uint(y);
  }
}

// Team schedule: what the blocks of a team, which are a thread-block cluster, do after their shares of the key tiles.  A block's
// piece -- unnormalised O, and (m, l), for every row -- is laid out in its own shared memory, over the rings, which are read no
// more: [warp of 32 rows][head_dim / 4][32] 16-byte vectors, R the unit's rows in whole warps.  Each block finishes some of the unit's output
// columns, in units of 8, over all the team's pieces: bulk copies bring it those columns of the others' pieces and their (m, l),
// counted in on a barrier of its own.
//   What bounds it is neither bytes nor the shared memory network but the number of instructions, run once and partly fetched for
// the first time: so it is short and in loops, what can be made ready before the last product is, and the reduction is spread over
// all eight softmax warps.  Cycles from the last product to the end of the block, 64 rows in teams of 4 in a step: straight from
// registers into the others' shared memory, 1500 unrolled instructions, 7900 (2450 to send, 1400 for the weights of 4 pieces, 1400 to
// reduce, 200 of waiting; in loops 6000: such stores move 16 - 18 bytes a cycle); bulk copies by one lane of the publisher 6100; by every
// warp as soon as its rows are laid out 5500.  Through L2 with counters, as before, a block of a team of 9 took 9800.
//   One-layer calls, before (through L2, keys not split) -> now, us: 256 active rows of Dream 16.4 -> 12.9, 8 sequences 16.9 -> 13.2, 4 13.2 -> 11.2,
// one 8.95 -> 8.55 (64 blocks instead of 144), 300 cached rows 7.7 -> 7.15, the tiny configuration 6.85 -> 6.65, 2 x 8 heads of 100 rows 10.6 ->
// 9.5, 4 sequences of 8 KV heads at 2000 rows 14.7 -> 13.4.  The split of the keys alone, with the exchange through L2: 8 sequences 16.9 ->
// 15.9, 4 13.2 -> 12.7, 64 rows and fewer equal (it is not used for whole units: an LLaDA layer, 64 rows a unit, is bound by HBM and took
// 0.2 us more).
__host__ __device__ inline int team_share(int head_dim, int team) { return (head_dim / 8 + team - 1) / team; }   // largest share, units
__host__ __device__ inline int team_bytes(int head_dim, int team, int rows) {
  return (team - 1) * team_share(head_dim, team) * rows * 32 + team * rows * 8;
}
struct TeamShape {
  FastDiv by_team;
  int team, rank, R, share;
  uint32_t sm_piece;     // the block's own piece
  uint32_t sm_x;         // the others': [team - 1][R / 32][share][2][32] vectors
  uint32_t sm_ml;        // [team][R] (m, l), the block's own last
  __device__ __forceinline__ int lo(int D, int r) const { return by_team.div(D / 8 * r); }   // first unit of rank r
};

// What the others will send: O those that have tiles (dealt so that no block has two before each has one), (m, l) all.
template <int D>
__device__ __forceinline__ void team_expect(const TeamShape& p, uint32_t bar_team, int T, bool has_tiles) {
  const int mine = p.lo(D, p.rank + 1) - p.lo(D, p.rank), with_tiles = min(T, p.team) - (has_tiles ? 1 : 0);
  mbar_expect_tx(bar_team, (uint32_t)(p.R * (with_tiles * mine * 32 + (p.team - 1) * 8)));
}

// What lane d of a warp sends block d of the warp's 32 rows (number `w` of the unit): the units that block finishes of [u0, u1), and,
// for every n_parts-th block from `part` on, the rows' (m, l).  Made ready while the block's first keys are on their way.
struct TeamParcel {
  uint32_t src, dst, bytes, ml_dst, bar;   // bytes, ml_dst: 0 for none
};
template <int D>
__device__ __forceinline__ TeamParcel team_parcel(const TeamShape& p, uint32_t bar_team, int w, int u0, int u1, int part, int n_parts) {
  const int d = threadIdx.x & 31;
  TeamParcel c = {0, 0, 0, 0, 0};
  if (d < p.team && d != p.rank) {
    const int lo_d = p.lo(D, d), lo = max(lo_d, u0), n = min(p.lo(D, d + 1), u1) - lo, slot = p.rank < d ? p.rank : p.rank - 1;
    c.src = p.sm_piece + (w * (D / 8) + lo) * 1024;
    c.dst = map_shared_rank(p.sm_x, d) + ((slot * (p.R >> 5) + w) * p.share + lo - lo_d) * 1024;
    c.bytes = n > 0 ? n * 1024 : 0;
    c.ml_dst = d % n_parts == part ? map_shared_rank(p.sm_ml, d) + (slot * p.R + w * 32) * 8 : 0;
    c.bar = map_shared_rank(bar_team, d);
  }
  return c;
}

// Softmax threads, all 256: row `row` of the unit and every n_groups-th unit of the block's columns from the group's on, two units
// and two pieces at a time (a unit or piece beyond the last is the last again, not stored or without weight).
template <int D>
__device__ __forceinline__ void team_reduce(const TeamShape& p, int row, int group, int n_groups, bool real, bool active, __nv_bfloat16* out, float* lse) {
  const int lo = p.lo(D, p.rank), n = p.lo(D, p.rank + 1) - lo, last = p.team - 1;
  const uint32_t at = (uint32_t)((row & 31) * 16), ml = p.sm_ml + row * 8, ml_step = p.R * 8, x_step = p.share * p.R * 32;
  const uint32_t x0 = p.sm_x + (uint32_t)((row >> 5) * p.share) * 1024 + at, own = p.sm_piece + (uint32_t)((row >> 5) * (D / 8) + lo) * 1024 + at;
  float m_all = -CUDART_INF_F;
#pragma unroll 4
  for (int s = 0; s <= last; ++s) m_all = fmaxf(m_all, ld_shared_f2(ml + s * ml_step).x);
#pragma unroll 1
  for (int u = group; u < n; u += 2 * n_groups) {
    const int u1 = min(u + n_groups, n - 1);
    float acc[2][8] = {}, l_all = 0.f;
#pragma unroll 1
    for (int s = 0; s <= last; s += 2) {
      float2 a[2];
      float4 x[2][2], y[2][2];
#pragma unroll
      for (int j = 0; j < 2; ++j) {
        const int sj = min(s + j, last);
        const uint32_t from = sj == last ? own : x0 + sj * x_step;
        a[j] = ld_shared_f2(ml + sj * ml_step);
        if (s + j > last) a[j].y = 0.f;
        x[j][0] = ld_shared_f4(from + u * 1024);
        y[j][0] = ld_shared_f4(from + u * 1024 + 512);
        x[j][1] = ld_shared_f4(from + u1 * 1024);
        y[j][1] = ld_shared_f4(from + u1 * 1024 + 512);
      }
#pragma unroll
      for (int j = 0; j < 2; ++j) {
        if (!__any_sync(0xffffffffu, a[j].y != 0.f)) continue;   // a piece without key tiles holds no O
        const float w = ex2_approx(a[j].x - m_all);
        l_all = fmaf(w, a[j].y, l_all);
#pragma unroll
        for (int i = 0; i < 2; ++i) {
          acc[i][0] = fmaf(w, x[j][i].x, acc[i][0]); acc[i][1] = fmaf(w, x[j][i].y, acc[i][1]);
          acc[i][2] = fmaf(w, x[j][i].z, acc[i][2]); acc[i][3] = fmaf(w, x[j][i].w, acc[i][3]);
          acc[i][4] = fmaf(w, y[j][i].x, acc[i][4]); acc[i][5] = fmaf(w, y[j][i].y, acc[i][5]);
          acc[i][6] = fmaf(w, y[j][i].z, acc[i][6]); acc[i][7] = fmaf(w, y[j][i].w, acc[i][7]);
        }
      }
    }
    const float inv = 1.f / l_all;
#pragma unroll
    for (int i = 0; i < 2; ++i) {
      uint32_t h[4];
#pragma unroll
      for (int j = 0; j < 4; ++j) h[j] = active ? pack_bf16(acc[i][2 * j] * inv, acc[i][2 * j + 1] * inv) : 0u;
      if (real) *reinterpret_cast<uint4*>(out + (lo + (i ? u1 : u)) * 8) = make_uint4(h[0], h[1], h[2], h[3]);
    }
    if (lo + u == 0 && real && lse) *lse = active ? (m_all + lg2_approx(l_all)) * 0.6931471805599453f : -CUDART_INF_F;
  }
}

// Teams that are no cluster: the exchange goes through L2.  The device runs 33 clusters of 4 blocks at a time, 15 of 9, 7 of 16, on 148
// SMs, and a cluster's blocks start together, once all of its SMs are free; two M tiles of heads of 128 have no room for the pieces
// in shared memory.  Where units are few and long, more blocks a unit are worth more than the shorter exchange.  Us between
// projections, the best other schedule -> this one: 2 layers of 3 sequences of 8 heads (2 KV heads) at 10000 cached rows 29.0 -> 24.5, 200 active
// rows of 2 sequences of Dream at 4000 46.8 -> 40.9, 8 layers of one sequence at 10000 58.2 -> 55.9.
// What a block of such a team works on after its share of the key tiles.  The team's pieces lie
// in the workspace as [rank][M tile][head_dim / 4][R rows] 16-byte vectors (4 columns of a row) and
// [rank][M tile][R rows] (m, l) pairs, R the unit's rows in an M tile rounded up to 32, 64 or 128; the unit's n_mt * head_dim / 4 * R
// output vectors are dealt to the ranks in that storage order, rank r reducing vectors [lo, hi) over all pieces.
// Everything the exchange needs, decoded by the caller and handed over by value.
struct WideArgs {
  __nv_bfloat16* out;
  float* lse;
  float* ws_o;
  float* ws_ml;
  unsigned int* arrive;        // the unit's two counters: blocks that have stored their piece ...
  unsigned int* depart;        // ... and blocks that are past their wait for the first
  size_t piece0;               // index of the team's first piece
  size_t qrow0;                // output row of the KV head's first query row
  FastDiv by_q_cap;
  int team, n_mt, rows, rows_total, rank, Lq;
  bool has_keys;
  int r0, lo, hi;              // r0: the row chunk's first row among the KV head's rows
  int r_shift;                 // log2 R
  __device__ __forceinline__ WideArgs(const AttnParams& p, const Segment& g, int D)
      : out(p.out), lse(p.lse), ws_o(p.ws_o), ws_ml(p.ws_ml), by_q_cap(p.by_q_cap), team(p.team), n_mt(p.n_mt), rows(p.rows),
        rows_total(p.rows_total), Lq(g.Lq), has_keys(g.T > 0) {
    const int unit = p.by_team.divmod(blockIdx.x, rank);
    r0 = g.rc * p.chunk_rows;
    qrow0 = (((size_t)g.lc_layer * p.batch + g.b) * p.n_q_heads + (size_t)g.kvh * p.group) * p.q_cap;
    arrive = p.tickets + unit;
    depart = arrive + kDlmMaxSplitUnits / 2;
    r_shift = p.rows > 64 ? 7 : p.rows > 32 ? 6 : 5;
    const int n_vec = (p.n_mt * (D / 4)) << r_shift;
    lo = p.by_team.div(n_vec * rank);          // n_vec <= 8192, team <= 16
    hi = p.by_team.div(n_vec * (rank + 1));
    piece0 = (size_t)unit * p.team * p.n_mt;
  }
};

// The two halves of the team schedule's exchange are functions of their own, not inlined: they run once per
// launch, and inlined they changed the register allocation of the kernel's main loops (measured: 2 - 3 % on the
// layer-batched calls, when all schedules were one kernel).
//
// Publisher warp, one thread: once every softmax thread of this block has stored its row of the block's piece
// (bar_pub), count the block in the unit's arrival counter; when the whole team has arrived, let the softmax threads go on
// (bar_team = bar_pub + 8).
template <bool kNoWait>
__device__ __noinline__ void wide_publish(const WideArgs p, uint32_t bar_pub, volatile int* abort_ptr) {
  constexpr uint64_t kLimit = kNoWait ? 0ull : kWaitLimitNs;
  if (!p.has_keys || !mbar_wait_limit(bar_pub, 0, abort_ptr, kLimit)) return;
  __threadfence();
  atomicAdd(p.arrive, 1u);
  if (!wait_counter(p.arrive, (unsigned int)p.team, abort_ptr, kLimit)) return;
  mbar_arrive(bar_pub + 8);
  // every block of the team is past its wait on the arrival counter when the last one gets here: the last
  // one clears both counters for the next launch
  if (atomicAdd(p.depart, 1u) == (unsigned int)p.team - 1u) {
    *p.arrive = 0;
    *p.depart = 0;
  }
}

// Softmax threads (all 256 of the block, whole warps).  Live ones store their row of the block's piece --
// unnormalised O from TMEM at t_o if the block had key tiles, and (m, l), which is (-inf, 0) if it had none
// (that piece's O is then never read).  Then all wait for the team and reduce this block's share of
// the unit's output vectors over the C pieces, in rank order.  A thread's vectors lie in one row of an M tile, whose weights it takes
// once, and what it needs of up to kMax pieces it asks L2 for at once: one round trip for the weights and the first vectors, one
// for each further pair or single vector.  (Bulk copies of the shares into shared memory, 2 C of them issued by one lane, took 2400 -
// 2900 cycles until they had landed, and the reduction from there 1400 - 6000.)  Returns false when a wait was given up.
template <int D, int kMax>
__device__ __forceinline__ void wide_reduce(const WideArgs& p) {
  constexpr int kVec = 16 / kMax;             // vectors in flight
  const int kVecs = (D / 4) << p.r_shift, R = 1 << p.r_shift;   // vectors of one M tile's piece
  const int tid = threadIdx.x, C = p.team;
  const int row = (p.lo + tid) & (R - 1);     // 256 is a multiple of R
  const float4* const o = reinterpret_cast<const float4*>(p.ws_o) + ((p.piece0 * (D / 4)) << p.r_shift);
  const size_t piece = (size_t)kVecs * p.n_mt;
  int mt = -1;
  bool real = false, active = false;
  float w[kMax], m_all = 0.f, l_all = 0.f, inv = 0.f;
  size_t qrow = 0;
  for (int i = p.lo + tid; i < p.hi; i += 256 * kVec) {
    float4 x[kVec][kMax];
#pragma unroll
    for (int u = 0; u < kVec; ++u)
#pragma unroll
      for (int c = 0; c < kMax; ++c)
        if (c < C && i + 256 * u < p.hi) x[u][c] = __ldcg(o + c * piece + i + 256 * u);
#pragma unroll
    for (int u = 0; u < kVec; ++u) {
      const int iu = i + 256 * u, mt_i = iu >= kVecs ? 1 : 0, qd = (iu - mt_i * kVecs) >> p.r_shift;
      if (iu >= p.hi) break;
      if (mt_i != mt) {
        mt = mt_i;
        const int r_unit = mt * 128 + row, r_kv = p.r0 + r_unit;
        real = r_unit < ((p.rows + 31) & ~31) && r_kv < p.rows_total;
        qrow = p.qrow0 + r_kv;                // rows of a KV head's query heads lie one after the other
        int ir;
        p.by_q_cap.divmod(r_kv, ir);
        active = ir < p.Lq;
        const float2* const a_ml = reinterpret_cast<const float2*>(p.ws_ml) + ((p.piece0 + mt) << p.r_shift) + row;
        float2 ml[kMax];
#pragma unroll
        for (int c = 0; c < kMax; ++c) ml[c] = c < C && real ? __ldcg(a_ml + (((size_t)c * p.n_mt) << p.r_shift)) : make_float2(-CUDART_INF_F, 0.f);
        m_all = -CUDART_INF_F;
#pragma unroll
        for (int c = 0; c < kMax; ++c)
          m_all = fmaxf(m_all, ml[c].x);
        l_all = 0.f;
#pragma unroll
        for (int c = 0; c < kMax; ++c) {
          w[c] = ml[c].y != 0.f ? ex2_approx(ml[c].x - m_all) : 0.f;
          l_all = fmaf(w[c], ml[c].y, l_all);
        }
        inv = active ? 1.f / l_all : 0.f;
      }
      if (!real) continue;
      float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
      for (int c = 0; c < kMax; ++c) {
        if (c < C && w[c] != 0.f) {           // a piece without keys holds no O
          acc.x = fmaf(w[c], x[u][c].x, acc.x);
          acc.y = fmaf(w[c], x[u][c].y, acc.y);
          acc.z = fmaf(w[c], x[u][c].z, acc.z);
          acc.w = fmaf(w[c], x[u][c].w, acc.w);
        }
      }
      const __nv_bfloat162 h0 = __floats2bfloat162_rn(active ? acc.x * inv : 0.f, active ? acc.y * inv : 0.f);
      const __nv_bfloat162 h1 = __floats2bfloat162_rn(active ? acc.z * inv : 0.f, active ? acc.w * inv : 0.f);
      *reinterpret_cast<uint2*>(p.out + qrow * D + qd * 4) =
          make_uint2(*reinterpret_cast<const uint32_t*>(&h0), *reinterpret_cast<const uint32_t*>(&h1));
      if (qd == 0 && p.lse) p.lse[qrow] = active ? (m_all + lg2_approx(l_all)) * 0.6931471805599453f : -CUDART_INF_F;
    }
  }
}

template <int D, bool kNoWait>
__device__ __noinline__ bool wide_exchange(const WideArgs p, uint32_t bar_pub, volatile int* abort_ptr, bool live, uint32_t t_o,
                                           bool has_tiles, float m_used, float l_run) {
  constexpr uint64_t kLimit = kNoWait ? 0ull : kWaitLimitNs;
  const int tid = threadIdx.x, mt = tid >> 7, row = tid & 127;
  if (live) {
    const size_t mine = p.piece0 + (size_t)p.rank * p.n_mt + mt;
    if (has_tiles) {
      float4* po = reinterpret_cast<float4*>(p.ws_o) + ((mine * (D / 4)) << p.r_shift) + row;
      uint32_t v[32];
#pragma unroll 1
      for (int c = 0; c < D / 32; ++c) {
        tmem_ld32(t_o + c * 32, v);
        tmem_ld_wait();
#pragma unroll
        for (int j = 0; j < 8; ++j)
          __stcg(po + ((c * 8 + j) << p.r_shift), make_float4(__uint_as_float(v[4 * j]), __uint_as_float(v[4 * j + 1]),
                                                              __uint_as_float(v[4 * j + 2]), __uint_as_float(v[4 * j + 3])));
      }
    }
    __stcg(reinterpret_cast<float2*>(p.ws_ml) + (mine << p.r_shift) + row, make_float2(m_used, l_run));
    // no fence here: the arrival below orders the stores before the publisher's wait (block scope), and the
    // publisher's fence before it counts the block in carries them to device scope
    mbar_arrive(bar_pub);
  }
  if (!mbar_wait_warp(bar_pub + 8, 0, abort_ptr, kLimit)) return false;
  if (p.team <= 8) wide_reduce<D, 8>(p); else wide_reduce<D, 16>(p);
  __syncwarp();
  return true;
}

// A key tile is processed in half-steps of up to 64 keys.  Each M tile has two 64-column score
// buffers in TMEM used alternately, so the scores of the half-step after next are computed by the
// tensor pipe while the softmax warps work on the current one: they never wait for scores in the
// steady state.  All roles enumerate the half-steps of a segment with this iterator.
constexpr int kHalfKeys = 64;
struct HalfStep {
  int t;          // key tile
  int k0;         // first key of the half-step within the tile (0 or 64)
  int nkeys;      // valid keys (1..64)
  bool first_of_tile, last_of_tile;
};
// In kernels that split the keys (kKeys) chain h has half-step h of every tile that reaches it.
template <bool kKeys>
struct HalfIter {
  const Segment& g;
  int fresh_box, t, h;
  __device__ HalfIter(const Segment& g_, int fresh_box_, int chain) : g(g_), fresh_box(fresh_box_), t(g_.t_begin), h(kKeys ? chain : 0) {}
  // kKeys: the chain has nothing in tile t
  __device__ __forceinline__ bool skips() const { return kKeys && h != 0 && t < g.t_end && tile_valid(g, t, fresh_box) <= kHalfKeys; }
  __device__ __forceinline__ bool get(HalfStep& s) const {
    if (t >= g.t_end) return false;
    const int valid = tile_valid(g, t, fresh_box);
    s.t = t;
    s.k0 = h * kHalfKeys;
    s.nkeys = min(kHalfKeys, valid - s.k0);
    s.first_of_tile = kKeys || (h == 0);
    s.last_of_tile = kKeys || (h == 1) || valid <= kHalfKeys;
    return true;
  }
  __device__ __forceinline__ void advance(const HalfStep& s) {
    if (kKeys) { ++t; return; }
    if (s.last_of_tile) { ++t; h = 0; } else { h = 1; }
  }
};

// Softmax of one half-step for the query row held by this thread (S row in TMEM -> P row in TMEM).
// O is rescaled only when the scores have outgrown the maximum in use by a lot: until then P is
// formed against the older, smaller maximum and may exceed 1 by a few powers of two, which bf16
// and the fp32 accumulators hold just as well; the final division by the row sum, taken against
// the same maximum, cancels it.  Ragged half-steps compare maxima (kRescaleThreshold, log2 units);
// full ones look at the row sum (kSumLimit).
constexpr float kRescaleThreshold = 8.0f;

// Rare path shared by both kinds of half-step: some row of the warp outgrew its maximum by more
// than the threshold, so the warp's O rows in TMEM are rescaled (rows that did not grow keep
// factor 1).  The P V product of the previous half-step may still be running: wait for it first.
template <int D>
__device__ __noinline__ bool rescale_o(uint32_t t_o, bool grow, float m_new, float& m_used, float& l_run,
                                       uint32_t bar_pv_done, uint32_t parity, volatile int* abort_ptr) {
  const bool ok = __all_sync(0xffffffffu, mbar_wait(bar_pv_done, parity, abort_ptr)) != 0;
  if (!ok) return false;
  tc_fence_after_sync();
  const float alpha = grow ? ex2_approx(m_used - m_new) : 1.0f;
  uint32_t v[32];
#pragma unroll 1
  for (int c = 0; c < D / 32; ++c) {
    tmem_ld32(t_o + c * 32, v);
    tmem_ld_wait();
#pragma unroll
    for (int j = 0; j < 32; ++j) v[j] = __float_as_uint(__uint_as_float(v[j]) * alpha);
    tmem_st32(t_o + c * 32, v);
  }
  tmem_st_wait();
  l_run *= alpha;
  if (grow) m_used = m_new;
  return true;
}

// Full half-step (64 valid keys): the score row sits in registers, so TMEM is read once and with a
// single wait.  Only the first half-step of a segment takes the row maximum before the
// exponentials; later ones form P against the maximum in use and look at the row sum afterwards:
// a sum above kSumLimit means some score outgrew that maximum by a lot, and only then (rare)
// is the maximum taken, O rescaled and P formed again.  The maximum pass, half-rate ALU work
// that both softmax groups of an SMSP would do at the same time, is gone from the steady state.
constexpr float kSumLimit = 1024.0f;   // 64 keys: some P is then above 16, and none was above 1024 before

template <int D>
__device__ __forceinline__ float row_max64(const uint32_t (&s)[64]) {
  float mx[8];   // independent chains: the maximum is latency-bound otherwise
#pragma unroll
  for (int c = 0; c < 8; ++c) mx[c] = __uint_as_float(s[c]);
#pragma unroll
  for (int j = 8; j < 64; j += 8) {
#pragma unroll
    for (int c = 0; c < 8; ++c) mx[c] = fmaxf(mx[c], __uint_as_float(s[j + c]));
  }
  return fmaxf(fmaxf(fmaxf(mx[0], mx[1]), fmaxf(mx[2], mx[3])), fmaxf(fmaxf(mx[4], mx[5]), fmaxf(mx[6], mx[7])));
}

// P = 2^(s * scale - m) for 32 scores, packed to bf16 pairs and written to 16 TMEM columns at t_p;
// adds to the two partial row sums.  (Variants measured in the kernel and found no faster at the
// configs' shapes: all 32 exponentials issued before the sums, and packing by integer add and byte
// permute instead of the conversion instruction, which shares the SFU's pipe.)
__device__ __forceinline__ void exp32_store(const uint32_t* s, float scale_log2, float m_used, uint32_t t_p, float& l0,
                                            float& l1) {
  uint32_t pk[16];
#pragma unroll
  for (int j = 0; j < 16; ++j) {
    const float p0 = ex2_approx(fmaf(__uint_as_float(s[2 * j]), scale_log2, -m_used));
    const float p1 = ex2_approx(fmaf(__uint_as_float(s[2 * j + 1]), scale_log2, -m_used));
    l0 += p0;
    l1 += p1;
    pk[j] = pack_bf16(p0, p1);
  }
  tmem_st16(t_p, pk);
}

// The same for 64 scores (32 TMEM columns at t_p); returns the row sum.
__device__ __forceinline__ float exp64_store(const uint32_t (&s)[64], float scale_log2, float m_used, uint32_t t_p) {
  float l0 = 0.f, l1 = 0.f;
  exp32_store(s, scale_log2, m_used, t_p, l0, l1);
  exp32_store(s + 32, scale_log2, m_used, t_p + 16, l0, l1);
  return l0 + l1;
}

template <int D>
__device__ __forceinline__ bool softmax_half_full(uint32_t t_s, uint32_t t_o, bool first, float scale_log2,
                                                  float& m_used, float& l_run, uint32_t bar_pv_done,
                                                  uint32_t pv_parity, volatile int* abort_ptr) {
  uint32_t s[64];
  tmem_ld32(t_s, s);
  tmem_ld32(t_s + 32, s + 32);
  tmem_ld_wait();
  if (first) {
    m_used = row_max64<D>(s) * scale_log2;
    l_run = 0.f;
  }
  float l_half = exp64_store(s, scale_log2, m_used, t_s);
  if (!first) {
    const bool grow = !(l_half <= kSumLimit);   // also catches a NaN sum
    if (__any_sync(0xffffffffu, grow)) {
      const float m_new = row_max64<D>(s) * scale_log2;
      tmem_st_wait();   // the P just written is replaced below
      if (!rescale_o<D>(t_o, grow, m_new, m_used, l_run, bar_pv_done, pv_parity, abort_ptr)) return false;
      l_half = exp64_store(s, scale_log2, m_used, t_s);
    }
  }
  l_run += l_half;
  tmem_st_wait();
  return true;
}

// Ragged half-step (fewer than 64 valid keys: the end of the cache rows, or the fresh rows): 32
// columns at a time, keys at or beyond `valid` masked out.
template <int D>
__device__ __noinline__ bool softmax_half_ragged(uint32_t t_s, uint32_t t_o, int valid, bool first, float scale_log2,
                                                 float& m_used, float& l_run, uint32_t bar_pv_done,
                                                 uint32_t pv_parity, volatile int* abort_ptr) {
  const int n_chunks = (valid + 31) >> 5;
  uint32_t v[32];
  float mx = -CUDART_INF_F;
  for (int c = 0; c < n_chunks; ++c) {
    tmem_ld32(t_s + c * 32, v);
    tmem_ld_wait();
#pragma unroll
    for (int j = 0; j < 32; ++j)
      if (c * 32 + j < valid) mx = fmaxf(mx, __uint_as_float(v[j]));
  }
  const float m_new = mx * scale_log2;
  if (first) {
    m_used = m_new;
    l_run = 0.f;
  } else {
    const bool grow = m_new > m_used + kRescaleThreshold;
    if (__any_sync(0xffffffffu, grow)) {
      if (!rescale_o<D>(t_o, grow, m_new, m_used, l_run, bar_pv_done, pv_parity, abort_ptr)) return false;
    }
  }
  float l_add = 0.f;
  for (int c = 0; c < n_chunks; ++c) {
    tmem_ld32(t_s + c * 32, v);
    tmem_ld_wait();
    uint32_t pk[16];
#pragma unroll
    for (int j = 0; j < 16; ++j) {
      float p0 = ex2_approx(fmaf(__uint_as_float(v[2 * j]), scale_log2, -m_used));
      float p1 = ex2_approx(fmaf(__uint_as_float(v[2 * j + 1]), scale_log2, -m_used));
      if (c * 32 + 2 * j >= valid) p0 = 0.f;
      if (c * 32 + 2 * j + 1 >= valid) p1 = 0.f;
      l_add += p0 + p1;
      pk[j] = pack_bf16(p0, p1);
    }
    tmem_st16(t_s + c * 16, pk);
  }
  l_run += l_add;
  tmem_st_wait();
  return true;
}

enum BlockWork { kManySegments, kOneUnit, kPartOfTeam, kPartOfWideTeam };   // what a block of a launch has

// kNoWait = true is the instantiation a test selects to run the give-up path: every wait on work still to come tests
// its barrier once and gives up if the data is not there yet (waits that let issued copies and MMAs finish keep the
// 2 s limit).  The limit is a compile-time constant because the waits sit on the critical path of the MMA issuers
// (a run-time limit cost 2 % at the Dream shape).
template <int D, int kChunk, BlockWork kWork, bool kNoWait>
__global__ void __launch_bounds__(kThreads, 1)
attn_step_sm100_kernel(const __grid_constant__ CUtensorMap tm_q, const __grid_constant__ CUtensorMap tm_kc,
                       const __grid_constant__ CUtensorMap tm_vc, const __grid_constant__ CUtensorMap tm_kn,
                       const __grid_constant__ CUtensorMap tm_vn, const __grid_constant__ AttnParams p) {
  using G = Geometry<D>;
  constexpr uint64_t kLimit = kNoWait ? 0ull : kWaitLimitNs;
  // One M tile per block: the two chains of warps that otherwise have an M tile each share it and split the keys, chain h taking
  // keys 64 h .. 64 h + 63 of every tile into an O, maximum and sum of its own, folded at the end.
  constexpr bool kSingle = kWork != kManySegments, kTeam = kWork == kPartOfTeam, kWide = kWork == kPartOfWideTeam, kKeys = kTeam && kChunk <= 128;
  const int n_chains = kKeys ? 2 : p.n_mt;
  // softmax threads that own a real query row, rounded up to whole warps (tid 0 .. n_live-1; keys split: of either half)
  const int n_live = (p.rows + 31) & ~31;
  // Shared memory of the block, all of it dynamic (the scheduling tables are sized by batch and grid):
  // [Q: n_mt tiles][K ring][V ring][barriers][flags][scheduling tables], from the first 1024-byte
  // boundary (the swizzled tiles need that alignment).
  extern __shared__ uint8_t smem_raw[];
  // compile-time ring depths: the MMA issuers' scalar code is on the critical path, and divisions by a
  // run-time depth in it cost 10 % at the LLaDA shape
  constexpr int KS = G::kStages, VS = G::kStages;
  const uint32_t smem_pad = (1024u - (smem_u32(smem_raw) & 1023u)) & 1023u;
  const uint32_t smem_base = smem_u32(smem_raw) + smem_pad;
  const uint32_t sm_q = smem_base;                               // [n_mt][kTileBytes]
  const uint32_t sm_k = sm_q + p.n_mt * G::kTileBytes;           // [KS][kTileBytes]
  const uint32_t sm_v = sm_k + KS * G::kTileBytes;               // [VS][kTileBytes]
  const uint32_t sm_bar = sm_v + VS * G::kTileBytes;             // barriers, 8 bytes each
  int* const flags = reinterpret_cast<int*>(smem_raw + smem_pad + (size_t)(p.n_mt + KS + VS) * G::kTileBytes + kBarrierBytes);
  volatile int* const abort_ptr = flags;        // raised by the first wait that gives up
  volatile int* const never_ptr = flags + 1;    // for waits that must not be cut short by an abort; raised by one that runs out
  uint32_t* const tmem_slot = reinterpret_cast<uint32_t*>(flags + 2);
  volatile int* const merge_ok = flags + 3;
  volatile int* const any_empty = flags + 4;    // some batch element has no key tile at all
  Sched sched;
  float2* const fold = reinterpret_cast<float2*>(flags + kFlagBytes / 4);   // [key half][row]
  const uint32_t sm_x = smem_u32(fold) + kFoldBytes;                        // kSingle: what the team's other blocks send (team_bytes)
  sched.prefix = flags + kFlagBytes / 4;
  sched.lc = sched.prefix + p.batch + 1;
  sched.lq = sched.lc + p.batch;
  if (smem_pad + (uint32_t)(p.n_mt + KS + VS) * G::kTileBytes + kBarrierBytes + kFlagBytes +
          (kTeam ? (uint32_t)(kFoldBytes + team_bytes(D, p.team, n_live)) : kSingle ? 0u : 4u * (uint32_t)sched_ints(p.batch)) > (uint32_t)p.smem_bytes ||
      (kTeam && cluster_nctarank() != (uint32_t)p.team)) {
    // cannot happen with the host's sizing (it leaves room for the largest pad) and launch; nothing has been touched yet
    if (threadIdx.x == 0) dlm_set_status(p.status, DLM_ERR_WORKSPACE);
    return;
  }

  const uint32_t bar_q_full = sm_bar, bar_q_empty = sm_bar + 8, bar_drain = sm_bar + 16;   // drain: [2]
  const uint32_t bar_k_full = sm_bar + 32, bar_k_empty = bar_k_full + 8 * kMaxStages;
  const uint32_t bar_v_full = bar_k_empty + 8 * kMaxStages, bar_v_empty = bar_v_full + 8 * kMaxStages;
  const uint32_t bar_s_ready = bar_v_empty + 8 * kMaxStages;             // [M tile][score buffer]: scores of a half-step written
  const uint32_t bar_p_ready = bar_s_ready + 32;                 // [M tile][score buffer]: P of a half-step written
  const uint32_t bar_pv_done = bar_p_ready + 32;                 // [M tile][half-step parity] P V product finished.  Two P V
                                                                 // products can be in flight, so consecutive half-steps use different
                                                                 // barriers: a parity wait cannot tell phases two apart
  const uint32_t bar_pub = bar_pv_done + 32;                   // partial result of a segment stored by every softmax thread
  const uint32_t bar_team = bar_pub + 8;                         // team schedule: the other blocks' pieces are there
  const uint32_t bar_fold = bar_team + 8;                        // teams: both chains are through (keys split: maxima and sums there too)
  const uint32_t bar_guess = bar_fold + 8;                       // K and V tile copied before the lengths were known [2]

  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;

  // ---- set-up: barriers, TMEM, descriptor prefetch and which unit is this block's first (they need no data), so that they
  // overlap the kernel before; then the lengths
  if (tid == 0) {
    *abort_ptr = 0; *never_ptr = 0; *merge_ok = 0; *any_empty = 0;
    mbar_init(bar_q_full, 1);
    mbar_init(bar_q_empty, (uint32_t)n_chains);     // one commit per MMA issuer
    mbar_init(bar_drain, 1);
    mbar_init(bar_drain + 8, 1);
    mbar_init(bar_pub, (uint32_t)(kTeam ? n_live / 32 * (kKeys ? 2 : 1) : n_live));   // clusters: one arrival per warp
    mbar_init(bar_team, 1);
    mbar_init(bar_guess, 1);
    mbar_init(bar_guess + 8, 1);
    mbar_init(bar_fold, (uint32_t)n_live / (kKeys ? 16 : 32));     // one arrival per live warp (keys split: of either half)
    for (int i = 0; i < KS; ++i) {
      mbar_init(bar_k_full + 8 * i, 1);
      mbar_init(bar_k_empty + 8 * i, (uint32_t)n_chains);
    }
    for (int i = 0; i < VS; ++i) {
      mbar_init(bar_v_full + 8 * i, 1);
      mbar_init(bar_v_empty + 8 * i, (uint32_t)n_chains);
    }
    for (int i = 0; i < 2; ++i) {
      const uint32_t live_i = (uint32_t)(kKeys ? n_live : max(32, min(128, n_live - 128 * i))) / 32;   // one arrival per live warp
      for (int u = 0; u < 2; ++u) {
        mbar_init(bar_s_ready + 16 * i + 8 * u, 1);
        mbar_init(bar_p_ready + 16 * i + 8 * u, live_i);
      }
      mbar_init(bar_pv_done + 16 * i, 1);
      mbar_init(bar_pv_done + 16 * i + 8, 1);
    }
    mbar_fence_init();
    fence_proxy_async_smem();
  }
  if (warp == 9) {
    tmem_alloc(smem_u32(tmem_slot), kTmemCols);
    tmem_relinquish();
  }
  if (warp == 8 && lane == 0) {
    prefetch_tensormap(&tm_q);
    prefetch_tensormap(&tm_kc);
    prefetch_tensormap(&tm_vc);
    prefetch_tensormap(&tm_kn);
    prefetch_tensormap(&tm_vn);
  }
  // Blocks of a single unit: the key tile that the block has first if the lengths are as expected is copied before they are read.  (Their
  // chain -- a round trip, the share, the copy's issue -- stood before a call's first scores: K was asked for 2300 cycles after the
  // wait for the kernel before, now 200.  One-layer calls: one sequence 8.55 -> 8.3 us, 32 KV heads 10.75 -> 10.25, an LLaDA layer 27.9 -> 27.6; 28
  // layers in one call 25.65 -> 24.95; every 400 cycles that the copy comes later cost 0.15 - 0.2 us.)  That copy has barriers of its own;
  // where the lengths are others, which all roles see alike, its data is dropped and the rings start as if it had not been.
  Segment one;
  int guess_first = 0, guess_n_ct = 0;
  bool ahead = false, hit = false;   // there is such a copy; it is what the block needs first
  if (kSingle) {
    decode_single(p, one);
    Segment guess = one;
    set_single_lengths(p, guess, p.hint_len, p.q_cap);
    ahead = guess.t_end > guess.t_begin;
    guess_first = guess.t_begin;
    guess_n_ct = guess.n_ct;
    if (tid == 0) {   // for the translation of their addresses, not their values
      prefetch_l2(p.cache_len + one.b);
      if (p.q_len) prefetch_l2(p.q_len + one.b);
    }
  }
  // barrier "full" of the i-th tile of a ring, and its phase: a copy made ahead takes the place of the first stage's first
  auto full_bar = [&](uint32_t ring, uint32_t guess, uint32_t i, uint32_t stages) { return kSingle && hit && i == 0 ? guess : ring + 8 * (i % stages); };
  auto full_parity = [&](uint32_t i, uint32_t stages) { return (i / stages - (kSingle && hit && i >= stages && i % stages == 0 ? 1u : 0u)) & 1u; };
  __syncwarp();
  tc_fence_before_sync();
  // the barriers exist and TMEM is there; in a team, so do the other blocks' barriers
  if (kTeam) cluster_sync(); else __syncthreads();
  tc_fence_after_sync();
  const uint32_t tmem = *tmem_slot;
  // Everything above needed no data.  Whole units and teams: which unit a block starts with does not depend on the lengths, so
  // the copy of its Q rows starts before they are read (about 1 us, and Q does not queue in front of the first K tile).  The
  // roles below consume this Q also when the unit turns out to have no key tile for this block.
  const bool early_q = kSingle || p.whole_units != 0;
  auto expect_q = [&]() { mbar_expect_tx(bar_q_full, (uint32_t)(p.n_mt * min(128, p.rows)) * 128u * G::kPanels); };   // a box counts in full
  auto copy_q = [&](int zq, int rc) {
    for (int mt = 0; mt < p.n_mt; ++mt)
      for (int pn = 0; pn < G::kPanels; ++pn)
        tma_load_3d(sm_q + mt * G::kTileBytes + pn * kPanelBytes, &tm_q, bar_q_full, pn * 64, rc * (kKeys ? p.chunk_rows : kChunk) + mt * 128, zq);
  };
  // From here on the inputs of the call are read: all threads wait for the kernel before.  In a block of a single unit each role
  // does so where it starts, so that the code up to there has been fetched by then, and reads its unit's lengths for itself.
  auto wait_for_inputs = [&]() {
    dlm_grid_dependency_wait();
    dlm_trigger_dependents();
  };
  auto read_lengths = [&]() {
    int Lc = p.cache_len[one.b], Lq = p.q_len ? p.q_len[one.b] : p.q_cap;
    if (Lc < 0 || Lc > p.capacity || Lq < 0 || Lq > p.q_cap) {
      if (tid == 0) dlm_set_status(p.status, DLM_ERR_CAPACITY);
      Lc = max(0, min(Lc, p.capacity));
      Lq = max(0, min(Lq, p.q_cap));
    }
    set_single_lengths(p, one, Lc, Lq);
    const bool same = one.t_begin < one.t_end && one.t_begin == guess_first && (guess_first < guess_n_ct ? guess_first < one.n_ct : guess_n_ct == one.n_ct);
    hit = ahead && same;
  };
  auto team_shape = [&]() {
    TeamShape a;
    a.by_team = p.by_team;
    a.team = p.team;
    p.by_team.divmod(blockIdx.x, a.rank);
    a.R = n_live;
    a.share = team_share(D, p.team);
    a.sm_piece = sm_k;
    a.sm_x = sm_x;
    a.sm_ml = sm_x + (uint32_t)((p.team - 1) * a.share * n_live * 32);
    return a;
  };
  if (!kSingle) {
    wait_for_inputs();
    if (early_q && warp == 8 && lane == 0) {
      int b, rc, kvh;
      const int lc_layer = p.by_kv_heads.divmod(p.by_rc.divmod(p.by_batch.divmod(blockIdx.x, b), rc), kvh);
      expect_q();
      copy_q((lc_layer * p.batch + b) * p.n_kv_heads + kvh, rc);
    }
  }
  // lengths and tile prefix, by one warp: lane = batch element
  if (!kSingle && warp == 0) {
    int acc = 0;
    for (int b0 = 0; b0 < p.batch; b0 += 32) {
      const int b = b0 + lane;
      int Lc = 0, Lq = 0, tiles = 0;
      if (b < p.batch) {
        Lc = p.cache_len[b];
        Lq = p.q_len ? p.q_len[b] : p.q_cap;
        if (Lc < 0 || Lc > p.capacity || Lq < 0 || Lq > p.q_cap) {
          dlm_set_status(p.status, DLM_ERR_CAPACITY);
          Lc = max(0, min(Lc, p.capacity));
          Lq = max(0, min(Lq, p.q_cap));
        }
        tiles = tiles_of(Lc, Lq, p.fresh_box);
        sched.lc[b] = Lc;
        sched.lq[b] = Lq;
      }
      int inc = tiles;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int v = __shfl_up_sync(0xffffffffu, inc, o);
        if (lane >= o) inc += v;
      }
      if (b < p.batch) sched.prefix[b] = acc + inc - tiles;
      if (__any_sync(0xffffffffu, b < p.batch && tiles == 0) && lane == 0) *any_empty = 1;
      acc += __shfl_sync(0xffffffffu, inc, 31);
    }
    if (lane == 0) sched.prefix[p.batch] = acc;
  }
  if (!kSingle) __syncthreads();
  // number of shares the item list is cut into (every share holds at least one item)
  int n_cta = (int)gridDim.x;
  sched.n_cta = n_cta;
  sched.share = sched.share_rem = 0;
  if (!kSingle && !p.whole_units) {
    const int total_items = sched.prefix[p.batch] * p.nl * p.n_kv_heads * p.n_rc;
    n_cta = min(n_cta, total_items);
    sched.n_cta = max(n_cta, 1);
    sched.share = total_items / sched.n_cta;
    sched.share_rem = total_items - sched.share * sched.n_cta;
  }
  const bool has_work = kSingle || p.whole_units || (int)blockIdx.x < n_cta;

  // The softmax warps keep a whole score row in registers; the other warpgroup needs few.
  // setmaxnreg.inc waits, without a bound, until the registers it asks for are free: the host
  // checks before the first launch that what the third warpgroup gives up covers what the two
  // softmax warpgroups take (kRegsSoftmax, kRegsOther against the kernel's register count).
  if (warp >= 8) {
    setmaxnreg_dec<kRegsOther>();
    if (warp == 8) {
      // ================================================================= TMA producer
      auto tile_bytes = [&](bool cache) { return (uint32_t)(cache ? min(kTileKeys, p.capacity) : p.fresh_box) * 128u * G::kPanels; };
      auto copy_tile = [&](uint32_t dst, const CUtensorMap* map, uint32_t bar, int row, int z) {
        for (int pn = 0; pn < G::kPanels; ++pn) tma_load_3d(dst + pn * kPanelBytes, map, bar, pn * 64, row, z);
      };
      if (kSingle) {
        const int zq = (one.lc_layer * p.batch + one.b) * p.n_kv_heads + one.kvh;
        const bool cache = guess_first < guess_n_ct;
        const int row = cache ? guess_first * kTileKeys : (guess_first - guess_n_ct) * p.fresh_box;
        const int z = cache ? zq + p.layer_begin * p.batch * p.n_kv_heads : zq;
        if (lane == 0) {
          expect_q();
          if (ahead) {
            mbar_expect_tx(bar_guess, tile_bytes(cache));
            mbar_expect_tx(bar_guess + 8, tile_bytes(cache));
          }
        }
        wait_for_inputs();
        if (lane == 0) {
          copy_q(zq, one.rc);
          if (ahead) {
            copy_tile(sm_k, cache ? &tm_kc : &tm_kn, bar_guess, row, z);
            copy_tile(sm_v, cache ? &tm_vc : &tm_vn, bar_guess + 8, row, z);
          }
        }
        __syncwarp();
        read_lengths();
        if (lane == 0 && ahead && !hit) {   // others go to the same shared memory, so not before these have landed
          mbar_wait(bar_guess, 0, never_ptr);
          mbar_wait(bar_guess + 8, 0, never_ptr);
        }
      }
      if (lane == 0 && has_work) {
        SegmentWalker<kSingle> walk(p, sched, blockIdx.x);
        Segment g = one;
        uint32_t kt = 0, vt = 0, seg = 0, q_issued = early_q ? 1 : 0;
        bool ok = true;
        bool q_ahead = early_q;   // the Q of the block's first unit is already on its way
        while (ok && walk.next(g, n_cta)) {
          const bool q_here = q_ahead;
          q_ahead = false;
          if (g.t_end <= g.t_begin) {
            if (q_here) ++seg;   // the issuers take and release that Q all the same
            continue;
          }
          const int zq = (g.lc_layer * p.batch + g.b) * p.n_kv_heads + g.kvh;
          const int zc = ((g.lc_layer + p.layer_begin) * p.batch + g.b) * p.n_kv_heads + g.kvh;
          if (!q_here) {
            if (seg > 0) ok = mbar_wait_limit(bar_q_empty, (seg - 1) & 1, abort_ptr, kLimit);
            if (!ok) break;
            expect_q();
            copy_q(zq, g.rc);
            ++q_issued;
          }
          for (int t = g.t_begin; t < g.t_end && ok; ++t) {
            const bool cache = t < g.n_ct;
            const int row = cache ? t * kTileKeys : (t - g.n_ct) * p.fresh_box;
            const int z = cache ? zc : zq;
            const uint32_t bytes = tile_bytes(cache);
            if (kSingle && kt == 0 && hit) {   // on its way already
              ++kt;
              ++vt;
              continue;
            }
            {
              const uint32_t s = kt % KS;
              if (kt >= (uint32_t)KS) ok = mbar_wait_limit(bar_k_empty + 8 * s, ((kt / KS) - 1) & 1, abort_ptr, kLimit);
              if (!ok) break;
              mbar_expect_tx(bar_k_full + 8 * s, bytes);
              copy_tile(sm_k + s * G::kTileBytes, cache ? &tm_kc : &tm_kn, bar_k_full + 8 * s, row, z);
              ++kt;
            }
            {
              const uint32_t s = vt % VS;
              if (vt >= (uint32_t)VS) ok = mbar_wait_limit(bar_v_empty + 8 * s, ((vt / VS) - 1) & 1, abort_ptr, kLimit);
              if (!ok) break;
              mbar_expect_tx(bar_v_full + 8 * s, bytes);
              copy_tile(sm_v + s * G::kTileBytes, cache ? &tm_vc : &tm_vn, bar_v_full + 8 * s, row, z);
              ++vt;
            }
          }
          ++seg;
        }
        // No copy lands after the block has released its shared memory: wait for those whose consumer may not have, also when
        // this lane itself never had to give up (its last copies were issued before another role did, or a unit without key
        // tiles has its Q on the way).  They have landed long since unless the block is unwinding.
        for (uint32_t i = (kt > (uint32_t)KS ? kt - KS : 0); i < kt; ++i)
          mbar_wait(full_bar(bar_k_full, bar_guess, i, KS), full_parity(i, KS), never_ptr);
        for (uint32_t i = (vt > (uint32_t)VS ? vt - VS : 0); i < vt; ++i)
          mbar_wait(full_bar(bar_v_full, bar_guess + 8, i, VS), full_parity(i, VS), never_ptr);
        if (q_issued > 0) mbar_wait(bar_q_full, (q_issued - 1) & 1, never_ptr);
      }
    } else if (warp == 9 || warp == 10) {
      // ============================================ MMA issuers: warp 9 for M tile (or key half) 0, warp 10 for 1
      // One warp per M tile, so that the scalar work around one tile's MMAs (barrier waits and
      // commits) runs while the tensor pipe executes the other tile's.  One elected lane runs the whole
      // loop, waits included: with the warp taking part in every wait and a lane elected per product, waits on
      // complete barriers and the elections stood between P's arrival and the products it releases (an LLaDA layer, one M tile
      // per block: 31.5 us, now 29.5; two M tiles, where the softmax warps bound the loop, 0 - 2 %).  The K, V and Q
      // buffers are released when every issuer has committed (their "empty" barriers count as many arrivals).
      const int mt = warp - 9;
      if (kSingle) {
        wait_for_inputs();
        read_lengths();
      }
      if (has_work && mt < n_chains && elect_one_sync()) {
        auto wait = [&](uint32_t bar, uint32_t parity) { return mbar_wait_limit(bar, parity, abort_ptr, kLimit); };
        SegmentWalker<kSingle> walk(p, sched, blockIdx.x);
        Segment g = one;
        uint32_t kt = 0, vt = 0, gt = 0, seg = 0;
        bool ok = true;
        const uint32_t idesc_pv = make_idesc_bf16(128, D, 1);
        // descriptors of the first K-step of each operand buffer; the loops only add constants
        const uint64_t desc_q = make_smem_desc_sw128(sm_q + (kKeys ? 0 : mt) * G::kTileBytes, 16, 1024);
        const uint64_t desc_k0 = make_smem_desc_sw128(sm_k, 16, 1024);
        const uint64_t desc_v0 = make_smem_desc_sw128(sm_v, kPanelBytes, 1024);
        const uint32_t t_o = tmem + G::kColO + mt * D;
        const uint32_t t_s = tmem + G::kColS + mt * 128;
        // S = Q K^T for the keys [k0, k0 + n16) of the tile in K stage `ks`, into score buffer `buf`
        auto issue_s = [&](uint32_t ks, int k0, int n16, uint32_t buf) {
          const uint32_t idesc = make_idesc_bf16(128, (uint32_t)n16, 0);
          const uint64_t dk = desc_offset(desc_k0, ks * G::kTileBytes + k0 * 128);
          const uint32_t d = t_s + buf * kHalfKeys;
#pragma unroll
          for (int k = 0; k < D / 16; ++k) {
            const uint32_t off = ((k >> 2) * kPanelBytes + (k & 3) * 32) >> 4;
            mma_ss_lo<false>(d, (uint32_t)desc_q + off, (uint32_t)dk + off, (uint32_t)(desc_q >> 32), idesc, k > 0 ? 1u : 0u);
          }
        };
        // O (+)= P V for the same keys, P in score buffer `buf`, V tile in stage `vs`
        auto issue_pv = [&](uint32_t vs, int k0, int n16, uint32_t buf, bool first) {
          const uint64_t dv = desc_offset(desc_v0, vs * G::kTileBytes + k0 * 128);
          const uint32_t a = t_s + buf * kHalfKeys;
          if (first) mma_ts<false>(t_o, a, dv, idesc_pv); else mma_ts<true>(t_o, a, dv, idesc_pv);
          if (n16 == kHalfKeys) {
#pragma unroll
            for (int st = 1; st < kHalfKeys / 16; ++st) mma_ts<true>(t_o, a + st * 8, desc_offset(dv, st * 2048), idesc_pv);
          } else {
            for (int st = 1; st < n16 / 16; ++st) mma_ts<true>(t_o, a + st * 8, desc_offset(dv, st * 2048), idesc_pv);
          }
        };
        uint32_t js = 0;   // half-steps whose scores have been issued (global count: buffer = js & 1)
        bool q_ahead = early_q;   // the Q of the block's first unit was copied before the lengths were known
        while (ok && walk.next(g, n_cta)) {
          const bool q_here = q_ahead;
          q_ahead = false;
          if (g.t_end <= g.t_begin) {
            if (q_here) {   // no key tile for this block after all: take that Q and release it
              ok = wait(bar_q_full, seg & 1);
              if (!ok) break;
              mbar_arrive(bar_q_empty);
              ++seg;
            }
            continue;
          }
          ok = wait(bar_q_full, seg & 1);
          if (!ok) break;
          HalfIter<kKeys> si(g, p.fresh_box, mt), pi(g, p.fresh_box, mt);
          // scores of the next half-step of the segment that has none yet, into buffer js & 1
          auto issue_next_s = [&]() -> bool {
            HalfStep hs;
            for (; si.skips(); ++si.t, ++kt) {   // (behind the copy, so that the arrival counts for this use of the buffer)
              if (!wait(full_bar(bar_k_full, bar_guess, kt, KS), full_parity(kt, KS))) return false;
              mbar_arrive(bar_k_empty + 8 * (kt % KS));
            }
            if (!si.get(hs)) return true;
            const uint32_t ks = kt % KS;
            if (hs.first_of_tile) {
              if (!wait(full_bar(bar_k_full, bar_guess, kt, KS), full_parity(kt, KS))) return false;
              tc_fence_after_sync();
            }
            issue_s(ks, hs.k0, (hs.nkeys + 15) & ~15, js & 1);
            tc_commit(bar_s_ready + 16 * mt + 8 * (js & 1));
            ++js;
            si.advance(hs);
            if (hs.last_of_tile) {
              tc_commit(bar_k_empty + 8 * ks);
              ++kt;
              if (si.t >= g.t_end) tc_commit(bar_q_empty);   // Q is not read again in this segment
            }
            return true;
          };
          ok = issue_next_s() && issue_next_s();   // both score buffers filled ahead
          bool first = true;
          HalfStep hs;
          auto skip_v = [&]() -> bool {
            for (; pi.skips(); ++pi.t, ++vt) {
              if (!wait(full_bar(bar_v_full, bar_guess + 8, vt, VS), full_parity(vt, VS))) return false;
              mbar_arrive(bar_v_empty + 8 * (vt % VS));
            }
            return true;
          };
          while (ok && (ok = skip_v()) && pi.get(hs)) {
            const uint32_t vs = vt % VS;
            if (hs.first_of_tile) {
              ok = wait(full_bar(bar_v_full, bar_guess + 8, vt, VS), full_parity(vt, VS));
              if (!ok) break;
            }
            ok = wait(bar_p_ready + 16 * mt + 8 * (gt & 1), (gt >> 1) & 1);
            if (!ok) break;
            tc_fence_after_sync();
            issue_pv(vs, hs.k0, (hs.nkeys + 15) & ~15, gt & 1, first);
            tc_commit(bar_pv_done + 16 * mt + 8 * (gt & 1));
            first = false;
            if (hs.last_of_tile) {
              tc_commit(bar_v_empty + 8 * vs);
              ++vt;
            }
            ++gt;
            pi.advance(hs);
            ok = issue_next_s();   // the buffer just consumed takes the half-step after next
          }
          ++seg;
        }
        // every MMA issued by this lane has finished before TMEM is released
        tc_commit(bar_drain + 8 * mt);
        mbar_wait(bar_drain + 8 * mt, 0, never_ptr);
      }
    } else {
      // ================================================================= publisher (warp 11)
      // A piece that some other block will merge: once every softmax thread has stored its row
      // (they arrive on bar_pub and move on), make the stores visible device-wide and count the
      // piece in its unit's counter.
      if (kSingle) {
        wait_for_inputs();
        read_lengths();
      }
      if (kTeam && lane == 0 && one.T > 0) {
        team_expect<D>(team_shape(), bar_team, one.T, one.t_end > one.t_begin);
      } else if (kWide && lane == 0) {
        wide_publish<kNoWait>(WideArgs(p, one, D), bar_pub, abort_ptr);
      } else if (!kSingle && lane == 0 && has_work && !p.whole_units) {
        SegmentWalker<kSingle> walk(p, sched, blockIdx.x);
        Segment g = one;
        uint32_t pub = 0;
        while (walk.next(g, n_cta)) {
          if (g.slot < 0 || g.merger || g.t_end <= g.t_begin) continue;
          if (!mbar_wait_limit(bar_pub, pub & 1, abort_ptr, kLimit)) break;
          ++pub;
          __threadfence();
          atomicAdd(p.tickets + ((g.lc_layer * p.n_kv_heads + g.kvh) * p.n_rc + g.rc) * p.batch + g.b, 1u);
        }
      }
    }
  } else {
    setmaxnreg_inc<kRegsSoftmax>();
    if (kSingle) {
      wait_for_inputs();
      read_lengths();
    }
    // teams: what this thread reduces, made ready while the first keys are on their way
    TeamShape sh;
    int red_row = 0, red_group = 0, red_groups = 0;
    bool red_real = false, red_active = false;
    __nv_bfloat16* red_out = nullptr;
    float* red_lse = nullptr;
    if (kTeam) {
      sh = team_shape();
      red_group = p.by_live.divmod(tid, red_row);
      red_groups = p.by_live.div(256);
      const int r_kv = one.rc * (kKeys ? p.chunk_rows : kChunk) + red_row;
      red_real = red_row < p.rows && r_kv < p.rows_total;
      red_active = red_real && r_kv - p.by_q_cap.div(r_kv) * p.q_cap < one.Lq;
      const size_t qrow = (((size_t)one.lc_layer * p.batch + one.b) * p.n_q_heads + (size_t)one.kvh * p.group) * p.q_cap + r_kv;
      red_out = p.out + qrow * D;
      if (p.lse) red_lse = p.lse + qrow;
    }
    if ((kKeys ? tid & 127 : tid) < n_live) {
      // ================================================= softmax warps (those that own real rows)
      const int mt = warp >> 2;
      const int row = (warp & 3) * 32 + lane;                 // row of the M tile = TMEM lane
      const uint32_t t_lane = (uint32_t)((warp & 3) * 32) << 16;
      const uint32_t t_s = tmem + t_lane + G::kColS + mt * 128;
      const uint32_t t_o = tmem + t_lane + G::kColO + mt * D;
      const int r_unit = kKeys ? row : mt * 128 + row;        // row within the unit
      const int n_live_mt = kKeys ? n_live : min(128, n_live - 128 * mt);   // live softmax threads of this M tile
      // the warp leaves a wait together, so the .sync.aligned TMEM instructions that follow
      // always see a converged warp, also when a wait is given up
      auto wait_warp = [&](uint32_t bar, uint32_t parity) { return mbar_wait_warp(bar, parity, abort_ptr, kLimit); };
      const int chunk_rows = kKeys ? p.chunk_rows : kChunk;
      // this thread's query row in row chunk rc of a KV head: which of its query heads, which active row
      // (rows of a KV head's query heads lie one after the other)
      auto out_row_of = [&](int lc_layer, int b, int kvh, int rc) {
        return (((size_t)lc_layer * p.batch + b) * p.n_q_heads + (size_t)kvh * p.group) * p.q_cap + rc * chunk_rows + r_unit;
      };
      constexpr int kCols = kKeys ? D / 2 : D;               // of O that this thread folds and stores
      const int c0 = kKeys ? mt * kCols : 0;
      TeamParcel parcel;
      if (kTeam) parcel = team_parcel<D>(sh, bar_team, r_unit >> 5, c0 / 8, (c0 + kCols) / 8, kKeys ? mt : 0, kKeys ? 2 : 1);
      // teams: the row's (m, l) and O to the block's piece; O complete in TMEM at t (and t2), or the block has no key tile
      auto lay_out_piece = [&](bool has_tiles, uint32_t t, uint32_t t2, const float (&w)[2], float m, float l) {
        st_shared_f2(sh.sm_ml + ((p.team - 1) * n_live + r_unit) * 8, m, l);
        if (has_tiles) {
          uint32_t to = sh.sm_piece + ((r_unit >> 5) * (D / 4) + c0 / 4) * 512 + lane * 16;
#pragma unroll 1
          for (int c = c0; c < c0 + kCols; c += 32) {
            uint32_t v[32];
            read_o<kKeys>(t + c, t2 + c, w, v);
#pragma unroll
            for (int j = 0; j < 32; j += 4, to += 512)
              st_shared_f4(to, __uint_as_float(v[j]), __uint_as_float(v[j + 1]), __uint_as_float(v[j + 2]), __uint_as_float(v[j + 3]));
          }
        }
        fence_proxy_async_smem();
        __syncwarp();
        if (lane == 0) mbar_arrive(bar_pub);   // for the block's own other warps
        if (parcel.ml_dst) bulk_copy_to_cluster(parcel.ml_dst, sh.sm_ml + ((p.team - 1) * n_live + (r_unit & ~31)) * 8, 256, parcel.bar);
        if (has_tiles && parcel.bytes) bulk_copy_to_cluster(parcel.dst, parcel.src, parcel.bytes, parcel.bar);
        __syncwarp();
      };
      auto zero_my_row = [&](size_t qrow, bool real_row) {
        if (real_row) {
          uint4* o = reinterpret_cast<uint4*>(p.out + qrow * D);
#pragma unroll
          for (int c = 0; c < D / 8; ++c) o[c] = make_uint4(0, 0, 0, 0);
          if (p.lse) p.lse[qrow] = -CUDART_INF_F;
        }
      };
      if (!kSingle && !p.whole_units && *any_empty) {
        // units without any key (inactive batch elements) appear in no share: zero them here
        const int n_units = p.nl * p.n_kv_heads * p.n_rc * p.batch;
        for (int unit = blockIdx.x; unit < n_units; unit += gridDim.x) {
          int b, rc, kvh;
          const int grp = p.by_batch.divmod(unit, b), lc_layer = p.by_kv_heads.divmod(p.by_rc.divmod(grp, rc), kvh);
          if (sched.prefix[b + 1] == sched.prefix[b])
            zero_my_row(out_row_of(lc_layer, b, kvh, rc), rc * chunk_rows + r_unit < p.rows_total);
        }
      }
      if (has_work) {
        SegmentWalker<kSingle> walk(p, sched, blockIdx.x);
        Segment g = one;
        uint32_t gt = 0, vt = 0;   // half-steps and key tiles done so far
        bool ok = true;
        while (ok && walk.next(g, n_cta)) {
          const int n = g.t_end - g.t_begin;
          if (n <= 0) {  // inactive batch element: the unit's rows are zero (team schedule: or no tile for this rank)
            if (g.T == 0) {
              zero_my_row(out_row_of(g.lc_layer, g.b, g.kvh, g.rc), g.rc * chunk_rows + r_unit < p.rows_total);
            } else if (kTeam) {   // a piece without key tiles
              const float none[2] = {0.f, 0.f};
              lay_out_piece(false, 0, 0, none, -CUDART_INF_F, 0.f);
            } else if (kWide) {
              ok = wide_exchange<D, kNoWait>(WideArgs(p, g, D), bar_pub, abort_ptr, true, t_o, false, -CUDART_INF_F, 0.f);
            }
            continue;
          }
          float m_used = -CUDART_INF_F, l_run = 0.f;
          bool first = true;
          const int n_whole = g.Lc / kTileKeys;   // tiles of 128 visible cache rows
          for (int t = g.t_begin; t < g.t_end && ok; ++t, ++vt) {
            const int valid = t < n_whole ? kTileKeys : tile_valid(g, t, p.fresh_box);
            const int n16 = (valid + 15) & ~15;
            const int k_begin = kKeys ? mt * kHalfKeys : 0, k_end = kKeys ? min(valid, k_begin + kHalfKeys) : valid;
            if (valid < n16 && k_begin < valid && k_end == valid) {
              // V rows in [valid, n16) would be multiplied by P = 0: clear them so that stale
              // NaN / Inf bit patterns cannot reach O.  Each M tile's warps do it before they
              // announce the P of the tile's first half-step, so it precedes that tile's P V
              // products (the two M tiles write the same zeros; with the keys split, the half that has them).
              const uint32_t vs = vt % VS;
              // (with the keys split, S of this tile does not show that the tile before the one before, whose V had the stage, is
              // through; a wait for a phase works only when the one before it is over)
              if (kKeys && gt > 0) ok = wait_warp(bar_pv_done + 16 * mt + 8 * ((gt - 1) & 1), ((gt - 1) >> 1) & 1);
              if (!ok) break;
              ok = wait_warp(full_bar(bar_v_full, bar_guess + 8, vt, VS), full_parity(vt, VS));
              if (!ok) break;
              const int per_row = G::kPanels * 8;
              for (int idx = row; idx < (n16 - valid) * per_row; idx += n_live_mt) {
                const int r = valid + idx / per_row, rem = idx % per_row;
                const uint32_t a = sm_v + vs * G::kTileBytes + (rem >> 3) * kPanelBytes + r * 128 + (rem & 7) * 16;
                asm volatile("st.shared.v4.b32 [%0], {%1, %1, %1, %1};" ::"r"(a), "r"(0u) : "memory");
              }
              fence_proxy_async_smem();
            }
            // the tile's half-steps (the same enumeration as HalfIter, which the MMA warps use)
            for (int k0 = k_begin; k0 < k_end && ok; k0 += kHalfKeys, ++gt) {
              const int nkeys = min(kHalfKeys, valid - k0);
              const uint32_t buf = gt & 1;
              ok = wait_warp(bar_s_ready + 16 * mt + 8 * buf, (gt >> 1) & 1);
              if (!ok) break;
              tc_fence_after_sync();
              if (nkeys == kHalfKeys)
                ok = softmax_half_full<D>(t_s + buf * kHalfKeys, t_o, first, p.scale_log2, m_used, l_run,
                                          bar_pv_done + 16 * mt + 8 * ((gt - 1) & 1), ((gt - 1) >> 1) & 1, abort_ptr);
              else
                ok = softmax_half_ragged<D>(t_s + buf * kHalfKeys, t_o, nkeys, first, p.scale_log2, m_used, l_run,
                                            bar_pv_done + 16 * mt + 8 * ((gt - 1) & 1), ((gt - 1) >> 1) & 1, abort_ptr);
              if (!ok) break;
              // every lane's P is stored (tcgen05.wait::st inside the softmax); one lane announces the warp's rows
              __syncwarp();
              if (lane == 0) {
                tc_fence_before_sync();
                mbar_arrive(bar_p_ready + 16 * mt + 8 * buf);
              }
              first = false;
            }
          }
          if (!ok) break;
          // ---- epilogue of the segment: O is complete once the last P V product has finished
          if (!kKeys || gt > 0) ok = wait_warp(bar_pv_done + 16 * mt + 8 * ((gt - 1) & 1), ((gt - 1) >> 1) & 1);
          if (!ok) break;
          tc_fence_after_sync();
          if (kTeam && !kKeys) {   // the piece is laid out over K tiles, which the other M tile's products may still read
            if (lane == 0) mbar_arrive(bar_fold);
            ok = wait_warp(bar_fold, 0);
            if (!ok) break;
          }
          float w[2] = {1.f, 0.f};                               // of the key halves' O, at t_first and t_second
          uint32_t t_first = t_o, t_second = t_o;
          if (kKeys) {
            // both halves' threads of a row learn of each other's maximum and sum ((-inf, 0) without keys); then each has
            // half of the columns
            fold[tid] = make_float2(m_used, l_run);
            tc_fence_before_sync();
            __syncwarp();
            if (lane == 0) mbar_arrive(bar_fold);
            ok = wait_warp(bar_fold, 0);
            if (!ok) break;
            tc_fence_after_sync();
            const float2 a = fold[row], b = fold[128 + row];
            m_used = fmaxf(a.x, b.x);
            w[0] = ex2_approx(a.x - m_used);
            w[1] = ex2_approx(b.x - m_used);     // 0 without keys
            l_run = fmaf(w[0], a.y, w[1] * b.y);
            t_first = t_second = t_o - mt * D;
            if (__any_sync(0xffffffffu, b.y != 0.f)) t_second += D;
            else w[0] = w[1] = 0.5f * w[0];
          }
          const size_t qrow = out_row_of(g.lc_layer, g.b, g.kvh, g.rc);
          const int r_kv = g.rc * chunk_rows + r_unit;           // row among all query rows of the KV head
          const bool real_row = r_kv < p.rows_total;
          const bool active = real_row && r_kv - p.by_q_cap.div(r_kv) * p.q_cap < g.Lq;
          uint32_t v[32];
          if (kTeam) {
            lay_out_piece(true, t_first, t_second, w, m_used, l_run);
          } else if (kWide) {
            ok = wide_exchange<D, kNoWait>(WideArgs(p, g, D), bar_pub, abort_ptr, true, t_o, true, m_used, l_run);
          } else if (kSingle || g.slot < 0) {
            const float inv = active ? 1.f / l_run : 0.f;
            constexpr int kChunks = kKeys ? D / 64 : D / 32;
            const int c0 = kKeys ? mt * kChunks : 0;
#pragma unroll 1
            for (int c = c0; c < c0 + kChunks; ++c) {
              read_o<kKeys>(t_first + c * 32, t_second + c * 32, w, v);
              if (real_row) {
                uint4* o = reinterpret_cast<uint4*>(p.out + qrow * D + c * 32);
#pragma unroll
                for (int q4 = 0; q4 < 4; ++q4) {
                  uint32_t w[4];
#pragma unroll
                  for (int j = 0; j < 4; ++j) {
                    const float a0 = active ? __uint_as_float(v[q4 * 8 + 2 * j]) * inv : 0.f;
                    const float a1 = active ? __uint_as_float(v[q4 * 8 + 2 * j + 1]) * inv : 0.f;
                    const __nv_bfloat162 h = __floats2bfloat162_rn(a0, a1);
                    w[j] = *reinterpret_cast<const uint32_t*>(&h);
                  }
                  o[q4] = make_uint4(w[0], w[1], w[2], w[3]);
                }
              }
            }
            if (real_row && p.lse && (!kKeys || mt == 0))
              p.lse[qrow] = active ? (m_used + lg2_approx(l_run)) * 0.6931471805599453f : -CUDART_INF_F;
          } else {
            // ---- a piece of a split unit.  Partial O is stored as 16-byte vectors of 4 columns,
            // [D/4][128 rows][4]: a warp's 32 rows of one vector are 512 contiguous bytes, for the
            // stores here and for the loads of the merge.
            if (!g.merger) {
              float4* po = reinterpret_cast<float4*>(p.ws_o) + ((size_t)g.slot * p.n_mt + mt) * (size_t)(D / 4 * 128) + row;
#pragma unroll 1
              for (int c = 0; c < D / 32; ++c) {
                tmem_ld32(t_o + c * 32, v);
                tmem_ld_wait();
#pragma unroll
                for (int j = 0; j < 8; ++j)
                  __stcg(po + (c * 8 + j) * 128, make_float4(__uint_as_float(v[4 * j]), __uint_as_float(v[4 * j + 1]),
                                                             __uint_as_float(v[4 * j + 2]), __uint_as_float(v[4 * j + 3])));
              }
              __stcg(reinterpret_cast<float2*>(p.ws_ml) + ((size_t)g.slot * p.n_mt + mt) * 128 + row,
                     make_float2(m_used, l_run));
              mbar_arrive(bar_pub);   // the publisher warp takes it from here
            } else {
              // ---- the unit's last piece: this block merges.  The other pieces belong to blocks
              // c_first .. this - 1, which computed them first thing; wait for their count, then fold
              // them into O (own piece first, then block order: the result does not depend on timing).
              const UnitPieces up(p, sched, g, blockIdx.x);
              const int n_others = up.c_last - up.c_first;
              const int unit = ((g.lc_layer * p.n_kv_heads + g.kvh) * p.n_rc + g.rc) * p.batch + g.b;
              if (tid == 0) {
                const bool came = wait_counter(p.tickets + unit, (unsigned int)n_others, abort_ptr, kLimit);
                if (came) p.tickets[unit] = 0;   // ready for the next launch
                *merge_ok = came ? 1 : 2;
              }
              // The other threads wait for thread 0's verdict on a flag, not on a hardware barrier: a warp that
              // gave up earlier never gets here, and a barrier would then wait for it for ever.  Thread 0 always
              // writes the flag within its own bounded wait; if its warp gave up before, the abort flag is up.
              for (uint32_t spin = 1; *merge_ok == 0; ++spin)
                if ((spin & 63u) == 0u && *abort_ptr) break;
              __syncwarp();
              const int verdict = __shfl_sync(0xffffffffu, *merge_ok, 0);   // one answer per warp: the code below is .aligned
              if (verdict != 1) { ok = false; break; }
              __threadfence();
              // maximum and sum over all pieces
              float m_all = m_used, l_all = l_run;
              for (int ib = 0; ib < n_others; ib += 4) {
                float2 ml[4];
#pragma unroll
                for (int j = 0; j < 4; ++j)
                  ml[j] = (ib + j < n_others)
                              ? __ldcg(reinterpret_cast<const float2*>(p.ws_ml) +
                                       ((size_t)up.slot_of(up.c_first + ib + j) * p.n_mt + mt) * 128 + row)
                              : make_float2(-CUDART_INF_F, 0.f);
                const float m_new = fmaxf(fmaxf(fmaxf(ml[0].x, ml[1].x), fmaxf(ml[2].x, ml[3].x)), m_all);
                l_all *= ex2_approx(m_all - m_new);
#pragma unroll
                for (int j = 0; j < 4; ++j) l_all += ml[j].y * ex2_approx(ml[j].x - m_new);
                m_all = m_new;
              }
              const float inv = active ? 1.f / l_all : 0.f;
              const float w_own = ex2_approx(m_used - m_all);
              if (real_row && p.lse)
                p.lse[qrow] = active ? (m_all + lg2_approx(l_all)) * 0.6931471805599453f : -CUDART_INF_F;
              // O: one other piece at a time, all of its row in flight at once (L2 latency, not
              // bandwidth, bounds a narrower loop); the running sum lives in TMEM between pieces
              for (int i = 0; i < n_others; ++i) {
                const size_t piece = (size_t)up.slot_of(up.c_first + i) * p.n_mt + mt;
                const float4* src = reinterpret_cast<const float4*>(p.ws_o) + piece * (size_t)(D / 4 * 128) + row;
                float4 x[D / 4];
#pragma unroll
                for (int j = 0; j < D / 4; ++j) x[j] = __ldcg(src + j * 128);
                const float w = ex2_approx(__ldcg(p.ws_ml + (piece * 128 + row) * 2) - m_all);
                const float w0 = (i == 0) ? w_own : 1.f;
                const bool last = (i == n_others - 1);
#pragma unroll
                for (int c = 0; c < D / 32; ++c) {
                  tmem_ld32(t_o + c * 32, v);
                  tmem_ld_wait();
#pragma unroll
                  for (int j = 0; j < 8; ++j) {
                    v[4 * j + 0] = __float_as_uint(fmaf(w, x[c * 8 + j].x, w0 * __uint_as_float(v[4 * j + 0])));
                    v[4 * j + 1] = __float_as_uint(fmaf(w, x[c * 8 + j].y, w0 * __uint_as_float(v[4 * j + 1])));
                    v[4 * j + 2] = __float_as_uint(fmaf(w, x[c * 8 + j].z, w0 * __uint_as_float(v[4 * j + 2])));
                    v[4 * j + 3] = __float_as_uint(fmaf(w, x[c * 8 + j].w, w0 * __uint_as_float(v[4 * j + 3])));
                  }
                  if (!last) {
                    tmem_st32(t_o + c * 32, v);
                  } else if (real_row) {
                    uint4* o = reinterpret_cast<uint4*>(p.out + qrow * D + c * 32);
#pragma unroll
                    for (int q4 = 0; q4 < 4; ++q4) {
                      uint32_t wd[4];
#pragma unroll
                      for (int j = 0; j < 4; ++j) {
                        const __nv_bfloat162 h =
                            __floats2bfloat162_rn(active ? __uint_as_float(v[q4 * 8 + 2 * j]) * inv : 0.f,
                                                  active ? __uint_as_float(v[q4 * 8 + 2 * j + 1]) * inv : 0.f);
                        wd[j] = *reinterpret_cast<const uint32_t*>(&h);
                      }
                      o[q4] = make_uint4(wd[0], wd[1], wd[2], wd[3]);
                    }
                  }
                }
                if (!last) tmem_st_wait();
              }
            }
          }
        }
      }
    }
    if (kWide && tid >= n_live && one.T > 0)   // warps without a row of their own help with the reduction
      wide_exchange<D, kNoWait>(WideArgs(p, one, D), bar_pub, abort_ptr, false, 0, false, 0.f, 0.f);
    if (kTeam && one.T > 0) {
      // teams: the columns that this block finishes, by all softmax threads
      if (mbar_wait_warp(bar_pub, 0, abort_ptr, kLimit) && mbar_wait_warp(bar_team, 0, abort_ptr, kLimit)) {
        if (red_group < red_groups) team_reduce<D>(sh, red_row, red_group, red_groups, red_real, red_active, red_out, red_lse);
      }
    }
  }
  // ---- teardown: nothing of this block is in flight any more.  A team's blocks leave together: none before the others have
  // stopped sending to its shared memory (every block gets here, also one that gave up, which then waits for what may be on its way).
  if (kTeam && tid == 0 && *abort_ptr && one.T > 0) mbar_wait(bar_team, 0, never_ptr);
  __syncwarp();
  if (kTeam) cluster_arrive();
  tc_fence_before_sync();
  __syncthreads();
  // behind the barrier: another role may give up after this thread has come this far, and then its rows are not written
  if (tid == 0 && (*abort_ptr || *never_ptr)) dlm_set_status(p.status, DLM_ERR_TIMEOUT);
  if (warp == 9) {
    tc_fence_after_sync();
    tmem_dealloc(tmem, kTmemCols);
    __syncwarp();
  }
  if (kTeam) cluster_wait();
}

// bf16 tensor viewed as [slabs][rows][D]; box = 64 elements x box_rows rows x 1 slab, 128-byte swizzle.
int encode_map(dlm_ctx* ctx, CUtensorMap* map, const void* base, int D, long long rows, long long slabs, int box_rows) {
  const cuuint64_t dims[3] = {(cuuint64_t)D, (cuuint64_t)rows, (cuuint64_t)slabs};
  const cuuint64_t strides[2] = {(cuuint64_t)D * 2, (cuuint64_t)rows * D * 2};
  const cuuint32_t box[3] = {64, (cuuint32_t)box_rows, 1};
  return dlm_tensor_map(ctx, map, base, 3, dims, strides, box) ? DLM_OK : DLM_ERR_CUDA;
}

// The kernel starts with `numRegs` registers per thread in all 12 warps.  The 8 softmax warps then
// ask for kRegsSoftmax each and block until they get them; only what the other 4 warps release
// is certain to be free, so the request must fit inside that.
bool register_budget_ok(const cudaFuncAttributes& a) {
  return a.numRegs >= kRegsOther && 8 * (kRegsSoftmax - a.numRegs) <= 4 * (a.numRegs - kRegsOther);
}

// The instantiations: head_dim 128 / 64; blocks of any number of segments, of one unit, parts of a team; units of up to 256 rows (two M
// tiles) / 128 (one; in teams with the keys split); normal / no-wait (test) waits.
using AttnKernel = void (*)(const CUtensorMap, const CUtensorMap, const CUtensorMap, const CUtensorMap, const CUtensorMap,
                            const AttnParams);
constexpr int kKernels = 16;
inline int kernel_index(int head_dim, const dlm_attn_plan& pl, bool no_wait) {
  const bool narrow = pl.single ? pl.n_mt == 1 : pl.chunk_rows == 128;
  return (head_dim == 128 ? 0 : 1) + (narrow ? 2 : 0) + (pl.wide ? 12 : pl.team > 1 ? 8 : pl.single ? 4 : 0) + (no_wait ? kKernels : 0);
}
template <bool kNoWait>
AttnKernel kernel_of_waits(int which) {
  switch (which) {
    case 0: return attn_step_sm100_kernel<128, 256, kManySegments, kNoWait>;
    case 1: return attn_step_sm100_kernel<64, 256, kManySegments, kNoWait>;
    case 2: return attn_step_sm100_kernel<128, 128, kManySegments, kNoWait>;
    case 3: return attn_step_sm100_kernel<64, 128, kManySegments, kNoWait>;
    case 4: return attn_step_sm100_kernel<128, 256, kOneUnit, kNoWait>;
    case 5: return attn_step_sm100_kernel<64, 256, kOneUnit, kNoWait>;
    case 6: return attn_step_sm100_kernel<128, 128, kOneUnit, kNoWait>;
    case 7: return attn_step_sm100_kernel<64, 128, kOneUnit, kNoWait>;
    case 9: return attn_step_sm100_kernel<64, 256, kPartOfTeam, kNoWait>;
    case 10: return attn_step_sm100_kernel<128, 128, kPartOfTeam, kNoWait>;
    case 11: return attn_step_sm100_kernel<64, 128, kPartOfTeam, kNoWait>;
    case 12: return attn_step_sm100_kernel<128, 256, kPartOfWideTeam, kNoWait>;
    case 13: return attn_step_sm100_kernel<64, 256, kPartOfWideTeam, kNoWait>;
    case 14: return attn_step_sm100_kernel<128, 128, kPartOfWideTeam, kNoWait>;
    case 15: return attn_step_sm100_kernel<64, 128, kPartOfWideTeam, kNoWait>;
    default: return nullptr;   // teams on two M tiles of heads of 128: their pieces have no room in shared memory
  }
}
AttnKernel kernel_of(int which) { return which >= kKernels ? kernel_of_waits<true>(which - kKernels) : kernel_of_waits<false>(which); }

// First use of an attention kernel on a context's device: checks the register budget and opts in to
// all the dynamic shared memory the device allows a block (less the kernel's static part).
int configure_kernel(dlm_ctx* ctx, int which, const void* kern) {
  if (ctx->attn_smem_limit[which] > 0) return DLM_OK;
  cudaFuncAttributes a;
  DLM_CUDA_TRY(cudaFuncGetAttributes(&a, kern));
  if (!register_budget_ok(a)) return DLM_ERR_UNSUPPORTED;
  const int limit = ctx->max_smem_optin - (int)a.sharedSizeBytes;
  if (limit <= 0) return DLM_ERR_UNSUPPORTED;
  DLM_CUDA_TRY(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, limit));
  if (which % kKernels >= 8 && which % kKernels < 12) DLM_CUDA_TRY(cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1));
  ctx->attn_smem_limit[which] = limit;
  return DLM_OK;
}

using Plan = dlm_attn_plan;

// Shared memory of a block: Q tiles, the K and V rings, barriers, flags, scheduling tables and up to
// 1023 bytes of alignment.  (Deeper rings were measured: 2 + 3 and 3 + 3 stages at head_dim 128 were
// 3 - 10 % slower on the configs' shapes, so the rest of the shared memory stays unused.)
bool plan_shared_memory(int smem_limit, int head_dim, int batch, Plan& pl) {
  const int tile = head_dim / 64 * kPanelBytes;
  const int stages = head_dim == 128 ? Geometry<128>::kStages : Geometry<64>::kStages;
  pl.smem_bytes = 1024 + (pl.n_mt + 2 * stages) * tile + kBarrierBytes + kFlagBytes +
                  (pl.team > 1 && !pl.wide ? kFoldBytes + team_bytes(head_dim, pl.team, (pl.rows + 31) & ~31) : pl.single ? 0 : 4 * sched_ints(batch));
  return pl.smem_bytes <= smem_limit;
}

// Device scratch of a call: room for the partial results of the split schedule and of teams through L2 whenever one of them is possible
// at all, whichever the hint and the cost estimate then pick.
struct WorkspaceSize {
  size_t o_bytes, ml_bytes;
};
WorkspaceSize workspace_size(const dlm_ctx* ctx, const dlm_kv_cache* cache, int nl, int n_q_heads, int q_cap) {
  const int rows_total = (n_q_heads / cache->n_kv_heads) * q_cap, sms = ctx->num_sms < kMaxGrid ? ctx->num_sms : kMaxGrid;
  const long long units = (long long)nl * cache->batch * cache->n_kv_heads * ((rows_total + 255) / 256);
  const size_t slots = units < 8LL * sms && units <= kDlmMaxSplitUnits ? 2 * (size_t)sms : 0, n_mt = rows_total > 128 ? 2 : 1;
  return {slots * n_mt * 128 * cache->head_dim * sizeof(float), slots * n_mt * 128 * 2 * sizeof(float)};
}

// Costs of a block's work in key tiles of two M tiles (2.2 us on a Dream-shaped layer): between units dealt whole and split, and between
// chunks of 256 and 128.
constexpr double kTileCost[2] = {0.86, 1.0};     // one key tile, for one / two M tiles: the softmax chain hardly gets longer
constexpr double kSplitCost[2] = {2.5, 4.0};     // the split schedule's partial store, wait and merge of one further piece ...
constexpr double kSplitPiece = 0.7;              // ... and of each piece beyond that
// With more units than SMs a block has whole units to compute while its first piece travels, and merges one unit at most.
// 40 layer-batched calls, split against whole: with two M tiles the split was 4 - 9 us slower where it saves one key tile a
// block, equal at two and 1 - 2 us faster at three (4 us at four: 5 layers x 2 x 419 rows 88.8 -> 84.5); with one M tile
// 2 - 4 us slower at one and two, equal at three, 1 - 2 us faster at four.
constexpr double kSplitManyCost[2] = {3.2, 2.7};

// A call of at most as many units as SMs in us, for each schedule, fitted to 515 calls (1 - 16 layers, 1 - 8 sequences, five models' heads of 128
// and 64, 8 - 200 active and 100 - 10000 cached rows) timed under every schedule, row chunk and team size that is possible, back to
// back and between projections (weighted 1 : 2, since most calls stand in a layer).  The teams' terms for rows and ragged tiles are rounded
// towards smaller chunks.  Between projections 28 of these calls were 3 - 34 % slower than before there were clusters, with costs that took heads
// of 64 for as dear as those of 128 and without teams through L2; now 10 are, by 3 - 7 %.  Back to back it was 79, now 18, most by 3 - 10 %;
// 8 - 32 units of 8 active rows at 4000 cached ones by 18 - 25 % (probably since a cluster waits for all of its SMs; not between projections).
struct CallShape {
  double t;      // key tiles of the block with the most, ragged ones by UnitTiles::cost
  double two;    // 1 with two M tiles a block, else 0
  double r;      // rows of a unit, in whole warps, / 128
  double d;      // head_dim / 128
  double g;      // blocks per SM
  double beyond; // 1 with more blocks than half of the SMs: the next call's cannot set themselves up beside them
};
double whole_us(const CallShape& c) { return 3.64 + c.t * (0.92 + 0.64 * c.two + 0.31 * c.d + 0.58 * c.g * c.d) + 0.73 * c.r; }
// full: the teams' part of the clusters that the device runs at a time; even: all blocks finish equally many columns
double team_us(const CallShape& c, int team, double full, bool even) {
  const double t = c.t * (1 + c.two);
  return 4.2 + t * (0.74 + 0.23 * c.d + 0.47 * c.d * c.g * c.g) + c.r * (1.2 + 0.9 * c.d) + 0.19 * team * full + (even ? 0.0 : 0.24) + 0.6 * c.beyond;
}
double wide_us(const CallShape& c) { return 5.08 + c.t * (1.16 + 0.62 * c.two + 0.4 * c.g * c.d) + 2.59 * c.r * c.d + 1.58 * c.beyond; }
// c.t: key tiles of a share, each counted in full; pieces: shares per unit
double split_us(const CallShape& c, double pieces) {
  return 8.42 + c.t * (1.04 + 0.59 * c.two - 0.36 * c.d + 1.11 * c.g * c.d) + 2.07 * c.two + 1.14 * pieces;
}
constexpr double kWholeCall = 3.2, kTileUs = 2.2;   // us of a call of more units than SMs: kWholeCall + kTileUs * its cost in key tiles

// A unit's key tiles: the cache's, then the fresh rows'.  (Where the keys are split over a block's two chains, half a tile takes nearly as long as
// a whole one.)
constexpr double kRagged = 0.5, kRaggedSplitKeys = 0.6;
struct UnitTiles {
  long long len, q_cap, box, n_cache, n;
  UnitTiles(long long len_, long long q_cap_) : len(len_), q_cap(q_cap_), box(q_cap_ < 128 ? q_cap_ : 128), n_cache((len_ + 127) / 128),
                                                n(n_cache + (q_cap_ + 127) / 128) {}
  // what tiles [from, to) cost: a ragged one `ragged` and the rest by its keys
  double cost(long long from, long long to, double ragged) const {
    double sum = 0;
    for (long long i = from; i < to; ++i) {
      const long long left = i < n_cache ? len - i * 128 : q_cap - (i - n_cache) * box, most = i < n_cache ? 128 : box;
      sum += ragged + (1.0 - ragged) / 128 * (double)(left < most ? left : most);
    }
    return sum;
  }
};

CallShape call_shape(const dlm_ctx* ctx, const Plan& pl, int head_dim, double tiles) {
  return {tiles, pl.n_mt == 2 ? 1.0 : 0.0, ((pl.rows + 31) & ~31) / 128.0, head_dim / 128.0, (double)pl.grid / ctx->num_sms, pl.grid * 2 > ctx->num_sms ? 1.0 : 0.0};
}

// The best plan of whole or split units with row chunks of `chunk_rows`, and its estimated cost.
double plan_chunked(const dlm_ctx* ctx, const dlm_kv_cache* cache, int nl, int n_q_heads, int q_cap, int len, int chunk_rows, Plan& pl) {
  pl.rows_total = (n_q_heads / cache->n_kv_heads) * q_cap;
  pl.chunk_rows = chunk_rows;
  pl.n_rc = (pl.rows_total + chunk_rows - 1) / chunk_rows;
  pl.rows = pl.rows_total < chunk_rows ? pl.rows_total : chunk_rows;
  pl.n_mt = (pl.rows + 127) / 128;
  const long long units = (long long)nl * cache->batch * cache->n_kv_heads * pl.n_rc;
  const int sms = ctx->num_sms < kMaxGrid ? ctx->num_sms : kMaxGrid;
  const bool may_split = units < 8LL * sms && units <= kDlmMaxSplitUnits;
  const long long tiles_unit = UnitTiles(len, q_cap).n;
  const double tile = kTileCost[pl.n_mt - 1];
  // units dealt whole: idle SMs when they do not fill a whole number of waves
  double best = (double)(((units + sms - 1) / sms) * tiles_unit) * tile;
  pl.whole_units = 1;
  pl.team = 1;
  pl.wide = 0;
  pl.grid = (int)(units < sms ? units : sms);
  if (!may_split) return best;
  // units split across blocks: equal shares, but a partial store per block and a merge per unit
  for (long long shares = units + 1; shares <= sms && shares <= units * tiles_unit; ++shares) {
    const double t = (double)((units * tiles_unit + shares - 1) / shares) * tile + kSplitCost[pl.n_mt - 1] +
                     kSplitPiece * ((double)shares / (double)units - 1.0);
    if (t < best) { best = t; pl.whole_units = 0; pl.grid = (int)shares; }
  }
  if (units > sms) {   // more units than SMs: the only split is over all SMs
    const double t = (double)((units * tiles_unit + sms - 1) / sms) * tile + kSplitManyCost[pl.n_mt - 1];
    if (t < best) { best = t; pl.whole_units = 0; pl.grid = sms; }
  }
  return best;
}

// The us of a plan of whole or split units of that cost.
double chunked_us(const dlm_ctx* ctx, const dlm_kv_cache* cache, int nl, int q_cap, int len, double cost, const Plan& pl) {
  const long long units = (long long)nl * cache->batch * cache->n_kv_heads * pl.n_rc;
  const UnitTiles tiles(len, q_cap);
  if (units > ctx->num_sms) return kWholeCall + kTileUs * cost;
  if (pl.whole_units) return whole_us(call_shape(ctx, pl, cache->head_dim, tiles.cost(0, tiles.n, kRagged)));
  return split_us(call_shape(ctx, pl, cache->head_dim, (double)((units * tiles.n + pl.grid - 1) / pl.grid)), (double)pl.grid / (double)units);
}

// How many clusters of `team` blocks, one block per SM, the device runs at a time (0: none).  It depends on which SMs a die has: 74 of 2,
// 45 of 3, 33 of 4, 26 of 5, 22 of 6, 15 of 7 - 9, 7 of 16 on one card.
int team_clusters(dlm_ctx* ctx, int team) {
  int& known = ctx->attn_clusters[team];
  if (known == 0) {
    constexpr int kTeamKernel = 10;   // head_dim 128, one M tile (kernel_index)
    const AttnKernel kern = kernel_of(kTeamKernel);
    known = -1;
    if (configure_kernel(ctx, kTeamKernel, reinterpret_cast<const void*>(kern)) == DLM_OK) {
      cudaLaunchConfig_t cfg = {};
      cfg.gridDim = dim3(team);
      cfg.blockDim = dim3(kThreads);
      cfg.dynamicSmemBytes = ctx->attn_smem_limit[kTeamKernel];
      cudaLaunchAttribute attr[1];
      attr[0].id = cudaLaunchAttributeClusterDimension;
      attr[0].val.clusterDim.x = team;
      attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
      cfg.attrs = attr;
      cfg.numAttrs = 1;
      int n = 0;
      if (cudaOccupancyMaxActiveClusters(&n, kern, &cfg) == cudaSuccess && n > 0) known = n;
      else cudaGetLastError();
    }
  }
  return known > 0 ? known : 0;
}

// The best plan with teams on row chunks of `chunk_rows`, and its estimated us (negative: there is none).
double plan_teams(dlm_ctx* ctx, const dlm_kv_cache* cache, int nl, int n_q_heads, int q_cap, int len, int chunk_rows, Plan& pl) {
  pl.rows_total = (n_q_heads / cache->n_kv_heads) * q_cap;
  pl.chunk_rows = chunk_rows;
  pl.n_rc = (pl.rows_total + chunk_rows - 1) / chunk_rows;
  pl.rows = pl.rows_total < chunk_rows ? pl.rows_total : chunk_rows;
  pl.n_mt = (pl.rows + 127) / 128;
  pl.whole_units = pl.single = 1;
  pl.wide = 0;
  const long long units = (long long)nl * cache->batch * cache->n_kv_heads * pl.n_rc;
  const UnitTiles tiles(len, q_cap);
  Plan at = pl;
  double best = -1;
  for (int team = 2; team <= kTeamMax && team <= ctx->attn_team_max && team <= tiles.n && units * team <= ctx->num_sms; ++team) {
    at.team = team;
    const int clusters = team_clusters(ctx, team);
    if (!plan_shared_memory(ctx->max_smem_optin, cache->head_dim, cache->batch, at) || units > clusters) continue;
    double most = 0;
    for (int r = 0; r < team; ++r)
      most = fmax(most, tiles.cost(tiles.n * r / team, tiles.n * (r + 1) / team, pl.n_mt == 1 ? kRaggedSplitKeys : kRagged));
    at.grid = (int)units * team;
    const double t = team_us(call_shape(ctx, at, cache->head_dim, most), team, (double)units / clusters, (cache->head_dim / 8) % team == 0);
    if (best < 0 || t < best) {
      best = t;
      pl.team = team;
      pl.grid = (int)units * team;
    }
  }
  return best;
}

// The best plan with teams that exchange through L2, and its estimated us (negative: there is none): the smallest team that reaches the
// fewest key tiles per block.  They meet in memory, so all blocks have to run at a time: one per SM.
double plan_wide(dlm_ctx* ctx, const dlm_kv_cache* cache, int nl, int n_q_heads, int q_cap, int len, int chunk_rows, Plan& pl) {
  pl.rows_total = (n_q_heads / cache->n_kv_heads) * q_cap;
  pl.chunk_rows = chunk_rows;
  pl.n_rc = (pl.rows_total + chunk_rows - 1) / chunk_rows;
  pl.rows = pl.rows_total < chunk_rows ? pl.rows_total : chunk_rows;
  pl.n_mt = (pl.rows + 127) / 128;
  pl.whole_units = pl.single = pl.wide = 1;
  const int sms = ctx->num_sms < kMaxGrid ? ctx->num_sms : kMaxGrid;
  const long long units = (long long)nl * cache->batch * cache->n_kv_heads * pl.n_rc;
  const UnitTiles tiles(len, q_cap);
  if (units * 2 > sms) return -1;
  long long team = ctx->attn_team_max < kTeamMax ? ctx->attn_team_max : kTeamMax;
  if (team > sms / units) team = sms / units;
  if (team > tiles.n) team = tiles.n;
  if (team <= 1) return -1;
  const long long per_block = (tiles.n + team - 1) / team;
  team = (tiles.n + per_block - 1) / per_block;
  if (team <= 1) return -1;
  pl.team = (int)team;
  pl.grid = (int)(units * team);
  double most = 0;
  for (int r = 0; r < team; ++r) most = fmax(most, tiles.cost(tiles.n * r / team, tiles.n * (r + 1) / team, kRagged));
  return wide_us(call_shape(ctx, pl, cache->head_dim, most));
}

// Row chunks of 256 (two M tiles sharing every K/V tile) read K/V once per KV head and cost little more per key tile than
// chunks of 128; those double the units that can be spread over the SMs and halve every partial result, the second read of
// K/V coming from L2.  Teams also come with chunks of 96 and 64, whose partial results are smaller still (one sequence of Dream,
// 224 rows a KV head, at 1024 cached rows: 9.3 us in chunks of 128, 8.7 of 96, 8.5 of 64, all in teams of 4; at 4096: 15.7, 12.5, 13.2 in
// the best teams that fit).  Whichever schedule of any has the least estimated cost, from the caller's cache length hint.
Plan make_plan(dlm_ctx* ctx, const dlm_kv_cache* cache, int nl, int n_q_heads, int q_cap, int cache_len_hint) {
  const int len = (cache_len_hint > 0 && cache_len_hint < cache->capacity) ? cache_len_hint : cache->capacity;
  Plan pl, other;
  double cost = plan_chunked(ctx, cache, nl, n_q_heads, q_cap, len, 256, pl);
  if (pl.n_mt == 2) {
    const double c = plan_chunked(ctx, cache, nl, n_q_heads, q_cap, len, 128, other);
    if (c < cost) { pl = other; cost = c; }
  }
  pl.single = pl.whole_units && (long long)nl * cache->batch * cache->n_kv_heads * pl.n_rc <= pl.grid;
  cost = chunked_us(ctx, cache, nl, q_cap, len, cost, pl);
  bool forced = ctx->attn_team_force;
  for (int chunk : {256, 128, 96, 64}) {
    if (chunk < 256 && pl.rows_total <= chunk) continue;   // all rows in one chunk: as with 256
    const double c = plan_teams(ctx, cache, nl, n_q_heads, q_cap, len, chunk, other);
    if (c >= 0 && (c < cost || forced)) { pl = other; cost = c; forced = false; }
  }
  for (int chunk : {256, 128}) {
    if (chunk < 256 && pl.rows_total <= chunk) continue;
    const double c = plan_wide(ctx, cache, nl, n_q_heads, q_cap, len, chunk, other);
    if (c >= 0 && (c < cost || forced)) { pl = other; cost = c; forced = false; }
  }
  const WorkspaceSize ws = workspace_size(ctx, cache, nl, n_q_heads, q_cap);
  pl.ws_o_bytes = ws.o_bytes;
  pl.ws_ml_bytes = ws.ml_bytes;
  return pl;
}

}  // namespace

extern "C" size_t dlm_attn_workspace_bytes(const dlm_ctx* ctx, const dlm_kv_cache* cache, int n_layers_in_call,
                                           int n_q_heads, int q_cap) {
  if (!ctx || !cache || n_layers_in_call <= 0 || n_q_heads <= 0 || q_cap <= 0 || cache->n_kv_heads <= 0 ||
      cache->batch <= 0 || n_q_heads % cache->n_kv_heads != 0)
    return 0;
  const WorkspaceSize ws = workspace_size(ctx, cache, n_layers_in_call, n_q_heads, q_cap);
  return ws.o_bytes + ws.ml_bytes + 256;
}

extern "C" int dlm_selftest_attn_schedule(const dlm_ctx* ctx, const dlm_kv_cache* cache, int n_layers_in_call, int n_q_heads,
                                          int q_cap, int cache_len_hint, int* grid, int* team, int* whole_units,
                                          int* chunk_rows) {
  if (!ctx || !cache || !grid || !team || !whole_units || !chunk_rows) return DLM_ERR_NULL;
  if (n_layers_in_call <= 0 || n_q_heads <= 0 || q_cap <= 0 || cache->n_kv_heads <= 0 || cache->batch <= 0 ||
      cache->capacity <= 0 || n_q_heads % cache->n_kv_heads != 0)
    return DLM_ERR_SHAPE;
  // (a plan may ask the device, once, how many clusters fit)
  const Plan pl = make_plan(const_cast<dlm_ctx*>(ctx), cache, n_layers_in_call, n_q_heads, q_cap, cache_len_hint);
  *grid = pl.grid;
  *team = pl.team;
  *whole_units = pl.whole_units;
  *chunk_rows = pl.chunk_rows;
  return DLM_OK;
}

extern "C" int dlm_freecache_attn_step(dlm_ctx* ctx, const dlm_kv_cache* cache, int layer_begin, int layer_end,
                                       const void* q, const void* k_new, const void* v_new, int n_q_heads,
                                       int q_cap, const int32_t* q_len, float softmax_scale, int cache_len_hint,
                                       void* out, float* lse, void* workspace, size_t workspace_bytes,
                                       void* stream) {
  if (!ctx || !cache || !cache->k || !cache->v || !cache->cache_len || !q || !k_new || !v_new || !out)
    return DLM_ERR_NULL;
  if (cache->n_layers <= 0 || cache->batch <= 0 || cache->n_kv_heads <= 0 || cache->capacity <= 0 ||
      n_q_heads <= 0 || q_cap <= 0)
    return DLM_ERR_SHAPE;
  if (layer_begin < 0 || layer_end > cache->n_layers || layer_begin >= layer_end) return DLM_ERR_SHAPE;
  const int D = cache->head_dim;
  if (D != 64 && D != 128) return DLM_ERR_UNSUPPORTED;
  if (n_q_heads % cache->n_kv_heads != 0) return DLM_ERR_UNSUPPORTED;
  const int group = n_q_heads / cache->n_kv_heads;
  if (q_cap > kMaxQCap || (long long)group * q_cap > (1 << 20) || cache->batch > kMaxBatch) return DLM_ERR_UNSUPPORTED;
  if (((uintptr_t)cache->k | (uintptr_t)cache->v | (uintptr_t)q | (uintptr_t)k_new | (uintptr_t)v_new |
       (uintptr_t)out) & 15)
    return DLM_ERR_UNSUPPORTED;
  DLM_DEVICE_TRY(ctx);
  const int nl = layer_end - layer_begin;
  const size_t need = dlm_attn_workspace_bytes(ctx, cache, nl, n_q_heads, q_cap);
  if (!workspace || workspace_bytes < need || ((uintptr_t)workspace & 255)) return DLM_ERR_WORKSPACE;
  const bool nw = ctx->wait_limit_ns == 0;
  // the plan of the last call serves the calls of a model's other layers too
  const dlm_attn_plan_key key = {nl, cache->batch, cache->n_kv_heads, cache->capacity, D, n_q_heads, q_cap, cache_len_hint,
                                 ctx->attn_team_max, ctx->attn_team_force ? 1 : 0, nw ? 1 : 0};
  if (memcmp(&key, &ctx->attn_plan_key, sizeof key) != 0) {
    Plan made = make_plan(ctx, cache, nl, n_q_heads, q_cap, cache_len_hint);
    const int which = kernel_index(D, made, nw);
    const int rc = configure_kernel(ctx, which, reinterpret_cast<const void*>(kernel_of(which)));
    if (rc != DLM_OK) return rc;
    if (!plan_shared_memory(ctx->attn_smem_limit[which], D, cache->batch, made)) return DLM_ERR_UNSUPPORTED;
    ctx->attn_plan = made;
    ctx->attn_plan_key = key;
  }
  const Plan& pl = ctx->attn_plan;
  {  // the split schedule counts (unit, key tile) items in 32 bits
    const long long tiles_per_unit = (cache->capacity + 127) / 128 + (q_cap + 127) / 128 + 1;
    if (!pl.whole_units && (long long)nl * cache->batch * cache->n_kv_heads * pl.n_rc * tiles_per_unit >= (1LL << 30))
      return DLM_ERR_UNSUPPORTED;
  }

  AttnParams p;
  p.cache_len = cache->cache_len;
  p.q_len = q_len;
  p.out = static_cast<__nv_bfloat16*>(out);
  p.lse = lse;
  p.ws_o = static_cast<float*>(workspace);
  p.ws_ml = reinterpret_cast<float*>(static_cast<uint8_t*>(workspace) + pl.ws_o_bytes);
  p.nl = nl;
  p.layer_begin = layer_begin;
  p.batch = cache->batch;
  p.n_kv_heads = cache->n_kv_heads;
  p.n_q_heads = n_q_heads;
  p.group = group;
  p.capacity = cache->capacity;
  p.q_cap = q_cap;
  p.rows = pl.rows;
  p.chunk_rows = pl.chunk_rows;
  p.rows_total = pl.rows_total;
  p.n_rc = pl.n_rc;
  p.n_mt = pl.n_mt;
  p.fresh_box = q_cap < 128 ? q_cap : 128;
  p.whole_units = pl.whole_units;
  p.team = pl.team;
  p.smem_bytes = pl.smem_bytes;
  const float scale = softmax_scale > 0.f ? softmax_scale : 1.0f / sqrtf((float)D);
  p.by_batch = make_fast_div(p.batch);
  p.by_rc = make_fast_div(p.n_rc);
  p.by_kv_heads = make_fast_div(p.n_kv_heads);
  p.by_q_cap = make_fast_div(q_cap);
  p.by_team = make_fast_div(pl.team);
  p.by_live = make_fast_div((pl.rows + 31) & ~31);
  // a hint of 1 is how a caller says that nothing is cached yet (0 leaves the length open)
  p.hint_len = cache_len_hint == 1 ? 0 : cache_len_hint > 0 && cache_len_hint < cache->capacity ? cache_len_hint : cache->capacity;
  p.scale_log2 = scale * 1.4426950408889634f;
  p.status = &ctx->words->status;
  p.tickets = ctx->words->attn_unit_tickets;

  CUtensorMap tm_q, tm_kc, tm_vc, tm_kn, tm_vn;
  const long long slabs_new = (long long)nl * cache->batch * cache->n_kv_heads;
  const long long slabs_cache = (long long)cache->n_layers * cache->batch * cache->n_kv_heads;
  const int cache_box = cache->capacity < 128 ? cache->capacity : 128;
  int rc = encode_map(ctx, &tm_q, q, D, pl.rows_total, slabs_new, pl.rows < 128 ? pl.rows : 128);
  if (rc == DLM_OK) rc = encode_map(ctx, &tm_kc, cache->k, D, cache->capacity, slabs_cache, cache_box);
  if (rc == DLM_OK) rc = encode_map(ctx, &tm_vc, cache->v, D, cache->capacity, slabs_cache, cache_box);
  if (rc == DLM_OK) rc = encode_map(ctx, &tm_kn, k_new, D, q_cap, slabs_new, p.fresh_box);
  if (rc == DLM_OK) rc = encode_map(ctx, &tm_vn, v_new, D, q_cap, slabs_new, p.fresh_box);
  if (rc != DLM_OK) return rc;

  cudaStream_t s = static_cast<cudaStream_t>(stream);
  DLM_CUDA_TRY(dlm_launch_cluster(kernel_of(kernel_index(D, pl, nw)), dim3(pl.grid), dim3(kThreads), (size_t)p.smem_bytes, s,
                                  (unsigned int)(pl.wide ? 1 : pl.team), tm_q, tm_kc, tm_vc, tm_kn, tm_vn, p));
  return dlm_launch_ok(ctx, 1);
}
