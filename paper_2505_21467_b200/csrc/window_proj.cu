// dlm_window_qkv_project / dlm_window_out_project: the dense projections either side of the attention
// step (Table 1 rows "Q/K/V projection" and "output projection"; Sec. 3.2.1 "Windowed Re-computation":
// the window's K/V are recomputed from its hidden states in every step).
//
// Y[rows x features] = X[rows x K] W[features x K]^T.  Activation rows are the MMA's M (one row per TMEM lane and
// epilogue thread), N features of one tile its N; a block (pair) sums the whole of K, so there is no workspace, no exchange
// between blocks and one summation order.  With the row in a thread, a head's features lie along the thread's registers: the
// rotary embedding pairs two of its own registers and every store is 16 bytes of one row.
//   up to 64 rows:  one block per tile, M = 64 (rows beyond the call's are never loaded, never read back), tiles of
//                   16 .. 128 features.  Bound by streaming the weights from HBM.
//   more rows:      chunks of up to 256 rows, each by a pair of blocks (cta_group::2, M = 256; M = 128 up to 128 rows): a block holds its half of
//                   the rows and its half of the tile's features, so it takes in half of what two separate blocks would;
//                   tiles of 64 .. 512 features.  Bound by the SM's intake from L2 at small tiles, by the tensor pipe from 256.
//                   Widths of 192 and beyond 256 exist so that a call's tiles fill the pairs once: 1280 rows of 4608 features
//                   are 90 tiles of 256, two rounds over 74 pairs (52.1 us), and 60 tiles of 384, one round (36.2 us).
// Measured (one call per layer over 28 / 32 layers' own weights, back to back, rotary embedding and staging on; before this
// form: one 128-feature block per tile with K split over blocks and partial tiles through the workspace):
//   rows x K -> features     32 x 3584 -> 4608   12.6 -> 8.5 us (3.9 TB/s of weights)    256 x 3584 -> 4608   25.1 -> 12.4 us
//                           256 x 4096 -> 12288   167 -> 28.6 us (900 TFLOP/s)          1280 x 3584 -> 4608   237 -> 36.1 us (1170 TFLOP/s)
// at SM clocks of 1927 - 1965 MHz (bursts of 12 ms); one call after the other for longer, the power cap brings 1280 rows to 1670
// MHz and 41 us, 256 x 4096 -> 12288 to 1600 MHz and 32 us.
// (Prefetching the tile's weights into L2 before the grid dependency wait, tried by rows and by stages, cost more than
// the head start gave: the stage loads queue behind it.  31 us without, 38 with, at LLaDA's 256 rows.  Prefetching
// 8 - 32 stages ahead as the loads go: 0 - 4 us slower too.)
// Both operands are K-major as they lie in memory.  A tensor map with K split into (64-element panel, panel index) lets one
// copy bring several panels of a stage: a producer's loop costs 200 - 340 cycles per iteration whatever it copies
// (barrier wait 100, expect 40, each copy 55), which bound the kernel when every 64 elements of K took an iteration.
//
// Block = 8 warps: warp 0 weight producer, warp 1 activation producer, warp 2 tcgen05.mma issuer (of the leader block),
// warp 3 TMEM and, for activations in many pieces, half of their copies, warps 4-7 the epilogue's tables; all eight write
// the results.
#include <cuda_bf16.h>

#include "common.cuh"
#include "sm100_ptx.cuh"

namespace {

using namespace sm100;

constexpr int kThreads = 256;
constexpr int kPanel = 64;                  // K elements of a 128-byte swizzled panel
constexpr int kMaxStages = 8;
constexpr int kMaxN = 512;                  // features of the widest tile (a block's whole TMEM)
constexpr int kMaxActRows = 256;            // rows of an output projection (one pair sees them all)
constexpr int kAuxBytes = 16 * kMaxStages + 16 + 32 + kMaxN * 4 + 128 * 32;   // barriers, flags, bias of the tile, row table

struct ProjParams {
  // destination: mode 0 = Q/K/V head by head ([B][heads][q_cap][D] each), mode 1 = row-major [rows][n_out]
  int mode;
  __nv_bfloat16* q_out;
  __nv_bfloat16* k_out;
  __nv_bfloat16* v_out;
  const __nv_bfloat16* bias;   // [n_out] or nullptr
  const float* rope_cos;       // mode 0: rotary embedding of the query and key heads, fp32 [B][q_cap][head_dim / 2],
  const float* rope_sin;       // or both nullptr
  // mode 0: K/V rows are also staged in the cache (one layer: [B][n_kv_heads][capacity][head_dim]) at row
  // cache_len[b] + i, the slot the commit's window mode uses; nullptr: no staging
  __nv_bfloat16* stage_k;
  __nv_bfloat16* stage_v;
  const int32_t* cache_len;    // [B]
  const int32_t* q_len;        // [B] rows of the window that are active (staged), or nullptr: all q_cap
  int capacity;
  int rows_total, q_cap, n_q_heads, n_kv_heads, head_dim, n_out, k_total;
  int batch;
  int act_heads;               // activations are [B][act_heads][q_cap][D] (0: plain [rows][K])
  int rc;                      // rows per block (a multiple of 8)
  int x_box_rows;              // rows per copy of head-split activations (rc: one copy brings all)
  int pieces;                  // copies that bring a panel of a block's activation rows
  int half_rows;               // features of a group's half: W is seen as [groups][2][half_rows][K]
  int w_box_rows;              // tiles of units: features per copy of the weights (32, or 64 where units lie in pairs)
  int n_stages, aux_offset;
  int head_shift;              // log2(head_dim), or -1
  int* status;
};

__host__ __device__ constexpr bool tile_of_units(int n) { return n == 192 || n > 256; }

// Where a row of the block goes: element offsets within q_out (or y), k_out / v_out and the staged layer (-1: not staged).
struct __align__(16) RowEntry {
  long long q, kv, stage;
};

// Feature tiles.  A tile takes N / 2 consecutive features from each half of a group of 2 half_rows features; with
// half_rows = head_dim / 2 a tile narrower than a head then holds both partners of every rotary pair it has.
// PAIR: each block of the pair loads one of the two halves, and D's columns are [half 0 | half 1] either way.
template <int N, int M, int KP>
__global__ void __launch_bounds__(kThreads, 1)
window_proj_kernel(const __grid_constant__ CUtensorMap tm_w, const __grid_constant__ CUtensorMap tm_x, const ProjParams p) {
  extern __shared__ uint8_t smem_raw[];
  constexpr bool PAIR = M > 64;
  constexpr int kRowTile = M == 64 ? 64 : M / 2;            // rows of the MMA in this block
  constexpr int kBlockN = PAIR ? N / 2 : N;                 // features whose weights this block loads
  constexpr uint32_t kWBytes = (uint32_t)KP * kBlockN * 128u;
  constexpr uint32_t kTmemCols = N <= 32 ? 32 : N <= 64 ? 64 : N <= 128 ? 128 : N <= 256 ? 256 : 512;
  // Tiles of units: a unit is 32 features of a group's first half and the 32 of the second half that they are paired with.
  // One MMA takes up to 256 columns; a wider tile is two, each [first halves | second halves] of its units.
  constexpr bool UNITS = tile_of_units(N);
  constexpr int kN0 = N > 256 ? (N / 64 + 1) / 2 * 64 : N, kN1 = N - kN0;
  const uint32_t pad = (1024u - (smem_u32(smem_raw) & 1023u)) & 1023u;
  const uint32_t base = smem_u32(smem_raw) + pad;
  const uint32_t x_panel = (uint32_t)p.rc * 128u, x_bytes = KP * x_panel;
  const uint32_t stage_bytes = kWBytes + x_bytes;
  // stages (and room behind them for the MMA's reads of rows that no copy fills, see make_proj_plan), then barriers, flags,
  // the tile's bias and the row table
  const uint32_t aux = p.aux_offset;
  const uint32_t bar_full = base + aux, bar_empty = bar_full + 8 * kMaxStages, bar_done = bar_full + 16 * kMaxStages;
  int* const flags = reinterpret_cast<int*>(smem_raw + pad + aux + 16 * kMaxStages + 16);
  volatile int* const abort_ptr = flags;
  volatile int* const never_ptr = flags + 1;
  uint32_t* const tmem_slot = reinterpret_cast<uint32_t*>(flags + 2);
  float* const bias_s = reinterpret_cast<float*>(flags + 8);
  RowEntry* const row_s = reinterpret_cast<RowEntry*>(bias_s + kMaxN);

  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const uint32_t rank = PAIR ? cluster_ctarank() : 0u;
  const int tile = PAIR ? (int)blockIdx.x >> 1 : (int)blockIdx.x;
  const int row0 = ((int)blockIdx.z * (PAIR ? 2 : 1) + (int)rank) * p.rc;   // this block's first row
  const int per_group = UNITS ? 1 : p.half_rows / (N / 2);
  const int group = tile / per_group, a0 = (tile % per_group) * (N / 2);
  const int feat0 = group * 2 * p.half_rows + a0, feat1 = feat0 + p.half_rows;   // first features of the two halves
  const int unit_shift = p.half_rows == 64 ? 1 : 0;          // UNITS: log2 of a group's units
  auto feature = [&](int c) {                                // output feature of column c
    if (!UNITS) return c < N / 2 ? feat0 + c : feat1 + c - N / 2;
    const int h = c < kN0 ? kN0 / 2 : kN1 / 2, cc = c < kN0 ? c : c - kN0, second = cc >= h ? 1 : 0;
    const int r = (c < kN0 ? 0 : kN0 / 2) + cc - second * h, unit = tile * (N / 64) + (r >> 5);
    return ((2 * (unit >> unit_shift) + second) << (5 + unit_shift)) + ((unit & unit_shift) << 5) + (r & 31);
  };
  const int n_panels = p.k_total / kPanel;
  const int n_k = (n_panels + KP - 1) / KP;                 // stages' worth of K; panels beyond the last are zero-filled

  if (tid == 0) {
    *abort_ptr = 0; *never_ptr = 0;
    for (int i = 0; i < p.n_stages; ++i) {
      mbar_init(bar_full + 8 * i, 2);
      mbar_init(bar_empty + 8 * i, 1);
    }
    mbar_init(bar_done, 1);
    mbar_fence_init();
    fence_proxy_async_smem();
  }
  if (warp == 0 && lane == 0) prefetch_tensormap(&tm_w);
  if (warp == 1 && lane == 0) prefetch_tensormap(&tm_x);
  if (warp == 3) {
    if (PAIR) {
      tmem_alloc_pair(smem_u32(tmem_slot), kTmemCols);
      tmem_relinquish_pair();
    } else {
      tmem_alloc(smem_u32(tmem_slot), kTmemCols);
      tmem_relinquish();
    }
  }
  __syncwarp();
  tc_fence_before_sync();
  if (PAIR) cluster_sync(); else __syncthreads();   // barriers exist (in both blocks), TMEM is there
  tc_fence_after_sync();
  const uint32_t tmem = *tmem_slot;
  dlm_grid_dependency_wait();
  dlm_trigger_dependents();

  int issued = 0;   // stages this producer warp has issued
  if (p.pieces > 1 && (warp == 1 || warp == 3)) {
    // ================================================================= activations in pieces of sequences
    // Head-split activations [B][heads][q_cap][D] whose rows of a block end inside a sequence.  A lane of warps 1 and 3 has its
    // copy of every stage, its coordinates but the panel's known beforehand (all by one lane, with the divisions in the loop
    // below: 125 cycles a copy).
    const uint32_t full0 = PAIR ? map_shared_rank(bar_full, 0) : bar_full;
    const int head_panels = p.head_dim / kPanel, item = (lane << 1) + (warp >> 1);
    const int my_kp = item / p.pieces, my_row = (item - my_kp * p.pieces) * p.x_box_rows;
    const int z = (row0 + my_row) / p.q_cap, y = row0 + my_row - z * p.q_cap;
    int head = my_kp / head_panels, panel = my_kp - head * head_panels, s = 0, round = 0;
    bool ok = true;
    for (int kc = 0; kc < n_k; ++kc) {
      if (round > 0) ok = mbar_wait_warp(bar_empty + 8 * s, (round - 1) & 1, abort_ptr);
      if (!ok) break;
      if (warp == 1 && rank == 0 && lane == 0) mbar_expect_tx(bar_full + 8 * s, x_bytes * 2u);   // pieces: always a pair
      __syncwarp();
      if (my_kp < KP)
        tma_load_4d<PAIR>(base + s * stage_bytes + my_kp * x_panel + my_row * 128, &tm_x, full0 + 8 * s, panel * kPanel, y, head, z);
      for (panel += KP; panel >= head_panels; panel -= head_panels) ++head;
      __syncwarp();
      ++issued;
      if (++s == p.n_stages) { s = 0; ++round; }
    }
  } else if (warp < 2) {
    // ================================================================= producers (0: weights, 1: activations)
    const uint32_t bytes = (warp == 0 ? kWBytes : x_bytes) * (PAIR ? 2u : 1u);   // what the leader's barrier gets from both blocks
    const uint32_t full0 = PAIR ? map_shared_rank(bar_full, 0) : bar_full;
    const int head_panels = p.act_heads ? p.head_dim / kPanel : 1;
    int head = 0, panel = 0;                                // head-split activations: where the next K panel lies
    const int y0 = p.batch > 1 ? row0 % p.q_cap : row0, z0 = p.batch > 1 ? row0 / p.q_cap : 0;
    bool ok = true;
    int s = 0, round = 0;
    for (int kc = 0; kc < n_k; ++kc) {
      if (round > 0) ok = mbar_wait_warp(bar_empty + 8 * s, (round - 1) & 1, abort_ptr);
      if (!ok) break;
      if (elect_one_sync()) {
        if (rank == 0) mbar_expect_tx(bar_full + 8 * s, bytes);
        const uint32_t dst = base + s * stage_bytes, bar = full0 + 8 * s;
        if (warp == 0 && UNITS) {
          for (int r = 0; r < kBlockN; r += p.w_box_rows) {   // units beyond the last are zero-filled
            const int unit = tile * (N / 64) + (r >> 5);
            tma_load_5d<PAIR>(dst + x_bytes + r * 128, &tm_w, bar, 0, (unit & unit_shift) << 5, (int)rank, kc, unit >> unit_shift);
          }
        } else if (warp == 0) {
          tma_load_5d<PAIR>(dst + x_bytes, &tm_w, bar, 0, a0, PAIR ? (int)rank : 0, kc * KP, group);
        } else if (p.act_heads == 0) {
          tma_load_4d<PAIR>(dst, &tm_x, bar, 0, row0, kc * KP, 0);
        } else {
          // activations [B][heads][q_cap][D]: panel k belongs to head k / (D / 64); rows of a box are (sequence, row)
          int h = head, pn = panel;
          for (int kp = 0; kp < KP; ++kp) {
            tma_load_4d<PAIR>(dst + kp * x_panel, &tm_x, bar, pn * kPanel, y0, h, z0);
            if (++pn == head_panels) { pn = 0; ++h; }
          }
        }
      }
      for (int kp = 0; kp < KP; ++kp)
        if (++panel == head_panels) { panel = 0; ++head; }
      __syncwarp();
      ++issued;
      if (++s == p.n_stages) { s = 0; ++round; }
    }
  } else if (warp == 2 && rank == 0) {
    // ================================================================= MMA issuer
    const uint32_t idesc = make_idesc_bf16(M, (uint32_t)kN0, 0), idesc1 = make_idesc_bf16(M, (uint32_t)(kN1 ? kN1 : 64), 0);
    const uint64_t desc = make_smem_desc_sw128(base, 16, 1024);
    const uint32_t desc_lo = (uint32_t)desc, desc_hi = (uint32_t)(desc >> 32);
    // One lane runs the whole loop, waits included, so that the MMAs of a stage follow one another at the tensor pipe's rate: with
    // the warp taking part in every wait and one lane elected per stage, a stage of 16 MMAs of 64 x 32 x 16 took 710 cycles, 320
    // more than the pipe needs (32 x 3584 -> 4608: 9.3 us, now 8.5; 32 x 3584 -> 3584: 8.5, now 7.5; with the weights in L2 8.1, now
    // 6.8).  Whether the next stage is there too is asked before this one's MMAs are issued, which hides the answer's latency.
    auto issue = [&](uint32_t off, bool first) {
      const uint32_t a_lo = desc_lo + (off >> 4), b_lo = a_lo + (x_bytes >> 4);
#pragma unroll
      for (int kp = 0; kp < KP; ++kp) {
#pragma unroll
        for (int k = 0; k < kPanel / 16; ++k) {
          const uint32_t add = !first || kp > 0 || k > 0 ? 1u : 0u, ka = a_lo + kp * (x_panel >> 4) + 2 * k, kb = b_lo + kp * (kBlockN * 8) + 2 * k;
          mma_ss_lo<PAIR>(tmem, ka, kb, desc_hi, idesc, add);
          if (kN1) mma_ss_lo<PAIR>(tmem + kN0, ka, kb + kN0 / 2 * 8, desc_hi, idesc1, add);
        }
      }
    };
    if (n_k <= 2) {   // K in one or two stages, each with a buffer of its own: nothing to overlap, and this way it takes 0.1 us less
      bool ok = true;
      for (int kc = 0; ok && kc < n_k; ++kc) {
        ok = mbar_wait_warp(bar_full + 8 * kc, 0, abort_ptr);
        tc_fence_after_sync();
        if (ok && elect_one_sync()) issue(kc * stage_bytes, kc == 0);
        __syncwarp();
      }
      if (elect_one_sync()) { if (PAIR) tc_commit_pair(bar_done); else tc_commit(bar_done); }
    } else if (elect_one_sync()) {
      int s = 0, round = 0;
      uint32_t off = 0;
      bool here = false;   // the stage's data has been seen to be there
      for (int kc = 0; kc < n_k; ++kc) {
        if (!here && !mbar_wait(bar_full + 8 * s, round & 1, abort_ptr)) break;
        tc_fence_after_sync();
        const uint32_t cur = off, bar = bar_empty + 8 * s;
        off += stage_bytes;
        if (++s == p.n_stages) { s = 0; off = 0; ++round; }
        here = kc + 1 < n_k && mbar_test_wait(bar_full + 8 * s, round & 1);
        issue(cur, kc == 0);
        if (PAIR) tc_commit_pair(bar); else tc_commit(bar);
      }
      if (PAIR) tc_commit_pair(bar_done); else tc_commit(bar_done);
    }
    __syncwarp();
  } else if (warp >= 4) {
    // ================================================================= tables of the epilogue
    const int t = tid - 128;
    for (int c = t; c < N; c += 128) bias_s[c] = p.bias && (!UNITS || feature(c) < p.n_out) ? __bfloat162float(p.bias[feature(c)]) : 0.f;
    const int row = row0 + t;
    if (t < p.rc && row < p.rows_total) {
      const int b = row / p.q_cap, i = row - b * p.q_cap;
      RowEntry e;
      e.q = p.mode == 1 ? (long long)row * p.n_out : ((long long)b * p.n_q_heads * p.q_cap + i) * p.head_dim;
      e.kv = ((long long)b * p.n_kv_heads * p.q_cap + i) * p.head_dim;
      e.stage = -1;   // cache row to stage at: none for an inactive row or one without room (reported)
      if (p.stage_k && feature(N - 1) >= p.n_q_heads * p.head_dim && (!p.q_len || i < p.q_len[b])) {
        const int pos = p.cache_len[b] + i;   // (not through the read-only path: the commit before may still be advancing it when this kernel starts)
        if (pos >= 0 && pos < p.capacity) e.stage = ((long long)b * p.n_kv_heads * p.capacity + pos) * p.head_dim;
        else dlm_set_status(p.status, DLM_ERR_CAPACITY);
      }
      row_s[t] = e;
    }
  }

  // ================================================================= epilogue, by all eight warps
  // fp32 columns pass through shared memory (free by then), in pieces of two segments of kCW columns (rotary pairs, or
  // just two runs), so that a store instruction writes whole sectors of neighbouring features.  One warp per scheduler runs
  // this code, so its length in dependent instructions is what counts: addresses are a per-row offset (table) plus a
  // per-segment pointer, two pieces pass between two barriers, and the rotary factors are in registers before the last
  // product is done (read piece by piece from L2: 36.4 us instead of 34.8 for 1280 rows of Dream).  (Rows kept in their threads, divisions and 64-bit products per store, four warps: 10 us for the
  // 256-feature tile.)
  {
    constexpr int kCW = N / 2 < 32 ? N / 2 : 32;              // columns of a segment
    constexpr int kPieces = N / (2 * kCW), kPR = kPieces > 1 ? 2 : 1;   // pieces of two segments; pieces per round
    constexpr uint32_t kPitch = 2 * kCW * 4 + 16;             // bytes of a staged row; the 16 spread rows over the banks
    constexpr uint32_t kPieceBytes = kRowTile * kPitch;
    constexpr int kLanes = kCW / 8, kRowsPerIt = kThreads / kLanes;
    constexpr int kIts = kRowTile > kRowsPerIt ? kRowTile / kRowsPerIt : 1;
    const int n_rows = min(p.rc, p.rows_total - row0);         // real rows of this block (may be <= 0)
    const int D = p.head_dim, half = D >> 1;
    const bool rope = p.rope_cos != nullptr;
    const int n_qk = p.n_q_heads + p.n_kv_heads;
    // first column of piece i and the distance from there to its second segment
    auto column = [&](int i, int& dist) {
      if (UNITS) {
        const bool second = i >= kN0 / 64;
        dist = second ? kN1 / 2 : kN0 / 2;
        return second ? kN0 + (i - kN0 / 64) * kCW : i * kCW;
      }
      dist = rope && N > D ? half : N / 2;
      if (dist == kCW) return i * 2 * kCW;
      return dist == N / 2 ? i * kCW : (i >> 1) * 2 * dist + (i & 1) * kCW;   // half a head: 32 or 64 columns
    };
    // cos / sin of this thread's rows and columns: every other piece has the same (a head's half is one or two segments), so
    // they are read once, while the products are still running
    float4 cs[kPR][kIts][2], sn[kPR][kIts][2];
    if (rope) {
#pragma unroll
      for (int pr = 0; pr < kPR; ++pr) {
        int dist;
        const int f = feature(column(pr, dist) + (tid % kLanes) * 8);
        if ((f >> p.head_shift) < n_qk) {
#pragma unroll
          for (int it = 0; it < kIts; ++it) {
            const int r = tid / kLanes + it * kRowsPerIt;
            if (r < n_rows) {
              const size_t a = (size_t)(row0 + r) * half + (f & (D - 1));
#pragma unroll
              for (int q = 0; q < 2; ++q) {
                cs[pr][it][q] = reinterpret_cast<const float4*>(p.rope_cos + a)[q];
                sn[pr][it][q] = reinterpret_cast<const float4*>(p.rope_sin + a)[q];
              }
            }
          }
        }
      }
    }
    // The last MMA is waited for whether or not a role of this block has given up: it reads the stages and writes TMEM.  (The
    // tables are there too.)  Who raised the abort flag sees it here.
    const bool clean = *abort_ptr == 0;
    const bool ok = __syncthreads_and(mbar_wait(bar_done, 0, never_ptr) && clean) != 0;
    tc_fence_after_sync();
    // Unwinding: the copies already issued land before the memory is released, also those of a producer that never had to wait
    // (the issuer may have given up behind it).  Both blocks' copies complete on the leader's barriers.  Otherwise the
    // issuer has waited for every one of them.
    if (!ok && rank == 0)
      for (int i = max(0, issued - p.n_stages); i < issued; ++i)
        mbar_wait(bar_full + 8 * (i % p.n_stages), (i / p.n_stages) & 1, never_ptr);
    if (ok && n_rows > 0) {
      // TMEM side: warps w and w + 4 read the lanes of quarter w % 4, one segment each.  The row of a lane: M = 64 puts 16
      // rows in each quarter; M = 128 as a pair puts rows 0-63 twice, lanes 64-127 holding the second half of the columns.
      const int quarter = warp & 3, seg = warp >> 2;
      const int my_row = M == 64 ? quarter * 16 + lane : M == 128 ? (quarter & 1) * 32 + lane : quarter * 32 + lane;
      const bool my_lane = (M != 64 || lane < 16) && my_row < n_rows;
      const uint32_t t_row = tmem + ((uint32_t)(quarter * 32) << 16);
      const uint32_t bias_a = smem_u32(bias_s);
      // store side: where features f .. f + 7 (one head) go
      struct Dest {
        __nv_bfloat16 *out, *stage;
        bool kv;
      };
      auto dest = [&](int f) {
        Dest d;
        d.stage = nullptr;
        d.kv = false;
        if (p.mode == 1) { d.out = p.q_out + f; return d; }
        const int head = p.head_shift >= 0 ? f >> p.head_shift : f / D, df = f - head * D;
        if (head < p.n_q_heads) { d.out = p.q_out + (size_t)head * p.q_cap * D + df; return d; }
        const bool is_k = head < n_qk;
        const size_t h = is_k ? head - p.n_q_heads : head - n_qk;
        d.kv = true;
        d.out = (is_k ? p.k_out : p.v_out) + h * p.q_cap * D + df;
        if (p.stage_k) d.stage = (is_k ? p.stage_k : p.stage_v) + h * p.capacity * D + df;
        return d;
      };
      auto store8 = [&](const Dest& d, const RowEntry& e, const float* y) {
        uint32_t w[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          const __nv_bfloat162 h = __floats2bfloat162_rn(y[2 * j], y[2 * j + 1]);
          w[j] = *reinterpret_cast<const uint32_t*>(&h);
        }
        const uint4 v = make_uint4(w[0], w[1], w[2], w[3]);
        *reinterpret_cast<uint4*>(d.out + (d.kv ? e.kv : e.q)) = v;
        if (d.stage && e.stage >= 0) *reinterpret_cast<uint4*>(d.stage + e.stage) = v;
      };
      uint32_t buf = base;
#pragma unroll 1
      for (int i0 = 0; i0 < kPieces; i0 += kPR) {
#pragma unroll
        for (int pr = 0; pr < kPR; ++pr) {
          if (kPieces % kPR != 0 && i0 + pr >= kPieces) break;
          int dist;
          int col = column(i0 + pr, dist);
          col += seg * dist;
          bool here = true;
          if (M == 128) {
            here = col / (N / 2) == quarter >> 1;            // warp-uniform
            col %= N / 2;
          }
          if (here) {
            uint32_t u[kCW];
            __syncwarp();
            if (kCW == 32) tmem_ld32(t_row + col, u);
            else if (kCW == 16) tmem_ld16(t_row + col, u);
            else tmem_ld8(t_row + col, u);
            tmem_ld_wait();
            if (my_lane) {
              const uint32_t a = buf + pr * kPieceBytes + my_row * kPitch + seg * kCW * 4;
#pragma unroll
              for (int j = 0; j < kCW; j += 4)
                st_shared_f4(a + j * 4, __uint_as_float(u[j]), __uint_as_float(u[j + 1]), __uint_as_float(u[j + 2]), __uint_as_float(u[j + 3]));
            }
          }
        }
        __syncthreads();
#pragma unroll
        for (int pr = 0; pr < kPR; ++pr) {
          if (kPieces % kPR != 0 && i0 + pr >= kPieces) break;
          int dist;
          const int cc = column(i0 + pr, dist) + (tid % kLanes) * 8;   // this thread's 8 columns, and the 8 at cc + dist
          const int f0 = feature(cc), f1 = feature(cc + dist);
          if (UNITS && f0 >= p.n_out) break;                 // the last tile's units beyond the last feature (uniform: one unit)
          const bool turn = rope && (f0 >> p.head_shift) < n_qk;
          const Dest d0 = dest(f0), d1 = dest(f1);
          float b0[8], b1[8];
#pragma unroll
          for (int j = 0; j < 8; j += 4) {
            const float4 x = ld_shared_f4(bias_a + (cc + j) * 4), y = ld_shared_f4(bias_a + (cc + dist + j) * 4);
            b0[j] = x.x; b0[j + 1] = x.y; b0[j + 2] = x.z; b0[j + 3] = x.w;
            b1[j] = y.x; b1[j + 1] = y.y; b1[j + 2] = y.z; b1[j + 3] = y.w;
          }
#pragma unroll
          for (int it = 0; it < kIts; ++it) {
            const int r = tid / kLanes + it * kRowsPerIt;
            if (r < n_rows) {
              const RowEntry e = row_s[r];
              const uint32_t a = buf + pr * kPieceBytes + r * kPitch + (tid % kLanes) * 32;
              float y0[8], y1[8];
#pragma unroll
              for (int j = 0; j < 2; ++j) {
                const float4 lo = ld_shared_f4(a + 16 * j), hi = ld_shared_f4(a + kCW * 4 + 16 * j);
                y0[4 * j] = lo.x; y0[4 * j + 1] = lo.y; y0[4 * j + 2] = lo.z; y0[4 * j + 3] = lo.w;
                y1[4 * j] = hi.x; y1[4 * j + 1] = hi.y; y1[4 * j + 2] = hi.z; y1[4 * j + 3] = hi.w;
              }
#pragma unroll
              for (int j = 0; j < 8; ++j) { y0[j] += b0[j]; y1[j] += b1[j]; }
              if (turn) {
                const float4 (&c4)[2] = cs[pr][it], (&s4)[2] = sn[pr][it];
                const float co[8] = {c4[0].x, c4[0].y, c4[0].z, c4[0].w, c4[1].x, c4[1].y, c4[1].z, c4[1].w};
                const float si[8] = {s4[0].x, s4[0].y, s4[0].z, s4[0].w, s4[1].x, s4[1].y, s4[1].z, s4[1].w};
#pragma unroll
                for (int j = 0; j < 8; ++j) {
                  const float lo = y0[j], hi = y1[j];
                  y0[j] = fmaf(-hi, si[j], lo * co[j]);
                  y1[j] = fmaf(lo, si[j], hi * co[j]);
                }
              }
              store8(d0, e, y0);
              store8(d1, e, y1);
            }
          }
        }
        buf = buf == base ? base + kPR * kPieceBytes : base;   // the next round's writes meet no reader of this one
      }
    }
  }
  // ---- teardown
  __syncwarp();
  if (tid == 0 && (*abort_ptr || *never_ptr)) dlm_set_status(p.status, DLM_ERR_TIMEOUT);
  tc_fence_before_sync();
  // a pair leaves together: the leader's MMAs read the other block's shared memory, both blocks' copies complete on the leader's barriers
  if (PAIR) cluster_sync(); else __syncthreads();
  if (warp == 3) {
    tc_fence_after_sync();
    if (PAIR) tmem_dealloc_pair(tmem, kTmemCols); else tmem_dealloc(tmem, kTmemCols);
  }
}

using ProjKernel = void (*)(const CUtensorMap, const CUtensorMap, const ProjParams);
struct ProjVariant {
  int n, m, kp;
  ProjKernel fn;
};
// N features, M rows, K panels per stage (stages of 16 - 40 KB)
const ProjVariant kVariants[] = {
    {16, 64, 4, window_proj_kernel<16, 64, 4>},     {32, 64, 4, window_proj_kernel<32, 64, 4>},
    {64, 64, 2, window_proj_kernel<64, 64, 2>},     {128, 64, 2, window_proj_kernel<128, 64, 2>},
    {64, 128, 2, window_proj_kernel<64, 128, 2>},   {128, 128, 2, window_proj_kernel<128, 128, 2>},
    {256, 128, 1, window_proj_kernel<256, 128, 1>}, {64, 256, 2, window_proj_kernel<64, 256, 2>},
    {128, 256, 1, window_proj_kernel<128, 256, 1>}, {192, 256, 1, window_proj_kernel<192, 256, 1>},
    {256, 256, 1, window_proj_kernel<256, 256, 1>}, {320, 256, 1, window_proj_kernel<320, 256, 1>},
    {384, 256, 1, window_proj_kernel<384, 256, 1>}, {448, 256, 1, window_proj_kernel<448, 256, 1>},
    {512, 256, 1, window_proj_kernel<512, 256, 1>},
};

struct ProjPlan {
  int variant, rc, x_box_rows, w_box_rows, chunks, tiles, half_rows, n_stages, aux_offset, smem_bytes;
};

// rows: activation rows of the call; heads_q_cap > 0: head-split activations (all rows in one chunk) with that many rows
// per sequence, `batch` sequences.
bool make_proj_plan(const dlm_ctx* ctx, int rows, int n_out, int k_total, int head_dim, int batch, int heads_q_cap, ProjPlan& pl) {
  // (head-split activations whose half of the sequences is more than the 64 rows of a pair's block take the wide pairs: one
  // copy per panel instead of pieces of a sequence)
  const bool wide = heads_q_cap > 0 && batch > 1 && (batch + 1) / 2 * heads_q_cap > 64;
  const int m = rows <= 64 ? 64 : rows <= 128 && !wide ? 128 : 256;
  const bool pair = m > 64;
  if (heads_q_cap > 0 && rows > kMaxActRows) return false;
  pl.chunks = pair ? (rows + 255) / 256 : 1;
  const int blocks_rows = pl.chunks * (pair ? 2 : 1);
  pl.rc = ((rows + blocks_rows - 1) / blocks_rows + 7) & ~7;
  pl.x_box_rows = pl.rc;
  if (heads_q_cap > 0 && batch > 1) {
    // one copy brings the rows of whole sequences; where the pair's split falls inside one, copies of the largest divisor of a
    // sequence (in eights) that leaves no block more than its rows.  With the common divisor of sequence and block, 14 copies of 8 rows a
    // panel at 3 x 72 rows, an output projection of Dream took 65.5 us; with the 5 of 24, dealt over lanes, 13.9.
    const int nb = (batch + blocks_rows - 1) / blocks_rows;
    if (nb * heads_q_cap <= (m == 128 ? 64 : 128)) {
      pl.rc = pl.x_box_rows = nb * heads_q_cap;
    } else {
      const int half = (rows + 1) / 2, limit = m == 128 ? 64 : 128;
      for (int d = heads_q_cap; d >= 8; d -= 8) {   // d = 8 always fits
        pl.x_box_rows = d;
        pl.rc = (half + d - 1) / d * d;
        if (heads_q_cap % d == 0 && pl.rc <= limit) break;
      }
    }
  }
  // The tile width: the one with the least estimate for the SM with the most blocks.  Per 16 elements of K a block's MMA takes
  // N / 2 cycles, or what its operands take at 128 bytes per cycle of shared memory, or what they take to arrive at 70 bytes
  // per cycle and SM; a block costs some fixed time on top.  It ranks widths and is not a time: HBM, latencies, the producers'
  // loop and the power cap are not in it, and calls take 1.3 to 3 times as long (32 x 3584 -> 4608: 4.0 us against 8.5
  // measured, 256 x 3584 -> 4608 9.2 against 12.4, 1280 x 3584 -> 4608 24.7 against 36.1, 256 x 4096 -> 12288 15.0 against 28.6,
  // and 28.5 with the weights in L2: it is not HBM that is missing there).  Of 98 calls with every width timed (seven
  // widths of five models, 1 - 3000 rows) it picks the fastest or one within 2 % in 92; the others are 2000 rows of 4096 -> 12288
  // (192: 203 us, 512: 174, under the power cap), 3000 of 256 -> 512 and 8 of 3584 -> 3584 (7 %), and three small ones (2 - 4 %).
  double best = 0;
  pl.variant = -1;
  for (int v = 0; v < (int)(sizeof(kVariants) / sizeof(kVariants[0])); ++v) {
    const ProjVariant& k = kVariants[v];
    if (k.m != m || (n_out % k.n != 0 && !tile_of_units(k.n))) continue;
    const long long blocks = (long long)((n_out + k.n - 1) / k.n) * blocks_rows;
    const double per_sm = (double)((blocks + ctx->num_sms - 1) / ctx->num_sms);
    const double mma = m == 256 ? k.n / 2.0 : k.n / 4.0, smem = ((m == 256 ? 4096.0 : 2048.0) * (k.n > 256 ? 2 : 1) + k.n * (pair ? 16.0 : 32.0)) / 128.0;
    const double intake = (pl.rc + k.n / (pair ? 2 : 1)) * 32.0 / 70.0;
    double cyc = mma > smem ? mma : smem;
    if (intake > cyc) cyc = intake;
    const double t = per_sm * (k_total / 16.0 * cyc + 1000.0 + 12.0 * k.n);
    if (pl.variant < 0 || t < best) { best = t; pl.variant = v; }
  }
  if (pl.variant < 0) return false;
  const ProjVariant& k = kVariants[pl.variant];
  pl.tiles = (n_out + k.n - 1) / k.n;
  // rotary pairs inside a tile: see the kernel
  if (tile_of_units(k.n)) {
    pl.half_rows = head_dim == 64 ? 32 : 64;
    pl.w_box_rows = pl.half_rows == 64 && k.n % 128 == 0 ? 64 : 32;
  } else {
    pl.half_rows = (head_dim == 64 || head_dim == 128) && k.n < head_dim ? head_dim / 2 : k.n / 2;
    pl.w_box_rows = k.n / 2;
  }
  const int stage = k.kp * 128 * (pl.rc + k.n / (pair ? 2 : 1));
  const int n_k = (k_total / kPanel + k.kp - 1) / k.kp;
  // Behind the stages: the MMA reads rows up to M of an activation panel, which no copy filled (their results are never
  // looked at); for the last panel of the last stage that may reach beyond the weights that follow it.
  const int row_tile = m == 64 ? 64 : m / 2, cw = k.n / 2 < 32 ? k.n / 2 : 32;
  const int beyond = (row_tile - pl.rc - k.kp * (k.n / (pair ? 2 : 1))) * 128, slack = beyond > 0 ? beyond : 0;
  const int fixed = 1024 + slack + kAuxBytes;
  // One block per SM, with depth (5 stages instead of 3: 20.2 -> 16.4 us at 256 Dream rows).  Two small ones per SM would let
  // the next kernel's blocks start beside this one's and prefetch their weights, but they also crowd onto the SMs that an
  // attention kernel before them leaves free: a 28-layer Dream step took 1137 us instead of 995.
  int stages = (220 * 1024 - fixed) / stage;
  if (stages < 3) stages = 3;
  if (stages > kMaxStages) stages = kMaxStages;
  if (stages > n_k) stages = n_k;
  pl.n_stages = stages;
  // the epilogue's two staging buffers, of one or two pieces each, lie over the stages
  const int staging = (k.n > 2 * cw ? 4 : 2) * row_tile * (2 * cw * 4 + 16);
  pl.aux_offset = stages * stage + slack;
  if (pl.aux_offset < staging) pl.aux_offset = (staging + 127) & ~127;
  pl.smem_bytes = 1024 + pl.aux_offset + kAuxBytes;
  return pl.smem_bytes <= ctx->max_smem_optin && pl.chunks <= 65535;
}

int launch_proj(dlm_ctx* ctx, const ProjPlan& pl, ProjParams& p, const CUtensorMap& tm_w, const CUtensorMap& tm_x, cudaStream_t s) {
  const ProjVariant& k = kVariants[pl.variant];
  const int cluster = k.m > 64 ? 2 : 1;
  if (!(ctx->proj_configured & (1u << pl.variant))) {
    DLM_CUDA_TRY(cudaFuncSetAttribute(k.fn, cudaFuncAttributeMaxDynamicSharedMemorySize, ctx->max_smem_optin));
    ctx->proj_configured |= 1u << pl.variant;
  }
  p.rc = pl.rc;
  p.x_box_rows = pl.x_box_rows;
  p.pieces = p.act_heads ? pl.rc / pl.x_box_rows : 1;
  p.half_rows = pl.half_rows;
  p.w_box_rows = pl.w_box_rows;
  p.n_stages = pl.n_stages;
  p.aux_offset = pl.aux_offset;
  p.head_shift = p.head_dim == 128 ? 7 : p.head_dim == 64 ? 6 : -1;
  p.status = &ctx->words->status;
  DLM_CUDA_TRY(dlm_launch_cluster(k.fn, dim3(pl.tiles * cluster, 1, pl.chunks), dim3(kThreads), (size_t)pl.smem_bytes, s,
                                  cluster, tm_w, tm_x, p));
  return dlm_launch_ok(ctx, 1);
}

// W seen as [groups][2][half_rows][K / 64][64]; a copy brings w_box_rows features of one half (pairs) or of both, kp panels.
bool encode_weights(dlm_ctx* ctx, CUtensorMap* map, const void* w, int n_out, int k_total, const ProjPlan& pl) {
  const ProjVariant& k = kVariants[pl.variant];
  const cuuint64_t row = (cuuint64_t)k_total * 2, a = (cuuint64_t)pl.half_rows;
  const cuuint64_t dims[5] = {(cuuint64_t)kPanel, a, 2, (cuuint64_t)(k_total / kPanel), (cuuint64_t)n_out / (2 * a)};
  const cuuint64_t strides[4] = {row, a * row, (cuuint64_t)kPanel * 2, 2 * a * row};
  const cuuint32_t box[5] = {(cuuint32_t)kPanel, (cuuint32_t)pl.w_box_rows, k.m > 64 ? 1u : 2u, (cuuint32_t)k.kp, 1};
  return dlm_tensor_map(ctx, map, w, 5, dims, strides, box);
}

}  // namespace

// The kernels sum all of K in one block (pair) and need no scratch; what is left is a non-zero answer for valid sizes.
extern "C" size_t dlm_window_proj_workspace_bytes(const dlm_ctx* ctx, int rows, int n_out, int k_total) {
  if (!ctx || rows <= 0 || n_out <= 0 || k_total <= 0 || n_out % 128 != 0 || k_total % kPanel != 0) return 0;
  return 256;
}

namespace {
int qkv_project(dlm_ctx* ctx, const void* x, const void* w, const void* bias, const float* rope_cos, const float* rope_sin,
                int batch, int q_cap, int d_model, int n_q_heads, int n_kv_heads, int head_dim, void* q_out, void* k_out,
                void* v_out, const dlm_kv_cache* cache, int layer, const int32_t* q_len, void* workspace, size_t workspace_bytes,
                void* stream);
}

extern "C" int dlm_window_qkv_project(dlm_ctx* ctx, const void* x, const void* w, const void* bias, int batch, int q_cap,
                                      int d_model, int n_q_heads, int n_kv_heads, int head_dim, void* q_out, void* k_out,
                                      void* v_out, void* workspace, size_t workspace_bytes, void* stream) {
  return qkv_project(ctx, x, w, bias, nullptr, nullptr, batch, q_cap, d_model, n_q_heads, n_kv_heads, head_dim, q_out, k_out,
                     v_out, nullptr, 0, nullptr, workspace, workspace_bytes, stream);
}

extern "C" int dlm_window_qkv_project_rope(dlm_ctx* ctx, const void* x, const void* w, const void* bias, const float* rope_cos,
                                           const float* rope_sin, int batch, int q_cap, int d_model, int n_q_heads,
                                           int n_kv_heads, int head_dim, void* q_out, void* k_out, void* v_out, void* workspace,
                                           size_t workspace_bytes, void* stream) {
  if (!rope_cos || !rope_sin) return DLM_ERR_NULL;
  // a tile's halves are a head's halves, or units of 32 features of either (make_proj_plan knows 64 and 128), and the factors
  // are read as 16-byte vectors
  if (head_dim != 64 && head_dim != 128) return DLM_ERR_UNSUPPORTED;
  if (((uintptr_t)rope_cos | (uintptr_t)rope_sin) & 15) return DLM_ERR_UNSUPPORTED;
  return qkv_project(ctx, x, w, bias, rope_cos, rope_sin, batch, q_cap, d_model, n_q_heads, n_kv_heads, head_dim, q_out, k_out,
                     v_out, nullptr, 0, nullptr, workspace, workspace_bytes, stream);
}

extern "C" int dlm_window_qkv_project_stage(dlm_ctx* ctx, const void* x, const void* w, const void* bias, const float* rope_cos,
                                            const float* rope_sin, int batch, int q_cap, int d_model, int n_q_heads,
                                            int n_kv_heads, int head_dim, const int32_t* q_len, void* q_out, void* k_out,
                                            void* v_out, const dlm_kv_cache* cache, int layer, void* workspace,
                                            size_t workspace_bytes, void* stream) {
  if (!cache || !cache->k || !cache->v || !cache->cache_len) return DLM_ERR_NULL;
  if ((rope_cos == nullptr) != (rope_sin == nullptr)) return DLM_ERR_NULL;
  if (rope_cos && head_dim != 64 && head_dim != 128) return DLM_ERR_UNSUPPORTED;
  if (((uintptr_t)rope_cos | (uintptr_t)rope_sin | (uintptr_t)cache->k | (uintptr_t)cache->v) & 15) return DLM_ERR_UNSUPPORTED;
  if (layer < 0 || layer >= cache->n_layers || cache->batch != batch || cache->n_kv_heads != n_kv_heads ||
      cache->head_dim != head_dim || cache->capacity <= 0)
    return DLM_ERR_SHAPE;
  return qkv_project(ctx, x, w, bias, rope_cos, rope_sin, batch, q_cap, d_model, n_q_heads, n_kv_heads, head_dim, q_out, k_out,
                     v_out, cache, layer, q_len, workspace, workspace_bytes, stream);
}

namespace {
int qkv_project(dlm_ctx* ctx, const void* x, const void* w, const void* bias, const float* rope_cos, const float* rope_sin,
                int batch, int q_cap, int d_model, int n_q_heads, int n_kv_heads, int head_dim, void* q_out, void* k_out,
                void* v_out, const dlm_kv_cache* cache, int layer, const int32_t* q_len, void* workspace, size_t workspace_bytes,
                void* stream) {
  if (!ctx || !x || !w || !q_out || !k_out || !v_out) return DLM_ERR_NULL;
  if (batch <= 0 || q_cap <= 0 || d_model <= 0 || n_q_heads <= 0 || n_kv_heads <= 0 || head_dim <= 0) return DLM_ERR_SHAPE;
  const long long n_out = (long long)(n_q_heads + 2 * n_kv_heads) * head_dim;
  const long long rows = (long long)batch * q_cap;
  if (n_out % 128 != 0 || d_model % kPanel != 0 || head_dim % 8 != 0 || rows > (1 << 20) || n_out > (1 << 24))
    return DLM_ERR_UNSUPPORTED;
  if (((uintptr_t)x | (uintptr_t)w | (uintptr_t)q_out | (uintptr_t)k_out | (uintptr_t)v_out) & 15) return DLM_ERR_UNSUPPORTED;
  DLM_DEVICE_TRY(ctx);
  ProjPlan pl;
  if (!make_proj_plan(ctx, (int)rows, (int)n_out, d_model, head_dim, batch, 0, pl)) return DLM_ERR_UNSUPPORTED;
  CUtensorMap tm_w, tm_x;
  if (!encode_weights(ctx, &tm_w, w, (int)n_out, d_model, pl)) return DLM_ERR_CUDA;
  {
    const cuuint64_t dims[4] = {(cuuint64_t)kPanel, (cuuint64_t)rows, (cuuint64_t)(d_model / kPanel), 1};
    const cuuint64_t strides[3] = {(cuuint64_t)d_model * 2, (cuuint64_t)kPanel * 2, (cuuint64_t)d_model * 2};
    const cuuint32_t box[4] = {(cuuint32_t)kPanel, (cuuint32_t)pl.rc, (cuuint32_t)kVariants[pl.variant].kp, 1};
    if (!dlm_tensor_map(ctx, &tm_x, x, 4, dims, strides, box)) return DLM_ERR_CUDA;
  }
  ProjParams p = {};
  p.mode = 0;
  p.q_out = static_cast<__nv_bfloat16*>(q_out);
  p.k_out = static_cast<__nv_bfloat16*>(k_out);
  p.v_out = static_cast<__nv_bfloat16*>(v_out);
  p.bias = static_cast<const __nv_bfloat16*>(bias);
  p.rope_cos = rope_cos;
  p.rope_sin = rope_sin;
  if (cache) {
    const size_t layer_elems = (size_t)batch * n_kv_heads * cache->capacity * head_dim;
    p.stage_k = static_cast<__nv_bfloat16*>(cache->k) + (size_t)layer * layer_elems;
    p.stage_v = static_cast<__nv_bfloat16*>(cache->v) + (size_t)layer * layer_elems;
    p.cache_len = cache->cache_len;
    p.q_len = q_len;
    p.capacity = cache->capacity;
  }
  p.rows_total = (int)rows; p.q_cap = q_cap; p.n_q_heads = n_q_heads; p.n_kv_heads = n_kv_heads; p.head_dim = head_dim;
  p.n_out = (int)n_out; p.k_total = d_model; p.batch = batch; p.act_heads = 0;
  return launch_proj(ctx, pl, p, tm_w, tm_x, static_cast<cudaStream_t>(stream));
}
}  // namespace

extern "C" int dlm_window_out_project(dlm_ctx* ctx, const void* o, const void* wo, const void* bias, int batch, int q_cap,
                                      int d_model, int n_q_heads, int head_dim, void* y, void* workspace,
                                      size_t workspace_bytes, void* stream) {
  if (!ctx || !o || !wo || !y) return DLM_ERR_NULL;
  if (batch <= 0 || q_cap <= 0 || d_model <= 0 || n_q_heads <= 0 || head_dim <= 0) return DLM_ERR_SHAPE;
  const long long k_total = (long long)n_q_heads * head_dim, rows = (long long)batch * q_cap;
  // a stage holds 64 features of one head for every row of the call: whole heads of 64-element panels, all rows in
  // one block (<= 256), and each batch element's rows starting on a swizzle-atom boundary (8 rows)
  if (d_model % 128 != 0 || head_dim % kPanel != 0 || rows > kMaxActRows || (batch > 1 && q_cap % 8 != 0))
    return DLM_ERR_UNSUPPORTED;
  if (((uintptr_t)o | (uintptr_t)wo | (uintptr_t)y) & 15) return DLM_ERR_UNSUPPORTED;
  DLM_DEVICE_TRY(ctx);
  ProjPlan pl;
  if (!make_proj_plan(ctx, (int)rows, d_model, (int)k_total, 0, batch, q_cap, pl)) return DLM_ERR_UNSUPPORTED;
  CUtensorMap tm_w, tm_x;
  if (!encode_weights(ctx, &tm_w, wo, d_model, (int)k_total, pl)) return DLM_ERR_CUDA;
  {
    // a box brings one 64-element panel of one head: the rows of whole sequences, or part of one sequence's rows
    const int box_seqs = batch > 1 && pl.x_box_rows % q_cap == 0 ? pl.x_box_rows / q_cap : 1;
    const cuuint64_t dims[4] = {(cuuint64_t)head_dim, (cuuint64_t)q_cap, (cuuint64_t)n_q_heads, (cuuint64_t)batch};
    const cuuint64_t strides[3] = {(cuuint64_t)head_dim * 2, (cuuint64_t)q_cap * head_dim * 2, (cuuint64_t)k_total * q_cap * 2};
    const cuuint32_t box[4] = {(cuuint32_t)kPanel, (cuuint32_t)(pl.x_box_rows / box_seqs), 1, (cuuint32_t)box_seqs};
    if (!dlm_tensor_map(ctx, &tm_x, o, 4, dims, strides, box)) return DLM_ERR_CUDA;
  }
  ProjParams p = {};
  p.mode = 1;
  p.q_out = static_cast<__nv_bfloat16*>(y);
  p.bias = static_cast<const __nv_bfloat16*>(bias);
  p.rows_total = (int)rows; p.q_cap = q_cap; p.n_q_heads = n_q_heads; p.n_kv_heads = 0; p.head_dim = head_dim;
  p.n_out = d_model; p.k_total = (int)k_total; p.batch = batch; p.act_heads = n_q_heads;
  return launch_proj(ctx, pl, p, tm_w, tm_x, static_cast<cudaStream_t>(stream));
}
