// Shared host/device declarations of the DLM FreeCache library (internal; the public
// interface is include/dlm.h).
#pragma once

#include <cuda.h>
#include <cuda_runtime.h>
#include <stdint.h>
#include <string.h>

#include "dlm.h"

// Device words owned by a context.  `status` holds the first data-dependent error code
// (0 = none); the ticket words let the last block of a kernel run a serial tail.
constexpr int kDlmUnmaskTickets = 1024;  // batch elements whose selection can run in the tail of the reduce kernel
constexpr int kDlmMaxSplitUnits = 2048;  // attention units that may be split across blocks in one call
struct dlm_device_words {
  int status;
  unsigned int commit_ticket;
  unsigned int pad[14];
  unsigned int unmask_tickets[kDlmUnmaskTickets];     // blocks of a batch element finished so far
  unsigned int attn_unit_tickets[kDlmMaxSplitUnits];  // pieces of a split unit finished so far
};

// TMA descriptors a context has built, by the sizes they describe and not by the tensor: a call copies the one of its sizes
// and writes its own address into the copy (9 ns; building one takes 57 ns, and an attention call has five), on new
// tensors as on old ones.  Direct-mapped and fixed in size.
struct dlm_map_key {
  cuuint64_t dims[5], strides[4];
  cuuint32_t box[5], rank;
};
constexpr int kDlmMapSlots = 128;
struct dlm_map_cache {
  dlm_map_key key[kDlmMapSlots];   // rank 0: empty
  CUtensorMap map[kDlmMapSlots];
};

// How an attention call's work is dealt out (attn_step.cu), and what that depends on.
struct dlm_attn_plan {
  int n_mt, rows, rows_total, n_rc, grid, whole_units, chunk_rows, team;
  int single;      // whole units or teams, and no block has more than one unit (or piece of one)
  int wide;        // teams that are no cluster: they exchange through L2
  int smem_bytes;
  size_t ws_o_bytes, ws_ml_bytes;
};
struct dlm_attn_plan_key {
  int nl, batch, n_kv_heads, capacity, head_dim, n_q_heads, q_cap, hint, team_max, team_force, no_wait;
};

struct dlm_ctx {
  int device;
  int num_sms;
  int max_smem_optin;       // largest dynamic shared memory a block may opt in to, bytes
  int64_t launches;
  dlm_device_words* words;  // device
  void* encode_tiled;       // cuTensorMapEncodeTiled and cuTensorMapReplaceAddress (driver API), resolved lazily
  void* replace_address;
  dlm_map_cache* maps;
  int commit_blocks_per_sm[2];  // resident blocks per SM of the two commit kernels (0 = not asked yet)
  unsigned long long wait_limit_ns;   // limit of the kernels' device-side waits (2 s; a test may shorten it)
  unsigned int proj_configured; // bit per projection kernel: shared-memory opt-in done on this context's device
  int attn_team_max;            // most blocks the attention call's team schedule may give one unit (1 = schedule off)
  bool attn_team_force;         // tests: take the team schedule wherever it is possible, whatever the cost estimate says
  dlm_attn_plan_key attn_plan_key;   // of the last call's plan (nl = 0: none yet)
  dlm_attn_plan attn_plan;
  int attn_clusters[17];        // clusters of so many attention blocks that the device runs at a time (0 = not asked yet, -1 = none)
  int attn_smem_limit[32];      // dynamic shared memory the attention kernels may use on this device (0 = not set up yet)
};

// Writes the descriptor of a bf16 tensor of `rank` dimensions (sizes, byte strides of dimensions 1 .., box), 128-byte swizzle,
// to `out`; false if the driver refuses it.  Defined in api.cu.
bool dlm_tensor_map(dlm_ctx* ctx, CUtensorMap* out, const void* base, int rank, const cuuint64_t* dims, const cuuint64_t* strides,
                    const cuuint32_t* box);

// Division by a divisor known on the host: one high multiply, an add and a shift (round-up reciprocal of Granlund and
// Montgomery, for dividends below 2^31).
struct FastDiv {
  uint32_t mul, shift;
  int d;
  __device__ __forceinline__ int div(int n) const { return (int)((__umulhi((uint32_t)n, mul) + (uint32_t)n) >> shift); }
  // quotient; `rem` gets the remainder
  __device__ __forceinline__ int divmod(int n, int& rem) const {
    const int q = div(n);
    rem = n - q * d;
    return q;
  }
};
static inline FastDiv make_fast_div(int d) {
  FastDiv f;
  f.d = d;
  f.shift = 0;
  while ((1ll << f.shift) < d) ++f.shift;
  f.mul = (uint32_t)((((1ull << 32) * ((1ull << f.shift) - (uint64_t)d)) / (uint64_t)d) + 1);
  return f;
}

#define DLM_CUDA_TRY(expr)                         \
  do {                                             \
    cudaError_t _e = (expr);                       \
    if (_e != cudaSuccess) return DLM_ERR_CUDA;    \
  } while (0)

// Records the first error seen by any thread of any kernel.
__device__ __forceinline__ void dlm_set_status(int* status, int code) { atomicCAS(status, 0, code); }

// Programmatic dependent launch.  Every kernel of the library is launched with the
// programmatic-stream-serialization attribute, calls dlm_grid_dependency_wait() before it touches
// anything a predecessor in the stream may have written, and lets its own dependents start
// launching early with dlm_trigger_dependents(): block scheduling and the dependents' data-free
// set-up then overlap the predecessor's tail instead of following it.  A dependent's wait still
// returns only when the predecessor grid has completed and its writes are visible, and the
// hardware starts dependents only once every block of the predecessor is running, so nothing is
// reordered.  Predecessors that know nothing of this (any other kernel) simply release their
// dependents when they finish.
__device__ __forceinline__ void dlm_grid_dependency_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void dlm_trigger_dependents() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

template <typename... KArgs, typename... Args>
static inline cudaError_t dlm_launch_cluster(void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t stream,
                                             unsigned int cluster, Args... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = stream;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  if (cluster > 1) {   // thread-block clusters of `cluster` consecutive blocks along x
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = cluster;
    attr[1].val.clusterDim.y = attr[1].val.clusterDim.z = 1;
    cfg.numAttrs = 2;
  }
  return cudaLaunchKernelEx(&cfg, kernel, static_cast<KArgs>(args)...);
}

template <typename... KArgs, typename... Args>
static inline cudaError_t dlm_launch(void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t stream,
                                     Args... args) {
  return dlm_launch_cluster(kernel, grid, block, smem, stream, 1, args...);
}

// The context's device must be the calling thread's current device: launches go to the current
// device, the context's words and the caller's pointers live on the context's.
static inline int dlm_check_device(const dlm_ctx* ctx) {
  int dev = -1;
  if (cudaGetDevice(&dev) != cudaSuccess) return DLM_ERR_CUDA;
  return dev == ctx->device ? DLM_OK : DLM_ERR_DEVICE;
}
#define DLM_DEVICE_TRY(ctx)                        \
  do {                                             \
    const int _d = dlm_check_device(ctx);          \
    if (_d != DLM_OK) return _d;                   \
  } while (0)

static inline int dlm_launch_ok(dlm_ctx* ctx, int n_kernels) {
  if (cudaGetLastError() != cudaSuccess) return DLM_ERR_CUDA;
  ctx->launches += n_kernels;
  return DLM_OK;
}
