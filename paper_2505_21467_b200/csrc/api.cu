// Context management of the DLM FreeCache library: creation, status word, error text.
#include <new>

#include "common.cuh"
#include "sm100_ptx.cuh"

extern "C" int dlm_create(dlm_ctx** out, int device) {
  if (!out) return DLM_ERR_NULL;
  *out = nullptr;
  int count = 0;
  if (cudaGetDeviceCount(&count) != cudaSuccess || device < 0 || device >= count) return DLM_ERR_CUDA;
  cudaDeviceProp prop;
  DLM_CUDA_TRY(cudaGetDeviceProperties(&prop, device));
  if (prop.major != 10) return DLM_ERR_UNSUPPORTED;  // the kernels are sm_100a only
  int prev = 0;
  DLM_CUDA_TRY(cudaGetDevice(&prev));
  DLM_CUDA_TRY(cudaSetDevice(device));
  dlm_ctx* ctx = new (std::nothrow) dlm_ctx();
  if (!ctx) return DLM_ERR_CUDA;
  ctx->device = device;
  ctx->num_sms = prop.multiProcessorCount;
  ctx->max_smem_optin = (int)prop.sharedMemPerBlockOptin;
  ctx->launches = 0;
  ctx->encode_tiled = ctx->replace_address = nullptr;
  ctx->maps = new (std::nothrow) dlm_map_cache();
  ctx->commit_blocks_per_sm[0] = ctx->commit_blocks_per_sm[1] = 0;
  for (int& limit : ctx->attn_smem_limit) limit = 0;
  for (int& n : ctx->attn_clusters) n = 0;
  ctx->proj_configured = 0;
  memset(&ctx->attn_plan_key, 0, sizeof ctx->attn_plan_key);
  ctx->wait_limit_ns = sm100::kWaitLimitNs;
  ctx->attn_team_max = 1 << 20;   // no limit beyond the schedule's own
  ctx->attn_team_force = false;
  if (!ctx->maps || cudaMalloc(&ctx->words, sizeof(dlm_device_words)) != cudaSuccess ||
      cudaMemset(ctx->words, 0, sizeof(dlm_device_words)) != cudaSuccess) {
    delete ctx->maps;
    delete ctx;
    cudaSetDevice(prev);
    return DLM_ERR_CUDA;
  }
  cudaSetDevice(prev);
  *out = ctx;
  return DLM_OK;
}

extern "C" int dlm_destroy(dlm_ctx* ctx) {
  if (!ctx) return DLM_ERR_NULL;
  cudaFree(ctx->words);
  delete ctx->maps;
  delete ctx;
  return DLM_OK;
}

extern "C" int dlm_get_status(dlm_ctx* ctx, void* stream) {
  if (!ctx) return DLM_ERR_NULL;
  DLM_DEVICE_TRY(ctx);
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  int code = 0;
  DLM_CUDA_TRY(cudaMemcpyAsync(&code, &ctx->words->status, sizeof(int), cudaMemcpyDeviceToHost, s));
  DLM_CUDA_TRY(cudaMemsetAsync(&ctx->words->status, 0, sizeof(int), s));
  DLM_CUDA_TRY(cudaStreamSynchronize(s));
  if (code != 0) {
    // a kernel that gave up may have left its ticket words half counted
    DLM_CUDA_TRY(cudaMemsetAsync(ctx->words, 0, sizeof(dlm_device_words), s));
    DLM_CUDA_TRY(cudaStreamSynchronize(s));
  }
  return code;
}

typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

typedef CUresult (*ReplaceAddressFn)(CUtensorMap*, void*);

static void* driver_entry(const char* name) {
  void* fn = nullptr;
  cudaDriverEntryPointQueryResult q;
  return cudaGetDriverEntryPoint(name, &fn, cudaEnableDefault, &q) == cudaSuccess && q == cudaDriverEntryPointSuccess ? fn : nullptr;
}

bool dlm_tensor_map(dlm_ctx* ctx, CUtensorMap* out, const void* base, int rank, const cuuint64_t* dims, const cuuint64_t* strides,
                    const cuuint32_t* box) {
  if (!ctx->encode_tiled) ctx->encode_tiled = driver_entry("cuTensorMapEncodeTiled");
  if (!ctx->replace_address) ctx->replace_address = driver_entry("cuTensorMapReplaceAddress");
  if (!ctx->encode_tiled || !ctx->replace_address) return false;
  dlm_map_key k;
  memset(&k, 0, sizeof k);
  k.rank = (cuuint32_t)rank;
  uint64_t h = (uint64_t)rank;
  for (int i = 0; i < rank; ++i) {
    k.dims[i] = dims[i];
    k.box[i] = box[i];
    if (i + 1 < rank) k.strides[i] = strides[i];
    h = (h ^ dims[i] ^ ((uint64_t)box[i] << 32)) * 0x9e3779b97f4a7c15ull;
  }
  const int slot = (int)(h >> 57);   // 7 bits
  static_assert(kDlmMapSlots == 128, "slots are picked by 7 bits");
  dlm_map_cache& c = *ctx->maps;
  if (memcmp(&c.key[slot], &k, sizeof k) != 0) {
    const cuuint32_t elem[5] = {1, 1, 1, 1, 1};
    c.key[slot].rank = 0;
    if (reinterpret_cast<EncodeTiledFn>(ctx->encode_tiled)(
            &c.map[slot], CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, (cuuint32_t)rank, const_cast<void*>(base), dims, strides, box, elem,
            CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
      return false;
    c.key[slot] = k;
  }
  *out = c.map[slot];
  return reinterpret_cast<ReplaceAddressFn>(ctx->replace_address)(out, const_cast<void*>(base)) == CUDA_SUCCESS;
}

extern "C" int64_t dlm_launch_count(const dlm_ctx* ctx) { return ctx ? ctx->launches : 0; }

extern "C" const char* dlm_strerror(int code) {
  switch (code) {
    case DLM_OK: return "ok";
    case DLM_ERR_NULL: return "a required pointer is NULL";
    case DLM_ERR_SHAPE: return "a size is non-positive or inconsistent";
    case DLM_ERR_UNSUPPORTED: return "configuration not supported";
    case DLM_ERR_CAPACITY: return "cache length or row count exceeds capacity";
    case DLM_ERR_WORKSPACE: return "workspace missing, misaligned or too small";
    case DLM_ERR_CUDA: return "a CUDA call failed";
    case DLM_ERR_TIMEOUT: return "a bounded device-side wait expired";
    case DLM_ERR_INDEX: return "a row index is out of range";
    case DLM_ERR_DEVICE: return "the current CUDA device is not the context's device";
    default: return "unknown error code";
  }
}

namespace {

// Waits on an mbarrier that nobody will ever arrive at, with the same bounded wait the kernels use.
__global__ void wait_probe_kernel(unsigned long long limit_ns, int* status) {
  __shared__ uint64_t bar;
  __shared__ int abort_flag;
  if (threadIdx.x == 0) {
    abort_flag = 0;
    sm100::mbar_init(sm100::smem_u32(&bar), 1);
    sm100::mbar_fence_init();
    if (!sm100::mbar_wait_limit(sm100::smem_u32(&bar), 0, &abort_flag, limit_ns)) dlm_set_status(status, DLM_ERR_TIMEOUT);
  }
}

}  // namespace

extern "C" int dlm_selftest_set_wait_limit(dlm_ctx* ctx, uint64_t limit_ns) {
  if (!ctx) return DLM_ERR_NULL;
  if (limit_ns > sm100::kWaitLimitNs) return DLM_ERR_SHAPE;
  if (limit_ns != 0 && limit_ns != sm100::kWaitLimitNs) return DLM_ERR_UNSUPPORTED;   // the two compiled-in limits
  ctx->wait_limit_ns = limit_ns;
  return DLM_OK;
}

extern "C" int dlm_selftest_set_attn_team_max(dlm_ctx* ctx, int max_blocks, int force) {
  if (!ctx) return DLM_ERR_NULL;
  if (max_blocks < 1 || (force != 0 && force != 1)) return DLM_ERR_SHAPE;
  ctx->attn_team_max = max_blocks;
  ctx->attn_team_force = force != 0;
  return DLM_OK;
}

extern "C" int dlm_selftest_wait_timeout(dlm_ctx* ctx, uint64_t limit_ns, void* stream) {
  if (!ctx) return DLM_ERR_NULL;
  if (limit_ns == 0 || limit_ns > 1000000000ull) return DLM_ERR_SHAPE;   // at most one second
  DLM_DEVICE_TRY(ctx);
  wait_probe_kernel<<<1, 32, 0, static_cast<cudaStream_t>(stream)>>>(limit_ns, &ctx->words->status);
  return dlm_launch_ok(ctx, 1);
}
