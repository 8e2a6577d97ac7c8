// dlm_unmask_select: confidence scoring over the vocabulary and top-k unmasking
// (Eq. 2: one logit row per masked position; Eq. 3: fill with the argmax;
//  M_{t-1} = M_t \ U_t).
// dlm_unmask_select_scored: the same ranked by one of several per-position scores computed
// in the same pass over the vocabulary (Sec. 3.1 names a MaskGIT-style, an entropy-based and a Top-K
// margin sampler beside plain confidence; the formulas are the readings given in include/dlm.h).
//
// The pass and the selection are in vocab_pass.cuh; a kind's kernel keeps only the statistics its score needs
//     m   maximum            idx  lowest index attaining it       s   sum exp(z - m)
//     negative entropy = t/s - ln s  with  t = sum (z - m) exp(z - m)
//     margin = (1 - exp(m2 - m)) / s  with  m2 the second largest entry
// (one kernel that kept all of them, 40 instructions per logit, took 66.6 us for 129 MB of logits).
#include "vocab_pass.cuh"

namespace {

int check(const float* logits, int batch, int block_len, int vocab, const uint8_t* masked, const int32_t* tokens, int k,
          const int32_t* tok, const float* conf, const int32_t* sel_idx, const int32_t* n_sel) {
  if (!logits || !masked || !tok || !conf) return DLM_ERR_NULL;
  if (k > 0 && (!tokens || !sel_idx || !n_sel)) return DLM_ERR_NULL;
  if (batch <= 0 || block_len <= 0 || vocab <= 0 || k < 0) return DLM_ERR_SHAPE;
  if (block_len > vocab::kMaxBlockLen || (long long)batch * block_len > vocab::kMaxRows) return DLM_ERR_UNSUPPORTED;
  if (((uintptr_t)logits & 3) != 0) return DLM_ERR_UNSUPPORTED;
  return DLM_OK;
}

vocab::Args make_args(const float* logits, int batch, int block_len, int vocab, uint8_t* masked, int32_t* tokens, int k, int32_t* tok,
                      float* conf, int32_t* sel_idx, int32_t* n_sel, void* entries) {
  vocab::Args a = {};
  a.logits = logits; a.rows = batch * block_len; a.block_len = block_len; a.vocab = vocab; a.k = k; a.masked = masked;
  a.tokens = tokens; a.tok = tok; a.conf = conf; a.sel_idx = sel_idx; a.n_sel = n_sel;
  a.entries = static_cast<vocab::Entry*>(entries);
  return a;
}

}  // namespace

extern "C" size_t dlm_unmask_workspace_bytes(const dlm_ctx* ctx, int batch, int block_len, int vocab) {
  (void)ctx;
  if (batch <= 0 || block_len <= 0 || vocab <= 0) return 0;
  const size_t n_chunks = ((size_t)vocab + vocab::kChunkUnit - 1) / vocab::kChunkUnit;
  return (size_t)batch * block_len * n_chunks * sizeof(vocab::Entry);
}

extern "C" int dlm_unmask_select(dlm_ctx* ctx, const float* logits, int batch, int block_len, int vocab,
                                 uint8_t* masked, int32_t* tokens, int k, int32_t* tok, float* conf,
                                 int32_t* sel_idx, int32_t* n_sel, void* workspace,
                                 size_t workspace_bytes, void* stream) {
  if (!ctx) return DLM_ERR_NULL;
  const int rc = check(logits, batch, block_len, vocab, masked, tokens, k, tok, conf, sel_idx, n_sel);
  if (rc != DLM_OK) return rc;
  const size_t need = dlm_unmask_workspace_bytes(ctx, batch, block_len, vocab);
  if (!workspace || workspace_bytes < need || ((uintptr_t)workspace & 15)) return DLM_ERR_WORKSPACE;
  DLM_DEVICE_TRY(ctx);
  vocab::Args a = make_args(logits, batch, block_len, vocab, masked, tokens, k, tok, conf, sel_idx, n_sel, workspace);
  a.tickets = batch <= kDlmUnmaskTickets ? ctx->words->unmask_tickets : nullptr;
  const int n = vocab::launch_kind<vocab::kConfidence>(a, DLM_SCORE_CONFIDENCE, batch, ctx->num_sms, static_cast<cudaStream_t>(stream));
  if (n < 0) return DLM_ERR_CUDA;
  return dlm_launch_ok(ctx, n);
}

// ---------------------------------------------------------------------------------------
extern "C" size_t dlm_unmask_scored_workspace_bytes(const dlm_ctx* ctx, int batch, int block_len, int vocab) {
  (void)ctx;
  if (batch <= 0 || block_len <= 0 || vocab <= 0) return 0;
  const size_t n_chunks = ((size_t)vocab + vocab::kChunkUnit - 1) / vocab::kChunkUnit;
  return (size_t)batch * block_len * n_chunks * sizeof(vocab::Entry);
}

extern "C" int dlm_unmask_select_scored(dlm_ctx* ctx, const float* logits, int batch, int block_len, int vocab,
                                        uint8_t* masked, int32_t* tokens, int k, int score_kind, const float* noise,
                                        int32_t* tok, float* conf, float* score, float* zmax, int32_t* sel_idx,
                                        int32_t* n_sel, void* workspace, size_t workspace_bytes, void* stream) {
  if (!ctx || !logits || !masked || !tok || !conf || !score || !zmax) return DLM_ERR_NULL;
  if (k > 0 && (!tokens || !sel_idx || !n_sel)) return DLM_ERR_NULL;
  if (batch <= 0 || block_len <= 0 || vocab <= 0 || k < 0) return DLM_ERR_SHAPE;
  if (score_kind < DLM_SCORE_CONFIDENCE || score_kind > DLM_SCORE_LOG_CONF_PLUS_NOISE) return DLM_ERR_SHAPE;
  if (score_kind == DLM_SCORE_LOG_CONF_PLUS_NOISE && !noise) return DLM_ERR_NULL;
  if (block_len > vocab::kMaxBlockLen || (long long)batch * block_len > vocab::kMaxRows) return DLM_ERR_UNSUPPORTED;
  if (((uintptr_t)logits & 3) != 0) return DLM_ERR_UNSUPPORTED;
  const size_t need = dlm_unmask_scored_workspace_bytes(ctx, batch, block_len, vocab);
  if (!workspace || workspace_bytes < need || ((uintptr_t)workspace & 15)) return DLM_ERR_WORKSPACE;
  DLM_DEVICE_TRY(ctx);
  vocab::Args a = {};
  a.logits = logits; a.rows = batch * block_len; a.block_len = block_len; a.vocab = vocab; a.k = k; a.masked = masked;
  a.tokens = tokens; a.tok = tok; a.conf = conf; a.sel_idx = sel_idx; a.n_sel = n_sel;
  a.score = score; a.zmax = zmax; a.noise = noise;
  a.entries = static_cast<vocab::Entry*>(workspace);
  a.tickets = batch <= kDlmUnmaskTickets ? ctx->words->unmask_tickets : nullptr;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  const int n = score_kind == DLM_SCORE_NEG_ENTROPY ? vocab::launch_kind<vocab::kEntropy>(a, score_kind, batch, ctx->num_sms, s)
              : score_kind == DLM_SCORE_MARGIN      ? vocab::launch_kind<vocab::kMargin>(a, score_kind, batch, ctx->num_sms, s)
                                                    : vocab::launch_kind<vocab::kConfidence>(a, score_kind, batch, ctx->num_sms, s);
  if (n < 0) return DLM_ERR_CUDA;
  return dlm_launch_ok(ctx, n);
}

// ---------------------------------------------------------------------------------------
// dlm_unmask_select_static: the same pass, with the per-row partial reductions kept in
// a fixed device array that is part of the library image, for callers that cannot allocate
// device memory at all.  Without a context there are no tickets: the selection is a second kernel.
namespace {

constexpr int kStaticEntries = 65536;  // 1 MiB: rows x chunks of one call may not exceed this
static __device__ __align__(256) vocab::Entry g_static[kStaticEntries];

constexpr int kMaxDevices = 64;
constexpr int kStaticSms = 148;              // blocks are dealt as on the device the kernels are written for
vocab::Entry* g_static_addr[kMaxDevices];   // device address of the array, per device (0 = not looked up yet)

}  // namespace

extern "C" int dlm_unmask_select_static(const float* logits, int batch, int block_len, int vocab,
                                        uint8_t* masked, int32_t* tokens, int k, int32_t* tok, float* conf,
                                        int32_t* sel_idx, int32_t* n_sel, void* stream) {
  const int rc = check(logits, batch, block_len, vocab, masked, tokens, k, tok, conf, sel_idx, n_sel);
  if (rc != DLM_OK) return rc;
  const int n_chunks = (vocab + vocab::kChunkUnit - 1) / vocab::kChunkUnit;
  if ((long long)batch * block_len * n_chunks > kStaticEntries) return DLM_ERR_WORKSPACE;
  int device = -1;
  DLM_CUDA_TRY(cudaGetDevice(&device));
  if (device < 0 || device >= kMaxDevices) return DLM_ERR_UNSUPPORTED;
  if (!g_static_addr[device]) {
    // In host code the array's name is only a handle; its address on the current device has to be
    // asked for, once per device.
    vocab::Entry* addr = nullptr;
    if (cudaGetSymbolAddress(reinterpret_cast<void**>(&addr), g_static) != cudaSuccess || !addr) return DLM_ERR_CUDA;
    g_static_addr[device] = addr;
  }
  vocab::Args a = make_args(logits, batch, block_len, vocab, masked, tokens, k, tok, conf, sel_idx, n_sel, g_static_addr[device]);
  if (vocab::launch_kind<vocab::kConfidence>(a, DLM_SCORE_CONFIDENCE, batch, kStaticSms, static_cast<cudaStream_t>(stream)) < 0)
    return DLM_ERR_CUDA;
  return cudaGetLastError() == cudaSuccess ? DLM_OK : DLM_ERR_CUDA;
}
