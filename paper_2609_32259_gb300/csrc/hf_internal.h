// Internal declarations shared by the library's translation units.
#pragma once

#include <cuda.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <mutex>
#include <string>

#include "heterofold.h"

namespace hf {

constexpr int kMaxReq = 1024;        // requests per call
constexpr int kMaxLayersR = 128;     // receiver layers
constexpr int kMaxSeg = 8;           // map input segments per receiver layer (Eq. 1: 3;
                                     // KV Ridge's layer routing: 8)
constexpr int kMaxTerms = 2;         // sender layers blended into one segment
constexpr int kMaxHeadDim = 256;
constexpr int kMaxBatch = 16;        // directions per hf_transfer_batch call

// One receiver layer's map input: n_seg segments of d_S features each;
// segment s is sum_t w[s][t] * (pooled sender layer layer[s][t]).
struct LayerSegs {
  int32_t n_seg;
  int32_t n_terms[kMaxSeg];
  int32_t layer[kMaxSeg][kMaxTerms];
  float w[kMaxSeg][kMaxTerms];
};

// Per-plan metadata that lives in the caller's device workspace.
struct WorkspaceLayout {
  size_t status;     // int32: device status bits
  size_t n_distinct; // int32: number of distinct alignment rows U
  size_t segs;       // LayerSegs[L_r]
  size_t inv_r;      // float[L_r * 2]  (1 / r)
  size_t inv_freq;   // float[D_r / 2]
  size_t inv_freq_s; // float[D_s / 2]: sender RoPE (sender_k_rotated)
  size_t r_tok_ptr;  // int32[n_req + 1]
  size_t r_pos0;     // int32[n_req]
  size_t s_tok_ptr;  // int32[n_req + 1]
  size_t s_pos0;     // int32[n_req]
  size_t spos;       // int32[T_s] sender RoPE positions (sender_k_rotated), else one word
  size_t s_row0;     // int32[n_req] sender-cache row of each request's span
  size_t srow;       // int32[T_s] sender-cache row of each aligned token (spans), else one word
  size_t run_ptr;    // int32[T_r + 1]: first receiver row of each distinct row
  size_t ucol;       // int32[T_r]: sender column of each distinct row (one-entry rows)
  size_t upos;       // int32[T_r]: RoPE position of each distinct row's first receiver row
  size_t pos;        // int32[T_r]: RoPE position of each receiver row
  size_t dst_row;    // int32[T_r]: destination row of each receiver row
  size_t new_flag;   // int32[T_r]: 1 where a receiver row starts a new distinct row, then its
                     // running sum: the one-based number of each row's distinct row
  // pooling after the map (overlap mean pooling): windows of 128 aligned
  // sender tokens with stride S = 128 - h, h the widest row's column span
  size_t win_info;   // int32[4]: h, S, number of windows, unused
  size_t row_key;    // int32[T_r]: first column of each row, then its running maximum
  size_t win_ptr;    // int32[T_s + 2]: first receiver row of each window
  size_t total;      // what a plan cannot do without
  // operand rows made before the transfer (see x_rows below), for as many
  // receiver layers as fit kOperandBytes, one at least
  size_t xbuf;
  size_t total_made; // total with them (equal to it where no rows are made)
  int64_t x_rows;
  int x_layers, made;
};

// Copied bf16 rows may take single-CTA tiles where at most kSingleRows distinct
// rows, one such tile's, are to be expected: in as many tokens on either side, and
// with Token Alignment, where about a quarter of the receiver's rows are distinct,
// in kSingleTokens receiver tokens.  A pair's 256-row tile is then mostly padding,
// and the maps, read once, are what bounds the transfer (256 tokens, Ministral ->
// Llama-shaped, whole step: 104 us with pairs, 95 us single, of which the maps'
// bytes take 60).  With a second block of rows every map is read twice: same-index
// Llama -> Ministral-shaped, 192 tokens 128 us in pairs, 146 single, 512 tokens 195
// and 226; Token Alignment, 512 tokens (129 distinct) 138 and 156.
constexpr int64_t kSingleRows = 128, kSingleTokens = 400;

// Bytes of made operand rows to aim at: receiver layers per launch, so that
// a launch's last round of tiles is a small part of it.
constexpr size_t kOperandBytes = static_cast<size_t>(512) << 20;

WorkspaceLayout workspace_layout(const hf_plan_desc& d);

// Constant tables copied into the workspace by the plan kernels.  They are
// passed by value as kernel parameters, so plan creation issues no host
// copies; the layer table goes to a kernel of its own because one launch's
// parameters are limited to 32 KB.
struct PlanConsts {
  int32_t L_r, D_r, D_s, n_req;
  float inv_r[2 * kMaxLayersR];
  float inv_freq[kMaxHeadDim / 2];
  float inv_freq_s[kMaxHeadDim / 2];
  int32_t r_tok_ptr[kMaxReq + 1];
  int32_t r_pos0[kMaxReq];
  int32_t s_tok_ptr[kMaxReq + 1];
  int32_t s_pos0[kMaxReq];
  int32_t s_row0[kMaxReq];
};
struct SegTables {
  int32_t L_r;
  LayerSegs segs[kMaxLayersR];
};
struct PlanTables {
  PlanConsts c;
  SegTables s;
};
static_assert(sizeof(PlanConsts) < 32000, "PlanConsts must fit the kernel parameter space");
static_assert(sizeof(SegTables) < 32000, "SegTables must fit the kernel parameter space");

}  // namespace hf

struct hf_plan_s {
  hf_plan_desc desc;  // host-array fields are cleared after copying
  int d_s, d_r, K, n_seg;
  int64_t T_s, T_r;
  int BN;
  bool gather;  // every map input row is a single unweighted sender row
  bool split;   // computed bf16 operand rows go to the tensor core as value + residual
  bool staged;  // split rows of one entry each: raw sender atoms staged by cp.async
  bool rope;    // receiver keys get RoPE
  bool unrot;   // sender keys carry RoPE and are rotated back in the builder
  bool span;    // aligned sender tokens are spans inside a longer sender cache
  bool pam;     // pooling after the map: map input rows are sender rows in windows
  bool wide;    // tiles of two 256-column blocks (operand rows built by the loader warps)
  // few distinct rows (kSingleRows): tiles of 128 rows x 256 columns on single
  // CTAs instead of 256 x 256 on pairs, where every plan of the launch has few
  bool few_rows;
  // bit c: the map input rows of role c (pooled, blended, weighted or rotated
  // back) are made by a pass of their own before the transfer, which then
  // copies them; x_rows rows (distinct rows, or sender tokens with pooling after
  // the map) of x_layers receiver layers at a time.  0 where rows are copies, in
  // fp32, and where the workspace holds only WorkspaceLayout::total bytes: the
  // loader warps then build what is not a copy, as they do in captured transfers.
  int made;
  int64_t x_rows;
  int x_layers;
  // The made rows are the plan's, not the call's: a transfer on another stream
  // takes them after x_done, the end of the transfer before it.
  std::mutex x_mutex;
  cudaEvent_t x_done = nullptr;
  int64_t s_rows;  // sender-cache rows per (layer, role)
  char* ws;
  size_t ws_bytes;
  hf::WorkspaceLayout lay;
  int32_t s_tok_ptr_last;
  int32_t max_sender_layer[hf::kMaxLayersR];  // highest sender layer each receiver layer reads
  // hf_transfer_host: copy streams and events, created on first use
  int aux_device = -1;
  cudaStream_t s_h2d = nullptr, s_d2h = nullptr;
  cudaEvent_t* events = nullptr;
  int n_events = 0;
};

namespace hf {

// Prologue kernels of a transfer (alignment, plan metadata) of at most
// kFusedRows tokens on either side and kFusedReq requests run as one launch.
// Their time is a chain of latencies, so a thread takes one row (four above
// 8,192 rows), and one CTA all of them up to 1,024 (the cluster's exchange
// costs about 1 us), a cluster of eight above.  The launch overlaps the end of
// the kernel before it (programmatic dependent launch).
constexpr int kFusedRows = 32768;
constexpr int kFusedReq = 64;
inline int fused_rows_per_thread(int64_t rows) { return rows <= 8192 ? 1 : 4; }
template <typename Kern, typename... Args>
cudaError_t launch_fused_rows(Kern kern, int64_t rows, cudaStream_t stream, const Args&... args) {
  const int ctas = rows <= 1024 ? 1 : 8, per = ctas * fused_rows_per_thread(rows);
  const int64_t threads = ((rows + per - 1) / per + 31) / 32 * 32;
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = static_cast<unsigned>(ctas);
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.gridDim = dim3(static_cast<unsigned>(ctas), 1, 1);
  cfg.blockDim = dim3(static_cast<unsigned>(threads < 128 ? 128 : threads), 1, 1);
  cfg.stream = stream;
  cfg.attrs = attr;
  cfg.numAttrs = 2;
  return cudaLaunchKernelEx(&cfg, kern, args...);
}

// A launch that may overlap the end of the kernel before it in the stream
// (programmatic dependent launch): the kernel calls depend_wait before its
// first global access.
template <typename Kern, typename... Args>
cudaError_t launch_dependent(Kern kern, dim3 grid, dim3 block, size_t smem, cudaStream_t stream,
                             const Args&... args) {
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = stream;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kern, args...);
}

void set_error(const std::string& msg);
hf_status cuda_fail(cudaError_t e, const char* what);
int device_sm_count();

hf_status launch_plan_kernels(hf_plan_s* p, const PlanTables& tables, cudaStream_t stream);
hf_status plan_build(const hf_plan_desc* desc, void* d_workspace, size_t workspace_bytes,
                     cudaStream_t stream, hf_plan_s* p, PlanTables* t);
// One transfer-kernel launch over receiver layers [l_begin, l_end) (l_end < 0: all).
// stall (test hook): the map producer withholds its first atom, so the
// launch ends through the bounded waits with HF_CHECK_TIMEOUT.
hf_status launch_transfer(hf_plan_s* p, const void* sender, void* receiver, cudaStream_t stream,
                          int l_begin = 0, int l_end = -1, bool stall = false);
// The operand rows of receiver layers [l_begin, l_end) of a plan with made rows.
hf_status launch_operands(const hf_plan_s* p, const void* sender, cudaStream_t stream, int l_begin,
                          int l_end);
// Several plans in one launch: they must share the dtype, the operand path
// and where the pooling happens, and make no operand rows (batch_compatible);
// n <= kMaxBatch.
bool batch_compatible(const hf_plan_s* const* plans, int n, cudaStream_t stream);
hf_status launch_transfer_batch(hf_plan_s* const* plans, const void* const* senders,
                                void* const* receivers, int n, cudaStream_t stream);

// Device buffers of gemm_f32 (part of hf_recolor_fit's workspace): the bf16
// planes of both operands, split-K partials, and an error word (set when a
// pipeline wait of the product kernel ran out).
struct GemmWork {
  void* planes_a;
  size_t planes_a_bytes;
  void* planes_b;
  size_t planes_b_bytes;
  float* partial;
  size_t partial_bytes;
  int32_t* err;
};
// Bytes of the three bf16 planes of an operand with `rows` rows and K columns.
size_t gemm_planes_bytes(int64_t rows, int64_t K);
// An operand that is already split: three planes of `rows_p` rows each,
// K-major bf16, the operand's row 0 at plane row `row0`.
struct GemmPlanes {
  const void* planes;
  int64_t rows_p;
  int row0;
};
// Which part of C a product writes.  tri: of the 256 x 256 tiles of row block
// m, those left of column diag_col and those that reach column diag_col +
// 256 m or beyond (diag_col 0: a symmetric product's upper triangle).  Columns
// in [fresh_lo, fresh_hi) (multiples of 64) take no C_in.
struct GemmShape {
  bool tri = false;
  int diag_col = 0;
  int fresh_lo = 0, fresh_hi = 0;
  int flush = 0;  // > 0: a sum over K goes to C in parts of this many 64-wide atoms (C += only)
};
// C = alpha op(A) op(B) + beta C_in + diag I of split operands with k_p
// columns (a multiple of 64, zero-padded).
hf_status gemm_planes(cudaStream_t s, const GemmWork& wk, int M, int N, int k_p, float alpha,
                      const GemmPlanes& a, const GemmPlanes& b, float beta, float* C, int64_t ldc,
                      const GemmShape& shape, const float* Cin = nullptr, float diag = 0.f);
// C[M x N] = alpha op(A) op(B) + beta C_in + diag I (row-major C and C_in,
// leading dimension ldc; C_in NULL = C), op(A)(i, k) = A[i * a_i + k * a_k],
// op(B)(k, j) = B[k * b_k + j * b_j], in fp32 accuracy on the tensor cores
// (hf_gemm.cu).  Asynchronous on s.
hf_status gemm_f32(cudaStream_t s, const GemmWork& wk, int M, int N, int K, float alpha,
                   const float* A, int64_t a_i, int64_t a_k, const float* B, int64_t b_k,
                   int64_t b_j, float beta, float* C, int64_t ldc, const float* Cin = nullptr,
                   float diag = 0.f);

// Tensor map of [n][rows][cols] bf16 with boxes of box_rows x 32 columns of one
// matrix, in the 64-byte swizzle.
hf_status bf16_strip_map(CUtensorMap* map, const void* base, uint64_t n, uint64_t rows,
                         uint64_t cols, uint32_t box_rows);

// Triangular factor of the symmetric positive definite n x n matrix W
// (row-major, leading dimension ld, n a multiple of kFactorBlock; the blocks on
// and above the diagonal are read): W = L L^T.  On return row i holds
// L^{-1}'s row i in columns 0 .. i (zeros to the end of the diagonal block,
// work values after it).  upper (or NULL, cleared before): L^T, n_upper x
// n_upper.  Tt: kFactorBlock^2 floats; planes: tri_factor_planes_bytes(n).  A
// pivot that is not above *thr sets *flag (cleared before) and the result is
// of no use.
// Up to two matrices are factored side by side: a chain of latencies each.
constexpr int kFactorBlock = 128;
size_t tri_factor_planes_bytes(int n);
struct TriProblem {
  float* W;
  int64_t ld;
  int n;
  float* Tt;
  void* planes;
  const float* thr;
  float* upper;
  int n_upper;
};
hf_status tri_factor(cudaStream_t s, const GemmWork& wk, const TriProblem* problems, int count,
                     int32_t* flag);

}  // namespace hf

#define HF_CUDA_TRY(expr, what)                      \
  do {                                               \
    cudaError_t e__ = (expr);                        \
    if (e__ != cudaSuccess) return hf::cuda_fail(e__, what); \
  } while (0)
