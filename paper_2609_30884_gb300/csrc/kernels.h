// Internal launcher interface between the C ABI layer (api.cu) and the kernels.
#pragma once

#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stddef.h>
#include <stdint.h>

#include <atomic>

namespace crf {

// One-time set-up that CUDA keeps per device (kernel attributes): bit d of the mask records
// device d. Host threads may race to do it; doing it twice is harmless.
class PerDevice {
 public:
  // Sets *dev to the current device; true while its set-up is still to do.
  bool pending(int* dev) const {
    if (cudaGetDevice(dev) != cudaSuccess) *dev = -1;
    return *dev < 0 || *dev >= 64 || !((mask_.load(std::memory_order_acquire) >> *dev) & 1u);
  }
  void done(int dev) {
    if (dev >= 0 && dev < 64) mask_.fetch_or(1ull << dev, std::memory_order_acq_rel);
  }

 private:
  std::atomic<uint64_t> mask_{0};
};

constexpr int kMaxReq = 32;   // equals CRF_MAX_REQUESTS
constexpr int kPage = 16;
constexpr int kRankPad = 16;  // LoRA rank padded to one K=16 MMA step
// The scaled LoRA down product is kept as a bf16 pair hi + lo (lo = bf16(v - hi)): module
// slot j holds hi at columns [32j, 32j + 16) and lo at [32j + 16, 32j + 32) of a [rows, kXaCols]
// buffer. A projection GEMM computes it for its rows and reads it back as one 64-wide K block
// against BX = [B | B] rows (kBxCols wide) of the module (the up product).
constexpr int kXaCols = 128;
constexpr int kBxCols = 64;

// Programmatic dependent launch for chains of short kernels. While a PdlScope is alive on the
// calling thread, the launchers below that go through launch_kernel() give their kernels the
// programmatic-stream-serialization attribute: such a kernel becomes resident while its
// predecessor in the stream still runs, sets itself up (a weight pass requests its first weights) and
// then waits for it (griddep_wait). Every kernel launched this way calls griddep_wait before it
// touches memory that an earlier kernel of the call may write, and before it ends, since the kernels
// behind it count on all before it having ended. Weights, and cached K/V pages that the call does not
// write, may be read before that wait, so a chain with such reads opens with an ordinary launch or a
// memset: what the caller enqueued before has then ended and is visible. Window calls, generation
// steps, the LM head pass of a KL call, the KL reduction over few rows and drift open a scope.
class PdlScope {
 public:
  PdlScope();
  ~PdlScope();
  PdlScope(const PdlScope&) = delete;
  PdlScope& operator=(const PdlScope&) = delete;

 private:
  bool prev_;
};
bool pdl_active();

template <typename... KArgs, typename... Args>
cudaError_t launch_kernel(void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem,
                          cudaStream_t stream, Args&&... args) {
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = stream;
  cfg.attrs = attr;
  cfg.numAttrs = pdl_active() ? 1 : 0;
  return cudaLaunchKernelEx(&cfg, kernel, static_cast<Args&&>(args)...);
}

// Rows of a batched activation matrix that belong to each request.
struct ReqTable {
  int n;
  int num_pages;  // pool size; page ids are checked against it in a CRF_DEBUG build
  int row0[kMaxReq];
  int len[kMaxReq];
  const int32_t* page_table[kMaxReq];
};

enum EpiKind : int {
  kEpiQkv = 1,        // +bias, RoPE(q,k); q -> qbuf, k/v -> KV pages    (Eq. S3)
  kEpiResid = 2,      // out = bf16(resid + acc)                         (o / down projection)
  kEpiSwiGLU = 3      // out = bf16(silu(gate) * up), tile = [gate | up]  (MLP)
};

// Host description of one GEMM  D[M, cols] = A[M, K] * B[cols, K]^T (+ LoRA ext) -> epilogue.
// Column space: `ngroups` groups laid side by side, each with its own weight
// matrix (plain mode, nseg == 1), or one group whose tiles stack `nseg` equal
// row segments of different matrices (paired / stacked mode, ngroups == 1).
struct GemmDesc {
  const void* A;          // [M, K]
  int M, K;
  int ngroups, nseg;
  const void* B[3];       // map index g + s; [B_rows, K]
  int B_rows[3];
  int group_cols[3];      // valid output columns per group (plain) / per segment (stacked)
  // Unmerged LoRA (Eq. S3), computed inside the same launch, which first forms XA[:, 32j .. 32j + 32) =
  // hi/lo of (alpha/r) x A_j^T for the n_slots adapted modules (LA[j] = A_j, [rank, K]) of each
  // 256-row block and raises xa_flags[row block]; every output tile of an adapted group then adds one K
  // block: XA[:, xa_base[g] .. + 64] against BX[i] (the module's [B | B] rows under its slot, zeros
  // elsewhere; [B_rows[i], kBxCols], map index i like B).
  void* XA;
  int n_slots;
  const void* LA[3];
  const void* BX[3];
  int rank;
  float scale;            // alpha / r
  int* xa_flags;          // [row blocks of 256], zero before the launch
  int ext_on[3];          // per group
  int ext_steps[3];       // K = 16 steps of the block that carry data (2 per module)
  int xa_base[3];
  // epilogue
  int epi;
  void* out;
  int ldo;
  const void* resid;
  int ld_resid;
  const void* bias[3];
  const float2* rope;     // (cos, sin) of pair i at position p: entry ((i / 2) rope_positions + p) 2 + i % 2
  int rope_positions;
  int head_dim, n_kv_heads;
  void* qbuf;
  int ldq;
  void* kpages;
  void* vpages;
  ReqTable req;
  int* status;
  const int* abort;       // per-call abort word (call_aborted), or null
};

// Launch the tcgen05 projection GEMM (CTA pairs; tiles of 256 rows and 256, 192 or 128 columns).
cudaError_t launch_gemm(const GemmDesc& d, int num_sms, cudaStream_t stream);

// ------------------------------------------------------------------ other kernels
struct RowPositions {
  int pos[kMaxReq];
};
// BX rows of up to 4 modules: out[m][r, :] = 0 except columns [col_off[m], col_off[m] + 32) =
// [B_m[r, 0:16] | B_m[r, 0:16]] (rank padded with zeros); a null B_m gives all-zero rows.
struct BextDesc {
  const __nv_bfloat16* B[4];
  __nv_bfloat16* out[4];
  int rows[4];
  int col_off[4];
  int n, rank;
};
// RMSNorm of `rows` rows; with `bx`, the same launch also builds those BX rows (extra blocks).
cudaError_t launch_rmsnorm(const __nv_bfloat16* x, const __nv_bfloat16* g, __nv_bfloat16* y,
                           int rows, int hidden, float eps, cudaStream_t stream,
                           const BextDesc* bx = nullptr);
// Token ids outside [0, vocab) read row 0 and set kStatusBounds in *status.
cudaError_t launch_embed(const __nv_bfloat16* embed, const int32_t* tokens, __nv_bfloat16* out,
                         int n, int hidden, int vocab, int* status, cudaStream_t stream);

// Causal GQA prefill attention over the paged cache of the current layer.
struct AttnDesc {
  const __nv_bfloat16* q;  // [rows, Hq*d] post-RoPE
  const __nv_bfloat16* kpages;  // [P][Hkv][16][d]
  const __nv_bfloat16* vpages;
  __nv_bfloat16* out;      // [rows, Hq*d]
  int ldo;
  int n_q_heads, n_kv_heads, head_dim;
  ReqTable req;
  int* status;
  const int* abort;
};
// tcgen05, S and O in TMEM: num_pages of the pool, total_rows of q (for the TMA maps).
cudaError_t launch_attention_tc(const AttnDesc& d, int num_pages, int total_rows, int num_sms,
                                cudaStream_t stream);

// ------------------------------------------------------------------ decode rows
// The last prefix row of each request through the layers after its window, and the rows of a
// generation step: fp32 rows, one weight pass (rows GEMM) for all of them, short kernels between.
constexpr int kRowsMax = 64;         // rows of one weight pass
constexpr int kRowsMaxSeg = 3;       // projections that share an input
constexpr int kRowsMaxSplits = 16;   // K splits of a weight tile
constexpr int kRowsRing = 150 * 1024;     // shared-memory ring of a pass inside a dependent chain
constexpr int kRowsRingMax = 200 * 1024;  // and of one alone on its SMs
// fp32 rows enter a weight pass as bf16 terms: three (exact) for one or two rows, two (about 16
// mantissa bits) from three rows on. Chosen by the rows of the whole call, so that equal rows in
// different passes stay equal.
inline int rows_terms(int total_rows) { return total_rows <= 2 ? 3 : 2; }

// How a weight pass over `nseg` projections is cut: 128-row weight tiles (tile0[s]: first of
// segment s; tile0[nseg]: the tile of the adapter's A rows, module i at its rows 16 i, if any) and
// K splits. Its output has `ncols` = 128 x tiles columns: output j of segment s is column
// 128 tile0[s] + j.
struct RowsPlan {
  int tile0[kRowsMaxSeg + 1];
  int tiles, splits, ncols;
  int kb, sub;  // K steps of a tile, each sub x 64 wide
};
RowsPlan rows_plan(int nseg, const int* outs, bool lora, int in_dim, int num_sms, bool split = true);
struct RowsGemmDesc {
  const __nv_bfloat16* W[kRowsMaxSeg];  // [out, in_dim]
  int out[kRowsMaxSeg];
  int nseg;
  const __nv_bfloat16* LA[kRowsMaxSeg];  // LoRA A rows [rank, in_dim] of the adapted modules
  int n_lora, rank;
  int in_dim;
  const __nv_bfloat16* x;  // [rows * terms, in_dim]: term t of row r at r * terms + t
  int rows, terms;
  float* y;                // [splits][rows][ncols] partial sums
  int ncols;               // 0: the plan's
  // when given: row r is scaled by rsqrt(sum_i nss[r][i] / in_dim + eps) (RMSNorm, rows enter as x * g)
  const float* nss;        // [rows, slices]
  int slices;
  float eps;
  int* status;
  const int* abort;        // per-call abort word, or null: a rejected call stores nothing
  bool alone;              // a long pass by itself (the LM head): the largest ring
};
cudaError_t launch_rows_gemm(const RowsGemmDesc& d, const RowsPlan& plan, int num_sms, cudaStream_t stream);

// A weight pass's output as its consumer reads it: element (r, col) is the sum over s of
// p[(s * rows + r) * ncols + col].
struct RowPart {
  const float* p;
  int splits, rows, ncols;
};
// The adapter's up product for decode rows, added where the projection's output is consumed:
// up[r, j] = sum_k B[j, k] (alpha / r) xa[r, k] with B [out_dim, rank] bf16 and xa the columns
// xa_col.. of the pass's output; a null B adds nothing.
struct RowUp {
  const __nv_bfloat16* B;
  int xa_col;
};
struct RowLora {
  int rank;
  float scale;  // alpha / r
};
// Where rows that join at this layer start: a bf16 row, or a token's embedding.
struct RowStart {
  const __nv_bfloat16* row[kMaxReq];
  const int32_t* token[kMaxReq];
  const __nv_bfloat16* embed;
  int vocab;
};
// The residual stream before a norm: x[r] = its start (rows >= up_rows), else x[r] + the pending
// pass's output (from column 0) + up product; then xs[r] = the terms of x[r] * g and nss[r][slice] =
// the slice's sum of squares, for the pass that applies 1 / rms. Token ids outside [0, vocab) read
// row 0 and set kStatusBounds.
int norm_slices(int dim);
cudaError_t launch_add_norm_rows(float* x, int dim, int rows, const RowPart& part, const RowUp& up, const RowLora& lora,
                                 int up_rows, const RowStart* start, const __nv_bfloat16* g, __nv_bfloat16* xs,
                                 int terms, float* nss, int* status, cudaStream_t stream);
// out[r] = bf16(x[r] + the last pass's output + up product) for every row with a non-null out.
struct RowOuts {
  __nv_bfloat16* out[kMaxReq];
};
cudaError_t launch_finish_rows(const float* x, int dim, int rows, const RowPart& part, const RowUp& up,
                               const RowLora& lora, const RowOuts& outs, const int* abort, cudaStream_t stream);
// ms[r] = the terms of silu(g) * u, g and u the pass's columns 0.. and up_col.. plus their up products.
cudaError_t launch_swiglu_rows(const RowPart& part, int up_col, int f, const RowUp& up_g, const RowUp& up_u,
                               const RowLora& lora, __nv_bfloat16* ms, int terms, cudaStream_t stream);
// LM-head inputs: rows [0, n_ref) of ref, then of cur (bf16): xs = the terms of h * g, nss as above.
cudaError_t launch_head_rows(const __nv_bfloat16* ref, const __nv_bfloat16* cur, int n_ref, int hidden,
                             const __nv_bfloat16* g, __nv_bfloat16* xs, int terms, float* nss, cudaStream_t stream);
// Single-query attention of `rows` decode rows (one per request) over pages [0, pos) plus own k/v.
struct DecodeAttnDesc {
  RowPart qkv;             // the q|k|v pass's output
  int col[3];              // its first columns of q, k, v
  RowUp up[3];
  RowLora lora;
  const __nv_bfloat16* bias[3];
  const float2* rope;      // launch_open_call's table, or [rows][head_dim / 2] with rope_by_row
  int rope_by_row, rope_positions;
  __nv_bfloat16* kpages;
  __nv_bfloat16* vpages;
  int write_kv;            // the row's own k, v go into slot pos % 16 of page page_table[pos / 16]
  const int32_t* page_table[kMaxReq];  // per decode row
  int pos[kMaxReq];        // position of the decode row (= number of cached keys before it)
  __nv_bfloat16* out;      // the terms of o: [rows * terms, Hq*d]
  int terms;
  float* part;             // scratch [rows, Hq, splits, d + 2]
  int rows, n_q_heads, n_kv_heads, head_dim, splits;
  int total_chunks, blocks, per_pair;  // set by launch_decode_attention
  const int* abort;        // per-call abort word, or null
};
// Decode attention: q, k, v finished from the pass's output (bias, up products, rotate-half RoPE),
// streamed over 128-position chunks (TMA-staged pages, one block per SM walking an equal run of
// the chunks of all rows and kv heads) + merge of the blocks' partials. `splits` in the descriptor must be at
// least decode_attention_splits(max position + 1).
cudaError_t launch_decode_attention(const DecodeAttnDesc& d, int num_pages, int num_sms, int* status,
                                    cudaStream_t stream);
int decode_attention_splits(int max_positions);
// One block whose wait on an mbarrier nothing arrives on runs out after the bounded-wait limit
// and raises kStatusTimeout in *status (the failure path, exercised without a fault).
cudaError_t launch_wait_selftest(int* status, cudaStream_t stream);
// out[r] = argmax of logits row r (lowest index among equal maxima). key, count: one entry per row, zero
// before the launch.
cudaError_t launch_argmax_rows(const float* logits, int rows, int vocab, unsigned long long* key, int* count,
                               int32_t* out, int num_sms, cudaStream_t stream, const int* abort);
// dst[0 .. n) = src[0 .. n) (bf16), unless the call's abort word is set.
cudaError_t launch_copy_rows(__nv_bfloat16* dst, const __nv_bfloat16* src, size_t n, const int* abort,
                             cudaStream_t stream);
// The first kernel of crf_recompute_window and crf_decode_step. With `check`: every id of every
// table in [0, num_pages) and no page twice across the tables; a failure sets *abort and raises
// kStatusPages in *status. `table` is scratch of (mask + 1) ints, mask + 1 a power of two at least
// twice the ids checked, zero before the launch. And the call's angles, (cos, sin) of rotation pair i
// at position p: for `rows`, angles[r][head_dim / 2] of n_pos = rows positions; else of positions
// 0 .. n_pos - 1 at angles[((i / 2) n_pos + p) 2 + i % 2], so that neighbouring rows of a projection
// read neighbouring entries.
struct PageCheck {
  const int32_t* pt[kMaxReq];
  int first[kMaxReq + 1];  // prefix of the tables' id counts
  int n;
};
cudaError_t launch_open_call(const PageCheck& pc, int num_pages, int* table, uint32_t mask, int* abort, int* status,
                             bool check, float2* angles, int n_pos, const RowPositions* rows, int head_dim,
                             double theta, cudaStream_t stream);

// Logits [rows, V] fp32 of rows given as terms and sums of squares (launch_head_rows, launch_add_norm_rows).
cudaError_t launch_lm_head(const __nv_bfloat16* W, const __nv_bfloat16* xs, int terms, const float* nss, int rows,
                           int vocab, int hidden, float eps, float* logits, int num_sms, int* status,
                           cudaStream_t stream, const int* abort = nullptr);
// KL per row from fp32 logits; part: scratch [rows][splits][5].
cudaError_t launch_kl(const float* zref, const float* zcur, int rows, int vocab, float* out,
                      float* part, int splits, int num_sms, cudaStream_t stream);
// Vocabulary splits per row of the KL reduction: about two blocks per SM over all rows, at least
// 1024 logits per split, at most kKlMaxSplits. Every KL entry point uses this count, so they
// reduce in the same order.
constexpr int kKlMaxSplits = 256;
inline int kl_split_count(int num_sms, int n_rows, int vocab) {
  int want = (2 * num_sms + n_rows - 1) / (n_rows > 0 ? n_rows : 1);
  const int by_vocab = (vocab + 1023) / 1024;
  want = want < by_vocab ? want : by_vocab;
  want = want < kKlMaxSplits ? want : kKlMaxSplits;
  return want < 1 ? 1 : want;
}

// Drift: per (layer, module) squared norms; see crf_drift.
struct DriftItem {
  const __nv_bfloat16* A0; const __nv_bfloat16* B0;
  const __nv_bfloat16* A1; const __nv_bfloat16* B1;
  int in_dim, out_dim;
  int out_index;           // layer * 7 + module
};
// Tensor-core drift (mma.sync Grams over the long dimensions, then a dependent-launched fp64
// combine per item); `workspace` is device scratch of drift_workspace_bytes(num_sms, rank,
// n_items) bytes (partial Grams). Launches drift_launches(n) kernels. out_sq holds n_out
// (layer, module) pairs; the entries of modules outside `adapted_mask` are cleared. A copy wait
// that exceeds its time limit sets kStatusTimeout in `status`.
size_t drift_workspace_bytes(int num_sms, int rank, int n_items);
int drift_launches(int n_items);
cudaError_t launch_drift(const DriftItem* items, int n_items, int rank, int n_out, int adapted_mask,
                         void* workspace, int num_sms, float* out_sq, int* status, cudaStream_t stream);

}  // namespace crf
