// The short kernels between the weight passes of the decode rows: residual update + RMSNorm,
// SwiGLU, the rows' way out, the LM head's inputs. Each adds a pass's K splits and the adapter's
// up product where it consumes the pass's output, and leaves its own output as the bf16 terms that
// the next pass multiplies. They are bound by latency (a few hundred KB at most): one element per
// thread, every load of a thread independent of its others, weights (norm gains, B rows) read
// before the wait for the kernel they depend on.
#include "rows.cuh"

namespace crf {

namespace {

constexpr int kSlice = 256;              // columns of one row per block
constexpr int kRowThreads = kSlice + 32;  // and a warp for the down products

__device__ __forceinline__ float block_sum(float v, float* red) {
  v = warp_sum(v);
  if ((threadIdx.x & 31) == 0 && threadIdx.x < kSlice) red[threadIdx.x >> 5] = v;
  __syncthreads();
  float t = 0.f;
#pragma unroll
  for (int w = 0; w < kSlice / 32; ++w) t += red[w];
  return t;
}

// The block's extra warp: the scaled down products of row r for one or two modules (16 lanes
// each), while the other warps add up their columns.
__device__ __forceinline__ void load_xa(const RowPart& part, int r, const RowUp& u0, const RowUp* u1,
                                        const RowLora& lora, float (*xa)[kRankPad]) {
  const int m = (threadIdx.x & 31) >> 4, k = threadIdx.x & 15;
  if (m < (u1 ? 2 : 1)) {
    const RowUp& u = m == 0 ? u0 : *u1;
    xa[m][k] = u.B && k < lora.rank ? part_sum(part, r, u.xa_col + k) * lora.scale : 0.f;
  }
}

template <int kTerms>
__global__ void __launch_bounds__(kRowThreads) add_norm_rows_kernel(float* __restrict__ x, int dim, const RowPart part,
                                                               const RowUp up, const RowLora lora, int up_rows,
                                                               const __grid_constant__ RowStart start,
                                                               const __nv_bfloat16* __restrict__ g,
                                                               __nv_bfloat16* __restrict__ xs, float* __restrict__ nss,
                                                               int slices, int* status) {
  __shared__ float red[kSlice / 32];
  __shared__ float xa[1][kRankPad];
  griddep_launch_dependents();
  const int r = blockIdx.x / slices, sl = blockIdx.x % slices;
  const bool col = threadIdx.x < kSlice;
  const int j = sl * kSlice + threadIdx.x;
  const bool in = col && j < dim, add = r < up_rows;
  const UpRow b = up_row(add ? up.B : nullptr, in ? j : 0, lora.rank);
  const float gv = in ? __bfloat162float(g[j]) : 0.f;
  griddep_wait();
  float v = 0.f;
  if (add) {
    if (in)
      v = x[static_cast<size_t>(r) * dim + j] + part_sum(part, r, j);
    else if (!col)
      load_xa(part, r, up, nullptr, lora, xa);
    __syncthreads();
    if (in && up.B) v += up_dot(b, xa[0]);
  } else {
    const __nv_bfloat16* row = start.row[r];
    if (start.token[r])
      row = start.embed + static_cast<size_t>(checked_token(*start.token[r], start.vocab,
                                                            sl == 0 && threadIdx.x == 0 ? status : nullptr)) * dim;
    if (in) v = __bfloat162float(row[j]);
  }
  if (in) {
    x[static_cast<size_t>(r) * dim + j] = v;
    store_terms<kTerms>(xs + static_cast<size_t>(r) * kTerms * dim + j, dim, v * gv);
  }
  const float ss = block_sum(v * v, red);
  if (threadIdx.x == 0) nss[r * slices + sl] = ss;
}

__global__ void __launch_bounds__(kRowThreads) finish_rows_kernel(const float* __restrict__ x, int dim, const RowPart part,
                                                             const RowUp up, const RowLora lora,
                                                             const __grid_constant__ RowOuts outs, int slices,
                                                             const int* abort) {
  __shared__ float xa[1][kRankPad];
  griddep_launch_dependents();
  const int r = blockIdx.x / slices;
  const bool col = threadIdx.x < kSlice;
  const int j = (blockIdx.x % slices) * kSlice + threadIdx.x;
  const bool in = col && j < dim;
  const UpRow b = up_row(up.B, in ? j : 0, lora.rank);
  griddep_wait();
  if (call_aborted(abort) || !outs.out[r]) return;
  float v = 0.f;
  if (in)
    v = x[static_cast<size_t>(r) * dim + j] + part_sum(part, r, j);
  else if (!col)
    load_xa(part, r, up, nullptr, lora, xa);
  __syncthreads();
  if (in && up.B) v += up_dot(b, xa[0]);
  if (in) outs.out[r][j] = __float2bfloat16_rn(v);
}

// kRows rows per block: each B row is read once for them, and their columns' loads are in flight
// together. One row a block leaves 32 rows of the 7B shape in four waves of blocks (11.9 us, 4 rows a
// block: one wave).
template <int kTerms, int kRows>
__global__ void __launch_bounds__(kRowThreads) swiglu_rows_kernel(const RowPart part, int up_col, int f, const RowUp up_g,
                                                                  const RowUp up_u, const RowLora lora,
                                                                  __nv_bfloat16* __restrict__ ms, int slices) {
  __shared__ float xa[kRows][2][kRankPad];
  griddep_launch_dependents();
  const int r0 = blockIdx.x / slices * kRows;
  const int j = (blockIdx.x % slices) * kSlice + threadIdx.x;
  const bool col = threadIdx.x < kSlice;
  const bool in = col && j < f;
  const UpRow bg = up_row(up_g.B, in ? j : 0, lora.rank), bu = up_row(up_u.B, in ? j : 0, lora.rank);
  griddep_wait();
  float g[kRows], u[kRows];
#pragma unroll
  for (int i = 0; i < kRows; ++i) {
    g[i] = u[i] = 0.f;
    if (r0 + i < part.rows) {
      if (in) {
        g[i] = part_sum(part, r0 + i, j);
        u[i] = part_sum(part, r0 + i, up_col + j);
      } else if (!col) {
        load_xa(part, r0 + i, up_g, &up_u, lora, xa[i]);
      }
    }
  }
  __syncthreads();
  if (!in) return;
#pragma unroll
  for (int i = 0; i < kRows; ++i) {
    if (r0 + i >= part.rows) break;
    if (up_g.B) g[i] += up_dot(bg, xa[i][0]);
    if (up_u.B) u[i] += up_dot(bu, xa[i][1]);
    store_terms<kTerms>(ms + static_cast<size_t>(r0 + i) * kTerms * f + j, f, g[i] / (1.f + __expf(-g[i])) * u[i]);
  }
}

template <int kTerms>
__global__ void __launch_bounds__(kSlice) head_rows_kernel(const __nv_bfloat16* __restrict__ ref,
                                                           const __nv_bfloat16* __restrict__ cur, int n_ref, int dim,
                                                           const __nv_bfloat16* __restrict__ g,
                                                           __nv_bfloat16* __restrict__ xs, float* __restrict__ nss,
                                                           int slices) {
  __shared__ float red[kSlice / 32];
  griddep_launch_dependents();
  griddep_wait();
  const int r = blockIdx.x / slices, sl = blockIdx.x % slices;
  const int j = sl * kSlice + threadIdx.x;
  const __nv_bfloat16* row = r < n_ref ? ref + static_cast<size_t>(r) * dim : cur + static_cast<size_t>(r - n_ref) * dim;
  float v = 0.f;
  if (j < dim) {
    v = __bfloat162float(row[j]);
    store_terms<kTerms>(xs + static_cast<size_t>(r) * kTerms * dim + j, dim, v * __bfloat162float(g[j]));
  }
  const float ss = block_sum(v * v, red);
  if (threadIdx.x == 0) nss[static_cast<size_t>(r) * slices + sl] = ss;
}

inline bool rank_ok(const RowLora& l) { return l.rank == 4 || l.rank == 8 || l.rank == 16; }

}  // namespace

int norm_slices(int dim) { return (dim + kSlice - 1) / kSlice; }

cudaError_t launch_add_norm_rows(float* x, int dim, int rows, const RowPart& part, const RowUp& up, const RowLora& lora,
                                 int up_rows, const RowStart* start, const __nv_bfloat16* g, __nv_bfloat16* xs,
                                 int terms, float* nss, int* status, cudaStream_t stream) {
  if (rows == 0) return cudaSuccess;
  if (!rank_ok(lora) || (up_rows < rows && !start)) return cudaErrorInvalidValue;
  RowStart s{};
  if (start) s = *start;
  const int slices = norm_slices(dim);
  auto kern = terms == 2 ? add_norm_rows_kernel<2> : add_norm_rows_kernel<3>;
  return launch_kernel(kern, dim3(rows * slices), dim3(kRowThreads), 0, stream, x, dim, part, up, lora, up_rows, s, g, xs, nss,
                       slices, status);
}

cudaError_t launch_finish_rows(const float* x, int dim, int rows, const RowPart& part, const RowUp& up,
                               const RowLora& lora, const RowOuts& outs, const int* abort, cudaStream_t stream) {
  if (rows == 0) return cudaSuccess;
  if (!rank_ok(lora)) return cudaErrorInvalidValue;
  const int slices = norm_slices(dim);
  return launch_kernel(finish_rows_kernel, dim3(rows * slices), dim3(kRowThreads), 0, stream, x, dim, part, up, lora, outs,
                       slices, abort);
}

cudaError_t launch_swiglu_rows(const RowPart& part, int up_col, int f, const RowUp& up_g, const RowUp& up_u,
                               const RowLora& lora, __nv_bfloat16* ms, int terms, cudaStream_t stream) {
  if (part.rows == 0) return cudaSuccess;
  if (!rank_ok(lora)) return cudaErrorInvalidValue;
  const int slices = norm_slices(f);
  auto launch = [&](auto kern, int rows) {
    return launch_kernel(kern, dim3((part.rows + rows - 1) / rows * slices), dim3(kRowThreads), 0, stream, part, up_col, f,
                         up_g, up_u, lora, ms, slices);
  };
  if (terms == 3) return launch(swiglu_rows_kernel<3, 1>, 1);
  return part.rows > 8 ? launch(swiglu_rows_kernel<2, 4>, 4) : launch(swiglu_rows_kernel<2, 1>, 1);
}

cudaError_t launch_head_rows(const __nv_bfloat16* ref, const __nv_bfloat16* cur, int n_ref, int hidden,
                             const __nv_bfloat16* g, __nv_bfloat16* xs, int terms, float* nss, cudaStream_t stream) {
  if (n_ref == 0) return cudaSuccess;
  const int slices = norm_slices(hidden);
  auto kern = terms == 2 ? head_rows_kernel<2> : head_rows_kernel<3>;
  return launch_kernel(kern, dim3(2 * n_ref * slices), dim3(kSlice), 0, stream, ref, cur, n_ref, hidden, g, xs, nss,
                       slices);
}

cudaError_t launch_lm_head(const __nv_bfloat16* W, const __nv_bfloat16* xs, int terms, const float* nss, int rows,
                           int vocab, int hidden, float eps, float* logits, int num_sms, int* status,
                           cudaStream_t stream, const int* abort) {
  const RowsPlan plan = rows_plan(1, &vocab, false, hidden, num_sms, /*split=*/false);
  const int slices = norm_slices(hidden);
  for (int r0 = 0; r0 < rows; r0 += kRowsMax) {
    RowsGemmDesc d{};
    d.W[0] = W;
    d.out[0] = vocab;
    d.nseg = 1;
    d.in_dim = hidden;
    d.x = xs + static_cast<size_t>(r0) * terms * hidden;
    d.rows = rows - r0 < kRowsMax ? rows - r0 : kRowsMax;
    d.terms = terms;
    d.y = logits + static_cast<size_t>(r0) * vocab;
    d.ncols = vocab;
    d.nss = nss + static_cast<size_t>(r0) * slices;
    d.slices = slices;
    d.eps = eps;
    d.status = status;
    d.abort = abort;
    d.alone = true;
    cudaError_t e = launch_rows_gemm(d, plan, num_sms, stream);
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

}  // namespace crf
