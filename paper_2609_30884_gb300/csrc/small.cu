// Memory-bound kernels: RMSNorm, embedding gather, RoPE angle tables, the page-table check, the
// greedy token and the first-step KL reduction (Section S2.1).
#include "common.cuh"
#include "kernels.h"

#include <algorithm>
#include <cfloat>
#include <cmath>
#include <cstdlib>
#include <cstring>
#include <optional>
#include <type_traits>

namespace crf {

namespace {

// ------------------------------------------------------------------ opening a call
// (cos, sin)(p * theta^(-2i/d)): the angle in turns, p * theta^(-2i/d) / (2 pi), is formed in fp64
// (per-frequency factors computed on the host in fp64), reduced to [0, 1) and evaluated with fp32
// sincospi.
struct RopeJob {
  double turns_per_pos[64];
  float2* table;
  int n, half;       // entries of the table, pairs per position
  int by_row;        // table [rows][half] for position pos[row]; else the position-minor table
  RowPositions pos;
};

// Blocks [0, check_blocks): one thread per page id; an id outside [0, num_pages), or already in the
// open-addressing table (zeros: empty; linear probing, at most mask + 1 probes), rejects the call.
// The blocks after them: the call's rotation angles.
__global__ void open_call_kernel(const __grid_constant__ PageCheck pc, int num_pages, int* table, uint32_t mask,
                                 int* abort, int* status, int check_blocks, const __grid_constant__ RopeJob rope) {
  griddep_launch_dependents();
  griddep_wait();
  if (static_cast<int>(blockIdx.x) >= check_blocks) {
    const int idx = (blockIdx.x - check_blocks) * blockDim.x + threadIdx.x;
    if (idx >= rope.n) return;
    int p, i;
    if (rope.by_row) {
      p = rope.pos.pos[idx / rope.half];
      i = idx % rope.half;
    } else {
      const int n_pos = rope.n / rope.half;
      p = idx / 2 % n_pos;
      i = idx / 2 / n_pos * 2 + idx % 2;
    }
    double turns = static_cast<double>(p) * rope.turns_per_pos[i];
    turns -= floor(turns);
    float s, c;
    sincospif(static_cast<float>(2.0 * turns), &s, &c);
    rope.table[idx] = make_float2(c, s);
    return;
  }
  const int idx = blockIdx.x * blockDim.x + threadIdx.x;
  if (idx >= pc.first[pc.n]) return;
  int i = 0;
  while (i + 1 < pc.n && idx >= pc.first[i + 1]) ++i;
  const int id = pc.pt[i][idx - pc.first[i]];
  bool bad = id < 0 || id >= num_pages;
  if (!bad) {
    uint32_t h = (static_cast<uint32_t>(id) * 0x9E3779B1u) & mask;
    for (uint32_t probe = 0; probe <= mask; ++probe) {
      const int prev = atomicCAS(table + h, 0, id + 1);
      if (prev == 0) break;
      if (prev == id + 1) {
        bad = true;
        break;
      }
      h = (h + 1) & mask;
    }
  }
  if (bad) {
    atomicExch(abort, 1);
    atomicOr(status, kStatusPages);
  }
}

// ------------------------------------------------------------------ RMSNorm (+ BX rows)
// One 16-byte chunk (8 columns) of a BX row per thread: the module's B row (rank values, zero
// padded to 16) at columns col_off .. col_off + 15 and again at col_off + 16 .. col_off + 31.
__device__ __forceinline__ void bext_chunk(const BextDesc& d, long idx) {
  int m = 0;
  long base = 0;
  while (m < d.n && idx >= base + static_cast<long>(d.rows[m]) * (kBxCols / 8)) {
    base += static_cast<long>(d.rows[m]) * (kBxCols / 8);
    ++m;
  }
  if (m >= d.n) return;
  const long k = idx - base;
  const int r = static_cast<int>(k / (kBxCols / 8));
  const int c0 = static_cast<int>(k % (kBxCols / 8)) * 8;
  const __nv_bfloat16* B = d.B[m];
  uint32_t w[4];
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    float v[2];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int c = c0 + 2 * j + h - d.col_off[m];
      const int q = c & 15;
      v[h] = (B && c >= 0 && c < 32 && q < d.rank) ? __bfloat162float(B[(size_t)r * d.rank + q]) : 0.f;
    }
    w[j] = pack_bf16(v[0], v[1]);
  }
  *reinterpret_cast<uint4*>(d.out[m] + (size_t)r * kBxCols + c0) = make_uint4(w[0], w[1], w[2], w[3]);
}

// Blocks [0, norm_blocks): one warp per row, y = x * rsqrt(mean(x^2) + eps) * g, fp32 math, bf16
// out. The row stays in registers (kVecs 16-byte pieces a lane, all loads in flight at once; 0: a
// row too wide for that is read twice). The blocks after them: the BX rows of `bx`, one chunk per
// thread.
// Bound by the trip of its loads in short calls: timed alone the register form is no faster (2003 rows
// of 1536: 8.7 us, 8.2 reading twice), but within a chain of launches prefill of 2003 tokens takes
// 1.49 ms, 1.57 reading twice.
template <int kVecs>
__global__ void rmsnorm_kernel(const __nv_bfloat16* __restrict__ x,
                               const __nv_bfloat16* __restrict__ g, __nv_bfloat16* __restrict__ y,
                               int rows, int hidden, float eps, const __grid_constant__ BextDesc bx,
                               int norm_blocks) {
  griddep_launch_dependents();
  griddep_wait();  // x comes from the kernel before, and earlier ones read y and the BX rows
  if (static_cast<int>(blockIdx.x) >= norm_blocks) {
    bext_chunk(bx, static_cast<long>(blockIdx.x - norm_blocks) * blockDim.x + threadIdx.x);
    return;
  }
  const int warp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int lane = threadIdx.x & 31;
  if (warp >= rows) return;
  const uint4* xr = reinterpret_cast<const uint4*>(x + (size_t)warp * hidden);
  const uint4* gr = reinterpret_cast<const uint4*>(g);
  uint4* yr = reinterpret_cast<uint4*>(y + (size_t)warp * hidden);
  const int nv = hidden / 8;
  float ss = 0.f;
  auto square = [&](const uint4& u) {
    const uint32_t w[4] = {u.x, u.y, u.z, u.w};
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const float a = bf16_lo(w[j]), b = bf16_hi(w[j]);
      ss += a * a + b * b;
    }
  };
  auto scale = [&](int i, const uint4& u, const uint4& gv, float inv) {
    const uint32_t w[4] = {u.x, u.y, u.z, u.w};
    const uint32_t gw[4] = {gv.x, gv.y, gv.z, gv.w};
    uint32_t o[4];
#pragma unroll
    for (int j = 0; j < 4; ++j)
      o[j] = pack_bf16(bf16_lo(w[j]) * inv * bf16_lo(gw[j]), bf16_hi(w[j]) * inv * bf16_hi(gw[j]));
    yr[i] = make_uint4(o[0], o[1], o[2], o[3]);
  };
  if constexpr (kVecs > 0) {
    uint4 u[kVecs];
#pragma unroll
    for (int k = 0; k < kVecs; ++k) {
      const int i = lane + 32 * k;
      u[k] = i < nv ? xr[i] : make_uint4(0, 0, 0, 0);
    }
#pragma unroll
    for (int k = 0; k < kVecs; ++k) square(u[k]);
    const float inv = rsqrtf(warp_sum(ss) / hidden + eps);
#pragma unroll
    for (int k = 0; k < kVecs; ++k) {
      const int i = lane + 32 * k;
      if (i < nv) scale(i, u[k], gr[i], inv);
    }
  } else {
    for (int i = lane; i < nv; i += 32) square(xr[i]);
    const float inv = rsqrtf(warp_sum(ss) / hidden + eps);
    for (int i = lane; i < nv; i += 32) scale(i, xr[i], gr[i], inv);
  }
}

// ------------------------------------------------------------------ embedding
__global__ void embed_kernel(const __nv_bfloat16* __restrict__ e, const int32_t* __restrict__ tok,
                             __nv_bfloat16* __restrict__ out, int n, int hidden, int vocab,
                             int* status) {
  const int nv = hidden / 8;
  const size_t idx = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (idx >= (size_t)n * nv) return;
  const int t = static_cast<int>(idx / nv), c = static_cast<int>(idx % nv);
  // Only the row's first chunk reports a bad id, so the status word sees one atomic per row.
  const int id = checked_token(tok[t], vocab, c == 0 ? status : nullptr);
  reinterpret_cast<uint4*>(out + (size_t)t * hidden)[c] =
      reinterpret_cast<const uint4*>(e + (size_t)id * hidden)[c];
}

// One T per thread and turn: 16 bytes, or 2 where a caller's row is not aligned to 16.
template <typename T>
__global__ void copy_rows_kernel(T* __restrict__ dst, const T* __restrict__ src, size_t n, const int* abort) {
  griddep_launch_dependents();
  griddep_wait();
  if (call_aborted(abort)) return;
  for (size_t i = blockIdx.x * static_cast<size_t>(blockDim.x) + threadIdx.x; i < n;
       i += static_cast<size_t>(gridDim.x) * blockDim.x)
    dst[i] = src[i];
}

// ------------------------------------------------------------------ KL
// Per (row, split): online (max, sum e^(z* - m), sum e^(z* - m)(z* - z)) for the
// reference and (max, sum e^(z - m)) for the current logits.
constexpr int kKlThreads = 256;
constexpr int kKlAhead = 8;

__global__ void __launch_bounds__(kKlThreads) kl_partial_kernel(const float* __restrict__ zr,
                                                                const float* __restrict__ zc,
                                                                int vocab, int splits,
                                                                float* __restrict__ part) {
  griddep_launch_dependents();
  griddep_wait();
  const int row = blockIdx.y, sp = blockIdx.x;
  const int per = (vocab + splits - 1) / splits;
  const int v0 = sp * per, v1 = min(vocab, v0 + per);
  const float* a = zr + (size_t)row * vocab;
  const float* b = zc + (size_t)row * vocab;
  float mr = -FLT_MAX, sr = 0.f, dr = 0.f, mc = -FLT_MAX, sc = 0.f;
  // the logits of eight turns in flight together, then added in order: one row pair has about two
  // turns a thread, 29 have 54, which took a memory latency each
  for (int i0 = v0 + threadIdx.x; i0 < v1; i0 += kKlAhead * kKlThreads) {
    float xs[kKlAhead], ys[kKlAhead];
#pragma unroll
    for (int u = 0; u < kKlAhead; ++u) {
      const int i = i0 + u * kKlThreads;
      xs[u] = i < v1 ? a[i] : 0.f;
      ys[u] = i < v1 ? b[i] : 0.f;
    }
#pragma unroll
    for (int u = 0; u < kKlAhead; ++u) {
      if (i0 + u * kKlThreads >= v1) break;
      const float x = xs[u], y = ys[u];
      if (x > mr) {
        const float f = __expf(mr - x);
        sr *= f;
        dr *= f;
        mr = x;
      }
      const float e = __expf(x - mr);
      sr += e;
      dr += e * (x - y);
      if (y > mc) {
        sc *= __expf(mc - y);
        mc = y;
      }
      sc += __expf(y - mc);
    }
  }
  // block combine
  __shared__ float s_mr[kKlThreads], s_sr[kKlThreads], s_dr[kKlThreads], s_mc[kKlThreads],
      s_sc[kKlThreads];
  s_mr[threadIdx.x] = mr;
  s_sr[threadIdx.x] = sr;
  s_dr[threadIdx.x] = dr;
  s_mc[threadIdx.x] = mc;
  s_sc[threadIdx.x] = sc;
  __syncthreads();
  for (int off = kKlThreads / 2; off > 0; off >>= 1) {
    if (threadIdx.x < off) {
      const int o = threadIdx.x + off;
      const float M = fmaxf(s_mr[threadIdx.x], s_mr[o]);
      const float f1 = s_mr[threadIdx.x] == -FLT_MAX ? 0.f : __expf(s_mr[threadIdx.x] - M);
      const float f2 = s_mr[o] == -FLT_MAX ? 0.f : __expf(s_mr[o] - M);
      s_sr[threadIdx.x] = s_sr[threadIdx.x] * f1 + s_sr[o] * f2;
      s_dr[threadIdx.x] = s_dr[threadIdx.x] * f1 + s_dr[o] * f2;
      s_mr[threadIdx.x] = M;
      const float Mc = fmaxf(s_mc[threadIdx.x], s_mc[o]);
      const float g1 = s_mc[threadIdx.x] == -FLT_MAX ? 0.f : __expf(s_mc[threadIdx.x] - Mc);
      const float g2 = s_mc[o] == -FLT_MAX ? 0.f : __expf(s_mc[o] - Mc);
      s_sc[threadIdx.x] = s_sc[threadIdx.x] * g1 + s_sc[o] * g2;
      s_mc[threadIdx.x] = Mc;
    }
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    float* p = part + ((size_t)row * splits + sp) * 5;
    p[0] = s_mr[0];
    p[1] = s_sr[0];
    p[2] = s_dr[0];
    p[3] = s_mc[0];
    p[4] = s_sc[0];
  }
}

// KL = D/S* + (M + log S) - (M* + log S*), combining the splits of one row (warp per row).
__global__ void kl_final_kernel(const float* part, int splits, float* out, int rows) {
  griddep_launch_dependents();
  griddep_wait();
  const int row = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int lane = threadIdx.x & 31;
  if (row >= rows) return;
  const float* p = part + (size_t)row * splits * 5;
  float Mr = -FLT_MAX, Mc = -FLT_MAX;
  for (int s = lane; s < splits; s += 32) {
    Mr = fmaxf(Mr, p[s * 5 + 0]);
    Mc = fmaxf(Mc, p[s * 5 + 3]);
  }
  Mr = warp_max(Mr);
  Mc = warp_max(Mc);
  float Sr = 0.f, Dr = 0.f, Sc = 0.f;
  for (int s = lane; s < splits; s += 32) {
    const float fr = p[s * 5 + 0] == -FLT_MAX ? 0.f : __expf(p[s * 5 + 0] - Mr);
    Sr += fr * p[s * 5 + 1];
    Dr += fr * p[s * 5 + 2];
    Sc += (p[s * 5 + 3] == -FLT_MAX ? 0.f : __expf(p[s * 5 + 3] - Mc)) * p[s * 5 + 4];
  }
  Sr = warp_sum(Sr);
  Dr = warp_sum(Dr);
  Sc = warp_sum(Sc);
  if (lane == 0) out[row] = Dr / Sr + (Mc + logf(Sc)) - (Mr + logf(Sr));
}

inline int cdiv(long a, long b) { return static_cast<int>((a + b - 1) / b); }

}  // namespace

cudaError_t launch_open_call(const PageCheck& pc, int num_pages, int* table, uint32_t mask, int* abort, int* status,
                             bool check, float2* angles, int n_pos, const RowPositions* rows, int head_dim,
                             double theta, cudaStream_t stream) {
  const int ids = check ? pc.first[pc.n] : 0;
  if (static_cast<uint32_t>(ids) > (mask + 1u) / 2u) return cudaErrorInvalidValue;
  RopeJob r{};
  r.half = head_dim / 2;
  if (r.half > 64 || n_pos < 0 || static_cast<long>(n_pos) * r.half > 0x7fffffffl) return cudaErrorInvalidValue;
  r.table = angles;
  r.n = n_pos * r.half;
  r.by_row = rows != nullptr;
  if (rows) r.pos = *rows;
  for (int i = 0; i < r.half; ++i)
    r.turns_per_pos[i] = std::pow(theta, -2.0 * i / head_dim) / (2.0 * 3.14159265358979323846);
  const int check_blocks = cdiv(ids, 256), blocks = check_blocks + cdiv(r.n, 256);
  if (blocks == 0) return cudaSuccess;
  return launch_kernel(open_call_kernel, dim3(blocks), dim3(256), 0, stream, pc, num_pages, table, mask, abort, status,
                       check_blocks, r);
}

cudaError_t launch_rmsnorm(const __nv_bfloat16* x, const __nv_bfloat16* g, __nv_bfloat16* y,
                           int rows, int hidden, float eps, cudaStream_t stream, const BextDesc* bx) {
  BextDesc d{};
  long chunks = 0;
  if (bx) {
    d = *bx;
    if (d.n < 0 || d.n > 4 || d.rank < 1 || d.rank > kRankPad) return cudaErrorInvalidValue;
    for (int m = 0; m < d.n; ++m) chunks += static_cast<long>(d.rows[m]) * (kBxCols / 8);
  }
  const int norm_blocks = cdiv(rows, 8);
  const int blocks = norm_blocks + static_cast<int>(cdiv(chunks, 256));
  if (blocks == 0) return cudaSuccess;
  auto launch = [&](auto kern) {
    return launch_kernel(kern, dim3(blocks), dim3(256), 0, stream, x, g, y, rows, hidden, eps, d, norm_blocks);
  };
  // Up to 6 pieces a lane (1536 columns) the row fits in 69 registers. 14 pieces (3584) need 135, one
  // block an SM: 16384 rows take 61 us against 46 reading twice. Between them, 8 and 10 pieces (2048 and
  // 2560 columns): 16384 rows 31 and 35 us against 25 and 32, the window even; prefill of 2003 rows 2.11 and
  // 2.55 ms against 2.16 and 2.62, so with few rows the line could lie higher.
  const int vecs = (hidden / 8 + 31) / 32;  // 16-byte pieces a lane
  if (vecs <= 2) return launch(rmsnorm_kernel<2>);
  if (vecs <= 6) return launch(rmsnorm_kernel<6>);
  return launch(rmsnorm_kernel<0>);
}

cudaError_t launch_embed(const __nv_bfloat16* embed, const int32_t* tokens, __nv_bfloat16* out,
                         int n, int hidden, int vocab, int* status, cudaStream_t stream) {
  const long total = (long)n * (hidden / 8);
  if (total == 0) return cudaSuccess;
  embed_kernel<<<cdiv(total, 256), 256, 0, stream>>>(embed, tokens, out, n, hidden, vocab, status);
  return cudaGetLastError();
}

namespace {
thread_local bool t_pdl = false;
}  // namespace

PdlScope::PdlScope() : prev_(t_pdl) { t_pdl = true; }
PdlScope::~PdlScope() { t_pdl = prev_; }
bool pdl_active() { return t_pdl; }

// Bounded-wait self-test: thread 0 waits on an mbarrier that nothing arrives on. The wait
// gives up after the library's limit, raises the status bit and the kernel returns, so the
// context stays usable (the same path every kernel's waits take).
__global__ void wait_selftest_kernel(int* status) {
  __shared__ __align__(8) uint64_t bar;
  __shared__ volatile int abort_flag;
  if (threadIdx.x == 0) {
    mbar_init(&bar, 1);
    abort_flag = 0;
    fence_barrier_init();
  }
  __syncthreads();
  if (threadIdx.x == 0) (void)mbar_wait(&bar, 0, &abort_flag, status);
}

cudaError_t launch_wait_selftest(int* status, cudaStream_t stream) {
  wait_selftest_kernel<<<1, 32, 0, stream>>>(status);
  return cudaGetLastError();
}

// out[r] = argmax_i logits[r, i], the lowest index among equal maxima; NaNs never win. Each row is cut
// over gridDim.x blocks (one block a row pulled 608 KB through one SM, about 8 us). A logit and its
// index make one 64-bit key that orders by value, then by the lower index; the blocks of a row meet in
// an atomic maximum, which no order of arrival changes, and the last of them writes the token.
constexpr int kArgmaxThreads = 256;
constexpr int kArgmaxAhead = 8;
__global__ void __launch_bounds__(kArgmaxThreads) argmax_rows_kernel(const float* __restrict__ logits, int vocab,
                                                                     unsigned long long* key, int* count, int32_t* out,
                                                                     const int* abort) {
  griddep_launch_dependents();
  griddep_wait();
  if (call_aborted(abort)) return;
  const int r = blockIdx.y;
  const float* z = logits + (size_t)r * vocab;
  const int per = (vocab + gridDim.x - 1) / gridDim.x;
  const int v0 = blockIdx.x * per, v1 = min(vocab, v0 + per);
  unsigned long long best = 0;
  for (int i0 = v0 + threadIdx.x; i0 < v1; i0 += kArgmaxAhead * kArgmaxThreads) {
    float v[kArgmaxAhead];
#pragma unroll
    for (int u = 0; u < kArgmaxAhead; ++u) {
      const int i = i0 + u * kArgmaxThreads;
      v[u] = i < v1 ? __ldg(z + i) : NAN;
    }
#pragma unroll
    for (int u = 0; u < kArgmaxAhead; ++u) {
      if (isnan(v[u])) continue;
      const uint32_t b = __float_as_uint(v[u] == 0.f ? 0.f : v[u]);  // both zeros are equal
      const uint32_t order = b >> 31 ? ~b : b | 0x80000000u;
      const unsigned long long k =
          static_cast<unsigned long long>(order) << 32 | ~static_cast<uint32_t>(i0 + u * kArgmaxThreads);
      if (k > best) best = k;
    }
  }
  __shared__ unsigned long long sb[kArgmaxThreads / 32];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const unsigned long long k = __shfl_xor_sync(0xffffffffu, best, o);
    if (k > best) best = k;
  }
  if ((threadIdx.x & 31) == 0) sb[threadIdx.x >> 5] = best;
  __syncthreads();
  if (threadIdx.x != 0) return;
#pragma unroll
  for (int w = 1; w < kArgmaxThreads / 32; ++w)
    if (sb[w] > best) best = sb[w];
  atomicMax(key + r, best);
  __threadfence();
  if (atomicAdd(count + r, 1) != static_cast<int>(gridDim.x) - 1) return;
  __threadfence();
  best = atomicMax(key + r, 0ull);
  out[r] = best == 0 ? 0x7fffffff : static_cast<int32_t>(~static_cast<uint32_t>(best));
}

cudaError_t launch_argmax_rows(const float* logits, int rows, int vocab, unsigned long long* key, int* count,
                               int32_t* out, int num_sms, cudaStream_t stream, const int* abort) {
  if (rows == 0) return cudaSuccess;
  // about two blocks per SM over all rows, at least 4096 logits each
  const int by_rows = std::max(1, 2 * num_sms / rows), by_vocab = (vocab + 4095) / 4096;
  return launch_kernel(argmax_rows_kernel, dim3(std::min(std::min(32, by_rows), by_vocab), rows), dim3(kArgmaxThreads), 0,
                       stream, logits, vocab, key, count, out, abort);
}

cudaError_t launch_copy_rows(__nv_bfloat16* dst, const __nv_bfloat16* src, size_t n, const int* abort,
                             cudaStream_t stream) {
  if (n == 0) return cudaSuccess;
  auto launch = [&](auto* d, const auto* f, size_t items) {
    const size_t want = (items + 255) / 256;
    return launch_kernel(copy_rows_kernel<std::remove_pointer_t<decltype(d)>>,
                         dim3(static_cast<unsigned>(want < 2048 ? want : 2048)), dim3(256), 0, stream, d, f, items, abort);
  };
  if (n % 8 == 0 && ((reinterpret_cast<uintptr_t>(dst) | reinterpret_cast<uintptr_t>(src)) & 15) == 0)
    return launch(reinterpret_cast<uint4*>(dst), reinterpret_cast<const uint4*>(src), n / 8);
  return launch(dst, src, n);
}

cudaError_t launch_kl(const float* zref, const float* zcur, int rows, int vocab, float* out,
                      float* part, int splits, int num_sms, cudaStream_t stream) {
  if (rows == 0) return cudaSuccess;
  // Launched early, one block per SM finds its SM free when the logits are done (one row pair, 7B: 168 ->
  // 162 us with the LM head); twice as many pile up on the first SMs with room and make the rest
  // wait (29 pairs, 1.5B: 103 -> 112 us), so those launch when the LM head has ended.
  std::optional<PdlScope> pdl;
  if (static_cast<long>(splits) * rows <= num_sms) pdl.emplace();
  const cudaError_t e =
      launch_kernel(kl_partial_kernel, dim3(splits, rows), dim3(kKlThreads), 0, stream, zref, zcur, vocab, splits, part);
  if (e != cudaSuccess) return e;
  return launch_kernel(kl_final_kernel, dim3(cdiv(rows, 8)), dim3(256), 0, stream, static_cast<const float*>(part),
                       splits, out, rows);
}

}  // namespace crf
