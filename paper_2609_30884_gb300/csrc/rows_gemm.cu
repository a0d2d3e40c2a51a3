// Weight passes of the decode rows (the first-step rows of a window, the rows of a generation
// step, the LM head): y[r, j] = sum_i W[j, i] x[r, i] for up to 64 fp32 rows x, every weight read
// once for all of them. Adapted projections of Eq. S3 for single rows (Section 3.1, Section S2.1).
//
// The work is bound by the weight bytes. tcgen05.mma takes the weights as the 128-row A operand,
// straight from the shared-memory ring that TMA fills, so no thread touches a weight. The rows are
// the B operand: each fp32 row enters as bf16 terms in rows of their own (kTerms per row, 2: about
// 16 mantissa bits, 3: the whole fp32 value), and the epilogue adds a row's term columns; products
// of bf16 values are exact in fp32, accumulation is fp32. The tensor core cuts its running
// sums off instead of rounding them, so a long sum drifts by half a unit a step: where the rows are
// exact (three terms: one or two rows), a unit's steps accumulate in groups of TMEM columns, and the
// rows, which fill at most 6 of an operand's 16 rows, change sides with every K block: an 8-row atom of
// zeros is the other half of the operand, reached through the descriptor's stride. So every block of a
// group has sums of its own, of four MMAs. (Boxes that start 8 rows early, zero-filled, did the same and
// took 2.5 us a pass more: 7B step of one row 3.30 ms, 3.03 so. An infinite weight makes its output NaN:
// infinity meets zeros.)
// Error of the logits against 64 bits, sums of 4 MMAs / of 32 to 60 / fp32 on CUDA cores: the LM head alone, one
// pair of rows, 7B 1.17e-7 / 4.48e-7 / 1.22e-7, 1.5B 1.01e-7 / 2.17e-7 / 1.10e-7; one layer and the head, one
// row, 7B 2.9e-7 / 1.2e-6 / 3.2e-7, 1.5B 2.5e-7 / 5.1e-7 / 2.6e-7.
// (Beyond 4096 columns a unit a sum holds up to eight: hidden 8192, ffn 28672, 3.4e-7 against 3.8e-7 on
// CUDA cores.)
//
// Units of work: (128-row weight tile, K split); a tile's `splits` units are spread over CTAs so
// that a narrow projection still fills the chip, and each writes its own partial sums
// [split][row][column]. The consumer of the output adds them in split order (part_sum), which it
// does while it adds the adapter's up product anyway: no reduction pass, no atomics. The adapter's
// A rows (up to three modules, 16 rows each) are one more tile of the pass, so the down products
// come out of it too. An RMSNorm's 1 / rms is a factor of the whole row: the rows enter as x * g
// and the epilogue multiplies by it (nss: the sums of squares by slice).
//
// One CTA per SM and dependent launch: the ring's first weights are requested before the wait for the
// kernel that makes x, so the copies run through the short kernels between two passes (a ring of 75
// KB for the short passes would fit beside decode attention's block and start earlier, but runs out
// sooner: 7B step of one row 3.08 against 3.01 ms, of 32 rows 4.64 against 4.37, before sums of four MMAs;
// asking L2 for more weights before the wait gained nothing). Weights are marked evict-first in L2, which keeps the
// rows' partial sums and the K/V pages there (3% of a 7B generation step).
//
// Measured alone and cold: LM head of the 7B shape, 2 rows, 1.09 GB in 164 us (6.6 TB/s); gate|up of one
// row, 272 MB in 46 us (5.9 TB/s; 56 us before); 58 rows of the 1.5B LM head 79 us in one pass (a pass
// for every 8 rows before: 779 us). Generation steps with all that this layout brought, CUDA-core and
// mma.sync passes of 8 rows before: 7B 1 row 4.06 -> 3.03 ms, 32 rows 18.2 -> 4.28 ms, 1.5B 8 rows 2.36 -> 1.35 ms.
#include "common.cuh"
#include "kernels.h"
#include "tma_map.h"

#include <algorithm>
#include <cstring>

namespace crf {

namespace {

constexpr int kTile = 128;
constexpr int kBlockK = 64;  // one 128-byte swizzled box; a step takes plan.sub of them side by side
constexpr int kExactGroups = 32;  // most accumulation groups of exact rows: all of TMEM
constexpr int kRgThreads = 192;  // producer, MMA and four epilogue warps
constexpr int kMaxStages = 12;
constexpr int kWBytes = kTile * kBlockK * 2;
constexpr int kAtom = 8 * kBlockK * 2;  // 8 operand rows; one of zeros on either side of the ring

struct RowsGemmArgs {
  CUtensorMap tmW[kRowsMaxSeg];
  CUtensorMap tmA[kRowsMaxSeg];  // LoRA A rows, box of 16
  CUtensorMap tmX;               // the rows' terms, box of 8 (exact rows) or n
  RowsPlan plan;
  int nseg, n_lora, units;
  int rows, n, stages, acc_cols, groups;
  uint32_t tmem_cols;
  float* y;
  const float* nss;
  int slices;
  float inv_dim, eps;
  int* status;
  const int* abort;
};

// The steps (K blocks) of this CTA's units, in order.
struct Steps {
  int u, tile, kb, end;
  __device__ __forceinline__ void at(const RowsGemmArgs& a, int unit) {
    u = unit;
    tile = unit / a.plan.splits;
    const int p = unit - tile * a.plan.splits;
    kb = p * a.plan.kb / a.plan.splits;
    end = (p + 1) * a.plan.kb / a.plan.splits;
  }
  __device__ __forceinline__ void next(const RowsGemmArgs& a) {
    if (++kb == end) at(a, u + gridDim.x);
  }
  __device__ __forceinline__ bool more(const RowsGemmArgs& a) const { return u < a.units; }
};

// s + e += x, the rounding error of s + x kept in e.
__device__ __forceinline__ void two_sum(float& s, float& e, float x) {
  const float t = __fadd_rn(s, x), b = __fsub_rn(t, s);
  e += __fadd_rn(__fsub_rn(s, __fsub_rn(t, b)), __fsub_rn(x, b));
  s = t;
}

// Groups of exact rows in the first of the two accumulators.
__device__ __forceinline__ int first_half(int groups) { return (groups + 1) / 2; }

// kExact: one or two rows in three terms (16 columns). A unit's steps fill both accumulators, half of
// its groups in each, so the epilogue reads the first while the second is multiplied. Else: two terms, and
// the accumulators take units in turn. kAlone: exact rows of a pass by itself (the LM head).
template <bool kExact, bool kAlone>
__global__ void __launch_bounds__(kRgThreads, 1) rows_gemm_kernel(const __grid_constant__ RowsGemmArgs a) {
  constexpr int kTerms = kExact ? 3 : 2;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* zero_lo = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) &
                                                ~static_cast<uintptr_t>(1023));
  uint8_t* smem = zero_lo + kAtom;  // the ring
  __shared__ __align__(8) uint64_t full[kMaxStages], empty[kMaxStages];
  __shared__ __align__(8) uint64_t tfull[2], tempty[2], drain_bar;
  __shared__ uint32_t tmem_base_sh;
  __shared__ float s_inv[kRowsMax];
  __shared__ volatile int abort_flag;

  griddep_launch_dependents();
  const int warp = __shfl_sync(0xffffffffu, threadIdx.x >> 5, 0), lane = threadIdx.x & 31;
  const int sub = a.plan.sub;
  const int x_bytes = kExact ? kAtom : a.n * kBlockK * 2;
  const int stage_bytes = sub * (kWBytes + x_bytes);
  uint8_t* zero_hi = smem + a.stages * stage_bytes;
  if (threadIdx.x == 0) {
    for (int i = 0; i < a.stages; ++i) {
      mbar_init(&full[i], 1);
      mbar_init(&empty[i], 1);
    }
    for (int i = 0; i < 2; ++i) {
      mbar_init(&tfull[i], 1);
      mbar_init(&tempty[i], 4);
    }
    mbar_init(&drain_bar, 1);
    abort_flag = 0;
    fence_barrier_init();
  }
  if (warp == 1) {
    tmem_alloc(&tmem_base_sh, a.tmem_cols);
    tmem_relinquish();
  }
  if (kExact && threadIdx.x < 2 * kAtom / 16) {
    uint8_t* z = threadIdx.x < kAtom / 16 ? zero_lo : zero_hi - kAtom;
    reinterpret_cast<uint4*>(z)[threadIdx.x] = make_uint4(0, 0, 0, 0);
    fence_proxy_async_smem();  // before the MMAs read them
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = tmem_base_sh;

  if (warp == 0) {
    // ---------------------------------------------------------------- producer
    // The whole warp runs the loop, one lane issues.
    const bool issuer = elect_one();
    const uint64_t once = l2_evict_first();
    auto load_w = [&](const Steps& s, int st) {
      uint8_t* dst = smem + st * stage_bytes;
      const bool lora = s.tile == a.plan.tile0[a.nseg];
      if (issuer)
        mbar_arrive_expect_tx(&full[st], sub * ((lora ? a.n_lora * 16 * kBlockK * 2 : kWBytes) + x_bytes));
      int seg = 0;
      while (seg + 1 < a.nseg && s.tile >= a.plan.tile0[seg + 1]) ++seg;
      for (int h = 0; h < sub; ++h, dst += kWBytes) {
        const int k = (s.kb * sub + h) * kBlockK;
        if (lora) {
          for (int i = 0; i < a.n_lora; ++i)
            if (issuer) tma_load_2d(dst + i * 16 * kBlockK * 2, &a.tmA[i], &full[st], k, 0);
        } else if (issuer) {
          tma_load_2d_hint(dst, &a.tmW[seg], &full[st], k, (s.tile - a.plan.tile0[seg]) * kTile, once);
        }
      }
    };
    auto load_x = [&](const Steps& s, int st) {
      for (int h = 0; h < sub; ++h)
        if (issuer)
          tma_load_2d(smem + st * stage_bytes + sub * kWBytes + h * x_bytes, &a.tmX, &full[st],
                      (s.kb * sub + h) * kBlockK, 0);
    };
    Steps w, x;
    w.at(a, blockIdx.x);
    x.at(a, blockIdx.x);
    // weights of the first stages before the wait, their rows after it
    int used = 0;  // stages filled so far
    for (; used < a.stages && w.more(a); ++used, w.next(a)) load_w(w, used);
    griddep_wait();
    asm volatile("fence.proxy.async.global;" ::: "memory");
    for (int i = 0; i < used; ++i, x.next(a)) load_x(x, i);
    bool ok = true;
    int st = 0;
    uint32_t ph = 1;
    for (; w.more(a); w.next(a)) {
      ok = mbar_wait_warp(&empty[st], ph ^ 1, &abort_flag, a.status);
      if (!ok) break;
      load_w(w, st);
      load_x(w, st);
      ++used;
      if (++st == a.stages) {
        st = 0;
        ph ^= 1;
      }
    }
    if (!ok) {
      // every copy issued lands before the CTA can exit: the last use of every stage
      volatile int never = 0;
      for (int i = 0; i < a.stages && i < used; ++i) {
        const int u = used - 1 - i;
        mbar_wait(&full[u % a.stages], static_cast<uint32_t>((u / a.stages) & 1), &never, nullptr);
      }
    }
  } else if (warp == 1) {
    // ---------------------------------------------------------------- MMA issuer
    // The whole warp runs the loop, one lane issues.
    const bool issuer = elect_one();
    const uint32_t idesc = idesc_bf16_f32(kTile, a.n);
    bool ok = true, issued = false;
    int st = 0, it = 0;
    uint32_t ph = 0;
    Steps s;
    for (s.at(a, blockIdx.x); ok && s.more(a); ++it) {
      int acc = kExact ? 0 : it & 1;
      const int turn = kExact ? it : it >> 1;
      if (!mbar_wait_warp(&tempty[acc], (turn & 1) ^ 1, &abort_flag, a.status)) {
        ok = false;
        break;
      }
      tc_fence_after();
      const int unit = s.u, len = s.end - s.kb;
      // accumulation group of step i: i * groups / len
      for (int i = 0, left = 0; s.u == unit; s.next(a), i += a.groups) {
        int group = kExact ? i / len : 0;
        const bool first = left != group + 1;
        left = group + 1;
        if (kExact && group >= first_half(a.groups)) {
          if (acc == 0) {
            if (issuer) mma_commit(&tfull[0]);
            if (!mbar_wait_warp(&tempty[1], (turn & 1) ^ 1, &abort_flag, a.status)) {
              ok = false;
              break;
            }
            tc_fence_after();
            acc = 1;
          }
          group -= first_half(a.groups);
        }
        const uint32_t d = tmem + acc * a.acc_cols + group * a.n;
        if (!mbar_wait_warp(&full[st], ph, &abort_flag, a.status)) {
          ok = false;
          break;
        }
        tc_fence_after();
        const uint32_t base = smem_u32(smem + st * stage_bytes);
        if (issuer) {
          for (int h = 0; h < sub; ++h) {
            const uint64_t wd = smem_desc(base + h * kWBytes, 16, 1024, kSwizzle128B);
            const uint32_t x = base + sub * kWBytes + h * x_bytes;
            uint64_t xd = smem_desc(x, 16, 1024, kSwizzle128B);
            if constexpr (kExact)  // the rows and 8 of zeros, or the other way round
              xd = ((s.kb * sub + h) & 1) == 0 ? smem_desc(x, 16, smem_u32(zero_hi) - x, kSwizzle128B)
                                               : smem_desc(smem_u32(zero_lo), 16, x - smem_u32(zero_lo), kSwizzle128B);
#pragma unroll
            for (int k = 0; k < kBlockK / 16; ++k)
              mma_bf16_ss(d, wd + 2 * k, xd + 2 * k, idesc, (!first || h > 0 || k > 0) ? 1u : 0u);
          }
          mma_commit(&empty[st]);
        }
        issued = true;
        if (++st == a.stages) {
          st = 0;
          ph ^= 1;
        }
      }
      if (ok && issuer) mma_commit(&tfull[acc]);
    }
    if (!ok && issued && issuer) {
      mma_commit(&drain_bar);
      volatile int never = 0;
      mbar_wait(&drain_bar, 0, &never, nullptr);
    }
  } else {
    // ---------------------------------------------------------------- epilogue (warps 2..5)
    griddep_wait();  // nss comes from the kernel before, and earlier kernels read y
    const int et = threadIdx.x - 64;
    if (et < a.rows) {
      float ss = 0.f;
      for (int i = 0; a.nss && i < a.slices; ++i) ss += __ldcg(a.nss + et * a.slices + i);
      s_inv[et] = a.nss ? rsqrtf(ss * a.inv_dim + a.eps) : 1.f;
    }
    const bool skip = call_aborted(a.abort);
    asm volatile("bar.sync 1, 128;" ::: "memory");
    const int quarter = warp & 3;
    const uint32_t lane_off = static_cast<uint32_t>(quarter * 32) << 16;
    int it = 0;
    bool ok = true;
    for (int u = blockIdx.x; ok && u < a.units; u += gridDim.x, ++it) {
      const int tile = u / a.plan.splits;
      const int col = tile * kTile + quarter * 32 + lane;
      float* y = a.y + static_cast<size_t>(u - tile * a.plan.splits) * a.rows * a.plan.ncols + col;
      const bool store = !skip && col < a.plan.ncols;
      auto put = [&](int c, const float (&v)[16]) {
#pragma unroll
        for (int i = 0; i < 16 / kTerms; ++i) {
          const int r = c / kTerms + i;
          float s = v[kTerms * i];
#pragma unroll
          for (int t = 1; t < kTerms; ++t) s += v[kTerms * i + t];
          if (store && r < a.rows) y[static_cast<size_t>(r) * a.plan.ncols] = s * s_inv[r];
        }
      };
      auto take = [&](int acc, int turn) {
        ok = __all_sync(0xffffffffu, mbar_wait(&tfull[acc], turn & 1, &abort_flag, a.status));
        tc_fence_after();
        return tmem + lane_off + acc * a.acc_cols;
      };
      auto release = [&](int acc) {
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(&tempty[acc]);
      };
      if constexpr (kExact) {
        // Four groups as a tree, the fours in order; in a pass by itself with the rounding errors of that sum
        // carried along (7B LM head's logits: 1.23e-7 without, 1.17e-7 with them).
        float v[16], e[16];
#pragma unroll
        for (int i = 0; i < 16; ++i) v[i] = e[i] = 0.f;
#pragma unroll 1
        for (int acc = 0; acc < 2; ++acc) {
          const int ng = acc == 0 ? first_half(a.groups) : a.groups - first_half(a.groups);
          if (ng == 0) break;
          const uint32_t t0 = take(acc, it);
          if (!ok) break;
#pragma unroll 1
          for (int k = 0; k < ng; k += 4) {
            // groups past the last hold what an earlier launch left: read, not used
            uint32_t w[4][16];
#pragma unroll
            for (int q = 0; q < 4; ++q) tmem_ld16(t0 + (k + q) * 16, w[q]);
            tmem_ld_wait();
#pragma unroll
            for (int i = 0; i < 16; ++i) {
              const float g1 = k + 1 < ng ? __uint_as_float(w[1][i]) : 0.f;
              const float g2 = k + 2 < ng ? __uint_as_float(w[2][i]) : 0.f;
              const float g3 = k + 3 < ng ? __uint_as_float(w[3][i]) : 0.f;
              const float f = (__uint_as_float(w[0][i]) + g1) + (g2 + g3);
              if constexpr (kAlone)
                two_sum(v[i], e[i], f);
              else
                v[i] += f;
            }
          }
          release(acc);
        }
        if (!ok) break;
        if constexpr (kAlone) {
#pragma unroll
          for (int i = 0; i < 16; ++i)
            if (isfinite(v[i])) v[i] += e[i];  // a sum that is not finite has no error term
        }
#pragma unroll
        for (int i = 0; i < 8; ++i) v[i] += v[8 + i];
        put(0, v);
      } else {
        const uint32_t t0 = take(it & 1, it >> 1);
        if (!ok) break;
        for (int c = 0; c < a.n; c += 16) {
          uint32_t w[16];
          tmem_ld16(t0 + c, w);
          tmem_ld_wait();
          float v[16];
#pragma unroll
          for (int i = 0; i < 16; ++i) v[i] = __uint_as_float(w[i]);
          put(c, v);
        }
        release(it & 1);
      }
    }
  }

  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc(tmem, a.tmem_cols);
  }
}

template <bool kExact, bool kAlone>
cudaError_t launch_form(const RowsGemmArgs& a, int grid, int smem, cudaStream_t stream) {
  static PerDevice once;
  int dev = 0;
  if (once.pending(&dev)) {
    cudaError_t e = cudaFuncSetAttribute(rows_gemm_kernel<kExact, kAlone>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         kRowsRingMax + 2 * kAtom + 1024);
    if (e != cudaSuccess) return e;
    once.done(dev);
  }
  return launch_kernel(rows_gemm_kernel<kExact, kAlone>, dim3(grid), dim3(kRgThreads), smem, stream, a);
}

}  // namespace

RowsPlan rows_plan(int nseg, const int* outs, bool lora, int in_dim, int num_sms, bool split) {
  RowsPlan p;
  std::memset(&p, 0, sizeof(p));
  for (int s = 0; s < nseg; ++s) {
    p.tile0[s] = p.tiles;
    p.tiles += (outs[s] + kTile - 1) / kTile;
  }
  p.tile0[nseg] = p.tiles;
  if (lora) ++p.tiles;
  p.ncols = p.tiles * kTile;
  const int blocks = (in_dim + kBlockK - 1) / kBlockK;
  // From 8 blocks a CTA on, steps are two blocks (256 contiguous bytes of each weight row, asked for
  // together): the rate is then set by how DRAM pages are visited. 7B shape: one generation step 3.69
  // -> 3.21 ms, LM head 184 -> 166 us; four blocks gain nothing more. Below it, one-block steps split
  // evenly over more CTAs.
  const long per_cta = (static_cast<long>(p.tiles) * blocks + num_sms - 1) / num_sms;
  p.sub = per_cta >= 8 ? 2 : 1;
  p.kb = (blocks + p.sub - 1) / p.sub;
  // splits: the fewest K blocks on the busiest CTA, a unit's fixed cost counted as three blocks
  // and each split's share of the consumer's sum as a quarter
  p.splits = 1;
  double best = 0;
  for (int s = 1; s <= (split ? std::min(kRowsMaxSplits, p.kb) : 1); ++s) {
    const double waves = (static_cast<long>(p.tiles) * s + num_sms - 1) / num_sms;
    const double cost = waves * (p.sub * ((p.kb + s - 1) / s) + 3) + 0.25 * s;
    if (s == 1 || cost < best) {
      best = cost;
      p.splits = s;
    }
  }
  return p;
}

cudaError_t launch_rows_gemm(const RowsGemmDesc& d, const RowsPlan& plan, int num_sms, cudaStream_t stream) {
  RowsGemmArgs a;
  std::memset(&a, 0, sizeof(a));
  if (d.rows < 1 || d.rows > kRowsMax || d.nseg < 1 || d.nseg > kRowsMaxSeg || d.n_lora < 0 || d.n_lora > kRowsMaxSeg ||
      (d.terms != 2 && d.terms != 3) || (d.terms == 3 && d.rows > 2) || d.in_dim % 8 != 0)
    return cudaErrorInvalidValue;
  for (int s = 0; s < kRowsMaxSeg; ++s) {
    const int src = s < d.nseg ? s : 0;  // unused maps alias a valid one
    if (!tensor_map_rows(&a.tmW[s], d.W[src], d.out[src], d.in_dim, kTile)) return cudaErrorInvalidValue;
    if (s < d.n_lora) {
      if (!tensor_map_rows(&a.tmA[s], d.LA[s], d.rank, d.in_dim, 16)) return cudaErrorInvalidValue;
    } else {
      a.tmA[s] = a.tmW[0];
    }
  }
  a.n = (d.rows * d.terms + 15) / 16 * 16;
  const int x_rows = d.terms == 3 ? 8 : a.n;
  if (!tensor_map_rows(&a.tmX, d.x, static_cast<long>(d.rows) * d.terms, d.in_dim, x_rows)) return cudaErrorInvalidValue;
  a.plan = plan;
  if (d.ncols > 0) a.plan.ncols = d.ncols;
  a.nseg = d.nseg;
  a.n_lora = d.n_lora;
  a.units = plan.tiles * plan.splits;
  a.rows = d.rows;
  // exact rows: a group for every two blocks of the longest unit, at least one step each, at most what TMEM
  // holds; half of them make an accumulator
  const bool exact = d.terms == 3;
  const int longest = (plan.kb + plan.splits - 1) / plan.splits * plan.sub;
  a.groups = exact ? std::min({kExactGroups, plan.kb / plan.splits, (longest + 1) / 2}) : 1;
  a.acc_cols = exact ? 16 * kExactGroups / 2 : 16;
  while (a.acc_cols < a.n) a.acc_cols *= 2;
  a.tmem_cols = 2 * a.acc_cols;
  const int stage = plan.sub * (kWBytes + x_rows * kBlockK * 2);
  const int ring = d.alone ? kRowsRingMax : kRowsRing;
  a.stages = std::min(kMaxStages, ring / stage);
  a.y = d.y;
  a.nss = d.nss;
  a.slices = d.slices;
  a.inv_dim = 1.f / d.in_dim;
  a.eps = d.eps;
  a.status = d.status;
  a.abort = d.abort;
  const int grid = std::min(num_sms, a.units);
  if (grid < 1) return cudaSuccess;
  const int smem = a.stages * stage + 2 * kAtom + 1024;
  if (!exact) return launch_form<false, false>(a, grid, smem, stream);
  return d.alone ? launch_form<true, true>(a, grid, smem, stream) : launch_form<true, false>(a, grid, smem, stream);
}

}  // namespace crf
