// Persistent tcgen05 GEMM for sm_103a with the unmerged LoRA product and fused epilogues.
//
//   D[256 x BN] = A[256 x K] * B[BN x K]^T  (+ XA[256 x 64] * BL^T),  BN = 256, 192 or 128
//
// A cluster of two CTAs on one TPC works on a 256 x BN tile with cta_group::2 MMAs. Each CTA
// stages its own 128 rows of A and its own half of the B rows, so the operand bytes each SM
// pulls through L2 per FLOP are two thirds of the single-CTA 128 x 256 tile's. The even CTA
// issues the MMAs; both CTAs hold 128 accumulator lanes in their own TMEM and drain them through
// the same epilogue.
//
// Per CTA: warp 0 loads operands into a STAGES-deep shared-memory ring (TMA: the warp runs the
// loop on voted waits, which keeps its state in the uniform registers that TMA and MMA operands live
// in, and one elected lane issues), warp 1 owns TMEM (two accumulators, so the epilogue of tile i overlaps the main loop of tile
// i+1) and, in the MMA-issuing CTA, issues tcgen05.mma the same way; warps 2..5 drain the
// accumulator (one TMEM lane = one output row per thread) through the fused epilogue. Operands
// are bf16, K-major, staged with 128-byte swizzle; accumulation is fp32 in TMEM.
//
// The adapter term (alpha/r) (x A^T) B^T of every adapted projection (Eq. S3, W = W0 + (alpha/r)
// B A kept unmerged) is computed in the same launch:
//  - XA items come first in the order of work: one per row block, an MMA of N = 16 per module over
//    the x rows against the LoRA A rows, whose epilogue warps store the product, scaled, as a bf16
//    pair [hi | lo] per module (16 + 16 columns of the XA buffer) and count themselves into the row
//    block's ready word;
//  - every output tile of an adapted module adds one 64-wide K block: A side = the XA columns of
//    its row block (copied once the ready word shows all its warps), B side = BX, the module's B
//    rows twice over ([B | B], against [hi | lo]) under the K steps of its slot and zeros under the
//    other slot, so one K block serves two stacked modules and the two halves of a pair alike. The
//    RMSNorm launch before the layer's projections builds the BX rows.
// An item takes about as long as a tile's main loop and starts with the first wave, so that wave
// hardly waits. Formed by each row block's first tile, in the other accumulator, the product took
// that tile 1.4 to 1.8 times a plain one's time and every other tile of the first wave waited for it
// (1.5B shape, 2003 rows: 7 of the 28 us of q|k|v, 19 of the 77 us of down). Items over a quarter of K
// each were slower: their sums met through memory.
//
// Measured (us a launch; first column: the XA product in each row block's first tile, 256-column tiles,
// one row a thread in the epilogue; then: XA items, epilogue through shared memory, 128 columns; last:
// loops run by whole warps, for o and down 192 columns, and silu() for the divide of SwiGLU):
//   1.5B,  2003 rows: q|k|v  34,  28,  25   o  33,  24,  20   gate|up   99,   88,   73   down   84,   60,   45
//   1.5B,  4096 rows:        45,  39,  33      48,  35,  29            164,  150,  127         131,  108,   81
//   7B,   16384 rows:       370, 358, 311     282, 283, 252           2582, 2546, 2289        1288, 1356, 1249
// (the last row in a one-layer window; in longer runs the power cap adds 4-7%)
#include "common.cuh"
#include "kernels.h"
#include "tma_map.h"

#include <algorithm>
#include <cstring>

namespace crf {

namespace {

constexpr int BM = 128;
constexpr int BK = 64;
constexpr int kRasterGroup = 8;
constexpr int kThreads = 192;
constexpr int kXaGroups = 8;     // epilogue warps of a pair: each stores 32 of a row block's XA rows

struct GemmArgs {
  CUtensorMap tmA;
  CUtensorMap tmB[3];
  CUtensorMap tmXA;
  CUtensorMap tmLA[3];  // LoRA A of XA slot j: the B operand of the XA product
  CUtensorMap tmBX[3];  // BX rows of map index i: the B side of the LoRA K block
  int M, K, num_kb;
  int ngroups, nseg;
  int group_tiles[3];
  int group_cols[3];
  int ext_on[3];      // per group: tile has the LoRA K block
  int ext_steps[3];   // per group: K = 16 steps of that block that carry data
  int xa_base[3];     // per group: first XA column of that block
  int row_tiles, total_n;
  int n_slots;        // adapted modules (XA slots); 0: no XA product
  int xa_n;           // N of the XA product: 16 per slot, two CTA halves of 16 x slots_per_cta
  int xa_items;        // XA items (row_tiles or none), before the tiles in the order
  int total_items;     // XA items and tiles
  int rank;
  __nv_bfloat16* xa;
  int* xa_flags;
  int epi;
  float scale;
  __nv_bfloat16* out;
  int ldo;
  const __nv_bfloat16* resid;
  int ld_resid;
  const __nv_bfloat16* bias[3];
  const float2* rope;
  int rope_positions;
  int head_dim, n_kv_heads;
  __nv_bfloat16* qbuf;
  int ldq;
  __nv_bfloat16* kpages;
  __nv_bfloat16* vpages;
  ReqTable req;
  int* status;
  const int* abort;
};

struct Tile {
  int m_blk, g, n_loc;
  bool xa;  // an XA item
};

// XA items first, row block by row block; then the output tiles in bands of kRasterGroup column
// tiles over every row block (the band's B rows stay in L2).
__device__ __forceinline__ Tile decode_tile(int t, const GemmArgs& a) {
  Tile r;
  r.xa = t < a.xa_items;
  if (r.xa) {
    r.m_blk = t;
    r.g = r.n_loc = 0;
    return r;
  }
  t -= a.xa_items;
  const int band_tiles = a.row_tiles * kRasterGroup;
  const int band = t / band_tiles;
  const int idx = t - band * band_tiles;
  const int n0 = band * kRasterGroup;
  const int width = min(kRasterGroup, a.total_n - n0);
  r.m_blk = idx / width;
  int n = n0 + (idx - r.m_blk * width);
  int g = 0;
  while (g < a.ngroups - 1 && n >= a.group_tiles[g]) {
    n -= a.group_tiles[g];
    ++g;
  }
  r.g = g;
  r.n_loc = n;
  return r;
}

__device__ __forceinline__ void store16_bf16(__nv_bfloat16* dst, const float (&v)[16]) {
  uint4 w0, w1;
  w0.x = pack_bf16(v[0], v[1]);
  w0.y = pack_bf16(v[2], v[3]);
  w0.z = pack_bf16(v[4], v[5]);
  w0.w = pack_bf16(v[6], v[7]);
  w1.x = pack_bf16(v[8], v[9]);
  w1.y = pack_bf16(v[10], v[11]);
  w1.z = pack_bf16(v[12], v[13]);
  w1.w = pack_bf16(v[14], v[15]);
  reinterpret_cast<uint4*>(dst)[0] = w0;
  reinterpret_cast<uint4*>(dst)[1] = w1;
}

// Find the request and position of batched row `row`; returns false if none.
__device__ __forceinline__ bool row_lookup(const ReqTable& rt, int row, int& pos,
                                           const int32_t*& pt) {
  for (int i = 0; i < rt.n; ++i) {
    const int r0 = rt.row0[i];
    if (row >= r0 && row < r0 + rt.len[i]) {
      pos = row - r0;
      pt = rt.page_table[i];
      return true;
    }
  }
  return false;
}

// Epilogue rows move through shared memory, 32 rows x 64 columns of a warp at a time: a thread owns a
// row of the accumulator, but 32 threads on 32 rows of a matrix cost 32 wavefronts an access, eight
// threads on 128 contiguous bytes of a row cost one. Slot (row, 16-byte unit u) of a warp's 4 KB scratch
// is at row * 128 + ((u ^ (row & 7)) << 4): no bank conflicts either way.
constexpr int kScratchBytes = 4 * 4096;
__device__ __forceinline__ uint4* scratch_at(uint8_t* s, int row, int u) {
  return reinterpret_cast<uint4*>(s + row * 128 + ((u ^ (row & 7)) << 4));
}
// Rows' 64 columns from scratch to the rows' own destinations (`dst`: this lane's row, null: none);
// units from `units` on are outside the matrix.
__device__ __forceinline__ void scratch_store(uint8_t* s, int lane, __nv_bfloat16* dst, int units) {
  __syncwarp();
  const unsigned long long p = reinterpret_cast<unsigned long long>(dst);
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const int r = 4 * i + (lane >> 3), u = lane & 7;
    uint4* q = reinterpret_cast<uint4*>(__shfl_sync(0xffffffffu, p, r));
    const uint4 v = *scratch_at(s, r, u);
    if (q != nullptr && u < units) q[u] = v;
  }
  __syncwarp();
}

// One row's share of a tile, 64 accumulator columns at a time, so that their TMEM loads and the
// residual's or rotation table's are in flight together (16 at a time and straight to memory, the
// epilogue of a 256-column tile took 8-10 us). Twice the epilogue warps instead was slower: they
// compete with the producer and the MMA thread.
template <int BN, int EPI>
__device__ __forceinline__ void epilogue_tile(const GemmArgs& a, const Tile& tl, uint32_t tacc, int row, int lane,
                                              uint8_t* scr) {
  const bool row_ok = row < a.M;

  if constexpr (EPI == kEpiResid) {
    const int col0 = tl.n_loc * BN;
    const int ncols = a.group_cols[tl.g];  // a multiple of 8
    __nv_bfloat16* out = row_ok ? a.out + (size_t)row * a.ldo : nullptr;
    const int row_w = row - lane;  // the warp's first row
#pragma unroll 1
    for (int c = 0; c < BN; c += 64) {
      const int col = col0 + c;
      uint32_t r[2][32];
      tmem_ld32(tacc + c, r[0]);
      tmem_ld32(tacc + c + 32, r[1]);
      const int units = (ncols - col) / 8;
      uint4 w[8];
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        const int rr = row_w + 4 * i + (lane >> 3), u = lane & 7;
        w[i] = rr < a.M && u < units
                   ? *(reinterpret_cast<const uint4*>(a.resid + (size_t)rr * a.ld_resid + col) + u)
                   : make_uint4(0, 0, 0, 0);
      }
#pragma unroll
      for (int i = 0; i < 8; ++i) *scratch_at(scr, 4 * i + (lane >> 3), lane & 7) = w[i];
      __syncwarp();
      tmem_ld_wait();
#pragma unroll
      for (int k = 0; k < 8; ++k) {
        const uint4 x = *scratch_at(scr, lane, k);
        const uint32_t u[4] = {x.x, x.y, x.z, x.w};
        uint32_t p[4];
#pragma unroll
        for (int e = 0; e < 4; ++e)
          p[e] = pack_bf16(bf16_lo(u[e]) + __uint_as_float(r[k >> 2][(8 * k + 2 * e) & 31]),
                           bf16_hi(u[e]) + __uint_as_float(r[k >> 2][(8 * k + 2 * e + 1) & 31]));
        *scratch_at(scr, lane, k) = make_uint4(p[0], p[1], p[2], p[3]);
      }
      scratch_store(scr, lane, out ? out + col : nullptr, units);
    }
    return;
  }

  if constexpr (EPI == kEpiSwiGLU) {
    constexpr int HALF = BN / 2;
    const int f0 = tl.n_loc * HALF;
    const int ffn = a.group_cols[0];  // a multiple of 8
#pragma unroll 1
    for (int c = 0; c < HALF; c += 64) {
#pragma unroll 1
      for (int h2 = 0; h2 < 64; h2 += 32) {
        uint32_t gt[32], up[32];
        tmem_ld32(tacc + c + h2, gt);
        tmem_ld32(tacc + HALF + c + h2, up);
        tmem_ld_wait();
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          uint32_t p[4];
#pragma unroll
          for (int e = 0; e < 4; ++e) {
            float v[2];
#pragma unroll
            for (int h = 0; h < 2; ++h)
              v[h] = silu(__uint_as_float(gt[8 * k + 2 * e + h])) * __uint_as_float(up[8 * k + 2 * e + h]);
            p[e] = pack_bf16(v[0], v[1]);
          }
          *scratch_at(scr, lane, h2 / 8 + k) = make_uint4(p[0], p[1], p[2], p[3]);
        }
      }
      scratch_store(scr, lane, row_ok ? a.out + (size_t)row * a.ldo + f0 + c : nullptr, (ffn - f0 - c) / 8);
    }
    return;
  }

  if constexpr (EPI == kEpiQkv) {
    // kEpiQkv: group 0 = q, 1 = k, 2 = v; tiles are head-aligned (BN % head_dim == 0). Per head 32
    // rotation pairs at a time: 32 columns from its first half and 32 from its second.
    const int d = a.head_dim;
    const int half = d >> 1;
    int pos = 0;
    const int32_t* pt = nullptr;
    const bool have = row_ok && row_lookup(a.req, row, pos, pt);
    const int g = tl.g;
    const __nv_bfloat16* bias = a.bias[g];
    __nv_bfloat16* dst_row = nullptr;
    size_t head_stride = 0;
    if (have) {
      if (g == 0) {
        dst_row = a.qbuf + (size_t)row * a.ldq;
        head_stride = d;
      } else {
        const int page = checked_page(pt[pos / kPage], a.req.num_pages, a.status);
        __nv_bfloat16* base = (g == 1) ? a.kpages : a.vpages;
        dst_row = base + ((size_t)page * a.n_kv_heads * kPage + (pos % kPage)) * d;
        head_stride = (size_t)kPage * d;
      }
    }
    const bool rot = have && g < 2;
    const float4* rope4 = reinterpret_cast<const float4*>(a.rope) + pos;
#pragma unroll 1
    for (int i0 = 0; i0 < half; i0 += 32) {
      float4 cs[16];  // (cos, sin) of two pairs each: consecutive positions are neighbours
      if (rot) {
#pragma unroll
        for (int k = 0; k < 16; ++k) cs[k] = rope4[(size_t)(i0 / 2 + k) * a.rope_positions];
      }
#pragma unroll 1
      for (int hh = 0; hh < BN / d; ++hh) {
        const int head = (tl.n_loc * BN) / d + hh;
        const int gcol = head * d;
        if (gcol >= a.group_cols[g]) break;
        uint32_t r0[32], r1[32];
        tmem_ld32(tacc + hh * d + i0, r0);
        tmem_ld32(tacc + hh * d + half + i0, r1);
        tmem_ld_wait();
#pragma unroll
        for (int k = 0; k < 4; ++k) {  // 8 pairs
          float v[8], w[8];
#pragma unroll
          for (int j = 0; j < 8; ++j) {
            v[j] = __uint_as_float(r0[8 * k + j]);
            w[j] = __uint_as_float(r1[8 * k + j]);
          }
          if (bias) {
            const uint4 b0 = *reinterpret_cast<const uint4*>(bias + gcol + i0 + 8 * k);
            const uint4 b1 = *reinterpret_cast<const uint4*>(bias + gcol + half + i0 + 8 * k);
            const uint32_t u0[4] = {b0.x, b0.y, b0.z, b0.w}, u1[4] = {b1.x, b1.y, b1.z, b1.w};
#pragma unroll
            for (int j = 0; j < 4; ++j) {
              v[2 * j] += bf16_lo(u0[j]);
              v[2 * j + 1] += bf16_hi(u0[j]);
              w[2 * j] += bf16_lo(u1[j]);
              w[2 * j + 1] += bf16_hi(u1[j]);
            }
          }
          if (g < 2) {
#pragma unroll
            for (int j = 0; j < 8; ++j) {
              const float4 q = cs[4 * k + (j >> 1)];
              const float c = (j & 1) ? q.z : q.x, sn = (j & 1) ? q.w : q.y;
              const float x1 = v[j], x2 = w[j];
              v[j] = x1 * c - x2 * sn;
              w[j] = x2 * c + x1 * sn;
            }
          }
          *scratch_at(scr, lane, k) = make_uint4(pack_bf16(v[0], v[1]), pack_bf16(v[2], v[3]), pack_bf16(v[4], v[5]),
                                                 pack_bf16(v[6], v[7]));
          *scratch_at(scr, lane, 4 + k) = make_uint4(pack_bf16(w[0], w[1]), pack_bf16(w[2], w[3]),
                                                     pack_bf16(w[4], w[5]), pack_bf16(w[6], w[7]));
        }
        // units 0..3: pairs' first elements, units 4..7: the second ones, half a head further on
        __nv_bfloat16* dst = dst_row ? dst_row + head * head_stride + i0 : nullptr;
        __syncwarp();
        const unsigned long long p = reinterpret_cast<unsigned long long>(dst);
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          const int r = 4 * i + (lane >> 3), u = lane & 7;
          __nv_bfloat16* q = reinterpret_cast<__nv_bfloat16*>(__shfl_sync(0xffffffffu, p, r));
          const uint4 x = *scratch_at(scr, r, u);
          if (q != nullptr) *reinterpret_cast<uint4*>(q + (u & 3) * 8 + (u >= 4 ? half : 0)) = x;
        }
        __syncwarp();
      }
    }
  }
}

// Bounded wait until *flag >= target (acquire at GPU scope). Gives up like mbar_wait.
__device__ __forceinline__ bool flag_wait(const int* flag, int target, volatile int* abort_flag, int* status) {
  unsigned long long t0 = 0;
  for (uint32_t it = 0;; ++it) {
    int v;
    asm volatile("ld.acquire.gpu.global.b32 %0, [%1];" : "=r"(v) : "l"(flag) : "memory");
    if (v >= target) return true;
    if (*abort_flag) return false;
    if ((it & 15u) == 0) {
      const unsigned long long now = globaltimer_ns();
      if (t0 == 0) {
        t0 = now;
      } else if (now - t0 > kWaitLimitNs) {
        *abort_flag = 1;
        if (status) atomicOr(status, kStatusTimeout);
        return false;
      }
    }
    __nanosleep(128);
  }
}

__device__ __forceinline__ void fence_proxy_async_global() {
  asm volatile("fence.proxy.async.global;" ::: "memory");
}

// Stage layout: the A tile (this CTA's 128 rows x 64) and the B tile (its BN / 2 rows x 64; in an XA
// item the LoRA A rows of its half of the XA product, up to 32); 128-byte swizzle.
constexpr int kPair = 2;
constexpr int kABytes = BM * BK * 2;
template <int BN>
constexpr int kBBytes = BN / kPair * BK * 2;
template <int BN>
constexpr int kStageBytes = kABytes + kBBytes<BN>;

// Ring position (stage, phase) and whether every wait so far succeeded.
struct Ring {
  int stage;
  uint32_t phase;
  int ok;
  int used;  // stages the producer has filled so far
};

template <int STAGES>
__device__ __forceinline__ void ring_next(Ring& r) {
  if (++r.stage == STAGES) {
    r.stage = 0;
    r.phase ^= 1;
  }
}

// B rows of an output tile staged by CTA `rank`: its share of the tile (plain) or its segment of
// the stacked tile; with the map index of the first of them.
template <int BN>
__device__ __forceinline__ void tile_b_rows(const GemmArgs& a, const Tile& tl, uint32_t rank, int& g0, int& nb,
                                            int& yb, int& b_step) {
  const int nseg = a.nseg;
  const int seg_rows = BN / nseg;
  const int per = nseg / kPair;
  g0 = nseg == 1 ? tl.g : tl.g + static_cast<int>(rank) * per;
  nb = nseg == 1 ? 1 : per;
  yb = nseg == 1 ? tl.n_loc * BN + static_cast<int>(rank) * (BN / kPair) : tl.n_loc * seg_rows;
  b_step = nseg == 1 ? 0 : seg_rows * BK * 2;
}

// Copies of an XA item: per K block the row block's x rows and the LoRA A rows of this
// CTA's half of the XA product (16 rows per XA slot; CTA r takes slots [r * spc, r * spc + spc)).
template <int BN, int STAGES>
__device__ __forceinline__ Ring load_xa_item(const GemmArgs& a, int m0, uint32_t rank, bool leader, bool issuer,
                                             uint8_t* smem, uint64_t* full_bar, uint64_t* empty_bar,
                                             volatile int* abort_flag, Ring ring) {
  const int spc = a.xa_n / (16 * kPair);
  const int s0 = static_cast<int>(rank) * spc, s1 = min(a.n_slots, s0 + spc);
  const uint32_t bytes = kPair * kABytes + a.n_slots * 16 * BK * 2;
  for (int kb = 0; kb < a.num_kb; ++kb) {
    if (!mbar_wait_warp(&empty_bar[ring.stage], ring.phase ^ 1, abort_flag, a.status)) {
      ring.ok = 0;
      return ring;
    }
    uint8_t* sa = smem + ring.stage * kStageBytes<BN>;
    uint8_t* sl = sa + kABytes;
    if (issuer) {
      if (leader) mbar_arrive_expect_tx(&full_bar[ring.stage], bytes);
      const uint32_t bar = mapa_shared(&full_bar[ring.stage], 0);
      tma_load_2d_pair(sa, &a.tmA, bar, kb * BK, m0);
      for (int j = s0; j < s1; ++j) tma_load_2d_pair(sl + (j - s0) * 16 * BK * 2, &a.tmLA[j], bar, kb * BK, 0);
    }
    ++ring.used;
    ring_next<STAGES>(ring);
  }
  return ring;
}

// The LoRA stage of an output tile: once the stage is free, wait (unless seen already) until the row
// block's XA rows are stored, and copy those rows (the A side of the K block) and the tile's BX rows
// (the B side).
template <int BN, int STAGES>
__device__ __forceinline__ Ring load_lora_stage(const GemmArgs& a, const Tile& tl, int m0, uint32_t rank, bool xa_ready,
                                                bool leader, bool issuer, uint8_t* smem, uint64_t* full_bar,
                                                uint64_t* empty_bar, volatile int* abort_flag, Ring ring) {
  if (!mbar_wait_warp(&empty_bar[ring.stage], ring.phase ^ 1, abort_flag, a.status)) {
    ring.ok = 0;
    return ring;
  }
  if (!xa_ready && !__all_sync(0xffffffffu, flag_wait(a.xa_flags + tl.m_blk, kXaGroups, abort_flag, a.status))) {
    ring.ok = 0;
    return ring;
  }
  int g0, nb, yb, b_step;
  tile_b_rows<BN>(a, tl, rank, g0, nb, yb, b_step);
  uint8_t* sa = smem + ring.stage * kStageBytes<BN>;
  if (issuer) {
    fence_proxy_async_global();  // the TMA copy below reads what the XA items' stores wrote
    if (leader) mbar_arrive_expect_tx(&full_bar[ring.stage], kPair * kStageBytes<BN>);
    const uint32_t bar = mapa_shared(&full_bar[ring.stage], 0);
    tma_load_2d_pair(sa, &a.tmXA, bar, a.xa_base[tl.g], m0);
    for (int j = 0; j < nb; ++j) tma_load_2d_pair(sa + kABytes + j * b_step, &a.tmBX[g0 + j], bar, 0, yb);
  }
  ++ring.used;
  ring_next<STAGES>(ring);
  return ring;
}

// MMAs of an XA item into d_tmem's first xa_n columns. One this narrow still takes about 115 cycles (a
// full tile's 128), the latency of the sum it adds to; spread over two or four accumulators they took
// longer (1.5B down, 2003 rows: 60 -> 76 us).
template <int BN, int STAGES>
__device__ __forceinline__ Ring mma_xa_item(const GemmArgs& a, uint32_t d_tmem, uint32_t idesc_xa, bool issuer,
                                            uint8_t* smem, uint64_t* full_bar, uint64_t* empty_bar,
                                            volatile int* abort_flag, Ring ring) {
  for (int kb = 0; kb < a.num_kb; ++kb) {
    if (!mbar_wait_warp(&full_bar[ring.stage], ring.phase, abort_flag, a.status)) {
      ring.ok = 0;
      return ring;
    }
    tc_fence_after();
    const uint32_t sa = smem_u32(smem + ring.stage * kStageBytes<BN>);
    const uint64_t ad = smem_desc(sa, 16, 1024, kSwizzle128B);
    const uint64_t ld = smem_desc(sa + kABytes, 16, 1024, kSwizzle128B);
    if (issuer) {
#pragma unroll
      for (int k = 0; k < BK / 16; ++k)
        mma_bf16_ss_pair(d_tmem, ad + 2 * k, ld + 2 * k, idesc_xa, (kb > 0 || k > 0) ? 1u : 0u);
      mma_commit_pair(&empty_bar[ring.stage], 0x3);
    }
    ring_next<STAGES>(ring);
  }
  return ring;
}

// XA item, after its MMAs: slot j (columns 16j .. 16j + 15 of tacc) is x A_j^T for this thread's row.
// Scaled by alpha / r it is stored as hi = bf16(v) at XA columns 32j.. and lo = bf16(v - hi) at
// 32j + 16.. (the pair carries about 16 mantissa bits); then the warp counts into the ready word.
__device__ __noinline__ void drain_xa(const GemmArgs& a, int m_blk, uint32_t tacc, int row, int lane) {
  uint32_t r[3][16];
#pragma unroll
  for (int j = 0; j < 3; ++j)
    if (j < a.n_slots) tmem_ld16(tacc + 16 * j, r[j]);
  tmem_ld_wait();
#pragma unroll
  for (int j = 0; j < 3; ++j) {
    if (j >= a.n_slots || row >= a.M) continue;
    float v[16], w[16];
#pragma unroll
    for (int i = 0; i < 16; ++i) {
      v[i] = __uint_as_float(r[j][i]) * a.scale;
      w[i] = v[i] - __bfloat162float(__float2bfloat16_rn(v[i]));
    }
    store16_bf16(a.xa + (size_t)row * kXaCols + 32 * j, v);
    store16_bf16(a.xa + (size_t)row * kXaCols + 32 * j + 16, w);
  }
  // XA rows visible to the tiles' copies (global, GPU scope)
  __threadfence();
  fence_proxy_async_global();
  __syncwarp();
  if (lane == 0) atomicAdd(a.xa_flags + m_blk, 1);
}

template <int BN, int STAGES, int EPI>
__global__ void __launch_bounds__(kThreads, 1) gemm_tc_kernel(const __grid_constant__ GemmArgs a) {
  static_assert(BN == 256 || BN == 128 || (BN == 192 && EPI == kEpiResid), "CTA-pair tiles");
  constexpr uint32_t TMEM_COLS = BN == 192 ? 512 : 2 * BN;  // two accumulators; a power of two
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) &
                                             ~static_cast<uintptr_t>(1023));
  __shared__ __align__(8) uint64_t full_bar[STAGES];
  __shared__ __align__(8) uint64_t empty_bar[STAGES];
  __shared__ __align__(8) uint64_t tfull_bar[2];
  __shared__ __align__(8) uint64_t tempty_bar[2];
  __shared__ __align__(8) uint64_t drain_bar;
  __shared__ uint32_t tmem_base_sh;
  __shared__ volatile int abort_flag;
  griddep_launch_dependents();
  const int warp = __shfl_sync(0xffffffffu, threadIdx.x >> 5, 0);  // uniform
  const int lane = threadIdx.x & 31;
  const uint32_t rank = cluster_ctarank();
  const bool leader = rank == 0;
  const int unit = blockIdx.x / kPair;
  const int n_units = gridDim.x / kPair;

  if (threadIdx.x == 0) {
    for (int s = 0; s < STAGES; ++s) {
      mbar_init(&full_bar[s], 1);
      mbar_init(&empty_bar[s], 1);
    }
    for (int i = 0; i < 2; ++i) {
      mbar_init(&tfull_bar[i], 1);
      mbar_init(&tempty_bar[i], 4 * kPair);
    }
    mbar_init(&drain_bar, 1);
    abort_flag = 0;
    fence_barrier_init();
  }
  if (warp == 0 && lane == 0) {
    tma_prefetch_desc(&a.tmA);
    for (int i = 0; i < 3; ++i) tma_prefetch_desc(&a.tmB[i]);
    if (a.n_slots > 0) {
      tma_prefetch_desc(&a.tmXA);
      for (int i = 0; i < a.n_slots; ++i) tma_prefetch_desc(&a.tmLA[i]);
      for (int i = 0; i < 3; ++i) tma_prefetch_desc(&a.tmBX[i]);
    }
  }
  if (warp == 1) {
    tmem_alloc_pair(&tmem_base_sh, TMEM_COLS);
    tmem_relinquish_pair();
  }
  tc_fence_before();
  cluster_sync();
  tc_fence_after();
  const uint32_t tmem_base = tmem_base_sh;
  griddep_wait();  // the set-up above touches nothing that the kernels before write
  // a rejected call: every CTA of every cluster sees the same word and has no work
  const int total_items = call_aborted(a.abort) ? 0 : a.total_items;

  if (warp == 0) {
    // ------------------------------------------------------------ TMA producer (every CTA)
    // The whole warp runs the loop, one lane issues.
    const bool issuer = elect_one();
    Ring ring{0, 0u, 1, 0};
    for (int t = unit; t < total_items && ring.ok; t += n_units) {
      const Tile tl = decode_tile(t, a);
      const int m0 = tl.m_blk * (BM * kPair) + static_cast<int>(rank) * BM;
      if (tl.xa) {
        ring = load_xa_item<BN, STAGES>(a, m0, rank, leader, issuer, smem, full_bar, empty_bar, &abort_flag, ring);
        continue;
      }
      int g0, nb, yb, b_step;
      tile_b_rows<BN>(a, tl, rank, g0, nb, yb, b_step);
      // Whether the row block's XA rows are stored, asked (acquire) while the stages already
      // copied still feed the MMAs; only a tile whose row block's XA items have not finished by
      // then waits at its LoRA stage.
      int xa_ready = 0;
      if (a.ext_on[tl.g]) {
        asm volatile("ld.acquire.gpu.global.b32 %0, [%1];" : "=r"(xa_ready) : "l"(a.xa_flags + tl.m_blk) : "memory");
        xa_ready = __all_sync(0xffffffffu, xa_ready >= kXaGroups);
      }
      int stage = ring.stage;
      uint32_t phase = ring.phase;
      const CUtensorMap* mB = &a.tmB[g0];
      for (int kb = 0; kb < a.num_kb; ++kb) {
        if (!mbar_wait_warp(&empty_bar[stage], phase ^ 1, &abort_flag, a.status)) {
          ring.ok = 0;
          break;
        }
        if (issuer) {
          uint8_t* sa = smem + stage * kStageBytes<BN>;
          uint8_t* sb = sa + kABytes;
          // the MMA-issuing CTA's full barrier counts the bytes of both CTAs
          if (leader) mbar_arrive_expect_tx(&full_bar[stage], kPair * kStageBytes<BN>);
          const uint32_t bar = mapa_shared(&full_bar[stage], 0);
          tma_load_2d_pair(sa, &a.tmA, bar, kb * BK, m0);
          for (int j = 0; j < nb; ++j) tma_load_2d_pair(sb + j * b_step, mB + j, bar, kb * BK, yb);
        }
        ++ring.used;
        if (++stage == STAGES) {
          stage = 0;
          phase ^= 1;
        }
      }
      ring.stage = stage;
      ring.phase = phase;
      if (ring.ok && a.ext_on[tl.g])
        ring = load_lora_stage<BN, STAGES>(a, tl, m0, rank, xa_ready != 0, leader, issuer, smem, full_bar, empty_bar,
                                           &abort_flag, ring);
    }
    if (!ring.ok) {
      if (leader) {
        // Let every copy already issued land before the CTA can exit: the last use of every stage.
        for (int s = 0; s < STAGES && s < ring.used; ++s) {
          const int u = ring.used - 1 - s;
          volatile int never = 0;
          mbar_wait(&full_bar[u % STAGES], static_cast<uint32_t>((u / STAGES) & 1), &never, nullptr);
        }
      } else {
        // The peer's copies complete on the other CTA's barriers: give them time to land.
        const unsigned long long t0 = globaltimer_ns();
        while (globaltimer_ns() - t0 < 200000ull) {
        }
      }
    }
  } else if (warp == 1) {
    // ------------------------------------------------------------ MMA issuer (even CTA)
    // The whole warp runs the loop, one lane issues.
    if (leader) {
      const bool issuer = elect_one();
      Ring ring{0, 0u, 1, 0};
      int it = 0;
      bool issued = false;
      const uint32_t idesc = idesc_bf16_f32(BM * kPair, BN);
      const uint32_t idesc_xa = idesc_bf16_f32(BM * kPair, a.n_slots > 0 ? a.xa_n : 32);
      for (int t = unit; t < total_items && ring.ok; t += n_units, ++it) {
        const Tile tl = decode_tile(t, a);
        const int acc = it & 1;
        const uint32_t acc_phase = (it >> 1) & 1;
        if (!mbar_wait_warp<true>(&tempty_bar[acc], acc_phase ^ 1, &abort_flag, a.status)) {
          ring.ok = 0;
          break;
        }
        tc_fence_after();
        const uint32_t d_tmem = tmem_base + acc * BN;
        issued = true;
        if (tl.xa) {
          ring = mma_xa_item<BN, STAGES>(a, d_tmem, idesc_xa, issuer, smem, full_bar, empty_bar, &abort_flag, ring);
          if (!ring.ok) break;
          if (issuer) mma_commit_pair(&tfull_bar[acc], 0x3);
          continue;
        }
        int stage = ring.stage;
        uint32_t phase = ring.phase;
        for (int kb = 0; kb < a.num_kb; ++kb) {
          if (!mbar_wait_warp(&full_bar[stage], phase, &abort_flag, a.status)) {
            ring.ok = 0;
            break;
          }
          tc_fence_after();
          const uint32_t sa = smem_u32(smem + stage * kStageBytes<BN>);
          const uint64_t ad = smem_desc(sa, 16, 1024, kSwizzle128B);
          const uint64_t bd = smem_desc(sa + kABytes, 16, 1024, kSwizzle128B);
          if (issuer) {
            // K = 16 steps advance 32 bytes = 2 units of the descriptor's start-address field
#pragma unroll
            for (int k = 0; k < BK / 16; ++k)
              mma_bf16_ss_pair(d_tmem, ad + 2 * k, bd + 2 * k, idesc, (kb > 0 || k > 0) ? 1u : 0u);
            mma_commit_pair(&empty_bar[stage], 0x3);
          }
          if (++stage == STAGES) {
            stage = 0;
            phase ^= 1;
          }
        }
        ring.stage = stage;
        ring.phase = phase;
        if (ring.ok && a.ext_on[tl.g]) {
          // the XA and BX copies have landed
          if (!mbar_wait_warp(&full_bar[ring.stage], ring.phase, &abort_flag, a.status)) {
            ring.ok = 0;
          } else {
            tc_fence_after();
            const uint32_t sa = smem_u32(smem + ring.stage * kStageBytes<BN>);
            const uint64_t ad = smem_desc(sa, 16, 1024, kSwizzle128B);
            const uint64_t bd = smem_desc(sa + kABytes, 16, 1024, kSwizzle128B);
            if (issuer) {
              for (int k = 0; k < a.ext_steps[tl.g]; ++k) mma_bf16_ss_pair(d_tmem, ad + 2 * k, bd + 2 * k, idesc, 1u);
              mma_commit_pair(&empty_bar[ring.stage], 0x3);
            }
            ring_next<STAGES>(ring);
          }
        }
        if (!ring.ok) break;
        if (issuer) mma_commit_pair(&tfull_bar[acc], 0x3);
      }
      if (!ring.ok && issued && issuer) {
        mma_commit_pair(&drain_bar, 0x1);
        volatile int never = 0;
        mbar_wait(&drain_bar, 0, &never, nullptr);
      }
    }
  } else {
    // ------------------------------------------------------------ epilogue (warps 2..5, every CTA)
    const int quarter = warp & 3;  // TMEM lane quarter this warp may access
    const int row_in_cta = quarter * 32 + lane;
    uint32_t tempty_addr[2];
    for (int i = 0; i < 2; ++i) tempty_addr[i] = mapa_shared(&tempty_bar[i], 0);
    int it = 0;
    for (int t = unit; t < total_items; t += n_units, ++it) {
      const Tile tl = decode_tile(t, a);
      const int acc = it & 1;
      const uint32_t acc_phase = (it >> 1) & 1;
      const int row = tl.m_blk * (BM * kPair) + static_cast<int>(rank) * BM + row_in_cta;
      // warp-uniform outcome: the TMEM loads of the epilogue are warp-collective
      if (!__all_sync(0xffffffffu, mbar_wait(&tfull_bar[acc], acc_phase, &abort_flag, a.status)))
        break;
      tc_fence_after();
      const uint32_t tacc = tmem_base + (static_cast<uint32_t>(quarter * 32) << 16) + acc * BN;
      if (tl.xa)
        drain_xa(a, tl.m_blk, tacc, row, lane);
      else
        epilogue_tile<BN, EPI>(a, tl, tacc, row, lane, smem + STAGES * kStageBytes<BN> + quarter * 4096);
      // the accumulator is free once this warp's TMEM loads have completed (tcgen05.wait::ld in
      // the epilogue); the tile's global stores need not be visible first, so the arrival on
      // the MMA-issuing CTA's barrier is relaxed
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive_cluster_relaxed(tempty_addr[acc]);
    }
  }

  tc_fence_before();
  cluster_sync();
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc_pair(tmem_base, TMEM_COLS);
  }
}

// ---------------------------------------------------------------- host side
template <int BN, int STAGES, int EPI>
cudaError_t launch_impl(GemmArgs& args, int num_sms, cudaStream_t stream) {
  constexpr int PAIR = kPair;
  constexpr int smem = STAGES * kStageBytes<BN> + kScratchBytes + 1024;
  auto kern = gemm_tc_kernel<BN, STAGES, EPI>;
  // the attributes and the co-resident cluster count are per device
  static PerDevice once;
  static std::atomic<int> units_of[64];
  int dev = 0, max_units = 0;
  if (!once.pending(&dev)) {
    max_units = units_of[dev].load(std::memory_order_relaxed);
  } else {
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e != cudaSuccess) return e;
    e = cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 0);
    if (e != cudaSuccess) return e;
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = PAIR;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.gridDim = dim3(num_sms);
    cfg.blockDim = dim3(kThreads);
    cfg.dynamicSmemBytes = smem;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    int clusters = 0;
    e = cudaOccupancyMaxActiveClusters(&clusters, kern, &cfg);
    if (e != cudaSuccess) return e;
    max_units = std::max(1, std::min(clusters, num_sms / PAIR));
    if (dev >= 0 && dev < 64) units_of[dev].store(max_units, std::memory_order_relaxed);
    once.done(dev);
  }
  // every unit of the grid is resident at once (one CTA per SM): a tile that waits for its row
  // block's XA items never waits on a unit that has not started, and every unit runs its XA items
  // before its tiles
  const int units = std::max(1, std::min(max_units, args.total_items));
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = PAIR;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.gridDim = dim3(PAIR * units);
  cfg.blockDim = dim3(kThreads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = stream;
  cfg.attrs = attr;
  cfg.numAttrs = pdl_active() ? 2 : 1;
  return cudaLaunchKernelEx(&cfg, kern, args);
}

int group_tiles(const GemmDesc& d, int g, int bn) {
  const int cols = d.nseg > 1 ? bn / d.nseg : bn;
  return (d.group_cols[g] + cols - 1) / cols;
}

// 256-column tiles run the MMAs at their best rate; narrower ones leave less of the last wave empty
// and less of the epilogue exposed at its end. Compared in K blocks of a 256-column tile, with factors
// from launches of the 1.5B and 7B shapes' widths (others were not timed): a tile's
// hand-over costs about two, the last epilogue 10 per 256 columns, a 192-column block 0.84 and a
// 128-column one 0.8 (its operands are half again as many bytes from L2 per FLOP: down of a 7B batch
// of 8228 rows takes 445 us on 256 columns, 754 on 128). 192 columns only where an epilogue has no
// heads or halves to keep together. Which one is taken changes no result: an element's K order is the
// same.
int tile_columns(const GemmDesc& d, int row_tiles, int num_kb, int units) {
  const int widths[3] = {256, 192, 128};
  const double block[3] = {1.0, 0.84, 0.8};
  int best = 0;
  double best_cost = 0;
  for (int i = 0; i < 3; ++i) {
    const int bn = widths[i];
    if (bn == 192 && d.epi != kEpiResid) continue;
    long tiles = 0;
    for (int g = 0; g < d.ngroups; ++g) tiles += static_cast<long>(group_tiles(d, g, bn)) * row_tiles;
    const long waves = (tiles + units - 1) / std::max(1, units);
    const double cost = waves * (num_kb * block[i] + 2) + 10.0 * bn / 256;
    if (i == 0 || cost < best_cost) {
      best = bn;
      best_cost = cost;
    }
  }
  return best;
}

}  // namespace

cudaError_t launch_gemm(const GemmDesc& d, int num_sms, cudaStream_t stream) {
  constexpr int pair = kPair;
  GemmArgs a;
  std::memset(&a, 0, sizeof(a));
  if (d.nseg != (d.epi == kEpiSwiGLU ? 2 : 1)) return cudaErrorInvalidValue;
  a.num_kb = (d.K + BK - 1) / BK;
  a.row_tiles = (d.M + BM * pair - 1) / (BM * pair);
  const int bn = tile_columns(d, a.row_tiles, a.num_kb, num_sms / pair);
  // rows of one B load: the CTA's share of the tile (plain) or one stacked segment
  const int b_box = d.nseg == 1 ? bn / pair : bn / d.nseg;
  if (!tensor_map_rows(&a.tmA, d.A, d.M, d.K, BM)) return cudaErrorInvalidValue;
  const int nmaps = d.ngroups + d.nseg - 1;
  for (int i = 0; i < 3; ++i) {
    const int src = i < nmaps ? i : 0;  // unused slots alias a valid map
    if (!tensor_map_rows(&a.tmB[i], d.B[src], d.B_rows[src], d.K, b_box)) return cudaErrorInvalidValue;
  }
  bool any_ext = false;
  for (int g = 0; g < d.ngroups; ++g) any_ext |= d.ext_on[g] != 0;
  if (any_ext != (d.n_slots > 0) || d.n_slots < 0 || d.n_slots > 3) return cudaErrorInvalidValue;
  if (any_ext) {
    if (!d.XA || !d.xa_flags || (d.rank != 4 && d.rank != 8 && d.rank != 16)) return cudaErrorInvalidValue;
    if (!tensor_map_rows(&a.tmXA, d.XA, d.M, kXaCols, BM)) return cudaErrorInvalidValue;
    for (int j = 0; j < 3; ++j) {
      const int src = j < d.n_slots ? j : 0;
      if (!d.LA[src] || !tensor_map_rows(&a.tmLA[j], d.LA[src], d.rank, d.K, 16))
        return cudaErrorInvalidValue;
    }
    for (int g = 0; g < d.ngroups; ++g) {
      if (!d.ext_on[g]) continue;
      // the 64-wide block must lie inside the XA row, 16-byte aligned (TMA x coordinate)
      if (d.xa_base[g] < 0 || d.xa_base[g] % 32 != 0 || d.xa_base[g] + BK > kXaCols ||
          d.ext_steps[g] < 1 || d.ext_steps[g] > BK / 16)
        return cudaErrorInvalidValue;
    }
    for (int i = 0; i < 3; ++i) {
      int src = (i < nmaps && d.BX[i]) ? i : -1;
      if (src < 0)
        for (int j = 0; j < nmaps; ++j)
          if (d.BX[j]) src = j;  // unused slots alias a valid map
      if (src < 0) return cudaErrorInvalidValue;
      if (!tensor_map_rows(&a.tmBX[i], d.BX[src], d.B_rows[src], kBxCols, b_box)) return cudaErrorInvalidValue;
    }
    for (int g = 0; g < d.ngroups; ++g)
      for (int s = 0; s < (d.ngroups == 1 ? d.nseg : 1); ++s)
        if (d.ext_on[g] && !d.BX[g + s]) return cudaErrorInvalidValue;
  } else {
    a.tmXA = a.tmA;
    for (int i = 0; i < 3; ++i) a.tmLA[i] = a.tmBX[i] = a.tmA;
  }
  a.M = d.M;
  a.K = d.K;
  a.ngroups = d.ngroups;
  a.nseg = d.nseg;
  a.total_n = 0;
  for (int g = 0; g < d.ngroups; ++g) {
    a.group_cols[g] = d.group_cols[g];
    a.group_tiles[g] = group_tiles(d, g, bn);
    a.total_n += a.group_tiles[g];
    a.ext_on[g] = d.ext_on[g];
    a.ext_steps[g] = d.ext_steps[g];
    a.xa_base[g] = d.xa_base[g];
  }
  a.n_slots = any_ext ? d.n_slots : 0;
  // two CTA halves of 16 x ceil(n_slots / 2) rows: N = 32 for one or two slots, 64 for three
  a.xa_n = 32 * ((a.n_slots + 1) / 2);
  a.rank = d.rank;
  a.xa = static_cast<__nv_bfloat16*>(d.XA);
  a.xa_flags = d.xa_flags;
  a.xa_items = a.n_slots > 0 ? a.row_tiles : 0;
  a.total_items = a.xa_items + a.row_tiles * a.total_n;
  a.epi = d.epi;
  a.scale = d.scale;
  a.out = static_cast<__nv_bfloat16*>(d.out);
  a.ldo = d.ldo;
  a.resid = static_cast<const __nv_bfloat16*>(d.resid);
  a.ld_resid = d.ld_resid;
  for (int i = 0; i < 3; ++i) a.bias[i] = static_cast<const __nv_bfloat16*>(d.bias[i]);
  a.rope = d.rope;
  a.rope_positions = d.rope_positions;
  a.head_dim = d.head_dim;
  a.n_kv_heads = d.n_kv_heads;
  a.qbuf = static_cast<__nv_bfloat16*>(d.qbuf);
  a.ldq = d.ldq;
  a.kpages = static_cast<__nv_bfloat16*>(d.kpages);
  a.vpages = static_cast<__nv_bfloat16*>(d.vpages);
  a.req = d.req;
  a.status = d.status;
  a.abort = d.abort;
  if (d.M == 0 || a.total_n == 0) return cudaSuccess;
  // one kernel per epilogue: each carries only its own epilogue code, which keeps the hot loops
  // of all its warps inside the SM's instruction cache
  if (bn == 192) return launch_impl<192, 7, kEpiResid>(a, num_sms, stream);
  if (bn == 128) switch (d.epi) {
      case kEpiQkv: return launch_impl<128, 8, kEpiQkv>(a, num_sms, stream);
      case kEpiResid: return launch_impl<128, 8, kEpiResid>(a, num_sms, stream);
      case kEpiSwiGLU: return launch_impl<128, 8, kEpiSwiGLU>(a, num_sms, stream);
      default: return cudaErrorInvalidValue;
    }
  switch (d.epi) {
    case kEpiQkv: return launch_impl<256, 6, kEpiQkv>(a, num_sms, stream);
    case kEpiResid: return launch_impl<256, 6, kEpiResid>(a, num_sms, stream);
    case kEpiSwiGLU: return launch_impl<256, 6, kEpiSwiGLU>(a, num_sms, stream);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace crf
