// Decode attention of single rows over the paged cache (the first-step rows carried
// through layers e..N-1: the hybrid execution of Section 3.1 that reads historical states
// from the window end on, and the generated tokens of Section S2.1): for each decode row at
// position pos and query head h,
//   o = softmax(q k^T / sqrt(d)) v over the cached keys 0..pos-1 of that layer plus the
//   row's own fresh (k, v) at position pos.
// The work is memory-bound (K and V of every cached position are read once): the positions
// are cut into chunks of 128 and streamed.
//   decode_attn_stream  one block per SM, walking a run of chunks: of one (row, kv head) pair, or, where
//                       rows are many or of uneven lengths, an equal run of all pairs' chunks
//                       laid end to end, which loads the SMs evenly at the price of a second pair's
//                       start and end in some blocks (the launcher weighs the two). A copy warp
//                       gathers K and V pages with TMA (128-byte swizzle) into a two-stage ring and
//                       does not wait for the kernel before: no kernel of the call writes the
//                       cached positions of the layer. Compute warps w and w + 4 take keys
//                       32 w .. 32 w + 31 of each chunk: both score them, each multiplies its half of
//                       V's columns. For each pair that its run meets, a block first finishes q
//                       (and, where the row's own position falls, k and v) from the q|k|v pass's
//                       partial sums: K splits, bias, up products, rotate-half RoPE, the row's K/V
//                       into its page slot in a generation step. The group's query heads (at most
//                       8) are rows 0..7 of the mma.sync m16n8k16 A operand as bf16(q) and rows
//                       8..15 as bf16(q - bf16(q)), so one product gives the score at fp32
//                       accuracy (K is exact in bf16); P enters P V as bf16. Every warp keeps
//                       an online-softmax state (max, sum and unnormalised o in registers) over
//                       its keys; at the pair's end the warps and the row's own key and value
//                       (scored and added in fp32) meet at the common max in a fixed order and
//                       the block writes one (max, sum, unnormalised o) partial in log2 units.
//   decode_attn_merge   one block per (query head, row, slice of columns): rescales the blocks' partials to the
//                       common max and normalises, every load of up to 32 partials in flight at
//                       once; o leaves as the o pass's bf16 terms.
#include "rows.cuh"
#include "tma_map.h"

#include <algorithm>
#include <cfloat>
#include <cstring>

namespace crf {

namespace {

constexpr int kChunk = 128;  // positions per chunk
constexpr int kStages = 2;   // 64 KB each at d = 128
constexpr int kComputeWarps = 8;
constexpr int kCompute = 32 * kComputeWarps;
constexpr int kThreadsStream = kCompute + 32;  // + one copy warp
constexpr int kMaxGroup = 8;
constexpr int kRedSlots = 4;  // 32-key slices of a chunk, whose o meet in shared memory

__device__ __forceinline__ void named_bar_sync_dec() {
  asm volatile("bar.sync 1, %0;" ::"n"(kCompute) : "memory");
}
// Named barrier that also ANDs a flag over its threads: the compute warps take every later
// barrier together even when one of them gave up on a timed-out wait.
__device__ __forceinline__ bool named_bar_and_dec(bool flag) {
  uint32_t out;
  asm volatile(
      "{\n\t.reg .pred pi, po;\n\t"
      "setp.ne.u32 pi, %1, 0;\n\t"
      "bar.red.and.pred po, 1, %2, pi;\n\t"
      "selp.u32 %0, 1, 0, po;\n\t}"
      : "=r"(out)
      : "r"(flag ? 1u : 0u), "n"(kCompute)
      : "memory");
  return out != 0;
}

struct DecodeArgs {
  CUtensorMap tmK;  // K pool of the layer viewed as [pages*Hkv*16, d], box {64, 16}
  CUtensorMap tmV;
  DecodeAttnDesc d;
  int num_pages;
  int* status;
};

__device__ __forceinline__ int row_chunks(const DecodeAttnDesc& p, int r) { return p.pos[r] / kChunk + 1; }

// With p.per_pair chunks (> 0) a block takes at most so many of one pair, in order: the blocks of a
// pair of row r.
__device__ __forceinline__ int pair_blocks(const DecodeAttnDesc& p, int r) {
  return (row_chunks(p, r) + p.per_pair - 1) / p.per_pair;
}
// Without: block b takes chunks [b total / blocks, (b + 1) total / blocks) of all pairs' chunks; the
// block that holds chunk x.
__device__ __forceinline__ int block_of_chunk(const DecodeAttnDesc& p, int x) {
  return static_cast<int>(((static_cast<long long>(x) + 1) * p.blocks - 1) / p.total_chunks);
}

// The chunk at index x of all pairs' chunks laid end to end (row, kv head, chunk), walked forward.
struct ChunkAt {
  int r, g, c, n;  // n: chunks of the row
  __device__ __forceinline__ void at(const DecodeAttnDesc& p, int x) {
    for (r = 0; r < p.rows; ++r) {
      n = row_chunks(p, r);
      if (x < n * p.n_kv_heads) break;
      x -= n * p.n_kv_heads;
    }
    g = x / n;
    c = x - g * n;
  }
  // This block's run [x0, x1) in the same order, placed at its first chunk.
  __device__ __forceinline__ void run(const DecodeAttnDesc& p, int& x0, int& x1) {
    if (p.per_pair == 0) {
      x0 = static_cast<int>(static_cast<long long>(blockIdx.x) * p.total_chunks / p.blocks);
      x1 = static_cast<int>((static_cast<long long>(blockIdx.x) + 1) * p.total_chunks / p.blocks);
      at(p, x0);
      return;
    }
    int b = blockIdx.x, per = 1;
    x0 = 0;
    for (r = 0; r < p.rows; ++r) {
      n = row_chunks(p, r);
      per = pair_blocks(p, r);
      if (b < per * p.n_kv_heads) break;
      b -= per * p.n_kv_heads;
      x0 += n * p.n_kv_heads;
    }
    g = b / per;
    b -= g * per;
    c = b * p.per_pair;
    x1 = x0 + g * n + min(n, c + p.per_pair);
    x0 += g * n + c;
  }
  __device__ __forceinline__ void next(const DecodeAttnDesc& p) {
    if (++c < n) return;
    c = 0;
    if (++g < p.n_kv_heads) return;
    g = 0;
    if (++r < p.rows) n = row_chunks(p, r);
  }
};

template <int D>
struct StreamSmem {
  static constexpr int HALVES = D / 64;
  static constexpr int HALF = kChunk * 128;   // bytes of one 64-column half of a K (or V) tile
  static constexpr int TILE = HALVES * HALF;
  // o of the kRedSlots slices at the pair's end; before it the finished q in fp32 and the A operand
  static constexpr int RED = kRedSlots * kMaxGroup * D * 4;
  static constexpr int QF = kMaxGroup * D * 4;
  static constexpr int QHALF = 16 * 128;      // one 64-column half of the 16-row A operand
  static_assert(kMaxGroup * D / 4 <= kCompute, "one thread per four columns of the group");
  static_assert(QF + HALVES * QHALF <= RED, "q fits the reduction scratch");
  static constexpr int kBytes = 2 * kStages * TILE + RED + 1024;
};

template <int D>
__global__ void __launch_bounds__(kThreadsStream, 1) decode_attn_stream(const __grid_constant__ DecodeArgs a) {
  using S = StreamSmem<D>;
  constexpr int HALVES = S::HALVES, HALF = S::HALF, TILE = S::TILE, HALF_D = D / 2;
  const DecodeAttnDesc& p = a.d;
  griddep_launch_dependents();
  int x0, x1;
  ChunkAt k;
  k.run(p, x0, x1);
  const int grp = p.n_q_heads / p.n_kv_heads;

  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) &
                                             ~static_cast<uintptr_t>(1023));
  uint8_t* sKV = smem;                                       // [kStages][K tile | V tile]
  uint8_t* sQ = smem + 2 * kStages * TILE;                   // A operand: [HALVES][16 rows][128 B], swizzled
  float (*s_q)[D] = reinterpret_cast<float (*)[D]>(sQ + HALVES * S::QHALF);
  float (*o_red)[kMaxGroup][D] = reinterpret_cast<float (*)[kMaxGroup][D]>(sQ);
  __shared__ float red_m[kRedSlots][kMaxGroup], red_l[kRedSlots][kMaxGroup];
  __shared__ float s_self[kMaxGroup];           // the row's own key, scored in fp32
  __shared__ float s_xa[3][kRankPad];           // the row's scaled down products of q, k, v
  __shared__ float s_k[D], s_v[D];              // own k and v
  __shared__ __align__(8) uint64_t full[kStages], empty[kStages];
  __shared__ volatile int abort_flag;

  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  if (tid == 0) {
    for (int i = 0; i < kStages; ++i) {
      mbar_init(&full[i], 1);
      mbar_init(&empty[i], kComputeWarps);
    }
    abort_flag = 0;
    fence_barrier_init();
  }
  __syncthreads();

  if (warp == kComputeWarps) {
    // ---------------------------------------------------------------- producer
    if (lane == 0) {
      int armed[kStages];
      for (int st = 0; st < kStages; ++st) armed[st] = -1;
      for (int x = x0; x < x1; ++x, k.next(p)) {
        const int i = x - x0, st = i % kStages;
        if (i >= kStages && !mbar_wait(&empty[st], (i / kStages - 1) & 1, &abort_flag, a.status)) break;
        const int t0 = k.c * kChunk;
        const int pages = (min(kChunk, p.pos[k.r] - t0) + kPage - 1) / kPage;
        uint8_t* sK = sKV + st * 2 * TILE;
        uint8_t* sV = sK + TILE;
        if (pages == 0) {
          mbar_arrive(&full[st]);  // only the row's own key here: nothing to copy
          armed[st] = -1;          // and nothing in flight (the stage's previous copies were consumed)
        } else {
          const int32_t* pt = p.page_table[k.r];
          mbar_arrive_expect_tx(&full[st], 2 * pages * HALVES * kPage * 128);
          for (int pg = 0; pg < pages; ++pg) {
            // read before the page check's verdict is known: of an id outside the pool the nearest page
            // is copied, inside the pool's rows (fewer than 2^31: they fit the GPU's memory), and the
            // block stops at the abort word before it uses it
            const int page = min(max(checked_page(pt[t0 / kPage + pg], a.num_pages, a.status), 0), a.num_pages - 1);
            const int row = (page * p.n_kv_heads + k.g) * kPage;
            for (int h = 0; h < HALVES; ++h) {
              const int off = h * HALF + pg * (kPage * 128);
              tma_load_2d(sK + off, &a.tmK, &full[st], 64 * h, row);
              tma_load_2d(sV + off, &a.tmV, &full[st], 64 * h, row);
            }
          }
          armed[st] = (i / kStages) & 1;
        }
      }
      // copies still in flight land before the block's shared memory is released
      volatile int never = 0;
      for (int st = 0; st < kStages; ++st)
        if (armed[st] >= 0) mbar_wait(&full[st], armed[st], &never, nullptr);
    }
    return;
  }

  // -------------------------------------------------------------------- compute warps 0..7
  const float qscale = 1.4426950408889634f * rsqrtf(static_cast<float>(D));  // scores in log2 units
  const uint32_t q_base = smem_u32(sQ);
  const int mi = lane >> 3, li = lane & 7;  // ldmatrix: matrix index, row within it
  const int r0 = lane >> 2, cq = 2 * (lane & 3);
  // a pair's elements, one per thread and turn: q of the group's heads, own k, own v (the last turn may
  // be part-filled: 2.5 turns of eight heads at D = 64). Their bias and B rows are weights: the first
  // pair's are read before the wait.
  constexpr int kTurns = ((kMaxGroup + 2) * D + kCompute - 1) / kCompute;
  static_assert(kTurns * kCompute >= (kMaxGroup + 2) * D, "every element of the largest group has a turn");
  UpRow u[kTurns];
  float val[kTurns];
  auto element = [&](int t, int g, int& m, int& j) {
    const int i = tid + t * kCompute;
    const int h = i / D;
    m = h < grp ? 0 : h - grp + 1;
    j = (m == 0 ? g * grp + h : g) * D + i % D;
  };
  auto load_weights = [&](int g, int n_el) {
#pragma unroll
    for (int t = 0; t < kTurns; ++t) {
      int m, j;
      element(t, g, m, j);
      val[t] = 0.f;
      if (tid + t * kCompute < n_el) {
        u[t] = up_row(p.up[m].B, j, p.lora.rank);
        if (p.bias[m]) val[t] = __bfloat162float(p.bias[m][j]);
      }
    }
  };
  load_weights(k.g, (grp + (k.c + (x1 - x0) >= k.n ? 2 : 0)) * D);
  griddep_wait();  // the q|k|v pass's output
  if (call_aborted(p.abort)) {
    abort_flag = 1;  // the producer stops and lets its copies land
    return;
  }
  bool ok = true;
  for (int x = x0; x < x1;) {
    const int r = k.r, g = k.g;
    const int pos = p.pos[r];
    const int n_run = min(x1 - x, k.n - k.c);       // chunks of this pair in the block's run
    const bool self_here = k.c + n_run == k.n;      // the run's last chunk holds the row's own position
    // partial slot: blocks of the pair before this one
    const int slot = p.per_pair ? k.c / p.per_pair
                                : static_cast<int>(blockIdx.x) - block_of_chunk(p, x - k.c);

    // 1. the elements' K splits (those of every turn in flight together), and meanwhile the down
    // products, whose up products follow
    {
      const int n_el = (grp + (self_here ? 2 : 0)) * D;
      if (x != x0) load_weights(g, n_el);
      const size_t stride = static_cast<size_t>(p.qkv.rows) * p.qkv.ncols;
      const float* row = p.qkv.p + static_cast<size_t>(r) * p.qkv.ncols;
      for (int s0 = 0; s0 < p.qkv.splits; s0 += 4) {
        float w[kTurns][4];
#pragma unroll
        for (int t = 0; t < kTurns; ++t) {
          int m, j;
          element(t, g, m, j);
          const float* src = row + s0 * stride + p.col[min(m, 2)] + j;
          const bool in = tid + t * kCompute < n_el;
#pragma unroll
          for (int q = 0; q < 4; ++q) w[t][q] = in && s0 + q < p.qkv.splits ? __ldcg(src + q * stride) : 0.f;
        }
        float xa = 0.f;
        const int m = tid / kRankPad, q = tid % kRankPad;
        const bool has_xa = tid < 3 * kRankPad && (m == 0 || self_here) && p.up[min(m, 2)].B && q < p.lora.rank;
        if (has_xa) {
          float z[4];
#pragma unroll
          for (int e = 0; e < 4; ++e)
            z[e] = s0 + e < p.qkv.splits ? __ldcg(row + (s0 + e) * stride + p.up[m].xa_col + q) : 0.f;
          xa = (z[0] + z[1]) + (z[2] + z[3]);
        }
        if (tid < 3 * kRankPad) s_xa[m][q] = (s0 > 0 ? s_xa[m][q] : 0.f) + xa * p.lora.scale;
#pragma unroll
        for (int t = 0; t < kTurns; ++t) val[t] += (w[t][0] + w[t][1]) + (w[t][2] + w[t][3]);
      }
      named_bar_sync_dec();
#pragma unroll
      for (int t = 0; t < kTurns; ++t) {
        const int i = tid + t * kCompute;
        const int h = i / D, e = i % D;
        const int m = h < grp ? 0 : h - grp + 1;
        if (i < n_el) {
          if (p.up[m].B) val[t] += up_dot(u[t], s_xa[m]);
          (m == 0 ? s_q[h] : m == 1 ? s_k : s_v)[e] = val[t];
        }
      }
      named_bar_sync_dec();
    }
    // 2. rotation; q scaled, kept in fp32 for the own key's score and split into the A operand
    auto angle = [&](int e) {
      return __ldg(p.rope + (p.rope_by_row ? static_cast<size_t>(r) * HALF_D + e
                                           : (static_cast<size_t>(e / 2) * p.rope_positions + pos) * 2 + e % 2));
    };
    for (int i = tid; i < kMaxGroup * HALF_D / 2; i += kCompute) {
      const int h = i / (HALF_D / 2), e = 2 * (i % (HALF_D / 2));
      float2 lo = make_float2(0.f, 0.f), hi = lo;  // elements e, e + 1 and their rotation partners
      if (h < grp) {
        const float2 c0 = angle(e), c1 = angle(e + 1);
        const float2 a0 = *reinterpret_cast<const float2*>(&s_q[h][e]);
        const float2 a1 = *reinterpret_cast<const float2*>(&s_q[h][e + HALF_D]);
        lo = make_float2((a0.x * c0.x - a1.x * c0.y) * qscale, (a0.y * c1.x - a1.y * c1.y) * qscale);
        hi = make_float2((a1.x * c0.x + a0.x * c0.y) * qscale, (a1.y * c1.x + a0.y * c1.y) * qscale);
        *reinterpret_cast<float2*>(&s_q[h][e]) = lo;
        *reinterpret_cast<float2*>(&s_q[h][e + HALF_D]) = hi;
      }
#pragma unroll
      for (int w = 0; w < 2; ++w) {
        const float2 q = w == 0 ? lo : hi;
        const int d = e + w * HALF_D;
        const float h0 = __bfloat162float(__float2bfloat16_rn(q.x)), h1 = __bfloat162float(__float2bfloat16_rn(q.y));
        const int c = (d % 64) / 8;
        const uint32_t off = (d / 64) * S::QHALF + h * 128 + ((c ^ h) << 4) + (d % 8) * 2;
        *reinterpret_cast<uint32_t*>(sQ + off) = pack_bf16(h0, h1);
        *reinterpret_cast<uint32_t*>(sQ + off + 8 * 128) = pack_bf16(q.x - h0, q.y - h1);
      }
    }
    if (self_here)
      for (int e = tid; e < HALF_D; e += kCompute) {
        const float2 cs = angle(e);
        const float a0 = s_k[e], a1 = s_k[e + HALF_D];
        s_k[e] = a0 * cs.x - a1 * cs.y;
        s_k[e + HALF_D] = a1 * cs.x + a0 * cs.y;
      }
    named_bar_sync_dec();
    uint32_t qf[D / 16][4];  // A fragments, for every chunk of the run
#pragma unroll
    for (int ks = 0; ks < D / 16; ++ks) {
      const int row = (mi & 1) * 8 + li, cc = 2 * (ks % 4) + (mi >> 1);
      ldsm_x4(q_base + (ks / 4) * S::QHALF + row * 128 + ((cc ^ (row & 7)) << 4), qf[ks][0], qf[ks][1], qf[ks][2],
              qf[ks][3]);
    }
    if (self_here) {
      // the row's own key, scored in fp32 (warp w takes head w)
      if (warp < grp) {
        float dot = 0.f;
        for (int d = lane; d < D; d += 32) dot += s_q[warp][d] * s_k[d];
        dot = warp_sum(dot);
        if (lane == 0) s_self[warp] = dot;
      }
      if (p.write_kv) {
        // this layer's copies may read the slot meanwhile: its score is masked and its V row zeroed
        const int page = checked_page(p.page_table[r][pos / kPage], a.num_pages, tid == 0 ? a.status : nullptr);
        const size_t dst = ((static_cast<size_t>(page) * p.n_kv_heads + g) * kPage + pos % kPage) * D;
        for (int e = tid; e < D; e += kCompute) {
          p.kpages[dst + e] = __float2bfloat16_rn(s_k[e]);
          p.vpages[dst + e] = __float2bfloat16_rn(s_v[e]);
        }
      }
    }

    // 3. the run's chunks. This warp's state over its 32 keys of every chunk: max and partial sum
    // of head r0 (log2 units), and its half of the unnormalised o's columns (cq, cq + 1 of every 8)
    float m0 = -INFINITY, l0 = 0.f;
    float O[D / 16][4];
#pragma unroll
    for (int dn = 0; dn < D / 16; ++dn)
#pragma unroll
      for (int e = 0; e < 4; ++e) O[dn][e] = 0.f;
    const int key0 = (warp & 3) * 32;
    const int u0 = (warp >> 2) * (D / 16);  // first 16-byte unit (8 columns) of this warp's half of V
    for (int q = 0; q < n_run; ++q, ++x, k.next(p)) {
      const int i = x - x0, st = i % kStages;
      const int n_cached = min(kChunk, pos - k.c * kChunk);  // cached keys of this chunk
      if (ok) ok = __all_sync(0xffffffffu, mbar_wait(&full[st], (i / kStages) & 1, &abort_flag, a.status));
      const uint32_t k_base = smem_u32(sKV + st * 2 * TILE), v_base = k_base + TILE;
      if (ok && key0 < n_cached && n_cached < key0 + 32) {
        // V rows from the row's own slot on are zeroed (its value is added in fp32 at the end, and
        // 0 * stale data must not produce NaN in P V); each warp reads its own rows and half only
        for (int w = lane; w < 32 * (D / 16); w += 32) {
          const int t2 = key0 + w / (D / 16), u = u0 + w % (D / 16);
          if (t2 >= n_cached)
            *reinterpret_cast<uint4*>(sKV + st * 2 * TILE + TILE + (u / 8) * HALF + t2 * 128 +
                                      (((u % 8) ^ (t2 & 7)) << 4)) = make_uint4(0, 0, 0, 0);
        }
        fence_proxy_async_smem();  // before the stage's next copies
        __syncwarp();
      }
      if (ok && key0 < n_cached) {
        // S = Q K^T for this warp's 32 keys: 4 n-tiles of 8 keys
        float sc[4][4];
#pragma unroll
        for (int nt = 0; nt < 4; ++nt)
#pragma unroll
          for (int e = 0; e < 4; ++e) sc[nt][e] = 0.f;
#pragma unroll
        for (int ks = 0; ks < D / 16; ++ks) {
          const int cc = 2 * (ks % 4) + (mi & 1);
#pragma unroll
          for (int np = 0; np < 2; ++np) {
            const int key = key0 + (2 * np + (mi >> 1)) * 8 + li;
            uint32_t b0, b1, b2, b3;
            ldsm_x4(k_base + (ks / 4) * HALF + key * 128 + ((cc ^ (key & 7)) << 4), b0, b1, b2, b3);
            mma16816(sc[2 * np], qf[ks], b0, b1);
            mma16816(sc[2 * np + 1], qf[ks], b2, b3);
          }
        }
        // high + low part, mask past this chunk's cached keys, online max / sum update
        float s[8];
        float c0 = -INFINITY;
#pragma unroll
        for (int e = 0; e < 8; ++e) {
          s[e] = sc[e >> 1][e & 1] + sc[e >> 1][2 + (e & 1)];
          if (key0 + (e >> 1) * 8 + cq + (e & 1) >= n_cached) s[e] = -INFINITY;
          c0 = fmaxf(c0, s[e]);
        }
#pragma unroll
        for (int o = 1; o <= 2; o <<= 1) c0 = fmaxf(c0, __shfl_xor_sync(0xffffffffu, c0, o));
        const float n0 = fmaxf(m0, c0);
        if (__any_sync(0xffffffffu, n0 > m0)) {
          // a slice with nothing valid so far keeps max -inf: no rescale, P = 0
          const float a0 = n0 == -INFINITY ? 1.f : ex2_approx(m0 - n0);
          m0 = n0;
          l0 *= a0;
#pragma unroll
          for (int dn = 0; dn < D / 16; ++dn) {
            O[dn][0] *= a0;
            O[dn][1] *= a0;
          }
        }
        const float z0 = m0 == -INFINITY ? 0.f : m0;
#pragma unroll
        for (int e = 0; e < 8; ++e) {
          s[e] = ex2_approx(s[e] - z0);
          l0 += s[e];
        }
        // O += P V: P from the score fragments, V by transposing loads
#pragma unroll
        for (int j = 0; j < 2; ++j) {
          const uint32_t pa[4] = {pack_bf16(s[4 * j], s[4 * j + 1]), 0u, pack_bf16(s[4 * j + 2], s[4 * j + 3]), 0u};
          const int vkey = key0 + 16 * j + (mi & 1) * 8 + li;
#pragma unroll
          for (int dp = 0; dp < D / 32; ++dp) {
            const int u = u0 + 2 * dp + (mi >> 1);  // 16-byte unit of the row (8 dims)
            uint32_t b0, b1, b2, b3;
            ldsm_x4_t(v_base + (u / 8) * HALF + vkey * 128 + (((u % 8) ^ (vkey & 7)) << 4), b0, b1, b2, b3);
            mma16816(O[2 * dp], pa, b0, b1);
            mma16816(O[2 * dp + 1], pa, b2, b3);
          }
        }
      }
      __syncwarp();
      if (lane == 0) mbar_arrive(&empty[st]);  // this warp is done with the stage
    }

    // 4. the slices' states (and the row's own key) meet at the common max, in a fixed order
#pragma unroll
    for (int o = 1; o <= 2; o <<= 1) l0 += __shfl_xor_sync(0xffffffffu, l0, o);
    if (warp < kRedSlots && (lane & 3) == 0) red_m[warp][r0] = m0;
    ok = named_bar_and_dec(ok);
    float M = self_here && r0 < grp ? s_self[r0] : -INFINITY;
#pragma unroll
    for (int w = 0; w < kRedSlots; ++w) M = fmaxf(M, red_m[w][r0]);
    const float f0 = m0 == -INFINITY ? 0.f : ex2_approx(m0 - M);
    if (warp < kRedSlots && (lane & 3) == 0) red_l[warp][r0] = l0 * f0;
#pragma unroll
    for (int dn = 0; dn < D / 16; ++dn)
      *reinterpret_cast<float2*>(&o_red[warp & 3][r0][8 * (u0 + dn) + cq]) = make_float2(O[dn][0] * f0, O[dn][1] * f0);
    named_bar_sync_dec();
    if (ok && tid < grp * (D / 4)) {  // four columns of one head per thread
      const int h = tid / (D / 4), d = 4 * (tid % (D / 4));
      float mx = self_here ? s_self[h] : -INFINITY, L = 0.f;
#pragma unroll
      for (int w = 0; w < kRedSlots; ++w) {
        mx = fmaxf(mx, red_m[w][h]);
        L += red_l[w][h];
      }
      const float ps = self_here ? ex2_approx(s_self[h] - mx) : 0.f;
      float o[4];
#pragma unroll
      for (int e = 0; e < 4; ++e) o[e] = self_here ? ps * s_v[d + e] : 0.f;
#pragma unroll
      for (int w = 0; w < kRedSlots; ++w) {
        const float4 v = *reinterpret_cast<const float4*>(&o_red[w][h][d]);
        o[0] += v.x;
        o[1] += v.y;
        o[2] += v.z;
        o[3] += v.w;
      }
      float* out = p.part + ((static_cast<size_t>(r) * p.n_q_heads + g * grp + h) * p.splits + slot) * (D + 2);
      *reinterpret_cast<float2*>(out + d) = make_float2(o[0], o[1]);
      *reinterpret_cast<float2*>(out + d + 2) = make_float2(o[2], o[3]);
      if (d == 0) {
        out[D] = mx;
        out[D + 1] = ps + L;
      }
    }
    if (x < x1) named_bar_sync_dec();  // the scratch is free for the next pair
  }
}

// One block per (query head, row, slice of kCols columns): 128 threads = kCols columns x groups of
// partials (group q takes partials q, q + groups, ...). Each thread folds its partials with an online
// max, eight loads in flight, then the groups meet in a fixed order. Blocks this small fit beside the
// stream kernel's, so they, and behind them the o pass's first weights, are there when it ends.
constexpr int kMergeThreads = 128;
template <int D, int kCols>
__global__ void __launch_bounds__(kMergeThreads) decode_attn_merge(const __grid_constant__ DecodeAttnDesc p) {
  constexpr int kGroups = kMergeThreads / kCols;
  griddep_launch_dependents();
  const int h = blockIdx.x, r = blockIdx.y, c = threadIdx.x % kCols, q = threadIdx.x / kCols;
  const int col = blockIdx.z * kCols + c;
  int first = 0;
  for (int i = 0; i < r; ++i) first += row_chunks(p, i) * p.n_kv_heads;
  const int n = row_chunks(p, r);
  first += h / (p.n_q_heads / p.n_kv_heads) * n;
  const int parts =
      p.per_pair ? pair_blocks(p, r) : block_of_chunk(p, first + n - 1) - block_of_chunk(p, first) + 1;
  const float* base = p.part + (static_cast<size_t>(r) * p.n_q_heads + h) * p.splits * (D + 2);
  __shared__ float red_m[kGroups], red_l[kGroups], red_o[kGroups][kCols];
  griddep_wait();  // the partials come from decode_attn_stream
  float m = -INFINITY, l = 0.f, acc = 0.f;
  for (int s0 = q; s0 < parts; s0 += 8 * kGroups) {
    float pm[8], pl[8], po[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const int s = s0 + i * kGroups;
      const float* ps = base + static_cast<size_t>(s) * (D + 2);
      const bool in = s < parts;
      pm[i] = in ? __ldcg(ps + D) : -INFINITY;
      pl[i] = in ? __ldcg(ps + D + 1) : 0.f;
      po[i] = in ? __ldcg(ps + col) : 0.f;
    }
    float nm = m;
#pragma unroll
    for (int i = 0; i < 8; ++i) nm = fmaxf(nm, pm[i]);
    const float f = m == -INFINITY ? 0.f : ex2_approx(m - nm);
    l *= f;
    acc *= f;
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const float e = pm[i] == -INFINITY ? 0.f : ex2_approx(pm[i] - nm);
      l += e * pl[i];
      acc += e * po[i];
    }
    m = nm;
  }
  red_o[q][c] = acc;
  if (c == 0) {
    red_m[q] = m;
    red_l[q] = l;
  }
  __syncthreads();
  if (q != 0) return;
  float M = red_m[0];
#pragma unroll
  for (int i = 1; i < kGroups; ++i) M = fmaxf(M, red_m[i]);
  float o = 0.f, L = 0.f;
#pragma unroll
  for (int i = 0; i < kGroups; ++i) {
    const float e = red_m[i] == -INFINITY ? 0.f : ex2_approx(red_m[i] - M);
    o += e * red_o[i][c];
    L += e * red_l[i];
  }
  const int qd = p.n_q_heads * D;
  __nv_bfloat16* dst = p.out + static_cast<size_t>(r) * p.terms * qd + h * D + col;
  if (p.terms == 2)
    store_terms<2>(dst, qd, o / L);
  else
    store_terms<3>(dst, qd, o / L);
}

template <int D>
cudaError_t launch_dec(const DecodeArgs& args, cudaStream_t stream) {
  constexpr int smem = StreamSmem<D>::kBytes;
  static PerDevice once;
  int dev = 0;
  if (once.pending(&dev)) {
    cudaError_t e = cudaFuncSetAttribute(decode_attn_stream<D>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e != cudaSuccess) return e;
    once.done(dev);
  }
  const DecodeAttnDesc& d = args.d;
  cudaError_t e = launch_kernel(decode_attn_stream<D>, dim3(d.blocks), dim3(kThreadsStream), smem, stream, args);
  if (e != cudaSuccess) return e;
  // many partials a head (few rows): four groups share them
  if (d.blocks > 8 * d.rows * d.n_kv_heads)
    return launch_kernel(decode_attn_merge<D, 32>, dim3(d.n_q_heads, d.rows, D / 32), dim3(kMergeThreads), 0, stream, d);
  return launch_kernel(decode_attn_merge<D, D>, dim3(d.n_q_heads, d.rows), dim3(kMergeThreads), 0, stream, d);
}

}  // namespace

int decode_attention_splits(int max_positions) { return std::max(1, (max_positions + kChunk - 1) / kChunk); }

cudaError_t launch_decode_attention(const DecodeAttnDesc& d, int num_pages, int num_sms, int* status,
                                    cudaStream_t stream) {
  if (d.rows < 1) return cudaSuccess;
  if (d.n_q_heads % d.n_kv_heads != 0 || d.n_q_heads / d.n_kv_heads > kMaxGroup)
    return cudaErrorInvalidValue;
  if (num_sms < 1) return cudaErrorInvalidValue;
  long total = 0;
  for (int r = 0; r < d.rows; ++r) {
    if (d.pos[r] / kChunk + 1 > d.splits) return cudaErrorInvalidValue;
    total += static_cast<long>(d.n_kv_heads) * (d.pos[r] / kChunk + 1);
  }
  if (total > 0x7fffffffl) return cudaErrorInvalidValue;
  DecodeArgs a;
  std::memset(&a, 0, sizeof(a));
  const long pool_rows = static_cast<long>(num_pages) * d.n_kv_heads * kPage;
  if (!tensor_map_rows(&a.tmK, d.kpages, pool_rows, d.head_dim, kPage) ||
      !tensor_map_rows(&a.tmV, d.vpages, pool_rows, d.head_dim, kPage))
    return cudaErrorInvalidValue;
  a.d = d;
  a.d.total_chunks = static_cast<int>(total);
  // One block per SM. Whole pairs: the fewest chunks a block that keep all blocks in one wave; a
  // pair's start and end cost about as much as three chunks (5 us against 1.5 us), and a run that
  // ignores the pairs pays them up to twice (7B shape, 32 rows of 1K-4K keys: 49 us against 62).
  a.d.blocks = static_cast<int>(std::min<long>(num_sms, total));
  int per = static_cast<int>((total + num_sms - 1) / num_sms);
  const int even = per;
  auto blocks_for = [&](int c) {
    long b = 0;
    for (int r = 0; r < d.rows; ++r) b += static_cast<long>(d.n_kv_heads) * ((d.pos[r] / kChunk + c) / c);
    return b;
  };
  const long least = static_cast<long>(d.rows) * d.n_kv_heads;  // blocks with a pair each
  while (least <= num_sms && blocks_for(per) > num_sms) ++per;
  if (least <= num_sms && per + 3 <= even + 6) {
    a.d.per_pair = per;
    a.d.blocks = static_cast<int>(blocks_for(per));
  } else {
    a.d.per_pair = 0;
  }
  a.num_pages = num_pages;
  a.status = status;
  if (d.head_dim == 128) return launch_dec<128>(a, stream);
  if (d.head_dim == 64) return launch_dec<64>(a, stream);
  return cudaErrorInvalidValue;
}

}  // namespace crf
