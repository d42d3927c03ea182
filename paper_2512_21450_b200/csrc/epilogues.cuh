// Epilogue functors of the GEMM engine.  An epilogue thread owns one row of the 128x256 accumulator
// tile (with eight warps: one row of one half of its columns) and receives it in chunks of 32 columns.
#pragma once
#include <math_constants.h>

#include "gemm_engine.cuh"

namespace rlh {

constexpr float kLog2e = 1.4426950408889634f;
constexpr float kLn2 = 0.6931471805599453f;

// One MUFU instruction: 2^x, denormal results flushed to zero (arguments here are <= 0 up to
// rounding, results in [0, 1]); -inf gives 0.
__device__ __forceinline__ float ex2_approx(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

// ---------------------------------------------------------------------------------------------
// Forward statistics (policy over the vocabulary, section 2.2): for its row and the vocabulary
// range of the work unit, keeps the running maximum M, S = sum exp(z-M), A = sum exp(z-M) z and
// the logit of the sampled token.  Logits never leave the chip; one float4 per (range, row) does.
struct RowStats {
  static constexpr bool kParts = false;
  static constexpr int kSideWarps = 0;
  static constexpr bool kFeeds = false, kAhead = false;
  static constexpr int kStagingBytes = 0;
  struct Params {
    const int* tokens_c;   // [rows] compact sampled-token ids
    float4* partials;      // [n_ranges][part_stride]
    int part_stride;
    int V;
  };
  struct State {
    float m, s, a, zy;
    int y;
  };
  __device__ static __forceinline__ void begin_unit(const Params& p, State& st, int m_tile, int, int row_in_tile,
                                                    int m_rows, int, int) {
    st.m = -CUDART_INF_F;
    st.s = 0.f;
    st.a = 0.f;
    st.zy = 0.f;
    const int row = m_tile * BM + row_in_tile;
    st.y = row < m_rows ? p.tokens_c[row] : -1;
  }
  __device__ static __forceinline__ void init(State&) {}
  __device__ static __forceinline__ void finish(State&) {}
  __device__ static __forceinline__ void chunk(const Params& p, State& st, int, int n_tile, int c, int, int,
                                               const float (&v)[32], const CUtensorMap*, uint32_t) {
    const int col0 = n_tile * BN + c * 32;
    const int nvalid = p.V - col0;
    if (nvalid <= 0) return;
    float cmax = -CUDART_INF_F;
    if (nvalid >= 32) {
#pragma unroll
      for (int i = 0; i < 32; i += 2) cmax = fmaxf(cmax, fmaxf(v[i], v[i + 1]));
    } else {
#pragma unroll
      for (int i = 0; i < 32; ++i) cmax = i < nvalid ? fmaxf(cmax, v[i]) : cmax;
    }
    const float newm = fmaxf(st.m, cmax);
    const float scale = ex2_approx((st.m - newm) * kLog2e);
    const float mL = newm * kLog2e;
    float cs = 0.f, ca = 0.f;
    if (nvalid >= 32) {
      // two columns per instruction (packed fp32 pairs): e = 2^(z*log2e - M*log2e), S += e, A += e*z
      const float2 l2 = make_float2(kLog2e, kLog2e), nm2 = make_float2(-mL, -mL);
      float2 cs2 = make_float2(0.f, 0.f), ca2 = make_float2(0.f, 0.f);
#pragma unroll
      for (int i = 0; i < 32; i += 2) {
        const float2 z2 = make_float2(v[i], v[i + 1]);
        const float2 t2 = __ffma2_rn(z2, l2, nm2);
        const float2 e2 = make_float2(ex2_approx(t2.x), ex2_approx(t2.y));
        cs2 = __fadd2_rn(cs2, e2);
        ca2 = __ffma2_rn(e2, z2, ca2);
      }
      cs = cs2.x + cs2.y;
      ca = ca2.x + ca2.y;
    } else {
#pragma unroll
      for (int i = 0; i < 32; ++i) {
        const float e = i < nvalid ? ex2_approx(fmaf(v[i], kLog2e, -mL)) : 0.f;
        cs += e;
        ca = fmaf(e, v[i], ca);
      }
    }
    st.s = fmaf(st.s, scale, cs);
    st.a = fmaf(st.a, scale, ca);
    st.m = newm;
    const unsigned rel = (unsigned)(st.y - col0);
    if (rel < 32u && (int)rel < nvalid) {
      float z = 0.f;
#pragma unroll
      for (int i = 0; i < 32; ++i) z = (rel == (unsigned)i) ? v[i] : z;
      st.zy = z;
    }
  }
  // the two column halves of a row: as the merge of two vocabulary ranges
  static constexpr int kMerge = 4;
  __device__ static __forceinline__ void pack(const State& st, float (&x)[kMerge]) {
    x[0] = st.m; x[1] = st.s; x[2] = st.a; x[3] = st.zy;
  }
  __device__ static __forceinline__ void merge(State& st, const float (&x)[kMerge]) {
    const float m = fmaxf(st.m, x[0]);
    // a half that saw no column inside the vocabulary has m = -inf and sums of 0
    const float a = st.m == m ? 1.f : ex2_approx((st.m - m) * kLog2e), b = x[0] == m ? 1.f : ex2_approx((x[0] - m) * kLog2e);
    st.s = fmaf(st.s, a, x[1] * b);
    st.a = fmaf(st.a, a, x[2] * b);
    st.zy += x[3];
    st.m = m;
  }
  __device__ static __forceinline__ void end_unit(const Params& p, State& st, int m_tile, int nr, int row_in_tile,
                                                  int m_rows) {
    const int row = m_tile * BM + row_in_tile;
    if (row < m_rows) p.partials[(size_t)nr * p.part_stride + row] = make_float4(st.m, st.s, st.a, st.zy);
  }
};

// With four epilogue warps (one per scheduler) their latencies are exposed and a tile's epilogue takes 3.8 us; with
// eight it takes 2.7, but they slow the MMA issuer down.  So eight where K is short: 8192 rows x 151936 words, score pass
// 908 / 1072 / 1377 / 1608 / 3072 us with four, 752 / 949 / 1250 / 1668 / 3718 with eight at d = 256 / 512 / 768 / 1024 / 2048.
constexpr int kEightWarpsMaxK = 896;
template <int W>
struct EpiStats : RowStats {
  static constexpr int kWarps = W;
};

// ---------------------------------------------------------------------------------------------
// 32 rows x 32 columns of 16-bit values (two per word, one row per lane) into one half of a 128-byte-swizzled 32 x 64
// box; c = index of the 32-column chunk.  The second half hands the box to the TMA unit.
template <int BUFS>   // boxes per warp
__device__ __forceinline__ void stage_half_box(const uint32_t (&w)[16], int c, uint32_t staging, uint32_t& n_issued,
                                               const CUtensorMap* map, int col, int row0) {
  const int lane = threadIdx.x & 31;
  const uint32_t buf = staging + (n_issued % BUFS) * kBoxBytes;
  if ((c & 1) == 0) {
    // first half of a new box: the last store issued from this buffer must have read it
    if (lane == 0) bulk_wait_group_read<BUFS - 1>();
    __syncwarp();
  }
  // row `lane` of the box is 128 bytes = 8 chunks of 8 values; chunk j sits at position j ^ (row & 7)
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    const uint32_t jj = uint32_t(4 * (c & 1) + j);
    const uint32_t addr = buf + lane * 128u + ((jj ^ uint32_t(lane & 7)) << 4);
    asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(addr), "r"(w[4 * j]), "r"(w[4 * j + 1]),
                 "r"(w[4 * j + 2]), "r"(w[4 * j + 3])
                 : "memory");
  }
  if (c & 1) {
    fence_proxy_async_smem();
    __syncwarp();
    if (lane == 0) {
      tma_store_2d(map, buf, col - 32, row0);
      bulk_commit_group();
    }
    n_issued++;
  }
}

// Forward statistics of EpiStats for one slab of rows, plus the logits themselves: kept in fp32 in the slab between the
// pass that forms them and the point where the row's log-sum-exp and loss coefficients are known, as two 16-bit planes so
// that the gradient can take the place of the upper halves.  Forming the logits once instead of twice (statistics, then
// recomputation for the gradient) leaves 6 d V tensor flops per token of 8 d V.  Both planes are seen through one map
// {columns, rows, planes} with boxes of 32 x 32, 64-byte swizzled.  6912 rows x 151936 words: 1.97 / 2.17 / 3.34 / 5.63 ms at
// d = 896 / 1024 / 2048 / 3584 (eight epilogue warps 1.94 / 2.17 / 3.52 / 5.98; stores straight from registers 1.96 / - / 3.48 / 5.75;
// the statistics alone 1.36 / 1.65 / 2.85 / 5.16).
struct EpiSweep {
  static constexpr bool kParts = false;
  static constexpr int kSideWarps = 0;
  static constexpr bool kFeeds = false, kAhead = false;
  static constexpr int kWarps = 4;
  static constexpr int kStagingBytes = kEpiStaging;
  using Params = RowStats::Params;
  struct State {
    RowStats::State s;
    uint32_t n_issued;
    int grow;   // compact row
  };
  __device__ static __forceinline__ void init(State& st) { st.n_issued = 0; }
  __device__ static __forceinline__ void finish(State& st) {
    if ((threadIdx.x & 31) == 0 && st.n_issued) bulk_wait_group_all();
    __syncwarp();
  }
  __device__ static __forceinline__ void begin_unit(const Params& p, State& st, int m_tile, int, int row_in_tile,
                                                    int m_rows, int slab_off, int) {
    const int rl = m_tile * BM + row_in_tile;
    const bool valid = rl < m_rows;
    st.grow = valid ? slab_off + rl : -1;
    st.s.m = -CUDART_INF_F;
    st.s.s = 0.f;
    st.s.a = 0.f;
    st.s.zy = 0.f;
    st.s.y = valid ? p.tokens_c[st.grow] : -1;
  }
  __device__ static __forceinline__ void chunk(const Params& p, State& st, int m_tile, int n_tile, int c,
                                               int row_in_tile, int m_rows, const float (&v)[32],
                                               const CUtensorMap* map, uint32_t staging) {
    // a CTA pair may own a 128-row tile that lies wholly past the slab's rows: nothing to write
    if (m_tile * BM >= ((m_rows + BM - 1) / BM) * BM) return;
    RowStats::chunk(p, st.s, 0, n_tile, c, 0, 0, v, map, staging);
    const int lane = threadIdx.x & 31;
    constexpr int kBufs = kStagingBytes / kWarps / kBoxBytes;
    const uint32_t buf = staging + (st.n_issued % kBufs) * kBoxBytes;   // 2 KB of upper halves, 2 KB of lower ones
    // the last stores issued from this buffer must have read it
    if (lane == 0) bulk_wait_group_read<kBufs - 1>();
    __syncwarp();
    // row `lane` of a box is 64 bytes = 4 chunks of 8 values; chunk j sits at position j ^ ((row >> 1) & 3)
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      uint32_t h[4], l[4];
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        const uint32_t a = __float_as_uint(v[8 * j + 2 * k]), b = __float_as_uint(v[8 * j + 2 * k + 1]);
        h[k] = __byte_perm(a, b, 0x7632);
        l[k] = __byte_perm(a, b, 0x5410);
      }
      const uint32_t addr = buf + lane * 64u + ((uint32_t(j) ^ (uint32_t(lane >> 1) & 3u)) << 4);
      asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(addr), "r"(h[0]), "r"(h[1]), "r"(h[2]), "r"(h[3]) : "memory");
      asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(addr + kBoxBytes / 2), "r"(l[0]), "r"(l[1]), "r"(l[2]), "r"(l[3])
                   : "memory");
    }
    fence_proxy_async_smem();
    __syncwarp();
    if (lane == 0) {
      const int col = n_tile * BN + c * 32, row0 = m_tile * BM + (row_in_tile - lane);
      tma_store_3d(map, buf, col, row0, 0);
      tma_store_3d(map, buf + kBoxBytes / 2, col, row0, 1);
      bulk_commit_group();
    }
    st.n_issued++;
  }
  static constexpr int kMerge = RowStats::kMerge;
  __device__ static __forceinline__ void pack(const State& st, float (&x)[kMerge]) { RowStats::pack(st.s, x); }
  __device__ static __forceinline__ void merge(State& st, const float (&x)[kMerge]) { RowStats::merge(st.s, x); }
  __device__ static __forceinline__ void end_unit(const Params& p, State& st, int, int nr, int, int) {
    if (st.grow >= 0)
      p.partials[(size_t)nr * p.part_stride + st.grow] = make_float4(st.s.m, st.s.s, st.s.a, st.s.zy);
  }
};

// ---------------------------------------------------------------------------------------------
// Gradient with respect to the logits for one slab of rows x vocabulary columns, rounded to
// bf16 and written to the slab scratch (row-major) by bulk tensor stores: each epilogue warp packs
// two consecutive 32-column chunks of its 32 rows into a 128-byte-swizzled 32x64 bf16 box in
// shared memory (two boxes per warp) and one lane hands the box to the TMA unit:
//   g_tj = cp_t (p_tj - 1[j = y_t]) + ce_t p_tj (log p_tj + Ent_t),  p_tj = exp(z_tj - lse_t)
// cp_t = -w_t dloss_t/dlogp_t and ce_t = w_t ent_coef come from the per-token loss kernel.
// Rows past the valid rows of the slab and columns past V are written as zero.
// Eight warps as in EpiStats: 708 / 661 / 772 / 894 us with four, 484 / 588 / 727 / 903 with eight at d = 256 / 512 / 768 / 1024
// (8192 rows x 75968 words).
struct GradParams {
  const int* tokens_c;
  const float* lse;
  const float* ent;
  const float* cp;
  const float* ce;
  int V;
  int vocab_base;  // global column of the slab's column 0
};
template <int W>
struct EpiGrad {
  static constexpr bool kParts = false;
  static constexpr int kSideWarps = 0;
  static constexpr bool kFeeds = false, kAhead = false;
  static constexpr int kWarps = W;
  static constexpr int kMerge = 0;
  static constexpr int kStagingBytes = kEpiStaging;
  using Params = GradParams;
  struct State {
    float lse, ent, cp, ce;
    int y;
    bool valid;
    uint32_t n_issued;   // boxes handed to the TMA unit so far (selects the staging buffer)
  };
  __device__ static __forceinline__ void begin_unit(const Params& p, State& st, int m_tile, int, int row_in_tile,
                                                    int m_rows, int slab_off, int) {
    const int rl = m_tile * BM + row_in_tile;
    st.valid = rl < m_rows;
    const int gr = slab_off + rl;   // compact row of this slab row
    st.lse = st.valid ? p.lse[gr] : 0.f;
    st.ent = st.valid ? p.ent[gr] : 0.f;
    st.cp = st.valid ? p.cp[gr] : 0.f;
    st.ce = st.valid ? p.ce[gr] : 0.f;
    st.y = st.valid ? p.tokens_c[gr] : -1;
  }
  __device__ static __forceinline__ void init(State& st) { st.n_issued = 0; }
  __device__ static __forceinline__ void finish(State& st) {
    if ((threadIdx.x & 31) == 0 && st.n_issued) bulk_wait_group_all();
    __syncwarp();
  }
  __device__ static __forceinline__ void chunk(const Params& p, State& st, int m_tile, int n_tile, int c,
                                               int row_in_tile, int m_rows, const float (&v)[32],
                                               const CUtensorMap* tmG, uint32_t staging) {
    // a CTA pair may own a 128-row tile that lies wholly past the slab's rows: nothing to write
    if (m_tile * BM >= ((m_rows + BM - 1) / BM) * BM) return;
    const int col_l = n_tile * BN + c * 32;
    const int col_g = p.vocab_base + col_l;
    const int nvalid = p.V - col_g;
    float g[32];
    if (!st.valid || nvalid <= 0) {
#pragma unroll
      for (int i = 0; i < 32; ++i) g[i] = 0.f;
    } else {
      if (st.ce == 0.f) {
        // packed fp32 pairs: p = 2^(z*log2e - lse*log2e), g = cp * p
        const float2 l2 = make_float2(kLog2e, kLog2e), nl2 = make_float2(-st.lse * kLog2e, -st.lse * kLog2e);
        const float2 cp2 = make_float2(st.cp, st.cp);
#pragma unroll
        for (int i = 0; i < 32; i += 2) {
          const float2 t2 = __ffma2_rn(make_float2(v[i], v[i + 1]), l2, nl2);
          const float2 g2 = __fmul2_rn(make_float2(ex2_approx(t2.x), ex2_approx(t2.y)), cp2);
          g[i] = g2.x;
          g[i + 1] = g2.y;
        }
      } else {
        // entropy term as well, still two columns per instruction:
        // g = p * (ce * (z - lse) + (ce * Ent + cp))
        const float2 l2 = make_float2(kLog2e, kLog2e), nl2 = make_float2(-st.lse * kLog2e, -st.lse * kLog2e);
        const float2 nlse2 = make_float2(-st.lse, -st.lse), ce2 = make_float2(st.ce, st.ce);
        const float k = fmaf(st.ce, st.ent, st.cp);
        const float2 k2 = make_float2(k, k);
#pragma unroll
        for (int i = 0; i < 32; i += 2) {
          const float2 z2 = make_float2(v[i], v[i + 1]);
          const float2 t2 = __ffma2_rn(z2, l2, nl2);
          const float2 e2 = make_float2(ex2_approx(t2.x), ex2_approx(t2.y));
          const float2 w2 = __ffma2_rn(ce2, __fadd2_rn(z2, nlse2), k2);
          const float2 g2 = __fmul2_rn(e2, w2);
          g[i] = g2.x;
          g[i + 1] = g2.y;
        }
      }
      const unsigned rel = (unsigned)(st.y - col_g);
      if (rel < 32u) {
#pragma unroll
        for (int i = 0; i < 32; ++i) g[i] = (rel == (unsigned)i) ? g[i] - st.cp : g[i];
      }
      if (nvalid < 32) {
#pragma unroll
        for (int i = 0; i < 32; ++i) g[i] = i < nvalid ? g[i] : 0.f;
      }
    }
    uint32_t w[16];
#pragma unroll
    for (int i = 0; i < 16; ++i) {
      const __nv_bfloat162 b = __floats2bfloat162_rn(g[2 * i], g[2 * i + 1]);
      w[i] = *reinterpret_cast<const uint32_t*>(&b);
    }
    const int lane = threadIdx.x & 31;
    stage_half_box<kStagingBytes / kWarps / kBoxBytes>(w, c, staging, st.n_issued, tmG, col_l, m_tile * BM + (row_in_tile - lane));
  }
  __device__ static __forceinline__ void end_unit(const Params&, State&, int, int, int, int) {}
};

// ---------------------------------------------------------------------------------------------
// Plain fp32 output tile: C[slice][row_base + row, col] = acc (+ previous value when accumulating).
// Each epilogue warp stages its 32x32 chunk in shared memory (128-byte swizzled, two buffers) and
// one lane hands it to the TMA unit: a bulk tensor store, or a bulk tensor reduce-add when
// accumulating.  The output is seen through a 3-D fp32 tensor map {columns, rows, K slices}, which
// also clips rows past the tensor.  Every element is written by exactly one tile per launch, so
// the result does not depend on timing.
struct AccParams {
  int n_cols;
  int accumulate;  // 0 store, 1 add, 2 (slabs walked from the last to the first): add unless this is the last slab that has rows
  const int* n_valid;                      // 2, and where side warps write dH (EpiAccScatter)
  int slab_cap, slab_one, slab_index;
  int row_base;
  int slice_add;   // stream-K launches: output slices past the first are always added to
  int tile_cols;   // > 0: k_slice > 0 names slot k_slice - 1, a box of tile_cols columns x tile_rows rows of its own
  int tile_rows;
};
// W: four warps, or eight for dW of few rows, where the time is the output's (K of a tile is short, and its 128 KB per CTA leave
// through the epilogue).  Adding, the boxes of this worker's next tile are brought to L2 meanwhile: the adds otherwise wait for
// DRAM one box at a time.  dW of 151936 words, d = 2048, four warps / eight: stores 282 / 264 us at 100 rows, 380 / 340 at 300, 468 / 430 at
// 512, and slower from 1000 rows on; adds 542 / 425, 587 / 446, 602 / 524 (the four without prefetches; with them 413 / 494 / 544; a
// plain kernel that adds in this order takes 400).
template <int W>
struct EpiAccW {
  static constexpr bool kParts = true;
  static constexpr int kSideWarps = 0;
  static constexpr bool kFeeds = false, kAhead = W == 8;
  static constexpr int kWarps = W;
  static constexpr int kMerge = 0;
  static constexpr int kStagingBytes = kEpiStaging;
  using Params = AccParams;
  struct State {
    int k_slice;
    int add;
    uint32_t n_issued;   // chunks handed to the TMA unit so far (selects the staging buffer)
    int next_row, next_col;   // this warp's part of the next tile (row -1: none)
  };
  __device__ static __forceinline__ void init(State& st) { st.n_issued = 0; }
  __device__ static __forceinline__ void finish(State& st) {
    if ((threadIdx.x & 31) == 0 && st.n_issued) bulk_wait_group_all();
    __syncwarp();
  }
  __device__ static __forceinline__ void begin_unit(const Params& p, State& st, int, int, int, int, int, int k_slice) {
    st.k_slice = k_slice;
    st.add = p.accumulate == 2 ? p.slab_index + 1 < slab_count(*p.n_valid, p.slab_cap, p.slab_one) : p.accumulate;
  }
  __device__ static __forceinline__ void chunk(const Params& p, State& st, int m_tile, int n_tile, int c,
                                               int row_in_tile, int m_rows, const float (&v)[32],
                                               const CUtensorMap* tmC, uint32_t staging) {
    const int lane = threadIdx.x & 31;
    const int row0 = m_tile * BM + (row_in_tile - lane);   // first row of this warp's 32
    const int col0 = n_tile * BN + c * 32;
    if (row0 >= m_rows || col0 >= p.n_cols) return;        // warp-uniform
    const bool part = p.tile_cols > 0 && st.k_slice > 0;
    constexpr int kBufs = kStagingBytes / kWarps / kBoxBytes;
    const uint32_t buf = staging + (st.n_issued % kBufs) * kBoxBytes;
    // the last store issued from this buffer must have finished reading it
    if (lane == 0) bulk_wait_group_read<kBufs - 1>();
    __syncwarp();
    if (kAhead && lane == 0 && st.add && st.next_row >= 0 && st.next_row < m_rows && st.next_col + c * 32 < p.n_cols)
      tma_prefetch_3d(tmC, st.next_col + c * 32, p.row_base + st.next_row, 0);
    // row `lane` of the box: 8 chunks of 16 bytes, chunk j stored at position j ^ (row & 7)
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      const uint32_t addr = buf + lane * 128u + (uint32_t((j ^ (lane & 7)) << 4));
      asm volatile("st.shared.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(addr), "f"(v[4 * j]), "f"(v[4 * j + 1]),
                   "f"(v[4 * j + 2]), "f"(v[4 * j + 3])
                   : "memory");
    }
    fence_proxy_async_smem();
    __syncwarp();
    if (lane == 0) {
      if (part) tma_store_3d(tmC, buf, col0 % p.tile_cols, row0 % p.tile_rows, st.k_slice - 1);
      else if (st.add || (p.slice_add && st.k_slice > 0)) tma_reduce_add_3d(tmC, buf, col0, p.row_base + row0, st.k_slice);
      else              tma_store_3d(tmC, buf, col0, p.row_base + row0, st.k_slice);
      bulk_commit_group();
    }
    st.n_issued++;
  }
  __device__ static __forceinline__ void end_unit(const Params&, State&, int, int, int, int) {}
};
using EpiAcc = EpiAccW<4>;

}  // namespace rlh
