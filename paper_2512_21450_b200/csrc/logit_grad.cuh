// One-sweep path: the fp32 logits of a slab become the bf16 gradient with respect to the logits, in the arithmetic of EpiGrad:
//   g_tj = cp_t (p_tj - 1[j = y_t]) + ce_t p_tj (log p_tj + Ent_t),
// with the full-distribution KL that of EpiGradKL, from the fp32 logits of both models:
//   g_tj = cp_t (p_tj - 1[j = y_t]) + cb_t p_tj (log p_tj - log q_tj - KL_t) + ce_t p_tj (log p_tj + Ent_t),
// written in place of the policy logits' upper halves; rows past the slab's valid rows (up to a multiple of 128) and
// columns past V become zero.  4 bytes in (8 with the KL) and 2 out per entry, nothing read twice: bound by memory.
// The work is done by extra warps of the dH kernel (EpiAccFed), which read and write DRAM while the tensor cores
// multiply what they have finished, or by a kernel of its own (logit_grad_kernel) where dH does not come next, where that does
// not pay (feed_pays) and with the full KL.
#pragma once
#include <type_traits>

#include "kl_epilogues.cuh"

namespace rlh {

struct LogitGradParams {
  uint16_t* slab;          // [slab rows][ld] upper halves of the logits, then the gradient
  const uint16_t* lo;      // lower halves
  int ld;                  // multiple of 256
  int V;
  int slab_cap, slab_one, slab_index;
  const int* tokens_c;     // per compact row, as the arrays below
  const float* lse;
  const float* ent;
  const float* cp;
  const float* ce;
  // full-distribution KL: the reference's logits
  const float* zr;
  const float* lse_ref;
  const float* kl;
  const float* cb;
};
// For a dH pass that may do it itself: its shape and grid.
struct FeedParams : LogitGradParams {
  GemmShape dh;
  int cg, workers;
  unsigned* ticket;        // jobs handed out; 0 when the launch starts
  unsigned* ready;         // [row tiles][column chunks]: jobs of the chunk that are done
};
// Words of the ticket (its own 16 bytes) and of the counters behind it.
inline size_t feed_words(long long rows, long long ld) {
  return (size_t)(4 + ((rows + BM - 1) / BM * ((ld + kFeedCols - 1) / kFeedCols) + 3) / 4 * 4);
}

// Whether dH pays for forming its operand itself, known once the rows are counted.  While its tiles run in whole waves, and
// where helpers are many or none; a few helpers ask for the ends of nearly all tiles at once, beside the parts, and where
// parts are many and short the start shows.  A whole step,
// apart against fed, sustained at the board's power limit, d = 2048: 4.71 / 7.78 / 9.09 / 11.06 ms against 4.51 / 7.60 / 8.82 / 10.75 at
// 2600 / 4864 / 5632 / 6912 rows (30 helpers, waves), level at 3500 (18 helpers: 5.93 / 5.90), but 3.40 / 6.66 against 3.51 / 6.78 at 2000 /
// 4096 (10 helpers); 45.3 against 44.4 at 16896 rows, d = 3584; 16.41 against 16.12 at 16896 rows, d = 1024; in 6 parts 1.49 against 1.47 at
// 1000 rows, d = 1536, in 9 and 12 1.24 against 1.26 at 447, d = 2048, and 0.89 against 0.90 at 700, d = 1024.
__host__ __device__ inline bool feed_pays(const GemmExtents& ex, int n_workers) {
  return ex.stream_k == 0 || ex.n_units > ex.cut || (ex.cut_len == 0 && ex.cut_parts <= 8) ||
         (ex.cut_len > 0 && (n_workers - ex.cut * ex.cut_parts) * 4 >= n_workers);
}

// The order in which (row tile, column chunk) pairs are worked on: that in which the dH pass reads them.  Its units of one
// wave walk their columns side by side, so the row tiles of a wave are taken together, one column chunk after the other
// (a row tile belongs to the wave that first needs it); tiles cut along K start at several columns at once, and so do
// theirs.  Any order is correct: whoever needs a chunk waits for it, and a job that was handed out never waits.
struct FeedOrder {
  int m_tiles, chunks, cg;
  int n_ranges, n_workers;    // units per row tile of cg * 128 rows, units per wave
  int plain_tiles;            // row tiles that a whole tile of dH needs first; the cut ones follow
};
__host__ __device__ inline FeedOrder feed_order(const GemmExtents& ex, int rows, int ld, int cg, int n_workers) {
  FeedOrder o;
  o.m_tiles = (rows + BM - 1) / BM;
  o.chunks = (ld + kFeedCols - 1) / kFeedCols;
  o.cg = cg;
  o.n_ranges = ex.n_ranges;
  o.n_workers = n_workers;
  const int plain = ex.n_units - ex.cut;
  o.plain_tiles = (plain + ex.n_ranges - 1) / ex.n_ranges * cg;
  if (o.plain_tiles > o.m_tiles) o.plain_tiles = o.m_tiles;
  return o;
}
// Cut tiles are read from several places of K on: parts[g & 1] chunks at least from the start of each range g on.
// Even ranges are the parts' own, odd ones (only where helpers work) the ends that helpers do.
__host__ __device__ inline int feed_cut_chunk(const GemmExtents& ex, const FeedOrder& o, int g) {
  const int per = ex.cut_len > 0 ? 2 : 1, s = g / per;
  return s < ex.cut_parts ? (cut_begin(ex, s) + (g % per ? ex.cut_len : 0)) * BK / kFeedCols : o.chunks;
}
// Pair number q of m_tiles * chunks.
__host__ __device__ inline void feed_pair(const GemmExtents& ex, const FeedOrder& o, int q, int& tile, int& chunk) {
  const int t = q / o.chunks;   // as if the tiles were taken one by one: in the right wave
  if (t < o.plain_tiles) {
    const int wave = t / o.cg * o.n_ranges / o.n_workers;
    const int lo = (wave * o.n_workers + o.n_ranges - 1) / o.n_ranges * o.cg;
    int hi = ((wave + 1) * o.n_workers + o.n_ranges - 1) / o.n_ranges * o.cg;
    if (hi > o.plain_tiles) hi = o.plain_tiles;
    const int r = q - lo * o.chunks;
    tile = lo + r % (hi - lo);
    chunk = r / (hi - lo);
    return;
  }
  const int n = o.m_tiles - o.plain_tiles, r = q - o.plain_tiles * o.chunks, pos = r / n;
  tile = o.plain_tiles + r % n;
  // a chunk of every range in turn, then of the longer ones, then what is left
  const int S = ex.cut_parts, per = ex.cut_len > 0 ? 2 : 1;
  if (S < 1) { chunk = pos; return; }
  const int len = ex.k_blocks / S, each[2] = {(per > 1 ? ex.cut_len : len) * BK / kFeedCols, (per > 1 ? len - ex.cut_len : 0) * BK / kFeedCols};
  const int both = each[0] < each[1] ? each[0] : each[1], more = each[0] + each[1] - 2 * both;
  if (pos < 2 * S * both) { chunk = feed_cut_chunk(ex, o, pos % (2 * S)) + pos / (2 * S); return; }
  int left = pos - 2 * S * both;
  if (left < S * more) { chunk = feed_cut_chunk(ex, o, left % S * per + (each[1] > each[0])) + both + left / S; return; }
  left -= S * more;
  for (int g = 0; g < S * per; ++g) {
    const int c0 = feed_cut_chunk(ex, o, g) + each[g % per], rest = feed_cut_chunk(ex, o, g + 1) - c0;
    if (left < rest) { chunk = c0 + left; return; }
    left -= rest;
  }
  chunk = o.chunks - 1;   // not reached
}

// What a row brings to its entries: log-sum-exp; cp, ce and the terms that do not depend on the column; with the KL the
// reference's log-sum-exp and cb.  valid: not a row of padding.
struct GradRow {
  float lse, cp, ce, rest, lse_ref, cb;
  int y;
  bool valid;
};
// Eight entries from column c on: halves of the logits (and the reference's logits) to the gradient.
template <bool KL>
__device__ __forceinline__ uint4 grad_words(const GradRow& r, const uint4& h, const uint4& l, const float (&zr)[8], int c, int V) {
  const uint32_t hw[4] = {h.x, h.y, h.z, h.w}, lw[4] = {l.x, l.y, l.z, l.w};
  const float k_lp = r.cb + r.ce;   // coefficient of log p_j
  float g[8];
#pragma unroll
  for (int j = 0; j < 8; ++j) {
    const float z = __uint_as_float(__byte_perm(lw[j / 2], hw[j / 2], j & 1 ? 0x7632 : 0x5410));
    if constexpr (KL) {
      const float lp = z - r.lse;
      g[j] = ex2_approx(lp * kLog2e) * (fmaf(k_lp, lp, r.rest) - r.cb * (zr[j] - r.lse_ref));
    } else {
      const float e = ex2_approx(fmaf(z, kLog2e, -r.lse * kLog2e));
      g[j] = r.ce == 0.f ? e * r.cp : e * fmaf(r.ce, z - r.lse, r.rest);
    }
  }
  const unsigned rel = (unsigned)(r.y - c);
  if (rel < 8u) {
#pragma unroll
    for (int j = 0; j < 8; ++j) g[j] = rel == (unsigned)j ? g[j] - r.cp : g[j];
  }
  if (!r.valid || c + 8 > V) {
#pragma unroll
    for (int j = 0; j < 8; ++j) g[j] = r.valid && c + j < V ? g[j] : 0.f;
  }
  uint32_t o[4];
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    const __nv_bfloat162 v = __floats2bfloat162_rn(g[2 * j], g[2 * j + 1]);
    o[j] = *reinterpret_cast<const uint32_t*>(&v);
  }
  return make_uint4(o[0], o[1], o[2], o[3]);
}
// Row i of the compact arrays.
template <bool KL>
__device__ __forceinline__ GradRow grad_row(const LogitGradParams& p, int i) {
  GradRow r = {p.lse[i], p.cp[i], p.ce[i], 0.f, 0.f, 0.f, p.tokens_c[i], true};
  if (KL) {
    r.lse_ref = p.lse_ref[i];
    r.cb = p.cb[i];
    r.rest = r.cp + r.ce * p.ent[i] - r.cb * p.kl[i];
  } else {
    r.rest = fmaf(r.ce, p.ent[i], r.cp);
  }
  return r;
}

// A launch of its own.  A warp takes kVecs * 256 consecutive columns of one row, all its 16-byte loads in flight before the
// first is used.  151936 columns: 17 / 45 / 146 / 556 / 986 us at 64 / 276 / 1000 / 4000 / 6912 rows, 5.5 TB/s at 276 and 6.3-6.6
// from 600 on (two pairs in flight 17 / 49 / 150 / 590 / 1089, eight 17 / 49 / 148 / 565 / 1012).  With the KL, four words per output:
// 68 / 232 / 462 us at 276 / 1000 / 2000 rows (one 256-column step: 72 / 247 / 481).
template <bool KL>
constexpr int kGradVecs = KL ? 2 : 4;
// Params: FeedParams where the dH pass may do it.
template <bool KL, class Params>
__global__ void __launch_bounds__(256) logit_grad_kernel(const Params p, const DevStatus* st) {
  chain_begin();
  constexpr int kVecs = kGradVecs<KL>;
  if constexpr (std::is_same<Params, FeedParams>::value) {
    if (feed_pays(gemm_extents(p.dh, st->n_valid, p.cg, p.workers), p.workers)) return;
  }
  int off, rows;
  slab_extent(st->n_valid, p.slab_cap, p.slab_one, p.slab_index, off, rows);
  const int rows_pad = (rows + 127) / 128 * 128;
  const int units_per_row = (p.ld + (kVecs * 256) - 1) / (kVecs * 256);
  const long long n_units = (long long)rows_pad * units_per_row;
  const int lane = threadIdx.x & 31;
  const long long n_warps = (long long)gridDim.x * (blockDim.x >> 5);
  for (long long u = (long long)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); u < n_units; u += n_warps) {
    const int r = (int)(u / units_per_row);
    const int c0 = (int)(u - (long long)r * units_per_row) * (kVecs * 256);
    const size_t at = (size_t)r * p.ld + c0;
    uint4* base = reinterpret_cast<uint4*>(p.slab + at) + lane;
    if (r >= rows) {
#pragma unroll
      for (int k = 0; k < kVecs; ++k)
        if (c0 + k * 256 < p.ld) base[k * 32] = make_uint4(0, 0, 0, 0);
      continue;
    }
    const uint4* low = reinterpret_cast<const uint4*>(p.lo + at) + lane;
    const float4* ref = reinterpret_cast<const float4*>(p.zr + (KL ? at : 0)) + 2 * lane;
    uint4 h[kVecs], l[kVecs];
    float4 z0[KL ? kVecs : 1], z1[KL ? kVecs : 1];
#pragma unroll
    for (int k = 0; k < kVecs; ++k)
      if (c0 + k * 256 < p.ld) {
        h[k] = base[k * 32];
        l[k] = __ldcs(low + k * 32);
        if (KL) {
          z0[k] = __ldcs(ref + k * 64);
          z1[k] = __ldcs(ref + k * 64 + 1);
        }
      }
    const GradRow row = grad_row<KL>(p, off + r);
#pragma unroll
    for (int k = 0; k < kVecs; ++k) {
      if (c0 + k * 256 >= p.ld) break;
      const int q = KL ? k : 0;
      const float zr[8] = {z0[q].x, z0[q].y, z0[q].z, z0[q].w, z1[q].x, z1[q].y, z1[q].z, z1[q].w};
      base[k * 32] = grad_words<KL>(row, h[k], l[k], zr, c0 + k * 256 + lane * 8, p.V);
    }
  }
}

// By warps of a tensor-core kernel: the jobs of one of them, as long as there are any.  The words of the next two rows are in
// flight while these are worked on, across jobs.  (Not with the KL: 8 bytes in per entry were too much beside the products, steps level.)
struct LogitGradWarp {
  static constexpr int kStepRows = 2;
  static constexpr int kSteps = kFeedRows / kStepRows;
  static constexpr int kVecs = kFeedCols / 256;    // 16-byte words per lane, row and plane
  struct Words {
    uint4 h[kStepRows][kVecs], l[kStepRows][kVecs];
  };
  struct Job {
    int r0, c0;       // first slab row, first column
    int flag;         // its counter
    GradRow row;      // slab row r0 + lane % kFeedRows
  };
  __device__ static __forceinline__ void load(const FeedParams& p, const Job& j, int step, int lane, Words& w) {
#pragma unroll
    for (int i = 0; i < kStepRows; ++i) {
      const size_t row = (size_t)(j.r0 + step * kStepRows + i) * p.ld;
#pragma unroll
      for (int k = 0; k < kVecs; ++k) {
        // without a branch, which costs the overlap of these loads; past the row's end the words before are loaded again
        const size_t at = row + (j.c0 + k * 256 < p.ld ? j.c0 + k * 256 : j.c0) + lane * 8;
        w.h[i][k] = __ldcs(reinterpret_cast<const uint4*>(p.slab + at));
        w.l[i][k] = __ldcs(reinterpret_cast<const uint4*>(p.lo + at));
      }
    }
  }
  __device__ static __forceinline__ void work(const FeedParams& p, const Job& j, int step, int lane, const Words& w) {
#pragma unroll
    for (int i = 0; i < kStepRows; ++i) {
      const int rj = step * kStepRows + i;
      auto of = [&](float x) { return __shfl_sync(0xffffffffu, x, rj); };
      GradRow row = {of(j.row.lse), of(j.row.cp), of(j.row.ce), of(j.row.rest), 0.f, 0.f, __shfl_sync(0xffffffffu, j.row.y, rj),
                     __shfl_sync(0xffffffffu, (int)j.row.valid, rj) != 0};
#pragma unroll
      for (int k = 0; k < kVecs; ++k) {
        if (j.c0 + k * 256 >= p.ld) break;
        const int c = j.c0 + k * 256 + lane * 8;
        *reinterpret_cast<uint4*>(p.slab + (size_t)(j.r0 + rj) * p.ld + c) = grad_words<false>(row, w.h[i][k], w.l[i][k], {}, c, p.V);
      }
    }
  }
  __device__ static __forceinline__ unsigned draw(const FeedParams& p, int lane) {
    unsigned t = 0;
    if (lane == 0) t = atomicAdd(p.ticket, 1u);
    return __shfl_sync(0xffffffffu, t, 0);
  }
  __device__ static __forceinline__ void open(const FeedParams& p, const GemmExtents& ex, const FeedOrder& o, unsigned t,
                                              int off, int rows, int lane, Job& j) {
    int tile, chunk;
    feed_pair(ex, o, (int)(t / kFeedJobs), tile, chunk);
    j.r0 = tile * BM + (int)(t % kFeedJobs) * kFeedRows;
    j.c0 = chunk * kFeedCols;
    j.flag = tile * o.chunks + chunk;
    const int r = j.r0 + (lane & (kFeedRows - 1));
    j.row = {};
    j.row.y = -1;
    if (r < rows) j.row = grad_row<false>(p, off + r);
  }
  __device__ static __forceinline__ void run(const FeedParams& p, const GemmExtents& ex, const FeedOrder& o, int off, int rows) {
    const int lane = threadIdx.x & 31;
    const unsigned n_jobs = (unsigned)o.m_tiles * o.chunks * kFeedJobs;
    unsigned t = draw(p, lane);
    if (t >= n_jobs) return;
    Job j;
    Words w[2];
    open(p, ex, o, t, off, rows, lane, j);
    load(p, j, 0, lane, w[0]);
    for (;;) {
      t = draw(p, lane);
      Job next = j;
#pragma unroll
      for (int s = 0; s < kSteps; ++s) {
        if (s + 1 < kSteps) {
          load(p, j, s + 1, lane, w[(s + 1) & 1]);
        } else if (t < n_jobs) {
          open(p, ex, o, t, off, rows, lane, next);
          load(p, next, 0, lane, w[(s + 1) & 1]);
        }
        work(p, j, s, lane, w[s & 1]);
      }
      // every lane's stores, then the counter; its reader copies the chunk through the TMA unit
      fence_proxy_async_global();
      __syncwarp();
      if (lane == 0) red_add_release(p.ready + j.flag, 1u);
      if (t >= n_jobs) return;
      j = next;
    }
  }
};

// dH of one slab while its operand G is still being formed: kSideWarps warps of every CTA do the jobs of LogitGradWarp, the
// producer waits for the chunks it is about to load.
struct EpiAccFed : EpiAcc {
  static constexpr int kSideWarps = 9;   // with the one that watches, sixteen warps in all: 128 registers a thread
  static constexpr bool kFeeds = true;
  struct Params : AccParams {
    FeedParams grad;
  };
  __device__ static __forceinline__ void side(const Params& p, const GemmExtents& ex, int cg, int n_workers, int) {
    LogitGradWarp::run(p.grad, ex, feed_order(ex, ex.m_rows, p.grad.ld, cg, n_workers), ex.slab_off, ex.m_rows);
  }
  __device__ static __forceinline__ bool feeds(const Params& p, const GemmExtents& ex, int n_workers) { return feed_pays(ex, n_workers); }
  // Counter of column chunk `chunk` of 128-row tile m
  __device__ static __forceinline__ const unsigned* feed_flag(const Params& p, int m, int chunk) {
    return p.grad.ready + m * ((p.grad.ld + kFeedCols - 1) / kFeedCols) + chunk;
  }
};

}  // namespace rlh
