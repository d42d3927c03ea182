// C ABI of the fused LM-head log-probability + GRPO policy-loss library: argument checks,
// workspace layout, tensor-map construction and the launch sequences.  All arithmetic of the
// path runs in the kernels of gemm_engine.cuh / epilogues.cuh / small_kernels.cuh.
#include <cuda.h>
#include <cuda_runtime.h>

#include <cstdio>
#include <cstring>
#include <mutex>
#include <new>

#include "rlhead.h"
#include "small_kernels.cuh"
#include "cluster_probe.cuh"

using namespace rlh;

typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

constexpr int kProfMax = 1 << 16;   // timed launch groups kept between two rl_profile_read calls
constexpr int kProfKinds = 9;    // 0 logits, 1 dlogits, 2 dH, 3 dW, 4 mask scan, 5 row preparation,
                                 // 6 merge + loss, 7 dH scatter, 8 advantages

struct rl_ctx {
  int device;
  int n_sm;
  cudaStream_t stream;
  DevStatus* dstatus;  // device
  void* ws;
  size_t ws_bytes;
  EncodeTiledFn encode;
  int slab_rows;  // rows of one gradient slab (multiple of 128)
  int slab_cols;  // vocabulary columns of one gradient slab (multiple of 256)
  int slab_auto;  // 1: rl_set_slab_limits() left the slab's shape to the library (whole rows where they fit)
  int cta_group;  // 1: one CTA per 128x256 tile; 2: CTA pairs on 256x256 tiles
  int dh_k_slices;  // upper bound on the K slices of the dH pass (1 = tiles are not cut)
  long long row_group_bytes;  // forward / dlogits: bytes of A panels walked together (0 = all row tiles at once)
  int wide_tiles;   // 1: dH and dW run on 256 x 512 tiles (both accumulators hold one tile)
  int dh_stream_k;  // 1: the dH pass balances its tiles over the SMs by stream-K (needs a second accumulator buffer)
  int grid[3];    // persistent grid for cta_group 1 and 2 (index = cta_group)
  int fixed_scratch;  // 1: the context of rl_token_logprobs_static, whose scratch has a documented size
  int grid_full[3];   // the same before rl_set_max_ctas() capped it
  rl_dw_slab_hook dw_hook;   // called after the launch that completes a slab of dW rows was enqueued
  void* dw_hook_user;
  long long launches;  // kernels launched by this context so far
  // optional per-kernel timing: event pairs around every tensor-core launch, by kernel kind
  int prof_on;
  int prof_used;
  // pipelined host-buffer steps: a copy stream, per-slot events and pinned result words (created on first use)
  cudaStream_t copy_stream;
  cudaEvent_t copy_done[2], step_done[2];
  float* pinned_out[2];
  int slot_busy[2];
  int* prof_kind;                 // [kProfMax], allocated when profiling is first switched on
  cudaEvent_t (*prof_ev)[2];      // [kProfMax][2], events created on first use
};

namespace {

constexpr long long kRowGroupBytes = 36ll << 20;   // A panels walked together by the rows-first passes (L2 is 126 MB)
constexpr int kSlabRowsMax = 32768;        // rows of one gradient slab
// Slab shape when the caller sets none: rows over the WHOLE vocabulary, at most kSlabBytes of them at 4 bytes an entry (8 with
// the full-distribution KL, 2 for a narrow head), and no more than kSlabRowBytes of compact hidden rows.  A row that is complete in the slab
// needs its logits formed only once.  Fewer rows per slab mean more passes over dW (8 bytes per entry and slab, beside 14
// bytes per entry of the slab itself): twice kSlabBytes takes 1.5 % off 16896 rows at d = 2048 and adds 1.3 % to 67244 rows
// at d = 3584.  More rows than L2 keeps make the dW pass re-read them from DRAM (7B-class step: 208 ms with 85 MB of rows
// per slab, 200 with 57; d = 2560: 178 ms with 70 MB, 173 with 60).  Below kSlabRowsMin rows a slab is cut by columns.
constexpr long long kSlabBytes = 1ll << 32;
constexpr long long kSlabRowBytes = 58ll << 20;
constexpr int kSlabRowsMin = 2048;
// Device words a context owns besides the workspace: the status record, a few scalars of the small kernels
// (byte 64: batch statistics, 96: longest response, kTicketOffset: ticket counters), the valid-row
// counts of rl_token_loss and, behind them, its block partials.
constexpr int kTokenLossBlocks = 1024;
constexpr size_t kCountOffset = 256;
constexpr size_t kSumsOffset = kCountOffset + kCountBlocks * sizeof(unsigned);
constexpr size_t kStatusBytes = kSumsOffset + (size_t)kTokenLossBlocks * kLossSums * sizeof(double);
constexpr int kAdvRowsMinGroups = 2048;     // from this many groups on, GRPO advantages run one thread per group
// Rows up to which the broadcast works the advantages out itself, once per thread and response it meets: one launch of 8.6-11.2 us
// in place of two of 10.7-15.6 up to 2^19 rows; at 2^20 / 2^21 rows 8.7-36 / 8.7-99 against 10.6-20 / 10.6-21 (16 to 2000 groups of 8 to 32).
constexpr int64_t kFusedAdvRows = 1 << 19;
constexpr int kWideGain = 96;              // time of a 256 x 512 tile, in % of two 256 x 256 tiles of the same K
constexpr int kMergeBlocks = 512;          // blocks per merge launch when a call makes several (kLossThreads threads each)
constexpr size_t kTicketOffset = 192;      // in the device block: blocks that are done, of the loss kernels of a step (cleared by
                                           // its row preparation) and of rl_token_loss (one launch: 0 whenever none runs)
constexpr int kDhSplitMax = 4;             // most K slices (separate fp32 accumulators) of the dH pass
constexpr int kSlabColsMax = 148 * 256;    // vocabulary columns of one gradient slab (148 tiles of 256: two per SM pair)

inline size_t align_up(size_t x, size_t a) { return (x + a - 1) / a * a; }

// fp32 accumulator buffers of the dH pass: one per K slice, or two when stream-K balancing is on
inline bool dh_uses_stream_k(const rl_ctx* c) { return c->dh_stream_k && c->dh_k_slices == 1; }
inline int dh_buffers(const rl_ctx* c) { return dh_uses_stream_k(c) ? 2 : c->dh_k_slices; }
// The merge of `rows` rows with at most `ranges` column ranges each (0: nothing to merge): a thread per row, else eight warps per
// 32 rows.  Merge and loss, thread against eight warps: 2 ranges 10.6 / 10.6 / 10.6 / 27 us against 12.1 / 15.0 / 20.9 / 101 at 8 / 16 /
// 32 / 524 thousand rows, 16 ranges 12.7 / 12.7 / 13.1 / 20.9 against 12.7 / 16.8 / 22.9 / 39.4 at 8 / 16 / 32 / 131 thousand, 75 ranges
// 14.1 / 22.9 / 25.0 / 24.8 / 39.5 against 11.9 / 12.7 / 18.8 / 26.6 / 42.7 at 4 / 8 / 16 / 32 / 65 thousand.
inline bool merge_by_thread(int64_t rows, int ranges) { return rows >= (ranges <= kMaxSplit ? 8192 : 32768) || ranges == 0; }
// Its blocks; all launches of a call together have at most kMergeBlocks * (1 + slabs).
inline int merge_blocks(int64_t rows, int slabs, int ranges) {
  const int64_t per = merge_by_thread(rows, ranges) ? kLossThreads : 32;
  const int64_t n = (rows + per - 1) / per, most = slabs > 1 ? kMergeBlocks : 2 * kMergeBlocks;
  return (int)(n < most ? n : most);
}
// Neither option set: the tiles of the dH pass's ragged last wave are cut into parts that lie in slots.
inline bool dh_cuts_tiles(const rl_ctx* c) { return !c->dh_stream_k && c->dh_k_slices == 1; }
// Full-distribution KL: two single-product passes that leave 6 bytes per logit pair behind, or two-product tiles formed
// twice.  The former trades 4 d + 4 d_ref tensor flops for 14 bytes of traffic per entry.  4096 rows, V = 151936: logits and
// their gradient take 3.3 / 3.5 / 4.9 / 8.3 ms against 2.5 / 4.3 / 8.2 / 17.2 ms at d = d_ref = 512 / 1024 / 2048 / 4096.
constexpr int64_t kKlSweepMinK = 1536;   // d + d_ref
inline bool kl_one_sweep(int64_t d, int64_t d_ref) { return d_ref > 0 && d + d_ref >= kKlSweepMinK; }
// Keeping the logits of a model takes 8 bytes of traffic per entry and a heavier epilogue, forming them again 2 d flops.
// Logits and their gradient, 6912 rows x 151936 words, kept against formed twice: 1.92 / 2.38 / 2.75 / 2.90 / 3.04 / 3.14 /
// 3.36 ms against 1.40 / 1.98 / 2.62 / 2.96 / 3.17 / 3.50 / 3.66 at d = 256 / 512 / 768 / 896 / 960 / 1024 / 1152.
constexpr int64_t kSweepMinK = 896;
// Bytes of a slab entry: fp32 logits that wait for the loss (two of them with the full KL) and leave room for the bf16
// gradient, or the gradient alone.
inline int slab_entry_bytes(int64_t d, int64_t d_ref) {
  return d_ref > 0 ? (kl_one_sweep(d, d_ref) ? 8 : 2) : (d >= kSweepMinK ? 4 : 2);
}
// Entries of a slab from which on dH may form its operand itself (feed_pays): below, the start of the feed shows, and a larger launch
// that does not feed 1 % of a call.  100 and 300 rows x 151936 words, d = 2048, 1 % slower and level; 256 rows of 40000 words 169 / 188 us.
constexpr long long kFeedEntries = 128 << 20;
// A narrow head keeps them too while they stay in L2, and up to 128 rows, where the logit pass is a stream of W: a whole call,
// kept against formed twice, 53.8 / 77.3 / 113 us against 58.6 / 79.4 / 106 at d = 256, 4 / 34 / 67 MB of logits (4096 words), 63.5 / 77.5 /
// 100.5 against 68.3 / 77.3 / 96.9 (16384 words, 17 / 34 / 67 MB), 188 / 192 / 253 against 215 / 200 / 232 at 64 / 128 / 256 rows of 151936 words.
constexpr size_t kKeepBytes = 40u << 20;
constexpr int kKeepRows = 128;
// 256 x 512 tiles: fewer operand bytes per flop, but a tile's epilogue does not overlap the next main loop, and a last
// tile that is half empty costs as much as a full one.  For dH, whose K is the vocabulary: 7 % of the pass (8.59 / 53.1 /
// 58.9 ms against 9.35 / 57.3 / 63.1 at d = 2048 / 2560 / 3584).  Not for dW, whose K is a slab of rows: 256 x 256 tiles
// take 54.5 / 62.1 / 133.6 ms against 56.3 / 63.7 / 137.0 at 10 / 8 / 14 thousand rows per slab.
inline bool use_wide(const rl_ctx* c, int64_t d) {
  const int64_t wide = (d + 2 * BN - 1) / (2 * BN) * 2, square = (d + BN - 1) / BN;
  return c->wide_tiles && c->cta_group == 2 && wide * kWideGain <= square * 100;
}
// Rows of a call up to which dW runs with eight epilogue warps (EpiAccW).  dW of 151936 words, d = 2048, four warps against eight, adding
// 577 / 449, 602 / 517, 604 / 572, 634 / 641 us at 300 / 512 / 640 / 768 rows, storing 368 / 336, 414 / 419, 515 / 504, 519 / 535; d = 3584, adding
// 1021 / 845, 1059 / 925, 1047 / 1018, 1112 / 1099: level at 700.  By the rows of the call, since how many are valid only the device knows: 300 valid
// rows among 1024 keep four (600 against 474 us adding).
constexpr int64_t kFewRows = 640;
// Whether dW's launch writes dH to the caller's rows as well (EpiAccScatter), or a launch of its own behind it does.  Four warps a CTA
// copy at 1.5 TB/s, a launch of its own at 4.7; beside, the copy is hidden as far as dW lasts, which is as long as the waves of its
// tiles: with few words and many columns it ends first.  Per row dW takes 7 ns a wave, a copy beside it 4.1 ps a column, one behind it
// 1.3: level near 2500 columns a wave.  A call, beside against behind: d = 3584, 16384 rows, 256 / 600 / 1000 / 1500 / 2000 words (1, 1, 1, 2,
// 2 waves) 487 / 560 / 592 / 708 / 826 us against 441 / 512 / 541 / 723 / 845, d = 4096, 1000 / 2000 / 3000 (1, 2, 3) 746 / 1008 / 1263 against
// 675 / 999 / 1318, d = 2048, 8192 rows, 256 / 1000 142 / 182 against 158 / 190.  Up to a thousand rows the launch saved is worth as much.
inline bool dH_beside_dW(const rl_ctx* c, int64_t T, int64_t d, int64_t cols) {
  const int64_t tiles = (d + BN - 1) / BN * ((cols + BN - 1) / BN) * 2;   // of 128 rows
  const int64_t waves = (tiles + c->grid[c->cta_group] - 1) / c->grid[c->cta_group];
  return T <= 1024 || d < 2000 * waves + 64;
}
// Width of a dH tile, and bytes of the slots its parts may need (two per worker).
inline int dh_tile_cols(const rl_ctx* c, int64_t d) { return use_wide(c, d) ? 2 * BN : BN; }
inline size_t dh_slot_bytes(const rl_ctx* c, int64_t d) {
  const int workers = c->grid_full[c->cta_group] / c->cta_group;
  return (size_t)2 * workers * BM * c->cta_group * dh_tile_cols(c, d) * 4;
}

struct WsLayout {
  int Tpad, Ts, Vs;   // rows; most rows and columns of a slab
  int Tc;             // rows of a slab when there are several
  size_t scan_counts, row_map, tokens_c, logp_c, lse_c, ent_c, cp_c, ce_c, partials, block_sums, Hc, G, dH_acc, staging, total;
  size_t row_pos;                                    // position of every row in the row map (T > kPrepRows)
  bool keeps_logits;                                 // one-sweep path: G's place first holds the upper halves of fp32 logits,
                                                     // the plane behind it their lower halves
  int part_ranges;                                   // column ranges per row that the partials have room for
  size_t dH_slots;                                   // parts of cut dH tiles (0: none)
  size_t feed, feed_bytes;                           // ticket and counters of the gradient jobs (logits are kept)
  int n_row_slabs;
  size_t Hc_ref, partials2, lse_ref_c, kl_c, cb_c;   // only with a reference model (full KL)
  size_t zr;                                         // the reference's logits of the slab (one-sweep form)
};

// Reference-model operands of the full-distribution KL (all NULL / 0 when it is not used).
struct KlRef {
  const void* H_ref;
  int64_t ldH_ref;
  const void* W_ref;
  int64_t ldW_ref;
  int64_t d_ref;
};

// Device copies of one step's host inputs (H, tokens, old, ref, adv, mask, rewards, offsets) and its result words.
struct HostStage {
  void* H;
  int32_t* tok;
  float *old_lp, *ref_lp, *adv;
  uint8_t* mask;
  float* out;       // [16]: loss, 7 unused, 8 metrics
  float *rew, *advseq;
  int32_t* off;
};
inline size_t carve_stage(char* base, int64_t T, int64_t d, HostStage* hs) {
  size_t o = 0;
  auto take = [&](size_t bytes) { size_t at = o; o = align_up(o + bytes, 1024); return base ? base + at : nullptr; };
  HostStage h;
  h.H = take((size_t)T * d * 2);
  h.tok = reinterpret_cast<int32_t*>(take((size_t)T * 4));
  h.old_lp = reinterpret_cast<float*>(take((size_t)T * 4));
  h.ref_lp = reinterpret_cast<float*>(take((size_t)T * 4));
  h.adv = reinterpret_cast<float*>(take((size_t)T * 4));
  h.mask = reinterpret_cast<uint8_t*>(take((size_t)T));
  h.out = reinterpret_cast<float*>(take(64));
  h.rew = reinterpret_cast<float*>(take((size_t)T * 4));
  h.advseq = reinterpret_cast<float*>(take((size_t)T * 4));
  h.off = reinterpret_cast<int32_t*>(take((size_t)(T + 1) * 4));
  if (hs) *hs = h;
  return o;
}

// host_slots > 0 adds room for that many sets of host-call inputs behind the scratch proper.
// by_columns: slabs of many rows and some columns even where whole rows would fit, for calls that form the logits twice
// whatever the slab's shape is: fewer, longer row slabs for dW (sequence-level ratio against the library that knew column slabs
// only: 74 thousand rows at d = 3584 1.4 % slower with slabs of whole rows, up to 2 % faster by columns; 37 thousand at d = 2048 level).
WsLayout ws_layout(const rl_ctx* c, int64_t T, int64_t d, int64_t V, int host_slots, int64_t d_ref = 0, bool by_columns = false) {
  WsLayout L;
  L.Tpad = (int)align_up((size_t)(T > 0 ? T : 1), 128);
  const int Vpad = (int)align_up((size_t)V, 256);
  long long rows = c->slab_rows, one = 0;
  L.Vs = Vpad < c->slab_cols ? Vpad : c->slab_cols;
  if (c->slab_auto && !by_columns) {
    // as many rows as kSlabBytes allows, and no more than keep the compact rows, which the dW pass reads once per row
    // panel of dW, in L2 beside the streamed slab
    long long whole = kSlabBytes / slab_entry_bytes(d, d_ref) / Vpad / 256 * 256;
    long long resident = kSlabRowBytes / (d * 2) / 256 * 256;
    if (resident < kSlabRowsMin) resident = kSlabRowsMin;
    if (whole >= kSlabRowsMin) {   // whatever T is: a smaller batch must not need more than a larger one
      if (whole > kSlabRowsMax) whole = kSlabRowsMax;
      rows = whole < resident ? whole : resident;
      one = whole < resident * 3 / 2 ? whole : resident * 3 / 512 * 256;
      L.Vs = Vpad;
    }
  }
  if (one < rows) one = rows;
  L.Ts = L.Tpad < one ? L.Tpad : (int)one;
  L.Tc = L.Tpad < rows ? L.Tpad : (int)rows;
  L.n_row_slabs = L.Tpad <= L.Ts ? 1 : (L.Tpad + L.Tc - 1) / L.Tc;
  size_t o = 0;
  size_t n_part_ranges = kMaxSplit, n_partials;
  auto take = [&](size_t bytes) { size_t at = o; o = align_up(o + bytes, 1024); return at; };
  L.scan_counts = take(((size_t)L.Tpad / 4096 + 2) * 4);
  L.row_map = take((size_t)L.Tpad * 4);
  L.row_pos = take(T > kPrepRows ? (size_t)T * 4 : 0);
  L.tokens_c = take((size_t)L.Tpad * 4);
  L.logp_c = take((size_t)L.Tpad * 4);
  L.lse_c = take((size_t)L.Tpad * 4);
  L.ent_c = take((size_t)L.Tpad * 4);
  L.cp_c = take((size_t)L.Tpad * 4);
  L.ce_c = take((size_t)L.Tpad * 4);
  {
    // one float4 per (column range, row): at most kMaxSplit ranges, or one per kFwdRange column tiles; with few rows
    // enough ranges to give every SM a unit
    const size_t tiles = (size_t)((V + BN - 1) / BN);
    const size_t by_range = (tiles + kFwdRange - 1) / kFwdRange;
    n_part_ranges = by_range > (size_t)kMaxSplit ? by_range : (size_t)kMaxSplit;
    n_partials = n_part_ranges * L.Tpad;
    if (!c->fixed_scratch) {
      const size_t most = tiles < (size_t)c->n_sm ? tiles : (size_t)c->n_sm, room = (size_t)c->n_sm * 512;
      const size_t fill = most * L.Tpad < room ? most : room / L.Tpad;
      if (n_part_ranges < fill) n_part_ranges = fill;
      // (sized by the room, not by the whole number of ranges that fit it, so that the size does not fall as T grows)
      const size_t n = most * L.Tpad < room ? most * L.Tpad : room;
      if (n_partials < n) n_partials = n;
    }
    L.part_ranges = (int)n_part_ranges;
    L.partials = take(n_partials * sizeof(float4));
  }
  L.block_sums = take((size_t)kMergeBlocks * (1 + L.n_row_slabs) * kLossSums * sizeof(double));
  L.Hc = take((size_t)L.Tpad * d * 2);
  const size_t entries = (size_t)L.Ts * L.Vs;
  const bool narrow = d_ref == 0 && d < kSweepMinK;
  const bool small = narrow && L.n_row_slabs == 1 && (L.Tpad <= kKeepRows || entries * 4 <= kKeepBytes);
  L.keeps_logits = L.Vs == Vpad && (slab_entry_bytes(d, d_ref) >= 4 || small);
  size_t slab = entries * (L.keeps_logits ? 4 : 2);
  // (so that the size does not fall where a batch gets too large for its logits to be kept)
  if (narrow && L.Vs == Vpad && slab < kKeepBytes) slab = entries * 4 < kKeepBytes ? entries * 4 : kKeepBytes;
  // what run_forward() touches lies before this point (without a reference model)
  L.G = take(slab);
  L.dH_acc = take((size_t)dh_buffers(c) * L.Ts * d * 4);
  L.dH_slots = dh_cuts_tiles(c) && L.Vs == Vpad ? take(dh_slot_bytes(c, d)) : 0;
  L.feed_bytes = L.keeps_logits ? feed_words(L.Ts, L.Vs) * 4 : 0;
  L.feed = take(L.feed_bytes);
  L.Hc_ref = L.partials2 = L.lse_ref_c = L.kl_c = L.cb_c = L.zr = 0;
  if (d_ref > 0) {
    L.Hc_ref = take((size_t)L.Tpad * d_ref * 2);
    L.partials2 = take(n_partials * sizeof(float4));
    L.lse_ref_c = take((size_t)L.Tpad * 4);
    L.kl_c = take((size_t)L.Tpad * 4);
    L.cb_c = take((size_t)L.Tpad * 4);
    if (L.keeps_logits) L.zr = take((size_t)L.Ts * L.Vs * 4);
  }
  L.staging = o;
  o += (size_t)host_slots * carve_stage(nullptr, T, d, nullptr);
  L.total = o;
  return L;
}

// Workspace of any call without a reference model: a loss per response may need either shape.
size_t ws_bytes(const rl_ctx* c, int64_t T, int64_t d, int64_t V) {
  const WsLayout L = ws_layout(c, T, d, V, 0);
  const size_t twice = L.n_row_slabs > 1 ? ws_layout(c, T, d, V, 0, 0, true).total : 0;
  return twice > L.total ? twice : L.total;
}

// K-major operand: global tensor [rows, k] with k contiguous, row stride ld elements.
bool map_kmajor(rl_ctx* c, CUtensorMap* m, const void* base, uint64_t rows, uint64_t k, uint64_t ld,
                uint32_t box_rows) {
  cuuint64_t dims[2] = {k, rows};
  cuuint64_t strides[1] = {ld * 2};
  cuuint32_t box[2] = {64, box_rows};
  cuuint32_t es[2] = {1, 1};
  return c->encode(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(base), dims, strides, box, es,
                   CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                   CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}
// MN-major operand: global tensor [k, mn] with mn contiguous (a multiple of 64), row stride ld.
// Seen by TMA as {64, k, mn/64} so that one box {64, 64, chunks} fetches `chunks` 64-wide panels.
bool map_mnmajor(rl_ctx* c, CUtensorMap* m, const void* base, uint64_t k_rows, uint64_t mn, uint64_t ld,
                 uint32_t chunks) {
  cuuint64_t dims[3] = {64, k_rows, mn / 64};
  cuuint64_t strides[2] = {ld * 2, 128};
  cuuint32_t box[3] = {64, 64, chunks};
  cuuint32_t es[3] = {1, 1, 1};
  return c->encode(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void*>(base), dims, strides, box, es,
                   CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                   CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// fp32 output seen by the accumulate epilogue: {cols, rows, slices} with 32x32 boxes, 128-byte
// swizzled in shared memory.  slices > 1: identical [rows, ld] buffers slice_rows rows apart.
bool map_out_f32(rl_ctx* c, CUtensorMap* m, const float* base, uint64_t rows, uint64_t cols, uint64_t ld,
                 uint64_t slices, uint64_t slice_rows) {
  cuuint64_t dims[3] = {cols, rows, slices};
  cuuint64_t strides[2] = {ld * 4, slice_rows * ld * 4};
  cuuint32_t box[3] = {32, 32, 1};
  cuuint32_t es[3] = {1, 1, 1};
  return c->encode(m, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 3, const_cast<float*>(base), dims, strides, box, es,
                   CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                   CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// bf16 [rows, cols] slab written by the dlogits epilogue in 32-row x 64-column boxes.
bool map_out_bf16(rl_ctx* c, CUtensorMap* m, const void* base, uint64_t rows, uint64_t cols, uint64_t ld) {
  cuuint64_t dims[2] = {cols, rows};
  cuuint64_t strides[1] = {ld * 2};
  cuuint32_t box[2] = {64, 32};
  cuuint32_t es[2] = {1, 1};
  return c->encode(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(base), dims, strides, box, es,
                   CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                   CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// The slab's two 16-bit planes of fp32 logits, rows * ld elements apart, written by the logit pass in 32 x 32 boxes, 64-byte swizzled.
bool map_out_planes(rl_ctx* c, CUtensorMap* m, const void* base, uint64_t rows, uint64_t ld) {
  cuuint64_t dims[3] = {ld, rows, 2};
  cuuint64_t strides[2] = {ld * 2, rows * ld * 2};
  cuuint32_t box[3] = {32, 32, 1};
  cuuint32_t es[3] = {1, 1, 1};
  return c->encode(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void*>(base), dims, strides, box, es,
                   CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_64B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                   CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// Dynamic shared memory of an instantiation: a constant of the build, known once its static size was asked for.
template <class Epi, int A_MN, int B_MN, int CG, int MODE>
int g_smem_bytes = 0;
template <class Epi, int A_MN, int B_MN, int CG, int MODE>
cudaError_t set_smem_attr_one() {
  cudaFuncAttributes fa;
  cudaError_t e = cudaFuncGetAttributes(&fa, gemm_kernel<Epi, A_MN, B_MN, CG, MODE>);
  if (e != cudaSuccess) return e;
  const int bytes = gemm_smem_bytes<CG, MODE, Epi::kStagingBytes>((int)fa.sharedSizeBytes);
  g_smem_bytes<Epi, A_MN, B_MN, CG, MODE> = bytes;
  return cudaFuncSetAttribute(gemm_kernel<Epi, A_MN, B_MN, CG, MODE>, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
}
// square tiles, single CTAs and CTA pairs
template <class Epi, int A_MN, int B_MN>
cudaError_t set_smem_attr() {
  cudaError_t e = set_smem_attr_one<Epi, A_MN, B_MN, 1, kTileSquare>();
  return e != cudaSuccess ? e : set_smem_attr_one<Epi, A_MN, B_MN, 2, kTileSquare>();
}
template <class Epi>
cudaError_t set_smem_attr_dual() {
  cudaError_t e = set_smem_attr_one<Epi, 0, 0, 1, kTileDual>();
  return e != cudaSuccess ? e : set_smem_attr_one<Epi, 0, 0, 2, kTileDual>();
}

// Rows of B that one CTA stages per k-slice (box height of a K-major B map) and the number of
// 64-wide panels of an MN-major B map, for the context's CTA grouping.
inline uint32_t b_box_rows(int cg) { return BN / cg; }
inline uint32_t b_box_rows(const rl_ctx* c) { return b_box_rows(c->cta_group); }
inline uint32_t b_box_panels(const rl_ctx* c) { return BN / 64 / c->cta_group; }

// CTAs per row tile of the passes that form logits: a pair would spend half its tensor work on padding when at most 128
// rows exist, and with so few rows the pass is a stream of W.
inline int fwd_cta_group(const rl_ctx* c, const WsLayout& L) { return L.Tpad <= BM ? 1 : c->cta_group; }

// Optional timing of a group of launches: event pair on the context's stream, tagged with a kind.
int prof_begin(rl_ctx* c, int kind) {
  if (!(c->prof_on && c->prof_ev && kind >= 0 && kind < kProfKinds && c->prof_used < kProfMax)) return -1;
  const int i = c->prof_used;
  for (int e = 0; e < 2; ++e)
    if (!c->prof_ev[i][e]) cudaEventCreate(&c->prof_ev[i][e]);
  cudaEventRecord(c->prof_ev[i][0], c->stream);
  return i;
}
void prof_end(rl_ctx* c, int i, int kind) {
  if (i < 0) return;
  cudaEventRecord(c->prof_ev[i][1], c->stream);
  c->prof_kind[i] = kind;
  c->prof_used = i + 1;
}

// One kernel launch on the context's stream that may be scheduled while the launch before it still runs (chain_begin()).
template <class... P, class... A>
void launch(rl_ctx* c, void (*kernel)(P...), int grid, int block, A&&... args) {
  cudaLaunchConfig_t cfg;
  memset(&cfg, 0, sizeof(cfg));
  cfg.gridDim = dim3(grid);
  cfg.blockDim = dim3(block);
  cfg.stream = c->stream;
  cudaLaunchAttribute attr;
  attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr.val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = &attr;
  cfg.numAttrs = 1;
  cudaLaunchKernelEx(&cfg, kernel, static_cast<P>(args)...);
}

// One launch of the tensor-core engine in tile mode MODE on the context's persistent grid (CTA pairs
// when cta_group is 2; wide tiles exist for pairs only).  a2 / b2 / k2_len: second product (kTileDual).
template <class Epi, int A_MN, int B_MN, int MODE>
void launch_tiles(rl_ctx* c, int cg, int kind, const CUtensorMap& a, const CUtensorMap& b, const CUtensorMap& a2,
                  const CUtensorMap& b2, const CUtensorMap& out, const GemmShape& sh, int k2_len,
                  const typename Epi::Params& ep) {
  const int prof = prof_begin(c, kind);
  cudaLaunchConfig_t cfg;
  memset(&cfg, 0, sizeof(cfg));
  cfg.gridDim = dim3(c->grid[cg]);
  cfg.blockDim = dim3(gemm_threads(Epi::kWarps, Epi::kSideWarps, Epi::kFeeds));
  cfg.stream = c->stream;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  attr[1].id = cudaLaunchAttributeClusterDimension;
  attr[1].val.clusterDim.x = 2;
  attr[1].val.clusterDim.y = 1;
  attr[1].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = cg == 2 ? 2 : 1;
  if (cg == 2) {
    cfg.dynamicSmemBytes = g_smem_bytes<Epi, A_MN, B_MN, 2, MODE>;
    cudaLaunchKernelEx(&cfg, gemm_kernel<Epi, A_MN, B_MN, 2, MODE>, a, b, a2, b2, out, sh, k2_len, ep, c->dstatus);
  } else if constexpr (MODE != kTileWide) {
    cfg.dynamicSmemBytes = g_smem_bytes<Epi, A_MN, B_MN, 1, MODE>;
    cudaLaunchKernelEx(&cfg, gemm_kernel<Epi, A_MN, B_MN, 1, MODE>, a, b, a2, b2, out, sh, k2_len, ep, c->dstatus);
  }
  c->launches++;
  prof_end(c, prof, kind);
}

// 256-column tiles, cg CTAs each; parts: the slots of cut tiles (any map where no tile is cut).
template <class Epi, int A_MN, int B_MN>
void launch_gemm(rl_ctx* c, int cg, int kind, const CUtensorMap& a, const CUtensorMap& b, const CUtensorMap& out,
                 const CUtensorMap& parts, const GemmShape& sh, const typename Epi::Params& ep) {
  launch_tiles<Epi, A_MN, B_MN, kTileSquare>(c, cg, kind, a, b, parts, b, out, sh, 0, ep);
}

// 256 x 512 tiles on CTA pairs; sh.n_tiles counts 512-wide column tiles.
template <class Epi, int A_MN, int B_MN>
void launch_wide(rl_ctx* c, int kind, const CUtensorMap& a, const CUtensorMap& b, const CUtensorMap& out,
                 const CUtensorMap& parts, const GemmShape& sh, const typename Epi::Params& ep) {
  launch_tiles<Epi, A_MN, B_MN, kTileWide>(c, 2, kind, a, b, parts, b, out, sh, 0, ep);
}

template <class Epi>
void launch_dual(rl_ctx* c, int kind, const CUtensorMap& a, const CUtensorMap& b, const CUtensorMap& a2,
                 const CUtensorMap& b2, const CUtensorMap& out, const GemmShape& sh, int k2_len,
                 const typename Epi::Params& ep) {
  launch_tiles<Epi, 0, 0, kTileDual>(c, c->cta_group, kind, a, b, a2, b2, out, sh, k2_len, ep);
}

rl_status check_hw(const void* H, int64_t ldH, const void* W, int64_t ldW, int64_t T, int64_t d, int64_t V) {
  if (T < 0 || d <= 0 || V <= 0) return RL_ERR_INVALID_ARG;
  if (T > 0 && (!H || !W)) return RL_ERR_INVALID_ARG;
  if (d % 64 != 0) return RL_ERR_SHAPE;
  if (T >= (int64_t(1) << 30) || V >= (int64_t(1) << 30)) return RL_ERR_SHAPE;
  if (ldH < d || ldW < d) return RL_ERR_SHAPE;
  if (ldH % 8 != 0 || ldW % 8 != 0) return RL_ERR_ALIGNMENT;
  if ((reinterpret_cast<uintptr_t>(H) & 15) || (reinterpret_cast<uintptr_t>(W) & 15)) return RL_ERR_ALIGNMENT;
  return RL_OK;
}

rl_status check_ws(rl_ctx* c, size_t bytes) {
  if (!c->ws || c->ws_bytes < bytes) return RL_ERR_WORKSPACE;
  return RL_OK;
}

// Vocabulary-parallel call: W holds the vocabulary ids [vocab_off, vocab_off + V) of V_total and the
// per-token statistics of the whole vocabulary come from the caller.
struct ShardArgs {
  int64_t vocab_off, V_total;
  const float* logp;
  const float* entropy;
  const float* lse;
};

// Row tiles per group for the rows-first passes: as many A panels (one row tile x K, bf16) as fit the byte budget.
inline int row_group_tiles(const rl_ctx* c, int64_t k) {
  if (c->row_group_bytes <= 0) return 0;
  const long long panel = (long long)BM * c->cta_group * k * 2;
  const long long n = c->row_group_bytes / panel;
  return n < 1 ? 1 : (n > (1 << 20) ? (1 << 20) : (int)n);
}

void launch_merge(rl_ctx* c, const LossParams& p, int64_t rows, int ranges, int slabs = 1) {
  const int blocks = merge_blocks(rows, slabs, ranges);
  auto merge = [&](auto plain, auto clearing) { launch(c, p.n_clear > 0 ? clearing : plain, blocks, kLossThreads, p, c->dstatus); };
  if (merge_by_thread(rows, ranges)) merge(combine_loss_kernel<1, false>, combine_loss_kernel<1, true>);
  else merge(combine_loss_kernel<kLossThreads / 32, false>, combine_loss_kernel<kLossThreads / 32, true>);
  c->launches++;
}

// Compute capability and SM count (cudaGetDeviceProperties takes 2.5 ms, these two queries a microsecond).
rl_status device_facts(int device, int* major, int* n_sm) {
  if (cudaDeviceGetAttribute(major, cudaDevAttrComputeCapabilityMajor, device) != cudaSuccess ||
      cudaDeviceGetAttribute(n_sm, cudaDevAttrMultiProcessorCount, device) != cudaSuccess)
    return RL_ERR_CUDA;
  return *major == 10 ? RL_OK : RL_ERR_UNSUPPORTED_ARCH;
}

inline rl_status cuda_ok() { return cudaGetLastError() == cudaSuccess ? RL_OK : RL_ERR_CUDA; }

// Mask scan of T rows in two launches (three for very many), row_pos may be NULL.
void launch_mask_scan(rl_ctx* c, const uint8_t* mask, int64_t T, int* block_counts, int* row_map, int* row_pos) {
  const int pr = prof_begin(c, 4);
  const int n_blocks = (int)((T + kScanRowsPerBlock - 1) / kScanRowsPerBlock);
  const int sums = n_blocks <= kScanSumBlocks ? 1 : 0;
  launch(c, mask_count_kernel, n_blocks, kScanThreads, mask, (int)T, block_counts);
  if (!sums) launch(c, mask_offsets_kernel, 1, 1024, block_counts, n_blocks, c->dstatus);
  launch(c, mask_write_kernel, n_blocks, kScanThreads, mask, (int)T, block_counts, sums, row_map, row_pos, c->dstatus);
  prof_end(c, pr, 4);
  c->launches += sums ? 2 : 3;
}

// Which part of the forward stage a call needs, and where its rows of W sit in the vocabulary.
struct FwdPlan {
  bool scan = true;          // mask scan (false: the row map of an earlier call on this workspace is reused)
  bool stats = true;         // tensor-core pass that leaves per-range statistics in the workspace
  int64_t vocab_off = 0;     // first vocabulary id of W's rows (vocabulary-parallel head)
  int64_t V_total = 0;       // size of the whole vocabulary for the token-range check (0: V)
  RowOutputs out = {};       // per-row outputs of the call, zeroed where the mask is 0
};

// Mask scan + row compaction + forward statistics.  Leaves per-range partials in the workspace.
rl_status run_forward(rl_ctx* c, const WsLayout& L, const void* H, int64_t ldH, const void* W, int64_t ldW,
                      const int32_t* tokens, const uint8_t* mask, int64_t T, int64_t d, int64_t V,
                      const KlRef* kl = nullptr, const FwdPlan& plan = FwdPlan()) {
  char* ws = static_cast<char*>(c->ws);
  int* row_map = reinterpret_cast<int*>(ws + L.row_map);
  int* tokens_c = reinterpret_cast<int*>(ws + L.tokens_c);
  __nv_bfloat16* Hc = reinterpret_cast<__nv_bfloat16*>(ws + L.Hc);
  PrepParams pp;
  memset(&pp, 0, sizeof(pp));
  pp.H = static_cast<const __nv_bfloat16*>(H);
  pp.ldH = ldH;
  pp.d = (int)d;
  pp.mask = mask;
  pp.T = (int)T;
  pp.tokens = tokens;
  pp.V = (int)(plan.V_total > 0 ? plan.V_total : V);
  pp.vocab_off = (int)plan.vocab_off;
  pp.Hc = Hc;
  pp.tokens_c = tokens_c;
  pp.row_map = row_map;
  pp.out = plan.out;
  pp.ticket = reinterpret_cast<unsigned*>(reinterpret_cast<char*>(c->dstatus) + kTicketOffset);
  if (T <= kPrepRows) {
    const int pr = prof_begin(c, 5);
    // a row per warp while that takes no more than four blocks per SM; at most 256: kPrepRows / (4 n_sm)
    int rows = (int)align_up((size_t)(T + c->n_sm * 4 - 1) / (c->n_sm * 4), 8);
    if (rows > 256) rows = 256;
    pp.rows_per_block = rows;
    launch(c, prep_rows_kernel<true>, (int)((T + rows - 1) / rows), 256, pp, c->dstatus);
    prof_end(c, pr, 5);
  } else {
    int* row_pos = reinterpret_cast<int*>(ws + L.row_pos);
    if (plan.scan) launch_mask_scan(c, mask, T, reinterpret_cast<int*>(ws + L.scan_counts), row_map, row_pos);
    pp.row_pos = row_pos;
    const int pr = prof_begin(c, 5);
    launch(c, prep_rows_kernel<false>, c->n_sm * 8, 256, pp, c->dstatus);
    prof_end(c, pr, 5);
  }
  c->launches += 1;
  __nv_bfloat16* Hc_ref = reinterpret_cast<__nv_bfloat16*>(ws + L.Hc_ref);
  if (kl) {   // full KL: compact the reference hidden states with the same row map
    launch(c, gather_plain_kernel, c->n_sm * 4, 256, static_cast<const __nv_bfloat16*>(kl->H_ref), kl->ldH_ref, (int)kl->d_ref,
           row_map, Hc_ref, c->dstatus);
    c->launches++;
  }
  if (!plan.stats) {
    return cuda_ok();
  }
  const int cg = kl ? c->cta_group : fwd_cta_group(c, L);
  CUtensorMap tmA, tmB;
  if (!map_kmajor(c, &tmA, Hc, (uint64_t)L.Tpad, (uint64_t)d, (uint64_t)d, BM)) return RL_ERR_CUDA;
  if (!map_kmajor(c, &tmB, W, (uint64_t)V, (uint64_t)d, (uint64_t)ldW, b_box_rows(cg))) return RL_ERR_CUDA;
  GemmShape sh;
  memset(&sh, 0, sizeof(sh));
  sh.n_valid = &c->dstatus->n_valid;
  sh.m_rows_cap = L.Tpad;
  sh.m_dyn = 1;
  sh.k_cap = (int)d;
  sh.n_tiles = (int)((V + BN - 1) / BN);
  sh.n_range = 0;  // split chosen on the device from the number of valid rows
  sh.n_split_max = L.part_ranges;
  sh.leaves_ranges = 1;
  sh.m_group = row_group_tiles(c, d + (kl ? kl->d_ref : 0));
  RowStats::Params ep;
  ep.tokens_c = tokens_c;
  ep.partials = reinterpret_cast<float4*>(ws + L.partials);
  ep.part_stride = L.Tpad;
  ep.V = (int)V;
  if (!kl) {
    if (d <= kEightWarpsMaxK) launch_gemm<EpiStats<8>, 0, 0>(c, cg, 0, tmA, tmB, tmA, tmA, sh, ep);
    else                      launch_gemm<EpiStats<4>, 0, 0>(c, cg, 0, tmA, tmB, tmA, tmA, sh, ep);   // no output map
  } else {
    // both logit tiles per output tile
    CUtensorMap tmA2, tmB2;
    if (!map_kmajor(c, &tmA2, Hc_ref, (uint64_t)L.Tpad, (uint64_t)kl->d_ref, (uint64_t)kl->d_ref, BM)) return RL_ERR_CUDA;
    if (!map_kmajor(c, &tmB2, kl->W_ref, (uint64_t)V, (uint64_t)kl->d_ref, (uint64_t)kl->ldW_ref, b_box_rows(c)))
      return RL_ERR_CUDA;
    EpiStatsKL::Params ek;
    ek.tokens_c = tokens_c;
    ek.partials = ep.partials;
    ek.partials2 = reinterpret_cast<float4*>(ws + L.partials2);
    ek.part_stride = L.Tpad;
    ek.V = (int)V;
    launch_dual<EpiStatsKL>(c, 0, tmA, tmB, tmA2, tmB2, tmA, sh, (int)kl->d_ref, ek);
  }
  return cuda_ok();
}

}  // namespace

extern "C" {

const char* rl_status_string(rl_status s) {
  switch (s) {
    case RL_OK: return "ok";
    case RL_ERR_INVALID_ARG: return "invalid argument";
    case RL_ERR_SHAPE: return "unsupported shape";
    case RL_ERR_ALIGNMENT: return "pointer or leading dimension not aligned for TMA";
    case RL_ERR_WORKSPACE: return "workspace missing or too small";
    case RL_ERR_CUDA: return "CUDA call failed";
    case RL_ERR_UNSUPPORTED_ARCH: return "device is not compute capability 10.x";
    case RL_ERR_TOKEN_RANGE: return "token id outside [0,V) on a valid row";
    case RL_ERR_TIMEOUT: return "bounded wait inside a kernel ran out";
  }
  return "unknown status";
}

rl_status rl_create(rl_ctx** out, int device) {
  if (!out) return RL_ERR_INVALID_ARG;
  *out = nullptr;
  int major = 0, n_sm = 0;
  rl_status sd = device_facts(device, &major, &n_sm);
  if (sd != RL_OK) return sd;
  if (cudaSetDevice(device) != cudaSuccess) return RL_ERR_CUDA;
  rl_ctx* c = new (std::nothrow) rl_ctx();
  if (!c) return RL_ERR_CUDA;
  c->device = device;
  c->n_sm = n_sm;
  c->stream = nullptr;
  c->ws = nullptr;
  c->ws_bytes = 0;
  c->slab_rows = kSlabRowsMax;
  c->slab_cols = kSlabColsMax;
  c->slab_auto = 1;
  c->cta_group = 1;
  c->dh_k_slices = 1;
  c->dh_stream_k = 0;
  c->wide_tiles = 1;
  c->row_group_bytes = kRowGroupBytes;
  c->fixed_scratch = 0;
  c->grid[0] = 0;
  c->grid[1] = c->n_sm;
  c->grid[2] = c->n_sm / 2 * 2;
  c->launches = 0;
  c->prof_on = 0;
  c->prof_used = 0;
  c->prof_kind = nullptr;
  c->prof_ev = nullptr;
  c->copy_stream = nullptr;
  for (int i = 0; i < 2; ++i) { c->copy_done[i] = nullptr; c->step_done[i] = nullptr; c->pinned_out[i] = nullptr; c->slot_busy[i] = 0; }
  void* fn = nullptr;
  cudaDriverEntryPointQueryResult qres;
  if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &fn, cudaEnableDefault, &qres) != cudaSuccess || !fn ||
      qres != cudaDriverEntryPointSuccess) {
    delete c;
    return RL_ERR_CUDA;
  }
  c->encode = reinterpret_cast<EncodeTiledFn>(fn);
  // device block: status word, then two doubles for batch statistics
  if (cudaMalloc(&c->dstatus, kStatusBytes) != cudaSuccess) { delete c; return RL_ERR_CUDA; }
  cudaMemset(c->dstatus, 0, kStatusBytes);
  bool ok = set_smem_attr<EpiStats<4>, 0, 0>() == cudaSuccess && set_smem_attr<EpiGrad<4>, 0, 0>() == cudaSuccess &&
            set_smem_attr<EpiStats<8>, 0, 0>() == cudaSuccess && set_smem_attr<EpiGrad<8>, 0, 0>() == cudaSuccess &&
            set_smem_attr<EpiSweep, 0, 0>() == cudaSuccess && set_smem_attr<EpiRefSweep, 0, 0>() == cudaSuccess &&
            set_smem_attr<EpiSweepKL, 0, 0>() == cudaSuccess &&
            set_smem_attr<EpiAcc, 0, 0>() == cudaSuccess && set_smem_attr<EpiAcc, 0, 1>() == cudaSuccess &&
            set_smem_attr<EpiAcc, 1, 0>() == cudaSuccess && set_smem_attr<EpiAcc, 1, 1>() == cudaSuccess &&
            set_smem_attr_dual<EpiStatsKL>() == cudaSuccess && set_smem_attr_dual<EpiGradKL>() == cudaSuccess &&
            set_smem_attr_one<EpiAcc, 0, 1, 2, kTileWide>() == cudaSuccess &&
            set_smem_attr<EpiAccScatter<4>, 1, 1>() == cudaSuccess && set_smem_attr<EpiAccScatter<8>, 1, 1>() == cudaSuccess && set_smem_attr<EpiAccFed, 0, 1>() == cudaSuccess &&
            set_smem_attr_one<EpiAccFed, 0, 1, 2, kTileWide>() == cudaSuccess;
  if (!ok) { cudaFree(c->dstatus); delete c; return RL_ERR_CUDA; }
  {
    // how many CTA pairs can be resident at once (pairs must share a TPC): the persistent grid
    // of the paired kernels must not exceed it
    cudaLaunchConfig_t cfg;
    memset(&cfg, 0, sizeof(cfg));
    cfg.gridDim = dim3(c->grid[2]);
    cfg.blockDim = dim3(gemm_threads(EpiAcc::kWarps, EpiAcc::kSideWarps, EpiAcc::kFeeds));
    cfg.dynamicSmemBytes = g_smem_bytes<EpiAcc, 0, 0, 2, kTileSquare>;
    cudaLaunchAttribute attr;
    attr.id = cudaLaunchAttributeClusterDimension;
    attr.val.clusterDim.x = 2;
    attr.val.clusterDim.y = 1;
    attr.val.clusterDim.z = 1;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    int n_clusters = 0;
    if (cudaOccupancyMaxActiveClusters(&n_clusters, gemm_kernel<EpiAcc, 0, 0, 2, kTileSquare>, &cfg) == cudaSuccess &&
        n_clusters > 0) {
      if (2 * n_clusters < c->grid[2]) c->grid[2] = 2 * n_clusters;
    } else {
      cudaGetLastError();
      c->grid[2] = 0;   // paired kernels unavailable
    }
    if (c->grid[2] >= 2) c->cta_group = 2;   // default: CTA pairs
  }
  for (int i = 0; i < 3; ++i) c->grid_full[i] = c->grid[i];
  c->dw_hook = nullptr;
  c->dw_hook_user = nullptr;
  *out = c;
  return RL_OK;
}

rl_status rl_destroy(rl_ctx* c) {
  if (!c) return RL_ERR_INVALID_ARG;
  if (c->prof_ev) {
    for (int i = 0; i < kProfMax; ++i)
      for (int e = 0; e < 2; ++e)
        if (c->prof_ev[i][e]) cudaEventDestroy(c->prof_ev[i][e]);
    delete[] c->prof_ev;
    delete[] c->prof_kind;
  }
  if (c->copy_stream) {
    cudaStreamSynchronize(c->copy_stream);
    cudaStreamDestroy(c->copy_stream);
    for (int i = 0; i < 2; ++i) {
      cudaEventDestroy(c->copy_done[i]);
      cudaEventDestroy(c->step_done[i]);
      cudaFreeHost(c->pinned_out[i]);
    }
  }
  cudaFree(c->dstatus);
  delete c;
  return RL_OK;
}

rl_status rl_set_stream(rl_ctx* c, void* s) {
  if (!c) return RL_ERR_INVALID_ARG;
  c->stream = static_cast<cudaStream_t>(s);
  return RL_OK;
}

rl_status rl_workspace_bytes(rl_ctx* c, int64_t T, int64_t d, int64_t V, size_t* bytes) {
  if (!c || !bytes || T < 0 || d <= 0 || V <= 0) return RL_ERR_INVALID_ARG;
  *bytes = ws_bytes(c, T, d, V);
  return RL_OK;
}

rl_status rl_workspace_bytes_logprobs(rl_ctx* c, int64_t T, int64_t d, int64_t V, size_t* bytes) {
  if (!c || !bytes || T < 0 || d <= 0 || V <= 0) return RL_ERR_INVALID_ARG;
  *bytes = ws_layout(c, T, d, V, false).G;
  return RL_OK;
}

rl_status rl_workspace_bytes_kl(rl_ctx* c, int64_t T, int64_t d, int64_t V, int64_t d_ref, size_t* bytes) {
  if (!c || !bytes || T < 0 || d <= 0 || V <= 0 || d_ref <= 0) return RL_ERR_INVALID_ARG;
  *bytes = ws_layout(c, T, d, V, false, d_ref).total;
  return RL_OK;
}

rl_status rl_workspace_bytes_host(rl_ctx* c, int64_t T, int64_t d, int64_t V, size_t* bytes) {
  if (!c || !bytes || T < 0 || d <= 0 || V <= 0) return RL_ERR_INVALID_ARG;
  *bytes = ws_layout(c, T, d, V, true).total;
  return RL_OK;
}

rl_status rl_set_cta_group(rl_ctx* c, int cta_group) {
  if (!c) return RL_ERR_INVALID_ARG;
  if (cta_group != 1 && cta_group != 2) return RL_ERR_INVALID_ARG;
  if (cta_group == 2 && c->grid[2] < 2) return RL_ERR_UNSUPPORTED_ARCH;
  c->cta_group = cta_group;
  return RL_OK;
}

rl_status rl_set_max_ctas(rl_ctx* c, int max_ctas) {
  if (!c || max_ctas < 0) return RL_ERR_INVALID_ARG;
  if (max_ctas == 0) {
    for (int i = 0; i < 3; ++i) c->grid[i] = c->grid_full[i];
    return RL_OK;
  }
  if (max_ctas < 2) return RL_ERR_INVALID_ARG;
  c->grid[1] = max_ctas < c->grid_full[1] ? max_ctas : c->grid_full[1];
  const int pairs = max_ctas / 2 * 2;
  c->grid[2] = pairs < c->grid_full[2] ? pairs : c->grid_full[2];
  return RL_OK;
}

rl_status rl_set_dw_slab_hook(rl_ctx* c, rl_dw_slab_hook hook, void* user) {
  if (!c) return RL_ERR_INVALID_ARG;
  c->dw_hook = hook;
  c->dw_hook_user = hook ? user : nullptr;
  return RL_OK;
}

rl_status rl_set_dh_k_slices(rl_ctx* c, int max_slices) {
  if (!c) return RL_ERR_INVALID_ARG;
  if (max_slices < 1 || max_slices > kDhSplitMax) return RL_ERR_INVALID_ARG;
  c->dh_k_slices = max_slices;
  return RL_OK;
}

rl_status rl_set_row_group_bytes(rl_ctx* c, int64_t bytes) {
  if (!c || bytes < 0) return RL_ERR_INVALID_ARG;
  c->row_group_bytes = bytes;
  return RL_OK;
}

rl_status rl_set_wide_tiles(rl_ctx* c, int on) {
  if (!c) return RL_ERR_INVALID_ARG;
  c->wide_tiles = on ? 1 : 0;
  return RL_OK;
}

rl_status rl_set_dh_stream_k(rl_ctx* c, int on) {
  if (!c) return RL_ERR_INVALID_ARG;
  c->dh_stream_k = on ? 1 : 0;
  return RL_OK;
}

rl_status rl_launch_count(rl_ctx* c, int64_t* n) {
  if (!c || !n) return RL_ERR_INVALID_ARG;
  *n = c->launches;
  return RL_OK;
}

rl_status rl_set_profiling(rl_ctx* c, int on) {
  if (!c) return RL_ERR_INVALID_ARG;
  if (on && !c->prof_ev) {
    c->prof_kind = new (std::nothrow) int[kProfMax];
    c->prof_ev = new (std::nothrow) cudaEvent_t[kProfMax][2];
    if (!c->prof_kind || !c->prof_ev) {
      delete[] c->prof_kind;
      delete[] c->prof_ev;
      c->prof_kind = nullptr;
      c->prof_ev = nullptr;
      return RL_ERR_CUDA;
    }
    memset(c->prof_ev, 0, sizeof(cudaEvent_t) * 2 * kProfMax);
  }
  c->prof_on = on ? 1 : 0;
  c->prof_used = 0;
  return RL_OK;
}

rl_status rl_profile_read(rl_ctx* c, double* ms, int64_t* launches) {
  if (!c || !ms || !launches) return RL_ERR_INVALID_ARG;
  if (cudaStreamSynchronize(c->stream) != cudaSuccess) return RL_ERR_CUDA;
  for (int k = 0; k < kProfKinds; ++k) { ms[k] = 0.0; launches[k] = 0; }
  for (int i = 0; i < c->prof_used; ++i) {
    float t = 0.f;
    if (cudaEventElapsedTime(&t, c->prof_ev[i][0], c->prof_ev[i][1]) != cudaSuccess) return RL_ERR_CUDA;
    ms[c->prof_kind[i]] += t;
    launches[c->prof_kind[i]]++;
  }
  c->prof_used = 0;
  return RL_OK;
}

rl_status rl_set_slab_limits(rl_ctx* c, int max_rows, int max_cols) {
  if (!c) return RL_ERR_INVALID_ARG;
  const int automatic = max_rows == 0 && max_cols == 0;
  if (max_rows == 0) max_rows = kSlabRowsMax;
  if (max_cols == 0) max_cols = kSlabColsMax;
  if (max_rows < 128 || max_rows % 128 != 0 || max_cols < 256 || max_cols % 256 != 0) return RL_ERR_SHAPE;
  if ((int64_t)max_rows * max_cols > (int64_t(1) << 31)) return RL_ERR_SHAPE;
  c->slab_rows = max_rows;
  c->slab_cols = max_cols;
  c->slab_auto = automatic;
  return RL_OK;
}

rl_status rl_set_workspace(rl_ctx* c, void* p, size_t bytes) {
  if (!c) return RL_ERR_INVALID_ARG;
  if (p && (reinterpret_cast<uintptr_t>(p) & 255)) return RL_ERR_ALIGNMENT;
  c->ws = p;
  c->ws_bytes = p ? bytes : 0;
  return RL_OK;
}

rl_status rl_last_device_status(rl_ctx* c, int32_t* detail) {
  if (!c) return RL_ERR_INVALID_ARG;
  DevStatus h;
  if (cudaStreamSynchronize(c->stream) != cudaSuccess) return RL_ERR_CUDA;
  if (cudaMemcpy(&h, c->dstatus, sizeof(h), cudaMemcpyDeviceToHost) != cudaSuccess) return RL_ERR_CUDA;
  if (detail) *detail = h.detail;
  if (h.code != 0) {
    int zero[2] = {0, 0};
    cudaMemcpy(c->dstatus, zero, sizeof(zero), cudaMemcpyHostToDevice);
  }
  return static_cast<rl_status>(h.code);
}

rl_status rl_grpo_advantages_ex(rl_ctx* c, const float* rewards, int64_t n_seq, int group_size, int ddof,
                                float eps_std, const int32_t* seq_offsets, int64_t T, float* adv_seq,
                                float* adv_tok) {
  if (!c || n_seq < 0 || (n_seq > 0 && (!rewards || !adv_seq))) return RL_ERR_INVALID_ARG;
  if ((ddof != 0 && ddof != 1) || !(eps_std >= 0.f)) return RL_ERR_INVALID_ARG;
  if ((adv_tok != nullptr) != (seq_offsets != nullptr) || T < 0) return RL_ERR_INVALID_ARG;
  if (group_size < 2 || n_seq % group_size != 0 || n_seq >= (int64_t(1) << 31)) return RL_ERR_SHAPE;
  if (n_seq == 0) return RL_OK;
  const int n_groups = (int)(n_seq / group_size);
  const int warps = 8;
  int seg = 32;   // lanes per group, as the kernel computes it
  while (seg > 1 && (seg >> 1) >= group_size) seg >>= 1;
  const int groups_per_block = warps * (32 / seg);
  const int pr_adv = prof_begin(c, 8);
  // many groups of 4, 8, ... 32 responses in 16-byte aligned arrays: one thread per group; else shuffle segments
  const bool rows_path = n_groups >= kAdvRowsMinGroups && group_size % 4 == 0 && group_size <= 32 &&
                         ((reinterpret_cast<uintptr_t>(rewards) | reinterpret_cast<uintptr_t>(adv_seq)) & 15) == 0;
  // few groups of few responses and rows: the broadcast works the advantages out itself
  const bool fused = adv_tok && T > 0 && T <= kFusedAdvRows && n_groups < kAdvRowsMinGroups && group_size <= 32 && rewards != adv_seq;
  if (fused) {
  } else if (rows_path) {
    const int blocks = (n_groups + 255) / 256;
    const float4* r4 = reinterpret_cast<const float4*>(rewards);
    float4* a4 = reinterpret_cast<float4*>(adv_seq);
    switch (group_size / 4) {
      case 1: launch(c, grpo_adv_rows_kernel<1>, blocks, 256, r4, n_groups, ddof, eps_std, a4); break;
      case 2: launch(c, grpo_adv_rows_kernel<2>, blocks, 256, r4, n_groups, ddof, eps_std, a4); break;
      case 3: launch(c, grpo_adv_rows_kernel<3>, blocks, 256, r4, n_groups, ddof, eps_std, a4); break;
      case 4: launch(c, grpo_adv_rows_kernel<4>, blocks, 256, r4, n_groups, ddof, eps_std, a4); break;
      case 5: launch(c, grpo_adv_rows_kernel<5>, blocks, 256, r4, n_groups, ddof, eps_std, a4); break;
      case 6: launch(c, grpo_adv_rows_kernel<6>, blocks, 256, r4, n_groups, ddof, eps_std, a4); break;
      case 7: launch(c, grpo_adv_rows_kernel<7>, blocks, 256, r4, n_groups, ddof, eps_std, a4); break;
      default: launch(c, grpo_adv_rows_kernel<8>, blocks, 256, r4, n_groups, ddof, eps_std, a4); break;
    }
  } else {
    launch(c, grpo_adv_kernel, (n_groups + groups_per_block - 1) / groups_per_block, warps * 32, rewards, n_groups, group_size, ddof, eps_std, adv_seq);
  }
  c->launches += fused ? 0 : 1;
  if (adv_tok && T > 0) {
    long long sweeps = T / (1024ll * 2 * c->n_sm);   // two blocks per SM before a block takes more than one sweep
    sweeps = sweeps < 1 ? 1 : (sweeps > kBroadcastSweeps ? kBroadcastSweeps : sweeps);
    long long blocks = (T + sweeps * 1024 - 1) / (sweeps * 1024);
    if (blocks > (long long)c->n_sm * 32) blocks = (long long)c->n_sm * 32;
    if (fused)
      launch(c, broadcast_adv_kernel<true>, (int)blocks, 256, rewards, group_size, ddof, eps_std, adv_seq, seq_offsets, (int)n_seq, (long long)T, (int)sweeps, adv_tok);
    else
      launch(c, broadcast_adv_kernel<false>, (int)blocks, 256, rewards, group_size, ddof, eps_std, adv_seq, seq_offsets, (int)n_seq, (long long)T, (int)sweeps, adv_tok);
    c->launches++;
  }
  prof_end(c, pr_adv, 8);
  return cuda_ok();
}

rl_status rl_advantages(rl_ctx* c, int estimator, const float* rewards, const int32_t* lengths, int64_t n_seq,
                        int group_size, float eps_std, float* adv_seq) {
  if (!c || n_seq < 0 || (n_seq > 0 && (!rewards || !adv_seq))) return RL_ERR_INVALID_ARG;
  if (estimator < RL_ADV_GRPO || estimator > RL_ADV_REINFORCE_PP || !(eps_std >= 0.f)) return RL_ERR_INVALID_ARG;
  if (estimator == RL_ADV_OPO && n_seq > 0 && !lengths) return RL_ERR_INVALID_ARG;
  if (estimator == RL_ADV_GRPO)
    return rl_grpo_advantages_ex(c, rewards, n_seq, group_size, 1, eps_std, nullptr, 0, adv_seq, nullptr);
  const int min_group = estimator == RL_ADV_RLOO ? 2 : 1;
  if (group_size < min_group || n_seq % group_size != 0 || n_seq >= (int64_t(1) << 31)) return RL_ERR_SHAPE;
  if (n_seq == 0) return RL_OK;
  const int n_groups = (int)(n_seq / group_size);
  const int warps = 8;
  const int pr = prof_begin(c, 8);
  launch(c, group_baseline_kernel, (n_groups + warps - 1) / warps, warps * 32, rewards, lengths, n_groups, group_size, estimator, adv_seq);
  c->launches++;
  if (estimator == RL_ADV_REINFORCE_PP) {
    double* stats = reinterpret_cast<double*>(reinterpret_cast<char*>(c->dstatus) + 64);
    launch(c, batch_stats_kernel, 1, 1024, adv_seq, (long long)n_seq, stats);
    int blocks = (int)((n_seq + 255) / 256);
    if (blocks > 4096) blocks = 4096;
    launch(c, batch_normalise_kernel, blocks, 256, adv_seq, (long long)n_seq, stats, eps_std);
    c->launches += 2;
  }
  prof_end(c, pr, 8);
  return cuda_ok();
}

rl_status rl_token_loss(rl_ctx* c, const float* logp, const float* entropy, const float* old_logp,
                        const float* ref_logp, const float* adv, const uint8_t* mask, int64_t T, float eps_low,
                        float eps_high, float beta, float ent_coef, const float* token_weight, const void* token_count,
                        float* loss, float* dlogp, float* dentropy, float* metrics_out) {
  if (!c || T < 0 || !loss) return RL_ERR_INVALID_ARG;
  if (!(eps_low >= 0.f && eps_low < 1.f) || !(eps_high >= 0.f) || !(beta >= 0.f) || !(ent_coef >= 0.f))
    return RL_ERR_INVALID_ARG;
  if (T > 0 && (!logp || !old_logp || !adv)) return RL_ERR_INVALID_ARG;
  if (T > 0 && beta != 0.f && !ref_logp) return RL_ERR_INVALID_ARG;
  if (T > 0 && ent_coef != 0.f && !entropy) return RL_ERR_INVALID_ARG;
  cudaStream_t st = c->stream;
  if (T == 0) {
    cudaMemsetAsync(loss, 0, 4, st);
    if (metrics_out) cudaMemsetAsync(metrics_out, 0, 32, st);
    return cuda_ok();
  }
  char* base = reinterpret_cast<char*>(c->dstatus);
  unsigned* counts = reinterpret_cast<unsigned*>(base + kCountOffset);
  double* block_sums = reinterpret_cast<double*>(base + kSumsOffset);
  const int pr = prof_begin(c, 6);
  long long cb = 0;
  if (mask) {
    cb = (T / 16 + 255) / 256 + 1;
    if (cb > kCountBlocks) cb = kCountBlocks;
    launch(c, count_valid_kernel, (int)cb, 256, mask, (long long)T, counts);
    c->launches++;
  }
  TokenLossParams p;
  memset(&p, 0, sizeof(p));
  p.logp = logp; p.entropy = entropy; p.old_logp = old_logp; p.ref_logp = beta != 0.f ? ref_logp : nullptr;
  p.adv = adv; p.mask = mask; p.token_weight = token_weight;
  p.counts = mask ? counts : nullptr;
  p.n_counts = (int)cb;
  p.token_count = reinterpret_cast<const unsigned long long*>(token_count);
  p.T = (long long)T;
  p.eps_low = eps_low; p.eps_high = eps_high; p.beta = beta; p.ent_coef = ent_coef;
  p.dlogp = dlogp; p.dentropy = dentropy;
  long long blocks = ((T + 3) / 4 + kLossThreads - 1) / kLossThreads;
  if (blocks > kTokenLossBlocks) blocks = kTokenLossBlocks;
  if (blocks > (long long)c->n_sm * 4) blocks = (long long)c->n_sm * 4;   // one wave: four blocks are resident per SM
  uintptr_t all = reinterpret_cast<uintptr_t>(logp) | reinterpret_cast<uintptr_t>(old_logp) | reinterpret_cast<uintptr_t>(adv) |
                  reinterpret_cast<uintptr_t>(entropy) | reinterpret_cast<uintptr_t>(p.ref_logp) |
                  reinterpret_cast<uintptr_t>(token_weight) | reinterpret_cast<uintptr_t>(dlogp) |
                  reinterpret_cast<uintptr_t>(dentropy);
  const bool vec = (all & 15) == 0 && (reinterpret_cast<uintptr_t>(mask) & 3) == 0;
  p.fin.block_sums = block_sums;
  p.fin.ticket = reinterpret_cast<unsigned*>(base + kTicketOffset) + 1;
  p.fin.base = 0;
  p.fin.total = (int)blocks;
  p.fin.loss = loss;
  p.fin.metrics = metrics_out;
  if (vec) launch(c, token_loss_kernel<true>, (int)blocks, kLossThreads, p);
  else     launch(c, token_loss_kernel<false>, (int)blocks, kLossThreads, p);
  c->launches += 1;
  prof_end(c, pr, 6);
  return cuda_ok();
}

rl_status rl_grpo_advantages(rl_ctx* c, const float* rewards, int64_t n_seq, int group_size, float* adv_seq) {
  return rl_grpo_advantages_ex(c, rewards, n_seq, group_size, 1, 1e-6f, nullptr, 0, adv_seq, nullptr);
}

rl_status rl_kl_shaped_returns(rl_ctx* c, const float* seq_value, const float* logp, const float* ref_logp,
                               const float* kl_tok, const uint8_t* mask, const int32_t* seq_offsets, int64_t n_seq,
                               int64_t T, float beta, float gamma, int kl_estimate, float* shaped_reward,
                               float* returns) {
  if (!c || n_seq < 0 || T < 0 || n_seq >= (int64_t(1) << 31) || T >= (int64_t(1) << 31)) return RL_ERR_INVALID_ARG;
  if (kl_estimate < RL_KL_K1 || kl_estimate > RL_KL_GIVEN || !(beta >= 0.f) || !(gamma >= 0.f)) return RL_ERR_INVALID_ARG;
  if (T == 0) return RL_OK;
  if (!returns) return RL_ERR_INVALID_ARG;
  if (n_seq == 0) {
    cudaMemsetAsync(returns, 0, (size_t)T * 4, c->stream);
    if (shaped_reward) cudaMemsetAsync(shaped_reward, 0, (size_t)T * 4, c->stream);
    return cuda_ok();
  }
  if (!seq_value || !seq_offsets) return RL_ERR_INVALID_ARG;
  if (kl_estimate == RL_KL_GIVEN ? !kl_tok : (!logp || !ref_logp)) return RL_ERR_INVALID_ARG;
  // A block per response, else a warp.  A block walks 512 rows at a time whether there are as many or not: with responses enough to
  // fill the machine either way it has to have them.  4096 / 32768 responses, block against warp: 21 / 158 us against 15 / 103 at 256 rows,
  // 22 / 164 against 19 / 146 at 384, 23 / 167 against 22 / 191 at 512, 34 / 281 against 25 / 227 at 600, 37 / 312 against 38 / 337 at 900;
  // 1024 responses: 10.8 against 12.7, 10.8 / 15.2, 10.9 / 18.8, 14.6 / 21.3, 14.7 / 29.2.
  constexpr int64_t kWarpRows = 32 * kShapeChunks, kBlockRows = kWarpRows * kShapeWarps;
  const int64_t mean_rows = T / n_seq, walked = (mean_rows + kBlockRows - 1) / kBlockRows * kBlockRows;
  const bool by_block = mean_rows >= kWarpRows && (n_seq <= (int64_t)c->n_sm * 8 || mean_rows * 16 >= walked * 13);
  int64_t blocks = by_block ? n_seq : (n_seq + kShapeWarps - 1) / kShapeWarps;
  if (blocks > (int64_t)c->n_sm * 64) blocks = (int64_t)c->n_sm * 64;
  const int pr = prof_begin(c, 8);
  auto shape = [&](auto kernel) {
    launch(c, kernel, (int)blocks, 32 * kShapeWarps, seq_value, logp, ref_logp, kl_tok, mask, seq_offsets, (int)n_seq,
                                                            (long long)T, beta, gamma, kl_estimate, shaped_reward, returns);
  };
  if (by_block) shape(kl_shaped_returns_kernel<kShapeWarps>);
  else          shape(kl_shaped_returns_kernel<1>);
  prof_end(c, pr, 8);
  c->launches += 1;
  return cuda_ok();
}

rl_status rl_mask_scan(rl_ctx* c, const uint8_t* mask, int64_t T, int32_t* row_map, int32_t* n_valid) {
  if (!c || T < 0 || T >= (int64_t(1) << 31) || !n_valid || (T > 0 && !row_map)) return RL_ERR_INVALID_ARG;
  if (T == 0) return cudaMemsetAsync(n_valid, 0, 4, c->stream) == cudaSuccess ? RL_OK : RL_ERR_CUDA;
  const int n_blocks = (int)((T + kScanRowsPerBlock - 1) / kScanRowsPerBlock);
  if (!c->ws || c->ws_bytes < ((size_t)n_blocks + 2) * 4) return RL_ERR_WORKSPACE;
  int* block_counts = static_cast<int*>(c->ws);
  launch_mask_scan(c, mask, T, block_counts, row_map, nullptr);
  if (cudaMemcpyAsync(n_valid, &c->dstatus->n_valid, 4, cudaMemcpyDeviceToDevice, c->stream) != cudaSuccess)
    return RL_ERR_CUDA;
  return cuda_ok();
}

rl_status rl_token_logprobs(rl_ctx* c, const void* H, int64_t ldH, const void* W, int64_t ldW, const int32_t* tokens,
                            const uint8_t* mask, int64_t T, int64_t d, int64_t V, float* logp, float* entropy,
                            float* lse) {
  if (!c) return RL_ERR_INVALID_ARG;
  rl_status s = check_hw(H, ldH, W, ldW, T, d, V);
  if (s != RL_OK) return s;
  if (T == 0) return RL_OK;
  if (!tokens || !logp) return RL_ERR_INVALID_ARG;
  const WsLayout L = ws_layout(c, T, d, V, false);
  if ((s = check_ws(c, L.G)) != RL_OK) return s;   // the forward arrays
  char* ws = static_cast<char*>(c->ws);
  FwdPlan plan;
  plan.out.value[0] = logp; plan.out.value[1] = entropy; plan.out.value[2] = lse;
  if ((s = run_forward(c, L, H, ldH, W, ldW, tokens, mask, T, d, V, nullptr, plan)) != RL_OK) return s;
  LossParams p;
  memset(&p, 0, sizeof(p));
  p.partials = reinterpret_cast<const float4*>(ws + L.partials);
  p.part_stride = L.Tpad;
  p.row_map = reinterpret_cast<const int*>(ws + L.row_map);
  p.with_loss = 0;
  p.lse_c = reinterpret_cast<float*>(ws + L.lse_c);
  p.ent_c = reinterpret_cast<float*>(ws + L.ent_c);
  p.logp_out = logp;
  p.ent_out = entropy;
  p.lse_out = lse;
  launch_merge(c, p, T, L.part_ranges);
  return cuda_ok();
}

// Body of rl_policy_loss_fwd_bwd_ex (shard == NULL) and of rl_policy_loss_shard_bwd.
static rl_status loss_fwd_bwd_impl(rl_ctx* c, const void* H, int64_t ldH, const void* W, int64_t ldW,
                                   const int32_t* tokens, const float* old_logp, const float* ref_logp,
                                   const float* adv, const uint8_t* mask, int64_t T, int64_t d, int64_t V,
                                   float eps_low, float eps_high, float beta, float* loss, void* dH, float* dW,
                                   const rl_loss_opts* opts, const ShardArgs* shard) {
  if (!c) return RL_ERR_INVALID_ARG;
  rl_status s = check_hw(H, ldH, W, ldW, T, d, V);
  if (s != RL_OK) return s;
  if (!(eps_low >= 0.f && eps_low < 1.f) || !(eps_high >= 0.f) || !(beta >= 0.f)) return RL_ERR_INVALID_ARG;
  if (!loss || !dW || !W) return RL_ERR_INVALID_ARG;
  if (T > 0 && (!tokens || !old_logp || !adv || !dH)) return RL_ERR_INVALID_ARG;
  rl_loss_opts o;
  memset(&o, 0, sizeof(o));
  if (opts) {
    if (opts->struct_size < sizeof(size_t) + sizeof(float) || opts->struct_size > sizeof(rl_loss_opts))
      return RL_ERR_INVALID_ARG;
    memcpy(&o, opts, opts->struct_size);
  }
  if (!(o.ent_coef >= 0.f)) return RL_ERR_INVALID_ARG;
  if (beta != 0.f && T > 0 && !ref_logp && !o.kl_full) return RL_ERR_INVALID_ARG;
  if (o.agg_mode < 0 || o.agg_mode > 2 || (o.dH_dtype != 0 && o.dH_dtype != 1)) return RL_ERR_INVALID_ARG;
  if ((o.sequence_level || (o.agg_mode != 0 && !o.token_weight)) && T > 0 &&
      (!o.seq_offsets || o.n_seq <= 0 || o.n_seq > T))
    return RL_ERR_INVALID_ARG;
  if ((reinterpret_cast<uintptr_t>(dH) & 15) || (reinterpret_cast<uintptr_t>(dW) & 15)) return RL_ERR_ALIGNMENT;
  const bool seq_path = o.sequence_level || (o.agg_mode != 0 && !o.token_weight);
  KlRef klref;
  memset(&klref, 0, sizeof(klref));
  if (shard) {
    if (o.kl_full) return RL_ERR_INVALID_ARG;
    if (shard->vocab_off < 0 || shard->V_total < shard->vocab_off + V || shard->V_total >= (int64_t(1) << 30))
      return RL_ERR_SHAPE;
    if (T > 0 && (!shard->logp || !shard->entropy || !shard->lse)) return RL_ERR_INVALID_ARG;
  }
  if (o.kl_full) {
    if (seq_path) return RL_ERR_INVALID_ARG;
    if (!o.W_ref || (T > 0 && !o.H_ref) || o.d_ref <= 0) return RL_ERR_INVALID_ARG;
    if (o.d_ref % 64 != 0 || o.ldH_ref < o.d_ref || o.ldW_ref < o.d_ref || o.ldH_ref % 8 != 0 || o.ldW_ref % 8 != 0)
      return RL_ERR_SHAPE;
    if ((reinterpret_cast<uintptr_t>(o.H_ref) & 15) || (reinterpret_cast<uintptr_t>(o.W_ref) & 15))
      return RL_ERR_ALIGNMENT;
    klref.H_ref = o.H_ref; klref.ldH_ref = o.ldH_ref;
    klref.W_ref = o.W_ref; klref.ldW_ref = o.ldW_ref;
    klref.d_ref = o.d_ref;
  }
  WsLayout L = ws_layout(c, T, d, V, 0, o.kl_full ? o.d_ref : 0);
  // the coefficients of a response's rows need rows of other slabs: the logits are formed twice
  if (seq_path && L.n_row_slabs > 1) L = ws_layout(c, T, d, V, 0, 0, true);
  if ((s = check_ws(c, L.total)) != RL_OK) return s;
  char* ws = static_cast<char*>(c->ws);
  cudaStream_t st = c->stream;

  if (T == 0) {
    cudaMemsetAsync(loss, 0, 4, st);
    if (!o.accumulate_dW) cudaMemsetAsync(dW, 0, (size_t)V * d * 4, st);
    if (o.metrics_out) cudaMemsetAsync(o.metrics_out, 0, 32, st);
    return cuda_ok();
  }

  // ---- forward: statistics per (row, vocabulary range).  One sweep: a slab that holds whole rows lets the pass that
  // forms their logits leave them there in fp32, and an elementwise pass turns them into the gradient once the rows'
  // coefficients are known.  Not where the coefficients of a row need rows of another slab, nor where the
  // statistics come from elsewhere: those paths form the logits a second time.
  const bool sweep = L.keeps_logits && !shard && (L.n_row_slabs == 1 || !seq_path);
  FwdPlan plan;
  plan.out.dH = dH;
  plan.out.dH_row_bytes = (long long)d * (o.dH_dtype ? 4 : 2);
  plan.out.value[0] = o.logp_out; plan.out.value[1] = o.entropy_out;
  plan.out.value[2] = o.kl_full ? o.kl_out : nullptr;
  if (sweep) plan.stats = false;
  if (shard) {
    // the statistics of the whole vocabulary are given: only the row compaction is needed
    plan.stats = false;
    plan.vocab_off = shard->vocab_off;
    plan.V_total = shard->V_total;
  }
  if ((s = run_forward(c, L, H, ldH, W, ldW, tokens, mask, T, d, V, o.kl_full ? &klref : nullptr, plan)) !=
      RL_OK)
    return s;

  // ---- merge + per-token loss, coefficients of the backward pass
  LossParams p;
  memset(&p, 0, sizeof(p));
  p.partials = reinterpret_cast<const float4*>(ws + L.partials);
  p.part_stride = L.Tpad;
  p.row_map = reinterpret_cast<const int*>(ws + L.row_map);
  p.old_logp = old_logp;
  p.ref_logp = ref_logp;
  p.adv = adv;
  p.token_weight = o.token_weight;
  p.eps_low = eps_low;
  p.eps_high = eps_high;
  p.beta = beta;
  p.ent_coef = o.ent_coef;
  p.token_count = reinterpret_cast<const long long*>(o.token_count);
  p.with_loss = 1;
  p.lse_c = reinterpret_cast<float*>(ws + L.lse_c);
  p.ent_c = reinterpret_cast<float*>(ws + L.ent_c);
  p.cp_c = reinterpret_cast<float*>(ws + L.cp_c);
  p.ce_c = reinterpret_cast<float*>(ws + L.ce_c);
  if (seq_path) p.logp_c = reinterpret_cast<float*>(ws + L.logp_c);
  p.logp_out = o.logp_out;
  p.ent_out = o.entropy_out;
  if (shard) {
    p.ext_logp = shard->logp;
    p.ext_ent = shard->entropy;
    p.ext_lse = shard->lse;
  }
  if (o.kl_full) {
    p.kl_full = 1;
    p.partials2 = reinterpret_cast<const float4*>(ws + L.partials2);
    p.lse_ref_c = reinterpret_cast<float*>(ws + L.lse_ref_c);
    p.kl_c = reinterpret_cast<float*>(ws + L.kl_c);
    p.cb_c = reinterpret_cast<float*>(ws + L.cb_c);
    p.kl_out = o.kl_out;
  }
  // merge of slab r (one sweep) or of all rows, then the loss and the coefficients of the backward pass
  LossFinish fin;
  fin.block_sums = reinterpret_cast<double*>(ws + L.block_sums);
  fin.ticket = reinterpret_cast<unsigned*>(reinterpret_cast<char*>(c->dstatus) + kTicketOffset);
  fin.loss = loss;
  fin.metrics = o.metrics_out;
  auto merge_and_loss = [&](int r) {
    const int slabs = sweep ? L.n_row_slabs : 1;
    const int64_t rows = sweep ? L.Ts : T;
    const int ranges = shard ? 0 : L.part_ranges;
    const int nb = merge_blocks(rows, slabs, ranges);
    const int pr_loss = prof_begin(c, 6);
    if (!seq_path) {
      p.fin = fin;
      p.fin.base = r * nb;
      p.fin.total = slabs * nb;
      launch_merge(c, p, rows, ranges, slabs);
    } else {
      // merge the statistics first, then one team per response forms weights, ratios and the loss; valid rows that lie
      // outside every response range take no part: their coefficients stay 0
      p.with_loss = 0;
      p.zero_coef = 1;
      launch_merge(c, p, rows, ranges, slabs);
      SeqParams q;
      memset(&q, 0, sizeof(q));
      q.seq_offsets = o.seq_offsets;
      q.n_seq = (int)o.n_seq;
      q.agg_mode = o.token_weight ? 0 : o.agg_mode;
      q.sequence_level = o.sequence_level ? 1 : 0;
      q.row_map = p.row_map;
      q.logp_c = p.logp_c;
      q.ent_c = p.ent_c;
      q.old_logp = old_logp;
      q.ref_logp = ref_logp;
      q.adv = adv;
      q.token_weight = o.token_weight;
      q.eps_low = eps_low; q.eps_high = eps_high; q.beta = beta; q.ent_coef = o.ent_coef;
      q.l_max = reinterpret_cast<int*>(reinterpret_cast<char*>(c->dstatus) + 96);
      q.cp_c = p.cp_c;
      q.ce_c = p.ce_c;
      q.fin = fin;
      q.fin.base = 0;
      if (q.agg_mode == 2) {
        launch(c, seq_lmax_kernel, 1, 1024, o.seq_offsets, (int)o.n_seq, q.l_max);
        c->launches++;
      }
      // A block per response, else a warp.  Merge and loss, block against warp: 64 responses 16.9 / 18.5 / 22.8 / 34 us against 17.1 /
      // 21.0 / 43 / 134 at 128 / 256 / 1024 / 4096 rows, 512 responses 22.8 / 25.2 / 34 / 72 against 21.0 / 27.1 / 56 / 204; 1024
      // responses 31.7 / 38.7 / 45.7 / 53 against 21.0 / 28.6 / 40.0 / 62 at 64 / 256 / 512 / 1024 rows, 8192 responses of 256 rows 190 against 79.
      const bool by_block = T >= 128 * o.n_seq && (o.n_seq <= (int64_t)c->n_sm * 4 || T >= 1024 * o.n_seq);
      const int64_t teams = by_block ? o.n_seq : (o.n_seq + kLossThreads / 32 - 1) / (kLossThreads / 32);
      q.fin.total = (int)(teams < 1024 ? teams : 1024);
      if (by_block) launch(c, seq_loss_kernel<kLossThreads>, q.fin.total, kLossThreads, q, c->dstatus);
      else          launch(c, seq_loss_kernel<32>, q.fin.total, kLossThreads, q, c->dstatus);
      c->launches++;
    }
    prof_end(c, pr_loss, 6);
  };
  if (!sweep) merge_and_loss(0);
  // ---- backward, one (row slab x vocabulary slab) at a time
  __nv_bfloat16* Hc = reinterpret_cast<__nv_bfloat16*>(ws + L.Hc);
  __nv_bfloat16* G = reinterpret_cast<__nv_bfloat16*>(ws + L.G);
  float* dH_acc = reinterpret_cast<float*>(ws + L.dH_acc);
  const int* row_map = reinterpret_cast<const int*>(ws + L.row_map);
  const int* n_valid = &c->dstatus->n_valid;

  CUtensorMap tmHc_k, tmW_k, tmG_k, tmW_mn, tmG_mn, tmHc_mn, tm_dH, tm_dW, tm_G_out, tmHr_k, tmWr_k, tm_slots, tmW_fwd,
      tmWr_fwd, tm_planes;
  if (o.kl_full) {
    if (!map_kmajor(c, &tmHr_k, ws + L.Hc_ref, (uint64_t)L.Tpad, (uint64_t)o.d_ref, (uint64_t)o.d_ref, BM) ||
        !map_kmajor(c, &tmWr_k, o.W_ref, (uint64_t)V, (uint64_t)o.d_ref, (uint64_t)o.ldW_ref, b_box_rows(c)))
      return RL_ERR_CUDA;
  }
  bool ok = map_kmajor(c, &tmHc_k, Hc, (uint64_t)L.Tpad, (uint64_t)d, (uint64_t)d, BM) &&
            map_kmajor(c, &tmW_k, W, (uint64_t)V, (uint64_t)d, (uint64_t)ldW, b_box_rows(c)) &&
            map_kmajor(c, &tmG_k, G, (uint64_t)L.Ts, (uint64_t)L.Vs, (uint64_t)L.Vs, BM) &&
            map_mnmajor(c, &tmW_mn, W, (uint64_t)V, (uint64_t)d, (uint64_t)ldW, b_box_panels(c)) &&
            map_mnmajor(c, &tmG_mn, G, (uint64_t)L.Ts, (uint64_t)L.Vs, (uint64_t)L.Vs, BM / 64) &&
            map_mnmajor(c, &tmHc_mn, Hc, (uint64_t)L.Tpad, (uint64_t)d, (uint64_t)d, b_box_panels(c)) &&
            map_out_bf16(c, &tm_G_out, G, (uint64_t)L.Ts, (uint64_t)L.Vs, (uint64_t)L.Vs) &&
            map_out_f32(c, &tm_dH, dH_acc, (uint64_t)L.Ts, (uint64_t)d, (uint64_t)d, (uint64_t)dh_buffers(c), (uint64_t)L.Ts) &&
            map_out_f32(c, &tm_dW, dW, (uint64_t)V, (uint64_t)d, (uint64_t)d, 1, (uint64_t)V);
  const int dh_tile_rows = BM * c->cta_group, dh_cols = dh_tile_cols(c, d);
  const int dh_workers = c->grid[c->cta_group] / c->cta_group;
  float* dH_slots = reinterpret_cast<float*>(ws + L.dH_slots);
  tm_slots = tm_dH;
  if (L.dH_slots)
    ok = ok && map_out_f32(c, &tm_slots, dH_slots, (uint64_t)dh_tile_rows, (uint64_t)dh_cols, (uint64_t)dh_cols,
                           (uint64_t)2 * dh_workers, (uint64_t)dh_tile_rows);
  const int cg_fwd = fwd_cta_group(c, L);
  tmW_fwd = tmW_k;
  if (cg_fwd != c->cta_group)
    ok = ok && map_kmajor(c, &tmW_fwd, W, (uint64_t)V, (uint64_t)d, (uint64_t)ldW, b_box_rows(cg_fwd));
  tmWr_fwd = tmWr_k;
  if (o.kl_full && cg_fwd != c->cta_group)
    ok = ok && map_kmajor(c, &tmWr_fwd, o.W_ref, (uint64_t)V, (uint64_t)o.d_ref, (uint64_t)o.ldW_ref, b_box_rows(cg_fwd));
  tm_planes = tm_G_out;
  if (sweep) ok = ok && map_out_planes(c, &tm_planes, G, (uint64_t)L.Ts, (uint64_t)L.Vs);
  if (!ok) return RL_ERR_CUDA;

  const int n_row_slabs = L.n_row_slabs;
  const int n_col_slabs = (int)((V + L.Vs - 1) / L.Vs);
  const int d_tiles = (int)((d + BN - 1) / BN);
  int hook_slab = 0;
  const bool dH_beside = dH_beside_dW(c, T, d, V - (int64_t)(n_col_slabs - 1) * L.Vs);
  // Slabs are sized for T rows, and how many of them have any is known to the device alone.  Whoever wants to be told as rows of dW
  // are completed has them walked from the last to the first, so that the one that completes them has rows: its dW launches, in
  // pieces and before its dH, are what is told about while they and dH still run.
  const bool reverse = c->dw_hook && n_row_slabs > 1;
  for (int q = 0; q < n_row_slabs; ++q) {
    const int r = reverse ? n_row_slabs - 1 - q : q;
    GemmShape dh_shape;
    memset(&dh_shape, 0, sizeof(dh_shape));
    DhSource src;
    src.acc = dH_acc;
    src.d = (int)d;
    src.cg = c->cta_group;
    src.workers = dh_workers;
    src.split_stride = (long long)L.Ts * d;
    src.slots = dH_slots;
    src.tile_rows = dh_tile_rows;
    src.tile_cols = dh_cols;
    src.row_map = row_map;
    src.dH = dH;
    src.f32 = o.dH_dtype;
    const int rows_cap = L.Ts;   // the valid rows are cut into equal slabs of at most Ts rows on the device
    // stream-K parts that finish a tile are added to the second accumulator buffer: it starts at zero
    if (dh_uses_stream_k(c)) cudaMemsetAsync(dH_acc + (size_t)L.Ts * d, 0, (size_t)L.Ts * d * 4, st);
    for (int cs = 0; cs < n_col_slabs; ++cs) {
      const int vocab_base = cs * L.Vs;
      const int cols = (int)((V - vocab_base) < L.Vs ? (V - vocab_base) : L.Vs);
      // dH may form its operand itself where it comes next and takes its tiles whole or cut; whether it does is decided on the
      // device (feed_pays), and logit_grad_kernel has nothing to do then
      const bool report = c->dw_hook && q == n_row_slabs - 1;
      const bool fed = sweep && !report && !o.kl_full && dh_cuts_tiles(c) && (long long)L.Ts * L.Vs >= kFeedEntries;
      // how tiles of dH are cut depends only on rows, d tiles and grid: same for every column slab
      dh_shape.n_valid = n_valid;
      dh_shape.m_rows_cap = rows_cap; dh_shape.m_dyn = 1; dh_shape.slab_cap = L.Tc; dh_shape.slab_one = L.Ts; dh_shape.slab_index = r;
      dh_shape.k_cap = cols;
      dh_shape.n_tiles = (int)((d + dh_cols - 1) / dh_cols);
      dh_shape.n_range = 1;
      dh_shape.b_k_off = vocab_base;
      dh_shape.n_fastest = 1;   // the CTAs that share a panel of G rows run together
      dh_shape.k_split_max = c->dh_k_slices;
      dh_shape.stream_k = dh_uses_stream_k(c) ? 1 : (L.dH_slots ? 2 : 0);
      FeedParams lg;
      memset(&lg, 0, sizeof(lg));
      // (1) the slab's G = dloss/dlogits as bf16: from the logits of a first pass, or by forming them again
      {
        if (sweep) {
          GemmShape sw;
          memset(&sw, 0, sizeof(sw));
          sw.n_valid = n_valid;
          sw.m_rows_cap = rows_cap; sw.m_dyn = 1; sw.slab_cap = L.Tc; sw.slab_one = L.Ts; sw.slab_index = r;
          sw.k_cap = (int)d;
          sw.n_tiles = (cols + BN - 1) / BN;
          sw.n_split_max = L.part_ranges;
          sw.leaves_ranges = 1;
          sw.a_mn_slab = 1;
          sw.m_group = row_group_tiles(c, d);
          float* zr = reinterpret_cast<float*>(ws + L.zr);
          uint16_t* z_hi = reinterpret_cast<uint16_t*>(G);
          uint16_t* z_lo = z_hi + (size_t)L.Ts * L.Vs;
          if (o.kl_full) {
            GemmShape sr = sw;
            sr.k_cap = (int)o.d_ref;
            sr.m_group = row_group_tiles(c, o.d_ref);
            EpiRefSweep::Params er;
            er.partials2 = reinterpret_cast<float4*>(ws + L.partials2);
            er.part_stride = L.Tpad;
            er.V = (int)V;
            er.slab = zr;
            er.ld = L.Vs;
            launch_gemm<EpiRefSweep, 0, 0>(c, cg_fwd, 0, tmHr_k, tmWr_fwd, tm_G_out, tm_G_out, sr, er);
          }
          RowStats::Params ep;
          ep.tokens_c = reinterpret_cast<const int*>(ws + L.tokens_c);
          ep.partials = reinterpret_cast<float4*>(ws + L.partials);
          ep.part_stride = L.Tpad;
          ep.V = (int)V;
          if (o.kl_full) {
            EpiSweepKL::Params ek;
            ek.stats = ep;
            ek.partials2 = reinterpret_cast<float4*>(ws + L.partials2);
            ek.zr = zr;
            ek.hi = z_hi;
            ek.lo = z_lo;
            ek.ld = L.Vs;
            launch_gemm<EpiSweepKL, 0, 0>(c, cg_fwd, 0, tmHc_k, tmW_fwd, tm_G_out, tm_G_out, sw, ek);
          } else {
            launch_gemm<EpiSweep, 0, 0>(c, cg_fwd, 0, tmHc_k, tmW_fwd, tm_planes, tm_planes, sw, ep);
          }
          p.slab_cap = L.Tc; p.slab_one = L.Ts;
          p.slab_index = r;
          p.clear = reinterpret_cast<uint4*>(ws + L.feed);
          p.n_clear = fed ? (int)(L.feed_bytes / 16) : 0;
          merge_and_loss(r);
          lg.slab = z_hi;
          lg.lo = z_lo;
          lg.ld = L.Vs;
          lg.V = (int)V;
          lg.slab_cap = L.Tc; lg.slab_one = L.Ts; lg.slab_index = r;
          lg.tokens_c = ep.tokens_c;
          lg.lse = p.lse_c; lg.ent = p.ent_c; lg.cp = p.cp_c; lg.ce = p.ce_c;
          lg.zr = zr;
          lg.lse_ref = p.lse_ref_c; lg.kl = p.kl_c; lg.cb = p.cb_c;
          if (fed) {
            lg.dh = dh_shape;
            lg.cg = c->cta_group;
            lg.workers = dh_workers;
            lg.ticket = reinterpret_cast<unsigned*>(ws + L.feed);
            lg.ready = lg.ticket + 4;
          }
          {
            const int pr_lg = prof_begin(c, 1);
            const long long padded = (long long)align_up(rows_cap, 128);
            const int unit = 256 * (o.kl_full ? kGradVecs<true> : kGradVecs<false>);
            long long grad_blocks = (padded * ((L.Vs + unit - 1) / unit) + 7) / 8;   // a warp each
            // many waves of blocks; two where dH may do it, 50 us of blocks that find nothing to do otherwise (6912 rows, d = 2048:
            // 11.03 -> 10.98 ms; 2000 and 4096 rows, which it does not do, level)
            const int most = c->n_sm * (fed ? 6 : 64);
            if (grad_blocks > most) grad_blocks = most;
            const LogitGradParams& alone = lg;
            if (fed)            launch(c, logit_grad_kernel<false, FeedParams>, (int)grad_blocks, 256, lg, c->dstatus);
            else if (o.kl_full) launch(c, logit_grad_kernel<true, LogitGradParams>, (int)grad_blocks, 256, alone, c->dstatus);
            else                launch(c, logit_grad_kernel<false, LogitGradParams>, (int)grad_blocks, 256, alone, c->dstatus);
            prof_end(c, pr_lg, 1);
            c->launches++;
          }
        } else {
          GemmShape sh;
          memset(&sh, 0, sizeof(sh));
          sh.n_valid = n_valid;
          sh.m_rows_cap = rows_cap; sh.m_dyn = 1; sh.slab_cap = L.Tc; sh.slab_one = L.Ts; sh.slab_index = r;
          sh.k_cap = (int)d;
          sh.n_tiles = (cols + BN - 1) / BN;
          sh.n_range = 0; sh.n_range_lo = 1; sh.n_range_hi = kFwdRange; sh.n_range_always = 1;   // chosen on the device
          sh.a_mn_slab = 1;
          sh.b_mn_off = vocab_base;
          sh.m_group = row_group_tiles(c, d + (o.kl_full ? o.d_ref : 0));
          if (!o.kl_full) {
            GradParams ep;
            ep.tokens_c = reinterpret_cast<const int*>(ws + L.tokens_c);
            ep.lse = p.lse_c; ep.ent = p.ent_c; ep.cp = p.cp_c; ep.ce = p.ce_c;
            ep.V = (int)V; ep.vocab_base = vocab_base;
            if (d <= kEightWarpsMaxK)
              launch_gemm<EpiGrad<8>, 0, 0>(c, c->cta_group, 1, tmHc_k, tmW_k, tm_G_out, tm_G_out, sh, ep);
            else
              launch_gemm<EpiGrad<4>, 0, 0>(c, c->cta_group, 1, tmHc_k, tmW_k, tm_G_out, tm_G_out, sh, ep);
          } else {
            EpiGradKL::Params ep;
            ep.tokens_c = reinterpret_cast<const int*>(ws + L.tokens_c);
            ep.lse = p.lse_c; ep.lse_ref = p.lse_ref_c; ep.ent = p.ent_c; ep.kl = p.kl_c;
            ep.cp = p.cp_c; ep.cb = p.cb_c; ep.ce = p.ce_c;
            ep.V = (int)V; ep.vocab_base = vocab_base;
            launch_dual<EpiGradKL>(c, 1, tmHc_k, tmW_k, tmHr_k, tmWr_k, tm_G_out, sh, (int)o.d_ref, ep);
          }
        }
      }
      // (2) dH_slab (+)= G * W_slab        [rows x d], K = vocabulary columns of the slab
      auto launch_dH = [&]() {
        const GemmShape& sh = dh_shape;
        AccParams ep = {};
        ep.n_cols = (int)d; ep.accumulate = cs > 0; ep.row_base = 0; ep.slice_add = sh.stream_k == 1;
        ep.tile_cols = sh.stream_k == 2 ? dh_cols : 0;
        ep.tile_rows = dh_tile_rows;
        auto tiles = [&](auto epi, const auto& params) {
          using Epi = decltype(epi);
          if (use_wide(c, d)) launch_wide<Epi, 0, 1>(c, 2, tmG_k, tmW_mn, tm_dH, tm_slots, sh, params);
          else launch_gemm<Epi, 0, 1>(c, c->cta_group, 2, tmG_k, tmW_mn, tm_dH, tm_slots, sh, params);
        };
        if (fed) {
          EpiAccFed::Params params = {};
          static_cast<AccParams&>(params) = ep;
          params.grad = lg;
          tiles(EpiAccFed(), params);
        } else {
          tiles(EpiAcc(), ep);
        }
      };
      // (3) dW_slab (+)= G^T * H_slab      [vocabulary rows x d], K = valid rows of the slab
      if (!report) launch_dH();
      const int step = report && cols > kSlabColsMax ? kSlabColsMax : cols;
      for (int c0 = 0; c0 < cols; c0 += step) {
        GemmShape sh;
        memset(&sh, 0, sizeof(sh));
        sh.n_valid = n_valid;
        sh.m_rows_cap = cols - c0 < step ? cols - c0 : step;
        sh.k_cap = rows_cap; sh.k_dyn = 1; sh.slab_cap = L.Tc; sh.slab_one = L.Ts; sh.slab_index = r;
        sh.n_tiles = d_tiles;
        sh.n_range = 1;
        sh.skip_if_k0 = (r > 0 || o.accumulate_dW) ? 1 : 0;
        sh.a_mn_off = c0;
        sh.b_k_slab = 1;
        sh.n_fastest = 1;
        AccParams ep = {};
        ep.n_cols = (int)d; ep.accumulate = o.accumulate_dW ? 1 : reverse ? 2 : (r > 0 ? 1 : 0);
        ep.n_valid = n_valid; ep.slab_cap = L.Tc; ep.slab_one = L.Ts; ep.slab_index = r;
        ep.row_base = vocab_base + c0; ep.slice_add = 0; ep.tile_cols = 0;
        if (dH_beside && !report && cs == n_col_slabs - 1) {
          src.shape = dh_shape;
          auto dW_and_dH = [&](auto epi) {
            typename decltype(epi)::Params es = {};
            static_cast<AccParams&>(es) = ep;
            es.dh = src;
            launch_gemm<decltype(epi), 1, 1>(c, c->cta_group, 3, tmG_mn, tmHc_mn, tm_dW, tm_dW, sh, es);
          };
          // (a worker with one or two tiles has nothing for more epilogue warps to overlap: the smallest step 52.2 -> 52.9 us)
          const long long tiles = (long long)d_tiles * ((cols + BN - 1) / BN);
          if (T <= kFewRows && tiles >= 4 * dh_workers) dW_and_dH(EpiAccScatter<8>());
          else                                          dW_and_dH(EpiAccScatter<4>());
        } else {
          launch_gemm<EpiAcc, 1, 1>(c, c->cta_group, 3, tmG_mn, tmHc_mn, tm_dW, tm_dW, sh, ep);
        }
        // these rows of dW are complete once the row slab that is walked last has added to them
        if (report) {
          const int64_t row0 = (int64_t)vocab_base + c0;
          c->dw_hook(c->dw_hook_user, hook_slab++, row0, row0 + sh.m_rows_cap);
        }
      }
      if (report) launch_dH();
    }
    // dW of the last column slab has written dH in passing, unless it came before dH or is too short for that
    if (!dH_beside || (c->dw_hook && q == n_row_slabs - 1)) {
      src.shape = dh_shape;
      const int pr_sc = prof_begin(c, 7);
      launch(c, scatter_dH_kernel, c->n_sm * 8, 256, src, c->dstatus);
      prof_end(c, pr_sc, 7);
      c->launches++;
    }
  }
  return cuda_ok();
}

rl_status rl_policy_loss_fwd_bwd_ex(rl_ctx* c, const void* H, int64_t ldH, const void* W, int64_t ldW,
                                    const int32_t* tokens, const float* old_logp, const float* ref_logp,
                                    const float* adv, const uint8_t* mask, int64_t T, int64_t d, int64_t V,
                                    float eps_low, float eps_high, float beta, float* loss, void* dH, float* dW,
                                    const rl_loss_opts* opts) {
  return loss_fwd_bwd_impl(c, H, ldH, W, ldW, tokens, old_logp, ref_logp, adv, mask, T, d, V, eps_low, eps_high, beta,
                           loss, dH, dW, opts, nullptr);
}

rl_status rl_policy_loss_shard_bwd(rl_ctx* c, const void* H, int64_t ldH, const void* W_shard, int64_t ldW,
                                   const int32_t* tokens, const float* old_logp, const float* ref_logp,
                                   const float* adv, const uint8_t* mask, int64_t T, int64_t d, int64_t V_shard,
                                   int64_t vocab_offset, int64_t V_total, const float* logp, const float* entropy,
                                   const float* lse, float eps_low, float eps_high, float beta, float* loss,
                                   void* dH_partial, float* dW_shard, const rl_loss_opts* opts) {
  ShardArgs sh;
  sh.vocab_off = vocab_offset;
  sh.V_total = V_total;
  sh.logp = logp;
  sh.entropy = entropy;
  sh.lse = lse;
  return loss_fwd_bwd_impl(c, H, ldH, W_shard, ldW, tokens, old_logp, ref_logp, adv, mask, T, d, V_shard, eps_low,
                           eps_high, beta, loss, dH_partial, dW_shard, opts, &sh);
}

rl_status rl_shard_logit_stats(rl_ctx* c, const void* H, int64_t ldH, const void* W_shard, int64_t ldW,
                               const int32_t* tokens, const uint8_t* mask, int64_t T, int64_t d, int64_t V_shard,
                               int64_t vocab_offset, int64_t V_total, float* stats) {
  if (!c) return RL_ERR_INVALID_ARG;
  rl_status s = check_hw(H, ldH, W_shard, ldW, T, d, V_shard);
  if (s != RL_OK) return s;
  if (vocab_offset < 0 || V_total < vocab_offset + V_shard || V_total >= (int64_t(1) << 30)) return RL_ERR_SHAPE;
  if (T == 0) return RL_OK;
  if (!tokens || !stats) return RL_ERR_INVALID_ARG;
  if (reinterpret_cast<uintptr_t>(stats) & 15) return RL_ERR_ALIGNMENT;
  const WsLayout L = ws_layout(c, T, d, V_shard, false);
  if ((s = check_ws(c, L.G)) != RL_OK) return s;   // the forward arrays
  char* ws = static_cast<char*>(c->ws);
  FwdPlan plan;
  plan.vocab_off = vocab_offset;
  plan.V_total = V_total;
  plan.out.stats = reinterpret_cast<float4*>(stats);
  if ((s = run_forward(c, L, H, ldH, W_shard, ldW, tokens, mask, T, d, V_shard, nullptr, plan)) != RL_OK)
    return s;
  LossParams p;
  memset(&p, 0, sizeof(p));
  p.partials = reinterpret_cast<const float4*>(ws + L.partials);
  p.part_stride = L.Tpad;
  p.row_map = reinterpret_cast<const int*>(ws + L.row_map);
  p.stats_out = reinterpret_cast<float4*>(stats);
  const int pr = prof_begin(c, 6);
  launch_merge(c, p, T, L.part_ranges);
  prof_end(c, pr, 6);
  return cuda_ok();
}

rl_status rl_merge_logit_stats(rl_ctx* c, const float* stats, int n_shards, const uint8_t* mask, int64_t T,
                               float* logp, float* entropy, float* lse) {
  if (!c || T < 0 || n_shards < 1 || n_shards > 4096) return RL_ERR_INVALID_ARG;
  if (T == 0) return RL_OK;
  if (!stats || !logp) return RL_ERR_INVALID_ARG;
  if (reinterpret_cast<uintptr_t>(stats) & 15) return RL_ERR_ALIGNMENT;
  int blocks = (int)((T + 255) / 256);
  if (blocks > 4096) blocks = 4096;
  const int pr = prof_begin(c, 6);
  launch(c, merge_shard_stats_kernel, blocks, 256, reinterpret_cast<const float4*>(stats), n_shards, (long long)T, mask, logp, entropy, lse);
  prof_end(c, pr, 6);
  c->launches++;
  return cuda_ok();
}

rl_status rl_token_logprobs_multi(rl_ctx* c, int n_models, const void* const* H, const int64_t* ldH,
                                  const void* const* W, const int64_t* ldW, const int64_t* d,
                                  const int32_t* tokens, const uint8_t* mask, int64_t T, int64_t V,
                                  float* const* logp, float* const* entropy) {
  if (!c || n_models < 1 || n_models > 16 || !H || !ldH || !W || !ldW || !d || !logp) return RL_ERR_INVALID_ARG;
  int64_t d_max = 0;
  for (int i = 0; i < n_models; ++i) {
    rl_status s = check_hw(H[i], ldH[i], W[i], ldW[i], T, d[i], V);
    if (s != RL_OK) return s;
    if (T > 0 && !logp[i]) return RL_ERR_INVALID_ARG;
    d_max = d[i] > d_max ? d[i] : d_max;
  }
  if (T == 0) return RL_OK;
  if (!tokens) return RL_ERR_INVALID_ARG;
  // one layout for all models: the compacted rows of the widest model fix the offsets
  const WsLayout L = ws_layout(c, T, d_max, V, false);
  rl_status s = check_ws(c, L.G);   // the forward arrays
  if (s != RL_OK) return s;
  char* ws = static_cast<char*>(c->ws);
  for (int i = 0; i < n_models; ++i) {
    FwdPlan plan;
    plan.out.value[0] = logp[i]; plan.out.value[1] = entropy ? entropy[i] : nullptr;
    plan.scan = i == 0;   // the mask is scanned once; every model reuses the row map
    if ((s = run_forward(c, L, H[i], ldH[i], W[i], ldW[i], tokens, mask, T, d[i], V, nullptr, plan)) != RL_OK)
      return s;
    LossParams p;
    memset(&p, 0, sizeof(p));
    p.partials = reinterpret_cast<const float4*>(ws + L.partials);
    p.part_stride = L.Tpad;
    p.row_map = reinterpret_cast<const int*>(ws + L.row_map);
    p.lse_c = reinterpret_cast<float*>(ws + L.lse_c);
    p.ent_c = reinterpret_cast<float*>(ws + L.ent_c);
    p.logp_out = logp[i];
    p.ent_out = entropy ? entropy[i] : nullptr;
    launch_merge(c, p, T, L.part_ranges);
  }
  return cuda_ok();
}

rl_status rl_policy_loss_fwd_bwd(rl_ctx* c, const void* H, int64_t ldH, const void* W, int64_t ldW,
                                 const int32_t* tokens, const float* old_logp, const float* ref_logp,
                                 const float* adv, const uint8_t* mask, int64_t T, int64_t d, int64_t V,
                                 float eps_low, float eps_high, float beta, float* loss, void* dH, float* dW) {
  return rl_policy_loss_fwd_bwd_ex(c, H, ldH, W, ldW, tokens, old_logp, ref_logp, adv, mask, T, d, V, eps_low,
                                   eps_high, beta, loss, dH, dW, nullptr);
}

// Arguments of one host-buffer step (all per-step inputs are host pointers).
struct HostStepArgs {
  const void* H_host;
  int64_t ldH;
  const void* W;
  int64_t ldW;
  const int32_t* tokens_host;
  const float *old_host, *ref_host, *adv_host, *rewards_host;
  int64_t n_seq;
  int group_size;
  const int32_t* seq_offsets_host;
  const uint8_t* mask_host;
  int64_t T, d, V;
  float eps_low, eps_high, beta, ent_coef;
  void* dH;
  float* dW;
};

static rl_status host_step_check(const rl_ctx* c, const HostStepArgs& a) {
  if (!c) return RL_ERR_INVALID_ARG;
  if (a.T < 0 || a.d <= 0 || a.V <= 0) return RL_ERR_INVALID_ARG;
  if (a.T > 0 && (!a.H_host || !a.tokens_host || !a.old_host)) return RL_ERR_INVALID_ARG;
  if (a.T > 0 && !a.adv_host && (!a.rewards_host || !a.seq_offsets_host || a.n_seq <= 0 || a.n_seq > a.T))
    return RL_ERR_INVALID_ARG;
  if (a.ldH != a.d) return RL_ERR_SHAPE;  // host rows are copied as one block
  // everything the advantage and loss calls would refuse is refused here, before a copy is enqueued
  if (a.d % 64 != 0 || a.ldW < a.d || a.T >= (int64_t(1) << 30) || a.V >= (int64_t(1) << 30)) return RL_ERR_SHAPE;
  if (a.ldW % 8 != 0 || (reinterpret_cast<uintptr_t>(a.W) & 15) || (reinterpret_cast<uintptr_t>(a.dH) & 15) ||
      (reinterpret_cast<uintptr_t>(a.dW) & 15))
    return RL_ERR_ALIGNMENT;
  if (!a.W || !a.dW || (a.T > 0 && !a.dH)) return RL_ERR_INVALID_ARG;
  if (!(a.eps_low >= 0.f && a.eps_low < 1.f) || !(a.eps_high >= 0.f) || !(a.beta >= 0.f) || !(a.ent_coef >= 0.f))
    return RL_ERR_INVALID_ARG;
  if (a.beta != 0.f && a.T > 0 && !a.ref_host) return RL_ERR_INVALID_ARG;
  if (a.T > 0 && !a.adv_host && (a.group_size < 2 || a.n_seq % a.group_size != 0)) return RL_ERR_SHAPE;
  return RL_OK;
}

// Copies the step's inputs into the stage on `copy` (the context's stream itself, or the copy stream, in
// which case the context's stream waits for copy_done) and enqueues advantages + loss forward/backward on
// the context's stream; the result words end up in hs.out.
static rl_status host_step_enqueue(rl_ctx* c, const HostStage& hs, cudaStream_t copy, cudaEvent_t copy_done,
                                   const HostStepArgs& a) {
  const int64_t T = a.T;
  if (T > 0) {
    cudaMemcpyAsync(hs.H, a.H_host, (size_t)T * a.d * 2, cudaMemcpyHostToDevice, copy);
    cudaMemcpyAsync(hs.tok, a.tokens_host, (size_t)T * 4, cudaMemcpyHostToDevice, copy);
    cudaMemcpyAsync(hs.old_lp, a.old_host, (size_t)T * 4, cudaMemcpyHostToDevice, copy);
    if (a.ref_host) cudaMemcpyAsync(hs.ref_lp, a.ref_host, (size_t)T * 4, cudaMemcpyHostToDevice, copy);
    if (a.adv_host) {
      cudaMemcpyAsync(hs.adv, a.adv_host, (size_t)T * 4, cudaMemcpyHostToDevice, copy);
    } else {
      cudaMemcpyAsync(hs.rew, a.rewards_host, (size_t)a.n_seq * 4, cudaMemcpyHostToDevice, copy);
      cudaMemcpyAsync(hs.off, a.seq_offsets_host, (size_t)(a.n_seq + 1) * 4, cudaMemcpyHostToDevice, copy);
    }
    if (a.mask_host) cudaMemcpyAsync(hs.mask, a.mask_host, (size_t)T, cudaMemcpyHostToDevice, copy);
  }
  if (copy != c->stream) {
    if (cudaEventRecord(copy_done, copy) != cudaSuccess || cudaStreamWaitEvent(c->stream, copy_done, 0) != cudaSuccess)
      return RL_ERR_CUDA;
  }
  if (T > 0 && !a.adv_host) {
    rl_status sa = rl_grpo_advantages_ex(c, hs.rew, a.n_seq, a.group_size, 1, 1e-6f, hs.off, T, hs.advseq, hs.adv);
    if (sa != RL_OK) return sa;
  }
  rl_loss_opts opts;
  memset(&opts, 0, sizeof(opts));
  opts.struct_size = sizeof(opts);
  opts.ent_coef = a.ent_coef;
  opts.metrics_out = hs.out + 8;
  return rl_policy_loss_fwd_bwd_ex(c, hs.H, a.d, a.W, a.ldW, hs.tok, hs.old_lp, a.ref_host ? hs.ref_lp : nullptr, hs.adv,
                                   a.mask_host ? hs.mask : nullptr, T, a.d, a.V, a.eps_low, a.eps_high, a.beta, hs.out,
                                   a.dH, a.dW, &opts);
}

rl_status rl_policy_loss_fwd_bwd_host(rl_ctx* c, const void* H_host, int64_t ldH, const void* W, int64_t ldW,
                                      const int32_t* tokens_host, const float* old_host, const float* ref_host,
                                      const float* adv_host, const float* rewards_host, int64_t n_seq,
                                      int group_size, const int32_t* seq_offsets_host,
                                      const uint8_t* mask_host, int64_t T, int64_t d,
                                      int64_t V, float eps_low, float eps_high, float beta, float ent_coef,
                                      float* loss_host, float* metrics_host, void* dH, float* dW) {
  if (!loss_host) return RL_ERR_INVALID_ARG;
  const HostStepArgs a = {H_host, ldH, W, ldW, tokens_host, old_host, ref_host, adv_host, rewards_host, n_seq, group_size,
                          seq_offsets_host, mask_host, T, d, V, eps_low, eps_high, beta, ent_coef, dH, dW};
  rl_status s = host_step_check(c, a);
  if (s != RL_OK) return s;
  const WsLayout L = ws_layout(c, T, d, V, 1);
  if ((s = check_ws(c, L.total)) != RL_OK) return s;
  HostStage hs;
  carve_stage(static_cast<char*>(c->ws) + L.staging, T, d, &hs);
  if ((s = host_step_enqueue(c, hs, c->stream, nullptr, a)) != RL_OK) return s;
  float h_out[16];
  if (cudaMemcpyAsync(h_out, hs.out, sizeof(h_out), cudaMemcpyDeviceToHost, c->stream) != cudaSuccess) return RL_ERR_CUDA;
  if (cudaStreamSynchronize(c->stream) != cudaSuccess) return RL_ERR_CUDA;
  loss_host[0] = h_out[0];
  if (metrics_host) memcpy(metrics_host, h_out + 8, 32);
  return RL_OK;
}

rl_status rl_workspace_bytes_host_pipelined(rl_ctx* c, int64_t T, int64_t d, int64_t V, size_t* bytes) {
  if (!c || !bytes || T < 0 || d <= 0 || V <= 0) return RL_ERR_INVALID_ARG;
  *bytes = ws_layout(c, T, d, V, 2).total;
  return RL_OK;
}

rl_status rl_policy_loss_fwd_bwd_host_submit(rl_ctx* c, int slot, const void* H_host, int64_t ldH, const void* W,
                                             int64_t ldW, const int32_t* tokens_host, const float* old_host,
                                             const float* ref_host, const float* adv_host,
                                             const float* rewards_host, int64_t n_seq, int group_size,
                                             const int32_t* seq_offsets_host, const uint8_t* mask_host, int64_t T,
                                             int64_t d, int64_t V, float eps_low, float eps_high, float beta,
                                             float ent_coef, void* dH, float* dW) {
  const HostStepArgs a = {H_host, ldH, W, ldW, tokens_host, old_host, ref_host, adv_host, rewards_host, n_seq, group_size,
                          seq_offsets_host, mask_host, T, d, V, eps_low, eps_high, beta, ent_coef, dH, dW};
  rl_status s = host_step_check(c, a);
  if (s != RL_OK) return s;
  if (slot < 0 || slot > 1 || c->slot_busy[slot]) return RL_ERR_INVALID_ARG;
  const WsLayout L = ws_layout(c, T, d, V, 2);
  if ((s = check_ws(c, L.total)) != RL_OK) return s;
  if (!c->copy_stream) {
    // first pipelined call on this context: the copy stream, two events and 64 pinned bytes per slot;
    // all of it or none of it, so that a later call never finds a half-made set
    cudaStream_t cs = nullptr;
    cudaEvent_t ev[4] = {nullptr, nullptr, nullptr, nullptr};
    float* pin[2] = {nullptr, nullptr};
    bool ok = cudaStreamCreateWithFlags(&cs, cudaStreamNonBlocking) == cudaSuccess;
    for (int i = 0; i < 4 && ok; ++i) ok = cudaEventCreateWithFlags(&ev[i], cudaEventDisableTiming) == cudaSuccess;
    for (int i = 0; i < 2 && ok; ++i)
      ok = cudaHostAlloc(reinterpret_cast<void**>(&pin[i]), 64, cudaHostAllocDefault) == cudaSuccess;
    if (!ok) {
      for (int i = 0; i < 2; ++i) if (pin[i]) cudaFreeHost(pin[i]);
      for (int i = 0; i < 4; ++i) if (ev[i]) cudaEventDestroy(ev[i]);
      if (cs) cudaStreamDestroy(cs);
      cudaGetLastError();
      return RL_ERR_CUDA;
    }
    for (int i = 0; i < 2; ++i) { c->copy_done[i] = ev[2 * i]; c->step_done[i] = ev[2 * i + 1]; c->pinned_out[i] = pin[i]; }
    c->copy_stream = cs;
  }
  HostStage hs;
  const size_t stage = carve_stage(nullptr, T, d, nullptr);
  carve_stage(static_cast<char*>(c->ws) + L.staging + (size_t)slot * stage, T, d, &hs);
  // the stage of this slot is free: its previous step was waited for (slot_busy is clear)
  if ((s = host_step_enqueue(c, hs, c->copy_stream, c->copy_done[slot], a)) != RL_OK) return s;
  if (cudaMemcpyAsync(c->pinned_out[slot], hs.out, 64, cudaMemcpyDeviceToHost, c->stream) != cudaSuccess ||
      cudaEventRecord(c->step_done[slot], c->stream) != cudaSuccess)
    return RL_ERR_CUDA;
  c->slot_busy[slot] = 1;
  return RL_OK;
}

rl_status rl_policy_loss_fwd_bwd_host_wait(rl_ctx* c, int slot, float* loss_host, float* metrics_host) {
  if (!c || slot < 0 || slot > 1 || !loss_host || !c->slot_busy[slot]) return RL_ERR_INVALID_ARG;
  if (cudaEventSynchronize(c->step_done[slot]) != cudaSuccess) return RL_ERR_CUDA;
  c->slot_busy[slot] = 0;
  loss_host[0] = c->pinned_out[slot][0];
  if (metrics_host) memcpy(metrics_host, c->pinned_out[slot] + 8, 32);
  return RL_OK;
}

rl_status rl_debug_schedule(int64_t n_valid, int64_t rows_cap, int64_t k_len, int64_t n_tiles, int n_range,
                            int n_fastest, int m_group, int stream_k, int k_split_max, int cta_group,
                            int n_workers, int32_t* units, int64_t max_units, int64_t* n_units) {
  if (!n_units || n_valid < 0 || rows_cap <= 0 || k_len < 0 || n_tiles <= 0 || n_workers <= 0 || max_units < 0 ||
      (cta_group != 1 && cta_group != 2) || (max_units > 0 && !units))
    return RL_ERR_INVALID_ARG;
  const int nv = (int)n_valid;
  GemmShape sh;
  memset(&sh, 0, sizeof(sh));
  sh.n_valid = &nv;
  sh.m_rows_cap = (int)rows_cap;
  sh.m_dyn = 1;
  sh.k_cap = (int)k_len;
  sh.n_tiles = (int)n_tiles;
  if (n_range >= 0) {
    sh.n_range = n_range;
  } else if (n_range <= -1000) {   // as the passes that form logits: at most -n_range - 1000 ranges per row tile
    sh.n_split_max = -n_range - 1000;
  } else if (n_range > -100) {   // as the gradient-of-the-logits pass: always chosen in [1, -n_range]
    sh.n_range_lo = 1; sh.n_range_hi = -n_range; sh.n_range_always = 1;
  } else {                       // as the forward pass: chosen in [8, -n_range - 100] when there is plenty of work
    sh.n_range_lo = kFwdRange; sh.n_range_hi = -n_range - 100;
  }
  sh.n_fastest = n_fastest;
  sh.m_group = m_group;
  sh.stream_k = stream_k;
  sh.k_split_max = k_split_max;
  const GemmExtents ex = gemm_extents(sh, nv, cta_group, n_workers);
  int64_t n = 0;
  for (int worker = 0; worker < n_workers; ++worker) {
    UnitWalk walk(sh, ex, worker, n_workers);
    int mu, nr, ks, kb0, kb1;
    while (walk.next(mu, nr, ks, kb0, kb1)) {
      if (n < max_units) {
        int32_t* o = units + n * 8;
        o[0] = worker; o[1] = mu; o[2] = nr * ex.n_range;
        o[3] = (nr + 1) * ex.n_range < sh.n_tiles ? (nr + 1) * ex.n_range : sh.n_tiles;
        o[4] = ks; o[5] = kb0; o[6] = kb1; o[7] = ex.k_blocks;
      }
      ++n;
    }
  }
  *n_units = n;
  return RL_OK;
}

// Extents of a dH pass over n_valid rows.
static GemmExtents dh_extents(int n_valid, int64_t k_len, int64_t n_tiles, int cta_group, int n_workers) {
  GemmShape sh;
  memset(&sh, 0, sizeof(sh));
  sh.m_rows_cap = n_valid;
  sh.m_dyn = 1;
  sh.k_cap = (int)k_len;
  sh.n_tiles = (int)n_tiles;
  sh.n_range = 1;
  sh.n_fastest = 1;
  sh.k_split_max = 1;
  sh.stream_k = 2;
  return gemm_extents(sh, n_valid, cta_group, n_workers);
}

rl_status rl_debug_tile_slots(int64_t n_valid, int64_t k_len, int64_t n_tiles, int cta_group, int n_workers, int32_t* slots,
                              int64_t max_slots, int64_t* n_slots) {
  if (!n_slots || n_valid <= 0 || k_len <= 0 || n_tiles <= 0 || n_workers <= 0 || max_slots < 0 ||
      (cta_group != 1 && cta_group != 2) || (max_slots > 0 && !slots))
    return RL_ERR_INVALID_ARG;
  const GemmExtents ex = dh_extents((int)n_valid, k_len, n_tiles, cta_group, n_workers);
  int64_t n = 0;
  auto put = [&](int tile, int slot) {
    if (n < max_slots) { slots[2 * n] = tile; slots[2 * n + 1] = slot; }
    ++n;
  };
  for (int r = 0; r < ex.cut; ++r)
    for (int s = 0; s < ex.cut_parts; ++s) {
      const CutSlots c = cut_slots(ex, n_workers, r, s);
      put(ex.n_units - ex.cut + r, c.main);
      for (int h = c.first; h <= c.last; ++h) put(ex.n_units - ex.cut + r, h);
    }
  *n_slots = n;
  return RL_OK;
}

rl_status rl_debug_feed_order(int64_t n_valid, int64_t k_len, int64_t ld, int64_t n_tiles, int cta_group, int n_workers,
                              int32_t* pairs, int64_t max_pairs, int64_t* n_pairs, int* pays) {
  if (!n_pairs || n_valid <= 0 || k_len <= 0 || ld < k_len || n_tiles <= 0 || n_workers <= 0 || max_pairs < 0 ||
      (cta_group != 1 && cta_group != 2) || (max_pairs > 0 && !pairs))
    return RL_ERR_INVALID_ARG;
  const GemmExtents ex = dh_extents((int)n_valid, k_len, n_tiles, cta_group, n_workers);
  const FeedOrder o = feed_order(ex, (int)n_valid, (int)ld, cta_group, n_workers);
  const int64_t n = (int64_t)o.m_tiles * o.chunks;
  for (int64_t q = 0; q < n && q < max_pairs; ++q) {
    int tile, chunk;
    feed_pair(ex, o, (int)q, tile, chunk);
    pairs[2 * q] = tile;
    pairs[2 * q + 1] = chunk;
  }
  *n_pairs = n;
  if (pays) *pays = feed_pays(ex, n_workers) ? 1 : 0;
  return RL_OK;
}

rl_status rl_debug_workspace(int64_t T, int64_t d, int64_t V, int64_t d_ref, int n_sm, int static_scratch, int64_t* bytes) {
  if (!bytes || T < 0 || d <= 0 || V <= 0 || d_ref < 0 || n_sm < 2) return RL_ERR_INVALID_ARG;
  rl_ctx c = {};
  c.n_sm = n_sm;
  c.slab_rows = kSlabRowsMax;
  c.slab_cols = kSlabColsMax;
  c.slab_auto = static_scratch ? 0 : 1;
  c.cta_group = static_scratch ? 1 : 2;
  c.dh_k_slices = 1;
  c.wide_tiles = static_scratch ? 0 : 1;
  c.fixed_scratch = static_scratch ? 1 : 0;
  c.grid_full[1] = n_sm;
  c.grid_full[2] = n_sm / 2 * 2;
  const WsLayout L = ws_layout(&c, T, d, V, 0, d_ref);
  bytes[0] = (int64_t)(d_ref > 0 || static_scratch ? L.total : ws_bytes(&c, T, d, V));
  bytes[1] = (int64_t)L.G;
  bytes[2] = (int64_t)(L.row_pos + (T > kPrepRows ? (size_t)T * 4 : 0));
  return RL_OK;
}

rl_status rl_selftest_wait_timeout(rl_ctx* c, int limit_ms) {
  if (!c || limit_ms < 1 || limit_ms > 1000) return RL_ERR_INVALID_ARG;
  wait_timeout_probe_kernel<<<1, 32, 0, c->stream>>>((unsigned long long)limit_ms * 1000000ull, c->dstatus);
  c->launches++;
  return cuda_ok();
}

rl_status rl_selftest_cluster_exchange(rl_ctx* c, int mode, int cluster_size, int iters, int bytes, int partner_xor,
                                       float* ms_host, int* n_clusters_host) {
  if (!c || !ms_host || (mode != 0 && mode != 1) || iters < 1 || iters > (1 << 20)) return RL_ERR_INVALID_ARG;
  if (cluster_size != 2 && cluster_size != 4 && cluster_size != 8) return RL_ERR_INVALID_ARG;
  size_t smem = 1024;
  if (mode == 0) {
    smem += (size_t)kProbeTile * kProbeTile * 6;
  } else {
    if (bytes < 16 || bytes % 16 != 0 || bytes > 48 * 1024 || partner_xor < 1 || partner_xor >= cluster_size)
      return RL_ERR_INVALID_ARG;
    smem += 4 * (size_t)bytes;
  }
  if (cudaFuncSetAttribute(cluster_exchange_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess)
    return RL_ERR_CUDA;
  cudaLaunchConfig_t cfg;
  memset(&cfg, 0, sizeof(cfg));
  cfg.gridDim = dim3(c->n_sm / cluster_size * cluster_size);
  cfg.blockDim = dim3(kProbeThreads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = c->stream;
  cudaLaunchAttribute attr;
  attr.id = cudaLaunchAttributeClusterDimension;
  attr.val.clusterDim.x = cluster_size;
  attr.val.clusterDim.y = 1;
  attr.val.clusterDim.z = 1;
  cfg.attrs = &attr;
  cfg.numAttrs = 1;
  int n_clusters = 0;
  if (cudaOccupancyMaxActiveClusters(&n_clusters, cluster_exchange_kernel, &cfg) != cudaSuccess || n_clusters < 1) {
    cudaGetLastError();
    return RL_ERR_UNSUPPORTED_ARCH;
  }
  if (n_clusters * cluster_size < (int)cfg.gridDim.x) cfg.gridDim = dim3(n_clusters * cluster_size);
  if (n_clusters_host) *n_clusters_host = (int)cfg.gridDim.x / cluster_size;
  float* sink = reinterpret_cast<float*>(reinterpret_cast<char*>(c->dstatus) + 128);   // never written in practice
  cudaEvent_t e0 = nullptr, e1 = nullptr;
  if (cudaEventCreate(&e0) != cudaSuccess || cudaEventCreate(&e1) != cudaSuccess) {
    if (e0) cudaEventDestroy(e0);
    return RL_ERR_CUDA;
  }
  rl_status rs = RL_OK;
  for (int pass = 0; pass < 2 && rs == RL_OK; ++pass) {   // one warm-up launch, one timed
    if (pass == 1) cudaEventRecord(e0, c->stream);
    if (cudaLaunchKernelEx(&cfg, cluster_exchange_kernel, mode, iters, bytes, partner_xor, sink, c->dstatus) != cudaSuccess)
      rs = RL_ERR_CUDA;
    c->launches++;
  }
  cudaEventRecord(e1, c->stream);
  if (rs == RL_OK && cudaEventSynchronize(e1) != cudaSuccess) rs = RL_ERR_CUDA;
  if (rs == RL_OK && cudaEventElapsedTime(ms_host, e0, e1) != cudaSuccess) rs = RL_ERR_CUDA;
  cudaEventDestroy(e0);
  cudaEventDestroy(e1);
  return rs;
}

rl_status rl_selftest_gemm(rl_ctx* c, const void* A, const void* B, float* C, int64_t M, int64_t N, int64_t K,
                           int a_mn, int b_mn, int accumulate) {
  if (!c || !A || !B || !C || M <= 0 || N <= 0 || K <= 0) return RL_ERR_INVALID_ARG;
  if (M % 128 != 0 || N % 256 != 0 || K % 8 != 0) return RL_ERR_SHAPE;
  CUtensorMap ta, tb;
  bool ok = a_mn ? map_mnmajor(c, &ta, A, (uint64_t)K, (uint64_t)M, (uint64_t)M, BM / 64)
                 : map_kmajor(c, &ta, A, (uint64_t)M, (uint64_t)K, (uint64_t)K, BM);
  ok = ok && (b_mn ? map_mnmajor(c, &tb, B, (uint64_t)K, (uint64_t)N, (uint64_t)N, b_box_panels(c))
                   : map_kmajor(c, &tb, B, (uint64_t)N, (uint64_t)K, (uint64_t)K, b_box_rows(c)));
  if (!ok) return RL_ERR_CUDA;
  GemmShape sh;
  memset(&sh, 0, sizeof(sh));
  sh.m_rows_cap = (int)M;
  sh.k_cap = (int)K;
  sh.n_tiles = (int)(N / BN);
  sh.n_range = 1;
  sh.n_fastest = 1;   // walk the column tiles of one row panel first, as the gradient passes do
  CUtensorMap tc;
  if (!map_out_f32(c, &tc, C, (uint64_t)M, (uint64_t)N, (uint64_t)N, 1, (uint64_t)M)) return RL_ERR_CUDA;
  AccParams ep = {};
  ep.n_cols = (int)N; ep.accumulate = accumulate; ep.row_base = 0; ep.slice_add = 0; ep.tile_cols = 0;
  if (c->wide_tiles && c->cta_group == 2 && !a_mn && b_mn) {   // the operand layout of dH, the one pass that has wide tiles
    sh.n_tiles = (int)((N + 2 * BN - 1) / (2 * BN));
    launch_wide<EpiAcc, 0, 1>(c, -1, ta, tb, tc, tc, sh, ep);
  } else if (!a_mn && !b_mn) launch_gemm<EpiAcc, 0, 0>(c, c->cta_group, -1, ta, tb, tc, tc, sh, ep);
  else if (!a_mn && b_mn) launch_gemm<EpiAcc, 0, 1>(c, c->cta_group, -1, ta, tb, tc, tc, sh, ep);
  else if (a_mn && !b_mn) launch_gemm<EpiAcc, 1, 0>(c, c->cta_group, -1, ta, tb, tc, tc, sh, ep);
  else launch_gemm<EpiAcc, 1, 1>(c, c->cta_group, -1, ta, tb, tc, tc, sh, ep);
  return cuda_ok();
}

// ---------------------------------------------------------------------------------------------
// Allocation-free variant of rl_token_logprobs.  Its scratch (compacted rows, row map, per-range
// softmax statistics, status word) lives in one file-scope device array instead of a caller
// workspace, so the call path contains no device allocation at all.
namespace {
constexpr size_t kStaticScratchBytes = size_t(16) << 20;   // 16 MiB per GPU that loads the library
constexpr size_t kStaticHeaderBytes = 256;                  // status word, then the workspace proper
constexpr int kStaticMaxDevices = 16;
static __device__ __align__(256) unsigned char g_static_scratch[kStaticScratchBytes];
struct StaticSlot {
  bool ready;
  rl_ctx ctx;
};
StaticSlot g_static_slot[kStaticMaxDevices];
std::mutex g_static_mutex;
}  // namespace

rl_status rl_token_logprobs_static(void* cuda_stream, const void* H, int64_t ldH, const void* W, int64_t ldW,
                                   const int32_t* tokens, const uint8_t* mask, int64_t T, int64_t d, int64_t V,
                                   float* logp, float* entropy, float* lse, int32_t* dev_status) {
  rl_status s = check_hw(H, ldH, W, ldW, T, d, V);
  if (s != RL_OK) return s;
  if (T > 0 && (!tokens || !logp)) return RL_ERR_INVALID_ARG;
  int device = -1;
  if (cudaGetDevice(&device) != cudaSuccess) return RL_ERR_CUDA;
  if (device < 0 || device >= kStaticMaxDevices) return RL_ERR_INVALID_ARG;
  std::lock_guard<std::mutex> lock(g_static_mutex);
  StaticSlot& slot = g_static_slot[device];
  if (!slot.ready) {
    // once per device, with that device current: the array's name is only a host-side handle;
    // the address kernels and memsets can use comes from cudaGetSymbolAddress
    int major = 0, n_sm = 0;
    if ((s = device_facts(device, &major, &n_sm)) != RL_OK) return s;
    unsigned char* base = nullptr;
    if (cudaGetSymbolAddress(reinterpret_cast<void**>(&base), g_static_scratch) != cudaSuccess || !base)
      return RL_ERR_CUDA;
    void* fn = nullptr;
    cudaDriverEntryPointQueryResult qres;
    if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &fn, cudaEnableDefault, &qres) != cudaSuccess || !fn ||
        qres != cudaDriverEntryPointSuccess)
      return RL_ERR_CUDA;
    if (set_smem_attr<EpiStats<4>, 0, 0>() != cudaSuccess || set_smem_attr<EpiStats<8>, 0, 0>() != cudaSuccess)
      return RL_ERR_CUDA;
    rl_ctx& c = slot.ctx;
    memset(&c, 0, sizeof(c));
    c.device = device;
    c.n_sm = n_sm;
    c.encode = reinterpret_cast<EncodeTiledFn>(fn);
    c.dstatus = reinterpret_cast<DevStatus*>(base);
    c.ws = base + kStaticHeaderBytes;
    c.ws_bytes = kStaticScratchBytes - kStaticHeaderBytes;
    c.slab_rows = kSlabRowsMax;
    c.slab_cols = kSlabColsMax;
    c.cta_group = 1;
    c.dh_k_slices = 1;
    c.dh_stream_k = 0;
    c.wide_tiles = 0;
    c.row_group_bytes = kRowGroupBytes;
    c.fixed_scratch = 1;
    c.grid[1] = c.n_sm;
    slot.ready = true;
  }
  rl_ctx* c = &slot.ctx;
  c->stream = static_cast<cudaStream_t>(cuda_stream);
  if (T == 0) {
    // nothing to compute, but the caller's status words must not keep stale contents
    if (dev_status && cudaMemsetAsync(dev_status, 0, 2 * sizeof(int32_t), c->stream) != cudaSuccess) return RL_ERR_CUDA;
    return RL_OK;
  }
  // only the forward part of the workspace layout is needed: everything before the gradient slab
  const WsLayout L = ws_layout(c, T, d, V, false);
  if (L.G > c->ws_bytes) return RL_ERR_WORKSPACE;
  char* ws = static_cast<char*>(c->ws);
  // the array keeps the previous call's contents: the status word and the valid-row count start at zero
  if (cudaMemsetAsync(c->dstatus, 0, sizeof(DevStatus), c->stream) != cudaSuccess) return RL_ERR_CUDA;
  FwdPlan plan;
  plan.out.value[0] = logp; plan.out.value[1] = entropy; plan.out.value[2] = lse;
  if ((s = run_forward(c, L, H, ldH, W, ldW, tokens, mask, T, d, V, nullptr, plan)) != RL_OK) return s;
  LossParams p;
  memset(&p, 0, sizeof(p));
  p.partials = reinterpret_cast<const float4*>(ws + L.partials);
  p.part_stride = L.Tpad;
  p.row_map = reinterpret_cast<const int*>(ws + L.row_map);
  p.with_loss = 0;
  p.lse_c = reinterpret_cast<float*>(ws + L.lse_c);
  p.ent_c = reinterpret_cast<float*>(ws + L.ent_c);
  p.logp_out = logp;
  p.ent_out = entropy;
  p.lse_out = lse;
  launch_merge(c, p, T, L.part_ranges);
  if (dev_status &&
      cudaMemcpyAsync(dev_status, c->dstatus, 2 * sizeof(int32_t), cudaMemcpyDeviceToDevice, c->stream) != cudaSuccess)
    return RL_ERR_CUDA;
  return cuda_ok();
}

}  // extern "C"
