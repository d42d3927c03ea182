// O(T) and O(B) kernels around the tensor-core passes: mask scan / row compaction
// (padding-free execution), GRPO advantages, merge of the per-range softmax statistics,
// per-token loss arithmetic with a deterministic two-stage reduction, and the final
// conversion of dH.  All of them are bandwidth- or latency-bound; loads are coalesced and
// vectorised where a row is wide enough to matter.
#pragma once
#include "logit_grad.cuh"

namespace rlh {

// ------------------------------------------------------------------------------------------
// Mask scan: row_map[i] = index of the i-th row with mask != 0 (ascending), n_valid = their number, and on request
// row_pos[t] = position of row t in the map, -1 for a masked row.  Each block owns 4096 consecutive rows, each thread 16
// of them (one 16-byte load when the mask is 16-byte aligned): (1) per-block counts, (2) every block adds up the counts
// before its own, scans its rows again and writes its indices.  From kScanSumBlocks blocks on, one block turns the counts
// into offsets in a launch between the two.  Up to kPrepRows rows none of this runs: prep_rows_kernel scans for itself.
constexpr int kScanSumBlocks = 1024;
constexpr int kScanThreads = 256;
constexpr int kScanRowsPerThread = 16;
constexpr int kScanRowsPerBlock = kScanThreads * kScanRowsPerThread;

// Bit i of the result = (mask[base + i] != 0), rows past T read as 0; mask == NULL means all valid.
__device__ __forceinline__ unsigned scan_load_bits(const uint8_t* __restrict__ mask, long long base, int T) {
  if (base >= T) return 0u;
  const int n = (int)min((long long)kScanRowsPerThread, (long long)T - base);
  if (!mask) return n == 16 ? 0xFFFFu : ((1u << n) - 1u);
  unsigned bits = 0;
  if (n == 16 && ((reinterpret_cast<uintptr_t>(mask + base) & 15) == 0)) {
    const uint4 q = __ldg(reinterpret_cast<const uint4*>(mask + base));
    const unsigned wds[4] = {q.x, q.y, q.z, q.w};
#pragma unroll
    for (int w = 0; w < 4; ++w)
#pragma unroll
      for (int b = 0; b < 4; ++b) bits |= ((wds[w] >> (8 * b)) & 0xFFu) ? (1u << (4 * w + b)) : 0u;
  } else {
    for (int i = 0; i < n; ++i) bits |= __ldg(mask + base + i) ? (1u << i) : 0u;
  }
  return bits;
}

__device__ __forceinline__ int block_exclusive_scan(int v, int* warp_sums, int* total) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  int incl = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int u = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += u;
  }
  if (lane == 31) warp_sums[warp] = incl;
  __syncthreads();
  if (warp == 0) {
    const int w = lane < (int)(blockDim.x >> 5) ? warp_sums[lane] : 0;
    int wi = w;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int u = __shfl_up_sync(0xffffffffu, wi, o);
      if (lane >= o) wi += u;
    }
    warp_sums[lane] = wi - w;
    if (lane == 31 && total) *total = wi;
  }
  __syncthreads();
  return warp_sums[warp] + incl - v;
}

__global__ void __launch_bounds__(kScanThreads) mask_count_kernel(const uint8_t* __restrict__ mask, int T,
                                                                  int* __restrict__ block_counts) {
  chain_begin();
  __shared__ int warp_sums[32];
  const long long base = ((long long)blockIdx.x * kScanThreads + threadIdx.x) * kScanRowsPerThread;
  int c = __popc(scan_load_bits(mask, base, T));
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) c += __shfl_xor_sync(0xffffffffu, c, o);
  if ((threadIdx.x & 31) == 0) warp_sums[threadIdx.x >> 5] = c;
  __syncthreads();
  if (threadIdx.x == 0) {
    int t = 0;
    for (int w = 0; w < kScanThreads / 32; ++w) t += warp_sums[w];
    block_counts[blockIdx.x] = t;
  }
}

// One block: block_counts[0..n) -> exclusive offsets in place, total -> st->n_valid.
__global__ void __launch_bounds__(1024) mask_offsets_kernel(int* __restrict__ block_counts, int n, DevStatus* st) {
  chain_begin();
  __shared__ int warp_sums[32];
  __shared__ int chunk_total;
  int carry = 0;
  for (int base = 0; base < n; base += 1024) {
    const int i = base + threadIdx.x;
    const int v = i < n ? block_counts[i] : 0;
    const int ex = block_exclusive_scan(v, warp_sums, &chunk_total);
    if (i < n) block_counts[i] = carry + ex;
    carry += chunk_total;
    __syncthreads();
  }
  if (threadIdx.x == 0) st->n_valid = carry;
}

// sums: block_offsets holds counts (to be added up here, total -> st->n_valid) instead of offsets.
__global__ void __launch_bounds__(kScanThreads) mask_write_kernel(const uint8_t* __restrict__ mask, int T,
                                                                  const int* __restrict__ block_offsets, int sums,
                                                                  int* __restrict__ row_map, int* __restrict__ row_pos,
                                                                  DevStatus* st) {
  chain_begin();
  __shared__ int warp_sums[32];
  __shared__ int block_total, before, all;
  __shared__ int staged[kScanRowsPerBlock];   // the block's valid rows, in order
  const long long base = ((long long)blockIdx.x * kScanThreads + threadIdx.x) * kScanRowsPerThread;
  unsigned bits = scan_load_bits(mask, base, T);
  int offset;
  if (sums) {
    if (threadIdx.x == 0) before = all = 0;
    __syncthreads();
    int c = 0, a = 0;
    for (int i = threadIdx.x; i < (int)gridDim.x; i += kScanThreads) {
      const int v = block_offsets[i];
      a += v;
      c += i < (int)blockIdx.x ? v : 0;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      c += __shfl_xor_sync(0xffffffffu, c, o);
      a += __shfl_xor_sync(0xffffffffu, a, o);
    }
    if ((threadIdx.x & 31) == 0) { atomicAdd(&before, c); atomicAdd(&all, a); }
    __syncthreads();
    offset = before;
    if (blockIdx.x == 0 && threadIdx.x == 0) st->n_valid = all;
  } else {
    offset = block_offsets[blockIdx.x];
  }
  int pos = block_exclusive_scan(__popc(bits), warp_sums, &block_total);
  if (row_pos) {
    int q = offset + pos;
#pragma unroll
    for (int i = 0; i < kScanRowsPerThread; ++i) {
      const bool v = (bits >> i) & 1u;
      if (base + i < T) row_pos[base + i] = v ? q : -1;
      q += v;
    }
  }
  while (bits) {
    const int i = __ffs(bits) - 1;
    bits &= bits - 1;
    staged[pos++] = (int)base + i;
  }
  __syncthreads();
  // coalesced copy of the block's indices to their place in the map
  int* dst = row_map + offset;
  for (int k = threadIdx.x; k < block_total; k += kScanThreads) dst[k] = staged[k];
}

// ------------------------------------------------------------------------------------------
// Row compaction: Hc[i,:] = H[row_map[i],:] for i < n_valid, zero rows up to the next multiple
// of 128 (so that tensor-core tiles never see stale data), compact token ids, and the
// token-range check.  One warp per row, 16-byte loads.  Token ids are checked against the whole
// vocabulary [0, V) and stored relative to vocab_off, the first id of the rows of W this call
// holds (0 unless the head is split by vocabulary): an id outside the held slice becomes a
// negative or too large column that no tile ever matches.  The rows are walked in their original order, so that the
// outputs of masked rows are zeroed in passing: nothing is cleared that is written again (a memset of dH cost as
// much as the copy itself, and each memset a launch).
// What a call returns per original row: zeroed where the mask is 0.
struct RowOutputs {
  void* dH;            // [T][dH_row_bytes], or NULL
  long long dH_row_bytes;
  float* value[4];     // [T] each, or NULL
  float4* stats;       // [T], or NULL
};

struct PrepParams {
  const __nv_bfloat16* H;
  long long ldH;
  int d;
  const uint8_t* mask;
  int T;
  int rows_per_block;     // scanning variant: at most 256
  const int* tokens;
  int V, vocab_off;
  __nv_bfloat16* Hc;
  int* tokens_c;
  int* row_map;           // written by the scanning variant
  const int* row_pos;     // read by the other
  RowOutputs out;
  unsigned* ticket;       // of the loss kernels that follow: cleared, whatever became of the call before
};

__device__ __forceinline__ void prep_row(const PrepParams& p, int t, int pos, int lane, DevStatus* st) {
  const int vec_per_row = p.d / 8;
  if (pos < 0) {
    if (p.out.dH) {
      uint4* q = reinterpret_cast<uint4*>(static_cast<char*>(p.out.dH) + (size_t)t * p.out.dH_row_bytes);
      const int n = (int)(p.out.dH_row_bytes / 16);
      for (int v = lane; v < n; v += 32) __stcs(q + v, make_uint4(0, 0, 0, 0));
    }
    if (lane < 4 && p.out.value[lane]) p.out.value[lane][t] = 0.f;
    if (lane == 4 && p.out.stats) p.out.stats[t] = make_float4(0.f, 0.f, 0.f, 0.f);
    return;
  }
  uint4* dst = reinterpret_cast<uint4*>(p.Hc + (size_t)pos * p.d);
  const uint4* src = reinterpret_cast<const uint4*>(p.H + (size_t)t * p.ldH);
#pragma unroll 8
  for (int v = lane; v < vec_per_row; v += 32) dst[v] = __ldg(src + v);
  if (lane == 0) {
    const int y = p.tokens[t];
    const bool in_range = y >= 0 && y < p.V;
    p.tokens_c[pos] = in_range ? y - p.vocab_off : -1;
    if (!in_range) latch_status(st, kStatusTokenRange, t);
  }
}

// SCAN: every block counts the mask itself (the rows before its own, and all of them), up to kPrepRows rows: one launch
// in place of three.  At 256 to 32768 rows the mask is 0.25 to 32 KB per block out of L2.
constexpr int kPrepRows = 32768;
template <bool SCAN>
__global__ void __launch_bounds__(256) prep_rows_kernel(const PrepParams p, DevStatus* st) {
  chain_begin();
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, warps = blockDim.x >> 5;
  if (blockIdx.x == 0 && threadIdx.x == 0) *p.ticket = 0;
  int n;
  if constexpr (SCAN) {
    __shared__ int warp_sums[32];
    __shared__ int before_s, all_s;
    __shared__ int pos_s[256];
    const int r0 = blockIdx.x * p.rows_per_block, rows = min(p.rows_per_block, p.T - r0);
    if (threadIdx.x == 0) before_s = all_s = 0;
    __syncthreads();
    int c = 0, a = 0;
    for (int g = threadIdx.x; g * 16 < p.T; g += blockDim.x) {
      const unsigned bits = scan_load_bits(p.mask, (long long)g * 16, p.T);
      const int before = r0 - g * 16;   // rows of this group that lie before the block's
      a += __popc(bits);
      c += before >= 16 ? __popc(bits) : (before > 0 ? __popc(bits & ((1u << before) - 1u)) : 0);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      c += __shfl_xor_sync(0xffffffffu, c, o);
      a += __shfl_xor_sync(0xffffffffu, a, o);
    }
    if (lane == 0) { atomicAdd(&before_s, c); atomicAdd(&all_s, a); }
    const int t = r0 + threadIdx.x;
    const bool valid = (int)threadIdx.x < rows && (!p.mask || p.mask[t] != 0);
    const int rank = block_exclusive_scan(valid ? 1 : 0, warp_sums, nullptr);
    const int pos = valid ? before_s + rank : -1;
    pos_s[threadIdx.x] = pos;
    if (valid) p.row_map[pos] = t;
    n = all_s;
    if (blockIdx.x == 0 && threadIdx.x == 0) st->n_valid = n;
    __syncthreads();
    for (int i = warp; i < rows; i += warps) prep_row(p, r0 + i, pos_s[i], lane, st);
  } else {
    n = st->n_valid;
    for (int t = blockIdx.x * warps + warp; t < p.T; t += gridDim.x * warps) prep_row(p, t, p.row_pos[t], lane, st);
  }
  const int n_pad = (n + 127) / 128 * 128;
  for (int i = n + blockIdx.x * warps + warp; i < n_pad; i += gridDim.x * warps) {
    uint4* dst = reinterpret_cast<uint4*>(p.Hc + (size_t)i * p.d);
    for (int v = lane; v < p.d / 8; v += 32) dst[v] = make_uint4(0, 0, 0, 0);
    if (lane == 0) p.tokens_c[i] = -1;
  }
}

// Row compaction of a second hidden-state matrix (the reference model's) with the same row map.
__global__ void __launch_bounds__(256) gather_plain_kernel(const __nv_bfloat16* __restrict__ H, long long ldH, int d,
                                                           const int* __restrict__ row_map,
                                                           __nv_bfloat16* __restrict__ Hc, const DevStatus* st) {
  chain_begin();
  const int n = st->n_valid;
  const int n_pad = (n + 127) / 128 * 128;
  const int lane = threadIdx.x & 31;
  const int warps_per_block = blockDim.x >> 5;
  const int vec_per_row = d / 8;
  for (int i = blockIdx.x * warps_per_block + (threadIdx.x >> 5); i < n_pad; i += gridDim.x * warps_per_block) {
    uint4* dst = reinterpret_cast<uint4*>(Hc + (size_t)i * d);
    if (i < n) {
      const uint4* src = reinterpret_cast<const uint4*>(H + (size_t)row_map[i] * ldH);
#pragma unroll 4
      for (int v = lane; v < vec_per_row; v += 32) dst[v] = __ldg(src + v);
    } else {
      for (int v = lane; v < vec_per_row; v += 32) dst[v] = make_uint4(0, 0, 0, 0);
    }
  }
}

// ------------------------------------------------------------------------------------------
// GRPO advantages (section 4.2 group-based normalisation), warp-shuffle segmented: a warp is cut
// into segments of seg = (smallest power of two >= G, at most 32) lanes, one group of G consecutive
// rewards per segment (a group of more than 32 responses takes a whole warp and strides over it).
// Mean, centred sum of squares (both in double) and the all-equal test are butterfly reductions that
// stay inside the segment.  For power-of-two G a warp reads and writes 128 contiguous bytes.
__global__ void __launch_bounds__(256) grpo_adv_kernel(const float* __restrict__ rewards, int n_groups, int G,
                                                       int ddof, float eps_std, float* __restrict__ adv_seq) {
  chain_begin();
  int seg = 32;
  while (seg > 1 && (seg >> 1) >= G) seg >>= 1;
  const int groups_per_warp = 32 / seg;
  const int lane = threadIdx.x & 31;
  const int sub = lane & (seg - 1);
  const long long warp_global = (long long)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  const long long g = warp_global * groups_per_warp + lane / seg;
  const bool live = g < n_groups;                 // lanes of groups past the end still take part in the shuffles
  const float* r = rewards + (size_t)(live ? g : 0) * G;
  // sums in double: a group whose rewards lie close together has a small sigma, and the rounding of
  // an fp32 mean divided by it would exceed the 1e-6 the advantages are held to
  double sum = 0.0;
  float mx = -CUDART_INF_F, mn = CUDART_INF_F;
  for (int i = sub; i < G && live; i += seg) {
    const float x = r[i];
    sum += (double)x;
    mx = fmaxf(mx, x);
    mn = fminf(mn, x);
  }
  for (int o = seg >> 1; o > 0; o >>= 1) {
    sum += __shfl_xor_sync(0xffffffffu, sum, o);
    mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    mn = fminf(mn, __shfl_xor_sync(0xffffffffu, mn, o));
  }
  const double mu = sum / (double)G;
  double ss = 0.0;
  for (int i = sub; i < G && live; i += seg) {
    const double c = (double)r[i] - mu;
    ss = fma(c, c, ss);
  }
  for (int o = seg >> 1; o > 0; o >>= 1) ss += __shfl_xor_sync(0xffffffffu, ss, o);
  const double sigma = sqrt(ss / (double)(G - ddof));
  const double inv = (mx == mn) ? 0.0 : 1.0 / (sigma + (double)eps_std);
  for (int i = sub; i < G && live; i += seg)
    adv_seq[(size_t)g * G + i] = (mx == mn) ? 0.f : (float)(((double)r[i] - mu) * inv);
}

// The same arithmetic with one THREAD per group, for batches of many groups whose size is a multiple of four
// (G = 4 * G4 <= 32): a thread reads its group as G4 16-byte words (a warp reads 32 * G * 4 contiguous bytes), keeps
// it in registers and needs no shuffles, so the double-precision mean / variance / square root / reciprocal are
// paid once per group instead of once per lane of a segment.  At 2^20 groups of 8 this is what lets the kernel
// run at memory speed; the shuffle kernel above serves small batches (one warp instruction covers 32 / seg groups,
// which keeps the launch short when there are only a few groups) and every other group size.
template <int G4>
__global__ void __launch_bounds__(256) grpo_adv_rows_kernel(const float4* __restrict__ rewards, int n_groups, int ddof,
                                                            float eps_std, float4* __restrict__ adv_seq) {
  chain_begin();
  constexpr int G = 4 * G4;
  const long long g = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (g >= n_groups) return;
  float x[G];
#pragma unroll
  for (int j = 0; j < G4; ++j) {
    const float4 v = rewards[g * G4 + j];
    x[4 * j] = v.x; x[4 * j + 1] = v.y; x[4 * j + 2] = v.z; x[4 * j + 3] = v.w;
  }
  double sum = 0.0;
  float mx = -CUDART_INF_F, mn = CUDART_INF_F;
#pragma unroll
  for (int i = 0; i < G; ++i) {
    sum += (double)x[i];
    mx = fmaxf(mx, x[i]);
    mn = fminf(mn, x[i]);
  }
  const double mu = sum / (double)G;
  double ss = 0.0;
#pragma unroll
  for (int i = 0; i < G; ++i) {
    const double c = (double)x[i] - mu;
    ss = fma(c, c, ss);
  }
  const double sigma = sqrt(ss / (double)(G - ddof));
  const double inv = (mx == mn) ? 0.0 : 1.0 / (sigma + (double)eps_std);
#pragma unroll
  for (int j = 0; j < G4; ++j) {
    float4 o;
    o.x = (mx == mn) ? 0.f : (float)(((double)x[4 * j] - mu) * inv);
    o.y = (mx == mn) ? 0.f : (float)(((double)x[4 * j + 1] - mu) * inv);
    o.z = (mx == mn) ? 0.f : (float)(((double)x[4 * j + 2] - mu) * inv);
    o.w = (mx == mn) ? 0.f : (float)(((double)x[4 * j + 3] - mu) * inv);
    adv_seq[g * G4 + j] = o;
  }
}

// Other critic-free estimators named in section 4.2 (no formula printed there; readings):
//   est 1 RLOO: A_i = r_i - mean of the other responses of the group
//   est 2 OPO : A_i = r_i - sum_j(len_j r_j) / sum_j(len_j)          (length-weighted baseline)
//   est 3     : c_i = r_i - group mean (first stage of REINFORCE++; batch normalisation follows)
// One warp per group, shuffle reductions.
__global__ void __launch_bounds__(256) group_baseline_kernel(const float* __restrict__ rewards,
                                                             const int* __restrict__ lengths, int n_groups, int G,
                                                             int est, float* __restrict__ adv_seq) {
  chain_begin();
  const int lane = threadIdx.x & 31;
  const int g = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  if (g >= n_groups) return;
  const float* r = rewards + (size_t)g * G;
  float sr = 0.f, sl = 0.f, slr = 0.f;
  for (int i = lane; i < G; i += 32) {
    const float x = r[i];
    const float l = (est == 2) ? (float)lengths[(size_t)g * G + i] : 1.f;
    sr += x;
    sl += l;
    slr = fmaf(l, x, slr);
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    sr += __shfl_xor_sync(0xffffffffu, sr, o);
    sl += __shfl_xor_sync(0xffffffffu, sl, o);
    slr += __shfl_xor_sync(0xffffffffu, slr, o);
  }
  for (int i = lane; i < G; i += 32) {
    const float x = r[i];
    float a;
    if (est == 1) a = x - (sr - x) / (float)(G - 1);
    else if (est == 2) a = x - (sl > 0.f ? slr / sl : 0.f);
    else a = x - sr / (float)G;
    adv_seq[(size_t)g * G + i] = a;
  }
}

// Batch statistics of c[n] in double, fixed order (one block): stats[0] = mean, stats[1] = population std.
__global__ void __launch_bounds__(1024) batch_stats_kernel(const float* __restrict__ c, long long n,
                                                           double* __restrict__ stats) {
  chain_begin();
  __shared__ double red[32];
  __shared__ double mean_s;
  double acc = 0.0;
  for (long long i = threadIdx.x; i < n; i += blockDim.x) acc += (double)c[i];
  for (int pass = 0; pass < 2; ++pass) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = acc;
    __syncthreads();
    if (threadIdx.x == 0) {
      double t = 0.0;
      for (int w = 0; w < 32; ++w) t += red[w];
      if (pass == 0) { mean_s = t / (double)n; stats[0] = mean_s; }
      else stats[1] = sqrt(t / (double)n);
    }
    __syncthreads();
    if (pass == 0) {
      const double mu = mean_s;
      acc = 0.0;
      for (long long i = threadIdx.x; i < n; i += blockDim.x) { const double dlt = (double)c[i] - mu; acc += dlt * dlt; }
    }
  }
}

__global__ void __launch_bounds__(256) batch_normalise_kernel(float* __restrict__ c, long long n,
                                                              const double* __restrict__ stats, float eps_std) {
  chain_begin();
  const double mu = stats[0];
  const double inv = 1.0 / (stats[1] + (double)eps_std);
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
    c[i] = (float)(((double)c[i] - mu) * inv);
}

// Broadcast of the per-response advantage to the rows of the response (outcome supervision).
// The row ranges [seq_offsets[s], seq_offsets[s+1]) are ascending and adjacent, so they partition
// [seq_offsets[0], seq_offsets[n_seq]); rows outside that span get 0.  A block owns
// kBroadcastSweeps * 1024 consecutive rows and walks them in sweeps of 1024; a thread owns four
// consecutive rows per sweep (one 16-byte store when the output is aligned).  It finds the response
// of its first row by binary search in its first sweep and from then on by a galloping search that starts
// at the response it ended the previous sweep in, so the cost per row does not depend on how long
// the responses are and almost all offset reads after the first sweep hit lines the block just used.
// Fewer sweeps per block when the rows would not fill the machine with eight.
// FUSED (few groups, at most 32 responses each): the response's advantage is worked out here, from the rewards of its
// group, instead of being read; the block's threads also write adv_seq.  One launch in place of two.
constexpr int kBroadcastSweeps = 8;

// Advantage of response s from the rewards of its group, in double as grpo_adv_rows_kernel.
__device__ __forceinline__ float group_advantage(const float* __restrict__ rewards, int G, int ddof, float eps_std, int s) {
  const float* r = rewards + (size_t)(s / G) * G;
  double sum = 0.0;
  float mx = -CUDART_INF_F, mn = CUDART_INF_F;
  for (int i = 0; i < G; ++i) {
    const float x = __ldg(r + i);
    sum += (double)x;
    mx = fmaxf(mx, x);
    mn = fminf(mn, x);
  }
  if (mx == mn) return 0.f;
  const double mu = sum / (double)G;
  double ss = 0.0;
  for (int i = 0; i < G; ++i) {
    const double c = (double)__ldg(r + i) - mu;
    ss = fma(c, c, ss);
  }
  return (float)(((double)__ldg(rewards + s) - mu) * (1.0 / (sqrt(ss / (double)(G - ddof)) + (double)eps_std)));
}

// Largest s in [s_from, n_seq) with seq_offsets[s] <= t, given seq_offsets[s_from] <= t < seq_offsets[n_seq].
__device__ __forceinline__ int seq_of_row(const int* __restrict__ seq_offsets, int n_seq, int s_from, long long t) {
  int lo = s_from, step = 1;
  while (lo + step < n_seq && seq_offsets[lo + step] <= t) { lo += step; step <<= 1; }
  int hi = min(lo + step, n_seq);        // seq_offsets[lo] <= t < seq_offsets[hi]
  while (hi - lo > 1) {
    const int mid = (lo + hi) >> 1;
    if (seq_offsets[mid] <= t) lo = mid; else hi = mid;
  }
  return lo;
}

template <bool FUSED>
__global__ void __launch_bounds__(256) broadcast_adv_kernel(const float* __restrict__ rewards, int G, int ddof, float eps_std,
                                                            float* adv_seq, const int* __restrict__ seq_offsets, int n_seq,
                                                            long long T, int sweeps, float* __restrict__ adv_tok) {
  chain_begin();
  if (FUSED)
    for (int s = blockIdx.x * blockDim.x + threadIdx.x; s < n_seq; s += gridDim.x * blockDim.x)
      adv_seq[s] = group_advantage(rewards, G, ddof, eps_std, s);
  auto value = [&](int s) { return FUSED ? group_advantage(rewards, G, ddof, eps_std, s) : adv_seq[s]; };
  const int first = seq_offsets[0], last = seq_offsets[n_seq];
  const bool vec_ok = (reinterpret_cast<uintptr_t>(adv_tok) & 15) == 0;
  const long long rows_per_block = (long long)sweeps * blockDim.x * 4;
  for (long long b0 = (long long)blockIdx.x * rows_per_block; b0 < T; b0 += (long long)gridDim.x * rows_per_block) {
    int s = -1, held = -1;                // response this thread was in last, -1: not searched yet; whose value a is
    float a = 0.f;
    for (int sweep = 0; sweep < sweeps; ++sweep) {
      const long long t0 = b0 + ((long long)sweep * blockDim.x + threadIdx.x) * 4;
      if (t0 >= T) break;
      float v[4] = {0.f, 0.f, 0.f, 0.f};
      if (t0 + 3 >= first && t0 < last) {
        const long long t_in = t0 < first ? first : t0;
        if (s < 0) {
          int lo = 0, hi = n_seq;         // seq_offsets[lo] <= t_in < seq_offsets[hi]
          // responses padded to one length: the first guess is right, and ten dependent loads are saved
          const int guess = (int)((float)(t_in - first) / (float)(last - first) * (float)n_seq);
          if (guess < n_seq) {
            const int o0 = seq_offsets[guess], o1 = seq_offsets[guess + 1];
            if (o0 <= t_in && t_in < o1) { lo = guess; hi = guess + 1; }
          }
          while (hi - lo > 1) {
            const int mid = (lo + hi) >> 1;
            if (seq_offsets[mid] <= t_in) lo = mid; else hi = mid;
          }
          s = lo;
        } else {
          s = seq_of_row(seq_offsets, n_seq, s, t_in);
        }
        int end = seq_offsets[s + 1];
        if (held != s) a = value(held = s);
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const long long t = t0 + i;
          if (t < first || t >= last) continue;
          while (t >= end) { ++s; end = seq_offsets[s + 1]; }   // empty ranges are skipped
          if (held != s) a = value(held = s);
          v[i] = a;
        }
      }
      if (vec_ok && t0 + 3 < T) {
        *reinterpret_cast<float4*>(adv_tok + t0) = make_float4(v[0], v[1], v[2], v[3]);
      } else {
        for (int i = 0; i < 4 && t0 + i < T; ++i) adv_tok[t0 + i] = v[i];
      }
    }
  }
}

// ------------------------------------------------------------------------------------------
// Token-level KL reward shaping (section 2.2 "Regularization": the KL-to-reference term applied as
// per-token rewards; the paper prints no formula, reading): every valid token t of a response gets
// the shaped reward r_t = -beta kl_t, its last valid token additionally the response's scalar
// seq_value, and the per-token value is the return-to-go ret_t = r_t + gamma ret_(next valid token).
// kl_t is the signed log-ratio logp - ref (kind 0), exp(delta) - delta - 1 with delta = ref - logp
// (kind 1), or a value handed in (kind 2).  Masked rows get 0 and are not a discount step.
// A block of four warps per response: it walks the response's rows from the end, 512 rows at a time (each warp 128,
// four 32-row chunks aligned to 128 bytes, all loaded before the first is used).  Every warp runs a suffix scan of the
// linear maps x -> v + g x (valid row: g = gamma, v = r_t; masked row: the identity) over its rows with shuffles, the
// warps' totals are chained through shared memory, and the return of the first valid row of the tile is carried to the
// next.  Per-token terms in fp32, sums in double.  (One warp per response walked 512 rows as a chain of four rounds:
// 26 us for 1024 responses; it stays for responses of less than a warp's 128 rows, and for many whose last 512 rows would be
// mostly empty.)  Rows outside every response range, [0, seq_offsets[0]) and [seq_offsets[n_seq], T), get 0.
constexpr int kShapeChunks = 4;
constexpr int kShapeWarps = 4;

// WARPS: warps per response, kShapeWarps or 1 (the block then works on kShapeWarps responses).
template <int WARPS>
__global__ void __launch_bounds__(32 * kShapeWarps) kl_shaped_returns_kernel(
    const float* __restrict__ seq_value, const float* __restrict__ logp, const float* __restrict__ ref_logp,
    const float* __restrict__ kl_tok, const uint8_t* __restrict__ mask, const int* __restrict__ seq_offsets, int n_seq,
    long long T, float beta, float gamma, int kind, float* __restrict__ shaped, float* __restrict__ ret) {
  chain_begin();
  __shared__ double g_s[WARPS], v_s[WARPS];
  __shared__ int live_s[WARPS];
  constexpr int kTeams = kShapeWarps / WARPS;
  const int lane = threadIdx.x & 31, warp = (threadIdx.x >> 5) % WARPS, team = (threadIdx.x >> 5) / WARPS;
  {
    const long long first = seq_offsets[0], last = seq_offsets[n_seq];
    const long long n_out = first + (T > last ? T - last : 0);
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n_out; i += (long long)gridDim.x * blockDim.x) {
      const long long t = i < first ? i : last + (i - first);
      ret[t] = 0.f;
      if (shaped) shaped[t] = 0.f;
    }
  }
  for (int sq = blockIdx.x * kTeams + team; sq < n_seq; sq += gridDim.x * kTeams) {
    const int lo = seq_offsets[sq], hi = seq_offsets[sq + 1];
    if (hi <= lo) continue;
    const double R = (double)seq_value[sq];
    double carry = 0.0;            // return-to-go of the first valid token after the tiles done so far
    bool terminal_done = false;    // the last valid token of the response has been found
    const int c_first = lo >> 5;
    for (int c_hi = (hi - 1) >> 5; c_hi >= c_first; c_hi -= kShapeChunks * WARPS) {
      const int c_warp = c_hi - warp * kShapeChunks;   // warp 0 has the last rows
      double g[kShapeChunks], v[kShapeChunks];
      float r[kShapeChunks];
      bool inside[kShapeChunks], valid[kShapeChunks];
      unsigned live[kShapeChunks], any = 0;
#pragma unroll
      for (int j = 0; j < kShapeChunks; ++j) {
        const int t = (c_warp - j) * 32 + lane;
        inside[j] = (c_warp - j) >= c_first && t >= lo && t < hi;
        valid[j] = inside[j] && (!mask || mask[t] != 0);
        double kl = 0.0;
        if (inside[j]) {
          if (kind == 2) {
            kl = (double)kl_tok[t];
          } else {
            // the difference of two fp32 values is exact in double; the exponential itself is taken in fp32
            // (expm1f keeps small log-ratios accurate to an ulp), the sums below run in double
            const double delta = (double)ref_logp[t] - (double)logp[t];
            const float df = (float)delta;
            kl = kind == 0 ? -delta : (double)expm1f(df) - delta;
          }
        }
        v[j] = valid[j] ? -(double)beta * kl : 0.0;
        live[j] = __ballot_sync(0xffffffffu, valid[j]);
        any |= live[j];
      }
      bool found = terminal_done, found_all = terminal_done || any != 0;
      if constexpr (WARPS > 1) {
        if (lane == 0) live_s[warp] = any != 0;
        __syncthreads();
#pragma unroll
        for (int w = 0; w < WARPS; ++w) {
          if (w < warp) found = found || live_s[w];
          found_all = found_all || live_s[w];
        }
      }
      double gw = 1.0, vw = 0.0;     // map of this warp's rows done so far, from the last row on
#pragma unroll
      for (int j = 0; j < kShapeChunks; ++j) {
        if (!found && live[j]) {
          if (lane == 31 - __clz(live[j])) v[j] += R;
          found = true;
        }
        r[j] = (float)v[j];
        g[j] = valid[j] ? (double)gamma : 1.0;
        if (gamma == 1.f) {
          // no discount: a plain suffix sum
#pragma unroll
          for (int o = 1; o < 32; o <<= 1) {
            const double v2 = __shfl_down_sync(0xffffffffu, v[j], o);
            if (lane + o < 32) v[j] += v2;
          }
          v[j] += vw;
        } else {
#pragma unroll
          for (int o = 1; o < 32; o <<= 1) {
            const double g2 = __shfl_down_sync(0xffffffffu, g[j], o);
            const double v2 = __shfl_down_sync(0xffffffffu, v[j], o);
            if (lane + o < 32) { v[j] = fma(g[j], v2, v[j]); g[j] *= g2; }
          }
          v[j] = fma(g[j], vw, v[j]);
          g[j] *= gw;
          gw = __shfl_sync(0xffffffffu, g[j], 0);
        }
        vw = __shfl_sync(0xffffffffu, v[j], 0);
      }
      double in = carry;             // return of the first valid row behind this warp's rows
      if constexpr (WARPS > 1) {
        if (lane == 0) { g_s[warp] = gw; v_s[warp] = vw; }
        __syncthreads();
#pragma unroll
        for (int w = 0; w < WARPS; ++w) {
          if (w == warp) in = carry;
          carry = fma(g_s[w], carry, v_s[w]);
        }
      } else {
        carry = fma(gw, carry, vw);
      }
      terminal_done = found_all;
#pragma unroll
      for (int j = 0; j < kShapeChunks; ++j) {
        if (!inside[j]) continue;
        const int t = (c_warp - j) * 32 + lane;
        ret[t] = valid[j] ? (float)fma(g[j], in, v[j]) : 0.f;
        if (shaped) shaped[t] = valid[j] ? r[j] : 0.f;
      }
    }
    if (WARPS > 1) __syncthreads();   // before the next response's tiles reuse the shared words
  }
}

// ------------------------------------------------------------------------------------------
// Merge of the per-range statistics and the per-token loss arithmetic (Eq. 6 with the clipped
// surrogate of section 3.1 and the k3 KL-to-reference term).
constexpr int kLossSums = 8;  // loss, pg, kl, ent, clip, ratio, ratio_max, unused
constexpr int kLossThreads = 256;   // eight warps: one per sum in the last stage

// Where the blocks of a loss kernel leave their sums; the block that draws the last ticket adds them up in a fixed
// order (so the result does not depend on which block that is), writes loss and metrics and returns the ticket counter to 0.
struct LossFinish {
  double* block_sums;     // [total][kLossSums]
  unsigned* ticket;
  int base, total;        // first entry of this launch, entries of all launches that share the sum
  float* loss;
  float* metrics;         // [8] or NULL
};

struct LossParams {
  // inputs
  const float4* partials;
  int part_stride;
  const int* row_map;
  const float* old_logp;   // [T] original rows; NULL in log-prob-only mode
  const float* ref_logp;   // [T] or NULL
  const float* adv;        // [T]
  const float* token_weight;  // [T] or NULL
  const long long* token_count;   // device scalar or NULL: divisor of the token mean (data-parallel global count)
  float eps_low, eps_high, beta, ent_coef;
  int with_loss;
  int zero_coef;           // the coefficients are written later, and not for every row
  // full-distribution KL to the reference policy (two-product forward): second partial per
  // (range, row) = {D, Mr, Sr, 0}; outputs lse_ref, KL_t and the coefficient cb_t = w_t beta
  const float4* partials2;
  int kl_full;
  float* lse_ref_c;
  float* kl_c;
  float* cb_c;
  // compact outputs
  float* lse_c;
  float* ent_c;
  float* logp_c;   // compact log-probabilities, or NULL
  float* cp_c;
  float* ce_c;
  // scattered outputs (original rows), any may be NULL
  float* logp_out;
  float* ent_out;
  float* lse_out;
  float* kl_out;
  LossFinish fin;
  // vocabulary-parallel head: stats_out != NULL -> only merge the ranges of this call's slice and
  // write (M, S, A, z_y) per original row; ext_lse != NULL -> the statistics of the whole
  // vocabulary come from the caller ([T], original rows) instead of the partials
  float4* stats_out;
  const float* ext_logp;
  const float* ext_ent;
  const float* ext_lse;
  // one row slab of the one-sweep path (slab_cap > 0): only its rows are merged
  int slab_cap, slab_one, slab_index;
  uint4* clear;            // ticket and counters of the gradient jobs that follow
  int n_clear;
};
// Fixed-order sum of column k of the block partials by one warp: lane l adds blocks l, l + 32, ... in order, then a
// butterfly over the lanes; the order depends on n_blocks alone, so the result is reproducible.
__device__ __forceinline__ double reduce_block_sums(const double* __restrict__ block_sums, int n_blocks, int k) {
  const int lane = threadIdx.x & 31;
  double v = 0.0;
  for (int b = lane; b < n_blocks; b += 32) {
    const double u = __ldcg(&block_sums[(size_t)b * kLossSums + k]);
    v = (k == 6) ? fmax(v, u) : v + u;
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const double u = __shfl_xor_sync(0xffffffffu, v, o);
    v = (k == 6) ? fmax(v, u) : v + u;
  }
  return v;
}


// Last stage of a loss kernel of kLossThreads threads: block sums, then (last block) the sums over blocks.
__device__ __forceinline__ void finish_loss(const double (&acc)[kLossSums], const LossFinish& f, float n_metric) {
  __shared__ double red[kLossThreads / 32][kLossSums];
  __shared__ int last;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
  for (int k = 0; k < kLossSums; ++k) {
    double v = acc[k];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      const double u = __shfl_xor_sync(0xffffffffu, v, o);
      v = (k == 6) ? fmax(v, u) : v + u;
    }
    if (lane == 0) red[warp][k] = v;
  }
  __syncthreads();
  if (threadIdx.x < kLossSums) {
    const int k = threadIdx.x;
    double v = red[0][k];
    for (int w = 1; w < kLossThreads / 32; ++w) v = (k == 6) ? fmax(v, red[w][k]) : v + red[w][k];
    f.block_sums[(size_t)(f.base + blockIdx.x) * kLossSums + k] = v;
    __threadfence();
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    last = atomicAdd(f.ticket, 1u) == (unsigned)(f.total - 1);
    if (last) *f.ticket = 0;
    __threadfence();
  }
  __syncthreads();
  if (!last) return;
  const double v = reduce_block_sums(f.block_sums, f.total, warp);
  if (lane != 0) return;
  if (warp == 0) f.loss[0] = (float)v;
  if (f.metrics) {
    if (warp >= 1 && warp <= 6) f.metrics[warp - 1] = (float)v;
    if (warp == 7) { f.metrics[6] = n_metric; f.metrics[7] = 0.f; }
  }
}

// A team of kW warps takes 32 rows at a time, lane = row, and shares their column ranges; its first warp goes on with the sums.
// What the loss needs besides is loaded before the merge, one round trip instead of three.  kW = 8 (a block) where rows are
// few: with one thread per row a call of a few hundred rows and 75 to 148 ranges was a chain of that many loads, 17 us.
// kW = 1 where there are rows enough to fill the machine, and where there is nothing to merge (merge_by_thread).
// CLEAR: the counters of gradient jobs that follow are cleared in passing.
template <int kW, bool CLEAR>
__global__ void __launch_bounds__(kLossThreads) combine_loss_kernel(const LossParams p, DevStatus* st) {
  chain_begin();
  constexpr int kTeams = kLossThreads / 32 / kW;
  __shared__ float part_s[2][7][kW][kW > 1 ? 32 : 1];
  if (CLEAR)
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < p.n_clear; i += gridDim.x * blockDim.x) p.clear[i] = make_uint4(0, 0, 0, 0);
  const int n = st->n_valid;
  const int n_ranges = p.ext_lse ? 0 : st->n_ranges;
  const int lane = threadIdx.x & 31, warp = (threadIdx.x >> 5) % kW, team = (threadIdx.x >> 5) / kW;
  double acc[kLossSums];
#pragma unroll
  for (int k = 0; k < kLossSums; ++k) acc[k] = 0.0;
  const long long n_mean = p.token_count ? *p.token_count : (long long)n;
  const float w_mean = n_mean > 0 ? (float)(1.0 / (double)n_mean) : 0.f;
  int i_begin = 0, i_end = n;
  if (p.slab_cap > 0) {
    slab_extent(n, p.slab_cap, p.slab_one, p.slab_index, i_begin, i_end);
    i_end += i_begin;
  }
  int turn = 0;
  for (int i0 = i_begin + (blockIdx.x * kTeams + team) * 32; i0 < i_end; i0 += gridDim.x * kTeams * 32, turn ^= 1) {
    const int i = i0 + lane;
    const bool in = i < i_end;
    float lse, logp, ent, kl = 0.f;
    float M = -CUDART_INF_F, S = 0.f, A = 0.f, zy = 0.f, Mr = -CUDART_INF_F, D = 0.f, Sr = 0.f;
    int row = 0;
    float A_t = 0.f, old_lp = 0.f, ref_lp = 0.f, tw = 0.f;
    if (warp == 0 && in) {
      row = p.row_map[i];
      if (p.with_loss) {
        A_t = p.adv[row];
        old_lp = p.old_logp[row];
        if (p.token_weight) tw = p.token_weight[row];
        if (p.beta != 0.f && !p.kl_full) ref_lp = p.ref_logp[row];
      }
    }
    if (p.ext_lse) {
      if (warp != 0 || !in) continue;
      lse = p.ext_lse[row];
      logp = p.ext_logp[row];
      ent = p.ext_ent[row];
    } else {
      const float4* q1 = p.partials + (in ? i : i_begin);
      const float4* q2 = p.partials2 + (in ? i : i_begin);
#pragma unroll 4
      for (int r = warp; r < n_ranges; r += kW) {
        const float4 q = q1[(size_t)r * p.part_stride];
        const float m = fmaxf(M, q.x), a = exp2f((M - m) * kLog2e), b = exp2f((q.x - m) * kLog2e);
        S = fmaf(S, a, q.y * b);
        A = fmaf(A, a, q.z * b);
        zy += q.w;
        if (p.kl_full) {
          const float4 k = q2[(size_t)r * p.part_stride];
          const float mr = fmaxf(Mr, k.y);
          D = fmaf(D, a, k.x * b);
          Sr = fmaf(Sr, exp2f((Mr - mr) * kLog2e), k.z * exp2f((k.y - mr) * kLog2e));
          Mr = mr;
        }
        M = m;
      }
      if constexpr (kW > 1) {
        auto ps = part_s[turn];   // the other buffer may still be read by warp 0
        ps[0][warp][lane] = M;
        ps[1][warp][lane] = S;
        ps[2][warp][lane] = A;
        ps[3][warp][lane] = zy;
        if (p.kl_full) {
          ps[4][warp][lane] = D;
          ps[5][warp][lane] = Mr;
          ps[6][warp][lane] = Sr;
        }
        __syncthreads();
        if (warp != 0) continue;
        float Mt = M, Mrt = Mr;
#pragma unroll
        for (int w = 1; w < kW; ++w) {
          Mt = fmaxf(Mt, ps[0][w][lane]);
          if (p.kl_full) Mrt = fmaxf(Mrt, ps[5][w][lane]);
        }
        S = A = zy = D = Sr = 0.f;
#pragma unroll
        for (int w = 0; w < kW; ++w) {
          const float m = ps[0][w][lane], b = m == -CUDART_INF_F ? 0.f : exp2f((m - Mt) * kLog2e);   // -inf: no range
          S = fmaf(ps[1][w][lane], b, S);
          A = fmaf(ps[2][w][lane], b, A);
          zy += ps[3][w][lane];
          if (p.kl_full) {
            const float mr = ps[5][w][lane];
            D = fmaf(ps[4][w][lane], b, D);
            Sr = fmaf(ps[6][w][lane], mr == -CUDART_INF_F ? 0.f : exp2f((mr - Mrt) * kLog2e), Sr);
          }
        }
        M = Mt;
        Mr = Mrt;
      }
      if (!in) continue;
      if (p.stats_out) {
        p.stats_out[row] = make_float4(M, S, A, zy);
        continue;
      }
      lse = M + logf(S);
      logp = zy - lse;
      ent = lse - A / S;
    }
    if (p.kl_full) {
      const float lse_ref = Mr + logf(Sr);
      kl = (A - D) / S - lse + lse_ref;      // sum_j p_j (z_j - zr_j) - lse + lse_ref
      p.lse_ref_c[i] = lse_ref;
      p.kl_c[i] = kl;
    }
    if (p.kl_out) p.kl_out[row] = kl;
    p.lse_c[i] = lse;
    p.ent_c[i] = ent;
    if (p.logp_c) p.logp_c[i] = logp;
    if (p.logp_out) p.logp_out[row] = logp;
    if (p.ent_out) p.ent_out[row] = ent;
    if (p.lse_out) p.lse_out[row] = lse;
    if (p.zero_coef) p.cp_c[i] = p.ce_c[i] = 0.f;
    if (p.with_loss) {
      const float w = p.token_weight ? tw : w_mean;
      const float rho = expf(logp - old_lp);
      const float clipped = fminf(fmaxf(rho, 1.f - p.eps_low), 1.f + p.eps_high);
      const float su = rho * A_t, sc = clipped * A_t;
      const bool active = su <= sc;          // unclipped branch is the minimum (ties: unclipped)
      const float s = active ? su : sc;
      float k3 = 0.f, dk3 = 0.f;
      if (p.kl_full) {
        k3 = kl;                              // its gradient is applied per vocabulary entry (cb)
        p.cb_c[i] = w * p.beta;
      } else if (p.beta != 0.f) {
        const float delta = ref_lp - logp;
        const float ed = expf(delta);
        k3 = ed - delta - 1.f;
        dk3 = 1.f - ed;
      }
      const float dlogp = -(active ? A_t * rho : 0.f) + p.beta * dk3;
      p.cp_c[i] = -w * dlogp;
      p.ce_c[i] = w * p.ent_coef;
      acc[0] += (double)w * (double)(-s + p.beta * k3 - p.ent_coef * ent);
      acc[1] += (double)w * (double)(-s);
      acc[2] += (double)w * (double)k3;
      acc[3] += (double)w * (double)ent;
      acc[4] += active ? 0.0 : (double)w;
      acc[5] += (double)w * (double)rho;
      acc[6] = fmax(acc[6], (double)rho);
    }
  }
  if (p.with_loss) finish_loss(acc, p.fin, (float)n);
}

// ------------------------------------------------------------------------------------------
// The per-token loss arithmetic on its own (Eq. 6 with the clipped surrogate of section 3.1 and the k3
// estimate of the KL term), for a caller that already holds the log-probability and entropy of every
// token: works on the original rows, four consecutive rows per thread (16-byte loads and stores when
// every array is 16-byte aligned), masked rows give zero derivatives.  Same arithmetic, in the same
// order, as combine_loss_kernel applies to the statistics it has merged.
constexpr int kCountBlocks = 256;   // most blocks of count_valid_kernel: one count per thread of its reader
__global__ void __launch_bounds__(256) count_valid_kernel(const uint8_t* __restrict__ mask, long long T,
                                                          unsigned* __restrict__ counts) {
  chain_begin();
  unsigned int n = 0;
  const bool vec = (reinterpret_cast<uintptr_t>(mask) & 15) == 0;
  const long long n16 = vec ? T / 16 : 0;
#pragma unroll 4
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n16; i += (long long)gridDim.x * blockDim.x) {
    const uint4 m = reinterpret_cast<const uint4*>(mask)[i];
    n += __popc(__vsetne4(m.x, 0)) + __popc(__vsetne4(m.y, 0)) + __popc(__vsetne4(m.z, 0)) + __popc(__vsetne4(m.w, 0));
  }
  for (long long t = n16 * 16 + (long long)blockIdx.x * blockDim.x + threadIdx.x; t < T;
       t += (long long)gridDim.x * blockDim.x)
    n += mask[t] != 0;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) n += __shfl_xor_sync(0xffffffffu, n, o);
  __shared__ unsigned int red[8];
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = n;
  __syncthreads();
  if (threadIdx.x == 0) {
    unsigned tot = 0;
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) tot += red[w];
    counts[blockIdx.x] = tot;
  }
}

struct TokenLossParams {
  const float* logp;
  const float* entropy;       // or NULL: taken as 0
  const float* old_logp;
  const float* ref_logp;      // or NULL (beta == 0)
  const float* adv;
  const uint8_t* mask;        // or NULL: every row valid
  const float* token_weight;  // or NULL: token mean
  const unsigned* counts;            // valid rows per block of count_valid_kernel, or NULL: every row is valid
  int n_counts;
  const unsigned long long* token_count;   // divisor of the token mean instead of the number of valid rows, or NULL
  long long T;
  float eps_low, eps_high, beta, ent_coef;
  float* dlogp;               // or NULL
  float* dentropy;            // or NULL
  LossFinish fin;
};

template <bool VEC>
__global__ void __launch_bounds__(kLossThreads, 4) token_loss_kernel(const TokenLossParams p) {
  chain_begin();
  double acc[kLossSums];
#pragma unroll
  for (int k = 0; k < kLossSums; ++k) acc[k] = 0.0;
  __shared__ unsigned long long valid_s;
  if (threadIdx.x == 0) valid_s = p.counts ? 0 : (unsigned long long)p.T;
  __syncthreads();
  if (p.counts) {
    unsigned long long v = (int)threadIdx.x < p.n_counts ? p.counts[threadIdx.x] : 0;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    if ((threadIdx.x & 31) == 0) atomicAdd(&valid_s, v);
    __syncthreads();
  }
  const unsigned long long n_valid = valid_s;
  const unsigned long long n_mean = p.token_count ? *p.token_count : n_valid;
  const float w_mean = n_mean > 0 ? (float)(1.0 / (double)n_mean) : 0.f;
  const long long n4 = (p.T + 3) / 4;
  for (long long q = (long long)blockIdx.x * blockDim.x + threadIdx.x; q < n4; q += (long long)gridDim.x * blockDim.x) {
    const long long t0 = q * 4;
    const int nrow = (int)(p.T - t0 < 4 ? p.T - t0 : 4);
    float lp[4], en[4], ol[4], rf[4], av[4], tw[4];
    unsigned int mk[4];
    if (VEC && nrow == 4) {
      const float4 a = *reinterpret_cast<const float4*>(p.logp + t0);
      const float4 b = *reinterpret_cast<const float4*>(p.old_logp + t0);
      const float4 c = *reinterpret_cast<const float4*>(p.adv + t0);
      lp[0] = a.x; lp[1] = a.y; lp[2] = a.z; lp[3] = a.w;
      ol[0] = b.x; ol[1] = b.y; ol[2] = b.z; ol[3] = b.w;
      av[0] = c.x; av[1] = c.y; av[2] = c.z; av[3] = c.w;
      const float4 z = make_float4(0.f, 0.f, 0.f, 0.f);
      const float4 e = p.entropy ? *reinterpret_cast<const float4*>(p.entropy + t0) : z;
      const float4 r = p.ref_logp ? *reinterpret_cast<const float4*>(p.ref_logp + t0) : z;
      const float4 w = p.token_weight ? *reinterpret_cast<const float4*>(p.token_weight + t0) : z;
      en[0] = e.x; en[1] = e.y; en[2] = e.z; en[3] = e.w;
      rf[0] = r.x; rf[1] = r.y; rf[2] = r.z; rf[3] = r.w;
      tw[0] = w.x; tw[1] = w.y; tw[2] = w.z; tw[3] = w.w;
      const unsigned int m4 = p.mask ? *reinterpret_cast<const unsigned int*>(p.mask + t0) : 0x01010101u;
#pragma unroll
      for (int i = 0; i < 4; ++i) mk[i] = (m4 >> (8 * i)) & 0xffu;
    } else {
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const bool in = i < nrow;
        lp[i] = in ? p.logp[t0 + i] : 0.f;
        ol[i] = in ? p.old_logp[t0 + i] : 0.f;
        av[i] = in ? p.adv[t0 + i] : 0.f;
        en[i] = (in && p.entropy) ? p.entropy[t0 + i] : 0.f;
        rf[i] = (in && p.ref_logp) ? p.ref_logp[t0 + i] : 0.f;
        tw[i] = (in && p.token_weight) ? p.token_weight[t0 + i] : 0.f;
        mk[i] = in ? (p.mask ? p.mask[t0 + i] : 1u) : 0u;
      }
    }
    float dl[4], de[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      dl[i] = 0.f;
      de[i] = 0.f;
      if (!mk[i]) continue;
      const float w = p.token_weight ? tw[i] : w_mean;
      const float rho = expf(lp[i] - ol[i]);
      const float clipped = fminf(fmaxf(rho, 1.f - p.eps_low), 1.f + p.eps_high);
      const float su = rho * av[i], sc = clipped * av[i];
      const bool active = su <= sc;          // unclipped branch is the minimum (ties: unclipped)
      const float s = active ? su : sc;
      float k3 = 0.f, dk3 = 0.f;
      if (p.beta != 0.f) {
        const float delta = rf[i] - lp[i];
        const float ed = expf(delta);
        k3 = ed - delta - 1.f;
        dk3 = 1.f - ed;
      }
      const float dlogp = -(active ? av[i] * rho : 0.f) + p.beta * dk3;
      dl[i] = w * dlogp;
      de[i] = -(w * p.ent_coef);
      acc[0] += (double)w * (double)(-s + p.beta * k3 - p.ent_coef * en[i]);
      acc[1] += (double)w * (double)(-s);
      acc[2] += (double)w * (double)k3;
      acc[3] += (double)w * (double)en[i];
      acc[4] += active ? 0.0 : (double)w;
      acc[5] += (double)w * (double)rho;
      acc[6] = fmax(acc[6], (double)rho);
    }
    if (VEC && nrow == 4) {
      if (p.dlogp) *reinterpret_cast<float4*>(p.dlogp + t0) = make_float4(dl[0], dl[1], dl[2], dl[3]);
      if (p.dentropy) *reinterpret_cast<float4*>(p.dentropy + t0) = make_float4(de[0], de[1], de[2], de[3]);
    } else {
      for (int i = 0; i < nrow; ++i) {
        if (p.dlogp) p.dlogp[t0 + i] = dl[i];
        if (p.dentropy) p.dentropy[t0 + i] = de[i];
      }
    }
  }
  finish_loss(acc, p.fin, (float)n_valid);
}

// ------------------------------------------------------------------------------------------
// Sequence-aware loss path: aggregation weights that depend on each response's valid length
// (the length normalisation by token weights of section 2.2) and the sequence-level importance
// ratio (the GSPO variant named in section 4.2; reading: rho_i = exp of the mean
// token log-ratio over the valid tokens of response i, used by every token of the response).
// One team of threads per response - a block, or a warp where responses are short; its valid tokens are the compact rows
// [lo, hi) found by binary search in the ascending row map.  (One warp per response always: 8 responses of 345 rows took
// 50 us in one block.)
struct SeqParams {
  const int* seq_offsets;   // [n_seq + 1] row range of each response
  int n_seq;
  int agg_mode;             // 0 token mean, 1 mean of per-response token means, 2 token sum / (B * L_max)
  int sequence_level;       // 1: sequence-level ratio
  const int* row_map;
  const float* logp_c;
  const float* ent_c;
  const float* old_logp;
  const float* ref_logp;
  const float* adv;
  const float* token_weight;  // overrides agg_mode when not NULL
  float eps_low, eps_high, beta, ent_coef;
  int* l_max;               // device scalar: longest row range
  float* cp_c;
  float* ce_c;
  LossFinish fin;
};

__global__ void __launch_bounds__(1024) seq_lmax_kernel(const int* __restrict__ seq_offsets, int n_seq, int* l_max) {
  chain_begin();
  __shared__ int red[32];
  int m = 0;
  for (int i = threadIdx.x; i < n_seq; i += blockDim.x) m = max(m, seq_offsets[i + 1] - seq_offsets[i]);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) m = max(m, __shfl_xor_sync(0xffffffffu, m, o));
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = m;
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int w = 1; w < 32; ++w) m = max(m, red[w]);
    *l_max = m;
  }
}

__device__ __forceinline__ int lower_bound_rows(const int* __restrict__ row_map, int n, int key) {
  int lo = 0, hi = n;
  while (lo < hi) {
    const int mid = (lo + hi) >> 1;
    if (row_map[mid] < key) lo = mid + 1; else hi = mid;
  }
  return lo;
}

// Sum over the TEAM threads of a team, the same value for all of them; every thread of the block calls it.
template <int TEAM>
__device__ __forceinline__ float team_sum(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  if (TEAM > 32) {
    __shared__ float part[TEAM / 32];
    __syncthreads();   // the previous sum has been read
    if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = v;
    __syncthreads();
    v = 0.f;
#pragma unroll
    for (int w = 0; w < TEAM / 32; ++w) v += part[w];
  }
  return v;
}

template <int TEAM>
__global__ void __launch_bounds__(kLossThreads) seq_loss_kernel(const SeqParams p, DevStatus* st) {
  chain_begin();
  const int n = st->n_valid;
  const int lane = threadIdx.x % TEAM, team = threadIdx.x / TEAM;
  constexpr int teams = kLossThreads / TEAM;
  double acc[kLossSums];
#pragma unroll
  for (int k = 0; k < kLossSums; ++k) acc[k] = 0.0;
  // token mean (agg_mode 0): over the valid rows that lie inside a response range, the ones that take part
  const int n_part = p.agg_mode == 0 ? lower_bound_rows(p.row_map, n, p.seq_offsets[p.n_seq]) -
                                           lower_bound_rows(p.row_map, n, p.seq_offsets[0])
                                     : 0;
  for (int sq = blockIdx.x * teams + team; sq < p.n_seq; sq += gridDim.x * teams) {
    const int lo = lower_bound_rows(p.row_map, n, p.seq_offsets[sq]);
    const int hi = lower_bound_rows(p.row_map, n, p.seq_offsets[sq + 1]);
    const int len = hi - lo;
    if (len <= 0) continue;
    float w_seq = 0.f;
    if (p.agg_mode == 0) w_seq = 1.f / (float)n_part;
    else if (p.agg_mode == 1) w_seq = 1.f / ((float)p.n_seq * (float)len);
    else w_seq = 1.f / ((float)p.n_seq * (float)max(*p.l_max, 1));
    float rho_seq = 1.f, seq_sum = 0.f;
    if (p.sequence_level) {
      float lr = 0.f;
      for (int k = lo + lane; k < hi; k += TEAM) lr += p.logp_c[k] - p.old_logp[p.row_map[k]];
      lr = team_sum<TEAM>(lr);
      rho_seq = expf(lr / (float)len);
      const float clipped = fminf(fmaxf(rho_seq, 1.f - p.eps_low), 1.f + p.eps_high);
      for (int k = lo + lane; k < hi; k += TEAM) {
        const int row = p.row_map[k];
        const float w = p.token_weight ? p.token_weight[row] : w_seq;
        const float A_t = p.adv[row];
        const bool active = rho_seq * A_t <= clipped * A_t;
        seq_sum += active ? w * A_t : 0.f;
      }
      seq_sum = team_sum<TEAM>(seq_sum);
    }
    for (int k = lo + lane; k < hi; k += TEAM) {
      const int row = p.row_map[k];
      const float w = p.token_weight ? p.token_weight[row] : w_seq;
      const float A_t = p.adv[row];
      const float logp = p.logp_c[k];
      const float ent = p.ent_c[k];
      const float rho = p.sequence_level ? rho_seq : expf(logp - p.old_logp[row]);
      const float clipped = fminf(fmaxf(rho, 1.f - p.eps_low), 1.f + p.eps_high);
      const float su = rho * A_t, sc = clipped * A_t;
      const bool active = su <= sc;
      const float s = active ? su : sc;
      float k3 = 0.f, dk3 = 0.f;
      if (p.beta != 0.f) {
        const float delta = p.ref_logp[row] - logp;
        const float ed = expf(delta);
        k3 = ed - delta - 1.f;
        dk3 = 1.f - ed;
      }
      // weighted d loss / d logp_t
      const float wdlogp = (p.sequence_level ? -(rho_seq / (float)len) * seq_sum : -(active ? w * A_t * rho : 0.f)) +
                           w * p.beta * dk3;
      p.cp_c[k] = -wdlogp;
      p.ce_c[k] = w * p.ent_coef;
      acc[0] += (double)w * (double)(-s + p.beta * k3 - p.ent_coef * ent);
      acc[1] += (double)w * (double)(-s);
      acc[2] += (double)w * (double)k3;
      acc[3] += (double)w * (double)ent;
      acc[4] += active ? 0.0 : (double)w;
      acc[5] += (double)w * (double)rho;
      acc[6] = fmax(acc[6], (double)rho);
    }
  }
  finish_loss(acc, p.fin, (float)n);
}

// ------------------------------------------------------------------------------------------
// Vocabulary-parallel head: merge of the per-row statistics (M, S, A, z_y) of the n_shards slices
// of a partition of the vocabulary (stats[s][t], original rows) into the log-probability of the
// sampled token, the entropy and the log-sum-exp over the whole vocabulary.  Rows with mask 0
// get 0.  One thread per row; the slices are visited in order, so the result is reproducible.
__global__ void __launch_bounds__(256) merge_shard_stats_kernel(const float4* __restrict__ stats, int n_shards,
                                                                long long T, const uint8_t* __restrict__ mask,
                                                                float* __restrict__ logp, float* __restrict__ ent,
                                                                float* __restrict__ lse) {
  chain_begin();
  for (long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x; t < T; t += (long long)gridDim.x * blockDim.x) {
    float o_logp = 0.f, o_ent = 0.f, o_lse = 0.f;
    if (!mask || mask[t]) {
      float M = -CUDART_INF_F;
      for (int s = 0; s < n_shards; ++s) M = fmaxf(M, __ldg(&stats[(size_t)s * T + t]).x);
      float S = 0.f, A = 0.f, zy = 0.f;
      for (int s = 0; s < n_shards; ++s) {
        const float4 q = __ldg(&stats[(size_t)s * T + t]);
        const float sc = exp2f((q.x - M) * kLog2e);
        S = fmaf(q.y, sc, S);
        A = fmaf(q.z, sc, A);
        zy += q.w;
      }
      o_lse = M + logf(S);
      o_logp = zy - o_lse;
      o_ent = o_lse - A / S;
    }
    logp[t] = o_logp;
    if (ent) ent[t] = o_ent;
    if (lse) lse[t] = o_lse;
  }
}

// ------------------------------------------------------------------------------------------
// dH of one row slab: fp32 accumulator rows -> rows of the caller's dH at their original positions, fp32 or bf16.  Done by four
// extra warps of the dW launch that follows (EpiAccScatter), or by a launch of its own where dW comes first.
// The dH pass may have cut K into slices that accumulate in separate buffers, split_stride elements apart, or cut the
// tiles of its last wave into parts that lie in slots: summed here in a fixed order.
struct DhSource {
  const float* acc;        // [slab rows][d]
  int d;
  GemmShape shape;         // the dH pass: together with its grid it fixes how tiles were cut
  int cg, workers;
  long long split_stride;
  const float* slots;      // [slots][tile_rows][tile_cols], tiles cut by stream_k == 2
  int tile_rows, tile_cols;
  const int* row_map;
  void* dH;
  int f32;                 // dH is fp32
};

__device__ __forceinline__ void add_piece(float4 (&x)[4], const float* q, int cols, int lane) {
#pragma unroll
  for (int k = 0; k < 2; ++k) {
    const int v = lane + 32 * k;
    if (v * 8 < cols) {
      const float4 a = __ldcs(reinterpret_cast<const float4*>(q) + 2 * v);
      const float4 b = __ldcs(reinterpret_cast<const float4*>(q) + 2 * v + 1);
      x[2 * k].x += a.x; x[2 * k].y += a.y; x[2 * k].z += a.z; x[2 * k].w += a.w;
      x[2 * k + 1].x += b.x; x[2 * k + 1].y += b.y; x[2 * k + 1].z += b.z; x[2 * k + 1].w += b.w;
    }
  }
}

// One warp per row and column tile (at most 512 columns: two groups of eight per lane); this is warp `warp` of n_warps.
__device__ __forceinline__ void scatter_rows(const DhSource& s, int n_valid, unsigned warp, unsigned n_warps) {
  int slab_base, rows;
  slab_extent(n_valid, s.shape.slab_cap, s.shape.slab_one, s.shape.slab_index, slab_base, rows);
  const GemmExtents ex = gemm_extents(s.shape, n_valid, s.cg, s.workers);
  const int slices = s.shape.stream_k == 1 ? 2 : ex.k_split;   // stream-K launches always keep two buffers
  const int lane = threadIdx.x & 31;
  const unsigned col_tiles = (s.d + s.tile_cols - 1) / s.tile_cols;
  const unsigned units = (unsigned)rows * col_tiles;
  for (unsigned u = warp; u < units; u += n_warps) {
    const int i = (int)(u / col_tiles), nt = (int)(u - i * col_tiles);
    const int cols = min(s.tile_cols, s.d - nt * s.tile_cols);
    const size_t col0 = (size_t)nt * s.tile_cols;
    float4 x[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) x[k] = make_float4(0.f, 0.f, 0.f, 0.f);
    const int r = i / s.tile_rows * ex.n_ranges + nt - (ex.n_units - ex.cut);
    if (ex.stream_k == 2 && r >= 0) {
      const int S = ex.cut_parts;
      const size_t slot = (size_t)s.tile_rows * s.tile_cols;
      const float* base = s.slots + (size_t)(i % s.tile_rows) * s.tile_cols;
      CutSlots at = {0, 1, 0};   // lane s: of part s
      if (ex.cut_len > 0 && lane < S) at = cut_slots(ex, s.workers, r, lane);
      for (int p = 0; p < S; ++p) {
        add_piece(x, base + slot * (r * S + p), cols, lane);
        if (ex.cut_len > 0) {
          const int a = __shfl_sync(0xffffffffu, at.first, p), b = __shfl_sync(0xffffffffu, at.last, p);
          for (int h = a; h <= b; ++h) add_piece(x, base + slot * h, cols, lane);
        }
      }
    } else {
      const float* q = s.acc + (size_t)i * s.d + col0;
      for (int k = 0; k < slices; ++k, q += s.split_stride) add_piece(x, q, cols, lane);
    }
    const size_t out = (size_t)s.row_map[slab_base + i] * s.d + col0;
#pragma unroll
    for (int k = 0; k < 2; ++k) {
      const int v = lane + 32 * k;
      if (v * 8 >= cols) break;
      const float4 a = x[2 * k], b = x[2 * k + 1];
      if (s.f32) {
        float4* dst = reinterpret_cast<float4*>(static_cast<float*>(s.dH) + out) + 2 * v;
        __stcs(dst, a);
        __stcs(dst + 1, b);
      } else {
        __nv_bfloat162 b0 = __floats2bfloat162_rn(a.x, a.y), b1 = __floats2bfloat162_rn(a.z, a.w);
        __nv_bfloat162 b2 = __floats2bfloat162_rn(b.x, b.y), b3 = __floats2bfloat162_rn(b.z, b.w);
        uint4 o;
        o.x = *reinterpret_cast<uint32_t*>(&b0);
        o.y = *reinterpret_cast<uint32_t*>(&b1);
        o.z = *reinterpret_cast<uint32_t*>(&b2);
        o.w = *reinterpret_cast<uint32_t*>(&b3);
        __stcs(reinterpret_cast<uint4*>(static_cast<__nv_bfloat16*>(s.dH) + out) + v, o);
      }
    }
  }
}

__global__ void __launch_bounds__(256) scatter_dH_kernel(const DhSource s, const DevStatus* st) {
  chain_begin();
  const unsigned per_block = blockDim.x >> 5;
  scatter_rows(s, st->n_valid, blockIdx.x * per_block + (threadIdx.x >> 5), gridDim.x * per_block);
}

// dW of one slab; extra warps write dH of the same slab, which the launch before has left, meanwhile: a launch less.
template <int W>
struct EpiAccScatter : EpiAccW<W> {
  static constexpr int kSideWarps = 4;
  struct Params : AccParams {
    DhSource dh;
  };
  __device__ static __forceinline__ void side(const Params& p, const GemmExtents&, int, int, int warp) {
    scatter_rows(p.dh, *p.n_valid, blockIdx.x * kSideWarps + warp, gridDim.x * kSideWarps);
  }
};

// ------------------------------------------------------------------------------------------
// Exercises the bounded waits, each with a short limit: on an mbarrier that nothing ever arrives on, on a counter in global memory and
// on a word in shared memory that nobody raises.  Each must come back with the abort flag raised; the detail's low bits name those that did not.
__device__ unsigned g_never_counted;
__global__ void __launch_bounds__(32) wait_timeout_probe_kernel(unsigned long long limit_ns, DevStatus* st) {
  __shared__ __align__(8) uint64_t bar;
  __shared__ int abort_flag, word;
  if (threadIdx.x == 0) {
    mbar_init(smem_u32(&bar), 1);
    word = 0;
    fence_mbar_init();
  }
  __syncwarp();
  if (threadIdx.x == 0) {
    volatile int *abort_p = &abort_flag, *word_p = &word;
    int kept = 0, seen;
    auto runs_out = [&](int bit, auto wait) {
      *abort_p = 0;
      if (wait() || *abort_p != 1) kept |= bit;
    };
    runs_out(1, [&] { return mbar_wait_bounded(smem_u32(&bar), 0, abort_p, limit_ns); });
    runs_out(2, [&] { return count_wait_bounded(&g_never_counted, 1, abort_p, limit_ns); });
    runs_out(4, [&] { return word_wait_bounded(word_p, 1, seen, abort_p, limit_ns); });
    latch_status(st, kStatusTimeout, 0x70000000 | kept);
  }
  __syncwarp();
}

}  // namespace rlh
