// Epilogues of the two-product tile mode of the GEMM engine: full-distribution KL(pi_theta || pi_ref) per token
// (section 2.2 "KL-to-reference", section 3.1 Omega) and its gradient with respect to the logits.
#pragma once
#include "epilogues.cuh"

namespace rlh {

// ---------------------------------------------------------------------------------------------
// Forward: the statistics of EpiStats for the policy logits z, plus
//   D  = sum_j exp(z_j - M) zr_j          (so that sum_j p_j (z_j - zr_j) = (A - D) / S)
//   Mr, Sr = running max and sum exp(zr - Mr) of the reference logits (for lse_ref).
// Two float4 per (range, row): {M, S, A, z_y} and {D, Mr, Sr, 0}.
// Eight epilogue warps in all passes of the full KL: their epilogues are the heavy ones (d = d_ref = 256 / 512 / 704 / 2048:
// statistics 1200 / 1474 / 1858 / 4775 us with four, 985 / 1246 / 1607 / 4395 with eight).
struct EpiStatsKL {
  static constexpr bool kParts = false;
  static constexpr int kSideWarps = 0;
  static constexpr bool kFeeds = false, kAhead = false;
  static constexpr int kWarps = 8;
  static constexpr int kStagingBytes = 0;
  struct Params {
    const int* tokens_c;
    float4* partials;
    float4* partials2;
    int part_stride;
    int V;
  };
  struct State {
    float m, s, a, zy, dsum, mr, sr;
    int y;
  };
  __device__ static __forceinline__ void init(State&) {}
  __device__ static __forceinline__ void finish(State&) {}
  __device__ static __forceinline__ void begin_unit(const Params& p, State& st, int m_tile, int, int row_in_tile,
                                                    int m_rows, int, int) {
    st.m = -CUDART_INF_F; st.s = 0.f; st.a = 0.f; st.zy = 0.f; st.dsum = 0.f;
    st.mr = -CUDART_INF_F; st.sr = 0.f;
    const int row = m_tile * BM + row_in_tile;
    st.y = row < m_rows ? p.tokens_c[row] : -1;
  }
  __device__ static __forceinline__ void chunk(const Params& p, State& st, int, int n_tile, int c, int, int,
                                               const float (&v)[32], const float (&vr)[32], const CUtensorMap*,
                                               uint32_t) {
    const int col0 = n_tile * BN + c * 32;
    const int nvalid = p.V - col0;
    if (nvalid <= 0) return;
    float cmax = -CUDART_INF_F, rmax = -CUDART_INF_F;
#pragma unroll
    for (int i = 0; i < 32; ++i) {
      cmax = i < nvalid ? fmaxf(cmax, v[i]) : cmax;
      rmax = i < nvalid ? fmaxf(rmax, vr[i]) : rmax;
    }
    const float newm = fmaxf(st.m, cmax), newr = fmaxf(st.mr, rmax);
    const float scale = ex2_approx((st.m - newm) * kLog2e), scale_r = ex2_approx((st.mr - newr) * kLog2e);
    const float mL = newm * kLog2e, rL = newr * kLog2e;
    float cs = 0.f, ca = 0.f, cd = 0.f, csr = 0.f;
#pragma unroll
    for (int i = 0; i < 32; ++i) {
      const float e = i < nvalid ? ex2_approx(fmaf(v[i], kLog2e, -mL)) : 0.f;
      const float er = i < nvalid ? ex2_approx(fmaf(vr[i], kLog2e, -rL)) : 0.f;
      cs += e;
      ca = fmaf(e, v[i], ca);
      cd = fmaf(e, vr[i], cd);
      csr += er;
    }
    st.s = fmaf(st.s, scale, cs);
    st.a = fmaf(st.a, scale, ca);
    st.dsum = fmaf(st.dsum, scale, cd);
    st.m = newm;
    st.sr = fmaf(st.sr, scale_r, csr);
    st.mr = newr;
    const unsigned rel = (unsigned)(st.y - col0);
    if (rel < 32u && (int)rel < nvalid) {
      float z = 0.f;
#pragma unroll
      for (int i = 0; i < 32; ++i) z = (rel == (unsigned)i) ? v[i] : z;
      st.zy = z;
    }
  }
  static constexpr int kMerge = 7;
  __device__ static __forceinline__ void pack(const State& st, float (&x)[kMerge]) {
    x[0] = st.m; x[1] = st.s; x[2] = st.a; x[3] = st.zy; x[4] = st.dsum; x[5] = st.mr; x[6] = st.sr;
  }
  __device__ static __forceinline__ void merge(State& st, const float (&x)[kMerge]) {
    const float m = fmaxf(st.m, x[0]), mr = fmaxf(st.mr, x[5]);
    // a half that saw no column inside the vocabulary has maxima of -inf and sums of 0
    const float a = st.m == m ? 1.f : ex2_approx((st.m - m) * kLog2e), b = x[0] == m ? 1.f : ex2_approx((x[0] - m) * kLog2e);
    const float ar = st.mr == mr ? 1.f : ex2_approx((st.mr - mr) * kLog2e), br = x[5] == mr ? 1.f : ex2_approx((x[5] - mr) * kLog2e);
    st.s = fmaf(st.s, a, x[1] * b);
    st.a = fmaf(st.a, a, x[2] * b);
    st.zy += x[3];
    st.dsum = fmaf(st.dsum, a, x[4] * b);
    st.sr = fmaf(st.sr, ar, x[6] * br);
    st.m = m;
    st.mr = mr;
  }
  __device__ static __forceinline__ void end_unit(const Params& p, State& st, int m_tile, int nr, int row_in_tile,
                                                  int m_rows) {
    const int row = m_tile * BM + row_in_tile;
    if (row < m_rows) {
      p.partials[(size_t)nr * p.part_stride + row] = make_float4(st.m, st.s, st.a, st.zy);
      p.partials2[(size_t)nr * p.part_stride + row] = make_float4(st.dsum, st.mr, st.sr, 0.f);
    }
  }
};

// ---------------------------------------------------------------------------------------------
// One-sweep form: the reference logits and the policy logits of a slab of whole rows are formed once each, in two
// single-product passes whose epilogues overlap the next tile's MMAs, and both stay in the slab in fp32 until the rows'
// log-sum-exps and loss coefficients are known: the reference logits as they are, the policy logits as two 16-bit planes,
// so that the gradient can take the place of the upper halves.  Forming both logits side by side (two-product tiles) left
// the epilogue exposed and had to be done twice: 4.2 + 4.0 ms at 4096 rows, d = d_ref = 2048, V = 151936.
__device__ __forceinline__ void ld_global_v8(const float* p, float (&v)[32], int i) {
  asm volatile("ld.global.v8.f32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
               : "=f"(v[i]), "=f"(v[i + 1]), "=f"(v[i + 2]), "=f"(v[i + 3]), "=f"(v[i + 4]), "=f"(v[i + 5]), "=f"(v[i + 6]),
                 "=f"(v[i + 7])
               : "l"(p + i)
               : "memory");
}
__device__ __forceinline__ void st_global_v8(float* p, const float* v) {
  asm volatile("st.global.v8.f32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(p), "f"(v[0]), "f"(v[1]), "f"(v[2]), "f"(v[3]),
               "f"(v[4]), "f"(v[5]), "f"(v[6]), "f"(v[7])
               : "memory");
}

// Upper and lower 16-bit halves of 32 consecutive logits of a row, to the two planes (32-byte stores, every sector whole).
__device__ __forceinline__ void st_planes(const float (&v)[32], uint16_t* hi, uint16_t* lo) {
  float h[16], l[16];
#pragma unroll
  for (int i = 0; i < 16; ++i) {
    const uint32_t a = __float_as_uint(v[2 * i]), b = __float_as_uint(v[2 * i + 1]);
    h[i] = __uint_as_float(__byte_perm(a, b, 0x7632));
    l[i] = __uint_as_float(__byte_perm(a, b, 0x5410));
  }
#pragma unroll
  for (int j = 0; j < 16; j += 8) {
    st_global_v8(reinterpret_cast<float*>(hi) + j, h + j);
    st_global_v8(reinterpret_cast<float*>(lo) + j, l + j);
  }
}

// Reference pass: zr to the slab, running max and sum of exp of the reference logits to partials2 = {-, Mr, Sr, -}.
// A thread holds 32 consecutive columns of its row: four 32-byte stores, every sector written whole.
struct EpiRefSweep {
  static constexpr bool kParts = false;
  static constexpr int kSideWarps = 0;
  static constexpr bool kFeeds = false, kAhead = false;
  static constexpr int kWarps = 8;
  static constexpr int kStagingBytes = 0;
  struct Params {
    float4* partials2;
    int part_stride;
    int V;
    float* slab;
    int ld;
  };
  struct State {
    RowStats::State s;
    float* row;
    int grow;
  };
  __device__ static __forceinline__ void init(State&) {}
  __device__ static __forceinline__ void finish(State&) {}
  __device__ static __forceinline__ void begin_unit(const Params& p, State& st, int m_tile, int, int row_in_tile,
                                                    int m_rows, int slab_off, int) {
    const int rl = m_tile * BM + row_in_tile;
    st.grow = rl < m_rows ? slab_off + rl : -1;
    st.row = rl < m_rows ? p.slab + (size_t)rl * p.ld : nullptr;
    st.s.m = -CUDART_INF_F;
    st.s.s = st.s.a = st.s.zy = 0.f;
    st.s.y = -1;
  }
  __device__ static __forceinline__ void chunk(const Params& p, State& st, int, int n_tile, int c, int, int,
                                               const float (&v)[32], const CUtensorMap* map, uint32_t staging) {
    RowStats::Params ps;
    ps.V = p.V;
    RowStats::chunk(ps, st.s, 0, n_tile, c, 0, 0, v, map, staging);
    if (st.row) {
      float* q = st.row + n_tile * BN + c * 32;
#pragma unroll
      for (int j = 0; j < 4; ++j) st_global_v8(q + 8 * j, v + 8 * j);
    }
  }
  static constexpr int kMerge = RowStats::kMerge;
  __device__ static __forceinline__ void pack(const State& st, float (&x)[kMerge]) { RowStats::pack(st.s, x); }
  __device__ static __forceinline__ void merge(State& st, const float (&x)[kMerge]) { RowStats::merge(st.s, x); }
  __device__ static __forceinline__ void end_unit(const Params& p, State& st, int, int nr, int, int) {
    if (st.grow >= 0) p.partials2[(size_t)nr * p.part_stride + st.grow] = make_float4(0.f, st.s.m, st.s.s, 0.f);
  }
};

// Policy pass: statistics of EpiStats, D = sum_j exp(z_j - M) zr_j (to partials2.x), and the planes of z.  The reference
// logits of the next 32 columns are loaded while these are worked on.
struct EpiSweepKL {
  static constexpr bool kParts = false;
  static constexpr int kSideWarps = 0;
  static constexpr bool kFeeds = false, kAhead = false;
  static constexpr int kWarps = 8;
  static constexpr int kStagingBytes = 0;
  struct Params {
    RowStats::Params stats;
    float4* partials2;
    const float* zr;       // reference logits of the slab
    uint16_t* hi;          // planes of the policy logits
    uint16_t* lo;
    int ld;                // whole tiles: columns past V are read and written as well
  };
  struct State {
    RowStats::State s;
    float d;
    long long at;    // start of this thread's row in the slab, -1: past the valid rows
    int grow;
    bool fresh;      // nothing loaded ahead yet
    float next[32];
  };
  __device__ static __forceinline__ void init(State&) {}
  __device__ static __forceinline__ void finish(State&) {}
  __device__ static __forceinline__ void begin_unit(const Params& p, State& st, int m_tile, int, int row_in_tile,
                                                    int m_rows, int slab_off, int) {
    const int rl = m_tile * BM + row_in_tile;
    const bool valid = rl < m_rows;
    st.grow = valid ? slab_off + rl : -1;
    st.at = valid ? (long long)rl * p.ld : -1;
    st.s.m = -CUDART_INF_F;
    st.s.s = st.s.a = st.s.zy = 0.f;
    st.d = 0.f;
    st.s.y = valid ? p.stats.tokens_c[st.grow] : -1;
    st.fresh = true;
  }
  __device__ static __forceinline__ void chunk(const Params& p, State& st, int, int n_tile, int c, int, int,
                                               const float (&v)[32], const CUtensorMap* map, uint32_t staging) {
    if (st.at < 0) return;
    const int col = n_tile * BN + c * 32;
    const float* q = p.zr + st.at + col;
    float zr[32];
    if (st.fresh) {
#pragma unroll
      for (int j = 0; j < 32; j += 8) ld_global_v8(q, zr, j);
      st.fresh = false;
    } else {
#pragma unroll
      for (int j = 0; j < 32; ++j) zr[j] = st.next[j];
    }
    // this warp's next columns: four chunks in a row, then the other half's four are passed over
    const int ahead = (c & 3) == 3 ? 32 + BN / 2 : 32;
    if (col + ahead < p.ld) {
#pragma unroll
      for (int j = 0; j < 32; j += 8) ld_global_v8(q + ahead, st.next, j);
    }
    const int nvalid = p.stats.V - col;
    const float m_old = st.s.m;
    RowStats::chunk(p.stats, st.s, 0, n_tile, c, 0, 0, v, map, staging);
    if (nvalid > 0) {
      // D with the same weights as A (the sum that EpiStats keeps), rescaled as A is
      const float mL = st.s.m * kLog2e;
      float2 cd2 = make_float2(0.f, 0.f);
      const float2 l2 = make_float2(kLog2e, kLog2e), nm2 = make_float2(-mL, -mL);
#pragma unroll
      for (int i = 0; i < 32; i += 2) {
        const float2 t2 = __ffma2_rn(make_float2(v[i], v[i + 1]), l2, nm2);
        const float e0 = i < nvalid ? ex2_approx(t2.x) : 0.f, e1 = i + 1 < nvalid ? ex2_approx(t2.y) : 0.f;
        cd2 = __ffma2_rn(make_float2(e0, e1), make_float2(zr[i], zr[i + 1]), cd2);
      }
      st.d = fmaf(st.d, ex2_approx((m_old - st.s.m) * kLog2e), cd2.x + cd2.y);
    }
    st_planes(v, p.hi + st.at + col, p.lo + st.at + col);
  }
  static constexpr int kMerge = RowStats::kMerge + 1;
  __device__ static __forceinline__ void pack(const State& st, float (&x)[kMerge]) {
    x[0] = st.s.m; x[1] = st.s.s; x[2] = st.s.a; x[3] = st.s.zy; x[4] = st.d;
  }
  __device__ static __forceinline__ void merge(State& st, const float (&x)[kMerge]) {
    const float y[RowStats::kMerge] = {x[0], x[1], x[2], x[3]}, m = fmaxf(st.s.m, x[0]);
    st.d = fmaf(st.d, st.s.m == m ? 1.f : ex2_approx((st.s.m - m) * kLog2e),
                x[4] * (x[0] == m ? 1.f : ex2_approx((x[0] - m) * kLog2e)));
    RowStats::merge(st.s, y);
  }
  __device__ static __forceinline__ void end_unit(const Params& p, State& st, int, int nr, int, int) {
    if (st.grow < 0) return;
    const size_t i = (size_t)nr * p.stats.part_stride + st.grow;
    p.stats.partials[i] = make_float4(st.s.m, st.s.s, st.s.a, st.s.zy);
    p.partials2[i].x = st.d;
  }
};

// ---------------------------------------------------------------------------------------------
// Backward: g_tj = cp_t (p_tj - 1[j = y_t]) + cb_t p_tj (log p_tj - log q_tj - KL_t)
//                  + ce_t p_tj (log p_tj + Ent_t),   cb_t = w_t beta,
// written to the bf16 slab exactly as EpiGrad does (swizzled staging + TMA bulk stores).
struct EpiGradKL {
  static constexpr bool kParts = false;
  static constexpr int kSideWarps = 0;
  static constexpr bool kFeeds = false, kAhead = false;
  static constexpr int kWarps = 8;
  static constexpr int kMerge = 0;
  static constexpr int kStagingBytes = kEpiStaging;
  struct Params {
    const int* tokens_c;
    const float* lse;
    const float* lse_ref;
    const float* ent;
    const float* kl;
    const float* cp;
    const float* cb;
    const float* ce;
    int V;
    int vocab_base;
  };
  struct State {
    float lse, lse_ref, ent, kl, cp, cb, ce;
    int y;
    bool valid;
    uint32_t n_issued;
  };
  __device__ static __forceinline__ void init(State& st) { st.n_issued = 0; }
  __device__ static __forceinline__ void finish(State& st) {
    if ((threadIdx.x & 31) == 0 && st.n_issued) bulk_wait_group_all();
    __syncwarp();
  }
  __device__ static __forceinline__ void begin_unit(const Params& p, State& st, int m_tile, int, int row_in_tile,
                                                    int m_rows, int slab_off, int) {
    const int rl = m_tile * BM + row_in_tile;
    st.valid = rl < m_rows;
    const int gr = slab_off + rl;
    st.lse = st.valid ? p.lse[gr] : 0.f;
    st.lse_ref = st.valid ? p.lse_ref[gr] : 0.f;
    st.ent = st.valid ? p.ent[gr] : 0.f;
    st.kl = st.valid ? p.kl[gr] : 0.f;
    st.cp = st.valid ? p.cp[gr] : 0.f;
    st.cb = st.valid ? p.cb[gr] : 0.f;
    st.ce = st.valid ? p.ce[gr] : 0.f;
    st.y = st.valid ? p.tokens_c[gr] : -1;
  }
  __device__ static __forceinline__ void chunk(const Params& p, State& st, int m_tile, int n_tile, int c,
                                               int row_in_tile, int m_rows, const float (&v)[32],
                                               const float (&vr)[32], const CUtensorMap* tmG, uint32_t staging) {
    if (m_tile * BM >= ((m_rows + BM - 1) / BM) * BM) return;
    const int col_l = n_tile * BN + c * 32;
    const int col_g = p.vocab_base + col_l;
    const int nvalid = p.V - col_g;
    float g[32];
    if (!st.valid || nvalid <= 0) {
#pragma unroll
      for (int i = 0; i < 32; ++i) g[i] = 0.f;
    } else {
      const float base = st.cp + st.ce * st.ent - st.cb * st.kl;   // terms that do not depend on j
      const float k_lp = st.cb + st.ce;                              // coefficient of log p_j
#pragma unroll
      for (int i = 0; i < 32; ++i) {
        const float lp = v[i] - st.lse;
        const float lq = vr[i] - st.lse_ref;
        g[i] = ex2_approx(lp * kLog2e) * (fmaf(k_lp, lp, base) - st.cb * lq);
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
    const int lane = threadIdx.x & 31;
    constexpr int kBufs = kStagingBytes / kWarps / kBoxBytes;
    const uint32_t buf = staging + (st.n_issued % kBufs) * kBoxBytes;
    if ((c & 1) == 0) {
      if (lane == 0) bulk_wait_group_read<kBufs - 1>();
      __syncwarp();
    }
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      __nv_bfloat162 b0 = __floats2bfloat162_rn(g[8 * j + 0], g[8 * j + 1]);
      __nv_bfloat162 b1 = __floats2bfloat162_rn(g[8 * j + 2], g[8 * j + 3]);
      __nv_bfloat162 b2 = __floats2bfloat162_rn(g[8 * j + 4], g[8 * j + 5]);
      __nv_bfloat162 b3 = __floats2bfloat162_rn(g[8 * j + 6], g[8 * j + 7]);
      const uint32_t jj = uint32_t(4 * (c & 1) + j);
      const uint32_t addr = buf + lane * 128u + ((jj ^ uint32_t(lane & 7)) << 4);
      asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(addr), "r"(*reinterpret_cast<uint32_t*>(&b0)),
                   "r"(*reinterpret_cast<uint32_t*>(&b1)), "r"(*reinterpret_cast<uint32_t*>(&b2)),
                   "r"(*reinterpret_cast<uint32_t*>(&b3))
                   : "memory");
    }
    if (c & 1) {
      fence_proxy_async_smem();
      __syncwarp();
      if (lane == 0) {
        tma_store_2d(tmG, buf, col_l - 32, m_tile * BM + (row_in_tile - lane));
        bulk_commit_group();
      }
      st.n_issued++;
    }
  }
  __device__ static __forceinline__ void end_unit(const Params&, State&, int, int, int, int) {}
};

}  // namespace rlh
