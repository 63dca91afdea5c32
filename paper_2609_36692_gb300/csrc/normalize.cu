// Fused momentum + relaxed tangent momentum + diagonal-Gram normalization
// (Algorithm 1 of the paper: M_t = mu M_{t-1} + G_t; x_i = m_i - <m_i, w_i> w_i
// for every active row; Psi = D(X)^{-1} X, Eq. 3).
//
// Row-active steps (k = 0): one CTA per stored row; the row of M and W stays in
// registers between the two block reductions (<m, w>, then ||x||^2), so the
// step reads G, M_{t-1}, W once and writes M_t, Psi once, with 16-byte vector
// accesses, or (rows that are not whole 16-byte pieces) one element per lane.
//
// Column-active steps (k = 1): the reduction runs down the columns of the
// row-major layout.  Pass A streams G, M_{t-1}, W once, writes M_t and per-
// (row block, column) partial sums of ||m||^2, <m, w> and ||w||^2; a small
// pass folds the partials (fp32 pairs, fixed order, no atomics on floats) into
// a_j = <m_j, w_j> and 1/||x_j|| with ||x||^2 = ||m||^2 - a^2 (2 - ||w||^2);
// pass B re-reads M_t and W and writes Psi.
//
// Zero active rows (undefined in Eq. 3) give zero rows of Psi; count[] gets
// the number of nonzero rows m' (so ||Psi||_F^2 = m').
//
// The tangent step subtracts c_i w_i with c_i = <m_i, w_i> (relaxed, the
// paper's), <m_i, w_i> / ||w_i||^2 (strict tangent ablation; 0 for a zero
// weight row) or 0 (no-tangent ablation), Table 5a.  The strict projection
// of a momentum row parallel to its weight row leaves only rounding, which
// would normalize to a unit row of noise: with the coefficient from fp32
// sums that residue is up to ~1e-5 of ||m_i||, so a strict-tangent row
// whose x_i is at most 1e-3 of ||m_i|| is taken as zero (the kernels'
// fp32 resolution of the projection).  Column-active strict steps sum
// ||x_j||^2 from the subtracted values in an extra pass (the closed form
// ||m||^2 - <m, w>^2 / ||w||^2 cancels for such columns).
#include <type_traits>

#include "common.cuh"
#include "internal.h"

namespace normpre {

constexpr int kColApplyRB = 64;   // rows per block of pass B (16 where that leaves SMs idle)
constexpr int kColThreads = 256;  // 32 column chunks of 8 x 8 row lanes

// The column sums are fp32 pairs (PairSum).  Folded in fp64 they gave the same
// steps bit for bit on every set of perf/cases.py and were 1.6 % slower on LLaMA
// 1B, 2.1 % on Qwen3 (24 additions and conversions per column of a block keep the
// fp64 pipe busy for 3 us).  The fold has the range of fp64 all the same: a
// block's sums whose pairs overflow (a column of entries of 1e18 has a squared
// norm of 1e36 times its rows, though its row lanes stay finite) are kept at
// 2^-4 of their size, marked by the sign bit of a sum that is never negative,
// and a column with a marked or overflowing sum is folded in fp64.
__device__ __forceinline__ float2* col_pairs(const NormLaunch& a) { return reinterpret_cast<float2*>(a.col_part); }
__device__ __forceinline__ float2 mark_wide(const PairSum& p) { return make_float2(copysignf(p.s, -1.f), p.e); }
__device__ __forceinline__ bool is_wide(float2 v) { return __float_as_int(v.x) < 0; }
__device__ __forceinline__ double wide_value(float s, float e, bool wide) {
  return (wide ? 16.0 : 1.0) * (static_cast<double>(s) + static_cast<double>(e));
}

// c_i of the tangent step for mode 0 relaxed, 1 none, 2 strict (mw = <m_i, w_i>,
// ww = ||w_i||^2).
__device__ __forceinline__ float tangent_coef(int mode, float mw, float ww) {
  if (mode == 0) return mw;
  if (mode == 2) return ww > 0.f ? mw / ww : 0.f;
  return 0.f;
}

// Rows per block of pass A: 256, halved down to 32 while the launch has fewer
// than four blocks per SM.  A block walks its rows in rounds of eight, each a
// round trip to HBM, so few tall blocks are latency-bound: one 256 x 1024
// matrix took 28 us in four 256-row blocks.
int col_stats_rows(int64_t rows, int64_t cols, int n) {
  int rb = kColStatsRB;
  const int64_t want = 4 * static_cast<int64_t>(device_sm_count());
  while (rb > 32 && cdiv(cols, 256) * cdiv(rows, rb) * n < want) rb /= 2;
  return rb;
}

size_t normalize_cols_part_bytes(int64_t rows, int64_t cols, int n, int rb) {
  return static_cast<size_t>(n) * cdiv(rows, rb) * cols * 3 * sizeof(double);
}

size_t normalize_cols_scratch_bytes(int64_t rows, int64_t cols, int n, int rb) {
  return normalize_cols_part_bytes(rows, cols, n, rb) + static_cast<size_t>(n) * cols * sizeof(float2) + 256;
}

// ---------------------------------------------------------------------------
// row-active, cols <= 16 * blockDim: 16 elements of the row per thread, in two
// 8-element pieces (VEC: cols % 8 == 0) or one by one, lane next to lane.  The
// element form keeps one pass over HBM for rows of any width (5461 columns,
// bf16 G, fp32 W and Psi: 416 us with the re-reading kernel below, which is
// left for rows past 16384).
// ---------------------------------------------------------------------------
template <typename T, bool VEC>
__device__ __forceinline__ void row_load(const T* p, int64_t j, int64_t cols, float* v) {
  if constexpr (VEC) {
    load8(p + j, v);
  } else {
#pragma unroll
    for (int e = 0; e < 8; ++e) {
      const int64_t je = j + static_cast<int64_t>(e) * blockDim.x;
      v[e] = je < cols ? to_f32(p[je]) : 0.f;
    }
  }
}
template <typename T, bool VEC>
__device__ __forceinline__ void row_store(T* p, int64_t j, int64_t cols, const float* v) {
  if constexpr (VEC) {
    store8(p + j, v);
  } else {
#pragma unroll
    for (int e = 0; e < 8; ++e) {
      const int64_t je = j + static_cast<int64_t>(e) * blockDim.x;
      if (je < cols) p[je] = from_f32<T>(v[e]);
    }
  }
}
// TRIGGER: the next kernel may come early.  Not behind rows of up to 256 columns,
// where at one CTA a row the trigger costs more than that gains (41 x 9728 rows of
// 8, a NormPre-G step: 1000 us with it, 865 without, 924 with plain launches; 20 x
// 2000 x 200 430 and 423; of 400 columns 393 and 398), and not in the element form,
// where it makes no difference; wider rows do not notice it, and other groups'
// kernels gain (13 layers of 384 to 2816 columns, two NormPre-L steps: 3110 us, 3125
// without).  A template parameter, since a branch takes the kernel from 58 to 64
// registers.
template <typename TG, typename TW, typename TP, bool VEC, bool TRIGGER>
__global__ void __launch_bounds__(1024) k_norm_rows(const __grid_constant__ NormLaunch a) {
  pdl_wait();
  if constexpr (TRIGGER) pdl_trigger();
  __shared__ float red[32];
  const int b = blockIdx.y;
  const int64_t row = blockIdx.x;
  const int64_t cols = a.cols;
  const TG* g = static_cast<const TG*>(a.G[b]) + row * cols;
  float* M = a.M[b] + row * cols;
  const TW* w = static_cast<const TW*>(a.W[b]) + row * cols;
  TP* psi = static_cast<TP*>(a.psi[b]) + row * a.psi_ld;
  float m[2][8], wv[2][8];
  float dot = 0.f, wsq = 0.f;
#pragma unroll
  for (int c = 0; c < 2; ++c) {
    const int64_t j = VEC ? (static_cast<int64_t>(c) * blockDim.x + threadIdx.x) * 8
                          : static_cast<int64_t>(c) * 8 * blockDim.x + threadIdx.x;
    if (j < cols) {
      float gv[8], mp[8];
      row_load<TG, VEC>(g, j, cols, gv);
      if constexpr (VEC) load8_cg(M + j, mp);
      else row_load<float, VEC>(M, j, cols, mp);
      row_load<TW, VEC>(w, j, cols, wv[c]);
#pragma unroll
      for (int e = 0; e < 8; ++e) {
        m[c][e] = fmaf(a.mu, mp[e], gv[e]);
        dot = fmaf(m[c][e], wv[c][e], dot);
        wsq = fmaf(wv[c][e], wv[c][e], wsq);
      }
      row_store<float, VEC>(M, j, cols, m[c]);
    } else {
#pragma unroll
      for (int e = 0; e < 8; ++e) { m[c][e] = 0.f; wv[c][e] = 0.f; }
    }
  }
  dot = block_sum(dot, red);
  if (a.tangent == 2) wsq = block_sum(wsq, red);
  const float coef = tangent_coef(a.tangent, dot, wsq);
  float ss = 0.f;
#pragma unroll
  for (int c = 0; c < 2; ++c)
#pragma unroll
    for (int e = 0; e < 8; ++e) {
      m[c][e] = fmaf(-coef, wv[c][e], m[c][e]);
      ss = fmaf(m[c][e], m[c][e], ss);
    }
  ss = block_sum(ss, red);
  if (a.tangent == 2) {
    float mm = 0.f;
#pragma unroll
    for (int c = 0; c < 2; ++c)
#pragma unroll
      for (int e = 0; e < 8; ++e) {
        const float mo = fmaf(coef, wv[c][e], m[c][e]);   // the momentum entry
        mm = fmaf(mo, mo, mm);
      }
    mm = block_sum(mm, red);
    if (ss <= 1e-6f * mm) ss = 0.f;
  }
  const float inv = ss > 0.f ? 1.f / sqrtf(ss) : 0.f;
#pragma unroll
  for (int c = 0; c < 2; ++c) {
    const int64_t j = VEC ? (static_cast<int64_t>(c) * blockDim.x + threadIdx.x) * 8
                          : static_cast<int64_t>(c) * 8 * blockDim.x + threadIdx.x;
    if (j < cols) {
      float v[8];
#pragma unroll
      for (int e = 0; e < 8; ++e) v[e] = m[c][e] * inv;
      row_store<TP, VEC>(psi, j, cols, v);
    }
  }
  if (threadIdx.x == 0) {
    if (ss > 0.f) atomicAdd(&a.count[a.mat_id[b]], 1);
    if (!isfinite(ss) || !isfinite(dot)) raise_flag(a.flags, kFlagNonfinite);
  }
}

// row-active, rows past 16 * 1024 columns: M is re-read by the thread that wrote it
template <typename TG, typename TW, typename TP>
__global__ void __launch_bounds__(256) k_norm_rows_scalar(const __grid_constant__ NormLaunch a) {
  pdl_wait();
  pdl_trigger();
  __shared__ float red[32];
  const int b = blockIdx.y;
  const int64_t row = blockIdx.x;
  const int64_t cols = a.cols;
  const TG* g = static_cast<const TG*>(a.G[b]) + row * cols;
  float* M = a.M[b] + row * cols;
  const TW* w = static_cast<const TW*>(a.W[b]) + row * cols;
  TP* psi = static_cast<TP*>(a.psi[b]) + row * a.psi_ld;
  float dot = 0.f, wsq = 0.f;
  for (int64_t j = threadIdx.x; j < cols; j += blockDim.x) {
    const float m = fmaf(a.mu, M[j], to_f32(g[j]));
    M[j] = m;
    const float wj = to_f32(w[j]);
    dot = fmaf(m, wj, dot);
    wsq = fmaf(wj, wj, wsq);
  }
  dot = block_sum(dot, red);
  if (a.tangent == 2) wsq = block_sum(wsq, red);
  const float coef = tangent_coef(a.tangent, dot, wsq);
  float ss = 0.f;
  float mm = 0.f;
  for (int64_t j = threadIdx.x; j < cols; j += blockDim.x) {
    const float x = fmaf(-coef, to_f32(w[j]), M[j]);
    ss = fmaf(x, x, ss);
    mm = fmaf(M[j], M[j], mm);
  }
  ss = block_sum(ss, red);
  if (a.tangent == 2) {
    mm = block_sum(mm, red);
    if (ss <= 1e-6f * mm) ss = 0.f;
  }
  const float inv = ss > 0.f ? 1.f / sqrtf(ss) : 0.f;
  for (int64_t j = threadIdx.x; j < cols; j += blockDim.x)
    psi[j] = from_f32<TP>(fmaf(-coef, to_f32(w[j]), M[j]) * inv);
  if (threadIdx.x == 0) {
    if (ss > 0.f) atomicAdd(&a.count[a.mat_id[b]], 1);
    if (!isfinite(ss) || !isfinite(dot)) raise_flag(a.flags, kFlagNonfinite);
  }
}

// ---------------------------------------------------------------------------
// column-active pass A: momentum + column partial sums (three pairs s + e per
// row block and column, 8 bytes each)
// grid (ceil(cols / 256), nrb, n); thread = (column chunk cc = tid % 32, row lane rl = tid / 32).
// ---------------------------------------------------------------------------
template <typename TG, typename TW, bool VEC>
__global__ void __launch_bounds__(kColThreads) k_norm_cols_stats(const __grid_constant__ NormLaunch a) {
  pdl_wait();
  pdl_trigger();
  __shared__ float part[8][3][256];
  const int b = blockIdx.z, rb = blockIdx.y;
  const int cc = threadIdx.x & 31, rl = threadIdx.x >> 5;
  const int64_t rows = a.rows, cols = a.cols;
  const int64_t r0 = static_cast<int64_t>(rb) * a.col_rb;
  const int64_t r1 = min(r0 + a.col_rb, rows);
  const TG* g = static_cast<const TG*>(a.G[b]);
  float* M = a.M[b];
  const TW* w = static_cast<const TW*>(a.W[b]);
  float smm[8], smw[8], sww[8];
#pragma unroll
  for (int e = 0; e < 8; ++e) { smm[e] = 0.f; smw[e] = 0.f; sww[e] = 0.f; }
  if (VEC) {
    const int64_t j0 = static_cast<int64_t>(blockIdx.x) * 256 + cc * 8;
    if (j0 < cols) {
      // a 32-bit counter takes the form with bf16 G and W from 82 registers (two
      // CTAs per SM) to 60: a Qwen3 NormPre-L pass of two steps 16660 and 16190 us;
      // with fp32 W it is slower (LLaMA 1B 16990 us, 16650 with 64 bits)
      using row_t = std::conditional_t<sizeof(TG) + sizeof(TW) == 4, int, int64_t>;
      const row_t end = static_cast<row_t>(r1);
#pragma unroll 4
      for (row_t r = static_cast<row_t>(r0) + rl; r < end; r += 8) {
        float gv[8], mp[8], wv[8];
        load8(g + r * cols + j0, gv);
        load8_cg(M + r * cols + j0, mp);
        load8(w + r * cols + j0, wv);
#pragma unroll
        for (int e = 0; e < 8; ++e) {
          const float m = fmaf(a.mu, mp[e], gv[e]);
          mp[e] = m;
          smm[e] = fmaf(m, m, smm[e]);
          smw[e] = fmaf(m, wv[e], smw[e]);
          sww[e] = fmaf(wv[e], wv[e], sww[e]);
        }
        store8(M + r * cols + j0, mp);
      }
    }
#pragma unroll
    for (int e = 0; e < 8; ++e) {
      part[rl][0][cc * 8 + e] = smm[e];
      part[rl][1][cc * 8 + e] = smw[e];
      part[rl][2][cc * 8 + e] = sww[e];
    }
  } else {
    // rows of any alignment: the thread's columns are cc + 32 e of the strip,
    // so that a warp reads 32 consecutive elements, all of a row's eight at
    // once (column by column, 5461 wide, took 503 us against the 140 of the
    // 16-byte form on as many elements)
    const int64_t j0 = static_cast<int64_t>(blockIdx.x) * 256 + cc;
    const int ne = static_cast<int>(min(static_cast<int64_t>(8), (cols - j0 + 31) / 32));   // <= 0: none
    // the next row's entries are loaded before this row's sums and its M's
    // write: with eight entries of three arrays in flight per thread the loads'
    // latency paced the loop (368 us a launch on 89 M elements, 284 with two
    // rows in flight; the 16-byte form would take 212)
    auto fetch = [&](int64_t r, float (&gv)[8], float (&mp)[8], float (&wv)[8]) {
      const int64_t o = r * cols + j0;
#pragma unroll
      for (int e = 0; e < 8; ++e) {
        const bool ok = e < ne && r < r1;
        gv[e] = ok ? to_f32(g[o + 32 * e]) : 0.f;
        mp[e] = ok ? M[o + 32 * e] : 0.f;
        wv[e] = ok ? to_f32(w[o + 32 * e]) : 0.f;
      }
    };
    float gv[8], mp[8], wv[8];
    fetch(r0 + rl, gv, mp, wv);
    for (int64_t r = r0 + rl; r < r1; r += 8) {
      float gn[8], mn[8], wn[8];
      fetch(r + 8, gn, mn, wn);
      const int64_t o = r * cols + j0;
#pragma unroll
      for (int e = 0; e < 8; ++e) {
        const float m = fmaf(a.mu, mp[e], gv[e]);
        if (e < ne) M[o + 32 * e] = m;
        smm[e] = fmaf(m, m, smm[e]);
        smw[e] = fmaf(m, wv[e], smw[e]);
        sww[e] = fmaf(wv[e], wv[e], sww[e]);
        gv[e] = gn[e]; mp[e] = mn[e]; wv[e] = wn[e];
      }
    }
#pragma unroll
    for (int e = 0; e < 8; ++e) {
      part[rl][0][cc + 32 * e] = smm[e];
      part[rl][1][cc + 32 * e] = smw[e];
      part[rl][2][cc + 32 * e] = sww[e];
    }
  }
  __syncthreads();
  // fold the 8 row lanes (fixed order) and write this block's partials
  const int col = threadIdx.x;   // 0..255
  const int64_t j = static_cast<int64_t>(blockIdx.x) * 256 + col;
  if (j < cols) {
    PairSum s0, s1, s2;
    bool wide = false;
#pragma unroll 1
    for (float f = 1.f;; f = 0.0625f) {
      s0 = s1 = s2 = PairSum();
#pragma unroll
      for (int l = 0; l < 8; ++l) {
        s0.add(f * part[l][0][col]);
        s1.add(f * part[l][1][col]);
        s2.add(f * part[l][2][col]);
      }
      wide = f != 1.f;
      if (wide || isfinite(s0.e + s1.e + s2.e)) break;   // an addition that overflows leaves NaN in e
    }
    const int64_t nrb = gridDim.y;
    float2* p = col_pairs(a) + ((static_cast<int64_t>(b) * nrb + rb) * cols + j) * 3;
    p[0] = make_float2(s0.s, s0.e); p[1] = make_float2(s1.s, s1.e);
    p[2] = wide ? mark_wide(s2) : make_float2(s2.s, s2.e);
  }
}

// column-active fold: per column a_j = <m_j, w_j>, inv_j = 1 / ||x_j||.
// stage 0: both from the pass-A sums (relaxed and no-tangent modes).
// stage 1 (strict): a_j = <m_j, w_j> / ||w_j||^2 only.
// stage 2 (strict): ||x_j||^2 from the direct sums of k_norm_cols_xsq (slot 1),
// ||m_j||^2 from pass A (slot 0), a_j kept.
// 32 columns per CTA (the few fp64 operations of a column spread over all SMs):
// one warp, or past four row blocks eight that take every eighth, since a thread
// walking a column's blocks alone waits for the loads.  65536 x 8, a step of
// NormPre-L: 450 us with eight, 505 with one (1024 blocks); 2048 x 2048, two
// matrices: 332 and 338 (64 blocks); 256 x 1024 228.6 and 229.7 (8).  Launches
// of more than eight warps per SM fill them with one (Qwen3: 11.5 us, 13 with eight)
constexpr int kColFinalWarps = 8, kColFinalOne = 4;   // warps, past as many row blocks
template <int NW>
__global__ void __launch_bounds__(32 * NW) k_norm_cols_final(const __grid_constant__ NormLaunch a, int nrb, int stage) {
  pdl_wait();
  pdl_trigger();
  __shared__ float2 part[NW][3][32];
  __shared__ bool part_wide[NW][32];
  const int b = blockIdx.y, lane = threadIdx.x, y = threadIdx.y;
  const int64_t cols = a.cols;
  const int64_t j = static_cast<int64_t>(blockIdx.x) * 32 + lane;
  const float2* sums = col_pairs(a) + (static_cast<int64_t>(b) * nrb * cols + j) * 3;
  PairSum p0, p1, p2;
  bool wide = false;
  if (j < cols) {
    const float2* p = sums + y * cols * 3;
#pragma unroll 8
    for (int rb = y; rb < nrb; rb += NW) {
      const float2 v0 = p[0], v1 = p[1], v2 = p[2];
      wide |= is_wide(v2) || (stage == 2 && is_wide(v1));
      p0.add(PairSum{v0.x, v0.y}); p1.add(PairSum{v1.x, v1.y}); p2.add(PairSum{v2.x, v2.y});
      p += NW * cols * 3;
    }
  }
  if constexpr (NW > 1) {
    part[y][0][lane] = make_float2(p0.s, p0.e);
    part[y][1][lane] = make_float2(p1.s, p1.e);
    part[y][2][lane] = make_float2(p2.s, p2.e);
    part_wide[y][lane] = wide;
    __syncthreads();
    if (y > 0) return;
#pragma unroll
    for (int w = 1; w < NW; ++w) {
      const float2 v0 = part[w][0][lane], v1 = part[w][1][lane], v2 = part[w][2][lane];
      wide |= part_wide[w][lane];
      p0.add(PairSum{v0.x, v0.y}); p1.add(PairSum{v1.x, v1.y}); p2.add(PairSum{v2.x, v2.y});
    }
  }
  float nz = 0.f;
  if (j < cols) {
    double s0, s1, s2;
    if (!wide && isfinite(p0.e + p1.e + p2.e)) {
      s0 = p0.value(); s1 = p1.value(); s2 = p2.value();
    } else {
      // stage 2: slot 1 has a mark of its own (k_norm_cols_xsq)
      s0 = s1 = s2 = 0;
      const float2* p = sums;
#pragma unroll 1
      for (int rb = 0; rb < nrb; ++rb, p += cols * 3) {
        const float2 v0 = p[0], v1 = p[1], v2 = p[2];
        const bool w2 = is_wide(v2);
        s0 += wide_value(v0.x, v0.y, w2);
        s1 += stage == 2 ? wide_value(fabsf(v1.x), v1.y, is_wide(v1)) : wide_value(v1.x, v1.y, w2);
        s2 += wide_value(fabsf(v2.x), v2.y, w2);
      }
    }
    float2* out = a.col_coef + static_cast<int64_t>(b) * cols + j;
    if (stage == 1) {
      // strict: only the projection coefficient; the norm comes from the direct pass
      *out = make_float2(s2 > 0.0 ? static_cast<float>(s1 / s2) : 0.f, 0.f);
    } else {
      // relaxed: a = S_mw, ||x||^2 = S_mm - a^2 (2 - S_ww); none: a = 0,
      // ||x||^2 = S_mm; strict (stage 2): S_xx summed directly
      double aa, d2;
      if (stage == 2) {
        aa = out->x;
        d2 = s1;
        if (d2 <= 1e-6 * s0) d2 = 0.0;   // parallel to the weight column: no tangent part
      }
      else if (a.tangent == 0) { aa = s1; d2 = s0 - aa * aa * (2.0 - s2); }
      else { aa = 0.0; d2 = s0; }
      if (!(d2 > 0.0)) d2 = (d2 == d2) ? 0.0 : d2;    // clamp rounding below zero, keep NaN
      const float inv = d2 > 0.0 ? static_cast<float>(1.0 / sqrt(d2)) : 0.f;
      *out = make_float2(static_cast<float>(aa), inv);
      nz = d2 > 0.0 ? 1.f : 0.f;
      if (!isfinite(d2) || !isfinite(aa)) raise_flag(a.flags, kFlagNonfinite);
    }
  }
  nz = warp_sum(nz);
  if (lane == 0 && nz > 0.f) atomicAdd(&a.count[a.mat_id[b]], static_cast<int>(nz));
}

// strict tangent, column-active: ||x_j||^2 of this block's rows summed from
// x_ij = m_ij - a_j w_ij itself (no cancellation), into slot 1 of the
// block's partials (the <m, w> sums, already folded into a_j).
// grid and thread layout as pass A.
template <typename TW, bool VEC>
__global__ void __launch_bounds__(kColThreads) k_norm_cols_xsq(const __grid_constant__ NormLaunch a) {
  pdl_wait();
  pdl_trigger();
  __shared__ float part[8][256];
  const int b = blockIdx.z, rb = blockIdx.y;
  const int cc = threadIdx.x & 31, rl = threadIdx.x >> 5;
  const int64_t rows = a.rows, cols = a.cols;
  const int64_t r0 = static_cast<int64_t>(rb) * a.col_rb;
  const int64_t r1 = min(r0 + a.col_rb, rows);
  const float* M = a.M[b];
  const TW* w = static_cast<const TW*>(a.W[b]);
  const float2* coef = a.col_coef + static_cast<int64_t>(b) * cols;
  if (VEC) {
    const int64_t j0 = static_cast<int64_t>(blockIdx.x) * 256 + cc * 8;
    float sx[8];
#pragma unroll
    for (int e = 0; e < 8; ++e) sx[e] = 0.f;
    if (j0 < cols) {
      float ca[8];
#pragma unroll
      for (int e = 0; e < 8; ++e) ca[e] = coef[j0 + e].x;
      for (int64_t r = r0 + rl; r < r1; r += 8) {
        float mv[8], wv[8];
        load8_cg(M + r * cols + j0, mv);
        load8(w + r * cols + j0, wv);
#pragma unroll
        for (int e = 0; e < 8; ++e) {
          const float x = fmaf(-ca[e], wv[e], mv[e]);
          sx[e] = fmaf(x, x, sx[e]);
        }
      }
    }
#pragma unroll
    for (int e = 0; e < 8; ++e) part[rl][cc * 8 + e] = sx[e];
  } else {
#pragma unroll
    for (int e = 0; e < 8; ++e) {
      const int64_t j = static_cast<int64_t>(blockIdx.x) * 256 + cc + 32 * e;
      float sx = 0.f;
      if (j < cols) {
        const float cj = coef[j].x;
        for (int64_t r = r0 + rl; r < r1; r += 8) {
          const float x = fmaf(-cj, to_f32(w[r * cols + j]), M[r * cols + j]);
          sx = fmaf(x, x, sx);
        }
      }
      part[rl][cc + 32 * e] = sx;
    }
  }
  __syncthreads();
  const int col = threadIdx.x;
  const int64_t j = static_cast<int64_t>(blockIdx.x) * 256 + col;
  if (j < cols) {
    PairSum s;
    bool wide = false;
#pragma unroll 1
    for (float f = 1.f;; f = 0.0625f) {
      s = PairSum();
#pragma unroll
      for (int l = 0; l < 8; ++l) s.add(f * part[l][col]);
      wide = f != 1.f;
      if (wide || isfinite(s.e)) break;
    }
    col_pairs(a)[((static_cast<int64_t>(b) * gridDim.y + rb) * cols + j) * 3 + 1] =
        wide ? mark_wide(s) : make_float2(s.s, s.e);
  }
}

// column-active pass B: Psi_ij = (m_ij - a_j w_ij) * inv_j
template <typename TW, typename TP, bool VEC>
__global__ void __launch_bounds__(kColThreads) k_norm_cols_apply(const __grid_constant__ NormLaunch a, int nrows) {
  pdl_wait();
  pdl_trigger();
  const int b = blockIdx.z, rb = blockIdx.y;
  const int cc = threadIdx.x & 31, rl = threadIdx.x >> 5;
  const int64_t rows = a.rows, cols = a.cols;
  const int64_t r0 = static_cast<int64_t>(rb) * nrows;
  const int64_t r1 = min(r0 + nrows, rows);
  const float* M = a.M[b];
  const TW* w = static_cast<const TW*>(a.W[b]);
  TP* psi = static_cast<TP*>(a.psi[b]);
  const float2* coef = a.col_coef + static_cast<int64_t>(b) * cols;
  if (VEC) {
    const int64_t j0 = static_cast<int64_t>(blockIdx.x) * 256 + cc * 8;
    if (j0 >= cols) return;
    float ca[8], ci[8];
#pragma unroll
    for (int e = 0; e < 8; ++e) { const float2 c = coef[j0 + e]; ca[e] = c.x; ci[e] = c.y; }
#pragma unroll 2
    for (int64_t r = r0 + rl; r < r1; r += 8) {
      float mv[8], wv[8];
      load8_cg(M + r * cols + j0, mv);
      load8(w + r * cols + j0, wv);
#pragma unroll
      for (int e = 0; e < 8; ++e) mv[e] = fmaf(-ca[e], wv[e], mv[e]) * ci[e];
      store8(psi + r * a.psi_ld + j0, mv);
    }
  } else {
    const int64_t j0 = static_cast<int64_t>(blockIdx.x) * 256 + cc;
    const int ne = static_cast<int>(min(static_cast<int64_t>(8), (cols - j0 + 31) / 32));   // <= 0: none
    float ca[8], ci[8];
#pragma unroll
    for (int e = 0; e < 8; ++e) {
      const float2 c = e < ne ? coef[j0 + 32 * e] : make_float2(0.f, 0.f);
      ca[e] = c.x; ci[e] = c.y;
    }
    for (int64_t r = r0 + rl; r < r1; r += 8) {
      const int64_t o = r * cols + j0;
      float mv[8], wv[8];
#pragma unroll
      for (int e = 0; e < 8; ++e) {
        mv[e] = e < ne ? M[o + 32 * e] : 0.f;
        wv[e] = e < ne ? to_f32(w[o + 32 * e]) : 0.f;
      }
#pragma unroll
      for (int e = 0; e < 8; ++e)
        if (e < ne) psi[r * a.psi_ld + j0 + 32 * e] = from_f32<TP>(fmaf(-ca[e], wv[e], mv[e]) * ci[e]);
    }
  }
}

// ---------------------------------------------------------------------------
// "Row+Column/Step" (orientation 3, Table 5b): after the row normalization,
// the columns of Psi (stored layout, row stride psi_ld) are normalized in
// place.  Pass 1 sums psi^2 per (block of kColStatsRB rows, column) into fp64
// partials; a fold (one CTA per matrix, fixed order) writes 1 / ||column||
// and sets count[] to the number of nonzero columns (then ||Psi||_F^2);
// pass 2 scales.
// ---------------------------------------------------------------------------
template <typename TP>
__global__ void __launch_bounds__(256) k_psi_colsq(const __grid_constant__ NormLaunch a) {
  pdl_wait();
  pdl_trigger();
  const int b = blockIdx.z, rb = blockIdx.y;
  const int64_t j = static_cast<int64_t>(blockIdx.x) * 256 + threadIdx.x;
  if (j >= a.cols) return;
  const TP* psi = static_cast<const TP*>(a.psi[b]);
  const int64_t r0 = static_cast<int64_t>(rb) * kColStatsRB, r1 = min(r0 + kColStatsRB, a.rows);
  float s = 0.f;
  for (int64_t r = r0; r < r1; ++r) {
    const float v = to_f32(psi[r * a.psi_ld + j]);
    s = fmaf(v, v, s);
  }
  a.col_part[(static_cast<int64_t>(b) * gridDim.y + rb) * a.cols + j] = s;
}

__global__ void __launch_bounds__(256) k_psi_colfold(const __grid_constant__ NormLaunch a, int nrb) {
  pdl_wait();
  pdl_trigger();
  __shared__ float red[32];
  const int b = blockIdx.x;
  float nz = 0.f;
  for (int64_t j = threadIdx.x; j < a.cols; j += blockDim.x) {
    double s = 0;
    for (int rb = 0; rb < nrb; ++rb) s += a.col_part[(static_cast<int64_t>(b) * nrb + rb) * a.cols + j];
    const float inv = s > 0.0 ? static_cast<float>(1.0 / sqrt(s)) : 0.f;
    a.col_coef[static_cast<int64_t>(b) * a.cols + j] = make_float2(0.f, inv);
    nz += s > 0.0 ? 1.f : 0.f;
  }
  nz = block_sum(nz, red);
  if (threadIdx.x == 0) a.count[a.mat_id[b]] = static_cast<int>(nz);
}

template <typename TP>
__global__ void __launch_bounds__(256) k_psi_colscale(const __grid_constant__ NormLaunch a) {
  pdl_wait();
  pdl_trigger();
  const int b = blockIdx.z;
  const int64_t j = static_cast<int64_t>(blockIdx.x) * 256 + threadIdx.x;
  if (j >= a.cols) return;
  const float inv = a.col_coef[static_cast<int64_t>(b) * a.cols + j].y;
  TP* psi = static_cast<TP*>(a.psi[b]);
  const int64_t r0 = static_cast<int64_t>(blockIdx.y) * kColApplyRB, r1 = min(r0 + kColApplyRB, a.rows);
  for (int64_t r = r0; r < r1; ++r) psi[r * a.psi_ld + j] = from_f32<TP>(to_f32(psi[r * a.psi_ld + j]) * inv);
}

cudaError_t launch_normalize_psi_cols(const NormLaunch& a, cudaStream_t s) {
  if (a.n <= 0 || a.rows <= 0 || a.cols <= 0) return cudaSuccess;
  const int nrb = static_cast<int>(cdiv(a.rows, kColStatsRB));
  const unsigned cb = static_cast<unsigned>(cdiv(a.cols, 256));
  if (a.psi_dtype == 1) k_psi_colsq<bf16><<<dim3(cb, nrb, a.n), 256, 0, s>>>(a);
  else k_psi_colsq<float><<<dim3(cb, nrb, a.n), 256, 0, s>>>(a);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  k_psi_colfold<<<a.n, 256, 0, s>>>(a, nrb);
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  const dim3 g2(cb, static_cast<unsigned>(cdiv(a.rows, kColApplyRB)), a.n);
  if (a.psi_dtype == 1) k_psi_colscale<bf16><<<g2, 256, 0, s>>>(a);
  else k_psi_colscale<float><<<g2, 256, 0, s>>>(a);
  return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// launchers
// ---------------------------------------------------------------------------
template <typename F>
static cudaError_t dispatch3(int g, int w, int p, F&& f) {
  // g, w, p: 0 = f32, 1 = bf16
  if (g == 0 && w == 0 && p == 0) return f((float*)0, (float*)0, (float*)0);
  if (g == 0 && w == 0 && p == 1) return f((float*)0, (float*)0, (bf16*)0);
  if (g == 0 && w == 1 && p == 0) return f((float*)0, (bf16*)0, (float*)0);
  if (g == 0 && w == 1 && p == 1) return f((float*)0, (bf16*)0, (bf16*)0);
  if (g == 1 && w == 0 && p == 0) return f((bf16*)0, (float*)0, (float*)0);
  if (g == 1 && w == 0 && p == 1) return f((bf16*)0, (float*)0, (bf16*)0);
  if (g == 1 && w == 1 && p == 0) return f((bf16*)0, (bf16*)0, (float*)0);
  return f((bf16*)0, (bf16*)0, (bf16*)0);
}

cudaError_t launch_normalize_rows(const NormLaunch& a, cudaStream_t s) {
  if (a.n <= 0 || a.rows <= 0 || a.cols <= 0) return cudaSuccess;
  const bool vec = (a.cols % 8 == 0) && (a.psi_ld % 8 == 0) && a.cols <= 16 * 1024;
  const dim3 grid(static_cast<unsigned>(a.rows), static_cast<unsigned>(a.n));
  return dispatch3(a.g_dtype, a.w_dtype, a.psi_dtype, [&](auto* tg, auto* tw, auto* tp) {
    using TG = std::remove_pointer_t<decltype(tg)>;
    using TW = std::remove_pointer_t<decltype(tw)>;
    using TP = std::remove_pointer_t<decltype(tp)>;
    const int threads = static_cast<int>(round_up(cdiv(a.cols, 16), 32));
    if (vec && a.cols > 256) {
      launch_pdl(a.overlap, k_norm_rows<TG, TW, TP, true, true>, dim3(grid), dim3(threads), 0, s, a);
    } else if (vec) {
      launch_pdl(a.overlap, k_norm_rows<TG, TW, TP, true, false>, dim3(grid), dim3(threads), 0, s, a);
    } else if (a.cols <= 16 * 1024) {
      launch_pdl(a.overlap, k_norm_rows<TG, TW, TP, false, false>, dim3(grid), dim3(threads), 0, s, a);
    } else {
      launch_pdl(a.overlap, k_norm_rows_scalar<TG, TW, TP>, dim3(grid), dim3(256), 0, s, a);
    }
    return cudaGetLastError();
  });
}

cudaError_t launch_normalize_cols(const NormLaunch& a, cudaStream_t s) {
  if (a.n <= 0 || a.rows <= 0 || a.cols <= 0) return cudaSuccess;
  const bool vec = (a.cols % 8 == 0) && (a.psi_ld % 8 == 0);
  const int nrb = static_cast<int>(cdiv(a.rows, a.col_rb));
  const dim3 grid(static_cast<unsigned>(cdiv(a.cols, 256)), static_cast<unsigned>(nrb),
                  static_cast<unsigned>(a.n));
  auto fold = [&](bool overlap, int stage) {
    const dim3 fgrid(static_cast<unsigned>(cdiv(a.cols, 32)), a.n);
    if (nrb > kColFinalOne && static_cast<int64_t>(fgrid.x) * a.n < 8 * static_cast<int64_t>(device_sm_count()))
      launch_pdl(overlap, k_norm_cols_final<kColFinalWarps>, fgrid, dim3(32, kColFinalWarps), 0, s, a, nrb, stage);
    else
      launch_pdl(overlap, k_norm_cols_final<1>, fgrid, dim3(32), 0, s, a, nrb, stage);
  };
  const int rb_b = grid.x * cdiv(a.rows, kColApplyRB) * a.n < 4 * static_cast<int64_t>(device_sm_count()) ? 16 : kColApplyRB;
  const dim3 grid_b(grid.x, static_cast<unsigned>(cdiv(a.rows, rb_b)), static_cast<unsigned>(a.n));
  return dispatch3(a.g_dtype, a.w_dtype, a.psi_dtype, [&](auto* tg, auto* tw, auto* tp) {
    using TG = std::remove_pointer_t<decltype(tg)>;
    using TW = std::remove_pointer_t<decltype(tw)>;
    using TP = std::remove_pointer_t<decltype(tp)>;
    if (vec) launch_pdl(a.overlap, k_norm_cols_stats<TG, TW, true>, dim3(grid), dim3(kColThreads), 0, s, a);
    else launch_pdl(a.overlap, k_norm_cols_stats<TG, TW, false>, dim3(grid), dim3(kColThreads), 0, s, a);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    if (a.tangent == 2) {
      // strict: the coefficient first, then ||x_j||^2 summed from x itself
      fold(a.overlap_next, 1);
      if ((e = cudaGetLastError()) != cudaSuccess) return e;
      if (vec) launch_pdl(a.overlap_next, k_norm_cols_xsq<TW, true>, dim3(grid), dim3(kColThreads), 0, s, a);
      else launch_pdl(a.overlap_next, k_norm_cols_xsq<TW, false>, dim3(grid), dim3(kColThreads), 0, s, a);
      if ((e = cudaGetLastError()) != cudaSuccess) return e;
      fold(a.overlap_next, 2);
    } else {
      fold(a.overlap_next, 0);
    }
    e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    if (vec) launch_pdl(a.overlap_next, k_norm_cols_apply<TW, TP, true>, dim3(grid_b), dim3(kColThreads), 0, s, a, rb_b);
    else launch_pdl(a.overlap_next, k_norm_cols_apply<TW, TP, false>, dim3(grid_b), dim3(kColThreads), 0, s, a, rb_b);
    return cudaGetLastError();
  });
}

}  // namespace normpre
