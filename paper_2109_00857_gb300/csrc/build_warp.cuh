// build_warp.cuh -- the FP32 build of groups of slices (steps a2-a6 fused) as
// device functions, shared by the single-model kernel (build_warp.cu) and the
// batched kernel (build_warp_batch.cu).
//
// The landing offset of realization w under action a along x is
// floor(u_w + d_a) (Sec. II-A move, cell(); u = 1/2 + w dt/dx from the DO
// velocity, Sec. II-C, d_a the action's displacement), taken for the exact sum
// of the two floats:
//   floor(u + d) = floor(u) + c_a + [u - floor(u) >= th_a]
// with per-action constants c_a, th_a (ActionTable).  Sorting the distinct
// th_a (T_0 < ... < T_{D-1}) gives each realization one fractional rank
// rho = #{T <= u - floor(u)} that decides the step for every action at once
// ([u - floor(u) >= th_a] = [rho >= le_a]).  So a realization needs one count,
// not one per action, at its fine coordinate X = floor(u) S + rho (S = D + 1)
// per axis, in the state's fine table.
//
// A CTA of NW warps builds a group of NW consecutive slices (NW spw states):
//   count    every warp covers all the group's states -- lane (q, i) state q,
//            realizations i, i + 32/spw, ... -- so a warp's loads touch only
//            32 / (NW spw) coefficient rows (one 128-byte wavefront per 16
//            bytes a lane; a warp on a state of its own needs eight), and
//            each row is read once per group, not once per state.  One pass:
//            the state's table is a window predicted from the coefficients'
//            spread, the exact extremes of u are tracked beside the counts
//            (three-input minima, one instruction per two realizations), and
//            the window is checked afterwards.  Table addresses are masked to
//            the state's power-of-two table, so a realization outside the
//            window corrupts only its own state's table, which is then
//            counted again with the exact window (recount_state; never on the
//            workloads measured: the windows hold 5 to 7 standard deviations,
//            N = 5000 draws reach 4).
//   prefix   warp v owns slice v: in-place 2-D inclusive prefix sums of its
//            states' tables over their exact extents.
//   emit     lane l = row (state q, action a): an offset bin (dx, dy) collects
//            exactly the fine cells X in [(dx - c_a - 1) S + le_a, + S) (and
//            likewise in y) -- a box whose count is four prefix lookups; two
//            scans of the row's bounding box count the entries (sink folded),
//            allocate the slice's columns and write the entry words in
//            ascending order with R(s,a) from the counts.
// Slices whose exact fine tables do not fit are appended to a list that the
// CTA kernel of build_fp32.cu finishes with a full-window histogram and the
// same landing offsets, so a slice's output does not depend on which kernel
// built it.
#pragma once
#include <climits>

#include "build_common.cuh"

namespace mdpgb {

__device__ __forceinline__ void red_add_shared(uint32_t addr, uint32_t v) {
  asm volatile("red.shared.add.u32 [%0], %1;" ::"r"(addr), "r"(v));
}
// NaN-propagating minima and maxima (a non-finite u must reach the extremes)
__device__ __forceinline__ float min_nan(float a, float b) {
  float r;
  asm("min.NaN.f32 %0, %1, %2;" : "=f"(r) : "f"(a), "f"(b));
  return r;
}
__device__ __forceinline__ float min_nan(float a, float b, float c) {
  float r;
  asm("min.NaN.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(b), "f"(c));
  return r;
}
__device__ __forceinline__ float max_nan(float a, float b, float c) {
  float r;
  asm("max.NaN.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(b), "f"(c));
  return r;
}

// Mode-count variants: KT > 0 exactly KT modes; KT == 0 up to kMaxModes (runtime).
template <int KT>
constexpr int kPhi = KT > 0 ? KT : kMaxModes;

// A realization's coefficient row in registers, with the widest loads its
// alignment allows (coeffs are 16-byte aligned).
template <int KT>
struct Row {
  float y[kPhi<KT>];
};
template <int KT>
__device__ __forceinline__ void load_row(const float *__restrict__ yw, int K, Row<KT> &r) {
  if constexpr (KT > 0 && KT % 4 == 0) {
#pragma unroll
    for (int k = 0; k < KT; k += 4) {
      const float4 v = __ldg(reinterpret_cast<const float4 *>(yw + k));
      r.y[k] = v.x; r.y[k + 1] = v.y; r.y[k + 2] = v.z; r.y[k + 3] = v.w;
    }
  } else if constexpr (KT > 0 && KT % 2 == 0) {
#pragma unroll
    for (int k = 0; k < KT; k += 2) {
      const float2 v = __ldg(reinterpret_cast<const float2 *>(yw + k));
      r.y[k] = v.x; r.y[k + 1] = v.y;
    }
  } else if constexpr (KT > 0) {
#pragma unroll
    for (int k = 0; k < KT; ++k) r.y[k] = __ldg(yw + k);
  } else {
#pragma unroll
    for (int k = 0; k < kMaxModes; ++k)
      if (k < K) r.y[k] = __ldg(yw + k);
  }
}

// u of one realization: the CTA kernel's FP32 operations (FMA chain over
// ascending k, then u = fma(w, lam, 1/2)).
template <int KT>
__device__ __forceinline__ float2 velocity_u(const Row<KT> &r, const float (&phx)[kPhi<KT>],
                                             const float (&phy)[kPhi<KT>], float vbx, float vby, int K, float lam) {
  float wx = vbx, wy = vby;
#pragma unroll
  for (int k = 0; k < kPhi<KT>; ++k) {
    if (KT > 0 || k < K) {
      wx = fmaf(r.y[k], phx[k], wx);
      wy = fmaf(r.y[k], phy[k], wy);
    }
  }
  return make_float2(fmaf(wx, lam, 0.5f), fmaf(wy, lam, 0.5f));
}

// ---- fractional ranks ----
// Per CTA, in shared memory: per axis the thresholds T[i] (2 for i >= D) and
// the lookup L[b] = 4 #{T in buckets < b} over kRankBuckets buckets of [0, 1]
// (entry kRankBuckets: f = 1 exactly, which counts like the last bucket).
struct RankTables {
  float T[2][kMaxActions + 4];
  uint8_t L[2][kRankBuckets + 4];
};
struct RankTab {
  const float *T;
  const uint8_t *L;
};
__device__ __forceinline__ RankTab rank_tab(const RankTables &rt, int axis) { return RankTab{rt.T[axis], rt.L[axis]}; }

// Copies a model's rank tables (whole CTA; the caller synchronises).
__device__ __forceinline__ void load_rank_tables(const BuildArgs &a, RankTables &rt) {
  for (int i = threadIdx.x; i < kMaxActions + 2; i += blockDim.x) {
    rt.T[0][i] = a.act.Tx[i];
    rt.T[1][i] = a.act.Ty[i];
  }
  for (int b = threadIdx.x; b <= kRankBuckets; b += blockDim.x) {
    rt.L[0][b] = (uint8_t)(4 * a.act.Lx[min(b, kRankBuckets - 1)]);
    rt.L[1][b] = (uint8_t)(4 * a.act.Ly[min(b, kRankBuckets - 1)]);
  }
}

// floor(u) and the rank of its fraction for |u| < kTame: the floor by adding
// 1.5 2^23 rounded down (its low mantissa bits are floor(u)), the bucket
// floor(128 f) by a product rounded down to a multiple of the smallest float
// (whose bits are the integer): no conversion instruction.  Any other u gives
// some fraction in [0, 1] (saturation; NaN gives 0), so the lookups stay in
// their tables.
constexpr float kTame = 16384.f;
constexpr float kFloorMagic = 12582912.f;          // 1.5 2^23
constexpr uint32_t kFloorBits = 0x4B400000u;       // its bits
struct FloorRank {
  uint32_t n;    // floor(u) + kFloorBits
  uint32_t r4;   // 4 rank
};
// DENSE: more than two thresholds in some bucket (the tail is scanned).
template <bool DENSE>
__device__ __forceinline__ FloorRank floor_rank(float u, const RankTab &rt) {
  const float t = __fadd_rd(u, kFloorMagic);
  const float f = __saturatef(u - (t - kFloorMagic));
  const uint32_t b = __float_as_uint(__fmul_rd(f, __uint_as_float((uint32_t)kRankBuckets)));
  uint32_t r4 = rt.L[b];
  const float *T = reinterpret_cast<const float *>(reinterpret_cast<const char *>(rt.T) + r4);
  // the thresholds below f's bucket come from the lookup; those in the bucket
  // follow them in T and every later one exceeds f, so with at most two per
  // bucket two comparisons finish it
  if constexpr (!DENSE) {
    r4 += (T[0] <= f ? 4u : 0u) + (T[1] <= f ? 4u : 0u);
  } else {
    while (*T <= f) {   // T[D] = 2 > f ends it
      ++T;
      r4 += 4u;
    }
  }
  return FloorRank{__float_as_uint(t), r4};
}
// Fine coordinate of u (|u| < kTame): floor(u) S + rank.
template <bool DENSE>
__device__ __forceinline__ int fine_coord(float u, int S, const RankTab &rt) {
  const FloorRank fr = floor_rank<DENSE>(u, rt);
  return (int)(fr.n - kFloorBits) * S + (int)(fr.r4 >> 2);
}

// A state's fine table over X in [xmin, xmin + gx), Y in [ymin, ymin + gy):
// prefix layout P[i * pitch + j], i <= gx, j <= gy, at word `base` of the
// slice's table memory (row 0 and column 0 stay zero; pitch is odd, so a
// warp's lanes walking rows i, i+1, ... hit distinct banks).
struct FineGeo {
  int xmin, ymin, gx, gy, pitch, base;
};

// ---- shared memory of a CTA ----
// GroupSmem (the batched kernel: with the model's arguments), the extremes
// [NW][NW spw] float4, then, aligned to a state's table, NW slices of `words`
// table words each; a state has words / spw of them, a power of two.
constexpr int kGroupWarps = 8;     // most warps (slices) per CTA
// Per-warp totals, added to the model's counters by warp_flush().
struct WarpAcc {
  unsigned long long samples, nnz, dom, maxrow;
};
struct GroupSmem {
  RankTables rt;
  int4 win[32];                    // [state]: the count window's (xmin, ymin, gx, pitch); gy = pitch - 1
  WarpAcc acc[kGroupWarps];        // per warp (in shared memory: the registers are the count loop's)
  long long next[2];               // next group of the work queue, alternating
  unsigned long long base[kGroupWarps];   // the slices' places in the pool
  int cols[kGroupWarps];           // and their columns
};
// Table words of a slice: the largest power of two <= cap_bins (at least one
// word per state, else 0: no slice fits and all go to the CTA kernel).
__host__ __device__ constexpr int table_words(int cap_bins, int spw) {
  int w = 1;
  while (2 * w <= cap_bins) w *= 2;
  return w >= 32 && w >= spw ? w : 0;
}
// A slice's table memory starts at a multiple of this: a state's table, for
// the address mask, and 16 bytes, for the vector stores that clear it.
__host__ __device__ constexpr uint32_t table_align(int words, int spw) {
  return 4u * (uint32_t)(words / spw) > 16u ? 4u * (uint32_t)(words / spw) : 16u;
}
__host__ __device__ constexpr int group_warps(int warps, int spw) {
  const int most = 32 / spw < kGroupWarps ? 32 / spw : kGroupWarps;   // at most one state per lane
  return warps < most ? warps : most;
}
// Bytes before the table memory is aligned: the head struct and the extremes.
__host__ __device__ constexpr uint32_t group_head_bytes(size_t head, int spw, int nw) {
  return (uint32_t)((head + 15) & ~(size_t)15) + 16u * (uint32_t)(nw * nw * spw);
}
// Dynamic shared memory of a CTA.  `reserved` bytes precede it in the shared
// window (the system's; the kernels have no static shared memory), so the
// head fills the gap below the first aligned table: 72 KB and three CTAs per
// SM at 2048 words, where reserving a worst-case gap allowed two.
inline size_t group_smem_bytes(size_t head, int reserved, int cap_bins, int spw, int nw) {
  const int words = table_words(cap_bins, spw);
  const uint32_t al = table_align(words, spw), hd = (uint32_t)reserved + group_head_bytes(head, spw, nw);
  return (size_t)((hd + al - 1) / al * al - (uint32_t)reserved) + (size_t)nw * 4u * (size_t)words;
}
inline cudaError_t reserved_smem(int *bytes) {
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(bytes, cudaDevAttrReservedSharedMemoryPerBlock, dev);
  return e;
}
// The CTA's table memory in its dynamic shared memory.  Should the tables not
// fit behind the alignment (another layout of the shared window), *words
// becomes 0: every sampled slice then goes to the CTA kernel.
__device__ __forceinline__ uint32_t *table_memory(unsigned char *smem, size_t head, int *words, int spw) {
  const int nw = blockDim.x >> 5;
  const uint32_t used = group_head_bytes(head, spw, nw), al = table_align(*words, spw);
  const uint32_t b = smem_u32(smem) + used, off = used + (((b + al - 1) & ~(al - 1)) - b);
  uint32_t size;
  asm("mov.u32 %0, %%dynamic_smem_size;" : "=r"(size));
  if (off + (uint32_t)nw * 4u * (uint32_t)*words > size) *words = 0;
  return reinterpret_cast<uint32_t *>(smem + off);
}
// (lane 0 of each warp owns its totals)
__device__ __forceinline__ void warp_clear(GroupSmem &sm) {
  if ((threadIdx.x & 31) == 0) sm.acc[threadIdx.x >> 5] = WarpAcc{0, 0, 0, 0};
}
__device__ __forceinline__ void warp_flush(const BuildArgs &a, GroupSmem &sm) {
  if ((threadIdx.x & 31) == 0) {
    const WarpAcc acc = sm.acc[threadIdx.x >> 5];
    if (acc.nnz) atomicAdd(&a.cnt[CNT_NNZ], acc.nnz);
    if (acc.dom) atomicAdd(&a.cnt[CNT_DOMAIN], acc.dom);
    if (acc.samples) atomicAdd(&a.cnt[CNT_SAMPLES], acc.samples);
    if (acc.maxrow) atomicMax(&a.cnt[CNT_MAXROW], acc.maxrow);
  }
  warp_clear(sm);
}
__device__ __forceinline__ void clear_tables(uint32_t *tabs, int words) {   // whole CTA
  for (int i = threadIdx.x; i < words * (int)(blockDim.x >> 5); i += blockDim.x) tabs[i] = 0u;
}

// The window a state's counts start from: centre and half width kSpread
// standard deviations (the coefficients' means and variances per layer through
// the state's modes), the half widths shrunk together until the table fits,
// spare rows split between both ends.  Measured need on the large workload:
// 921 cells on average, 1739 at most, of 2048.
constexpr float kSpread = 7.f;
template <int KT, bool DENSE>
__device__ __forceinline__ FineGeo predict_window(const BuildArgs &a, int64_t t, const float (&phx)[kPhi<KT>],
                                                  const float (&phy)[kPhi<KT>], float vbx, float vby, int K, int Sx,
                                                  int Sy, const RankTables &rt, int words) {
  float cx = vbx, cy = vby, vx = 0.f, vy = 0.f;
#pragma unroll
  for (int k = 0; k < kPhi<KT>; ++k) {
    if (KT > 0 || k < K) {
      float m = 0.f, v = a.coef_var[k];
      if (a.mom) {
        const float2 mv = __ldg(a.mom + (size_t)t * K + k);
        m = mv.x;
        v = mv.y;
      }
      cx = fmaf(m, phx[k], cx);
      cy = fmaf(m, phy[k], cy);
      vx = fmaf(v * phx[k], phx[k], vx);
      vy = fmaf(v * phy[k], phy[k], vy);
    }
  }
  const float lim = 0.5f * kTame;
  cx = fmaf(cx, a.lam, 0.5f);
  cy = fmaf(cy, a.lam, 0.5f);
  if (!(fabsf(cx) < lim)) cx = 0.f;
  if (!(fabsf(cy) < lim)) cy = 0.f;
  // standard deviations in cells, at least one fine cell and at most 64 cells
  const float sx = fminf(fmaxf(a.lam * sqrtf(vx), 1.f / (float)Sx), 64.f);
  const float sy = fminf(fmaxf(a.lam * sqrtf(vy), 1.f / (float)Sy), 64.f);
  // (2 h sx Sx + 2)(2 h sy Sy + 2) <= words for the half width h (in standard deviations)
  const float p = 2.f * sx * (float)Sx, q = 2.f * sy * (float)Sy, s = p + q;
  const float h = fminf(kSpread, (sqrtf(s * s + p * q * ((float)words - 4.f)) - s) / (p * q));
  FineGeo g;
  g.ymin = fine_coord<DENSE>(cy - h * sy, Sy, rank_tab(rt, 1));
  g.gy = min(fine_coord<DENSE>(cy + h * sy, Sy, rank_tab(rt, 1)) - g.ymin + 1, words / 2 - 2);
  g.gy = max(g.gy, 1);
  g.pitch = (g.gy + 1) | 1;
  g.gy = g.pitch - 1;
  g.gx = words / g.pitch - 1;
  const int x0 = fine_coord<DENSE>(cx - h * sx, Sx, rank_tab(rt, 0));
  const int x1 = fine_coord<DENSE>(cx + h * sx, Sx, rank_tab(rt, 0));
  g.xmin = x0 - (g.gx - (x1 - x0 + 1)) / 2;
  g.base = 0;
  return g;
}

// Counts state s again with the exact table g (the warp owning its slice;
// tab: the state's table memory).  Rare: see the file comment.
template <int KT, bool DENSE>
__device__ __noinline__ void recount_state(const BuildArgs &a, const RankTables &rt, int64_t s, const FineGeo g,
                                           uint32_t *tab, int words) {
  const int lane = threadIdx.x & 31, K = KT > 0 ? KT : a.K;
  const RankTab rx = rank_tab(rt, 0), ry = rank_tab(rt, 1);
  const int Sx = a.act.Dx + 1, Sy = a.act.Dy + 1;
  const int64_t t = s / a.Nc, c = s % a.Nc;
  const float *vbar = static_cast<const float *>(a.vbar), *modes = static_cast<const float *>(a.modes);
  const float *Yt = static_cast<const float *>(a.Y) + (size_t)t * a.N * K;
  float phx[kPhi<KT>], phy[kPhi<KT>];
#pragma unroll
  for (int k = 0; k < kPhi<KT>; ++k) {
    phx[k] = phy[k] = 0.f;
    if (KT > 0 || k < K) {
      const float2 ph = *reinterpret_cast<const float2 *>(modes + 2 * ((t * K + k) * a.Nc + c));
      phx[k] = ph.x;
      phy[k] = ph.y;
    }
  }
  const float vbx = vbar[2 * s], vby = vbar[2 * s + 1];
  for (int i = lane; i < words; i += 32) tab[i] = 0u;
  __syncwarp();
  for (int w = lane; w < a.N; w += 32) {
    Row<KT> y;
    load_row<KT>(Yt + (size_t)w * K, K, y);
    const float2 u = velocity_u<KT>(y, phx, phy, vbx, vby, K, a.lam);
    const int X = fine_coord<DENSE>(u.x, Sx, rx) - g.xmin, Y = fine_coord<DENSE>(u.y, Sy, ry) - g.ymin;
    red_add_shared(smem_u32(tab) + 4u * (uint32_t)((X + 1) * g.pitch + Y + 1), 1u);
  }
  __syncwarp();
}

// In-place 2-D inclusive prefix sums of a counted table (whole warp): P[i][j] =
// sum of the counts X' < i, Y' < j.  Lanes take rows, then columns, four
// cells loaded before they are stored (a lane's loads overlap).
__device__ __forceinline__ void prefix_table(uint32_t *P, const FineGeo &g) {
  const int lane = threadIdx.x & 31;
  __syncwarp();
  for (int i = 1 + lane; i <= g.gx; i += 32) {
    uint32_t *p = P + i * g.pitch + 1;
    uint32_t v = 0;
    int j = 0;
    for (; j + 4 <= g.gy; j += 4, p += 4) {
      uint32_t x0 = p[0], x1 = p[1], x2 = p[2], x3 = p[3];
      x0 += v; x1 += x0; x2 += x1; x3 += x2;
      p[0] = x0; p[1] = x1; p[2] = x2; p[3] = x3;
      v = x3;
    }
    for (; j < g.gy; ++j, ++p) {
      v += *p;
      *p = v;
    }
  }
  __syncwarp();
  for (int j = 1 + lane; j <= g.gy; j += 32) {
    uint32_t *p = P + g.pitch + j;
    uint32_t v = 0;
    int i = 0;
    for (; i + 4 <= g.gx; i += 4, p += 4 * g.pitch) {
      uint32_t x0 = p[0], x1 = p[g.pitch], x2 = p[2 * g.pitch], x3 = p[3 * g.pitch];
      x0 += v; x1 += x0; x2 += x1; x3 += x2;
      p[0] = x0; p[g.pitch] = x1; p[2 * g.pitch] = x2; p[3 * g.pitch] = x3;
      v = x3;
    }
    for (; i < g.gx; ++i, p += g.pitch) {
      v += *p;
      *p = v;
    }
  }
  __syncwarp();
}

// One row of a slice (lane l = row (q, a)) and its state's prefix table.
struct RowGeo {
  FineGeo g;                 // prefix table of the row's state, base relative to the slice's memory
  int kind;
  bool rows;                 // a sampled row inside the sub-grid
  int lox, hix, loy, hiy;    // its landing offsets
};
// What the emit's first half finds: the row's in-domain successors and sink count.
struct RowCount {
  int e;
  uint32_t sink;
};
// The slice's place in the pool.
struct SlicePlace {
  unsigned long long base;
  int W;
  bool fits;
};
struct SliceTotals {
  int dom, sinks;
};

// The emit's end: the sink's share of R, the slice's and the row's fields.
// e: the row's stored successors, ell of them in the ELL columns.
__device__ __forceinline__ SliceTotals emit_tail(const BuildArgs &a, int64_t sl, const RowGeo &r, int e, int ell,
                                                 uint32_t sink, const SlicePlace &pl, float (&R)[3]) {
  const int lane = threadIdx.x & 31;
  const float invN = 1.0f / (float)a.N;
#pragma unroll
  for (int o = 0; o < 3; ++o) {
    if (r.rows && sink) R[o] = fmaf((float)sink * invN, a.rw.f_r_out, R[o]);
    if (r.kind == KIND_SINK) R[o] = a.rw.f_r_out;
  }
  if (e > ell) atomicMax(&a.cnt[CNT_MAXLEN], (unsigned long long)e);
  if (!pl.fits) sink = 0;
  if (lane == 0) {
    a.slice_off[sl] = (pl.fits && pl.W > 0) ? (uint32_t)pl.base : kNoSlice;
    a.slice_w[sl] = (pl.fits && pl.W > 0) ? (uint8_t)pl.W : (uint8_t)0;
  }
  const int64_t ir = sl * 32 + lane;
  a.nnz[ir] = (uint8_t)ell;
  a.sinkc[ir] = (uint16_t)sink;
#pragma unroll
  for (int o = 0; o < 3; ++o)
    if (o < a.rw.n_obj) static_cast<float *>(a.R)[(int64_t)o * a.rows_pad + ir] = R[o];
  return SliceTotals{__reduce_add_sync(0xffffffffu, e), __popc(__ballot_sync(0xffffffffu, sink > 0))};
}

// ---- the emit for any row: two scans of the row's whole bounding box, the
// class of every landing cell from memory ----
template <class F>
__device__ __forceinline__ void scan_row(const BuildArgs &a, int64_t sl, const uint32_t *grid, const RowGeo &r, F &&f) {
  const int lane = threadIdx.x & 31, a_l = lane % a.A_pad;
  const int64_t s_l = sl * a.spw + lane / a.A_pad, Nc = a.Nc;
  const int nx = a.nx, ny = a.ny;
  const int Sx = a.act.Dx + 1, Sy = a.act.Dy + 1;
  const FineGeo &gl = r.g;
  // count of offset bin (di, dj) of this lane's row: a box of the prefix table
  const uint32_t *P = grid + gl.base;
  const int xoff = (-a.act.cx[a_l] - 1) * Sx + a.act.lex[a_l] - gl.xmin;
  const int yoff = (-a.act.cy[a_l] - 1) * Sy + a.act.ley[a_l] - gl.ymin;
  const int64_t t = s_l / Nc, c = s_l % Nc;
  const int ci = (int)(c % nx), cj = (int)(c / nx);
  const int64_t nxt = (t + 1) * Nc;
  for (int dj = r.loy; dj <= r.hiy; ++dj) {
    const int jp = cj + dj, y0 = dj * Sy + yoff;
    const int j0 = min(max(y0, 0), gl.gy), j1 = min(max(y0 + Sy, 0), gl.gy);
    for (int di = r.lox; di <= r.hix; ++di) {
      const int x0 = di * Sx + xoff;
      const int r0 = min(max(x0, 0), gl.gx) * gl.pitch, r1 = min(max(x0 + Sx, 0), gl.gx) * gl.pitch;
      const uint32_t n = P[r1 + j1] - P[r0 + j1] - P[r1 + j0] + P[r0 + j0];
      if (n == 0) continue;
      const int ip = ci + di;
      const bool inside = ip >= 0 && ip < nx && jp >= 0 && jp < ny;
      const int64_t cell = nxt + (int64_t)jp * nx + ip;
      f(dj * nx + di, n, inside ? a.cls[cell] : (uint8_t)CLS_OBSTACLE, cell);
    }
  }
}
template <bool HYB>   // (as write_general; one definition per kernel)
__device__ __noinline__ RowCount count_general(const BuildArgs &a, int64_t sl, const uint32_t *grid, const RowGeo r) {
  RowCount rc{0, 0u};
  if (r.rows)
    scan_row(a, sl, grid, r, [&](int, uint32_t n, uint8_t cc, int64_t) {
      if (cc & CLS_OBSTACLE) rc.sink += n;
      else ++rc.e;
    });
  return rc;
}
// The first row_cap in-domain successors go to the ELL columns, the rest to
// the slice's spill block (HYB); without spill (the batched build) such a row
// is counted and left empty.
template <bool HYB>
__device__ __noinline__ SliceTotals write_general(const BuildArgs &a, int64_t sl, const uint32_t *grid,
                                                  const RowGeo r, const RowCount rc, const SlicePlace pl) {
  const int lane = threadIdx.x & 31, a_l = lane % a.A_pad;
  const float *__restrict__ gbar = static_cast<const float *>(a.gbar);
  const float invN = 1.0f / (float)a.N;
  const bool cap_hit = !HYB && rc.e > a.row_cap;
  if (cap_hit) atomicAdd(&a.cnt[CNT_ROW_CAP], 1ULL);
  int e = cap_hit ? 0 : rc.e, ell = min(e, a.row_cap);
  int64_t sp_at = -1;
  if constexpr (HYB) sp_at = spill_alloc(a, sl, e - ell);
  uint32_t *dst = a.pool + pl.base * 32 + lane;
  const bool write = pl.fits && !cap_hit;
  float R[3] = {0.f, 0.f, 0.f};
  if (r.rows) {
    int k = 0;
    const float F = a.act.F[a_l], g_s = gbar ? gbar[sl * a.spw + lane / a.A_pad] : 0.f;
    scan_row(a, sl, grid, r, [&](int off, uint32_t n, uint8_t cc, int64_t cell) {
      if (cc & CLS_OBSTACLE) return;
      const uint32_t wd = entry_word(off, n);
      if (k < ell) {
        if (write) dst[(size_t)k * 32] = wd;
      } else if (sp_at >= 0) {
        a.spill[sp_at + (k - ell)] = wd;
      }
      ++k;
      const float g_sp = gbar ? gbar[cell] : 0.f, p = (float)n * invN;
      for (int o = 0; o < a.rw.n_obj; ++o)
        R[o] = fmaf(p, step_reward32(a.rw, a.rw.objs[o], F, g_s, g_sp, (cc & CLS_TARGET) != 0), R[o]);
    });
  }
  if (!write) e = ell = 0;
  if (write)   // zero padding up to the slice width
    for (int kk = ell; kk < pl.W; ++kk) dst[(size_t)kk * 32] = 0u;
  return emit_tail(a, sl, r, e, ell, rc.sink, pl, R);
}

// ---- the usual slice: every state's landings in a box of at most 8 x 8
// cells, at most 32 offset bins per row, no row beyond row_cap ----
// The classes of a state's box come as bit masks (one coalesced read per state
// instead of one byte per entry and scan); one scan finds the row's nonzero
// in-domain bins as a mask, with two prefix lookups per bin (a bin's upper edge
// is the next one's lower edge); the write then walks the set bits in step:
// column k of all 32 rows, padding included, is one 128-byte store.
constexpr int kBox = 8;
struct SmallRow {
  uint32_t mask;      // nonzero in-domain bins, bit dj mbx + di
  int mbx;            // bins per mask row; 0: the slice takes the general emit
  int xoff, yoff;     // table coordinates of the first bin's lower edges
  uint32_t tg0, tg1;  // targets in the state's box (bit cy 8 + cx)
  int bit0;           // box bit of the row's first bin
};
template <int SPW>
__device__ __forceinline__ RowCount count_small(const BuildArgs &a, int64_t sl, const uint32_t *grid, const RowGeo &r,
                                                SmallRow &sr) {
  const int lane = threadIdx.x & 31;
  const int spw = SPW > 0 ? SPW : a.spw, A_pad = 32 / spw, q_l = lane / A_pad, a_l = lane % A_pad;
  const int nx = a.nx, ny = a.ny;
  const int64_t Nc = a.Nc;
  const int Sx = a.act.Dx + 1, Sy = a.act.Dy + 1;
  sr = SmallRow{};
  // bounding box of the state's rows
  int bx0 = r.rows ? r.lox : INT_MAX, bx1 = r.rows ? r.hix : INT_MIN;
  int by0 = r.rows ? r.loy : INT_MAX, by1 = r.rows ? r.hiy : INT_MIN;
#pragma unroll
  for (int off = A_pad >> 1; off >= 1; off >>= 1) {
    bx0 = min(bx0, __shfl_xor_sync(0xffffffffu, bx0, off));
    bx1 = max(bx1, __shfl_xor_sync(0xffffffffu, bx1, off));
    by0 = min(by0, __shfl_xor_sync(0xffffffffu, by0, off));
    by1 = max(by1, __shfl_xor_sync(0xffffffffu, by1, off));
  }
  const int nbx = r.rows ? r.hix - r.lox + 1 : 0, nby = r.rows ? r.hiy - r.loy + 1 : 0;
  const int mbx = __reduce_max_sync(0xffffffffu, nbx), mby = __reduce_max_sync(0xffffffffu, nby);
  const bool small = bx1 < bx0 || (bx1 - bx0 < kBox && by1 - by0 < kBox);
  RowCount rc{0, r.kind == KIND_SINK ? (uint32_t)a.N : 0u};
  if (!__all_sync(0xffffffffu, small) || mbx * mby > 32) return rc;
  sr.mbx = max(mbx, 1);
  // blocked (outside or obstacle) and target cells of the boxes
  uint32_t blk0 = 0, blk1 = 0;
  for (int q = 0; q < spw; ++q) {
    const int src = q * A_pad;
    const int x0 = __shfl_sync(0xffffffffu, bx0, src), y0 = __shfl_sync(0xffffffffu, by0, src);
    const int x1 = __shfl_sync(0xffffffffu, bx1, src), y1 = __shfl_sync(0xffffffffu, by1, src);
    if (x1 < x0) continue;
    const int64_t s = sl * spw + q, t = layer_of(s, Nc, a.nS), c = s - t * Nc;
    const int cj = (int)layer_of(c, nx, a.nS), ci = (int)(c - (int64_t)cj * nx);
    const uint8_t *cn = a.cls + (t + 1) * Nc;
#pragma unroll
    for (int half = 0; half < 2; ++half) {
      const int cx = lane % kBox, cy = lane / kBox + 4 * half;
      const int ip = ci + x0 + cx, jp = cj + y0 + cy;
      uint8_t cc = CLS_OBSTACLE;
      if (x0 + cx <= x1 && y0 + cy <= y1 && ip >= 0 && ip < nx && jp >= 0 && jp < ny) cc = cn[(int64_t)jp * nx + ip];
      const uint32_t b = __ballot_sync(0xffffffffu, (cc & CLS_OBSTACLE) != 0);
      const uint32_t g = __ballot_sync(0xffffffffu, (cc & CLS_TARGET) != 0);
      if (q == q_l) {
        if (half) { blk1 = b; sr.tg1 = g; }
        else { blk0 = b; sr.tg0 = g; }
      }
    }
  }
  const FineGeo &gl = r.g;
  const uint32_t *P = grid + gl.base;
  if (r.rows) {
    sr.xoff = (r.lox - a.act.cx[a_l] - 1) * Sx + a.act.lex[a_l] - gl.xmin;
    sr.yoff = (r.loy - a.act.cy[a_l] - 1) * Sy + a.act.ley[a_l] - gl.ymin;
    sr.bit0 = (r.loy - by0) * kBox + (r.lox - bx0);
  }
  int j0 = 0, y = sr.yoff, bin = 0, row0 = sr.bit0;   // the first bins start at or below the table's edge
  for (int dj = 0; dj < mby; ++dj, row0 += kBox) {
    y += Sy;
    const int j1 = min(y, gl.gy);
    const bool vj = dj < nby;
    uint32_t prev = 0;
    int x = sr.xoff;
    for (int di = 0; di < mbx; ++di, ++bin) {
      x += Sx;
      if (vj && di < nbx) {
        const int row = min(x, gl.gx) * gl.pitch;   // x > 0: the first bin holds the state's extreme
        const uint32_t v = P[row + j1] - P[row + j0], n = v - prev;
        prev = v;
        const int bit = row0 + di;
        if (((bit & 32 ? blk1 : blk0) >> (bit & 31)) & 1u) rc.sink += n;
        else if (n) sr.mask |= 1u << bin;
      }
    }
    j0 = j1;
  }
  rc.e = __popc(sr.mask);
  if (!__all_sync(0xffffffffu, rc.e <= a.row_cap)) sr.mbx = 0;
  return rc;
}
template <int SPW, bool HYB>
__device__ __forceinline__ SliceTotals write_small(const BuildArgs &a, int64_t sl, const uint32_t *grid,
                                                   const RowGeo &r, const RowCount &rc, const SmallRow &sr,
                                                   const SlicePlace &pl) {
  const int lane = threadIdx.x & 31;
  const int spw = SPW > 0 ? SPW : a.spw, A_pad = 32 / spw, q_l = lane / A_pad, a_l = lane % A_pad;
  const int Sx = a.act.Dx + 1, Sy = a.act.Dy + 1, nx = a.nx;
  if constexpr (HYB) {
    if (lane == 0 && a.spill_off) a.spill_off[sl] = kNoSlice;
  }
  const FineGeo &gl = r.g;
  const uint32_t *P = grid + gl.base;
  const float *__restrict__ gbar = static_cast<const float *>(a.gbar);
  const float *gn = gbar + sl * spw + q_l + a.Nc;   // the state's cell, one layer on
  const float invN = 1.0f / (float)a.N;
  const int n_obj = a.rw.n_obj;
  float rb[3] = {0.f, 0.f, 0.f};   // the rewards' parts known from the row
  bool net = false;
  {
    const float F = r.rows ? a.act.F[a_l] : 0.f;
    const float g_s = r.rows && gbar ? gbar[sl * spw + q_l] : 0.f;
#pragma unroll
    for (int o = 0; o < 3; ++o) {
      if (o < n_obj) {
        rb[o] = reward_base32(a.rw, a.rw.objs[o], F, g_s);
        net |= a.rw.objs[o] == MDP_OBJ_NET_ENERGY;
      }
    }
  }
  const int div = (65536 + sr.mbx - 1) / sr.mbx;   // bin / mbx for bin < 32
  const bool any_target = __any_sync(0xffffffffu, (sr.tg0 | sr.tg1) != 0);
  uint32_t *dst = a.pool + pl.base * 32 + lane;
  uint32_t mask = sr.mask;
  float R[3] = {0.f, 0.f, 0.f};
  for (int k = 0; k < pl.W; ++k, dst += 32) {
    uint32_t wd = 0u;
    if (mask) {
      const int bin = __ffs(mask) - 1;
      mask &= mask - 1;
      const int dj = (bin * div) >> 16, di = bin - dj * sr.mbx;
      const int x0 = sr.xoff + di * Sx, y0 = sr.yoff + dj * Sy;
      const int r0 = max(x0, 0) * gl.pitch, r1 = min(x0 + Sx, gl.gx) * gl.pitch;
      const int j0 = max(y0, 0), j1 = min(y0 + Sy, gl.gy);
      const uint32_t n = P[r1 + j1] - P[r0 + j1] - P[r1 + j0] + P[r0 + j0];
      const int off = (r.loy + dj) * nx + r.lox + di;
      wd = entry_word(off, n);
      const float p = (float)n * invN;
      const float g_sp = net ? gn[off] : 0.f;
      bool is_t = false;
      if (any_target) {
        const int bit = sr.bit0 + dj * kBox + di;
        is_t = (((bit & 32 ? sr.tg1 : sr.tg0) >> (bit & 31)) & 1u) != 0;
      }
#pragma unroll
      for (int o = 0; o < 3; ++o)
        if (o < n_obj) R[o] = fmaf(p, reward_cell32(a.rw, a.rw.objs[o], rb[o], g_sp, is_t), R[o]);
    }
    if (pl.fits) *dst = wd;
  }
  const int e = pl.fits ? rc.e : 0;
  return emit_tail(a, sl, r, e, e, rc.sink, pl, R);
}

// The CTA builds the slices [sl0, sl0 + NW) of model a (those below
// a.slice_end), NW = blockDim.x / 32 with NW SPW <= 32 states; every thread
// calls it, and the caller synchronises before sm is used again.  ext: the
// extremes' exchange, (min x, min y, -max x, -max y) of u.  tabs: the
// slices' table memory (all zero on entry and on return), `words` words each.
// SPW > 0: states per slice fixed at compile time; SPW == 0: runtime spw.
// KT: see kPhi.  HYB: rows beyond row_cap keep their tail in the slice's spill
// block; without it (the batched build, whose models keep no spill area) such
// a row is counted in CNT_ROW_CAP and left empty.
// next_group: thread 0's next work-queue index, published in sm.next[par]
// (taken before the count, so its latency is hidden).
template <int KT, int SPW, bool HYB, bool DENSE>
__device__ __forceinline__ void group_slices(const BuildArgs &a, int64_t sl0, GroupSmem &sm, float4 *ext,
                                             uint32_t *tabs, int words, long long next_group, int par) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, NW = blockDim.x >> 5;
  const int spw = SPW > 0 ? SPW : a.spw;
  const int K = KT > 0 ? KT : a.K;
  // model scalars in registers: the loops below also store to memory, so
  // loads through `a` (shared memory in the batched kernel) would repeat
  const int N = a.N;
  const int64_t Nc = a.Nc;
  const float lam = a.lam;
  const RankTab rx = rank_tab(sm.rt, 0), ry = rank_tab(sm.rt, 1);
  const int Sx = a.act.Dx + 1, Sy = a.act.Dy + 1;
  const int swords = words / spw;   // a state's table (power of two)
  const int G = NW * spw, lps = 32 / G;

  // ---- count: lane (q_t, i) state q_t of the group
  {
    const int q_t = lane / lps, w0 = warp * lps + lane % lps;
    const int64_t s_t = sl0 * spw + q_t;
    const bool sample = q_t < G && s_t < a.slice_end * spw && state_kind(a, s_t) == KIND_SAMPLE;
    float mnx = INFINITY, mny = INFINITY, mxx = -INFINITY, mxy = -INFINITY;
    if (sample && swords > 0) {
      const int64_t t = layer_of(s_t, Nc, a.nS), c = s_t - t * Nc;
      const float vbx = static_cast<const float *>(a.vbar)[2 * s_t], vby = static_cast<const float *>(a.vbar)[2 * s_t + 1];
      const float *modes = static_cast<const float *>(a.modes);
      float phx[kPhi<KT>], phy[kPhi<KT>];
#pragma unroll
      for (int k = 0; k < kPhi<KT>; ++k) {
        phx[k] = phy[k] = 0.f;
        if (KT > 0 || k < K) {
          const float2 ph = *reinterpret_cast<const float2 *>(modes + 2 * ((t * K + k) * Nc + c));
          phx[k] = ph.x;
          phy[k] = ph.y;
        }
      }
      const FineGeo win = predict_window<KT, DENSE>(a, t, phx, phy, vbx, vby, K, Sx, Sy, sm.rt, swords);
      if (threadIdx.x < 32 && lane % lps == 0) sm.win[q_t] = make_int4(win.xmin, win.ymin, win.gx, win.pitch);
      // byte address of fine cell (X, Y): base | (4 ((X - xmin + 1) pitch + Y - ymin + 1) mod the table),
      // X = (n - kFloorBits) S + r4 / 4, the constants folded modulo 2^32
      const uint32_t base = smem_u32(tabs + (size_t)q_t * swords), mask = 4u * (uint32_t)(swords - 1);
      const uint32_t cX = 4u * (uint32_t)(Sx * win.pitch), cY = 4u * (uint32_t)Sy, pitch = (uint32_t)win.pitch;
      const uint32_t c0 = 4u * ((uint32_t)(1 - win.xmin) * pitch + (uint32_t)(1 - win.ymin)) - kFloorBits * (cX + cY);
      auto count = [&](float2 u) {
        const FloorRank fx = floor_rank<DENSE>(u.x, rx), fy = floor_rank<DENSE>(u.y, ry);
        const uint32_t lin = fx.n * cX + fx.r4 * pitch + fy.n * cY + (fy.r4 + c0);
        red_add_shared((lin & mask) | base, 1u);
      };
      const int step = 32 / spw;
      const float *yp = static_cast<const float *>(a.Y) + ((size_t)t * N + w0) * K;
      // two realizations per trip; their rows are loaded one trip ahead
      int w = w0;
      Row<KT> y0, y1;
      if (w + step < N) {
        load_row<KT>(yp, K, y0);
        load_row<KT>(yp + (size_t)step * K, K, y1);
      }
#pragma unroll 1
      for (; w + step < N; w += 2 * step) {
        yp += (size_t)(2 * step) * K;
        const float2 u0 = velocity_u<KT>(y0, phx, phy, vbx, vby, K, lam);
        const float2 u1 = velocity_u<KT>(y1, phx, phy, vbx, vby, K, lam);
        if (w + 3 * step < N) {
          load_row<KT>(yp, K, y0);
          load_row<KT>(yp + (size_t)step * K, K, y1);
        }
        mnx = min_nan(mnx, u0.x, u1.x);
        mny = min_nan(mny, u0.y, u1.y);
        mxx = max_nan(mxx, u0.x, u1.x);
        mxy = max_nan(mxy, u0.y, u1.y);
        count(u0);
        count(u1);
      }
      if (w < N) {   // the last realization of an odd number
        load_row<KT>(yp, K, y0);
        const float2 u0 = velocity_u<KT>(y0, phx, phy, vbx, vby, K, lam);
        mnx = min_nan(mnx, u0.x);
        mny = min_nan(mny, u0.y);
        mxx = max_nan(mxx, u0.x, u0.x);
        mxy = max_nan(mxy, u0.y, u0.y);
        count(u0);
      }
    }
    float nxx = -mxx, nxy = -mxy;
    for (int off = lps >> 1; off >= 1; off >>= 1) {
      mnx = min_nan(mnx, __shfl_xor_sync(0xffffffffu, mnx, off));
      mny = min_nan(mny, __shfl_xor_sync(0xffffffffu, mny, off));
      nxx = min_nan(nxx, __shfl_xor_sync(0xffffffffu, nxx, off));
      nxy = min_nan(nxy, __shfl_xor_sync(0xffffffffu, nxy, off));
    }
    if (q_t < G && lane % lps == 0) ext[warp * G + q_t] = make_float4(mnx, mny, nxx, nxy);
    if (threadIdx.x == 0) sm.next[par] = next_group;
  }
  __syncthreads();

  // ---- warp v: slice v, lane l = row (q_l, a_l)
  const int64_t sl = sl0 + warp;
  uint32_t *grid = tabs + (size_t)warp * words;
  RowGeo r{};
  r.hix = r.hiy = -1;
  bool build = sl < a.slice_end, defer = false;
  if (build) {
    const int q_l = lane / (32 / spw), a_l = lane % (32 / spw);
    r.kind = a_l < a.A ? state_kind(a, sl * spw + q_l) : (int)KIND_NONE;
    r.rows = r.kind == KIND_SAMPLE;
    for (int q = 0; q < spw; ++q) {
      const int qg = warp * spw + q;
      const int64_t s = sl * spw + q;
      if (state_kind(a, s) != KIND_SAMPLE) continue;
      // the state's extremes over all warps: lane (i, v) warp i's component v
      const int i = lane >> 2;
      float m = i < NW ? reinterpret_cast<const float *>(&ext[i * G + qg])[lane & 3] : INFINITY;
      m = min_nan(m, __shfl_xor_sync(0xffffffffu, m, 4));
      m = min_nan(m, __shfl_xor_sync(0xffffffffu, m, 8));
      m = min_nan(m, __shfl_xor_sync(0xffffffffu, m, 16));
      const float mnx = __shfl_sync(0xffffffffu, m, 0), mny = __shfl_sync(0xffffffffu, m, 1);
      const float mxx = -__shfl_sync(0xffffffffu, m, 2), mxy = -__shfl_sync(0xffffffffu, m, 3);
      // non-finite or far velocities: the CTA kernel's path
      const bool tame = mnx > -kTame && mxx < kTame && mny > -kTame && mxy < kTame;
      if (!tame || swords == 0) {
        defer = true;
        continue;
      }
      if (q == q_l && r.rows) {
        const int cxa = a.act.cx[a_l], cya = a.act.cy[a_l];
        const float thxa = a.act.thx[a_l], thya = a.act.thy[a_l];
        r.lox = land_offset(mnx, cxa, thxa); r.hix = land_offset(mxx, cxa, thxa);
        r.loy = land_offset(mny, cya, thya); r.hiy = land_offset(mxy, cya, thya);
        if (r.lox < -a.h || r.hix > a.h || r.loy < -a.h || r.hiy > a.h) {   // sub-grid overflow
          r.rows = false;
          atomicAdd(&a.cnt[CNT_OVERFLOW], 1ULL);
        }
      }
      // the exact table inside the window (its pitch, its own origin)
      FineGeo g;
      g.xmin = fine_coord<DENSE>(mnx, Sx, rx);
      g.ymin = fine_coord<DENSE>(mny, Sy, ry);
      g.gx = fine_coord<DENSE>(mxx, Sx, rx) - g.xmin + 1;
      g.gy = fine_coord<DENSE>(mxy, Sy, ry) - g.ymin + 1;
      const int4 win = sm.win[qg];
      g.pitch = win.w;
      g.base = q * swords + (g.xmin - win.x) * g.pitch + (g.ymin - win.y);
      if (g.xmin < win.x || g.ymin < win.y || g.xmin + g.gx > win.x + win.z || g.ymin + g.gy >= win.y + win.w) {
        // outside the predicted window: the exact table, if it fits
        const long long pitch = ((long long)g.gy + 1) | 1;
        if (((long long)g.gx + 1) * pitch > (long long)swords) {
          defer = true;
          continue;
        }
        g.pitch = (int)pitch;
        g.base = q * swords;
        if (!defer) recount_state<KT, DENSE>(a, sm.rt, s, g, grid + g.base, swords);
      }
      if (q == q_l) r.g = g;
      if (!defer) prefix_table(grid + g.base, g);
    }
    if (defer) {   // too wide (or not finite): the CTA kernel builds the slice
      build = false;
      if (lane == 0) {
        const unsigned long long i = atomicAdd(&a.cnt[CNT_DEFER_N], 1ULL);
        a.defer[i] = (uint32_t)sl;
      }
    }
  }
  RowCount rc{};
  SmallRow sr{};
  SlicePlace pl{};
  if (build) {
    rc = count_small<SPW>(a, sl, grid, r, sr);
    if (!sr.mbx) {
      const uint32_t sink = r.kind == KIND_SINK ? (uint32_t)N : 0u;
      rc = count_general<HYB>(a, sl, grid, r);
      rc.sink += sink;
    }
    // (a row the batched build leaves empty takes no columns)
    pl.W = __reduce_max_sync(0xffffffffu, HYB || rc.e <= a.row_cap ? min(rc.e, a.row_cap) : 0);
  }
  // ---- the group's columns: one atomic per group, slices back to back (one
  // per slice is bound by the one address: 4 ns each, 600,000 slices 2.4 ms)
  if (lane == 0) sm.cols[warp] = pl.W;
  __syncthreads();
  if (warp == 0) {
    const int w = lane < NW ? sm.cols[lane] : 0;
    int incl = w;
#pragma unroll
    for (int d = 1; d < kGroupWarps; d <<= 1) {
      const int x = __shfl_up_sync(0xffffffffu, incl, d);
      if (lane >= d) incl += x;
    }
    const int total = __shfl_sync(0xffffffffu, incl, kGroupWarps - 1);
    unsigned long long base = 0;
    if (lane == 0 && total > 0) base = atomicAdd(&a.cnt[CNT_POOL_COLS], (unsigned long long)total);
    base = __shfl_sync(0xffffffffu, base, 0);
    if (lane < NW) sm.base[lane] = base + (unsigned long long)(incl - w);
  }
  __syncthreads();
  if (build) {
    pl.base = sm.base[warp];
    pl.fits = pl.W == 0 || pl.base + (unsigned long long)pl.W <= a.pool_cap_cols;
    if (!pl.fits && lane == 0) atomicAdd(&a.cnt[CNT_POOL_FULL], 1ULL);
    const SliceTotals tot = sr.mbx ? write_small<SPW, HYB>(a, sl, grid, r, rc, sr, pl)
                                   : write_general<HYB>(a, sl, grid, r, rc, pl);
    const int sampled = __popc(__ballot_sync(0xffffffffu, r.rows));
    if (lane == 0) {
      WarpAcc &acc = sm.acc[warp];
      acc.nnz += (unsigned long long)(tot.dom + tot.sinks);
      acc.dom += (unsigned long long)tot.dom;
      acc.samples += (unsigned long long)sampled * (unsigned long long)N;
      if ((unsigned long long)pl.W > acc.maxrow) acc.maxrow = pl.W;
    }
  }
  // the slice's tables are zero again
  __syncwarp();
  uint4 *p = reinterpret_cast<uint4 *>(grid);
  for (int i = lane; i < words / 4; i += 32) p[i] = make_uint4(0u, 0u, 0u, 0u);
}

}  // namespace mdpgb
