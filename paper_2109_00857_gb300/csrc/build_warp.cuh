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
//   count    every warp covers all the group's states: lane (i, p) the states 2 p
//            and 2 p + 1, realizations i, i + 64/spw, ...  The LSU returns 128
//            bytes a cycle to the lanes whatever the addresses, so what a
//            realization's row costs is set by how many states a lane applies
//            it to: two (a third would not fit the registers).  One pass: the
//            state's table is a window predicted from the coefficients' spread,
//            the exact extremes of u are tracked beside the counts (three-input
//            minima, one instruction per two realizations), and the window is
//            checked afterwards.  Table addresses are taken modulo the state's
//            power-of-two table, so a realization outside the window corrupts
//            only its own state's table, which is then counted again with the
//            exact window (recount_slice; rare: the windows hold 5 to 7 standard
//            deviations, N = 5000 draws reach 4).  A state's table is an equal
//            share of the slice's words; a slice with a state that needs more has
//            all its states' exact tables packed and counted again (recount_slice).
//            Bound by issue and the LSU: 46 warp instructions and 11 LSU
//            wavefronts per 32 (state, realization) items -- 17 FMAs, 4 lookups,
//            3 wavefronts of shared counts, 4 of coefficients (the earlier
//            kernel, one state per lane and warp, 128 and 45 over its two passes).
//   prefix   warp v owns slice v: in-place 2-D inclusive prefix sums of its
//            states' tables over their exact extents.
//   emit     lane l = row (state q, action a): an offset bin (dx, dy) collects
//            exactly the fine cells X in [(dx - c_a - 1) S + le_a, + S) (and
//            likewise in y) -- a box of the prefix table.  One scan of the row's
//            bins stages its entry words in ascending order (sink folded), the
//            group allocates its columns, and the rows are copied out with
//            R(s,a) from the counts.
// Slices whose exact fine tables do not fit together are appended to a list that the
// CTA kernel of build_fp32.cu finishes with a full-window histogram and the
// same landing offsets, so a slice's output does not depend on which kernel
// built it.
#pragma once
#include <climits>
#include <cstddef>

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

// Two floats in one 64-bit register pair and their packed operations: one
// instruction works on both (each half rounds like the scalar operation, so a
// realization's u does not depend on the pairing).
using f2 = unsigned long long;
__device__ __forceinline__ f2 pack2(float a, float b) {
  f2 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
  return r;
}
__device__ __forceinline__ float2 unpack2(f2 v) {
  float2 r;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(v));
  return r;
}
__device__ __forceinline__ f2 fma2_down(f2 a, f2 b, f2 c) {
  f2 r;
  asm("fma.rm.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
  return r;
}
__device__ __forceinline__ f2 add2(f2 a, f2 b) {
  f2 r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ f2 add2_down(f2 a, f2 b) {
  f2 r;
  asm("add.rm.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}

// Mode-count variants: KT > 0 exactly KT modes; KT == 0 up to kMaxModes (runtime);
// KT == kNoModes: none, so that all realizations are the same -- a state is counted
// once, by N (100 x 90 cells, 20 layers, 32 actions, N = 500: 1.55 ms as a run-time
// mode count of 0).
constexpr int kNoModes = -1;
template <int KT>
constexpr int kPhi = KT > 0 ? KT : (KT == kNoModes ? 1 : kMaxModes);
template <int KT>
__device__ __forceinline__ int mode_count(int K) {
  return KT > 0 ? KT : (KT == kNoModes ? 0 : K);
}

// A realization's coefficient row, with the widest loads its alignment allows
// (coeffs are 16-byte aligned).
template <int KT>
__device__ __forceinline__ void load_row(const float *__restrict__ yw, int K, float (&y)[kPhi<KT>]) {
  if constexpr (KT > 0 && KT % 4 == 0) {
#pragma unroll
    for (int k = 0; k < KT; k += 4) {
      const float4 v = __ldg(reinterpret_cast<const float4 *>(yw + k));
      y[k] = v.x; y[k + 1] = v.y; y[k + 2] = v.z; y[k + 3] = v.w;
    }
  } else if constexpr (KT > 0 && KT % 2 == 0) {
#pragma unroll
    for (int k = 0; k < KT; k += 2) {
      const float2 v = __ldg(reinterpret_cast<const float2 *>(yw + k));
      y[k] = v.x; y[k + 1] = v.y;
    }
  } else {
#pragma unroll
    for (int k = 0; k < kPhi<KT>; ++k)
      if (KT > 0 || k < K) y[k] = __ldg(yw + k);
  }
}
// Warps (slices of a group) per CTA, and the CTAs per SM that the registers have
// to allow: five CTAs of four warps at 96 registers, two realizations of two
// states in flight per lane.  Measured (build kernel of the large, energy and
// 16-action CSR workloads): 62.8 / 2.81 / 1.04 ms; four CTAs at 128 registers
// 61.2 / 2.95 / 1.08; two CTAs of eight warps 66.4 / 3.08 / 1.17; one realization
// in flight 70.6 / 3.08 / 1.12.
constexpr int kGroupWarps = 4;
template <int KT>
constexpr int kMinCtas = KT == 0 ? 4 : 5;

// ---- fractional ranks ----
// Per CTA, in shared memory: per axis T[1 + i] the thresholds (T[0] = -1, 2
// after the last) and the lookup L[b] = 4 * (thresholds up to and including
// bucket b; MODE 2 and 3: below bucket b) over act.rank_buckets buckets of
// [0, 1]; f = 1 has its own.  The displacements' per-action constants.
struct RankTables {
  float T[2][kMaxActions + 4];
  uint8_t L[2][kMaxBuckets + 4];
  int c[2][kMaxActions], le[2][kMaxActions];
  float th[2][kMaxActions], F[kMaxActions];
};

// Fills a model's tables (whole CTA; the caller synchronises).  (The action
// constants are read per lane: from the constant bank that would be one
// access per distinct action.)
__device__ __forceinline__ void load_rank_tables(const BuildArgs &a, RankTables &rt) {
  const int B = a.act.rank_buckets;
  for (int i = threadIdx.x; i < kMaxActions + 3; i += blockDim.x) {
    rt.T[0][i] = i == 0 ? -1.f : (i <= a.act.Dx ? a.act.Tx[i - 1] : 2.f);
    rt.T[1][i] = i == 0 ? -1.f : (i <= a.act.Dy ? a.act.Ty[i - 1] : 2.f);
  }
  for (int i = threadIdx.x; i < kMaxActions; i += blockDim.x) {
    rt.c[0][i] = a.act.cx[i]; rt.c[1][i] = a.act.cy[i];
    rt.le[0][i] = a.act.lex[i]; rt.le[1][i] = a.act.ley[i];
    rt.th[0][i] = a.act.thx[i]; rt.th[1][i] = a.act.thy[i];
    rt.F[i] = a.act.F[i];
  }
  const bool upto = a.act.rank_mode == 1;
  for (int b = threadIdx.x; b <= B; b += blockDim.x) {
    int nx = 0, ny = 0;
    for (int i = 0; i < a.act.Dx; ++i) nx += (int)(a.act.Tx[i] * (float)B) < b + (upto ? 1 : 0) ? 1 : 0;
    for (int i = 0; i < a.act.Dy; ++i) ny += (int)(a.act.Ty[i] * (float)B) < b + (upto ? 1 : 0) ? 1 : 0;
    if (a.act.rank_mode == 2 && b == 0) {   // all but the first bucket's last two (see ActionTable)
      int mx = 0, my = 0;
      for (int i = 0; i < a.act.Dx; ++i) mx += (int)(a.act.Tx[i] * (float)B) == 0 ? 1 : 0;
      for (int i = 0; i < a.act.Dy; ++i) my += (int)(a.act.Ty[i] * (float)B) == 0 ? 1 : 0;
      nx = max(mx - 2, 0);
      ny = max(my - 2, 0);
    }
    rt.L[0][b] = (uint8_t)(4 * nx);
    rt.L[1][b] = (uint8_t)(4 * ny);
  }
}

// floor(u) for |u| < kTame by adding 1.5 2^23 rounded down: the low mantissa
// bits of the sum are floor(u).
constexpr float kTame = 1e6f;
constexpr float kFloorMagic = 12582912.f;          // 1.5 2^23
constexpr uint32_t kFloorBits = 0x4B400000u;       // its bits
// An integer i < 2^23 as the float whose bits it is (i times the smallest
// float): a product or sum of such floats rounded down is integer arithmetic.
__device__ __forceinline__ float int_float(uint32_t i) { return __uint_as_float(i); }

// Fine coordinate of u (|u| < kTame) along an axis: floor(u) S + rank, rank =
// #{T <= u - floor(u)}; exact for any table.
template <int MODE>
__device__ __forceinline__ int fine_coord(float u, int S, const RankTables &rt, int axis, int buckets) {
  const float t = __fadd_rd(u, kFloorMagic);
  const float f = __saturatef(u - (t - kFloorMagic));
  int r = rt.L[axis][__float_as_uint(__fmul_rd(f, int_float((uint32_t)buckets)))] >> 2;
  const float *T = rt.T[axis] + 1;
  if constexpr (MODE <= 2) {
    while (r > 0 && T[r - 1] > f) --r;
  }
  if constexpr (MODE >= 2) {
    while (T[r] <= f) ++r;   // T[D] = 2 > f ends it
  }
  return (int)(__float_as_uint(t) - kFloorBits) * S + r;
}

// 4 rank of f, its lookup entry at shared address `l`; AXIS selects the
// tables, which follow one another.  MODE 1 is one comparison with the last
// threshold up to f's bucket, MODE 2 two with those in it.
template <int MODE, int AXIS>
__device__ __forceinline__ uint32_t rank4(uint32_t l, float f, uint32_t t_base) {
  uint32_t r;
  if constexpr (MODE == 1) {
    asm volatile(
        "{\n\t.reg .pred p;\n\t.reg .f32 t;\n\t.reg .u32 a;\n\t"
        "ld.shared.u8 %0, [%1 + %4];\n\tadd.u32 a, %0, %3;\n\tld.shared.f32 t, [a + %5];\n\t"
        "setp.lt.f32 p, %2, t;\n\t@p sub.u32 %0, %0, 4;\n\t}"
        : "=&r"(r)
        : "r"(l), "f"(f), "r"(t_base), "n"(AXIS * (int)sizeof(RankTables::L[0])), "n"(AXIS * (int)sizeof(RankTables::T[0])));
  } else {
    asm volatile(
        "{\n\t.reg .pred p, q;\n\t.reg .f32 t, v;\n\t.reg .u32 a;\n\t"
        "ld.shared.u8 %0, [%1 + %4];\n\tadd.u32 a, %0, %3;\n\tld.shared.f32 t, [a + %5];\n\t"
        "ld.shared.f32 v, [a + %6];\n\tsetp.le.f32 p, t, %2;\n\tsetp.le.f32 q, v, %2;\n\t"
        "@p add.u32 %0, %0, 4;\n\t@q add.u32 %0, %0, 4;\n\t}"
        : "=&r"(r)
        : "r"(l), "f"(f), "r"(t_base), "n"(AXIS * (int)sizeof(RankTables::L[0])),
          "n"(AXIS * (int)sizeof(RankTables::T[0]) + 4), "n"(AXIS * (int)sizeof(RankTables::T[0]) + 8));
  }
  return r;
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
// [NW][NW spw] float4, then NW slices of `words` table words each.  A state
// counts into its share of them, a power of two; a slice with a state that needs
// more than its share has its states' exact tables packed into the whole
// (recount_slice).
// Per-warp totals, added to the model's counters by warp_flush().
struct WarpAcc {
  unsigned long long samples, nnz, dom, maxrow;
};
// A state's count set-up.  Its table address of fine cell (X, Y), X = n S + rank
// with n = floor(u) as the bits n + kFloorBits and r4 = 4 rank: the cell index
// modulo the table by 32-bit overflow, lin = n_x aN + r4_x aR + n_y bN + r4_y bR +
// c0 in units of 2^32 / words, its byte offset the high half of lin * bytes.
struct StateSetup {
  int4 win;              // the window's (xmin, ymin, gx, pitch); gy = pitch - 1
  float4 u;              // extremes of u: (min x, min y, max x, max y)
  int4 X;                // and their fine coordinates
  int32_t off;           // the window's first word in the slice's table memory
  uint32_t base, bytes, aN, aR, c0;
  int32_t layer;         // time layer; -1: not sampled
  int32_t kind;          // state_kind
  float vbx, vby;
};
struct GroupSmem {
  RankTables rt;
  WarpAcc acc[kGroupWarps];        // per warp (in shared memory: the registers are the count loop's)
  long long next[2];               // next group of the work queue, alternating
  unsigned long long base[kGroupWarps];   // the slices' places in the pool
  int cols[kGroupWarps];           // and their columns
  uint32_t dummy[32];              // where lanes without a state to count put their counts
  unsigned int trap;               // states to count again (a fraction below act.rank_trap)
  StateSetup st[32];               // the group's states (last: only NW spw are laid out)
};
// Table words of a slice (whole 16-byte vectors), and a state's share: the largest
// power of two that leaves every state one, if that is at least 16 words (else
// 0: nothing is counted at first, and every slice is packed).
__host__ __device__ constexpr int slice_words(int cap_bins) { return (cap_bins + 3) & ~3; }
__host__ __device__ constexpr int share_words(int cap_bins, int spw) {
  int w = 16;
  while (2 * w * spw <= cap_bins) w *= 2;
  return w * spw <= cap_bins ? w : 0;
}
__host__ __device__ constexpr int group_warps(int warps, int spw) {
  const int most = 32 / spw < kGroupWarps ? 32 / spw : kGroupWarps;   // at most one state per lane
  return warps < most ? warps : most;
}
// Entries per row that the emit stages, 1.5 KB per warp (the workloads' longest row: 12).
// A slice with a longer row is written by a second scan; with more staged, a fifth CTA
// would no longer fit an SM from 18 on.
constexpr int kStage = 12;
// Bytes before the table memory (the head, the extremes, the entry stages), and
// of a CTA's dynamic shared memory.
// `before`: bytes the kernel puts in front of GroupSmem (a multiple of 16).
__host__ __device__ constexpr uint32_t group_ext_offset(uint32_t before, int spw, int nw) {
  return (before + (uint32_t)offsetof(GroupSmem, st) + (uint32_t)(nw * spw) * (uint32_t)sizeof(StateSetup) + 15u) & ~15u;
}
__host__ __device__ constexpr uint32_t group_head_bytes(uint32_t before, int spw, int nw) {
  return group_ext_offset(before, spw, nw) + 16u * (uint32_t)(nw * nw * spw) + 128u * (uint32_t)(nw * kStage);
}
inline size_t group_smem_bytes(uint32_t before, int cap_bins, int spw, int nw) {
  return group_head_bytes(before, spw, nw) + (size_t)nw * 4u * (size_t)slice_words(cap_bins);
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
// 921 cells on average, 1739 at most, of 2048.  The table is rotated by up to
// 31 words (base) so that the group's states have their centres in different
// banks: the counts of a warp then meet 3.4-fold conflicts, not 4.7.
constexpr float kSpread = 7.f;
__host__ __device__ constexpr int window_words(int words) { return words >= 256 ? words - 32 : words; }
// Warp v's part for the group whose first slice is sl0: the set-up of its
// slice's states, 32 / spw lanes per state over the modes (so that the count
// loop's warps, which all work on all states, find it in shared memory).  In
// two halves: the loads are issued before the previous group's write and used
// after it.
struct SetupLoads {
  int kind;
  int64_t t;
  float2 vb, ph;   // the state's mean flow; mode lane % per
};
template <int SPW>
__device__ __forceinline__ SetupLoads setup_load(const BuildArgs &a, int64_t sl0) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, spw = SPW > 0 ? SPW : a.spw, per = 32 / spw;
  const int64_t sl = sl0 + warp, s = sl * spw + lane / per, Nc = a.Nc;
  SetupLoads l{KIND_NONE, 0, make_float2(0.f, 0.f), make_float2(0.f, 0.f)};
  if (sl < a.slice_end && s < a.nS) {
    l.kind = state_kind(a, s);
    l.t = layer_of(s, Nc, a.nS);
    l.vb = __ldg(reinterpret_cast<const float2 *>(a.vbar) + s);
    const int k = lane % per;
    if (k < a.K) l.ph = __ldg(reinterpret_cast<const float2 *>(a.modes) + l.t * (a.K - 1) * Nc + s + k * Nc);
  }
  return l;
}
__device__ __forceinline__ float sqrt_fast(float x) {   // (where a window lies, not a result)
  float r;
  asm("sqrt.approx.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}
template <int SPW, int MODE>
__device__ __forceinline__ void setup_slice(const BuildArgs &a, GroupSmem &sm, int64_t sl0, const SetupLoads &ld,
                                            uint32_t *tabs, int words, int table) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, NW = blockDim.x >> 5;
  const int spw = SPW > 0 ? SPW : a.spw, per = 32 / spw, K = a.K, G = NW * spw;
  const int q = warp * spw + lane / per;   // state of the group
  const int64_t t = ld.t;
  const bool sample = ld.kind == KIND_SAMPLE;
  float mx = 0.f, my = 0.f, vx = 0.f, vy = 0.f;
  if (sample) {
    for (int k = lane % per; k < K; k += per) {
      const float2 ph = k < per ? ld.ph
                                : reinterpret_cast<const float2 *>(a.modes)[t * (K - 1) * a.Nc + sl0 * spw + q + k * a.Nc];
      float v = a.coef_var[k];
      if (a.mom) {
        const float2 mv = __ldg(a.mom + (size_t)t * K + k);
        v = mv.y;
        mx = fmaf(mv.x, ph.x, mx);
        my = fmaf(mv.x, ph.y, my);
      }
      vx = fmaf(v * ph.x, ph.x, vx);
      vy = fmaf(v * ph.y, ph.y, vy);
    }
  }
#pragma unroll
  for (int off = 16; off >= 1; off >>= 1) {
    if (off >= per) continue;
    vx += __shfl_xor_sync(0xffffffffu, vx, off);
    vy += __shfl_xor_sync(0xffffffffu, vy, off);
    if (a.mom) {
      mx += __shfl_xor_sync(0xffffffffu, mx, off);
      my += __shfl_xor_sync(0xffffffffu, my, off);
    }
  }
  const int Sx = a.act.Dx + 1, Sy = a.act.Dy + 1, room = window_words(table);
  const float lam = a.lam, lim = 0.5f * kTame;
  float cx = fmaf(ld.vb.x + mx, lam, 0.5f), cy = fmaf(ld.vb.y + my, lam, 0.5f);
  if (!(fabsf(cx) < lim)) cx = 0.f;
  if (!(fabsf(cy) < lim)) cy = 0.f;
  // the window's size in fine cells: h standard deviations (at least half a
  // fine cell each, at most 64 cells) to either side, the fine cells taken as even,
  //   (2 h sx Sx + 2)(2 h sy Sy + 2) <= room
  const float p = 2.f * fminf(fmaxf(lam * sqrt_fast(vx) * (float)Sx, 1.f), 64.f * (float)Sx);
  const float r = 2.f * fminf(fmaxf(lam * sqrt_fast(vy) * (float)Sy, 1.f), 64.f * (float)Sy);
  const float d = p + r, h = fminf(kSpread, __fdividef(sqrt_fast(d * d + p * r * ((float)room - 4.f)) - d, p * r));
  const int gy0 = max(min((int)(h * r) + 2, room / 2 - 2), 1), pitch = (gy0 + 1) | 1, gy = pitch - 1;
  int gx = (int)__fdividef((float)room, (float)pitch);   // rows: room / pitch, one of them the border
  gx -= gx * pitch > room ? 2 : 1;
  // the centre's fine coordinates (x on even lanes, y on odd ones of the state;
  // one lane per state does both)
  int Xc, Yc;
  if (SPW > 0 && SPW <= 16) {
    const bool odd = lane & 1;
    const int c = fine_coord<MODE>(odd ? cy : cx, odd ? Sy : Sx, sm.rt, odd, a.act.rank_buckets);
    const int o = __shfl_xor_sync(0xffffffffu, c, 1);
    Xc = odd ? o : c;
    Yc = odd ? c : o;
  } else {
    Xc = fine_coord<MODE>(cx, Sx, sm.rt, 0, a.act.rank_buckets);
    Yc = fine_coord<MODE>(cy, Sy, sm.rt, 1, a.act.rank_buckets);
  }
  const int xmin = Xc - gx / 2, ymin = Yc - gy / 2;
  const int centre = (Xc - xmin + 1) * pitch + Yc - ymin + 1;
  const int rot = room < table ? (q * 32 / G - centre) & 31 : 0;
  if (lane % per != 0) return;
  StateSetup st;
  st.win = make_int4(xmin, ymin, gx, pitch);
  st.off = lane / per * table + rot;
  st.layer = sample ? (int32_t)t : -1;
  st.kind = ld.kind;
  st.vbx = ld.vb.x;
  st.vby = ld.vb.y;
  const uint32_t sc = table > 0 ? 0x80000000u / (uint32_t)(table / 2) : 0u;   // 2^32 / table
  st.base = table > 0 ? smem_u32(tabs + warp * words + lane / per * table) : smem_u32(&sm.dummy[q]);
  st.bytes = 4u * (uint32_t)table;
  st.aN = (uint32_t)(Sx * pitch) * sc;
  st.aR = (uint32_t)pitch * (sc / 4);
  st.c0 = ((uint32_t)(1 - xmin) * (uint32_t)pitch + (uint32_t)(1 - ymin + rot)) * sc - kFloorBits * (st.aN + (uint32_t)Sy * sc);
  sm.st[q] = st;
}

// Counts state s, the group's q-th, again with the exact table g (the warp owning its
// slice), in the `words` words at g.base of the slice's memory.  Rare where windows hold 5 standard deviations and more, but every
// second state or so where a share is small for its states (few actions, wide
// spreads): hence the counting loop's lookups and two rows in flight.
template <int KT, int MODE>
__device__ __forceinline__ void recount_state(const BuildArgs &a, const GroupSmem &sm, int64_t s, int q, const FineGeo &g,
                                              uint32_t *grid, int words) {
  const RankTables &rt = sm.rt;
  const StateSetup &st = sm.st[q];
  uint32_t *tab = grid + g.base;
  const bool care = MODE <= 2 && (sm.trap >> q & 1u);   // some fraction lies below act.rank_trap
  const int lane = threadIdx.x & 31, K = mode_count<KT>(a.K), B = a.act.rank_buckets, N = a.N;
  const int Sx = a.act.Dx + 1, Sy = a.act.Dy + 1;
  for (int i = lane; i < words; i += 32) tab[i] = 0u;
  __syncwarp();
  if (g.gx == 1 && g.gy == 1) {   // every realization in one cell
    if (lane == 0) tab[g.pitch + 1] = (uint32_t)N;
    return;
  }
  const int64_t t = st.layer;
  const float *Yt = static_cast<const float *>(a.Y) + (size_t)t * N * K;
  const float vbx = st.vbx, vby = st.vby, lam = a.lam, bk = int_float((uint32_t)B);
  float phx[kPhi<KT>], phy[kPhi<KT>];
#pragma unroll
  for (int k = 0; k < kPhi<KT>; ++k) {
    phx[k] = phy[k] = 0.f;
    if (KT > 0 || k < K) {
      const float2 ph = __ldg(reinterpret_cast<const float2 *>(a.modes) + t * (K - 1) * a.Nc + s + k * a.Nc);
      phx[k] = ph.x;
      phy[k] = ph.y;
    }
  }
  // byte address of fine cell (n S + rank, ...), n as its floor's bits (modulo 2^32)
  const uint32_t pitch = (uint32_t)g.pitch, aN = 4u * (uint32_t)Sx * pitch, bN = 4u * (uint32_t)Sy;
  const uint32_t c0 = smem_u32(tab) + 4u * ((uint32_t)(1 - g.xmin) * pitch + (uint32_t)(1 - g.ymin)) - kFloorBits * (aN + bN);
  auto rank4c = [&](float f, int axis) -> uint32_t {   // (rank4; the compiler may interleave it)
    const uint32_t l = rt.L[axis][__float_as_uint(__fmul_rd(f, bk))];
    const float *T = rt.T[axis] + (l >> 2);
    if (MODE == 1) return f < T[0] ? l - 4u : l;
    return l + (T[1] <= f ? 4u : 0u) + (T[2] <= f ? 4u : 0u);
  };
  auto cell = [&](const float (&y)[kPhi<KT>]) -> uint32_t {
    float wx = vbx, wy = vby;
#pragma unroll
    for (int k = 0; k < kPhi<KT>; ++k) {
      if (KT > 0 || k < K) {
        wx = fmaf(y[k], phx[k], wx);
        wy = fmaf(y[k], phy[k], wy);
      }
    }
    const float ux = fmaf(wx, lam, 0.5f), uy = fmaf(wy, lam, 0.5f);
    if (MODE > 2 || care) {
      const int X = fine_coord<MODE>(ux, Sx, rt, 0, B), Y = fine_coord<MODE>(uy, Sy, rt, 1, B);
      return c0 + kFloorBits * (aN + bN) + 4u * ((uint32_t)X * pitch + (uint32_t)Y);
    }
    const float tx = __fadd_rd(ux, kFloorMagic), ty = __fadd_rd(uy, kFloorMagic);
    const uint32_t rx = rank4c(__saturatef(ux - (tx - kFloorMagic)), 0), ry = rank4c(__saturatef(uy - (ty - kFloorMagic)), 1);
    return c0 + __float_as_uint(tx) * aN + rx * pitch + __float_as_uint(ty) * bN + ry;
  };
  constexpr int kRows = KT == 0 ? 1 : 2;
  int w = lane;
  for (; w + 32 * (kRows - 1) < N; w += 32 * kRows) {
    float y[kRows][kPhi<KT>];
    uint32_t at[kRows];
#pragma unroll
    for (int i = 0; i < kRows; ++i) load_row<KT>(Yt + (size_t)(w + 32 * i) * K, K, y[i]);
#pragma unroll
    for (int i = 0; i < kRows; ++i) at[i] = cell(y[i]);
#pragma unroll
    for (int i = 0; i < kRows; ++i) red_add_shared(at[i], 1u);
  }
  for (; w < N; w += 32) {
    float y[kPhi<KT>];
    load_row<KT>(Yt + (size_t)w * K, K, y);
    red_add_shared(cell(y), 1u);
  }
  __syncwarp();
}

// In-place 2-D inclusive prefix sums of a counted table (whole warp): P[i][j] =
// sum of the counts X' < i, Y' < j.  Lanes take rows, then columns, four
// cells loaded before they are stored (a lane's loads overlap).  A few lines
// beyond a multiple of 32 (kScanLines) are scanned across the lanes instead:
// another trip would have them on a few lanes (large workload: 33 x 31 cells
// on average).
constexpr int kScanLines = 8;
__device__ __forceinline__ void prefix_lines(uint32_t *P, int lines, int line_step, int cells, int step) {
  const int lane = threadIdx.x & 31;
  const int tail = (lines & 31) <= kScanLines && cells <= 64 ? lines & 31 : 0, by_lane = lines - tail;
  for (int i = 1 + lane; i <= by_lane; i += 32) {
    uint32_t *p = P + i * line_step + step;
    uint32_t v = 0;
    int j = 0;
    for (; j + 4 <= cells; j += 4, p += 4 * step) {
      uint32_t x0 = p[0], x1 = p[step], x2 = p[2 * step], x3 = p[3 * step];
      x0 += v; x1 += x0; x2 += x1; x3 += x2;
      p[0] = x0; p[step] = x1; p[2 * step] = x2; p[3 * step] = x3;
      v = x3;
    }
    for (; j < cells; ++j, p += step) {
      v += *p;
      *p = v;
    }
  }
  for (int i = by_lane + 1; i <= lines; ++i) {   // lane l: cells 2 l and 2 l + 1 of the line
    uint32_t *p = P + i * line_step + (2 * lane + 1) * step;
    const uint32_t x0 = 2 * lane < cells ? p[0] : 0u, x1 = 2 * lane + 1 < cells ? p[step] : 0u;
    uint32_t incl = x0 + x1;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      const uint32_t x = __shfl_up_sync(0xffffffffu, incl, d);
      if (lane >= d) incl += x;
    }
    if (2 * lane < cells) p[0] = incl - x1;
    if (2 * lane + 1 < cells) p[step] = incl;
  }
  __syncwarp();
}
__device__ __forceinline__ void prefix_table(uint32_t *P, const FineGeo &g) {
  __syncwarp();
  prefix_lines(P, g.gx, g.pitch, g.gy, 1);
  prefix_lines(P, g.gy, 1, g.gx, g.pitch);
}

// A state's extreme over all warps, component lane & 3 of (min x, min y, max x, max y)
// (whole warp: lane (i, v) reads warp i's component v).
__device__ __forceinline__ float state_extreme(const float4 *ext, int qg, int NW, int G) {
  const int lane = threadIdx.x & 31, i = lane >> 2;
  float m = i < NW ? reinterpret_cast<const float *>(&ext[i * G + qg])[lane & 3] : INFINITY;
  m = min_nan(m, __shfl_xor_sync(0xffffffffu, m, 4));
  m = min_nan(m, __shfl_xor_sync(0xffffffffu, m, 8));
  m = min_nan(m, __shfl_xor_sync(0xffffffffu, m, 16));
  return lane & 2 ? -m : m;
}
// The table of exactly a state's extremes, base unset.
__device__ __forceinline__ FineGeo exact_table(const StateSetup &st) {
  FineGeo g;
  g.xmin = st.X.x;
  g.ymin = st.X.y;
  g.gx = st.X.z - st.X.x + 1;
  g.gy = st.X.w - st.X.y + 1;
  g.pitch = (g.gy + 1) | 1;
  g.base = 0;
  return g;
}
__device__ __forceinline__ long long table_cells(const FineGeo &g) { return (long long)(g.gx + 1) * g.pitch; }

// Counts again the states `missed` (bits q) of a slice, whose predicted windows did not
// hold them, each with its exact table in its share of the slice's memory -- or, if
// one of them needs more, every sampled state, the tables back to back in all `words`
// words: what a state leaves is another's.  These tables become the states' windows
// (false: they do not fit together).  Whole warp.
template <int KT, int MODE>
__device__ __noinline__ bool recount_slice(const BuildArgs &a, GroupSmem &sm, int64_t sl, uint32_t *grid, int words,
                                           int share, int spw, uint32_t missed) {
  const int lane = threadIdx.x & 31, first = (threadIdx.x >> 5) * spw;
  StateSetup *st = sm.st + first;
  bool pack = false;
  for (uint32_t left = missed; left; left &= left - 1u)
    pack |= table_cells(exact_table(st[__ffs(left) - 1])) > (long long)share;
  if (pack) {
    missed = 0u;
    long long total = 0;
    for (int q = 0; q < spw; ++q) {
      if (st[q].layer < 0) continue;
      missed |= 1u << q;
      total += table_cells(exact_table(st[q]));
    }
    if (total > (long long)words) return false;
  }
  int base = 0;
  for (uint32_t left = missed; left; left &= left - 1u) {
    const int q = __ffs(left) - 1;
    FineGeo g = exact_table(st[q]);
    const int cells = (int)table_cells(g);
    g.base = pack ? base : q * share;
    base += cells;
    recount_state<KT, MODE>(a, sm, sl * spw + q, first + q, g, grid, pack ? cells : share);
    __syncwarp();
    if (lane == 0) {
      st[q].win = make_int4(g.xmin, g.ymin, g.gx, g.pitch);
      st[q].off = g.base;
    }
  }
  __syncwarp();
  return true;
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
// cells, at most 32 offset bins and kStage entries per row ----
// The classes of a state's box come as bit masks (one coalesced read per state
// instead of one byte per entry and scan); one branch-free scan over the
// row's bins, two prefix lookups per bin (a bin's upper edge is the next one's
// lower edge; bins past the row's end come out empty), stages the entry words in
// shared memory; once the columns are allocated, the rows are copied out in
// step -- column k of all 32 rows, padding included, is one 128-byte store --
// and R is formed from the staged counts.
constexpr int kBox = 8;
struct SmallRow {
  bool small;         // else the slice takes the general emit
  bool any_target;    // some state of the slice may land on a target
};
// The box's part: classes loaded (and turned into masks by ballots later).
struct BoxCells {
  int bx0, by0, mbx, mby;   // the state's box, most bins of a row per axis
  uint8_t cc[2];            // SPW == 1: the lane's two cells
};
template <int SPW>
__device__ __forceinline__ BoxCells box_cells(const BuildArgs &a, int64_t sl, const RowGeo &r, SmallRow &sr,
                                              uint64_t &blk) {
  const int lane = threadIdx.x & 31;
  const int spw = SPW > 0 ? SPW : a.spw, A_pad = 32 / spw, q_l = lane / A_pad;
  const int nx = a.nx, ny = a.ny;
  const int64_t Nc = a.Nc;
  sr = SmallRow{false, false};
  blk = 0;
  // bounding box of the state's rows
  int bx0 = r.rows ? r.lox : INT_MAX, bx1 = r.rows ? r.hix : INT_MIN;
  int by0 = r.rows ? r.loy : INT_MAX, by1 = r.rows ? r.hiy : INT_MIN;
  if (SPW == 1) {
    bx0 = __reduce_min_sync(0xffffffffu, bx0);
    bx1 = __reduce_max_sync(0xffffffffu, bx1);
    by0 = __reduce_min_sync(0xffffffffu, by0);
    by1 = __reduce_max_sync(0xffffffffu, by1);
  } else {
#pragma unroll
    for (int off = A_pad >> 1; off >= 1; off >>= 1) {
      bx0 = min(bx0, __shfl_xor_sync(0xffffffffu, bx0, off));
      bx1 = max(bx1, __shfl_xor_sync(0xffffffffu, bx1, off));
      by0 = min(by0, __shfl_xor_sync(0xffffffffu, by0, off));
      by1 = max(by1, __shfl_xor_sync(0xffffffffu, by1, off));
    }
  }
  const int nbx = r.rows ? r.hix - r.lox + 1 : 0, nby = r.rows ? r.hiy - r.loy + 1 : 0;
  BoxCells bc{bx0, by0, (int)__reduce_max_sync(0xffffffffu, nbx), (int)__reduce_max_sync(0xffffffffu, nby), {0, 0}};
  const bool small = bx1 < bx0 || (bx1 - bx0 < kBox && by1 - by0 < kBox);
  sr.small = __all_sync(0xffffffffu, small) && bc.mbx * bc.mby <= 32;
  if (!sr.small) return bc;
  for (int q = 0; q < spw; ++q) {
    const int src = q * A_pad;
    const int x0 = SPW == 1 ? bx0 : __shfl_sync(0xffffffffu, bx0, src), y0 = SPW == 1 ? by0 : __shfl_sync(0xffffffffu, by0, src);
    const int x1 = SPW == 1 ? bx1 : __shfl_sync(0xffffffffu, bx1, src), y1 = SPW == 1 ? by1 : __shfl_sync(0xffffffffu, by1, src);
    if (x1 < x0) continue;
    const int64_t s = sl * spw + q, t = layer_of(s, Nc, a.nS), c = s - t * Nc;
    const int cj = (int)layer_of(c, nx, a.nS), ci = (int)(c - (int64_t)cj * nx);
    const uint8_t *cn = a.cls + (t + 1) * Nc;
    uint8_t cc[2];
#pragma unroll
    for (int half = 0; half < 2; ++half) {
      const int cx = lane % kBox, cy = lane / kBox + 4 * half;
      const int ip = ci + x0 + cx, jp = cj + y0 + cy;
      cc[half] = CLS_OBSTACLE;
      if (x0 + cx <= x1 && y0 + cy <= y1 && ip >= 0 && ip < nx && jp >= 0 && jp < ny) cc[half] = cn[(int64_t)jp * nx + ip];
    }
    if (SPW == 1) {
      bc.cc[0] = cc[0];
      bc.cc[1] = cc[1];
    } else {
      const uint32_t b0 = __ballot_sync(0xffffffffu, (cc[0] & CLS_OBSTACLE) != 0);
      const uint32_t b1 = __ballot_sync(0xffffffffu, (cc[1] & CLS_OBSTACLE) != 0);
      sr.any_target |= __any_sync(0xffffffffu, ((cc[0] | cc[1]) & CLS_TARGET) != 0) != 0;
      if (q == q_l) blk = (uint64_t)b1 << 32 | b0;
    }
  }
  return bc;
}
template <int SPW>
__device__ __forceinline__ RowCount count_small(const BuildArgs &a, const RankTables &rt, const uint32_t *grid,
                                                const RowGeo &r, const BoxCells &bc, uint64_t blk, uint32_t *stage,
                                                SmallRow &sr) {
  const int lane = threadIdx.x & 31;
  const int A_pad = SPW > 0 ? 32 / SPW : 32 / a.spw, a_l = lane % A_pad;
  const int Sx = a.act.Dx + 1, Sy = a.act.Dy + 1, nx = a.nx, mbx = bc.mbx, mby = bc.mby;
  RowCount rc{0, r.kind == KIND_SINK ? (uint32_t)a.N : 0u};
  if (SPW == 1) {
    const uint32_t b0 = __ballot_sync(0xffffffffu, (bc.cc[0] & CLS_OBSTACLE) != 0);
    const uint32_t b1 = __ballot_sync(0xffffffffu, (bc.cc[1] & CLS_OBSTACLE) != 0);
    sr.any_target = __any_sync(0xffffffffu, ((bc.cc[0] | bc.cc[1]) & CLS_TARGET) != 0) != 0;
    blk = (uint64_t)b1 << 32 | b0;
  }
  const FineGeo &gl = r.g;   // (all zero in rows without a table: every bin comes out empty)
  const uint32_t *P = grid + gl.base;
  int xoff = 0, y = 0, off = 0;
  if (r.rows) {
    xoff = (r.lox - rt.c[0][a_l] - 1) * Sx + rt.le[0][a_l] - gl.xmin;
    y = (r.loy - rt.c[1][a_l] - 1) * Sy + rt.le[1][a_l] - gl.ymin;
    blk >>= (r.loy - bc.by0) * kBox + (r.lox - bc.bx0);
    off = r.loy * nx + r.lox;
  }
  const int gx = r.rows ? gl.gx : 0, gy = r.rows ? gl.gy : 0;
  const uint32_t *p0 = P;   // the first bins start at or below the table's edge
  uint32_t *st = stage + lane;
  for (int dj = 0; dj < mby; ++dj) {
    y += Sy;
    const uint32_t *p1 = P + min(y, gy);
    uint32_t prev = 0, bits = (uint32_t)blk;
    int x = xoff;
    for (int d0 = 0; d0 < mbx; d0 += 4) {   // four bins' lookups in flight
      uint32_t v[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        x += Sx;
        const int row = min(x, gx) * gl.pitch;   // x > 0: the first bin holds the state's extreme
        v[i] = p1[row] - p0[row];
      }
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const uint32_t n = v[i] - prev;
        prev = v[i];
        if (n) {
          if (bits & 1u) {
            rc.sink += n;
          } else {
            if (rc.e < kStage) *st = entry_word(off + d0 + i, n);
            st += 32;
            ++rc.e;
          }
        }
        bits >>= 1;
      }
    }
    p0 = p1;
    blk >>= kBox;
    off += nx;
  }
  sr.small = __all_sync(0xffffffffu, rc.e <= min(a.row_cap, kStage));
  return rc;
}
template <int SPW, bool HYB>
__device__ __forceinline__ SliceTotals write_small(const BuildArgs &a, const RankTables &rt, int64_t sl,
                                                   const RowGeo &r, const RowCount &rc, const uint32_t *stage,
                                                   const SmallRow &sr, const SlicePlace &pl) {
  const int lane = threadIdx.x & 31;
  const int spw = SPW > 0 ? SPW : a.spw, A_pad = 32 / spw, q_l = lane / A_pad, a_l = lane % A_pad;
  if constexpr (HYB) {
    if (lane == 0 && a.spill_off) a.spill_off[sl] = kNoSlice;
  }
  const float *__restrict__ gbar = static_cast<const float *>(a.gbar);
  const int64_t next = sl * spw + q_l + a.Nc;   // the state's cell, one layer on
  const float invN = 1.0f / (float)a.N;
  const int n_obj = a.rw.n_obj;
  // the rewards' parts known from the row; net energy's (the same for every
  // objective slot that asks for it) is finished per cell
  float rb[3] = {0.f, 0.f, 0.f}, rb_net = 0.f;
  bool is_net[3] = {false, false, false};
  bool net = false;
  {
    const float F = rt.F[a_l];
    const float g_s = r.rows && gbar ? gbar[next - a.Nc] : 0.f;
#pragma unroll
    for (int o = 0; o < 3; ++o) {
      if (o < n_obj) {
        rb[o] = reward_base32(a.rw, a.rw.objs[o], F, g_s);
        is_net[o] = a.rw.objs[o] == MDP_OBJ_NET_ENERGY;
        if (is_net[o]) rb_net = rb[o];
        net |= is_net[o];
      }
    }
  }
  uint32_t *dst = a.pool + pl.base * 32 + lane;
  const uint32_t *st = stage + lane;
  float R[3] = {0.f, 0.f, 0.f};
  for (int k0 = 0; k0 < pl.W; k0 += 4, dst += 128, st += 128) {   // four columns' loads in flight
    uint32_t wd[4];
    float g[4];
    uint8_t cc[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const bool in = k0 + i < rc.e;
      wd[i] = in ? st[32 * i] : 0u;
      const int off = (int)(int16_t)(wd[i] & 0xFFFFu);
      g[i] = net && in ? gbar[next + off] : 0.f;
      cc[i] = sr.any_target && in ? a.cls[next + off] : (uint8_t)0;
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      if (pl.fits && k0 + i < pl.W) dst[32 * i] = wd[i];
      if (k0 + i < rc.e) {
        const float p = (float)(wd[i] >> 16) * invN;
        const float rn = reward_cell32(a.rw, MDP_OBJ_NET_ENERGY, rb_net, g[i], false);
#pragma unroll
        for (int o = 0; o < 3; ++o) {
          float x = is_net[o] ? rn : rb[o];
          if (sr.any_target && (cc[i] & CLS_TARGET)) x = __fadd_rn(x, a.rw.f_r_term);
          R[o] = fmaf(p, x, R[o]);
        }
      }
    }
  }
  const int e = pl.fits ? rc.e : 0;
  return emit_tail(a, sl, r, e, e, rc.sink, pl, R);
}

// (set up by setup_slice, synchronised)
// The CTA builds the slices [sl0, sl0 + NW) of model a (those below
// a.slice_end), NW = blockDim.x / 32 with NW SPW <= 32 states; every thread
// calls it, and the caller synchronises before sm is used again.  ext: the
// extremes' exchange, (min x, min y, -max x, -max y) of u.  tabs: the
// slices' table memory (all zero on entry and on return), `words` words each,
// `share` of them a state's.
// SPW > 0: states per slice fixed at compile time; SPW == 0: runtime spw.
// KT: see kPhi.  HYB: rows beyond row_cap keep their tail in the slice's spill
// block; without it (the batched build, whose models keep no spill area) such
// a row is counted in CNT_ROW_CAP and left empty.
// next_group: thread 0's next work-queue index, published in sm.next[par]
// (taken before the count, so its latency is hidden).
// next_first(g): the first slice of queue index g if it belongs to the same
// model and is to be set up here, else -1.
template <int KT, int SPW, bool HYB, int MODE, class F>
__device__ __forceinline__ void group_slices(const BuildArgs &a, int64_t sl0, GroupSmem &sm, float4 *ext,
                                             uint32_t *tabs, int words, int share, long long next_group, int par,
                                             F &&next_first) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, NW = blockDim.x >> 5;
  const int spw = SPW > 0 ? SPW : a.spw;
  const int K = mode_count<KT>(a.K);
  // model scalars in registers: the loops below also store to memory, so
  // loads through `a` (shared memory in the batched kernel) would repeat
  const int N = a.N;
  const int64_t Nc = a.Nc;
  const float lam = a.lam;
  const int B = a.act.rank_buckets;
  const int Sx = a.act.Dx + 1, Sy = a.act.Dy + 1;
  const int G = NW * spw;           // states of the group (even, <= 32)

  // ---- count: lane (i, p) states 2 p and 2 p + 1 of the group, realizations
  // i, i + step, ...; the two states are the halves of every packed operation
  {
    const int np = G / 2, p_t = lane % np, sub = lane / np, subs = 32 / np;
    const int w0 = warp * subs + sub, step = 64 / spw;   // step = NW subs
    const float *modes = static_cast<const float *>(a.modes);
    const int layer0 = sm.st[2 * p_t].layer, layer1 = sm.st[2 * p_t + 1].layer;
    const bool split = layer0 >= 0 && layer1 >= 0 && layer0 != layer1;
    float phx[2][kPhi<KT>], phy[2][kPhi<KT>];
    {
      // neighbouring cells of a layer, unless the pair is split
      const int64_t s0 = sl0 * spw + 2 * p_t;
      const int la = layer0 >= 0 ? layer0 : max(layer1, 0);
      const float *m0 = modes + 2 * ((int64_t)la * (K - 1) * Nc + s0);   // (la K + k) Nc + (s0 - la Nc) at k = 0
      const float *m1 = split ? modes + 2 * ((int64_t)layer1 * (K - 1) * Nc + s0 + 1) : m0 + 2;
#pragma unroll
      for (int k = 0; k < kPhi<KT>; ++k) {
        float2 p0 = make_float2(0.f, 0.f), p1 = p0;
        if (KT > 0 || k < K) {
          if (layer0 >= 0) p0 = __ldg(reinterpret_cast<const float2 *>(m0));
          if (layer1 >= 0) p1 = __ldg(reinterpret_cast<const float2 *>(m1));
          m0 += 2 * Nc;
          m1 += 2 * Nc;
        }
        phx[0][k] = p0.x;
        phy[0][k] = p0.y;
        phx[1][k] = p1.x;
        phy[1][k] = p1.y;
      }
    }
    const uint32_t sc = share > 0 ? 0x80000000u / (uint32_t)(share / 2) : 0u;
    const uint32_t bN = (uint32_t)Sy * sc, bR = sc / 4;
    const uint32_t t_base = smem_u32(&sm.rt.T[0][0]);
    const float lut = int_float(smem_u32(&sm.rt.L[0][0])), bk = int_float((uint32_t)B);
    const f2 lut2 = pack2(lut, lut), bk2 = pack2(bk, bk);
    const f2 magic2 = pack2(kFloorMagic, kFloorMagic), nmagic2 = pack2(-kFloorMagic, -kFloorMagic);
    // a pair of states on both sides of a layer boundary: the second on its own
    // layer's coefficients, in a second round
    const int rounds = __any_sync(0xffffffffu, split) ? 2 : 1;
#pragma unroll 1
    for (int round = 0; round < rounds; ++round) {
      const int t = round == 0 && layer0 >= 0 ? layer0 : layer1;
      const bool on0 = layer0 >= 0 && round == 0, on1 = layer1 >= 0 && (split ? round == 1 : round == 0);
      const StateSetup *st = &sm.st[2 * p_t];
      const uint32_t dummy = smem_u32(&sm.dummy[lane]);
      const uint32_t base0 = on0 ? st[0].base : dummy, base1 = on1 ? st[1].base : dummy;
      const uint32_t bytes0 = on0 ? st[0].bytes : 0u, bytes1 = on1 ? st[1].bytes : 0u;
      const uint32_t aN0 = st[0].aN, aN1 = st[1].aN, aR0 = st[0].aR, aR1 = st[1].aR, c00 = st[0].c0, c01 = st[1].c0;
      const float vbx0 = st[0].vbx, vby0 = st[0].vby, vbx1 = st[1].vbx, vby1 = st[1].vby;
      float mnx0 = INFINITY, mny0 = INFINITY, mnx1 = INFINITY, mny1 = INFINITY;
      float mxx0 = -INFINITY, mxy0 = -INFINITY, mxx1 = -INFINITY, mxy1 = -INFINITY;
      float fmn = 2.f;
      auto red = [&](uint32_t lin, uint32_t bytes, uint32_t base) {
        uint32_t addr;
        asm("mad.hi.u32 %0, %1, %2, %3;" : "=r"(addr) : "r"(lin), "r"(bytes), "r"(base));
        red_add_shared(addr, KT == kNoModes ? (uint32_t)N : 1u);
      };
      // u of a realization for both states (FMA chain over ascending k, then u =
      // fma(w, lam, 1/2): the CTA kernel's operations)
      // (scalar: packed FMAs of the two states would need every coefficient
      // twice in a register pair, two moves each)
      auto velocity = [&](const float (&y)[kPhi<KT>], f2 &ux, f2 &uy) {
        float wx[2] = {vbx0, vbx1}, wy[2] = {vby0, vby1};
#pragma unroll
        for (int k = 0; k < kPhi<KT>; ++k) {
          if (KT > 0 || k < K) {
#pragma unroll
            for (int h = 0; h < 2; ++h) {
              wx[h] = fmaf(y[k], phx[h][k], wx[h]);
              wy[h] = fmaf(y[k], phy[h][k], wy[h]);
            }
          }
        }
        ux = pack2(fmaf(wx[0], lam, 0.5f), fmaf(wx[1], lam, 0.5f));
        uy = pack2(fmaf(wy[0], lam, 0.5f), fmaf(wy[1], lam, 0.5f));
      };
      auto count = [&](f2 wx, f2 wy) {
        const float2 ux = unpack2(wx), uy = unpack2(wy);
        // floor by the magic sum; the fraction saturated to [0, 1] (NaN: 0), so
        // that the lookups stay in their tables whatever u is
        const f2 tx = add2_down(wx, magic2), ty = add2_down(wy, magic2);
        const float2 nx = unpack2(add2(tx, nmagic2)), ny = unpack2(add2(ty, nmagic2));
        const float fx0 = __saturatef(ux.x - nx.x), fx1 = __saturatef(ux.y - nx.y);
        const float fy0 = __saturatef(uy.x - ny.x), fy1 = __saturatef(uy.y - ny.y);
        if constexpr (MODE <= 2) {
          fmn = fminf(fmn, fminf(fx0, fy0));
          fmn = fminf(fmn, fminf(fx1, fy1));
        }
        uint32_t rx0, rx1, ry0, ry1;
        if constexpr (MODE <= 2) {
          // lookup addresses L + floor(B f): integer arithmetic on float bits
          const float2 lx = unpack2(fma2_down(pack2(fx0, fx1), bk2, lut2));
          const float2 ly = unpack2(fma2_down(pack2(fy0, fy1), bk2, lut2));
          rx0 = rank4<MODE, 0>(__float_as_uint(lx.x), fx0, t_base);
          ry0 = rank4<MODE, 1>(__float_as_uint(ly.x), fy0, t_base);
          rx1 = rank4<MODE, 0>(__float_as_uint(lx.y), fx1, t_base);
          ry1 = rank4<MODE, 1>(__float_as_uint(ly.y), fy1, t_base);
        } else {
          auto r4 = [&](float f, int axis) {
            int r = sm.rt.L[axis][__float_as_uint(__fmul_rd(f, bk))] >> 2;
            while (sm.rt.T[axis][r + 1] <= f) ++r;
            return 4u * (uint32_t)r;
          };
          rx0 = r4(fx0, 0); ry0 = r4(fy0, 1);
          rx1 = r4(fx1, 0); ry1 = r4(fy1, 1);
        }
        const float2 bx = unpack2(tx), by = unpack2(ty);
        red(__float_as_uint(bx.x) * aN0 + rx0 * aR0 + __float_as_uint(by.x) * bN + ry0 * bR + c00, bytes0, base0);
        red(__float_as_uint(bx.y) * aN1 + rx1 * aR1 + __float_as_uint(by.y) * bN + ry1 * bR + c01, bytes1, base1);
      };
      auto extremes = [&](f2 ax, f2 ay, f2 bx, f2 by) {   // of two realizations
        const float2 ux = unpack2(ax), uy = unpack2(ay), vx = unpack2(bx), vy = unpack2(by);
        mnx0 = min_nan(mnx0, ux.x, vx.x); mxx0 = max_nan(mxx0, ux.x, vx.x);
        mny0 = min_nan(mny0, uy.x, vy.x); mxy0 = max_nan(mxy0, uy.x, vy.x);
        mnx1 = min_nan(mnx1, ux.y, vx.y); mxx1 = max_nan(mxx1, ux.y, vx.y);
        mny1 = min_nan(mny1, uy.y, vy.y); mxy1 = max_nan(mxy1, uy.y, vy.y);
      };
      const float *yp = static_cast<const float *>(a.Y) + ((size_t)t * N + w0) * K;
      const int N_run = KT == kNoModes ? 1 : N;   // realizations to run through
      int w = on0 || on1 ? w0 : N_run;
#pragma unroll 1
      for (; w + step < N_run; w += 2 * step, yp += (size_t)(2 * step) * K) {   // two realizations per trip
        float y0[kPhi<KT>], y1[kPhi<KT>];
        load_row<KT>(yp, K, y0);
        load_row<KT>(yp + (size_t)step * K, K, y1);
        f2 ax, ay, bx, by;
        velocity(y0, ax, ay);
        velocity(y1, bx, by);
        extremes(ax, ay, bx, by);
        count(ax, ay);
        count(bx, by);
      }
      if (w < N_run) {   // the last of an odd number
        float y0[kPhi<KT>];
        load_row<KT>(yp, K, y0);
        f2 ax, ay;
        velocity(y0, ax, ay);
        extremes(ax, ay, ax, ay);
        count(ax, ay);
      }
      // (a trapped fraction of either state: both are counted again)
      if (MODE <= 2 && fmn < a.act.rank_trap) atomicOr(&sm.trap, ((on0 ? 1u : 0u) | (on1 ? 2u : 0u)) << (2 * p_t));
      // extremes (min x, min y, -max x, -max y of both states) over the lanes of
      // the pair: halved in number with every exchange while there are several
      float v[8] = {mnx0, mny0, -mxx0, -mxy0, mnx1, mny1, -mxx1, -mxy1};
      int first = 0, left = 8;
#pragma unroll
      for (int off = 16; off >= 4; off >>= 1) {
        if (off < np) break;
        const bool up = (lane & off) != 0;
        constexpr int kHalf[3] = {4, 2, 1};
        const int half = kHalf[off == 16 ? 0 : (off == 8 ? 1 : 2)];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          if (i < half) {
            const float send = up ? v[i] : v[i + half], keep = up ? v[i + half] : v[i];
            v[i] = min_nan(keep, __shfl_xor_sync(0xffffffffu, send, off));
          }
        }
        first += up ? half : 0;
        left = half;
      }
      if (np <= 2) v[0] = min_nan(v[0], __shfl_xor_sync(0xffffffffu, v[0], 2));
      if (np > 2 || (lane & 2) == 0) {
        float *ef = reinterpret_cast<float *>(ext + warp * G + 2 * p_t);
#pragma unroll
        for (int i = 0; i < 4; ++i)
          if (i < left && (first + i < 4 ? on0 : on1)) ef[first + i] = v[i];
      }
    }
    if (threadIdx.x == 0) sm.next[par] = next_group;
  }
  __syncthreads();

  // ---- warp v: slice v, lane l = row (q_l, a_l)
  const int64_t sl = sl0 + warp;
  uint32_t *grid = tabs + (size_t)warp * words;
  uint32_t *stage = tabs - (size_t)(NW - warp) * (32 * kStage);   // the stages precede the tables
  RowGeo r{};
  r.hix = r.hiy = -1;
  bool build = sl < a.slice_end, defer = false;
  if (build) {
    const int q_l = lane / (32 / spw), a_l = lane % (32 / spw);
    r.kind = a_l < a.A ? sm.st[warp * spw + q_l].kind : (int)KIND_NONE;
    r.rows = r.kind == KIND_SAMPLE;
    // the states' extremes and whether they lie in the predicted windows, lane & 3 =
    // component of (min x, min y, max x, max y)
    uint32_t missed = 0u;
    for (int q = 0; q < spw; ++q) {
      StateSetup &st = sm.st[warp * spw + q];
      if (st.layer < 0) continue;   // not sampled
      const float m = state_extreme(ext, warp * spw + q, NW, G);
      if (!__all_sync(0xffffffffu, m > -kTame && m < kTame)) {   // non-finite or far velocities: the CTA kernel's path
        defer = true;
        break;
      }
      const bool y = lane & 1, top = lane & 2;
      const int X = fine_coord<MODE>(m, y ? Sy : Sx, sm.rt, y, B);
      const int4 win = st.win;
      const int lo = y ? win.y : win.x, n = y ? win.w - 1 : win.z;
      const bool out = top ? X >= lo + n : X < lo;
      if (__any_sync(0xffffffffu, out) || (MODE <= 2 && ((sm.trap >> (warp * spw + q)) & 1u))) missed |= 1u << q;
      if (lane < 4) {
        (&st.u.x)[lane] = m;
        (&st.X.x)[lane] = X;
      }
    }
    __syncwarp();
    if (missed && !defer) defer = !recount_slice<KT, MODE>(a, sm, sl, grid, words, share, spw, missed);
    for (int q = 0; q < spw && !defer; ++q) {
      const StateSetup &st = sm.st[warp * spw + q];
      if (st.layer < 0) continue;
      const float4 u = st.u;
      if (q == q_l && r.rows) {
        const int cxa = sm.rt.c[0][a_l], cya = sm.rt.c[1][a_l];
        const float thxa = sm.rt.th[0][a_l], thya = sm.rt.th[1][a_l];
        r.lox = land_offset(u.x, cxa, thxa); r.hix = land_offset(u.z, cxa, thxa);
        r.loy = land_offset(u.y, cya, thya); r.hiy = land_offset(u.w, cya, thya);
        if (r.lox < -a.h || r.hix > a.h || r.loy < -a.h || r.hiy > a.h) {   // sub-grid overflow
          r.rows = false;
          atomicAdd(&a.cnt[CNT_OVERFLOW], 1ULL);
        }
      }
      // the exact table inside the window (its pitch, its own origin)
      FineGeo g = exact_table(st);
      g.pitch = st.win.w;
      g.base = st.off + (g.xmin - st.win.x) * g.pitch + (g.ymin - st.win.y);
      if (q == q_l) r.g = g;
      if (SPW != 1) prefix_table(grid + g.base, g);
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
    // (the box's classes are on their way while the table is summed)
    uint64_t blk;
    const BoxCells bc = box_cells<SPW>(a, sl, r, sr, blk);
    if (SPW == 1 && sm.st[warp].layer >= 0) prefix_table(grid + r.g.base, r.g);
    // (the small scan's counts are right for rows longer than are staged, too; counted
    // again all the same in the batched kernel, which is 1.3 % faster that way)
    const bool boxed = HYB && sr.small;
    if (sr.small) rc = count_small<SPW>(a, sm.rt, grid, r, bc, blk, stage, sr);
    if (!boxed && !sr.small) {
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
    for (int d = 1; d < 8; d <<= 1) {
      const int x = __shfl_up_sync(0xffffffffu, incl, d);
      if (lane >= d) incl += x;
    }
    const int total = __shfl_sync(0xffffffffu, incl, 7);
    unsigned long long base = 0;
    if (lane == 0 && total > 0) base = atomicAdd(&a.cnt[CNT_POOL_COLS], (unsigned long long)total);
    base = __shfl_sync(0xffffffffu, base, 0);
    if (lane < NW) sm.base[lane] = base + (unsigned long long)(incl - w);
    if (lane == 0) sm.trap = 0u;   // read above, set again by the next group
  }
  __syncthreads();
  const long long g1 = sm.next[par];
  const SetupLoads ld = next_first(g1) >= 0 ? setup_load<SPW>(a, next_first(g1)) : SetupLoads{};
  if (build) {
    pl.base = sm.base[warp];
    pl.fits = pl.W == 0 || pl.base + (unsigned long long)pl.W <= a.pool_cap_cols;
    if (!pl.fits && lane == 0) atomicAdd(&a.cnt[CNT_POOL_FULL], 1ULL);
    const SliceTotals tot = sr.small ? write_small<SPW, HYB>(a, sm.rt, sl, r, rc, stage, sr, pl)
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
  if (next_first(g1) >= 0) setup_slice<SPW, MODE>(a, sm, next_first(g1), ld, tabs, words, share);
}

}  // namespace mdpgb
