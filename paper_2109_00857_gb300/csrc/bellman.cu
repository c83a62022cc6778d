// bellman.cu -- sparse value iteration (steps a7-a8) and the small helper
// kernels of the build (cell classes, sub-grid offset table, field extremes).
//
// Bellman backup (Sec. II-B): Q(s,a) = R(s,a) + sum_j P_j V(s'_j),
// V_{k+1}(s) = max_a Q(s,a), pi(s) = argmax_a Q(s,a) (lowest index wins ties).
// The slices' entry columns reach shared memory by TMA bulk copies and the
// successors' values V(s') are gathered from the next time layer.  Three
// sweeps with the same results bit for bit: the warp-specialized sweep for
// one state per slice (a producer warp copies rounds of slices into three
// slots, 31 consumer warps each sum one slice, lane l row l, and take the max
// and argmax with one redux.sync key per objective); warp per slice for
// several states per slice (a segmented butterfly over the A_pad lanes of a
// state) and for the smaller layers of backward passes; and the grouped sweep,
// kept for the batch's one-state-per-slice class (four states per warp step,
// each lane summing four rows and keeping a running max, a 3-step shuffle per
// state).  Residual max|V_{k+1} - V_k|
// is reduced on the device; a sweep whose predecessor met the tolerance
// exits at once, so a fixed launch sequence needs no host round trip between
// sweeps.
#include <algorithm>
#include <cmath>
#include <cfloat>

#include "build_common.cuh"

namespace mdpgb {

// ------------------------------------------------------------ prepare ----
__global__ void prepare_kernel(const uint8_t *__restrict__ obstacle, const uint8_t *__restrict__ target,
                               uint8_t *__restrict__ cls, int64_t Nc, int64_t n, int32_t *delta,
                               int L, int nx) {
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += stride) {
    uint8_t c = 0;
    if (obstacle[i]) c |= CLS_OBSTACLE;
    if (target[i % Nc]) c |= CLS_TARGET;
    cls[i] = c;
  }
  if (blockIdx.x == 0) {
    const int h = (L - 1) / 2;
    for (int b = threadIdx.x; b < L * L; b += blockDim.x) delta[b] = (b / L - h) * nx + (b % L - h);
  }
}

cudaError_t launch_prepare(const uint8_t *obstacle, const uint8_t *target, uint8_t *cls, int nx,
                           int ny, int nt, int32_t *delta, int L, cudaStream_t st) {
  const int64_t Nc = (int64_t)nx * ny, n = Nc * nt;
  int64_t blocks = (n + 255) / 256;
  if (blocks > 4096) blocks = 4096;
  if (blocks < 1) blocks = 1;
  prepare_kernel<<<(unsigned)blocks, 256, 0, st>>>(obstacle, target, cls, Nc, n, delta, L, nx);
  return cudaGetLastError();
}

// ------------------------------------------------------ field extremes ----
// out[g*C + c] = max |x| over the elements of group g, component c, for data
// laid out [outer][G][inner][C].  Non-negative floats order like their bits
// (a NaN above all).
// A block takes pieces of one group's runs of inner C elements; a thread's
// elements are a multiple of C apart, so it keeps one maximum in a register and
// memory sees an atomic per block, piece and component where the maximum is
// still to be raised.  (One atomic per element, all on a few addresses, made
// the three launches of 37 layers of 77 x 45 cells and five modes 530 us;
// 17 us so.)
constexpr int kAbsThreads = 256, kAbsLoads = 16;
template <typename T>
__global__ void __launch_bounds__(kAbsThreads) absmax_kernel(const T *__restrict__ x, int64_t runs, int G, int64_t run,
                                                             int64_t pieces, int C, unsigned int *out) {
  __shared__ unsigned int top[kAbsThreads];   // per component (C <= kAbsThreads)
  const int width = kAbsThreads / C * C;      // threads taking part
  const int c = threadIdx.x % C;
  for (int64_t item = blockIdx.x; item < runs * pieces; item += gridDim.x) {
    const int64_t r = item / pieces, begin = item % pieces * ((int64_t)kAbsLoads * width);
    const T *p = x + r * run;
    if (threadIdx.x < C) top[threadIdx.x] = 0u;
    __syncthreads();
    unsigned int m = 0u;
    if (threadIdx.x < width) {
#pragma unroll
      for (int i = 0; i < kAbsLoads; ++i) {
        const int64_t at = begin + (int64_t)i * width + threadIdx.x;
        if (at < run) m = max(m, __float_as_uint(fabsf((float)p[at])));
      }
      if (m > 0u) atomicMax(&top[c], m);
    }
    __syncthreads();
    if (threadIdx.x < C) {
      unsigned int *o = &out[(int)(r % G) * C + threadIdx.x];
      const unsigned int v = top[threadIdx.x];
      if (v > *reinterpret_cast<volatile unsigned int *>(o)) atomicMax(o, v);
    }
    __syncthreads();
  }
}

cudaError_t launch_absmax(const void *x, int precision, int64_t n, int G, int64_t inner, int C,
                          unsigned int *out, cudaStream_t st) {
  if (n < 1) return cudaSuccess;
  if (inner == 1) {   // groups of single elements: components of one group
    C *= G;
    G = 1;
  }
  if (C < 1 || C > kAbsThreads) return cudaErrorInvalidValue;
  if (G == 1) inner = n / C;   // one group: one run
  const int64_t run = inner * C, runs = n / run;
  const int64_t piece = (int64_t)kAbsLoads * (kAbsThreads / C * C), pieces = (run + piece - 1) / piece;
  const unsigned blocks = (unsigned)std::min<int64_t>(runs * pieces, (int64_t)num_sms() * 8);
  if (precision == MDP_FP64_CHECK)
    absmax_kernel<double><<<blocks, kAbsThreads, 0, st>>>(static_cast<const double *>(x), runs, G, run, pieces, C, out);
  else
    absmax_kernel<float><<<blocks, kAbsThreads, 0, st>>>(static_cast<const float *>(x), runs, G, run, pieces, C, out);
  return cudaGetLastError();
}

// ------------------------------------------------------------- backups ----
template <typename RT>
struct Acc;
template <>
struct Acc<float> {
  float v = 0.f;
  __device__ __forceinline__ void add(uint32_t cnt, float V, int) { v = fmaf((float)cnt, V, v); }
  __device__ __forceinline__ float q(float R, float invN) const { return fmaf(v, invN, R); }
};
template <>
struct Acc<double> {
  double v = 0.0;
  // the oracle's order: acc = acc + (count/N) * V(s'), then Q = R + acc
  __device__ __forceinline__ void add(uint32_t cnt, double V, int N) {
    v = __dadd_rn(v, __dmul_rn(__ddiv_rn((double)cnt, (double)N), V));
  }
  __device__ __forceinline__ double q(double R, double) const { return __dadd_rn(R, v); }
};

// ---- mbarrier / bulk-copy helpers (PTX) ----
__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint32_t bar, uint32_t bytes) {
  asm volatile("{\n\t.reg .b64 st;\n\tmbarrier.arrive.expect_tx.shared::cta.b64 st, [%0], %1;\n\t}" ::"r"(bar),
               "r"(bytes)
               : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
  asm volatile("{\n\t.reg .b64 st;\n\tmbarrier.arrive.shared::cta.b64 st, [%0];\n\t}" ::"r"(bar) : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint32_t bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(bar), "r"(parity)
      : "memory");
  return ok != 0;
}
// Bounded wait: gives up after ~2 s of clock cycles so a lost arrival can
// never hang the GPU; the caller reports the timeout through the error word.
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity, long long limit = 4000000000LL) {
  if (mbar_try_wait(bar, parity)) return true;   // usual case: the data is there
  const long long t0 = clock64();
  while (!mbar_try_wait(bar, parity)) {
    if (clock64() - t0 > limit) return false;
  }
  return true;
}
// The same bounded wait, but each test may suspend the warp (up to ~20 us,
// resumed as soon as the phase completes) instead of spinning, so waiting
// warps leave the issue slots to the others.
__device__ __forceinline__ bool mbar_try_wait_suspend(uint32_t bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %3;\n\tselp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(bar), "r"(parity), "r"(20000u)
      : "memory");
  return ok != 0;
}
__device__ __forceinline__ bool mbar_wait_suspend(uint32_t bar, uint32_t parity, long long limit) {
  if (mbar_try_wait(bar, parity)) return true;
  const long long t0 = clock64();
  while (!mbar_try_wait_suspend(bar, parity)) {
    if (clock64() - t0 > limit) return false;
  }
  return true;
}
__device__ __forceinline__ void bulk_g2s(uint32_t dst, const void *src, uint32_t bytes, uint32_t bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst),
               "l"(src), "r"(bytes), "r"(bar)
               : "memory");
}
// The same copy marked for early L2 eviction (policy from l2_evict_first):
// the entry stream is read once per sweep and should not push the value
// tables, which every sweep gathers from, out of L2.
__device__ __forceinline__ void bulk_g2s_stream(uint32_t dst, const void *src, uint32_t bytes, uint32_t bar,
                                                uint64_t policy) {
  asm volatile(
      "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint [%0], [%1], %2, [%3], %4;" ::"r"(
          dst),
      "l"(src), "r"(bytes), "r"(bar), "l"(policy)
      : "memory");
}
__device__ __forceinline__ uint64_t l2_evict_first() {
  uint64_t p;
  asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(p));
  return p;
}

constexpr int kWarps = 8;     // warps per CTA
constexpr int kDepth = 2;     // slices each warp keeps in flight

struct PipeRange {
  int64_t sl_lo, sl_hi;   // slices of this launch
  int64_t s_lo, s_hi;     // states whose V this launch writes
  int stage_bytes;        // bytes per stage
  int zero_second;        // two-chain pass: the second chain's values of this layer are 0
  // two-chain pass: this layer's slots, layer t + 1's (nullptr: there is none) and
  // where their union goes; the largest float <= SolveArgs::tol
  ChainSlot *slots;
  const ChainSlot *next_slots;
  uint32_t *next_above;
  int first;              // layer 0: the slots take the largest differences themselves, too
  float tol;
  SolveStop stop;
  int grouped;            // 1: bellman_body_g (kGS states per warp step, batched sweeps); 2: bellman_kernel_ws
                          // (stage_bytes = entry bytes per slot)
};

// one stage holds a slice's entry columns (at most wcap of them)
static int stage_bytes_for(int wcap) { return wcap * 128; }

// A CTA streams a contiguous block of slices (so its V(s') gathers stay in a
// small window of layer t+1 that L1 keeps); warp w takes slices w, w+8, ...
// and keeps kDepth of them in flight in private stages: lane 0 copies a
// slice's entry columns with cp.async.bulk (TMA) into a stage whose mbarrier
// counts the bytes, while the warp works on an earlier stage: gathers V(s'),
// forms Q, reduces max/argmax over each state's A_pad lanes and writes V and
// the policy.  The slice's R values (one per row and objective) come with
// plain coalesced loads issued one slice ahead; slice offsets and widths of
// the next 32 slices are read in one coalesced load.
// res != nullptr: Jacobi sweep k (exits at once if sweep k-1 met the
// tolerance) with the residual reduced into res[k-1].
// One CTA, slices [b_lo, b_hi) of one model (all threads call it).
// Values of NC components of one state (the objectives of a fused solve; of a
// two-chain pass, the objectives' values and then their second chain's),
// stored side by side and padded to a power of two so that vector loads gather
// V(s') of every component.
template <typename RT, int NC>
struct alignas(sizeof(RT) * (NC <= 2 ? NC : (NC <= 4 ? 4 : 8))) VPack {
  static constexpr int W = NC <= 2 ? NC : (NC <= 4 ? 4 : 8);
  RT v[W];
};

// Per-objective operands of one Bellman launch.  NO objectives share the
// streamed transition slices (each slice is copied once per sweep), each
// with its own R, policy and residual slots; their values live in one
// packed table (in = V_k, out = V_{k+1}; equal for the in-place layered
// pass).  A layered pass has no res (no residual, no early
// exit).
// P == kChains: a two-chain layered pass (launch_two_chains): components NO..2 NO - 1
// are a second chain of values with the same R, whose policy is not kept.
// (What a launch is for is fixed at compile time: chosen at run time, the full
// sweeps took 2 to 3 % longer -- 100 x 100 cells, 60 layers, 32 actions 8.66 ms
// against 8.47.)
enum Pass : int { kSweep = 0, kLayer = 1, kChains = 2 };
template <typename RT, int NO, Pass P = kSweep>
struct VSet {
  static constexpr int NC = P == kChains ? 2 * NO : NO;
  const RT *R[NO];
  const VPack<RT, NC> *in;
  VPack<RT, NC> *out;
  int16_t *pol[NO];
  unsigned long long *res[NO];
};

// The tail of row `lane` of slice sl that the build put in the slice's spill
// block (HYB), added to the row's sums in its stored (ascending) order after
// the ELL columns: the same sum as over one plain row.  Called only for
// models with a spill area (a.spill_off != nullptr).
template <typename RT, int NC>
__device__ __forceinline__ void add_spill(const SolveArgs &a, int64_t sl, int lane, const VPack<RT, NC> *Vn,
                                          Acc<RT> (&acc)[NC]) {
  const uint32_t off = __ldg(a.spill_off + sl);
  if (off == kNoSlice) return;
  const uint32_t *blk = a.spill + off;
  const uint32_t b = __ldg(blk + lane), e = __ldg(blk + lane + 1);
  for (uint32_t i = b; i < e; ++i) {
    const uint32_t w = __ldg(blk + kSpillHdr + i);
    const VPack<RT, NC> g = Vn[(int)(int16_t)(w & 0xFFFFu)];
#pragma unroll
    for (int o = 0; o < NC; ++o) acc[o].add(w >> 16, g.v[o], a.N);
  }
}

// Programmatic dependent launch: a layer's kernel may start while the previous
// layer's finishes -- its prologue and first entry copies touch nothing that
// kernel writes -- and waits here before it reads V.  A sweep waits at once (it
// starts from the previous one's residuals): that hides a launch's latency alone.
// Both return at once in kernels launched without the attribute.
__device__ __forceinline__ void pdl_trigger() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// A CTA whose solve has timed out or proven nothing (its error word is set) gives
// up before it waits on anything.  The word may be set while the CTA starts -- by the layer
// that a dependent launch overlaps, or by another CTA of the same launch -- so
// one thread reads it for all: threads that disagreed would leave the others
// with barriers nobody initialized.  A dependent launch still waits for the
// kernel before it, so that the stream's next work (a copy, a free) starts after
// every layer has ended.  (CTAs without slices may leave without that wait: the
// launch has one with slices, which does not.)  Synchronises the CTA.
__device__ __forceinline__ bool cta_gives_up(const SolveArgs &a) {
  if (!__syncthreads_or(threadIdx.x == 0 && *(volatile int *)a.err != 0)) return false;
  pdl_wait();
  return true;
}

// A two-chain pass ends as soon as it proves nothing for any objective.  Every CTA
// says in a slot of its layer for which objectives it saw differences above tol
// (the CTAs spread over the slots: 608 stores to one address took 6 us a layer,
// more than the layer itself).  The first warp of the next layer's launch unites
// the slots -- the loads are issued with the first gathers and used at the end,
// so no layer waits for them -- and, where there is nothing, tells the layers
// still to start, by the error word, and the host, which stops launching them.
__device__ __forceinline__ uint32_t chains_look(const PipeRange &pr) {   // one warp
  return pr.next_slots ? __ldcg(&pr.next_slots[threadIdx.x & 31].above) : 1u;
}
__device__ __forceinline__ void chains_tell(const SolveArgs &a, const PipeRange &pr, uint32_t above) {
  if (!pr.next_slots) return;
  above = __reduce_or_sync(0xffffffffu, above);
  if ((threadIdx.x & 31) != 0) return;
  *pr.next_above = above;
  if (above != 0u) return;
  atomicOr(a.err, kErrNotProven);
  if (pr.stop.host) *(volatile unsigned int *)pr.stop.host = pr.stop.token;
}
// A sweep that finds nothing left to do: no more need be launched.
__device__ __forceinline__ void tell_host(const PipeRange &pr) {
  if (pr.stop.host && blockIdx.x == 0 && threadIdx.x == 0) *(volatile unsigned int *)pr.stop.host = pr.stop.token;
}
// Publishes the largest differences m[o] of the chains over a CTA's states (wmax:
// shared memory for a value per warp and objective; all threads call it).  In
// floats and their bits: FP64 maxima like the sweeps' would cost 2 us a layer.
// (It takes 0.3 us of a layer of 40,000 slices, 14.9 us before; told by each warp as
// soon as it is seen, 0.9 us.)
template <int NO, int WARPS>
__device__ __forceinline__ void chains_publish(const PipeRange &pr, const float (&m)[NO], double *wmax) {
  unsigned int *top = reinterpret_cast<unsigned int *>(wmax);
  const int tid = threadIdx.x, warp = tid >> 5;
#pragma unroll
  for (int o = 0; o < NO; ++o) {
    const unsigned int x = __reduce_max_sync(0xffffffffu, __float_as_uint(m[o]));
    if ((tid & 31) == 0 && warp < WARPS) top[warp * NO + o] = x;
  }
  __syncthreads();
  if (warp == 0) {
    unsigned int x = 0u;   // lane o: objective o's
#pragma unroll
    for (int o = 0; o < NO; ++o) {
      const unsigned int y = __reduce_max_sync(0xffffffffu, tid < WARPS ? top[tid * NO + o] : 0u);
      if (tid == o) x = y;
    }
    ChainSlot *slot = pr.slots + (blockIdx.x % kChainSlots);
    const unsigned int above = __ballot_sync(0xffffffffu, __uint_as_float(x) > pr.tol);
    if (tid == 0 && above) atomicOr(&slot->above, above);
    if (pr.first && tid < NO) atomicMax(&slot->first[tid], x);
  }
}

template <typename RT, int NO, Pass P = kSweep>
__device__ __forceinline__ void bellman_body(const SolveArgs &a, const VSet<RT, NO, P> &v, int k, int64_t b_lo,
                                             int64_t b_hi, const PipeRange &pr, unsigned char *sm,
                                             double *wmax, int *wst_s) {
  using Pk = VPack<RT, VSet<RT, NO, P>::NC>;
  constexpr int NC = VSet<RT, NO, P>::NC;
  constexpr bool layered = P != kSweep;
  if (layered) pdl_trigger();
  // objectives whose previous sweep met the tolerance are finished
  unsigned live = (1u << NO) - 1u;
  if (!layered && k > 1) {
#pragma unroll
    for (int o = 0; o < NO; ++o)
      if (__longlong_as_double((long long)v.res[o][k - 2]) <= a.tol) live &= ~(1u << o);
  }
  if (!live) {
    tell_host(pr);
    return;
  }
  uint64_t *full = reinterpret_cast<uint64_t *>(sm);   // [kWarps][kDepth]
  unsigned char *ring = sm + 256;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int64_t n_local = b_hi - b_lo;
  if (n_local <= 0) return;

  if (tid < kWarps * kDepth) mbar_init(smem_u32(full + tid), 1);
  if (tid == 0) asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  if (cta_gives_up(a)) return;
  if (a.work && k >= 1 && blockIdx.x == 0 && tid == 0) a.work[k - 1] = (unsigned long long)(pr.sl_hi - pr.sl_lo);
  unsigned char *myring = ring + (size_t)warp * kDepth * pr.stage_bytes;

  // 32-bit slice/state indices (the host guarantees |S| + Nc < 2^31)
  const int n_mine = (n_local > warp) ? (int)((n_local - warp + kWarps - 1) / kWarps) : 0;
  const int sl0 = (int)b_lo + warp;                       // my j-th slice: sl0 + j*kWarps
  const uint32_t ring0 = smem_u32(myring), bar0 = smem_u32(full + warp * kDepth);
  uint32_t m_off = 0, m_w = 0;   // lane l: metadata of my slice 32*(j/32) + l
  const uint64_t stream_policy = l2_evict_first();
  const long long wait_limit = a.wait_cycles > 0 ? a.wait_cycles : 4000000000LL;   // ~2 s

  // issue(j, st): copy my j-th slice into stage st = j % kDepth (whole warp calls it)
  auto issue = [&](int j, int st) {
    if ((j & 31) == 0) {
      const int jj = j + lane;
      if (jj < n_mine) {
        const int sl = sl0 + jj * kWarps;
        m_off = __ldg(a.slice_off + sl);
        m_w = __ldg(a.slice_w + sl);
      }
    }
    const uint32_t off = __shfl_sync(0xffffffffu, m_off, j & 31);
    const uint32_t W = __shfl_sync(0xffffffffu, m_w, j & 31);
    if (lane == 0) {
      wst_s[warp * kDepth + st] = (int)W;
      const uint32_t sbase = ring0 + (uint32_t)(st * pr.stage_bytes);
      const uint32_t fb = bar0 + 8u * (uint32_t)st;
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");   // earlier reads of the stage
      // (a.test_extra_tx: bytes that never arrive, on CTA 0's first slice -- failure
      // injection for tests)
      mbar_expect_tx(fb, W * 128u + (j == 0 && warp == 0 && blockIdx.x == 0 ? a.test_extra_tx : 0u));
      if (W) bulk_g2s_stream(sbase, a.pool + (size_t)off * 32, W * 128u, fb, stream_policy);
    }
    __syncwarp();
  };
  // R of my j-th slice, lane = row: one coalesced 128-byte load per objective,
  // issued one slice ahead of its use
  auto load_r = [&](int j, RT (&Rr)[NO]) {
    const size_t sl = (size_t)(sl0 + j * kWarps);
#pragma unroll
    for (int o = 0; o < NO; ++o) Rr[o] = __ldcs(v.R[o] + sl * 32 + lane);   // streamed: read once
  };

  const int q = lane / a.A_pad, act = lane % a.A_pad;
  const int nS = (int)a.nS, Nc = (int)a.Nc;
  const int s_lo = (int)pr.s_lo, s_hi = (int)pr.s_hi;
  const RT invN = (RT)1 / (RT)a.N;
  float rf[NO];      // FP32 residuals
  double r[NO];      // FP64 residuals
#pragma unroll
  for (int o = 0; o < NO; ++o) {
    rf[o] = 0.f;
    r[o] = 0.0;
  }
  for (int j = 0; j < kDepth && j < n_mine; ++j) issue(j, j);
  RT Rn[NO];   // R of the next slice
#pragma unroll
  for (int o = 0; o < NO; ++o) Rn[o] = (RT)0;
  if (n_mine > 0) load_r(0, Rn);
  if (layered) pdl_wait();   // from here on V of the next layer is read
  uint32_t next_above = 0u;
  if (P == kChains && blockIdx.x == 0 && warp == 0) next_above = chains_look(pr);
  int st = 0;
  uint32_t phase = 0;
  int s = sl0 * a.spw + q;                      // state of this lane's row in my j-th slice
  const int s_step = kWarps * a.spw;
  // active-layer Jacobi: layer t_cur of my state s (s < t_end = (t_cur+1) Nc)
  // and whether any of its values changed in this sweep
  uint8_t *chg_out = a.lflags ? a.lflags + (size_t)(k % 3) * (a.nt + 1) : nullptr;
  int t_cur = s / Nc, t_end = (t_cur + 1) * Nc;
  bool chg = false;
  for (int j = 0; j < n_mine; ++j, s += s_step) {
    if (!mbar_wait(bar0 + 8u * (uint32_t)st, phase, wait_limit)) {
      if (lane == 0) atomicOr(a.err, kErrTimeout);
      // drain: wait (bounded) for the copies still in flight into my stages
      for (int jj = j + 1; jj < j + kDepth && jj < n_mine; ++jj)
        mbar_wait(bar0 + 8u * (uint32_t)(jj % kDepth), (uint32_t)(jj / kDepth) & 1, wait_limit);
      break;
    }
    const unsigned char *sb = myring + st * pr.stage_bytes;
    const uint32_t *ent = reinterpret_cast<const uint32_t *>(sb) + lane;
    const bool valid = s >= s_lo && s < s_hi && act < a.A;
    RT Rv[NO];
#pragma unroll
    for (int o = 0; o < NO; ++o) Rv[o] = Rn[o];
    if (j + 1 < n_mine) load_r(j + 1, Rn);
    const int W = wst_s[warp * kDepth + st];
    Acc<RT> acc[NC];
    // successor layer base of this state; rows without successors (last
    // layer, padding lanes) hold only padding words and read V[|S|] = 0
    const int sn = (s + Nc <= nS) ? s + Nc : nS;
    const Pk *Vn = v.in + sn;
#pragma unroll 4
    for (int kk = 0; kk < W; ++kk) {   // every column of the slice, ascending
      const uint32_t w = ent[kk * 32];
      const Pk g = Vn[(int)(int16_t)(w & 0xFFFFu)];
#pragma unroll
      for (int o = 0; o < NC; ++o) acc[o].add(w >> 16, g.v[o], a.N);
    }
    if (a.spill_off) add_spill<RT, NC>(a, sl0 + (int64_t)j * kWarps, lane, Vn, acc);
    __syncwarp();
    if (j + kDepth < n_mine) issue(j + kDepth, st);   // refill the stage just read
    if (++st == kDepth) {
      st = 0;
      phase ^= 1u;
    }
    const bool head = act == 0 && s >= s_lo && s < s_hi;   // the lane that writes state s
    const bool term = head && __ldg(a.cls + s) != CLS_FREE;
    Pk old{}, nv;
    if (head && !layered) old = v.in[s];
#pragma unroll
    for (int o = 0; o < NC; ++o) {
      RT qv = valid ? acc[o].q(Rv[o % NO], invN) : -(RT)INFINITY;
      int qa = act;
      if (sizeof(RT) == 4 && a.A_pad == 32) {
        // one state per warp: order-preserving integer key, warp max in one
        // redux, lowest lane (= lowest action) among the maxima by ballot
        const uint32_t bits = __float_as_uint((float)qv + 0.0f);   // -0 keys like +0
        const uint32_t key = (bits & 0x80000000u) ? ~bits : (bits | 0x80000000u);
        const uint32_t kmax = __reduce_max_sync(0xffffffffu, key);
        qa = __ffs(__ballot_sync(0xffffffffu, key == kmax)) - 1;
        qv = __shfl_sync(0xffffffffu, qv, qa);
      } else {
        for (int m = 1; m < a.A_pad; m <<= 1) {
          const RT oq = __shfl_xor_sync(0xffffffffu, qv, m);
          const int oa = __shfl_xor_sync(0xffffffffu, qa, m);
          if (oq > qv || (oq == qv && oa < qa)) {
            qv = oq;
            qa = oa;
          }
        }
      }
      if (o >= NO) {   // second chain: the value alone
        nv.v[o] = pr.zero_second ? (RT)0 : qv;
        continue;
      }
      // a finished objective carries its value forward unchanged
      const bool upd = (live >> o) & 1u;
      nv.v[o] = upd ? qv : old.v[o];
      if (head && upd) {
        v.pol[o % NO][s] = term ? (int16_t)-1 : (int16_t)qa;
        if constexpr (layered) continue;
        else if constexpr (sizeof(RT) == 4) rf[o % NO] = fmaxf(rf[o % NO], fabsf(qv - old.v[o]));
        else r[o % NO] = fmax(r[o % NO], fabs(qv - old.v[o]));
      }
    }
#pragma unroll
    for (int o = NC; o < Pk::W; ++o) nv.v[o] = (RT)0;
    if (head) {
      v.out[s] = nv;
      if constexpr (P == kChains) {
#pragma unroll
        for (int o = 0; o < NO; ++o) rf[o] = fmaxf(rf[o], fabsf(nv.v[o] - nv.v[NO + o]));
      }
      if (!layered && chg_out) {
        if (s >= t_end) {   // entered a later layer: publish the finished one
          if (chg) chg_out[t_cur] = 1;
          chg = false;
          do { ++t_cur; t_end += Nc; } while (s >= t_end);
        }
#pragma unroll
        for (int o = 0; o < NO; ++o) {   // bitwise: -0 vs +0 counts as a change
          if constexpr (sizeof(RT) == 4) chg |= __float_as_uint(nv.v[o]) != __float_as_uint(old.v[o]);
          else chg |= __double_as_longlong(nv.v[o]) != __double_as_longlong(old.v[o]);
        }
      }
    }
  }
  if (chg_out && chg) chg_out[t_cur] = 1;
  if constexpr (P == kChains) {
    if (blockIdx.x == 0 && warp == 0) chains_tell(a, pr, next_above);
    chains_publish<NO, kWarps>(pr, rf, wmax);
  }
  if (!layered) {
#pragma unroll
    for (int o = 0; o < NO; ++o) {
      double ro = (sizeof(RT) == 4) ? (double)rf[o] : r[o];
      for (int m = 16; m > 0; m >>= 1) ro = fmax(ro, __shfl_xor_sync(0xffffffffu, ro, m));
      if (lane == 0) wmax[warp * NO + o] = ro;
    }
    __syncthreads();
#pragma unroll
    for (int o = 0; o < NO; ++o) {   // thread o publishes objective o (no dynamic index into v)
      if (tid == o) {
        double m = 0.0;
        for (int i = 0; i < kWarps; ++i) m = fmax(m, wmax[i * NO + o]);
        if (m > 0.0) atomicMax(&v.res[o][k - 1], (unsigned long long)__double_as_longlong(m));
      }
    }
  }
}

// Active-layer Jacobi sweep k: layer t needs recomputing if its own values
// or those of layer t+1 changed in sweep k-1 (otherwise V_{k+1} = V_k on it
// and the output table already holds that value from sweep k-1).  Sets
// [sl_lo, sl_hi) to the slices of the first through the last such layer
// (layers in between are recomputed, which yields their unchanged values).
// The leader CTA (one per model) clears the flags that sweep k+1 will set.
// Returns false when no layer changed: V_{k+1} = V_k, the residual stays 0.
// All threads of the CTA call it.
__device__ __forceinline__ bool active_range(const SolveArgs &a, int k, PipeRange &pr, bool leader) {
  const int nt = a.nt;
  const uint8_t *prev = a.lflags + (size_t)((k - 1) % 3) * (nt + 1);
  if (leader) {
    uint8_t *clr = a.lflags + (size_t)((k + 1) % 3) * (nt + 1);
    for (int t = threadIdx.x; t <= nt; t += blockDim.x) clr[t] = 0;
  }
  __shared__ int s_tlo, s_thi;
  if (threadIdx.x == 0) {
    s_tlo = nt;
    s_thi = -1;
  }
  __syncthreads();
  for (int t = threadIdx.x; t < nt; t += blockDim.x) {
    if (prev[t] | prev[t + 1]) {
      atomicMin(&s_tlo, t);
      atomicMax(&s_thi, t);
    }
  }
  __syncthreads();
  const int tlo = s_tlo, thi = s_thi;
  if (thi < 0) return false;
  pr.sl_lo = (int64_t)tlo * a.Nc / a.spw;
  pr.sl_hi = min(a.n_slices, ((int64_t)(thi + 1) * a.Nc + a.spw - 1) / a.spw);
  return true;
}

template <typename RT, int NO, Pass P>
__global__ void __launch_bounds__(32 * kWarps, P == kChains && NO == 3 ? 3 : 4) bellman_kernel(SolveArgs a, VSet<RT, NO, P> v,
                                                                                   int k, PipeRange pr) {
  extern __shared__ __align__(128) unsigned char sm[];
  __shared__ double wmax[kWarps * NO];
  __shared__ int wst_s[kWarps * kDepth];   // columns of the slice in each stage
  if (P == kSweep) {
    pdl_trigger();
    pdl_wait();
    if (a.lflags && !active_range(a, k, pr, blockIdx.x == 0)) {
      tell_host(pr);
      return;
    }
  }
  const int64_t total = pr.sl_hi - pr.sl_lo;
  const int64_t per_cta = (total + gridDim.x - 1) / gridDim.x;
  const int64_t b_lo = pr.sl_lo + (int64_t)blockIdx.x * per_cta;
  const int64_t b_hi = min(pr.sl_hi, b_lo + per_cta);
  bellman_body<RT, NO, P>(a, v, k, b_lo, b_hi, pr, sm, wmax, wst_s);
}

// ---- grouped sweep: kGS states per warp step (models with A_pad = 32) ----
// One slice per state (A_pad = 32) makes the per-slice epilogue of
// bellman_body (a max/argmax over 32 lanes per objective, the stage refill,
// the writes) cost as much as the slice's backups.  Here a warp takes kGS
// consecutive slices at a time: lane (q, g) owns state q of the group and the
// actions g, g + kGL, g + 2 kGL, ... (ascending), forms their Q values one
// after another in registers and keeps the running maximum (strict >, so the
// lowest action wins ties); a log2(kGL)-step shuffle reduction over the kGL
// lanes of each state finishes the max/argmax.  Each row is still summed by
// one lane in ascending column order, so values and policy equal
// bellman_body's bit for bit.  The kGS slices of a group are copied into
// fixed slots of one stage (slot = wcap columns + 32 bytes: the 8-bank skew
// between slots keeps the lanes' shared-memory reads conflict-free).
constexpr int kGS = 4;           // states (slices) per group
constexpr int kGL = 32 / kGS;    // lanes per state
constexpr int kWarpsG = 16;      // warps per CTA: one CTA per SM (one V(s') window per L1)

static int slot_bytes_g(int wcap) { return wcap * 128 + 32; }
static size_t grouped_smem(int wcap) { return 256 + (size_t)kWarpsG * kDepth * kGS * slot_bytes_g(wcap); }
// dynamic shared memory the grouped kernel may take: the opt-in maximum per
// CTA (227 KB) less its static arrays and a margin
constexpr size_t kGroupedSmemMax = 227 * 1024 - 2048;

template <typename RT, int NO>
__device__ __forceinline__ void bellman_body_g(const SolveArgs &a, const VSet<RT, NO> &v, int k, int64_t b_lo,
                                               int64_t b_hi, const PipeRange &pr, unsigned char *sm,
                                               double *wmax, int *wst_s) {
  unsigned live = (1u << NO) - 1u;
  if (k > 1) {
#pragma unroll
    for (int o = 0; o < NO; ++o)
      if (v.res[o] && __longlong_as_double((long long)v.res[o][k - 2]) <= a.tol) live &= ~(1u << o);
  }
  if (!live) return;
  uint64_t *full = reinterpret_cast<uint64_t *>(sm);   // [kWarpsG][kDepth]
  unsigned char *ring = sm + 256;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int64_t n_local = b_hi - b_lo;
  if (n_local <= 0) return;

  if (tid < kWarpsG * kDepth) mbar_init(smem_u32(full + tid), 1);
  if (tid == 0) asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  if (cta_gives_up(a)) return;
  if (a.work && k >= 1 && blockIdx.x == 0 && tid == 0) a.work[k - 1] = (unsigned long long)(pr.sl_hi - pr.sl_lo);
  const int slot = pr.stage_bytes / kGS;
  unsigned char *myring = ring + (size_t)warp * kDepth * pr.stage_bytes;
  const int n_groups = (int)((n_local + kGS - 1) / kGS);
  const int n_mine = (n_groups > warp) ? (n_groups - warp + kWarpsG - 1) / kWarpsG : 0;
  const int first0 = (int)b_lo + warp * kGS;      // first slice of my j-th group: first0 + j*gstep
  const int gstep = kWarpsG * kGS;
  const int hi = (int)b_hi;
  const uint32_t ring0 = smem_u32(myring), bar0 = smem_u32(full + warp * kDepth);
  const uint64_t stream_policy = l2_evict_first();
  const int q = lane / kGL, g = lane % kGL;

  // lane l: metadata of slice l % kGS of my group 32/kGS * (j / (32/kGS)) + l / kGS
  constexpr int kMetaG = 32 / kGS;
  uint32_t m_off = 0, m_w = 0;
  // issue(j, st): lanes 0..kGS-1 copy the slices of my j-th group into their
  // slots of stage st (whole warp calls it)
  auto issue = [&](int j, int st) {
    if (j % kMetaG == 0) {   // one coalesced load for the next kMetaG groups
      const int sl = first0 + (j + lane / kGS) * gstep + lane % kGS;
      m_off = 0;
      m_w = 0;
      if (sl < hi) {
        m_off = __ldg(a.slice_off + sl);
        m_w = __ldg(a.slice_w + sl);
      }
    }
    const int src = (j % kMetaG) * kGS + (lane % kGS);
    const uint32_t off = __shfl_sync(0xffffffffu, m_off, src);
    uint32_t W = __shfl_sync(0xffffffffu, m_w, src);
    if (lane >= kGS) W = 0;
    uint32_t tot = W;
#pragma unroll
    for (int m = 1; m < kGS; m <<= 1) tot += __shfl_xor_sync(0xffffffffu, tot, m);
    const uint32_t fb = bar0 + 8u * (uint32_t)st;
    if (lane < kGS) wst_s[(warp * kDepth + st) * kGS + lane] = (int)W;
    if (lane == 0) {
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");   // earlier reads of the stage
      mbar_expect_tx(fb, tot * 128u);
    }
    __syncwarp();
    if (lane < kGS && W) {
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      bulk_g2s_stream(ring0 + (uint32_t)(st * pr.stage_bytes + lane * slot), a.pool + (size_t)off * 32, W * 128u,
                      fb, stream_policy);
    }
    __syncwarp();
  };
  // R of my j-th group (lane (q, g): rows g + i*kGL of slice q) and, on the
  // head lanes, the state's current values and class: loaded one group ahead
  auto load_r = [&](int j, RT (&Rr)[kGS][NO], VPack<RT, NO> &old, uint8_t &cls) {
    const int sl = first0 + j * gstep + q;
    if (sl < hi) {
#pragma unroll
      for (int i = 0; i < kGS; ++i)
#pragma unroll
        for (int o = 0; o < NO; ++o) Rr[i][o] = __ldcs(v.R[o] + (size_t)sl * 32 + i * kGL + g);
      if (g == 0) {
        old = v.in[sl];
        cls = __ldg(a.cls + sl);
      }
    }
  };

  const int nS = (int)a.nS, Nc = (int)a.Nc;
  const int s_lo = (int)pr.s_lo, s_hi = (int)pr.s_hi;
  const RT invN = (RT)1 / (RT)a.N;
  float rf[NO];
  double r[NO];
#pragma unroll
  for (int o = 0; o < NO; ++o) {
    rf[o] = 0.f;
    r[o] = 0.0;
  }
  for (int j = 0; j < kDepth && j < n_mine; ++j) issue(j, j);
  RT Rn[kGS][NO];
#pragma unroll
  for (int i = 0; i < kGS; ++i)
#pragma unroll
    for (int o = 0; o < NO; ++o) Rn[i][o] = (RT)0;
  VPack<RT, NO> old_n{};
  uint8_t cls_n = 0;
  if (n_mine > 0) load_r(0, Rn, old_n, cls_n);
  int st = 0;
  uint32_t phase = 0;
  int s = first0 + q;   // spw = 1: state = slice
  uint8_t *chg_out = a.lflags ? a.lflags + (size_t)(k % 3) * (a.nt + 1) : nullptr;
  int t_cur = s / Nc, t_end = (t_cur + 1) * Nc;
  bool chg = false;
  for (int j = 0; j < n_mine; ++j, s += gstep) {
    if (!mbar_wait(bar0 + 8u * (uint32_t)st, phase)) {
      if (lane == 0) atomicOr(a.err, kErrTimeout);
      for (int jj = j + 1; jj < j + kDepth && jj < n_mine; ++jj)
        mbar_wait(bar0 + 8u * (uint32_t)(jj % kDepth), (uint32_t)(jj / kDepth) & 1);
      break;
    }
    const uint32_t *ent = reinterpret_cast<const uint32_t *>(myring + st * pr.stage_bytes + q * slot) + g;
    const int Wq = wst_s[(warp * kDepth + st) * kGS + q];
    RT Rv[kGS][NO];
#pragma unroll
    for (int i = 0; i < kGS; ++i)
#pragma unroll
      for (int o = 0; o < NO; ++o) Rv[i][o] = Rn[i][o];
    const VPack<RT, NO> old = old_n;
    const uint8_t cls_s = cls_n;
    if (j + 1 < n_mine) load_r(j + 1, Rn, old_n, cls_n);
    const bool in_rng = s < hi && s >= s_lo && s < s_hi;
    const int sn = (s + Nc <= nS) ? s + Nc : nS;
    const VPack<RT, NO> *Vn = v.in + sn;
    Acc<RT> acc[kGS][NO];
#pragma unroll(NO == 1 ? 4 : 1)
    for (int kk = 0; kk < Wq; ++kk) {   // every column of the slice, ascending
#pragma unroll
      for (int i = 0; i < kGS; ++i) {
        const uint32_t w = ent[kk * 32 + i * kGL];
        const VPack<RT, NO> gv = Vn[(int)(int16_t)(w & 0xFFFFu)];
#pragma unroll
        for (int o = 0; o < NO; ++o) acc[i][o].add(w >> 16, gv.v[o], a.N);
      }
    }
    __syncwarp();
    if (j + kDepth < n_mine) issue(j + kDepth, st);   // refill the stage just read
    if (++st == kDepth) {
      st = 0;
      phase ^= 1u;
    }
    // running max over my actions (ascending, strict >: the lowest wins ties)
    RT qv[NO];
    int qa[NO];
    // (states outside the range are not written, so only padding actions
    // need masking)
    const bool full_a = a.A == 32;
#pragma unroll
    for (int i = 0; i < kGS; ++i) {
      const int act = i * kGL + g;
      const bool valid = full_a || act < a.A;
#pragma unroll
      for (int o = 0; o < NO; ++o) {
        const RT x = valid ? acc[i][o].q(Rv[i][o], invN) : -(RT)INFINITY;
        if (i == 0 || x > qv[o]) {
          qv[o] = x;
          qa[o] = act;
        }
      }
    }
#pragma unroll
    for (int o = 0; o < NO; ++o) {
#pragma unroll
      for (int m = 1; m < kGL; m <<= 1) {
        const RT oq = __shfl_xor_sync(0xffffffffu, qv[o], m);
        const int oa = __shfl_xor_sync(0xffffffffu, qa[o], m);
        if (oq > qv[o] || (oq == qv[o] && oa < qa[o])) {
          qv[o] = oq;
          qa[o] = oa;
        }
      }
    }
    const bool head = g == 0 && in_rng;   // the lane that writes state s
    const bool term = head && cls_s != CLS_FREE;
    VPack<RT, NO> nv;
#pragma unroll
    for (int o = 0; o < NO; ++o) {
      const bool upd = (live >> o) & 1u;
      nv.v[o] = upd ? qv[o] : old.v[o];
      if (head && upd) {
        v.pol[o][s] = term ? (int16_t)-1 : (int16_t)qa[o];
        if constexpr (sizeof(RT) == 4) rf[o] = fmaxf(rf[o], fabsf(qv[o] - old.v[o]));
        else r[o] = fmax(r[o], fabs(qv[o] - old.v[o]));
      }
    }
#pragma unroll
    for (int o = NO; o < VPack<RT, NO>::W; ++o) nv.v[o] = (RT)0;
    if (head) {
      v.out[s] = nv;
      if (chg_out) {
        if (s >= t_end) {
          if (chg) chg_out[t_cur] = 1;
          chg = false;
          do { ++t_cur; t_end += Nc; } while (s >= t_end);
        }
#pragma unroll
        for (int o = 0; o < NO; ++o) {
          if constexpr (sizeof(RT) == 4) chg |= __float_as_uint(nv.v[o]) != __float_as_uint(old.v[o]);
          else chg |= __double_as_longlong(nv.v[o]) != __double_as_longlong(old.v[o]);
        }
      }
    }
  }
  if (chg_out && chg) chg_out[t_cur] = 1;
  if (v.res[0]) {
#pragma unroll
    for (int o = 0; o < NO; ++o) {
      double ro = (sizeof(RT) == 4) ? (double)rf[o] : r[o];
      for (int m = 16; m > 0; m >>= 1) ro = fmax(ro, __shfl_xor_sync(0xffffffffu, ro, m));
      if (lane == 0) wmax[warp * NO + o] = ro;
    }
    __syncthreads();
#pragma unroll
    for (int o = 0; o < NO; ++o) {
      if (tid == o) {
        double m = 0.0;
        for (int i = 0; i < kWarpsG; ++i) m = fmax(m, wmax[i * NO + o]);
        if (m > 0.0) atomicMax(&v.res[o][k - 1], (unsigned long long)__double_as_longlong(m));
      }
    }
  }
}

// ---- warp-specialized sweep: a producer warp stages rounds of slices ----
// Models with one state per slice (A_pad = 32).  Each CTA has kWsCons
// consumer warps and one producer warp, and walks its block of consecutive
// slices in rounds: a round holds up to kWsCons consecutive slices (as many as
// fit a slot's entry capacity) and consumer warp w takes slice w of every
// round, so the CTA's warps gather V(s') from one small window of layer t+1
// that L1 keeps.  The producer copies a round into one of kWsSlots
// shared-memory slots with TMA bulk copies -- the slices' entry columns (one
// copy when the pool is in slice order, else one per slice), then for every
// objective the round's R values in one copy (consecutive slices have
// consecutive R rows) -- completing on the slot's full barrier, and writes
// each slice's columns, cell class and current values (loaded one round
// ahead) into the slot's table; the consumers arrive on the slot's empty
// barrier once they have read it, and the producer refills it.  Slots are
// sized by the bytes the slices really have, not by the widest slice.  Lane l
// of a consumer sums row l (action l) in ascending column order, so every Q is
// the same float as in the other kernels, and the max over the 32 actions is
// one redux.sync on an order-preserving key with the lowest winning action by
// ballot (FP64: a butterfly): values and policy equal theirs bit for bit.
constexpr int kWsCons = 31;     // consumer warps per CTA (+ 1 producer = 1024 threads)
constexpr int kWsSlots = 3;     // round slots
// slices per consumer warp and round (warp w takes slices w, w + 31, ...;
// its slices' column loops run interleaved).  Measured on the large
// workload: 1 (rounds of 31 slices in three slots) 99.5 ms per solve, 2
// (rounds of 62 in two slots) 108-117 ms.
constexpr int kWsPer = 1;
constexpr int kWsRound = kWsCons * kWsPer;   // most slices in a round
constexpr int kWsTab = 32 * kWsPer;          // table entries per slot

struct WsHdr {
  uint64_t full[kWsSlots];      // producer arrival + the round's copied bytes
  uint64_t empty[kWsSlots];     // one arrival per consumer warp
  int2 round[kWsSlots];         // (first slice, slices in the round); 0 slices ends the block
  int2 slice[kWsSlots][kWsTab]; // (entry byte offset in the slot, W | cell class << 8) per slice
};
__host__ __device__ constexpr size_t ws_hdr_bytes() { return (sizeof(WsHdr) + 127) & ~(size_t)127; }
// the slices' current values, [kWsSlots][kWsTab]
template <typename RT, int NO>
__host__ __device__ constexpr size_t ws_old_bytes() { return (kWsSlots * kWsTab * sizeof(VPack<RT, NO>) + 127) & ~(size_t)127; }
template <typename RT>
__host__ __device__ constexpr int ws_r_bytes(int n_obj) { return n_obj * kWsTab * 32 * (int)sizeof(RT); }

// Work of the slices [lo, x) of a slice-ordered pool, in entry columns: their
// columns plus kWsSliceWork per slice (a slice's own cost -- its R rows, its
// state's values, the max over the actions -- weighed in columns).
constexpr int64_t kWsSliceWork = 24;

// CTA b of G takes the slices [ws_cut(b), ws_cut(b + 1)) of [lo, hi): the cut
// is the first x whose work from lo reaches b/G of the whole, so every CTA
// gets the same work however the widths vary (a pool in slice order has
// slice_off = the prefix sums of the widths: the work is monotone in x).  A
// 32-ary search over slice_off, about five dependent loads.  One warp calls it
// with its lanes converged; every lane returns the cut.
__device__ int64_t ws_cut(const SolveArgs &a, int64_t lo, int64_t hi, int64_t b, int64_t G) {
  if (b <= 0) return lo;
  if (b >= G) return hi;
  const int lane = threadIdx.x & 31;
  const uint32_t c0 = __ldg(a.slice_off + lo);
  const int64_t c_end = (int64_t)__ldg(a.slice_off + hi - 1) + (int64_t)__ldg(a.slice_w + hi - 1);
  const int64_t total = (c_end - (int64_t)c0) + kWsSliceWork * (hi - lo);
  const int64_t tgt = total * b / G;   // < total: the cut lies in (lo, hi) or is hi
  if (tgt <= 0) return lo;
  // invariant: work(l) < tgt <= work(h)
  int64_t l = lo, h = hi;
  while (h - l > 1) {
    const int64_t step = (h - l + 31) / 32;   // probes l + step, l + 2 step, ... below h
    const int64_t x = l + (int64_t)(lane + 1) * step;
    bool below = false;
    if (x < h) below = (int64_t)(__ldg(a.slice_off + x) - c0) + kWsSliceWork * (x - lo) < tgt;
    const int c = __popc(__ballot_sync(0xffffffffu, below));   // a prefix of the lanes
    const int64_t nh = min(h, l + (int64_t)(c + 1) * step);
    l += (int64_t)c * step;
    h = nh;
  }
  return h;
}

template <typename RT, int NO, Pass P>
__device__ __forceinline__ void bellman_body_ws(const SolveArgs &a, const VSet<RT, NO, P> &v, int k,
                                                const PipeRange &pr, unsigned char *sm, double *wmax, int *s_flag,
                                                int64_t *s_cut) {
  constexpr int NC = VSet<RT, NO, P>::NC;
  using Pk = VPack<RT, NC>;
  // (A layer's kernel asks at run time: with the sweeps' code left out at compile
  // time, a layer of 40,000 slices took 16.3 us instead of 13.5, three objectives
  // 17.1 or 29.5 instead of 17.5 from one version of the code to the next.)
  const bool layered = P != kSweep && v.res[0] == nullptr;
  if (layered) pdl_trigger();
  unsigned live = (1u << NO) - 1u;
  if (!layered && k > 1) {
#pragma unroll
    for (int o = 0; o < NO; ++o)
      if (__longlong_as_double((long long)v.res[o][k - 2]) <= a.tol) live &= ~(1u << o);
  }
  if (!live) {
    tell_host(pr);
    return;
  }
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  // one read of the error word for the whole CTA (an earlier launch timed out)
  if (tid == 0) *s_flag = *(volatile int *)a.err;
  // this CTA's slices: equal work (slice-ordered pool) or equal counts
  if (warp < 2) {
    int64_t x;
    if (a.pool_ordered && pr.sl_hi > pr.sl_lo) {
      x = ws_cut(a, pr.sl_lo, pr.sl_hi, (int64_t)blockIdx.x + warp, gridDim.x);
    } else {
      const int64_t per_cta = (pr.sl_hi - pr.sl_lo + gridDim.x - 1) / gridDim.x;
      x = min(pr.sl_hi, pr.sl_lo + ((int64_t)blockIdx.x + warp) * per_cta);
    }
    if (lane == 0) s_cut[warp] = x;
  }
  __syncthreads();
  if (*s_flag) {   // (see cta_gives_up)
    if (layered) pdl_wait();
    return;
  }
  if (a.work && k >= 1 && blockIdx.x == 0 && tid == 0) a.work[k - 1] = (unsigned long long)(pr.sl_hi - pr.sl_lo);
  const int64_t b_lo = s_cut[0], b_hi = s_cut[1];
  if (b_hi <= b_lo) return;

  WsHdr *hdr = reinterpret_cast<WsHdr *>(sm);
  Pk *olds = reinterpret_cast<Pk *>(sm + ws_hdr_bytes());   // [kWsSlots][32]
  constexpr int kRB = 32 * (int)sizeof(RT);                // one objective's R values of a slice
  constexpr int kRBytes = ws_r_bytes<RT>(NO);
  const int ecap = pr.stage_bytes;                         // entry bytes per slot
  const int slot_bytes = kRBytes + ecap;
  unsigned char *slots = sm + ws_hdr_bytes() + ws_old_bytes<RT, NC>();
  if (tid < kWsSlots) {
    mbar_init(smem_u32(&hdr->full[tid]), 1);
    mbar_init(smem_u32(&hdr->empty[tid]), kWsCons);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncthreads();
  const uint32_t full0 = smem_u32(&hdr->full[0]), empty0 = smem_u32(&hdr->empty[0]);
  const long long wait_limit = a.wait_cycles > 0 ? a.wait_cycles : 4000000000LL;   // ~2 s
  const uint32_t slots0 = smem_u32(slots);

  float diff[NO];   // a consumer's largest differences of the chains
#pragma unroll
  for (int o = 0; o < NO; ++o) diff[o] = 0.f;
  if (warp == kWsCons) {
    // ---------------------------------------------------------- producer
    const uint64_t stream_policy = l2_evict_first();
    const RT *myR = nullptr;   // lane o copies objective o's R rows
#pragma unroll
    for (int o = 0; o < NO; ++o)
      if (lane == o) myR = v.R[o];
    int64_t sl = b_lo;
    bool failed = false;
    // lane l: slices sl + l + 32 i of the next round -- pool column, columns, cell
    // class and current values -- loaded before the wait for its slot
    uint32_t off[kWsPer];
    int W[kWsPer], cls[kWsPer];
    Pk old[kWsPer];
    auto fetch = [&]() {
#pragma unroll
      for (int i = 0; i < kWsPer; ++i) {
        off[i] = 0;
        W[i] = 0;
        cls[i] = 0;
        if (lane + 32 * i < kWsRound && sl + lane + 32 * i < b_hi) {
          const int64_t x = sl + lane + 32 * i;
          off[i] = __ldg(a.slice_off + x);
          W[i] = __ldg(a.slice_w + x);
          cls[i] = __ldg(a.cls + x);   // spw = 1: state = slice
          if (!layered) old[i] = v.in[x];
        }
      }
    };
    fetch();
    int slot = 0;
    uint32_t ph = 0;   // phase parity of the slot's current round
    for (int r = 0;; ++r) {
      // (a layer's consumers free no slot before the layer it overlaps has ended: the
      // wait's limit starts then)
      if (layered && r == kWsSlots) pdl_wait();
      if (r >= kWsSlots && !mbar_wait_suspend(empty0 + 8u * (uint32_t)slot, ph ^ 1u, wait_limit)) {
        if (lane == 0) atomicOr(a.err, kErrTimeout);
        failed = true;
        break;
      }
      int n = 0, tot = 0, e[kWsPer];
      const uint32_t off0 = __shfl_sync(0xffffffffu, off[0], 0);
#pragma unroll
      for (int i = 0; i < kWsPer; ++i) e[i] = 0;
      if (sl < b_hi) {
        int carry = 0;
        bool open = true;
#pragma unroll
        for (int i = 0; i < kWsPer; ++i) {
          int cum = W[i] * 128;   // inclusive scan of the entry bytes
#pragma unroll
          for (int d = 1; d < 32; d <<= 1) {
            const int x = __shfl_up_sync(0xffffffffu, cum, d);
            if (lane >= d) cum += x;
          }
          cum += carry;
          const bool valid = open && lane + 32 * i < kWsRound && sl + lane + 32 * i < b_hi;
          const int ni = __popc(__ballot_sync(0xffffffffu, valid && cum <= ecap));   // a prefix of the lanes
          if (ni > 0) tot = __shfl_sync(0xffffffffu, cum, ni - 1);
          e[i] = cum - W[i] * 128;
          if (lane < ni) {
            hdr->slice[slot][32 * i + lane] = make_int2(e[i], W[i] | (cls[i] << 8));
            if (!layered) olds[slot * kWsTab + 32 * i + lane] = old[i];
          }
          n += ni;
          if (ni < 32) open = false;
          carry = __shfl_sync(0xffffffffu, cum, 31);
        }
      }
      __syncwarp();   // the slot's table is written before lane 0 arrives (release)
      const uint32_t fb = full0 + 8u * (uint32_t)slot;
      if (lane == 0) {
        hdr->round[slot] = make_int2((int)sl, n);
        if (n > 0) {
          asm volatile("fence.proxy.async.shared::cta;" ::: "memory");   // the slot's earlier reads
          // (a.test_extra_tx: bytes that never arrive, on the first round of CTA 0,
          // so that a bounded wait runs out -- failure injection for tests)
          const uint32_t extra = (r == 0 && blockIdx.x == 0) ? a.test_extra_tx : 0u;
          mbar_expect_tx(fb, (uint32_t)(tot + NO * n * kRB) + extra);
        } else {
          mbar_arrive(fb);   // no more rounds: the consumers stop here
        }
      }
      __syncwarp();
      if (n == 0) break;
      const uint32_t sbase = slots0 + (uint32_t)(slot * slot_bytes);
      if (a.pool_ordered) {
        // the round's slices are back to back in the pool: one copy
        if (lane == 0 && tot > 0) {
          asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
          bulk_g2s_stream(sbase + (uint32_t)kRBytes, a.pool + (size_t)off0 * 32, (uint32_t)tot, fb, stream_policy);
        }
      } else {
#pragma unroll
        for (int i = 0; i < kWsPer; ++i) {
          if (lane + 32 * i < n && W[i] > 0) {
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            bulk_g2s_stream(sbase + (uint32_t)(kRBytes + e[i]), a.pool + (size_t)off[i] * 32, (uint32_t)W[i] * 128u,
                            fb, stream_policy);
          }
        }
      }
      if (lane < NO) {
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        bulk_g2s_stream(sbase + (uint32_t)(lane * kWsTab * kRB), myR + (size_t)sl * 32, (uint32_t)(n * kRB), fb,
                        stream_policy);
      }
      __syncwarp();
      sl += n;
      fetch();   // the next round's slices
      if (++slot == kWsSlots) {
        slot = 0;
        ph ^= 1u;
      }
    }
    // After a timeout the consumers may have stopped reading: wait (bounded)
    // for the copies of the last rounds issued, whose slots were not reused,
    // so that none is still in flight when the CTA exits.  (Normally every
    // round was waited for by the consumers, and the end-of-block round has
    // reused one of these slots, so this must not run then.)
    if (failed) {
      for (int i = 0; i < kWsSlots; ++i) {
        slot = (slot + kWsSlots - 1) % kWsSlots;   // the last rounds, newest first
        if (slot == kWsSlots - 1) ph ^= 1u;
        mbar_wait_suspend(full0 + 8u * (uint32_t)slot, ph, wait_limit);
      }
    }
  } else {
    // ---------------------------------------------------------- consumers
    if (layered) pdl_wait();   // from here on V of the next layer is read
    uint32_t next_above = 0u;
    if (P == kChains && blockIdx.x == 0 && warp == 0) next_above = chains_look(pr);
    const int nS = (int)a.nS, Nc = (int)a.Nc;
    const int s_lo = (int)pr.s_lo, s_hi = (int)pr.s_hi;
    const RT invN = (RT)1 / (RT)a.N;
    const bool act_ok = lane < a.A;
    int16_t *mypol = v.pol[0];   // lane o < NO writes objective o's policy
#pragma unroll
    for (int o = 1; o < NO; ++o)
      if (lane == o) mypol = v.pol[o];
    const bool mylive = lane < NO && ((live >> lane) & 1u);
    float rf[NO];
    double rd[NO];
#pragma unroll
    for (int o = 0; o < NO; ++o) {
      rf[o] = 0.f;
      rd[o] = 0.0;
    }
    uint8_t *chg_out = a.lflags ? a.lflags + (size_t)(k % 3) * (a.nt + 1) : nullptr;
    int t_cur = -1, t_end = 0;
    bool chg = false;
    int slot = 0;
    uint32_t ph = 0;
    for (;;) {
      if (!mbar_wait_suspend(full0 + 8u * (uint32_t)slot, ph, wait_limit)) {
        if (lane == 0) atomicOr(a.err, kErrTimeout);
        break;
      }
      const int2 rdesc = hdr->round[slot];
      if (rdesc.y == 0) break;
      Acc<RT> accs[kWsPer][NC];
      RT Rvs[kWsPer][NO];
      Pk olds_i[kWsPer];
      int wcs[kWsPer], Ws[kWsPer];
      const uint32_t *ents[kWsPer];
      const Pk *Vns[kWsPer];
      const unsigned char *sb = slots + (size_t)slot * slot_bytes;
      int Wm = 0;
#pragma unroll
      for (int i = 0; i < kWsPer; ++i) {
        const int j = warp + kWsCons * i;
        Ws[i] = 0;
        wcs[i] = 0;
        ents[i] = nullptr;
        Vns[i] = v.in;
        if (j < rdesc.y) {
          const int si = rdesc.x + j;
          const int2 sd = hdr->slice[slot][j];
          wcs[i] = sd.y;
          Ws[i] = sd.y & 0xFF;
          ents[i] = reinterpret_cast<const uint32_t *>(sb + kRBytes + sd.x) + lane;
          Vns[i] = v.in + ((si + Nc <= nS) ? si + Nc : nS);
          const RT *Rs = reinterpret_cast<const RT *>(sb) + j * 32 + lane;
#pragma unroll
          for (int o = 0; o < NO; ++o) Rvs[i][o] = Rs[o * kWsTab * 32];
          if (!layered) olds_i[i] = olds[slot * kWsTab + j];
        }
        Wm = max(Wm, Ws[i]);
      }
#pragma unroll 2
      for (int kk = 0; kk < Wm; ++kk) {   // every column of each slice, ascending
#pragma unroll
        for (int i = 0; i < kWsPer; ++i) {
          if (kk < Ws[i]) {
            const uint32_t w = ents[i][kk * 32];
            const Pk g = Vns[i][(int)(int16_t)(w & 0xFFFFu)];
#pragma unroll
            for (int o = 0; o < NC; ++o) accs[i][o].add(w >> 16, g.v[o], a.N);
          }
        }
      }
      __syncwarp();
      if (lane == 0) mbar_arrive(empty0 + 8u * (uint32_t)slot);   // the slot is read
      if (++slot == kWsSlots) {
        slot = 0;
        ph ^= 1u;
      }
#pragma unroll
      for (int i = 0; i < kWsPer; ++i) {
        if (warp + kWsCons * i >= rdesc.y) continue;
        const int s = rdesc.x + warp + kWsCons * i;
        Acc<RT> (&acc)[NC] = accs[i];
        RT (&Rv)[NO] = Rvs[i];
        const Pk old = olds_i[i];
        const int wc = wcs[i];
        if (a.spill_off) add_spill<RT, NC>(a, s, lane, v.in + ((s + Nc <= nS) ? s + Nc : nS), acc);
        RT qv[NC];
        int qa[NO];
#pragma unroll
        for (int o = 0; o < NC; ++o) {
          RT q = act_ok ? acc[o].q(Rv[o % NO], invN) : -(RT)INFINITY;
          int ia = lane;
          if constexpr (sizeof(RT) == 4) {
            // order-preserving key (-0 keys like +0): the max in one redux,
            // the lowest lane (= lowest action) among the maxima by ballot
            const uint32_t bits = __float_as_uint((float)q + 0.0f);
            const uint32_t key = bits ^ ((uint32_t)((int32_t)bits >> 31) | 0x80000000u);
            const uint32_t kmax = __reduce_max_sync(0xffffffffu, key);
            if (o >= NO) {   // second chain: the value alone, from its key
              qv[o] = __uint_as_float(kmax ^ ((uint32_t)((int32_t)~kmax >> 31) | 0x80000000u));
              continue;
            }
            ia = __ffs(__ballot_sync(0xffffffffu, key == kmax)) - 1;
            q = __shfl_sync(0xffffffffu, q, ia);
          } else {
#pragma unroll
            for (int m = 1; m < 32; m <<= 1) {
              const RT oq = __shfl_xor_sync(0xffffffffu, q, m);
              const int oa = __shfl_xor_sync(0xffffffffu, ia, m);
              if (oq > q || (oq == q && oa < ia)) {
                q = oq;
                ia = oa;
              }
            }
          }
          qv[o] = q;
          if (o < NO) qa[o % NO] = ia;
        }
        if (s < s_lo || s >= s_hi) continue;
        const bool term = (wc >> 8) != CLS_FREE;
        Pk nv;
#pragma unroll
        for (int o = 0; o < NO; ++o) {
          const bool upd = (live >> o) & 1u;
          nv.v[o] = upd ? qv[o] : old.v[o];
          if (upd) {
            if constexpr (sizeof(RT) == 4) rf[o] = fmaxf(rf[o], fabsf(qv[o] - old.v[o]));
            else rd[o] = fmax(rd[o], fabs(qv[o] - old.v[o]));
          }
        }
#pragma unroll
        for (int o = NO; o < Pk::W; ++o) nv.v[o] = (o < NC && !pr.zero_second) ? qv[o < NC ? o : 0] : (RT)0;
        if constexpr (P == kChains) {
#pragma unroll
          for (int o = 0; o < NO; ++o) diff[o] = fmaxf(diff[o], fabsf(nv.v[o] - nv.v[NO + o]));
        }
        int myqa = qa[0];
#pragma unroll
        for (int o = 1; o < NO; ++o)
          if (lane == o) myqa = qa[o];
        if (mylive) mypol[s] = term ? (int16_t)-1 : (int16_t)myqa;
        if (lane == 0) v.out[s] = nv;
        if (chg_out) {
          if (s >= t_end) {   // entered a later layer: publish the finished one
            if (chg && lane == 0) chg_out[t_cur] = 1;
            chg = false;
            t_cur = s / Nc;
            t_end = (t_cur + 1) * Nc;
          }
#pragma unroll
          for (int o = 0; o < NO; ++o) {   // bitwise: -0 vs +0 counts as a change
            if constexpr (sizeof(RT) == 4) chg |= __float_as_uint(nv.v[o]) != __float_as_uint(old.v[o]);
            else chg |= __double_as_longlong(nv.v[o]) != __double_as_longlong(old.v[o]);
          }
        }
      }
    }
    if (chg_out && chg && lane == 0) chg_out[t_cur] = 1;
    if (P == kChains && blockIdx.x == 0 && warp == 0) chains_tell(a, pr, next_above);
    if (!layered && lane == 0) {
#pragma unroll
      for (int o = 0; o < NO; ++o) wmax[warp * NO + o] = (sizeof(RT) == 4) ? (double)rf[o] : rd[o];
    }
  }
  if constexpr (P == kChains) chains_publish<NO, kWsCons>(pr, diff, wmax);
  if (!layered) {
    __syncthreads();
#pragma unroll
    for (int o = 0; o < NO; ++o) {   // thread o publishes objective o
      if (tid == o) {
        double m = 0.0;
        for (int i = 0; i < kWsCons; ++i) m = fmax(m, wmax[i * NO + o]);
        if (m > 0.0) atomicMax(&v.res[o][k - 1], (unsigned long long)__double_as_longlong(m));
      }
    }
  }
}

template <typename RT, int NO, Pass P>
__global__ void __launch_bounds__(32 * (kWsCons + 1), 1) bellman_kernel_ws(SolveArgs a, VSet<RT, NO, P> v, int k,
                                                                         PipeRange pr) {
  extern __shared__ __align__(128) unsigned char sm[];
  __shared__ double wmax[kWsCons * NO];
  __shared__ int s_flag;
  __shared__ int64_t s_cut[2];
  if (P == kSweep) {
    pdl_trigger();
    pdl_wait();
    if (a.lflags && !active_range(a, k, pr, blockIdx.x == 0)) {
      tell_host(pr);
      return;
    }
  }
  bellman_body_ws<RT, NO, P>(a, v, k, pr, sm, wmax, &s_flag, s_cut);
}

// Plan of batched Jacobi sweep k (one block): per model, the slices of the
// layers whose inputs changed in sweep k-1 (nothing once the model met the
// tolerance or ran max_sweeps), with the model's flags for sweep k+1
// cleared.  Then the total is cut into chunks of about total / G slices,
// each model's range into whole chunks, so every CTA entry of the sweep
// holds one model's contiguous range (entries past the last: item -1).
// n <= blockDim.x.
__global__ void plan_batch_kernel(const BatchSolveItem *items, int n, int k, BatchCta *ctas, int G,
                                  int n_entries) {
  __shared__ long long s_cnt[1024];
  __shared__ int s_ctas[1024];
  __shared__ long long s_chunk;
  const int i = threadIdx.x;
  long long lo = 0, hi = 0, s_lo = 0, s_hi = 0;
  if (i < n) {
    const BatchSolveItem &it = items[i];
    const SolveArgs &a = it.a;
    s_hi = a.nS;
    const bool done = k > it.max_sweeps ||
                      (k > 1 && __longlong_as_double((long long)it.res[k - 2]) <= a.tol) ||
                      *(volatile int *)a.err;
    if (a.lflags) {
      const int nt = a.nt;
      const uint8_t *prev = a.lflags + (size_t)((k - 1) % 3) * (nt + 1);
      uint8_t *clr = a.lflags + (size_t)((k + 1) % 3) * (nt + 1);
      int tlo = nt, thi = -1;
      for (int t = 0; t < nt; ++t) {
        if (prev[t] | prev[t + 1]) {
          tlo = min(tlo, t);
          thi = t;
        }
      }
      for (int t = 0; t <= nt; ++t) clr[t] = 0;
      if (thi >= 0 && !done) {
        lo = (long long)tlo * a.Nc / a.spw;
        hi = min((long long)a.n_slices, ((long long)(thi + 1) * a.Nc + a.spw - 1) / a.spw);
      }
    } else if (!done) {
      hi = a.n_slices;
    }
  }
  s_cnt[i] = hi - lo;
  __syncthreads();
  if (i == 0) {
    long long tot = 0;
    for (int j = 0; j < n; ++j) tot += s_cnt[j];
    s_chunk = max(32LL, (tot + G - 1) / G);
  }
  __syncthreads();
  const long long chunk = s_chunk;
  s_ctas[i] = (i < n) ? (int)((s_cnt[i] + chunk - 1) / chunk) : 0;
  __syncthreads();
  if (i < n) {
    int first = 0;
    for (int j = 0; j < i; ++j) first += s_ctas[j];
    for (int c = 0; c < s_ctas[i] && first + c < n_entries; ++c) {
      const long long a0 = lo + (long long)c * chunk;
      ctas[first + c] = BatchCta{i, a0, min(hi, a0 + chunk), s_lo, s_hi};
    }
  }
  if (i == n) {   // unused entries
    int used = 0;
    for (int j = 0; j < n; ++j) used += s_ctas[j];
    for (int e = used; e < n_entries; ++e) ctas[e] = BatchCta{-1, 0, 0, 0, 0};
  }
}

// CTA b's share of step k of a layered batch: layer nt - k of every model that has
// it, cut like the plan's ranges (at least min_chunk slices a CTA).  The layers'
// sizes are known beforehand, so every CTA works its share out itself (one warp,
// two passes over the models; with a planning launch before each of their 148
// steps, 16 uneven models took 43.4 ms, 42.1 so).  The whole CTA calls it.
__device__ BatchCta layer_share(const BatchSolveItem *items, int n, int k, int G, int min_chunk, BatchCta *share) {
  if (threadIdx.x < 32) {
    const int lane = threadIdx.x;
    auto range = [&](int i, int64_t &lo, int64_t &hi, int64_t &s_lo, int64_t &s_hi) {
      lo = hi = 0;
      if (i >= n) return;
      const SolveArgs &a = items[i].a;
      const int t = a.nt - k;
      if (t < 0) return;
      s_lo = (int64_t)t * a.Nc;
      s_hi = s_lo + a.Nc;
      const int sh = __ffs(a.spw) - 1;   // (a power of two)
      lo = s_lo >> sh;
      hi = min((int64_t)a.n_slices, (s_hi + a.spw - 1) >> sh);
    };
    if (lane == 0) share->item = -1;
    long long tot = 0;
    int64_t lo, hi, s_lo = 0, s_hi = 0;
    for (int b = 0; b < n; b += 32) {
      range(b + lane, lo, hi, s_lo, s_hi);
      tot += hi - lo;
    }
    for (int m = 16; m > 0; m >>= 1) tot += __shfl_xor_sync(0xffffffffu, tot, m);
    const unsigned chunk = (unsigned)max((long long)min_chunk, (tot + G - 1) / G);
    int first = 0;
    for (int b = 0; b < n; b += 32) {
      range(b + lane, lo, hi, s_lo, s_hi);
      const int c = (int)(((unsigned)(hi - lo) + chunk - 1) / chunk);
      int incl = c;
      for (int d = 1; d < 32; d <<= 1) {
        const int x = __shfl_up_sync(0xffffffffu, incl, d);
        if (lane >= d) incl += x;
      }
      const int mine = (int)blockIdx.x - (first + incl - c);
      if (mine >= 0 && mine < c) {
        const int64_t a0 = lo + (int64_t)mine * chunk;
        *share = BatchCta{b + lane, a0, min(hi, a0 + (int64_t)chunk), s_lo, s_hi};
      }
      first += __shfl_sync(0xffffffffu, incl, 31);
    }
  }
  __syncthreads();
  return *share;
}

// Batched Jacobi sweep k over many models: CTA b works on ctas[b] (one
// model's contiguous slice range, from the plan); each model stops on its
// own residual.
template <bool layered>
__global__ void __launch_bounds__(32 * kWarps, 4) bellman_batch_kernel(const BatchSolveItem *items,
                                                                    const BatchCta *ctas, int k,
                                                                    int stage_bytes, int n, int G) {
  extern __shared__ __align__(128) unsigned char sm[];
  __shared__ double wmax[kWarps];
  __shared__ int wst_s[kWarps * kDepth];
  __shared__ BatchCta share;
  const BatchCta c = layered ? layer_share(items, n, k, G, kWarps, &share) : ctas[blockIdx.x];
  if (c.item < 0) return;
  const BatchSolveItem &it = items[c.item];
  PipeRange pr{};
  pr.sl_lo = c.sl_lo;
  pr.sl_hi = c.sl_hi;
  pr.s_lo = c.s_lo;
  pr.s_hi = c.s_hi;
  pr.stage_bytes = stage_bytes;
  pr.zero_second = 0;
  pr.grouped = 0;
  VSet<float, 1, layered ? kLayer : kSweep> v;
  v.R[0] = static_cast<const float *>(it.a.R);
  // Jacobi: ping-pong (sweep k reads Va when k is odd); layered: in place in Va
  v.in = reinterpret_cast<const VPack<float, 1> *>((layered || (k & 1)) ? it.Va : it.Vb);
  v.out = reinterpret_cast<VPack<float, 1> *>((layered || !(k & 1)) ? it.Va : it.Vb);
  v.pol[0] = it.policy;
  v.res[0] = layered ? nullptr : it.res;
  bellman_body(it.a, v, layered ? 0 : k, pr.sl_lo, pr.sl_hi, pr, sm, wmax, wst_s);
}

// The same over models with one state per slice, by the grouped sweep.
template <bool layered>
__global__ void __launch_bounds__(32 * kWarpsG, 1) bellman_batch_kernel_g(const BatchSolveItem *items,
                                                                       const BatchCta *ctas, int k,
                                                                       int stage_bytes, int n, int G) {
  extern __shared__ __align__(128) unsigned char sm[];
  __shared__ double wmax[kWarpsG];
  __shared__ int wst_s[kWarpsG * kDepth * kGS];
  __shared__ BatchCta share;
  const BatchCta c = layered ? layer_share(items, n, k, G, 8 * kGS, &share) : ctas[blockIdx.x];
  if (c.item < 0) return;
  const BatchSolveItem &it = items[c.item];
  PipeRange pr{};
  pr.sl_lo = c.sl_lo;
  pr.sl_hi = c.sl_hi;
  pr.s_lo = c.s_lo;
  pr.s_hi = c.s_hi;
  pr.stage_bytes = stage_bytes;
  pr.zero_second = 0;
  pr.grouped = 1;
  VSet<float, 1> v;
  v.R[0] = static_cast<const float *>(it.a.R);
  // Jacobi: ping-pong (sweep k reads Va when k is odd); layered: in place in Va
  v.in = reinterpret_cast<const VPack<float, 1> *>((layered || (k & 1)) ? it.Va : it.Vb);
  v.out = reinterpret_cast<VPack<float, 1> *>((layered || !(k & 1)) ? it.Va : it.Vb);
  v.pol[0] = it.policy;
  v.res[0] = layered ? nullptr : it.res;
  bellman_body_g<float, 1>(it.a, v, layered ? 0 : k, pr.sl_lo, pr.sl_hi, pr, sm, wmax, wst_s);
}

// Per model (one block each): sweeps and residual, final iterate into Va.
__global__ void finalize_batch_kernel(const BatchSolveItem *items, int layered) {
  const BatchSolveItem &it = items[blockIdx.x];
  __shared__ int s_sweeps;
  if (layered) {   // one pass, in place in Va
    if (threadIdx.x == 0) {
      it.stats[0] = 1.0;
      it.stats[1] = 0.0;
    }
    return;
  }
  if (threadIdx.x == 0) {
    int sw = it.max_sweeps;
    for (int k = 1; k <= it.max_sweeps; ++k)
      if (__longlong_as_double((long long)it.res[k - 1]) <= it.a.tol) { sw = k; break; }
    s_sweeps = sw;
    it.stats[0] = (double)sw;
    it.stats[1] = sw > 0 ? __longlong_as_double((long long)it.res[sw - 1]) : 0.0;
  }
  __syncthreads();
  if ((s_sweeps & 1) == 0) return;
  for (int64_t i = threadIdx.x; i <= it.a.nS; i += blockDim.x) it.Va[i] = it.Vb[i];
}

cudaError_t launch_bellman_batch(const BatchSolveItem *items_d, int n, BatchCta *ctas_d, int G, int k,
                                 int stage_bytes, int grouped, int layered, cudaStream_t st) {
  if (n > 1023) return cudaErrorInvalidValue;
  if (!layered) {
    plan_batch_kernel<<<1, 1024, 0, st>>>(items_d, n, k, ctas_d, G, G + n);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
  }
  if (grouped) {
    const size_t smem = 256 + (size_t)kWarpsG * kDepth * stage_bytes;
    auto *fn = layered ? bellman_batch_kernel_g<true> : bellman_batch_kernel_g<false>;
    fn<<<G + n, 32 * kWarpsG, smem, st>>>(items_d, ctas_d, k, stage_bytes, n, G);
  } else {
    const size_t smem = 256 + (size_t)kWarps * kDepth * stage_bytes;
    auto *fn = layered ? bellman_batch_kernel<true> : bellman_batch_kernel<false>;
    fn<<<G + n, 32 * kWarps, smem, st>>>(items_d, ctas_d, k, stage_bytes, n, G);
  }
  return cudaGetLastError();
}

cudaError_t launch_finalize_batch(const BatchSolveItem *items_d, int n, int layered, cudaStream_t st) {
  finalize_batch_kernel<<<n, 256, 0, st>>>(items_d, layered);
  return cudaGetLastError();
}

bool bellman_grouped_fits(int spw, int wcap) { return spw == 1 && grouped_smem(wcap) <= kGroupedSmemMax; }

cudaError_t prepare_bellman_batch(int wcap, int grouped, int layered, int *stage_bytes, int *per_sm) {
  if (grouped) {
    *stage_bytes = kGS * slot_bytes_g(wcap);
    const size_t smem = grouped_smem(wcap);
    if (smem > kGroupedSmemMax) return cudaErrorInvalidConfiguration;
    auto *fn = layered ? bellman_batch_kernel_g<true> : bellman_batch_kernel_g<false>;
    cudaError_t e = allow_max_smem((const void *)fn);
    if (e != cudaSuccess) return e;
    return cudaOccupancyMaxActiveBlocksPerMultiprocessor(per_sm, fn, 32 * kWarpsG, smem);
  }
  *stage_bytes = stage_bytes_for(wcap);
  const size_t smem = 256 + (size_t)kWarps * kDepth * (*stage_bytes);
  if (smem > 227 * 1024) return cudaErrorInvalidConfiguration;
  auto *fn = layered ? bellman_batch_kernel<true> : bellman_batch_kernel<false>;
  cudaError_t e = allow_max_smem((const void *)fn);
  if (e != cudaSuccess) return e;
  return cudaOccupancyMaxActiveBlocksPerMultiprocessor(per_sm, fn, 32 * kWarps, smem);
}

// stats_d[0] = sweeps, [1] = residual of the last sweep.  Copies the final
// iterate into Va when it ended in Vb.
template <typename RT>
__global__ void finalize_kernel(const unsigned long long *res, int max_sweeps, double tol, RT *Va,
                                const RT *Vb, int64_t n, double *stats_d) {
  __shared__ int s_sweeps;
  if (threadIdx.x == 0) {
    int sw = max_sweeps;
    for (int k = 1; k <= max_sweeps; ++k)
      if (__longlong_as_double((long long)res[k - 1]) <= tol) { sw = k; break; }
    s_sweeps = sw;
    if (blockIdx.x == 0) {
      stats_d[0] = (double)sw;
      stats_d[1] = sw > 0 ? __longlong_as_double((long long)res[sw - 1]) : 0.0;
    }
  }
  __syncthreads();
  if ((s_sweeps & 1) == 0) return;   // V_sweeps lives in Va already
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
    Va[i] = Vb[i];
}

// Warp-specialized sweep: per slot the R rows of up to 32 slices and the
// entry bytes of a round; three slots of ~53 KB (FP32, three objectives) keep
// two full rounds of copies in flight while one is read and leave ~60 KB of
// the SM's 256 KB to L1 for the V(s') window.  A slot always holds the widest
// slice.  (Measured on the large instance: 132 KB 114 ms, 160 KB 104 ms,
// 190 KB 104 ms, 215 KB 107 ms per fused solve; four or five slots in the
// same memory make shorter rounds and are slower.)
constexpr size_t kWsSmem = 160 * 1024;

template <typename RT, int NO, Pass P>
static int ws_entry_bytes(int wcap, int smem_kb) {
  const size_t budget = smem_kb > 0 ? (size_t)smem_kb * 1024 : kWsSmem;
  const long per_slot = (long)((budget - ws_hdr_bytes() - ws_old_bytes<RT, VSet<RT, NO, P>::NC>()) / kWsSlots) - ws_r_bytes<RT>(NO);
  long e = std::max<long>(per_slot, (long)wcap * 128);
  return (int)(e & ~127L);
}

// Launch shape of a sweep over `slices` slices, or of a layer of a backward pass (a
// launch per layer).
// A layer is as long as its longest warp, so the warp-per-slice kernel spreads
// one over all the warps it can (a sweep gives a warp at least four slices, which
// keeps its copies ahead of its sums).  Measured per layer, two chains: 200 slices
// 6.3 us with four slices a warp, 3.3 with one; 1733 slices 7.6 and 3.4;
// 12,800 slices 10.4 and 7.5.
// For one state per slice that kernel also takes the layers up to kLayerSlices
// slices per resident warp from the warp-specialized one, whose rounds of 31 slices
// pay off above (us a layer of 10,000 / 40,000 slices, 32 actions: one objective, two
// chains 6.1 / 14.9 against 7.6 / 14.5; three objectives, one chain 7.1 / 18.6
// against 8.3 / 16.5, two chains 9.4 / 28.9 against 10.4 / 22.2).
template <int NC>
constexpr int kLayerSlices = NC <= 2 ? 7 : 3;
template <typename RT, int NO, Pass P>
static cudaError_t pipe_config(const SolveArgs &a, int64_t slices, PipeRange *pr, size_t *smem, int *blocks) {
  constexpr bool layer = P != kSweep;
  pr->zero_second = 0;
  // the warp-per-slice kernel's stages
  const int stage = stage_bytes_for(a.wcap);
  const size_t warp_smem = 256 + (size_t)kWarps * kDepth * stage;
  const bool ws = a.spw == 1 && !a.small_ctas;   // one state per slice: the warp-specialized sweep, any width
  int per_sm = 0;
  if (warp_smem <= 227 * 1024 && (!ws || (layer && sizeof(RT) == 4))) {
    cudaError_t e = allow_max_smem((const void *)bellman_kernel<RT, NO, P>);
    if (e != cudaSuccess) return e;
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, bellman_kernel<RT, NO, P>, 32 * kWarps, warp_smem);
    if (e != cudaSuccess) return e;
  }
  if (ws && slices > (int64_t)num_sms() * per_sm * kWarps * kLayerSlices<VSet<RT, NO, P>::NC>) {
    pr->grouped = 2;
    pr->stage_bytes = ws_entry_bytes<RT, NO, P>(a.wcap, a.sweep_smem_kb);
    *smem = ws_hdr_bytes() + ws_old_bytes<RT, VSet<RT, NO, P>::NC>() + (size_t)kWsSlots * (ws_r_bytes<RT>(NO) + pr->stage_bytes);
    cudaError_t e = allow_max_smem((const void *)bellman_kernel_ws<RT, NO, P>);
    if (e != cudaSuccess) return e;
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, bellman_kernel_ws<RT, NO, P>, 32 * (kWsCons + 1), *smem);
    if (e != cudaSuccess) return e;
    if (per_sm < 1) return cudaErrorInvalidConfiguration;
    int64_t b = (int64_t)num_sms() * per_sm;
    const int64_t want = (slices + 2 * kWsRound - 1) / (2 * kWsRound);   // >= 2 rounds per CTA
    if (b > want) b = want;
    if (b < 1) b = 1;
    *blocks = (int)b;
    return cudaSuccess;
  }
  pr->grouped = 0;   // the warp-per-slice kernel
  pr->stage_bytes = stage;
  *smem = warp_smem;
  if (per_sm < 1) return cudaErrorInvalidConfiguration;
  int64_t b = (int64_t)num_sms() * per_sm;
  const int per_warp = layer ? 1 : 4;
  const int64_t want = (slices + per_warp * kWarps - 1) / (per_warp * kWarps);
  if (b > want) b = want;
  if (b < 1) b = 1;
  *blocks = (int)b;
  return cudaSuccess;
}

// Fused solve epilogue: objective o's sweep count is the first k whose
// residual met tol (else max_sweeps); the table of the last executed sweep
// (the largest count; 0 = the initial table) holds every objective's final
// values, since a finished objective is carried forward unchanged.  Writes
// the stats and copies objective o's column into V[o][0..n).
template <typename RT, int NO>
struct VOut {
  RT *V[NO];
};
template <typename RT, int NO>
__global__ void finalize_multi_kernel(const double *stats_base, size_t blk, int max_sweeps, double tol,
                                      const VPack<RT, NO> *ta, const VPack<RT, NO> *tb, VOut<RT, NO> out,
                                      int64_t n, double *stats_out, int layered) {
  __shared__ int s_last;
  if (threadIdx.x == 0) {
    int last = 0;
    for (int o = 0; o < NO; ++o) {
      const unsigned long long *res = reinterpret_cast<const unsigned long long *>(stats_base + o * blk + 4);
      int sw = max_sweeps;
      if (!layered) {
        for (int k = 1; k <= max_sweeps; ++k)
          if (__longlong_as_double((long long)res[k - 1]) <= tol) { sw = k; break; }
      }
      last = max(last, sw);
      if (blockIdx.x == 0 && !layered) {
        stats_out[o * blk + 0] = (double)sw;
        stats_out[o * blk + 1] = sw > 0 ? __longlong_as_double((long long)res[sw - 1]) : 0.0;
      }
    }
    s_last = layered ? 0 : last;
  }
  __syncthreads();
  const VPack<RT, NO> *t = (s_last & 1) ? tb : ta;   // sweep k writes tb when k is odd
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    const VPack<RT, NO> p = t[i];
#pragma unroll
    for (int o = 0; o < NO; ++o) out.V[o][i] = p.v[o];
  }
}

// pdl: the launch may start while the previous kernel of the stream finishes
// (the layers of a layered pass).
template <typename RT, int NO, Pass P>
static void launch_sweep(const SolveArgs &a, const VSet<RT, NO, P> &v, int k, const PipeRange &pr, int blocks,
                         size_t smem, cudaStream_t st, bool pdl = false) {
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3((unsigned)blocks);
  cfg.blockDim = dim3(pr.grouped == 2 ? 32 * (kWsCons + 1) : 32 * kWarps);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute at{};
  at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at.val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = &at;
  cfg.numAttrs = pdl ? 1 : 0;
  if (pr.grouped == 2) cudaLaunchKernelEx(&cfg, bellman_kernel_ws<RT, NO, P>, a, v, k, pr);
  else cudaLaunchKernelEx(&cfg, bellman_kernel<RT, NO, P>, a, v, k, pr);
}

constexpr int64_t kOverlapSlices = 500000;
static bool stop_told(const SolveStop &s) { return s.host && *(volatile unsigned int *)s.host == s.token; }

// Objective o's status block: stats_d + o*(4 + max_sweeps) holds sweeps,
// residual, (objective 0: the error word), spare, then one residual slot
// per sweep.  NO = 1 iterates in the caller's V and io.Vtmp[0]; NO > 1 in
// the packed tables io.table[0..1], copied out to V[o] at the end.
// stop.host != nullptr: no more sweeps are launched once one has found nothing left
// to do (21 x 27 cells, 103 layers: the empty launches of a run that ends in sweep
// 24 took a fifth of its time); a sweep that was not launched leaves its residual 0
// like one that did nothing.
template <typename RT, int NO>
static cudaError_t jacobi_t(const SolveArgs &a, int max_sweeps, const SolveIO &io, double *stats_d,
                            const SolveStop &stop, cudaStream_t st) {
  using Pk = VPack<RT, NO>;
  const size_t blk = 4 + (size_t)max_sweeps;
  Pk *ta = static_cast<Pk *>(NO == 1 ? io.V[0] : io.table[0]);
  Pk *tb = static_cast<Pk *>(NO == 1 ? io.Vtmp[0] : io.table[1]);
  VSet<RT, NO> odd, even;   // sweep k reads ta when k is odd, tb when even
  odd.in = ta;
  odd.out = tb;
  even.in = tb;
  even.out = ta;
  for (int o = 0; o < NO; ++o) {
    unsigned long long *res = reinterpret_cast<unsigned long long *>(stats_d + o * blk + 4);
    cudaError_t e = cudaMemsetAsync(res, 0, sizeof(unsigned long long) * (size_t)max_sweeps, st);
    if (e != cudaSuccess) return e;
    odd.R[o] = even.R[o] = static_cast<const RT *>(io.R[o]);
    odd.pol[o] = even.pol[o] = io.policy[o];
    odd.res[o] = even.res[o] = res;
  }
  if (a.lflags) {   // sweep 1 recomputes every layer
    cudaError_t e = cudaMemsetAsync(a.lflags, 1, (size_t)a.nt, st);
    if (e == cudaSuccess) e = cudaMemsetAsync(a.lflags + a.nt, 0, (size_t)a.nt + 2, st);
    if (e == cudaSuccess && a.work) e = cudaMemsetAsync(a.work, 0, sizeof(unsigned long long) * max_sweeps, st);
    if (e != cudaSuccess) return e;
  }
  PipeRange pr{};
  size_t smem = 0;
  int blocks = 1;
  cudaError_t e = pipe_config<RT, NO, kSweep>(a, a.n_slices, &pr, &smem, &blocks);
  if (e != cudaSuccess) return e;
  pr.sl_lo = 0;
  pr.sl_hi = a.n_slices;
  pr.s_lo = 0;
  pr.s_hi = a.nS;
  pr.stop = stop;
  SolveArgs rest = a;   // a test's injected failure is for the first launch alone
  rest.test_extra_tx = 0;
  // A sweep starts while the one before ends, unless it is long and its CTAs fill an SM
  // each: they then take the SMs in the order these fall free, which costs more than
  // the launch (us a full sweep with and without, 32 actions: 58,000 slices 20.3 and
  // 22.6, 490,000 113.7 and 114.1, 600,000 141 and 139, 4.8 million 1219 and 1092).
  const bool pdl = pr.grouped != 2 || a.n_slices <= kOverlapSlices;
  for (int k = 1; k <= max_sweeps && !stop_told(stop); ++k)
    launch_sweep(k > 1 ? rest : a, (k & 1) ? odd : even, k, pr, blocks, smem, st, pdl && k > 1);
  e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  int64_t fb = (a.nS + 1 + 255) / 256;
  if (fb > 1024) fb = 1024;
  if constexpr (NO == 1) {
    finalize_kernel<RT><<<(unsigned)fb, 256, 0, st>>>(odd.res[0], max_sweeps, a.tol, static_cast<RT *>(io.V[0]),
                                                       static_cast<const RT *>(io.Vtmp[0]), a.nS + 1, stats_d);
  } else {
    VOut<RT, NO> out;
    for (int o = 0; o < NO; ++o) out.V[o] = static_cast<RT *>(io.V[o]);
    finalize_multi_kernel<RT, NO><<<(unsigned)fb, 256, 0, st>>>(stats_d, blk, max_sweeps, a.tol, ta, tb, out,
                                                                 a.nS + 1, stats_d, 0);
  }
  return cudaGetLastError();
}

template <typename RT>
static cudaError_t jacobi_n(const SolveArgs &a, int max_sweeps, const SolveIO &io, double *stats_d,
                            const SolveStop &stop, cudaStream_t st) {
  switch (io.n) {
    case 1: return jacobi_t<RT, 1>(a, max_sweeps, io, stats_d, stop, st);
    case 2: return jacobi_t<RT, 2>(a, max_sweeps, io, stats_d, stop, st);
    case 3: return jacobi_t<RT, 3>(a, max_sweeps, io, stats_d, stop, st);
    default: return cudaErrorInvalidValue;
  }
}

cudaError_t launch_jacobi_multi(const SolveArgs &a, int precision, int max_sweeps, const SolveIO &io,
                                double *stats_d, const SolveStop &stop, cudaStream_t st) {
  if (precision == MDP_FP64_CHECK) return jacobi_n<double>(a, max_sweeps, io, stats_d, stop, st);
  return jacobi_n<float>(a, max_sweeps, io, stats_d, stop, st);
}

cudaError_t launch_jacobi(const SolveArgs &a, int precision, int max_sweeps, void *Va, void *Vb,
                          int16_t *policy, double *stats_d, cudaStream_t st) {
  SolveIO io{};
  io.n = 1;
  io.R[0] = a.R;
  io.V[0] = Va;
  io.Vtmp[0] = Vb;
  io.policy[0] = policy;
  return launch_jacobi_multi(a, precision, max_sweeps, io, stats_d, SolveStop{nullptr, 0}, st);
}

// In place: layer t reads layer t+1, finished by the previous launch.
template <typename RT, int NO>
static cudaError_t layered_t(const SolveArgs &a, int nt, const SolveIO &io, double *stats_d,
                             cudaStream_t st) {
  using Pk = VPack<RT, NO>;
  PipeRange pr0{};
  size_t smem = 0;
  int blocks = 1;
  // every layer has the same number of slices (up to one straddling slice)
  cudaError_t e = pipe_config<RT, NO, kLayer>(a, (a.Nc + a.spw - 1) / a.spw + 1, &pr0, &smem, &blocks);
  if (e != cudaSuccess) return e;
  VSet<RT, NO, kLayer> v;
  Pk *t = static_cast<Pk *>(NO == 1 ? io.V[0] : io.table[0]);
  v.in = t;
  v.out = t;
  for (int o = 0; o < NO; ++o) {
    v.R[o] = static_cast<const RT *>(io.R[o]);
    v.pol[o] = io.policy[o];
    v.res[o] = nullptr;
  }
  SolveArgs rest = a;   // a test's injected failure is for the first launch alone
  rest.test_extra_tx = 0;
  for (int t_ = nt - 1; t_ >= 0; --t_) {
    PipeRange pr = pr0;
    pr.s_lo = (int64_t)t_ * a.Nc;
    pr.s_hi = pr.s_lo + a.Nc;
    pr.sl_lo = pr.s_lo / a.spw;
    pr.sl_hi = (pr.s_hi + a.spw - 1) / a.spw;
    launch_sweep(t_ < nt - 1 ? rest : a, v, 0, pr, blocks, smem, st, t_ < nt - 1);
  }
  e = cudaGetLastError();
  if (e != cudaSuccess || NO == 1) return e;
  VOut<RT, NO> out;
  for (int o = 0; o < NO; ++o) out.V[o] = static_cast<RT *>(io.V[o]);
  int64_t fb = (a.nS + 1 + 255) / 256;
  if (fb > 1024) fb = 1024;
  finalize_multi_kernel<RT, NO><<<(unsigned)fb, 256, 0, st>>>(stats_d, 0, 0, a.tol, t, t, out, a.nS + 1,
                                                               stats_d, 1);
  return cudaGetLastError();
}

// ---- the Jacobi result by two chains ----
// What a cold-started Jacobi run (V_0 = 0) to tolerance tol >= 0 returns, from
// one pass over P instead of nt + 1 sweeps, when that is certain.  In this
// time-layered MDP V_k = V* on the layers t >= nt - k, bit for bit (layer nt-1
// has no successors, and layer t's values are computed from layer t+1's by the
// same operations in every sweep).  Let W(t) = V_{nt-t-1}(t) be layer t's last
// iterate before that: W(nt-1) = 0 and W(t) = T W(t+1), a second backward
// chain.  Sweep k = nt - t changes layer t from W(t) to V*(t), so its residual
// is at least d_t = max |V*(t) - W(t)|.  If every d_t exceeds tol, no sweep
// 1..nt stops the run, and sweep nt + 1 changes nothing: the run ends there
// with V*, its greedy policy, nt + 1 sweeps and residual 0.  If only d_0 does
// not, sweep nt ends the run with the same V and policy: it changes no other
// layer, so its residual is d_0.  (Otherwise the caller runs the sweeps.)  Both
// chains share the entry stream, so the pass costs little more than a layered
// one; a run whose tolerance is met earlier pays for the layers up to there
// (21 x 27 cells, 103 layers, 16 actions, met in sweep 24: 0.25 ms when all
// layers ran).
//
// Copies the first chain to V[o], if the pass was not given up.
template <int NO>
__global__ void finalize_two_kernel(const VPack<float, 2 * NO> *tab, VOut<float, NO> out, int64_t n, ChainWords *w,
                                    const ChainSlot *slots, uint32_t *above) {
  if (*(volatile const int *)&w->err) return;
  if (blockIdx.x == 0 && threadIdx.x < 32) {   // layer 0
    const ChainSlot c = slots[threadIdx.x];
    const unsigned any = __reduce_or_sync(0xffffffffu, c.above);
    if (threadIdx.x == 0) above[0] = any;
    for (int o = 0; o < 3; ++o) {
      const unsigned d = __reduce_max_sync(0xffffffffu, c.first[o]);
      if (threadIdx.x == 0) w->first[o] = d;
    }
  }
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    const VPack<float, 2 * NO> p = tab[i];
#pragma unroll
    for (int o = 0; o < NO; ++o) out.V[o][i] = p.v[o];
  }
}

// io.table[0]: the packed table of 2 n components per state, its last entry zeroed by
// the caller like w.
template <int NO>
static cudaError_t two_chains_t(const SolveArgs &a, int nt, const SolveIO &io, ChainWords *w, const SolveStop &stop,
                                cudaStream_t st) {
  PipeRange pr0{};
  size_t smem = 0;
  int blocks = 1;
  cudaError_t e = pipe_config<float, NO, kChains>(a, (a.Nc + a.spw - 1) / a.spw + 1, &pr0, &smem, &blocks);
  if (e != cudaSuccess) return e;
  VSet<float, NO, kChains> v;
  auto *t = static_cast<VPack<float, 2 * NO> *>(io.table[0]);
  v.in = t;
  v.out = t;
  VOut<float, NO> out;
  for (int o = 0; o < NO; ++o) {
    v.R[o] = static_cast<const float *>(io.R[o]);
    v.pol[o] = io.policy[o];
    v.res[o] = nullptr;
    out.V[o] = static_cast<float *>(io.V[o]);
  }
  SolveArgs rest = a;   // a test's injected failure is for the first launch alone
  rest.test_extra_tx = 0;
  pr0.stop = stop;
  uint32_t *above = chain_above(w);
  ChainSlot *slots = chain_slots(w, nt);
  pr0.tol = (float)a.tol;
  if ((double)pr0.tol > a.tol) pr0.tol = std::nextafter(pr0.tol, -1.f);
  for (int t_ = nt - 1; t_ >= 0; --t_) {
    if (stop_told(stop)) break;   // given up
    PipeRange pr = pr0;
    pr.s_lo = (int64_t)t_ * a.Nc;
    pr.s_hi = pr.s_lo + a.Nc;
    pr.sl_lo = pr.s_lo / a.spw;
    pr.sl_hi = (pr.s_hi + a.spw - 1) / a.spw;
    pr.zero_second = t_ == nt - 1;
    pr.slots = slots + (size_t)t_ * kChainSlots;
    pr.next_slots = t_ < nt - 1 ? pr.slots + kChainSlots : nullptr;
    pr.next_above = above + t_ + 1;
    pr.first = t_ == 0;
    launch_sweep(t_ < nt - 1 ? rest : a, v, 0, pr, blocks, smem, st, t_ < nt - 1);
  }
  e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  const int64_t fb = std::min<int64_t>((a.nS + 256) / 256, (int64_t)num_sms() * 8);
  finalize_two_kernel<NO><<<(unsigned)fb, 256, 0, st>>>(t, out, a.nS + 1, w, slots, above);
  return cudaGetLastError();
}

cudaError_t launch_two_chains(const SolveArgs &a, int nt, const SolveIO &io, ChainWords *w, const SolveStop &stop,
                              cudaStream_t st) {
  switch (io.n) {
    case 1: return two_chains_t<1>(a, nt, io, w, stop, st);
    case 2: return two_chains_t<2>(a, nt, io, w, stop, st);
    case 3: return two_chains_t<3>(a, nt, io, w, stop, st);
    default: return cudaErrorInvalidValue;
  }
}

template <typename RT>
static cudaError_t layered_n(const SolveArgs &a, int nt, const SolveIO &io, double *stats_d,
                             cudaStream_t st) {
  switch (io.n) {
    case 1: return layered_t<RT, 1>(a, nt, io, stats_d, st);
    case 2: return layered_t<RT, 2>(a, nt, io, stats_d, st);
    case 3: return layered_t<RT, 3>(a, nt, io, stats_d, st);
    default: return cudaErrorInvalidValue;
  }
}

cudaError_t launch_layered_multi(const SolveArgs &a, int precision, int nt, const SolveIO &io,
                                 double *stats_d, cudaStream_t st) {
  if (precision == MDP_FP64_CHECK) return layered_n<double>(a, nt, io, stats_d, st);
  return layered_n<float>(a, nt, io, stats_d, st);
}

}  // namespace mdpgb
