// export.cu -- the pool's compaction into slice order and the paper-layout
// export (CSR over row = a |S| + s), with the prefix sums both need.
#include <algorithm>

#include "build_common.cuh"

namespace mdpgb {

// ------------------------------------------------------ prefix sums ----
// Exclusive sums over tiles of kTile values: x[i] holds the sum within the tile,
// tile[i / kTile] the sum of the tiles before (after scan_offsets), so that the
// consumer adds the two and no pass over x is spent on it.  x is a plain array or
// scattered over another one (At: where value i lies).
constexpr int kScanThreads = 512, kScanItems = 8, kTile = kScanThreads * kScanItems;

template <class Load, class At>
__global__ void __launch_bounds__(kScanThreads) scan_tiles_kernel(Load load, int64_t n, At x, int64_t *tile) {
  __shared__ int64_t wsum[kScanThreads / 32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int64_t base = (int64_t)blockIdx.x * kTile + warp * (32 * kScanItems);   // a warp's values are consecutive
  int64_t v[kScanItems], run = 0;
#pragma unroll
  for (int i = 0; i < kScanItems; ++i) {
    const int64_t at = base + 32 * i + lane;
    v[i] = at < n ? load(at) : 0;
  }
#pragma unroll
  for (int i = 0; i < kScanItems; ++i) {
    int64_t s = v[i];
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      const int64_t o = __shfl_up_sync(0xffffffffu, s, d);
      if (lane >= d) s += o;
    }
    v[i] = run + s - v[i];
    run += __shfl_sync(0xffffffffu, s, 31);
  }
  if (lane == 0) wsum[warp] = run;
  __syncthreads();
  int64_t before = 0, all = 0;
  for (int w = 0; w < kScanThreads / 32; ++w) {
    if (w < warp) before += wsum[w];
    all += wsum[w];
  }
#pragma unroll
  for (int i = 0; i < kScanItems; ++i) {
    const int64_t at = base + 32 * i + lane;
    if (at < n) *x(at) = v[i] + before;
  }
  if (threadIdx.x == 0) tile[blockIdx.x] = all;
}

__global__ void scan_add_kernel(int64_t *x, int64_t n, const int64_t *tile) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
    x[i] += tile[i / kTile];
}

struct Words {
  int64_t *x;
  __device__ __forceinline__ int64_t *operator()(int64_t i) const { return x + i; }
};
template <class At>
struct LoadWords {
  At at;
  __device__ __forceinline__ int64_t operator()(int64_t i) const { return *at(i); }
};
struct LoadBytes {
  const uint8_t *x;
  __device__ __forceinline__ int64_t operator()(int64_t i) const { return x[i]; }
};

// words of `tile` memory that n values need
static int64_t scan_words(int64_t n) {
  int64_t need = 0;
  do {
    n = (n + kTile - 1) / kTile;
    need += n;
  } while (n > 1);
  return need;
}

// x and tile as above (load may read x itself: a thread reads its values before it writes them)
template <class Load, class At>
static cudaError_t scan_offsets(Load load, int64_t n, At x, int64_t *tile, cudaStream_t st) {
  const int64_t tiles = (n + kTile - 1) / kTile;
  scan_tiles_kernel<<<(unsigned)tiles, kScanThreads, 0, st>>>(load, n, x, tile);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  if (tiles == 1) return cudaMemsetAsync(tile, 0, sizeof(int64_t), st);
  int64_t *up = tile + tiles;
  e = scan_offsets(LoadWords<Words>{{tile}}, tiles, Words{tile}, up, st);
  if (e != cudaSuccess || tiles <= kTile) return e;   // one tile of tiles: its offset is 0
  scan_add_kernel<<<(unsigned)std::min<int64_t>((tiles + 255) / 256, 8192), 256, 0, st>>>(tile, tiles, up);
  return cudaGetLastError();
}

// ------------------------------------------------------- compaction ----
// One warp per slice: the slice's W columns are W*128 contiguous bytes in
// both pools, copied as 16-byte vectors; then the new offset is recorded.
__global__ void pool_reorder_kernel(const uint32_t *__restrict__ pool, uint32_t *__restrict__ out,
                                    uint32_t *slice_off, const uint8_t *__restrict__ slice_w,
                                    const int64_t *__restrict__ new_off, const int64_t *__restrict__ tile,
                                    int64_t n_slices) {
  const int lane = threadIdx.x & 31;
  const int64_t wid = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
  const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
  for (int64_t sl = wid; sl < n_slices; sl += nwarps) {
    const int W = slice_w[sl];
    const int64_t no = new_off[sl] + tile[sl / kTile];
    if (W) {
      const uint4 *src = reinterpret_cast<const uint4 *>(pool + (size_t)slice_off[sl] * 32);
      uint4 *dst = reinterpret_cast<uint4 *>(out + (size_t)no * 32);
      for (int i = lane; i < W * 8; i += 32) dst[i] = src[i];
    }
    __syncwarp();
    if (lane == 0) slice_off[sl] = (uint32_t)no;
  }
}

cudaError_t launch_pool_reorder(const uint32_t *pool, uint32_t *out, uint32_t *slice_off, const uint8_t *slice_w,
                                int64_t n_slices, cudaStream_t st) {
  if (n_slices < 1) return cudaSuccess;
  int64_t *x = nullptr;
  cudaError_t e = dev_alloc((void **)&x, sizeof(int64_t) * (size_t)(n_slices + scan_words(n_slices)), st);
  if (e != cudaSuccess) return e;
  int64_t *tile = x + n_slices;
  e = scan_offsets(LoadBytes{slice_w}, n_slices, Words{x}, tile, st);
  if (e == cudaSuccess) {
    const int64_t blocks = std::min<int64_t>(num_sms() * 16, (n_slices + 7) / 8);
    pool_reorder_kernel<<<(unsigned)blocks, 256, 0, st>>>(pool, out, slice_off, slice_w, x, tile, n_slices);
    e = cudaGetLastError();
  }
  dev_free(x, st);
  return e;
}

// ----------------------------------------------------------- export ----
// The model stores a state's rows side by side, the paper layout an action's: a
// block of kXState states by all actions is transposed through shared memory.
// Bound by memory: the entries are read once (4 bytes) and written once (12).
//   lengths   per (action, block) the sum of its rows' lengths; scanned over
//             a nb + b, it is where the block's rows of action a begin.
//             (Where there is no memory for the sums, they lie in the caller's
//             rowptr, each where its block's first row ends up; always there,
//             the exports below took 10 to 18 % longer.)
//   fill      the block's slices are staged in shared memory, words of slice j
//             rotated by j so that reading one action's row of every state
//             meets every bank once; warp by action, lane by state, the row's
//             entries are staged in output order and leave as whole lines.
// (One thread per row wrote the entries 8 bytes at a time to rows |S| apart, and
// two scans over all rows took as long: 90 x 90 cells, 40 layers, 16 actions,
// 5.2 million rows: 0.80 ms for an export with entries and one without,
// 0.32 ms so.)
constexpr int kXState = 32;      // states of a block
constexpr int kXWarps = 8;
constexpr int kXCols = 320;      // staged columns of the block's slices (40 KB)
constexpr int kXStage = 384;     // staged entries of a warp's action (12 a row)

struct ExportArgs {
  const uint32_t *pool, *slice_off, *spill, *spill_off;
  const uint8_t *slice_w, *nnz;
  const uint16_t *sinkc;
  int64_t nS, Nc, n_slices, blocks;
  int32_t A, A_pad, spw;
  int64_t *sums;          // of (action, block) at act * sum_act + block * sum_block, then their scan
  int64_t sum_act, sum_block;
  const int64_t *tile;
  int64_t *rowptr, *col;
  int32_t *count;
};

__device__ __forceinline__ int spill_len(const ExportArgs &a, int64_t sl, int lane) {
  if (!a.spill_off) return 0;
  const uint32_t off = a.spill_off[sl];
  return off == kNoSlice ? 0 : (int)(a.spill[off + lane + 1] - a.spill[off + lane]);
}

// Sum i = a nb + b of the lengths (and its scan) in rowptr.
struct RowptrSums {
  int64_t *rowptr;
  int64_t nS, blocks;
  __device__ __forceinline__ int64_t *operator()(int64_t i) const {
    const int64_t act = layer_of(i, blocks, nS);   // (i <= nS)
    return rowptr + act * nS + (i - act * blocks) * kXState;
  }
};

// warp per block: lane = row of a slice
__global__ void __launch_bounds__(256) export_lengths_kernel(ExportArgs a) {
  const int lane = threadIdx.x & 31, act = lane % a.A_pad, q = lane / a.A_pad;
  const int per = kXState / a.spw;   // slices of a block
  const int64_t warps = (int64_t)gridDim.x * (blockDim.x >> 5);
  for (int64_t b = blockIdx.x * (int64_t)(blockDim.x >> 5) + (threadIdx.x >> 5); b < a.blocks; b += warps) {
    unsigned long long len = 0;
    const int64_t sl0 = b * per;
#pragma unroll 4
    for (int j = 0; j < per; ++j) {
      const int64_t sl = sl0 + j, ir = sl * 32 + lane;
      if (sl < a.n_slices && sl * a.spw + q < a.nS && act < a.A)
        len += (unsigned)(a.nnz[ir] + spill_len(a, sl, lane) + (a.sinkc[ir] ? 1 : 0));
    }
    for (int off = a.A_pad; off < 32; off <<= 1) len += __shfl_xor_sync(0xffffffffu, len, off);
    if (q == 0 && act < a.A) a.sums[(int64_t)act * a.sum_act + b * a.sum_block] = (int64_t)len;
  }
}

template <typename RT>
struct ExportSmem {
  uint32_t cols[kXCols * 32];
  unsigned long long stage[kXWarps][kXStage];   // state of the block, entry word
  uint32_t row[kXState * 32];                   // [slice][rotated lane]: entries | sink count << 8
  RT R[kXState * 32];
  int first[kXState + 1];                       // first staged column of each slice
  uint32_t off[kXState];
};

template <typename RT>
__global__ void __launch_bounds__(32 * kXWarps) export_fill_kernel(const ExportArgs a, const RT *__restrict__ Rsrc,
                                                                   RT *__restrict__ Rdst) {
  extern __shared__ __align__(16) unsigned char xsm[];
  ExportSmem<RT> &sm = *reinterpret_cast<ExportSmem<RT> *>(xsm);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int spw = a.spw, per = kXState / spw;
  const bool entries = a.col || a.count;
  for (int64_t b = blockIdx.x; b < a.blocks; b += gridDim.x) {
    const int64_t sl0 = b * per, s0 = b * kXState;
    const int n_sl = (int)min((int64_t)per, a.n_slices - sl0);
    if (warp == 0) {
      const int W = lane < n_sl ? a.slice_w[sl0 + lane] : 0;
      int incl = W;
#pragma unroll
      for (int d = 1; d < 32; d <<= 1) {
        const int o = __shfl_up_sync(0xffffffffu, incl, d);
        if (lane >= d) incl += o;
      }
      sm.first[lane] = incl - W;
      if (lane == 31) sm.first[32] = incl;
      if (lane < n_sl) sm.off[lane] = a.slice_off[sl0 + lane];
    }
    for (int j = warp; j < n_sl; j += kXWarps) {
      const int64_t ir = (sl0 + j) * 32 + lane;
      const int at = j * 32 + ((lane + j) & 31);
      sm.row[at] = (uint32_t)a.nnz[ir] | (uint32_t)a.sinkc[ir] << 8;
      if (Rdst) sm.R[at] = Rsrc[ir];
    }
    __syncthreads();
    const bool staged = sm.first[32] <= kXCols;
    if (entries && staged) {
      for (int j = warp; j < n_sl; j += kXWarps) {
        const int f = sm.first[j], W = sm.first[j + 1] - f, to = (lane + j) & 31;
        const uint32_t *src = a.pool + (size_t)sm.off[j] * 32 + lane;
#pragma unroll 4
        for (int k = 0; k < W; ++k) sm.cols[(f + k) * 32 + to] = src[(size_t)k * 32];
      }
      __syncthreads();
    }
    // warp = action, lane = state
    const int64_t s = s0 + lane;
    const int j = lane / spw, q = lane % spw;
    for (int act = warp; act < a.A; act += kXWarps) {
      const int64_t begin = a.sums[(int64_t)act * a.sum_act + b * a.sum_block] + a.tile[((int64_t)act * a.blocks + b) / kTile];
      __syncwarp();   // (the sum's place may be a row's of this block)
      const int l = q * a.A_pad + act, to = (l + j) & 31;
      const bool on = s < a.nS;
      const uint32_t rw = on ? sm.row[j * 32 + to] : 0u;
      const int e = (int)(rw & 0xFFu), sp = on ? spill_len(a, sl0 + j, l) : 0;
      const uint32_t sink = rw >> 8;
      const int len = e + sp + (sink ? 1 : 0);
      int incl = len;
#pragma unroll
      for (int d = 1; d < 32; d <<= 1) {
        const int o = __shfl_up_sync(0xffffffffu, incl, d);
        if (lane >= d) incl += o;
      }
      const int total = __shfl_sync(0xffffffffu, incl, 31), mine = incl - len;
      const int64_t r = (int64_t)act * a.nS + s;
      if (on) {
        a.rowptr[r] = begin + mine;
        if (act == a.A - 1 && s == a.nS - 1) a.rowptr[r + 1] = begin + incl;
        if (Rdst) Rdst[r] = sm.R[j * 32 + to];
      }
      if (!entries) continue;
      const uint32_t *src = staged ? sm.cols + sm.first[min(j, n_sl - 1)] * 32 + to
                                   : a.pool + (on && e ? (size_t)sm.off[j] * 32 : (size_t)0) + l;
      const uint32_t *tail = sp ? a.spill + a.spill_off[sl0 + j] + kSpillHdr + a.spill[a.spill_off[sl0 + j] + l] : nullptr;
      if (total <= kXStage) {
        unsigned long long *st = sm.stage[warp] + mine;
        const unsigned long long who = (unsigned long long)(unsigned)lane << 32;
        for (int k = 0; k < e; ++k) *st++ = who | src[(size_t)k * 32];
        for (int k = 0; k < sp; ++k) *st++ = who | tail[k];   // (ascending order continues)
        if (sink) *st = 1ULL << 63 | sink;
        __syncwarp();
        for (int k = lane; k < total; k += 32) {
          const unsigned long long v = sm.stage[warp][k];
          const uint32_t w = (uint32_t)v;
          const bool is_sink = (v >> 63) != 0;
          if (a.col)
            a.col[begin + k] = is_sink ? a.nS : s0 + (int64_t)(v >> 32) + a.Nc + (int64_t)(int16_t)(w & 0xFFFFu);
          if (a.count) a.count[begin + k] = is_sink ? (int32_t)w : (int32_t)(w >> 16);
        }
        __syncwarp();
      } else {   // longer rows: each lane writes its own
        const int64_t o = begin + mine;
        for (int k = 0; k < e + sp; ++k) {
          const uint32_t w = k < e ? src[(size_t)k * 32] : tail[k - e];
          if (a.col) a.col[o + k] = s + a.Nc + (int64_t)(int16_t)(w & 0xFFFFu);
          if (a.count) a.count[o + k] = (int32_t)(w >> 16);
        }
        if (sink) {
          if (a.col) a.col[o + e + sp] = a.nS;
          if (a.count) a.count[o + e + sp] = (int32_t)sink;
        }
      }
    }
    __syncthreads();
  }
}

template <typename RT>
static cudaError_t fill_t(const ExportArgs &a, const mdp_model_t *m, int obj, void *R, cudaStream_t st) {
  cudaError_t e = allow_max_smem((const void *)export_fill_kernel<RT>);
  if (e != cudaSuccess) return e;
  int per_sm = 0;
  const size_t smem = sizeof(ExportSmem<RT>);
  e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, export_fill_kernel<RT>, 32 * kXWarps, smem);
  if (e != cudaSuccess) return e;
  if (per_sm < 1) return cudaErrorInvalidConfiguration;
  const int64_t blocks = std::min<int64_t>(a.blocks, (int64_t)num_sms() * per_sm * 4);
  export_fill_kernel<RT><<<(unsigned)blocks, 32 * kXWarps, smem, st>>>(
      a, static_cast<const RT *>(m->R) + (size_t)obj * m->rows_pad, static_cast<RT *>(R));
  return cudaGetLastError();
}

cudaError_t launch_export(const mdp_model_t *m, int obj, int64_t *rowptr, int64_t *col,
                          int32_t *count, void *R, cudaStream_t st) {
  ExportArgs a{};
  a.pool = m->pool; a.slice_off = m->slice_off; a.spill = m->spill; a.spill_off = m->spill_off;
  a.slice_w = m->slice_w; a.nnz = m->nnz; a.sinkc = m->sinkc;
  a.nS = m->nS; a.Nc = m->Nc; a.n_slices = m->n_slices; a.A = m->A; a.A_pad = m->A_pad; a.spw = m->spw;
  a.blocks = (m->nS + kXState - 1) / kXState;
  a.rowptr = rowptr; a.col = col; a.count = count;
  const int64_t n = a.A * a.blocks;
  int64_t *x = nullptr;
  a.sum_act = a.blocks;
  a.sum_block = 1;
  cudaError_t e = dev_alloc((void **)&x, sizeof(int64_t) * (size_t)(n + scan_words(n)), st);
  const bool in_rowptr = e == cudaErrorMemoryAllocation;
  if (in_rowptr) {
    cudaGetLastError();   // (it is not the call's)
    a.sum_act = m->nS;
    a.sum_block = kXState;
    e = dev_alloc((void **)&x, sizeof(int64_t) * (size_t)scan_words(n), st);
  }
  if (e != cudaSuccess) return e;
  a.sums = in_rowptr ? rowptr : x;
  int64_t *tile = in_rowptr ? x : x + n;
  a.tile = tile;
  const RowptrSums scattered{rowptr, m->nS, a.blocks};
  export_lengths_kernel<<<(unsigned)std::min<int64_t>((a.blocks + 7) / 8, (int64_t)num_sms() * 8), 256, 0, st>>>(a);
  e = cudaGetLastError();
  if (e == cudaSuccess)
    e = in_rowptr ? scan_offsets(LoadWords<RowptrSums>{scattered}, n, scattered, tile, st)
                  : scan_offsets(LoadWords<Words>{{x}}, n, Words{x}, tile, st);
  if (e == cudaSuccess)
    e = m->precision == MDP_FP64_CHECK ? fill_t<double>(a, m, obj, R, st) : fill_t<float>(a, m, obj, R, st);
  dev_free(x, st);
  return e;
}

}  // namespace mdpgb
