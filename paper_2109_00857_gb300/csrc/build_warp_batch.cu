// build_warp_batch.cu -- the FP32 group build over many models in one
// persistent launch (mdp_batch_*); the algorithm is in build_warp.cuh.
#include "build_warp.cuh"

namespace mdpgb {

// The current model's arguments in shared memory: BuildArgs up to the action
// constants that the group build reads.  The whole of it would leave four CTAs
// an SM instead of five (16 uneven models: 38.3 ms of kernels; 42 ms so).
static_assert(sizeof(BuildArgs) % 16 == 0, "an array of them is copied as 16-byte vectors");
constexpr uint32_t kArgsBytes = (uint32_t)((offsetof(BuildArgs, act) + offsetof(ActionTable, dxl) + 15) & ~(size_t)15);

// Many models: persistent CTAs pull global group indices, a few consecutive
// ones at a time; g -> (model m, group g - prefix[m]), by binary search over
// the prefix sums when g leaves the current model.  The models of one launch
// share the mode count (KT > 0; KT == 0: runtime, up to kMaxModes), the states
// per slice (SPW; 0: runtime, but one value per launch) and the rank lookup's
// mode.
template <int KT, int SPW, int MODE>
__global__ void __launch_bounds__(32 * kGroupWarps, kMinCtas<KT>)
    build_group_batch_kernel(const BuildArgs *__restrict__ items, const int64_t *__restrict__ prefix, int n,
                             unsigned long long *work, int words, int share, int spw) {
  extern __shared__ __align__(16) unsigned char gsm[];
  const BuildArgs &a = *reinterpret_cast<const BuildArgs *>(gsm);
  GroupSmem &sm = *reinterpret_cast<GroupSmem *>(gsm + kArgsBytes);
  const int NW = blockDim.x >> 5, states = SPW > 0 ? SPW : spw;
  float4 *ext = reinterpret_cast<float4 *>(gsm + group_ext_offset(kArgsBytes, states, NW));
  uint32_t *tabs = reinterpret_cast<uint32_t *>(gsm + group_head_bytes(kArgsBytes, states, NW));
  const int64_t total = prefix[n];
  // groups per queue grab (see launch_g)
  const unsigned long long chunk = (unsigned long long)max((int64_t)1, min((int64_t)8, total / (16 * (int64_t)gridDim.x)));
  clear_tables(tabs, words);
  warp_clear(sm);
  if (threadIdx.x == 0) {
    sm.next[0] = (long long)atomicAdd(work, chunk);
    sm.trap = 0u;
  }
  __syncthreads();
  // the model of group g: last m with prefix[m] <= g; [lo, hi) the current one's groups
  auto model_of = [&](long long g) {
    int x = 0, y = n - 1;
    while (x < y) {
      const int mid = (x + y + 1) >> 1;
      if (prefix[mid] <= g) x = mid; else y = mid - 1;
    }
    return x;
  };
  int cur = -1, left = (int)chunk - 1;   // left: groups of the last grab still to do (thread 0)
  int64_t lo = 0, hi = 0;
  for (int par = 0;; par ^= 1) {
    const long long g = sm.next[par];
    if (g >= total) break;
    if (g < lo || g >= hi) {
      if (cur >= 0) warp_flush(items[cur], sm);
      cur = model_of(g);
      lo = prefix[cur];
      hi = prefix[cur + 1];
      const uint4 *src = reinterpret_cast<const uint4 *>(items + cur);
      uint4 *dst = reinterpret_cast<uint4 *>(gsm);
      for (int i = threadIdx.x; i < (int)(kArgsBytes / 16); i += blockDim.x) dst[i] = src[i];
      load_rank_tables(items[cur], sm.rt);
      __syncthreads();
      setup_slice<SPW, MODE>(a, sm, (g - lo) * NW, setup_load<SPW>(a, (g - lo) * NW), tabs, words, share);
      __syncthreads();
    }
    long long next = total;
    if (threadIdx.x == 0) {
      if (left > 0) {
        next = g + 1;
        --left;
      } else {
        next = (long long)atomicAdd(work, chunk);
        left = (int)chunk - 1;
      }
    }
    group_slices<KT, SPW, false, MODE>(a, (g - lo) * NW, sm, ext, tabs, words, share, next, par ^ 1,
                                       [&](long long g1) {   // (another model's group is set up after the switch)
                                         return g1 >= lo && g1 < hi ? (int64_t)(g1 - lo) * NW : (int64_t)-1;
                                       });
    __syncthreads();
  }
  if (cur >= 0) warp_flush(items[cur], sm);
}

template <int KT, int SPW, int MODE>
static cudaError_t launch_gb(const BuildArgs *items_d, const int64_t *prefix_d, int n, unsigned long long *work_d,
                             int cap, int spw, cudaStream_t st) {
  const int nw = batch_group_slices(spw), words = slice_words(cap);
  const size_t smem = group_smem_bytes(kArgsBytes, cap, spw, nw);
  cudaError_t e = allow_max_smem((const void *)build_group_batch_kernel<KT, SPW, MODE>);
  if (e != cudaSuccess) return e;
  int per_sm = 0;
  e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, build_group_batch_kernel<KT, SPW, MODE>, nw * 32, smem);
  if (e != cudaSuccess) return e;
  if (per_sm < 1) return cudaErrorInvalidConfiguration;
  build_group_batch_kernel<KT, SPW, MODE>
      <<<num_sms() * per_sm, nw * 32, smem, st>>>(items_d, prefix_d, n, work_d, words, share_words(cap, spw), spw);
  return cudaGetLastError();
}

template <int SPW, int MODE>
static cudaError_t launch_gb_k(const BuildArgs *items_d, const int64_t *prefix_d, int n, unsigned long long *work_d,
                               int cap_bins, int K, int spw, cudaStream_t st) {
  switch (K) {
    case 0: return launch_gb<kNoModes, 0, MODE>(items_d, prefix_d, n, work_d, cap_bins, spw, st);
    case 1: return launch_gb<1, SPW, MODE>(items_d, prefix_d, n, work_d, cap_bins, spw, st);
    case 2: return launch_gb<2, SPW, MODE>(items_d, prefix_d, n, work_d, cap_bins, spw, st);
    case 3: return launch_gb<3, SPW, MODE>(items_d, prefix_d, n, work_d, cap_bins, spw, st);
    case 4: return launch_gb<4, SPW, MODE>(items_d, prefix_d, n, work_d, cap_bins, spw, st);
    case 5: return launch_gb<5, SPW, MODE>(items_d, prefix_d, n, work_d, cap_bins, spw, st);
    case 6: return launch_gb<6, SPW, MODE>(items_d, prefix_d, n, work_d, cap_bins, spw, st);
    case 7: return launch_gb<7, SPW, MODE>(items_d, prefix_d, n, work_d, cap_bins, spw, st);
    case 8: return launch_gb<8, SPW, MODE>(items_d, prefix_d, n, work_d, cap_bins, spw, st);
    default: return MODE == 1 ? launch_gb<0, 0, 1>(items_d, prefix_d, n, work_d, cap_bins, spw, st)
                              : launch_gb<0, 0, 2>(items_d, prefix_d, n, work_d, cap_bins, spw, st);
  }
}

int batch_group_slices(int spw) { return group_warps(kGroupWarps, spw); }

// (the single-model kernel's instantiations)
cudaError_t launch_build_warp_batch(const BuildArgs *items_d, const int64_t *prefix_d, int n,
                                    unsigned long long *work_d, int cap_bins, int K, int spw, int rank_mode,
                                    cudaStream_t st) {
  if (rank_mode == 1) {
    if (spw == 1) return launch_gb_k<1, 1>(items_d, prefix_d, n, work_d, cap_bins, K, spw, st);
    if (spw == 2) return launch_gb_k<2, 1>(items_d, prefix_d, n, work_d, cap_bins, K, spw, st);
    return launch_gb_k<0, 1>(items_d, prefix_d, n, work_d, cap_bins, K, spw, st);
  }
  if (rank_mode == 2) {
    if (spw == 1) return launch_gb_k<1, 2>(items_d, prefix_d, n, work_d, cap_bins, K, spw, st);
    if (spw == 2) return launch_gb_k<2, 2>(items_d, prefix_d, n, work_d, cap_bins, K, spw, st);
    return K == 0 ? launch_gb<kNoModes, 0, 2>(items_d, prefix_d, n, work_d, cap_bins, spw, st)
                  : launch_gb<0, 0, 2>(items_d, prefix_d, n, work_d, cap_bins, spw, st);
  }
  return launch_gb<0, 0, 3>(items_d, prefix_d, n, work_d, cap_bins, spw, st);
}

}  // namespace mdpgb
