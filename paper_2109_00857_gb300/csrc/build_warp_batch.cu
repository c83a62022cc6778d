// build_warp_batch.cu -- the FP32 group build over many models in one
// persistent launch (mdp_batch_*); the algorithm is in build_warp.cuh.
#include "build_warp.cuh"

namespace mdpgb {

// Many models: persistent CTAs pull global group indices; g -> (model m,
// group g - prefix[m]) by binary search over the prefix sums.  The models of
// one launch share the mode count (KT > 0; KT == 0: runtime, up to
// kMaxModes), the states per slice (SPW; 0: runtime, but one value per launch)
// and the density of their thresholds.
struct BatchSmem {
  GroupSmem g;
  BuildArgs a;   // the current model's arguments
};

template <int KT, int SPW, bool DENSE>
__global__ void __launch_bounds__(32 * kGroupWarps, KT == 0 ? 2 : 3)
    build_group_batch_kernel(const BuildArgs *__restrict__ items, const int64_t *__restrict__ prefix, int n,
                             unsigned long long *work, int words, int spw) {
  extern __shared__ __align__(16) unsigned char gsm[];
  BatchSmem &sm = *reinterpret_cast<BatchSmem *>(gsm);
  float4 *ext = reinterpret_cast<float4 *>(gsm + ((sizeof(BatchSmem) + 15) & ~(size_t)15));
  uint32_t *tabs = table_memory(gsm, sizeof(BatchSmem), &words, SPW > 0 ? SPW : spw);
  const int NW = blockDim.x >> 5;
  const int64_t total = prefix[n];
  clear_tables(tabs, words);
  warp_clear(sm.g);
  if (threadIdx.x == 0) sm.g.next[0] = (long long)atomicAdd(work, 1ULL);
  __syncthreads();
  int cur = -1;
  for (int par = 0;; par ^= 1) {
    const long long g = sm.g.next[par];
    if (g >= total) break;
    long long next = total;
    if (threadIdx.x == 0) next = (long long)atomicAdd(work, 1ULL);
    int lo = 0, hi = n - 1;   // last m with prefix[m] <= g
    while (lo < hi) {
      const int mid = (lo + hi + 1) >> 1;
      if (prefix[mid] <= g) lo = mid; else hi = mid - 1;
    }
    if (lo != cur) {
      if (cur >= 0) warp_flush(items[cur], sm.g);
      cur = lo;
      static_assert(sizeof(BuildArgs) % 8 == 0, "copied as 64-bit words");
      const uint64_t *src = reinterpret_cast<const uint64_t *>(items + lo);
      uint64_t *dst = reinterpret_cast<uint64_t *>(&sm.a);
      for (int i = threadIdx.x; i < (int)(sizeof(BuildArgs) / 8); i += blockDim.x) dst[i] = src[i];
      load_rank_tables(items[lo], sm.g.rt);
      __syncthreads();
    }
    group_slices<KT, SPW, false, DENSE>(sm.a, (g - prefix[lo]) * NW, sm.g, ext, tabs, words, next, par ^ 1);
    __syncthreads();
  }
  if (cur >= 0) warp_flush(items[cur], sm.g);
}

template <int KT, int SPW, bool DENSE = false>
static cudaError_t launch_gb(const BuildArgs *items_d, const int64_t *prefix_d, int n, unsigned long long *work_d,
                             int cap, int spw, cudaStream_t st) {
  const int nw = batch_group_slices(spw), words = table_words(cap, spw);
  int reserved = 0;
  cudaError_t e = reserved_smem(&reserved);
  if (e != cudaSuccess) return e;
  const size_t smem = group_smem_bytes(sizeof(BatchSmem), reserved, cap, spw, nw);
  e = allow_max_smem((const void *)build_group_batch_kernel<KT, SPW, DENSE>);
  if (e != cudaSuccess) return e;
  int per_sm = 0;
  e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, build_group_batch_kernel<KT, SPW, DENSE>, nw * 32, smem);
  if (e != cudaSuccess) return e;
  if (per_sm < 1) return cudaErrorInvalidConfiguration;
  build_group_batch_kernel<KT, SPW, DENSE>
      <<<num_sms() * per_sm, nw * 32, smem, st>>>(items_d, prefix_d, n, work_d, words, spw);
  return cudaGetLastError();
}

template <int SPW>
static cudaError_t launch_gb_k(const BuildArgs *items_d, const int64_t *prefix_d, int n, unsigned long long *work_d,
                               int cap_bins, int K, int spw, cudaStream_t st) {
  switch (K) {
    case 1: return launch_gb<1, SPW>(items_d, prefix_d, n, work_d, cap_bins, spw, st);
    case 2: return launch_gb<2, SPW>(items_d, prefix_d, n, work_d, cap_bins, spw, st);
    case 3: return launch_gb<3, SPW>(items_d, prefix_d, n, work_d, cap_bins, spw, st);
    case 4: return launch_gb<4, SPW>(items_d, prefix_d, n, work_d, cap_bins, spw, st);
    case 5: return launch_gb<5, SPW>(items_d, prefix_d, n, work_d, cap_bins, spw, st);
    case 6: return launch_gb<6, SPW>(items_d, prefix_d, n, work_d, cap_bins, spw, st);
    case 7: return launch_gb<7, SPW>(items_d, prefix_d, n, work_d, cap_bins, spw, st);
    case 8: return launch_gb<8, SPW>(items_d, prefix_d, n, work_d, cap_bins, spw, st);
    default: return launch_gb<0, SPW>(items_d, prefix_d, n, work_d, cap_bins, spw, st);
  }
}

int batch_group_slices(int spw) { return group_warps(kGroupWarps, spw); }

cudaError_t launch_build_warp_batch(const BuildArgs *items_d, const int64_t *prefix_d, int n,
                                    unsigned long long *work_d, int cap_bins, int K, int spw, bool dense,
                                    cudaStream_t st) {
  if (dense) return launch_gb<0, 0, true>(items_d, prefix_d, n, work_d, cap_bins, spw, st);
  if (spw == 1) return launch_gb_k<1>(items_d, prefix_d, n, work_d, cap_bins, K, spw, st);
  if (spw == 2) return launch_gb_k<2>(items_d, prefix_d, n, work_d, cap_bins, K, spw, st);
  return launch_gb_k<0>(items_d, prefix_d, n, work_d, cap_bins, K, spw, st);
}

}  // namespace mdpgb
