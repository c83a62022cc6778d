// build_warp.cu -- production FP32 MDP build, the group kernel (single-model
// kernel and launchers; the algorithm is in build_warp.cuh, the batched kernel
// in build_warp_batch.cu).
#include <algorithm>

#include "build_warp.cuh"

namespace mdpgb {

// Per layer and mode the mean and variance of a caller's coefficient table
// (the library's own draws have mean 0 and variance sigma^2): what the count
// windows are predicted from.  One block per layer.
__global__ void coeff_moments_kernel(const float *__restrict__ Y, int N, int K, float2 *__restrict__ mom) {
  __shared__ float s1[8], s2[8];
  const float *Yt = Y + (size_t)blockIdx.x * N * K;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  for (int k = 0; k < K; ++k) {
    float a = 0.f, b = 0.f;
    for (int w = threadIdx.x; w < N; w += blockDim.x) {
      const float y = Yt[(size_t)w * K + k];
      a += y;
      b = fmaf(y, y, b);
    }
    for (int off = 16; off >= 1; off >>= 1) {
      a += __shfl_xor_sync(0xffffffffu, a, off);
      b += __shfl_xor_sync(0xffffffffu, b, off);
    }
    if (lane == 0) {
      s1[warp] = a;
      s2[warp] = b;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
      for (int i = 1; i < (int)(blockDim.x >> 5); ++i) {
        a += s1[i];
        b += s2[i];
      }
      const float m = a / (float)N;
      mom[(size_t)blockIdx.x * K + k] = make_float2(m, fmaxf(b / (float)N - m * m, 0.f));
    }
    __syncthreads();
  }
}

cudaError_t launch_coeff_moments(const float *Y, int nt, int N, int K, float2 *mom, cudaStream_t st) {
  coeff_moments_kernel<<<nt, 256, 0, st>>>(Y, N, K, mom);
  return cudaGetLastError();
}

// Single model: CTAs pull groups of slices from the model's work queue --
// persistent CTAs, or at most a.slices_per_warp groups each (the grid then
// covers the model, so every group is taken).
template <int KT, int SPW, bool DENSE>
__global__ void __launch_bounds__(32 * kGroupWarps, KT == 0 ? 2 : 3) build_group_kernel(const __grid_constant__ BuildArgs a, int words) {
  extern __shared__ __align__(16) unsigned char gsm[];
  GroupSmem &sm = *reinterpret_cast<GroupSmem *>(gsm);
  float4 *ext = reinterpret_cast<float4 *>(gsm + ((sizeof(GroupSmem) + 15) & ~(size_t)15));
  uint32_t *tabs = table_memory(gsm, sizeof(GroupSmem), &words, SPW > 0 ? SPW : a.spw);
  const int NW = blockDim.x >> 5;
  const long long n_groups = (a.slice_end - a.slice_begin + NW - 1) / NW;
  clear_tables(tabs, words);
  warp_clear(sm);
  load_rank_tables(a, sm.rt);
  if (threadIdx.x == 0) sm.next[0] = (long long)atomicAdd(&a.cnt[CNT_WORK], 1ULL);
  __syncthreads();
  for (int n = 1, par = 0;; ++n, par ^= 1) {
    const long long g = sm.next[par];
    if (g >= n_groups) break;
    long long next = n_groups;   // this CTA's share may end with this group
    if (threadIdx.x == 0 && (a.slices_per_warp == 0 || n < a.slices_per_warp))
      next = (long long)atomicAdd(&a.cnt[CNT_WORK], 1ULL);
    group_slices<KT, SPW, true, DENSE>(a, a.slice_begin + g * NW, sm, ext, tabs, words, next, par ^ 1);
    __syncthreads();
  }
  warp_flush(a, sm);
}

template <int KT, int SPW, bool DENSE = false>
static cudaError_t launch_g(const BuildArgs &a, int warps, int sms, cudaStream_t st) {
  const int nw = group_warps(warps, a.spw), words = table_words(a.cap_bins, a.spw);
  int reserved = 0;
  cudaError_t e = reserved_smem(&reserved);
  if (e != cudaSuccess) return e;
  const size_t smem = group_smem_bytes(sizeof(GroupSmem), reserved, a.cap_bins, a.spw, nw);
  e = allow_max_smem((const void *)build_group_kernel<KT, SPW, DENSE>);
  if (e != cudaSuccess) return e;
  int per_sm = 0;
  e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, build_group_kernel<KT, SPW, DENSE>, nw * 32, smem);
  if (e != cudaSuccess) return e;
  if (per_sm < 1) return cudaErrorInvalidConfiguration;
  const int64_t groups = (a.slice_end - a.slice_begin + nw - 1) / nw;
  int64_t blocks = std::min<int64_t>((int64_t)sms * per_sm, groups);
  if (a.slices_per_warp > 0)   // bounded CTAs: a grid that covers every group
    blocks = (groups + a.slices_per_warp - 1) / a.slices_per_warp;
  build_group_kernel<KT, SPW, DENSE><<<(unsigned)std::max<int64_t>(blocks, 1), nw * 32, smem, st>>>(a, words);
  return cudaGetLastError();
}

template <int SPW>
static cudaError_t launch_spw(const BuildArgs &a, int warps, int sms, cudaStream_t st) {
  switch (a.K) {
    case 1: return launch_g<1, SPW>(a, warps, sms, st);
    case 2: return launch_g<2, SPW>(a, warps, sms, st);
    case 3: return launch_g<3, SPW>(a, warps, sms, st);
    case 4: return launch_g<4, SPW>(a, warps, sms, st);
    case 5: return launch_g<5, SPW>(a, warps, sms, st);
    case 6: return launch_g<6, SPW>(a, warps, sms, st);
    case 7: return launch_g<7, SPW>(a, warps, sms, st);
    case 8: return launch_g<8, SPW>(a, warps, sms, st);
    default: return launch_g<0, SPW>(a, warps, sms, st);
  }
}

cudaError_t launch_build_warp(const BuildArgs &a, int warps, int sms, cudaStream_t st) {
  if (a.act.Mx > 2 || a.act.My > 2) return launch_g<0, 0, true>(a, warps, sms, st);   // dense thresholds
  if (a.spw == 1) return launch_spw<1>(a, warps, sms, st);
  if (a.spw == 2) return launch_spw<2>(a, warps, sms, st);
  return launch_spw<0>(a, warps, sms, st);
}

}  // namespace mdpgb
