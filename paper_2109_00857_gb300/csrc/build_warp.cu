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
// persistent CTAs, or at most a.groups_per_cta groups each (the grid then
// covers the model, so every group is taken).
template <int KT, int SPW, int MODE>
__global__ void __launch_bounds__(32 * kGroupWarps, kMinCtas<KT>) build_group_kernel(const __grid_constant__ BuildArgs a, int words,
                                                                                int share, int chunk) {
  extern __shared__ __align__(16) unsigned char gsm[];
  GroupSmem &sm = *reinterpret_cast<GroupSmem *>(gsm);
  const int NW = blockDim.x >> 5, spw = SPW > 0 ? SPW : a.spw;
  float4 *ext = reinterpret_cast<float4 *>(gsm + group_ext_offset(0, spw, NW));
  uint32_t *tabs = reinterpret_cast<uint32_t *>(gsm + group_head_bytes(0, spw, NW));
  const long long n_groups = (a.slice_end - a.slice_begin + NW - 1) / NW;
  clear_tables(tabs, words);
  warp_clear(sm);
  load_rank_tables(a, sm.rt);
  if (threadIdx.x == 0) {
    sm.next[0] = (long long)atomicAdd(&a.cnt[CNT_WORK], (unsigned long long)chunk);
    sm.trap = 0u;
  }
  __syncthreads();
  // queue index g: chunk consecutive groups; the first slice of a group, or -1
  auto first_slice = [&](long long g) { return g < n_groups ? a.slice_begin + g * NW : (int64_t)-1; };
  if (first_slice(sm.next[0]) >= 0)
    setup_slice<SPW, MODE>(a, sm, first_slice(sm.next[0]), setup_load<SPW>(a, first_slice(sm.next[0])), tabs, words,
                           share);
  __syncthreads();
  int left = chunk - 1;   // thread 0: groups of its last queue grab still to do
  for (int n = 1, par = 0;; ++n, par ^= 1) {
    const long long g = sm.next[par];
    if (g >= n_groups) break;
    long long next = n_groups;   // this CTA's share may end with this group
    if (threadIdx.x == 0 && (a.groups_per_cta == 0 || n < a.groups_per_cta)) {
      if (left > 0) {
        next = g + 1;
        --left;
      } else {
        next = (long long)atomicAdd(&a.cnt[CNT_WORK], (unsigned long long)chunk);
        left = chunk - 1;
      }
    }
    group_slices<KT, SPW, true, MODE>(a, a.slice_begin + g * NW, sm, ext, tabs, words, share, next, par ^ 1,
                                        first_slice);
    __syncthreads();
  }
  warp_flush(a, sm);
}

template <int KT, int SPW, int MODE>
static cudaError_t launch_g(const BuildArgs &a, int warps, int sms, cudaStream_t st) {
  const int nw = group_warps(warps, a.spw), words = slice_words(a.cap_bins);
  const size_t smem = group_smem_bytes(0, a.cap_bins, a.spw, nw);
  cudaError_t e = allow_max_smem((const void *)build_group_kernel<KT, SPW, MODE>);
  if (e != cudaSuccess) return e;
  int per_sm = 0;
  e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, build_group_kernel<KT, SPW, MODE>, nw * 32, smem);
  if (e != cudaSuccess) return e;
  if (per_sm < 1) return cudaErrorInvalidConfiguration;
  const int64_t groups = (a.slice_end - a.slice_begin + nw - 1) / nw;
  int64_t blocks = std::min<int64_t>((int64_t)sms * per_sm, groups);
  // groups per queue grab: at least 32 grabs a CTA, at most 8 groups (the
  // queue's one address takes about 2 ns per grab)
  int chunk = (int)std::min<int64_t>(8, std::max<int64_t>(1, groups / (32 * blocks)));
  if (a.groups_per_cta > 0) chunk = 1;
  if (a.groups_per_cta > 0)   // bounded CTAs: a grid that covers every group
    blocks = (groups + a.groups_per_cta - 1) / a.groups_per_cta;
  build_group_kernel<KT, SPW, MODE><<<(unsigned)std::max<int64_t>(blocks, 1), nw * 32, smem, st>>>(
      a, words, share_words(a.cap_bins, a.spw), chunk);
  return cudaGetLastError();
}

template <int SPW, int MODE>
static cudaError_t launch_k(const BuildArgs &a, int warps, int sms, cudaStream_t st) {
  switch (a.K) {
    case 0: return launch_g<kNoModes, 0, MODE>(a, warps, sms, st);
    case 1: return launch_g<1, SPW, MODE>(a, warps, sms, st);
    case 2: return launch_g<2, SPW, MODE>(a, warps, sms, st);
    case 3: return launch_g<3, SPW, MODE>(a, warps, sms, st);
    case 4: return launch_g<4, SPW, MODE>(a, warps, sms, st);
    case 5: return launch_g<5, SPW, MODE>(a, warps, sms, st);
    case 6: return launch_g<6, SPW, MODE>(a, warps, sms, st);
    case 7: return launch_g<7, SPW, MODE>(a, warps, sms, st);
    case 8: return launch_g<8, SPW, MODE>(a, warps, sms, st);
    default: return MODE == 1 ? launch_g<0, 0, 1>(a, warps, sms, st) : launch_g<0, 0, 2>(a, warps, sms, st);
  }
}

// Instantiations: 32 and 16 actions (one and two states per slice) with the
// one- and the two-comparison lookup and up to eight modes; fewer actions with
// the one-comparison lookup; no modes with either; everything else with runtime
// sizes.
cudaError_t launch_build_warp(const BuildArgs &a, int warps, int sms, cudaStream_t st) {
  const int mode = a.act.rank_mode;
  if (mode == 1) {
    if (a.spw == 1) return launch_k<1, 1>(a, warps, sms, st);
    if (a.spw == 2) return launch_k<2, 1>(a, warps, sms, st);
    return launch_k<0, 1>(a, warps, sms, st);
  }
  if (mode == 2) {
    if (a.spw == 1) return launch_k<1, 2>(a, warps, sms, st);
    if (a.spw == 2) return launch_k<2, 2>(a, warps, sms, st);
    return a.K == 0 ? launch_g<kNoModes, 0, 2>(a, warps, sms, st) : launch_g<0, 0, 2>(a, warps, sms, st);
  }
  return launch_g<0, 0, 3>(a, warps, sms, st);
}

}  // namespace mdpgb
