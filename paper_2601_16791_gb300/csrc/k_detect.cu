// k_detect.cu -- close-encounter detection and pair compaction
// (arXiv 2601.16791, Sec. 2.1.2, mce_snif listing: a pair is flagged when
// min(d0, d1, d2min) <= rc^2, rc = max(rcrit_i, rcrit_j)).
//
// One thread per target body against the big bodies of its system, staged in
// shared memory as FP32 copies of the endpoint states (with fewer than
// kDetMinScreen of them, the FP64 states too).  Two provably conservative FP32
// screens discard far pairs (mx_encounter.cuh; the first, by reach, from
// kDetMinScreen big bodies on); surviving pairs are decided in FP64 with the
// closed-form minimum of the cubic Hermite interpolant of the squared separation.
// Each target keeps its flagged big bodies (ascending) and writes them as one
// contiguous run, with one atomic per warp; runs of different targets come in
// any order.  The step groups runs as they are; callers that want the pairs
// in order sort the keys (k_sort_keys).
#include "mx_common.cuh"
#include "mx_detect_body.cuh"
#include "mx_kernels.h"

namespace mx {

template <bool FEW>
__global__ void __launch_bounds__(kThreads) k_detect(Dev d, const double* xv0, const double* xv1,
                                                     unsigned char* flags,
                                                     unsigned long long* keys, int* count,
                                                     int cap, int runs) {
  extern __shared__ __align__(16) unsigned char dsm_det[];
  detect_tile<FEW>(d, xv0, xv1, flags, keys, count, cap, runs, blockIdx.x, dsm_det);
}

// The step's (small-flag, j, i) key as an (i, j) key.
__device__ __forceinline__ unsigned long long swapped(unsigned long long k) {
  return ((k & 0xffffffffull) << 32) | ((k >> 32) & 0x7fffffffull);
}

// Ranks of up to kRankMax keys, all SMs together: a key's place is the number
// of smaller ones (the keys are distinct pairs), counted by eight lanes.  The
// n^2 compares of 5,500 keys (2,000 big bodies + 200,000 planetesimals) and the
// copy back take 44 + 6 us, where one block's bitonic sort takes 120; 1,000 keys
// 13 + 3 against 14, 16,384 keys 189 + 11 against 250.  kRankMax is the size of
// the scratch; the sort beyond it runs in global memory (16,385 keys: 960 us).
constexpr int kRankMax = kSortTmp;
__global__ void __launch_bounds__(256) k_rank_keys(const unsigned long long* keys, const int* count,
                                                   int cap, int swap_ij, unsigned long long* out) {
  const int n = min(*count, cap);
  if (n > kRankMax) return;
  const int sub = threadIdx.x & 7;
  const unsigned gmask = 0xffu << (threadIdx.x & 24);
  const int per = (gridDim.x * blockDim.x) >> 3;
  for (int i = (blockIdx.x * blockDim.x + threadIdx.x) >> 3; i < n; i += per) {
    const unsigned long long k = swap_ij ? swapped(keys[i]) : keys[i];
    int r = 0;
#pragma unroll 8
    for (int m = sub; m < n; m += 8) r += ((swap_ij ? swapped(keys[m]) : keys[m]) < k) ? 1 : 0;
    for (int o = 4; o > 0; o >>= 1) r += __shfl_xor_sync(gmask, r, o);
    if (sub == 0) out[r] = k;
  }
}

// Sorts min(*count, cap) keys ascending in one block (bitonic; shared memory
// up to kSortSmem keys, global memory beyond), or copies them back from
// `ranked`, where k_rank_keys has put them.  swap_ij turns the step's
// (small-flag, j, i) keys into (i, j) keys first.
constexpr int kSortSmem = 4096;   // 32 KB of static shared memory
__global__ void __launch_bounds__(1024) k_sort_keys(unsigned long long* keys, const int* count,
                                                    int cap, int swap_ij,
                                                    const unsigned long long* ranked) {
  __shared__ unsigned long long sk[kSortSmem];
  const int n = min(*count, cap);
  if (n <= 0) return;
  if (ranked && n <= kRankMax) {
    for (int i = threadIdx.x; i < n; i += blockDim.x) keys[i] = ranked[i];
    return;
  }
  if (swap_ij) {
    for (int i = threadIdx.x; i < n; i += blockDim.x) keys[i] = swapped(keys[i]);
    __syncthreads();
  }
  int P2 = 1;
  while (P2 < n) P2 <<= 1;
  const bool in_smem = P2 <= kSortSmem;
  unsigned long long* a = in_smem ? sk : keys;
  if (in_smem) {
    for (int i = threadIdx.x; i < P2; i += blockDim.x) sk[i] = (i < n) ? keys[i] : ~0ull;
  } else {
    for (int i = n + threadIdx.x; i < P2; i += blockDim.x) keys[i] = ~0ull;
  }
  __syncthreads();
  for (int k = 2; k <= P2; k <<= 1) {
    for (int jj = k >> 1; jj > 0; jj >>= 1) {
      for (int i = threadIdx.x; i < P2; i += blockDim.x) {
        const int ixj = i ^ jj;
        if (ixj > i) {
          const unsigned long long x = a[i], y = a[ixj];
          const bool up = (i & k) == 0;
          if ((x > y) == up) {
            a[i] = y;
            a[ixj] = x;
          }
        }
      }
      __syncthreads();
    }
  }
  if (in_smem)
    for (int i = threadIdx.x; i < n; i += blockDim.x) keys[i] = sk[i];
}

// (i, j) int pairs from sorted (i << 32 | j) keys.
__global__ void k_keys_to_pairs(const unsigned long long* keys, const int* count, int cap,
                                int* pairs) {
  const int n = min(*count, cap);
  for (int p = blockIdx.x * blockDim.x + threadIdx.x; p < n; p += gridDim.x * blockDim.x) {
    const unsigned long long k = keys[p];
    pairs[2 * p] = (int)(k >> 32);
    pairs[2 * p + 1] = (int)(k & 0xffffffffull);
  }
}

void launch_keys_to_pairs(const unsigned long long* keys, const int* count, int cap, int* pairs,
                          cudaStream_t st) {
  k_keys_to_pairs<<<64, 256, 0, st>>>(keys, count, cap, pairs);
}

void launch_detect(const Dev& d, const double* xv0, const double* xv1, unsigned char* flags,
                   unsigned long long* keys, int* count, int cap, int runs, cudaStream_t st) {
  const bool few = det_few(d.big_max);
  const size_t sm = det_smem_bytes(det_chunk(d.tile, d.big_max), few);
  auto* k = few ? k_detect<true> : k_detect<false>;
  k<<<d.ntiles, d.tile, sm, st>>>(d, xv0, xv1, flags, keys, count, cap, runs);
}

void launch_sort_keys(unsigned long long* keys, const int* count, int cap, int swap_ij,
                      unsigned long long* tmp, cudaStream_t st) {
  if (tmp) k_rank_keys<<<256, 256, 0, st>>>(keys, count, cap, swap_ij, tmp);
  k_sort_keys<<<1, 1024, 0, st>>>(keys, count, cap, swap_ij, tmp);
}

// The kernels of a step share one shared-memory carveout (the largest), so
// the SMs are not reconfigured between consecutive kernels with different
// shared-memory needs (measured: ~12 us bubbles before k_detect and the kick).
void configure_detect() {
  for (auto* k : {k_detect<true>, k_detect<false>})
    cudaFuncSetAttribute(k, cudaFuncAttributePreferredSharedMemoryCarveout,
                         cudaSharedmemCarveoutMaxShared);
}

}  // namespace mx
