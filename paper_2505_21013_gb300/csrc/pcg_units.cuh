// Helpers of the PCG kernels whose CTAs own 32-row units (pcg_rd.cu, pcg_su.cu): the split of
// the rows, and the halo of a CTA found on the device.
#pragma once

#include <cuda_runtime.h>

namespace ppn {

// the posts [rd_post0(b), rd_post0(b + 1)) of CTA b
__host__ __device__ inline int rd_post0(int b, int n_posts, int grid) { return (int)(((long long)b * n_posts) / grid); }

// smallest power of two >= 2 n (at least 64)
__host__ __device__ inline int rd_hash_size(int n) {
  int h = 64;
  while (h < 2 * n) h *= 2;
  return h;
}
__device__ __forceinline__ unsigned rd_hash(int j) { return (unsigned)j * 2654435761u >> 8; }
// inserts j into the table of hs keys (-1: free); false when it is full
__device__ __forceinline__ bool rd_insert(int* key, int hs, int j) {
  unsigned h = rd_hash(j) & (unsigned)(hs - 1);
  for (int n = 0; n < hs; ++n, h = (h + 1) & (unsigned)(hs - 1)) {
    const int k = atomicCAS(&key[h], -1, j);
    if (k == -1 || k == j) return true;
  }
  return false;
}

// The inserted keys' ranks (ascending) as their indices, and the sorted list, by the whole CTA of NT
// threads; *n (zero before) receives their count, of which only the first cap are listed (idx: hs >= 2 cap
// entries).  Ascending halo rows make the exchange's loads whole runs (allocation-free solve of 32000 rows
// 9.4 -> 8.3 us per CG iteration, FP64 scene of 256 rows 7.3 -> 7.0, against the hash's order).
// A few keys are compared all with all (125 FP64 vertices 584 us a step, 588 sorted; 756 mixed ones 1638
// and 1687).  More of them, up to 4096 on a mesh without an order, go through a bitonic sort and a search
// per key.  One solve of one iteration, all pairs -> sorted, by the halo rows of a CTA: 295 84 -> 83 us,
// 422 88 -> 83, 1678 225 -> 112, 3378 627 -> 156.
constexpr int RD_RANK_MAX = 256;
template <int NT>
__device__ __forceinline__ void rd_rank(const int* key, int* idx, int* list, int hs, int cap, int* n) {
  static_assert(RD_RANK_MAX <= NT, "a thread per key");
  for (int h = threadIdx.x; h < hs; h += NT)
    if (key[h] >= 0) {
      const int k = atomicAdd(n, 1);
      if (k < cap) idx[k] = key[h];
    }
  __syncthreads();
  const int m = *n;
  if (m > cap) return;  // (the caller refuses it)
  if (m <= RD_RANK_MAX) {
    if ((int)threadIdx.x < m) list[threadIdx.x] = idx[threadIdx.x];
    __syncthreads();
    for (int h = threadIdx.x; h < hs; h += NT)
      if (key[h] >= 0) {
        int r = 0;
        const int j = key[h];
#pragma unroll 8
        for (int k = 0; k < m; ++k) r += list[k] < j;
        idx[h] = r;
      }
    __syncthreads();
    for (int h = threadIdx.x; h < hs; h += NT)
      if (key[h] >= 0) list[idx[h]] = key[h];
    __syncthreads();
    return;
  }
  int p = 64;
  while (p < m) p *= 2;
  for (int k = m + threadIdx.x; k < p; k += NT) idx[k] = 0x7fffffff;
  __syncthreads();
  for (int size = 2; size <= p; size *= 2)
    for (int stride = size / 2; stride > 0; stride /= 2) {
      for (int i = threadIdx.x; i < p / 2; i += NT) {
        const int a = 2 * i - (i & (stride - 1)), b = a + stride;
        const int x = idx[a], y = idx[b];
        if ((x > y) == ((a & size) == 0)) {
          idx[a] = y;
          idx[b] = x;
        }
      }
      // the pairs of a warp's 32 threads lie in 64 entries of their own once stride <= 32
      if (stride > 32 || (stride == 1 && size >= 64))
        __syncthreads();
      else
        __syncwarp();
    }
  for (int k = threadIdx.x; k < m; k += NT) list[k] = idx[k];
  __syncthreads();
  for (int h = threadIdx.x; h < hs; h += NT)
    if (key[h] >= 0) {
      int lo = 0;  // the last entry that is not above the key
      for (int o = p / 2; o > 0; o /= 2)
        if (lo + o < m && list[lo + o] <= key[h]) lo += o;
      idx[h] = lo;
    }
  __syncthreads();
}

}  // namespace ppn
