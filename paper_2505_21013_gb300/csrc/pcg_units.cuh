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
// threads; *n (zero before) receives their count, of which only the first cap are listed.
// Ascending halo rows make the exchange's loads whole runs (allocation-free solve of 32000 rows 9.4 ->
// 8.3 us per CG iteration, FP64 scene of 256 rows 7.3 -> 7.0, against the hash's order).  Every key is
// compared with every other: a few hundred rows, about a microsecond per solve.
template <int NT>
__device__ __forceinline__ void rd_rank(const int* key, int* idx, int* list, int hs, int cap, int* n) {
  for (int h = threadIdx.x; h < hs; h += NT)
    if (key[h] >= 0) {
      const int k = atomicAdd(n, 1);
      if (k < cap) list[k] = key[h];
    }
  __syncthreads();
  const int m = *n;
  if (m <= cap)
    for (int h = threadIdx.x; h < hs; h += NT)
      if (key[h] >= 0) {
        int r = 0;
        for (int k = 0; k < m; ++k) r += list[k] < key[h];
        idx[h] = r;
      }
  __syncthreads();
  if (m <= cap)
    for (int h = threadIdx.x; h < hs; h += NT)
      if (key[h] >= 0) list[idx[h]] = key[h];
  __syncthreads();
}

}  // namespace ppn
