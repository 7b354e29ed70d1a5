// The units of work of many entries (tiles, column groups) as one list, of
// which every block of a grid takes an equal run.  Dealing out blocks by entry
// instead gives each entry the same number: the largest entry's blocks then
// run alone at the end, and those of entries without work still start.
#pragma once
#include <cstdint>

namespace peps {

// `mine` is the unit count of entry threadIdx.x of the first 256, count(j) any
// entry's, body(j, a, b) does units a .. b of entry j.  At least 256 threads;
// called and left by the whole block.
template <class Count, class Body>
__device__ __forceinline__ void for_block_share(int n, int64_t mine, Count count, Body body) {
  __shared__ int64_t ends[256], wsum[8];   // where each entry's units end in the list
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
  int64_t total = 0;
  if (n > 256) {
    int64_t v = tid < 256 ? mine : 0;
    if (tid < 256)
      for (int j = tid + 256; j < n; j += 256) v += count(j);
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    if (lane == 0 && w < 8) wsum[w] = v;
    __syncthreads();
    for (int i = 0; i < 8; ++i) total += wsum[i];
  }
  int64_t before = 0;   // units of the entries before the 256 looked at
  for (int c0 = 0; c0 < n; c0 += 256) {
    const int nc = n - c0 < 256 ? n - c0 : 256;
    int64_t v = 0;
    if (tid < nc) v = c0 == 0 ? mine : count(c0 + tid);
    for (int o = 1; o < 32; o <<= 1) {
      const int64_t x = __shfl_up_sync(0xffffffffu, v, o);
      if (lane >= o) v += x;
    }
    __syncthreads();   // wsum and ends of the 256 before are read
    if (lane == 31 && w < 8) wsum[w] = v;
    __syncthreads();
    if (tid < 256) {
      v += before;
      for (int i = 0; i < w; ++i) v += wsum[i];
      ends[tid] = v;
    }
    __syncthreads();
    if (n <= 256) total = ends[255];
    const int64_t lo = total * blockIdx.x / gridDim.x, hi = total * (blockIdx.x + 1) / gridDim.x;
    if (before >= hi || lo >= hi) return;
    int first = 0, last = nc;   // the first entry that ends after lo
    while (first < last) {
      const int mid = (first + last) >> 1;
      if (ends[mid] > lo) last = mid;
      else first = mid + 1;
    }
    for (int j = first; j < nc; ++j) {
      const int64_t begin = j > 0 ? ends[j - 1] : before;
      if (begin >= hi) break;
      const int64_t a = lo > begin ? lo : begin, b = hi < ends[j] ? hi : ends[j];
      if (a < b) body(c0 + j, (int)(a - begin), (int)(b - begin));
    }
    before = ends[nc - 1];
  }
}

}  // namespace peps
