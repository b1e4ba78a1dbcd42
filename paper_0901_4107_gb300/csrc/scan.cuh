// Exclusive scan of int counts over the whole grid: block sums, their scan by
// one CTA, then every block scans its own part from its offset.  (One CTA
// scanning 262 k counts alone took 490 us; three launches take about 12.)
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

namespace amm {

constexpr int SCAN_THREADS = 256, SCAN_PER = 8, SCAN_BLOCK = SCAN_THREADS * SCAN_PER;

// ints of scratch that exclusive_scan needs for m counts
inline int64_t scan_scratch(int64_t m) { return (m + SCAN_BLOCK - 1) / SCAN_BLOCK + 1; }

// inclusive scan of x over the CTA (NT threads); total: the CTA's sum
template <int NT>
__device__ __forceinline__ int scan_cta(int x, int& total) {
  __shared__ int ws[NT / 32];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int y = __shfl_up_sync(0xffffffffu, x, o);
    if (lane >= o) x += y;
  }
  if (lane == 31) ws[w] = x;
  __syncthreads();
  int before = 0;
  total = 0;
  for (int q = 0; q < NT / 32; q++) {
    const int s = ws[q];
    before += q < w ? s : 0;
    total += s;
  }
  __syncthreads();   // ws is reused
  return x + before;
}

static __global__ void __launch_bounds__(SCAN_THREADS) k_scan_sums(const int* count, int64_t m, int* part) {
  const int64_t b = (int64_t)blockIdx.x * SCAN_BLOCK;
  int s = 0;
#pragma unroll
  for (int q = 0; q < SCAN_PER; q++) {
    const int64_t k = b + q * SCAN_THREADS + threadIdx.x;
    s += k < m ? count[k] : 0;
  }
  int total;
  scan_cta<SCAN_THREADS>(s, total);
  if (threadIdx.x == 0) part[blockIdx.x] = total;
}

// in place: part[0..nb) to its exclusive scan, part[nb] the sum
static __global__ void __launch_bounds__(1024) k_scan_parts(int* part, int nb) {
  int run = 0;
  for (int b = 0; b < nb; b += 1024) {
    const int k = b + (int)threadIdx.x;
    const int x = k < nb ? part[k] : 0;
    int total;
    const int inc = scan_cta<1024>(x, total);
    if (k < nb) part[k] = run + inc - x;
    run += total;
  }
  if (threadIdx.x == 0) part[nb] = run;
}

static __global__ void __launch_bounds__(SCAN_THREADS) k_scan_write(const int* count, int64_t m, const int* part, int nb,
                                                                  int* start) {
  const int64_t b = (int64_t)blockIdx.x * SCAN_BLOCK;
  int run = part[blockIdx.x];
#pragma unroll 1
  for (int q = 0; q < SCAN_PER; q++) {
    const int64_t k = b + q * SCAN_THREADS + threadIdx.x;
    const int x = k < m ? count[k] : 0;
    int total;
    const int inc = scan_cta<SCAN_THREADS>(x, total);
    if (k < m) start[k] = run + inc - x;
    run += total;
  }
  if (blockIdx.x == 0 && threadIdx.x == 0) start[m] = part[nb];
}

// start[0..m] of count[0..m), m >= 1; part: scan_scratch(m) ints
inline cudaError_t exclusive_scan(const int* count, int* start, int64_t m, int* part, cudaStream_t st) {
  const int nb = (int)((m + SCAN_BLOCK - 1) / SCAN_BLOCK);
  k_scan_sums<<<nb, SCAN_THREADS, 0, st>>>(count, m, part);
  k_scan_parts<<<1, 1024, 0, st>>>(part, nb);
  k_scan_write<<<nb, SCAN_THREADS, 0, st>>>(count, m, part, nb, start);
  return cudaGetLastError();
}

}  // namespace amm
