// Exclusive scans of int64 counts (compaction offsets of the classification and of the solver's
// cell lists): exact integer sums, the same in any order.
#pragma once

#include <cuda_runtime.h>

namespace ibm {

constexpr int SCAN_BLOCK = 1024;

// inclusive scan of one value per thread of a SCAN_BLOCK-thread block; total: their sum.  Warps
// scan by shuffles and every warp scans the 32 warp totals for itself; tot: two buffers that
// consecutive calls alternate, so one barrier per call suffices.
__device__ __forceinline__ long long block_scan_incl(long long v, long long (&tot)[32], long long &total) {
  const unsigned full = 0xffffffffu;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  for (int o = 1; o < 32; o <<= 1) {
    const long long u = __shfl_up_sync(full, v, o);
    if (lane >= o) v += u;
  }
  if (lane == 31) tot[warp] = v;
  __syncthreads();
  long long w = tot[lane];
  for (int o = 1; o < 32; o <<= 1) {
    const long long u = __shfl_up_sync(full, w, o);
    if (lane >= o) w += u;
  }
  const long long before = __shfl_sync(full, w, (warp + 31) & 31);   // totals of the warps before this one
  total = __shfl_sync(full, w, 31);
  return v + (warp > 0 ? before : 0);
}

// out[0 .. n) = exclusive prefix sums of in[0 .. n), out[n] = the total; one block.  Bound by
// latency, about 1 us per SCAN_BLOCK values: one value per thread, so every load and store is
// coalesced, and the next values' load is issued before the scan of these.
static __global__ void __launch_bounds__(SCAN_BLOCK) k_block_scan(const long long *in, long long *out, int n) {
  __shared__ long long tot[2][32];
  long long run = 0;
  long long x = (int)threadIdx.x < n ? in[threadIdx.x] : 0;
  for (int b = 0, s = 0; b < n; b += SCAN_BLOCK, s ^= 1) {
    const int i = b + (int)threadIdx.x;
    const long long next = n - i > SCAN_BLOCK ? in[i + SCAN_BLOCK] : 0;
    long long total;
    const long long v = block_scan_incl(x, tot[s], total);
    if (i < n) out[i] = run + v - x;
    run += total;
    x = next;
  }
  if (threadIdx.x == 0) out[n] = run;
}

// the same in tiles: one block scans SCAN_TILE values and writes their total ...
constexpr int SCAN_PER = 4, SCAN_TILE = SCAN_BLOCK * SCAN_PER;
static __global__ void __launch_bounds__(SCAN_BLOCK) k_tile_scan(const long long *in, long long *out, int n, long long *tile) {
  __shared__ long long tot[32];
  const int b = blockIdx.x * SCAN_TILE + SCAN_PER * (int)threadIdx.x;
  long long x[SCAN_PER], sum = 0, total;
  for (int q = 0; q < SCAN_PER; ++q) {
    x[q] = b + q < n ? in[b + q] : 0;
    sum += x[q];
  }
  long long run = block_scan_incl(sum, tot, total) - sum;
  for (int q = 0; q < SCAN_PER; ++q) {
    if (b + q < n) out[b + q] = run;
    run += x[q];
  }
  if (threadIdx.x == 0) tile[blockIdx.x] = total;
}

// ... and then the tiles' offsets (tile: their scan, nt + 1 values) are added
static __global__ void __launch_bounds__(SCAN_BLOCK) k_tile_add(long long *out, int n, const long long *tile, int nt) {
  const int b = blockIdx.x * SCAN_TILE + (int)threadIdx.x;
  const long long add = tile[blockIdx.x];
  for (int q = 0; q < SCAN_PER; ++q)
    if (b + q * SCAN_BLOCK < n) out[b + q * SCAN_BLOCK] += add;
  if (blockIdx.x == 0 && threadIdx.x == 0) out[n] = tile[nt];
}

// scratch (in int64 values) that launch_scan needs for n counts
inline size_t scan_scratch(long long n) { return 2 * (size_t)((n + SCAN_TILE - 1) / SCAN_TILE) + 1; }

// Exclusive scan of n counts on st.  Up to 2 SCAN_TILE values one block takes them in at most
// 8 us; above, three launches take less (classification of twelve spheres at 512^3, about 500,000
// bins: 520 us in one block, 7 us in tiles.  The earlier scan, one contiguous chunk per thread
// and one thread adding the chunk totals, took 1917 us).
inline void launch_scan(const long long *in, long long *out, int n, long long *scratch, cudaStream_t st) {
  if (n <= 2 * SCAN_TILE) {
    k_block_scan<<<1, SCAN_BLOCK, 0, st>>>(in, out, n);
    return;
  }
  const int nt = (n + SCAN_TILE - 1) / SCAN_TILE;
  long long *sums = scratch, *offs = scratch + nt;
  k_tile_scan<<<nt, SCAN_BLOCK, 0, st>>>(in, out, n, sums);
  k_block_scan<<<1, SCAN_BLOCK, 0, st>>>(sums, offs, nt);
  k_tile_add<<<nt, SCAN_BLOCK, 0, st>>>(out, n, offs, nt);
}

}  // namespace ibm
