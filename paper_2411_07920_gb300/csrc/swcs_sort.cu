// Determinants ordered by bitstring for the copy-out: a least-significant-digit
// radix sort of (bitstring, FP64 value) pairs, 8 bits a pass over the n_so bits
// that a determinant can have set.
//
// A pass is three kernels: digit counts per tile of 4,096 pairs, their scan
// (digit-major, so that a tile's first place of a digit follows the lower
// digits of all tiles and the same digit of the tiles before), and the stable
// scatter.  Inside a tile each warp owns 512 consecutive pairs: it counts its
// digits, the warps' counts are scanned per digit, and the warp places its
// pairs 32 at a time in order, equal digits ranked by a match over the warp.
// Bound by the launches up to 10^5 pairs (0.1 ms at 40 spin-orbitals; std::sort
// on the host took 5.5 ms of the call), by memory above.
#include <algorithm>
#include <cstdint>
#include <cuda_runtime.h>

#include "swcs_kernels.h"

namespace swcs {

namespace {

constexpr int kSortThreads = 256, kSortWarps = kSortThreads / 32;
constexpr int kSortTile = 4096, kSortPerWarp = kSortTile / kSortWarps;  // 512 pairs, 16 rounds of 32

__global__ void __launch_bounds__(kSortThreads) sort_count_kernel(const uint64_t* keys, int64_t n, int shift,
                                                                  uint32_t* counts, int tiles) {
  __shared__ unsigned h[256];
  h[threadIdx.x] = 0;
  __syncthreads();
  const int64_t b = (int64_t)blockIdx.x * kSortTile, e = min(n, b + kSortTile);
  for (int64_t i = b + threadIdx.x; i < e; i += kSortThreads) atomicAdd(&h[(keys[i] >> shift) & 255u], 1u);
  __syncthreads();
  counts[(size_t)threadIdx.x * tiles + blockIdx.x] = h[threadIdx.x];
}

// Exclusive scan of 256 * tiles counts in place, one CTA.
__global__ void __launch_bounds__(1024) sort_scan_kernel(uint32_t* counts, int64_t m) {
  __shared__ unsigned sums[32];
  __shared__ unsigned carry;
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  if (threadIdx.x == 0) carry = 0;
  __syncthreads();
  for (int64_t b = 0; b < m; b += 4096) {
    const int64_t i = b + 4 * (int64_t)threadIdx.x;
    unsigned v[4], loc = 0;
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      v[q] = i + q < m ? counts[i + q] : 0u;
      loc += v[q];
    }
    unsigned inc = loc;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const unsigned x = __shfl_up_sync(0xffffffffu, inc, o);
      if (lane >= o) inc += x;
    }
    if (lane == 31) sums[wid] = inc;
    __syncthreads();
    unsigned run = carry + inc - loc;
    for (int w = 0; w < wid; ++w) run += sums[w];
#pragma unroll
    for (int q = 0; q < 4; ++q)
      if (i + q < m) {
        counts[i + q] = run;
        run += v[q];
      }
    __syncthreads();
    if (threadIdx.x == 1023) carry = run;
    __syncthreads();
  }
}

__global__ void __launch_bounds__(kSortThreads) sort_scatter_kernel(const uint64_t* keys, const double* vals, int64_t n,
                                                                    int shift, const uint32_t* first, int tiles,
                                                                    uint64_t* out_keys, double* out_vals) {
  __shared__ unsigned h[kSortWarps][256];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  for (int w = 0; w < kSortWarps; ++w) h[w][threadIdx.x] = 0;
  __syncthreads();
  const int64_t b = (int64_t)blockIdx.x * kSortTile + (int64_t)warp * kSortPerWarp;
  for (int r = 0; r < kSortPerWarp; r += 32) {
    const int64_t i = b + r + lane;
    if (i < n) atomicAdd(&h[warp][(keys[i] >> shift) & 255u], 1u);
  }
  __syncthreads();
  {  // a digit per thread: where each warp's pairs of that digit begin
    unsigned run = first[(size_t)threadIdx.x * tiles + blockIdx.x];
    for (int w = 0; w < kSortWarps; ++w) {
      const unsigned c = h[w][threadIdx.x];
      h[w][threadIdx.x] = run;
      run += c;
    }
  }
  __syncthreads();
  for (int r = 0; r < kSortPerWarp; r += 32) {
    const int64_t i = b + r + lane;
    const bool live = i < n;
    const uint64_t k = live ? keys[i] : 0ull;
    const unsigned d = live ? (unsigned)(k >> shift) & 255u : 256u;
    const unsigned same = __match_any_sync(0xffffffffu, d);
    const unsigned rank = __popc(same & ((1u << lane) - 1u));
    unsigned at = 0;
    if (live) at = h[warp][d] + rank;
    __syncwarp();
    if (live && rank == 0) h[warp][d] += __popc(same);
    __syncwarp();
    if (live) {
      out_keys[at] = k;
      out_vals[at] = vals[i];
    }
  }
}

}  // namespace

size_t sort_count_words(int64_t n) { return (size_t)256 * (size_t)((n + kSortTile - 1) / kSortTile); }

// Sorts n pairs by the low `bits` bits of their keys (the rest zero): (k0, v0) holds the input, which is left as it
// is; the passes go between (k1, v1) and (k2, v2).  *in_k2: whether the result is in (k2, v2).
cudaError_t launch_sort_pairs(const uint64_t* k0, const double* v0, uint64_t* k1, double* v1, uint64_t* k2, double* v2,
                              int64_t n, int bits, uint32_t* counts, bool* in_k2, cudaStream_t st) {
  const int tiles = (int)((n + kSortTile - 1) / kSortTile);
  const uint64_t* ki = k0;
  const double* vi = v0;
  bool second = true;
  for (int shift = 0; shift < bits; shift += 8) {
    second = !second;
    uint64_t* ko = second ? k2 : k1;
    double* vo = second ? v2 : v1;
    sort_count_kernel<<<tiles, kSortThreads, 0, st>>>(ki, n, shift, counts, tiles);
    sort_scan_kernel<<<1, 1024, 0, st>>>(counts, (int64_t)256 * tiles);
    sort_scatter_kernel<<<tiles, kSortThreads, 0, st>>>(ki, vi, n, shift, counts, tiles, ko, vo);
    ki = ko;
    vi = vo;
  }
  *in_k2 = second;
  return cudaGetLastError();
}

}  // namespace swcs
