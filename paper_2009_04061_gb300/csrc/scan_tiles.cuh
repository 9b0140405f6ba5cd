// Exclusive scan of int32 values in two launches, shared by the library's own
// offsets (k_util.cu) and the scan for callers that may not allocate
// (k_noalloc.cu). The first launch only reads: it sums tiles of 4,096 values. In
// the second, each CTA adds up the sums of the tiles before its own (at most
// kDirectTiles of them, out of L2) and scans its tile from there, so the values are
// read twice and written once, and no launch scans the sums or adds them in a
// pass of its own (3,000,001 values: 10.7 + 2.7 + 8.9 us in three launches). Of more
// tiles the sums are scanned first, by the same two launches: adding them up in
// every CTA grows with the square of their number (2,048 tiles 26 us against 27
// with the sums scanned first, 4,096 42 against 40, 16,384 168 against 149, 524,288
// 22.7 against 4.0 ms).
// What bounds it is memory; values move as 16-byte vectors where the buffer
// allows.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

namespace gpa {
namespace scan {

constexpr int kThreads = 512;
constexpr int kItems = 8;                 // two 16-byte vectors a thread
constexpr int kTile = kThreads * kItems;  // 4,096 values
constexpr int kDirectTiles = 4096;

// Tiles of n values (0 <= n <= INT32_MAX), at least one.
constexpr int tiles_of(int64_t n) { return n <= kTile ? 1 : (int)((n + kTile - 1) / kTile); }
static_assert(tiles_of(0) == 1 && tiles_of(kTile) == 1 && tiles_of(kTile + 1) == 2 && tiles_of(INT32_MAX) == 524288,
              "up to the largest count");

// Loads this thread's kItems values of the tile at `off` (0 past n).
__device__ __forceinline__ void load_items(const int32_t* buf, int64_t off, int64_t n, bool vec, int32_t* v) {
  const int64_t base = off + (int64_t)threadIdx.x * kItems;
  if (vec && base + kItems <= n) {
    const int4 a = *reinterpret_cast<const int4*>(buf + base);
    const int4 b = *reinterpret_cast<const int4*>(buf + base + 4);
    v[0] = a.x; v[1] = a.y; v[2] = a.z; v[3] = a.w;
    v[4] = b.x; v[5] = b.y; v[6] = b.z; v[7] = b.w;
  } else {
#pragma unroll
    for (int t = 0; t < kItems; ++t) v[t] = base + t < n ? buf[base + t] : 0;
  }
}

// Sum over the CTA (every thread gets it); red: kThreads / 32 ints.
__device__ __forceinline__ int32_t cta_sum(int32_t x, int32_t* red) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = x;
  __syncthreads();
  int32_t s = 0;
#pragma unroll
  for (int w = 0; w < kThreads / 32; ++w) s += red[w];
  __syncthreads();
  return s;
}

// The tile's sum goes to sums[blockIdx.x].
__device__ __forceinline__ void tile_sum(const int32_t* buf, int64_t n, int32_t* sums) {
  __shared__ int32_t red[kThreads / 32];
  const bool vec = (reinterpret_cast<uintptr_t>(buf) & 15u) == 0;
  int32_t v[kItems], local = 0;
  load_items(buf, (int64_t)blockIdx.x * kTile, n, vec, v);
#pragma unroll
  for (int t = 0; t < kItems; ++t) local += v[t];
  const int32_t s = cta_sum(local, red);
  if (threadIdx.x == 0) sums[blockIdx.x] = s;
}

// Scans the tile in place from the sum of sums[0, blockIdx.x), or from
// sums[blockIdx.x] where they are scanned already (kScanned); the last tile's CTA
// writes the total (total may be null).
template <bool kScanned>
__device__ __forceinline__ void tile_scan(int32_t* buf, int64_t n, const int32_t* sums, int32_t* total) {
  __shared__ int32_t red[kThreads / 32];
  __shared__ int32_t warp_off[kThreads / 32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const bool vec = (reinterpret_cast<uintptr_t>(buf) & 15u) == 0;
  const int64_t off = (int64_t)blockIdx.x * kTile;
  int32_t v[kItems], local = 0;
  load_items(buf, off, n, vec, v);
  int32_t before = 0;
  if (kScanned) {
    before = sums[blockIdx.x];
  } else {
    for (unsigned t = threadIdx.x; t < blockIdx.x; t += kThreads) before += sums[t];
    before = cta_sum(before, red);
  }
#pragma unroll
  for (int t = 0; t < kItems; ++t) local += v[t];
  int32_t incl = local;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int32_t y = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += y;
  }
  if (lane == 31) warp_off[warp] = incl;
  __syncthreads();
  int32_t run = before + incl - local;
#pragma unroll
  for (int w = 0; w < kThreads / 32; ++w) run += w < warp ? warp_off[w] : 0;
  const int64_t base = off + (int64_t)threadIdx.x * kItems;
  int32_t out[kItems];
#pragma unroll
  for (int t = 0; t < kItems; ++t) {
    out[t] = run;
    run += v[t];
  }
  if (vec && base + kItems <= n) {
    *reinterpret_cast<int4*>(buf + base) = make_int4(out[0], out[1], out[2], out[3]);
    *reinterpret_cast<int4*>(buf + base + 4) = make_int4(out[4], out[5], out[6], out[7]);
  } else {
#pragma unroll
    for (int t = 0; t < kItems; ++t)
      if (base + t < n) buf[base + t] = out[t];
  }
  // (values past n count as 0, so the last thread's running sum is the total)
  if (total && blockIdx.x == gridDim.x - 1 && threadIdx.x == kThreads - 1) *total = run;
}

}  // namespace scan
}  // namespace gpa
