// Layout derivations done once per loaded program (predecessor lists, the
// block of each instruction, loop depths) and a device exclusive scan.
#include <algorithm>

#include "gpa_internal.cuh"
#include "scan_tiles.cuh"

namespace gpa {

namespace {

__global__ void __launch_bounds__(scan::kThreads) k_scan_sums(const int32_t* buf, int n, int32_t* sums) {
  scan::tile_sum(buf, n, sums);
}
template <bool kScanned>
__global__ void __launch_bounds__(scan::kThreads) k_scan_tiles(int32_t* buf, int n, const int32_t* sums) {
  scan::tile_scan<kScanned>(buf, n, sums, buf + n);
}

__global__ void k_instr_block(Prog P) {
  for (int b = blockIdx.x * blockDim.x + threadIdx.x; b < P.nb; b += gridDim.x * blockDim.x)
    for (int x = P.block_instr_off[b]; x < P.block_instr_off[b + 1]; ++x) ((int32_t*)P.instr_block)[x] = b;
}

// Thread per block, its function by binary search (a thread per function wrote a
// large function's blocks one by one: 96 us for 61 functions).
__global__ void k_block_func(Prog P) {
  for (int b = blockIdx.x * blockDim.x + threadIdx.x; b < P.nb; b += gridDim.x * blockDim.x) {
    int lo = 0, hi = P.nf;  // func_block_off[lo] <= b < func_block_off[hi]
    while (hi - lo > 1) {
      const int mid = (lo + hi) >> 1;
      if (P.func_block_off[mid] <= b) lo = mid;
      else hi = mid;
    }
    ((int32_t*)P.block_func)[b] = lo;
  }
}

__global__ void k_pred_count(Prog P, int n_succ, int32_t* pred_cnt) {
  for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < n_succ; e += gridDim.x * blockDim.x)
    atomicAdd(&pred_cnt[P.succ[e]], 1);
}

__global__ void k_pred_fill(Prog P, int32_t* cursor) {
  for (int b = blockIdx.x * blockDim.x + threadIdx.x; b < P.nb; b += gridDim.x * blockDim.x)
    for (int e = P.succ_off[b]; e < P.succ_off[b + 1]; ++e) {
      int s = P.succ[e];
      int at = atomicAdd(&cursor[s], 1);
      ((int32_t*)P.pred)[P.pred_off[s] + at] = b;
    }
}

// Predecessor lists in ascending block order (they are short).
__global__ void k_pred_sort(Prog P) {
  for (int b = blockIdx.x * blockDim.x + threadIdx.x; b < P.nb; b += gridDim.x * blockDim.x) {
    int32_t* a = (int32_t*)P.pred + P.pred_off[b];
    const int n = P.pred_off[b + 1] - P.pred_off[b];
    for (int i = 1; i < n; ++i) {
      int v = a[i], k = i - 1;
      while (k >= 0 && a[k] > v) { a[k + 1] = a[k]; --k; }
      a[k + 1] = v;
    }
  }
}

__global__ void k_loop_depth(Prog P) {
  for (int l = blockIdx.x * blockDim.x + threadIdx.x; l < P.nl; l += gridDim.x * blockDim.x) {
    int d = 0;
    for (int q = l; q >= 0 && d <= P.nl; q = P.loop_parent[q]) ++d;
    ((int32_t*)P.loop_depth)[l] = d;
  }
}

// Event lists for the backward scans, one segment per (block, resource bucket
// k = ev_bucket(r)): for each instruction of the block from the last to the
// first, its defs of the bucket's resources (with kind and guard) and, if
// unguarded, its reads of them. A scan for resource r reads only its bucket's
// segment (about 2.6 events on the batched workload, against 21.5 for the
// whole block); the events of r appear in it in the order of a bottom-up walk
// of the block (an instruction's defs before its reads). ev_off is the CSR over
// (block, bucket) pairs: segment (b, k) is [ev_off[b * 16 + k], ev_off[b * 16 + k + 1]).
// Both kernels walk a block once, a thread per block, with the 16 buckets'
// counters or cursors in shared memory (interleaved by thread); walking the
// block again for each bucket took 140 us for 29,000 blocks.
constexpr int kEvThreads = 128;
__global__ void __launch_bounds__(kEvThreads) k_ev_count(Prog P, int32_t* cnt) {
  __shared__ int32_t c[kEvBuckets][kEvThreads];
  const int tid = threadIdx.x;
  for (int b = blockIdx.x * kEvThreads + tid; b < P.nb; b += gridDim.x * kEvThreads) {
#pragma unroll
    for (int k = 0; k < kEvBuckets; ++k) c[k][tid] = 0;
    const int x0 = P.block_instr_off[b], x1 = P.block_instr_off[b + 1];
    // the block's defs are consecutive entries
    const int d1 = P.def_off[x1];
    for (int e = P.def_off[x0]; e < d1; ++e) ++c[ev_bucket(P.def_res[e] & 0x1FF)][tid];
    int u0 = P.use_off[x0];
    for (int x = x0; x < x1; ++x) {
      const int u1 = P.use_off[x + 1];
      if (P.guard[x] == 0)
        for (int e = u0; e < u1; ++e) ++c[ev_bucket(P.use_res[e] & 0x1FF)][tid];
      u0 = u1;
    }
    int4* out = reinterpret_cast<int4*>(cnt + (size_t)b * kEvBuckets);
#pragma unroll
    for (int k = 0; k < kEvBuckets; k += 4)
      out[k / 4] = make_int4(c[k][tid], c[k + 1][tid], c[k + 2][tid], c[k + 3][tid]);
  }
}

__global__ void __launch_bounds__(kEvThreads) k_ev_fill(Prog P, const int32_t* ev_off, uint32_t* events) {
  __shared__ int32_t cur[kEvBuckets][kEvThreads];
  const int tid = threadIdx.x;
  for (int b = blockIdx.x * kEvThreads + tid; b < P.nb; b += gridDim.x * kEvThreads) {
    const int4* in = reinterpret_cast<const int4*>(ev_off + (size_t)b * kEvBuckets);
#pragma unroll
    for (int k = 0; k < kEvBuckets; k += 4) {
      const int4 v = in[k / 4];
      cur[k][tid] = v.x; cur[k + 1][tid] = v.y; cur[k + 2][tid] = v.z; cur[k + 3][tid] = v.w;
    }
    const int first = P.block_instr_off[b];
    int x = P.block_instr_off[b + 1] - 1;
    int d1 = P.def_off[x + 1], u1 = P.use_off[x + 1];
    for (; x >= first; --x) {
      const uint32_t pos = (uint32_t)(x - first) << 16;
      const uint32_t g = P.guard[x];
      const int d0 = P.def_off[x], u0 = P.use_off[x];
      for (int e = d0; e < d1; ++e) {
        const uint32_t v = P.def_res[e];
        events[cur[ev_bucket(v & 0x1FFu)][tid]++] = (v & 0x1FFu) | 0x200u | (((v >> 12) & 3u) << 10) | (g << 12) | pos;
      }
      if (g == 0)
        for (int e = u0; e < u1; ++e) {
          const uint32_t v = P.use_res[e] & 0x1FFu;
          events[cur[ev_bucket(v)][tid]++] = v | pos;
        }
      d1 = d0;
      u1 = u0;
    }
  }
}

}  // namespace

void launch_build_events(const Prog& P, int32_t* ev_off, uint32_t* events, int32_t* tmp, cudaStream_t st, int sms,
                         int64_t* launches) {
  k_ev_count<<<grid_for(P.nb, kEvThreads, sms), kEvThreads, 0, st>>>(P, ev_off);
  ++*launches;
  scan_exclusive_inplace(ev_off, P.nb * kEvBuckets, tmp, st, launches);
  k_ev_fill<<<grid_for(P.nb, kEvThreads, sms), kEvThreads, 0, st>>>(P, ev_off, events);
  ++*launches;
}

__global__ void k_block_meta(Prog P, int4* meta) {
  for (int b = blockIdx.x * blockDim.x + threadIdx.x; b < P.nb; b += gridDim.x * blockDim.x) {
    meta[2 * (size_t)b] = make_int4(P.block_instr_off[b], P.block_instr_off[b + 1], P.ev_off[(size_t)b * kEvBuckets],
                                    P.ev_off[(size_t)(b + 1) * kEvBuckets]);
    const int q0 = P.pred_off[b], q1 = P.pred_off[b + 1];
    meta[2 * (size_t)b + 1] = make_int4(q0, q1, q1 > q0 ? P.pred[q0] : -1, q1 > q0 + 1 ? P.pred[q0 + 1] : -1);
  }
}

void launch_build_meta(const Prog& P, int4* meta, cudaStream_t st, int sms, int64_t* launches) {
  k_block_meta<<<grid_for(P.nb, 256, sms), 256, 0, st>>>(P, meta);
  ++*launches;
}

namespace {
__global__ void k_store_u64(unsigned long long* p, unsigned long long v) { *p = v; }
}  // namespace

void launch_store_u64(unsigned long long* p, unsigned long long v, cudaStream_t st, int64_t* launches) {
  k_store_u64<<<1, 1, 0, st>>>(p, v);
  ++*launches;
}

int grid_for(int64_t n, int threads, int sms) {
  int64_t g = (n + threads - 1) / threads;
  int64_t cap = (int64_t)sms * 8;
  if (g > cap) g = cap;
  return (int)(g < 1 ? 1 : g);
}

// The tiles' sums and their total, and the same again for those beyond kDirectTiles.
size_t scan_tmp_ints(int n) { return (size_t)scan::tiles_of(n) + scan::tiles_of(scan::tiles_of(n)) + 16; }

// buf has n + 1 entries; on return buf[k] = sum of the first k inputs and
// buf[n] = the total (the input buf[n] is ignored).
void scan_exclusive_inplace(int32_t* buf, int n, int32_t* tmp, cudaStream_t st, int64_t* launches) {
  const int tiles = scan::tiles_of(n);
  if (tiles > 1) {
    k_scan_sums<<<tiles, scan::kThreads, 0, st>>>(buf, n, tmp);
    ++*launches;
  }
  if (tiles > scan::kDirectTiles) {
    scan_exclusive_inplace(tmp, tiles, tmp + tiles + 1, st, launches);
    k_scan_tiles<true><<<tiles, scan::kThreads, 0, st>>>(buf, n, tmp);
  } else {
    k_scan_tiles<false><<<tiles, scan::kThreads, 0, st>>>(buf, n, tmp);
  }
  ++*launches;
}

void launch_build_layout(const Prog& P, cudaStream_t st, int sms, int64_t* launches) {
  k_instr_block<<<grid_for(P.nb, 256, sms), 256, 0, st>>>(P);
  k_loop_depth<<<grid_for(P.nl > 0 ? P.nl : 1, 256, sms), 256, 0, st>>>(P);
  k_block_func<<<grid_for(P.nb, 256, sms), 256, 0, st>>>(P);
  *launches += 3;
}

// Predecessor CSR: count, scan, fill, sort. pred_cnt has nb + 1 ints and
// ends up holding pred_off; cursor has nb ints.
void launch_build_preds(const Prog& P, int n_succ, int32_t* pred_off, int32_t* cursor, int32_t* tmp, cudaStream_t st,
                        int sms, int64_t* launches) {
  cudaMemsetAsync(pred_off, 0, sizeof(int32_t) * (P.nb + 1), st);
  cudaMemsetAsync(cursor, 0, sizeof(int32_t) * P.nb, st);
  k_pred_count<<<grid_for(n_succ > 0 ? n_succ : 1, 256, sms), 256, 0, st>>>(P, n_succ, pred_off);
  ++*launches;
  scan_exclusive_inplace(pred_off, P.nb, tmp, st, launches);
  k_pred_fill<<<grid_for(P.nb, 256, sms), 256, 0, st>>>(P, cursor);
  k_pred_sort<<<grid_for(P.nb, 256, sms), 256, 0, st>>>(P);
  *launches += 2;
}

}  // namespace gpa
