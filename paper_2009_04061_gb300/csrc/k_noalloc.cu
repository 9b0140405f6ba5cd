// gpa_exclusive_scan_noalloc: the library's exclusive prefix sum (the scan
// behind its edge, event and predecessor offsets) for callers that must not
// allocate device memory. Its scratch (the per-tile sums) is a fixed static
// device array instead of a cudaMalloc'd buffer; see include/gpa.h.
#include <cuda_runtime.h>

#include <mutex>

#include "gpa_internal.cuh"
#include "scan_tiles.cuh"

namespace {

using gpa::scan::kThreads;
using gpa::scan::kTile;                         // 4096 values per tile
constexpr int kMaxTiles = gpa::scan::kDirectTiles;  // so n <= 16,777,216
constexpr int kMaxDevices = 64;

// Tile sums of the last call. Every call writes each entry it reads before
// reading it, so nothing is cleared.
static __device__ __align__(256) int32_t g_scan_scratch[kMaxTiles + 64];

std::mutex g_mu;
int32_t* g_scratch_addr[kMaxDevices] = {nullptr};

__global__ void __launch_bounds__(kThreads) k_na_scan_sums(const int32_t* buf, int n, int32_t* scratch) {
  gpa::scan::tile_sum(buf, n, scratch);
}
__global__ void __launch_bounds__(kThreads) k_na_scan_tiles(int32_t* buf, int n, const int32_t* scratch,
                                                            int32_t* total) {
  gpa::scan::tile_scan<false>(buf, n, scratch, total);
}

// Device address of the scratch array on the current device, resolved once per
// device (host code cannot use the symbol itself as a device pointer).
gpa_status scratch_address(int32_t** out) {
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return GPA_ERR_CUDA;
  if (dev < 0 || dev >= kMaxDevices) return GPA_ERR_INVALID_ARG;
  std::lock_guard<std::mutex> lock(g_mu);
  if (!g_scratch_addr[dev]) {
    int32_t* p = nullptr;
    if (cudaGetSymbolAddress(reinterpret_cast<void**>(&p), g_scan_scratch) != cudaSuccess || !p)
      return GPA_ERR_CUDA;
    g_scratch_addr[dev] = p;
  }
  *out = g_scratch_addr[dev];
  return GPA_OK;
}

}  // namespace

extern "C" gpa_status gpa_exclusive_scan_noalloc(int32_t* dev_buf, int64_t n, int32_t* dev_total, gpa_stream stream) {
  if (n < 0 || (n > 0 && !dev_buf) || !dev_total) return GPA_ERR_INVALID_ARG;
  if (n > (int64_t)kMaxTiles * kTile) return GPA_ERR_CAPACITY;
  int32_t* scratch = nullptr;
  const gpa_status s = scratch_address(&scratch);
  if (s) return s;
  // An error left pending by an earlier, unrelated call is not ours to clear:
  // report it (it stays pending for its owner) and launch nothing.
  if (cudaPeekAtLastError() != cudaSuccess) return GPA_ERR_CUDA;
  cudaStream_t st = (cudaStream_t)stream;
  if (n == 0) return cudaMemsetAsync(dev_total, 0, sizeof(int32_t), st) == cudaSuccess ? GPA_OK : GPA_ERR_CUDA;
  const int tiles = gpa::scan::tiles_of(n);
  if (tiles > 1) {  // (a single tile has nothing before it)
    k_na_scan_sums<<<tiles, kThreads, 0, st>>>(dev_buf, (int)n, scratch);
    if (cudaGetLastError() != cudaSuccess) return GPA_ERR_CUDA;
  }
  k_na_scan_tiles<<<tiles, kThreads, 0, st>>>(dev_buf, (int)n, scratch, dev_total);
  return cudaGetLastError() == cudaSuccess ? GPA_OK : GPA_ERR_CUDA;
}
