// Host runtime behind the C ABI in include/gpa.h: context and program
// registry, input validation, device memory, stream-ordered launches, the
// chunked host-sample ingest, status words and parity getters.
#include <cuda_runtime.h>

#include <algorithm>
#include <climits>
#include <cstddef>
#include <cstdio>
#include <cstring>
#include <map>
#include <mutex>
#include <new>
#include <vector>

#include "gpa_internal.cuh"

using namespace gpa;

namespace {

struct ProgramRec {
  Prog P{};
  bool dry = false;                     // count bytes only (gpa_program_footprint)
  // Like the program's block, these come from the pool in stream order.
  int4* xbuf = nullptr;                 // export buffer of gpa_export_unpruned_edges (grown on demand)
  int64_t xbuf_cap = 0, x_n = 0;
  void* xout = nullptr;                 // the ordered export and its scratch, for xout_cap edges
  int64_t xout_cap = 0;
  cudaStream_t build = nullptr;         // stream of the stream-ordered allocations and copies
  int64_t bytes = 0;                    // device bytes requested for the program
  cudaGraphExec_t step_exec = nullptr;  // captured step (gpa_step_capture)
  LaunchRec* launch = nullptr;          // launch statistics (gpa_set_launch_stats)
  int64_t step_launches = 0;            // kernels in it
  int32_t *pred_off = nullptr, *cursor = nullptr, *ev_off = nullptr;  // build scratch kept from allocation
  uint32_t* events = nullptr;
  int4* meta = nullptr;
  int n_succ = 0, n_def = 0, n_use = 0;
  int32_t* scan_tmp = nullptr;
  void* block = nullptr;                // the program's device memory, one allocation
  size_t zero_at = 0, zero_bytes = 0;   // its part that starts as zeros
};

// What a load asks for, gathered before anything is allocated: the arrays to
// copy first, then those that start as zeros, then the rest. The vectors hold
// derived arrays until they are copied.
struct Layout {
  struct Item {
    void** slot;
    const void* src;  // host array to copy, or nullptr
    size_t bytes;
    bool zero;
  };
  std::vector<Item> items;
  std::vector<int32_t> order, minreach, tile_off, tile_func;
  std::vector<uint8_t> natural, iflags;
};

}  // namespace

struct gpa_ctx {
  int device = 0;
  int sms = 0;
  Arch arch{};
  gpa_options opts{};
  SearchArena tier[3]{};
  cudaEvent_t scratch_ev = nullptr;
  std::map<gpa_pid, ProgramRec*> progs;
  gpa_pid next_pid = 1;
  int64_t launches = 0;
  // staging for gpa_ingest_host_samples
  uint64_t* stage[2] = {nullptr, nullptr};
  size_t stage_n = 0;
  cudaStream_t copy_stream = nullptr;
  cudaStream_t capture_stream = nullptr;  // private stream for gpa_step_capture
  cudaStream_t build_stream = nullptr;    // program allocation, copies and layout builds
  cudaMemPool_t pool = nullptr;           // programs' memory, shared by the device's contexts (take_pool)
  char* load_stage = nullptr;             // pinned staging of a load's copies (kLoadStage bytes, on first use)
  char* advice_stage = nullptr;           // and of advice into pageable arrays (kAdviceStage bytes)
  cudaEvent_t ev_copied[2] = {nullptr, nullptr}, ev_used[2] = {nullptr, nullptr};
  gpa::SearchFork fork{};  // larger searches beside tiers 1-2
};

namespace {

constexpr size_t kStageSamples = (size_t)64 << 20;  // 64M samples (512 MB) per staging buffer

#define CK(x)                                   \
  do {                                          \
    if ((x) != cudaSuccess) return GPA_ERR_CUDA; \
  } while (0)

constexpr size_t kPoolKeep = (size_t)1 << 30;   // program memory a device's pool holds on to
constexpr size_t kLoadStage = (size_t)32 << 20;  // loads with at most this much to copy go through one copy

constexpr size_t kAdviceStage = (size_t)4 << 20;

template <class T>
void dev_alloc(Layout& L, T** p, size_t n, bool zero = false) {
  L.items.push_back({(void**)p, nullptr, std::max<size_t>(n, 1) * sizeof(T), zero});
}
template <class T>
void dev_copy(Layout& L, const T** dst, const T* src, size_t n) {
  if (n) L.items.push_back({(void**)dst, src, n * sizeof(T), false});
  else dev_alloc(L, const_cast<T**>(dst), 1);
}

// Offsets of the items in the program's one allocation (256-byte aligned).
size_t lay_out(const Layout& L, ProgramRec* R, std::vector<size_t>* at, size_t* copy_bytes) {
  at->assign(L.items.size(), 0);
  size_t off = 0;
  for (int pass = 0; pass < 3; ++pass) {
    if (pass == 1) R->zero_at = off;
    for (size_t k = 0; k < L.items.size(); ++k) {
      const Layout::Item& it = L.items[k];
      if ((it.src ? 0 : it.zero ? 1 : 2) != pass) continue;
      (*at)[k] = off;
      off += (it.bytes + 255) & ~(size_t)255;
    }
    if (pass == 0) *copy_bytes = off;
    if (pass == 1) R->zero_bytes = off - R->zero_at;
  }
  R->bytes = (int64_t)off;
  return off;
}

// Programs' memory comes from a pool of the library's own, one a device for all of
// the process's contexts, that holds on to up to kPoolKeep of it (the device's
// default pool returns all that unloaded programs gave back at the next
// synchronization, so every session mapped its memory anew). With a pool for each
// context, a server's eight slots could hold 8 GB that only they could reuse. The
// first context creates the pool, the last one gives it back.
struct DevicePool {
  cudaMemPool_t pool = nullptr;
  int users = 0;
};
std::mutex g_pool_mu;
std::map<int, DevicePool>& device_pools() {
  static auto* pools = new std::map<int, DevicePool>();  // (contexts may outlive the program's static objects)
  return *pools;
}
// The device's pool, nullptr if it cannot be had (programs take the default pool then).
cudaMemPool_t take_pool(int device) {
  std::lock_guard<std::mutex> lock(g_pool_mu);
  DevicePool& d = device_pools()[device];
  if (d.users == 0) {
    cudaMemPoolProps props{};
    props.allocType = cudaMemAllocationTypePinned;
    props.location.type = cudaMemLocationTypeDevice;
    props.location.id = device;
    uint64_t keep = kPoolKeep;
    if (cudaMemPoolCreate(&d.pool, &props) != cudaSuccess) {
      cudaGetLastError();
      return nullptr;
    }
    if (cudaMemPoolSetAttribute(d.pool, cudaMemPoolAttrReleaseThreshold, &keep) != cudaSuccess) {
      cudaGetLastError();
      cudaMemPoolDestroy(d.pool);
      return nullptr;
    }
  }
  ++d.users;
  return d.pool;
}
void drop_pool(int device, cudaMemPool_t pool) {
  if (!pool) return;
  std::lock_guard<std::mutex> lock(g_pool_mu);
  DevicePool& d = device_pools()[device];
  if (--d.users == 0) cudaMemPoolDestroy(d.pool);
}

// Stream-ordered memory from the pool, nullptr if there is none.
void* pool_alloc(const gpa_ctx* ctx, size_t bytes, cudaStream_t st) {
  void* p = nullptr;
  if ((ctx->pool ? cudaMallocFromPoolAsync(&p, bytes, ctx->pool, st) : cudaMallocAsync(&p, bytes, st)) == cudaSuccess)
    return p;
  cudaGetLastError();
  return nullptr;
}

// Frees a program whose work has finished (the callers synchronize first).
void free_program(ProgramRec* R) {
  if (R->step_exec) cudaGraphExecDestroy(R->step_exec);
  if (R->xbuf) cudaFree(R->xbuf);
  if (R->xout) cudaFree(R->xout);
  if (R->launch) cudaFree(R->launch);
  if (R->build) cudaStreamSynchronize(R->build);
  if (R->block) cudaFree(R->block);
  delete R;
}

// Vectorised sweeps of the validation (no early exit).
__attribute__((optimize("O3"))) bool any_above(const uint8_t* a, int64_t n, int limit) {
  int bad = 0;
  for (int64_t i = 0; i < n; ++i) bad |= a[i] > limit;
  return bad;
}
__attribute__((optimize("O3"))) bool any_above(const uint16_t* a, int64_t n, int limit) {
  int bad = 0;
  for (int64_t i = 0; i < n; ++i) bad |= a[i] > limit;
  return bad;
}
__attribute__((optimize("O3"))) bool any_outside(const int32_t* a, int64_t n, int32_t limit) {  // 0 <= a < limit
  int bad = 0;
  for (int64_t i = 0; i < n; ++i) bad |= (uint32_t)a[i] >= (uint32_t)limit;
  return bad;
}
__attribute__((optimize("O3"))) bool bad_defs(const uint16_t* a, int64_t n) {
  int bad = 0;
  for (int64_t i = 0; i < n; ++i) {
    const int r = a[i] & 0x1FF, kind = a[i] >> 12;
    bad |= (r >= kNumRes) | ((a[i] & 0x0E00) != 0) | (kind > 2) | ((kind != 0) & (r < kBarBase));
  }
  return bad;
}
__attribute__((optimize("O3"))) bool not_ascending(const int32_t* a, int64_t n, int least_step) {
  int bad = 0;
  for (int64_t i = 0; i < n; ++i) bad |= (int64_t)a[i + 1] - a[i] < least_step;
  return bad;
}
// Entries of one list that name the same resource `step` apart: apart[e] becomes
// nonzero once a list starts among the entries e + 1 .. e + step.
__attribute__((optimize("O3"))) bool repeats_at(const uint16_t* a, const uint8_t* first, uint8_t* apart, int64_t n,
                                                int step) {
  uint16_t bad = 0;
  for (int64_t e = 0; e + step < n; ++e) {
    const uint8_t s = (uint8_t)(apart[e] | first[e + step]);
    apart[e] = s;
    bad |= (uint16_t)((((a[e] ^ a[e + step]) & 0x1FF) == 0) & (s == 0));
  }
  return bad;
}
// A resource named twice in one of n lists (CSR: off, a). The lists are short and
// of unpredictable length, so entries are compared with their neighbours in
// vectorised sweeps, one per distance (list by list it was three quarters of the
// validation); a list longer than 16 is marked in a bitmap.
bool any_repeats(const int32_t* off, const uint16_t* a, int n) {
  int most = 0;
  for (int x = 0; x < n; ++x) most = std::max(most, off[x + 1] - off[x]);
  if (most < 2) return false;
  const int64_t m = off[n];
  std::vector<uint8_t> first((size_t)m + 1, 0), apart((size_t)m, 0);
  for (int x = 0; x < n; ++x) first[off[x]] = 1;  // (an empty list marks the next one's start again)
  for (int step = 1; step < std::min(most, 16); ++step)
    if (repeats_at(a, first.data(), apart.data(), m, step)) return true;
  if (most <= 16) return false;
  for (int x = 0; x < n; ++x) {
    const int k = off[x + 1] - off[x];
    if (k <= 16) continue;
    uint32_t seen[16] = {};
    for (int i = 0; i < k; ++i) {
      const unsigned r = a[off[x] + i] & 0x1FFu;
      if (seen[r >> 5] >> (r & 31) & 1u) return true;
      seen[r >> 5] |= 1u << (r & 31);
    }
  }
  return false;
}

ProgramRec* find(gpa_ctx* ctx, gpa_pid pid) {
  if (!ctx) return nullptr;
  auto it = ctx->progs.find(pid);
  return it == ctx->progs.end() ? nullptr : it->second;
}

// ---------------------------------------------------------------- validation
gpa_status validate(const gpa_program_desc* d, const Arch& A) {
  const int nf = d->n_functions, ni = d->n_instr, nb = d->n_blocks, nl = d->n_loops;
  if (nf < 1 || nf >= 65536 || ni < 1 || nb < nf || nl < 0 || d->n_lines < 1 || d->n_succ < 0 || d->n_def < 0 ||
      d->n_use < 0)
    return GPA_ERR_INVALID_PROGRAM;
  if ((int64_t)ni * kCnt >= ((int64_t)1 << 32)) return GPA_ERR_INVALID_PROGRAM;
  // event lists: int32 offsets over (block, resource bucket) segments and events
  if ((int64_t)nb * kEvBuckets >= INT32_MAX || (int64_t)d->n_def + d->n_use >= INT32_MAX)
    return GPA_ERR_INVALID_PROGRAM;
  if (!d->func_instr_off || !d->func_block_off || !d->func_loop_off || !d->block_instr_off || !d->succ_off ||
      !d->opclass || !d->guard || !d->iflags || !d->line || !d->def_off || !d->use_off || !d->block_loop)
    return GPA_ERR_INVALID_ARG;
  if ((d->n_succ && !d->succ) || (d->n_def && !d->def_res) || (d->n_use && !d->use_res) ||
      (nl && (!d->loop_parent || !d->loop_header)) || d->n_calls < 0 ||
      (d->n_calls && (!d->call_site || !d->call_callee)))
    return GPA_ERR_INVALID_ARG;
  for (int c = 0; c < d->n_calls; ++c) {
    const int x = d->call_site[c], g = d->call_callee[c];
    if (x < -1 || x >= ni || g < -1 || g >= nf || (x < 0 && g < 0)) return GPA_ERR_INVALID_PROGRAM;
    if (c && (x < d->call_site[c - 1] || (x >= 0 && x == d->call_site[c - 1]))) return GPA_ERR_INVALID_PROGRAM;
  }
  auto mono = [](const int32_t* a, int n, int last, bool strict) {
    return a[0] == 0 && a[n] == last && !not_ascending(a, n, strict ? 1 : 0);
  };
  if (!mono(d->func_instr_off, nf, ni, true) || !mono(d->func_block_off, nf, nb, true) ||
      !mono(d->func_loop_off, nf, nl, false) || !mono(d->block_instr_off, nb, ni, true) ||
      !mono(d->succ_off, nb, d->n_succ, false) || !mono(d->def_off, ni, d->n_def, false) ||
      !mono(d->use_off, ni, d->n_use, false))
    return GPA_ERR_INVALID_PROGRAM;
  std::vector<int> bfunc(nb), lfunc(nl);
  for (int b = 0; b < nb; ++b)
    if (d->block_instr_off[b + 1] - d->block_instr_off[b] > 65535) return GPA_ERR_INVALID_PROGRAM;
  for (int f = 0; f < nf; ++f) {
    if (d->func_instr_off[f + 1] - d->func_instr_off[f] >= (1 << 24)) return GPA_ERR_INVALID_PROGRAM;
    if (d->block_instr_off[d->func_block_off[f]] != d->func_instr_off[f]) return GPA_ERR_INVALID_PROGRAM;
    for (int b = d->func_block_off[f]; b < d->func_block_off[f + 1]; ++b) bfunc[b] = f;
    for (int l = d->func_loop_off[f]; l < d->func_loop_off[f + 1]; ++l) lfunc[l] = f;
  }
  if (any_above(d->opclass, ni, A.n_op - 1) || any_above(d->guard, ni, 14) || any_outside(d->line, ni, d->n_lines) ||
      bad_defs(d->def_res, d->n_def) || any_above(d->use_res, d->n_use, kNumRes - 1))
    return GPA_ERR_INVALID_PROGRAM;
  if (any_repeats(d->def_off, d->def_res, ni) || any_repeats(d->use_off, d->use_res, ni)) return GPA_ERR_INVALID_PROGRAM;
  for (int l = 0; l < nl; ++l) {
    const int p = d->loop_parent[l], h = d->loop_header[l];
    if (p < -1 || p >= nl || p == l || (p >= 0 && lfunc[p] != lfunc[l])) return GPA_ERR_INVALID_PROGRAM;
    if (h < 0 || h >= nb || bfunc[h] != lfunc[l]) return GPA_ERR_INVALID_PROGRAM;
    int depth = 0;
    for (int q = l; q >= 0; q = d->loop_parent[q])
      if (++depth > nl) return GPA_ERR_INVALID_PROGRAM;  // parent cycle
  }
  auto in_loop = [&](int b, int l) {
    for (int q = d->block_loop[b]; q >= 0; q = d->loop_parent[q])
      if (q == l) return true;
    return false;
  };
  for (int b = 0; b < nb; ++b) {
    const int q = d->block_loop[b];
    if (q < -1 || q >= nl || (q >= 0 && lfunc[q] != bfunc[b])) return GPA_ERR_INVALID_PROGRAM;
  }
  for (int l = 0; l < nl; ++l)
    if (!in_loop(d->loop_header[l], l)) return GPA_ERR_INVALID_PROGRAM;
  for (int u = 0; u < nb; ++u) {
    for (int e = d->succ_off[u]; e < d->succ_off[u + 1]; ++e) {
      const int v = d->succ[e];
      if (v < 0 || v >= nb || bfunc[v] != bfunc[u]) return GPA_ERR_INVALID_PROGRAM;
      for (int e2 = d->succ_off[u]; e2 < e; ++e2)
        if (d->succ[e2] == v) return GPA_ERR_INVALID_PROGRAM;
      if (v <= u) {  // must be a back edge: v heads a loop that contains u
        bool ok = false;
        for (int q = d->block_loop[u]; q >= 0 && !ok; q = d->loop_parent[q]) ok = d->loop_header[q] == v;
        if (!ok) return GPA_ERR_INVALID_PROGRAM;
      }
    }
  }
  // every block reachable from its function's entry
  std::vector<char> reach(nb, 0);
  std::vector<int> st;
  for (int f = 0; f < nf; ++f) {
    st.push_back(d->func_block_off[f]);
    reach[d->func_block_off[f]] = 1;
  }
  while (!st.empty()) {
    int b = st.back();
    st.pop_back();
    for (int e = d->succ_off[b]; e < d->succ_off[b + 1]; ++e)
      if (!reach[d->succ[e]]) { reach[d->succ[e]] = 1; st.push_back(d->succ[e]); }
  }
  for (int b = 0; b < nb; ++b)
    if (!reach[b]) return GPA_ERR_INVALID_PROGRAM;
  return GPA_OK;
}

gpa_status status_from(unsigned long long st) {
  if (st & ST_NOT_CONVERGED) return GPA_ERR_NOT_CONVERGED;
  if (st & (ST_CAPACITY | ST_OVERFLOW)) return GPA_ERR_CAPACITY;
  if (st & ST_TIMEOUT) return GPA_ERR_TIMEOUT;
  return GPA_OK;
}

// Default opcode classes (order documented in gpa.h).
const int32_t kDefLat[21] = {4, 5, 4, 4, 2, 0, 32, 32, 1024, 1024, 32, 32, 1024, 1024, 64, 1024, 16, 16, 8, 0, 1024};
const uint32_t kDefFlags[21] = {
    0, 0, 0, 0, 0, 0, GPA_F_SYNC, GPA_F_SYNC,
    GPA_F_MEM | GPA_F_GLOBAL | GPA_F_VARLAT, GPA_F_MEM | GPA_F_GLOBAL | GPA_F_VARLAT,
    GPA_F_SHARED | GPA_F_VARLAT, GPA_F_SHARED | GPA_F_VARLAT,
    GPA_F_MEM | GPA_F_LOCAL | GPA_F_VARLAT, GPA_F_MEM | GPA_F_LOCAL | GPA_F_VARLAT,
    GPA_F_MEM | GPA_F_CONST | GPA_F_VARLAT, GPA_F_MEM | GPA_F_GLOBAL | GPA_F_VARLAT,
    GPA_F_LONG_ARITH | GPA_F_VARLAT, GPA_F_LONG_ARITH | GPA_F_VARLAT, 0, 0, 0};

}  // namespace

extern "C" {

const char* gpa_status_string(gpa_status s) {
  switch (s) {
    case GPA_OK: return "ok";
    case GPA_ERR_INVALID_ARG: return "invalid argument";
    case GPA_ERR_INVALID_PROGRAM: return "invalid program";
    case GPA_ERR_CUDA: return "CUDA runtime error";
    case GPA_ERR_NOT_CONVERGED: return "reaching-definitions fixpoint did not converge";
    case GPA_ERR_CAPACITY: return "capacity exceeded";
    case GPA_ERR_TIMEOUT: return "device wait timed out";
    case GPA_ERR_NO_PROGRAM: return "no such program";
    case GPA_ERR_OOM: return "out of device memory";
    default: return "unknown status";
  }
}

gpa_status gpa_arch_default(gpa_arch_desc* arch) {
  if (!arch) return GPA_ERR_INVALID_ARG;
  arch->n_opclasses = 21;
  arch->latency = kDefLat;
  arch->flags = kDefFlags;
  return GPA_OK;
}

gpa_status gpa_create(const gpa_arch_desc* arch, const gpa_options* opts, gpa_ctx** out) {
  if (!arch || !out || arch->n_opclasses < 1 || arch->n_opclasses > GPA_MAX_OPCLASSES || !arch->latency ||
      !arch->flags)
    return GPA_ERR_INVALID_ARG;
  for (int o = 0; o < arch->n_opclasses; ++o)
    if (arch->latency[o] < 0) return GPA_ERR_INVALID_ARG;
  gpa_options o{};
  if (opts) {
    o = *opts;
    if (o.max_fixpoint_sweeps < 0 || o.max_search_nodes < 0 || o.search_slots < 0 || o.max_sources_per_use < 0 ||
        o.max_sources_per_use > kBigSrc || o.small_search_nodes < 0 || o.mid_search_nodes < 0 ||
        o.hist_variant < 0 || o.hist_variant > 3 || o.large_search_nodes < 0 || o.hist_chunk < 0 ||
        o.hist_chunk > 4096 || o.reach_schedule < 0 || o.reach_schedule > 1 || o.small_search_warps < 0 ||
        o.small_search_warps > 32 || o.small_search_warps % 4 != 0)
      return GPA_ERR_INVALID_ARG;
  }
  auto* c = new (std::nothrow) gpa_ctx();
  if (!c) return GPA_ERR_OOM;
  if (cudaGetDevice(&c->device) != cudaSuccess ||
      cudaDeviceGetAttribute(&c->sms, cudaDevAttrMultiProcessorCount, c->device) != cudaSuccess) {
    delete c;
    return GPA_ERR_CUDA;
  }
  c->arch.n_op = arch->n_opclasses;
  for (int k = 0; k < arch->n_opclasses; ++k) { c->arch.lat[k] = arch->latency[k]; c->arch.flags[k] = arch->flags[k]; }
  if (o.max_fixpoint_sweeps == 0) o.max_fixpoint_sweeps = 64;
  if (o.max_search_nodes == 0) o.max_search_nodes = 32768;
  // Global-memory search warps: as many as the search kernel keeps resident
  // (its registers allow 24 one-warp CTAs per SM on GB300). Many warps on
  // global-memory arenas hide latency better than few on shared memory.
  if (o.search_slots == 0) o.search_slots = search_warps_per_sm() * c->sms;
  if (o.max_sources_per_use == 0) o.max_sources_per_use = kBigSrc;
  if (o.small_search_nodes == 0) o.small_search_nodes = 16;
  if (o.small_search_warps == 0) o.small_search_warps = 24;
  c->opts = o;
  // Tiers 1 and 2: one search a lane over shared-memory arenas, as many one-warp
  // CTAs per SM as their arenas fit. Tier 3: warps with global-memory arenas
  // for the searches beyond that. Node capacities are powers of two (hash
  // masks); a lane's arena holds at most 128 (byte indices).
  int n1 = 2, n3 = 2;
  while (n1 < o.small_search_nodes && n1 < kLaneNodes) n1 <<= 1;
  while (n3 < o.max_search_nodes) n3 <<= 1;
  int n2 = n1;
  const int want2 = o.mid_search_nodes ? o.mid_search_nodes : 64;
  while (n2 < want2 && n2 < kLaneNodes) n2 <<= 1;
  SearchArena* T = c->tier;
  auto lane_tier = [&](int nodes, int most) {
    SearchArena t{};
    t.nodes = nodes;
    t.bytes = search_lane_bytes(nodes);
    // a CTA's arena and the 1 KB the system reserves for it, in 227 KB of an SM
    t.warps = c->sms * (int)std::max<int64_t>(1, std::min<int64_t>(most, 227 * 1024 / (t.bytes + 1024)));
    return t;
  };
  T[0] = lane_tier(n1, o.small_search_warps);
  T[1] = lane_tier(n2, 32);
  T[2].nodes = n3; T[2].src = std::min(n3, 1024); T[2].layers = kMaxLayers; T[2].warps = o.search_slots;
  T[2].bytes = search_arena_bytes(T[2].nodes, T[2].src, T[2].layers, false);
  gpa_status s = GPA_OK;
  if (!s && cudaMalloc(&T[2].global, (size_t)T[2].bytes * T[2].warps) != cudaSuccess) {
    T[2].global = nullptr;
    s = GPA_ERR_OOM;
  }
  if (!s && cudaMemset(T[2].global, 0, (size_t)T[2].bytes * T[2].warps) != cudaSuccess) s = GPA_ERR_CUDA;
  // The third tier's node hashes start empty (-1); every search leaves them so.
  const size_t hash_bytes = sizeof(int32_t) * 2 * (size_t)T[2].nodes * T[2].warps;
  if (!s && cudaMalloc(&T[2].hash, hash_bytes) != cudaSuccess) {
    T[2].hash = nullptr;
    s = GPA_ERR_OOM;
  }
  if (!s && cudaMemset(T[2].hash, 0xFF, hash_bytes) != cudaSuccess) s = GPA_ERR_CUDA;
  if (!s && cudaEventCreateWithFlags(&c->scratch_ev, cudaEventDisableTiming) != cudaSuccess) s = GPA_ERR_CUDA;
  if (!s) c->pool = take_pool(c->device);
  if (!s && cudaStreamCreateWithFlags(&c->build_stream, cudaStreamNonBlocking) != cudaSuccess) s = GPA_ERR_CUDA;
  if (!s && cudaEventCreateWithFlags(&c->fork.fork, cudaEventDisableTiming) != cudaSuccess) s = GPA_ERR_CUDA;
  for (int k = 0; k < 3; ++k) {
    if (!s && cudaStreamCreateWithFlags(&c->fork.side[k], cudaStreamNonBlocking) != cudaSuccess) s = GPA_ERR_CUDA;
    if (!s && cudaEventCreateWithFlags(&c->fork.join[k], cudaEventDisableTiming) != cudaSuccess) s = GPA_ERR_CUDA;
  }
  if (s) {
    if (c->tier[2].global) cudaFree(c->tier[2].global);
    if (c->tier[2].hash) cudaFree(c->tier[2].hash);
    if (c->scratch_ev) cudaEventDestroy(c->scratch_ev);
    drop_pool(c->device, c->pool);
    if (c->build_stream) cudaStreamDestroy(c->build_stream);
    if (c->fork.fork) cudaEventDestroy(c->fork.fork);
    for (int k = 0; k < 3; ++k) {
      if (c->fork.side[k]) cudaStreamDestroy(c->fork.side[k]);
      if (c->fork.join[k]) cudaEventDestroy(c->fork.join[k]);
    }
    delete c;
    return s;
  }
  *out = c;
  return GPA_OK;
}

gpa_status gpa_destroy(gpa_ctx* ctx) {
  if (!ctx) return GPA_ERR_INVALID_ARG;
  cudaDeviceSynchronize();
  for (auto& kv : ctx->progs) free_program(kv.second);
  drop_pool(ctx->device, ctx->pool);
  if (ctx->load_stage) cudaFreeHost(ctx->load_stage);
  if (ctx->advice_stage) cudaFreeHost(ctx->advice_stage);
  if (ctx->tier[2].global) cudaFree(ctx->tier[2].global);
  if (ctx->tier[2].hash) cudaFree(ctx->tier[2].hash);
  for (int k = 0; k < 2; ++k) {
    if (ctx->stage[k]) cudaFree(ctx->stage[k]);
    if (ctx->ev_copied[k]) cudaEventDestroy(ctx->ev_copied[k]);
    if (ctx->ev_used[k]) cudaEventDestroy(ctx->ev_used[k]);
  }
  if (ctx->copy_stream) cudaStreamDestroy(ctx->copy_stream);
  if (ctx->capture_stream) cudaStreamDestroy(ctx->capture_stream);
  if (ctx->build_stream) cudaStreamDestroy(ctx->build_stream);
  if (ctx->scratch_ev) cudaEventDestroy(ctx->scratch_ev);
  if (ctx->fork.fork) cudaEventDestroy(ctx->fork.fork);
  for (int k = 0; k < 3; ++k) {
    if (ctx->fork.side[k]) cudaStreamDestroy(ctx->fork.side[k]);
    if (ctx->fork.join[k]) cudaEventDestroy(ctx->fork.join[k]);
  }
  delete ctx;
  return GPA_OK;
}

// Gathers the program's device arrays and derives those that are computed on
// the host (with R->dry, only their sizes). pool_bytes: the context's search
// arenas, which the fourth tier uses when they hold more than its own would.
static void plan_program(const gpa_program_desc* d, ProgramRec* R, Layout& L, int tier3_nodes, int64_t pool_bytes,
                         int sms) {
  Prog& P = R->P;
  P.nf = d->n_functions; P.ni = d->n_instr; P.nb = d->n_blocks; P.nl = d->n_loops; P.n_lines = d->n_lines;
  // Staged fixpoint: the largest per-function need within the cap (edges stay
  // inside their function, so a function's predecessor entries are its
  // blocks' successor entries).
  auto reach_need = [&](int f) {
    const int b0 = d->func_block_off[f], b1 = d->func_block_off[f + 1];
    return reach_smem_need(b1 - b0, (int64_t)d->succ_off[b1] - d->succ_off[b0],
                           (int64_t)d->func_loop_off[f + 1] - d->func_loop_off[f]);
  };
  // Staged fixpoint: functions needing at most this much shared memory (the
  // others go by mask words where their loops are natural ones and a word a block
  // fits, else to the windowed global-memory kernel).
  P.reach_smem = 0;
  for (int f = 0; f < d->n_functions; ++f) {
    const int64_t need = reach_need(f);
    if (need <= kReachClassCap[0] && need > P.reach_smem) P.reach_smem = (int32_t)need;
  }
  R->n_succ = d->n_succ; R->n_def = d->n_def; R->n_use = d->n_use;
  const size_t ni = P.ni, nb = P.nb, nl = P.nl, nf = P.nf;
  dev_copy(L, &P.func_instr_off, d->func_instr_off, nf + 1);
  {
    // The staged fixpoint takes the functions by shared memory need, largest
    // first, in four launches by size class (kReachClassCap): class c holds the
    // needs in (cap[c + 1], cap[c]], and its launch sizes its stage for the
    // largest of them. Functions beyond cap[0] are left to the kernels by mask words
    // and by windows (reach_windowed of them).
    std::vector<int64_t> need(nf);
    for (size_t f = 0; f < nf; ++f) need[f] = reach_need((int)f);
    std::vector<int32_t>& order = L.order;
    order.resize(nf);
    for (size_t f = 0; f < nf; ++f) order[f] = (int32_t)f;
    std::stable_sort(order.begin(), order.end(), [&](int32_t a, int32_t b) { return need[a] > need[b]; });
    dev_copy(L, &P.reach_order, order.data(), nf);
    int q = 0;
    while (q < (int)nf && need[order[q]] > kReachClassCap[0]) ++q;
    for (int c = 0; c < 4; ++c) {
      P.reach_cls[c] = q;
      P.reach_cls_smem[c] = 0;
      const int64_t lo = c < 3 ? kReachClassCap[c + 1] : -1;
      while (q < (int)nf && need[order[q]] > lo) {
        P.reach_cls_smem[c] = std::max<int32_t>(P.reach_cls_smem[c], (int32_t)need[order[q]]);
        ++q;
      }
    }
    P.reach_cls[4] = q;
    // Natural loops: a loop body is the header and the blocks that reach one of
    // its latches (a body block with an edge to the header) without passing the
    // header. Then every body block reaches every other one, which lets the
    // fixpoint seed a block with the definitions of its enclosing loops.
    std::vector<uint8_t>& natural = L.natural;
    natural.assign(nf, 1);
    if (!R->dry) {  // (a footprint needs only the sizes)
      std::vector<int32_t> pcnt(nb + 1, 0), pl((size_t)d->n_succ);
      for (size_t u = 0; u < nb; ++u)
        for (int e = d->succ_off[u]; e < d->succ_off[u + 1]; ++e) ++pcnt[d->succ[e] + 1];
      for (size_t b = 0; b < nb; ++b) pcnt[b + 1] += pcnt[b];
      std::vector<int32_t> fill(pcnt.begin(), pcnt.end() - 1);
      for (size_t u = 0; u < nb; ++u)
        for (int e = d->succ_off[u]; e < d->succ_off[u + 1]; ++e) pl[fill[d->succ[e]]++] = (int32_t)u;
      auto in_body = [&](int b, int l) {
        for (int q = d->block_loop[b]; q >= 0; q = d->loop_parent[q])
          if (q == l) return true;
        return false;
      };
      std::vector<int32_t> body_n(nl, 0), stamp(nb, -1), st;
      for (size_t b = 0; b < nb; ++b)
        for (int q = d->block_loop[b]; q >= 0; q = d->loop_parent[q]) ++body_n[q];
      for (size_t f = 0; f < nf; ++f)
        for (int l = d->func_loop_off[f]; l < d->func_loop_off[f + 1] && natural[f]; ++l) {
          const int h = d->loop_header[l];
          int seen = 1;
          stamp[h] = l;
          st.clear();
          for (int e = pcnt[h]; e < pcnt[h + 1]; ++e)
            if (in_body(pl[e], l) && stamp[pl[e]] != l) { stamp[pl[e]] = l; ++seen; st.push_back(pl[e]); }
          while (!st.empty() && natural[f]) {
            const int x = st.back();
            st.pop_back();
            if (!in_body(x, l)) { natural[f] = 0; break; }
            for (int e = pcnt[x]; e < pcnt[x + 1]; ++e)
              if (stamp[pl[e]] != l) { stamp[pl[e]] = l; ++seen; st.push_back(pl[e]); }
          }
          if (seen != body_n[l]) natural[f] = 0;
        }
    }
    dev_copy(L, &P.func_natural, natural.data(), nf);
    P.reach_windowed = 0;
    for (int k = 0; k < P.reach_cls[0]; ++k) {
      const int f = order[k];
      const int64_t nbf = d->func_block_off[f + 1] - d->func_block_off[f],
                    nlf = d->func_loop_off[f + 1] - d->func_loop_off[f];
      if (!natural[f] || reach_words_need(nbf, nlf) > kReachSmemCap) ++P.reach_windowed;
    }
    // Smallest block reachable from each block: a min fixpoint over
    // successors, swept in descending block order (forward edges point up, so
    // each sweep settles every forward path; back edges need a few more).
    std::vector<int32_t>& mr = L.minreach;
    mr.resize(nb);
    for (size_t b = 0; b < nb; ++b) mr[b] = (int32_t)b;
    for (bool changed = !R->dry; changed;) {
      changed = false;
      for (size_t b = nb; b-- > 0;)
        for (int e = d->succ_off[b]; e < d->succ_off[b + 1]; ++e)
          if (mr[d->succ[e]] < mr[b]) { mr[b] = mr[d->succ[e]]; changed = true; }
    }
    dev_copy(L, &P.block_minreach, mr.data(), nb);
  }
  dev_copy(L, &P.func_block_off, d->func_block_off, nf + 1);
  dev_copy(L, &P.func_loop_off, d->func_loop_off, nf + 1);
  dev_copy(L, &P.block_instr_off, d->block_instr_off, nb + 1);
  dev_copy(L, &P.succ_off, d->succ_off, nb + 1);
  dev_copy(L, &P.succ, d->succ, (size_t)d->n_succ);
  dev_copy(L, &P.opclass, d->opclass, ni);
  dev_copy(L, &P.guard, d->guard, ni);
  {
    // Instruction flags on the device: bit 0 math-library code (the caller's
    // bit 0), bit 1 call site, bit 2 in a device function (a function some call
    // site calls): Function Inlining matches bits 1-2.
    std::vector<uint8_t>& fl = L.iflags;
    fl.resize(ni);
    std::vector<char> dev(nf, 0);
    for (int c = 0; c < d->n_calls; ++c)
      if (d->call_callee[c] >= 0) dev[d->call_callee[c]] = 1;
    for (size_t f = 0; f < nf; ++f)
      for (int x = d->func_instr_off[f]; x < d->func_instr_off[f + 1]; ++x)
        fl[x] = (uint8_t)((d->iflags[x] & 1) | (dev[f] ? 4 : 0));
    for (int c = 0; c < d->n_calls; ++c)
      if (d->call_site[c] >= 0) fl[d->call_site[c]] |= 2;
    dev_copy(L, &P.iflags, fl.data(), ni);
  }
  dev_copy(L, &P.line, d->line, ni);
  dev_copy(L, &P.def_off, d->def_off, ni + 1);
  dev_copy(L, &P.def_res, d->def_res, (size_t)d->n_def);
  dev_copy(L, &P.use_off, d->use_off, ni + 1);
  dev_copy(L, &P.use_res, d->use_res, (size_t)d->n_use);
  dev_copy(L, &P.block_loop, d->block_loop, nb);
  dev_copy(L, &P.loop_parent, d->loop_parent, nl);
  dev_copy(L, &P.loop_header, d->loop_header, nl);
  auto alloc_const = [&](const int32_t** q, size_t n) { dev_alloc(L, const_cast<int32_t**>(q), n); };
  alloc_const(&P.pred_off, nb + 1);
  alloc_const(&P.pred, (size_t)d->n_succ);
  dev_alloc(L, &R->cursor, nb);
  alloc_const(&P.loop_depth, nl);
  alloc_const(&P.instr_block, ni);
  alloc_const(&P.block_func, nb);
  alloc_const(&P.ev_off, nb * kEvBuckets + 1);
  dev_alloc(L, &R->events, (size_t)d->n_def + (size_t)d->n_use);
  dev_alloc(L, &P.res_maxlat, 2 * nf * kNumRes);  // and res_guards
  dev_alloc(L, &R->scan_tmp, scan_tmp_ints((int)std::max(ni, nb * kEvBuckets) + 1));
  dev_alloc(L, &P.cnt, ni * kCnt, true);
  dev_alloc(L, &P.stats, (size_t)SS_N, true);
  dev_alloc(L, &P.def_mask, nb * kWords);
  dev_alloc(L, &P.touch_mask, nb * kWords);
  dev_alloc(L, &R->meta, 2 * nb);
  dev_alloc(L, &P.rin, nb * kWords);
  dev_alloc(L, &P.rout, nb * kWords);
  dev_alloc(L, &P.head, ni);
  P.raw_cap = 2 * (int64_t)d->n_use + 1024;
  dev_alloc(L, &P.raw, (size_t)P.raw_cap);
  P.queue_cap = (int64_t)d->n_use + 1;
  for (int k = 0; k < 8; ++k) dev_alloc(L, &P.queue[k], (size_t)P.queue_cap);
  dev_alloc(L, &P.tasks, (size_t)std::max<int64_t>(d->n_use, 1));
  for (int k = 0; k < 2; ++k) dev_alloc(L, &P.tier_hint[k], (size_t)std::max<int64_t>(d->n_use, 1), true);
  dev_alloc(L, &P.cov_cnt, (size_t)std::max<int64_t>(d->n_use, 1));
  P.diag = 0;
  dev_alloc(L, &P.edge_off, ni + 1, true);
  dev_alloc(L, &P.big_use, ni);
  dev_alloc(L, &P.suse, ni);
  P.edge_cap = P.raw_cap;
  dev_alloc(L, &P.e_use, (size_t)P.edge_cap);
  dev_alloc(L, &P.e_def, (size_t)P.edge_cap);
  dev_alloc(L, &P.e_dmin, (size_t)P.edge_cap);
  dev_alloc(L, &P.e_dlong, (size_t)P.edge_cap);
  dev_alloc(L, &P.e_flags, (size_t)P.edge_cap);
  dev_alloc(L, &P.e_share, (size_t)P.edge_cap * 8);
  dev_alloc(L, &P.blame, ni * kCnt);
  dev_alloc(L, &P.a_totals, nf * 4);
  dev_alloc(L, &P.a_matched, nf * GPA_NUM_OPT);
  dev_alloc(L, &P.a_speedup, nf * GPA_NUM_OPT);
  dev_alloc(L, &P.a_rank, nf * GPA_NUM_OPT);
  dev_alloc(L, &P.a_nhot, nf * GPA_NUM_OPT);
  dev_alloc(L, &P.a_hot, nf * GPA_NUM_OPT * 5 * 6);
  dev_alloc(L, &P.a_loop_speedup, nl);
  {
    P.adv_tile = adv_tile_size(P.ni, sms);
    std::vector<int32_t>&off = L.tile_off, &func = L.tile_func;
    off.assign(nf + 1, 0);
    for (size_t f = 0; f < nf; ++f) {
      const int n = (d->func_instr_off[f + 1] - d->func_instr_off[f] + P.adv_tile - 1) / P.adv_tile;
      off[f + 1] = off[f] + n;
      func.insert(func.end(), (size_t)n, (int32_t)f);
    }
    P.adv_tiles = off[nf];
    dev_copy(L, &P.adv_tile_off, off.data(), nf + 1);
    dev_copy(L, &P.adv_tile_func, func.data(), func.size());
    dev_alloc(L, &P.adv_tops, (size_t)P.adv_tiles * GPA_NUM_OPT * 5);
    P.adv_zero = (int64_t)(nf * kAdvAcc + 4 * nl + 2 * (size_t)P.n_lines);
    dev_alloc(L, &P.adv_acc, (size_t)P.adv_zero);
  }
  dev_alloc(L, &P.a_par_match, nf * 2);
  dev_alloc(L, &P.a_par_speedup, nf * 2);
  dev_alloc(L, &P.a_par_warps, nf * 4);
  dev_alloc(L, &P.a_par_limit, nf);
  P.launch = nullptr;
  P.sm = SmModel{};
  // Fourth search tier: room for 64 literal sets per block of the largest
  // function (at most 2^22 nodes), when that is more than the context's
  // third tier holds; fewer CTAs for bigger arenas (about 2 GB at most).
  {
    int64_t mb = 1;
    for (int f = 0; f < d->n_functions; ++f) mb = std::max<int64_t>(mb, d->func_block_off[f + 1] - d->func_block_off[f]);
    int64_t n4 = 2;
    while (n4 < 64 * mb && n4 < ((int64_t)1 << 22)) n4 <<= 1;
    P.t4_nodes = 0; P.t4_arena = nullptr; P.t4_bytes = 0; P.t4_ctas = 0; P.t4_src = 0;
    if (n4 > tier3_nodes) {
      P.t4_nodes = (int32_t)n4;
      P.t4_src = (int32_t)std::min<int64_t>(n4, 4096);
      P.t4_ctas = n4 <= ((int64_t)1 << 18) ? 16 : n4 <= ((int64_t)1 << 20) ? 8 : 4;
      P.t4_bytes = search_arena_bytes(P.t4_nodes, P.t4_src, kMaxLayers, true);
      // arenas of its own only where the context's pool holds no more of them
      if (pool_bytes / P.t4_bytes <= P.t4_ctas) dev_alloc(L, &P.t4_arena, (size_t)P.t4_bytes * P.t4_ctas);
    }
  }
}

// Pointers into other allocations, once these have theirs.
static void derive_pointers(ProgramRec* R) {
  Prog& P = R->P;
  R->pred_off = const_cast<int32_t*>(P.pred_off);
  R->ev_off = const_cast<int32_t*>(P.ev_off);
  P.events = R->events;
  P.block_meta = R->meta;
  P.res_guards = reinterpret_cast<uint32_t*>(P.res_maxlat) + (size_t)P.nf * kNumRes;
  P.adv_own_active = P.adv_acc + (size_t)P.nf * kAdvAcc;
  P.adv_own_matched = P.adv_own_active + P.nl;
  P.a_loop_active = P.adv_own_matched + P.nl;
  P.a_loop_matched = P.a_loop_active + P.nl;
  P.a_line_stall = P.a_loop_matched + P.nl;
  P.a_line_lat = P.a_line_stall + P.n_lines;
}

static int64_t arena_pool_bytes(const gpa_ctx* ctx) { return (int64_t)ctx->tier[2].bytes * ctx->tier[2].warps; }

// Allocates the program's memory and queues its copies and clears on the build
// stream: one allocation (eighty of them, and as many pageable copies, were
// most of a small program's load), the arrays gathered in pinned memory for one
// copy unless they are large. On failure the caller frees R.
static gpa_status place_program(gpa_ctx* ctx, ProgramRec* R, const Layout& L) {
  std::vector<size_t> at;
  size_t copy_bytes = 0;
  const size_t total = lay_out(L, R, &at, &copy_bytes);
  cudaStream_t st = R->build;
  R->block = pool_alloc(ctx, total, st);
  if (!R->block) return GPA_ERR_OOM;
  char* base = static_cast<char*>(R->block);
  for (size_t k = 0; k < L.items.size(); ++k) *L.items[k].slot = base + at[k];
  derive_pointers(R);
  if (!ctx->load_stage && cudaMallocHost(&ctx->load_stage, kLoadStage) != cudaSuccess) {
    cudaGetLastError();
    ctx->load_stage = nullptr;  // (copied array by array then)
  }
  const bool staged = ctx->load_stage && copy_bytes <= kLoadStage;
  for (size_t k = 0; k < L.items.size(); ++k) {
    const Layout::Item& it = L.items[k];
    if (!it.src) continue;
    if (staged) std::memcpy(ctx->load_stage + at[k], it.src, it.bytes);
    else if (cudaMemcpyAsync(base + at[k], it.src, it.bytes, cudaMemcpyHostToDevice, st) != cudaSuccess) return GPA_ERR_CUDA;
  }
  if (staged && cudaMemcpyAsync(base, ctx->load_stage, copy_bytes, cudaMemcpyHostToDevice, st) != cudaSuccess)
    return GPA_ERR_CUDA;
  if (cudaMemsetAsync(base + R->zero_at, 0, R->zero_bytes, st) != cudaSuccess) return GPA_ERR_CUDA;
  return GPA_OK;
}

gpa_status gpa_program_footprint(gpa_ctx* ctx, const gpa_program_desc* d, int64_t* bytes) {
  if (!ctx || !d || !bytes) return GPA_ERR_INVALID_ARG;
  gpa_status s = validate(d, ctx->arch);
  if (s) return s;
  ProgramRec R;
  R.dry = true;
  Layout L;
  plan_program(d, &R, L, ctx->tier[2].nodes, arena_pool_bytes(ctx), ctx->sms);
  std::vector<size_t> at;
  size_t copy_bytes = 0;
  lay_out(L, &R, &at, &copy_bytes);
  *bytes = R.bytes;
  return GPA_OK;
}

gpa_status gpa_program_bytes(gpa_ctx* ctx, gpa_pid pid, int64_t* bytes) {
  ProgramRec* R = find(ctx, pid);
  if (!R) return GPA_ERR_NO_PROGRAM;
  if (!bytes) return GPA_ERR_INVALID_ARG;
  *bytes = R->bytes;
  return GPA_OK;
}

gpa_status gpa_load_program(gpa_ctx* ctx, const gpa_program_desc* d, gpa_pid* out) {
  if (!ctx || !d || !out) return GPA_ERR_INVALID_ARG;
  gpa_status s = validate(d, ctx->arch);
  if (s) return s;
  auto* R = new (std::nothrow) ProgramRec();
  if (!R) return GPA_ERR_OOM;
  R->build = ctx->build_stream;
  Layout L;
  plan_program(d, R, L, ctx->tier[2].nodes, arena_pool_bytes(ctx), ctx->sms);
  s = place_program(ctx, R, L);
  if (s) { free_program(R); return s; }
  Prog& P = R->P;
  for (int c = 0; c < kClasses; ++c) P.class_limit[c] = smem_class_limit(c, ctx->sms);
  // Everything of the load runs on the context's build stream, which is then
  // synchronized: other streams' work is not waited for.
  cudaStream_t st = R->build;
  launch_build_layout(P, st, ctx->sms, &ctx->launches);
  launch_build_preds(P, R->n_succ, R->pred_off, R->cursor, R->scan_tmp, st, ctx->sms, &ctx->launches);
  launch_build_events(P, R->ev_off, R->events, R->scan_tmp, st, ctx->sms, &ctx->launches);
  launch_build_meta(P, R->meta, st, ctx->sms, &ctx->launches);
  if (cudaStreamSynchronize(st) != cudaSuccess || cudaGetLastError() != cudaSuccess) {
    free_program(R);
    return GPA_ERR_CUDA;
  }
  const gpa_pid pid = ctx->next_pid++;
  ctx->progs[pid] = R;
  *out = pid;
  return GPA_OK;
}

gpa_status gpa_unload_program(gpa_ctx* ctx, gpa_pid pid) {
  ProgramRec* R = find(ctx, pid);
  if (!R) return GPA_ERR_NO_PROGRAM;
  cudaDeviceSynchronize();
  free_program(R);
  ctx->progs.erase(pid);
  return GPA_OK;
}

gpa_status gpa_unload_program_async(gpa_ctx* ctx, gpa_pid pid, gpa_stream stream) {
  ProgramRec* R = find(ctx, pid);
  if (!R) return GPA_ERR_NO_PROGRAM;
  cudaStream_t st = (cudaStream_t)stream;
  // The captured graph, if any, is freed when an in-flight launch completes.
  if (R->step_exec) cudaGraphExecDestroy(R->step_exec);
  R->step_exec = nullptr;
  gpa_status s = GPA_OK;
  for (void* p : {R->block, (void*)R->xbuf, R->xout, (void*)R->launch})
    if (p && cudaFreeAsync(p, st) != cudaSuccess) s = GPA_ERR_CUDA;
  delete R;
  ctx->progs.erase(pid);
  return s;
}

gpa_status gpa_reset_counts(gpa_ctx* ctx, gpa_pid pid, gpa_stream stream) {
  ProgramRec* R = find(ctx, pid);
  if (!R) return GPA_ERR_NO_PROGRAM;
  cudaStream_t st = (cudaStream_t)stream;
  CK(cudaMemsetAsync(R->P.cnt, 0, (size_t)R->P.ni * kCnt * sizeof(unsigned long long), st));
  CK(cudaMemsetAsync(R->P.stats, 0, SS_N * sizeof(unsigned long long), st));
  return GPA_OK;
}

gpa_status gpa_copy_counts(gpa_ctx* ctx, gpa_pid pid, uint64_t* dev_dst, gpa_stream stream) {
  ProgramRec* R = find(ctx, pid);
  if (!R) return GPA_ERR_NO_PROGRAM;
  if (!dev_dst || (reinterpret_cast<uintptr_t>(dev_dst) & 7u)) return GPA_ERR_INVALID_ARG;
  CK(cudaMemcpyAsync(dev_dst, R->P.cnt, (size_t)R->P.ni * kCnt * sizeof(unsigned long long),
                     cudaMemcpyDeviceToDevice, (cudaStream_t)stream));
  return GPA_OK;
}

gpa_status gpa_set_counts(gpa_ctx* ctx, gpa_pid pid, const uint64_t* dev_counts, uint64_t invalid,
                          gpa_stream stream) {
  ProgramRec* R = find(ctx, pid);
  if (!R) return GPA_ERR_NO_PROGRAM;
  if (!dev_counts || (reinterpret_cast<uintptr_t>(dev_counts) & 7u)) return GPA_ERR_INVALID_ARG;
  cudaStream_t st = (cudaStream_t)stream;
  CK(cudaMemsetAsync(R->P.stats, 0, SS_N * sizeof(unsigned long long), st));
  CK(cudaMemcpyAsync(R->P.cnt, dev_counts, (size_t)R->P.ni * kCnt * sizeof(unsigned long long),
                     cudaMemcpyDeviceToDevice, st));
  launch_store_u64(&R->P.stats[SS_INVALID], (unsigned long long)invalid, st, &ctx->launches);
  CK(cudaGetLastError());
  return GPA_OK;
}

gpa_status gpa_ingest_samples(gpa_ctx* ctx, gpa_pid pid, const uint64_t* dev_samples, size_t n, gpa_stream stream) {
  ProgramRec* R = find(ctx, pid);
  if (!R) return GPA_ERR_NO_PROGRAM;
  if (n == 0) return GPA_OK;
  if (!dev_samples || (reinterpret_cast<uintptr_t>(dev_samples) & 7u)) return GPA_ERR_INVALID_ARG;
  launch_histogram(R->P, dev_samples, n, (cudaStream_t)stream, ctx->sms, &ctx->launches, ctx->opts.hist_variant,
                   ctx->opts.hist_chunk);
  CK(cudaGetLastError());
  return GPA_OK;
}

constexpr int kHostIngestCtas = 32;  // SMs an ingest over the host link takes

gpa_status gpa_ingest_host_samples(gpa_ctx* ctx, gpa_pid pid, const uint64_t* host, size_t n, gpa_stream stream) {
  ProgramRec* R = find(ctx, pid);
  if (!R) return GPA_ERR_NO_PROGRAM;
  if (n == 0) return GPA_OK;
  if (!host) return GPA_ERR_INVALID_ARG;
  cudaStream_t st = (cudaStream_t)stream;
  // Pinned host memory that this device can address (page-locked allocations
  // are mapped under unified addressing) is read by the aggregation kernel
  // itself over the host link: no staging buffer, no copy engine. The link
  // (about 210 GB/s) needs far fewer SMs than HBM (about 23 GB/s an SM), so the
  // launch takes at most kHostIngestCtas of them and leaves the rest to other
  // work, such as the blame of the batch before. Other memory goes through the
  // staging buffers.
  cudaPointerAttributes at{};
  int dev = -1;
  if (cudaPointerGetAttributes(&at, host) == cudaSuccess && at.type == cudaMemoryTypeHost && at.devicePointer &&
      cudaGetDevice(&dev) == cudaSuccess && dev == ctx->device) {
    launch_histogram(R->P, static_cast<const uint64_t*>(at.devicePointer), n, st,
                     std::min(ctx->sms, kHostIngestCtas), &ctx->launches, ctx->opts.hist_variant,
                     ctx->opts.hist_chunk);
    CK(cudaGetLastError());
    return GPA_OK;
  }
  cudaGetLastError();  // a failed query is not an error here
  if (!ctx->stage[0]) {
    ctx->stage_n = kStageSamples;
    for (int k = 0; k < 2; ++k) {
      if (cudaMalloc(&ctx->stage[k], ctx->stage_n * sizeof(uint64_t)) != cudaSuccess) return GPA_ERR_OOM;
      CK(cudaEventCreateWithFlags(&ctx->ev_copied[k], cudaEventDisableTiming));
      CK(cudaEventCreateWithFlags(&ctx->ev_used[k], cudaEventDisableTiming));
      CK(cudaEventRecord(ctx->ev_used[k], st));
    }
    CK(cudaStreamCreateWithFlags(&ctx->copy_stream, cudaStreamNonBlocking));
  }
  // Double buffering: the copy of chunk c+1 overlaps the aggregation of chunk c.
  CK(cudaStreamWaitEvent(ctx->copy_stream, ctx->ev_used[0], 0));
  CK(cudaStreamWaitEvent(ctx->copy_stream, ctx->ev_used[1], 0));
  size_t off = 0;
  for (int c = 0; off < n; ++c) {
    const int k = c & 1;
    const size_t m = std::min(ctx->stage_n, n - off);
    CK(cudaStreamWaitEvent(ctx->copy_stream, ctx->ev_used[k], 0));
    CK(cudaMemcpyAsync(ctx->stage[k], host + off, m * sizeof(uint64_t), cudaMemcpyHostToDevice, ctx->copy_stream));
    CK(cudaEventRecord(ctx->ev_copied[k], ctx->copy_stream));
    CK(cudaStreamWaitEvent(st, ctx->ev_copied[k], 0));
    launch_histogram(R->P, ctx->stage[k], m, st, ctx->sms, &ctx->launches, ctx->opts.hist_variant,
                     ctx->opts.hist_chunk);
    CK(cudaEventRecord(ctx->ev_used[k], st));
    off += m;
  }
  CK(cudaGetLastError());
  return GPA_OK;
}

// Steps (b)-(c) on stream st. With order_scratch, waits for and marks the
// context's shared search scratch (a captured step does this around its
// graph launch instead).
static gpa_status blame_body(gpa_ctx* ctx, ProgramRec* R, cudaStream_t st, bool order_scratch) {
  // per-step counters: general searches, largest search, sweeps, raw edges, queues
  CK(cudaMemsetAsync(R->P.stats + SS_GENERAL, 0, sizeof(unsigned long long) * 3, st));
  CK(cudaMemsetAsync(R->P.stats + SS_RAW_N, 0, sizeof(unsigned long long) * (SS_N - SS_RAW_N), st));
  // The search scratch and the side streams are shared by the context's
  // programs: order their users.
  if (order_scratch) CK(cudaStreamWaitEvent(st, ctx->scratch_ev, 0));
  launch_dataflow(R->P, ctx->arch, ctx->opts.max_fixpoint_sweeps, ctx->opts.reach_schedule, &ctx->fork, st, ctx->sms,
                  &ctx->launches);
  launch_blame(R->P, ctx->arch, ctx->tier, &ctx->fork, ctx->opts.max_sources_per_use, R->scan_tmp, st, ctx->sms,
               &ctx->launches);
  if (order_scratch) CK(cudaEventRecord(ctx->scratch_ev, st));
  CK(cudaGetLastError());
  return GPA_OK;
}

gpa_status gpa_blame(gpa_ctx* ctx, gpa_pid pid, gpa_stream stream) {
  ProgramRec* R = find(ctx, pid);
  if (!R) return GPA_ERR_NO_PROGRAM;
  return blame_body(ctx, R, (cudaStream_t)stream, true);
}

// The counting run of the searches (P.diag = 1) behind gpa_dependency_coverage
// and gpa_export_unpruned_edges; h receives the stats words.
static gpa_status coverage_run(gpa_ctx* ctx, ProgramRec* R, cudaStream_t st, int diag, unsigned long long* h) {
  Prog D = R->P;
  D.diag = diag;
  D.xedges = R->xbuf;
  D.xcap = diag == 2 ? R->xbuf_cap : 0;
  if (diag == 1) CK(cudaMemsetAsync(D.cov_cnt, 0, sizeof(uint32_t) * (size_t)std::max(R->n_use, 1), st));
  CK(cudaMemsetAsync(D.stats + SS_GENERAL, 0, sizeof(unsigned long long) * 3, st));
  CK(cudaMemsetAsync(D.stats + SS_RAW_N, 0, sizeof(unsigned long long) * (SS_N - SS_RAW_N), st));
  CK(cudaStreamWaitEvent(st, ctx->scratch_ev, 0));
  launch_dataflow(D, ctx->arch, ctx->opts.max_fixpoint_sweeps, ctx->opts.reach_schedule, &ctx->fork, st, ctx->sms,
                  &ctx->launches);
  launch_coverage(D, ctx->arch, ctx->tier, &ctx->fork, st, ctx->sms, &ctx->launches);
  CK(cudaEventRecord(ctx->scratch_ev, st));
  CK(cudaGetLastError());
  CK(cudaStreamSynchronize(st));
  CK(cudaMemcpy(h, D.stats, sizeof(unsigned long long) * SS_N, cudaMemcpyDeviceToHost));
  return status_from(h[SS_STATUS]);
}

gpa_status gpa_dependency_coverage(gpa_ctx* ctx, gpa_pid pid, gpa_stream stream, int64_t* out) {
  ProgramRec* R = find(ctx, pid);
  if (!R) return GPA_ERR_NO_PROGRAM;
  if (!out) return GPA_ERR_INVALID_ARG;
  unsigned long long h[SS_N];
  const gpa_status s = coverage_run(ctx, R, (cudaStream_t)stream, 1, h);
  out[0] = (int64_t)h[SS_COV];
  out[1] = (int64_t)h[SS_COV + 1];
  out[2] = (int64_t)h[SS_COV + 2];
  return s;
}

// The ordered export's arrays in xout: seven columns of xout_cap int32 (the last is
// scratch: ids, then ni + 1 offsets, ni cursors and the list of large buckets), then
// the bytes.
static ExportOut export_out(const ProgramRec* R, int32_t** ids) {
  int32_t* p = static_cast<int32_t*>(R->xout);
  const size_t c = (size_t)R->xout_cap;
  if (ids) *ids = p + 6 * c;
  return ExportOut{p, p + c, p + 2 * c, p + 3 * c, p + 4 * c, p + 5 * c,
                   reinterpret_cast<uint8_t*>(p + 7 * c + 2 * (size_t)R->P.ni + 1 + export_big_ints(R->xout_cap))};
}

gpa_status gpa_export_unpruned_edges(gpa_ctx* ctx, gpa_pid pid, gpa_stream stream, int64_t* n_edges) {
  ProgramRec* R = find(ctx, pid);
  if (!R) return GPA_ERR_NO_PROGRAM;
  if (!n_edges) return GPA_ERR_INVALID_ARG;
  cudaStream_t st = (cudaStream_t)stream;
  unsigned long long h[SS_N];
  *n_edges = 0;
  R->x_n = 0;
  auto grow = [&](int64_t need) {
    if (R->xbuf) cudaFreeAsync(R->xbuf, st);
    R->xbuf = static_cast<int4*>(pool_alloc(ctx, sizeof(int4) * 2 * (size_t)need, st));
    R->xbuf_cap = R->xbuf ? need : 0;
    return R->xbuf != nullptr;
  };
  // A first buffer of an edge per use entry (32 MB at most) holds most exports;
  // the run counts every edge, so a buffer that proves too small (or could not be
  // had) is made to measure and the run repeated. The buffer is kept.
  if (!R->xbuf) grow(std::min<int64_t>(std::max(R->n_use, 1), (int64_t)1 << 20));
  gpa_status s = coverage_run(ctx, R, st, 2, h);
  if (s) return s;
  if ((int64_t)h[SS_XN] > R->xbuf_cap) {
    if (!grow((int64_t)h[SS_XN])) return GPA_ERR_OOM;
    s = coverage_run(ctx, R, st, 2, h);
    if (s) return s;
  }
  const int64_t n = std::min<int64_t>((int64_t)h[SS_XN], R->xbuf_cap);
  if (n > INT32_MAX) {  // beyond the device's 32-bit offsets: ordered on the host (gpa_get_unpruned_edges)
    R->x_n = *n_edges = n;
    return GPA_OK;
  }
  if (n > R->xout_cap) {
    if (R->xout) cudaFreeAsync(R->xout, st);
    R->xout = pool_alloc(
        ctx, (size_t)n * 29 + sizeof(int32_t) * (2 * (size_t)R->P.ni + 1 + (size_t)export_big_ints(n)), st);
    R->xout_cap = R->xout ? n : 0;
    if (!R->xout) return GPA_ERR_OOM;
  }
  int32_t* ids = nullptr;
  const ExportOut out = export_out(R, &ids);
  int32_t* off = ids + R->xout_cap;
  int32_t* cursor = off + R->P.ni + 1;
  launch_order_export(R->xbuf, n, R->P.ni, off, cursor, ids, cursor + R->P.ni, out, R->scan_tmp, st, ctx->sms,
                      &ctx->launches);
  CK(cudaGetLastError());
  CK(cudaStreamSynchronize(st));
  R->x_n = n;
  *n_edges = n;
  return GPA_OK;
}

gpa_status gpa_get_unpruned_edges(gpa_ctx* ctx, gpa_pid pid, int32_t* use, int32_t* def, int32_t* res,
                                  int32_t* dmin, int32_t* back_edges, int32_t* dlong, uint8_t* dom, gpa_stream stream) {
  ProgramRec* R = find(ctx, pid);
  if (!R) return GPA_ERR_NO_PROGRAM;
  CK(cudaStreamSynchronize((cudaStream_t)stream));
  const size_t n = (size_t)R->x_n;
  if (!n) return GPA_OK;
  if (n > INT32_MAX) {
    std::vector<int4> x(2 * n);
    CK(cudaMemcpy(x.data(), R->xbuf, sizeof(int4) * x.size(), cudaMemcpyDeviceToHost));
    std::vector<size_t> order(n);
    for (size_t k = 0; k < n; ++k) order[k] = k;
    std::sort(order.begin(), order.end(), [&](size_t a, size_t b) {
      const int4 &p = x[2 * a], &q = x[2 * b];
      return p.x != q.x ? p.x < q.x : p.z != q.z ? p.z < q.z : p.y < q.y;
    });
    for (size_t t = 0; t < n; ++t) {
      const int4 a = x[2 * order[t]], b = x[2 * order[t] + 1];
      if (use) use[t] = a.x;
      if (def) def[t] = a.y;
      if (res) res[t] = a.z;
      if (dmin) dmin[t] = a.w;
      if (back_edges) back_edges[t] = b.x;
      if (dlong) dlong[t] = b.y;
      if (dom) dom[t] = (uint8_t)b.z;
    }
    return GPA_OK;
  }
  const ExportOut x = export_out(R, nullptr);
  int32_t* const dst[6] = {use, def, res, dmin, back_edges, dlong};
  const int32_t* const src[6] = {x.use, x.def, x.res, x.dmin, x.back, x.dlong};
  for (int k = 0; k < 6; ++k)
    if (dst[k]) CK(cudaMemcpy(dst[k], src[k], n * sizeof(int32_t), cudaMemcpyDeviceToHost));
  if (dom) CK(cudaMemcpy(dom, x.dom, n, cudaMemcpyDeviceToHost));
  return GPA_OK;
}

gpa_status gpa_step_capture(gpa_ctx* ctx, gpa_pid pid, const uint64_t* dev_samples, size_t n) {
  ProgramRec* R = find(ctx, pid);
  if (!R) return GPA_ERR_NO_PROGRAM;
  if (n && (!dev_samples || (reinterpret_cast<uintptr_t>(dev_samples) & 7u))) return GPA_ERR_INVALID_ARG;
  if (!ctx->capture_stream) CK(cudaStreamCreateWithFlags(&ctx->capture_stream, cudaStreamNonBlocking));
  cudaStream_t cs = ctx->capture_stream;
  const int64_t l0 = ctx->launches;
  CK(cudaStreamBeginCapture(cs, cudaStreamCaptureModeThreadLocal));
  gpa_status s = GPA_OK;
  if (cudaMemsetAsync(R->P.cnt, 0, (size_t)R->P.ni * kCnt * sizeof(unsigned long long), cs) != cudaSuccess ||
      cudaMemsetAsync(R->P.stats, 0, SS_N * sizeof(unsigned long long), cs) != cudaSuccess)
    s = GPA_ERR_CUDA;
  if (!s && n)
    launch_histogram(R->P, dev_samples, n, cs, ctx->sms, &ctx->launches, ctx->opts.hist_variant,
                     ctx->opts.hist_chunk);
  if (!s) s = blame_body(ctx, R, cs, false);
  if (!s) launch_advise(R->P, ctx->arch, cs, &ctx->launches);
  cudaGraph_t g = nullptr;
  const cudaError_t e = cudaStreamEndCapture(cs, &g);
  const int64_t kernels = ctx->launches - l0;
  ctx->launches = l0;  // nothing ran yet
  if (s || e != cudaSuccess || !g) {
    if (g) cudaGraphDestroy(g);
    cudaGetLastError();
    return s ? s : GPA_ERR_CUDA;
  }
  cudaGraphExec_t ex = nullptr;
  const cudaError_t ei = cudaGraphInstantiate(&ex, g, 0);
  cudaGraphDestroy(g);
  if (ei != cudaSuccess) { cudaGetLastError(); return GPA_ERR_CUDA; }
  if (R->step_exec) cudaGraphExecDestroy(R->step_exec);
  R->step_exec = ex;
  R->step_launches = kernels;
  return GPA_OK;
}

gpa_status gpa_step_launch(gpa_ctx* ctx, gpa_pid pid, gpa_stream stream) {
  ProgramRec* R = find(ctx, pid);
  if (!R) return GPA_ERR_NO_PROGRAM;
  if (!R->step_exec) return GPA_ERR_INVALID_ARG;
  cudaStream_t st = (cudaStream_t)stream;
  CK(cudaStreamWaitEvent(st, ctx->scratch_ev, 0));
  CK(cudaGraphLaunch(R->step_exec, st));
  CK(cudaEventRecord(ctx->scratch_ev, st));
  ctx->launches += R->step_launches;
  return GPA_OK;
}

static gpa_status copy_advice(gpa_ctx* ctx, ProgramRec* R, const gpa_advice* out, cudaStream_t st) {
  const Prog& P = R->P;
  const size_t nf = P.nf, no = GPA_NUM_OPT;
  OutList L{};
  void* user[kOutItems];
  size_t total = 0;
  auto add = [&](void* dst, const void* src, size_t bytes) {
    if (!dst || !bytes) return;
    L.src[L.n] = src;
    L.bytes[L.n] = (int64_t)bytes;
    user[L.n++] = dst;
    total += (bytes + 15) & ~(size_t)15;
  };
  add(out->totals, P.a_totals, nf * 4 * 8);
  add(out->matched, P.a_matched, nf * no * 8);
  add(out->speedup, P.a_speedup, nf * no * 8);
  add(out->rank, P.a_rank, nf * no * 4);
  add(out->n_hot, P.a_nhot, nf * no * 4);
  add(out->hot, P.a_hot, nf * no * 5 * 6 * 8);
  add(out->loop_active, P.a_loop_active, (size_t)P.nl * 8);
  add(out->loop_matched, P.a_loop_matched, (size_t)P.nl * 8);
  add(out->loop_speedup, P.a_loop_speedup, (size_t)P.nl * 8);
  add(out->line_stall, P.a_line_stall, (size_t)P.n_lines * 8);
  add(out->line_latency, P.a_line_lat, (size_t)P.n_lines * 8);
  add(out->par_match, P.a_par_match, nf * 2 * 4);
  add(out->par_speedup, P.a_par_speedup, nf * 2 * 8);
  add(out->par_warps, P.a_par_warps, nf * 4 * 8);
  add(out->par_limit, P.a_par_limit, nf * 4);
  // Page-locked destinations that this device can address are written by one
  // kernel; others of up to kAdviceStage in all through page-locked staging, and
  // larger ones array by array.
  bool direct = true, on_host = true;
  for (int k = 0; k < L.n; ++k) {
    // (the last byte too: a caller may have registered only part of an array)
    cudaPointerAttributes at{}, end{};
    const bool known = cudaPointerGetAttributes(&at, user[k]) == cudaSuccess;
    direct = direct && known && at.type == cudaMemoryTypeHost && at.devicePointer &&
             (reinterpret_cast<uintptr_t>(at.devicePointer) & 3u) == 0 &&
             cudaPointerGetAttributes(&end, static_cast<const char*>(user[k]) + L.bytes[k] - 1) == cudaSuccess &&
             end.type == cudaMemoryTypeHost &&
             end.devicePointer == static_cast<char*>(at.devicePointer) + L.bytes[k] - 1;
    on_host = on_host && known && at.type != cudaMemoryTypeDevice;
    L.dst[k] = at.devicePointer;
  }
  cudaGetLastError();  // a failed query is not an error here
  bool staged = false;
  if (!direct && on_host && total <= kAdviceStage) {
    if (!ctx->advice_stage && cudaMallocHost(&ctx->advice_stage, kAdviceStage) != cudaSuccess) {
      cudaGetLastError();
      ctx->advice_stage = nullptr;
    }
    staged = ctx->advice_stage != nullptr;
    size_t off = 0;
    for (int k = 0; k < L.n && staged; ++k) {
      L.dst[k] = ctx->advice_stage + off;
      off += ((size_t)L.bytes[k] + 15) & ~(size_t)15;
    }
  }
  if (direct || staged) {
    launch_copy_out(L, st, &ctx->launches);
    CK(cudaGetLastError());
  } else {
    for (int k = 0; k < L.n; ++k)
      CK(cudaMemcpyAsync(user[k], L.src[k], (size_t)L.bytes[k], cudaMemcpyDeviceToHost, st));
  }
  CK(cudaStreamSynchronize(st));
  if (staged)
    for (int k = 0; k < L.n; ++k) std::memcpy(user[k], L.dst[k], (size_t)L.bytes[k]);
  return GPA_OK;
}

static_assert(sizeof(LaunchRec) == sizeof(gpa_launch_stats) && offsetof(gpa_launch_stats, threads_per_block) == 8 &&
                  offsetof(LaunchRec, threads) == 8 && offsetof(gpa_launch_stats, smem_per_block) == 16 &&
                  offsetof(LaunchRec, smem) == 16,
              "LaunchRec mirrors gpa_launch_stats");

gpa_status gpa_set_launch_stats(gpa_ctx* ctx, gpa_pid pid, const gpa_launch_stats* stats, const gpa_sm_model* sm) {
  ProgramRec* R = find(ctx, pid);
  if (!R) return GPA_ERR_NO_PROGRAM;
  Prog& P = R->P;
  if (stats) {
    if (!sm || sm->n_sms < 1 || sm->schedulers_per_sm < 1 || sm->max_warps_per_sm < 1 || sm->max_blocks_per_sm < 1 ||
        sm->regs_per_sm < 1 || sm->reg_alloc_unit < 1 || sm->smem_per_sm < 1 || sm->smem_alloc_unit < 1 ||
        sm->smem_reserved_per_block < 0)
      return GPA_ERR_INVALID_ARG;
    for (int f = 0; f < P.nf; ++f) {
      const gpa_launch_stats& L = stats[f];
      if (L.blocks < 1 || L.threads_per_block < 1 || L.threads_per_block > 1024 || L.regs_per_thread < 0 ||
          L.regs_per_thread > 255 || L.smem_per_block < 0 || L.reserved != 0)
        return GPA_ERR_INVALID_ARG;
    }
  }
  // Kernels of earlier calls may read the old statistics; a captured step
  // holds the old ones and is dropped (capture it again).
  CK(cudaDeviceSynchronize());
  if (R->step_exec) {
    cudaGraphExecDestroy(R->step_exec);
    R->step_exec = nullptr;
  }
  if (!stats) {
    P.launch = nullptr;
    return GPA_OK;
  }
  const size_t bytes = sizeof(LaunchRec) * (size_t)std::max(P.nf, 1);
  if (!R->launch) R->launch = static_cast<LaunchRec*>(pool_alloc(ctx, bytes, ctx->build_stream));
  if (!R->launch) return GPA_ERR_OOM;
  CK(cudaMemcpyAsync(R->launch, stats, sizeof(LaunchRec) * (size_t)P.nf, cudaMemcpyHostToDevice, ctx->build_stream));
  CK(cudaStreamSynchronize(ctx->build_stream));
  P.launch = R->launch;
  P.sm = SmModel{sm->n_sms, sm->schedulers_per_sm, sm->max_warps_per_sm, sm->max_blocks_per_sm, sm->regs_per_sm,
                 sm->reg_alloc_unit, sm->smem_per_sm, sm->smem_alloc_unit, sm->smem_reserved_per_block};
  return GPA_OK;
}

gpa_status gpa_sm_model_of_device(int device, gpa_sm_model* out) {
  if (!out) return GPA_ERR_INVALID_ARG;
  cudaDeviceProp d{};
  CK(cudaGetDeviceProperties(&d, device));
  out->n_sms = d.multiProcessorCount;
  out->schedulers_per_sm = 4;
  out->max_warps_per_sm = d.maxThreadsPerMultiProcessor / 32;
  out->max_blocks_per_sm = d.maxBlocksPerMultiProcessor;
  out->regs_per_sm = d.regsPerMultiprocessor;
  out->reg_alloc_unit = 256;
  out->smem_per_sm = (int32_t)d.sharedMemPerMultiprocessor;
  out->smem_alloc_unit = 128;
  out->smem_reserved_per_block = (int32_t)d.reservedSharedMemPerBlock;
  return GPA_OK;
}

gpa_status gpa_advise(gpa_ctx* ctx, gpa_pid pid, const gpa_advice* out, gpa_stream stream) {
  ProgramRec* R = find(ctx, pid);
  if (!R) return GPA_ERR_NO_PROGRAM;
  cudaStream_t st = (cudaStream_t)stream;
  launch_advise(R->P, ctx->arch, st, &ctx->launches);
  CK(cudaGetLastError());
  if (out) return copy_advice(ctx, R, out, st);
  return GPA_OK;
}

gpa_status gpa_get_advice(gpa_ctx* ctx, gpa_pid pid, const gpa_advice* out, gpa_stream stream) {
  ProgramRec* R = find(ctx, pid);
  if (!R) return GPA_ERR_NO_PROGRAM;
  if (!out) return GPA_ERR_INVALID_ARG;
  return copy_advice(ctx, R, out, (cudaStream_t)stream);
}

gpa_status gpa_sync_status(gpa_ctx* ctx, gpa_pid pid, gpa_stream stream, int64_t* info) {
  ProgramRec* R = find(ctx, pid);
  if (!R) return GPA_ERR_NO_PROGRAM;
  cudaStream_t st = (cudaStream_t)stream;
  unsigned long long h[SS_N];
  CK(cudaStreamSynchronize(st));
  CK(cudaMemcpy(h, R->P.stats, sizeof h, cudaMemcpyDeviceToHost));
  if (info) {
    info[0] = (int64_t)h[SS_INVALID];
    info[1] = (int64_t)h[SS_GENERAL];
    info[2] = (int64_t)h[SS_MAX_NODES];
    info[3] = (int64_t)h[SS_SWEEPS];
    info[4] = (int64_t)h[SS_OVF_N];
    // each search once: handed on by the lanes, or queued straight for a larger tier
    info[5] = (int64_t)(h[SS_OVF2_N] + h[SS_HINT3_N] + h[SS_WIDE_N] + h[SS_DIRECT_N]);
    for (int c = 0; c < kClasses; ++c)
      info[5] += (int64_t)std::min<unsigned long long>(h[SS_A1_N + c], (unsigned long long)R->P.class_limit[c]);
    info[6] = (int64_t)(h[SS_MAX_TASK] & 0x7FFFFFFFull);     // use of the largest search
    info[7] = (int64_t)((h[SS_MAX_TASK] >> 31) & 0x1FFull);  // its resource
  }
  return status_from(h[SS_STATUS]);
}

gpa_status gpa_get_search_profile(gpa_ctx* ctx, gpa_pid pid, uint64_t* out, gpa_stream stream) {
  ProgramRec* R = find(ctx, pid);
  if (!R) return GPA_ERR_NO_PROGRAM;
  if (!out) return GPA_ERR_INVALID_ARG;
  CK(cudaStreamSynchronize((cudaStream_t)stream));
  CK(cudaMemcpy(out, R->P.stats + SS_PHASE, 42 * sizeof(uint64_t), cudaMemcpyDeviceToHost));
  CK(cudaMemcpy(out + 42, R->P.stats + SS_SIZE_CYC, 16 * sizeof(uint64_t), cudaMemcpyDeviceToHost));
  CK(cudaMemcpy(out + 58, R->P.stats + SS_FAILBITS, sizeof(uint64_t), cudaMemcpyDeviceToHost));
  return GPA_OK;
}

gpa_status gpa_get_counts(gpa_ctx* ctx, gpa_pid pid, uint64_t* counts, uint64_t* invalid, gpa_stream stream) {
  ProgramRec* R = find(ctx, pid);
  if (!R) return GPA_ERR_NO_PROGRAM;
  cudaStream_t st = (cudaStream_t)stream;
  CK(cudaStreamSynchronize(st));
  if (counts) CK(cudaMemcpy(counts, R->P.cnt, (size_t)R->P.ni * kCnt * 8, cudaMemcpyDeviceToHost));
  if (invalid) CK(cudaMemcpy(invalid, R->P.stats + SS_INVALID, 8, cudaMemcpyDeviceToHost));
  return GPA_OK;
}

gpa_status gpa_get_reaching(gpa_ctx* ctx, gpa_pid pid, uint32_t* rin, uint32_t* rout, gpa_stream stream) {
  ProgramRec* R = find(ctx, pid);
  if (!R) return GPA_ERR_NO_PROGRAM;
  CK(cudaStreamSynchronize((cudaStream_t)stream));
  if (rin) CK(cudaMemcpy(rin, R->P.rin, (size_t)R->P.nb * kWords * 4, cudaMemcpyDeviceToHost));
  if (rout) CK(cudaMemcpy(rout, R->P.rout, (size_t)R->P.nb * kWords * 4, cudaMemcpyDeviceToHost));
  return GPA_OK;
}

gpa_status gpa_get_blame(gpa_ctx* ctx, gpa_pid pid, uint64_t* blame, gpa_stream stream) {
  ProgramRec* R = find(ctx, pid);
  if (!R) return GPA_ERR_NO_PROGRAM;
  if (!blame) return GPA_ERR_INVALID_ARG;
  CK(cudaStreamSynchronize((cudaStream_t)stream));
  CK(cudaMemcpy(blame, R->P.blame, (size_t)R->P.ni * kCnt * 8, cudaMemcpyDeviceToHost));
  return GPA_OK;
}

gpa_status gpa_get_edges(gpa_ctx* ctx, gpa_pid pid, int64_t* n_edges, int64_t cap, int32_t* use, int32_t* def,
                         int32_t* dmin, int32_t* dlong, uint32_t* flags, uint64_t* share, gpa_stream stream) {
  ProgramRec* R = find(ctx, pid);
  if (!R) return GPA_ERR_NO_PROGRAM;
  if (!n_edges) return GPA_ERR_INVALID_ARG;
  CK(cudaStreamSynchronize((cudaStream_t)stream));
  int32_t total = 0;
  CK(cudaMemcpy(&total, R->P.edge_off + R->P.ni, 4, cudaMemcpyDeviceToHost));
  if (total > R->P.edge_cap) total = (int32_t)R->P.edge_cap;
  *n_edges = total;
  const size_t m = (size_t)std::min<int64_t>(total, cap < 0 ? 0 : cap);
  if (m) {
    if (use) CK(cudaMemcpy(use, R->P.e_use, m * 4, cudaMemcpyDeviceToHost));
    if (def) CK(cudaMemcpy(def, R->P.e_def, m * 4, cudaMemcpyDeviceToHost));
    if (dmin) CK(cudaMemcpy(dmin, R->P.e_dmin, m * 4, cudaMemcpyDeviceToHost));
    if (dlong) CK(cudaMemcpy(dlong, R->P.e_dlong, m * 4, cudaMemcpyDeviceToHost));
    if (flags) CK(cudaMemcpy(flags, R->P.e_flags, m * 4, cudaMemcpyDeviceToHost));
    if (share) CK(cudaMemcpy(share, R->P.e_share, m * 8 * 8, cudaMemcpyDeviceToHost));
  }
  return GPA_OK;
}

int64_t gpa_launch_count(gpa_ctx* ctx) { return ctx ? ctx->launches : -1; }

}  // extern "C"
