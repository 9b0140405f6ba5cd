// Internal device-side layout and helpers of libgpa (not part of the C ABI).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "gpa.h"

namespace gpa {

constexpr int kNumRes = 268;     // R0..R254, P0..P6, B0..B5
constexpr int kPredBase = 255;
constexpr int kBarBase = 262;
constexpr int kWords = 9;        // 268 bits in 32-bit words
constexpr int kEvBuckets = 16;   // event segments per block: resources by r mod 16
__host__ __device__ inline int ev_bucket(int r) { return r & (kEvBuckets - 1); }
constexpr int kCnt = 24;         // counters per instruction: class * 2 + latency flag
constexpr uint16_t kAllLits = 0xFFFF;
constexpr int kLaneNodes = 128;  // most nodes of a one-lane search (first and second tier)
constexpr int kMaxLayers = 8;    // back-edge layers for longest paths (K <= 7)
constexpr int kMaxSrc = 64;      // merged sources per stalled use in the thread-per-use kernels
constexpr int kBigSrc = 2048;    // merged sources per stalled use (hard upper bound; beyond kMaxSrc
                                 // a CTA per use with shared-memory arrays)

// Bits of the per-program device status word.
enum : unsigned long long {
  ST_NOT_CONVERGED = 1, ST_CAPACITY = 2, ST_TIMEOUT = 4, ST_OVERFLOW = 8
};
// Slots of the per-program stats array (unsigned long long).
enum {
  SS_INVALID = 0, SS_GENERAL = 1, SS_MAX_NODES = 2, SS_SWEEPS = 3, SS_STATUS = 4,
  SS_RAW_N = 5, SS_QUEUE_N = 6, SS_QUEUE_HEAD = 7, SS_OVF_N = 8, SS_OVF_HEAD = 9, SS_OVF2_N = 10,
  SS_OVF2_HEAD = 11, SS_MAX_TASK = 12,
  // Per-tier search phase cycles (3 tiers x 6; the fourth tier adds to the
  // third's), filled only when built with -DGPA_PHASE_TIMING: graph,
  // distances, sources, rule 2, longest paths, and the count of rule-2
  // reachability runs.
  // With -DGPA_PHASE_TIMING also: searches by log2 of their node count (16
  // slots) and the searches that needed pass B (1 slot).
  // And the slowest search: (cycles << 20 | nodes), its rule-2 runs and the
  // cycles of its five phases.
  SS_PHASE = 13, SS_SIZES = 31, SS_PASSB = 47, SS_SLOW = 48,
  SS_DIRECT_N = 55,  // searches queued straight for the CTAs beyond max_search_nodes (queues 4 and 7)
  // 56, 57: unused
  SS_SIZE_CYC = 58,  // with -DGPA_PHASE_TIMING: cycles of the searches by log2 of their node count (16)
  SS_HINT3_N = 74,   // searches beyond a class's limit (from the top of queue[3])
  SS_FAILBITS = 75,  // why a step reported GPA_ERR_CAPACITY: the last search tier ran out of
                     // 1 nodes, 2 edges, 3 occurrences, 4 sources, 5 back-edge layers,
                     // 6 hash rounds; 8 queue, 9 sources per use, 10 merged edges,
                     // 11 distance range, 12 raw edges, 13 no path length
  SS_BIG_N = 76,     // uses with more than kMaxSrc distinct sources (listed in big_use)
  SS_COV = 77,       // gpa_dependency_coverage: stalled uses, single before, single after pruning
  // 80: unused
  SS_XN = 81,        // unpruned edges written by the export pass
  SS_HIST_HEAD = 82, // next chunk of the run-aware aggregation kernel (reset before each launch)
  SS_HINT3_HEAD = 83,  // next of them
  SS_T4_N = 84, SS_T4_HEAD = 85,  // searches for the fourth tier (queue[4])
  SS_REACH_CLS = 86,   // next entry of reach_order for each of the staged fixpoint's 4 launches
  SS_SUSE_N = 90,      // entries of suse (the stalled uses of this step)
  // 91: unused
  // searches queued straight for a size class of the shared-memory warps
  SS_A1_N = 92, SS_A1_HEAD = 97,  // kClasses of each
  SS_WIDE_N = 102, SS_WIDE_HEAD = 103,    // searches for the CTAs of 128 threads: known ones (bottom of queue[6])
  SS_WIDE2_N = 104, SS_WIDE2_HEAD = 105,  // and what the shared-memory warps hand on (its top)
  SS_T5_N = 106, SS_T5_HEAD = 107,        // searches beyond 2^18 nodes (queue[7])
  SS_N = 108
};
// Size classes of the shared-memory search warps (k_search_smem.cu), and the
// queue and region of each class's searches known from an earlier step.
constexpr int kClasses = 5;
__host__ __device__ inline int class_nodes(int c, int most) {
  const int n = c < 4 ? 320 << c : 5632;
  return n < most ? n : most;
}
__host__ __device__ constexpr int class_queue(int c) { return c < 3 ? c : c == 3 ? 2 : 5; }
__host__ __device__ constexpr bool class_top(int c) { return c != 2 && c != 4; }
// Values of tier_hint: the queue that a use entry's search belongs to.
enum { kHintLane2 = 2, kHintA1 = 3, kHintWide = kHintA1 + kClasses, kHintCta, kHintGiant };

struct Arch {
  int32_t n_op;
  int32_t lat[GPA_MAX_OPCLASSES];
  uint32_t flags[GPA_MAX_OPCLASSES];
};

// Device view of one loaded program and its per-step buffers.
// One function's launch statistics (the layout of gpa_launch_stats) and the
// SM of the occupancy model (the fields of gpa_sm_model).
struct LaunchRec {
  long long blocks;
  int32_t threads, regs, smem, reserved;
};
// Instructions of an advice tile: 1,024, or 256 for programs of fewer tiles than
// the chip has SMs (a tile is a chain of its warps' passes: Rodinia-shaped step
// 520 us with tiles of 1,024, 497 with 256; thousand-function step 6.63 and
// 6.73 ms, advice over 301 functions 318 and 337 us).
inline int adv_tile_size(int64_t n_instr, int sms) { return n_instr <= 1024ll * sms ? 256 : 1024; }
constexpr int kAdvAcc = 14;     // per-function sums of the advice kernel, and its tiles that are done
// A hotspot candidate of a tile.
struct AdvCand {
  unsigned long long v;
  int32_t def, use, dist, pad;
};
struct SmModel {
  int32_t n_sms, schedulers, max_warps, max_blocks, regs, reg_unit, smem, smem_unit, smem_reserved;
};

struct Prog {
  int32_t nf, ni, nb, nl, n_lines;
  int32_t diag;                   // 1: the searches count sources (gpa_dependency_coverage), 2: they export
                                  // every source (gpa_export_unpruned_edges); both emit no raw edges
  int4* xedges;                   // export: 2 per edge, {use, def, resource, dmin}, {K, dlong, dom, 0}
  int64_t xcap;                   // edges the export buffer holds
  uint32_t* cov_cnt;              // n_use: that run's sources per use entry, before pruning (low 16 bits)
                                  // and kept after pruning (high 16 bits)
  int32_t reach_smem;             // shared memory of the staged fixpoint: the largest need that fits
  int32_t reach_cls[5];           // the staged fixpoint's launches: reach_order[reach_cls[c], reach_cls[c + 1])
  int32_t reach_cls_smem[4];      // and the largest need among them (0: no launch)
  const uint8_t* func_natural;    // nf: 1 when every loop body of the function is a natural loop
  int32_t reach_windowed;         // functions that only the windowed kernel takes (too large for the other two,
                                  // or large with other loops)
  // Fourth search tier, sized for this program's largest function (0 nodes:
  // none): searches that outgrow the context's third tier, a CTA each.
  int32_t t4_nodes, t4_src, t4_ctas;
  int64_t t4_bytes;               // per CTA
  char* t4_arena;                 // t4_ctas * t4_bytes, global memory
  const int32_t* func_instr_off;
  const int32_t* func_block_off;
  const int32_t* func_loop_off;
  const int32_t* block_instr_off;
  const int32_t* succ_off;
  const int32_t* succ;
  const int32_t* pred_off;
  const int32_t* pred;
  const uint8_t* opclass;
  const uint8_t* guard;
  const uint8_t* iflags;          // bit 0 math-library code, 1 call site, 2 in a device function
  const int32_t* line;
  const int32_t* def_off;
  const uint16_t* def_res;
  const int32_t* use_off;
  const uint16_t* use_res;
  const int32_t* block_loop;
  const int32_t* loop_parent;
  const int32_t* loop_header;
  const int32_t* loop_depth;
  const int32_t* instr_block;
  const int32_t* block_func;
  const int32_t* reach_order;     // nf: functions by the staged fixpoint's shared memory need, largest first
  const int32_t* block_minreach;  // nb: smallest block reachable from the block (itself included)
  const int4* block_meta;         // 2 per block: {first instr, end instr, first event, end event},
                                  // {first pred, end pred, first two predecessors or -1} (one
                                  // 32-byte line for the searches)
  const int32_t* ev_off;          // nb * 16 + 1: event segments of (block, resource bucket)
  const uint32_t* events;         // per segment, the defs and unguarded reads of the bucket's
                                  // resources, bottom-up: resource | def << 9 | kind << 10 |
                                  // guard << 12 | position in block << 16
  // step state
  unsigned long long* cnt;        // ni * 24
  unsigned long long* stats;      // SS_N
  uint32_t* def_mask;             // nb * 9: resources defined in the block
  uint32_t* touch_mask;           // nb * 9: resources defined or read by an unguarded instruction (blocks a search
                                  // must scan)
  int32_t* res_maxlat;            // nf * 268: largest latency of any def of the resource in the function
  uint32_t* res_guards;           // nf * 268, right behind res_maxlat: guard literals of the resource's defs in the function
  uint32_t* rin;                  // nb * 9
  uint32_t* rout;                 // nb * 9
  int32_t* head;                  // ni: raw-edge list head per use (-1 = none)
  int4* raw;                      // raw edges: def, next, dmin, dlong | flags << 24
  int64_t raw_cap;
  // General searches. A task is named by its use entry e; tasks[e] = {use,
  // resource | start literal set << 9 | blocked << 25}. Each queue has queue_cap
  // entries: 0 first tier from the bottom (after it the second tier's overflow),
  // first size class of the shared-memory warps from the top; 1 second tier,
  // second class; 2 third class, fourth class; 3 (top) what is beyond a class's limit;
  // 4 CTAs of 512 threads; 5 fifth class; 6 CTAs of 128 threads, what the
  // shared-memory warps hand on; 7 beyond 2^18 nodes. An entry is in one region of a
  // queue at a time, so the two regions never meet.
  int2* tasks;                    // n_use
  int32_t* queue[8];
  int32_t class_limit[kClasses];  // searches a class takes in a step; the rest go to the global-memory warps
  // n_use each: the queue known to hold the entry's search (0: none), kept
  // across steps (a search's size depends only on the program); [1] of the
  // diagnostics' searches, which have no latency bound.
  uint8_t* tier_hint[2];
  int64_t queue_cap;
  int32_t* big_use;               // ni: uses with more than kMaxSrc sources (SS_BIG_N of them)
  int32_t* suse;                  // ni: the stalled uses of this step, SS_SUSE_N of them (any order)
  int32_t* edge_off;              // ni + 1: edges per use, scanned in place
  int32_t* e_use;
  int32_t* e_def;
  int32_t* e_dmin;
  int32_t* e_dlong;
  uint32_t* e_flags;
  unsigned long long* e_share;    // edges * 8
  int64_t edge_cap;
  unsigned long long* blame;      // ni * 24
  // advice: tiles of at most adv_tile instructions of one function
  int32_t adv_tile, adv_tiles;
  const int32_t* adv_tile_off;    // nf + 1: first tile of each function
  const int32_t* adv_tile_func;   // adv_tiles
  AdvCand* adv_tops;              // adv_tiles * 9 * 5
  // one block of adv_zero counters, cleared at once: adv_acc, the loops' own
  // samples, then a_loop_active, a_loop_matched, a_line_stall, a_line_lat
  int64_t adv_zero;
  unsigned long long* adv_acc;    // nf * kAdvAcc
  unsigned long long *adv_own_active, *adv_own_matched;
  unsigned long long* a_totals;   // nf * 4
  unsigned long long* a_matched;  // nf * 8
  double* a_speedup;              // nf * 8
  int32_t* a_rank;                // nf * 8
  int32_t* a_nhot;                // nf * 8
  long long* a_hot;               // nf * 8 * 5 * 6
  unsigned long long* a_loop_active;
  unsigned long long* a_loop_matched;
  double* a_loop_speedup;
  unsigned long long* a_line_stall;
  unsigned long long* a_line_lat;
  // parallel optimizers (Table 2, Eqs. 6-10): launch statistics per function
  // (nullptr: none set) and the SM they ran on
  const LaunchRec* launch;
  SmModel sm;
  int32_t* a_par_match;           // nf * 2
  double* a_par_speedup;          // nf * 2
  double* a_par_warps;            // nf * 4
  int32_t* a_par_limit;           // nf
};

// Arenas of the general (multi-block) search: one search a lane in the first
// two tiers (bytes: shared memory of a warp), per group in the others.
struct SearchArena {
  int32_t nodes, src, layers, warps;  // warps: search groups (the fourth tier's are CTAs)
  int64_t bytes;   // per warp or group
  char* global;    // global-memory tiers: warps * bytes
  int* hash;       // third tier: warps * 2 * nodes ints, empty (-1) between searches; else nullptr
};

__device__ __forceinline__ void set_status(const Prog& P, unsigned long long bits) {
  atomicOr(&P.stats[SS_STATUS], bits);
}
// GPA_ERR_CAPACITY with its reason (bit `why` of SS_FAILBITS).
__device__ __forceinline__ void capacity(const Prog& P, int why) {
  atomicOr(&P.stats[SS_STATUS], (unsigned long long)ST_CAPACITY);
  atomicOr(&P.stats[SS_FAILBITS], 1ull << why);
}

// ---------------------------------------------------------------- Sec. 4 predicate literals
// Literal set: bit i = Pi, bit 7+i = !Pi; kAllLits = the set holds "_".
__device__ __forceinline__ uint16_t add_literal(uint16_t S, int g) {
  if (S == kAllLits || g == 0) return kAllLits;
  S = (uint16_t)(S | (1u << (g - 1)));  // literal 1..7 -> bit 0..6 (Pi), 8..14 -> bit 7..13 (!Pi)
  uint32_t pos = S & 0x7Fu, neg = (S >> 7) & 0x7Fu;
  return (pos & neg) ? kAllLits : S;
}
// Literals of a set that can still matter to a search for a use guarded by
// g through a resource whose defs carry the guard literals `guards`: g
// itself, and each literal whose complement some def may still add (only
// such a literal can complete a Pi / !Pi pair). Dropping the others merges
// literal sets that give every continuation the same coverage outcomes.
__device__ __forceinline__ uint16_t live_literals(uint32_t guards, int g) {
  const uint32_t comp = ((guards & 0x7Fu) << 7) | ((guards >> 7) & 0x7Fu);
  return (uint16_t)(comp | (g ? 1u << (g - 1) : 0u));
}
__device__ __forceinline__ uint16_t keep_literals(uint16_t S, uint16_t live) {
  return S == kAllLits ? S : (uint16_t)(S & live);
}
// "P contains p'": p' in P or "_" in P.
__device__ __forceinline__ bool contains(uint16_t S, int g) {
  if (S == kAllLits) return true;
  if (g == 0) return false;
  return (S >> (g - 1)) & 1u;
}

// Rule 1, opcode pruning: can instruction class op cause stalls of class cls?
__device__ __forceinline__ bool opcode_keeps(const Arch& A, int cls, int op) {
  if (cls == GPA_MEMORY_DEPENDENCY || cls == GPA_CONSTANT_MEMORY_DEPENDENCY) return (A.flags[op] & GPA_F_MEM) != 0;
  if (cls == GPA_SYNC) return (A.flags[op] & GPA_F_SYNC) != 0;
  return true;
}
// Rule 1 for the coverage count: does op survive for some dependency class stalled at j?
__device__ __forceinline__ bool keeps_any(const Prog& P, const Arch& A, int j, int op) {
  const unsigned long long* c = P.cnt + (size_t)j * kCnt;
  return ((c[2 * GPA_EXEC_DEPENDENCY] | c[2 * GPA_EXEC_DEPENDENCY + 1]) && opcode_keeps(A, GPA_EXEC_DEPENDENCY, op)) ||
         ((c[2 * GPA_MEMORY_DEPENDENCY] | c[2 * GPA_MEMORY_DEPENDENCY + 1]) && opcode_keeps(A, GPA_MEMORY_DEPENDENCY, op)) ||
         ((c[2 * GPA_SYNC] | c[2 * GPA_SYNC + 1]) && opcode_keeps(A, GPA_SYNC, op)) ||
         ((c[2 * GPA_CONSTANT_MEMORY_DEPENDENCY] | c[2 * GPA_CONSTANT_MEMORY_DEPENDENCY + 1]) &&
          opcode_keeps(A, GPA_CONSTANT_MEMORY_DEPENDENCY, op));
}
// Later steps queue entry e's search for (at least) the queue `hint`. (An entry's
// search runs in one place at a time.)
__device__ __forceinline__ void raise_hint(const Prog& P, int e, uint32_t hint) {
  uint8_t* h = P.tier_hint[P.diag ? 1 : 0] + e;
  if (*h < hint) *h = (uint8_t)hint;
}
// One unpruned edge for the export (counted only when the buffer is full: the
// host makes it larger and runs the export again).
__device__ __forceinline__ void xemit(const Prog& P, int j, int i, int r, int dmin, int K, int dlong, bool dom) {
  const unsigned long long k = atomicAdd(&P.stats[SS_XN], 1ull);
  if (k >= (unsigned long long)P.xcap) return;
  P.xedges[2 * k] = make_int4(j, i, r, dmin);
  P.xedges[2 * k + 1] = make_int4(K, dlong, dom ? 1 : 0, 0);
}
// Adds a (use entry) contribution to the coverage count (the export has none).
__device__ __forceinline__ void cov_add(const Prog& P, int e, int n_all, int n_kept) {
  if (P.diag != 1) return;
  atomicAdd(&P.cov_cnt[e], (uint32_t)min(n_all, 0xFFFF) | ((uint32_t)min(n_kept, 0xFFFF) << 16));
}

// Def kind of resource r at instruction x: -1 not defined, else 0/1/2.
__device__ __forceinline__ int def_kind(const Prog& P, int x, int r) {
  const int e1 = P.def_off[x + 1];
  for (int e = P.def_off[x]; e < e1; ++e) {
    uint32_t v = P.def_res[e];
    if ((int)(v & 0x1FFu) == r) return (int)((v >> 12) & 3u);
  }
  return -1;
}
__device__ __forceinline__ bool uses_res(const Prog& P, int x, int r) {
  const int e1 = P.use_off[x + 1];
  for (int e = P.use_off[x]; e < e1; ++e)
    if ((int)(P.use_res[e] & 0x1FFu) == r) return true;
  return false;
}

__device__ __forceinline__ bool stalled(const Prog& P, int j) {
  const unsigned long long* c = P.cnt + (size_t)j * kCnt;
  return (c[4] | c[5] | c[6] | c[7] | c[10] | c[11] | c[12] | c[13]) != 0ull;
}

// Raw edge (j <- i through r) onto j's list.
__device__ __forceinline__ void emit_raw(const Prog& P, const Arch& A, int j, int i, int r, int kind, int dmin,
                                         int dlong) {
  uint32_t fl = r >= kBarBase ? 2u : (r >= kPredBase ? 8u : 4u);
  // Write-after-read (Sec. 4, Fig. 6): the variable-latency def reads a
  // register that the use writes, and they are linked through a read barrier.
  if (r >= kBarBase && kind == 2 && (A.flags[P.opclass[i]] & GPA_F_VARLAT)) {
    for (int e = P.def_off[j]; e < P.def_off[j + 1]; ++e) {
      const int rr = P.def_res[e] & 0x1FF;
      if (rr < kPredBase && uses_res(P, i, rr)) { fl |= 1u; break; }
    }
  }
  if (dmin >= (1 << 24) || dlong >= (1 << 24)) { capacity(P, 11); return; }
  const unsigned long long slot = atomicAdd(&P.stats[SS_RAW_N], 1ull);
  if (slot >= (unsigned long long)P.raw_cap) { capacity(P, 12); return; }
  const int next = atomicExch(&P.head[j], (int)slot);
  P.raw[slot] = make_int4(i, next, dmin, dlong | (int)(fl << 24));
}

// ---------------------------------------------------------------- launchers
int grid_for(int64_t n, int threads, int sms);
// The exported edges, ordered (launch_order_export): arrays of n entries.
struct ExportOut {
  int32_t *use, *def, *res, *dmin, *back, *dlong;
  uint8_t* dom;
};
constexpr int kExportRank = 1024;  // most edges of a use that are ordered by comparing each with all
inline int64_t export_big_ints(int64_t n) { return n / kExportRank + 2; }  // the uses with more, and their number
void launch_order_export(const int4* x, int64_t n, int ni, int32_t* off, int32_t* cursor, int32_t* ids, int32_t* big,
                         const ExportOut& out, int32_t* scan_tmp, cudaStream_t st, int sms, int64_t* launches);
void launch_build_layout(const Prog& P, cudaStream_t st, int sms, int64_t* launches);
void launch_store_u64(unsigned long long* p, unsigned long long v, cudaStream_t st, int64_t* launches);
void launch_build_preds(const Prog& P, int n_succ, int32_t* pred_off, int32_t* cursor, int32_t* tmp, cudaStream_t st,
                        int sms, int64_t* launches);
void launch_histogram(const Prog& P, const uint64_t* samples, size_t n, cudaStream_t st, int sms, int64_t* launches,
                      int variant, int hist_chunk);

// Lets kernel func take up to the device's opt-in shared memory per block.
// Every launch and captured graph node of a kernel then sees the same limit
// (each requests only what it uses), whatever ran before it.
// The dynamic limit is the opt-in maximum less the kernel's static shared memory.
template <class F>
inline void allow_max_smem(F func) {
  int dev = 0, optin = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
  cudaFuncAttributes fa{};
  cudaFuncGetAttributes(&fa, func);
  cudaFuncSetAttribute(func, cudaFuncAttributeMaxDynamicSharedMemorySize, optin - (int)fa.sharedSizeBytes);
}

// Shared memory of the staged fixpoint for a function of nbf blocks, ne
// predecessor entries and nlf loops: ROUT (9 words a block) and a row of zeros,
// a 16-byte record per block (16-byte aligned: up to 12 bytes of padding), the
// predecessor CSR, each block's innermost loop, and per loop its parent and two
// 9-word masks (the definitions in its body; those of its body and enclosing
// loops; of the latter also a row of zeros).
__host__ __device__ inline int64_t reach_smem_need(int64_t nbf, int64_t ne, int64_t nlf) {
  return 4 * kWords * (nbf + 1) + 12 + 16 * nbf + 4 * (nbf + 1) + 4 * ne + 4 * nbf + 4 * nlf +
         2 * 4 * kWords * nlf + 4 * kWords;
}
// Shared memory of the fixpoint by function and word: two chunks of 512 records,
// a word per block and a zero, two per loop.
__host__ __device__ inline int64_t reach_words_need(int64_t nbf, int64_t nlf) {
  return 2 * 512 * 16 + 4 * (nbf + 1) + 8 * nlf;
}
// Size classes of the staged fixpoint's launches (upper bounds of the need):
// the larger a function, the fewer warps per SM its launch runs.
constexpr int64_t kReachClassCap[4] = {200 * 1024, 64 * 1024, 28 * 1024, 12 * 1024};
constexpr int64_t kReachSmemCap = 220 * 1024;  // of a CTA per function and word
// Three more streams (and their events) on which the searches queued straight
// for the larger tiers run beside the first two.
struct SearchFork {
  cudaStream_t side[3];
  cudaEvent_t fork, join[3];
};
void launch_dataflow(const Prog& P, const Arch& A, int max_sweeps, int schedule, const SearchFork* fork,
                     cudaStream_t st, int sms, int64_t* launches);
void launch_blame(const Prog& P, const Arch& A, const SearchArena* tiers, const SearchFork* fork, int max_src,
                  int32_t* scan_tmp, cudaStream_t st, int sms, int64_t* launches);
void launch_search(const Prog& P, const Arch& A, const SearchArena* tiers, const SearchFork* fork, cudaStream_t st,
                   int sms, int64_t* launches);
void launch_coverage(const Prog& P, const Arch& A, const SearchArena* tiers, const SearchFork* fork, cudaStream_t st,
                     int sms, int64_t* launches);
int64_t search_arena_bytes(int nodes, int src, int layers, bool own_hash);
int search_lane_width(int nodes);      // lanes of a warp that search, for arenas of so many nodes
int64_t search_lane_bytes(int nodes);  // their arenas, in bytes a warp
void launch_search_lanes(const Prog& P, const Arch& A, const SearchArena& T, int tier, cudaStream_t st,
                         int64_t* launches);
int smem_class_limit(int c, int sms);
void launch_search_smem(const Prog& P, const Arch& A, int most_nodes, int part, cudaStream_t st, int sms,
                        int64_t* launches);
int search_warps_per_sm();  // resident one-warp CTAs of the search kernel per SM (global-memory tiers)
void launch_build_meta(const Prog& P, int4* meta, cudaStream_t st, int sms, int64_t* launches);
void launch_build_events(const Prog& P, int32_t* ev_off, uint32_t* events, int32_t* tmp, cudaStream_t st, int sms,
                         int64_t* launches);
void launch_advise(const Prog& P, const Arch& A, cudaStream_t st, int64_t* launches);
// Copies up to kOutItems device arrays (4-byte multiples) to memory the device
// can write, in one launch.
constexpr int kOutItems = 15;
struct OutList {
  const void* src[kOutItems];
  void* dst[kOutItems];
  int64_t bytes[kOutItems];
  int n;
};
void launch_copy_out(const OutList& L, cudaStream_t st, int64_t* launches);
// Exclusive scan of n int32 values in place over buf[0..n], buf[n] receives the total.
void scan_exclusive_inplace(int32_t* buf, int n, int32_t* tmp, cudaStream_t st, int64_t* launches);
size_t scan_tmp_ints(int n);

}  // namespace gpa
