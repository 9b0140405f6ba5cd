// Step (b)/(c), general backward searches (Sec. 4): immediate sources of a
// stalled use j through resource r whose value may come from outside j's
// block, with the three pruning rules evaluated over the set of source paths.
//
// The search tiers in global memory: one search group per (use, resource) task, a
// warp for what the shared-memory warps leave of their largest classes, a CTA of
// 128 threads for up to 32,768 nodes (max_search_nodes), a CTA of 512 threads for
// up to 2^18 nodes and for what is larger still; searches of up to 64 nodes run one to a lane
// before them (k_search_lanes.cu), those of up to 5,632 one to a warp in shared
// memory (k_search_smem.cu). The graph of (block, literal set) nodes lives
// in the group's arena in global memory. The group's threads scan node blocks in parallel
// through per-block event lists (defs and unguarded reads, bottom-up), insert
// nodes and sources into open-addressing hashes together, relax distances and
// propagate reachability bits over frontiers with atomics, and run the
// layered longest paths as level-synchronous frontiers; rank 0 only resets
// counters between steps.
//
// Node 0 is the part of j's block above j, already scanned by the local pass
// (its sources are settled there). A node's d is the shortest distance from
// the last instruction of its block to j. Pass A grows the graph in distance
// order up to `bound`, the largest latency of any def of r in the function: a
// source farther than that fails rule 3 whatever the rest of the graph holds.
// Only if some source is within its latency does pass B complete the graph,
// which rule 2 and the longest paths need; when pass B adds no node, pass A's
// distances are already those of the whole graph. A CTA's search mostly gets by
// with a part of it (kLayers below).
#include <algorithm>

#include "gpa_internal.cuh"

namespace gpa {

namespace {

constexpr int kInf = 0x3FFFFFFF;
constexpr uint32_t kBackBit = 0x80000000u;
constexpr int kExpanded = 1;

struct Arena {
  int N, E, O, SRC, L;
  int *blk, *S, *wall, *k, *e0, *e1, *fl, *seen, *ord, *tmp, *grp, *q;  // per node
  unsigned long long* dpk;  // (shortest distance << 32) | parent node
  unsigned long long* sdb;  // per source: (shortest distance << 32) | nearest occurrence
  int *dl, *ht, *hused, *eto, *on, *ox, *onext;
  int *wblk, *wpos, *wneed;
  int *si, *sk, *sp, *shead;
  int* ctr;  // 0 nodes, 1 edges, 2 occurrences, 3 hash slots used, 4 overflow, 5 scratch
};

// own_hash: the node hash (2 * N ints) lies in the arena; otherwise it is kept
// apart (SearchArena::hash).
__host__ __device__ inline int64_t arena_bytes(int N, int SRC, int L, bool own_hash) {
  const int64_t E = 2 * (int64_t)N, O = N;
  int64_t ints = 12 * (int64_t)N + (int64_t)L * N + (own_hash ? 2 * (int64_t)N : 0) + N + E + 3 * O + 3 * (int64_t)N +
                 4 * (int64_t)SRC + 8;
  return 8 * (int64_t)N + 8 * (int64_t)SRC + ((ints * 4 + 15) & ~(int64_t)15);
}

__device__ Arena carve(char* base, int* hash, int N, int SRC, int L, int* ctr) {
  Arena a;
  a.N = N; a.E = 2 * N; a.O = N; a.SRC = SRC; a.L = L;
  a.dpk = reinterpret_cast<unsigned long long*>(base);
  a.sdb = a.dpk + N;
  int* p = reinterpret_cast<int*>(base + 8 * (int64_t)N + 8 * (int64_t)SRC);
  int** node_arrays[12] = {&a.blk, &a.S, &a.wall, &a.k, &a.e0, &a.e1, &a.fl, &a.seen, &a.ord, &a.tmp, &a.grp, &a.q};
  for (int t = 0; t < 12; ++t) { *node_arrays[t] = p; p += N; }
  a.dl = p; p += (int64_t)L * N;
  a.ht = hash;
  if (!hash) { a.ht = p; p += 2 * N; }
  a.hused = p; p += N;
  a.eto = p; p += a.E;
  a.on = p; p += a.O; a.ox = p; p += a.O; a.onext = p; p += a.O;
  a.wblk = p; p += N; a.wpos = p; p += N; a.wneed = p; p += N;
  a.si = p; p += SRC; a.sk = p; p += SRC; a.sp = p; p += SRC; a.shead = p; p += SRC;
  a.ctr = ctr;
  return a;
}

__device__ __forceinline__ uint32_t node_hash(int blk, int S) {
  uint32_t h = (uint32_t)blk * 0x9E3779B1u ^ ((uint32_t)S * 0x85EBCA77u);
  h ^= h >> 15;
  return h;
}

// A hint that brings the line holding p into this SM's L1 (no register is
// written, so nothing waits for it).
__device__ __forceinline__ void prefetch_l1(const void* p) {
  asm volatile("prefetch.global.L1 [%0];" ::"l"(__cvta_generic_to_global(p)));
}

__device__ __forceinline__ int dist_of(const Arena& a, int u) { return (int)(a.dpk[u] >> 32); }
__device__ __forceinline__ int par_of(const Arena& a, int u) { return (int)(a.dpk[u] & 0xFFFFFFFFull); }

// The threads that run one search together: a warp or a whole CTA
// (the very large searches). Both give the search the same
// steps: a barrier, an any-vote, exclusive prefix counts, inclusive sums and
// reductions over the group, a read of a shared flag that every thread takes
// before any of them may change it, and a broadcast from rank 0.
struct WarpGroup {
  static constexpr int kSize = 32;
  __device__ __forceinline__ int rank() const { return threadIdx.x & 31; }
  __device__ __forceinline__ void sync() const { __syncwarp(); }
  __device__ __forceinline__ bool any(bool p) const { return __any_sync(0xffffffffu, p); }
  // exclusive prefix count of `pred`: this thread's slot; *total over the group
  __device__ __forceinline__ int slot(bool pred, int* total) const {
    const unsigned m = __ballot_sync(0xffffffffu, pred);
    *total = __popc(m);
    return __popc(m & ((1u << (threadIdx.x & 31)) - 1u));
  }
  __device__ __forceinline__ int inclusive_sum(int x, int* total) const {
    const int lane = threadIdx.x & 31;
    for (int o = 1; o < 32; o <<= 1) {
      const int y = __shfl_up_sync(0xffffffffu, x, o);
      if (lane >= o) x += y;
    }
    *total = __shfl_sync(0xffffffffu, x, 31);
    return x;
  }
  __device__ __forceinline__ int sum(int x) const {
    for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
    return x;
  }
  __device__ __forceinline__ int max(int x) const {
    for (int o = 16; o > 0; o >>= 1) x = ::max(x, __shfl_xor_sync(0xffffffffu, x, o));
    return x;
  }
  __device__ __forceinline__ int min(int x) const {
    for (int o = 16; o > 0; o >>= 1) x = ::min(x, __shfl_xor_sync(0xffffffffu, x, o));
    return x;
  }
  __device__ __forceinline__ int read(const volatile int* p) const {
    const int v = *p;
    __syncwarp();
    return v;
  }
  __device__ __forceinline__ unsigned long long broadcast(unsigned long long v) const {
    return __shfl_sync(0xffffffffu, v, 0);
  }
};

// A CTA of NT threads as one search group. `red` is shared scratch of NT / 32
// ints, `cast` a shared 64-bit slot for broadcasts. Every collective ends with
// a barrier, so the scratch is free again when it returns.
template <int NT>
struct CtaGroup {
  static constexpr int kSize = NT;
  static constexpr int kWarps = NT / 32;
  int* red;
  unsigned long long* cast;
  __device__ __forceinline__ int rank() const { return threadIdx.x; }
  __device__ __forceinline__ void sync() const { __syncthreads(); }
  __device__ __forceinline__ bool any(bool p) const { return __syncthreads_or(p) != 0; }
  // a value per warp (its last lane's) -> the sum over the warps before this
  // thread's; *total: the sum over all warps
  __device__ __forceinline__ int warp_offsets(int v, int* total) const {
    const int w = threadIdx.x >> 5;
    if ((threadIdx.x & 31) == 31) red[w] = v;
    __syncthreads();
    int before = 0, all = 0;
#pragma unroll
    for (int i = 0; i < kWarps; ++i) {
      const int c = red[i];
      before += i < w ? c : 0;
      all += c;
    }
    __syncthreads();
    *total = all;
    return before;
  }
  __device__ __forceinline__ int slot(bool pred, int* total) const {
    const unsigned m = __ballot_sync(0xffffffffu, pred);
    const int lane = threadIdx.x & 31;
    return warp_offsets(__popc(m), total) + __popc(m & ((1u << lane) - 1u));
  }
  __device__ __forceinline__ int inclusive_sum(int x, int* total) const {
    const int lane = threadIdx.x & 31;
    for (int o = 1; o < 32; o <<= 1) {
      const int y = __shfl_up_sync(0xffffffffu, x, o);
      if (lane >= o) x += y;
    }
    return warp_offsets(x, total) + x;
  }
  template <class Op>
  __device__ __forceinline__ int reduce(int x, Op op) const {
    for (int o = 16; o > 0; o >>= 1) x = op(x, __shfl_xor_sync(0xffffffffu, x, o));
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = x;
    __syncthreads();
    int v = red[0];
#pragma unroll
    for (int i = 1; i < kWarps; ++i) v = op(v, red[i]);
    __syncthreads();
    return v;
  }
  __device__ __forceinline__ int sum(int x) const { return reduce(x, [](int p, int q) { return p + q; }); }
  __device__ __forceinline__ int max(int x) const { return reduce(x, [](int p, int q) { return ::max(p, q); }); }
  __device__ __forceinline__ int min(int x) const { return reduce(x, [](int p, int q) { return ::min(p, q); }); }
  __device__ __forceinline__ int read(const volatile int* p) const {
    const int v = *p;
    __syncthreads();
    return v;
  }
  __device__ __forceinline__ unsigned long long broadcast(unsigned long long v) const {
    if (threadIdx.x == 0) *cast = v;
    __syncthreads();
    v = *cast;
    __syncthreads();
    return v;
  }
};

// Rule 2 on the function's blocks alone, for the sources within their latency
// (sp 2): bit b of reach[B] says block B is reached
// from the root's predecessors without passing the wall of the batch's b-th
// needed group (ord holds the nl groups). A block whose own defs of r cover j's
// guard passes nothing on, whatever literal set comes in. Every path of the graph
// is such a path of blocks, so a source whose block is not reached past some
// wall is cut (sp 3). Returns how many were. A function has tens of thousands of blocks where the
// graph has hundreds of thousands of nodes. Uses dl's second and third layer, q
// and tmp.
template <class G>
__device__ int cut_by_blocks(const G& g, const Prog& P, const Arena& a, int b0, int r, int gj, int nsrc, int nl,
                             int undecided) {
  const int me = g.rank();
  const int f = P.block_func[b0], fb = P.func_block_off[f], nblk = P.func_block_off[f + 1] - fb;
  if (nblk > a.N || a.L < 4) return 0;
  volatile int* ctr = a.ctr;
  int* reach = a.dl + a.N;
  int* mark = a.dl + 2 * (int64_t)a.N;  // the batch's bit + 1 of the block's group; 64: queued; 128: covers
  const int w = r >> 5;
  const uint32_t bit = 1u << (r & 31);
  auto offer = [&](int p, unsigned m, int* nxt) {
    if (!(P.rout[(size_t)p * kWords + w] & bit)) return;
    const unsigned add = m & ~(unsigned)reach[p - fb];
    if (!add) return;
    const unsigned old = (unsigned)atomicOr(&reach[p - fb], (int)add);
    if ((old | add) != old && !(atomicOr(&mark[p - fb], 64) & 64)) nxt[atomicAdd((int*)&ctr[5], 1)] = p - fb;
  };
  for (int t = me; t < nblk; t += G::kSize) {
    const size_t B = fb + t;
    uint16_t S = 0;
    if (P.touch_mask[B * kWords + w] & bit) {
      const size_t seg = B * kEvBuckets + ev_bucket(r);
      for (int e = P.ev_off[seg]; e < P.ev_off[seg + 1]; ++e) {
        const uint32_t ev = P.events[e];
        if ((int)(ev & 0x1FFu) == r && (ev & 0x200u)) S = add_literal(S, (int)((ev >> 12) & 0xFu));
      }
    }
    mark[t] = contains(S, gj) ? 128 : 0;
  }
  int cut = 0;
  for (int w0 = 0; w0 < nl && cut < undecided; w0 += 32) {
    const int nbits = min(32, nl - w0);
    const unsigned full = nbits == 32 ? 0xFFFFFFFFu : ((1u << nbits) - 1u);
    for (int t = me; t < nblk; t += G::kSize) reach[t] = 0;
    if (me == 0) ctr[5] = 0;
    g.sync();
    if (me < nbits) mark[a.wblk[a.ord[w0 + me]] - fb] |= me + 1;
    g.sync();
    int* cur = a.q;
    int* nxt = a.tmp;
    const int4 pm0 = P.block_meta[2 * (size_t)b0 + 1];
    for (int q = pm0.x + me; q < pm0.y; q += G::kSize) offer(P.pred[q], full, cur);
    g.sync();
    int fsize = g.read(&ctr[5]);
    while (fsize > 0) {
      if (me == 0) ctr[5] = 0;
      for (int t = me; t < fsize; t += G::kSize) atomicAnd(&mark[cur[t]], ~64);
      g.sync();
      for (int t = me; t < fsize; t += G::kSize) {
        const int B = cur[t];
        unsigned m = (unsigned)atomicOr(&reach[B], 0);
        const int mk = mark[B], wb = mk & 63;
        if (mk & 128) continue;
        if (wb) m &= ~(1u << (wb - 1));
        if (!m) continue;
        const int4 pm = P.block_meta[2 * (size_t)(fb + B) + 1];
        for (int q = pm.x; q < pm.y; ++q) offer(P.pred[q], m, nxt);
      }
      g.sync();
      fsize = g.read(&ctr[5]);
      int* sw = cur; cur = nxt; nxt = sw;
    }
    int now = 0;
    for (int m = me; m < nsrc; m += G::kSize) {
      if (a.sp[m] != 2) continue;
      const int x = a.si[m], B = P.instr_block[x] - fb;
      unsigned ok = (unsigned)reach[B];
      const int wb = mark[B] & 63;
      if (wb && x < a.wpos[a.ord[w0 + wb - 1]]) ok &= ~(1u << (wb - 1));
      if ((ok & full) != full) { a.sp[m] = 3; ++now; }
    }
    cut += g.sum(now);
    if (me < nbits) mark[a.wblk[a.ord[w0 + me]] - fb] &= 128;
    g.sync();
  }
  return cut;
}

// Returns false when the search outgrew the arena (nothing emitted).
// With P.diag, the search counts the sources of (j, r) before and after
// pruning into use entry e (`blocked`: an unguarded reader above j in its
// block prunes them all by rule 2) and emits nothing. `unsized`: the search takes
// its whole graph, whose size tells later steps its shared-memory class, unless that
// turns out larger than the last of them.
template <class G>
__device__ bool group_search(const G& g, const Prog& P, const Arch& A, const Arena& a, int j, int r, uint16_t S0,
                             int bound, uint16_t live, int tier, int e, bool blocked, bool unsized) {
  const int me = g.rank();
#ifdef GPA_PHASE_TIMING
  long long t_prev = clock64();
  const long long t_begin = t_prev;
  long long t_prev_total = t_prev;
  unsigned long long ph[5] = {0, 0, 0, 0, 0};
  unsigned long long r2runs = 0;
  auto phase = [&](int i) {
    if (me == 0) {
      const long long t = clock64();
      atomicAdd(&P.stats[SS_PHASE + (min(tier, 3) - 1) * 6 + i], (unsigned long long)(t - t_prev));
      ph[i] = (unsigned long long)(t - t_prev);
      t_prev = t;
      if (i == 4 || i == 0) {
        const int nn = max(((volatile int*)a.ctr)[0], 1);
        if (i == 4 || i == 0)
          atomicAdd(&P.stats[SS_SIZE_CYC + min(15, 31 - __clz(nn))], (unsigned long long)(t - t_prev_total));
        t_prev_total = t;
        const unsigned long long key = ((unsigned long long)(t - t_begin) << 20) | (unsigned long long)min(((volatile int*)a.ctr)[0], 0xFFFFF);
        if (atomicMax(&P.stats[SS_SLOW], key) < key) {
          P.stats[SS_SLOW + 1] = r2runs;
          for (int q = 0; q < 5; ++q) P.stats[SS_SLOW + 2 + q] = ph[q];
        }
      }
    }
  };
#else
  auto phase = [](int) {};
#endif
  const int gj = P.guard[j];
  const int b0 = P.instr_block[j];
  const int first0 = P.block_meta[2 * (size_t)b0].x;
  const int w = r >> 5;
  const uint32_t bit = 1u << (r & 31);
  const uint32_t hmask = (uint32_t)(2 * a.N - 1);
  volatile int* ctr = a.ctr;

  // Unexpanded nodes are kept in a list (alternating between seen and tmp,
  // both free until rule 2): ubuf holds ctr[6] of them.
  int* ubuf = a.seen;
  int* ukeep = a.tmp;
  if (me == 0) {
    ctr[0] = 1; ctr[1] = 0; ctr[2] = 0; ctr[3] = 0; ctr[4] = 0; ctr[5] = 0; ctr[6] = 1;
    ubuf[0] = 0;
    S0 = keep_literals(S0, live);
    a.blk[0] = b0; a.S[0] = (int)S0 | ((int)S0 << 16); a.wall[0] = -1; a.fl[0] = 0;
    a.dpk[0] = 0ull; a.k[0] = 0; a.e0[0] = 0; a.e1[0] = 0;
  }
  g.sync();

  // Self-checks of the arena invariants before indexed accesses: an edge
  // range inside [0, edges) here, each target inside [0, nodes) where it is
  // read (target_ok). A violation is recorded as ST_OVERFLOW and the access
  // skipped.
  auto edges_ok = [&](int u, int) {
    const int e0 = a.e0[u], e1 = a.e1[u];
    if (e0 < 0 || e1 < e0 || e1 > a.E || e1 > ctr[1]) { set_status(P, ST_OVERFLOW); return false; }
    return true;
  };
  auto target_ok = [&](int v, int n_now) {
    if ((unsigned)v < (unsigned)n_now) return true;
    set_status(P, ST_OVERFLOW);
    return false;
  };
  auto wout = [&](int u) {
    if (u == 0) return j - first0 + 1;
    const int4 m = P.block_meta[2 * (size_t)a.blk[u]];
    return m.y - m.x;
  };
  auto last_of = [&](int u) { return P.block_meta[2 * (size_t)a.blk[u]].y - 1; };

  // Scan node u's block bottom-up through its events of r's bucket (one
  // thread). Records occurrences, the literal set leaving the top and the first
  // unguarded reader of r met (the wall). Sets a.fl[u] bit 2 if the scan
  // stopped (covered). `first` is the block's first instruction and
  // [ev_beg, ev_end) its segment of r's bucket, empty when no instruction of
  // the block defines r or reads it unguarded (loaded by the caller together
  // with the block's other records).
  auto scan = [&](int u, int first, int ev_beg, int ev_end) {
    uint16_t S = (uint16_t)(a.S[u] & 0xFFFF);
    bool stop = false;
    if (u != 0) {
      const int B = a.blk[u];
      int wall = -1;
      {
        int last_def_pos = -1;
        // Events four at a time: independent read-only loads in flight together
        // (a sentinel resource 511 pads the last group).
        for (int e0 = ev_beg; e0 < ev_end && !stop; e0 += 4) {
          uint32_t evs[4];
#pragma unroll
          for (int q = 0; q < 4; ++q) evs[q] = e0 + q < ev_end ? __ldg(&P.events[e0 + q]) : 0x1FFu;
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            const uint32_t ev = evs[q];
            if (stop || (int)(ev & 0x1FFu) != r) continue;
            const int pos = (int)(ev >> 16), x = first + pos;
            if (ev & 0x200u) {  // def of r
              last_def_pos = pos;
              if (!contains(S, gj) && !(B == b0 && x < j)) {  // sources above j in its block are settled
                const int o = atomicAdd((int*)&a.ctr[2], 1);
                if (o < a.O) { a.on[o] = u; a.ox[o] = x; } else { a.ctr[4] = 3; }
              }
              S = add_literal(S, (int)((ev >> 12) & 0xFu));
              if (contains(S, gj)) stop = true;
            } else if (wall < 0 && pos != last_def_pos && x != j) {  // unguarded reader of r
              wall = x;
            }
          }
        }
      }
      a.wall[u] = wall;
    }
    a.S[u] = (a.S[u] & 0xFFFF) | ((int)keep_literals(S, live) << 16);
    a.fl[u] |= kExpanded | (stop ? 4 : 0);
  };

  // Link the predecessors of the listed nodes, lanes over nodes. Edge ranges
  // come from a warp prefix count; the (block, literal set) nodes are found or
  // added with a warp-synchronous insert: a lane claims an empty slot with
  // atomicCAS, allocates and publishes the node in the same round, and lanes
  // that met a claim in progress retry the slot in the next round.
  // pm: the node's predecessor record (range, first two predecessors);
  // ro0 / ro1: the reach words of those two (loaded before the scan).
  auto link_chunk = [&](const int* lst, int cnt, int4 pm, uint32_t ro0, uint32_t ro1, bool relax) {
    const bool mine = me < cnt;
    const int u = mine ? lst[me] : 0;
    const int B = mine ? a.blk[u] : 0;
    const int Sout = mine ? ((a.S[u] >> 16) & 0xFFFF) : 0;
    const bool open = mine && !(a.fl[u] & 4);
    if (!open) pm = make_int4(0, 0, -1, -1);
    // whether a def of r reaches out of the predecessor at q, and that predecessor
    auto reaches = [&](int q) -> bool {
      const int k = q - pm.x;
      if (k == 0) return ro0 & bit;
      if (k == 1) return ro1 & bit;
      return P.rout[(size_t)__ldg(&P.pred[q]) * kWords + w] & bit;
    };
    auto pred_at = [&](int q) -> int {
      const int k = q - pm.x;
      return k == 0 ? pm.z : k == 1 ? pm.w : __ldg(&P.pred[q]);
    };
    int deg = 0;
    for (int q = pm.x; q < pm.y; ++q) deg += reaches(q) ? 1 : 0;
    int total;
    const int incl = g.inclusive_sum(deg, &total);
    const int ne = ctr[1];
    if (ne + total > a.E) { if (me == 0) ctr[4] = 2; g.sync(); return; }
    if (mine) { a.e0[u] = ne + incl - deg; a.e1[u] = ne + incl; }
    const int maxdeg = g.max(deg);
    // Pass A relaxes each new edge as it is linked, from u's distance now
    // (packed with u as the parent); an expanded target that improves is
    // queued in ord for relax_from, which carries the change on. A node whose
    // own distance improves meanwhile is such a target, so its edges are
    // relaxed again from the better distance.
    unsigned long long nd_u = ~0ull;
    if (relax && mine) {
      const int du = dist_of(a, u);
      if (du < kInf) nd_u = ((unsigned long long)(du + wout(u)) << 32) | (unsigned)u;
    }
    int qp = pm.x;
    for (int kk = 0; kk < maxdeg; ++kk) {
      bool pending = kk < deg;
      int p = -1;
      if (pending) {
        while (!reaches(qp)) ++qp;
        p = pred_at(qp++);
      }
      uint32_t h = pending ? (node_hash(p, Sout) & hmask) : 0;
      int v = -1;
      for (int round = 0; round < 4 * (int)hmask + 64; ++round) {
        if (!g.any(pending)) break;
        if (pending) {
          const int c = a.ht[h];
          if (c >= 0) {
            if (a.blk[c] == p && (a.S[c] & 0xFFFF) == Sout) { v = c; pending = false; }
            else h = (h + 1) & hmask;
          } else if (c == -1) {
            if (atomicCAS(&a.ht[h], -1, -2 - me) == -1) {
              const int nv = atomicAdd((int*)&a.ctr[0], 1);
              if (nv >= a.N) {
                a.ctr[4] = 1; a.ht[h] = -1; pending = false;
              } else {
                a.blk[nv] = p; a.S[nv] = Sout; a.wall[nv] = -1; a.fl[nv] = 0; a.k[nv] = kInf;
                a.e0[nv] = 0; a.e1[nv] = 0;  // no out-edges until the node is expanded
                a.dpk[nv] = ((unsigned long long)kInf << 32) | 0xFFFFFFFFull;
                a.hused[atomicAdd((int*)&a.ctr[3], 1)] = (int)h;
                ubuf[atomicAdd((int*)&a.ctr[6], 1)] = nv;
                __threadfence_block();
                a.ht[h] = nv;
                v = nv; pending = false;
              }
            }
          }  // c <= -2: another lane is publishing this slot; look again next round
        }
        g.sync();
      }
      if (pending) a.ctr[4] = 6;  // the round limit is a bound, not expected to be reached
      if (kk < deg && v >= 0) a.eto[a.e0[u] + kk] = v | (p >= B ? (int)kBackBit : 0);
      if (relax && kk < deg && v >= 0 && nd_u < a.dpk[v] && atomicMin(&a.dpk[v], nd_u) > nd_u &&
          (a.fl[v] & kExpanded) && !(atomicOr(&a.fl[v], 8) & 8))
        a.ord[atomicAdd((int*)&a.ctr[5], 1)] = v;
    }
    g.sync();
    if (me == 0) ctr[1] = ne + total;
    g.sync();
  };

  // Expand every listed node: parallel scans, then parallel linking.
  auto expand_list = [&](const int* list, int cnt, bool relax) {
    for (int c0 = 0; c0 < cnt; c0 += G::kSize) {
      int4 pm = make_int4(0, 0, -1, -1);
      uint32_t ro0 = 0u, ro1 = 0u;
      if (c0 + me < cnt) {
        const int u = list[c0 + me];
        const int B = a.blk[u];
        // First round of loads, all independent: the block's two records, the
        // touch word of r and the bounds of r's event segment.
        pm = __ldg(&P.block_meta[2 * (size_t)B + 1]);
        const int first = __ldg(&P.block_meta[2 * (size_t)B].x);
        const uint32_t tw = __ldg(&P.touch_mask[(size_t)B * kWords + w]);
        const size_t seg = (size_t)B * kEvBuckets + ev_bucket(r);
        const int ev_beg = __ldg(&P.ev_off[seg]);
        int ev_end = __ldg(&P.ev_off[seg + 1]);
        ev_end = (tw & bit) ? ev_end : ev_beg;  // an untouched block has nothing to scan
        // Second round: the reach words of the first two predecessors (read
        // when linking), and the first two predecessors' records, fetched into
        // L1 for the wave that expands them; the scan's event loads follow.
        if (pm.z >= 0) {
          ro0 = P.rout[(size_t)pm.z * kWords + w];
          prefetch_l1(&P.block_meta[2 * (size_t)pm.z]);
          prefetch_l1(&P.touch_mask[(size_t)pm.z * kWords + w]);
          prefetch_l1(&P.ev_off[(size_t)pm.z * kEvBuckets + ev_bucket(r)]);
        }
        if (pm.w >= 0) {
          ro1 = P.rout[(size_t)pm.w * kWords + w];
          prefetch_l1(&P.block_meta[2 * (size_t)pm.w]);
          prefetch_l1(&P.touch_mask[(size_t)pm.w * kWords + w]);
          prefetch_l1(&P.ev_off[(size_t)pm.w * kEvBuckets + ev_bucket(r)]);
        }
        scan(u, first, ev_beg, ev_end);
      }
      g.sync();
      if (ctr[4]) return;
      link_chunk(list + c0, min(G::kSize, cnt - c0), pm, ro0, ro1, relax);
      if (g.read(&ctr[4])) return;  // the next chunk's scans may set it
    }
  };

  // Worklist relaxation from the listed nodes: improved targets join the next
  // frontier once (flag bit 8 of fl). mode 0: shortest distance with parent
  // (64-bit atomicMin on (d << 32) | parent); mode 1: fewest back edges.
  // Frontiers live in ord / grp, which are free until rule 2.
  auto relax_from = [&](const int* start, int cnt, int mode) {
    int* cur = a.ord;
    int* nxt = a.grp;
    for (int t = me; t < cnt; t += G::kSize) cur[t] = start[t];
    if (me == 0) ctr[5] = 0;
    g.sync();
    int fsize = cnt;
    while (fsize > 0) {
      for (int f0 = 0; f0 < fsize; f0 += G::kSize) {
        if (f0 + me >= fsize) continue;
        const int u = cur[f0 + me];
        atomicAnd(&a.fl[u], ~8);
        const int n_now = ctr[0];
        if (!edges_ok(u, n_now)) continue;
        if (mode == 0) {
          const int du = dist_of(a, u);
          if (du >= kInf) continue;
          const unsigned long long nd = (unsigned long long)(du + wout(u)) << 32 | (unsigned)u;
          for (int e = a.e0[u]; e < a.e1[u]; ++e) {
            const int v = a.eto[e] & 0x7FFFFFFF;
            if (!target_ok(v, n_now)) break;
            if (nd < a.dpk[v] && atomicMin(&a.dpk[v], nd) > nd && !(atomicOr(&a.fl[v], 8) & 8))
              nxt[atomicAdd((int*)&a.ctr[5], 1)] = v;
          }
        } else {
          const int ku = a.k[u];
          if (ku >= kInf) continue;
          for (int e = a.e0[u]; e < a.e1[u]; ++e) {
            const int v = a.eto[e] & 0x7FFFFFFF;
            if (!target_ok(v, n_now)) break;
            const int kb = ku + (int)((uint32_t)a.eto[e] >> 31);
            if (kb < a.k[v] && atomicMin(&a.k[v], kb) > kb && !(atomicOr(&a.fl[v], 8) & 8))
              nxt[atomicAdd((int*)&a.ctr[5], 1)] = v;
          }
        }
      }
      g.sync();
      fsize = ctr[5];
      g.sync();
      if (me == 0) ctr[5] = 0;
      int* sw = cur; cur = nxt; nxt = sw;
      g.sync();
    }
  };

  // Pass B only needs the nodes that can lie on a path from a candidate
  // source up to j: the node's block must be reachable in the CFG from the
  // candidate's block, so it is not below that block's smallest reachable
  // block. cand_low is the least of these over the candidates.
  int cand_low = 0;
  auto relevant = [&](int u) { return a.blk[u] >= cand_low; };

  // How the graph grows. kNear (pass A): the nodes within the bound. kLayers:
  // those that paths of at most k_max back edges to a live candidate can pass,
  // where k_max is the most that the candidates' occurrences in pass A need:
  // nodes of fewer back edges, and of k_max where the block is not above every
  // candidate's (from there on only forward edges are left, and block indices
  // fall along them). kAll (pass B): every node on a path to a candidate.
  enum { kNear, kLayers, kAll };
  constexpr bool kParts = G::kSize > 32;
  int k_max = 0, blk_low = 0;
  auto in_layers = [&](int u) { return a.k[u] < k_max || (a.k[u] == k_max && a.blk[u] >= blk_low); };

  // Split unexpanded nodes: those to expand now (into list) and the rest, which
  // stay unexpanded (beyond pass A, nodes off every candidate's paths are
  // dropped for good). kLayers sets the rest aside in `defer` (the layers of
  // the longest paths are free until then), so its waves do not read them again.
  int* list = a.q;
  int* const defer = a.dl;
  int n_defer = 0;
  auto split = [&](const int* from, int m, int* rest, int grow, int* kept_out) {
    int cnt = 0, kept = 0;
    for (int i0 = 0; i0 < m; i0 += G::kSize) {
      const int i = i0 + me;
      const int u = i < m ? from[i] : 0;
      const bool now = i < m && (grow == kNear ? dist_of(a, u) <= bound : relevant(u) && (!kParts || grow == kAll || in_layers(u)));
      const bool keep = i < m && !now && (grow == kNear || (kParts && grow == kLayers && relevant(u)));
      int tot_now, tot_keep;
      const int at_now = g.slot(now, &tot_now);
      const int at_keep = g.slot(keep, &tot_keep);
      if (now) list[cnt + at_now] = u;
      if (keep) rest[kept + at_keep] = u;
      cnt += tot_now;
      kept += tot_keep;
    }
    g.sync();
    *kept_out = kept;
    return cnt;
  };
  auto take_wave = [&](int grow) {
    int kept;
    int cnt = split(ubuf, g.read(&ctr[6]), kParts && grow == kLayers ? defer + n_defer : ukeep, grow, &kept);
    int* sw = ubuf; ubuf = ukeep; ukeep = sw;
    if (kParts && grow == kLayers) {
      n_defer += kept;
      kept = 0;
      // nodes whose fewest back edges fell meanwhile (compacted in place: a
      // chunk is read before any of it is written, and writes stay below it)
      if (cnt == 0) cnt = split(defer, n_defer, defer, grow, &n_defer);
    }
    if (me == 0) ctr[6] = kept;
    g.sync();
    return cnt;
  };

  // Pass A expands in waves the nodes within the bound, relaxing as they
  // link. Only if some source is within its latency does the graph grow on.
  // A CTA's searches then first drop the sources that rule 2 cuts on the
  // function's blocks already (cut_by_blocks), and grow the layers of what is
  // left: the longest paths need no more, and a source that reaches past every
  // wall there survives. Only where some does not is the graph completed
  // (`whole`). Counted on kernels of 45,000 to 200,000 instructions: six in ten
  // sources go on the blocks, a search is left with one wall to test on the graph
  // instead of dozens, and one or no search in 2,000 needs the whole graph.
  // Blame with 5M samples of 120,000 instructions: 480 -> 330 ms; 60,000: 54 ->
  // 46 ms; 200,000 (20M samples): 340 -> 250 ms. The warps' searches, whose size
  // tells later steps their shared-memory class, take the whole graph at once.
  // All growth runs in this one loop, so the wave code exists once in the kernel.
  bool cand = false, grew_b = false, whole = !kParts || P.diag || unsized, again = false;
  bool sizing = kParts && unsized && !P.diag;
  int grow = kNear;
  int nsrc, nl, alive, n_cut = 0;
  int* const cut_list = a.dl + 3 * (int64_t)a.N;  // sources cut on the blocks
  auto candidate = [&](int o) {
    const int u = a.on[o];
    return dist_of(a, u) + (last_of(u) - a.ox[o]) <= A.lat[P.opclass[a.ox[o]]];
  };
  // Puts the nodes back into the hash and the list in `defer` back into ubuf.
  auto resume = [&](int n) {
    for (int u = 1 + me; u < n; u += G::kSize) {
      uint32_t h = node_hash(a.blk[u], a.S[u] & 0xFFFF) & hmask;
      for (uint32_t t = 0; t <= hmask && atomicCAS(&a.ht[h], -1, u) != -1; ++t) h = (h + 1) & hmask;
      a.hused[u - 1] = (int)h;
    }
    for (int t = me; t < n_defer; t += G::kSize) a.seen[t] = defer[t];
    ubuf = a.seen;
    ukeep = a.tmp;
    if (me == 0) { ctr[3] = n - 1; ctr[5] = 0; ctr[6] = n_defer; }
    g.sync();
    n_defer = 0;
    again = true;
  };
  while (true) {  // once; a CTA's search: pass A, the layers, and the whole graph if need be
  while (!ctr[4]) {
    const int cnt = take_wave(grow);
    if (cnt > 0) {
      grew_b |= grow != kNear;
      expand_list(list, cnt, grow == kNear);
      if (ctr[4]) break;
      // pass A relaxed the wave's edges as they were linked; carry on from the
      // expanded nodes that improved (queued in ord, counted in ctr[5])
      // (every thread reads the count before relax_from's rank 0 clears it)
      if (grow == kNear) {
        const int n_dirty = g.read(&ctr[5]);
        if (n_dirty > 0) relax_from(a.ord, n_dirty, 0);
      } else if (kParts && grow == kLayers) {
        relax_from(list, cnt, 1);
      } else if (kParts && sizing && g.read(&ctr[0]) > class_nodes(kClasses - 1, a.N)) {
        // Of no class: on with the parts, from a graph that is pass A's and some more
        // (which adds only paths of the whole graph; k is not set yet, like after pass A).
        sizing = whole = false;
        grow = kNear;
        break;
      }
      continue;
    }
    if (grow != kNear) break;
    // End of pass A. A source within its latency? (Every candidate is found
    // by pass A: a source farther than the bound fails rule 3.)
    const int no = min(ctr[2], a.O);
    int low = 0x7FFFFFFF;
    for (int o = me; o < no; o += G::kSize) {
      if (candidate(o)) {
        cand = true;
        low = min(low, P.block_minreach[a.blk[a.on[o]]]);
      }
    }
    cand = g.any(cand);
    cand_low = g.min(low);
    if (!cand) break;
    if (kParts && !whole) break;
    grow = kAll;
  }
  // Clear the hash slots this search used.
  const int nh = ctr[3];
  for (int t = me; t < nh; t += G::kSize) a.ht[a.hused[t]] = -1;
  g.sync();
  const int n = ctr[0];
  if (me == 0) {
    if (!again) atomicAdd(&P.stats[SS_GENERAL], 1ull);
    atomicMax(&P.stats[SS_MAX_NODES], (unsigned long long)n);
    atomicMax(&P.stats[SS_MAX_TASK], ((unsigned long long)n << 40) | ((unsigned long long)r << 31) | (unsigned)j);
#ifdef GPA_PHASE_TIMING
    atomicAdd(&P.stats[SS_SIZES + min(15, 31 - __clz(max(n, 1)))], 1ull);
    if (cand) atomicAdd(&P.stats[SS_PASSB], 1ull);
#endif
  }
  phase(0);
  if (ctr[4]) {
    if (me == 0) ctr[7] = ctr[4];
    g.sync();
    return false;
  }
  if (!cand && !P.diag) return true;

  // Shortest distance with parents, and fewest back edges, over the whole
  // graph. When pass B expanded no node, every edge of the graph was relaxed
  // to the fixpoint in pass A, whose (distance, parent) minimum over the same
  // edges is this one. On the layers both are there already: the back edges
  // were relaxed as they grew, and the distances of pass A's nodes are final
  // (any path within the bound stays in them; a node beyond it keeps a distance
  // beyond it, so its occurrences fail rule 3 as they should).
  const bool fresh_d = (!kParts || whole) && grew_b;
  if (!kParts || whole) {
    for (int u = me; u < n; u += G::kSize) {
      if (fresh_d) a.dpk[u] = u == 0 ? 0ull : (((unsigned long long)kInf << 32) | 0xFFFFFFFFull);
      a.k[u] = u == 0 ? 0 : kInf;
      a.fl[u] &= ~8;
    }
    if (me == 0) a.q[0] = 0;
    g.sync();
#pragma unroll 1
    for (int mode = fresh_d ? 0 : 1; mode < 2; ++mode) relax_from(a.q, 1, mode);
  }
  phase(1);

  // Sources: a warp-synchronous hash keyed by instruction gives each source an
  // index; per source, 64-bit atomicMin keeps (shortest distance, its
  // occurrence), atomicMin the fewest back edges, and the occurrences are
  // chained into a list.
  const int no = ctr[2];
  if (me == 0) { ctr[3] = 0; ctr[5] = 0; }
  g.sync();
  const uint32_t smask = (uint32_t)(2 * a.SRC - 1);
  for (int o0 = 0; o0 < no; o0 += G::kSize) {
    const int o = o0 + me;
    bool pending = o < no;
    const int x = pending ? a.ox[o] : -1;
    uint32_t h = pending ? (((uint32_t)x * 0x9E3779B1u) >> 7) & smask : 0;
    int m = -1;
    for (int round = 0; round < 4 * (int)smask + 64; ++round) {
      if (!g.any(pending)) break;
      if (pending) {
        const int c = a.ht[h];
        if (c >= 0) {
          if (a.si[c] == x) { m = c; pending = false; } else h = (h + 1) & smask;
        } else if (c == -1) {
          if (atomicCAS(&a.ht[h], -1, -2 - me) == -1) {
            const int nm = atomicAdd((int*)&a.ctr[5], 1);
            if (nm >= a.SRC) {
              a.ctr[4] = 4; a.ht[h] = -1; pending = false;
            } else {
              a.si[nm] = x; a.sk[nm] = kInf; a.shead[nm] = -1; a.sp[nm] = 0;
              a.sdb[nm] = ~0ull;
              a.hused[atomicAdd((int*)&a.ctr[3], 1)] = (int)h;
              __threadfence_block();
              a.ht[h] = nm;
              m = nm; pending = false;
            }
          }
        }
      }
      g.sync();
    }
    if (pending) a.ctr[4] = 6;
    if (m >= 0) {
      const int u = a.on[o];
      const int dist = dist_of(a, u) + (last_of(u) - x);
      atomicMin(&a.sdb[m], ((unsigned long long)dist << 32) | (unsigned)o);
      atomicMin(&a.sk[m], a.k[u]);
      a.onext[o] = atomicExch(&a.shead[m], o);
    }
    g.sync();
  }
  {
    const int nh2 = ctr[3];
    for (int t = me; t < nh2; t += G::kSize) a.ht[a.hused[t]] = -1;
  }
  g.sync();
  if (ctr[4]) {
    if (me == 0) ctr[7] = ctr[4];
    g.sync();
    return false;
  }
  nsrc = g.read(&ctr[5]);
  alive = 0;
  for (int m = me; m < nsrc; m += G::kSize) {
    a.sp[m] = (int)(a.sdb[m] >> 32) > A.lat[P.opclass[a.si[m]]] ? 1 : 0;  // rule 3
    if (P.diag == 1 && (blocked || !keeps_any(P, A, j, P.opclass[a.si[m]]))) a.sp[m] = 1;  // rule 2 above j, rule 1
    if (P.diag == 2) a.sp[m] = 0;  // export: rule 2 for every source
    if (kParts && !a.sp[m])
      for (int t = 0; t < n_cut; ++t)
        if (cut_list[t] == a.si[m]) { a.sp[m] = 1; break; }
    alive += a.sp[m] ? 0 : 1;
  }
  alive = g.sum(alive);
  phase(2);
  if (alive == 0) {
    if (P.diag == 1 && me == 0) cov_add(P, e, nsrc, 0);
    return true;
  }

  // Rule 2. Wall groups, one per block: a hash keyed by block with atomicMax
  // of the positions (the unguarded reader met first from the bottom truncates
  // at least as much as any other reader of that block). A wall can only block
  // source i if it lies on the parent chain of i's nearest occurrence.
  if (me == 0) { ctr[3] = 0; ctr[5] = 0; }
  g.sync();
  for (int u0 = 0; u0 < n; u0 += G::kSize) {
    const int u = u0 + me;
    bool pending = u < n && u != 0 && a.wall[u] >= 0;
    const int B = pending ? a.blk[u] : -1;
    uint32_t h = pending ? (((uint32_t)B * 0x9E3779B1u) >> 5) & hmask : 0;
    int wg = -1;
    for (int round = 0; round < 4 * (int)hmask + 64; ++round) {
      if (!g.any(pending)) break;
      if (pending) {
        const int c = a.ht[h];
        if (c >= 0) {
          if (a.wblk[c] == B) { wg = c; pending = false; } else h = (h + 1) & hmask;
        } else if (c == -1) {
          if (atomicCAS(&a.ht[h], -1, -2 - me) == -1) {
            const int ng = atomicAdd((int*)&a.ctr[5], 1);
            a.wblk[ng] = B; a.wpos[ng] = -1; a.wneed[ng] = 0;
            a.hused[atomicAdd((int*)&a.ctr[3], 1)] = (int)h;
            __threadfence_block();
            a.ht[h] = ng;
            wg = ng; pending = false;
          }
        }
      }
      g.sync();
    }
    if (pending) a.ctr[4] = 6;
    if (u < n) a.grp[u] = wg;
    if (wg >= 0) atomicMax(&a.wpos[wg], a.wall[u]);
    g.sync();
  }
  {
    const int nh2 = ctr[3];
    for (int t = me; t < nh2; t += G::kSize) a.ht[a.hused[t]] = -1;
  }
  g.sync();
  if (ctr[4]) {
    if (me == 0) ctr[7] = ctr[4];
    g.sync();
    return false;
  }
  const int nw = ctr[5];
  for (int m = me; m < nsrc; m += G::kSize) {
    if (a.sp[m]) continue;
    const int o = (int)(a.sdb[m] & 0xFFFFFFFFull), u = a.on[o];
    if (u != 0 && a.wall[u] > a.ox[o]) a.wneed[a.grp[u]] = 1;
    for (int v = par_of(a, u), hops = 0; v > 0 && hops < n; v = par_of(a, v), ++hops)
      if (a.wall[v] >= 0) a.wneed[a.grp[v]] = 1;
  }
  g.sync();
  // The needed groups, compacted into ord (free until the longest paths).
  nl = 0;
  for (int t0 = 0; t0 < nw; t0 += G::kSize) {
    const bool need = t0 + me < nw && a.wneed[t0 + me];
    int tot;
    const int at = g.slot(need, &tot);
    if (need) a.ord[nl + at] = t0 + me;
    nl += tot;
  }
  for (int t = me; t < nw; t += G::kSize) a.wneed[t] = 0;
  g.sync();
  if (kParts && grow == kNear && !whole) {
    // Pass A is done: rule 2 on the blocks, then the layers of the survivors.
    n_defer = g.read(&ctr[6]);
    for (int t = me; t < n_defer; t += G::kSize) defer[t] = ubuf[t];
    for (int m = me; m < nsrc; m += G::kSize) if (!a.sp[m]) a.sp[m] = 2;
    g.sync();
    alive -= cut_by_blocks(g, P, a, b0, r, gj, nsrc, nl, alive);
    phase(3);
    if (alive == 0) return true;
    if (me == 0) { ctr[5] = 0; a.q[0] = 0; }
    g.sync();
    for (int m = me; m < nsrc; m += G::kSize)
      if (a.sp[m] == 3) cut_list[atomicAdd((int*)&a.ctr[5], 1)] = a.si[m];
    g.sync();
    n_cut = g.read(&ctr[5]);
    relax_from(a.q, 1, 1);
    int most = 0, low_blk = 0x7FFFFFFF, low_reach = 0x7FFFFFFF;
    for (int m = me; m < nsrc; m += G::kSize) {
      if (a.sp[m] != 2) continue;
      const int B = P.instr_block[a.si[m]];
      low_blk = min(low_blk, B);
      low_reach = min(low_reach, P.block_minreach[B]);
      for (int o = a.shead[m]; o >= 0; o = a.onext[o])
        if (candidate(o)) most = max(most, a.k[a.on[o]]);
    }
    k_max = g.max(most);
    blk_low = g.min(low_blk);
    cand_low = g.min(low_reach);
    whole = k_max >= a.L;
    grow = whole ? kAll : kLayers;
    resume(n);
    continue;
  }
  // Bit-parallel reachability over up to 32 groups at a time: bit b of
  // reach[u] (kept in seen) says u is reachable from the root without passing
  // the wall of the batch's b-th group. A node truncated by a group (each node
  // of its block that has a wall) passes every bit on but that group's.
  // wneed[g] holds g's bit + 1 while g is in the batch.
  int* reach = a.seen;
  const int undecided = alive;
  for (int w0 = 0; w0 < nl && alive > 0; w0 += 32) {
    const int nbits = min(32, nl - w0);
    const unsigned full = nbits == 32 ? 0xFFFFFFFFu : ((1u << nbits) - 1u);
#ifdef GPA_PHASE_TIMING
    if (me == 0) atomicAdd(&P.stats[SS_PHASE + (min(tier, 3) - 1) * 6 + 5], 1ull);
    ++r2runs;
#endif
    if (me < nbits) a.wneed[a.ord[w0 + me]] = me + 1;
    for (int u = me; u < n; u += G::kSize) reach[u] = u == 0 ? (int)full : 0;
    g.sync();
    auto pass_mask = [&](int u) {
      const int wg = u != 0 ? a.grp[u] : -1;
      const int b = wg >= 0 ? a.wneed[wg] : 0;
      return b ? ~(1u << (b - 1)) : 0xFFFFFFFFu;
    };
    int* cur = a.q;
    int* nxt = a.tmp;
    if (me == 0) { cur[0] = 0; ctr[5] = 0; }
    int fsize = 1;
    g.sync();
    while (fsize > 0) {
      // Clear the queued flags of the whole frontier first: bits that arrive
      // at a frontier node during this round queue it again.
      for (int f = me; f < fsize; f += G::kSize) atomicAnd(&a.fl[cur[f]], ~8);
      g.sync();
      for (int f0 = 0; f0 < fsize; f0 += G::kSize) {
        if (f0 + me >= fsize) continue;
        const int u = cur[f0 + me];
        if (!edges_ok(u, n)) continue;
        const unsigned m = (unsigned)atomicOr(&reach[u], 0) & pass_mask(u);
        if (!m) continue;
        for (int e = a.e0[u]; e < a.e1[u]; ++e) {
          const int v = a.eto[e] & 0x7FFFFFFF;
          if (!target_ok(v, n)) break;
          const unsigned add = m & ~(unsigned)reach[v];
          if (!add) continue;
          const unsigned old = (unsigned)atomicOr(&reach[v], (int)add);
          if ((old | add) != old && !(atomicOr(&a.fl[v], 8) & 8)) nxt[atomicAdd((int*)&a.ctr[5], 1)] = v;
        }
      }
      g.sync();
      fsize = ctr[5];
      g.sync();
      if (me == 0) ctr[5] = 0;
      int* sw = cur; cur = nxt; nxt = sw;
      g.sync();
    }
    // A source survives the batch if, for every group, one of its occurrences
    // is reached without passing that group's wall (an occurrence above the
    // wall inside a truncated node is cut too).
    int dropped = 0;
    for (int m = me; m < nsrc; m += G::kSize) {
      if (a.sp[m]) continue;
      unsigned ok = 0;
      for (int o = a.shead[m]; o >= 0 && (ok & full) != full; o = a.onext[o]) {
        const int u = a.on[o];
        unsigned r = (unsigned)reach[u];
        const int wg = u != 0 ? a.grp[u] : -1;
        if (wg >= 0 && a.wneed[wg] && a.ox[o] < a.wpos[wg]) r &= ~(1u << (a.wneed[wg] - 1));
        ok |= r;
      }
      if ((ok & full) != full) { a.sp[m] = !kParts || whole ? 1 : 2; ++dropped; }
    }
    alive -= g.sum(dropped);
    g.sync();
    if (me < nbits) a.wneed[a.ord[w0 + me]] = 0;
    g.sync();
  }
  phase(3);
  // A path found on the layers is a path of the whole graph, so a source that
  // survived there survives. Where one did not, the whole graph decides.
  if (kParts && !whole && undecided > alive) {
    if (n_defer > 0) {
      whole = true;
      grow = kAll;
      resume(n);
      continue;
    }
    for (int m = me; m < nsrc; m += G::kSize) if (a.sp[m] == 2) a.sp[m] = 1;  // the layers are the whole graph
    g.sync();
  }
  break;
  }
  const int n = g.read(&ctr[0]);
  if (P.diag == 1) {
    if (me == 0) cov_add(P, e, nsrc, alive);
    return true;
  }
  // The export keeps every source: sp marks the rule-2 cuts (its dom flag).
  const bool every = P.diag == 2;
  if (alive == 0 && !every) return true;

  // Longest path with exactly K back edges: layer = back edges used. Each
  // layer is a DAG over the forward edges, processed in topological order by
  // level-synchronous Kahn frontiers; back edges feed the next layer.
  int maxK = 0;
  for (int m = me; m < nsrc; m += G::kSize) if (!a.sp[m] || every) maxK = max(maxK, a.sk[m]);
  maxK = g.max(maxK);
  if (maxK >= a.L) {
    if (me == 0) ctr[7] = 5;
    g.sync();
    return false;
  }
  for (int t = me; t < (maxK + 1) * n; t += G::kSize) a.dl[(t / n) * a.N + (t % n)] = -1;
  for (int u = me; u < n; u += G::kSize) a.ord[u] = 0;
  g.sync();
  for (int u = me; u < n; u += G::kSize)
    for (int e = a.e0[u]; e < a.e1[u]; ++e)
      if (!((uint32_t)a.eto[e] >> 31)) atomicAdd(&a.ord[a.eto[e] & 0x7FFFFFFF], 1);
  if (me == 0) a.dl[0] = 0;
  g.sync();
  for (int l = 0; l <= maxK; ++l) {
    int* dll = a.dl + (int64_t)l * a.N;
    if (me == 0) ctr[5] = 0;
    g.sync();
    for (int u = me; u < n; u += G::kSize) {
      a.seen[u] = a.ord[u];  // remaining forward in-edges
      if (a.ord[u] == 0) a.q[atomicAdd((int*)&a.ctr[5], 1)] = u;
    }
    g.sync();
    int fsize = ctr[5];
    int* cur = a.q;
    int* nxt = a.tmp;
    g.sync();
    if (me == 0) ctr[5] = 0;
    g.sync();
    while (fsize > 0) {
      for (int f0 = 0; f0 < fsize; f0 += G::kSize) {
        if (f0 + me < fsize) {
          const int u = cur[f0 + me];
          const int cv = dll[u];
          const int nd = cv + wout(u);
          for (int e = a.e0[u]; e < a.e1[u]; ++e) {
            const int v = a.eto[e] & 0x7FFFFFFF;
            const bool back = (uint32_t)a.eto[e] >> 31;
            if (back) {
              if (cv >= 0 && l + 1 <= maxK) atomicMax(&a.dl[(int64_t)(l + 1) * a.N + v], nd);
            } else {
              if (cv >= 0) atomicMax(&dll[v], nd);
              if (atomicSub(&a.seen[v], 1) == 1) nxt[atomicAdd((int*)&a.ctr[5], 1)] = v;
            }
          }
        }
      }
      g.sync();
      fsize = ctr[5];
      g.sync();
      if (me == 0) ctr[5] = 0;
      int* sw = cur; cur = nxt; nxt = sw;
      g.sync();
    }
  }
  for (int m = me; m < nsrc; m += G::kSize) {
    if (a.sp[m] && !every) continue;
    const int K = a.sk[m];
    int best = -1;
    for (int o = a.shead[m]; o >= 0; o = a.onext[o]) {
      const int u = a.on[o];
      const int dlu = a.dl[(int64_t)K * a.N + u];
      if (dlu >= 0) best = max(best, dlu + last_of(u) - a.ox[o]);
    }
    if (best < 1) { capacity(P, 13); continue; }
    if (every) xemit(P, j, a.si[m], r, (int)(a.sdb[m] >> 32), K, best, a.sp[m] || blocked);
    else emit_raw(P, A, j, a.si[m], r, def_kind(P, a.si[m], r), (int)(a.sdb[m] >> 32), best);
  }
  g.sync();
  phase(4);
  return true;
}

// A queue region of searches and where those that outgrow the arenas go.
struct Route {
  int q, n_slot, h_slot;   // queue, its count and head
  bool top;                // read down from the top of the queue
  int next_q, next_slot;   // -1: the last tier (it records why it ran out)
  bool next_top;
  uint32_t next_hint;
};

// The task loop of a search group: claim (use, resource) tasks from one
// queue until it is empty. An arena that holds its own hash (`clear`) has it
// emptied when the group's first task arrives, so a group that finds none touches
// no memory.
template <class G>
__device__ void run_tasks(const G& g, const Prog& P, const Arch& A, const Arena& a, const Route& R, int tier,
                          bool clear) {
  const int me = g.rank();
  const unsigned long long cap = (unsigned long long)P.queue_cap;
  const int32_t* q = P.queue[R.q];
  const unsigned long long nt = min(P.stats[R.n_slot], cap);
  while (true) {
    unsigned long long t = 0;
    if (me == 0) t = atomicAdd(&P.stats[R.h_slot], 1ull);
    t = g.broadcast(t);
    if (t >= nt) break;
    if (clear) {
      for (int k = me; k < 2 * a.N; k += G::kSize) a.ht[k] = -1;
      g.sync();
      clear = false;
    }
    const int e = q[R.top ? cap - 1 - t : t];
    const int2 task = P.tasks[e];
    const int r = task.y & 0x1FF;
    const int f = P.block_func[P.instr_block[task.x]];
    // The coverage count needs every source: no latency bound.
    const int bound = P.diag ? kInf - 1 : P.res_maxlat[(size_t)f * kNumRes + r];
    const uint16_t live = live_literals(P.res_guards[(size_t)f * kNumRes + r], P.guard[task.x]);
    // What a CTA gets from a full list may be of any class yet. (Every thread reads
    // the hint before rank 0 raises it: the search's barriers lie between.)
    const bool unsized = G::kSize > 32 && P.tier_hint[P.diag ? 1 : 0][e] < kHintWide;
    const bool ok = group_search(g, P, A, a, task.x, r, (uint16_t)((uint32_t)task.y >> 9), bound, live, tier, e,
                                 (task.y >> 25) & 1, unsized);
    if (me != 0) continue;
    if (ok) {
      // Later steps queue the search for the class of its graph.
      if (tier == 3 || unsized) {
        int c = 0;
        while (c < kClasses && class_nodes(c, a.N) < ((volatile int*)a.ctr)[0]) ++c;
        raise_hint(P, e, (uint32_t)(kHintA1 + c));
      }
      continue;
    }
    if (R.next_q < 0) {
      capacity(P, a.ctr[7] > 0 ? a.ctr[7] : 1);
      continue;
    }
    raise_hint(P, e, R.next_hint);
    const unsigned long long o = atomicAdd(&P.stats[R.next_slot], 1ull);
    if (o < cap) P.queue[R.next_q][R.next_top ? cap - 1 - o : o] = e;
    else capacity(P, 8);
  }
}

// Persistent work-stealing warps, one search each: what the shared-memory
// warps' largest classes are known to have beyond three rounds of the chip. (Of
// unknown size, searches of up to 32,768 nodes would come here: those go to the CTAs.)
// 80 registers a thread, so 24 one-warp CTAs fit an SM: the searches are chains of
// dependent loads, and more warps in flight finish more of them (measured: 40.7
// against 41.9 ms a step with 96).
__global__ void __launch_bounds__(32, 24) k_search_warp(Prog P, Arch A, SearchArena SA, Route R) {
  // The search counters live in shared memory (the arena is in global memory):
  // frontier sizes are read after every round.
  __shared__ int s_ctr[8];
  // The node hashes lie apart from the arenas (whose pool the largest searches lay
  // out anew) and are empty between searches: every search empties the slots it
  // used, also when it outgrew its arena. They were cleared with the context,
  // so a launch clears nothing. (A launch that began by clearing its warps'
  // 256 KB hashes wrote 956 MB and took 145 us with no search to run.)
  const Arena a = carve(SA.global + (int64_t)blockIdx.x * SA.bytes, SA.hash + (int64_t)blockIdx.x * 2 * SA.nodes,
                        SA.nodes, SA.src, SA.layers, s_ctr);
  run_tasks(WarpGroup{}, P, A, a, R, 3, false);
}

// A CTA per search: the waves, frontiers and source lists of these searches
// are wide enough for its threads. 128 threads for searches of 5,633 to 32,768
// nodes (a warp took 31 ms for the largest of them) and for what the shared-memory
// warps' full lists hand on, whose size is not known yet (first step of 20,000, 30,000
// and 45,000 instructions: 26, 35 and 70 ms of blame with those by the warps, 16, 17
// and 41 by CTAs; 200,000 with 20M samples 194 and 184, with 300M, where most of them
// outgrow these arenas too, 266 and 271); 512 for larger ones, two of
// these CTAs on an SM (64 registers), 1,024 for those beyond 2^18 nodes, whose
// arenas are too large for a CTA on every SM. Both are chains of barriers and
// arena latency, so what counts is threads in flight: on the 120,000-instruction
// kernel 330 ms of blame with one CTA of 512 an SM for both, 298 with two,
// 247 with 1,024 threads for the largest. (256 threads, three CTAs: 233 there, but
// 31.6 against 28.1 ms at 45,000 instructions, where the searches do not fill
// the chip; 128 threads, six CTAs: slower everywhere.)
template <int NT>
__global__ void __launch_bounds__(NT, NT == 128 ? 4 : 1024 / NT) k_search_cta(Prog P, Arch A, SearchArena SA, Route R) {
  __shared__ int s_ctr[8];
  __shared__ int s_red[CtaGroup<NT>::kWarps];
  __shared__ unsigned long long s_cast;
  const CtaGroup<NT> g{s_red, &s_cast};
  int* hash = SA.hash ? SA.hash + (int64_t)blockIdx.x * 2 * SA.nodes : nullptr;
  const Arena a = carve(SA.global + (int64_t)blockIdx.x * SA.bytes, hash, SA.nodes, SA.src, SA.layers, s_ctr);
  run_tasks(g, P, A, a, R, 4, hash == nullptr);
}

}  // namespace

int64_t search_arena_bytes(int nodes, int src, int layers, bool own_hash) {
  return arena_bytes(nodes, src, layers, own_hash);
}

int search_warps_per_sm() {
  int n = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, k_search_warp, 32, 0) != cudaSuccess || n < 1) n = 4;
  return n;
}

void launch_search(const Prog& P, const Arch& A, const SearchArena* tiers, const SearchFork* fork, cudaStream_t st,
                   int sms, int64_t* launches) {
  // The searches queued straight for the larger tiers depend on nothing the
  // first two tiers do: with further streams they run beside them (no kernel
  // waits on another; the joins only order the parts that share arenas or
  // storage after them). They are submitted first, so that the largest searches
  // start first and the first tiers' CTAs fill the SMs as they come free.
  cudaStream_t s[4] = {st, st, st, st};
  if (fork) {
    cudaEventRecord(fork->fork, st);
    for (int k = 0; k < 3; ++k) {
      s[k] = fork->side[k];
      cudaStreamWaitEvent(s[k], fork->fork, 0);
    }
  }
  // The CTAs of 128 threads take the first of the arenas, the warps the others
  // (with a single arena they take turns).
  SearchArena wide = tiers[2], narrow = tiers[2];
  wide.warps = std::max(1, std::min(tiers[2].warps / 2, 4 * sms));
  if (tiers[2].warps > 1) {
    narrow.warps -= wide.warps;
    narrow.global += (int64_t)wide.warps * narrow.bytes;
    narrow.hash += (int64_t)wide.warps * 2 * narrow.nodes;
  } else {
    s[2] = s[1];
  }
  const bool big = P.t4_nodes > 0;
  const int q4 = big ? 4 : -1;
  const Route wide1{6, SS_WIDE_N, SS_WIDE_HEAD, false, q4, SS_T4_N, false, kHintCta};
  const Route wide2{6, SS_WIDE2_N, SS_WIDE2_HEAD, true, q4, SS_T4_N, false, kHintCta};
  const Route warp1{3, SS_HINT3_N, SS_HINT3_HEAD, true, q4, SS_T4_N, false, kHintCta};
  // No launch takes more groups than there can be tasks (one per use entry).
  auto groups = [&](int n) { return (int)std::max<int64_t>(1, std::min<int64_t>(n, P.queue_cap)); };
  launch_search_smem(P, A, tiers[2].nodes, 1, s[0], sms, launches);
  k_search_cta<128><<<groups(wide.warps), 128, 0, s[1]>>>(P, A, wide, wide1);
  k_search_warp<<<groups(narrow.warps), 32, 0, s[2]>>>(P, A, narrow, warp1);
  launch_search_lanes(P, A, tiers[0], 1, st, launches);
  launch_search_lanes(P, A, tiers[1], 2, st, launches);
  if (fork)
    for (int k = 0; k < 3; ++k) {
      cudaEventRecord(fork->join[k], fork->side[k]);
      cudaStreamWaitEvent(st, fork->join[k], 0);
    }
  launch_search_smem(P, A, tiers[2].nodes, 2, st, sms, launches);
  k_search_cta<128><<<groups(wide.warps), 128, 0, st>>>(P, A, wide, wide2);
  *launches += 3;
  if (big) {
    // Larger searches run after the others on this stream, so the third tier's
    // arena pool is free by then and they carve their arenas from it (at most two
    // CTAs per SM): first those of up to 2^18 nodes (most of them; arenas for the
    // program's largest function would be so big that the pool holds few), then
    // the rest in arenas of t4_nodes, from the pool when it holds more of them
    // than the program's own.
    const int64_t pool = tiers[2].global ? (int64_t)tiers[2].warps * tiers[2].bytes : 0;
    SearchArena own{P.t4_nodes, P.t4_src, kMaxLayers, P.t4_arena ? P.t4_ctas : 0, P.t4_bytes, P.t4_arena, nullptr};
    if (pool / P.t4_bytes > own.warps) {
      own.warps = (int)std::min<int64_t>(pool / P.t4_bytes, std::max(sms, 1));
      own.global = tiers[2].global;
    }
    const int mid_nodes = 1 << 18;
    SearchArena mid{mid_nodes, 4096, kMaxLayers, 0, arena_bytes(mid_nodes, 4096, kMaxLayers, true), tiers[2].global,
                    nullptr};
    mid.warps = (int)std::min<int64_t>(pool / mid.bytes, 2 * std::max(sms, 1));
    Route r4{4, SS_T4_N, SS_T4_HEAD, false, -1, 0, false, 0};
    if (P.t4_nodes > mid_nodes && mid.warps > own.warps) {
      r4.next_q = 7; r4.next_slot = SS_T5_N; r4.next_hint = kHintGiant;
      k_search_cta<512><<<groups(mid.warps), 512, 0, st>>>(P, A, mid, r4);
      ++*launches;
      const Route r5{7, SS_T5_N, SS_T5_HEAD, false, -1, 0, false, 0};
      k_search_cta<1024><<<groups(own.warps), 1024, 0, st>>>(P, A, own, r5);
    } else {
      k_search_cta<512><<<groups(own.warps), 512, 0, st>>>(P, A, own, r4);
    }
    ++*launches;
  }
}

}  // namespace gpa
