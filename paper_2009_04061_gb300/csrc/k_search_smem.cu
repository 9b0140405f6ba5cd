// Step (b)/(c), general backward searches (Sec. 4), the middle tier: one search
// per warp over an arena in shared memory, up to 5,632 (block, literal set)
// nodes.
//
// These searches grow four or five nodes a wave over hundreds of waves, and
// each of their later steps (fewest back edges, rule 2's reachability, longest
// paths) walks the graph's depth level by level, so a search is a chain of
// thousands of dependent accesses to its own arena and the largest one decides
// how long a step takes. What bounds it is the latency of that arena: in global
// memory (k_search_warp, 700 cycles an access) a search of 227 nodes took 650 us
// and one of 5,269 took 6.4 ms. So the arena is laid out small enough for shared
// memory: 36.5 bytes a node (16-bit node, edge and list indices; distance and
// parent in one word; words that later steps reuse) plus the hash, and holds the
// block lengths that the global-memory search reads from the program again and
// again.
//
// One CTA of 16 warps per SM gives its 227 KB to one size class after another:
// 1 search of 5,632 nodes, 2 of 2,560, 4 of 1,280, 8 of 640, 16 of 320. Searches
// that an earlier step of the program found to be of a class are queued for it
// and run largest class first; a search that outgrows its class goes on a list of
// its CTA, which works off its lists in ascending order at the end. Beyond the
// last class, and where a list is full, CTAs of 128 threads over global memory take
// over. One-warp searches there take what the three largest classes are known to have
// beyond three rounds of the chip: a search takes three times as long, but 3,648 run
// at once (see smem_class_limit).
// Registers: 80 a thread, so that global-memory searches (which use no shared
// memory) find room beside this CTA.
//
// The graph, the passes and the rules are those of k_search.cu's group search;
// like the one-lane search (k_search_lanes.cu) it ends early when its only
// unexpanded node meets an unguarded reader of r before any def was met.
#include <algorithm>
#include <climits>

#include "gpa_internal.cuh"

namespace gpa {

namespace {

constexpr int kWarps = 16;
constexpr int kLocalList = 256;      // searches a CTA keeps for its own next class
constexpr int kDistBits = 19, kIdxBits = 13;
constexpr uint32_t kFar = (1u << kDistBits) - 1u;  // no distance yet
constexpr uint32_t kIdxMask = (1u << kIdxBits) - 1u;
constexpr uint32_t kNoWall = 0xFFFFu;
constexpr uint32_t F_EXP = 1u << 24, F_QUE = 1u << 25, F_NEED = 1u << 26, F_BACK = 1u << 27;
constexpr int kSearchInf = 0x7FFFFFFF;

__host__ __device__ inline int class_warps(int c) { return 16 >> c; }
// Searches of class c that a CTA keeps for itself: rounds of the largest
// classes, bounded so that a list does not outlast the CTAs that take the rest.
__device__ inline int local_list(int c) {
  return c < 2 ? kLocalList : (c == 2 ? 8 : c == 3 ? 4 : 3) * class_warps(c);
}
__host__ __device__ inline int hash_slots(int n) {  // a power of two, at least 1.4 n
  int h = 16;
  while (5 * h < 7 * n) h <<= 1;
  return h;
}
__host__ __device__ inline int n_occ(int n) { return n / 4 < 8 ? 8 : (n / 4 + 1) & ~1; }
__host__ __device__ inline int n_src(int n) { return n / 8 < 8 ? 8 : n / 8; }
__host__ __device__ inline int n_edge(int n) { return (3 * n / 2 + 3) & ~1; }
__host__ __device__ inline int64_t warp_arena_bytes(int n) {
  const int64_t nn = (n + 1) & ~1;
  const int64_t b = 4 * (6 * nn + n_occ(n) + 4 * (int64_t)n_src(n)) +
                    2 * (3 * nn + n_edge(n) + hash_slots(n) + n_occ(n));
  return (b + 15) & ~(int64_t)15;
}

struct WArena {
  int n, occs, srcs, edges;
  uint32_t hmask;
  uint32_t *key;   // block (relative to the function) | literal set << 16
  uint32_t *dp;    // distance << 13 | parent; then the reach mask; then a layer's longest distance
  uint32_t *wl;    // wall position (kNoWall: none) | instructions of the block << 16
  uint32_t *ef;    // first edge | edges << 16 | flags << 24
  uint32_t *kk;    // fewest back edges; then forward in-edges | in-edges left << 16
  uint32_t *gx;    // two 16-bit lists; then the wall group + 1; then the next layer's longest distance
  uint32_t *oc;    // per occurrence: position | node << 16 | def kind << 29
  uint32_t *si, *sd, *sk, *sh;  // per source: block | position << 16; distance << 13 | nearest occurrence;
                                // fewest back edges | cut << 31; first occurrence
  uint16_t *l0, *l1, *l2;  // node lists
  uint16_t *ed;    // edges: target | back << 15
  uint16_t *ht;    // node (or source) hash: 0xFFFF empty, marks while a slot is being filled
  uint16_t *on;    // per occurrence: the next of its source
  volatile int *ctr;  // 2 occurrences, 4 too small, 5 sources
  uint16_t *wpos;  // 32 wall positions (while the graph grows: which edge a lane takes)
};

__device__ WArena carve(char* base, int n, int* ctr, uint16_t* wpos) {
  WArena a;
  const int nn = (n + 1) & ~1;
  a.n = n; a.occs = n_occ(n); a.srcs = n_src(n); a.edges = n_edge(n);
  const int hs = hash_slots(n);
  a.hmask = (uint32_t)hs - 1u;
  uint32_t* p = reinterpret_cast<uint32_t*>(base);
  a.key = p; p += nn; a.dp = p; p += nn; a.wl = p; p += nn;
  a.ef = p; p += nn; a.kk = p; p += nn; a.gx = p; p += nn;
  a.oc = p; p += a.occs;
  a.si = p; p += a.srcs; a.sd = p; p += a.srcs; a.sk = p; p += a.srcs; a.sh = p; p += a.srcs;
  uint16_t* q = reinterpret_cast<uint16_t*>(p);
  a.l0 = q; q += nn; a.l1 = q; q += nn; a.l2 = q; q += nn;
  a.ed = q; q += a.edges;
  a.ht = q; q += hs;
  a.on = q;
  a.ctr = ctr;
  a.wpos = wpos;
  return a;
}

__device__ __forceinline__ uint32_t mix(uint32_t k) {
  uint32_t h = (k & 0xFFFFu) * 0x9E3779B1u ^ ((k >> 16) * 0x85EBCA77u);
  return h ^ (h >> 15);
}
// One search by one warp. Returns 0 when it is done, else why its arena is too
// small (nothing was emitted); *nodes: the nodes met.
// A warp that has an SM's scheduler to itself is bound by the instructions of a
// wave, one after another, so list appends are ballots over uniform loops (the
// counts stay in registers), a wave's edges are spread over the lanes whatever
// node they belong to, and lanes that look for the same node let one of them
// probe.
__device__ int warp_search(const Prog& P, const Arch& A, const WArena& a, int j, int r, uint16_t S0, int e_use,
                           bool blocked, int* nodes) {
  constexpr unsigned kAll = 0xFFFFFFFFu;
  const int lane = threadIdx.x & 31;
  const unsigned lt = (1u << lane) - 1u;
  volatile int* ctr = a.ctr;
  const int gj = P.guard[j];
  const int b0 = P.instr_block[j];
  const int f = P.block_func[b0];
  const int fb = P.func_block_off[f];
  *nodes = 0;
  if (P.func_block_off[f + 1] - fb > 0xFFFF) return 1;  // its blocks need more than the arena's 16 bits
  const size_t fr = (size_t)f * kNumRes + r;
  const int bound = P.diag ? kSearchInf : P.res_maxlat[fr];
  const uint16_t live = live_literals(P.res_guards[fr], gj);
  const int w = r >> 5;
  const uint32_t bit = 1u << (r & 31);
  S0 = keep_literals(S0, live);
  auto clear_hash = [&]() {
    uint32_t* h = reinterpret_cast<uint32_t*>(a.ht);
    for (uint32_t i = lane; i <= a.hmask / 2; i += 32) h[i] = 0xFFFFFFFFu;
  };
  auto dist_of = [&](int u) { return *(volatile uint32_t*)&a.dp[u] >> kIdxBits; };
  auto len_of = [&](int u) { return a.wl[u] >> 16; };
  auto wall_of = [&](int u) { return a.wl[u] & 0xFFFFu; };
  auto occ_node = [&](int o) { return (int)((a.oc[o] >> 16) & kIdxMask); };
  auto occ_pos = [&](int o) { return (int)(a.oc[o] & 0xFFFFu); };
  // An improved distance of an expanded node, which is not queued yet.
  auto improves = [&](bool has, int v, uint32_t nd) -> bool {
    return has && nd < *(volatile uint32_t*)&a.dp[v] && atomicMin(&a.dp[v], nd) > nd &&
           (*(volatile uint32_t*)&a.ef[v] & F_EXP) && !(atomicOr(&a.ef[v], F_QUE) & F_QUE);
  };

#ifdef GPA_PHASE_TIMING
  long long t_prev = clock64();
  auto phase = [&](int i) {  // (the second tier's row of the search profile)
    if (lane == 0) {
      const long long t = clock64();
      atomicAdd(&P.stats[SS_PHASE + 6 + i], (unsigned long long)(t - t_prev));
      t_prev = t;
    }
  };
#else
  auto phase = [](int) {};
#endif
  clear_hash();
  if (lane == 0) {
    ctr[2] = 0; ctr[4] = 0;
    a.key[0] = (uint32_t)(b0 - fb) | ((uint32_t)S0 << 16);
    a.dp[0] = 0u; a.wl[0] = kNoWall; a.ef[0] = 0u;
    a.l0[0] = 0;
  }
  __syncwarp();
  int nn = 1, ne = 0, nu = 1;   // nodes, edges, unexpanded nodes (all lanes hold the same)
  bool has_back = false;
  uint16_t* ub = a.l0;          // the unexpanded nodes
  uint16_t* uk = a.l1;
  uint16_t* cur = reinterpret_cast<uint16_t*>(a.gx);  // nodes to relax from
  uint16_t* nxt = cur + a.n;

  bool cand = false, pass_b = false;
  int low = 0;
  while (true) {
    // A wave: the unexpanded nodes within the bound (pass B: those that can lie
    // on a path from a source within its latency; the others are dropped).
    const bool only = nu == 1 && ctr[2] == 0 && !pass_b && !P.diag;
    int cnt = 0, kept = 0;
    for (int i0 = 0; i0 < nu; i0 += 32) {
      const int i = i0 + lane;
      const int u = i < nu ? ub[i] : 0;
      const bool now = i < nu && (pass_b ? fb + (int)(a.key[u] & 0xFFFFu) >= low : (int)dist_of(u) <= bound);
      const bool keep = i < nu && !now && !pass_b;
      const unsigned mn = __ballot_sync(kAll, now), mk = __ballot_sync(kAll, keep);
      if (now) a.l2[cnt + __popc(mn & lt)] = (uint16_t)u;
      if (keep) uk[kept + __popc(mk & lt)] = (uint16_t)u;
      cnt += __popc(mn);
      kept += __popc(mk);
    }
    __syncwarp();
    uint16_t* sw = ub; ub = uk; uk = sw;
    nu = kept;
    if (cnt == 0) {
      if (pass_b) break;
      // End of pass A: a source within its latency? (A source farther than the
      // bound fails rule 3.)
      const int no = ctr[2];
      int lo = kSearchInf;
      for (int o = lane; o < no; o += 32) {
        const int u = occ_node(o);
        const int d = (int)dist_of(u) + (int)len_of(u) - 1 - occ_pos(o);
        if (d > bound) continue;
        const int B = fb + (int)(a.key[u] & 0xFFFFu);
        if (d <= A.lat[P.opclass[P.block_meta[2 * (size_t)B].x + occ_pos(o)]]) lo = min(lo, P.block_minreach[B]);
      }
      low = __reduce_min_sync(kAll, lo);
      cand = low != kSearchInf;
      if (!cand) break;
      pass_b = true;
      continue;
    }
    int nq = 0;  // nodes to relax from, in cur
    for (int c0 = 0; c0 < cnt; c0 += 32) {
      // Expand up to 32 nodes: parallel scans ...
      const bool mine = c0 + lane < cnt;
      const int u = mine ? a.l2[c0 + lane] : 0;
      const uint32_t key = a.key[u];
      const int B = fb + (int)(key & 0xFFFFu);
      uint16_t S = (uint16_t)(key >> 16);
      int deg = 0, pA = 0, pB = 0;  // the first two predecessors that a def of r leaves
      int q0 = 0;                   // (the predecessor list, for more than two)
      bool cut = false;
      uint32_t nd = 0;
      if (mine) {
        const int4 m0 = __ldg(&P.block_meta[2 * (size_t)B]);
        const int4 pm = __ldg(&P.block_meta[2 * (size_t)B + 1]);
        const uint32_t tw = __ldg(&P.touch_mask[(size_t)B * kWords + w]);
        const size_t seg = (size_t)B * kEvBuckets + ev_bucket(r);
        const int ev_beg = __ldg(&P.ev_off[seg]);
        int ev_end = __ldg(&P.ev_off[seg + 1]);
        if (!(tw & bit) || u == 0) ev_end = ev_beg;
        const uint32_t ro0 = pm.z >= 0 ? P.rout[(size_t)pm.z * kWords + w] & bit : 0u;
        const uint32_t ro1 = pm.w >= 0 ? P.rout[(size_t)pm.w * kWords + w] & bit : 0u;
        uint32_t wall = kNoWall;
        int last_def = -1;
        bool any_def = false, stop = false;
        for (int e0 = ev_beg; e0 < ev_end && !stop; e0 += 4) {
          uint32_t evs[4];
#pragma unroll
          for (int q = 0; q < 4; ++q) evs[q] = e0 + q < ev_end ? __ldg(&P.events[e0 + q]) : 0x1FFu;
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            const uint32_t ev = evs[q];
            if (stop || (int)(ev & 0x1FFu) != r) continue;
            const int pos = (int)(ev >> 16), x = m0.x + pos;
            if (ev & 0x200u) {  // def of r
              last_def = pos;
              if (!contains(S, gj) && !(B == b0 && x < j)) {  // sources above j in its block are settled
                any_def = true;
                const int o = atomicAdd((int*)&ctr[2], 1);
                if (o < a.occs) a.oc[o] = (uint32_t)pos | ((uint32_t)u << 16) | (((ev >> 10) & 3u) << 29);
              }
              S = add_literal(S, (int)((ev >> 12) & 0xFu));
              if (contains(S, gj)) stop = true;
            } else if (wall == kNoWall && pos != last_def && x != j) {  // unguarded reader of r
              wall = (uint32_t)pos;
              cut |= only && !any_def;
            }
          }
        }
        const uint32_t len = (uint32_t)(u == 0 ? j - m0.x + 1 : m0.y - m0.x);
        a.wl[u] = wall | (len << 16);
        nd = dist_of(u) + len;
        if (!stop) {
          deg = (ro0 ? 1 : 0) + (ro1 ? 1 : 0);
          pA = ro0 ? pm.z : pm.w;
          pB = pm.w;
          q0 = pm.x;
          for (int q = pm.x + 2; q < pm.y; ++q) {
            const int p = __ldg(&P.pred[q]);
            if (!(P.rout[(size_t)p * kWords + w] & bit)) continue;
            if (deg == 0) pA = p;
            if (deg == 1) pB = p;
            ++deg;
          }
        }
      }
      __syncwarp();
      // With `only`, the single node dominates everything beyond it: when it meets
      // an unguarded reader before any def, every source lies beyond that reader.
      if (__any_sync(kAll, cut)) { *nodes = nn; return 0; }
      if (ctr[2] > a.occs) { *nodes = nn; return 3; }
      if (__any_sync(kAll, mine && nd >= kFar)) { *nodes = nn; return 1; }
      nd = (nd << kIdxBits) | (uint32_t)u;
      // ... then linking. The edge ranges from a prefix sum of the degrees (two
      // ballots, as long as none exceeds three).
      int excl, total;
      if (__any_sync(kAll, deg > 3)) {
        int incl = deg;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
          const int y = __shfl_up_sync(kAll, incl, o);
          if (lane >= o) incl += y;
        }
        total = __shfl_sync(kAll, incl, 31);
        excl = incl - deg;
        if (__any_sync(kAll, deg > 255)) { *nodes = nn; return 2; }
      } else {
        const unsigned m1 = __ballot_sync(kAll, deg & 1), m2 = __ballot_sync(kAll, deg & 2);
        excl = __popc(m1 & lt) + 2 * __popc(m2 & lt);
        total = __popc(m1) + 2 * __popc(m2);
      }
      if (ne + total > a.edges) { *nodes = nn; return 2; }
      if (mine) a.ef[u] = (uint32_t)(ne + excl) | ((uint32_t)deg << 16) | F_EXP;
      const int Sout = (int)keep_literals(S, live);
      __syncwarp();
      for (int e0 = 0; e0 < total; e0 += 32) {
        // lane i takes edge e0 + i: its node's lane and which predecessor it is
        for (int k = 0; k < deg; ++k) {
          const int i = excl + k - e0;
          if (i >= 0 && i < 32) a.wpos[i] = (uint16_t)(lane | (k << 5));
        }
        __syncwarp();
        const bool pend = e0 + lane < total;
        const int mp = pend ? a.wpos[lane] : 0;
        const int src = mp & 31, k = mp >> 5;
        const int p0 = __shfl_sync(kAll, pA, src), p1 = __shfl_sync(kAll, pB, src);
        const int Bu = __shfl_sync(kAll, B, src), So = __shfl_sync(kAll, Sout, src), qu = __shfl_sync(kAll, q0, src);
        const uint32_t ndu = __shfl_sync(kAll, nd, src);
        int p = k == 0 ? p0 : p1;
        if (pend && k >= 2) {  // the k-th predecessor that a def of r leaves
          int left = k;
          for (int q = qu;; ++q) {
            p = __ldg(&P.pred[q]);
            if ((P.rout[(size_t)p * kWords + w] & bit) && left-- == 0) break;
          }
        }
        const uint32_t pk = (uint32_t)(p - fb) | ((uint32_t)So << 16);
        // One lane per node looked for probes the hash. A lane that finds an
        // empty slot leaves its mark there; the one whose mark stays adds the node.
        const unsigned pm_ = __ballot_sync(kAll, pend);
        const unsigned peers = __match_any_sync(kAll, pk) & pm_;
        const int lead = __ffs(peers) - 1;
        bool act = pend && lane == lead;
        uint32_t h = mix(pk) & a.hmask;
        int v = -1;
        while (__any_sync(kAll, act)) {  // ends: the hash has more slots than there can be nodes
          const uint32_t c = act ? *(volatile uint16_t*)&a.ht[h] : 0u;
          const bool empty = act && c == 0xFFFFu;
          if (act && !empty) {
            if (a.key[c] == pk) { v = (int)c; act = false; }
            else h = (h + 1) & a.hmask;
          }
          __syncwarp();  // every slot is read before any is marked
          if (empty) *(volatile uint16_t*)&a.ht[h] = (uint16_t)(0x8000 | lane);
          __syncwarp();
          const bool won = empty && *(volatile uint16_t*)&a.ht[h] == (0x8000 | lane);
          const unsigned wm = __ballot_sync(kAll, won);
          if (wm) {
            if (nn + __popc(wm) > a.n) { *nodes = a.n; return 1; }
            if (won) {
              v = nn + __popc(wm & lt);
              a.key[v] = pk; a.wl[v] = kNoWall; a.ef[v] = 0u; a.dp[v] = 0xFFFFFFFFu;
              ub[nu + __popc(wm & lt)] = (uint16_t)v;
              *(volatile uint16_t*)&a.ht[h] = (uint16_t)v;
              act = false;
            }
            nn += __popc(wm);
            nu += __popc(wm);
          }
          __syncwarp();
        }
        v = __shfl_sync(kAll, v, lead < 0 ? 0 : lead);
        const bool back = pend && p >= Bu;
        has_back |= __any_sync(kAll, back);
        if (pend) a.ed[ne + e0 + lane] = (uint16_t)(v | (back ? 0x8000 : 0));
        // The new edges relax their targets; an expanded one that improves is
        // queued to carry the change on.
        const bool q = improves(pend, v, ndu);
        const unsigned qm = __ballot_sync(kAll, q);
        if (q) cur[nq + __popc(qm & lt)] = (uint16_t)v;
        nq += __popc(qm);
        __syncwarp();
      }
      ne += total;
    }
    // Carry improved distances on over the expanded nodes' edges.
    while (nq > 0) {
      int nq2 = 0;
      bool far = false;
      for (int i0 = 0; i0 < nq; i0 += 32) {
        const bool in = i0 + lane < nq;
        const int u = in ? cur[i0 + lane] : 0;
        const uint32_t ef = in ? atomicAnd(&a.ef[u], ~F_QUE) : 0u;
        const uint32_t d = dist_of(u) + len_of(u);
        far |= in && d >= kFar;
        const uint32_t ndu = (d << kIdxBits) | (uint32_t)u;
        const int deg = (int)((ef >> 16) & 0xFFu), e0 = (int)(ef & 0xFFFFu);
        const int md = __reduce_max_sync(kAll, deg);
        for (int k = 0; k < md; ++k) {
          const int v = k < deg ? a.ed[e0 + k] & 0x7FFF : 0;
          const bool q = improves(k < deg && !far, v, ndu);
          const unsigned qm = __ballot_sync(kAll, q);
          if (q) nxt[nq2 + __popc(qm & lt)] = (uint16_t)v;
          nq2 += __popc(qm);
        }
      }
      __syncwarp();
      if (__any_sync(kAll, far)) { *nodes = nn; return 1; }
      uint16_t* s2 = cur; cur = nxt; nxt = s2;
      nq = nq2;
    }
  }
  *nodes = nn;
  phase(0);
  if (!cand && !P.diag) return 0;
  const int n = nn, no = ctr[2];

  // Fewest back edges from j: layer by layer, forward edges within a layer,
  // back edges into the next (every node is listed once).
  if (has_back) {
    for (int u = lane; u < n; u += 32) a.kk[u] = u == 0 ? 0u : 0xFFFFu;
    if (lane == 0) a.l0[0] = 0;
    __syncwarp();
    int fs = 1, nb = 0;
    cur = a.l0;
    nxt = a.l1;
    for (uint32_t k = 0; fs > 0; ++k) {
      while (fs > 0) {
        int f2 = 0;
        for (int i0 = 0; i0 < fs; i0 += 32) {
          const bool in = i0 + lane < fs;
          const uint32_t ef = in ? *(volatile uint32_t*)&a.ef[cur[i0 + lane]] : 0u;
          const int deg = (int)((ef >> 16) & 0xFFu), e0 = (int)(ef & 0xFFFFu);
          const int md = __reduce_max_sync(kAll, deg);
          for (int q = 0; q < md; ++q) {
            const int ed = q < deg ? a.ed[e0 + q] : 0, v = ed & 0x7FFF;
            const bool un = q < deg && *(volatile uint32_t*)&a.kk[v] > k;
            const bool bk = un && (ed & 0x8000) && !(atomicOr(&a.ef[v], F_BACK) & F_BACK);
            const bool fw = un && !(ed & 0x8000) && atomicMin(&a.kk[v], k) > k;
            const unsigned bm = __ballot_sync(kAll, bk), fm = __ballot_sync(kAll, fw);
            if (bk) a.l2[nb + __popc(bm & lt)] = (uint16_t)v;
            if (fw) nxt[f2 + __popc(fm & lt)] = (uint16_t)v;
            nb += __popc(bm);
            f2 += __popc(fm);
          }
        }
        __syncwarp();
        uint16_t* sw = cur; cur = nxt; nxt = sw;
        fs = f2;
      }
      // the back edges' targets that no fewer back edges reached
      for (int i0 = 0; i0 < nb; i0 += 32) {
        const bool in = i0 + lane < nb;
        const int v = in ? a.l2[i0 + lane] : 0;
        if (in) atomicAnd(&a.ef[v], ~F_BACK);
        const bool fw = in && atomicMin(&a.kk[v], k + 1) > k + 1;
        const unsigned fm = __ballot_sync(kAll, fw);
        if (fw) cur[fs + __popc(fm & lt)] = (uint16_t)v;
        fs += __popc(fm);
      }
      nb = 0;
      __syncwarp();
    }
  }
  phase(1);

  // Sources: a hash keyed by (block, position) gives each an index; per source
  // the shortest distance with its occurrence, the fewest back edges, and its
  // occurrences chained.
  clear_hash();
  if (lane == 0) ctr[5] = 0;
  __syncwarp();
  for (int o0 = 0; o0 < no; o0 += 32) {
    const int o = o0 + lane;
    bool pending = o < no;
    const int u = pending ? occ_node(o) : 0;
    const uint32_t id = pending ? (a.key[u] & 0xFFFFu) | ((uint32_t)occ_pos(o) << 16) : 0u;
    uint32_t h = mix(id) & a.hmask;
    int m = -1;
    for (int round = 0; round < 4 * (int)a.hmask + 64; ++round) {
      if (!__any_sync(0xffffffffu, pending)) break;
      if (pending) {
        const uint32_t c = *(volatile uint16_t*)&a.ht[h];
        if (c < 0xFFFEu) {
          if (*(volatile uint32_t*)&a.si[c] == id) { m = (int)c; pending = false; }
          else h = (h + 1) & a.hmask;
        } else if (c == 0xFFFFu) {
          if (atomicCAS((unsigned short*)&a.ht[h], (unsigned short)0xFFFF, (unsigned short)0xFFFE) == 0xFFFF) {
            const int nm = atomicAdd((int*)&ctr[5], 1);
            pending = false;
            if (nm >= a.srcs) {
              ctr[4] = 4;
              *(volatile uint16_t*)&a.ht[h] = 0xFFFF;
            } else {
              a.si[nm] = id; a.sd[nm] = 0xFFFFFFFFu; a.sk[nm] = 0xFFFFu; a.sh[nm] = 0xFFFFu;
              __threadfence_block();
              *(volatile uint16_t*)&a.ht[h] = (uint16_t)nm;
              m = nm;
            }
          }
        }
      }
      __syncwarp();
    }
    if (pending) ctr[4] = 6;
    if (m >= 0) {
      const uint32_t d = dist_of(u) + len_of(u) - 1u - (uint32_t)occ_pos(o);
      atomicMin(&a.sd[m], (d << kIdxBits) | (uint32_t)o);
      atomicMin(&a.sk[m], has_back ? a.kk[u] : 0u);
      a.on[o] = (uint16_t)atomicExch(&a.sh[m], (uint32_t)o);
    }
    __syncwarp();
  }
  const int why = ctr[4];
  __syncwarp();
  if (why) return why;
  const int nsrc = ctr[5];
  auto src_instr = [&](int m) {
    return P.block_meta[2 * (size_t)(fb + (int)(a.si[m] & 0xFFFFu))].x + (int)(a.si[m] >> 16);
  };
  int alive = 0;
  for (int m = lane; m < nsrc; m += 32) {
    const int op = P.opclass[src_instr(m)];
    bool drop = (int)(a.sd[m] >> kIdxBits) > A.lat[op];                    // rule 3
    if (P.diag == 1 && (blocked || !keeps_any(P, A, j, op))) drop = true;  // rule 2 above j, rule 1
    if (P.diag == 2) drop = false;                                         // export: rule 2 for every source
    if (drop) a.sk[m] |= 1u << 31;
    alive += drop ? 0 : 1;
  }
  alive = __reduce_add_sync(0xffffffffu, alive);
  if (alive == 0) {
    if (P.diag == 1 && lane == 0) cov_add(P, e_use, nsrc, 0);
    return 0;
  }

  phase(2);
  // Rule 2. The walls that can cut a source lie on the parent chain of its
  // nearest occurrence: mark their nodes.
  __syncwarp();
  for (int m = lane; m < nsrc; m += 32) {
    if (a.sk[m] >> 31) continue;
    const int o = (int)(a.sd[m] & kIdxMask), u = occ_node(o);
    if (wall_of(u) != kNoWall && (int)wall_of(u) > occ_pos(o)) atomicOr(&a.ef[u], F_NEED);
    for (int v = (int)(a.dp[u] & kIdxMask), hops = 0; v > 0 && hops < n; v = (int)(a.dp[v] & kIdxMask), ++hops)
      if (wall_of(v) != kNoWall) atomicOr(&a.ef[v], F_NEED);
  }
  __syncwarp();
  for (int u = lane; u < n; u += 32) a.gx[u] = 0u;
  __syncwarp();
  // Up to 32 wall groups at a time, one per block (the reader met first from
  // the bottom over the block's nodes): bit g of a node's mask says it is reached
  // without passing group g's wall; a node of the group passes every bit on but
  // its own.
  int scan0 = 0;
  while (alive > 0) {
    int ng = 0;
    while (scan0 < n && ng < 32) {
      const int u = scan0 + lane;
      const unsigned need = __ballot_sync(0xffffffffu, u < n && (*(volatile uint32_t*)&a.ef[u] & F_NEED));
      if (!need) { scan0 += 32; continue; }
      const uint32_t B = a.key[scan0 + __ffs(need) - 1] & 0xFFFFu;
      int wp = 0;
      for (int v = lane; v < n; v += 32) {
        if (v == 0 || (a.key[v] & 0xFFFFu) != B || wall_of(v) == kNoWall) continue;
        a.gx[v] = (uint32_t)(ng + 1);
        atomicAnd(&a.ef[v], ~F_NEED);
        wp = max(wp, (int)wall_of(v));
      }
      wp = __reduce_max_sync(0xffffffffu, wp);
      if (lane == 0) a.wpos[ng] = (uint16_t)wp;
      ++ng;
      __syncwarp();
    }
    if (ng == 0) break;
    const uint32_t full = ng == 32 ? 0xFFFFFFFFu : (1u << ng) - 1u;
    for (int u = lane; u < n; u += 32) a.dp[u] = u == 0 ? full : 0u;
    if (lane == 0) a.l0[0] = 0;
    __syncwarp();
    cur = a.l0;
    nxt = a.l1;
    int fs = 1;
    while (fs > 0) {
      // The whole frontier's queued flags first: bits that reach a frontier node
      // during this round queue it again.
      for (int i = lane; i < fs; i += 32) atomicAnd(&a.ef[cur[i]], ~F_QUE);
      __syncwarp();
      int f2 = 0;
      for (int i0 = 0; i0 < fs; i0 += 32) {
        const bool in = i0 + lane < fs;
        const int u = in ? cur[i0 + lane] : 0;
        const uint32_t g = a.gx[u];
        const uint32_t mk = in ? *(volatile uint32_t*)&a.dp[u] & (g ? ~(1u << (g - 1)) : 0xFFFFFFFFu) : 0u;
        const uint32_t ef = mk ? *(volatile uint32_t*)&a.ef[u] : 0u;
        const int deg = (int)((ef >> 16) & 0xFFu), e0 = (int)(ef & 0xFFFFu);
        const int md = __reduce_max_sync(kAll, deg);
        for (int k = 0; k < md; ++k) {
          const int v = k < deg ? a.ed[e0 + k] & 0x7FFF : 0;
          bool q = k < deg && (mk & ~*(volatile uint32_t*)&a.dp[v]);
          if (q) {
            const uint32_t old = atomicOr(&a.dp[v], mk);
            q = (old | mk) != old && !(atomicOr(&a.ef[v], F_QUE) & F_QUE);
          }
          const unsigned qm = __ballot_sync(kAll, q);
          if (q) nxt[f2 + __popc(qm & lt)] = (uint16_t)v;
          f2 += __popc(qm);
        }
      }
      __syncwarp();
      uint16_t* sw = cur; cur = nxt; nxt = sw;
      fs = f2;
    }
    // A source survives if, for every group, one of its occurrences is reached
    // without passing that group's wall.
    int dropped = 0;
    for (int m = lane; m < nsrc; m += 32) {
      if (a.sk[m] >> 31) continue;
      uint32_t ok = 0u;
      for (uint32_t o = a.sh[m]; o != 0xFFFFu && ok != full; o = a.on[o]) {
        const int u = occ_node((int)o);
        const uint32_t g = a.gx[u];
        uint32_t rr = a.dp[u];
        if (g && occ_pos((int)o) < (int)a.wpos[g - 1]) rr &= ~(1u << (g - 1));
        ok |= rr;
      }
      if (ok != full) { a.sk[m] |= 1u << 31; ++dropped; }
    }
    alive -= __reduce_add_sync(0xffffffffu, dropped);
    if (scan0 >= n) break;
    __syncwarp();
    for (int u = lane; u < n; u += 32) a.gx[u] = 0u;
    __syncwarp();
  }
  if (P.diag == 1) {
    if (lane == 0) cov_add(P, e_use, nsrc, alive);
    return 0;
  }
  const bool every = P.diag == 2;  // the export keeps every source (the cut is its dom flag)
  if (alive == 0 && !every) return 0;

  phase(3);
  // Longest path with exactly K back edges: one layer per back edge, each a DAG
  // of forward edges processed in Kahn's order; back edges feed the next layer.
  __syncwarp();
  int maxk = 0;
  for (int m = lane; m < nsrc; m += 32)
    if (!(a.sk[m] >> 31) || every) maxk = max(maxk, (int)(a.sk[m] & 0xFFFFu));
  maxk = __reduce_max_sync(0xffffffffu, maxk);
  if (maxk >= kMaxLayers) return 5;
  for (int u = lane; u < n; u += 32) {
    a.kk[u] = 0u;
    a.dp[u] = u == 0 ? 0u : 0xFFFFFFFFu;
    a.gx[u] = 0xFFFFFFFFu;
  }
  __syncwarp();
  for (int e = lane; e < ne; e += 32) {
    const int ed = a.ed[e];
    if (!(ed & 0x8000)) atomicAdd(&a.kk[ed], 1u);
  }
  __syncwarp();
  for (int l = 0; l <= maxk; ++l) {
    int fs = 0;
    for (int u0 = 0; u0 < n; u0 += 32) {
      const int u = u0 + lane;
      const uint32_t in = u < n ? a.kk[u] & 0xFFFFu : 1u;
      const unsigned z = __ballot_sync(0xffffffffu, in == 0u);
      if (u < n) a.kk[u] = in | (in << 16);
      if (in == 0u) a.l0[fs + __popc(z & lt)] = (uint16_t)u;
      fs += __popc(z);
    }
    cur = a.l0;
    nxt = a.l1;
    __syncwarp();
    while (fs > 0) {
      int f2 = 0;
      for (int i0 = 0; i0 < fs; i0 += 32) {
        const bool in = i0 + lane < fs;
        const int u = in ? cur[i0 + lane] : 0;
        const int cv = *(volatile int*)&a.dp[u];
        const int nd = cv + (int)len_of(u);
        const uint32_t ef = in ? a.ef[u] : 0u;
        const int deg = (int)((ef >> 16) & 0xFFu), e0 = (int)(ef & 0xFFFFu);
        const int md = __reduce_max_sync(kAll, deg);
        for (int k = 0; k < md; ++k) {
          const int ed = k < deg ? a.ed[e0 + k] : 0x8000, v = ed & 0x7FFF;
          bool q = false;
          if (ed & 0x8000) {
            if (k < deg && cv >= 0 && l < maxk) atomicMax((int*)&a.gx[v], nd);
          } else {
            if (cv >= 0) atomicMax((int*)&a.dp[v], nd);
            q = (atomicSub(&a.kk[v], 1u << 16) >> 16) == 1u;
          }
          const unsigned qm = __ballot_sync(kAll, q);
          if (q) nxt[f2 + __popc(qm & lt)] = (uint16_t)v;
          f2 += __popc(qm);
        }
      }
      __syncwarp();
      uint16_t* sw = cur; cur = nxt; nxt = sw;
      fs = f2;
    }
    for (int m = lane; m < nsrc; m += 32) {
      const bool cut = a.sk[m] >> 31;
      if ((cut && !every) || (int)(a.sk[m] & 0xFFFFu) != l) continue;
      int best = -1;
      uint32_t kind = 0;
      for (uint32_t o = a.sh[m]; o != 0xFFFFu; o = a.on[o]) {
        const int u = occ_node((int)o), d = *(volatile int*)&a.dp[u];
        kind = (a.oc[o] >> 29) & 3u;
        if (d >= 0) best = max(best, d + (int)len_of(u) - 1 - occ_pos((int)o));
      }
      if (best < 1) { capacity(P, 13); continue; }
      const int dmin = (int)(a.sd[m] >> kIdxBits);
      if (every) xemit(P, j, src_instr(m), r, dmin, l, best, cut || blocked);
      else emit_raw(P, A, j, src_instr(m), r, (int)kind, dmin, best);
    }
    __syncwarp();
    if (l < maxk) {
      for (int u = lane; u < n; u += 32) {
        a.dp[u] = a.gx[u];
        a.gx[u] = 0xFFFFFFFFu;
      }
      __syncwarp();
    }
  }
  phase(4);
  return 0;
}

// part 1: the searches queued for a class, largest class first (beside tiers 1
// and 2); part 2: the second tier's overflow, from the first class up.
__global__ void __launch_bounds__(768, 1) k_search_smem(Prog P, Arch A, int most_nodes, int part) {
  extern __shared__ __align__(16) char smem[];
  __shared__ int s_ctr[kWarps][8];
  __shared__ uint16_t s_wpos[kWarps][32];
  __shared__ int s_local[kClasses][kLocalList];  // use entries to redo in class c
  __shared__ int s_nlocal[kClasses], s_hlocal[kClasses];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const unsigned long long cap = (unsigned long long)P.queue_cap;
  // tasks of class c: queued by the local pass (at most its limit, the rest went
  // to the global-memory warps), or the second tier's overflow for the first class
  auto n_tasks = [&](int c) -> unsigned long long {
    if (part == 1) return min(P.stats[SS_A1_N + c], min(cap, (unsigned long long)P.class_limit[c]));
    return c == 0 ? min(P.stats[SS_OVF2_N], cap) : 0ull;
  };
  // Beside tiers 1 and 2 (part 1) no more SMs are taken than give every search a
  // warp at once: a CTA holds its SM's shared memory, which those tiers need too
  // (259 searches spread over all SMs kept them waiting).
  unsigned long long need = 0;
  for (int c = 0; c < kClasses; ++c) need += (n_tasks(c) + class_warps(c) - 1) / class_warps(c);
  if (need == 0 || (part == 1 && blockIdx.x >= need)) return;
  if (threadIdx.x < kClasses) { s_nlocal[threadIdx.x] = 0; s_hlocal[threadIdx.x] = 0; }
  __syncthreads();
  unsigned long long runs = 0, most = 0, most_task = 0;

  auto run_class = [&](int c, bool local) {
    const int n = class_nodes(c, most_nodes);
    if (warp < class_warps(c)) {
      const WArena a = carve(smem + warp * warp_arena_bytes(n), n, s_ctr[warp], s_wpos[warp]);
      const int32_t* q = P.queue[part == 1 ? class_queue(c) : 0];  // (queue 0: the second tier's overflow)
      const bool top = part == 1 && class_top(c);
      const int head = part == 1 ? SS_A1_HEAD + c : SS_OVF2_HEAD;
      const unsigned long long nt = n_tasks(c);
      const int list = local_list(c);
      while (true) {
        int e = -1;
        if (lane == 0) {
          if (local) {
            const int t = atomicAdd(&s_hlocal[c], 1);
            if (t < min(s_nlocal[c], list)) e = s_local[c][t];
          } else {
            const unsigned long long t = atomicAdd(&P.stats[head], 1ull);
            if (t < nt) e = q[top ? cap - 1 - t : t];
          }
        }
        e = __shfl_sync(0xffffffffu, e, 0);
        if (e < 0) break;
        const int2 task = P.tasks[e];
        const int j = task.x, r = task.y & 0x1FF;
        int met = 0;
        const int over = warp_search(P, A, a, j, r, (uint16_t)((uint32_t)task.y >> 9), e, (task.y >> 25) & 1, &met);
        const unsigned long long nn = (unsigned long long)met;
        __syncwarp();
        ++runs;
        most = max(most, nn);
        most_task = max(most_task, (nn << 40) | ((unsigned long long)r << 31) | (unsigned)j);
        if (lane != 0) continue;
#ifdef GPA_PHASE_TIMING
        atomicAdd(&P.stats[SS_SIZES + min(15, 31 - __clz(max((int)nn, 1)))], 1ull);
#endif
        if (!over) continue;
        int next = c + 1;  // the next class that is larger than this one
        while (next < kClasses && class_nodes(next, most_nodes) == n) ++next;
        raise_hint(P, e, (uint32_t)(kHintA1 + next));
        if (next < kClasses) {
          const int t = atomicAdd(&s_nlocal[next], 1);
          if (t < local_list(next)) { s_local[next][t] = e; continue; }
        }
        // beyond the last class, or the CTA's list is full
        const unsigned long long o = atomicAdd(&P.stats[SS_WIDE2_N], 1ull);
        if (o < cap) P.queue[6][cap - 1 - o] = e;
        else capacity(P, 8);
      }
    }
    __syncthreads();
  };
  if (part == 1) {
    for (int c = kClasses - 1; c >= 0; --c)
      if (n_tasks(c)) run_class(c, false);
  } else {
    run_class(0, false);
  }
  for (int c = 1; c < kClasses; ++c)
    if (s_nlocal[c]) run_class(c, true);
  if (lane == 0 && runs) {
    atomicAdd(&P.stats[SS_GENERAL], runs);
    atomicMax(&P.stats[SS_MAX_NODES], most);
    atomicMax(&P.stats[SS_MAX_TASK], most_task);
  }
}

}  // namespace

int smem_class_limit(int c, int sms) { return c < 2 ? INT_MAX : 3 * class_warps(c) * sms; }

void launch_search_smem(const Prog& P, const Arch& A, int most_nodes, int part, cudaStream_t st, int sms,
                        int64_t* launches) {
  size_t smem = 0;
  for (int c = 0; c < kClasses; ++c)
    smem = std::max(smem, (size_t)(class_warps(c) * warp_arena_bytes(class_nodes(c, most_nodes))));
  static_assert(kWarps * 32 <= 768, "the launch bound (768 threads: at most 80 registers each)");
  allow_max_smem(k_search_smem);
  const int grid = (int)std::max<int64_t>(1, std::min<int64_t>(sms, P.queue_cap));
  k_search_smem<<<grid, kWarps * 32, smem, st>>>(P, A, most_nodes, part);
  ++*launches;
}

}  // namespace gpa
