// Step (b)/(c), general backward searches (Sec. 4), first and second tier: one
// search per lane, its whole state in shared memory.
//
// Nine searches in ten meet fewer than 128 (block, literal set) nodes, most of
// them fewer than 16, and grow two or three nodes at a time, so a warp spent on
// one of them keeps one lane busy. Here every lane of a warp runs its own search:
// an arena of 9 words a node, interleaved by lane (word w of the lane's arena
// lies at w * LPW + lane), so whatever nodes the lanes are at, a warp's access
// touches one bank per lane. What bounds the kernel is the chain of dependent
// loads of each search (a block's record, then its events and its predecessors'
// reach words), so what counts is how many searches an SM has in flight: 352 of
// 16 nodes (eleven warps of 32 lanes) or 96 of 64 nodes (twelve warps of 8 lanes),
// as many as their arenas fit in shared memory. Searches of up to 64 nodes of the
// thousand-function step: 3.88 ms with a warp each, 0.42 + 1.01 ms in these two.
//
// The lanes of a warp are kept together by state, not by search: a step
// expands one node of every lane that is building its graph; lanes whose graph
// is complete wait until a quarter of the warp has one and finish theirs
// together (sources, rules 2 and 3, longest paths); idle lanes take new tasks
// together in the same way.
//
// The graph and its rules are those of the group search (k_search.cu): node 0 is
// the part of j's block above j; pass A expands nodes by distance, nearest first,
// up to `bound`; if some source is within its latency, pass B completes the
// graph with the nodes that can lie on a path from such a source. Two things
// differ, neither in what survives:
//  * nearest first, a node's distance is final when it is expanded, so edges are
//    relaxed once;
//  * a search ends when its only unexpanded node meets an unguarded reader of r
//    before any def of r was met: every path to every source passes that reader,
//    so none survives rule 2 (a third of the searches on the batched workload).
// Searches that outgrow the arena go on to the next tier.
#include <algorithm>

#include "gpa_internal.cuh"

namespace gpa {

namespace {

// A node's words.
enum {
  W_KEY = 0,   // block (relative to the function) | literal set << 16
  W_DIST = 1,  // shortest distance << 8 | parent; then rule 2's reach mask; then a layer's longest distance
  W_INFO = 2,  // wall position (0xFFFF: none) | fewest back edges << 16 | flags << 24
  W_EDGE = 3,  // first edge | edges << 8 | forward in-edges << 16 | wall group + 1, or in-edges left << 24
  W_LEN = 4,   // instructions of the block (node 0: up to and including j) | list entry << 16
  W_NEXT = 5,  // the next layer's longest distance
  kNodeWords = 6
};
enum { F_QUEUED = 1 };
constexpr uint32_t kFar = 0xFFFFFFu;  // no distance yet (distances are below 128 * 65,535)
constexpr int kOccWords = 3;          // position | node << 16 | def kind << 24; distance << 8 | nearest
                                      // occurrence; source | back edges << 8 | within latency << 16 | kept << 17

__host__ __device__ inline int lane_occs(int n) { return n / 2 + 4; }
__host__ __device__ inline int lane_words(int n) {
  // nodes, 2n edge bytes, 2n hash bytes (at least a word each), occurrences
  return kNodeWords * n + 2 * ((2 * n + 3) / 4) + kOccWords * lane_occs(n);
}

__device__ __forceinline__ uint32_t lane_hash(int blk, int S) {
  uint32_t h = (uint32_t)blk * 0x9E3779B1u ^ ((uint32_t)S * 0x85EBCA77u);
  return h ^ (h >> 15);
}

// The arena of one lane: words at stride LPW, bytes and half words within them.
template <int LPW>
struct LaneArena {
  uint32_t* w;       // this lane's word 0
  int n, edges, hash, occ;  // nodes; word offsets of the edge bytes, the hash bytes, the occurrences
  __device__ __forceinline__ uint32_t& word(int i) const { return w[i * LPW]; }
  __device__ __forceinline__ uint32_t& node(int u, int f) const { return w[(u * kNodeWords + f) * LPW]; }
  __device__ __forceinline__ uint16_t& half(int u, int f, int k) const {
    return reinterpret_cast<uint16_t*>(&w[(u * kNodeWords + f) * LPW])[k];
  }
  __device__ __forceinline__ uint8_t& byte(int u, int f, int k) const {
    return reinterpret_cast<uint8_t*>(&w[(u * kNodeWords + f) * LPW])[k];
  }
  __device__ __forceinline__ uint8_t& edge(int e) const {
    return reinterpret_cast<uint8_t*>(&w[(edges + (e >> 2)) * LPW])[e & 3];
  }
  __device__ __forceinline__ uint8_t& slot(int h) const {
    return reinterpret_cast<uint8_t*>(&w[(hash + (h >> 2)) * LPW])[h & 3];
  }
  __device__ __forceinline__ uint16_t& wallpos(int g) const {  // over the hash, once the graph is complete
    return reinterpret_cast<uint16_t*>(&w[(hash + (g >> 1)) * LPW])[g & 1];
  }
  __device__ __forceinline__ uint32_t& o(int i, int f) const { return w[(occ + i * kOccWords + f) * LPW]; }
  __device__ __forceinline__ uint8_t& list(int i) const { return byte(i, W_LEN, 2); }
};

enum { L_IDLE = 0, L_GROW = 1, L_FINISH = 2, L_NONE = 3 };

// One lane's search.
template <int LPW>
struct LaneSearch {
  LaneArena<LPW> a;
  int state;
  int j, r, gj, e_use, b0, fb, bound, low;  // low: pass B's least block
  uint16_t live;
  bool blocked, pass_b, back;               // back: the graph has a back edge
  int nn, ne, no, nl;                       // nodes, edges, occurrences, unexpanded nodes
  int over;                                 // why the arena is too small (0: it is not)

  __device__ __forceinline__ void begin(const Prog& P, int e) {
    const int2 task = P.tasks[e];
    e_use = e;
    j = task.x;
    r = task.y & 0x1FF;
    blocked = (task.y >> 25) & 1;
    gj = P.guard[j];
    b0 = P.instr_block[j];
    const int f = P.block_func[b0];
    fb = P.func_block_off[f];
    const size_t fr = (size_t)f * kNumRes + r;
    bound = P.diag ? 0x7FFFFFFF : P.res_maxlat[fr];  // the coverage count needs every source
    live = live_literals(P.res_guards[fr], gj);
    const uint16_t S0 = keep_literals((uint16_t)((uint32_t)task.y >> 9), live);
    over = P.func_block_off[f + 1] - fb > 0xFFFF ? 1 : 0;
    for (int h = 0; h < a.occ - a.hash; ++h) a.word(a.hash + h) = 0u;
    a.node(0, W_KEY) = (uint32_t)(b0 - fb) | ((uint32_t)S0 << 16);
    a.node(0, W_DIST) = 0u;
    a.node(0, W_INFO) = 0xFFFFu;
    a.node(0, W_EDGE) = 0u;
    a.node(0, W_LEN) = 0u;
    a.list(0) = 0;
    nn = 1; ne = 0; no = 0; nl = 1;
    pass_b = false; back = false; low = 0;
    state = over ? L_FINISH : L_GROW;
  }

  // Expands the nearest unexpanded node.
  __device__ void grow(const Prog& P) {
    int at = -1;
    uint32_t dk = 0xFFFFFFFFu;
    for (int i = 0; i < nl; ++i) {
      const uint32_t d = a.node(a.list(i), W_DIST);
      if (d < dk) { dk = d; at = i; }
    }
    if (at < 0 || (!pass_b && (int)(dk >> 8) > bound)) { state = L_FINISH; return; }
    const int u = a.list(at);
    a.list(at) = a.list(--nl);
    const bool only = nl == 0 && no == 0 && !pass_b && !P.diag;  // every path on passes u, no source yet
    const uint32_t key = a.node(u, W_KEY);
    const int B = fb + (int)(key & 0xFFFFu);
    uint16_t S = (uint16_t)(key >> 16);
    const int w = r >> 5;
    const uint32_t bit = 1u << (r & 31);
    // First round of loads: the block's record, the touch word of r, the bounds
    // of r's event segment. Second round: the reach words of its first two
    // predecessors and the events.
    const int4 m0 = __ldg(&P.block_meta[2 * (size_t)B]);
    const int4 pm = __ldg(&P.block_meta[2 * (size_t)B + 1]);
    const uint32_t tw = __ldg(&P.touch_mask[(size_t)B * kWords + w]);
    const size_t seg = (size_t)B * kEvBuckets + ev_bucket(r);
    const int ev_beg = __ldg(&P.ev_off[seg]);
    int ev_end = __ldg(&P.ev_off[seg + 1]);
    if (!(tw & bit) || u == 0) ev_end = ev_beg;  // nothing to scan (node 0: the local pass has)
    const uint32_t ro0 = pm.z >= 0 ? P.rout[(size_t)pm.z * kWords + w] : 0u;
    const uint32_t ro1 = pm.w >= 0 ? P.rout[(size_t)pm.w * kWords + w] : 0u;
    bool stop = false, cut = false;
    int wall = 0xFFFF, last_def = -1;
    for (int e0 = ev_beg; e0 < ev_end && !stop && !cut; e0 += 4) {
      uint32_t evs[4];
#pragma unroll
      for (int q = 0; q < 4; ++q) evs[q] = e0 + q < ev_end ? __ldg(&P.events[e0 + q]) : 0x1FFu;
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const uint32_t ev = evs[q];
        if (stop || cut || (int)(ev & 0x1FFu) != r) continue;
        const int pos = (int)(ev >> 16), x = m0.x + pos;
        if (ev & 0x200u) {  // def of r
          last_def = pos;
          if (!contains(S, gj) && !(B == b0 && x < j)) {  // sources above j in its block are settled
            if (no < lane_occs(a.n)) a.o(no, 0) = (uint32_t)pos | ((uint32_t)u << 16) | (((ev >> 10) & 3u) << 24);
            else over = 3;
            ++no;
          }
          S = add_literal(S, (int)((ev >> 12) & 0xFu));
          if (contains(S, gj)) stop = true;
        } else if (wall == 0xFFFF && pos != last_def && x != j) {  // unguarded reader of r
          wall = pos;
          if (only && no == 0) cut = true;
        }
      }
    }
    if (cut) { no = 0; pass_b = true; state = L_FINISH; return; }  // nothing survives: see finish()
    const int len = u == 0 ? j - m0.x + 1 : m0.y - m0.x;
    a.half(u, W_INFO, 0) = (uint16_t)wall;
    a.half(u, W_LEN, 0) = (uint16_t)len;
    a.byte(u, W_EDGE, 0) = (uint8_t)ne;
    const int Sout = (int)keep_literals(S, live);
    const uint32_t nd = (((dk >> 8) + (uint32_t)len) << 8) | (uint32_t)u;
    const int ne0 = ne;
    if (!stop && !over) {
      const int hm = 2 * a.n - 1;
      for (int q = pm.x; q < pm.y; ++q) {
        const int k = q - pm.x;
        const int p = k == 0 ? pm.z : k == 1 ? pm.w : __ldg(&P.pred[q]);
        const uint32_t ro = k == 0 ? ro0 : k == 1 ? ro1 : P.rout[(size_t)p * kWords + w];
        if (!(ro & bit)) continue;
        if (ne >= 2 * a.n) { over = 2; break; }
        const uint32_t pk = (uint32_t)(p - fb) | ((uint32_t)Sout << 16);
        int h = (int)(lane_hash(p, Sout) & (uint32_t)hm);
        int v = a.slot(h);
        while (v && a.node(v, W_KEY) != pk) {  // ends: at most n of the 2n slots are taken
          h = (h + 1) & hm;
          v = a.slot(h);
        }
        if (!v) {
          if (nn >= a.n) { over = 1; break; }
          v = nn++;
          a.slot(h) = (uint8_t)v;
          a.node(v, W_KEY) = pk;
          a.node(v, W_DIST) = kFar << 8;
          a.node(v, W_INFO) = 0xFFFFu | (0xFFu << 16);
          a.node(v, W_EDGE) = 0u;
          a.half(v, W_LEN, 0) = 0;
          if (!pass_b || p >= low) a.list(nl++) = (uint8_t)v;
        }
        if (nd < a.node(v, W_DIST)) a.node(v, W_DIST) = nd;
        back |= p >= B;
        a.edge(ne++) = (uint8_t)(v | (p >= B ? 0x80 : 0));
      }
    }
    a.byte(u, W_EDGE, 1) = (uint8_t)(ne - ne0);
    if (over) state = L_FINISH;
  }

  __device__ __forceinline__ int wall_of(int u) const { return a.half(u, W_INFO, 0); }
  __device__ __forceinline__ int len_of(int u) const { return a.half(u, W_LEN, 0); }
  __device__ __forceinline__ int occ_node(int o) const { return (a.o(o, 0) >> 16) & 0xFF; }
  __device__ __forceinline__ int occ_pos(int o) const { return a.o(o, 0) & 0xFFFF; }
  __device__ __forceinline__ int block_of(int u) const { return (int)(a.node(u, W_KEY) & 0xFFFFu); }
  __device__ __forceinline__ int occ_dist(int o) const {
    const int u = occ_node(o);
    return (int)(a.node(u, W_DIST) >> 8) + len_of(u) - 1 - occ_pos(o);
  }
  __device__ __forceinline__ int occ_instr(const Prog& P, int o) const {
    return P.block_meta[2 * (size_t)(fb + block_of(occ_node(o)))].x + occ_pos(o);
  }
  __device__ __forceinline__ int source_of(int o) const { return a.o(o, 2) & 0xFF; }
  __device__ __forceinline__ bool kept(int o) const { return (a.o(o, 2) >> 17) & 1u; }

  // The graph is complete up to this pass: returns true when the search goes
  // on with pass B, false when it is done (over: why it has to be redone in the
  // next tier).
  __device__ bool finish(const Prog& P, const Arch& A) {
    if (over) return false;
    if (!pass_b) {
      int lo = 0x7FFFFFFF;
      for (int o = 0; o < no; ++o) {
        const int d = occ_dist(o);
        bool within = false;
        if (d <= bound) {
          within = d <= A.lat[P.opclass[occ_instr(P, o)]];
          if (within) lo = min(lo, P.block_minreach[fb + block_of(occ_node(o))]);
        }
        a.o(o, 2) = within ? 1u << 16 : 0u;
      }
      if (lo == 0x7FFFFFFF && !P.diag) return false;
      // Pass B: the unexpanded nodes that can lie on a path from such a source.
      // (The diagnostics have no bound: pass A left no node unexpanded.)
      pass_b = true;
      low = lo;
      int keep = 0;
      for (int i = 0; i < nl; ++i) {
        const int u = a.list(i);
        if (fb + block_of(u) >= low) a.list(keep++) = (uint8_t)u;
      }
      nl = keep;
      if (nl > 0) {
        // occurrences of pass B lie beyond the bound: none is within its latency
        for (int o = no; o < lane_occs(a.n); ++o) a.o(o, 2) = 0u;
        return true;
      }
    }
    if (no == 0) {
      if (P.diag == 1) cov_add(P, e_use, 0, 0);
      return false;
    }

    // Fewest back edges from j (all zero without a back edge in the graph).
    a.byte(0, W_INFO, 2) = 0;
    if (back) {
      int head = 0, tail = 1 == a.n ? 0 : 1, inq = 1;
      a.list(0) = 0;
      while (inq > 0) {
        const int u = a.list(head);
        head = head + 1 == a.n ? 0 : head + 1;
        --inq;
        a.byte(u, W_INFO, 3) &= ~F_QUEUED;
        const int ku = a.byte(u, W_INFO, 2);
        const int e0 = a.byte(u, W_EDGE, 0), e1 = e0 + a.byte(u, W_EDGE, 1);
        for (int e = e0; e < e1; ++e) {
          const int ed = a.edge(e), v = ed & 0x7F, k = ku + (ed >> 7);
          if (k >= a.byte(v, W_INFO, 2)) continue;
          a.byte(v, W_INFO, 2) = (uint8_t)k;
          if (a.byte(v, W_INFO, 3) & F_QUEUED) continue;
          a.byte(v, W_INFO, 3) |= F_QUEUED;
          a.list(tail) = (uint8_t)v;
          tail = tail + 1 == a.n ? 0 : tail + 1;
          ++inq;
        }
      }
    }

    // Sources: the occurrences of one instruction (same block and position)
    // belong to the first of them, which keeps the shortest distance, the nearest
    // occurrence and the fewest back edges. Rule 3.
    int nsrc = 0, alive = 0;
    for (int o = 0; o < no; ++o) {
      const int u = occ_node(o), B = block_of(u), pos = occ_pos(o);
      int s = 0;
      while (s < o && !(source_of(s) == s && occ_pos(s) == pos && block_of(occ_node(s)) == B)) ++s;
      const uint32_t db = ((uint32_t)occ_dist(o) << 8) | (uint32_t)o;
      const uint32_t k = back ? a.byte(u, W_INFO, 2) : 0u;
      const uint32_t within = a.o(o, 2) & (1u << 16);
      if (s == o) {
        ++nsrc;
        a.o(o, 1) = db;
        a.o(o, 2) = (uint32_t)o | (k << 8) | within;
      } else {
        if (db < a.o(s, 1)) a.o(s, 1) = db;
        const uint32_t t = a.o(s, 2);
        a.o(s, 2) = (t & ~0xFF00u) | (min(k, (t >> 8) & 0xFFu) << 8) | within;
        a.o(o, 2) = (uint32_t)s;
      }
    }
    for (int s = 0; s < no; ++s) {
      if (source_of(s) != s) continue;
      bool ok = (a.o(s, 2) >> 16) & 1u;
      // coverage: rule 2 above j and rule 1; the export tests rule 2 for every source
      if (P.diag == 1 && ok && (blocked || !keeps_any(P, A, j, P.opclass[occ_instr(P, s)]))) ok = false;
      if (P.diag == 2) ok = true;
      if (ok) { a.o(s, 2) |= 1u << 17; ++alive; }
    }
    if (alive == 0) {
      if (P.diag == 1) cov_add(P, e_use, nsrc, 0);
      return false;
    }

    // Rule 2. A block's wall group: the unguarded reader met first from the
    // bottom over its nodes. It can cut a source only if it lies on the parent
    // chain of the source's nearest occurrence; the groups needed get a bit each.
    int ng = 0;
    auto need = [&](int u) {
      if (a.byte(u, W_EDGE, 3)) return;  // its block's group has a bit
      if (ng == 32) { over = 1; return; }
      const int B = block_of(u);
      int wp = 0;
      for (int v = 1; v < nn; ++v) {
        if (block_of(v) != B || wall_of(v) == 0xFFFF) continue;
        a.byte(v, W_EDGE, 3) = (uint8_t)(ng + 1);
        wp = max(wp, wall_of(v));
      }
      a.wallpos(ng++) = (uint16_t)wp;
    };
    for (int s = 0; s < no; ++s) {
      if (source_of(s) != s || !kept(s)) continue;
      const int o = (int)(a.o(s, 1) & 0xFFu);
      const int u = occ_node(o);
      const int wu = wall_of(u);
      if (wu != 0xFFFF && wu > occ_pos(o)) need(u);
      for (int v = (int)(a.node(u, W_DIST) & 0xFFu), hops = 0; v > 0 && hops < nn;
           v = (int)(a.node(v, W_DIST) & 0xFFu), ++hops)
        if (wall_of(v) != 0xFFFF) need(v);
    }
    if (over) return false;
    if (ng > 0) {
      // Bit g of a node's reach mask: reached without passing group g's wall. A
      // node of the group passes every bit on but its own.
      const uint32_t full = ng == 32 ? 0xFFFFFFFFu : (1u << ng) - 1u;
      for (int u = 1; u < nn; ++u) a.node(u, W_DIST) = 0u;
      a.node(0, W_DIST) = full;
      int head = 0, tail = 1 == a.n ? 0 : 1, inq = 1;
      a.list(0) = 0;
      while (inq > 0) {
        const int u = a.list(head);
        head = head + 1 == a.n ? 0 : head + 1;
        --inq;
        a.byte(u, W_INFO, 3) &= ~F_QUEUED;
        const int gu = u ? a.byte(u, W_EDGE, 3) : 0;
        const uint32_t m = a.node(u, W_DIST) & (gu ? ~(1u << (gu - 1)) : 0xFFFFFFFFu);
        const int e0 = a.byte(u, W_EDGE, 0), e1 = e0 + a.byte(u, W_EDGE, 1);
        for (int e = e0; e < e1; ++e) {
          const int v = a.edge(e) & 0x7F;
          const uint32_t old = a.node(v, W_DIST);
          if (!(m & ~old)) continue;
          a.node(v, W_DIST) = old | m;
          if (a.byte(v, W_INFO, 3) & F_QUEUED) continue;
          a.byte(v, W_INFO, 3) |= F_QUEUED;
          a.list(tail) = (uint8_t)v;
          tail = tail + 1 == a.n ? 0 : tail + 1;
          ++inq;
        }
      }
      for (int s = 0; s < no; ++s) {
        if (source_of(s) != s || !kept(s)) continue;
        uint32_t ok = 0u;
        for (int o = s; o < no && ok != full; ++o) {
          if (source_of(o) != s) continue;
          const int u = occ_node(o), gu = a.byte(u, W_EDGE, 3);
          uint32_t m = a.node(u, W_DIST);
          if (gu && occ_pos(o) < (int)a.wallpos(gu - 1)) m &= ~(1u << (gu - 1));
          ok |= m;
        }
        if (ok != full) { a.o(s, 2) &= ~(1u << 17); --alive; }
      }
    }
    if (P.diag == 1) {
      cov_add(P, e_use, nsrc, alive);
      return false;
    }
    const bool every = P.diag == 2;  // the export keeps every source (rule 2's cut is its dom flag)
    if (alive == 0 && !every) return false;

    // Longest path with exactly K back edges, layer by layer: Kahn's order over
    // the forward edges; back edges feed the next layer.
    int maxk = 0;
    for (int s = 0; s < no; ++s)
      if (source_of(s) == s && (kept(s) || every)) maxk = max(maxk, (int)((a.o(s, 2) >> 8) & 0xFFu));
    if (maxk >= kMaxLayers) { over = 5; return false; }
    for (int u = 0; u < nn; ++u) {
      a.half(u, W_EDGE, 1) = 0;
      a.node(u, W_DIST) = 0xFFFFFFFFu;
      a.node(u, W_NEXT) = 0xFFFFFFFFu;
    }
    for (int e = 0; e < ne; ++e) {
      const int ed = a.edge(e);
      if (!(ed & 0x80)) a.byte(ed, W_EDGE, 2) = (uint8_t)(a.byte(ed, W_EDGE, 2) + 1);
    }
    a.node(0, W_DIST) = 0u;
    for (int l = 0; l <= maxk; ++l) {
      int tail = 0;
      for (int u = 0; u < nn; ++u) {
        const uint8_t in = a.byte(u, W_EDGE, 2);
        a.byte(u, W_EDGE, 3) = in;
        if (in == 0) a.list(tail++) = (uint8_t)u;
      }
      for (int head = 0; head < tail; ++head) {
        const int u = a.list(head);
        const int cv = (int)a.node(u, W_DIST);
        const int nd = cv + len_of(u);
        const int e0 = a.byte(u, W_EDGE, 0), e1 = e0 + a.byte(u, W_EDGE, 1);
        for (int e = e0; e < e1; ++e) {
          const int ed = a.edge(e), v = ed & 0x7F;
          if (ed & 0x80) {
            if (cv >= 0 && l < maxk && nd > (int)a.node(v, W_NEXT)) a.node(v, W_NEXT) = (uint32_t)nd;
          } else {
            if (cv >= 0 && nd > (int)a.node(v, W_DIST)) a.node(v, W_DIST) = (uint32_t)nd;
            const uint8_t left = (uint8_t)(a.byte(v, W_EDGE, 3) - 1);
            a.byte(v, W_EDGE, 3) = left;
            if (left == 0) a.list(tail++) = (uint8_t)v;
          }
        }
      }
      for (int s = 0; s < no; ++s) {
        if (source_of(s) != s || !(kept(s) || every) || (int)((a.o(s, 2) >> 8) & 0xFFu) != l) continue;
        int best = -1;
        for (int o = s; o < no; ++o) {
          if (source_of(o) != s) continue;
          const int u = occ_node(o), d = (int)a.node(u, W_DIST);
          if (d >= 0) best = max(best, d + len_of(u) - 1 - occ_pos(o));
        }
        if (best < 1) { capacity(P, 13); continue; }
        const int i = occ_instr(P, s), dmin = (int)(a.o(s, 1) >> 8);
        if (every) xemit(P, j, i, r, dmin, l, best, !kept(s) || blocked);
        else emit_raw(P, A, j, i, r, (int)((a.o(s, 0) >> 24) & 3u), dmin, best);
      }
      if (l < maxk)
        for (int u = 0; u < nn; ++u) {
          a.node(u, W_DIST) = a.node(u, W_NEXT);
          a.node(u, W_NEXT) = 0xFFFFFFFFu;
        }
    }
    return false;
  }
};

// Persistent one-warp CTAs over one queue of (use, resource) tasks: the first
// tier reads the local pass's queue, the second the first tier's overflow.
template <int LPW>
__global__ void __launch_bounds__(32) k_search_lanes(Prog P, Arch A, int nodes, int tier) {
  extern __shared__ __align__(16) uint32_t lane_sm[];
  const int lane = threadIdx.x;
  const unsigned long long cap = (unsigned long long)P.queue_cap;
  const int32_t* queue = P.queue[tier - 1];
  const unsigned long long n_tasks = min(P.stats[tier == 1 ? SS_QUEUE_N : SS_OVF_N], cap);
  unsigned long long* head = &P.stats[tier == 1 ? SS_QUEUE_HEAD : SS_OVF_HEAD];
  if (n_tasks == 0) return;

  LaneSearch<LPW> s;
  s.a.w = lane_sm + lane;
  s.a.n = nodes;
  s.a.edges = kNodeWords * nodes;
  s.a.hash = s.a.edges + (2 * nodes + 3) / 4;
  s.a.occ = s.a.hash + (2 * nodes + 3) / 4;
  // Few tasks are spread over the warps: fewer lanes of each take part.
  const int width = (int)min((unsigned long long)LPW, (n_tasks + gridDim.x - 1) / gridDim.x);
  const int batch = max(1, width / 4);
  s.state = lane < width ? L_IDLE : L_NONE;
  bool more = true;              // the queue may hold another task
  unsigned long long runs = 0, most = 0, most_task = 0;
  while (true) {
    const unsigned idle = __ballot_sync(0xffffffffu, s.state == L_IDLE);
    const unsigned growing = __ballot_sync(0xffffffffu, s.state == L_GROW);
    const unsigned done = __ballot_sync(0xffffffffu, s.state == L_FINISH);
    if (done && (__popc(done) >= batch || !growing)) {
      if (s.state == L_FINISH) {
        if (s.finish(P, A)) {
          s.state = L_GROW;  // pass B
        } else {
          s.state = L_IDLE;
          ++runs;
          const unsigned long long t =
              ((unsigned long long)s.nn << 40) | ((unsigned long long)s.r << 31) | (unsigned)s.j;
          most_task = max(most_task, t);
          most = max(most, (unsigned long long)s.nn);
#ifdef GPA_PHASE_TIMING
          atomicAdd(&P.stats[SS_SIZES + min(15, 31 - __clz(s.nn))], 1ull);
#endif
          if (s.over) {
            raise_hint(P, s.e_use, (uint32_t)(tier + 1));
            // first tier -> bottom of queue 1; second tier -> bottom of queue 0
            const unsigned long long o = atomicAdd(&P.stats[tier == 1 ? SS_OVF_N : SS_OVF2_N], 1ull);
            if (o < cap) P.queue[2 - tier][o] = s.e_use;
            else capacity(P, 8);
          }
        }
      }
      __syncwarp();
    } else if (more && idle && (__popc(idle) >= batch || !growing)) {
      unsigned long long t = 0;
      const int first = __ffs(idle) - 1;
      if (lane == first) t = atomicAdd(head, (unsigned long long)__popc(idle));
      t = __shfl_sync(0xffffffffu, t, first);
      more = t + (unsigned long long)__popc(idle) < n_tasks;
      if (s.state == L_IDLE) {
        t += (unsigned long long)__popc(idle & ((1u << lane) - 1u));
        if (t < n_tasks) s.begin(P, queue[t]);
      }
      __syncwarp();
    } else if (growing) {
      if (s.state == L_GROW) s.grow(P);
      __syncwarp();
    } else {
      break;
    }
  }
  for (int o = 16; o > 0; o >>= 1) {
    runs += __shfl_xor_sync(0xffffffffu, runs, o);
    most = max(most, __shfl_xor_sync(0xffffffffu, most, o));
    most_task = max(most_task, __shfl_xor_sync(0xffffffffu, most_task, o));
  }
  if (lane == 0 && runs) {
    atomicAdd(&P.stats[SS_GENERAL], runs);
    atomicMax(&P.stats[SS_MAX_NODES], most);
    atomicMax(&P.stats[SS_MAX_TASK], most_task);
  }
}

}  // namespace

// How the lanes are packed in warps matters little, since their arenas alone
// decide how many searches an SM holds: 16 lanes of 16 nodes or 4 of 64 measured
// the same on the thousand-function step (6.83-6.87 ms), 16 of 64 7.16 ms.
int search_lane_width(int nodes) { return nodes <= 32 ? 32 : 8; }
int64_t search_lane_bytes(int nodes) { return 4ll * lane_words(nodes) * search_lane_width(nodes); }

void launch_search_lanes(const Prog& P, const Arch& A, const SearchArena& T, int tier, cudaStream_t st,
                         int64_t* launches) {
  const int grid = (int)std::max<int64_t>(1, std::min<int64_t>(T.warps, P.queue_cap));
  if (search_lane_width(T.nodes) == 32) {
    cudaFuncSetAttribute(k_search_lanes<32>, cudaFuncAttributePreferredSharedMemoryCarveout, 100);
    k_search_lanes<32><<<grid, 32, (size_t)T.bytes, st>>>(P, A, T.nodes, tier);
  } else {
    cudaFuncSetAttribute(k_search_lanes<8>, cudaFuncAttributePreferredSharedMemoryCarveout, 100);
    k_search_lanes<8><<<grid, 32, (size_t)T.bytes, st>>>(P, A, T.nodes, tier);
  }
  ++*launches;
}

}  // namespace gpa
