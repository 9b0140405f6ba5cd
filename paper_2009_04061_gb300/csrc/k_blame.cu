// Steps (b) and (c), Sec. 4: backward slicing with virtual barrier registers
// and predicate coverage, the three pruning rules, and Eq. 1 apportioning.
//
// For each stalled use j and each resource r it reads, the immediate sources
// are the defs of r reached backwards from j while the union P of the guard
// literals of the defs met so far does not contain j's guard (Sec. 4,
// "Predicated instructions"); "_" is contained by everything and Pi with !Pi
// makes "_". A source i survives if (rule 2) no single unguarded reader k of r
// (k not i, j) lies on every source path from i to j, and (rule 3) its
// shortest source path is at most latency(i). Sources reached through several
// resources merge into one source i; Eq. 1 then splits each dependency class
// and latency flag of j by issue_i / longest_path_i among the sources that
// (rule 1) match the class's opcode rule.
//
// Work split:
//  * k_search_local: four threads per stalled use, one linear scan per
//    resource inside j's block. It settles every source of that block
//    (their only path is the straight segment) and stops at coverage or at
//    the first unguarded reader of r (that reader lies on every path beyond,
//    so nothing further can survive rule 2). If every predecessor block
//    through which a def of r arrives covers j's guard, those predecessors
//    are settled here too (one path per source); otherwise the (use,
//    resource) pair is queued.
//  * k_search_lanes, k_search_smem, k_search_warp, k_search_cta: persistent
//    lanes, warps and CTAs pull queued (use, resource) pairs and explore the
//    (block, literal set) graph, by its size.
//  * k_merge_count / scan / k_apportion: merge sources per use, apportion in
//    integers, scatter blame with 64-bit atomics.
#include <algorithm>

#include "gpa_internal.cuh"

namespace gpa {

namespace {

__device__ __forceinline__ int dep_class(int ci) {
  return ci == 0 ? GPA_EXEC_DEPENDENCY : ci == 1 ? GPA_MEMORY_DEPENDENCY : ci == 2 ? GPA_SYNC : GPA_CONSTANT_MEMORY_DEPENDENCY;
}

// Scans predecessor block p of j's block b0 bottom-up for resource r, from
// the literal set S left at the top of b0. Returns true if p covers j's
// guard. With emit, emits p's sources that survive rules 2 and 3: when every
// predecessor covers, a source has exactly one def-clear path (from j up to
// the top of b0, into p at its bottom and up to the source), so its shortest
// and longest distances are that path's length d0 + (last(p) - x), and
// rule 2 reduces to an unguarded reader of r below it in p (met first in the
// bottom-up scan). Defs above j in b0 are settled by the in-block scan.
__device__ bool scan_pred(const Prog& P, const Arch& A, int j, int r, int gj, int b0, int p, uint16_t S, int d0,
                          bool emit, int* n_all = nullptr, int* n_kept = nullptr, bool blocked = false) {
  const int first = P.block_instr_off[p], last = P.block_instr_off[p + 1] - 1;
  bool wall = false;
  int last_def_pos = -1;
  const size_t seg = (size_t)p * kEvBuckets + ev_bucket(r);  // p's events of r's bucket
  const int ev1 = P.ev_off[seg + 1];
  for (int t = P.ev_off[seg]; t < ev1; ++t) {
    const uint32_t ev = P.events[t];
    if ((int)(ev & 0x1FFu) != r) continue;
    const int pos = (int)(ev >> 16), x = first + pos;
    if (ev & 0x200u) {
      last_def_pos = pos;
      if (!contains(S, gj) && !(p == b0 && x < j)) {
        const int d = d0 + (last - x);
        const bool keep = !wall && d <= A.lat[P.opclass[x]];
        if (emit && keep) emit_raw(P, A, j, x, r, (int)((ev >> 10) & 3u), d, d);
        if (n_all) {  // coverage count
          ++*n_all;
          if (keep && !blocked && keeps_any(P, A, j, P.opclass[x])) ++*n_kept;
        }
        if (P.diag == 2 && n_all) xemit(P, j, x, r, d, p >= b0 ? 1 : 0, d, wall || blocked);
      }
      S = add_literal(S, (int)((ev >> 12) & 0xFu));
      if (contains(S, gj)) return true;
    } else if (!wall && pos != last_def_pos && x != j) {
      wall = true;
    }
  }
  return false;
}

// The stalled uses (instructions with dependency-class samples), appended a
// warp at a time: a tenth of the instructions on the batched workload, so the
// kernels that work per stalled use take them from this list with every lane
// busy instead of striding over all instructions. With `init`, the pass also
// starts the blame: the samples outside the dependency classes stay where they
// were taken, the others are apportioned later. A warp takes 32 rows of 24
// counters, 6 KB, as twelve coalesced 16-byte loads a lane (a pair is one class of
// one row), and marks the rows with stalls in shared memory; reading the rows
// again for the list alone took 114 us on 3.3M instructions.
__global__ void __launch_bounds__(256) k_stalled_list(Prog P, int init) {
  __shared__ int s_row[8][32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int x0 = (blockIdx.x * 8 + warp) * 32;
  if (x0 >= P.ni) return;
  s_row[warp][lane] = 0;
  __syncwarp();
  const ulonglong2* c = reinterpret_cast<const ulonglong2*>(P.cnt + (size_t)x0 * kCnt);
  ulonglong2* b = reinterpret_cast<ulonglong2*>(P.blame + (size_t)x0 * kCnt);
  const int pairs = min(32, P.ni - x0) * (kCnt / 2);
#pragma unroll
  for (int i = 0; i < kCnt / 2; ++i) {
    const int p = i * 32 + lane;
    if (p < pairs) {
      const ulonglong2 v = c[p];
      const int row = p / (kCnt / 2), cls = p - row * (kCnt / 2);
      const bool dep = cls == GPA_EXEC_DEPENDENCY || cls == GPA_MEMORY_DEPENDENCY || cls == GPA_SYNC ||
                       cls == GPA_CONSTANT_MEMORY_DEPENDENCY;
      if (dep && (v.x | v.y)) s_row[warp][row] = 1;
      if (init) b[p] = dep ? make_ulonglong2(0ull, 0ull) : v;
    }
  }
  if (init && x0 + lane < P.ni) P.head[x0 + lane] = -1;
  __syncwarp();
  const bool s = s_row[warp][lane];
  const unsigned m = __ballot_sync(0xffffffffu, s);
  if (!m) return;
  unsigned long long base = 0;
  if (lane == 0) base = atomicAdd(&P.stats[SS_SUSE_N], (unsigned long long)__popc(m));
  base = __shfl_sync(0xffffffffu, base, 0);
  if (s) P.suse[base + __popc(m & ((1u << lane) - 1u))] = x0 + lane;
}

// Four threads per stalled use (from the stalled-use list), each taking every
// fourth resource the use reads: a resource's scans are a chain of dependent
// loads, so a thread per use ran its two or three of them one after another
// (55 us for a 200-instruction program).
constexpr int kLocalLanes = 4;
__global__ void k_search_local(Prog P, Arch A) {
  const int n_suse = (int)P.stats[SS_SUSE_N];
  for (int64_t kk = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; kk < (int64_t)n_suse * kLocalLanes;
       kk += (int64_t)gridDim.x * blockDim.x) {
    const int j = P.suse[kk / kLocalLanes];
    const int gj = P.guard[j];
    const int b0 = P.instr_block[j];
    const int first = P.block_instr_off[b0];
    const int pj = j - first;
    const int e_end = P.use_off[j + 1];
    for (int e = P.use_off[j] + (int)(kk % kLocalLanes); e < e_end; e += kLocalLanes) {
      const int r = P.use_res[e] & 0x1FF;
      const size_t seg = (size_t)b0 * kEvBuckets + ev_bucket(r);  // b0's events of r's bucket
      const int ev0 = P.ev_off[seg], ev1 = P.ev_off[seg + 1];
      uint16_t S = 0;
      bool blocked = false, covered = false;
      int last_def_pos = -1;
      int n_all = 0, n_kept = 0;  // coverage count (P.diag)
      for (int t = ev0; t < ev1; ++t) {  // bottom-up
        const uint32_t ev = P.events[t];
        const int pos = (int)(ev >> 16);
        if (pos >= pj || (int)(ev & 0x1FFu) != r) continue;
        const int x = first + pos;
        if (ev & 0x200u) {
          last_def_pos = pos;
          if (!contains(S, gj)) {
            const int d = pj - pos;
            if (!P.diag) {
              if (d <= A.lat[P.opclass[x]]) emit_raw(P, A, j, x, r, (int)((ev >> 10) & 3u), d, d);
            } else {
              ++n_all;
              if (!blocked && d <= A.lat[P.opclass[x]] && keeps_any(P, A, j, P.opclass[x])) ++n_kept;
              if (P.diag == 2) xemit(P, j, x, r, d, 0, d, blocked);
            }
          }
          S = add_literal(S, (int)((ev >> 12) & 0xFu));
          if (contains(S, gj)) { covered = true; break; }
        } else if (pos != last_def_pos && !blocked) {
          // An unguarded reader on every path beyond this point: nothing
          // further survives rule 2 (the coverage count still counts it).
          blocked = true;
          if (!P.diag) break;
        }
      }
      if (P.diag && covered) { cov_add(P, e, n_all, n_kept); continue; }
      if (covered || (blocked && !P.diag)) continue;
      // Predecessors through which a def of r reaches b0 (distinct blocks).
      // If each covers j's guard inside itself, resolve here; otherwise queue
      // the general search.
      const int w = r >> 5;
      const uint32_t bit = 1u << (r & 31);
      const int q0 = P.pred_off[b0], q1 = P.pred_off[b0 + 1];
      auto counts = [&](int q) {
        const int p = P.pred[q];
        if (!(P.rout[(size_t)p * kWords + w] & bit)) return false;
        for (int q2 = q0; q2 < q; ++q2) if (P.pred[q2] == p) return false;
        return true;
      };
      bool any = false, all_cover = true;
      for (int q = q0; q < q1 && all_cover; ++q) {
        if (!counts(q)) continue;
        any = true;
        all_cover = scan_pred(P, A, j, r, gj, b0, P.pred[q], S, pj + 1, false);
      }
      if (!any) {
        if (P.diag) cov_add(P, e, n_all, n_kept);
        continue;
      }
      if (all_cover) {
        for (int q = q0; q < q1; ++q)
          if (counts(q))
            scan_pred(P, A, j, r, gj, b0, P.pred[q], S, pj + 1, !P.diag, P.diag ? &n_all : nullptr, &n_kept, blocked);
        if (P.diag) cov_add(P, e, n_all, n_kept);
        continue;
      }
      if (P.diag) cov_add(P, e, n_all, n_kept);  // the in-block part; the search adds the rest
      // A search known to outgrow the first tier goes straight to the queue
      // that held it before (see Prog::queue).
      const uint32_t hint = P.tier_hint[P.diag ? 1 : 0][e];
      P.tasks[e] = make_int2(j, r | ((int)S << 9) | (blocked ? 1 << 25 : 0));
      int slot = SS_QUEUE_N, q = 0;
      bool top = false, placed = false;
      unsigned long long t = 0;
      if (hint >= kHintCta && P.t4_nodes > 0) {
        const bool giant = hint >= kHintGiant;
        slot = giant ? SS_T5_N : SS_T4_N;
        q = giant ? 7 : 4;
        atomicAdd(&P.stats[SS_DIRECT_N], 1ull);
      } else if (hint >= kHintWide) { slot = SS_WIDE_N; q = 6; }
      else if (hint >= kHintA1) {
        const int c = (int)hint - kHintA1;
        slot = SS_A1_N + c;
        q = class_queue(c);
        top = class_top(c);
        t = atomicAdd(&P.stats[slot], 1ull);
        placed = t < (unsigned long long)P.class_limit[c];
        if (!placed) { slot = SS_HINT3_N; q = 3; top = true; }  // the warps
      } else if (hint == kHintLane2) { slot = SS_OVF_N; q = 1; }
      if (!placed) t = atomicAdd(&P.stats[slot], 1ull);
      if (t < (unsigned long long)P.queue_cap) P.queue[q][top ? P.queue_cap - 1 - (int64_t)t : (int64_t)t] = e;
      else capacity(P, 8);
    }
  }
}

// ---------------------------------------------------------------- merge and apportion
// (The lanes of a warp hold neighbouring uses, whose sources are mostly
// different instructions: partitioning them by address first cost more than the
// few atomics it saved.)
__device__ __forceinline__ void blame_add(unsigned long long* addr, unsigned long long v) { atomicAdd(addr, v); }

// Distinct sources of use j over its raw edge list, using ids[cap] as scratch:
// the count, or -1 if there are more than cap.
__device__ int distinct_sources(const Prog& P, int j, int* ids, int cap) {
  int c = 0;
  for (int t = P.head[j]; t >= 0; t = P.raw[t].y) {
    const int i = P.raw[t].x;
    bool seen = false;
    for (int q = 0; q < c; ++q) seen |= ids[q] == i;
    if (seen) continue;
    if (c >= cap) return -1;
    ids[c++] = i;
  }
  return c;
}

// Uses with more distinct sources than a thread's arrays hold are listed for
// k_merge_big / k_apportion_big (shared-memory arrays, one CTA per use).
__global__ void k_merge_count(Prog P, int max_src) {
  for (int j = blockIdx.x * blockDim.x + threadIdx.x; j < P.ni; j += gridDim.x * blockDim.x) {
    int ids[kMaxSrc];
    int c = distinct_sources(P, j, ids, min(max_src, kMaxSrc));
    if (c < 0 && max_src > kMaxSrc) {
      const unsigned long long k = atomicAdd(&P.stats[SS_BIG_N], 1ull);
      P.big_use[k] = j;  // k < ni: each use is listed at most once
      c = 0;             // k_merge_big writes the count
    } else if (c < 0) {
      capacity(P, 9);
      c = 0;
    }
    P.edge_off[j] = c;
  }
}

__global__ void k_merge_big(Prog P, int max_src) {
  __shared__ int ids[kBigSrc];
  const unsigned long long nbig = P.stats[SS_BIG_N];
  for (unsigned long long k = blockIdx.x; k < nbig; k += gridDim.x) {
    if (threadIdx.x == 0) {
      const int j = P.big_use[k];
      int c = distinct_sources(P, j, ids, min(max_src, kBigSrc));
      if (c < 0) { capacity(P, 9); c = 0; }
      P.edge_off[j] = c;
    }
    __syncthreads();
  }
}

// Merged edges of use j (ascending def index) and Eq. 1 shares of each of its
// dependency classes and latency flags, with arrays of capacity cap.
__device__ void apportion_use(const Prog& P, const Arch& A, int j, int off, int c, int* mi, int* md, int* ml,
                              uint32_t* mf, uint32_t* mo, unsigned long long* mc, int* sel,
                              unsigned long long* wt, unsigned __int128* rem, unsigned long long* sh) {
  // the eight dependency counters of j, and of each source its opcode's flags
  // and issue count: loaded once, the sources' while the list is walked
  static_assert(2 * GPA_EXEC_DEPENDENCY == 4 && 2 * GPA_MEMORY_DEPENDENCY == 6 && 2 * GPA_SYNC == 10 &&
                    2 * GPA_CONSTANT_MEMORY_DEPENDENCY == 12,
                "dependency-class words 4-7 and 10-13");
  const ulonglong2* cj2 = reinterpret_cast<const ulonglong2*>(P.cnt + (size_t)j * kCnt);
  const ulonglong2 cj[4] = {cj2[2], cj2[3], cj2[5], cj2[6]};
  int m = 0;
  if (c > 0) {
    for (int t = P.head[j]; t >= 0; t = P.raw[t].y) {
      const int4 R = P.raw[t];
      const int dl = R.w & 0xFFFFFF;
      const uint32_t fl = (uint32_t)R.w >> 24;
      int q = 0;
      while (q < m && mi[q] != R.x) ++q;
      if (q == m) {
        if (m >= c) continue;  // capacity already reported by the count pass
        mi[m] = R.x; md[m] = R.z; ml[m] = dl; mf[m] = fl;
        mo[m] = A.flags[P.opclass[R.x]];
        mc[m] = P.cnt[(size_t)R.x * kCnt];
        ++m;
      } else {
        md[q] = min(md[q], R.z); ml[q] = max(ml[q], dl); mf[q] |= fl;
      }
    }
    // ascending def index
    for (int a = 1; a < m; ++a) {
      const int xi = mi[a], xd = md[a], xl = ml[a];
      const uint32_t xf = mf[a], xo = mo[a];
      const unsigned long long xc = mc[a];
      int b = a - 1;
      while (b >= 0 && mi[b] > xi) {
        mi[b + 1] = mi[b]; md[b + 1] = md[b]; ml[b + 1] = ml[b]; mf[b + 1] = mf[b]; mo[b + 1] = mo[b]; mc[b + 1] = mc[b];
        --b;
      }
      mi[b + 1] = xi; md[b + 1] = xd; ml[b + 1] = xl; mf[b + 1] = xf; mo[b + 1] = xo; mc[b + 1] = xc;
    }
    for (int t = 0; t < m; ++t) {
      const int64_t e = off + t;
      P.e_use[e] = j; P.e_def[e] = mi[t]; P.e_dmin[e] = md[t]; P.e_dlong[e] = ml[t]; P.e_flags[e] = mf[t];
#pragma unroll
      for (int q = 0; q < 8; ++q) P.e_share[e * 8 + q] = 0ull;
    }
  }
  for (int ci = 0; ci < 4; ++ci) {
    const int cls = dep_class(ci);
    // rule 1 (opcode_keeps): the flag a source of this class carries
    const uint32_t keeps = ci == 1 || ci == 3 ? (uint32_t)GPA_F_MEM : ci == 2 ? (uint32_t)GPA_F_SYNC : 0u;
    for (int lat = 0; lat < 2; ++lat) {
      const unsigned long long S = lat ? cj[ci].y : cj[ci].x;
      if (!S) continue;
      int ns = 0;
      for (int t = 0; t < m; ++t)
        if (!keeps || (mo[t] & keeps)) sel[ns++] = t;
      if (ns == 0) {  // no surviving source: the samples stay on j
        blame_add(P.blame + (size_t)j * kCnt + cls * 2 + lat, S);
        continue;
      }
      if (ns == 1) {  // a single source takes them all, whatever its weight
        const int t = sel[0];
        if (mc[t] >> 43) set_status(P, ST_OVERFLOW);
        P.e_share[(int64_t)(off + t) * 8 + ci * 2 + lat] = S;
        blame_add(P.blame + (size_t)mi[t] * kCnt + cls * 2 + lat, S);
        continue;
      }
      // Eq. 1: weight = issued samples / longest path, in units of 2^-20.
      unsigned __int128 W = 0;
      for (int q = 0; q < ns; ++q) {
        const unsigned long long issue = mc[sel[q]];
        const unsigned long long len = (unsigned long long)max(ml[sel[q]], 1);
        if (issue >> 43) set_status(P, ST_OVERFLOW);
        // (len < 2^24, so a 64-bit division does for issue counts below 2^44)
        wt[q] = issue >> 44 ? (unsigned long long)(((unsigned __int128)issue << 20) / len) : (issue << 20) / len;
        W += wt[q];
      }
      if (W == 0) {
        for (int q = 0; q < ns; ++q) {
          wt[q] = (1ull << 20) / (unsigned long long)max(ml[sel[q]], 1);
          W += wt[q];
        }
      }
      if (W == 0) {
        for (int q = 0; q < ns; ++q) wt[q] = 1ull;
        W = (unsigned __int128)ns;
      }
      // S * wt and W mostly fit 64 bits, whose division is a tenth of the work.
      unsigned long long given = 0;
      const bool narrow = !(W >> 64);
      for (int q = 0; q < ns; ++q) {
        const unsigned __int128 num = (unsigned __int128)S * wt[q];
        if (narrow && !(num >> 64)) {
          const unsigned long long a = (unsigned long long)num, b = (unsigned long long)W;
          sh[q] = a / b;
          rem[q] = a - sh[q] * b;
        } else {
          sh[q] = (unsigned long long)(num / W);
          rem[q] = num % W;
        }
        given += sh[q];
      }
      // Largest remainders get the leftover units; ties go to the lower def index.
      unsigned long long left = S - given;
      while (left > 0) {
        int best = -1;
        for (int q = 0; q < ns; ++q) {
          if (rem[q] == (unsigned __int128)-1) continue;
          if (best < 0 || rem[q] > rem[best]) best = q;  // sel is in ascending def order
        }
        if (best < 0) break;  // cannot happen: fewer leftover units than sources
        sh[best] += 1;
        rem[best] = (unsigned __int128)-1;
        --left;
      }
      for (int q = 0; q < ns; ++q) {
        const int t = sel[q];
        P.e_share[(int64_t)(off + t) * 8 + ci * 2 + lat] = sh[q];
        if (sh[q]) blame_add(P.blame + (size_t)mi[t] * kCnt + cls * 2 + lat, sh[q]);
      }
    }
  }
}

// Thread per stalled use (a use with edges is stalled: searches run for
// stalled uses only).
__global__ void k_apportion(Prog P, Arch A, int max_src) {
  const int n_suse = (int)P.stats[SS_SUSE_N];
  for (int k = blockIdx.x * blockDim.x + threadIdx.x; k < n_suse; k += gridDim.x * blockDim.x) {
    const int j = P.suse[k];
    const int off = P.edge_off[j];
    int c = P.edge_off[j + 1] - off;
    if (c > kMaxSrc) continue;  // k_apportion_big
    if (off + c > P.edge_cap) { capacity(P, 10); c = 0; }
    int mi[kMaxSrc], md[kMaxSrc], ml[kMaxSrc], sel[kMaxSrc];
    uint32_t mf[kMaxSrc], mo[kMaxSrc];
    unsigned long long mc[kMaxSrc], wt[kMaxSrc], sh[kMaxSrc];
    unsigned __int128 rem[kMaxSrc];
    apportion_use(P, A, j, off, c, mi, md, ml, mf, mo, mc, sel, wt, rem, sh);
  }
}

__global__ void k_apportion_big(Prog P, Arch A) {
  extern __shared__ __align__(16) unsigned char big_sm[];
  unsigned __int128* rem = reinterpret_cast<unsigned __int128*>(big_sm);
  unsigned long long* wt = reinterpret_cast<unsigned long long*>(rem + kBigSrc);
  unsigned long long* sh = wt + kBigSrc;
  int* mi = reinterpret_cast<int*>(sh + kBigSrc);
  int* md = mi + kBigSrc;
  int* ml = md + kBigSrc;
  int* sel = ml + kBigSrc;
  uint32_t* mf = reinterpret_cast<uint32_t*>(sel + kBigSrc);
  uint32_t* mo = mf + kBigSrc;
  unsigned long long* mc = reinterpret_cast<unsigned long long*>(mo + kBigSrc);
  const unsigned long long nbig = P.stats[SS_BIG_N];
  for (unsigned long long k = blockIdx.x; k < nbig; k += gridDim.x) {
    if (threadIdx.x == 0) {
      const int j = P.big_use[k];
      const int off = P.edge_off[j];
      int c = P.edge_off[j + 1] - off;
      if (off + c > P.edge_cap) { capacity(P, 10); c = 0; }
      if (c > kMaxSrc) apportion_use(P, A, j, off, c, mi, md, ml, mf, mo, mc, sel, wt, rem, sh);
    }
    __syncthreads();
  }
}

// Single dependency coverage: a stalled use is a single dependency node when
// no resource it reads has more than one source (before pruning) or more than
// one kept source (after).
__global__ void k_coverage(Prog P) {
  unsigned long long nodes = 0, before = 0, after = 0;
  for (int j = blockIdx.x * blockDim.x + threadIdx.x; j < P.ni; j += gridDim.x * blockDim.x) {
    if (!stalled(P, j)) continue;
    uint32_t most_all = 0, most_kept = 0;
    for (int e = P.use_off[j]; e < P.use_off[j + 1]; ++e) {
      const uint32_t c = P.cov_cnt[e];
      most_all = max(most_all, c & 0xFFFFu);
      most_kept = max(most_kept, c >> 16);
    }
    ++nodes;
    before += most_all <= 1u;
    after += most_kept <= 1u;
  }
  for (int o = 16; o > 0; o >>= 1) {
    nodes += __shfl_xor_sync(0xffffffffu, nodes, o);
    before += __shfl_xor_sync(0xffffffffu, before, o);
    after += __shfl_xor_sync(0xffffffffu, after, o);
  }
  if ((threadIdx.x & 31) == 0 && nodes) {
    atomicAdd(&P.stats[SS_COV], nodes);
    atomicAdd(&P.stats[SS_COV + 1], before);
    atomicAdd(&P.stats[SS_COV + 2], after);
  }
}

// Ordering the export by (use, resource, def): edges counted per use, scanned,
// dropped into their use's bucket, and each edge's rank within its bucket taken
// by comparing it with the others there (a use has a handful). Buckets of more than
// kExportRank edges (guarded defs can give a use tens of thousands) are listed and
// merge-sorted instead, a CTA each: comparing is quadratic (60 uses of 32,001 sources:
// the export and its copy out 203 ms by comparing, 53 ms sorted; 2,050 sources 2.0 and
// 1.8 ms, 1,025 the same).
__global__ void k_export_count(const int4* x, int64_t n, int32_t* cnt) {
  for (int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; k < n; k += (int64_t)gridDim.x * blockDim.x)
    atomicAdd(&cnt[x[2 * k].x], 1);
}
__global__ void k_export_bucket(const int4* x, int64_t n, const int32_t* off, int32_t* cursor, int32_t* ids,
                                int32_t* big) {
  for (int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; k < n; k += (int64_t)gridDim.x * blockDim.x) {
    const int j = x[2 * k].x;
    const int at = atomicAdd(&cursor[j], 1);
    ids[off[j] + at] = (int32_t)k;
    if (at == 0 && off[j + 1] - off[j] > kExportRank) big[1 + atomicAdd(&big[0], 1)] = j;
  }
}
__global__ void k_export_order(const int4* x, int64_t n, const int32_t* off, const int32_t* ids, ExportOut out) {
  for (int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; k < n; k += (int64_t)gridDim.x * blockDim.x) {
    const int4 a = x[2 * k], b = x[2 * k + 1];
    const int q0 = off[a.x], q1 = off[a.x + 1];
    if (q1 - q0 > kExportRank) continue;  // k_export_sort
    int at = q0;
    for (int q = q0; q < q1; ++q) {
      const int4 c = x[2 * (int64_t)ids[q]];
      at += c.z < a.z || (c.z == a.z && c.y < a.y) ? 1 : 0;
    }
    out.use[at] = a.x; out.def[at] = a.y; out.res[at] = a.z; out.dmin[at] = a.w;
    out.back[at] = b.x; out.dlong[at] = b.y; out.dom[at] = (uint8_t)b.z;
  }
}
// The listed buckets: runs of 1, 2, 4, ... merged pairwise, each element placed by a
// binary search in the run beside its own (an earlier run's elements come first among
// equals). The use column serves as the other buffer until it is written.
__global__ void __launch_bounds__(1024) k_export_sort(const int4* x, const int32_t* off, int32_t* ids,
                                                      const int32_t* big, ExportOut out) {
  for (int t = blockIdx.x; t < big[0]; t += gridDim.x) {
    const int j = big[1 + t], q0 = off[j], m = off[j + 1] - q0;
    int32_t *a = ids + q0, *b = out.use + q0;
    for (int64_t w = 1; w < m; w *= 2) {
      for (int i = threadIdx.x; i < m; i += blockDim.x) {
        const int id = a[i];
        const int4 v = x[2 * (int64_t)id];
        const bool right = (i / w) & 1;
        const int64_t base = i / w * w, other = right ? base - w : base + w;
        int64_t lo = min(other, (int64_t)m), hi = min(other + w, (int64_t)m);
        const int64_t first = lo;
        while (lo < hi) {
          const int64_t mid = (lo + hi) / 2;
          const int4 c = x[2 * (int64_t)a[mid]];
          const bool before = c.z != v.z ? c.z < v.z : c.y < v.y || (right && c.y == v.y);
          if (before) lo = mid + 1;
          else hi = mid;
        }
        b[min(base, other) + (i - base) + (lo - first)] = id;
      }
      __syncthreads();
      int32_t* sw = a; a = b; b = sw;
    }
    for (int i = threadIdx.x; i < m; i += blockDim.x) {
      const int64_t id = a[i];
      const int4 v = x[2 * id], u = x[2 * id + 1];
      const int at = q0 + i;
      out.use[at] = v.x; out.def[at] = v.y; out.res[at] = v.z; out.dmin[at] = v.w;
      out.back[at] = u.x; out.dlong[at] = u.y; out.dom[at] = (uint8_t)u.z;
    }
    __syncthreads();
  }
}

}  // namespace

// n <= INT32_MAX; off and cursor have ni + 1 and ni entries, ids n, big export_big_ints(n).
void launch_order_export(const int4* x, int64_t n, int ni, int32_t* off, int32_t* cursor, int32_t* ids, int32_t* big,
                         const ExportOut& out, int32_t* scan_tmp, cudaStream_t st, int sms, int64_t* launches) {
  if (n <= 0) return;
  cudaMemsetAsync(off, 0, sizeof(int32_t) * (size_t)(ni + 1), st);
  cudaMemsetAsync(cursor, 0, sizeof(int32_t) * (size_t)ni, st);
  cudaMemsetAsync(big, 0, sizeof(int32_t), st);
  const int g = grid_for(n, 256, sms);
  k_export_count<<<g, 256, 0, st>>>(x, n, off);
  scan_exclusive_inplace(off, ni, scan_tmp, st, launches);
  k_export_bucket<<<g, 256, 0, st>>>(x, n, off, cursor, ids, big);
  k_export_order<<<g, 256, 0, st>>>(x, n, off, ids, out);
  *launches += 3;
  if (n > kExportRank) {
    k_export_sort<<<sms, 1024, 0, st>>>(x, off, ids, big, out);
    ++*launches;
  }
}

void launch_coverage(const Prog& P, const Arch& A, const SearchArena* tiers, const SearchFork* fork, cudaStream_t st,
                     int sms, int64_t* launches) {
  const int threads = 128;
  const int g_local = std::max(1, std::min(sms * 64, (int)(((int64_t)P.ni * kLocalLanes + threads - 1) / threads)));
  k_stalled_list<<<(P.ni + 255) / 256, 256, 0, st>>>(P, 0);
  k_search_local<<<g_local, threads, 0, st>>>(P, A);
  *launches += 2;
  launch_search(P, A, tiers, fork, st, sms, launches);
  if (P.diag != 1) return;
  k_coverage<<<grid_for(P.ni, threads, sms), threads, 0, st>>>(P);
  ++*launches;
}

void launch_blame(const Prog& P, const Arch& A, const SearchArena* tiers, const SearchFork* fork, int max_src,
                  int32_t* scan_tmp, cudaStream_t st, int sms, int64_t* launches) {
  const int threads = 128;
  const int g_instr = grid_for(P.ni, threads, sms);
  // The per-use kernels take the stalled-use list (its length is known on the
  // device only): enough CTAs for every SM to hold as many warps as their
  // registers allow, each thread taking about one use on the batched workload.
  const int g_use = std::max(1, std::min(grid_for(P.ni, threads, sms) * 4, (P.ni + threads - 1) / threads));
  const int g_local = std::max(1, std::min(sms * 64, (int)(((int64_t)P.ni * kLocalLanes + threads - 1) / threads)));
  k_stalled_list<<<(P.ni + 255) / 256, 256, 0, st>>>(P, 1);
  k_search_local<<<g_local, threads, 0, st>>>(P, A);
  *launches += 2;
  launch_search(P, A, tiers, fork, st, sms, launches);
  k_merge_count<<<g_instr, threads, 0, st>>>(P, max_src);
  k_merge_big<<<sms, 32, 0, st>>>(P, max_src);
  *launches += 2;
  scan_exclusive_inplace(P.edge_off, P.ni, scan_tmp, st, launches);
  k_apportion<<<g_use, threads, 0, st>>>(P, A, max_src);
  const size_t big_smem = (size_t)kBigSrc * (16 + 8 + 8 + 4 * 6 + 8);
  allow_max_smem(k_apportion_big);
  k_apportion_big<<<sms, 32, big_smem, st>>>(P, A);
  *launches += 2;
}

}  // namespace gpa
