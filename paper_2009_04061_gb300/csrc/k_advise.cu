// Step (d), Sec. 5: roll blame up to lines, loops and functions, match the
// code optimizers of Table 2 (Function Inlining from the program's call
// table), estimate their speedups (Eq. 2 for stall elimination, Eq. 4 for
// latency hiding, Eq. 5 per loop scope), rank them and
// pick each optimizer's top five hotspots (def, use, distance); with launch
// statistics, the parallel optimizers (Eqs. 6-10).
//
// One CTA per tile of 1,024 (or 256) instructions of one function, so that a large
// function is spread over the chip (one CTA a function left a 20,000-instruction
// function 880 us behind the others and a 120,000-instruction one 4.3 ms). A tile
// reads its instructions' counters and blame and its edges (contiguous, since
// edges are ordered by use) once: sums, loop and line roll-ups, and all nine
// optimizers' top five together, each kept by a warp in its first five lanes
// (candidates that beat the fifth are inserted best first, by a ballot and a shift). The
// function's last tile to finish merges the tiles' lists and writes its results.
// What bounds it is the counters' and blame's 384 bytes an instruction.
#include "gpa_internal.cuh"

namespace gpa {

namespace {

constexpr int kThreads = 128;
constexpr int kWarpsA = kThreads / 32;
constexpr int kHot = 5;
enum { O_RR = 0, O_SR, O_FS, O_FM, O_WB, O_MT, O_LU, O_CR, O_FI, N_O = 9 };
constexpr int kAcc = kAdvAcc - 1;  // per-function sums, see k_advise; then the tiles that are done

struct Cand { unsigned long long v; int def, use, dist; };

__device__ __forceinline__ bool better(const Cand& a, const Cand& b) {  // a ranks before b
  if (a.v != b.v) return a.v > b.v;
  if (a.def != b.def) return a.def < b.def;
  return a.use < b.use;
}
__device__ __forceinline__ Cand shfl_cand(const Cand& c, int src) {
  return Cand{__shfl_sync(0xffffffffu, c.v, src), __shfl_sync(0xffffffffu, c.def, src),
              __shfl_sync(0xffffffffu, c.use, src), __shfl_sync(0xffffffffu, c.dist, src)};
}
// A warp's top five, best first, in lanes 0-4 (v == 0: none): takes in every
// lane's candidate (v == 0: none), best first, until one does not make the five
// (in lane order a warp full of candidates cost 32 insertions). Candidates are
// distinct, so the order is total.
__device__ __forceinline__ void top_insert(Cand& top, const Cand& c) {
  const int lane = threadIdx.x & 31;
  const Cand fifth = shfl_cand(top, kHot - 1);
  unsigned m = __ballot_sync(0xffffffffu, c.v != 0ull && better(c, fifth));
  while (m) {
    // the best of the lanes in m: largest v, then smallest def, then smallest use
    unsigned best = m;
    const uint32_t hi = (uint32_t)(c.v >> 32), lo = (uint32_t)c.v;
    const uint32_t mh = __reduce_max_sync(0xffffffffu, (m >> lane) & 1u ? hi : 0u);
    best &= __ballot_sync(0xffffffffu, hi == mh);
    const uint32_t ml = __reduce_max_sync(0xffffffffu, (best >> lane) & 1u ? lo : 0u);
    best &= __ballot_sync(0xffffffffu, lo == ml);
    if (best & (best - 1)) {
      const int md = __reduce_min_sync(0xffffffffu, (best >> lane) & 1u ? c.def : 0x7FFFFFFF);
      best &= __ballot_sync(0xffffffffu, c.def == md);
      const int mu = __reduce_min_sync(0xffffffffu, (best >> lane) & 1u ? c.use : 0x7FFFFFFF);
      best &= __ballot_sync(0xffffffffu, c.use == mu);
    }
    const int src = __ffs(best) - 1;
    m &= ~(1u << src);
    const Cand x = shfl_cand(c, src);
    const int rank = __popc(__ballot_sync(0xffffffffu, lane < kHot && better(top, x)));
    if (rank == kHot) break;  // the others rank below it
    const Cand up{__shfl_up_sync(0xffffffffu, top.v, 1), __shfl_up_sync(0xffffffffu, top.def, 1),
                  __shfl_up_sync(0xffffffffu, top.use, 1), __shfl_up_sync(0xffffffffu, top.dist, 1)};
    if (lane > rank) top = up;  // (lanes past the fifth hold what fell out; they never rank)
    if (lane == rank) top = x;
  }
}
// Adds v to dst[l] for every lane with l >= 0, one atomic per distinct l of the
// warp (neighbouring instructions mostly share their loop).
__device__ __forceinline__ void add_by_loop(unsigned long long* dst, int l, unsigned long long v) {
  unsigned m = __ballot_sync(0xffffffffu, l >= 0 && v != 0ull);
  while (m) {
    const int L = __shfl_sync(0xffffffffu, l, __ffs(m) - 1);
    const bool mine = l == L;
    unsigned long long s = mine ? v : 0ull;
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if ((threadIdx.x & 31) == 0) atomicAdd(&dst[L], s);
    m &= ~__ballot_sync(0xffffffffu, mine);
  }
}

__device__ __forceinline__ double est(unsigned long long T, unsigned long long M) {
  if (T == 0) return 1.0;
  if (T == M) return __longlong_as_double(0x7FF0000000000000LL);  // +inf
  return (double)T / (double)(T - M);
}

__device__ int innermost_loop(const Prog& P, int x) { return P.block_loop[P.instr_block[x]]; }

__device__ int lca_loop(const Prog& P, int a, int b) {
  if (a < 0 || b < 0) return -1;
  int da = P.loop_depth[a], db = P.loop_depth[b];
  while (da > db) { a = P.loop_parent[a]; --da; }
  while (db > da) { b = P.loop_parent[b]; --db; }
  while (a != b && a >= 0 && b >= 0) { a = P.loop_parent[a]; b = P.loop_parent[b]; }
  return (a == b) ? a : -1;
}

// Matched samples of an edge per edge-based optimizer. Shares are indexed
// class slot (exec, memory, sync, constant memory) * 2 + latency flag. The
// def and use's innermost common loop goes to `lca`.
struct EdgeMatch { unsigned long long rr, sr, lu, cr; };
__device__ __forceinline__ EdgeMatch edge_match(const Prog& P, const Arch& A, int64_t e, int def, int use, int* lca) {
  const ulonglong2* sh = reinterpret_cast<const ulonglong2*>(P.e_share + e * 8);
  const ulonglong2 s0 = sh[0], s1 = sh[1], s3 = sh[3];
  const uint32_t fl = A.flags[P.opclass[def]];
  const bool local = fl & GPA_F_LOCAL;
  const bool global_mem = !local && !(fl & GPA_F_CONST);  // constant-memory stalls are never global
  EdgeMatch m;
  m.rr = local ? (s1.x + s1.y + s3.x + s3.y) : 0ull;           // Register Reuse
  m.sr = (fl & GPA_F_LONG_ARITH) ? (s0.x + s0.y) : 0ull;      // Strength Reduction
  m.cr = s0.y + (global_mem ? s1.y : 0ull);                   // latency samples
  *lca = m.cr ? lca_loop(P, innermost_loop(P, def), innermost_loop(P, use)) : -1;
  m.lu = *lca >= 0 ? m.cr : 0ull;
  return m;
}

// Parallel optimizers of function f (Table 2; Sec. 5.2, Eqs. 6-10 with f = 1),
// from its launch statistics, the SM model and its totals (T samples, issued).
// Occupancy: blocks per SM is the least of the warp, register, shared-memory
// and block-count limits (the binding one is reported, lowest id on ties).
// W = resident blocks per SM * warps per block / schedulers; R_I = issued / T;
// I(W) = 1 - (1 - R_I)^W (Eqs. 8-9).
//  Block Increase (fewer blocks than SMs): the same threads in one block per
//  SM, W_new = W * blocks / SMs; every SM runs one wave, so a scheduler's
//  warps over the run are its resident warps: C_W = W_new / W (Eq. 6).
//  Thread Increase (the block-count limit binds, and the grid reaches it): the
//  same threads in larger blocks, W_new = the warps per SM the warp, register
//  and shared-memory limits (per warp) and the grid allow, / schedulers; a
//  scheduler's warps over the run are unchanged: C_W = 1.
//  S = (1 / C_W) * C_I (Eq. 10), C_I = I(W_new) / I(W) (Eq. 7).
__device__ void parallel_advice(const Prog& P, int f, unsigned long long T, unsigned long long issued) {
  int match[2] = {0, 0}, limit = -1;
  double sp[2] = {1.0, 1.0}, w[4] = {0.0, 0.0, 0.0, 0.0};
  if (P.launch) {
    const LaunchRec L = P.launch[f];
    const SmModel& M = P.sm;
    const long long big = 1ll << 40;
    const long long wpb = (L.threads + 31) / 32;
    long long lim[4];
    lim[0] = M.max_warps / wpb;
    long long warps_by_regs = M.max_warps;  // warps per SM the registers allow
    if (L.regs > 0) {
      const long long rpw = ((long long)L.regs * 32 + M.reg_unit - 1) / M.reg_unit * M.reg_unit;
      warps_by_regs = (long long)M.schedulers * ((M.regs / M.schedulers) / rpw);
      lim[1] = warps_by_regs / wpb;
    } else {
      lim[1] = big;
    }
    long long warps_by_smem = big;          // warps per SM the shared memory allows
    if (L.smem > 0) {
      const long long per = ((long long)L.smem + M.smem_reserved + M.smem_unit - 1) / M.smem_unit * M.smem_unit;
      lim[2] = M.smem / per;
      warps_by_smem = lim[2] * wpb;
    } else {
      lim[2] = big;
    }
    lim[3] = M.max_blocks;
    long long bps = lim[0];
    limit = 0;
    for (int q = 1; q < 4; ++q)
      if (lim[q] < bps) { bps = lim[q]; limit = q; }
    const long long per_sm = (L.blocks + M.n_sms - 1) / M.n_sms;  // blocks per SM the grid gives
    const long long rb = bps < per_sm ? bps : per_sm;
    const double W = (double)(rb * wpb) / (double)M.schedulers;
    match[0] = L.blocks < M.n_sms;
    match[1] = limit == 3 && per_sm >= bps;
    double Wn[2] = {0.0, 0.0};
    Wn[0] = W * (double)L.blocks / (double)M.n_sms;
    long long wn = M.max_warps;
    if (warps_by_regs < wn) wn = warps_by_regs;
    if (warps_by_smem < wn) wn = warps_by_smem;
    const long long grid_warps = (L.blocks * wpb + M.n_sms - 1) / M.n_sms;
    if (grid_warps < wn) wn = grid_warps;
    Wn[1] = (double)wn / (double)M.schedulers;
    // an estimate needs a resident warp and an issue rate above zero
    const bool est_ok = bps > 0 && T > 0 && issued > 0;
    const double R = T ? (double)issued / (double)T : 0.0;
    const double I = 1.0 - pow(1.0 - R, W);
    for (int k = 0; k < 2; ++k) {
      if (!match[k]) continue;
      w[2 * k] = W;
      w[2 * k + 1] = Wn[k];
      if (!est_ok) continue;
      const double cw = k == 0 ? Wn[0] / W : 1.0, ci = (1.0 - pow(1.0 - R, Wn[k])) / I;
      sp[k] = (1.0 / cw) * ci;
    }
  }
  for (int k = 0; k < 2; ++k) {
    P.a_par_match[(size_t)f * 2 + k] = match[k];
    P.a_par_speedup[(size_t)f * 2 + k] = sp[k];
  }
  for (int k = 0; k < 4; ++k) P.a_par_warps[(size_t)f * 4 + k] = w[k];
  P.a_par_limit[f] = limit;
}

__global__ void __launch_bounds__(kThreads) k_advise(Prog P, Arch A) {
  __shared__ unsigned long long red[kAcc][kWarpsA];
  __shared__ unsigned long long tot[kAcc];
  __shared__ Cand wtop[N_O][kWarpsA][kHot];  // each warp's top five (v == 0: none)
  __shared__ bool s_last;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int f = P.adv_tile_func[blockIdx.x];
  const int t0 = P.adv_tile_off[f], nt = P.adv_tile_off[f + 1] - t0;
  const int i0 = P.func_instr_off[f];
  const int x0 = i0 + ((int)blockIdx.x - t0) * P.adv_tile, x1 = min(P.func_instr_off[f + 1], x0 + P.adv_tile);
  // Edge ranges are clamped to the edge capacity (overflow is reported in the status word).
  const int64_t e0 = min((int64_t)P.edge_off[x0], P.edge_cap), e1 = min((int64_t)P.edge_off[x1], P.edge_cap);
  unsigned long long acc[kAcc];
#pragma unroll
  for (int q = 0; q < kAcc; ++q) acc[q] = 0ull;
  Cand top[N_O];
#pragma unroll
  for (int o = 0; o < N_O; ++o) top[o] = Cand{0ull, 0, 0, 0};
  // acc: 0 T, 1 A, 2 L, 3 issued, 4 FS, 5 FM, 6 WB, 7 MT, 8 RR, 9 SR, 10 LU, 11 CR, 12 FI
  for (int xb = x0 + warp * 32; xb < x1; xb += kThreads) {
    const int x = xb + lane;
    const bool in = x < x1;
    unsigned long long a = 0, l = 0, stall = 0, fs = 0, wb = 0, mt = 0, bs = 0, bl = 0, c0 = 0, c1 = 0;
    int loop = -1;
    uint32_t ifl = 0, fl = 0;
    if (in) {
      const ulonglong2* c = reinterpret_cast<const ulonglong2*>(P.cnt + (size_t)x * kCnt);
      const ulonglong2* b = reinterpret_cast<const ulonglong2*>(P.blame + (size_t)x * kCnt);
      ifl = P.iflags[x];
      fl = A.flags[P.opclass[x]];
      loop = innermost_loop(P, x);
#pragma unroll
      for (int k = 0; k < kCnt / 2; ++k) {
        const ulonglong2 v = c[k];
        a += v.x;
        l += v.y;
        if (k == 0) c0 = v.x, c1 = v.y;
        else stall += v.x + v.y;
        if (k == 1) fs = v.x + v.y;
        if (k == 5) wb = v.x + v.y;
        if (k == 8) mt = v.x + v.y;
      }
#pragma unroll
      for (int k = 1; k < kCnt / 2; ++k) {
        const ulonglong2 v = b[k];
        bs += v.x + v.y;
        bl += v.y;
      }
      acc[0] += a + l; acc[1] += a; acc[2] += l; acc[3] += c0;
      if (bs) atomicAdd(&P.a_line_stall[P.line[x]], bs);
      if (bl) atomicAdd(&P.a_line_lat[P.line[x]], bl);
    }
    const unsigned long long fm = (ifl & 1) ? stall : 0ull;
    const unsigned long long fi = (ifl & 6) ? l : 0ull;  // latency stalls in a device function or at a call site
    if (!(fl & GPA_F_GLOBAL)) mt = 0ull;
    acc[4] += fs; acc[5] += fm; acc[6] += wb; acc[7] += mt; acc[12] += fi;
    add_by_loop(P.adv_own_active, loop, a);
    const int pc = x - i0;
    top_insert(top[O_FS], Cand{fs, pc, pc, 0});
    top_insert(top[O_FM], Cand{fm, pc, pc, 0});
    top_insert(top[O_WB], Cand{wb, pc, pc, 0});
    top_insert(top[O_MT], Cand{mt, pc, pc, 0});
    top_insert(top[O_FI], Cand{fi ? fi - c1 : 0ull, pc, pc, 0});  // a hotspot counts no SELECTED samples
  }
  for (int64_t eb = e0 + warp * 32; eb < e1; eb += kThreads) {
    const int64_t e = eb + lane;
    EdgeMatch m{0ull, 0ull, 0ull, 0ull};
    int q = -1, def = 0, use = 0, dist = 0;
    if (e < e1) {
      def = P.e_def[e];
      use = P.e_use[e];
      dist = P.e_dmin[e];
      m = edge_match(P, A, e, def, use, &q);
    }
    acc[8] += m.rr; acc[9] += m.sr; acc[10] += m.lu; acc[11] += m.cr;
    add_by_loop(P.adv_own_matched, q, m.lu);
    def -= i0;
    use -= i0;
    top_insert(top[O_RR], Cand{m.rr, def, use, dist});
    top_insert(top[O_SR], Cand{m.sr, def, use, dist});
    top_insert(top[O_LU], Cand{m.lu, def, use, dist});
    top_insert(top[O_CR], Cand{m.cr, def, use, dist});
  }
#pragma unroll
  for (int q = 0; q < kAcc; ++q) {
    unsigned long long v = acc[q];
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    if (lane == 0) red[q][warp] = v;
  }
#pragma unroll
  for (int o = 0; o < N_O; ++o)
    if (lane < kHot) wtop[o][warp][lane] = top[o];
  __syncthreads();
  if (tid < kAcc) {
    unsigned long long v = 0;
    for (int w = 0; w < kWarpsA; ++w) v += red[tid][w];
    tot[tid] = v;
  }
  // The tile's top five, a warp per optimizer in turn.
  for (int o = warp; o < N_O; o += kWarpsA) {
    static_assert(kWarpsA * kHot <= 32, "one lane per entry of the warps' lists");
    Cand best{0ull, 0, 0, 0};
    top_insert(best, lane < kWarpsA * kHot ? wtop[o][lane / kHot][lane % kHot] : Cand{0ull, 0, 0, 0});
    if (nt == 1) {
      __syncwarp();  // (read before it is overwritten)
      if (lane < kHot) wtop[o][0][lane] = best;
    } else if (lane < kHot) {
      AdvCand* out = P.adv_tops + ((size_t)blockIdx.x * N_O + o) * kHot + lane;
      *out = AdvCand{best.v, best.def, best.use, best.dist, 0};
    }
  }
  __syncthreads();
  if (nt > 1) {
    // The last of the function's tiles finishes it.
    unsigned long long* fa = P.adv_acc + (size_t)f * kAdvAcc;
    if (tid < kAcc && tot[tid]) atomicAdd(&fa[tid], tot[tid]);
    __threadfence();
    __syncthreads();
    if (tid == 0) s_last = atomicAdd(&fa[kAcc], 1ull) == (unsigned long long)(nt - 1);
    __syncthreads();
    if (!s_last) return;
    __threadfence();
    if (tid < kAcc) tot[tid] = __ldcg(&fa[tid]);
    for (int o = warp; o < N_O; o += kWarpsA) {
      Cand best{0ull, 0, 0, 0};
      for (int k = 0; k < nt * kHot; k += 32) {
        Cand c{0ull, 0, 0, 0};
        const int q = k + lane;
        if (q < nt * kHot) {
          const int4* in = reinterpret_cast<const int4*>(P.adv_tops + ((size_t)(t0 + q / kHot) * N_O + o) * kHot + q % kHot);
          const int2 v = __ldcg(reinterpret_cast<const int2*>(in));
          const int2 du = __ldcg(reinterpret_cast<const int2*>(in) + 1);
          c.v = (unsigned long long)(uint32_t)v.x | ((unsigned long long)(uint32_t)v.y << 32);
          c.def = du.x;
          c.use = du.y;
          c.dist = __ldcg(reinterpret_cast<const int*>(in) + 4);
        }
        top_insert(best, c);
      }
      if (lane < kHot) wtop[o][0][lane] = best;
    }
    __syncthreads();
  }
  const unsigned long long T = tot[0], Aact = tot[1];
  // Results: the hotspots, a thread per entry; the estimates and the ranking, one
  // thread; the parallel optimizers, another.
  if (tid < N_O * kHot) {
    const int o = tid / kHot, h = tid % kHot;
    const Cand b = wtop[o][0][h];
    long long* out = P.a_hot + ((size_t)f * N_O + o) * kHot * 6 + h * 6;
    if (b.v != 0ull) {
      out[0] = b.def; out[1] = b.use;
      out[2] = P.line[i0 + b.def]; out[3] = P.line[i0 + b.use];
      out[4] = b.dist; out[5] = (long long)b.v;
    } else {
      for (int q = 0; q < 6; ++q) out[q] = -1;
    }
    if (h == 0) {
      int nb = 0;
      while (nb < kHot && wtop[o][0][nb].v != 0ull) ++nb;
      P.a_nhot[(size_t)f * N_O + o] = nb;
    }
  }
  if (tid == 64) {
    unsigned long long M[N_O];
    M[O_RR] = tot[8]; M[O_SR] = tot[9]; M[O_FS] = tot[4]; M[O_FM] = tot[5];
    M[O_WB] = tot[6]; M[O_MT] = tot[7]; M[O_LU] = tot[10]; M[O_CR] = tot[11]; M[O_FI] = tot[12];
    double sp[N_O];
    for (int o = 0; o < N_O; ++o) {
      const bool hide = (o == O_LU || o == O_CR || o == O_FI);
      sp[o] = est(T, hide ? min(Aact, M[o]) : M[o]);
      P.a_matched[(size_t)f * N_O + o] = M[o];
      P.a_speedup[(size_t)f * N_O + o] = sp[o];
    }
    int ord[N_O];
    for (int o = 0; o < N_O; ++o) ord[o] = o;
    for (int a = 1; a < N_O; ++a) {  // stable: ties keep the lower id first
      int v = ord[a], b = a - 1;
      while (b >= 0 && sp[ord[b]] < sp[v]) { ord[b + 1] = ord[b]; --b; }
      ord[b + 1] = v;
    }
    for (int o = 0; o < N_O; ++o) P.a_rank[(size_t)f * N_O + o] = ord[o];
    for (int q = 0; q < 4; ++q) P.a_totals[(size_t)f * 4 + q] = tot[q];
  }
  if (tid == 96) parallel_advice(P, f, T, tot[3]);
  // Eq. 5 per loop scope: each loop's own samples go to it and to the loops
  // around it (this CTA alone reads and writes the function's loop counters now).
  const int l0 = P.func_loop_off[f], l1 = P.func_loop_off[f + 1];
  for (int lp = l0 + tid; lp < l1; lp += kThreads) {
    const unsigned long long al = __ldcg(&P.adv_own_active[lp]), ml = __ldcg(&P.adv_own_matched[lp]);
    for (int q = lp; q >= 0; q = P.loop_parent[q]) {
      if (al) atomicAdd(&P.a_loop_active[q], al);
      if (ml) atomicAdd(&P.a_loop_matched[q], ml);
    }
  }
  __threadfence_block();
  __syncthreads();
  for (int lp = l0 + tid; lp < l1; lp += kThreads)
    P.a_loop_speedup[lp] = est(T, min(__ldcg(&P.a_loop_active[lp]), __ldcg(&P.a_loop_matched[lp])));
}

// Results out in one launch: the arrays are cut into pieces of 4 KB, a CTA per
// piece, written straight into page-locked host memory over the host link (a
// copy per array was fifteen, a few microseconds each: most of the advice call of
// a small program).
constexpr int64_t kOutPiece = 4096;
__global__ void __launch_bounds__(128) k_copy_out(OutList L) {
  int64_t piece = blockIdx.x;
  int k = 0;
  while (k < L.n - 1 && piece >= (L.bytes[k] + kOutPiece - 1) / kOutPiece) piece -= (L.bytes[k++] + kOutPiece - 1) / kOutPiece;
  const int64_t at = piece * kOutPiece, n = min(kOutPiece, L.bytes[k] - at);
  const char* src = static_cast<const char*>(L.src[k]) + at;
  char* dst = static_cast<char*>(L.dst[k]) + at;
  const bool vec = ((reinterpret_cast<uintptr_t>(src) | reinterpret_cast<uintptr_t>(dst)) & 15u) == 0;
  const int64_t nv = vec ? n / 16 : 0;
  for (int64_t i = threadIdx.x; i < nv; i += blockDim.x)
    reinterpret_cast<int4*>(dst)[i] = reinterpret_cast<const int4*>(src)[i];
  for (int64_t i = nv * 4 + threadIdx.x; i < n / 4; i += blockDim.x)
    reinterpret_cast<int*>(dst)[i] = reinterpret_cast<const int*>(src)[i];
}

}  // namespace

void launch_copy_out(const OutList& L, cudaStream_t st, int64_t* launches) {
  int64_t pieces = 0;
  for (int k = 0; k < L.n; ++k) pieces += (L.bytes[k] + kOutPiece - 1) / kOutPiece;
  if (pieces == 0) return;
  k_copy_out<<<(unsigned)pieces, 128, 0, st>>>(L);
  ++*launches;
}

void launch_advise(const Prog& P, const Arch& A, cudaStream_t st, int64_t* launches) {
  // every counter that is added to, in one block
  cudaMemsetAsync(P.adv_acc, 0, sizeof(unsigned long long) * (size_t)P.adv_zero, st);
  k_advise<<<P.adv_tiles, kThreads, 0, st>>>(P, A);
  ++*launches;
}

}  // namespace gpa
