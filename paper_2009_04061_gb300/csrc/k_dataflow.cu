// Step (b), first half: per-block resource summaries and the reaching-
// definitions fixpoint at resource granularity (Sec. 4, backward slicing over
// registers, predicates and virtual barrier registers).
//
// The classic def-site reaching definitions projected on resources reduces to
// reachability of definitions: some def of r reaches the exit of b iff b
// defines r or some def of r reaches its entry (an unpredicated def kills the
// earlier defs of r but itself reaches on), and reaches the entry iff it
// reaches the exit of a predecessor. So
//   RIN[b] = OR over preds p of ROUT[p],   ROUT[b] = DEF[b] | RIN[b],
// 268-bit masks in 9 words. The backward searches use ROUT to skip blocks no
// def of the searched resource can leave.
#include <algorithm>

#include "gpa_internal.cuh"

namespace gpa {

namespace {

// Thread per basic block, over the block's events: its 16 bucket segments lie
// one after another and hold exactly its defs and its unguarded reads, so the
// loads are independent of one another (walking the instructions' operand lists
// was a chain of three dependent loads an instruction: 24 us for a 12-block
// program, 135 us for 3.3M instructions). The masks stay in registers, each
// resource's bit added to its word by a compare per word (no indexed register
// array), then the 9 words of each mask stored.
__global__ void k_block_masks(Prog P, int windowed) {
  for (int b = blockIdx.x * blockDim.x + threadIdx.x; b < P.nb; b += gridDim.x * blockDim.x) {
    uint32_t dm[kWords], um[kWords];
#pragma unroll
    for (int w = 0; w < kWords; ++w) { dm[w] = 0; um[w] = 0; }
    const int4 m = P.block_meta[2 * (size_t)b];  // (z, w: the block's events)
    for (int e0 = m.z; e0 < m.w; e0 += 4) {
      uint32_t evs[4];
#pragma unroll
      for (int q = 0; q < 4; ++q) evs[q] = e0 + q < m.w ? __ldg(&P.events[e0 + q]) : 0x1FFu;
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const int r = (int)(evs[q] & 0x1FFu);  // (the filler's word 15 is none of the nine)
        const uint32_t bit = 1u << (r & 31);
        const uint32_t db = (evs[q] & 0x200u) ? bit : 0u, ub = (evs[q] & 0x200u) ? 0u : bit;
#pragma unroll
        for (int w = 0; w < kWords; ++w) {
          dm[w] |= (r >> 5) == w ? db : 0u;
          um[w] |= (r >> 5) == w ? ub : 0u;
        }
      }
    }
    const size_t o = (size_t)b * kWords;
#pragma unroll
    for (int w = 0; w < kWords; ++w) {
      P.def_mask[o + w] = dm[w];
      P.touch_mask[o + w] = dm[w] | um[w];
      if (windowed) {  // its fixpoint starts from these; the other kernels write every word
        P.rin[o + w] = 0u;
        P.rout[o + w] = dm[w];
      }
    }
  }
}

// Largest latency of any def of each resource in each function (the
// distance beyond which no def of that resource can pass the latency rule),
// and the guard literals its defs carry there.
__global__ void k_res_maxlat(Prog P, Arch A) {
  for (int x = blockIdx.x * blockDim.x + threadIdx.x; x < P.ni; x += gridDim.x * blockDim.x) {
    const int f = P.block_func[P.instr_block[x]];
    const int lat = A.lat[P.opclass[x]];
    const int g = P.guard[x];
    for (int e = P.def_off[x]; e < P.def_off[x + 1]; ++e) {
      const size_t k = (size_t)f * kNumRes + (P.def_res[e] & 0x1FF);
      atomicMax(&P.res_maxlat[k], lat);
      if (g) atomicOr(&P.res_guards[k], 1u << (g - 1));
    }
  }
}

// One CTA per function, the function staged in shared memory: ROUT (9 words
// per block, starting at DEF), and per block a record of its first two
// predecessors other than the block before it, its innermost loop, and flags
// (the block before it is a predecessor; more predecessors in the CSR). ROUT
// only grows, so ROUT[b] = ROUT[b] | OR of the predecessors' ROUT needs no
// separate DEF. A sweep visits the blocks one after another in layout order (a
// topological order of the forward edges, so one sweep carries a def along any
// forward path), lanes 0-8 of the first warp over the 9 words, with the
// previous block's ROUT in a register. A block's other predecessors are never
// the block just before it, so their words for the next block are loaded
// before this block's ROUT is stored, through a record that was loaded one
// block earlier still (missing predecessors point at a row of zeros): the
// sweep's chain per block is one shared-memory load. The rest (staging, records, loop masks, RIN and the copy-out) is
// spread over the CTA's threads.
// When every loop body of the function is a natural loop (or it has none),
// each block also takes in, from the start, the defs of the bodies of the loops
// around it: every block of a natural loop reaches every other one through the
// back edge, and a def from outside a loop enters it through its header, which
// precedes the body in layout order. With that, the first sweep gives every
// block all the defs that reach it: the least fixpoint, in one sweep. Other
// functions sweep until a sweep changes nothing (max_sweeps at most). Then RIN
// = OR of the predecessors' ROUT and both go to global memory. The launch
// takes reach_order[q_lo, q_hi) from the counter at `head`; functions needing
// more than `cap` bytes are left to another launch.
__device__ __forceinline__ void cp_async4(void* smem_dst, const void* src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"((uint32_t)__cvta_generic_to_shared(smem_dst)),
               "l"(src)
               : "memory");
}
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_all;" ::: "memory"); }

__global__ void __launch_bounds__(256) k_reaching_smem(Prog P, int max_sweeps, int q_lo, int q_hi, int head, int cap) {
  extern __shared__ __align__(16) uint32_t sm[];
  __shared__ int s_f;
  const int tid = threadIdx.x, nt = blockDim.x;
  while (true) {
    // Functions are taken largest first, so the long ones start early.
    __syncthreads();  // every thread has read s_f and left the previous function's stage
    if (tid == 0) {
      const unsigned long long q = atomicAdd(&P.stats[head], 1ull) + (unsigned long long)q_lo;
      s_f = q < (unsigned long long)q_hi ? P.reach_order[q] : -1;
    }
    __syncthreads();
    const int f = s_f;
    if (f < 0) break;
    const int b0 = P.func_block_off[f], b1 = P.func_block_off[f + 1], nbf = b1 - b0;
    const int e0 = P.pred_off[b0], ne = P.pred_off[b1] - e0;
    const int l0 = P.func_loop_off[f], nlf = P.func_loop_off[f + 1] - l0;
    if (nbf == 0 || reach_smem_need(nbf, ne, nlf) > cap) continue;  // the same for every thread
    const bool exact = P.func_natural[f];  // one seeded sweep is the fixpoint
    const bool seed = exact && nlf > 0;
    uint32_t* so = sm;
    const int rows = nbf * kWords + kWords;  // ROUT and a row of zeros
    int4* rec = reinterpret_cast<int4*>(so + ((rows + 3) & ~3));
    int* spo = reinterpret_cast<int*>(rec + nbf);
    int* sp = spo + nbf + 1;
    int* sloop = sp + ne;
    int* spar = sloop + nbf;
    uint32_t* ldef = reinterpret_cast<uint32_t*>(spar + nlf);
    uint32_t* lin = ldef + (size_t)nlf * kWords;  // (and a row of zeros)
    // Staging: asynchronous 4-byte copies, all in flight together, then the
    // global indices rebased to the function in place.
    for (int t = tid; t < nbf * kWords; t += nt) cp_async4(so + t, P.def_mask + (size_t)b0 * kWords + t);
    for (int t = tid; t <= nbf; t += nt) cp_async4(spo + t, P.pred_off + b0 + t);
    for (int t = tid; t < ne; t += nt) cp_async4(sp + t, P.pred + e0 + t);
    if (seed) {
      for (int t = tid; t < nbf; t += nt) cp_async4(sloop + t, P.block_loop + b0 + t);
      for (int t = tid; t < nlf; t += nt) cp_async4(spar + t, P.loop_parent + l0 + t);
    }
    if (tid < kWords) { so[nbf * kWords + tid] = 0u; lin[(size_t)(seed ? nlf : 0) * kWords + tid] = 0u; }
    cp_async_wait_all();
    __syncthreads();
    for (int t = tid; t <= nbf; t += nt) spo[t] -= e0;
    for (int t = tid; t < ne; t += nt) sp[t] -= b0;
    if (seed) {
      for (int t = tid; t < nbf; t += nt) sloop[t] = sloop[t] >= 0 ? sloop[t] - l0 : -1;
      for (int t = tid; t < nlf; t += nt) spar[t] = spar[t] >= 0 ? spar[t] - l0 : -1;
      for (int t = tid; t < nlf * kWords; t += nt) ldef[t] = 0u;
    }
    __syncthreads();
    for (int b = tid; b < nbf; b += nt) {
      int p1 = -1, p2 = -1, fl = 0;
      for (int e = spo[b]; e < spo[b + 1]; ++e) {
        const int p = sp[e];
        if (p == b - 1) fl |= 1;
        else if (p1 < 0) p1 = p;
        else if (p2 < 0) p2 = p;
        else fl |= 2;
      }
      // word offsets of the two predecessors' rows and the loop's row
      const int l = seed ? sloop[b] : -1;
      rec[b] = make_int4((p1 >= 0 ? p1 : nbf) * kWords, (p2 >= 0 ? p2 : nbf) * kWords,
                         (l >= 0 ? l : (seed ? nlf : 0)) * kWords, fl);
    }
    if (seed) {
      // the defs of each loop's body, nested loops included
      for (int t = tid; t < nbf * kWords; t += nt) {
        const uint32_t v = so[t];
        if (!v) continue;
        const int w = t % kWords;
        for (int l = sloop[t / kWords]; l >= 0; l = spar[l]) atomicOr(&ldef[l * kWords + w], v);
      }
      __syncthreads();
      // and of the enclosing loops' bodies
      for (int t = tid; t < nlf * kWords; t += nt) {
        const int w = t % kWords;
        uint32_t v = 0u;
        for (int l = t / kWords; l >= 0; l = spar[l]) v |= ldef[l * kWords + w];
        lin[t] = v;
      }
    }
    __syncthreads();
    if (tid < 32) {
      const int lane = tid;
      bool converged = false;
      int sweep = 0;
      const int limit = exact ? 1 : max_sweeps;
      for (; sweep < limit && !converged; ++sweep) {
        bool ch = false;
        if (lane < kWords) {
          // words from the record's two predecessors and the enclosing loops
          auto pre = [&](const int4& r) -> uint32_t { return lin[r.z + lane] | so[r.x + lane] | so[r.y + lane]; };
          uint32_t prev = 0u;
          int4 r = rec[0], rn = rec[nbf > 1 ? 1 : 0];
          uint32_t old = so[lane];
          uint32_t in_r = pre(r);
          for (int b = 0; b < nbf; ++b) {
            // (the last iterations load their own block's words again)
            const int bn = b + 1 < nbf ? b + 1 : b;
            const int4 rnn = rec[b + 2 < nbf ? b + 2 : b];
            const uint32_t oldn = so[bn * kWords + lane];
            const uint32_t in_n = pre(rn);  // its rows are not b's: not written below
            uint32_t in = in_r;
            if (r.w & 1) in |= prev;
            if (r.w & 2)
              for (int e = spo[b]; e < spo[b + 1]; ++e) in |= so[sp[e] * kWords + lane];
            const uint32_t o = old | in;
            ch |= o != old;
            so[b * kWords + lane] = o;
            prev = o;
            r = rn;
            rn = rnn;
            old = oldn;
            in_r = in_n;
          }
        }
        converged = exact || !__any_sync(0xffffffffu, ch);
      }
      if (lane == 0) {
        if (!converged) set_status(P, ST_NOT_CONVERGED);
        atomicMax(&P.stats[SS_SWEEPS], (unsigned long long)sweep);
      }
    }
    __syncthreads();
    for (int t = tid; t < nbf * kWords; t += nt) {
      const int b = t / kWords, w = t - b * kWords;
      uint32_t in = 0u;
      for (int e = spo[b]; e < spo[b + 1]; ++e) in |= so[sp[e] * kWords + w];
      P.rin[(size_t)b0 * kWords + t] = in;
      P.rout[(size_t)b0 * kWords + t] = so[t];
    }
  }
}

// Functions of natural loops whose stage does not fit an SM's shared memory
// (more than about 3,000 blocks): a CTA per function and word of the masks, so
// that one word per block fits (51,000 blocks). One thread runs the seeded sweep
// over the word; the other warps prepare the records of the next 512 blocks
// meanwhile (the two predecessors other than the block before, the enclosing
// loops' defs, the flags). 17,000 blocks: 50 ms with the kernel below on one
// warp, the sweep's chain of a shared-memory load a block now.
constexpr int kRecChunk = 512;
__global__ void __launch_bounds__(256) k_reaching_words(Prog P, int cap) {
  extern __shared__ __align__(16) uint32_t sm[];
  const int tid = threadIdx.x, nt = blockDim.x, w = blockIdx.y;
  const int f = P.reach_order[blockIdx.x];
  const int b0 = P.func_block_off[f], nbf = P.func_block_off[f + 1] - b0;
  const int l0 = P.func_loop_off[f], nlf = P.func_loop_off[f + 1] - l0;
  if (!P.func_natural[f] || reach_words_need(nbf, nlf) > cap) return;  // left to k_reaching
  int4* rec = reinterpret_cast<int4*>(sm);          // two chunks
  uint32_t* so = sm + 2 * kRecChunk * 4;            // nbf words, then a zero
  uint32_t* ldef = so + nbf + 1;                    // per loop: the defs of its body
  uint32_t* lin = ldef + nlf;                       // and of its body and the loops around it
  for (int b = tid; b < nbf; b += nt) so[b] = P.def_mask[(size_t)(b0 + b) * kWords + w];
  if (tid == 0) so[nbf] = 0u;
  for (int l = tid; l < nlf; l += nt) ldef[l] = 0u;
  __syncthreads();
  if (nlf > 0) {
    for (int b = tid; b < nbf; b += nt) {
      const uint32_t v = so[b];
      if (v)
        for (int l = P.block_loop[b0 + b]; l >= 0; l = P.loop_parent[l]) atomicOr(&ldef[l - l0], v);
    }
    __syncthreads();
    for (int l = tid; l < nlf; l += nt) {
      uint32_t v = 0u;
      for (int q = l + l0; q >= 0; q = P.loop_parent[q]) v |= ldef[q - l0];
      lin[l] = v;
    }
    __syncthreads();
  }
  auto build = [&](int c, int t0, int step) {  // records of chunk c
    const int n = min(kRecChunk, nbf - c * kRecChunk);
    for (int i = t0; i < n; i += step) {
      const int b = c * kRecChunk + i;
      int p1 = nbf, p2 = nbf, fl = 0;
      const int q1 = P.pred_off[b0 + b + 1];
      for (int q = P.pred_off[b0 + b]; q < q1; ++q) {
        const int p = P.pred[q] - b0;
        if (p == b - 1) fl |= 1;
        else if (p1 == nbf) p1 = p;
        else if (p2 == nbf) p2 = p;
        else fl |= 2;
      }
      const int l = nlf > 0 ? P.block_loop[b0 + b] : -1;
      rec[(c & 1) * kRecChunk + i] = make_int4(p1, p2, l >= 0 ? (int)lin[l - l0] : 0, fl);
    }
  };
  const int chunks = (nbf + kRecChunk - 1) / kRecChunk;
  build(0, tid, nt);
  __syncthreads();
  uint32_t prev = 0u;
  for (int c = 0; c < chunks; ++c) {
    if (tid == 0) {
      const int4* rc = rec + (c & 1) * kRecChunk;
      const int first = c * kRecChunk, n = min(kRecChunk, nbf - first);
      int4 r = rc[0], rn = rc[n > 1 ? 1 : 0];
      uint32_t in_r = so[first] | so[r.x] | so[r.y] | (uint32_t)r.z;
      for (int i = 0; i < n; ++i) {
        const int b = first + i;
        const int4 rnn = rc[i + 2 < n ? i + 2 : i];
        const uint32_t in_n = so[i + 1 < n ? b + 1 : b] | so[rn.x] | so[rn.y] | (uint32_t)rn.z;
        uint32_t o = in_r;
        if (r.w & 1) o |= prev;
        if (r.w & 2)
          for (int q = P.pred_off[b0 + b]; q < P.pred_off[b0 + b + 1]; ++q) o |= so[P.pred[q] - b0];
        so[b] = o;
        prev = o;
        r = rn;
        rn = rnn;
        in_r = in_n;
      }
    } else if (tid >= 32 && c + 1 < chunks) {
      build(c + 1, tid - 32, nt - 32);
    }
    __syncthreads();
  }
  for (int b = tid; b < nbf; b += nt) {
    uint32_t in = 0u;
    for (int q = P.pred_off[b0 + b]; q < P.pred_off[b0 + b + 1]; ++q) in |= so[P.pred[q] - b0];
    P.rin[(size_t)(b0 + b) * kWords + w] = in;
    P.rout[(size_t)(b0 + b) * kWords + w] = so[b];
  }
  if (tid == 0) atomicMax(&P.stats[SS_SWEEPS], 1ull);
}

// Warp per function. Blocks are visited in layout order (a topological order
// of the forward edges) 32 at a time, lane per block; inside a window the
// lanes iterate until __ballot_sync reports no change, then move on. A full
// pass without change ends the fixpoint; max_sweeps passes without reaching it
// set ST_NOT_CONVERGED. Monotone OR updates from 0 make the result the least
// fixpoint regardless of the visiting order. Takes the functions the staged
// kernel does not (every function with `all`).
__global__ void k_reaching(Prog P, int max_sweeps, int all) {
  const int lane = threadIdx.x & 31;
  const int warp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int n_warps = (gridDim.x * blockDim.x) >> 5;
  for (int f = warp; f < P.nf; f += n_warps) {
    const int b0 = P.func_block_off[f], b1 = P.func_block_off[f + 1];
    if (!all && b1 > b0 &&
        reach_smem_need(b1 - b0, P.pred_off[b1] - P.pred_off[b0], P.func_loop_off[f + 1] - P.func_loop_off[f]) <=
            P.reach_smem)
      continue;
    if (!all && P.func_natural[f] &&
        reach_words_need(b1 - b0, P.func_loop_off[f + 1] - P.func_loop_off[f]) <= kReachSmemCap)
      continue;
    bool converged = false;
    int sweep = 0;
    for (; sweep < max_sweeps && !converged; ++sweep) {
      bool changed_any = false;
      for (int w0 = b0; w0 < b1; w0 += 32) {
        const int b = w0 + lane;
        const bool mine = b < b1;
        for (int it = 0; it < 64; ++it) {
          bool ch = false;
          if (mine) {
            uint32_t in[kWords];
#pragma unroll
            for (int w = 0; w < kWords; ++w) in[w] = 0u;
            for (int e = P.pred_off[b]; e < P.pred_off[b + 1]; ++e) {
              const volatile uint32_t* ro = P.rout + (size_t)P.pred[e] * kWords;
#pragma unroll
              for (int w = 0; w < kWords; ++w) in[w] |= ro[w];
            }
            volatile uint32_t* ri = P.rin + (size_t)b * kWords;
            volatile uint32_t* ro = P.rout + (size_t)b * kWords;
            const uint32_t* dm = P.def_mask + (size_t)b * kWords;
#pragma unroll
            for (int w = 0; w < kWords; ++w) {
              const uint32_t o = dm[w] | in[w];
              if (in[w] != ri[w] || o != ro[w]) ch = true;
              ri[w] = in[w];
              ro[w] = o;
            }
          }
          __syncwarp();
          if (!__ballot_sync(0xffffffffu, ch)) break;
          changed_any = true;
        }
      }
      converged = !changed_any;
    }
    if (lane == 0) {
      if (!converged) set_status(P, ST_NOT_CONVERGED);
      atomicMax(&P.stats[SS_SWEEPS], (unsigned long long)sweep);
    }
  }
}

}  // namespace

void launch_dataflow(const Prog& P, const Arch& A, int max_sweeps, int schedule, const SearchFork* fork,
                     cudaStream_t st, int sms, int64_t* launches) {
  k_block_masks<<<(P.nb + 127) / 128, 128, 0, st>>>(P, schedule == 1 || P.reach_windowed > 0);
  ++*launches;
  const bool staged = schedule == 0 && P.reach_smem > 0;
  const int n_big = schedule == 0 ? P.reach_cls[0] : P.nf;  // functions beyond the staged kernel
  // The launches write different functions' masks, so they run side by side: a
  // function's sweep is one warp's chain, and each launch lasts as long as its
  // largest function's.
  int parts = n_big > 0 ? 1 : 0;
  for (int c = 0; staged && c < 4; ++c) parts += P.reach_cls[c + 1] > P.reach_cls[c] ? 1 : 0;
  const bool split = parts > 1;
  cudaStream_t on[4] = {st, st, st, st};
  if (split) {
    on[1] = on[3] = fork->side[0];
    on[2] = fork->side[1];
    cudaEventRecord(fork->fork, st);
    cudaStreamWaitEvent(fork->side[0], fork->fork, 0);
    cudaStreamWaitEvent(fork->side[1], fork->fork, 0);
  }
  int part = 0;
  if (n_big > 0) {
    if (schedule == 0) {
      allow_max_smem(k_reaching_words);
      k_reaching_words<<<dim3(n_big, kWords), 256, kReachSmemCap, on[0]>>>(P, (int)kReachSmemCap);
      ++*launches;
    }
    if (schedule == 1 || P.reach_windowed) {
      int fblocks = (P.nf * 32 + 127) / 128;
      if (fblocks > sms * 16) fblocks = sms * 16;
      if (fblocks < 1) fblocks = 1;
      k_reaching<<<fblocks, 128, 0, on[0]>>>(P, max_sweeps, schedule == 1 ? 1 : 0);
      ++*launches;
    }
    ++part;
  }
  if (staged) {
    // One launch per size class: the larger the functions, the more shared
    // memory each warp stages and the fewer warps per SM.
    allow_max_smem(k_reaching_smem);
    for (int c = 0; c < 4; ++c) {
      const int n = P.reach_cls[c + 1] - P.reach_cls[c];
      if (n <= 0 || P.reach_cls_smem[c] <= 0) continue;
      const int smem = P.reach_cls_smem[c];
      const int per_sm = std::max(1, std::min(32, (int)((200 * 1024) / (smem + 1024))));
      const int g = std::min(n, sms * per_sm);
      // the larger the functions, the more threads share a function's
      // staging, records and copy-out (its sweep is one warp's in any case)
      const int threads = c == 0 ? 256 : c == 1 ? 128 : c == 2 ? 64 : 32;
      k_reaching_smem<<<g, threads, smem, on[part & 3]>>>(P, max_sweeps, P.reach_cls[c], P.reach_cls[c + 1],
                                                          SS_REACH_CLS + c, smem);
      ++part;
      ++*launches;
    }
  }
  cudaMemsetAsync(P.res_maxlat, 0, 2 * sizeof(int32_t) * (size_t)P.nf * kNumRes, st);  // and res_guards, behind it
  k_res_maxlat<<<grid_for(P.ni, 256, sms), 256, 0, st>>>(P, A);
  ++*launches;
  if (split) {
    for (int k = 0; k < 2; ++k) {
      cudaEventRecord(fork->join[k], fork->side[k]);
      cudaStreamWaitEvent(st, fork->join[k], 0);
    }
  }
}

}  // namespace gpa
