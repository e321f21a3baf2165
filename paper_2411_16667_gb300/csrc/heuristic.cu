// Ideal-point heuristic (Sec. 4; the "heuristics H" input of Algorithms 1-2):
// h_k(v) = length of the shortest v -> goal path under objective k alone.
//
// One thread block computes one (goal, k) pair by a bucketed label-correcting
// single-source shortest-path search from the goal over the reversed arcs
// (near/far variant of delta-stepping): nodes whose tentative distance is
// below the current threshold are relaxed in rounds until none improves, the
// threshold then moves delta past the smallest pending distance. The distances
// are exact shortest distances (label-correcting converges to them);
// unreachable nodes keep 0xFFFFFFFF.
//
// What bounds it: a round is one chain of dependent accesses (list entry, node,
// arc, distance, minimum, list) and there are hundreds of rounds, so the time
// is rounds x chain, not bytes. Hence a group of lanes takes one node and a
// lane one arc (a thread that walked its node's arcs one after the other made
// the chain eight times longer), and everything the chain touches twice stays
// in shared memory when it fits:
//   kDistShared    distances, list flags and the heads of the near lists (the
//                  returning atomics of a round take ~100 cycles instead of
//                  ~650 at the L2): up to kDistNodes nodes
//   kFlagsShared   list flags (two bits a node) and list heads: up to
//                  kFlagsNodes nodes
//   kFlagsGlobal   list heads only: larger graphs
// Measured, one thread per node and all lists in global memory -> here: 97x89
// ship grid, d = 3 (distances shared) 1.37 -> 0.28 ms; 160x160 2.7 -> 0.52;
// 256x256, d = 5 (flags shared) 4.4 -> 1.5; road-like graph of 199,809 nodes,
// d = 4 (flags shared) 16 -> 4.8 ms: 1,400 rounds of 3.4 us.
//
// Scratch per block: near, next, far, far2 (n each) and flags (n).
#include "opmos_dev.cuh"
#include "search.cuh"

namespace opmos {

namespace {

// A full block (two to an SM, 32 registers a thread): a round's wide frontiers
// are bound by the loads one SM has in flight (512 threads were 1.5 times slower).
constexpr unsigned kHeurThreads = 1024;
constexpr unsigned kNearShared = 2048;  // entries of each near list kept in shared memory

enum HeurMode { kFlagsGlobal = 0, kFlagsShared = 1, kDistShared = 2 };

// Words of dynamic shared memory a mode takes for n nodes.
size_t heur_words(HeurMode mode, size_t n) {
  const size_t bits = 2 * ((n + 31) / 32);
  return 2 * kNearShared + (mode >= kFlagsShared ? bits : 0) + (mode == kDistShared ? n : 0);
}

template <HeurMode MODE>
__global__ void __launch_bounds__(kHeurThreads, 2)
    heuristic_kernel(GraphDev G, const HJob* jobs, unsigned njobs, uint32_t* scratch, size_t spb,
                     const uint32_t* delta, unsigned* next_job, unsigned* err, unsigned lpn) {
  extern __shared__ uint32_t dyn[];
  __shared__ unsigned s_job, s_near_n, s_next_n, s_far_n, s_far2_n, s_fmin;
  const unsigned n = G.n, tid = threadIdx.x, nt = blockDim.x;
  uint32_t* base = scratch + (size_t)blockIdx.x * spb;
  const unsigned words = (n + 31) / 32;
  // near list l = 0, 1: entry i at dyn[l * kNearShared + i] while i < kNearShared, at base[l * n + i] beyond
  uint32_t* const nbit = MODE >= kFlagsShared ? dyn + 2 * kNearShared : base + 4 * (size_t)n;
  uint32_t* const fbit = MODE >= kFlagsShared ? nbit + words : nullptr;
  uint32_t* const sdist = nbit + 2 * words;  // kDistShared
  // a group of lpn lanes (a power of two) takes one node
  const unsigned grp = tid / lpn, gl = tid % lpn, ngrp = nt / lpn;
  for (;;) {
    if (tid == 0) s_job = atomicAdd(next_job, 1u);
    __syncthreads();
    const unsigned job = s_job;
    __syncthreads();
    if (job >= njobs) return;
    const unsigned k = jobs[job].k, goal = jobs[job].goal;
    uint32_t* const out = jobs[job].h_out;
    uint32_t* const dist = MODE == kDistShared ? sdist : out;
    const uint32_t* rc = G.rcost + (size_t)k * G.m;
    const unsigned long long dk = delta[k] ? delta[k] : 1u;
    auto at = [&](uint32_t w) -> uint32_t { return MODE == kDistShared ? dist[w] : __ldcg(dist + w); };
    // Sets node w's flag in the near (far) list; true if it was not set.
    // kFlagsGlobal keeps both flags of a node in one word.
    auto mark = [&](uint32_t w, bool far) -> bool {
      if (MODE == kFlagsGlobal) return !(atomicOr(&nbit[w], far ? 2u : 1u) & (far ? 2u : 1u));
      const uint32_t b = 1u << (w & 31);
      return !(atomicOr((far ? fbit : nbit) + (w >> 5), b) & b);
    };
    auto unmark = [&](uint32_t w, bool far) {
      if (MODE == kFlagsGlobal)
        atomicAnd(&nbit[w], far ? ~2u : ~1u);
      else
        atomicAnd((far ? fbit : nbit) + (w >> 5), ~(1u << (w & 31)));
    };
    for (unsigned v = tid; v < n; v += nt) dist[v] = kInf;
    for (unsigned x = tid; x < (MODE == kFlagsGlobal ? n : 2 * words); x += nt) nbit[x] = 0;
    __syncthreads();
    unsigned cur = 0;  // near list in use
    uint32_t* far = base + 2 * (size_t)n;
    uint32_t* far2 = base + 3 * (size_t)n;
    auto put = [&](unsigned l, unsigned i, uint32_t w) {
      if (i < kNearShared)
        dyn[l * kNearShared + i] = w;
      else
        base[(size_t)l * n + i] = w;
    };
    auto get = [&](unsigned l, unsigned i) -> uint32_t {
      return i < kNearShared ? dyn[l * kNearShared + i] : __ldcg(base + (size_t)l * n + i);
    };
    if (tid == 0) {
      dist[goal] = 0;
      put(0, 0, goal);
      mark(goal, false);
      s_near_n = 1;
      s_next_n = 0;
      s_far_n = 0;
      s_fmin = kInf;
    }
    __syncthreads();
    unsigned long long thr = dk;  // near holds distances < thr
    unsigned long long rounds = 0;
    const unsigned long long max_rounds = 64ull * n + 4096;
    for (;;) {
      for (;;) {
        const unsigned nn = s_near_n;
        if (nn == 0) break;
        if (++rounds > max_rounds) {
          if (tid == 0) atomicCAS(err, 0u, (unsigned)OPMOS_ERR_TIMEOUT);
          return;
        }
        // flags down first: a node improved from here on joins the next list
        for (unsigned i = tid; i < nn; i += nt) unmark(get(cur, i), false);
        __syncthreads();
        for (unsigned i = grp; i < nn; i += ngrp) {
          const uint32_t u = get(cur, i);
          const uint32_t j0 = __ldg(G.rrowptr + u), j1 = __ldg(G.rrowptr + u + 1);
          const uint32_t du = at(u);
          for (uint32_t j = j0 + gl; j < j1; j += lpn) {
            const uint32_t w = __ldg(G.rsrc + j);
            const uint32_t nd = du + __ldg(rc + j);
            // no look at dist[w] first: it would be one more link of the chain
            if (nd < atomicMin(&dist[w], nd)) {
              if (nd < thr) {
                if (mark(w, false)) put(cur ^ 1u, atomicAdd(&s_next_n, 1u), w);
              } else {
                atomicMin(&s_fmin, nd);
                if (mark(w, true)) far[atomicAdd(&s_far_n, 1u)] = w;
              }
            }
          }
        }
        __syncthreads();
        cur ^= 1u;
        if (tid == 0) {
          s_near_n = s_next_n;
          s_next_n = 0;
        }
        __syncthreads();
      }
      const unsigned fn = s_far_n;
      if (fn == 0) break;
      // pending distances below the old threshold are final; s_fmin is at most
      // the smallest of the others
      const unsigned long long settled = thr;
      thr = max((unsigned long long)s_fmin, settled) + dk;
      __syncthreads();
      if (tid == 0) {
        s_far2_n = 0;
        s_fmin = kInf;
      }
      __syncthreads();
      for (unsigned i = tid; i < fn; i += nt) {
        const uint32_t w = __ldcg(far + i);
        const uint32_t dw = at(w);
        if (dw < thr) {
          unmark(w, true);
          if (dw >= settled) {
            mark(w, false);
            put(cur, atomicAdd(&s_near_n, 1u), w);
          }
        } else {
          atomicMin(&s_fmin, dw);
          far2[atomicAdd(&s_far2_n, 1u)] = w;
        }
      }
      __syncthreads();
      uint32_t* t = far;
      far = far2;
      far2 = t;
      if (tid == 0) s_far_n = s_far2_n;
      __syncthreads();
    }
    if (MODE == kDistShared) {
      for (unsigned v = tid; v < n; v += nt) out[v] = dist[v];
      __syncthreads();
    }
  }
}

// The mode of a graph of n nodes: everything in shared memory while it fits.
HeurMode heuristic_mode(size_t n, size_t smem) {
  if (heur_words(kDistShared, n) * 4 <= smem) return kDistShared;
  if (heur_words(kFlagsShared, n) * 4 <= smem) return kFlagsShared;
  return kFlagsGlobal;
}

template <HeurMode MODE>
cudaError_t launch_mode(const GraphDev& G, const HJob* jobs, unsigned njobs, uint32_t* scratch,
                        size_t scratch_words_per_block, unsigned blocks, const uint32_t* delta, unsigned* next_job,
                        unsigned* err, cudaStream_t s) {
  const size_t smem = heur_words(MODE, G.n) * 4;
  const cudaError_t e = cudaFuncSetAttribute((const void*)heuristic_kernel<MODE>,
                                             cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  // lanes a node: as many as its arcs on average, so one round takes most nodes
  unsigned lpn = 4;
  while (lpn < 32 && (unsigned long long)lpn * G.n < G.m) lpn <<= 1;
  heuristic_kernel<MODE><<<blocks, kHeurThreads, smem, s>>>(G, jobs, njobs, scratch, scratch_words_per_block, delta,
                                                            next_job, err, lpn);
  return cudaGetLastError();
}

}  // namespace

cudaError_t launch_heuristic(const GraphDev& G, const HJob* jobs, unsigned njobs, uint32_t* scratch,
                             size_t scratch_words_per_block, unsigned blocks, const uint32_t* delta,
                             unsigned* next_job, unsigned* err, cudaStream_t s, size_t smem) {
  switch (heuristic_mode(G.n, smem)) {
    case kDistShared:
      return launch_mode<kDistShared>(G, jobs, njobs, scratch, scratch_words_per_block, blocks, delta, next_job, err, s);
    case kFlagsShared:
      return launch_mode<kFlagsShared>(G, jobs, njobs, scratch, scratch_words_per_block, blocks, delta, next_job, err, s);
    default:
      return launch_mode<kFlagsGlobal>(G, jobs, njobs, scratch, scratch_words_per_block, blocks, delta, next_job, err, s);
  }
}

}  // namespace opmos
