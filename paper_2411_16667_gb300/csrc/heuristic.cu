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
// ship grid, d = 3 (distances shared) 1.37 -> 0.26 ms; 160x160 2.7 -> 0.49;
// 256x256, d = 5 (flags shared) 4.4 -> 1.44; road-like graph of 199,809 nodes,
// d = 4 (flags shared) 16 -> 4.6 ms: 1,400 rounds of 3.3 us. Larger graphs with
// SMs to spare go to a cluster of blocks below.
//
// Scratch per block: near, next, far, far2 (n each) and flags (n).
#include <algorithm>

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

// ---------------------------------------------------------------------------
// One (goal, k) pair by a cluster of kHeurCluster blocks: for graphs whose
// distances do not fit one SM's shared memory, while there are SMs to spare
// (a query's own d pairs; a batch has a pair for every SM). The same search, the
// nodes dealt out to the blocks (node v is number v / kHeurCluster of block
// v % kHeurCluster, so neighbours of a grid go to different blocks), each
// block with its nodes' distances, flags and the heads of their lists in its
// shared memory.
//
// A step: every block relaxes the next nodes of its near list, one arc a lane,
// and writes the (node, distance) each arc gives into the inbox of the node's
// block; one cluster barrier; every block takes the minima of its inbox and
// lists what improved. Only stores and that barrier cross SMs. (Improving the
// distances by atomics on the other blocks' shared memory was a chain of three
// returning atomics a round: 1.35 ms instead of 1.12 on the 256x256 grid below.) Inboxes are two by step parity, with a row for
// every sender, so a slot is a count in the sender's own memory.
//
// A single block's round was a chain of ~7,000 cycles, 5,000 of them scattered
// returning atomics at the L2 for ~130 nodes; a step is 3,600 (1,700 until the
// last arc is sent, 1,400 for the barrier and the slowest block, 300 for the
// inbox). Measured, one block -> cluster: 256x256 ship grid, d = 5: 1.44 -> 1.12
// ms; road-like graph of 199,809 nodes, d = 4: 4.6 -> 2.8 ms, d = 2: 4.1 -> 2.5
// ms. 256 threads a block were 15-25% slower, 1,024 up to 15%.
// ---------------------------------------------------------------------------
constexpr unsigned kHeurCluster = 8;
constexpr unsigned kClusterThreads = 512;  // also the messages of one block to another in a step
constexpr unsigned kClusterNear = 1024;    // entries of each near list kept in shared memory
constexpr unsigned kInboxWords = 2 * kHeurCluster * kClusterThreads * 2;

constexpr size_t cluster_nodes(size_t n) { return (n + kHeurCluster - 1) / kHeurCluster; }
constexpr size_t cluster_words(size_t n) {
  return kInboxWords + 2 * kClusterNear + cluster_nodes(n) + 2 * ((cluster_nodes(n) + 31) / 32);
}

// The address of this block's shared p in block `rank` of the cluster, and
// stores there.
__device__ __forceinline__ unsigned peer(const void* p, unsigned rank) {
  unsigned a;
  asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"((unsigned)__cvta_generic_to_shared(p)), "r"(rank));
  return a;
}
__device__ __forceinline__ void peer_store(unsigned a, unsigned x, unsigned y) {
  asm volatile("st.shared::cluster.v2.u32 [%0], {%1, %2};" ::"r"(a), "r"(x), "r"(y) : "memory");
}
__device__ __forceinline__ void cluster_sync() {
  asm volatile("barrier.cluster.arrive.release;\n\tbarrier.cluster.wait.acquire;" ::: "memory");
}

__global__ void __launch_bounds__(kClusterThreads, 1) __cluster_dims__(kHeurCluster, 1, 1)
    heuristic_cluster_kernel(GraphDev G, const HJob* jobs, uint32_t* scratch, const uint32_t* delta, unsigned* err,
                             unsigned lpn) {
  extern __shared__ __align__(8) uint32_t dyn[];
  __shared__ unsigned s_n[2], s_far_n, s_far2_n, s_fmin;  // entries of the near lists and the far list; smallest far distance
  __shared__ unsigned s_sent[kHeurCluster], s_near, s_low;  // a step's messages: number to each block, any for a near list, smallest far one
  __shared__ uint2 s_info[2][kHeurCluster];  // by step parity, from every block: messages | more << 31, smallest far distance
  const unsigned n = G.n, tid = threadIdx.x, lane = tid & 31u;
  const unsigned rank = blockIdx.x % kHeurCluster, job = blockIdx.x / kHeurCluster;
  const unsigned npc = (n + kHeurCluster - 1) / kHeurCluster, words = (npc + 31) / 32;
  uint2* const inbox = reinterpret_cast<uint2*>(dyn);  // [parity][sender][slot]
  uint32_t* const heads = dyn + kInboxWords;           // of the near lists
  uint32_t* const dist = heads + 2 * kClusterNear;
  uint32_t* const nbit = dist + npc;
  uint32_t* const fbit = nbit + words;
  // the ends of the near lists and the far list twice, npc entries each
  uint32_t* const base = scratch + (size_t)blockIdx.x * 4 * npc;
  auto append = [&](unsigned l, uint32_t lv) {
    const unsigned at = atomicAdd(&s_n[l], 1u);
    if (at < kClusterNear)
      heads[l * kClusterNear + at] = lv;
    else
      base[(size_t)l * npc + at] = lv;
  };
  auto mark = [&](uint32_t* bits, uint32_t lv) -> bool {
    const uint32_t b = 1u << (lv & 31);
    return !(atomicOr(bits + (lv >> 5), b) & b);
  };
  auto unmark = [&](uint32_t* bits, uint32_t lv) { atomicAnd(bits + (lv >> 5), ~(1u << (lv & 31))); };
  const unsigned grp = tid / lpn, gl = tid % lpn, ngrp = kClusterThreads / lpn;
  const unsigned k = jobs[job].k, goal = jobs[job].goal;
  uint32_t* const out = jobs[job].h_out;
  const uint32_t* rc = G.rcost + (size_t)k * G.m;
  const unsigned long long dk = delta[k] ? delta[k] : 1u;
  for (unsigned v = tid; v < npc; v += kClusterThreads) dist[v] = kInf;
  for (unsigned x = tid; x < 2 * words; x += kClusterThreads) nbit[x] = 0;
  if (tid < kHeurCluster) s_sent[tid] = 0;
  if (tid == 0) {
    s_n[0] = s_n[1] = s_far_n = s_near = 0;
    s_fmin = s_low = kInf;
  }
  __syncthreads();
  if (tid == 0 && goal % kHeurCluster == rank) {
    dist[goal / kHeurCluster] = 0;
    mark(nbit, goal / kHeurCluster);
    append(1u, goal / kHeurCluster);
  }
  cluster_sync();  // nobody writes into a block before its start
  // the near list being relaxed, the next entry of it and its end (the other
  // list is being filled); arcs of the lanes' nodes are left
  unsigned cur = 0, pos = 0, nn = 0, ip = 0, fsel = 0;
  int left = 0;
  uint32_t jb = 0, je = 0, du = 0;  // the group's node: next arcs, their end, its distance
  unsigned long long thr = dk;      // the near lists hold distances < thr
  unsigned long long steps = 0;
  const unsigned long long max_steps = 128ull * n + 4096;
  // every block takes every branch of this loop's end alike: they depend on what
  // all have exchanged
  for (;;) {
    if (++steps > max_steps) {
      if (tid == 0) atomicCAS(err, 0u, (unsigned)OPMOS_ERR_TIMEOUT);
      return;
    }
    if (!left) {
      if (pos >= nn) {  // this list is done
        cur ^= 1u;
        pos = 0;
        nn = s_n[cur];
        if (tid == 0) s_n[cur ^ 1u] = 0;
      }
      jb = je = 0;
      if (pos + grp < nn) {
        const unsigned i = pos + grp;
        const uint32_t lu = i < kClusterNear ? heads[cur * kClusterNear + i] : base[(size_t)cur * npc + i];
        const uint32_t u = lu * kHeurCluster + rank;
        jb = __ldg(G.rrowptr + u);
        je = __ldg(G.rrowptr + u + 1);
        du = dist[lu];
        if (gl == 0) unmark(nbit, lu);  // an improvement from here on lists it again
      }
      pos += ngrp;
    }
    if (jb + gl < je) {
      const uint32_t w = __ldg(G.rsrc + jb + gl);
      const uint32_t nd = du + __ldg(rc + jb + gl);
      const unsigned o = w % kHeurCluster;
      const unsigned slot = atomicAdd(&s_sent[o], 1u);
      peer_store(peer(inbox + (ip * kHeurCluster + rank) * kClusterThreads + slot, o), w / kHeurCluster, nd);
      if (nd < thr)
        s_near = 1;
      else
        atomicMin(&s_low, nd);
    }
    jb += lpn;
    left = __syncthreads_or(jb < je);
    if (tid < kHeurCluster) {
      const bool more = left || pos < nn || s_n[cur ^ 1u] || s_near;
      peer_store(peer(&s_info[ip][rank], tid), s_sent[tid] | (more ? 0x80000000u : 0u), min(s_fmin, s_low));
    }
    cluster_sync();
    unsigned more = 0, fmin = kInf;
#pragma unroll
    for (unsigned r = 0; r < kHeurCluster; ++r) {
      more |= s_info[ip][r].x;
      fmin = min(fmin, s_info[ip][r].y);
    }
    if (tid < kHeurCluster) s_sent[tid] = 0;
    if (tid == 0) {
      s_near = 0;
      s_low = kInf;
    }
    // the inbox, two warps a sender
    {
      constexpr unsigned kWarps = kClusterThreads / 32;
      const unsigned from = (tid >> 5) % kHeurCluster;
      const unsigned c = s_info[ip][from].x & 0x7FFFFFFFu;
      const uint2* in = inbox + (ip * kHeurCluster + from) * kClusterThreads;
      for (unsigned i = (tid >> 5) / kHeurCluster * 32 + lane; i < c; i += kWarps / kHeurCluster * 32) {
        const uint2 m = in[i];
        if (m.y < atomicMin(dist + m.x, m.y)) {
          if (m.y < thr) {
            if (mark(nbit, m.x)) append(cur ^ 1u, m.x);
          } else {
            atomicMin(&s_fmin, m.y);
            if (mark(fbit, m.x)) base[(size_t)(2 + fsel) * npc + atomicAdd(&s_far_n, 1u)] = m.x;
          }
        }
      }
    }
    ip ^= 1u;
    __syncthreads();
    if (more & 0x80000000u) continue;
    if (fmin == kInf) break;  // no block has a pending distance
    // pending distances below the old threshold are final; fmin is at most the
    // smallest of the others. Each block sorts its own far list.
    const unsigned long long settled = thr;
    thr = max((unsigned long long)fmin, settled) + dk;
    const unsigned fn = s_far_n;
    const uint32_t* const far = base + (size_t)(2 + fsel) * npc;
    fsel ^= 1u;
    uint32_t* const far2 = base + (size_t)(2 + fsel) * npc;
    __syncthreads();
    if (tid == 0) {
      s_far2_n = 0;
      s_fmin = kInf;
    }
    __syncthreads();
    for (unsigned i = tid; i < fn; i += kClusterThreads) {
      const uint32_t lw = far[i], dw = dist[lw];
      if (dw < thr) {
        unmark(fbit, lw);
        if (dw >= settled && mark(nbit, lw)) append(cur ^ 1u, lw);
      } else {
        atomicMin(&s_fmin, dw);
        far2[atomicAdd(&s_far2_n, 1u)] = lw;
      }
    }
    __syncthreads();
    if (tid == 0) s_far_n = s_far2_n;
    __syncthreads();
  }
  for (unsigned lv = tid; lv < npc; lv += kClusterThreads) {
    const unsigned v = lv * kHeurCluster + rank;
    if (v < n) out[v] = dist[lv];
  }
}

// The mode of a graph of n nodes: everything in shared memory while it fits.
HeurMode heuristic_mode(size_t n, size_t smem) {
  if (heur_words(kDistShared, n) * 4 <= smem) return kDistShared;
  if (heur_words(kFlagsShared, n) * 4 <= smem) return kFlagsShared;
  return kFlagsGlobal;
}

// Lanes a node: as many as its arcs on average, so one round takes most nodes.
unsigned lanes_per_node(const GraphDev& G) {
  unsigned lpn = 4;
  while (lpn < 32 && (unsigned long long)lpn * G.n < G.m) lpn <<= 1;
  return lpn;
}

// Allows a kernel as much dynamic shared memory as any launch of it may take.
// The bound belongs to the kernel, not to the launch, and other threads launch
// it for other graphs (opmos_heuristic_noalloc holds no lock): one that fitted
// this launch could be lowered by another thread just before it.
cudaError_t allow_smem(const void* kernel) {
  return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kHeurSmem);
}

template <HeurMode MODE>
cudaError_t launch_mode(const GraphDev& G, const HJob* jobs, unsigned njobs, uint32_t* scratch,
                        size_t scratch_words_per_block, unsigned blocks, const uint32_t* delta, unsigned* next_job,
                        unsigned* err, cudaStream_t s) {
  const size_t smem = heur_words(MODE, G.n) * 4;
  const cudaError_t e = allow_smem((const void*)heuristic_kernel<MODE>);
  if (e != cudaSuccess) return e;
  heuristic_kernel<MODE><<<blocks, kHeurThreads, smem, s>>>(G, jobs, njobs, scratch, scratch_words_per_block, delta,
                                                            next_job, err, lanes_per_node(G));
  return cudaGetLastError();
}

}  // namespace

Residents residents;

cudaError_t load_heuristic(unsigned* ctr, cudaStream_t s) {
  GraphDev G{};
  G.n = 1;
  cudaError_t e = launch_mode<kDistShared>(G, nullptr, 0, nullptr, 0, 1, nullptr, ctr, ctr + 1, s);
  if (e == cudaSuccess) e = launch_mode<kFlagsShared>(G, nullptr, 0, nullptr, 0, 1, nullptr, ctr, ctr + 1, s);
  if (e == cudaSuccess) e = launch_mode<kFlagsGlobal>(G, nullptr, 0, nullptr, 0, 1, nullptr, ctr, ctr + 1, s);
  return e;
}

cudaError_t launch_heuristic(const GraphDev& G, const HJob* jobs, unsigned njobs, uint32_t* scratch,
                             size_t scratch_words_per_block, unsigned blocks, const uint32_t* delta,
                             unsigned* next_job, unsigned* err, cudaStream_t s, size_t smem, unsigned sms) {
  std::lock_guard<std::mutex> lk(residents.mu);
  if (residents.servers != 0) {
    smem = std::min(smem, kHeurSmemServed);
    sms = 0;
  }
  // a cluster a pair where the distances do not fit one block but fit eight,
  // while every cluster has its SMs at once
  if (heuristic_mode(G.n, smem) != kDistShared && njobs * kHeurCluster <= sms &&
      cluster_words(G.n) * 4 <= smem) {
    const size_t bytes = cluster_words(G.n) * 4;
    const cudaError_t e = allow_smem((const void*)heuristic_cluster_kernel);
    if (e != cudaSuccess) return e;
    heuristic_cluster_kernel<<<njobs * kHeurCluster, kClusterThreads, bytes, s>>>(G, jobs, scratch, delta, err,
                                                                                 lanes_per_node(G));
    return cudaGetLastError();
  }
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
