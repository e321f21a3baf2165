// Ordered-parallel multi-objective label-setting search (Sec. 5, Algorithm 2)
// on one GPU, pipelined as in Sec. 5.1. One "team" of threads works on one
// query: the whole cooperative grid for a single query, or a share of the
// grid's blocks per query in the multi-query kernel.
//
// Step i of the search is ONE phase between two team barriers, in which two
// things run side by side on the team's warps (Sec. 5.1: the next batch is
// extracted while the current one is processed):
//
//   merge (window i)     the candidates produced by expanding window i are
//                        merged node by node, one warp per target node (split
//                        into parts of one warp each when there is much to
//                        compare):
//                        resolved against each other (in-batch dominance and
//                        duplicates), against the node's frontier alpha(v')
//                        (Algorithm 1: weakly dominated candidates are dropped,
//                        strictly dominated frontier labels are pruned), then
//                        against P on F (Algorithm 1); survivors become labels,
//                        join alpha(v') and the next OPEN. Extracted goal
//                        labels reach a virtual node n standing for P, whose
//                        merge applies the goal branch of Algorithm 1 and
//                        appends survivors to the P log.
//   extract (window i+1) OPEN_i is scanned once: the window is every live entry
//                        in the lowest histogram bins of (F[0], F[1]) whose
//                        cumulative count stays within W (the NUM_POP of
//                        Sec. 5); pruned entries are dropped (lazy OPEN delete,
//                        Sec. 5.1) and so are entries whose F a logged solution
//                        weakly dominates (PruneOPEN of Algorithm 1, applied
//                        lazily); window labels are expanded at once along
//                        their out-arcs (g' = g + c(e), dropped when h(v') is
//                        infinite or a champion of the node -- one of its best
//                        accepted labels -- dominates it) into the other candidate set;
//                        all other entries are carried to OPEN_{i+1}.
//
// Labels created by merge i therefore become extractable from window i+2 on:
// the same one-step lag as the paper's asynchronous scheme, which leaves the
// result exact (only the amount of work changes).
//
// The histogram of OPEN_{i+1} is built while its entries are written (carried
// entries and new labels), on bins fixed at the start of step i. Its F[0]
// origin is a lower bound on every key OPEN_{i+1} can hold: with a consistent
// heuristic a child's F is at least its parent's, so min F[0] over OPEN plus
// the window in flight never decreases. A bin holds 2^s2 consecutive cells
// q * 256 + x, q the F[0] bucket and x the F[1] cell of a key, so that every
// bin prefix is a lexicographic prefix of OPEN.
//
// Determinism: a label pruned in step j is still extractable in step j (its
// ldead word records j, and extraction drops labels with ldead < i), equal
// candidates at a node keep the smallest arc id, a label created in step i
// that an equal candidate with a smaller arc id meets takes that candidate's
// parent and arc, and a label created and pruned within one step is taken
// back out of the histogram. Given the launch parameters, the windows, the
// fronts and the paths do not depend on the timing of the threads.
//
// The F-against-P tests use an index of P rebuilt once P has grown by 32 +
// a fraction of its indexed count: P sorted along a Z-order curve over
// objectives 1..3 in tiles of 32, each with its componentwise minimum, plus
// the goal costs logged since; a rebuild runs over three steps (rank,
// scatter, tiles) and is then published.
//
// A node's frontier is only ever written by one warp per step (the parts of a
// split merge read it, and the last one to finish writes), so updates need no
// locks. All waits are bounded (see GridTeam::sync).
#pragma once

#include "opmos_dev.cuh"
#include "search.cuh"

#include <algorithm>

namespace opmos {
namespace detail {

__device__ __forceinline__ unsigned warp_min(unsigned x) { return __reduce_min_sync(0xffffffffu, x); }

__device__ __forceinline__ unsigned warp_max(unsigned x) { return __reduce_max_sync(0xffffffffu, x); }

__device__ __forceinline__ unsigned long long warp_min64(unsigned long long x) {
  const unsigned hi = warp_min((unsigned)(x >> 32));
  const unsigned lo = warp_min((unsigned)(x >> 32) == hi ? (unsigned)x : 0xffffffffu);
  return (unsigned long long)hi << 32 | lo;
}

// Block-wide exclusive scan of one value per thread; returns the block total.
__device__ inline unsigned block_exclusive_scan(unsigned x, unsigned* s_warp, unsigned& total) {
  const unsigned lane = lane_id(), w = threadIdx.x >> 5, nw = blockDim.x >> 5;
  unsigned incl = x;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    unsigned y = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= (unsigned)o) incl += y;
  }
  if (lane == 31) s_warp[w] = incl;
  __syncthreads();
  if (w == 0) {
    unsigned v = lane < nw ? s_warp[lane] : 0;
    unsigned vi = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      unsigned y = __shfl_up_sync(0xffffffffu, vi, o);
      if (lane >= (unsigned)o) vi += y;
    }
    if (lane < nw) s_warp[lane] = vi - v;
    if (lane == nw - 1) s_warp[32] = vi;
  }
  __syncthreads();
  const unsigned r = s_warp[w] + incl - x;
  total = s_warp[32];
  __syncthreads();
  return r;
}

// Dynamic shared memory of the search kernels: 32 rows of DP words a warp (see
// Search::rows).
__device__ __forceinline__ uint32_t* row_space() {
  extern __shared__ __align__(16) uint32_t s_rows[];
  return s_rows;
}

struct Shared {
  alignas(16) unsigned hist[kNB];  // this block's share of the next OPEN's histogram
  unsigned warp[33];
  unsigned f_min, b1_max;  // see select_window
  unsigned pmax[3];
  // what this block's extraction items found (next bins), added to the global
  // record once a step
  unsigned long long min_key;
  unsigned win_min, win_max, f1lo, f1hi;
  unsigned rec[32];    // the step's record (RecWord)
  PIdx pd;             // the P index as this step sees it
  // this block's counters since the last flush, cnt + (high << 16) each (see flush_counts)
  unsigned cnt[kNStat], high[kNStat];
  unsigned tmax[5];    // this block's longest merge part, merge, extraction item (ns); most
                       // candidates and largest frontier of its split merges
};

// Adds the block's counters to the query's. Every thread calls it, between
// block barriers that separate it from the counting. (Counters in shared memory
// are added to by one lane a work item; 26 of 64 bits in every thread took 52
// registers.) With `full` set only the ones that large are added. A step adds
// less than 2^31 labels or candidates to a block's counters; of what may be more,
// times and comparisons, see Search::count_big.
constexpr unsigned kFlushAt = 1u << 30;  // at a step's end
__device__ __forceinline__ void flush_counts(QCtl* C, Shared& S, unsigned full = 1u) {
  const unsigned i = threadIdx.x - 64u;
  if (i < (unsigned)kNStat && (S.cnt[i] | S.high[i]) >= full) {
    atomicAdd(&C->stats[i], S.cnt[i] + ((unsigned long long)S.high[i] << 16));
    S.cnt[i] = S.high[i] = 0;
  }
}
__device__ __forceinline__ void clear_counts(Shared& S) {
  if (threadIdx.x < kNStat) S.cnt[threadIdx.x] = S.high[threadIdx.x] = 0;
}

// Histogram bin of an OPEN key (F0 << 32 | F1): the key's cell is
// q * kSub + x, q = (F0 - b0) / delta its F[0] bucket and x = (F1 - b1) >> s1
// (at most kSub - 1) its F[1] cell; a bin is 2^s2 consecutive cells, and the
// last bin collects every key beyond. Monotone in lexicographic (F0, F1)
// order for F0 >= b0, so every prefix of bins is a lexicographic prefix of
// OPEN.
struct BinParams {
  uint32_t b0, b1, s1, delta, s2;
};
__device__ __forceinline__ unsigned bin_of(uint64_t key, const BinParams& bp) {
  const uint32_t F0 = (uint32_t)(key >> 32), F1 = (uint32_t)key;
  const uint32_t f = F0 > bp.b0 ? F0 - bp.b0 : 0u;
  const uint64_t q = bp.delta == 1u ? f : f / bp.delta;
  const uint32_t x = F1 > bp.b1 ? min((F1 - bp.b1) >> bp.s1, (unsigned)kSub - 1) : 0u;
  return (unsigned)min((q * kSub + x) >> bp.s2, (uint64_t)(kNB - 1));
}

// Z-order ("Morton") comparison without interleaving: the dimension whose
// values differ in the highest bit decides.
__device__ __forceinline__ bool msb_less(uint32_t a, uint32_t b) { return a < b && a < (a ^ b); }
template <int MD>
__device__ __forceinline__ bool z_less(const uint32_t (&a)[MD], const uint32_t (&b)[MD]) {
  int dim = 0;
  uint32_t x = 0;
#pragma unroll
  for (int k = 0; k < MD; ++k) {
    const uint32_t y = a[k] ^ b[k];
    if (msb_less(x, y)) {
      dim = k;
      x = y;
    }
  }
  return a[dim] < b[dim];
}

// kMany: nodes may have several champions (A.nchamps); a test for it at run time
// made short steps 1% slower.
template <int D, bool kMany = false>
struct Search {
  static constexpr int DP = row_words(D);      // words of a champion's row
  static constexpr int CW = row_words(D + 2);  // words of a candidate's record: costs, arc, parent
  // frontier tiles loaded per round of a scan: fewer at high d (registers)
  static constexpr int kU = D <= 4 ? 4 : (D <= 12 ? 2 : 1);
  static constexpr int kPT = D <= 4 ? 4 : (D <= 8 ? 2 : 1);  // P-index tiles loaded per round
  static constexpr unsigned kMaxScale = 24;  // see next_scale

  const GraphDev& G;
  const QArena& A;
  QCtl* C;
  const QParams& P;
  const OutPool& O;
  Shared& S;
  // fixed for one step
  unsigned cyc = 0;    // step number i
  unsigned psnap = 0;  // P-log prefix every F-against-P test of step i uses
  unsigned lbase = 0;  // labels that existed when step i began
  unsigned fifo_head = 0;  // FIFO: the oldest ring position still in use in step i
  unsigned pscale = 0;     // parts listed in step i are of P.part_work << pscale comparisons
  BinParams bpn{};     // bins of the next OPEN's histogram

  __device__ Search(const GraphDev& g, const QArena& a, QCtl* c, const QParams& p, const OutPool& o,
                    Shared& s)
      : G(g), A(a), C(c), P(p), O(o), S(s) {}

  __device__ __forceinline__ void count(int what, unsigned n) const { atomicAdd(&S.cnt[what], n); }
  // A counter that a step may carry past 32 bits (times, comparisons), at most
  // once a work item: 16 bits go to one word, the others to a second, which a
  // step of less than the barrier's time limit cannot fill; empty_counts comes
  // before the first is full. (Looking whether an addition wrapped made steps 2%
  // longer, adding large values to the query's counter instead 1%.)
  __device__ __forceinline__ void count_big(int what, unsigned long long n) const {
    atomicAdd(&S.cnt[what], (unsigned)n & 0xFFFFu);
    atomicAdd(&S.high[what], (unsigned)(n >> 16));
  }
  static constexpr unsigned kFlushItems = 1024;
  static_assert((unsigned long long)(kGridThreads / 32) * kFlushItems * 0xFFFFu + kFlushAt < 1ull << 32 &&
                    kGridWideThreads <= kGridThreads && kMultiThreads <= kGridThreads, "a step's counts");
  // By one warp beside others that count, every kFlushItems of its work items.
  __device__ void empty_counts() const {
    const unsigned i = lane_id();
    if (i >= (unsigned)kNStat) return;
    const unsigned long long n = atomicExch(&S.cnt[i], 0u) + ((unsigned long long)atomicExch(&S.high[i], 0u) << 16);
    if (n) atomicAdd(&C->stats[i], n);
  }
  // One lane counts for the warp.
  __device__ __forceinline__ void count_lane0(int what, unsigned n) const {
    if (lane_id() == 0 && n) atomicAdd(&S.cnt[what], n);
  }

  // h_k(v) and c_k(e); objectives the query does not use read as 0, which
  // leaves every dominance relation of the used ones unchanged
  __device__ __forceinline__ uint32_t hk(int k, uint32_t v) const {
    return (uint32_t)k < P.qd ? __ldg(P.h + (size_t)k * G.n + v) : 0u;
  }
  __device__ __forceinline__ uint32_t ck(int k, uint32_t e) const {
    return (uint32_t)k < P.qd ? __ldg(G.cost + (size_t)k * G.m + e) : 0u;
  }
  __device__ __forceinline__ uint64_t key_of(const uint32_t (&g)[D], uint32_t v) const {
    return ((uint64_t)(g[0] + hk(0, v)) << 32) | (D > 1 ? g[1 % D] + hk(1 % D, v) : 0u);
  }

  // ---------------- initialisation (Algorithm 1) ----------------
  // Empty frontiers, candidate sets and histograms (the empty sets Algorithm
  // 1 starts from). The team must pass a barrier before init_seed.
  // Whole arrays in turn, 16 bytes a thread: a batch starts a query on one block,
  // and every other query of the iteration waits for it. (A thread
  // that set its node's words in every array wrote 32 sectors an instruction;
  // 400 queries on 128x128 nodes took 41.3 ms instead of 35.0.) Stores that are
  // the first to leave the L2, for most nodes are not reached soon: with plain
  // ones the next query's heuristic found its graph evicted (447x447 road
  // graph: 2.75 ms instead of 2.36).
  template <class Team>
  __device__ void init_zero(const Team& T) {
    const size_t n = G.n + 1ull;  // n real nodes + P
    fill(T, A.fcount, n, 0u);
    fill(T, A.fcap, n, 0u);
    fill(T, A.fbase, 2 * n, 0u);
#pragma unroll
    for (int b = 0; b < 2; ++b) {
      fill(T, A.champ[b], n * A.nchamps * DP, kInf);
      fill(T, A.cs[b].node_head, n << A.lsub, (uint32_t)kNil);
      fill(T, A.cs[b].ncand, n, 0u);
      fill(T, A.cs[b].hflag, n, 0u);
      fill(T, A.cs[b].hcnt, n, 0u);
    }
    fill(T, A.hist, 3u * kNB, 0u);
    fill(T, A.prank, kPSMax, 0u);
  }
  // words words at p (16-byte aligned) set to x
  template <class Team>
  __device__ __forceinline__ static void fill(const Team& T, void* p, size_t words, uint32_t x) {
    for (size_t i = T.tid(); i < words / 4; i += T.nthreads()) __stcs(static_cast<uint4*>(p) + i, make_uint4(x, x, x, x));
    for (size_t i = words / 4 * 4 + T.tid(); i < words; i += T.nthreads()) static_cast<uint32_t*>(p)[i] = x;
  }

  __device__ static void clear_cycle(CycleCtl& K) {
    K.open_count.v = 0;
    K.min_key.v = ~0ull;
    K.win_count.v = 0;
    K.win_min.v = kInf;
    K.win_max.v = 0;
    K.cand_count.v = 0;
    K.touched_count.v = 0;
    K.work_next.v = 0;
    K.part_count.v = 0;
    K.part_scale.v = 0;
    K.f1lo.v = kInf;
    K.f1hi.v = 0;
    K.plen.v = 0;
    K.lbase.v = 0;
    for (int j = 0; j < 5; ++j) K.tmax[j] = 0;
    K.head.v = 0;
  }

  // l_s = (v_s, 0) into OPEN_0 and G_OP(v_s) (Algorithm 1), control reset.
  template <class Team>
  __device__ void init_seed(const Team& T, bool reset_ctl) {
    if (!T.leader()) return;
    if (reset_ctl) {
      C->bar.error = 0;
      C->done = 0;
      C->res_count = C->res_status = 0;
      C->res_off = C->res_path = C->res_total = 0;
      for (int i = 0; i < kNStat; ++i) C->stats[i] = 0;
    }
    C->step = 0;
    C->t_start = globaltimer();
    const uint32_t s = P.start, t = P.goal, tile = P.tile;
#pragma unroll
    for (int k = 0; k < D; ++k) A.lg[(size_t)k * A.label_cap] = 0;
    A.lnode[0] = s;
    A.lparent[0] = kInf;
    A.ledge[0] = kInf;
    A.lpver[0] = 0;
    A.ldead[0] = kAlive;
    const uint32_t fs = (s == t) ? G.n : s;  // start == goal: l_s is the solution
    A.fbase[fs] = 0;
    A.fcap[fs] = tile;
    A.fcount[fs] = 1;
#pragma unroll
    for (int k = 0; k < D; ++k) A.fpool[(size_t)k * tile] = 0;
    A.fpool[(size_t)D * tile] = 0;
    C->f_words.v = (unsigned long long)(D + 1) * tile;
    C->n_labels.v = 1;
    for (int r = 0; r < 3; ++r) {
      clear_cycle(C->cyc[r]);
      C->cyc[r].win_prev.v = kInf;
    }
    for (int b = 0; b < 2; ++b) C->pidx[b] = PIdx{};
    const uint32_t h0 = hk(0, s);
    const uint64_t key = ((uint64_t)h0 << 32) | (D > 1 ? hk(1, s) : 0u);
    CycleCtl& K = C->cyc[0];
    K.lbase.v = 1;
    // the bins of OPEN_0's histogram put l_s in bin 0
    C->bins[0] = BinLimits{h0, (uint32_t)key, 0u, P.delta, 0u};
    if (s != t && h0 != kInf) {  // start == goal: P = {l_s}; h(s) = inf: goal unreachable
      A.okey[0][0] = key;
      A.oid[0][0] = 0;
      K.open_count.v = 1;
      K.min_key.v = key;
      K.f1lo.v = K.f1hi.v = (uint32_t)key;
      A.hist[0] = 1;
    }
    if (s == t) {
#pragma unroll
      for (int k = 0; k < D; ++k) A.plog[(size_t)k * A.plog_cap] = 0;
    }
    C->fifo_tail.v = K.open_count.v;
    C->plog_len.v = (s == t) ? 1u : 0u;
    K.plen.v = C->plog_len.v;
    count(S_INSERTED, 1u);
  }

  // ---------------- window selection (Algorithm 2: NUM_POP lowest labels) ----------------
  // OPEN's histogram in registers: the block's first 8 warps take 512 bins each,
  // lane l the bins 4 (32 j + l) .. + 3 of them in q[j] (16-byte loads, whole
  // lines). Other SMs added to it: read past L1. A step issues the loads before
  // it waits for its record, which says whether they are needed.
  struct Bins {
    uint4 q[4];
  };
  static_assert(kNB == 8 * 512 && kGridThreads >= 256 && kGridWideThreads >= 256 && kMultiThreads >= 256, "Bins");
  __device__ __forceinline__ static Bins load_bins(const unsigned* gh) {
    Bins h;
    const uint4* g4 = reinterpret_cast<const uint4*>(gh) + (threadIdx.x >> 5) * 128 + lane_id();
#pragma unroll
    for (int j = 0; j < 4; ++j) h.q[j] = threadIdx.x < 256u ? __ldcg(g4 + 32 * j) : make_uint4(0u, 0u, 0u, 0u);
    return h;
  }
  // The window is the bins [0, b*], b* the largest bin whose cumulative count is
  // <= W, but at least the first non-empty bin (the overflow bin is never
  // taken). all: OPEN holds at most W entries, so every bin but the last has a
  // cumulative count within W. Every block finds the same b*; bstar() gives it
  // after the next block barrier. One thread holds the bin where the count
  // passes W and one the first entry, so they write without atomics. (Loading
  // the bins after the record, staging them in shared memory, a block scan and
  // atomics by every thread made a step of the 160x160 ship grid 13.5 us
  // instead of 12.5, one of the 32x32 grid 11.5 instead of 10.9.)
  __device__ void select_window(const Bins& h, bool all) {
    if (threadIdx.x == 0) {
      S.b1_max = all ? kNB - 2 : 0;
      S.f_min = kNB;
    }
    if (all) return;
    const unsigned w = threadIdx.x >> 5, lane = lane_id();
    unsigned sum[4], incl[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) sum[j] = incl[j] = h.q[j].x + h.q[j].y + h.q[j].z + h.q[j].w;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1)
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const unsigned y = __shfl_up_sync(0xffffffffu, incl[j], o);
        if (lane >= (unsigned)o) incl[j] += y;
      }
    unsigned tot[4], all4 = 0;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      tot[j] = __shfl_sync(0xffffffffu, incl[j], 31);
      all4 += tot[j];
    }
    if (lane == 0 && w < 8) S.warp[w] = all4;
    __syncthreads();
    if (w >= 8) return;
    unsigned before = 0;
#pragma unroll
    for (unsigned x = 0; x < 8; ++x) before += x < w ? S.warp[x] : 0u;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      unsigned run = before + incl[j] - sum[j];  // the count before the lane's four bins
      const unsigned c[4] = {h.q[j].x, h.q[j].y, h.q[j].z, h.q[j].w};
#pragma unroll
      for (int x = 0; x < 4; ++x) {
        const unsigned bin = w * 512 + j * 128 + lane * 4 + x;
        if (run == 0 && c[x] && bin < kNB - 1) S.f_min = bin;
        if (run <= P.window && (run + c[x] > P.window || bin == kNB - 1)) S.b1_max = bin ? bin - 1 : 0u;
        run += c[x];
      }
      before += tot[j];
    }
  }
  __device__ __forceinline__ unsigned bstar() const {
    return max(S.b1_max, S.f_min == (unsigned)kNB ? 0u : S.f_min);
  }

  // Bins of the histogram of OPEN_{i+1}, from what step i-1 measured (the
  // same on every block). F[0] origin: the smallest F[0] among the entries
  // carried into OPEN_i, window i (whose children merge i creates) and window
  // i-1 (whose children are OPEN_i's other entries). F[1] cells: the F[1]
  // range of the entries carried into OPEN_i in 256 cells. Cells per bin: the
  // bins cover the F[0] buckets from the origin to window i's largest F[0]
  // and three times window i's F[0] extent beyond.
  struct Measured {
    unsigned long long min_key;
    unsigned f1lo, f1hi, wmin, wprev, wmax;
  };
  __device__ BinParams next_bins(const Measured& m) const {
    BinParams b;
    b.b0 = min(min((uint32_t)(m.min_key >> 32), m.wmin), m.wprev);
    if (b.b0 == kInf) b.b0 = 0;
    b.b1 = m.f1lo <= m.f1hi ? m.f1lo : (m.min_key != ~0ull ? (uint32_t)m.min_key : 0u);
    const unsigned span = m.f1lo <= m.f1hi ? m.f1hi - m.f1lo : 0u;
    constexpr int kSubBits = 8;
    static_assert(kSub == 1 << kSubBits, "cells per bucket");
    b.s1 = (unsigned)max(0, 32 - kSubBits - __clz((int)span));  // the smallest with span >> s1 < kSub
    b.delta = P.delta;
    const uint32_t wmin = min(m.wmin, m.wmax);
    uint32_t q0 = m.wmax > b.b0 ? m.wmax - b.b0 : 0u, q1 = m.wmax - wmin;
    if (b.delta != 1u) {
      q0 /= b.delta;
      q1 /= b.delta;
    }
    const uint64_t rows = (uint64_t)q0 + 1 + 3ull * ((uint64_t)q1 + 1);
    b.s2 = 0;
    while (b.s2 < 30 && ((uint64_t)(kNB - 1) << b.s2) >> kSubBits < rows) ++b.s2;
    return b;
  }

  // n-th (0-based) set bit of m, 32 if there is none.
  __device__ __forceinline__ unsigned nth_bit(unsigned m, unsigned n) {
    for (unsigned i = 0; i < n && m; ++i) m &= m - 1;
    return m ? __ffs(m) - 1 : 32u;
  }

  // ---------------- expansion (Algorithm 1) ----------------
  // The candidates of one round of the whole warp (lane's candidate when
  // alive: target v2, parent, arc e, costs g2; fc = fcount[v2]). The two
  // returning atomics a candidate needs -- its record and its rank at the
  // node -- are in flight together.
  __device__ __forceinline__ void add_candidates(const CandSet& cs, CycleCtl& K1, bool alive, uint32_t v2,
                                                 uint32_t parent, uint32_t e, const uint32_t (&g2)[D], unsigned fc) {
    const unsigned am = __ballot_sync(0xffffffffu, alive);
    if (!am) return;
    const unsigned lead = __ffs(am) - 1;
    unsigned c = 0, pos = 0;
    if (lane_id() == lead) c = atomicAdd(&K1.cand_count.v, __popc(am));
    if (alive) pos = atomicAdd(&cs.ncand[v2], 1u);
    c = __shfl_sync(0xffffffffu, c, lead) + __popc(am & lanemask_lt());
    if (alive) {
      uint32_t rec[CW];
#pragma unroll
      for (int k = 0; k < CW; ++k) rec[k] = k < D ? g2[k % D] : k == D ? e : k == D + 1 ? parent : 0u;
      vec_store(cs.crow + (size_t)c * CW, rec);
      cs.cflag[c] = 0u;
      if (pos < A.nslots) {
        cs.cslot[(size_t)v2 * A.nslots + pos] = (int)c;
      } else {  // list (pos - nslots) mod 2^lsub of the node, so all its lists grow evenly
        const unsigned j = (pos - A.nslots) & ((1u << A.lsub) - 1u);
        cs.cnext[c] = atomicExch(&cs.node_head[((size_t)v2 << A.lsub) + j], (int)c);
        count(S_OVF, 1u);
      }
    }
    // Every node is listed once, on its first candidate (one warp merges it). A
    // node with much to compare has its merge split into hflag[v] parts, listed
    // apart; its own item is skipped then.
    const unsigned fm = __ballot_sync(0xffffffffu, alive && pos == 0);
    if (fm) {
      const unsigned l0 = __ffs(fm) - 1;
      unsigned t = 0;
      if (lane_id() == l0) t = atomicAdd(&K1.touched_count.v, __popc(fm));
      t = __shfl_sync(0xffffffffu, t, l0) + __popc(fm & lanemask_lt());
      if (alive && pos == 0) cs.touched[t] = v2;
    }
    // A merge is split once its candidates x what each is compared with (and
    // the 128 or so comparisons' time it costs anyway) exceed P.part_work: looked at as the candidates reach 1, 2, 4, 8, ... A candidate
    // meets the frontier and, if it survives, P: few entries of P with few
    // objectives (the index tiles cover three), most of it with many. At the
    // goal node n there is P alone.
    if (alive && ((pos + 1u) & pos) == 0u) {
      const unsigned want = parts_for(pos + 1u, 128u + pos + (v2 == G.n ? psnap >> kPGoal : fc + (psnap >> kPNode)),
                                      v2 == G.n ? 0u : fc);
      if (want > 1u) split_merge(cs, K1, v2, want);
    }
  }

  // Parts a merge of nc candidates of F comparisons each is split into: a power
  // of two, each part about P.part_work << pscale comparisons or fewer. scan: the
  // frontier entries the candidates meet. However few they are, one warp takes a
  // round of loads for 32 kU entries, 0.5 us, so an entry beyond the first four
  // rounds counts as kScanCands comparisons by itself. (One candidate against 4,000
  // entries took 20 us, and every step of the 256x256 grid, d = 3, had one: W =
  // 1,024 1,111 ms instead of 1,299, W = 256 3,410 instead of 3,980. Counted from
  // the first entry on, graphs of small frontiers split merges for nothing: 110x110,
  // d = 5, W = 256 51.5 ms instead of 46.9.)
  static constexpr unsigned kScanCands = 7, kScanFree = 128 * kU;
  static constexpr unsigned kPNode = D <= 4 ? 5 : (D <= 6 ? 3 : (D <= 8 ? 2 : 0)), kPGoal = D <= 4 ? 2 : (D <= 6 ? 1 : 0);
  __device__ unsigned parts_for(unsigned nc, unsigned F, unsigned scan) const {
    unsigned long long w = (unsigned long long)nc * F;
    if (scan > kScanFree) w += kScanCands * (scan - kScanFree);
    unsigned k = 1;
    while (k < A.kparts && w > ((unsigned long long)P.part_work << pscale) * k) k <<= 1;
    return k;
  }
  // The scale of the parts listed in this step, from the places asked for in the
  // last one (asked) at scale s: doubled until half the list would have held
  // them and the grid's warps had had kPartsPerWarp each, halved when an eighth
  // of that would do.
  // The list is filled first come first served, and a merge that finds it full is
  // left to one warp: with many objectives and a large front every node asks for
  // all its parts (d = 12 route of 1,153 nodes, 16,268 solutions, W = 4,096:
  // 100,000 places of 9,232 a step, one-warp merges of 3.7 ms each step, 310 ms
  // instead of 46).
  // And once the warps have their parts, what a part costs by itself counts:
  // 256x256 grid d=3 at W = 131,072 133 -> 129 ms, second seed 228 -> 208. (Parts of
  // twice the work for every window from 131,072 on, whatever there was to do, made
  // that 134 and 212 ms, and steps of fewer parts longer: 96x96 d=5 10.0 ms instead
  // of 8.6, 128x128 d=3 11.0 instead of 9.8.)
  __device__ __forceinline__ unsigned next_scale(unsigned asked, unsigned s) const {
    if (asked < P.parts_most / 8) return s ? s - 1u : 0u;
    for (; asked > P.parts_most && s < kMaxScale; asked >>= 1) ++s;
    return s;
  }

  // Raises the parts node v's merge is split into to want, and lists the new
  // ones. Candidates arrive together, so the node's count of parts is raised by
  // one atomic maximum whose return tells which parts are new (a protocol in
  // which one candidate listed the node and later ones raised it lost most
  // raises: nodes of 400 candidates were merged in 2 parts, 190 us). The
  // places of the list are claimed first: a count never exceeds the parts
  // listed, and when the list is full the node keeps the parts it has (none:
  // one warp merges it). Places claimed in vain hold kNoPart.
  __device__ void split_merge(const CandSet& cs, CycleCtl& K1, uint32_t v, unsigned want) {
    const unsigned seen = ld_volatile(&cs.hflag[v]);
    if (want <= seen) return;
    const unsigned j = atomicAdd(&K1.part_count.v, want - seen), end = j + (want - seen);
    unsigned old = want;  // nothing new when the list is full
    if (end <= A.xcap) old = atomicMax(&cs.hflag[v], want);
    for (unsigned x = j; x < min(end, A.xcap); ++x)
      cs.xpart[x] = old + (x - j) < want ? make_uint2(v, old + (x - j)) : make_uint2(kNoPart, 0u);
  }

  // A window label as its lane holds it.
  struct Label {
    uint32_t id, v;
    uint32_t e0, e1;  // its out-arcs
    uint32_t g[D];
    unsigned since;   // P-log length at its last F-against-P test
  };
  // Everything extraction needs of label id, in two rounds of loads.
  __device__ __forceinline__ Label load_label(bool want, uint32_t id) const {
    Label l;
    l.id = id;
    l.v = l.e0 = l.e1 = 0;
    l.since = kInf;
#pragma unroll
    for (int k = 0; k < D; ++k) l.g[k] = 0;
    if (want) {
      l.v = A.lnode[id];
#pragma unroll
      for (int k = 0; k < D; ++k) l.g[k] = A.lg[(size_t)k * A.label_cap + id];
      l.since = A.lpver[id];
      l.e0 = __ldg(G.rowptr + l.v);
      l.e1 = __ldg(G.rowptr + l.v + 1);
    }
    return l;
  }
  // Lazy PruneOPEN: F against the goal costs logged since the label's last
  // check (through the P index when that check predates it).
  __device__ __forceinline__ bool still_open(bool want, const Label& l, unsigned long long& pcmp) {
    const unsigned since = warp_min(want ? l.since : kInf);
    bool alive = want;
    if (since < psnap) {
      const PIdx& pd = S.pd;
      uint32_t F[D];
#pragma unroll
      for (int k = 0; k < D; ++k) F[k] = want ? l.g[k] + hk(k, l.v) : 0u;
      if (pd.count && since < pd.mark)
        p_filter(alive, F, pd.mark, psnap, pd.count, 0, pd.ntiles, pd.cur, pcmp);
      else
        p_filter(alive, F, since, psnap, 0, 0, 0, 0, pcmp);
    }
    return alive;
  }

  // Expansion of the window labels the warp's lanes hold (take): 32 / L of
  // them side by side, one per group of L lanes, one round of out-arcs at a
  // time with every lane taking part: g' = g + c(e), dropped when h(v') is
  // infinite (Algorithm 1). A goal label is not expanded (Algorithm 1); it
  // becomes a candidate at the virtual node n. L is P.lanes, or more when the
  // labels leave lane groups idle (one label on a node of degree 24: one round
  // of 32 lanes instead of three of 8).
  __device__ void expand_labels(bool take, const Label& own, const CandSet& cs, CycleCtl& K1) {
    unsigned hits = __ballot_sync(0xffffffffu, take);
    unsigned L = P.lanes;
    while (L < 32u && __popc(hits) * L <= 16u) L <<= 1;
    const unsigned lane = lane_id(), groups = 32u / L, grp = lane / L, gl = lane % L;
    unsigned arcs = 0;
    while (hits) {
      const unsigned src = nth_bit(hits, grp);
      const bool has = src < 32u;
      const unsigned from = has ? src : 0u;
      const uint32_t lid = __shfl_sync(0xffffffffu, own.id, from), v = __shfl_sync(0xffffffffu, own.v, from);
      const uint32_t e0 = __shfl_sync(0xffffffffu, own.e0, from), e1 = __shfl_sync(0xffffffffu, own.e1, from);
      uint32_t g[D];
#pragma unroll
      for (int k = 0; k < D; ++k) g[k] = __shfl_sync(0xffffffffu, own.g[k], from);
      const bool goal = has && v == P.goal;
      const unsigned deg = has ? (goal ? 1u : e1 - e0) : 0u;
      const unsigned rounds = warp_max(deg);
      for (unsigned r = 0; r < rounds; r += L) {
        bool alive = gl + r < deg;
        arcs += __popc(__ballot_sync(0xffffffffu, alive && !goal));
        uint32_t v2 = G.n, par = lid, e = e0 + gl + r, g2[D];
#pragma unroll
        for (int k = 0; k < D; ++k) g2[k] = g[k];
        unsigned fc = 0;
        if (alive) {
          if (goal) {
            par = A.lparent[lid];
            e = A.ledge[lid];
          } else {
            v2 = __ldg(G.col + e);
#pragma unroll
            for (int k = 0; k < D; ++k) g2[k] += ck(k, e);
          }
          fc = A.fcount[v2];
          if (!goal) {
            // dropped when the goal is unreachable from v2, or a champion v2 had
            // when the step began dominates it
            uint32_t ch[D];
            champion(A.champ[cyc & 1u], v2, ch);
            alive = hk(0, v2) != kInf && !weakly_le<D>(ch, g2);
            if (kMany && A.nchamps > 1u && alive) {
#pragma unroll
              for (unsigned q = 1; q < kChamps; ++q) {
                champion(A.champ[cyc & 1u], plane(q) + v2, ch);
                alive = alive && !weakly_le<D>(ch, g2);
              }
            }
          }
        }
        add_candidates(cs, K1, alive, v2, par, e, g2, fc);
      }
      for (unsigned r = 0; r < groups && hits; ++r) hits &= hits - 1;
    }
    count_lane0(S_CAND, arcs);
  }

  // ---------------- extraction of window i+1 from OPEN_i ----------------
  // Entries one work item (one warp) takes: as many labels as one round of
  // the warp's lanes expands (an item of 32 labels is eight rounds of
  // dependent loads and atomics one after the other: 10 us at 8 lanes a label
  // and degree 8, 45 us at degree 24, while most of the warps had no item),
  // more only when there are more entries than warps hold then.
  // Measured: longest extraction item of a step 10 -> 3 us and step 22 -> 13 us
  // (97x89 ship grid, d = 3), 17 -> 2.4 us and 34 -> 17 us (241-node route, d = 8).
  __device__ __forceinline__ unsigned item_entries(unsigned n, unsigned nwarps) const {
    unsigned per = 32u;
    while (per > 1u && (32u / per) < G.maxdeg) per >>= 1;
    return min(kChunk, max(per, (n + nwarps - 1) / nwarps));
  }

  // One warp, the `per` entries chunk, chunk + nchunks, chunk + 2 nchunks,
  // ... (a merge appends a node's new labels side by side and they tend to
  // fall in the same window, so strided chunks spread the window's labels
  // over the work items): dead entries are dropped (lazy OPEN delete), window
  // entries whose F a logged solution weakly dominates are dropped (lazy
  // PruneOPEN), the other window entries are taken and expanded at once by
  // lane groups; every other entry is carried to OPEN_{i+1} and counted in
  // its histogram.
  __device__ void extract_chunk(unsigned chunk, unsigned n_in, unsigned per, const BinParams& bp, CycleCtl& K1) {
    const unsigned cur = cyc & 1u, nxt = cur ^ 1u;
    const CandSet& cs = A.cs[nxt];
    const unsigned lane = lane_id();
    const unsigned nchunks = (n_in + per - 1) / per;
    const unsigned i = chunk + lane * nchunks;
    const bool valid = lane < per && i < n_in;
    uint64_t key = 0;
    uint32_t id = 0;
    unsigned dead = 0;
    bool want = false, keep = false;
    if (valid) {
      key = A.okey[cur][i];
      id = A.oid[cur][i];
      dead = A.ldead[id];
      want = bin_of(key, bp) <= bstar();
    }
    const Label own = load_label(want, id);
    const bool gone = valid && dead < cyc;
    if (gone)
      want = false;
    else
      keep = valid && !want;
    unsigned long long pcmp = 0;
    bool take = still_open(want, own, pcmp);
    if (lane_id() == 0 && pcmp) count_big(S_PCMP, pcmp);
    count_lane0(S_OSCAN, __popc(__ballot_sync(0xffffffffu, valid)));
    count_lane0(S_DEAD, __popc(__ballot_sync(0xffffffffu, gone)));
    count_lane0(S_GOALPRUNED, __popc(__ballot_sync(0xffffffffu, want && !take)));
    if (n_in > A.win_cap && take) {  // else the window cannot be full
      if (agg_inc(&K1.win_count.v) >= A.win_cap) {
        take = false;
        keep = true;  // window full: stays in OPEN for the next step
      }
    }
    // places in the next OPEN are claimed before the expansion and used
    // after it
    const unsigned km = __ballot_sync(0xffffffffu, keep);
    unsigned ob = 0;
    if (km && lane == 0) ob = atomicAdd(&K1.open_count.v, __popc(km));
    const unsigned tm = __ballot_sync(0xffffffffu, take);
    if (tm) {
      count_lane0(S_EXTRACTED, __popc(tm));
      const unsigned wmin = warp_min(take ? (unsigned)(key >> 32) : kInf);
      const unsigned wmax = warp_max(take ? (unsigned)(key >> 32) : 0u);
      if (lane == 0) {
        atomicMin(&S.win_min, wmin);
        atomicMax(&S.win_max, wmax);
      }
      expand_labels(take, own, cs, K1);
    }
    if (km) {
      const unsigned o = __shfl_sync(0xffffffffu, ob, 0) + __popc(km & lanemask_lt());
      bool inbins = false;
      if (keep) {
        if (o < A.open_cap) {
          A.okey[nxt][o] = key;
          A.oid[nxt][o] = id;
          const unsigned b = bin_of(key, bpn);
          atomicAdd(&S.hist[b], 1u);
          inbins = b < (unsigned)kNB - 1;
        } else {
          set_error(C, OPMOS_ERR_CAPACITY);
        }
      }
      count_lane0(S_OKEEP, __popc(km));
      const unsigned long long kmin = warp_min64(keep ? key : ~0ull);
      const unsigned f1lo = warp_min(inbins ? (uint32_t)key : kInf), f1hi = warp_max(inbins ? (uint32_t)key : 0u);
      if (lane == 0) {
        atomicMin(&S.min_key, kmin);
        if (f1lo != kInf) {
          atomicMin(&S.f1lo, f1lo);
          atomicMax(&S.f1hi, f1hi);
        }
      }
    }
  }

  // FIFO order (OPMOS_FLAG_FIFO): one warp takes the ring positions
  // [p0, p1) of window i+1 (at most 32) -- the oldest entries -- and expands
  // every one that is alive and not dominated by a logged solution on F.
  // Nothing is carried: the rest of the ring stays where it is.
  __device__ void extract_fifo(unsigned p0, unsigned p1, CycleCtl& K1) {
    const CandSet& cs = A.cs[(cyc & 1u) ^ 1u];
    const unsigned pos = p0 + lane_id();
    uint32_t id = 0;
    unsigned dead = 0;
    const bool valid = pos < p1;
    if (valid) {
      id = A.oid[0][pos % A.open_cap];
      dead = A.ldead[id];
    }
    const Label own = load_label(valid, id);
    const bool want = valid && dead >= cyc;
    unsigned long long pcmp = 0;
    const bool take = still_open(want, own, pcmp);
    if (lane_id() == 0 && pcmp) count_big(S_PCMP, pcmp);
    count_lane0(S_OSCAN, __popc(__ballot_sync(0xffffffffu, valid)));
    count_lane0(S_DEAD, __popc(__ballot_sync(0xffffffffu, valid && !want)));
    count_lane0(S_GOALPRUNED, __popc(__ballot_sync(0xffffffffu, want && !take)));
    count_lane0(S_EXTRACTED, __popc(__ballot_sync(0xffffffffu, take)));
    expand_labels(take, own, cs, K1);
  }

  // ---------------- rows: up to 32 vectors every lane of the warp reads ----------------
  // A warp keeps the vectors it tests against many others (candidates with
  // their arcs, or their F) in shared memory, one row of RP words each: a lane
  // holds one entry of the other side, and the row all lanes read comes in
  // RP / 4 loads instead of D shuffles.
  static constexpr int RP = row_words(D + 1);
  __device__ __forceinline__ uint32_t* rows() const { return row_space() + (threadIdx.x & ~31u) * RP; }
  __device__ __forceinline__ void put_row(const uint32_t (&x)[D], uint32_t edge = 0) const {
    uint32_t r[RP];
#pragma unroll
    for (int k = 0; k < RP; ++k) r[k] = k < D ? x[k % D] : k == D ? edge : 0u;
    __syncwarp();  // earlier readers are done
    vec_store(rows() + lane_id() * RP, r);
    __syncwarp();
  }
  __device__ __forceinline__ void get_row(unsigned j, uint32_t (&x)[D]) const {
    uint32_t r[RP];
    vec_load(rows() + j * RP, r);
#pragma unroll
    for (int k = 0; k < D; ++k) x[k] = r[k];
  }
  __device__ __forceinline__ void get_row(unsigned j, uint32_t (&x)[D], uint32_t& edge) const {
    uint32_t r[RP];
    vec_load(rows() + j * RP, r);
#pragma unroll
    for (int k = 0; k < D; ++k) x[k] = r[k];
    edge = r[D];
  }
  // Rows of W words, 16 bytes at a time (W = 1 or a multiple of 2).
  template <int W>
  __device__ __forceinline__ static void vec_load(const uint32_t* r, uint32_t (&x)[W]) {
    if constexpr (W % 4 == 0) {
#pragma unroll
      for (int q = 0; q < W / 4; ++q) {
        const uint4 v = reinterpret_cast<const uint4*>(r)[q];
        x[4 * q] = v.x;
        x[4 * q + 1] = v.y;
        x[4 * q + 2] = v.z;
        x[4 * q + 3] = v.w;
      }
    } else if constexpr (W % 2 == 0) {
#pragma unroll
      for (int q = 0; q < W / 2; ++q) {
        const uint2 v = reinterpret_cast<const uint2*>(r)[q];
        x[2 * q] = v.x;
        x[2 * q + 1] = v.y;
      }
    } else {
#pragma unroll
      for (int k = 0; k < W; ++k) x[k] = r[k];
    }
  }
  template <int W>
  __device__ __forceinline__ static void vec_store(uint32_t* r, const uint32_t (&x)[W]) {
    if constexpr (W % 4 == 0) {
#pragma unroll
      for (int q = 0; q < W / 4; ++q)
        reinterpret_cast<uint4*>(r)[q] = make_uint4(x[4 * q], x[4 * q + 1], x[4 * q + 2], x[4 * q + 3]);
    } else {
#pragma unroll
      for (int k = 0; k < W; ++k) r[k] = x[k];
    }
  }

  // F against tiles [tlo, thi) of the P index (pcount entries) + the logged goal
  // costs log[t0, t1): clears alive for candidates a solution weakly dominates
  // (Algorithm 1). Every lane of the warp calls it (its rows are overwritten);
  // pcmp counts vector comparisons (lane 0's count is the warp's).
  //
  // The chain is what it costs (a handful of candidates, tiles in L2): the log's
  // tail and the tile minima are loaded together, every candidate's passing
  // tiles are found first (lane j keeps candidate j's), and then kPT of those
  // tiles are loaded at a time, whichever candidates they belong to. (Scanning
  // the entries outright with more than six objectives, where most tiles of a
  // small front pass, was five times the comparisons on a large one: 7x7 grid,
  // d = 16, 17,539 solutions 101 ms instead of 80; 6x8x24 route, d = 12, 16,268
  // solutions 65 instead of 52, 1,381 solutions 3.7 instead of 3.6.)
  __device__ void p_filter(bool& alive, const uint32_t (&F)[D], unsigned t0, unsigned t1, unsigned pcount,
                           unsigned tlo, unsigned thi, unsigned pbuf, unsigned long long& pcmp) {
    const unsigned lane = lane_id();
    unsigned cnt = 0;
    unsigned am = __ballot_sync(0xffffffffu, alive);
    if (!am || (t0 >= t1 && tlo >= thi)) return;
    const uint32_t* ps = A.ps[pbuf];
    const uint32_t* pst = A.pst[pbuf];
    const size_t tcap = A.plog_cap / 32 + 1;
    uint32_t tm[D];  // tile minima, one tile a lane
#pragma unroll
    for (int k = 0; k < D; ++k) tm[k] = tlo + lane < thi ? pst[(size_t)k * tcap + tlo + lane] : kInf;
    put_row(F);
    p_scan(am, A.plog, t0, t1, cnt);
    for (unsigned tg = tlo; tg < thi && am; tg += 32) {
      if (tg != tlo) {
#pragma unroll
        for (int k = 0; k < D; ++k) tm[k] = tg + lane < thi ? pst[(size_t)k * tcap + tg + lane] : kInf;
      }
      cnt += __popc(am) * min(32u, thi - tg);
      unsigned pm = 0;  // lane j: the tiles candidate j still has to be tested against
      for (unsigned todo = am; todo;) {
        unsigned j[2];
        next_two(todo, j);
#pragma unroll
        for (int x = 0; x < 2; ++x) {
          uint32_t Fj[D];
          get_row(j[x], Fj);
          const unsigned m = __ballot_sync(0xffffffffu, tg + lane < thi && weakly_le<D>(tm, Fj));
          if (lane == j[x]) pm = m;
        }
      }
      // (candidate, tile) pairs, one tile of up to kPT candidates a round -- or
      // several tiles of one candidate when fewer are left
      for (;;) {
        unsigned open = __ballot_sync(0xffffffffu, pm != 0u);
        if (!open) break;
        unsigned jq[kPT], eq[kPT];
        unsigned turn = open;
#pragma unroll
        for (int q = 0; q < kPT; ++q) {
          if (!turn) turn = open;
          jq[q] = 32u;
          eq[q] = pcount;
          if (open) {
            jq[q] = __ffs(turn) - 1;
            turn &= turn - 1;
            const unsigned m = __shfl_sync(0xffffffffu, pm, jq[q]);
            eq[q] = (tg + __ffs(m) - 1) * 32 + lane;
            if (lane == jq[q]) pm &= pm - 1;
            if (!(m & (m - 1))) {  // that was its last tile
              open &= ~(1u << jq[q]);
              turn &= ~(1u << jq[q]);
            }
            cnt += 32;
          }
        }
        uint32_t p[kPT][D];
#pragma unroll
        for (int q = 0; q < kPT; ++q)
#pragma unroll
          for (int k = 0; k < D; ++k) p[q][k] = eq[q] < pcount ? ps[(size_t)k * A.plog_cap + eq[q]] : kInf;
        unsigned gone = 0;
#pragma unroll
        for (int q = 0; q < kPT; ++q) {
          if (jq[q] > 31u) break;
          uint32_t Fj[D];
          get_row(jq[q], Fj);
          if (eq[q] < pcount && weakly_le<D>(p[q], Fj)) gone |= 1u << jq[q];
        }
        gone = __reduce_or_sync(0xffffffffu, gone);
        am &= ~gone;
        if ((gone >> lane) & 1u) pm = 0;
      }
    }
    alive = (am >> lane) & 1u;
    if (lane == 0) pcmp += cnt;
  }

  // The rows of am against entries [t0, t1) of a list of goal costs, all of them.
  __device__ __forceinline__ void p_scan(unsigned& am, const uint32_t* list, unsigned t0, unsigned t1,
                                         unsigned& cnt) const {
    const unsigned lane = lane_id();
    for (unsigned r0 = t0; r0 < t1 && am; r0 += 32 * kU) {
      uint32_t pt[kU][D];
#pragma unroll
      for (int u = 0; u < kU; ++u) {
        const unsigned jj = r0 + u * 32 + lane;
#pragma unroll
        for (int k = 0; k < D; ++k) pt[u][k] = jj < t1 ? list[(size_t)k * A.plog_cap + jj] : kInf;
      }
      cnt += __popc(am) * min(32u * kU, t1 - r0);
      const int nu = (int)min((unsigned)kU, (t1 - r0 + 31) / 32);
      for (unsigned todo = am; todo;) {
        unsigned j[2];
        next_two(todo, j);
        uint32_t Fj[2][D];
        bool wd[2] = {false, false};
#pragma unroll
        for (int x = 0; x < 2; ++x) {
          get_row(j[x], Fj[x]);
#pragma unroll
          for (int u = 0; u < kU; ++u) {
            if (u >= nu) break;
            wd[x] |= r0 + u * 32 + lane < t1 && weakly_le<D>(pt[u], Fj[x]);
          }
        }
        am &= ~__reduce_or_sync(0xffffffffu, (wd[0] ? 1u << j[0] : 0u) | (wd[1] ? 1u << j[1] : 0u));
      }
    }
  }

  // The next two set bits of todo, taken out of it (the last one twice).
  __device__ __forceinline__ static void next_two(unsigned& todo, unsigned (&j)[2]) {
    j[0] = j[1] = __ffs(todo) - 1;
    todo &= todo - 1;
    if (todo) {
      j[1] = __ffs(todo) - 1;
      todo &= todo - 1;
    }
  }

  // ---------------- merge of window i's candidates (Algorithm 1: frontier checks, goal branch) ----------------
  // Up to 32 candidates of one node, lane j holding candidate j (and its row).
  struct Batch {
    uint32_t c[D];
    uint32_t edge, par;
    bool alive;
  };
  // kU tiles of 32 frontier entries, lane l holding entry l of each.
  struct Round {
    uint32_t m[kU][D];
    uint32_t mid[kU];
  };
  __device__ __forceinline__ Round load_round(unsigned r0, unsigned hi, uint64_t fb, unsigned cap, bool ids) const {
    Round t;
#pragma unroll
    for (int u = 0; u < kU; ++u) {
      const unsigned i = r0 + u * 32 + lane_id();
      const bool vm = i < hi;
#pragma unroll
      for (int k = 0; k < D; ++k) t.m[u][k] = vm ? A.fpool[fb + (size_t)k * cap + i] : kInf;
      t.mid[u] = ids && vm ? A.fpool[fb + (size_t)D * cap + i] : 0u;
    }
    return t;
  }
  // The lanes' candidates (kNil: none).
  __device__ __forceinline__ Batch load_batch(const CandSet& cs, int mine) const {
    Batch b;
    b.alive = mine != kNil;
    uint32_t rec[CW];
#pragma unroll
    for (int k = 0; k < CW; ++k) rec[k] = kInf;
    if (b.alive) vec_load(cs.crow + (size_t)mine * CW, rec);
#pragma unroll
    for (int k = 0; k < D; ++k) b.c[k] = rec[k];
    b.edge = rec[D];
    b.par = rec[D + 1];
    return b;
  }
  // A batch against itself: a candidate another one strictly dominates, or that
  // equals one with a smaller arc id, is dropped (a dropped one drops nothing
  // more: what it dominates is dominated by what dropped it). Leaves the batch
  // in the rows.
  __device__ __forceinline__ void resolve_batch(Batch& b) const {
    const unsigned lane = lane_id();
    put_row(b.c, b.edge);
    unsigned am = __ballot_sync(0xffffffffu, b.alive);
    for (unsigned todo = am; todo;) {
      unsigned j[2];
      next_two(todo, j);
      uint32_t cj[2][D], ej[2];
      bool dies = false;
#pragma unroll
      for (int x = 0; x < 2; ++x) {
        get_row(j[x], cj[x], ej[x]);
        if (lane != j[x] && weakly_le<D>(cj[x], b.c))
          dies |= !weakly_le<D>(b.c, cj[x]) || ej[x] < b.edge || (ej[x] == b.edge && j[x] < lane);
      }
      const unsigned gone = __ballot_sync(0xffffffffu, dies);
      am &= ~gone;
      todo &= ~gone;
    }
    b.alive = (am >> lane) & 1u;
  }

  // A label created in this step and pruned in it is taken back out of the
  // next OPEN's histogram (its OPEN entry is dropped at the next extraction).
  __device__ __forceinline__ void unhist(const uint32_t (&g)[D], uint32_t v, uint32_t id) {
    if (id >= lbase && v != G.n) atomicSub(&S.hist[bin_of(key_of(g, v), bpn)], 1u);
  }

  // The batch against frontier entries [lo, hi) at fb, cap: candidates an entry
  // weakly dominates die, entries a candidate strictly dominates are pruned
  // (label dead from the next step on). WRITE: the entries that stay are moved together from lo on, and the
  // end of them is returned; an entry created in this step (id >= lbase) that
  // a candidate equals takes its parent and arc if its arc id is smaller, so
  // the path kept for a cost does not depend on the order in which candidates
  // arrived. Otherwise the entries are only read (several warps share the
  // frontier), and pruned tells whether one was marked.
  //
  // kU tiles of 32 entries are loaded per round (t: the first round, loaded by
  // the caller beside the candidates) and every live candidate's row is read
  // once a round: 2 D compares a pair and a vote for two candidates.
  template <bool WRITE>
  __device__ unsigned scan_frontier(uint32_t v, Batch& b, unsigned lo, unsigned hi, uint64_t fb, unsigned cap,
                                    Round& t, bool& pruned_any, unsigned long long& fcmp) {
    constexpr int U = kU;
    const unsigned lane = lane_id();
    unsigned am = __ballot_sync(0xffffffffu, b.alive), out = lo;
    const uint32_t(&m)[U][D] = t.m;
    const uint32_t(&mid)[U] = t.mid;
    for (unsigned r0 = lo; r0 < hi; r0 += 32 * U) {
      if (!am && (!WRITE || out == r0)) {  // nothing left to test and nothing moved: the rest stays in place
        out = hi;
        break;
      }
      if (r0 != lo) t = load_round(r0, hi, fb, cap, WRITE);  // (the caller has loaded the first)
      const int nu = (int)min((unsigned)U, (hi - r0 + 31) / 32);  // tiles of the round that hold entries
      bool pr[U];
#pragma unroll
      for (int u = 0; u < U; ++u) pr[u] = false;
      fcmp += __popc(am) * min(32u * U, hi - r0);
      // two candidates an iteration (the last one twice when they are odd): a
      // warp alone waits for its own chain of compares and votes
      for (unsigned todo = am; todo;) {
        unsigned j[2];
        next_two(todo, j);
        uint32_t cj[2][D];
        get_row(j[0], cj[0]);
        get_row(j[1], cj[1]);
        bool dies[2] = {false, false}, same = false;
#pragma unroll
        for (int u = 0; u < U; ++u) {
          if (u >= nu) break;
          const bool vm = r0 + u * 32 + lane < hi;
#pragma unroll
          for (int x = 0; x < 2; ++x) {
            const bool le_mc = vm && weakly_le<D>(m[u], cj[x]);
            const bool le_cm = vm && weakly_le<D>(cj[x], m[u]);
            dies[x] |= le_mc;
            pr[u] |= le_cm && !le_mc;
            if (WRITE) same |= le_cm && le_mc && mid[u] >= lbase;
          }
        }
        const unsigned gone = __reduce_or_sync(0xffffffffu, (dies[0] ? 1u << j[0] : 0u) | (dies[1] ? 1u << j[1] : 0u));
        if (!gone) continue;
        am &= ~gone;
        if (WRITE && __any_sync(0xffffffffu, same)) {
#pragma unroll
          for (int x = 0; x < 2; ++x) {
            const uint32_t ej = __shfl_sync(0xffffffffu, b.edge, j[x]), pj = __shfl_sync(0xffffffffu, b.par, j[x]);
#pragma unroll
            for (int u = 0; u < U; ++u) {
              const bool eq = r0 + u * 32 + lane < hi && mid[u] >= lbase && weakly_le<D>(m[u], cj[x]) &&
                              weakly_le<D>(cj[x], m[u]);
              if (eq && ej < A.ledge[mid[u]]) {
                A.ledge[mid[u]] = ej;
                A.lparent[mid[u]] = pj;
              }
            }
          }
        }
      }
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const unsigned i = r0 + u * 32 + lane;
        if (pr[u]) {
          const uint32_t id = WRITE ? mid[u] : A.fpool[fb + (size_t)D * cap + i];
          A.ldead[id] = cyc;
          if (WRITE) unhist(m[u], v, id);
          count(S_PRUNED, 1u);
          pruned_any = true;
        }
      }
      if (WRITE) {
#pragma unroll
        for (int u = 0; u < U; ++u) {
          const unsigned i = r0 + u * 32 + lane;
          const bool keep = i < hi && !pr[u];
          const unsigned km = __ballot_sync(0xffffffffu, keep);
          const unsigned pos = out + __popc(km & lanemask_lt());
          // (every lane's entries of the round are in registers: a tile's
          // places may overwrite entries of its round only)
          if (keep && pos != i) {
#pragma unroll
            for (int k = 0; k < D; ++k) A.fpool[fb + (size_t)k * cap + pos] = m[u][k];
            A.fpool[fb + (size_t)D * cap + pos] = mid[u];
          }
          out += __popc(km);
        }
      }
    }
    b.alive = (am >> lane) & 1u;
    __syncwarp();
    return out;
  }

  // F against share x of n of P (Algorithm 1) for the batch: the index's tiles
  // and the log behind it, up to t1. hv: the node's heuristic, 0 at the goal
  // node n.
  __device__ __forceinline__ void batch_ptest(const uint32_t (&hv)[D], Batch& b, unsigned t1, unsigned x, unsigned n,
                                              unsigned long long& pcmp) {
    if (!__any_sync(0xffffffffu, b.alive)) return;
    const PIdx& pd = S.pd;
    uint32_t F[D];
#pragma unroll
    for (int k = 0; k < D; ++k) F[k] = b.alive ? b.c[k] + hv[k] : kInf;
    const unsigned t0 = pd.count ? pd.mark : 0u, tiles = pd.count ? pd.ntiles : 0u, tail = t1 - min(t0, t1);
    p_filter(b.alive, F, t0 + (unsigned)((uint64_t)tail * x / n), t0 + (unsigned)((uint64_t)tail * (x + 1) / n), pd.count,
             (unsigned)((uint64_t)tiles * x / n), (unsigned)((uint64_t)tiles * (x + 1) / n), pd.cur, pcmp);
  }

  // A node's champion is the accepted label of the smallest cost sum; further ones
  // (A.nchamps) are those of sums in which one objective weighs four times the
  // others, then a quarter. A candidate one of them weakly dominates would be
  // dropped by the merge (a label once accepted is in the frontier or was pruned by
  // one that dominates whatever it dominates), so the expansion drops it at once: a third to two thirds of all candidates
  // (two thirds to three quarters are dominated by some label). The rows are a
  // pair by step parity: step i reads rows i & 1 and writes the others, so a row
  // is never read half written; an older champion is as valid as a new one.
  __device__ __forceinline__ static void champion(const uint32_t* rows, size_t v, uint32_t (&x)[D]) {
    uint32_t r[DP];
    vec_load(rows + v * DP, r);
#pragma unroll
    for (int k = 0; k < D; ++k) x[k] = r[k];
  }
  // Champion q of node v is row plane(q) + v.
  __device__ __forceinline__ size_t plane(unsigned q) const { return (size_t)q * (G.n + 1ull); }
  // The cost sum champion Q is the smallest of.
  template <unsigned Q>
  __device__ __forceinline__ static uint32_t cost_sum(const uint32_t (&x)[D]) {
    unsigned long long sum = 0;
#pragma unroll
    for (int k = 0; k < D; ++k) sum += x[k];
    if constexpr (Q > 0) {
      constexpr unsigned k = (Q - 1) % D;
      sum = Q <= (unsigned)D ? sum + 3ull * x[k] : 4ull * sum - 3ull * x[k];
    }
    return (uint32_t)min(sum, (unsigned long long)kInf);
  }
  template <unsigned Q>
  __device__ __forceinline__ void update_champion(uint32_t v, const Batch& b) {
    uint32_t c0[D], c1[D];
    const size_t row = plane(Q) + v;
    uint32_t* const next = A.champ[(cyc & 1u) ^ 1u] + row * DP;
    champion(A.champ[cyc & 1u], row, c0);
    champion(A.champ[(cyc & 1u) ^ 1u], row, c1);
    const uint32_t mine = b.alive ? cost_sum<Q>(b.c) : kInf;
    const uint32_t best = warp_min(mine);
    const unsigned who = __ballot_sync(0xffffffffu, b.alive && mine == best);
    const uint32_t s0 = cost_sum<Q>(c0), s1 = cost_sum<Q>(c1);
    __syncwarp();  // the rows are read before one is written
    if (best < min(s0, s1)) {
      if (lane_id() == (unsigned)__ffs(who) - 1) {
#pragma unroll
        for (int k = 0; k < D; ++k) next[k] = b.c[k];
      }
    } else if (s0 < s1 && lane_id() == 0) {
#pragma unroll
      for (int k = 0; k < D; ++k) next[k] = c0[k];
    }
  }

  // The batch's survivors become labels and join alpha(v) -- `out` live entries
  // at fb, cap, moved to a block of twice the size when full -- and the next
  // OPEN, or at the goal node n the P log. Returns alpha(v)'s new size. The
  // warp is the only one at the node. A candidate P rejected has still pruned
  // the frontier entries it dominates (as in Algorithm 1, where Prune precedes
  // the P test).
  __device__ unsigned insert_batch(uint32_t v, const uint32_t (&hv)[D], const Batch& b, unsigned out, uint64_t& fb,
                                   unsigned& cap, CycleCtl& K1, unsigned nc) {
    const unsigned lane = lane_id();
    const bool is_goal = v == G.n, fifo = (P.flags & OPMOS_FLAG_FIFO) != 0;
    const unsigned smask = __ballot_sync(0xffffffffu, b.alive);
    const unsigned ns = __popc(smask);
    if (!ns) return out;
    // label ids and places in the next OPEN, claimed side by side
    unsigned lb = 0, ob = 0, plen = 0;
    if (lane == 0) {
      lb = atomicAdd(&C->n_labels.v, ns);
      if (!is_goal) ob = atomicAdd(fifo ? &C->fifo_tail.v : &K1.open_count.v, ns);
      if (is_goal) plen = ld_volatile(&C->plog_len.v);  // this warp is the log's only writer
    }
    if (!is_goal) {
      update_champion<0>(v, b);
      if (kMany && A.nchamps > 1u && nc >= kChampCands) {
        static_assert(kChamps == 4, "one call each");
        update_champion<1>(v, b);
        update_champion<2>(v, b);
        update_champion<3>(v, b);
      }
    }
    lb = __shfl_sync(0xffffffffu, lb, 0);
    ob = __shfl_sync(0xffffffffu, ob, 0);
    plen = __shfl_sync(0xffffffffu, plen, 0);
    if (lb + ns > A.label_cap || lb + ns > P.label_budget) {
      if (lane == 0) set_error(C, (lb + ns > A.label_cap) ? OPMOS_ERR_CAPACITY : OPMOS_ERR_BUDGET);
      return out;
    }
    if (is_goal ? plen + ns > A.plog_cap : (fifo ? ob - fifo_head : ob) + ns > A.open_cap) {
      if (lane == 0) set_error(C, OPMOS_ERR_CAPACITY);
      return out;
    }
    if (lane == 0) atomicMax(&K1.lbase.v, lb + ns);
    const unsigned need = out + ns;
    if (need > cap) {
      // grow: new block of twice the size, copy the live entries
      const unsigned tile = P.tile;
      unsigned ncap = max(2u * need, tile);
      ncap = (ncap + tile - 1) / tile * tile;
      unsigned long long nb0 = 0;
      if (lane == 0) nb0 = atomicAdd(&C->f_words.v, (unsigned long long)(D + 1) * ncap);
      nb0 = __shfl_sync(0xffffffffu, nb0, 0);
      if (nb0 + (unsigned long long)(D + 1) * ncap > A.fpool_words) {
        if (lane == 0) set_error(C, OPMOS_ERR_CAPACITY);
        return out;
      }
      for (unsigned i = lane; i < out; i += 32) {
#pragma unroll
        for (int k = 0; k <= D; ++k) A.fpool[nb0 + (size_t)k * ncap + i] = A.fpool[fb + (size_t)k * cap + i];
      }
      fb = nb0;
      cap = ncap;
      if (lane == 0) {
        A.fbase[v] = fb;
        A.fcap[v] = cap;
      }
    }
    if (b.alive) {
      const unsigned r = __popc(smask & lanemask_lt());
      const unsigned id = lb + r;
#pragma unroll
      for (int k = 0; k < D; ++k) A.lg[(size_t)k * A.label_cap + id] = b.c[k];
      A.lnode[id] = is_goal ? P.goal : v;
      A.lparent[id] = b.par;
      A.ledge[id] = b.edge;
      A.lpver[id] = psnap;
      A.ldead[id] = kAlive;
#pragma unroll
      for (int k = 0; k < D; ++k) A.fpool[fb + (size_t)k * cap + out + r] = b.c[k];
      A.fpool[fb + (size_t)D * cap + out + r] = id;
      if (is_goal) {
#pragma unroll
        for (int k = 0; k < D; ++k) A.plog[(size_t)k * A.plog_cap + plen + r] = b.c[k];
      } else if (fifo) {
        // the ring's tail (positions [head, tail) of this step are never written over)
        A.oid[0][(ob + r) % A.open_cap] = id;
      } else {
        // the array of step i+1, counted in its histogram
        const uint64_t key = ((uint64_t)(b.c[0] + hv[0]) << 32) | (D > 1 ? b.c[1 % D] + hv[1 % D] : 0u);
        const unsigned nxt = (cyc & 1u) ^ 1u;
        A.okey[nxt][ob + r] = key;
        A.oid[nxt][ob + r] = id;
        atomicAdd(&S.hist[bin_of(key, bpn)], 1u);
      }
    }
    __syncwarp();
    if (lane == 0) {
      if (is_goal) {  // the log entries are written before they are published
        __threadfence();
        *reinterpret_cast<volatile unsigned*>(&C->plog_len.v) = plen + ns;
        atomicMax(&K1.plen.v, plen + ns);
      } else if (fifo) {
        atomicMax(&K1.open_count.v, ob + ns);
      }
      count(S_INSERTED, ns);
    }
    return need;
  }

  // A node's candidates of one step in groups of up to 32: first the slots, 32
  // at a time, then 32 / L rounds of its L = 2^lsub lists at a time: lane x
  // walks list x mod L and holds its candidate of round x / L of the group.
  struct Groups {
    uint32_t v;
    unsigned in_slots, nslot_groups;
    int lcur;        // the lane's position in its list
    unsigned lnext;  // the list group lcur stands at
  };
  __device__ __forceinline__ unsigned ngroups(unsigned nc) const {
    const unsigned ns = min(nc, A.nslots);
    return (ns + 31) / 32 + (nc - ns + 31) / 32;
  }
  __device__ __forceinline__ int list_step(const CandSet& cs, int c, unsigned n) const {
    for (; n && c != kNil; --n) c = cs.cnext[c];
    return c;
  }
  __device__ __forceinline__ Groups open_groups(const CandSet& cs, uint32_t v, unsigned nc) const {
    Groups q;
    q.v = v;
    q.in_slots = min(nc, A.nslots);
    q.nslot_groups = (q.in_slots + 31) / 32;
    q.lnext = 0;
    q.lcur = kNil;
    if (nc > q.in_slots) {
      const unsigned list = lane_id() & ((1u << A.lsub) - 1u);
      q.lcur = list_step(cs, cs.node_head[((size_t)v << A.lsub) + list], lane_id() >> A.lsub);
    }
    return q;
  }
  // The lane's candidate of group g (kNil: none); g must not decrease.
  __device__ __forceinline__ int group(const CandSet& cs, Groups& q, unsigned g) const {
    if (g < q.nslot_groups) {
      const unsigned s = g * 32 + lane_id();
      return s < q.in_slots ? cs.cslot[(size_t)q.v * A.nslots + s] : kNil;
    }
    q.lcur = list_step(cs, q.lcur, (g - q.nslot_groups - q.lnext) << (5 - A.lsub));
    q.lnext = g - q.nslot_groups;
    return q.lcur;
  }
  // The node's candidate set is empty again (the set is reused two steps later).
  __device__ __forceinline__ void clear_groups(const CandSet& cs, uint32_t v, unsigned nc) const {
    const unsigned lane = lane_id();
    __syncwarp();  // every lane has read what it needs
    if (lane == 0) cs.ncand[v] = 0;
    if (nc > A.nslots && lane < (1u << A.lsub)) cs.node_head[((size_t)v << A.lsub) + lane] = kNil;
  }

  __device__ __forceinline__ void node_h(uint32_t v, uint32_t (&hv)[D]) const {
#pragma unroll
    for (int k = 0; k < D; ++k) hv[k] = v == G.n ? 0u : hk(k, v);
  }

  // One node's merge by one warp, 32 candidates at a time:
  // (b) against the frontier alpha(v), compacted in place; at the goal node n
  // alpha is P: one weak-dominance test against the P index and every goal
  // cost logged since it was built (P members a new solution dominates are
  // dropped once, at output: Prune(P, l) of Algorithm 1); (c) F against P;
  // (d) survivors join alpha(v) and the next OPEN.
  __device__ void merge_node(uint32_t v, CycleCtl& K1) {
    const CandSet& cs = A.cs[cyc & 1u];
    const unsigned lane = lane_id();
    // the node's words and its first slots, in one round of loads
    const unsigned nc = cs.ncand[v];
    uint64_t fb = A.fbase[v];
    unsigned cap = A.fcap[v], fc = A.fcount[v];
    const unsigned fc0 = fc;
    const int slot0 = lane < A.nslots ? cs.cslot[(size_t)v * A.nslots + lane] : kNil;
    const uint32_t split = cs.hflag[v];
    uint32_t hv[D];
    node_h(v, hv);
    __syncwarp();  // every lane has read the word before lane 0 changes it
    if (split) {   // merged in parts this step; this item or the last part clears the word
      if (lane == 0 && (atomicOr(&cs.hflag[v], kSplitSeen) & kSplitDone)) cs.hflag[v] = 0;
      return;
    }
    Groups q = open_groups(cs, v, nc);
    const unsigned ng = ngroups(nc);
    unsigned long long fcmp = 0, pcmp = 0;
    bool pruned = false;
    for (unsigned g = 0; g < ng; ++g) {
      const int mine = g ? group(cs, q, g) : (lane < q.in_slots ? slot0 : kNil);
      Batch b = load_batch(cs, mine);
      Round t = load_round(0u, v == G.n ? 0u : fc, fb, cap, true);
      resolve_batch(b);
      // Where parts have grown, merges of several groups are left to one warp, and a
      // label that a later group's candidate prunes again has cost its place in the
      // arena: the later groups are looked at first (256x256 grid, d = 3, W = 262,144,
      // 58.2 -> 56.5 M labels, same time). For single queries with large windows only,
      // whose arenas fill; elsewhere it made searches 1% longer.
      if (kMany && pscale && ng <= 16u && g + 1u < ng) test_groups(cs, v, nc, b, g + 1u, ng);
      if (v == G.n) {
        batch_ptest(hv, b, __shfl_sync(0xffffffffu, ld_volatile(&C->plog_len.v), 0), 0u, 1u, pcmp);
      } else {
        fc = scan_frontier<true>(v, b, 0u, fc, fb, cap, t, pruned, fcmp);
        batch_ptest(hv, b, psnap, 0u, 1u, pcmp);
      }
      fc = insert_batch(v, hv, b, fc, fb, cap, K1, nc);
    }
    clear_groups(cs, v, nc);
    if (lane == 0) {
      if (fc != fc0) A.fcount[v] = fc;
      count_big(S_FCMP, fcmp);
      count_big(S_PCMP, pcmp);
    }
  }

  // The batch's live candidates (in the rows) against the node's candidates of
  // groups [glo, ghi): one that another strictly dominates, or that equals one
  // with a smaller arc id, dies (no two candidates of a node have the same
  // costs and the same arc). The next group's records are loaded while one is tested.
  __device__ void test_groups(const CandSet& cs, uint32_t v, unsigned nc, Batch& b, unsigned glo, unsigned ghi) {
    const unsigned lane = lane_id();
    unsigned am = __ballot_sync(0xffffffffu, b.alive);
    Groups q = open_groups(cs, v, nc);
    int o = glo < ghi ? group(cs, q, glo) : kNil;
    Batch t = load_batch(cs, o);
    for (unsigned g = glo; g < ghi && am; ++g) {
      const int o2 = g + 1 < ghi ? group(cs, q, g + 1) : kNil;
      const Batch t2 = load_batch(cs, o2);
      for (unsigned todo = am; todo;) {
        unsigned j[2];
        next_two(todo, j);
        unsigned gone = 0;
#pragma unroll
        for (int x = 0; x < 2; ++x) {
          uint32_t cj[D], ej;
          get_row(j[x], cj, ej);
          if (t.alive && weakly_le<D>(t.c, cj)) {
            // (one that equals it in cost and arc is the candidate itself)
            if (!weakly_le<D>(cj, t.c) || t.edge < ej) gone |= 1u << j[x];
          }
        }
        am &= ~__reduce_or_sync(0xffffffffu, gone);
      }
      t = t2;
    }
    b.alive = (am >> lane) & 1u;
  }

  // Part r of a merge split into k parts (a power of two; decided while the
  // node's candidates arrived), one warp. What can drop a candidate -- the
  // node's other candidates, the frontier, P -- is only read, so the parts are
  // independent: ka shares of the candidates (groups a, a + ka, ... of 32, or
  // 16, 8 or 4 lanes of one group while there are more parts than groups)
  // times kb ranges of all three. Shares of the candidates come first, as a
  // candidate's early exit stays within one part then, while they hold about
  // kShareCands candidates. Frontier entries a
  // candidate strictly dominates are marked pruned (ldead = cyc); candidates
  // that die get cflag set. Dominance is transitive and the frontier is an
  // antichain, so it does not matter that a part does not see the deaths of the
  // others. The last part to finish (a counter per node; nobody waits) compacts
  // the frontier if a part pruned, and inserts what no part dropped.
  //
  // One warp a part, not a block: a block merge of the same work was 40 us of
  // block barriers and round trips between them for 3 us of comparisons, while
  // warps wait for nobody and many share an SM.
  static constexpr unsigned kShareCands = 4;
  __device__ void merge_part(uint32_t v, unsigned r, unsigned k, CycleCtl& K1) {
    const CandSet& cs = A.cs[cyc & 1u];
    const unsigned lane = lane_id();
    const bool goal = v == G.n;
    const unsigned nc = cs.ncand[v], F = A.fcount[v];
    uint64_t fb = A.fbase[v];
    unsigned cap = A.fcap[v];
    uint32_t hv[D];
    node_h(v, hv);
    const unsigned plen = goal ? __shfl_sync(0xffffffffu, ld_volatile(&C->plog_len.v), 0) : psnap;
    const unsigned ng = ngroups(nc);
    unsigned ka = k, sub = 1;  // sub: shares of a group of 32
    while (ka > 1u && ka / 2 >= ng) {
      ka >>= 1;
      if (sub < kPartShares && sub * kShareCands < nc) sub <<= 1;
    }
    const unsigned ks = ka * sub, kb = k / ks;
    const unsigned a = (r % ks) / sub, bb = r / ks;
    const unsigned width = 32u / sub, l0 = (r % ks) % sub * width;  // this part's lanes of a group
    const unsigned lo = (unsigned)((uint64_t)F * bb / kb), hi = goal ? 0u : (unsigned)((uint64_t)F * (bb + 1) / kb);
    unsigned long long fcmp = 0, pcmp = 0;
    bool pruned = false;
    {
      Groups q = open_groups(cs, v, nc);
      // (parts beyond the shares times the ranges have nothing to do)
      for (unsigned g = r < ks * kb ? a : ng; g < ng; g += ka) {
        const int mine = group(cs, q, g);
        Batch b = load_batch(cs, mine);
        Round t = load_round(lo, hi, fb, cap, false);
        const bool own = lane - l0 < width;
        b.alive = b.alive && own;
        put_row(b.c, b.edge);
        if (!goal) scan_frontier<false>(v, b, lo, hi, fb, cap, t, pruned, fcmp);
        test_groups(cs, v, nc, b, ng * bb / kb, ng * (bb + 1) / kb);
        batch_ptest(hv, b, plen, bb, kb, pcmp);
        if (own && mine != kNil && !b.alive) cs.cflag[mine] = 1u;
      }
    }
    // the part counter's low 16 bits count finished parts; kPartPruned is
    // added by a part that pruned a frontier entry
    const unsigned pr = __any_sync(0xffffffffu, pruned) ? kPartPruned : 0u;
    __threadfence();
    __syncwarp();
    unsigned done = 0;
    if (lane == 0) done = atomicAdd(&cs.hcnt[v], 1u + pr) + 1u + pr;
    done = __shfl_sync(0xffffffffu, done, 0);
    if ((done & (kPartPruned - 1u)) == k) {
      __threadfence();
      unsigned out = F;
      if (done >= kPartPruned) out = compact_pruned(fb, cap, F);
      Groups q = open_groups(cs, v, nc);
      int pend = kNil;  // lanes 0 .. np-1: survivors to insert
      unsigned np = 0;
      for (unsigned g0 = 0; g0 < ng; g0 += 4) {  // four groups' flags side by side
        int mine[4];
        uint32_t gone[4];
#pragma unroll
        for (int x = 0; x < 4; ++x) mine[x] = g0 + x < ng ? group(cs, q, g0 + x) : kNil;
#pragma unroll
        for (int x = 0; x < 4; ++x) gone[x] = mine[x] != kNil ? __ldcg(cs.cflag + mine[x]) : 1u;
#pragma unroll
        for (int x = 0; x < 4; ++x) {
          const unsigned bal = __ballot_sync(0xffffffffu, gone[x] == 0u), cnt = __popc(bal);
          if (np + cnt > 32u) {
            out = insert_batch(v, hv, load_batch(cs, pend), out, fb, cap, K1, nc);
            pend = kNil;
            np = 0;
          }
          const unsigned t = lane - np;  // this lane receives the t-th survivor of the group
          const bool recv = lane >= np && t < cnt;
          const int got = __shfl_sync(0xffffffffu, mine[x], recv ? nth_bit(bal, t) : 0u);
          if (recv) pend = got;
          np += cnt;
        }
      }
      if (np) out = insert_batch(v, hv, load_batch(cs, pend), out, fb, cap, K1, nc);
      clear_groups(cs, v, nc);
      if (lane == 0) {
        cs.hcnt[v] = 0;
        if (out != F) A.fcount[v] = out;
        if (atomicOr(&cs.hflag[v], kSplitDone) & kSplitSeen) cs.hflag[v] = 0;
      }
    }
    if (lane == 0) {
      count_big(S_FCMP, fcmp);
      count_big(S_PCMP, pcmp);
    }
  }

  // Compaction of a frontier after a split merge, by one warp: the entries
  // whose label was pruned in this step (ldead == cyc, written by other warps:
  // read past L1) are removed; returns the live count. Two dependent loads a
  // round are what it costs, so a round is eight tiles of label ids and their
  // words, and costs are read only from the first removed entry on. (Four tiles
  // with their costs made a step of the 256x256 grid, d = 3, W = 1,024, whose
  // largest frontiers have thousands of entries, 55.1 us instead of 52.6.)
  __device__ unsigned compact_pruned(uint64_t fb, unsigned cap, unsigned F) {
    constexpr int U = 8;
    const unsigned lane = lane_id();
    uint32_t* const ids = A.fpool + fb + (size_t)D * cap;
    unsigned out = 0;
    for (unsigned r0 = 0; r0 < F; r0 += 32 * U) {
      uint32_t mid[U];
      unsigned km[U];
#pragma unroll
      for (int u = 0; u < U; ++u) mid[u] = r0 + u * 32 + lane < F ? ids[r0 + u * 32 + lane] : 0u;
      unsigned kept = 0;
#pragma unroll
      for (int u = 0; u < U; ++u) km[u] = r0 + u * 32 + lane < F ? __ldcg(A.ldead + mid[u]) : cyc;
#pragma unroll
      for (int u = 0; u < U; ++u) {
        km[u] = __ballot_sync(0xffffffffu, km[u] != cyc);
        kept += __popc(km[u]);
      }
      if (out == r0 && kept == min(32u * U, F - r0)) {  // nothing removed yet: the entries stay in place
        out += kept;
        continue;
      }
#pragma unroll
      for (int u0 = 0; u0 < U; u0 += kU) {
        uint32_t m[kU][D];
#pragma unroll
        for (int u = 0; u < kU; ++u) {
          const bool keep = (km[u0 + u] >> lane) & 1u;
#pragma unroll
          for (int k = 0; k < D; ++k)
            m[u][k] = keep ? A.fpool[fb + (size_t)k * cap + r0 + (u0 + u) * 32 + lane] : 0u;
        }
        __syncwarp();  // read before any of their places is written
#pragma unroll
        for (int u = 0; u < kU; ++u) {
          const unsigned pos = out + __popc(km[u0 + u] & lanemask_lt());
          if ((km[u0 + u] >> lane) & 1u) {
#pragma unroll
            for (int k = 0; k < D; ++k) A.fpool[fb + (size_t)k * cap + pos] = m[u][k];
            ids[pos] = mid[u0 + u];
          }
          out += __popc(km[u0 + u]);
        }
        __syncwarp();
      }
    }
    __syncwarp();
    return out;
  }

  // ---------------- P index rebuild (three steps, then published) ----------------
  // Rank item: the Z-order rank contributions of 32 logged goal costs (one
  // per lane) from kRankQ others, added into prank.
  __device__ void rank_item(unsigned item) {
    if constexpr (D >= 2) {
      constexpr int MD = D - 1 < 3 ? D - 1 : 3;
      const PIdx& pd = S.pd;
      const unsigned k = pd.k;
      const unsigned nq = (k + kRankQ - 1) / kRankQ;
      const unsigned eb = item / nq, qc = item % nq;
      const unsigned lane = lane_id();
      const unsigned i = eb * 32 + lane;
      const bool vi = i < k;
      const size_t pc = A.plog_cap;
      uint32_t lo[MD], zi[MD];
#pragma unroll
      for (int j = 0; j < MD; ++j) {
        lo[j] = hk(j + 1, P.start);
        zi[j] = vi ? (A.plog[(size_t)(j + 1) * pc + i] - lo[j]) >> pd.shift[j] : 0u;
      }
      unsigned rank = 0;
      const unsigned q1 = min(k, (qc + 1) * kRankQ);
      for (unsigned q = qc * kRankQ; q < q1; ++q) {
        uint32_t zq[MD];
#pragma unroll
        for (int j = 0; j < MD; ++j) zq[j] = (A.plog[(size_t)(j + 1) * pc + q] - lo[j]) >> pd.shift[j];
        rank += z_less<MD>(zq, zi) || (q < i && !z_less<MD>(zi, zq));
      }
      if (vi && rank) atomicAdd(&A.prank[i], rank);
    }
  }

  template <class Team>
  __device__ void index_strided_work(const Team& T) {
    if constexpr (D >= 2) {
      const PIdx& pd = S.pd;
      const unsigned k = pd.k, nb = pd.nb;
      const size_t pc = A.plog_cap;
      if (pd.state == 2) {  // scatter every logged cost to its rank
        for (unsigned x = T.tid(); x < k; x += T.nthreads()) {
          const unsigned r = A.prank[x];
#pragma unroll
          for (int kk = 0; kk < D; ++kk) A.ps[nb][(size_t)kk * pc + r] = A.plog[(size_t)kk * pc + x];
        }
      } else if (pd.state == 3) {  // tile minima; ranks cleared for the next rebuild
        const unsigned nt = (k + 31) / 32;
        const size_t tcap = pc / 32 + 1;
        for (unsigned t = T.tid(); t < nt; t += T.nthreads()) {
          uint32_t mn[D];
#pragma unroll
          for (int kk = 0; kk < D; ++kk) mn[kk] = kInf;
          for (unsigned e = t * 32; e < min(k, t * 32 + 32); ++e)
#pragma unroll
            for (int kk = 0; kk < D; ++kk) mn[kk] = min(mn[kk], A.ps[nb][(size_t)kk * pc + e]);
#pragma unroll
          for (int kk = 0; kk < D; ++kk) A.pst[nb][(size_t)kk * tcap + t] = mn[kk];
        }
        for (unsigned x = T.tid(); x < k; x += T.nthreads()) A.prank[x] = 0;
      }
    }
  }

  // The P index as step i+1 will see it (leader block, all threads): a
  // rebuild advances rank -> scatter -> tiles -> published; with none in
  // progress, one starts once the log has outgrown the index by 32 + its
  // count >> ps_grow (each F-against-P test also scans the unindexed tail).
  __device__ void index_transition(unsigned i) {
    PIdx nd = S.pd;
    bool plan = false;
    if (nd.state == 1) {
      nd.state = 2;
    } else if (nd.state == 2) {
      nd.state = 3;
    } else if (nd.state == 3) {
      nd.cur = nd.nb;
      nd.count = nd.k;
      nd.mark = nd.k;
      nd.ntiles = (nd.k + 31) / 32;
      nd.state = 0;
    } else if (D >= 2) {
      plan = psnap - nd.mark > 32u + (nd.count >> P.ps_grow) && psnap <= kPSMax;
    }
    if (plan) {
      constexpr int MD = D - 1 < 3 ? D - 1 : 3;
      if (threadIdx.x == 0) S.pmax[0] = S.pmax[1] = S.pmax[2] = 0;
      __syncthreads();
      unsigned mx[3] = {0, 0, 0};
      for (unsigned x = threadIdx.x; x < psnap; x += blockDim.x)
#pragma unroll
        for (int j = 0; j < MD; ++j)
          mx[j] = max(mx[j], A.plog[(size_t)(j + 1) * A.plog_cap + x] - hk(j + 1, P.start));
#pragma unroll
      for (int j = 0; j < MD; ++j) atomicMax(&S.pmax[j], mx[j]);
      __syncthreads();
      int bl[3] = {0, 0, 0}, mn = 32;
#pragma unroll
      for (int j = 0; j < MD; ++j) {
        bl[j] = 32 - __clz(S.pmax[j]);
        mn = min(mn, bl[j]);
      }
#pragma unroll
      for (int j = 0; j < 3; ++j) nd.shift[j] = j < MD ? (unsigned)(bl[j] - mn) : 0u;
      nd.state = 1;
      nd.nb = nd.cur ^ 1u;
      nd.k = psnap;
    }
    if (threadIdx.x == 0) C->pidx[(i + 1) & 1u] = nd;
  }

  // ---------------- one step ----------------
  // Returns false (on every block alike) when the search is over: OPEN_i
  // holds no entry and window i produced no candidate.
  template <class Team>
  __device__ bool step(const Team& T, unsigned i, unsigned long long* tlap) {
    const unsigned r0 = i % 3, r1 = (i + 1) % 3, r2 = (i + 2) % 3;
    const unsigned cur = i & 1u;
    CycleCtl& K0 = C->cyc[r0];
    CycleCtl& K1 = C->cyc[r1];
    CycleCtl& K2 = C->cyc[r2];
    const bool fifo = (P.flags & OPMOS_FLAG_FIFO) != 0;
    const Bins bins = load_bins(A.hist + r0 * kNB);
    // Everything the step reads of its record, by one warp a block in one round
    // of loads, a lane a word (every warp reading every word was 36,000 loads
    // of 15 lines a step: 2.7 us).
    if (threadIdx.x < kRecWords) {
      static_assert(sizeof(BinLimits) == 5 * 4 && sizeof(PIdx) == 10 * 4, "RecWord");
      static_assert(offsetof(CycleCtl, min_key) == RW_KEYLO * 128, "RecWord");
      const unsigned l = threadIdx.x;
      const unsigned* src = reinterpret_cast<const unsigned*>(&K0) + l * 32u;
      if (l == RW_KEYHI) src -= 31;
      if (l >= RW_BINS) src = reinterpret_cast<const unsigned*>(&C->bins[r0]) + (l - RW_BINS);
      if (l >= RW_PIDX) src = reinterpret_cast<const unsigned*>(&C->pidx[cur]) + (l - RW_PIDX);
      const unsigned x = __ldcg(src);
      S.rec[l] = x;
      if (l >= RW_PIDX) reinterpret_cast<unsigned*>(&S.pd)[l - RW_PIDX] = x;
      if (l < 5) S.tmax[l] = 0;
      if (l == 0) {
        S.min_key = ~0ull;
        S.win_min = S.f1lo = kInf;
        S.win_max = S.f1hi = 0;
      }
    }
    __syncthreads();
    const unsigned* rec = S.rec;
    const unsigned head = rec[RW_HEAD], tail = rec[RW_OPEN];
    const unsigned nt = rec[RW_TOUCHED], np = min(rec[RW_PARTS], A.xcap);
    const Measured ms{(unsigned long long)rec[RW_KEYHI] << 32 | rec[RW_KEYLO], rec[RW_F1LO], rec[RW_F1HI],
                      rec[RW_WMIN], rec[RW_WPREV], rec[RW_WMAX]};
    const unsigned n_in = min(tail - head, A.open_cap);  // FIFO: ring tail - head
    if (n_in == 0 && nt == 0) return false;
    cyc = i;
    fifo_head = head;
    const unsigned fwin = min(n_in, P.window);  // FIFO: ring positions window i+1 takes
    psnap = rec[RW_PLEN];
    lbase = rec[RW_LBASE];
    // bins OPEN_i's histogram was built on
    const BinParams bp{rec[RW_BINS], rec[RW_BINS + 1], rec[RW_BINS + 2], rec[RW_BINS + 3], rec[RW_BINS + 4]};
    bpn = next_bins(ms);
    pscale = next_scale(rec[RW_PARTS], rec[RW_SCALE]);
    select_window(bins, fifo || n_in <= P.window);
    for (unsigned x = T.tid(); x < kNB; x += T.nthreads()) A.hist[r2 * kNB + x] = 0;
    if (T.leader_block()) {
      if (threadIdx.x == 64) {
        // the longest tasks of step i-1 (its slot is K2)
        count_big(S_MAXH, K2.tmax[0]);
        count_big(S_MAXL, K2.tmax[1]);
        count_big(S_MAXX, K2.tmax[2]);
        count_big(S_MAXNC, K2.tmax[3]);
        count_big(S_MAXF, K2.tmax[4]);
        clear_cycle(K2);
        // values step i+1 starts from; the writers of this step raise them
        atomicMax(&K1.plen.v, psnap);
        atomicMax(&K1.lbase.v, lbase);
        K1.win_prev.v = ms.wmin;
        K1.part_scale.v = pscale;
        C->bins[r1] = BinLimits{bpn.b0, bpn.b1, bpn.s1, bpn.delta, bpn.s2};
        if (fifo) {
          K1.head.v = head + fwin;
          atomicMax(&K1.open_count.v, head + n_in);
        }
      }
      index_transition(i);
    }
    __syncthreads();
    if (T.leader() && tlap) {
      const unsigned long long t = globaltimer();
      count_big(S_TSEL, t - *tlap);
      *tlap = t;
    }
    // work items, one warp each: parts of split merges (the longest), index-rank
    // items, merges, extraction chunks
    const PIdx& pd = S.pd;
    const unsigned nrank = (D >= 2 && pd.state == 1) ? ((pd.k + 31) / 32) * ((pd.k + kRankQ - 1) / kRankQ) : 0u;
    const unsigned nopen = fifo ? fwin : n_in, nwarps = T.nwarps();
    const unsigned per = item_entries(nopen, nwarps);
    const unsigned nchunks = (nopen + per - 1) / per;
    const unsigned nitems = np + nrank + nt + nchunks;
    const unsigned lane = lane_id();
    unsigned done = 0;  // items of this warp
    // The first item of a warp goes by its number, neighbouring items to
    // different blocks; the rest is claimed (claims by every warp at once queue
    // on one counter: 2 us).
    for (unsigned t = (threadIdx.x >> 5) * T.nblocks() + T.block(); t < nitems;) {
      const unsigned long long t0 = globaltimer();
      if (t < np) {
        const uint2 x = A.cs[cur].xpart[t];
        const uint32_t v = x.x;
        if (v != kNoPart) {
          const unsigned r = x.y, k = A.cs[cur].hflag[v] & kSplitParts;
          if (lane == 0 && r == 0) {  // read before the merge clears them
            atomicMax(&S.tmax[3], A.cs[cur].ncand[v]);
            atomicMax(&S.tmax[4], A.fcount[v]);
            count(S_NHEAVY, 1u);
          }
          __syncwarp();
          merge_part(v, r, k, K1);
          if (lane == 0) {
            const unsigned long long dt = globaltimer() - t0;
            atomicMax(&S.tmax[0], (unsigned)min(dt, 0xFFFFFFFFull));
            count_big(S_SUMH, dt);
          }
        }
      } else if (t < np + nrank) {
        rank_item(t - np);
      } else if (t < np + nrank + nt) {
        const uint32_t v = A.cs[cur].touched[t - np - nrank];
        merge_node(v, K1);
        if (lane == 0) {
          const unsigned long long dt = globaltimer() - t0;
          atomicMax(&S.tmax[1], (unsigned)min(dt, 0xFFFFFFFFull));
          count_big(S_SUML, dt);
        }
      } else {
        const unsigned c = t - np - nrank - nt;
        if (fifo)
          extract_fifo(head + c * per, head + min(fwin, (c + 1) * per), K1);
        else
          extract_chunk(c, n_in, per, bp, K1);
        if (lane == 0) {
          const unsigned long long dt = globaltimer() - t0;
          atomicMax(&S.tmax[2], (unsigned)min(dt, 0xFFFFFFFFull));
          count_big(S_SUMX, dt);
        }
      }
      if (nitems <= nwarps) break;
      if (++done % kFlushItems == 0) empty_counts();
      if (lane == 0) t = nwarps + atomicAdd(&K0.work_next.v, 1u);
      t = __shfl_sync(0xffffffffu, t, 0);
    }
    index_strided_work(T);
    __syncthreads();
    if (threadIdx.x < 5 && S.tmax[threadIdx.x]) atomicMax(&K0.tmax[threadIdx.x], S.tmax[threadIdx.x]);
    flush_counts(C, S, kFlushAt);
    if (threadIdx.x == 32) {
      if (S.min_key != ~0ull) atomicMin(&K1.min_key.v, S.min_key);
      if (S.win_min != kInf) {
        atomicMin(&K1.win_min.v, S.win_min);
        atomicMax(&K1.win_max.v, S.win_max);
      }
      if (S.f1lo != kInf) {
        atomicMin(&K1.f1lo.v, S.f1lo);
        atomicMax(&K1.f1hi.v, S.f1hi);
      }
    }
    // (a thread empties what it adds: S.hist is zero again for the next step)
    for (unsigned x = threadIdx.x; x < kNB / 4; x += blockDim.x) {
      uint4& q = reinterpret_cast<uint4*>(S.hist)[x];
      const uint4 h = q;
      if (!(h.x | h.y | h.z | h.w)) continue;
      q = make_uint4(0u, 0u, 0u, 0u);
      unsigned* to = A.hist + r1 * kNB + 4 * x;
      if (h.x) atomicAdd(to, h.x);
      if (h.y) atomicAdd(to + 1, h.y);
      if (h.z) atomicAdd(to + 2, h.z);
      if (h.w) atomicAdd(to + 3, h.w);
    }
    if (T.leader() && tlap) {
      const unsigned long long t = globaltimer();
      count_big(S_TWORK, t - *tlap);
      *tlap = t;
    }
    return true;
  }

  // ---------------- output: P without dominated members, sorted, with paths ----------------
  // Four parts separated by team barriers (single query) or by iterations of
  // the multi-query kernel: filter | rank | scan | paths. Regions of the
  // output pool: res_off holds k'*D costs then k'+1 path offsets; res_path
  // holds the path nodes then their arcs.

  // (1) Prune(P, l) deferred from the search: drop members another member
  // dominates; C->res_count must be 0 beforehand.
  template <class Team>
  __device__ void out_filter(const Team& T) {
    const uint32_t t = G.n;  // P
    const unsigned k = A.fcount[t];
    const uint64_t fb = A.fbase[t];
    const unsigned cap = A.fcap[t];
    unsigned kept = 0;
    for (unsigned i = T.tid(); i < k; i += T.nthreads()) {
      uint32_t ci[D];
#pragma unroll
      for (int kk = 0; kk < D; ++kk) ci[kk] = A.fpool[fb + (size_t)kk * cap + i];
      bool dom = false;
      for (unsigned j = 0; j < k && !dom; ++j) {
        uint32_t cj[D];
#pragma unroll
        for (int kk = 0; kk < D; ++kk) cj[kk] = A.fpool[fb + (size_t)kk * cap + j];
        dom = dominates<D>(cj, ci);
      }
      if (dom) {
        A.ldead[A.fpool[fb + (size_t)D * cap + i]] = 0;
        count(S_PRUNED, 1u);
      } else {
        ++kept;
      }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) kept += __shfl_xor_sync(0xffffffffu, kept, o);
    if (lane_id() == 0 && kept) atomicAdd(&C->res_count, kept);
  }

  // (2a) region 1 allocation, one thread.
  __device__ void out_alloc1() {
    const unsigned kk_live = ld_volatile(&C->res_count);
    const unsigned long long words = (unsigned long long)kk_live * D + kk_live + 1;
    const unsigned long long off = atomicAdd(O.used, words);
    if (off + words > O.cap) set_error(C, OPMOS_ERR_CAPACITY);
    C->res_off = off;
  }

  // (2b) lexicographic rank of every kept member; costs and path lengths.
  template <class Team>
  __device__ void out_rank(const Team& T) {
    const uint32_t t = G.n;  // P
    const unsigned k = A.fcount[t];
    const uint64_t fb = A.fbase[t];
    const unsigned cap = A.fcap[t];
    const bool paths = !(P.flags & OPMOS_FLAG_NO_PATHS);
    const unsigned kk_live = ld_volatile(&C->res_count);
    const unsigned long long off = C->res_off;
    for (unsigned i = T.tid(); i < k; i += T.nthreads()) {
      const uint32_t idi = A.fpool[fb + (size_t)D * cap + i];
      if (A.ldead[idi] != kAlive) continue;
      uint32_t ci[D];
#pragma unroll
      for (int kk = 0; kk < D; ++kk) ci[kk] = A.fpool[fb + (size_t)kk * cap + i];
      unsigned rank = 0;
      for (unsigned j = 0; j < k; ++j) {
        uint32_t cj[D];
#pragma unroll
        for (int kk = 0; kk < D; ++kk) cj[kk] = A.fpool[fb + (size_t)kk * cap + j];
        if ((lex_less<D>(cj, ci) || (j < i && equal<D>(cj, ci))) &&
            A.ldead[A.fpool[fb + (size_t)D * cap + j]] == kAlive)
          ++rank;
      }
      if (rank >= kk_live || off + (unsigned long long)kk_live * D + kk_live + 1 > O.cap) {
        set_error(C, OPMOS_ERR_CAPACITY);  // never write outside the allocated region
        continue;
      }
#pragma unroll
      for (int kk = 0; kk < D; ++kk) O.words[off + (size_t)rank * D + kk] = ci[kk];
      unsigned len = 0;
      if (paths)
        for (uint32_t x = idi; x != kInf; x = A.lparent[x]) ++len;
      O.words[off + (size_t)kk_live * D + rank] = len;
      A.lpver[idi] = rank;  // remembered for the path pass
    }
  }

  // (3) exclusive scan of the path lengths and region 2 allocation; one block.
  __device__ void out_scan() {
    const bool paths = !(P.flags & OPMOS_FLAG_NO_PATHS);
    const unsigned kk_live = ld_volatile(&C->res_count);
    const unsigned long long off = C->res_off;
    uint32_t* lens = O.words + off + (size_t)kk_live * D;
    unsigned carry = 0;
    for (unsigned b0 = 0; b0 < kk_live + 1; b0 += blockDim.x) {
      const unsigned i = b0 + threadIdx.x;
      const unsigned x = i < kk_live ? lens[i] : 0;
      unsigned total;
      const unsigned ex = block_exclusive_scan(x, S.warp, total);
      if (i <= kk_live) lens[i] = carry + ex;
      carry += total;
    }
    if (threadIdx.x == 0) {
      const unsigned long long total = carry;
      const unsigned long long words = paths ? 2 * total - kk_live : 0;
      unsigned long long p0 = 0;
      if (words) {
        p0 = atomicAdd(O.used, words);
        if (p0 + words > O.cap) set_error(C, OPMOS_ERR_CAPACITY);
      }
      C->res_path = p0;
      C->res_total = total;
    }
  }

  // (4) parent-chain walks: nodes start..goal and the arcs between them.
  template <class Team>
  __device__ void out_paths(const Team& T) {
    if (P.flags & OPMOS_FLAG_NO_PATHS) return;
    const uint32_t t = G.n;  // P
    const unsigned k = A.fcount[t];
    const uint64_t fb = A.fbase[t];
    const unsigned cap = A.fcap[t];
    const unsigned kk_live = ld_volatile(&C->res_count);
    const unsigned long long off = C->res_off, p0 = C->res_path, total = C->res_total;
    const uint32_t* offs = O.words + off + (size_t)kk_live * D;
    if (p0 + 2 * total > O.cap + kk_live) return;  // region 2 was not granted
    for (unsigned i = T.tid(); i < k; i += T.nthreads()) {
      const uint32_t idi = A.fpool[fb + (size_t)D * cap + i];
      if (A.ldead[idi] != kAlive) continue;
      const unsigned rank = A.lpver[idi];
      if (rank >= kk_live) continue;
      const unsigned a = offs[rank], b = offs[rank + 1];
      // nodes at p0 + [a, b); arcs at p0 + total + [a - rank, b - rank - 1)
      unsigned pos = b;
      for (uint32_t x = idi; x != kInf && pos > a; x = A.lparent[x]) {
        --pos;
        O.words[p0 + pos] = A.lnode[x];
        if (A.lparent[x] != kInf) O.words[p0 + total + pos - rank - 1] = A.ledge[x];
      }
    }
  }

  template <class Team>
  __device__ bool output(const Team& T) {
    out_filter(T);
    if (!T.sync(C)) return false;
    if (T.leader()) out_alloc1();
    if (!T.sync(C)) return false;
    out_rank(T);
    if (!T.sync(C)) return false;
    if (T.leader_block()) out_scan();
    if (!T.sync(C)) return false;
    out_paths(T);
    return true;
  }
};

// ---------------------------------------------------------------------------
// Single query on the whole cooperative grid
// ---------------------------------------------------------------------------
template <int D, bool kMany>
__device__ void run_grid(const GraphDev& G, const QArena& A, QCtl* C, const QParams& P, const OutPool& O,
                         QResult* R) {
  __shared__ Shared S;
  const GridTeam T;
  Search<D, kMany> X(G, A, C, P, O, S);
  clear_counts(S);
  for (unsigned x = threadIdx.x; x < kNB; x += blockDim.x) S.hist[x] = 0;
  X.init_zero(T);
  bool ok = T.sync(C);
  X.init_seed(T, false);
  ok = ok && T.sync(C);
  unsigned step = 0;
  unsigned long long tph = globaltimer();
  while (ok) {
    if (T.leader() && globaltimer() - C->t_start > P.time_limit_ns) set_error(C, OPMOS_ERR_TIMEOUT);
    if (!X.step(T, step, &tph)) break;
    ok = T.sync(C);
    if (T.leader()) {
      const unsigned long long t = globaltimer();
      X.count_big(S_TSYNC, t - tph);
      tph = t;
    }
    ++step;
  }
  if (ok) {
    if (T.leader()) C->res_count = 0;
    ok = T.sync(C) && X.output(T);
    if (T.leader()) X.count_big(S_TOUT, globaltimer() - tph);
  }
  if (T.leader()) {
    X.count(S_STEPS, step);
    X.count(S_GOALINS, ld_volatile(&C->plog_len.v));
  }
  __syncthreads();
  flush_counts(C, S);
  T.sync(C);
  if (T.leader()) {
    __threadfence();
    R->status = *reinterpret_cast<volatile unsigned*>(&C->bar.error);
    R->count = C->res_count;
    R->off = C->res_off;
    R->path = C->res_path;
    R->total = C->res_total;
    R->labels = C->n_labels.v;
    R->f_words = C->f_words.v;
    for (int i = 0; i < kNStat; ++i) R->stats[i] = C->stats[i];
  }
}

template <int D, unsigned NT, unsigned NB>
__global__ void __launch_bounds__(NT, NB) search_grid_kernel(GraphDev G, QArena A, QCtl* C, QParams P, OutPool O,
                                                             QResult* R) {
  run_grid<D, (NB > 1)>(G, A, C, P, O, R);
}

// ---------------------------------------------------------------------------
// Multi-query persistent kernel (batch and serving): continuous batching of
// many independent queries, each a slot. Every iteration:
//   P0  block 0 retires finished slots and admits queued queries into free
//       slots (FREE -> INIT -> RUN -> OUT -> FREE), and advances every
//       running slot by one step;
//   P1  INIT slots are initialised, OUT slots write one part of their
//       result, RUN slots run one search step (merge of window i beside the
//       extraction of window i+1).
// In P1 every block reads the same assignment of "virtual blocks" to slots,
// made in P0 (a running slot gets a share of the grid in proportion to its
// work, at least one block), so large and small queries advance side by side.
// ---------------------------------------------------------------------------
struct SubTeam {
  unsigned j, nb;
  __device__ __forceinline__ unsigned tid() const { return j * blockDim.x + threadIdx.x; }
  __device__ __forceinline__ unsigned nthreads() const { return nb * blockDim.x; }
  __device__ __forceinline__ unsigned wid() const { return tid() >> 5; }
  __device__ __forceinline__ unsigned nwarps() const { return nthreads() >> 5; }
  __device__ __forceinline__ unsigned block() const { return j; }
  __device__ __forceinline__ unsigned nblocks() const { return nb; }
  __device__ __forceinline__ bool leader_block() const { return j == 0; }
  __device__ __forceinline__ bool leader() const { return j == 0 && threadIdx.x == 0; }
};

__device__ inline bool mq_barrier(MCtl* M, unsigned& target) {
  __shared__ unsigned s_ok;
  __syncthreads();
  if (threadIdx.x == 0) {
    target += gridDim.x;
    s_ok = grid_barrier(&M->bar, target);
  }
  __syncthreads();
  return s_ok != 0;
}

__device__ inline void mq_write_result(const MSlot& sl, unsigned slot, QCtl* C, QResult* results,
                                       unsigned* done_flags, unsigned qcap) {
  const unsigned ri = sl.qidx % qcap;
  QResult* R = &results[ri];
  R->status = ld_volatile(&C->bar.error);
  R->slot = slot;
  R->count = C->res_count;
  R->off = C->res_off;
  R->path = C->res_path;
  R->total = C->res_total;
  R->labels = C->n_labels.v;
  R->f_words = C->f_words.v;
  C->stats[S_STEPS] = C->step;
  C->stats[S_GOALINS] = C->plog_len.v;
  unsigned long long st[kNStat];
#pragma unroll
  for (int i = 0; i < kNStat; ++i) st[i] = __ldcg(&C->stats[i]);
#pragma unroll
  for (int i = 0; i < kNStat; ++i) R->stats[i] = st[i];
  if (done_flags) {
    __threadfence_system();  // the record is visible before its completion flag
    *reinterpret_cast<volatile unsigned*>(&done_flags[ri]) = 1u;
    __threadfence_system();
  }
}

template <int D>
__device__ void mq_alloc_region1(const MSlot& sl, QCtl* C) {
  const OutPool& O = sl.O;
  const unsigned kk_live = ld_volatile(&C->res_count);
  const unsigned long long words = (unsigned long long)kk_live * D + kk_live + 1;
  const unsigned long long off = atomicAdd(O.used, words);
  if (off + words > O.cap) set_error(C, OPMOS_ERR_CAPACITY);
  C->res_off = off;
}

// Virtual blocks of the iteration, from every slot's weight (block 0; w[x]: the
// work units of slot threadIdx.x + x * blockDim.x, 0 for none, kOneBlock for
// work of one block). Every slot with work gets one block, and the blocks left
// are shared out in proportion to the work: no more virtual blocks than blocks,
// as long as there are blocks for all, since one that takes two makes the
// iteration twice as long for everyone. M->pref holds the prefix sums. One block
// computes them for all: a block that read the weights for itself could see
// counters the iteration's work already moves, and take another slot's work.
constexpr unsigned kOneBlock = 0xFFFFFFFFu;
constexpr unsigned kSlotsPerThread = (kMaxSlots + kMultiThreads - 1) / kMultiThreads;
__device__ inline void mq_assign(const unsigned (&w)[kSlotsPerThread], unsigned nslots, MCtl* M) {
  __shared__ unsigned long long s_wtot;
  __shared__ unsigned s_active, s_scan[33];
  if (threadIdx.x == 0) {
    s_wtot = 0;
    s_active = 0;
  }
  __syncthreads();
  unsigned long long wloc = 0;
  unsigned active = 0;
#pragma unroll
  for (unsigned x = 0; x < kSlotsPerThread; ++x) {
    active += w[x] != 0u;
    if (w[x] != kOneBlock) wloc += w[x];
  }
  if (wloc) atomicAdd(&s_wtot, wloc);
  if (active) atomicAdd(&s_active, active);
  __syncthreads();
  const unsigned long long wtot = s_wtot > 0 ? s_wtot : 1;
  const unsigned long long spare = gridDim.x > s_active ? gridDim.x - s_active : 0u;
  unsigned carry = 0;
#pragma unroll
  for (unsigned x = 0; x < kSlotsPerThread; ++x) {
    const unsigned q = threadIdx.x + x * blockDim.x;
    if (x * blockDim.x >= nslots) break;
    const unsigned nbq = w[x] == 0u ? 0u : w[x] == kOneBlock ? 1u : 1u + (unsigned)(w[x] * spare / wtot);
    unsigned total;
    const unsigned ex = block_exclusive_scan(nbq, s_scan, total);
    if (q < nslots) M->pref[q] = carry + ex;
    carry += total;
  }
  if (threadIdx.x == 0) M->pref[nslots] = carry;
}

// P0: slot transitions and admission (block 0).
template <int D>
__device__ void mq_schedule(MSlot* slots, QCtl* ctls, unsigned nslots, const MQuery* queue, unsigned* hctl,
                            const GraphDev* graphs, MCtl* M, QResult* results, unsigned* done_flags) {
  __shared__ unsigned s_busy;
  if (threadIdx.x == 0) s_busy = 0;
  __syncthreads();
  const unsigned q_count = ld_volatile(&hctl[HC_TAIL]);
  const unsigned qcap = M->qcap;
  const unsigned after_out = M->hold ? SL_HELD : SL_FREE;
  unsigned w[kSlotsPerThread];  // work units of this thread's slots in the iteration
#pragma unroll
  for (unsigned x = 0; x < kSlotsPerThread; ++x) {
    w[x] = 0;
    const unsigned q = threadIdx.x + x * blockDim.x;
    if (q >= nslots) continue;
    MSlot& sl = slots[q];
    QCtl* C = &ctls[q];
    unsigned st = sl.state;
    if (st == SL_RUN || st == SL_INIT) {
      // the step that comes next, from one round of loads
      const unsigned step = st == SL_RUN ? __ldcg(&C->step) + 1u : 0u;
      const CycleCtl& K = C->cyc[step % 3];
      const unsigned err = ld_volatile(&C->bar.error), open = __ldcg(&K.open_count.v) - __ldcg(&K.head.v),
                     touched = __ldcg(&K.touched_count.v);
      const unsigned parts = min(__ldcg(&K.part_count.v), sl.A.xcap);  // (asked for; the list holds so many)
      const bool late = st == SL_RUN && globaltimer() - C->t_start > sl.P.time_limit_ns;
      C->step = step;
      if (err || (open == 0 && touched == 0)) {
        st = SL_OUT1;
      } else if (late) {
        set_error(C, OPMOS_ERR_TIMEOUT);
        st = SL_OUT1;
      } else {
        st = SL_RUN;
        w[x] = max(1u, open / 4u + touched + parts);
      }
      if (st == SL_OUT1) C->res_count = 0;
    } else if (st == SL_OUT1 || st == SL_OUT2 || st == SL_OUT3 || st == SL_OUT4) {
      // one output part per iteration; an error ends the output early
      if (ld_volatile(&C->bar.error) || st == SL_OUT4) {
        mq_write_result(sl, q, C, results, done_flags, qcap);
        st = after_out;
      } else if (st == SL_OUT1) {
        mq_alloc_region1<D>(sl, C);
        if (ld_volatile(&C->bar.error)) {  // no room for the result: report, never write
          mq_write_result(sl, q, C, results, done_flags, qcap);
          st = after_out;
        } else {
          st = SL_OUT2;
        }
      } else {
        st = st + 1;
      }
    } else if (st == SL_HELD && ld_volatile(&hctl[HC_RELEASE + q])) {
      hctl[HC_RELEASE + q] = 0;  // the host has collected the result
      st = SL_FREE;
    }
    if (st == SL_FREE) {
      unsigned qn = ld_volatile(&M->q_next);
      while (qn < q_count) {
        const unsigned got = atomicCAS(&M->q_next, qn, qn + 1);
        if (got == qn) break;
        qn = got;
      }
      if (qn < q_count) {
        MQuery Q;
        {
          const volatile MQuery* src = &queue[qn % qcap];
          Q.graph = src->graph;
          Q.start = src->start;
          Q.goal = src->goal;
          Q.d = src->d;
          Q.h = src->h;
        }
        sl.P.start = Q.start;
        sl.P.goal = Q.goal;
        sl.P.h = Q.h;
        sl.P.qd = Q.d;
        sl.G = graphs[Q.graph];
        sl.d = Q.d;
        sl.qidx = qn;
        if (M->hold) *sl.O.used = 0;  // serving: the slot's own pool starts empty (batch pools are shared)
        st = SL_INIT;
      }
    }
    sl.state = st;
    if (st == SL_INIT || st == SL_OUT3)
      w[x] = kOneBlock;
    else if (st == SL_OUT1 || st == SL_OUT2 || st == SL_OUT4)
      w[x] = max(1u, __ldcg(sl.A.fcount + sl.G.n) / 4u);
    if (st != SL_FREE) atomicAdd(&s_busy, 1u);
  }
  __syncthreads();
  mq_assign(w, nslots, M);
  if (threadIdx.x == 0) {
    M->iter++;
    const unsigned closing = ld_volatile(&hctl[HC_CLOSING]);
    if (closing >= 2 || (closing && s_busy == 0 && ld_volatile(&M->q_next) >= ld_volatile(&hctl[HC_TAIL])))
      M->done = 1;  // 1: drain then stop; 2: stop now
  }
}

template <int D>
__device__ void mq_work(MSlot* slots, QCtl* ctls, unsigned q, unsigned j, unsigned nb, Shared& S, MSlot& s_slot) {
  // the slot's record in shared memory (a copy in every thread's local memory
  // was 500 bytes a thread an iteration)
  static_assert(sizeof(MSlot) % 4 == 0, "MSlot");
  for (unsigned x = threadIdx.x; x < sizeof(MSlot) / 4; x += blockDim.x)
    reinterpret_cast<unsigned*>(&s_slot)[x] = __ldcg(reinterpret_cast<const unsigned*>(&slots[q]) + x);
  __syncthreads();
  const unsigned st = s_slot.state;
  QCtl* C = &ctls[q];
  Search<D> X(s_slot.G, s_slot.A, C, s_slot.P, s_slot.O, S);
  if (st == SL_INIT) {
    const BlockTeam T;
    X.init_zero(T);
    if (threadIdx.x == 0) C->bar.error = 0;
    __syncthreads();
    X.init_seed(T, true);
    __syncthreads();
  } else if (st == SL_OUT1) {
    X.out_filter(SubTeam{j, nb});
  } else if (st == SL_OUT2) {
    X.out_rank(SubTeam{j, nb});
  } else if (st == SL_OUT3) {
    X.out_scan();
  } else if (st == SL_OUT4) {
    X.out_paths(SubTeam{j, nb});
  } else if (st == SL_RUN) {
    X.step(SubTeam{j, nb}, C->step, nullptr);
  }
  __syncthreads();
  flush_counts(C, S);
}

template <int D>
__device__ void mq_phase(MSlot* slots, QCtl* ctls, unsigned nslots, MCtl* M, Shared& S, MSlot& s_slot,
                         unsigned* s_pref) {
  for (unsigned q = threadIdx.x; q <= nslots; q += blockDim.x) s_pref[q] = ld_volatile(&M->pref[q]);
  __syncthreads();
  const unsigned B = gridDim.x;
  const unsigned VB = s_pref[nslots];
  for (unsigned v = blockIdx.x; v < VB; v += B) {
    unsigned lo = 0, hi = nslots;  // last q with s_pref[q] <= v
    while (hi - lo > 1) {
      const unsigned mid = (lo + hi) / 2;
      if (s_pref[mid] <= v) lo = mid; else hi = mid;
    }
    const unsigned q = lo;
    const unsigned j = v - s_pref[q], nb = s_pref[q + 1] - s_pref[q];
    mq_work<D>(slots, ctls, q, j, nb, S, s_slot);
    __syncthreads();
  }
}

template <int D>
__global__ void __launch_bounds__(kMultiThreads, 2)
    multi_kernel(MSlot* slots, QCtl* ctls, unsigned nslots, const MQuery* queue, unsigned* hctl,
                 const GraphDev* graphs, QResult* results, unsigned* done_flags, MCtl* M) {
  __shared__ Shared S;
  __shared__ MSlot s_slot;
  __shared__ unsigned s_pref[kMaxSlots + 1];
  clear_counts(S);
  for (unsigned x = threadIdx.x; x < kNB; x += blockDim.x) S.hist[x] = 0;
  unsigned target = 0;
  for (;;) {
    if (blockIdx.x == 0) mq_schedule<D>(slots, ctls, nslots, queue, hctl, graphs, M, results, done_flags);
    if (!mq_barrier(M, target)) return;
    if (ld_volatile(&M->done)) return;
    mq_phase<D>(slots, ctls, nslots, M, S, s_slot, s_pref);
    if (!mq_barrier(M, target)) return;
  }
}

}  // namespace detail

// ---------------------------------------------------------------------------
// host launchers, explicitly instantiated per objective count
// ---------------------------------------------------------------------------
// Dynamic shared memory of a block of nt threads: the warps' rows, or at_least
// when that is more. The kernel is allowed the most that any launch of it takes
// (a server's block), as batches and servers launch it from several threads.
template <int D>
size_t row_bytes(const void* kernel, unsigned nt, size_t at_least = 0) {
  const size_t rows = (size_t)nt * detail::Search<D>::RP * 4;
  cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)std::max(rows, kServeBlockSmem));
  return std::max(rows, at_least);
}

template <int D>
cudaError_t launch_grid(const GraphDev& G, const QArena& A, QCtl* C, const QParams& P, const OutPool& O,
                        QResult* R, bool wide, unsigned blocks, cudaStream_t s) {
  void* args[] = {(void*)&G, (void*)&A, (void*)&C, (void*)&P, (void*)&O, (void*)&R};
  const void* kernel = wide ? (const void*)detail::search_grid_kernel<D, kGridWideThreads, kGridWideBlocksPerSM>
                            : (const void*)detail::search_grid_kernel<D, kGridThreads, 1>;
  const unsigned nt = wide ? kGridWideThreads : kGridThreads;
  return cudaLaunchCooperativeKernel(kernel, dim3(blocks), dim3(nt), args, row_bytes<D>(kernel, nt), s);
}

template <int D>
int grid_occupancy(bool wide) {
  const void* kernel = wide ? (const void*)detail::search_grid_kernel<D, kGridWideThreads, kGridWideBlocksPerSM>
                            : (const void*)detail::search_grid_kernel<D, kGridThreads, 1>;
  const unsigned nt = wide ? kGridWideThreads : kGridThreads;
  int nb = 0;
  cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, kernel, (int)nt, row_bytes<D>(kernel, nt));
  return nb;
}

template <int D>
cudaError_t launch_multi_d(MSlot* slots, QCtl* ctls, unsigned nslots, const MQuery* queue, unsigned* hctl,
                           const GraphDev* graphs, QResult* results, unsigned* done_flags, MCtl* M, unsigned blocks,
                           size_t smem, cudaStream_t s) {
  void* args[] = {(void*)&slots, (void*)&ctls, (void*)&nslots, (void*)&queue, (void*)&hctl,
                  (void*)&graphs, (void*)&results, (void*)&done_flags, (void*)&M};
  const void* kernel = (const void*)detail::multi_kernel<D>;
  return cudaLaunchCooperativeKernel(kernel, dim3(blocks), dim3(kMultiThreads), args,
                                     row_bytes<D>(kernel, kMultiThreads, smem), s);
}

template <int D>
int multi_occupancy_d(size_t smem) {
  const void* kernel = (const void*)detail::multi_kernel<D>;
  int nb = 0;
  cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, kernel, (int)kMultiThreads,
                                                row_bytes<D>(kernel, kMultiThreads, smem));
  return nb;
}

}  // namespace opmos
