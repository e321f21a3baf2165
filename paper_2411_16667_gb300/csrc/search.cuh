// Host-visible declarations shared by the search kernels and the C ABI layer.
#pragma once
#include <mutex>

#include "opmos_dev.cuh"

namespace opmos {

// Multi-query kernel (batch and serving) --------------------------------------
constexpr unsigned kMultiThreads = 256;  // threads per block
constexpr unsigned kMaxSlots = 1024;     // concurrent queries
enum SlotState : unsigned {
  SL_FREE = 0, SL_INIT = 1, SL_RUN = 2, SL_OUT1 = 3, SL_OUT2 = 4, SL_OUT3 = 5, SL_OUT4 = 6,
  SL_HELD = 7  // result written, waiting for the host to collect it (serving)
};

struct MSlot {     // one concurrent query: its arena and current parameters
  QArena A;
  QParams P;
  GraphDev G;
  OutPool O;       // where its result goes (shared in batch mode, its own when serving)
  unsigned d, state, qidx, pad;  // d: objectives the query uses (<= the kernel's)
};

struct MQuery {    // a queued query
  uint32_t graph, start, goal, d;
  const uint32_t* h;  // d * n heuristic toward goal (device)
};

struct MCtl {      // grid-wide control of the multi-query kernel
  Barrier bar;  // the grid barrier
  unsigned done, pad;
  unsigned q_next, iter, qcap, hold;  // hold: keep slots until the host releases them
  unsigned pref[kMaxSlots + 1];       // virtual blocks of the iteration: prefix sums over the slots
};

// Host control words (host-mapped memory when serving): [0] queries queued
// so far, [1] closing (no more queries will come), [2 + slot] release flag.
enum { HC_TAIL = 0, HC_CLOSING = 1, HC_RELEASE = 2 };

// Result descriptor of one query, written by the team leader at the end.
// Output words (in the OutPool): at off, count*d costs (lexicographic) then
// count+1 path offsets; at path, total node ids then total-count arc ids.
struct QResult {
  unsigned status;
  unsigned slot;    // slot whose output pool holds the result
  unsigned count;
  unsigned pad;
  unsigned long long off;
  unsigned long long path;
  unsigned long long total;
  unsigned long long labels;
  unsigned long long f_words;
  unsigned long long stats[kNStat];
};

// Kernel launchers of one objective count D (search_inst.cu instantiates them,
// one object per group of D values); the kernel of a query with qd < D
// objectives reads objectives qd..D-1 as 0.
// wide: the grid of two 256-thread blocks per SM (large windows) instead
// of one 384-thread block per SM.
template <int D>
cudaError_t launch_grid(const GraphDev& G, const QArena& A, QCtl* C, const QParams& P, const OutPool& O,
                        QResult* R, bool wide, unsigned blocks, cudaStream_t s);
template <int D>
int grid_occupancy(bool wide);
template <int D>
cudaError_t launch_multi_d(MSlot* slots, QCtl* ctls, unsigned nslots, const MQuery* queue, unsigned* hctl,
                           const GraphDev* graphs, QResult* results, unsigned* done_flags, MCtl* M, unsigned blocks,
                           size_t smem, cudaStream_t s);
template <int D>
int multi_occupancy_d(size_t smem);

// Dispatch on the objective count, 1..OPMOS_MAX_D (search_dispatch.cu).
cudaError_t launch_search_grid(unsigned d, const GraphDev& G, const QArena& A, QCtl* C, const QParams& P,
                               const OutPool& O, QResult* R, bool wide, unsigned blocks, cudaStream_t s);
int search_occupancy(unsigned d, bool wide);
cudaError_t launch_multi(unsigned d, MSlot* slots, QCtl* ctls, unsigned nslots, const MQuery* queue,
                         unsigned* hctl, const GraphDev* graphs, QResult* results, unsigned* done_flags, MCtl* M,
                         unsigned blocks, size_t smem, cudaStream_t s);
int multi_occupancy(unsigned d, size_t smem);

// Ideal-point heuristic jobs: h_out[v] = shortest v->goal distance under
// objective k (Sec. 4), one thread block per job.
struct HJob {
  uint32_t goal, k;
  uint32_t* h_out;  // n entries
};
// Sets the calling thread's opmos_last_error() message; returns code.
int record_error(int code, const char* msg);

// smem: shared memory a block may take. kHeurSmem by default; kHeurSmemServed
// beside a resident multi-query kernel, which leaves a block's place (its
// shared memory, registers and threads) free on the SMs it does not fill: the
// server launches its kernel with kServeBlockSmem a block for that.
constexpr size_t kHeurSmem = 200u << 10;
constexpr size_t kServeBlockSmem = 72u << 10;
constexpr size_t kHeurSmemServed = 68u << 10;
// Resident server kernels of this process. While there is one, the heuristic
// takes blocks that fit beside it: a cluster, or a block with most of an SM's
// shared memory, would wait for the server's end. A heuristic looks and launches
// under mu, and a server's kernel is launched and counted under it, so that none
// starts in between.
struct Residents {
  std::mutex mu;
  int servers = 0;
};
extern Residents residents;
// Loads the heuristic's kernels that run beside a server, by launches without
// jobs (ctr: two zero words of device memory).
cudaError_t load_heuristic(unsigned* ctr, cudaStream_t s);
cudaError_t launch_heuristic(const GraphDev& G, const HJob* jobs, unsigned njobs, uint32_t* scratch,
                             size_t scratch_words_per_block, unsigned blocks, const uint32_t* delta,
                             unsigned* next_job, unsigned* err, cudaStream_t s, size_t smem = kHeurSmem,
                             unsigned sms = 0);

}  // namespace opmos
