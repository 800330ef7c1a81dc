// Host-side engine state of a Pkd-tree (device memory it owns, streams,
// tuning knobs, kernel timers).
#pragma once

#include <cuda_runtime.h>

#include <algorithm>
#include <atomic>
#include <functional>
#include <mutex>
#include <string>
#include <vector>

#include "common.cuh"
#include "ids.cuh"

namespace pkd {

// Tunables; none of them changes any result.
struct Knobs {
  long long fail_alloc_after = -1;  // >= 0: allocations fail after this many more (fault injection)
  long long wait_cycles = 4000000000ll;  // limit of the streaming sieve's waits (clock cycles, ~2 s)
  int base_cap = 0;   // 0: derived from d and the shared memory per block
  int skel_cap = 0;   // 0: derived
  int tile = 2048;    // points per tile in the sieve kernels
  int base_kernel = 0;  // base case: 0 presorted lists, 1 radix select per node
  int sieve_kernel = 0;  // sieve: 0 persistent with bulk copies and recorded
                         // buckets, 2 persistent re-walking, 1 one tile per CTA
  int graph_rounds = -1;  // build rounds: 1 decided on the device (one CUDA graph
                          // with conditional nodes), 0 sequenced by the host,
                          // -1 (not set) a graph when there can be rounds
  long long front_cap = 0;  // > 0: first capacity of an update's flatten lists (testing)
};
Knobs& knobs();

// Device memory of one tree.
//
// Node slots: [0, shared_cap) is a shared region handed out by an atomic
// counter (skeleton nodes of sieve rounds, tree roots); slot
// shared_cap + 2*pos + k (k < 2) belongs to arena position pos, so the
// nodes of a subproblem finished in shared memory over positions
// [s, s + L) live in [shared_cap + 2s, shared_cap + 2s + 2L) without any
// global coordination (a binary tree over L >= 1 points has <= 2L - 1 nodes).
struct TreeMem {
  Params p{};
  int device = 0;
  Pts A{};                 // point arena (SoA), capacity `cap`
  uint64_t cap = 0;
  uint64_t top = 0;        // arena positions [0, top) are in use or garbage
  Node* nodes = nullptr;
  uint8_t* ndim = nullptr;
  uint64_t shared_cap = 0;
  uint64_t node_cap = 0;   // shared_cap + 2*cap
  uint32_t* shared_next = nullptr;  // device: next free slot of the shared region
  uint32_t root = 0;
  uint64_t size = 0;
  uint8_t* dead = nullptr;          // delete scratch: per arena position (kept zero)
  uint32_t* aux = nullptr;          // delete scratch: per node slot (kept zero)
  bool scratch_dirty = false;       // a delete has set marks it has not cleared yet
  DevStatus* st = nullptr;          // device status word
  DevStatus* st_host = nullptr;     // pinned mirror
  uint32_t query_slots = 0;         // slots of st->refused that a running call holds (atomic)
  IdTable ids;                      // id -> coordinates of the stored points
  int32_t* bbox = nullptr;          // stored bounding boxes (boxes.cu), node_cap * 2d
  uint64_t bbox_cap = 0;            // node slots bbox covers
  bool bbox_on = false;             // kept current after every update; queries prune with them
  // the last use of the tree on every stream a call queued work on (an event
  // recorded after that work), so that freeing the tree waits for exactly
  // that work; untracked: a use that could not record one (a call that may
  // not allocate), after which freeing waits for the whole device
  std::vector<std::pair<cudaStream_t, cudaEvent_t>> uses;
  bool untracked = false;
};

// Small host values into device memory, in stream order, by a kernel that
// takes them as arguments (bytes: a multiple of 4, dst 4-byte aligned).  A
// host-to-device copy would queue behind whatever large copy the caller has
// on the same copy engine (the next step's input, say) and hold the stream
// back for its whole duration; a kernel does not.  Up to 4 KiB; larger
// values go through cudaMemcpyAsync.
int dev_store(void* dst, const void* src, size_t bytes, cudaStream_t s);
// n words from device to device the same way (a small copy).
int dev_copy_words(uint32_t* dst, const uint32_t* src, uint32_t n, cudaStream_t s);
// bytes of dst set to `value` by a kernel (for the same reason: a fill that
// the runtime may hand to a copy engine would wait for the caller's copies).
int dev_fill(void* dst, int value, size_t bytes, cudaStream_t s);

// Records the use of tree t by the work queued so far on stream s.
void tree_touch(TreeMem& t, cudaStream_t s, bool noalloc = false);
// Orders the legacy default stream after every recorded use (or, after an
// untracked one, waits for the device) and forgets the uses.
void tree_wait_uses(TreeMem& t);

// Records the tree's use by the calling entry point when it returns (every
// return path, after its last enqueue).
struct TreeTouch {
  TreeMem* t;
  cudaStream_t s;
  bool noalloc = false;
  ~TreeTouch() {
    if (t) tree_touch(*t, s, noalloc);
  }
};

// Every kernel launch of the library goes through PKD_LAUNCH, which counts
// it (pkd_kernel_stats("launches", ...) reports the count).
void count_launch();
#define PKD_LAUNCH(...)        \
  do {                         \
    ::pkd::count_launch();     \
    __VA_ARGS__;               \
  } while (0)

// Host-side tracing: with PKD_TRACE=1 in the environment, trace_mark()
// synchronises the stream and prints the wall time since the previous mark.
void trace_mark(cudaStream_t s, const char* what);

// Testing: a thread that comes to one of these points sleeps there, as often and
// as long as the option of that name says, so that a test can place another
// thread's call in between.
enum PausePoint {
  PAUSE_ROUNDS,  // "pause_rounds": a rebuild whose rounds the host sequences, in front of the first
  PAUSE_SMEM,    // "pause_smem": a kernel with raised shared memory, in front of its launch
  PAUSE_QUERY,   // "pause_query": a query, between its check and its search
  PAUSE_POINTS
};
void test_pause(PausePoint p);

// Lets kernel K be launched with `bytes` of dynamic shared memory on the
// current device.  The limit is the process's, so it is only ever raised, under
// a lock: set to what each launch needs it could be lowered by another thread
// between this thread's setting and its launch, which then fails.
template <auto K>
void allow_smem(size_t bytes) {
  constexpr int DEVICES = 64;
  static std::atomic<int> limit[DEVICES];
  static std::mutex mu;
  int dev = 0;
  cudaGetDevice(&dev);
  if (limit[dev % DEVICES].load(std::memory_order_acquire) < (int)bytes) {
    std::lock_guard<std::mutex> g(mu);
    if (limit[dev % DEVICES].load(std::memory_order_relaxed) < (int)bytes &&
        cudaFuncSetAttribute(K, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes) == cudaSuccess)
      limit[dev % DEVICES].store((int)bytes, std::memory_order_release);
  }
  test_pause(PAUSE_SMEM);
}

// Error helpers.
int cuda_err(cudaError_t e);
#define PKD_CUDA(x)                          \
  do {                                       \
    cudaError_t _e = (x);                    \
    if (_e != cudaSuccess) return cuda_err(_e); \
  } while (0)

// The library's stream-ordered memory pool on the current device.  Its
// release threshold is unlimited: memory freed by one build stays mapped for
// the next instead of being returned to the driver at every synchronisation.
cudaMemPool_t mem_pool();

// Large blocks (tree arenas and node arrays) go through a small cache in
// front of the pool: a freed block is kept with an event recorded on the
// freeing stream and handed to the next request it fits (the requesting
// stream waits on that event), so building, updating and freeing trees in a
// loop does not map and unmap gigabytes each time.  Blocks below
// BIG_BLOCK_MIN go straight to the pool.  On exhaustion the cache is
// emptied and the request retried once.
constexpr size_t BIG_BLOCK_MIN = (size_t)64 << 20;
cudaError_t big_alloc(void** p, size_t bytes, cudaStream_t s);
void big_free(void* p, cudaStream_t s);
// The same for a block that must start zeroed: *zero says whether the block
// handed out is known to be zero over `bytes` (a cached block released with
// big_free_zeroed); otherwise the caller clears it.
cudaError_t big_alloc_zeroed(void** p, size_t bytes, cudaStream_t s, bool* zero);
void big_free_zeroed(void* p, size_t zeroed, cudaStream_t s);

// Every device allocation of the library goes through pool_alloc: a
// stream-ordered allocation from the pool above that is counted (reported by
// pkd_kernel_stats("allocations")) and that fails with
// cudaErrorMemoryAllocation, without allocating, once the option
// "fail_alloc_after" is set to k >= 0 and k allocations have succeeded since
// (host-side fault injection for the out-of-memory paths).
cudaError_t pool_alloc(void** p, size_t bytes, cudaStream_t s);

// Stream-ordered allocation from that pool.
template <class T>
int dalloc(T** p, size_t n, cudaStream_t s) {
  *p = nullptr;
  if (n == 0) n = 1;
  cudaError_t e = pool_alloc((void**)p, n * sizeof(T), s);
  if (e == cudaErrorMemoryAllocation) {
    cudaGetLastError();
    return PKD_ENOMEM;
  }
  return e == cudaSuccess ? PKD_OK : cuda_err(e);
}
template <class T>
void dfree(T*& p, cudaStream_t s) {
  if (p) cudaFreeAsync(p, s);
  p = nullptr;
}

// Scratch buffers of one call, freed in stream order when it returns.  Small
// buffers are cut from blocks of BLOCK bytes: an update asks for a few hundred
// of them, at about 1.5 us of host time each when every one was an allocation.
struct Scratch {
  static constexpr size_t BLOCK = 256 << 10;
  cudaStream_t s;
  std::vector<void*> ptrs;   // every buffer handed out, in order
  std::vector<void*> owned;  // what has to be freed
  char* cur = nullptr;
  size_t left = 0;
  ~Scratch() {
    for (void* p : owned) cudaFreeAsync(p, s);
  }
  template <class T>
  int get(T** p, size_t n) {
    *p = nullptr;
    const size_t bytes = (std::max<size_t>(n, 1) * sizeof(T) + 255) & ~(size_t)255;
    char* q = nullptr;
    if (bytes > BLOCK / 4) {
      const int e = dalloc(&q, bytes, s);
      if (e != PKD_OK) return e;
      owned.push_back(q);
    } else {
      if (left < bytes) {
        const int e = dalloc(&cur, BLOCK, s);
        left = e == PKD_OK ? BLOCK : 0;
        if (e != PKD_OK) return e;
        owned.push_back(cur);
      }
      q = cur;
      cur += bytes;
      left -= bytes;
    }
    *p = (T*)q;
    ptrs.push_back(q);
    return PKD_OK;
  }
};

// Pinned host blocks of PINNED_BLOCK bytes from a library-owned pool that
// grows by whole chunks and is never returned (pinning and unpinning memory
// are slow, synchronising driver calls).  nullptr when pinning fails.
constexpr size_t PINNED_BLOCK = 256;
void* pinned_get();
void pinned_put(void* p);

// A pinned block of PINNED_BLOCK bytes owned by one scope.  Whoever lets the
// device write to it waits for that write before the scope ends: the block
// goes straight back to the pool.  (Handing it back by a host function queued
// on the stream held the stream for about 25 us, twice in a build.)
struct PinnedBlock {
  void* p = nullptr;
  PinnedBlock() : p(pinned_get()) {}
  ~PinnedBlock() { pinned_put(p); }
  PinnedBlock(const PinnedBlock&) = delete;
  PinnedBlock& operator=(const PinnedBlock&) = delete;
};

// Reads the device status word; PKD_OK or the mapped error.
int check_status(TreeMem& t, cudaStream_t s);
int status_code(int err, int detail);

// Kernel timing (CUDA events on the launching stream).
struct KTimer {
  bool on = false;
  cudaEvent_t a = nullptr, b = nullptr;
  std::string name;
  uint64_t items = 0;
  cudaStream_t s = nullptr;
};
void ktimer_begin(KTimer& k, const char* name, uint64_t items, cudaStream_t s);
void ktimer_end(KTimer& k);
bool ktiming_enabled();
// While timing is on, add `items` to the counter family `name` (a count
// with no kernel time, e.g. the points a batch update rebuilt).
void stat_items(const char* name, uint64_t items);
// A host-side duration (ms) under a timer family (e.g. recording a graph).
void stat_host_ms(const char* name, double ms, uint64_t items);

// A build of independent subproblems ("segments"): every segment's points
// sit at arena positions [start, start+len) of A (or of the caller's input
// when `input_coords` is set), its root goes to node slot `root`, its depth
// salts the samples.  On return each segment's points are in A in leaf order
// and its subtree is written to the node arrays.
struct BuildJob {
  const int32_t* input_coords = nullptr;  // point-major input (segments IN_INPUT)
  const uint32_t* input_ids = nullptr;
  uint64_t base = 0;       // lowest arena position of any segment
  uint64_t extent = 0;     // highest position + 1 - base
  std::vector<Seg> segs;   // host list of root segments, or:
  const Seg* dsegs = nullptr;  // device list of root segments (dsegs_n of them)
  uint64_t dsegs_n = 0;
  uint64_t max_len = 0;    // longest segment, when the caller knows it (0: unknown)
  // Called once on the host when the shared-memory base cases have been
  // queued or recorded (work that should overlap them, which are bound by
  // instruction issue rather than memory traffic, is queued from here).  The
  // argument is an event that completes when they may start (null: the work
  // queued so far on the stream).
  std::function<void(cudaEvent_t)> before_base;
};
int run_build(TreeMem& t, const BuildJob& job, cudaStream_t s);

// Waits for the whole device, never while another thread records a graph
// (CUDA forbids that: the wait fails and ends the recording).
cudaError_t device_wait();

// Builds whose rounds ran from one graph launch (since the library was loaded).
int graph_builds();
// ... of them, the builds that launched a graph recorded by an earlier build.
int graph_reuses();

// True while this host thread records a CUDA graph (kernel timers are off).
bool& flow_capturing();

// Derived shared-memory capacities.
int base_cap_for(int d);
int skel_cap_for(int d);

}  // namespace pkd
