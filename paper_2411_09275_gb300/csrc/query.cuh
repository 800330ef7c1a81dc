// Shared by the query kernels (knn.cu, query.cu): their arguments, and the
// depth-first stacks' memory.
#pragma once

#include <algorithm>

#include "engine.hpp"
#include "tree_impl.hpp"

namespace pkd {

constexpr int QSTACK = 128;    // trees of height below QSTACK - 2: stacks in shared memory
constexpr int QTHREADS = 128;

struct QueryArgs {
  const Node* nodes;
  const uint8_t* ndim;
  Pts A;
  uint32_t root;
  const int32_t* q;
  const int32_t* hi;
  uint64_t nq;
  int k;
  uint32_t* out_ids;
  int64_t* out_d2;
  uint64_t* out_cnt;
  DevStatus* st;
  const int32_t* box;  // stored bounding boxes (node slot * 2d), or null
  unsigned long long call;  // the search does nothing when this call was refused (0: checked before)
  int slot;                 // where its refusal stands
  int cap;             // stack entries per query
  bool given_offsets;  // report: the offsets are the caller's (no verdict on the tree when they do not fit)
  uint32_t* deep;      // deep trees: the queries' stacks, one after another
};

// The checks in front of a query: the coordinates' range (c1, and c2 unless
// null) and the tree's status word, in one kernel.  The search is queued right
// behind it and does nothing when the check refuses the call; the host waits
// for the check alone, so it costs the search one kernel instead of a round
// trip to the host (a fill, a kernel, two copies and two waits before: 45 us
// in front of the search, now about 5).
// The refusal is the call's number in a slot of the status block that no other
// call on the tree holds until this one returns, and a refused call returns
// after its search.  (An accepted call's search may still run by then: it only
// looks for its own number.)  With every slot taken the host waits for the check
// before the search is queued.
struct QueryHost {  // written by the check into pinned memory
  int err, detail, bad;
};
class QueryCheck {
 public:
  QueryCheck(TreeMem& tree, cudaStream_t stream) : t(tree), s(stream) {}
  ~QueryCheck();
  QueryCheck(const QueryCheck&) = delete;
  QueryCheck& operator=(const QueryCheck&) = delete;
  int begin(const int32_t* c1, uint64_t n1, const int32_t* c2, uint64_t n2);
  int end();  // waits for the check: PKD_OK, PKD_EINVAL or the tree's error
  unsigned long long call = 0;
  int slot = -1;

 private:
  int verdict();
  TreeMem& t;
  cudaStream_t s;
  bool ended = false;
  volatile QueryHost* h = nullptr;
  cudaEvent_t ev = nullptr;
};
// PKD_OK, or the error for a stream that is being captured: before anything is
// recorded on it, as a call that waits for the stream could not return anything
// else (and a graph must not keep the call's pinned blocks).
int refuse_capture(cudaStream_t s);

// In the searches: was the call refused?  (The same answer in all lanes.)
__device__ __forceinline__ bool query_refused(const QueryArgs& a) {
  const bool no = a.call && (pkd_failed(a.st) || *(volatile const unsigned long long*)&a.st->refused[a.slot] == a.call);
  return __any_sync(0xffffffffu, no);
}

#define PKD_QDISPATCH(d, F, ...)      \
  switch (d) {                        \
    case 1: F<1>(__VA_ARGS__); break; \
    case 2: F<2>(__VA_ARGS__); break; \
    case 3: F<3>(__VA_ARGS__); break; \
    case 4: F<4>(__VA_ARGS__); break; \
    case 5: F<5>(__VA_ARGS__); break; \
    case 6: F<6>(__VA_ARGS__); break; \
    case 7: F<7>(__VA_ARGS__); break; \
    default: F<8>(__VA_ARGS__); break; \
  }

// A depth-first search holds at most one waiting sibling per level.
inline bool query_height_ok(const TreeMem& t) {
  return t.st_host && t.st_host->max_depth + 2 < (uint32_t)QSTACK;
}
inline int query_stack_cap(const TreeMem& t) { return (int)((t.st_host->max_depth + 3) & ~1u); }

// Runs fn(args, first query) over the queries of `a`: one call with the
// stacks in shared memory, or, for a tree too deep for that, chunks of
// queries whose stacks (`words` 32-bit words per entry, `extra` entries more
// than the height) live in a global scratch buffer of at most DEEP_SCRATCH
// bytes.
constexpr uint64_t DEEP_SCRATCH = 1ull << 30;

template <class F>
int for_query_chunks(const TreeMem& t, const QueryArgs& a, int words, int extra, cudaStream_t s, F&& fn) {
  if (!t.st_host || t.st_host->max_depth > (1u << 30)) return PKD_EINTERNAL;
  QueryArgs ac = a;
  ac.cap = query_stack_cap(t) + extra;
  if (query_height_ok(t)) {
    fn(ac, 0);
    return PKD_OK;
  }
  const uint64_t per = (uint64_t)ac.cap * (uint64_t)words;
  const uint64_t chunk = std::max<uint64_t>(1, std::min<uint64_t>(a.nq, DEEP_SCRATCH / (4 * per)));
  uint32_t* deep = nullptr;
  PKD_TRY_(dalloc(&deep, chunk * per, s));
  for (uint64_t c0 = 0; c0 < a.nq; c0 += chunk) {
    ac.nq = std::min<uint64_t>(chunk, a.nq - c0);
    ac.q = a.q + c0 * (uint64_t)t.p.d;
    if (a.hi) ac.hi = a.hi + c0 * (uint64_t)t.p.d;
    ac.deep = deep;
    fn(ac, c0);
  }
  dfree(deep, s);
  return PKD_OK;
}

// Launches a kernel with `smb` bytes of dynamic shared memory (above 48 KiB
// only for trees of a height far above the usual).
template <auto K, class... A>
void launch_query(uint64_t blocks, size_t smb, cudaStream_t s, A... args) {
  if (smb > 48 * 1024) allow_smem<K>(smb);
  PKD_LAUNCH((K<<<(unsigned)blocks, QTHREADS, smb, s>>>(args...)));
}

}  // namespace pkd
