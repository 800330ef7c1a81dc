// Range count and range report (Sec. 5 "Queries" of the paper): the subtrees
// that meet the box are searched from the root; a subtree whose subspace lies
// inside the box adds its stored size (count) or all of its points (report).
//
// One warp answers one box: its lanes test up to 32 waiting nodes at once,
// and up to four leaves at once, eight lanes each (eight points of a
// coordinate are one 32-byte sector).  No subspace is stored: a child meets
// the box exactly when its parent does and the box reaches its side of the
// splitter, and it lies inside the box once every one of the 2d faces has
// been passed by a splitter, so a waiting node is its slot and a mask of the
// faces still to pass.
//
// What bounds it: the loads' latency (a window of 32 nodes, then its leaves,
// is one chain of dependent loads; the boxes' warps overlap theirs).  One
// thread per box (before) walked node after node with the subspace's 2d
// bounds in a local-memory stack; 1e4 boxes of about 300 points in 3e6
// clustered 2-D points: count 0.45-0.60 -> 0.033 ms, report 3.2 -> 0.13 ms.
#include <atomic>

#include "coords.cuh"
#include "query.cuh"

namespace pkd {

// Waiting nodes of a box: windows of 32 while at most RANGE_WIDE wait, one at
// a time above (depth first, at most one more per level), so RANGE_EXTRA
// entries more than the height always suffice.
constexpr int RANGE_WIDE = 256, RANGE_EXTRA = RANGE_WIDE + 32;

// What a lane finds out about its node.
struct RangeNode {
  Node nd;
  int dm;       // split dimension (inner nodes)
  bool leaf, inner;
  bool inside;  // every point lies in the box (leaf, or any node when counting)
  bool go_l, go_r;
  uint32_t ml, mr;  // the children's masks
};

// Face masks: bit j while the subspace may reach below lo[j], bit 16 + j
// while it may reach above hi[j].  lo_lane / hi_lane: lane j's bounds.
template <int D>
__device__ __forceinline__ uint32_t range_root_mask(int32_t lo_lane, int32_t hi_lane, int lane) {
  const unsigned below = __ballot_sync(0xffffffffu, lane < D && lo_lane > 0);
  const unsigned above = __ballot_sync(0xffffffffu, lane < D && hi_lane < PKD_COORD_LIMIT - 1);
  return below | (above << 16);
}

template <int D>
__device__ __forceinline__ RangeNode range_node(const QueryArgs& a, bool on, uint32_t v, uint32_t mask, int32_t lo_lane,
                                                int32_t hi_lane) {
  constexpr unsigned FULL = 0xffffffffu;
  RangeNode r{};
  if (on) {
    r.nd = a.nodes[v];
    r.dm = a.ndim[v];
  }
  if (a.box) {  // the tight box of the node's points decides earlier than the splitters
    bool out = false, in = true;
#pragma unroll
    for (int j = 0; j < D; ++j) {
      const int32_t lo = __shfl_sync(FULL, lo_lane, j), hi = __shfl_sync(FULL, hi_lane, j);
      if (on) {
        const int32_t blo = a.box[(uint64_t)v * 2 * D + j], bhi = a.box[(uint64_t)v * 2 * D + D + j];
        out |= (bhi < lo) | (blo > hi) | (bhi < blo);
        in &= (blo >= lo) & (bhi <= hi);
      }
    }
    if (out) on = false;
    if (in) mask = 0;
  }
  r.leaf = on && r.dm == PKD_LEAF;
  r.inner = on && r.dm != PKD_LEAF;
  r.inside = on && mask == 0;
  const int j = r.inner ? r.dm : 0;
  const int32_t lo = __shfl_sync(FULL, lo_lane, j), hi = __shfl_sync(FULL, hi_lane, j);
  r.go_l = r.inner && lo < r.nd.split;
  r.go_r = r.inner && hi >= r.nd.split;
  r.ml = hi >= r.nd.split - 1 ? mask & ~(1u << (16 + j)) : mask;
  r.mr = lo <= r.nd.split ? mask & ~(1u << j) : mask;
  return r;
}

// The (g + 1)-th set bit of m, g < 4 (-1 when there are fewer).
__device__ __forceinline__ int nth_bit(unsigned m, int g) {
#pragma unroll
  for (int i = 0; i < 3; ++i)
    if (i < g) m &= m - 1;
  return m ? __ffs((int)m) - 1 : -1;
}

// Does point g of the arena lie in the box?
template <int D>
__device__ __forceinline__ bool range_in(const Pts& A, uint64_t g, const int32_t* lo, const int32_t* hi) {
  bool in = true;
#pragma unroll
  for (int j = 0; j < D; ++j) {
    const int32_t x = A.c[(uint64_t)j * A.stride + g];
    in &= (x >= lo[j]) & (x <= hi[j]);
  }
  return in;
}

#define RANGE_PROLOGUE                                                                              \
  constexpr unsigned FULL = 0xffffffffu;                                                            \
  extern __shared__ __align__(16) unsigned char sm[];                                               \
  if (query_refused(a)) return;                                                                     \
  const int lane = threadIdx.x & 31;                                                                \
  const uint64_t qi = (uint64_t)blockIdx.x * (QTHREADS / 32) + threadIdx.x / 32;                    \
  if (qi >= a.nq) return;                                                                           \
  uint2* st; /* waiting nodes: slot, mask */                                                        \
  if constexpr (DEEP) st = (uint2*)a.deep + qi * (uint64_t)a.cap;                                   \
  else st = (uint2*)sm + (size_t)(threadIdx.x / 32) * a.cap;                                        \
  int32_t lo[D], hi[D];                                                                             \
  _Pragma("unroll") for (int j = 0; j < D; ++j) {                                                   \
    lo[j] = a.q[qi * D + j];                                                                        \
    hi[j] = a.hi[qi * D + j];                                                                       \
  }                                                                                                 \
  const int32_t lo_lane = lane < D ? a.q[qi * D + lane] : 0;                                        \
  const int32_t hi_lane = lane < D ? a.hi[qi * D + lane] : 0;                                       \
  /* an empty box (hi < lo) or one without a point of the domain holds nothing */                   \
  const bool none = __any_sync(FULL, lane < D && hi_lane < lo_lane);                                \
  const uint32_t mask0 = range_root_mask<D>(lo_lane, hi_lane, lane);                                \
  if (lane == 0) st[0] = make_uint2(a.root, mask0);                                                 \
  int sp = none ? 0 : 1;                                                                            \
  __syncwarp();

template <int D, bool DEEP>
__global__ void __launch_bounds__(QTHREADS) k_range_count(QueryArgs a) {
  RANGE_PROLOGUE
  const int g = lane >> 3, gl = lane & 7;  // four leaves at once
  unsigned long long cnt = 0;              // per lane
  while (sp > 0) {
    const int p = sp > RANGE_WIDE ? 1 : min(sp, 32);
    const uint2 e = lane < p ? st[sp - 1 - lane] : make_uint2(0, 0);
    __syncwarp();  // read before the entries are written again
    const RangeNode r = range_node<D>(a, lane < p, e.x, e.y, lo_lane, hi_lane);
    if (r.inside) cnt += r.nd.size;
    const unsigned bl = __ballot_sync(FULL, r.go_l && !r.inside), br = __ballot_sync(FULL, r.go_r && !r.inside);
    const unsigned under = (1u << lane) - 1u;
    sp -= p;
    if (sp + __popc(bl) + __popc(br) > a.cap) {
      if (lane == 0) set_error(a.st, DERR_STACK, 901);
      break;
    }
    if (bl >> lane & 1) st[sp + __popc(bl & under)] = make_uint2(r.nd.a, r.ml);
    sp += __popc(bl);
    if (br >> lane & 1) st[sp + __popc(br & under)] = make_uint2(r.nd.b, r.mr);
    sp += __popc(br);
    unsigned lv = __ballot_sync(FULL, r.leaf && !r.inside);
    while (lv) {
      const int src = nth_bit(lv, g);
      const uint32_t la = __shfl_sync(FULL, r.nd.a, src & 31);
      uint32_t ls = __shfl_sync(FULL, r.nd.size, src & 31);
      if (src < 0) ls = 0;
#pragma unroll
      for (int i = 0; i < 4; ++i) lv &= lv - 1;
      for (uint32_t b = gl; b < ls; b += 32) {  // no collective inside: the groups may part
        bool in[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) in[u] = b + 8 * u < ls && range_in<D>(a.A, (uint64_t)la + b + 8 * u, lo, hi);
        cnt += (unsigned)in[0] + in[1] + in[2] + in[3];
      }
    }
    __syncwarp();
  }
#pragma unroll
  for (int o = 16; o; o >>= 1) cnt += __shfl_xor_sync(FULL, cnt, o);
  if (lane == 0) a.out_cnt[qi] = cnt;
}

// Range report: the ids of box qi from out_ids[offsets[qi]], in depth-first
// leaf order.  The waiting nodes stand in that order, the first on top; each
// step expands the inner nodes among the top 32 in place and writes out the
// leaves in front of the first inner node.  (A subtree inside the box is
// walked to its leaves too: after updates its points need not be contiguous
// in the arena.)
template <int D, bool DEEP>
__global__ void __launch_bounds__(QTHREADS) k_range_report(QueryArgs a, const uint64_t* offsets, uint32_t* out_ids,
                                                             uint64_t ids_cap) {
  RANGE_PROLOGUE
  const int g = lane >> 3, gl = lane & 7;
  uint64_t pos = offsets[qi];
  const uint64_t end = min(offsets[qi + 1], ids_cap);
  while (sp > 0) {
    const int p = sp > RANGE_WIDE ? 1 : min(sp, 32);
    const uint2 e = lane < p ? st[sp - 1 - lane] : make_uint2(0, 0);
    __syncwarp();  // read before the entries are written again
    const RangeNode r = range_node<D>(a, lane < p, e.x, e.y, lo_lane, hi_lane);
    // the leaves (and nodes that dropped out) in front of the first inner node
    const unsigned inner = __ballot_sync(FULL, r.inner);
    const int np = inner ? __ffs((int)inner) - 1 : p;
    const bool keep = r.leaf && lane >= np;  // a leaf whose turn has not come
    const int c = keep ? 1 : (int)r.go_l + (int)r.go_r;
    int inc = c;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int t = __shfl_up_sync(FULL, inc, o);
      if (lane >= o) inc += t;
    }
    const int total = __shfl_sync(FULL, inc, 31);
    sp += total - p;
    if (sp > a.cap) {
      if (lane == 0) set_error(a.st, DERR_STACK, 903);
      return;
    }
    int at = sp - 1 - (inc - c);
    if (keep) st[at] = e;
    if (r.go_l) st[at--] = make_uint2(r.nd.a, r.ml);
    if (r.go_r) st[at] = make_uint2(r.nd.b, r.mr);
    unsigned lv = __ballot_sync(FULL, r.leaf && lane < np);
    while (lv) {
      const int src = nth_bit(lv, g);
      const uint32_t la = __shfl_sync(FULL, r.nd.a, src & 31);
      uint32_t ls = __shfl_sync(FULL, r.nd.size, src & 31);
      const bool all = __shfl_sync(FULL, r.inside, src & 31);
      if (src < 0) ls = 0;
      const bool four = !__any_sync(FULL, ls > 32);
      if (four) {
#pragma unroll
        for (int i = 0; i < 4; ++i) lv &= lv - 1;
        uint32_t id[4];
        bool in[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          const uint32_t b = gl + 8 * u;
          in[u] = b < ls && (all || range_in<D>(a.A, (uint64_t)la + b, lo, hi));
          id[u] = b < ls ? a.A.id[(uint64_t)la + b] : 0;
        }
        // ranks: leaf by leaf (g), then eight points at a time (u)
        unsigned m[4];
        int mine = 0;
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          m[u] = __ballot_sync(FULL, in[u]);
          mine += __popc(m[u] >> (8 * g) & 0xFFu);
        }
        int before = 0, tot = 0;
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          const int t = __shfl_sync(FULL, mine, 8 * k);
          if (k < g) before += t;
          tot += t;
        }
        if (pos > end || (uint64_t)tot > end - pos) {  // more points than counted: the tree changed
          if (lane == 0 && !a.given_offsets) set_error(a.st, DERR_STATE, 902);
          return;
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          const unsigned mu = m[u] >> (8 * g) & 0xFFu;
          if (in[u]) out_ids[pos + before + __popc(mu & ((1u << gl) - 1u))] = id[u];
          before += __popc(mu);
        }
        pos += tot;
      } else {  // the first leaf alone, by the whole warp
        const uint32_t a0 = __shfl_sync(FULL, la, 0), s0 = __shfl_sync(FULL, ls, 0);
        const bool all0 = __shfl_sync(FULL, all, 0);
        lv &= lv - 1;
        for (uint32_t b0 = 0; b0 < s0; b0 += 32) {
          const uint32_t b = b0 + lane;
          const bool in = b < s0 && (all0 || range_in<D>(a.A, (uint64_t)a0 + b, lo, hi));
          const unsigned m = __ballot_sync(FULL, in);
          if (pos > end || (uint64_t)__popc(m) > end - pos) {
            if (lane == 0 && !a.given_offsets) set_error(a.st, DERR_STATE, 902);
            return;
          }
          if (in) out_ids[pos + __popc(m & ((1u << lane) - 1u))] = a.A.id[(uint64_t)a0 + b];
          pos += __popc(m);
        }
      }
    }
    __syncwarp();
  }
}

// Exclusive scan of q 64-bit counts into offsets[0..q] (offsets[q] = total,
// also stored to host_total): one block for up to SCAN64_ONE counts (a launch
// instead of three and, with the total stored to pinned memory, no copy back),
// else per-block sums, one block over the sums, then the blocks again.
constexpr int SCAN64_THREADS = 256, SCAN64_PER = 8, SCAN64_TILE = SCAN64_THREADS * SCAN64_PER;
constexpr uint64_t SCAN64_ONE = 16 * SCAN64_TILE;

__device__ __forceinline__ uint64_t block_scan64(uint64_t v, uint64_t* sh, uint64_t* total) {
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  uint64_t inc = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint64_t t = __shfl_up_sync(0xffffffffu, inc, o);
    if (lane >= o) inc += t;
  }
  if (lane == 31) sh[w] = inc;
  __syncthreads();
  uint64_t before = 0, tot = 0;
  for (int k = 0; k < SCAN64_THREADS / 32; ++k) {
    if (k < w) before += sh[k];
    tot += sh[k];
  }
  __syncthreads();
  *total = tot;
  return before + inc - v;
}

__global__ void k_scan64_reduce(const uint64_t* in, uint64_t n, uint64_t* partial) {
  __shared__ uint64_t sh[SCAN64_THREADS / 32];
  const uint64_t base = (uint64_t)blockIdx.x * SCAN64_TILE + (uint64_t)threadIdx.x * SCAN64_PER;
  uint64_t s = 0;
  for (int k = 0; k < SCAN64_PER; ++k)
    if (base + k < n) s += in[base + k];
  uint64_t tot;
  block_scan64(s, sh, &tot);
  if (threadIdx.x == 0) partial[blockIdx.x] = tot;
}

__global__ void k_scan64_partials(uint64_t* partial, uint64_t nb) {
  __shared__ uint64_t sh[SCAN64_THREADS / 32];
  uint64_t carry = 0;
  for (uint64_t b0 = 0; b0 < nb; b0 += SCAN64_THREADS) {
    const uint64_t i = b0 + threadIdx.x;
    const uint64_t v = i < nb ? partial[i] : 0;
    uint64_t tot;
    const uint64_t ex = block_scan64(v, sh, &tot);
    if (i < nb) partial[i] = carry + ex;
    carry += tot;
  }
  if (threadIdx.x == 0) partial[nb] = carry;
}

// Tile blockIdx.x + k * gridDim.x of the scan; `partial` null: one block over all tiles.
__global__ void k_scan64_apply(QueryArgs a, const uint64_t* in, uint64_t n, const uint64_t* partial, uint64_t* out,
                               uint64_t* host_total) {
  __shared__ uint64_t sh[SCAN64_THREADS / 32];
  if (__syncthreads_or(threadIdx.x < 32 && query_refused(a))) return;  // no counts were written
  uint64_t carry = partial ? partial[blockIdx.x] : 0;
  for (uint64_t tile = blockIdx.x; tile * SCAN64_TILE < n; tile += gridDim.x) {
    const uint64_t base = tile * SCAN64_TILE + (uint64_t)threadIdx.x * SCAN64_PER;
    uint64_t v[SCAN64_PER], s = 0;
    for (int k = 0; k < SCAN64_PER; ++k) {
      v[k] = base + k < n ? in[base + k] : 0;
      s += v[k];
    }
    uint64_t tot;
    uint64_t run = carry + block_scan64(s, sh, &tot);
    for (int k = 0; k < SCAN64_PER; ++k) {
      if (base + k < n) out[base + k] = run;
      run += v[k];
    }
    carry += tot;
  }
  if (blockIdx.x == gridDim.x - 1 && threadIdx.x == 0) {
    out[n] = carry;
    *(volatile uint64_t*)host_total = carry;
  }
}

__global__ void k_query_check(const int32_t* c1, uint64_t n1, const int32_t* c2, uint64_t n2, DevStatus* st,
                              unsigned long long call, int slot, QueryHost* h) {
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    h->err = st->err;
    h->detail = st->detail;
  }
  const unsigned b = coord_bits(c1, n1) | (c2 ? coord_bits(c2, n2) : 0);
  if (__any_sync(0xffffffffu, (b >> 30) != 0) && (threadIdx.x & 31) == 0) {
    if (slot >= 0) *(volatile unsigned long long*)&st->refused[slot] = call;
    *(volatile int*)&h->bad = 1;
  }
}

int refuse_capture(cudaStream_t s) {
  cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
  PKD_CUDA(cudaStreamIsCapturing(s, &cap));
  if (cap == cudaStreamCaptureStatusNone) return PKD_OK;
  const cudaError_t e = cudaStreamSynchronize(s);  // ends the capture with an error
  cudaGetLastError();
  return e != cudaSuccess ? cuda_err(e) : PKD_ECUDA;
}

int QueryCheck::begin(const int32_t* c1, uint64_t n1, const int32_t* c2, uint64_t n2) {
  static std::atomic<unsigned long long> calls{0};
  PKD_TRY_(refuse_capture(s));
  h = (volatile QueryHost*)pinned_get();
  if (!h) return PKD_ENOMEM;
  h->bad = 0;
  call = ++calls;
  uint32_t held = __atomic_load_n(&t.query_slots, __ATOMIC_RELAXED);
  while (~held & ((1u << QUERY_SLOTS) - 1u)) {
    const int k = __builtin_ctz(~held);
    if (__atomic_compare_exchange_n(&t.query_slots, &held, held | 1u << k, true, __ATOMIC_ACQUIRE, __ATOMIC_RELAXED)) {
      slot = k;
      break;
    }
  }
  KTimer kt;
  ktimer_begin(kt, "validate", n1 + (c2 ? n2 : 0), s);
  PKD_LAUNCH(k_query_check<<<coord_blocks(n1), 256, 0, s>>>(c1, n1, c2, n2, t.st, call, slot, (QueryHost*)h));
  ktimer_end(kt);
  if (cudaEventCreateWithFlags(&ev, cudaEventDisableTiming) != cudaSuccess || cudaEventRecord(ev, s) != cudaSuccess) {
    cudaGetLastError();
    PKD_CUDA(cudaStreamSynchronize(s));
    if (ev) cudaEventDestroy(ev);
    ev = nullptr;
  }
  test_pause(PAUSE_QUERY);
  if (slot < 0) {
    call = 0;
    return verdict();
  }
  return PKD_OK;
}

int QueryCheck::verdict() {
  if (ev) PKD_CUDA(cudaEventSynchronize(ev));
  if (h->bad) return PKD_EINVAL;
  return status_code(h->err, h->detail);
}

int QueryCheck::end() {
  const int e = verdict();
  if (slot >= 0 && h->bad) PKD_CUDA(cudaStreamSynchronize(s));  // the search has read its slot
  ended = true;
  return e;
}

QueryCheck::~QueryCheck() {
  if (ev) {
    cudaEventSynchronize(ev);  // the check writes to the block until then
    cudaEventDestroy(ev);
  }
  if (slot >= 0) {
    if (!ended) cudaStreamSynchronize(s);
    __atomic_fetch_and(&t.query_slots, ~(1u << slot), __ATOMIC_RELEASE);
  }
  if (h) pinned_put((void*)h);
}

template <int D>
static void launch_report(const QueryArgs& a, const uint64_t* offsets, uint32_t* ids, uint64_t ids_cap,
                          cudaStream_t s) {
  constexpr int WPB = QTHREADS / 32;
  const uint64_t g = (a.nq + WPB - 1) / WPB;
  KTimer kt;
  ktimer_begin(kt, "range_report", a.nq, s);
  if (a.deep) launch_query<k_range_report<D, true>>(g, 0, s, a, offsets, ids, ids_cap);
  else launch_query<k_range_report<D, false>>(g, (size_t)WPB * a.cap * sizeof(uint2), s, a, offsets, ids,
                    ids_cap);
  ktimer_end(kt);
}

template <int D>
static void launch_rc(const QueryArgs& a, cudaStream_t s) {
  constexpr int WPB = QTHREADS / 32;
  const uint64_t g = (a.nq + WPB - 1) / WPB;
  KTimer kt;
  ktimer_begin(kt, "range_count", a.nq, s);
  if (a.deep) launch_query<k_range_count<D, true>>(g, 0, s, a);
  else launch_query<k_range_count<D, false>>(g, (size_t)WPB * a.cap * sizeof(uint2), s, a);
  ktimer_end(kt);
}

}  // namespace pkd

using namespace pkd;

namespace {

// A box query's arguments.
QueryArgs range_args(const TreeMem& t, const QueryCheck& check, const int32_t* lo, const int32_t* hi, uint64_t q) {
  QueryArgs a{};
  a.call = check.call;
  a.slot = check.slot;
  a.nodes = t.nodes;
  a.ndim = t.ndim;
  a.A = t.A;
  a.root = t.root;
  a.q = lo;
  a.hi = hi;
  a.nq = q;
  a.st = t.st;
  a.box = t.bbox_on ? t.bbox : nullptr;
  return a;
}

int range_counts(const TreeMem& t, const QueryArgs& a, uint64_t* counts, cudaStream_t s) {
  return for_query_chunks(t, a, 2, RANGE_EXTRA, s, [&](QueryArgs ac, uint64_t c0) {
    ac.out_cnt = counts + c0;
    PKD_QDISPATCH(t.p.d, launch_rc, ac, s);
  });
}

int range_ids(const TreeMem& t, const QueryArgs& a, const uint64_t* offsets, uint32_t* ids, uint64_t cap,
              cudaStream_t s) {
  return for_query_chunks(t, a, 2, RANGE_EXTRA, s, [&](QueryArgs ac, uint64_t c0) {
    PKD_QDISPATCH(t.p.d, launch_report, ac, offsets + c0, ids, cap, s);
  });
}

}  // namespace

extern "C" {

int pkd_range_count(const pkd_tree* tc, const int32_t* lo, const int32_t* hi, uint64_t q,
                    uint64_t* out_counts, void* stream) {
  if (!tc) return PKD_EINVAL;
  if (q == 0) return PKD_OK;
  if (!lo || !hi || !out_counts) return PKD_EINVAL;
  TreeMem& t = const_cast<TreeMem&>(tc->m);
  cudaStream_t s = (cudaStream_t)stream;
  TreeTouch touch{&t, s};
  const uint64_t nc = q * (uint64_t)t.p.d;
  QueryCheck check(t, s);
  PKD_TRY_(check.begin(lo, nc, hi, nc));
  PKD_TRY_(range_counts(t, range_args(t, check, lo, hi, q), out_counts, s));
  PKD_CUDA(cudaGetLastError());
  return check.end();
}

int pkd_range_report(const pkd_tree* tc, const int32_t* lo, const int32_t* hi, uint64_t q, uint64_t* offsets,
                     uint32_t* ids, uint64_t ids_cap, uint64_t* total, void* stream) {
  if (!tc || !total) return PKD_EINVAL;
  *total = 0;
  if (q == 0) return PKD_OK;
  if (!lo || !hi || !offsets) return PKD_EINVAL;
  TreeMem& t = const_cast<TreeMem&>(tc->m);
  cudaStream_t s = (cudaStream_t)stream;
  TreeTouch touch{&t, s};
  const uint64_t nc = q * (uint64_t)t.p.d;
  QueryCheck check(t, s);
  PKD_TRY_(check.begin(lo, nc, hi, nc));
  // pass 1: counts, scanned into offsets[0..q]
  const uint64_t nb = q <= SCAN64_ONE ? 1 : (q + SCAN64_TILE - 1) / SCAN64_TILE;
  Scratch sc{s, {}};
  uint64_t *counts, *partial = nullptr;
  PKD_TRY_(sc.get(&counts, q));
  if (nb > 1) PKD_TRY_(sc.get(&partial, nb + 1));
  PinnedBlock tot;
  if (!tot.p) return PKD_ENOMEM;
  const QueryArgs a = range_args(t, check, lo, hi, q);
  PKD_TRY_(range_counts(t, a, counts, s));
  if (nb > 1) {
    PKD_LAUNCH(k_scan64_reduce<<<(unsigned)nb, SCAN64_THREADS, 0, s>>>(counts, q, partial));
    PKD_LAUNCH(k_scan64_partials<<<1, SCAN64_THREADS, 0, s>>>(partial, nb));
  }
  PKD_LAUNCH(k_scan64_apply<<<(unsigned)nb, SCAN64_THREADS, 0, s>>>(a, counts, q, partial, offsets, (uint64_t*)tot.p));
  PKD_CUDA(cudaStreamSynchronize(s));
  PKD_TRY_(check.end());  // a refused call's counts were not written
  *total = *(volatile uint64_t*)tot.p;
  if (*total > ids_cap || (*total > 0 && !ids)) return PKD_EINVAL;
  // pass 2: the ids
  PKD_TRY_(range_ids(t, a, offsets, ids, ids_cap, s));
  PKD_CUDA(cudaGetLastError());
  return PKD_OK;
}

int pkd_range_report_ids(const pkd_tree* tc, const int32_t* lo, const int32_t* hi, uint64_t q, const uint64_t* offsets,
                         uint32_t* ids, uint64_t ids_cap, void* stream) {
  if (!tc) return PKD_EINVAL;
  if (q == 0) return PKD_OK;
  if (!lo || !hi || !offsets || (ids_cap > 0 && !ids)) return PKD_EINVAL;
  TreeMem& t = const_cast<TreeMem&>(tc->m);
  cudaStream_t s = (cudaStream_t)stream;
  TreeTouch touch{&t, s};
  const uint64_t nc = q * (uint64_t)t.p.d;
  QueryCheck check(t, s);
  PKD_TRY_(check.begin(lo, nc, hi, nc));
  QueryArgs a = range_args(t, check, lo, hi, q);
  a.given_offsets = true;
  PKD_TRY_(range_ids(t, a, offsets, ids, ids_cap, s));
  PKD_CUDA(cudaGetLastError());
  return check.end();
}

}  // extern "C"
