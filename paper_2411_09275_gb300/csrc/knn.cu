// k nearest neighbours (Sec. 5 "Queries" of the paper): depth-first search,
// near child first, a subtree pruned when its subspace is strictly farther
// than the current k-th candidate.
//
// A group of G lanes answers one query: the leaf's points are spread over the
// lanes (8 lanes read one 32-byte sector per coordinate), the k best pairs
// (squared distance, id) sit sorted in the lanes' registers, S per lane, and
// the stack of waiting far children in shared memory.  One thread per query
// (before) kept all three in local memory and walked every leaf point by
// point behind dependent loads.  The subspace of a node is not stored as a
// box: lane j holds the query's offset to it in dimension j, and going to the
// far side of a splitter changes one offset, so the bound of a child is the
// parent's minus the old offset squared plus the new one squared (the same
// number as the distance to the box that the splitters imply).
//
// What bounds it: dependent loads (37% of the stalls with 4 lanes a query, 50%
// of the L1's misses hit L2, 20% of the DRAM bandwidth) and instructions (the SMs
// 60% busy, about a third of it list insertions); small batches are bound by the chain of
// dependent loads down the tree (about 20 us for one 10-NN query in 1e6 2-D
// points).  One thread per query (before) kept the stack, with the 2d bounds
// of every waiting subspace, and the k entries in local memory.  10-NN, time
// before -> now: 1e6 uniform queries in 1e7 3-D points 7.5 -> 1.85 ms; a call of
// 1e5 queries in clustered 1e7 3-D points 0.81 to 1.9 -> 0.20 to 0.62 ms by the
// draw of the points (3.0 to 4.0 times); 64 queries in 1e6 2-D points 170 -> 20
// us; 100-NN of 2000 queries in 2e5 8-D points 91 -> 2.0 ms.
#include <cstdio>
#include <mutex>

#include "query.cuh"

namespace pkd {

// (ad, ai) < (bd, bi) for distances >= 0: the borrow of a 96-bit subtraction.
__device__ __forceinline__ bool pair_less(long long ad, uint32_t ai, long long bd, uint32_t bi) {
  int32_t h;
  asm("{.reg .u32 t;\n\t"
      "sub.cc.u32 t, %1, %2;\n\t"
      "subc.cc.u32 t, %3, %4;\n\t"
      "subc.u32 %0, %5, %6;}"
      : "=r"(h)
      : "r"(ai), "r"(bi), "r"((uint32_t)ad), "r"((uint32_t)bd), "r"((uint32_t)(ad >> 32)), "r"((uint32_t)(bd >> 32)));
  return h < 0;
}

// Up to this many queries get a whole warp each when k <= 16: a leaf is then
// one step and the chip still has warps to spare.  More queries share a warp
// (4 lanes each up to d = 4, 8 above, a lane per dimension): the steps down the
// tree and the insertions of several queries run together.  10-NN in 1e7 3-D
// points, a warp against 4 lanes: 26 / 50 us at 64 queries, 54 / 60 us at
// 8000, 84 / 70 us at 16000, 268 / 168 us at 64000; 6-D, a warp against 8
// lanes: 165 / 270 us at 64, 325 / 355 us at 8000, 399 / 372 us at 16000.
// Above k = 16 the list needs the 32 lanes.
constexpr uint64_t KNN_WARP_QUERIES = 8192;

template <int D, int G, int S, bool DEEP>
__global__ void __launch_bounds__(QTHREADS) k_knn(QueryArgs a) {
  constexpr unsigned FULL = 0xffffffffu;
  constexpr unsigned GBITS = G == 32 ? FULL : (1u << (G & 31)) - 1u;
  constexpr int U = 32 / G;  // points per lane and step
  static_assert(D <= G, "a lane per dimension");
  extern __shared__ __align__(16) unsigned char sm[];
  if (query_refused(a)) return;
  const int lane = threadIdx.x & (G - 1);
  const int gshift = (threadIdx.x & 31) & ~(G - 1);
  const uint64_t qi = (uint64_t)blockIdx.x * (QTHREADS / G) + threadIdx.x / G;
  bool act = qi < a.nq;
  const int cap = a.cap;

  // the group's stack: bound, slot and offsets of every waiting child
  unsigned char* sb;
  if constexpr (DEEP) sb = (unsigned char*)(a.deep + (act ? qi : 0) * (uint64_t)cap * (3 + D));
  else sb = sm + (size_t)(threadIdx.x / G) * cap * (12 + 4 * D);
  long long* const s_lb = (long long*)sb;
  uint32_t* const s_v = (uint32_t*)(s_lb + cap);
  int32_t* const s_off = (int32_t*)(s_v + cap);

  int32_t qa[D];
#pragma unroll
  for (int j = 0; j < D; ++j) qa[j] = act ? a.q[qi * D + j] : 0;
  const int32_t q = act && lane < D ? a.q[qi * D + lane] : 0;
  int32_t off = 0;

  // position lane * S + s of the sorted list; the k real entries are the last
  // k positions, so that the k-th best is always the last lane's last entry
  // (the positions in front hold (0, 0), which no pair is below)
  long long bd[S];
  uint32_t bi[S];
#pragma unroll
  for (int s = 0; s < S; ++s) {
    const bool real = lane * S + s >= G * S - a.k;
    bd[s] = real ? LLONG_MAX : 0;
    bi[s] = real ? 0xFFFFFFFFu : 0;
  }
  long long kd = LLONG_MAX;
  uint32_t ki = 0xFFFFFFFFu;

  uint32_t v = a.root;
  long long cur = 0;
  int sp = 0;
  while (__any_sync(FULL, act)) {
    // down to a leaf, the groups of the warp level by level together
    Node nd{};
    bool inner = false;
    int dm = 0;
    if (act) {
      nd = a.nodes[v];
      dm = a.ndim[v];
      inner = dm != PKD_LEAF;
    }
    while (__any_sync(FULL, inner)) {
      const int j = inner ? dm : 0;
      const int32_t qd = __shfl_sync(FULL, q, j, G), od = __shfl_sync(FULL, off, j, G);
      if (inner) {
        const bool left = qd < nd.split;
        const int32_t no = left ? nd.split - qd : qd - (nd.split - 1);
        const uint32_t far = left ? nd.b : nd.a;
        v = left ? nd.a : nd.b;
        const long long fd = cur - (long long)od * od + (long long)no * no;
        nd = a.nodes[v];
        dm = a.ndim[v];
        if (fd <= kd) {
          if (sp >= cap) {
            set_error(a.st, DERR_STACK, 900);
            act = false;
          } else {
            if (lane == 0) {
              s_lb[sp] = fd;
              s_v[sp] = far;
            }
            if (lane < D) s_off[sp * D + lane] = lane == j ? no : off;
            ++sp;
          }
        }
        inner = act && dm != PKD_LEAF;
      }
    }
    // the leaf's points, U per lane at a time
    const uint32_t size = act ? nd.size : 0;
    for (uint32_t base = 0; __any_sync(FULL, base < size); base += G * U) {
      long long d2[U];
      uint32_t id[U];
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const uint32_t i = base + u * G + lane;
        d2[u] = LLONG_MAX;
        id[u] = 0xFFFFFFFFu;
        if (i < size) {
          const uint64_t g = (uint64_t)nd.a + i;
          long long t2 = 0;
#pragma unroll
          for (int j = 0; j < D; ++j) {
            const long long t = a.A.c[(uint64_t)j * a.A.stride + g] - qa[j];
            t2 += t * t;
          }
          d2[u] = t2;
          id[u] = a.A.id[g];
        }
      }
#pragma unroll
      for (int u = 0; u < U; ++u) {
        bool better = pair_less(d2[u], id[u], kd, ki);
        unsigned m = __ballot_sync(FULL, better);
        while (m) {  // one candidate of every group that has one
          const unsigned gm = (m >> gshift) & GBITS;
          const int src = gm ? __ffs((int)gm) - 1 : 0;
          long long cd = __shfl_sync(FULL, d2[u], src, G);
          uint32_t ci = __shfl_sync(FULL, id[u], src, G);
          if (!gm) {  // goes behind every entry: no change
            cd = LLONG_MAX;
            ci = 0xFFFFFFFFu;
          }
          if (lane == src) better = false;
          const long long pd = __shfl_up_sync(FULL, bd[S - 1], 1, G);
          const uint32_t pi = __shfl_up_sync(FULL, bi[S - 1], 1, G);
          bool lt = pair_less(cd, ci, bd[S - 1], bi[S - 1]);
#pragma unroll
          for (int s = S - 1; s > 0; --s) {
            const bool ltp = pair_less(cd, ci, bd[s - 1], bi[s - 1]);
            if (lt) {
              bd[s] = ltp ? bd[s - 1] : cd;
              bi[s] = ltp ? bi[s - 1] : ci;
            }
            lt = ltp;
          }
          const bool ltp = lane > 0 && pair_less(cd, ci, pd, pi);
          if (lt) {
            bd[0] = ltp ? pd : cd;
            bi[0] = ltp ? pi : ci;
          }
          kd = __shfl_sync(FULL, bd[S - 1], G - 1, G);
          ki = __shfl_sync(FULL, bi[S - 1], G - 1, G);
          better = better && pair_less(d2[u], id[u], kd, ki);
          m = __ballot_sync(FULL, better);
        }
      }
    }
    // the waiting child on top that can still hold a neighbour: the lanes
    // test G entries at once
    bool need = act;
    __syncwarp();
    while (__any_sync(FULL, need)) {
      const int e = sp - 1 - lane;
      const long long lb = need && e >= 0 ? s_lb[e] : LLONG_MAX;
      const bool can = need && e >= 0 && lb <= kd;
      const unsigned gm = (__ballot_sync(FULL, can) >> gshift) & GBITS;
      if (need) {
        if (gm) {
          sp -= __ffs((int)gm);
          cur = s_lb[sp];
          v = s_v[sp];
          if (lane < D) off = s_off[sp * D + lane];
          need = false;
        } else {
          sp -= G;
          if (sp <= 0) act = need = false;
        }
      }
      if (a.box) {  // the tight box of its points may be farther than its subspace
        const bool test = act && !need && lane < D;
        int32_t lo = 0, hi = 0;
        if (test) {
          const int32_t* p = a.box + (uint64_t)v * 2 * D;
          lo = p[lane];
          hi = p[D + lane];
        }
        long long t = test ? (q < lo ? lo - q : (q > hi ? q - hi : 0)) : 0;
        t *= t;
        if (lo > hi) t = LLONG_MAX >> 4;  // an empty subtree: past every distance, without overflow in the sum
#pragma unroll
        for (int o = 1; o < 8 && o < G; o <<= 1) t += __shfl_xor_sync(FULL, t, o, G);
        t = __shfl_sync(FULL, t, 0, G);
        if (act && !need && t > kd) need = true;
      }
    }
    __syncwarp();
  }
  if (qi < a.nq) {
#pragma unroll
    for (int s = 0; s < S; ++s) {
      const int p = lane * S + s - (G * S - a.k);
      if (p >= 0) {
        a.out_d2[qi * a.k + p] = bd[s];
        a.out_ids[qi * a.k + p] = bi[s];
      }
    }
  }
}

// The k-NN kernel for k neighbours of a.nq queries.
template <int D, int G, int S, bool DEEP>
static void launch_knn_as(const QueryArgs& a, cudaStream_t s) {
  constexpr int GPB = QTHREADS / G;
  launch_query<k_knn<D, G, S, DEEP>>((a.nq + GPB - 1) / GPB, DEEP ? 0 : (size_t)GPB * a.cap * (12 + 4 * D), s, a);
}
template <int D, bool DEEP>
static void launch_knn_(const QueryArgs& a, cudaStream_t s) {
  constexpr int G = D <= 4 ? 4 : 8;
  if (!DEEP && a.k <= 16 && a.nq > KNN_WARP_QUERIES) {
    if (a.k <= G) launch_knn_as<D, G, 1, false>(a, s);
    else if (D <= 4 && a.k <= 12) launch_knn_as<D, G, D <= 4 ? 3 : 2, false>(a, s);
    else launch_knn_as<D, G, 16 / G, false>(a, s);
  } else if (a.k <= 32) launch_knn_as<D, 32, 1, DEEP>(a, s);
  else if (a.k <= 64) launch_knn_as<D, 32, 2, DEEP>(a, s);
  else launch_knn_as<D, 32, 4, DEEP>(a, s);
}
template <int D>
static void launch_knn_any(const QueryArgs& a, cudaStream_t s) {
  if (a.deep) launch_knn_<D, true>(a, s);
  else launch_knn_<D, false>(a, s);
}
template <int D>
static void launch_knn(const QueryArgs& a, cudaStream_t s) {
  KTimer kt;
  ktimer_begin(kt, "knn", a.nq, s);
  launch_knn_any<D>(a, s);
  ktimer_end(kt);
}

}  // namespace pkd

using namespace pkd;

extern "C" {

int pkd_knn(const pkd_tree* tc, const int32_t* queries, uint64_t q, int k, uint32_t* out_ids,
            int64_t* out_d2, void* stream) {
  if (!tc) return PKD_EINVAL;
  TreeMem& t = const_cast<TreeMem&>(tc->m);
  return knn_on(t, t.root, queries, q, k, out_ids, out_d2, (cudaStream_t)stream);
}

}  // extern "C"

int pkd::knn_on(TreeMem& t, uint32_t root, const int32_t* queries, uint64_t q, int k, uint32_t* out_ids,
                int64_t* out_d2, cudaStream_t s) {
  if (k < 1 || k > 128) return PKD_EINVAL;
  if (q == 0) return PKD_OK;
  if (!queries || !out_ids || !out_d2) return PKD_EINVAL;
  TreeTouch touch{&t, s};
  QueryCheck check(t, s);
  PKD_TRY_(check.begin(queries, q * (uint64_t)t.p.d, nullptr, 0));
  QueryArgs a{};
  a.call = check.call;
  a.slot = check.slot;
  a.nodes = t.nodes;
  a.ndim = t.ndim;
  a.A = t.A;
  a.root = root;
  a.q = queries;
  a.nq = q;
  a.k = k;
  a.out_ids = out_ids;
  a.out_d2 = out_d2;
  a.st = t.st;
  a.box = (t.bbox_on && root == t.root) ? t.bbox : nullptr;
  PKD_TRY_(for_query_chunks(t, a, t.p.d + 3, 0, s, [&](QueryArgs ac, uint64_t c0) {
    ac.out_ids = out_ids + c0 * (uint64_t)k;
    ac.out_d2 = out_d2 + c0 * (uint64_t)k;
    PKD_QDISPATCH(t.p.d, launch_knn, ac, s);
  }));
  PKD_CUDA(cudaGetLastError());
  return check.end();
}


// ----------------------------------------------------------------------------
// k-NN ids without any allocation (the paper has no counterpart)
// ----------------------------------------------------------------------------
// pkd_knn takes a status word from the library's memory pool for its
// coordinate check and needs a caller buffer for the distances.  Some callers
// can do neither: a server that has handed all spare device memory to its
// trees and may not let a pool grow while a request is in flight, or one that
// needs the latency of a query call free of allocator and mapping work.  This
// variant keeps both in a fixed scratch array compiled into the library:
//
//   bytes [0, 4)                          coordinate-check flag; must be zero
//                                         when the check kernel starts (each
//                                         call clears it on its stream first)
//   bytes [256, 256 + 8 * q * k)          the k distances of every query; no
//                                         initial value needed (written by
//                                         the search before anything reads it)
//
// The scratch is one array per device, shared by every call: two calls whose
// work overlaps on the device (different streams, or different host threads)
// race on it.  Calls issued one after the other on one stream are ordered.
// The first call on a device is the set-up: it resolves the array's address
// and launches every kernel the call uses once on an empty query set, which
// loads them and lets the driver size its local-memory reservation for the
// largest; make that call before any region in which the caller may not
// allocate.

namespace pkd {

static __device__ __align__(256) unsigned char g_knn_noalloc_scratch[256 + 8 * (uint64_t)PKD_NOALLOC_MAX_PAIRS];

__global__ void k_noalloc_check(const int32_t* c, uint64_t cnt, unsigned* bad) {
  uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
  int b = 0;
  for (; i < cnt; i += stride) {
    const int32_t v = c[i];
    b |= (v < 0) | (v >= PKD_COORD_LIMIT);
  }
  if (__any_sync(0xffffffffu, b) && (threadIdx.x & 31) == 0) atomicOr(bad, 1u);
}

constexpr int NOALLOC_MAX_DEVICES = 64;
static std::mutex g_noalloc_mu;
static unsigned char* g_noalloc_ptr[NOALLOC_MAX_DEVICES] = {};

// Every kernel this entry point can launch, run once on an empty query set:
// under lazy module loading a kernel's first launch loads it, and a kernel
// with more local memory per thread than any launched before makes the driver
// enlarge the device's local-memory reservation.  Both must happen in the
// set-up, not in a later call.
template <int D, int G, int S>
static void noalloc_warm_as(cudaStream_t s) {
  QueryArgs a{};
  a.nq = 0;
  a.k = 1;
  a.cap = 2;
  PKD_LAUNCH((k_knn<D, G, S, false><<<1, QTHREADS, (size_t)(QTHREADS / G) * 2 * (12 + 4 * D), s>>>(a)));
}
template <int D>
static void noalloc_warm(cudaStream_t s) {
  constexpr int G = D <= 4 ? 4 : 8;
  noalloc_warm_as<D, G, 1>(s);
  noalloc_warm_as<D, G, D <= 4 ? 3 : 2>(s);
  noalloc_warm_as<D, G, 16 / G>(s);
  noalloc_warm_as<D, 32, 1>(s);
  noalloc_warm_as<D, 32, 2>(s);
  noalloc_warm_as<D, 32, 4>(s);
}

// Set-up, once per device, with that device current: the scratch address,
// and every kernel of the call loaded with its local memory reserved.
static int noalloc_scratch(int dev, cudaStream_t s, unsigned char** out) {
  std::lock_guard<std::mutex> g(g_noalloc_mu);
  if (!g_noalloc_ptr[dev]) {
    void* p = nullptr;
    const cudaError_t e = cudaGetSymbolAddress(&p, g_knn_noalloc_scratch);
    if (e != cudaSuccess || p == nullptr) {
      fprintf(stderr, "pkd_knn_ids_noalloc: scratch address on device %d: %s\n", dev,
              cudaGetErrorString(e));
      return e != cudaSuccess ? cuda_err(e) : PKD_ECUDA;
    }
    PKD_LAUNCH(k_noalloc_check<<<1, 256, 0, s>>>(nullptr, 0, nullptr));
    noalloc_warm<1>(s);
    noalloc_warm<2>(s);
    noalloc_warm<3>(s);
    noalloc_warm<4>(s);
    noalloc_warm<5>(s);
    noalloc_warm<6>(s);
    noalloc_warm<7>(s);
    noalloc_warm<8>(s);
    PKD_CUDA(cudaGetLastError());
    PKD_CUDA(cudaStreamSynchronize(s));
    g_noalloc_ptr[dev] = (unsigned char*)p;
  }
  *out = g_noalloc_ptr[dev];
  return PKD_OK;
}

}  // namespace pkd

extern "C" int pkd_knn_ids_noalloc(const pkd_tree* tc, const int32_t* queries, uint64_t q, int k,
                                   uint32_t* out_ids, void* stream) {
  if (!tc || k < 1 || k > 128) return PKD_EINVAL;
  if (q == 0) return PKD_OK;
  if (!queries || !out_ids) return PKD_EINVAL;
  if (q > (uint64_t)PKD_NOALLOC_MAX_PAIRS / (uint64_t)k) {
    fprintf(stderr,
            "pkd_knn_ids_noalloc: q*k = %llu exceeds the fixed scratch of %llu (query, neighbour) "
            "pairs; split the batch or use pkd_knn\n",
            (unsigned long long)q * (unsigned long long)k, (unsigned long long)PKD_NOALLOC_MAX_PAIRS);
    return PKD_EINVAL;
  }
  TreeMem& t = const_cast<TreeMem&>(tc->m);
  int dev = -1;
  PKD_CUDA(cudaGetDevice(&dev));
  if (dev != t.device || dev < 0 || dev >= NOALLOC_MAX_DEVICES) return PKD_EINVAL;
  unsigned char* scratch = nullptr;
  PKD_TRY_(noalloc_scratch(dev, (cudaStream_t)stream, &scratch));
  cudaStream_t s = (cudaStream_t)stream;
  TreeTouch touch{&t, s, true};  // may not create an event
  unsigned* bad = (unsigned*)scratch;
  PKD_CUDA(cudaMemsetAsync(bad, 0, sizeof(unsigned), s));
  PKD_LAUNCH(k_noalloc_check<<<152 * 8, 256, 0, s>>>(queries, q * (uint64_t)t.p.d, bad));
  unsigned h = 0;
  PKD_CUDA(cudaMemcpyAsync(&h, bad, sizeof(unsigned), cudaMemcpyDeviceToHost, s));
  PKD_CUDA(cudaStreamSynchronize(s));
  if (h != 0) return PKD_EINVAL;
  PKD_TRY_(check_status(t, s));
  if (!query_height_ok(t)) return PKD_EINTERNAL;
  QueryArgs a{};
  a.nodes = t.nodes;
  a.ndim = t.ndim;
  a.A = t.A;
  a.root = t.root;
  a.q = queries;
  a.nq = q;
  a.k = k;
  a.out_ids = out_ids;
  a.out_d2 = (int64_t*)(scratch + 256);
  a.st = t.st;
  a.cap = query_stack_cap(t);
  PKD_QDISPATCH(t.p.d, launch_knn_any, a, s);
  PKD_CUDA(cudaGetLastError());
  return PKD_OK;
}
