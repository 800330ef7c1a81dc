// Routing a batch update: every batch point goes down the tree to its leaf,
// lambda levels a round, and on the way the update is decided.
//
// An item is a tree node with the batch points below it (a contiguous range
// of the batch buffers).  One team answers an item in one pass: it fetches the
// "skeleton at T" (the node and the lambda levels below it that points reach,
// Alg. 2) into shared memory while its points step down, counts the points of
// every node, tests the alpha balance top-down (a reached node's new size is
// its size plus or minus its points: an id that a delete has taken is stored,
// so every routed point is found), and emits
//   stay     nodes that stay, with their new sizes (written to the tree once
//            nothing can fail any more)
//   items    subtrees to rebuild: unbalanced nodes, and the leaves an insert
//            reaches; their arena ranges are assigned here
//   groups   leaves a delete reaches: gout to compact in place, gin inside
//            subtrees that are rebuilt
//   next     items of the next round, by size
// The points below an item that ends here go to their final place in F,
// those of a next item to the other batch buffer, each once.
//
// Teams: a warp up to SMALL_ITEM points, a CTA up to MID_ITEM.  Larger items
// are sieved by the count / scan / scatter kernels of the build between
// k_big_fetch and k_big_emit.  The four passes over every item's skeleton in
// global memory that this replaces (fetch, emit, count, decide, with the
// sieve for every item above SMALL_ITEM) were bound by the latency of their
// dependent loads, and a batch of a thousand points took 17 launches and a
// host read per round.
//
// What bounds it: the chain of lambda dependent node loads of an item, hidden
// by 32 warps per SM (64 registers), and the instructions around them.  The
// last round of 1e7 random points in 1e8 (262144 items of 38 points): 0.64 ms;
// the round before (4096 items of 2441): 0.35 ms.  Four passes: 0.9-1.2 ms and
// 0.5 ms with the sieve.
#pragma once

#include "sieve_tma.cuh"

namespace pkd {

struct LeafGroup {
  uint32_t slot;   // the leaf's node slot
  uint32_t len;    // routed batch points
  uint64_t start;  // the first of them (position in F)
};

struct __align__(16) RebuildItem {  // (arena and batch positions are below 2^31)
  uint32_t slot;
  uint32_t depth;
  uint32_t size;      // points after the update
  uint32_t old_live;  // stored points that remain
  uint32_t pos;       // arena position assigned
  uint32_t ws;        // the first of its batch points (insert) in F
  uint32_t nw;        // their number
  uint32_t leaf;      // 1: the old subtree is a leaf of at most BIG_LEAF points
};

// Leaves of more than BIG_LEAF points are copied one block each.
constexpr uint32_t BIG_LEAF = 1024;

constexpr uint32_t SMALL_ITEM = 256;  // one warp, 8 points a lane
constexpr uint32_t MID_ITEM = 4096;   // one CTA of MID_TEAM threads, 16 points each
constexpr int MID_TEAM = 256, BIG_TEAM = 128, WARP_TEAMS = 4;
constexpr uint32_t ITEM_FLAG = 0x80000000u;  // in a Seg's depth: inside a rebuilt subtree
constexpr int CONT_FLAG = 0x100;             // in an external entry's x: its points go on

// Counters of an update (U_*) and of a round (R_*), 32-bit words on the device.
enum : int {
  U_INNER = 0, U_TOTAL = 2 /* u64: items << 32 | their points */, U_ITEMS = 3, U_INNER_PTS = 4 /* u64 */, U_MAX = 6, U_MAXNEW = 7,
  U_GOUT = 8, U_GIN = 9, U_FOUND = 10, U_WORDS = 16
};
enum : int { R_BIG = 0, R_MID = 1, R_SMALL = 2, R_TILES = 3, R_BIGPTS = 4, R_STAY = 5, R_AUX = 6, R_COPY = 7, R_WORDS = 8 };
// The blocks of counters lie 128 bytes apart: atomics on one line serialise.
constexpr uint32_t CTL_STRIDE = 32;

struct RouteArgs {
  Params p;
  int lam, NB, HN, TILE;
  int insert;
  int last;  // no further round: an item for one is an error
  const Node* nodes;
  const uint8_t* ndim;
  uint32_t* aux;  // [node slot] deleted points below, inside rebuilt subtrees (delete)
  DevStatus* st;
  Pts src, dst, F;
  uint64_t top;    // arena position of the first rebuild item
  uint32_t* u;     // U_* counters
  uint32_t* cur;   // this round's R_* counters (stay, aux, copy)
  uint32_t* next;  // the next round's
  Seg *big, *mid, *small;  // the next round's items
  uint32_t big_cap, mid_cap, small_cap;
  uint2* stay;  // (slot, new size)
  uint32_t stay_cap;
  uint32_t* auxs;  // slots whose aux word was set
  uint32_t aux_cap;
  uint2* copy;  // big items: (first, count) of ended ranges, at most TILE points each
  uint32_t copy_cap;
  RebuildItem* items;
  LeafGroup *gout, *gin;
  uint32_t item_cap, group_cap;
};

// An item's skeleton in shared memory, by heap index (level-lambda position
// for st).
struct Skel {
  int2* sk;         // split (internal) or split dimension (external), meta
  uint32_t* sl;     // node slot
  uint32_t* sz;     // node size
  uint32_t* st;     // batch points before the position
  uint32_t* under;  // bits: inside a subtree that is rebuilt
};
__host__ __device__ inline size_t skel_bytes(int HN, int NB) {
  return (size_t)HN * 16 + (size_t)NB * 4 + (size_t)(HN < 128 ? 4 : HN / 32) * 4;
}
__device__ __forceinline__ Skel skel_at(unsigned char* p, int HN, int NB) {
  Skel S;
  S.sk = (int2*)p;
  S.sl = (uint32_t*)(S.sk + HN);
  S.sz = S.sl + HN;
  S.st = S.sz + HN;
  S.under = S.st + NB;
  return S;
}

template <int T>
__device__ __forceinline__ void team_sync() {
  if constexpr (T == 32) __syncwarp();
  else __syncthreads();
}
template <int T>
__device__ __forceinline__ int team_rank() {
  return T == 32 ? lane_id() : (int)threadIdx.x;
}
__device__ __forceinline__ int heap_level(int v) { return 31 - __clz(v); }
// First level-lambda position below heap index v: its number as a bucket.
__device__ __forceinline__ int heap_pos(int v, int lam) {
  const int j = heap_level(v);
  return (v - (1 << j)) << (lam - j);
}

// Batch points below heap entry v of an item of `len` points: the starts of the
// positions below it are consecutive.
__device__ __forceinline__ uint32_t heap_count(const Skel& S, int v, int lam, uint32_t len) {
  const int lo = heap_pos(v, lam), hi = lo + (1 << (lam - heap_level(v)));
  return (hi == (1 << lam) ? len : S.st[hi]) - S.st[lo];
}

// Nodes of one skeleton level: every defined heap entry is loaded; one that
// points reach (or any, `all`) becomes internal and defines its children
// unless it is a leaf or on the last level.  Returns whether this thread saw
// an internal entry.
template <int T>
__device__ __forceinline__ bool skel_level(const RouteArgs& a, const Skel& S, int j, bool all) {
  bool any = false;
  for (int v = (1 << j) + team_rank<T>(); v < (2 << j); v += T) {
    const int2 e = S.sk[v];
    if (sk_state(e.y) == SK_NONE) continue;
    const uint32_t slot = S.sl[v];
    const int dm = a.ndim[slot];
    const Node nd = a.nodes[slot];
    S.sz[v] = nd.size;
    if (j == a.lam || dm == PKD_LEAF || !(all || e.x)) {
      S.sk[v] = make_int2(dm, sk_meta(SK_BUCKET, 0, heap_pos(v, a.lam)));
      continue;
    }
    any = true;
    S.sk[v] = make_int2(nd.split, sk_meta(SK_INTERNAL, dm, 0));
    S.sl[2 * v] = nd.a;
    S.sl[2 * v + 1] = nd.b;
    S.sk[2 * v] = S.sk[2 * v + 1] = make_int2(0, sk_meta(SK_BUCKET, 0, 0));  // x: points reach it
  }
  return any;
}

template <int T>
__device__ __forceinline__ void skel_clear(const RouteArgs& a, const Skel& S) {
  for (int v = team_rank<T>(); v < a.HN; v += T) S.sk[v] = make_int2(0, sk_meta(SK_NONE, 0, 0));
  for (int b = team_rank<T>(); b < a.NB; b += T) S.st[b] = 0;
  for (int w = team_rank<T>(); w < max(4, a.HN / 32); w += T) S.under[w] = 0;
}

// What the team decided about an internal entry (in sk[v].x, the split is not
// needed any more).
enum : int { ACT_NONE = 0, ACT_STAY = 1, ACT_AUX = 2, ACT_REBUILD = 3 };

// With the positions' starts in st: the balance test of every internal entry,
// and everything the item emits.  On return the x of an external entry has
// CONT_FLAG when its points go on to another round.
template <int T>
__device__ __forceinline__ void route_tail(const RouteArgs& a, const Skel& S, const Seg& it, uint2& seen,
                                           bool is_big) {
  const int tid = team_rank<T>();
  const bool ins = a.insert != 0;
  const uint32_t depth0 = it.depth & ~ITEM_FLAG;
  // all tests at once: a rebuilt node (rare) covers the ones below it afterwards
  bool fix = (it.depth & ITEM_FLAG) != 0;
  for (int v = 1 + tid; v < a.NB; v += T) {
    if (sk_state(S.sk[v].y) != SK_INTERNAL) continue;
    const uint32_t c = heap_count(S, v, a.lam, it.len);
    int act = ACT_NONE;
    if (c) {
      const uint32_t lc = heap_count(S, 2 * v, a.lam, it.len);
      const uint32_t N = ins ? S.sz[v] + c : S.sz[v] - c;
      const uint32_t L = ins ? S.sz[2 * v] + lc : S.sz[2 * v] - lc;
      act = N > 0 && is_balanced(L, N, a.p.alpha_num, a.p.alpha_den) ? ACT_STAY : ACT_REBUILD;
      fix |= act == ACT_REBUILD;
    }
    S.sk[v].x = act;
  }
  if constexpr (T == 32) {
    fix = __any_sync(FULL_MASK, fix);
    __syncwarp();
  } else {
    fix = __syncthreads_or(fix);
  }
  if (fix) {
    if (tid == 0 && (it.depth & ITEM_FLAG)) S.under[0] |= 2u;
    team_sync<T>();
    for (int j = 0; j < a.lam; ++j) {
      for (int v = (1 << j) + tid; v < (2 << j); v += T) {
        if (sk_state(S.sk[v].y) != SK_INTERNAL || S.sk[v].x == ACT_NONE) continue;
        const bool und = (S.under[v >> 5] >> (v & 31)) & 1u;
        if (und) S.sk[v].x = ins ? ACT_NONE : ACT_AUX;
        if (und || S.sk[v].x == ACT_REBUILD) atomicOr(&S.under[(2 * v) >> 5], 3u << ((2 * v) & 31));
      }
      team_sync<T>();
    }
  }
  // Emission, a warp at a time over its share of the heap, in two passes: the
  // totals, one atomic per counter for all of them (on different lanes, so that
  // they overlap), then the entries.  Appending through one counter serialises
  // at its address (about 1.3 ns each): with an update of every counter per 64
  // heap entries the last round of a 1e7-point insert took 1.35 ms, now 0.64.
  const int lane = lane_id();
  const int step = 32 * (T / 32), vw = T == 32 ? 0 : 32 * warp_id();
  const unsigned lt = lanemask_lt();
  // What heap entry v emits: a list (kind), its points, a size.
  //   0 rebuild items, 1 small, 2 mid, 3 big, 4 gout, 5 gin, 6 stay
  struct Out {
    int kind;
    bool inner, aux;
    uint32_t len, size;
  };
  auto what = [&](int v) {
    Out o{-1, false, false, 0, 0};
    if (v < 1 || v >= a.HN) return o;
    const int2 e = S.sk[v];
    const int st = sk_state(e.y);
    if (st == SK_NONE || (st == SK_INTERNAL && e.x == ACT_NONE)) return o;
    o.len = heap_count(S, v, a.lam, it.len);
    if (o.len == 0) return o;
    const uint32_t old = S.sz[v];
    if (st == SK_INTERNAL) {
      if (e.x == ACT_AUX) {
        o.aux = true;
      } else {
        o.kind = e.x == ACT_STAY ? 6 : 0;
        o.size = ins ? old + o.len : old - o.len;
        o.inner = true;
      }
      return o;
    }
    const bool und = (S.under[v >> 5] >> (v & 31)) & 1u;
    if (ins && und) return o;  // the rebuilt subtree takes the range as it is
    if (e.x == PKD_LEAF) {
      if (ins) {
        o.kind = 0;
        o.size = old + o.len;
        o.inner = old > BIG_LEAF;
      } else {
        o.kind = und ? 5 : 4;
        o.aux = und;
      }
    } else {
      o.kind = o.len > MID_ITEM ? 3 : (o.len > SMALL_ITEM ? 2 : 1);
    }
    return o;
  };
  uint32_t nsz = 0, imax = 0, nmax = 0, tiles = 0, bpts = 0, ninner = 0;
  unsigned long long ipts = 0, cnt = 0;  // cnt: a byte per list, 7: aux words
  for (int v0 = vw; v0 < a.HN; v0 += step) {
    const Out o = what(v0 + lane);
    if (o.kind >= 0) cnt += 1ull << (8 * o.kind);
    if (o.aux) cnt += 1ull << 56;
    if (o.kind == 0) {
      nsz += o.size;
      imax = max(imax, o.size);
      if (ins) nmax = max(nmax, o.len);
      ninner += o.inner;
      if (sk_state(S.sk[v0 + lane].y) == SK_INTERNAL) ipts += S.sz[v0 + lane];
    } else if (o.kind == 3) {
      tiles += (o.len + a.TILE - 1) / a.TILE;
      bpts += o.len;
    }
  }
  unsigned present = 0;
#pragma unroll
  for (int k = 0; k < 8; ++k)
    if ((cnt >> (8 * k)) & 0xFFu) present |= 1u << k;
  present = __reduce_or_sync(FULL_MASK, present);
  uint32_t amount = 0;  // lane k: entries of list k
#pragma unroll
  for (int k = 0; k < 8; ++k) {
    if (!((present >> k) & 1u)) continue;  // warp-uniform
    const uint32_t t = __reduce_add_sync(FULL_MASK, (uint32_t)(cnt >> (8 * k)) & 0xFFu);
    if (lane == k) amount = t;
  }
  uint32_t first = 0, pos32 = 0;
  if (present & 1u) {
    nsz = __reduce_add_sync(FULL_MASK, nsz);
    imax = __reduce_max_sync(FULL_MASK, imax);
    nmax = __reduce_max_sync(FULL_MASK, nmax);
    ninner = __reduce_add_sync(FULL_MASK, ninner);
    if (ninner) {
      for (int o = 16; o; o >>= 1) ipts += __shfl_xor_sync(FULL_MASK, ipts, o);
      if (lane == 9) atomicAdd((unsigned long long*)(a.u + U_INNER_PTS), ipts);
      if (lane == 10) atomicAdd(a.u + U_INNER, ninner);
    }
    // the maxima seldom grow: only what this warp has not sent yet
    if (imax > seen.x) {
      seen.x = imax;
      if (lane == 11) atomicMax(a.u + U_MAX, imax);
    }
    if (nmax > seen.y) {
      seen.y = nmax;
      if (lane == 12) atomicMax(a.u + U_MAXNEW, nmax);
    }
  }
  if (present & 8u) {
    tiles = __reduce_add_sync(FULL_MASK, tiles);
    bpts = __reduce_add_sync(FULL_MASK, bpts);
    if (lane == 13) atomicAdd(a.next + R_TILES, tiles);
    if (lane == 14) atomicAdd(a.next + R_BIGPTS, bpts);
  }
  if (amount) {  // the lists hold every entry by construction
    uint32_t* c = nullptr;
    uint32_t cap = 0;
    switch (lane) {
      case 0: cap = a.item_cap; break;
      case 1: c = a.next + R_SMALL, cap = a.small_cap; break;
      case 2: c = a.next + R_MID, cap = a.mid_cap; break;
      case 3: c = a.next + R_BIG, cap = a.big_cap; break;
      case 4: c = a.u + U_GOUT, cap = a.group_cap; break;
      case 5: c = a.u + U_GIN, cap = a.group_cap; break;
      case 6: c = a.cur + R_STAY, cap = a.stay_cap; break;
      default: c = a.cur + R_AUX, cap = a.aux_cap; break;
    }
    if (lane == 0) {  // items (high word) and their arena positions (fewer than 2^31) in one
      const unsigned long long r =
          atomicAdd((unsigned long long*)(a.u + U_TOTAL), ((unsigned long long)amount << 32) | nsz);
      first = (uint32_t)(r >> 32);
      pos32 = (uint32_t)r;
    } else {
      first = atomicAdd(c, amount);
    }
    if (first + amount > cap || first + amount < first) {
      set_error(a.st, DERR_CAPACITY, 800 + lane);
      first = 0xFFFFFFFFu;
    }
    if (a.last && lane >= 1 && lane <= 3) {
      set_error(a.st, DERR_STATE, 820 + lane);
      first = 0xFFFFFFFFu;
    }
  }
  uint32_t at[8];
#pragma unroll
  for (int k = 0; k < 8; ++k) at[k] = __shfl_sync(FULL_MASK, first, k);
  uint64_t pos = a.top + __shfl_sync(FULL_MASK, pos32, 0);
  if (present || is_big)
    for (int v0 = vw; v0 < a.HN; v0 += step) {
      const int v = v0 + lane;
      const Out o = what(v);
      if (!__any_sync(FULL_MASK, o.len != 0)) continue;
      const uint64_t b0 = o.len ? it.start + S.st[heap_pos(v, a.lam)] : 0;
      const uint32_t slot = o.len ? S.sl[v] : 0, dep = depth0 + (uint32_t)heap_level(max(v, 1));
#pragma unroll
      for (int k = 0; k < 7; ++k) {
        if (!((present >> k) & 1u) || at[k] == 0xFFFFFFFFu) continue;  // warp-uniform
        const unsigned bits = __ballot_sync(FULL_MASK, o.kind == k);
        const uint32_t i = at[k] + __popc(bits & lt);
        at[k] += __popc(bits);
        if (k == 0) {
          if (!bits) continue;
          const uint32_t mine = o.kind == 0 ? o.size : 0u;
          const uint32_t incl = (uint32_t)warp_incl_scan((int)mine);
          if (o.kind == 0)
            a.items[i] = RebuildItem{slot, dep, o.size, ins ? S.sz[v] : o.size, (uint32_t)(pos + incl - mine),
                                     (uint32_t)b0, ins ? o.len : 0u, o.inner ? 0u : 1u};
          pos += __shfl_sync(FULL_MASK, incl, 31);
        } else if (o.kind == k) {
          if (k <= 3) {
            const bool und = (S.under[v >> 5] >> (v & 31)) & 1u;
            (k == 1 ? a.small : k == 2 ? a.mid : a.big)[i] = Seg{b0, o.len, dep | (und ? ITEM_FLAG : 0u), slot, IN_B};
            S.sk[v].x |= CONT_FLAG;
          } else if (k <= 5) {
            (k == 4 ? a.gout : a.gin)[i] = LeafGroup{slot, o.len, b0};
          } else {
            a.stay[i] = make_uint2(slot, o.size);
          }
        }
      }
      if ((present >> 7 & 1u) && at[7] != 0xFFFFFFFFu) {
        const unsigned bits = __ballot_sync(FULL_MASK, o.aux);
        if (o.aux) {
          a.auxs[at[7] + __popc(bits & lt)] = slot;
          a.aux[slot] = o.len;
        }
        at[7] += __popc(bits);
      }
      // the sieve moved every point of a big item to the other buffer: the
      // ranges that end here are copied to F afterwards, TILE points at a time
      if (is_big && o.len && sk_state(S.sk[v].y) == SK_BUCKET && !(S.sk[v].x & CONT_FLAG)) {
        const uint32_t nc = (o.len + a.TILE - 1) / a.TILE;
        const uint32_t i = atomicAdd(a.cur + R_COPY, nc);
        if (i + nc > a.copy_cap) set_error(a.st, DERR_CAPACITY, 810);
        else
          for (uint32_t k = 0; k < nc; ++k)
            a.copy[i + k] = make_uint2((uint32_t)b0 + k * a.TILE, min((uint32_t)a.TILE, o.len - k * a.TILE));
      }
    }
  team_sync<T>();
}

template <int D, int T>
__global__ void __launch_bounds__(T == 32 ? 32 * WARP_TEAMS : T, T == 32 ? 8 : 4) k_route(RouteArgs a, const Seg* list,
                                                                         const uint32_t* n) {
  constexpr int PER = (int)(T == 32 ? SMALL_ITEM : MID_ITEM) / T;
  constexpr int TEAMS = T == 32 ? WARP_TEAMS : 1;
  extern __shared__ __align__(16) unsigned char route_sm[];
  if (pkd_failed_block(a.st)) return;
  const int tid = team_rank<T>(), team = T == 32 ? warp_id() : 0;
  const Skel S = skel_at(route_sm + (size_t)team * skel_bytes(a.HN, a.NB), a.HN, a.NB);
  const uint32_t nn = *n;
  uint2 seen = make_uint2(0, 0);  // (reading the counters would queue behind the atomics on their line)
  for (uint32_t i = blockIdx.x * TEAMS + team; i < nn; i += gridDim.x * TEAMS) {
    const Seg it = list[i];
    const int len = (int)it.len;
    skel_clear<T>(a, S);
    // Heap index of every point, then also its rank within the external entry
    // << 12.  The coordinates are read again where they are needed (from L1 or
    // L2): held in registers they made the warps' kernel spill at 3-D, with the
    // same time.
    uint32_t hr[PER];
#pragma unroll
    for (int q = 0; q < PER; ++q) hr[q] = q * T + tid < len ? 1 : 0;
    team_sync<T>();
    if (tid == 0) {
      S.sl[1] = it.root;
      S.sk[1] = make_int2(1, sk_meta(SK_BUCKET, 0, 0));
    }
    team_sync<T>();
    for (int j = 0; j <= a.lam; ++j) {
      const bool mine = skel_level<T>(a, S, j, false);
      bool any;
      if constexpr (T == 32) {
        any = __any_sync(FULL_MASK, mine);
        __syncwarp();
      } else {
        any = __syncthreads_or(mine);
      }
      if (!any) break;  // every point is at its external entry
#pragma unroll
      for (int q = 0; q < PER; ++q) {
        if (q * T >= len) break;
        const int h = (int)hr[q];
        if (!h) continue;
        const int2 e = S.sk[h];
        if (sk_state(e.y) != SK_INTERNAL) continue;
        const int32_t xv = a.src.c[(uint64_t)sk_dim(e.y) * a.src.stride + it.start + q * T + tid];
        const int c = 2 * h + (xv >= e.x);
        hr[q] = (uint32_t)c;
        S.sk[c].x = 1;
      }
      team_sync<T>();
    }
#pragma unroll
    for (int q = 0; q < PER; ++q) {
      if (q * T >= len) break;
      if (hr[q]) hr[q] |= atomicAdd(&S.st[heap_pos((int)hr[q], a.lam)], 1u) << 12;
    }
    team_sync<T>();
    if (tid < 32) {  // starts: exclusive scan of the positions' counts
      unsigned carry = 0;
      for (int b0 = 0; b0 < a.NB; b0 += 32) {
        const int b = b0 + tid;
        const unsigned c = b < a.NB ? S.st[b] : 0;
        const unsigned incl = (unsigned)warp_incl_scan((int)c);
        __syncwarp();
        if (b < a.NB) S.st[b] = carry + incl - c;
        carry += __shfl_sync(FULL_MASK, incl, 31);
      }
    }
    team_sync<T>();
    route_tail<T>(a, S, it, seen, false);
#pragma unroll
    for (int q = 0; q < PER; ++q) {
      if (q * T >= len) break;
      if (!hr[q]) continue;
      const int v = (int)(hr[q] & 0xFFFu);
      const uint64_t g = it.start + q * T + tid;
      const uint64_t o = it.start + S.st[heap_pos(v, a.lam)] + (hr[q] >> 12);
      const Pts& P = (S.sk[v].x & CONT_FLAG) ? a.dst : a.F;
#pragma unroll
      for (int j = 0; j < D; ++j) P.c[(uint64_t)j * P.stride + o] = a.src.c[(uint64_t)j * a.src.stride + g];
      P.id[o] = a.src.id[g];
    }
    team_sync<T>();
  }
}

// Big items: the whole skeleton, for the sieve (skel, with an external
// entry's bucket = its position) and for k_big_emit.
static __global__ void __launch_bounds__(BIG_TEAM) k_big_fetch(RouteArgs a, const Seg* list, int2* skel, uint32_t* slots,
                                                        uint32_t* sizes) {
  extern __shared__ __align__(16) unsigned char route_sm[];
  const Skel S = skel_at(route_sm, a.HN, a.NB);
  skel_clear<BIG_TEAM>(a, S);
  __syncthreads();
  if (threadIdx.x == 0) {
    S.sl[1] = list[blockIdx.x].root;
    S.sk[1] = make_int2(0, sk_meta(SK_BUCKET, 0, 0));
  }
  __syncthreads();
  for (int j = 0; j <= a.lam; ++j)
    if (!__syncthreads_or(skel_level<BIG_TEAM>(a, S, j, true))) break;
  __syncthreads();
  const uint64_t o = (uint64_t)blockIdx.x * a.HN;
  for (int v = threadIdx.x; v < a.HN; v += BIG_TEAM) {
    skel[o + v] = S.sk[v];
    slots[o + v] = S.sl[v];
    sizes[o + v] = S.sz[v];
  }
}

// ... and, with the bucket-major scan of the tile histograms, their counts,
// decisions and emission.
static __global__ void __launch_bounds__(BIG_TEAM) k_big_emit(RouteArgs a, RoundArgs r, const uint32_t* slots,
                                                       const uint32_t* sizes) {
  extern __shared__ __align__(16) unsigned char route_sm[];
  if (pkd_failed_block(a.st)) return;
  const Skel S = skel_at(route_sm, a.HN, a.NB);
  const Seg it = r.big[blockIdx.x];
  skel_clear<BIG_TEAM>(a, S);
  __syncthreads();
  const uint64_t o = (uint64_t)blockIdx.x * a.HN;
  for (int v = threadIdx.x; v < a.HN; v += BIG_TEAM) {
    S.sk[v] = r.skel[o + v];
    S.sl[v] = slots[o + v];
    S.sz[v] = sizes[o + v];
  }
  const uint64_t nt = (it.len + r.TILE - 1) / r.TILE, hb = (uint64_t)r.tile0[blockIdx.x] * r.NB;
  const uint32_t base = r.hscan[hb];
  for (int b = threadIdx.x; b < a.NB; b += BIG_TEAM) S.st[b] = r.hscan[hb + (uint64_t)b * nt] - base;
  __syncthreads();
  uint2 seen = make_uint2(0, 0);
  route_tail<BIG_TEAM>(a, S, it, seen, true);
}

// The ranges of the big items that ended, from the sieve's destination to F.
static __global__ void k_copy_ended(RouteArgs a, const uint32_t* n) {
  if (pkd_failed_block(a.st)) return;
  const uint32_t nn = min(*n, a.copy_cap);
  const int d = a.p.d;
  for (uint32_t i = blockIdx.x; i < nn; i += gridDim.x) {
    const uint2 c = a.copy[i];
    for (uint32_t k = threadIdx.x; k < c.y; k += blockDim.x) {
      const uint64_t p = (uint64_t)c.x + k;
      for (int j = 0; j < d; ++j) a.F.c[(uint64_t)j * a.F.stride + p] = a.dst.c[(uint64_t)j * a.dst.stride + p];
      a.F.id[p] = a.dst.id[p];
    }
  }
}

}  // namespace pkd
