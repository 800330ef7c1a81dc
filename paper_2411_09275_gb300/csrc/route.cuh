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
#pragma once

#include "sieve_tma.cuh"

namespace pkd {

struct LeafGroup {
  uint32_t slot;   // the leaf's node slot
  uint32_t len;    // routed batch points
  uint64_t start;  // the first of them (position in F)
};

struct RebuildItem {
  uint32_t slot;
  uint32_t depth;
  uint32_t size;      // points after the update
  uint32_t old_live;  // stored points that remain
  uint64_t ws, we;    // batch points (insert) in F
  uint64_t pos;       // arena position assigned
  uint32_t leaf;      // 1: the old subtree is a leaf of at most BIG_LEAF points
  uint32_t pad;
};

// Leaves of more than BIG_LEAF points are copied one block each.
constexpr uint32_t BIG_LEAF = 1024;

constexpr uint32_t SMALL_ITEM = 256;  // one warp, 8 points a lane
constexpr uint32_t MID_ITEM = 4096;   // one CTA of MID_TEAM threads, 16 points each
constexpr int MID_TEAM = 256, BIG_TEAM = 128, WARP_TEAMS = 4;
constexpr uint32_t ITEM_FLAG = 0x80000000u;  // in a Seg's depth: inside a rebuilt subtree
constexpr uint32_t CONT_FLAG = 0x80000000u;  // in a count: the node's points go on

// Counters of an update (U_*) and of a round (R_*), 32-bit words on the device.
enum : int {
  U_ITEMS = 0, U_INNER = 1, U_TOTAL = 2 /* u64 */, U_INNER_PTS = 4 /* u64 */, U_MAX = 6, U_MAXNEW = 7,
  U_GOUT = 8, U_GIN = 9, U_FOUND = 10, U_WORDS = 16
};
enum : int { R_BIG = 0, R_MID = 1, R_SMALL = 2, R_TILES = 3, R_BIGPTS = 4, R_STAY = 5, R_AUX = 6, R_COPY = 7, R_WORDS = 8 };

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
  uint32_t* f;      // batch points below
  uint32_t* st;     // batch points before the position
  uint32_t* under;  // bits: inside a subtree that is rebuilt
};
__host__ __device__ inline size_t skel_bytes(int HN, int NB) {
  return (size_t)HN * 20 + (size_t)NB * 4 + (size_t)(HN < 128 ? 4 : HN / 32) * 4;
}
__device__ __forceinline__ Skel skel_at(unsigned char* p, int HN, int NB) {
  Skel S;
  S.sk = (int2*)p;
  S.sl = (uint32_t*)(S.sk + HN);
  S.sz = S.sl + HN;
  S.f = S.sz + HN;
  S.st = S.f + HN;
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
  for (int v = team_rank<T>(); v < a.HN; v += T) {
    S.sk[v] = make_int2(0, sk_meta(SK_NONE, 0, 0));
    S.f[v] = 0;
  }
  for (int b = team_rank<T>(); b < a.NB; b += T) S.st[b] = 0;
  for (int w = team_rank<T>(); w < max(4, a.HN / 32); w += T) S.under[w] = 0;
}

// What the team decided about an internal entry (in sk[v].x, the split is not
// needed any more).
enum : int { ACT_NONE = 0, ACT_STAY = 1, ACT_AUX = 2, ACT_REBUILD = 3 };

// With the points of every external entry in f and the positions' starts in
// st: counts bottom-up, the balance test top-down, and everything the item
// emits.  On return f[v] of an external entry has CONT_FLAG when its points
// go on to another round.
template <int T>
__device__ __forceinline__ void route_tail(const RouteArgs& a, const Skel& S, const Seg& it, bool is_big) {
  const int tid = team_rank<T>();
  const bool ins = a.insert != 0;
  const uint32_t depth0 = it.depth & ~ITEM_FLAG;
  for (int j = a.lam - 1; j >= 0; --j) {
    for (int v = (1 << j) + tid; v < (2 << j); v += T)
      if (sk_state(S.sk[v].y) == SK_INTERNAL) S.f[v] = S.f[2 * v] + S.f[2 * v + 1];
    team_sync<T>();
  }
  if (tid == 0 && (it.depth & ITEM_FLAG)) S.under[0] |= 2u;
  team_sync<T>();
  for (int j = 0; j < a.lam; ++j) {
    for (int v = (1 << j) + tid; v < (2 << j); v += T) {
      if (sk_state(S.sk[v].y) != SK_INTERNAL) continue;
      const uint32_t c = S.f[v];
      int act = ACT_NONE;
      if (c) {
        const int c0 = 2 * v;  // the children share a word of `under`
        if ((S.under[v >> 5] >> (v & 31)) & 1u) {
          act = ins ? ACT_NONE : ACT_AUX;
          atomicOr(&S.under[c0 >> 5], 3u << (c0 & 31));
        } else {
          const uint32_t N = ins ? S.sz[v] + c : S.sz[v] - c;
          const uint32_t L = ins ? S.sz[c0] + S.f[c0] : S.sz[c0] - S.f[c0];
          if (N > 0 && is_balanced(L, N, a.p.alpha_num, a.p.alpha_den)) {
            act = ACT_STAY;
          } else {
            act = ACT_REBUILD;
            atomicOr(&S.under[c0 >> 5], 3u << (c0 & 31));
          }
        }
      }
      S.sk[v].x = act;
    }
    team_sync<T>();
  }
  // Emission, a warp at a time over 32 * PER heap entries: one atomic per
  // counter for all of them, on different lanes so that they overlap.
  constexpr int PER = 4;
  const int lane = lane_id();
  const int w = T == 32 ? 0 : warp_id();
  const unsigned lt = lanemask_lt();
  for (int v0 = 32 * PER * w; v0 < a.HN; v0 += 32 * PER * (T / 32)) {
    uint32_t len[PER], size[PER];
    // lists: 0 rebuild items, 1 small, 2 mid, 3 big, 4 gout, 5 gin, 6 stay, 7 aux
    int kind[PER];
    bool inner[PER], aux[PER];
    uint32_t nsz = 0, imax = 0, nmax = 0, tiles = 0, bpts = 0, ninner = 0;
    unsigned long long ipts = 0;
#pragma unroll
    for (int u = 0; u < PER; ++u) {
      const int v = v0 + 32 * u + lane;
      kind[u] = -1;
      len[u] = size[u] = 0;
      inner[u] = aux[u] = false;
      if (v < 1 || v >= a.HN) continue;
      const int2 e = S.sk[v];
      const int st = sk_state(e.y);
      if (st == SK_NONE) continue;
      len[u] = S.f[v];
      if (len[u] == 0) continue;
      const uint32_t old = S.sz[v];
      if (st == SK_INTERNAL) {
        if (e.x == ACT_REBUILD) {
          kind[u] = 0;
          size[u] = ins ? old + len[u] : old - len[u];
          inner[u] = true;
          ipts += old;
        } else if (e.x == ACT_STAY) {
          kind[u] = 6;
          size[u] = ins ? old + len[u] : old - len[u];
        } else if (e.x == ACT_AUX) {
          aux[u] = true;
        }
        continue;
      }
      const bool und = (S.under[v >> 5] >> (v & 31)) & 1u;
      if (ins && und) continue;  // the rebuilt subtree takes the range as it is
      if (e.x == PKD_LEAF) {
        if (ins) {
          kind[u] = 0;
          size[u] = old + len[u];
          inner[u] = old > BIG_LEAF;
        } else {
          kind[u] = und ? 5 : 4;
          aux[u] = und;
        }
        continue;
      }
      kind[u] = len[u] > MID_ITEM ? 3 : (len[u] > SMALL_ITEM ? 2 : 1);
      S.f[v] = len[u] | CONT_FLAG;
      if (kind[u] == 3) {
        tiles += (len[u] + a.TILE - 1) / a.TILE;
        bpts += len[u];
      }
    }
    uint32_t tot[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) tot[k] = 0;
    bool anything = false;
#pragma unroll
    for (int u = 0; u < PER; ++u) {
      if (kind[u] == 0) {
        nsz += size[u];
        imax = max(imax, size[u]);
        nmax = max(nmax, ins ? len[u] : 0u);
        ninner += inner[u];
      }
      anything |= kind[u] >= 0 || aux[u] || (is_big && len[u]);
    }
    if (!__any_sync(FULL_MASK, anything)) continue;
#pragma unroll
    for (int u = 0; u < PER; ++u) {
#pragma unroll
      for (int k = 0; k < 7; ++k) tot[k] += __popc(__ballot_sync(FULL_MASK, kind[u] == k));
      tot[7] += __popc(__ballot_sync(FULL_MASK, aux[u]));
    }
    uint32_t incl = 0, first = 0;
    unsigned long long pos0 = 0;
    if (tot[0]) {
      incl = (uint32_t)warp_incl_scan((int)nsz);
      imax = __reduce_max_sync(FULL_MASK, imax);
      nmax = __reduce_max_sync(FULL_MASK, nmax);
      ninner = __reduce_add_sync(FULL_MASK, ninner);
      for (int o = 16; o; o >>= 1) ipts += __shfl_xor_sync(FULL_MASK, ipts, o);
      const uint32_t all = __shfl_sync(FULL_MASK, incl, 31);
      if (lane == 8) pos0 = atomicAdd((unsigned long long*)(a.u + U_TOTAL), (unsigned long long)all);
      if (lane == 9 && ipts) atomicAdd((unsigned long long*)(a.u + U_INNER_PTS), ipts);
      if (lane == 10) atomicMax(a.u + U_MAX, imax);
      if (lane == 11 && nmax) atomicMax(a.u + U_MAXNEW, nmax);
      if (lane == 12 && ninner) atomicAdd(a.u + U_INNER, ninner);
    }
    if (tot[3]) {
      tiles = __reduce_add_sync(FULL_MASK, tiles);
      bpts = __reduce_add_sync(FULL_MASK, bpts);
      if (lane == 13) atomicAdd(a.next + R_TILES, tiles);
      if (lane == 14) atomicAdd(a.next + R_BIGPTS, bpts);
    }
    {
      uint32_t n = 0;
      uint32_t* c = nullptr;
#pragma unroll
      for (int k = 0; k < 8; ++k)
        if (lane == k) n = tot[k];
      switch (lane) {
        case 0: c = a.u + U_ITEMS; break;
        case 1: c = a.next + R_SMALL; break;
        case 2: c = a.next + R_MID; break;
        case 3: c = a.next + R_BIG; break;
        case 4: c = a.u + U_GOUT; break;
        case 5: c = a.u + U_GIN; break;
        case 6: c = a.cur + R_STAY; break;
        case 7: c = a.cur + R_AUX; break;
        default: break;
      }
      if (n) first = atomicAdd(c, n);
      if (n) {  // the lists hold every entry by construction
        const uint32_t cap = lane == 0 ? a.item_cap : lane == 1 ? a.small_cap : lane == 2 ? a.mid_cap
                             : lane == 3 ? a.big_cap : lane <= 5 ? a.group_cap : lane == 6 ? a.stay_cap : a.aux_cap;
        if (first + n > cap || first + n < first) {
          set_error(a.st, DERR_CAPACITY, 800 + lane);
          first = 0xFFFFFFFFu;
        }
        if (a.last && lane >= 1 && lane <= 3) {
          set_error(a.st, DERR_STATE, 820 + lane);
          first = 0xFFFFFFFFu;
        }
      }
    }
    uint32_t at[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) at[k] = __shfl_sync(FULL_MASK, first, k);
    uint64_t pos = a.top + __shfl_sync(FULL_MASK, pos0, 8) + incl - nsz;
#pragma unroll
    for (int u = 0; u < PER; ++u) {
      const int v = v0 + 32 * u + lane;
#pragma unroll
      for (int k = 0; k < 7; ++k) {
        if (tot[k] == 0 || at[k] == 0xFFFFFFFFu) continue;  // warp-uniform
        const unsigned bits = __ballot_sync(FULL_MASK, kind[u] == k);
        if (kind[u] == k) {
          const uint32_t o = at[k] + __popc(bits & lt);
          const uint64_t b0 = it.start + S.st[heap_pos(v, a.lam)];
          const uint32_t dep = depth0 + (uint32_t)heap_level(v), slot = S.sl[v];
          if (k == 0) {
            a.items[o] = RebuildItem{slot, dep, size[u], ins ? S.sz[v] : size[u], b0, b0 + (ins ? len[u] : 0u), pos,
                                     inner[u] ? 0u : 1u, 0u};
            pos += size[u];
          } else if (k <= 3) {
            const bool und = (S.under[v >> 5] >> (v & 31)) & 1u;
            (k == 1 ? a.small : k == 2 ? a.mid : a.big)[o] = Seg{b0, len[u], dep | (und ? ITEM_FLAG : 0u), slot, IN_B};
          } else if (k <= 5) {
            (k == 4 ? a.gout : a.gin)[o] = LeafGroup{slot, len[u], b0};
          } else {
            a.stay[o] = make_uint2(slot, size[u]);
          }
        }
        at[k] += __popc(bits);
      }
      if (tot[7] && at[7] != 0xFFFFFFFFu) {
        const unsigned bits = __ballot_sync(FULL_MASK, aux[u]);
        if (aux[u]) {
          a.auxs[at[7] + __popc(bits & lt)] = S.sl[v];
          a.aux[S.sl[v]] = len[u];
        }
        at[7] += __popc(bits);
      }
      // the sieve moved every point of a big item to the other buffer: the
      // ranges that end here are copied to F afterwards, TILE points at a time
      if (is_big && v >= 1 && v < a.HN && len[u] && sk_state(S.sk[v].y) == SK_BUCKET && !(S.f[v] & CONT_FLAG)) {
        const uint32_t nc = (len[u] + a.TILE - 1) / a.TILE;
        const uint32_t o = atomicAdd(a.cur + R_COPY, nc);
        const uint32_t b0 = (uint32_t)it.start + S.st[heap_pos(v, a.lam)];
        if (o + nc > a.copy_cap) set_error(a.st, DERR_CAPACITY, 810);
        else
          for (uint32_t k = 0; k < nc; ++k)
            a.copy[o + k] = make_uint2(b0 + k * a.TILE, min((uint32_t)a.TILE, len[u] - k * a.TILE));
      }
    }
  }
  team_sync<T>();
}

template <int D, int T>
__global__ void __launch_bounds__(T == 32 ? 32 * WARP_TEAMS : T, T == 32 ? 5 : 2) k_route(RouteArgs a, const Seg* list,
                                                                         const uint32_t* n) {
  constexpr int PER = (int)(T == 32 ? SMALL_ITEM : MID_ITEM) / T;
  constexpr int TEAMS = T == 32 ? WARP_TEAMS : 1;
  constexpr bool REGS = T == 32 && D <= 3;  // the points' coordinates stay in registers
  extern __shared__ __align__(16) unsigned char route_sm[];
  if (pkd_failed_block(a.st)) return;
  const int tid = team_rank<T>(), team = T == 32 ? warp_id() : 0;
  const Skel S = skel_at(route_sm + (size_t)team * skel_bytes(a.HN, a.NB), a.HN, a.NB);
  const uint32_t nn = *n;
  for (uint32_t i = blockIdx.x * TEAMS + team; i < nn; i += gridDim.x * TEAMS) {
    const Seg it = list[i];
    const int len = (int)it.len;
    skel_clear<T>(a, S);
    int32_t x[PER][REGS ? D : 1];
    uint32_t hr[PER];  // heap index, then also the rank within the external entry << 12
#pragma unroll
    for (int q = 0; q < PER; ++q) {
      hr[q] = 0;
      if (q * T + tid < len) {
        hr[q] = 1;
        if constexpr (REGS) {
#pragma unroll
          for (int j = 0; j < D; ++j) x[q][j] = a.src.c[(uint64_t)j * a.src.stride + it.start + q * T + tid];
        }
      }
    }
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
        const int dm = sk_dim(e.y);
        int32_t xv;
        if constexpr (REGS) {
          xv = x[q][0];
#pragma unroll
          for (int k = 1; k < D; ++k)
            if (dm == k) xv = x[q][k];
        } else {
          xv = a.src.c[(uint64_t)dm * a.src.stride + it.start + q * T + tid];
        }
        const int c = 2 * h + (xv >= e.x);
        hr[q] = (uint32_t)c;
        S.sk[c].x = 1;
      }
      team_sync<T>();
    }
#pragma unroll
    for (int q = 0; q < PER; ++q) {
      if (q * T >= len) break;
      if (hr[q]) hr[q] |= atomicAdd(&S.f[hr[q]], 1u) << 12;
    }
    team_sync<T>();
    for (int v = 1 + tid; v < a.HN; v += T)
      if (sk_state(S.sk[v].y) == SK_BUCKET && S.f[v]) S.st[heap_pos(v, a.lam)] = S.f[v];
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
    route_tail<T>(a, S, it, false);
#pragma unroll
    for (int q = 0; q < PER; ++q) {
      if (q * T >= len) break;
      if (!hr[q]) continue;
      const int v = (int)(hr[q] & 0xFFFu);
      const uint64_t g = it.start + q * T + tid;
      const uint64_t o = it.start + S.st[heap_pos(v, a.lam)] + (hr[q] >> 12);
      const Pts& P = (S.f[v] & CONT_FLAG) ? a.dst : a.F;
#pragma unroll
      for (int j = 0; j < D; ++j) {
        int32_t xv;
        if constexpr (REGS) xv = x[q][j];
        else xv = a.src.c[(uint64_t)j * a.src.stride + g];
        P.c[(uint64_t)j * P.stride + o] = xv;
      }
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
  for (int v = 1 + threadIdx.x; v < a.HN; v += BIG_TEAM)
    if (sk_state(S.sk[v].y) == SK_BUCKET) {
      const int b = heap_pos(v, a.lam);
      S.f[v] = (b + 1 < a.NB ? S.st[b + 1] : it.len) - S.st[b];
    }
  __syncthreads();
  route_tail<BIG_TEAM>(a, S, it, true);
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
