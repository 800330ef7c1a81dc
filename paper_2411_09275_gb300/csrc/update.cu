// Batch updates of a Pkd-tree: BatchInsert (Alg. 2, Sec. 4.1) and the
// two-round BatchDelete (Sec. 4.2).
//
//  route    the batch goes down the tree lambda levels a round (route.cuh); on
//           the way a node that receives updates stays (its new size is
//           recorded) when it is still alpha-balanced, otherwise it is rebuilt
//           with Build on all its (live) points plus the new ones.  A reached
//           leaf is rebuilt (insert: Build(leaf + new)) or compacted (delete).
//  delete   every stored point of a reached leaf is compared with the batch
//           points routed there; the matches go (round 1 of Sec. 4.2).
//  rebuild  old subtrees are flattened by a parallel breadth-first walk into
//           fresh arena ranges, new points appended, and every rebuild item
//           becomes a root segment of one multi-segment build (build.cu).
#include <algorithm>
#include <cstdio>
#include <vector>

#include "query.cuh"
#include "route.cuh"
#include "tree_impl.hpp"

namespace pkd {

// The per-leaf kernels below give each warp UPW leaves (or rebuild items):
// lanes 0..UPW-1 fetch the descriptors together, and for leaves of at most
// 32 points every load of the UPW leaves is issued before the first store,
// so a warp keeps UPW dependent chains in flight instead of one.
constexpr int UPW = 4;
constexpr int UPW_WARPS = 8;  // warps per CTA
static_assert(32 % UPW == 0, "lanes split evenly between a warp's leaves");
__host__ __device__ inline unsigned upw_blocks(uint32_t n) {
  return (unsigned)(((uint64_t)n + UPW * UPW_WARPS - 1) / (UPW * UPW_WARPS));
}

// Deletion round 1 at the leaves: stored points equal to a routed batch point
// (coordinates and id) go.  MARK: the leaves of rebuilt subtrees, whose points
// the flatten copies: they are only marked (dead).  Otherwise the survivors
// move to the front of the leaf and its size is rewritten at once, in the pass
// that has its points in registers (marking every leaf and compacting in a
// second pass read each leaf twice: 0.55 + 0.89 ms for the 1e7 random deletes
// in 1e8 points).  *total counts the points that go.  Bound by HBM and by the
// latency of a warp's loads: eight CTAs per SM up to three dimensions, which
// spill a few registers, against six and four: 3.11, 3.16 and 3.33 ms for the
// whole delete.
template <int D, bool MARK>
__global__ void __launch_bounds__(UPW_WARPS * 32, (D <= 3 ? 8 : 1)) k_delete_leaves(const LeafGroup* groups,
                                                          const uint32_t* ngroups, Node* nodes, Pts A, Pts F,
                                                          uint8_t* dead, uint32_t* total) {
  __shared__ uint32_t sum_sh[UPW_WARPS];
  const uint32_t n = *ngroups;
  const uint32_t k0 = (blockIdx.x * UPW_WARPS + warp_id()) * UPW;
  const int lane = lane_id();
  uint32_t gone = 0;  // of the warp
  uint32_t slot = 0, a = 0, sz = 0, glen = 0;
  unsigned long long gst = 0;
  if (lane < UPW && k0 + lane < n) {
    const LeafGroup G = groups[k0 + lane];
    const Node leaf = nodes[G.slot];
    slot = G.slot;
    gst = G.start;
    glen = G.len;
    a = leaf.a;
    sz = leaf.size;
  }
  // common case: every leaf of the warp holds at most 32 points and
  // receives at most 32 / UPW batch points; all loads are issued at once
  constexpr int PER = 32 / UPW;
  uint32_t qa[UPW], qsz[UPW], qlen[UPW];
  bool small = true;
#pragma unroll
  for (int q = 0; q < UPW; ++q) {
    qa[q] = __shfl_sync(FULL_MASK, a, q);
    qsz[q] = __shfl_sync(FULL_MASK, sz, q);
    qlen[q] = __shfl_sync(FULL_MASK, glen, q);
    small &= qsz[q] <= 32 && qlen[q] <= (uint32_t)PER;
  }
  if (small) {
    int32_t x[UPW][D];
    uint32_t id[UPW];
#pragma unroll
    for (int q = 0; q < UPW; ++q) {
      id[q] = 0;
      if ((uint32_t)lane < qsz[q]) {
#pragma unroll
        for (int j = 0; j < D; ++j) x[q][j] = A.c[(uint64_t)j * A.stride + qa[q] + lane];
        id[q] = A.id[(uint64_t)qa[q] + lane];
      }
    }
    // lane q * PER + e holds batch point e of leaf q
    const int mq = lane / PER, me = lane % PER;
    const unsigned long long myst = __shfl_sync(FULL_MASK, gst, mq);
    const uint32_t mylen = __shfl_sync(FULL_MASK, glen, mq);
    int32_t fx[D];
    uint32_t fid = 0xFFFFFFFFu;
    if ((uint32_t)me < mylen) {
      const uint64_t r = myst + (uint64_t)me;
#pragma unroll
      for (int j = 0; j < D; ++j) fx[j] = F.c[(uint64_t)j * F.stride + r];
      fid = F.id[r];
    }
#pragma unroll
    for (int q = 0; q < UPW; ++q) {
      bool hit = false;
      for (int t = 0; t < (int)qlen[q]; ++t) {
        const int src = q * PER + t;
        bool same = __shfl_sync(FULL_MASK, fid, src) == id[q];
#pragma unroll
        for (int j = 0; j < D; ++j) same &= __shfl_sync(FULL_MASK, fx[j], src) == x[q][j];
        hit |= same;
      }
      const bool in = (uint32_t)lane < qsz[q];
      hit &= in;
      gone += __popc(__ballot_sync(FULL_MASK, hit));
      if constexpr (MARK) {
        if (hit) dead[(uint64_t)qa[q] + lane] = 1;
      } else {  // the whole leaf is in registers: survivors to the front, in order
        const unsigned m = __ballot_sync(FULL_MASK, in && !hit);
        if (in && !hit) {
          const uint64_t o = (uint64_t)qa[q] + __popc(m & lanemask_lt());
          if (o != (uint64_t)qa[q] + lane) {
#pragma unroll
            for (int j = 0; j < D; ++j) A.c[(uint64_t)j * A.stride + o] = x[q][j];
            A.id[o] = id[q];
          }
        }
        const uint32_t qslot = __shfl_sync(FULL_MASK, slot, q);
        if (lane == 0 && qsz[q]) nodes[qslot].size = (uint32_t)__popc(m);
      }
    }
  } else {
#pragma unroll 1
    for (int q = 0; q < UPW; ++q) {
      if (k0 + q >= n) break;
      const uint32_t qslot = __shfl_sync(FULL_MASK, slot, q);
      const uint32_t qa_ = __shfl_sync(FULL_MASK, a, q), qsz_ = __shfl_sync(FULL_MASK, sz, q);
      const uint32_t qlen_ = __shfl_sync(FULL_MASK, glen, q);
      const unsigned long long qst = __shfl_sync(FULL_MASK, gst, q);
      uint32_t out = 0;
      for (uint32_t base = 0; base < qsz_; base += 32) {
        const uint32_t i = base + lane;
        bool hit = false;
        int32_t x[D];
        uint32_t id = 0;
        if (i < qsz_) {
          const uint64_t p = (uint64_t)qa_ + i;
#pragma unroll
          for (int j = 0; j < D; ++j) x[j] = A.c[(uint64_t)j * A.stride + p];
          id = A.id[p];
        }
        // the routed batch points, 32 at a time, broadcast lane by lane
        for (uint32_t b0 = 0; b0 < qlen_; b0 += 32) {
          const uint32_t rb = b0 + lane;
          int32_t fx[D];
          uint32_t fid = 0xFFFFFFFFu;
          if (rb < qlen_) {
            const uint64_t r = qst + rb;
#pragma unroll
            for (int j = 0; j < D; ++j) fx[j] = F.c[(uint64_t)j * F.stride + r];
            fid = F.id[r];
          }
          const int cnt = (int)min(32u, qlen_ - b0);
          for (int t = 0; t < cnt; ++t) {
            bool same = __shfl_sync(FULL_MASK, fid, t) == id;
#pragma unroll
            for (int j = 0; j < D; ++j) same &= __shfl_sync(FULL_MASK, fx[j], t) == x[j];
            hit |= same;
          }
        }
        hit &= i < qsz_;
        gone += __popc(__ballot_sync(FULL_MASK, hit));
        if constexpr (MARK) {
          if (hit) dead[(uint64_t)qa_ + i] = 1;
        } else {
          const bool keep = i < qsz_ && !hit;
          const unsigned m = __ballot_sync(FULL_MASK, keep);
          __syncwarp();
          if (keep) {
            const uint64_t o = (uint64_t)qa_ + out + __popc(m & lanemask_lt());
#pragma unroll
            for (int j = 0; j < D; ++j) A.c[(uint64_t)j * A.stride + o] = x[j];
            A.id[o] = id;
          }
          out += __popc(m);
          __syncwarp();
        }
      }
      if (!MARK && lane == 0) nodes[qslot].size = out;
    }
  }
  if (lane == 0) sum_sh[warp_id()] = gone;
  __syncthreads();
  if (threadIdx.x == 0) {
    uint32_t t = 0;
    for (int w = 0; w < UPW_WARPS; ++w) t += sum_sh[w];
    if (t) atomicAdd(total, t);
  }
}

// The marks of a delete's rebuilt subtrees, cleared: one warp per leaf (its
// node record, in the old subtree, is still there).
__global__ void k_clear_dead(const LeafGroup* groups, const uint32_t* ngroups, const Node* nodes, uint8_t* dead) {
  const uint32_t n = *ngroups;
  for (uint32_t g = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; g < n; g += (gridDim.x * blockDim.x) >> 5) {
    const Node nd = nodes[groups[g].slot];
    for (uint32_t i = lane_id(); i < nd.size; i += 32) dead[(uint64_t)nd.a + i] = 0;
  }
}

// The node of every item of at most phi points: a leaf over its new range.
// (Its depth is that of the old subtree's root, so the tree's depth bound
// needs no update.)
__global__ void k_item_leaves(const RebuildItem* it, const uint32_t* n, Node* nodes, uint8_t* ndim, uint32_t phi) {
  const uint32_t i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= *n) return;
  const RebuildItem x = it[i];
  if (x.size > phi) return;
  nodes[x.slot] = Node{0, x.size, x.pos, 0};
  ndim[x.slot] = PKD_LEAF;
}

// Breadth-first flatten of the old subtrees of the rebuild items: every
// frontier entry is (node, item, offset of its live points within the item).
struct Front {
  uint32_t slot;
  uint32_t item;
  uint64_t off;
};

constexpr int FRONT_BATCH = 8;  // frontier levels launched per host check

__global__ void k_front_init(const RebuildItem* it, const uint32_t* n, Front* f, uint32_t* nf) {
  const uint32_t i = blockIdx.x * blockDim.x + threadIdx.x;
  const bool e = i < *n && !it[i].leaf && it[i].old_live != 0;
  const uint32_t c[1] = {e ? 1u : 0u};
  uint32_t* const ctrs[1] = {nf};
  uint32_t first[1];
  block_reserve<1>(c, ctrs, first);
  if (e) f[first[0]] = Front{it[i].slot, i, 0};
}

// One level of the frontier: the grid strides over the device-side count
// *nf (block-uniform), so the host launches a batch of levels without
// reading any count in between; a level with an empty frontier does nothing.
// An entry past a list's capacity is not written: it sets *ovf, and the
// host redoes the flatten with larger lists.  The counts still include such
// entries, so a level reads at most `cap` entries of its frontier, rounded down
// to whole pairs: children are written in pairs from even positions, and a pair
// that does not fit whole is not written (the attempt is redone anyway).  The
// roots always fit with room to spare.
__global__ void k_front_expand(const Front* f, const uint32_t* nf, Front* g, uint32_t* ng, Front* leaves,
                               uint32_t* nleaves, Front* bigleaves, uint32_t* nbig, const Node* nodes,
                               const uint8_t* ndim, const uint32_t* aux, int use_aux, uint32_t cap, uint32_t bcap,
                               uint32_t* ovf) {
  const uint32_t n = min(*nf, cap & ~1u);
  for (uint32_t base = blockIdx.x * blockDim.x; base < n; base += gridDim.x * blockDim.x) {
    const uint32_t i = base + threadIdx.x;
    const bool have = i < n;
    Front e{};
    bool leaf = false, big = false;
    if (have) {
      e = f[i];
      leaf = ndim[e.slot] == PKD_LEAF;
      big = leaf && nodes[e.slot].size > BIG_LEAF;
    }
    const uint32_t c[3] = {have && leaf && !big ? 1u : 0u, have && !leaf ? 2u : 0u, big ? 1u : 0u};
    uint32_t* const ctrs[3] = {nleaves, ng, nbig};
    uint32_t first[3];
    block_reserve<3>(c, ctrs, first);
    if (!have) continue;
    if (leaf) {
      const uint32_t k = big ? first[2] : first[0];
      if (k < (big ? bcap : cap)) (big ? bigleaves : leaves)[k] = e;
      else atomicOr(ovf, 1u);
      continue;
    }
    const Node nd = nodes[e.slot];
    const uint32_t llive = nodes[nd.a].size - (use_aux ? aux[nd.a] : 0u);
    const uint32_t k = first[1];
    if (k + 2 > cap) {
      atomicOr(ovf, 1u);
      continue;
    }
    g[k] = Front{nd.a, e.item, e.off};
    g[k + 1] = Front{nd.b, e.item, e.off + llive};
  }
}

// The whole flatten of a small update in one block: the roots, then level after
// level, the lists' lengths in shared memory (a rebuilt subtree of a few hundred
// points has four levels; as launches, the roots, a batch of levels and their
// counters took 14 of 4 us each).  Returns after FRONT_LEVELS levels at most,
// with what is left of the frontier in f and its length in fc[0].
constexpr uint64_t FRONT_SMALL_POINTS = 8192, FRONT_SMALL_ITEMS = 16384;
constexpr int FRONT_LEVELS = 128;  // even: f holds the frontier at the end
__global__ void __launch_bounds__(512) k_front_small(const RebuildItem* it, const uint32_t* n, Front* f, Front* g,
                                                     uint32_t* fc, Front* leaves, Front* bigleaves, const Node* nodes,
                                                     const uint8_t* ndim, const uint32_t* aux, int use_aux,
                                                     uint32_t cap, uint32_t bcap) {
  __shared__ uint32_t nf[2], nl, nb, ovf;
  if (threadIdx.x == 0) nf[0] = nf[1] = nl = nb = ovf = 0;
  __syncthreads();
  for (uint32_t i = threadIdx.x; i < *n; i += blockDim.x)
    if (!it[i].leaf && it[i].old_live != 0) f[atomicAdd(&nf[0], 1u)] = Front{it[i].slot, i, 0};  // the roots fit
  __syncthreads();
  int lev = 0;
  for (; lev < FRONT_LEVELS; ++lev) {
    const uint32_t c = min(nf[lev & 1], cap & ~1u);
    if (c == 0 || ovf) break;  // uniform: nothing changes them before the barrier below
    __syncthreads();
    if (threadIdx.x == 0) nf[(lev + 1) & 1] = 0;
    __syncthreads();
    for (uint32_t i = threadIdx.x; i < c; i += blockDim.x) {
      const Front e = f[i];
      const Node nd = nodes[e.slot];
      if (ndim[e.slot] == PKD_LEAF) {
        const bool big = nd.size > BIG_LEAF;
        const uint32_t k = atomicAdd(big ? &nb : &nl, 1u);
        if (k < (big ? bcap : cap)) (big ? bigleaves : leaves)[k] = e;
        else ovf = 1;
        continue;
      }
      const uint32_t llive = nodes[nd.a].size - (use_aux ? aux[nd.a] : 0u);
      const uint32_t k = atomicAdd(&nf[(lev + 1) & 1], 2u);
      if (k + 2 > cap) {
        ovf = 1;
        continue;
      }
      g[k] = Front{nd.a, e.item, e.off};
      g[k + 1] = Front{nd.b, e.item, e.off + llive};
    }
    __syncthreads();
    Front* t = f;
    f = g;
    g = t;
  }
  if (threadIdx.x == 0) {
    fc[0] = lev == FRONT_LEVELS ? nf[0] : 0u;
    fc[1] = ovf;
    fc[2] = nl;
    fc[3] = nb;
  }
}

// Flattened leaves, UPW per warp: copy their live points to the item's range.
template <int D>
__global__ void __launch_bounds__(UPW_WARPS * 32) k_copy_leaves(const Front* lv, const uint32_t* n,
                                                                const RebuildItem* items, const Node* nodes, Pts A,
                                                                const uint8_t* dead, int use_dead) {
  const uint32_t nn = *n;
  const uint32_t k0 = (blockIdx.x * UPW_WARPS + warp_id()) * UPW;
  if (k0 >= nn) return;
  const int lane = lane_id();
  uint32_t a = 0, sz = 0;
  unsigned long long d0 = 0;
  if (lane < UPW && k0 + lane < nn) {
    const Front e = lv[k0 + lane];
    const Node nd = nodes[e.slot];
    a = nd.a;
    sz = nd.size;
    d0 = (uint64_t)items[e.item].pos + e.off;
  }
  uint32_t qa[UPW], qsz[UPW];
  unsigned long long qd[UPW];
  bool small = true;
#pragma unroll
  for (int q = 0; q < UPW; ++q) {
    qa[q] = __shfl_sync(FULL_MASK, a, q);
    qsz[q] = __shfl_sync(FULL_MASK, sz, q);
    qd[q] = __shfl_sync(FULL_MASK, d0, q);
    small &= qsz[q] <= 32;
  }
  if (small) {
    int32_t x[UPW][D];
    uint32_t id[UPW];
    bool keep[UPW];
#pragma unroll
    for (int q = 0; q < UPW; ++q) {
      keep[q] = lane < qsz[q];
      if (keep[q]) {
        const uint64_t src = (uint64_t)qa[q] + lane;
        if (use_dead) keep[q] = !dead[src];
#pragma unroll
        for (int j = 0; j < D; ++j) x[q][j] = A.c[(uint64_t)j * A.stride + src];
        id[q] = A.id[src];
      }
    }
#pragma unroll
    for (int q = 0; q < UPW; ++q) {
      const unsigned m = __ballot_sync(FULL_MASK, keep[q]);
      if (keep[q]) {
        const uint64_t dst = qd[q] + __popc(m & lanemask_lt());
#pragma unroll
        for (int j = 0; j < D; ++j) A.c[(uint64_t)j * A.stride + dst] = x[q][j];
        A.id[dst] = id[q];
      }
    }
    return;
  }
#pragma unroll 1
  for (int q = 0; q < UPW; ++q) {
    uint32_t out = 0;
    for (uint32_t base = 0; base < qsz[q]; base += 32) {
      const uint32_t i = base + lane;
      const bool keep = i < qsz[q] && !(use_dead && dead[(uint64_t)qa[q] + i]);
      const unsigned m = __ballot_sync(FULL_MASK, keep);
      if (keep) {
        const uint64_t src = (uint64_t)qa[q] + i, dst = qd[q] + out + __popc(m & lanemask_lt());
#pragma unroll
        for (int j = 0; j < D; ++j) A.c[(uint64_t)j * A.stride + dst] = A.c[(uint64_t)j * A.stride + src];
        A.id[dst] = A.id[src];
      }
      out += __popc(m);
    }
  }
}

// Rebuild items, UPW per warp: the item's build segment; a leaf item's stored
// points (an insert's items are mostly leaves) and the new points of an item
// with at most NEW_BIG of them go to its arena range.  The larger ones are
// left to k_copy_new_flat, the other old subtrees to the flatten.
// An item of at most phi points is a leaf again (Build wraps it): its segment
// is skipped by the rebuild, which then only visits the items that split, and
// k_item_leaves writes its node once its points are in place.
constexpr uint64_t NEW_BIG = 256;
template <int D>
__global__ void __launch_bounds__(UPW_WARPS * 32, (D <= 3 ? 6 : 1)) k_copy_items(const RebuildItem* items,
                                                            const uint32_t* n, const Node* nodes, Pts F, Pts A,
                                                            Seg* segs, uint32_t phi) {
  const uint32_t nn = *n;
  const uint32_t k0 = (blockIdx.x * UPW_WARPS + warp_id()) * UPW;
  if (k0 >= nn) return;
  const int lane = lane_id();
  unsigned long long ws = 0, cnt = 0, pos = 0;
  uint32_t a = 0, sz = 0, live = 0;
  if (lane < UPW && k0 + lane < nn) {
    const RebuildItem it = items[k0 + lane];
    ws = it.ws;
    cnt = it.nw;
    pos = it.pos;
    live = it.old_live;
    if (it.leaf) {
      const Node nd = nodes[it.slot];
      a = nd.a;
      sz = nd.size;
    }
    segs[k0 + lane] = Seg{it.pos, it.size <= phi ? SEG_SKIP : it.size, it.depth, it.slot, IN_A};
  }
  // common case: leaves of at most 32 points, at most 32 / UPW new points per
  // item, one per lane: every load before the first store
  constexpr int PER = 32 / UPW;
  const int mq = lane / PER, me = lane % PER;
  const unsigned long long mws = __shfl_sync(FULL_MASK, ws, mq), mcnt = __shfl_sync(FULL_MASK, cnt, mq);
  const unsigned long long md = __shfl_sync(FULL_MASK, pos, mq) + __shfl_sync(FULL_MASK, live, mq);
  const bool few = __all_sync(FULL_MASK, mcnt <= (unsigned long long)PER);
  if (few && __all_sync(FULL_MASK, sz <= 32)) {
    int32_t x[UPW][D], fx[D];
    uint32_t id[UPW], fid = 0;
#pragma unroll
    for (int q = 0; q < UPW; ++q) {
      const uint32_t qa = __shfl_sync(FULL_MASK, a, q), qsz = __shfl_sync(FULL_MASK, sz, q);
      if ((uint32_t)lane < qsz) {
#pragma unroll
        for (int j = 0; j < D; ++j) x[q][j] = A.c[(uint64_t)j * A.stride + qa + lane];
        id[q] = A.id[(uint64_t)qa + lane];
      }
    }
    if ((unsigned long long)me < mcnt) {
#pragma unroll
      for (int j = 0; j < D; ++j) fx[j] = F.c[(uint64_t)j * F.stride + mws + me];
      fid = F.id[mws + me];
    }
#pragma unroll
    for (int q = 0; q < UPW; ++q) {
      const uint32_t qsz = __shfl_sync(FULL_MASK, sz, q);
      const unsigned long long o = __shfl_sync(FULL_MASK, pos, q) + lane;
      if ((uint32_t)lane < qsz) {
#pragma unroll
        for (int j = 0; j < D; ++j) A.c[(uint64_t)j * A.stride + o] = x[q][j];
        A.id[o] = id[q];
      }
    }
    if ((unsigned long long)me < mcnt) {
#pragma unroll
      for (int j = 0; j < D; ++j) A.c[(uint64_t)j * A.stride + md + me] = fx[j];
      A.id[md + me] = fid;
    }
    return;
  }
#pragma unroll 1
  for (int q = 0; q < UPW; ++q) {
    const unsigned long long qws = __shfl_sync(FULL_MASK, ws, q), qcnt = __shfl_sync(FULL_MASK, cnt, q);
    const unsigned long long qpos = __shfl_sync(FULL_MASK, pos, q);
    const uint32_t qa = __shfl_sync(FULL_MASK, a, q), qsz = __shfl_sync(FULL_MASK, sz, q);
    const uint32_t qlive = __shfl_sync(FULL_MASK, live, q);
    for (uint32_t i = lane; i < qsz; i += 32) {
      const uint64_t src = (uint64_t)qa + i, dst = qpos + i;
#pragma unroll
      for (int j = 0; j < D; ++j) A.c[(uint64_t)j * A.stride + dst] = A.c[(uint64_t)j * A.stride + src];
      A.id[dst] = A.id[src];
    }
    if (qcnt > NEW_BIG) continue;  // k_copy_new_flat copies these
    for (uint64_t i = lane; i < qcnt; i += 32) {
      const uint64_t src = qws + i, dst = qpos + qlive + i;
#pragma unroll
      for (int j = 0; j < D; ++j) A.c[(uint64_t)j * A.stride + dst] = F.c[(uint64_t)j * F.stride + src];
      A.id[dst] = F.id[src];
    }
  }
}

// Insert: every new batch point of the rebuild items with more than NEW_BIG
// of them, one thread each: cnt[i] = those points of item i (0 for the
// others), off = their exclusive scan, so point j of
// the flat order belongs to the item whose range [off[i], off[i] + cnt[i])
// holds it (binary search).  A clustered batch can put millions of points
// into one item; this keeps all of them in flight instead of one warp's.
__global__ void k_item_newcounts(const RebuildItem* it, const uint32_t* n, uint32_t* cnt) {
  const uint32_t i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < *n) {
    const uint32_t c = it[i].nw;
    cnt[i] = c > NEW_BIG ? c : 0u;  // the items k_copy_items leaves out
  }
}

template <int D>
__global__ void __launch_bounds__(256) k_copy_new_flat(const RebuildItem* items, const uint32_t* n,
                                                       const uint32_t* off, const uint32_t* cnt, uint64_t m, Pts F,
                                                       Pts A) {
  const uint32_t ni = *n;
  if (ni == 0) return;
  const uint64_t total = (uint64_t)off[ni - 1] + cnt[ni - 1];
  for (uint64_t j = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; j < total && j < m;
       j += (uint64_t)gridDim.x * blockDim.x) {
    uint32_t lo = 0, hi = ni;  // the last item whose offset is <= j
    while (hi - lo > 1) {
      const uint32_t mid = (lo + hi) >> 1;
      if (off[mid] <= j) lo = mid;
      else hi = mid;
    }
    const RebuildItem it = items[lo];
    const uint64_t k = j - off[lo];
    const uint64_t src = it.ws + k, dst = (uint64_t)it.pos + it.old_live + k;
#pragma unroll
    for (int q = 0; q < D; ++q) A.c[(uint64_t)q * A.stride + dst] = F.c[(uint64_t)q * F.stride + src];
    A.id[dst] = F.id[src];
  }
}

// Flattened leaves of more than BIG_LEAF points (heavy leaves, or leaves
// after skewed updates), one block each: live points keep their leaf's
// relative order, compacted by a block-wide ballot scan per 256 points.

template <int D>
__global__ void __launch_bounds__(256) k_copy_big_leaves(const Front* lv, const uint32_t* n,
                                                         const RebuildItem* items, const Node* nodes, Pts A,
                                                         const uint8_t* dead, int use_dead) {
  __shared__ int wsum[8];
  const uint32_t nn = *n;
  for (uint32_t k = blockIdx.x; k < nn; k += gridDim.x) {
    const Front e = lv[k];
    const Node nd = nodes[e.slot];
    const uint64_t d0 = (uint64_t)items[e.item].pos + e.off;
    uint64_t out = 0;
    for (uint32_t base = 0; base < nd.size; base += 256) {
      const uint32_t i = base + threadIdx.x;
      const uint64_t src = (uint64_t)nd.a + i;
      const bool keep = i < nd.size && !(use_dead && dead[src]);
      int32_t x[D];
      uint32_t id = 0;
      if (keep) {
#pragma unroll
        for (int q = 0; q < D; ++q) x[q] = A.c[(uint64_t)q * A.stride + src];
        id = A.id[src];
      }
      const unsigned m = __ballot_sync(FULL_MASK, keep);
      if (lane_id() == 0) wsum[warp_id()] = __popc(m);
      __syncthreads();
      int before = 0, tot = 0;
      for (int w = 0; w < 8; ++w) {
        if (w < warp_id()) before += wsum[w];
        tot += wsum[w];
      }
      if (keep) {
        const uint64_t dst = d0 + out + before + __popc(m & lanemask_lt());
#pragma unroll
        for (int q = 0; q < D; ++q) A.c[(uint64_t)q * A.stride + dst] = x[q];
        A.id[dst] = id;
      }
      out += tot;
      __syncthreads();
    }
  }
}

template <int D>
static void launch_copy_new_flat(const RebuildItem* items, const uint32_t* n, const uint32_t* off,
                                 const uint32_t* cnt, uint64_t m, Pts F, Pts A, cudaStream_t s) {
  const unsigned g = (unsigned)std::min<uint64_t>((m + 255) / 256, 152ull * 32);
  PKD_LAUNCH(k_copy_new_flat<D><<<std::max(g, 1u), 256, 0, s>>>(items, n, off, cnt, m, F, A));
}
template <int D>
static void launch_copy_big_leaves(const Front* lv, const uint32_t* n, uint32_t nh, const RebuildItem* items,
                                   const Node* nodes, Pts A, const uint8_t* dead, int use_dead, cudaStream_t s) {
  const unsigned g = std::min<uint32_t>(nh, 152u * 8);
  PKD_LAUNCH(k_copy_big_leaves<D><<<std::max(g, 1u), 256, 0, s>>>(lv, n, items, nodes, A, dead, use_dead));
}

template <int D>
static void launch_delete(bool mark, const LeafGroup* g, const uint32_t* ng, uint32_t n, Node* nodes, Pts A, Pts F,
                          uint8_t* dead, uint32_t* total, cudaStream_t s) {
  if (mark) PKD_LAUNCH((k_delete_leaves<D, true><<<upw_blocks(n), UPW_WARPS * 32, 0, s>>>(g, ng, nodes, A, F, dead, total)));
  else PKD_LAUNCH((k_delete_leaves<D, false><<<upw_blocks(n), UPW_WARPS * 32, 0, s>>>(g, ng, nodes, A, F, dead, total)));
}
template <int D>
static void launch_copy_leaves(const Front* lv, const uint32_t* n, uint32_t nh, const RebuildItem* items,
                               const Node* nodes, Pts A, const uint8_t* dead, int use_dead, cudaStream_t s) {
  PKD_LAUNCH(k_copy_leaves<D><<<upw_blocks(nh), UPW_WARPS * 32, 0, s>>>(lv, n, items, nodes, A, dead, use_dead));
}
template <int D>
static void launch_copy_items(const RebuildItem* items, const uint32_t* n, uint32_t nh, const Node* nodes, Pts F, Pts A,
                              Seg* segs, uint32_t phi, cudaStream_t s) {
  PKD_LAUNCH(k_copy_items<D><<<upw_blocks(nh), UPW_WARPS * 32, 0, s>>>(items, n, nodes, F, A, segs, phi));
}

// The items of a round that one team answers each; nmid and nsmall bound (or
// are) their numbers.
template <int D>
static void launch_route(const RouteArgs& a, const Seg* mid, const uint32_t* d_nmid, uint32_t nmid, const Seg* small,
                         const uint32_t* d_nsmall, uint32_t nsmall, cudaStream_t s) {
  const size_t per = skel_bytes(a.HN, a.NB), warps = per * WARP_TEAMS;
  if (warps > 48 * 1024) allow_smem<k_route<D, 32>>(warps);  // (a CTA's one skeleton: 37 KB at lambda = 10)
  if (nmid) PKD_LAUNCH((k_route<D, MID_TEAM><<<nmid, MID_TEAM, per, s>>>(a, mid, d_nmid)));
  if (nsmall) {
    // persistent warps: each remembers the largest sizes that it has sent
    const unsigned g = std::min<unsigned>((nsmall + WARP_TEAMS - 1) / WARP_TEAMS, (unsigned)sm_count() * 8);
    PKD_LAUNCH((k_route<D, 32><<<g, 32 * WARP_TEAMS, warps, s>>>(a, small, d_nsmall)));
  }
}

// The recorded sizes of the nodes that stay, applied once the update can no
// longer fail for lack of memory.
__global__ void k_apply_sizes(const uint2* stay, const uint32_t* n, uint32_t cap, Node* nodes) {
  const uint32_t nn = min(*n, cap);
  for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < nn; i += gridDim.x * blockDim.x)
    nodes[stay[i].x].size = stay[i].y;
}

__global__ void k_clear_aux(const uint32_t* slots, const uint32_t* n, uint32_t cap, uint32_t* aux) {
  const uint32_t nn = min(*n, cap);
  for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < nn; i += gridDim.x * blockDim.x) aux[slots[i]] = 0;
}

// The counters of an update, zeroed, and its first round: one item, the root.
__global__ void k_update_init(uint32_t* ctl, uint32_t words, Seg root, Seg* list, int which) {
  for (uint32_t i = threadIdx.x; i < words; i += blockDim.x) ctl[i] = (int)i == which ? 1u : 0u;
  if (threadIdx.x == 0) *list = root;
}

__global__ void k_stage(const int32_t* coords, const uint32_t* ids, uint64_t m, int d, Pts W) {
  const uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= m) return;
  for (int j = 0; j < d; ++j) W.c[(uint64_t)j * W.stride + i] = coords[i * d + j];
  W.id[i] = ids[i];
}

// ---------------------------------------------------------------------------
// host
// ---------------------------------------------------------------------------

// Grow the arena (and the per-position node region) to hold `need` more
// points; node slots do not move, so the tree stays valid.
static int ensure_capacity(TreeMem& t, uint64_t need, cudaStream_t s) {
  if (t.top + need <= t.cap) return PKD_OK;
  uint64_t ncap = std::max<uint64_t>(t.cap + t.cap / 2, t.top + need + 4096);
  const uint64_t nnode = t.shared_cap + 2 * ncap;
  if (nnode >= 0xFFFFFFF0ull) return PKD_ENOMEM;
  Pts A2{};
  Node* n2 = nullptr;
  uint8_t* d2 = nullptr;
  cudaError_t e = big_alloc((void**)&A2.c, (size_t)t.p.d * ncap * 4, s);
  if (e == cudaSuccess) e = big_alloc((void**)&A2.id, (size_t)ncap * 4, s);
  if (e == cudaSuccess) e = big_alloc((void**)&n2, (size_t)nnode * sizeof(Node), s);
  if (e == cudaSuccess) e = big_alloc((void**)&d2, (size_t)nnode, s);
  if (e != cudaSuccess) {
    cudaGetLastError();
    for (void* q : {(void*)A2.c, (void*)A2.id, (void*)n2, (void*)d2}) big_free(q, s);
    return PKD_ENOMEM;
  }
  A2.stride = ncap;
  for (int j = 0; j < t.p.d; ++j)
    PKD_CUDA(cudaMemcpyAsync(A2.c + (uint64_t)j * ncap, t.A.c + (uint64_t)j * t.cap, t.top * 4,
                             cudaMemcpyDeviceToDevice, s));
  PKD_CUDA(cudaMemcpyAsync(A2.id, t.A.id, t.top * 4, cudaMemcpyDeviceToDevice, s));
  const uint64_t used = t.shared_cap + 2 * t.top;
  PKD_CUDA(cudaMemcpyAsync(n2, t.nodes, used * sizeof(Node), cudaMemcpyDeviceToDevice, s));
  PKD_CUDA(cudaMemcpyAsync(d2, t.ndim, used, cudaMemcpyDeviceToDevice, s));
  // delete scratch grows with the arena and keeps its marks
  uint8_t* dead2 = nullptr;
  uint32_t* aux2 = nullptr;
  if (t.dead) e = big_alloc((void**)&dead2, ncap, s);
  if (e == cudaSuccess && t.aux) e = big_alloc((void**)&aux2, nnode * 4, s);
  if (e != cudaSuccess) {  // nothing of the tree has changed
    cudaGetLastError();
    for (void* q : {(void*)A2.c, (void*)A2.id, (void*)n2, (void*)d2, (void*)dead2, (void*)aux2}) big_free(q, s);
    return PKD_ENOMEM;
  }
  if (dead2) {
    PKD_TRY(dev_fill(dead2, 0, ncap, s));
    PKD_CUDA(cudaMemcpyAsync(dead2, t.dead, t.cap, cudaMemcpyDeviceToDevice, s));
  }
  if (aux2) {
    PKD_TRY(dev_fill(aux2, 0, nnode * 4, s));
    PKD_CUDA(cudaMemcpyAsync(aux2, t.aux, t.node_cap * 4, cudaMemcpyDeviceToDevice, s));
  }
  for (void* q : {(void*)t.A.c, (void*)t.A.id, (void*)t.nodes, (void*)t.ndim, (void*)t.dead, (void*)t.aux})
    big_free(q, s);
  t.dead = dead2;
  t.aux = aux2;
  t.A = A2;
  t.nodes = n2;
  t.ndim = d2;
  t.cap = ncap;
  t.node_cap = nnode;
  return PKD_OK;
}

// The delete scratch: aux before the batch is routed, dead when a subtree is
// rebuilt.
static int ensure_aux(TreeMem& t, cudaStream_t s) {
  if (t.aux) return PKD_OK;
  bool zero = false;
  PKD_CUDA(big_alloc_zeroed((void**)&t.aux, t.node_cap * 4, s, &zero));
  if (!zero) PKD_TRY(dev_fill(t.aux, 0, t.node_cap * 4, s));
  else stat_items("scratch_zeroed", t.node_cap * 4);
  return PKD_OK;
}
static int ensure_dead(TreeMem& t, cudaStream_t s) {
  if (t.dead) return PKD_OK;
  bool zero = false;
  PKD_CUDA(big_alloc_zeroed((void**)&t.dead, t.cap, s, &zero));
  if (!zero) PKD_TRY(dev_fill(t.dead, 0, t.cap, s));
  return PKD_OK;
}

// One round of a route: its lists of recorded sizes and of aux words.
struct RouteRound {
  uint2* stay = nullptr;
  uint32_t stay_cap = 0;
  uint32_t* auxs = nullptr;
  uint32_t aux_cap = 0;
  const uint32_t* ctl = nullptr;  // the round's R_* counters
};

static unsigned list_blocks(uint64_t n) {
  return (unsigned)std::max<uint64_t>(1, std::min<uint64_t>((n + 255) / 256, 152 * 8));
}

// The batch comes either point-major from the caller (coords, ids) or
// already staged in structure-of-arrays form (`staged`, a buffer of at least
// m positions that the route may overwrite).  Returns after its work has
// finished, with the tree's status read; *idflags (insert): the id table's
// flags of the batch, nothing of the tree has changed when they are set.
static int run_update(TreeMem& t, const int32_t* coords, const uint32_t* ids, const Pts* staged, uint64_t m,
                      bool insert, uint64_t* n_changed, int* idflags, cudaStream_t s) {
  const Params& p = t.p;
  const int d = p.d, lam = p.lambda, NB = 1 << lam, HN = 2 << lam;
  const int TILE = std::min(std::max(knobs().tile, 256), 4096);
  Scratch sc{s, {}};
  trace_mark(s, insert ? "insert: enter" : "delete: enter");
  if (!insert) PKD_TRY(ensure_aux(t, s));
  trace_mark(s, "upd: delete scratch");

  // batch buffers: W0/W1 ping-pong between the rounds, F final positions
  int32_t *wc[3] = {nullptr, nullptr, nullptr};
  uint32_t* wid[3] = {nullptr, nullptr, nullptr};
  for (int k = staged ? 1 : 0; k < 3; ++k) {
    PKD_TRY(sc.get(&wc[k], (size_t)d * m));
    PKD_TRY(sc.get(&wid[k], m));
  }
  Pts W[2] = {staged ? *staged : Pts{wc[0], wid[0], m}, Pts{wc[1], wid[1], m}};
  Pts F{wc[2], wid[2], m};
  if (!staged) PKD_LAUNCH(k_stage<<<(unsigned)((m + 255) / 256), 256, 0, s>>>(coords, ids, m, d, W[0]));

  // A batch of at most MID_ITEM points needs no sieve: its rounds, at most
  // the tree's height / lambda, are queued one after another on bounds of
  // their lists' lengths, and the host reads the counters once at the end.
  // A larger one reads them after every round, for the next round's sieve
  // and list sizes (about 20 us each), and so does one into a tree too tall for
  // the searches' stacks in shared memory: its rounds are counted by the tallest
  // path, which few batches go down, and the bounds on the lists grow with it
  // (4096 points at a height of 1e5: 3.3 GB and 17000 rounds).
  const bool queued = m <= MID_ITEM && query_height_ok(t);
  const uint32_t height = t.st_host->max_depth;  // an upper bound
  const int max_rounds = (int)std::max<uint64_t>(1, ((uint64_t)height + lam - 1) / lam);
  const uint32_t ctl_words = (uint32_t)(max_rounds + 3) * CTL_STRIDE;
  uint32_t* ctl;
  PKD_TRY(sc.get(&ctl, ctl_words));
  PinnedBlock hblk;
  uint32_t* hu = (uint32_t*)hblk.p;
  if (!hu) return PKD_ENOMEM;
  static_assert((U_WORDS + R_WORDS) * 4 <= PINNED_BLOCK, "counters");
  auto rc = [&](int r) { return ctl + (uint32_t)(r + 1) * CTL_STRIDE; };

  // every routed point ends in one leaf group or rebuild item
  const uint32_t group_cap = (uint32_t)m;
  RouteArgs ra{};
  ra.p = p;
  ra.lam = lam;
  ra.NB = NB;
  ra.HN = HN;
  ra.TILE = TILE;
  ra.insert = insert ? 1 : 0;
  ra.nodes = t.nodes;
  ra.ndim = t.ndim;
  ra.aux = t.aux;
  ra.st = t.st;
  ra.F = F;
  ra.top = t.top;
  ra.u = ctl;
  ra.group_cap = ra.item_cap = group_cap;
  PKD_TRY(sc.get(&ra.items, group_cap));
  if (!insert) {
    PKD_TRY(sc.get(&ra.gout, group_cap));
    PKD_TRY(sc.get(&ra.gin, group_cap));
  }

  // ---- route ----
  std::vector<RouteRound> rounds;
  const Seg root{0, (uint32_t)m, 0, t.root, IN_B};
  Seg* first;
  PKD_TRY(sc.get(&first, 1));
  uint32_t nbig = m > MID_ITEM, nmid = !nbig && m > SMALL_ITEM, nsmall = !nbig && !nmid;
  uint32_t tiles = nbig ? (uint32_t)((m + TILE - 1) / TILE) : 0;
  uint64_t big_pts = nbig ? m : 0;  // points the round's sieve kernels move
  Seg *big = first, *mid = first, *small = first;
  PKD_LAUNCH(k_update_init<<<1, 256, 0, s>>>(ctl, ctl_words, root, first,
                                             (int)CTL_STRIDE + (nbig ? R_BIG : (nmid ? R_MID : R_SMALL))));
  RouteRound all{};  // queued rounds share their lists
  if (queued) {
    // a point's path has at most `height` inner nodes, and a node is listed once
    all.stay_cap = (uint32_t)std::min<uint64_t>(m * std::max<uint32_t>(height, 1), t.node_cap);
    PKD_TRY(sc.get(&all.stay, all.stay_cap));
    if (!insert) {
      all.aux_cap = (uint32_t)std::min<uint64_t>(m * (height + 1ull), t.node_cap);
      PKD_TRY(sc.get(&all.auxs, all.aux_cap));
    }
    all.ctl = rc(max_rounds + 1);
    rounds.push_back(all);
  }
  // From here on, every exit clears the marks a delete sets (the scratch
  // must be zero for the next call).
  struct ClearMarks {
    TreeMem& t;
    const std::vector<RouteRound>& rounds;
    cudaStream_t s;
    bool on;
    const LeafGroup* gin = nullptr;  // the groups whose points were marked
    const uint32_t* ngin = nullptr;
    uint32_t most = 0;
    bool aux = true;  // the routed rounds may have set aux words
    void clear() {
      if (!on) return;
      on = false;
      if (gin) PKD_LAUNCH(k_clear_dead<<<list_blocks((uint64_t)most * 32), 256, 0, s>>>(gin, ngin, t.nodes, t.dead));
      if (!aux) return;
      for (const auto& R : rounds)
        PKD_LAUNCH(k_clear_aux<<<list_blocks(R.aux_cap), 256, 0, s>>>(R.auxs, R.ctl + R_AUX, R.aux_cap, t.aux));
    }
    ~ClearMarks() {
      if (!on) return;
      clear();
      if (cudaPeekAtLastError() == cudaSuccess) t.scratch_dirty = false;
    }
  } marks{t, rounds, s, !insert};
  if (!insert) t.scratch_dirty = true;

  auto read_flags = [&]() {  // the tree's status, with the batch's id flags
    PKD_CUDA(cudaMemcpyAsync(t.st_host, t.st, sizeof(DevStatus), cudaMemcpyDeviceToHost, s));
    PKD_CUDA(cudaStreamSynchronize(s));
    if (idflags) *idflags = t.st_host->idflags;
    return status_code(t.st_host->err, t.st_host->detail);
  };
  int w = 0, r = 0;
  for (;; ++r) {
    const uint64_t nitems = (uint64_t)nbig + nmid + nsmall;  // or a bound
    if (queued ? r == max_rounds : nitems == 0) break;
    if (r > max_rounds) return PKD_EINTERNAL;
    ra.src = W[w];
    ra.dst = W[w ^ 1];
    ra.next = rc(r + 1);
    ra.last = queued && r + 1 == max_rounds;
    ra.cur = queued ? rc(max_rounds + 1) : rc(r);
    if (queued) {
      ra.stay = all.stay;
      ra.stay_cap = all.stay_cap;
      ra.auxs = all.auxs;
      ra.aux_cap = all.aux_cap;
    } else {
      RouteRound R{};
      R.stay_cap = (uint32_t)std::min({m * (uint64_t)lam, nitems * (uint64_t)(NB - 1), t.node_cap});
      PKD_TRY(sc.get(&R.stay, R.stay_cap));
      if (!insert) {
        R.aux_cap = (uint32_t)std::min({m * (uint64_t)(lam + 1), nitems * (uint64_t)(HN - 1), t.node_cap});
        PKD_TRY(sc.get(&R.auxs, R.aux_cap));
      }
      R.ctl = rc(r);
      ra.stay = R.stay;
      ra.stay_cap = R.stay_cap;
      ra.auxs = R.auxs;
      ra.aux_cap = R.aux_cap;
      rounds.push_back(R);
    }
    ra.small = ra.mid = ra.big = nullptr;
    ra.small_cap = ra.mid_cap = ra.big_cap = 0;
    if (!ra.last) {  // every item has NB external nodes and a point at least
      ra.small_cap = (uint32_t)std::min<uint64_t>(m, nitems * NB);
      ra.mid_cap = (uint32_t)std::min<uint64_t>(ra.small_cap, m / (SMALL_ITEM + 1));
      ra.big_cap = queued ? 0 : (uint32_t)std::min<uint64_t>(ra.small_cap, m / (MID_ITEM + 1));
      PKD_TRY(sc.get(&ra.small, ra.small_cap));
      PKD_TRY(sc.get(&ra.mid, ra.mid_cap));
      if (ra.big_cap) PKD_TRY(sc.get(&ra.big, ra.big_cap));
    }
    if (nbig) {
      // big items: fetch, tile histograms, bucket-major scan, emit, scatter
      RoundArgs sa{};
      uint32_t *slots, *sizes, *hist, *hscan, *partial;
      const uint64_t nh = (uint64_t)tiles * NB;
      PKD_TRY(sc.get(&sa.skel, (size_t)nbig * HN));
      PKD_TRY(sc.get(&slots, (size_t)nbig * HN));
      PKD_TRY(sc.get(&sizes, (size_t)nbig * HN));
      PKD_TRY(sc.get(&sa.tile0, nbig));
      PKD_TRY(sc.get(&sa.excl, nbig));
      PKD_TRY(sc.get(&hist, nh));
      PKD_TRY(sc.get(&hscan, nh));
      PKD_TRY(sc.get(&partial, (nh + SCAN_TILE - 1) / SCAN_TILE + 1));
      if (record_buckets(NB)) PKD_TRY(sc.get(&sa.bkt, (size_t)tiles * TILE));
      ra.copy_cap = (uint32_t)(tiles + (uint64_t)nbig * NB);
      PKD_TRY(sc.get(&ra.copy, ra.copy_cap));
      sa.wait_cycles = knobs().wait_cycles;
      sa.p = p;
      sa.lam = lam;
      sa.NB = NB;
      sa.HN = HN;
      sa.TILE = TILE;
      sa.src.soa = W[w];
      sa.dst = W[w ^ 1];
      sa.st = t.st;
      sa.big = big;
      sa.nbig = rc(r) + R_BIG;
      sa.hist = hist;
      sa.hscan = hscan;
      const size_t per = skel_bytes(HN, NB);
      if (per > 48 * 1024) return PKD_EINTERNAL;  // (37 KB at lambda = 10)
      PKD_LAUNCH(k_big_fetch<<<nbig, BIG_TEAM, per, s>>>(ra, big, sa.skel, slots, sizes));
      PKD_LAUNCH(k_big_prefix<<<1, 1024, 0, s>>>(big, sa.nbig, (uint32_t)TILE, sa.tile0, sa.excl));
      PKD_DISPATCH_D(d, launch_count, sa, tiles, big_pts, "count_route", s);
      device_excl_scan(hist, hscan, nh, partial, s);
      PKD_LAUNCH(k_big_emit<<<nbig, BIG_TEAM, per, s>>>(ra, sa, slots, sizes));
      PKD_DISPATCH_D(d, launch_scatter, sa, tiles, big_pts, "scatter_route", s);
      PKD_LAUNCH(k_copy_ended<<<std::min<uint32_t>(ra.copy_cap, 152 * 8), 256, 0, s>>>(ra, rc(r) + R_COPY));
    }
    PKD_DISPATCH_D(d, launch_route, ra, mid, rc(r) + R_MID, nmid, small, rc(r) + R_SMALL, nsmall, s);
    if (queued) {
      nmid = ra.mid_cap;
      nsmall = ra.small_cap;
    } else {
      PKD_CUDA(cudaMemcpyAsync(hu + U_WORDS, rc(r + 1), R_WORDS * 4, cudaMemcpyDeviceToHost, s));
      PKD_TRY(read_flags());
      if (idflags && *idflags) return PKD_OK;
      const uint32_t* nx = hu + U_WORDS;
      nbig = nx[R_BIG];
      nmid = nx[R_MID];
      nsmall = nx[R_SMALL];
      tiles = nx[R_TILES];
      big_pts = nx[R_BIGPTS];
    }
    big = ra.big;
    mid = ra.mid;
    small = ra.small;
    w ^= 1;
  }
  PKD_CUDA(cudaMemcpyAsync(hu, ctl, U_WORDS * 4, cudaMemcpyDeviceToHost, s));
  PKD_TRY(read_flags());
  if (idflags && *idflags) return PKD_OK;
  const uint32_t nitems = hu[U_ITEMS], ninner = hu[U_INNER], ngout = hu[U_GOUT], ngin = hu[U_GIN];
  const uint64_t total = hu[U_TOTAL];
  const uint64_t inner_total = *(unsigned long long*)(hu + U_INNER_PTS);
  marks.aux = ninner != 0;
  const uint32_t* d_nitems = ctl + U_ITEMS;
  const RebuildItem* items = ra.items;
  stat_items(insert ? "rebuilt_insert" : "rebuilt_delete", total);
  trace_mark(s, "upd: route");

  // ---- rebuild ----
  // Nothing the tree shows has changed so far: the new sizes are recorded,
  // the leaves to compact are listed.  The new subtrees are built in fresh
  // arena positions (past top), and every allocation, the build's included,
  // comes before the first write to a node, so PKD_ENOMEM leaves the tree as
  // it was.
  if (nitems) {
    PKD_TRY(ensure_capacity(t, total, s));
    trace_mark(s, "upd: ensure capacity");
    if (ngin) {  // a delete's marks in the subtrees that are rebuilt
      PKD_TRY(ensure_dead(t, s));
      PKD_DISPATCH_D(d, launch_delete, true, ra.gin, ctl + U_GIN, ngin, t.nodes, t.A, F, t.dead, ctl + U_FOUND, s);
      marks.gin = ra.gin;
      marks.ngin = ctl + U_GIN;
      marks.most = ngin;
    }
    Seg* segs;
    PKD_TRY(sc.get(&segs, nitems));
    const unsigned gi = (nitems + 127) / 128;
    PKD_DISPATCH_D(d, launch_copy_items, items, d_nitems, nitems, t.nodes, F, t.A, segs, (uint32_t)p.phi, s);
    if (hu[U_MAXNEW] > NEW_BIG) {
      uint32_t *ncnt, *noff, *npart;
      PKD_TRY(sc.get(&ncnt, nitems));
      PKD_TRY(sc.get(&noff, nitems));
      PKD_TRY(sc.get(&npart, ((uint64_t)nitems + SCAN_TILE - 1) / SCAN_TILE + 1));
      PKD_LAUNCH(k_item_newcounts<<<gi, 128, 0, s>>>(items, d_nitems, ncnt));
      device_excl_scan(ncnt, noff, nitems, npart, s);
      PKD_DISPATCH_D(d, launch_copy_new_flat, items, d_nitems, noff, ncnt, m, F, t.A, s);
    }
    if (ninner) {
      // Flatten the old subtrees that are not single leaves, breadth first.
      // Capacity of the lists: every node of the old subtrees appears once: a
      // subtree of P stored points has at most 2P - 1 nodes unless deletes
      // left empty leaves in it.  When a level overflows that, the flatten is
      // redone with four entries per stored point of the tree.  The levels run
      // in batches whose counts stay on the device; the host reads the
      // frontier once per batch (a rebuilt subtree is many levels deep).
      const uint64_t big_fcap = 4 * ((uint64_t)t.size + (uint64_t)nitems) + 1024;
      uint64_t fcap = 2 * inner_total + (uint64_t)ninner + 1024;
      if (knobs().front_cap > 0) fcap = (uint64_t)knobs().front_cap;
      fcap = std::max<uint64_t>(std::min(fcap, big_fcap), (uint64_t)ninner + 1024);  // the roots always fit
      Front *fa = nullptr, *fb = nullptr, *leaves = nullptr, *bigleaves = nullptr;
      uint32_t* fc;  // [0] frontier, [1] overflow, [2] leaves, [3] big leaves
      uint32_t* lc;  // the frontier of every level of a batch
      PKD_TRY(sc.get(&fc, 4));
      PKD_TRY(sc.get(&lc, FRONT_BATCH + 1));
      const unsigned gexp = (unsigned)sm_count() * 8;
      uint32_t* hf = hu + U_WORDS;
      for (;;) {
        const uint32_t fcap32 = (uint32_t)std::min<uint64_t>(fcap, 0xFFFFFFF0ull);
        const uint32_t bcap32 = (uint32_t)std::min<uint64_t>(fcap / BIG_LEAF + 16 + ninner, 0xFFFFFFF0ull);
        PKD_TRY(sc.get(&fa, fcap32));
        PKD_TRY(sc.get(&fb, fcap32));
        PKD_TRY(sc.get(&leaves, fcap32));
        PKD_TRY(sc.get(&bigleaves, bcap32));
        int levels = 0;
        if (inner_total <= FRONT_SMALL_POINTS && nitems <= FRONT_SMALL_ITEMS) {
          PKD_LAUNCH(k_front_small<<<1, 512, 0, s>>>(items, d_nitems, fa, fb, fc, leaves, bigleaves, t.nodes, t.ndim,
                                                     t.aux, insert ? 0 : 1, fcap32, bcap32));
          levels = FRONT_LEVELS;
          PKD_CUDA(cudaMemcpyAsync(hf, fc, 16, cudaMemcpyDeviceToHost, s));
          PKD_CUDA(cudaStreamSynchronize(s));
        } else {
          PKD_TRY(dev_fill(fc, 0, 16, s));
          PKD_LAUNCH(k_front_init<<<gi, 128, 0, s>>>(items, d_nitems, fa, fc));
          hf[0] = 1;
          hf[1] = 0;
        }
        while (hf[0] != 0 && hf[1] == 0) {
          if (levels > 100000) return PKD_EINTERNAL;
          PKD_TRY(dev_fill(lc + 1, 0, (size_t)FRONT_BATCH * 4, s));
          PKD_TRY(dev_copy_words(lc, fc, 1, s));
          for (int k = 0; k < FRONT_BATCH; ++k) {
            PKD_LAUNCH(k_front_expand<<<gexp, 128, 0, s>>>(fa, lc + k, fb, lc + k + 1, leaves, fc + 2, bigleaves,
                                                            fc + 3, t.nodes, t.ndim, t.aux, insert ? 0 : 1, fcap32,
                                                            bcap32, fc + 1));
            std::swap(fa, fb);
          }
          levels += FRONT_BATCH;
          PKD_TRY(dev_copy_words(fc, lc + FRONT_BATCH, 1, s));
          PKD_CUDA(cudaMemcpyAsync(hf, fc, 16, cudaMemcpyDeviceToHost, s));
          PKD_CUDA(cudaStreamSynchronize(s));
        }
        if (hf[1] == 0) break;
        // a list overflowed: nothing the tree shows has changed yet
        if (fcap >= big_fcap) return PKD_EINTERNAL;
        stat_items("front_retries", 1);
        fcap = big_fcap;
      }
      if (hf[2])
        PKD_DISPATCH_D(d, launch_copy_leaves, leaves, fc + 2, hf[2], items, t.nodes, t.A, t.dead, ngin ? 1 : 0, s);
      if (hf[3])
        PKD_DISPATCH_D(d, launch_copy_big_leaves, bigleaves, fc + 3, hf[3], items, t.nodes, t.A, t.dead, ngin ? 1 : 0,
                       s);
    }
    trace_mark(s, "upd: flatten + gather");
    BuildJob job;
    job.base = t.top;
    job.extent = std::max<uint64_t>(total, 1);
    job.dsegs = segs;
    job.dsegs_n = nitems;
    job.max_len = hu[U_MAX];
    PKD_TRY(run_build(t, job, s));
    PKD_LAUNCH(k_item_leaves<<<gi, 128, 0, s>>>(items, d_nitems, t.nodes, t.ndim, (uint32_t)p.phi));
    trace_mark(s, "upd: rebuild");
  }

  // ---- the visible changes: nothing below allocates ----
  if (ngout)  // delete: the reached leaves lose their deleted points
    PKD_DISPATCH_D(d, launch_delete, false, ra.gout, ctl + U_GOUT, ngout, t.nodes, t.A, F, nullptr, ctl + U_FOUND, s);
  for (const auto& R : rounds)
    PKD_LAUNCH(k_apply_sizes<<<list_blocks(R.stay_cap), 256, 0, s>>>(R.stay, R.ctl + R_STAY, R.stay_cap, t.nodes));
  t.top += total;
  marks.clear();
  PKD_CUDA(cudaMemcpyAsync(hu, ctl, U_WORDS * 4, cudaMemcpyDeviceToHost, s));
  const int e = read_flags();  // waits for everything
  if (!insert && cudaPeekAtLastError() == cudaSuccess) t.scratch_dirty = false;  // every mark is cleared
  trace_mark(s, "upd: cleanup");
  if (n_changed) *n_changed = insert ? m : hu[U_FOUND];
  return e;
}

}  // namespace pkd

using namespace pkd;

extern "C" {

int pkd_batch_insert(pkd_tree* tc, const int32_t* coords, const uint32_t* ids, uint64_t m, void* stream) {
  if (!tc) return PKD_EINVAL;
  if (m == 0) return PKD_OK;
  if (!coords || !ids) return PKD_EINVAL;
  TreeMem& t = tc->m;
  if (t.size + m >= (1ull << 31)) return PKD_EINVAL;
  cudaStream_t s = (cudaStream_t)stream;
  TreeTouch touch{&t, s};
  {
    QueryCheck check(t, s);
    PKD_TRY_(check.begin(coords, m * (uint64_t)t.p.d, nullptr, 0));
    PKD_TRY_(check.end());
  }
  // the batch's ids take their slots first: a stored or repeated id rejects
  // the whole batch before the tree changes (the flags are read with the
  // route's counters)
  PKD_TRY_(ids_reserve(t, m, s));
  uint64_t* slots = nullptr;
  PKD_TRY_(dalloc(&slots, m, s));
  ids_claim(t, coords, ids, m, slots, s);
  t.ids.used += m;
  int fl = 0;
  int e = run_update(t, coords, ids, nullptr, m, true, nullptr, &fl, s);
  if (e != PKD_OK || fl) {  // the flags, read and cleared: a bad batch is told as such
    const int ec = read_idflags(t, s, &fl);
    if (fl && (e == PKD_OK || e == PKD_ENOMEM)) e = (fl & IDF_FULL) ? PKD_EINTERNAL : PKD_EINVAL;
    if (ec != PKD_OK) e = ec;
  }
  if (e == PKD_OK) {
    t.size += m;
    t.ids.live += m;
    if (t.bbox_on) e = boxes_compute(t, s);
  } else {
    ids_unclaim(t, slots, m, s);
  }
  dfree(slots, s);
  return e;
}

int pkd_batch_delete(pkd_tree* tc, const uint32_t* ids, uint64_t m, uint64_t* n_deleted, void* stream) {
  if (!tc) return PKD_EINVAL;
  if (n_deleted) *n_deleted = 0;
  if (m == 0) return PKD_OK;
  if (!ids) return PKD_EINVAL;
  TreeMem& t = tc->m;
  if (m >= (1ull << 31)) return PKD_EINVAL;
  cudaStream_t s = (cudaStream_t)stream;
  PKD_TRY_(refuse_capture(s));
  TreeTouch touch{&t, s};
  // ids -> coordinates: every LIVE id of the batch is taken once (repeats and
  // unknown or deleted ids are skipped) and staged for the sieve; whatever
  // refuses the call after that gives them back
  PinnedBlock hb;
  if (!hb.p) return PKD_ENOMEM;
  Scratch sc{s, {}};
  const int d = t.p.d;
  int32_t* wc;
  uint32_t *wid, *cnt;
  uint64_t* wslots;
  PKD_TRY(sc.get(&wc, (size_t)d * m));
  PKD_TRY(sc.get(&wid, m));
  PKD_TRY(sc.get(&wslots, m));
  PKD_TRY(sc.get(&cnt, 1));
  PKD_TRY(dev_fill(cnt, 0, 4, s));
  Pts W{wc, wid, m};
  ids_take(t, ids, m, W, wslots, cnt, s);
  PKD_CUDA(cudaMemcpyAsync(hb.p, cnt, 4, cudaMemcpyDeviceToHost, s));
  int fl = 0;
  PKD_TRY(read_idflags(t, s, &fl));  // synchronises s
  int e = status_code(t.st_host->err, t.st_host->detail);
  const uint32_t taken = *(const uint32_t*)hb.p;
  if (e == PKD_OK && fl) e = PKD_EINTERNAL;
  if (e != PKD_OK) {
    ids_restore(t, wslots, taken, s);
    return e;
  }
  stat_items("delete_gather", taken);
  if (taken == 0) return PKD_OK;
  uint64_t removed = 0;
  e = run_update(t, nullptr, nullptr, &W, taken, false, &removed, nullptr, s);
  if (e == PKD_OK && removed != taken) {
    fprintf(stderr, "pkd: delete removed %llu points for %u live ids\n", (unsigned long long)removed, taken);
    e = PKD_EINTERNAL;
  }
  if (e != PKD_OK) ids_restore(t, wslots, taken, s);
  if (e == PKD_OK) {
    t.size -= removed;
    t.ids.live -= removed;
    if (n_deleted) *n_deleted = removed;
    if (t.bbox_on) e = boxes_compute(t, s);
  }
  return e;
}

}  // extern "C"
