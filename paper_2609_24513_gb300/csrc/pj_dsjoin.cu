// Dataset-level join: the paper's own formulation (Sec. 3.1-3.5), next to
// the per-pair refinement of the rest of the library.
//
//   * one BVH over all triangles of a dataset (the same LBVH build as the
//     per-mesh trees, run on the dataset as one mesh; each triangle record
//     then carries its owning mesh -- the paper's triangle-to-object map);
//   * Alg. 1 in both directions (Sec. 3.2 "Bidirectional tracing"): every
//     owned edge of one dataset is tested against the other's triangles around
//     it -- found by walking the two BVHs together, or (a self join, dense
//     data) by sending packets of 32 triangles through the other BVH -- with
//     the exact strict segment/triangle test, and every crossing is recorded:
//     an edge may pierce several objects, so nothing stops at the first hit
//     (the multi-hit loop of Alg. 1);
//   * containment (Sec. 3.3-3.4): each object casts one ray from its
//     lexicographically first vertex through the other dataset's BVH and
//     toggles a parity bit for every object whose triangle it crosses; an
//     odd count records the pair;
//   * materialisation (Sec. 3.5): a hashmap sized by the selectivity
//     estimate (one pass, a relaunch with twice the slots on overflow), the
//     counting two-pass strategy (count, prefix sum, emit, sort, unique), or
//     a hashmap of a fixed size.
//
// Exactness.  The per-pair join's containment test uses, for each pair, the
// first vertex of B_j that is not on A_i's surface.  A parity ray from the
// first vertex decides every pair whose surface does not pass through that
// vertex; pairs whose surface does (checked exactly at the triangles the ray
// meets, which include every triangle holding the vertex), and all pairs of
// a ray that meets more candidate objects than it can track, are handed to
// the per-pair join.  The result therefore equals the per-pair join over the
// bounding-box candidates, which the tests check against the oracle.
#include <cub/cub.cuh>

#include <algorithm>
#include <cstring>
#include <vector>

#include "pj_geom.cuh"
#include "pj_internal.cuh"

namespace pj {

constexpr unsigned long long kHashEmpty = ~0ull;
constexpr int kDsStack = 192;     // plain depth-first order's stack entries
constexpr int kParList = 48;      // objects a parity ray tracks
constexpr int kHashProbes = 2048;  // probes before a hashmap counts as full

enum { DS_EDGES = 0, DS_NODES, DS_TRIS, DS_HITS, DS_RAYS, DS_OVERFLOW, DS_ERR, DS_NREC,
       DS_NOBJ, DS_FULL, DS_NSTAT };

struct DsSide {
  int64_t M, F;
  const float4 *mrec;    // per mesh: box, first lexicographic vertex
  const float *aabb;     // per mesh: closed box
  const float *nodes;    // dataset BVH
  const float4 *trirec;  // its triangle records, .w of the third = owning mesh
};

// where a pair goes: a hashmap, a per-item count, or a slot of a flat buffer
enum { SINK_HASH = 0, SINK_COUNT = 1, SINK_EMIT = 2 };
struct Sink {
  int mode;
  unsigned long long *table;  // SINK_HASH
  unsigned long long mask;    // slots - 1 (a power of two)
  int64_t *cnt;               // SINK_COUNT: per item
  const int64_t *off;         // SINK_EMIT: per item
  unsigned long long *keys;   // SINK_EMIT
  int64_t base;               // this launch's first item index
};

// pairs handed to the per-pair join, and objects whose rays overflowed
struct Recheck {
  int2 *pairs;
  int32_t *objs;
  unsigned long long cap;
};

// MurmurHash3's 64-bit finaliser (Appleby), to spread pair keys over slots
__device__ __forceinline__ unsigned long long mix64(unsigned long long x) {
  x ^= x >> 33;
  x *= 0xff51afd7ed558ccdull;
  x ^= x >> 33;
  x *= 0xc4ceb9fe1a85ec53ull;
  x ^= x >> 33;
  return x;
}

__device__ __forceinline__ void hash_insert(const Sink &k, unsigned long long key,
                                            unsigned long long *st) {
  unsigned long long h = mix64(key) & k.mask;
  for (int i = 0; i < kHashProbes; ++i) {
    // a plain read first: most records repeat a pair already present
    const unsigned long long cur = __ldcg(k.table + h);
    if (cur == key) return;
    if (cur == kHashEmpty) {
      const unsigned long long prev = atomicCAS(k.table + h, kHashEmpty, key);
      if (prev == kHashEmpty || prev == key) return;
    }
    h = (h + 1) & k.mask;
  }
  atomicExch(st + DS_OVERFLOW, 1ull);  // relaunched with more slots
}

__device__ __forceinline__ int64_t mesh_of(const int64_t *off, int64_t M, int64_t e) {
  int64_t lo = 0, hi = M - 1;
  while (lo < hi) {
    int64_t mid = (lo + hi + 1) >> 1;
    if (off[mid] <= e) lo = mid; else hi = mid - 1;
  }
  return lo;
}

__device__ __forceinline__ unsigned long long pair_key(int a, int b, int self_join) {
  if (self_join && a > b) {
    const int t = a;
    a = b;
    b = t;
  }
  return ((unsigned long long)(unsigned)a << 32) | (unsigned)b;
}

__device__ __forceinline__ void flush_stats(unsigned long long *st, const unsigned long long *v,
                                            int n) {
  for (int i = 0; i < n; ++i) {
    unsigned long long x = v[i];
    for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
    if ((threadIdx.x & 31) == 0 && x) atomicAdd(st + i, x);
  }
}

// Alg. 1 in both directions: every owned edge of S through T's BVH, every
// strict crossing recorded; S = A, T = B and the reverse (a self join: S = T =
// A once).
//
// A warp takes a packet of 32 source triangles, consecutive in S's own BVH
// order (so that they mostly lie together), one per lane.  It walks T's BVH
// once for all of them: the children of up to 32 / W nodes, one to a lane, are
// tested against the box around the packet, and each that meets it against
// every lane's triangle; a part of T that no lane meets is never entered.
// Where a child is smaller than the triangle, its owned edges are tested too
// (a vessel's triangle is larger than most of a nucleus: by boxes alone it met
// thousands of leaves that its edges pass by).  A leaf and a lane that meet
// are listed in shared memory and the list is worked off a pair to a lane: box
// tests, then the exact test.
//
// Boxes are compared open: a strict crossing has strictly overlapping boxes
// on every axis (an edge and a triangle whose boxes only touch meet at an
// extreme of one of them, which lies in no relative interior).
//
// What bounds it: the packets' node tests (issue), then reading S's records
// once.  An edge per thread with a stack of its own (no packets, S in input
// order) visited 94.6 M nodes on 1,200 nuclei x 60 vessels (25 M edges) and
// took 2,685 us in both directions, memory latency at every visit:
// 1,100 now.  Packets of 256 triangles (8 a lane, one box) measured
// 3,000-12,000: where the order jumps or triangles are large, 8 triangles'
// box meets far more leaves than they do.
constexpr int kDsPacket = 32;              // source triangles of a warp
constexpr int kDsWarps = 4;                // warps of a block

__device__ __forceinline__ bool open_overlap(F3 alo, F3 ahi, F3 blo, F3 bhi) {
  return alo.x < bhi.x && blo.x < ahi.x && alo.y < bhi.y && blo.y < ahi.y && alo.z < bhi.z &&
         blo.z < ahi.z;
}

struct DsTri {
  F3 v[3];
  int edges, mesh;  // owned-edge bits, owning mesh
};
__device__ __forceinline__ DsTri ds_tri(const float4 *rec, int64_t i) {
  const float4 r0 = __ldg(rec + 3 * i), r1 = __ldg(rec + 3 * i + 1), r2 = __ldg(rec + 3 * i + 2);
  DsTri t;
  t.v[0] = mkf3(r0.x, r0.y, r0.z);
  t.v[1] = mkf3(r0.w, r1.x, r1.y);
  t.v[2] = mkf3(r1.z, r1.w, r2.x);
  t.edges = __float_as_int(r2.y);
  t.mesh = __float_as_int(r2.w);
  return t;
}
__device__ __forceinline__ F3 min3(F3 a, F3 b) {
  return mkf3(fminf(a.x, b.x), fminf(a.y, b.y), fminf(a.z, b.z));
}
__device__ __forceinline__ F3 max3(F3 a, F3 b) {
  return mkf3(fmaxf(a.x, b.x), fmaxf(a.y, b.y), fmaxf(a.z, b.z));
}

__device__ __forceinline__ float warp_min(float v) {
  for (int o = 16; o > 0; o >>= 1) v = fminf(v, __shfl_xor_sync(0xffffffffu, v, o));
  return v;
}

template <int W>
__global__ void __launch_bounds__(32 * kDsWarps, 4) k_ds_edges(DsSide A, DsSide B, int self_join,
                                                               Sink sink,
                                                               unsigned long long *st) {
  constexpr int kDsList = 128;  // listed (lane, leaf) pairs of a warp
  // plain depth-first order (a node at a time) needs at most kDsStack entries;
  // up to 32 / W nodes at a time are taken while no more are used, so one such
  // step and that order on top of it always fit
  constexpr int kCap = 2 * kDsStack + 32;
  __shared__ uint32_t s_stack[kDsWarps][kCap];
  __shared__ uint32_t s_leaf[kDsWarps][kDsList];
  __shared__ uint8_t s_lane[kDsWarps][kDsList];
  const unsigned full = 0xffffffffu;
  const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
  const unsigned lt = (1u << lane) - 1u;
  uint32_t *stk = s_stack[wib];
  uint32_t *leaf = s_leaf[wib];
  uint8_t *leaf_lane = s_lane[wib];
  unsigned long long c_edges = 0, c_nodes = 0, c_tris = 0, c_hits = 0;
  const int SW = node_stride_words(W);
  // B's packets first: there are usually fewer of them with more to do each
  const int64_t nA = (A.F + kDsPacket - 1) / kDsPacket;
  const int64_t nB = self_join ? 0 : (B.F + kDsPacket - 1) / kDsPacket;
  for (int64_t w = blockIdx.x * (int64_t)kDsWarps + wib; w < nA + nB;
       w += gridDim.x * (int64_t)kDsWarps) {
    const int dir = w < nB;
    const int64_t pk = dir ? w : w - nB, item = sink.base + (dir ? nA + pk : pk);
    const float4 *srec = dir ? B.trirec : A.trirec, *trec = dir ? A.trirec : B.trirec;
    const float *tnodes = dir ? A.nodes : B.nodes;
    const int64_t SF = dir ? B.F : A.F;
    int64_t n_rec = 0;  // the packet's records (the same in every lane)
    const int64_t f0 = pk * kDsPacket;
    // this lane's triangle, its box (no owned edge: lo > hi, which overlaps
    // nothing)
    F3 lo = mkf3(3e38f, 3e38f, 3e38f), hi = mkf3(-3e38f, -3e38f, -3e38f);
    float side = 0.f;
    if (f0 + lane < SF) {
      const DsTri tri = ds_tri(srec, f0 + lane);
      if (tri.edges) {
        c_edges += __popc(tri.edges);
        lo = min3(tri.v[0], min3(tri.v[1], tri.v[2]));
        hi = max3(tri.v[0], max3(tri.v[1], tri.v[2]));
        side = fmaxf(hi.x - lo.x, fmaxf(hi.y - lo.y, hi.z - lo.z));
      }
    }
    // the box around the packet's
    F3 ulo, uhi;
    ulo.x = warp_min(lo.x);
    ulo.y = warp_min(lo.y);
    ulo.z = warp_min(lo.z);
    uhi.x = -warp_min(-hi.x);
    uhi.y = -warp_min(-hi.y);
    uhi.z = -warp_min(-hi.z);
    int sp = 1, nl = 0;
    unsigned pend = 0;  // children that meet the packet's box, not yet seen to
    F3 blo, bhi;        // this lane's child
    uint32_t word = 0;
    if (lane == 0) stk[0] = 0u;
    __syncwarp();
    for (;;) {
      // work off the listed pairs when a child's might not fit, or nothing
      // else is left
      if (nl + 32 > kDsList || (sp == 0 && !pend)) {
        if (nl == 0) break;
        for (int i0 = 0; i0 < nl; i0 += 32) {
          const int i = i0 + lane;
          DsTri a;
          int cnt = 0;
          int64_t first = 0;
          F3 alo = mkf3(0.f, 0.f, 0.f), ahi = alo;
          if (i < nl) {
            a = ds_tri(srec, f0 + leaf_lane[i]);
            alo = min3(a.v[0], min3(a.v[1], a.v[2]));
            ahi = max3(a.v[0], max3(a.v[1], a.v[2]));
            first = (leaf[i] >> 3) & 0x0FFFFFFFu;
            cnt = (int)(leaf[i] & 7u) + 1;
          }
          const int most = __reduce_max_sync(full, cnt);
          for (int t = 0; t < most; ++t) {
            DsTri b;
            unsigned ek = 0;  // edges whose box overlaps the triangle's
            if (t < cnt) {
              b = ds_tri(trec, first + t);
              const F3 blo = min3(b.v[0], min3(b.v[1], b.v[2]));
              const F3 bhi = max3(b.v[0], max3(b.v[1], b.v[2]));
              if (open_overlap(alo, ahi, blo, bhi) && !(self_join && a.mesh == b.mesh)) {
#pragma unroll
                for (int k = 0; k < 3; ++k) {
                  const F3 p = a.v[k], q = a.v[k == 2 ? 0 : k + 1];
                  if (((a.edges >> k) & 1) && open_overlap(min3(p, q), max3(p, q), blo, bhi))
                    ek |= 1u << k;
                }
              }
            }
            if (!__any_sync(full, ek != 0)) continue;
#pragma unroll 1
            for (int k = 0; k < 3; ++k) {
              bool hit = false;
              if ((ek >> k) & 1) {
                const F3 p = k == 0 ? a.v[0] : (k == 1 ? a.v[1] : a.v[2]);
                const F3 q = k == 0 ? a.v[1] : (k == 1 ? a.v[2] : a.v[0]);
                bool ex = false;
                c_tris += 1;
                hit = segtri_filtered(p, q, b.v[0], b.v[1], b.v[2], &ex);
              }
              const unsigned m = __ballot_sync(full, hit);
              if (!m) continue;
              if (hit) {
                c_hits += 1;
                const unsigned long long key = dir == 0 ? pair_key(a.mesh, b.mesh, self_join)
                                                        : pair_key(b.mesh, a.mesh, self_join);
                if (sink.mode == SINK_HASH) hash_insert(sink, key, st);
                else if (sink.mode == SINK_EMIT)
                  sink.keys[sink.off[item] + n_rec + __popc(m & lt)] = key;
              }
              n_rec += __popc(m);
            }
          }
        }
        __syncwarp();
        nl = 0;
        continue;
      }
      if (!pend) {
        // the next nodes' children, one to a lane, against the packet's box
        const int n = sp <= kDsStack ? min(sp, 32 / W) : 1;
        c_nodes += lane == 0 ? n : 0;
        bool in = false;
        if (lane < n * W) {
          const float4 *slot = reinterpret_cast<const float4 *>(
              tnodes + (int64_t)stk[sp - 1 - lane / W] * SW + 8 + 8 * (lane % W));
          const float4 q0 = __ldg(slot), q1 = __ldg(slot + 1);
          blo = mkf3(q0.x, q0.y, q0.z);
          bhi = mkf3(q0.w, q1.x, q1.y);
          word = __float_as_uint(q1.z);
          in = open_overlap(ulo, uhi, blo, bhi);  // an empty slot's box is inverted
        }
        pend = __ballot_sync(full, in);
        sp -= n;
        continue;
      }
      // one child against every lane's triangle
      const int src = __ffs(pend) - 1;
      pend &= pend - 1;
      const F3 clo = mkf3(__shfl_sync(full, blo.x, src), __shfl_sync(full, blo.y, src),
                          __shfl_sync(full, blo.z, src));
      const F3 chi = mkf3(__shfl_sync(full, bhi.x, src), __shfl_sync(full, bhi.y, src),
                          __shfl_sync(full, bhi.z, src));
      const uint32_t ch = __shfl_sync(full, word, src);
      bool meets = open_overlap(lo, hi, clo, chi);
      if (meets && fmaxf(chi.x - clo.x, fmaxf(chi.y - clo.y, chi.z - clo.z)) < side) {
        meets = false;
        const DsTri tri = ds_tri(srec, f0 + lane);  // again (cached): few lanes get here
#pragma unroll 1
        for (int k = 0; k < 3; ++k) {
          const F3 p = k == 0 ? tri.v[0] : (k == 1 ? tri.v[1] : tri.v[2]);
          const F3 q = k == 0 ? tri.v[1] : (k == 1 ? tri.v[2] : tri.v[0]);
          if ((tri.edges >> k) & 1) meets = meets || slab_hit(make_seg(p, q), clo, chi);
        }
      }
      const unsigned m = __ballot_sync(full, meets);
      if (!m) continue;
      if (ch & kLeafBit) {
        if (meets) {
          leaf[nl + __popc(m & lt)] = ch;
          leaf_lane[nl + __popc(m & lt)] = (uint8_t)lane;
        }
        nl += __popc(m);
      } else if (sp >= kCap) {
        if (lane == 0) atomicExch(st + DS_ERR, 1ull);
      } else {
        if (lane == 0) stk[sp] = ch;
        ++sp;
      }
      __syncwarp();
    }
    if (sink.mode == SINK_COUNT && lane == 0) sink.cnt[item] = n_rec;
  }
  const unsigned long long v[4] = {c_edges, c_nodes, c_tris, c_hits};
  flush_stats(st, v, 4);
}

// ---------------------------------------------------------------------------
// Alg. 1 in both directions at once for two datasets: the two BVHs walked
// together.  A queue entry is a pair of items, one of each dataset, whose
// boxes overlap (open): a node of either BVH, or a leaf.  A step replaces it
// by the overlapping pairs of the children of the larger node, or of both
// where they are of similar size; pairs of two leaves go to a list, and the
// edges of each against the other's triangles are tested from there.  Each
// part of one dataset thus meets only the parts of the other that lie around
// it, wherever the walk is, instead of being looked for from the root: 1,200
// nuclei x 60 vessels take 64,000 pairs, where packets of 32 triangles
// (k_ds_edges) took 2.0 M node visits and 1,100 us; 190 now.
//
// The walk is breadth first, a launch per level, the narrow ones in one block.
// What bounds it is each level's launch and chain of dependent reads.  Queues
// and list are of fixed size, 10,000 x 500 tissue meshes put 3.9 M entries in
// all through them; where they do not suffice (DS_FULL: dense data) the packets
// trace the edges after all, as they do for a self join, in which every
// triangle meets its own mesh's (16 x 16 spheres of 20,480 triangles crossing
// each other: 6.0 ms of tracing with the walk that is given up, 28 for an edge
// per thread).
// ---------------------------------------------------------------------------
constexpr uint32_t kDsOpen = 0x40000000u;   // the item's children are taken
constexpr uint32_t kDsIdx = 0x3FFFFFFFu;    // node, or node * W + k of a leaf
constexpr unsigned kDsQueue = 1u << 22;     // entries of a queue
constexpr unsigned kDsLeaves = 1u << 23;    // leaf pairs
constexpr int kDsLevelT = 512;              // threads of a block of the walk
constexpr unsigned kDsNarrow = 64;          // entries of a level that one block takes
constexpr int kDsLevels = 192;              // levels of the walk

__device__ __forceinline__ float ds_side(F3 lo, F3 hi) {
  return fmaxf(hi.x - lo.x, fmaxf(hi.y - lo.y, hi.z - lo.z));
}

// an entry of two items with these sizes: which of them the next step opens
__device__ __forceinline__ uint2 ds_entry(uint32_t a, float sa, uint32_t b, float sb) {
  const bool la = a & kLeafBit, lb = b & kLeafBit;
  return make_uint2(a | (!la && (lb || !(sb > 2.f * sa)) ? kDsOpen : 0u),
                    b | (!lb && (la || !(sa > 2.f * sb)) ? kDsOpen : 0u));
}

// child slot k of an open item, or the item's own box and word
template <int W>
__device__ __forceinline__ void ds_slot(const float *nodes, uint32_t item, int k, F3 &lo, F3 &hi,
                                        uint32_t &word, uint32_t &child) {
  const int SW = node_stride_words(W);
  const uint32_t ix = item & kDsIdx;
  const bool open = item & kDsOpen, leaf = item & kLeafBit;
  const float4 *p = reinterpret_cast<const float4 *>(
      nodes + (open ? (int64_t)ix * SW + 8 * (k + 1)
                    : leaf ? (int64_t)(ix / W) * SW + 8 * (ix % W + 1) : (int64_t)ix * SW));
  const float4 q0 = __ldg(p), q1 = __ldg(p + 1);
  lo = mkf3(q0.x, q0.y, q0.z);
  hi = mkf3(q0.w, q1.x, q1.y);
  word = __float_as_uint(q1.z);
  child = !open ? item : ((word & kLeafBit) ? (kLeafBit | (ix * W + k)) : word);
}

// A warp's part of a list: entries wait in shared memory until there are 32
// for one reservation.  A reservation per step, of about two entries, queued
// the wide levels up at the list's counter: 10,000 nuclei x 500 vessels, 3.9 M
// entries, took 2.07 ms of walk, leaves and rays; 1.34 now, the widest level
// 352 us and now 129 (1,200 x 60: the join 485 and now 471).
struct DsOut {
  uint2 *buf;  // 64 entries
  int n;       // of them waiting
  uint2 *list;
  unsigned *count, cap;
  __device__ __forceinline__ void put(bool on, unsigned m, uint2 e, unsigned long long *st,
                                      int lane) {
    if (on) buf[n + __popc(m & ((1u << lane) - 1u))] = e;
    n += __popc(m);
    if (n >= 32) flush(32, st, lane);
  }
  __device__ __forceinline__ void flush(int k, unsigned long long *st, int lane) {
    __syncwarp();
    unsigned at = 0;
    if (lane == 0) at = atomicAdd(count, (unsigned)k);
    at = __shfl_sync(0xffffffffu, at, 0) + lane;
    n -= k;
    if (lane < k) {
      if (at < cap) list[at] = buf[n + lane];
      else st[DS_FULL] = 1ull;
    }
    __syncwarp();
  }
};

// one entry's child pair r (of at most W x W) per lane: leaf pairs to the
// list, others to the next queue
template <int W>
__device__ __forceinline__ void ds_step(const float *nodesA, const float *nodesB, uint2 e, int r,
                                        bool on, DsOut &next_q, DsOut &leaf_q,
                                        unsigned long long *st, int lane) {
  const int nA = (e.x & kDsOpen) ? W : 1, nB = (e.y & kDsOpen) ? W : 1;
  on = on && r < nA * nB;
  bool ok = false;
  uint2 next = make_uint2(0u, 0u), pair = next;
  if (on) {
    F3 alo, ahi, blo, bhi;
    uint32_t wa, wb, ca, cb;
    ds_slot<W>(nodesA, e.x, r / nB, alo, ahi, wa, ca);
    ds_slot<W>(nodesB, e.y, r % nB, blo, bhi, wb, cb);
    ok = open_overlap(alo, ahi, blo, bhi);  // an empty slot's box is inverted
    next = ds_entry(ca, ds_side(alo, ahi), cb, ds_side(blo, bhi));
    pair = make_uint2(wa, wb);  // of two leaves: their descriptors
  }
  const bool leaf = ok && (next.x & next.y & kLeafBit);
  const unsigned m1 = __ballot_sync(0xffffffffu, ok && !leaf);
  const unsigned m2 = __ballot_sync(0xffffffffu, leaf);
  if (m1) next_q.put(ok && !leaf, m1, next, st, lane);
  if (m2) leaf_q.put(leaf, m2, pair, st, lane);
}

// A launch of the walk.  Launch i finds its level in at[i] and leaves the next
// one's in at[i + 1]; cnt[l] counts the entries of level l (queues alternate).
// A level of more than kDsNarrow entries is taken by the whole grid; narrower
// ones, the first and the last few, by one block, level after level until one
// is wide or none is left (the join took 628, 533 and 509 us with 1,024, 256
// and 64 entries as the line, 588 with the first levels in a kernel of their
// own and a launch for each further one).
// Launches that find nothing return at once; they are queued ahead
// (programmatic launches), as many as the trees have levels.
template <int W>
__global__ void __launch_bounds__(kDsLevelT) k_ds_level(const float *nodesA, const float *nodesB,
                                                        uint2 *q0, uint2 *q1, unsigned *cnt,
                                                        unsigned *at, int i, uint2 *leaves,
                                                        unsigned *n_leaves, unsigned queue_cap,
                                                        unsigned leaf_cap,
                                                        unsigned long long *st) {
  asm volatile("griddepcontrol.wait;" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  constexpr int G = W * W < 32 ? W * W : 32, PER = W * W / G;
  __shared__ uint2 s_buf[kDsLevelT / 32][2][64];
  const int lane = threadIdx.x & 31;
  uint2 *buf = s_buf[threadIdx.x >> 5][0];
  DsOut leaf_q{buf + 64, 0, leaves, n_leaves, leaf_cap};
  int lv = (int)__ldcg(at + i);
  unsigned n = __ldcg(cnt + lv);
  const bool wide = n > kDsNarrow;
  if (!wide && blockIdx.x > 0) return;
  unsigned long long visited = 0;
  if (i == 0) {  // the pair of roots
    if (threadIdx.x == 0) {
      const float4 *a = reinterpret_cast<const float4 *>(nodesA);
      const float4 *b = reinterpret_cast<const float4 *>(nodesB);
      const float4 a0 = a[0], a1 = a[1], b0 = b[0], b1 = b[1];
      q0[0] = ds_entry(0u, ds_side(mkf3(a0.x, a0.y, a0.z), mkf3(a0.w, a1.x, a1.y)), 0u,
                       ds_side(mkf3(b0.x, b0.y, b0.z), mkf3(b0.w, b1.x, b1.y)));
      __threadfence();
    }
    __syncthreads();
    n = 1;
  }
  const unsigned threads = wide ? gridDim.x * kDsLevelT : kDsLevelT;
  const unsigned t0 = (wide ? blockIdx.x * kDsLevelT : 0u) + threadIdx.x - lane;
  while (n > 0 && lv < kDsLevels - 1) {
    n = min(n, queue_cap);
    visited += 2ull * n;
    const uint2 *qin = lv & 1 ? q1 : q0;
    DsOut next_q{buf, 0, lv & 1 ? q0 : q1, cnt + lv + 1, queue_cap};
    for (unsigned e0 = t0 / G; e0 < n; e0 += threads / G) {
      const unsigned e = e0 + lane / G;
      const uint2 x = e < n ? __ldcg(qin + e) : make_uint2(0u, 0u);
#pragma unroll
      for (int j = 0; j < PER; ++j)
        ds_step<W>(nodesA, nodesB, x, lane % G + j * G, e < n, next_q, leaf_q, st, lane);
    }
    if (next_q.n > 0) next_q.flush(next_q.n, st, lane);
    ++lv;
    if (wide) break;
    __threadfence();
    __syncthreads();
    n = __ldcg(cnt + lv);
    if (n > kDsNarrow) break;
  }
  if (leaf_q.n > 0) leaf_q.flush(leaf_q.n, st, lane);
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    at[i + 1] = (unsigned)lv;
    if (visited) atomicAdd(st + DS_NODES, visited);
  }
}

// The listed leaf pairs: 2 L lanes to a pair, one source triangle of either
// side to a lane, its owned edges against the other leaf's triangles; the
// tests that box comparisons leave are listed and run 32 at a time.  Records
// are counted and placed per warp of the grid.
__global__ void __launch_bounds__(32 * kDsWarps) k_ds_leaf(DsSide A, DsSide B, const uint2 *leaves,
                                                           const unsigned *n_leaves,
                                                          unsigned leaf_cap, int lshift,
                                                           Sink sink, unsigned long long *st) {
  __shared__ unsigned s_list[kDsWarps][128 * 3];
  const unsigned full = 0xffffffffu;
  const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5, L = 1 << lshift;
  const unsigned lt = (1u << lane) - 1u;
  unsigned *list = s_list[wib];
  const int64_t warp = blockIdx.x * (int64_t)kDsWarps + wib, nw = gridDim.x * (int64_t)kDsWarps;
  const int64_t item = sink.base + warp;
  const unsigned n = min(*n_leaves, leaf_cap);
  unsigned long long c_tris = 0, c_hits = 0;
  int64_t n_rec = 0;
  int ntest = 0;
  // the last m listed: (source triangle, side | edge << 1, target triangle)
  auto run = [&](int m) {
    ntest -= m;
    bool hit = false;
    unsigned long long key = 0;
    if (lane < m) {
      const unsigned *e = list + 3 * (ntest + lane);
      const bool dir = e[1] & 1u;
      const int k = (int)(e[1] >> 1);
      const DsTri a = ds_tri(dir ? B.trirec : A.trirec, e[0]);
      const DsTri b = ds_tri(dir ? A.trirec : B.trirec, e[2]);
      const F3 p = k == 0 ? a.v[0] : (k == 1 ? a.v[1] : a.v[2]);
      const F3 q = k == 0 ? a.v[1] : (k == 1 ? a.v[2] : a.v[0]);
      bool ex = false;
      c_tris += 1;
      hit = segtri_filtered(p, q, b.v[0], b.v[1], b.v[2], &ex);
      key = dir ? pair_key(b.mesh, a.mesh, 0) : pair_key(a.mesh, b.mesh, 0);
    }
    const unsigned mh = __ballot_sync(full, hit);
    if (hit) {
      c_hits += 1;
      if (sink.mode == SINK_HASH) hash_insert(sink, key, st);
      else if (sink.mode == SINK_EMIT) sink.keys[sink.off[item] + n_rec + __popc(mh & lt)] = key;
    }
    n_rec += __popc(mh);
    __syncwarp();
  };
  const int per = 16 >> lshift;  // pairs of a step
  for (int64_t p0 = warp * per; p0 < n; p0 += nw * per) {
    const int64_t p = p0 + (lane >> (lshift + 1));
    const int si = lane & (L - 1);
    const unsigned dir = (lane >> lshift) & 1;
    const uint2 e = p < n ? leaves[p] : make_uint2(0u, 0u);
    const uint32_t sw = dir ? e.y : e.x, tw = dir ? e.x : e.y;
    const int64_t s0 = (sw >> 3) & 0x0FFFFFFFu, t0 = (tw >> 3) & 0x0FFFFFFFu;
    const int nt = (int)(tw & 7u) + 1;
    DsTri a;
    a.edges = 0;
    if (p < n && si <= (int)(sw & 7u)) a = ds_tri(dir ? B.trirec : A.trirec, s0 + si);
    for (int t = 0; t < L; ++t) {
      F3 blo = mkf3(0.f, 0.f, 0.f), bhi = blo;
      unsigned own = 0;
      if (a.edges && t < nt) {
        const DsTri b = ds_tri(dir ? A.trirec : B.trirec, t0 + t);
        blo = min3(b.v[0], min3(b.v[1], b.v[2]));
        bhi = max3(b.v[0], max3(b.v[1], b.v[2]));
        own = (unsigned)a.edges;
      }
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        const F3 u = a.v[k], v = a.v[k == 2 ? 0 : k + 1];
        const bool keep = ((own >> k) & 1u) && open_overlap(min3(u, v), max3(u, v), blo, bhi);
        const unsigned m = __ballot_sync(full, keep);
        if (keep) {
          unsigned *w = list + 3 * (ntest + __popc(m & lt));
          w[0] = (unsigned)(s0 + si);
          w[1] = dir | (unsigned)(k << 1);
          w[2] = (unsigned)(t0 + t);
        }
        ntest += __popc(m);
      }
      __syncwarp();
      while (ntest >= 32) run(32);
    }
  }
  if (ntest > 0) run(ntest);
  if (sink.mode == SINK_COUNT && lane == 0) sink.cnt[item] = n_rec;
  const unsigned long long v[2] = {c_tris, c_hits};
  flush_stats(st + DS_TRIS, v, 2);
}

// Containment rays (Sec. 3.3): a warp per object of Q, one ray from its first
// lexicographic vertex through T's BVH along the axis direction that leaves
// T's dataset box soonest (parity is the same in every direction for a closed
// mesh and a point off it).  Only objects whose closed box holds the vertex
// can contain it; up to kParList of them are tracked with a parity bit and an
// on-surface bit.  Q = B, T = A, then the reverse (a self join: Q = T = A
// once).  The children of up to 32 / W nodes are tested at a time, and a
// leaf's triangles one per lane; a thread per object walked alone (150 us for
// 1,260 objects, 21 now).
constexpr int kParLeaves = 64;  // listed leaves of a warp

template <int W>
__global__ void __launch_bounds__(32 * kDsWarps) k_ds_parity(DsSide A, DsSide B, int self_join,
                                                             Sink sink, Recheck rc,
                                                             bool first_pass, int lshift,
                                                             unsigned long long *st) {
  constexpr int kCap = 2 * kDsStack + 32;  // as in k_ds_edges
  __shared__ uint32_t s_stack[kDsWarps][kCap], s_leaf[kDsWarps][kParLeaves];
  __shared__ int s_obj[kDsWarps][kParList];
  __shared__ unsigned s_bits[kDsWarps][kParList];
  const unsigned full = 0xffffffffu;
  const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5, SW = node_stride_words(W);
  const unsigned lt = (1u << lane) - 1u;
  uint32_t *stk = s_stack[wib], *leaf = s_leaf[wib];
  int *lobj = s_obj[wib];
  unsigned *lbits = s_bits[wib];
  unsigned long long c_rays = 0, c_nodes = 0, c_tris = 0;
  const int64_t nB = self_join ? A.M : B.M, nA = self_join ? 0 : A.M;
  for (int64_t w = blockIdx.x * (int64_t)kDsWarps + wib; w < nB + nA;
       w += gridDim.x * (int64_t)kDsWarps) {
    const bool rev = w >= nB;  // an object of A against B
    const int64_t iq = rev ? w - nB : w;
    const float4 *qrec = (rev || self_join ? A.mrec : B.mrec) + 3 * iq;
    const float *tnodes = rev ? B.nodes : A.nodes, *taabb = rev ? B.aabb : A.aabb;
    const float4 *trec = rev ? B.trirec : A.trirec;
    int64_t n_rec = 0;
    const float4 q0 = qrec[0], q1 = qrec[1], q2 = qrec[2];
    const F3 vf = mkf3(q0.w, q1.w, q2.x);
    // T's dataset box: the root's own slot
    const float4 b0 = __ldg(reinterpret_cast<const float4 *>(tnodes));
    const float4 b1 = __ldg(reinterpret_cast<const float4 *>(tnodes) + 1);
    const F3 tlo = mkf3(b0.x, b0.y, b0.z), thi = mkf3(b0.w, b1.x, b1.y);
    if (vf.x >= tlo.x && vf.x <= thi.x && vf.y >= tlo.y && vf.y <= thi.y && vf.z >= tlo.z &&
        vf.z <= thi.z) {
      c_rays += lane == 0;
      const I3 v = toi(vf);
      int ax, dr;
      ray_axis_choice(vf, tlo, thi, ax, dr);
      int nl = 0, sp = 1, nlf = 0;
      bool over = false;
      if (lane == 0) stk[0] = 0u;
      __syncwarp();
      while (sp > 0 || nlf > 0) {
        if (sp == 0 || nlf + 32 > kParLeaves) {
          // the listed leaves' triangles, L lanes to a leaf
          for (int i0 = 0; i0 < nlf; i0 += 32 >> lshift) {
            const int i = i0 + (lane >> lshift), t = lane & ((1 << lshift) - 1);
            bool in = false;
            int ot = 0;
            unsigned bits = 0;
            if (i < nlf && t <= (int)(leaf[i] & 7u)) {
              const DsTri x = ds_tri(trec, ((leaf[i] >> 3) & 0x0FFFFFFFu) + t);
              ot = x.mesh;
              if (!(self_join && ot == (int)iq)) {
                // an object whose box does not hold the vertex cannot contain it
                const float *ob = taabb + 6 * (int64_t)ot;
                in = !(vf.x < ob[0] || vf.x > ob[3] || vf.y < ob[1] || vf.y > ob[4] ||
                       vf.z < ob[2] || vf.z > ob[5]);
              }
              if (in) {
                c_tris += 1;
                const I3 a = toi(x.v[0]), b = toi(x.v[1]), c = toi(x.v[2]);
                bits = (on_triangle(v, a, b, c) ? 2u : 0u) |
                       (ray_axis_hit(v, a, b, c, ax, dr) ? 1u : 0u);
              }
            }
            // (an object is tracked from the first triangle on, hit or not)
            for (unsigned m = __ballot_sync(full, in); m; m &= m - 1) {
              const int l = __ffs(m) - 1;
              const int o = __shfl_sync(full, ot, l);
              const unsigned bt = __shfl_sync(full, bits, l);
              int li = -1;
              for (int j0 = 0; j0 < nl; j0 += 32) {
                const unsigned f = __ballot_sync(full, j0 + lane < nl && lobj[j0 + lane] == o);
                if (f) li = j0 + __ffs(f) - 1;
              }
              if (li < 0) {
                if (nl == kParList) {
                  over = true;
                  continue;
                }
                li = nl++;
                if (lane == 0) {
                  lobj[li] = o;
                  lbits[li] = 0;
                }
              }
              if (lane == 0) lbits[li] = ((lbits[li] | bt) & 2u) | ((lbits[li] ^ bt) & 1u);
              __syncwarp();
            }
          }
          __syncwarp();
          nlf = 0;
          continue;
        }
        const int n = sp <= kDsStack ? min(sp, 32 / W) : 1;
        c_nodes += lane == 0 ? n : 0;
        bool in = false;
        uint32_t ch = 0;
        if (lane < n * W) {
          const float4 *slot = reinterpret_cast<const float4 *>(
              tnodes + (int64_t)stk[sp - 1 - lane / W] * SW + 8 + 8 * (lane % W));
          const float4 s0 = __ldg(slot), s1 = __ldg(slot + 1);
          ch = __float_as_uint(s1.z);
          Box bx;
          bx.lo = mkf3(s0.x, s0.y, s0.z);
          bx.hi = mkf3(s0.w, s1.x, s1.y);
          in = ch != kEmpty && ray_axis_box(vf, bx, ax, dr);
        }
        const bool lf = in && (ch & kLeafBit);
        const unsigned m1 = __ballot_sync(full, in && !lf), m2 = __ballot_sync(full, lf);
        sp -= n;
        if (sp + __popc(m1) > kCap) {
          if (lane == 0) atomicExch(st + DS_ERR, 1ull);
          break;
        }
        if (in && !lf) stk[sp + __popc(m1 & lt)] = ch;
        if (lf) leaf[nlf + __popc(m2 & lt)] = ch;
        sp += __popc(m1);
        nlf += __popc(m2);
        __syncwarp();
      }
      if (over && first_pass && lane == 0) {
        // every candidate of this object goes to the per-pair join
        const unsigned long long i = atomicAdd(st + DS_NOBJ, 1ull);
        if (i < rc.cap) rc.objs[i] = (int32_t)iq;
        else atomicExch(st + DS_ERR, 2ull);
      }
      for (int j0 = 0; j0 < nl; j0 += 32) {
        const int j = j0 + lane;
        const unsigned bits = j < nl ? lbits[j] : 0u;
        const int o = j < nl ? lobj[j] : 0;
        const int a = rev ? (int)iq : o, b = rev ? o : (int)iq;
        if ((bits & 2) && first_pass && !over) {
          // the vertex lies on this object's surface: the pair's own test
          const unsigned long long i = atomicAdd(st + DS_NREC, 1ull);
          if (i < rc.cap) rc.pairs[i] = make_int2(a, b);
          else atomicExch(st + DS_ERR, 2ull);
        }
        const bool rec = bits == 1u;
        const unsigned m = __ballot_sync(full, rec);
        if (rec) {
          const unsigned long long key = pair_key(a, b, self_join);
          if (sink.mode == SINK_HASH) hash_insert(sink, key, st);
          else if (sink.mode == SINK_EMIT)
            sink.keys[sink.off[sink.base + w] + n_rec + __popc(m & lt)] = key;
        }
        n_rec += __popc(m);
      }
      __syncwarp();
    }
    if (sink.mode == SINK_COUNT && lane == 0) sink.cnt[sink.base + w] = n_rec;
  }
  unsigned long long x[1] = {c_rays};
  flush_stats(st + DS_RAYS, x, 1);
  x[0] = c_nodes;
  flush_stats(st + DS_NODES, x, 1);
  x[0] = c_tris;
  flush_stats(st + DS_TRIS, x, 1);
}

// the occupied slots of a hashmap, in any order
__global__ void k_hash_extract(const unsigned long long *table, int64_t slots,
                               unsigned long long *keys, unsigned long long *n) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < slots;
       i += (int64_t)gridDim.x * blockDim.x) {
    const unsigned long long k = table[i];
    const bool has = k != kHashEmpty;
    const unsigned m = __ballot_sync(0xffffffffu, has);
    unsigned long long base = 0;
    if ((threadIdx.x & 31) == 0 && m) base = atomicAdd(n, (unsigned long long)__popc(m));
    base = __shfl_sync(0xffffffffu, base, 0);
    if (has) keys[base + __popc(m & ((1u << (threadIdx.x & 31)) - 1u))] = k;
  }
}

__global__ void k_keys_to_pairs(const unsigned long long *keys, const int64_t *n, int32_t *out) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < *n;
       i += (int64_t)gridDim.x * blockDim.x) {
    out[2 * i] = (int32_t)(keys[i] >> 32);
    out[2 * i + 1] = (int32_t)(keys[i] & 0xFFFFFFFFull);
  }
}

// the owning mesh of every triangle record of a dataset BVH
__global__ void k_set_owner(float4 *trirec, const int32_t *sorted, const int64_t *toff, int64_t M,
                            int64_t F) {
  for (int64_t s = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; s < F;
       s += (int64_t)gridDim.x * blockDim.x)
    trirec[3 * s + 2].w = __int_as_float((int)mesh_of(toff, M, sorted[s]));
}

// The dataset BVH of (W, L): the per-mesh build run on the dataset as a
// single mesh (borrowing its vertex, triangle and edge arrays), then the
// owning meshes written into the triangle records.
static pj_status dataset_bvh(Ctx *ctx, Dataset *ds, int W, int L, cudaStream_t s, Bvh **out) {
  auto it = ds->dbvhs.find({W, L});
  if (it != ds->dbvhs.end()) {
    *out = &it->second;
    return PJ_OK;
  }
  if (ds->F >= (1ll << 28))
    return fail(ctx, PJ_ERR_INVALID_ARG, "dataset too large for the dataset-level BVH (2^28 triangles)");
  Dataset flat;
  flat.M = 1;
  flat.V = ds->V;
  flat.F = ds->F;
  flat.d_xyz = ds->d_xyz;
  flat.d_tris = ds->d_tris;
  flat.d_emask = ds->d_emask;
  flat.h_toff = {0, ds->F};
  flat.h_voff = {0, ds->V};
  float box[6] = {3.4e38f, 3.4e38f, 3.4e38f, -3.4e38f, -3.4e38f, -3.4e38f};
  for (int64_t m = 0; m < ds->M; ++m)
    for (int d = 0; d < 3; ++d) {
      box[d] = std::min(box[d], ds->h_aabb[6 * m + d]);
      box[3 + d] = std::max(box[3 + d], ds->h_aabb[6 * m + 3 + d]);
    }
  int64_t toff[2] = {0, ds->F};
  TmpMem tmp(ctx, s);
  PJ_CK(tmp.get(&flat.d_toff, 2));
  PJ_CK(tmp.get(&flat.d_aabb, 6));
  PJ_CK(cudaMemcpyAsync(flat.d_toff, toff, sizeof(toff), cudaMemcpyHostToDevice, s));
  PJ_CK(cudaMemcpyAsync(flat.d_aabb, box, sizeof(box), cudaMemcpyHostToDevice, s));
  pj_status st = build_bvh(ctx, &flat, W, L, s);
  cudaStreamSynchronize(s);
  if (st != PJ_OK) return st;
  Bvh b = flat.bvhs[{W, L}];
  k_set_owner<<<blocks_for(ds->F, 256), 256, 0, s>>>(b.d_trirec, b.d_tri_order, ds->d_toff, ds->M,
                                                     ds->F);
  PJ_CK(cudaGetLastError());
  PJ_CK(cudaStreamSynchronize(s));
  ds->dbvhs[{W, L}] = b;
  *out = &ds->dbvhs[{W, L}];
  return PJ_OK;
}

static DsSide ds_side(Dataset *d, Bvh *b) {
  DsSide x;
  x.M = d->M;
  x.F = d->F;
  x.mrec = d->d_mrec;
  x.aabb = d->d_aabb;
  x.nodes = b->d_nodes;
  x.trirec = b->d_trirec;
  return x;
}

typedef void (*DsEdgeKernel)(DsSide, DsSide, int, Sink, unsigned long long *);
typedef void (*DsParKernel)(DsSide, DsSide, int, Sink, Recheck, bool, int, unsigned long long *);

pj_status run_dataset_join(Ctx *ctx, Dataset *A, Dataset *B, int self_join,
                           const pj_dsjoin_opts *o, pj_pairs *out, pj_dsjoin_stats *stats,
                           cudaStream_t s) {
  const int W = o->width ? o->width : 4, L = o->leaf_size ? o->leaf_size : 2;
  if (!(W == 2 || W == 4 || W == 8) || !(L == 1 || L == 2 || L == 4 || L == 8))
    return fail(ctx, PJ_ERR_INVALID_ARG, "width must be 2, 4 or 8 and leaf size 1, 2, 4 or 8");
  if (o->predicate != PJ_PRED_INTERSECTS && o->predicate != PJ_PRED_OVERLAP)
    return fail(ctx, PJ_ERR_INVALID_ARG, "the dataset-level join evaluates intersects or overlap");
  if (o->materialize < PJ_MAT_ESTIMATED || o->materialize > PJ_MAT_FIXED)
    return fail(ctx, PJ_ERR_INVALID_ARG, "unknown materialisation");
  const bool parity = o->predicate == PJ_PRED_INTERSECTS;
  pj_dsjoin_stats S;
  memset(&S, 0, sizeof(S));
  // events of its own: the estimate and the per-pair join record the
  // context's phase events
  struct Events {
    cudaEvent_t e[6] = {};
    ~Events() {
      for (auto x : e)
        if (x) cudaEventDestroy(x);
    }
  } evs;
  for (auto &x : evs.e) PJ_CK(cudaEventCreate(&x));
  cudaEvent_t *ev = evs.e;
  PJ_CK(cudaEventRecord(ev[0], s));
  // 1. the dataset BVHs (built once per W, L; not part of the timed join)
  Bvh *bA = nullptr, *bB = nullptr;
  pj_status st;
  if ((st = dataset_bvh(ctx, A, W, L, s, &bA)) != PJ_OK) return st;
  if ((st = dataset_bvh(ctx, B, W, L, s, &bB)) != PJ_OK) return st;
  if (1 + (W - 1) * std::max(bA->max_depth, bB->max_depth) > kDsStack)
    return fail(ctx, PJ_ERR_INTERNAL, "dataset BVH too deep for the traversal stack");
  const DsSide sA = ds_side(A, bA), sB = ds_side(B, bB);
  DsEdgeKernel ke = W == 2 ? k_ds_edges<2> : (W == 4 ? k_ds_edges<4> : k_ds_edges<8>);
  DsParKernel kp = W == 2 ? k_ds_parity<2> : (W == 4 ? k_ds_parity<4> : k_ds_parity<8>);
  PJ_CK(cudaEventRecord(ev[1], s));
  // 2. the estimate (sizes the hashmap)
  float ms_est = 0.f;
  int64_t slots = 0;
  if (o->materialize == PJ_MAT_ESTIMATED) {
    pj_estimate e;
    if ((st = run_estimate(ctx, A, B, o->grid, nullptr, &e, s)) != PJ_OK) return st;
    S.estimate = e.e_final;
    ms_est = e.ms;
    slots = (int64_t)std::min(e.slots, 1e12);
  } else if (o->materialize == PJ_MAT_FIXED) {
    slots = o->fixed_slots > 0 ? o->fixed_slots : (int64_t(1) << 26);
  }
  unsigned long long *d_st = (unsigned long long *)ws_get(ctx, "ds_stats", 8 * DS_NSTAT, &st);
  if (!d_st) return st;
  const unsigned long long rc_cap = 1 << 20;
  int2 *rc_pairs = (int2 *)ws_get(ctx, "ds_recheck", sizeof(int2) * rc_cap, &st);
  if (!rc_pairs) return st;
  int32_t *rc_objs = (int32_t *)ws_get(ctx, "ds_recheck_obj", sizeof(int32_t) * rc_cap, &st);
  if (!rc_objs) return st;
  Recheck rc{rc_pairs, rc_objs, rc_cap};
  const int lshift = L == 1 ? 0 : (L == 2 ? 1 : (L == 4 ? 2 : 3));
  // edges by the walk of both BVHs, or in packets (see k_ds_level)
  const int levels = bA->max_depth + bB->max_depth;
  bool dual = !self_join && levels + 2 < kDsLevels;
  const unsigned walk = (unsigned)std::max(0, ctx->limits.dataset_walk);
  const unsigned queue_cap = walk ? std::min(walk, kDsQueue) : kDsQueue;
  const unsigned leaf_cap = walk ? std::min(walk, kDsLeaves) : kDsLeaves;
  uint2 *q0 = nullptr, *q1 = nullptr, *leaves = nullptr;
  unsigned *lv_cnt = nullptr;  // entries per level, the leaf pairs, the launches' levels
  if (dual) {
    q0 = (uint2 *)ws_get(ctx, "ds_queue0", sizeof(uint2) * (size_t)kDsQueue, &st);
    if (q0) q1 = (uint2 *)ws_get(ctx, "ds_queue1", sizeof(uint2) * (size_t)kDsQueue, &st);
    if (q1) leaves = (uint2 *)ws_get(ctx, "ds_leaves", sizeof(uint2) * (size_t)kDsLeaves, &st);
    if (leaves) lv_cnt = (unsigned *)ws_get(ctx, "ds_levels", 4 * (2 * kDsLevels + 1), &st);
    if (!lv_cnt) {  // no room for the walk's 168 MB: the packets need none
      dual = false;
      clear_err(ctx);
    }
  }
  // one tracing pass over every item: the warps that test the leaf pairs, or
  // A's packets of triangles and B's; B's objects, A's objects (count / emit
  // arrays are indexed in this order)
  // (its registers let 6 blocks of k_ds_leaf onto an SM; 8 an SM left a third
  // of a round to the end: 1.33 ms of tracing against 1.21 on 10,000 x 500;
  // 64 registers for 8 blocks: 1.26)
  const int leaf_grid = ctx->num_sms * 6;
  auto packets = [](int64_t F) { return (F + kDsPacket - 1) / kDsPacket; };
  const int64_t nPack = packets(A->F) + (self_join ? 0 : packets(B->F));
  const int64_t nObj = !parity ? 0 : (self_join ? A->M : A->M + B->M);
  auto edge_items = [&]() { return dual ? (int64_t)leaf_grid * kDsWarps : nPack; };
  auto trace = [&](Sink k, bool first_pass) -> pj_status {
    k.base = 0;
    if (dual) {
      unsigned *n_leaves = lv_cnt + kDsLevels;
      if (first_pass) {
        const auto kl = W == 2 ? k_ds_level<2> : (W == 4 ? k_ds_level<4> : k_ds_level<8>);
        PJ_CK(cudaMemsetAsync(lv_cnt, 0, 4 * (2 * kDsLevels + 1), s));
        cudaLaunchAttribute attr{};
        attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
        attr.val.programmaticStreamSerializationAllowed = 1;
        cudaLaunchConfig_t cfg{};
        cfg.gridDim = dim3(ctx->num_sms * 4);
        cfg.blockDim = dim3(kDsLevelT);
        cfg.stream = s;
        cfg.attrs = &attr;
        for (int l = 0; l < levels; ++l) {
          cfg.numAttrs = l > 0;
          PJ_CK(cudaLaunchKernelEx(&cfg, kl, sA.nodes, sB.nodes, q0, q1, lv_cnt,
                                   lv_cnt + kDsLevels + 1, l, leaves, n_leaves, queue_cap,
                                   leaf_cap, d_st));
        }
        ctx->launches += levels;
      }
      k_ds_leaf<<<leaf_grid, 32 * kDsWarps, 0, s>>>(sA, sB, leaves, n_leaves, leaf_cap, lshift, k,
                                                    d_st);
    } else {
      // enough warps to spread the costly packets, few enough that their
      // counters' atomics do not queue up
      const int egrid = (int)std::min<int64_t>((nPack + kDsWarps - 1) / kDsWarps,
                                               ctx->num_sms * 32);
      ke<<<egrid, 32 * kDsWarps, 0, s>>>(sA, self_join ? sA : sB, self_join, k, d_st);
    }
    if (parity) {
      k.base = edge_items();
      kp<<<(int)std::min<int64_t>((nObj + kDsWarps - 1) / kDsWarps, ctx->num_sms * 32),
           32 * kDsWarps, 0, s>>>(sA, self_join ? sA : sB, self_join, k, rc, first_pass, lshift,
                                  d_st);
    }
    ctx->launches += parity ? 2 : 1;
    PJ_CK(cudaGetLastError());
    return PJ_OK;
  };
  unsigned long long h_st[DS_NSTAT];
  unsigned long long *keys = nullptr;
  int64_t n_keys = 0;
  float ms_trace = 0.f;
  if (o->materialize != PJ_MAT_TWO_PASS) {
    // single pass into a hashmap; on overflow twice the slots and again
    // slots rounded up to a power of two (at least 16 for a fixed size,
    // 1,024 for an estimate)
    int64_t cap = o->materialize == PJ_MAT_FIXED ? 16 : 1024;
    while (cap < slots) cap *= 2;
    for (;;) {
      unsigned long long *table =
          (unsigned long long *)ws_get(ctx, "ds_hash", 8 * (size_t)cap, &st);
      if (!table) return st;
      PJ_CK(cudaMemsetAsync(table, 0xff, 8 * (size_t)cap, s));
      PJ_CK(cudaMemsetAsync(d_st, 0, 8 * DS_NSTAT, s));
      PJ_CK(cudaEventRecord(ev[2], s));
      Sink k{SINK_HASH, table, (unsigned long long)(cap - 1), nullptr, nullptr, nullptr, 0};
      if ((st = trace(k, true)) != PJ_OK) return st;
      PJ_CK(cudaEventRecord(ev[4], s));
      PJ_CK(cudaMemcpyAsync(h_st, d_st, sizeof(h_st), cudaMemcpyDeviceToHost, s));
      PJ_CK(cudaStreamSynchronize(s));
      cudaEventElapsedTime(&ms_trace, ev[2], ev[4]);
      if (dual && h_st[DS_FULL]) {
        dual = false;  // too dense for the walk's queue or list
        continue;
      }
      if (!h_st[DS_OVERFLOW]) {
        keys = (unsigned long long *)ws_get(ctx, "ds_keys", 8 * (size_t)cap + 8, &st);
        if (!keys) return st;
        unsigned long long *d_n = keys + cap;
        PJ_CK(cudaMemsetAsync(d_n, 0, 8, s));
        k_hash_extract<<<(int)std::min<int64_t>(blocks_for(cap, 256), ctx->num_sms * 16), 256, 0,
                         s>>>(table, cap, keys, d_n);
        ++ctx->launches;
        unsigned long long n = 0;
        PJ_CK(cudaMemcpyAsync(&n, d_n, 8, cudaMemcpyDeviceToHost, s));
        PJ_CK(cudaStreamSynchronize(s));
        n_keys = (int64_t)n;
        S.slots = cap;
        break;
      }
      if (++S.relaunches > 12) return fail(ctx, PJ_ERR_NO_MEMORY, "hashmap overflow after 12 doublings");
      cap *= 2;
    }
  } else {
    // count, prefix sum, emit
    int64_t *off = nullptr;
    int64_t items = 0;
    for (;;) {
      items = edge_items() + nObj;
      int64_t *cnt = (int64_t *)ws_get(ctx, "ds_count", 8 * (size_t)(items + 1), &st);
      if (!cnt) return st;
      off = (int64_t *)ws_get(ctx, "ds_off", 8 * (size_t)(items + 1), &st);
      if (!off) return st;
      PJ_CK(cudaMemsetAsync(d_st, 0, 8 * DS_NSTAT, s));
      PJ_CK(cudaMemsetAsync(cnt, 0, 8 * (size_t)(items + 1), s));
      PJ_CK(cudaEventRecord(ev[2], s));
      Sink kc{SINK_COUNT, nullptr, 0, cnt, nullptr, nullptr, 0};
      if ((st = trace(kc, true)) != PJ_OK) return st;
      size_t tb = 0;
      PJ_CK(cub::DeviceScan::ExclusiveSum(nullptr, tb, cnt, off, (int)(items + 1), s));
      void *tmp = ws_get(ctx, "ds_scan_tmp", tb, &st);
      if (!tmp) return st;
      PJ_CK(cub::DeviceScan::ExclusiveSum(tmp, tb, cnt, off, (int)(items + 1), s));
      if (!dual) break;
      PJ_CK(cudaMemcpyAsync(h_st, d_st, sizeof(h_st), cudaMemcpyDeviceToHost, s));
      PJ_CK(cudaStreamSynchronize(s));
      if (!h_st[DS_FULL]) break;
      dual = false;  // too dense for the walk's queue or list
    }
    int64_t total = 0;
    PJ_CK(cudaMemcpyAsync(&total, off + items, 8, cudaMemcpyDeviceToHost, s));
    PJ_CK(cudaStreamSynchronize(s));
    keys = (unsigned long long *)ws_get(ctx, "ds_keys", 8 * (size_t)std::max<int64_t>(total, 1) + 8, &st);
    if (!keys) return st;
    Sink ke2{SINK_EMIT, nullptr, 0, nullptr, off, keys, 0};
    // the stats count both passes: keep the first pass's
    PJ_CK(cudaMemcpyAsync(h_st, d_st, sizeof(h_st), cudaMemcpyDeviceToHost, s));
    if ((st = trace(ke2, false)) != PJ_OK) return st;
    PJ_CK(cudaEventRecord(ev[4], s));
    PJ_CK(cudaStreamSynchronize(s));
    unsigned long long h2[DS_NSTAT];
    PJ_CK(cudaMemcpyAsync(h2, d_st, sizeof(h2), cudaMemcpyDeviceToHost, s));
    PJ_CK(cudaStreamSynchronize(s));
    h_st[DS_ERR] |= h2[DS_ERR];
    cudaEventElapsedTime(&ms_trace, ev[2], ev[4]);
    n_keys = total;
    S.slots = total;
    ctx->launches += 1;
  }
  if (h_st[DS_ERR] == 1) return fail(ctx, PJ_ERR_INTERNAL, "dataset BVH traversal stack exceeded");
  if (h_st[DS_ERR] == 2) return fail(ctx, PJ_ERR_NO_MEMORY, "too many parity rays to recheck");
  S.edges = A->E + (self_join ? 0 : B->E);  // every owned edge
  S.node_visits = (int64_t)h_st[DS_NODES];
  S.tri_tests = (int64_t)h_st[DS_TRIS];
  S.hits = (int64_t)h_st[DS_HITS];
  S.parity_rays = (int64_t)h_st[DS_RAYS];
  // 3. pairs the parity rays left to the per-pair join: candidates of the
  // overflowing objects and the listed pairs, refined by run_join
  std::vector<int32_t> rchk;
  {
    const int64_t np = (int64_t)std::min<unsigned long long>(h_st[DS_NREC], rc_cap);
    const int64_t no = (int64_t)std::min<unsigned long long>(h_st[DS_NOBJ], rc_cap);
    std::vector<int2> hp(np);
    std::vector<int32_t> ho(no);
    if (np) PJ_CK(cudaMemcpyAsync(hp.data(), rc_pairs, sizeof(int2) * np, cudaMemcpyDeviceToHost, s));
    if (no) PJ_CK(cudaMemcpyAsync(ho.data(), rc_objs, sizeof(int32_t) * no, cudaMemcpyDeviceToHost, s));
    PJ_CK(cudaStreamSynchronize(s));
    for (auto &p : hp) {
      int a = p.x, b = p.y;
      if (self_join && a > b) std::swap(a, b);
      rchk.push_back(a);
      rchk.push_back(b);
    }
    // an overflowing object: its bounding-box candidates on the other side.
    // (Object ids from both directions share this list; the kernels of one
    // direction write ids of their own casting side, told apart here by
    // trying both sides' boxes, which only adds candidates.)
    auto meet = [](const float *x, const float *y) {
      return x[0] <= y[3] && y[0] <= x[3] && x[1] <= y[4] && y[1] <= x[4] && x[2] <= y[5] &&
             y[2] <= x[5];
    };
    for (int32_t q : ho) {
      if (q < B->M)
        for (int64_t i = 0; i < A->M; ++i)
          if (meet(&A->h_aabb[6 * i], &B->h_aabb[6 * (int64_t)q])) {
            int a = (int)i, b = q;
            if (self_join && a > b) std::swap(a, b);
            if (!(self_join && a == b)) {
              rchk.push_back(a);
              rchk.push_back(b);
            }
          }
      if (!self_join && q < A->M)
        for (int64_t j = 0; j < B->M; ++j)
          if (meet(&A->h_aabb[6 * (int64_t)q], &B->h_aabb[6 * j])) {
            rchk.push_back(q);
            rchk.push_back((int)j);
          }
    }
  }
  std::vector<unsigned long long> extra;
  S.recheck_pairs = (int64_t)rchk.size() / 2;
  if (!rchk.empty()) {
    pj_join_opts po{};
    po.width = W;
    po.leaf_size = L;
    po.out_host = 1;
    // the per-pair join needs both datasets' per-mesh BVH of this shape
    for (Dataset *D : {A, B})
      if (D->bvhs.find({W, L}) == D->bvhs.end()) {
        if ((st = build_bvh(ctx, D, W, L, s)) != PJ_OK) return st;
      }
    pj_pairs r;
    memset(&r, 0, sizeof(r));
    if ((st = run_join(ctx, A, B, rchk.data(), nullptr, (int64_t)rchk.size() / 2, 0, 0, &po, s,
                       &r)) != PJ_OK)
      return st;
    for (int64_t k = 0; k < r.count; ++k)
      extra.push_back(((unsigned long long)(unsigned)r.pairs[2 * k] << 32) |
                      (unsigned)r.pairs[2 * k + 1]);
    pairs_release(ctx, &r);
  }
  // 4. sort and unique (with the rechecked pairs), then (idA, idB)
  PJ_CK(cudaEventRecord(ev[5], s));
  const int64_t n_all = n_keys + (int64_t)extra.size();
  unsigned long long *k2 = (unsigned long long *)ws_get(ctx, "ds_keys2", 8 * (size_t)std::max<int64_t>(n_all, 1), &st);
  if (!k2) return st;
  unsigned long long *k3 = (unsigned long long *)ws_get(ctx, "ds_keys3", 8 * (size_t)std::max<int64_t>(n_all, 1), &st);
  if (!k3) return st;
  if (!extra.empty()) {
    // the traced keys and the rechecked pairs in one buffer
    unsigned long long *k1 = (unsigned long long *)ws_get(ctx, "ds_keys1", 8 * (size_t)n_all, &st);
    if (!k1) return st;
    if (n_keys > 0)
      PJ_CK(cudaMemcpyAsync(k1, keys, 8 * (size_t)n_keys, cudaMemcpyDeviceToDevice, s));
    PJ_CK(cudaMemcpyAsync(k1 + n_keys, extra.data(), 8 * extra.size(), cudaMemcpyHostToDevice, s));
    PJ_CK(cudaStreamSynchronize(s));  // extra is a host vector
    keys = k1;
  }
  int64_t *d_nu = (int64_t *)ws_get(ctx, "ds_nunique", 8, &st);
  if (!d_nu) return st;
  int64_t K = 0;
  if (n_all > 0) {
    size_t tb = 0, tb2 = 0;
    PJ_CK(cub::DeviceRadixSort::SortKeys(nullptr, tb, keys, k2, (int)n_all, 0, 64, s));
    PJ_CK(cub::DeviceSelect::Unique(nullptr, tb2, k2, k3, d_nu, (int)n_all, s));
    void *tmp = ws_get(ctx, "ds_sort_tmp", std::max(tb, tb2), &st);
    if (!tmp) return st;
    PJ_CK(cub::DeviceRadixSort::SortKeys(tmp, tb, keys, k2, (int)n_all, 0, 64, s));
    PJ_CK(cub::DeviceSelect::Unique(tmp, tb2, k2, k3, d_nu, (int)n_all, s));
    PJ_CK(cudaMemcpyAsync(&K, d_nu, 8, cudaMemcpyDeviceToHost, s));
    PJ_CK(cudaStreamSynchronize(s));
  }
  cudaError_t pe;
  int32_t *d_out = (int32_t *)pool_get(ctx, 8 * (size_t)std::max<int64_t>(K, 1), &pe);
  PJ_CK(pe);
  if (K > 0) {
    k_keys_to_pairs<<<(int)std::min<int64_t>(blocks_for(K, 256), ctx->num_sms * 8), 256, 0, s>>>(
        k3, d_nu, d_out);
    ++ctx->launches;
  }
  PJ_CK(cudaEventRecord(ev[3], s));
  PJ_CK(cudaStreamSynchronize(s));
  memset(out, 0, sizeof(*out));
  out->count = K;
  out->n_candidates = 0;
  if (o->out_host) {
    PJ_CK(cudaMallocHost((void **)&out->pairs, 8 * (size_t)std::max<int64_t>(K, 1)));
    if (K > 0) PJ_CK(cudaMemcpy(out->pairs, d_out, 8 * (size_t)K, cudaMemcpyDeviceToHost));
    pool_put(ctx, d_out);
    out->on_device = 0;
  } else {
    out->pairs = d_out;
    out->on_device = 1;
  }
  float ms_all = 0.f, ms_mat = 0.f;
  cudaEventElapsedTime(&ms_all, ev[1], ev[3]);
  cudaEventElapsedTime(&ms_mat, ev[5], ev[3]);
  out->device_ms = ms_all;
  S.ms_total = ms_all;
  S.ms_estimate = ms_est;
  S.ms_trace = ms_trace;
  S.ms_materialize = ms_mat;
  if (stats) *stats = S;
  return PJ_OK;
}

}  // namespace pj
