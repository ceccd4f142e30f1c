// Per-mesh BVH build on the GPU: an LBVH (Karras, "Maximizing Parallelism in
// the Construction of BVHs, Octrees, and k-d Trees", HPG 2012) over 30-bit
// Morton codes of triangle centroids normalised to the mesh box, exact
// integer-valued boxes by a bottom-up refit, then a top-down collapse of the
// binary tree into W-wide nodes whose leaves hold at most L triangles (a leaf
// is a subtree, so its triangles are contiguous in the sorted order).
//
// The paper builds one OptiX acceleration structure per dataset (Sec. 4.1);
// here each mesh gets its own tree because the refinement works per
// candidate pair.  Build time is not part of the query time (Sec. 4.2
// "Measurement").
#include <cub/cub.cuh>

#include <algorithm>
#include <vector>

#include "pj_internal.cuh"

namespace pj {

__device__ __forceinline__ uint32_t spread10(uint32_t v) {
  v &= 0x3ffu;
  v = (v | (v << 16)) & 0x030000FFu;
  v = (v | (v << 8)) & 0x0300F00Fu;
  v = (v | (v << 4)) & 0x030C30C3u;
  v = (v | (v << 2)) & 0x09249249u;
  return v;
}

// Morton keys, kWarpSpan triangles per warp.  The grid cell of a centroid is
// floor(1024 (c - lo) / ext) in integers (sums of three coordinates, below
// 2^20): the FP64 quotients this replaces gave the same cells and took most
// of 1,104 us for 11 M triangles (90 now), with a binary search of
// the mesh per triangle.
__global__ void __launch_bounds__(256) k_morton(const float *xyz, const int32_t *tris, int64_t F,
                                                const int64_t *toff, int64_t M,
                                                const float *aabb, uint64_t *keys,
                                                int32_t *ids) {
  const int lane = threadIdx.x & 31;
  const int64_t w = blockIdx.x * (int64_t)8 + (threadIdx.x >> 5);
  const int64_t t0 = w * kWarpSpan, t1 = min(t0 + kWarpSpan, F);
  if (t0 >= t1) return;
  int64_t m = warp_mesh_of(toff, M, t0, lane), end = toff[m + 1];
  for (int64_t t = t0 + lane; t < t1; t += 32) {
    while (end <= t) end = toff[++m + 1];
    const int64_t a = tris[3 * t], b = tris[3 * t + 1], c = tris[3 * t + 2];
    uint32_t q[3];
#pragma unroll
    for (int d = 0; d < 3; ++d) {
      const int sum = (int)xyz[3 * a + d] + (int)xyz[3 * b + d] + (int)xyz[3 * c + d];
      const int lo = 3 * (int)aabb[6 * m + d];
      const unsigned ext = (unsigned)(3 * (int)aabb[6 * m + 3 + d] - lo);
      q[d] = ext > 0 ? min(((unsigned)(sum - lo) << 10) / ext, 1023u) : 0u;
    }
    uint32_t code = (spread10(q[0]) << 2) | (spread10(q[1]) << 1) | spread10(q[2]);
    keys[t] = ((uint64_t)m << 30) | code;
    ids[t] = (int32_t)t;
  }
}

// binary radix tree node arrays (per dataset, internal nodes of mesh m at
// [ioff[m], ioff[m] + n_m - 1) with ioff[m] = toff[m] - m)
struct BinTree {
  int2 *child;             // >= 0 local internal index, < 0: leaf -(pos + 1)
  int2 *range;             // first and last local sorted position
  int32_t *par_int;        // parent (global internal) of internal node, -1 root
  int32_t *par_leaf;       // parent (global internal) of sorted leaf, -1 none
  float2 *box;             // 3 per internal node: (lo x, lo y) (lo z, hi x) (hi y, hi z)
  float2 *leaf_box;        // 3 per sorted leaf
  int32_t *visits;
};

struct Box6 {
  float2 a, b, c;
};
__device__ __forceinline__ Box6 ld_box(const float2 *p) {
  Box6 r;
  r.a = __ldcg(p);
  r.b = __ldcg(p + 1);
  r.c = __ldcg(p + 2);
  return r;
}
__device__ __forceinline__ void st_box(float2 *p, const Box6 &r) {
  __stcg(p, r.a);
  __stcg(p + 1, r.b);
  __stcg(p + 2, r.c);
}
__device__ __forceinline__ Box6 join(const Box6 &x, const Box6 &y) {
  Box6 r;
  r.a = make_float2(fminf(x.a.x, y.a.x), fminf(x.a.y, y.a.y));
  r.b = make_float2(fminf(x.b.x, y.b.x), fmaxf(x.b.y, y.b.y));
  r.c = make_float2(fmaxf(x.c.x, y.c.x), fmaxf(x.c.y, y.c.y));
  return r;
}

__device__ __forceinline__ int delta(const uint64_t *keys, int64_t base, int n,
                                     int i, int j) {
  if (j < 0 || j >= n) return -1;
  uint32_t ki = (uint32_t)(keys[base + i] & 0x3FFFFFFFu);
  uint32_t kj = (uint32_t)(keys[base + j] & 0x3FFFFFFFu);
  if (ki != kj) return __clz(ki ^ kj);
  return 32 + __clz((uint32_t)i ^ (uint32_t)j);
}

// the tree's nodes, one per thread (a chain of dependent key reads each: a
// span of 256 per warp took 54 us for 0.6 M triangles); *big counts those
// with more than L triangles
__global__ void __launch_bounds__(256) k_karras(const uint64_t *keys, const int64_t *toff,
                                                const int64_t *ioff, int64_t M, int64_t n_int,
                                                BinTree T, int L, unsigned long long *big) {
  __shared__ unsigned s_big;
  if (threadIdx.x == 0) s_big = 0;
  __syncthreads();
  const int lane = threadIdx.x & 31;
  const int64_t g0 = blockIdx.x * (int64_t)blockDim.x + threadIdx.x - lane, g = g0 + lane;
  unsigned nbig = 0;
  int64_t m = g0 < n_int ? warp_mesh_of(ioff, M, g0, lane) : 0;
  if (g < n_int) {
    while (ioff[m + 1] <= g) ++m;
    int64_t base = toff[m];
    int n = (int)(toff[m + 1] - toff[m]);
    int i = (int)(g - ioff[m]);
    int d = (delta(keys, base, n, i, i + 1) - delta(keys, base, n, i, i - 1)) >= 0 ? 1 : -1;
    int dmin = delta(keys, base, n, i, i - d);
    int lmax = 2;
    while (delta(keys, base, n, i, i + lmax * d) > dmin) lmax <<= 1;
    int l = 0;
    for (int t = lmax >> 1; t >= 1; t >>= 1)
      if (delta(keys, base, n, i, i + (l + t) * d) > dmin) l += t;
    int j = i + l * d;
    int dnode = delta(keys, base, n, i, j);
    int s = 0;
    for (int div = 2;; div <<= 1) {
      int t = (l + div - 1) / div;
      if (delta(keys, base, n, i, i + (s + t) * d) > dnode) s += t;
      if (t <= 1) break;
    }
    int gamma = i + s * d + min(d, 0);
    int lo = min(i, j), hi = max(i, j);
    int64_t ib = ioff[m];
    int32_t left, right;
    if (lo == gamma) {
      left = -(gamma + 1);
      T.par_leaf[base + gamma] = (int32_t)g;
    } else {
      left = gamma;
      T.par_int[ib + gamma] = (int32_t)g;
    }
    if (hi == gamma + 1) {
      right = -(gamma + 2);
      T.par_leaf[base + gamma + 1] = (int32_t)g;
    } else {
      right = gamma + 1;
      T.par_int[ib + gamma + 1] = (int32_t)g;
    }
    T.child[g] = make_int2(left, right);
    T.range[g] = make_int2(lo, hi);
    if (i == 0) T.par_int[g] = -1;
    nbig += hi - lo + 1 > L;
  }
  nbig = __reduce_add_sync(0xffffffffu, nbig);
  if (lane == 0 && nbig) atomicAdd(&s_big, nbig);
  __syncthreads();
  if (threadIdx.x == 0 && s_big) atomicAdd(big, (unsigned long long)s_big);
}

// the sorted triangles: their boxes and their records (the key holds the mesh)
__global__ void __launch_bounds__(256) k_leaves(const float *xyz, const int32_t *tris,
                                                const int32_t *sorted, const uint64_t *keys,
                                                const uint8_t *emask, const int64_t *toff,
                                                int64_t F, float2 *leaf_box, float4 *rec) {
  for (int64_t s = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; s < F;
       s += (int64_t)gridDim.x * blockDim.x) {
    const int64_t t = sorted[s], m = (int64_t)(keys[s] >> 30);
    const float *a = xyz + 3 * (int64_t)tris[3 * t], *b = xyz + 3 * (int64_t)tris[3 * t + 1],
                *c = xyz + 3 * (int64_t)tris[3 * t + 2];
    const float ax = a[0], ay = a[1], az = a[2], bx = b[0], by = b[1], bz = b[2];
    const float cx = c[0], cy = c[1], cz = c[2];
    rec[3 * s] = make_float4(ax, ay, az, bx);
    rec[3 * s + 1] = make_float4(by, bz, cx, cy);
    rec[3 * s + 2] = make_float4(cz, __int_as_float((int)emask[t]),
                                 __int_as_float((int)(t - toff[m])), 0.f);
    leaf_box[3 * s] = make_float2(fminf(ax, fminf(bx, cx)), fminf(ay, fminf(by, cy)));
    leaf_box[3 * s + 1] = make_float2(fminf(az, fminf(bz, cz)), fmaxf(ax, fmaxf(bx, cx)));
    leaf_box[3 * s + 2] = make_float2(fmaxf(ay, fmaxf(by, cy)), fmaxf(az, fmaxf(bz, cz)));
  }
}

// Bottom-up union of child boxes; the second thread to reach a node computes
// it (no waiting: the first one stops).  A block takes kRefitT consecutive
// leaves.  Nodes whose triangles all lie among them -- all but a few per
// block -- are met and united in shared memory; only above them do threads
// meet through global memory.  A node's
// number is one end of its range, so it is also its place in the block.  The
// version without blocks, with a binary search of the mesh at every step,
// took 1,910 us for 11 M triangles, 661 now.
constexpr int kRefitT = 256;

__global__ void __launch_bounds__(kRefitT) k_refit(const uint64_t *keys, const int64_t *toff,
                                                   const int64_t *ioff, int64_t F, BinTree T) {
  __shared__ Box6 s_leaf[kRefitT], s_node[kRefitT];
  __shared__ int s_visit[kRefitT];
  const int tid = threadIdx.x;
  const int64_t b0 = blockIdx.x * (int64_t)kRefitT, s = b0 + tid;
  const int64_t b1 = min(b0 + kRefitT, F);
  s_visit[tid] = 0;
  if (s < F) s_leaf[tid] = ld_box(T.leaf_box + 3 * s);
  __syncthreads();
  if (s >= F) return;
  const int64_t m = (int64_t)(keys[s] >> 30), base = toff[m], ib = ioff[m];
  const int shift = (int)(base - b0);  // local position + shift: place in the block
  int32_t g = T.par_leaf[s];
  while (g >= 0) {
    const int2 rg = T.range[g];
    if (base + rg.x < b0 || base + rg.y >= b1) break;
    const int at = (int)(g - ib) + shift;
    __threadfence_block();
    if (atomicAdd(&s_visit[at], 1) == 0) return;
    __threadfence_block();
    const int2 ch = T.child[g];
    const volatile float2 *p0 = reinterpret_cast<volatile float2 *>(
        ch.x < 0 ? &s_leaf[-ch.x - 1 + shift] : &s_node[ch.x + shift]);
    const volatile float2 *p1 = reinterpret_cast<volatile float2 *>(
        ch.y < 0 ? &s_leaf[-ch.y - 1 + shift] : &s_node[ch.y + shift]);
    Box6 x, y;
    x.a = make_float2(p0[0].x, p0[0].y);
    x.b = make_float2(p0[1].x, p0[1].y);
    x.c = make_float2(p0[2].x, p0[2].y);
    y.a = make_float2(p1[0].x, p1[0].y);
    y.b = make_float2(p1[1].x, p1[1].y);
    y.c = make_float2(p1[2].x, p1[2].y);
    const Box6 r = join(x, y);
    s_node[at] = r;
    st_box(T.box + 3 * (int64_t)g, r);
    g = T.par_int[g];
  }
  while (g >= 0) {
    // releases this thread's box, acquires the sibling's
    int seen;
    asm volatile("atom.add.acq_rel.gpu.global.s32 %0, [%1], 1;"
                 : "=r"(seen) : "l"(T.visits + g) : "memory");
    if (seen == 0) break;
    const int2 ch = T.child[g];
    const Box6 x = ld_box(ch.x < 0 ? T.leaf_box + 3 * (base + (-ch.x - 1)) : T.box + 3 * (ib + ch.x));
    const Box6 y = ld_box(ch.y < 0 ? T.leaf_box + 3 * (base + (-ch.y - 1)) : T.box + 3 * (ib + ch.y));
    st_box(T.box + 3 * (int64_t)g, join(x, y));
    g = T.par_int[g];
  }
}

// Wide node `id`, to be filled from binary node `bin`: >= 0 local internal,
// < 0 leaf -(pos + 1).  The entries of one level have consecutive ids.
struct QEntry {
  int32_t bin;
  int32_t mesh;
};

// One level of the top-down collapse: the entries [start[lv], start[lv] +
// cnt[lv]) become wide nodes; their inner children get the ids after the
// level's last, a warp's at a time, and are counted in cnt[lv + 1].  The
// levels follow each other on the device, several to a host round trip (an
// empty level returns at once): a host wait and a queue per level, and an
// atomic per child and entry on single words, took 1,939 us for 11 M
// triangles, 737 now.
constexpr int kCollapseBatch = 8;

template <int W>
__global__ void __launch_bounds__(256) k_collapse(QEntry *q, unsigned *start, unsigned *cnt,
                                                  int lv, int64_t node_cap, const int64_t *toff,
                                                  const int64_t *ioff, BinTree T, float *nodes,
                                                  int L, int *err) {
  const int64_t e0 = start[lv], next = e0 + cnt[lv];
  const int64_t n = min(next, node_cap) - e0;  // (the capacity is never passed)
  if (blockIdx.x == 0 && threadIdx.x == 0) start[lv + 1] = (unsigned)next;
  const int lane = threadIdx.x & 31;
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  // warp-uniform trips: the warp's new nodes are numbered together
  for (int64_t k0 = blockIdx.x * (int64_t)blockDim.x + threadIdx.x - lane; k0 < n; k0 += stride) {
    const bool on = k0 + lane < n;
    int32_t fr[W];
    int2 rg[W];  // their ranges
    int nf = 0, inner = 0;
    int64_t base = 0, ib = 0;
    QEntry e{0, 0};
    auto range_of = [&](int32_t r) {
      return r < 0 ? make_int2(-r - 1, -r - 1) : T.range[ib + r];
    };
    auto box_of = [&](int32_t r) {
      return r < 0 ? T.leaf_box + 3 * (base + (-r - 1)) : T.box + 3 * (ib + r);
    };
    auto area_of = [&](int32_t r) {
      const Box6 b = ld_box(box_of(r));
      const float dx = b.b.y - b.a.x, dy = b.c.x - b.a.y, dz = b.c.y - b.b.x;
      return dx * dy + dy * dz + dz * dx;
    };
    if (on) {
      e = q[e0 + k0 + lane];
      base = toff[e.mesh];
      ib = ioff[e.mesh];
      float area[W];  // of those that may be opened, else -1
      auto put = [&](int k, int32_t r) {
        const int2 x = range_of(r);
        const float a = x.y - x.x + 1 <= L ? -1.f : area_of(r);
#pragma unroll
        for (int j = 0; j < W; ++j)
          if (j == k) {
            fr[j] = r;
            rg[j] = x;
            area[j] = a;
          }
      };
      const int2 er = range_of(e.bin);
      if (er.y - er.x + 1 <= L) {
        put(nf++, e.bin);
      } else {
        const int2 c = T.child[ib + e.bin];
        put(nf++, c.x);
        put(nf++, c.y);
        while (nf < W) {
          int best = -1;
          int32_t br = 0;
          float best_a = -1.f;
#pragma unroll
          for (int k = 0; k < W; ++k)
            if (k < nf && area[k] > best_a) {
              best_a = area[k];
              best = k;
              br = fr[k];
            }
          if (best < 0) break;
          const int2 c2 = T.child[ib + br];
          put(best, c2.x);
          put(nf++, c2.y);
        }
      }
#pragma unroll
      for (int k = 0; k < W; ++k) inner += k < nf && rg[k].y - rg[k].x + 1 > L;
    }
    // ids of this lane's inner children
    int incl = inner;
    for (int o = 1; o < 32; o <<= 1) {
      const int v = __shfl_up_sync(0xffffffffu, incl, o);
      if (lane >= o) incl += v;
    }
    const int tot = __shfl_sync(0xffffffffu, incl, 31);
    unsigned first = 0;
    if (lane == 0 && tot) first = atomicAdd(cnt + lv + 1, (unsigned)tot);
    int64_t id = next + __shfl_sync(0xffffffffu, first, 0) + (incl - inner);
    if (!on) continue;
    float4 *node = reinterpret_cast<float4 *>(nodes + (e0 + k0 + lane) * node_stride_words(W));
    {
      const Box6 b = ld_box(box_of(e.bin));
      node[0] = make_float4(b.a.x, b.a.y, b.b.x, b.b.y);
      node[1] = make_float4(b.c.x, b.c.y, 0.f, 0.f);
    }
#pragma unroll
    for (int k = 0; k < W; ++k) {
      if (k >= nf) {
        node[2 * k + 2] = make_float4(3e38f, 3e38f, 3e38f, -3e38f);
        node[2 * k + 3] = make_float4(-3e38f, -3e38f, __uint_as_float(kEmpty), 0.f);
        continue;
      }
      uint32_t word;
      const int c = rg[k].y - rg[k].x + 1;
      if (c <= L) {
        word = kLeafBit | ((uint32_t)rg[k].x << 3) | (uint32_t)(c - 1);
      } else if (id >= node_cap) {
        atomicExch(err, 1);
        word = kEmpty;
        ++id;
      } else {
        word = (uint32_t)id;
        q[id] = QEntry{fr[k], e.mesh};
        ++id;
      }
      const Box6 b = ld_box(box_of(fr[k]));
      node[2 * k + 2] = make_float4(b.a.x, b.a.y, b.b.x, b.b.y);
      node[2 * k + 3] = make_float4(b.c.x, b.c.y, __uint_as_float(word), 0.f);
    }
  }
}

__global__ void k_iota_roots(int32_t *roots, int64_t M) {
  for (int64_t m = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; m < M;
       m += (int64_t)gridDim.x * blockDim.x)
    roots[m] = (int32_t)m;
}

__global__ void k_init_queue(QEntry *q, int64_t M, const int64_t *toff, unsigned *start,
                             unsigned *cnt) {
  for (int64_t m = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; m < M;
       m += (int64_t)gridDim.x * blockDim.x)
    q[m] = QEntry{(toff[m + 1] - toff[m] > 1) ? 0 : -1, (int32_t)m};  // internal 0 is the root
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    start[0] = 0;
    cnt[0] = (unsigned)M;
  }
}

pj_status build_bvh(Ctx *ctx, Dataset *ds, int W, int L, cudaStream_t s) {
  const int64_t M = ds->M, F = ds->F;
  const int64_t n_int = F - M;
  auto nb = [&](int64_t n) {
    int64_t b = (n + 255) / 256, cap = (int64_t)ctx->num_sms * 32;
    return (int)std::max<int64_t>(1, std::min(b, cap));
  };
  TmpMem tmp(ctx, s);
  Bvh bvh;
  bvh.W = W;
  bvh.L = L;
  // 1. Morton keys, sorted per mesh
  uint64_t *k0, *k1;
  int32_t *i0;
  PJ_CK(tmp.get(&k0, F));
  PJ_CK(tmp.get(&k1, F));
  PJ_CK(tmp.get(&i0, F));
  PJ_CK(mem_get(ctx, (void **)&bvh.d_tri_order, sizeof(int32_t) * (size_t)std::max<int64_t>(F, 1), s));
  struct Guard {
    Ctx *ctx;
    Bvh *b;
    cudaStream_t s;
    bool ok = false;
    ~Guard() {
      if (ok) return;
      for (void *p : {(void *)b->d_nodes, (void *)b->d_roots, (void *)b->d_tri_order,
                      (void *)b->d_trirec})
        mem_put(ctx, p, s);
    }
  } guard{ctx, &bvh, s};
  k_morton<<<span_blocks(F), 256, 0, s>>>(ds->d_xyz, ds->d_tris, F, ds->d_toff, M, ds->d_aabb, k0, i0);
  int mbits = 1;
  while ((1ll << mbits) <= M) ++mbits;
  size_t tb = 0;
  PJ_CK(cub::DeviceRadixSort::SortPairs(nullptr, tb, k0, k1, i0, bvh.d_tri_order, (int)F, 0,
                                        30 + mbits, s));
  char *tstore;
  PJ_CK(tmp.get(&tstore, (int64_t)tb));
  PJ_CK(cub::DeviceRadixSort::SortPairs(tstore, tb, k0, k1, i0, bvh.d_tri_order, (int)F, 0,
                                        30 + mbits, s));
  // 2. binary radix trees
  std::vector<int64_t> h_ioff(M + 1);
  for (int64_t m = 0; m <= M; ++m) h_ioff[m] = ds->h_toff[m] - m;
  int64_t *d_ioff;
  PJ_CK(tmp.get(&d_ioff, M + 1));
  PJ_CK(cudaMemcpyAsync(d_ioff, h_ioff.data(), sizeof(int64_t) * (M + 1),
                        cudaMemcpyHostToDevice, s));
  BinTree T;
  PJ_CK(tmp.get(&T.child, n_int));
  PJ_CK(tmp.get(&T.range, n_int));
  PJ_CK(tmp.get(&T.par_int, n_int));
  PJ_CK(tmp.get(&T.par_leaf, F));
  PJ_CK(tmp.get(&T.box, 3 * n_int));
  PJ_CK(tmp.get(&T.leaf_box, 3 * F));
  PJ_CK(tmp.get(&T.visits, n_int));
  unsigned long long *d_big;  // binary nodes with more than L triangles
  PJ_CK(tmp.get(&d_big, 1));
  PJ_CK(cudaMemsetAsync(d_big, 0, 8, s));
  PJ_CK(cudaMemsetAsync(T.par_leaf, 0xff, sizeof(int32_t) * F, s));
  PJ_CK(cudaMemsetAsync(T.visits, 0, sizeof(int32_t) * std::max<int64_t>(n_int, 1), s));
  if (n_int > 0)
    k_karras<<<blocks_for(n_int, 256), 256, 0, s>>>(k1, ds->d_toff, d_ioff, M, n_int, T, L, d_big);
  // triangle boxes and records in leaf order
  PJ_CK(mem_get(ctx, (void **)&bvh.d_trirec, sizeof(float4) * 3 * (size_t)std::max<int64_t>(F, 1), s));
  k_leaves<<<nb(F), 256, 0, s>>>(ds->d_xyz, ds->d_tris, bvh.d_tri_order, k1, ds->d_emask,
                                 ds->d_toff, F, T.leaf_box, bvh.d_trirec);
  // 3. exact boxes bottom-up
  if (n_int > 0)
    k_refit<<<blocks_for(F, kRefitT), kRefitT, 0, s>>>(k1, ds->d_toff, d_ioff, F, T);
  PJ_CK(cudaGetLastError());
  // 4. collapse to W-wide nodes
  unsigned long long big = 0;
  PJ_CK(cudaMemcpyAsync(&big, d_big, 8, cudaMemcpyDeviceToHost, s));
  PJ_CK(cudaStreamSynchronize(s));
  const int64_t node_cap = (int64_t)big + M;
  const int sw = node_stride_words(W);
  float *nodes_tmp;
  PJ_CK(tmp.get(&nodes_tmp, node_cap * sw));
  QEntry *q;
  PJ_CK(tmp.get(&q, node_cap));
  constexpr int kMaxLevels = 4096;
  unsigned *lvl;  // first entry and number of entries of each level
  int *dflag;     // node capacity exceeded
  PJ_CK(tmp.get(&lvl, 2 * (kMaxLevels + 1)));
  PJ_CK(tmp.get(&dflag, 1));
  unsigned *start = lvl, *cnt = lvl + kMaxLevels + 1;
  PJ_CK(cudaMemsetAsync(lvl, 0, sizeof(unsigned) * 2 * (kMaxLevels + 1), s));
  PJ_CK(cudaMemsetAsync(dflag, 0, 4, s));
  k_init_queue<<<nb(M), 256, 0, s>>>(q, M, ds->d_toff, start, cnt);
  const auto kc = W == 2 ? k_collapse<2> : (W == 4 ? k_collapse<4> : k_collapse<8>);
  const int cgrid = (int)std::min<int64_t>(nb(node_cap), (int64_t)ctx->num_sms * 8);
  int levels = 0;  // levels with nodes
  int64_t n_nodes = 0;
  for (int lv = 0;;) {
    if (lv + kCollapseBatch > kMaxLevels)
      return fail(ctx, PJ_ERR_INTERNAL, "BVH collapse did not terminate");
    for (int k = 0; k < kCollapseBatch; ++k, ++lv)
      kc<<<cgrid, 256, 0, s>>>(q, start, cnt, lv, node_cap, ds->d_toff, d_ioff, T, nodes_tmp, L,
                               dflag);
    PJ_CK(cudaGetLastError());
    unsigned h[kCollapseBatch + 1];  // the levels after the batch's first
    PJ_CK(cudaMemcpyAsync(h, cnt + lv - kCollapseBatch, sizeof(h), cudaMemcpyDeviceToHost, s));
    int over = 0;
    PJ_CK(cudaMemcpyAsync(&over, dflag, 4, cudaMemcpyDeviceToHost, s));
    PJ_CK(cudaStreamSynchronize(s));
    if (over) return fail(ctx, PJ_ERR_INTERNAL, "BVH node capacity exceeded");
    for (int k = 0; k < kCollapseBatch && h[k]; ++k) {
      n_nodes += h[k];
      ++levels;
    }
    if (h[kCollapseBatch] == 0) break;
  }
  if (n_nodes * W >= (1ll << 30))
    return fail(ctx, PJ_ERR_INVALID_ARG, "dataset too large for 30-bit BVH slot ids");
  bvh.n_nodes = n_nodes;
  bvh.max_depth = levels;
  PJ_CK(mem_get(ctx, (void **)&bvh.d_nodes, sizeof(float) * (size_t)n_nodes * sw, s));
  PJ_CK(cudaMemcpyAsync(bvh.d_nodes, nodes_tmp, sizeof(float) * (size_t)n_nodes * sw,
                        cudaMemcpyDeviceToDevice, s));
  PJ_CK(mem_get(ctx, (void **)&bvh.d_roots, sizeof(int32_t) * (size_t)M, s));
  k_iota_roots<<<nb(M), 256, 0, s>>>(bvh.d_roots, M);
  PJ_CK(cudaGetLastError());
  PJ_CK(cudaStreamSynchronize(s));
  bvh.bytes = (int64_t)n_nodes * sw * 4 + 4 * M + 4 * F + 48 * F;
  guard.ok = true;
  ds->bvhs[{W, L}] = bvh;
  return PJ_OK;
}

}  // namespace pj
