// C-ABI entry points: contexts, dataset loading (quantisation check, closed-
// manifold check and unique edges, per-mesh boxes, lexicographic vertex
// order), exports and counters.
//
// Loading follows the paper's preprocessing/loading split (Sec. 4.2): each
// dataset becomes flat triangles with a triangle-to-object map (here: per-mesh
// offset ranges) and a per-object unique-edge set (Sec. 3.1 Step I: interior
// edges of a closed manifold are shared by exactly two triangles, so each is
// kept once, owned by one of its triangles).
#include <cub/cub.cuh>

#include <algorithm>
#include <cstdio>
#include <cstring>

#include "pj_internal.cuh"

namespace pj {

thread_local Exec *t_exec = nullptr;

// a serving thread keeps its own message; API calls set the context's
pj_status fail(Ctx *c, pj_status code, const std::string &msg) {
  if (t_exec) {
    t_exec->err = msg;
  } else if (c) {
    std::lock_guard<std::mutex> lk(c->err_mu);
    c->err = msg;
  }
  return code;
}

void clear_err(Ctx *c) {
  std::lock_guard<std::mutex> lk(c->err_mu);
  c->err.clear();
}

pj_status cuda_fail(Ctx *c, cudaError_t e, const char *what) {
  std::string m = std::string("CUDA error ") + cudaGetErrorName(e) + " (" +
                  cudaGetErrorString(e) + ") in " + what;
  return fail(c, e == cudaErrorMemoryAllocation ? PJ_ERR_NO_MEMORY : PJ_ERR_CUDA, m);
}

pj_status exec_init(Ctx *ctx, Exec *e) {
  cudaError_t r = cudaMalloc(&e->d_misc, kExecBytes);
  if (r == cudaSuccess) r = cudaMemset(e->d_misc, 0, kExecBytes);
  if (r == cudaSuccess) e->d_err = reinterpret_cast<int *>(e->d_misc + 8);
  if (r == cudaSuccess) r = cudaMallocHost(&e->h_pinned, 4096 + 8 * kFirstPairs);
  for (auto &ev : e->ev)
    if (r == cudaSuccess) r = cudaEventCreate(&ev);
  if (r != cudaSuccess) return cuda_fail(ctx, r, "exec_init");
  return PJ_OK;
}

void exec_free(Exec *e) {
  if (e->stream) {
    for (auto &kv : e->ws)
      if (kv.second.ptr) cudaFreeAsync(kv.second.ptr, e->stream);
    cudaStreamSynchronize(e->stream);
  } else {
    for (auto &kv : e->ws) cudaFree(kv.second.ptr);
  }
  e->ws.clear();
  cudaFree(e->d_misc);
  cudaFreeHost(e->h_pinned);
  for (auto &ev : e->ev)
    if (ev) cudaEventDestroy(ev);
  e->d_misc = nullptr;
  e->d_err = nullptr;
  e->h_pinned = nullptr;
  for (auto &ev : e->ev) ev = nullptr;
}

void *ws_get(Ctx *ctx, const char *name, size_t bytes, pj_status *st) {
  *st = PJ_OK;
  Exec *ex = cur_exec(ctx);
  Workspace &w = ex->ws[name];
  if (bytes == 0) bytes = 16;
  if (w.cap >= bytes) return w.ptr;
  const size_t old_cap = w.cap;
  w.zeroed = false;  // a new block, even at the same address, holds anything
  size_t want = bytes + bytes / 4;
  cudaError_t e;
  if (ex->stream) {
    // a serving slot: the old block is released and the new one taken in
    // the slot's stream order, so a growth does not wait for the batches of
    // the other slots (cudaFree would wait for the whole device); it grows
    // at least twofold, so that it grows a few times at most
    want = std::max(want, 2 * old_cap);
    if (w.ptr) cudaFreeAsync(w.ptr, ex->stream);
    w.ptr = nullptr;
    w.cap = 0;
    e = cudaMallocAsync(&w.ptr, want, ex->stream);
    if (e == cudaErrorMemoryAllocation) {
      mem_trim(ctx);
      e = cudaMallocAsync(&w.ptr, want, ex->stream);
    }
  } else {
    if (w.ptr) cudaFree(w.ptr);
    w.ptr = nullptr;
    w.cap = 0;
    e = cudaMalloc(&w.ptr, want);
    if (e == cudaErrorMemoryAllocation) {
      mem_trim(ctx);
      e = cudaMalloc(&w.ptr, want);
    }
  }
  if (e != cudaSuccess) {
    cudaGetLastError();
    w.ptr = nullptr;
    *st = cuda_fail(ctx, e, name);
    return nullptr;
  }
  w.cap = want;
  // workspaces back captured graphs: a new address invalidates them (only
  // the context's own scratch is ever captured)
  if (ex == &ctx->main) {
    for (auto &g : ctx->graphs) cudaGraphExecDestroy(g.second);
    ctx->graphs.clear();
  }
  return w.ptr;
}

void *ws_get_zeroed(Ctx *ctx, const char *name, size_t bytes, cudaStream_t s, pj_status *st) {
  Workspace &w = cur_exec(ctx)->ws[name];
  const void *before = w.ptr;
  void *p = ws_get(ctx, name, bytes, st);
  if (!p) return nullptr;
  if (p != before || !w.zeroed) {
    cudaError_t e = cudaMemsetAsync(p, 0, w.cap, s);
    if (e != cudaSuccess) {
      *st = cuda_fail(ctx, e, name);
      return nullptr;
    }
    w.zeroed = true;
  }
  return p;
}

void ws_mark_dirty(Ctx *ctx, const char *name) { cur_exec(ctx)->ws[name].zeroed = false; }

void *pool_get(Ctx *ctx, size_t bytes, cudaError_t *e) {
  *e = cudaSuccess;
  auto it = ctx->pool.lower_bound(bytes);
  if (it != ctx->pool.end() && it->first <= 4 * std::max<size_t>(bytes, 4096)) {
    void *p = it->second;
    ctx->pool_bytes -= it->first;
    ctx->pool.erase(it);
    return p;
  }
  size_t cap = 4096;
  while (cap < bytes) cap *= 2;
  void *p = nullptr;
  *e = cudaMalloc(&p, cap);
  if (*e == cudaErrorMemoryAllocation) {
    mem_trim(ctx);
    *e = cudaMalloc(&p, cap);
  }
  if (*e != cudaSuccess) {
    cudaGetLastError();
    return nullptr;
  }
  ctx->pool_cap[p] = cap;
  return p;
}

void pool_put(Ctx *ctx, void *p) {
  if (!p) return;
  auto it = ctx->pool_cap.find(p);
  if (it == ctx->pool_cap.end()) {
    cudaFree(p);
    return;
  }
  if (ctx->pool_bytes + it->second > (size_t(1) << 30)) {
    cudaFree(p);
    ctx->pool_cap.erase(it);
    return;
  }
  ctx->pool.emplace(it->second, p);
  ctx->pool_bytes += it->second;
}

void pool_release(Ctx *ctx) {
  for (auto &kv : ctx->pool) {
    cudaFree(kv.second);
    ctx->pool_cap.erase(kv.second);
  }
  ctx->pool.clear();
  ctx->pool_bytes = 0;
  for (auto &kv : ctx->hpool) {
    cudaFreeHost(kv.second);
    ctx->hpool_cap.erase(kv.second);
  }
  ctx->hpool.clear();
  ctx->hpool_bytes = 0;
}

void *hpool_get(Ctx *ctx, size_t bytes, cudaError_t *e) {
  *e = cudaSuccess;
  auto it = ctx->hpool.lower_bound(bytes);
  if (it != ctx->hpool.end() && it->first <= 4 * std::max<size_t>(bytes, 4096)) {
    void *p = it->second;
    ctx->hpool_bytes -= it->first;
    ctx->hpool.erase(it);
    return p;
  }
  size_t cap = 4096;
  while (cap < bytes) cap *= 2;
  void *p = nullptr;
  *e = cudaMallocHost(&p, cap);
  if (*e != cudaSuccess) {
    cudaGetLastError();
    return nullptr;
  }
  ctx->hpool_cap[p] = cap;
  return p;
}

void hpool_put(Ctx *ctx, void *p) {
  if (!p) return;
  auto it = ctx->hpool_cap.find(p);
  if (it == ctx->hpool_cap.end()) {
    cudaFreeHost(p);
    return;
  }
  if (ctx->hpool_bytes + it->second > (size_t(1) << 28)) {
    cudaFreeHost(p);
    ctx->hpool_cap.erase(it);
    return;
  }
  ctx->hpool.emplace(it->second, p);
  ctx->hpool_bytes += it->second;
}

void pairs_release(Ctx *ctx, pj_pairs *r) {
  if (r->pairs) {
    if (r->on_device) pool_put(ctx, r->pairs);
    else if (r->pairs_malloc) free(r->pairs);
    else hpool_put(ctx, r->pairs);
  }
  pool_put(ctx, r->flags);
  pool_put(ctx, r->cycles);
  memset(r, 0, sizeof(*r));
}

// ---------------------------------------------------------------------------
// Load kernels
// ---------------------------------------------------------------------------
__device__ __forceinline__ int64_t mesh_of(const int64_t *off, int64_t M, int64_t e) {
  // largest m with off[m] <= e (meshes may be empty)
  int64_t lo = 0, hi = M - 1;
  while (lo < hi) {
    int64_t mid = (lo + hi + 1) >> 1;
    if (off[mid] <= e) lo = mid; else hi = mid - 1;
  }
  return lo;
}

// sentinel boxes of meshes without vertices, and the start of the minima
__global__ void k_init_aabb(float *aabb, int64_t M) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < 6 * M;
       i += (int64_t)gridDim.x * blockDim.x)
    aabb[i] = i % 6 < 3 ? 3e38f : -3e38f;
}

// The quantisation check and every mesh's closed box in one pass over the
// vertices, kWarpSpan of them per warp (a block per mesh took 35 us for 15
// meshes of 13,000 vertices: too few blocks).  Coordinates that pass the check
// are not negative, so their order is that of their bits, and the sentinels'.
__global__ void __launch_bounds__(256) k_validate_boxes(const float *xyz, int64_t V,
                                                        const int64_t *voff, int64_t M,
                                                        int *aabb, unsigned long long *bad) {
  const int lane = threadIdx.x & 31;
  const int64_t w = blockIdx.x * (int64_t)8 + (threadIdx.x >> 5);
  const int64_t v0 = w * kWarpSpan, v1 = min(v0 + kWarpSpan, V);
  if (v0 >= v1) return;
  int64_t m = mesh_of(voff, M, v0);  // meshes may have no vertices
  for (int64_t f0 = v0; f0 < v1; ++m) {
    const int64_t f1 = min(voff[m + 1], v1);
    int lo[3] = {__float_as_int(3e38f), __float_as_int(3e38f), __float_as_int(3e38f)};
    int hi[3] = {__float_as_int(-3e38f), __float_as_int(-3e38f), __float_as_int(-3e38f)};
    for (int64_t v = f0 + lane; v < f1; v += 32)
#pragma unroll
      for (int d = 0; d < 3; ++d) {
        const float f = xyz[3 * v + d];
        if (!((f >= 0.f) && (f < 262144.f) && (f == floorf(f))))
          atomicMin(bad, (unsigned long long)(3 * v + d));
        // + 0: a negative zero counts as zero
        const int b = __float_as_int(f + 0.f);
        lo[d] = min(lo[d], b);
        hi[d] = max(hi[d], b);
      }
    if (f1 > f0) {
#pragma unroll
      for (int d = 0; d < 3; ++d) {
        const int a = __reduce_min_sync(0xffffffffu, lo[d]), b = __reduce_max_sync(0xffffffffu, hi[d]);
        if (lane == 0) {
          atomicMin(aabb + 6 * m + d, a);
          atomicMax(aabb + 6 * m + 3 + d, b);
        }
      }
      f0 = f1;
    }
  }
}

// the largest box extent on each axis over all meshes, to ext[0..2]
__global__ void __launch_bounds__(256) k_max_extent(const float *aabb, int64_t M,
                                                    unsigned long long *ext) {
  int e[3] = {0, 0, 0};
  for (int64_t m = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; m < M;
       m += (int64_t)gridDim.x * blockDim.x)
    for (int d = 0; d < 3; ++d) {
      const float x = aabb[6 * m + 3 + d] - aabb[6 * m + d];
      if (x > 0.f && x < 262144.f) e[d] = max(e[d], (int)x);
    }
  for (int d = 0; d < 3; ++d) {
    const int x = __reduce_max_sync(0xffffffffu, e[d]);
    if ((threadIdx.x & 31) == 0 && x) atomicMax(ext + d, (unsigned long long)x);
  }
}

// Global vertex ids of the triangles, their check, and the first step of the
// unique edges: a half-edge (lo, hi) takes a place in the list of its lower
// vertex (its rank there; ranks from kMaxRank set *big, see load_impl).
constexpr unsigned kMaxRank = 255;

__global__ void __launch_bounds__(256) k_convert_tris(const int32_t *tris_local, int64_t F,
                                                      const int64_t *voff, const int64_t *toff,
                                                      int64_t M, int32_t *tris_g, unsigned *deg,
                                                      uint8_t *rank, unsigned long long *bad,
                                                      unsigned long long *big) {
  const int lane = threadIdx.x & 31;
  const int64_t w = blockIdx.x * (int64_t)8 + (threadIdx.x >> 5);
  const int64_t t0 = w * kWarpSpan, t1 = min(t0 + kWarpSpan, F);
  if (t0 >= t1) return;
  int64_t m = warp_mesh_of(toff, M, t0, lane);
  int64_t end = toff[m + 1], vo = voff[m], nv = voff[m + 1] - vo;
  for (int64_t t = t0 + lane; t < t1; t += 32) {
    while (end <= t) {
      ++m;
      end = toff[m + 1];
      vo = voff[m];
      nv = voff[m + 1] - vo;
    }
    int id[3] = {tris_local[3 * t], tris_local[3 * t + 1], tris_local[3 * t + 2]};
    const bool ok = id[0] >= 0 && id[1] >= 0 && id[2] >= 0 && id[0] < nv && id[1] < nv &&
                    id[2] < nv && id[0] != id[1] && id[1] != id[2] && id[0] != id[2];
    if (!ok) {
      atomicMin(bad, (unsigned long long)t);
      id[0] = id[1] = id[2] = 0;
    }
#pragma unroll
    for (int k = 0; k < 3; ++k) tris_g[3 * t + k] = (int32_t)(vo + id[k]);
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      const unsigned r = atomicAdd(deg + vo + min(id[k], id[k == 2 ? 0 : k + 1]), 1u);
      rank[3 * t + k] = (uint8_t)min(r, kMaxRank);
      if (r >= kMaxRank) *big = 1ull;
    }
  }
}

// the half-edges into their lower vertices' lists: (higher vertex, half-edge)
__global__ void __launch_bounds__(256) k_edge_lists(const int32_t *tris_g, int64_t F,
                                                    const unsigned *off, const uint8_t *rank,
                                                    uint2 *list) {
  for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < F;
       t += (int64_t)gridDim.x * blockDim.x) {
    const unsigned id[3] = {(unsigned)tris_g[3 * t], (unsigned)tris_g[3 * t + 1],
                            (unsigned)tris_g[3 * t + 2]};
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      const unsigned a = id[k], b = id[k == 2 ? 0 : k + 1];
      list[off[min(a, b)] + rank[3 * t + k]] = make_uint2(max(a, b), (unsigned)(3 * t + k));
    }
  }
}

// One entry of a vertex's list: if it is the first with its higher vertex,
// the edge's half-edges are counted; the one that comes first among the
// triangles owns the edge, any number but two is an open or shared edge.
__device__ __forceinline__ bool edge_entry(const uint2 *e, int d, int i, unsigned *emask,
                                           unsigned long long *bad) {
  const unsigned hi = e[i].x;
  unsigned own = 0xffffffffu;
  int n = 0;
  for (int j = 0; j < d; ++j) {
    const uint2 q = e[j];
    if (q.x != hi) continue;
    if (j < i) return false;
    ++n;
    own = min(own, q.y);
  }
  if (n != 2) atomicMin(bad, (unsigned long long)own);
  const unsigned t = own / 3;
  atomicOr(emask + (t >> 2), 1u << (8 * (t & 3) + own % 3));
  return true;
}

// a thread per vertex; a warp for each of the few with long lists (poles)
constexpr int kLongList = 24;

__global__ void __launch_bounds__(256) k_edge_match(const uint2 *list, const unsigned *off,
                                                    int64_t V, unsigned *emask,
                                                    unsigned long long *n_unique,
                                                    unsigned long long *bad) {
  const int lane = threadIdx.x & 31;
  unsigned long long n = 0;
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t v0 = blockIdx.x * (int64_t)blockDim.x + threadIdx.x - lane; v0 < V; v0 += stride) {
    const int64_t v = v0 + lane;
    const unsigned b = v < V ? off[v] : 0u;
    const int d = v < V ? (int)(off[v + 1] - b) : 0;
    if (d <= kLongList)
      for (int i = 0; i < d; ++i) n += edge_entry(list + b, d, i, emask, bad);
    for (unsigned m = __ballot_sync(0xffffffffu, d > kLongList); m; m &= m - 1) {
      const int l = __ffs(m) - 1;
      const unsigned lb = __shfl_sync(0xffffffffu, b, l);
      const int ld = __shfl_sync(0xffffffffu, d, l);
      for (int i = lane; i < ld; i += 32) n += edge_entry(list + lb, ld, i, emask, bad);
    }
  }
  for (int o = 16; o > 0; o >>= 1) n += __shfl_xor_sync(0xffffffffu, n, o);
  __shared__ unsigned long long s_n[8];
  if (lane == 0) s_n[threadIdx.x >> 5] = n;
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int w = 1; w < 8; ++w) n += s_n[w];
    if (n) atomicAdd(n_unique, n);
  }
}

// per-mesh record (see Dataset::d_mrec); runs after the boxes and the
// lexicographic order exist
__global__ void k_mesh_rec(const float *aabb, const float *xyz, const int32_t *lexorder,
                           const int64_t *voff, const int64_t *toff, int64_t M, float4 *rec) {
  for (int64_t m = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; m < M;
       m += (int64_t)gridDim.x * blockDim.x) {
    const float *b = aabb + 6 * m;
    const int64_t v0 = voff[m], nv = voff[m + 1] - v0;
    float x = 0.f, y = 0.f, z = 0.f;
    if (nv > 0) {
      const int64_t g = lexorder[v0];
      x = xyz[3 * g];
      y = xyz[3 * g + 1];
      z = xyz[3 * g + 2];
    }
    rec[3 * m] = make_float4(b[0], b[1], b[2], x);
    rec[3 * m + 1] = make_float4(b[3], b[4], b[5], y);
    rec[3 * m + 2] = make_float4(z, __int_as_float((int)toff[m]), __int_as_float((int)v0),
                                 __int_as_float((int)nv));
  }
}

__global__ void k_halfedges(const int32_t *tris_g, int64_t F, uint64_t *keys,
                            uint32_t *vals) {
  for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < F;
       t += (int64_t)gridDim.x * blockDim.x) {
    for (int k = 0; k < 3; ++k) {
      uint32_t a = (uint32_t)tris_g[3 * t + k], b = (uint32_t)tris_g[3 * t + (k + 1) % 3];
      uint32_t lo = a < b ? a : b, hi = a < b ? b : a;
      keys[3 * t + k] = ((uint64_t)lo << 32) | hi;
      vals[3 * t + k] = (uint32_t)(3 * t + k);
    }
  }
}

// sorted half-edges: every key must occur exactly twice; the first of each
// run owns the edge
__global__ void k_edge_runs(const uint64_t *keys, const uint32_t *vals, int64_t n,
                            uint32_t *owner_bits, unsigned long long *n_unique,
                            unsigned long long *bad) {
  unsigned long long local = 0;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x) {
    uint64_t k = keys[i];
    if (i > 0 && keys[i - 1] == k) continue;  // not a run head
    bool two = (i + 1 < n) && keys[i + 1] == k && !((i + 2 < n) && keys[i + 2] == k);
    if (!two) atomicMin(bad, (unsigned long long)vals[i]);
    uint32_t v = vals[i];
    atomicOr(&owner_bits[v / 3], 1u << (v % 3));
    ++local;
  }
  for (int o = 16; o > 0; o >>= 1) local += __shfl_xor_sync(0xffffffffu, local, o);
  if ((threadIdx.x & 31) == 0 && local) atomicAdd(n_unique, local);
}

__global__ void k_pack_u8(const uint32_t *in, uint8_t *out, int64_t n) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x)
    out[i] = (uint8_t)in[i];
}

__global__ void k_lex_keys(const float *xyz, int64_t V, const int64_t *voff,
                           int64_t M, uint64_t *kxyz, uint32_t *kmesh,
                           int32_t *ids) {
  for (int64_t v = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; v < V;
       v += (int64_t)gridDim.x * blockDim.x) {
    uint64_t x = (uint64_t)xyz[3 * v], y = (uint64_t)xyz[3 * v + 1],
             z = (uint64_t)xyz[3 * v + 2];
    kxyz[v] = (x << 36) | (y << 18) | z;
    kmesh[v] = (uint32_t)mesh_of(voff, M, v);
    ids[v] = (int32_t)v;
  }
}

// mesh, x, y, z in one key: coordinates from the mesh's box, as many bits as
// the largest box takes on each axis
__global__ void __launch_bounds__(256) k_lex_keys_box(const float *xyz, int64_t V,
                                                      const int64_t *voff, int64_t M,
                                                      const float *aabb, int bx, int by, int bz,
                                                      uint64_t *key, int32_t *ids) {
  const int lane = threadIdx.x & 31;
  const int64_t w = blockIdx.x * (int64_t)8 + (threadIdx.x >> 5);
  const int64_t v0 = w * kWarpSpan, v1 = min(v0 + kWarpSpan, V);
  if (v0 >= v1) return;
  int64_t m = mesh_of(voff, M, v0);  // meshes may have no vertices
  for (int64_t v = v0 + lane; v < v1; v += 32) {
    while (voff[m + 1] <= v) ++m;
    const float *b = aabb + 6 * m;
    const uint64_t x = (uint64_t)(xyz[3 * v] - b[0]), y = (uint64_t)(xyz[3 * v + 1] - b[1]),
                   z = (uint64_t)(xyz[3 * v + 2] - b[2]);
    key[v] = (((((uint64_t)m << bx) | x) << by | y) << bz) | z;
    ids[v] = (int32_t)v;
  }
}

__global__ void k_gather_u32(const uint32_t *src, const int32_t *idx, uint32_t *dst,
                             int64_t n) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x)
    dst[i] = src[idx[i]];
}

static int nblk(Ctx *ctx, int64_t n, int t = 256) {
  int64_t b = (n + t - 1) / t;
  int64_t cap = (int64_t)ctx->num_sms * 32;
  if (b > cap) b = cap;
  if (b < 1) b = 1;
  return (int)b;
}

cudaError_t mem_get(Ctx *ctx, void **p, size_t bytes, cudaStream_t s) {
  cudaError_t e = cudaMallocFromPoolAsync(p, std::max<size_t>(bytes, 16), ctx->mem, s);
  if (e != cudaSuccess) {
    cudaGetLastError();
    *p = nullptr;
  }
  return e;
}

void mem_put(Ctx *ctx, void *p, cudaStream_t s) {
  (void)ctx;
  if (p) cudaFreeAsync(p, s);
}

void mem_trim(Ctx *ctx) {
  cudaGetLastError();
  // buffers given back in its order (a serving thread must not wait on a
  // stream that an API call may be capturing)
  if (!t_exec) cudaStreamSynchronize(ctx->stream);
  cudaMemPoolTrimTo(ctx->mem, 0);
}

void free_bvh(Ctx *ctx, Bvh &b) {
  for (void *p : {(void *)b.d_nodes, (void *)b.d_roots, (void *)b.d_tri_order, (void *)b.d_trirec})
    mem_put(ctx, p, ctx->stream);
  b = Bvh();
}

void free_dataset(Ctx *ctx, Dataset *d) {
  for (auto &kv : d->bvhs) free_bvh(ctx, kv.second);
  for (auto &kv : d->dbvhs) free_bvh(ctx, kv.second);
  for (void *p : {(void *)d->d_xyz, (void *)d->d_tris, (void *)d->d_voff, (void *)d->d_toff,
                  (void *)d->d_aabb, (void *)d->d_lexorder, (void *)d->d_emask,
                  (void *)d->d_mrec})
    mem_put(ctx, p, ctx->stream);
}

pj_status mesh_boxes(Ctx *ctx, const float *xyz, const int64_t *voff, int64_t M, float *box,
                     bool *ok) {
  cudaStream_t s = ctx->stream;
  const int64_t v0 = voff[0], V = voff[M] - v0;
  std::vector<int64_t> off(voff, voff + M + 1);
  for (auto &o : off) o -= v0;
  TmpMem tmp(ctx, s);
  int64_t *d_off;
  float *d_box;
  unsigned long long *d_bad, bad = 0;
  PJ_CK(tmp.get(&d_off, M + 1));
  PJ_CK(tmp.get(&d_box, 6 * M));
  PJ_CK(tmp.get(&d_bad, 1));
  PJ_CK(cudaMemcpyAsync(d_off, off.data(), sizeof(int64_t) * (M + 1), cudaMemcpyHostToDevice, s));
  PJ_CK(cudaMemsetAsync(d_bad, 0xff, 8, s));
  k_init_aabb<<<nblk(ctx, 6 * M), 256, 0, s>>>(d_box, M);
  k_validate_boxes<<<span_blocks(V), 256, 0, s>>>(xyz + 3 * v0, V, d_off, M,
                                                  reinterpret_cast<int *>(d_box), d_bad);
  PJ_CK(cudaGetLastError());
  PJ_CK(cudaMemcpyAsync(box, d_box, sizeof(float) * 6 * M, cudaMemcpyDeviceToHost, s));
  PJ_CK(cudaMemcpyAsync(&bad, d_bad, 8, cudaMemcpyDeviceToHost, s));
  PJ_CK(cudaStreamSynchronize(s));
  *ok = bad == ~0ull;
  return PJ_OK;
}

pj_status load_impl(Ctx *ctx, const float *xyz, int64_t V,
                           const int32_t *tris, int64_t F, const int64_t *voff,
                           const int64_t *toff, int64_t M, int dev_ptrs,
                           Dataset *d) {
  cudaStream_t s = ctx->stream;
  if (M <= 0) return fail(ctx, PJ_ERR_INVALID_ARG, "n_meshes must be positive");
  if (!voff || !toff) return fail(ctx, PJ_ERR_INVALID_ARG, "offset arrays are required");
  if (voff[0] != 0 || toff[0] != 0 || voff[M] != V || toff[M] != F)
    return fail(ctx, PJ_ERR_INVALID_ARG, "offsets must start at 0 and end at n_verts / n_tris");
  for (int64_t m = 0; m < M; ++m) {
    if (voff[m + 1] < voff[m] || toff[m + 1] < toff[m])
      return fail(ctx, PJ_ERR_INVALID_ARG, "offsets must be non-decreasing");
    if (toff[m + 1] - toff[m] > (1 << 28) - 2)
      return fail(ctx, PJ_ERR_INVALID_ARG, "a mesh has more than 2^28 - 2 triangles");
    if (toff[m + 1] == toff[m])
      return fail(ctx, PJ_ERR_NOT_MANIFOLD, "mesh " + std::to_string(m) + " has no triangles");
  }
  if (V >= (1ll << 31) - 1 || F >= (1ll << 31) - 1 || 3 * F >= (1ll << 32))
    return fail(ctx, PJ_ERR_INVALID_ARG, "dataset too large (2^31 - 1 vertices / triangles)");
  if ((V > 0 && !xyz) || (F > 0 && !tris)) return fail(ctx, PJ_ERR_INVALID_ARG, "null input");

  d->M = M; d->V = V; d->F = F;
  d->h_voff.assign(voff, voff + M + 1);
  d->h_toff.assign(toff, toff + M + 1);
  auto keep = [&](auto **p, int64_t n) {
    return mem_get(ctx, (void **)p, sizeof(**p) * (size_t)std::max<int64_t>(n, 1), s);
  };
  PJ_CK(keep(&d->d_xyz, 3 * V));
  PJ_CK(keep(&d->d_tris, 3 * F));
  PJ_CK(keep(&d->d_voff, M + 1));
  PJ_CK(keep(&d->d_toff, M + 1));
  PJ_CK(keep(&d->d_aabb, 6 * M));
  PJ_CK(keep(&d->d_lexorder, V));
  PJ_CK(keep(&d->d_emask, F + 3));  // written in words
  PJ_CK(keep(&d->d_mrec, 3 * M));
  d->bytes = 12 * V + 12 * F + 16 * (M + 1) + 24 * M + 4 * V + F + 48 * M;

  TmpMem tmp(ctx, s);
  int32_t *tris_local = nullptr;
  cudaMemcpyKind k = dev_ptrs ? cudaMemcpyDeviceToDevice : cudaMemcpyHostToDevice;
  PJ_CK(cudaMemcpyAsync(d->d_xyz, xyz, sizeof(float) * 3 * V, k, s));
  PJ_CK(tmp.get(&tris_local, 3 * F));
  PJ_CK(cudaMemcpyAsync(tris_local, tris, sizeof(int32_t) * 3 * F, k, s));
  PJ_CK(cudaMemcpyAsync(d->d_voff, voff, sizeof(int64_t) * (M + 1), cudaMemcpyHostToDevice, s));
  PJ_CK(cudaMemcpyAsync(d->d_toff, toff, sizeof(int64_t) * (M + 1), cudaMemcpyHostToDevice, s));

  // [0] bad coord, [1] bad tri, [2] bad edge, [3] n unique, [4] a long list,
  // [5..7] largest box extents
  unsigned long long *d_flags = nullptr;
  PJ_CK(tmp.get(&d_flags, 8));
  unsigned long long init[8] = {~0ull, ~0ull, ~0ull, 0ull, 0ull, 0ull, 0ull, 0ull};
  PJ_CK(cudaMemcpyAsync(d_flags, init, sizeof(init), cudaMemcpyHostToDevice, s));

  unsigned *deg, *deg_off;  // per vertex: half-edges whose lower vertex it is
  uint8_t *rank;
  PJ_CK(tmp.get(&deg, V + 1));  // (a bad triangle's ids may be one past the end)
  PJ_CK(tmp.get(&deg_off, V + 1));
  PJ_CK(tmp.get(&rank, 3 * F));
  PJ_CK(cudaMemsetAsync(deg, 0, sizeof(unsigned) * (V + 1), s));
  k_init_aabb<<<nblk(ctx, 6 * M), 256, 0, s>>>(d->d_aabb, M);
  if (V > 0)
    k_validate_boxes<<<span_blocks(V), 256, 0, s>>>(d->d_xyz, V, d->d_voff, M,
                                                    reinterpret_cast<int *>(d->d_aabb), d_flags);
  k_max_extent<<<std::min(nblk(ctx, M), ctx->num_sms), 256, 0, s>>>(d->d_aabb, M, d_flags + 5);
  k_convert_tris<<<span_blocks(F), 256, 0, s>>>(tris_local, F, d->d_voff, d->d_toff, M, d->d_tris,
                                                deg, rank, d_flags + 1, d_flags + 4);
  PJ_CK(cudaGetLastError());
  unsigned long long hf[8];
  PJ_CK(cudaMemcpyAsync(hf, d_flags, sizeof(hf), cudaMemcpyDeviceToHost, s));
  PJ_CK(cudaStreamSynchronize(s));
  if (hf[0] != ~0ull) {
    int64_t i = (int64_t)hf[0];
    char buf[160];
    snprintf(buf, sizeof(buf), "vertex %lld coordinate %lld is not an integer in [0, 2^18)",
             (long long)(i / 3), (long long)(i % 3));
    return fail(ctx, PJ_ERR_NOT_QUANTIZED, buf);
  }
  if (hf[1] != ~0ull) {
    int64_t t = (int64_t)hf[1];
    int64_t m = std::upper_bound(d->h_toff.begin(), d->h_toff.end(), t) - d->h_toff.begin() - 1;
    char buf[200];
    snprintf(buf, sizeof(buf), "triangle %lld of mesh %lld has a vertex id out of range "
             "or repeats a vertex", (long long)(t - d->h_toff[m]), (long long)m);
    return fail(ctx, PJ_ERR_NOT_MANIFOLD, buf);
  }

  // Unique edges and the closed-manifold check.  Half-edges meet in the list
  // of their lower vertex, about three long: a count (with the conversion
  // above), a scan, a scatter and a comparison within the lists, each about
  // one pass over the triangles.  A radix sort of all half-edges by 64-bit
  // keys made sixteen, and its run count queued a million atomics: 3,050 us
  // for 11 M triangles, 560 now (conversion included).  Lists are compared
  // entry by entry, so with a vertex of 255 half-edges or more the sort still
  // does it.
  if (hf[4] == 0) {
    uint2 *list;
    PJ_CK(tmp.get(&list, 3 * F));
    size_t tb = 0;
    PJ_CK(cub::DeviceScan::ExclusiveSum(nullptr, tb, deg, deg_off, V + 1, s));
    char *tstore;
    PJ_CK(tmp.get(&tstore, (int64_t)tb));
    PJ_CK(cub::DeviceScan::ExclusiveSum(tstore, tb, deg, deg_off, V + 1, s));
    PJ_CK(cudaMemsetAsync(d->d_emask, 0, (size_t)(F + 3) / 4 * 4, s));
    k_edge_lists<<<nblk(ctx, F), 256, 0, s>>>(d->d_tris, F, deg_off, rank, list);
    if (V > 0)
      k_edge_match<<<nblk(ctx, V), 256, 0, s>>>(list, deg_off, V,
                                                reinterpret_cast<unsigned *>(d->d_emask),
                                                d_flags + 3, d_flags + 2);
    PJ_CK(cudaGetLastError());
  } else {
    int64_t n = 3 * F;
    uint64_t *k0, *k1;
    uint32_t *v0, *v1, *bits;
    PJ_CK(tmp.get(&k0, n));
    PJ_CK(tmp.get(&k1, n));
    PJ_CK(tmp.get(&v0, n));
    PJ_CK(tmp.get(&v1, n));
    PJ_CK(tmp.get(&bits, F));
    PJ_CK(cudaMemsetAsync(bits, 0, sizeof(uint32_t) * F, s));
    k_halfedges<<<nblk(ctx, F), 256, 0, s>>>(d->d_tris, F, k0, v0);
    size_t tb = 0;
    PJ_CK(cub::DeviceRadixSort::SortPairs(nullptr, tb, k0, k1, v0, v1, (int)n, 0, 64, s));
    void *tstore;
    PJ_CK(tmp.get((char **)&tstore, (int64_t)tb));
    PJ_CK(cub::DeviceRadixSort::SortPairs(tstore, tb, k0, k1, v0, v1, (int)n, 0, 64, s));
    k_edge_runs<<<nblk(ctx, n), 256, 0, s>>>(k1, v1, n, bits, d_flags + 3, d_flags + 2);
    k_pack_u8<<<nblk(ctx, F), 256, 0, s>>>(bits, d->d_emask, F);
    PJ_CK(cudaGetLastError());
  }
  // Per-mesh lexicographic vertex order.  One stable sort where mesh, x, y
  // and z (from the mesh's box) fit 64 bits, of just those bits: 46 bits, six
  // passes, on 700 nuclei, against eleven of two sorts (by x, y, z, then by
  // mesh), which larger datasets of large meshes still take.
  auto bits = [](unsigned long long x) {
    int b = 0;
    while (x >> b) ++b;
    return b;
  };
  const int bx = bits(hf[5]), by = bits(hf[6]), bz = bits(hf[7]);
  const int mb = bits((unsigned long long)(M - 1));
  if (V > 0) {
    uint64_t *kx, *kx2;
    int32_t *ids;
    PJ_CK(tmp.get(&kx, V));
    PJ_CK(tmp.get(&kx2, V));
    PJ_CK(tmp.get(&ids, V));
    size_t tb = 0;
    char *tstore;
    if (mb + bx + by + bz <= 64) {
      const int end = std::max(1, mb + bx + by + bz);
      k_lex_keys_box<<<span_blocks(V), 256, 0, s>>>(d->d_xyz, V, d->d_voff, M, d->d_aabb, bx, by,
                                                    bz, kx, ids);
      PJ_CK(cub::DeviceRadixSort::SortPairs(nullptr, tb, kx, kx2, ids, d->d_lexorder, (int)V, 0,
                                            end, s));
      PJ_CK(tmp.get(&tstore, (int64_t)tb));
      PJ_CK(cub::DeviceRadixSort::SortPairs(tstore, tb, kx, kx2, ids, d->d_lexorder, (int)V, 0,
                                            end, s));
    } else {
      uint32_t *km, *km2;
      int32_t *ids2;
      PJ_CK(tmp.get(&km, V));
      PJ_CK(tmp.get(&km2, V));
      PJ_CK(tmp.get(&ids2, V));
      k_lex_keys<<<nblk(ctx, V), 256, 0, s>>>(d->d_xyz, V, d->d_voff, M, kx, km, ids);
      size_t tb2 = 0;
      PJ_CK(cub::DeviceRadixSort::SortPairs(nullptr, tb, kx, kx2, ids, ids2, (int)V, 0, 54, s));
      PJ_CK(cub::DeviceRadixSort::SortPairs(nullptr, tb2, km, km2, ids2, d->d_lexorder, (int)V, 0,
                                            mb, s));
      PJ_CK(tmp.get(&tstore, (int64_t)std::max(tb, tb2)));
      PJ_CK(cub::DeviceRadixSort::SortPairs(tstore, tb, kx, kx2, ids, ids2, (int)V, 0, 54, s));
      // mesh ids in the xyz-sorted order
      k_gather_u32<<<nblk(ctx, V), 256, 0, s>>>(km, ids2, km2, V);
      PJ_CK(cub::DeviceRadixSort::SortPairs(tstore, tb2, km2, km, ids2, d->d_lexorder, (int)V, 0,
                                            mb, s));
    }
    PJ_CK(cudaGetLastError());
  }
  if (M > 0) {
    k_mesh_rec<<<nblk(ctx, M), 256, 0, s>>>(d->d_aabb, d->d_xyz, d->d_lexorder, d->d_voff,
                                            d->d_toff, M, d->d_mrec);
    PJ_CK(cudaGetLastError());
  }
  PJ_CK(cudaMemcpyAsync(hf, d_flags, sizeof(hf), cudaMemcpyDeviceToHost, s));
  PJ_CK(cudaStreamSynchronize(s));
  if (hf[2] != ~0ull) {
    int64_t t = (int64_t)(hf[2] / 3);
    int64_t m = std::upper_bound(d->h_toff.begin(), d->h_toff.end(), t) - d->h_toff.begin() - 1;
    char buf[200];
    snprintf(buf, sizeof(buf), "mesh %lld is not a closed manifold: an edge of its triangle "
             "%lld is not shared by exactly two triangles", (long long)m,
             (long long)(t - d->h_toff[m]));
    return fail(ctx, PJ_ERR_NOT_MANIFOLD, buf);
  }
  d->E = (int64_t)hf[3];
  d->h_aabb.resize(6 * (size_t)M);
  if (M > 0)
    PJ_CK(cudaMemcpy(d->h_aabb.data(), d->d_aabb, sizeof(float) * 6 * M, cudaMemcpyDeviceToHost));
  // the admission grid: per cell the meshes whose box touches it, then the
  // summed-area table of those counts
  const int G = kOccG, G1 = kOccG + 1;
  const double cw = 262144.0 / G;
  std::vector<int64_t> cnt((size_t)G * G * G, 0);
  for (int64_t m = 0; m < M; ++m) {
    int lo[3], hi[3];
    for (int k = 0; k < 3; ++k) {
      lo[k] = std::min(G - 1, std::max(0, (int)(d->h_aabb[6 * m + k] / cw)));
      hi[k] = std::min(G - 1, std::max(0, (int)(d->h_aabb[6 * m + 3 + k] / cw)));
    }
    for (int x = lo[0]; x <= hi[0]; ++x)
      for (int y = lo[1]; y <= hi[1]; ++y)
        for (int z = lo[2]; z <= hi[2]; ++z) cnt[((size_t)x * G + y) * G + z] += 1;
  }
  d->occ_sat.assign((size_t)G1 * G1 * G1, 0);
  auto S = [&](int x, int y, int z) -> int64_t & { return d->occ_sat[((size_t)x * G1 + y) * G1 + z]; };
  for (int x = 1; x <= G; ++x)
    for (int y = 1; y <= G; ++y)
      for (int z = 1; z <= G; ++z)
        S(x, y, z) = cnt[((size_t)(x - 1) * G + (y - 1)) * G + (z - 1)] + S(x - 1, y, z) +
                     S(x, y - 1, z) + S(x, y, z - 1) - S(x - 1, y - 1, z) - S(x - 1, y, z - 1) -
                     S(x, y - 1, z - 1) + S(x - 1, y - 1, z - 1);
  return PJ_OK;
}

int64_t window_mesh_bound(const Dataset *d, const int32_t *wlo, const int32_t *whi) {
  const int G = kOccG, G1 = kOccG + 1;
  if (d->occ_sat.size() != (size_t)G1 * G1 * G1) return d->M;
  const double cw = 262144.0 / G;
  int a[3], b[3];
  for (int k = 0; k < 3; ++k) {
    a[k] = std::min(G - 1, std::max(0, (int)(wlo[k] / cw)));
    b[k] = std::min(G - 1, std::max(0, (int)(whi[k] / cw))) + 1;
  }
  auto S = [&](int x, int y, int z) { return d->occ_sat[((size_t)x * G1 + y) * G1 + z]; };
  const int64_t sum = S(b[0], b[1], b[2]) - S(a[0], b[1], b[2]) - S(b[0], a[1], b[2]) -
                      S(b[0], b[1], a[2]) + S(a[0], a[1], b[2]) + S(a[0], b[1], a[2]) +
                      S(b[0], a[1], a[2]) - S(a[0], a[1], a[2]);
  return std::min(sum, d->M);
}

}  // namespace pj

using namespace pj;

// ---------------------------------------------------------------------------
// C ABI
// ---------------------------------------------------------------------------
extern "C" {

pj_status pj_create(const pj_config *cfg, pj_ctx **out) {
  if (!out) return PJ_ERR_INVALID_ARG;
  *out = nullptr;
  Ctx *ctx = new (std::nothrow) Ctx();
  if (!ctx) return PJ_ERR_NO_MEMORY;
  if (cfg) ctx->cfg = *cfg;
  ctx->device = cfg ? cfg->device : 0;
  cudaError_t e = cudaSetDevice(ctx->device);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&ctx->num_sms, cudaDevAttrMultiProcessorCount, ctx->device);
  if (e == cudaSuccess) e = cudaStreamCreateWithFlags(&ctx->stream, cudaStreamNonBlocking);
  if (e == cudaSuccess) {
    cudaMemPoolProps props{};
    props.allocType = cudaMemAllocationTypePinned;
    props.location.type = cudaMemLocationTypeDevice;
    props.location.id = ctx->device;
    e = cudaMemPoolCreate(&ctx->mem, &props);
    unsigned long long keep = kMemKeep;
    if (e == cudaSuccess)
      e = cudaMemPoolSetAttribute(ctx->mem, cudaMemPoolAttrReleaseThreshold, &keep);
  }
  if (e == cudaSuccess) e = cudaMalloc(&ctx->d_counters, sizeof(unsigned long long) * C_NUM);
  if (e == cudaSuccess) e = cudaMemset(ctx->d_counters, 0, sizeof(unsigned long long) * C_NUM);
  if (e != cudaSuccess || exec_init(ctx, &ctx->main) != PJ_OK) {
    cudaGetLastError();
    exec_free(&ctx->main);
    if (ctx->mem) cudaMemPoolDestroy(ctx->mem);
    delete ctx;
    return e == cudaErrorMemoryAllocation ? PJ_ERR_NO_MEMORY : PJ_ERR_CUDA;
  }
  *out = reinterpret_cast<pj_ctx *>(ctx);
  return PJ_OK;
}

pj_status pj_destroy(pj_ctx *h) {
  Ctx *ctx = reinterpret_cast<Ctx *>(h);
  if (!ctx) return PJ_ERR_INVALID_ARG;
  cudaSetDevice(ctx->device);
  serve_stop(ctx);
  // work that reads the datasets may sit on any stream of the device (the
  // allocation-free join runs on the caller's), so wait for all of it
  cudaDeviceSynchronize();
  for (auto &kv : ctx->datasets) free_dataset(ctx, kv.second.get());
  for (auto &g : ctx->graphs) cudaGraphExecDestroy(g.second);
  exec_free(&ctx->main);
  pool_release(ctx);
  cudaFree(ctx->d_counters);
  cudaStreamSynchronize(ctx->stream);  // the datasets' buffers are back
  cudaMemPoolDestroy(ctx->mem);
  cudaStreamDestroy(ctx->stream);
  delete ctx;
  return PJ_OK;
}

const char *pj_last_error(pj_ctx *h) {
  Ctx *ctx = reinterpret_cast<Ctx *>(h);
  if (!ctx) return "null context";
  return ctx->err.c_str();
}

pj_status pj_load_meshes(pj_ctx *h, const float *xyz, int64_t n_verts,
                         const int32_t *tris, int64_t n_tris,
                         const int64_t *mesh_vert_off, const int64_t *mesh_tri_off,
                         int64_t n_meshes, int32_t ptr_is_device, pj_dataset *out) {
  Ctx *ctx = reinterpret_cast<Ctx *>(h);
  if (!ctx || !out) return PJ_ERR_INVALID_ARG;
  std::lock_guard<std::mutex> lk(ctx->mu);
  clear_err(ctx);
  if (n_verts < 0 || n_tris < 0) return fail(ctx, PJ_ERR_INVALID_ARG, "negative size");
  cudaSetDevice(ctx->device);
  std::unique_ptr<Dataset> d(new Dataset());
  pj_status st = load_impl(ctx, xyz, n_verts, tris, n_tris, mesh_vert_off, mesh_tri_off,
                           n_meshes, ptr_is_device, d.get());
  if (st != PJ_OK) {
    cudaStreamSynchronize(ctx->stream);
    free_dataset(ctx, d.get());
    return st;
  }
  std::unique_lock<std::shared_mutex> wl(ctx->ds_rw);
  int id = ctx->next_ds++;
  ctx->datasets[id] = std::move(d);
  *out = id;
  return PJ_OK;
}

static Dataset *get_ds(Ctx *ctx, pj_dataset id) {
  auto it = ctx->datasets.find(id);
  return it == ctx->datasets.end() ? nullptr : it->second.get();
}

pj_status pj_free_dataset(pj_ctx *h, pj_dataset id) {
  Ctx *ctx = reinterpret_cast<Ctx *>(h);
  if (!ctx) return PJ_ERR_INVALID_ARG;
  std::lock_guard<std::mutex> lk(ctx->mu);
  std::unique_lock<std::shared_mutex> wl(ctx->ds_rw);
  Dataset *d = get_ds(ctx, id);
  if (!d) return fail(ctx, PJ_ERR_INVALID_ARG, "unknown dataset");
  if (serve_uses(ctx, d))
    return fail(ctx, PJ_ERR_BUSY, "serving queries on this dataset have not been polled yet");
  cudaSetDevice(ctx->device);
  // joins that read this dataset may still run on a caller's stream (the
  // allocation-free join returns once its work is queued): wait for the
  // whole device, not only the context's stream
  cudaDeviceSynchronize();
  free_dataset(ctx, d);
  ctx->datasets.erase(id);
  for (auto &g : ctx->graphs) cudaGraphExecDestroy(g.second);
  ctx->graphs.clear();
  return PJ_OK;
}

pj_status pj_build_bvh(pj_ctx *h, pj_dataset id, const pj_bvh_params *p) {
  Ctx *ctx = reinterpret_cast<Ctx *>(h);
  if (!ctx) return PJ_ERR_INVALID_ARG;
  std::lock_guard<std::mutex> lk(ctx->mu);
  std::unique_lock<std::shared_mutex> wl(ctx->ds_rw);
  clear_err(ctx);
  Dataset *d = get_ds(ctx, id);
  if (!d) return fail(ctx, PJ_ERR_INVALID_ARG, "unknown dataset");
  int W = p && p->width ? p->width : 4, L = p && p->leaf_size ? p->leaf_size : 4;
  if (!(W == 2 || W == 4 || W == 8) || !(L == 1 || L == 2 || L == 4 || L == 8))
    return fail(ctx, PJ_ERR_INVALID_ARG, "width must be 2, 4 or 8 and leaf size 1, 2, 4 or 8");
  cudaSetDevice(ctx->device);
  if (d->bvhs.count({W, L})) {
    d->last_bvh = {W, L};
    return PJ_OK;
  }
  pj_status st = build_bvh(ctx, d, W, L, ctx->stream);
  if (st == PJ_OK) d->last_bvh = {W, L};
  return st;
}

pj_status pj_dataset_info_get(pj_ctx *h, pj_dataset id, pj_dataset_info *out) {
  Ctx *ctx = reinterpret_cast<Ctx *>(h);
  if (!ctx || !out) return PJ_ERR_INVALID_ARG;
  std::lock_guard<std::mutex> lk(ctx->mu);
  Dataset *d = get_ds(ctx, id);
  if (!d) return fail(ctx, PJ_ERR_INVALID_ARG, "unknown dataset");
  memset(out, 0, sizeof(*out));
  out->n_meshes = d->M;
  out->n_verts = d->V;
  out->n_tris = d->F;
  out->n_edges = d->E;
  out->device_bytes = d->bytes;
  auto it = d->bvhs.find(d->last_bvh);
  if (it != d->bvhs.end()) {
    out->bvh_nodes = it->second.n_nodes;
    out->bvh_width = it->second.W;
    out->bvh_leaf_size = it->second.L;
    out->bvh_max_depth = it->second.max_depth;
  }
  for (auto &kv : d->bvhs) out->device_bytes += kv.second.bytes;
  return PJ_OK;
}

pj_status pj_join_intersects(pj_ctx *h, pj_dataset a, pj_dataset b,
                             const int32_t *cand, int64_t n_cand, int32_t self_join,
                             void *stream, pj_pairs *out) {
  return pj_join_intersects_ex(h, a, b, cand, nullptr, n_cand, 0, self_join, nullptr,
                               stream, out);
}

pj_status pj_join_intersects_ex(pj_ctx *h, pj_dataset a, pj_dataset b,
                                const int32_t *cand, const int32_t *cand_off,
                                int64_t n_cand, int32_t cand_on_device,
                                int32_t self_join, const pj_join_opts *opts,
                                void *stream, pj_pairs *out) {
  Ctx *ctx = reinterpret_cast<Ctx *>(h);
  if (!ctx || !out) return PJ_ERR_INVALID_ARG;
  std::lock_guard<std::mutex> lk(ctx->mu);
  clear_err(ctx);
  memset(out, 0, sizeof(*out));
  Dataset *A = get_ds(ctx, a), *B = get_ds(ctx, b);
  if (!A || !B) return fail(ctx, PJ_ERR_INVALID_ARG, "unknown dataset");
  if (self_join && a != b) return fail(ctx, PJ_ERR_INVALID_ARG, "self_join needs a == b");
  if (cand && n_cand < 0) return fail(ctx, PJ_ERR_INVALID_ARG, "negative n_cand");
  if (!cand && cand_off) return fail(ctx, PJ_ERR_INVALID_ARG, "offsets need explicit candidates");
  cudaSetDevice(ctx->device);
  pj_join_opts o{};
  if (opts) o = *opts;
  return run_join(ctx, A, B, cand, cand_off, cand ? n_cand : -1, cand_on_device, self_join,
                  &o, stream ? (cudaStream_t)stream : ctx->stream, out);
}

pj_status pj_join_intersects_noalloc(pj_ctx *h, pj_dataset a, pj_dataset b,
                                     const int32_t *d_cand, int64_t n_cand, uint8_t *d_flags,
                                     int32_t *d_pairs, int64_t *d_count, void *stream) {
  Ctx *ctx = reinterpret_cast<Ctx *>(h);
  if (!ctx) return PJ_ERR_INVALID_ARG;
  std::lock_guard<std::mutex> lk(ctx->mu);
  clear_err(ctx);
  Dataset *A = get_ds(ctx, a), *B = get_ds(ctx, b);
  if (!A || !B) return fail(ctx, PJ_ERR_INVALID_ARG, "unknown dataset");
  cudaSetDevice(ctx->device);
  return run_join_noalloc(ctx, A, B, d_cand, n_cand, d_flags, d_pairs, d_count,
                          stream ? (cudaStream_t)stream : ctx->stream);
}

pj_status pj_join_tiled(pj_ctx *h, const pj_host_meshes *a, const pj_host_meshes *b,
                        int32_t self_join, const pj_tiled_opts *opts, pj_pairs *out,
                        pj_tiled_stats *stats) {
  Ctx *ctx = reinterpret_cast<Ctx *>(h);
  if (!ctx || !out || !a || (!self_join && !b)) return PJ_ERR_INVALID_ARG;
  std::lock_guard<std::mutex> lk(ctx->mu);
  clear_err(ctx);
  memset(out, 0, sizeof(*out));
  cudaSetDevice(ctx->device);
  pj_tiled_opts o{};
  if (opts) o = *opts;
  return run_join_tiled(ctx, a, b, self_join, &o, out, stats);
}

pj_status pj_dataset_join(pj_ctx *h, pj_dataset a, pj_dataset b, int32_t self_join,
                          const pj_dsjoin_opts *opts, pj_pairs *out, pj_dsjoin_stats *stats) {
  Ctx *ctx = reinterpret_cast<Ctx *>(h);
  if (!ctx || !out) return PJ_ERR_INVALID_ARG;
  std::lock_guard<std::mutex> lk(ctx->mu);
  clear_err(ctx);
  memset(out, 0, sizeof(*out));
  Dataset *A = get_ds(ctx, a), *B = get_ds(ctx, b);
  if (!A || !B) return fail(ctx, PJ_ERR_INVALID_ARG, "unknown dataset");
  if (self_join && a != b) return fail(ctx, PJ_ERR_INVALID_ARG, "self_join needs a == b");
  cudaSetDevice(ctx->device);
  pj_dsjoin_opts o{};
  if (opts) o = *opts;
  return run_dataset_join(ctx, A, B, self_join, &o, out, stats, ctx->stream);
}

pj_status pj_estimate_join(pj_ctx *h, pj_dataset a, pj_dataset b, int32_t grid,
                           double *cells_out, pj_estimate *out) {
  Ctx *ctx = reinterpret_cast<Ctx *>(h);
  if (!ctx || !out) return PJ_ERR_INVALID_ARG;
  std::lock_guard<std::mutex> lk(ctx->mu);
  clear_err(ctx);
  Dataset *A = get_ds(ctx, a), *B = get_ds(ctx, b);
  if (!A || !B) return fail(ctx, PJ_ERR_INVALID_ARG, "unknown dataset");
  if (grid < 0) return fail(ctx, PJ_ERR_INVALID_ARG, "negative grid");
  cudaSetDevice(ctx->device);
  return run_estimate(ctx, A, B, grid, cells_out, out, ctx->stream);
}

pj_status pj_submit(pj_ctx *h, const pj_query *q, pj_ticket *out) {
  Ctx *ctx = reinterpret_cast<Ctx *>(h);
  if (!ctx || !q || !out) return PJ_ERR_INVALID_ARG;
  *out = 0;
  std::shared_lock<std::shared_mutex> rl(ctx->ds_rw);
  auto ia = ctx->datasets.find(q->a), ib = ctx->datasets.find(q->b);
  if (ia == ctx->datasets.end() || ib == ctx->datasets.end()) return PJ_ERR_INVALID_ARG;
  if (q->self_join && q->a != q->b) return PJ_ERR_INVALID_ARG;
  return serve_submit(ctx, ia->second.get(), ib->second.get(), q, out);
}

pj_status pj_poll(pj_ctx *h, pj_ticket t, int32_t wait, pj_pairs *out, pj_query_stats *stats) {
  Ctx *ctx = reinterpret_cast<Ctx *>(h);
  if (!ctx || !out) return PJ_ERR_INVALID_ARG;
  return serve_poll(ctx, t, wait, out, stats);
}

pj_status pj_free_pairs(pj_ctx *h, pj_pairs *res) {
  Ctx *ctx = reinterpret_cast<Ctx *>(h);
  if (!ctx || !res) return PJ_ERR_INVALID_ARG;
  std::lock_guard<std::mutex> lk(ctx->mu);
  cudaSetDevice(ctx->device);
  pairs_release(ctx, res);
  return PJ_OK;
}

pj_status pj_autotune(pj_ctx *h, pj_dataset a, pj_dataset b, const int32_t *cand,
                      int64_t n_cand, int32_t self_join, const pj_tune_space *space,
                      pj_join_opts *best, pj_tune_entry *table, int32_t table_cap,
                      int32_t *table_n) {
  Ctx *ctx = reinterpret_cast<Ctx *>(h);
  if (!ctx || !space || !best) return PJ_ERR_INVALID_ARG;
  std::lock_guard<std::mutex> lk(ctx->mu);
  std::unique_lock<std::shared_mutex> wl(ctx->ds_rw);
  clear_err(ctx);
  Dataset *A = get_ds(ctx, a), *B = get_ds(ctx, b);
  if (!A || !B) return fail(ctx, PJ_ERR_INVALID_ARG, "unknown dataset");
  if (self_join && a != b) return fail(ctx, PJ_ERR_INVALID_ARG, "self_join needs a == b");
  cudaSetDevice(ctx->device);
  int n = 0;
  pj_status st = run_autotune(ctx, A, B, cand, cand ? n_cand : -1, self_join, space, best, table,
                              table ? table_cap : 0, &n);
  if (table_n) *table_n = n;
  return st;
}

pj_status pj_set_test_limits(pj_ctx *h, const pj_test_limits *limits) {
  Ctx *ctx = reinterpret_cast<Ctx *>(h);
  if (!ctx) return PJ_ERR_INVALID_ARG;
  std::lock_guard<std::mutex> lk(ctx->mu);
  ctx->limits = limits ? *limits : pj_test_limits{};
  for (auto &g : ctx->graphs) cudaGraphExecDestroy(g.second);  // captured with the old ones
  ctx->graphs.clear();
  return PJ_OK;
}

pj_status pj_get_counters(pj_ctx *h, pj_counters *out) {
  Ctx *ctx = reinterpret_cast<Ctx *>(h);
  if (!ctx || !out) return PJ_ERR_INVALID_ARG;
  std::lock_guard<std::mutex> lk(ctx->mu);
  cudaSetDevice(ctx->device);
  unsigned long long c[C_NUM];
  cudaError_t e = cudaMemcpy(c, ctx->d_counters, sizeof(c), cudaMemcpyDeviceToHost);
  if (e != cudaSuccess) return cuda_fail(ctx, e, "pj_get_counters");
  memset(out, 0, sizeof(*out));
  out->pairs_refined = c[C_PAIRS];
  out->node_pairs = c[C_NODE_PAIRS];
  out->box_tests = c[C_BOX_TESTS];
  out->leaf_pairs = c[C_LEAF_PAIRS];
  out->edge_slab_tests = c[C_SLAB_TESTS];
  out->segtri_tests = c[C_SEGTRI];
  out->exact_fallbacks = c[C_FALLBACK];
  out->parity_rays = c[C_PARITY_RAYS];
  out->parity_nodes = c[C_PARITY_NODES];
  out->parity_tri_tests = c[C_PARITY_TRIS];
  out->bytes_fetched = c[C_BYTES];
  out->pairs_hit = c[C_HITS];
  out->kernel_launches = ctx->launches.load();
  out->tasks_spilled = c[C_SPILLED];
  out->tasks_resumed = c[C_TASKS];
  out->bytes_tasks = c[C_BYTES_TASKS];
  out->bytes_parity = c[C_BYTES_PARITY];
  out->bytes_expand = c[C_BYTES_EXPAND];
  out->bytes_leaf = c[C_BYTES_LEAF];
  out->parity_handed_over = c[C_PAR_HANDOVER];
  return PJ_OK;
}

pj_status pj_reset_counters(pj_ctx *h) {
  Ctx *ctx = reinterpret_cast<Ctx *>(h);
  if (!ctx) return PJ_ERR_INVALID_ARG;
  std::lock_guard<std::mutex> lk(ctx->mu);
  cudaSetDevice(ctx->device);
  cudaError_t e = cudaMemset(ctx->d_counters, 0, sizeof(unsigned long long) * C_NUM);
  ctx->launches = 0;
  return e == cudaSuccess ? PJ_OK : cuda_fail(ctx, e, "pj_reset_counters");
}

pj_status pj_segtri_batch(pj_ctx *h, const float *pq, const float *abc, int64_t n,
                          int32_t mode, uint8_t *res, int64_t *n_fallback, void *stream) {
  Ctx *ctx = reinterpret_cast<Ctx *>(h);
  if (!ctx || n < 0 || (n > 0 && (!pq || !abc || !res))) return PJ_ERR_INVALID_ARG;
  if (mode != PJ_LEAF_FILTERED && mode != PJ_LEAF_EXACT && mode != PJ_LEAF_STATIC)
    return PJ_ERR_INVALID_ARG;
  std::lock_guard<std::mutex> lk(ctx->mu);
  clear_err(ctx);
  cudaSetDevice(ctx->device);
  return run_segtri_batch(ctx, pq, abc, n, mode, res, n_fallback,
                          stream ? (cudaStream_t)stream : ctx->stream);
}

pj_status pj_export_bvh(pj_ctx *h, pj_dataset id, int32_t W, int32_t L, int32_t *nodes,
                        int32_t *roots, int32_t *tri_order, int64_t *n_nodes) {
  Ctx *ctx = reinterpret_cast<Ctx *>(h);
  if (!ctx || !n_nodes) return PJ_ERR_INVALID_ARG;
  std::lock_guard<std::mutex> lk(ctx->mu);
  Dataset *d = get_ds(ctx, id);
  if (!d) return fail(ctx, PJ_ERR_INVALID_ARG, "unknown dataset");
  auto it = d->bvhs.find({W, L});
  if (it == d->bvhs.end()) return fail(ctx, PJ_ERR_INVALID_ARG, "no BVH with that width / leaf size");
  Bvh &b = it->second;
  cudaSetDevice(ctx->device);
  *n_nodes = b.n_nodes;
  int sw = node_stride_words(W);
  if (nodes) PJ_CK(cudaMemcpy(nodes, b.d_nodes, 4 * (size_t)b.n_nodes * sw, cudaMemcpyDeviceToHost));
  if (roots) PJ_CK(cudaMemcpy(roots, b.d_roots, 4 * d->M, cudaMemcpyDeviceToHost));
  if (tri_order) {
    PJ_CK(cudaMemcpy(tri_order, b.d_tri_order, 4 * d->F, cudaMemcpyDeviceToHost));
    for (int64_t m = 0; m < d->M; ++m)
      for (int64_t t = d->h_toff[m]; t < d->h_toff[m + 1]; ++t)
        tri_order[t] -= (int32_t)d->h_toff[m];
  }
  return PJ_OK;
}

pj_status pj_export_mesh_data(pj_ctx *h, pj_dataset id, float *aabb, int32_t *lex_first,
                              uint8_t *edge_owner) {
  Ctx *ctx = reinterpret_cast<Ctx *>(h);
  if (!ctx) return PJ_ERR_INVALID_ARG;
  std::lock_guard<std::mutex> lk(ctx->mu);
  Dataset *d = get_ds(ctx, id);
  if (!d) return fail(ctx, PJ_ERR_INVALID_ARG, "unknown dataset");
  cudaSetDevice(ctx->device);
  if (aabb) PJ_CK(cudaMemcpy(aabb, d->d_aabb, sizeof(float) * 6 * d->M, cudaMemcpyDeviceToHost));
  if (edge_owner) PJ_CK(cudaMemcpy(edge_owner, d->d_emask, d->F, cudaMemcpyDeviceToHost));
  if (lex_first) {
    std::vector<int32_t> lo((size_t)d->V);
    PJ_CK(cudaMemcpy(lo.data(), d->d_lexorder, 4 * d->V, cudaMemcpyDeviceToHost));
    for (int64_t m = 0; m < d->M; ++m)
      lex_first[m] = d->h_voff[m + 1] > d->h_voff[m]
                         ? lo[d->h_voff[m]] - (int32_t)d->h_voff[m] : -1;
  }
  return PJ_OK;
}

}  // extern "C"
