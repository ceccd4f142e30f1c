// Bounding-box filter join by a sweep along x (Sec. 3.1, the filter step: the
// candidate pairs are the mesh pairs whose closed boxes overlap).
//
// For joins whose all-pairs count is large (tens of thousands of meshes a
// side) testing every pair costs more than the refinement; here the boxes of
// both sides are put in order of the x bucket their low x falls in (2^14
// buckets of 16 grid units, a counting sort), and each box is tested only
// against the boxes after it in that order up to the last one of its high x's
// bucket -- every pair of boxes that overlap on x meets exactly once that
// way, from the one that comes first.  A warp takes a box and tests 32 others
// a step; boxes with long ranges are listed and shared by several warps.  The
// pairs found are listed, counted per mesh of side A, placed in A's order by
// a scan of the counts, and each mesh's few are ordered by B, so that the
// result has the (id A, id B) order of the all-pairs join and every later
// step sees the same candidate list.
//
// What bounds it: launches and one host wait (for the pairs' number, which
// sizes the join's buffers); the test pass is about 33 us on 55,000 urban
// meshes.  Radix sorts of the boxes (4 passes) and of the pairs (8), the test
// run twice and two host waits before this took 359 us there, 116 now
// (267 and 85 on 6,007 x 9,001 cells and nuclei).  The sort of
// the pairs is still taken when a mesh has kSwMost pairs or more: ordering
// its list compares all of them with each other.
#include <cub/cub.cuh>

#include "pj_internal.cuh"

namespace pj {

constexpr int SW_T = 256;
constexpr int kSwShift = 4;                           // grid units per bucket: 2^4
constexpr int kSwBuckets = 1 << (18 - kSwShift);      // coordinates lie in [0, 2^18)
constexpr int kSwShort = 16;                          // steps a box's own warp takes
constexpr int kSwMost = 1024;                         // pairs of a mesh ordered in place

__device__ __forceinline__ int sw_bucket(float x) { return (int)x >> kSwShift; }

__device__ __forceinline__ const float *sw_box(const float *aabbA, int64_t MA, const float *aabbB,
                                               int64_t i) {
  return i < MA ? aabbA + 6 * i : aabbB + 6 * (i - MA);
}

// each box's rank in its bucket
__global__ void __launch_bounds__(SW_T) k_sw_rank(const float *aabbA, int64_t MA,
                                                  const float *aabbB, int64_t n, int *hist,
                                                  int *rank) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x)
    rank[i] = atomicAdd(hist + sw_bucket(sw_box(aabbA, MA, aabbB, i)[0]), 1);
}

// one block: off[b] = boxes in buckets before b, off[kSwBuckets] = all
__global__ void __launch_bounds__(1024) k_sw_offsets(const int *hist, int *off) {
  constexpr int PER = kSwBuckets / 1024;
  __shared__ int s_w[32];
  const int t = threadIdx.x, lane = t & 31;
  int v[PER], sum = 0;
#pragma unroll
  for (int k = 0; k < PER; k += 4) {
    const int4 q = reinterpret_cast<const int4 *>(hist)[(t * PER + k) / 4];
    v[k] = q.x;
    v[k + 1] = q.y;
    v[k + 2] = q.z;
    v[k + 3] = q.w;
  }
#pragma unroll
  for (int k = 0; k < PER; ++k) {
    const int x = v[k];
    v[k] = sum;
    sum += x;
  }
  int incl = sum;
  for (int o = 1; o < 32; o <<= 1) {
    const int x = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += x;
  }
  if (lane == 31) s_w[t >> 5] = incl;
  __syncthreads();
  if (t < 32) {
    int x = s_w[t];
    for (int o = 1; o < 32; o <<= 1) {
      const int y = __shfl_up_sync(0xffffffffu, x, o);
      if (t >= o) x += y;
    }
    s_w[t] = x;
  }
  __syncthreads();
  const int before = (t >= 32 ? s_w[(t >> 5) - 1] : 0) + incl - sum;
#pragma unroll
  for (int k = 0; k < PER; k += 4)
    reinterpret_cast<int4 *>(off)[(t * PER + k) / 4] =
        make_int4(before + v[k], before + v[k + 1], before + v[k + 2], before + v[k + 3]);
  if (t == 1023) off[kSwBuckets] = before + sum;
}

// the ordered boxes, two float4 each: (lo x, lo y, lo z, hi x), (hi y, hi z,
// id, end of its range) with id < MA for side A and MA + j for mesh j of B
__global__ void __launch_bounds__(SW_T) k_sw_place(const float *aabbA, int64_t MA,
                                                   const float *aabbB, int64_t n, const int *off,
                                                   const int *rank, float4 *sb) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x) {
    const float *b = sw_box(aabbA, MA, aabbB, i);
    const int64_t p = off[sw_bucket(b[0])] + rank[i];
    sb[2 * p] = make_float4(b[0], b[1], b[2], b[3]);
    sb[2 * p + 1] = make_float4(b[4], b[5], __int_as_float((int)i),
                                __int_as_float(off[sw_bucket(b[3]) + 1]));
  }
}

// [0] pairs found, [1] boxes with long ranges, [2] a mesh of kSwMost pairs
enum { SW_PAIRS = 0, SW_LONG, SW_MANY, SW_WORDS };

// A warp's part of the pair list: hits wait in shared memory until there are
// 32 for one reservation.
struct SwOut {
  uint64_t *keys;   // (id A << 32 | id B), the first `cap` found
  int64_t cap;
  int *cnt;         // per mesh of A
  unsigned long long *words;
};

__device__ __forceinline__ void sw_flush(const SwOut &o, uint64_t *buf, int &nbuf, int n,
                                         int lane) {
  unsigned long long base = 0;
  if (lane == 0) base = atomicAdd(o.words + SW_PAIRS, (unsigned long long)n);
  base = __shfl_sync(0xffffffffu, base, 0);
  if (lane < n && (int64_t)(base + lane) < o.cap) o.keys[base + lane] = buf[lane];
  __syncwarp();
  const bool more = lane < nbuf - n;
  const uint64_t k = more ? buf[n + lane] : 0;
  __syncwarp();
  if (more) buf[lane] = k;
  nbuf -= n;
  __syncwarp();
}

// box (P0, P1) against box q of the order; the pair goes to the list
__device__ __forceinline__ void sw_step(const float4 *sb, const float4 &P0, const float4 &P1,
                                        int64_t q, bool on, int64_t MA, int self_join,
                                        const SwOut &o, uint64_t *buf, int &nbuf, int lane) {
  bool hit = false;
  int vp = __float_as_int(P1.z), vq = 0;
  if (on) {
    const float4 Q0 = sb[2 * q], Q1 = sb[2 * q + 1];
    vq = __float_as_int(Q1.z);
    hit = (self_join || (vp < MA) != (vq < MA)) && P0.x <= Q0.w && Q0.x <= P0.w &&
          P0.y <= Q1.x && Q0.y <= P1.x && P0.z <= Q1.y && Q0.z <= P1.y;
  }
  const unsigned m = __ballot_sync(0xffffffffu, hit);
  if (!m) return;
  if (hit) {
    int a, b;
    if (self_join) {
      a = min(vp, vq);
      b = max(vp, vq);
    } else {
      a = vp < MA ? vp : vq;
      b = (vp < MA ? vq : vp) - (int)MA;
    }
    if (atomicAdd(o.cnt + a, 1) + 1 >= kSwMost) o.words[SW_MANY] = 1ull;
    buf[nbuf + __popc(m & ((1u << lane) - 1u))] = ((uint64_t)(uint32_t)a << 32) | (uint32_t)b;
  }
  nbuf += __popc(m);
  __syncwarp();
  if (nbuf >= 32) sw_flush(o, buf, nbuf, 32, lane);
}

// a warp per box; those of more than kSwShort steps go to `longs`
__global__ void __launch_bounds__(SW_T) k_sw_short(const float4 *sb, int64_t n, int64_t MA,
                                                   int self_join, SwOut o, int *longs) {
  __shared__ uint64_t s_buf[SW_T / 32][64];
  const int lane = threadIdx.x & 31;
  uint64_t *buf = s_buf[threadIdx.x >> 5];
  int nbuf = 0;
  const int64_t nw = (int64_t)gridDim.x * (SW_T / 32);
  for (int64_t p = blockIdx.x * (int64_t)(SW_T / 32) + (threadIdx.x >> 5); p < n; p += nw) {
    const float4 P0 = sb[2 * p], P1 = sb[2 * p + 1];
    const int64_t end = __float_as_int(P1.w);
    if (end - p - 1 > 32 * kSwShort) {
      if (lane == 0) longs[atomicAdd(o.words + SW_LONG, 1ull)] = (int)p;
      continue;
    }
    for (int64_t q0 = p + 1; q0 < end; q0 += 32)
      sw_step(sb, P0, P1, q0 + lane, q0 + lane < end, MA, self_join, o, buf, nbuf, lane);
  }
  if (nbuf > 0) sw_flush(o, buf, nbuf, nbuf, lane);
}

// the listed boxes, as many warps to each as there are for it
__global__ void __launch_bounds__(SW_T) k_sw_long(const float4 *sb, int64_t MA, int self_join,
                                                  SwOut o, const int *longs) {
  __shared__ uint64_t s_buf[SW_T / 32][64];
  const int lane = threadIdx.x & 31;
  uint64_t *buf = s_buf[threadIdx.x >> 5];
  int nbuf = 0;
  const int64_t nw = (int64_t)gridDim.x * (SW_T / 32);
  const int64_t w = blockIdx.x * (int64_t)(SW_T / 32) + (threadIdx.x >> 5);
  const int64_t nl = (int64_t)o.words[SW_LONG];
  if (nl == 0) return;
  const int64_t g = max((int64_t)1, nw / nl);  // warps to a box
  if (w >= nw / g * g) return;
  for (int64_t l = w / g; l < nl; l += nw / g) {
    const int64_t p = longs[l];
    const float4 P0 = sb[2 * p], P1 = sb[2 * p + 1];
    const int64_t end = __float_as_int(P1.w);
    for (int64_t q0 = p + 1 + 32 * (w % g); q0 < end; q0 += 32 * g)
      sw_step(sb, P0, P1, q0 + lane, q0 + lane < end, MA, self_join, o, buf, nbuf, lane);
  }
  if (nbuf > 0) sw_flush(o, buf, nbuf, nbuf, lane);
}

// the listed pairs to their mesh's places (counting its count down), any order
__global__ void __launch_bounds__(SW_T) k_sw_scatter(const uint64_t *keys, int64_t n,
                                                     const int *off, int *cnt, int2 *cand) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x) {
    const int a = (int)(keys[i] >> 32);
    cand[off[a] + atomicSub(cnt + a, 1) - 1] = make_int2(a, (int)(keys[i] & 0xffffffffull));
  }
}

// each mesh's pairs by B: a thread sorts up to kSwInsert, a warp places more
// by their rank (each pair's B compared with all of them)
constexpr int kSwInsert = 8;

__global__ void __launch_bounds__(SW_T) k_sw_order(const int *off, int64_t MA, int2 *cand) {
  __shared__ int s_b[SW_T / 32][kSwMost];
  const int lane = threadIdx.x & 31;
  int *sb = s_b[threadIdx.x >> 5];
  const int64_t stride = (int64_t)gridDim.x * SW_T;
  for (int64_t a0 = blockIdx.x * (int64_t)SW_T + threadIdx.x - lane; a0 < MA; a0 += stride) {
    const int64_t a = a0 + lane;
    const int at = a < MA ? off[a] : 0, k = a < MA ? off[a + 1] - at : 0;
    if (k > 1 && k <= kSwInsert)
      for (int i = 1; i < k; ++i) {
        const int2 v = cand[at + i];
        int j = i;
        for (; j > 0; --j) {
          const int2 u = cand[at + j - 1];
          if (u.y <= v.y) break;
          cand[at + j] = u;
        }
        cand[at + j] = v;
      }
    for (unsigned m = __ballot_sync(0xffffffffu, k > kSwInsert); m; m &= m - 1) {
      const int l = __ffs(m) - 1;
      const int la = __shfl_sync(0xffffffffu, at, l), lk = __shfl_sync(0xffffffffu, k, l);
      for (int i = lane; i < lk; i += 32) sb[i] = cand[la + i].y;
      __syncwarp();
      for (int i = lane; i < lk; i += 32) {
        const int b = sb[i];
        int r = 0;  // B ids are distinct
        for (int j = 0; j < lk; ++j) r += sb[j] < b;
        cand[la + r] = make_int2((int)(a0 + l), b);
      }
      __syncwarp();
    }
  }
}

__global__ void k_sw_unpack(const uint64_t *keys, int64_t n, int32_t *cand) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x) {
    const uint64_t k = keys[i];
    cand[2 * i] = (int32_t)(k >> 32);
    cand[2 * i + 1] = (int32_t)(k & 0xFFFFFFFFu);
  }
}

pj_status mbb_sweep(Ctx *ctx, const Dataset *A, const Dataset *B, bool self_join,
                    cudaStream_t s, int64_t *d_count, int32_t **d_cand, int64_t *C) {
  *d_cand = nullptr;
  *C = 0;
  const int64_t MA = A->M, MB = self_join ? 0 : B->M, n = MA + MB;
  pj_status st = PJ_OK;
  auto get = [&](const char *name, size_t bytes) { return ws_get(ctx, name, bytes, &st); };
  auto cand_ws = [&](int64_t c) -> pj_status {
    *d_cand = (int32_t *)get("cand", sizeof(int32_t) * 2 * (size_t)std::max<int64_t>(c, 1));
    return *d_cand ? PJ_OK : st;
  };
  if (n < 2) {  // the device count (read by every later kernel) is zero
    PJ_CK(cudaMemsetAsync(d_count, 0, sizeof(int64_t), s));
    return cand_ws(0);
  }
  if (n > INT32_MAX) return fail(ctx, PJ_ERR_NO_MEMORY, "more than 2^31 meshes to sweep");
  const float *aA = A->d_aabb, *aB = self_join ? nullptr : B->d_aabb;
  const int grid = std::min(blocks_for(n, SW_T), ctx->num_sms * 16);
  // cleared together: bucket counts, words, pairs per mesh of A
  int *hist = (int *)get("sw_counts", 4 * ((size_t)kSwBuckets + (size_t)MA + 1) + 8 * SW_WORDS);
  int *off = (int *)get("sw_off", 4 * ((size_t)kSwBuckets + 1));
  int *rank = (int *)get("sw_rank", 4 * (size_t)n);
  int *longs = (int *)get("sw_long", 4 * (size_t)n);
  int *offA = (int *)get("sw_offsets", 4 * ((size_t)MA + 1));
  float4 *sb = (float4 *)get("sw_boxes", 32 * (size_t)n);
  if (!hist || !off || !rank || !longs || !offA || !sb) return st;
  unsigned long long *words = (unsigned long long *)(hist + kSwBuckets);
  int *cnt = (int *)(words + SW_WORDS);
  size_t tb = 0;
  PJ_CK(cub::DeviceScan::ExclusiveSum(nullptr, tb, cnt, offA, (int)(MA + 1), s));
  void *tmp = get("sw_scan", tb);
  if (!tmp) return st;
  // room for the list: what it held before, at first four pairs a box
  int64_t cap = std::max<int64_t>(4 * n, (int64_t)(cur_exec(ctx)->ws["sw_list"].cap / 8));
  unsigned long long *h = (unsigned long long *)cur_exec(ctx)->h_pinned;
  uint64_t *keys = nullptr;
  bool placed = false;
  for (;;) {
    keys = (uint64_t *)get("sw_list", 8 * (size_t)cap);
    if (!keys) return st;
    if (!placed) {
      PJ_CK(cudaMemsetAsync(hist, 0, 4 * ((size_t)kSwBuckets + (size_t)MA + 1) + 8 * SW_WORDS, s));
      k_sw_rank<<<grid, SW_T, 0, s>>>(aA, MA, aB, n, hist, rank);
      k_sw_offsets<<<1, 1024, 0, s>>>(hist, off);
      k_sw_place<<<grid, SW_T, 0, s>>>(aA, MA, aB, n, off, rank, sb);
      ctx->launches += 3;
      placed = true;
    } else {
      PJ_CK(cudaMemsetAsync(words, 0, 8 * SW_WORDS + 4 * ((size_t)MA + 1), s));
    }
    const SwOut o{keys, cap, cnt, words};
    const int pgrid = (int)std::min<int64_t>((n + SW_T / 32 - 1) / (SW_T / 32),
                                             (int64_t)ctx->num_sms * 8);
    k_sw_short<<<pgrid, SW_T, 0, s>>>(sb, n, MA, self_join ? 1 : 0, o, longs);
    k_sw_long<<<ctx->num_sms * 8, SW_T, 0, s>>>(sb, MA, self_join ? 1 : 0, o, longs);
    ctx->launches += 2;
    PJ_CK(cudaGetLastError());
    PJ_CK(cub::DeviceScan::ExclusiveSum(tmp, tb, cnt, offA, (int)(MA + 1), s));
    PJ_CK(cudaMemcpyAsync(d_count, words + SW_PAIRS, 8, cudaMemcpyDeviceToDevice, s));
    PJ_CK(cudaMemcpyAsync(h, words, 8 * SW_WORDS, cudaMemcpyDeviceToHost, s));
    PJ_CK(cudaStreamSynchronize(s));
    if (h[SW_PAIRS] > INT32_MAX) return fail(ctx, PJ_ERR_NO_MEMORY, "more than 2^31 candidate pairs");
    if ((int64_t)h[SW_PAIRS] <= cap) break;
    cap = (int64_t)h[SW_PAIRS];
  }
  const int64_t c = (int64_t)h[SW_PAIRS];
  if ((st = cand_ws(c)) != PJ_OK) return st;
  *C = c;
  if (c == 0) return PJ_OK;
  const int cgrid = std::min(blocks_for(c, SW_T), ctx->num_sms * 16);
  if (!h[SW_MANY]) {
    k_sw_scatter<<<cgrid, SW_T, 0, s>>>(keys, c, offA, cnt, (int2 *)*d_cand);
    k_sw_order<<<std::min(blocks_for(MA, SW_T), ctx->num_sms * 6), SW_T, 0, s>>>(
        offA, MA, (int2 *)*d_cand);
    ctx->launches += 2;
  } else {
    uint64_t *q1 = (uint64_t *)get("sw_q1", 8 * (size_t)c);
    if (!q1) return st;
    size_t tb2 = 0;
    PJ_CK(cub::DeviceRadixSort::SortKeys(nullptr, tb2, keys, q1, (int)c, 0, 63, s));
    void *tmp2 = get("sw_sort", tb2);
    if (!tmp2) return st;
    PJ_CK(cub::DeviceRadixSort::SortKeys(tmp2, tb2, keys, q1, (int)c, 0, 63, s));
    k_sw_unpack<<<cgrid, SW_T, 0, s>>>(q1, c, *d_cand);
    ctx->launches += 1;
  }
  PJ_CK(cudaGetLastError());
  return PJ_OK;
}

}  // namespace pj
