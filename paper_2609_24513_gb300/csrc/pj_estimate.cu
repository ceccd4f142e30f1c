// Selectivity estimate of a join on the device (paper Sec. 3.5, "Result
// Materialization"): the expected number of intersecting object pairs, from
// per-cell statistics of a regular grid laid over both datasets.  It sizes
// the deduplicating hashmap of the dataset-level join (pj_dataset_join).
//
// Per cell and dataset k: N_k objects whose closed box touches the cell, S_k
// their mean box side (the three extents averaged), VolRatio_k their mean
// mesh-to-box volume ratio.  Two objects are treated as cubes of the mean
// sides; their centres fall in the interaction volume (S_1 + S_2 + eps)^3
// (the Minkowski sum of the two cubes) with probability P_base = V_int /
// V_cell; the shape factor (sqrt(VolRatio_1 VolRatio_2))^gamma discounts
// boxes that are mostly empty; P = min(P_base F_shape, 1), E_i = N_1 N_2 P,
// E_final = sum of E_i over the cells.
//
// Readings (the paper leaves them open): lengths in units of the grid's full
// extent (coordinates / (2^18 - 1)); the grid spans the box of both datasets
// in G^3 equal cells; "touches" is closed; a mesh's volume is the
// divergence-theorem sum |sum det[a, b, c]| / 6 after shifting the mesh by its
// first vertex (summed exactly, then rounded to float64).
#include <algorithm>
#include <cmath>

#include "pj_internal.cuh"

namespace pj {

constexpr double kQ = 262143.0;  // 2^18 - 1

// Six times the signed volume of each mesh: sum over its triangles of
// (a - p0) . ((b - p0) x (c - p0)), p0 its first vertex, as an exact integer.
//
// What bounds it: the index and vertex reads (12 B a triangle, and 12 B a
// vertex once the caches have merged its six uses).  Three choices follow.
//   - Integer arithmetic.  Coordinates are integers below 2^18, so a term is
//     exact in 64 bits (below 2^57); this GPU issues few FP64 operations per
//     cycle, and the ~23 a term takes in FP64 cost more than its reads.  A
//     term is added as its low 32 bits and its high part (low: at most 2^31
//     terms of 32 bits, high: 2^31 terms of 26 bits), so no sum can overflow
//     however the surface winds, and the result does not depend on the order.
//   - Work split by triangles, kVolTris per warp, not by meshes: a mesh may
//     hold 12 triangles or 50,000, and a warp per mesh left the GPU waiting
//     for the longest (and had one triangle's dependent loads in flight).
//   - Four triangles of a lane in flight, the next four's indices loaded
//     before they are summed, and the first mesh found by 32 probes a step
//     (278 us with 512 triangles a warp, a binary search and no such overlap:
//     the loads' latency, not the arithmetic, was waited for; 2,048 triangles
//     a warp measured the same as 1,024).
// Measured on 3,000 nuclei and 150 vessels (42.6 M triangles, 765 MB): 190 us
// (4.0 TB/s) against 6,162 us for a warp per mesh in FP64.
constexpr int kVolTris = 1024;

struct VolSide {
  const float *xyz;
  const int32_t *tris;
  const int64_t *voff, *toff;
  int64_t M, F, warps;           // warps: kVolTris triangles each
  unsigned long long *acc;       // 2 per mesh: low and high parts
};

// an integer-valued float below 2^18 as an integer, offset by a constant
// that cancels in differences (an addition; the conversion instruction
// issues at a quarter of its rate)
__device__ __forceinline__ int coord_bits(float x) { return __float_as_int(x + 8388608.f); }

__global__ void __launch_bounds__(256) k_mesh_volume(VolSide A, VolSide B) {
  const int lane = threadIdx.x & 31;
  int64_t w = blockIdx.x * (int64_t)(blockDim.x / 32) + (threadIdx.x >> 5);
  if (w >= A.warps + B.warps) return;
  const VolSide S = w < A.warps ? A : B;
  if (w >= A.warps) w -= A.warps;
  const int64_t t0 = w * kVolTris, t1 = min(t0 + kVolTris, S.F);
  int64_t m = warp_mesh_of(S.toff, S.M, t0, lane);
  for (int64_t f0 = t0; f0 < t1; ++m) {
    const int64_t f1 = min(S.toff[m + 1], t1);
    const float *p0 = S.xyz + 3 * S.voff[m];
    const int ox = coord_bits(p0[0]), oy = coord_bits(p0[1]), oz = coord_bits(p0[2]);
    unsigned long long s_lo = 0;
    long long s_hi = 0;
    int32_t id[4][3];
    auto load_ids = [&](int64_t f) {
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        // past the end: the last triangle again, not added
        const int32_t *q = S.tris + 3 * min(f + 32 * u, f1 - 1);
#pragma unroll
        for (int k = 0; k < 3; ++k) id[u][k] = q[k];
      }
    };
    load_ids(f0 + lane);
    for (int64_t f = f0 + lane; f < f1; f += 4 * 32) {
      float v[4][9];
#pragma unroll
      for (int u = 0; u < 4; ++u)
#pragma unroll
        for (int k = 0; k < 3; ++k) {
          const float *q = S.xyz + 3 * (int64_t)id[u][k];
          v[u][3 * k] = q[0];
          v[u][3 * k + 1] = q[1];
          v[u][3 * k + 2] = q[2];
        }
      if (f + 4 * 32 < f1) load_ids(f + 4 * 32);
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        if (f + 32 * u >= f1) break;
        const int ax = coord_bits(v[u][0]) - ox, ay = coord_bits(v[u][1]) - oy;
        const int az = coord_bits(v[u][2]) - oz, bx = coord_bits(v[u][3]) - ox;
        const int by = coord_bits(v[u][4]) - oy, bz = coord_bits(v[u][5]) - oz;
        const int cx = coord_bits(v[u][6]) - ox, cy = coord_bits(v[u][7]) - oy;
        const int cz = coord_bits(v[u][8]) - oz;
        const long long d = ax * ((long long)by * cz - (long long)bz * cy) +
                            ay * ((long long)bz * cx - (long long)bx * cz) +
                            az * ((long long)bx * cy - (long long)by * cx);
        s_lo += (unsigned)d;
        s_hi += d >> 32;
      }
    }
    for (int o = 16; o > 0; o >>= 1) {
      s_lo += __shfl_xor_sync(0xffffffffu, s_lo, o);
      s_hi += __shfl_xor_sync(0xffffffffu, s_hi, o);
    }
    if (lane == 0) {
      atomicAdd(S.acc + 2 * m, s_lo);
      atomicAdd(S.acc + 2 * m + 1, (unsigned long long)s_hi);
    }
    f0 = f1;
  }
}

// |hi 2^32 + lo| / 6, the sum rounded once
__device__ __forceinline__ double volume_of(const unsigned long long *acc) {
  const long long hi = (long long)acc[1] + (long long)(acc[0] >> 32);
  return fabs((double)hi * 4294967296.0 + (double)(acc[0] & 0xffffffffull)) / 6.0;
}

struct Grid {
  double g0[3], cw[3];
  int G;
};

struct StatSide {
  const float *aabb;
  const unsigned long long *acc;
  int64_t M;
  unsigned long long *N;
  double *S, *R;
};

// Every cell a mesh's closed box touches gets N += 1, S += the mean box side,
// R += the volume ratio.  A block takes kStatMeshes meshes: one thread per
// mesh works out its cells and values (some twenty FP64 divisions; by every
// lane of a warp per mesh they took most of the kernel, 43 us), then a warp
// per mesh spreads the cells over its lanes (a vessel touches hundreds, and a
// thread per mesh issued their atomics one after another).  16 us against
// 83 us for a thread per mesh, on the 3,150 meshes above.
constexpr int kStatMeshes = 16, kStatT = 256;

__global__ void __launch_bounds__(kStatT) k_cell_stats(StatSide A, StatSide B, Grid g) {
  __shared__ int s_i0[kStatMeshes][3], s_n[kStatMeshes][3];
  __shared__ double s_side[kStatMeshes], s_ratio[kStatMeshes];
  const int64_t m0 = blockIdx.x * (int64_t)kStatMeshes;
  if (threadIdx.x < kStatMeshes && m0 + threadIdx.x < A.M + B.M) {
    int64_t m = m0 + threadIdx.x;
    const StatSide &D = m < A.M ? A : B;
    if (m >= A.M) m -= A.M;
    double ext[3];
    for (int d = 0; d < 3; ++d) {
      const double lo = D.aabb[6 * m + d] / kQ, hi = D.aabb[6 * m + 3 + d] / kQ;
      ext[d] = hi - lo;
      const int i0 = (int)fmin(fmax(floor((lo - g.g0[d]) / g.cw[d]), 0.0), (double)(g.G - 1));
      const int i1 = (int)fmin(fmax(floor((hi - g.g0[d]) / g.cw[d]), 0.0), (double)(g.G - 1));
      s_i0[threadIdx.x][d] = i0;
      s_n[threadIdx.x][d] = i1 - i0 + 1;
    }
    const double box = ext[0] * ext[1] * ext[2];
    s_side[threadIdx.x] = (ext[0] + ext[1] + ext[2]) / 3.0;
    s_ratio[threadIdx.x] =
        box > 0.0 ? volume_of(D.acc + 2 * m) / (kQ * kQ * kQ) / box : 0.0;
  }
  __syncthreads();
  const int lane = threadIdx.x & 31;
  for (int k = threadIdx.x >> 5; k < kStatMeshes && m0 + k < A.M + B.M; k += kStatT / 32) {
    const StatSide &D = m0 + k < A.M ? A : B;
    const int ny = s_n[k][1], nz = s_n[k][2], cells = s_n[k][0] * ny * nz;  // at most 256^3
    for (int i = lane; i < cells; i += 32) {
      const int yz = i / nz, x = s_i0[k][0] + yz / ny, y = s_i0[k][1] + yz % ny;
      const int64_t c = ((int64_t)x * g.G + y) * g.G + s_i0[k][2] + i % nz;
      atomicAdd(D.N + c, 1ull);
      atomicAdd(D.S + c, s_side[k]);
      atomicAdd(D.R + c, s_ratio[k]);
    }
  }
}

// per cell: E_i = N_1 N_2 min(P_base F_shape, 1); their sum and the number of
// cells holding objects of both datasets
__global__ void k_cell_estimate(const unsigned long long *N1, const double *S1, const double *R1,
                                const unsigned long long *N2, const double *S2, const double *R2,
                                int64_t cells, double v_cell, double eps, double gamma,
                                double *E, double *sum, unsigned long long *occupied) {
  double acc = 0.0;
  unsigned long long occ = 0;
  for (int64_t c = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; c < cells;
       c += (int64_t)gridDim.x * blockDim.x) {
    double e = 0.0;
    if (N1[c] > 0 && N2[c] > 0) {
      const double n1 = (double)N1[c], n2 = (double)N2[c];
      const double m1 = S1[c] / n1, m2 = S2[c] / n2, r1 = R1[c] / n1, r2 = R2[c] / n2;
      const double s = m1 + m2 + eps;
      const double p_base = s * s * s / v_cell;
      const double f_shape = pow(sqrt(r1 * r2), gamma);
      e = n1 * n2 * fmin(p_base * f_shape, 1.0);
      occ += 1;
    }
    if (E) E[c] = e;
    acc += e;
  }
  for (int o = 16; o > 0; o >>= 1) {
    acc += __shfl_xor_sync(0xffffffffu, acc, o);
    occ += __shfl_xor_sync(0xffffffffu, occ, o);
  }
  if ((threadIdx.x & 31) == 0) {
    atomicAdd(sum, acc);
    atomicAdd(occupied, occ);
  }
}

pj_status run_estimate(Ctx *ctx, Dataset *A, Dataset *B, int G, double *cells_out,
                       pj_estimate *out, cudaStream_t s) {
  if (G <= 0) G = 16;
  if (G > 256) return fail(ctx, PJ_ERR_INVALID_ARG, "grid must be at most 256 cells per axis");
  if (A->M == 0 || B->M == 0) {
    memset(out, 0, sizeof(*out));
    out->grid = G;
    return PJ_OK;
  }
  // the grid over both datasets' boxes (host copies of the mesh boxes)
  Grid g;
  g.G = G;
  for (int d = 0; d < 3; ++d) {
    float flo = 3e38f, fhi = -3e38f;
    for (const Dataset *D : {A, B})
      for (int64_t m = 0; m < D->M; ++m) {
        flo = std::min(flo, D->h_aabb[6 * m + d]);
        fhi = std::max(fhi, D->h_aabb[6 * m + 3 + d]);
      }
    const double lo = flo / kQ, hi = fhi / kQ;
    g.g0[d] = lo;
    g.cw[d] = std::max(hi - lo, 1.0 / kQ) / G;
  }
  const int64_t cells = (int64_t)G * G * G;
  pj_status st;
  // one buffer: the two sides' volume sums, then per dataset N, S, R, then
  // E, sum, occupied.  A dataset against itself is measured once.
  const bool same = A == B;
  const int64_t MB = same ? 0 : B->M;
  const size_t words = 2 * ((size_t)A->M + (size_t)MB) + 8 * (size_t)cells + 2;
  unsigned long long *buf = (unsigned long long *)ws_get(ctx, "estimate", 8 * words, &st);
  if (!buf) return st;
  unsigned long long *accA = buf, *accB = accA + 2 * A->M;
  unsigned long long *N1 = accB + 2 * MB;
  double *S1 = (double *)(N1 + cells), *R1 = S1 + cells;
  unsigned long long *N2 = (unsigned long long *)(R1 + cells);
  double *S2 = (double *)(N2 + cells), *R2 = S2 + cells;
  double *E = R2 + cells, *sum = E + cells;
  unsigned long long *occ = (unsigned long long *)(sum + 1);
  cudaEvent_t *ev = cur_exec(ctx)->ev;
  PJ_CK(cudaEventRecord(ev[0], s));
  PJ_CK(cudaMemsetAsync(buf, 0, 8 * words, s));
  auto vol_side = [](const Dataset *D, unsigned long long *acc) {
    return VolSide{D->d_xyz, D->d_tris, D->d_voff, D->d_toff, D->M, D->F,
                   (D->F + kVolTris - 1) / kVolTris, acc};
  };
  VolSide va = vol_side(A, accA), vb = vol_side(B, accB);
  if (same) vb.warps = 0;
  k_mesh_volume<<<blocks_for(va.warps + vb.warps, 8), 256, 0, s>>>(va, vb);
  const StatSide sa{A->d_aabb, accA, A->M, N1, S1, R1}, sb{B->d_aabb, accB, MB, N2, S2, R2};
  k_cell_stats<<<blocks_for(A->M + MB, kStatMeshes), kStatT, 0, s>>>(sa, sb, g);
  if (same) {
    N2 = N1;
    S2 = S1;
    R2 = R1;
  }
  const double v_cell = g.cw[0] * g.cw[1] * g.cw[2];
  // small blocks: the cells of an ordinary grid (4,096) then reach most SMs,
  // whose few FP64 units evaluate the power
  k_cell_estimate<<<(int)std::min<int64_t>(blocks_for(cells, 32), ctx->num_sms * 32), 32, 0, s>>>(
      N1, S1, R1, N2, S2, R2, cells, v_cell, 1e-3, 0.8, E, sum, occ);
  ctx->launches += 3;
  PJ_CK(cudaGetLastError());
  PJ_CK(cudaEventRecord(ev[3], s));
  double h[2];
  PJ_CK(cudaMemcpyAsync(h, sum, 16, cudaMemcpyDeviceToHost, s));
  if (cells_out) PJ_CK(cudaMemcpyAsync(cells_out, E, 8 * (size_t)cells, cudaMemcpyDeviceToHost, s));
  PJ_CK(cudaStreamSynchronize(s));
  memset(out, 0, sizeof(*out));
  out->e_final = h[0];
  out->slots = h[0] / 0.5;
  unsigned long long o;
  memcpy(&o, &h[1], 8);
  out->cells_occupied = (int64_t)o;
  out->grid = G;
  cudaEventElapsedTime(&out->ms, ev[0], ev[3]);
  return PJ_OK;
}

}  // namespace pj
