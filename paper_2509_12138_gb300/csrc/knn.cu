// a9 (first half): exact k nearest neighbours of the isosurface points on a
// uniform grid.  Their distances give the plain initial scale (mean 3-NN
// distance) and, with k = 16, the geometry features of the learned initialiser.
//
// Build: count points per cell (each point keeping its rank in its cell),
// exclusive scan, scatter the points (as float4 with the index in .w) into cell
// order.  Query: one thread per point, taken in cell order so that a warp's
// points search the same cells; the cells of one (z, y) row are consecutive, so
// a run of them is one range of the sorted points.  Cubes of cells of growing
// radius R are searched, rows that lie farther than the k-th best skipped,
// until the k-th best distance is smaller than the distance from the point to
// the outside of the cube.  A first search keeps the k smallest squared
// distances alone, in registers (two min / max per slot and candidate, where
// (distance, index) pairs would cost compares and selects); a second one over
// the same rows collects the points within the k-th distance, and one sort
// orders them.  Ties in distance are broken by the smaller index, so the result
// is unique.
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include "common.cuh"

using namespace gs;

namespace {

__host__ __device__ inline size_t a256(size_t x) { return (x + 255) & ~(size_t)255; }

struct Grid {
  float lo[3];
  float h, inv_h;
  int dim[3];
  float slack;  // bounds the rounding of cell boundaries and of the points' cells
};

struct KnnWs {
  size_t start, rank, scan, sorted, total;
};
KnnWs knn_ws(int64_t n, int64_t cells) {
  KnnWs L;
  size_t o = 0;
  L.start = o; o += a256(sizeof(uint32_t) * (size_t)(cells + 1));
  L.rank = o; o += a256(sizeof(uint32_t) * (size_t)(n > 0 ? n : 1));
  L.scan = o; o += a256(gs_scan_ws_bytes(cells));
  L.sorted = o; o += a256(sizeof(float4) * (size_t)(n > 0 ? n : 1));
  L.total = o;
  return L;
}

__device__ __forceinline__ int cell_coord(float x, float lo, float inv_h, int dim) {
  int c = (int)floorf((x - lo) * inv_h);
  return min(max(c, 0), dim - 1);
}

__device__ __forceinline__ int64_t cell_of(const Grid& g, float x, float y, float z) {
  const int cx = cell_coord(x, g.lo[0], g.inv_h, g.dim[0]);
  const int cy = cell_coord(y, g.lo[1], g.inv_h, g.dim[1]);
  const int cz = cell_coord(z, g.lo[2], g.inv_h, g.dim[2]);
  return ((int64_t)cz * g.dim[1] + cy) * g.dim[0] + cx;
}

__global__ void k_cell_count(const float* __restrict__ pts, int64_t n, Grid g, uint32_t* __restrict__ count,
                             uint32_t* __restrict__ rank) {
  gs_wait_previous();
  int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i >= n) return;
  rank[i] = atomicAdd(&count[cell_of(g, pts[3 * i], pts[3 * i + 1], pts[3 * i + 2])], 1u);
}

__global__ void k_cell_scatter(const float* __restrict__ pts, int64_t n, Grid g, const uint32_t* __restrict__ start,
                               const uint32_t* __restrict__ rank, float4* __restrict__ sorted) {
  gs_wait_previous();
  int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i >= n) return;
  float x = pts[3 * i], y = pts[3 * i + 1], z = pts[3 * i + 2];
  sorted[start[cell_of(g, x, y, z)] + rank[i]] = make_float4(x, y, z, __int_as_float((int)i));
}

// squared distance, one rounding order for both searches
__device__ __forceinline__ float dist2(float4 a, float4 b) {
  const float ex = a.x - b.x, ey = a.y - b.y, ez = a.z - b.z;
  return __fmaf_rn(ez, ez, __fmaf_rn(ey, ey, __fmul_rn(ex, ex)));
}

// distance along one axis from p to the points held by cells c0 .. c1 (0 inside).  Points from outside the grid are
// held by its outermost cells, so those reach on without end.
__device__ __forceinline__ float axis_gap(float p, float lo, const Grid& g, int c0, int c1, int dim) {
  const float below = c0 > 0 ? lo + (float)c0 * g.h - p : 0.f;
  const float above = c1 < dim - 1 ? p - (lo + (float)(c1 + 1) * g.h) : 0.f;
  return fmaxf(0.f, fmaxf(below, above) - g.slack);
}

// Calls f(point) for the points of the cells that cube radius R adds to radius
// R - 1 (all of the cube when `whole`), except runs of cells farther from p
// than the squared distance limit().
template <typename F, typename L>
__device__ __forceinline__ void visit(const Grid& g, const uint32_t* __restrict__ start,
                                      const float4* __restrict__ sorted, const int* c, const float* p, int R,
                                      bool whole, L limit, F f) {
  auto run = [&](int64_t row, float d2yz, int xa, int xb) {
    xa = max(xa, 0);
    xb = min(xb, g.dim[0] - 1);
    if (xa > xb) return;
    const float gx = axis_gap(p[0], g.lo[0], g, xa, xb, g.dim[0]);
    if ((d2yz + gx * gx) * 0.999f > limit()) return;
    const uint32_t e = start[row + xb + 1];
    for (uint32_t q = start[row + xa]; q < e; ++q) f(sorted[q]);
  };
  for (int dz = -R; dz <= R; ++dz) {
    const int z = c[2] + dz;
    if (z < 0 || z >= g.dim[2]) continue;
    const float gz = axis_gap(p[2], g.lo[2], g, z, z, g.dim[2]);
    for (int dy = -R; dy <= R; ++dy) {
      const int y = c[1] + dy;
      if (y < 0 || y >= g.dim[1]) continue;
      const float gy = axis_gap(p[1], g.lo[1], g, y, y, g.dim[1]);
      const float d2 = gz * gz + gy * gy;
      const int64_t row = ((int64_t)z * g.dim[1] + y) * g.dim[0];
      if (whole || dz == -R || dz == R || dy == -R || dy == R) {
        run(row, d2, c[0] - R, c[0] + R);
      } else {
        run(row, d2, c[0] - R, c[0] - R);
        run(row, d2, c[0] + R, c[0] + R);
      }
    }
  }
}

// Bound by instruction issue (59% of cycles) with 12 of 32 lanes active, the
// warp's points' rows ending at different lengths.  1M points of an interface, k
// = 16: 1721 us with sorted (distance, index) insertions, cells visited one by
// one and points in input order, 673 us.
constexpr int KNN_T = 128;
template <int K>
__global__ void __launch_bounds__(KNN_T) k_knn_query(int64_t n, Grid g, const uint32_t* __restrict__ start,
                                                     const float4* __restrict__ sorted, int vec,
                                                     int* __restrict__ out_idx, float* __restrict__ out_dist) {
  gs_wait_previous();
  __shared__ unsigned long long s_best[K][KNN_T];
  const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (t >= n) return;
  const float4 me = sorted[t];
  const int i = __float_as_int(me.w);
  const float p[3] = {me.x, me.y, me.z};
  int c[3];
  #pragma unroll
  for (int a = 0; a < 3; ++a) c[a] = cell_coord(p[a], g.lo[a], g.inv_h, g.dim[a]);
  float b[K];  // the K smallest squared distances so far, ascending
  #pragma unroll
  for (int q = 0; q < K; ++q) b[q] = INFINITY;
  auto kth = [&]() { return b[K - 1]; };
  const int maxdim = max(g.dim[0], max(g.dim[1], g.dim[2]));
  int R = 1;
  for (;; ++R) {
    visit(g, start, sorted, c, p, R, R == 1, kth, [&](float4 o) {
      const float d = dist2(o, me);
      if (d < b[K - 1] && __float_as_int(o.w) != i) {
        #pragma unroll
        for (int q = K - 1; q > 0; --q) b[q] = fminf(b[q], fmaxf(b[q - 1], d));
        b[0] = fminf(b[0], d);
      }
    });
    // distance from p to the outside of the searched cube of cells
    float guard = INFINITY;
    bool whole = true;
    #pragma unroll
    for (int a = 0; a < 3; ++a) {
      int lo = c[a] - R, hi = c[a] + R;
      if (lo > 0) guard = fminf(guard, p[a] - (g.lo[a] + lo * g.h));
      if (hi < g.dim[a] - 1) guard = fminf(guard, (g.lo[a] + (hi + 1) * g.h) - p[a]);
      whole = whole && lo <= 0 && hi >= g.dim[a] - 1;
    }
    // the k-th best must be strictly inside: a point outside the cube is at least `guard` away
    if (whole || R >= maxdim || b[K - 1] < guard * guard * 0.999f) break;
  }
  // the points within the k-th distance: `below` nearer ones, and the smallest indices at it in the other slots
  const float last = b[K - 1];
  int below = 0;
  #pragma unroll
  for (int q = 0; q < K; ++q) below += b[q] < last ? 1 : 0;
  #pragma unroll
  for (int q = 0; q < K; ++q) s_best[q][threadIdx.x] = ~0ull;
  int n1 = 0, n2 = 0;
  visit(g, start, sorted, c, p, R, true, kth, [&](float4 o) {
    const float d = dist2(o, me);
    const int j = __float_as_int(o.w);
    if (!(d <= last) || !(d < INFINITY) || j == i) return;  // (a distance past the float range is no neighbour's)
    const unsigned long long key = ((unsigned long long)__float_as_uint(d) << 32) | (uint32_t)j;
    if (d < last) {
      if (n1 < K) s_best[n1++][threadIdx.x] = key;
    } else if (below + n2 < K) {
      s_best[below + n2++][threadIdx.x] = key;
    } else {  // more ties than slots: replace the largest index held
      int w = below;
      for (int q = below + 1; q < K; ++q)
        if (s_best[q][threadIdx.x] > s_best[w][threadIdx.x]) w = q;
      if (w < K && key < s_best[w][threadIdx.x]) s_best[w][threadIdx.x] = key;
    }
  });
  // ascending (distance, index): odd-even transposition for K = 3, a bitonic network otherwise
  unsigned long long v[K];
  #pragma unroll
  for (int q = 0; q < K; ++q) v[q] = s_best[q][threadIdx.x];
  auto order = [&](unsigned long long& x, unsigned long long& y) {
    const bool sw = y < x;
    const unsigned long long lo = sw ? y : x, hi = sw ? x : y;
    x = lo; y = hi;
  };
  if ((K & (K - 1)) != 0) {
    #pragma unroll
    for (int r = 0; r < K; ++r)
      #pragma unroll
      for (int q = r & 1; q + 1 < K; q += 2) order(v[q], v[q + 1]);
  } else {
    #pragma unroll
    for (int k = 2; k <= K; k *= 2)
      #pragma unroll
      for (int j = k / 2; j > 0; j /= 2)
        #pragma unroll
        for (int q = 0; q < K; ++q) {
          const int o = q ^ j;
          if (o > q) {
            if ((q & k) == 0) order(v[q], v[o]); else order(v[o], v[q]);
          }
        }
  }
  int ri[K];
  float rd[K];
  #pragma unroll
  for (int q = 0; q < K; ++q) {
    const bool ok = v[q] != ~0ull;
    ri[q] = ok ? (int)(uint32_t)v[q] : -1;
    rd[q] = ok ? sqrtf(__uint_as_float((uint32_t)(v[q] >> 32))) : INFINITY;
  }
  int* oi = out_idx + (int64_t)i * K;
  float* od = out_dist + (int64_t)i * K;
  if (K % 4 == 0 && vec) {
    #pragma unroll
    for (int q = 0; q + 3 < K; q += 4) {
      reinterpret_cast<int4*>(oi)[q / 4] = make_int4(ri[q], ri[q + 1], ri[q + 2], ri[q + 3]);
      reinterpret_cast<float4*>(od)[q / 4] = make_float4(rd[q], rd[q + 1], rd[q + 2], rd[q + 3]);
    }
  } else {
    #pragma unroll
    for (int q = 0; q < K; ++q) { oi[q] = ri[q]; od[q] = rd[q]; }
  }
}

}  // namespace

GS_API size_t gs_knn_workspace_size(int64_t n, const int32_t* grid_dims) {
  if (n < 0 || !grid_dims || grid_dims[0] < 1 || grid_dims[1] < 1 || grid_dims[2] < 1) return 0;
  int64_t cells = (int64_t)grid_dims[0] * grid_dims[1] * grid_dims[2];
  return knn_ws(n, cells).total;
}

GS_API int gs_knn(const float* points, int64_t n, int k, const float* grid_lo, float cell_size,
                  const int32_t* grid_dims, void* workspace, size_t workspace_bytes, int32_t* idx, float* dist,
                  gs_stream_t stream) {
  GS_RANGE("gs_knn");
  if (!points || !idx || !dist || !grid_lo || !grid_dims || !workspace || n < 0 || !(cell_size > 0.f) ||
      !(k == 3 || k == 8 || k == 16))
    return GS_ERR_INVALID;
  Grid g;
  for (int a = 0; a < 3; ++a) {
    if (grid_dims[a] < 1) return GS_ERR_INVALID;
    g.lo[a] = grid_lo[a];
    g.dim[a] = grid_dims[a];
  }
  g.h = cell_size;
  g.inv_h = 1.0f / cell_size;
  g.slack = 0.f;
  for (int a = 0; a < 3; ++a) g.slack = fmaxf(g.slack, 1e-6f * (fabsf(g.lo[a]) + (float)g.dim[a] * cell_size));
  int64_t cells = (int64_t)g.dim[0] * g.dim[1] * g.dim[2];
  if (cells >= (int64_t)UINT32_MAX) return GS_ERR_INVALID;
  KnnWs L = knn_ws(n, cells);
  if (workspace_bytes < L.total || ((uintptr_t)workspace & 255u)) return GS_ERR_INVALID;
  if (n == 0) return GS_OK;
  cudaStream_t s = (cudaStream_t)stream;
  char* ws = (char*)workspace;
  uint32_t* start = (uint32_t*)(ws + L.start);
  uint32_t* rank = (uint32_t*)(ws + L.rank);
  float4* sorted = (float4*)(ws + L.sorted);
  if (cudaMemsetAsync(start, 0, sizeof(uint32_t) * cells, s) != cudaSuccess) return GS_ERR_CUDA;
  unsigned nb = (unsigned)((n + 255) / 256);
  gs_launch(k_cell_count, nb, 256, 0, s, points, n, g, start, rank);
  // start[c] = exclusive prefix (in place); start[cells] = n
  int r = gs_scan_u32(start, start, cells, ws + L.scan, start + cells, s);
  if (r != GS_OK) return r;
  gs_launch(k_cell_scatter, nb, 256, 0, s, points, n, g, start, rank, sorted);
  unsigned qb = (unsigned)((n + KNN_T - 1) / KNN_T);
  const int vec = (((uintptr_t)idx | (uintptr_t)dist) & 15u) == 0;
#define GS_KQ(K) gs_launch(k_knn_query<K>, qb, KNN_T, 0, s, n, g, start, sorted, vec, idx, dist)
  switch (k) {
    case 3: GS_KQ(3); break;
    case 8: GS_KQ(8); break;
    default: GS_KQ(16); break;
  }
#undef GS_KQ
  return gs_check_launch();
}
