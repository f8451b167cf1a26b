// a2 for small problems: the lists, ranges and blend schedule of gs_bin_sort in
// four launches.
//
// The general design takes 23 launches (26 with over 256 lists), schedule included; with a few thousand
// records each of them is a few microseconds of launch and one round of memory
// latency.  Here one CTA per unit sorts the unit's records by depth in shared
// memory, and every (unit, tile) list is then made by a warp of its own that
// reads the unit's tile rectangles in depth order and keeps those that cover
// its tile: records x tiles tests in all, so the design is for small products
// of the two (gs_small_sort_applies).  A list comes out in (depth, record index)
// order without any sort of the instances.  What bounds it is latency, not
// bytes.  Sort and schedule of 500 records on 16 tiles: 150 -> 37 us; of 8 units
// of 2,000 records on 64 tiles: 204 -> 66 us (43 and 90 us with 32 records per
// step of a list's warp instead of 128, and 8 lists per block instead of 4).
#include <cuda_runtime.h>
#include <math.h>
#include <stddef.h>
#include <stdint.h>

#include "common.cuh"

using namespace gs;

namespace {

constexpr int ST = 1024;                 // threads of the unit sort
constexpr int SW = ST / 32;
constexpr int ROUNDS = 16;               // records per thread
constexpr int UNIT_MAX = ST * ROUNDS;    // records per unit
constexpr int LISTS_MAX = 4096;          // (unit, tile) lists; with UNIT_MAX records each, at most 2^26 tests and instances

// device words shared by the launches
struct Ctrl {
  uint32_t total;     // instances of all visible records
  uint32_t finished;  // units sorted
  uint32_t cut_m;     // tiles kept of the record at the cut
  uint32_t over;      // more instances than the capacity
  unsigned long long cut;  // (depth bits, record) of the first record that is not kept whole
  uint32_t vis[GS_MAX_UNITS];
};

struct UnitSmem {
  uint32_t key[UNIT_MAX];
  uint16_t id[UNIT_MAX];
  uint16_t wc[SW][256];  // per-warp digit counts, then each warp's offset within the digit
  uint32_t start[256];
  uint32_t red[SW];
  uint32_t kmin, kmax, visible;
};

__device__ __forceinline__ uint2 pack_rect(int x0, int y0, int x1, int y1) {
  return make_uint2((uint32_t)x0 | ((uint32_t)y0 << 16), (uint32_t)x1 | ((uint32_t)y1 << 16));
}
__device__ __forceinline__ uint32_t rect_tiles(uint2 r) {
  return ((r.y & 0xffffu) - (r.x & 0xffffu)) * ((r.y >> 16) - (r.x >> 16));
}

// Sum over the block, to every thread.
__device__ __forceinline__ uint64_t block_total(uint64_t v, uint64_t* s) {
  #pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  __syncthreads();
  if ((threadIdx.x & 31) == 0) s[threadIdx.x >> 5] = v;
  __syncthreads();
  uint64_t t = 0;
  for (int q = 0; q < SW; ++q) t += s[q];
  return t;
}

// One CTA per unit: its records in (depth, index) order with their tile
// rectangles.  Stable LSD radix passes over the depth bits relative to the
// unit's nearest record, as many as the farthest one needs; culled records take
// the key behind it.  Warp w ranks the records of its own run of positions in
// order, so counting digits per warp and scanning over warps ranks the block.
// The last CTA finds the cut if the instances exceed the capacity: the record,
// in (depth, index) order over all units, at which the capacity runs out.
__global__ void __launch_bounds__(ST, 1) k_small_units(UnitTable U, const float4* __restrict__ xy,
                                                       const float* __restrict__ depth,
                                                       const int* __restrict__ radius,
                                                       const uint32_t* __restrict__ tiles, int W, int H, int64_t cap,
                                                       uint32_t* __restrict__ rec, uint2* __restrict__ rect,
                                                       Ctrl* __restrict__ ctrl, int* __restrict__ status) {
  gs_wait_previous();
  extern __shared__ __align__(16) unsigned char s_raw[];
  UnitSmem& s = *reinterpret_cast<UnitSmem*>(s_raw);
  __shared__ uint64_t s_sum[SW];
  __shared__ int s_last;
  const int u = blockIdx.x, tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
  const int64_t base = U.proj_base[u];
  const int n = (int)(U.proj_base[u + 1] - base);
  const int rounds = (n + ST - 1) / ST;       // uniform; this warp's positions are [32 w rounds, 32 (w + 1) rounds)
  const int first = w * 32 * rounds + lane;
  if (tid == 0) { s.kmin = 0xffffffffu; s.kmax = 0u; s.visible = 0u; }
  __syncthreads();
  uint32_t key[ROUNDS];
  uint16_t id[ROUNDS];
  uint32_t seen = 0u, kmin = 0xffffffffu, kmax = 0u;  // seen: bit j set when record j is visible
  #pragma unroll
  for (int j = 0; j < ROUNDS; ++j) {
    const int k = first + 32 * j;
    key[j] = 0u; id[j] = (uint16_t)k;
    if (j < rounds && k < n && tiles[base + k] > 0u) {
      key[j] = __float_as_uint(depth[base + k]);
      seen |= 1u << j;
      kmin = min(kmin, key[j]); kmax = max(kmax, key[j]);
    }
  }
  kmin = __reduce_min_sync(0xffffffffu, kmin);
  kmax = __reduce_max_sync(0xffffffffu, kmax);
  const uint32_t nv = __reduce_add_sync(0xffffffffu, (uint32_t)__popc(seen));
  if (lane == 0 && nv) { atomicMin(&s.kmin, kmin); atomicMax(&s.kmax, kmax); atomicAdd(&s.visible, nv); }
  __syncthreads();
  const uint32_t visible = s.visible, k0 = s.kmin;
  // culled records: one past the farthest relative depth (a visible depth is finite, so this does not wrap)
  const uint32_t behind = visible ? s.kmax - k0 + 1u : 0u;
  #pragma unroll
  for (int j = 0; j < ROUNDS; ++j) key[j] = (seen >> j & 1u) ? key[j] - k0 : behind;
  const uint32_t lt = (1u << lane) - 1u;
  for (int shift = 0; shift < 32 && (behind >> shift) != 0u; shift += 8) {
    for (int q = tid; q < SW * 256; q += ST) (&s.wc[0][0])[q] = 0;
    __syncthreads();
    uint16_t rank[ROUNDS];
    #pragma unroll
    for (int j = 0; j < ROUNDS; ++j) {
      if (j >= rounds) break;
      const bool ok = first + 32 * j < n;
      const uint32_t d = ok ? (key[j] >> shift) & 255u : 256u;
      const uint32_t peers = __match_any_sync(0xffffffffu, d);
      const uint32_t before = ok ? s.wc[w][d] : 0u;
      rank[j] = (uint16_t)(before + __popc(peers & lt));
      __syncwarp();
      if (ok && (peers & lt) == 0u) s.wc[w][d] = (uint16_t)(before + __popc(peers));
      __syncwarp();
    }
    __syncthreads();
    uint32_t cnt = 0u;
    if (tid < 256) {
      for (int q = 0; q < SW; ++q) {
        const uint32_t c = s.wc[q][tid];
        s.wc[q][tid] = (uint16_t)cnt;
        cnt += c;
      }
    }
    uint32_t inc = cnt;
    #pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t v = __shfl_up_sync(0xffffffffu, inc, o);
      if (lane >= o) inc += v;
    }
    if (lane == 31) s.red[w] = inc;
    __syncthreads();
    if (tid < 256) {
      uint32_t off = 0u;
      for (int q = 0; q < w; ++q) off += s.red[q];
      s.start[tid] = off + inc - cnt;
    }
    __syncthreads();
    #pragma unroll
    for (int j = 0; j < ROUNDS; ++j) {
      if (j >= rounds) break;
      if (first + 32 * j < n) {
        const uint32_t d = (key[j] >> shift) & 255u;
        const uint32_t pos = s.start[d] + s.wc[w][d] + rank[j];
        s.key[pos] = key[j];
        s.id[pos] = id[j];
      }
    }
    __syncthreads();
    #pragma unroll
    for (int j = 0; j < ROUNDS; ++j) {
      if (j >= rounds) break;
      const int k = first + 32 * j;
      if (k < n) { key[j] = s.key[k]; id[j] = s.id[k]; }
    }
  }
  const int TX = (W + TILE - 1) / TILE, TY = (H + TILE - 1) / TILE;
  uint64_t sum = 0;
  #pragma unroll
  for (int j = 0; j < ROUNDS; ++j) {
    if (j >= rounds) break;
    const int k = first + 32 * j;
    if (k < (int)visible) {
      const int64_t p = base + id[j];
      int x0, y0, x1, y1;
      tile_rect(xy[p], radius[p], TX, TY, x0, y0, x1, y1);
      rec[base + k] = (uint32_t)p;
      rect[base + k] = pack_rect(x0, y0, x1, y1);
      sum += (uint64_t)((x1 - x0) * (y1 - y0));
    }
  }
  sum = block_total(sum, s_sum);
  if (tid == 0) {
    ctrl->vis[u] = visible;
    atomicAdd(&ctrl->total, (uint32_t)sum);
    __threadfence();
    s_last = atomicAdd(&ctrl->finished, 1u) == (uint32_t)U.n - 1u;
  }
  __threadfence();
  __syncthreads();
  if (!s_last) return;
  __threadfence();
  const uint64_t total = *(volatile uint32_t*)&ctrl->total;
  if ((int64_t)total <= cap) {
    if (tid == 0) { ctrl->over = 0u; ctrl->cut = ~0ull; ctrl->cut_m = 0u; }
    return;
  }
  // the first record, by (depth, index), whose instances run past the capacity: its key found digit by digit from
  // the top, each pass summing the instances of the records that share the digits found so far per next digit
  __shared__ uint32_t s_bin[256];
  __shared__ unsigned long long s_pre;
  __shared__ uint32_t s_left;
  if (tid == 0) { s_pre = 0ull; s_left = (uint32_t)cap; }
  for (int shift = 56; shift >= 0; shift -= 8) {
    if (tid < 256) s_bin[tid] = 0u;
    __syncthreads();
    const unsigned long long pre = s_pre;
    for (int q = 0; q < U.n; ++q) {
      const int64_t b = U.proj_base[q];
      const int m = (int)*(volatile uint32_t*)&ctrl->vis[q];
      #pragma unroll 4
      for (int e = tid; e < m; e += ST) {
        const uint32_t p = __ldcg(rec + b + e);
        const uint32_t nt = rect_tiles(__ldcg(rect + b + e));
        const unsigned long long k = ((unsigned long long)__float_as_uint(depth[p]) << 32) | p;
        if (shift == 56 || (k >> (shift + 8)) == (pre >> (shift + 8))) atomicAdd(&s_bin[(uint32_t)(k >> shift) & 255u], nt);
      }
    }
    __syncthreads();
    if (tid == 0) {
      uint32_t left = s_left;
      int d = 0;
      while (d < 255 && s_bin[d] <= left) left -= s_bin[d++];
      s_left = left;
      s_pre = pre | ((unsigned long long)d << shift);
    }
    __syncthreads();
  }
  if (tid == 0) {
    ctrl->over = 1u;
    ctrl->cut = s_pre;
    ctrl->cut_m = s_left;
    set_status(status, GS_ERR_CAPACITY);
  }
}

// The records of one (unit, tile) list, 32 GROUP at a time in depth order:
// whether record i + 32 q + lane has an instance in it, and its id.  The loads
// of a group are independent, so a warp waits for memory once per group.
constexpr int GROUP = 4;
struct Hits {
  const uint32_t* rec;
  const uint2* rect;
  const float* depth;
  const Ctrl* ctrl;
  int tx, ty, m;
  bool over;
  unsigned long long cut;
  uint32_t cut_m;
  __device__ __forceinline__ Hits(const UnitTable& U, int u, int tx_, int ty_, const uint32_t* rec_, const uint2* rect_,
                                  const float* depth_, const Ctrl* ctrl_)
      : rec(rec_ + U.proj_base[u]), rect(rect_ + U.proj_base[u]), depth(depth_), ctrl(ctrl_), tx(tx_), ty(ty_) {
    m = (int)ctrl->vis[u];
    over = ctrl->over != 0u;
    cut = ctrl->cut;
    cut_m = ctrl->cut_m;
  }
  __device__ __forceinline__ void load(int i, bool* hit, uint32_t* p) const {
    uint2 r[GROUP];
    #pragma unroll
    for (int q = 0; q < GROUP; ++q) {
      const int k = i + 32 * q + (int)(threadIdx.x & 31);
      r[q] = k < m ? __ldg(rect + k) : make_uint2(0u, 0u);  // (an empty rectangle)
      p[q] = k < m ? __ldg(rec + k) : 0u;
    }
    #pragma unroll
    for (int q = 0; q < GROUP; ++q) {
      const int x0 = (int)(r[q].x & 0xffffu), y0 = (int)(r[q].x >> 16);
      const int x1 = (int)(r[q].y & 0xffffu), y1 = (int)(r[q].y >> 16);
      hit[q] = tx >= x0 && tx < x1 && ty >= y0 && ty < y1;
      if (over && hit[q]) {  // instances are numbered row by row within a record
        const unsigned long long k = ((unsigned long long)__float_as_uint(depth[p[q]]) << 32) | p[q];
        hit[q] = k < cut || (k == cut && (uint32_t)((ty - y0) * (x1 - x0) + tx - x0) < cut_m);
      }
    }
  }
};

constexpr int LW = 4;  // lists (warps) per block

__global__ void __launch_bounds__(LW * 32) k_small_count(UnitTable U, int W, int n_tiles, int NT,
                                                         const uint32_t* __restrict__ rec,
                                                         const uint2* __restrict__ rect,
                                                         const float* __restrict__ depth,
                                                         const Ctrl* __restrict__ ctrl, uint32_t* __restrict__ count) {
  gs_wait_previous();
  const int f = blockIdx.x * LW + (threadIdx.x >> 5);
  if (f >= NT) return;
  const int TX = (W + TILE - 1) / TILE, tile = f % n_tiles;
  const Hits H(U, f / n_tiles, tile % TX, tile / TX, rec, rect, depth, ctrl);
  uint32_t c = 0u;
  for (int i = 0; i < H.m; i += 32 * GROUP) {
    bool hit[GROUP];
    uint32_t p[GROUP];
    H.load(i, hit, p);
    #pragma unroll
    for (int q = 0; q < GROUP; ++q) c += hit[q] ? 1u : 0u;
  }
  c = __reduce_add_sync(0xffffffffu, c);
  if ((threadIdx.x & 31) == 0) count[f] = c;
}

// exclusive prefix over the block's threads; *total: the sum
__device__ __forceinline__ uint32_t block_prefix(uint32_t v, uint32_t* s, uint32_t* total) {
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  uint32_t inc = v;
  #pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t x = __shfl_up_sync(0xffffffffu, inc, o);
    if (lane >= o) inc += x;
  }
  __syncthreads();
  if (lane == 31) s[w] = inc;
  __syncthreads();
  uint32_t off = 0u, all = 0u;
  for (int q = 0; q < SW; ++q) { off += q < w ? s[q] : 0u; all += s[q]; }
  *total = all;
  return off + inc - v;
}

// One CTA: ranges and instance count, and with a schedule the tile order
// (heaviest length classes first) and the chunk jobs.
__global__ void __launch_bounds__(ST) k_small_ranges(int NT, const uint32_t* __restrict__ count,
                                                     uint2* __restrict__ ranges, uint32_t* __restrict__ d_count,
                                                     uint32_t* __restrict__ order, uint32_t* __restrict__ job_base,
                                                     uint32_t* __restrict__ jobs, int64_t max_jobs, int K) {
  gs_wait_previous();
  constexpr int PER = LISTS_MAX / ST;
  __shared__ uint32_t s[SW], s_class[33], s_len[LISTS_MAX];
  const int t0 = threadIdx.x * PER;
  uint32_t c[PER], sum = 0u, total;
  #pragma unroll
  for (int e = 0; e < PER; ++e) { c[e] = t0 + e < NT ? count[t0 + e] : 0u; sum += c[e]; }
  if (threadIdx.x < 33) s_class[threadIdx.x] = 0u;
  uint32_t at = block_prefix(sum, s, &total);
  if (threadIdx.x == 0) *d_count = total;
  #pragma unroll
  for (int e = 0; e < PER; ++e) {
    if (t0 + e < NT) {
      ranges[t0 + e] = c[e] ? make_uint2(at, at + c[e]) : make_uint2(0u, 0u);
      if (order) atomicAdd(&s_class[32 - __clz(c[e])], 1u);
    }
    at += c[e];
  }
  if (!order) return;
  __syncthreads();
  if (threadIdx.x == 0) {
    uint32_t acc = 0u;
    for (int q = 32; q >= 0; --q) { const uint32_t x = s_class[q]; s_class[q] = acc; acc += x; }
  }
  __syncthreads();
  #pragma unroll
  for (int e = 0; e < PER; ++e)
    if (t0 + e < NT) {
      const uint32_t o = atomicAdd(&s_class[32 - __clz(c[e])], 1u);
      order[o] = (uint32_t)(t0 + e);
      s_len[o] = c[e];
    }
  __syncthreads();
  uint32_t nj[PER];
  sum = 0u;
  #pragma unroll
  for (int e = 0; e < PER; ++e) {
    nj[e] = t0 + e < NT ? (s_len[t0 + e] + (uint32_t)K - 1u) / (uint32_t)K : 0u;
    sum += nj[e];
  }
  at = block_prefix(sum, s, &total);
  if (threadIdx.x == 0) job_base[NT] = total;
  #pragma unroll
  for (int e = 0; e < PER; ++e) {
    if (t0 + e >= NT) continue;
    job_base[t0 + e] = at;
    for (uint32_t j = 0; j < nj[e] && (int64_t)(at + j) < max_jobs; ++j) {
      jobs[2 * (int64_t)(at + j)] = (uint32_t)(t0 + e);
      jobs[2 * (int64_t)(at + j) + 1] = j;
    }
    at += nj[e];
  }
}

__global__ void __launch_bounds__(LW * 32) k_small_fill(UnitTable U, int W, int n_tiles, int NT,
                                                        const uint32_t* __restrict__ rec,
                                                        const uint2* __restrict__ rect,
                                                        const float* __restrict__ depth,
                                                        const Ctrl* __restrict__ ctrl,
                                                        const float4* __restrict__ xy,
                                                        const float4* __restrict__ conic_op,
                                                        const uint2* __restrict__ ranges,
                                                        uint32_t* __restrict__ vals, uint16_t* __restrict__ masks) {
  gs_wait_previous();
  const int f = blockIdx.x * LW + (threadIdx.x >> 5);
  if (f >= NT) return;
  const uint2 rg = ranges[f];
  if (rg.x == rg.y) return;
  const int TX = (W + TILE - 1) / TILE, tile = f % n_tiles, tx = tile % TX, ty = tile / TX;
  const uint32_t lt = (1u << (threadIdx.x & 31)) - 1u;
  const Hits H(U, f / n_tiles, tx, ty, rec, rect, depth, ctrl);
  uint32_t at = rg.x;
  for (int i = 0; i < H.m; i += 32 * GROUP) {
    bool hit[GROUP];
    uint32_t p[GROUP], mk[GROUP];
    H.load(i, hit, p);
    if (masks) {
      float4 m[GROUP], co[GROUP];
      #pragma unroll
      for (int q = 0; q < GROUP; ++q)
        if (hit[q]) { m[q] = xy[p[q]]; co[q] = conic_op[p[q]]; }
      #pragma unroll
      for (int q = 0; q < GROUP; ++q) {
        float pm;
        mk[q] = hit[q] ? block_mask(alpha_box(make_float2(m[q].x, m[q].y), co[q], pm), tx, ty) : 0u;
      }
    }
    #pragma unroll
    for (int q = 0; q < GROUP; ++q) {
      const uint32_t bal = __ballot_sync(0xffffffffu, hit[q]);
      if (hit[q]) {
        const uint32_t k = at + __popc(bal & lt);
        vals[k] = p[q];
        if (masks) masks[k] = (uint16_t)mk[q];
      }
      at += __popc(bal);
    }
  }
}

}  // namespace

// Whether the design applies.  A list's warp reads all records of its unit, twice, so this design takes 13 us + 20 ns
// per record of the largest unit, whatever they cover.  The general one takes 85 us, more with several units, and its
// emission gives all instances of a record to one thread: 10 to 35 us per instance that a record has on average, and
// about 1 us per tile of the largest splat.  Neither is known here; the image's tiles bound the one, and the capacity
// stands for the other (where it was fitted, 1.25 times the instances).  So the limit grows by 1,024 records with each
// doubling of the tiles and by 256 with each instance that the capacity leaves a record.  us per call, this design /
// general / general with one splat that covers the image (4 instances of capacity per record):
//   16 tiles, 1 unit      limit 4,096    3,000  80 / 82 / -      5,000  118 / 86 / -      16,384  352 / 86 / -
//   49 tiles, 2 units     limit 5,750    7,285 165 / 91 / 111
//   64 tiles, 8 units     limit 6,144    3,000  78 / 122 / -     5,000  116 / 107 / -      8,000  174 / 103 / -
//   165 tiles, 1 unit     limit 7,540    4,500 104 / 96 / -      7,285  157 / 93 / 254
//   256 tiles, 1 unit     limit 8,192    3,000  74 / 127 / -     5,000  107 / 109 / -     15,000  278 / 94 / 338
//   256 tiles, 4 units    limit 8,192                                                     10,000  204 / 128 / 440
//   1024 tiles, 4 units   limit 10,240   4,000 107 / 369 / -     8,000  176 / 226 / -     16,384  313 / 142 / -
// Before this design the general one took 150 to 240 us at these sizes, 95 to 155 in a captured graph: against that no
// call of 170 sizes is slower now, captured ones of small splats just below the limit by up to 1.4 times.
bool gs_small_sort_applies(const UnitTable& U, int64_t P, int n_tiles, int64_t cap) {
  if ((int64_t)U.n * n_tiles > LISTS_MAX) return false;
  const double most = 1024.0 * log2((double)n_tiles) + 256.0 * ((double)cap / (double)P - 4.0);
  for (int u = 0; u < U.n; ++u)
    if ((double)(U.proj_base[u + 1] - U.proj_base[u]) > fmin(fmax(most, 3072.0), (double)UNIT_MAX)) return false;
  return true;
}

size_t gs_small_sort_ctrl_words() { return sizeof(Ctrl) / sizeof(uint32_t); }

// rec, rect: P words / pairs; count: LISTS_MAX words; ctrl: gs_small_sort_ctrl_words() words, 8-byte aligned.
int gs_small_sort(const UnitTable& U, const gs_proj* proj, int width, int height, int64_t cap, uint32_t* rec,
                  uint2* rect, uint32_t* count, void* ctrl_ws, uint32_t* sorted_vals, uint32_t* ranges,
                  uint32_t* d_num_instances, const gs_schedule* sched, int* d_status, cudaStream_t s) {
  Ctrl* ctrl = (Ctrl*)ctrl_ws;
  const int n_tiles = ((width + TILE - 1) / TILE) * ((height + TILE - 1) / TILE), NT = n_tiles * U.n;
  if (cudaMemsetAsync(ctrl, 0, offsetof(Ctrl, cut_m), s) != cudaSuccess ||
      cudaFuncSetAttribute(k_small_units, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(UnitSmem)) !=
          cudaSuccess)
    return GS_ERR_CUDA;
  gs_launch(k_small_units, (unsigned)U.n, ST, sizeof(UnitSmem), s, U, (const float4*)proj->xy, proj->depth,
      proj->radius, proj->tiles, width, height, cap, rec, rect, ctrl, d_status);
  const unsigned lb = (unsigned)((NT + LW - 1) / LW);
  gs_launch(k_small_count, lb, LW * 32, 0, s, U, width, n_tiles, NT, rec, rect, proj->depth, ctrl, count);
  gs_launch(k_small_ranges, 1, ST, 0, s, NT, count, (uint2*)ranges, d_num_instances,
      sched ? sched->tile_order : nullptr, sched ? sched->job_base : nullptr, sched ? sched->jobs : nullptr,
      sched ? sched->max_jobs : 0, sched ? sched->chunk : 32);
  gs_launch(k_small_fill, lb, LW * 32, 0, s, U, width, n_tiles, NT, rec, rect, proj->depth, ctrl,
      (const float4*)proj->xy, (const float4*)proj->conic_op, (const uint2*)ranges, sorted_vals,
      sched ? sched->block_masks : nullptr);
  return gs_check_launch();
}
