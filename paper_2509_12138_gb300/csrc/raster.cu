// a3 / a5: front-to-back alpha blending per 16x16 tile and its reverse replay.
//
// One thread per pixel; each warp owns a BW x (32/BW) pixel block of a 16x16
// tile (BW = 8, 16 or 4: the tunable variant).  With the sort's block masks
// every (tile, pixel block) is a one-warp CTA; without them one CTA covers a
// tile.  Each warp walks the tile's list
// independently of the other warps (no block barriers: warps whose block few
// splats reach do not wait for the busy ones).  A record is blended by a warp
// only if the bounding box of the ellipse where its alpha can reach 1/255
// meets the warp's block; this skips only (pixel, record) pairs that the
// per-pixel alpha test would reject anyway, so results are unchanged.
#include <cuda_runtime.h>
#include <limits.h>
#include <stdint.h>

#include "common.cuh"

using namespace gs;

namespace {

__device__ __forceinline__ void atomic_add2(float* p, float a, float b) {
#if __CUDA_ARCH__ >= 900
  atomicAdd(reinterpret_cast<float2*>(p), make_float2(a, b));
#else
  atomicAdd(p, a); atomicAdd(p + 1, b);
#endif
}
__device__ __forceinline__ void atomic_add4(float* p, float a, float b, float c, float d) {
#if __CUDA_ARCH__ >= 900
  atomicAdd(reinterpret_cast<float4*>(p), make_float4(a, b, c, d));
#else
  atomicAdd(p, a); atomicAdd(p + 1, b); atomicAdd(p + 2, c); atomicAdd(p + 3, d);
#endif
}

// Deterministic mode: gradients accumulate as int64 fixed point (value x 2^40,
// rounded to nearest).  Integer addition is associative, so the sums do not
// depend on the order in which warps add their contributions.  |value| is
// clamped to 2^22 (|value| 2^40 stays below 2^62); NaN adds 0.
constexpr float FIX_SCALE = 1099511627776.0f;  // 2^40
constexpr float FIX_LIMIT = 4194304.0f;        // 2^22
__device__ __forceinline__ unsigned long long to_fixed(float v) {
  float c = (v == v) ? fminf(fmaxf(v, -FIX_LIMIT), FIX_LIMIT) : 0.f;
  return (unsigned long long)__float2ll_rn(c * FIX_SCALE);
}

// One lane's nine gradient values of record pr (dx, dy | dA, dB, dC, dopacity | dr, dg, db).
__device__ __forceinline__ void add_lane(float* dxy, float* dco, float* drgb, unsigned long long* fixed, int64_t pr,
                                         const float* v) {
  if (fixed) {
    #pragma unroll
    for (int q = 0; q < 9; ++q) atomicAdd(fixed + 9 * pr + q, to_fixed(v[q]));
  } else {
    atomic_add2(dxy + 2 * pr, v[0], v[1]);
    atomic_add4(dco + 4 * pr, v[2], v[3], v[4], v[5]);
    atomic_add4(drgb + 4 * pr, v[6], v[7], v[8], 0.f);
  }
}

// Value q (0..8, order as above) of record pr.
__device__ __forceinline__ void add_one(float* dxy, float* dco, float* drgb, unsigned long long* fixed, int64_t pr,
                                        int q, float x) {
  if (fixed) {
    atomicAdd(fixed + 9 * pr + q, to_fixed(x));
    return;
  }
  float* dst = q < 2 ? dxy + 2 * pr + q : (q < 6 ? dco + 4 * pr + (q - 2) : drgb + 4 * pr + (q - 6));
  atomicAdd(dst, x);
}

__device__ __forceinline__ bool box_misses(float4 b, float x0, float x1, float y0, float y1) {
  return b.y < x0 || b.x > x1 || b.w < y0 || b.z > y1;
}

// Per-warp staging of one round of 32 records in shared memory: lane k writes
// record k, then every hit is read back as a broadcast.
struct __align__(16) Rec {
  float4 a;  // x, y, A, B
  float4 b;  // C, opacity, power floor, record id (bits)
  float4 c;  // r, g, b, unused
};

// Block index -> (unit, tile): heaviest tiles first when an order is given.
__device__ __forceinline__ void block_tile(const uint32_t* __restrict__ order, int n_tiles, int& u, int& tile) {
  uint32_t f = order ? order[blockIdx.x] : blockIdx.x;
  u = (int)(f / (uint32_t)n_tiles);
  tile = (int)(f % (uint32_t)n_tiles);
}

// Forward.  Each warp walks its tile's list on its own, 32 records per round
// (one per lane): a lane loads a record and tests its alpha box against the
// warp's pixel block; the records that hit are taken in list order, read back
// from the warp's staging area.  The next round's loads are issued before the
// current round is blended.
template <int BW>
__global__ void __launch_bounds__(TILE_PIX) k_render_fwd(const uint2* __restrict__ ranges,
                                                         const uint32_t* __restrict__ order,
                                                         const uint32_t* __restrict__ vals,
                                                         const float4* __restrict__ xy,
                                                         const float4* __restrict__ conic_op,
                                                         const float4* __restrict__ rgb, int W, int H, int TX,
                                                         int n_tiles, float bg0, float bg1, float bg2,
                                                         float* __restrict__ img, float* __restrict__ final_T,
                                                         uint32_t* __restrict__ n_contrib) {
  gs_wait_previous();
  const unsigned FULL = 0xffffffffu;
  __shared__ Rec s_rec[TILE_PIX / 32][32];
  int u, tile;
  block_tile(order, n_tiles, u, tile);
  int tx = tile % TX, ty = tile / TX;
  constexpr int BH = 32 / BW, NWX = TILE / BW;
  int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  float wx0 = (float)(tx * TILE + (w % NWX) * BW), wy0 = (float)(ty * TILE + (w / NWX) * BH);
  float wx1 = wx0 + (float)(BW - 1), wy1 = wy0 + (float)(BH - 1);
  int px = (int)wx0 + (lane % BW), py = (int)wy0 + (lane / BW);
  bool inside = px < W && py < H;
  uint2 rg = ranges[(int64_t)u * n_tiles + tile];
  int n = (int)(rg.y - rg.x);
  float T = 1.f, c0 = 0.f, c1 = 0.f, c2 = 0.f;
  int last = 0;
  bool done = !inside;
  // pixel offsets from the tile's corner, the origin of the staged record positions (rel_pos)
  float tox = (float)(tx * TILE), toy = (float)(ty * TILE);
  float fx = (float)(px - tx * TILE), fy = (float)(py - ty * TILE);
  Rec* my = &s_rec[w][0];
  uint32_t p_n = 0;
  float4 m_n = make_float4(0.f, 0.f, 0.f, 0.f);
  float4 co_n = make_float4(0.f, 0.f, 0.f, 0.f), c_n = co_n;
  if (lane < n) { p_n = vals[rg.x + lane]; m_n = xy[p_n]; co_n = conic_op[p_n]; c_n = rgb[p_n]; }
  for (int base = 0; base < n; base += 32) {
    if (__all_sync(FULL, done)) break;
    float4 m = m_n;
    float4 co = co_n, c = c_n;
    bool valid = base + lane < n;
    int kn = base + 32 + lane;
    if (kn < n) { p_n = vals[rg.x + kn]; m_n = xy[p_n]; co_n = conic_op[p_n]; c_n = rgb[p_n]; }
    float pmin = 0.f;
    bool hit = false;
    if (valid) {
      float4 b = alpha_box(make_float2(m.x, m.y), co, pmin);
      hit = !box_misses(b, wx0, wx1, wy0, wy1);
    }
    unsigned mask = __ballot_sync(FULL, hit);
    if (hit) {
      my[lane].a = make_float4(rel_pos(m.x, m.z, tox), rel_pos(m.y, m.w, toy), co.x, co.y);
      my[lane].b = make_float4(co.z, co.w, pmin, 0.f);
      my[lane].c = c;
    }
    __syncwarp();
    while (mask) {
      int j = __ffs(mask) - 1;
      mask &= mask - 1;
      if (done) continue;
      float4 ra = my[j].a, rb = my[j].b;
      float power = splat_power(ra.z, ra.w, rb.x, ra.x - fx, ra.y - fy);
      if (power > 0.f || power < rb.z) continue;
      float alpha = fminf(ALPHA_MAX, rb.y * __expf(power));
      if (alpha < ALPHA_MIN) continue;
      float tT = T * (1.f - alpha);
      if (tT < T_MIN) { done = true; continue; }
      float4 rc = my[j].c;
      float wgt = alpha * T;
      c0 += rc.x * wgt; c1 += rc.y * wgt; c2 += rc.z * wgt;
      T = tT;
      last = base + j + 1;
    }
    __syncwarp();
  }
  if (inside) {
    int64_t plane = (int64_t)W * H;
    int64_t pix = (int64_t)py * W + px;
    float* im = img + (int64_t)u * 3 * plane;
    im[pix] = c0 + T * bg0;
    im[plane + pix] = c1 + T * bg1;
    im[2 * plane + pix] = c2 + T * bg2;
    final_T[(int64_t)u * plane + pix] = T;
    n_contrib[(int64_t)u * plane + pix] = (uint32_t)last;
  }
}

// Sum of 8 values over the warp in 9 shuffles: each butterfly level halves the
// set of values a lane carries; afterwards lane l holds the total of value
// 4 bit4(l) + 2 bit3(l) + bit2(l).
__device__ __forceinline__ float reduce8(const float* v, int lane) {
  const unsigned FULL = 0xffffffffu;
  float a[4], b[2];
  bool h = lane & 16;
  #pragma unroll
  for (int i = 0; i < 4; ++i) {
    float send = h ? v[i] : v[i + 4], keep = h ? v[i + 4] : v[i];
    a[i] = keep + __shfl_xor_sync(FULL, send, 16);
  }
  h = lane & 8;
  #pragma unroll
  for (int i = 0; i < 2; ++i) {
    float send = h ? a[i] : a[i + 2], keep = h ? a[i + 2] : a[i];
    b[i] = keep + __shfl_xor_sync(FULL, send, 8);
  }
  h = lane & 4;
  float send = h ? b[0] : b[1], keep = h ? b[1] : b[0];
  float c = keep + __shfl_xor_sync(FULL, send, 4);
  c += __shfl_xor_sync(FULL, c, 2);
  c += __shfl_xor_sync(FULL, c, 1);
  return c;
}

// Backward.  Each warp replays its tile's list back to front from the largest
// n_contrib among its pixels, in rounds of 32 records; hits are taken in
// reverse list order.  The 9 gradient values of a record (d xy, d conic,
// d opacity, d rgb) are summed over the warp (butterfly for 8, a plain xor
// tree for the ninth) only if some lane contributed, and the lanes holding
// the totals add them to the record's gradients with one atomic instruction.
template <int BW>
__global__ void __launch_bounds__(TILE_PIX) k_render_bwd(const uint2* __restrict__ ranges,
                                                         const uint32_t* __restrict__ order,
                                                         const uint32_t* __restrict__ vals,
                                                         const float4* __restrict__ xy,
                                                         const float4* __restrict__ conic_op,
                                                         const float4* __restrict__ rgb, int W, int H, int TX,
                                                         int n_tiles, float bg0, float bg1, float bg2,
                                                         const float* __restrict__ final_T,
                                                         const uint32_t* __restrict__ n_contrib,
                                                         const float* __restrict__ dimg,
                                                         const float* __restrict__ dLdT, float* __restrict__ dxy,
                                                         float* __restrict__ dco, float* __restrict__ drgb,
                                                           unsigned long long* __restrict__ fixed) {
  gs_wait_previous();
  const unsigned FULL = 0xffffffffu;
  __shared__ Rec s_rec[TILE_PIX / 32][32];
  int u, tile;
  block_tile(order, n_tiles, u, tile);
  int tx = tile % TX, ty = tile / TX;
  constexpr int BH = 32 / BW, NWX = TILE / BW;
  int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  float wx0 = (float)(tx * TILE + (w % NWX) * BW), wy0 = (float)(ty * TILE + (w / NWX) * BH);
  float wx1 = wx0 + (float)(BW - 1), wy1 = wy0 + (float)(BH - 1);
  int px = (int)wx0 + (lane % BW), py = (int)wy0 + (lane / BW);
  bool inside = px < W && py < H;
  uint2 rg = ranges[(int64_t)u * n_tiles + tile];
  int64_t plane = (int64_t)W * H;
  int64_t pix = (int64_t)py * W + px;
  float T = 1.f, g0 = 0.f, g1 = 0.f, g2 = 0.f;
  float qT = 0.f;  // dL/dT_final x T_final: a blended entry adds -qT / (1 - alpha) to dL/dalpha
  int last = 0;
  if (inside) {
    T = final_T[(int64_t)u * plane + pix];
    last = (int)n_contrib[(int64_t)u * plane + pix];
    const float* d = dimg + (int64_t)u * 3 * plane;
    g0 = d[pix]; g1 = d[plane + pix]; g2 = d[2 * plane + pix];
    if (dLdT) qT = dLdT[(int64_t)u * plane + pix] * T;
  }
  int n = min(__reduce_max_sync(FULL, last), (int)(rg.y - rg.x));
  float S0 = bg0, S1 = bg1, S2 = bg2;  // colour behind the current entry
  float tox = (float)(tx * TILE), toy = (float)(ty * TILE);
  float fx = (float)(px - tx * TILE), fy = (float)(py - ty * TILE);
  Rec* my = &s_rec[w][0];
  // lanes (l & 3) == 0 hold butterfly value q(l); value 8 (d blue) is held by all lanes
  int q = ((lane >> 4) & 1) * 4 + ((lane >> 3) & 1) * 2 + ((lane >> 2) & 1);
  for (int top = n; top > 0; top -= 32) {
    int base = top - 32;
    int k = base + lane;
    bool hit = false;
    if (k >= 0) {
      uint32_t p = vals[rg.x + k];
      float4 m = xy[p];
      float4 co = conic_op[p];
      float pm;
      float4 b = alpha_box(make_float2(m.x, m.y), co, pm);
      hit = !box_misses(b, wx0, wx1, wy0, wy1);
      if (hit) {
        my[lane].a = make_float4(rel_pos(m.x, m.z, tox), rel_pos(m.y, m.w, toy), co.x, co.y);
        my[lane].b = make_float4(co.z, co.w, pm, __uint_as_float(p));
        my[lane].c = rgb[p];
      }
    }
    unsigned mask = __ballot_sync(FULL, hit);
    __syncwarp();
    while (mask) {
      int j = 31 - __clz(mask);
      mask &= ~(1u << j);
      int pos = base + j;
      float v[9];
      #pragma unroll
      for (int e = 0; e < 9; ++e) v[e] = 0.f;
      bool contrib = false;
      float4 ra = my[j].a, rb = my[j].b;
      if (pos < last) {
        float dx = ra.x - fx, dy = ra.y - fy;
        float A = ra.z, B = ra.w, Cc = rb.x, op = rb.y;
        float power = splat_power(A, B, Cc, dx, dy);
        if (power <= 0.f && power >= rb.z) {
          float G = __expf(power);
          float araw = op * G;
          bool clamped = araw > ALPHA_MAX;
          float alpha = clamped ? ALPHA_MAX : araw;
          if (alpha >= ALPHA_MIN) {
            contrib = true;
            float4 rc = my[j].c;
            T = __fdividef(T, 1.f - alpha);  // transmittance in front of this entry
            float wgt = alpha * T;
            v[6] = wgt * g0; v[7] = wgt * g1; v[8] = wgt * g2;
            float dalpha = T * ((rc.x - S0) * g0 + (rc.y - S1) * g1 + (rc.z - S2) * g2);
            if (qT != 0.f) dalpha -= __fdividef(qT, 1.f - alpha);
            S0 = alpha * rc.x + (1.f - alpha) * S0;
            S1 = alpha * rc.y + (1.f - alpha) * S1;
            S2 = alpha * rc.z + (1.f - alpha) * S2;
            if (!clamped) {
              v[5] = G * dalpha;
              float dp = araw * dalpha;
              v[2] = -0.5f * dx * dx * dp;
              v[3] = -dx * dy * dp;
              v[4] = -0.5f * dy * dy * dp;
              v[0] = -(A * dx + B * dy) * dp;
              v[1] = -(Cc * dy + B * dx) * dp;
            }
          }
        }
      }
      unsigned cm = __ballot_sync(FULL, contrib);
      if (cm) {
        int64_t pr = (int64_t)__float_as_uint(rb.w);
        if ((cm & (cm - 1)) == 0) {
          // a single contributing lane: no reduction
          if (contrib) add_lane(dxy, dco, drgb, fixed, pr, v);
        } else {
          float tot = reduce8(v, lane);
          float e8 = v[8];
          #pragma unroll
          for (int o = 16; o > 0; o >>= 1) e8 += __shfl_xor_sync(FULL, e8, o);
          if ((lane & 3) == 0) {
            add_one(dxy, dco, drgb, fixed, pr, q, tot);
          } else if (lane == 1) {
            add_one(dxy, dco, drgb, fixed, pr, 8, e8);
          }
        }
      }
    }
    __syncwarp();
  }
}

// Bits of the 4x4 pixel blocks that a warp's BW x (32/BW) pixel block overlaps.
template <int BW>
__device__ __forceinline__ uint32_t warp_block_bits(int w) {
  constexpr int BH = 32 / BW, NWX = TILE / BW;
  int ox = (w % NWX) * BW, oy = (w / NWX) * BH;
  uint32_t bits = 0;
  #pragma unroll
  for (int by = 0; by < 4; ++by)
    #pragma unroll
    for (int bx = 0; bx < 4; ++bx)
      if (4 * bx <= ox + BW - 1 && 4 * bx + 3 >= ox && 4 * by <= oy + BH - 1 && 4 * by + 3 >= oy)
        bits |= 1u << (4 * by + bx);
  return bits;
}

// Transpose of a 32 x 32 bit matrix held one row per lane: bit j of the
// result in lane p is bit p of lane j's word (five butterfly exchanges of
// 16-, 8-, 4-, 2- and 1-bit blocks).
__device__ __forceinline__ uint32_t transpose32(uint32_t x) {
  const int lane = threadIdx.x & 31;
  const uint32_t MS[5] = {0x0000ffffu, 0x00ff00ffu, 0x0f0f0f0fu, 0x33333333u, 0x55555555u};
  #pragma unroll
  for (int k = 0; k < 5; ++k) {
    const int s = 16 >> k;
    const uint32_t m = MS[k];
    const uint32_t y = __shfl_xor_sync(0xffffffffu, x, s);
    x = (lane & s) ? (((y & ~m) >> s) | (x & ~m)) : ((x & m) | ((y & m) << s));
  }
  return x;
}

// The pixels of a warp's block (BW x 32 / BW from tile-local origin (ox, oy))
// whose centre lies in a superset of a record's alpha >= 1/255 box, so that
// every pixel outside it has alpha < 1/255 and would be skipped by the blend:
// columns c0 .. c1 and rows r0 .. r1 of the block (none: c1 < c0).  (rx, ry):
// the record's tile-local position; co: conic and opacity; pf: its power floor
// (rgb.w), which is at most -(ln(255 o) + 1e-3), so -pf takes the place of
// alpha_box's logarithm.  The approximate divide stays far inside the 0.1% +
// 0.01 px margin.
struct HitBox {
  int c0, c1, r0, r1;
};
template <int BW>
__device__ __forceinline__ HitBox hit_box(float rx, float ry, float4 co, float pf, float ox, float oy) {
  constexpr int BH = 32 / BW;
  HitBox h = {0, -1, 0, -1};
  const float det = co.x * co.z - co.y * co.y;
  if (!(pf < 0.f) || !(det > 0.f)) return h;
  const float k = __fdividef(-2.f * pf, det);
  const float ex = sqrtf(k * co.z) * 1.001f + 0.01f, ey = sqrtf(k * co.x) * 1.001f + 0.01f;
  const float c0 = fmaxf(ceilf(rx - ex - ox), 0.f), c1 = fminf(floorf(rx + ex - ox), (float)(BW - 1));
  const float r0 = fmaxf(ceilf(ry - ey - oy), 0.f), r1 = fminf(floorf(ry + ey - oy), (float)(BH - 1));
  if (!(c0 <= c1) || !(r0 <= r1)) return h;
  h.c0 = (int)c0; h.c1 = (int)c1; h.r0 = (int)r0; h.r1 = (int)r1;
  return h;
}

// Record-major evaluation: a record's o G at every pixel of its box that can
// blend (alpha >= 1/255), to row[pixel]; returns the mask of those pixels.
// CLAMP stores min(0.99, o G).  Only the rows and columns that hold pixels of
// `act` are evaluated (pixels outside it may be).  The pixel coordinates are exact small integers
// stepped in float (integer conversions share the exponential's quarter-rate
// unit).
template <int BW, bool CLAMP>
__device__ __forceinline__ uint32_t eval_hit(float rx, float ry, float4 co, float pf, float ox, float oy, uint32_t act,
                                             float* row) {
  HitBox h = hit_box<BW>(rx, ry, co, pf, ox, oy);
  uint32_t valid = 0u, cols = act;  // columns of act: its rows folded onto each other
  #pragma unroll
  for (int q = 16; q >= BW; q >>= 1) cols |= cols >> q;
  cols &= (1u << BW) - 1u;
  h.c0 = max(h.c0, __ffs(cols) - 1);
  h.c1 = min(h.c1, 31 - __clz(cols));
  h.r0 = max(h.r0, (__ffs(act) - 1) / BW);
  h.r1 = min(h.r1, (31 - __clz(act)) / BW);
  if (h.c1 < h.c0 || h.r1 < h.r0) return 0u;
  const int w = h.c1 - h.c0 + 1;
  const int n = w * (h.r1 - h.r0 + 1);
  const float x0 = ox + (float)h.c0, x1 = ox + (float)h.c1;
  float x = x0, y = oy + (float)h.r0;
  int px = h.r0 * BW + h.c0;
  #pragma unroll 2
  for (int k = 0; k < n; ++k) {
    const float power = splat_power(co.x, co.y, co.z, rx - x, ry - y);
    const float a = co.w * __expf(power), alpha = fminf(ALPHA_MAX, a);
    const bool hit = !(power > 0.f) && !(alpha < ALPHA_MIN);
    if (hit) row[px] = CLAMP ? alpha : a;
    valid |= (hit ? 1u : 0u) << px;
    const bool wrap = x >= x1;  // next column, or the next row's first
    x = wrap ? x0 : x + 1.f;
    y = wrap ? y + 1.f : y;
    px += wrap ? BW + 1 - w : 1;
  }
  return valid;
}

// ---- the walks of one warp over a list: hits gathered 32 at a time
//
// With sub-pixel splats a list entry reaches few of a tile's eight pixel
// blocks (about 5 of 32 at 10M Gaussians and 1080p) and few pixels of a block
// it reaches (about 9 of 32).  So the warp first reads the 2-byte block masks
// of SCAN entries at a time and queues the entries that reach its block, and
// works on batches of up to 32 queued hits, in two lane assignments:
//   record-major: lane j holds hit j's record in registers and evaluates its
//     alpha at the pixels its box reaches, into a (hit, pixel) matrix in shared
//     memory (row stride 33: neither assignment has regular bank conflicts);
//   pixel-major: the 32 x 32 bits of accepted pairs are transposed across the
//     warp, and lane p composites the hits of its pixel in list order, reading
//     one alpha and a colour per pair (the colours lie 32 to a bank row, so any
//     mix of hits is read without conflicts).
// Each phase runs as often as its busiest lane has pairs.  Every pair's alpha
// and the order of a pixel's compositing are those of a sequential walk.  Bound
// by instruction issue (47-70% of cycles on a 2M scene) and, on edge-on views,
// by the longest block's serial walk.  Forward stage at one lane per pixel and
// hit -> this: 200k at 960x540 134 -> 72 us, 1M at 1080p 319 -> 181 us.  Where a
// splat covers whole blocks, one lane per pixel and hit evaluates as few pairs
// and is the faster one by 5 to 20% (whole lists of 1M splats of 6 pixels at
// 1080p 730 us, this 854; of a few dozen entries at 800x600 18, this 30), but a
// choice per batch or per list within the kernel cost the small splats 3 to 10%
// in registers, and a second kernel more than that.  Three
// or four pairs per step of the pixel-major loop, or four pixels per step of the
// record-major one, cost registers and were slower (10M at 1080p 1157 us with
// two, 1208, 1302 and 1264).
constexpr int SCAN = 256;            // entries whose masks are read at a time (8 per lane)
constexpr int QUEUE_CAP = SCAN + 32; // queued entries: a full scan behind at most 31 left over
constexpr int MROW = 33;             // row stride of the (hit, pixel) matrices

struct FwdScratch {
  float alpha[32 * MROW];
  float r[32], g[32], b[32];
  uint32_t q[QUEUE_CAP];
};

// Queues the entries of [s, min(s + SCAN, end)) (DOWN: of (max(s - SCAN, beg),
// s], from s down) whose block mask meets wbits behind the qn queued ones, in
// walking order; returns the new number.  masks: of the list's first entry on.
template <bool DOWN>
__device__ __forceinline__ int scan_hits(const uint16_t* __restrict__ masks, int s, int bound, uint32_t wbits,
                                         uint32_t* q, int qn) {
  const unsigned FULL = 0xffffffffu;
  const int lane = threadIdx.x & 31;
  const uint32_t lt = (1u << lane) - 1u;
  uint32_t mk[SCAN / 32];
  #pragma unroll
  for (int r = 0; r < SCAN / 32; ++r) {
    const int k = DOWN ? s - 32 * r - lane : s + 32 * r + lane;
    mk[r] = (DOWN ? k >= bound : k < bound) ? masks[k] : 0u;
  }
  #pragma unroll
  for (int r = 0; r < SCAN / 32; ++r) {
    if (DOWN ? s - 32 * r < bound : s + 32 * r >= bound) break;
    const bool h = (mk[r] & wbits) != 0u;
    const unsigned bal = __ballot_sync(FULL, h);
    if (h) q[qn + __popc(bal & lt)] = (uint32_t)(DOWN ? s - 32 * r - lane : s + 32 * r + lane);
    qn += __popc(bal);
  }
  return qn;
}

__device__ __forceinline__ void prefetch_l1(const void* p) { asm volatile("prefetch.global.L1 [%0];" ::"l"(p)); }

// Front-to-back walk of list entries [beg, end) (indices from the list's
// start `off`) for one warp's pixel block (tile-local origin (ox, oy)):
// composites into (T, c, last) of the lanes that are not done; a lane whose
// transmittance would fall below T_MIN stops (done).  DUAL: also composites
// the same pairs from T = 1 into loc = (T, c), the walk's partial.
template <int BW, bool DUAL>
__device__ __forceinline__ void walk_fwd(const uint32_t* __restrict__ vals, const uint16_t* __restrict__ masks,
                                         const float4* __restrict__ xy, const float4* __restrict__ conic_op,
                                         const float4* __restrict__ rgb, uint32_t off, int beg, int end,
                                         uint32_t wbits, float tox, float toy, float ox, float oy, FwdScratch& sc,
                                         float& T, float& c0, float& c1, float& c2, int& last, bool& done,
                                         float4& loc) {
  const unsigned FULL = 0xffffffffu;
  const int lane = threadIdx.x & 31;
  vals += off;
  masks += off;
  int scan = beg, qn = 0, qh = 0;  // next entry to scan; queued entries are q[qh .. qn)
  // Queues the next batch's entries and starts its records on their way to L1, one batch ahead of their use, and the
  // masks and ids of the following scan (the next chunk's too: no gain).  The warps that fit (20 per SM at 96
  // registers) do not cover the latency of masks, ids and records in turn: waiting for each, the forward stage took 4
  // to 8% longer (10M at 1080p, two views, 1203, 1515 -> 1147, 1398 us; merged 100M at 4K 7462 -> 7092; 6M at 400x300
  // 1249 -> 1151).
  auto next_batch = [&]() -> uint32_t {
    if (qn - qh < 32 && scan < end) {
      // the left-over entries to the front, then whole scans until a batch is full
      const uint32_t keep = qh + lane < qn ? sc.q[qh + lane] : 0u;
      __syncwarp();
      qn -= qh;
      qh = 0;
      if (lane < qn) sc.q[lane] = keep;
      do {
        qn = scan_hits<false>(masks, scan, end, wbits, sc.q, qn);
        scan += SCAN;
      } while (qn < 32 && scan < end);
      __syncwarp();
      // one lane per 128 bytes: 64 masks or 32 ids
      const int ahead = scan + (lane < SCAN / 64 ? 64 * lane : 32 * (lane - SCAN / 64));
      if (lane < SCAN / 64 + SCAN / 32 && ahead < end) {
        if (lane < SCAN / 64) prefetch_l1(masks + ahead);
        else prefetch_l1(vals + ahead);
      }
    }
    uint32_t p = 0u;
    if (qh + lane < qn) {
      p = vals[sc.q[qh + lane]];
      prefetch_l1(xy + p);
      prefetch_l1(conic_op + p);
      prefetch_l1(rgb + p);
    }
    return p;
  };
  uint32_t pn = next_batch();
  for (;;) {
    const uint32_t act = __ballot_sync(FULL, !done);
    if (!act) break;
    const int nb = min(32, qn - qh);
    if (nb == 0) break;
    const uint32_t p = pn, entry = lane < nb ? sc.q[qh + lane] : 0u;
    qh += nb;
    pn = next_batch();
    // record-major: alpha of hit `lane` at the pixels its box reaches
    uint32_t valid = 0u;
    if (lane < nb) {
      const float4 m = xy[p], co = conic_op[p], c = rgb[p];
      const float rx = rel_pos(m.x, m.z, tox), ry = rel_pos(m.y, m.w, toy);
      sc.r[lane] = c.x; sc.g[lane] = c.y; sc.b[lane] = c.z;
      valid = eval_hit<BW, true>(rx, ry, co, c.w, ox, oy, act, sc.alpha + lane * MROW);
    }
    __syncwarp();
    // pixel-major: this pixel's pairs in list order
    uint32_t mine = transpose32(valid);
    int lj = -1;
    if (done) mine = 0u;
    // as many steps as the busiest lane has pairs, two at a time; a lane without one takes alpha 0.  No branch
    // inside, so the loads and bit scans of the next pairs overlap this one's chain through T.
    for (int it = (int)__reduce_max_sync(FULL, (uint32_t)__popc(mine)); it > 0; it -= 2) {
      int j[2];
      float al[2], cr[2], cg[2], cb[2];
      #pragma unroll
      for (int e = 0; e < 2; ++e) {
        j[e] = mine ? __ffs(mine) - 1 : 0;
        al[e] = mine ? sc.alpha[j[e] * MROW + lane] : 0.f;
        cr[e] = sc.r[j[e]]; cg[e] = sc.g[j[e]]; cb[e] = sc.b[j[e]];
        mine &= mine - 1;
      }
      #pragma unroll
      for (int e = 0; e < 2; ++e) {
        const float om = 1.f - al[e], tT = T * om;
        const bool pair = al[e] > 0.f && !done;
        const bool blend = pair && !(tT < T_MIN);
        done = done || (pair && tT < T_MIN);
        const float wgt = blend ? al[e] * T : 0.f;
        if (blend) {
          c0 += cr[e] * wgt; c1 += cg[e] * wgt; c2 += cb[e] * wgt;
          T = tT;
          lj = j[e];
        }
        if (DUAL) {
          const float lw = al[e] * loc.x;
          if (blend) {
            loc.y += cr[e] * lw; loc.z += cg[e] * lw; loc.w += cb[e] * lw;
            loc.x *= om;
          }
        }
      }
    }
    const int at = (int)__shfl_sync(FULL, entry, max(lj, 0));
    if (lj >= 0) last = at + 1;
    __syncwarp();
  }
  __syncwarp();
}

// ---- scheduled forward: sequential fronts, chunk-parallel remainders
//
// Per pixel, front-to-back compositing over a list is a product of (1 - alpha)
// factors and a sum of colours weighted by the running product, so chunks of
// K entries can be composited independently from T = 1 and combined:
// C += T C_c, T *= T_c.  Composited that way, everything behind a pixel's early
// stop is work for nothing (at 10M Gaussians and 1080p 50-65% of the entries lie
// behind the last stop of their block); walked in order, a list of a hundred
// chunks is one warp's serial work.  So:
//   front  (list, block warps): chunks 0 .. M - 1 in order with the early stop.
//           A list that ends there, or whose pixels all stop there, is final.
//           Otherwise the block's later chunks are queued;
//   chunks (queued jobs): partial (T_c, C_c, last_c | stop) of every such chunk;
//   combine (queued blocks): applies the partials in order, finds each pixel's
//           stop chunk c* (the first with T T_c < T_MIN or a stop of its own),
//           writes the checkpoints in front of it, finishes the pixels that
//           never stop and marks the stop chunks' queue entries;
//   stop   (marked jobs): walks c* again from the true incoming state for the
//           pixels that stop there and writes their remaining checkpoints.
// Per pixel the blended entries and the stop decision are those of the
// sequential walk; the combine changes only the rounding order of T and C.
// gs_schedule.walk_whole_lists is M = infinity.
// M depends on the lists and on how many warps the device holds, not on the
// timing (a split that followed it would change the rounding of the checkpoints
// from run to run).  With the blocks of lists with entries and the smaller of
// the resident warps and the image's blocks:
//   all lists of at most 8 chunks (by the heaviest's class): no split, the
//     passes behind the front would cost more than its last blocks' walks;
//   fewer blocks than that (a small image with empty lists), or fewer than an
//     eighth of the resident warps (any image of up to 47 tiles): 1, a serial
//     walk leaves warps idle;
//   else the chunks or blocks a warp gets, the fewer, 4 to 16, so that a serial
//     walk is no longer than the whole pass; the parallel passes walk chunks
//     behind stops, so as much as that bound allows stays in front.
// Forward stage, two views each (us), M = 1 / 4 / 16 -> by this rule: 10M at
// 1080p 1846, 1626 / 1687, 1592 / 1144, 1351 -> 1142, 1342; 1M at 1080p 268, 309
// / 179, 280 / 180, 218 -> 180, 220; 8 partitions of 2.8M at 1080p 726, 678 /
// 703, 665 / 779, 704 -> 762, 696; 4M at 1800x1300 696, 768 / 668, 723 / 525,
// 673 -> 522, 674; 3M in 3 partitions at 400x300, two views, 1119, 1089 / 1223,
// 1197 / 1754, 1559 -> 1113, 1093; 6M at 400x300 1120, 1069 / 1299, 1240 / 1648,
// 1643 -> 1124, 1079; 1M there 368, 369 / 429, 450 / 415, 542 -> 366, 370.
// Images covered by lists of many chunks, M = 1 / 4 / 8: 32x32, 50,000 faint
// splats, 116 / 178 / 266; 64x64, 1M, 226 / 353 / 497 (but 50,000 opaque ones
// 98 / 89 / 66, so the line is not exact); 128x128, 300,000 of some pixels, 451 /
// 375 / 270; 256x256, 50,000 of many, 368 / 126 / 126.
// Where the capacity bounds every list to FRONT_CHUNKS chunks, the passes behind
// the front are not launched at all (5 us each with nothing to do).
constexpr int FRONT_CHUNKS = 16;
__device__ __forceinline__ int front_chunks(const uint2* __restrict__ ranges, const uint32_t* __restrict__ order,
                                            uint32_t jobs, uint32_t lists, uint32_t NT, uint32_t resident, int K) {
  if (lists == 0u) return FRONT_CHUNKS;
  const uint32_t units = 8u * lists;
  const uint2 first = ranges[order[0]];  // of the heaviest lists' class: less than twice its length is the longest
  const uint32_t longest = 2u << (31 - __clz((int)max(first.y - first.x, 1u)));
  if (longest <= 8u * (uint32_t)K) return FRONT_CHUNKS;
  const uint32_t warps = min(resident, 8u * NT);
  if (units < warps || 8u * units <= resident) return 1;
  return (int)min((uint32_t)FRONT_CHUNKS, max(4u, 8u * min(jobs, units) / warps));
}
constexpr uint32_t STOP_BIT = 0x80000000u;  // partial or front state: the pixel has stopped
constexpr uint32_t REWALK_BIT = 0x80000000u;  // n_contrib between combine and stop pass: stop chunk pending,
                                             // the stop chunk c* in the bits below it
constexpr uint32_t MARK_BIT = 0x80000000u;  // queue entry (chunk job << 3 | block): some pixel stops in it

// The warp's pixel of (list o, block w) and its geometry.
template <int BW>
struct PixelOf {
  int u, tile, tx, ty, px, py, pix_local, ox, oy;  // (ox, oy): the block's tile-local origin
  bool inside;
  uint32_t wbits;  // the 4x4 blocks of the warp's pixels
  __device__ __forceinline__ PixelOf(const uint32_t* __restrict__ order, int o, int w, int n_tiles, int TX, int W,
                                     int H) {
    uint32_t f = order[o];
    u = (int)(f / (uint32_t)n_tiles);
    tile = (int)(f % (uint32_t)n_tiles);
    tx = tile % TX;
    ty = tile / TX;
    constexpr int BH = 32 / BW, NWX = TILE / BW;
    int lane = threadIdx.x & 31;
    ox = (w % NWX) * BW;
    oy = (w / NWX) * BH;
    px = tx * TILE + ox + (lane % BW);
    py = ty * TILE + oy + (lane / BW);
    pix_local = (py - ty * TILE) * TILE + (px - tx * TILE);
    inside = px < W && py < H;
    wbits = warp_block_bits<BW>(w);
  }
};

// Lists without entries: the background.  One block per (unit, tile); block 0
// also zeroes the work counters of the passes behind it.
__global__ void __launch_bounds__(TILE_PIX) k_render_fwd_empty(const uint2* __restrict__ ranges, int W, int H, int TX,
                                                               int n_tiles, float bg0, float bg1, float bg2,
                                                               float* __restrict__ img, float* __restrict__ final_T,
                                                               uint32_t* __restrict__ n_contrib,
                                                               uint32_t* __restrict__ tickets,
                                                               uint32_t* __restrict__ qcount) {
  gs_wait_previous();
  if (blockIdx.x == 0 && threadIdx.x == 0) { tickets[0] = 0u; tickets[1] = 0u; *qcount = 0u; }
  const uint2 rg = ranges[blockIdx.x];
  if (rg.y > rg.x) return;
  const int u = (int)(blockIdx.x / (unsigned)n_tiles), tile = (int)(blockIdx.x % (unsigned)n_tiles);
  const int px = (tile % TX) * TILE + (int)(threadIdx.x % TILE), py = (tile / TX) * TILE + (int)(threadIdx.x / TILE);
  if (px >= W || py >= H) return;
  const int64_t plane = (int64_t)W * H, pix = (int64_t)py * W + px;
  float* im = img + (int64_t)u * 3 * plane;
  im[pix] = bg0; im[plane + pix] = bg1; im[2 * plane + pix] = bg2;
  final_T[(int64_t)u * plane + pix] = 1.f;
  n_contrib[(int64_t)u * plane + pix] = 0u;
}

// Number of lists with entries: they come first in tile order, so it is the
// first order position from which job_base stays at its total (a 32-way search
// by the warp).
__device__ __forceinline__ int lists_in_use(const uint32_t* __restrict__ job_base, int NT) {
  const uint32_t total = job_base[NT];
  int lo = 0, hi = NT;  // the answer lies in [lo, hi]
  while (lo < hi) {
    const int step = (hi - lo + 31) / 32;
    const int at = lo + step * (int)(threadIdx.x & 31);
    const uint32_t full = __ballot_sync(0xffffffffu, at >= hi || job_base[min(at, NT)] == total);
    const int f = full ? __ffs(full) - 1 : 32;  // first probe at or past the answer
    const int nlo = f == 0 ? lo : lo + step * (f - 1) + 1;
    hi = f == 0 ? lo : min(hi, lo + step * f);
    lo = nlo;
  }
  return lo;
}

// Checkpoints of boundaries [lo, hi] of a pixel, back to front: boundary b's
// slot holds chunk b's partial (T_b, C_b) and chunk_last the T in front of it;
// it becomes (that T, colour behind the boundary per unit T).  S: the colour
// behind boundary hi + 1, updated.  Loads are issued CB boundaries at a time.
constexpr int CB = 4;
__device__ __forceinline__ void close_checkpoints(float4* __restrict__ cpp, const uint32_t* __restrict__ clp, int lo,
                                                  int hi, float& S0, float& S1, float& S2) {
  for (int bb = hi; bb >= lo; bb -= CB) {
    float4 ptv[CB];
    uint32_t tv[CB];
    #pragma unroll
    for (int q = 0; q < CB; ++q)
      if (bb - q >= lo) {
        ptv[q] = cpp[(int64_t)(bb - q - 1) * TILE_PIX];
        tv[q] = clp[(int64_t)(bb - q - 1) * TILE_PIX];
      }
    #pragma unroll
    for (int q = 0; q < CB; ++q) {
      if (bb - q < lo) break;
      const float4 pt = ptv[q];
      S0 = pt.y + pt.x * S0; S1 = pt.z + pt.x * S1; S2 = pt.w + pt.x * S2;
      cpp[(int64_t)(bb - q - 1) * TILE_PIX] = make_float4(__uint_as_float(tv[q]), S0, S1, S2);
    }
  }
}

// One chunk from the state (T, c): walked in order, its partial from T = 1 to
// *slot and the incoming T to *tslot (slots of the boundary in front of it).
template <int BW>
__device__ __forceinline__ float4 walk_chunk(const uint32_t* __restrict__ vals, const uint16_t* __restrict__ masks,
                                             const float4* __restrict__ xy, const float4* __restrict__ conic_op,
                                             const float4* __restrict__ rgb, uint32_t off, int beg, int end,
                                             uint32_t wbits, float tox, float toy, float ox, float oy, FwdScratch& sc,
                                             float& T, float& c0, float& c1, float& c2, int& last, bool& done,
                                             bool store, float4* slot, uint32_t* tslot) {
  if (store) *tslot = __float_as_uint(T);
  float4 loc = make_float4(1.f, 0.f, 0.f, 0.f);
  walk_fwd<BW, true>(vals, masks, xy, conic_op, rgb, off, beg, end, wbits, tox, toy, ox, oy, sc, T, c0, c1, c2, last,
                     done, loc);
  if (store) *slot = loc;
  return loc;
}

// Front pass: unit (list o, block w) walks chunks 0 .. min(nch, M) - 1 in
// order.  The resident warps take the units, heaviest lists first: the first
// one by the block's number, the others from a ticket counter, the next ticket
// fetched while a unit runs.  (With the first one from the counter too a warp
// drew two before it began, and with up to two units per warp half of the warps
// got two units and the others none: 200k at 960x540 89 -> 72 us, whole lists 71
// -> 59; 600k at 256x256 175 -> 113; 8 views of 2,000 at 128x128 47 -> 36.)
template <int BW>
__global__ void __launch_bounds__(32) k_render_fwd_front(const uint2* __restrict__ ranges,
                                                         const uint32_t* __restrict__ order,
                                                         const uint32_t* __restrict__ job_base, int K, bool whole,
                                                         uint32_t resident, int NT,
                                                         float4* __restrict__ ckpt, uint32_t* __restrict__ chunk_last,
                                                         const uint32_t* __restrict__ vals,
                                                         const uint16_t* __restrict__ masks,
                                                         const float4* __restrict__ xy,
                                                         const float4* __restrict__ conic_op,
                                                         const float4* __restrict__ rgb, int W, int H, int TX,
                                                         int n_tiles, float bg0, float bg1, float bg2,
                                                         float* __restrict__ img, float* __restrict__ final_T,
                                                         uint32_t* __restrict__ n_contrib,
                                                         uint32_t* __restrict__ queue, uint32_t qcap,
                                                         uint32_t* __restrict__ ticket) {
  gs_wait_previous();
  __shared__ FwdScratch s_walk;
  const int lane = threadIdx.x & 31;
  const int lists = lists_in_use(job_base, NT);
  const uint32_t total = (uint32_t)lists * 8u;
  const int M = resident ? front_chunks(ranges, order, job_base[NT], (uint32_t)lists, (uint32_t)NT, resident, K)
                         : INT_MAX;
  auto unit = [&](uint32_t vb) {
    const int o = (int)(vb >> 3), w = (int)(vb & 7u);
    PixelOf<BW> P(order, o, w, n_tiles, TX, W, H);
    const uint32_t jb = job_base[o];
    const int nch = (int)(job_base[o + 1] - jb);
    const uint2 rg = ranges[(int64_t)P.u * n_tiles + P.tile];
    const int L = (int)(rg.y - rg.x);
    const int64_t cp0 = (int64_t)jb - o;
    float4* cpp = ckpt + cp0 * TILE_PIX + P.pix_local;  // slot of boundary b: cpp[(b - 1) * TILE_PIX]
    uint32_t* clp = chunk_last + cp0 * TILE_PIX + P.pix_local;
    const int upto = min(nch, M);
    float T = 1.f, c0 = 0.f, c1 = 0.f, c2 = 0.f;
    int last = 0, c = 0;
    bool done = !P.inside, in_order = whole;
    for (; c < upto; ++c) {
      if (__all_sync(0xffffffffu, done)) break;
      const float Tin = T, i0 = c0, i1 = c1, i2 = c2;
      const bool was = done;
      const float4 loc = walk_chunk<BW>(vals, masks, xy, conic_op, rgb, rg.x, c * K, min(c * K + K, L), P.wbits,
                                        (float)(P.tx * TILE), (float)(P.ty * TILE), (float)P.ox, (float)P.oy, s_walk,
                                        T, c0, c1, c2, last, done, c > 0 && P.inside,
                                        cpp + (int64_t)(c - 1) * TILE_PIX, clp + (int64_t)(c - 1) * TILE_PIX);
      // a chunk without a stop enters by its partial, as the combine's do, so that images do not depend on M (but for
      // a pixel whose stop falls on the two sides of one rounding); from a stop chunk on (and in whole-list walks) the
      // walked state counts
      in_order = in_order || !(Tin * loc.x >= T_MIN);
      if (!in_order && !done && !was) {
        T = Tin * loc.x;
        c0 = i0 + Tin * loc.y; c1 = i1 + Tin * loc.z; c2 = i2 + Tin * loc.w;
      }
    }
    const int64_t plane = (int64_t)W * H;
    const int64_t pix = (int64_t)P.py * W + P.px;
    float* im = img + (int64_t)P.u * 3 * plane;
    if (c < nch && !__all_sync(0xffffffffu, done)) {
      // the rest of the list in parallel: this block's state in front of chunk M, and its later chunks' jobs
      uint32_t base = lane == 0 ? atomicAdd(queue + qcap, (uint32_t)(nch - c)) : 0u;
      base = __shfl_sync(0xffffffffu, base, 0);
      for (int q = c + lane; q < nch; q += 32) queue[base + (uint32_t)(q - c)] = ((jb + (uint32_t)q) << 3) | (uint32_t)w;
      if (!P.inside) return;
      im[pix] = c0; im[plane + pix] = c1; im[2 * plane + pix] = c2;
      final_T[(int64_t)P.u * plane + pix] = T;
      n_contrib[(int64_t)P.u * plane + pix] = (uint32_t)last | (done ? STOP_BIT : 0u);
      return;
    }
    if (!P.inside) return;
    for (int b = nch - 1; b >= max(c, 1); --b)
      cpp[(int64_t)(b - 1) * TILE_PIX] = make_float4(T, bg0, bg1, bg2);  // behind the stop: final state
    float S0 = bg0, S1 = bg1, S2 = bg2;
    close_checkpoints(cpp, clp, 1, c - 1, S0, S1, S2);
    im[pix] = c0 + T * bg0;
    im[plane + pix] = c1 + T * bg1;
    im[2 * plane + pix] = c2 + T * bg2;
    final_T[(int64_t)P.u * plane + pix] = T;
    n_contrib[(int64_t)P.u * plane + pix] = (uint32_t)last;
  };
  const bool lead = lane == 0;
  uint32_t vb = blockIdx.x;
  while (vb < total) {
    const uint32_t nxt = lead ? gridDim.x + atomicAdd(ticket, 1u) : 0u;
    unit(vb);
    vb = __shfl_sync(0xffffffffu, nxt, 0);
  }
}

// Chunk pass: queued job (list o, chunk c, block w) composites its entries
// from T = 1 for the pixels that have not stopped in front of chunk M; the
// partial goes to checkpoint slot c - 1 and chunk_last.
template <int BW>
__global__ void __launch_bounds__(32) k_render_fwd_chunk(const uint2* __restrict__ ranges,
                                                         const uint32_t* __restrict__ order,
                                                         const uint32_t* __restrict__ job_base,
                                                         const uint32_t* __restrict__ jobs, int K,
                                                         float4* __restrict__ ckpt, uint32_t* __restrict__ chunk_last,
                                                         const uint32_t* __restrict__ vals,
                                                         const uint16_t* __restrict__ masks,
                                                         const float4* __restrict__ xy,
                                                         const float4* __restrict__ conic_op,
                                                         const float4* __restrict__ rgb, int W, int H, int TX,
                                                         int n_tiles, const uint32_t* __restrict__ n_contrib,
                                                         const uint32_t* __restrict__ queue, uint32_t qcap,
                                                         uint32_t* __restrict__ ticket) {
  gs_wait_previous();
  __shared__ FwdScratch s_walk;
  const uint32_t total = queue[qcap];
  auto job = [&](uint32_t ent) {
    const uint32_t jid = ent >> 3;
    const int w = (int)(ent & 7u), o = (int)jobs[2 * (int64_t)jid], ch = (int)jobs[2 * (int64_t)jid + 1];
    PixelOf<BW> P(order, o, w, n_tiles, TX, W, H);
    const uint2 rg = ranges[(int64_t)P.u * n_tiles + P.tile];
    const int L = (int)(rg.y - rg.x);
    float T = 1.f, c0 = 0.f, c1 = 0.f, c2 = 0.f;
    int last = 0;
    bool done = !P.inside;
    if (P.inside) done = (n_contrib[((int64_t)P.u * H + P.py) * W + P.px] & STOP_BIT) != 0u;
    float4 none;
    walk_fwd<BW, false>(vals, masks, xy, conic_op, rgb, rg.x, ch * K, min(ch * K + K, L), P.wbits,
                        (float)(P.tx * TILE), (float)(P.ty * TILE), (float)P.ox, (float)P.oy, s_walk, T, c0, c1, c2,
                        last, done, none);
    if (!P.inside) return;
    const int64_t slot = ((int64_t)job_base[o] - o + ch - 1) * TILE_PIX + P.pix_local;
    ckpt[slot] = make_float4(T, c0, c1, c2);
    chunk_last[slot] = (uint32_t)last | (done ? STOP_BIT : 0u);
  };
  const bool lead = (threadIdx.x & 31) == 0;
  uint32_t e = __shfl_sync(0xffffffffu, lead ? atomicAdd(ticket, 1u) : 0u, 0);
  while (e < total) {
    uint32_t nxt = lead ? atomicAdd(ticket, 1u) : 0u;
    job(queue[e]);
    e = __shfl_sync(0xffffffffu, nxt, 0);
  }
}

// The combine of one pixel of a queued block: the partials of chunks m .. nch - 1
// applied to the front's state; cstar receives the pixel's stop chunk (-1: none,
// or a stop in the front).  The per-chunk loads are issued CB chunks at a time:
// for lists of hundreds of chunks the walk is otherwise one load latency per chunk.
__device__ __forceinline__ void combine_pixel(int m, int nch, int64_t plane, int64_t pix, float* im, float* fT,
                                              uint32_t* nc, float4* __restrict__ cpp, uint32_t* __restrict__ clp,
                                              float bg0, float bg1, float bg2, int& cstar) {
  float c0 = im[pix], c1 = im[plane + pix], c2 = im[2 * plane + pix];
  float T = fT[pix];
  const uint32_t lw0 = nc[pix];
  int last = (int)(lw0 & ~STOP_BIT);
  const bool done = (lw0 & STOP_BIT) != 0u;  // a stop in the front is exact
  for (int cb = m; cb < nch && cstar < 0; cb += CB) {
    uint32_t lwv[CB];
    float4 ptv[CB];
    #pragma unroll
    for (int q = 0; q < CB; ++q) {
      int c = cb + q;
      if (c < nch && !done) {
        lwv[q] = clp[(int64_t)(c - 1) * TILE_PIX];
        ptv[q] = cpp[(int64_t)(c - 1) * TILE_PIX];
      }
    }
    #pragma unroll
    for (int q = 0; q < CB; ++q) {
      int c = cb + q;
      if (c >= nch || cstar >= 0) break;
      clp[(int64_t)(c - 1) * TILE_PIX] = __float_as_uint(T);  // T in front of chunk c (final once done)
      if (done) continue;
      float4 pt = ptv[q];
      float Tn = T * pt.x;
      if ((lwv[q] & STOP_BIT) == 0u && !(Tn < T_MIN)) {
        c0 += T * pt.y; c1 += T * pt.z; c2 += T * pt.w;
        T = Tn;
        uint32_t lc = lwv[q] & ~STOP_BIT;
        if (lc) last = (int)lc;
      } else {
        cstar = c;  // the stop pass walks chunk c for this pixel and writes the rest
      }
    }
  }
  if (cstar >= 1) {
    // boundaries in front of the stop chunk: S_b = A_b + B_b S_c* (the stop pass knows S_c*)
    float A0 = 0.f, A1 = 0.f, A2 = 0.f, B = 1.f;
    for (int bb = cstar - 1; bb >= 1; bb -= CB) {
      float4 ptv[CB];
      #pragma unroll
      for (int q = 0; q < CB; ++q)
        if (bb - q >= 1) ptv[q] = cpp[(int64_t)(bb - q - 1) * TILE_PIX];
      #pragma unroll
      for (int q = 0; q < CB; ++q) {
        if (bb - q < 1) break;
        float4 pt = ptv[q];
        A0 = pt.y + pt.x * A0; A1 = pt.z + pt.x * A1; A2 = pt.w + pt.x * A2;
        B = pt.x * B;
        cpp[(int64_t)(bb - q - 1) * TILE_PIX] = make_float4(B, A0, A1, A2);
      }
    }
    im[pix] = c0; im[plane + pix] = c1; im[2 * plane + pix] = c2;
    fT[pix] = T;
    clp[(int64_t)(cstar - 1) * TILE_PIX] = (uint32_t)last;  // the stop pass reads it and puts T back
    nc[pix] = (uint32_t)cstar | REWALK_BIT;
  } else {
    // checkpoint b: (T in front of chunk b, colour behind boundary b per unit T there); a pixel that
    // stopped in the front has the background behind every boundary from chunk m on
    float S0 = bg0, S1 = bg1, S2 = bg2;
    if (done)
      for (int b = nch - 1; b >= m; --b) cpp[(int64_t)(b - 1) * TILE_PIX] = make_float4(T, bg0, bg1, bg2);
    close_checkpoints(cpp, clp, 1, done ? m - 1 : nch - 1, S0, S1, S2);
    im[pix] = c0 + T * bg0;
    im[plane + pix] = c1 + T * bg1;
    im[2 * plane + pix] = c2 + T * bg2;
    fT[pix] = T;
    nc[pix] = (uint32_t)last;
  }
}

// Combine pass: one warp per queued block; the entry of its first queued chunk
// stands for it (a block's entries are consecutive, so it is one whose
// predecessor is not the same block's previous chunk).  The first block also
// zeroes the stop pass's ticket.
template <int BW>
__global__ void __launch_bounds__(32) k_render_fwd_combine(const uint32_t* __restrict__ order,
                                                           const uint32_t* __restrict__ job_base,
                                                           const uint32_t* __restrict__ jobs,
                                                           float4* __restrict__ ckpt,
                                                           uint32_t* __restrict__ chunk_last, int W, int H, int TX,
                                                           int n_tiles, float bg0, float bg1, float bg2,
                                                           float* __restrict__ img, float* __restrict__ final_T,
                                                           uint32_t* __restrict__ n_contrib,
                                                           uint32_t* __restrict__ queue, uint32_t qcap,
                                                           uint32_t* __restrict__ ticket) {
  gs_wait_previous();
  if (blockIdx.x == 0 && threadIdx.x == 0) *ticket = 0u;
  const uint32_t total = queue[qcap];
  for (uint32_t e = blockIdx.x; e < total; e += gridDim.x) {
    const uint32_t ent = queue[e] & ~MARK_BIT;  // (marks are set by the warp of the entry's block)
    if (e > 0 && ((queue[e - 1] & ~MARK_BIT) + 8u) == ent) continue;
    const uint32_t jid = ent >> 3;
    const int w = (int)(ent & 7u), o = (int)jobs[2 * (int64_t)jid], m = (int)jobs[2 * (int64_t)jid + 1];
    const uint32_t jb = job_base[o];
    const int nch = (int)(job_base[o + 1] - jb);
    PixelOf<BW> P(order, o, w, n_tiles, TX, W, H);
    const int64_t plane = (int64_t)W * H, pix = (int64_t)P.py * W + P.px, cp0 = (int64_t)jb - o;
    int cstar = -1;
    if (P.inside)
      combine_pixel(m, nch, plane, pix, img + (int64_t)P.u * 3 * plane, final_T + (int64_t)P.u * plane,
                    n_contrib + (int64_t)P.u * plane, ckpt + cp0 * TILE_PIX + P.pix_local,
                    chunk_last + cp0 * TILE_PIX + P.pix_local, bg0, bg1, bg2, cstar);
    // mark the block's queue entries the stop pass walks: one per distinct stop chunk of its pixels
    const unsigned peers = __match_any_sync(0xffffffffu, cstar);
    if (cstar >= 1 && (int)(threadIdx.x & 31) == __ffs(peers) - 1) queue[e + (uint32_t)(cstar - m)] |= MARK_BIT;
    __syncwarp();
  }
}

// Stop pass: the marked queue entries, (list o, chunk c, block w) with some
// pixel of block w stopping in chunk c: walks chunk c again for those pixels
// from the state the combine left, and writes their final image, final_T,
// n_contrib and the checkpoints after c (final state).
template <int BW>
__global__ void __launch_bounds__(32) k_render_fwd_stop(const uint2* __restrict__ ranges,
                                                              const uint32_t* __restrict__ order,
                                                              const uint32_t* __restrict__ job_base,
                                                              const uint32_t* __restrict__ jobs, int K,
                                                              float4* __restrict__ ckpt,
                                                              uint32_t* __restrict__ chunk_last,
                                                              const uint32_t* __restrict__ vals,
                                                              const uint16_t* __restrict__ masks,
                                                              const float4* __restrict__ xy,
                                                              const float4* __restrict__ conic_op,
                                                              const float4* __restrict__ rgb, int W, int H, int TX,
                                                              int n_tiles, float bg0, float bg1, float bg2,
                                                              float* __restrict__ img, float* __restrict__ final_T,
                                                              uint32_t* __restrict__ n_contrib,
                                                              const uint32_t* __restrict__ queue, uint32_t qcap,
                                                              uint32_t* __restrict__ ticket) {
  gs_wait_previous();
  __shared__ FwdScratch s_walk;
  const uint32_t total = queue[qcap];
  auto job = [&](uint32_t ent) {
    uint32_t jid = ent >> 3;
    int o = (int)jobs[2 * (int64_t)jid], ch = (int)jobs[2 * (int64_t)jid + 1];
    if (ch == 0) return;
    int nch = (int)(job_base[o + 1] - job_base[o]);
    int w = (int)(ent & 7u);
    PixelOf<BW> P(order, o, w, n_tiles, TX, W, H);
    uint2 rg = ranges[(int64_t)P.u * n_tiles + P.tile];
    int L = (int)(rg.y - rg.x);
    int64_t plane = (int64_t)W * H;
    int64_t pix = (int64_t)P.py * W + P.px;
    float* im = img + (int64_t)P.u * 3 * plane;
    float* fT = final_T + (int64_t)P.u * plane;
    uint32_t* nc = n_contrib + (int64_t)P.u * plane;
    bool mine = false;
    float T = 1.f, c0 = 0.f, c1 = 0.f, c2 = 0.f;
    int last = 0;
    int64_t cp0 = (int64_t)job_base[o] - o;
    if (P.inside) {
      uint32_t lw = nc[pix];
      mine = (lw & REWALK_BIT) != 0u && (int)(lw & ~REWALK_BIT) == ch;
      if (mine) {
        last = (int)chunk_last[(cp0 + ch - 1) * TILE_PIX + P.pix_local];  // left there by the combine
        c0 = im[pix]; c1 = im[plane + pix]; c2 = im[2 * plane + pix];
        T = fT[pix];
      }
    }
    // only the 4x4 pixel blocks of this warp's walking pixels: records whose block mask misses them
    // cannot reach those pixels
    uint32_t my_block = mine ? 1u << (4 * ((P.py - P.ty * TILE) >> 2) + ((P.px - P.tx * TILE) >> 2)) : 0u;
    uint32_t wbits = __reduce_or_sync(0xffffffffu, my_block);
    if (!wbits) return;
    bool done = !mine;
    // walk chunk c* (and, should the pixel not stop there after all, the chunks after it), keeping each
    // walked chunk's partial and the T in front of it; chunks behind the stop get the identity partial
    int c = ch;
    for (; c < nch; ++c) {
      walk_chunk<BW>(vals, masks, xy, conic_op, rgb, rg.x, c * K, min(c * K + K, L), wbits, (float)(P.tx * TILE),
                     (float)(P.ty * TILE), (float)P.ox, (float)P.oy, s_walk, T, c0, c1, c2, last, done, mine,
                     ckpt + (cp0 + c - 1) * TILE_PIX + P.pix_local, chunk_last + (cp0 + c - 1) * TILE_PIX + P.pix_local);
      if (__all_sync(0xffffffffu, done)) break;
    }
    if (!mine) return;
    // checkpoints: (T in front of boundary b, colour behind it per unit T), composited back to front
    float4* cpp = ckpt + cp0 * TILE_PIX + P.pix_local;  // slot of boundary b: cpp[(b - 1) * TILE_PIX]
    const uint32_t* clp = chunk_last + cp0 * TILE_PIX + P.pix_local;
    for (int b = nch - 1; b > c; --b)
      cpp[(int64_t)(b - 1) * TILE_PIX] = make_float4(T, bg0, bg1, bg2);  // behind the stop: final state
    float S0 = bg0, S1 = bg1, S2 = bg2;
    close_checkpoints(cpp, clp, ch, min(c, nch - 1), S0, S1, S2);  // walked chunks
    for (int bb = 1; bb < ch; bb += CB) {  // in front of c*: S_b = A_b + B_b S_c* as left by the combine
      float4 abv[CB];
      uint32_t tv[CB];
      #pragma unroll
      for (int q = 0; q < CB; ++q)
        if (bb + q < ch) {
          abv[q] = cpp[(int64_t)(bb + q - 1) * TILE_PIX];
          tv[q] = clp[(int64_t)(bb + q - 1) * TILE_PIX];
        }
      #pragma unroll
      for (int q = 0; q < CB; ++q) {
        if (bb + q >= ch) break;
        float4 ab = abv[q];
        cpp[(int64_t)(bb + q - 1) * TILE_PIX] = make_float4(__uint_as_float(tv[q]), ab.y + ab.x * S0,
                                                            ab.z + ab.x * S1, ab.w + ab.x * S2);
      }
    }
    im[pix] = c0 + T * bg0;
    im[plane + pix] = c1 + T * bg1;
    im[2 * plane + pix] = c2 + T * bg2;
    fT[pix] = T;
    nc[pix] = (uint32_t)last;
  };
  const bool lead = (threadIdx.x & 31) == 0;
  uint32_t e = __shfl_sync(0xffffffffu, lead ? atomicAdd(ticket, 1u) : 0u, 0);
  while (e < total) {
    uint32_t nxt = lead ? atomicAdd(ticket, 1u) : 0u;
    const uint32_t ent = queue[e];
    if (ent & MARK_BIT) job(ent & ~MARK_BIT);
    e = __shfl_sync(0xffffffffu, nxt, 0);
  }
}


// Lanes of a warp's pixel block (bw x 32 / bw pixels from tile-local origin
// (ox, oy), lane = row bw + column) whose pixel centre lies in a record's
// alpha >= 1/255 box (alpha_box: conservative, so every pixel outside it has
// alpha < 1/255 and would be skipped by the blend).  (rx, ry): the record's
// tile-local position; co: conic and opacity.
__device__ __forceinline__ uint32_t hit_lanes(float rx, float ry, float4 co, float ox, float oy, int bw) {
  float pm;
  const float4 b = alpha_box(make_float2(rx, ry), co, pm);
  if (!(b.x <= b.y)) return 0u;
  const int bh = 32 / bw;
  const float c0 = fmaxf(ceilf(b.x - ox), 0.f), c1 = fminf(floorf(b.y - ox), (float)(bw - 1));
  const float r0 = fmaxf(ceilf(b.z - oy), 0.f), r1 = fminf(floorf(b.w - oy), (float)(bh - 1));
  if (!(c0 <= c1) || !(r0 <= r1)) return 0u;
  const int lo = (int)c0, rl = (int)r0, rh = (int)r1;
  const uint32_t cm = ((2u << ((int)c1 - lo)) - 1u) << lo;
  uint32_t m = 0u;
  for (int r = rl; r <= rh; ++r) m |= cm << (r * bw);
  return m;
}

// Contributing lanes up to which the scheduled backward skips the warp
// reduction of a record's nine gradient values and lets each lane issue its
// own vector atomics.  L2 absorbs these well: at 1M and 10M Gaussians per
// 1080p view every threshold from 3 to 32 was faster than the one below it;
// 16 keeps the same-address atomics of a record bounded for large splats.
constexpr int DIRECT_LANES = 16;

// Position and conic terms of one (pixel, record) pair's gradient from the
// pixel offset (dx, dy), dp = o G dL/dalpha and the conic (A, B, C):
// v = (dx, dy | dA, dB, dC) in the order add_lane expects.
__device__ __forceinline__ void pos_conic_terms(float dx, float dy, float dp, float A, float B, float Cc, float* v) {
  v[2] = -0.5f * dx * dx * dp;
  v[3] = -dx * dy * dp;
  v[4] = -0.5f * dy * dy * dp;
  v[0] = -(A * dx + B * dy) * dp;
  v[1] = -(Cc * dy + B * dx) * dp;
}

// Rounds with at least this many hits walk per-lane hit lists: each lane takes
// only the hits whose alpha box reaches its pixel.  Below it the box and the
// transpose cost more than the hits they spare (10M Gaussians at 1080p,
// thresholds swept over 1-24).
constexpr int HIT_LISTS_BWD = 8;

// Ring of deferred (pixel, record) pairs of the scheduled backward, per warp.
constexpr int QCAP = 64;

// Lanes 0..count-1 finish entries head .. head + count - 1 of the ring: the
// position and conic terms, then the record's three vector atomics.
__device__ __forceinline__ void bwd_queue_flush(const float4* s_q, int head, int count, int lane, float* dxy,
                                                float* dco, float* drgb) {
  if (lane < count) {
    int e = (head + lane) & (QCAP - 1);
    float4 a = s_q[e], b = s_q[QCAP + e], c = s_q[2 * QCAP + e];
    float v[5];
    pos_conic_terms(a.x, a.y, a.z, b.x, b.y, b.z, v);
    int64_t pr = (int64_t)__float_as_uint(b.w);
    atomic_add2(dxy + 2 * pr, v[0], v[1]);
    atomic_add4(dco + 4 * pr, v[2], v[3], v[4], a.w);
    atomic_add4(drgb + 4 * pr, c.x, c.y, c.z, 0.f);
  }
}

// Backward over chunk jobs: job (list, chunk c, pixel block) replays entries
// [c K, min((c + 1) K, L)) of the list back to front.  It starts from the
// forward's checkpoint at the chunk's end (T in front of it and the colour
// behind it per unit T), or from final_T and the background for the last
// chunk.  Masks and ids are read two rounds of 32 entries ahead, hit records one
// round ahead.  The gradient terms of sparse hits go through a per-warp ring
// (float accumulation; k_render_bwd_det has the deterministic one).
template <int BW>
__global__ void __launch_bounds__(32, 32) k_render_bwd_m(const uint2* __restrict__ ranges,
                                                           const uint32_t* __restrict__ order,
                                                           const uint32_t* __restrict__ job_base,
                                                           const uint32_t* __restrict__ jobs, int K,
                                                           const float4* __restrict__ ckpt,
                                                           const uint32_t* __restrict__ vals,
                                                           const uint16_t* __restrict__ masks,
                                                           const float4* __restrict__ xy,
                                                           const float4* __restrict__ conic_op,
                                                           const float4* __restrict__ rgb, int W, int H, int TX,
                                                           int n_tiles, int NT, float bg0, float bg1, float bg2,
                                                           const float* __restrict__ img,
                                                           const float* __restrict__ final_T,
                                                           const uint32_t* __restrict__ n_contrib,
                                                           const float* __restrict__ dimg,
                                                           const float* __restrict__ dLdT, float* __restrict__ dxy,
                                                           float* __restrict__ dco, float* __restrict__ drgb,
                                                           uint32_t* __restrict__ ticket) {
  gs_wait_previous();
  const unsigned FULL = 0xffffffffu;
  __shared__ Rec s_rec[32];
  // the resident warps take the (chunk job, pixel block) units from a ticket counter (zeroed before
  // the launch), the next ticket fetched while a unit runs: no block of a grid sized for the capacity
  // sits idle, and units of very different cost still spread as they finish
  const uint32_t total = job_base[NT] * 8u;
  auto job = [&](uint32_t vb) {
    uint32_t jid = vb >> 3;
    int w = (int)(vb & 7u);
    int o = (int)jobs[2 * (int64_t)jid], ch = (int)jobs[2 * (int64_t)jid + 1];
    uint32_t f = order[o];
    int u = (int)(f / (uint32_t)n_tiles), tile = (int)(f % (uint32_t)n_tiles);
    int nch = (int)(job_base[o + 1] - job_base[o]);
    int tx = tile % TX, ty = tile / TX;
    constexpr int BH = 32 / BW, NWX = TILE / BW;
    int lane = threadIdx.x & 31;
    int px = tx * TILE + (w % NWX) * BW + (lane % BW), py = ty * TILE + (w / NWX) * BH + (lane / BW);
    uint32_t wbits = warp_block_bits<BW>(w);
    bool inside = px < W && py < H;
    float tox = (float)(tx * TILE), toy = (float)(ty * TILE);  // origin of the staged record positions
    float lx = (float)(px - tx * TILE), ly = (float)(py - ty * TILE);
    uint2 rg = ranges[(int64_t)u * n_tiles + tile];
    int L = (int)(rg.y - rg.x);
    int cbeg = ch * K, cend = min(cbeg + K, L);
    int64_t plane = (int64_t)W * H;
    int64_t pix = (int64_t)py * W + px;
    float T = 1.f, g0 = 0.f, g1 = 0.f, g2 = 0.f, S0 = bg0, S1 = bg1, S2 = bg2;
    float qT = 0.f;  // dL/dT_final x T_final: a blended entry adds -qT / (1 - alpha) to dL/dalpha
    int last = 0;
    if (inside) last = (int)n_contrib[(int64_t)u * plane + pix];
    // entries this warp replays: [cbeg, min(cend, max over its pixels of last)); a chunk behind the last stop has none
    const int n = min(__reduce_max_sync(FULL, last), cend);
    if (n <= cbeg) return;
    if (inside) {
      const float* d = dimg + (int64_t)u * 3 * plane;
      g0 = d[pix]; g1 = d[plane + pix]; g2 = d[2 * plane + pix];
      if (dLdT) qT = dLdT[(int64_t)u * plane + pix] * final_T[(int64_t)u * plane + pix];
      if (ch + 1 < nch && last > cbeg) {
        // the forward's checkpoint at the chunk's end: T there and the colour behind it per unit T
        int pix_local = (py - ty * TILE) * TILE + (px - tx * TILE);
        float4 cp = ckpt[((int64_t)job_base[o] - o + ch) * TILE_PIX + pix_local];
        T = cp.x;
        S0 = cp.y; S1 = cp.z; S2 = cp.w;
      } else {
        T = final_T[(int64_t)u * plane + pix];
      }
    }
    Rec* my = &s_rec[0];
    int q = ((lane >> 4) & 1) * 4 + ((lane >> 3) & 1) * 2 + ((lane >> 2) & 1);
    bool h1 = false;
    uint32_t p1 = 0;
    float4 m1 = make_float4(0.f, 0.f, 0.f, 0.f);
    float4 co1 = make_float4(0.f, 0.f, 0.f, 0.f), cc1 = co1;
    uint32_t mk2 = 0, pk2 = 0;
    {
      int k = n - 32 + lane;
      if (n > cbeg && k >= cbeg) {
        uint32_t mk = masks[rg.x + k];
        if (mk & wbits) {
          p1 = vals[rg.x + k];
          h1 = true; m1 = xy[p1]; co1 = conic_op[p1]; cc1 = rgb[p1];
        }
      }
      int k2 = n - 64 + lane;
      if (n - 32 > cbeg && k2 >= cbeg) { mk2 = masks[rg.x + k2]; pk2 = vals[rg.x + k2]; }
    }
    // pairs of hits with at most DIRECT_LANES contributing lanes go to a ring of
    // (dx, dy, dp, dopacity | A, B, C, id | dr, dg, db) entries; every 32 entries all
    // lanes finish one pair each (conic and position terms, vector atomics).  The
    // per-pixel state (T, colour behind) is still updated at the hit in list order.
    __shared__ float4 s_q[3 * QCAP];
    int qh = 0, qt = 0;  // ring head and tail (warp-uniform)
    for (int top = n; top > cbeg; top -= 32) {
      int base = top - 32;
      bool hit = h1;
      uint32_t p = p1;
      float4 m = m1;
      float4 co = co1, c = cc1;
      h1 = (mk2 & wbits) != 0;
      if (h1) { p1 = pk2; m1 = xy[pk2]; co1 = conic_op[pk2]; cc1 = rgb[pk2]; }
      int k2 = top - 96 + lane;
      mk2 = 0;
      if (top - 64 > cbeg && k2 >= cbeg) { mk2 = masks[rg.x + k2]; pk2 = vals[rg.x + k2]; }
      unsigned mask = __ballot_sync(FULL, hit);
      const float rx = rel_pos(m.x, m.z, tox), ry = rel_pos(m.y, m.w, toy);
      if (hit) {
        my[lane].a = make_float4(rx, ry, co.x, co.y);
        my[lane].b = make_float4(co.z, co.w, c.w, __uint_as_float(p));
        my[lane].c = c;
      }
      __syncwarp();
      if (__popc(mask) >= HIT_LISTS_BWD) {
        // per-lane hit lists, back to front: bit j of `mine` = hit j's alpha box reaches this lane's
        // pixel and the entry lies in front of the pixel's last contribution; every pair goes to the ring
        uint32_t mine = transpose32(hit ? hit_lanes(rx, ry, co, (float)((w % NWX) * BW), (float)((w / NWX) * BH), BW)
                                        : 0u);
        const int upto = last - base;
        mine &= upto >= 32 ? 0xffffffffu : (upto > 0 ? (1u << upto) - 1u : 0u);
        while (__any_sync(FULL, mine != 0u)) {
          const bool act = mine != 0u;
          const int j = act ? 31 - __clz(mine) : 0;
          if (act) mine &= ~(1u << j);
          bool contrib = false;
          float dx = 0.f, dy = 0.f, dp = 0.f, v5 = 0.f, v6 = 0.f, v7 = 0.f, v8 = 0.f;
          float4 ra = my[j].a, rb = my[j].b;
          if (act) {
            dx = ra.x - lx; dy = ra.y - ly;
            float power = splat_power(ra.z, ra.w, rb.x, dx, dy);
            if (power <= 0.f && power >= rb.z) {
              float G = __expf(power);
              float araw = rb.y * G;
              bool clamped = araw > ALPHA_MAX;
              float alpha = clamped ? ALPHA_MAX : araw;
              if (alpha >= ALPHA_MIN) {
                contrib = true;
                float4 rc = my[j].c;
                T = __fdividef(T, 1.f - alpha);
                float wgt = alpha * T;
                v6 = wgt * g0; v7 = wgt * g1; v8 = wgt * g2;
                float dalpha = T * ((rc.x - S0) * g0 + (rc.y - S1) * g1 + (rc.z - S2) * g2);
                if (qT != 0.f) dalpha -= __fdividef(qT, 1.f - alpha);
                S0 = alpha * rc.x + (1.f - alpha) * S0;
                S1 = alpha * rc.y + (1.f - alpha) * S1;
                S2 = alpha * rc.z + (1.f - alpha) * S2;
                if (!clamped) {
                  v5 = G * dalpha;
                  dp = araw * dalpha;
                }
              }
            }
          }
          unsigned cm = __ballot_sync(FULL, contrib);
          if (!cm) continue;
          if (contrib) {
            int e = (qt + __popc(cm & ((1u << lane) - 1u))) & (QCAP - 1);
            s_q[e] = make_float4(dx, dy, dp, v5);
            s_q[QCAP + e] = make_float4(ra.z, ra.w, rb.x, rb.w);
            s_q[2 * QCAP + e] = make_float4(v6, v7, v8, 0.f);
          }
          qt += __popc(cm);
          if (qt - qh >= 32) {
            __syncwarp();
            bwd_queue_flush(s_q, qh, 32, lane, dxy, dco, drgb);
            qh += 32;
            __syncwarp();
          }
        }
        mask = 0u;  // every hit of the round is done
      }
      while (mask) {
        int j = 31 - __clz(mask);
        mask &= ~(1u << j);
        int pos = base + j;
        bool contrib = false;
        float dx = 0.f, dy = 0.f, dp = 0.f, v5 = 0.f, v6 = 0.f, v7 = 0.f, v8 = 0.f;
        float4 ra = my[j].a, rb = my[j].b;
        if (pos < last) {
          dx = ra.x - lx; dy = ra.y - ly;
          float power = splat_power(ra.z, ra.w, rb.x, dx, dy);
          if (power <= 0.f && power >= rb.z) {
            float G = __expf(power);
            float araw = rb.y * G;
            bool clamped = araw > ALPHA_MAX;
            float alpha = clamped ? ALPHA_MAX : araw;
            if (alpha >= ALPHA_MIN) {
              contrib = true;
              float4 rc = my[j].c;
              T = __fdividef(T, 1.f - alpha);
              float wgt = alpha * T;
              v6 = wgt * g0; v7 = wgt * g1; v8 = wgt * g2;
              float dalpha = T * ((rc.x - S0) * g0 + (rc.y - S1) * g1 + (rc.z - S2) * g2);
              if (qT != 0.f) dalpha -= __fdividef(qT, 1.f - alpha);
              S0 = alpha * rc.x + (1.f - alpha) * S0;
              S1 = alpha * rc.y + (1.f - alpha) * S1;
              S2 = alpha * rc.z + (1.f - alpha) * S2;
              if (!clamped) {  // a clamped alpha passes no gradient to opacity, conic or position
                v5 = G * dalpha;
                dp = araw * dalpha;
              }
            }
          }
        }
        unsigned cm = __ballot_sync(FULL, contrib);
        if (!cm) continue;
        int nc = __popc(cm);
        if (nc <= DIRECT_LANES) {
          if (contrib) {
            int e = (qt + __popc(cm & ((1u << lane) - 1u))) & (QCAP - 1);
            s_q[e] = make_float4(dx, dy, dp, v5);
            s_q[QCAP + e] = make_float4(ra.z, ra.w, rb.x, rb.w);
            s_q[2 * QCAP + e] = make_float4(v6, v7, v8, 0.f);
          }
          qt += nc;
          if (qt - qh >= 32) {
            __syncwarp();
            bwd_queue_flush(s_q, qh, 32, lane, dxy, dco, drgb);
            qh += 32;
            __syncwarp();
          }
          continue;
        }
        int64_t pr = (int64_t)__float_as_uint(rb.w);
        float v[9];
        pos_conic_terms(dx, dy, dp, ra.z, ra.w, rb.x, v);
        v[5] = v5; v[6] = v6; v[7] = v7; v[8] = v8;
        {
          float tot = reduce8(v, lane);
          float e8 = v[8];
          #pragma unroll
          for (int oo = 16; oo > 0; oo >>= 1) e8 += __shfl_xor_sync(FULL, e8, oo);
          if ((lane & 3) == 0) {
            add_one(dxy, dco, drgb, nullptr, pr, q, tot);
          } else if (lane == 1) {
            add_one(dxy, dco, drgb, nullptr, pr, 8, e8);
          }
        }
      }
      __syncwarp();
    }
    if (qt > qh) bwd_queue_flush(s_q, qh, qt - qh, lane, dxy, dco, drgb);
  };
  const bool lead = (threadIdx.x & 31) == 0;
  uint32_t vb = __shfl_sync(0xffffffffu, lead ? atomicAdd(ticket, 1u) : 0u, 0);
  while (vb < total) {
    uint32_t nxt = lead ? atomicAdd(ticket, 1u) : 0u;
    job(vb);
    vb = __shfl_sync(0xffffffffu, nxt, 0);
  }
}

struct __align__(16) BwdScratch {
  float w[32 * MROW];   // o G of an accepted (hit, pixel) pair, then its colour weight alpha T (few hits: their Rec)
  float dp[32 * MROW];  // dL/dpower of the pair (0 when alpha was clamped)
  float r[32], g[32], b[32];     // the batch's colours
  float g0[32], g1[32], g2[32];  // dL/dimg of the block's pixels
  uint32_t q[QUEUE_CAP];
};

// The deterministic backward over the same chunk jobs.  Its cost is the int64
// atomics, nine per record and addition, so it sums each hit over the block's
// pixels first: hits are gathered back to front into batches of 32 and
// evaluated record-major, then replayed pixel-major, as in the forward walk;
// the replay leaves each pair's colour weight alpha T and dL/dpower in shared
// memory, and a third, record-major phase forms the pairs' gradients and sums
// them in its lane's registers, in pixel order, so that nothing depends on
// scheduling.  700k at 1011x757: 578 us with a warp reduction per hit, 240 us.
// A record-major phase lasts as long as the widest hit has pixels (32 where it
// covers the block), however few hits there are, so batches of up to FEW_HITS
// take the warp reduction per hit.  Lists of 3 entries of some pixels each, at
// 1080p: 74 us record-major, 42 this way (39 with a reduction for every hit); of
// 6 entries 79, 50 (45); up to 4, 6, 8 and 12 hits the worst of 150 scenes took
// 1.36, 1.19, 1.12 and 1.06 times what reductions throughout take, but with 12
// some scenes more than record-major phases throughout (1.14; 1.05 with 8).
constexpr int FEW_HITS = 8;
template <int BW>
__global__ void __launch_bounds__(32, 20) k_render_bwd_det(const uint2* __restrict__ ranges,
                                                           const uint32_t* __restrict__ order,
                                                           const uint32_t* __restrict__ job_base,
                                                           const uint32_t* __restrict__ jobs, int K,
                                                           const float4* __restrict__ ckpt,
                                                           const uint32_t* __restrict__ vals,
                                                           const uint16_t* __restrict__ masks,
                                                           const float4* __restrict__ xy,
                                                           const float4* __restrict__ conic_op,
                                                           const float4* __restrict__ rgb, int W, int H, int TX,
                                                           int n_tiles, int NT, float bg0, float bg1, float bg2,
                                                           const float* __restrict__ img,
                                                           const float* __restrict__ final_T,
                                                           const uint32_t* __restrict__ n_contrib,
                                                           const float* __restrict__ dimg,
                                                           const float* __restrict__ dLdT,
                                                           unsigned long long* __restrict__ fixed,
                                                           uint32_t* __restrict__ ticket) {
  gs_wait_previous();
  const unsigned FULL = 0xffffffffu;
  __shared__ BwdScratch sc;
  // the resident warps take the (chunk job, pixel block) units from a ticket counter (zeroed before
  // the launch), the next ticket fetched while a unit runs: no block of a grid sized for the capacity
  // sits idle, and units of very different cost still spread as they finish
  const uint32_t total = job_base[NT] * 8u;
  auto job = [&](uint32_t vb) {
    uint32_t jid = vb >> 3;
    int w = (int)(vb & 7u);
    int o = (int)jobs[2 * (int64_t)jid], ch = (int)jobs[2 * (int64_t)jid + 1];
    PixelOf<BW> P(order, o, w, n_tiles, TX, W, H);
    int nch = (int)(job_base[o + 1] - job_base[o]);
    const int lane = threadIdx.x & 31;
    const float tox = (float)(P.tx * TILE), toy = (float)(P.ty * TILE);  // origin of the record positions
    const float ox = (float)P.ox, oy = (float)P.oy, bx = 8388608.f - ox, by = 8388608.f - oy;
    uint2 rg = ranges[(int64_t)P.u * n_tiles + P.tile];
    int L = (int)(rg.y - rg.x);
    int cbeg = ch * K, cend = min(cbeg + K, L);
    int64_t plane = (int64_t)W * H;
    int64_t pix = (int64_t)P.py * W + P.px;
    float T = 1.f, g0 = 0.f, g1 = 0.f, g2 = 0.f, S0 = bg0, S1 = bg1, S2 = bg2;
    float qT = 0.f;  // dL/dT_final x T_final: a blended entry adds -qT / (1 - alpha) to dL/dalpha
    // entries this warp replays: [cbeg, min(cend, max over its pixels of last))
    const int last = P.inside ? (int)n_contrib[(int64_t)P.u * plane + pix] : 0;
    const int n = min(__reduce_max_sync(FULL, last), cend);
    if (n <= cbeg) return;
    if (P.inside) {
      const float* d = dimg + (int64_t)P.u * 3 * plane;
      g0 = d[pix]; g1 = d[plane + pix]; g2 = d[2 * plane + pix];
      if (dLdT) qT = dLdT[(int64_t)P.u * plane + pix] * final_T[(int64_t)P.u * plane + pix];
      if (ch + 1 < nch && last > cbeg) {
        // the forward's checkpoint at the chunk's end: T there and the colour behind it per unit T
        float4 cp = ckpt[((int64_t)job_base[o] - o + ch) * TILE_PIX + P.pix_local];
        T = cp.x;
        S0 = cp.y; S1 = cp.z; S2 = cp.w;
      } else {
        T = final_T[(int64_t)P.u * plane + pix];
      }
    }
    sc.g0[lane] = g0; sc.g1[lane] = g1; sc.g2[lane] = g2;
    const uint32_t act = __ballot_sync(FULL, last > cbeg);  // pixels with an entry to replay
    const uint32_t* lv = vals + rg.x;
    const uint16_t* lm = masks + rg.x;
    int scan = n - 1, qn = 0, qh = 0;  // next entry to scan (downwards); queued entries are q[qh .. qn)
    for (;;) {
      if (qn - qh < 32 && scan >= cbeg) {
        const uint32_t keep = qh + lane < qn ? sc.q[qh + lane] : 0u;
        __syncwarp();
        qn -= qh;
        qh = 0;
        if (lane < qn) sc.q[lane] = keep;
        do {
          qn = scan_hits<true>(lm, scan, cbeg, P.wbits, sc.q, qn);
          scan -= SCAN;
        } while (qn < 32 && scan >= cbeg);
        __syncwarp();
      }
      const int nb = min(32, qn - qh);
      if (nb == 0) break;
      if (nb <= FEW_HITS) {
        // each lane its own pixel's share of every hit, summed over the warp per hit
        Rec* rec = reinterpret_cast<Rec*>(sc.w);
        if (lane < nb) {
          const uint32_t id = lv[sc.q[qh + lane]];
          const float4 m = xy[id], k = conic_op[id];
          rec[lane].a = make_float4(rel_pos(m.x, m.z, tox), rel_pos(m.y, m.w, toy), k.x, k.y);
          rec[lane].b = make_float4(k.z, k.w, 0.f, __uint_as_float(id));
          rec[lane].c = rgb[id];
        }
        __syncwarp();
        for (int j = 0; j < nb; ++j) {
          const float4 ra = rec[j].a, rb = rec[j].b;
          const float dx = ra.x - (ox + (float)(lane & (BW - 1))), dy = ra.y - (oy + (float)(lane / BW));
          const float power = splat_power(ra.z, ra.w, rb.x, dx, dy);
          const float G = __expf(power), araw = rb.y * G;
          const bool clamped = araw > ALPHA_MAX;  // a clamped alpha passes no gradient to opacity, conic or position
          const float alpha = clamped ? ALPHA_MAX : araw;
          const bool pair = !(power > 0.f) && !(alpha < ALPHA_MIN) && (int)sc.q[qh + j] < last;
          const unsigned cm = __ballot_sync(FULL, pair);
          if (!cm) continue;
          float v[9];
          #pragma unroll
          for (int e = 0; e < 9; ++e) v[e] = 0.f;
          if (pair) {
            const float4 rc = rec[j].c;
            const float om = 1.f - alpha;
            T = __fdividef(T, om);  // transmittance in front of this entry
            const float wgt = alpha * T;
            v[6] = wgt * g0; v[7] = wgt * g1; v[8] = wgt * g2;
            float dalpha = T * ((rc.x - S0) * g0 + (rc.y - S1) * g1 + (rc.z - S2) * g2);
            if (qT != 0.f) dalpha -= __fdividef(qT, om);
            S0 = alpha * rc.x + om * S0; S1 = alpha * rc.y + om * S1; S2 = alpha * rc.z + om * S2;
            if (!clamped) {
              v[5] = G * dalpha;
              pos_conic_terms(dx, dy, araw * dalpha, ra.z, ra.w, rb.x, v);
            }
          }
          const int64_t id = (int64_t)__float_as_uint(rb.w);
          if ((cm & (cm - 1)) == 0) {
            if (pair) add_lane(nullptr, nullptr, nullptr, fixed, id, v);
          } else {
            const float tot = reduce8(v, lane);
            float e8 = v[8];
            #pragma unroll
            for (int d = 16; d > 0; d >>= 1) e8 += __shfl_xor_sync(FULL, e8, d);
            const int slot = ((lane >> 4) & 1) * 4 + ((lane >> 3) & 1) * 2 + ((lane >> 2) & 1);
            if ((lane & 3) == 0) add_one(nullptr, nullptr, nullptr, fixed, id, slot, tot);
            else if (lane == 1) add_one(nullptr, nullptr, nullptr, fixed, id, 8, e8);
          }
        }
        qh += nb;
        __syncwarp();
        continue;
      }
      // record-major: o G of hit `lane` at the pixels its box reaches
      uint32_t pr = 0u, valid = 0u;
      float rx = 0.f, ry = 0.f;
      float4 co = make_float4(0.f, 0.f, 0.f, 1.f);
      if (lane < nb) {
        pr = lv[sc.q[qh + lane]];
        const float4 m = xy[pr], c = rgb[pr];
        co = conic_op[pr];
        rx = rel_pos(m.x, m.z, tox); ry = rel_pos(m.y, m.w, toy);
        sc.r[lane] = c.x; sc.g[lane] = c.y; sc.b[lane] = c.z;
        valid = eval_hit<BW, false>(rx, ry, co, c.w, ox, oy, act, sc.w + lane * MROW);
      }
      __syncwarp();
      // pixel-major: this pixel's pairs back to front, those in front of its last contribution
      uint32_t mine = transpose32(valid);
      if (mine && (int)sc.q[qh] >= last) {
        int a = 0, b = nb;  // first hit with an entry below `last` (entries fall with j)
        while (a < b) {
          const int mid = (a + b) >> 1;
          if ((int)sc.q[qh + mid] >= last) a = mid + 1; else b = mid;
        }
        mine &= a < 32 ? 0xffffffffu << a : 0u;
      }
      const uint32_t con = mine;
      while (mine) {
        const int j = __ffs(mine) - 1;
        mine &= mine - 1;
        const float araw = sc.w[j * MROW + lane];
        const bool clamped = araw > ALPHA_MAX;  // a clamped alpha passes no gradient to opacity, conic or position
        const float alpha = clamped ? ALPHA_MAX : araw;
        const float om = 1.f - alpha;
        T = __fdividef(T, om);  // transmittance in front of this entry
        const float cr = sc.r[j], cg = sc.g[j], cb = sc.b[j];
        float dalpha = T * ((cr - S0) * g0 + (cg - S1) * g1 + (cb - S2) * g2);
        if (qT != 0.f) dalpha -= __fdividef(qT, om);
        S0 = alpha * cr + om * S0; S1 = alpha * cg + om * S1; S2 = alpha * cb + om * S2;
        sc.w[j * MROW + lane] = alpha * T;
        sc.dp[j * MROW + lane] = clamped ? 0.f : araw * dalpha;
      }
      __syncwarp();
      // record-major: the sums over hit `lane`'s pixels, then its atomics
      uint32_t pm = transpose32(con);
      if (pm) {
        float v[9];
        #pragma unroll
        for (int q = 0; q < 9; ++q) v[q] = 0.f;
        while (pm) {
          const int px = __ffs(pm) - 1;
          pm &= pm - 1;
          const float wgt = sc.w[lane * MROW + px], dp = sc.dp[lane * MROW + px];
          // 2^23 + integer, minus the origin's offset: the pixel's coordinates without an integer conversion
          const float dx = rx - (__int_as_float(0x4b000000 | (px & (BW - 1))) - bx);
          const float dy = ry - (__int_as_float(0x4b000000 | (px / BW)) - by);
          v[0] += (co.x * dx + co.y * dy) * dp;
          v[1] += (co.z * dy + co.y * dx) * dp;
          v[2] += dx * dx * dp; v[3] += dx * dy * dp; v[4] += dy * dy * dp;
          v[5] += dp;
          v[6] += wgt * sc.g0[px]; v[7] += wgt * sc.g1[px]; v[8] += wgt * sc.g2[px];
        }
        v[0] = -v[0]; v[1] = -v[1];
        v[2] *= -0.5f; v[3] = -v[3]; v[4] *= -0.5f;
        v[5] /= co.w;
        add_lane(nullptr, nullptr, nullptr, fixed, (int64_t)pr, v);
      }
      qh += nb;
      __syncwarp();
    }
    __syncwarp();
  };
  const bool lead = (threadIdx.x & 31) == 0;
  uint32_t vb = __shfl_sync(0xffffffffu, lead ? atomicAdd(ticket, 1u) : 0u, 0);
  while (vb < total) {
    uint32_t nxt = lead ? atomicAdd(ticket, 1u) : 0u;
    job(vb);
    vb = __shfl_sync(0xffffffffu, nxt, 0);
  }
}

// Tile order: heaviest lists first (counting sort of (unit, tile) by the
// bit length of the list length; order within a class is arbitrary and the
// blend results do not depend on it).
__global__ void k_order_hist(const uint2* __restrict__ ranges, int n, uint32_t* __restrict__ hist) {
  gs_wait_previous();
  __shared__ uint32_t s[33];
  if (threadIdx.x < 33) s[threadIdx.x] = 0;
  __syncthreads();
  int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) {
    uint2 r = ranges[i];
    uint32_t len = r.y - r.x;
    atomicAdd(&s[32 - __clz(len)], 1u);  // class 0: empty; class c: 2^(c-1) <= len < 2^c
  }
  __syncthreads();
  if (threadIdx.x < 33 && s[threadIdx.x]) atomicAdd(&hist[threadIdx.x], s[threadIdx.x]);
}

__global__ void k_order_scatter(const uint2* __restrict__ ranges, int n, const uint32_t* __restrict__ hist,
                                uint32_t* __restrict__ cursor, uint32_t* __restrict__ order) {
  gs_wait_previous();
  __shared__ uint32_t s_base[33], s_cnt[33];
  if (threadIdx.x < 33) { s_base[threadIdx.x] = hist[threadIdx.x]; s_cnt[threadIdx.x] = 0u; }
  __syncthreads();
  if (threadIdx.x == 0) {
    uint32_t acc = 0;
    for (int c = 32; c >= 0; --c) { const uint32_t h = s_base[c]; s_base[c] = acc; acc += h; }  // heavy classes first
  }
  int i = blockIdx.x * blockDim.x + threadIdx.x;
  int c = 0;
  uint32_t rank = 0u;
  if (i < n) {
    uint2 r = ranges[i];
    c = 32 - __clz(r.y - r.x);
    rank = atomicAdd(&s_cnt[c], 1u);
  }
  __syncthreads();
  // one global atomic per block and class (most lists are empty: one per list queued up on that class's counter)
  if (threadIdx.x < 33 && s_cnt[threadIdx.x]) s_base[threadIdx.x] += atomicAdd(&cursor[threadIdx.x], s_cnt[threadIdx.x]);
  __syncthreads();
  if (i < n) order[s_base[c] + rank] = (uint32_t)i;
}

// Work counters of one rendered view (diagnostic, outside any timed region):
// counts[0] = blended (pixel, record) pairs (records before n_contrib whose
// alpha reaches 1/255); counts[1] = (pixel, list entry) pairs the sequential
// front-to-back walk evaluates, up to and including the entry that stops the
// pixel; counts[2] = sum of n_contrib, the entries the reverse replay walks
// per pixel; counts[3], counts[4] = the pairs of counts[1] and counts[2]
// whose block mask reaches the pixel's 4x4 block (0 without masks): the
// (pixel, entry) pairs a walk that skips masked-out records must evaluate.
__global__ void __launch_bounds__(TILE_PIX) k_blend_pairs(const uint2* __restrict__ ranges,
                                                          const uint32_t* __restrict__ vals,
                                                          const float4* __restrict__ xy,
                                                          const float4* __restrict__ conic_op, int W, int H, int TX,
                                                          int n_tiles, const uint32_t* __restrict__ n_contrib,
                                                          const uint16_t* __restrict__ masks,
                                                          unsigned long long* __restrict__ counts) {
  gs_wait_previous();
  int tile = blockIdx.x, u = blockIdx.y;
  int tx = tile % TX, ty = tile / TX;
  int px = tx * TILE + (threadIdx.x & 15), py = ty * TILE + (threadIdx.x >> 4);
  const uint32_t blk = 1u << (4 * ((threadIdx.x >> 4) >> 2) + ((threadIdx.x & 15) >> 2));
  unsigned long long c = 0, visited = 0, replay = 0, m_visited = 0, m_replay = 0;
  if (px < W && py < H) {
    uint2 rg = ranges[(int64_t)u * n_tiles + tile];
    int L = (int)(rg.y - rg.x);
    int last = (int)n_contrib[(int64_t)u * W * H + (int64_t)py * W + px];
    replay = (unsigned long long)last;
    float T = 1.f;
    int j = 0;
    for (; j < L; ++j) {
      bool in_mask = masks && (masks[rg.x + j] & blk);
      m_visited += in_mask ? 1 : 0;
      m_replay += (in_mask && j < last) ? 1 : 0;
      uint32_t p = vals[rg.x + j];
      float4 m = xy[p];
      float4 co = conic_op[p];
      float dx = rel_pos(m.x, m.z, (float)(tx * TILE)) - (float)(px - tx * TILE);
      float dy = rel_pos(m.y, m.w, (float)(ty * TILE)) - (float)(py - ty * TILE);
      float power = splat_power(co.x, co.y, co.z, dx, dy);
      if (power > 0.f) continue;
      float alpha = fminf(ALPHA_MAX, co.w * __expf(power));
      if (alpha < ALPHA_MIN) continue;
      if (j < last) ++c;
      float tT = T * (1.f - alpha);
      if (tT < T_MIN) break;
      T = tT;
    }
    visited = (unsigned long long)min(j + 1, L);
    // the remaining entries up to n_contrib count for the replay (none after a stop, which ends the list)
    for (int k = j + 1; k < min(last, L); ++k) m_replay += (masks && (masks[rg.x + k] & blk)) ? 1 : 0;
  }
  #pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    c += __shfl_xor_sync(0xffffffffu, c, o);
    visited += __shfl_xor_sync(0xffffffffu, visited, o);
    replay += __shfl_xor_sync(0xffffffffu, replay, o);
    m_visited += __shfl_xor_sync(0xffffffffu, m_visited, o);
    m_replay += __shfl_xor_sync(0xffffffffu, m_replay, o);
  }
  if ((threadIdx.x & 31) == 0) {
    if (c) atomicAdd(&counts[0], c);
    if (visited) atomicAdd(&counts[1], visited);
    if (replay) atomicAdd(&counts[2], replay);
    if (m_visited) atomicAdd(&counts[3], m_visited);
    if (m_replay) atomicAdd(&counts[4], m_replay);
  }
}

// Deterministic mode: the int64 fixed-point sums back to the float screen-space gradients.
__global__ void k_fixed_to_grad2d(const unsigned long long* __restrict__ fixed, int64_t P, float* __restrict__ dxy,
                                  float* __restrict__ dco, float* __restrict__ drgb) {
  gs_wait_previous();
  int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (p >= P) return;
  float g[9];
  #pragma unroll
  for (int q = 0; q < 9; ++q) g[q] = __ll2float_rn((long long)fixed[9 * p + q]) * (1.0f / FIX_SCALE);
  reinterpret_cast<float2*>(dxy)[p] = make_float2(g[0], g[1]);
  reinterpret_cast<float4*>(dco)[p] = make_float4(g[2], g[3], g[4], g[5]);
  reinterpret_cast<float4*>(drgb)[p] = make_float4(g[6], g[7], g[8], 0.f);
}

// The two ticket words of the scheduled blend kernels: the jobs array's last entry, which no job uses
// (a list of L entries has ceil(L / K) < L / K + 1 jobs, so there are fewer than max_jobs - 1).
inline uint32_t* sched_ticket(const gs_schedule* sched) {
  return sched->jobs + 2 * (sched->max_jobs - 1);
}

}  // namespace

int gs_render_fwd_impl(const gs_proj* proj, const uint32_t* sorted_vals, const uint32_t* ranges, int n_units,
                       int width, int height, const float* bg, float* img, float* final_T, uint32_t* n_contrib,
                       int variant, const gs_schedule* sched, cudaStream_t s) {
  if (!proj || !proj->xy || !proj->conic_op || !proj->rgb || !sorted_vals || !ranges || !bg || !img ||
      !final_T || !n_contrib || n_units < 1 || n_units > GS_MAX_UNITS || width <= 0 || height <= 0 ||
      variant < 0 || variant > 2)
    return GS_ERR_INVALID;
  int TX = (width + TILE - 1) / TILE, TY = (height + TILE - 1) / TILE;
  dim3 grid(TX * TY * n_units);
  // the queue of the forward's later passes holds at most one entry per (chunk job, pixel block); its count follows it
  const uint32_t qcap = sched ? (uint32_t)(8 * sched->max_jobs) : 0u;
#define GS_FWD(BW)                                                                                                  \
  if (sched) {                                                                                                        \
    const bool later = !sched->walk_whole_lists && sched->max_checkpoints > FRONT_CHUNKS;                             \
    uint32_t* tk = sched_ticket(sched);                                                                               \
    uint32_t* q = sched->stop_queue;                                                                                  \
    float4* ck = (float4*)sched->checkpoints;                                                                         \
    const float4 *pxy = (const float4*)proj->xy, *pco = (const float4*)proj->conic_op, *prgb = (const float4*)proj->rgb;\
    const uint2* rg = (const uint2*)ranges;                                                                           \
    gs_launch(k_render_fwd_empty, grid, TILE_PIX, 0, s, rg, width, height, TX, TX * TY, bg[0], bg[1], bg[2],       \
        img, final_T, n_contrib, tk, q + qcap);                                                                    \
    const unsigned resident = gs_resident_grid<k_render_fwd_front<BW>, 32>(INT_MAX);                               \
    gs_launch(k_render_fwd_front<BW>, resident < 8 * grid.x ? resident : 8 * grid.x, 32, 0, s, rg, sched->tile_order, \
        sched->job_base, sched->chunk, sched->walk_whole_lists != 0, later ? resident : 0u, (int)grid.x, ck,          \
        sched->chunk_last, sorted_vals, sched->block_masks, pxy, pco, prgb, width, height, TX, TX * TY, bg[0], bg[1], \
        bg[2], img, final_T, n_contrib, q, qcap, tk);                                                                 \
    if (later) {                                                                                                      \
      gs_launch(k_render_fwd_chunk<BW>, gs_resident_grid<k_render_fwd_chunk<BW>, 32>((int64_t)qcap), 32, 0,        \
          s, rg, sched->tile_order, sched->job_base, sched->jobs, sched->chunk, ck, sched->chunk_last,             \
          sorted_vals, sched->block_masks, pxy, pco, prgb, width, height, TX, TX * TY, n_contrib, q, qcap,         \
          tk + 1);                                                                                                 \
      gs_launch(k_render_fwd_combine<BW>, gs_resident_grid<k_render_fwd_combine<BW>, 32>((int64_t)qcap), 32,       \
          0, s, sched->tile_order, sched->job_base, sched->jobs, ck, sched->chunk_last, width, height, TX,         \
          TX * TY, bg[0], bg[1], bg[2], img, final_T, n_contrib, q, qcap, tk);                                     \
      gs_launch(k_render_fwd_stop<BW>, gs_resident_grid<k_render_fwd_stop<BW>, 32>((int64_t)qcap), 32, 0, s,       \
          rg, sched->tile_order, sched->job_base, sched->jobs, sched->chunk, ck, sched->chunk_last,                \
          sorted_vals, sched->block_masks, pxy, pco, prgb, width, height, TX, TX * TY, bg[0], bg[1], bg[2],        \
          img, final_T, n_contrib, q, qcap, tk);                                                                   \
    }                                                                                                                 \
  } else                                                                                                            \
    gs_launch(k_render_fwd<BW>, grid, TILE_PIX, 0, s, (const uint2*)ranges, nullptr, sorted_vals,                  \
        (const float4*)proj->xy, (const float4*)proj->conic_op, (const float4*)proj->rgb, width, height, TX,       \
        TX * TY, bg[0], bg[1], bg[2], img, final_T, n_contrib)
  if (variant == 0) { GS_FWD(8); } else if (variant == 1) { GS_FWD(16); } else { GS_FWD(4); }
#undef GS_FWD
  return gs_check_launch();
}

GS_API int gs_render_fwd(const gs_proj* proj, const uint32_t* sorted_vals, const uint32_t* ranges, int n_units,
                         int width, int height, const float* bg, float* img, float* final_T, uint32_t* n_contrib,
                         int variant, const gs_schedule* sched, gs_stream_t stream) {
  GS_RANGE("gs_render_fwd");
  return gs_render_fwd_impl(proj, sorted_vals, ranges, n_units, width, height, bg, img, final_T, n_contrib, variant,
                            sched, (cudaStream_t)stream);
}

int gs_blend_bwd_impl(const gs_proj* proj, const uint32_t* sorted_vals, const uint32_t* ranges, int n_units,
                      int width, int height, const float* bg, const float* final_T, const uint32_t* n_contrib,
                      const float* dL_dimg, const float* dL_dT, const gs_grad2d* g2d, int64_t n_proj, int variant,
                      const gs_schedule* sched, const float* img, cudaStream_t s) {
  if (!proj || !proj->xy || !proj->conic_op || !proj->rgb || !sorted_vals || !ranges || !bg || !final_T ||
      !n_contrib || !dL_dimg || !g2d || !g2d->dxy || !g2d->dconic_op || !g2d->drgb || n_units < 1 || (sched && !img) ||
      n_units > GS_MAX_UNITS || width <= 0 || height <= 0 || n_proj < 0 || variant < 0 || variant > 2)
    return GS_ERR_INVALID;
  unsigned long long* fixed = g2d->fixed;
  if (fixed) {
    if (cudaMemsetAsync(fixed, 0, sizeof(unsigned long long) * 9 * (size_t)n_proj, s) != cudaSuccess)
      return GS_ERR_CUDA;
  } else if (cudaMemsetAsync(g2d->dxy, 0, sizeof(float) * 2 * (size_t)n_proj, s) != cudaSuccess ||
             cudaMemsetAsync(g2d->dconic_op, 0, sizeof(float) * 4 * (size_t)n_proj, s) != cudaSuccess ||
             cudaMemsetAsync(g2d->drgb, 0, sizeof(float) * 4 * (size_t)n_proj, s) != cudaSuccess) {
    return GS_ERR_CUDA;
  }
  int TX = (width + TILE - 1) / TILE, TY = (height + TILE - 1) / TILE;
  dim3 grid(TX * TY * n_units);
#define GS_BWD(BW)                                                                                                   \
  if (sched)                                                                                                         \
    {                                                                                                              \
      if (cudaMemsetAsync(sched_ticket(sched), 0, sizeof(uint32_t), s) != cudaSuccess) return GS_ERR_CUDA;        \
      if (fixed) {                                                                                                   \
        gs_launch(k_render_bwd_det<BW>, gs_resident_grid<k_render_bwd_det<BW>, 32>(sched->max_jobs * 8), 32,       \
            0, s, (const uint2*)ranges, sched->tile_order, sched->job_base, sched->jobs, sched->chunk,             \
            (const float4*)sched->checkpoints, sorted_vals, sched->block_masks, (const float4*)proj->xy,           \
            (const float4*)proj->conic_op, (const float4*)proj->rgb, width, height, TX, TX * TY,                   \
            TX * TY * n_units, bg[0], bg[1], bg[2], img, final_T, n_contrib, dL_dimg, dL_dT, fixed,                \
            sched_ticket(sched));                                                                                  \
      } else {                                                                                                       \
        gs_launch(k_render_bwd_m<BW>, gs_resident_grid<k_render_bwd_m<BW>, 32>(sched->max_jobs * 8), 32, 0,        \
            s, (const uint2*)ranges, sched->tile_order, sched->job_base, sched->jobs, sched->chunk,                \
            (const float4*)sched->checkpoints, sorted_vals, sched->block_masks, (const float4*)proj->xy,           \
            (const float4*)proj->conic_op, (const float4*)proj->rgb, width, height, TX, TX * TY,                   \
            TX * TY * n_units, bg[0], bg[1], bg[2], img, final_T, n_contrib, dL_dimg, dL_dT, g2d->dxy,             \
            g2d->dconic_op, g2d->drgb, sched_ticket(sched));                                                       \
      }                                                                                                              \
    }                                                                                                              \
  else                                                                                                               \
    gs_launch(k_render_bwd<BW>, grid, TILE_PIX, 0, s, (const uint2*)ranges, nullptr, sorted_vals,                  \
        (const float4*)proj->xy, (const float4*)proj->conic_op, (const float4*)proj->rgb, width, height, TX,       \
        TX * TY, bg[0], bg[1], bg[2], final_T, n_contrib, dL_dimg, dL_dT, g2d->dxy, g2d->dconic_op, g2d->drgb,     \
        fixed)
  if (variant == 0) { GS_BWD(8); } else if (variant == 1) { GS_BWD(16); } else { GS_BWD(4); }
#undef GS_BWD
  if (fixed && n_proj > 0)
    gs_launch(k_fixed_to_grad2d, (unsigned)((n_proj + 255) / 256), 256, 0, s, fixed, n_proj, g2d->dxy,
        g2d->dconic_op, g2d->drgb);
  return gs_check_launch();
}

GS_API int gs_blend_pairs(const gs_proj* proj, const uint32_t* sorted_vals, const uint32_t* ranges, int n_units,
                          int width, int height, const uint32_t* n_contrib, const uint16_t* block_masks,
                          unsigned long long* d_count, gs_stream_t stream) {
  GS_RANGE("gs_blend_pairs");
  if (!proj || !proj->xy || !proj->conic_op || !sorted_vals || !ranges || !n_contrib || !d_count || n_units < 1 ||
      n_units > GS_MAX_UNITS || width <= 0 || height <= 0)
    return GS_ERR_INVALID;
  cudaStream_t s = (cudaStream_t)stream;
  if (cudaMemsetAsync(d_count, 0, 5 * sizeof(unsigned long long), s) != cudaSuccess) return GS_ERR_CUDA;
  int TX = (width + TILE - 1) / TILE, TY = (height + TILE - 1) / TILE;
  gs_launch(k_blend_pairs, dim3(TX * TY, n_units), TILE_PIX, 0, s, (const uint2*)ranges, sorted_vals,
      (const float4*)proj->xy, (const float4*)proj->conic_op, width, height, TX, TX * TY, n_contrib, block_masks,
      d_count);
  return gs_check_launch();
}

// Heaviest-first order of the (unit, tile) blocks from the tile ranges.
// ws: 2 x 33 uint32 of scratch.
int gs_tile_order_impl(const uint32_t* ranges, int n, uint32_t* ws, uint32_t* order, cudaStream_t s) {
  if (cudaMemsetAsync(ws, 0, sizeof(uint32_t) * 66, s) != cudaSuccess) return GS_ERR_CUDA;
  unsigned nb = (unsigned)((n + 255) / 256);
  gs_launch(k_order_hist, nb, 256, 0, s, (const uint2*)ranges, n, ws);
  gs_launch(k_order_scatter, nb, 256, 0, s, (const uint2*)ranges, n, ws, ws + 33, order);
  return gs_check_launch();
}
