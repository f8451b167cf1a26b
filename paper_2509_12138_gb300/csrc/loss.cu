// a4: masked L1 + SSIM photometric loss and its image gradient.
//
// The mask restricts the loss to the pixels a partition owns (paper Sec. II,
// "Image Rendering and Masking").  SSIM uses the 11x11 Gaussian window
// (sigma 1.5) as a separable, zero-padded "same" convolution; each 32x32
// output tile stages its (32+10)^2 input halo in shared memory.  The SSIM
// gradient w.r.t. the rendered image is the adjoint convolution of three
// per-pixel factor maps (dS/dmu_x, dS/dE[x^2], dS/dE[xy] times the mask
// weight), again separable and zero padded.
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include "common.cuh"

using namespace gs;

namespace {

constexpr int LT = 32;           // output tile edge
constexpr int R = 5;             // window radius
constexpr int HT = LT + 2 * R;   // halo tile edge (42)
constexpr int PAD = 8;           // columns staged in front of the output tile: a multiple of 4 pixels, at least R
constexpr int HW = LT + 2 * PAD; // staged columns (48), in groups of 4
constexpr int SEG = 4;           // outputs per thread along each pass
constexpr int LOSS_T = 256;      // LT columns x (LT / SEG) strips
// Row strides in shared memory: 8 threads of a 16-byte access take 4 segments of 2 rows (seg_task), whose banks
// differ when the rows of pairs (8 bytes) start 4 banks apart and those of single values 16 banks apart.
constexpr int HS2 = 50, TS2 = 34;  // pairs: staged rows, horizontal sums
constexpr int HS1 = 48, TS1 = 48;  // single values
static_assert(LT * (LT / SEG) == LOSS_T && HT % 2 == 0 && PAD >= R + 2 && HW <= HS2 && HW <= HS1, "thread layout");
constexpr float C1 = 0.01f * 0.01f;
constexpr float C2 = 0.03f * 0.03f;

// Normalised 11-tap Gaussian window (sigma 1.5), computed by each block.
__device__ __forceinline__ void load_window(float* w) {
  if (threadIdx.x < 11) {
    float s = 0.f;
    for (int t = 0; t < 11; ++t) s += expf(-(t - 5.f) * (t - 5.f) / (2.f * 1.5f * 1.5f));
    float d = threadIdx.x - 5.f;
    w[threadIdx.x] = expf(-d * d / (2.f * 1.5f * 1.5f)) / s;
  }
}

__host__ __device__ inline size_t a256(size_t x) { return (x + 255) & ~(size_t)255; }

struct LossWs {
  size_t msum, l1, ss, fac, total;
};
LossWs loss_ws(int U, int W, int H) {
  LossWs L;
  size_t o = 0;
  L.msum = o; o += a256(sizeof(uint32_t) * U);
  L.l1 = o; o += a256(sizeof(double) * U);
  L.ss = o; o += a256(sizeof(double) * U);
  L.fac = o; o += a256(sizeof(float) * 3 * 3 * (size_t)U * W * H);
  L.total = o;
  return L;
}

__device__ __forceinline__ float block_sum(float v, float* s) {
  #pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  __syncthreads();
  if (lane == 0) s[w] = v;
  __syncthreads();
  float t = 0.f;
  if (threadIdx.x == 0)
    for (int q = 0; q < (int)(blockDim.x >> 5); ++q) t += s[q];
  return t;  // valid in thread 0
}

// Mask pixels per unit.  vec: the units' masks start on 16 bytes and hold a multiple of 16 (16-byte loads).
__global__ void k_mask_count(const uint8_t* __restrict__ mask, int64_t plane, int vec, uint32_t* msum) {
  gs_wait_previous();
  __shared__ float s[32];
  int u = blockIdx.y;
  uint32_t c = 0;
  const int64_t stride = (int64_t)gridDim.x * blockDim.x, first = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (vec) {
    const uint4* m4 = reinterpret_cast<const uint4*>(mask + (int64_t)u * plane);
    auto nonzero = [](uint32_t x) { return (uint32_t)__popc(__vcmpne4(x, 0u)) >> 3; };
    for (int64_t k = first; k < plane / 16; k += stride) {
      const uint4 x = __ldg(m4 + k);
      c += nonzero(x.x) + nonzero(x.y) + nonzero(x.z) + nonzero(x.w);
    }
  } else {
    for (int64_t k = first; k < plane; k += stride) c += mask[(int64_t)u * plane + k] ? 1u : 0u;
  }
  float t = block_sum((float)c, s);
  if (threadIdx.x == 0 && t > 0.f) atomicAdd(&msum[u], (uint32_t)t);
}

// L1 part only (lambda = 0): gradient and loss sums
__global__ void k_l1(const float* __restrict__ img, const float* __restrict__ gt, const uint8_t* __restrict__ mask,
                     int64_t plane, const uint32_t* __restrict__ msum, float w1, float invU, double* l1sum,
                     float* __restrict__ dimg) {
  gs_wait_previous();
  __shared__ float s[32];
  int u = blockIdx.y;
  float acc = 0.f;
  float nm = (float)msum[u];
  float scale = nm > 0.f ? w1 * invU / (3.f * nm) : 0.f;
  for (int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k < plane; k += (int64_t)gridDim.x * blockDim.x) {
    bool in = mask[(int64_t)u * plane + k] != 0;
    #pragma unroll
    for (int c = 0; c < 3; ++c) {
      int64_t q = ((int64_t)u * 3 + c) * plane + k;
      float d = img[q] - gt[q];
      float sg = d > 0.f ? 1.f : (d < 0.f ? -1.f : 0.f);
      dimg[q] = in ? scale * sg : 0.f;
      if (in) acc += fabsf(d);
    }
  }
  float t = block_sum(acc, s);
  if (threadIdx.x == 0 && t != 0.f) atomicAdd(&l1sum[u], (double)t);
}

// Two quantities that go through the same window travel as a pair, which
// Blackwell multiplies and adds in one instruction (each half rounded as the
// scalar operation would).
using pair = unsigned long long;
__device__ __forceinline__ pair make_pair(float a, float b) {
  pair r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
  return r;
}
__device__ __forceinline__ float2 halves(pair v) {
  float2 r;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(v));
  return r;
}
__device__ __forceinline__ pair fma2(pair a, pair b, pair c) {
  pair r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
  return r;
}
__device__ __forceinline__ pair mul2(pair a, pair b) {
  pair r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}

// Separable 11-tap window, SEG outputs per thread along each pass: a thread
// reads its 14 inputs once and multiplies from registers, where one output per
// thread would read 11 values for 11 multiplications.  Taps are added in
// ascending order from zero, one fused multiply-add each.
__device__ __forceinline__ void taps(const float* w, const float* in, float* out) {
  #pragma unroll
  for (int e = 0; e < SEG; ++e) {
    float a = 0.f;
    #pragma unroll
    for (int t = 0; t < 11; ++t) a = fmaf(w[t], in[e + t], a);
    out[e] = a;
  }
}
__device__ __forceinline__ void taps2(const pair* w, const pair* in, pair* out) {
  #pragma unroll
  for (int e = 0; e < SEG; ++e) {
    pair a = 0ull;
    #pragma unroll
    for (int t = 0; t < 11; ++t) a = fma2(w[t], in[e + t], a);
    out[e] = a;
  }
}
// the window's inputs of the outputs SEG g .. SEG g + 3 of a staged row: columns SEG g + PAD - R on, from the aligned
// column in front of them (v[1] and v[3] are the first)
__device__ __forceinline__ void load_seg2(const pair* row, int g, pair* v) {
  #pragma unroll
  for (int q = 0; q < 8; ++q) {
    const ulonglong2 x = reinterpret_cast<const ulonglong2*>(row + SEG * g + 2)[q];
    v[2 * q] = x.x; v[2 * q + 1] = x.y;
  }
}
__device__ __forceinline__ void load_seg(const float* row, int g, float* v) {
  #pragma unroll
  for (int q = 0; q < 5; ++q) {
    const float4 x = reinterpret_cast<const float4*>(row + SEG * g)[q];
    v[4 * q] = x.x; v[4 * q + 1] = x.y; v[4 * q + 2] = x.z; v[4 * q + 3] = x.w;
  }
}
__device__ __forceinline__ void store_seg2(pair* row, int g, const pair* v) {
  ulonglong2* r = reinterpret_cast<ulonglong2*>(row + SEG * g);
  r[0] = make_ulonglong2(v[0], v[1]);
  r[1] = make_ulonglong2(v[2], v[3]);
}
__device__ __forceinline__ void store_seg(float* row, int g, const float* v) {
  reinterpret_cast<float4*>(row)[g] = make_float4(v[0], v[1], v[2], v[3]);
}
// horizontal task k: (halo row, segment), so that 8 threads in a row take 2 rows x 4 segments
constexpr int SEG_TASKS = HT * (LT / SEG);
__device__ __forceinline__ void seg_task(int k, int& r, int& g) {
  const int hi = k >> 3;
  r = 2 * (hi >> 1) + ((k >> 2) & 1);
  g = 4 * (hi & 1) + (k & 3);
}
static_assert(LT / SEG == 8, "seg_task");

// vertical pass: the SEG outputs of column lx from row SEG strip of the horizontal sums
__device__ __forceinline__ void taps_down(const float* w, const float (*tmp)[TS1], int lx, int strip, float* out) {
  float v[SEG + 10];
  #pragma unroll
  for (int t = 0; t < SEG + 10; ++t) v[t] = tmp[SEG * strip + t][lx];
  taps(w, v, out);
}
__device__ __forceinline__ void taps_down2(const pair* w, const pair (*tmp)[TS2], int lx, int strip, pair* out) {
  pair v[SEG + 10];
  #pragma unroll
  for (int t = 0; t < SEG + 10; ++t) v[t] = tmp[SEG * strip + t][lx];
  taps2(w, v, out);
}

// Calls f(staged row, first staged column, image column, row in the image?,
// offset in the plane) for every group of 4 staged pixels.  Where the plane's
// rows start on 16 bytes (vec) a group lies inside the image or outside and is
// one load per array; otherwise its pixels are read one at a time.
template <typename F>
__device__ __forceinline__ void for_groups(int bx, int by, int W, int H, F f) {
  for (int k = threadIdx.x; k < HT * (HW / 4); k += LOSS_T) {
    const int r = k / (HW / 4), q = 4 * (k % (HW / 4));
    const int gx = bx * LT - PAD + q, gy = by * LT - R + r;
    f(r, q, gx, gy >= 0 && gy < H, (int64_t)gy * W + gx);
  }
}

// SSIM statistics, loss sums and the three factor maps.  Bound by fp32 issue
// (127 multiply-adds per pixel and channel with the halo rows, 76 instructions
// as pairs); the rest is staging and the divisions of the epilogue.  The whole
// loss at 2048x2048, a random half of the pixels in the mask: 650 us with one
// output per thread -> 280; 8 views of 1920x1080, 20% mask: 360 us with scalar
// multiply-adds and pixel-by-pixel staging -> 234, one view 85 -> 66.
__global__ void __launch_bounds__(LOSS_T) k_ssim_stats(const float* __restrict__ img, const float* __restrict__ gt,
                                                       const uint8_t* __restrict__ mask, int W, int H, int vec,
                                                       const uint32_t* __restrict__ msum, float lam, float invU,
                                                       double* l1sum, double* ssum, float* __restrict__ fac) {
  gs_wait_previous();
  __shared__ __align__(16) pair s_xy[HT][HS2];       // (image, GT)
  __shared__ __align__(16) pair s_mu[HT][TS2], s_sq[HT][TS2];  // horizontal sums of (x, y) and (x^2, y^2)
  __shared__ __align__(16) float s_c[HT][TS1];       // of x y
  __shared__ float s_red[32];
  __shared__ float s_win[11];
  int tiles_x = (W + LT - 1) / LT;
  int bx = blockIdx.x % tiles_x, by = blockIdx.x / tiles_x;
  int c = blockIdx.y, u = blockIdx.z;
  int64_t plane = (int64_t)W * H;
  const int lx = threadIdx.x % LT, strip = threadIdx.x / LT;
  const int px = bx * LT + lx, py = by * LT + SEG * strip;  // this thread's outputs: rows py .. py + SEG - 1
  bool in[SEG], any = false;
  #pragma unroll
  for (int e = 0; e < SEG; ++e) {
    in[e] = px < W && py + e < H && mask[(int64_t)u * plane + (int64_t)(py + e) * W + px] != 0;
    any = any || in[e];
  }
  // a tile without mask pixels adds nothing to the loss and has no factor map entries
  if (!__syncthreads_or(any)) return;
  load_window(s_win);
  const float* X = img + ((int64_t)u * 3 + c) * plane;
  const float* Y = gt + ((int64_t)u * 3 + c) * plane;
  for_groups(bx, by, W, H, [&](int r, int q, int gx, bool row_in, int64_t off) {
    float4 a = make_float4(0.f, 0.f, 0.f, 0.f), b = a;
    if (vec) {
      if (row_in && gx >= 0 && gx < W) {
        a = __ldg(reinterpret_cast<const float4*>(X + off));
        b = __ldg(reinterpret_cast<const float4*>(Y + off));
      }
    } else if (row_in) {
      auto get = [&](int e, float& av, float& bv) {
        if (gx + e >= 0 && gx + e < W) { av = X[off + e]; bv = Y[off + e]; }
      };
      get(0, a.x, b.x); get(1, a.y, b.y); get(2, a.z, b.z); get(3, a.w, b.w);
    }
    ulonglong2* dst = reinterpret_cast<ulonglong2*>(&s_xy[r][q]);
    dst[0] = make_ulonglong2(make_pair(a.x, b.x), make_pair(a.y, b.y));
    dst[1] = make_ulonglong2(make_pair(a.z, b.z), make_pair(a.w, b.w));
  });
  __syncthreads();
  float w[11];
  pair w2[11];
  #pragma unroll
  for (int t = 0; t < 11; ++t) { w[t] = s_win[t]; w2[t] = make_pair(w[t], w[t]); }
  for (int k = threadIdx.x; k < SEG_TASKS; k += LOSS_T) {
    int r, g;
    seg_task(k, r, g);
    pair v[16], o2[SEG];
    float p[SEG + 10], o[SEG];
    load_seg2(s_xy[r], g, v);
    taps2(w2, v + 1, o2);
    store_seg2(s_mu[r], g, o2);
    #pragma unroll
    for (int t = 0; t < SEG + 10; ++t) {
      const float2 ab = halves(v[t + 1]);
      p[t] = __fmul_rn(ab.x, ab.y);
    }
    taps(w, p, o);
    store_seg(s_c[r], g, o);
    #pragma unroll
    for (int t = 0; t < SEG + 10; ++t) v[t + 1] = mul2(v[t + 1], v[t + 1]);
    taps2(w2, v + 1, o2);
    store_seg2(s_sq[r], g, o2);
  }
  __syncthreads();
  pair mu[SEG], sq[SEG];
  float cr[SEG];
  taps_down2(w2, s_mu, lx, strip, mu);
  taps_down2(w2, s_sq, lx, strip, sq);
  taps_down(w, s_c, lx, strip, cr);
  float nm = (float)msum[u];
  float sacc = 0.f, lacc = 0.f;
  #pragma unroll
  for (int e = 0; e < SEG; ++e) {
    if (!in[e]) continue;  // the factor maps are zero off the mask; only mask pixels are stored and read
    float fmu = 0.f, fxx = 0.f, fxy = 0.f;
    if (nm > 0.f) {
      const float2 m = halves(mu[e]), q2 = halves(sq[e]);
      float ux = m.x, uy = m.y;
      float vx = q2.x - ux * ux, vy = q2.y - uy * uy, cxy = cr[e] - ux * uy;
      float A1 = 2.f * ux * uy + C1, A2 = 2.f * cxy + C2;
      float B1 = ux * ux + uy * uy + C1, B2 = vx + vy + C2;
      float S = (A1 * A2) / (B1 * B2);
      sacc += S;
      const float2 xy = halves(s_xy[SEG * strip + e + R][lx + PAD]);
      lacc += fabsf(xy.x - xy.y);
      float wp = -lam * invU / (3.f * nm);  // d loss / d S_p
      fmu = wp * S * (2.f * uy / A1 - 2.f * ux / B1 - 2.f * uy / A2 + 2.f * ux / B2);
      fxx = wp * S * (-1.f / B2);
      fxy = wp * S * (2.f / A2);
    }
    int64_t base = ((int64_t)u * 3 + c) * plane + (int64_t)(py + e) * W + px;
    int64_t fs = (int64_t)3 * plane * gridDim.z;  // stride between the three factor maps
    fac[base] = fmu;
    fac[fs + base] = fxx;
    fac[2 * fs + base] = fxy;
  }
  float ts = block_sum(sacc, s_red);
  if (threadIdx.x == 0 && ts != 0.f) atomicAdd(&ssum[u], (double)ts);
  float tl = block_sum(lacc, s_red);
  if (threadIdx.x == 0 && tl != 0.f) atomicAdd(&l1sum[u], (double)tl);
}

// dL/dimg = L1 part + conv(fmu) + 2 x conv(fxx) + y conv(fxy).  76
// multiply-adds per pixel and channel, 51 instructions as pairs.
__global__ void __launch_bounds__(LOSS_T) k_ssim_grad(const float* __restrict__ img, const float* __restrict__ gt,
                                                      const uint8_t* __restrict__ mask, int W, int H, int vec,
                                                      const uint32_t* __restrict__ msum, float w1, float invU,
                                                      const float* __restrict__ fac, float* __restrict__ dimg) {
  gs_wait_previous();
  __shared__ __align__(16) pair s_in[HT][HS2];    // (fmu, fxx)
  __shared__ __align__(16) float s_in1[HT][HS1];  // fxy
  __shared__ __align__(16) pair s_tmp[HT][TS2];
  __shared__ __align__(16) float s_tmp1[HT][TS1];
  __shared__ float s_win[11];
  int tiles_x = (W + LT - 1) / LT;
  int bx = blockIdx.x % tiles_x, by = blockIdx.x / tiles_x;
  int c = blockIdx.y, u = blockIdx.z;
  int64_t plane = (int64_t)W * H;
  int64_t off = ((int64_t)u * 3 + c) * plane;
  int64_t fs = (int64_t)3 * plane * gridDim.z;
  const int lx = threadIdx.x % LT, strip = threadIdx.x / LT;
  const int px = bx * LT + lx, py = by * LT + SEG * strip;
  const uint8_t* M = mask + (int64_t)u * plane;
  // factor maps are nonzero only at mask pixels: zero elsewhere, whatever the maps' memory holds there
  bool any = false;
  for_groups(bx, by, W, H, [&](int r, int q, int gx, bool row_in, int64_t o) {
    float4 a = make_float4(0.f, 0.f, 0.f, 0.f), b = a, d = a;
    if (vec) {
      const uint32_t m = row_in && gx >= 0 && gx < W ? __ldg(reinterpret_cast<const uint32_t*>(M + o)) : 0u;
      if (m) {
        // (the outer 3 of the staged columns are beyond the window's reach)
        any = any || (q == 0 ? m >> 24 : q == HW - 4 ? m & 0xffu : m) != 0u;
        a = __ldg(reinterpret_cast<const float4*>(fac + off + o));
        b = __ldg(reinterpret_cast<const float4*>(fac + fs + off + o));
        d = __ldg(reinterpret_cast<const float4*>(fac + 2 * fs + off + o));
        if (!(m & 0xffu)) a.x = b.x = d.x = 0.f;
        if (!(m & 0xff00u)) a.y = b.y = d.y = 0.f;
        if (!(m & 0xff0000u)) a.z = b.z = d.z = 0.f;
        if (!(m & 0xff000000u)) a.w = b.w = d.w = 0.f;
      }
    } else if (row_in) {
      auto get = [&](int e, float& av, float& bv, float& dv) {
        if (gx + e >= 0 && gx + e < W && M[o + e] != 0) {
          const int64_t pix = off + o + e;
          av = fac[pix]; bv = fac[fs + pix]; dv = fac[2 * fs + pix];
          any = any || (q + e >= PAD - R && q + e < PAD + LT + R);
        }
      };
      get(0, a.x, b.x, d.x); get(1, a.y, b.y, d.y); get(2, a.z, b.z, d.z); get(3, a.w, b.w, d.w);
    }
    ulonglong2* dst = reinterpret_cast<ulonglong2*>(&s_in[r][q]);
    dst[0] = make_ulonglong2(make_pair(a.x, b.x), make_pair(a.y, b.y));
    dst[1] = make_ulonglong2(make_pair(a.z, b.z), make_pair(a.w, b.w));
    *reinterpret_cast<float4*>(&s_in1[r][q]) = d;
  });
  // no mask pixel within the window's reach: both gradient terms vanish
  if (!__syncthreads_or(any)) {
    #pragma unroll
    for (int e = 0; e < SEG; ++e)
      if (px < W && py + e < H) dimg[off + (int64_t)(py + e) * W + px] = 0.f;
    return;
  }
  load_window(s_win);
  __syncthreads();
  float w[11];
  pair w2[11];
  #pragma unroll
  for (int t = 0; t < 11; ++t) { w[t] = s_win[t]; w2[t] = make_pair(w[t], w[t]); }
  for (int k = threadIdx.x; k < SEG_TASKS; k += LOSS_T) {
    int r, g;
    seg_task(k, r, g);
    pair v[16], o2[SEG];
    float a[20], o[SEG];
    load_seg2(s_in[r], g, v);
    taps2(w2, v + 1, o2);
    store_seg2(s_tmp[r], g, o2);
    load_seg(s_in1[r], g, a);
    taps(w, a + 3, o);
    store_seg(s_tmp1[r], g, o);
  }
  __syncthreads();
  pair cv[SEG];
  float cv1[SEG];
  taps_down2(w2, s_tmp, lx, strip, cv);
  taps_down(w, s_tmp1, lx, strip, cv1);
  float nm = (float)msum[u];
  #pragma unroll
  for (int e = 0; e < SEG; ++e) {
    if (!(px < W && py + e < H)) continue;
    int64_t pix = (int64_t)(py + e) * W + px;
    float x = img[off + pix], y = gt[off + pix];
    bool in = M[pix] != 0;
    float d = x - y;
    float sg = d > 0.f ? 1.f : (d < 0.f ? -1.f : 0.f);
    float gl1 = (in && nm > 0.f) ? w1 * invU / (3.f * nm) * sg : 0.f;
    const float2 f = halves(cv[e]);
    dimg[off + pix] = gl1 + f.x + 2.f * x * f.y + y * cv1[e];
  }
}

// the units' losses, one per lane (a thread summing them alone waits for each unit's loads in turn)
__global__ void __launch_bounds__(32) k_loss_final(const uint32_t* msum, const double* l1sum, const double* ssum, int U,
                                                   float lam, float* out) {
  gs_wait_previous();
  double acc = 0.0;
  for (int u = threadIdx.x; u < U; u += 32) {
    double nm = (double)msum[u];
    if (nm <= 0.0) continue;
    double l1 = l1sum[u] / (3.0 * nm);
    double v = (1.0 - lam) * l1;
    if (lam > 0.f) v += lam * (1.0 - ssum[u] / (3.0 * nm));
    acc += v;
  }
  #pragma unroll
  for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
  if (threadIdx.x == 0) *out = (float)(acc / U);
}

// Background-opacity penalty (variant of the mask): per unit, the number of pixels outside the mask
// and the sum of their rendered opacity 1 - T_final (one atomic per warp).
__global__ void __launch_bounds__(256) k_bg_sum(const float* __restrict__ final_T, const uint8_t* __restrict__ mask,
                                                int64_t plane, unsigned long long* __restrict__ cnt,
                                                double* __restrict__ sum) {
  gs_wait_previous();
  int u = blockIdx.y;
  const float* T = final_T + (int64_t)u * plane;
  const uint8_t* m = mask + (int64_t)u * plane;
  unsigned c = 0;
  double a = 0.0;
  for (int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; k < plane; k += (int64_t)gridDim.x * blockDim.x)
    if (m[k] == 0) { ++c; a += (double)(1.f - T[k]); }
  for (int o = 16; o > 0; o >>= 1) {
    c += __shfl_down_sync(0xffffffffu, c, o);
    a += __shfl_down_sync(0xffffffffu, a, o);
  }
  if ((threadIdx.x & 31) == 0 && c) {
    atomicAdd(&cnt[u], (unsigned long long)c);
    atomicAdd(&sum[u], a);
  }
}

// dpenalty/dT_final: -lambda / (U n_bg) at the unit's background pixels, 0 at mask pixels
__global__ void __launch_bounds__(256) k_bg_grad(const uint8_t* __restrict__ mask, int64_t plane,
                                                 const unsigned long long* __restrict__ cnt, float lam, float invU,
                                                 float* __restrict__ dLdT) {
  gs_wait_previous();
  int u = blockIdx.y;
  unsigned long long n = cnt[u];
  float g = n ? -lam * invU / (float)n : 0.f;
  const uint8_t* m = mask + (int64_t)u * plane;
  float* d = dLdT + (int64_t)u * plane;
  for (int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; k < plane; k += (int64_t)gridDim.x * blockDim.x)
    d[k] = m[k] == 0 ? g : 0.f;
}

__global__ void k_bg_final(const unsigned long long* cnt, const double* sum, int U, float lam, float* out) {
  gs_wait_previous();
  double acc = 0.0;
  for (int u = 0; u < U; ++u)
    if (cnt[u]) acc += sum[u] / (double)cnt[u];
  *out += (float)(lam * acc / U);
}

}  // namespace

GS_API size_t gs_bg_penalty_workspace_size(int n_units) {
  if (n_units < 1) return 0;
  return a256(sizeof(unsigned long long) * (size_t)n_units) + a256(sizeof(double) * (size_t)n_units);
}

GS_API int gs_bg_penalty(const float* final_T, const uint8_t* mask, int n_units, int width, int height,
                         float lambda_bg, void* workspace, size_t workspace_bytes, float* d_loss, float* dL_dT,
                         gs_stream_t stream) {
  GS_RANGE("gs_bg_penalty");
  if (!final_T || !mask || !d_loss || !dL_dT || !workspace || n_units < 1 || n_units > GS_MAX_UNITS || width <= 0 ||
      height <= 0 || !(lambda_bg >= 0.f) || !isfinite(lambda_bg))
    return GS_ERR_INVALID;
  size_t need = gs_bg_penalty_workspace_size(n_units);
  if (workspace_bytes < need || ((uintptr_t)workspace & 255u)) return GS_ERR_INVALID;
  cudaStream_t s = (cudaStream_t)stream;
  unsigned long long* cnt = (unsigned long long*)workspace;
  double* sum = (double*)((char*)workspace + a256(sizeof(unsigned long long) * (size_t)n_units));
  if (cudaMemsetAsync(workspace, 0, need, s) != cudaSuccess) return GS_ERR_CUDA;
  int64_t plane = (int64_t)width * height;
  int gx = (int)((plane + 255) / 256);
  if (gx > 1024) gx = 1024;
  gs_launch(k_bg_sum, dim3(gx, n_units), 256, 0, s, final_T, mask, plane, cnt, sum);
  gs_launch(k_bg_grad, dim3(gx, n_units), 256, 0, s, mask, plane, cnt, lambda_bg, 1.f / n_units, dL_dT);
  gs_launch(k_bg_final, 1, 1, 0, s, cnt, sum, n_units, lambda_bg, d_loss);
  return gs_check_launch();
}

GS_API size_t gs_loss_workspace_size(int n_units, int width, int height) {
  if (n_units < 1 || width <= 0 || height <= 0) return 0;
  return loss_ws(n_units, width, height).total;
}

GS_API int gs_loss(const float* img, const float* gt, const uint8_t* mask, int n_units, int width, int height,
                   float lambda_ssim, void* workspace, size_t workspace_bytes, float* d_loss, float* dL_dimg,
                   gs_stream_t stream) {
  GS_RANGE("gs_loss");
  if (!img || !gt || !mask || !d_loss || !dL_dimg || !workspace || n_units < 1 || width <= 0 || height <= 0 ||
      !(lambda_ssim >= 0.f && lambda_ssim <= 1.f))
    return GS_ERR_INVALID;
  LossWs L = loss_ws(n_units, width, height);
  if (workspace_bytes < L.total || ((uintptr_t)workspace & 255u)) return GS_ERR_INVALID;
  cudaStream_t s = (cudaStream_t)stream;
  char* ws = (char*)workspace;
  uint32_t* msum = (uint32_t*)(ws + L.msum);
  double* l1 = (double*)(ws + L.l1);
  double* ss = (double*)(ws + L.ss);
  float* fac = (float*)(ws + L.fac);
  if (cudaMemsetAsync(ws, 0, L.fac, s) != cudaSuccess) return GS_ERR_CUDA;
  int64_t plane = (int64_t)width * height;
  float invU = 1.f / n_units;
  int gx = (int)((plane + 255) / 256);
  if (gx > 1024) gx = 1024;
  const int vec = ((uintptr_t)mask & 15u) == 0 && plane % 16 == 0;
  gs_launch(k_mask_count, dim3(gx, n_units), 256, 0, s, mask, plane, vec, msum);
  if (lambda_ssim == 0.f) {
    gs_launch(k_l1, dim3(gx, n_units), 256, 0, s, img, gt, mask, plane, msum, 1.f, invU, l1, dL_dimg);
  } else {
    int tiles = ((width + LT - 1) / LT) * ((height + LT - 1) / LT);
    dim3 grid(tiles, 3, n_units);
    // rows, and with them every group of 4 pixels, start on 16 bytes (the mask's on 4)
    const int rows = width % 4 == 0 && (((uintptr_t)img | (uintptr_t)gt) & 15u) == 0 && ((uintptr_t)mask & 3u) == 0;
    gs_launch(k_ssim_stats, grid, LOSS_T, 0, s, img, gt, mask, width, height, rows, msum, lambda_ssim, invU, l1, ss,
        fac);
    gs_launch(k_ssim_grad, grid, LOSS_T, 0, s, img, gt, mask, width, height, rows, msum, 1.f - lambda_ssim, invU,
        fac, dL_dimg);
  }
  gs_launch(k_loss_final, 1, 32, 0, s, msum, l1, ss, n_units, lambda_ssim, d_loss);
  return gs_check_launch();
}

// ---- backward entry points (blend + projection)
int gs_blend_bwd_impl(const gs_proj* proj, const uint32_t* sorted_vals, const uint32_t* ranges, int n_units,
                      int width, int height, const float* bg, const float* final_T, const uint32_t* n_contrib,
                      const float* dL_dimg, const float* dL_dT, const gs_grad2d* g2d, int64_t n_proj, int variant,
                      const gs_schedule* sched, const float* img, cudaStream_t s);

GS_API int gs_blend_bwd(const gs_proj* proj, const uint32_t* sorted_vals, const uint32_t* ranges, int n_units,
                        int width, int height, const float* bg, const float* img, const float* final_T,
                        const uint32_t* n_contrib, const float* dL_dimg, const float* dL_dT, const gs_grad2d* g2d,
                        int64_t n_proj, int variant, const gs_schedule* sched, gs_stream_t stream) {
  GS_RANGE("gs_blend_bwd");
  return gs_blend_bwd_impl(proj, sorted_vals, ranges, n_units, width, height, bg, final_T, n_contrib, dL_dimg,
                           dL_dT, g2d, n_proj, variant, sched, img, (cudaStream_t)stream);
}

GS_API int gs_render_bwd(const float* params, int64_t n_gauss, int sh_degree, const gs_units* units,
                         const gs_camera* cams, const gs_proj* proj, const uint32_t* sorted_vals,
                         const uint32_t* ranges, int width, int height, const float* bg, const float* img,
                         const float* final_T, const uint32_t* n_contrib, const float* dL_dimg,
                         const float* dL_dT, const gs_grad2d* g2d, float* grads, int variant,
                         const gs_schedule* sched, gs_stream_t stream) {
  GS_RANGE("gs_render_bwd");
  UnitTable U;
  int64_t P = 0;
  if (gs_fill_units(units, U, &P) != GS_OK) return GS_ERR_INVALID;
  int r = gs_blend_bwd_impl(proj, sorted_vals, ranges, U.n, width, height, bg, final_T, n_contrib, dL_dimg, dL_dT,
                            g2d, P, variant, sched, img, (cudaStream_t)stream);
  if (r != GS_OK) return r;
  return gs_project_bwd(params, n_gauss, sh_degree, units, cams, proj, g2d, grads, stream);
}
