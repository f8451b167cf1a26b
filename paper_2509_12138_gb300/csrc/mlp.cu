// a9 (second half): the learned initialiser.  A 3-layer MLP maps each
// isosurface point's kNN geometry to its initial log-scale (relative to the
// mean 3-NN distance), rotation and opacity.
//
// Network: X[112] -> relu(X W1 + b1)[64] -> relu(. W2 + b2)[64] -> . W3 + b3 [8].
// Features (built in shared memory, never stored): the 16 neighbour offsets
// divided by the mean neighbour distance (48), the 16 neighbour normals (48),
// the point's own normal (3), zero padding to 112.  GEMM operands are bf16
// (round to nearest even), products accumulate in fp32 on the tensor cores
// (mma.sync m16n8k16 / m16n8k8); activations are rounded to bf16 where they
// become the next GEMM's operand, and back-propagated signals likewise.
//
// Batches of 128 points, 16 per warp.  Layer outputs stay in registers: the
// accumulator layout of two adjacent n8 tiles is the A-operand layout of one
// k16 step, so layers chain without shared memory; the other operands come
// from bf16 tiles in shared memory by ldmatrix.  Weight gradients are
// tensor-core GEMMs over the batch's points, summed in fp32 registers over all
// of a CTA's batches and added to the global gradient once per CTA.
//
// The arithmetic (23 kFLOP per point forward) is small for the tensor cores,
// and the 300 gathered bytes per point are small for HBM; what bounds the
// stage is latency: index load -> gather -> tile -> chained mma.  So the
// training kernel gives the gathers to warps of their own, one batch ahead of
// the warps that multiply, and mma.sync, whose operands and results are
// registers, suffices.
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include "common.cuh"

using namespace gs;

namespace {

constexpr int KIN = 112, HID = 64, KOUT = 8, KNN = 16;
constexpr int W1_OFF = 0, B1_OFF = W1_OFF + KIN * HID, W2_OFF = B1_OFF + HID, B2_OFF = W2_OFF + HID * HID;
constexpr int W3_OFF = B2_OFF + HID, B3_OFF = W3_OFF + HID * KOUT, NPARAM = B3_OFF + KOUT;  // 11912
constexpr int BATCH = 128;       // points per batch
constexpr int FWD_T = 256;        // threads of the forward kernels: 8 warps build, then multiply 16 points each
constexpr int PROD_T = 128;       // training kernel: 4 warps that build the next batch's features,
constexpr int CONS_T = 256;       // 8 warps that multiply
constexpr int LDX = 120;  // bf16 row stride of the feature tile and of W1^T (240 B: 8 rows hit 8 bank groups)
constexpr int LDH = 72;   // bf16 row stride of 64-wide tiles (144 B: likewise)
constexpr int LDI = 17;   // row stride of the staged neighbour indices

static_assert(NPARAM == 11912, "parameter layout");
static_assert(CONS_T / 32 * 16 == BATCH && FWD_T / 32 * 16 == BATCH, "16 points per warp");

// shared-memory layout (bytes)
struct Smem {
  static constexpr int W1t = 0;                          // [64][LDX] bf16  W1^T
  static constexpr int W2t = W1t + HID * LDX * 2;        // [64][LDH] bf16  W2^T
  static constexpr int W3t = W2t + HID * LDH * 2;        // [8][LDH]  bf16  W3^T
  static constexpr int Bias = W3t + KOUT * LDH * 2;      // fp32 b1[64] b2[64] b3[8]
  static constexpr int Idx = Bias + (2 * HID + KOUT) * 4;  // int [BATCH][LDI]
  static constexpr int Dbar = Idx + BATCH * LDI * 4;     // float2 [BATCH]: mean distance, its reciprocal
  static constexpr int X = Dbar + BATCH * 8;             // [BATCH][LDX] bf16 features
  static constexpr int FWD_END = X + BATCH * LDX * 2;
  static constexpr int Y = FWD_END;                      // fp32 [BATCH][8] outputs (initialiser)
  static constexpr int INIT_END = Y + BATCH * KOUT * 4;
  static constexpr int X2 = FWD_END;                     // training: the second feature tile
  static constexpr int W2 = X2 + BATCH * LDX * 2;        // [64][LDH] bf16  W2 (in-major)
  static constexpr int W3 = W2 + HID * LDH * 2;          // [64][8]   bf16  W3 (in-major)
  static constexpr int H1 = W3 + HID * KOUT * 2;         // [BATCH][LDH] bf16
  static constexpr int H2 = H1 + BATCH * LDH * 2;
  static constexpr int dH1 = H2 + BATCH * LDH * 2;
  static constexpr int dH2 = dH1 + BATCH * LDH * 2;
  static constexpr int dY = dH2 + BATCH * LDH * 2;       // [BATCH][8] bf16
  static constexpr int TRAIN_END = dY + BATCH * KOUT * 2;
};
static_assert(Smem::X % 16 == 0 && Smem::X2 % 16 == 0 && Smem::W2 % 16 == 0 && Smem::H1 % 16 == 0 &&
              Smem::dY % 16 == 0 && Smem::W2t % 16 == 0 && Smem::W3t % 16 == 0, "ldmatrix rows are 16-byte aligned");

__device__ __forceinline__ uint16_t bf(float x) { return __bfloat16_as_ushort(__float2bfloat16_rn(x)); }
__device__ __forceinline__ uint32_t pack(float lo, float hi) {
  return (uint32_t)bf(lo) | ((uint32_t)bf(hi) << 16);
}
__device__ __forceinline__ uint32_t ld32(const uint16_t* p) { return *reinterpret_cast<const uint32_t*>(p); }
// Four 8x8 bf16 matrices, lane l giving the address of row l & 7 of matrix l >> 3; TRANS: transposed.
template <bool TRANS = false>
__device__ __forceinline__ void ldsm4(uint32_t (&r)[4], const uint16_t* p) {
  const unsigned a = (unsigned)__cvta_generic_to_shared(p);
  if (TRANS)
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];\n"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(a) : "memory");
  else
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];\n"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(a) : "memory");
}
__device__ __forceinline__ void ldsm2t(uint32_t& r0, uint32_t& r1, const uint16_t* p) {
  const unsigned a = (unsigned)__cvta_generic_to_shared(p);
  asm volatile("ldmatrix.sync.aligned.m8n8.x2.trans.shared.b16 {%0,%1}, [%2];\n" : "=r"(r0), "=r"(r1) : "r"(a) : "memory");
}

__device__ __forceinline__ void mma16816(float* d, const uint32_t* a, uint32_t b0, uint32_t b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
      "{%0,%1,%2,%3};\n"
      : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}
__device__ __forceinline__ void mma1688(float* d, uint32_t a0, uint32_t a1, uint32_t b0) {
  asm volatile(
      "mma.sync.aligned.m16n8k8.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5}, {%6}, {%0,%1,%2,%3};\n"
      : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
      : "r"(a0), "r"(a1), "r"(b0));
}

// Stage the fp32 master weights as bf16 (transposed copies where the
// B operand needs them) and the biases as fp32.
__device__ void stage_weights(const float* __restrict__ w, char* sm, bool train) {
  uint16_t* W1t = (uint16_t*)(sm + Smem::W1t);
  uint16_t* W2t = (uint16_t*)(sm + Smem::W2t);
  uint16_t* W2 = (uint16_t*)(sm + Smem::W2);
  uint16_t* W3t = (uint16_t*)(sm + Smem::W3t);
  uint16_t* W3 = (uint16_t*)(sm + Smem::W3);
  float* bias = (float*)(sm + Smem::Bias);
  for (int q = threadIdx.x; q < KIN * HID; q += blockDim.x) {
    int k = q / HID, o = q % HID;
    W1t[o * LDX + k] = bf(w[W1_OFF + q]);
  }
  for (int q = threadIdx.x; q < HID * HID; q += blockDim.x) {
    int k = q / HID, o = q % HID;
    uint16_t v = bf(w[W2_OFF + q]);
    W2t[o * LDH + k] = v;
    if (train) W2[k * LDH + o] = v;
  }
  for (int q = threadIdx.x; q < HID * KOUT; q += blockDim.x) {
    int k = q / KOUT, o = q % KOUT;
    uint16_t v = bf(w[W3_OFF + q]);
    W3t[o * LDH + k] = v;
    if (train) W3[k * KOUT + o] = v;
  }
  for (int q = threadIdx.x; q < 2 * HID + KOUT; q += blockDim.x) {
    int src = q < HID ? B1_OFF + q : (q < 2 * HID ? B2_OFF + q - HID : B3_OFF + q - 2 * HID);
    bias[q] = w[src];
  }
}

// The 16 neighbour indices and distances of a point, loaded ahead of their use.
struct KnnRow {
  int idx[KNN];
  float dist[KNN];
};
__device__ __forceinline__ void load_row(KnnRow& r, const int* __restrict__ knn_idx,
                                         const float* __restrict__ knn_dist, int64_t n, int64_t i, bool vec) {
  if (i < n) {
    if (vec) {  // rows are 64 bytes: 16-byte loads when the arrays start on 16 bytes
      #pragma unroll
      for (int q = 0; q < KNN / 4; ++q) {
        const int4 a = __ldg(reinterpret_cast<const int4*>(knn_idx + i * KNN) + q);
        const float4 b = __ldg(reinterpret_cast<const float4*>(knn_dist + i * KNN) + q);
        r.idx[4 * q] = a.x; r.idx[4 * q + 1] = a.y; r.idx[4 * q + 2] = a.z; r.idx[4 * q + 3] = a.w;
        r.dist[4 * q] = b.x; r.dist[4 * q + 1] = b.y; r.dist[4 * q + 2] = b.z; r.dist[4 * q + 3] = b.w;
      }
    } else {
      #pragma unroll
      for (int a = 0; a < KNN; ++a) { r.idx[a] = knn_idx[i * KNN + a]; r.dist[a] = knn_dist[i * KNN + a]; }
    }
  } else {
    #pragma unroll
    for (int a = 0; a < KNN; ++a) { r.idx[a] = -1; r.dist[a] = 0.f; }
  }
}
__device__ __forceinline__ void stage_row(const KnnRow& r, int p, int* s_idx, float2* s_dbar) {
  float s = 0.f;
  #pragma unroll
  for (int a = 0; a < KNN; ++a) { s_idx[p * LDI + a] = r.idx[a]; s += r.dist[a]; }
  float d = s / (float)KNN;
  d = d > 1e-12f ? d : 1e-12f;
  s_dbar[p] = make_float2(d, 1.f / d);
}

// bf16 of the float quotient o / d, given r = 1 / d: the product o r is within
// two units in the last place of the quotient, so both round to the same bf16
// unless the product lies within a few units of the midpoint of two bf16
// values; only then (about one value in 4000) the division is carried out.
__device__ __forceinline__ uint16_t bf_quotient(float o, float d, float r) {
  float q = o * r;
  if (((__float_as_uint(q) & 0xffffu) - 0x7ff8u) < 0x11u) q = o / d;
  return bf(q);
}

// Features of the batch's points into the bf16 tile X[BATCH][LDX] by NT
// threads, from the staged neighbour rows.  A thread takes single (point,
// neighbour, component) values: consecutive lanes read the components of one
// neighbour and write consecutive features, so a warp's gather touches a third
// of the sectors that whole neighbours per lane would.  Three rounds of NT
// values cover STEP points, so a round's neighbour and component are the same
// for all of a thread's points; GRP gathers are in flight per thread, since the
// builders' time is the gathers' latency (a step of 2M points: 4 in flight 842
// us, 16 784 us; with the division of every value 923 us).
template <int NT>
__device__ __forceinline__ void build_features(int tid, const float* __restrict__ pts, const float* __restrict__ nrm,
                                               int64_t n, int64_t base, const int* s_idx, const float2* s_dbar,
                                               uint16_t* X) {
  constexpr int STEP = NT * 3 / 48, GRP = BATCH / STEP < 16 ? BATCH / STEP : 16;
  static_assert(NT * 3 % 48 == 0 && BATCH % (STEP * GRP) == 0, "rounds repeat every STEP points");
  #pragma unroll 1
  for (int r = 0; r < 3; ++r) {
    const int p0 = (tid + NT * r) / 48, f = (tid + NT * r) % 48, c = f % 3;
    const int* idx = s_idx + p0 * LDI + f / 3;
    const float2* dbar = s_dbar + p0;
    const float* own = pts + 3 * (base + p0) + c;
    uint16_t* x = X + p0 * LDX + f;
    #pragma unroll 1
    for (int q = 0; q < BATCH / STEP; q += GRP) {
      float o[GRP], nn[GRP];
      #pragma unroll
      for (int e = 0; e < GRP; ++e) {
        const int j = idx[e * STEP * LDI];
        o[e] = nn[e] = 0.f;
        if (j >= 0) {  // (-1 for the points past n too)
          o[e] = __ldg(pts + 3 * (int64_t)j + c) - __ldg(own + e * STEP * 3);
          nn[e] = __ldg(nrm + 3 * (int64_t)j + c);
        }
      }
      #pragma unroll
      for (int e = 0; e < GRP; ++e) {
        const float2 d = dbar[e * STEP];  // mean neighbour distance and its reciprocal
        x[e * STEP * LDX] = bf_quotient(o[e], d.x, d.y);
        x[e * STEP * LDX + 48] = bf(nn[e]);
      }
      idx += GRP * STEP * LDI;
      dbar += GRP * STEP;
      own += GRP * STEP * 3;
      x += GRP * STEP * LDX;
    }
  }
  for (int e = tid; e < BATCH * (KIN - 96); e += NT) {
    const int p = e / (KIN - 96), f = 96 + e % (KIN - 96);
    const float v = (f < 99 && base + p < n) ? __ldg(nrm + 3 * (base + p) + (f - 96)) : 0.f;
    X[p * LDX + f] = bf(v);
  }
}

// Forward pass of the warp's 16 rows (m0 .. m0+15 of the batch).  h1, h2 are
// the post-ReLU fp32 activations in accumulator layout; y the outputs.
__device__ __forceinline__ void forward_rows(const char* sm, const uint16_t* X, int m0, float (&h1)[8][4],
                                             float (&h2)[8][4], float (&y)[4]) {
  const int lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3, l8 = lane & 7, mi = lane >> 3;
  // ldmatrix rows: A tiles (rows 0-7 | 8-15) x (k 0-7 | 8-15); weight tiles two n8 tiles x (k 0-7 | 8-15)
  const uint16_t* ax = X + (m0 + l8 + (mi & 1) * 8) * LDX + (mi >> 1) * 8;
  const uint16_t* w1 = (const uint16_t*)(sm + Smem::W1t) + (l8 + (mi >> 1) * 8) * LDX + (mi & 1) * 8;
  const uint16_t* w2 = (const uint16_t*)(sm + Smem::W2t) + (l8 + (mi >> 1) * 8) * LDH + (mi & 1) * 8;
  const uint16_t* W3t = (const uint16_t*)(sm + Smem::W3t);
  const float* bias = (const float*)(sm + Smem::Bias);
  #pragma unroll
  for (int j = 0; j < 8; ++j) h1[j][0] = h1[j][1] = h1[j][2] = h1[j][3] = 0.f;
  #pragma unroll
  for (int s = 0; s < KIN / 16; ++s) {
    uint32_t a[4];
    ldsm4(a, ax + 16 * s);
    #pragma unroll
    for (int j = 0; j < 8; j += 2) {
      uint32_t b[4];
      ldsm4(b, w1 + 8 * j * LDX + 16 * s);
      mma16816(h1[j], a, b[0], b[1]);
      mma16816(h1[j + 1], a, b[2], b[3]);
    }
  }
  #pragma unroll
  for (int j = 0; j < 8; ++j) {
    float b0 = bias[8 * j + 2 * t], b1 = bias[8 * j + 2 * t + 1];
    h1[j][0] = fmaxf(h1[j][0] + b0, 0.f); h1[j][1] = fmaxf(h1[j][1] + b1, 0.f);
    h1[j][2] = fmaxf(h1[j][2] + b0, 0.f); h1[j][3] = fmaxf(h1[j][3] + b1, 0.f);
  }
  #pragma unroll
  for (int j = 0; j < 8; ++j) h2[j][0] = h2[j][1] = h2[j][2] = h2[j][3] = 0.f;
  #pragma unroll
  for (int s = 0; s < HID / 16; ++s) {
    uint32_t a[4] = {pack(h1[2 * s][0], h1[2 * s][1]), pack(h1[2 * s][2], h1[2 * s][3]),
                     pack(h1[2 * s + 1][0], h1[2 * s + 1][1]), pack(h1[2 * s + 1][2], h1[2 * s + 1][3])};
    #pragma unroll
    for (int j = 0; j < 8; j += 2) {
      uint32_t b[4];
      ldsm4(b, w2 + 8 * j * LDH + 16 * s);
      mma16816(h2[j], a, b[0], b[1]);
      mma16816(h2[j + 1], a, b[2], b[3]);
    }
  }
  #pragma unroll
  for (int j = 0; j < 8; ++j) {
    float b0 = bias[HID + 8 * j + 2 * t], b1 = bias[HID + 8 * j + 2 * t + 1];
    h2[j][0] = fmaxf(h2[j][0] + b0, 0.f); h2[j][1] = fmaxf(h2[j][1] + b1, 0.f);
    h2[j][2] = fmaxf(h2[j][2] + b0, 0.f); h2[j][3] = fmaxf(h2[j][3] + b1, 0.f);
  }
  y[0] = y[1] = y[2] = y[3] = 0.f;
  #pragma unroll
  for (int s = 0; s < HID / 16; ++s) {
    uint32_t a[4] = {pack(h2[2 * s][0], h2[2 * s][1]), pack(h2[2 * s][2], h2[2 * s][3]),
                     pack(h2[2 * s + 1][0], h2[2 * s + 1][1]), pack(h2[2 * s + 1][2], h2[2 * s + 1][3])};
    int k0 = 16 * s + 2 * t;
    mma16816(y, a, ld32(W3t + g * LDH + k0), ld32(W3t + g * LDH + k0 + 8));
  }
  float b0 = bias[2 * HID + 2 * t], b1 = bias[2 * HID + 2 * t + 1];
  y[0] += b0; y[1] += b1; y[2] += b0; y[3] += b1;
}

// Rows of a batch staged, then its features (all FWD_T threads of a forward kernel).
__device__ __forceinline__ void build_batch(const float* __restrict__ pts, const float* __restrict__ nrm,
                                            const int* __restrict__ knn_idx, const float* __restrict__ knn_dist,
                                            int64_t n, int64_t base, bool vec, char* sm) {
  if (threadIdx.x < BATCH) {
    KnnRow r;
    load_row(r, knn_idx, knn_dist, n, base + threadIdx.x, vec);
    stage_row(r, threadIdx.x, (int*)(sm + Smem::Idx), (float2*)(sm + Smem::Dbar));
  }
  __syncthreads();
  build_features<FWD_T>(threadIdx.x, pts, nrm, n, base, (const int*)(sm + Smem::Idx), (const float2*)(sm + Smem::Dbar),
                        (uint16_t*)(sm + Smem::X));
  __syncthreads();
}

// y rows (m0+g, m0+g+8), cols (2t, 2t+1) -> out[row][col]
__global__ void __launch_bounds__(FWD_T, 3) k_mlp_forward(const float* __restrict__ pts, const float* __restrict__ nrm,
                                                         const int* __restrict__ knn_idx,
                                                         const float* __restrict__ knn_dist, int64_t n, bool vec,
                                                         const float* __restrict__ w, float* __restrict__ out) {
  gs_wait_previous();
  extern __shared__ __align__(16) char sm[];
  stage_weights(w, sm, false);
  int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
  int64_t nb = (n + BATCH - 1) / BATCH;
  for (int64_t b = blockIdx.x; b < nb; b += gridDim.x) {
    int64_t base = b * BATCH;
    build_batch(pts, nrm, knn_idx, knn_dist, n, base, vec, sm);
    float h1[8][4], h2[8][4], y[4];
    int m0 = warp * 16;
    forward_rows(sm, (const uint16_t*)(sm + Smem::X), m0, h1, h2, y);
    int64_t r0 = base + m0 + g, r1 = r0 + 8;
    if (r0 < n) { out[r0 * KOUT + 2 * t] = y[0]; out[r0 * KOUT + 2 * t + 1] = y[1]; }
    if (r1 < n) { out[r1 * KOUT + 2 * t] = y[2]; out[r1 * KOUT + 2 * t + 1] = y[3]; }
    __syncthreads();  // the feature tile is rebuilt next iteration
  }
}

// Initial Gaussian parameters: plane 1 (log-scale, logit opacity) and plane 2
// (rotation).  Plain form: isotropic log(mean 3-NN distance), identity rotation,
// logit_default.  With the MLP: log-scale = log(d3) + y[0:3], rotation y[3:7],
// logit y[7]; any non-finite output (or a rotation of norm < 1e-6) falls back to
// the plain values for that Gaussian.
__device__ __forceinline__ void write_init(float4* __restrict__ params, int64_t N, int64_t i, float d3, const float* y,
                                           bool have_y, float logit_default) {
  float ls = logf(fmaxf(d3, 1e-7f));
  float4 sop = make_float4(ls, ls, ls, logit_default);
  float4 q = make_float4(1.f, 0.f, 0.f, 0.f);
  if (have_y) {
    bool ok = true;
    for (int c = 0; c < KOUT; ++c) ok = ok && isfinite(y[c]);
    float qn = sqrtf(y[3] * y[3] + y[4] * y[4] + y[5] * y[5] + y[6] * y[6]);
    ok = ok && qn > 1e-6f;
    if (ok) {
      sop = make_float4(ls + y[0], ls + y[1], ls + y[2], y[7]);
      q = make_float4(y[3], y[4], y[5], y[6]);
    }
  }
  params[N + i] = sop;
  params[2 * N + i] = q;
}

__global__ void k_plain_init(const float* __restrict__ knn_dist, int k, int64_t n, float logit_default,
                             float4* __restrict__ params, int64_t N) {
  gs_wait_previous();
  int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i >= n) return;
  float d3 = (knn_dist[i * k] + knn_dist[i * k + 1] + knn_dist[i * k + 2]) / 3.f;
  write_init(params, N, i, d3, nullptr, false, logit_default);
}

__global__ void __launch_bounds__(FWD_T, 3) k_mlp_init(const float* __restrict__ pts, const float* __restrict__ nrm,
                                                      const int* __restrict__ knn_idx,
                                                      const float* __restrict__ knn_dist, int64_t n, bool vec,
                                                      const float* __restrict__ w, float logit_default,
                                                      float4* __restrict__ params, int64_t N) {
  gs_wait_previous();
  extern __shared__ __align__(16) char sm[];
  stage_weights(w, sm, false);
  int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
  float* ybuf = (float*)(sm + Smem::Y);  // [BATCH][8] fp32 staging of the outputs
  int64_t nb = (n + BATCH - 1) / BATCH;
  for (int64_t b = blockIdx.x; b < nb; b += gridDim.x) {
    int64_t base = b * BATCH;
    build_batch(pts, nrm, knn_idx, knn_dist, n, base, vec, sm);
    float h1[8][4], h2[8][4], y[4];
    int m0 = warp * 16;
    forward_rows(sm, (const uint16_t*)(sm + Smem::X), m0, h1, h2, y);
    ybuf[(m0 + g) * KOUT + 2 * t] = y[0];
    ybuf[(m0 + g) * KOUT + 2 * t + 1] = y[1];
    ybuf[(m0 + g + 8) * KOUT + 2 * t] = y[2];
    ybuf[(m0 + g + 8) * KOUT + 2 * t + 1] = y[3];
    __syncthreads();
    if (threadIdx.x < BATCH && base + threadIdx.x < n) {
      int64_t i = base + threadIdx.x;
      float d3 = (knn_dist[i * KNN] + knn_dist[i * KNN + 1] + knn_dist[i * KNN + 2]) / 3.f;
      write_init(params, N, i, d3, ybuf + threadIdx.x * KOUT, true, logit_default);
    }
  }
}

__device__ __forceinline__ void bar_sync(int id, int threads) {
  asm volatile("bar.sync %0, %1;\n" ::"r"(id), "r"(threads) : "memory");
}

// One training step's gradients: forward, loss (sum of squared errors times
// `scale`), backward; dW accumulated into `grad` (zeroed by the caller).
//
// One CTA per SM (183 KB of tiles): 8 warps multiply batch t while 4 warps
// build the features of batch t + 1 into the other tile (with the neighbour
// rows of t + 2 already loading), one block barrier per batch.  The weight
// gradients' 92 m16n8 tiles are split over the 8 warps as (half of the rows) x
// (16 columns), at most 12 tiles each, so every operand fragment serves several
// mma; a batch's tiles are summed from zero on the tensor cores and added to
// fp32 registers, which leave for memory once, at the end.  Bias gradients are
// the same columns multiplied by a fragment of ones.  2M points: 3792 us with
// one warp group per SM doing both in turn, operands read as 16-bit scalars
// and gradients kept in shared memory; 784 us.
__global__ void __launch_bounds__(CONS_T + PROD_T, 1)
    k_mlp_train(const float* __restrict__ pts, const float* __restrict__ nrm, const int* __restrict__ knn_idx,
                const float* __restrict__ knn_dist, const float* __restrict__ target, int64_t n, bool vec,
                const float* __restrict__ w, float scale, float* __restrict__ grad, float* __restrict__ loss) {
  gs_wait_previous();
  extern __shared__ __align__(16) char sm[];
  int* s_idx = (int*)(sm + Smem::Idx);
  float2* s_dbar = (float2*)(sm + Smem::Dbar);
  const int64_t nb = (n + BATCH - 1) / BATCH;
  const int64_t b0 = blockIdx.x;
  const int steps = b0 < nb ? (int)((nb - b0 + gridDim.x - 1) / gridDim.x) : 0;
  auto base_of = [&](int k) { return (b0 + (int64_t)k * gridDim.x) * BATCH; };
  auto tile = [&](int k) { return (uint16_t*)(sm + ((k & 1) ? Smem::X2 : Smem::X)); };
  // the barrier of both roles, which meet in it from different places of the code
  auto both_roles = []() { bar_sync(0, CONS_T + PROD_T); };
  stage_weights(w, sm, true);
  __syncthreads();
  if (threadIdx.x >= CONS_T) {
    // ---- feature builders
    const int tid = threadIdx.x - CONS_T;
    KnnRow row;
    if (steps > 0) load_row(row, knn_idx, knn_dist, n, base_of(0) + tid, vec);
    for (int k = 0; k < steps; ++k) {  // batch k, while the other warps multiply batch k - 1
      stage_row(row, tid, s_idx, s_dbar);
      if (k + 1 < steps) load_row(row, knn_idx, knn_dist, n, base_of(k + 1) + tid, vec);
      bar_sync(2, PROD_T);
      build_features<PROD_T>(tid, pts, nrm, n, base_of(k), s_idx, s_dbar, tile(k));
      both_roles();
    }
    both_roles();  // the last batch is multiplied
    return;
  }
  // ---- multipliers
  uint16_t* sH1 = (uint16_t*)(sm + Smem::H1);
  uint16_t* sH2 = (uint16_t*)(sm + Smem::H2);
  uint16_t* sdH1 = (uint16_t*)(sm + Smem::dH1);
  uint16_t* sdH2 = (uint16_t*)(sm + Smem::dH2);
  uint16_t* sdY = (uint16_t*)(sm + Smem::dY);
  const uint16_t* W2 = (const uint16_t*)(sm + Smem::W2);
  const uint16_t* W3 = (const uint16_t*)(sm + Smem::W3);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
  const int l8 = lane & 7, mi = lane >> 3;
  const int m0 = warp * 16;
  // weight-gradient tiles of this warp: rows 64 half .. of dW1 (4 or 3 m16 tiles), 32 half .. of dW2, 16 nq .. of
  // dW3 (half 1), all in columns 16 nq ..
  const int half = warp & 1, nq = warp >> 1;
  float g1[4][2][4], g2[2][2][4], g3[4], gb[2][2], gb3[2];
  #pragma unroll
  for (int e = 0; e < 4; ++e) {
    #pragma unroll
    for (int m = 0; m < 4; ++m) g1[m][0][e] = g1[m][1][e] = 0.f;
    #pragma unroll
    for (int m = 0; m < 2; ++m) g2[m][0][e] = g2[m][1][e] = 0.f;
    g3[e] = 0.f;
  }
  gb[0][0] = gb[0][1] = gb[1][0] = gb[1][1] = gb3[0] = gb3[1] = 0.f;
  const uint32_t ONES[4] = {0x3f803f80u, 0x3f803f80u, 0x3f803f80u, 0x3f803f80u};
  float lsum = 0.f;
  for (int k = 0; k < steps; ++k) {
    both_roles();  // batch k's features are in its tile; every warp is done with batch k - 1
    const uint16_t* X = tile(k);
    const int64_t r0 = base_of(k) + m0 + g, r1 = r0 + 8;
    float tg[4] = {0.f, 0.f, 0.f, 0.f};
    if (r0 < n) { tg[0] = __ldg(target + r0 * KOUT + 2 * t); tg[1] = __ldg(target + r0 * KOUT + 2 * t + 1); }
    if (r1 < n) { tg[2] = __ldg(target + r1 * KOUT + 2 * t); tg[3] = __ldg(target + r1 * KOUT + 2 * t + 1); }
    uint32_t on1 = 0u, on2 = 0u;  // active ReLUs, bit 4 j + e
    uint32_t ady0, ady1;
    {
      float h1[8][4], h2[8][4], y[4];
      forward_rows(sm, X, m0, h1, h2, y);
      float dy[4];
      #pragma unroll
      for (int e = 0; e < 4; ++e) {
        const float d = (e < 2 ? r0 : r1) < n ? y[e] - tg[e] : 0.f;
        lsum += d * d;
        dy[e] = 2.f * d * scale;
      }
      ady0 = pack(dy[0], dy[1]); ady1 = pack(dy[2], dy[3]);
      *reinterpret_cast<uint32_t*>(sdY + (m0 + g) * KOUT + 2 * t) = ady0;
      *reinterpret_cast<uint32_t*>(sdY + (m0 + g + 8) * KOUT + 2 * t) = ady1;
      // activations as bf16 tiles for the weight gradients
      #pragma unroll
      for (int j = 0; j < 8; ++j) {
        *reinterpret_cast<uint32_t*>(sH1 + (m0 + g) * LDH + 8 * j + 2 * t) = pack(h1[j][0], h1[j][1]);
        *reinterpret_cast<uint32_t*>(sH1 + (m0 + g + 8) * LDH + 8 * j + 2 * t) = pack(h1[j][2], h1[j][3]);
        *reinterpret_cast<uint32_t*>(sH2 + (m0 + g) * LDH + 8 * j + 2 * t) = pack(h2[j][0], h2[j][1]);
        *reinterpret_cast<uint32_t*>(sH2 + (m0 + g + 8) * LDH + 8 * j + 2 * t) = pack(h2[j][2], h2[j][3]);
        #pragma unroll
        for (int e = 0; e < 4; ++e) {
          on1 |= (h1[j][e] > 0.f ? 1u : 0u) << (4 * j + e);
          on2 |= (h2[j][e] > 0.f ? 1u : 0u) << (4 * j + e);
        }
      }
    }
    {
      // dH2 = dY W3^T, masked by the ReLU of layer 2, rounded to bf16
      uint32_t d2[8][2];
      #pragma unroll
      for (int j = 0; j < 8; ++j) {
        float d[4] = {0.f, 0.f, 0.f, 0.f};
        mma1688(d, ady0, ady1, ld32(W3 + (8 * j + g) * KOUT + 2 * t));
        #pragma unroll
        for (int e = 0; e < 4; ++e) d[e] = (on2 >> (4 * j + e)) & 1u ? d[e] : 0.f;
        d2[j][0] = pack(d[0], d[1]); d2[j][1] = pack(d[2], d[3]);
        *reinterpret_cast<uint32_t*>(sdH2 + (m0 + g) * LDH + 8 * j + 2 * t) = d2[j][0];
        *reinterpret_cast<uint32_t*>(sdH2 + (m0 + g + 8) * LDH + 8 * j + 2 * t) = d2[j][1];
      }
      // dH1 = dH2 W2^T, masked by the ReLU of layer 1
      float d1[8][4];
      #pragma unroll
      for (int j = 0; j < 8; ++j) d1[j][0] = d1[j][1] = d1[j][2] = d1[j][3] = 0.f;
      const uint16_t* w2 = W2 + (l8 + (mi >> 1) * 8) * LDH + (mi & 1) * 8;
      #pragma unroll
      for (int s = 0; s < HID / 16; ++s) {
        const uint32_t a[4] = {d2[2 * s][0], d2[2 * s][1], d2[2 * s + 1][0], d2[2 * s + 1][1]};
        #pragma unroll
        for (int j = 0; j < 8; j += 2) {
          uint32_t b[4];
          ldsm4(b, w2 + 8 * j * LDH + 16 * s);
          mma16816(d1[j], a, b[0], b[1]);
          mma16816(d1[j + 1], a, b[2], b[3]);
        }
      }
      #pragma unroll
      for (int j = 0; j < 8; ++j) {
        #pragma unroll
        for (int e = 0; e < 4; ++e) d1[j][e] = (on1 >> (4 * j + e)) & 1u ? d1[j][e] : 0.f;
        *reinterpret_cast<uint32_t*>(sdH1 + (m0 + g) * LDH + 8 * j + 2 * t) = pack(d1[j][0], d1[j][1]);
        *reinterpret_cast<uint32_t*>(sdH1 + (m0 + g + 8) * LDH + 8 * j + 2 * t) = pack(d1[j][2], d1[j][3]);
      }
    }
    bar_sync(1, CONS_T);
    // weight gradients over the batch's points: dW1 = X^T dH1, dW2 = H1^T dH2, dW3 = H2^T dY; both operands
    // transposed on the way into registers (ldmatrix rows: points)
    const int arow = l8 + (mi >> 1) * 8, acol = (mi & 1) * 8;  // A: (points 0-7 | 8-15) x (rows 0-7 | 8-15)
    const int brow = l8 + (mi & 1) * 8, bcol = 16 * nq + (mi >> 1) * 8;
    {
      float a1[4][2][4], s1[2][4];
      #pragma unroll
      for (int e = 0; e < 4; ++e) {
        #pragma unroll
        for (int m = 0; m < 4; ++m) a1[m][0][e] = a1[m][1][e] = 0.f;
        s1[0][e] = s1[1][e] = 0.f;
      }
      #pragma unroll 2
      for (int s = 0; s < BATCH / 16; ++s) {
        uint32_t b[4];
        ldsm4<true>(b, sdH1 + (16 * s + brow) * LDH + bcol);
        #pragma unroll
        for (int m = 0; m < 4; ++m) {
          if (half == 1 && m == 3) continue;  // 7 row tiles: 4 and 3
          uint32_t a[4];
          ldsm4<true>(a, X + (16 * s + arow) * LDX + 64 * half + 16 * m + acol);
          mma16816(a1[m][0], a, b[0], b[1]);
          mma16816(a1[m][1], a, b[2], b[3]);
        }
        if (half == 0) {
          mma16816(s1[0], ONES, b[0], b[1]);
          mma16816(s1[1], ONES, b[2], b[3]);
        }
      }
      #pragma unroll
      for (int q = 0; q < 2; ++q) {
        #pragma unroll
        for (int e = 0; e < 4; ++e)
          #pragma unroll
          for (int m = 0; m < 4; ++m) g1[m][q][e] += a1[m][q][e];
        if (half == 0) { gb[q][0] += s1[q][0]; gb[q][1] += s1[q][1]; }
      }
    }
    {
      float a2[2][2][4], a3[4], s2[2][4], s3[4];
      #pragma unroll
      for (int e = 0; e < 4; ++e) {
        a2[0][0][e] = a2[0][1][e] = a2[1][0][e] = a2[1][1][e] = 0.f;
        a3[e] = s2[0][e] = s2[1][e] = s3[e] = 0.f;
      }
      #pragma unroll 2
      for (int s = 0; s < BATCH / 16; ++s) {
        uint32_t b[4];
        ldsm4<true>(b, sdH2 + (16 * s + brow) * LDH + bcol);
        #pragma unroll
        for (int m = 0; m < 2; ++m) {
          uint32_t a[4];
          ldsm4<true>(a, sH1 + (16 * s + arow) * LDH + 32 * half + 16 * m + acol);
          mma16816(a2[m][0], a, b[0], b[1]);
          mma16816(a2[m][1], a, b[2], b[3]);
        }
        if (half == 1) {
          mma16816(s2[0], ONES, b[0], b[1]);
          mma16816(s2[1], ONES, b[2], b[3]);
          uint32_t a[4], y0, y1;
          ldsm2t(y0, y1, sdY + (16 * s + (lane & 15)) * KOUT);
          ldsm4<true>(a, sH2 + (16 * s + arow) * LDH + 16 * nq + acol);
          mma16816(a3, a, y0, y1);
          if (nq == 0) mma16816(s3, ONES, y0, y1);
        }
      }
      #pragma unroll
      for (int q = 0; q < 2; ++q) {
        #pragma unroll
        for (int e = 0; e < 4; ++e) { g2[0][q][e] += a2[0][q][e]; g2[1][q][e] += a2[1][q][e]; }
        if (half == 1) { gb[q][0] += s2[q][0]; gb[q][1] += s2[q][1]; }
      }
      #pragma unroll
      for (int e = 0; e < 4; ++e) g3[e] += a3[e];
      gb3[0] += s3[0]; gb3[1] += s3[1];
    }
  }
  both_roles();  // (the builders' last barrier)
  // accumulator element e of a tile: row g (+ 8 for e >= 2), column 2 t + (e & 1)
  auto put = [&](int off, int ncols, int row, int col, const float* v) {
    #pragma unroll
    for (int e = 0; e < 4; ++e) {
      const int r = row + g + (e >> 1) * 8, c = col + 2 * t + (e & 1);
      if (v[e] != 0.f) atomicAdd(grad + off + r * ncols + c, v[e]);
    }
  };
  #pragma unroll
  for (int q = 0; q < 2; ++q) {
    #pragma unroll
    for (int m = 0; m < 4; ++m)
      if (half == 0 || m < 3) put(W1_OFF, HID, 64 * half + 16 * m, 16 * nq + 8 * q, g1[m][q]);
    #pragma unroll
    for (int m = 0; m < 2; ++m) put(W2_OFF, HID, 32 * half + 16 * m, 16 * nq + 8 * q, g2[m][q]);
    if (g == 0) {  // every row of a ones product holds the column sums
      float* gbias = grad + (half == 0 ? B1_OFF : B2_OFF) + 16 * nq + 8 * q + 2 * t;
      atomicAdd(gbias, gb[q][0]);
      atomicAdd(gbias + 1, gb[q][1]);
    }
  }
  if (half == 1) put(W3_OFF, KOUT, 16 * nq, 0, g3);
  if (half == 1 && nq == 0 && g == 0) {
    atomicAdd(grad + B3_OFF + 2 * t, gb3[0]);
    atomicAdd(grad + B3_OFF + 2 * t + 1, gb3[1]);
  }
  #pragma unroll
  for (int o = 16; o > 0; o >>= 1) lsum += __shfl_xor_sync(0xffffffffu, lsum, o);
  if (lane == 0 && lsum != 0.f) atomicAdd(loss, lsum * scale);
}

__global__ void __launch_bounds__(FWD_T) k_features_out(const float* __restrict__ pts, const float* __restrict__ nrm,
                                                        const int* __restrict__ knn_idx,
                                                        const float* __restrict__ knn_dist, int64_t n, bool vec,
                                                        uint16_t* __restrict__ X) {
  gs_wait_previous();
  extern __shared__ __align__(16) char sm[];
  int64_t nb = (n + BATCH - 1) / BATCH;
  const uint16_t* sX = (const uint16_t*)(sm + Smem::X);
  for (int64_t b = blockIdx.x; b < nb; b += gridDim.x) {
    int64_t base = b * BATCH;
    build_batch(pts, nrm, knn_idx, knn_dist, n, base, vec, sm);
    for (int q = threadIdx.x; q < BATCH * KIN; q += blockDim.x) {
      int p = q / KIN, f = q % KIN;
      if (base + p < n) X[(base + p) * KIN + f] = sX[p * LDX + f];
    }
  }
}

int grid_for(int64_t n, int per_sm) {
  int dev = 0, sms = 148;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  int64_t nb = (n + BATCH - 1) / BATCH;
  int64_t cap = (int64_t)sms * per_sm;
  return (int)(nb < cap ? (nb > 0 ? nb : 1) : cap);
}

template <typename K>
int set_smem(K kernel, int bytes) {
  return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes) == cudaSuccess ? GS_OK
                                                                                                          : GS_ERR_CUDA;
}

bool rows_aligned(const int32_t* idx, const float* dist) { return (((uintptr_t)idx | (uintptr_t)dist) & 15u) == 0; }

bool knn_args_ok(const float* pts, const float* nrm, const int32_t* idx, const float* dist, int64_t n) {
  return pts && nrm && idx && dist && n >= 0;
}

}  // namespace

GS_API int gs_mlp_param_count(void) { return NPARAM; }

GS_API int gs_mlp_features(const float* points, const float* normals, const int32_t* knn_idx, const float* knn_dist,
                           int64_t n, uint16_t* features, gs_stream_t stream) {
  GS_RANGE("gs_mlp_features");
  if (!knn_args_ok(points, normals, knn_idx, knn_dist, n) || !features) return GS_ERR_INVALID;
  if (n == 0) return GS_OK;
  if (set_smem(k_features_out, Smem::FWD_END) != GS_OK) return GS_ERR_CUDA;
  gs_launch(k_features_out, grid_for(n, 3), FWD_T, Smem::FWD_END, (cudaStream_t)stream, points, normals, knn_idx,
      knn_dist, n, rows_aligned(knn_idx, knn_dist), features);
  return gs_check_launch();
}

GS_API int gs_mlp_forward(const float* points, const float* normals, const int32_t* knn_idx, const float* knn_dist,
                          int64_t n, const float* weights, float* out, gs_stream_t stream) {
  GS_RANGE("gs_mlp_forward");
  if (!knn_args_ok(points, normals, knn_idx, knn_dist, n) || !weights || !out) return GS_ERR_INVALID;
  if (n == 0) return GS_OK;
  if (set_smem(k_mlp_forward, Smem::FWD_END) != GS_OK) return GS_ERR_CUDA;
  gs_launch(k_mlp_forward, grid_for(n, 3), FWD_T, Smem::FWD_END, (cudaStream_t)stream, points, normals, knn_idx,
      knn_dist, n, rows_aligned(knn_idx, knn_dist), weights, out);
  return gs_check_launch();
}

GS_API int gs_mlp_train_step(const float* points, const float* normals, const int32_t* knn_idx,
                             const float* knn_dist, const float* targets, int64_t n, float* weights, float* grad,
                             float* m, float* v, float lr, const int32_t* d_step, float* d_loss, gs_stream_t stream) {
  GS_RANGE("gs_mlp_train_step");
  if (!knn_args_ok(points, normals, knn_idx, knn_dist, n) || !targets || !weights || !grad || !m || !v ||
      !d_step || !d_loss || n < 1 || !(lr > 0.f))
    return GS_ERR_INVALID;
  cudaStream_t s = (cudaStream_t)stream;
  if (cudaMemsetAsync(grad, 0, sizeof(float) * NPARAM, s) != cudaSuccess ||
      cudaMemsetAsync(d_loss, 0, sizeof(float), s) != cudaSuccess)
    return GS_ERR_CUDA;
  if (set_smem(k_mlp_train, Smem::TRAIN_END) != GS_OK) return GS_ERR_CUDA;
  float scale = 1.0f / (8.0f * (float)n);
  gs_launch(k_mlp_train, grid_for(n, 1), CONS_T + PROD_T, Smem::TRAIN_END, s, points, normals, knn_idx, knn_dist,
      targets, n, rows_aligned(knn_idx, knn_dist), weights, scale, grad, d_loss);
  int r = gs_check_launch();
  if (r != GS_OK) return r;
  float lr4[4] = {lr, lr, lr, lr};
  return gs_adam_step(weights, grad, m, v, NPARAM / 4, 1, lr4, lr4, 0, 0.9f, 0.999f, 1e-8f, d_step, 0, nullptr,
                      stream);
}

GS_API int gs_init_gaussians(const float* points, const float* normals, const int32_t* knn_idx,
                             const float* knn_dist, int knn_k, int64_t n, const float* weights, float logit_default,
                             float* params, int64_t n_gauss, gs_stream_t stream) {
  GS_RANGE("gs_init_gaussians");
  if (!points || !knn_dist || !params || n < 0 || n > n_gauss || knn_k < 3) return GS_ERR_INVALID;
  if (weights && (!normals || !knn_idx || knn_k != KNN)) return GS_ERR_INVALID;
  if (n == 0) return GS_OK;
  cudaStream_t s = (cudaStream_t)stream;
  // means = the points
  if (cudaMemcpy2DAsync(params, 4 * sizeof(float), points, 3 * sizeof(float), 3 * sizeof(float), (size_t)n,
                        cudaMemcpyDeviceToDevice, s) != cudaSuccess)
    return GS_ERR_CUDA;
  if (!weights) {
    gs_launch(k_plain_init, (unsigned)((n + 255) / 256), 256, 0, s, knn_dist, knn_k, n, logit_default,
        (float4*)params, n_gauss);
  } else {
    if (set_smem(k_mlp_init, Smem::INIT_END) != GS_OK) return GS_ERR_CUDA;
    gs_launch(k_mlp_init, grid_for(n, 3), FWD_T, Smem::INIT_END, s, points, normals, knn_idx, knn_dist, n,
        rows_aligned(knn_idx, knn_dist), weights, logit_default, (float4*)params, n_gauss);
  }
  return gs_check_launch();
}
