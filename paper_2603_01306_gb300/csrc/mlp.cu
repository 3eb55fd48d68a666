// Per-coordinate warm-start network: 5 -> 64 -> 64 -> 1, ReLU after both
// hidden layers, inputs standardised as (x - shift) / scale; the child's
// starting point is beta^P_j + f(x_j) (the parent warm start of Sec. 5.3 plus a
// learned correction).  Weights live in one FP32 vector (layout in
// include/warmstart.h); with bf16 != 0 every kernel evaluates the network
// with the trainable entries rounded to BF16, accumulating in FP32.
//
// forward: BF16 weights: the 64 x 64 layer on the tensor cores (mma.sync
//          m16n8k16, BF16 operands, FP32 accumulation), 16 rows per warp:
//          each lane computes layer 1 for the A-fragment entries it holds and
//          splits them into three BF16 planes (exactly the FP32 value), so the
//          products are exact and only the FP32 sums round; layer 2's bias,
//          ReLU and the output layer follow on the accumulator fragments.
//          FP32 weights (the reference build of the network): one thread per
//          row on the CUDA cores, layer 2 fused with the output layer.
// grad:    tiles of 128 (64) rows per CTA, the three 64 x 64 products of a tile
//          register-tiled in FP32; one partial per CTA, summed in a fixed
//          order by a second kernel, so the gradient is bit-reproducible for a
//          given row count.
// adam:    one thread per trainable entry (Kingma and Ba, 2015).
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <cmath>
#include <cstdint>

#include "common.cuh"
#include "warmstart.h"

namespace {

constexpr int NIN = 5, NH = 64;
constexpr int O_W1 = 0, O_B1 = NH * NIN, O_W2 = O_B1 + NH, O_B2 = O_W2 + NH * NH, O_W3 = O_B2 + NH,
              O_B3 = O_W3 + NH, O_SHIFT = O_B3 + 1, O_SCALE = O_SHIFT + NIN;
static_assert(O_SHIFT == RELAX_MLP_NTRAIN, "layout");
static_assert(O_SCALE + NIN == RELAX_MLP_NPARAM, "layout");

constexpr int FWD_THREADS = 128;
constexpr int GRAD_T = 256;     // threads of the gradient kernel
constexpr int W2P = NH + 4;     // its padded row stride in shared memory (16-byte rows, distinct banks)

__device__ __forceinline__ float wround(float w, int bf16) {
  return bf16 ? __bfloat162float(__float2bfloat16_rn(w)) : w;
}

// the network's parameters in shared memory, FP32 (BF16-rounded when asked)
struct SW {
  float W1[NH * NIN], b1[NH], W2[NH * NH], b2[NH], w3[NH], b3, shift[NIN], iscale[NIN];
};

__device__ void load_weights(SW& s, const float* theta, int bf16) {
  for (int i = threadIdx.x; i < NH * NIN; i += blockDim.x) s.W1[i] = wround(theta[O_W1 + i], bf16);
  for (int i = threadIdx.x; i < NH * NH; i += blockDim.x) s.W2[i] = wround(theta[O_W2 + i], bf16);
  for (int i = threadIdx.x; i < NH; i += blockDim.x) {
    s.b1[i] = wround(theta[O_B1 + i], bf16);
    s.b2[i] = wround(theta[O_B2 + i], bf16);
    s.w3[i] = wround(theta[O_W3 + i], bf16);
  }
  if (threadIdx.x < NIN) {
    s.shift[threadIdx.x] = theta[O_SHIFT + threadIdx.x];
    s.iscale[threadIdx.x] = 1.0f / theta[O_SCALE + threadIdx.x];
  }
  if (threadIdx.x == 0) s.b3 = wround(theta[O_B3], bf16);
}

// layer 1 of one row: h1 = relu(W1 xs + b1)
__device__ __forceinline__ void layer1(const SW& s, const float* xs, float* h1) {
#pragma unroll
  for (int h = 0; h < NH; ++h) {
    float a = s.b1[h];
#pragma unroll
    for (int i = 0; i < NIN; ++i) a = fmaf(s.W1[h * NIN + i], xs[i], a);
    h1[h] = a > 0.f ? a : 0.f;
  }
}

__device__ __forceinline__ float dot64(const float* w, const float* h) {
  float a0 = 0.f, a1 = 0.f, a2 = 0.f, a3 = 0.f;
#pragma unroll
  for (int k = 0; k < NH; k += 4) {
    a0 = fmaf(w[k], h[k], a0);
    a1 = fmaf(w[k + 1], h[k + 1], a1);
    a2 = fmaf(w[k + 2], h[k + 2], a2);
    a3 = fmaf(w[k + 3], h[k + 3], a3);
  }
  return (a0 + a1) + (a2 + a3);
}

// ---- tensor-core forward (BF16 weights)
__device__ __forceinline__ uint32_t pack_bf16(__nv_bfloat16 lo, __nv_bfloat16 hi) {
  return (uint32_t)__bfloat16_as_ushort(lo) | ((uint32_t)__bfloat16_as_ushort(hi) << 16);
}
// x = p0 + p1 + p2 exactly (8 + 8 + 8 significand bits of an FP32 value)
__device__ __forceinline__ void split3_f32(float x, __nv_bfloat16 (&q)[3]) {
  q[0] = __float2bfloat16_rn(x);
  const float r1 = x - __bfloat162float(q[0]);
  q[1] = __float2bfloat16_rn(r1);
  q[2] = __float2bfloat16_rn(r1 - __bfloat162float(q[1]));
}
__device__ __forceinline__ void mma_bf16_16816(float (&d)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, "
      "{%0, %1, %2, %3};"
      : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

constexpr int MMA_WARPS = 4;
constexpr int W2LD = NH + 8;   // padded row of W2 in shared memory: the 8 row groups hit distinct banks

__global__ void __launch_bounds__(32 * MMA_WARPS) mlp_forward_mma_kernel(const float* theta, const float* feat,
                                                                        const float* base, int64_t rows, float* out) {
  __shared__ SW s;
  __shared__ __align__(16) __nv_bfloat16 W2b[NH * W2LD];   // W2 [o][h], exact in BF16
  load_weights(s, theta, 1);
  for (int i = threadIdx.x; i < NH * NH; i += blockDim.x) W2b[(i / NH) * W2LD + i % NH] = __float2bfloat16_rn(s.W2[i]);
  __syncthreads();
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int g = lane >> 2, t4 = lane & 3;   // fragment row group, column pair
  const int64_t ntiles = (rows + 15) / 16;
  for (int64_t tile = (int64_t)blockIdx.x * MMA_WARPS + warp; tile < ntiles; tile += (int64_t)gridDim.x * MMA_WARPS) {
    const int64_t r0 = tile * 16 + g, r1 = r0 + 8;
    float x0[NIN], x1[NIN];
#pragma unroll
    for (int i = 0; i < NIN; ++i) {
      x0[i] = r0 < rows ? (feat[r0 * NIN + i] - s.shift[i]) * s.iscale[i] : 0.f;
      x1[i] = r1 < rows ? (feat[r1 * NIN + i] - s.shift[i]) * s.iscale[i] : 0.f;
    }
    // A fragments of layer 2's input h1 (rows r0, r1 x 64 hidden units), three planes
    uint32_t A[3][4][4];
#pragma unroll
    for (int kc = 0; kc < 4; ++kc) {
#pragma unroll
      for (int hh = 0; hh < 2; ++hh) {            // columns 2 t4 (+1) and 2 t4 + 8 (+1)
        __nv_bfloat16 q00[3], q01[3], q10[3], q11[3];
        const int h = kc * 16 + 2 * t4 + 8 * hh;
        float a00 = s.b1[h], a01 = s.b1[h + 1], a10 = s.b1[h], a11 = s.b1[h + 1];
#pragma unroll
        for (int i = 0; i < NIN; ++i) {
          a00 = fmaf(s.W1[h * NIN + i], x0[i], a00);
          a01 = fmaf(s.W1[(h + 1) * NIN + i], x0[i], a01);
          a10 = fmaf(s.W1[h * NIN + i], x1[i], a10);
          a11 = fmaf(s.W1[(h + 1) * NIN + i], x1[i], a11);
        }
        split3_f32(a00 > 0.f ? a00 : 0.f, q00);
        split3_f32(a01 > 0.f ? a01 : 0.f, q01);
        split3_f32(a10 > 0.f ? a10 : 0.f, q10);
        split3_f32(a11 > 0.f ? a11 : 0.f, q11);
#pragma unroll
        for (int pl = 0; pl < 3; ++pl) {
          A[pl][kc][2 * hh] = pack_bf16(q00[pl], q01[pl]);       // row g
          A[pl][kc][2 * hh + 1] = pack_bf16(q10[pl], q11[pl]);   // row g + 8
        }
      }
    }
    float y0 = 0.f, y1 = 0.f;
#pragma unroll
    for (int nt = 0; nt < NH / 8; ++nt) {
      float d[4] = {0.f, 0.f, 0.f, 0.f};
      const __nv_bfloat16* wrow = W2b + (nt * 8 + g) * W2LD;   // output unit nt*8+g, k contiguous
#pragma unroll
      for (int kc = 0; kc < 4; ++kc) {
        const uint32_t b0 = *reinterpret_cast<const uint32_t*>(wrow + kc * 16 + 2 * t4);
        const uint32_t b1 = *reinterpret_cast<const uint32_t*>(wrow + kc * 16 + 2 * t4 + 8);
#pragma unroll
        for (int pl = 2; pl >= 0; --pl) mma_bf16_16816(d, A[pl][kc], b0, b1);   // small planes first
      }
      // d: (row g, cols o, o+1), (row g + 8, cols o, o+1), o = nt*8 + 2 t4
      const int o = nt * 8 + 2 * t4;
      const float h00 = d[0] + s.b2[o], h01 = d[1] + s.b2[o + 1];
      const float h10 = d[2] + s.b2[o], h11 = d[3] + s.b2[o + 1];
      if (h00 > 0.f) y0 = fmaf(s.w3[o], h00, y0);
      if (h01 > 0.f) y0 = fmaf(s.w3[o + 1], h01, y0);
      if (h10 > 0.f) y1 = fmaf(s.w3[o], h10, y1);
      if (h11 > 0.f) y1 = fmaf(s.w3[o + 1], h11, y1);
    }
    // the four lanes of a row group hold disjoint output units: sum them
    y0 += __shfl_xor_sync(0xffffffffu, y0, 1);
    y0 += __shfl_xor_sync(0xffffffffu, y0, 2);
    y1 += __shfl_xor_sync(0xffffffffu, y1, 1);
    y1 += __shfl_xor_sync(0xffffffffu, y1, 2);
    if (t4 == 0) {
      if (r0 < rows) {
        const float y = s.b3 + y0;
        out[r0] = base ? (feat[r0 * NIN + 2] < -0.5f ? 0.f : base[r0] + y) : y;
      }
      if (r1 < rows) {
        const float y = s.b3 + y1;
        out[r1] = base ? (feat[r1 * NIN + 2] < -0.5f ? 0.f : base[r1] + y) : y;
      }
    }
  }
}

__global__ void __launch_bounds__(FWD_THREADS) mlp_forward_kernel(const float* theta, int bf16, const float* feat,
                                                                 const float* base, int64_t rows, float* out) {
  __shared__ SW s;
  load_weights(s, theta, bf16);
  __syncthreads();
  // one row per thread (no row loop: the compiler would hoist the weights out
  // of it into registers)
  const int64_t r = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (r < rows) {
    float xs[NIN], h1[NH];
#pragma unroll
    for (int i = 0; i < NIN; ++i) xs[i] = (feat[r * NIN + i] - s.shift[i]) * s.iscale[i];
    layer1(s, xs, h1);
    float y = s.b3;
#pragma unroll 1
    for (int o = 0; o < NH; ++o) {
      const float a = s.b2[o] + dot64(&s.W2[o * NH], h1);
      if (a > 0.f) y = fmaf(s.w3[o], a, y);
    }
    // a start: zero on the child's J0 (fix feature -1), base + f elsewhere
    out[r] = base ? (feat[r * NIN + 2] < -0.5f ? 0.f : base[r] + y) : y;
  }
}

// per-CTA partial gradient: part[blockIdx.x][0 .. NTRAIN) and the partial mean
// of squared residuals at part[blockIdx.x][NTRAIN].  16 x 16 threads; the three
// products of a tile (layer 2, its transpose in the backward sweep, the W2
// gradient) are register-tiled: a thread holds RPT rows x 4 units, or 4 x 4
// weights, and reads its operands as float4 (one shared-memory read per eight
// to ten FMAs; a thread per row, with a read per FMA and four warps per SM, was
// bound by those reads).  16384 rows, gradient and Adam step: 56.5 -> 34.3 us
// (the partials' sum, one thread per entry before, included).
template <int TILE>
struct GradSm {
  SW s;
  alignas(16) float W2T[NH * W2P];        // [h][o]
  alignas(16) float W2R[NH * W2P];        // [o][h]
  alignas(16) float H1[TILE * W2P];       // [row][h]
  alignas(16) float DA2[TILE * W2P];      // [row][o] dL/da2
  float XS[TILE * 8];         // [row] standardised inputs
  float comb[16][NH * (NIN + 3)];
};

template <int TILE>
__global__ void __launch_bounds__(GRAD_T) mlp_grad_kernel(const float* theta, int bf16, const float* feat,
                                                         const float* base, const float* target, int64_t rows,
                                                         float* part) {
  constexpr int RPT = TILE / 16;   // rows per thread
  extern __shared__ __align__(16) unsigned char grad_raw[];
  GradSm<TILE>& m = *reinterpret_cast<GradSm<TILE>*>(grad_raw);
  const int t = threadIdx.x, tr = t >> 4, tc = t & 15;
  load_weights(m.s, theta, bf16);
  __syncthreads();
  for (int i = t; i < NH * NH; i += GRAD_T) {
    const int o = i / NH, h = i % NH;
    const float w = m.s.W2[i];
    m.W2R[o * W2P + h] = w;
    m.W2T[h * W2P + o] = w;
  }
  const float inv_n = 1.0f / (float)rows;
  // accumulators: W2 entries (o = 4 tr + i, h = 4 tc + j); units 4 tc + j over
  // this thread's rows: b2, w3, b1, W1
  float gW2[4][4] = {}, gb2[4] = {}, gw3[4] = {}, gb1[4] = {}, gW1[4][NIN] = {};
  float gb3 = 0.f;
  double sq = 0.0;
  const int64_t ntiles = (rows + TILE - 1) / TILE;
  for (int64_t tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
    const int64_t r0 = tile * TILE;
    __syncthreads();   // the last tile's operands are read; the weights are in place
    for (int i = t; i < TILE * NIN; i += GRAD_T) {
      const int r = i / NIN, c = i % NIN;
      m.XS[r * 8 + c] = r0 + r < rows ? (feat[r0 * NIN + i] - m.s.shift[c]) * m.s.iscale[c] : 0.f;
    }
    __syncthreads();
    // ---- layer 1
    for (int i = t; i < TILE * NH; i += GRAD_T) {
      const int r = i / NH, h = i % NH;
      float a = m.s.b1[h];
#pragma unroll
      for (int c = 0; c < NIN; ++c) a = fmaf(m.s.W1[h * NIN + c], m.XS[r * 8 + c], a);
      m.H1[r * W2P + h] = a > 0.f ? a : 0.f;
    }
    __syncthreads();
    // ---- layer 2, output, residual: rows tr RPT + i, units 4 tc + j
    float acc[RPT][4];
    {
      const float4 b = *reinterpret_cast<const float4*>(&m.s.b2[4 * tc]);
#pragma unroll
      for (int i = 0; i < RPT; ++i) { acc[i][0] = b.x; acc[i][1] = b.y; acc[i][2] = b.z; acc[i][3] = b.w; }
    }
#pragma unroll 2
    for (int k = 0; k < NH; k += 4) {
      float4 w[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) w[u] = *reinterpret_cast<const float4*>(&m.W2T[(k + u) * W2P + 4 * tc]);
#pragma unroll
      for (int i = 0; i < RPT; ++i) {
        const float4 h = *reinterpret_cast<const float4*>(&m.H1[(tr * RPT + i) * W2P + k]);
        const float hv[4] = {h.x, h.y, h.z, h.w};
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          acc[i][0] = fmaf(w[u].x, hv[u], acc[i][0]);
          acc[i][1] = fmaf(w[u].y, hv[u], acc[i][1]);
          acc[i][2] = fmaf(w[u].z, hv[u], acc[i][2]);
          acc[i][3] = fmaf(w[u].w, hv[u], acc[i][3]);
        }
      }
    }
    const float4 w3 = *reinterpret_cast<const float4*>(&m.s.w3[4 * tc]);
    const float w3v[4] = {w3.x, w3.y, w3.z, w3.w};
#pragma unroll
    for (int i = 0; i < RPT; ++i) {
      const int r = tr * RPT + i;
      const int64_t row = r0 + r;
      float y = 0.f;
#pragma unroll
      for (int j = 0; j < 4; ++j)
        if (acc[i][j] > 0.f) y = fmaf(w3v[j], acc[i][j], y);
#pragma unroll
      for (int o = 8; o > 0; o >>= 1) y += __shfl_xor_sync(0xffffffffu, y, o);
      float d = 0.f;
      if (row < rows) {
        const float res = base[row] + (m.s.b3 + y) - target[row];
        d = 2.0f * res * inv_n;
        if (tc == 0) {
          sq += (double)res * (double)res;
          gb3 += d;
        }
      }
      float4 da;
      float* dv = &da.x;
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const float h2 = acc[i][j] > 0.f ? acc[i][j] : 0.f;
        dv[j] = h2 > 0.f ? d * w3v[j] : 0.f;
        gb2[j] += dv[j];
        gw3[j] = fmaf(d, h2, gw3[j]);
      }
      *reinterpret_cast<float4*>(&m.DA2[r * W2P + 4 * tc]) = da;
    }
    __syncthreads();
    // ---- backward through layer 2: dL/dh1 = W2' dL/da2, rows tr RPT + i, units 4 tc + j
#pragma unroll
    for (int i = 0; i < RPT; ++i) acc[i][0] = acc[i][1] = acc[i][2] = acc[i][3] = 0.f;
#pragma unroll 2
    for (int k = 0; k < NH; k += 4) {
      float4 w[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) w[u] = *reinterpret_cast<const float4*>(&m.W2R[(k + u) * W2P + 4 * tc]);
#pragma unroll
      for (int i = 0; i < RPT; ++i) {
        const float4 d = *reinterpret_cast<const float4*>(&m.DA2[(tr * RPT + i) * W2P + k]);
        const float dv[4] = {d.x, d.y, d.z, d.w};
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          acc[i][0] = fmaf(w[u].x, dv[u], acc[i][0]);
          acc[i][1] = fmaf(w[u].y, dv[u], acc[i][1]);
          acc[i][2] = fmaf(w[u].z, dv[u], acc[i][2]);
          acc[i][3] = fmaf(w[u].w, dv[u], acc[i][3]);
        }
      }
    }
#pragma unroll
    for (int i = 0; i < RPT; ++i) {
      const int r = tr * RPT + i;
      const float4 h = *reinterpret_cast<const float4*>(&m.H1[r * W2P + 4 * tc]);
      const float hv[4] = {h.x, h.y, h.z, h.w};
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const float da1 = hv[j] > 0.f ? acc[i][j] : 0.f;
        gb1[j] += da1;
#pragma unroll
        for (int c = 0; c < NIN; ++c) gW1[j][c] = fmaf(da1, m.XS[r * 8 + c], gW1[j][c]);
      }
    }
    // ---- the W2 gradient over the tile's rows, in row order
#pragma unroll 4
    for (int r = 0; r < TILE; ++r) {
      const float4 d = *reinterpret_cast<const float4*>(&m.DA2[r * W2P + 4 * tr]);
      const float4 h = *reinterpret_cast<const float4*>(&m.H1[r * W2P + 4 * tc]);
      const float dv[4] = {d.x, d.y, d.z, d.w}, hv[4] = {h.x, h.y, h.z, h.w};
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) gW2[i][j] = fmaf(dv[i], hv[j], gW2[i][j]);
    }
  }
  float* P = part + (size_t)blockIdx.x * (RELAX_MLP_NTRAIN + 1);
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) P[O_W2 + (4 * tr + i) * NH + 4 * tc + j] = gW2[i][j];
  // the sums over the 16 row groups, in order
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    float* c = &m.comb[tr][(4 * tc + j) * (NIN + 3)];
    c[0] = gb2[j];
    c[1] = gw3[j];
    c[2] = gb1[j];
#pragma unroll
    for (int i = 0; i < NIN; ++i) c[3 + i] = gW1[j][i];
  }
  __shared__ double sqs[16];
  __shared__ float b3s[16];
  if (tc == 0) {
    sqs[tr] = sq;
    b3s[tr] = gb3;
  }
  __syncthreads();
  for (int i = t; i < NH * (NIN + 3); i += GRAD_T) {
    float v = 0.f;
#pragma unroll
    for (int g = 0; g < 16; ++g) v += m.comb[g][i];
    const int u = i / (NIN + 3), f = i % (NIN + 3);
    P[f == 0 ? O_B2 + u : f == 1 ? O_W3 + u : f == 2 ? O_B1 + u : O_W1 + u * NIN + (f - 3)] = v;
  }
  if (t == 0) {
    double v = 0.0;
    float b = 0.f;
    for (int g = 0; g < 16; ++g) {
      v += sqs[g];
      b += b3s[g];
    }
    P[RELAX_MLP_NTRAIN] = (float)(v / (double)rows);
    P[O_B3] = b;
  }
}

// grad[i] = sum over CTAs of part[c][i], loss = sum of the partial means: 32
// entries per CTA, warp w taking the CTAs w, w + 8, ... in order and the warps
// summed in order (a thread per entry walked all the partials alone)
__global__ void __launch_bounds__(256) mlp_reduce_kernel(const float* part, int nparts, float* grad, float* loss) {
  __shared__ float sh[8][32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int i = blockIdx.x * 32 + lane;
  float a = 0.f;
  if (i <= RELAX_MLP_NTRAIN) {
#pragma unroll 8
    for (int c = warp; c < nparts; c += 8) a += part[(size_t)c * (RELAX_MLP_NTRAIN + 1) + i];
  }
  sh[warp][lane] = a;
  __syncthreads();
  if (warp != 0) return;
  float v = 0.f;
#pragma unroll
  for (int w = 0; w < 8; ++w) v += sh[w][lane];
  if (i < RELAX_MLP_NTRAIN) grad[i] = v;
  else if (i == RELAX_MLP_NTRAIN && loss) *loss = v;
  if (i >= RELAX_MLP_NTRAIN && i < RELAX_MLP_NPARAM) grad[i] = 0.f;   // shift and scale are not trained
}

// b1, b2 and their complements come separately: 1 - b in FP32 from an FP32 b
// near 1 would carry b's rounding error magnified (0.999f: 1.3e-5 relative)
__global__ void mlp_adam_kernel(float* theta, const float* grad, float* m, float* v, float lr, float b1, float omb1,
                                float b2, float omb2, float eps, float c1, float c2) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= RELAX_MLP_NTRAIN) return;
  const float g = grad[i];
  const float mi = b1 * m[i] + omb1 * g;
  const float vi = b2 * v[i] + omb2 * g * g;
  m[i] = mi;
  v[i] = vi;
  theta[i] -= lr * (mi / c1) / (sqrtf(vi / c2) + eps);
}

int sm_count() {
  int dev = 0, n = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev);
  return n > 0 ? n : 1;
}

relax_status cuda_status(cudaError_t e) {
  if (e == cudaSuccess) return RELAX_OK;
  return e == cudaErrorMemoryAllocation ? RELAX_ENOMEM : RELAX_ECUDA;
}

}  // namespace

extern "C" {

relax_status relax_mlp_forward(const float* theta, int32_t bf16, const float* feat, const float* base, int64_t rows,
                               float* out, void* stream) {
  if (!theta || !feat || !out || rows < 0) return RELAX_EINVAL;
  if (rows == 0) return RELAX_OK;
  if (bf16) {   // BF16 weights: the tensor-core forward, grid-stride over 16-row tiles
    const int64_t tiles = (rows + 15) / 16;
    const int64_t want = (tiles + MMA_WARPS - 1) / MMA_WARPS;
    const unsigned grid = (unsigned)(want < 8 * sm_count() ? want : 8 * sm_count());
    mlp_forward_mma_kernel<<<grid, 32 * MMA_WARPS, 0, (cudaStream_t)stream>>>(theta, feat, base, rows, out);
    return cuda_status(cudaGetLastError());
  }
  const int64_t grid = (rows + FWD_THREADS - 1) / FWD_THREADS;
  if (grid > INT32_MAX) return RELAX_ENOTSUP;
  mlp_forward_kernel<<<(unsigned)grid, FWD_THREADS, 0, (cudaStream_t)stream>>>(theta, 0, feat, base, rows, out);
  return cuda_status(cudaGetLastError());
}

relax_status relax_mlp_grad(const float* theta, int32_t bf16, const float* feat, const float* base,
                            const float* target, int64_t rows, float* grad, float* loss, void* stream) {
  if (!theta || !feat || !base || !target || !grad || rows <= 0) return RELAX_EINVAL;
  cudaStream_t st = (cudaStream_t)stream;
  // tiles of 128 rows, of 64 where those would leave half of the SMs idle
  const int sms = sm_count();
  const int tile = rows * 2 < (int64_t)128 * sms ? 64 : 128;
  const auto kernel = tile == 128 ? mlp_grad_kernel<128> : mlp_grad_kernel<64>;
  const size_t smem = tile == 128 ? sizeof(GradSm<128>) : sizeof(GradSm<64>);
  // per device (the current one): cheap, so set on every call
  cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return cuda_status(e);
  const int64_t ntiles = (rows + tile - 1) / tile;
  const int nparts = (int)(ntiles < sms ? ntiles : sms);
  float* part = nullptr;
  e = relax::pool_alloc((void**)&part, (size_t)nparts * (RELAX_MLP_NTRAIN + 1) * sizeof(float), st);
  if (e != cudaSuccess) return cuda_status(e);
  kernel<<<nparts, GRAD_T, smem, st>>>(theta, bf16 ? 1 : 0, feat, base, target, rows, part);
  e = cudaGetLastError();
  if (e == cudaSuccess) {
    mlp_reduce_kernel<<<(RELAX_MLP_NPARAM + 31) / 32, 256, 0, st>>>(part, nparts, grad, loss);
    e = cudaGetLastError();
  }
  cudaFreeAsync(part, st);
  return cuda_status(e);
}

relax_status relax_mlp_adam(float* theta, const float* grad, float* m, float* v, int32_t t, double lr, double beta1,
                            double beta2, double eps, void* stream) {
  if (!theta || !grad || !m || !v || t < 1 || !(lr >= 0.0) || !(beta1 >= 0.0 && beta1 < 1.0) ||
      !(beta2 >= 0.0 && beta2 < 1.0) || !(eps >= 0.0))
    return RELAX_EINVAL;
  const double c1 = 1.0 - std::pow(beta1, (double)t), c2 = 1.0 - std::pow(beta2, (double)t);
  mlp_adam_kernel<<<(RELAX_MLP_NTRAIN + 255) / 256, 256, 0, (cudaStream_t)stream>>>(
      theta, grad, m, v, (float)lr, (float)beta1, (float)(1.0 - beta1), (float)beta2, (float)(1.0 - beta2), (float)eps,
      (float)c1, (float)c2);
  return cuda_status(cudaGetLastError());
}

}  // extern "C"
