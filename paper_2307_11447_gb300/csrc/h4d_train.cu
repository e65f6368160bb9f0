// h4d_train.cu -- training of the learned insertion-site proposal on the GPU: minibatch
// gather from the trial records, BF16 forward and backward through the 96-64-64-2 network
// on mma.sync tiles (FP32 accumulation), weight-gradient GEMMs over the batch, Adam.
//
// Loss of a batch of n records (each a cation row and an anion row):
//   L = (1/n) sum_records [BCE(logit_cation(f_c), t) + BCE(logit_anion(f_a), t)]
// with the soft target t = min(1, exp(y - y0)) of the record's insertion-direction
// Metropolis exponent y.  Every reduction runs in a fixed order, so a step is
// bit-reproducible.
#include <cuda_runtime.h>

#include <cstdint>

#include "h4d_engine.cuh"
#include "h4d_philox.cuh"
#include "h4d_prop.cuh"

namespace h4d {

// ---- weight packing: FP32 masters -> bf16 B fragments --------------------------------
// item ranges: w1 [0,1536), w2 [1536,2560), w3 [2560,2688), w2t [2688,3712),
// w3r [3712,3840), b [3840,3970)
__global__ void prop_pack_kernel(const float* __restrict__ w, uint2* w1, uint2* w2, uint2* w3, uint2* w2t,
                                 float* w3r, float* b) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  const float* W1 = w;
  const float* W2 = w + kPropOffW2;
  const float* W3 = w + kPropOffW3;
  if (i < 1536) {  // W1: K = 96 (6 k-steps), N = 64 (8 n-tiles)
    const int lane = i & 31, nt = (i >> 5) & 7, ks = i >> 8, g = lane >> 2, t = lane & 3;
    const int n = 8 * nt + g, k = 16 * ks + 2 * t;
    w1[i] = make_uint2(pack_bf16(W1[k * 64 + n], W1[(k + 1) * 64 + n]),
                       pack_bf16(W1[(k + 8) * 64 + n], W1[(k + 9) * 64 + n]));
  } else if (i < 2560) {  // W2: K = 64, N = 64
    const int j = i - 1536, lane = j & 31, nt = (j >> 5) & 7, ks = j >> 8, g = lane >> 2, t = lane & 3;
    const int n = 8 * nt + g, k = 16 * ks + 2 * t;
    w2[j] = make_uint2(pack_bf16(W2[k * 64 + n], W2[(k + 1) * 64 + n]),
                       pack_bf16(W2[(k + 8) * 64 + n], W2[(k + 9) * 64 + n]));
  } else if (i < 2688) {  // W3: K = 64, N = 8 (columns 2..7 zero)
    const int j = i - 2560, lane = j & 31, ks = j >> 5, g = lane >> 2, t = lane & 3;
    const int k = 16 * ks + 2 * t;
    float v0 = 0.f, v1 = 0.f, v2 = 0.f, v3 = 0.f;
    if (g < 2) {
      v0 = W3[k * 2 + g]; v1 = W3[(k + 1) * 2 + g]; v2 = W3[(k + 8) * 2 + g]; v3 = W3[(k + 9) * 2 + g];
    }
    w3[j] = make_uint2(pack_bf16(v0, v1), pack_bf16(v2, v3));
  } else if (i < 3712) {  // W2^T: B[k][n] = W2[n][k]
    const int j = i - 2688, lane = j & 31, nt = (j >> 5) & 7, ks = j >> 8, g = lane >> 2, t = lane & 3;
    const int n = 8 * nt + g, k = 16 * ks + 2 * t;
    w2t[j] = make_uint2(pack_bf16(W2[n * 64 + k], W2[n * 64 + k + 1]),
                        pack_bf16(W2[n * 64 + k + 8], W2[n * 64 + k + 9]));
  } else if (i < 3840) {
    const int j = i - 3712;
    w3r[j] = bf16_lo(pack_bf16(W3[j], 0.f));
  } else if (i < 3970) {
    const int j = i - 3840;
    b[j] = j < 64 ? w[kPropOffB1 + j] : (j < 128 ? w[kPropOffB2 + j - 64] : w[kPropOffB3 + j - 128]);
  }
}

int launch_prop_pack(const float* w, uint2* w1, uint2* w2, uint2* w3, uint2* w2t, float* w3r, float* b,
                     void* stream) {
  prop_pack_kernel<<<(3970 + 255) / 256, 256, 0, (cudaStream_t)stream>>>(w, w1, w2, w3, w2t, w3r, b);
  return cudaGetLastError() == cudaSuccess ? H4D_OK : H4D_ECUDA;
}

// ---- loss and gradient -------------------------------------------------------------------
// Row r is record r/2, species r%2 (0 = cation row, 1 = anion row); feat is [rows][96],
// tgt [rows].  A CTA takes blocks of 128 rows: forward and backward of 16-row tiles, one per
// warp, with the activations and their gradients kept in shared memory as bf16, transposed
// (the batch row is the K index of the weight-gradient products), and then the CTA's part of
// dW = A^T B over those rows, 84 output tiles of 16 x 8 spread over the warps, accumulated in
// registers from block to block.  Each CTA writes one partial gradient; a second kernel adds
// the partials in CTA order, so a step is bit-reproducible.
// A training step moves 3 MB and does 0.5 GFLOP: it is bound by latency, hence one pass over
// the batch and sums split over CTAs.  With the activations written to global memory and one
// warp per output tile (one lane per bias and for the loss) walking all rows, loss and gradient
// of 4096 records took 0.9 ms; now a training step takes 52 us instead of 917.
constexpr int kBlockRows = 128, kLd = kBlockRows + 8;  // + 8: conflict-free fragment loads
constexpr int kGradTiles = 84;  // dW1 6 x 8, dW2 4 x 8, dW3 4 x 1
struct GradSmem {
  uint16_t xT[96 * kLd], h1T[64 * kLd], dz1T[64 * kLd], h2T[64 * kLd], dz2T[64 * kLd], dlT[8 * kLd];
  float loss[kBlockRows];
};

__device__ __forceinline__ void st_bf16(uint16_t* p, float v) { *p = (uint16_t)(pack_bf16(v, 0.f) & 0xffffu); }

// store the bf16 pairs of an A fragment (rows q0, q1; columns c, c+1) transposed
__device__ __forceinline__ void st_pairT(uint16_t* T, int c, int q0, int q1, unsigned lo, unsigned hi) {
  T[c * kLd + q0] = (uint16_t)(lo & 0xffffu);
  T[(c + 1) * kLd + q0] = (uint16_t)(lo >> 16);
  T[c * kLd + q1] = (uint16_t)(hi & 0xffffu);
  T[(c + 1) * kLd + q1] = (uint16_t)(hi >> 16);
}
__device__ __forceinline__ unsigned ld_pair(const uint16_t* base, int row, int k) {
  return *reinterpret_cast<const unsigned*>(base + row * kLd + k);
}

__global__ void __launch_bounds__(256) prop_grad_kernel(PropNet net, const float* __restrict__ feat,
                                                        const float* __restrict__ tgt, int rows, float inv_n,
                                                        int n_blocks, int blocks_per_cta, float* __restrict__ part,
                                                        double* __restrict__ part_loss) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  GradSmem& S = *reinterpret_cast<GradSmem*>(smem_raw);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, g = lane >> 2, t = lane & 3;
  const int q0 = 16 * warp + g, q1 = q0 + 8;  // this lane's rows of the block
  float dw[11][4];
#pragma unroll
  for (int i = 0; i < 11; ++i) dw[i][0] = dw[i][1] = dw[i][2] = dw[i][3] = 0.f;
  float db = 0.f;       // threads 0..129: one bias each
  double loss = 0.0;    // warp 7
  for (int k = threadIdx.x; k < 6 * kLd; k += 256) S.dlT[2 * kLd + k] = 0;  // rows 2..7 of dl
  const int b0 = blockIdx.x * blocks_per_cta, b1 = min(n_blocks, b0 + blocks_per_cta);
  for (int blk = b0; blk < b1; ++blk) {
    const int r0 = kBlockRows * blk + q0, r1 = r0 + 8;
    const bool v0 = r0 < rows, v1 = r1 < rows;
    // ---- layer 1 ----
    float acc1[8][4];
#pragma unroll
    for (int i = 0; i < 8; ++i) acc1[i][0] = acc1[i][1] = acc1[i][2] = acc1[i][3] = 0.f;
#pragma unroll
    for (int ks = 0; ks < 6; ++ks) {
      const int k = 16 * ks + 2 * t;
      const float2 z2 = make_float2(0.f, 0.f);
      const float2 f00 = v0 ? *reinterpret_cast<const float2*>(feat + (size_t)r0 * 96 + k) : z2;
      const float2 f10 = v1 ? *reinterpret_cast<const float2*>(feat + (size_t)r1 * 96 + k) : z2;
      const float2 f01 = v0 ? *reinterpret_cast<const float2*>(feat + (size_t)r0 * 96 + k + 8) : z2;
      const float2 f11 = v1 ? *reinterpret_cast<const float2*>(feat + (size_t)r1 * 96 + k + 8) : z2;
      unsigned a[4] = {pack_bf16(f00.x, f00.y), pack_bf16(f10.x, f10.y), pack_bf16(f01.x, f01.y),
                       pack_bf16(f11.x, f11.y)};
      st_pairT(S.xT, k, q0, q1, a[0], a[1]);
      st_pairT(S.xT, k + 8, q0, q1, a[2], a[3]);
#pragma unroll
      for (int nt = 0; nt < 8; ++nt) mma_bf16(acc1[nt], a, net.w1[(ks * 8 + nt) * 32 + lane]);
    }
    unsigned mask1 = 0;  // bit 4*nt + e: pre-activation > 0
#pragma unroll
    for (int nt = 0; nt < 8; ++nt) {
      const float b0 = net.b[8 * nt + 2 * t], b1 = net.b[8 * nt + 2 * t + 1];
      acc1[nt][0] += b0; acc1[nt][1] += b1; acc1[nt][2] += b0; acc1[nt][3] += b1;
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        if (acc1[nt][e] > 0.f) mask1 |= 1u << (4 * nt + e);
        else acc1[nt][e] = 0.f;
      }
    }
    unsigned a2[4][4];
#pragma unroll
    for (int ks = 0; ks < 4; ++ks) c_to_a(acc1[2 * ks], acc1[2 * ks + 1], a2[ks]);
#pragma unroll
    for (int nt = 0; nt < 8; ++nt)
      st_pairT(S.h1T, 8 * nt + 2 * t, q0, q1, a2[nt >> 1][(nt & 1) * 2], a2[nt >> 1][(nt & 1) * 2 + 1]);
    // ---- layer 2 ----
    float acc2[8][4];
#pragma unroll
    for (int i = 0; i < 8; ++i) acc2[i][0] = acc2[i][1] = acc2[i][2] = acc2[i][3] = 0.f;
#pragma unroll
    for (int ks = 0; ks < 4; ++ks)
#pragma unroll
      for (int nt = 0; nt < 8; ++nt) mma_bf16(acc2[nt], a2[ks], net.w2[(ks * 8 + nt) * 32 + lane]);
    unsigned mask2 = 0;
#pragma unroll
    for (int nt = 0; nt < 8; ++nt) {
      const float b0 = net.b[64 + 8 * nt + 2 * t], b1 = net.b[64 + 8 * nt + 2 * t + 1];
      acc2[nt][0] += b0; acc2[nt][1] += b1; acc2[nt][2] += b0; acc2[nt][3] += b1;
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        if (acc2[nt][e] > 0.f) mask2 |= 1u << (4 * nt + e);
        else acc2[nt][e] = 0.f;
      }
    }
    unsigned a3[4][4];
#pragma unroll
    for (int ks = 0; ks < 4; ++ks) c_to_a(acc2[2 * ks], acc2[2 * ks + 1], a3[ks]);
#pragma unroll
    for (int nt = 0; nt < 8; ++nt)
      st_pairT(S.h2T, 8 * nt + 2 * t, q0, q1, a3[nt >> 1][(nt & 1) * 2], a3[nt >> 1][(nt & 1) * 2 + 1]);
    // ---- layer 3, loss and dL/dlogit ----
    float lg[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
    for (int ks = 0; ks < 4; ++ks) mma_bf16(lg, a3[ks], net.w3[ks * 32 + lane]);
    const int s = r0 & 1;  // rows g and g+8 have the same species
    float dl0 = 0.f, dl1 = 0.f;
    if (t == 0) {
      const float b3 = net.b[128 + s];
      const float l0 = (s ? lg[1] : lg[0]) + b3, l1 = (s ? lg[3] : lg[2]) + b3;
      const float t0 = v0 ? tgt[r0] : 0.f, t1 = v1 ? tgt[r1] : 0.f;
      dl0 = v0 ? (1.f / (1.f + expf(-l0)) - t0) * inv_n : 0.f;
      dl1 = v1 ? (1.f / (1.f + expf(-l1)) - t1) * inv_n : 0.f;
      S.loss[q0] = v0 ? fmaxf(l0, 0.f) - l0 * t0 + log1pf(expf(-fabsf(l0))) : 0.f;
      S.loss[q1] = v1 ? fmaxf(l1, 0.f) - l1 * t1 + log1pf(expf(-fabsf(l1))) : 0.f;
      st_bf16(S.dlT + s * kLd + q0, dl0);
      st_bf16(S.dlT + s * kLd + q1, dl1);
      st_bf16(S.dlT + (1 - s) * kLd + q0, 0.f);
      st_bf16(S.dlT + (1 - s) * kLd + q1, 0.f);
    }
    dl0 = __shfl_sync(0xffffffffu, dl0, lane & ~3);
    dl1 = __shfl_sync(0xffffffffu, dl1, lane & ~3);
    // the backward pass uses dL/dlogit rounded to bf16, as the weight-gradient GEMM does
    dl0 = bf16_lo(pack_bf16(dl0, 0.f));
    dl1 = bf16_lo(pack_bf16(dl1, 0.f));
    // ---- dz2 = (dl W3^T) * [z2 > 0] ----
    float dz2[8][4];
#pragma unroll
    for (int nt = 0; nt < 8; ++nt) {
      const int c = 8 * nt + 2 * t;
      const float w0 = net.w3r[c * 2 + s], w1 = net.w3r[(c + 1) * 2 + s];
      dz2[nt][0] = (mask2 >> (4 * nt + 0) & 1) ? dl0 * w0 : 0.f;
      dz2[nt][1] = (mask2 >> (4 * nt + 1) & 1) ? dl0 * w1 : 0.f;
      dz2[nt][2] = (mask2 >> (4 * nt + 2) & 1) ? dl1 * w0 : 0.f;
      dz2[nt][3] = (mask2 >> (4 * nt + 3) & 1) ? dl1 * w1 : 0.f;
    }
    unsigned ad[4][4];
#pragma unroll
    for (int ks = 0; ks < 4; ++ks) c_to_a(dz2[2 * ks], dz2[2 * ks + 1], ad[ks]);
#pragma unroll
    for (int nt = 0; nt < 8; ++nt)
      st_pairT(S.dz2T, 8 * nt + 2 * t, q0, q1, ad[nt >> 1][(nt & 1) * 2], ad[nt >> 1][(nt & 1) * 2 + 1]);
    // ---- dz1 = (dz2 W2^T) * [z1 > 0] ----
    float acc[8][4];
#pragma unroll
    for (int i = 0; i < 8; ++i) acc[i][0] = acc[i][1] = acc[i][2] = acc[i][3] = 0.f;
#pragma unroll
    for (int ks = 0; ks < 4; ++ks)
#pragma unroll
      for (int nt = 0; nt < 8; ++nt) mma_bf16(acc[nt], ad[ks], net.w2t[(ks * 8 + nt) * 32 + lane]);
#pragma unroll
    for (int nt = 0; nt < 8; ++nt)
#pragma unroll
      for (int e = 0; e < 4; ++e)
        if (!(mask1 >> (4 * nt + e) & 1)) acc[nt][e] = 0.f;
#pragma unroll
    for (int nt = 0; nt < 8; ++nt)
      st_pairT(S.dz1T, 8 * nt + 2 * t, q0, q1, pack_bf16(acc[nt][0], acc[nt][1]),
               pack_bf16(acc[nt][2], acc[nt][3]));
    __syncthreads();
    // ---- weight gradients over the block's rows ----
#pragma unroll
    for (int i = 0; i < 11; ++i) {
      const int task = warp + 8 * i;
      if (task < kGradTiles) {
        const uint16_t* A = task < 48 ? S.xT : (task < 80 ? S.h1T : S.h2T);
        const uint16_t* B = task < 48 ? S.dz1T : (task < 80 ? S.dz2T : S.dlT);
        const int mt = task < 48 ? task >> 3 : (task < 80 ? (task - 48) >> 3 : task - 80);
        const int nt = task < 80 ? task & 7 : 0;
        const int ra = 16 * mt + g, rb = 8 * nt + g;
#pragma unroll
        for (int k0 = 0; k0 < kBlockRows; k0 += 16) {
          const int k = k0 + 2 * t;
          const unsigned a[4] = {ld_pair(A, ra, k), ld_pair(A, ra + 8, k), ld_pair(A, ra, k + 8), ld_pair(A, ra + 8, k + 8)};
          mma_bf16(dw[i], a, make_uint2(ld_pair(B, rb, k), ld_pair(B, rb, k + 8)));
        }
      }
    }
    if (threadIdx.x < 130) {
      const int j = threadIdx.x;
      const uint16_t* D = j < 64 ? S.dz1T + j * kLd : (j < 128 ? S.dz2T + (j - 64) * kLd : S.dlT + (j - 128) * kLd);
      float s0 = 0.f, s1 = 0.f;
      for (int k = 0; k < kBlockRows; k += 2) {
        const unsigned d = *reinterpret_cast<const unsigned*>(D + k);
        s0 += bf16_lo(d);
        s1 += bf16_hi(d);
      }
      db += s0 + s1;
    } else if (warp == 7) {
      double s = 0.0;
      for (int k = lane; k < kBlockRows; k += 32) s += (double)S.loss[k];
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
      loss += s;
    }
    __syncthreads();
  }
  float* out = part + (size_t)blockIdx.x * kPropNW;
#pragma unroll
  for (int i = 0; i < 11; ++i) {
    const int task = warp + 8 * i;
    if (task < kGradTiles) {
      const int off = task < 48 ? 0 : (task < 80 ? kPropOffW2 : kPropOffW3);
      const int mt = task < 48 ? task >> 3 : (task < 80 ? (task - 48) >> 3 : task - 80);
      const int ld = task < 80 ? 64 : 2, c = task < 80 ? 8 * (task & 7) + 2 * t : 2 * t;
      if (c < ld) {
        out[off + (16 * mt + g) * ld + c] = dw[i][0];
        out[off + (16 * mt + g) * ld + c + 1] = dw[i][1];
        out[off + (16 * mt + g + 8) * ld + c] = dw[i][2];
        out[off + (16 * mt + g + 8) * ld + c + 1] = dw[i][3];
      }
    }
  }
  if (threadIdx.x < 130)
    out[threadIdx.x < 64 ? kPropOffB1 + threadIdx.x
                         : (threadIdx.x < 128 ? kPropOffB2 + threadIdx.x - 64 : kPropOffB3 + threadIdx.x - 128)] = db;
  if (threadIdx.x == 224) part_loss[blockIdx.x] = loss;
}

__global__ void __launch_bounds__(128) prop_grad_reduce(const float* __restrict__ part, const double* __restrict__ part_loss,
                                                        int n_parts, float* __restrict__ grad, double* __restrict__ loss) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < kPropNW) {
    double s = 0.0;
    for (int p = 0; p < n_parts; ++p) s += (double)part[(size_t)p * kPropNW + i];
    grad[i] = (float)s;
  } else if (i == kPropNW) {
    double s = 0.0;
    for (int p = 0; p < n_parts; ++p) s += part_loss[p];
    *loss = s;
  }
}

// CTAs of a batch: one per 128 rows up to one per SM
int prop_grad_parts(int rows) {
  const int n_blocks = (rows + kBlockRows - 1) / kBlockRows;
  const int per_cta = (n_blocks + 151) / 152;
  return (n_blocks + per_cta - 1) / per_cta;
}

int launch_prop_grad(const PropNet& net, const float* feat, const float* tgt, int n_rec, float inv_n, float* part,
                     double* part_loss, float* grad, double* loss, void* stream) {
  cudaStream_t st = (cudaStream_t)stream;
  const int rows = 2 * n_rec, n_blocks = (rows + kBlockRows - 1) / kBlockRows;
  const int parts = prop_grad_parts(rows), per_cta = (n_blocks + 151) / 152;
  if (cudaFuncSetAttribute(prop_grad_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(GradSmem)) !=
      cudaSuccess)
    return H4D_ECUDA;
  prop_grad_kernel<<<parts, 256, sizeof(GradSmem), st>>>(net, feat, tgt, rows, inv_n, n_blocks, per_cta, part, part_loss);
  prop_grad_reduce<<<(kPropNW + 1 + 127) / 128, 128, 0, st>>>(part, part_loss, parts, grad, loss);
  return cudaGetLastError() == cudaSuccess ? H4D_OK : H4D_ECUDA;
}

// ---- Adam (Kingma and Ba, 2015) on the FP32 masters ---------------------------------------
__global__ void prop_adam_kernel(float* w, float* m, float* v, const float* __restrict__ grad, float c1, float c2,
                                 float lr) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= kPropNW) return;
  const float gi = grad[i];
  const float mi = 0.9f * m[i] + 0.1f * gi;
  const float vi = 0.999f * v[i] + 0.001f * gi * gi;
  m[i] = mi;
  v[i] = vi;
  w[i] -= lr * (mi * c1) / (sqrtf(vi * c2) + 1e-8f);
}

int launch_prop_adam(float* w, float* m, float* v, const float* grad, int step, float lr, void* stream) {
  const float c1 = (float)(1.0 / (1.0 - pow(0.9, step)));
  const float c2 = (float)(1.0 / (1.0 - pow(0.999, step)));
  prop_adam_kernel<<<(kPropNW + 255) / 256, 256, 0, (cudaStream_t)stream>>>(w, m, v, grad, c1, c2, lr);
  return cudaGetLastError() == cudaSuccess ? H4D_OK : H4D_ECUDA;
}

// ---- valid records, in ring order: status 0 and a finite exponent -------------------------
__global__ void __launch_bounds__(1024) prop_compact_kernel(const int2* __restrict__ meta,
                                                           const double* __restrict__ y, int n_rec, int* valid,
                                                           int* n_valid) {
  __shared__ int warp_tot[32];
  __shared__ int base;
  if (threadIdx.x == 0) base = 0;
  __syncthreads();
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  for (int c0 = 0; c0 < n_rec; c0 += 1024) {
    const int i = c0 + threadIdx.x;
    const bool ok = i < n_rec && meta[i].y == 0 && isfinite(y[i]);
    const unsigned bal = __ballot_sync(0xffffffffu, ok);
    if (lane == 0) warp_tot[warp] = __popc(bal);
    __syncthreads();
    int off = base;
    for (int w = 0; w < warp; ++w) off += warp_tot[w];
    off += __popc(bal & ((1u << lane) - 1u));
    if (ok) valid[off] = i;
    __syncthreads();
    if (threadIdx.x == 0) {
      int s = 0;
      for (int w = 0; w < 32; ++w) s += warp_tot[w];
      base += s;
    }
    __syncthreads();
  }
  if (threadIdx.x == 0) *n_valid = base;
}

int launch_prop_compact(const int2* meta, const double* y, int n_rec, int* valid, int* n_valid, void* stream) {
  prop_compact_kernel<<<1, 1024, 0, (cudaStream_t)stream>>>(meta, y, n_rec, valid, n_valid);
  return cudaGetLastError() == cudaSuccess ? H4D_OK : H4D_ECUDA;
}

// ---- minibatch gather ---------------------------------------------------------------------
// Record b of the batch is valid[pick(draw)] with draw word b%4 of Philox counter
// {step, b/4, kPurTrain, 0} under key {seed, kTrainKey}; with n_batch >= n_valid the batch
// is every valid record in order.  feat [n][2][96], tgt [n][2] = min(1, exp(y - y0)).
__global__ void prop_gather_kernel(const float* __restrict__ rec_feat, const double* __restrict__ rec_y,
                                   const int* __restrict__ valid, int n_valid, int n_batch, u64 seed,
                                   long long step, float y0, float* feat, float* tgt) {
  const int b = blockIdx.x;
  if (b >= n_batch || n_valid <= 0) return;
  int idx;
  if (n_batch >= n_valid) {
    if (b >= n_valid) return;
    idx = valid[b];
  } else {
    u64 r[4];
    draw4(seed, kTrainKey, (u64)step, (u64)(b >> 2), kPurTrain, r);
    idx = valid[pick_index(r[b & 3], n_valid)];
  }
  for (int k = threadIdx.x; k < 192; k += blockDim.x) feat[(size_t)b * 192 + k] = rec_feat[(size_t)idx * 192 + k];
  if (threadIdx.x < 2) tgt[2 * b + threadIdx.x] = (float)exp(fmin(rec_y[idx] - (double)y0, 0.0));
}

int launch_prop_gather(const float* rec_feat, const double* rec_y, const int* valid, int n_valid, int n_batch,
                       unsigned long long seed, long long step, float y0, float* feat, float* tgt, void* stream) {
  if (n_batch <= 0) return H4D_OK;
  prop_gather_kernel<<<n_batch, 64, 0, (cudaStream_t)stream>>>(rec_feat, rec_y, valid, n_valid, n_batch, seed, step,
                                                               y0, feat, tgt);
  return cudaGetLastError() == cudaSuccess ? H4D_OK : H4D_ECUDA;
}

}  // namespace h4d
