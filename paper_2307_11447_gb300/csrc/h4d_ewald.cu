// h4d_ewald.cu -- long-range Coulomb term of Sec. II.B.2 (Eqs. 9-10): the reciprocal-space
// Ewald sum and the self energy of one configuration, scaled by the altitude screening
// g^lr(wbar) = exp(-kappa_lr wbar):
//   - structure factor: S(k) = sum_j q_j exp(i k.r_j) for every k of one half space;
//   - forces: F_j = g (8 pi K q_j / V) sum_half A_k k [Re S sin(k.r_j) - Im S cos(k.r_j)].
// The phase k.r_j / 2 pi = (n_x X_j + n_y Y_j + n_z Z_j) / 2^32 is formed in 32-bit integer
// arithmetic from the fixed-point coordinates X = round(x/L 2^32) (wrap-around is the
// periodicity).
//
// The k-vectors are taken as columns (n_x, n_y) of the half space times n_z = -kmax..kmax:
// exp(i k.r) = a b with a = exp(2 pi i (n_x X + n_y Y)) and b = exp(2 pi i n_z Z), so a term
// is a product of tabulated phases instead of a sine and a cosine, and n_z and -n_z share
// theirs.  Both passes are then small matrix products: the structure factors contract
// columns x n_z over the atoms, the forces contract columns x atoms over n_z.  Bound: the FP32
// pipe and, at about a quarter of the instructions, the sines and cosines of the tables.  A call for 9110
// atoms at kmax 14 with forces: 993 -> 156 us, of which the kernels take 78 us (one
// sincospif per term, the k-space weights on the host and a copy each way between the passes took
// 330 us of kernels); error of the forces against 64 bits 6.3e-6 -> 1.9e-6.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdint>
#include <cstring>
#include <new>
#include <vector>

#include "h4d_engine.cuh"

namespace {

constexpr int kColT = 32;      // columns of a structure-factor tile
constexpr int kMT = 16;        // n_z values of a tile (and of the force kernel's register table)
constexpr int kStage = 64;     // atoms staged in shared memory per step
constexpr int kSkWarps = 8;    // warps of a structure-factor block, each with its share of the atoms
constexpr int kTileVals = kColT * kMT * 4;  // partial sums of a tile
constexpr int kFStage = 16;    // columns staged per step of the force kernel
constexpr int kFThreads = 128;
constexpr int kSlots = 152 * 2;   // resident structure-factor blocks (registers: two per SM)
constexpr int kFSlots = 152 * 4;  // resident force blocks
constexpr size_t kPartBytes = (size_t)64 << 20;  // structure-factor partials of one batch of atoms
constexpr int kMaxK = 64;

struct KGeom {
  int kmax, ncol, nct, nmt;  // largest |n|, columns, column tiles, n_z tiles
  double k1sq;               // (2 pi / L)^2
  double e[kMaxK + 1];       // exp(-(2 pi m / L)^2 / (4 alpha^2)): A_k = e e e / k^2
};

// column c of the half space: n_x = 0 with n_y = 0..kmax, then n_x = 1..kmax with all n_y
// (of column 0 only n_z > 0 belongs to it)
__device__ __forceinline__ int2 column(int c, int kmax) {
  if (c <= kmax) return make_int2(0, c);
  const int k = c - (kmax + 1), w = 2 * kmax + 1;
  return make_int2(1 + k / w, k % w - kmax);
}

// cos and sin of 2 pi ph / 2^32: the nearest quarter turn is taken off in integers, and on the
// remaining eighth of a turn either side the Taylor polynomials (first omitted terms: 2e-9 of
// the sine, 1.2e-10 of the cosine) need no further reduction.  Half the instructions of
// sincospif on the converted phase, whose conversion also rounds a whole turn to 24 bits.
__device__ __forceinline__ void phase_cs(unsigned ph, float& c, float& s) {
  const unsigned k = ph + 0x20000000u;  // its top two bits: the quarter turn
  const float t = (float)((int)(k & 0x3FFFFFFFu) - 0x20000000) * 1.4629180792671596e-09f;  // 2 pi / 2^32
  const float z = t * t;
  float a = fmaf(z, 2.7557319e-6f, -1.9841270e-4f);
  a = fmaf(a, z, 8.3333333e-3f);
  a = fmaf(a, z, -1.6666667e-1f);
  a = fmaf(a * z, t, t);
  float b = fmaf(z, -2.7557319e-7f, 2.4801587e-5f);
  b = fmaf(b, z, -1.3888889e-3f);
  b = fmaf(b, z, 4.1666667e-2f);
  b = fmaf(b, z, -0.5f);
  b = fmaf(b, z, 1.0f);
  const bool odd = k & 0x40000000u;
  // quarter 0: (b, a), 1: (-a, b), 2: (-b, -a), 3: (a, -b)
  c = __uint_as_float(__float_as_uint(odd ? a : b) ^ ((k + 0x40000000u) & 0x80000000u));
  s = __uint_as_float(__float_as_uint(odd ? b : a) ^ (k & 0x80000000u));
}

struct Charges {
  float q[4];
};

// positions on the 32-bit grid, one coordinate per thread, and charges (32 atoms per block: two
// FP64 divisions each, so the block count decides)
__global__ void __launch_bounds__(96) ewald_atoms(const double* __restrict__ x, int n, int nw3, int single, double L,
                                                  Charges Q, uint4* __restrict__ xq) {
  const int a = blockIdx.x * 32 + threadIdx.x / 3, d = threadIdx.x % 3;
  if (a >= n) return;
  const double v = x[3 * (size_t)a + d];
  const double y = v - L * floor(v / L);
  unsigned* o = reinterpret_cast<unsigned*>(xq + a);
  o[d] = (unsigned)(unsigned long long)rint(y / L * 4294967296.0);
  if (d == 0)
    o[3] = __float_as_uint(a < nw3 ? (a % 3 == 0 ? Q.q[2] : Q.q[3])
                                   : (single || ((a - nw3) & 1) == 0 ? Q.q[0] : Q.q[1]));
}

// Structure-factor partials of one tile (32 columns x 16 n_z) and one chunk of atoms.  The
// block tabulates q a and b of 64 atoms in shared memory; each warp takes eight of them and
// accumulates the whole tile, a lane 4 columns x 4 n_z x 4 products (64 accumulators for 6
// wide shared loads an atom, two products per instruction).  A warp adds at most 64 atoms in
// FP32, then the eight warps' tiles are added pairwise and the chunks in FP64.
__global__ void __launch_bounds__(32 * kSkWarps, 2)
    ewald_sk_kernel(const uint4* __restrict__ xq, int n, KGeom G, int chunk_atoms, float* __restrict__ part) {
  extern __shared__ float4 sm4[];
  float* At = reinterpret_cast<float*>(sm4);  // [64 atoms][2][8 lanes][2 columns][re, im]
  float* Bt = At + kStage * 2 * kColT;        // [64 atoms][16 n_z][c, c, s, s]
  const int ct = blockIdx.x % G.nct, mt = blockIdx.x / G.nct;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, cg = lane & 7, mg = lane >> 3;
  const int a0 = blockIdx.y * chunk_atoms, a1 = min(n, a0 + chunk_atoms);
  const int2 mycol = column(min(ct * kColT + lane, G.ncol - 1), G.kmax);  // the column this lane tabulates
  float2 acc[4][4][2];
#pragma unroll
  for (int u = 0; u < 4; ++u)
#pragma unroll
    for (int v = 0; v < 4; ++v) acc[u][v][0] = acc[u][v][1] = make_float2(0.f, 0.f);
  // plane, lane and half of this lane's column in At
  float* const Aw = At + ((lane & 2) >> 1) * 32 + (lane >> 2) * 4 + (lane & 1) * 2;
  for (int t0 = a0; t0 < a1; t0 += kStage) {
    // (all of the stage's loads ahead of its arithmetic: one wait for L2 instead of four)
    uint4 p[kStage / kSkWarps];
    unsigned z[kStage * kMT / (32 * kSkWarps)];
#pragma unroll
    for (int r = 0; r < kStage / kSkWarps; ++r) {
      const int a = t0 + warp + r * kSkWarps;
      p[r] = a < a1 ? xq[a] : make_uint4(0u, 0u, 0u, 0u);
    }
#pragma unroll
    for (int r = 0; r < kStage * kMT / (32 * kSkWarps); ++r) {
      const int a = t0 + threadIdx.x / kMT + r * (32 * kSkWarps / kMT);
      z[r] = a < a1 ? xq[a].z : 0u;
    }
    __syncthreads();  // the tables of the stage before are done with
#pragma unroll
    for (int r = 0; r < kStage / kSkWarps; ++r) {
      const float q = __uint_as_float(p[r].w);
      float c, s;
      phase_cs((unsigned)mycol.x * p[r].x + (unsigned)mycol.y * p[r].y, c, s);
      *reinterpret_cast<float2*>(Aw + (warp + r * kSkWarps) * 64) = make_float2(q * c, q * s);
    }
#pragma unroll
    for (int r = 0; r < kStage * kMT / (32 * kSkWarps); ++r) {
      const int a = threadIdx.x / kMT + r * (32 * kSkWarps / kMT), m = threadIdx.x % kMT;
      float c, s;
      phase_cs((unsigned)(mt * kMT + m) * z[r], c, s);
      *reinterpret_cast<float4*>(Bt + a * 64 + 4 * m) = make_float4(c, c, s, s);
    }
    __syncthreads();
#pragma unroll 1
    for (int a = warp; a < kStage; a += kSkWarps) {
      float4 A[2], B[4];
#pragma unroll
      for (int h = 0; h < 2; ++h) A[h] = *reinterpret_cast<const float4*>(At + a * 64 + h * 32 + cg * 4);
#pragma unroll
      for (int v = 0; v < 4; ++v) B[v] = *reinterpret_cast<const float4*>(Bt + a * 64 + mg * 4 + v * 16);
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const float4 Ah = A[u >> 1];
        const float2 z = (u & 1) ? make_float2(Ah.z, Ah.w) : make_float2(Ah.x, Ah.y);
#pragma unroll
        for (int v = 0; v < 4; ++v) {
          acc[u][v][0] = __ffma2_rn(z, make_float2(B[v].x, B[v].y), acc[u][v][0]);
          acc[u][v][1] = __ffma2_rn(z, make_float2(B[v].z, B[v].w), acc[u][v][1]);
        }
      }
    }
  }
  // add the warps' tiles; value r of lane l is entry 32 r + l
  __syncthreads();
  float* red = reinterpret_cast<float*>(sm4);
#pragma unroll
  for (int u = 0; u < 4; ++u)
#pragma unroll
    for (int v = 0; v < 4; ++v)
#pragma unroll
      for (int k = 0; k < 2; ++k) {
        const int r = (u * 4 + v) * 4 + 2 * k;
        red[warp * kTileVals + r * 32 + lane] = acc[u][v][k].x;
        red[warp * kTileVals + (r + 1) * 32 + lane] = acc[u][v][k].y;
      }
  __syncthreads();
  float* o = part + ((size_t)blockIdx.y * gridDim.x + blockIdx.x) * kTileVals;
  for (int e = threadIdx.x; e < kTileVals; e += 32 * kSkWarps) {
    float s[kSkWarps];
#pragma unroll
    for (int w = 0; w < kSkWarps; ++w) s[w] = red[w * kTileVals + e];
    o[e] = ((s[0] + s[1]) + (s[2] + s[3])) + ((s[4] + s[5]) + (s[6] + s[7]));
  }
}

// Sums over the chunks, the energy, and the weights of the force pass.  A block takes 32
// (column, n_z) entries of a tile, one product each per warp: q a b = (re c, im c, re s, im s)
// sums give S(n_z) = (re c - im s, im c + re s) and S(-n_z) = (re c + im s, im c - re s).
// With W = A S of both, the force pass needs D = conj W(+) + conj W(-) and
// E = i (conj W(+) - conj W(-)), stored as (Re D, Re E, Im D, Im E).  run (if given) carries
// the sums over batches of atoms; the last batch writes the results.
__global__ void __launch_bounds__(128) ewald_sk_reduce(const float* __restrict__ part, KGeom G, int n_chunks, int first,
                                                       int last, double* __restrict__ run, float4* __restrict__ W,
                                                       double* __restrict__ u_part) {
  __shared__ double sum[4][32];
  const int tiles = G.nct * G.nmt, tile = blockIdx.x >> 4, uv = blockIdx.x & 15;
  const int k = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const size_t e = (size_t)tile * kTileVals + (uv * 4 + k) * 32 + lane;
  double s = first ? 0.0 : run[e];
#pragma unroll 8
  for (int c = 0; c < n_chunks; ++c) s += (double)part[(size_t)c * tiles * kTileVals + e];
  if (!last) {
    run[e] = s;
    return;
  }
  sum[k][lane] = s;
  __syncthreads();
  if (k != 0) return;
  const int u = uv >> 2, v = uv & 3;
  const int ct = tile % G.nct, mt = tile / G.nct;
  // the lane's columns in At: plane u / 2, half u % 2 of its group of four
  const int c = ct * kColT + (lane & 7) * 4 + u, m = mt * kMT + v * 4 + (lane >> 3);
  double en = 0.0;
  float4 w = make_float4(0.f, 0.f, 0.f, 0.f);
  if (c < G.ncol && m <= G.kmax && (c > 0 || m > 0)) {
    const int2 xy = column(c, G.kmax);
    const double A = G.e[xy.x] * G.e[abs(xy.y)] * G.e[m] /
                     (G.k1sq * (double)(xy.x * xy.x + xy.y * xy.y + m * m));
    const double rc = sum[0][lane], ic = sum[1][lane], rs = sum[2][lane], is = sum[3][lane];
    const double pr = rc - is, pi = ic + rs;
    double mr = rc + is, mi = ic - rs;
    if (c == 0 || m == 0) mr = mi = 0.0;  // -n_z is not in the half space, or is n_z itself
    en = A * ((pr * pr + pi * pi) + (mr * mr + mi * mi));
    w = make_float4((float)(A * (pr + mr)), (float)(A * (pi - mi)), (float)(-A * (pi + mi)), (float)(A * (pr - mr)));
  }
  if (c < G.ncol) W[(size_t)c * (G.nmt * kMT) + m] = w;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) en += __shfl_xor_sync(0xffffffffu, en, o);
  if (lane == 0) u_part[blockIdx.x] = en;
}

// Force partials of 128 atoms (one per thread) and one chunk of columns.  A thread keeps
// (cos, sin) and (-m sin, m cos) of its 16 n_z in registers; a column's weights are broadcast
// from shared memory, four packed FMAs per 16 bytes:
//   T = sum_m D c + E s,  T' = sum_m m (-i E c + i D s),
//   F_x += n_x Im(a T), F_y += n_y Im(a T), F_z += Im(a T').
// 16 columns (sums of up to 32 terms each) are added in FP32, the rest in FP64.
__global__ void __launch_bounds__(kFThreads, 4)
    ewald_force_kernel(const uint4* __restrict__ xq, int n, KGeom G, const float4* __restrict__ W, int chunk_cols,
                       double* __restrict__ part) {
  __shared__ float4 w[kFStage][kMT];
  __shared__ int2 col[kFStage];
  const int j = blockIdx.x * kFThreads + threadIdx.x;
  const uint4 p = j < n ? xq[j] : make_uint4(0u, 0u, 0u, 0u);
  const int c0 = blockIdx.y * chunk_cols, c1 = min(G.ncol, c0 + chunk_cols);
  double gx = 0.0, gy = 0.0, gz = 0.0;
  for (int mt = 0; mt < G.nmt; ++mt) {
    const int mn = min(kMT, G.kmax + 1 - mt * kMT);
    float2 b[kMT], bm[kMT];
#pragma unroll
    for (int m = 0; m < kMT; ++m) {
      float c, s;
      phase_cs((unsigned)(mt * kMT + m) * p.z, c, s);
      const float fm = (float)(mt * kMT + m);
      b[m] = make_float2(c, s);
      bm[m] = make_float2(-fm * s, fm * c);
    }
    for (int t0 = c0; t0 < c1; t0 += kFStage) {
      const int cn = min(kFStage, c1 - t0);
      __syncthreads();
      for (int e = threadIdx.x; e < cn * kMT; e += kFThreads)
        w[e / kMT][e % kMT] = W[(size_t)(t0 + e / kMT) * (G.nmt * kMT) + mt * kMT + e % kMT];
      if (threadIdx.x < cn) col[threadIdx.x] = column(t0 + threadIdx.x, G.kmax);
      __syncthreads();
      float fx = 0.f, fy = 0.f, fz = 0.f;
#pragma unroll 1
      for (int k = 0; k < cn; ++k) {
        const int2 xy = col[k];
        float ac, as;
        phase_cs((unsigned)xy.x * p.x + (unsigned)xy.y * p.y, ac, as);
        float2 tr = make_float2(0.f, 0.f), ti = tr, zr = tr, zi = tr;  // zi is the negative
#pragma unroll
        for (int m4 = 0; m4 < kMT; m4 += 4) {
          if (m4 >= mn) break;
#pragma unroll
          for (int m = m4; m < m4 + 4; ++m) {  // weights beyond kmax are zero
            const float4 q = w[k][m];
            const float2 re = make_float2(q.x, q.y), im = make_float2(q.z, q.w);
            tr = __ffma2_rn(re, b[m], tr);
            ti = __ffma2_rn(im, b[m], ti);
            zr = __ffma2_rn(im, bm[m], zr);
            zi = __ffma2_rn(re, bm[m], zi);
          }
        }
        const float f = fmaf(ac, ti.x + ti.y, as * (tr.x + tr.y));
        fx = fmaf((float)xy.x, f, fx);
        fy = fmaf((float)xy.y, f, fy);
        fz += fmaf(-ac, zi.x + zi.y, as * (zr.x + zr.y));
      }
      gx += (double)fx;
      gy += (double)fy;
      gz += (double)fz;
    }
  }
  if (j < n) {
    double* o = part + (size_t)blockIdx.y * 3 * n + j;
    o[0] = gx;
    o[(size_t)n] = gy;
    o[2 * (size_t)n] = gz;
  }
}

__global__ void __launch_bounds__(128) ewald_force_reduce(const uint4* __restrict__ xq, const double* __restrict__ part,
                                                          int n, int n_chunks, double pref, double* __restrict__ F) {
  const int j = blockIdx.x * blockDim.x + threadIdx.x, d = blockIdx.y;
  if (j >= n) return;
  double g = 0.0;
  for (int c = 0; c < n_chunks; ++c) g += part[((size_t)c * 3 + d) * n + j];
  F[3 * (size_t)j + d] = pref * (double)__uint_as_float(xq[j].w) * g;
}

size_t carve(size_t& off, size_t bytes) {
  const size_t o = off;
  off += (bytes + 255) & ~(size_t)255;
  return o;
}

int type_of_host(int a, int nw3) { return a < nw3 ? ((a % 3 == 0) ? 2 : 3) : ((a - nw3) & 1); }

int ceil_div(int a, int b) { return a / b + (a % b != 0); }

}  // namespace

extern "C" int h4d_ewald_lr(const h4d_params* params, double L, int32_t n_water, int32_t n, const double* x,
                            double alpha, int32_t kmax, double wbar, double kappa_lr, double* U_recip,
                            double* U_self, double* F, double* t_kernel_ms) {
  if (!params || !x || n < 0 || n_water < 0 || 3 * n_water > n || !(L > 0) || !(alpha > 0) || kmax < 1 ||
      kmax > kMaxK || !(wbar >= 0) || !(kappa_lr >= 0))
    return H4D_EINVAL;
  if (t_kernel_ms) *t_kernel_ms = 0.0;
  if (n == 0) {
    if (U_recip) *U_recip = 0.0;
    if (U_self) *U_self = 0.0;
    return H4D_OK;
  }
  const int single = params->exchange == H4D_EXCHANGE_SINGLE;
  const int nw3 = 3 * n_water;
  const double K = params->kcoul, V = L * L * L;
  const double g = std::exp(-kappa_lr * wbar);  // Eq. 10
  KGeom G;
  G.kmax = kmax;
  G.ncol = (kmax + 1) + kmax * (2 * kmax + 1);
  G.nct = ceil_div(G.ncol, kColT);
  G.nmt = ceil_div(kmax + 1, kMT);
  G.k1sq = (2.0 * M_PI / L) * (2.0 * M_PI / L);
  for (int m = 0; m <= kmax; ++m) G.e[m] = std::exp(-G.k1sq * m * m / (4.0 * alpha * alpha));
  Charges Q;
  for (int t = 0; t < 4; ++t) Q.q[t] = (float)params->q[t];
  // Atoms in chunks, so that tiles x chunks is one wave of resident blocks, of 1 to 8 stages
  // (eight: the longest FP32 sums); batches of chunks bound the partials' memory
  const int tiles = G.nct * G.nmt, stages = ceil_div(n, kStage);
  const int chunk = kStage * std::min(8, std::max(1, ceil_div(stages, std::max(1, kSlots / tiles))));
  const int n_chunks = ceil_div(n, chunk);
  const int batch = std::min(n_chunks, std::max(1, (int)(kPartBytes / (sizeof(float) * kTileVals * (size_t)tiles))));
  // columns in chunks of at least eight, one wave again; at most 32 chunks to add up
  const int ablocks = ceil_div(n, kFThreads);
  const int want = std::min(std::min(32, ceil_div(G.ncol, 8)), std::max(1, kFSlots / ablocks));
  const int chunk_c = ceil_div(G.ncol, want), nch_c = ceil_div(G.ncol, chunk_c);
  const int n_u = tiles * 16;
  const size_t na = (size_t)n;
  size_t off = 0;
  const size_t o_x = carve(off, na * 3 * sizeof(double));  // later the forces
  const size_t o_xq = carve(off, na * sizeof(uint4));
  const size_t o_u = carve(off, n_u * sizeof(double));
  const size_t o_w = carve(off, (size_t)G.ncol * G.nmt * kMT * sizeof(float4));
  const size_t o_run = carve(off, batch < n_chunks ? (size_t)tiles * kTileVals * sizeof(double) : 0);
  const size_t o_part = carve(off, std::max((size_t)batch * tiles * kTileVals * sizeof(float),
                                            F ? (size_t)nch_c * 3 * na * sizeof(double) : 0));
  std::vector<double> u;
  try {
    u.resize(n_u);
  } catch (const std::bad_alloc&) {
    return H4D_ECUDA;
  }
  void* slab = nullptr;
  if (h4d::scratch_alloc(&slab, off) != H4D_OK) return H4D_ECUDA;
  unsigned char* b = static_cast<unsigned char*>(slab);
  uint4* xq = reinterpret_cast<uint4*>(b + o_xq);
  double* d_x = reinterpret_cast<double*>(b + o_x);
  double* d_u = reinterpret_cast<double*>(b + o_u);
  float4* d_w = reinterpret_cast<float4*>(b + o_w);
  double* d_run = batch < n_chunks ? reinterpret_cast<double*>(b + o_run) : nullptr;
  cudaEvent_t ev[2] = {nullptr, nullptr};
  const size_t smem = sizeof(float) * kSkWarps * kTileVals;
  auto ok = [](cudaError_t e) { return e == cudaSuccess; };
  bool good = ok(cudaFuncSetAttribute(ewald_sk_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
  if (t_kernel_ms)
    for (auto& e : ev) good = good && ok(cudaEventCreate(&e));
  good = good && ok(cudaMemcpyAsync(d_x, x, na * 3 * sizeof(double), cudaMemcpyHostToDevice, 0));
  if (good) {
    if (t_kernel_ms) cudaEventRecord(ev[0]);
    ewald_atoms<<<ceil_div(n, 32), 96>>>(d_x, n, nw3, single, L, Q, xq);
    for (int c0 = 0; c0 < n_chunks; c0 += batch) {
      const int nc = std::min(batch, n_chunks - c0);
      const int a0 = c0 * chunk;
      float* part = reinterpret_cast<float*>(b + o_part);
      ewald_sk_kernel<<<dim3(tiles, nc), 32 * kSkWarps, smem>>>(xq + a0, n - a0, G, chunk, part);
      ewald_sk_reduce<<<n_u, 128>>>(part, G, nc, c0 == 0, c0 + nc == n_chunks, d_run, d_w, d_u);
    }
    if (F) {
      // F_j = g (4 pi K q_j / V) sum_{all k} A_k k [Re S sin - Im S cos]: twice the half space
      double* part = reinterpret_cast<double*>(b + o_part);
      ewald_force_kernel<<<dim3(ablocks, nch_c), kFThreads>>>(xq, n, G, d_w, chunk_c, part);
      ewald_force_reduce<<<dim3(ceil_div(n, 128), 3), 128>>>(xq, part, n, nch_c,
                                                            g * 8.0 * M_PI * K / V * (2.0 * M_PI / L), d_x);
    }
    if (t_kernel_ms) cudaEventRecord(ev[1]);
    good = ok(cudaGetLastError());
  }
  double qq = 0.0;  // on the host while the kernels run
  for (int a = 0; a < n; ++a) {
    const double q = params->q[single && a >= nw3 ? 0 : type_of_host(a, nw3)];
    qq += q * q;
  }
  good = good && ok(cudaMemcpy(u.data(), d_u, n_u * sizeof(double), cudaMemcpyDeviceToHost));
  if (F) good = good && ok(cudaMemcpy(F, d_x, na * 3 * sizeof(double), cudaMemcpyDeviceToHost));
  if (good && t_kernel_ms) {
    float ms = 0.f;
    good = ok(cudaEventElapsedTime(&ms, ev[0], ev[1]));
    *t_kernel_ms = ms;
  }
  if (!good) cudaStreamSynchronize(0);
  for (auto& e : ev)
    if (e) cudaEventDestroy(e);
  h4d::scratch_free(b, off);
  if (!good) return H4D_ECUDA;
  double sum = 0.0;
  for (int k = 0; k < n_u; ++k) sum += u[k];
  // U_recip = (2 pi K / V) sum_{all k != 0} A_k |S_k|^2 = (4 pi K / V) sum_half A_k |S_k|^2
  if (U_recip) *U_recip = g * 4.0 * M_PI * K / V * sum;
  if (U_self) *U_self = -g * K * alpha / std::sqrt(M_PI) * qq;
  return H4D_OK;
}
