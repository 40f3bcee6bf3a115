// Training of the closure network (5 -> 64 -> 64 -> 64 -> 6, tanh on the
// hidden layers): forward, backward and the parameter update in FP32 on the
// CUDA cores.  Parameters (FP32): W1[64][5] b1 W2[64][64] b2 W3[64][64] b3
// W4[6][64] b4.  Each layer's input (x, h1, h2, h3) is rounded to bfloat16
// (or left as it is in the FP32 test mode); products and sums are FP32.
//
// The work is 26 k multiply-adds per sample against 44 bytes of input.  A CTA of
// 128 threads takes chunks of 64 samples; every product of the chunk is a small
// matrix product with 32 accumulators per thread (8 x 4), whose operands come
// from shared memory as 16-byte loads (three per 32 multiply-adds), and the
// gradient of the two 64 x 64 layers stays in registers from chunk to chunk.
// Two CTAs share an SM, so one fills the other's barriers.  Batch of 65536:
// gradient 1019 -> 127 us (one sample per thread, weights by broadcast loads,
// before; the FP32 pipes alone would take 45 us), with the sliced reduction and
// Adam 1121 -> 137 us.  Shared-memory loads are what bounds it: a 16-byte load
// takes four wavefronts however many lanes share an address.
//
// FP32 sums are short whatever the batch: 64 samples of a chunk, then at most
// kRun chunks of a CTA, whose totals are added in FP64; no term passes through
// more than 78 additions, and the rounding of a sum of equal terms (the worst
// case) is that of 128 terms in a row.  (One running sum per resident CTA has no
// such bound: of 2^21 equal samples, 108 chunks per CTA, it was off by 26 units
// of 2^-24.)  The further CTAs cost 2 % at a batch of 2^20: 1.68 -> 1.71 ms.
#include <cuda_bf16.h>

#include "internal.h"
#include "mlp_train.cuh"

namespace fftk {

namespace mlpcc {

constexpr int kChunk = 64;      // samples per chunk
constexpr int kThreads = 128;
constexpr int kLd = kChunk + 4;  // row length of [feature][sample] and [out][in] tiles: 16-byte rows, 4 banks apart
constexpr int kPerSm = 2;        // CTAs per SM (shared memory)
constexpr int kWave = 152 * kPerSm;
constexpr int kRun = 14;         // chunks of one CTA at most
// offsets in the parameter vector
constexpr int oW1 = 0, oB1 = 320, oW2 = 384, oB2 = 4480, oW3 = 4544, oB3 = 8640, oW4 = 8704, oB4 = 9088;

struct Smem {
  float w1[64 * 8];    // rows padded to 8
  float w2[64 * kLd];
  float w3[64 * kLd];
  float w4[6 * kLd];
  float b1[64], b2[64], b3[64], b4[8];
  float x[5 * kLd];           // layer inputs, [feature][sample]
  float a[3][64 * kLd];       // h1, h2, h3, overwritten by their deltas on the way back
  float d4[6 * kLd];          // output deltas
  double loss[kThreads / 32];
};

__device__ __forceinline__ float bf16r(float x) { return __bfloat162float(__float2bfloat16_rn(x)); }
// a layer input as the network defines it (BF16), or unrounded in the FP32
// test mode that isolates the kernels' arithmetic from the BF16 rounding
template <bool BF16>
__device__ __forceinline__ float act_round(float x) {
  return BF16 ? bf16r(x) : x;
}

__device__ __forceinline__ float4 ld4(const float* p) { return *reinterpret_cast<const float4*>(p); }

__device__ void load_params(Smem& s, const float* __restrict__ p) {
  const int t = threadIdx.x;
  for (int e = t; e < 320; e += kThreads) s.w1[(e / 5) * 8 + e % 5] = p[oW1 + e];
  for (int e = t; e < 4096; e += kThreads) {
    s.w2[(e >> 6) * kLd + (e & 63)] = p[oW2 + e];
    s.w3[(e >> 6) * kLd + (e & 63)] = p[oW3 + e];
  }
  for (int e = t; e < 384; e += kThreads) s.w4[(e >> 6) * kLd + (e & 63)] = p[oW4 + e];
  if (t < 64) {
    s.b1[t] = p[oB1 + t];
    s.b2[t] = p[oB2 + t];
    s.b3[t] = p[oB3 + t];
    if (t < 6) s.b4[t] = p[oB4 + t];
  }
}

// Outputs o = og + 8 q (q < 8) of 4 samples from b0: z = bias, then the
// products in the order of the inputs; tanh and the rounding into `out`.
// og = lane & 7: the 8 rows of W read together lie 4 banks apart.
template <bool BF16>
__device__ __forceinline__ void hidden_layer(const float* W, const float* bias, const float* in, float* out, int og,
                                             int b0) {
  float z[8][4];
#pragma unroll
  for (int q = 0; q < 8; ++q) {
    const float b = bias[og + 8 * q];
#pragma unroll
    for (int c = 0; c < 4; ++c) z[q][c] = b;
  }
#pragma unroll 1
  for (int i = 0; i < 64; i += 4) {
    const float4 a0 = ld4(in + i * kLd + b0), a1 = ld4(in + (i + 1) * kLd + b0);
    const float4 a2 = ld4(in + (i + 2) * kLd + b0), a3 = ld4(in + (i + 3) * kLd + b0);
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      const float4 w = ld4(W + (og + 8 * q) * kLd + i);
      z[q][0] = fmaf(w.w, a3.x, fmaf(w.z, a2.x, fmaf(w.y, a1.x, fmaf(w.x, a0.x, z[q][0]))));
      z[q][1] = fmaf(w.w, a3.y, fmaf(w.z, a2.y, fmaf(w.y, a1.y, fmaf(w.x, a0.y, z[q][1]))));
      z[q][2] = fmaf(w.w, a3.z, fmaf(w.z, a2.z, fmaf(w.y, a1.z, fmaf(w.x, a0.z, z[q][2]))));
      z[q][3] = fmaf(w.w, a3.w, fmaf(w.z, a2.w, fmaf(w.y, a1.w, fmaf(w.x, a0.w, z[q][3]))));
    }
  }
#pragma unroll
  for (int q = 0; q < 8; ++q)
    *reinterpret_cast<float4*>(out + (og + 8 * q) * kLd + b0) =
        make_float4(act_round<BF16>(tanhf(z[q][0])), act_round<BF16>(tanhf(z[q][1])),
                    act_round<BF16>(tanhf(z[q][2])), act_round<BF16>(tanhf(z[q][3])));
}

// Forward of the chunk's samples base .. base + nb - 1 (zeros beyond); y: the
// outputs 3 (t >> 6) + {0, 1, 2} of sample t & 63.
template <bool BF16>
__device__ __forceinline__ void chunk_forward(Smem& s, const float* __restrict__ x, long long base, int nb,
                                              float (&y)[3]) {
  const int t = threadIdx.x, lane = t & 31;
  const int og = lane & 7, b0 = 4 * ((lane >> 3) + 4 * (t >> 5));
  for (int e = t; e < 5 * kChunk; e += kThreads) {
    const int b = e / 5, i = e - 5 * b;
    s.x[i * kLd + b] = b < nb ? act_round<BF16>(x[base * 5 + e]) : 0.f;
  }
  __syncthreads();
  {
    float4 a[5];
#pragma unroll
    for (int i = 0; i < 5; ++i) a[i] = ld4(s.x + i * kLd + b0);
#pragma unroll 2
    for (int q = 0; q < 8; ++q) {
      const int o = og + 8 * q;
      const float4 w = ld4(s.w1 + o * 8);
      const float w4 = s.w1[o * 8 + 4], b = s.b1[o];
      const float z0 = fmaf(w4, a[4].x, fmaf(w.w, a[3].x, fmaf(w.z, a[2].x, fmaf(w.y, a[1].x, fmaf(w.x, a[0].x, b)))));
      const float z1 = fmaf(w4, a[4].y, fmaf(w.w, a[3].y, fmaf(w.z, a[2].y, fmaf(w.y, a[1].y, fmaf(w.x, a[0].y, b)))));
      const float z2 = fmaf(w4, a[4].z, fmaf(w.w, a[3].z, fmaf(w.z, a[2].z, fmaf(w.y, a[1].z, fmaf(w.x, a[0].z, b)))));
      const float z3 = fmaf(w4, a[4].w, fmaf(w.w, a[3].w, fmaf(w.z, a[2].w, fmaf(w.y, a[1].w, fmaf(w.x, a[0].w, b)))));
      *reinterpret_cast<float4*>(s.a[0] + o * kLd + b0) =
          make_float4(act_round<BF16>(tanhf(z0)), act_round<BF16>(tanhf(z1)), act_round<BF16>(tanhf(z2)),
                      act_round<BF16>(tanhf(z3)));
    }
  }
  __syncthreads();
  hidden_layer<BF16>(s.w2, s.b2, s.a[0], s.a[1], og, b0);
  __syncthreads();
  hidden_layer<BF16>(s.w3, s.b3, s.a[1], s.a[2], og, b0);
  __syncthreads();
  const int b = t & 63, o0 = 3 * (t >> 6);
#pragma unroll
  for (int o = 0; o < 3; ++o) y[o] = s.b4[o0 + o];
#pragma unroll 4
  for (int i = 0; i < 64; i += 4) {
    const float h0 = s.a[2][i * kLd + b], h1 = s.a[2][(i + 1) * kLd + b];
    const float h2 = s.a[2][(i + 2) * kLd + b], h3 = s.a[2][(i + 3) * kLd + b];
#pragma unroll
    for (int o = 0; o < 3; ++o) {
      const float4 w = ld4(s.w4 + (o0 + o) * kLd + i);
      y[o] = fmaf(w.w, h3, fmaf(w.z, h2, fmaf(w.y, h1, fmaf(w.x, h0, y[o]))));
    }
  }
}

// Delta of a layer's input for inputs i = 4 og + {0..3} and 32 + 4 og + {0..3}
// of 4 samples from b0: sum over the layer's ROWS outputs, in their order.
template <int ROWS>
__device__ __forceinline__ void back_rows(const float* W, const float* d, int og, int b0, float (&acc)[8][4]) {
#pragma unroll
  for (int q = 0; q < 8; ++q)
#pragma unroll
    for (int c = 0; c < 4; ++c) acc[q][c] = 0.f;
#pragma unroll 2
  for (int o = 0; o < ROWS; ++o) {
    const float4 dv = ld4(d + o * kLd + b0);
    const float4 wa = ld4(W + o * kLd + 4 * og), wb = ld4(W + o * kLd + 32 + 4 * og);
    const float w[8] = {wa.x, wa.y, wa.z, wa.w, wb.x, wb.y, wb.z, wb.w};
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      acc[q][0] = fmaf(w[q], dv.x, acc[q][0]);
      acc[q][1] = fmaf(w[q], dv.y, acc[q][1]);
      acc[q][2] = fmaf(w[q], dv.z, acc[q][2]);
      acc[q][3] = fmaf(w[q], dv.w, acc[q][3]);
    }
  }
}

// the same thread's elements of h, replaced by delta = acc (1 - h^2)
__device__ __forceinline__ void back_store(float* h, int og, int b0, const float (&acc)[8][4]) {
#pragma unroll
  for (int q = 0; q < 8; ++q) {
    float* p = h + ((q < 4 ? 4 * og + q : 32 + 4 * og + q - 4) * kLd) + b0;
    const float4 v = ld4(p);
    *reinterpret_cast<float4*>(p) =
        make_float4(acc[q][0] * (1.f - v.x * v.x), acc[q][1] * (1.f - v.y * v.y), acc[q][2] * (1.f - v.z * v.z),
                    acc[q][3] * (1.f - v.w * v.w));
  }
}

// The chunk's gradient of a 64 x 64 layer, o = og + 8 q, i = ig + 16 r, summed
// over its samples in their order and added to the running sum g.
__device__ __forceinline__ void outer64(const float* d, const float* h, int og, int ig, float (&g)[8][4]) {
  float acc[8][4];
#pragma unroll
  for (int q = 0; q < 8; ++q)
#pragma unroll
    for (int r = 0; r < 4; ++r) acc[q][r] = 0.f;
#pragma unroll 1
  for (int k = 0; k < kChunk; k += 4) {
    float4 hv[4];
#pragma unroll
    for (int r = 0; r < 4; ++r) hv[r] = ld4(h + (ig + 16 * r) * kLd + k);
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      const float4 dv = ld4(d + (og + 8 * q) * kLd + k);
#pragma unroll
      for (int r = 0; r < 4; ++r)
        acc[q][r] = fmaf(dv.w, hv[r].w, fmaf(dv.z, hv[r].z, fmaf(dv.y, hv[r].y, fmaf(dv.x, hv[r].x, acc[q][r]))));
    }
  }
#pragma unroll
  for (int q = 0; q < 8; ++q)
#pragma unroll
    for (int r = 0; r < 4; ++r) g[q][r] += acc[q][r];
}

__device__ __forceinline__ float row_sum(const float* row) {
  float acc = 0.f;
#pragma unroll
  for (int k = 0; k < kChunk; k += 4) {
    const float4 v = ld4(row + k);
    acc = acc + v.x;
    acc = acc + v.y;
    acc = acc + v.z;
    acc = acc + v.w;
  }
  return acc;
}

// sum over the chunk of d[k] h[k]
__device__ __forceinline__ float row_dot(const float* d, const float* h) {
  float acc = 0.f;
#pragma unroll 4
  for (int k = 0; k < kChunk; k += 4) {
    const float4 a = ld4(d + k), b = ld4(h + k);
    acc = fmaf(a.w, b.w, fmaf(a.z, b.z, fmaf(a.y, b.y, fmaf(a.x, b.x, acc))));
  }
  return acc;
}

}  // namespace mlpcc

// Chunks c = blockIdx.x, blockIdx.x + gridDim.x, ... of 64 samples: forward,
// backward, and this CTA's gradient and loss (sum of squared errors) over
// them into part[blockIdx.x], loss_part[blockIdx.x].
template <bool BF16>
__global__ void __launch_bounds__(mlpcc::kThreads, mlpcc::kPerSm)
    k_mlp_grad(const float* __restrict__ params, const float* __restrict__ x, const float* __restrict__ t, int B,
               int chunks, float* __restrict__ part, double* __restrict__ loss_part) {
  pdl_wait();
  using namespace mlpcc;
  extern __shared__ __align__(16) unsigned char smem_mlp[];
  Smem& s = *reinterpret_cast<Smem*>(smem_mlp);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int og = lane & 7, b0 = 4 * ((lane >> 3) + 4 * warp), ig = (lane >> 3) + 4 * warp;
  const int lo = tid & 63, half = tid >> 6;  // row and half of the small layers' products
  load_params(s, params);
  float g2[8][4], g3[8][4];
#pragma unroll
  for (int q = 0; q < 8; ++q)
#pragma unroll
    for (int r = 0; r < 4; ++r) g2[q][r] = g3[q][r] = 0.f;
  float g4[3] = {0.f, 0.f, 0.f}, g1[3] = {0.f, 0.f, 0.f};
  float gb23 = 0.f, gb4 = 0.f;  // b3 rows on the first 64 threads, b2 rows on the others; b4 on the first 6
  const float g = 2.f / (6.f * (float)B);
  double l2 = 0.0;
#pragma unroll 1
  for (int c = blockIdx.x; c < chunks; c += gridDim.x) {
    const long long base = (long long)c * kChunk;
    const int nb = min((long long)kChunk, (long long)B - base);
    float y[3];
    chunk_forward<BF16>(s, x, base, nb, y);
    // output error: dL/dz4 = 2 (y - t) / (6 B)
#pragma unroll
    for (int o = 0; o < 3; ++o) {
      const int oo = 3 * half + o;
      float e = 0.f;
      if (lo < nb) e = y[o] - t[(base + lo) * 6 + oo];
      l2 += (double)e * e;
      s.d4[oo * kLd + lo] = e * g;
    }
    __syncthreads();
    float acc[8][4];
    // layer 4 (its gradient reads h3, which its delta then replaces)
#pragma unroll
    for (int o = 0; o < 3; ++o) g4[o] += row_dot(s.d4 + (3 * half + o) * kLd, s.a[2] + lo * kLd);
    if (tid < 6) gb4 += row_sum(s.d4 + tid * kLd);
    back_rows<6>(s.w4, s.d4, og, b0, acc);
    __syncthreads();
    back_store(s.a[2], og, b0, acc);
    __syncthreads();
    // layer 3
    outer64(s.a[2], s.a[1], og, ig, g3);
    if (half == 0) gb23 += row_sum(s.a[2] + lo * kLd);
    back_rows<64>(s.w3, s.a[2], og, b0, acc);
    __syncthreads();
    back_store(s.a[1], og, b0, acc);
    __syncthreads();
    // layer 2
    outer64(s.a[1], s.a[0], og, ig, g2);
    if (half == 1) gb23 += row_sum(s.a[1] + lo * kLd);
    back_rows<64>(s.w2, s.a[1], og, b0, acc);
    __syncthreads();
    back_store(s.a[0], og, b0, acc);
    __syncthreads();
    // layer 1: inputs 0, 1, 2 on the first 64 threads; 3, 4 and the bias on the others
#pragma unroll
    for (int r = 0; r < 3; ++r) {
      const int i = 3 * half + r;
      g1[r] += i < 5 ? row_dot(s.a[0] + lo * kLd, s.x + i * kLd) : row_sum(s.a[0] + lo * kLd);
    }
    __syncthreads();  // the next chunk overwrites x
  }
  float* out = part + (long long)blockIdx.x * kNP;
#pragma unroll
  for (int q = 0; q < 8; ++q)
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      const int e = (og + 8 * q) * 64 + ig + 16 * r;
      out[oW2 + e] = g2[q][r];
      out[oW3 + e] = g3[q][r];
    }
#pragma unroll
  for (int o = 0; o < 3; ++o) out[oW4 + (3 * half + o) * 64 + lo] = g4[o];
#pragma unroll
  for (int r = 0; r < 3; ++r) {
    const int i = 3 * half + r;
    out[i < 5 ? oW1 + lo * 5 + i : oB1 + lo] = g1[r];
  }
  out[(half == 0 ? oB3 : oB2) + lo] = gb23;
  if (tid < 6) out[oB4 + tid] = gb4;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) l2 += __shfl_down_sync(0xffffffffu, l2, o);
  if (lane == 0) s.loss[warp] = l2;
  __syncthreads();
  if (tid == 0) loss_part[blockIdx.x] = (s.loss[0] + s.loss[1]) + (s.loss[2] + s.loss[3]);
}

// the forward pass alone, the arithmetic of k_mlp_grad's forward: y[B][6]
template <bool BF16>
__global__ void __launch_bounds__(mlpcc::kThreads, mlpcc::kPerSm)
    k_mlp_forward_cc(const float* __restrict__ params, const float* __restrict__ x, float* __restrict__ y, int B,
                     int chunks) {
  using namespace mlpcc;
  extern __shared__ __align__(16) unsigned char smem_mlp[];
  Smem& s = *reinterpret_cast<Smem*>(smem_mlp);
  const int lo = threadIdx.x & 63, half = threadIdx.x >> 6;
  load_params(s, params);
#pragma unroll 1
  for (int c = blockIdx.x; c < chunks; c += gridDim.x) {
    const long long base = (long long)c * kChunk;
    const int nb = min((long long)kChunk, (long long)B - base);
    float y3[3];
    chunk_forward<BF16>(s, x, base, nb, y3);
    if (lo < nb) {
#pragma unroll
      for (int o = 0; o < 3; ++o) y[(base + lo) * 6 + 3 * half + o] = y3[o];
    }
  }
}

// Adam (Kingma and Ba 2015) with bias corrections for parameter i
__device__ __forceinline__ void adam_update(const AdamStep& a, int i, float gi) {
  const float mi = a.b1 * a.m[i] + (1.f - a.b1) * gi;
  const float vi = a.b2 * a.v[i] + (1.f - a.b2) * gi * gi;
  a.m[i] = mi;
  a.v[i] = vi;
  a.params[i] -= a.lr * (mi / a.c1) / (sqrtf(vi / a.c2) + a.eps);
}

// Sums of the per-CTA partials in a fixed order, FP64: 32 parameters per
// block, eight threads each for every eighth partial, their sums in order.
// Bound by the read of the partials (11 MB up to 272384 samples, 36 KB per 896
// more; L2 holds those of 3 million).
constexpr int kRedCols = 32, kRedRows = 8;
template <bool ADAM>
__global__ void __launch_bounds__(kRedCols* kRedRows)
    k_mlp_reduce(const float* __restrict__ part, int nblk, float* __restrict__ grad,
                 const double* __restrict__ loss_part, double* __restrict__ loss, double inv_count, AdamStep adam) {
  pdl_wait();
  __shared__ double sum[kRedRows][kRedCols + 1];
  const int col = threadIdx.x % kRedCols, row = threadIdx.x / kRedCols;
  const int i = blockIdx.x * kRedCols + col;
  double acc = 0.0;
  if (i < kNP) {
#pragma unroll 8
    for (int k = row; k < nblk; k += kRedRows) acc += (double)part[(long long)k * kNP + i];
  }
  sum[row][col] = acc;
  __syncthreads();
  if (row == 0 && i < kNP) {
    double tot = 0.0;
#pragma unroll
    for (int r = 0; r < kRedRows; ++r) tot += sum[r][col];
    const float gi = (float)tot;
    grad[i] = gi;
    if constexpr (ADAM) adam_update(adam, i, gi);
  }
  if (loss && blockIdx.x == 0 && row == 1) {  // one warp: every 32nd partial, then the lanes in pairs
    double l = 0.0;
    for (int k = col; k < nblk; k += 32) l += loss_part[k];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) l += __shfl_down_sync(0xffffffffu, l, o);
    if (col == 0) *loss = l * inv_count;
  }
}

__global__ void k_adam(AdamStep a, const float* __restrict__ g, int n) {
  pdl_wait();
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) adam_update(a, i, g[i]);
}

// ------------------------------------------------------------ host side ----
static int mlp_chunks(long long B) { return (int)((B + mlpcc::kChunk - 1) / mlpcc::kChunk); }

// whole waves of CTAs from the first one on, as many as keep each to kRun chunks
int mlp_grad_blocks(long long B) {
  using namespace mlpcc;
  const int c = mlp_chunks(B);
  return c < kWave ? c : kWave * ((c + kWave * kRun - 1) / (kWave * kRun));
}

static cudaError_t mlp_cc_attrs() {
  static PerDevice once;
  return once.run([](int) {
    const int n = (int)sizeof(mlpcc::Smem);
    cudaError_t e = cudaFuncSetAttribute(k_mlp_grad<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, n);
    if (e == cudaSuccess)
      e = cudaFuncSetAttribute(k_mlp_grad<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, n);
    if (e == cudaSuccess)
      e = cudaFuncSetAttribute(k_mlp_forward_cc<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, n);
    if (e == cudaSuccess)
      e = cudaFuncSetAttribute(k_mlp_forward_cc<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, n);
    return e;
  });
}

cudaError_t launch_mlp_grad(bool bf16, const float* params, const float* x, const float* t, int B, float* part,
                            double* loss_part, cudaStream_t st) {
  const cudaError_t e = mlp_cc_attrs();
  if (e != cudaSuccess) return e;
  const int blocks = mlp_grad_blocks(B), chunks = mlp_chunks(B);
  if (bf16)
    launch_pdl(k_mlp_grad<true>, blocks, mlpcc::kThreads, sizeof(mlpcc::Smem), st, params, x, t, B, chunks, part,
               loss_part);
  else
    launch_pdl(k_mlp_grad<false>, blocks, mlpcc::kThreads, sizeof(mlpcc::Smem), st, params, x, t, B, chunks, part,
               loss_part);
  return cudaGetLastError();
}

cudaError_t launch_mlp_reduce(int B, const float* part, const double* loss_part, float* grad, double* loss,
                              const AdamStep* adam, cudaStream_t st) {
  const int blocks = (kNP + kRedCols - 1) / kRedCols, nblk = mlp_grad_blocks(B);
  const double inv = 1.0 / (6.0 * (double)B);
  if (adam)
    launch_pdl(k_mlp_reduce<true>, blocks, kRedCols * kRedRows, 0, st, part, nblk, grad, loss_part, loss, inv, *adam);
  else
    launch_pdl(k_mlp_reduce<false>, blocks, kRedCols * kRedRows, 0, st, part, nblk, grad, loss_part, loss, inv,
               AdamStep{});
  return cudaGetLastError();
}

cudaError_t launch_mlp_forward_cc(bool bf16, const float* params, const float* x, float* y, int B, cudaStream_t st) {
  const cudaError_t e = mlp_cc_attrs();
  if (e != cudaSuccess) return e;
  const int chunks = mlp_chunks(B), blocks = chunks < mlpcc::kWave ? chunks : mlpcc::kWave;
  if (bf16)
    k_mlp_forward_cc<true><<<blocks, mlpcc::kThreads, sizeof(mlpcc::Smem), st>>>(params, x, y, B, chunks);
  else
    k_mlp_forward_cc<false><<<blocks, mlpcc::kThreads, sizeof(mlpcc::Smem), st>>>(params, x, y, B, chunks);
  return cudaGetLastError();
}

cudaError_t launch_adam(const AdamStep& a, const float* grad, cudaStream_t st) {
  launch_pdl(k_adam, (kNP + 255) / 256, 256, 0, st, a, grad, kNP);
  return cudaGetLastError();
}

}  // namespace fftk
