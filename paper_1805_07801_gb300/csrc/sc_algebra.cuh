// Point algebra of the sine/cosine transforms (fft_sc.cu states the method).
#pragma once

#include "fft_engine.cuh"

namespace fftk {

__device__ __forceinline__ int sc_perm(int r, int L) { return r < L / 2 ? 2 * r : 2 * (L - 1 - r) + 1; }
// position r of element i in the permuted line
__device__ __forceinline__ int sc_unperm(int i, int L) { return (i & 1) ? L - 1 - (i >> 1) : (i >> 1); }

// C_k from V_k, V_{L-k} and W_k
__device__ __forceinline__ float2 sc_post(float2 vk, float2 vn, float2 w) {
  const float2 a = cmul(w, vk), b = cmulc(vn, w);  // W V_k, conj(W) V_{L-k}
  return make_float2(0.5f * (a.x + b.x), 0.5f * (a.y + b.y));
}

// V_k = conj(W_k) (C_k - i C_{L-k})
__device__ __forceinline__ float2 sc_pre(float2 ck, float2 cn, float2 w) {
  const float2 d = make_float2(ck.x + cn.y, ck.y - cn.x);  // C_k - i C_{L-k}
  return cmulc(d, w);
}

}  // namespace fftk
