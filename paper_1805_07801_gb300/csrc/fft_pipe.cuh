// Pieces of the pipelined strided passes (fft_stream.cu, ns_ypass.cu):
// persistent CTAs whose next tile of T = 16 columns x L rows streams into a
// staging buffer while this one is transformed in registers.
//
// Tiles are handed out in order: queue[0] counts them, each CTA draws one
// ahead (atomicAdd returns the next one after the first gridDim tiles), and
// the last CTA to leave sets the counters back to zero.  Were each CTA to take
// every gridDim-th tile, the CTAs would drift apart over a long pass, and
// neighbouring tiles, which share the lines of misaligned rows and the pages
// of DRAM, would no longer be worked on at the same time (1024^3 per pass: x
// 1.60 against 1.35 ms, y 2.14 against 1.37 ms).
#pragma once

#include "fft_engine.cuh"

namespace fftk {

__device__ __forceinline__ void pipe_leave(int* queue) {  // one thread of each CTA
  if (atomicAdd(queue + 1, 1) == (int)gridDim.x - 1) {
    queue[0] = 0;
    queue[1] = 0;
  }
}

// Slot of (row, column) in the half-size exchange buffer.  A warp holds two
// rows: rows G apart (the stores of the first stage) and neighbouring rows (the
// loads) each fall into different halves of the banks.
template <int G, int T>
__device__ __forceinline__ int pipe_slot(int pos, int c) {
  return ((pos ^ ((pos / G) & 1)) * T) + c;
}

// Two-stage transform (radix G, then R2 = L / G) of the line held in v (natural
// pattern v[m] = x[j + m S], S = L / G) by S threads, with one exchange through
// L T floats: real parts first, then imaginary parts.  stw: exp(-2 pi i m / L).
// The exchange buffer must be free on entry and may be in use on exit (a
// barrier comes before it is written again).  Natural pattern out, except with
// MIRROR (two butterflies per thread): thread j takes the second-stage
// butterflies j and G - j (of j = 0: 0 and G / 2), v[i + 2 r] = X[b_i + G r],
// so that every output's mirror is its own.
template <int L, int G, int SIGN, int T, bool MIRROR = false>
__device__ __forceinline__ void pipe_transform(float2 (&v)[G], int j, int c, float* ex, const float2* stw) {
  constexpr int S = L / G, R2 = L / G, B = G / R2;
  static_assert(G * R2 == L && B * R2 == G && (!MIRROR || B == 2), "two stages");
  auto bf = [&](int i) { return MIRROR && i == 1 ? (j == 0 ? G / 2 : G - j) : j + i * S; };
  dftR<G, SIGN>(v);
#pragma unroll
  for (int r = 0; r < G; ++r) ex[pipe_slot<G, T>(j * G + r, c)] = v[r].x;
  __syncthreads();
#pragma unroll
  for (int m = 0; m < G; ++m) v[m].x = ex[pipe_slot<G, T>(bf(m % B) + m / B * G, c)];
  __syncthreads();
#pragma unroll
  for (int r = 0; r < G; ++r) ex[pipe_slot<G, T>(j * G + r, c)] = v[r].y;
  __syncthreads();
#pragma unroll
  for (int m = 0; m < G; ++m) v[m].y = ex[pipe_slot<G, T>(bf(m % B) + m / B * G, c)];
  // second stage: butterfly i takes the values i + r B
#pragma unroll
  for (int i = 0; i < B; ++i) {
    float2 a[R2];
#pragma unroll
    for (int r = 0; r < R2; ++r) a[r] = v[i + r * B];
#pragma unroll
    for (int r = 1; r < R2; ++r) {
      const float2 w = stw[r * bf(i)];
      a[r] = SIGN < 0 ? cmul(a[r], w) : cmulc(a[r], w);
    }
    dftR<R2, SIGN>(a);
#pragma unroll
    for (int r = 0; r < R2; ++r) v[i + r * B] = a[r];
  }
}

}  // namespace fftk
