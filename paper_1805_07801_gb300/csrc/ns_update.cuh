// The per-mode update of the Navier-Stokes right-hand side, shared by the
// fused forward x pass (ns_fwdx.cuh) and the split-precision path (ns.cu).
#pragma once

#include "fft_engine.cuh"
#include "fft_pipe.cuh"
#include "ns_common.cuh"

namespace fftk {
// Base shape of the x passes of powers of two: 8 values per thread.
template <int N>
struct NFCfg {
  static constexpr int G = N < 8 ? N : 8;
  static constexpr int S = N / G;
  static constexpr int T = S >= 32 ? (S == 32 ? 16 : (S == 64 ? 8 : 4)) : 16;
};

// ----------------------------------------------------- x pass + update -----

struct NSUpdate {
  const float2* etab;  // exp(-nu k^2 dt) = hi + lo (two FP32 parts), indexed by integer k^2;
                       // exp(-nu k^2 dt/2) follows at offset etab_len (the RK4 half steps)
  int etab_len;
  float2* acc;         // RK4 accumulator (3 fields)
  const double* ef;    // forced-mode energy (device scalar)
  double feps;         // injected power (0 = off)
  int k2min, k2max;
  float dt;
  float scale;         // 1 / n^3
};

// One kept mode (k_x, k_y, k_z) at index idx of each field: N = P[n] (Eq. (8)),
// + subgrid force, + forcing, then
//   RHS:    out = N
//   STAGE1: out = E (u0 + dt N)                      (out = u1)
//   STAGE2: out = 1/2 E u0 + 1/2 (u1 + dt N)         (out = u0, in place)
// or one stage of RK4 with H = exp(-nu k^2 dt/2), state u0, stage state u1,
// accumulator A (N from the stage's input: u0 in RK4_1, u1 after):
//   RK4_1:  A = E u0 + dt/6 E N,   out = H (u0 + dt/2 N)   (out = u1)
//   RK4_2:  A += dt/3 H N,         out = H u0 + dt/2 N     (out = u1)
//   RK4_3:  A += dt/3 H N,         out = E u0 + dt H N     (out = u1)
//   RK4_4:  out = A + dt/6 N                                (out = u0)
// in two steps, so that a thread can have the loads of several modes in
// flight before the first store (out may be u0, which orders loads after
// stores): what a mode reads,
struct NSModeIn {
  float2 E, H;  // integrating factors, hi + lo
  float2 a[3];  // u0
  float2 b[3];  // u1 (STAGE2) or the accumulator (RK4)
};

__device__ __forceinline__ void ns_mode_load(NSModeIn& in, int k2, long long idx, long long M, const NSUpdate& upd,
                                             int mode, const float2* u0, const float2* u1) {
  if (mode == NS_RHS) return;
  if (mode != NS_RK4_2 && mode != NS_RK4_4) in.E = __ldg(&upd.etab[k2]);
  if (mode >= NS_RK4_1 && mode != NS_RK4_4) in.H = __ldg(&upd.etab[upd.etab_len + k2]);
  if (mode != NS_RK4_4) {
#pragma unroll
    for (int f = 0; f < 3; ++f) in.a[f] = u0[idx + f * M];
  }
  if (mode == NS_STAGE2 || mode >= NS_RK4_2) {
    const float2* b = mode == NS_STAGE2 ? u1 : upd.acc;
#pragma unroll
    for (int f = 0; f < 3; ++f) in.b[f] = b[idx + f * M];
  }
}

// v * (hi + lo), one rounding: E = hi + lo carries the factor to ~2^-48, so
// repeated steps do not bias the decay
__device__ __forceinline__ float2 ns_mul_pair(float2 v, float2 E) {
  return make_float2(fmaf(v.x, E.x, v.x * E.y), fmaf(v.y, E.x, v.y * E.y));
}

// and the update from it
__device__ __forceinline__ void ns_mode_update(const NSModeIn& in, float2 nx, float2 ny, float2 nz, int kx, int ky,
                                               int kz, long long idx, long long M, const NSUpdate& upd, int mode,
                                               float gforce, const float2* u0, const float2* u1,
                                               const float2* __restrict__ extra, float2* out) {
  const int k2 = kx * kx + ky * ky + kz * kz;
  if (k2 == 0) {
    nx = ny = nz = make_float2(0.f, 0.f);
  } else {
    const float fkx = (float)kx, fky = (float)ky, fkz = (float)kz;
    const float inv = 1.f / (float)k2;
    const float2 kn = make_float2((fkx * nx.x + fky * ny.x + fkz * nz.x) * inv,
                                  (fkx * nx.y + fky * ny.y + fkz * nz.y) * inv);
    nx = csub(nx, cscale(kn, fkx));
    ny = csub(ny, cscale(kn, fky));
    nz = csub(nz, cscale(kn, fkz));
  }
  if (extra) {  // subgrid force, already dealiased and projected
    nx = cadd(nx, extra[idx]);
    ny = cadd(ny, extra[idx + M]);
    nz = cadd(nz, extra[idx + 2 * M]);
  }
  if (gforce != 0.f && k2 >= upd.k2min && k2 <= upd.k2max) {  // forced
    const float2* ucur = (mode == NS_STAGE2 || mode >= NS_RK4_2) ? u1 : u0;
    nx = cadd(nx, cscale(ucur[idx], gforce));
    ny = cadd(ny, cscale(ucur[idx + M], gforce));
    nz = cadd(nz, cscale(ucur[idx + 2 * M], gforce));
  }
  const float dt = upd.dt;
  const float2 n3[3] = {nx, ny, nz};
#pragma unroll
  for (int f = 0; f < 3; ++f) {
    const long long i = idx + f * M;
    const float2 nv = n3[f];
    if (mode == NS_RHS) {
      out[i] = nv;
    } else if (mode == NS_STAGE1) {
      const float2 a = in.a[f];
      out[i] = ns_mul_pair(make_float2(a.x + dt * nv.x, a.y + dt * nv.y), in.E);
    } else if (mode == NS_STAGE2) {
      const float2 ea = ns_mul_pair(in.a[f], in.E), b = in.b[f];
      out[i] = make_float2(0.5f * (ea.x + (b.x + dt * nv.x)), 0.5f * (ea.y + (b.y + dt * nv.y)));
    } else if (mode == NS_RK4_4) {
      const float2 c = in.b[f];
      out[i] = make_float2(fmaf(dt / 6.f, nv.x, c.x), fmaf(dt / 6.f, nv.y, c.y));
    } else if (mode == NS_RK4_1) {
      const float2 a = in.a[f], ea = ns_mul_pair(a, in.E), en = ns_mul_pair(nv, in.E);
      upd.acc[i] = make_float2(fmaf(dt / 6.f, en.x, ea.x), fmaf(dt / 6.f, en.y, ea.y));
      out[i] = ns_mul_pair(make_float2(a.x + 0.5f * dt * nv.x, a.y + 0.5f * dt * nv.y), in.H);
    } else {
      const float2 a = in.a[f], c = in.b[f], hn = ns_mul_pair(nv, in.H);
      upd.acc[i] = make_float2(fmaf(dt / 3.f, hn.x, c.x), fmaf(dt / 3.f, hn.y, c.y));
      if (mode == NS_RK4_2) {
        const float2 ha = ns_mul_pair(a, in.H);
        out[i] = make_float2(fmaf(0.5f * dt, nv.x, ha.x), fmaf(0.5f * dt, nv.y, ha.y));
      } else {
        const float2 ea = ns_mul_pair(a, in.E);
        out[i] = make_float2(fmaf(dt, hn.x, ea.x), fmaf(dt, hn.y, ea.y));
      }
    }
  }
}

// Transform of an x pass with its tile's buffers at `sm`: the line engine with
// an exchange buffer of the tile's size, or (TWO) two long-radix stages with a
// half-size buffer and the twiddles behind it.
template <int N, int G, int SIGN, int T, bool TWO>
struct XTransform {
  static constexpr size_t WORDS = TWO ? (size_t)N * T / 2 + N : (size_t)N * T;  // float2 at sm
  __device__ __forceinline__ static void init(float2* sm, const float2* tw, const float2* t3) {
    if constexpr (TWO)
      for (int i = threadIdx.x; i < N; i += N / G * T) sm[(size_t)N * T / 2 + i] = N % 3 == 0 ? t3[N + i] : tw[i];
  }
  __device__ __forceinline__ static void run(float2 (&v)[G], int j, int c, float2* sm, const float2* tw,
                                             const float2* t3) {
    if constexpr (TWO) {
      __syncthreads();  // the buffer may still be read
      pipe_transform<N, G, SIGN, T>(v, j, c, reinterpret_cast<float*>(sm), sm + (size_t)N * T / 2);
    } else {
      fft_line<N, G, SIGN>(v, j, ColX<T>{sm, c}, tw, t3);
    }
  }
};

// The forward x pass with the update of `mode` (ns_fwdx.cu, ns_fwdx3.cu).
cudaError_t ns_fwdx(fftk_plan p, const float2* nh, const float2* u0, const float2* u1, float2* out,
                    const NSUpdate& upd, int mode, const float2* extra, cudaStream_t st);
cudaError_t ns_fwdx3(fftk_plan p, const float2* nh, const float2* u0, const float2* u1, float2* out,
                     const NSUpdate& upd, int mode, const float2* extra, cudaStream_t st);

}  // namespace fftk
