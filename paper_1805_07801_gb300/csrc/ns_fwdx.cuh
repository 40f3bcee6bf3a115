// The fused forward x pass of the Navier-Stokes right-hand side: instantiated
// for powers of two in ns_fwdx.cu and for 3 * 2^m in ns_fwdx3.cu.
#pragma once

#include <mutex>

#include "ns_update.cuh"

namespace fftk {

// The pass moves three fields in and, with the stage state and the accumulator,
// three to twelve more fields of kept modes, and is bound by the latency of
// those accesses: its one CTA per SM (the exchange buffer and the two parked
// fields fill the shared memory) loads, transforms and updates in turn.
// 512^3, RK2: 648 us per launch with the update's loads one mode at a time,
// 567 us with the loads of two modes in flight (the mode a template argument,
// so that they fit into 64 registers), 484 us with the L2 prefetches below
// (546 us with all of them at the start), 468 us with two long-radix stages
// instead of three; 64^3: 12.6 -> 8.3 us; 768^3: 2.87 -> 2.26 ms, with radix 48
// and 16 instead of 8, 8, 12 1.76 ms.
//
// One field is in registers and two are parked.  From n = 256 on, two stages with
// the half-size exchange (XTransform) on 256 threads, 16 columns per tile (8 at n =
// 1024, whose parked fields fill the shared memory); below, and at 384, whose 24
// values hold no whole number of radix-16 butterflies, the line engine with 24
// (3 * 2^m) or 8 values per thread and 16 columns.  RK2 / RK4 step with 8 values
// and so: 256^3 833 / 1706 -> 820 / 1682 us, 1024^3 62.6 / 128.8 -> 61.6 / 127.0 ms
// (64 registers spilled up to 64 bytes there).  With two stages and for 3 * 2^m
// only the slots m whose rows j + m S can be kept by the 2/3 rule are parked, the
// first LOW and those from HIGH on.
template <int N>
struct NUCfg {
  static constexpr bool TWO = N >= 256 && N != 384;  // radix 48, 32 or 16, then 16 (32 at 1024)
  static constexpr int G = N == 768 ? 48 : N == 256 ? 16 : TWO ? 32 : (N % 3 == 0 ? elems_per_thread(N) : NFCfg<N>::G);
  static constexpr int S = N / G;
  static constexpr int T = N == 1024 ? 8 : 16;
  static constexpr int THREADS = T * S;
  static constexpr int KD = (N - 1) / 3;
  static constexpr int LOW = N % 3 != 0 && !TWO ? G : KD / S + 1;
  static constexpr int HIGH = (N - KD) / S > LOW ? (N - KD) / S : LOW;
  static constexpr int SLOTS = LOW + G - HIGH;
  using X = XTransform<N, G, -1, T, TWO>;
  static constexpr size_t SMEM = sizeof(float2) * (X::WORDS + 2 * (size_t)SLOTS * THREADS);
  static constexpr int MINB = TWO          ? (N == 256 ? 2 : 1)
                              : N % 3 == 0 ? (THREADS <= 128 ? 4 : (THREADS <= 256 ? 2 : 1))
                                           : (512 / THREADS < 8 ? 512 / THREADS : 8);
  static constexpr int GROUP = 4;  // modes whose loads are in flight together
  __host__ __device__ static constexpr bool parked(int m) { return m < LOW || m >= HIGH; }
  __host__ __device__ static constexpr int slot(int m) { return m < LOW ? m : m - HIGH + LOW; }
};

// 5. forward x pass of the 3 nonlinear fields, then on every kept mode:
//    N = P[n] (Eq. (8)), + forcing, and
//    RHS:    out = N
//    STAGE1: out = E (u0 + dt N)                      (out = u1)
//    STAGE2: out = 1/2 E u0 + 1/2 (u1 + dt N)         (out = u0, in place)
template <int N, int MODE>
__global__ void __launch_bounds__(NUCfg<N>::THREADS, NUCfg<N>::MINB)
    k_ns_fwdx(const float2* __restrict__ nh, const float2* u0, const float2* u1, float2* out,
              int ktiles, NSUpdate upd, const float2* __restrict__ extra, const float2* __restrict__ tw,
              const float2* __restrict__ t3) {
  pdl_wait();
  constexpr long long H1 = N / 2 + 1, MM = (long long)N * N * H1;  // geometry of the n^3 grid
  constexpr long long HW = ns_row(N), MW = (long long)N * N * HW;  // the padded workspace (nh)
  constexpr int KD = (N - 1) / 3;                                  // largest kept |k| (2/3 rule)
  using C = NUCfg<N>;
  constexpr int G = C::G, S = C::S, T = C::T;
  extern __shared__ float2 smn[];
  const int c = threadIdx.x % T, j = threadIdx.x / T;
  const int dky = blockIdx.x / ktiles;
  const int ay = dense_to_a(dky, N, KD);
  const int kz = (blockIdx.x - dky * ktiles) * T + c;
  const bool valid = kz < (KD + 1);
  const long long q = (long long)ay * H1 + kz;
  const long long rs = (long long)N * H1;
  const long long qw = (long long)ay * HW + kz, rw = (long long)N * HW;
  // fields 0 and 1 are parked in shared memory after their transforms (this
  // thread's slots only), so one field at a time is held in registers
  float2* park = smn + C::X::WORDS + threadIdx.x;
  C::X::init(smn, tw, t3);
  const float2* bsrc = MODE == NS_STAGE2 ? u1 : upd.acc;
  constexpr bool A0 = MODE != NS_RHS && MODE != NS_RK4_4, B0 = MODE == NS_STAGE2 || MODE >= NS_RK4_2;
  float2 V[G];
#pragma unroll 1
  for (int f = 0; f < 3; ++f) {
#pragma unroll
    for (int m = 0; m < G; ++m)
      V[m] = valid ? nh[f * MW + (j + m * S) * rw + qw] : make_float2(0.f, 0.f);
    if constexpr (N >= 256) {
      // The next field, and with the last two the update's reads, go to L2
      // while this field is transformed: one CTA holds the SM, so nothing else
      // covers those loads.  (All at once at the start would fill the L2.)
      if (f < 2)
        for (int r = threadIdx.x; r < N; r += C::THREADS) prefetch_l2(nh + (f + 1) * MW + r * rw + qw - c);
      if ((A0 && f == 1) || (B0 && f == 2)) {
        const float2* src = f == 1 ? u0 : bsrc;
        for (int r = threadIdx.x; r < 2 * KD + 1; r += C::THREADS) {
          const long long o = dense_to_a(r, N, KD) * rs + q - c;
#pragma unroll
          for (int i = 0; i < 3; ++i) prefetch_l2(src + i * MM + o);
        }
      }
    }
    C::X::run(V, j, c, smn, tw, t3);
    if (f < 2) {
#pragma unroll
      for (int m = 0; m < G; ++m)
        if (C::parked(m)) park[(f * C::SLOTS + C::slot(m)) * C::THREADS] = V[m];
    }
  }
  if (!valid) return;
  const int ky = kwav(ay, N);
  float gforce = 0.f;
  if (upd.feps > 0.0) {
    const double ef = *upd.ef;
    gforce = ef > 0.0 ? (float)(upd.feps / (2.0 * ef)) : 0.f;
  }
  constexpr int NG = C::GROUP;
#pragma unroll
  for (int m0 = 0; m0 < G; m0 += NG) {
    NSModeIn in[NG];
#pragma unroll
    for (int i = 0; i < NG; ++i) {
      const int m = m0 + i, pos = j + m * S, kx = kwav(pos, N);
      if (C::parked(m) && kept_xy(pos, N, KD))
        ns_mode_load(in[i], kx * kx + ky * ky + kz * kz, pos * rs + q, MM, upd, MODE, u0, u1);
    }
#pragma unroll
    for (int i = 0; i < NG; ++i) {
      const int m = m0 + i, pos = j + m * S;
      if (!C::parked(m) || !kept_xy(pos, N, KD)) continue;
      ns_mode_update(in[i], cscale(park[C::slot(m) * C::THREADS], upd.scale),
                     cscale(park[(C::SLOTS + C::slot(m)) * C::THREADS], upd.scale), cscale(V[m], upd.scale),
                     kwav(pos, N), ky, kz, pos * rs + q, MM, upd, MODE, gforce, u0, u1, extra, out);
    }
  }
}

template <int N, int MODE>
static cudaError_t fwdx_nm(fftk_plan p, const float2* nh, const float2* u0, const float2* u1, float2* out,
                           const NSUpdate& upd, const float2* extra, cudaStream_t st) {
  using U = NUCfg<N>;
  static PerDevice once;
  const cudaError_t e = once.run([](int) {
    return cudaFuncSetAttribute(k_ns_fwdx<N, MODE>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)U::SMEM);
  });
  if (e != cudaSuccess) return e;
  constexpr int KD = (N - 1) / 3, KT = (KD + U::T) / U::T;  // k_z tiles of KD + 1 columns
  LaunchScope ls(p, KK_NS_FWDX, st);
  launch_pdl(k_ns_fwdx<N, MODE>, (2 * KD + 1) * KT, U::THREADS, U::SMEM, st, nh, u0, u1, out, KT, upd, extra,
                                                                  twiddles(p, 1 << Log2<N>::value), p->d_tw3);
  return cudaGetLastError();
}

template <int N>
static cudaError_t fwdx_n(fftk_plan p, const float2* nh, const float2* u0, const float2* u1, float2* out,
                          const NSUpdate& upd, int mode, const float2* extra, cudaStream_t st) {
  switch (mode) {
#define MODE(m) \
  case m:       \
    return fwdx_nm<N, m>(p, nh, u0, u1, out, upd, extra, st);
    MODE(NS_RHS) MODE(NS_STAGE1) MODE(NS_STAGE2) MODE(NS_RK4_1) MODE(NS_RK4_2) MODE(NS_RK4_3) MODE(NS_RK4_4)
#undef MODE
  }
  return cudaErrorInvalidValue;
}

}  // namespace fftk
