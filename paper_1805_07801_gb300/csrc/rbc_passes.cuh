// The fused passes of the convection right-hand side (rbc.cu describes the
// method), as templates on the grid size: instantiated for powers of two in
// rbc_pow2.cu and for 3 * 2^m in rbc_radix3.cu.  The workspace has the fused
// Navier-Stokes passes' padded rows (ns_row).
#pragma once

#include <mutex>

#include "ns_passes.cuh"

namespace fftk {

struct RBCUpdate {
  const float2* tab;  // E_nu, E_kappa, H_nu, H_kappa at offsets 0, L, 2L, 3L
  int tab_len;
  float dt;
};

__device__ __forceinline__ float2 mul_pair(float2 v, float2 E) {  // v * (hi + lo), one rounding
  return make_float2(fmaf(v.x, E.x, v.x * E.y), fmaf(v.y, E.x, v.y * E.y));
}

// the update of entry i of one field in mode MODE (the modes of
// ns_mode_update): N = n, a = u0, b = the stage state or the accumulator; i is
// the entry of out, ia that of the accumulator
template <int MODE>
__device__ __forceinline__ void rbc_entry_store(long long i, long long ia, float2 n, float2 a, float2 b, float2 E, float2 H, float dt,
                                                float2* acc, float2* out) {
  if constexpr (MODE == NS_RHS) {
    out[i] = n;
  } else if constexpr (MODE == NS_STAGE1) {
    out[i] = mul_pair(make_float2(a.x + dt * n.x, a.y + dt * n.y), E);
  } else if constexpr (MODE == NS_STAGE2) {
    const float2 ea = mul_pair(a, E);
    out[i] = make_float2(0.5f * (ea.x + (b.x + dt * n.x)), 0.5f * (ea.y + (b.y + dt * n.y)));
  } else if constexpr (MODE == NS_RK4_4) {
    out[i] = make_float2(fmaf(dt / 6.f, n.x, b.x), fmaf(dt / 6.f, n.y, b.y));
  } else if constexpr (MODE == NS_RK4_1) {
    const float2 ea = mul_pair(a, E), en = mul_pair(n, E);
    acc[ia] = make_float2(fmaf(dt / 6.f, en.x, ea.x), fmaf(dt / 6.f, en.y, ea.y));
    out[i] = mul_pair(make_float2(a.x + 0.5f * dt * n.x, a.y + 0.5f * dt * n.y), H);
  } else {
    const float2 hn = mul_pair(n, H);
    acc[ia] = make_float2(fmaf(dt / 3.f, hn.x, b.x), fmaf(dt / 3.f, hn.y, b.y));
    if constexpr (MODE == NS_RK4_2) {
      const float2 ha = mul_pair(a, H);
      out[i] = make_float2(fmaf(0.5f * dt, n.x, ha.x), fmaf(0.5f * dt, n.y, ha.y));
    } else {
      const float2 ea = mul_pair(a, E);
      out[i] = make_float2(fmaf(dt, hn.x, ea.x), fmaf(dt, hn.y, ea.y));
    }
  }
}

// Slots of the workspace: in[7] = u_x, u_y, u_z, omega_x, omega_y, omega_z,
// theta; out[6] = n_x, n_y, n_z, u_x theta, u_y theta, u_z theta.
struct RBCSlots {
  int in[7];
  int out[6];
};

// What the launchers of one stage need besides the plan.
struct RBCStage {
  float2* w;          // 7 fields, padded rows
  const float2* x;    // the stage's input state (the stage state from the second stage on)
  const float2* u0;   // the step's state
  const float2* s1;   // stage state, padded rows
  float2* acc;        // RK4 accumulator, padded rows
  float2* out;
  RBCUpdate upd;
  int mode;
  float scale;        // 1 / n^3
};

// the fused z pass on the padded workspace
cudaError_t rbc_z(fftk_plan p, float2* w, const RBCSlots& sl, cudaStream_t st);
cudaError_t rbc_z3(fftk_plan p, float2* w, const RBCSlots& sl, cudaStream_t st);
// periodic cube: the inverse x pass with the curl (state -> 7 fields), and the
// forward x pass with the update (6 fields -> out)
// (padded: x is the stage state)
cudaError_t rbc_invx(fftk_plan p, const float2* x, bool padded, float2* w, cudaStream_t st);
cudaError_t rbc_invx3(fftk_plan p, const float2* x, bool padded, float2* w, cudaStream_t st);
cudaError_t rbc_fwdx(fftk_plan p, const RBCStage& s, cudaStream_t st);
cudaError_t rbc_fwdx3(fftk_plan p, const RBCStage& s, cudaStream_t st);

// ---- fused z pass (both bases: z is Fourier in each) ----------------------
// Per (x, y) line: c2r of u, theta (parked in shared memory) and of the three
// vorticity components (folded into the accumulators of n = u x omega), then
// r2c of n and of u theta: thirteen transforms, in place (a slot is written
// after it has been read).  Like the Navier-Stokes z pass it is bound by its
// instructions; it shares that pass's shape (NZCfg): few long-radix stages,
// the inputs staged by bulk copies two fields ahead, Hermitian-split factors
// from one table load per thread.  512^3: 2031 us per launch with 8 values per
// thread and plain loads, 1679 us so; 256^3: 265 and 225 us.
template <int N>
struct RZCfg {
  using Z = NZCfg<N, 4096>;  // (with 24 values only one CTA of four parked fields would fit)
  static constexpr int H = Z::H, HB = Z::HB, G = Z::G, S = Z::S, LPC = Z::LPC, NBUF = Z::NBUF, THREADS = Z::THREADS;
  static constexpr bool WARP = Z::WARP;
  static constexpr int KC = Z::KC, KCP = Z::KCP;
  static constexpr size_t FIELDS = sizeof(float2) * (size_t)LPC * (HB + 4 * H);  // exchange + 4 parked fields
  static constexpr size_t STAGE = Z::STAGE;
  static constexpr size_t SMEM = FIELDS + STAGE + sizeof(uint64_t) * NBUF * LPC;
  static constexpr int MINB = G == 12 ? 2 : (N == 256 ? 4 : Z::MINB);
};

template <int N>
__global__ void __launch_bounds__(RZCfg<N>::THREADS, RZCfg<N>::MINB)
    k_rbc_z(float2* w, RBCSlots sl, const float2* __restrict__ tw, const float2* __restrict__ t3, int* err) {
  pdl_wait();
  constexpr long long HW = ns_row(N), MM = (long long)N * N * HW;
  using C = RZCfg<N>;
  constexpr int H = C::H, G = C::G, S = C::S, KC = C::KC, NB = C::NBUF;
  constexpr int LOGN = Log2<N>::value;
  extern __shared__ __align__(16) float2 smz[];
  const int li = threadIdx.x / S, j = threadIdx.x % S;
  const long long line = (long long)blockIdx.x * C::LPC + li;
  const bool valid = line < (long long)N * N;
  const LineX<C::WARP, S, G> xc{smz + li * C::HB, line_xor<S>(li)};
  float2* park = smz + C::LPC * C::HB + li * 4 * H + j;  // [4][G][S]: u_x, u_y, u_z, theta
  float2* stage = smz + C::FIELDS / sizeof(float2) + li * NB * C::KCP;
  uint64_t* bar = reinterpret_cast<uint64_t*>(smz + (C::FIELDS + C::STAGE) / sizeof(float2)) + NB * li;

  // the inputs in the order of their use: u, theta, omega; a line's rows start
  // on 128-byte lines, a copy is KC values rounded up to even
  constexpr uint32_t bytes = (uint32_t)(sizeof(float2) * ((KC + 1) & ~1));
  auto issue = [&](int f) {  // one thread of the line; buffer f % NB was last read NB fields ago
    const int slot = sl.in[f < 3 ? f : (f == 3 ? 6 : f - 1)];
    uint64_t* b = bar + f % NB;
    tcg::fence_smem_async();
    tcg::mbar_expect(b, bytes);
    tcg::bulk_g2s(stage + (f % NB) * C::KCP, w + slot * MM + line * HW, bytes, b);
  };
  bool ok = true;
  auto arrive = [&](int f) {  // wait for input f's copy (bounded; an expired wait is reported)
    if (!valid) return;
    const uint32_t par = (uint32_t)((f / NB) & 1);
    if (!tcg::mbar_wait(bar + f % NB, par)) {
      if (j == 0 && ok) atomicOr(err, 1);
      ok = false;
      tcg::mbar_wait(bar + f % NB, par);  // once more for the copy still in flight
    }
  };
  if (j == 0 && valid) {
    for (int b = 0; b < NB; ++b) tcg::mbar_init(bar + b);
    for (int b = 0; b < NB; ++b) issue(b);
  }
  xc.sync();  // the barriers are initialised before anyone polls them
  const SplitFactors<N, G> twk(N % 3 == 0 ? t3 + N : tw, j);

  auto c2r = [&](int f, float2(&U)[G]) {
    const float2* src = stage + (f % NB) * C::KCP;
    arrive(f);
#pragma unroll
    for (int m = 0; m < G; ++m) {
      const int k = j + m * S;
      float2 A = make_float2(0.f, 0.f), B = make_float2(0.f, 0.f);
      if (k < KC) A = src[k];
      if (H - k < KC) B = src[H - k];
      if (k == 0) {
        A.y = 0.f;
        B.y = 0.f;
      }
      const float2 Bc = cconj(B);
      const float2 E = cadd(A, Bc);
      const float2 O = cmulc(csub(A, Bc), twk(m));
      U[m] = make_float2(E.x - O.y, E.y + O.x);
    }
    if constexpr (S == 1) xc.sync();  // (one thread per line: the transform has no exchange)
    fft_line<H, G, +1, LOGN>(U, j, xc, tw, t3);
    if (f + NB < 7 && j == 0 && valid) issue(f + NB);
  };
  auto r2c = [&](int slot, float2(&U)[G]) {
    fft_line<H, G, -1, LOGN>(U, j, xc, tw, t3);
#pragma unroll
    for (int m = 0; m < G; ++m) xc.st_run(j + m * S, U[m]);
    xc.sync();
    float2* dst = w + slot * MM + line * HW;
#pragma unroll
    for (int m = 0; m < G; ++m) {
      const int k = j + m * S;
      const float2 Bc = cconj(xc.ld_run(mirror<H>(k)));
      const float2 E = cscale(cadd(U[m], Bc), 0.5f);
      const float2 D = csub(U[m], Bc);
      const float2 O = make_float2(0.5f * D.y, -0.5f * D.x);
      if (valid && k < KC) dst[k] = cadd(E, cmul(twk(m), O));
    }
    xc.sync();
  };
  auto pk = [&](int f, int m) -> float2& { return park[(f * G + m) * S]; };
  auto neg = [](float2 a) { return make_float2(-a.x, -a.y); };
  {
    float2 U[G];
#pragma unroll 1
    for (int f = 0; f < 4; ++f) {
      c2r(f, U);
#pragma unroll
      for (int m = 0; m < G; ++m) pk(f, m) = U[m];
    }
  }
  // n = u x omega, two real points per slot (see k_ns_z)
  float2 Ny[G], Nx[G];
  {
    float2 Nz[G];
    {
      float2 W[G];
      c2r(4, W);  // omega_x
#pragma unroll
      for (int m = 0; m < G; ++m) {
        Ny[m] = __fmul2_rn(pk(2, m), W[m]);
        Nz[m] = __fmul2_rn(neg(pk(1, m)), W[m]);
      }
      c2r(5, W);  // omega_y
#pragma unroll
      for (int m = 0; m < G; ++m) {
        Nx[m] = __fmul2_rn(neg(pk(2, m)), W[m]);
        Nz[m] = __ffma2_rn(pk(0, m), W[m], Nz[m]);
      }
    }
    r2c(sl.out[2], Nz);
  }
  {
    float2 W[G];
    c2r(6, W);  // omega_z
#pragma unroll
    for (int m = 0; m < G; ++m) {
      Nx[m] = __ffma2_rn(pk(1, m), W[m], Nx[m]);
      Ny[m] = __ffma2_rn(neg(pk(0, m)), W[m], Ny[m]);
    }
  }
  r2c(sl.out[0], Nx);
  r2c(sl.out[1], Ny);
#pragma unroll 1
  for (int i = 0; i < 3; ++i) {
    float2 P[G];
#pragma unroll
    for (int m = 0; m < G; ++m) P[m] = __fmul2_rn(pk(i, m), pk(3, m));
    r2c(sl.out[3 + i], P);
  }
}

// ---- forward x pass with the update (periodic cube) ------------------------
// As the Navier-Stokes forward x pass (ns_fwdx.cuh), with six fields and three
// parked arrays: the divergence k . F(u theta), then n_x and n_y.  k_y and k_z
// are constant along a line, so k_y u_y theta + k_z u_z theta is formed before
// its transform: five transforms for six fields.  512^3, per launch: forward x pass 528 us and
// update 922 us as kernels of their own, 1135 us fused (1607 us with all its L2
// prefetches at the start instead of one field ahead, 1351 us with radices 8, 8,
// 8 on 1024 threads instead of 32, 16 on 256), 1088 us with padded rows for the
// stage state and the accumulator, 1052 us with the loads of four modes in
// flight in the update, 1014 us with five transforms (256^3 126 -> 119 us, 384^3
// 388 -> 363 us).  Its six fields and eighteen kept arrays would take 632
// us: eight warps do not cover the loads of each field and the exchanges.
// Two stages at n = 512 and 1024 (step at 1024^3, RK2 / RK4: 97.8 / 205.3 ->
// 91.7 / 192.2 ms).  Not at 256, where 16 values on 128 registers spill up to 268
// bytes (RK4 2345 -> 2403 us), nor at 768, where three parked fields leave room
// for eight columns and so for four warps (74.9 -> 74.3 ms, below 1 %).
template <int N>
struct RUCfg {
  static constexpr bool TWO = N == 512 || N == 1024;  // radix 32, then 16 or 32
  static constexpr int G = TWO ? 32 : (N % 3 == 0 ? elems_per_thread(N) : NFCfg<N>::G);
  static constexpr int S = N / G;
  static constexpr int T = N == 512 ? 16 : (N >= 768 ? 8 : (N % 3 == 0 ? 16 : NFCfg<N>::T));
  static constexpr int THREADS = T * S;
  static constexpr int KD = (N - 1) / 3;
  static constexpr int LOW = KD / S + 1;
  static constexpr int HIGH = (N - KD) / S > LOW ? (N - KD) / S : LOW;
  static constexpr int SLOTS = LOW + G - HIGH;
  using X = XTransform<N, G, -1, T, TWO>;
  static constexpr size_t SMEM = sizeof(float2) * (X::WORDS + 3 * (size_t)SLOTS * THREADS);
  static constexpr int MINB = THREADS >= 512 ? 1 : (THREADS == 256 ? (N == 768 || TWO ? 1 : 2) : 4);
  // modes whose loads are in flight together (four at 3 * 2^m spill, 384^3 422 us
  // against 388 with two and 405 with one)
  static constexpr int GROUP = N % 3 == 0 ? 2 : 4;
  __host__ __device__ static constexpr bool parked(int m) { return m < LOW || m >= HIGH; }
  __host__ __device__ static constexpr int slot(int m) { return m < LOW ? m : m - HIGH + LOW; }
};

template <int N, int MODE>
__global__ void __launch_bounds__(RUCfg<N>::THREADS, RUCfg<N>::MINB)
    k_rbc_fwdx(const float2* __restrict__ w, const float2* x, const float2* u0, const float2* s1, float2* acc,
               float2* out, int ktiles, RBCUpdate upd, float scale, const float2* __restrict__ tw,
               const float2* __restrict__ t3) {
  pdl_wait();
  constexpr long long H1 = N / 2 + 1, MM = (long long)N * N * H1;  // geometry of the n^3 grid
  constexpr long long HW = ns_row(N), MW = (long long)N * N * HW;  // the padded workspace
  constexpr int KD = (N - 1) / 3;
  constexpr bool A0 = MODE != NS_RHS && MODE != NS_RK4_4;             // reads the step's state
  constexpr bool B0 = MODE == NS_STAGE2 || MODE >= NS_RK4_2;           // reads the stage state or the accumulator
  using C = RUCfg<N>;
  constexpr int G = C::G, S = C::S, T = C::T;
  extern __shared__ float2 smn[];
  const int c = threadIdx.x % T, j = threadIdx.x / T;
  const int dky = blockIdx.x / ktiles;
  const int ay = dense_to_a(dky, N, KD);
  const int kz = (blockIdx.x - dky * ktiles) * T + c;
  const bool valid = kz < (KD + 1);
  const long long q = (long long)ay * H1 + kz, rs = (long long)N * H1;
  const long long qw = (long long)ay * HW + kz, rw = (long long)N * HW;
  float2* park = smn + C::X::WORDS + threadIdx.x;
  C::X::init(smn, tw, t3);
  const int ky = kwav(ay, N);
  const float2* bsrc = MODE == NS_STAGE2 ? s1 : acc;
  // the caller's state has rows of n/2 + 1, the stage state and the accumulator
  // padded ones: entry (row pos, this column) of a field
  constexpr bool XP = MODE == NS_STAGE2 || MODE >= NS_RK4_2;                        // x
  constexpr bool OP = MODE == NS_STAGE1 || (MODE >= NS_RK4_1 && MODE != NS_RK4_4);  // out
  constexpr long long XM = XP ? MW : MM, OM = OP ? MW : MM;
  float2 V[G];
#pragma unroll 1
  for (int i = 0; i < 5; ++i) {
    // u_x theta, k_y u_y theta + k_z u_z theta, then n
    const int f = i < 2 ? 3 + i : i - 2;
#pragma unroll
    for (int m = 0; m < G; ++m)
      V[m] = valid ? w[f * MW + (j + m * S) * rw + qw] : make_float2(0.f, 0.f);
    if (i == 1) {
#pragma unroll
      for (int m = 0; m < G; ++m) {
        const float2 t = valid ? w[5 * MW + (j + m * S) * rw + qw] : make_float2(0.f, 0.f);
        V[m] = make_float2(fmaf((float)kz, t.x, (float)ky * V[m].x), fmaf((float)kz, t.y, (float)ky * V[m].y));
      }
    }
    if constexpr (N >= 256) {  // the next field, and at last the update's reads, go to L2 meanwhile (see k_ns_fwdx)
      if (i < 4) {
        const int nf = i == 0 ? 4 : i - 1;
        for (int r = threadIdx.x; r < N; r += C::THREADS) {
          prefetch_l2(w + nf * MW + r * rw + qw - c);
          if (i == 0) prefetch_l2(w + 5 * MW + r * rw + qw - c);
        }
      }
      if (i == 3 || i == 4)
        for (int r = threadIdx.x; r < 2 * KD + 1; r += C::THREADS) {
          const long long o = dense_to_a(r, N, KD) * rs + q - c, ow = dense_to_a(r, N, KD) * rw + qw - c;
          if (i == 3) {
            prefetch_l2(x + 2 * XM + (XP ? ow : o));
            prefetch_l2(x + 3 * XM + (XP ? ow : o));
          }
#pragma unroll
          for (int f2 = 0; f2 < 4; ++f2) {
            if (A0 && i == 3) prefetch_l2(u0 + f2 * MM + o);
            if (B0 && i == 4) prefetch_l2(bsrc + f2 * MW + ow);
          }
        }
    }
    C::X::run(V, j, c, smn, tw, t3);
    if (i < 2) {
#pragma unroll
      for (int m = 0; m < G; ++m)
        if (C::parked(m)) {
          float2& d = park[C::slot(m) * C::THREADS];
          const float2 v = cscale(V[m], scale);
          d = i == 0 ? cscale(v, (float)kwav(j + m * S, N)) : cadd(d, v);
        }
    } else if (i < 4) {
#pragma unroll
      for (int m = 0; m < G; ++m)
        if (C::parked(m)) park[((i - 1) * C::SLOTS + C::slot(m)) * C::THREADS] = V[m];
    }
  }
  if (!valid) return;
  const float fky = (float)ky, fkz = (float)kz, dt = upd.dt;
  // out may be x or u0, which orders loads after stores: the loads of GROUP
  // modes come before their first store
  constexpr int NG = C::GROUP;
  static_assert(G % NG == 0, "groups of modes");
  float2 ga[NG][4], gb[NG][4], gx[NG][2], gE[NG][2], gH[NG][2];
#pragma unroll
  for (int m = 0; m < G; ++m) {
    if (m % NG == 0) {
#pragma unroll
      for (int i = 0; i < NG; ++i) {
        const int pos = j + (m + i) * S;
        if (!C::parked(m + i) || !kept_xy(pos, N, KD)) continue;
        const long long idx = pos * rs + q, idw = pos * rw + qw;
        const int kx = kwav(pos, N), k2 = kx * kx + ky * ky + kz * kz;
        gx[i][0] = x[(XP ? idw : idx) + 2 * XM];
        gx[i][1] = x[(XP ? idw : idx) + 3 * XM];
#pragma unroll
        for (int f = 0; f < 4; ++f) {
          if (A0) ga[i][f] = u0[idx + f * MM];
          if (B0) gb[i][f] = bsrc[idw + f * MW];
        }
#pragma unroll
        for (int t = 0; t < 2; ++t) {
          if (MODE != NS_RHS && MODE != NS_RK4_4) gE[i][t] = __ldg(&upd.tab[t * upd.tab_len + k2]);
          if (MODE >= NS_RK4_1 && MODE != NS_RK4_4) gH[i][t] = __ldg(&upd.tab[(2 + t) * upd.tab_len + k2]);
        }
      }
    }
    const int pos = j + m * S, gi = m % NG;
    if (!C::parked(m) || !kept_xy(pos, N, KD)) continue;
    const long long idx = pos * rs + q, idw = pos * rw + qw;
    const int kx = kwav(pos, N), k2 = kx * kx + ky * ky + kz * kz;
    const float2 uz = gx[gi][0], th = gx[gi][1];
    const float2 *a = ga[gi], *b = gb[gi], *E = gE[gi], *H = gH[gi];
    const float2 dv = park[C::slot(m) * C::THREADS];
    float2 px = cscale(park[(C::SLOTS + C::slot(m)) * C::THREADS], scale);
    float2 py = cscale(park[(2 * C::SLOTS + C::slot(m)) * C::THREADS], scale);
    float2 pz = cadd(cscale(V[m], scale), th);  // n + theta z, then the projection
    float2 nv[4];
    if (k2 == 0) {
      nv[0] = nv[1] = nv[2] = nv[3] = make_float2(0.f, 0.f);
    } else {
      const float fkx = (float)kx, inv = 1.f / (float)k2;
      const float2 kn = make_float2((fkx * px.x + fky * py.x + fkz * pz.x) * inv,
                                    (fkx * px.y + fky * py.y + fkz * pz.y) * inv);
      nv[0] = csub(px, cscale(kn, fkx));
      nv[1] = csub(py, cscale(kn, fky));
      nv[2] = csub(pz, cscale(kn, fkz));
      nv[3] = make_float2(dv.y + uz.x, -dv.x + uz.y);  // -i k . F(u theta) + u_z
    }
#pragma unroll
    for (int f = 0; f < 4; ++f)
      rbc_entry_store<MODE>((OP ? idw : idx) + f * OM, idw + f * MW, nv[f], a[f], b[f], E[f == 3 ? 1 : 0],
                            H[f == 3 ? 1 : 0], dt, acc, out);
  }
}

// ------------------------------------------------------------ launchers ----
template <int N, bool PADDED>
static cudaError_t rbc_invx_np(fftk_plan p, const float2* x, float2* w, cudaStream_t st) {
  using I = NICfg<N>;
  static PerDevice once;
  const cudaError_t e = once.run([](int) {
    return cudaFuncSetAttribute(k_ns_invx<N, true, PADDED>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)I::SMEM);
  });
  if (e != cudaSuccess) return e;
  constexpr int KD = (N - 1) / 3, KT = (KD + I::T) / I::T;
  LaunchScope ls(p, KK_X_INV, st);
  launch_pdl(k_ns_invx<N, true, PADDED>, (2 * KD + 1) * KT, I::THREADS, I::SMEM, st, x, w, KT,
             twiddles(p, 1 << Log2<N>::value), p->d_tw3);
  return cudaGetLastError();
}

template <int N>
static cudaError_t rbc_invx_n(fftk_plan p, const float2* x, bool padded, float2* w, cudaStream_t st) {
  return padded ? rbc_invx_np<N, true>(p, x, w, st) : rbc_invx_np<N, false>(p, x, w, st);
}

template <int N>
static cudaError_t rbc_z_n(fftk_plan p, float2* w, const RBCSlots& sl, cudaStream_t st) {
  using C = RZCfg<N>;
  static PerDevice once;
  const cudaError_t e = once.run([](int) {
    return cudaFuncSetAttribute(k_rbc_z<N>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)C::SMEM);
  });
  if (e != cudaSuccess) return e;
  const long long lines = (long long)N * N;
  LaunchScope ls(p, KK_RBC_Z, st);
  launch_pdl(k_rbc_z<N>, (unsigned)((lines + C::LPC - 1) / C::LPC), C::THREADS, C::SMEM, st, w, sl, twiddles(p,
             1 << Log2<N>::value), p->d_tw3, p->d_err);
  return cudaGetLastError();
}

template <int N, int MODE>
static cudaError_t rbc_fwdx_nm(fftk_plan p, const RBCStage& s, cudaStream_t st) {
  using U = RUCfg<N>;
  static PerDevice once;
  const cudaError_t e = once.run([](int) {
    return cudaFuncSetAttribute(k_rbc_fwdx<N, MODE>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)U::SMEM);
  });
  if (e != cudaSuccess) return e;
  constexpr int KD = (N - 1) / 3, KT = (KD + U::T) / U::T;
  LaunchScope ls(p, KK_RBC_UPDATE, st);
  launch_pdl(k_rbc_fwdx<N, MODE>, (2 * KD + 1) * KT, U::THREADS, U::SMEM, st, s.w, s.x, s.u0, s.s1, s.acc, s.out, KT,
             s.upd,
                                                                   s.scale, twiddles(p, 1 << Log2<N>::value),
                                                                   p->d_tw3);
  return cudaGetLastError();
}
template <int N>
static cudaError_t rbc_fwdx_n(fftk_plan p, const RBCStage& s, cudaStream_t st) {
  switch (s.mode) {
#define MODE(m) \
  case m:       \
    return rbc_fwdx_nm<N, m>(p, s, st);
    MODE(NS_RHS) MODE(NS_STAGE1) MODE(NS_STAGE2) MODE(NS_RK4_1) MODE(NS_RK4_2) MODE(NS_RK4_3) MODE(NS_RK4_4)
#undef MODE
  }
  return cudaErrorInvalidValue;
}

}  // namespace fftk
