// The fused passes of the Navier-Stokes right-hand side (ns.cu describes the
// method), as templates on the grid size: instantiated for powers of two in
// ns.cu and for 3 * 2^m in ns_radix3.cu.
#pragma once

#include "fft_engine.cuh"
#include "internal.h"
#include "ns_common.cuh"
#include "ns_update.cuh"
#include "tcgen05.cuh"

namespace fftk {
// ------------------------------------------------------------ x/y config ---
// Single-field passes (both y passes): the strided FFT pass configuration,
// 16 k_z columns per tile (128-byte row segments); powers of two: 16 values
// per thread, 32 warps per SM at <= 64 registers; 3 * 2^m: 24 values, 128
// registers.
template <int N>
struct NXCfg {
  static constexpr int G = elems_per_thread(N);
  static constexpr int S = N / G;
  static constexpr int T = S <= 16 ? 16 : (S <= 64 ? 16 : 1024 / S);
  static constexpr int THREADS = T * S;
  static constexpr int MINB = N % 3 == 0 ? (THREADS <= 128 ? 4 : (THREADS <= 256 ? 2 : 1))
                                         : (THREADS <= 512 ? (THREADS <= 256 ? 4 : 2) : 1);
  static constexpr size_t SMEM = sizeof(float2) * (size_t)N * T;
};

// 2./4. y pass, columns (x, k_z < kc), blockIdx -> (field, x, k_z tile).
//    SIGN=+1: only kept k_y rows are read, every y row is written;
//    SIGN=-1: every y row is read, only kept k_y rows are written.
template <int N, int SIGN>
__global__ void __launch_bounds__(NXCfg<N>::THREADS, NXCfg<N>::MINB)
    k_ns_ypass(const float2* w, float2* wo, int ktiles, const float2* __restrict__ tw,
               const float2* __restrict__ t3) {  // wo may be w
  pdl_wait();
  constexpr long long H1 = ns_row(N), MM = (long long)N * N * H1;  // the padded workspace
  constexpr int KD = (N - 1) / 3;                                  // largest kept |k| (2/3 rule)
  using C = NXCfg<N>;
  constexpr int G = C::G, S = C::S, T = C::T;
  extern __shared__ float2 smn[];
  const int c = threadIdx.x % T, j = threadIdx.x / T;
  const int kt = blockIdx.x % ktiles;
  const int rest = blockIdx.x / ktiles;
  const int x = rest % N;
  const int f = rest / N;
  const int kz = kt * T + c;
  const bool valid = kz < (KD + 1);
  const long long off = f * MM + (long long)x * N * H1 + kz;
  float2 v[G];
#pragma unroll
  for (int m = 0; m < G; ++m) {
    const int pos = j + m * S;
    const bool rd = valid && (SIGN < 0 || kept_xy(pos, N, KD));
    v[m] = rd ? w[off + (long long)pos * H1] : make_float2(0.f, 0.f);
  }
  fft_line<N, G, SIGN>(v, j, ColX<T>{smn, c}, tw, t3);
  if (valid) {
#pragma unroll
    for (int m = 0; m < G; ++m) {
      const int pos = j + m * S;
      if (SIGN > 0 || kept_xy(pos, N, KD)) wo[off + (long long)pos * H1] = v[m];
    }
  }
}

// Inverse x pass.  Powers of two hold two fields at once, 16 values per thread
// for n >= 512 with 16 columns per tile (128-byte row segments) at n = 512 and
// 8 at n = 1024.  3 * 2^m lines (24 values per thread, 16 columns) hold one
// and park the other in shared memory.
template <int N>
struct NICfg {
  static constexpr bool PARK = N % 3 == 0;
  static constexpr int G = PARK ? elems_per_thread(N) : (N >= 512 ? 16 : NFCfg<N>::G);
  static constexpr int S = N / G;
  static constexpr int T = PARK || N == 512 ? 16 : (N == 1024 ? 8 : NFCfg<N>::T);
  static constexpr int THREADS = T * S;
  static constexpr int MINB = PARK ? (THREADS <= 128 ? 4 : (THREADS <= 256 ? 2 : 1)) : (THREADS <= 256 ? 2 : 1);
  using X = XTransform<N, G, +1, T, false>;
  static constexpr size_t SMEM = sizeof(float2) * (X::WORDS + (PARK ? (size_t)N * T : 0));
};

// 1. inverse x pass with the curl.  Columns: kept (k_y, k_z); rows: k_x.
//    U_c = F^-1_x(u_c), D_c = F^-1_x(i k_x u_c), then
//    omega_x = i (k_y U_z - k_z U_y), omega_y = i k_z U_x - D_z,
//    omega_z = D_y - i k_y U_x   (five transforms instead of six).
//    Output field order: u_x, u_y, u_z, omega_x, omega_y, omega_z.
//    THETA (convection): field 3 of u, the temperature, goes to field 6 of w.
//    PADDED: u has the padded rows of the stage states.
template <int N, bool THETA = false, bool PADDED = false>
__global__ void __launch_bounds__(NICfg<N>::THREADS, NICfg<N>::MINB)
    k_ns_invx(const float2* __restrict__ u, float2* __restrict__ w, int ktiles, const float2* __restrict__ tw,
              const float2* __restrict__ t3) {
  pdl_wait();
  constexpr long long HW = ns_row(N), MW = (long long)N * N * HW;  // the padded workspace
  constexpr long long H1 = PADDED ? HW : N / 2 + 1, MM = (long long)N * N * H1;  // u
  constexpr int KD = (N - 1) / 3;                                  // largest kept |k| (2/3 rule)
  using C = NICfg<N>;
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
  const float ky = (float)kwav(ay, N), kzf = (float)kz;
  auto load = [&](int f, float2(&v)[G], bool ikx) {
#pragma unroll
    for (int m = 0; m < G; ++m) {
      const int pos = j + m * S;
      float2 a = make_float2(0.f, 0.f);
      if (valid && kept_xy(pos, N, KD)) a = u[f * MM + pos * rs + q];
      v[m] = ikx ? mul_i(a, (float)kwav(pos, N)) : a;
    }
  };
  auto store = [&](int f, const float2(&v)[G]) {
    if (valid) {
#pragma unroll
      for (int m = 0; m < G; ++m) w[f * MW + (j + m * S) * rw + qw] = v[m];
    }
  };
  if constexpr (C::PARK) {
    float2* park = smn + C::X::WORDS + threadIdx.x;  // this thread's slots
    C::X::init(smn, tw, t3);
    float2 a[G];
    load(0, a, false);
    C::X::run(a, j, c, smn, tw, t3);  // U_x
    store(0, a);
#pragma unroll
    for (int m = 0; m < G; ++m) park[m * C::THREADS] = a[m];
    load(1, a, true);
    C::X::run(a, j, c, smn, tw, t3);  // D_y
#pragma unroll
    for (int m = 0; m < G; ++m) a[m] = csub(a[m], mul_i(park[m * C::THREADS], ky));  // omega_z
    store(5, a);
    load(2, a, true);
    C::X::run(a, j, c, smn, tw, t3);  // D_z
#pragma unroll
    for (int m = 0; m < G; ++m) a[m] = csub(mul_i(park[m * C::THREADS], kzf), a[m]);  // omega_y
    store(4, a);
    load(1, a, false);
    C::X::run(a, j, c, smn, tw, t3);  // U_y
    store(1, a);
#pragma unroll
    for (int m = 0; m < G; ++m) park[m * C::THREADS] = a[m];
    load(2, a, false);
    C::X::run(a, j, c, smn, tw, t3);  // U_z
    store(2, a);
#pragma unroll
    for (int m = 0; m < G; ++m) {
      const float2 y = park[m * C::THREADS];
      a[m] = make_float2(-(ky * a[m].y - kzf * y.y), ky * a[m].x - kzf * y.x);  // omega_x
    }
    store(3, a);
    if constexpr (THETA) {
      load(3, a, false);
      C::X::run(a, j, c, smn, tw, t3);
      store(6, a);
    }
  } else {
    float2 a[G], b[G];
    load(1, a, true);
    C::X::run(a, j, c, smn, tw, t3);  // D_y
    load(0, b, false);
    C::X::run(b, j, c, smn, tw, t3);  // U_x
    store(0, b);
  #pragma unroll
    for (int m = 0; m < G; ++m) a[m] = csub(a[m], mul_i(b[m], ky));  // omega_z
    store(5, a);
    load(2, a, true);
    C::X::run(a, j, c, smn, tw, t3);  // D_z
  #pragma unroll
    for (int m = 0; m < G; ++m) a[m] = csub(mul_i(b[m], kzf), a[m]);  // omega_y
    store(4, a);
    load(1, a, false);
    C::X::run(a, j, c, smn, tw, t3);  // U_y
    store(1, a);
    load(2, b, false);
    C::X::run(b, j, c, smn, tw, t3);  // U_z
    store(2, b);
  #pragma unroll
    for (int m = 0; m < G; ++m)
      b[m] = make_float2(-(ky * b[m].y - kzf * a[m].y), ky * b[m].x - kzf * a[m].x);  // omega_x
    store(3, b);
    if constexpr (THETA) {
      load(3, a, false);
      C::X::run(a, j, c, smn, tw, t3);
      store(6, a);
    }
  }
}

// ------------------------------------------------------------- z product ---
// The z kernel holds a 256-point line (n = 512) as 16 values per thread on 16
// threads, two lines per warp: each transform is two radix-16 stages with one
// exchange through shared memory (8 values per thread would need three stages
// and two exchanges, and the exchanges dominated the L1 traffic).  A thread
// holds up to four such arrays (u x omega accumulators and a vorticity
// component), 230 registers at n = 512: two CTAs of 128 threads per SM.
// Small grids have few lines: below n = 512 a line goes to more threads with
// fewer values (8 at 128 and 256, 4 below), which fills the chip (per RK2 step,
// 16 values -> these: 32^3 82 -> 53 us, 64^3 101 -> 62 us, 128^3 180 -> 139 us,
// 256^3 929 -> 843 us).
// 3 * 2^m lines: 12 values per thread, at n = 768 24 (radices 8, 8, 6 instead of
// 4, 4, 4, 6) with one staging buffer, so that two CTAs fit: 5.95 -> 4.85 ms
// per launch (at 384 and 192 with 24: 3.06 against 3.03 ms, 514 against 479 us
// per step).
// Measured and dropped: three CTAs per SM with one staging buffer (168
// registers, 1.120 against 1.126 ms), CTAs of 64 or 32 threads with five or
// ten per SM (spills; 1.20 ms), the velocity parked in TMEM (slower).
template <int N, int MIN24 = 768>  // MIN24: 3 * 2^m lines from here on hold 24 values per thread
struct NZCfg {
  static constexpr int H = N / 2;
  static constexpr int HB = line_slots(H);        // exchange slots per line
  static constexpr int G = N % 3 == 0 ? (N >= MIN24 ? 24 : (H >= 48 ? 12 : 6))
                                      : (N >= 512 ? 16 : (N >= 128 ? 8 : (H < 4 ? H : 4)));
  static constexpr int S = H / G;
  static constexpr int LPC = S >= 128 ? 1 : 128 / S;
  static constexpr int NBUF = G == 24 ? 1 : 2;    // staging buffers per line
  static constexpr int THREADS = LPC * S;
  static constexpr bool WARP = S <= 32;
  static constexpr int KC = (N - 1) / 3 + 1;      // kept k_z count (2/3 rule)
  static constexpr int KCP = (KC + 2) & ~1;       // staged values per line and buffer (KC + alignment slack)
  static constexpr size_t FIELDS = sizeof(float2) * (size_t)LPC * (HB + 3 * H);  // exchange + 3 parked fields
  static constexpr size_t STAGE = sizeof(float2) * (size_t)LPC * NBUF * KCP;  // staging buffers
  static constexpr size_t SMEM = FIELDS + STAGE + sizeof(uint64_t) * NBUF * LPC;  // + one mbarrier per buffer
  static constexpr int MINB = G == 16 || G == 24 ? 2 : (G == 12 || N == 256 ? 3 : 4);  // CTAs per SM
};

// 3. per (x, y) line: the six c2r transforms, the product n = u x omega and
//    the three r2c transforms.  Reads k_z < kc of fields 0..5 of w, writes
//    k_z < kc of fields 0..2 of wo (wo may be w: a line is fully read before
//    it is written).
//    The three velocity components are parked in real space in shared memory;
//    each vorticity component is then transformed and folded into the
//    accumulators of n, so at most 4 fields are held in registers.
//    A line's kept coefficients of each input field arrive by one bulk
//    asynchronous copy into one of two staging buffers, issued two fields
//    ahead of their use, so the global loads' latency overlaps the transforms
//    of the field before; the c2r reads X[k] and its mirror X[H - k] from there.
template <int N, int HW>  // HW: row length of the workspace (n/2 + 1, or the fused path's padded rows)
__global__ void __launch_bounds__(NZCfg<N>::THREADS, NZCfg<N>::MINB)
    k_ns_z(const float2* w, float2* wo, const float2* __restrict__ tw, const float2* __restrict__ t3, int* err) {
  pdl_wait();
  constexpr long long H1 = HW, MM = (long long)N * N * H1;  // geometry of the workspace
  using C = NZCfg<N>;
  constexpr int H = C::H, G = C::G, S = C::S;
  constexpr int LOGN = Log2<N>::value;
  constexpr int KC = C::KC;  // kept k_z count
  extern __shared__ __align__(16) float2 smz[];
  const int li = threadIdx.x / S, j = threadIdx.x % S;
  const long long line = (long long)blockIdx.x * C::LPC + li;
  const bool valid = line < (long long)N * N;
  // (dft3 with multiply-adds would spill 24 bytes at 96 points: step 64.7 -> 67.5 us)
  const LineX<C::WARP, S, G, (N % 3 == 0 && G == 12)> xc{smz + li * C::HB, line_xor<S>(li)};
  float2* park = smz + C::LPC * C::HB + li * 3 * H + j;  // [3][G][S] per line, this thread's column
  constexpr int NB = C::NBUF;
  float2* stage = smz + C::FIELDS / sizeof(float2) + li * NB * C::KCP;  // this line's buffers
  uint64_t* bar = reinterpret_cast<uint64_t*>(smz + (C::FIELDS + C::STAGE) / sizeof(float2)) + NB * li;

  // Field f's element k of this line sits at element f MM + line H1 + k.  MM
  // is even; with H1 odd (rows of n/2 + 1) the line starts 16-byte aligned for
  // even lines and 8 bytes past a 16-byte boundary for odd ones: the copy then
  // starts `lead` elements early (the previous line's last value, k_z = n/2,
  // which this kernel never writes) and ends at k_z <= kc, inside the line.
  // With padded rows (H1 a multiple of 16) every line is aligned.
  const int lead = (int)((line * H1) & 1);
  const uint32_t bytes = (uint32_t)(sizeof(float2) * ((KC + lead + 1) & ~1));
  auto issue = [&](int f) {  // one thread of the line; buffer f % NB was last read NB fields ago
    uint64_t* b = bar + f % NB;
    tcg::fence_smem_async();
    tcg::mbar_expect(b, bytes);
    tcg::bulk_g2s(stage + (f % NB) * C::KCP, w + f * MM + line * H1 - lead, bytes, b);
  };
  bool ok = true;
  auto arrive = [&](int f) {  // wait for field f's copy (bounded; an expired wait is reported)
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

  // inverse z transform of field f (half-complex -> N real points, two per slot)
  auto c2r = [&](int f, float2 (&U)[G]) {
    const float2* src = stage + (f % NB) * C::KCP + lead;
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
    // every thread of the line has passed an exchange barrier since it read
    // the buffer: refill it with field f + NB
    if (f + NB < 6 && j == 0 && valid) issue(f + NB);
  };

  {
    float2 U[G];
#pragma unroll 1
    for (int f = 0; f < 3; ++f) {
      c2r(f, U);
#pragma unroll
      for (int m = 0; m < G; ++m) park[(f * G + m) * S] = U[m];
    }
  }
  // forward z transforms of n (N real points -> half-complex), k_z < kc written
  auto r2c = [&](int f, float2 (&U)[G]) {
    fft_line<H, G, -1, LOGN>(U, j, xc, tw, t3);
#pragma unroll
    for (int m = 0; m < G; ++m) xc.st_run(j + m * S, U[m]);
    xc.sync();
    float2* dst = wo + f * MM + line * H1;
#pragma unroll
    for (int m = 0; m < G; ++m) {
      const int k = j + m * S;
      const float2 A = U[m];
      const float2 Bc = cconj(xc.ld_run(mirror<H>(k)));
      const float2 E = cscale(cadd(A, Bc), 0.5f);
      const float2 D = csub(A, Bc);
      const float2 O = make_float2(0.5f * D.y, -0.5f * D.x);
      if (valid && k < KC) dst[k] = cadd(E, cmul(twk(m), O));
    }
    xc.sync();
  };
  // n = u x omega at the two real points held by each slot (elementwise
  // products of the (even, odd) point pairs, paired FP32 instructions):
  //   n_x = u_y w_z - u_z w_y,  n_y = u_z w_x - u_x w_z,  n_z = u_x w_y - u_y w_x
  // n_z is complete after omega_y and is transformed before omega_z is loaded.
  auto neg = [](float2 a) { return make_float2(-a.x, -a.y); };
  float2 Ny[G], Nx[G];
  {
    float2 Nz[G];
    {
      float2 W[G];
      c2r(3, W);  // omega_x
#pragma unroll
      for (int m = 0; m < G; ++m) {
        const float2 uy = park[(1 * G + m) * S], uz = park[(2 * G + m) * S];
        Ny[m] = __fmul2_rn(uz, W[m]);
        Nz[m] = __fmul2_rn(neg(uy), W[m]);
      }
      c2r(4, W);  // omega_y
#pragma unroll
      for (int m = 0; m < G; ++m) {
        const float2 ux = park[(0 * G + m) * S], uz = park[(2 * G + m) * S];
        Nx[m] = __fmul2_rn(neg(uz), W[m]);
        Nz[m] = __ffma2_rn(ux, W[m], Nz[m]);
      }
    }
    r2c(2, Nz);
  }
  {
    float2 W[G];
    c2r(5, W);  // omega_z
#pragma unroll
    for (int m = 0; m < G; ++m) {
      const float2 ux = park[(0 * G + m) * S], uy = park[(1 * G + m) * S];
      Nx[m] = __ffma2_rn(uy, W[m], Nx[m]);
      Ny[m] = __ffma2_rn(neg(ux), W[m], Ny[m]);
    }
  }
  r2c(0, Nx);
  r2c(1, Ny);
}

// y pass of `fields` fields on padded rows (ns_ypass.cu): sign +1 reads the kept
// rows and writes every row, -1 reads every row and writes the kept ones; out
// may be in.
cudaError_t ns_ypass(fftk_plan p, const float2* in, float2* out, int fields, int sign, int kind, cudaStream_t st);

// One right-hand side and update on a cube of 3 * 2^m points (ns_radix3.cu).
cudaError_t ns_rhs_radix3(fftk_plan p, const float2* u, const float2* u0, const float2* u1, float2* out,
                          const NSUpdate& upd, int mode, const float2* extra, cudaStream_t st);

// --------------------------------------------------------------- launchers --
template <int N>
struct NSLaunch {
  static cudaError_t attrs() {
    static PerDevice once;
    return once.run([](int) {
      cudaError_t err = cudaFuncSetAttribute(k_ns_invx<N>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             (int)NICfg<N>::SMEM);
      if (err == cudaSuccess)
        err = cudaFuncSetAttribute(k_ns_z<N, (int)ns_row(N)>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                   (int)NZCfg<N>::SMEM);
      if constexpr (N % 3 != 0)
        if (err == cudaSuccess)
          err = cudaFuncSetAttribute(k_ns_z<N, N / 2 + 1>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                     (int)NZCfg<N>::SMEM);
      return err;
    });
  }

  // The fused z pass alone (c2r of the six fields in s->w, u x omega, r2c of
  // n into fields 0..2), for the split-precision right-hand side.
  static cudaError_t z(fftk_plan p, cudaStream_t st) {
    using Z = NZCfg<N>;
    cudaError_t e = attrs();
    if (e != cudaSuccess) return e;
    NSWork* s = p->ns;
    LaunchScope ls(p, KK_NS_Z, st);
    const long long lines = (long long)N * N;
    launch_pdl(k_ns_z<N, N / 2 + 1>, (unsigned)((lines + Z::LPC - 1) / Z::LPC), Z::THREADS, Z::SMEM, st, s->w, s->w,
               twiddles(p, N), nullptr, p->d_err);
    return cudaGetLastError();
  }

  // One evaluation of N(u) followed by the update selected by `mode`.
  static cudaError_t rhs(fftk_plan p, const float2* u, const float2* u0, const float2* u1,
                         float2* out, const NSUpdate& upd, int mode, const float2* extra,
                         cudaStream_t st) {
    using Z = NZCfg<N>;
    cudaError_t e = attrs();
    if (e != cudaSuccess) return e;
    NSWork* s = p->ns;
    const NSGeom g = s->g;
    using I = NICfg<N>;
    const int ki = (g.kc + I::T - 1) / I::T;
    // invx u -> A, inverse y A -> B, z B -> A (fields 0..2), forward y A -> A,
    // forward x A -> out.  The inverse y pass out of place measured 0.684 ->
    // 0.647 ms at 512^3; the forward y pass, which writes only the kept rows,
    // measured slower out of place (0.313 -> 0.331 ms), so it stays in place.
    e = ns_second_workspace(p);
    if (e != cudaSuccess) return e;
    float2* A = s->w;
    float2* Bw = s->w2;
    const float2* tw = twiddles(p, 1 << Log2<N>::value);
    const float2* t3 = p->d_tw3;
    {
      LaunchScope ls(p, KK_NS_INVX, st);
      launch_pdl(k_ns_invx<N>, g.nk * ki, I::THREADS, I::SMEM, st, u, A, ki, tw, t3);
    }
    e = ns_ypass(p, A, Bw, 6, +1, KK_NS_INVY, st);
    if (e != cudaSuccess) return e;
    {
      LaunchScope ls(p, KK_NS_Z, st);
      const long long lines = (long long)N * N;
      launch_pdl(k_ns_z<N, (int)ns_row(N)>, (unsigned)((lines + Z::LPC - 1) / Z::LPC), Z::THREADS, Z::SMEM, st, Bw, A,
                 tw, t3, p->d_err);
    }
    e = cudaGetLastError();
    if (e == cudaSuccess) e = ns_ypass(p, A, A, 3, -1, KK_NS_FWDY, st);
    return e == cudaSuccess ? ns_fwdx(p, A, u0, u1, out, upd, mode, extra, st) : e;
  }
};

}  // namespace fftk
