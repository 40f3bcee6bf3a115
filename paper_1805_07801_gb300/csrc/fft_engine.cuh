// Device-side 1D FFT engine shared by every pass kernel.
//
// A line of length L (a power of two, or three times one) is held by S = L/G
// threads, G complex values per thread in the "natural" pattern
// v[m] = x[j + m*S] (j = thread index within the line).  The transform is a
// sequence of self-sorting (Stockham) radix-R stages (stage_radix): every
// thread runs G/R radix-R butterflies in registers, and consecutive stages
// exchange data through a shared-memory buffer.  Lines of 3 * 2^m points take
// their factor 3 in the last stage, as a radix-3, 6, 12 or 24 butterfly, so
// every stage before it spans a power of two.  After the last stage the output is
// again in the natural pattern, so a pass can load and store global memory
// directly from registers with the same coalesced pattern.
//
// This replaces the FFTW 1D line transforms used by FFTK (paper Sec. 3);
// the factorisation is fixed at compile time by Stage below.
//
// Sign convention: SIGN = -1 computes X[k] = sum_n x[n] exp(-2 pi i n k / L)
// (forward), SIGN = +1 the unnormalised inverse.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

// Complex sums and real scalings use the paired FP32 instructions of sm_100
// and later (two correctly rounded operations per instruction: the results
// are those of the scalar operations).  They cut the instruction count of
// the issue-bound kernels (the fused Navier-Stokes passes); a translation
// unit whose kernels are bound by their global accesses instead (the plain
// strided passes, measured slower with them) defines FFTK_PAIRED_FP32 as 0
// before including this header.  2: the rotations by constants take one too
// (the fused passes of powers of two: without it the 512-point inverse x pass
// spills 8 bytes; the sine/cosine passes and the shell transfer run 1 to 7 %
// slower with it).  The engine lives in an inline namespace named after the
// choice, so the forms never meet at link time.
#ifndef FFTK_PAIRED_FP32
#define FFTK_PAIRED_FP32 1
#endif

namespace fftk {
#if FFTK_PAIRED_FP32 == 2
inline namespace paired_rot_fp32 {
#elif FFTK_PAIRED_FP32
inline namespace paired_fp32 {
#else
inline namespace scalar_fp32 {
#endif

// ---------------------------------------------------------------- complex --
#if FFTK_PAIRED_FP32
__device__ __forceinline__ float2 cadd(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float2 csub(float2 a, float2 b) { return __fadd2_rn(a, make_float2(-b.x, -b.y)); }
#else
__device__ __forceinline__ float2 cadd(float2 a, float2 b) { return make_float2(a.x + b.x, a.y + b.y); }
__device__ __forceinline__ float2 csub(float2 a, float2 b) { return make_float2(a.x - b.x, a.y - b.y); }
#endif
__device__ __forceinline__ float2 cmul(float2 a, float2 b) {
  return make_float2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
}
// a * conj(b)
__device__ __forceinline__ float2 cmulc(float2 a, float2 b) {
  return make_float2(a.x * b.x + a.y * b.y, a.y * b.x - a.x * b.y);
}
#if FFTK_PAIRED_FP32
__device__ __forceinline__ float2 cscale(float2 a, float s) { return __fmul2_rn(a, make_float2(s, s)); }
// a s + b
__device__ __forceinline__ float2 cscale_add(float2 a, float s, float2 b) { return __ffma2_rn(a, make_float2(s, s), b); }
#else
__device__ __forceinline__ float2 cscale(float2 a, float s) { return make_float2(a.x * s, a.y * s); }
__device__ __forceinline__ float2 cscale_add(float2 a, float s, float2 b) { return make_float2(fmaf(a.x, s, b.x), fmaf(a.y, s, b.y)); }
#endif
__device__ __forceinline__ float2 cconj(float2 a) { return make_float2(a.x, -a.y); }
// a * (SIGN * i)
template <int SIGN>
__device__ __forceinline__ float2 mul_si(float2 a) {
  return SIGN < 0 ? make_float2(a.y, -a.x) : make_float2(-a.y, a.x);
}

template <int N>
struct Log2 {
  static constexpr int value = 1 + Log2<N / 2>::value;
};
template <>
struct Log2<1> {
  static constexpr int value = 0;
};

// Mathematical constants of the 8- and 16-point DFTs (in FP64: rot rounds them).
#define FFTK_C8 0.70710678118654752440   // cos(pi/4)
#define FFTK_C16 0.92387953251128675613  // cos(pi/8)
#define FFTK_S16 0.38268343236508977173  // sin(pi/8)

// a * exp(SIGN i theta) with (cos, sin) = (c, s), constants after inlining.  The
// larger of the two is applied as 1 + (c - 1), a multiply-add in place of the
// product: rounded to FP32, the cosines of pi/16, pi/8 and pi/4 are all below the
// true ones, by 3.0e-8, 3.1e-8 and 1.7e-8, so that every factor shrinks its value
// and the losses add up over a transform and its inverse; the rounding of c - 1
// weighs a third of that at most.  Round-trip error of a line, rounded -> so: 1024
// points (32 x 32) 1.65e-7 -> 1.46e-7, 512 (32 x 16) 1.50e-7 -> 1.37e-7, 256
// (16 x 16) 1.38e-7 -> 1.28e-7, in the same number of operations.  (pi/4, where
// both components are the larger one, gains nothing and is left.)
template <int SIGN>
__device__ __forceinline__ float2 rot(float2 a, double c, double s) {
  const double t = SIGN * s, ac = c < 0. ? -c : c, at = t < 0. ? -t : t;
  const float fc = (float)c, ft = (float)t;
  if (ac == at) return cmul(a, make_float2(fc, ft));
  const float m = (float)((ac > at ? ac : at) - 1.);
#if FFTK_PAIRED_FP32 == 2
  const float2 z = cscale_add(a, m, a);
#else
  const float2 z = make_float2(fmaf(a.x, m, a.x), fmaf(a.y, m, a.y));
#endif
  if (ac > at) return make_float2(fmaf(-a.y, ft, c < 0. ? -z.x : z.x), fmaf(a.x, ft, c < 0. ? -z.y : z.y));
  return make_float2(fmaf(a.x, fc, t < 0. ? z.y : -z.y), fmaf(a.y, fc, t < 0. ? -z.x : z.x));
}

// cos and sin of pi/16 and 3 pi/16
#define FFTK_C32A 0.98078528040323044913
#define FFTK_S32A 0.19509032201612826785
#define FFTK_C32B 0.83146961230254523708
#define FFTK_S32B 0.55557023301960222474

// a * exp(-2 pi i q / 32) for a q (0 <= q < 32) known at compile time after
// unrolling: the eighth-turn remainder by its (cos, sin) constants, then the
// quarter and half turns exactly.  The Hermitian-split factor exp(-2 pi i k / N)
// of a real line of N = 2 G S points at k = j + m S (G values per thread on S
// threads) is W_j mul_root32 by q = m 16 / G: one table load per thread.
__device__ __forceinline__ float2 mul_root32(float2 a, int q) {
  float2 r;
  switch (q & 7) {
    case 0: r = a; break;
    case 1: r = rot<-1>(a, FFTK_C32A, FFTK_S32A); break;
    case 2: r = rot<-1>(a, FFTK_C16, FFTK_S16); break;
    case 3: r = rot<-1>(a, FFTK_C32B, FFTK_S32B); break;
    case 4: r = rot<-1>(a, FFTK_C8, FFTK_C8); break;
    case 5: r = rot<-1>(a, FFTK_S32B, FFTK_C32B); break;
    case 6: r = rot<-1>(a, FFTK_S16, FFTK_C16); break;
    default: r = rot<-1>(a, FFTK_S32A, FFTK_C32A); break;
  }
  if (q & 8) r = mul_si<-1>(r);
  return (q & 16) ? make_float2(-r.x, -r.y) : r;
}

// cos and sin of pi/24, 2 pi/24 and 5 pi/24
#define FFTK_C48A 0.99144486137381041114
#define FFTK_S48A 0.13052619222005159155
#define FFTK_C48B 0.96592582628906828675
#define FFTK_S48B 0.25881904510252076235
#define FFTK_C48E 0.79335334029123516458
#define FFTK_S48E 0.60876142900872063942
#define FFTK_C6 0.86602540378443864676  // cos(pi/6) = sin(pi/3)

// a * exp(-2 pi i m / NR) for m in [0, NR/2) known at compile time, NR a power
// of two up to 32 (mul_root32), 12, 24 or 48 (the same split for lines of
// 3 * 2^m values: steps of pi/24 by their constants, the quarter turn exactly)
template <int NR>
__device__ __forceinline__ float2 mul_root(float2 a, int m) {
  if constexpr (NR % 3 != 0) {
    return mul_root32(a, m * (32 / NR));
  } else {
    const int q = m * (48 / NR);
    float2 r;
    switch (q % 12) {
      case 0: r = a; break;
      case 1: r = rot<-1>(a, FFTK_C48A, FFTK_S48A); break;
      case 2: r = rot<-1>(a, FFTK_C48B, FFTK_S48B); break;
      case 3: r = rot<-1>(a, FFTK_C16, FFTK_S16); break;
      case 4: r = rot<-1>(a, FFTK_C6, 0.5); break;
      case 5: r = rot<-1>(a, FFTK_C48E, FFTK_S48E); break;
      case 6: r = rot<-1>(a, FFTK_C8, FFTK_C8); break;
      case 7: r = rot<-1>(a, FFTK_S48E, FFTK_C48E); break;
      case 8: r = rot<-1>(a, 0.5, FFTK_C6); break;
      case 9: r = rot<-1>(a, FFTK_S16, FFTK_C16); break;
      case 10: r = rot<-1>(a, FFTK_S48B, FFTK_C48B); break;
      default: r = rot<-1>(a, FFTK_S48A, FFTK_C48A); break;
    }
    return q >= 12 ? mul_si<-1>(r) : r;
  }
}

// The Hermitian-split factors exp(-2 pi i k / N), k = j + m S, of a thread with G
// values of a packed line (N = 2 G S points; t: the size-N table).  With four
// values one correctly rounded load for each; else W_j times the roots of order
// 2 G, whose product adds a rounding of its own.  (At 16 values per thread in
// k_ns_z one load per value and use instead: 1.190 against 1.126 ms per launch at
// 512^3.)
template <int N, int G, bool TABLE = G == 4>
struct SplitFactors {
  static constexpr int S = N / (2 * G), LOADS = TABLE ? G : 1;
  float2 w[LOADS];
  __device__ __forceinline__ SplitFactors(const float2* __restrict__ t, int j) {
#pragma unroll
    for (int m = 0; m < LOADS; ++m) w[m] = __ldg(&t[j + m * S]);
  }
  __device__ __forceinline__ float2 operator()(int m) const {
    if constexpr (TABLE) {
      return w[m];
    } else {
      return mul_root<2 * G>(w[0], m);
    }
  }
};

// index of the mirror H - k of entry k of a packed line of H values (k = 0: itself)
template <int H>
__device__ __forceinline__ int mirror(int k) {
  if constexpr ((H & (H - 1)) == 0) {
    return (H - k) & (H - 1);
  } else {
    return k == 0 ? 0 : H - k;
  }
}

// --------------------------------------------------------------- codelets --
// In-place DFT of R values held in registers, natural order in and out.
template <int SIGN>
__device__ __forceinline__ void dft2(float2& x0, float2& x1) {
  float2 t = x0;
  x0 = cadd(t, x1);
  x1 = csub(t, x1);
}

template <int SIGN>
__device__ __forceinline__ void dft4(float2& x0, float2& x1, float2& x2, float2& x3) {
  float2 a = cadd(x0, x2), b = csub(x0, x2);
  float2 c = cadd(x1, x3), d = mul_si<SIGN>(csub(x1, x3));
  x0 = cadd(a, c);
  x2 = csub(a, c);
  x1 = cadd(b, d);
  x3 = csub(b, d);
}

template <int SIGN>
__device__ __forceinline__ void dft8(float2 (&x)[8]) {
  dft4<SIGN>(x[0], x[2], x[4], x[6]);  // even samples: E0..E3 in x0,x2,x4,x6
  dft4<SIGN>(x[1], x[3], x[5], x[7]);  // odd samples:  O0..O3 in x1,x3,x5,x7
  float2 e0 = x[0], e1 = x[2], e2 = x[4], e3 = x[6];
  float2 o0 = x[1];
  float2 o1 = rot<SIGN>(x[3], FFTK_C8, FFTK_C8);   // W8^1
  float2 o2 = mul_si<SIGN>(x[5]);                  // W8^2
  float2 o3 = rot<SIGN>(x[7], -FFTK_C8, FFTK_C8);  // W8^3
  x[0] = cadd(e0, o0);
  x[4] = csub(e0, o0);
  x[1] = cadd(e1, o1);
  x[5] = csub(e1, o1);
  x[2] = cadd(e2, o2);
  x[6] = csub(e2, o2);
  x[3] = cadd(e3, o3);
  x[7] = csub(e3, o3);
}

// 16 = 4 x 4: X[k1 + 4 k2] = sum_{n2} W16^{n2 k1} W4^{n2 k2} sum_{n1} x[4 n1 + n2] W4^{n1 k1}
template <int SIGN>
__device__ __forceinline__ void dft16(float2 (&x)[16]) {
#pragma unroll
  for (int n2 = 0; n2 < 4; ++n2) dft4<SIGN>(x[n2], x[4 + n2], x[8 + n2], x[12 + n2]);
  // y[n2][k1] now sits at x[n2 + 4 k1]; apply W16^{n2 k1}
  x[5] = rot<SIGN>(x[5], FFTK_C16, FFTK_S16);      // n2=1,k1=1: W^1
  x[9] = rot<SIGN>(x[9], FFTK_C8, FFTK_C8);        // n2=1,k1=2: W^2
  x[13] = rot<SIGN>(x[13], FFTK_S16, FFTK_C16);    // n2=1,k1=3: W^3
  x[6] = rot<SIGN>(x[6], FFTK_C8, FFTK_C8);        // n2=2,k1=1: W^2
  x[10] = mul_si<SIGN>(x[10]);                     // n2=2,k1=2: W^4
  x[14] = rot<SIGN>(x[14], -FFTK_C8, FFTK_C8);     // n2=2,k1=3: W^6
  x[7] = rot<SIGN>(x[7], FFTK_S16, FFTK_C16);      // n2=3,k1=1: W^3
  x[11] = rot<SIGN>(x[11], -FFTK_C8, FFTK_C8);     // n2=3,k1=2: W^6
  x[15] = rot<SIGN>(x[15], -FFTK_C16, -FFTK_S16);  // n2=3,k1=3: W^9
#pragma unroll
  for (int k1 = 0; k1 < 4; ++k1) dft4<SIGN>(x[4 * k1], x[4 * k1 + 1], x[4 * k1 + 2], x[4 * k1 + 3]);
  // X[k1 + 4 k2] sits at x[4 k1 + k2]: transpose the 4x4 index grid
  float2 t[16];
#pragma unroll
  for (int i = 0; i < 16; ++i) t[i] = x[i];
#pragma unroll
  for (int k1 = 0; k1 < 4; ++k1)
#pragma unroll
    for (int k2 = 0; k2 < 4; ++k2) x[k1 + 4 * k2] = t[4 * k1 + k2];
}

// a * exp(SIGN 2 pi i q / 32), q known at compile time after unrolling
template <int SIGN>
__device__ __forceinline__ float2 rot32(float2 a, int q) {
  return mul_root32(a, SIGN < 0 ? q : (32 - q) & 31);
}

// 32 = 4 x 8: X[k1 + 4 k2] = sum_{n2} W32^{n2 k1} W8^{n2 k2} sum_{n1} x[8 n1 + n2] W4^{n1 k1}
template <int SIGN>
__device__ __forceinline__ void dft32(float2 (&x)[32]) {
#pragma unroll
  for (int n2 = 0; n2 < 8; ++n2) dft4<SIGN>(x[n2], x[8 + n2], x[16 + n2], x[24 + n2]);
  float2 o[32];
#pragma unroll
  for (int k1 = 0; k1 < 4; ++k1) {
    float2 t[8];
#pragma unroll
    for (int n2 = 0; n2 < 8; ++n2) t[n2] = rot32<SIGN>(x[8 * k1 + n2], n2 * k1);
    dft8<SIGN>(t);
#pragma unroll
    for (int k2 = 0; k2 < 8; ++k2) o[k1 + 4 * k2] = t[k2];
  }
#pragma unroll
  for (int k = 0; k < 32; ++k) x[k] = o[k];
}

// X1,2 = a - (b + c)/2 +- SIGN i sin(pi/3) (b - c).  FUSED: the last product and
// sum as one multiply-add each, a rounding less.
template <int SIGN, bool FUSED>
__device__ __forceinline__ void dft3(float2& a, float2& b, float2& c) {
  const float2 s = cadd(b, c), d = mul_si<SIGN>(csub(b, c));
  const float2 t = make_float2(fmaf(-0.5f, s.x, a.x), fmaf(-0.5f, s.y, a.y));
  a = cadd(a, s);
  if constexpr (FUSED) {
    b = cscale_add(d, (float)FFTK_C6, t);
    c = cscale_add(make_float2(-d.x, -d.y), (float)FFTK_C6, t);
  } else {
    const float2 h = cscale_add(d, (float)(FFTK_C6 - 1.), d);  // as in rot
    b = cadd(t, h);
    c = csub(t, h);
  }
}

template <int R, int SIGN, bool FUSED = true>
__device__ __forceinline__ void dftR(float2 (&a)[R]) {
  if constexpr (R % 3 == 0) {
    // R = 3 P, P = 1, 2, 4, 8 or 16: 3 and P have no common factor, so the DFT is
    // the two-dimensional 3 x P one without twiddles (Good's mapping):
    // n = P n1 + 3 n2, k = k1 (mod 3) = k2 (mod P)
    constexpr int P = R / 3;
    constexpr int E1 = P == 1 ? 1 : (P >= 8 ? 16 : 4), E2 = P == 1 ? 0 : (P == 2 ? 3 : (P == 16 ? 33 : 9));
#pragma unroll
    for (int n2 = 0; n2 < P; ++n2) dft3<SIGN, FUSED>(a[3 * n2], a[(P + 3 * n2) % R], a[(2 * P + 3 * n2) % R]);
    float2 o[R];
#pragma unroll
    for (int k1 = 0; k1 < 3; ++k1) {
      float2 t[P];
#pragma unroll
      for (int n2 = 0; n2 < P; ++n2) t[n2] = a[(P * k1 + 3 * n2) % R];
      if constexpr (P > 1) dftR<P, SIGN>(t);
#pragma unroll
      for (int k2 = 0; k2 < P; ++k2) o[(E1 * k1 + E2 * k2) % R] = t[k2];
    }
#pragma unroll
    for (int k = 0; k < R; ++k) a[k] = o[k];
  } else if constexpr (R == 2) {
    dft2<SIGN>(a[0], a[1]);
  } else if constexpr (R == 4) {
    dft4<SIGN>(a[0], a[1], a[2], a[3]);
  } else if constexpr (R == 8) {
    dft8<SIGN>(a);
  } else if constexpr (R == 16) {
    dft16<SIGN>(a);
  } else if constexpr (R == 32) {
    dft32<SIGN>(a);
  }
}

// --------------------------------------------------------- smem swizzle ----
// Position `pos` of a tile with T columns (T a power of two; column c added by
// the caller).  For T < 16 the 16/T rows that share a 16-element block are
// placed by an XOR fold of pos's digits, so every access pattern of the engine
// (unit-stride rows, and radix-R strided rows) is bank-conflict free for
// 64-bit accesses (a half warp covers all 32 banks once).
template <int T>
__device__ __forceinline__ int swz(int pos) {
  if constexpr (T >= 16) {
    return pos * T;
  } else {
    constexpr int t = Log2<T>::value;
    constexpr int s = 4 - t;
    int f = pos;
#pragma unroll
    for (int sh = s; sh < 16; sh += s) f ^= pos >> sh;
    f &= (1 << s) - 1;
    return ((pos >> s) << 4) + (f << t);
  }
}

// Exchange buffer for a column tile: element (pos, c) of a [L][T] tile.
template <int T>
struct ColX {
  static constexpr bool kTight = false;
  static constexpr bool kStageTables = false;  // a warp spans 32/T butterflies: gathers are near-broadcasts
  float2* s;
  int c;
  __device__ __forceinline__ void st(int pos, float2 v) const { s[swz<T>(pos) + c] = v; }
  __device__ __forceinline__ float2 ld(int pos) const { return s[swz<T>(pos) + c]; }
  __device__ __forceinline__ void sync() const { __syncthreads(); }
};

// Position of element `pos` of one contiguous line: an XOR permutation within
// each 16-element block, keyed by the block index B = pos >> 4 through the
// map bits(B) -> {1, 2, 12, 8, then 1, 2, 4, 8, ...}.  Block bit 2 flips slot
// bits 2 and 3, which makes the radix-8 exchanges (8 values per thread) as
// well as the radix-16 ones conflict free for 64-bit accesses.
__device__ __forceinline__ int swz_line(int pos) {
  const int b = pos >> 4;
  const int lo = b & 15;
  const int h = lo ^ ((lo & 4) << 1) ^ (b >> 4) ^ (b >> 8);
  return (pos & ~15) | ((pos ^ h) & 15);
}

// The same with the map {7, 10, 12, 8, ...}, which also keeps the radix-4
// exchanges (4 or 12 values per thread) free of conflicts, at a few more
// integer operations.
__device__ __forceinline__ int swz_line4(int pos) {
  const int b = pos >> 4;
  const int lo = b & 15;
  const int h = lo ^ ((lo & 1) * 6) ^ ((lo & 2) << 2) ^ ((lo & 4) << 1) ^ (b >> 4) ^ (b >> 8);
  return (pos & ~15) | ((pos ^ h) & 15);
}

// Lines of S < 16 threads share a half warp: line li of a CTA permutes its
// slots by one more XOR, so that the lines' equal positions lie in different
// banks.  (Simulated over all exchanges, packed lines of 48 values on 4
// threads: 4.0 -> 1.25 times the least number of wavefronts; 96 on 8: 2.4 ->
// 1.15; 192 on 16 through swz_line4: 1.67 -> 1.17.)
template <int S>
__device__ __forceinline__ int line_xor(int li) {
  if constexpr (S == 8) return (li & 1) * 9;
  if constexpr (S == 4) return ((li & 1) * 5) ^ ((li & 2) * 5);
  if constexpr (S == 2) return (li & 7) * 2;
  return 0;
}

// Exchange buffer for one contiguous line of S threads with G values each;
// WARP_SYNC when a line's threads live in one warp.  TIGHT: a kernel without
// registers to spare (see dft3).
template <bool WARP_SYNC, int S = 32, int G = 16, bool TIGHT = false>
struct LineX {
  static constexpr bool kTight = TIGHT;
  static constexpr bool kStageTables = true;  // a warp spans 32 consecutive butterflies
  static constexpr bool kMap4 = G != 16 && (S < 16 || G % 8 != 0);
  float2* s;
  int x = 0;  // line_xor
  __device__ __forceinline__ int at(int pos) const { return (kMap4 ? swz_line4(pos) : swz_line(pos)) ^ x; }
  __device__ __forceinline__ void st(int pos, float2 v) const { s[at(pos)] = v; }
  __device__ __forceinline__ float2 ld(int pos) const { return s[at(pos)]; }
  // unpermuted, for a line that is stored in the natural pattern and read as
  // its mirror H - k: both are runs of consecutive slots (the permuted mirror
  // took two wavefronts for one)
  __device__ __forceinline__ void st_run(int pos, float2 v) const { s[pos ^ x] = v; }
  __device__ __forceinline__ float2 ld_run(int pos) const { return s[pos ^ x]; }
  __device__ __forceinline__ void sync() const {
    if constexpr (WARP_SYNC)
      __syncwarp();
    else
      __syncthreads();
  }
};

// brings the line of p (a valid global address) into L2
__device__ __forceinline__ void prefetch_l2(const void* p) { asm volatile("prefetch.global.L2 [%0];" ::"l"(p)); }

// ---------------------------------------------------------------- engine ---
// Twiddle tables: the plan holds, for every power of two L' <= 4 LT, the
// table exp(-2 pi i m / L'), m < L', at offset L' of one array (entries
// computed in FP64 on the host and rounded once to FP32).  A kernel gets the
// table of size 2^TL >= L, which locates the array's base at compile time.
//
// A stage of span M = NS R (radix R after NS points) multiplies input r of
// butterfly k by exp(-2 pi i r k / M).  In a contiguous line (LineX) one warp
// holds 32 consecutive butterflies, and a gather from the size-L table at
// index r k L / M spreads each load over up to 32 scattered entries; so the
// plan also stores, for every M <= 4096 and R in {2, 4, 8, 16}, the table
// exp(-2 pi i r k / M) r-major (entry r NS + k), which those stages read.
// These tables lie kStageTwiddles entries below the base of the pyramid (the
// same FP64-built values, rounded the same way).  Column tiles (ColX) keep the
// pyramid: their warps span 32/T butterflies, so the gathers are already
// near-broadcasts.
constexpr int kStageTwiddles = 32768;
__host__ __device__ constexpr int stage_tw_offset(int M, int R) {
  return 4 * M + (R == 2 ? 0 : (R == 4 ? 1 : (R == 8 ? 2 : 3))) * M;
}

// The last stage of a line of M = 3 * 2^j points has radix R in {3, 6, 12, 24}.
// The plan holds exp(-2 pi i m / M), m < M, for every M = 3 * 2^j up to its
// longest such axis at offset M of one array, and below that array the r-major
// tables of the pairs (M, R) for contiguous lines, laid out as above.
constexpr int kStage3Twiddles = 24576;
__host__ __device__ constexpr int stage3_tw_offset(int M, int R) {
  return 4 * M + (R == 3 ? 0 : (R == 6 ? 1 : (R == 12 ? 2 : 3))) * M;
}

__host__ __device__ constexpr int fftk_min3(int a, int b, int c) {
  return a < b ? (a < c ? a : c) : (b < c ? b : c);
}

// Radix of the stage that takes up `rem` remaining points at g values per
// thread: min(16, g, rem) for powers of two; while the factor 3 remains, all
// of rem if one butterfly can hold it, else the largest power of two in g.
__host__ __device__ constexpr int stage_radix(int rem, int g) {
  if (rem % 3 != 0) return fftk_min3(16, g, rem);
  if (rem <= g && g % rem == 0) return rem;
  return fftk_min3(16, g & -g, rem / 3);
}

template <int L, int G, int SIGN, int NS, int TL>
struct Stage {
  template <class X>
  __device__ __forceinline__ static void run(float2 (&v)[G], int j, const X& xc, const float2* __restrict__ tw,
                                             const float2* __restrict__ t3) {
    if constexpr (NS < L) {
      constexpr int REM = L / NS;
      constexpr int R = stage_radix(REM, G);
      constexpr int B = G / R;   // butterflies per thread
      constexpr int S = L / G;   // threads per line
      static_assert(B * R == G && REM % R == 0, "radix");
      constexpr bool LAST = (NS * R == L);
#pragma unroll
      for (int t = 0; t < B; ++t) {
        const int b = j + t * S;   // butterfly index in [0, L/R)
        const int k = b & (NS - 1);
        float2 a[R];
#pragma unroll
        for (int r = 0; r < R; ++r) a[r] = v[t + r * B];
        if constexpr (NS > 1 && R % 3 == 0) {
          // exp(SIGN 2 pi i r k / L) of the last stage, L = NS R = 3 * 2^m
          const float2* ts = t3 - kStage3Twiddles + stage3_tw_offset(L, R);
          const float2* tg = t3 + L;
#pragma unroll
          for (int r = 1; r < R; ++r) {
            const float2 w = X::kStageTables ? __ldg(&ts[r * NS + k]) : __ldg(&tg[r * k]);
            a[r] = SIGN < 0 ? cmul(a[r], w) : cmulc(a[r], w);
          }
        } else if constexpr (NS > 1) {
          // exp(SIGN 2 pi i r k / (NS R)): from this stage's r-major table for
          // contiguous lines, else from the size-2^TL table (tw, at offset 2^TL
          // of the pyramid) at index r k 2^TL / (NS R)
          constexpr int LOG_NSR = Log2<NS * R>::value;
          const float2* ts = tw - (1 << TL) - kStageTwiddles + stage_tw_offset(NS * R, R);
#pragma unroll
          for (int r = 1; r < R; ++r) {
            const float2 w = X::kStageTables ? __ldg(&ts[r * NS + k]) : __ldg(&tw[(r * k) << (TL - LOG_NSR)]);
            a[r] = SIGN < 0 ? cmul(a[r], w) : cmulc(a[r], w);
          }
        }
        dftR<R, SIGN, !X::kTight>(a);
        if constexpr (LAST) {
#pragma unroll
          for (int r = 0; r < R; ++r) v[t + r * B] = a[r];
        } else {
          const int base = (b - k) * R + k;  // (b / NS) * NS * R + k
#pragma unroll
          for (int r = 0; r < R; ++r) xc.st(base + r * NS, a[r]);
        }
      }
      if constexpr (!LAST) {
        xc.sync();
#pragma unroll
        for (int m = 0; m < G; ++m) v[m] = xc.ld(j + m * S);
        xc.sync();
        Stage<L, G, SIGN, NS * R, TL>::run(v, j, xc, tw, t3);
      }
    }
  }
};

// Full L-point transform of the line held in v (natural pattern in and out).
// The exchange buffer must be free on entry; it is free again on exit.
// tw: the power-of-two twiddle table of size 2^TL (by default the largest one
// not longer than L); t3: the plan's 3 * 2^m tables (such lines only).
template <int L, int G, int SIGN, int TL = Log2<L>::value, class X>
__device__ __forceinline__ void fft_line(float2 (&v)[G], int j, const X& xc, const float2* __restrict__ tw,
                                         const float2* __restrict__ t3 = nullptr) {
  static_assert((1 << TL) >= (L % 3 == 0 ? L / 3 : L), "twiddle table too short");
  Stage<L, G, SIGN, 1, TL>::run(v, j, xc, tw, t3);
}

// Elements per thread used by the strided passes for a line of length L: 16,
// and 24 (radices 8, 8, 12 at 768) for lines of 3 * 2^m points that are long
// enough to spread over several threads.
__host__ __device__ constexpr int elems_per_thread(int L) {
  if (L % 3 == 0) return L >= 96 ? 24 : (L >= 12 ? 12 : L);
  return L < 16 ? L : 16;
}
// slots of the exchange buffer of one contiguous line of H values (the
// permutations stay within blocks of 16)
__host__ __device__ constexpr int line_slots(int H) { return (H + 15) / 16 * 16; }

}  // inline namespace
}  // namespace fftk
