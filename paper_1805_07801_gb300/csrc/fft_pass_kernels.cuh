// The three 1D pass kinds of the 3D transform (paper Sec. 3), as templates on
// the line length: instantiated for powers of two in fft_passes.cu and for
// 3 * 2^m in fft_radix3.cu.  The z pass (real <-> half complex) works on
// contiguous lines, the strided complex pass serves y and x.
// The paper's MPI_Alltoall exchanges between passes are absent:
// every pass reads its lines in place, batched across the contiguous index
// (the transpose-free layout of Appendix A), so no reorder pass exists.
#pragma once

#include <mutex>

#include "fft_engine.cuh"
#include "internal.h"

namespace fftk {

// ------------------------------------------------------------------ z pass --
// Values per thread of a packed line of H: 16, fewer on short lines, so that at
// least eight threads share a line of 16 or more (64-byte pieces, more threads
// for small grids); 24 or 12 for 3 * 2^m.  Pairs with 16 values -> these:
// 64^3 35.6 -> 24.6 us, 64 fields of 64^3 308 -> 217 us, 8 of 256 x 256 x 128
// 818 -> 683 us, 16 of 256^3 2508 -> 2406 us, 16 of 512 x 512 x 32 2369 -> 1709 us; H = 256 is
// slower with 8 (two 512^3 fields 2277 against 2190 us).
__host__ __device__ constexpr int z_elems(int H) {
  if (H % 3 == 0) return H >= 192 ? 24 : (H >= 48 ? 12 : 6);
  if (H < 16) return H < 2 ? H : 2;
  return H <= 64 ? 4 : (H <= 128 ? 8 : 16);
}

template <int N>
struct ZCfg {
  static constexpr int H = N / 2;                  // complex length of the packed line
  static constexpr int HB = line_slots(H);         // its exchange slots
  static constexpr int G = z_elems(H);
  static constexpr int S = H / G;                  // threads per line
  static constexpr int MAXT = N % 3 == 0 ? 128 : 256;
  static constexpr int LPC = S >= MAXT ? 1 : MAXT / S;  // lines per CTA
  static constexpr int THREADS = LPC * S;
  static constexpr bool WARP = S <= 32;
  // split factors from the table: lines of 24 points have 3 % less error so (and
  // those of 48 would take 4 % longer for half a percent)
  static constexpr bool TABLE = G == 4 || (G == 6 && S <= 2);
  static constexpr int MINB = 4;  // 32 warps per SM at <= 64 registers (3 * 2^m: 16 at <= 128)
};

// Real-to-complex along z.  The N reals of a line are packed as H = N/2
// complex values z[n] = x[2n] + i x[2n+1]; after the H-point transform Z,
//   X[k] = (Z[k] + conj Z[H-k])/2 + exp(-2 pi i k/N) (Z[k] - conj Z[H-k])/(2i),
// k = 0..H (Z[H] = Z[0]).
template <int N>
__global__ void __launch_bounds__(ZCfg<N>::THREADS, ZCfg<N>::MINB)
    k_z_r2c(const float* __restrict__ in, float2* __restrict__ out, long long nlines,
            const float2* __restrict__ tw, const float2* __restrict__ t3, float scale) {  // tw: size-2^LOGN table
  pdl_wait();
  using C = ZCfg<N>;
  constexpr int H = C::H, G = C::G, S = C::S;
  constexpr int LOGN = Log2<N>::value;
  __shared__ float2 sm[C::LPC * C::HB];
  const int li = threadIdx.x / S, j = threadIdx.x % S;
  const long long line = (long long)blockIdx.x * C::LPC + li;
  const bool valid = line < nlines;
  const LineX<C::WARP, S, G> xc{sm + li * C::HB, line_xor<S>(li)};
  float2 v[G];
  const float2* src = reinterpret_cast<const float2*>(in + line * N);
#pragma unroll
  for (int m = 0; m < G; ++m) v[m] = valid ? src[j + m * S] : make_float2(0.f, 0.f);
  fft_line<H, G, -1, LOGN>(v, j, xc, tw, t3);
#pragma unroll
  for (int m = 0; m < G; ++m) xc.st_run(j + m * S, v[m]);
  xc.sync();
  if (valid) {
    float2* dst = out + line * (H + 1);
    const SplitFactors<N, G, C::TABLE> split(N % 3 == 0 ? t3 + N : tw, j);
#pragma unroll
    for (int m = 0; m < G; ++m) {
      const int k = j + m * S;
      const float2 A = v[m];
      const float2 Bc = cconj(xc.ld_run(mirror<H>(k)));
      const float2 E = cscale(cadd(A, Bc), 0.5f);
      const float2 D = csub(A, Bc);
      const float2 O = make_float2(0.5f * D.y, -0.5f * D.x);  // D / (2i)
      dst[k] = cscale(cadd(E, cmul(split(m), O)), scale);
    }
    if (j == 0) dst[H] = make_float2((v[0].x - v[0].y) * scale, 0.f);
  }
}

// Complex-to-real along z: the inverse of the packing above.  With
// E = X[k] + conj X[H-k] and O = (X[k] - conj X[H-k]) exp(+2 pi i k/N),
// Z[k] = E + i O, and the unnormalised H-point inverse of Z gives
// x[2n] + i x[2n+1].  Im X[0] and Im X[H] are ignored (line-wise c2r).
template <int N>
__global__ void __launch_bounds__(ZCfg<N>::THREADS, ZCfg<N>::MINB)
    k_z_c2r(const float2* __restrict__ in, float* __restrict__ out, long long nlines,
            const float2* __restrict__ tw, const float2* __restrict__ t3) {  // tw: size-2^LOGN table
  pdl_wait();
  using C = ZCfg<N>;
  constexpr int H = C::H, G = C::G, S = C::S;
  constexpr int LOGN = Log2<N>::value;
  __shared__ float2 sm[C::LPC * C::HB];
  const int li = threadIdx.x / S, j = threadIdx.x % S;
  const long long line = (long long)blockIdx.x * C::LPC + li;
  const bool valid = line < nlines;
  const LineX<C::WARP, S, G> xc{sm + li * C::HB, line_xor<S>(li)};
  const float2* src = in + line * (H + 1);
  // X[0..H-1] of the line pass through the exchange buffer once, so the
  // mirror X[H - k] is read from there instead of a second global load
  // (X[H] itself, the k = 0 mirror, is one broadcast load)
  float2 v[G];
#pragma unroll
  for (int m = 0; m < G; ++m) {
    v[m] = valid ? src[j + m * S] : make_float2(0.f, 0.f);
    xc.st_run(j + m * S, v[m]);
  }
  const float2 XH = valid ? src[H] : make_float2(0.f, 0.f);
  const SplitFactors<N, G, C::TABLE> split(N % 3 == 0 ? t3 + N : tw, j);
  xc.sync();
#pragma unroll
  for (int m = 0; m < G; ++m) {
    const int k = j + m * S;
    float2 A = v[m];
    float2 B = k == 0 ? XH : xc.ld_run(H - k);
    if (k == 0) {
      A.y = 0.f;
      B.y = 0.f;
    }
    const float2 Bc = cconj(B);
    const float2 E = cadd(A, Bc);
    const float2 O = cmulc(csub(A, Bc), split(m));
    v[m] = make_float2(E.x - O.y, E.y + O.x);
  }
  xc.sync();  // every mirror has been read before the transform's exchanges
  fft_line<H, G, +1, LOGN>(v, j, xc, tw, t3);
  if (valid) {
    float2* dst = reinterpret_cast<float2*>(out + line * N);
#pragma unroll
    for (int m = 0; m < G; ++m) dst[j + m * S] = v[m];
  }
}

// ------------------------------------------------------- strided c2c pass --
// Tile = T adjacent columns (contiguous index q) x the full line (L rows of
// stride Q).  Loads and stores are T-wide row segments, coalesced along q.
// Tile width T per line length: 16 columns (128-byte rows) where the 227 KB of
// shared memory allows and at least 64 threads come together; 32 warps per SM at
// <= 64 registers per thread.  (256 threads per CTA with up to 256 columns, two
// CTAs per SM: y passes of short rows left most columns empty.  Pairs: 64 fields
// of 32^3 39 -> 25 us, 64 of 64^3 186 -> 149 us, 8 of 128^3 174 -> 140 us.)
// Lines of 3 * 2^m points hold 24 values per thread at <= 128 registers, 512
// threads per SM.
template <int L>
struct CCfg {
  static constexpr int G = elems_per_thread(L);
  static constexpr int S = L / G;
  static constexpr int MAXT = L % 3 == 0 ? 512 : 1024;
  static constexpr int T = S <= 16 ? (L % 3 == 0 ? 16 : (S >= 4 ? 16 : 64 / S)) : (16 * S <= MAXT ? 16 : MAXT / S);
  static constexpr int THREADS = T * S;
  static constexpr int MINB = L % 3 == 0 ? (THREADS <= 128 ? 4 : (THREADS <= 256 ? 2 : 1)) : (1024 / THREADS < 16 ? 1024 / THREADS : 16);
  static constexpr size_t SMEM = sizeof(float2) * (size_t)L * T;
};

// AHEAD > 0: while it transforms, the CTA asks for the rows of the tile AHEAD
// places on (the one that comes next on some SM) in L2.  For lines that leave
// room for one CTA per SM, whose loads nothing else covers.
template <int L, int SIGN, int AHEAD>
__global__ void __launch_bounds__(CCfg<L>::THREADS, CCfg<L>::MINB)
    k_cpass(const float2* in, float2* out, long long Q, long long qtiles,
            const float2* __restrict__ tw, const float2* __restrict__ t3, float scale) {
  pdl_wait();
  using C = CCfg<L>;
  constexpr int G = C::G, S = C::S, T = C::T;
  extern __shared__ float2 smc[];
  const int c = threadIdx.x % T, j = threadIdx.x / T;
  const long long tile = blockIdx.x;
  const long long p = tile / qtiles;
  const long long q = (tile - p * qtiles) * T + c;
  const bool valid = q < Q;
  const long long base = p * (long long)L * Q + q;
  float2 v[G];
#pragma unroll
  for (int m = 0; m < G; ++m)
    v[m] = valid ? in[base + (long long)(j + m * S) * Q] : make_float2(0.f, 0.f);
  if constexpr (AHEAD > 0) {
    const long long nt = tile + AHEAD;
    if (nt < (long long)gridDim.x) {
      const long long np = nt / qtiles;
      const float2* src = in + np * (long long)L * Q + (nt - np * qtiles) * T;
      for (int r = threadIdx.x; r < L; r += C::THREADS) prefetch_l2(src + (long long)r * Q);
    }
  }
  fft_line<L, G, SIGN>(v, j, ColX<T>{smc, c}, tw, t3);
  if (valid) {
#pragma unroll
    for (int m = 0; m < G; ++m) out[base + (long long)(j + m * S) * Q] = cscale(v[m], scale);
  }
}

// ----------------------------------------------------------- launchers -----
template <int N>
static cudaError_t z_r2c_n(fftk_plan p, const float* in, float2* out, long long nl, float scale,
                           cudaStream_t st) {
  using C = ZCfg<N>;
  const long long blocks = (nl + C::LPC - 1) / C::LPC;
  LaunchScope ls(p, KK_Z_R2C, st);
  launch_pdl(k_z_r2c<N>, (unsigned)blocks, C::THREADS, 0, st, in, out, nl, twiddles(p, 1 << Log2<N>::value), p->d_tw3,
             scale);
  return cudaGetLastError();
}

template <int N>
static cudaError_t z_c2r_n(fftk_plan p, const float2* in, float* out, long long nl,
                           cudaStream_t st) {
  using C = ZCfg<N>;
  const long long blocks = (nl + C::LPC - 1) / C::LPC;
  LaunchScope ls(p, KK_Z_C2R, st);
  launch_pdl(k_z_c2r<N>, (unsigned)blocks, C::THREADS, 0, st, in, out, nl, twiddles(p, 1 << Log2<N>::value), p->d_tw3);
  return cudaGetLastError();
}

template <int L, int SIGN, int AHEAD>
static cudaError_t cpass_la(fftk_plan p, const float2* in, float2* out, long long P, long long Q, float scale,
                            int kind, cudaStream_t st) {
  using C = CCfg<L>;
  static PerDevice once;
  const cudaError_t attr_err = once.run([](int) {
    return cudaFuncSetAttribute(k_cpass<L, SIGN, AHEAD>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)C::SMEM);
  });
  if (attr_err != cudaSuccess) return attr_err;
  const long long qtiles = (Q + C::T - 1) / C::T;
  const long long blocks = P * qtiles;
  LaunchScope ls(p, kind, st);
  launch_pdl(k_cpass<L, SIGN, AHEAD>, (unsigned)blocks, C::THREADS, C::SMEM, st, in, out, Q, qtiles,
             twiddles(p, 1 << Log2<L>::value), p->d_tw3, scale);
  return cudaGetLastError();
}

template <int L, int SIGN>
static cudaError_t cpass_l(fftk_plan p, const float2* in, float2* out, long long P, long long Q, float scale,
                           int kind, cudaStream_t st) {
  // rows further apart than a few pages (the x pass) only where 24 values per
  // thread leave 16 warps on the SM (1024^3, before its pipelined pass: y 2.07 ->
  // 1.95 ms, but x, with 32 warps, 2.01 against 2.12 ms).  Of the lines that
  // fft_stream.cu takes unless the array is narrow or small, 768 points keep it
  // (1000 planes of 9 columns, inverse 65.3 -> 62.4 us), 1536 do not (21.8 against
  // 23.0 us, 57.2 against 60.0, 192 against 188), and 1024 would spill.
  if constexpr (L == 768 || L >= 2048)
    if (Q <= 4096 || L % 3 == 0) return cpass_la<L, SIGN, 152>(p, in, out, P, Q, scale, kind, st);
  return cpass_la<L, SIGN, 0>(p, in, out, P, Q, scale, kind, st);
}

}  // namespace fftk
