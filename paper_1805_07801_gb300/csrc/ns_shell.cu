// Shell-to-shell energy transfer (paper Sec. 1 and Sec. 3: the scale-by-scale
// analysis): per giver shell the advection term (u . grad) u_g through passes
// that touch only the modes at hand.
//
// With the giver's modes inside |k_i| <= kb, the inverse passes read and write
// columns and rows up to kb only, and the real gradient never reaches memory:
//   x: U_i = F^-1_x u_g,i and D_i = F^-1_x (i k_x u_g,i)
//   y: U_i, i k_y U_i and D_i (each written where the z pass reads it)
//   z: per line, for each i: the three gradient components (i k_z applied to
//      U_i here) to real space, their products with u summed, and back
//   y, x forward on the kept modes, then the reduction over the receivers.
// 256^3, eight octave shells: 12.6 ms through 25 inverse and 8 forward
// transforms of three full fields, 3.8 ms so (32^3: 1.03 and 0.31 ms).
#include <cmath>
#include <mutex>
#include <vector>

#include "ns_passes.cuh"

namespace fftk {

// the integers k^2 of the modes with lo <= nint|k| < hi (|k| >= b - 1/2 exactly
// when k^2 >= b^2 - b + 1, for b >= 1)
struct ShellRange {
  int k2lo, k2hi;  // inclusive
  int kb;          // largest |k_i| of the shell's kept modes
};

// x: fields 0..2 of w get U_i, fields 3..5 D_i; blockIdx -> (i, k_y, k_z tile)
template <int N>
__global__ void __launch_bounds__(NXCfg<N>::THREADS, NXCfg<N>::MINB)
    k_shell_invx(const float2* __restrict__ u, float2* __restrict__ w, ShellRange sh, int ktiles,
                 const float2* __restrict__ tw) {
  pdl_wait();
  constexpr long long H1 = N / 2 + 1, MM = (long long)N * N * H1;
  constexpr long long HW = ns_row(N), MW = (long long)N * N * HW;
  using C = NXCfg<N>;
  constexpr int G = C::G, S = C::S, T = C::T;
  extern __shared__ float2 sms[];
  const int c = threadIdx.x % T, j = threadIdx.x / T;
  const int kt = blockIdx.x % ktiles, rest = blockIdx.x / ktiles;
  const int nk = 2 * sh.kb + 1;
  const int i = rest / nk, ay = dense_to_a(rest - i * nk, N, sh.kb);
  const int kz = kt * T + c, ky = kwav(ay, N);
  const bool valid = kz <= sh.kb;
  const float2* src = u + i * MM + (long long)ay * H1 + kz;
  float2* dst = w + i * MW + (long long)ay * HW + kz;
  float2 v[G];
#pragma unroll 1
  for (int d = 0; d < 2; ++d) {  // U_i, then D_i
#pragma unroll
    for (int m = 0; m < G; ++m) {
      const int pos = j + m * S, kx = kwav(pos, N), k2 = kx * kx + ky * ky + kz * kz;
      float2 a = make_float2(0.f, 0.f);
      if (valid && kept_xy(pos, N, sh.kb) && k2 >= sh.k2lo && k2 <= sh.k2hi) a = src[(long long)pos * N * H1];
      v[m] = d ? mul_i(a, (float)kx) : a;
    }
    fft_line<N, G, +1>(v, j, ColX<T>{sms, c}, tw);
    if (valid) {
#pragma unroll
      for (int m = 0; m < G; ++m) dst[3 * d * MW + (long long)(j + m * S) * N * HW] = v[m];
    }
  }
}

// y: blockIdx -> (f, x, k_z tile); f < 3: U_f of a to fields f (U_f) and 3 + f
// (i k_y U_f) of b; f >= 3: D in place in a
template <int N>
__global__ void __launch_bounds__(NXCfg<N>::THREADS, NXCfg<N>::MINB)
    k_shell_invy(float2* a, float2* __restrict__ b, int kb, int ktiles, const float2* __restrict__ tw) {
  pdl_wait();
  constexpr long long HW = ns_row(N), MW = (long long)N * N * HW;
  using C = NXCfg<N>;
  constexpr int G = C::G, S = C::S, T = C::T;
  extern __shared__ float2 sms[];
  const int c = threadIdx.x % T, j = threadIdx.x / T;
  const int kt = blockIdx.x % ktiles, rest = blockIdx.x / ktiles;
  const int x = rest % N, f = rest / N;
  const int kz = kt * T + c;
  const bool valid = kz <= kb;
  const long long off = (long long)x * N * HW + kz;
  const float2* src = a + f * MW + off;
  float2 v[G];
#pragma unroll 1
  for (int d = 0; d < (f < 3 ? 2 : 1); ++d) {
#pragma unroll
    for (int m = 0; m < G; ++m) {
      const int pos = j + m * S;
      float2 t = make_float2(0.f, 0.f);
      if (valid && kept_xy(pos, N, kb)) t = src[(long long)pos * HW];
      v[m] = d ? mul_i(t, (float)kwav(pos, N)) : t;
    }
    fft_line<N, G, +1>(v, j, ColX<T>{sms, c}, tw);
    if (valid) {
      float2* dst = (f < 3 ? b + (3 * d + f) * MW : a + f * MW) + off;
#pragma unroll
      for (int m = 0; m < G; ++m) dst[(long long)(j + m * S) * HW] = v[m];
    }
  }
}

// z: per (x, y) line A_i = sum_j u_j d_j u_g,i and back, k_z < kc written to
// fields 0..2 of a (the U of the x pass, read by then).  ur: u in real space.
template <int N>
struct SZCfg3 {
  using Z = NZCfg<N>;
  static constexpr size_t SMEM = sizeof(float2) * (size_t)Z::LPC * (Z::HB + 3 * Z::H);  // exchange + u
  static constexpr int MINB = Z::G >= 16 ? 2 : 4;
};

template <int N>
__global__ void __launch_bounds__(NZCfg<N>::THREADS, SZCfg3<N>::MINB)
    k_shell_z(float2* a, const float2* __restrict__ b, const float* __restrict__ ur, int kb,
              const float2* __restrict__ tw) {
  pdl_wait();
  constexpr long long HW = ns_row(N), MW = (long long)N * N * HW, R = (long long)N * N * N;
  using C = NZCfg<N>;
  constexpr int H = C::H, G = C::G, S = C::S, KC = C::KC;
  constexpr int LOGN = Log2<N>::value;
  extern __shared__ float2 sms[];
  const int li = threadIdx.x / S, j = threadIdx.x % S;
  const long long line = (long long)blockIdx.x * C::LPC + li;
  const bool valid = line < (long long)N * N;
  const LineX<C::WARP, S, G> xc{sms + li * C::HB, line_xor<S>(li)};
  const SplitFactors<N, G> twk(tw, j);
  float2* park = sms + C::LPC * C::HB + li * 3 * H + j;  // u, [3][G][S], two real points per slot
#pragma unroll
  for (int q = 0; q < 3; ++q) {
    const float2* src = reinterpret_cast<const float2*>(ur + q * R + line * N);
#pragma unroll
    for (int m = 0; m < G; ++m) park[(q * G + m) * S] = valid ? src[j + m * S] : make_float2(0.f, 0.f);
  }
#pragma unroll 1
  for (int i = 0; i < 3; ++i) {
    float2 acc[G];
#pragma unroll
    for (int m = 0; m < G; ++m) acc[m] = make_float2(0.f, 0.f);
#pragma unroll
    for (int q = 0; q < 3; ++q) {
      const float2* src = (q == 0 ? a + (3 + i) * MW : b + (q == 1 ? 3 + i : i) * MW) + line * HW;
      float2 W[G];
#pragma unroll
      for (int m = 0; m < G; ++m) {
        const int k = j + m * S;
        float2 A = make_float2(0.f, 0.f), B = make_float2(0.f, 0.f);
        if (valid && k <= kb) A = src[k];
        if (valid && H - k <= kb) B = src[H - k];
        if (q == 2) {  // d_z
          A = mul_i(A, (float)k);
          B = mul_i(B, (float)(H - k));
        }
        if (k == 0) {
          A.y = 0.f;
          B.y = 0.f;
        }
        const float2 Bc = cconj(B);
        const float2 E = cadd(A, Bc);
        const float2 O = cmulc(csub(A, Bc), twk(m));
        W[m] = make_float2(E.x - O.y, E.y + O.x);
      }
      fft_line<H, G, +1, LOGN>(W, j, xc, tw);
      if constexpr (S == 1) xc.sync();
#pragma unroll
      for (int m = 0; m < G; ++m) acc[m] = __ffma2_rn(park[(q * G + m) * S], W[m], acc[m]);
    }
    fft_line<H, G, -1, LOGN>(acc, j, xc, tw);
#pragma unroll
    for (int m = 0; m < G; ++m) xc.st_run(j + m * S, acc[m]);
    xc.sync();
    float2* dst = a + i * MW + line * HW;
#pragma unroll
    for (int m = 0; m < G; ++m) {
      const int k = j + m * S;
      const float2 Bc = cconj(xc.ld_run(mirror<H>(k)));
      const float2 E = cscale(cadd(acc[m], Bc), 0.5f);
      const float2 D = csub(acc[m], Bc);
      const float2 O = make_float2(0.5f * D.y, -0.5f * D.x);
      if (valid && k < KC) dst[k] = cadd(E, cmul(twk(m), O));
    }
    xc.sync();
  }
}

// forward x pass of three fields, kept rows of kept columns, into rows of n/2 + 1
template <int N>
__global__ void __launch_bounds__(NXCfg<N>::THREADS, NXCfg<N>::MINB)
    k_shell_fwdx(const float2* __restrict__ a, float2* __restrict__ out, int ktiles, float scale,
                 const float2* __restrict__ tw) {
  pdl_wait();
  constexpr long long H1 = N / 2 + 1, MM = (long long)N * N * H1;
  constexpr long long HW = ns_row(N), MW = (long long)N * N * HW;
  constexpr int KD = (N - 1) / 3, NK = 2 * KD + 1;
  using C = NXCfg<N>;
  constexpr int G = C::G, S = C::S, T = C::T;
  extern __shared__ float2 sms[];
  const int c = threadIdx.x % T, j = threadIdx.x / T;
  const int kt = blockIdx.x % ktiles, rest = blockIdx.x / ktiles;
  const int f = rest / NK, ay = dense_to_a(rest - f * NK, N, KD);
  const int kz = kt * T + c;
  const bool valid = kz <= KD;
  const float2* src = a + f * MW + (long long)ay * HW + kz;
  float2 v[G];
#pragma unroll
  for (int m = 0; m < G; ++m) v[m] = valid ? src[(long long)(j + m * S) * N * HW] : make_float2(0.f, 0.f);
  fft_line<N, G, -1>(v, j, ColX<T>{sms, c}, tw);
  if (valid) {
    float2* dst = out + f * MM + (long long)ay * H1 + kz;
#pragma unroll
    for (int m = 0; m < G; ++m) {
      const int pos = j + m * S;
      if (kept_xy(pos, N, KD)) dst[(long long)pos * N * H1] = cscale(v[m], scale);
    }
  }
}

// (u . grad) u_g of one giver on the kept modes: u -> out (rows of n/2 + 1)
template <int N>
static cudaError_t shell_advect_n(fftk_plan p, const float2* u, const float* ur, const ShellRange& sh, float2* out,
                                  cudaStream_t st) {
  using X = NXCfg<N>;
  using Z = NZCfg<N>;
  static PerDevice once;
  const cudaError_t e = once.run([](int) {
    const int sx = (int)X::SMEM;
    cudaError_t err = cudaFuncSetAttribute(k_shell_invx<N>, cudaFuncAttributeMaxDynamicSharedMemorySize, sx);
    if (err == cudaSuccess)
      err = cudaFuncSetAttribute(k_shell_invy<N>, cudaFuncAttributeMaxDynamicSharedMemorySize, sx);
    if (err == cudaSuccess)
      err = cudaFuncSetAttribute(k_shell_fwdx<N>, cudaFuncAttributeMaxDynamicSharedMemorySize, sx);
    if (err == cudaSuccess)
      err = cudaFuncSetAttribute(k_shell_z<N>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)SZCfg3<N>::SMEM);
    return err;
  });
  if (e != cudaSuccess) return e;
  constexpr int KD = (N - 1) / 3, KT = (KD + X::T) / X::T;
  const int kt = (sh.kb + X::T) / X::T;  // tiles of kb + 1 columns
  const float2* tw = twiddles(p, N);
  float2* A = p->ns->w;
  float2* B = p->ns->w2;
  {
    LaunchScope ls(p, KK_X_INV, st);
    launch_pdl(k_shell_invx<N>, 3 * (2 * sh.kb + 1) * kt, X::THREADS, X::SMEM, st, u, A, sh, kt, tw);
  }
  {
    LaunchScope ls(p, KK_Y_INV, st);
    launch_pdl(k_shell_invy<N>, 6 * N * kt, X::THREADS, X::SMEM, st, A, B, sh.kb, kt, tw);
  }
  {
    LaunchScope ls(p, KK_AUX, st);
    launch_pdl(k_shell_z<N>, (unsigned)(((long long)N * N + Z::LPC - 1) / Z::LPC), Z::THREADS, SZCfg3<N>::SMEM, st, A,
               B, ur, sh.kb, tw);
  }
  const cudaError_t ey = ns_ypass(p, A, A, 3, -1, KK_Y_FWD, st);
  if (ey != cudaSuccess) return ey;
  {
    LaunchScope ls(p, KK_X_FWD, st);
    launch_pdl(k_shell_fwdx<N>, 3 * (2 * KD + 1) * KT, X::THREADS, X::SMEM, st, A, out, KT,
               (float)(1.0 / ((double)N * N * N)), tw);
  }
  return cudaGetLastError();
}

static cudaError_t shell_advect(fftk_plan p, const float2* u, const float* ur, const ShellRange& sh, float2* out,
                                cudaStream_t st) {
  switch (p->nx) {
#define CASE(n) \
  case n:       \
    return shell_advect_n<n>(p, u, ur, sh, out, st);
    CASE(8) CASE(16) CASE(32) CASE(64) CASE(128) CASE(256) CASE(512) CASE(1024)
#undef CASE
  }
  return cudaErrorInvalidValue;
}

}  // namespace fftk

using namespace fftk;

extern "C" fftk_status tarang_shell_transfer(fftk_plan p, const void* uhat, int nshells, const int* bounds,
                                             double* out_host, void* cuda_stream) {
  if (!p || !uhat || !bounds || !out_host || misaligned16(uhat)) return FFTK_ERR_INVALID_ARG;
  if (p->nx != p->ny || p->nx != p->nz || p->nx < 8 || p->nx > 1024 || !is_pow2(p->nx)) return FFTK_ERR_UNSUPPORTED_SIZE;
  const int kmax = ns_kmax(p->nx);
  if (nshells < 1 || nshells > kmax + 1 || bounds[0] < 0 || bounds[nshells] > kmax + 1)
    return FFTK_ERR_INVALID_ARG;
  for (int i = 0; i < nshells; ++i)
    if (bounds[i + 1] <= bounds[i]) return FFTK_ERR_INVALID_ARG;
  fftk_status st0 = ns_ensure(p);
  if (st0 != FFTK_OK) return st0;
  cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
  NSWork* s = p->ns;
  const NSGeom g = s->g;
  const long long R = (long long)g.n * g.n * g.n;
  const int nb = s->kmax + 1, width = 2 + nb;
  cudaError_t e = ns_second_workspace(p);
  if (e == cudaSuccess && !s->r3) {
    e = cudaMalloc(&s->r3, sizeof(float) * 3 * (size_t)R);
    if (e != cudaSuccess) s->r3 = nullptr;
  }
  if (e == cudaSuccess && s->sout_rows < nshells) {
    cudaFree(s->sout);
    s->sout = nullptr;
    s->sout_rows = 0;
    e = cudaMalloc(&s->sout, sizeof(double) * (size_t)nshells * width);
    if (e == cudaSuccess)
      s->sout_rows = nshells;
    else
      s->sout = nullptr;
  }
  if (e != cudaSuccess) {
    cudaGetLastError();
    return e == cudaErrorMemoryAllocation ? FFTK_ERR_OOM : FFTK_ERR_CUDA;
  }
  const float2* u = static_cast<const float2*>(uhat);
  // the largest nint|k| among the kept modes: givers beyond it are empty
  const int kd = g.kd;
  const int kfar = (int)std::floor(std::sqrt(3.0 * kd * kd) + 0.5);
  if (fftk_c2r(p, u, s->r3, 3, cuda_stream) != FFTK_OK) return FFTK_ERR_CUDA;
  std::vector<char> live(nshells, 0);
  for (int gi = 0; gi < nshells && e == cudaSuccess; ++gi) {
    const int lo = bounds[gi], hi = bounds[gi + 1];
    if (lo > kfar) continue;
    live[gi] = 1;
    const ShellRange sh{lo > 0 ? lo * lo - lo + 1 : 0, hi * hi - hi, hi - 1 < kd ? hi - 1 : kd};
    e = shell_advect(p, u, s->r3, sh, s->u1, st);
    if (e == cudaSuccess) e = diag_launch(p, u, s->u1, 0.0, st, 3, s->sout + (size_t)gi * width);
  }
  std::vector<double> h((size_t)nshells * width, 0.0);
  if (e == cudaSuccess)
    e = cudaMemcpyAsync(h.data(), s->sout, sizeof(double) * h.size(), cudaMemcpyDeviceToHost, st);
  if (e == cudaSuccess) e = cudaStreamSynchronize(st);
  if (e != cudaSuccess) return from_cuda(e);
  // T[r][g] = -sum over the receiver's integer shells of w Re(conj(u) . (u . grad) u_g)
  bool finite = true;
  for (int r = 0; r < nshells; ++r)
    for (int gi = 0; gi < nshells; ++gi) {
      double t = 0.0;
      if (live[gi])
        for (int K = bounds[r]; K < bounds[r + 1]; ++K) t -= h[(size_t)gi * width + 2 + K];
      out_host[(size_t)r * nshells + gi] = t;
      finite = finite && std::isfinite(t);
    }
  return finite ? FFTK_OK : FFTK_ERR_NONFINITE;
}
