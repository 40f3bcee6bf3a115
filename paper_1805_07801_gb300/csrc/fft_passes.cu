// The 1D passes of the 3D transform for power-of-two lines
// (fft_pass_kernels.cuh) and their dispatch.

// these passes are bound by their 8-byte global accesses; scalar FP32 sums
// measured faster here than the paired ones (see fft_engine.cuh)
#define FFTK_PAIRED_FP32 0
#include "fft_pass_kernels.cuh"

namespace fftk {

#define FFTK_SIZES(X) X(2) X(4) X(8) X(16) X(32) X(64) X(128) X(256) X(512) X(1024) X(2048) X(4096)

cudaError_t launch_z_r2c(fftk_plan p, const float* in, float2* out, long long nlines, float scale,
                         cudaStream_t st) {
  if (nlines <= 0) return cudaSuccess;
  if (!is_pow2(p->nz)) return launch_z3(p, true, in, out, nlines, scale, st);
  switch (p->nz) {
#define CASE(n) \
  case n:       \
    return z_r2c_n<n>(p, in, out, nlines, scale, st);
    FFTK_SIZES(CASE)
#undef CASE
  }
  return cudaErrorInvalidValue;
}

cudaError_t launch_z_c2r(fftk_plan p, const float2* in, float* out, long long nlines,
                         cudaStream_t st) {
  if (nlines <= 0) return cudaSuccess;
  if (!is_pow2(p->nz)) return launch_z3(p, false, in, out, nlines, 1.f, st);
  switch (p->nz) {
#define CASE(n) \
  case n:       \
    return z_c2r_n<n>(p, in, out, nlines, st);
    FFTK_SIZES(CASE)
#undef CASE
  }
  return cudaErrorInvalidValue;
}

cudaError_t launch_cpass(fftk_plan p, int L, int sign, const float2* in, float2* out, long long P,
                         long long Q, float scale, int kind, cudaStream_t st) {
  if (P <= 0 || Q <= 0) return cudaSuccess;
  if (sign < 0) {
    switch (L) {
#define CASE(n) \
  case n:       \
    return cpass_l<n, -1>(p, in, out, P, Q, scale, kind, st);
      FFTK_SIZES(CASE)
#undef CASE
    }
  } else {
    switch (L) {
#define CASE(n) \
  case n:       \
    return cpass_l<n, +1>(p, in, out, P, Q, scale, kind, st);
      FFTK_SIZES(CASE)
#undef CASE
    }
  }
  return cudaErrorInvalidValue;
}

}  // namespace fftk
