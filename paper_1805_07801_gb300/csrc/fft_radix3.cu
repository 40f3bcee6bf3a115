// The 1D passes for lines of 3 * 2^m points (the paper's 768^3, 1536^3 and
// 3072^3 grids of the Cray XC40 runs, Sec. 5): the kernels of
// fft_pass_kernels.cuh on lines whose last stage takes the factor 3, with 24
// values per thread (12 for short lines).  Against three sub-lines combined
// through shared memory by a radix-3 step: five fields of 384 x 64 x 192, z
// r2c 168 -> 55 us, c2r 137 -> 55 us (its 3-strided loads and table gathers
// bound it); 768^3 pair 5.94 -> 4.87 ms.
#include "fft_pass_kernels.cuh"

namespace fftk {

cudaError_t launch_cpass3(fftk_plan p, int L, int sign, const float2* in, float2* out, long long P, long long Q,
                          float scale, int kind, cudaStream_t st) {
  if (P <= 0 || Q <= 0) return cudaSuccess;
#define CASE(n)                                                                                   \
  case n:                                                                                         \
    return sign < 0 ? cpass_l<n, -1>(p, in, out, P, Q, scale, kind, st)                           \
                    : cpass_l<n, +1>(p, in, out, P, Q, scale, kind, st);
  switch (L) {
    CASE(6) CASE(12) CASE(24) CASE(48) CASE(96) CASE(192) CASE(384) CASE(768) CASE(1536) CASE(3072)
  }
#undef CASE
  return cudaErrorInvalidValue;
}

cudaError_t launch_z3(fftk_plan p, bool fwd, const void* in, void* out, long long nlines, float scale,
                      cudaStream_t st) {
  if (nlines <= 0) return cudaSuccess;
#define CASE(n)                                                                                                   \
  case n:                                                                                                         \
    return fwd ? z_r2c_n<n>(p, static_cast<const float*>(in), static_cast<float2*>(out), nlines, scale, st)       \
               : z_c2r_n<n>(p, static_cast<const float2*>(in), static_cast<float*>(out), nlines, st);
  switch (p->nz) { CASE(12) CASE(24) CASE(48) CASE(96) CASE(192) CASE(384) CASE(768) CASE(1536) CASE(3072) }
#undef CASE
  return cudaErrorInvalidValue;
}

}  // namespace fftk
