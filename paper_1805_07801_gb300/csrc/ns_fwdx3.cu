// The forward x pass of the Navier-Stokes solver (ns_fwdx.cuh) for cubes of 3 * 2^m points.
#include "ns_fwdx.cuh"

namespace fftk {

cudaError_t ns_fwdx3(fftk_plan p, const float2* nh, const float2* u0, const float2* u1, float2* out,
                     const NSUpdate& upd, int mode, const float2* extra, cudaStream_t st) {
  switch (p->nx) {
#define CASE(n) \
  case n:       \
    return fwdx_n<n>(p, nh, u0, u1, out, upd, mode, extra, st);
    CASE(12) CASE(24) CASE(48) CASE(96) CASE(192) CASE(384) CASE(768)
#undef CASE
  }
  return cudaErrorInvalidValue;
}

}  // namespace fftk
