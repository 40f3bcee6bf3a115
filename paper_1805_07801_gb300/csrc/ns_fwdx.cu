// The forward x pass of the Navier-Stokes solver (ns_fwdx.cuh) for powers of two.
#include "ns_fwdx.cuh"

namespace fftk {

cudaError_t ns_fwdx(fftk_plan p, const float2* nh, const float2* u0, const float2* u1, float2* out,
                    const NSUpdate& upd, int mode, const float2* extra, cudaStream_t st) {
  switch (p->nx) {
#define CASE(n) \
  case n:       \
    return fwdx_n<n>(p, nh, u0, u1, out, upd, mode, extra, st);
    CASE(8) CASE(16) CASE(32) CASE(64) CASE(128) CASE(256) CASE(512) CASE(1024)
#undef CASE
    default:
      return ns_fwdx3(p, nh, u0, u1, out, upd, mode, extra, st);
  }
}

}  // namespace fftk
