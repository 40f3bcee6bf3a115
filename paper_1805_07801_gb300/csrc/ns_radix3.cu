// The fused Navier-Stokes passes on cubes of 3 * 2^m points (the paper's XC40
// runs use 768^3, Sec. 6): the kernels of ns_passes.cuh on lines whose last
// stage takes the factor 3.  768^3 RK2 step: 64.8 ms through the plan's full
// transforms with the products in real space, 30.2 ms fused (384^3: 8.07 and
// 3.24 ms, 96^3: 0.26 and 0.12 ms), 22.1 ms with the y and forward x passes in
// two long-radix stages (ns_ypass.cu, ns_fwdx3.cu) and 24 values per thread in
// the z lines.
#include <mutex>

#include "ns_passes.cuh"

namespace fftk {

cudaError_t ns_rhs_radix3(fftk_plan p, const float2* u, const float2* u0, const float2* u1, float2* out,
                          const NSUpdate& upd, int mode, const float2* extra, cudaStream_t st) {
  switch (p->nx) {
#define CASE(n) \
  case n:       \
    return NSLaunch<n>::rhs(p, u, u0, u1, out, upd, mode, extra, st);
    CASE(12) CASE(24) CASE(48) CASE(96) CASE(192) CASE(384) CASE(768)
#undef CASE
  }
  return cudaErrorInvalidValue;
}

}  // namespace fftk
