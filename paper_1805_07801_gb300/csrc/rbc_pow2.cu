// The fused convection passes (rbc_passes.cuh) for powers of two.
#include "rbc_passes.cuh"

namespace fftk {

cudaError_t rbc_invx(fftk_plan p, const float2* x, bool padded, float2* w, cudaStream_t st) {
  switch (p->nx) {
#define CASE(n) \
  case n:       \
    return rbc_invx_n<n>(p, x, padded, w, st);
    CASE(8) CASE(16) CASE(32) CASE(64) CASE(128) CASE(256) CASE(512) CASE(1024)
#undef CASE
    default:
      return rbc_invx3(p, x, padded, w, st);
  }
}

cudaError_t rbc_z(fftk_plan p, float2* w, const RBCSlots& sl, cudaStream_t st) {
  switch (p->nx) {
#define CASE(n) \
  case n:       \
    return rbc_z_n<n>(p, w, sl, st);
    CASE(8) CASE(16) CASE(32) CASE(64) CASE(128) CASE(256) CASE(512) CASE(1024)
#undef CASE
    default:
      return rbc_z3(p, w, sl, st);
  }
}

cudaError_t rbc_fwdx(fftk_plan p, const RBCStage& s, cudaStream_t st) {
  switch (p->nx) {
#define CASE(n) \
  case n:       \
    return rbc_fwdx_n<n>(p, s, st);
    CASE(8) CASE(16) CASE(32) CASE(64) CASE(128) CASE(256) CASE(512) CASE(1024)
#undef CASE
    default:
      return rbc_fwdx3(p, s, st);
  }
}

}  // namespace fftk
