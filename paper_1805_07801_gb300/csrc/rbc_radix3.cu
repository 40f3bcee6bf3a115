// The fused convection passes (rbc_passes.cuh) for cubes of 3 * 2^m points.
#include "rbc_passes.cuh"

namespace fftk {

cudaError_t rbc_invx3(fftk_plan p, const float2* x, bool padded, float2* w, cudaStream_t st) {
  switch (p->nx) {
#define CASE(n) \
  case n:       \
    return rbc_invx_n<n>(p, x, padded, w, st);
    CASE(12) CASE(24) CASE(48) CASE(96) CASE(192) CASE(384) CASE(768)
#undef CASE
  }
  return cudaErrorInvalidValue;
}

cudaError_t rbc_z3(fftk_plan p, float2* w, const RBCSlots& sl, cudaStream_t st) {
  switch (p->nx) {
#define CASE(n) \
  case n:       \
    return rbc_z_n<n>(p, w, sl, st);
    CASE(12) CASE(24) CASE(48) CASE(96) CASE(192) CASE(384) CASE(768)
#undef CASE
  }
  return cudaErrorInvalidValue;
}

cudaError_t rbc_fwdx3(fftk_plan p, const RBCStage& s, cudaStream_t st) {
  switch (p->nx) {
#define CASE(n) \
  case n:       \
    return rbc_fwdx_n<n>(p, s, st);
    CASE(12) CASE(24) CASE(48) CASE(96) CASE(192) CASE(384) CASE(768)
#undef CASE
  }
  return cudaErrorInvalidValue;
}

}  // namespace fftk
