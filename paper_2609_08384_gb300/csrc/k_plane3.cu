// Plane pass of three fields: instantiations (a translation unit of their own so
// that they compile beside those of two fields).
#include "plane.cuh"

namespace brahms {

cudaError_t run_plane3(int nx, int ny, const XPassArgs& a, const float2* twy, cudaStream_t s) {
#define BRAHMS_PL_CASE(X, Y) \
  if (nx == X && ny == Y) return launch_plane<X, Y, 3>(a, twy, s);
  BRAHMS_FOR_EACH_PLANE(BRAHMS_PL_CASE)
#undef BRAHMS_PL_CASE
  return cudaErrorInvalidValue;
}

}  // namespace brahms
