// Plane pass of two fields: instantiations, and the dispatch.
#include "plane.cuh"

namespace brahms {

cudaError_t run_plane(int nx, int ny, int nf, const XPassArgs& a, const float2* twy, cudaStream_t s) {
  if (nf == 3) return run_plane3(nx, ny, a, twy, s);
#define BRAHMS_PL_CASE(X, Y) \
  if (nx == X && ny == Y) return launch_plane<X, Y, 2>(a, twy, s);
  BRAHMS_FOR_EACH_PLANE(BRAHMS_PL_CASE)
#undef BRAHMS_PL_CASE
  return cudaErrorInvalidValue;
}

bool plane_supported(int nx, int ny) {
#define BRAHMS_PS_CASE(X, Y) \
  if (nx == X && ny == Y) return true;
  BRAHMS_FOR_EACH_PLANE(BRAHMS_PS_CASE)
#undef BRAHMS_PS_CASE
  return false;
}

}  // namespace brahms
