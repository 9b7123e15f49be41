// Grouped plane pass of the batched form: one launch applies the plane pass to
// the planes of every active instance of one grid shape (see k_xgroup.cu for the
// layout and the per-instance tables).
#include "plane.cuh"

namespace brahms {

template <int NX, int NY>
__global__ void __launch_bounds__(kPlaneThreads, plane_min_blocks<NX>())
    plane_group_kernel(const XPassArgs base, const float2* twy, const GroupInst* __restrict__ gi,
                       const float2* __restrict__ ecoef, int stride, int step, int planes) {
  extern __shared__ float4 sm4[];
  chain_begin();
  const int i = (int)(blockIdx.x / (unsigned)planes), k = (int)(blockIdx.x % (unsigned)planes);
  const GroupInst g = gi[i];
  XPassArgs p = base;
  p.dz = g.dz;
  p.kh[0] = g.kh[0];
  p.kh[1] = g.kh[1];
  p.kh2[0] = g.kh2[0];
  p.kh2[1] = g.kh2[1];
  p.mode = step < 0 ? XM_NL_FIRST : (step == g.nz - 1 ? XM_NL_LAST : XM_NL_MID);
  plane_tile<NX, NY, 2>(p, base.data + (long long)i * 2 * base.fstride + (long long)k * NX * NY,
                        ecoef + (long long)i * stride + (step + 1) * kStageFactors, twy, reinterpret_cast<float2*>(sm4));
}

template <int NX, int NY>
static cudaError_t launch_plane_group(const XPassArgs& base, const float2* twy, const GroupInst* gi, const float2* ecoef,
                                      int stride, int step, int ninst, cudaStream_t s) {
  constexpr size_t smem = (size_t)plane_smem<NX, NY>(2);
  static SmemOnce once;
  const cudaError_t e = raise_smem_limit(plane_group_kernel<NX, NY>, smem, once);
  const int planes = (int)(base.rows / NY);
  if (e != cudaSuccess || planes <= 0 || ninst <= 0) return e;
  return launch_chained(plane_group_kernel<NX, NY>, dim3((unsigned)planes * (unsigned)ninst), kPlaneThreads, smem, s, base,
                        twy, gi, ecoef, stride, step, planes);
}

cudaError_t run_plane_group(int nx, int ny, const XPassArgs& base, const float2* twy, const GroupInst* gi,
                            const float2* ecoef, int stride, int step, int ninst, cudaStream_t s) {
#define BRAHMS_PG_CASE(X, Y) \
  if (nx == X && ny == Y) return launch_plane_group<X, Y>(base, twy, gi, ecoef, stride, step, ninst, s);
  BRAHMS_FOR_EACH_PLANE(BRAHMS_PG_CASE)
#undef BRAHMS_PG_CASE
  return cudaErrorInvalidValue;
}

}  // namespace brahms
