// Single transforms of the fields, one axis at a time: what brahms_transform and the
// spectral-phase gradient call.  Nothing takes these transforms back, so their turns
// are products with hi + lo floats (TwProduct) where those of a z-step are shears that
// its inverse transforms undo.  Forward error against FP64 of 64 columns of 16, 256 and
// 4096 random points 9.8e-8, 1.16e-7 and 1.34e-7; by shears 1.05e-7, 1.27e-7, 1.47e-7.
#include "kernels.cuh"
#include "launch_cfg.h"

namespace brahms {

template <int NX, bool INV>
__global__ void __launch_bounds__(xpass_threads<NX>()) xline_kernel(const XLineArgs p) {
  using PL = FftPlan<NX>;
  constexpr int E = PL::E, T = PL::T, ROWS = xpass_rows<NX>();
  constexpr int R0 = fft_radix<PL, INV>(0), RL = fft_radix<PL, INV>(PL::NP - 1);
  using SY = typename std::conditional<xpass_warp_sync<NX>(), SyncWarp, SyncBlock>::type;
  extern __shared__ float4 sm4[];
  const int t = threadIdx.x % T, rl = threadIdx.x / T;
  const long long row = (long long)blockIdx.x * ROWS + rl;
  const bool act = row < p.rows;
  const XchRow xr{reinterpret_cast<float2*>(sm4) + rl * XchRow::pitch(NX)};
  float2* line = p.data + (act ? row : 0) * NX;
  chain_begin();
  float2 v[E];
#pragma unroll
  for (int b = 0; b < E / R0; ++b)
#pragma unroll
    for (int r = 0; r < R0; ++r)
      v[b * R0 + r] = act ? __ldcg(line + pos_first<PL, INV>(t + b * T, r)) : make_float2(0.f, 0.f);
  fft_run<PL, INV, 0, XchRow, SY, TwProduct>(v, t, xr, TwProduct{p.twp});
  if (!act) return;
#pragma unroll
  for (int b = 0; b < E / RL; ++b)
#pragma unroll
    for (int r = 0; r < RL; ++r) {
      float2 w = v[b * RL + r];
      if constexpr (INV) w = __ffma2_rn(w, dup(p.scale), __fmul2_rn(w, dup(p.scale_lo)));
      line[pos_last<PL, INV>(t + b * T, r)] = w;
    }
}

template <int NX, bool INV>
static cudaError_t launch_xline(const XLineArgs& a, cudaStream_t s) {
  constexpr size_t smem = (size_t)xpass_smem_floats2<NX>(1) * sizeof(float2);
  static SmemOnce once;
  const cudaError_t e = raise_smem_limit(xline_kernel<NX, INV>, smem, once);
  const long long grid = (a.rows + xpass_rows<NX>() - 1) / xpass_rows<NX>();
  if (e != cudaSuccess || grid <= 0) return e;
  return launch_chained(xline_kernel<NX, INV>, dim3((unsigned)grid), xpass_threads<NX>(), smem, s, a);
}

cudaError_t run_xline_fft(int nx, bool inv, const XLineArgs& a, cudaStream_t s) {
  switch (nx) {
#define BRAHMS_XL_CASE(N) \
  case N:                 \
    return inv ? launch_xline<N, true>(a, s) : launch_xline<N, false>(a, s);
    BRAHMS_FOR_EACH_SIZE(BRAHMS_XL_CASE)
#undef BRAHMS_XL_CASE
    default:
      return cudaErrorInvalidValue;
  }
}

template <class PL, bool INV, int AXIS>
__global__ void __launch_bounds__(tiles_per_cta<PL>() * tile_threads<PL>()) axis_fft_kernel(const AxisArgs p) {
  extern __shared__ float4 sm4[];
  chain_begin();
  axis_tile<PL, INV, AXIS, tiles_per_cta<PL>() * tile_threads<PL>()>(p, blockIdx.x, TwProduct{p.twp},
                                                                    reinterpret_cast<float2*>(sm4));
}

template <int N, bool INV, int AXIS>
static cudaError_t launch_axis(const AxisArgs& a, cudaStream_t s) {
  using PL = AxisPlan<N, AXIS>;
  constexpr int TPC = tiles_per_cta<PL>();
  constexpr size_t smem = (size_t)(TPC * PL::N * ColTile<PL>::value) * sizeof(float2);
  static SmemOnce once;
  const cudaError_t e = raise_smem_limit(axis_fft_kernel<PL, INV, AXIS>, smem, once);
  const long long grid = (a.ntiles + TPC - 1) / TPC;
  if (e != cudaSuccess || grid <= 0) return e;
  return launch_chained(axis_fft_kernel<PL, INV, AXIS>, dim3((unsigned)grid), TPC * tile_threads<PL>(), smem, s, a);
}

cudaError_t run_axis_fft(int n, int axis, bool inv, const AxisArgs& a, cudaStream_t s) {
  switch (n) {
#define BRAHMS_A_CASE(N)                                                                        \
  case N:                                                                                       \
    if (axis == 1) return inv ? launch_axis<N, true, 1>(a, s) : launch_axis<N, false, 1>(a, s); \
    return inv ? launch_axis<N, true, 2>(a, s) : launch_axis<N, false, 2>(a, s);
    BRAHMS_FOR_EACH_SIZE(BRAHMS_A_CASE)
#undef BRAHMS_A_CASE
    default:
      return cudaErrorInvalidValue;
  }
}

}  // namespace brahms
