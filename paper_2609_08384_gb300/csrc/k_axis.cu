// y-pass and tau-pass instantiations and dispatch.
#include <cmath>
#include <vector>

#include "kernels.cuh"
#include "launch_cfg.h"

namespace brahms {

template <int N, bool INV>
static cudaError_t launch_ypass(const AxisArgs& a, cudaStream_t s) {
  using PL = AxisPlan<N, 1>;
  constexpr int TPC = tiles_per_cta<PL>();
  constexpr int THREADS = TPC * tile_threads<PL>();
  const size_t smem = (size_t)ypass_smem_floats2<PL, INV>() * sizeof(float2);
  static SmemOnce once;
  cudaError_t e = raise_smem_limit(ypass_kernel<PL, INV>, smem, once);
  if (e != cudaSuccess) return e;
  const long long grid = (a.ntiles + TPC - 1) / TPC;
  if (grid <= 0) return cudaSuccess;
  return launch_chained(ypass_kernel<PL, INV>, dim3((unsigned)grid), THREADS, smem, s, a);
}

// The pipelined tau-pass: one wave of persistent CTAs over tiles of its own width.
template <class PL, bool SCALED>
static cudaError_t launch_tprop_pipe(const AxisArgs& a0, cudaStream_t s) {
  constexpr int TX = tau_pipe_cols<PL>();
  constexpr size_t smem = (size_t)tau_pipe_smem<PL>();
  static SmemOnce once;
  cudaError_t e = raise_smem_limit(tpass_pipe_kernel<PL, SCALED>, smem, once);
  if (e != cudaSuccess || a0.ntiles <= 0) return e;
  AxisArgs a = a0;
  const long long lines = a0.ntiles / a0.xtiles;  // (field, y) lines
  a.xtiles = (a0.nx + TX - 1) / TX;
  a.ntiles = lines * a.xtiles;
  const long long wave = 152 * tau_pipe_ctas<PL>();
  const long long grid = a.ntiles < wave ? a.ntiles : wave;
  return launch_chained(tpass_pipe_kernel<PL, SCALED>, dim3((unsigned)grid), tau_pipe_threads<PL>(), smem, s, a);
}

template <int N, bool SCALED>
static cudaError_t launch_tprop(const AxisArgs& a, cudaStream_t s) {
  using PL = TauPlan<N>;
  if constexpr (tau_pipe<PL>()) {
    return launch_tprop_pipe<PL, SCALED>(a, s);
  } else {
    constexpr int TPC = tiles_per_cta<PL>();
    constexpr int THREADS = TPC * tile_threads<PL>();
    const size_t smem = (size_t)axis_smem_floats2<PL>() * sizeof(float2);
    static SmemOnce once;
    cudaError_t e = raise_smem_limit(tpass_prop_kernel<PL, SCALED>, smem, once);
    if (e != cudaSuccess) return e;
    const long long grid = (a.ntiles + TPC - 1) / TPC;
    if (grid <= 0) return cudaSuccess;
    return launch_chained(tpass_prop_kernel<PL, SCALED>, dim3((unsigned)grid), THREADS, smem, s, a);
  }
}

cudaError_t run_ypass(int ny, bool inv, const AxisArgs& a, cudaStream_t s) {
  switch (ny) {
#define BRAHMS_A_CASE(N) \
  case N:                \
    return inv ? launch_ypass<N, true>(a, s) : launch_ypass<N, false>(a, s);
    BRAHMS_FOR_EACH_SIZE(BRAHMS_A_CASE)
#undef BRAHMS_A_CASE
    default:
      return cudaErrorInvalidValue;
  }
}

cudaError_t run_tpass_prop(int nt, const AxisArgs& a, cudaStream_t s) {
  switch (nt) {
#define BRAHMS_T_CASE(N)                                       \
  case N:                                                      \
    if constexpr ((N & (N - 1)) == 0)                          \
      if (!a.scaled) return launch_tprop<N, false>(a, s); \
    return launch_tprop<N, true>(a, s);
    BRAHMS_FOR_EACH_SIZE(BRAHMS_T_CASE)
#undef BRAHMS_T_CASE
    default:
      return cudaErrorInvalidValue;
  }
}

int tw_table_size_of(int n, int axis) {
  switch (n) {
#define BRAHMS_W_CASE(N) \
  case N:                \
    return axis == 0   ? tw_table_size<AxisPlan<N, 0>>()  \
           : axis == 1 ? tw_table_size<AxisPlan<N, 1>>()  \
                       : tw_table_size<AxisPlan<N, 2>>();
    BRAHMS_FOR_EACH_SIZE(BRAHMS_W_CASE)
#undef BRAHMS_W_CASE
    default:
      return 0;
  }
}

template <class PL>
static int radices(int* r) {
  for (int p = 0; p < PL::NP; ++p) r[p] = PL::r(p);
  return PL::NP;
}
static int plan_radices(int n, int axis, int* r) {
  switch (n) {
#define BRAHMS_R_CASE(N) \
  case N:                \
    return axis == 0 ? radices<AxisPlan<N, 0>>(r) : axis == 1 ? radices<AxisPlan<N, 1>>(r) : radices<AxisPlan<N, 2>>(r);
    BRAHMS_FOR_EACH_SIZE(BRAHMS_R_CASE)
#undef BRAHMS_R_CASE
    default:
      return 0;
  }
}

static int centred(int d, int n) { return d >= (n + 1) / 2 ? d - n : d; }

static float2 entry(double phi, const float2*) { return make_float2((float)-std::tan(0.5 * phi), (float)std::sin(phi)); }
static float4 entry(double phi, const float4*) {
  const double c = std::cos(phi), sn = std::sin(phi);
  const float ch = (float)c, sh = (float)sn;
  return make_float4(ch, sh, (float)(c - (double)ch), (float)(sn - (double)sh));
}

// Per-pass twiddle blocks (the layout of tw_pass_off): for each pass P >= 1 with
// radix R after stride NS, entries [r][m] = the shears (-tan(phi/2), sin(phi)) of
// phi = -2 pi r' m' / (NS R), or its cosine and sine as hi + lo, the digits of r and m
// centred, evaluated in FP64.
template <class T>
static bool fill(T* h, int n, int axis) {
  int rad[8];
  const int np = plan_radices(n, axis, rad);
  if (np <= 0) return false;
  h[0] = entry(0.0, h);  // a plan of one pass has no turns
  int ns = 1;
  for (int q = 0; q < np; ++q) {
    if (q > 0) {
      for (int r = 0; r < rad[q]; ++r)
        for (int m = 0; m < ns; ++m) {
          int mc = 0, w = 1, rest = m;
          for (int p = 0; p < q; ++p) {
            mc += w * centred(rest % rad[p], rad[p]);
            rest /= rad[p];
            w *= rad[p];
          }
          *h = entry(-6.283185307179586476925286766559 * (double)(centred(r, rad[q]) * mc) / (double)(ns * rad[q]), h);
          ++h;
        }
    }
    ns *= rad[q];
  }
  return true;
}
bool fill_twiddles(float2* h, int n, int axis) { return fill(h, n, axis); }
bool fill_twiddles(float4* h, int n, int axis) { return fill(h, n, axis); }
cudaError_t upload_twiddles(float2* tw, int n, int axis, cudaStream_t s) {
  std::vector<float2> h((size_t)tw_table_size_of(n, axis));
  if (h.empty() || !fill_twiddles(h.data(), n, axis)) return cudaErrorInvalidValue;
  const cudaError_t e = cudaMemcpyAsync(tw, h.data(), sizeof(float2) * h.size(), cudaMemcpyHostToDevice, s);
  if (e != cudaSuccess) return e;
  return cudaStreamSynchronize(s);  // h is a local buffer
}

int tau_col_tile_of(int n) {
  switch (n) {
#define BRAHMS_TC_CASE(N) \
  case N:                 \
    return ColTile<TauPlan<N>>::value;
    BRAHMS_FOR_EACH_SIZE(BRAHMS_TC_CASE)
#undef BRAHMS_TC_CASE
    default:
      return 0;
  }
}

int col_tile_of(int n) {
  switch (n) {
#define BRAHMS_C_CASE(N) \
  case N:                \
    return ColTile<ColPlan<N>>::value;
    BRAHMS_FOR_EACH_SIZE(BRAHMS_C_CASE)
#undef BRAHMS_C_CASE
    default:
      return 0;
  }
}

}  // namespace brahms
