// Plane pass: for grids whose whole (x, y) plane of all fields fits in shared
// memory, the y-inverse, the x-pass and the y-forward of a z-step are one kernel,
// one CTA per tau-plane, so that a step is two passes over the fields (this one
// and the tau-pass) instead of four.
//
// The CTA's threads take the plane's columns (y transforms, the exchanges in the
// plane's own buffer), then its rows (inverse x transform, park, the RK4 half
// steps, forward x transform: the x-pass's steps, see kernels.cuh), then its
// columns again.  Fields go from and to global memory in the column phases,
// straight from and to registers, 8 bytes a lane along x.
#pragma once

#include "kernels.cuh"
#include "launch_cfg.h"

namespace brahms {

constexpr int kPlaneThreads = 256;

// Resident CTAs asked for: two (every plane fits), four (64 registers) where a row is
// one thread's, as the compiler took by itself with fewer stage factors (62 registers;
// at 66 a step of 3 x 16x16x512 takes 17.6 us instead of 13.5).
template <int NX>
__host__ __device__ constexpr int plane_min_blocks() { return FftPlan<NX>::T == 1 ? 4 : 2; }

// one column of a plane buffer whose rows are PITCH apart
template <int PITCH>
struct XchPlane {
  static constexpr bool kSplit = false;
  float2* base;
  __device__ __forceinline__ void st(int pos, float2 v) const { base[pos * PITCH] = v; }
  __device__ __forceinline__ float2 ld(int pos) const { return base[pos * PITCH]; }
};

template <int NX, int NY>
__host__ __device__ constexpr int plane_smem(int nf) {
  return nf * NY * XchRow::pitch(NX) * (int)sizeof(float2);
}

// The plan of the columns: the y axis's own, whose twiddle table the launch is given
// (another plan of the same length would read its entries in another order).
template <int NY>
using PlaneColumnPlan = AxisPlan<NY, 1>;

// Columns of all fields: from global memory (or the buffer) through one
// transform along y into the buffer (or global memory).
template <int NX, int NY, int F, bool INV>
__device__ __forceinline__ void plane_columns(float2* buf, float2* data, long long fstride, const float2* twy) {
  using PL = PlaneColumnPlan<NY>;
  constexpr int PITCH = XchRow::pitch(NX);
  constexpr int COLS = kPlaneThreads / PL::T;  // columns at a time
  constexpr int R0 = fft_radix<PL, INV>(0), RL = fft_radix<PL, INV>(PL::NP - 1);
  const int t = threadIdx.x / COLS;
#pragma unroll 1
  for (int c0 = 0; c0 < F * NX; c0 += COLS) {
    const int c = c0 + threadIdx.x % COLS;
    const bool act = c < F * NX;
    const int f = act ? c / NX : 0, x = act ? c % NX : 0;
    float2* col = buf + f * NY * PITCH + x;
    float2* glob = data + f * fstride + x;
    const XchPlane<PITCH> xc{col};
    float2 v[PL::E];
#pragma unroll
    for (int b = 0; b < PL::E / R0; ++b)
#pragma unroll
      for (int r = 0; r < R0; ++r) {
        const int pos = pos_first<PL, INV>(t + b * PL::T, r);
        v[b * R0 + r] = !act ? make_float2(0.f, 0.f) : INV ? __ldcg(glob + pos * NX) : col[pos * PITCH];
      }
    if constexpr (PL::NP == 1) {
      dft<R0, INV>(v);
    } else {
      // an inactive thread's exchanges stay off the buffer
      fft_run<PL, INV, 0, XchGuard<XchPlane<PITCH>>, SyncBlock, TwGlobal>(v, t, XchGuard<XchPlane<PITCH>>{xc, act},
                                                                          TwGlobal{twy});
    }
    __syncthreads();  // the column's last exchange has been read
    if (act) {
#pragma unroll
      for (int b = 0; b < PL::E / RL; ++b)
#pragma unroll
        for (int r = 0; r < RL; ++r) {
          const int pos = pos_last<PL, INV>(t + b * PL::T, r);
          if constexpr (INV) col[pos * PITCH] = v[b * RL + r];
          else glob[pos * NX] = v[b * RL + r];
        }
    }
  }
}

// The pass on one tau-plane; data: the plane of field 0.
template <int NX, int NY, int F>
__device__ __forceinline__ void plane_tile(const XPassArgs& p, float2* data, const float2* coef, const float2* twy,
                                           float2* buf) {
  using PL = FftPlan<NX>;
  constexpr int PITCH = XchRow::pitch(NX), E = PL::E, T = PL::T;
  constexpr int ROWS = kPlaneThreads / T;  // rows at a time
  constexpr int RF0 = fft_radix<PL, false>(0), RFL = fft_radix<PL, false>(PL::NP - 1);
  static_assert(xpass_warp_sync<NX>(), "a row's threads lie in one warp");
  const TwGlobal tw{p.tw};
  const int mode = p.mode;
  if (mode != XM_NL_FIRST) {
    plane_columns<NX, NY, F, true>(buf, data, p.fstride, twy);
    __syncthreads();
  }
  const int t = threadIdx.x % T;
  const Stages<false> B = stages_of(coef), A = stages_of(coef + 3);
#pragma unroll 1
  for (int y0 = 0; y0 < NY; y0 += ROWS) {
    const int y = y0 + threadIdx.x / T;
    if (y >= NY) continue;  // whole rows: a row's threads stay together
    float2* row = buf + y * PITCH;  // field f at row + f NY PITCH
#pragma unroll 1
    for (int f = 0; f < F; ++f) {
      float2* my = row + f * NY * PITCH;
      const XchRow xr{my};
      float2 v[E];
      if (mode != XM_NL_FIRST) {
#pragma unroll
        for (int b = 0; b < E / RFL; ++b)
#pragma unroll
          for (int r = 0; r < RFL; ++r) v[b * RFL + r] = my[pos_first<PL, true>(t + b * T, r)];
        fft_run<PL, true, 0, XchRow, SyncRow<T>, TwGlobal>(v, t, xr, tw);
      } else {
        const float2* src = data + f * p.fstride + y * NX;
#pragma unroll
        for (int b = 0; b < E / RF0; ++b)
#pragma unroll
          for (int r = 0; r < RF0; ++r) v[b * RF0 + r] = __ldcg(src + pos_first<PL, false>(t + b * T, r));
      }
      SyncRow<T>::sync();
      park<PL>(my, t, v);
    }
#pragma unroll 1
    for (int q = 0; q < E / 2; ++q) {
      Pair a[F];
#pragma unroll
      for (int f = 0; f < F; ++f) {
        const float4 w = *park_place<PL>(row + f * NY * PITCH, t, q);
        a[f] = {make_float2(w.x, w.y), make_float2(w.z, w.w)};
      }
      if (mode != XM_NL_FIRST) rk4<F>(a, B, p.kh, p.kh2);
      if (mode != XM_NL_LAST) rk4<F>(a, A, p.kh, p.kh2);
#pragma unroll
      for (int f = 0; f < F; ++f)
        *park_place<PL>(row + f * NY * PITCH, t, q) = make_float4(a[f].re.x, a[f].re.y, a[f].im.x, a[f].im.y);
    }
#pragma unroll 1
    for (int f = 0; f < F; ++f) {
      float2* my = row + f * NY * PITCH;
      const XchRow xr{my};
      float2 v[E];
      unpark<PL>(my, t, v);
      if (mode == XM_NL_LAST) {
        float2* dst = data + f * p.fstride + y * NX;
#pragma unroll
        for (int b = 0; b < E / RF0; ++b)
#pragma unroll
          for (int r = 0; r < RF0; ++r) dst[pos_first<PL, false>(t + b * T, r)] = v[b * RF0 + r];
      } else {
        fft_run<PL, false, 0, XchRow, SyncRow<T>, TwGlobal>(v, t, xr, tw);
        SyncRow<T>::sync();
#pragma unroll
        for (int b = 0; b < E / RFL; ++b)
#pragma unroll
          for (int r = 0; r < RFL; ++r) my[pos_last<PL, false>(t + b * T, r)] = v[b * RFL + r];
      }
    }
  }
  if (mode != XM_NL_LAST) {
    __syncthreads();
    plane_columns<NX, NY, F, false>(buf, data, p.fstride, twy);
  }
}

template <int NX, int NY, int F>
__global__ void __launch_bounds__(kPlaneThreads, plane_min_blocks<NX>()) plane_kernel(const XPassArgs p, const float2* twy) {
  extern __shared__ float4 sm4[];
  chain_begin();
  plane_tile<NX, NY, F>(p, p.data + (long long)blockIdx.x * NX * NY, p.ecoef, twy, reinterpret_cast<float2*>(sm4));
}

template <int NX, int NY, int F>
cudaError_t launch_plane(const XPassArgs& a0, const float2* twy, cudaStream_t s) {
  XPassArgs a = a0;
  fill_stage_factors(a);
  constexpr size_t smem = (size_t)plane_smem<NX, NY>(F);
  static SmemOnce once;
  const cudaError_t e = raise_smem_limit(plane_kernel<NX, NY, F>, smem, once);
  if (e != cudaSuccess) return e;
  return launch_chained(plane_kernel<NX, NY, F>, dim3((unsigned)(a.rows / NY)), kPlaneThreads, smem, s, a, twy);
}

}  // namespace brahms
