// The reverse x-pass of the adjoint: takes the adjoint through one boundary
// between z-steps (the recording forward x-pass is in k_xrec.cu).
//
// Forward, the x-pass at boundary b (between steps b-1 and b) maps the state
// a2 = L(N_A(A_{b-1})) (after its inverse x-FFT) through N_B of step b-1 to
// A_b and through N_A of step b.  In reverse the same boundary takes the
// adjoint through the inverse x-FFT, the reverse of N_A at A_b, the reverse
// of N_B at a2 and the forward x-FFT -- the structure of the forward x-pass
// with each RK4 replaced by its vector-Jacobian product (rk4_vjp).
// Between two such passes the adjoint of the linear step, IDFT3(conj(P)
// DFT3), runs as the usual y-forward, tau-propagator (conjugated) and
// y-inverse passes.
//
// MAP: under a transverse mismatch map every point has its own stage phases,
// T V^s (s = 0, 1, 2), from the same tables as the forward x-pass.  The
// sensitivities to the stage phases keep their meaning: the map term of
// Phi(x, y, z) does not depend on the per-step mismatch.  Instantiated by
// k_xadj.cu (map-free) and k_xadj_map.cu.
#pragma once

#include "launch_cfg.h"
#include "vjp.cuh"

namespace brahms {

// points 2 q and 2 q + 1 of thread t from a row in place order (as recorded) or in
// row order
template <class PL>
__device__ __forceinline__ float4 load_points(const float2* row, bool row_order, int t, int q) {
  if (!row_order) return __ldcg(reinterpret_cast<const float4*>(row) + q * PL::T + t);
  const float2 a = __ldcg(row + point_pos<PL>(t, 2 * q)), b = __ldcg(row + point_pos<PL>(t, 2 * q + 1));
  return make_float4(a.x, b.x, a.y, b.y);
}

// The tile of the forward x-pass (kernels.cuh: rows by asynchronous copies, parked
// two points together), with the two RK4 half steps in reverse, on two points at a
// time.  The recorded states come in place order, one 16-byte load a field and two
// points.  Backward of the 2 x 128x128x256 state over 36 steps 10.65 -> 10.13 ms (so
// about 14 of 75 us of this pass), 3 x 128x128x256 over 25 steps 11.58 -> 10.79, under
// a map 11.87 -> 11.51 and 12.59 -> 11.74; with all stage factors from FP64 10.28, 10.96,
// 11.59 and 11.83.  What bounds it: the FP32 pipe (196 operations a point and half step
// of two fields) beside 48 B a point and field of memory traffic against the forward
// pass's 16.
template <int NX, int F, int THREADS, bool MAP>
__device__ __forceinline__ void xpass_adj_tile(const XAdjArgs& p, long long tile, float2* rowbuf, float (&sens)[6]) {
  using PL = FftPlan<NX>;
  constexpr int E = PL::E;
  constexpr int T = PL::T;
  constexpr int ROWS = xtile_rows<NX, THREADS>();
  constexpr int PITCH = XchRow::pitch(NX);
  constexpr int RF0 = fft_radix<PL, false>(0);
  constexpr int RFL = fft_radix<PL, false>(PL::NP - 1);
  using SY = typename std::conditional<xpass_warp_sync<NX>(), SyncWarp, SyncBlock>::type;
  static_assert(ROWS >= 1 && ROWS * T == THREADS, "CTA must hold whole rows");
  const TwGlobal tw{p.tw};

  const int t = threadIdx.x % T;
  const int rl = threadIdx.x / T;
  const long long row = tile * ROWS + rl;
  const bool act = row < p.rows;
  float2* myrow = rowbuf + rl * PITCH;

  // 1. every field: load, inverse transform (from k-space), park
#pragma unroll
  for (int f = 0; f < F; ++f) {
    if (act) copy_row<PL>(myrow + f * ROWS * PITCH, p.g + f * p.fstride + row * NX, t);
    cp_async_commit();
  }
#pragma unroll 1
  for (int f = 0; f < F; ++f) {
    const XchRow xr{myrow + f * ROWS * PITCH};
    if (f == F - 1) cp_async_wait<0>();
    else if (f == F - 2) cp_async_wait<1>();
    else cp_async_wait<2>();
    SY::sync();
    float2 v[E];
    if (p.from_k) {
#pragma unroll
      for (int b = 0; b < E / RFL; ++b)
#pragma unroll
        for (int r = 0; r < RFL; ++r) v[b * RFL + r] = xr.base[pos_first<PL, true>(t + b * T, r)];
      fft_run<PL, true, 0, XchRow, SY, TwGlobal>(v, t, xr, tw);
    } else {
#pragma unroll
      for (int b = 0; b < E / RF0; ++b)
#pragma unroll
        for (int r = 0; r < RF0; ++r) v[b * RF0 + r] = xr.base[pos_first<PL, false>(t + b * T, r)];
    }
    SY::sync();  // the row's last reads are done
    park<PL>(xr.base, t, v);
  }

  // 2. reverse of N_A (at xa), then of N_B (at xb), two points at a time; the states
  // (and under a map the stage-factor tables) of the next points are requested
  // while these are reversed
  if (act) {
    const long long nxy = (long long)p.ny * NX;
    const float2* emap = MAP ? p.emap + (row % p.ny) * NX : nullptr;
    float4 na[F], nb[F];
    float2 nm[4][2];
    const float4 none = make_float4(0.f, 0.f, 0.f, 0.f);
    const auto request = [&](int q) {
#pragma unroll
      for (int f = 0; f < F; ++f) {
        const long long at = f * p.fstride + row * NX;
        na[f] = p.xa ? load_points<PL>(p.xa + at, p.xa_row_order, t, q) : none;
        nb[f] = p.xb ? load_points<PL>(p.xb + at, false, t, q) : none;
      }
      if constexpr (MAP) {
#pragma unroll
        for (int m = 0; m < 4; ++m)
#pragma unroll
          for (int u = 0; u < 2; ++u) nm[m][u] = __ldcg(emap + m * nxy + point_pos<PL>(t, 2 * q + u));
      }
    };
    Stages<MAP> B, A;
    if constexpr (!MAP) {
      B = stages_of(p.ecoef);
      A = stages_of(p.ecoef + 3);
    }
    float2 s[6];
#pragma unroll
    for (int k = 0; k < 6; ++k) s[k] = make_float2(0.f, 0.f);
    request(0);
#pragma unroll 1
    for (int q = 0; q < E / 2; ++q) {
      Pair g[F], x[F], xbv[F];
#pragma unroll
      for (int f = 0; f < F; ++f) {
        const float4 w = *park_place<PL>(myrow + f * ROWS * PITCH, t, q);
        g[f] = {make_float2(w.x, w.y), make_float2(w.z, w.w)};
        x[f] = {make_float2(na[f].x, na[f].y), make_float2(na[f].z, na[f].w)};
        xbv[f] = {make_float2(nb[f].x, nb[f].y), make_float2(nb[f].z, nb[f].w)};
      }
      if constexpr (MAP) {
        const auto pair_of = [](const float2* m) { return Pair{make_float2(m[0].x, m[1].x), make_float2(m[0].y, m[1].y)}; };
        B.e0 = pair_of(nm[0]);
        B.v = pair_of(nm[1]);
        A.e0 = pair_of(nm[2]);
        A.v = pair_of(nm[3]);
      }
      if (q + 1 < E / 2) request(q + 1);
      if (p.xa) rk4_vjp<F>(x, g, A, p.kh, p.kh2, s);
      if (p.xb) rk4_vjp<F>(xbv, g, B, p.kh, p.kh2, s + 3);
#pragma unroll
      for (int f = 0; f < F; ++f)
        *park_place<PL>(myrow + f * ROWS * PITCH, t, q) = make_float4(g[f].re.x, g[f].re.y, g[f].im.x, g[f].im.y);
    }
#pragma unroll
    for (int k = 0; k < 6; ++k) sens[k] = s[k].x + s[k].y;
  }

  // 3. every field: unpark, forward transform (or leave in real space), store
#pragma unroll 1
  for (int f = 0; f < F; ++f) {
    const XchRow xr{myrow + f * ROWS * PITCH};
    float2* dst = p.g + f * p.fstride + (act ? row : 0) * NX;
    float2 v[E];
    unpark<PL>(xr.base, t, v);
    if (!p.to_k) {
      if (act) {
#pragma unroll
        for (int b = 0; b < E / RF0; ++b)
#pragma unroll
          for (int r = 0; r < RF0; ++r) dst[pos_first<PL, false>(t + b * T, r)] = v[b * RF0 + r];
      }
    } else {
      fft_run<PL, false, 0, XchRow, SY, TwGlobal>(v, t, xr, tw);
      if (act) {
#pragma unroll
        for (int b = 0; b < E / RFL; ++b)
#pragma unroll
          for (int r = 0; r < RFL; ++r) dst[pos_last<PL, false>(t + b * T, r)] = v[b * RFL + r];
      }
    }
    SY::sync();
  }
}

// Resident CTAs of 128 threads: four (128 registers) hold two fields without spills,
// three fields or the tables of a map need three (168).  Both together spill there (at 18
// of 20 lengths) and take two CTAs where a thread has more than 16 points: mean of the
// recording and the reverse x-pass with three and two, 3 x 512x128x128 276 and 245 us,
// 3 x 192x128x256 214 and 191; with up to 16 the warps weigh more, 3 x 256x128x256 206
// and 222, 3 x 128x128x256 112 and 125.
template <int NX, int F, bool MAP>
__host__ __device__ constexpr int xadj_min_blocks() {
  return xpass_threads<NX>() > 128
             ? 1
             : (F == 3 && MAP && FftPlan<NX>::E > 16 ? 2 : F == 3 || MAP ? 3 : 4) * 128 / xpass_threads<NX>();
}
template <int NX, int F, bool MAP>
__global__ void __launch_bounds__(xpass_threads<NX>(), xadj_min_blocks<NX, F, MAP>())
    xpass_adj_kernel(const XAdjArgs p) {
  constexpr int THREADS = xpass_threads<NX>();
  extern __shared__ float4 sm4[];
  float2* rowbuf = reinterpret_cast<float2*>(sm4);
  __shared__ double red[THREADS / 32][6];
  chain_begin();
  float sens[6] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
  // rows from the last tau-plane down, as the forward x-pass
  xpass_adj_tile<NX, F, THREADS, MAP>(p, (long long)gridDim.x - 1 - blockIdx.x, rowbuf, sens);
  // block sums in FP64, fixed order (deterministic)
#pragma unroll
  for (int k = 0; k < 6; ++k) {
    double v = (double)sens[k];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5][k] = v;
  }
  __syncthreads();
  if (threadIdx.x < 6) {
    double v = 0.0;
#pragma unroll
    for (int w = 0; w < THREADS / 32; ++w) v += red[w][threadIdx.x];
    p.partial[(long long)blockIdx.x * 6 + threadIdx.x] = v;
  }
}

template <int NX, int F, bool MAP>
cudaError_t launch_adjoint(const XAdjArgs& a, long long* ncta, cudaStream_t s) {
  constexpr int ROWS = xpass_rows<NX>();
  constexpr int THREADS = xpass_threads<NX>();
  const size_t smem = (size_t)xpass_smem_floats2<NX>(F) * sizeof(float2);
  static SmemOnce once;
  cudaError_t e = raise_smem_limit(xpass_adj_kernel<NX, F, MAP>, smem, once);
  if (e != cudaSuccess) return e;
  const long long grid = (a.rows + ROWS - 1) / ROWS;
  *ncta = grid;
  if (grid <= 0) return cudaSuccess;
  return launch_chained(xpass_adj_kernel<NX, F, MAP>, dim3((unsigned)grid), THREADS, smem, s, a);
}


}  // namespace brahms
