// Set-up tables, the energy reduction and dtype conversions.
#include "kernels.cuh"
#include "launch_cfg.h"
#include "map_seg.h"

namespace brahms {

// 2 pi * numpy.fft.fftfreq(n, d)[m]; the Nyquist bin is negative.
__device__ __forceinline__ double ang_freq(int m, int n, double d) {
  const int mm = (m < (n + 1) / 2) ? m : m - n;
  return 6.283185307179586476925286766559 * (double)mm / ((double)n * d);
}

// amp * exp(i phi) - 1 ("delta form"), formed in FP64 and rounded once:
//   amp cos(phi) - 1 = (amp - 1) - 2 amp sin^2(phi/2),   amp sin(phi).
// Stored this way, a factor with a small phase keeps |1 + D| = amp to FP32
// relative precision of the small part, so repeated application does not
// bias the field energy.  (amp - 1 can be as small as the rest of a norm: a sine
// rounded to a float first would swallow it, always.)
__device__ __forceinline__ float2 delta_phase(double phi, double amp_m1) {
  const double two_pi = 6.283185307179586476925286766559;
  const double r = phi - two_pi * rint(phi / two_pi);
  const double sh = sin(0.5 * r), amp = 1.0 + amp_m1;
  return make_float2((float)(amp_m1 - 2.0 * amp * sh * sh), (float)(amp * sin(r)));
}

// Separable factors of the linear propagator over dz (Eqs. dispOp, diffOp,
// with d/dx -> i kx, d/dtau -> i Omega, diffraction +(i/2k) Laplacian and the
// unitary third-order term), each stored as D = P - 1:
//   Px = exp(-i dz [kx^2/(2k) + tan(rho) kx])
//   Py = exp(-i dz ky^2/(2k))
//   Pt = exp(dz [-alpha/2 - i delta Omega + i k2/2 Omega^2 - i k3/6 Omega^3])
__global__ void prop_tables_kernel(const TableArgs a) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  const int per = a.nx + a.ny + a.nt;
  if (i >= per * a.nf) return;
  const int f = i / per;
  int m = i % per;
  const bool cw = a.nt == 1 && a.ny > 1;
  if (m < a.nx) {
    const double kx = ang_freq(m, a.nx, a.dx);
    const double ph = -a.dz * (kx * kx / (2.0 * a.k[f]) + tan(a.rho[f]) * kx);
    a.px[f * a.nx + m] = delta_phase(ph, 0.0);
    return;
  }
  m -= a.nx;
  if (m < a.ny) {
    const double ky = ang_freq(m, a.ny, a.dy);
    a.py[f * a.ny + m] = delta_phase(-a.dz * ky * ky / (2.0 * a.k[f]), cw ? a.rest : 0.0);
    return;
  }
  m -= a.ny;
  const double om = ang_freq(m, a.nt, a.dt);
  const double ph = a.dz * (-a.delta[f] * om + 0.5 * a.k2[f] * om * om - a.k3[f] / 6.0 * om * om * om);
  const double loss = expm1(-0.5 * a.alpha[f] * a.dz), rest = cw ? 0.0 : a.rest;
  a.pt[f * a.nt + m] = delta_phase(ph, loss + rest + loss * rest);
}

// ---------------------------------------------- mismatch-map tables
__device__ __forceinline__ float2 phase_plus(double phi) {
  const float2 em = phase_minus(phi);
  return make_float2(em.x, -em.y);
}

__global__ void map_tables_kernel(const MapArgs a) {
  chain_begin();
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < a.nxy;
       i += (long long)gridDim.x * blockDim.x) {
    const double mb = a.mapB[i], ma = a.mapA[i];
    const double p = a.mphase[i];
    a.emap[i] = phase_plus(a.phiB + a.dkB * 0.5 * a.dz + p + mb * (a.zB - a.zp + 0.5 * a.dz));
    a.emap[a.nxy + i] = phase_plus((a.dkB + mb) * 0.25 * a.dz);
    double pa = p, zpa = a.zp;
    if (a.advance) {
      pa = p + mb * (a.zA - a.zp);
      zpa = a.zA;
      a.mphase[i] = pa;
    }
    a.emap[2 * a.nxy + i] = phase_plus(a.phiA + pa + ma * (a.zA - zpa));
    a.emap[3 * a.nxy + i] = phase_plus((a.dkA + ma) * 0.25 * a.dz);
  }
}

cudaError_t run_map_tables(const MapArgs& a, cudaStream_t s) {
  long long g = (a.nxy + 255) / 256;
  if (g > 152 * 8) g = 152 * 8;
  return launch_chained(map_tables_kernel, dim3((unsigned)g), 256, 0, s, a);
}

__global__ void map_phase_advance_kernel(double* mphase, const double* m, double len, long long nxy) {
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < nxy; i += (long long)gridDim.x * blockDim.x)
    mphase[i] += m[i] * len;
}

cudaError_t run_map_phase_advance(double* mphase, const double* m, double len, long long nxy, cudaStream_t s) {
  long long g = (nxy + 255) / 256;
  if (g > 152 * 8) g = 152 * 8;
  map_phase_advance_kernel<<<(unsigned)g, 256, 0, s>>>(mphase, m, len, nxy);
  return cudaPeekAtLastError();
}

// B: the second half of step jB (starting at its midpoint), A: the first half
// of step jA; the same four tables as map_tables_kernel.
__global__ void map_tables_seg_kernel(const MapSegArgs a) {
  chain_begin();
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < a.nxy;
       i += (long long)gridDim.x * blockDim.x) {
    double qb = 0.0, qa = 0.0;
    for (int s = 0; s < a.nseg; ++s) {
      const double m = a.maps[s * a.nxy + i];
      qb += a.cB[s] * m;
      qa += a.cA[s] * m;
    }
    const double mb = a.maps[a.sB * a.nxy + i], ma = a.maps[a.sA * a.nxy + i];
    a.emap[i] = phase_plus(a.phiB + a.dkB * 0.5 * a.dz + qb + mb * (0.5 * a.dz));
    a.emap[a.nxy + i] = phase_plus((a.dkB + mb) * 0.25 * a.dz);
    a.emap[2 * a.nxy + i] = phase_plus(a.phiA + qa);
    a.emap[3 * a.nxy + i] = phase_plus((a.dkA + ma) * 0.25 * a.dz);
  }
}

cudaError_t run_map_tables_seg(const MapSegArgs& a, cudaStream_t s) {
  if (a.nseg < 1 || a.nseg > kMapSegMax) return cudaErrorInvalidValue;
  long long g = (a.nxy + 255) / 256;
  if (g > 152 * 8) g = 152 * 8;
  return launch_chained(map_tables_seg_kernel, dim3((unsigned)g), 256, 0, s, a);
}

cudaError_t run_prop_tables(const TableArgs& a, cudaStream_t s) {
  const int n = (a.nx + a.ny + a.nt) * a.nf;
  prop_tables_kernel<<<(n + 255) / 256, 256, 0, s>>>(a);
  return cudaPeekAtLastError();
}

// ------------------------------------------------------------- energy
// Per-field sum of |A|^2: two complex values per 16-byte load, squares
// summed in FP32 over eight points (round-to-nearest, unbiased) and added to an FP64
// accumulator: one FP64 addition per eight points.  Bound by memory: 805 MB read in 122
// us (6.6 TB/s).
__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
  return v;
}

// COPY: the fields read are also written to dst, so that a field brought in or
// handed out is read once for both.  The last block to finish adds the partial
// sums in their fixed order and writes the sums and the device error word to
// the pinned host words as well, so a check is one launch and no copies.
template <bool COPY>
__global__ void __launch_bounds__(256) energy_kernel(const EnergyArgs p) {
  const int f = blockIdx.y, nf = gridDim.y;
  const float4* a4 = reinterpret_cast<const float4*>(f == 0 ? p.src[0] : f == 1 ? p.src[1] : p.src[2]);
  float4* d4 = reinterpret_cast<float4*>(f == 0 ? p.dst[0] : f == 1 ? p.dst[1] : p.dst[2]);
  double own = 0.0;
  // pairs (every length is even, so a field holds whole 16-byte pairs)
  const long long n2 = p.n / 2;
  const long long stride = (long long)gridDim.x * blockDim.x;
  const long long i0 = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  long long i = i0;
  // independent pairs per round, four to an FP64 addition: the loads overlap; eight
  // where the fields are copied, four (37 registers, all CTAs resident) where they are
  // only read
  constexpr int U = COPY ? 8 : 4;
  const auto square = [](float4 v) { return fmaf(v.x, v.x, fmaf(v.y, v.y, fmaf(v.z, v.z, v.w * v.w))); };
  for (; i + (U - 1) * stride < n2; i += U * stride) {
    float4 v[U];
#pragma unroll
    for (int u = 0; u < U; ++u) v[u] = __ldcg(a4 + i + u * stride);
#pragma unroll
    for (int u = 0; u < U; ++u)
      if constexpr (COPY) d4[i + u * stride] = v[u];
#pragma unroll
    for (int u = 0; u < U; u += 4)
      own += (double)((square(v[u]) + square(v[u + 1])) + (square(v[u + 2]) + square(v[u + 3])));
  }
  for (; i < n2; i += stride) {
    const float4 v = __ldcg(a4 + i);
    if constexpr (COPY) d4[i] = v;
    own += (double)square(v);
  }
  __shared__ double red[8][3];
  __shared__ bool last;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  own = warp_sum(own);
  if (lane == 0) red[warp][0] = own;
  __syncthreads();
  if (warp == 0) {
    const double s = warp_sum(lane < 8 ? red[lane][0] : 0.0);
    if (lane == 0) {
      p.partial[f * gridDim.x + blockIdx.x] = s;
      __threadfence();
      // wraps to zero for the next launch
      last = atomicInc(p.count, gridDim.x * nf - 1) == gridDim.x * nf - 1;
    }
  }
  __syncthreads();
  if (!last) return;
  __threadfence();
  // the fields' partial sums side by side (one field after the other took 3 us longer)
  double v[3] = {0.0, 0.0, 0.0};
  for (int k = threadIdx.x; k < (int)gridDim.x; k += 256)
#pragma unroll
    for (int g = 0; g < 3; ++g)
      if (g < nf) v[g] += __ldcg(p.partial + g * gridDim.x + k);
#pragma unroll
  for (int g = 0; g < 3; ++g) {
    v[g] = warp_sum(v[g]);
    if (lane == 0) red[warp][g] = v[g];
  }
  __syncthreads();
  if (threadIdx.x < nf) {
    double e = 0.0;
    for (int w = 0; w < 8; ++w) e += red[w][threadIdx.x];
    p.host[threadIdx.x] = e;
  }
  if (threadIdx.x == 3) *reinterpret_cast<int*>(p.host + 3) = *p.err;
}

cudaError_t run_energy(const EnergyArgs& a, int nf, int nblocks, cudaStream_t s) {
  if (a.dst[0]) energy_kernel<true><<<dim3(nblocks, nf), 256, 0, s>>>(a);
  else energy_kernel<false><<<dim3(nblocks, nf), 256, 0, s>>>(a);
  return cudaPeekAtLastError();
}

// ---------------------------------------------------------- conversions
__global__ void c128_to_c64_kernel(const double2* __restrict__ in, float2* __restrict__ out, long long n) {
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
    const double2 v = in[i];
    out[i] = make_float2((float)v.x, (float)v.y);
  }
}
__global__ void c64_to_c128_kernel(const float2* __restrict__ in, double2* __restrict__ out, long long n) {
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
    const float2 v = in[i];
    out[i] = make_double2((double)v.x, (double)v.y);
  }
}

// two fields of n points (even) in one launch, 16-byte pairs
__global__ void copy_pair_kernel(const float4* __restrict__ s0, float4* __restrict__ d0, const float4* __restrict__ s1,
                                 float4* __restrict__ d1, long long n2) {
  const float4* s = blockIdx.y ? s1 : s0;
  float4* d = blockIdx.y ? d1 : d0;
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n2; i += (long long)gridDim.x * blockDim.x)
    d[i] = __ldcg(s + i);
}

static int grid_for(long long n) {
  long long g = (n + 255) / 256;
  return (int)(g > 152 * 16 ? 152 * 16 : (g < 1 ? 1 : g));
}

// ------------------------------------------------ pointwise linear step
// The linear step of a single row (ny = nt = 1: neither a y nor a tau transform): the
// multiply
// P = (1 + Dx)(1 + Dy)(1 + Dt) / N of the tau-pass, element by element, with
// the tau-pass's arithmetic, on the (kx, ky)-domain state.
__global__ void prop_pointwise_kernel(const AxisArgs p, int nf) {
  chain_begin();
  const long long plane = (long long)p.nx * p.ny;
  const long long per_field = plane * p.nt;
  const long long n = per_field * nf;
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
    const int f = (int)(i / per_field);
    const long long r = i - (long long)f * per_field;
    const int x = (int)(r % p.nx);
    const int y = (int)((r / p.nx) % p.ny);
    const int t = (int)(r / plane);
    const float2 dx = p.px[f * p.nx + x], dy = p.py[f * p.ny + y], dt = p.pt[f * p.nt + t];
    float2* q = p.data + (long long)f * p.fstride + r;
    *q = !p.scaled ? ColumnProp<false>(p, dx, dy)(p, *q, dt) : ColumnProp<true>(p, dx, dy)(p, *q, dt);
  }
}

cudaError_t run_prop_pointwise(const AxisArgs& a, int nf, cudaStream_t s) {
  return launch_chained(prop_pointwise_kernel, dim3((unsigned)grid_for((long long)a.nx * a.ny * a.nt * nf)), 256, 0, s, a,
                        nf);
}

cudaError_t run_copy_pair(const float2* s0, float2* d0, const float2* s1, float2* d1, long long n, cudaStream_t s) {
  copy_pair_kernel<<<dim3(grid_for(n / 2), 2), 256, 0, s>>>(
      reinterpret_cast<const float4*>(s0), reinterpret_cast<float4*>(d0), reinterpret_cast<const float4*>(s1),
      reinterpret_cast<float4*>(d1), n / 2);
  return cudaPeekAtLastError();
}

cudaError_t run_c128_to_c64(const double2* in, float2* out, long long n, cudaStream_t s) {
  c128_to_c64_kernel<<<grid_for(n), 256, 0, s>>>(in, out, n);
  return cudaPeekAtLastError();
}
cudaError_t run_c64_to_c128(const float2* in, double2* out, long long n, cudaStream_t s) {
  c64_to_c128_kernel<<<grid_for(n), 256, 0, s>>>(in, out, n);
  return cudaPeekAtLastError();
}

}  // namespace brahms
