// Kernels of one split-step z-step (Sec. 3.1, Eq. expon) on the layout
// fields[f][tau][y][x] (x fastest), complex64.
//
// A z-step is four passes over memory per field:
//   x-pass  inverse x-FFT, the second RK4 half step of step j, the first RK4
//           half step of step j+1, forward x-FFT (all fields of a row at once,
//           the nonlinear coupling is pointwise across fields)
//   y-pass  forward y-FFT
//   t-pass  forward tau-FFT, multiply by the linear propagator
//           P = Px(kx) Py(ky) Pt(Omega) / (NX NY NT), inverse tau-FFT
//   y-pass  inverse y-FFT
// On the small planes of BRAHMS_FOR_EACH_PLANE the y-inverse, x-pass and y-forward
// are one kernel (plane.cuh), and on cw grids (nt = 1, ny > 1) the linear step is one
// pass along y (the tau-pass's kernel on the axes x, tau, y).
// Between calls the state is in real space; the first and the last step of
// a call peel the x-pass (NL_FIRST / NL_LAST).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include <type_traits>

#include "fft_core.cuh"

namespace brahms {

enum XMode : int { XM_NL_FIRST = 2, XM_NL_MID = 3, XM_NL_LAST = 4 };

constexpr int kStageFactors = 6;  // of an x-pass: the start, middle and end of both half steps

struct XPassArgs {
  float2* data;        // [nf][rows][nx]
  long long fstride;   // elements between fields
  long long rows;      // ny * nt
  const float2* tw;    // per-pass twiddle table of the x transform
  int mode;            // XMode
  double phiA, dkA;    // step whose first half is applied: Phi(z_j), dk_j
  double phiB, dkB;    // step whose second half is applied
  double dz;
  float kh[3];         // kappa_f * dz/2, including the 1/2 SH factor for 2 fields
  float kh2[3];        // kh / 2 (exact)
  // transverse mismatch map: per-(x, y) stage phase factors [4][ny][nx]
  // (B start, B quarter-step, A start, A quarter-step; see run_map_tables),
  // or NULL for a mismatch uniform across the grid
  const float2* emap;
  int ny;
  // recording (adjoint recomputation): real-space copies of the state that
  // enters the B half step and of the state that enters the A half step, or NULL;
  // each row in place order (park_place), as the reverse x-pass reads it
  float2* rec_b;
  float2* rec_a;
  // the stage factors of both half steps from the phases above, written by the
  // host dispatchers in FP64 (map-free x-passes read them instead of computing
  // them per CTA): e^{+i Phi} at the start, middle and end of the B half and of the A
  // half
  float2 ecoef[kStageFactors];
};
// Host: the stage factors of an x-pass from its phases (FP64 phase, reduced
// mod 2 pi, cos and sin in FP64, rounded to float).
void fill_stage_factors(XPassArgs& a);

struct AxisArgs {
  float2* data;
  int nx, ny, nt;
  long long fstride;
  long long ntiles;
  int xtiles;
  const float2* tw;    // twiddles of the transformed axis
  const float4* twp;   // the same as products (single transforms, the spectrum)
  const float2* px;    // [nf][nx] propagator factors (t-pass only)
  const float2* py;    // [nf][ny]
  const float2* pt;    // [nf][nt]
  float scale;            // 1/(nx ny nt) as a float
  int scaled;             // it is no power of two: see ColumnProp
  int conj_p;             // apply conj(P) (the adjoint of the linear step)
};

// plan of length N on an axis (0 x, 1 y, 2 tau)
template <int N, int AXIS>
using AxisPlan = typename std::conditional<AXIS == 0, FftPlan<N>,
                                           typename std::conditional<AXIS == 1, ColPlan<N>, TauPlan<N>>::type>::type;

// ------------------------------------------------------------ tile shapes
template <int N>
__host__ __device__ constexpr int fft_threads() { return FftPlan<N>::T; }

// x-pass CTA: 128 threads, or one row when a row needs 64 threads or more (its block
// barriers then wait for one row alone: x-pass of 2 x 1024x256x64 197 -> 188 us with
// one row of 64 threads instead of two, 3 x 1024x64x64 82.6 -> 79.0, step of 2 x
// 1024x1024x1 31.9 -> 30.9); rows whose threads lie inside one warp synchronise
// their exchanges with __syncwarp.
template <int N>
__host__ __device__ constexpr int xpass_threads() { return fft_threads<N>() >= 64 ? fft_threads<N>() : 128; }
template <int N>
__host__ __device__ constexpr int xpass_rows() { return xpass_threads<N>() / fft_threads<N>(); }
template <int N>
__host__ __device__ constexpr bool xpass_warp_sync() { return fft_threads<N>() <= 32 && 32 % fft_threads<N>() == 0; }
// shared memory in float2 units: a row buffer per field and row
template <int N>
__host__ __device__ constexpr int xpass_smem_floats2(int nf) {
  return nf * xpass_rows<N>() * XchRow::pitch(N);
}
// resident CTAs the x-pass asks the register allocator for: 6 (80 registers)
// where six CTAs' shared memory fits in an SM and rows are at most 256 long, 5 there for
// three fields under a map (at 80 registers rows of 4, 6, 8, 32 and 64 points spill:
// step of 3 x 8, 32 and 64 points along x 155.2, 199.4 and 171.6 us with 6, 150.9, 193.6
// and 168.5 with 5; the other lengths alike); otherwise 4, or 8 of 64 threads (128
// registers)
template <int N, int F, bool MAP>
__host__ __device__ constexpr int xpass_min_blocks() {
  return xpass_threads<N>() > 128                                                ? 1
         : (N <= 256 && 6 * (xpass_smem_floats2<N>(F) * 8 + 1024) <= 228 * 1024) ? (MAP && F == 3 ? 5 : 6)
         : xpass_threads<N>() == 64                                              ? 8
                                                                                 : 4;
}

// Strided pencils: tiles of TX neighbouring columns (128-byte rows up to
// N = 1024) times the plan's T threads per pencil.
__host__ __device__ constexpr int col_tile_n(int n) { return n <= 1024 ? 16 : (n <= 2048 ? 8 : 4); }
// columns per tile of a plan's strided-pencil kernels
template <class PL>
struct ColTile {
  static constexpr int value = col_tile_n(PL::N);
};
template <class PL>
__host__ __device__ constexpr int tile_threads() { return PL::T * ColTile<PL>::value; }
template <class PL>
__host__ __device__ constexpr int tiles_per_cta() { return tile_threads<PL>() >= 256 ? 1 : 256 / tile_threads<PL>(); }
// twiddle tables of up to 2560 entries (20 KB: lengths up to 1024) are copied to
// shared memory; larger ones are read through L1
template <class PL>
__host__ __device__ constexpr bool tw_in_smem() { return tw_table_size<PL>() <= 2560; }
template <class PL>
__host__ __device__ constexpr int axis_smem_floats2() {
  return (tw_in_smem<PL>() ? tw_table_size<PL>() : 0) + tiles_per_cta<PL>() * PL::N * ColTile<PL>::value;
}
// The forward y-pass reads its twiddles through L1 instead of staging them in
// shared memory per CTA: measured on the 3 x 256x256x512 state, 285 -> 253 us
// per launch (the inverse y-pass, 259 -> 266, measured the other way and keeps the
// staging; now 231 and 237, 7.0 and 6.8 TB/s).
template <class PL, bool INV>
__host__ __device__ constexpr bool axis_tw_staged() { return tw_in_smem<PL>() && INV; }
template <class PL, bool INV>
__host__ __device__ constexpr int ypass_smem_floats2() {
  return (axis_tw_staged<PL, INV>() ? tw_table_size<PL>() : 0) +
         tiles_per_cta<PL>() * PL::N * ColTile<PL>::value;
}

// -------------------------------------------------------- nonlinear step
// Two grid points at once: real and imaginary parts as FP32 pairs, so that the
// arithmetic of both points is one packed instruction (see fft_core.cuh).
struct Pair {
  float2 re, im;
};
__device__ __forceinline__ float2 dup(float a) { return make_float2(a, a); }
__device__ __forceinline__ float2 neg(float2 a) { return make_float2(-a.x, -a.y); }
__device__ __forceinline__ Pair pair_mul(Pair a, Pair b) {
  return {__ffma2_rn(a.re, b.re, neg(__fmul2_rn(a.im, b.im))), __ffma2_rn(a.re, b.im, __fmul2_rn(a.im, b.re))};
}
// a conj(b)
__device__ __forceinline__ Pair pair_mulc(Pair a, Pair b) {
  return {__ffma2_rn(a.re, b.re, __fmul2_rn(a.im, b.im)), __ffma2_rn(a.im, b.re, neg(__fmul2_rn(a.re, b.im)))};
}
// i a conj(b)
__device__ __forceinline__ Pair pair_imulc(Pair a, Pair b) {
  return {__ffma2_rn(a.re, b.im, neg(__fmul2_rn(a.im, b.re))), __ffma2_rn(a.re, b.re, __fmul2_rn(a.im, b.im))};
}
// a + c b and a + i c b for a real c
__device__ __forceinline__ Pair pair_axpy(Pair a, float c, Pair b) {
  return {__ffma2_rn(dup(c), b.re, a.re), __ffma2_rn(dup(c), b.im, a.im)};
}
__device__ __forceinline__ Pair pair_iaxpy(Pair a, float c, Pair b) {
  return {__ffma2_rn(dup(-c), b.im, a.re), __ffma2_rn(dup(c), b.re, a.im)};
}
__device__ __forceinline__ Pair pair_add(Pair a, Pair b) { return {cadd(a.re, b.re), cadd(a.im, b.im)}; }

// Products of the coupling at one stage: the driving term of field 0 (A_s A_i,
// or A_F^2), without its phase, and i times the slopes of the others, i u
// conj(A_i), i u conj(A_s) (or i u conj(A_F)), u = e^{+i Phi} A_0.
template <int F>
__device__ __forceinline__ Pair nl_drive(const Pair* t) {
  if constexpr (F == 3) return pair_mul(t[0], t[1]);
  else return {__ffma2_rn(t[0].re, t[0].re, neg(__fmul2_rn(t[0].im, t[0].im))),
               __fmul2_rn(cadd(t[0].re, t[0].re), t[0].im)};
}
template <int F>
__device__ __forceinline__ void nl_slopes(Pair u, const Pair* t, Pair* n) {
  if constexpr (F == 3) {
    n[0] = pair_imulc(u, t[1]);
    n[1] = pair_imulc(u, t[0]);
  } else {
    n[0] = pair_imulc(u, t[0]);
  }
}

// Stage factors of a half step of length h: e0, em, e1 = e^{+i Phi} at its start,
// middle and end, and v = e^{+i dk h/2}.  Uniform over the grid, all three come from the
// host, formed in FP64, and v from them; under a map a point has e0 and v (MAP), and em
// and e1 are e0 v and e0 v^2.
template <bool MAP>
struct Stages {
  Pair e0, em, e1, v;
};
__device__ __forceinline__ Pair pair_dup(float2 c) { return {dup(c.x), dup(c.y)}; }
__device__ __forceinline__ Stages<false> stages_of(const float2* coef) {
  const Pair e0 = pair_dup(coef[0]), em = pair_dup(coef[1]);
  return {e0, em, pair_dup(coef[2]), pair_mulc(em, e0)};
}

// Classical RK4 over one half step h (Sec. 3.1) of Eqs. CEp/CEs/CEi (fields p,
// s, i) or of the degenerate pair (SH, F) at two points; kh = kappa h and kh2 = kh/2
// per field.
// Field 0 enters the others' slopes only through u = e A_0, so its stage values
// are carried as u directly, with m the driving terms of stages 1..4:
//   u1 = e0 A_0,  w = em A_0,  u2 = w + i kh2 v m1,  u3 = w + i kh2 m2,
//   u4 = e1 A_0 + i kh v m3,  A_0 += i kh/6 (conj(e0) m1 + conj(em) 2 (m2 + m3) + conj(e1) m4),
// 128 operations a point for three fields; under a map w = v u1, u4 = v (w + i kh m3)
// and the sum nested in v, 124, where forming em and e1 of every point would take 8 more.
// Every stage and the final combination use the same kh_f, and the 1/6 weight is
// common to all fields: field-dependent rounding of the weights would break the
// Manley-Rowe balance the exact scheme keeps and let the total energy drift step
// after step.
template <int F, bool MAP>
__device__ __forceinline__ void rk4(Pair (&a)[F], const Stages<MAP>& c, const float* kh, const float* kh2) {
  constexpr int G = F - 1;
  Pair t[G], n[G], acc[G];
  const Pair u1 = pair_mul(c.e0, a[0]);
  const Pair w = MAP ? pair_mul(c.v, u1) : pair_mul(c.em, a[0]);
  const Pair m1 = nl_drive<F>(a + 1);
  nl_slopes<F>(u1, a + 1, acc);
#pragma unroll
  for (int g = 0; g < G; ++g) t[g] = pair_axpy(a[g + 1], kh2[g + 1], acc[g]);
  const Pair m2 = nl_drive<F>(t);
  nl_slopes<F>(pair_iaxpy(w, kh2[0], pair_mul(c.v, m1)), t, n);
#pragma unroll
  for (int g = 0; g < G; ++g) {
    acc[g] = pair_axpy(acc[g], 2.f, n[g]);
    t[g] = pair_axpy(a[g + 1], kh2[g + 1], n[g]);
  }
  const Pair m3 = nl_drive<F>(t);
  nl_slopes<F>(pair_iaxpy(w, kh2[0], m2), t, n);
#pragma unroll
  for (int g = 0; g < G; ++g) {
    acc[g] = pair_axpy(acc[g], 2.f, n[g]);
    t[g] = pair_axpy(a[g + 1], kh[g + 1], n[g]);
  }
  const Pair m4 = nl_drive<F>(t);
  nl_slopes<F>(MAP ? pair_mul(c.v, pair_iaxpy(w, kh[0], m3)) : pair_iaxpy(pair_mul(c.e1, a[0]), kh[0], pair_mul(c.v, m3)), t, n);
#pragma unroll
  for (int g = 0; g < G; ++g) {
    const Pair q = pair_add(acc[g], n[g]);
    a[g + 1] = pair_axpy(a[g + 1], kh[g + 1], {__fmul2_rn(q.re, dup(1.f / 6.f)), __fmul2_rn(q.im, dup(1.f / 6.f))});
  }
  Pair m;
  if constexpr (MAP) {
    m = pair_axpy(pair_mulc(m4, c.v), 2.f, pair_add(m2, m3));
    m = pair_mulc(pair_add(m1, pair_mulc(m, c.v)), c.e0);
  } else {
    m = pair_axpy(pair_mulc(m1, c.e0), 2.f, pair_mulc(pair_add(m2, m3), c.em));
    m = pair_add(m, pair_mulc(m4, c.e1));
  }
  a[0] = pair_iaxpy(a[0], kh[0], {__fmul2_rn(m.re, dup(1.f / 6.f)), __fmul2_rn(m.im, dup(1.f / 6.f))});
}

// e^{-i Phi} with Phi in FP64, reduced to [-pi, pi] before the FP32 sincos.
__device__ __forceinline__ float2 phase_minus(double phi) {
  const double two_pi = 6.283185307179586476925286766559;
  double r = phi - two_pi * rint(phi / two_pi);
  float s, c;
  sincosf((float)r, &s, &c);
  return make_float2(c, -s);
}

// ------------------------------------------------------------------ x-pass
// One row (y, tau) of every field per T threads; a CTA of THREADS threads
// handles THREADS/T rows per tile.  Each field of a row has its own row buffer
// in shared memory, used both as that field's FFT exchange space and to park the
// field between the transforms: after the inverse transform every thread parks
// its values, the pointwise RK4 pair then reads all F values of each owned point,
// and the forward transform starts from the owned points again.  No thread ever
// reads a value another thread parked, so parking needs no barrier, and the
// fields and the points are processed in loops rather than unrolled, which keeps
// the kernel small enough for the instruction cache.  Two points of a thread
// are parked together as (re, re, im, im) in 16 bytes, which is the form the
// packed RK4 works in.  The rows of all fields are requested together, by
// asynchronous copies straight into the row buffers, so a field's row arrives
// while the one before it is transformed and no registers wait for it (108 ->
// 92 registers for three fields of 256; 482 -> 421 us per launch on
// 3 x 256x256x512, 350 -> 326 on 2 x 512x512x128; 423 and 333 now).  What bounds it:
// the FP32 pipe, 131 operations a point and field (46 of the two transforms of 256
// points, 85 of the RK4 half steps), 337 us at its measured rate on that state.
// Twiddles are read through L1.
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() {
  asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}
// the thread's share of a row, 16 bytes (two points) at a time
template <class PL>
__device__ __forceinline__ void copy_row(float2* dst, const float2* src, int t) {
  const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
#pragma unroll
  for (int q = 0; q < PL::E / 2; ++q)
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(d + 16 * (t + q * PL::T)), "l"(src + 2 * (t + q * PL::T))
                 : "memory");
}
// points 2 q and 2 q + 1 of thread t in a row buffer
template <class PL>
__device__ __forceinline__ float4* park_place(float2* row, int t, int q) {
  return reinterpret_cast<float4*>(row) + q * PL::T + t;
}
template <class PL>
__device__ __forceinline__ void park(float2* row, int t, const float2 (&v)[PL::E]) {
#pragma unroll
  for (int q = 0; q < PL::E / 2; ++q)
    *park_place<PL>(row, t, q) = make_float4(v[2 * q].x, v[2 * q + 1].x, v[2 * q].y, v[2 * q + 1].y);
}
template <class PL>
__device__ __forceinline__ void unpark(float2* row, int t, float2 (&v)[PL::E]) {
#pragma unroll
  for (int q = 0; q < PL::E / 2; ++q) {
    const float4 a = *park_place<PL>(row, t, q);
    v[2 * q] = make_float2(a.x, a.z);
    v[2 * q + 1] = make_float2(a.y, a.w);
  }
}
// position on the row of point e of thread t between the transforms
template <class PL>
__device__ __forceinline__ int point_pos(int t, int e) {
  constexpr int R0 = fft_radix<PL, false>(0);
  return pos_first<PL, false>(t + (e / R0) * PL::T, e % R0);
}
template <int NX, int THREADS>
__host__ __device__ constexpr int xtile_rows() { return THREADS / FftPlan<NX>::T; }
template <int NX, int THREADS>
__host__ __device__ constexpr int xtile_smem_floats2(int nf) {
  return nf * xtile_rows<NX, THREADS>() * XchRow::pitch(NX);
}

template <int NX, int F, int THREADS, bool MAP = false, bool REC = false>
__device__ __forceinline__ void xpass_tile(const XPassArgs& p, long long tile, const float2* coef, float2* rowbuf) {
  using PL = FftPlan<NX>;
  constexpr int E = PL::E;
  constexpr int T = PL::T;
  constexpr int ROWS = xtile_rows<NX, THREADS>();
  constexpr int PITCH = XchRow::pitch(NX);
  constexpr int RF0 = fft_radix<PL, false>(0);           // forward first radix
  constexpr int RFL = fft_radix<PL, false>(PL::NP - 1);  // forward last radix
  using SY = typename std::conditional<xpass_warp_sync<NX>(), SyncWarp, SyncBlock>::type;
  static_assert(ROWS >= 1 && ROWS * T == THREADS, "CTA must hold whole rows");
  const TwGlobal tw{p.tw};

  const int t = threadIdx.x % T;
  const int rl = threadIdx.x / T;
  const long long row = tile * ROWS + rl;
  const bool act = row < p.rows;
  float2* myrow = rowbuf + rl * PITCH;  // field f at myrow + f ROWS PITCH
  const int mode = p.mode;
  const bool from_k = mode != XM_NL_FIRST;

  // 1. every field's row lands in its buffer by asynchronous copies, all requested
  // up front; then field by field inverse transform (from k-space) and park
#pragma unroll
  for (int f = 0; f < F; ++f) {
    if (act) copy_row<PL>(myrow + f * ROWS * PITCH, p.data + f * p.fstride + row * NX, t);
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
    if (from_k) {
#pragma unroll
      for (int b = 0; b < E / RFL; ++b)
#pragma unroll
        for (int r = 0; r < RFL; ++r) v[b * RFL + r] = xr.base[pos_first<PL, true>(t + b * T, r)];
      // the inverse's outputs lie at the forward first pass's positions
      fft_run<PL, true, 0, XchRow, SY, TwGlobal>(v, t, xr, tw);
    } else {
#pragma unroll
      for (int b = 0; b < E / RF0; ++b)
#pragma unroll
        for (int r = 0; r < RF0; ++r) v[b * RF0 + r] = xr.base[pos_first<PL, false>(t + b * T, r)];
    }
    SY::sync();  // the row's last reads (of the copy or of the last exchange) are done
    park<PL>(xr.base, t, v);
  }

  // 2. the RK4 half steps, two points at a time over the owned points
  {
    const long long nxy = (long long)p.ny * NX;
    const float2* emap = MAP ? p.emap + (act ? row % p.ny : 0) * NX : nullptr;
    // MAP: the next points' stage-factor tables are requested while these points'
    // RK4 pair runs
    float2 nm[4][2];
    Stages<MAP> B, A;
    if constexpr (MAP) {
#pragma unroll
      for (int q = 0; q < 4; ++q)
#pragma unroll
        for (int u = 0; u < 2; ++u) nm[q][u] = __ldcg(emap + q * nxy + point_pos<PL>(t, u));
    } else {
      B = stages_of(coef);
      A = stages_of(coef + 3);
    }
#pragma unroll 1
    for (int e = 0; e < E; e += 2) {
      if constexpr (MAP) {
        const auto pair_of = [](const float2* m) { return Pair{make_float2(m[0].x, m[1].x), make_float2(m[0].y, m[1].y)}; };
        B.e0 = pair_of(nm[0]);
        B.v = pair_of(nm[1]);
        A.e0 = pair_of(nm[2]);
        A.v = pair_of(nm[3]);
        if (e + 2 < E) {
#pragma unroll
          for (int q = 0; q < 4; ++q)
#pragma unroll
            for (int u = 0; u < 2; ++u) nm[q][u] = __ldcg(emap + q * nxy + point_pos<PL>(t, e + 2 + u));
        }
      }
      Pair a[F];
#pragma unroll
      for (int f = 0; f < F; ++f) {
        const float4 w = *park_place<PL>(myrow + f * ROWS * PITCH, t, e / 2);
        a[f] = {make_float2(w.x, w.y), make_float2(w.z, w.w)};
      }
      const auto record = [&](float2* rec) {
        if (!act) return;
#pragma unroll
        for (int f = 0; f < F; ++f)
          *park_place<PL>(rec + f * p.fstride + row * NX, t, e / 2) =
              make_float4(a[f].re.x, a[f].re.y, a[f].im.x, a[f].im.y);
      };
      if (mode != XM_NL_FIRST) {
        if constexpr (REC) {
          if (p.rec_b) record(p.rec_b);
        }
        rk4<F>(a, B, p.kh, p.kh2);
      }
      if (mode != XM_NL_LAST) {
        if constexpr (REC) {
          if (p.rec_a) record(p.rec_a);
        }
        rk4<F>(a, A, p.kh, p.kh2);
      }
#pragma unroll
      for (int f = 0; f < F; ++f)
        *park_place<PL>(myrow + f * ROWS * PITCH, t, e / 2) =
            make_float4(a[f].re.x, a[f].re.y, a[f].im.x, a[f].im.y);
    }
  }

  // 3. every field: unpark, forward transform (but on the last x-pass of a call), store
#pragma unroll 1
  for (int f = 0; f < F; ++f) {
    const XchRow xr{myrow + f * ROWS * PITCH};
    float2* dst = p.data + f * p.fstride + (act ? row : 0) * NX;
    float2 v[E];
    unpark<PL>(xr.base, t, v);
    if (mode == XM_NL_LAST) {
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
    SY::sync();  // the next field's exchanges use another buffer; keep the warp together
  }
}

// MAP: per-point stage phases from a transverse mismatch map (p.emap);
// REC: record the half steps' input states (p.rec_b, p.rec_a)
template <int NX, int F, bool MAP, bool REC = false>
__global__ void __launch_bounds__(xpass_threads<NX>(), xpass_min_blocks<NX, F, MAP>())
    xpass_kernel(const XPassArgs p) {
  constexpr int THREADS = xpass_threads<NX>();
  extern __shared__ float4 sm4[];
  float2* rowbuf = reinterpret_cast<float2*>(sm4);
  chain_begin();
  // stage factors from the launch (formed on the host in FP64: a per-CTA FP64
  // phase reduction stalled every CTA's first warps)
  // rows from the last tau-plane down (see the note on pass order above)
  xpass_tile<NX, F, THREADS, MAP, REC>(p, (long long)gridDim.x - 1 - blockIdx.x, p.ecoef, rowbuf);
}

// ------------------------------------------------- strided-axis passes
// AXIS 1: pencils along y (stride nx), tiles over (f, tau, x-tile).
// AXIS 2: pencils along tau (stride nx ny), tiles over (f, y, x-tile).
// Order across passes: the x-pass walks its rows from the last tau-plane
// down and the y-passes from the first up, so the x-pass starts on planes the
// y-inverse wrote last and the y-forward on planes the x-pass wrote last,
// still in L2 (read there, and overwritten there before they are written
// back).  Measured on the 3 x 256x256x512 state: 1603 -> 1592 ms per
// 1000-step call; a tau-major y order (every field of a plane together)
// made the y-passes 20 us slower and the step 1622 ms.  The tau-propagator
// also walks its tiles from the last down (tau 476 -> 473, y-inverse
// 258 -> 257 us).  (The step now takes 1310 us on that state.)
template <int N, int AXIS, int TX>
struct AxisTile {
  float2* base;  // element (x, pencil index 0)
  long long stride;
  int f, other, x;
  bool act;
  __device__ __forceinline__ AxisTile(const AxisArgs& p, long long tile, int tx) {
    const int xt = (int)(tile % p.xtiles);
    const long long rest = tile / p.xtiles;
    const int no = AXIS == 1 ? p.nt : p.ny;
    other = (int)(rest % no);
    f = (int)(rest / no);
    x = xt * TX + tx;
    act = tile < p.ntiles && x < p.nx;
    stride = AXIS == 1 ? (long long)p.nx : (long long)p.nx * p.ny;
    const long long off = AXIS == 1 ? (long long)other * p.nx * p.ny + x : (long long)other * p.nx + x;
    base = p.data + (act ? (long long)f * p.fstride + off : 0);
  }
};

// A pencil's registers from and to memory at the positions of the first pass of
// a direction (which are those of the other direction's last pass): input r of
// butterfly j at n + r N/R0, n centred, input 0 wrapped when n < 0.
template <class PL, bool INV>
__device__ __forceinline__ void load_pencil(float2 (&v)[PL::E], const float2* base, long long stride, int t, bool act) {
  constexpr int R0 = fft_radix<PL, INV>(0);
#pragma unroll
  for (int b = 0; b < PL::E / R0; ++b) {
    const int n = centred_first<PL, INV>(t + b * PL::T);
    const float2* q = base + n * stride;
#pragma unroll
    for (int r = 0; r < R0; ++r)
      v[b * R0 + r] = act ? __ldcg(r == 0 && n < 0 ? q + PL::N * stride : q + (r * (PL::N / R0)) * stride)
                          : make_float2(0.f, 0.f);
  }
}
template <class PL, bool INV>
__device__ __forceinline__ void store_pencil(const float2 (&v)[PL::E], float2* base, long long stride, int t) {
  constexpr int R0 = fft_radix<PL, INV>(0);
#pragma unroll
  for (int b = 0; b < PL::E / R0; ++b) {
    const int n = centred_first<PL, INV>(t + b * PL::T);
    float2* q = base + n * stride;
#pragma unroll
    for (int r = 0; r < R0; ++r)
      *(r == 0 && n < 0 ? q + PL::N * stride : q + (r * (PL::N / R0)) * stride) = v[b * R0 + r];
  }
}

// Tiles per CTA of THREADS threads for strided pencils.
template <class PL, int THREADS>
__host__ __device__ constexpr int tiles_per_cta_t() { return THREADS / tile_threads<PL>(); }

template <class PL, bool INV, int AXIS, int THREADS, class TW = TwShared>
__device__ __forceinline__ void axis_tile(const AxisArgs& p, long long cta_tile, const TW& tw, float2* xch) {
  constexpr int N = PL::N, T = PL::T, TX = ColTile<PL>::value;
  constexpr int TPC = tiles_per_cta_t<PL, THREADS>();
  static_assert(TPC >= 1 && TPC * T * TX == THREADS, "CTA must hold whole tiles");
  const int lt = threadIdx.x % (T * TX), tl = threadIdx.x / (T * TX);
  const int tx = lt % TX, t = lt / TX;
  const AxisTile<N, AXIS, TX> a(p, cta_tile * TPC + tl, tx);
  const XchCol<TX> xc{xch + tl * N * TX, tx};
  float2 v[PL::E];
  load_pencil<PL, INV>(v, a.base, a.stride, t, a.act);
  fft_run<PL, INV, 0, XchCol<TX>, SyncBlock, TW>(v, t, xc, tw);
  if (a.act) store_pencil<PL, !INV>(v, a.base, a.stride, t);
}

// The propagator P = (1 + Dx)(1 + Dy)(1 + Dt) / (nx ny nt) of one column, the
// factors in delta form.  With 1 + Dxy = (1 + Dx)(1 + Dy) a value w becomes
//   c w + w E(Omega),  E = g0 + Dt g1,  g0 = c Dxy,  g1 = c (1 + Dxy),
// c = 1/(nx ny nt) = scale where that is a power of two.  Where it is not (SCALED), c = 1
// and the result is scaled, scale w + scale w E, and the transformed axis's table carries
// what the float is short of 1/(nx ny nt), a factor 1 + rest of its entries, which are
// rounded once either way.  (With such a scale in g0 and g1 their rounding came on top of
// Dxy's, the same one in every step: the parametric run of 48x256x128 points ended 12 %
// further from FP64, and noise on a grid of 3 2^k points gained 6e-8 of its energy per
// step.  Scaling w by hi + lo floats before the product rounds w once more; after it they
// take two more operations a value, 450 instead of 406 us on 2 x 512x256x384.)
// The small product w E is formed first and c w added with one rounding.  (Folding w into the FMA chain rounds w.x - w.y E.y before the
// second-order term w.x (cos phi - 1) arrives; for small phases that term is below
// half an ulp and is then always lost, so |1 + E| acts as 1 + phi^2 / 2 and the
// energy grows step after step.)
// conj(P) (the adjoint) turns the sign of E's imaginary part, which sits in its
// three constants gi.
template <bool SCALED>
struct ColumnProp {
  float c;
  float2 g0, g1;
  float3 gi;  // E.y = gi.x + Dt.x gi.y + Dt.y gi.z, the sign of conj(P) in it
  __device__ __forceinline__ ColumnProp(const AxisArgs& p, float2 dx, float2 dy) {
    const float2 dxy = cadd(cadd(dx, dy), cmul(dx, dy));
    c = SCALED ? 1.f : p.scale;
    g0 = cscale(dxy, c);
    g1 = make_float2(c * (1.f + dxy.x), g0.y);
    const float sg = p.conj_p ? -1.f : 1.f;
    gi = make_float3(sg * g0.y, sg * g1.y, sg * g1.x);
  }
  __device__ __forceinline__ float2 operator()(const AxisArgs& p, float2 w, float2 dt) const {
    const float ex = fmaf(dt.x, g1.x, fmaf(-dt.y, g1.y, g0.x));
    const float ey = fmaf(dt.x, gi.y, fmaf(dt.y, gi.z, gi.x));
    const float2 we = make_float2(fmaf(w.x, ex, -w.y * ey), fmaf(w.x, ey, w.y * ex));
    if constexpr (SCALED)
      return __ffma2_rn(w, dup(p.scale), __fmul2_rn(we, dup(p.scale)));
    else return __ffma2_rn(w, dup(c), we);
  }
};

// The propagator on a column's registers, which hold A_hat(kx, ky, Omega_k) at
// k = pos_last; pt: the field's tau factors.  (The kernels are instantiated for both
// kinds of grid where the plan has 2^k points: a branch here cost grids of 2^k points
// 2 to 8 % of their step.)
template <class PL, bool SCALED>
__device__ __forceinline__ void apply_prop(float2 (&v)[PL::E], const AxisArgs& p, const ColumnProp<SCALED>& g,
                                           const float2* pt, int t) {
  constexpr int RL = fft_radix<PL, false>(PL::NP - 1);
#pragma unroll
  for (int b = 0; b < PL::E / RL; ++b)
#pragma unroll
    for (int r = 0; r < RL; ++r)
      v[b * RL + r] = g(p, v[b * RL + r], pt[pos_last<PL, false>(t + b * PL::T, r)]);
}

// Resident CTAs of 256 threads that the plain tau-pass asks the register allocator for;
// larger CTAs (2048 and 4096 points, 1024 threads) have 64 registers a thread anyway.
// What takes it are the plans that the pipelined one below leaves: measured per step
// with 1, 2, 3 and 4, lengths of up to 48 points lie within 2 % of each other, 32 points
// gain 1.5 % from 4 (63.3 us against 64.3 on 2 x 128x512x32) and 96 points lose 10 % to
// it (2 x 256x96x1: 10.7 us with 1 and 2, 11.1 with 3, 11.9 with 4).
template <class PL>
__host__ __device__ constexpr int tprop_min_blocks() {
  return tiles_per_cta<PL>() * tile_threads<PL>() > 256 ? 1 : PL::E > 16 ? 2 : PL::E > 8 ? 3 : 4;
}

// Forward tau-FFT, propagator multiply, inverse tau-FFT, in one pass.
template <class PL, bool SCALED, int THREADS, class TW = TwShared>
__device__ __forceinline__ void tprop_tile(const AxisArgs& p, long long cta_tile, const TW& tw, float2* xch) {
  constexpr int N = PL::N, T = PL::T, TX = ColTile<PL>::value;
  constexpr int TPC = tiles_per_cta_t<PL, THREADS>();
  static_assert(TPC >= 1 && TPC * T * TX == THREADS, "CTA must hold whole tiles");
  const int lt = threadIdx.x % (T * TX), tl = threadIdx.x / (T * TX);
  const int tx = lt % TX, t = lt / TX;
  const AxisTile<N, 2, TX> a(p, cta_tile * TPC + tl, tx);
  const XchCol<TX> xc{xch + tl * N * TX, tx};
  float2 v[PL::E];
  load_pencil<PL, false>(v, a.base, a.stride, t, a.act);
  fft_run<PL, false, 0, XchCol<TX>, SyncBlock, TW>(v, t, xc, tw);
  const float2 zero = make_float2(0.f, 0.f);
  const ColumnProp<SCALED> g(p, a.act ? p.px[a.f * p.nx + a.x] : zero, a.act ? p.py[a.f * p.ny + a.other] : zero);
  apply_prop<PL>(v, p, g, p.pt + (a.act ? a.f * p.nt : 0), t);
  // the inverse's first pass reads exactly these positions
  fft_run<PL, true, 0, XchCol<TX>, SyncBlock, TW>(v, t, xc, tw);
  if (a.act) store_pencil<PL, false>(v, a.base, a.stride, t);
}

// ------------------------------------------------- pipelined tau-pass
// The same pass by persistent CTAs that copy their next tile (cp.async, 16
// bytes) into one buffer while they transform the current one in the other, so
// the wait for memory overlaps the transforms.  Tiles are 8 columns wide (rows of
// 64 bytes) for the plans of 16 or more threads per pencil and 128/T for those of
// 8, small enough for two buffers and several CTAs per SM, and the exchanges run
// in the tile's own buffer.
// Taken by the two-pass plans (one exchange per transform) and by the plans of 32
// threads per pencil, whose 16-column tile leaves room for one CTA per SM.
// Measured per launch, plain tau-pass against this one: 512 points (three fields
// of 256x256) 463 -> 415 us, 256 (three of 128x128) 57 -> 49, 128 (two of 512x512)
// 231 -> 212, 64 (two of 1024x256) 127 -> 115, 768 (two of 192x192, then in four
// passes) 388 -> 348.  (Plans of four passes, replaced since, lost 1 to 5 % on 192 and
// 384 points to their block barriers.)
// What bounds it: latency between the phases of a tile at 12 to 16 warps per SM
// (512 points: issue 47 %, FP32 pipe 43 %, shared memory 47 %, DRAM 47 %); plans
// with 16 values per thread and twice the warps were slower (494 to 580 us).
template <class PL>
__host__ __device__ constexpr bool tau_pipe() { return PL::T >= 8 && PL::T <= 32 && (PL::NP == 2 || PL::T == 32); }
template <class PL>
__host__ __device__ constexpr int tau_pipe_cols() { return PL::T >= 16 ? 8 : 128 / PL::T; }
template <class PL>
__host__ __device__ constexpr int tau_pipe_threads() { return PL::T * tau_pipe_cols<PL>(); }
template <class PL>
__host__ __device__ constexpr int tau_pipe_smem() {
  return (2 * PL::N * tau_pipe_cols<PL>() + tw_table_size<PL>()) * (int)sizeof(float2);
}
// Resident CTAs: as many as shared memory holds, at most 512 threads per SM (128
// registers) where a thread's values or its tile of 8 columns need them, 768 (80)
// for the 128-point plan, 1024 for 64 points.  (256 points: 49 us with 512
// threads, 53 with 640, 57 with 768; 128 points: 226, 218, 212.)
template <class PL>
__host__ __device__ constexpr int tau_pipe_ctas() {
  const int fit = 227 * 1024 / (tau_pipe_smem<PL>() + 1024);
  const int most = (PL::E <= 8 ? 1024 : PL::T == 8 ? 768 : 512) / tau_pipe_threads<PL>();
  return fit < most ? fit : most;
}

// tile number `tile` of a pipelined tau kernel: its (field, y, x) and its first
// column in memory
template <int TX>
struct PipeTile {
  int f, y, x;
  float2* base;
  __device__ __forceinline__ PipeTile(const AxisArgs& p, long long tile) {
    x = (int)(tile % p.xtiles) * TX;
    const long long rest = tile / p.xtiles;
    y = (int)(rest % p.ny);
    f = (int)(rest / p.ny);
    base = p.data + (long long)f * p.fstride + (long long)y * p.nx + x;
  }
};
// requests the thread's share of a tile, in 16-byte pieces, into [tau][column]
template <class PL>
__device__ __forceinline__ void pipe_copy(const AxisArgs& p, long long tile, float2* buf) {
  constexpr int TX = tau_pipe_cols<PL>();
  constexpr int PAIRS = TX / 2, ROWS = tau_pipe_threads<PL>() / PAIRS;  // pieces per row, rows per copy step
  const PipeTile<TX> a(p, tile);
  const long long plane = (long long)p.nx * p.ny;
  const int c = 2 * (threadIdx.x % PAIRS), row = threadIdx.x / PAIRS;
  if (a.x + c >= p.nx) return;  // nx is even
  const float2* src = a.base + c + row * plane;
  const unsigned dst = (unsigned)__cvta_generic_to_shared(buf + row * TX + c);
#pragma unroll
  for (int q = 0; q < PL::N / ROWS; ++q)
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst + q * ROWS * TX * 8),
                 "l"(src + (long long)(q * ROWS) * plane)
                 : "memory");
}
template <class PL>
using PipeXch = typename std::conditional<tau_pipe_cols<PL>() == 8, XchCol8, XchCol<tau_pipe_cols<PL>()>>::type;
// the thread's first-pass inputs of a tile that has arrived
template <class PL>
__device__ __forceinline__ void pipe_take(float2 (&v)[PL::E], const PipeXch<PL>& xc, int t) {
  constexpr int R0 = fft_radix<PL, false>(0);
#pragma unroll
  for (int i = 0; i < PL::E / R0; ++i)
#pragma unroll
    for (int r = 0; r < R0; ++r) v[i * R0 + r] = xc.ld(pos_first<PL, false>(t + i * PL::T, r));
}

template <class PL, bool SCALED>
__global__ void __launch_bounds__(tau_pipe_threads<PL>(), tau_pipe_ctas<PL>())
    tpass_pipe_kernel(const AxisArgs p) {
  constexpr int N = PL::N, TX = tau_pipe_cols<PL>(), THREADS = tau_pipe_threads<PL>();
  using X = PipeXch<PL>;
  extern __shared__ float4 sm4[];
  float2* buf = reinterpret_cast<float2*>(sm4);
  float2* tw = buf + 2 * N * TX;
  for (int i = threadIdx.x; i < tw_table_size<PL>(); i += THREADS) tw[i] = p.tw[i];
  const long long plane = (long long)p.nx * p.ny;
  const int tx = threadIdx.x % TX, t = threadIdx.x / TX;
  long long k = blockIdx.x;  // tiles from the last down
  chain_begin();
  if (k < p.ntiles) pipe_copy<PL>(p, p.ntiles - 1 - k, buf);
  cp_async_commit();
  for (int b = 0; k < p.ntiles; k += gridDim.x, b ^= 1) {
    cp_async_wait<0>();
    __syncthreads();  // the tile is there, and the last one's buffer is free
    if (k + gridDim.x < p.ntiles) pipe_copy<PL>(p, p.ntiles - 1 - (k + gridDim.x), buf + (b ^ 1) * N * TX);
    cp_async_commit();
    const PipeTile<TX> a(p, p.ntiles - 1 - k);
    const bool act = a.x + tx < p.nx;
    // the column's factors, requested ahead of the forward transform
    const float2 dx = act ? p.px[a.f * p.nx + a.x + tx] : make_float2(0.f, 0.f), dy = p.py[a.f * p.ny + a.y];
    const X xc{buf + b * N * TX, tx};
    float2 v[PL::E];
    pipe_take<PL>(v, xc, t);
      fft_run<PL, false, 0, X, SyncBlock, TwShared>(v, t, xc, TwShared{tw});
    apply_prop<PL>(v, p, ColumnProp<SCALED>(p, dx, dy), p.pt + a.f * p.nt, t);
    fft_run<PL, true, 0, X, SyncBlock, TwShared>(v, t, xc, TwShared{tw});
    if (act) store_pencil<PL, false>(v, a.base + tx, plane, t);
  }
}

// y-pass of a z-step
template <class PL, bool INV>
__global__ void __launch_bounds__(tiles_per_cta<PL>() * tile_threads<PL>())
    ypass_kernel(const AxisArgs p) {
  constexpr int THREADS = tiles_per_cta<PL>() * tile_threads<PL>();
  extern __shared__ float4 sm4[];
  if constexpr (axis_tw_staged<PL, INV>()) {
    float2* tw = reinterpret_cast<float2*>(sm4);
    for (int i = threadIdx.x; i < tw_table_size<PL>(); i += blockDim.x) tw[i] = p.tw[i];
    __syncthreads();
    chain_begin();
    axis_tile<PL, INV, 1, THREADS>(p, blockIdx.x, TwShared{tw}, tw + tw_table_size<PL>());
  } else {
    chain_begin();
    axis_tile<PL, INV, 1, THREADS>(p, blockIdx.x, TwGlobal{p.tw}, reinterpret_cast<float2*>(sm4));
  }
}

template <class PL, bool SCALED>
__global__ void __launch_bounds__(tiles_per_cta<PL>() * tile_threads<PL>(), tprop_min_blocks<PL>())
    tpass_prop_kernel(const AxisArgs p) {
  constexpr int THREADS = tiles_per_cta<PL>() * tile_threads<PL>();
  extern __shared__ float4 sm4[];
  if constexpr (tw_in_smem<PL>()) {
    float2* tw = reinterpret_cast<float2*>(sm4);
    for (int i = threadIdx.x; i < tw_table_size<PL>(); i += blockDim.x) tw[i] = p.tw[i];
    __syncthreads();
    chain_begin();
    // tiles from the last down: the pass ends on the first field's low-y
    // pencils, which the y-inverse then reads first
    tprop_tile<PL, SCALED, THREADS>(p, (long long)gridDim.x - 1 - blockIdx.x, TwShared{tw},
                            tw + tw_table_size<PL>());
  } else {
    chain_begin();
    tprop_tile<PL, SCALED, THREADS>(p, blockIdx.x, TwGlobal{p.tw}, reinterpret_cast<float2*>(sm4));
  }
}

// ------------------------------------------------------------ dispatchers
// Each returns cudaErrorInvalidValue for an unsupported length.
cudaError_t run_xpass(int nx, int nf, const XPassArgs& a, cudaStream_t s);
cudaError_t run_ypass(int ny, bool inv, const AxisArgs& a, cudaStream_t s);
cudaError_t run_tpass_prop(int nt, const AxisArgs& a, cudaStream_t s);
bool size_supported(int n);
int col_tile_of(int n);      // columns per tile of the y/tau FFT kernels
int tau_col_tile_of(int n);  // columns per tile of the tau propagator kernel

// grouped x-pass of the batched form (k_xgroup.cu): the same x-pass for
// ninst instances of one shape stored one after another (2 fields each,
// base.data the first, base.fstride between fields, base.rows = ny nt rows
// per instance, base.tw the x twiddles); the instance parameters come from
// gi[0..ninst); step < 0 is the first half step of step 0.
struct GroupInst {
  float kh[2], kh2[2];  // kappa_f dz/2 (1/2 on the SH equation) and half of it
  double dk, dz;
  int nz;
};
// ecoef: the instances' stage factors, instance i's for step j at
// ecoef[i stride + (j + 1) kStageFactors + 0..]
cudaError_t run_xpass_group(int nx, const XPassArgs& base, const GroupInst* gi, const float2* ecoef, int stride,
                            int step, int ninst, cudaStream_t s);
// the same pass of the grouped form on ninst instances (k_planegroup.cu)
cudaError_t run_plane_group(int nx, int ny, const XPassArgs& base, const float2* twy, const GroupInst* gi,
                            const float2* ecoef, int stride, int step, int ninst, cudaStream_t s);
int xpass_rows_of(int nx);  // rows per CTA of the x-pass of length nx

// plane pass (k_plane.cu): y-inverse, x-pass and y-forward of a step in one
// kernel, for the (nx, ny) below; a.mode NL_FIRST, NL_MID or NL_LAST, no map
bool plane_supported(int nx, int ny);
cudaError_t run_plane(int nx, int ny, int nf, const XPassArgs& a, const float2* twy, cudaStream_t s);
cudaError_t run_plane3(int nx, int ny, const XPassArgs& a, const float2* twy, cudaStream_t s);

// single transforms (k_single.cu), the turns as products (TwProduct): rows of x (rows:
// of all fields, one behind another; the output times scale + scale_lo) and, with
// a.twp, the y axis or the tau axis
struct XLineArgs {
  float2* data;
  long long rows;
  const float4* twp;
  float scale, scale_lo;
};
cudaError_t run_xline_fft(int nx, bool inv, const XLineArgs& a, cudaStream_t s);
cudaError_t run_axis_fft(int n, int axis, bool inv, const AxisArgs& a, cudaStream_t s);

// misc kernels (k_misc.cu)
// TMA tau-pass (k_tma.cu)
bool tma_tau_supported(int nx, int nt);
cudaError_t make_tau_tensor_map(void* map128, const float2* data, int nx, int ny, int nt, int nf, int tx);
// wait_ns bounds each wait for a tile's copy; on expiry *err is set
cudaError_t run_tpass_prop_tma(int nt, int tx, const void* map128, const AxisArgs& a, int* err,
                               unsigned long long wait_ns, cudaStream_t s);

// per-pass twiddle table of the plan of length n on an axis (0 x, 1 y, 2 tau), built on
// the host in FP64, and its size in entries: the turns as shears, or as products (cosine
// and sine as hi + lo floats); fill_twiddles is false for an unsupported length
int tw_table_size_of(int n, int axis);
bool fill_twiddles(float2* host, int n, int axis);
bool fill_twiddles(float4* host, int n, int axis);
cudaError_t upload_twiddles(float2* tw, int n, int axis, cudaStream_t s);
// 1/n = scale (1 + rest); rest = 0 for a power of two
struct Norm {
  float scale;
  double rest;
};
inline Norm norm_of(double n) {
  const float scale = (float)(1.0 / n);
  return {scale, 1.0 / n / (double)scale - 1.0};
}
// rest (of 1/(nx ny nt)) goes into pt, or into py on a cw grid (nt = 1, ny > 1), whose
// linear step transforms y
struct TableArgs {
  float2* px;
  float2* py;
  float2* pt;
  int nx, ny, nt, nf;
  double dx, dy, dt, dz;
  double k[3], rho[3], delta[3], k2[3], k3[3], alpha[3];
  double rest;
};
cudaError_t run_prop_tables(const TableArgs& a, cudaStream_t s);
// Stage phase factors of one x-pass under a transverse mismatch map m(x, y):
// Phi(x, y, z) = Phi(z) + m z.  With zj the distance of the B step's start
// (phiB = Phi there, dkB its mismatch) and zA that of the A step's start,
//   emap[0] = e^{i (phiB + dkB dz/2 + m (zj + dz/2))},  emap[1] = e^{i (dkB + m) dz/4},
//   emap[2] = e^{i (phiA + m zA)},                        emap[3] = e^{i (dkA + m) dz/4},
// each [ny][nx]; phases in FP64 reduced mod 2 pi before the FP32 sincos.
// The map's share of the coupling phase at a point is Q = P + m (z - zp):
// P the integral of the maps in effect before zp, m the map in effect since.
// mapB is the map of the step whose B half step this x-pass applies, mapA
// that of the next step's A half step; when they differ (advance != 0) the
// kernel brings P up to zA (P += mapB (zA - zp)) and the A factors start
// from there.
struct MapArgs {
  const double* mapB;
  const double* mapA;
  double* mphase;  // P [ny][nx]
  float2* emap;
  long long nxy;
  double phiB, dkB, zB, phiA, dkA, zA, dz, zp;
  int advance;
};
cudaError_t run_map_tables(const MapArgs& a, cudaStream_t s);
// P += m * len at every point (a map replaced between propagations)
cudaError_t run_map_phase_advance(double* mphase, const double* m, double len, long long nxy, cudaStream_t s);
// the linear step's multiply element by element (grids with ny = nt = 1)
cudaError_t run_prop_pointwise(const AxisArgs& a, int nf, cudaStream_t s);
// diagnostics (k_diag.cu): out[f nt + k] = sum_{x,y} |A_f(tau_k)|^2, and
// out[f nt + m] += sum_{x,y} |DFT_tau A_f|^2 (m) (out zeroed by the caller;
// a: tau-axis arguments without the propagator)
cudaError_t run_power_trace(const float2* data, int nx, int ny, int nt, int nf, long long fstride, double* out,
                            cudaStream_t s);
cudaError_t run_tau_spectrum(int nt, const AxisArgs& a, double* out, cudaStream_t s);

// thermal model (k_thermal.cu)
struct HeatArgs {
  const float2* data;
  long long fstride;
  int nx, ny, nt, nf;
  double c[3];  // weight * alpha_f * 1/2 c eps0 n_f (* rep_rate dt for nt > 1)
  double* heat;  // [ny][nx], accumulated into
};
cudaError_t run_heat_load(const HeatArgs& a, cudaStream_t s);
// sine-transform tables for one axis of even length n > 1: 2n entries
cudaError_t run_sine_twiddles(double2* tw, int n, cudaStream_t s);
bool sine_length_supported(int n);
struct ThermalArgs {
  const double* heat;  // [ny][nx] W/m^3
  double* temp;        // [ny][nx] K, output (also the transform's work array)
  const double2* twx;  // sine-transform tables of nx and ny
  const double2* twy;
  int nx, ny;
  double dx, dy, kappa;
  double dkdT;
  double* dkmap;  // [ny][nx] 1/m, output
  int* bad;       // set if a temperature is not finite
};
cudaError_t run_thermal_solve(const ThermalArgs& a, int* nlaunch, cudaStream_t s);
// Per-field sums of |A|^2 over n points (even) of src[f], 16-byte aligned, into
// host[f] (pinned), with the device error word in host[3]; dst[f] not NULL: the
// field is copied there too.  partial: nf x nblocks; *count is zero before the
// first launch and after every one.
struct EnergyArgs {
  const float2* src[3];
  float2* dst[3];
  long long n;
  double* partial;
  double* host;
  unsigned int* count;
  const int* err;
};
cudaError_t run_energy(const EnergyArgs& a, int nf, int nblocks, cudaStream_t s);
// d0 = s0 and d1 = s1, n points (even) each, 16-byte aligned
cudaError_t run_copy_pair(const float2* s0, float2* d0, const float2* s1, float2* d1, long long n, cudaStream_t s);
cudaError_t run_c128_to_c64(const double2* in, float2* out, long long n, cudaStream_t s);
cudaError_t run_c64_to_c128(const float2* in, double2* out, long long n, cudaStream_t s);

// adjoint recomputation and reverse x-pass (k_xadj.cu)
// x-pass that also records the states entering its half steps (a.rec_b, a.rec_a)
cudaError_t run_xpass_record(int nx, int nf, const XPassArgs& a, cudaStream_t s);
cudaError_t run_xpass_record_map(int nx, int nf, const XPassArgs& a, cudaStream_t s);
// Reverse of one x-pass boundary: the adjoint g, in (kx, y, tau) when
// from_k (else real space), goes through the inverse x-FFT, the reverse of
// the A half step at state xa (if xa), the reverse of the B half step at
// state xb (if xb), and the forward x-FFT when to_k.  Each CTA writes its
// six stage-phase sensitivity sums (A: start, middle, end; B: the same) to
// partial[blockIdx.x][6]; *ncta receives the CTA count.
struct XAdjArgs {
  float2* g;
  const float2* xa;
  const float2* xb;
  int xa_row_order;    // xa lies in row order (a checkpoint), not as recorded
  long long fstride, rows;
  const float2* tw;
  int from_k, to_k;
  double phiA, dkA, phiB, dkB, dz;  // phase at the start and mismatch of the steps b (A) and b - 1 (B), as in XPassArgs
  float kh[3];                     // kappa_f h (1/2 on the SH equation for two fields)
  float kh2[3];                    // kh / 2 (exact)
  double* partial;
  // transverse mismatch map: the per-(x, y) stage phase factors of this
  // boundary's B and A half steps [4][ny][nx] (as in XPassArgs), or NULL
  const float2* emap;
  int ny;
  // map-free: the stage factors as in XPassArgs, written by the host dispatcher in
  // FP64 from the phases above
  float2 ecoef[kStageFactors];
};
cudaError_t run_xpass_adjoint(int nx, int nf, const XAdjArgs& a, long long* ncta, cudaStream_t s);
cudaError_t run_xpass_adjoint_map(int nx, int nf, const XAdjArgs& a, long long* ncta, cudaStream_t s);
// sensA[k] = sum_c partial[c][k], sensB[k] = sum_c partial[c][3 + k] (either may be NULL)
cudaError_t run_sens_boundary(const double* partial, long long ncta, double* sensA, double* sensB, cudaStream_t s);
long long xpass_adjoint_ctas(int nx, long long rows);

// adjoint kernels (k_adjoint.cu)
cudaError_t run_scale_fields(const float2* a, float2* g, long long n, int nf, long long fstride, const float* s,
                             cudaStream_t st);
cudaError_t run_phase_grad(const float2* gh, const float2* ah, long long plane, int nt, double* acc, cudaStream_t s);
cudaError_t run_phase_tables(float2* px, int nx, float2* py, int ny, float2* pt, int nt, const double* phi, int sign,
                             double rest, cudaStream_t s);

}  // namespace brahms

// Supported transform lengths (each needs an FftPlan).
#define BRAHMS_FOR_EACH_SIZE(X) \
  X(2) X(4) X(8) X(16) X(32) X(64) X(128) X(256) X(512) X(1024) X(2048) X(4096) \
  X(6) X(12) X(24) X(48) X(96) X(192) X(384) X(768)

// Planes with a plane-pass kernel: rows of 16 to 64 points and columns of 8 to 64, up to
// 1536 points.  (On other planes of up to 1536 points, with rows of up to 12 points or of
// 96 and more or columns of up to 6, it has not been tried; they take the four passes.)
// A larger plane keeps one CTA busy for longer than the three passes take over the
// whole GPU.
// Time per z-step of the plane pass with the tau-pass against the four passes, 64 / 512
// planes: two fields 16x16 7.0 against 13.6 us / 12.3 against 17.7, 32x32 7.4 against
// 10.5 / 17.8 against 22.6, 24x64 10.6 against 12.8 / 29.0 against 32.4; three fields
// 32x32 10.1 against 12.0 / 26.7 against 29.5, 24x64 13.8 against 15.6 / 39.0 against
// 43.9, 48x32 13.1 against 14.2 / 40.2 against 41.2, 64x24 12.6 against 12.7 / 40.9
// against 40.4.  Where it loses, by up to 5 %, are 512 planes and more: 24x24 with two
// fields (21.3 against 20.6), 32x8, 48x8 and 48x24 with three (15.8 against 15.2).  Past
// 1536 points, two fields: 48x48 14.6 against 14.4 / 48.0 against 47.0, 64x64 17.2
// against 14.0 / 56.9 against 55.7, 96x96 45.5 against 29.2 / 197 against 161.
#define BRAHMS_FOR_EACH_PLANE(X)                                        \
  X(16, 8) X(16, 12) X(16, 16) X(16, 24) X(16, 32) X(16, 48) X(16, 64)  \
  X(24, 8) X(24, 12) X(24, 16) X(24, 24) X(24, 32) X(24, 48) X(24, 64)  \
  X(32, 8) X(32, 12) X(32, 16) X(32, 24) X(32, 32) X(32, 48)            \
  X(48, 8) X(48, 12) X(48, 16) X(48, 24) X(48, 32)                      \
  X(64, 8) X(64, 12) X(64, 16) X(64, 24)
