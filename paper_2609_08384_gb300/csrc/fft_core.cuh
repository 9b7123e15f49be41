// Register-resident mixed-radix Stockham FFT building blocks for sm_103a.
//
// A pencil of length N is owned by T = N/E threads; each thread keeps E
// complex values in registers.  One Stockham pass of radix R (Govindaraju et
// al., "High performance discrete Fourier transforms on graphics processors",
// SC'08, autosort formulation) combines the R sub-transforms of butterfly j,
// multiplying number r by W_{NS R}^{r m} (NS the product of the radices of the
// earlier passes, m = j mod NS), with a radix-R DFT, and writes the results to
// (j/NS) NS R + m + k NS.  Between passes the values are exchanged through
// shared memory; the first pass reads its inputs straight from global memory
// and the last pass leaves the outputs in registers, so a kernel stores them
// with coalesced writes and never stages the whole pencil twice.
//
// Centred indices.  The digits of both indices of a twiddle are taken in
// centred form (digit d of radix R as d or d - R, in [-R/2, R/2)), so that no
// twiddle turns by much more than a quarter of the circle.  A sub-transform of
// r - R takes its inputs one place later than that of r, and with m' in the
// place of m output k is number m' + k NS: the butterflies and exchanges stay
// as they are, and only the positions of the first pass's inputs and of the
// last pass's outputs move (pos_first, pos_last).
//
// Twiddles as shears.  A turn by phi is the product of three shears,
//   x += p y,  y += s x,  x += p y,  p = -tan(phi / 2), s = sin(phi)
// (the lifting form of a plane rotation; Buneman's tan/sin twiddles): three
// FMAs where the product with a twiddle held as hi + lo floats took eight.
// Each shear has determinant 1 whatever the rounding of p and s, and the same
// three shears with the signs turned are its exact inverse.  The inverse
// transform is built as the exact mirror of the forward one (decimation in
// frequency against decimation in time: the same twiddles on the same values,
// and codelets whose inner factors mirror each other), so what the rounded
// twiddles do to a field the way back undoes, and the energy of a field that
// passes them again and again does not drift.  (With c and s rounded to single
// floats |c + i s| differs from 1 and it does; a pair of directions that are
// not each other's mirror let the energy of the 3 x 256x256x512 parametric run
// fall by 7e-9 per step.)  |phi| <= 1/4 turn, or a little more in plans of three
// passes, keeps p near 1 or below.
// Error against FP64 of 3D transforms of random fields by shears: forward 1.6e-7 (by
// products with hi + lo twiddles 1.5e-7), forward and inverse 2.11e-7 (2.10e-7); energy
// of smooth beams over 100 z-steps: rms 1.6e-9 to 2.6e-9 per step (1.7e-9 to 5.6e-9).
// Transforms that nothing takes back turn by products (TwProduct, k_single.cu).
//
// Packed arithmetic.  A complex value is an aligned register pair, and sums of
// complex values are single add/sub.f32x2 instructions.  One FFMA2 occupies the
// FP32 pipe as long as two FFMA but takes one issue slot, so packed sums leave
// issue slots to the loads, address arithmetic and exchanges (measured per 16
// FMA lanes and warp: FFMA with 4 logic operations 10.9 ns, FFMA2 with 4 logic
// operations 8.5 ns, either alone 8.0 - 8.3 ns).
//
// The forward transform is unnormalised with e^{-2 pi i m n / N}; the inverse
// uses e^{+...} and the radix order reversed, so that the inverse's first
// pass reads exactly the positions the forward's last pass produced.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include <type_traits>

namespace brahms {

// First call of a kernel launched with launch_chained: waits until the grids
// before it on the stream have ended and their writes are visible.  Only tables
// that no kernel of the chain writes may be read before it.  (No kernel releases
// its dependents early: launch_dependents at the start of every kernel made steps
// on states beyond the L2 8 to 11 % slower, 1306 -> 1432 us on 3 x 256x256x512,
// and small ones no faster.)
__device__ __forceinline__ void chain_begin() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

__device__ __forceinline__ float2 cadd(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float2 csub(float2 a, float2 b) {
  float2 d;
  asm("{\n .reg .b64 x, y, z;\n mov.b64 x, {%2, %3};\n mov.b64 y, {%4, %5};\n sub.rn.f32x2 z, x, y;\n"
      " mov.b64 {%0, %1}, z;\n}"
      : "=f"(d.x), "=f"(d.y)
      : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
  return d;
}
__device__ __forceinline__ float2 cmul(float2 a, float2 b) {
  return make_float2(fmaf(a.x, b.x, -a.y * b.y), fmaf(a.x, b.y, a.y * b.x));
}
__device__ __forceinline__ float2 cscale(float2 a, float s) { return make_float2(a.x * s, a.y * s); }
// a + t^Q b, t = -i (forward) or +i (inverse), Q taken mod 4: a quarter turn of
// b is a choice of the components that are added or subtracted
template <bool INV, int Q>
__device__ __forceinline__ float2 add_turned(float2 a, float2 b) {
  constexpr int q = ((INV ? -Q : Q) % 4 + 4) % 4;
  if constexpr (q == 0) return cadd(a, b);
  else if constexpr (q == 2) return csub(a, b);
  else if constexpr (q == 1) return make_float2(a.x + b.y, a.y - b.x);
  else return make_float2(a.x - b.y, a.y + b.x);
}

// a turn by the three shears of (p, s) (see the header)
__device__ __forceinline__ float2 shear_turn(float2 a, float p, float s) {
  const float x = fmaf(p, a.y, a.x);
  const float y = fmaf(s, x, a.y);
  return make_float2(fmaf(p, y, x), y);
}

// A turn by a table entry, and the turn back: by the shears of w, or by the product
// with (cos + i sin) as hi + lo floats, w = (cos hi, sin hi, cos lo, sin lo), which
// single transforms take (TwProduct)
__device__ __forceinline__ float2 turn(float2 a, float2 w) { return shear_turn(a, w.x, w.y); }
__device__ __forceinline__ float2 turn_back(float2 a, float2 w) { return shear_turn(a, -w.x, -w.y); }
__device__ __forceinline__ float2 turn(float2 a, float4 w) {
  return make_float2(fmaf(w.x, a.x, fmaf(-w.y, a.y, fmaf(w.z, a.x, -w.w * a.y))),
                     fmaf(w.x, a.y, fmaf(w.y, a.x, fmaf(w.z, a.y, w.w * a.x))));
}
__device__ __forceinline__ float2 turn_back(float2 a, float4 w) {
  return turn(a, make_float4(w.x, -w.y, w.z, -w.w));
}

// ---------------------------------------------------------------- codelets
// tan(pi k / 32), sin(pi k / 16) and cos(pi k / 16), k = 0..4
__host__ __device__ constexpr double tan_pi32(int k) {
  return k == 0 ? 0.0
       : k == 1 ? 0.098491403357164253077197521291327
       : k == 2 ? 0.19891236737965800691159762264468
       : k == 3 ? 0.30334668360734239167588394694130
                : 0.41421356237309504880168872420970;
}
__host__ __device__ constexpr double sin_pi16(int k) {
  return k == 0 ? 0.0
       : k == 1 ? 0.19509032201612826784828486847702
       : k == 2 ? 0.38268343236508977172845998403040
       : k == 3 ? 0.55557023301960222474283081394853
                : 0.70710678118654752440084436210485;
}
__host__ __device__ constexpr double cos_pi16(int k) {
  return k == 0 ? 1.0
       : k == 1 ? 0.98078528040323044912618223613424
       : k == 2 ? 0.92387953251128675612818318939679
       : k == 3 ? 0.83146961230254523707878837761791
                : 0.70710678118654752440084436210485;
}
// W32^E = (-/+ i)^quarter(E) W32^rest(E), rest in [-3, 4]
__host__ __device__ constexpr int w32_quarter(int e) { return ((e + 3) / 8) % 4; }
__host__ __device__ constexpr int w32_rest(int e) { return e - 8 * ((e + 3) / 8); }
// a times W32^rest(E); the quarter turns are left to the additions that follow.
// PROD: the product with hi + lo floats, for single transforms
template <bool INV, int E, bool PROD>
__device__ __forceinline__ float2 w32_turn(float2 a) {
  constexpr int k = w32_rest(E);
  if constexpr (k == 0) return a;
  else {
    constexpr int ak = k < 0 ? -k : k;
    // forward: phi = -2 pi k / 32
    constexpr bool pos = (k < 0) != INV;
    if constexpr (ak == 4) {
      // one eighth of a turn: (x -/+ y) / sqrt 2 with the factor as hi + lo.  The
      // turn most used is kept exact: as rounded shears it is 1.9e-8 short of
      // orthogonal, and smooth beams lost 7e-9 of their energy per z-step
      const float2 d = pos ? make_float2(a.x - a.y, a.x + a.y) : make_float2(a.x + a.y, a.y - a.x);
      constexpr float ch = (float)sin_pi16(4), cl = (float)(sin_pi16(4) - (double)ch);
      return __ffma2_rn(d, make_float2(ch, ch), __fmul2_rn(d, make_float2(cl, cl)));
    } else if constexpr (PROD) {
      constexpr double c = cos_pi16(ak), sn = pos ? sin_pi16(ak) : -sin_pi16(ak);
      constexpr float ch = (float)c, sh = (float)sn;
      return turn(a, make_float4(ch, sh, (float)(c - (double)ch), (float)(sn - (double)sh)));
    } else {
      // one sixteenth of a turn: p one float off tan(pi/16) makes the pair of
      // floats eight times nearer to orthogonal (7e-10 against 6e-9) for an angle
      // 6e-8 off, which the way back undoes: energy of the 1000-step parametric
      // run +2.3e-7 instead of -7.4e-7 (a single transform shows it: 8 % more error
      // at 256 and 512 points)
      constexpr float pk = ak == 2 ? 0.198912397f : (float)tan_pi32(ak);
      constexpr float sk = ak == 2 ? 0.382683486f : (float)sin_pi16(ak);
      return shear_turn(a, pos ? -pk : pk, pos ? sk : -sk);
    }
  }
}

template <bool INV>
__device__ __forceinline__ void dft2(float2& a, float2& b) {
  float2 t = a;
  a = cadd(t, b);
  b = csub(t, b);
}

// four-point DFT of v0, t^Q1 v1, t^Q2 v2, t^Q3 v3 (pending quarter turns)
template <bool INV, int Q1 = 0, int Q2 = 0, int Q3 = 0>
__device__ __forceinline__ void dft4(float2& v0, float2& v1, float2& v2, float2& v3) {
  const float2 a = add_turned<INV, Q2>(v0, v2), b = add_turned<INV, Q2 + 2>(v0, v2);
  const float2 c = add_turned<INV, Q3 - Q1>(v1, v3), d = add_turned<INV, Q3 - Q1 + 2>(v1, v3);
  v0 = add_turned<INV, Q1>(a, c);
  v2 = add_turned<INV, Q1 + 2>(a, c);
  v1 = add_turned<INV, Q1 + 1>(b, d);
  v3 = add_turned<INV, Q1 + 3>(b, d);
}

// sin(pi/3) as hi + lo floats: in the three-point DFT it is a factor, not a
// turn, so its rounding would change the energy of a field a little each time
constexpr double kS3d = 0.86602540378443864676372317075294;
constexpr float kS3 = (float)kS3d, kS3lo = (float)(kS3d - (double)(float)kS3d);

template <bool INV>
__device__ __forceinline__ void dft3(float2& v0, float2& v1, float2& v2) {
  const float2 s = cadd(v1, v2);
  const float2 t = __ffma2_rn(s, make_float2(-0.5f, -0.5f), v0);
  const float2 d = csub(v1, v2);
  const float2 u = __ffma2_rn(d, make_float2(kS3, kS3), __fmul2_rn(d, make_float2(kS3lo, kS3lo)));
  v0 = cadd(v0, s);
  v1 = add_turned<INV, 1>(t, u);
  v2 = add_turned<INV, 3>(t, u);
}

// Radix 8: forward n = 4 n1 + n2, k = k1 + 2 k2 as sums over n1, turns by
// W8^{n2 k1}, four-point transforms over n2; the inverse takes the same steps
// backwards (its input number k may carry a pending quarter turn Qk).
template <bool PROD, int Q1 = 0, int Q2 = 0, int Q3 = 0, int Q4 = 0, int Q5 = 0, int Q6 = 0, int Q7 = 0>
__device__ __forceinline__ void idft8(float2* v) {
  static_assert(Q1 == 0, "number 1 carries no turn");
  dft4<true, Q2, Q4, Q6>(v[0], v[2], v[4], v[6]);
  dft4<true, Q3, Q5, Q7>(v[1], v[3], v[5], v[7]);
  const float2 y0[4] = {v[0], v[2], v[4], v[6]};
  const float2 y1[4] = {v[1], w32_turn<true, 4, PROD>(v[3]), v[5], w32_turn<true, 12, PROD>(v[7])};
  v[0] = cadd(y0[0], y1[0]);
  v[4] = csub(y0[0], y1[0]);
  v[1] = cadd(y0[1], y1[1]);
  v[5] = csub(y0[1], y1[1]);
  v[2] = add_turned<true, 1>(y0[2], y1[2]);
  v[6] = add_turned<true, 3>(y0[2], y1[2]);
  v[3] = add_turned<true, 1>(y0[3], y1[3]);
  v[7] = add_turned<true, 3>(y0[3], y1[3]);
}
template <bool INV, bool PROD>
__device__ __forceinline__ void dft8(float2* v) {
  if constexpr (INV) {
    idft8<PROD>(v);
  } else {
    float2 y0[4], y1[4];
#pragma unroll
    for (int n2 = 0; n2 < 4; ++n2) {
      y0[n2] = cadd(v[n2], v[n2 + 4]);
      y1[n2] = csub(v[n2], v[n2 + 4]);
    }
    y1[1] = w32_turn<false, 4, PROD>(y1[1]);
    y1[3] = w32_turn<false, 12, PROD>(y1[3]);
    dft4<false>(y0[0], y0[1], y0[2], y0[3]);
    dft4<false, w32_quarter(4), w32_quarter(8), w32_quarter(12)>(y1[0], y1[1], y1[2], y1[3]);
#pragma unroll
    for (int k2 = 0; k2 < 4; ++k2) {
      v[2 * k2] = y0[k2];
      v[2 * k2 + 1] = y1[k2];
    }
  }
}

// Radix 4 M (M = 4 or 8): n = 4 n1 + n2 (n1 < M, n2 < 4), k = k1 + M k2: M-point
// transforms over n1, turns by W_{4M}^{n2 k1}, four-point transforms over n2
// (radix 16 is its own mirror; radix 32's inverse runs them backwards)
template <bool INV, int M, int K1, bool PROD>
__device__ __forceinline__ void dft4m_column(float2 (&y)[4][M], float2* v) {
  constexpr int U = 8 / M;  // W_{4M} = W32^U
  float2 b0 = y[0][K1], b1 = w32_turn<INV, U * K1, PROD>(y[1][K1]), b2 = w32_turn<INV, 2 * U * K1, PROD>(y[2][K1]),
         b3 = w32_turn<INV, 3 * U * K1, PROD>(y[3][K1]);
  dft4<INV, w32_quarter(U * K1), w32_quarter(2 * U * K1), w32_quarter(3 * U * K1)>(b0, b1, b2, b3);
  v[K1] = b0;
  v[K1 + M] = b1;
  v[K1 + 2 * M] = b2;
  v[K1 + 3 * M] = b3;
  if constexpr (K1 + 1 < M) dft4m_column<INV, M, K1 + 1, PROD>(y, v);
}
template <bool INV, bool PROD>
__device__ __forceinline__ void dft16(float2* v) {
  float2 y[4][4];
#pragma unroll
  for (int n2 = 0; n2 < 4; ++n2) {
#pragma unroll
    for (int n1 = 0; n1 < 4; ++n1) y[n2][n1] = v[4 * n1 + n2];
    dft4<INV>(y[n2][0], y[n2][1], y[n2][2], y[n2][3]);
  }
  dft4m_column<INV, 4, 0, PROD>(y, v);
}
// row n2 of the inverse radix 32: turns by W32^{n2 k1}, eight points over k1
template <int N2, bool PROD>
__device__ __forceinline__ void idft32_row(float2 (&y)[4][8], float2* v) {
  float2* z = y[N2];
  z[1] = w32_turn<true, N2, PROD>(z[1]);
  z[2] = w32_turn<true, 2 * N2, PROD>(z[2]);
  z[3] = w32_turn<true, 3 * N2, PROD>(z[3]);
  z[4] = w32_turn<true, 4 * N2, PROD>(z[4]);
  z[5] = w32_turn<true, 5 * N2, PROD>(z[5]);
  z[6] = w32_turn<true, 6 * N2, PROD>(z[6]);
  z[7] = w32_turn<true, 7 * N2, PROD>(z[7]);
  idft8<PROD, w32_quarter(N2), w32_quarter(2 * N2), w32_quarter(3 * N2), w32_quarter(4 * N2), w32_quarter(5 * N2),
        w32_quarter(6 * N2), w32_quarter(7 * N2)>(z);
#pragma unroll
  for (int n1 = 0; n1 < 8; ++n1) v[4 * n1 + N2] = z[n1];
}
template <bool INV, bool PROD>
__device__ __forceinline__ void dft32(float2* v) {
  float2 y[4][8];
  if constexpr (INV) {
#pragma unroll
    for (int k1 = 0; k1 < 8; ++k1) {
#pragma unroll
      for (int k2 = 0; k2 < 4; ++k2) y[k2][k1] = v[k1 + 8 * k2];
      dft4<true>(y[0][k1], y[1][k1], y[2][k1], y[3][k1]);
    }
    idft32_row<0, PROD>(y, v);
    idft32_row<1, PROD>(y, v);
    idft32_row<2, PROD>(y, v);
    idft32_row<3, PROD>(y, v);
  } else {
#pragma unroll
    for (int n2 = 0; n2 < 4; ++n2) {
#pragma unroll
      for (int n1 = 0; n1 < 8; ++n1) y[n2][n1] = v[4 * n1 + n2];
      dft8<false, PROD>(y[n2]);
    }
    dft4m_column<false, 8, 0, PROD>(y, v);
  }
}

// Radix 3 M (M = 2, 4, 8) by the prime-factor mapping (Good 1958): with
// n = M n1 + 3 n2 and k = M (1/M mod 3) k1 + 3 (1/3 mod M) k2, both mod 3 M, the
// transform is M-point transforms over n2 and three-point ones over n1 with no
// turns between them.
template <bool INV, int M, bool PROD>
__device__ __forceinline__ void dft3m(float2* v) {
  constexpr int N = 3 * M, K1 = M * (M % 3 == 1 ? 1 : 2), K2 = 3 * (M == 2 ? 1 : 3);
  float2 y[3][M];
#pragma unroll
  for (int n1 = 0; n1 < 3; ++n1) {
#pragma unroll
    for (int n2 = 0; n2 < M; ++n2) y[n1][n2] = v[(M * n1 + 3 * n2) % N];
    if constexpr (M == 2) dft2<INV>(y[n1][0], y[n1][1]);
    else if constexpr (M == 4) dft4<INV>(y[n1][0], y[n1][1], y[n1][2], y[n1][3]);
    else dft8<INV, PROD>(y[n1]);
  }
#pragma unroll
  for (int k2 = 0; k2 < M; ++k2) {
    dft3<INV>(y[0][k2], y[1][k2], y[2][k2]);
#pragma unroll
    for (int k1 = 0; k1 < 3; ++k1) v[(K1 * k1 + K2 * k2) % N] = y[k1][k2];
  }
}

template <int R, bool INV, bool PROD = false>
__device__ __forceinline__ void dft(float2* v) {
  if constexpr (R == 2) dft2<INV>(v[0], v[1]);
  else if constexpr (R == 3) dft3<INV>(v[0], v[1], v[2]);
  else if constexpr (R == 4) dft4<INV>(v[0], v[1], v[2], v[3]);
  else if constexpr (R == 6) dft3m<INV, 2, PROD>(v);
  else if constexpr (R == 8) dft8<INV, PROD>(v);
  else if constexpr (R == 12) dft3m<INV, 4, PROD>(v);
  else if constexpr (R == 24) dft3m<INV, 8, PROD>(v);
  else if constexpr (R == 16) dft16<INV, PROD>(v);
  else if constexpr (R == 32) dft32<INV, PROD>(v);
  else static_assert(R == 2, "unsupported radix");
}

// ------------------------------------------------------------------- plans
// A plan: length N, registers per thread E (a multiple of every radix), and
// the forward radix sequence.  Kernels pick a plan per length.
template <int N_, int E_, int NP_, int R0_, int R1_ = 0, int R2_ = 0, int R3_ = 0>
struct Plan {
  static constexpr int N = N_;
  static constexpr int E = E_;
  static constexpr int NP = NP_;
  static constexpr int T = N_ / E_;  // threads per pencil
  __host__ __device__ static constexpr int r(int p) { return p == 0 ? R0_ : p == 1 ? R1_ : p == 2 ? R2_ : R3_; }
};

// default plans
template <int N>
struct FftPlan;
template <> struct FftPlan<2> : Plan<2, 2, 1, 2> {};
template <> struct FftPlan<4> : Plan<4, 4, 1, 4> {};
template <> struct FftPlan<8> : Plan<8, 8, 1, 8> {};
template <> struct FftPlan<16> : Plan<16, 16, 1, 16> {};
template <> struct FftPlan<32> : Plan<32, 8, 2, 4, 8> {};
template <> struct FftPlan<64> : Plan<64, 8, 2, 8, 8> {};
template <> struct FftPlan<128> : Plan<128, 16, 2, 16, 8> {};
template <> struct FftPlan<256> : Plan<256, 16, 2, 16, 16> {};
// 512 = 32 x 16 (two passes, one exchange): measured on GB300 for the tau
// propagator of the 3 x 256x256x512 state, 473 us per launch against 546 for
// 8 x 8 x 8 and 610 for 16 x 32
template <> struct FftPlan<512> : Plan<512, 32, 2, 32, 16> {};
template <> struct FftPlan<1024> : Plan<1024, 16, 3, 16, 8, 8> {};
template <> struct FftPlan<2048> : Plan<2048, 16, 3, 16, 16, 8> {};
template <> struct FftPlan<4096> : Plan<4096, 16, 3, 16, 16, 16> {};
template <> struct FftPlan<6> : Plan<6, 6, 1, 6> {};
template <> struct FftPlan<12> : Plan<12, 12, 1, 12> {};
template <> struct FftPlan<24> : Plan<24, 12, 2, 12, 2> {};
template <> struct FftPlan<48> : Plan<48, 12, 2, 12, 4> {};
template <> struct FftPlan<96> : Plan<96, 12, 3, 12, 4, 2> {};
template <> struct FftPlan<192> : Plan<192, 24, 2, 24, 8> {};
template <> struct FftPlan<384> : Plan<384, 24, 3, 8, 12, 4> {};
template <> struct FftPlan<768> : Plan<768, 24, 3, 8, 24, 4> {};

// The lengths 3 2^k take radices 6, 12 and 24, which need one exchange where 3 x 4
// x 4 x 4 needs three: those four-pass plans were bound by shared memory (x-pass of
// 3 x 48x192x384: 82 % of its wavefronts, FP32 pipe 47 %).  Step of 2 x 96x96x192
// 72 -> 55 us, of 3 x 48x192x384 192 -> 147, of 2 x 192x192x768 1063 -> 875.
//
// Plans of y and tau where they differ from the rows'.  1024 points as 32 x 32
// (one exchange, 32 threads per pencil): tau-pass of 2 x 256x256x1024 833 -> 658
// us, step of 2 x 512x1024x1 25 -> 20 us; on rows it needs twice the rows for the
// same threads (2 x 1024x128x1: 11 -> 15 us).  96 as 24 x 4: y-passes of 2 x
// 96x96x192 14.4 + 14.6 -> 12.2 + 13.1 us, tau-pass of 3 x 96x384x96 46 -> 40 (rows
// 26.9 against 27.3).  384 as 24 x 16: y-passes of 3 x 96x384x96 63.5 -> 61.4,
// tau-pass of 3 x 48x192x384 53.5 -> 47.8 (rows of 2 x 384x48x192 46 against 55).
// 192 as 8 x 24 along y: y-passes of 2 x 192x192x768 305 -> 278 us (its tau-pass
// and rows are better as 24 x 8: 18.5 against 20.4 us on 2 x 96x96x192).
template <int N>
struct ColPlan : FftPlan<N> {};
template <>
struct ColPlan<96> : Plan<96, 24, 2, 24, 4> {};
template <>
struct ColPlan<192> : Plan<192, 24, 2, 8, 24> {};
template <>
struct ColPlan<384> : Plan<384, 48, 2, 24, 16> {};
template <>
struct ColPlan<1024> : Plan<1024, 32, 2, 32, 32> {};
template <int N>
struct TauPlan : ColPlan<N> {};
template <>
struct TauPlan<192> : FftPlan<192> {};

template <class PL, bool INV>
__host__ __device__ constexpr int fft_radix(int p) {
  return INV ? PL::r(PL::NP - 1 - p) : PL::r(p);
}
template <class PL, bool INV>
__host__ __device__ constexpr int fft_ns(int p) {
  int s = 1;
  for (int q = 0; q < p; ++q) s *= fft_radix<PL, INV>(q);
  return s;
}

// Centred number of butterfly j's first-pass inputs in a direction (input r of
// butterfly j is number centred_first(j) + r N/R0 of the pencil): the lowest
// digit of j belongs to the last pass, the highest to pass 1.
template <class PL, bool INV>
__host__ __device__ __forceinline__ int centred_first(int j) {
  int n = 0, w = 1;
#pragma unroll
  for (int p = PL::NP - 1; p >= 1; --p) {
    const int R = fft_radix<PL, INV>(p);
    const int d = j % R;
    n += w * (d >= (R + 1) / 2 ? d - R : d);
    j /= R;
    w *= R;
  }
  return n;
}
// Position of input r of butterfly j in the first pass of a direction; output r
// of butterfly j in the last pass of the other direction lies at the same place.
template <class PL, bool INV>
__device__ __forceinline__ int pos_first(int j, int r) {
  constexpr int S0 = PL::N / fft_radix<PL, INV>(0);
  const int n = centred_first<PL, INV>(j) + r * S0;
  return r == 0 && n < 0 ? n + PL::N : n;
}
template <class PL, bool INV>
__device__ __forceinline__ int pos_last(int j, int k) {
  return pos_first<PL, !INV>(j, k);
}

// ---------------------------------------------------------------- exchange
// Contiguous pencil (one row of x): one padding slot per 16 entries; rows start
// on 16-byte boundaries.
struct XchRow {
  static constexpr bool kSplit = false;
  float2* base;
  __device__ __forceinline__ void st(int pos, float2 v) const { base[pos + (pos >> 4)] = v; }
  __device__ __forceinline__ float2 ld(int pos) const { return base[pos + (pos >> 4)]; }
  __host__ __device__ static constexpr int pitch(int n) { return (n + n / 16 + 2) / 2 * 2; }
};
// Strided pencils: TX neighbouring columns, column index fastest.
template <int TX>
struct XchCol {
  static constexpr bool kSplit = false;
  float2* base;
  int tx;
  __device__ __forceinline__ void st(int pos, float2 v) const { base[pos * TX + tx] = v; }
  __device__ __forceinline__ float2 ld(int pos) const { return base[pos * TX + tx]; }
};
// Tiles of 8 columns: a row is 64 bytes, so the two rows of a half-warp's access
// must differ in parity.  The writes of pass 0 go to rows R0 j + r, whose parity
// is the same for every j: there row pos is kept at pos ^ ((pos / R0) & 1).
struct XchCol8 {
  static constexpr bool kSplit = false;
  float2* base;
  int tx;
  __device__ __forceinline__ void st(int pos, float2 v) const { base[pos * 8 + tx] = v; }
  __device__ __forceinline__ float2 ld(int pos) const { return base[pos * 8 + tx]; }
};
// The same layout for one real component at a time: the exchange runs in two
// rounds (real parts, then imaginary parts) through half the shared memory.
template <int TX>
struct XchColSplit {
  static constexpr bool kSplit = true;
  float* base;
  int tx;
  __device__ __forceinline__ void st(int pos, float v) const { base[pos * TX + tx] = v; }
  __device__ __forceinline__ float ld(int pos) const { return base[pos * TX + tx]; }
};

// Per-pass twiddle layout: forward pass P >= 1 with radix R and stride NS owns the
// R x NS block [r][m] of the shears (p, s) of the turn by -2 pi r' m' / (NS R), r'
// the centred r and m' the number of m with its digits centred (lowest digit:
// pass 0), so the threads of a warp, whose butterflies have consecutive m, read
// consecutive entries.  The inverse turns its outputs k of pass NP-1-P by the
// same entries [k][j / NS] with the signs turned.
template <class PL>
__host__ __device__ constexpr int tw_pass_off(int P) {
  int o = 0, ns = 1;
  for (int q = 0; q < P; ++q) {
    const int r = PL::r(q);
    if (q > 0) o += r * ns;
    ns *= r;
  }
  return o;
}
template <class PL>
__host__ __device__ constexpr int tw_table_size() {
  return PL::NP > 1 ? tw_pass_off<PL>(PL::NP) : 1;
}

// twiddle access from shared memory or, read-only, through L1
struct TwShared {
  static constexpr bool kProduct = false;
  const float2* p;
  __device__ __forceinline__ float2 operator()(int i) const { return p[i]; }
};
struct TwGlobal {
  static constexpr bool kProduct = false;
  const float2* p;
  __device__ __forceinline__ float2 operator()(int i) const { return __ldg(p + i); }
};
// the same turns as products with hi + lo floats (codelets too), for transforms that
// nothing undoes: the spectrum, single transforms, the spectral-phase gradient
struct TwProduct {
  static constexpr bool kProduct = true;
  const float4* p;
  __device__ __forceinline__ float4 operator()(int i) const { return __ldg(p + i); }
};
struct TwProductShared {
  static constexpr bool kProduct = true;
  const float4* p;
  __device__ __forceinline__ float4 operator()(int i) const { return p[i]; }
};

// Barrier used around shared-memory exchanges: the whole CTA, or only the
// warp when every pencil's threads lie inside one warp.
struct SyncBlock {
  __device__ __forceinline__ static void sync() { __syncthreads(); }
};
struct SyncWarp {
  __device__ __forceinline__ static void sync() { __syncwarp(); }
};
// the T threads of one row inside a warp (T a power of two)
template <int T>
struct SyncRow {
  __device__ __forceinline__ static void sync() {
    if constexpr (T == 32) __syncwarp();
    else if constexpr (T > 1) __syncwarp(((1u << T) - 1u) << (threadIdx.x & 31 & ~(T - 1)));
  }
};
// an exchange that only active threads take part in (all keep the barriers)
template <class X>
struct XchGuard {
  static constexpr bool kSplit = X::kSplit;
  X x;
  bool act;
  __device__ __forceinline__ void st(int pos, float2 v) const {
    if (act) x.st(pos, v);
  }
  __device__ __forceinline__ float2 ld(int pos) const { return act ? x.ld(pos) : make_float2(0.f, 0.f); }
};

// Passes P..NP-1 of a length-N transform on the registers v (see header).
// Every thread that shares a barrier of type S must call this.
template <class PL, bool INV, int P, class X, class S = SyncBlock, class TW = TwShared>
__device__ __forceinline__ void fft_run(float2 (&v)[PL::E], int t, const X& x, const TW& tw) {
  constexpr int N = PL::N;
  constexpr int NP = PL::NP;
  constexpr int E = PL::E;
  constexpr int T = PL::T;
  constexpr int R = fft_radix<PL, INV>(P);
  constexpr int NS = fft_ns<PL, INV>(P);
  constexpr int B = E / R;
  static_assert(E % R == 0, "E must be a multiple of every radix");
  if constexpr (!INV && P > 0) {
#pragma unroll
    for (int b = 0; b < B; ++b) {
      const int m = (t + b * T) % NS;
#pragma unroll
      for (int r = 1; r < R; ++r) {
        v[b * R + r] = turn(v[b * R + r], tw(tw_pass_off<PL>(P) + r * NS + m));
      }
    }
  }
#pragma unroll
  for (int b = 0; b < B; ++b) dft<R, INV, TW::kProduct>(&v[b * R]);
  if constexpr (INV && P + 1 < NP) {
    constexpr int REST = N / (NS * R);
#pragma unroll
    for (int b = 0; b < B; ++b) {
      const int q = (t + b * T) / NS;
#pragma unroll
      for (int k = 1; k < R; ++k) {
        v[b * R + k] = turn_back(v[b * R + k], tw(tw_pass_off<PL>(NP - 1 - P) + k * REST + q));
      }
    }
  }
  if constexpr (P + 1 < NP) {
    constexpr int R2 = fft_radix<PL, INV>(P + 1);
    constexpr int B2 = E / R2;
    if constexpr (X::kSplit) {
      // real parts, then imaginary parts, through the same buffer
      float re[E];
#pragma unroll
      for (int c = 0; c < 2; ++c) {
        S::sync();  // earlier readers of the exchange buffer are done
#pragma unroll
        for (int b = 0; b < B; ++b) {
          const int j = t + b * T;
          const int m = j % NS;
          const int d = (j / NS) * NS * R + m;
#pragma unroll
          for (int r = 0; r < R; ++r) x.st(d + r * NS, c == 0 ? v[b * R + r].x : v[b * R + r].y);
        }
        S::sync();
#pragma unroll
        for (int b = 0; b < B2; ++b) {
          const int j = t + b * T;
#pragma unroll
          for (int r = 0; r < R2; ++r) {
            const float u = x.ld(j + r * (N / R2));
            if (c == 0)
              re[b * R2 + r] = u;
            else
              v[b * R2 + r] = make_float2(re[b * R2 + r], u);
          }
        }
      }
    } else {
      S::sync();  // earlier readers of the exchange buffer are done
      // exchange of pass 0 in 8-column tiles: rows in turned parity (XchCol8)
      constexpr bool kTurn = std::is_same<X, XchCol8>::value && P == 0 && R % 2 == 0;
      constexpr int K = N / R2;
#pragma unroll
      for (int b = 0; b < B; ++b) {
        const int j = t + b * T;
        const int m = j % NS;
        const int d = (j / NS) * NS * R + m;
#pragma unroll
        for (int r = 0; r < R; ++r) {
          if constexpr (kTurn) x.st(d + r + (r % 2 ? -(j & 1) : (j & 1)), v[b * R + r]);
          else x.st(d + r * NS, v[b * R + r]);
        }
      }
      S::sync();
#pragma unroll
      for (int b = 0; b < B2; ++b) {
        const int j = t + b * T;
#pragma unroll
        for (int r = 0; r < R2; ++r) {
          if constexpr (kTurn && K % R == 0 && K <= R) v[b * R2 + r] = x.ld(((r * (K / R)) % 2 ? (j ^ 1) : j) + r * K);
          else if constexpr (kTurn) v[b * R2 + r] = x.ld((j + r * K) ^ (((j + r * K) / R) & 1));
          else v[b * R2 + r] = x.ld(j + r * K);
        }
      }
    }
    fft_run<PL, INV, P + 1, X, S, TW>(v, t, x, tw);
  }
}

}  // namespace brahms
