// Reverse mode of the RK4 half step (Sec. 3.1) at two grid points, the nonlinear
// part of the reverse x-pass.
//
// Complex gradients follow G_z = dJ/dRe z + i dJ/dIm z.  For y = f(x):
//   G_x = sum_y [ conj(G_y) dy/dconj(x) + G_y conj(dy/dx) ].
// The stages are recomputed in registers from the state at the start of the half
// step, in the form of rk4 (kernels.cuh): field 0 as u = e^{i Phi} A_0 of the
// stage, m the driving term of field 0 and n the slopes of the others, so that no
// product of a stage carries a phase or a coupling.  The sensitivity to a stage's
// phase is
//   dJ/dPhi = sum_f Re( conj(G_k_f) dk_f/dPhi ),  dk_0/dPhi = -i k_0,
//   dk_f/dPhi = +i k_f (f >= 1),
// which is Im(conj(G_m) m) - sum_f Im(conj(G_n_f) n_f); the second sum equals
// Im(conj(G_u) u), G_u the gradient that the stage's slopes give u, and the first
// Im(conj(X) t) of the part X of a field's gradient that comes from m (half of it
// for two fields), so that neither m nor n is kept.
#pragma once

#include "kernels.cuh"

namespace brahms {

// Im(conj(a) b)
__device__ __forceinline__ float im_cb(float2 a, float2 b) { return a.x * b.y - a.y * b.x; }
// acc + Im(conj(a) b)
__device__ __forceinline__ float2 add_im_cb(float2 acc, Pair a, Pair b) {
  return __ffma2_rn(a.re, b.im, __ffma2_rn(neg(a.im), b.re, acc));
}
// c g and -i c g for a real c; a - i c g
__device__ __forceinline__ Pair pair_scale(float c, Pair g) { return {__fmul2_rn(dup(c), g.re), __fmul2_rn(dup(c), g.im)}; }
__device__ __forceinline__ Pair pair_niscale(float c, Pair g) {
  return {__fmul2_rn(dup(c), g.im), __fmul2_rn(dup(-c), g.re)};
}
__device__ __forceinline__ Pair pair_niaxpy(Pair a, float c, Pair g) {
  return {__ffma2_rn(dup(c), g.im, a.re), __ffma2_rn(dup(-c), g.re, a.im)};
}
// acc + i a conj(b)
__device__ __forceinline__ Pair pair_add_imulc(Pair acc, Pair a, Pair b) {
  return {__ffma2_rn(a.re, b.im, __ffma2_rn(neg(a.im), b.re, acc.re)),
          __ffma2_rn(a.re, b.re, __ffma2_rn(a.im, b.im, acc.im))};
}
// -i a b, and acc - i a b
__device__ __forceinline__ Pair pair_nimul(Pair a, Pair b) {
  return {__ffma2_rn(a.re, b.im, __fmul2_rn(a.im, b.re)), __ffma2_rn(a.im, b.im, neg(__fmul2_rn(a.re, b.re)))};
}
__device__ __forceinline__ Pair pair_add_nimul(Pair acc, Pair a, Pair b) {
  return {__ffma2_rn(a.re, b.im, __ffma2_rn(a.im, b.re, acc.re)),
          __ffma2_rn(a.im, b.im, __ffma2_rn(neg(a.re), b.re, acc.im))};
}

// Reverse of one stage's products at (u, t): from the gradients gm of the driving
// term (twice it for two fields) and gn of the slopes to those of u and t; s gains
// the sensitivity to the stage's phase.
template <int F>
__device__ __forceinline__ void nl_vjp(Pair u, const Pair* t, Pair gm, const Pair* gn, Pair& gu, Pair* gt, float2& s) {
  const Pair x = pair_mulc(gm, t[F - 2]);  // what field 1's driving term takes from gm
  if constexpr (F == 3) {
    gu = pair_add_nimul(pair_nimul(t[1], gn[0]), t[0], gn[1]);
    s = add_im_cb(s, x, t[0]);
    gt[0] = pair_add_imulc(x, u, gn[1]);
    gt[1] = pair_add_imulc(pair_mulc(gm, t[0]), u, gn[0]);
  } else {
    gu = pair_nimul(t[0], gn[0]);
    s = __ffma2_rn(dup(0.5f), add_im_cb(make_float2(0.f, 0.f), x, t[0]), s);
    gt[0] = pair_add_imulc(x, u, gn[0]);
  }
  s = add_im_cb(s, {neg(gu.re), neg(gu.im)}, u);
}

// One RK4 half step in reverse at two points: x is the forward state at the start
// of the half step, c, kh and kh2 as in rk4; g enters as the gradient with respect
// to the end state and leaves as the gradient with respect to x.  s[0], s[1], s[2]
// gain the sensitivities to the stage phases at the start, the midpoint (both middle
// stages) and the end.  The gradients of the stages' u are kept in the stage's own
// frame; the stage factors take them to x, v from one stage to the next.
template <int F, bool MAP>
__device__ __forceinline__ void rk4_vjp(const Pair (&x)[F], Pair (&g)[F], const Stages<MAP>& c, const float* kh,
                                        const float* kh2, float2* s) {
  constexpr int G = F - 1;
  const Pair v = c.v;
  const Pair* t1 = x + 1;
  Pair t2[G], t3[G], t4[G], n[G];
  const Pair u1 = pair_mul(c.e0, x[0]);
  const Pair w = MAP ? pair_mul(v, u1) : pair_mul(c.em, x[0]);
  nl_slopes<F>(u1, t1, n);
#pragma unroll
  for (int f = 0; f < G; ++f) t2[f] = pair_axpy(t1[f], kh2[f + 1], n[f]);
  const Pair u2 = pair_iaxpy(w, kh2[0], pair_mul(v, nl_drive<F>(t1)));
  nl_slopes<F>(u2, t2, n);
#pragma unroll
  for (int f = 0; f < G; ++f) t3[f] = pair_axpy(t1[f], kh2[f + 1], n[f]);
  const Pair u3 = pair_iaxpy(w, kh2[0], nl_drive<F>(t2));
  nl_slopes<F>(u3, t3, n);
#pragma unroll
  for (int f = 0; f < G; ++f) t4[f] = pair_axpy(t1[f], kh[f + 1], n[f]);
  const Pair u4 = MAP ? pair_mul(v, pair_iaxpy(w, kh[0], nl_drive<F>(t3)))
                      : pair_iaxpy(pair_mul(c.e1, x[0]), kh[0], pair_mul(v, nl_drive<F>(t3)));

  // direct shares of the end state: 1/6 of its gradient to stages 1 and 4, 1/3 to 2
  // and 3; the driving term's in the frame of the stage's u
  const float kd = F == 2 ? 2.f * kh[0] : kh[0], kd2 = F == 2 ? kh[0] : kh2[0];
  const Pair p1 = pair_mul(c.e0, g[0]);
  const Pair p2 = MAP ? pair_mul(v, p1) : pair_mul(c.em, g[0]);
  const Pair p4 = MAP ? pair_mul(v, p2) : pair_mul(c.e1, g[0]);
  const Pair d23 = pair_niscale(kd * (1.f / 3.f), p2);
  Pair dn[G], gn[G], gt[G], gu;
#pragma unroll
  for (int f = 0; f < G; ++f) {
    dn[f] = pair_scale(kh[f + 1] * (1.f / 3.f), g[f + 1]);
    gn[f] = pair_scale(0.5f, dn[f]);
  }
  // stage 4: u4 = e1 A_0 + i kh v m3, t4 = A + kh n3
  nl_vjp<F>(u4, t4, pair_niscale(kd * (1.f / 6.f), p4), gn, gu, gt, s[2]);
  Pair gw = pair_mulc(gu, v);  // MAP: the gradient of w
  if constexpr (!MAP) g[0] = pair_add(g[0], pair_mulc(gu, c.e1));
#pragma unroll
  for (int f = 0; f < G; ++f) {
    g[f + 1] = pair_add(g[f + 1], gt[f]);
    gn[f] = pair_axpy(dn[f], kh[f + 1], gt[f]);
  }
  // stage 3: u3 = w + i kh/2 m2, t3 = A + kh/2 n2
  nl_vjp<F>(u3, t3, pair_niaxpy(d23, kd, gw), gn, gu, gt, s[1]);
  gw = MAP ? pair_add(gw, gu) : gu;
#pragma unroll
  for (int f = 0; f < G; ++f) {
    g[f + 1] = pair_add(g[f + 1], gt[f]);
    gn[f] = pair_axpy(dn[f], kh2[f + 1], gt[f]);
  }
  // stage 2: u2 = w + i kh/2 v m1, t2 = A + kh/2 n1
  nl_vjp<F>(u2, t2, pair_niaxpy(d23, kd2, gu), gn, gu, gt, s[1]);
  const Pair r = pair_mulc(gu, v);
  if constexpr (!MAP) g[0] = pair_add(g[0], pair_mulc(pair_add(gw, gu), c.em));
#pragma unroll
  for (int f = 0; f < G; ++f) {
    g[f + 1] = pair_add(g[f + 1], gt[f]);
    gn[f] = pair_axpy(pair_scale(0.5f, dn[f]), kh2[f + 1], gt[f]);
  }
  // stage 1: u1 = e0 A_0
  nl_vjp<F>(u1, t1, pair_niaxpy(pair_niscale(kd * (1.f / 6.f), p1), kd2, r), gn, gu, gt, s[0]);
#pragma unroll
  for (int f = 0; f < G; ++f) g[f + 1] = pair_add(g[f + 1], gt[f]);
  if constexpr (MAP) gu = pair_add(pair_add(gu, r), pair_mulc(gw, v));
  g[0] = pair_add(g[0], pair_mulc(gu, c.e0));
}

}  // namespace brahms
