// Reverse-mode derivatives of the pair arithmetic (hweno_pair.cuh), for the adjoint of a 2D Euler stage.
//
// Where the corrections of a face or a cell may be taken from pairs, the adjoint splits in the same
// way: the transposes of the linear scheme and of the fluxes in FP64, the transpose of the correction
// in pairs.  The correction's derivatives are of the order of max(t_l) as well, so their pairs (2^-42)
// add less than the rounding of the linear part.  Adjoints can have any size: a thread divides its
// seeds by the power of two of the largest on their way into pairs and multiplies on the way out.
#pragma once
#include "hweno_adjoint.cuh"

namespace hw {

// p_from and d_from with the power of two 2^(sh >> 20) taken out and put back
__device__ __forceinline__ P2 p_from_scaled(double x, int sh) {
  const int H = __double2hiint(x), L = __double2loint(x);
  const unsigned int u = (unsigned int)((H & 0x7fffffff) - 0x38000000 - sh);
  unsigned int b = __funnelshift_l((unsigned int)L, u, 3);
  if (u >= 0x0ff00000u) b = (int)u < 0 ? 0u : 0x7fc00000u;
  b |= (unsigned int)H & 0x80000000u;
  const float unit = __fmul_rn(__uint_as_float(b & 0xff800000u), 0x1p-52f);
  return P2{__uint_as_float(b), __fmul_rn(__uint2float_rn((unsigned int)L & 0x1fffffffu), unit)};
}
__device__ __forceinline__ double d_from_scaled(float x, int sh) {
  const unsigned int b = __float_as_uint(x), m = b & 0x7fffffffu;
  const unsigned int hi = m < 0x00800000u ? 0u : (m >> 3) + 0x38000000u + (unsigned int)sh;
  return __hiloint2double((int)(hi | (b & 0x80000000u)), m < 0x00800000u ? 0 : (int)(b << 29));
}
__device__ __forceinline__ double d_from_scaled(P2 x, int sh, const FU& f) {
  return f.add(d_from_scaled(x.h, sh), d_from_scaled(x.l, sh));
}
// The exponent (in place, of the largest of n numbers, less the bias) as a scale for the two above.
// Returns false where the seeds are not finite or so small that the scaled results would leave the
// normal range.
__device__ __forceinline__ bool seed_scale(unsigned int big, int& sh) {
  sh = (int)(big & 0x7ff00000u) - 0x3ff00000;
  if (big == 0u) sh = 0;
  return sh < (900 << 20) && sh > -(800 << 20);
}
__device__ __forceinline__ unsigned int seed_bits(double x) { return (unsigned int)__double2hiint(x) & 0x7fffffffu; }

// x += a b
template <class F>
__device__ __forceinline__ void p_acc(P<F>& x, P<F> a, P<F> b) {
  x = p_add(x, p_mul(a, b));
}
template <class F>
__device__ __forceinline__ void p_dec(P<F>& x, P<F> a, P<F> b) {
  x = p_sub(x, p_mul(a, b));
}

// The kinds of correction: h times the modified derivative; the two sides of a face (lane 0 the right
// face of its stencil, lane 1 the left face)
enum { CORR_LIMITED, CORR_FACE };

// Backward of p_stencil and the correction of a kind: nb the adjoint of the correction; the adjoints
// of d01, d12, y0, y2 are written, the correction itself is returned, and ok is cleared where it may
// not be taken from pairs.  The tie |X| = |Y| takes half of
// each, as d|x| = 0 at 0 does.  SMALL32: the small term of the denominator, tau (G Q + e0 (e1 + e2)), in FP32.  The
// derivatives, beside the linear part's of order one, are right to 2^-55 with 1/gamma_1 = 200, and 2^-53 with
// 40, 2^-49 with 4; in pairs (the limiter, with its 1/d_1 of 20, and faces below kSmall32) to 2^-53 or better
// whatever the linear weights.
constexpr float kSmall32 = 100.0f;
template <int KIND, bool SMALL32>
__device__ __forceinline__ P4 p_correction_vjp(P4 d01, P4 d12, P4 y0, P4 y2, P4 h, P4 eps, P4 inv_l, P4 G, P4 nb,
                                               P4& d01b, P4& d12b, P4& y0b, P4& y2b, bool& ok) {
  // forward, as p_stencil and p_correction
  const P4 e1 = p_add(p_sqr(d01), eps), e2 = p_add(p_sqr(d12), eps);
  const P4 du = p_renorm(p_add(d01, d12)), d2 = p_renorm(p_sub(d12, d01));
  const P4 hdv = p_mul(h, p_sub(y0, y2));
  const P4 w = p_renorm(p_sub(p_mul(h, p_add(y0, y2)), du));
  const P4 z = p_renorm(p_add(hdv, p_scale(d2, 2.0f)));
  constexpr double k1_ = 9.0 / 256.0 + 781.0 / 320.0, k3_ = (13.0 / 3.0) * (67.0 / 520.0);
  constexpr double k2_ = (13.0 / 3.0) * (67.0 / 520.0) * (67.0 / 520.0) + 1421461.0 / 36400.0;
  const P4 k1 = p_const<F2>(k1_), k2 = p_const<F2>(k2_), k3 = p_const<F2>(k3_), k56 = p_const<F2>(5.0 / 6.0);
  const P4 k1w = p_mul(k1, w), k56d = p_mul(k56, d2), k2z = p_mul(k2, z);
  const P4 r1 = p_sub(k1w, p_mulf(du, 0.1875f)), r2 = p_add(k56d, p_mul(k3, z));
  const P4 X = p_renorm(p_add(p_add(p_mul(w, r1), p_mul(d2, r2)), p_mul(k2z, z)));
  const P4 Y = p_renorm(p_scale(p_mul(du, d2), 0.5f));
  const P4 tau = p_sqr(p_maxabs(X, Y));
  const P4 A1 = p_add(X, Y), A2 = p_sub(X, Y), e0 = p_add(e1, A1);
  const P4 S1 = p_mul(A1, e2), S2 = p_mul(A2, e1), Q = p_mul(e1, e2), PP = p_mul(e0, Q);
  const P4 e12 = p_add(e1, e2);
  P4 GQR;
  if (!SMALL32)
    GQR = p_add(p_mul(Q, G), p_mul(e0, e12));
  else
    GQR.h = f_fma(G.h, Q.h, f_mul(e0.h, e12.h));
  ok = p_smooth(tau.h, e0.h, e1.h, e2.h, PP.h) && ok;
  P4 q1, q2;
  if (KIND == CORR_LIMITED) {
    const P4 c = p_scale(w, 0.25f), d = p_scale(d2, 0.5f);
    q1 = p_sub(c, d);
    q2 = p_add(c, d);
  } else {
    const P4 a = p_sub(p_scale(d2, 0.03125f), p_mulf(hdv, 0.046875f)), a2 = p_sub(a, p_scale(d2, 0.5f));
    const P4 b = p_scalev(p_mulf(w, 0.09375f), f_pack(1.0f, -1.0f));
    q1 = p_add(p_mix(a2, a), b);
    q2 = p_add(p_mix(a, a2), b);
  }
  P4 den = p_mul(inv_l, PP);
  if (!SMALL32)
    den = p_add(den, p_mul(tau, GQR));
  else
    den.l = f_fma(tau.h, GQR.h, den.l);
  den = p_renorm(den);
  const P4 quo = p_div(p_add(p_mul(S1, q1), p_mul(S2, q2)), den);
  const P4 n = p_mul(tau, quo);
  // backward: n = tau N / den, N = S1 q1 + S2 q2, den = P / l + tau (G Q + R)
  const P4 Nb = p_mul(nb, p_div(tau, den)), denb = p_neg(p_mul(Nb, quo));
  P4 taub = p_mul(nb, quo);
  const P4 q1b = p_mul(Nb, S1), q2b = p_mul(Nb, S2), S1b = p_mul(Nb, q1), S2b = p_mul(Nb, q2);
  const P4 Pb = p_mul(inv_l, denb);
  P4 Qb = p_mul(Pb, e0), e0b = p_mul(Pb, Q), e1b, e2b;
  if (!SMALL32) {
    const P4 Rb = p_mul(denb, tau), t = p_mul(Rb, e0);
    p_acc(taub, denb, GQR);
    p_acc(Qb, Rb, G);
    p_acc(e0b, Rb, e12);
    e1b = p_add(p_add(p_mul(Qb, e2), p_mul(S2b, A2)), t);
    e2b = p_add(p_add(p_mul(Qb, e1), p_mul(S1b, A1)), t);
  } else {
    const F2 Rb = f_mul(denb.h, tau.h);
    taub.l = f_fma(denb.h, GQR.h, taub.l);
    Qb.l = f_fma(Rb, G.h, Qb.l);
    e0b.l = f_fma(Rb, e12.h, e0b.l);
    e1b = p_add(p_mul(Qb, e2), p_mul(S2b, A2));
    e2b = p_add(p_mul(Qb, e1), p_mul(S1b, A1));
    e1b.l = f_fma(Rb, e0.h, e1b.l);
    e2b.l = f_fma(Rb, e0.h, e2b.l);
  }
  e1b = p_add(e1b, e0b);
  const P4 A1b = p_add(p_mul(S1b, e2), e0b), A2b = p_mul(S2b, e1);
  P4 Xb = p_add(A1b, A2b), Yb = p_sub(A1b, A2b);
  {
    auto part = [](float xh, float xl, float yh, float yl) {
      const float d = f_add(f_sub(fabsf(xh), fabsf(yh)), f_sub(xh < 0.0f ? -xl : xl, yh < 0.0f ? -yl : yl));
      return d > 0.0f ? 2.0f : (d < 0.0f ? 0.0f : 1.0f);
    };
    const float w0 = part(f_lane0(X.h), f_lane0(X.l), f_lane0(Y.h), f_lane0(Y.l));
    const float w1 = part(f_lane1(X.h), f_lane1(X.l), f_lane1(Y.h), f_lane1(Y.l));
    p_acc(Xb, taub, p_scalev(X, f_pack(w0, w1)));
    p_acc(Yb, taub, p_scalev(Y, f_pack(2.0f - w0, 2.0f - w1)));
  }
  P4 wb = p_mul(Xb, p_add(r1, k1w));
  P4 dub = p_sub(p_scale(p_mul(Yb, d2), 0.5f), p_mulf(p_mul(Xb, w), 0.1875f));
  P4 d2b = p_add(p_mul(Xb, p_add(r2, k56d)), p_scale(p_mul(Yb, du), 0.5f));
  const P4 zb = p_mul(Xb, p_add(p_mul(k3, d2), p_scale(k2z, 2.0f)));
  P4 hdvb = zb;
  d2b = p_add(d2b, p_scale(zb, 2.0f));
  const P4 qs = p_add(q1b, q2b);
  if (KIND == CORR_LIMITED) {
    wb = p_add(wb, p_scale(qs, 0.25f));
    d2b = p_add(d2b, p_scale(p_sub(q2b, q1b), 0.5f));
  } else {
    wb = p_add(wb, p_scalev(p_mulf(qs, 0.09375f), f_pack(1.0f, -1.0f)));
    d2b = p_add(d2b, p_sub(p_scale(qs, 0.03125f), p_scale(p_mix(q1b, q2b), 0.5f)));
    hdvb = p_sub(hdvb, p_mulf(qs, 0.046875f));
  }
  const P4 svb = p_mul(h, wb), dvb = p_mul(h, hdvb);
  dub = p_sub(dub, wb);
  y0b = p_add(svb, dvb);
  y2b = p_sub(svb, dvb);
  d01b = p_add(p_sub(dub, d2b), p_mul(p_scale(d01, 2.0f), e1b));
  d12b = p_add(p_add(dub, d2b), p_mul(p_scale(d12, 2.0f), e2b));
  return n;
}

// Adjoints of the variables of an EigP<4>
template <class F>
struct EigPBar {
  P<F> u, v, H, c, hb1, hb2, hic, uc, hq2;
  __device__ __forceinline__ void zero() { u = v = H = c = hb1 = hb2 = hic = uc = hq2 = p_const<F>(0.0); }
};
// w = transposed right eigenvectors times qb
template <class F>
__device__ __forceinline__ void p_back_t(const EigP<4, F>& e, const P<F>* qb, P<F>* w) {
  const P<F> q0b = p_add(qb[0], p_add(p_mul(e.v, qb[2]), p_mul(e.u, qb[1])));
  const P<F> sg = p_add(p_mul(e.H, qb[3]), q0b), dl = p_add(p_mul(e.uc, qb[3]), p_mul(e.c, qb[1]));
  w[0] = p_sub(sg, dl);
  w[1] = p_add(p_mul(e.hq2, qb[3]), q0b);
  w[2] = p_add(p_mul(e.v, qb[3]), qb[2]);
  w[3] = p_add(sg, dl);
}
// the adjoints of the basis of q = R w
template <class F>
__device__ __forceinline__ void p_back_eig(const P<F>* w, const P<F>* qb, EigPBar<F>& b) {
  const P<F> sg = p_add(w[0], w[3]), dl = p_sub(w[3], w[0]), q0 = p_add(sg, w[1]);
  p_acc(b.H, qb[3], sg);
  p_acc(b.hq2, qb[3], w[1]);
  p_acc(b.v, qb[3], w[2]);
  p_acc(b.uc, qb[3], dl);
  p_acc(b.v, qb[2], q0);
  p_acc(b.u, qb[1], q0);
  p_acc(b.c, qb[1], dl);
}
// w = L q: the adjoint of q, and those of the basis
template <class F>
__device__ __forceinline__ void p_project_vjp(const EigP<4, F>& e, const P<F>* q, const P<F>* wb, P<F>* qb,
                                              EigPBar<F>& b) {
  const P<F> k = p_add(p_sub(p_mul(e.u, q[1]), q[3]), p_mul(e.v, q[2])), m = p_sub(p_mul(e.u, q[0]), q[1]);
  const P<F> thb = p_sub(p_add(wb[0], wb[3]), p_scale(wb[1], 2.0f)), shb = p_sub(wb[0], wb[3]);
  const P<F> kb = p_neg(p_mul(thb, e.hb1)), mb = p_mul(shb, e.hic);
  p_acc(b.hb2, thb, q[0]);
  p_dec(b.hb1, thb, k);
  p_acc(b.hic, shb, m);
  p_acc(b.u, mb, q[0]);
  p_acc(b.u, kb, q[1]);
  p_acc(b.v, kb, q[2]);
  p_dec(b.v, wb[2], q[0]);
  const P<F> w2 = wb[2];
  qb[0] = p_add(p_sub(wb[1], p_mul(e.v, w2)), p_add(p_mul(thb, e.hb2), p_mul(mb, e.u)));
  qb[1] = p_sub(p_mul(kb, e.u), mb);
  qb[2] = p_add(w2, p_mul(kb, e.v));
  qb[3] = p_neg(kb);
}
// to the velocities, the enthalpy and c^2 that the basis was set up from
template <class F>
__device__ __forceinline__ void p_setup_vjp(const EigP<4, F>& e, P<F> gm1, EigPBar<F>& b, P<F>& c2b) {
  const P<F> ic = p_scale(e.hic, 2.0f);
  p_acc(b.hb1, b.hb2, e.hq2);
  p_acc(b.hq2, b.hb2, e.hb1);
  p_acc(b.u, b.hq2, e.u);
  p_acc(b.v, b.hq2, e.v);
  p_acc(b.u, b.uc, e.c);
  p_acc(b.c, b.uc, e.u);
  // c = sqrt(c2), ic = 1/c, hic = ic/2, hb1 = gm1 ic^2 / 2
  const P<F> icb = p_add(p_mul(p_mul(gm1, ic), b.hb1), p_scale(b.hic, 0.5f));
  c2b = p_mul(p_scale(ic, 0.5f), p_sub(b.c, p_mul(icb, p_sqr(ic))));
}
// Given the adjoints of 1/rho, u, v, p of a state U (normal frame), those of U are added
template <class F>
__device__ __forceinline__ void p_prim_vjp(const P<F>* U, P<F> ir, P<F> u, P<F> v, P<F> gm1, P<F> irb, P<F> ub,
                                           P<F> vb, P<F> pb, P<F>* Ub) {
  const P<F> gp = p_mul(gm1, pb), keb = p_scale(gp, -0.5f);
  Ub[3] = p_add(Ub[3], gp);
  p_acc(ub, keb, U[1]);
  p_acc(vb, keb, U[2]);
  Ub[1] = p_add(Ub[1], p_add(p_mul(keb, u), p_mul(ub, ir)));
  Ub[2] = p_add(Ub[2], p_add(p_mul(keb, v), p_mul(vb, ir)));
  p_acc(irb, ub, U[1]);
  p_acc(irb, vb, U[2]);
  p_dec(Ub[0], irb, p_sqr(ir));
}
// sums over the two lanes
__device__ __forceinline__ P2 p_sum(P4 x) { return p_add(p_lane0(x), p_lane1(x)); }

}  // namespace hw
