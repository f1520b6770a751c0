// The nonlinear part of the HWENO interpolation in pairs of FP32 values, for the FP64 kernels.
//
// What bounds the stage kernels is the FP64 pipe: one warp instruction takes 68 cycles of its
// scheduler (a DFMA, a DADD and a conversion between FP64 and FP32 alike, however many lanes are
// active), in which 50 to 60 FP32 instructions issue beside it.  The interpolation is therefore
// split into its linear part and a correction,
//   sum_l omega_l p_l = p_0 + gamma_1 [ (W1 - W0)(p_1 - p_0) + (W2 - W0)(p_2 - p_0) ] / W,
//   W_l = 1 + t_l, t_l = tau / (beta_l + eps), W = gamma_0 W0 + gamma_1 (W1 + W2),
// exactly (p_0 is the linear-weights value, and the three candidates' deviations from it cancel in
// the linear weights).  p_0 is linear in the stencil, so it needs no characteristic fields: it is
// formed in conserved variables in FP64, as all of the linear scheme is.  The correction is at most
// max(t_l) times a second difference, and where max(t_l) <= kPairMaxT = 2^-14 (that is where the
// second difference of a characteristic field is below about 6e-3: smooth flow, at any distance
// from a captured front) it needs only 40 bits to be right to the last bit of the sum: it is
// evaluated, with its characteristic projections, on values hi + lo of two FP32 numbers (48 bits).
// Everywhere else (and whenever a value leaves the FP32 range, is not finite or is not physical)
// the FP64 code evaluates the weights as written.  Error: the pair arithmetic below is accurate to
// about 2^-42 of the stencil's differences, the correction is below 2^-14 of them, so its error
// stays under 2^-54 of the differences, which are what the FP64 evaluation rounds at 2^-53.
//
// The indicators enter through their differences.  With du = u_{i+1} - u_{i-1},
// d2 = u_{i+1} - 2 u_i + u_{i-1}, w = h (v_{i-1} + v_{i+1}) - du, z = h (v_{i-1} - v_{i+1}) + 2 d2
// (of third and fourth order on smooth data), Eq. (GHYZ) is
//   beta0 = (du/2 - 3 w/16)^2 + 781/320 w^2 + 13/3 (d2/2 + 67 z/520)^2 + 1421461/36400 z^2,
//   beta1 = (du - d2)^2 / 4,  beta2 = (du + d2)^2 / 4,
// so that beta0 - beta1 = X + Y and beta0 - beta2 = X - Y with Y = du d2 / 2 and
//   X = w (k1 w - 3 du/16) + d2 (5 d2/6 + k3 z) + k2 z^2,
// free of the cancellation of the indicators themselves, and tau of Eq. (nonlinear),
// (|X + Y| + |X - Y|)^2 / 4, is max(|X|, |Y|)^2.
#pragma once
#include "hweno_math.cuh"

namespace hw {

// Two FP32 lanes in one register pair: fma.rn.f32x2 and its kin do both in one instruction.  The FP32
// work beside the FP64 pipe is limited by its latency (three warps per scheduler), so it is done for
// two stencils at a time: the two sides of a face, the two directions of a cell.
struct F2 {
  unsigned long long v;
};
__device__ __forceinline__ F2 f_pack(float x, float y) {
  F2 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r.v) : "f"(x), "f"(y));
  return r;
}
__device__ __forceinline__ float f_lane0(F2 a) { return __uint_as_float((unsigned int)a.v); }
__device__ __forceinline__ float f_lane1(F2 a) { return __uint_as_float((unsigned int)(a.v >> 32)); }
__device__ __forceinline__ F2 f_add(F2 a, F2 b) {
  F2 r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
  return r;
}
__device__ __forceinline__ F2 f_mul(F2 a, F2 b) {
  F2 r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
  return r;
}
__device__ __forceinline__ F2 f_fma(F2 a, F2 b, F2 c) {
  F2 r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r.v) : "l"(a.v), "l"(b.v), "l"(c.v));
  return r;
}
__device__ __forceinline__ F2 f_sub(F2 a, F2 b) { return f_fma(b, f_pack(-1.0f, -1.0f), a); }
__device__ __forceinline__ F2 f_neg(F2 a) { return f_mul(a, f_pack(-1.0f, -1.0f)); }
__device__ __forceinline__ float f_add(float a, float b) { return __fadd_rn(a, b); }
__device__ __forceinline__ float f_sub(float a, float b) { return __fsub_rn(a, b); }
__device__ __forceinline__ float f_mul(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ float f_fma(float a, float b, float c) { return __fmaf_rn(a, b, c); }
__device__ __forceinline__ float f_neg(float a) { return -a; }
// a constant in every lane
template <class F>
__device__ __forceinline__ F f_all(float x);
template <>
__device__ __forceinline__ float f_all<float>(float x) {
  return x;
}
template <>
__device__ __forceinline__ F2 f_all<F2>(float x) {
  return f_pack(x, x);
}
__device__ __forceinline__ float f_rcp(float x) {
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}
__device__ __forceinline__ F2 f_rcp(F2 a) { return f_pack(f_rcp(f_lane0(a)), f_rcp(f_lane1(a))); }
__device__ __forceinline__ float f_rsqrt(float x) {
  float r;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}
__device__ __forceinline__ F2 f_rsqrt(F2 a) { return f_pack(f_rsqrt(f_lane0(a)), f_rsqrt(f_lane1(a))); }

// A value h + l per lane; l is of the order of h's last bits, or of those of what h was cancelled from.  Sums are
// Knuth's two-sum (The Art of Computer Programming 2, 4.2.2), products take the low part from an FMA and
// quotients one correction from the exact remainder (Dekker, Numer. Math. 18, 1971), the low parts
// added in plain FP32.
template <class F>
struct P {
  F h, l;
};
using P2 = P<float>;
using P4 = P<F2>;

__device__ __forceinline__ P4 p_pack(P2 x, P2 y) { return P4{f_pack(x.h, y.h), f_pack(x.l, y.l)}; }
__device__ __forceinline__ P2 p_lane0(P4 x) { return P2{f_lane0(x.h), f_lane0(x.l)}; }
__device__ __forceinline__ P2 p_lane1(P4 x) { return P2{f_lane1(x.h), f_lane1(x.l)}; }
// lane 0 of x and lane 1 of y
__device__ __forceinline__ P4 p_mix(P4 x, P4 y) { return p_pack(p_lane0(x), p_lane1(y)); }
// a double literal, and a pair of PairGrid, in every lane
template <class F>
__device__ __forceinline__ P<F> p_const(double x) {
  const float h = (float)x;
  return P<F>{f_all<F>(h), f_all<F>((float)(x - (double)h))};
}
template <class F>
__device__ __forceinline__ P<F> p_const(const float (&x)[2]) {
  return P<F>{f_all<F>(x[0]), f_all<F>(x[1])};
}

template <class F>
__device__ __forceinline__ P<F> p_renorm(P<F> x) {
  const F s = f_add(x.h, x.l);
  return P<F>{s, f_add(x.l, f_sub(x.h, s))};
}
template <class F>
__device__ __forceinline__ P<F> p_neg(P<F> x) {
  return P<F>{f_neg(x.h), f_neg(x.l)};
}
template <class F>
__device__ __forceinline__ P<F> p_add(P<F> x, P<F> y) {
  const F s = f_add(x.h, y.h), t = f_sub(s, x.h);
  const F e = f_add(f_sub(x.h, f_sub(s, t)), f_sub(y.h, t));
  return P<F>{s, f_add(e, f_add(x.l, y.l))};
}
template <class F>
__device__ __forceinline__ P<F> p_sub(P<F> x, P<F> y) {
  const F s = f_sub(x.h, y.h), t = f_sub(s, x.h);
  const F e = f_sub(f_sub(x.h, f_sub(s, t)), f_add(y.h, t));
  return P<F>{s, f_add(e, f_sub(x.l, y.l))};
}
template <class F>
__device__ __forceinline__ P<F> p_mul(P<F> x, P<F> y) {
  const F p = f_mul(x.h, y.h);
  return P<F>{p, f_fma(x.l, y.h, f_fma(x.h, y.l, f_fma(x.h, y.h, f_neg(p))))};
}
template <class F>
__device__ __forceinline__ P<F> p_sqr(P<F> x) {
  const F p = f_mul(x.h, x.h);
  return P<F>{p, f_fma(f_add(x.h, x.h), x.l, f_fma(x.h, x.h, f_neg(p)))};
}
// times a number that FP32 holds exactly
template <class F>
__device__ __forceinline__ P<F> p_mulf(P<F> x, float c_) {
  const F c = f_all<F>(c_), p = f_mul(x.h, c);
  return P<F>{p, f_fma(x.l, c, f_fma(x.h, c, f_neg(p)))};
}
// times a power of two (per lane)
template <class F>
__device__ __forceinline__ P<F> p_scalev(P<F> x, F c) {
  return P<F>{f_mul(x.h, c), f_mul(x.l, c)};
}
template <class F>
__device__ __forceinline__ P<F> p_scale(P<F> x, float c) {
  return p_scalev(x, f_all<F>(c));
}
// x / y: the quotient of the leading parts and one correction from its exact remainder
template <class F>
__device__ __forceinline__ P<F> p_div(P<F> x, P<F> y) {
  const F r = f_rcp(y.h), q = f_mul(x.h, r), n = f_neg(q);
  const F e = f_add(f_fma(n, y.l, x.l), f_fma(n, y.h, x.h));
  return P<F>{q, f_mul(e, r)};
}
template <class F>
__device__ __forceinline__ P<F> p_rcp(P<F> y) {
  const F r = f_rcp(y.h), n = f_neg(r);
  const F e = f_fma(n, y.l, f_fma(n, y.h, f_all<F>(1.0f)));
  return P<F>{r, f_mul(e, r)};
}
// sqrt(x) and 1/sqrt(x)
template <class F>
__device__ __forceinline__ P<F> p_sqrt(P<F> x, P<F>& inv) {
  const F r = f_rsqrt(x.h), s = f_mul(x.h, r);
  const F e = f_mul(f_add(f_fma(f_neg(s), s, x.h), x.l), f_mul(f_all<F>(0.5f), r));
  const P<F> q = p_renorm(P<F>{s, e});
  inv = p_rcp(q);
  return q;
}
// the larger of |x| and |y|
__device__ __forceinline__ P2 p_maxabs(P2 x, P2 y) {
  const P2 a = x.h < 0.0f ? p_neg(x) : x, b = y.h < 0.0f ? p_neg(y) : y;
  return f_add(f_sub(a.h, b.h), f_sub(a.l, b.l)) > 0.0f ? a : b;
}
__device__ __forceinline__ P4 p_maxabs(P4 x, P4 y) {
  return p_pack(p_maxabs(p_lane0(x), p_lane0(y)), p_maxabs(p_lane1(x), p_lane1(y)));
}

// An FP64 number as a pair, through the integer pipe (a conversion instruction takes an FP64 slot):
// the leading 24 bits of the significand (truncated) and the other 29, rounded to 24.  Below the
// normal FP32 range: zero; above it, or not finite: NaN, which no test of p_smooth passes.
__device__ __forceinline__ P2 p_from(double x) {
  const int H = __double2hiint(x), L = __double2loint(x);
  const unsigned int u = (unsigned int)(H & 0x7fffffff) - 0x38000000u;  // exponent rebiased, in place
  unsigned int b = __funnelshift_l((unsigned int)L, u, 3);
  if (u >= 0x0ff00000u) b = (int)u < 0 ? 0u : 0x7fc00000u;
  b |= (unsigned int)H & 0x80000000u;
  const float unit = __fmul_rn(__uint_as_float(b & 0xff800000u), 0x1p-52f);  // +-1 ulp of x
  return P2{__uint_as_float(b), __fmul_rn(__uint2float_rn((unsigned int)L & 0x1fffffffu), unit)};
}
// An FP32 number as FP64 through the integer pipe (denormals become zero)
__device__ __forceinline__ double d_from(float x) {
  const unsigned int b = __float_as_uint(x), m = b & 0x7fffffffu;
  const unsigned int hi = m < 0x00800000u ? 0u : (m >> 3) + 0x38000000u;
  return __hiloint2double((int)(hi | (b & 0x80000000u)), m < 0x00800000u ? 0 : (int)(b << 29));
}

// The largest t_l at which the correction is evaluated in pairs (see above), and the range of
// e0 e1 e2 (e_l = beta_l + eps) in which its products keep their last bits: at the default
// eps = 1e-10 the smallest product is 1e-30.
constexpr float kPairMaxT = 0x1p-14f, kPairMinP = 5e-31f, kPairMax = 1e37f;

// What a stencil's corrections share: S1 = (e0 - e1) e2, S2 = (e0 - e2) e1, e0 e1 e2, tau, and the
// FP32 values Q = e1 e2 and R = e0 (e1 + e2) of the small terms of the denominators.
template <class F>
struct PStencil {
  P<F> tau, S1, S2, P_, d2, w, hdv;
  F Q, R;
};
// not true for a NaN: e0 e1 e2 holds those of every input
__device__ __forceinline__ bool p_smooth(float tau, float e0, float e1, float e2, float p) {
  return tau <= f_mul(kPairMaxT, fminf(e0, fminf(e1, e2))) && p >= kPairMinP;
}
__device__ __forceinline__ bool p_smooth(F2 tau, F2 e0, F2 e1, F2 e2, F2 p) {
  return p_smooth(f_lane0(tau), f_lane0(e0), f_lane0(e1), f_lane0(e2), f_lane0(p)) &&
         p_smooth(f_lane1(tau), f_lane1(e0), f_lane1(e1), f_lane1(e2), f_lane1(p));
}
// The stencil with differences d01, d12, end derivatives y0, y2, mesh size h; e1 = d01^2 + eps,
// e2 = d12^2 + eps.  Returns whether its corrections may be taken from pairs (in every lane).
template <class F>
__device__ __forceinline__ bool p_stencil(P<F> d01, P<F> d12, P<F> y0, P<F> y2, P<F> e1, P<F> e2, P<F> h,
                                          PStencil<F>& s) {
  const P<F> du = p_add(d01, d12), d2 = p_sub(d12, d01);
  s.hdv = p_mul(h, p_sub(y0, y2));
  s.d2 = d2;
  s.w = p_sub(p_mul(h, p_add(y0, y2)), du);
  const P<F> z = p_add(s.hdv, p_scale(d2, 2.0f));
  constexpr double k1 = 9.0 / 256.0 + 781.0 / 320.0, k3 = (13.0 / 3.0) * (67.0 / 520.0);
  constexpr double k2 = (13.0 / 3.0) * (67.0 / 520.0) * (67.0 / 520.0) + 1421461.0 / 36400.0;
  const P<F> a = p_mul(s.w, p_sub(p_mul(p_const<F>(k1), s.w), p_mulf(du, 0.1875f)));
  const P<F> b = p_mul(d2, p_add(p_mul(p_const<F>(5.0 / 6.0), d2), p_mul(p_const<F>(k3), z)));
  const P<F> X = p_renorm(p_add(p_add(a, b), p_mul(p_const<F>(k2), p_sqr(z))));
  const P<F> Y = p_renorm(p_scale(p_mul(du, d2), 0.5f));
  s.tau = p_sqr(p_maxabs(X, Y));
  const P<F> A1 = p_add(X, Y), A2 = p_sub(X, Y);
  const P<F> e0 = p_add(e1, A1);
  s.S1 = p_mul(A1, e2);
  s.S2 = p_mul(A2, e1);
  const P<F> Q = p_mul(e1, e2);
  s.P_ = p_mul(e0, Q);
  s.Q = Q.h;
  s.R = f_mul(e0.h, f_add(e1.h, e2.h));
  return p_smooth(s.tau.h, e0.h, e1.h, e2.h, s.P_.h);
}
// The correction from the candidates' deviations q1, q2 from the linear value: inv_l = 1/gamma_1 (or
// 1/d_1), G = gamma_0/gamma_1 (or d_0/d_1).  The quotient comes before the factor tau, whose
// smallest values would leave the FP32 range in the numerator.
template <class F>
__device__ __forceinline__ P<F> p_correction(const PStencil<F>& s, P<F> q1, P<F> q2, P<F> inv_l, float G) {
  P<F> den = p_mul(inv_l, s.P_);
  den.l = f_fma(s.tau.h, f_fma(f_all<F>(G), s.Q, s.R), den.l);
  return p_mul(s.tau, p_div(p_add(p_mul(s.S1, q1), p_mul(s.S2, q2)), p_renorm(den)));
}
// u at the stencil's right face and at its left face: the deviations of the candidates are
// a - d2/2 + b, a + b and a - b, a - d2/2 - b with a = d2/32 - 3 h dv/64, b = 3 w/32
template <class F>
__device__ __forceinline__ void p_deviations(const PStencil<F>& s, P<F>& a, P<F>& a2, P<F>& b) {
  a = p_sub(p_scale(s.d2, 0.03125f), p_mulf(s.hdv, 0.046875f));
  a2 = p_sub(a, p_scale(s.d2, 0.5f));
  b = p_mulf(s.w, 0.09375f);
}
template <class F>
__device__ __forceinline__ P<F> p_right_value(const PStencil<F>& s, P<F> inv_l, float G) {
  P<F> a, a2, b;
  p_deviations(s, a, a2, b);
  return p_correction(s, p_add(a2, b), p_add(a, b), inv_l, G);
}
template <class F>
__device__ __forceinline__ P<F> p_left_value(const PStencil<F>& s, P<F> inv_l, float G) {
  P<F> a, a2, b;
  p_deviations(s, a, a2, b);
  return p_correction(s, p_sub(a, b), p_sub(a2, b), inv_l, G);
}
// the right face of the stencil in lane 0 and the left face of that in lane 1: the two sides of a face
__device__ __forceinline__ P4 p_face_values(const PStencil<F2>& s, P4 inv_l, float G) {
  P4 a, a2, b;
  p_deviations(s, a, a2, b);
  b = p_scalev(b, f_pack(1.0f, -1.0f));
  return p_correction(s, p_add(p_mix(a2, a), b), p_add(p_mix(a, a2), b), inv_l, G);
}
// h times the modified derivative: deviations w/4 - d2/2 and w/4 + d2/2
template <class F>
__device__ __forceinline__ P<F> p_limited(const PStencil<F>& s, P<F> inv_l, float G) {
  const P<F> c = p_scale(s.w, 0.25f), d = p_scale(s.d2, 0.5f);
  return p_correction(s, p_sub(c, d), p_add(c, d), inv_l, G);
}

// ---------------------------------------------------------------------------------------------
// The characteristic fields of Eig in pairs.
template <int NC, class F>
struct EigP {
  P<F> u, v, H, c, hb1, hb2, hic, uc, hq2;

  // from the velocities, the enthalpy and c^2; gm1 = gamma - 1
  __device__ __forceinline__ void setup(P<F> u_, P<F> v_, P<F> H_, P<F> c2, P<F> gm1) {
    u = u_;
    v = v_;
    H = H_;
    P<F> ic;
    c = p_sqrt(c2, ic);
    hq2 = p_scale(NC == 4 ? p_add(p_sqr(u), p_sqr(v)) : p_sqr(u), 0.5f);
    hic = p_scale(ic, 0.5f);
    hb1 = p_scale(p_mul(gm1, p_sqr(ic)), 0.5f);
    hb2 = p_mul(hb1, hq2);
    uc = p_mul(u, c);
  }
  // the Roe average of two cells from their primitives (sqrt(rho), u[, v], H)
  __device__ __forceinline__ void setup_roe(const P<F>* A, const P<F>* B, P<F> gm1) {
    const P<F> iw = p_rcp(p_renorm(p_add(A[0], B[0])));
    const P<F> a = p_mul(A[0], iw), b = p_mul(B[0], iw);
    const P<F> ub = p_add(p_mul(a, A[1]), p_mul(b, B[1])), Hb = p_add(p_mul(a, A[NC - 1]), p_mul(b, B[NC - 1]));
    const P<F> vb = NC == 4 ? p_add(p_mul(a, A[2]), p_mul(b, B[2])) : p_const<F>(0.0);
    const P<F> q2 = NC == 4 ? p_add(p_sqr(ub), p_sqr(vb)) : p_sqr(ub);
    setup(ub, vb, Hb, p_renorm(p_mul(gm1, p_sub(Hb, p_scale(q2, 0.5f)))), gm1);
  }
  __device__ __forceinline__ void project(const P<F>* q, P<F>* w) const {
    P<F> k = p_sub(p_mul(u, q[1]), q[NC - 1]);
    if (NC == 4) k = p_add(k, p_mul(v, q[2]));
    const P<F> th = p_sub(p_mul(hb2, q[0]), p_mul(hb1, k));
    const P<F> sh = p_mul(p_sub(p_mul(u, q[0]), q[1]), hic);
    const P<F> q0 = q[0];
    if (NC == 4) w[2] = p_sub(q[2], p_mul(v, q0));
    w[0] = p_add(th, sh);
    w[1] = p_sub(q0, p_scale(th, 2.0f));
    w[NC - 1] = p_sub(th, sh);
  }
  __device__ __forceinline__ void back(const P<F>* w, P<F>* q) const {
    const P<F> sg = p_add(w[0], w[NC - 1]), dl = p_sub(w[NC - 1], w[0]);
    q[0] = p_add(sg, w[1]);
    q[1] = p_add(p_mul(u, q[0]), p_mul(c, dl));
    P<F> e = p_add(p_mul(H, sg), p_add(p_mul(hq2, w[1]), p_mul(uc, dl)));
    if (NC == 4) {
      q[2] = p_add(p_mul(v, q[0]), w[2]);
      e = p_add(e, p_mul(v, w[2]));
    }
    q[NC - 1] = e;
  }
};

// Velocities and enthalpy of a state (normal frame), and p/rho
template <int NC>
__device__ __forceinline__ void p_prim(const P2* U, P2 gm1, P2& u, P2& v, P2& H, P2& pr) {
  const P2 ir = p_rcp(U[0]);
  u = p_mul(U[1], ir);
  v = NC == 4 ? p_mul(U[2], ir) : P2{0.0f, 0.0f};
  const P2 ke = NC == 4 ? p_add(p_mul(U[1], u), p_mul(U[2], v)) : p_mul(U[1], u);
  const P2 p = p_mul(gm1, p_sub(U[NC - 1], p_scale(ke, 0.5f)));
  H = p_mul(p_add(U[NC - 1], p), ir);
  pr = p_mul(p, ir);
}

// A thread's pairs in shared memory, 16 bytes a slot: the arrays of the loops over vectors and
// characteristic fields, which stay loops.  Unrolled, the kernels' code is several times the
// instruction cache's reach and its fetches are waited for.  at: this thread's first slot.
struct PairSlots {
  ulonglong2* at;
  __device__ __forceinline__ P4 get(int k) const {
    const ulonglong2 t = at[k * kThreads];
    return P4{F2{t.x}, F2{t.y}};
  }
  __device__ __forceinline__ void set(int k, P4 x) const { at[k * kThreads] = make_ulonglong2(x.h.v, x.l.v); }
};
constexpr int kStencilSlots = 16;  // four vectors of four components

// Projects the four vectors of slots v NC + k in place.  A field that is small beside its vector comes
// out of the products with h and l of like size: they are renormalised for the squares that follow.
template <int NC>
__device__ __forceinline__ void p_project_slots(const EigP<NC, F2>& e, const PairSlots& sm) {
#pragma unroll 1
  for (int v = 0; v < 4; ++v) {
    P4 q[NC];
#pragma unroll
    for (int k = 0; k < NC; ++k) q[k] = sm.get(v * NC + k);
    e.project(q, q);
#pragma unroll
    for (int k = 0; k < NC; ++k) sm.set(v * NC + k, p_renorm(q[k]));
  }
}

// Whether the corrections are finite: a denominator that left the FP32 range shows in them
template <int NC>
__device__ __forceinline__ bool p_finite(const P4* n) {
  float s = 0.0f;
#pragma unroll
  for (int k = 0; k < NC; ++k) s = f_add(s, f_add(fabsf(f_lane0(n[k].h)), fabsf(f_lane1(n[k].h))));
  return s < kPairMax;
}

// The corrections of one face (normal frame), U^- = p_0^- + n^-, U^+ = p_0^+ + n^+ (n: lane 0 and lane
// 1), from the cell differences dU of the cells k-1..k+2 and their derivatives Z along the sweep; e:
// the characteristic fields at the face (unused for a scalar law).  For the Euler equations also
// sum = U^- + U^+ less the two centre values, dif = U^+ - U^-, hdif = h (D^+ - D^-) and size, the
// largest of the differences and h times the derivatives that they are formed from, per component.
// These are small beside the states, so pairs hold them to the last bit of the states; hdif has to be
// right to the last bit of h D as well, so the differences that it is made of, dU0 - dU2 (da), Z3 - Z0
// (zo) and Z2 - Z1 (zi), are taken in FP64.  Returns false where any field needs the FP64 weights.
template <int NC, int SYS>
__device__ __forceinline__ bool p_face(const double (&dU)[3][NC], const double (&Z)[4][NC], const double* da_,
                                       const double* zo_, const double* zi_, const EigP<NC, F2>& e,
                                       const PairGrid& pg, int dir, const PairSlots& sm, P4* n, P2* sum, P2* dif, P2* hdif,
                                       float* size) {
  const P4 h = p_const<F2>(pg.h[dir]), eps = p_const<F2>(pg.eps), ig = p_const<F2>(pg.ig1);
  P4 d1, d2, y1, y2;  // a scalar law's, per side: the differences and end derivatives of its stencil
  {
    P2 d[3][NC], z[4][NC];
#pragma unroll
    for (int k = 0; k < NC; ++k) {
#pragma unroll
      for (int q = 0; q < 3; ++q) d[q][k] = p_from(dU[q][k]);
#pragma unroll
      for (int q = 0; q < 4; ++q) z[q][k] = p_from(Z[q][k]);
    }
    if (SYS == SYS_EULER) {
      // two components at a time:
      // U^+ + U^- - U_k - U_{k+1} = (dU0 - dU2)/8 + 3h/64 (z3 - z0 - 3 (z2 - z1)) + n^+ + n^-,
      // U^+ - U^- = -(dU0 + dU1 + dU2)/8 + 3h/64 (z0 + z3 + 3 (z1 + z2)) + n^+ - n^- and
      // D^+ - D^- = 3/(16 h) (dU0 - dU2) + (z3 - z0 + 3 (z2 - z1))/16
#pragma unroll
      for (int k = 0; k < NC; k += 2) {
        const int k1 = k + 1 < NC ? k + 1 : k;
        const P4 a0 = p_pack(d[0][k], d[0][k1]), a1 = p_pack(d[1][k], d[1][k1]), a2 = p_pack(d[2][k], d[2][k1]);
        const P4 z0 = p_pack(z[0][k], z[0][k1]), z1 = p_pack(z[1][k], z[1][k1]);
        const P4 z2 = p_pack(z[2][k], z[2][k1]), z3 = p_pack(z[3][k], z[3][k1]);
        const P4 sz = p_add(p_add(z0, z3), p_mulf(p_add(z1, z2), 3.0f));
        const P4 zo = p_pack(p_from(zo_[k]), p_from(zo_[k1]));
        const P4 zi = p_mulf(p_pack(p_from(zi_[k]), p_from(zi_[k1])), 3.0f);
        const P4 da = p_pack(p_from(da_[k]), p_from(da_[k1]));
        const P4 t = p_add(p_scale(da, 0.125f), p_mulf(p_mul(h, p_sub(zo, zi)), 0.046875f));
        const P4 x = p_add(p_scale(p_add(p_add(a0, a2), a1), -0.125f), p_mulf(p_mul(h, sz), 0.046875f));
        const P4 y = p_add(p_mulf(da, 0.1875f), p_scale(p_mul(h, p_add(zo, zi)), 0.0625f));
        sum[k] = p_lane0(t);
        sum[k1] = k1 == k ? sum[k] : p_lane1(t);
        dif[k] = p_lane0(x);
        hdif[k] = p_lane0(y);
        dif[k1] = k1 == k ? dif[k] : p_lane1(x);
        hdif[k1] = k1 == k ? hdif[k] : p_lane1(y);
      }
#pragma unroll
      for (int k = 0; k < NC; ++k) {
        const float a = fmaxf(fmaxf(fabsf(z[0][k].h), fabsf(z[1][k].h)), fmaxf(fabsf(z[2][k].h), fabsf(z[3][k].h)));
        size[k] = fmaxf(fmaxf(fabsf(d[0][k].h), fmaxf(fabsf(d[1][k].h), fabsf(d[2][k].h))), a * pg.h[dir][0]);
      }
    }
    if (SYS == SYS_EULER) {
#pragma unroll
      for (int k = 0; k < NC; ++k) {
        sm.set(0 * NC + k, p_pack(d[0][k], d[1][k]));
        sm.set(1 * NC + k, p_pack(d[1][k], d[2][k]));
        sm.set(2 * NC + k, p_pack(z[0][k], z[1][k]));
        sm.set(3 * NC + k, p_pack(z[2][k], z[3][k]));
      }
    } else {
      d1 = p_pack(d[0][0], d[1][0]);
      d2 = p_pack(d[1][0], d[2][0]);
      y1 = p_pack(z[0][0], z[1][0]);
      y2 = p_pack(z[2][0], z[3][0]);
    }
  }
  P4 c[NC];
  bool ok = true;
  if (SYS == SYS_EULER) {
    p_project_slots<NC>(e, sm);
#pragma unroll 1
    for (int s = 0; s < NC; ++s) {
      PStencil<F2> st;
      d1 = sm.get(s);
      d2 = sm.get(NC + s);
      ok = p_stencil(d1, d2, sm.get(2 * NC + s), sm.get(3 * NC + s), p_add(p_sqr(d1), eps), p_add(p_sqr(d2), eps), h,
                     st) &&
           ok;
      sm.set(s, p_face_values(st, ig, pg.G));
    }
#pragma unroll
    for (int s = 0; s < NC; ++s) c[s] = sm.get(s);
  } else {
    PStencil<F2> st;
    ok = p_stencil(d1, d2, y1, y2, p_add(p_sqr(d1), eps), p_add(p_sqr(d2), eps), h, st);
    c[0] = p_face_values(st, ig, pg.G);
  }
  if (SYS == SYS_EULER) {
    e.back(c, n);
#pragma unroll
    for (int k = 0; k < NC; ++k) {
      const P2 a = p_lane0(n[k]), b = p_lane1(n[k]);
      sum[k] = p_add(sum[k], p_add(a, b));
      dif[k] = p_add(dif[k], p_sub(b, a));
    }
  } else {
    n[0] = c[0];
  }
  return ok && p_finite<NC>(n);
}

// The corrections of one cell in both directions (lane d: direction d, in its normal frame; in 1D the
// lanes are the same) from the cells i-1..i+1: nt of h times the modified derivative and, FACES (R2),
// nm and np of the values at the right and the left face.  Slots: the two differences and the two end
// derivatives.
template <int NC, int SYS, bool FACES>
__device__ __forceinline__ bool p_cell(const PairSlots& sm, const EigP<NC, F2>& e, P4 h, const PairGrid& pg, P4* nm,
                                       P4* np, P4* nt) {
  if (SYS == SYS_EULER) p_project_slots<NC>(e, sm);
  const P4 eps = p_const<F2>(pg.eps), ig = p_const<F2>(pg.ig1), id = p_const<F2>(pg.id1);
  P4 cm[NC], cp[NC], ct[NC];
  bool ok = true;
#pragma unroll 1
  for (int s = 0; s < NC; ++s) {
    PStencil<F2> st;
    const P4 d1 = sm.get(s), d2 = sm.get(NC + s);
    ok = p_stencil(d1, d2, sm.get(2 * NC + s), sm.get(3 * NC + s), p_add(p_sqr(d1), eps), p_add(p_sqr(d2), eps), h,
                   st) &&
         ok;
    sm.set(s, p_limited(st, id, pg.Gd));
    if (FACES) {
      sm.set(NC + s, p_right_value(st, ig, pg.G));
      sm.set(2 * NC + s, p_left_value(st, ig, pg.G));
    }
  }
#pragma unroll
  for (int s = 0; s < NC; ++s) {
    ct[s] = sm.get(s);
    if (FACES) {
      cm[s] = sm.get(NC + s);
      cp[s] = sm.get(2 * NC + s);
    }
  }
  if (SYS == SYS_EULER) {
    e.back(ct, nt);
    if (FACES) {
      e.back(cm, nm);
      e.back(cp, np);
    }
  } else {
    nt[0] = ct[0];
  }
  return ok && p_finite<NC>(nt) && (!FACES || (p_finite<NC>(nm) && p_finite<NC>(np)));
}

// The square of a change's size beside a state with 1/rho = ir and 1/E = ie (the momentum's beside
// sqrt(rho E)); each factor beside the state, so that no square leaves the FP32 range before it is compared
template <int NC>
__device__ __forceinline__ float p_rel2(const float* x, float ir, float ie) {
  const float a = x[0] * ir, b = x[NC - 1] * ie;
  float m2 = (x[1] * ir) * (x[1] * ie);
  if (NC == 4) m2 += (x[2] * ir) * (x[2] * ie);
  return fmaxf(fmaxf(a * a, b * b), m2);
}

// Whether pairs hold an Euler state with density rho and energy E, its fluxes and their derivatives on the
// mesh to the last bit: what d_from leaves out is below 2^-126, and has to stay below 2^-53 (here
// 2^-62) of the smallest of rho, E, rho c, E c and of these over h (rho c^2 ~ E); the upper bounds keep
// 1/rho^2 and the products of p_flux_pair inside FP32.  Not true for rho <= 0, E <= 0, infinities and NaN.
// On the exponents, in the integer pipe (hexp: the larger mesh size's, not below 0).
__device__ __forceinline__ bool p_units(double rho, double E, int hexp) {
  const int a = (__double2hiint(rho) >> 20) - 1023, b = (__double2hiint(E) >> 20) - 1023;
  const int low = min(min(2 * a, 2 * b), min(a + b, 3 * b - a));
  return a >= -50 && a <= 40 && b >= -50 && b <= 60 && b - a >= -40 && b - a <= 60 && low - 2 * hexp >= -128;
}

// The Lax-Friedrichs flux of an Euler face whose two states are close, from the sums U = U^- + U^+,
// D = D^- + D^+ and the differences dif = U^+ - U^-, hdif = h (D^+ - D^-).  With f homogeneous of
// degree one,
//   f(U^-) + f(U^+) = f(U) + q(U; dif) + O(dif^4),  q(U; r) = f''(U)[r, r] / 2,
//   f'(U^-) D^- + f'(U^+) D^+ = f'(U) D + q'(U; dif) + ..., q' the derivative of q along (D, D^+ - D^-)
// (the odd orders cancel).  q and q' are so small beside the fluxes where they are used that FP32
// carries them; where the differences are larger, or where the pairs' noise in them (2^-48 of size,
// what they were formed from) would show beside the rounding of the states, the FP64 code takes both
// states.
// Returns vf and vh: minus half of alpha times the differences plus half of q and q'; false where any of
// these is not held by FP32.
template <int NC>
__device__ __forceinline__ bool p_flux_pair(const double* U, const double* D, const P2* dif, const P2* hdif,
                                            const float* size, double alpha, P2 ih, const PairGrid& pg, const FU& f,
                                            double* vf, double* vh) {
  constexpr int E = NC - 1;
  float u_[NC], d_[NC];
#pragma unroll
  for (int k = 0; k < NC; ++k) {
    u_[k] = p_from(U[k]).h;
    d_[k] = p_from(D[k]).h;
  }
  const float rho = u_[0], gm1 = pg.gm1[0], ir = f_rcp(rho), ie = f_rcp(u_[E]);
  float r[NC], s[NC];  // the differences and the differences of the derivatives (h and l overlap)
#pragma unroll
  for (int k = 0; k < NC; ++k) {
    r[k] = f_add(dif[k].h, dif[k].l);
    s[k] = f_add(hdif[k].h, hdif[k].l);
  }
  // q is below 2^-32 of the fluxes, q' of the derivatives' fluxes
  const float r2 = p_rel2<NC>(r, ir, ie), d2 = p_rel2<NC>(size, ir, ie);
  if (!(r2 <= 0x1p-34f && d2 <= 0x1p-12f && r2 * p_rel2<NC>(s, ir, ie) <= 0x1p-64f * d2)) return false;
#pragma unroll
  for (int k = 0; k < NC; ++k) s[k] *= ih.h;
  // first-order changes of the velocities and of the pressure, second-order ones, and their
  // derivatives (t after a name)
  const float irt = -ir * ir * d_[0];
  const float u = u_[1] * ir, ut = (d_[1] - u * d_[0]) * ir;
  const float du = (r[1] - u * r[0]) * ir, dut = (s[1] - ut * r[0] - u * s[0] - du * d_[0]) * ir;
  float q2 = du * du, q2t = 2.0f * du * dut, ke = u * u, ket = 2.0f * u * ut;
  float ur = u * r[1], urt = ut * r[1] + u * s[1];
  float v = 0.0f, vt = 0.0f, dv = 0.0f, dvt = 0.0f;
  if (NC == 4) {
    v = u_[2] * ir;
    vt = (d_[2] - v * d_[0]) * ir;
    dv = (r[2] - v * r[0]) * ir;
    dvt = (s[2] - vt * r[0] - v * s[0] - dv * d_[0]) * ir;
    q2 += dv * dv;
    q2t += 2.0f * dv * dvt;
    ke += v * v;
    ket += 2.0f * v * vt;
    ur += v * r[2];
    urt += vt * r[2] + v * s[2];
  }
  const float p = gm1 * (u_[E] - 0.5f * rho * ke), pt = gm1 * (d_[E] - 0.5f * (d_[0] * ke + rho * ket));
  const float p1 = gm1 * (r[E] - ur + 0.5f * ke * r[0]), p1t = gm1 * (s[E] - urt + 0.5f * (ket * r[0] + ke * s[0]));
  const float p2 = -0.5f * gm1 * rho * q2, p2t = -0.5f * gm1 * (d_[0] * q2 + rho * q2t);
  const float a = du * r[0], at = dut * r[0] + du * s[0], hp = u_[E] + p, hpt = d_[E] + pt;
  float q[NC], t[NC];
  q[0] = t[0] = 0.0f;
  q[1] = rho * du * du + p2;
  t[1] = d_[0] * du * du + 2.0f * rho * du * dut + p2t;
  if (NC == 4) {
    q[2] = rho * du * dv;
    t[2] = d_[0] * du * dv + rho * (dut * dv + du * dvt);
  }
  q[E] = (r[E] + p1) * du - hp * a * ir + p2 * u;
  t[E] = (s[E] + p1t) * du + (r[E] + p1) * dut - (hpt * a + hp * at) * ir - hp * a * irt + p2t * u + p2 * ut;
  const P2 ma = p_scale(p_from(alpha), -0.5f);
  // an alpha outside the FP32 range (a NaN here, which d_from would make a number), or a product with it
  float big = fabsf(ma.h);
#pragma unroll
  for (int k = 0; k < NC; ++k) {
    P2 x = p_mul(ma, dif[k]), y = p_mul(p_mul(ma, hdif[k]), ih);
    x.l += 0.5f * q[k];
    y.l += 0.5f * t[k];
    big = f_add(big, f_add(f_add(fabsf(x.h), fabsf(x.l)), f_add(fabsf(y.h), fabsf(y.l))));
    vf[k] = f.add(d_from(x.h), d_from(x.l));
    vh[k] = f.add(d_from(y.h), d_from(y.l));
  }
  return big < kPairMax;
}

}  // namespace hw
