"""The reverse mode of the pair corrections (csrc/hweno_adjoint_pair.cuh) compiled for the host, its few
device instructions replaced by plain C++ (approximate reciprocals by ones that are off by 1e-7), against
forward-mode derivatives of the same correction in long double: right to 2^-53 of the linear part's
coefficients (which are of order one) whatever the linear weights, where a kernel would take pairs."""
import os
import re
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2411_11229_gb300", "csrc")

SHIM = r"""
#pragma once
#include <algorithm>
#include <cmath>
#include <cstdint>
#include <cstring>
#define __device__
#define __forceinline__ inline
using std::fma; using std::fmax; using std::fmin; using std::max; using std::min;
template <class A, class B> A bits(B b) { A a; std::memcpy(&a, &b, sizeof a); return a; }
static float __fadd_rn(float a, float b) { return a + b; }
static float __fsub_rn(float a, float b) { return a - b; }
static float __fmul_rn(float a, float b) { return a * b; }
static float __fmaf_rn(float a, float b, float c) { return std::fmaf(a, b, c); }
static int __double2hiint(double x) { return (int)(bits<int64_t>(x) >> 32); }
static int __double2loint(double x) { return (int)bits<int64_t>(x); }
static double __hiloint2double(int h, int l) { return bits<double>(((uint64_t)(uint32_t)h << 32) | (uint32_t)l); }
static unsigned __funnelshift_l(unsigned l, unsigned h, unsigned s) { return (unsigned)((((uint64_t)h << 32 | l) << s) >> 32); }
static float __uint_as_float(unsigned b) { return bits<float>(b); }
static unsigned __float_as_uint(float f) { return bits<unsigned>(f); }
static float __uint2float_rn(unsigned u) { return (float)u; }
static long long __double_as_longlong(double x) { return bits<long long>(x); }
static unsigned long long two(float x, float y) { return __float_as_uint(x) | (unsigned long long)__float_as_uint(y) << 32; }
static unsigned long long each(unsigned long long a, unsigned long long b, unsigned long long c, int op) {
  float r[2];
  for (int i = 0; i < 2; ++i) {
    const float x = bits<float>((unsigned)(a >> 32 * i)), y = bits<float>((unsigned)(b >> 32 * i));
    r[i] = op == 0 ? x + y : op == 1 ? x * y : std::fmaf(x, y, bits<float>((unsigned)(c >> 32 * i)));
  }
  return two(r[0], r[1]);
}
struct ulonglong2 { unsigned long long x, y; };
static ulonglong2 make_ulonglong2(unsigned long long a, unsigned long long b) { return {a, b}; }
static double rsqrt(double x) { return 1.0 / std::sqrt(x); }
"""

MAIN = r"""
#include <cstdio>
#include <random>
using namespace hw;
using R = long double;
struct D { R v, d; };
static D operator+(D a, D b) { return {a.v + b.v, a.d + b.d}; }
static D operator-(D a, D b) { return {a.v - b.v, a.d - b.d}; }
static D operator*(D a, D b) { return {a.v * b.v, a.d * b.v + a.v * b.d}; }
static D operator/(D a, D b) { const R q = a.v / b.v; return {q, (a.d - q * b.d) / b.v}; }
static D operator*(R k, D a) { return {k * a.v, k * a.d}; }
static D operator+(R k, D a) { return {k + a.v, a.d}; }
static D mag(D a) { return a.v < 0 ? D{-a.v, -a.d} : a; }
// nonlinear less linear value: 0 h times the modified derivative, 1 right face, 2 left face
static D correction(int kind, D a, D b, D hl, D hr, R g0) {
  const R g1 = (1 - g0) / 2, eps = 1e-10L;
  const D du = a + b, d2 = b - a, sv = hl + hr, dv = hl - hr;
  const D A = (R)11 / 16 * du - (R)3 / 16 * sv, B = (R)67 / 520 * dv + (R)197 / 260 * d2, C = (R)1 / 4 * (sv - du);
  const D E = (R)1 / 4 * (dv + (R)2 * d2);
  const D b0 = A * A + (R)13 / 3 * B * B + (R)781 / 20 * C * C + (R)1421461 / 2275 * E * E, b1 = a * a, b2 = b * b;
  const D s = (R)0.5 * (mag(b0 - b1) + mag(b0 - b2)), tau = s * s;
  const D W0 = (R)1 + tau / (eps + b0), W1 = (R)1 + tau / (eps + b1), W2 = (R)1 + tau / (eps + b2);
  const D mir[4] = {(R)-1 * b, (R)-1 * a, hr, hl};  // the stencil seen from the left face
  const D x = kind == 2 ? mir[0] : a, y = kind == 2 ? mir[1] : b, l = kind == 2 ? (R)-1 * mir[2] : hl, r = kind == 2 ? (R)-1 * mir[3] : hr;
  const D V1 = kind == 2 ? W2 : W1, V2 = kind == 2 ? W1 : W2;
  const D p0 = kind == 0 ? (R)0.75 * du - (R)0.25 * sv
                         : (R)0.125 * x + (R)0.5625 * y - (R)3 / 64 * l - (R)9 / 64 * r;
  const D p1 = kind == 0 ? a : (R)0.5 * x, p2 = kind == 0 ? b : (R)0.5 * y;
  return (W0 * (p0 - g1 * (p1 + p2)) + g1 * (V1 * p1 + V2 * p2)) / (g0 * W0 + g1 * (V1 + V2)) - p0;
}
static P4 pair(double x) { float p[2] = {(float)x, 0.0f}; p[1] = (float)(x - p[0]); return p_const<F2>(p); }
template <int KIND, bool SMALL32>
static void run(double g0) {
  std::mt19937_64 rng(5);
  auto u = [&] { return 2.0 * (double)(rng() >> 11) * 0x1p-53 - 1.0; };
  const double g1 = 0.5 * (1.0 - g0), G = g0 / g1, h = 1.0 / 64;
  R worst = 0;
  int used = 0;
  for (int it = 0; it < 60000; ++it) {
    const double a = std::exp(-2.0 - 6.0 * std::fabs(u())), b = a * (1.0 + 0.1 * u()) + 0.01 * u(), sg = it % 2 ? -1.0 : 1.0;
    const double x[4] = {sg * a, sg * b, sg * (a + 0.02 * u()) / h, sg * (b + 0.02 * u()) / h};
    P4 v[4], o[4];
    for (int q = 0; q < 4; ++q) v[q] = p_pack(p_from(x[q]), p_from(x[q]));
    bool ok = true;
    p_correction_vjp<KIND, SMALL32>(v[0], v[1], v[2], v[3], pair(h), pair(1e-10), pair(G + 2.0), pair(G), pair(1.0), o[0],
                                    o[1], o[2], o[3], ok);
    if (!ok) continue;
    ++used;
    for (int lane = 0; lane < 2; ++lane)
      for (int q = 0; q < 4; ++q) {
        D in[4];
        for (int m = 0; m < 4; ++m) in[m] = D{(R)x[m] * (m < 2 ? 1 : (R)h), m == q ? (m < 2 ? 1 : (R)h) : (R)0};
        const D c = correction(KIND == CORR_LIMITED ? 0 : 1 + lane, in[0], in[1], in[2], in[3], g0);
        const P2 t = lane ? p_lane1(o[q]) : p_lane0(o[q]);
        worst = std::max(worst, std::fabs(c.d - ((R)t.h + (R)t.l)) * (q < 2 ? 1 : 1 / (R)h));
      }
  }
  std::printf("%d %.3f %d %.2f\n", KIND, g0, used, (double)std::log2(worst));
}
int main() {
  // the form that the kernels choose
  for (double g0 : {0.99, 0.985, 0.95, 0.5, 0.02}) {
    if (2.0 / (1.0 - g0) >= kSmall32) run<CORR_FACE, true>(g0);
    else run<CORR_FACE, false>(g0);
  }
  for (double d0 : {0.9, 0.7, 0.5, 0.02}) run<CORR_LIMITED, false>(d0);
}
"""


def _host(name):
    s = open(os.path.join(CSRC, name)).read()
    for instr, call in (("rcp.approx.ftz.f32", "r = (1.0f / x) * (1.0f + 1e-7f);"),
                        ("rsqrt.approx.ftz.f32", "r = (1.0f / std::sqrt(x)) * (1.0f - 1e-7f);"),
                        ("rcp.approx.ftz.f64", "r = 1.0 / x;"), ("rsqrt.approx.ftz.f64", "r = 1.0 / std::sqrt(x);"),
                        ("mov.b64", "r.v = two(x, y);"), ("add.rn.f32x2", "r.v = each(a.v, b.v, 0, 0);"),
                        ("mul.rn.f32x2", "r.v = each(a.v, b.v, 0, 1);"), ("fma.rn.f32x2", "r.v = each(a.v, b.v, c.v, 2);")):
        s = re.sub(r'asm\("' + re.escape(instr) + r'[^;]*;[^;]*;', call, s)
    assert "asm(" not in s
    return re.sub(r'#(include "hweno_[^"]*"|pragma once).*', "", s)


@pytest.mark.skipif(shutil.which("g++") is None, reason="needs g++")
def test_derivatives_of_the_corrections(tmp_path):
    src = SHIM.replace("#pragma once", "") + "".join(
        _host(f) for f in ("hweno_math.cuh", "hweno_pair.cuh", "hweno_adjoint_pair.cuh")) + MAIN
    (tmp_path / "t.cpp").write_text(src)
    subprocess.run(["g++", "-std=c++17", "-O1", "-ffp-contract=off", "-w", "-o", str(tmp_path / "t"), str(tmp_path / "t.cpp")],
                   check=True)
    out = subprocess.run([str(tmp_path / "t")], check=True, capture_output=True, text=True).stdout
    rows = [r.split() for r in out.splitlines()]
    assert len(rows) == 9
    for kind, weight, used, err in rows:
        assert int(used) > 200, rows
        assert float(err) <= -53.0, rows
