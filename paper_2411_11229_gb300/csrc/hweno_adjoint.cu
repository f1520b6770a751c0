// Adjoint of one SSP-RK3 step of the Euler equations (1D and 2D), hand-written: see
// include/hweno.h (hweno_adjoint_step) for the contract.
//
// The vector-Jacobian product of one stage operator, lam = (dM/dS)^T muM + (dL/dS)^T muL at a
// stage input S with alpha fixed, is the transpose of the forward kernels:
//   k_adj_cell   per cell and direction: backward of the modified derivative (Eq. limiter in the
//                cell's characteristic fields): contributions to U of cells i-1..i+1 and to the
//                derivative of cells i-1, i+1;
//   k_adj_face   per face: recomputes the face and back-propagates the flux adjoint
//                nu = (muL[right cell] - muL[left cell]) / h through the LF fluxes at U^+-, the
//                back projection, the HWENO weights and smoothness indicators, the projections,
//                the eigenvectors and the Roe average: contributions to U and to the derivative
//                of the four cells of the face;
//   k_adj_gather per cell: collects those contributions, applies the transposes of the (linear)
//                D-terms and mixed fluxes to the flux adjoints and the nodal flux VJPs, and adds
//                the identity part of M.
// Contributions are stored per face / per cell and gathered (no atomics: deterministic).
// In 2D, k_adj_cell_pair and k_adj_face_pair form the same contributions with the transposes of the
// nonlinear part in pairs (hweno_adjoint_pair.cuh) and list the cells and faces that need the FP64 weights
// for k_adj_cell and k_adj_face.  1D grids, and 2D ones up to kAdjPairMinCells, are too small to fill the FP64 pipe and keep the FP64 kernels.
#include <cmath>
#include "hweno_adjoint.cuh"
#include "hweno_adjoint_pair.cuh"
#include "hweno_host.cuh"

using namespace hwh;

namespace hw {

struct AdjWork {
  double* CU;  // face contributions to U: [dir][face][4 cells][NC] (original frame)
  double* CD;  // face contributions to the own-direction derivative, same layout
  double* CM;  // modified-derivative contributions: [dir][cell][3 U + 2 D][NC] (original frame)
  const double* scal;  // the handle's scalars; [4..7] are zero (read by fu_of)
  // 2D: the cells and faces that k_adj_cell_pair and k_adj_face_pair leave to the FP64 kernels:
  // count[0] cells * 2 + direction in cells, count[1] faces of both directions in faces
  unsigned int* count;
  unsigned int *cells, *faces;
};

// -------------------------------------------------------------------------------------------
template <int DIM>
__device__ __forceinline__ void adj_cell(const Grid& g, const double* __restrict__ S, const double* __restrict__ muM,
                                         const AdjWork& aw, int d, long long p) {
  constexpr int NC = DIM == 1 ? 3 : 4;
  const long long plane = g.plane;
  const int i = (int)(p % g.nx), j = (int)(p / g.nx);
  const int n = d == 0 ? g.nx : g.ny;
  const int a0 = d == 0 ? i : j;
  const int fld = d == 0 ? 1 : 2;
  const double ih = g.ih[d];
  const FU fu = fu_of(aw.scal);
  // the derivatives enter unscaled, as in the forward cell kernel (h folded into the constants)
  double U3[3][NC], D3[3][NC];
  long long pc[3];
  bool refl[3];
#pragma unroll
  for (int q = 0; q < 3; ++q) {
    const int ac = bc_map(a0 - 1 + q, n, g.bc, refl[q]);
    pc[q] = HW_IDX(d == 0 ? (long long)j * g.nx + ac : (long long)ac * g.nx + i, plane);
#pragma unroll
    for (int k = 0; k < NC; ++k) {
      U3[q][k] = S[k * plane + pc[q]];
      D3[q][k] = S[(fld * NC + k) * plane + pc[q]];
    }
    if (d == 1) {
      swap_frame<NC>(U3[q]);
      swap_frame<NC>(D3[q]);
    }
    mirror_U<NC>(U3[q], refl[q]);
    mirror_D<NC>(D3[q], refl[q]);
  }
  // forward: eigenvectors of the cell's own state
  const Prim<NC> pr = prim_of<NC>(U3[1], g.gm1, fu);
  const double H = (U3[1][NC - 1] + pr.p) * pr.ir;
  const double c2 = g.gamma * pr.p * pr.ir;
  const double ic = rsqrt(c2);
  const double c = c2 * ic;
  Eig<NC> e;
  e.setup(pr.u, pr.v, H, c, ic, g.gm1);
  // the limiter sees the characteristic fields only through differences of neighbouring cells
  double dU[2][NC], Dq[2][NC], Zm[NC], Zp[NC], ht[NC];
#pragma unroll
  for (int q = 0; q < 2; ++q)
#pragma unroll
    for (int k = 0; k < NC; ++k) dU[q][k] = fu.sub(U3[q + 1][k], U3[q][k]);
  e.project(dU[0], Dq[0], fu);
  e.project(dU[1], Dq[1], fu);
  e.project(D3[0], Zm, fu);
  e.project(D3[2], Zp, fu);
  // forward intermediates of the limiter, per field, kept in this thread's shared-memory slots
  extern __shared__ double adj_cell_sm[];
  double* const svb = adj_cell_sm + threadIdx.x;
  const AdjK ak = adj_k(g, d, fu);
#pragma unroll
  for (int s = 0; s < NC; ++s)
    ht[s] = cell_field_save(Dq[0][s], Dq[1][s], Zm[s], Zp[s], ak, svb + s * kCellSaved * kThreads, kThreads, fu) * ih;
  // backward from the adjoint of the modified derivative of this cell
  double ob[NC];
#pragma unroll
  for (int k = 0; k < NC; ++k) ob[k] = muM[(fld * NC + k) * plane + p];
  if (d == 1) swap_frame<NC>(ob);
  EigBar eb = {0.0, 0.0, 0.0, 0.0, 0.0};
  double hq2b = 0.0, ucb = 0.0, hb1b = 0.0, hb2b = 0.0, hicb = 0.0;
  double htb[NC];
#pragma unroll
  for (int s = 0; s < NC; ++s) htb[s] = 0.0;
  back_bwd<NC>(e, ht, ob, htb, hq2b, ucb, eb, fu);
  double Dqb[2][NC], Zmb[NC], Zpb[NC];
#pragma unroll
  for (int s = 0; s < NC; ++s) {
    double db[2] = {0.0, 0.0};
    Zmb[s] = Zpb[s] = 0.0;
    cell_field_bwd_saved(Dq[0][s], Dq[1][s], Zm[s], Zp[s], ak, htb[s] * ih, svb + s * kCellSaved * kThreads,
                         kThreads, db, Zmb[s], Zpb[s], fu);
    Dqb[0][s] = db[0];
    Dqb[1][s] = db[1];
  }
  double dUb[2][NC], Ub[3][NC], Dmb[NC], Dpb[NC];
#pragma unroll
  for (int k = 0; k < NC; ++k) {
    dUb[0][k] = dUb[1][k] = 0.0;
    Dmb[k] = Dpb[k] = 0.0;
  }
#pragma unroll
  for (int q = 0; q < 2; ++q) project_bwd<NC>(e, dU[q], Dqb[q], dUb[q], hb1b, hb2b, hicb, eb, fu);
  project_bwd<NC>(e, D3[0], Zmb, Dmb, hb1b, hb2b, hicb, eb, fu);
  project_bwd<NC>(e, D3[2], Zpb, Dpb, hb1b, hb2b, hicb, eb, fu);
#pragma unroll
  for (int k = 0; k < NC; ++k) {
    Ub[0][k] = -dUb[0][k];
    Ub[1][k] = fu.sub(dUb[0][k], dUb[1][k]);
    Ub[2][k] = dUb[1][k];
  }
  setup_bwd<NC>(e, g.gm1, ic, hb1b, hb2b, hicb, hq2b, ucb, eb);
  // c = sqrt(c2), ic = 1/sqrt(c2), c2 = gamma p ir, H = (E + p) ir
  const double c2b = 0.5 * ic * (eb.c - eb.ic * ic * ic);
  double pb = c2b * g.gamma * pr.ir + eb.H * pr.ir;
  double irb = c2b * g.gamma * pr.p + eb.H * (U3[1][NC - 1] + pr.p);
  Ub[1][NC - 1] += eb.H * pr.ir;
  prim_bwd<NC>(U3[1], pr, g.gm1, irb, eb.u, eb.v, pb, Ub[1], fu);
  // a mirrored neighbour was read through the sign table: its contributions go back through it
  // (the table is its own transpose)
#pragma unroll
  for (int q = 0; q < 3; ++q) mirror_U<NC>(Ub[q], refl[q]);
  mirror_D<NC>(Dmb, refl[0]);
  mirror_D<NC>(Dpb, refl[2]);
  // store (original frame): 3 U contributions, then the derivative adjoints of cells i-1, i+1
  double* out = aw.CM + ((long long)d * plane + p) * 5 * NC;
#pragma unroll
  for (int q = 0; q < 3; ++q) {
    if (d == 1) swap_frame<NC>(Ub[q]);
#pragma unroll
    for (int k = 0; k < NC; ++k) out[q * NC + k] = Ub[q][k];
  }
  if (d == 1) {
    swap_frame<NC>(Dmb);
    swap_frame<NC>(Dpb);
  }
#pragma unroll
  for (int k = 0; k < NC; ++k) {
    out[3 * NC + k] = Dmb[k];
    out[4 * NC + k] = Dpb[k];
  }
}

// 1D: every cell; 2D: the cells of the list, or every one where there is no list
template <int DIM>
__global__ void __launch_bounds__(kThreads) k_adj_cell(Grid g, const double* __restrict__ S, const double* __restrict__ muM,
                                                       AdjWork aw) {
  long long k = (long long)blockIdx.x * kThreads + threadIdx.x;
  if (DIM == 1) {
    if (k < g.plane) adj_cell<1>(g, S, muM, aw, 0, k);
    return;
  }
  const long long n = aw.cells ? min((long long)aw.count[0], 2 * g.plane) : 2 * g.plane;
  for (; k < n; k += (long long)gridDim.x * kThreads) {
    const unsigned int c = aw.cells ? aw.cells[HW_IDX(k, 2 * g.plane)] : (unsigned int)k;
    if ((long long)(c >> 1) < g.plane) adj_cell<DIM>(g, S, muM, aw, (int)(c & 1u), HW_IDX(c >> 1, g.plane));
  }
}

// -------------------------------------------------------------------------------------------
template <int DIM>
__device__ __forceinline__ void adj_face(const Grid& g, const double* __restrict__ S, const double* __restrict__ muL,
                                         const AdjWork& aw, const double* __restrict__ alpha2, int dir, long long f) {
  constexpr int NC = DIM == 1 ? 3 : 4;
  const long long plane = g.plane;
  const int n = dir == 0 ? g.nx : g.ny;
  int fa, line;
  if (dir == 0) {
    line = (int)(f / (n + 1));
    fa = (int)(f % (n + 1));
  } else {
    fa = (int)(f / g.nx);
    line = (int)(f % g.nx);
  }
  long long pc[4];
  bool refl[4];
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const int a = bc_map(fa - 2 + q, n, g.bc, refl[q]);
    pc[q] = HW_IDX(dir == 0 ? (long long)line * g.nx + a : (long long)a * g.nx + line, plane);
  }
  const int fown = dir == 0 ? 1 : 2;
  // 1/(2h): the flux adjoints below are differences (mu_L[right] - mu_L[left]) without their 1/h,
  // which this coefficient carries together with the 1/2 of the LF fluxes
  const double hih = g.hih[dir];
  const double k21 = g.uvd[dir][0], k3 = g.uvd[dir][1];
  const double alpha = alpha2[dir];
  const FU fu = fu_of(aw.scal);
  double Uq[4][NC], Zq[4][NC];
#pragma unroll
  for (int q = 0; q < 4; ++q) {
#pragma unroll
    for (int k = 0; k < NC; ++k) {
      Uq[q][k] = S[k * plane + pc[q]];
      Zq[q][k] = S[(fown * NC + k) * plane + pc[q]];  // unscaled, as in the forward face kernel
    }
    if (dir == 1) {
      swap_frame<NC>(Uq[q]);
      swap_frame<NC>(Zq[q]);
    }
    mirror_U<NC>(Uq[q], refl[q]);
    mirror_D<NC>(Zq[q], refl[q]);
  }
  // adjoints of the face fluxes of U and of the own derivative (normal frame)
  double nuf[NC], nuh[NC];
  {
    const bool hasL = fa - 1 >= 0, hasR = fa <= n - 1;
    // (an outer face has one cell inside: its address serves both loads)
    const int aL = hasL ? fa - 1 : fa, aR = hasR ? fa : fa - 1;
    const long long cL = HW_IDX(dir == 0 ? (long long)line * g.nx + aL : (long long)aL * g.nx + line, plane);
    const long long cR = HW_IDX(dir == 0 ? (long long)line * g.nx + aR : (long long)aR * g.nx + line, plane);
#pragma unroll
    for (int k = 0; k < NC; ++k) {
      const double rf = muL[k * plane + cR], lf = muL[k * plane + cL];
      const double rh = muL[(fown * NC + k) * plane + cR], lh = muL[(fown * NC + k) * plane + cL];
      nuf[k] = fu.sub(hasR ? rf : 0.0, hasL ? lf : 0.0);
      nuh[k] = fu.sub(hasR ? rh : 0.0, hasL ? lh : 0.0);
    }
    if (dir == 1) {
      swap_frame<NC>(nuf);
      swap_frame<NC>(nuh);
    }
  }
  // ---- forward recomputation
  const Prim<NC> pl = prim_of<NC>(Uq[1], g.gm1, fu), prr = prim_of<NC>(Uq[2], g.gm1, fu);
  const double sl = sqrt(Uq[1][0]), sr = sqrt(Uq[2][0]);
  const double Hl = (Uq[1][NC - 1] + pl.p) * pl.ir, Hr = (Uq[2][NC - 1] + prr.p) * prr.ir;
  const double iw = rcp(fu.add(sl, sr), fu);
  const double ub = fu.mul(fma(sl, pl.u, fu.mul(sr, prr.u)), iw);
  const double vb = NC == 4 ? fu.mul(fma(sl, pl.v, fu.mul(sr, prr.v)), iw) : 0.0;
  const double Hb = fu.mul(fma(sl, Hl, fu.mul(sr, Hr)), iw);
  const double c2 = g.gm1 * fma(-0.5, NC == 4 ? fma(ub, ub, vb * vb) : ub * ub, Hb);
  const double ic = rsqrt(c2);
  Eig<NC> e;
  e.setup(ub, vb, Hb, c2 * ic, ic, g.gm1);
  // the interpolation sees the characteristic fields only through differences of neighbouring
  // cells; the interface derivatives (Eq. P'xi) are linear in the stencil and formed in conserved
  // variables (k21 = 21/(16 h), k3 = 3/(16 h))
  double dU[3][NC], Dm[NC], Dp[NC];
#pragma unroll
  for (int q = 0; q < 3; ++q)
#pragma unroll
    for (int k = 0; k < NC; ++k) dU[q][k] = fu.sub(Uq[q + 1][k], Uq[q][k]);
#pragma unroll
  for (int k = 0; k < NC; ++k) {
    Dm[k] = fma(k21, dU[1][k], fma(-k3, dU[0][k], fma(0.0625, Zq[0][k], -0.1875 * Zq[2][k])));
    Dp[k] = fma(k21, dU[1][k], fma(-k3, dU[2][k], fma(-0.1875, Zq[1][k], 0.0625 * Zq[3][k])));
  }
  double Dq[3][NC], Yq[4][NC];
#pragma unroll
  for (int q = 0; q < 3; ++q) e.project(dU[q], Dq[q], fu);
#pragma unroll
  for (int q = 0; q < 4; ++q) e.project(Zq[q], Yq[q], fu);
  double cm[NC], cp[NC];
  // forward intermediates of the interpolation, per field, kept in this thread's shared-memory slots
  extern __shared__ double adj_face_sm[];
  double* const svb = adj_face_sm + threadIdx.x;
  const AdjK ak = adj_k(g, dir, fu);
#pragma unroll
  for (int s = 0; s < NC; ++s)
    face_field_save(Dq[0][s], Dq[1][s], Dq[2][s], Yq[0][s], Yq[1][s], Yq[2][s], Yq[3][s], ak, cm[s], cp[s],
                    svb + s * kFaceSaved * kThreads, kThreads, fu);
  // interface states: centre states plus the back-projected corrections
  double Um[NC], Up[NC];
  e.back_add(cm, Uq[1], Um, fu);
  e.back_add(cp, Uq[2], Up, fu);
  // ---- backward: fh = (FUm + FUp - alpha (Up - Um)) / 2 + Df, hh = (HDm + HDp - alpha (Dp - Dm)) / 2
  // + Dh, with the flux adjoints nuf / h and nuh / h
  double Umb[NC], Upb[NC], Dmb[NC], Dpb[NC], Fb[NC], Hb2[NC];
  const double ha = hih * alpha;
#pragma unroll
  for (int k = 0; k < NC; ++k) {
    Umb[k] = ha * nuf[k];
    Upb[k] = -Umb[k];
    Dmb[k] = ha * nuh[k];
    Dpb[k] = -Dmb[k];
    Fb[k] = hih * nuf[k];
    Hb2[k] = hih * nuh[k];
  }
  {
    // the primitives of each interface state, shared by its flux and Jacobian-product backward
    const Prim<NC> qm = prim_of<NC>(Um, g.gm1, fu), qp = prim_of<NC>(Up, g.gm1, fu);
    flux_bwd<NC>(Um, qm, g.gm1, Fb, Umb, fu);
    flux_bwd<NC>(Up, qp, g.gm1, Fb, Upb, fu);
    jvp_bwd<NC>(Um, qm, Dm, g.gm1, Hb2, Umb, Dmb, fu);
    jvp_bwd<NC>(Up, qp, Dp, g.gm1, Hb2, Upb, Dpb, fu);
  }
  EigBar eb = {0.0, 0.0, 0.0, 0.0, 0.0};
  double hq2b = 0.0, ucb = 0.0, hb1b = 0.0, hb2b = 0.0, hicb = 0.0;
  double cmb[NC], cpb[NC];
#pragma unroll
  for (int s = 0; s < NC; ++s) cmb[s] = cpb[s] = 0.0;
  back_bwd<NC>(e, cm, Umb, cmb, hq2b, ucb, eb, fu);
  back_bwd<NC>(e, cp, Upb, cpb, hq2b, ucb, eb, fu);
  double Uqb[4][NC], Zqb[4][NC], dUb[3][NC];
#pragma unroll
  for (int k = 0; k < NC; ++k) {
    // the centre states enter Um, Up directly; the derivatives linearly
    Uqb[0][k] = Uqb[3][k] = 0.0;
    Uqb[1][k] = Umb[k];
    Uqb[2][k] = Upb[k];
    dUb[0][k] = -k3 * Dmb[k];
    dUb[1][k] = k21 * fu.add(Dmb[k], Dpb[k]);
    dUb[2][k] = -k3 * Dpb[k];
    Zqb[0][k] = 0.0625 * Dmb[k];
    Zqb[1][k] = -0.1875 * Dpb[k];
    Zqb[2][k] = -0.1875 * Dmb[k];
    Zqb[3][k] = 0.0625 * Dpb[k];
  }
  double Dqb[3][NC], Yb[4][NC];
#pragma unroll
  for (int s = 0; s < NC; ++s) {
    double db[3] = {0.0, 0.0, 0.0}, yb[4] = {0.0, 0.0, 0.0, 0.0};
    face_field_bwd_saved(Dq[0][s], Dq[1][s], Dq[2][s], Yq[0][s], Yq[1][s], Yq[2][s], Yq[3][s], ak, cmb[s], cpb[s],
                         svb + s * kFaceSaved * kThreads, kThreads, db, yb, fu);
#pragma unroll
    for (int q = 0; q < 3; ++q) Dqb[q][s] = db[q];
#pragma unroll
    for (int q = 0; q < 4; ++q) Yb[q][s] = yb[q];
  }
#pragma unroll
  for (int q = 0; q < 3; ++q) project_bwd<NC>(e, dU[q], Dqb[q], dUb[q], hb1b, hb2b, hicb, eb, fu);
#pragma unroll
  for (int q = 0; q < 4; ++q) project_bwd<NC>(e, Zq[q], Yb[q], Zqb[q], hb1b, hb2b, hicb, eb, fu);
#pragma unroll
  for (int q = 0; q < 3; ++q)
#pragma unroll
    for (int k = 0; k < NC; ++k) {
      Uqb[q + 1][k] = fu.add(Uqb[q + 1][k], dUb[q][k]);
      Uqb[q][k] = fu.sub(Uqb[q][k], dUb[q][k]);
    }
  setup_bwd<NC>(e, g.gm1, ic, hb1b, hb2b, hicb, hq2b, ucb, eb);
  // c = sqrt(c2), ic = 1/sqrt(c2); c2 = gm1 (Hb - (ub^2 + vb^2)/2)
  const double c2b = 0.5 * ic * (eb.c - eb.ic * ic * ic);
  const double Hbb = eb.H + g.gm1 * c2b;
  const double ubb = eb.u - g.gm1 * ub * c2b;
  const double vbb = eb.v - g.gm1 * vb * c2b;
  // Roe average: x_b = (sl x_l + sr x_r) iw for x in (u, v, H)
  const double iwb = ubb * fma(sl, pl.u, sr * prr.u) + (NC == 4 ? vbb * fma(sl, pl.v, sr * prr.v) : 0.0) +
                     Hbb * fma(sl, Hl, sr * Hr);
  const double slb = iw * (ubb * pl.u + (NC == 4 ? vbb * pl.v : 0.0) + Hbb * Hl) - iwb * iw * iw;
  const double srb = iw * (ubb * prr.u + (NC == 4 ? vbb * prr.v : 0.0) + Hbb * Hr) - iwb * iw * iw;
  // cells 1 and 2: sqrt(rho), u, v, H = (E + p) ir; d sqrt(rho) / d rho = sqrt(rho) ir / 2
  {
    const double Hlb = Hbb * sl * iw;
    Uqb[1][0] += slb * (0.5 * sl) * pl.ir;
    Uqb[1][NC - 1] += Hlb * pl.ir;
    prim_bwd<NC>(Uq[1], pl, g.gm1, Hlb * (Uq[1][NC - 1] + pl.p), ubb * sl * iw, vbb * sl * iw, Hlb * pl.ir, Uqb[1]);
    const double Hrb = Hbb * sr * iw;
    Uqb[2][0] += srb * (0.5 * sr) * prr.ir;
    Uqb[2][NC - 1] += Hrb * prr.ir;
    prim_bwd<NC>(Uq[2], prr, g.gm1, Hrb * (Uq[2][NC - 1] + prr.p), ubb * sr * iw, vbb * sr * iw, Hrb * prr.ir,
                 Uqb[2]);
  }
  // store (original frame): the contributions to U and to the unscaled derivative of the direction
  const long long fo = HW_IDX(dir == 0 ? (long long)line * (g.nx + 1) + fa : (long long)fa * g.nx + line,
                              dir == 0 ? (long long)(g.nx + 1) * g.ny : (long long)(g.ny + 1) * g.nx);
  const long long base = ((dir == 0 ? 0 : (long long)(g.nx + 1) * g.ny) + fo) * 4 * NC;
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    mirror_U<NC>(Uqb[q], refl[q]);
    mirror_D<NC>(Zqb[q], refl[q]);
    if (dir == 1) {
      swap_frame<NC>(Uqb[q]);
      swap_frame<NC>(Zqb[q]);
    }
#pragma unroll
    for (int k = 0; k < NC; ++k) {
      aw.CU[base + q * NC + k] = Uqb[q][k];
      aw.CD[base + q * NC + k] = Zqb[q][k];
    }
  }
}

// 1D: every face; 2D: the faces of the list, or every one where there is no list
template <int DIM>
__global__ void __launch_bounds__(kThreads) k_adj_face(Grid g, const double* __restrict__ S, const double* __restrict__ muL,
                                                       AdjWork aw, const double* __restrict__ alpha2) {
  long long k = (long long)blockIdx.x * kThreads + threadIdx.x;
  const long long nfx = (long long)(g.nx + 1) * g.ny;
  if (DIM == 1) {
    if (k < nfx) adj_face<1>(g, S, muL, aw, alpha2, 0, k);
    return;
  }
  const long long all = nfx + (long long)(g.ny + 1) * g.nx;
  const long long n = aw.faces ? min((long long)aw.count[1], all) : all;
  for (; k < n; k += (long long)gridDim.x * kThreads) {
    const long long f = HW_IDX(aw.faces ? (long long)aw.faces[HW_IDX(k, all)] : k, all);
    if (f < all) adj_face<DIM>(g, S, muL, aw, alpha2, f < nfx ? 0 : 1, f < nfx ? f : f - nfx);
  }
}

// -------------------------------------------------------------------------------------------
// The pairs of a thread in shared memory (unrolled, k_adj_face_pair's 96 KB of instructions waited for
// themselves: 5.2 of 14 stall cycles, 1.14 ms per 512^2 launch against 0.52 ms)
// slots: vector v, component k; field s, vector v; one per field
constexpr int kPairSlots = 36;
__device__ __forceinline__ int slot_q(int v, int k) { return v * 4 + k; }
__device__ __forceinline__ int slot_w(int s, int v) { return 16 + s * 4 + v; }
__device__ __forceinline__ int slot_c(int s) { return 32 + s; }

// The same contributions of a 2D cell (both directions: the lanes of its pairs) with the transpose of
// the limiter's nonlinear part in pairs; false where the FP64 kernel is needed.
__device__ __forceinline__ bool adj_cell_pair(const Grid& g, const double* __restrict__ S,
                                              const double* __restrict__ muM, const AdjWork& aw, long long p,
                                              const PairSlots& sm) {
  constexpr int NC = 4;
  const long long plane = g.plane;
  const FU fu = fu_of(aw.scal);
  const int i = (int)(p % g.nx), j = (int)(p / g.nx);
  bool refl[2][2], units;
  double ob[2][NC];
  P4 U1[NC];
  {
    // the differences in FP64: the derivatives of the weights see them relative to themselves
    P2 du[2][2][NC], z[2][2][NC];
    double Uc[NC];
#pragma unroll
    for (int k = 0; k < NC; ++k) Uc[k] = S[k * plane + p];
    units = p_units(Uc[0], Uc[NC - 1], g.pg.hexp);
#pragma unroll
    for (int d = 0; d < 2; ++d) {
      const int n = d == 0 ? g.nx : g.ny, a0 = d == 0 ? i : j, fld = d == 0 ? 1 : 2;
#pragma unroll
      for (int q = 0; q < 2; ++q) {  // the neighbours i - 1, i + 1
        const int ac = bc_map(a0 - 1 + 2 * q, n, g.bc, refl[d][q]);
        const long long pc = HW_IDX(d == 0 ? (long long)j * g.nx + ac : (long long)ac * g.nx + i, plane);
        double U[NC], D[NC];
#pragma unroll
        for (int k = 0; k < NC; ++k) {
          U[k] = S[k * plane + pc];
          D[k] = S[(fld * NC + k) * plane + pc];
        }
        if (d == 1) {
          swap_frame<NC>(U);
          swap_frame<NC>(D);
        }
        mirror_U<NC>(U, refl[d][q]);
        mirror_D<NC>(D, refl[d][q]);
#pragma unroll
        for (int k = 0; k < NC; ++k) {
          const double c = Uc[d == 1 && (k == 1 || k == 2) ? 3 - k : k];
          du[q][d][k] = p_from(q == 0 ? fu.sub(c, U[k]) : fu.sub(U[k], c));
          z[q][d][k] = p_from(D[k]);
        }
      }
#pragma unroll
      for (int k = 0; k < NC; ++k) ob[d][k] = muM[(fld * NC + k) * plane + p];
      if (d == 1) swap_frame<NC>(ob[d]);
    }
#pragma unroll
    for (int k = 0; k < NC; ++k) {
      U1[k] = p_pack(p_from(Uc[k]), p_from(Uc[k == 1 || k == 2 ? 3 - k : k]));
#pragma unroll
      for (int q = 0; q < 2; ++q) {
        sm.set(slot_q(q, k), p_pack(du[q][0][k], du[q][1][k]));
        sm.set(slot_q(2 + q, k), p_pack(z[q][0][k], z[q][1][k]));
      }
    }
  }
  unsigned int big = 0u;
#pragma unroll
  for (int k = 0; k < NC; ++k) big = max(big, max(seed_bits(ob[0][k]), seed_bits(ob[1][k])));
  int sh;
  if (!seed_scale(big, sh)) return false;
  const P4 gm1 = p_const<F2>(g.pg.gm1);
  // the cell's characteristic fields
  const P4 ir = p_rcp(U1[0]), u = p_mul(U1[1], ir), v = p_mul(U1[2], ir);
  const P4 pr = p_mul(gm1, p_sub(U1[3], p_scale(p_add(p_mul(U1[1], u), p_mul(U1[2], v)), 0.5f)));
  const P4 ep = p_add(U1[3], pr), prir = p_mul(pr, ir);
  EigP<NC, F2> e;
  e.setup(u, v, p_mul(ep, ir), p_renorm(p_add(prir, p_mul(gm1, prir))), gm1);
  // seeds: of h v~ in the characteristic fields
  const P4 h = p_pack(p_const<float>(g.pg.h[0]), p_const<float>(g.pg.h[1]));
  const P4 ih = p_pack(p_const<float>(g.pg.ih[0]), p_const<float>(g.pg.ih[1]));
  P4 qb[NC], c[NC];
#pragma unroll
  for (int k = 0; k < NC; ++k) qb[k] = p_mul(p_pack(p_from_scaled(ob[0][k], sh), p_from_scaled(ob[1][k], sh)), ih);
  p_back_t(e, qb, c);
#pragma unroll
  for (int s = 0; s < NC; ++s) sm.set(slot_c(s), c[s]);
#pragma unroll 1
  for (int v = 0; v < 4; ++v) {
    P4 q[NC];
#pragma unroll
    for (int k = 0; k < NC; ++k) q[k] = sm.get(slot_q(v, k));
    e.project(q, q);
#pragma unroll
    for (int k = 0; k < NC; ++k) sm.set(slot_w(k, v), p_renorm(q[k]));
  }
  const P4 eps = p_const<F2>(g.pg.eps), id = p_const<F2>(g.pg.id1), Gd = p_const<F2>(g.pg.Gdp);
  bool ok = true;
#pragma unroll 1
  for (int s = 0; s < NC; ++s) {
    P4 w0, w1, w2, w3;
    sm.set(slot_c(s), p_correction_vjp<CORR_LIMITED, false>(sm.get(slot_w(s, 0)), sm.get(slot_w(s, 1)),
                                                            sm.get(slot_w(s, 2)), sm.get(slot_w(s, 3)), h, eps, id, Gd,
                                                            sm.get(slot_c(s)), w0, w1, w2, w3, ok));
    sm.set(slot_w(s, 0), w0);
    sm.set(slot_w(s, 1), w1);
    sm.set(slot_w(s, 2), w2);
    sm.set(slot_w(s, 3), w3);
  }
#pragma unroll
  for (int s = 0; s < NC; ++s) c[s] = sm.get(slot_c(s));
  if (!units || !ok || !p_finite<NC>(c)) return false;
  EigPBar<F2> eb;
  eb.zero();
  p_back_eig(c, qb, eb);
#pragma unroll 1
  for (int v = 0; v < 4; ++v) {
    P4 q[NC], wb[NC], t[NC];
#pragma unroll
    for (int k = 0; k < NC; ++k) {
      q[k] = sm.get(slot_q(v, k));
      wb[k] = sm.get(slot_w(k, v));
    }
    p_project_vjp(e, q, wb, t, eb);
#pragma unroll
    for (int k = 0; k < NC; ++k) sm.set(slot_q(v, k), t[k]);
  }
  P4 c2b;
  p_setup_vjp(e, gm1, eb, c2b);
  // c^2 = gamma p / rho, H = (E + p) / rho
  const P4 gc = p_add(c2b, p_mul(gm1, c2b)), Hi = p_mul(eb.H, ir);
  P4 Ub[NC];
#pragma unroll
  for (int k = 0; k < NC; ++k) Ub[k] = p_sub(sm.get(slot_q(0, k)), sm.get(slot_q(1, k)));
  Ub[3] = p_add(Ub[3], Hi);
  p_prim_vjp(U1, ir, u, v, gm1, p_add(p_mul(gc, pr), p_mul(eb.H, ep)), eb.u, eb.v, p_add(p_mul(gc, ir), Hi), Ub);
  if (!p_finite<NC>(Ub)) return false;
#pragma unroll
  for (int d = 0; d < 2; ++d) {
    auto lane = [&](P4 x) { return d_from_scaled(d == 0 ? p_lane0(x) : p_lane1(x), sh, fu); };
    double o[5][NC];
#pragma unroll
    for (int k = 0; k < NC; ++k) {
      // the linear part of v~: 3/4 (u_{i+1} - u_{i-1})/h - (v_{i-1} + v_{i+1})/4
      o[0][k] = fma(-g.l34[d], ob[d][k], -lane(sm.get(slot_q(0, k))));
      o[1][k] = lane(Ub[k]);
      o[2][k] = fma(g.l34[d], ob[d][k], lane(sm.get(slot_q(1, k))));
      o[3][k] = fma(-0.25, ob[d][k], lane(sm.get(slot_q(2, k))));
      o[4][k] = fma(-0.25, ob[d][k], lane(sm.get(slot_q(3, k))));
    }
    // mirrored neighbours: back through the sign table
    mirror_U<NC>(o[0], refl[d][0]);
    mirror_U<NC>(o[2], refl[d][1]);
    mirror_D<NC>(o[3], refl[d][0]);
    mirror_D<NC>(o[4], refl[d][1]);
    double* out = aw.CM + ((long long)d * plane + p) * 5 * NC;
#pragma unroll
    for (int q = 0; q < 5; ++q) {
      if (d == 1) swap_frame<NC>(o[q]);
#pragma unroll
      for (int k = 0; k < NC; ++k) out[q * NC + k] = o[q][k];
    }
  }
  return true;
}

// Bound by its FP32 work (54 % of the FMA pipe, FP64 26 %): three blocks of 128 per SM (168 registers, 74 KB
// of slots each).  2D Euler 1024^2: 0.51 ms per launch against 2.32 ms for the FP64 kernel.
__global__ void __launch_bounds__(kThreads, 3) k_adj_cell_pair(Grid g, const double* __restrict__ S,
                                                               const double* __restrict__ muM, AdjWork aw) {
  const long long p = (long long)blockIdx.x * kThreads + threadIdx.x;
  extern __shared__ ulonglong2 adj_pair_slots[];
  if (p < g.plane && !adj_cell_pair(g, S, muM, aw, HW_IDX(p, g.plane), PairSlots{adj_pair_slots + threadIdx.x})) {
    const unsigned int k = atomicAdd(aw.count, 2u);
    aw.cells[HW_IDX(k, 2 * g.plane)] = (unsigned int)p * 2u;
    aw.cells[HW_IDX((long long)k + 1, 2 * g.plane)] = (unsigned int)p * 2u + 1u;
  }
}

// -------------------------------------------------------------------------------------------
// The contributions of a 2D face with the transpose of the interpolation's nonlinear part in pairs;
// false where the FP64 kernel is needed.
template <bool SMALL32>
__device__ __forceinline__ bool adj_face_pair(const Grid& g, const double* __restrict__ S,
                                              const double* __restrict__ muL, const AdjWork& aw,
                                              const double* __restrict__ alpha2, int dir, long long f, const PairSlots& sm) {
  constexpr int NC = 4;
  const long long plane = g.plane;
  const int n = dir == 0 ? g.nx : g.ny;
  int fa, line;
  if (dir == 0) {
    line = (int)(f / (n + 1));
    fa = (int)(f % (n + 1));
  } else {
    fa = (int)(f / g.nx);
    line = (int)(f % g.nx);
  }
  const FU fu = fu_of(aw.scal);
  const int fown = dir == 0 ? 1 : 2;
  bool refl[4];
  double Uq[2][NC];                  // the inner cells
  double Um[NC], Up[NC], Dm[NC], Dp[NC];  // interface states less the corrections
  const double k21 = g.uvd[dir][0], k3 = g.uvd[dir][1], l3 = g.l3[dir], l9 = g.l9[dir];
  bool units;
  {
    double U[4][NC], Z[4][NC];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int a = bc_map(fa - 2 + q, n, g.bc, refl[q]);
      const long long pc = HW_IDX(dir == 0 ? (long long)line * g.nx + a : (long long)a * g.nx + line, plane);
#pragma unroll
      for (int k = 0; k < NC; ++k) {
        U[q][k] = S[k * plane + pc];
        Z[q][k] = S[(fown * NC + k) * plane + pc];
      }
      if (dir == 1) {
        swap_frame<NC>(U[q]);
        swap_frame<NC>(Z[q]);
      }
      mirror_U<NC>(U[q], refl[q]);
      mirror_D<NC>(Z[q], refl[q]);
    }
    units = p_units(U[1][0], U[1][NC - 1], g.pg.hexp) && p_units(U[2][0], U[2][NC - 1], g.pg.hexp);
#pragma unroll
    for (int k = 0; k < NC; ++k) {
      const double a = fu.sub(U[1][k], U[0][k]), b = fu.sub(U[2][k], U[1][k]), c = fu.sub(U[3][k], U[2][k]);
      Um[k] = fma(0.125, a, fma(0.5625, b, fma(-l3, Z[0][k], -l9 * Z[2][k])));
      Up[k] = fma(-0.125, c, fma(-0.5625, b, fma(l3, Z[3][k], l9 * Z[1][k])));
      Dm[k] = fma(k21, b, fma(-k3, a, fma(0.0625, Z[0][k], -0.1875 * Z[2][k])));
      Dp[k] = fma(k21, b, fma(-k3, c, fma(-0.1875, Z[1][k], 0.0625 * Z[3][k])));
      Uq[0][k] = U[1][k];
      Uq[1][k] = U[2][k];
      const P2 pb = p_from(b);
      // per side (lane): the differences and the end derivatives of its stencil
      sm.set(slot_q(0, k), p_pack(p_from(a), pb));
      sm.set(slot_q(1, k), p_pack(pb, p_from(c)));
      sm.set(slot_q(2, k), p_pack(p_from(Z[0][k]), p_from(Z[1][k])));
      sm.set(slot_q(3, k), p_pack(p_from(Z[2][k]), p_from(Z[3][k])));
    }
  }
  // primitives of the two inner cells (lanes) and their Roe average
  const P4 gm1 = p_const<F2>(g.pg.gm1);
  P4 UI[NC];
#pragma unroll
  for (int k = 0; k < NC; ++k) UI[k] = p_pack(p_from(Uq[0][k]), p_from(Uq[1][k]));
  P4 inv;
  const P4 ir = p_rcp(UI[0]), u = p_mul(UI[1], ir), v = p_mul(UI[2], ir), sq = p_sqrt(UI[0], inv);
  const P4 pr = p_mul(gm1, p_sub(UI[3], p_scale(p_add(p_mul(UI[1], u), p_mul(UI[2], v)), 0.5f)));
  const P4 ep = p_add(UI[3], pr), H = p_mul(ep, ir);
  const P2 iw_ = p_rcp(p_renorm(p_sum(sq)));
  const P4 iw = p_pack(iw_, iw_), wt = p_mul(sq, iw);  // the weights of the average
  const P2 ub = p_sum(p_mul(wt, u)), vb = p_sum(p_mul(wt, v)), Hb = p_sum(p_mul(wt, H));
  EigP<NC, F2> e;
  {
    const P2 q2 = p_add(p_sqr(ub), p_sqr(vb));
    const P2 c2 = p_renorm(p_mul(p_const<float>(g.pg.gm1), p_sub(Hb, p_scale(q2, 0.5f))));
    e.setup(p_pack(ub, ub), p_pack(vb, vb), p_pack(Hb, Hb), p_pack(c2, c2), gm1);
  }
  const P4 h = p_const<F2>(g.pg.h[dir]), eps = p_const<F2>(g.pg.eps), ig = p_const<F2>(g.pg.ig1);
#pragma unroll 1
  for (int v = 0; v < 4; ++v) {
    P4 q[NC];
#pragma unroll
    for (int k = 0; k < NC; ++k) q[k] = sm.get(slot_q(v, k));
    e.project(q, q);
#pragma unroll
    for (int k = 0; k < NC; ++k) sm.set(slot_w(k, v), p_renorm(q[k]));
  }
  P4 nb[NC];
  {
    P4 c[NC], nn[NC];
    bool ok = true;
#pragma unroll 1
    for (int s = 0; s < NC; ++s) {
      PStencil<F2> st;
      const P4 w0 = sm.get(slot_w(s, 0)), w1 = sm.get(slot_w(s, 1));
      ok = p_stencil(w0, w1, sm.get(slot_w(s, 2)), sm.get(slot_w(s, 3)), p_add(p_sqr(w0), eps), p_add(p_sqr(w1), eps),
                     h, st) &&
           ok;
      sm.set(slot_c(s), p_face_values(st, ig, g.pg.G));
    }
#pragma unroll
    for (int s = 0; s < NC; ++s) c[s] = sm.get(slot_c(s));
    e.back(c, nn);
    if (!units || !ok || !p_finite<NC>(nn)) return false;
#pragma unroll
    for (int k = 0; k < NC; ++k) {
      const P2 a = p_lane0(nn[k]), b = p_lane1(nn[k]);
      Um[k] = fu.add(Uq[0][k], fu.add(Um[k], fu.add(d_from(a.h), d_from(a.l))));
      Up[k] = fu.add(Uq[1][k], fu.add(Up[k], fu.add(d_from(b.h), d_from(b.l))));
    }
  }
  // FP64: the fluxes' transposes, as in adj_face
  double Umb[NC], Upb[NC], Dmb[NC], Dpb[NC];
  {
    double Fb[NC], Hb2[NC];
    const double hih = g.hih[dir], ha = hih * alpha2[dir];
    const bool hasL = fa - 1 >= 0, hasR = fa <= n - 1;
    // (an outer face has one cell inside: its address serves both loads)
    const int aL = hasL ? fa - 1 : fa, aR = hasR ? fa : fa - 1;
    const long long cL = HW_IDX(dir == 0 ? (long long)line * g.nx + aL : (long long)aL * g.nx + line, plane);
    const long long cR = HW_IDX(dir == 0 ? (long long)line * g.nx + aR : (long long)aR * g.nx + line, plane);
    double nuf[NC], nuh[NC];
#pragma unroll
    for (int k = 0; k < NC; ++k) {
      const double rf = muL[k * plane + cR], lf = muL[k * plane + cL];
      const double rh = muL[(fown * NC + k) * plane + cR], lh = muL[(fown * NC + k) * plane + cL];
      nuf[k] = fu.sub(hasR ? rf : 0.0, hasL ? lf : 0.0);
      nuh[k] = fu.sub(hasR ? rh : 0.0, hasL ? lh : 0.0);
    }
    if (dir == 1) {
      swap_frame<NC>(nuf);
      swap_frame<NC>(nuh);
    }
#pragma unroll
    for (int k = 0; k < NC; ++k) {
      Umb[k] = ha * nuf[k];
      Upb[k] = -Umb[k];
      Dmb[k] = ha * nuh[k];
      Dpb[k] = -Dmb[k];
      Fb[k] = hih * nuf[k];
      Hb2[k] = hih * nuh[k];
    }
    const Prim<NC> qm = prim_of<NC>(Um, g.gm1, fu), qp = prim_of<NC>(Up, g.gm1, fu);
    flux_bwd<NC>(Um, qm, g.gm1, Fb, Umb, fu);
    flux_bwd<NC>(Up, qp, g.gm1, Fb, Upb, fu);
    jvp_bwd<NC>(Um, qm, Dm, g.gm1, Hb2, Umb, Dmb, fu);
    jvp_bwd<NC>(Up, qp, Dp, g.gm1, Hb2, Upb, Dpb, fu);
  }
  // pairs: the transpose of the corrections
  unsigned int big = 0u;
#pragma unroll
  for (int k = 0; k < NC; ++k) big = max(big, max(seed_bits(Umb[k]), seed_bits(Upb[k])));
  int sh;
  if (!seed_scale(big, sh)) return false;
#pragma unroll
  for (int k = 0; k < NC; ++k) nb[k] = p_pack(p_from_scaled(Umb[k], sh), p_from_scaled(Upb[k], sh));
  P4 c[NC];
  p_back_t(e, nb, c);
#pragma unroll
  for (int s = 0; s < NC; ++s) sm.set(slot_c(s), c[s]);
#pragma unroll 1
  for (int s = 0; s < NC; ++s) {
    bool ok = true;
    P4 w0, w1, w2, w3;
    sm.set(slot_c(s), p_correction_vjp<CORR_FACE, SMALL32>(sm.get(slot_w(s, 0)), sm.get(slot_w(s, 1)),
                                                           sm.get(slot_w(s, 2)), sm.get(slot_w(s, 3)), h, eps, ig,
                                                           p_const<F2>(g.pg.Gp), sm.get(slot_c(s)), w0, w1, w2, w3, ok));
    sm.set(slot_w(s, 0), w0);
    sm.set(slot_w(s, 1), w1);
    sm.set(slot_w(s, 2), w2);
    sm.set(slot_w(s, 3), w3);
  }
#pragma unroll
  for (int s = 0; s < NC; ++s) c[s] = sm.get(slot_c(s));
  EigPBar<F2> eb;
  eb.zero();
  p_back_eig(c, nb, eb);
#pragma unroll 1
  for (int v = 0; v < 4; ++v) {
    P4 q[NC], wb[NC];
#pragma unroll
    for (int k = 0; k < NC; ++k) {
      q[k] = sm.get(slot_q(v, k));
      wb[k] = sm.get(slot_w(k, v));
    }
    P4 b[NC];
    p_project_vjp(e, q, wb, b, eb);
#pragma unroll
    for (int k = 0; k < NC; ++k) sm.set(slot_q(v, k), b[k]);
  }
  P4 c2b, UIb[NC];
  p_setup_vjp(e, gm1, eb, c2b);
  {
    // both lanes held the same basis: the sums of their adjoints; c^2 = gm1 (H - (u^2 + v^2)/2), then the
    // Roe average x = (s_l x_l + s_r x_r) iw
    const P2 gc = p_mul(p_const<float>(g.pg.gm1), p_sum(c2b));
    const P2 Hs = p_add(p_sum(eb.H), gc);
    const P2 us = p_sub(p_sum(eb.u), p_mul(gc, ub)), vs = p_sub(p_sum(eb.v), p_mul(gc, vb));
    const P4 H4 = p_pack(Hs, Hs), u4 = p_pack(us, us), v4 = p_pack(vs, vs);
    const P4 t = p_add(p_mul(u4, u), p_add(p_mul(v4, v), p_mul(H4, H)));
    const P2 iwb_ = p_sum(p_mul(sq, t));
    const P4 iwb = p_mul(p_pack(iwb_, iwb_), p_sqr(iw));
    const P4 sb = p_sub(p_mul(iw, t), iwb);
    const P4 Hl = p_mul(H4, wt), Hi = p_mul(Hl, ir);
    const P2 zero = p_const<float>(0.0);
    UIb[0] = p_mul(p_mul(sb, p_scale(sq, 0.5f)), ir);
    UIb[1] = UIb[2] = p_pack(zero, zero);
    UIb[3] = Hi;
    p_prim_vjp(UI, ir, u, v, gm1, p_mul(Hl, ep), p_mul(u4, wt), p_mul(v4, wt), Hi, UIb);
  }
  if (!p_finite<NC>(UIb)) return false;
  // FP64: the transposes of the linear parts, and the pairs added
  const long long fo = HW_IDX(dir == 0 ? (long long)line * (g.nx + 1) + fa : (long long)fa * g.nx + line,
                              dir == 0 ? (long long)(g.nx + 1) * g.ny : (long long)(g.ny + 1) * g.nx);
  const long long base = ((dir == 0 ? 0 : (long long)(g.nx + 1) * g.ny) + fo) * 4 * NC;
  double Ub[4][NC], Zb[4][NC];
#pragma unroll
  for (int k = 0; k < NC; ++k) {
    const P4 b1 = sm.get(slot_q(0, k)), b2 = sm.get(slot_q(1, k)), z1 = sm.get(slot_q(2, k)), z2 = sm.get(slot_q(3, k));
    const P2 a0 = p_lane0(b1), a1 = p_add(p_lane1(b1), p_lane0(b2)), a2 = p_lane1(b2);
    const double m0 = d_from_scaled(p_neg(a0), sh, fu);
    const double m1 = d_from_scaled(p_add(p_sub(a0, a1), p_lane0(UIb[k])), sh, fu);
    const double m2 = d_from_scaled(p_add(p_sub(a1, a2), p_lane1(UIb[k])), sh, fu);
    const double m3 = d_from_scaled(a2, sh, fu);
    const double c1 = fma(0.5625, fu.sub(Umb[k], Upb[k]), k21 * fu.add(Dmb[k], Dpb[k]));
    Ub[0][k] = fma(-0.125, Umb[k], fma(k3, Dmb[k], m0));
    Ub[1][k] = fma(1.125, Umb[k], fma(-k3, Dmb[k], fu.sub(m1, c1)));
    Ub[2][k] = fma(1.125, Upb[k], fma(k3, Dpb[k], fu.add(m2, c1)));
    Ub[3][k] = fma(-0.125, Upb[k], fma(-k3, Dpb[k], m3));
    Zb[0][k] = fma(-l3, Umb[k], fma(0.0625, Dmb[k], d_from_scaled(p_lane0(z1), sh, fu)));
    Zb[1][k] = fma(l9, Upb[k], fma(-0.1875, Dpb[k], d_from_scaled(p_lane1(z1), sh, fu)));
    Zb[2][k] = fma(-l9, Umb[k], fma(-0.1875, Dmb[k], d_from_scaled(p_lane0(z2), sh, fu)));
    Zb[3][k] = fma(l3, Upb[k], fma(0.0625, Dpb[k], d_from_scaled(p_lane1(z2), sh, fu)));
  }
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    mirror_U<NC>(Ub[q], refl[q]);
    mirror_D<NC>(Zb[q], refl[q]);
    if (dir == 1) {
      swap_frame<NC>(Ub[q]);
      swap_frame<NC>(Zb[q]);
    }
#pragma unroll
    for (int k = 0; k < NC; ++k) {
      aw.CU[base + q * NC + k] = Ub[q][k];
      aw.CD[base + q * NC + k] = Zb[q][k];
    }
  }
  return true;
}

// Bound by the FP64 pipe (72 % busy; the fluxes' transposes) with the pairs' latency between.  1024^2: 2.0 ms
// per launch against 5.95 ms for the FP64 kernel; two or four blocks per SM: the adjoint step 11.6 and
// 11.7 ms against 11.4 ms.
template <bool SMALL32>
__global__ void __launch_bounds__(kThreads, 3) k_adj_face_pair(Grid g, const double* __restrict__ S,
                                                               const double* __restrict__ muL, AdjWork aw,
                                                               const double* __restrict__ alpha2) {
  const int dir = blockIdx.y;
  const long long nfx = (long long)(g.nx + 1) * g.ny, nf = dir == 0 ? nfx : (long long)(g.ny + 1) * g.nx;
  const long long f = (long long)blockIdx.x * kThreads + threadIdx.x;
  extern __shared__ ulonglong2 adj_pair_slots[];
  if (f < nf && !adj_face_pair<SMALL32>(g, S, muL, aw, alpha2, dir, f, PairSlots{adj_pair_slots + threadIdx.x}))
    aw.faces[HW_IDX(atomicAdd(aw.count + 1, 1u), nfx + (long long)(g.ny + 1) * g.nx)] =
        (unsigned int)(f + (dir == 0 ? 0 : nfx));
}

// -------------------------------------------------------------------------------------------
// aliases of cell a (0 <= a < n) among the unmapped indices -2 .. n+1 of the stencils
__device__ __forceinline__ int aliases(int a, int n, int bc, int* x) {
  int k = 0;
  x[k++] = a;
  if (bc == BC_PERIODIC) {
    if (a + n <= n + 1) x[k++] = a + n;
    if (a - n >= -2) x[k++] = a - n;
  } else if (bc == BC_REFLECTIVE) {
    // ghost -1-a mirrors cell a (a = 0, 1), ghost 2n-1-a mirrors it (a = n-1, n-2)
    if (-1 - a >= -2) x[k++] = -1 - a;
    if (2 * n - 1 - a <= n + 1) x[k++] = 2 * n - 1 - a;
  } else {
    if (a == 0) {
      x[k++] = -1;
      x[k++] = -2;
    }
    if (a == n - 1) {
      x[k++] = n;
      x[k++] = n + 1;
    }
  }
  return k;
}

template <int DIM>
__global__ void __launch_bounds__(kThreads, 4) k_adj_gather(Grid g, const double* __restrict__ S,
                                                         const double* __restrict__ muM, const double* __restrict__ muL,
                                                         AdjWork aw, double* __restrict__ lam) {
  constexpr int NC = DIM == 1 ? 3 : 4;
  constexpr int NF = DIM + 1;
  const long long plane = g.plane;
  const long long p = (long long)blockIdx.x * kThreads + threadIdx.x;
  if (p >= plane) return;
  const FU fu = fu_of(aw.scal);
  const int i = (int)(p % g.nx), j = (int)(p / g.nx);
  double lb[NF][NC];
#pragma unroll
  for (int k = 0; k < NC; ++k) {
    lb[0][k] = muM[k * plane + p];  // M = (U, ...): identity part
#pragma unroll
    for (int f = 1; f < NF; ++f) lb[f][k] = 0.0;
  }
  double U[NC], V[NF - 1][NC];
#pragma unroll
  for (int k = 0; k < NC; ++k) {
    U[k] = S[k * plane + p];
#pragma unroll
    for (int f = 1; f < NF; ++f) V[f - 1][k] = S[(f * NC + k) * plane + p];
  }
  const Prim<NC> qc = prim_of<NC>(U, g.gm1, fu);  // original frame
  const long long oplx = (long long)g.ny * (g.nx + 1);
#pragma unroll
  for (int d = 0; d < DIM; ++d) {
    const int n = d == 0 ? g.nx : g.ny;
    const int a0 = d == 0 ? i : j;
    const int fown = d == 0 ? 1 : 2, foth = d == 0 ? 2 : 1;
    const double ih = g.ih[d];
    int xs[3];
    const int nx_ = aliases(a0, n, g.bc, xs);
    double nf[NC], nh[NC], no[NC];
#pragma unroll
    for (int k = 0; k < NC; ++k) nf[k] = nh[k] = no[k] = 0.0;
    // the normal momentum (original frame) and the nodal sign tables of a mirrored alias: f and
    // the mixed value change sign except for the normal momentum, h only for it
    const int km = d == 0 ? 1 : 2;
    const double cf_ih = DCoef::cf * ih, ef_ih = g.efih[d] * ih, eg_ih = g.egih[d] * ih;
    const double ch_ih = g.chh[d] * ih, eh_ih = DCoef::eh * ih;
    const double m7_ih = (7.0 / 12.0) * ih, m1_ih = (-1.0 / 12.0) * ih;
    for (int t = 0; t < nx_; ++t) {
      const int x = xs[t];
      const bool mir = g.bc == BC_REFLECTIVE && (x < 0 || x >= n);
      // faces fa = x + 2 - q hold this cell at position q
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const int fa = x + 2 - q;
        if (fa < 0 || fa > n) continue;
        const int line = d == 0 ? j : i;
        const long long fo = HW_IDX(d == 0 ? (long long)line * (g.nx + 1) + fa : (long long)fa * g.nx + line,
                                    d == 0 ? oplx : (long long)(g.ny + 1) * g.nx);
        const long long base = ((d == 0 ? 0 : oplx) + fo) * 4 * NC + q * NC;
#pragma unroll
        for (int k = 0; k < NC; ++k) {
          lb[0][k] = fu.add(lb[0][k], aw.CU[base + k]);
          lb[fown][k] = fu.add(lb[fown][k], aw.CD[base + k]);
        }
        // flux adjoints of this face, for the nodal values (D-terms, mixed flux)
        const bool hasL = fa - 1 >= 0, hasR = fa <= n - 1;
        const long long cL = d == 0 ? (long long)line * g.nx + (fa - 1) : (long long)(fa - 1) * g.nx + line;
        const long long cR = d == 0 ? (long long)line * g.nx + fa : (long long)fa * g.nx + line;
        // the transposed D-term and mixed-flux coefficients of position q, with the 1/h of the flux
        // adjoints folded in (only the outer positions carry h in Eq. Cd-1)
        const double s1 = (q == 0 || q == 3) ? cf_ih : -cf_ih;
        const double sdh = q == 0 ? ef_ih : (q == 1 ? -eg_ih : (q == 2 ? eg_ih : -ef_ih));
        const double mq = (q == 1 || q == 2) ? m7_ih : m1_ih;
#pragma unroll
        for (int k = 0; k < NC; ++k) {
          auto dmu = [&](int fld) {
            const double r = hasR ? muL[(fld * NC + k) * plane + HW_IDX(cR, plane)] : 0.0;
            const double l = hasL ? muL[(fld * NC + k) * plane + HW_IDX(cL, plane)] : 0.0;
            return fu.sub(r, l);
          };
          // a mirrored alias takes the nodal sign tables: f and the mixed value flip except for the
          // normal momentum, h only for it (sign flips in the integer pipe)
          const bool flip_f = mir && k != km, flip_h = mir && k == km;
          const double nfh = dmu(0), nhh = dmu(fown);
          nf[k] = fma(s1, neg_if(nfh, flip_f), fma(sdh, neg_if(nhh, flip_f), nf[k]));
          if (q == 0 || q == 3)
            nh[k] = fma(q == 0 ? ch_ih : -ch_ih, neg_if(nfh, flip_h), fma(eh_ih, neg_if(nhh, flip_h), nh[k]));
          if (DIM == 2) no[k] = fma(mq, neg_if(dmu(foth), flip_f), no[k]);
        }
      }
      // modified derivatives of cells c = x + 1 - q hold this cell at stencil position q
#pragma unroll
      for (int q = 0; q < 3; ++q) {
        const int c = x + 1 - q;
        if (c < 0 || c > n - 1) continue;
        const long long pcl = HW_IDX(d == 0 ? (long long)j * g.nx + c : (long long)c * g.nx + i, plane);
        const double* cm = aw.CM + ((long long)d * plane + pcl) * 5 * NC;
#pragma unroll
        for (int k = 0; k < NC; ++k) lb[0][k] = fu.add(lb[0][k], cm[q * NC + k]);
        if (q == 0) {
#pragma unroll
          for (int k = 0; k < NC; ++k) lb[fown][k] = fu.add(lb[fown][k], cm[3 * NC + k]);
        } else if (q == 2) {
#pragma unroll
          for (int k = 0; k < NC; ++k) lb[fown][k] = fu.add(lb[fown][k], cm[4 * NC + k]);
        }
      }
    }
    // nodal VJPs at this cell (normal frame): f(U), A(U) D_own, A(U) D_other
    double Un[NC], Dn[NC], On[NC], Ub[NC], Db[NC], Ob[NC];
#pragma unroll
    for (int k = 0; k < NC; ++k) {
      Un[k] = U[k];
      Dn[k] = V[fown - 1][k];
      On[k] = DIM == 2 ? V[foth - 1][k] : 0.0;
      Ub[k] = Db[k] = Ob[k] = 0.0;
    }
    if (d == 1) {
      swap_frame<NC>(Un);
      swap_frame<NC>(Dn);
      swap_frame<NC>(On);
      swap_frame<NC>(nf);
      swap_frame<NC>(nh);
      swap_frame<NC>(no);
    }
    // the cell's primitives in the direction's frame (the velocities exchanged in y), shared by
    // the three nodal backward passes and computed once for both directions
    Prim<NC> qn = qc;
    if (d == 1) {
      qn.u = qc.v;
      qn.v = qc.u;
    }
    flux_bwd<NC>(Un, qn, g.gm1, nf, Ub, fu);
    jvp_bwd<NC>(Un, qn, Dn, g.gm1, nh, Ub, Db, fu);
    if (DIM == 2) jvp_bwd<NC>(Un, qn, On, g.gm1, no, Ub, Ob, fu);
    if (d == 1) {
      swap_frame<NC>(Ub);
      swap_frame<NC>(Db);
      swap_frame<NC>(Ob);
    }
#pragma unroll
    for (int k = 0; k < NC; ++k) {
      lb[0][k] = fu.add(lb[0][k], Ub[k]);
      lb[fown][k] = fu.add(lb[fown][k], Db[k]);
      if (DIM == 2) lb[foth][k] = fu.add(lb[foth][k], Ob[k]);
    }
  }
#pragma unroll
  for (int f = 0; f < NF; ++f)
#pragma unroll
    for (int k = 0; k < NC; ++k) lam[(f * NC + k) * plane + p] = lb[f][k];
}

// The transposes of the Runge-Kutta combinations of Eq. (2Dfully-hweno), value by value, one pass
// each (every array has n values):
//   k_rk_seed:  muM = c1 x, muL = c2 x                       (the last stage's seeds from lam_in)
//   k_rk_mid:   lamB = c0 y + c1 x, muM = c2 x, muL = c3 x    (x = the last stage's VJP, y = lam_in)
//   k_rk_first: muM = x + y, muL = c3 x                       (x = the middle stage's VJP, y = lamB)
__global__ void k_rk_seed(long long n, double* __restrict__ muM, double* __restrict__ muL, double c1, double c2,
                          const double* __restrict__ x) {
  const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const double v = x[i];
  muM[i] = c1 * v;
  muL[i] = c2 * v;
}
__global__ void k_rk_mid(long long n, double* __restrict__ lamB, double* __restrict__ muM, double* __restrict__ muL,
                         double c0, double c1, double c2, double c3, const double* __restrict__ x,
                         const double* __restrict__ y) {
  const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const double v = x[i];
  lamB[i] = fma(c0, y[i], c1 * v);
  muM[i] = c2 * v;
  muL[i] = c3 * v;
}
__global__ void k_rk_first(long long n, double* __restrict__ muM, double* __restrict__ muL, double c3,
                           const double* __restrict__ x, const double* __restrict__ y) {
  const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const double v = x[i];
  muM[i] = v + y[i];
  muL[i] = c3 * v;
}

}  // namespace hw

namespace hwh {
unsigned int bounds_take_adjoint(int* line) {
#ifdef HWENO_BOUNDS_CHECK
  return hw::bounds_take(line);
#else
  if (line) *line = 0;
  return 0;
#endif
}
}  // namespace hwh

namespace {

struct AdjLayout {
  size_t S1, S2, lam2, lam1, lamB, muM, muL, CU, CD, CM, lists, total;
};

AdjLayout adj_layout(const hweno_ctx* h) {
  const size_t nst = hweno_state_doubles(h) * 8;
  const size_t nc = nc_of(h);
  const size_t nfx = (size_t)(h->nx + 1) * h->ny, nfy = h->dim == 2 ? (size_t)(h->ny + 1) * h->nx : 0;
  AdjLayout l;
  l.S1 = l.S2 = l.lam2 = l.lam1 = l.lamB = l.muM = l.muL = align_up(nst);
  l.CU = l.CD = align_up((nfx + nfy) * 4 * nc * 8);
  l.CM = align_up((size_t)h->dim * h->nx * h->ny * 5 * nc * 8);
  // the counts, then the lists of cells (two directions each) and faces
  l.lists = h->dim == 2 ? align_up((64 + 2 * (size_t)h->nx * h->ny + nfx + nfy) * sizeof(unsigned int)) : 0;
  l.total = 7 * l.S1 + l.CU + l.CD + l.CM + l.lists;
  return l;
}

struct AdjPtrs {
  double *S1, *S2, *lam2, *lam1, *lamB, *muM, *muL;
  hw::AdjWork aw;
};

AdjPtrs adj_ptrs(const hweno_ctx* h, void* ws) {
  const AdjLayout l = adj_layout(h);
  unsigned char* p = static_cast<unsigned char*>(ws);
  AdjPtrs a;
  double** arr[7] = {&a.S1, &a.S2, &a.lam2, &a.lam1, &a.lamB, &a.muM, &a.muL};
  for (int k = 0; k < 7; ++k) {
    *arr[k] = reinterpret_cast<double*>(p);
    p += l.S1;
  }
  a.aw.CU = reinterpret_cast<double*>(p);
  p += l.CU;
  a.aw.CD = reinterpret_cast<double*>(p);
  p += l.CD;
  a.aw.CM = reinterpret_cast<double*>(p);
  p += l.CM;
  a.aw.count = reinterpret_cast<unsigned int*>(p);
  a.aw.cells = a.aw.count + 64;
  a.aw.faces = a.aw.cells + 2 * h->nx * h->ny;
  a.aw.scal = h->w.scal;
  return a;
}

// From this many cells on a 2D grid's VJP takes the pairs: below it there is at most one warp of faces to a
// scheduler, whose FP64 pipe waits for that warp's chain of instructions, the longer one in pairs, and the
// kernels of the lists find little or nothing to do.  One step forward and back at 46x146 1.23 ms in FP64,
// 1.50 in pairs; at 128^2 1.49 and 1.51, at 160^2 1.96 and 1.64.
constexpr long long kAdjPairMinCells = hw::kSMs * 4LL * 32 / 2;

template <int DIM>
int stage_vjp(hweno_ctx* h, const Grid& g, const double* S, const double* alpha2, const double* muM,
              const double* muL, const hw::AdjWork& aw, double* lam) {
  const cudaStream_t st = h->stream;
  const unsigned bc = blocks_for(g.plane);
  // the FP64 kernels' shared memory for the saved forward intermediates: one slot per thread and value
  constexpr int NC = DIM == 1 ? 3 : 4;
  constexpr size_t cell_sm = (size_t)hw::kCellSaved * NC * hw::kThreads * sizeof(double);
  constexpr size_t face_sm = (size_t)hw::kFaceSaved * NC * hw::kThreads * sizeof(double);
  if (cudaFuncSetAttribute(hw::k_adj_face<DIM>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)face_sm) !=
          cudaSuccess ||
      cudaFuncSetAttribute(hw::k_adj_cell<DIM>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)cell_sm) !=
          cudaSuccess)
    return HWENO_ECUDA;
  const long long nfx = (long long)(g.nx + 1) * g.ny;
  const long long nfy = DIM == 2 ? (long long)(g.ny + 1) * g.nx : 0;
  const unsigned bf = blocks_for(nfx > nfy ? nfx : nfy);
  if (DIM == 1) {
    hw::k_adj_cell<1><<<bc, hw::kThreads, cell_sm, st>>>(g, S, muM, aw);
    hw::k_adj_face<1><<<bf, hw::kThreads, face_sm, st>>>(g, S, muL, aw, alpha2);
  } else {
    // most of the work in pairs, the rest (listed on the way) in FP64: two blocks per SM take it in turn
    const unsigned bl = 2u * hw::kSMs;
    constexpr size_t pair_sm = (size_t)hw::kPairSlots * hw::kThreads * sizeof(ulonglong2);
    const auto face_pair = g.pg.ig1[0] >= hw::kSmall32 ? hw::k_adj_face_pair<true> : hw::k_adj_face_pair<false>;
    if (cudaFuncSetAttribute(face_pair, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)pair_sm) !=
            cudaSuccess ||
        cudaFuncSetAttribute(hw::k_adj_cell_pair, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)pair_sm) !=
            cudaSuccess)
      return HWENO_ECUDA;
    hw::AdjWork fw = aw;
    if (g.plane >= kAdjPairMinCells && pair_mesh(h)) {
      if (cudaMemsetAsync(aw.count, 0, 2 * sizeof(unsigned int), st) != cudaSuccess) return HWENO_ECUDA;
      hw::k_adj_cell_pair<<<bc, hw::kThreads, pair_sm, st>>>(g, S, muM, aw);
      face_pair<<<dim3(bf, 2), hw::kThreads, pair_sm, st>>>(g, S, muL, aw, alpha2);
      h->launches += 2;
    } else {
      fw.cells = fw.faces = nullptr;
    }
    hw::k_adj_cell<DIM><<<bl < 2 * bc ? bl : 2 * bc, hw::kThreads, cell_sm, st>>>(g, S, muM, fw);
    hw::k_adj_face<DIM><<<bl < 2 * bf ? bl : 2 * bf, hw::kThreads, face_sm, st>>>(g, S, muL, fw, alpha2);
  }
  hw::k_adj_gather<DIM><<<bc, hw::kThreads, 0, st>>>(g, S, muM, muL, aw, lam);
  h->launches += 3;
  return cudaGetLastError() == cudaSuccess ? HWENO_OK : HWENO_ECUDA;
}

unsigned rk_blocks(const hweno_ctx* h) { return (unsigned)((hweno_state_doubles(h) + 255) / 256); }
long long rk_n(const hweno_ctx* h) { return (long long)hweno_state_doubles(h); }
int launch_status() { return cudaGetLastError() == cudaSuccess ? HWENO_OK : HWENO_ECUDA; }

}  // namespace

extern "C" size_t hweno_adjoint_workspace_bytes(const hweno_t* h) { return h ? adj_layout(h).total : 0; }

namespace {

// the three stage VJPs of one step, given the stage inputs S^n, S1, S2
int adjoint_from_stages(hweno_t* h, const AdjPtrs& a, const double* Sn, const double* S1, const double* S2, double dt,
                        const double* alpha6, const double* lam_in, double* lam_out) {
  const Grid g = grid_of(h);
  int rc;
  auto vjp = [&](const double* S, int st, const double* muM, const double* muL, double* lam) {
    return h->dim == 1 ? stage_vjp<1>(h, g, S, alpha6 + 2 * st, muM, muL, a.aw, lam)
                       : stage_vjp<2>(h, g, S, alpha6 + 2 * st, muM, muL, a.aw, lam);
  };
  // S^{n+1} = 1/3 B + 2/3 (M(S2) + dt L(S2)):  muM = 2/3 lam_in, muL = 2/3 dt lam_in
  hw::k_rk_seed<<<rk_blocks(h), 256, 0, h->stream>>>(rk_n(h), a.muM, a.muL, 2.0 / 3.0, 2.0 / 3.0 * dt, lam_in);
  if ((rc = launch_status())) return rc;
  if ((rc = vjp(S2, 2, a.muM, a.muL, a.lam2))) return rc;
  // S2 = 3/4 B + 1/4 (M(S1) + dt L(S1)):  lamB = 1/3 lam_in + 3/4 lam2, muM = 1/4 lam2, muL = 1/4 dt lam2
  hw::k_rk_mid<<<rk_blocks(h), 256, 0, h->stream>>>(rk_n(h), a.lamB, a.muM, a.muL, 1.0 / 3.0, 0.75, 0.25, 0.25 * dt,
                                                    a.lam2, lam_in);
  if ((rc = launch_status())) return rc;
  if ((rc = vjp(S1, 1, a.muM, a.muL, a.lam1))) return rc;
  // S1 = M(S^n) + dt L(S^n), B = M(S^n):  muM = lam1 + lamB, muL = dt lam1
  hw::k_rk_first<<<rk_blocks(h), 256, 0, h->stream>>>(rk_n(h), a.muM, a.muL, dt, a.lam1, a.lamB);
  if ((rc = launch_status())) return rc;
  if ((rc = vjp(Sn, 0, a.muM, a.muL, lam_out))) return rc;
  h->launches += 3;
  return HWENO_OK;
}

}  // namespace

extern "C" {

int hweno_adjoint_step(hweno_t* h, const double* Sn, double dt, const double* alpha6, const double* lam_in,
                       double* lam_out, void* adj_ws) {
  if (!h || !Sn || !alpha6 || !lam_in || !lam_out || !adj_ws) return HWENO_EINVAL;
  if (h->system != HWENO_EULER || h->var != 0) return HWENO_EINVAL;
  if (!(dt > 0.0) || ((uintptr_t)adj_ws & 255)) return HWENO_EINVAL;
  if (!h->ws) return HWENO_ESTATE;
  const AdjPtrs a = adj_ptrs(h, adj_ws);
  const size_t bytes = hweno_state_doubles(h) * 8;
  // forward stages 1 and 2 from S^n with the recorded alphas (the forward workspace is scratch)
  if (cudaMemcpyAsync(a.S1, Sn, bytes, cudaMemcpyDeviceToDevice, h->stream) != cudaSuccess) return HWENO_ECUDA;
  int rc = stage_replay(h, a.S1, 0, dt, alpha6);
  if (rc) return rc;
  if (cudaMemcpyAsync(a.S2, a.S1, bytes, cudaMemcpyDeviceToDevice, h->stream) != cudaSuccess) return HWENO_ECUDA;
  rc = stage_replay(h, a.S2, 1, dt, alpha6 + 2);
  if (rc) return rc;
  return adjoint_from_stages(h, a, Sn, a.S1, a.S2, dt, alpha6, lam_in, lam_out);
}

int hweno_adjoint_step_stages(hweno_t* h, const double* Sn, const double* S1, const double* S2, double dt,
                              const double* alpha6, const double* lam_in, double* lam_out, void* adj_ws) {
  if (!h || !Sn || !S1 || !S2 || !alpha6 || !lam_in || !lam_out || !adj_ws) return HWENO_EINVAL;
  if (h->system != HWENO_EULER || h->var != 0) return HWENO_EINVAL;
  if (!(dt > 0.0) || ((uintptr_t)adj_ws & 255)) return HWENO_EINVAL;
  if (!h->ws) return HWENO_ESTATE;  // the kernels read the bound workspace's scalars
  return adjoint_from_stages(h, adj_ptrs(h, adj_ws), Sn, S1, S2, dt, alpha6, lam_in, lam_out);
}

int hweno_step_replay_stages(hweno_t* h, double dt, const double* alpha6, double* S1_out, double* S2_out) {
  if (!h || !alpha6 || !S1_out || !S2_out || !(dt > 0.0)) return HWENO_EINVAL;
  if (!h->ws || !h->state) return HWENO_ESTATE;
  const size_t bytes = hweno_state_doubles(h) * 8;
  for (int st = 0; st < 3; ++st) {
    int rc = stage(h, h->state, h->state, 0, st, dt, st, nullptr, nullptr, alpha6 + 2 * st);
    if (rc) return rc;
    if (st < 2 && cudaMemcpyAsync(st == 0 ? S1_out : S2_out, h->state, bytes, cudaMemcpyDeviceToDevice,
                                  h->stream) != cudaSuccess)
      return HWENO_ECUDA;
  }
  return HWENO_OK;
}

int hweno_step_stages(hweno_t* h, double dt, double* S1_out, double* S2_out) {
  if (!h || !S1_out || !S2_out || !std::isfinite(dt)) return HWENO_EINVAL;
  if (!h->ws || !h->state) return HWENO_ESTATE;
  if (((uintptr_t)S1_out & 15) || ((uintptr_t)S2_out & 15)) return HWENO_EINVAL;
  const size_t bytes = hweno_state_doubles(h) * 8;
  for (int st = 0; st < 3; ++st) {
    int rc = stage(h, h->state, h->state, 0, st, dt, st, nullptr, nullptr);
    if (rc) return rc;
    if (st < 2 && cudaMemcpyAsync(st == 0 ? S1_out : S2_out, h->state, bytes, cudaMemcpyDeviceToDevice,
                                  h->stream) != cudaSuccess)
      return HWENO_ECUDA;
  }
  return HWENO_OK;
}

int hweno_step_replay(hweno_t* h, double dt, const double* alpha6) {
  if (!h || !alpha6 || !(dt > 0.0)) return HWENO_EINVAL;
  if (!h->ws || !h->state) return HWENO_ESTATE;
  for (int st = 0; st < 3; ++st) {
    int rc = stage(h, h->state, h->state, 0, st, dt, st, nullptr, nullptr, alpha6 + 2 * st);
    if (rc) return rc;
  }
  return HWENO_OK;
}

int hweno_step_record(hweno_t* h, double* rec7) {
  if (!h || !rec7) return HWENO_EINVAL;
  if (!h->ws) return HWENO_ESTATE;
  // dt of the last step, then the wavespeed slots of its three stages (bit patterns of doubles)
  if (cudaMemcpyAsync(rec7, h->w.scal, sizeof(double), cudaMemcpyDeviceToDevice, h->stream) != cudaSuccess ||
      cudaMemcpyAsync(rec7 + 1, h->w.alpha, 6 * sizeof(double), cudaMemcpyDeviceToDevice, h->stream) != cudaSuccess)
    return HWENO_ECUDA;
  return HWENO_OK;
}

int hweno_stage_vjp(hweno_t* h, const double* S, const double* alpha2, const double* muM, const double* muL,
                    double* lam, void* adj_ws) {
  if (!h || !S || !alpha2 || !muM || !muL || !lam || !adj_ws) return HWENO_EINVAL;
  if (h->system != HWENO_EULER || h->var != 0) return HWENO_EINVAL;
  if ((uintptr_t)adj_ws & 255) return HWENO_EINVAL;
  if (!h->ws) return HWENO_ESTATE;
  const AdjPtrs a = adj_ptrs(h, adj_ws);
  const Grid g = grid_of(h);
  return h->dim == 1 ? stage_vjp<1>(h, g, S, alpha2, muM, muL, a.aw, lam)
                     : stage_vjp<2>(h, g, S, alpha2, muM, muL, a.aw, lam);
}

}  // extern "C"
