// Stage kernels of the HWENO-I scheme (Xie, Tao, Jiao, Zhang, arXiv 2411.11229) for sm_103a.
//
// One Runge-Kutta stage is three launches over the grid, and on 2D grids from 2^15 cells a fourth (k_left)
// for the cells and faces whose nonlinear part needs the FP64 weights:
//   k_cell   per cell : wavespeed (LF alpha of the stage input), nodal fluxes f, h = f'(u) v (and
//                       the mixed-flux nodal values in 2D) for the D-terms (Eqs. Cd-1, DfDh, mixed),
//                       Euler primitives for the Roe averages, and the modified derivative v~
//                       (Eq. limiter) in the local characteristic fields of the cell.
//   k_face   per face : characteristic projection with the Roe-averaged eigenvectors, the HWENO
//                       interpolation of u and v to both sides of the face (Eqs. Pxi, P'xi, GHYZ,
//                       nonlinear, interp), back projection, and the numerical fluxes
//                       (Eqs. flux-1d, flux-LF, DfDh, mixed).
//   k_update per cell : conservative differences (Eqs. odeH / ode2H) and the SSP-RK3 combination
//                       with the modified derivative in the base (Eqs. fully-hweno, 2Dfully-hweno),
//                       in place; or L and M written out (rhs mode).
// The path is bound by the FP64 pipe (a few thousand FP64 operations per cell and stage against
// roughly a kilobyte of traffic), so the split keeps every warp's lanes busy on one kind of work
// and exchanges intermediates through L2/HBM, which has bandwidth to spare.
//
// VAR selects the scheme: 0 is the scheme of the paper with one boundary type on every side;
// 1 adds the runtime options (per-side boundary types with fixed-state sides, v^+/- with the
// nonlinear weights, the D-terms of Eq. Cd-2, the gravity source of Eq. euler2d-s); 2 is 1 with
// the per-cell characteristic decomposition (R2): k_cell interpolates both faces of every cell in
// the cell's own characteristic fields and k_face only forms the fluxes; k_r2_ghost supplies the
// face states of the ghost cells at the ends of every line.
#pragma once
#include "hweno_math.cuh"
#include "hweno_pair.cuh"

namespace hw {

// Device views into the caller's workspace.
struct Work {
  double* B;     // stage base M(S^n): [NF][NC][plane]
  double* MD;    // modified derivatives (V~, W~): [DIM][NC][plane]
  double* NOD;   // nodal values per direction, normal frame: [DIM][NG][NC][plane]
  float2* PRIM;  // Euler primitives (sqrt(rho), u[, v], H): [NP][plane], as pairs (hweno_pair.cuh) where the
                 // faces take pairs (Grid::face_pairs), else in FP64 in the same bytes
  double* FX;    // x-face fluxes, original frame: [NF][NC][ny][nx+1]
  double* FY;    // y-face fluxes: [NF][NC][ny+1][nx]
  unsigned long long* alpha;  // wavespeed slots (bit patterns of non-negative doubles): slot s of
                              // direction d at alpha[s * astride + d]
  double* scal;               // [0] dt of the current step, [1] t, [2] t_end, [3] steps taken,
                              // [4..7] zero (read by fu_of; never written after creation)
  unsigned int* status;       // [0] bit 0: non-physical state met; [2], [3] entries in left_cells and
                              // left_faces (zero between stages)
  long long astride;          // distance between slots (2 for a single grid)
  // R2 only: face states of every cell, normal frame:
  // FS [DIM][4][NC][plane] = (u^- and v^- at the right face, u^+ and v^+ at the left face);
  // GFS [DIM][2 ends][2][NC][gstride] = the low ghost's right-face and the high ghost's
  // left-face states of every line.
  double* FS;
  double* GFS;
  long long gstride;
  // local LF coefficients only: the spectral radius of every cell per direction [DIM][plane]
  double* WS;
  // listed grids only: cell * 2 + direction of the cells, x faces then y faces of the faces, that k_cell
  // and k_face leave to k_left
  unsigned int *left_cells, *left_faces;
};


// The units of FU in thread registers: a zero read at a per-thread address of the zeroed slots
// scal[4..7], so that the compiler can neither fold it nor keep it in a uniform register.
__device__ __forceinline__ FU fu_of(const double* scal) {
  const double z = scal[4 + (threadIdx.x & 3)];
  return FU{1.0 + z, -z, __double2hiint(z)};
}

template <int NC>
__device__ __forceinline__ void swap_frame(double* q) {
  if (NC == 4) {
    const double t = q[1];
    q[1] = q[2];
    q[2] = t;
  }
}

// The bit pattern of a wavespeed (non-negative, so its order is the numbers'), 0 for a NaN
__device__ __forceinline__ unsigned long long speed_bits(double x) {
  const unsigned long long b = dbl_bits(x);
  return b <= 0x7ff0000000000000ull ? b : 0ull;
}
__device__ __forceinline__ unsigned long long warp_max(unsigned long long b) {
  const unsigned int hi = __reduce_max_sync(0xffffffffu, (unsigned int)(b >> 32));
  const unsigned int lo = __reduce_max_sync(0xffffffffu, (unsigned int)(b >> 32) == hi ? (unsigned int)b : 0u);
  return ((unsigned long long)hi << 32) | lo;
}
// max over the block of the wavespeeds (a, b), then one atomicMax per block, all on the bit patterns
// (a maximum of FP64 numbers is an instruction of the FP64 pipe)
__device__ __forceinline__ void block_max2(double a, double b, unsigned long long* dst) {
  __shared__ unsigned long long sm[2][32];
  unsigned long long x = warp_max(speed_bits(a)), y = warp_max(speed_bits(b));
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  if (lane == 0) {
    sm[0][wid] = x;
    sm[1][wid] = y;
  }
  __syncthreads();
  if (wid == 0) {
    const int nw = blockDim.x >> 5;
    x = warp_max(lane < nw ? sm[0][lane] : 0ull);
    y = warp_max(lane < nw ? sm[1][lane] : 0ull);
    if (lane == 0) {
      atomicMax(dst, x);
      atomicMax(dst + 1, y);
    }
  }
}
// whether x is a finite number, and whether it is greater than zero, in the integer pipe
__device__ __forceinline__ bool finite_bits(double x) { return (__double2hiint(x) & 0x7ff00000) != 0x7ff00000; }
__device__ __forceinline__ bool positive_bits(double x) {
  const unsigned long long b = dbl_bits(x);
  return b - 1ull < 0x7ff0000000000000ull;
}

// ---------------------------------------------------------------------------------------------
// Modified derivative of one cell in one direction (normal frame).  U3/D3: cells i-1, i, i+1
// (D = derivative along the sweep; only i-1 and i+1 enter).  e: eigenvectors of the cell.  The
// limiter needs the characteristic fields only through the differences of neighbouring cells, so
// the two conserved differences are projected (equal neighbours give exactly zero).
template <int NC, int SYS>
__device__ __forceinline__ void modified_derivative(const double (&U3)[3][NC], const double (&D3)[3][NC],
                                                    const Eig<NC>& e, int dir, const Grid& g, double* out,
                                                    const FU& f) {
  double dU[2][NC], Dq[2][NC], Zm[NC], Zp[NC];
#pragma unroll
  for (int q = 0; q < 2; ++q)
#pragma unroll
    for (int k = 0; k < NC; ++k) dU[q][k] = f.sub(U3[q + 1][k], U3[q][k]);
  if (SYS == SYS_EULER) {
    e.project(dU[0], Dq[0], f);
    e.project(dU[1], Dq[1], f);
    e.project(D3[0], Zm, f);
    e.project(D3[2], Zp, f);
  } else {
    Dq[0][0] = dU[0][0];
    Dq[1][0] = dU[1][0];
    Zm[0] = D3[0][0];
    Zp[0] = D3[2][0];
  }
  double ht[NC];
  const StencilK k = stencil_k(g, dir, f);
#pragma unroll
  for (int s = 0; s < NC; ++s) ht[s] = f.mul(cell_field_d(Dq[0][s], Dq[1][s], Zm[s], Zp[s], k, f), k.ih);
  if (SYS == SYS_EULER) {
    e.back(ht, out, f);
  } else {
    out[0] = ht[0];
  }
}

// The ghost cell of a fixed-state side: the side's state (normal frame), zero derivatives.
template <int NC, int SYS>
__device__ __forceinline__ void load_fixed(const Grid& g, int side, int dir, double* U, double* D) {
#pragma unroll
  for (int k = 0; k < NC; ++k) {
    U[k] = g.fixU[side][k];
    D[k] = 0.0;
  }
  if (SYS == SYS_EULER && dir == 1) swap_frame<NC>(U);
}

// The three cells i-1, i, i+1 of cell (i, j) along direction d, through the boundary map (normal
// frame, mirrored or fixed where the map says so).  U3[1] is taken from Uc (already loaded).
template <int DIM, int SYS, int VAR, int NC>
__device__ __forceinline__ void load_stencil3(const Grid& g, const double* __restrict__ S, int d, int i, int j,
                                              int a0, const double* Uc, double (&U3)[3][NC], double (&D3)[3][NC]) {
  const long long plane = g.plane;
  const int n = d == 0 ? g.nx : g.ny;
  const int fld = d == 0 ? 1 : 2;
#pragma unroll
  for (int q = 0; q < 3; ++q) {
    bool refl, fixed = false;
    const int ac = VAR ? bc_map_ext(a0 - 1 + q, n, g.side[2 * d], g.side[2 * d + 1], refl, fixed)
                       : bc_map(a0 - 1 + q, n, g.bc, refl);
    const long long pc = HW_IDX(d == 0 ? (long long)j * g.nx + ac : (long long)ac * g.nx + i, plane);
#pragma unroll
    for (int k = 0; k < NC; ++k) {
      U3[q][k] = (q == 1 && Uc) ? Uc[k] : S[k * plane + pc];
      D3[q][k] = S[(fld * NC + k) * plane + pc];
    }
    if (SYS == SYS_EULER && d == 1) {
      swap_frame<NC>(U3[q]);
      swap_frame<NC>(D3[q]);
    }
    if (SYS == SYS_EULER) {
      mirror_U<NC>(U3[q], refl);
      mirror_D<NC>(D3[q], refl);
    }
    if (VAR && fixed) load_fixed<NC, SYS>(g, 2 * d + (a0 - 1 + q < 0 ? 0 : 1), d, U3[q], D3[q]);
  }
}

// R2: the modified derivative and the face states of one cell in one direction from its own
// stencil in its own characteristic fields (normal frame, derivatives unscaled).  The face values
// are the cell's state plus back-projected corrections; without the weighted-derivative option the
// face derivatives are linear in the stencil and are formed in conserved variables.
template <int NC, int SYS, bool VW>
__device__ __forceinline__ void r2_cell_vw(const double (&U3)[3][NC], const double (&D3)[3][NC], const Eig<NC>& e,
                                           int dir, const Grid& g, double* md, double (&fs)[4][NC], const FU& f) {
  double dU[2][NC], Dq[2][NC], Zm[NC], Zp[NC];
#pragma unroll
  for (int q = 0; q < 2; ++q)
#pragma unroll
    for (int k = 0; k < NC; ++k) dU[q][k] = f.sub(U3[q + 1][k], U3[q][k]);
  if (!VW) {
    // the Hermite derivative of Eq. (P'xi) at the two faces (linear in the stencil)
    const double k21 = g.uvd[dir][0], k3 = g.uvd[dir][1];
#pragma unroll
    for (int k = 0; k < NC; ++k) {
      fs[1][k] = fma(k21, dU[1][k], fma(-k3, dU[0][k], fma(0.0625, D3[0][k], -0.1875 * D3[2][k])));
      fs[3][k] = fma(k21, dU[0][k], fma(-k3, dU[1][k], fma(-0.1875, D3[0][k], 0.0625 * D3[2][k])));
    }
  }
  if (SYS == SYS_EULER) {
    e.project(dU[0], Dq[0], f);
    e.project(dU[1], Dq[1], f);
    e.project(D3[0], Zm, f);
    e.project(D3[2], Zp, f);
  } else {
    Dq[0][0] = dU[0][0];
    Dq[1][0] = dU[1][0];
    Zm[0] = D3[0][0];
    Zp[0] = D3[2][0];
  }
  const double bc = SYS == SYS_EULER ? 0.0 : U3[1][0];
  const StencilK k = stencil_k(g, dir, f);
  double cm[NC], chm[NC], cp[NC], chp[NC], ht[NC];
#pragma unroll
  for (int s = 0; s < NC; ++s) {
    cell_faces_field<VW>(Dq[0][s], Dq[1][s], Zm[s], Zp[s], bc, k, g, dir, cm[s], chm[s], cp[s], chp[s], ht[s], f);
    ht[s] = f.mul(ht[s], k.ih);
  }
  if (SYS == SYS_EULER) {
    e.back_add(cm, U3[1], fs[0], f);
    e.back_add(cp, U3[1], fs[2], f);
    e.back(ht, md, f);
  } else {
    fs[0][0] = cm[0];
    fs[2][0] = cp[0];
    md[0] = ht[0];
  }
  if (VW) {
    if (SYS == SYS_EULER) {
      e.back(chm, fs[1], f);
      e.back(chp, fs[3], f);
    } else {
      fs[1][0] = chm[0];
      fs[3][0] = chp[0];
    }
  }
}

// r2_cell_vw with the weighted-derivative option read from the grid's flags (one code path each)
template <int NC, int SYS>
__device__ __forceinline__ void r2_cell(const double (&U3)[3][NC], const double (&D3)[3][NC], const Eig<NC>& e,
                                        int dir, const Grid& g, double* md, double (&fs)[4][NC], const FU& f) {
  if (g.flags & FLAG_V_WEIGHTED)
    r2_cell_vw<NC, SYS, true>(U3, D3, e, dir, g, md, fs, f);
  else
    r2_cell_vw<NC, SYS, false>(U3, D3, e, dir, g, md, fs, f);
}

// Velocities, pressure, 1/rho of a cell, and its wavespeeds per direction; ROOT: 1/c as well (the FP64
// weights' fields need both, and one chain of instructions gives both; in 1D, whose steps in one launch
// give the two to different warps, they are apart: 849 us against 856 for ten steps of 16383 cells)
template <int DIM, int SYS, bool ROOT>
struct CellState {
  double u = 0.0, v = 0.0, pr = 0.0, ir = 0.0, c = 0.0, ic = 0.0;
  __device__ __forceinline__ bool speeds(double& wsx, double& wsy, const FU& f) const {
    wsx = f.add(fabs(u), c);
    wsy = DIM == 2 ? f.add(fabs(v), c) : 0.0;
    return finite_bits(wsx) && finite_bits(wsy);
  }
  // returns whether the state is physical
  __device__ __forceinline__ bool set(const double* U, const Grid& g, const FU& f, double& wsx, double& wsy) {
    constexpr int NC = Traits<DIM, SYS>::NC;
    if (SYS == SYS_EULER) {
      ir = rcp(U[0], f);
      u = f.mul(U[1], ir);
      if (DIM == 2) v = f.mul(U[2], ir);
      const double ke = DIM == 2 ? fma(U[1], u, f.mul(U[2], v)) : f.mul(U[1], u);
      pr = g.gm1 * fma(-0.5, ke, U[NC - 1]);
      const double c2 = f.mul(g.gamma * pr, ir);
      if (ROOT) ic = rsqrt_fast(c2, f);
      c = ROOT ? f.mul(c2, ic) : sqrt_fast(c2, f);
      bool ok = speeds(wsx, wsy, f) && positive_bits(U[0]) && positive_bits(pr);
      if (!ok && denormal_bits(c2)) {  // off the usual way: the other cells do not pay for it
        if (ROOT) ic = rsqrt_full(c2, f);
        c = sqrt_full(c2, f);
        ok = speeds(wsx, wsy, f) && positive_bits(U[0]) && positive_bits(pr);
      }
      return ok;
    }
    if (SYS == SYS_BURGERS) {
      wsx = fabs(U[0]);
      wsy = DIM == 2 ? wsx : 0.0;
      return finite_bits(wsx);
    }
    wsx = fabs(g.ax);
    wsy = DIM == 2 ? fabs(g.ay) : 0.0;
    return true;
  }
};

// The modified derivative of cell p in direction d (and, for R2, the cell's face states) with the FP64
// weights, from the cell's state U and what CellState holds of it.
template <int DIM, int SYS, int VAR>
__device__ __forceinline__ void cell_limiter_of(const Grid& g, const double* __restrict__ S, const Work& w, long long p,
                                                int i, int j, int d, const double* U,
                                                const CellState<DIM, SYS, DIM == 2>& c,
                                                const FU& f) {
  constexpr int NC = Traits<DIM, SYS>::NC;
  const long long plane = g.plane;
  double U3[3][NC], D3[3][NC];
  load_stencil3<DIM, SYS, VAR, NC>(g, S, d, i, j, d == 0 ? i : j, U, U3, D3);
  Eig<NC> e;
  if (SYS == SYS_EULER) {
    double cc = c.c, ic = c.ic;
    if (DIM == 1) {
      const double c2 = f.mul(g.gamma * c.pr, c.ir);
      ic = rsqrt_full(c2, f);
      cc = f.mul(c2, ic);
    }
    e.setup(d == 0 ? c.u : c.v, d == 0 ? c.v : c.u, f.mul(f.add(U[NC - 1], c.pr), c.ir), cc, ic, g.gm1);
  }
  double out[NC];
  if (VAR == 2) {
    double fs[4][NC];
    r2_cell<NC, SYS>(U3, D3, e, d, g, out, fs, f);
    double* FSd = w.FS + (long long)d * 4 * NC * plane;
#pragma unroll
    for (int q = 0; q < 4; ++q)
#pragma unroll
      for (int k = 0; k < NC; ++k) FSd[(q * NC + k) * plane + p] = fs[q][k];
  } else {
    modified_derivative<NC, SYS>(U3, D3, e, d, g, out, f);
  }
  if (SYS == SYS_EULER && d == 1) swap_frame<NC>(out);
#pragma unroll
  for (int k = 0; k < NC; ++k) w.MD[((long long)d * NC + k) * plane + p] = out[k];
}

// The same from the cell alone: the cells that the pairs leave to the FP64 weights.
template <int DIM, int SYS, int VAR>
__device__ __forceinline__ void cell_limiter(const Grid& g, const double* __restrict__ S, const Work& w, long long p,
                                             int d) {
  constexpr int NC = Traits<DIM, SYS>::NC;
  const FU f = fu_of(w.scal);
  double U[NC], wx, wy;
#pragma unroll
  for (int k = 0; k < NC; ++k) U[k] = S[k * g.plane + p];
  CellState<DIM, SYS, DIM == 2> c;
  c.set(U, g, f, wx, wy);
  cell_limiter_of<DIM, SYS, VAR>(g, S, w, p, (int)(p % g.nx), (int)(p / g.nx), d, U, c, f);
}

// The same in every direction with the nonlinear part in pairs (hweno_pair.cuh): U, pu, pv, pH, pc2 the
// cell's state and its velocities, enthalpy and c^2.  Returns false, having written nothing, where
// the FP64 weights are needed.
template <int DIM, int SYS, int VAR>
__device__ __forceinline__ bool cell_limiter_pair(const Grid& g, const double* __restrict__ S, const Work& w,
                                                  long long p, int i, int j, const double* U, P2 pu, P2 pv, P2 pH,
                                                  P2 pc2, const PairSlots& sm, const FU& f) {
  constexpr int NC = Traits<DIM, SYS>::NC;
  const long long plane = g.plane;
  // (asked for last: a return here would hold up the loads of the neighbours, 2 % of a smooth 1024^2 stage)
  const bool units = SYS != SYS_EULER || p_units(U[0], U[NC - 1], g.pg.hexp);
  // FP64: p_0'(x_i) = 3/4 (u_{i+1} - u_{i-1})/h - (v_{i-1} + v_{i+1})/4 and (R2) the derivatives at the two
  // faces; the linear parts of R2's values less the centre value in pairs, which hold them to the last
  // bit of the states where the stencil's differences are small beside these
  double md[DIM][NC], dm[DIM][NC], dp[DIM][NC];
  P4 um[NC], up[NC];
  bool small = true;
  {
    P2 uc[NC], du[2][DIM][NC], z[2][DIM][NC];
#pragma unroll
    for (int k = 0; k < NC; ++k) uc[k] = p_from(U[k]);
#pragma unroll
    for (int d = 0; d < DIM; ++d) {
      double U3[3][NC], D3[3][NC];
      load_stencil3<DIM, SYS, VAR, NC>(g, S, d, i, j, d == 0 ? i : j, U, U3, D3);
      const double k21 = g.uvd[d][0], k3 = g.uvd[d][1];
#pragma unroll
      for (int k = 0; k < NC; ++k) {
        md[d][k] = fma(g.l34[d], f.sub(U3[2][k], U3[0][k]), -0.25 * f.add(D3[0][k], D3[2][k]));
        // the differences are taken between pairs: U to 48 bits is enough for the correction
        const P2 u1 = uc[SYS == SYS_EULER && NC == 4 && d == 1 && (k == 1 || k == 2) ? 3 - k : k];
        if (VAR != 2) {
          du[0][d][k] = p_renorm(p_sub(u1, p_from(U3[0][k])));
          du[1][d][k] = p_renorm(p_sub(p_from(U3[2][k]), u1));
        }
        z[0][d][k] = p_from(D3[0][k]);
        z[1][d][k] = p_from(D3[2][k]);
        if (VAR == 2) {
          const double d0 = f.sub(U3[1][k], U3[0][k]), d1 = f.sub(U3[2][k], U3[1][k]);
          du[0][d][k] = p_from(d0);  // its face values want the differences themselves
          du[1][d][k] = p_from(d1);
          dm[d][k] = fma(k21, d1, fma(-k3, d0, fma(0.0625, D3[0][k], -0.1875 * D3[2][k])));
          dp[d][k] = fma(k21, d0, fma(-k3, d1, fma(-0.1875, D3[0][k], 0.0625 * D3[2][k])));
        }
      }
    }
#pragma unroll
    for (int q = 0; q < 2; ++q)
#pragma unroll
      for (int k = 0; k < NC; ++k) {
        sm.set(q * NC + k, p_pack(du[q][0][k], du[q][DIM - 1][k]));
        sm.set((2 + q) * NC + k, p_pack(z[q][0][k], z[q][DIM - 1][k]));
      }
    if (VAR == 2) {
      const P4 hq = p_pack(p_const<float>(g.pg.h[0]), p_const<float>(g.pg.h[DIM - 1]));
      float size[DIM][NC], u_[NC];
#pragma unroll
      for (int k = 0; k < NC; ++k) {
        const P4 d0 = sm.get(k), d1 = sm.get(NC + k);
        const P4 z0 = p_mul(hq, sm.get(2 * NC + k)), z1 = p_mul(hq, sm.get(3 * NC + k));
        // d0/8 + 9 d1/16 - 3 z0/64 - 9 z1/64 and, mirrored, -d1/8 - 9 d0/16 + 3 z1/64 + 9 z0/64
        um[k] = p_add(p_add(p_scale(d0, 0.125f), p_mulf(d1, 0.5625f)), p_neg(p_mulf(p_add(z0, p_mulf(z1, 3.0f)), 0.046875f)));
        up[k] = p_sub(p_mulf(p_add(z1, p_mulf(z0, 3.0f)), 0.046875f), p_add(p_scale(d1, 0.125f), p_mulf(d0, 0.5625f)));
        u_[k] = uc[k].h;
        size[0][k] = fmaxf(fmaxf(fabsf(f_lane0(d0.h)), fabsf(f_lane0(d1.h))), fmaxf(fabsf(f_lane0(z0.h)), fabsf(f_lane0(z1.h))));
        size[DIM - 1][k] =
            fmaxf(fmaxf(fabsf(f_lane1(d0.h)), fabsf(f_lane1(d1.h))), fmaxf(fabsf(f_lane1(z0.h)), fabsf(f_lane1(z1.h))));
      }
      const float ir = f_rcp(u_[0]), ie = f_rcp(u_[NC - 1]);
#pragma unroll
      for (int d = 0; d < DIM; ++d) small = small && p_rel2<NC>(size[d], ir, ie) <= 0x1p-12f;
    }
  }
  if (!small) return false;
  EigP<NC, F2> e;
  if (SYS == SYS_EULER) {
    const P2 un = DIM == 2 ? pv : pu, ut = DIM == 2 ? pu : pv;
    e.setup(p_pack(pu, un), p_pack(pv, ut), p_pack(pH, pH), p_pack(pc2, pc2), p_const<F2>(g.pg.gm1));
  }
  const P4 h = p_pack(p_const<float>(g.pg.h[0]), p_const<float>(g.pg.h[DIM - 1]));
  P4 nm[NC], np[NC], nt[NC];
  if (!p_cell<NC, SYS, VAR == 2>(sm, e, h, g.pg, nm, np, nt) || !units) return false;
#pragma unroll
  for (int d = 0; d < DIM; ++d) {
    const P2 ih = p_const<float>(g.pg.ih[d]);
    double out[NC];
#pragma unroll
    for (int k = 0; k < NC; ++k) {
      const P2 n = p_mul(d == 0 ? p_lane0(nt[k]) : p_lane1(nt[k]), ih);
      out[k] = f.add(md[d][k], f.add(d_from(n.h), d_from(n.l)));
    }
    if (VAR == 2) {
      double* FSd = w.FS + (long long)d * 4 * NC * plane;
#pragma unroll
      for (int k = 0; k < NC; ++k) {
        const P4 a4 = p_add(um[k], nm[k]), b4 = p_add(up[k], np[k]);
        const P2 a = d == 0 ? p_lane0(a4) : p_lane1(a4), b = d == 0 ? p_lane0(b4) : p_lane1(b4);
        const double u1 = U[SYS == SYS_EULER && NC == 4 && d == 1 && (k == 1 || k == 2) ? 3 - k : k];
        FSd[k * plane + p] = f.add(u1, f.add(d_from(a.h), d_from(a.l)));
        FSd[(NC + k) * plane + p] = dm[d][k];
        FSd[(2 * NC + k) * plane + p] = f.add(u1, f.add(d_from(b.h), d_from(b.l)));
        FSd[(3 * NC + k) * plane + p] = dp[d][k];
      }
    }
    if (SYS == SYS_EULER && d == 1) swap_frame<NC>(out);
#pragma unroll
    for (int k = 0; k < NC; ++k) w.MD[((long long)d * NC + k) * plane + p] = out[k];
  }
  return true;
}

// How a kernel takes the nonlinear part of the interpolation: all of it with the FP64 weights; or in pairs,
// with what the pairs leave to the FP64 weights taken block by block or listed for k_left.
enum { MODE_FP64 = 0, MODE_BLOCK = 1, MODE_LISTED = 2 };

// Cell work of one stage at cell p: wavespeeds (returned in wsx, wsy), primitives, nodal values per
// direction and, LIMITER, modified derivatives (and, for R2, the face states of the cell).  Returns
// false where the modified derivatives are left to cell_limiter (PAIRS).
template <int DIM, int SYS, int VAR, bool PAIRS, bool LIMITER>
__device__ __forceinline__ bool cell_body(const Grid& g, const double* __restrict__ S, const Work& w, long long p,
                                          double& wsx, double& wsy, const PairSlots& sm) {
  using T = Traits<DIM, SYS>;
  constexpr int NC = T::NC, NG = T::NG;
  const long long plane = g.plane;
  const FU f = fu_of(w.scal);
  {
    const int i = (int)(p % g.nx), j = (int)(p / g.nx);
    double U[NC], V[NC], Wd[NC];
#pragma unroll
    for (int k = 0; k < NC; ++k) {
      U[k] = S[k * plane + p];
      V[k] = S[(NC + k) * plane + p];
      if (DIM == 2) Wd[k] = S[(2 * NC + k) * plane + p];
    }
    // primitives and wavespeeds
    CellState<DIM, SYS, !PAIRS && DIM == 2> c;
    if (!c.set(U, g, f, wsx, wsy)) atomicOr(w.status, 1u);
    const double u = c.u, v = c.v, pr = c.pr, ir = c.ir;
    if (VAR && (g.flags & FLAG_ALPHA_LOCAL)) {
      w.WS[p] = wsx;
      if (DIM == 2) w.WS[plane + p] = wsy;
    }
    // primitive derivatives along V and W (2D Euler: shared by the Jacobians of both directions)
    double pdV[3] = {0.0, 0.0, 0.0}, pdW[3] = {0.0, 0.0, 0.0};
    if (SYS == SYS_EULER && DIM == 2) {
      Phys<2, SYS_EULER>::prim_deriv(U, u, v, ir, V, g.gm1, pdV[0], pdV[1], pdV[2], f);
      Phys<2, SYS_EULER>::prim_deriv(U, u, v, ir, Wd, g.gm1, pdW[0], pdW[1], pdW[2], f);
    }
    // nodal values per direction (normal frame)
#pragma unroll
    for (int d = 0; d < DIM; ++d) {
      double Un[NC], Dn[NC], On[NC], F[NC], Hn[NC], Mx[NC];
#pragma unroll
      for (int k = 0; k < NC; ++k) {
        Un[k] = U[k];
        Dn[k] = d == 0 ? V[k] : Wd[k];
        On[k] = d == 0 ? Wd[k] : V[k];
      }
      const double a = d == 0 ? g.ax : g.ay;
      if (SYS == SYS_EULER) {
        if (d == 1) {
          swap_frame<NC>(Un);
          swap_frame<NC>(Dn);
          swap_frame<NC>(On);
        }
        const double un = d == 0 ? u : v;
        F[0] = Un[1];
        F[1] = fma(Un[1], un, pr);
        if (DIM == 2) F[2] = f.mul(Un[2], un);
        F[NC - 1] = f.mul(f.add(Un[NC - 1], pr), un);
        if (DIM == 2) {
          // own-direction field (V in x, W in y) and the other one, each with its normal-velocity
          // derivative (u' in x, v' in y)
          const double* po = d == 0 ? pdV : pdW;
          const double* pt = d == 0 ? pdW : pdV;
          const double hp = f.add(U[NC - 1], pr);
          Phys<2, SYS_EULER>::jvp_apply(Un, Dn, un, po[d], po[2], hp, Hn, f);
          Phys<2, SYS_EULER>::jvp_apply(Un, On, un, pt[d], pt[2], hp, Mx, f);
        } else {
          Phys<1, SYS_EULER>::jvp_prim(Un, un, pr, ir, Dn, Hn, g.gm1, f);
        }
      } else {
        Phys<DIM, SYS>::flux(Un, F, a, g.gm1);
        Phys<DIM, SYS>::jvp(Un, Dn, Hn, a, g.gm1);
        if (DIM == 2) Phys<DIM, SYS>::jvp(Un, On, Mx, a, g.gm1);
      }
      double* nod = w.NOD + (long long)d * NG * NC * plane;
#pragma unroll
      for (int k = 0; k < NC; ++k) {
        nod[k * plane + p] = F[k];
        nod[(NC + k) * plane + p] = Hn[k];
        if (DIM == 2) nod[(2 * NC + k) * plane + p] = Mx[k];
      }
    }
    if (SYS == SYS_EULER && VAR != 2 && !(PAIRS && (VAR == 0 || g.face_pairs))) {
      double* P = reinterpret_cast<double*>(w.PRIM);
      P[p] = sqrt_fast(U[0], f);
      P[plane + p] = u;
      if (DIM == 2) P[2 * plane + p] = v;
      P[DIM * plane + plane + p] = f.mul(f.add(U[NC - 1], pr), ir);
    }
    // modified derivatives (Eq. limiter), one per direction
    if constexpr (!PAIRS) {
      if (LIMITER)
#pragma unroll
        for (int d = 0; d < DIM; ++d) cell_limiter_of<DIM, SYS, VAR>(g, S, w, p, i, j, d, U, c, f);
      return true;
    }
    P2 pu = {0.0f, 0.0f}, pv = pu, pH = pu, pc2 = pu;
    if (SYS == SYS_EULER) {
      P2 q[NC], inv;
#pragma unroll
      for (int k = 0; k < NC; ++k) q[k] = p_from(U[k]);
      const P2 gm1 = P2{g.pg.gm1[0], g.pg.gm1[1]};
      p_prim<NC>(q, gm1, pu, pv, pH, pc2);
      pc2 = p_add(pc2, p_mul(gm1, pc2));  // gamma p / rho
      if (VAR == 0 || (VAR == 1 && g.face_pairs)) {
        const P2 sr = p_sqrt(q[0], inv);
        w.PRIM[p] = make_float2(sr.h, sr.l);
        w.PRIM[plane + p] = make_float2(pu.h, pu.l);
        if (DIM == 2) w.PRIM[2 * plane + p] = make_float2(pv.h, pv.l);
        w.PRIM[DIM * plane + plane + p] = make_float2(pH.h, pH.l);
      }
    }
    return cell_limiter_pair<DIM, SYS, VAR>(g, S, w, p, i, j, U, pu, pv, pH, p_renorm(pc2), sm, f);
  }
}

// The cells or faces of one block whose nonlinear weights are to be evaluated in FP64: the block's
// threads take them in turn afterwards, so that a warp with a single one of them does not run the
// FP64 path for its other lanes (an FP64 warp instruction costs the same with one lane active).  A
// block that has any keeps its place on the SM for one more pass of FP64 work in one or two warps;
// listed grids append theirs to one list instead, which k_left takes in full warps.
struct Leftover {
  int n;
  unsigned short item[2 * kThreads];
};

// The cells p0 .. p0 + kThreads - 1 of a block, one per thread; every thread of the block calls it.
// reused: the block calls it again with the same list.
template <int DIM, int SYS, int VAR, int MODE>
__device__ __forceinline__ void cell_tile(const Grid& g, const double* __restrict__ S, const Work& w, long long p0,
                                          double& wsx, double& wsy, Leftover& lo, const PairSlots& sm, bool reused) {
  const long long p = p0 + threadIdx.x;
  if (MODE == MODE_LISTED) {
    // (one atomic per thread: collected by warp, the kernel takes 3 % longer with nothing to append)
    if (p < g.plane && !cell_body<DIM, SYS, VAR, true, true>(g, S, w, HW_IDX(p, g.plane), wsx, wsy, sm)) {
      const unsigned int k = atomicAdd(w.status + 2, (unsigned int)DIM);
#pragma unroll
      for (unsigned int d = 0; d < DIM; ++d)
        w.left_cells[HW_IDX((long long)k + d, DIM * g.plane)] = (unsigned int)p * 2u + d;
    }
    return;
  }
  if (MODE == MODE_FP64) {
    if (p < g.plane) cell_body<DIM, SYS, VAR, false, true>(g, S, w, HW_IDX(p, g.plane), wsx, wsy, sm);
    return;
  }
  if (reused) __syncthreads();
  if (threadIdx.x == 0) lo.n = 0;
  __syncthreads();
  if (p < g.plane) {
    if (!cell_body<DIM, SYS, VAR, true, true>(g, S, w, HW_IDX(p, g.plane), wsx, wsy, sm)) {
      const int k = atomicAdd(&lo.n, DIM);
#pragma unroll
      for (int d = 0; d < DIM; ++d) lo.item[k + d] = (unsigned short)(threadIdx.x * 2 + d);
    }
  }
  __syncthreads();
  for (int k = threadIdx.x; k < lo.n; k += kThreads) {
    const int it = lo.item[k];
    cell_limiter<DIM, SYS, VAR>(g, S, w, HW_IDX(p0 + (it >> 1), g.plane), it & 1);
  }
}

// Bound by the FP64 pipe (85 % busy): 123 FP64 instructions per 2D Euler cell against 545 with the FP64
// weights; 1024^2 0.24 ms per launch against 0.97 ms.  MODE_FP64 is the form of the grids that wait for one
// thread's chain of instructions (pairs_of): no pair code, no slots, 130 registers and no spills (48^2
// 24.3 us a launch; inside the kernel with the pairs 26.8 us).
template <int DIM, int SYS, int VAR, int MODE>
__global__ void __launch_bounds__(kThreads, MODE == MODE_FP64 ? 3 : 4) k_cell(Grid g, const double* __restrict__ S,
                                                                             Work w, int slot) {
  __shared__ Leftover lo;
  __shared__ ulonglong2 slots[MODE == MODE_FP64 ? 1 : 4 * Traits<DIM, SYS>::NC * kThreads];
  double wsx = 0.0, wsy = 0.0;
  cell_tile<DIM, SYS, VAR, MODE>(g, S, w, (long long)blockIdx.x * kThreads, wsx, wsy, lo,
                                 PairSlots{slots + (MODE == MODE_FP64 ? 0 : threadIdx.x)}, false);
  block_max2(wsx, wsy, w.alpha + slot * w.astride);
}

// R1 face states: the interface values and derivatives from both sides of face k+1/2, from the
// states Uq and derivatives Zq (normal frame) of the cells k-1..k+2, interpolated in the
// characteristic fields of e (the Roe average at the face; unused for a scalar law).  The
// interpolation needs the fields only through differences of neighbouring cells and the
// derivatives: the three conserved differences are projected and the centre states added back in
// conserved variables.  VW: the weighted-derivative option.
template <int NC, int SYS, bool VW>
__device__ __forceinline__ void r1_face_states(const double (&Uq)[4][NC], const double (&Zq)[4][NC],
                                               const Eig<NC>& e, const Grid& g, int dir, double* Um, double* Up,
                                               double* Dm, double* Dp, const FU& f) {
  double dU[3][NC];
#pragma unroll
  for (int q = 0; q < 3; ++q)
#pragma unroll
    for (int k = 0; k < NC; ++k) dU[q][k] = f.sub(Uq[q + 1][k], Uq[q][k]);
  if (!VW) {
    // the Hermite derivative of Eq. (P'xi) at the face from both sides (linear in the stencil,
    // formed first so that the differences and derivatives are not held through the fields)
    const double k21 = g.uvd[dir][0], k3 = g.uvd[dir][1];
#pragma unroll
    for (int k = 0; k < NC; ++k) {
      Dm[k] = fma(k21, dU[1][k], fma(-k3, dU[0][k], fma(0.0625, Zq[0][k], -0.1875 * Zq[2][k])));
      Dp[k] = fma(k21, dU[1][k], fma(-k3, dU[2][k], fma(-0.1875, Zq[1][k], 0.0625 * Zq[3][k])));
    }
  }
  double Dq[3][NC], Yq[4][NC];
  if (SYS == SYS_EULER) {
#pragma unroll
    for (int q = 0; q < 3; ++q) e.project(dU[q], Dq[q], f);
#pragma unroll
    for (int q = 0; q < 4; ++q) e.project(Zq[q], Yq[q], f);
  } else {
#pragma unroll
    for (int q = 0; q < 3; ++q) Dq[q][0] = dU[q][0];
#pragma unroll
    for (int q = 0; q < 4; ++q) Yq[q][0] = Zq[q][0];
  }
  // HWENO interpolation in each characteristic field: u^- from the stencil of cell k, u^+ from the
  // stencil of cell k+1 (mirror image)
  const double bm = SYS == SYS_EULER ? 0.0 : Uq[1][0], bp = SYS == SYS_EULER ? 0.0 : Uq[2][0];
  double cm[NC], chm[NC], cp[NC], chp[NC];
  const StencilK k = stencil_k(g, dir, f);
#pragma unroll
  for (int s = 0; s < NC; ++s)
    face_field_d<VW>(Dq[0][s], Dq[1][s], Dq[2][s], Yq[0][s], Yq[1][s], Yq[2][s], Yq[3][s], bm, bp, k, g, dir, cm[s],
                     chm[s], cp[s], chp[s], f);
  // back to conserved variables
  if (SYS == SYS_EULER) {
    e.back_add(cm, Uq[1], Um, f);
    e.back_add(cp, Uq[2], Up, f);
  } else {
    Um[0] = cm[0];
    Up[0] = cp[0];
  }
  if (VW) {
    if (SYS == SYS_EULER) {
      e.back(chm, Dm, f);
      e.back(chp, Dp, f);
    } else {
      Dm[0] = chm[0];
      Dp[0] = chp[0];
    }
  }
}

// ---------------------------------------------------------------------------------------------
// Face work of one stage: face f of direction dir (x faces: f = j (nx+1) + i; y faces:
// f = j nx + i), alpha = the LF coefficient of that direction.  PAIR: the nonlinear part of the
// interpolation in pairs (hweno_pair.cuh); returns false, having written the mixed flux at most, where the
// FP64 weights are needed (R2: the flux of two close states in pairs).  STORED: the primitives were stored in
// FP64; else they are formed from the states.
template <int DIM, int SYS, int VAR, bool PAIR, bool STORED = false>
__device__ __forceinline__ bool face_body(const Grid& g, const double* __restrict__ S, const Work& w, int dir,
                                          long long f, double alpha, const PairSlots& sm) {
  using T = Traits<DIM, SYS>;
  constexpr int NC = T::NC, NG = T::NG;
  const long long plane = g.plane;
  const FU fu = fu_of(w.scal);
  const int n = dir == 0 ? g.nx : g.ny;
  int fa, line;
  if (dir == 0) {
    line = (int)(f / (n + 1));
    fa = (int)(f % (n + 1));
  } else {
    fa = (int)(f / g.nx);
    line = (int)(f % g.nx);
  }
  // cells fa-2 .. fa+1 around face fa (between cells fa-1 and fa)
  long long pc[4];
  bool refl[4], fixed[4];
  int fside[4];
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    fixed[q] = false;
    fside[q] = 2 * dir + (fa - 2 + q < 0 ? 0 : 1);
    const int a = VAR ? bc_map_ext(fa - 2 + q, n, g.side[2 * dir], g.side[2 * dir + 1], refl[q], fixed[q])
                      : bc_map(fa - 2 + q, n, g.bc, refl[q]);
    pc[q] = HW_IDX(dir == 0 ? (long long)line * g.nx + a : (long long)a * g.nx + line, plane);
  }
  const int fown = dir == 0 ? 1 : 2, foth = dir == 0 ? 2 : 1;
  // local LF: the larger spectral radius of the two cells of the face
  if (VAR && (g.flags & FLAG_ALPHA_LOCAL)) {
    const double al = fixed[1] ? g.fixA[fside[1]] : w.WS[dir * plane + pc[1]];
    const double ar = fixed[2] ? g.fixA[fside[2]] : w.WS[dir * plane + pc[2]];
    alpha = fmax(al, ar);
  }
  const double* nod = w.NOD + (long long)dir * NG * NC * plane;
  double* out = dir == 0 ? w.FX : w.FY;
  const long long oplane = dir == 0 ? (long long)g.ny * (g.nx + 1) : (long long)(g.ny + 1) * g.nx;
  const long long fo = HW_IDX(dir == 0 ? (long long)line * (g.nx + 1) + fa : (long long)fa * g.nx + line, oplane);
  // Eq. (mixed), linear in the nodal values: independent of everything below.  Nodal values of mirrored
  // neighbours (normal frame): f and the mixed value change sign except for the normal momentum, the
  // normal-derivative flux changes sign only for the normal momentum.  First where registers are short
  // (PAIR) and for R2 (100^2: 75.7 us an evaluation, 77.2 at the end); else with the other nodal values, so
  // that the loads of the primitives do not wait for its stores (96x170: 84.8 us, first 85.8).
  constexpr bool kMixedFirst = PAIR || VAR == 2;
  auto mixed = [&] {
    if (DIM != 2) return;
#pragma unroll
    for (int k = 0; k < NC; ++k) {
      double o[4];
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        o[q] = neg_if(nod[(2 * NC + k) * plane + pc[q]], refl[q] && k != 1);
        if (VAR && fixed[q]) o[q] = 0.0;
      }
      const int ko = SYS == SYS_EULER && dir == 1 && (k == 1 || k == 2) ? 3 - k : k;
      out[(foth * NC + ko) * oplane + fo] = fma(7.0 / 12.0, fu.add(o[1], o[2]), (-1.0 / 12.0) * fu.add(o[0], o[3]));
    }
  };
  if (kMixedFirst) mixed();
  const double a_adv = dir == 0 ? g.ax : g.ay;
  const P2 ih = p_const<float>(g.pg.ih[dir]);
  double Um[NC], Up[NC], Dm[NC], Dp[NC];
  // Lax-Friedrichs fluxes (Eq. flux-LF): FS/2 + vf and HS/2 + vh, with FS = f(U^-) + f(U^+),
  // vf = -alpha (U^+ - U^-)/2, HS and vh likewise from f'(U) D and D.  Where the two states of an
  // Euler face are close (PAIR, and the near faces of R2), FS and HS are the flux and the Jacobian
  // product of the sums of the states and derivatives (both are homogeneous of degree one), and what
  // the mean of the two fluxes differs by joins vf and vh (p_flux_pair): half of the flux arithmetic.
  double FS[NC], HS[NC], vf[NC], vh[NC];
  bool summed = false;
  if (VAR == 2) {
    // R2: the face states were formed per cell (the low and high ghosts by k_r2_ghost)
    const double* FSd = w.FS + (long long)dir * 4 * NC * plane;
    const long long gs = w.gstride;
    const double* Glo = w.GFS + (long long)(dir * 2 + 0) * 2 * NC * gs;
    const double* Ghi = w.GFS + (long long)(dir * 2 + 1) * 2 * NC * gs;
    const long long gl = HW_IDX(line, gs);
#pragma unroll
    for (int k = 0; k < NC; ++k) {
      Um[k] = fa >= 1 ? FSd[(0 * NC + k) * plane + pc[1]] : Glo[(0 * NC + k) * gs + gl];
      Dm[k] = fa >= 1 ? FSd[(1 * NC + k) * plane + pc[1]] : Glo[(1 * NC + k) * gs + gl];
      Up[k] = fa < n ? FSd[(2 * NC + k) * plane + pc[2]] : Ghi[(0 * NC + k) * gs + gl];
      Dp[k] = fa < n ? FSd[(3 * NC + k) * plane + pc[2]] : Ghi[(1 * NC + k) * gs + gl];
    }
  } else {
    double Uq[4][NC], Zq[4][NC];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
#pragma unroll
      for (int k = 0; k < NC; ++k) {
        Uq[q][k] = S[k * plane + pc[q]];
        Zq[q][k] = S[(fown * NC + k) * plane + pc[q]];
      }
      if (SYS == SYS_EULER && dir == 1) {
        swap_frame<NC>(Uq[q]);
        swap_frame<NC>(Zq[q]);
      }
      if (SYS == SYS_EULER) {
        mirror_U<NC>(Uq[q], refl[q]);
        mirror_D<NC>(Zq[q], refl[q]);
      }
      if (VAR && fixed[q]) load_fixed<NC, SYS>(g, fside[q], dir, Uq[q], Zq[q]);
    }
    if (PAIR) {
      const bool units = SYS != SYS_EULER || (p_units(Uq[1][0], Uq[1][NC - 1], g.pg.hexp) &&
                                              p_units(Uq[2][0], Uq[2][NC - 1], g.pg.hexp));
      double dU[3][NC];
#pragma unroll
      for (int q = 0; q < 3; ++q)
#pragma unroll
        for (int k = 0; k < NC; ++k) dU[q][k] = fu.sub(Uq[q + 1][k], Uq[q][k]);
      // the Hermite derivatives of Eq. (P'xi), which are linear in the stencil, and the linear parts of
      // the interface values less the centre values; for the Euler equations the sums of both sides,
      // the values' linear part among the pairs
      const double k21 = g.uvd[dir][0], k3 = g.uvd[dir][1], l3 = g.l3[dir], l9 = g.l9[dir];
      double Us[NC], Ds[NC], da[NC], zo[NC], zi[NC];
      if (SYS == SYS_EULER) {
        const double k42 = 2.0 * k21;
#pragma unroll
        for (int k = 0; k < NC; ++k) {
          Us[k] = fu.add(Uq[1][k], Uq[2][k]);
          da[k] = fu.sub(dU[0][k], dU[2][k]);
          zo[k] = fu.sub(Zq[3][k], Zq[0][k]);
          zi[k] = fu.sub(Zq[2][k], Zq[1][k]);
          Ds[k] = fma(k42, dU[1][k],
                      fma(-k3, fu.add(dU[0][k], dU[2][k]),
                          fma(0.0625, fu.add(Zq[0][k], Zq[3][k]), -0.1875 * fu.add(Zq[1][k], Zq[2][k]))));
        }
      } else {
        Um[0] = fma(0.125, dU[0][0], fma(0.5625, dU[1][0], fma(-l3, Zq[0][0], -l9 * Zq[2][0])));
        Up[0] = fma(-0.125, dU[2][0], fma(-0.5625, dU[1][0], fma(l3, Zq[3][0], l9 * Zq[1][0])));
        Dm[0] = fma(k21, dU[1][0], fma(-k3, dU[0][0], fma(0.0625, Zq[0][0], -0.1875 * Zq[2][0])));
        Dp[0] = fma(k21, dU[1][0], fma(-k3, dU[2][0], fma(-0.1875, Zq[1][0], 0.0625 * Zq[3][0])));
      }
      EigP<NC, F2> e;
      if (SYS == SYS_EULER) {
        // Roe average of the two adjacent cells from their primitives; a mirrored neighbour has the
        // opposite normal velocity
        P4 c[2][NC];
#pragma unroll
        for (int q = 0; q < 2; ++q) {
#pragma unroll
          for (int k = 0; k < NC; ++k) {
            const int kn = NC == 4 && dir == 1 && (k == 1 || k == 2) ? 3 - k : k;
            const float2 t = w.PRIM[kn * plane + pc[1 + q]];
            P2 x = P2{t.x, t.y};
            if (VAR && fixed[1 + q]) x = p_from(g.fixP[fside[1 + q]][kn]);
            if (k == 1 && refl[1 + q]) x = p_neg(x);
            c[q][k] = p_pack(x, x);
          }
        }
        e.setup_roe(c[0], c[1], p_const<F2>(g.pg.gm1));
      }
      P4 n[NC];
      P2 sum[NC], dif[NC], hdif[NC];
      float size[NC];
      if (!p_face<NC, SYS>(dU, Zq, da, zo, zi, e, g.pg, dir, sm, n, sum, dif, hdif, size) || !units) return false;
      if (SYS == SYS_EULER) {
#pragma unroll
        for (int k = 0; k < NC; ++k) {
          Us[k] = fu.add(Us[k], fu.add(d_from(sum[k].h), d_from(sum[k].l)));
        }
        if (!p_flux_pair<NC>(Us, Ds, dif, hdif, size, alpha, ih, g.pg, fu, vf, vh)) return false;
        Phys<DIM, SYS>::flux_jvp(Us, Ds, FS, HS, a_adv, g.gm1, fu);
        summed = true;
      } else {
        const P2 a = p_lane0(n[0]), b = p_lane1(n[0]);
        Um[0] = fu.add(Uq[1][0], fu.add(Um[0], fu.add(d_from(a.h), d_from(a.l))));
        Up[0] = fu.add(Uq[2][0], fu.add(Up[0], fu.add(d_from(b.h), d_from(b.l))));
      }
    } else {
      // characteristic fields at the face: Roe average of the two adjacent cells
      Eig<NC> e;
      if (SYS == SYS_EULER) {
        double sq[2], uq[2], vq[2], Hq[2];
#pragma unroll
        for (int q = 0; q < 2; ++q) {
          const double* U = Uq[1 + q];
          if (STORED) {
            const double* P = reinterpret_cast<const double*>(w.PRIM);
            const bool fx = VAR && fixed[1 + q];
            const double* F = g.fixP[fside[1 + q]];
            const int kn = DIM == 2 && dir == 1 ? 2 : 1;  // the normal velocity
            sq[q] = fx ? F[0] : P[pc[1 + q]];
            uq[q] = neg_if(fx ? F[kn] : P[kn * plane + pc[1 + q]], refl[1 + q]);
            vq[q] = DIM == 1 ? 0.0 : (fx ? F[3 - kn] : P[(3 - kn) * plane + pc[1 + q]]);
            Hq[q] = fx ? F[DIM + 1] : P[(DIM + 1) * plane + pc[1 + q]];
            continue;
          }
          const double ir = rcp(U[0], fu);
          uq[q] = fu.mul(U[1], ir);
          vq[q] = DIM == 2 ? fu.mul(U[2], ir) : 0.0;
          const double ke = DIM == 2 ? fma(U[1], uq[q], fu.mul(U[2], vq[q])) : fu.mul(U[1], uq[q]);
          Hq[q] = fu.mul(fu.add(U[NC - 1], g.gm1 * fma(-0.5, ke, U[NC - 1])), ir);
          sq[q] = sqrt_fast(U[0], fu);
        }
        const double iw = rcp(fu.add(sq[0], sq[1]), fu);
        const double ub = fu.mul(fma(sq[0], uq[0], fu.mul(sq[1], uq[1])), iw);
        const double vb = DIM == 2 ? fu.mul(fma(sq[0], vq[0], fu.mul(sq[1], vq[1])), iw) : 0.0;
        const double Hb = fu.mul(fma(sq[0], Hq[0], fu.mul(sq[1], Hq[1])), iw);
        const double c2 = g.gm1 * fma(-0.5, DIM == 2 ? fma(ub, ub, fu.mul(vb, vb)) : fu.mul(ub, ub), Hb);
        const double ic = rsqrt_full(c2, fu);
        e.setup(ub, vb, Hb, fu.mul(c2, ic), ic, g.gm1);
      }
      if (VAR && (g.flags & FLAG_V_WEIGHTED))
        r1_face_states<NC, SYS, true>(Uq, Zq, e, g, dir, Um, Up, Dm, Dp, fu);
      else
        r1_face_states<NC, SYS, false>(Uq, Zq, e, g, dir, Um, Up, Dm, Dp, fu);
    }
  }
  if (VAR == 2 && PAIR) {
    double Us[NC], Ds[NC];
    P2 dif[NC], hdif[NC];
    float size[NC];
    const P2 h = p_const<float>(g.pg.h[dir]);
#pragma unroll
    for (int k = 0; k < NC; ++k) {
      Us[k] = fu.add(Um[k], Up[k]);
      Ds[k] = fu.add(Dm[k], Dp[k]);
      dif[k] = p_from(fu.sub(Up[k], Um[k]));
      hdif[k] = p_mul(h, p_from(fu.sub(Dp[k], Dm[k])));
      size[k] = p_from(Ds[k]).h * h.h;
    }
    if (p_units(Us[0], Us[NC - 1], g.pg.hexp) && p_flux_pair<NC>(Us, Ds, dif, hdif, size, alpha, ih, g.pg, fu, vf, vh)) {
      Phys<DIM, SYS>::flux_jvp(Us, Ds, FS, HS, a_adv, g.gm1, fu);
      summed = true;
    }
  }
  if (!summed) {
    double FUm[NC], FUp[NC], HDm[NC], HDp[NC];
    Phys<DIM, SYS>::flux_jvp(Um, Dm, FUm, HDm, a_adv, g.gm1, fu);
    Phys<DIM, SYS>::flux_jvp(Up, Dp, FUp, HDp, a_adv, g.gm1, fu);
    const double ma = -0.5 * alpha;
#pragma unroll
    for (int k = 0; k < NC; ++k) {
      FS[k] = fu.add(FUm[k], FUp[k]);
      HS[k] = fu.add(HDm[k], HDp[k]);
      vf[k] = fu.mul(ma, fu.sub(Up[k], Um[k]));
      vh[k] = fu.mul(ma, fu.sub(Dp[k], Dm[k]));
    }
  }
  const bool cd2 = VAR && (g.flags & FLAG_CD2) != 0;
  if (!kMixedFirst) mixed();
  double fh[NC], hh[NC];
#pragma unroll
  for (int k = 0; k < NC; ++k) {
    const bool nm = k == 1;
    const bool s0 = refl[0] && !nm, s1 = refl[1] && !nm, s2 = refl[2] && !nm, s3 = refl[3] && !nm;
    double f0 = neg_if(nod[k * plane + pc[0]], s0), f1 = neg_if(nod[k * plane + pc[1]], s1);
    double f2 = neg_if(nod[k * plane + pc[2]], s2), f3 = neg_if(nod[k * plane + pc[3]], s3);
    // h at the outer nodes (Eq. Cd-1) or, for Cd-2, at the inner ones
    double ha = neg_if(nod[(NC + k) * plane + pc[cd2 ? 1 : 0]], refl[cd2 ? 1 : 0] && nm);
    double hb = neg_if(nod[(NC + k) * plane + pc[cd2 ? 2 : 3]], refl[cd2 ? 2 : 3] && nm);
    if (VAR) {
      // a fixed-state ghost: the side's flux, zero derivative fluxes
      if (fixed[0]) f0 = g.fixF[fside[0]][k];
      if (fixed[1]) f1 = g.fixF[fside[1]][k];
      if (fixed[2]) f2 = g.fixF[fside[2]][k];
      if (fixed[3]) f3 = g.fixF[fside[3]][k];
      if (fixed[cd2 ? 1 : 0]) ha = 0.0;
      if (fixed[cd2 ? 2 : 3]) hb = 0.0;
    }
    double Df, Dh;
    if (cd2) {
      // D-terms (Eqs. Cd-2, DfDh), with the viscous part
      Df = fma(DCoef2::cf, fu.add(fu.sub(f0, f1), fu.sub(f3, f2)), fma(g.c2h[dir], fu.sub(ha, hb), vf[k]));
      Dh = fma(g.e2fih[dir], fu.sub(f0, f3), fma(g.e2gih[dir], fu.sub(f1, f2), fma(DCoef2::eh, fu.add(ha, hb), vh[k])));
    } else {
      // D-terms (Eqs. Cd-1, DfDh), with the viscous part
      Df = fma(DCoef::cf, fu.add(fu.sub(f0, f1), fu.sub(f3, f2)), fma(g.chh[dir], fu.sub(ha, hb), vf[k]));
      Dh = fma(g.efih[dir], fu.sub(f0, f3), fma(g.egih[dir], fu.sub(f2, f1), fma(DCoef::eh, fu.add(ha, hb), vh[k])));
    }
    fh[k] = fma(0.5, FS[k], Df);
    hh[k] = fma(0.5, HS[k], Dh);
  }
  if (SYS == SYS_EULER && dir == 1) {
    swap_frame<NC>(fh);
    swap_frame<NC>(hh);
  }
#pragma unroll
  for (int k = 0; k < NC; ++k) {
    out[k * oplane + fo] = fh[k];
    out[(fown * NC + k) * oplane + fo] = hh[k];
  }
  return true;
}

// The faces f0 .. f0 + kThreads - 1 (of nf) of direction dir, one per thread; every thread of the
// block calls it.  reused: as cell_tile.
template <int DIM, int SYS, int VAR, int MODE>
__device__ __forceinline__ void face_tile(const Grid& g, const double* __restrict__ S, const Work& w, int dir,
                                          long long f0, long long nf, double alpha, Leftover& lo,
                                          const PairSlots& sm, bool reused) {
  const long long f = f0 + threadIdx.x;
  // R2: only the fluxes (k_cell formed the face states)
  if (MODE == MODE_FP64 || VAR == 2) {
    if (f < nf) face_body<DIM, SYS, VAR, MODE != MODE_FP64, true>(g, S, w, dir, f, alpha, sm);
    return;
  }
  if (MODE == MODE_LISTED) {
    if (f < nf && !face_body<DIM, SYS, VAR, true>(g, S, w, dir, f, alpha, sm)) {
      const long long nfx = (long long)(g.nx + 1) * g.ny, all = nfx + (DIM == 2 ? (long long)(g.ny + 1) * g.nx : 0);
      w.left_faces[HW_IDX(atomicAdd(w.status + 3, 1u), all)] = (unsigned int)(f + (dir == 0 ? 0 : nfx));
    }
    return;
  }
  if (reused) __syncthreads();
  if (threadIdx.x == 0) lo.n = 0;
  __syncthreads();
  if (f < nf && !face_body<DIM, SYS, VAR, true>(g, S, w, dir, f, alpha, sm))
    lo.item[atomicAdd(&lo.n, 1)] = (unsigned short)threadIdx.x;
  __syncthreads();
  for (int k = threadIdx.x; k < lo.n; k += kThreads)
    face_body<DIM, SYS, VAR, false>(g, S, w, dir, f0 + lo.item[k], alpha, sm);
}

// Bound by the FP64 pipe (86 % busy at 1024^2; about 170 FP64 instructions per 2D Euler face against 666
// with the FP64 weights everywhere), with the latency of the pairs' FP32 work between: four blocks of 128
// per SM (128 registers) cover it better than three or five (2D Euler 2048^2 with k_cell likewise: 4.70
// against 4.75 and 4.94 ms per stage, before the pairs' loops).  2D Euler 1024^2: 0.70 ms per launch
// against 2.33 ms with the FP64 weights.
// MODE_FP64 (small grids; the weighted derivative, which needs the weights everywhere): three blocks per SM,
// 166 registers without spills.  The same form inside the kernel with the pairs had 128 registers and 496 B
// of spills (916 B with the variants): 48^2 30.8 us a launch against 30.3; the weighted derivative at
// 1024^2 2.67 ms against 2.56.
template <int DIM, int SYS, int VAR, int MODE>
__global__ void __launch_bounds__(kThreads, MODE == MODE_FP64 && DIM == 2 ? 3 : 4) k_face(
    Grid g, const double* __restrict__ S, Work w, int slot) {
  constexpr bool kSlots = SYS == SYS_EULER && VAR != 2 && MODE != MODE_FP64;  // the others use none
  __shared__ Leftover lo;
  __shared__ ulonglong2 slots[kSlots ? 4 * Traits<DIM, SYS>::NC * kThreads : 1];
  const int dir = blockIdx.y;
  const int n = dir == 0 ? g.nx : g.ny;
  const int nlines = dir == 0 ? g.ny : g.nx;
  face_tile<DIM, SYS, VAR, MODE>(g, S, w, dir, (long long)blockIdx.x * kThreads, (long long)(n + 1) * nlines,
                                 __longlong_as_double((long long)w.alpha[slot * w.astride + dir]), lo,
                                 PairSlots{slots + (kSlots ? threadIdx.x : 0)}, false);
}

// The listed cells and faces of a stage with the FP64 weights, in full warps (faces first, then cells): a
// fixed grid, three blocks of 128 per SM as the FP64 path's registers allow.  It is bound by the FP64
// pipe (about 560 instructions a face) and idle when the lists are empty.
template <int DIM, int SYS, int VAR>
__global__ void __launch_bounds__(kThreads, 3) k_left(Grid g, const double* __restrict__ S, Work w, int slot) {
  const long long nfx = (long long)(g.nx + 1) * g.ny, all = nfx + (DIM == 2 ? (long long)(g.ny + 1) * g.nx : 0);
  const long long nf = min((long long)w.status[3], all), nfw = (nf + 31) / 32 * 32;
  const long long nc = min((long long)w.status[2], DIM * g.plane);
  const PairSlots none{nullptr};
  for (long long k = (long long)blockIdx.x * kThreads + threadIdx.x; k < nfw + nc; k += (long long)gridDim.x * kThreads) {
    if (k < nf) {
      const long long f = HW_IDX(w.left_faces[HW_IDX(k, all)], all);
      const int dir = f < nfx ? 0 : 1;
      if (f < all)
        face_body<DIM, SYS, VAR, false>(g, S, w, dir, f - (dir == 0 ? 0 : nfx),
                                        __longlong_as_double((long long)w.alpha[slot * w.astride + dir]), none);
    } else if (k >= nfw) {
      const unsigned int c = w.left_cells[HW_IDX(k - nfw, DIM * g.plane)];
      if ((long long)(c >> 1) < g.plane) cell_limiter<DIM, SYS, VAR>(g, S, w, HW_IDX(c >> 1, g.plane), (int)(c & 1u));
    }
  }
}

// ---------------------------------------------------------------------------------------------
// Update of one cell p.  mode 0: Runge-Kutta stage in place, S = a B + b (M + dt L) (stage 0:
// B := M, S = M + dt L).  mode 1: write L and M to Lout, Mout.
template <int DIM, int SYS, int VAR = 0>
__device__ __forceinline__ void update_body(const Grid& g, double* __restrict__ S, const Work& w, int mode, int stage,
                                            double a_k, double b_k, double dt, long long p_in,
                                            double* __restrict__ Lout, double* __restrict__ Mout) {
  using T = Traits<DIM, SYS>;
  constexpr int NC = T::NC, NF = T::NF;
  // the gravity source, where it is possible (tested in the integer pipe)
  const bool src = VAR != 0 && DIM == 2 && SYS == SYS_EULER && (dbl_bits(g.grav) << 1) != 0;
  const long long plane = g.plane;
  const long long p = HW_IDX(p_in, plane);
  const int i = (int)(p % g.nx), j = (int)(p / g.nx);
  const long long oplx = (long long)g.ny * (g.nx + 1), oply = (long long)(g.ny + 1) * g.nx;
  const long long px = HW_IDX((long long)j * (g.nx + 1) + i, oplx - 1);  // faces px and px + 1
  // the stage's constants copied into thread registers (exactly: c 1 + (-0) = c), so that every
  // FP64 instruction below has register operands (see FU)
  const FU fu = fu_of(w.scal);
  const double mix = fu.reg(-g.inv_dx), miy = fu.reg(-g.inv_dy);
  const double akr = fu.reg(a_k), bkr = fu.reg(b_k);
  // the Runge-Kutta stage b (M + dt L) with dt L = (dt mix) dF + (dt miy) dG (+ dt source): the
  // coefficients of the two flux differences taken as one product each, b dt (-1/h) (b = 1 at the
  // first stage)
  const double bdt = fu.mul(bkr, fu.reg(dt));
  const double cx = fu.mul(bdt, mix), cy = fu.mul(bdt, miy);
#pragma unroll
  for (int f = 0; f < NF; ++f) {
    // Eq. (euler2d-s): field f gains g (0, 0, S_f[rho], S_f[rho nu]) (read before S is overwritten)
    double src2 = 0.0, src3 = 0.0;
    if (src) {
      src2 = g.grav * S[(f * NC + 0) * plane + p];
      src3 = g.grav * S[(f * NC + 2) * plane + p];
    }
#pragma unroll
    for (int k = 0; k < NC; ++k) {
      const int fk = f * NC + k;
      const double dF = fu.sub(w.FX[fk * oplx + px + 1], w.FX[fk * oplx + px]);
      const double dG = DIM == 2 ? fu.sub(w.FY[fk * oply + p + g.nx], w.FY[fk * oply + p]) : 0.0;
      const double M = f == 0 ? S[fk * plane + p] : w.MD[((long long)(f - 1) * NC + k) * plane + p];
      if (mode == 1) {
        // L = -(F_{i+1/2} - F_{i-1/2}) / dx [- (G_{j+1/2} - G_{j-1/2}) / dy] [+ source]
        double L = fu.mul(dF, mix);
        if (DIM == 2) L = fma(dG, miy, L);
        if (src && k == 2) L = fu.add(L, src2);
        if (src && k == 3) L = fu.add(L, src3);
        Lout[fk * plane + p] = L;
        Mout[fk * plane + p] = M;
        continue;
      }
      // b M + b dt L
      double v = stage == 0 ? M : fu.mul(bkr, M);
      if (src && k == 2) v = fma(bdt, src2, v);
      if (src && k == 3) v = fma(bdt, src3, v);
      if (DIM == 2) v = fma(cy, dG, v);
      v = fma(cx, dF, v);
      if (stage == 0) {
        w.B[fk * plane + p] = M;
        S[fk * plane + p] = v;
      } else {
        S[fk * plane + p] = fma(akr, w.B[fk * plane + p], v);
      }
    }
  }
}

// The CFL step for the wavespeeds axs, ays at time t, clamped to the end time te (if positive)
template <int DIM>
__device__ __forceinline__ double cfl_dt(const Grid& g, double axs, double ays, double t, double te) {
  double dt = DIM == 2 ? g.cfl / fma(axs, g.inv_dx, ays * g.inv_dy) : g.cfl * g.dx / axs;
  if (te > 0.0 && t + dt > te) dt = fmax(te - t, 0.0);
  return dt;
}

// The step size of a stage: dt_fixed > 0, or (dt_fixed <= 0) at stage 0 the CFL step from the
// wavespeed slot (clamped to t_end); stages 1 and 2 reuse the value stored in scal[0].
template <int DIM>
__device__ __forceinline__ double stage_dt(const Grid& g, const Work& w, int stage, double dt_fixed, int slot) {
  if (stage != 0) return w.scal[0];
  if (dt_fixed > 0.0) return dt_fixed;
  return cfl_dt<DIM>(g, __longlong_as_double((long long)w.alpha[slot * w.astride]),
                     __longlong_as_double((long long)w.alpha[slot * w.astride + 1]), w.scal[1], w.scal[2]);
}

// dt of stage 0 is stored in scal[0] by block 0 and reused by stages 1 and 2; the time advances
// at stage 2.
template <int DIM, int SYS, int VAR>
__global__ void __launch_bounds__(kThreads) k_update(Grid g, double* __restrict__ S, Work w, int mode, int stage,
                                                      double a_k, double b_k, double dt_fixed, int slot,
                                                      double* __restrict__ Lout, double* __restrict__ Mout) {
  __shared__ double s_dt;
  if (g.listed && blockIdx.x == 0 && threadIdx.x == 0) w.status[2] = w.status[3] = 0u;
  if (mode == 0) {
    if (threadIdx.x == 0) {
      const double dt = stage_dt<DIM>(g, w, stage, dt_fixed, slot);
      if (stage == 0 && blockIdx.x == 0) w.scal[0] = dt;
      s_dt = dt;
    }
    __syncthreads();
  }
  const long long p = (long long)blockIdx.x * kThreads + threadIdx.x;
  if (p >= g.plane) return;
  const double dt = mode == 0 ? s_dt : 0.0;
  // a CFL step at the end time has dt = 0: it leaves the state as it is, so that steps issued
  // past the end time (without waiting for the host) change nothing
  if (mode == 0 && dt_fixed <= 0.0 && dt == 0.0) return;
  update_body<DIM, SYS, VAR>(g, S, w, mode, stage, a_k, b_k, dt, p, Lout, Mout);
  if (mode == 0 && stage == 2 && p == 0) {
    w.scal[1] += dt;
    w.scal[3] += 1.0;  // steps taken
  }
}

// R2: face states of the ghost cells at both ends of every line (the low ghost's right-face
// state, the high ghost's left-face state), from the ghost's own stencil and characteristic
// fields through the boundary map.  Threads: [dir][end][line], gstride lines per (dir, end).
template <int DIM>
__global__ void __launch_bounds__(kThreads) k_r2_ghost(Grid g, const double* __restrict__ S, Work w) {
  constexpr int NC = Traits<DIM, SYS_EULER>::NC;
  const long long gs = w.gstride;
  const long long t = (long long)blockIdx.x * kThreads + threadIdx.x;
  const int dir = (int)(t / (2 * gs));
  const int end = (int)((t / gs) % 2);
  const int line = (int)(t % gs);
  if (dir >= DIM) return;
  const int n = dir == 0 ? g.nx : g.ny, nlines = dir == 0 ? g.ny : g.nx;
  if (line >= nlines) return;
  const int a0 = end == 0 ? -1 : n;
  const int i = dir == 0 ? 0 : line, j = dir == 0 ? line : 0;  // the line's coordinates
  double U3[3][NC], D3[3][NC];
  load_stencil3<DIM, SYS_EULER, 1, NC>(g, S, dir, i, j, a0, nullptr, U3, D3);
  // eigenvectors of the ghost's own state (normal frame)
  const double* U = U3[1];
  const double ir = rcp(U[0]);
  const double u = U[1] * ir, v = DIM == 2 ? U[2] * ir : 0.0;
  const double ke = DIM == 2 ? fma(U[1], u, U[2] * v) : U[1] * u;
  const double pr = g.gm1 * fma(-0.5, ke, U[NC - 1]);
  const double H = (U[NC - 1] + pr) * ir;
  const double c2 = g.gamma * pr * ir;
  const double ic = rsqrt(c2);
  Eig<NC> e;
  e.setup(u, v, H, c2 * ic, ic, g.gm1);
  double md[NC], fs[4][NC];
  r2_cell<NC, SYS_EULER>(U3, D3, e, dir, g, md, fs, fu_of(w.scal));
  double* G = w.GFS + (long long)(dir * 2 + end) * 2 * NC * gs;
  const int q0 = end == 0 ? 0 : 2;
  const long long gl = HW_IDX(line, gs);
#pragma unroll
  for (int k = 0; k < NC; ++k) {
    G[(0 * NC + k) * gs + gl] = fs[q0][k];
    G[(1 * NC + k) * gs + gl] = fs[q0 + 1][k];
  }
}

// alpha of a state only (hweno_max_wavespeed)
template <int DIM, int SYS>
__global__ void __launch_bounds__(kThreads) k_wavespeed(Grid g, const double* __restrict__ S, Work w, int slot) {
  constexpr int NC = Traits<DIM, SYS>::NC;
  const long long plane = g.plane;
  const long long p = (long long)blockIdx.x * kThreads + threadIdx.x;
  double wsx = 0.0, wsy = 0.0;
  if (p < plane) {
    if (SYS == SYS_EULER) {
      double U[NC];
#pragma unroll
      for (int k = 0; k < NC; ++k) U[k] = S[k * plane + p];
      const double ir = rcp(U[0]);
      const double u = U[1] * ir, v = DIM == 2 ? U[2] * ir : 0.0;
      const double ke = DIM == 2 ? fma(U[1], u, U[2] * v) : U[1] * u;
      const double pr = g.gm1 * fma(-0.5, ke, U[NC - 1]);
      const double c = sqrt(g.gamma * pr * ir);
      wsx = fabs(u) + c;
      wsy = DIM == 2 ? fabs(v) + c : 0.0;
      if (!(U[0] > 0.0) || !(pr > 0.0) || !isfinite(wsx) || !isfinite(wsy)) atomicOr(w.status, 1u);
    } else if (SYS == SYS_BURGERS) {
      wsx = fabs(S[p]);
      wsy = DIM == 2 ? wsx : 0.0;
    } else {
      wsx = fabs(g.ax);
      wsy = DIM == 2 ? fabs(g.ay) : 0.0;
    }
  }
  block_max2(wsx, wsy, w.alpha + slot * w.astride);
}

}  // namespace hw
