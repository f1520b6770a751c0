// CFL or fixed-dt steps of one small 1D grid in one cooperative launch.
//
// A 1D grid of up to 152 x 124 cells cannot fill the GPU: its three kernels per stage each wait for one
// thread's chain of FP64 instructions (68 cycles each, however many lanes are active), for the launch
// and for the loads from L2 that replace what the previous kernel knew.  Here every block keeps its
// cells in shared memory for all stages of all steps; per stage there is one grid barrier, before which
// the blocks publish the two cells at each of their ends and the largest wavespeed of their updated
// cells.  The arithmetic is that of the stage kernels with the FP64 weights, operation for operation, on a
// block-local grid whose ghost cells are filled in.
//
// What bounds it is the chain of one warp: each of an SM's four schedulers has its own FP64 pipe, so a
// block of four warps is four chains side by side.  Two forms:
//   ROLES = 1: each thread one cell and one face, 124 cells a block; about 750 FP64 instructions per
//              Euler stage and warp, 25 us of the 28 us that a stage takes.
//   ROLES = 4 (up to 152 x 28 cells): the four warps of a block share 28 cells: the two sides of the
//              faces, the nodal values and D-terms, the modified derivatives at once, then the values
//              of the fluxes and of the update dealt out: about 290 instructions.
// Ten CFL steps of 1D Euler at 2048 cells: 1.235 ms by stage kernels, 0.844 ms with ROLES = 1, 0.351 ms
// with 4 (11.7 us a stage); at 16383 cells 1.236 to 0.851 ms (ROLES = 1); the 267 steps of advection at
// 160 cells 14.3, 7.1 and 4.0 ms (5.0 us a stage).
#include <cooperative_groups.h>

#include "hweno_host.cuh"

namespace cg = cooperative_groups;
using namespace hwh;

namespace hw {

// the wavespeed slots and the toggle that the launches take in turn, behind the stage slots
// alpha[0..7]: [8] the number of launches, [9 + 4 set + slot] the slots of a set, all zero between
// launches of that set
constexpr int kLineToggle = 8, kLineSlots = 9;
static_assert(kLineSlots + 2 * 4 <= hwh::kAlphaWords, "the layout holds both sets");

struct LineArgs {
  int nsteps;
  double dt_fixed;
  double* halo;  // [2][block][2 ends][2 cells][fields x components]
};

// One side of the faces 2 .. m + 2 of a block (normal frame): the state and derivative at face fa from
// the cells fa-2 .. fa (side 0) or fa-1 .. fa+1 (side 1) of S (stride W), as r1_face_states takes them,
// and their flux and Jacobian product.  Lane l of the warp holds face l + 2 and the primitives of cell
// l + 1, up to lane m + 1's cell m + 2; the lanes behind repeat what the last ones do.
template <int SYS, int W>
__device__ __forceinline__ void line_side(const Grid& g, const double* S, int side, int lane, int m, const FU& f,
                                          double* U, double* D, double* F, double* H) {
  constexpr int NC = Traits<1, SYS>::NC;
  const int c = (lane <= m ? lane : m) + 1 + side;  // the stencil's centre
  const int pc = (lane <= m ? lane : m + 1) + 1;    // the cell of the primitives
  double dl[NC], dr[NC], yl[NC], yr[NC];
#pragma unroll
  for (int k = 0; k < NC; ++k) {
    const double u = S[k * W + c];
    dl[k] = f.sub(u, S[k * W + c - 1]);
    dr[k] = f.sub(S[k * W + c + 1], u);
    yl[k] = S[(NC + k) * W + c - 1];
    yr[k] = S[(NC + k) * W + c + 1];
    const double k21 = g.uvd[0][0], k3 = g.uvd[0][1];
    D[k] = side == 0 ? fma(k21, dr[k], fma(-k3, dl[k], fma(0.0625, yl[k], -0.1875 * yr[k])))
                     : fma(k21, dl[k], fma(-k3, dr[k], fma(-0.1875, yl[k], 0.0625 * yr[k])));
  }
  Eig<NC> e;
  double wl[NC], wr[NC], zl[NC], zr[NC], w[NC];
  if (SYS == SYS_EULER) {
    // those of cell fa from the next lane; their Roe average
    double q[NC];
#pragma unroll
    for (int k = 0; k < NC; ++k) q[k] = S[k * W + pc];
    const double ir = rcp(q[0], f), ul = f.mul(q[1], ir);
    const double pr = g.gm1 * fma(-0.5, f.mul(q[1], ul), q[NC - 1]);
    const double Hl = f.mul(f.add(q[NC - 1], pr), ir), sl = sqrt_fast(q[0], f);
    const double ur = __shfl_down_sync(0xffffffffu, ul, 1), Hr = __shfl_down_sync(0xffffffffu, Hl, 1);
    const double sr = __shfl_down_sync(0xffffffffu, sl, 1);
    const double iw = rcp(f.add(sl, sr), f);
    const double ub = f.mul(fma(sl, ul, f.mul(sr, ur)), iw), Hb = f.mul(fma(sl, Hl, f.mul(sr, Hr)), iw);
    const double c2 = g.gm1 * fma(-0.5, f.mul(ub, ub), Hb), ic = rsqrt_full(c2, f);
    e.setup(ub, 0.0, Hb, f.mul(c2, ic), ic, g.gm1);
    e.project(dl, wl, f);
    e.project(dr, wr, f);
    e.project(yl, zl, f);
    e.project(yr, zr, f);
  } else {
    wl[0] = dl[0];
    wr[0] = dr[0];
    zl[0] = yl[0];
    zr[0] = yr[0];
  }
  const StencilK k = stencil_k(g, 0, f);
  const double half = side == 0 ? k.half : -k.half;
#pragma unroll
  for (int s = 0; s < NC; ++s) {
    double du, sv;
    const double e0 = beta0_eps(wl[s], wr[s], zl[s], zr[s], k, du, sv, f);
    const Wts wt = weights_e(e0, fma(wl[s], wl[s], k.eps), fma(wr[s], wr[s], k.eps), k.quarter, f);
    const double* co = side == 0 ? k.cm : k.cp;
    const double r = fma(co[0], wl[s], fma(co[1], wr[s], fma(co[2], zl[s], f.mul(co[3], zr[s]))));
    const double sl = fma(wt.W1, wl[s], f.mul(wt.W2, wr[s]));
    const double rden = rcp(fma(k.G, wt.W0, f.add(wt.W1, wt.W2)), f);
    w[s] = fma(fma(wt.W0, r, f.mul(half, sl)), rden, SYS == SYS_EULER ? 0.0 : S[c]);
  }
  double base[NC];
#pragma unroll
  for (int q = 0; q < NC; ++q) base[q] = S[q * W + c];
  if (SYS == SYS_EULER)
    e.back_add(w, base, U, f);
  else
    U[0] = w[0];
  Phys<1, SYS>::flux_jvp(U, D, F, H, g.ax, g.gm1, f);
}

template <int SYS, int ROLES>
__global__ void __launch_bounds__(kThreads) k_line_steps(Grid g, double* __restrict__ S, Work w, LineArgs a) {
  constexpr int NC = Traits<1, SYS>::NC, NV = 2 * NC, W = kThreads / ROLES;  // W: a block's cells and four ghosts
  __shared__ double sS[NV * W], sB[NV * W], sMD[NC * W], sNOD[NV * W], sFX[NV * (W + 1)];
  __shared__ float2 sPRIM[NC * W];
  __shared__ double sSide[ROLES == 4 ? 2 * 4 * NC * W : 1], sD[ROLES == 4 ? 5 * NC * W : 1], s_dt;
  __shared__ unsigned long long s_max[kThreads / 32];
  cg::grid_group grid = cg::this_grid();
  const int nb = gridDim.x, b = blockIdx.x, t = threadIdx.x, lane = t % W, role = t / W;
  // the block's cells: n0 .. n0 + m - 1 at local indices 2 .. m + 1
  const int base = g.nx / nb, extra = g.nx % nb;
  const int n0 = b * base + (b < extra ? b : extra), m = base + (b < extra ? 1 : 0);
  Grid gl = g;
  gl.nx = m + 4;
  gl.plane = W;
  gl.bc = BC_TRANSMISSIVE;  // never met by what is used: the ghost cells are there
  Work wl = w;
  wl.B = sB;
  wl.MD = sMD;
  wl.NOD = sNOD;
  wl.PRIM = sPRIM;
  wl.FX = sFX;
  const PairSlots none{nullptr};
  const FU f = fu_of(w.scal);
  const bool own = role == 0 && lane < m, owner = b == 0 && t == 0;

  // own cells, and the ghost cells of the first stage through the boundary map
  if (lane < m + 4) {
    bool refl;
    const long long p = HW_IDX(bc_map(n0 + lane - 2, g.nx, g.bc, refl), g.plane);
    for (int v = role; v < NV; v += ROLES) {
      const bool flip = refl && ((v < NC) == (v % NC == 1));
      sS[v * W + lane] = neg_if(S[v * g.plane + p], SYS == SYS_EULER && flip);
    }
  }
  const unsigned int launches = (unsigned int)w.alpha[kLineToggle];
  unsigned long long* const slots = w.alpha + kLineSlots + 4 * (launches & 1u);
  unsigned long long* const next = w.alpha + kLineSlots + 4 * (~launches & 1u);
  double time = w.scal[1], steps = w.scal[3], dt = 0.0;
  const double t_end = w.scal[2];
  __syncthreads();

  // the largest wavespeed of the block's cells into a slot
  auto publish_speed = [&](unsigned long long* slot) {
    double ws = 0.0, wy;
    if (own) {
      double U[NC];
#pragma unroll
      for (int k = 0; k < NC; ++k) U[k] = sS[k * W + lane + 2];
      CellState<1, SYS, false>().set(U, g, f, ws, wy);
    }
    if (ROLES == 4) {
      if (role == 0) {
        const unsigned long long x = warp_max(speed_bits(ws));
        if (lane == 0) atomicMax(slot, x);
      }
      return;
    }
    const unsigned long long x = warp_max(speed_bits(ws));
    if ((t & 31) == 0) s_max[t >> 5] = x;
    __syncthreads();
    if (t == 0) {
      unsigned long long y = s_max[0];
#pragma unroll
      for (int q = 1; q < kThreads / 32; ++q) y = s_max[q] > y ? s_max[q] : y;
      atomicMax(slot, y);
    }
  };
  publish_speed(slots);
  grid.sync();
  if (owner) {
    w.alpha[kLineToggle] = launches + 1u;
    next[0] = next[1] = next[2] = 0ull;
  }

  const double a_k[3] = {0.0, 0.75, 1.0 / 3.0}, b_k[3] = {1.0, 0.25, 2.0 / 3.0};
  const int stages = 3 * a.nsteps;
  for (int s = 0, st = 0; s < stages; ++s, st = st == 2 ? 0 : st + 1) {
    const unsigned long long bits = __ldcg(slots + s % 3);
    const double alpha = __longlong_as_double((long long)bits);
    if (owner) {
      slots[(s + 2) % 3] = 0ull;
      w.alpha[2 * st] = bits;
    }
    if (st == 0 && (ROLES == 1 || role == 3)) {
      dt = a.dt_fixed > 0.0 ? a.dt_fixed : cfl_dt<1>(g, alpha, 0.0, time, t_end);
      if (ROLES == 4 && lane == 0) s_dt = dt;
    }
    if (ROLES == 1) {
      // cells: the nodal values of all, the modified derivatives of the block's own; then faces 2 .. m + 2
      double wsx = 0.0, wsy = 0.0;
      if (t < m + 4) {
        cell_body<1, SYS, 0, false, false>(gl, sS, wl, t, wsx, wsy, none);
        if (t >= 2 && t < m + 2) cell_limiter<1, SYS, 0>(gl, sS, wl, t, 0);
      }
      __syncthreads();
      if (t <= m) face_body<1, SYS, 0, false, true>(gl, sS, wl, 0, t + 2, alpha, none);
      __syncthreads();
    } else {
      if (role < 2) {
        double U[NC], D[NC], F[NC], H[NC];
        line_side<SYS, W>(gl, sS, role, lane, m, f, U, D, F, H);
        if (lane <= m)
#pragma unroll
          for (int k = 0; k < NC; ++k) {
            double* o = sSide + ((role * 4) * NC + k) * W + lane;
            o[0] = U[k];
            o[NC * W] = D[k];
            o[2 * NC * W] = F[k];
            o[3 * NC * W] = H[k];
          }
      } else if (role == 2) {
        double wsx = 0.0, wsy = 0.0;
        if (lane < m + 4) cell_body<1, SYS, 0, false, false>(gl, sS, wl, lane, wsx, wsy, none);
        __syncwarp();
        if (lane <= m)
#pragma unroll
          for (int k = 0; k < NC; ++k) {
            // the sums of the D-terms (Eqs. Cd-1, DfDh) of face lane + 2
            const double *n0_ = sNOD + k * W + lane, *n1 = n0_ + NC * W;
            const double f0 = n0_[0], f1 = n0_[1], f2 = n0_[2], f3 = n0_[3], ha = n1[0], hb = n1[3];
            double* o = sD + 5 * k * W + lane;
            o[0] = f.add(f.sub(f0, f1), f.sub(f3, f2));
            o[W] = f.sub(ha, hb);
            o[2 * W] = f.sub(f0, f3);
            o[3 * W] = f.sub(f2, f1);
            o[4 * W] = f.add(ha, hb);
          }
      } else if (lane >= 2 && lane < m + 2) {
        cell_limiter<1, SYS, 0>(gl, sS, wl, lane, 0);
      }
      __syncthreads();
      dt = s_dt;
    }
    if (st == 0) {
      if (owner) w.scal[0] = dt;
      if (a.dt_fixed <= 0.0 && dt == 0.0) {  // the end time is reached: nothing changes any more
        if (owner) w.alpha[2] = w.alpha[4] = bits;
        break;
      }
    }
    if (ROLES == 1) {
      if (own) update_body<1, SYS, 0>(gl, sS, wl, 0, st, a_k[st], b_k[st], dt, t + 2, nullptr, nullptr);
    } else {
      // the fluxes (Eq. flux-LF), a value per warp in turn, then the update of the same value
      const double bdt = f.mul(b_k[st], dt), cx = f.mul(bdt, -g.inv_dx);
      for (int v = role; v < NV; v += 4) {
        const int fld = v < NC ? 0 : 1, k = v - fld * NC;
        double F = 0.0;
        if (lane <= m) {
          const double *lo = sSide + (fld * NC + k) * W + lane, *hi = lo + 4 * NC * W, *q = sD + 5 * k * W + lane;
          const double vis = f.mul(-0.5 * alpha, f.sub(hi[0], lo[0]));
          const double D = fld == 0 ? fma(DCoef::cf, q[0], fma(g.chh[0], q[W], vis))
                                    : fma(g.efih[0], q[2 * W], fma(g.egih[0], q[3 * W], fma(DCoef::eh, q[4 * W], vis)));
          F = fma(0.5, f.add(lo[2 * NC * W], hi[2 * NC * W]), D);
        }
        const double Fr = __shfl_down_sync(0xffffffffu, F, 1);
        if (lane < m) {
          const int l = lane + 2;
          const double M = fld == 0 ? sS[v * W + l] : sMD[k * W + l];
          const double x = fma(cx, f.sub(Fr, F), st == 0 ? M : f.mul(b_k[st], M));
          if (st == 0) {
            sB[v * W + l] = M;
            sS[v * W + l] = x;
          } else {
            sS[v * W + l] = fma(a_k[st], sB[v * W + l], x);
          }
        }
      }
    }
    if (st == 2) {
      time += dt;
      steps += 1.0;
    }
    if (s + 1 == stages) break;
    __syncthreads();
    // publish, meet, fill the ghost cells
    double* const halo = a.halo + (size_t)(s & 1) * nb * 4 * NV;
    const int ht = kThreads - 1 - t;  // the last threads: the first warp has the wavespeeds to do
    if (ht < 4 * NV) {  // end, cell, value
      const int end = ht / (2 * NV), c = ht / NV % 2, v = ht % NV;
      halo[((size_t)b * 4 + end * 2 + c) * NV + v] = sS[v * W + (end == 0 ? 2 + c : m + c)];
    }
    publish_speed(slots + (s + 1) % 3);
    grid.sync();
    if (t < 4 * NV) {
      const int end = t / (2 * NV), c = t / NV % 2, v = t % NV;  // ghost cells c = 0, 1 from the left
      const int l = end == 0 ? c : m + 2 + c;
      const bool edge = end == 0 ? b == 0 : b == nb - 1;
      double x;
      if (!edge || g.bc == BC_PERIODIC) {
        const int o = end == 0 ? (b == 0 ? nb - 1 : b - 1) : (b == nb - 1 ? 0 : b + 1);
        x = __ldcg(&halo[((size_t)o * 4 + (1 - end) * 2 + c) * NV + v]);
      } else if (g.bc == BC_TRANSMISSIVE) {
        x = sS[v * W + (end == 0 ? 2 : m + 1)];
      } else {  // mirrored about the wall
        x = neg_if(sS[v * W + (end == 0 ? 3 - c : m + 1 - c)], SYS == SYS_EULER && ((v < NC) == (v % NC == 1)));
      }
      sS[v * W + l] = x;
    }
    __syncthreads();
  }
  if (owner) {
    w.scal[1] = time;
    w.scal[3] = steps;
  }
  __syncthreads();
  if (lane < m)
    for (int v = role; v < NV; v += ROLES) S[v * g.plane + HW_IDX(n0 + lane, g.plane)] = sS[v * W + lane + 2];
}

}  // namespace hw

namespace hwh {

unsigned int bounds_take_line(int* line) {
#ifdef HWENO_BOUNDS_CHECK
  return hw::bounds_take(line);
#else
  if (line) *line = 0;
  return 0;
#endif
}

// Declared in hweno_host.cuh.
int line_steps(hweno_ctx* h, double dt, int nsteps, bool* done) {
  *done = false;
  if (h->dim != 1 || h->var != 0 || h->profiling || h->nx > kLineMaxCells || nsteps <= 0) return HWENO_OK;
  int dev = 0, sms = 0;
  if (cudaGetDevice(&dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
    return HWENO_ECUDA;
  // four warps to 28 cells while there are SMs for the blocks (28 to 12 us a stage of 1D Euler), else a
  // thread to a cell: a second block on an SM would share the schedulers' FP64 pipes with the first
  const bool roles = h->nx <= (int64_t)sms * (hw::kThreads / 4 - 4);
  const int cells = (roles ? hw::kThreads / 4 : hw::kThreads) - 4;
  const int nb = (int)((h->nx + cells - 1) / cells);
  if (nb > sms) return HWENO_OK;
  hw::LineArgs a;
  a.dt_fixed = dt;
  // free on this path, and large enough: 2 x blocks x 4 cells' values in (nx + 1) cells' rounded up to 256 bytes
  a.halo = h->w.FX;
  static void (*const kern[2][3])(Grid, double*, Work, hw::LineArgs) = {
      {hw::k_line_steps<hw::SYS_ADV, 1>, hw::k_line_steps<hw::SYS_BURGERS, 1>, hw::k_line_steps<hw::SYS_EULER, 1>},
      {hw::k_line_steps<hw::SYS_ADV, 4>, hw::k_line_steps<hw::SYS_BURGERS, 4>, hw::k_line_steps<hw::SYS_EULER, 4>}};
  const Grid g = grid_of(h);
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)nb);
  cfg.blockDim = dim3(hw::kThreads);
  cfg.stream = h->stream;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeCooperative;
  attr[0].val.cooperative = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  constexpr int kMost = 4096;  // steps of one launch
  for (int k = 0; k < nsteps; k += kMost) {
    a.nsteps = nsteps - k < kMost ? nsteps - k : kMost;
    const cudaError_t e = cudaLaunchKernelEx(&cfg, kern[roles ? 1 : 0][h->system], g, h->state, h->w, a);
    if (e == cudaErrorCooperativeLaunchTooLarge && k == 0) {
      cudaGetLastError();  // fewer SMs than the device's: the stage kernels
      return HWENO_OK;
    }
    if (e != cudaSuccess) return HWENO_ECUDA;
    h->launches += 1;
  }
  *done = true;
  return HWENO_OK;
}

}  // namespace hwh
