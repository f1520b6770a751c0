// CFL or fixed-dt steps of one small 1D grid in one cooperative launch.
//
// A 1D grid of up to 152 x 124 cells cannot fill the GPU: its three kernels per stage each wait for one
// thread's chain of FP64 instructions (68 cycles each, however many lanes are active), for the launch
// and for the loads from L2 that replace what the previous kernel knew.  Here every block keeps its
// cells in shared memory for all stages of all steps and each thread one cell and one face; per stage
// there is one grid barrier, before which the blocks publish the two cells at each of their ends and
// the largest wavespeed of their updated cells.  The arithmetic is that of the stage kernels with the
// FP64 weights (the same device functions on a block-local grid whose ghost cells are filled in), so
// the results are theirs.  What bounds it is that chain: about 520 FP64 instructions of one warp per Euler
// stage, 17 us.  Ten CFL steps of 1D Euler at 2048 cells 1.235 to 0.844 ms (28 us a stage against 41), at
// 16383 cells 1.239 to 0.844 ms; 267 steps of advection at 160 cells 14.4 to 7.1 ms (8.8 us a stage).
#include <cooperative_groups.h>

#include "hweno_host.cuh"

namespace cg = cooperative_groups;
using namespace hwh;

namespace hw {

constexpr int kLineStride = kThreads;  // a block's cells and two ghost cells at each end

// the wavespeed slots and the toggle that the launches take in turn, behind the stage slots
// alpha[0..7]: [8] the number of launches, [9 + 4 set + slot] the slots of a set, all zero between
// launches of that set
constexpr int kLineToggle = 8, kLineSlots = 9;

struct LineArgs {
  int nsteps;
  double dt_fixed;
  double* halo;  // [2][block][2 ends][2 cells][fields x components]
};

template <int SYS>
__global__ void __launch_bounds__(kThreads) k_line_steps(Grid g, double* __restrict__ S, Work w, LineArgs a) {
  constexpr int NC = Traits<1, SYS>::NC, NV = 2 * NC, W = kLineStride;
  __shared__ double sS[NV * W], sB[NV * W], sMD[NC * W], sNOD[NV * W], sFX[NV * (W + 1)];
  __shared__ float2 sPRIM[NC * W];
  __shared__ unsigned long long s_max[kThreads / 32];
  cg::grid_group grid = cg::this_grid();
  const int nb = gridDim.x, b = blockIdx.x, t = threadIdx.x;
  // the block's cells: n0 .. n0 + m - 1 at local indices 2 .. m + 1
  const int base = g.nx / nb, extra = g.nx % nb;
  const int n0 = b * base + (b < extra ? b : extra), m = base + (b < extra ? 1 : 0);
  Grid gl = g;
  gl.nx = m + 4;
  gl.plane = W;
  gl.bc = BC_TRANSMISSIVE;  // never met by what is used: the ghost cells are there
  gl.pairs = 0;
  Work wl = w;
  wl.B = sB;
  wl.MD = sMD;
  wl.NOD = sNOD;
  wl.PRIM = sPRIM;
  wl.FX = sFX;
  const PairSlots none{nullptr};
  const FU f = fu_of(w.scal);
  const bool own = t < m, owner = b == 0 && t == 0;

  // own cells, and the ghost cells of the first stage through the boundary map
  for (int l = t; l < m + 4; l += kThreads) {
    bool refl;
    const long long p = HW_IDX(bc_map(n0 + l - 2, g.nx, g.bc, refl), g.plane);
    for (int v = 0; v < NV; ++v) {
      const bool flip = refl && ((v < NC) == (v % NC == 1));
      sS[v * W + l] = neg_if(S[v * g.plane + p], SYS == SYS_EULER && flip);
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
      for (int k = 0; k < NC; ++k) U[k] = sS[k * W + t + 2];
      CellState<1, SYS>().set(U, g, f, ws, wy);
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
    if (st == 0) {
      dt = a.dt_fixed;
      if (dt <= 0.0) {
        dt = cfl_dt<1>(g, alpha, 0.0, time, t_end);
        if (dt == 0.0) {  // the end time is reached: nothing changes any more
          if (owner) {
            w.scal[0] = 0.0;
            w.alpha[2] = w.alpha[4] = bits;
          }
          break;
        }
      }
      if (owner) w.scal[0] = dt;
    }
    // cells: the nodal values of all, the modified derivatives of the block's own
    double wsx = 0.0, wsy = 0.0;
    if (t < m + 4) {
      cell_body<1, SYS, 0>(gl, sS, wl, t, wsx, wsy, none);
      if (t >= 2 && t < m + 2) cell_limiter<1, SYS, 0>(gl, sS, wl, t, 0);
    }
    __syncthreads();
    // faces 2 .. m + 2
    if (t <= m) face_body<1, SYS, 0, false>(gl, sS, wl, 0, t + 2, alpha, none);
    __syncthreads();
    if (own) update_body<1, SYS, 0>(gl, sS, wl, 0, st, a_k[st], b_k[st], dt, t + 2, nullptr, nullptr);
    if (st == 2) {
      time += dt;
      steps += 1.0;
    }
    if (s + 1 == stages) break;
    __syncthreads();
    // publish, meet, fill the ghost cells
    double* const halo = a.halo + (size_t)(s & 1) * nb * 4 * NV;
    if (t < 4 * NV) {  // end, cell, value
      const int end = t / (2 * NV), c = t / NV % 2, v = t % NV;
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
  if (own)
    for (int v = 0; v < NV; ++v) S[v * g.plane + HW_IDX(n0 + t, g.plane)] = sS[v * W + t + 2];
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
  constexpr int kCells = hw::kLineStride - 4;
  const int nb = (int)((h->nx + kCells - 1) / kCells);
  if (nb > sms) return HWENO_OK;
  hw::LineArgs a;
  a.dt_fixed = dt;
  a.halo = h->w.FX;  // free on this path: 2 x blocks x 4 cells of at most (nx + 1) cells' values
  static void (*const kern[3])(Grid, double*, Work, hw::LineArgs) = {
      hw::k_line_steps<hw::SYS_ADV>, hw::k_line_steps<hw::SYS_BURGERS>, hw::k_line_steps<hw::SYS_EULER>};
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
    const cudaError_t e = cudaLaunchKernelEx(&cfg, kern[h->system], g, h->state, h->w, a);
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
