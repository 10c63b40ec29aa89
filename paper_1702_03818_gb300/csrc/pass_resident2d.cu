// Whole-job kernel for small FP64 2D grids (fixed conductivity): every stage of every step in one cooperative
// launch, the state in registers.  With a launch per stage a 256^2 stage takes 4.7 us, of which its FP64 work is
// 1.7: the rest is launch, ramp and load latency.
//
// The grid is cut into UC x UR units of at most 16 columns and R rows, one warp each: lanes 0 .. 15 hold U of a
// unit's columns, lanes 16 .. 31 V (the FP64 pipe of an SM sub-partition takes 64 clocks for a warp instruction
// whatever its lanes do, so half-warp columns spread a grid more evenly over the 4 x SMs sub-partitions: 256^2 is
// 1216 units of 3 or 4 rows, 34 FP64 instructions a stage for each and 2 units a sub-partition).  A CTA is cw x rh
// neighbouring units, at most one CTA an SM.  256^2: 5.9 us a stage as one launch each at the full grid, 4.7 with the
// launches spread over the SMs, 3.0 here: 2.1 of FP64 issue and about 0.9 for the edges' trip through L2.
// Per stage a warp publishes its four edges, forms the differences inside the unit, takes its neighbours' edges and
// updates its cells (a cell's operations and their order are those of the streaming pass, whose unrolled rows the
// compiler contracts in either of two ways: the same bits or 4e-15 apart).  Edges go to
// warps of the same CTA through shared memory, at one CTA barrier a stage, and to other CTAs as 16-byte packets,
// two 64-bit words that hold half a value and the stage number each: a reader that sees the number has the
// value (resident2d.cuh), so there is no fence, flag or second trip through L2.  A slot is written again two stages on; by then the
// writer has read the neighbour's edge of the stage between, which the neighbour published after reading the
// slot.  Every wait is bounded: when it runs out the warp latches the time-out status and goes on without
// waiting, so the launch ends.
#include <algorithm>
#include <memory>

#include <cuda_runtime.h>

#include "frkc2_internal.h"
#include "resident2d.cuh"

namespace frkc2 {
namespace {

constexpr int RS_MAXS = 1024;
constexpr int RS_RMAX = 8;
constexpr int RS_WMAX = 16;  // warps (units) of a CTA

struct Resident2dArgs {
  double* u;            // caller's real state, read at the start and written at the end
  const double* fx;     // [ny][nx + 1], face x between columns x - 1 and x
  const double* fy;     // [ny + 1][nx]
  ulonglong2* pk;       // packets, zeroed before the launch
  unsigned* status;
  int nx, ny, periodic;
  int nstrip, nband, cw, rh;  // CTAs across and up, units of a CTA across and up
  int nsteps, s;
  int fault_inject;     // testing only: the first wait is for a stage number that nothing publishes
  long long wait_limit; // polls
  double ca[RS_MAXS];   // dt Re a_l / dx^2
  double cb[RS_MAXS];   // dt Im a_l / dx^2
};

// packets of a CTA: [parity][N: cw x 32, S: cw x 32, E: rh x 2R, W: rh x 2R]
__host__ __device__ inline int packet_half(int cw, int rh, int R) { return 64 * cw + 4 * R * rh; }

template <int R>
__global__ void __launch_bounds__(32 * RS_WMAX, 1) k_resident2d(const Resident2dArgs a) {
  __shared__ double edge[2][RS_WMAX][4][32];  // [parity][receiving warp][side]
  constexpr unsigned FULL = 0xffffffffu;
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, comp = lane >> 4, slot = lane & 15;
  const int nx = a.nx, ny = a.ny, cw = a.cw, rh = a.rh;
  const int UC = a.nstrip * cw, UR = a.nband * rh;
  const int ui = int(blockIdx.x) % a.nstrip * cw + wid % cw, uj = int(blockIdx.x) / a.nstrip * rh + wid / cw;
  const int x0 = int((long long)ui * nx / UC), w = int((long long)(ui + 1) * nx / UC) - x0;
  const int y0 = int((long long)uj * ny / UR), rv = int((long long)(uj + 1) * ny / UR) - y0;
  const int x = x0 + slot;
  const bool colv = slot < w, full = rv == R;  // (a unit has R or R - 1 rows)

  // the four sides: where this warp's edge goes and where the neighbour's arrives
  const int half = packet_half(cw, rh, R);
  const int off[4] = {0, 32 * cw, 64 * cw, 64 * cw + 2 * R * rh};
  int mode[4];
  int to_warp[4];
  int put[4], get[4];  // packet indices
#pragma unroll
  for (int d = 0; d < 4; ++d) {
    int ni = ui + (d == SIDE_E) - (d == SIDE_W), nj = uj + (d == SIDE_N) - (d == SIDE_S);
    mode[d] = EDGE_REMOTE;
    if (a.periodic) {
      ni = ni < 0 ? UC - 1 : (ni == UC ? 0 : ni);
      nj = nj < 0 ? UR - 1 : (nj == UR ? 0 : nj);
    } else if (ni < 0 || ni >= UC || nj < 0 || nj >= UR) {
      mode[d] = EDGE_NONE;
      ni = ui;
      nj = uj;
    }
    const int nb = nj / rh * a.nstrip + ni / cw;
    to_warp[d] = nj % rh * cw + ni % cw;
    if (mode[d] == EDGE_REMOTE && nb == int(blockIdx.x)) mode[d] = EDGE_LOCAL;
    const int o = d ^ 1;  // the neighbour's side
    const int row_in = d < 2 ? wid % cw * 32 + lane : wid / cw * 2 * R + comp * R + min(slot, R - 1);
    const int row_out = d < 2 ? ni % cw * 32 + lane : nj % rh * 2 * R + comp * R;
    get[d] = int(blockIdx.x) * 2 * half + off[d] + row_in;
    put[d] = nb * 2 * half + off[o] + row_out;
  }

  double X[R], kE[R], kW[R], kN[R], kS = 0.0;
#pragma unroll
  for (int r = 0; r < R; ++r) {
    X[r] = kE[r] = kW[r] = kN[r] = 0.0;
    if (colv && r < rv && in_bounds(x < nx && y0 + r < ny, a.status)) {
      const size_t y = size_t(y0 + r);
      if (comp == 0) X[r] = a.u[y * nx + x];
      kE[r] = a.fx[y * (nx + 1) + x + 1];
      kW[r] = a.fx[y * (nx + 1) + x];
      kN[r] = a.fy[(y + 1) * nx + x];
      if (r == 0) kS = a.fy[y * nx + x];
    }
  }

  bool bad = false, wait = true;
  unsigned seq = 0;
  int par = 0;
  for (int step = 0; step < a.nsteps; ++step) {
    for (int l = 0; l < a.s; ++l, par ^= 1) {
      ++seq;
      // publish the edges
      const double top = full ? X[R - 1] : X[R > 1 ? R - 2 : 0];
      if (mode[SIDE_N] == EDGE_REMOTE) {
        if (colv) put_packet(a.pk + put[SIDE_N] + par * half, top, seq);
      } else if (mode[SIDE_N] == EDGE_LOCAL) {
        edge[par][to_warp[SIDE_N]][SIDE_S][lane] = top;
      }
      if (mode[SIDE_S] == EDGE_REMOTE) {
        if (colv) put_packet(a.pk + put[SIDE_S] + par * half, X[0], seq);
      } else if (mode[SIDE_S] == EDGE_LOCAL) {
        edge[par][to_warp[SIDE_S]][SIDE_N][lane] = X[0];
      }
      if (slot == w - 1) {
#pragma unroll
        for (int r = 0; r < R; ++r) {
          if (r < R - 1 || full) {
            if (mode[SIDE_E] == EDGE_REMOTE)
              put_packet(a.pk + put[SIDE_E] + par * half + r, X[r], seq);
            else if (mode[SIDE_E] == EDGE_LOCAL)
              edge[par][to_warp[SIDE_E]][SIDE_W][comp * 16 + r] = X[r];
          }
        }
      }
      if (slot == 0) {
#pragma unroll
        for (int r = 0; r < R; ++r) {
          if (r < R - 1 || full) {
            if (mode[SIDE_W] == EDGE_REMOTE)
              put_packet(a.pk + put[SIDE_W] + par * half + r, X[r], seq);
            else if (mode[SIDE_W] == EDGE_LOCAL)
              edge[par][to_warp[SIDE_W]][SIDE_E][comp * 16 + r] = X[r];
          }
        }
      }
      // differences inside the unit, and the west column's values on the lanes that take the west edge (lane
      // comp * 16 + r takes row r of the west and east edges)
      double dN[R], xw = 0.0;
#pragma unroll
      for (int r = 0; r < R; ++r) {
        dN[r] = r + 1 < R ? X[r + 1 < R ? r + 1 : r] - X[r] : 0.0;
        const double v = __shfl_sync(FULL, X[r], 0, 16);
        if (slot == r) xw = v;
      }
      // the neighbours' edges
      __syncthreads();
      double h[4];
#pragma unroll
      for (int d = 0; d < 4; ++d) h[d] = mode[d] == EDGE_LOCAL ? edge[par][wid][d][lane] : 0.0;
      if (wait) {
        const unsigned want = a.fault_inject ? FULL : seq;
        long long polls = 0;
        while (true) {
          bool ready = true;
#pragma unroll
          for (int d = 0; d < 4; ++d)
            if (mode[d] == EDGE_REMOTE && (d < 2 ? colv : slot < rv)) ready &= get_packet(a.pk + get[d] + par * half, h[d], want);
          if (__all_sync(FULL, ready)) break;
          if (++polls > a.wait_limit) {
            if (lane == 0) atomicOr(a.status, ST_TIMEOUT);
            wait = false;
            break;
          }
        }
      }
      const double dWe = xw - h[SIDE_W];
      const double dTop = h[SIDE_N] - top;
      double dS = X[0] - h[SIDE_S];
      const double ca = a.ca[l], cb = flip(a.cb[l], comp == 0);
      const bool last = l == a.s - 1;
      double ks = kS;
#pragma unroll
      for (int r = 0; r < R; ++r) {
        double e = __shfl_down_sync(FULL, X[r], 1, 16);
        const double eh = __shfl_sync(FULL, h[SIDE_E], r, 16), wh = __shfl_sync(FULL, dWe, r, 16);
        if (slot == w - 1) e = eh;
        const double dE = e - X[r];
        double dW = __shfl_up_sync(FULL, dE, 1, 16);
        if (slot == 0) dW = wh;
        if (r == R - 1 || (r == R - 2 && !full)) dN[r] = dTop;
        const double f = fma(kE[r], dE, fma(-kW[r], dW, fma(kN[r], dN[r], -__dmul_rn(ks, dS))));
        const double fo = __shfl_xor_sync(FULL, f, 16);  // the other component's
        const double v = fma(cb, fo, fma(ca, f, X[r]));
        if (colv && (r < R - 1 || full)) {
          if (last) {  // step output: the real part
            if (comp == 0) bad |= (__double2hiint(v) & 0x7ff00000) == 0x7ff00000;
            X[r] = comp ? 0.0 : v;
          } else {
            X[r] = v;
          }
        }
        dS = dN[r];
        ks = kN[r];
      }
    }
  }
#pragma unroll
  for (int r = 0; r < R; ++r)
    if (comp == 0 && colv && r < rv && in_bounds(x < nx && y0 + r < ny, a.status)) a.u[size_t(y0 + r) * nx + x] = X[r];
  if (bad) atomicOr(a.status, ST_NONFINITE);
}

struct ResidentShape {
  int cw, rh, nstrip, nband, R;  // R 0: no shape
  double us;                     // modelled, a stage
};

// The shape of the least modelled time, fitted to 250 shapes at 13 grids from 33 x 21 to 700 x 400 (it picks the
// fastest, or one within 1 %, at each): FP64 instructions a stage of the fullest sub-partition (64 clocks each; a
// single warp there doesn't keep the pipe busy), a warp's own chain of them, and a cost per warp of the CTA for
// barrier and edges.  256^2: 8 warps of 4 rows 3.10 us, 10 of 3 3.16, 14 of 2 3.24, 4 of 7 4.09; 100^2: 5 of 1 row
// 1.33, 4 of 2 1.79.
ResidentShape resident_shape(int nx, int ny, int sms, size_t bytes) {
  ResidentShape best{};
  for (int cw = 1; cw <= 4; cw *= 2)
    for (int rh = 1; cw * rh <= RS_WMAX; ++rh) {
      const int nw = cw * rh, nstrip = (nx + 16 * cw - 1) / (16 * cw);
      if (nstrip > sms || nstrip * cw > nx || ny < rh) continue;
      const int nband = std::min(sms / nstrip, ny / rh), R = (ny + nband * rh - 1) / (nband * rh);
      if (R > RS_RMAX) continue;
      if (size_t(nstrip) * nband * 2 * packet_half(cw, rh, R) * sizeof(ulonglong2) > bytes) continue;
      const double us = 0.56 + (0.027 * std::max(1.5, double((nw + 3) / 4)) + 0.015) * (8 * R + 2) + 0.03 * nw;
      if (!best.R || us <= best.us) best = {cw, rh, nstrip, nband, R, us};
    }
  return best;
}

template <int R>
cudaError_t launch_r(const Resident2dArgs& a, cudaStream_t st) {
  void* args[] = {const_cast<Resident2dArgs*>(&a)};
  const cudaError_t e =
      cudaLaunchCooperativeKernel((const void*)k_resident2d<R>, dim3(a.nstrip * a.nband), dim3(32 * a.cw * a.rh), args, 0, st);
  if (e == cudaSuccess) count_launch();
  return e;
}

}  // namespace

// Wherever a shape fits (up to about 550^2: 16 warps of 8 rows on every SM; not narrower or lower than the units of a
// CTA): us a stage, resident against a launch of the streaming pass per stage: 8 x 5 0.86 / 2.8, 100^2 1.3 / 3.0,
// 256^2 3.1 / 4.7, 512^2 8.9 / 10.8, 700 x 400 10.1 / 11.5.  The clearing of the packets and the cooperative launch
// take what they save in 4 stages at the largest grids (500^2, one step: s = 4 59.5 us against 59.1; 130 x 97 26 / 30).
bool resident2d_wins(const frkc2_problem& p, int s, int nsteps, size_t packet_bytes) {
  if (p.ndim != 2 || p.precision != FRKC2_FP64 || p.kappa_kind == FRKC2_KAPPA_POWER || s > RS_MAXS) return false;
  if ((long long)nsteps * s < 4) return false;
  if ((long long)nsteps * s >= 0x7fffffffll || p.n[0] * p.n[1] > (1 << 20)) return false;
  const CoopDevice d = coop_device();
  return d.coop && resident_shape(int(p.n[0]), int(p.n[1]), d.sms, packet_bytes).R > 0;
}

cudaError_t launch_resident2d(const frkc2_problem& p, const frkc2_plan_s& plan, double dt, int nsteps, void* u, const void* fx,
                              const void* fy, void* packets, size_t packet_bytes, unsigned* status, long long wait_limit,
                              int fault_inject, cudaStream_t st) {
  const ResidentShape sh = resident_shape(int(p.n[0]), int(p.n[1]), coop_device().sms, packet_bytes);
  if (!sh.R) return cudaErrorInvalidValue;
  const size_t used = size_t(sh.nstrip) * sh.nband * 2 * packet_half(sh.cw, sh.rh, sh.R) * sizeof(ulonglong2);
  const cudaError_t e = cudaMemsetAsync(packets, 0, used, st);
  if (e != cudaSuccess) return e;
  auto a = std::make_unique<Resident2dArgs>();
  a->u = static_cast<double*>(u);
  a->fx = static_cast<const double*>(fx);
  a->fy = static_cast<const double*>(fy);
  a->pk = static_cast<ulonglong2*>(packets);
  a->status = status;
  a->nx = int(p.n[0]);
  a->ny = int(p.n[1]);
  a->periodic = p.bc == FRKC2_BC_PERIODIC;
  a->nstrip = sh.nstrip;
  a->nband = sh.nband;
  a->cw = sh.cw;
  a->rh = sh.rh;
  a->nsteps = nsteps;
  a->s = plan.s;
  a->fault_inject = fault_inject;
  a->wait_limit = wait_limit > 0 ? wait_limit : RESIDENT_WAIT;
  const double h2 = p.dx * p.dx;
  for (int l = 0; l < plan.s; ++l) {
    a->ca[l] = dt * plan.a_re[l] / h2;
    a->cb[l] = dt * plan.a_im[l] / h2;
  }
  switch (sh.R) {
    case 1: return launch_r<1>(*a, st);
    case 2: return launch_r<2>(*a, st);
    case 3: return launch_r<3>(*a, st);
    case 4: return launch_r<4>(*a, st);
    case 5: return launch_r<5>(*a, st);
    case 6: return launch_r<6>(*a, st);
    case 7: return launch_r<7>(*a, st);
    default: return launch_r<8>(*a, st);
  }
}

}  // namespace frkc2
