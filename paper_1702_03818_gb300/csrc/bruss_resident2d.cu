// Brusselator whole job in FP64 for small grids: every stage of every step in one cooperative launch, the state in
// registers.  The persistent kernel of bruss2d.cu spends a 200^2 stage of 5.8 us on 3.9 us of FP64 issue (264 cells an
// SM are 9 warps, 3 of them on one sub-partition, 41 FP64 instructions of 64 clocks each) and on storing the stage,
// a fence, a flag, its polling and reading the stage back through L2.
//
// Units, edges and packets are those of pass_resident2d.cu, with the two species on the two half-warps: lanes 0 .. 15
// hold the complex v of 16 columns, lanes 16 .. 31 the complex w, and the halves share the reaction terms (one forms
// Re v^2 and Re v^2 w, the other the imaginary parts).  That is 21 FP64 instructions a row of 16 cells against 20.5,
// in pieces that spread over the sub-partitions; a cell's operations are those of k_bruss2d (results 2e-14 apart: the
// compiler contracts other products there).  The reaction terms, which need no neighbour, are formed while the edges
// travel.  us a stage, persistent kernel / here: 64^2 4.2 / 2.0, 200^2 5.8 / 4.4, 300^2 9.4 / 8.0, 388 x 535 22.3 / 18.5;
// of the 4.4 at 200^2, 3.3 are FP64 issue, the rest the edges' trip, the barrier and the chain of a row.
#include <algorithm>
#include <memory>

#include <cuda_runtime.h>

#include "frkc2.h"
#include "frkc2_internal.h"
#include "resident2d.cuh"

namespace frkc2 {
namespace {

constexpr int BZ_MAXS = 1024;
constexpr int BZ_RMAX = 7;  // (8 rows a warp spill, and no grid is faster with them than in the persistent kernel)
constexpr int bz_wmax(int R) { return R <= 2 ? 24 : 16; }  // warps (units) of a CTA

struct BrussResidentArgs {
  double* v;            // caller's real state, read at the start and written at the end
  double* w;
  ulonglong2* pk;       // packets, zeroed before the launch
  unsigned* status;
  int nx, ny, periodic;
  int nstrip, nband, cw, rh;  // CTAs across and up, units of a CTA across and up
  int nsteps, s;
  int fault_inject;     // testing only: the first wait is for a stage number that nothing publishes
  long long wait_limit; // polls
  double Dd, A, B1, B;  // D / dx^2, A, B + 1, B
  double hr[BZ_MAXS];   // dt Re a_l
  double hi[BZ_MAXS];   // dt Im a_l
};

// packets of a CTA: [parity][N: cw x 32, S: cw x 32, E: rh x 2R, W: rh x 2R][real, imaginary]
__host__ __device__ inline int bz_packet_half(int cw, int rh, int R) { return 128 * cw + 8 * R * rh; }

template <int R>
__global__ void __launch_bounds__(32 * bz_wmax(R), 1) k_bruss_resident(const BrussResidentArgs a) {
  extern __shared__ double edge[];  // [parity][receiving warp][side][real, imaginary][32]
  constexpr unsigned FULL = 0xffffffffu;
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5, sp = lane >> 4, slot = lane & 15;
  const int nx = a.nx, ny = a.ny, cw = a.cw, rh = a.rh;
  const int UC = a.nstrip * cw, UR = a.nband * rh;
  const int ui = int(blockIdx.x) % a.nstrip * cw + wid % cw, uj = int(blockIdx.x) / a.nstrip * rh + wid / cw;
  const int x0 = int((long long)ui * nx / UC), w = int((long long)(ui + 1) * nx / UC) - x0;
  const int y0 = int((long long)uj * ny / UR), rv = int((long long)(uj + 1) * ny / UR) - y0;
  const int x = x0 + slot;
  const bool colv = slot < w, full = rv == R;  // (a unit has R or R - 1 rows)
  auto local = [&](int par, int warp, int side) { return edge + (((par * nw + warp) * 4 + side) * 2) * 32; };

  // the four sides: where this warp's edge goes and where the neighbour's arrives
  const int half = bz_packet_half(cw, rh, R);
  const int off[4] = {0, 64 * cw, 128 * cw, 128 * cw + 4 * R * rh};
  int mode[4], to_warp[4], put[4], get[4];  // packet indices
#pragma unroll
  for (int d = 0; d < 4; ++d) {
    int ni = ui + (d == SIDE_E) - (d == SIDE_W), nj = uj + (d == SIDE_N) - (d == SIDE_S);
    mode[d] = EDGE_REMOTE;
    if (a.periodic) {
      ni = ni < 0 ? UC - 1 : (ni == UC ? 0 : ni);
      nj = nj < 0 ? UR - 1 : (nj == UR ? 0 : nj);
    } else if (ni < 0 || ni >= UC || nj < 0 || nj >= UR) {
      mode[d] = EDGE_NONE;  // zero flux: the ghost cell repeats the boundary cell
      ni = ui;
      nj = uj;
    }
    const int nb = nj / rh * a.nstrip + ni / cw;
    to_warp[d] = nj % rh * cw + ni % cw;
    if (mode[d] == EDGE_REMOTE && nb == int(blockIdx.x)) mode[d] = EDGE_LOCAL;
    const int row_in = d < 2 ? wid % cw * 32 + lane : wid / cw * 2 * R + sp * R + min(slot, R - 1);
    const int row_out = d < 2 ? ni % cw * 32 + lane : nj % rh * 2 * R + sp * R;
    get[d] = int(blockIdx.x) * 2 * half + off[d] + 2 * row_in;
    put[d] = nb * 2 * half + off[d ^ 1] + 2 * row_out;
  }

  double Xr[R], Xi[R];  // the lane's species
  double* __restrict__ state = sp ? a.w : a.v;
#pragma unroll
  for (int r = 0; r < R; ++r) {
    Xr[r] = Xi[r] = 0.0;
    if (colv && r < rv && in_bounds(x < nx && y0 + r < ny, a.status)) Xr[r] = state[size_t(y0 + r) * nx + x];
  }
  // the lanes whose east / west neighbour is another unit's, or the wall's ghost cell
  const bool east = slot == w - 1 && mode[SIDE_E] != EDGE_NONE, east_wall = slot == w - 1 && !east;
  const bool west = slot == 0 && mode[SIDE_W] != EDGE_NONE, west_wall = slot == 0 && !west;
  const double cR = sp ? a.B : -a.B1;  // the linear reaction term's coefficient of v

  bool bad = false, wait = true;
  unsigned seq = 0;
  int par = 0;
  for (int step = 0; step < a.nsteps; ++step) {
    for (int l = 0; l < a.s; ++l, par ^= 1) {
      ++seq;
      // publish the edges
      const double topr = full ? Xr[R - 1] : Xr[R > 1 ? R - 2 : 0], topi = full ? Xi[R - 1] : Xi[R > 1 ? R - 2 : 0];
#pragma unroll
      for (int d = 0; d < 2; ++d) {
        const double er = d == SIDE_N ? topr : Xr[0], ei = d == SIDE_N ? topi : Xi[0];
        if (mode[d] == EDGE_REMOTE) {
          if (colv) {
            put_packet(a.pk + put[d] + par * half, er, seq);
            put_packet(a.pk + put[d] + par * half + 1, ei, seq);
          }
        } else if (mode[d] == EDGE_LOCAL) {
          double* q = local(par, to_warp[d], d ^ 1);
          q[lane] = er;
          q[32 + lane] = ei;
        }
      }
#pragma unroll
      for (int d = 2; d < 4; ++d)
        if (slot == (d == SIDE_E ? w - 1 : 0)) {
          double* q = local(par, to_warp[d], d ^ 1);
#pragma unroll
          for (int r = 0; r < R; ++r)
            if (r < R - 1 || full) {
              if (mode[d] == EDGE_REMOTE) {
                put_packet(a.pk + put[d] + par * half + 2 * r, Xr[r], seq);
                put_packet(a.pk + put[d] + par * half + 2 * r + 1, Xi[r], seq);
              } else if (mode[d] == EDGE_LOCAL) {
                q[sp * 16 + r] = Xr[r];
                q[32 + sp * 16 + r] = Xi[r];
              }
            }
        }
      // the reaction terms, a third of the FP64 work, while the edges travel
      double gr[R], gi[R];
#pragma unroll
      for (int r = 0; r < R; ++r) {
        const double xr = Xr[r], xi = Xi[r];
        // v^2 and v^2 w: the v half forms the real parts, the w half the imaginary ones
        const double or_ = __shfl_xor_sync(FULL, xr, 16), oi = __shfl_xor_sync(FULL, xi, 16);
        const double vr = sp ? or_ : xr, vi = sp ? oi : xi;
        const double t = __dmul_rn(sp ? vr : vi, vi);
        const double q = fma(sp ? t : vr, sp ? 1.0 : vr, flip(t, !sp));
        const double qo = __shfl_xor_sync(FULL, q, 16);
        const double qr = sp ? qo : q, qi = sp ? q : qo;
        const double wR = sp ? xr : or_, wI = sp ? xi : oi;
        const double u = __dmul_rn(qi, sp ? wR : wI);
        const double p = fma(qr, sp ? wI : wR, flip(u, !sp));
        const double po = __shfl_xor_sync(FULL, p, 16);
        const double pr = sp ? po : p, pi = sp ? p : po;
        gr[r] = __dadd_rn(fma(cR, vr, sp ? flip(pr, true) : a.A), sp ? 0.0 : pr);
        gi[r] = fma(cR, vi, flip(pi, sp));
      }
      __syncthreads();
      // the neighbours' edges (lane sp * 16 + r takes row r of the west and east ones)
      double hr[4], hi[4];
#pragma unroll
      for (int d = 0; d < 4; ++d) {
        const double* q = local(par, wid, d);
        hr[d] = mode[d] == EDGE_LOCAL ? q[lane] : (d == SIDE_N ? topr : Xr[0]);
        hi[d] = mode[d] == EDGE_LOCAL ? q[32 + lane] : (d == SIDE_N ? topi : Xi[0]);
      }
      if (wait) {
        const unsigned want = a.fault_inject ? FULL : seq;
        long long polls = 0;
        bool miss[4];
#pragma unroll
        for (int d = 0; d < 4; ++d) miss[d] = mode[d] == EDGE_REMOTE && (d < 2 ? colv : slot < rv);
        while (true) {
#pragma unroll
          for (int d = 0; d < 4; ++d)
            if (miss[d]) {
              const bool re = get_packet(a.pk + get[d] + par * half, hr[d], want);
              miss[d] = !(get_packet(a.pk + get[d] + par * half + 1, hi[d], want) && re);
            }
          if (!__any_sync(FULL, miss[0] || miss[1] || miss[2] || miss[3])) break;
          if (++polls > a.wait_limit) {
            if (lane == 0) atomicOr(a.status, ST_TIMEOUT);
            wait = false;
            break;
          }
        }
      }
      const double cr = a.hr[l], ci = a.hi[l];
      const bool last = l == a.s - 1;
      double Sr = hr[SIDE_S], Si = hi[SIDE_S];
#pragma unroll
      for (int r = 0; r < R; ++r) {
        const double xr = Xr[r], xi = Xi[r];
        double Er = __shfl_down_sync(FULL, xr, 1, 16), Ei = __shfl_down_sync(FULL, xi, 1, 16);
        double Wr = __shfl_up_sync(FULL, xr, 1, 16), Wi = __shfl_up_sync(FULL, xi, 1, 16);
        const double er = __shfl_sync(FULL, hr[SIDE_E], r, 16), ei = __shfl_sync(FULL, hi[SIDE_E], r, 16);
        const double wr_ = __shfl_sync(FULL, hr[SIDE_W], r, 16), wi_ = __shfl_sync(FULL, hi[SIDE_W], r, 16);
        Er = east ? er : (east_wall ? xr : Er);
        Ei = east ? ei : (east_wall ? xi : Ei);
        Wr = west ? wr_ : (west_wall ? xr : Wr);
        Wi = west ? wi_ : (west_wall ? xi : Wi);
        const bool top = r == R - 1 || (r == R - 2 && !full);
        const double Nr = (top ? hr[SIDE_N] : Xr[r + 1 < R ? r + 1 : r]), Ni = (top ? hi[SIDE_N] : Xi[r + 1 < R ? r + 1 : r]);
        const double Lr = fma(-4.0, xr, __dadd_rn(__dadd_rn(Er, Wr), __dadd_rn(Nr, Sr)));
        const double Li = fma(-4.0, xi, __dadd_rn(__dadd_rn(Ei, Wi), __dadd_rn(Ni, Si)));
        const double fr = fma(a.Dd, Lr, gr[r]);
        const double fi = fma(a.Dd, Li, gi[r]);
        const double nr = fma(-ci, fi, fma(cr, fr, xr)), ni = fma(ci, fr, fma(cr, fi, xi));
        Sr = xr;
        Si = xi;
        const bool live = colv && (r < R - 1 || full);
        Xr[r] = (live ? nr : xr);
        Xi[r] = live && !last ? ni : 0.0;  // step output: the real part
        bad |= last && live && (__double2hiint(nr) & 0x7ff00000) == 0x7ff00000;
      }
    }
  }
#pragma unroll
  for (int r = 0; r < R; ++r)
    if (colv && r < rv && in_bounds(x < nx && y0 + r < ny, a.status)) state[size_t(y0 + r) * nx + x] = Xr[r];
  if (bad) atomicOr(a.status, ST_NONFINITE);
}

struct BrussResidentShape {
  int cw, rh, nstrip, nband, R;  // R 0: no shape
  double us;                     // modelled, a stage
};

// The shape of the least modelled time, fitted to 300 shapes at 11 grids from 33 x 21 to 700 x 200 (mean deviation 5 %;
// it picks the fastest at each): FP64 instructions of the SM (16 clocks each over its sub-partitions), a warp's own chain
// of them, barrier and edges per warp.  200^2: 20 warps of 1 row 4.49 us, 10 of 2 4.67, 7 of 3 4.98, 4 of 5 5.94.
BrussResidentShape bruss_resident_shape(int nx, int ny, int sms, size_t bytes) {
  BrussResidentShape best{};
  for (int cw = 1; cw <= 4; cw *= 2)
    for (int rh = 1; cw * rh <= bz_wmax(1); ++rh) {
      const int nw = cw * rh, nstrip = (nx + 16 * cw - 1) / (16 * cw);
      if (nstrip > sms || nstrip * cw > nx || ny < rh) continue;
      const int nband = std::min(sms / nstrip, ny / rh), R = (ny + nband * rh - 1) / (nband * rh);
      if (R > BZ_RMAX || nw > bz_wmax(R)) continue;
      if (size_t(nstrip) * nband * 2 * bz_packet_half(cw, rh, R) * sizeof(ulonglong2) > bytes) continue;
      const double us = 0.31 + (0.145 * nw + 0.59) * R + 0.045 * nw;
      if (!best.R || us <= best.us) best = {cw, rh, nstrip, nband, R, us};
    }
  return best;
}

template <int R>
cudaError_t launch_r(const BrussResidentArgs& a, cudaStream_t st) {
  constexpr size_t per_warp = 2 * 4 * 2 * 32 * sizeof(double);
  static SmemLimit smem;
  const cudaError_t attr = smem.raise(k_bruss_resident<R>, per_warp * bz_wmax(R));
  if (attr != cudaSuccess) return attr;
  void* args[] = {const_cast<BrussResidentArgs*>(&a)};
  const cudaError_t e = cudaLaunchCooperativeKernel((const void*)k_bruss_resident<R>, dim3(a.nstrip * a.nband),
                                                    dim3(32 * a.cw * a.rh), args, per_warp * a.cw * a.rh, st);
  if (e == cudaSuccess) count_launch();
  return e;
}

}  // namespace

// Where the model's time, with 3 % for its error (8 % for 7 rows, whose registers spill), is below what the
// persistent kernel takes at least, the lower edge of 60 grids measured with both: 2.8 us + 0.0625 per 1000 cells, at
// least 4.2, and steps with its CTAs a SM above that (resident / persistent us: 64 x 53 3.4 / 4.4, 183 x 176 3.8 / 5.2,
// 395 x 238 8.7 / 9.6, 255 x 720 16.3 / 19.2; on the other side 420 x 269 11.3 / 10.4, 147 x 1816 26.3 / 22.6: strips and
// bands of uneven units).
bool bruss_resident_wins(const frkc2_bruss_problem& p, int s, int nsteps, size_t packet_bytes) {
  if (p.precision != FRKC2_FP64 || s > BZ_MAXS || (long long)nsteps * s >= 0x7fffffffll) return false;
  if (p.nx * p.ny > (1 << 20)) return false;
  const CoopDevice d = coop_device();
  if (!d.coop) return false;
  const BrussResidentShape sh = bruss_resident_shape(int(p.nx), int(p.ny), d.sms, packet_bytes);
  const double cells = double(p.nx) * double(p.ny), per_sm = cells / (256.0 * d.sms);
  const double persistent = per_sm > 6.0 ? 22.4 : per_sm > 4.0 ? 19.0 : std::max(4.2, 2.8 + 0.0625e-3 * cells);
  return sh.R > 0 && sh.us * (sh.R >= 7 ? 1.08 : 1.03) <= persistent;
}

cudaError_t launch_bruss_resident(const frkc2_bruss_problem& p, const frkc2_plan_s& plan, double dt, int nsteps, double* v, double* w,
                                  void* packets, size_t packet_bytes, unsigned* status, long long wait_limit, int fault_inject,
                                  cudaStream_t st) {
  const BrussResidentShape sh = bruss_resident_shape(int(p.nx), int(p.ny), coop_device().sms, packet_bytes);
  if (!sh.R) return cudaErrorInvalidValue;
  const size_t used = size_t(sh.nstrip) * sh.nband * 2 * bz_packet_half(sh.cw, sh.rh, sh.R) * sizeof(ulonglong2);
  const cudaError_t e = cudaMemsetAsync(packets, 0, used, st);
  if (e != cudaSuccess) return e;
  auto a = std::make_unique<BrussResidentArgs>();
  a->v = v;
  a->w = w;
  a->pk = static_cast<ulonglong2*>(packets);
  a->status = status;
  a->nx = int(p.nx);
  a->ny = int(p.ny);
  a->periodic = p.bc == FRKC2_BC_PERIODIC;
  a->nstrip = sh.nstrip;
  a->nband = sh.nband;
  a->cw = sh.cw;
  a->rh = sh.rh;
  a->nsteps = nsteps;
  a->s = plan.s;
  a->fault_inject = fault_inject;
  a->wait_limit = wait_limit > 0 ? wait_limit : RESIDENT_WAIT;
  a->Dd = p.D / (p.dx * p.dx);
  a->A = p.A;
  a->B1 = p.B + 1.0;
  a->B = p.B;
  for (int l = 0; l < plan.s; ++l) {
    a->hr[l] = dt * plan.a_re[l];
    a->hi[l] = dt * plan.a_im[l];
  }
  switch (sh.R) {
    case 1: return launch_r<1>(*a, st);
    case 2: return launch_r<2>(*a, st);
    case 3: return launch_r<3>(*a, st);
    case 4: return launch_r<4>(*a, st);
    case 5: return launch_r<5>(*a, st);
    case 6: return launch_r<6>(*a, st);
    default: return launch_r<7>(*a, st);
  }
}

}  // namespace frkc2
