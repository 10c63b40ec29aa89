// 3D single-stage pass (k = 1) streaming along z, for every conductivity kind and precision.
//
// A CTA is nw warps; warp w holds the RY grid rows y = by OY + w RY - 1 .. + RY - 1 and lane l is
// column x = bx 30 + l - 1, so the CTA covers a 32 x (RY nw) column block whose outer lanes and rows
// are halo: it outputs the 30 x OY columns inside, OY = RY nw - 2.  It walks up z; each thread keeps
// its RY columns' W and conductivity at z and z + 1 and the flux through their down faces in
// registers.  Per plane:
//   - each cell forms the fluxes through its east, north and up faces, F = kappa_f (W_nb - W_c); the
//     west flux is lane - 1's east flux (shuffle), the down flux the up flux of the plane below
//     (register), and inside a thread's rows the south flux is the north flux of the row below:
//     f = (F_e - F_w) + (F_n - F_s) + (F_u - F_d), every face flux formed once (MIXED: see flux);
//   - between warps, the y exchange runs one plane ahead: a warp publishes its first row's W and
//     kappa of plane z + 1 and its last row's north flux of plane z (formed during plane z - 1) in
//     the same double-buffered shared write, so one barrier a plane serves both directions;
//   - for kappa(u) = 1 + c u^p every cell's kappa(W) is evaluated once per stage (when its plane is
//     loaded); for FIELD / CONST the cell conductivities are read (4 or 8 bytes a cell, where the
//     three face arrays are 12 or 24).  A face takes kappa_c + kappa_nb, the factor 1/2 folded into
//     the stage coefficients (exact).
// Rows that are halo, or lie outside the grid, skip the x and z fluxes and the update.
//
// Work split: column blocks x chunks along z; neighbouring blocks of one chunk are neighbours in the
// launch order, so CTAs that run together read the same planes and share halo columns and lines in L2
// (one contiguous range of (block, z) per CTA instead: FP32 256^3 104 us a pass against 94).  nw is chosen
// per grid so that the blocks cover ny with the fewest rows, the chunk count so that the waves are full.
//
// What bounds it: the FP64 pipe.  FP64 kappa(u) takes about 62 FP64 instructions a computed cell (24 for
// kappa(W), 38 for the stencil and the update), FIELD / CONST 24; computed / output cells 1.14 x the
// columns lost at ragged edges.  A pass over 160^3: FP64 kappa(u) 959 -> 668 us, MIXED 266 -> 139 us;
// FP64 periodic FIELD 71 x 90 x 123, a step of 8 stages: 1433 -> 582 us (single rows per warp, two
// barriers a plane, 32-plane chunks, three face arrays before).  FP32: pass_stream3d_f32.cu.
//
// MIXED: double state and differences, float conductivities and fluxes.  Its conversions between
// double and float go through the integer pipe (frkc2_math.cuh), bit for bit the hardware's, because
// a conversion takes a slot of the FP64 pipe like an addition: 10 FP64-pipe instructions a cell
// instead of 20 (121 x 150 x 97, kappa(u), two steps of 16 stages: 5.68 -> 1.91 ms).
#include <algorithm>
#include <type_traits>

#include <cuda_runtime.h>

#include "frkc2_internal.h"
#include "frkc2_math.cuh"

namespace frkc2 {
namespace {

constexpr int S3_OX = 30;          // output columns per CTA
constexpr int S3_CHUNK = 32;       // MIXED: see flux
constexpr int K3_FIELD = 0;        // FIELD / CONST: real conductivity read from memory (or a constant)
constexpr int K3_POWER = 1;        // kappa(u), general exponent
constexpr int K3_P25 = 2;          // kappa(u), exponent 2.5

template <class T> struct V2s;
template <> struct V2s<double> { using type = double2; };
template <> struct V2s<float> { using type = float2; };

__device__ __forceinline__ bool nonfinite3(double v) { return (__double2hiint(v) & 0x7ff00000) == 0x7ff00000; }

// Rows of one thread and the most warps of a CTA.  160^3, kappa(u), a pass: 16 warps FP64 668 us /
// MIXED 139 us; FP64 with 12 warps 669 us, 8 warps (2 CTAs per SM) 703 us, 4 warps (4 CTAs) 771 us:
// with the FP64 pipe the bound, the halo rows of smaller CTAs cost more than they hide.
constexpr int S3_RY = 2, S3_MAXW = 16;

struct S3Args {
  int nx, ny, nz;
  int oy;                   // output rows per CTA
  int bxn;                  // column blocks along x
  int chunks;               // chunks along z
  int in_real, out_real;    // the pass reads / writes the real state instead of interleaved (U, V)
  int check_finite;
  const void* in;
  void* out;
  const void* kappa;        // FIELD: cell conductivities; nullptr: the constant kc
  double kc, kp;
  double ca, cb;            // dt a_l / (2 dx^2): the face factor 1/2 folded in
  unsigned* status;
};

template <class S, class A, int KIND, bool PERIODIC>
__global__ void __launch_bounds__(32 * S3_MAXW) k_stream3d(const S3Args p) {
  constexpr int RY = S3_RY, MAXW = S3_MAXW;
  constexpr bool POWER = KIND != K3_FIELD;
  constexpr bool MIX = !std::is_same<S, A>::value;
  using S2 = typename V2s<S>::type;
  using A2 = typename V2s<A>::type;
  __shared__ S2 shW[2][MAXW][32];   // first row's W of the next plane
  __shared__ A2 shK[2][MAXW][32];   // and its conductivity
  __shared__ A2 shF[2][MAXW][32];   // last row's north flux of this plane
  // launched with programmatic stream serialization: the next launch may start its CTAs as this
  // one's exit, and every global load below comes after the previous launch has completed
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  asm volatile("griddepcontrol.wait;" ::: "memory");
  const int lane = threadIdx.x, w = threadIdx.y, nw = blockDim.y;
  const int nx = p.nx, ny = p.ny, nz = p.nz;
  const size_t plane = size_t(nx) * ny;
  const bool in_real = p.in_real, out_real = p.out_real;
  const S ca = S(p.ca), cb = S(p.cb);
  const A kc = A(p.kc), kp = A(p.kp);
  const S* __restrict__ Ur = static_cast<const S*>(p.in);
  const S2* __restrict__ Wi = static_cast<const S2*>(p.in);
  const A* __restrict__ Kf = static_cast<const A*>(p.kappa);

  const A2 a0 = {A(0), A(0)};
  auto kap = [&](S2 v) -> A2 {
    A2 k = a0;
    if constexpr (KIND == K3_P25) {
      A vx, vy;
      if constexpr (MIX) {
        bool slow = false;
        vx = narrow_fast(v.x, slow);
        vy = narrow_fast(v.y, slow);
        while (__any_sync(0xffffffffu, slow)) {
          vx = narrow_hw(v.x);
          vy = narrow_hw(v.y);
          slow = false;
        }
        kappa_power25_mixed(vx, vy, kc, k.x, k.y);
      } else {
        kappa_power25_fast(v.x, v.y, kc, k.x, k.y);
      }
    } else if constexpr (KIND == K3_POWER) {
      kappa_power<A>(A(v.x), A(v.y), kc, kp, k.x, k.y);
    }
    return k;
  };
  // sum of the two conductivities of a face, and the (twice the) flux
  auto ksum = [&](A2 a, A2 b) -> A2 {
    A2 k = a0;
    k.x = a.x + b.x;
    if (POWER) k.y = a.y + b.y;
    return k;
  };
  // (Which product of the imaginary part is fused is fixed here, so that results depend neither on the
  // compiler's choice nor on where the chunks along z begin: the x and y faces one way, the z faces the
  // other.  MIXED only: plane 32 j takes its down face as the x and y faces, so that this one face of 32 has
  // two fluxes, a float rounding apart.  These are the results that MIXED has had since its chunks were of 32
  // planes; with one flux there the state moves by 5e-9 in norm, 121 x 150 x 97, 32 stages, more than double results may.)
  auto flux = [&](A2 kf, A dr, A di, bool zface) -> A2 {
    A2 F;
    if (POWER) {
      F.x = fma(kf.x, dr, -mul_rn(kf.y, di));
      F.y = zface ? fma(kf.y, dr, mul_rn(kf.x, di)) : fma(kf.x, di, mul_rn(kf.y, dr));
    } else {
      F.x = kf.x * dr;
      F.y = kf.x * di;
    }
    return F;
  };
  // difference of two states in the arithmetic precision
  auto diff = [&](S2 a, S2 b, bool& slow) -> A2 {
    A2 d;
    if constexpr (MIX) {
      d.x = narrow_fast(a.x - b.x, slow);
      d.y = narrow_fast(a.y - b.y, slow);
    } else {
      d.x = a.x - b.x;
      d.y = a.y - b.y;
    }
    return d;
  };
  auto diff_exact = [&](S2 a, S2 b) -> A2 {
    A2 d;
    d.x = narrow_hw(a.x - b.x);
    d.y = narrow_hw(a.y - b.y);
    return d;
  };
  // the flux of one face on its own (the y faces between warps, and the priming planes)
  auto face = [&](S2 a, S2 b, A2 ka, A2 kb, bool zface) -> A2 {
    bool slow = false;
    A2 d = diff(a, b, slow);
    while (MIX && __any_sync(0xffffffffu, slow)) {
      d = diff_exact(a, b);
      slow = false;
    }
    return flux(ksum(ka, kb), d.x, d.y, zface);
  };

  int b = 0;  // exchange buffer
  bool bad = false;
  const int blk = blockIdx.x, z0 = int((long long)blockIdx.y * nz / p.chunks), z1 = int((long long)(blockIdx.y + 1) * nz / p.chunks);
  {
    const int gx = (blk % p.bxn) * S3_OX + lane - 1;
    const int gy0 = (blk / p.bxn) * p.oy + w * RY - 1;
    const bool out_x = lane >= 1 && lane <= 30 && gx < nx;
    // per row: the in-plane offset read (wrapped, or clamped to the grid: the conductivity of a
    // Dirichlet ghost is its interior cell's), whether the row is in the grid / an output row, and
    // whether a neighbour needs it
    size_t col[RY];
    unsigned inside = 0, act = 0, need = 0;  // bits by row; act and need are warp-uniform
    const bool xin = PERIODIC || (gx >= 0 && gx < nx);
    const int xr = PERIODIC ? wrap3(gx, nx) : min(max(gx, 0), nx - 1);
#pragma unroll
    for (int r = 0; r < RY; ++r) {
      const int gy = gy0 + r, R = w * RY + r;
      const int yr = PERIODIC ? wrap3(gy, ny) : min(max(gy, 0), ny - 1);
      col[r] = size_t(yr) * nx + xr;
      if (xin && (PERIODIC || (gy >= 0 && gy < ny))) inside |= 1u << r;
      if (R >= 1 && R <= p.oy && gy < ny) act |= 1u << r;
      if (gy <= ny) need |= 1u << r;
    }
    auto zrow = [&](int z) -> size_t { return size_t(PERIODIC ? wrap3(z, nz) : min(max(z, 0), nz - 1)) * plane; };
    auto load = [&](int z, size_t zo, int r) -> S2 {
      S2 v;
      v.x = v.y = S(0);
      if (!PERIODIC && (z < 0 || z >= nz)) return v;
      if (!(inside >> r & 1) || !in_bounds(zo + col[r] < size_t(nz) * plane, p.status)) return v;
      if (in_real)
        v.x = __ldg(Ur + zo + col[r]);
      else
        v = __ldg(Wi + zo + col[r]);
      return v;
    };
    auto loadk = [&](size_t zo, int r) -> A2 {  // FIELD / CONST
      A2 k = a0;
      k.x = kc;
      if (Kf && in_bounds(zo + col[r] < size_t(nz) * plane, p.status)) k.x = __ldg(Kf + zo + col[r]);
      return k;
    };

    // prime: W and kappa of z0 and z0 + 1, the fluxes through the down faces of z0, and the last
    // row's north flux of plane z0
    S2 Wc[RY], Wp[RY];
    A2 Kc[RY], Kp[RY], Fd[RY], Ft;
    {
      const size_t zm = zrow(z0 - 1), zc = zrow(z0), zp = zrow(z0 + 1);
#pragma unroll
      for (int r = 0; r < RY; ++r) {
        const S2 Wm = load(z0 - 1, zm, r);
        Wc[r] = load(z0, zc, r);
        Wp[r] = load(z0 + 1, zp, r);
        A2 Km;
        if (POWER) {
          Km = kap(Wm);
          Kc[r] = kap(Wc[r]);
          Kp[r] = kap(Wp[r]);
        } else {
          Km = loadk(zm, r);
          Kc[r] = loadk(zc, r);
          Kp[r] = loadk(zp, r);
        }
        Fd[r] = face(Wc[r], Wm, Kc[r], Km, !MIX || z0 % S3_CHUNK != 0);
      }
      shW[b][w][lane] = Wc[0];
      shK[b][w][lane] = Kc[0];
      __syncthreads();
      const int wn = w + 1 < nw ? w + 1 : w;  // (the top halo row's north flux is not used)
      Ft = face(shW[b][wn][lane], Wc[RY - 1], Kc[RY - 1], shK[b][wn][lane], false);
      b ^= 1;
    }
    for (int z = z0; z < z1; ++z) {
      const bool more = z + 1 < z1;
      S2 Wl[RY];  // the plane after next, issued early
      A2 Kl[RY];
      const size_t zl = zrow(z + 2);
#pragma unroll
      for (int r = 0; r < RY; ++r) {
        Wl[r].x = Wl[r].y = S(0);
        Kl[r] = a0;
        if (more) {
          Wl[r] = load(z + 2, zl, r);
          if (!POWER) Kl[r] = loadk(zl, r);
        }
      }
      shW[b][w][lane] = Wp[0];
      shK[b][w][lane] = Kp[0];
      shF[b][w][lane] = Ft;
      __syncthreads();
      A2 Fs = shF[b][w > 0 ? w - 1 : w][lane];  // (the bottom halo row's south flux is not used)
      const int wn = w + 1 < nw ? w + 1 : w;
      const S2 Wnn = shW[b][wn][lane];
      const A2 Knn = shK[b][wn][lane];
      b ^= 1;
      const size_t zo = size_t(z) * plane;
#pragma unroll
      for (int r = 0; r < RY; ++r) {
        A2 Fn = Ft;
        if (r + 1 < RY) Fn = face(Wc[r + 1], Wc[r], Kc[r], Kc[r + 1], false);
        if (act >> r & 1) {
          S2 We;
          A2 Ke = a0;
          We.x = __shfl_down_sync(0xffffffffu, Wc[r].x, 1);
          We.y = __shfl_down_sync(0xffffffffu, Wc[r].y, 1);
          Ke.x = __shfl_down_sync(0xffffffffu, Kc[r].x, 1);
          if (POWER) Ke.y = __shfl_down_sync(0xffffffffu, Kc[r].y, 1);
          bool slow = false;
          A2 dE = diff(We, Wc[r], slow), dU = diff(Wp[r], Wc[r], slow);
          while (MIX && __any_sync(0xffffffffu, slow)) {
            dE = diff_exact(We, Wc[r]);
            dU = diff_exact(Wp[r], Wc[r]);
            slow = false;
          }
          const A2 Fe = flux(ksum(Kc[r], Ke), dE.x, dE.y, false);
          const A2 Fu = flux(ksum(Kc[r], Kp[r]), dU.x, dU.y, true);
          A2 Fw;
          Fw.x = __shfl_up_sync(0xffffffffu, Fe.x, 1);
          Fw.y = __shfl_up_sync(0xffffffffu, Fe.y, 1);
          const A fR = ((Fe.x - Fw.x) + (Fn.x - Fs.x)) + (Fu.x - Fd[r].x);
          const A fI = ((Fe.y - Fw.y) + (Fn.y - Fs.y)) + (Fu.y - Fd[r].y);
          Fd[r] = Fu;
          if (MIX && POWER && (z + 1) % S3_CHUNK == 0) Fd[r] = flux(ksum(Kc[r], Kp[r]), dU.x, dU.y, false);
          S sR, sI;
          if constexpr (MIX) {
            bool sl = false;
            sR = widen_fast(fR, sl);
            sI = widen_fast(fI, sl);
            while (__any_sync(0xffffffffu, sl)) {
              sR = widen_hw(fR);
              sI = widen_hw(fI);
              sl = false;
            }
          } else {
            sR = fR;
            sI = fI;
          }
          if (out_x && in_bounds(zo + col[r] < size_t(nz) * plane, p.status)) {
            const S un = Wc[r].x + ca * sR - cb * sI;
            if (out_real) {
              static_cast<S*>(p.out)[zo + col[r]] = un;
            } else {
              S2 o;
              o.x = un;
              o.y = Wc[r].y + ca * sI + cb * sR;
              static_cast<S2*>(p.out)[zo + col[r]] = o;
            }
            if (p.check_finite) bad |= nonfinite3(un);
          }
        }
        Fs = Fn;
      }
      if (more) {
        Ft = face(Wnn, Wp[RY - 1], Kp[RY - 1], Knn, false);
#pragma unroll
        for (int r = 0; r < RY; ++r) {
          Wc[r] = Wp[r];
          Kc[r] = Kp[r];
          Wp[r] = Wl[r];
          if (!POWER)
            Kp[r] = Kl[r];
          else if (need >> r & 1)
            Kp[r] = kap(Wl[r]);
        }
      }
    }
  }
  if (bad) atomicOr(p.status, ST_NONFINITE);
}

template <class S, class A, int KIND, bool PERIODIC>
cudaError_t launch_t(S3Args a, cudaStream_t st) {
  constexpr int RY = S3_RY, MAXW = S3_MAXW;
  const auto kern = k_stream3d<S, A, KIND, PERIODIC>;
  struct Res {
    cudaError_t err;
    int sms, per_sm[S3_MAXW + 1];
  };
  static const Res res = [kern] {
    Res r{};
    for (int n = 1; n <= MAXW; ++n) {
      const Residency q = query_residency(kern, 32 * n, 0);
      if (q.err != cudaSuccess) r.err = q.err;
      r.sms = q.sms;
      r.per_sm[n] = q.per_sm;
    }
    return r;
  }();
  if (res.err != cudaSuccess) return res.err;
  // warps per CTA: at least half of the most (fewer leave too few rows between the halo rows), the
  // count that covers ny with the fewest rows, the larger of equal ones
  int nw = 0;
  long long best = 0;
  for (int n = MAXW; n >= MAXW / 2; --n) {
    const int oy = RY * n - 2;
    const long long rows = (long long)((a.ny + oy - 1) / oy) * RY * n;
    if (nw == 0 || rows < best) {
      nw = n;
      best = rows;
    }
  }
  a.oy = RY * nw - 2;
  a.bxn = (a.nx + S3_OX - 1) / S3_OX;
  const long long blocks = (long long)a.bxn * ((a.ny + a.oy - 1) / a.oy);
  a.chunks = stream3d_chunks(blocks, a.nz, (long long)res.sms * res.per_sm[nw]);
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(unsigned(blocks), a.chunks, 1);
  cfg.blockDim = dim3(32, nw, 1);
  cfg.dynamicSmemBytes = 0;
  cfg.stream = st;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  const cudaError_t le = cudaLaunchKernelEx(&cfg, kern, a);
  count_launch();
  return le != cudaSuccess ? le : cudaGetLastError();
}

template <class S, class A>
cudaError_t launch_s(const frkc2_problem& p, const S3Args& a, cudaStream_t st) {
  const bool per = p.bc == FRKC2_BC_PERIODIC;
  if (p.kappa_kind != FRKC2_KAPPA_POWER) return per ? launch_t<S, A, K3_FIELD, true>(a, st) : launch_t<S, A, K3_FIELD, false>(a, st);
  if (a.kp == 2.5) return per ? launch_t<S, A, K3_P25, true>(a, st) : launch_t<S, A, K3_P25, false>(a, st);
  return per ? launch_t<S, A, K3_POWER, true>(a, st) : launch_t<S, A, K3_POWER, false>(a, st);
}

}  // namespace

// Chunks along z: of 1 .. min(nz, 256), the count whose waves of CTAs (slots resident at once) take the fewest planes,
// two more per chunk for its priming, the smallest of equal ones.  Column blocks of one chunk are neighbours in the launch
// order, so the CTAs that run together read the same planes and share their halo columns and lines in L2.
// Every stage's launch asks, so it looks only at the smallest count with the chunk length of the most chunks that w waves
// hold, until w waves take more planes however long their chunks are (nz = 250: 1.2 us of the host for a look at every count).
int stream3d_chunks(long long blocks, int nz, long long slots) {
  const int most = std::min(nz, 256);
  int best = 1;
  long long least = (blocks + slots - 1) / slots * (nz + 2);  // one chunk
  for (long long w = (blocks + slots - 1) / slots; blocks * nz + 2 * w * slots < least * slots; ++w) {
    const long long c = std::min<long long>(most, w * slots / blocks), length = (nz + c - 1) / c;
    if (w * (length + 2) < least) {
      best = int((nz + length - 1) / length);
      least = w * (length + 2);
    }
    if (c == most) break;
  }
  return best;
}

cudaError_t launch_pass_stream3d(const frkc2_problem& p, const PassArgs& a, cudaStream_t st) {
  S3Args s{};
  s.nx = a.nx;
  s.ny = a.ny;
  s.nz = a.nz;
  s.in_real = a.in_mode == PASS_IO_REAL;
  s.out_real = a.out_mode == PASS_IO_REAL;
  s.check_finite = a.check_finite;
  s.in = a.U_in;
  s.out = a.U_out;
  s.kappa = p.kappa_kind == FRKC2_KAPPA_FIELD ? p.kappa : nullptr;
  s.kc = a.kc;
  s.kp = a.kp;
  s.ca = 0.5 * a.ca[0];
  s.cb = 0.5 * a.cb[0];
  s.status = a.status;
  switch (p.precision) {
    case FRKC2_FP64: return launch_s<double, double>(p, s, st);
    case FRKC2_FP32:  // (its offsets in a plane are 32-bit, in bytes)
      return p.n[0] * p.n[1] <= (int64_t(1) << 29) ? launch_pass_stream3d_f32(p, a, st) : launch_s<float, float>(p, s, st);
    default: return launch_s<double, float>(p, s, st);
  }
}

}  // namespace frkc2
