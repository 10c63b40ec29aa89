// 3D single-stage pass (k = 1) in FP32, streaming along z: the scheme of pass_stream3d.cu (columns of
// warps, the y exchange one plane ahead, one barrier a plane, full waves of chunks along z) with the arithmetic as packed two-lane instructions.
//
// The pass is issue bound (a cell-stage of kappa(u) is about 58 FP32 operations against 16 bytes), so a thread
// holds its four rows as two pairs (rows 0, 1 and rows 2, 3): x and z neighbours of a pair are pairs
// themselves, and differences, conductivity sums, complex fluxes, the face sums, the update and all of
// kappa(W) but its square roots, absolute values and sign selects run two cells to an instruction
// (add / mul / fma .f32x2, sm_100 family).  Only the y faces, which would need shifted pairs, take
// scalar instructions.  A packed negation is not free, so the complex products take one difference in both signs.
// The plane loop is unrolled by three with the roles of the three planes held rotated (no register
// moves), and the passes between a step's first and last are instantiated for interleaved state.
// 256^3, kappa(u), s = 32: 125 -> 79 us a pass (40 us at the copy bandwidth; 90 instructions a computed
// cell against 239 an output cell before, at 66 % issue).
#include <algorithm>

#include <cuda_runtime.h>

#include "frkc2_internal.h"
#include "frkc2_math.cuh"

namespace frkc2 {
namespace {

constexpr int F3_OX = 30;     // output columns per CTA
// Rows of a thread, most warps of a CTA, CTAs per SM.  Small CTAs wait less at the plane's barrier, which
// outweighs their halo rows: 256^3, s = 32, kappa(u), a pass (rows, warps, CTAs): (4, 4, 4) 85.7 us, (2, 8, 3)
// 86.9, (2, 12, 2) 88.6, (4, 8, 2) 93.4, (4, 4, 5) 95.2, (2, 8, 4) 97.8.
constexpr int F3_RY = 4, F3_MAXW = 4, F3_CTAS = 4;
// Planes by which the prefetch into L2 (one instruction of a warp a plane) runs ahead of the load: from DRAM a load
// took longer than the plane of work between it and its use (36 % of the warps' time).  256^3, s = 32, kappa(u), a step:
// none 2750 us, 1 2568, 2 2542, 3 2550, 5 2570.  Only where the two states and the conductivities don't stay in L2
// anyway, above F3_L2 bytes (s = 16, 2 steps, without / with: 160^3, 66 MB 753 / 770, with a field, 82 MB 626 / 647;
// 176^3, 87 MB 989 / 987, field 928 / 894; 224^3 1975 / 1859, field 1789 / 1572).
constexpr size_t F3_L2 = 86000000;
constexpr int F3_AHEAD = 2;
constexpr int F3_H = F3_RY / 2;  // a thread's pairs of rows
constexpr int K3_FIELD = 0, K3_POWER = 1, K3_P25 = 2;  // as in pass_stream3d.cu

struct F3Args {
  int nx, ny, nz;
  int oy;                   // output rows per CTA
  int bxn;                  // column blocks along x
  int chunks;               // chunks along z
  int in_real, out_real;    // the pass reads / writes the real state instead of interleaved (U, V)
  int check_finite;
  int prefetch;             // prefetch planes into L2
  const void* in;
  void* out;
  const float* kappa;       // FIELD: cell conductivities; nullptr: the constant kc
  float kc, kp;
  float ca, cb;             // dt a_l / (2 dx^2): the face factor 1/2 folded in
  unsigned* status;
};

__device__ __forceinline__ float2 sub2(float2 a, float2 b) { return __ffma2_rn(make_float2(-1.f, -1.f), b, a); }  // exact product

// One plane of a thread's rows: two pairs of complex states and conductivities.
struct Plane3 {
  float2 U[F3_H], V[F3_H], KR[F3_H], KI[F3_H];
};

// (twice the) complex flux of a pair of faces: kf (d), d given as (dr, di) with ndi = -di
template <bool POWER>
__device__ __forceinline__ void flux2(float2 kr, float2 ki, float2 dr, float2 di, float2 ndi, float2& fr, float2& fi) {
  if (POWER) {
    fr = fma2(kr, dr, mul2(ki, ndi));
    fi = fma2(kr, di, mul2(ki, dr));
  } else {
    fr = mul2(kr, dr);
    fi = mul2(kr, di);
  }
}

// CC: input and output interleaved (else as the arguments say)
template <int KIND, bool PERIODIC, bool CC>
__global__ void __launch_bounds__(32 * F3_MAXW, F3_CTAS) k_stream3d_f32(const F3Args p) {
  constexpr int RY = F3_RY;
  constexpr bool POWER = KIND != K3_FIELD;
  __shared__ float4 shW[2][F3_MAXW][32];  // first row's (U, V, Re kappa, Im kappa) of the next plane
  __shared__ float2 shF[2][F3_MAXW][32];  // last row's north flux of this plane
  // launched with programmatic stream serialization: the next launch may start its CTAs as this
  // one's exit, and every global load below comes after the previous launch has completed
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  asm volatile("griddepcontrol.wait;" ::: "memory");
  const int lane = threadIdx.x, w = threadIdx.y, nw = blockDim.y;
  const int nx = p.nx, ny = p.ny, nz = p.nz;
  const size_t plane = size_t(nx) * ny;  // at most 2^29 (launch_pass_stream3d): offsets in a plane are 32-bit
  const bool in_real = !CC && p.in_real, out_real = !CC && p.out_real;
  const float2 ca2 = make_float2(p.ca, p.ca), cb2 = make_float2(p.cb, p.cb), ncb2 = make_float2(-p.cb, -p.cb);
  const float kc = p.kc, cs = p.kc * 0.70710678118654752440f;
  const int wn = w + 1 < nw ? w + 1 : w;  // (the top halo row's north flux is not used)
  const int ws = w > 0 ? w - 1 : w;       // (the bottom halo row's south flux is not used)
  const float2 z2 = make_float2(0.f, 0.f);

  // conductivities of a loaded plane; Dirichlet ghosts (read at the clamped cell) become zero first
  auto kap = [&](Plane3& q, unsigned in) {
    if (!PERIODIC && __any_sync(0xffffffffu, in != (1u << F3_RY) - 1)) {
#pragma unroll
      for (int h = 0; h < F3_H; ++h) {
        if (!(in >> (2 * h) & 1)) q.U[h].x = q.V[h].x = 0.f;
        if (!(in >> (2 * h + 1) & 1)) q.U[h].y = q.V[h].y = 0.f;
      }
    }
#pragma unroll
    for (int h = 0; h < F3_H; ++h) {
      if constexpr (KIND == K3_P25) {
        kappa25_pair(q.U[h], q.V[h], cs, q.KR[h], q.KI[h]);
      } else if constexpr (KIND == K3_POWER) {
        kappa_power<float>(q.U[h].x, q.V[h].x, kc, p.kp, q.KR[h].x, q.KI[h].x);
        kappa_power<float>(q.U[h].y, q.V[h].y, kc, p.kp, q.KR[h].y, q.KI[h].y);
      }
    }
  };

  int b = 0;  // exchange buffer
  bool bad = false;
  const int blk = blockIdx.x, z0 = int((long long)blockIdx.y * nz / p.chunks), z1 = int((long long)(blockIdx.y + 1) * nz / p.chunks);
  {
    const int gx = (blk % p.bxn) * F3_OX + lane - 1;
    const int gy0 = (blk / p.bxn) * p.oy + w * RY - 1;
    const bool out_x = lane >= 1 && lane <= 30 && gx < nx;
    // per row: the byte offset of its column in a plane of the state (wrapped, or clamped to the grid:
    // the conductivity of a Dirichlet ghost is its interior cell's); bit r of `inside`: the cell is in
    // the grid, of `outm`: it is an output
    unsigned off[RY], inside = 0, outm = 0;
    const bool xin = PERIODIC || (gx >= 0 && gx < nx);
    const int xr = PERIODIC ? wrap3(gx, nx) : min(max(gx, 0), nx - 1);
#pragma unroll
    for (int r = 0; r < RY; ++r) {
      const int gy = gy0 + r, R = w * RY + r;
      const int yr = PERIODIC ? wrap3(gy, ny) : min(max(gy, 0), ny - 1);
      off[r] = (unsigned(yr) * unsigned(nx) + unsigned(xr)) * 8u;
      if (xin && (PERIODIC || (gy >= 0 && gy < ny))) inside |= 1u << r;
      if (out_x && R >= 1 && R <= p.oy && gy < ny) outm |= 1u << r;
    }
    auto zin = [&](int z) -> unsigned { return PERIODIC || (z >= 0 && z < nz) ? inside : 0u; };
    // the lane's 32 bytes of the warp's four rows in a plane, for the prefetch into L2
    unsigned poff;
    {
      const int gy = gy0 + (lane >> 3), px = gx - lane + 4 * (lane & 7);
      poff = (unsigned(PERIODIC ? wrap3(gy, ny) : min(max(gy, 0), ny - 1)) * unsigned(nx) +
              unsigned(PERIODIC ? wrap3(px, nx) : min(max(px, 0), nx - 1))) * 8u;
    }
    auto prefetch = [&](int z) {
      const char* base = static_cast<const char*>(p.in) + size_t(PERIODIC ? wrap3(z, nz) : min(max(z, 0), nz - 1)) * plane * 8;
      if (in_bounds(poff / 8 < plane, p.status)) {
        asm volatile("prefetch.global.L2 [%0];" ::"l"(base + poff));
        if (!POWER && p.kappa && (lane & 1) == 0)
          asm volatile("prefetch.global.L2 [%0];" ::"l"(reinterpret_cast<const char*>(p.kappa) +
                                                        (base - static_cast<const char*>(p.in)) / 2 + poff / 2));
      }
    };
    // W (and FIELD / CONST conductivities) of plane z; the offsets are 32-bit against a uniform base
    auto load = [&](int z, Plane3& q) {
      const size_t zo = size_t(PERIODIC ? wrap3(z, nz) : min(max(z, 0), nz - 1)) * plane;
      const char* base = static_cast<const char*>(p.in) + zo * (in_real ? 4 : 8);
      const char* kbase = reinterpret_cast<const char*>(p.kappa) + zo * 4;
#pragma unroll
      for (int r = 0; r < RY; ++r) {
        float2 v = z2;
        if (in_bounds(off[r] / 8 < plane, p.status)) {
          if (in_real)
            v.x = __ldg(reinterpret_cast<const float*>(base + off[r] / 2));
          else
            v = __ldg(reinterpret_cast<const float2*>(base + off[r]));
        }
        (r & 1 ? q.U[r >> 1].y : q.U[r >> 1].x) = v.x;
        (r & 1 ? q.V[r >> 1].y : q.V[r >> 1].x) = v.y;
        if (!POWER) {
          float k = kc;
          if (p.kappa && in_bounds(off[r] / 8 < plane, p.status)) k = __ldg(reinterpret_cast<const float*>(kbase + off[r] / 2));
          (r & 1 ? q.KR[r >> 1].y : q.KR[r >> 1].x) = k;
        }
      }
    };
    // fluxes of a pair of z faces between planes a (below) and c (above)
    auto zflux = [&](const Plane3& a, const Plane3& c, int h, float2& fr, float2& fi) {
      const float2 dr = sub2(c.U[h], a.U[h]), di = sub2(c.V[h], a.V[h]), ndi = POWER ? sub2(a.V[h], c.V[h]) : z2;
      flux2<POWER>(add2(a.KR[h], c.KR[h]), POWER ? add2(a.KI[h], c.KI[h]) : z2, dr, di, ndi, fr, fi);
    };
    // flux of one y face between cells (u0, v0, kr0, ki0) and the one north of it
    auto yflux = [&](float u0, float v0, float kr0, float ki0, float u1, float v1, float kr1, float ki1, float& fr, float& fi) {
      const float kr = kr0 + kr1, dr = u1 - u0, di = v1 - v0;
      if (POWER) {
        const float ki = ki0 + ki1;
        fr = fmaf(kr, dr, -(ki * di));
        fi = fmaf(kr, di, ki * dr);
      } else {
        fr = kr * dr;
        fi = kr * di;
      }
    };
    // north flux of the thread's last row, from the next warp's first row
    auto topflux = [&](const Plane3& a, float4 n) -> float2 {
      float2 f;
      yflux(a.U[F3_H - 1].y, a.V[F3_H - 1].y, a.KR[F3_H - 1].y, POWER ? a.KI[F3_H - 1].y : 0.f, n.x, n.y, n.z, n.w, f.x, f.y);
      return f;
    };
    auto publish = [&](const Plane3& q) {
      shW[b][w][lane] = make_float4(q.U[0].x, q.V[0].x, q.KR[0].x, POWER ? q.KI[0].x : 0.f);
    };

    // three planes in registers: z and z + 1 with their conductivities, z + 2 as it was loaded
    Plane3 A, B, C;
    float2 FdR[F3_H], FdI[F3_H], Ft;
    // prime: the fluxes through the down faces of z0 and the last row's north flux
    load(z0 - 1, C);
    load(z0, A);
    load(z0 + 1, B);
    kap(C, zin(z0 - 1));
    kap(A, zin(z0));
    kap(B, zin(z0 + 1));
#pragma unroll
    for (int h = 0; h < F3_H; ++h) zflux(C, A, h, FdR[h], FdI[h]);
    publish(A);
    __syncthreads();
    Ft = topflux(A, shW[b][wn][lane]);
    b ^= 1;
    load(z0 + 2, C);
    // one plane: c = plane z, u = plane z + 1, l = plane z + 2, which gets its conductivities; c then
    // takes the load of plane z + 3 (used a whole plane later)
    auto step = [&](int z, Plane3& c, Plane3& u, Plane3& l) {
      publish(u);
      shF[b][w][lane] = Ft;
      __syncthreads();
      const float2 Fs = shF[b][ws][lane];
      const float4 Nn = shW[b][wn][lane];
      b ^= 1;
      // y part of f: the faces inside the thread, the exchanged fluxes outside
      float2 yR[F3_H], yI[F3_H];
      {
        float pr = Fs.x, pi = Fs.y;
#pragma unroll
        for (int h = 0; h < F3_H; ++h) {
          float r0, i0, r1 = Ft.x, i1 = Ft.y;
          yflux(c.U[h].x, c.V[h].x, c.KR[h].x, POWER ? c.KI[h].x : 0.f, c.U[h].y, c.V[h].y, c.KR[h].y, POWER ? c.KI[h].y : 0.f, r0, i0);
          if (h + 1 < F3_H)
            yflux(c.U[h].y, c.V[h].y, c.KR[h].y, POWER ? c.KI[h].y : 0.f, c.U[h + 1].x, c.V[h + 1].x, c.KR[h + 1].x, POWER ? c.KI[h + 1].x : 0.f, r1, i1);
          yR[h] = make_float2(r0 - pr, r1 - r0);
          yI[h] = make_float2(i0 - pi, i1 - i0);
          pr = r1;
          pi = i1;
        }
      }
      char* obase = static_cast<char*>(p.out) + size_t(z) * plane * (out_real ? 4 : 8);
#pragma unroll
      for (int h = 0; h < F3_H; ++h) {
        float2 eU, eV, eKR, eKI = z2;
        eU.x = __shfl_down_sync(0xffffffffu, c.U[h].x, 1);
        eU.y = __shfl_down_sync(0xffffffffu, c.U[h].y, 1);
        eV.x = __shfl_down_sync(0xffffffffu, c.V[h].x, 1);
        eV.y = __shfl_down_sync(0xffffffffu, c.V[h].y, 1);
        eKR.x = __shfl_down_sync(0xffffffffu, c.KR[h].x, 1);
        eKR.y = __shfl_down_sync(0xffffffffu, c.KR[h].y, 1);
        if (POWER) {
          eKI.x = __shfl_down_sync(0xffffffffu, c.KI[h].x, 1);
          eKI.y = __shfl_down_sync(0xffffffffu, c.KI[h].y, 1);
        }
        float2 FeR, FeI, FuR, FuI, FwR, FwI;
        flux2<POWER>(add2(c.KR[h], eKR), POWER ? add2(c.KI[h], eKI) : z2, sub2(eU, c.U[h]), sub2(eV, c.V[h]),
                     POWER ? sub2(c.V[h], eV) : z2, FeR, FeI);
        FwR.x = __shfl_up_sync(0xffffffffu, FeR.x, 1);
        FwR.y = __shfl_up_sync(0xffffffffu, FeR.y, 1);
        FwI.x = __shfl_up_sync(0xffffffffu, FeI.x, 1);
        FwI.y = __shfl_up_sync(0xffffffffu, FeI.y, 1);
        zflux(c, u, h, FuR, FuI);
        const float2 fR = add2(add2(sub2(FeR, FwR), yR[h]), sub2(FuR, FdR[h]));
        const float2 fI = add2(add2(sub2(FeI, FwI), yI[h]), sub2(FuI, FdI[h]));
        FdR[h] = FuR;
        FdI[h] = FuI;
        const float2 un = fma2(ncb2, fI, fma2(ca2, fR, c.U[h]));
        const float2 vn = fma2(cb2, fR, fma2(ca2, fI, c.V[h]));
#pragma unroll
        for (int e = 0; e < 2; ++e) {
          const int r = 2 * h + e;
          const float uu = e ? un.y : un.x, vv = e ? vn.y : vn.x;
          if ((outm >> r & 1) && in_bounds(off[r] / 8 < plane, p.status)) {
            if (out_real)
              *reinterpret_cast<float*>(obase + off[r] / 2) = uu;
            else
              *reinterpret_cast<float2*>(obase + off[r]) = make_float2(uu, vv);
            if (!CC && p.check_finite) bad |= (__float_as_uint(uu) & 0x7f800000u) == 0x7f800000u;
          }
        }
      }
      Ft = topflux(u, Nn);
      if (z + 3 <= z1) load(z + 3, c);
      if (CC && p.prefetch && z + 3 + F3_AHEAD <= z1) prefetch(z + 3 + F3_AHEAD);
      kap(l, zin(z + 2));
    };
    for (int z = z0; z < z1; z += 3) {
      step(z, A, B, C);
      if (z + 1 >= z1) break;
      step(z + 1, B, C, A);
      if (z + 2 >= z1) break;
      step(z + 2, C, A, B);
    }
  }
  if (bad) atomicOr(p.status, ST_NONFINITE);
}

template <int KIND, bool PERIODIC, bool CC>
cudaError_t launch_t(F3Args a, cudaStream_t st) {
  const auto kern = k_stream3d_f32<KIND, PERIODIC, CC>;
  struct Res {
    cudaError_t err;
    int sms, per_sm[F3_MAXW + 1];
  };
  static const Res res = [kern] {
    Res r{};
    for (int n = 1; n <= F3_MAXW; ++n) {
      const Residency q = query_residency(kern, 32 * n, 0);
      if (q.err != cudaSuccess) r.err = q.err;
      r.sms = q.sms;
      r.per_sm[n] = q.per_sm;
    }
    return r;
  }();
  if (res.err != cudaSuccess) return res.err;
  // warps per CTA: the count of at least half the most that covers ny with the fewest rows, each warp
  // less counted as 2 % (fewer warps hide less latency)
  int nw = 0;
  long long best = 0;
  for (int n = F3_MAXW; n >= F3_MAXW / 2; --n) {
    const int oy = F3_RY * n - 2;
    const long long rows = (long long)((a.ny + oy - 1) / oy) * F3_RY * n * (50 + F3_MAXW - n);
    if (nw == 0 || rows < best) {
      nw = n;
      best = rows;
    }
  }
  a.oy = F3_RY * nw - 2;
  a.bxn = (a.nx + F3_OX - 1) / F3_OX;
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

template <int KIND>
cudaError_t launch_k(const F3Args& a, bool per, cudaStream_t st) {
  if (!a.in_real && !a.out_real && !a.check_finite)
    return per ? launch_t<KIND, true, true>(a, st) : launch_t<KIND, false, true>(a, st);
  return per ? launch_t<KIND, true, false>(a, st) : launch_t<KIND, false, false>(a, st);
}

}  // namespace

cudaError_t launch_pass_stream3d_f32(const frkc2_problem& p, const PassArgs& a, cudaStream_t st) {
  F3Args s{};
  s.nx = a.nx;
  s.ny = a.ny;
  s.nz = a.nz;
  s.in_real = a.in_mode == PASS_IO_REAL;
  s.out_real = a.out_mode == PASS_IO_REAL;
  s.check_finite = a.check_finite;
  s.in = a.U_in;
  s.out = a.U_out;
  s.kappa = p.kappa_kind == FRKC2_KAPPA_FIELD ? static_cast<const float*>(p.kappa) : nullptr;
  s.kc = float(a.kc);
  s.kp = float(a.kp);
  s.ca = float(0.5 * a.ca[0]);
  s.cb = float(0.5 * a.cb[0]);
  s.prefetch = size_t(a.nx) * a.ny * a.nz * (s.kappa ? 20 : 16) > F3_L2;
  s.status = a.status;
  const bool per = p.bc == FRKC2_BC_PERIODIC;
  if (p.kappa_kind != FRKC2_KAPPA_POWER) return launch_k<K3_FIELD>(s, per, st);
  return s.kp == 2.5f ? launch_k<K3_P25>(s, per, st) : launch_k<K3_POWER>(s, per, st);
}

}  // namespace frkc2
