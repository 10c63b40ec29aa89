// 2D temporally blocked pass for FP32 (fixed conductivity) with the state in registers:
// k stages of Sec. 3, Eq. 13 per HBM round trip.
//
// A CTA of 16 x 16 threads owns a region of 16C x 16C cells, C = 4 or 2: its output tile
// (16C - 2k)^2 plus a k-cell halo recomputed redundantly (region-edge values go stale one cell per
// stage, which never reaches the output tile).  Thread (tx, ty) owns the C x C cells at columns
// C tx, rows C ty and keeps, for all k stages, their complex state (32 floats for C = 4) and their
// face conductivities (40) in registers.  C = 4 recomputes least and serves grids that fill the
// chip; C = 2 gives four times the CTAs for grids that would leave SMs idle (128^2: 0.78 -> 0.34 us a
// stage, 256^2 0.80 -> 0.51; the region size and k are chosen by tb2d_shape).  Launches of less than a
// wave are spread evenly over the SMs (spread_smem).  Rows are read and written as vectors (2048^2, k = 8, a pass:
// 61 -> 50 us; faces and state buffers have rows padded to a multiple of 4 cells).  Per stage:
//   - the thread's bottom and top rows go to shared memory (double-buffered by stage parity,
//     one barrier per stage); its south and north neighbour rows come back from the threads
//     below and above;
//   - the columns beyond its own come from the adjacent threads by 16-lane shuffles, one row
//     at a time, before that row is updated;
//   - every neighbour difference inside the block is formed once and used by both cells of
//     the face: f = k_n d_n - k_s d_s + k_e d_e - k_w d_w, then the complex update;
//   - the cells are held as horizontal pairs (float2), so the y differences, the y terms of f
//     and the complex update run as packed two-lane FP32 instructions (add / fma .f32x2, new
//     with the sm_100 family), two cells per instruction; the x differences and x terms, whose
//     pairs would straddle the register pairs, stay scalar: 11.5 FP32 instructions per
//     cell-stage for 16.5 floating-point operations.
// Shared memory traffic: 8 bytes per cell-stage (the two exchanged rows), against the full
// state of a shared-memory ping-pong.
// The batched launch runs the same region computation from tb2d_region.cuh; this kernel keeps
// its own copy because, written as that shared device function, it compiled to an 11 % slower
// pass (4.15e11 against 4.61e11 cell-stage/s at 2048^2, k = 8) with the same registers.
#include <algorithm>
#include <cstdint>
#include <type_traits>

#include <cuda_runtime.h>

#include "frkc2_internal.h"

namespace frkc2 {
namespace {

constexpr int RT_THREADS = 256;   // 16 x 16 threads of C x C cells

// a row of C cells of one component, as it goes through shared memory, and as cell pairs
template <int C> struct Row;
template <> struct Row<4> { using type = float4; };
template <> struct Row<2> { using type = float2; };
__device__ __forceinline__ float4 row_of(const float2 (&a)[2]) { return make_float4(a[0].x, a[0].y, a[1].x, a[1].y); }
__device__ __forceinline__ float2 row_of(const float2 (&a)[1]) { return a[0]; }
__device__ __forceinline__ void row_get(float4 v, float2 (&a)[2]) {
  a[0] = make_float2(v.x, v.y);
  a[1] = make_float2(v.z, v.w);
}
__device__ __forceinline__ void row_get(float2 v, float2 (&a)[1]) { a[0] = v; }
// a row of four cells as vectors of VEC cells
// (plain loads throughout: with __ldg the compiler kept them in order and a pass of single cells took 8 % longer)
template <int VEC, int H>
__device__ __forceinline__ void row_load(const float* p, float2 (&a)[H]) {
  if constexpr (VEC == 4) {
    row_get(*reinterpret_cast<const float4*>(p), a);
  } else {
#pragma unroll
    for (int h = 0; h < H; ++h) a[h] = *(reinterpret_cast<const float2*>(p) + h);
  }
}
template <int VEC, int H>
__device__ __forceinline__ void row_store(float* p, const float2 (&a)[H]) {
  if constexpr (VEC == 4) {
    *reinterpret_cast<float4*>(p) = row_of(a);
  } else {
#pragma unroll
    for (int h = 0; h < H; ++h) *(reinterpret_cast<float2*>(p) + h) = a[h];
  }
}

__device__ __forceinline__ int wrap_r(int g, int n) {
  if (g >= 0 && g < n) return g;
  if (g < 0 && g >= -n) return g + n;
  if (g >= n && g < 2 * n) return g - n;
  const int r = g % n;
  return r < 0 ? r + n : r;
}

// a - b on both halves in one packed instruction (sm_100 family)
__device__ __forceinline__ float2 sub2(float2 a, float2 b) { return __fadd2_rn(a, make_float2(-b.x, -b.y)); }

// VEC: a thread's rows move as vectors of so many cells where they lie in the grid in one piece (not across the
// periodic wrap); 1: single cells throughout.  k a multiple of VEC keeps the rows aligned.
template <int C, bool PERIODIC, int VEC>
__global__ void __launch_bounds__(RT_THREADS, C == 4 ? 2 : 4) k_tb2d_reg(const PassArgs p, const TbIo io) {
  using R = typename Row<C>::type;
  constexpr int H = C / 2, RT_R = 16 * C;  // pairs of a row; region edge (cells)
  __shared__ R sh_bot[2][2][16][16];  // [stage parity][U, V][ty][tx]: the thread's first row
  __shared__ R sh_top[2][2][16][16];  // its last row
  const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
  const int k = p.k;
  const int T = RT_R - 2 * k;
  const int x0 = blockIdx.x * T - k, y0 = blockIdx.y * T - k;
  const int nx = p.nx, ny = p.ny;
  // the next pass may be launched as soon as every CTA of this one is running (it then loads
  // its face conductivities, which no pass writes, and waits below for this pass's state)
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  const float* __restrict__ Uin = static_cast<const float*>(p.U_in);
  const float* __restrict__ Vin = static_cast<const float*>(p.V_in);
  const bool padded = io.fxp != nullptr;
  const float* __restrict__ FX = padded ? io.fxp : static_cast<const float*>(p.fx);
  const float* __restrict__ FY = padded ? io.fyp : static_cast<const float*>(p.fy);
  const int pfx = padded ? io.fpitch : nx + 1, pfy = padded ? io.fpitch : nx, pin = io.in_pitch;

  // wrapped (periodic) or raw (Dirichlet) grid rows / columns of the thread's cells; the last
  // entry is the next row / column (north and east faces)
  int gyr[C + 1], gxc[C + 1];
  bool yin[C + 1], xin[C + 1];
#pragma unroll
  for (int i = 0; i < C + 1; ++i) {
    const int gx = x0 + C * tx + i, gy = y0 + C * ty + i;
    gxc[i] = PERIODIC ? wrap_r(gx, nx) : gx;
    gyr[i] = PERIODIC ? wrap_r(gy, ny) : gy;
    xin[i] = gx >= 0 && gx < nx;
    yin[i] = gy >= 0 && gy < ny;
  }
  unsigned inside = 0;  // Dirichlet: bit C r + c set if cell (r, c) lies in the grid
#pragma unroll
  for (int r = 0; r < C; ++r)
#pragma unroll
    for (int c = 0; c < C; ++c)
      if (xin[c] && yin[r]) inside |= 1u << (C * r + c);
  const bool run = VEC > 1 && (gxc[0] & (VEC - 1)) == 0 && gxc[C - 1] == gxc[0] + C - 1 && (PERIODIC || (xin[0] && xin[C - 1]));
  // fx[r][c]: x face c of row r (the west face of cell c; c = C is the east face of the last cell);
  // FY2[r]: y faces r as cell pairs (the south faces of row r; r = C the north faces of the last row)
  float fx[C][C + 1];
  float2 FY2[C + 1][H];
  if (VEC > 1 && padded && run) {
#pragma unroll
    for (int r = 0; r < C + 1; ++r) {
#pragma unroll
      for (int h = 0; h < H; ++h) FY2[r][h] = make_float2(0.f, 0.f);
      if (PERIODIC || (gyr[r] >= 0 && gyr[r] <= ny)) {
        const size_t fi = size_t(gyr[r]) * pfy + gxc[0];
        if (in_bounds(fi + C <= size_t(ny + 1) * pfy, p.status)) row_load<VEC>(FY + fi, FY2[r]);
      }
      if (r < C) {
        float2 e[H];
#pragma unroll
        for (int h = 0; h < H; ++h) e[h] = make_float2(0.f, 0.f);
        fx[r][C] = 0.f;
        if (PERIODIC || yin[r]) {
          const size_t fi = size_t(gyr[r]) * pfx + gxc[0];
          if (in_bounds(fi + C < size_t(ny) * pfx, p.status)) {
            row_load<VEC>(FX + fi, e);
            fx[r][C] = FX[fi + C];  // (periodic face nx repeats face 0)
          }
        }
#pragma unroll
        for (int h = 0; h < H; ++h) {
          fx[r][2 * h] = e[h].x;
          fx[r][2 * h + 1] = e[h].y;
        }
      }
    }
  } else {
#pragma unroll
    for (int r = 0; r < C + 1; ++r) {
#pragma unroll
      for (int c = 0; c < C + 1; ++c) {
        if (r < C) {
          float v = 0.f;
          if (PERIODIC || (yin[r] && gxc[c] >= 0 && gxc[c] <= nx)) {
            const size_t fi = size_t(gyr[r]) * pfx + gxc[c];
            if (in_bounds(fi < size_t(ny) * pfx, p.status)) v = FX[fi];
          }
          fx[r][c] = v;
        }
        if (c < C) {
          float v = 0.f;
          if (PERIODIC || (xin[c] && gyr[r] >= 0 && gyr[r] <= ny)) {
            const size_t fi = size_t(gyr[r]) * pfy + gxc[c];
            if (in_bounds(fi < size_t(ny + 1) * pfy, p.status)) v = FY[fi];
          }
          (c & 1 ? FY2[r][c >> 1].y : FY2[r][c >> 1].x) = v;
        }
      }
    }
  }
  // the previous pass's state is complete and visible after this (a no-op for a launch
  // without the programmatic-serialization attribute)
  asm volatile("griddepcontrol.wait;" ::: "memory");
  // the state as horizontal cell pairs: U2[r][h] = (U[r][2h], U[r][2h + 1])
  float2 U2[C][H], V2[C][H];
  const bool vin = VEC > 1 && (pin & (VEC - 1)) == 0 && (reinterpret_cast<uintptr_t>(Uin) & (4 * VEC - 1)) == 0;
  if (vin && run) {
#pragma unroll
    for (int r = 0; r < C; ++r) {
#pragma unroll
      for (int h = 0; h < H; ++h) U2[r][h] = V2[r][h] = make_float2(0.f, 0.f);
      const size_t g = size_t(gyr[r]) * pin + gxc[0];
      if ((PERIODIC || yin[r]) && in_bounds(g + C <= size_t(pin) * ny, p.status)) {
        row_load<VEC>(Uin + g, U2[r]);
        if (Vin) row_load<VEC>(Vin + g, V2[r]);
      }
    }
  } else {
#pragma unroll
    for (int r = 0; r < C; ++r)
#pragma unroll
      for (int c = 0; c < C; ++c) {
        float uu = 0.f, vv = 0.f;
        if (PERIODIC || (inside & (1u << (C * r + c)))) {
          const size_t g = size_t(gyr[r]) * pin + gxc[c];
          if (in_bounds(g < size_t(pin) * ny, p.status)) {
            uu = Uin[g];
            if (Vin) vv = Vin[g];
          }
        }
        (c & 1 ? U2[r][c >> 1].y : U2[r][c >> 1].x) = uu;
        (c & 1 ? V2[r][c >> 1].y : V2[r][c >> 1].x) = vv;
      }
  }

  const float2 z2 = make_float2(0.f, 0.f);
  // MASK: the region reaches beyond a Dirichlet grid, whose cells outside stay zero
  auto stages = [&](auto mask) {
  constexpr bool MASK = decltype(mask)::value;
  for (int j = 0; j < k; ++j) {
    const int b = j & 1;
    sh_bot[b][0][ty][tx] = row_of(U2[0]);
    sh_bot[b][1][ty][tx] = row_of(V2[0]);
    sh_top[b][0][ty][tx] = row_of(U2[C - 1]);
    sh_top[b][1][ty][tx] = row_of(V2[C - 1]);
    __syncthreads();
    // the region's outermost thread rows have no neighbour row here: their edge goes stale
    float2 su2[H], sv2[H], nu2[H], nv2[H];
#pragma unroll
    for (int h = 0; h < H; ++h) su2[h] = sv2[h] = nu2[h] = nv2[h] = z2;
    if (ty > 0) {
      row_get(sh_top[b][0][ty - 1][tx], su2);
      row_get(sh_top[b][1][ty - 1][tx], sv2);
    }
    if (ty < 15) {
      row_get(sh_bot[b][0][ty + 1][tx], nu2);
      row_get(sh_bot[b][1][ty + 1][tx], nv2);
    }
    const float ca = p.caf[j], cb = p.cbf[j];
    const float2 ca2 = make_float2(ca, ca), cb2 = make_float2(cb, cb), ncb2 = make_float2(-cb, -cb);
    // differences across the south faces of the current row: W(r) - W(r - 1)
    float2 dsU[H], dsV[H];
#pragma unroll
    for (int h = 0; h < H; ++h) {
      dsU[h] = sub2(U2[0][h], su2[h]);
      dsV[h] = sub2(V2[0][h], sv2[h]);
    }
#pragma unroll
    for (int r = 0; r < C; ++r) {
      // columns beyond the thread's own, before this row is updated
      const float wU = __shfl_up_sync(0xffffffffu, U2[r][H - 1].y, 1, 16);
      const float wV = __shfl_up_sync(0xffffffffu, V2[r][H - 1].y, 1, 16);
      const float eU = __shfl_down_sync(0xffffffffu, U2[r][0].x, 1, 16);
      const float eV = __shfl_down_sync(0xffffffffu, V2[r][0].x, 1, 16);
      float u[C + 2], v[C + 2];
      u[0] = wU;
      v[0] = wV;
#pragma unroll
      for (int h = 0; h < H; ++h) {
        u[2 * h + 1] = U2[r][h].x;
        u[2 * h + 2] = U2[r][h].y;
        v[2 * h + 1] = V2[r][h].x;
        v[2 * h + 2] = V2[r][h].y;
      }
      u[C + 1] = eU;
      v[C + 1] = eV;
      // dx[c]: across x face c, W(c) - W(c - 1), each formed once for the two cells of the face
      float dxU[C + 1], dxV[C + 1];
#pragma unroll
      for (int c = 0; c < C + 1; ++c) {
        dxU[c] = u[c + 1] - u[c];
        dxV[c] = v[c + 1] - v[c];
      }
      // x part of f per cell, written straight into the halves of the pairs
      float2 fU[H], fV[H];
#pragma unroll
      for (int h = 0; h < H; ++h) {
        const int c = 2 * h;
        fU[h].x = fx[r][c + 1] * dxU[c + 1] - fx[r][c] * dxU[c];
        fU[h].y = fx[r][c + 2] * dxU[c + 2] - fx[r][c + 1] * dxU[c + 1];
        fV[h].x = fx[r][c + 1] * dxV[c + 1] - fx[r][c] * dxV[c];
        fV[h].y = fx[r][c + 2] * dxV[c + 2] - fx[r][c + 1] * dxV[c + 1];
      }
#pragma unroll
      for (int h = 0; h < H; ++h) {
        const float2 nU = r < C - 1 ? U2[r < C - 1 ? r + 1 : r][h] : nu2[h];
        const float2 nV = r < C - 1 ? V2[r < C - 1 ? r + 1 : r][h] : nv2[h];
        const float2 dnU = sub2(nU, U2[r][h]), dnV = sub2(nV, V2[r][h]);
        // y part, two cells per instruction: f += k_n d_n - k_s d_s
        const float2 nks = make_float2(-FY2[r][h].x, -FY2[r][h].y);
        fU[h] = __ffma2_rn(nks, dsU[h], __ffma2_rn(FY2[r + 1][h], dnU, fU[h]));
        fV[h] = __ffma2_rn(nks, dsV[h], __ffma2_rn(FY2[r + 1][h], dnV, fV[h]));
        // W += (ca + i cb) f
        float2 un = __ffma2_rn(ncb2, fV[h], __ffma2_rn(ca2, fU[h], U2[r][h]));
        float2 vn = __ffma2_rn(cb2, fU[h], __ffma2_rn(ca2, fV[h], V2[r][h]));
        if (MASK) {
          if (!(inside & (1u << (C * r + 2 * h)))) un.x = vn.x = 0.f;
          if (!(inside & (1u << (C * r + 2 * h + 1)))) un.y = vn.y = 0.f;
        }
        U2[r][h] = un;
        V2[r][h] = vn;
        dsU[h] = dnU;
        dsV[h] = dnV;
      }
    }
  }
  };
  if (!PERIODIC && (x0 < 0 || y0 < 0 || x0 + RT_R > nx || y0 + RT_R > ny))
    stages(std::true_type{});
  else
    stages(std::false_type{});

  // store the output tile: region cells at distance >= k from the region edge
  float* __restrict__ Uo = static_cast<float*>(p.U_out);
  float* __restrict__ Vo = static_cast<float*>(p.V_out);
  const int pout = io.out_pitch, gx0 = x0 + C * tx;
  const bool vout = VEC > 1 && (pout & (VEC - 1)) == 0 && (reinterpret_cast<uintptr_t>(Uo) & (4 * VEC - 1)) == 0 &&
                    (gx0 & (VEC - 1)) == 0 && C * tx >= k && C * tx + C <= RT_R - k && gx0 + C <= nx;
  bool bad = false;
#pragma unroll
  for (int r = 0; r < C; ++r) {
    const int ry = C * ty + r;
    const int gy = y0 + ry;
    if (ry < k || ry >= RT_R - k || gy >= ny) continue;
    const size_t row = size_t(gy) * pout;
    if (vout && in_bounds(row + gx0 + C <= size_t(pout) * ny, p.status)) {
      row_store<VEC>(Uo + row + gx0, U2[r]);
      if (Vo) row_store<VEC>(Vo + row + gx0, V2[r]);
    }
#pragma unroll
    for (int c = 0; c < C; ++c) {
      const int rx = C * tx + c;
      const int gx = gx0 + c;
      if (rx < k || rx >= RT_R - k || gx >= nx) continue;
      const float uu = (c & 1) ? U2[r][c >> 1].y : U2[r][c >> 1].x;
      if (!vout && in_bounds(row + gx < size_t(pout) * ny, p.status)) {
        Uo[row + gx] = uu;
        if (Vo) Vo[row + gx] = (c & 1) ? V2[r][c >> 1].y : V2[r][c >> 1].x;
      }
      if (p.check_finite) bad |= (__float_as_uint(uu) & 0x7f800000u) == 0x7f800000u;
    }
  }
  if (bad) atomicOr(p.status, ST_NONFINITE);
}

template <int C, bool PERIODIC, int VEC>
Residency tb_residency() {
  static SpreadKernel own;
  return spread_residency(own, k_tb2d_reg<C, PERIODIC, VEC>, RT_THREADS, 0, sizeof(typename Row<C>::type) * 2 * 2 * 2 * 256);
}

template <int C, bool PERIODIC, int VEC>
cudaError_t launch_c(const PassArgs& a, const TbIo& io, cudaStream_t st, bool overlap_previous) {
  const Residency res = tb_residency<C, PERIODIC, VEC>();
  if (res.err != cudaSuccess) return res.err;
  const int T = 16 * C - 2 * a.k;
  const size_t stat = sizeof(typename Row<C>::type) * 2 * 2 * 2 * 256;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((a.nx + T - 1) / T, (a.ny + T - 1) / T, 1);
  cfg.blockDim = dim3(RT_THREADS, 1, 1);
  cfg.dynamicSmemBytes = spread_smem(stat, (long long)cfg.gridDim.x * cfg.gridDim.y, res.sms, res.per_sm) - stat;
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = overlap_previous ? 1 : 0;
  const cudaError_t e = cudaLaunchKernelEx(&cfg, k_tb2d_reg<C, PERIODIC, VEC>, a, io);
  count_launch();
  return e != cudaSuccess ? e : cudaGetLastError();
}

}  // namespace

// Time of a pass of k stages over `regions` regions in us, fitted to measurements on periodic grids of 64^2 to
// 4096^2 (k = 2 .. 12): a wave by the CTAs an SM holds (C = 4: by the vectors that k allows), and waves that
// overlap by c at their ends.  Model / measured: C = 2, k = 8, 128^2 3.2 / 3.1, 256^2 4.1 / 4.3; C = 4, k = 6, 1021 x 777
// 8.8 / 8.8, k = 8, 1024^2 16.6 / 16.4, 2048^2 50.5 / 50.2, 4096^2 188 / 184.
static double tb2d_pass_us(int C, int k, long long regions, int sms) {
  auto wave = [&](long long ctas) {
    const long long r = (ctas + sms - 1) / sms;  // CTAs per SM
    if (C == 4) {
      if (k % 4 == 0) return r <= 1 ? 3.3 + 0.35 * k : 4.0 + 0.66 * k;
      if (k % 2 == 0) return r <= 1 ? 3.7 + 0.39 * k : 4.4 + 0.73 * k;
      return r <= 1 ? 4.3 + 0.32 * k : 5.5 + 0.67 * k;
    }
    return r <= 1 ? 2.0 + 0.15 * k : r == 2 ? 2.4 + 0.21 * k : r == 3 ? 2.4 + 0.38 * k : 2.0 + 0.64 * k;
  };
  const double c = C == 4 ? 0.3 + 0.2 * k : 0.3 * k;
  const long long slots = (long long)(C == 4 ? 2 : 4) * sms, full = regions / slots, rest = regions % slots;
  return double(full) * (wave(slots) - c) + (rest ? wave(rest) : c);
}

static TbShape tb2d_best(int C, int nx, int ny, int s, int kmin, int kstep, int kmax) {
  const int sms = model_sms();
  TbShape best{C, kmin, 0.0};
  for (int k = kmin; k <= std::min(s, kmax); k += kstep) {
    auto pass = [&](int q) {
      const int T = 16 * C - 2 * q;
      // A launch's y axis ends at 65535: tall grids take regions high enough, up to 4 million rows.  (Regions along one
      // axis would have no such end, but the registers of their division cost a 2048^2 pass 6 %: 3931 -> 4176 us, s = 64, 10 steps.)
      if ((ny + T - 1) / T > 65535) return 1e30;
      return tb2d_pass_us(C, q, (long long)((nx + T - 1) / T) * ((ny + T - 1) / T), sms);
    };
    const double us = (s / k) * pass(k) + (s % k ? pass(s % k) : 0.0);
    if (k == kmin || us < best.us) best = TbShape{C, k, us};
  }
  return best;
}

TbShape tb2d_shape(int nx, int ny, int s) {
  const TbShape a = tb2d_best(2, nx, ny, s, 1, 1, 10), b = tb2d_best(4, nx, ny, s, 1, 1, 12);
  return a.us < b.us ? a : b;
}

TbShape tb2d_shape_even(int nx, int ny, int s) { return tb2d_best(4, nx, ny, s, 2, 2, 12); }

bool tb2d_supported(const frkc2_problem& p, int k) {
  return p.ndim == 2 && p.precision == FRKC2_FP32 && p.kappa_kind != FRKC2_KAPPA_POWER && k >= 1 && 2 * k < 64;
}

cudaError_t launch_pass_tb2d(const frkc2_problem& p, const PassArgs& a, const TbIo& io, cudaStream_t st,
                             bool overlap_previous, int cells) {
  (void)p;
  const bool per = a.bc == FRKC2_BC_PERIODIC;
  if (cells == 2) return per ? launch_c<2, true, 1>(a, io, st, overlap_previous) : launch_c<2, false, 1>(a, io, st, overlap_previous);
  if (a.k % 4 == 0) return per ? launch_c<4, true, 4>(a, io, st, overlap_previous) : launch_c<4, false, 4>(a, io, st, overlap_previous);
  if (a.k % 2 == 0) return per ? launch_c<4, true, 2>(a, io, st, overlap_previous) : launch_c<4, false, 2>(a, io, st, overlap_previous);
  return per ? launch_c<4, true, 1>(a, io, st, overlap_previous) : launch_c<4, false, 1>(a, io, st, overlap_previous);
}

}  // namespace frkc2
