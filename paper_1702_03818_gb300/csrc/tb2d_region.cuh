// 2D temporally blocked stage pass for FP32 (fixed conductivity) with the state in registers:
// the computation of one 64 x 64 region for the batched persistent launch (batched.cu), and
// the region constants and helpers (RT_R, RT_THREADS, wrap_r, sub2) of the other register-
// tiled kernels.  The single-problem FP32 pass (pass_tb2d.cu) keeps its own copy of the same
// computation, which compiles to a faster kernel than this function inlined into one.
//
// A CTA of 16 x 16 threads owns a 64 x 64 region: its output tile (64 - 2k)^2 plus a k-cell
// halo recomputed redundantly (region-edge values go stale one cell per stage, which never
// reaches the output tile).  Thread (tx, ty) owns the 4 x 4 cells at columns 4tx..4tx+3,
// rows 4ty..4ty+3 and keeps, for all k stages, their complex state (32 floats) and their 40
// face conductivities in registers.  Per stage:
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
#pragma once

#include <cstdint>

#include <cuda_runtime.h>

namespace frkc2 {

constexpr int RT_R = 64;         // region edge (cells)
constexpr int RT_THREADS = 256;  // 16 x 16 threads of 4 x 4 cells

struct RegionShared {
  float4 bot[2][2][16][16];  // [stage parity][U, V][ty][tx]: the thread's row 0
  float4 top[2][2][16][16];  // its row 3
};

__device__ __forceinline__ int wrap_r(int g, int n) {
  if (g >= 0 && g < n) return g;
  if (g < 0 && g >= -n) return g + n;
  if (g >= n && g < 2 * n) return g - n;
  const int r = g % n;
  return r < 0 ? r + n : r;
}

// a - b on both halves in one packed instruction (sm_100 family)
__device__ __forceinline__ float2 sub2(float2 a, float2 b) { return __fadd2_rn(a, make_float2(-b.x, -b.y)); }

// One 64 x 64 region: load, kq stages, store the cells at distance >= k from the region edge.
// x0, y0: grid coordinates of the region's corner (tile origin - k).  coef(j, ca, cb) gives the
// stage coefficients.  L1BYPASS: state loads through L2 only (buffers written by other CTAs
// of the same launch).  Returns true if a stored value is not finite (when check_finite).
// pfx, pfy, pin, pout: row pitches of the faces and of the state read and written.  A thread's rows move as
// 16-byte vectors where pitch, k and pointer keep them aligned and they lie in the grid in one piece.
template <bool PERIODIC, bool L1BYPASS, class Coef>
__device__ __forceinline__ bool tb2d_region(RegionShared& sh, int nx, int ny, int k, int kq, int x0, int y0,
                                            const float* __restrict__ Uin, const float* __restrict__ Vin,
                                            float* __restrict__ Uo, float* __restrict__ Vo,
                                            const float* __restrict__ FX, const float* __restrict__ FY,
                                            int pfx, int pfy, int pin, int pout, Coef coef, bool check_finite) {
  const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;

  // wrapped (periodic) or raw (Dirichlet) grid rows / columns of the thread's cells; the fifth
  // entry is the next row / column (north and east faces)
  int gyr[5], gxc[5];
  bool yin[5], xin[5];
#pragma unroll
  for (int i = 0; i < 5; ++i) {
    const int gx = x0 + 4 * tx + i, gy = y0 + 4 * ty + i;
    gxc[i] = PERIODIC ? wrap_r(gx, nx) : gx;
    gyr[i] = PERIODIC ? wrap_r(gy, ny) : gy;
    xin[i] = gx >= 0 && gx < nx;
    yin[i] = gy >= 0 && gy < ny;
  }
  unsigned inside = 0;  // Dirichlet: bit 4r + c set if cell (r, c) lies in the grid
#pragma unroll
  for (int r = 0; r < 4; ++r)
#pragma unroll
    for (int c = 0; c < 4; ++c)
      if (xin[c] && yin[r]) inside |= 1u << (4 * r + c);
  const bool run = (gxc[0] & 3) == 0 && gxc[3] == gxc[0] + 3 && (PERIODIC || (xin[0] && xin[3]));
  // fx[r][c]: x face c of row r (the west face of cell c; c = 4 is the east face of cell 3);
  // FY2[r]: y faces r as cell pairs (the south faces of row r; r = 4 the north faces of row 3)
  float fx[4][5];
  float2 FY2[5][2];
  if (run && ((pfx | pfy) & 3) == 0) {
#pragma unroll
    for (int r = 0; r < 5; ++r) {
      float4 y = make_float4(0.f, 0.f, 0.f, 0.f), x = y;
      float x4 = 0.f;
      if (PERIODIC || (gyr[r] >= 0 && gyr[r] <= ny)) y = *reinterpret_cast<const float4*>(FY + size_t(gyr[r]) * pfy + gxc[0]);
      FY2[r][0] = make_float2(y.x, y.y);
      FY2[r][1] = make_float2(y.z, y.w);
      if (r < 4) {
        if (PERIODIC || yin[r]) {
          const float* q = FX + size_t(gyr[r]) * pfx + gxc[0];
          x = *reinterpret_cast<const float4*>(q);
          x4 = q[4];  // (periodic face nx repeats face 0)
        }
        fx[r][0] = x.x;
        fx[r][1] = x.y;
        fx[r][2] = x.z;
        fx[r][3] = x.w;
        fx[r][4] = x4;
      }
    }
  } else {
#pragma unroll
    for (int r = 0; r < 5; ++r) {
#pragma unroll
      for (int c = 0; c < 5; ++c) {
        if (r < 4) {
          float v = 0.f;
          if (PERIODIC || (yin[r] && gxc[c] >= 0 && gxc[c] <= nx)) v = FX[size_t(gyr[r]) * pfx + gxc[c]];
          fx[r][c] = v;
        }
        if (c < 4) {
          float v = 0.f;
          if (PERIODIC || (xin[c] && gyr[r] >= 0 && gyr[r] <= ny)) v = FY[size_t(gyr[r]) * pfy + gxc[c]];
          (c & 1 ? FY2[r][c >> 1].y : FY2[r][c >> 1].x) = v;
        }
      }
    }
  }
  // the state as horizontal cell pairs: U2[r][h] = (U[r][2h], U[r][2h + 1])
  float2 U2[4][2], V2[4][2];
  if (run && (pin & 3) == 0 && (reinterpret_cast<uintptr_t>(Uin) & 15) == 0) {
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      float4 u = make_float4(0.f, 0.f, 0.f, 0.f), v = u;
      if (PERIODIC || yin[r]) {
        const size_t g = size_t(gyr[r]) * pin + gxc[0];
        const float4* qu = reinterpret_cast<const float4*>(Uin + g);
        u = L1BYPASS ? __ldcg(qu) : *qu;
        if (Vin) {
          const float4* qv = reinterpret_cast<const float4*>(Vin + g);
          v = L1BYPASS ? __ldcg(qv) : *qv;
        }
      }
      U2[r][0] = make_float2(u.x, u.y);
      U2[r][1] = make_float2(u.z, u.w);
      V2[r][0] = make_float2(v.x, v.y);
      V2[r][1] = make_float2(v.z, v.w);
    }
  } else {
#pragma unroll
    for (int r = 0; r < 4; ++r)
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        float uu = 0.f, vv = 0.f;
        if (PERIODIC || (inside & (1u << (4 * r + c)))) {
          const size_t g = size_t(gyr[r]) * pin + gxc[c];
          uu = L1BYPASS ? __ldcg(Uin + g) : Uin[g];
          if (Vin) vv = L1BYPASS ? __ldcg(Vin + g) : Vin[g];
        }
        (c & 1 ? U2[r][c >> 1].y : U2[r][c >> 1].x) = uu;
        (c & 1 ? V2[r][c >> 1].y : V2[r][c >> 1].x) = vv;
      }
  }

  const float4 z4 = make_float4(0.f, 0.f, 0.f, 0.f);
  for (int j = 0; j < kq; ++j) {
    const int b = j & 1;
    sh.bot[b][0][ty][tx] = make_float4(U2[0][0].x, U2[0][0].y, U2[0][1].x, U2[0][1].y);
    sh.bot[b][1][ty][tx] = make_float4(V2[0][0].x, V2[0][0].y, V2[0][1].x, V2[0][1].y);
    sh.top[b][0][ty][tx] = make_float4(U2[3][0].x, U2[3][0].y, U2[3][1].x, U2[3][1].y);
    sh.top[b][1][ty][tx] = make_float4(V2[3][0].x, V2[3][0].y, V2[3][1].x, V2[3][1].y);
    __syncthreads();
    // the region's outermost thread rows have no neighbour row here: their edge goes stale
    const float4 su4 = ty > 0 ? sh.top[b][0][ty - 1][tx] : z4, sv4 = ty > 0 ? sh.top[b][1][ty - 1][tx] : z4;
    const float4 nu4 = ty < 15 ? sh.bot[b][0][ty + 1][tx] : z4, nv4 = ty < 15 ? sh.bot[b][1][ty + 1][tx] : z4;
    float ca, cb;
    coef(j, ca, cb);
    const float2 ca2 = make_float2(ca, ca), cb2 = make_float2(cb, cb), ncb2 = make_float2(-cb, -cb);
    const float2 su2[2] = {make_float2(su4.x, su4.y), make_float2(su4.z, su4.w)};
    const float2 sv2[2] = {make_float2(sv4.x, sv4.y), make_float2(sv4.z, sv4.w)};
    const float2 nu2[2] = {make_float2(nu4.x, nu4.y), make_float2(nu4.z, nu4.w)};
    const float2 nv2[2] = {make_float2(nv4.x, nv4.y), make_float2(nv4.z, nv4.w)};
    // differences across the south faces of the current row: W(r) - W(r - 1)
    float2 dsU[2], dsV[2];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      dsU[h] = sub2(U2[0][h], su2[h]);
      dsV[h] = sub2(V2[0][h], sv2[h]);
    }
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      // columns beyond the thread's own, before this row is updated
      const float wU = __shfl_up_sync(0xffffffffu, U2[r][1].y, 1, 16);
      const float wV = __shfl_up_sync(0xffffffffu, V2[r][1].y, 1, 16);
      const float eU = __shfl_down_sync(0xffffffffu, U2[r][0].x, 1, 16);
      const float eV = __shfl_down_sync(0xffffffffu, V2[r][0].x, 1, 16);
      const float u[6] = {wU, U2[r][0].x, U2[r][0].y, U2[r][1].x, U2[r][1].y, eU};
      const float v[6] = {wV, V2[r][0].x, V2[r][0].y, V2[r][1].x, V2[r][1].y, eV};
      // dx[c]: across x face c, W(c) - W(c - 1), each formed once for the two cells of the face
      float dxU[5], dxV[5];
#pragma unroll
      for (int c = 0; c < 5; ++c) {
        dxU[c] = u[c + 1] - u[c];
        dxV[c] = v[c + 1] - v[c];
      }
      // x part of f per cell, written straight into the halves of the pairs
      float2 fU[2], fV[2];
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int c = 2 * h;
        fU[h].x = fx[r][c + 1] * dxU[c + 1] - fx[r][c] * dxU[c];
        fU[h].y = fx[r][c + 2] * dxU[c + 2] - fx[r][c + 1] * dxU[c + 1];
        fV[h].x = fx[r][c + 1] * dxV[c + 1] - fx[r][c] * dxV[c];
        fV[h].y = fx[r][c + 2] * dxV[c + 2] - fx[r][c + 1] * dxV[c + 1];
      }
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const float2 nU = r < 3 ? U2[r + 1][h] : nu2[h];
        const float2 nV = r < 3 ? V2[r + 1][h] : nv2[h];
        const float2 dnU = sub2(nU, U2[r][h]), dnV = sub2(nV, V2[r][h]);
        // y part, two cells per instruction: f += k_n d_n - k_s d_s
        const float2 nks = make_float2(-FY2[r][h].x, -FY2[r][h].y);
        fU[h] = __ffma2_rn(nks, dsU[h], __ffma2_rn(FY2[r + 1][h], dnU, fU[h]));
        fV[h] = __ffma2_rn(nks, dsV[h], __ffma2_rn(FY2[r + 1][h], dnV, fV[h]));
        // W += (ca + i cb) f
        float2 un = __ffma2_rn(ncb2, fV[h], __ffma2_rn(ca2, fU[h], U2[r][h]));
        float2 vn = __ffma2_rn(cb2, fU[h], __ffma2_rn(ca2, fV[h], V2[r][h]));
        if (!PERIODIC) {
          if (!(inside & (1u << (4 * r + 2 * h)))) un.x = vn.x = 0.f;
          if (!(inside & (1u << (4 * r + 2 * h + 1)))) un.y = vn.y = 0.f;
        }
        U2[r][h] = un;
        V2[r][h] = vn;
        dsU[h] = dnU;
        dsV[h] = dnV;
      }
    }
  }

  // store the output tile: region cells at distance >= k from the region edge
  bool bad = false;
  const int gx0 = x0 + 4 * tx;
  const bool vout = (pout & 3) == 0 && (reinterpret_cast<uintptr_t>(Uo) & 15) == 0 && (gx0 & 3) == 0 && 4 * tx >= k &&
                    4 * tx + 4 <= RT_R - k && gx0 + 4 <= nx;
#pragma unroll
  for (int r = 0; r < 4; ++r) {
    const int ry = 4 * ty + r;
    const int gy = y0 + ry;
    if (ry < k || ry >= RT_R - k || gy >= ny) continue;
    const size_t row = size_t(gy) * pout;
    if (vout) {
      *reinterpret_cast<float4*>(Uo + row + gx0) = make_float4(U2[r][0].x, U2[r][0].y, U2[r][1].x, U2[r][1].y);
      if (Vo) *reinterpret_cast<float4*>(Vo + row + gx0) = make_float4(V2[r][0].x, V2[r][0].y, V2[r][1].x, V2[r][1].y);
    }
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      const int rx = 4 * tx + c;
      const int gx = gx0 + c;
      if (rx < k || rx >= RT_R - k || gx >= nx) continue;
      const float uu = (c & 1) ? U2[r][c >> 1].y : U2[r][c >> 1].x;
      if (!vout) {
        Uo[row + gx] = uu;
        if (Vo) Vo[row + gx] = (c & 1) ? V2[r][c >> 1].y : V2[r][c >> 1].x;
      }
      if (check_finite) bad |= (__float_as_uint(uu) & 0x7f800000u) == 0x7f800000u;
    }
  }
  return bad;
}

}  // namespace frkc2
