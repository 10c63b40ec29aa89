// Temporally blocked Brusselator pass (FP32): k stages of Sec. 3, Eq. 13 on the complex pair (v, w) per round
// trip through memory, the state in registers.
//
// The per-stage forms (bruss2d.cu) move 32 bytes a cell-stage; this one moves 32 bytes a cell and k stages.
// A CTA of 16 x 16 threads owns a region of 16C x 16C cells: its output tile (16C - 2k)^2 plus a k-cell halo
// that it recomputes (region-edge values go stale one cell a stage and never reach the output tile).  Thread
// (tx, ty) keeps the C x C cells at columns C tx, rows C ty -- 4 C^2 floats -- for all k stages; per stage its
// bottom and top rows go through shared memory (double-buffered by stage parity, one barrier a stage) and the
// columns beyond its own come from the adjacent threads by 16-lane shuffles.  Every cell is updated by the
// operations of k_bruss2d in their order, so the results are bit for bit those of the per-stage forms.
//
// What bounds it: FP32 issue (57 instructions a computed cell-stage, 41 of them arithmetic, at 65 % issue), and on
// grids of less than a wave the latency of a stage.  C = 4 (64 registers of state, 2 CTAs per SM) recomputes
// least and serves large grids; at its 128 registers it spills (88 bytes stored and 220
// loaded a thread, zero flux 148 and 288).  C = 2 gives four times as many CTAs, for grids that would leave SMs idle.
// 2048^2, s = 16, 10 steps: 6165 -> 2218 us (41 % of the FP32 rate counting the halo); 200^2, 42 steps: 1859 ->
// 450 us; 700 x 611 zero flux, 10 steps: 875 -> 436 us.
#include <algorithm>

#include <cuda_runtime.h>

#include "frkc2_internal.h"

namespace frkc2 {
namespace {

constexpr int BT_THREADS = 256;  // 16 x 16 threads of C x C cells
constexpr int BT_KMAX = 8;

// a row of C cells of one component
template <int C> struct Row;
template <> struct Row<4> { using type = float4; };
template <> struct Row<2> { using type = float2; };
__device__ __forceinline__ void row_get(float4 v, float (&a)[4]) { a[0] = v.x; a[1] = v.y; a[2] = v.z; a[3] = v.w; }
__device__ __forceinline__ void row_get(float2 v, float (&a)[2]) { a[0] = v.x; a[1] = v.y; }
__device__ __forceinline__ float4 row_of(const float (&a)[4]) { return make_float4(a[0], a[1], a[2], a[3]); }
__device__ __forceinline__ float2 row_of(const float (&a)[2]) { return make_float2(a[0], a[1]); }

struct BrTbArgs {
  const float* in[4];   // Re v, Im v, Re w, Im w; the imaginary parts nullptr: zero
  float* out[4];        // the imaginary parts nullptr: not stored
  int nx, ny, k;
  float Dd, A, B1, B;   // D / dx^2, A, B + 1, B
  int check_finite;
  int vec;              // rows of C cells are aligned and never wrap: whole-row loads and stores
  unsigned* status;
  float hr[BT_KMAX], hi[BT_KMAX];  // dt a_l of the pass's stages
};

template <int C>
struct BrTbShared {
  typename Row<C>::type bot[2][4][16][16];  // [stage parity][component][ty][tx]: the thread's first row
  typename Row<C>::type top[2][4][16][16];  // its last row
};

__device__ __forceinline__ int bt_wrap(int g, int n) {
  if (g < 0) g += n;
  if (g >= n) g -= n;
  if (g >= 0 && g < n) return g;
  g %= n;
  return g < 0 ? g + n : g;
}

// EDGE (zero flux only): the region touches the grid's boundary, where a neighbour outside is the cell
// itself.  nb: bits i the columns whose west, 4 + i whose east, 8 + i the rows whose south, 12 + i whose
// north neighbour is outside.
template <int C, bool EDGE>
__device__ __forceinline__ void bt_stages(BrTbShared<C>& sh, const BrTbArgs& p, float (&W)[4][C][C], unsigned nb) {
  const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
  const float Dd = p.Dd, A = p.A, B1 = p.B1, B = p.B;
  for (int j = 0; j < p.k; ++j) {
    const int b = j & 1;
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      sh.bot[b][c][ty][tx] = row_of(W[c][0]);
      sh.top[b][c][ty][tx] = row_of(W[c][C - 1]);
    }
    __syncthreads();
    const float hr = p.hr[j], hi = p.hi[j];
    // the region's outermost thread rows have no neighbour row here: their edge goes stale
    const int ts = ty > 0 ? ty - 1 : 0, tn = ty < 15 ? ty + 1 : 15;
    float S[4][C];  // the old values of the row below
#pragma unroll
    for (int c = 0; c < 4; ++c) row_get(sh.top[b][c][ts][tx], S[c]);
#pragma unroll
    for (int r = 0; r < C; ++r) {
      float L[4][C];  // Laplacian sums of the row
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        float N[C];
        if (r == C - 1) {
          row_get(sh.bot[b][c][tn][tx], N);
        } else {
#pragma unroll
          for (int i = 0; i < C; ++i) N[i] = W[c][r < C - 1 ? r + 1 : r][i];
        }
        const float w = __shfl_up_sync(0xffffffffu, W[c][r][C - 1], 1, 16);
        const float e = __shfl_down_sync(0xffffffffu, W[c][r][0], 1, 16);
#pragma unroll
        for (int i = 0; i < C; ++i) {
          const float m = W[c][r][i];
          float E = i < C - 1 ? W[c][r][i < C - 1 ? i + 1 : i] : e, Wt = i > 0 ? W[c][r][i > 0 ? i - 1 : 0] : w;
          float No = N[i], So = S[c][i];
          if (EDGE) {
            if (nb >> i & 1) Wt = m;
            if (nb >> (4 + i) & 1) E = m;
            if (nb >> (8 + r) & 1) So = m;
            if (nb >> (12 + r) & 1) No = m;
          }
          L[c][i] = ((E + Wt) + (No + So)) - 4.f * m;
        }
      }
#pragma unroll
      for (int i = 0; i < C; ++i) {
        const float vr = W[0][r][i], vi = W[1][r][i], wr = W[2][r][i], wi = W[3][r][i];
        const float qr = vr * vr - vi * vi;
        const float qi = (vr + vr) * vi;
        const float pr = qr * wr - qi * wi;
        const float pi = qr * wi + qi * wr;
        const float fvr = Dd * L[0][i] + ((A - B1 * vr) + pr);
        const float fvi = Dd * L[1][i] + (pi - B1 * vi);
        const float fwr = Dd * L[2][i] + (B * vr - pr);
        const float fwi = Dd * L[3][i] + (B * vi - pi);
        S[0][i] = vr;
        S[1][i] = vi;
        S[2][i] = wr;
        S[3][i] = wi;
        W[0][r][i] = vr + hr * fvr - hi * fvi;
        W[1][r][i] = vi + hr * fvi + hi * fvr;
        W[2][r][i] = wr + hr * fwr - hi * fwi;
        W[3][r][i] = wi + hr * fwi + hi * fwr;
      }
    }
  }
}

template <int C, bool PERIODIC>
__global__ void __launch_bounds__(BT_THREADS, C == 4 ? 2 : 4) k_bruss_tb2d(const BrTbArgs p) {
  using R = typename Row<C>::type;
  constexpr int BT_R = 16 * C;  // region edge (cells)
  extern __shared__ __align__(16) unsigned char smem_raw[];
  BrTbShared<C>& sh = *reinterpret_cast<BrTbShared<C>*>(smem_raw);
  const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
  const int k = p.k, T = BT_R - 2 * k, nx = p.nx, ny = p.ny;
  const int rx = blockIdx.x * T - k, ry = blockIdx.y * T - k;  // the region's corner
  const int x0 = rx + C * tx, y0 = ry + C * ty;
  // launched with programmatic stream serialization: the next pass may start its CTAs as this one's
  // exit, and every global load below comes after the previous launch has completed
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  asm volatile("griddepcontrol.wait;" ::: "memory");
  int gx[C];
  unsigned nb = 0;
#pragma unroll
  for (int i = 0; i < C; ++i) {
    gx[i] = PERIODIC ? bt_wrap(x0 + i, nx) : min(max(x0 + i, 0), nx - 1);
    if (!PERIODIC) {
      if (x0 + i == 0) nb |= 1u << i;
      if (x0 + i == nx - 1) nb |= 16u << i;
      if (y0 + i == 0) nb |= 256u << i;
      if (y0 + i == ny - 1) nb |= 4096u << i;
    }
  }
  float W[4][C][C];
  // (a row of C cells outside a zero-flux grid is loaded from inside it: its values are not used)
  const int gv = PERIODIC ? gx[0] : min(max(x0, 0), nx - C);
#pragma unroll
  for (int r = 0; r < C; ++r) {
    const int gy = PERIODIC ? bt_wrap(y0 + r, ny) : min(max(y0 + r, 0), ny - 1);
    const size_t row = size_t(gy) * nx;
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      if (p.vec && p.in[c]) {
        row_get(__ldg(reinterpret_cast<const R*>(p.in[c] + row + gv)), W[c][r]);
      } else {
#pragma unroll
        for (int i = 0; i < C; ++i) W[c][r][i] = p.in[c] ? __ldg(p.in[c] + row + gx[i]) : 0.f;
      }
    }
  }
  if (!PERIODIC && (rx <= 0 || ry <= 0 || rx + BT_R >= nx || ry + BT_R >= ny))
    bt_stages<C, true>(sh, p, W, nb);
  else
    bt_stages<C, false>(sh, p, W, nb);
  bool bad = false;
#pragma unroll
  for (int r = 0; r < C; ++r) {
    const int yy = C * ty + r, gy = y0 + r;
    if (yy < k || yy >= BT_R - k || gy >= ny) continue;
    const size_t row = size_t(gy) * nx;
    if (p.vec) {  // (k is then a multiple of C, so a row of C cells is output as a whole or not at all)
      if (C * tx < k || C * tx >= BT_R - k || x0 >= nx) continue;
#pragma unroll
      for (int c = 0; c < 4; ++c)
        if (p.out[c]) *reinterpret_cast<R*>(p.out[c] + row + x0) = row_of(W[c][r]);
    }
#pragma unroll
    for (int i = 0; i < C; ++i) {
      const int xx = C * tx + i, gc = x0 + i;
      if (xx < k || xx >= BT_R - k || gc >= nx) continue;
      if (!p.vec) {
#pragma unroll
        for (int c = 0; c < 4; ++c)
          if (p.out[c]) p.out[c][row + gc] = W[c][r][i];
      }
      if (p.check_finite)
        bad |= (__float_as_uint(W[0][r][i]) & 0x7f800000u) == 0x7f800000u || (__float_as_uint(W[2][r][i]) & 0x7f800000u) == 0x7f800000u;
    }
  }
  if (bad) atomicOr(p.status, ST_NONFINITE);
}

template <int C, bool PERIODIC>
Residency bt_residency() {
  static SpreadKernel own;
  return spread_residency(own, k_bruss_tb2d<C, PERIODIC>, BT_THREADS, sizeof(BrTbShared<C>), 0);
}

template <int C, bool PERIODIC>
cudaError_t bt_launch(const BrTbArgs& a, cudaStream_t st, bool overlap_previous) {
  const Residency res = bt_residency<C, PERIODIC>();
  if (res.err != cudaSuccess) return res.err;
  const int T = 16 * C - 2 * a.k;
  const long long regions = (long long)((a.nx + T - 1) / T) * ((a.ny + T - 1) / T);
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((a.nx + T - 1) / T, (a.ny + T - 1) / T, 1);
  cfg.blockDim = dim3(BT_THREADS, 1, 1);
  cfg.dynamicSmemBytes = spread_smem(sizeof(BrTbShared<C>), regions, res.sms, res.per_sm);
  cfg.stream = st;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at;
  cfg.numAttrs = overlap_previous ? 1 : 0;
  const cudaError_t e = cudaLaunchKernelEx(&cfg, k_bruss_tb2d<C, PERIODIC>, a);
  count_launch();
  return e != cudaSuccess ? e : cudaGetLastError();
}

}  // namespace

// Cells per thread and stages per pass, from a model of a pass's time in us fitted to measurements (periodic,
// s = 16): regions of 32 x 32 (C = 2) take 2.1 + 0.32 k alone on an SM and 2.7 + 0.77 k with all 4 resident,
// regions of 64 x 64 (C = 4) 3.0 + 0.8 k and 5.8 + 1.32 k with both, and unaligned rows 0.7 / 4.5 more.
// (2048^2: C = 4, k = 4 55.5 us a pass; 192^2: C = 2, k = 8 4.3 us.)
BrussTb bruss_tb2d_shape(int nx, int ny, int s) {
  BrussTb best{0, 0};
  double least = 0.0;
  for (int C = 2; C <= 4; C += 2) {
    const Residency res = C == 2 ? bt_residency<2, true>() : bt_residency<4, true>();
    if (res.err != cudaSuccess) return BrussTb{0, 0};
    const long long slots = (long long)res.sms * res.per_sm;
    auto pass = [&](int k) {
      const int T = 16 * C - 2 * k;
      const long long regions = (long long)((nx + T - 1) / T) * ((ny + T - 1) / T);
      const double waves = double((regions + slots - 1) / slots);
      const double r = double(std::min<long long>(res.per_sm, (regions + res.sms - 1) / res.sms));
      const double one = C == 2 ? 1.9 + 0.2 * r + (0.17 + 0.15 * r) * k : (r < 2.0 ? 3.0 + 0.8 * k : 5.8 + 1.32 * k);
      return waves * (one + (k % C || nx % C ? (C == 2 ? 0.7 : 4.5) : 0.0));
    };
    for (int k = 1; k <= std::min(BT_KMAX, s / 2); ++k) {
      const double cost = (s / k) * pass(k) + (s % k ? pass(s % k) : 0.0);
      if (best.k == 0 || cost < least) {
        best.cells = C;
        best.k = k;
        least = cost;
      }
    }
  }
  // A launch's y axis ends at 65535: where the regions of a pass are more (from 1.5 million rows on), the persistent
  // kernel.  (Regions along one axis would have no such end, but 2048^2, s = 16, 10 steps, takes 2213 -> 2250 us with them.)
  for (int k : {best.k, best.k ? s % best.k : 0})
    if (k > 0 && (ny - 1) / (16 * best.cells - 2 * k) >= 65535) return BrussTb{0, 0};
  return best;
}

cudaError_t launch_bruss_tb2d(const frkc2_bruss_problem& p, const frkc2_plan_s& plan, double dt, int nsteps, BrussTb shape,
                              float* v, float* w, void* const P[2][4], unsigned* status, cudaStream_t st) {
  BrTbArgs a{};
  a.nx = int(p.nx);
  a.ny = int(p.ny);
  a.Dd = float(p.D / (p.dx * p.dx));
  a.A = float(p.A);
  a.B1 = float(p.B + 1.0);
  a.B = float(p.B);
  a.status = status;
  const int s = plan.s, C = shape.cells, npass = (s + shape.k - 1) / shape.k;  // at least two: no pass writes what it reads
  const bool per = p.bc == FRKC2_BC_PERIODIC;
  const uintptr_t base = reinterpret_cast<uintptr_t>(v) | reinterpret_cast<uintptr_t>(w);
  for (int n = 0; n < nsteps; ++n)
    for (int q = 0; q < npass; ++q) {
      const NvtxRange pass_range("frkc2 pass");
      const bool first = q == 0, last = q == npass - 1;
      const int l0 = q * shape.k;
      a.k = std::min(shape.k, s - l0);
      for (int c = 0; c < 4; ++c) {
        a.in[c] = first ? (c == 0 ? v : c == 2 ? w : nullptr) : static_cast<const float*>(P[(q - 1) & 1][c]);
        a.out[c] = last ? (c == 0 ? v : c == 2 ? w : nullptr) : static_cast<float*>(P[q & 1][c]);
      }
      a.check_finite = last;
      a.vec = a.k % C == 0 && a.nx % C == 0 && (base & (4 * C - 1)) == 0;
      for (int j = 0; j < a.k; ++j) {
        a.hr[j] = float(dt * plan.a_re[l0 + j]);
        a.hi[j] = float(dt * plan.a_im[l0 + j]);
      }
      const bool ov = n > 0 || q > 0;
      const cudaError_t e = C == 2 ? (per ? bt_launch<2, true>(a, st, ov) : bt_launch<2, false>(a, st, ov))
                                   : (per ? bt_launch<4, true>(a, st, ov) : bt_launch<4, false>(a, st, ov));
      if (e != cudaSuccess) return e;
    }
  return cudaSuccess;
}

}  // namespace frkc2
