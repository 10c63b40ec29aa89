// Internal declarations shared by the FRKC2 host code and kernels (not part of the C ABI).
#pragma once

#include <algorithm>
#include <atomic>
#include <cstddef>
#include <cstdint>
#include <mutex>
#include <vector>

#include <cuda_runtime.h>
#include <nvtx3/nvToolsExt.h>

#include "frkc2.h"

struct frkc2_plan_s {
  int s = 0;
  double beta = 0.0;
  double Q = 0.0;
  int n_iter = 0;
  std::vector<int> order;     // root index of each stage
  std::vector<double> a_re;   // step sizes in stage order
  std::vector<double> a_im;
  bool paired = false;        // conjugates adjacent: stages 2p, 2p+1 form one real pair
  double gain = 0.0;          // rounding gain of the stage order (frkc2_plan_rounding_gain)
};

namespace frkc2 {

// NVTX range for the enclosing scope (host timeline: a call, a step, a pass; no cost without a
// tool attached)
struct NvtxRange {
  explicit NvtxRange(const char* name) { nvtxRangePushA(name); }
  ~NvtxRange() { nvtxRangePop(); }
  NvtxRange(const NvtxRange&) = delete;
  NvtxRange& operator=(const NvtxRange&) = delete;
};

constexpr int KMAX = 16;                 // most stages in one pass
constexpr unsigned ST_NONFINITE = 1u;    // status word bits
constexpr unsigned ST_TIMEOUT = 2u;
constexpr unsigned ST_BOUNDS = 4u;       // bounds-checking build: an index left its array

// Index checks of the bounds-checking build (FRKC2_DEBUG_BOUNDS, libfrkc2_debug.so): false
// and ST_BOUNDS latched in *status when ok is false, the caller then skipping the access.  In
// the normal build it is the constant true and the check compiles away.
#ifdef FRKC2_DEBUG_BOUNDS
__device__ __forceinline__ bool in_bounds(bool ok, unsigned* status) {
  if (!ok) atomicOr(status, ST_BOUNDS);
  return ok;
}
#else
__device__ __forceinline__ constexpr bool in_bounds(bool, unsigned*) { return true; }
#endif

// state layouts a pass reads or writes (the streaming pass honours them; the tile kernels
// always use planar U, V)
constexpr int PASS_IO_REAL = 0;     // U only (imaginary part zero on input, dropped on output)
constexpr int PASS_IO_PLANAR = 1;   // separate U and V arrays
constexpr int PASS_IO_COMPLEX = 2;  // one interleaved (U, V) array at U_in / U_out

inline size_t align256(size_t b) { return (b + 255) & ~size_t(255); }

// One k-stage pass over the grid: read (U, V), apply k stages, write (U, V).
struct PassArgs {
  int ndim, bc;
  int nx, ny, nz;         // grid extents (1 past ndim)
  int tx, ty, tz;         // output tile of one CTA
  int hx, hy, hz;         // halo width per axis: k along present axes, 0 otherwise
  int k;                  // stages in this pass
  int check_finite;       // flag non-finite outputs in the status word
  int in_mode, out_mode;  // PASS_IO_* (streaming pass only)
  const void* U_in;       // real part of the pass input
  const void* V_in;       // imaginary part; nullptr = zero (first pass of a step)
  void* U_out;
  void* V_out;            // nullptr = not stored (last pass of a step)
  const void* H_in;       // embedded first-order solution (tile kernel only); nullptr = none
  void* H_out;
  const void* fx;         // face conductivities (FIELD / CONST), layouts in faces_layout()
  const void* fy;
  const void* fz;
  double kc, kp;          // POWER: kappa(w) = 1 + kc * w^kp
  unsigned* status;
  double ca[KMAX];        // dt Re(a_l) / dx^2 for the pass's stages
  double cb[KMAX];        // dt Im(a_l) / dx^2
  float caf[KMAX];        // the same, rounded to float once on the host
  float cbf[KMAX];
};

// Face arrays: x faces [nz][ny][nx+1], y faces [nz][ny+1][nx], z faces [nz+1][ny][nx];
// face index i along an axis lies between cells i-1 and i.
struct FaceLayout {
  size_t nfx, nfy, nfz;   // element counts (0 for absent axes)
};
FaceLayout faces_layout(const frkc2_problem& p);

// Workspace layout of frkc2_step (byte offsets from the workspace base).
struct StepLayout {
  size_t status, fx, fy, fz, fen, ua, va, ub, vb, total;
};
StepLayout step_layout(const frkc2_problem& p);

size_t state_bytes(int precision);
size_t arith_bytes(int precision);
size_t cells(const frkc2_problem& p);

// Launchers (return cudaGetLastError()).
cudaError_t launch_faces(const frkc2_problem& p, void* fx, void* fy, void* fz, cudaStream_t st);
cudaError_t launch_rho(const frkc2_problem& p, const void* u, double* rho_dev, cudaStream_t st);
cudaError_t launch_pass_generic(const frkc2_problem& p, const PassArgs& a, cudaStream_t st);
cudaError_t launch_err_sum(const frkc2_problem& p, const void* u, const void* h, double* out, cudaStream_t st);
cudaError_t launch_pass_stream2d(const frkc2_problem& p, const PassArgs& a, const void* fen, cudaStream_t st);
size_t face_pair_bytes(const frkc2_problem& p);
cudaError_t launch_face_pairs(const frkc2_problem& p, const void* fx, const void* fy, void* out, cudaStream_t st);
// overlap_previous: the launch may start while the previous launch on the stream (a pass of
// the same kind) finishes; its CTAs read the pass input only after that launch completes.
// cells: a thread's cells along each axis, 4 (64 x 64 regions) or 2 (32 x 32, k < 16)
struct TbIo {
  const float* fxp;  // x faces [ny][fpitch], y faces [ny + 1][fpitch] in rows padded to a multiple of 4 (launch_faces_padded),
  const float* fyp;  // or nullptr: the unpadded arrays of PassArgs
  int fpitch;
  int in_pitch, out_pitch;  // row pitch of the state read and written
};
cudaError_t launch_pass_tb2d(const frkc2_problem& p, const PassArgs& a, const TbIo& io, cudaStream_t st,
                             bool overlap_previous, int cells = 4);
cudaError_t launch_faces_padded(const frkc2_problem& p, float* fxp, float* fyp, int pitch, cudaStream_t st);
// region size and stages per pass for a grid and a plan of s stages, with the model's us a step
struct TbShape {
  int cells, k;
  double us;
};
TbShape tb2d_shape(int nx, int ny, int s);
// 64 x 64 regions and an even k: a cell's column keeps its parity in its thread, and with it its rounding
TbShape tb2d_shape_even(int nx, int ny, int s);
bool small1d_supported(const frkc2_problem& p, int s);
// 2D FP32 wavefront pass (pass_wf2d.cu): CTAs of WF_NW warps stream column strips of
// 64 WF_NW cells up the grid with up to WF_KMAX stage levels in flight; rows arrive by TMA.
constexpr int WF_NW = 4;
int wf2d_face_pitch(int nx);
// computed / output cell-stages of the wavefront pass at its default launch
double wf2d_recompute(int nx, int ny, int k);
double wf2d_pass8_us(int nx, int ny);
// k stages per pass and s stages per step: every pass (the last may be shorter) needs an
// instantiated stage count (1, 2, 4, 6, 8, 10 or 12)
bool wf2d_supported(const frkc2_problem& p, int k, int s, const void* u);
cudaError_t launch_faces_wf(const frkc2_problem& p, const void* fx, const void* fy, void* out, cudaStream_t st);
// chunk_rows: rows per CTA (0 = one wave of two CTAs per SM); in_real / out_real: the pass reads
// / writes the real state (float [ny][nx]) instead of interleaved (U, V) float2 [ny][nx]
cudaError_t launch_pass_wf2d(const frkc2_problem& p, const PassArgs& a, const void* faces_wf, int chunk_rows,
                             bool in_real, bool out_real, cudaStream_t st, bool overlap_previous,
                             long long wait_limit = 0, int fault_inject = 0);
cudaError_t launch_small1d(const frkc2_problem& p, const frkc2_plan_s& plan, double dt, int nsteps, void* u,
                           const void* fx, unsigned* status, cudaStream_t st, int cluster, int stages_per_exchange,
                           int threads_per_cta);
// FP64 2D whole job in one cooperative launch (pass_resident2d.cu): whether it is the choice for the problem, given
// the room for packets; and the launch (packets: 256-byte aligned, zeroed by the call)
bool resident2d_wins(const frkc2_problem& p, int s, int nsteps, size_t packet_bytes);
cudaError_t launch_resident2d(const frkc2_problem& p, const frkc2_plan_s& plan, double dt, int nsteps, void* u, const void* fx,
                              const void* fy, void* packets, size_t packet_bytes, unsigned* status, long long wait_limit,
                              int fault_inject, cudaStream_t st);
// A cooperative launch that the context cannot hold at once (it may have fewer SMs than the device): nothing has run,
// and the caller takes the form of a launch a stage.
inline bool coop_refused(cudaError_t e) {
  const bool refused = e == cudaErrorCooperativeLaunchTooLarge || e == cudaErrorNotSupported || e == cudaErrorLaunchOutOfResources;
  if (refused) (void)cudaGetLastError();
  return refused;
}
// the same for the Brusselator in FP64 (bruss_resident2d.cu; refused: the persistent kernel)
bool bruss_resident_wins(const frkc2_bruss_problem& p, int s, int nsteps, size_t packet_bytes);
cudaError_t launch_bruss_resident(const frkc2_bruss_problem& p, const frkc2_plan_s& plan, double dt, int nsteps, double* v, double* w,
                                  void* packets, size_t packet_bytes, unsigned* status, long long wait_limit, int fault_inject,
                                  cudaStream_t st);
int stream3d_chunks(long long blocks, int nz, long long slots);
cudaError_t launch_pass_stream3d_f32(const frkc2_problem& p, const PassArgs& a, cudaStream_t st);
cudaError_t launch_pass_stream3d(const frkc2_problem& p, const PassArgs& a, cudaStream_t st);
// faces in padded rows (a.fx, a.fy of pitch fpitch), the pair state between passes as four planes of `plane` floats in
// rows of `pitch` (both pitches and the plane multiples of 4)
cudaError_t launch_pass_tb2d_df(const frkc2_problem& p, const PassArgs& a, int fpitch, int pitch, size_t plane, cudaStream_t st,
                                bool overlap_previous);
cudaError_t launch_pass_stream2d_df(const frkc2_problem& p, const PassArgs& a, const void* fen, cudaStream_t st);
cudaError_t launch_pass_paired2d(const frkc2_problem& p, const PassArgs& a, const void* fen, cudaStream_t st);
bool tb2d_supported(const frkc2_problem& p, int k);
size_t generic_smem_bytes(const frkc2_problem& p, const PassArgs& a);
void default_tiles(const frkc2_problem& p, int k, int* tx, int* ty, int* tz);

// One streamed 2D adjoint stage (fixed conductivity).
struct AdjStreamArgs {
  int nx, ny;
  const void* fen;    // face pairs
  const void* W;      // stage state W^l
  int w_complex;      // 0: real array (imaginary part 0), 1: interleaved (U, V)
  const void* L_in;   // lam^{l+1}
  int l_complex;      // 0: real array, 1: interleaved, 2: real part of an interleaved array
  void* L_out;        // lam^l, interleaved
  double* dk;         // dJ/dkappa accumulator or nullptr
  double ca, cb;      // dt a_l / dx^2
};
cudaError_t launch_adj_stream2d(const frkc2_problem& p, const AdjStreamArgs& a, cudaStream_t st);

// Temporally blocked FP32 adjoint (2D fixed conductivity): one pass of nst <= k stages.
struct AdjTbPass {
  int nst;
  // tape pass: forward stages from W^{l0}; out[j] receives W^{l0+1+j} (interleaved), the last
  // as a real array when last_real (the step output)
  const void* in;
  int in_complex;
  void* out[16];
  int last_real;
  // reverse pass: stage j is the j-th from the end; W[j] its tape entry (real when !w_complex)
  const void* W[16];
  int w_complex[16];
  const void* L_in;
  int l_mode;  // 0: real array, 1: interleaved, 2: real part of an interleaved array
  void* L_out;
  double* dk;
  double ca[16], cb[16];  // dt a_l / dx^2 of stage j
};
bool adj_tb2d_supported(const frkc2_problem& p, int k);
int adj_tb2d_k(const frkc2_problem& p, int s, bool rev);  // stages of a tape or reverse pass
cudaError_t launch_tape_tb2d(const frkc2_problem& p, int k, const AdjTbPass& t, const void* fx, const void* fy,
                             unsigned* status, cudaStream_t st);
cudaError_t launch_adjrev_tb2d(const frkc2_problem& p, int k, const AdjTbPass& t, const void* fx, const void* fy,
                               unsigned* status, cudaStream_t st);

// Temporally blocked Brusselator (FP32, bruss_tb2d.cu): the shape for a grid and plan (k = 0: not
// available), and the steps.
struct BrussTb {
  int cells;  // cells of a thread along each axis: 2 or 4 (regions of 32 x 32 or 64 x 64)
  int k;      // most stages per pass
};
BrussTb bruss_tb2d_shape(int nx, int ny, int s);
cudaError_t launch_bruss_tb2d(const frkc2_bruss_problem& p, const frkc2_plan_s& plan, double dt, int nsteps, BrussTb shape,
                              float* v, float* w, void* const P[2][4], unsigned* status, cudaStream_t st);

void count_launch(int n = 1);

// SM count and resident CTAs per SM of a kernel (at least 1).  Launchers keep the result in a
// function-local static, initialised once and thread-safely on the first call -- which must
// not be inside a stream capture; the library assumes one GPU model per process.
struct Residency {
  cudaError_t err;
  int sms;
  int per_sm;
};
template <class K>
Residency query_residency(K kern, int threads, size_t smem) {
  Residency r{cudaSuccess, 0, 0};
  int dev = 0;
  r.err = cudaGetDevice(&dev);
  if (r.err == cudaSuccess) r.err = cudaDeviceGetAttribute(&r.sms, cudaDevAttrMultiProcessorCount, dev);
  if (r.err == cudaSuccess) r.err = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&r.per_sm, kern, threads, smem);
  if (r.per_sm < 1) r.per_sm = 1;
  return r;
}

// SMs for the models of a pass's time: the device's, or 152 where it cannot be asked.
inline int model_sms() {
  static const int sms = [] {
    int dev = 0, n = 152;
    if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
      n = 152;
    return n;
  }();
  return sms;
}

// Dynamic shared memory that spreads a launch of `ctas` CTAs over the SMs: where they fit in one wave, as
// much as leaves room for just ceil(ctas / sms) of them per SM.  CTAs of a dependent launch that starts
// early (programmatic stream serialization) are otherwise packed onto the SMs that empty first: a pass of
// 144 CTAs of the FP32 Brusselator on 152 SMs took 9.5 us, and 4.3 us with one CTA per SM.  The kernel's
// MaxDynamicSharedMemorySize must be SPREAD_SMEM.
constexpr int SPREAD_SMEM = 226 * 1024;
inline size_t spread_smem(size_t need, long long ctas, int sms, int per_sm) {
  const long long want = (ctas + sms - 1) / sms;  // CTAs per SM
  if (want >= per_sm) return need;
  const size_t room = size_t(SPREAD_SMEM) / size_t(want);  // want CTAs fit (each with its 1 KB), want + 1 do not
  return std::max(need, want == 1 ? room : (room - 1024) / 1024 * 1024);
}

// A launch of persistent CTAs over `work` CTAs' worth of warp rows: the same number r of CTAs on every SM,
// r the fewest that give every warp at most one row (at most per_sm), spread as above.  (256^2 FP64, a
// stage: 5.9 us with 288 CTAs as they fell, 4.7 with 304 spread; 100^2 4.5 -> 3.05.)
struct SpreadGrid {
  unsigned grid;
  size_t smem;
};
inline SpreadGrid spread_grid(long long work, int sms, int per_sm) {
  const long long r = std::max<long long>(1, std::min<long long>(per_sm, (work + sms - 1) / sms));
  return {unsigned(r * sms), spread_smem(0, r * sms, sms, per_sm)};
}
// A kernel's MaxDynamicSharedMemorySize belongs to the device that is current when it is set: one of these per kernel
// sets it once on each device that launches the kernel (from the 65th on at every launch).
class SmemLimit {
  std::atomic<unsigned long long> done_{0};

 public:
  template <class K>
  cudaError_t raise(K kern, size_t bytes) {
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    const unsigned long long bit = dev < 64 ? 1ull << dev : 0ull;
    if (done_.load(std::memory_order_relaxed) & bit) return cudaSuccess;
    e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, int(bytes));
    if (e == cudaSuccess) done_.fetch_or(bit, std::memory_order_relaxed);
    return e;
  }
};

// query_residency for a kernel launched with such padding: `fixed` bytes of static shared memory.  `own`: the kernel's.
struct SpreadKernel {
  SmemLimit smem;
  std::once_flag once;
  Residency res{cudaSuccess, 0, 0};
};
template <class K>
Residency spread_residency(SpreadKernel& own, K kern, int threads, size_t smem, size_t fixed) {
  const cudaError_t e = own.smem.raise(kern, SPREAD_SMEM - fixed);
  std::call_once(own.once, [&] { own.res = query_residency(kern, threads, smem); });
  Residency r = own.res;
  if (e != cudaSuccess) r.err = e;
  return r;
}

}  // namespace frkc2
