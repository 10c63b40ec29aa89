// What the resident 2D kernels share: the sides of a unit and the packets in which CTAs pass each other its edges.
// A packet is two 64-bit words, each half a value and the stage number; 64-bit relaxed accesses are single-copy
// atomic, so a reader that sees the number in both words has the value.
#pragma once
#include <cuda_runtime.h>

namespace frkc2 {
namespace {

enum { SIDE_N = 0, SIDE_S = 1, SIDE_E = 2, SIDE_W = 3 };  // the opposite side: side ^ 1
enum { EDGE_NONE = 0, EDGE_LOCAL = 1, EDGE_REMOTE = 2 };

__device__ __forceinline__ void put_packet(ulonglong2* p, double v, unsigned seq) {
  asm volatile(
      "{\n\t.reg .b64 a, b;\n\tmov.b64 a, {%1, %3};\n\tmov.b64 b, {%2, %3};\n\t"
      "st.relaxed.gpu.global.v2.b64 [%0], {a, b};\n\t}" ::"l"(p), "r"(__double2loint(v)), "r"(__double2hiint(v)), "r"(seq)
      : "memory");
}
__device__ __forceinline__ bool get_packet(const ulonglong2* p, double& v, unsigned seq) {
  unsigned lo, hi, s0, s1;
  asm volatile(
      "{\n\t.reg .b64 a, b;\n\tld.relaxed.gpu.global.v2.b64 {a, b}, [%4];\n\t"
      "mov.b64 {%0, %2}, a;\n\tmov.b64 {%1, %3}, b;\n\t}"
      : "=r"(lo), "=r"(hi), "=r"(s0), "=r"(s1)
      : "l"(p)
      : "memory");
  v = __hiloint2double(int(hi), int(lo));
  return s0 == seq && s1 == seq;
}

// v or -v, on the integer pipe (a negation outside an FP64 instruction would take an FP64 slot)
__device__ __forceinline__ double flip(double v, bool negate) {
  return __hiloint2double(__double2hiint(v) ^ (negate ? int(0x80000000u) : 0), __double2loint(v));
}

// Polls of a wait by default: 62 s (233 ns a poll, 64^2) to 120 s (447 ns, 200^2 Brusselator).  The CTAs of a launch may be
// placed one by one as a long launch on another stream leaves the SMs, and the first of them wait for the last: a batch of
// 512 FP64 problems takes 7 s, which 2^25 polls (8 s) hardly outlast.
constexpr long long RESIDENT_WAIT = 1ll << 28;

struct CoopDevice {
  int sms, coop;
};
// queried once, on the first (eager) call
inline CoopDevice coop_device() {
  static const CoopDevice d = [] {
    CoopDevice v{0, 0};
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&v.sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&v.coop, cudaDevAttrCooperativeLaunch, dev) != cudaSuccess)
      v.sms = v.coop = 0;
    return v;
  }();
  return d;
}

}  // namespace
}  // namespace frkc2
