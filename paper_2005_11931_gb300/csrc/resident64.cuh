// Shared by the FP64 passes that keep a grid on chip (k_step_res64.cu, k_adjoint_res64.cu): the tiling, and
// the values that travel between CTAs with the number of the step that wrote them.
#pragma once
#include "async_copy.cuh"
#include "tsu_internal.h"

namespace tsu {
namespace dev {

constexpr int kR64Warps = 8, kR64Threads = kR64Warps * 32;
constexpr int kR64Out = 30;    // own columns of a strip: 30 s + 1 .. 30 s + 30
constexpr int kR64Rows = 128;  // most rows of a tile
constexpr uint64_t kR64WaitNs = 10000000000ull;
// rims: [2][CTA][2][kR64Rows] first and last own column, [2][CTA][2][32] first and last own row
constexpr size_t kR64RimBytes = (size_t)2 * kResMaxCtas * 2 * (kR64Rows + 32) * sizeof(uint4);
inline int64_t r64_strips(int64_t nx) { return (nx - 2 + kR64Out - 1) / kR64Out; }

__device__ __forceinline__ void put64(uint4* d, const double x, const uint32_t tag) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(x);
  asm volatile("st.volatile.global.v4.u32 [%0], {%1, %2, %3, %2};" ::"l"(d), "r"((uint32_t)b), "r"(tag),
               "r"((uint32_t)(b >> 32))
               : "memory");
}
__device__ __forceinline__ uint4 try64(const uint4* d) {
  uint4 x;
  asm volatile("ld.volatile.global.v4.u32 {%0, %1, %2, %3}, [%4];"
               : "=r"(x.x), "=r"(x.y), "=r"(x.z), "=r"(x.w)
               : "l"(d)
               : "memory");
  return x;
}
// the value of x, read again until both its halves carry the tag (bounded)
__device__ __forceinline__ double get64(uint4 x, const uint4* d, const uint32_t tag, bool& dead) {
  if (!(x.y == tag && x.w == tag) && !dead) {
    const uint64_t t0 = global_ns();
    long long it = 0;
    for (; it < kSpinCap; ++it) {
      x = try64(d);
      if (x.y == tag && x.w == tag) break;
      if ((it & 63) == 63 && global_ns() - t0 > kR64WaitNs) it = kSpinCap;
    }
    dead = it >= kSpinCap;
  }
  if (dead) return __longlong_as_double(0x7ff8000000000000ll);  // a wait ran out: nothing that follows is valid
  return __longlong_as_double((long long)((unsigned long long)x.z << 32 | x.x));
}

}  // namespace dev
}  // namespace tsu
