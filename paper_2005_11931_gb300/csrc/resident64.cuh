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
// rims: [2][CTA][2][kR64Rows] first and last own column, [2][CTA][2][32] first and last own row; the word of
// expired waits (PollLimit) in the last 128 bytes
constexpr size_t kR64RimBytes = (size_t)2 * kResMaxCtas * 2 * (kR64Rows + 32) * sizeof(ulonglong2) + 128;
inline PollLimit r64_limit(void* rims, bool hold) {
  return PollLimit{hold ? kPollHookNs : kPollNs, (int*)((char*)rims + kR64RimBytes - 128)};
}
inline int64_t r64_strips(int64_t nx) { return (nx - 2 + kR64Out - 1) / kR64Out; }

// A double travels as two 64-bit words, each half of it with the tag in the upper 32 bits (an aligned 8-byte
// element of a vector access is read and written whole, a 32-bit one would be on its own).
__device__ __forceinline__ void put64(ulonglong2* d, const double x, const uint32_t tag) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(x), t = (unsigned long long)tag << 32;
  asm volatile("st.volatile.global.v2.b64 [%0], {%1, %2};" ::"l"(d), "l"(t | (uint32_t)b), "l"(t | b >> 32) : "memory");
}
__device__ __forceinline__ ulonglong2 try64(const ulonglong2* d) {
  ulonglong2 x;
  asm volatile("ld.volatile.global.v2.b64 {%0, %1}, [%2];" : "=l"(x.x), "=l"(x.y) : "l"(d) : "memory");
  return x;
}
__device__ __forceinline__ bool has_tag(const ulonglong2& x, const uint32_t tag) {
  return (uint32_t)(x.x >> 32) == tag && (uint32_t)(x.y >> 32) == tag;
}
// the value of x, read again until both its halves carry the tag (bounded)
__device__ __forceinline__ double get64(ulonglong2 x, const ulonglong2* d, const uint32_t tag, const PollLimit& w,
                                        bool& dead) {
  if (!has_tag(x, tag) && !dead) {
    const uint64_t t0 = global_ns();
    dead = true;
    for (int it = 0; it < kPollCap; ++it) {
      x = try64(d);
      if (has_tag(x, tag)) {
        dead = false;
        break;
      }
      if ((it & 63) == 63 && poll_over(w, t0)) break;
    }
  }
  if (dead) return __longlong_as_double(0x7ff8000000000000ll);  // a wait ran out: nothing that follows is valid
  return __longlong_as_double((long long)(x.y << 32 | (uint32_t)x.x));
}

}  // namespace dev
}  // namespace tsu
