// ||v|| of value rows (App. A.1.3): what the kernel of its own and the scoring kernel's spare CTAs share.
#pragma once

#include "kvc_internal.cuh"

namespace kvc {

// A row is kLpr = row bytes / 16 lanes wide (16 for the 256-byte rows of a bf16 head of 128), so a warp carries 32 / kLpr
// rows at a time and every lane loads; each lane has kNormRows such rows in flight (one 16-byte load each) before it
// adds anything, and a warp's rows are consecutive.
constexpr int kNormRows = 8;
template <int kLpr>
constexpr int kNormBlock = kNormRows * (32 / kLpr);            // rows of a warp

// Two fp32 values in one register pair.
__device__ __forceinline__ unsigned long long norm_pair(uint32_t a, uint32_t b) {
  unsigned long long r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "r"(a), "r"(b));
  return r;
}
__device__ __forceinline__ unsigned long long norm_square(unsigned long long x, unsigned long long acc) {
  unsigned long long d;
  asm("fma.rn.f32x2 %0, %1, %1, %2;" : "=l"(d) : "l"(x), "l"(acc));
  return d;
}

// The norms of the warp's kNormBlock rows from `first` on, whose pieces are in w, to out[first ..].  The squares are added in one
// order everywhere: a lane's elements in ascending order, then the lanes by halving distances.  Instructions count here (the
// scoring kernel's spare CTAs are bound by them as much as by HBM): two rows' squares go into one packed multiply-add, and at every
// distance a lane hands half of its rows on and keeps the other half (8 shuffles for 8 rows instead of 32; both sides of an
// exchange would have come to the same sum).
template <typename T, int kLpr>
__device__ __forceinline__ void norm_store(const uint4 (&w)[kNormRows], float* out, long long first, long long N) {
  constexpr int kGroups = 32 / kLpr, kPer = kLpr / kNormRows;   // kPer lanes hold a row's norm in the end
  static_assert(kNormRows == 8 && kPer >= 1, "three exchanges leave one row");
  const int lane = threadIdx.x & 31, sub = lane & (kLpr - 1), grp = lane / kLpr;
  float v[kNormRows];
#pragma unroll
  for (int u = 0; u < kNormRows; u += 2) {
    const uint32_t a[4] = {w[u].x, w[u].y, w[u].z, w[u].w}, b[4] = {w[u + 1].x, w[u + 1].y, w[u + 1].z, w[u + 1].w};
    unsigned long long acc = 0ull;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      if (sizeof(T) == 2) {
        // a bf16 is the upper half of the fp32 with the same value
        acc = norm_square(norm_pair(a[i] << 16, b[i] << 16), acc);
        acc = norm_square(norm_pair(a[i] & 0xffff0000u, b[i] & 0xffff0000u), acc);
      } else {
        acc = norm_square(norm_pair(a[i], b[i]), acc);
      }
    }
    asm("mov.b64 {%0, %1}, %2;" : "=f"(v[u]), "=f"(v[u + 1]) : "l"(acc));
  }
  int o = kLpr / 2;
#pragma unroll
  for (int rows = kNormRows / 2; rows > 0; rows >>= 1, o >>= 1) {
    const bool upper = (sub & o) != 0;                           // keeps the upper half of the rows
#pragma unroll
    for (int j = 0; j < rows; ++j) {
      const float sent = __shfl_xor_sync(0xffffffffu, upper ? v[j] : v[j + rows], o);
      v[j] = (upper ? v[j + rows] : v[j]) + sent;
    }
  }
#pragma unroll
  for (; o > 0; o >>= 1) v[0] += __shfl_xor_sync(0xffffffffu, v[0], o);
  const long long c = first + grp + sub / kPer * kGroups;
  if (sub % kPer == 0 && c < N) out[c] = sqrtf(v[0]);
}

}  // namespace kvc
