// Batcher's odd-even merge sort as a compile-time network: every index is a template constant, so the
// array stays in registers.  N a power of two; LIMIT < N prunes the network to its first LIMIT inputs
// (valid where the inputs from LIMIT on would sit last, since a compare-exchange with such an input
// changes nothing).  OP::ce(a, b) leaves what goes first in a; DescF / DescU sort in descending order.
#pragma once
#include <stdint.h>

struct DescF {
  static __device__ __forceinline__ void ce(float& a, float& b) { const float hi = fmaxf(a, b), lo = fminf(a, b); a = hi; b = lo; }
};
struct DescU {
  static __device__ __forceinline__ void ce(uint32_t& a, uint32_t& b) { const uint32_t hi = max(a, b), lo = min(a, b); a = hi; b = lo; }
};
template <int LO, int N, int R, class OP, int LIMIT> struct OEMerge {
  template <class T> static __device__ __forceinline__ void run(T* x) {
    constexpr int M = R * 2;
    if constexpr (M < N) {
      OEMerge<LO, N, M, OP, LIMIT>::run(x);
      OEMerge<LO + R, N, M, OP, LIMIT>::run(x);
#pragma unroll
      for (int i = LO + R; i + R < LO + N; i += M)
        if (i + R < LIMIT) OP::ce(x[i], x[i + R]);
    } else {
      if constexpr (LO + R < LIMIT) OP::ce(x[LO], x[LO + R]);
    }
  }
};
template <int LO, int N, class OP, int LIMIT> struct OESort {
  template <class T> static __device__ __forceinline__ void run(T* x) {
    if constexpr (N > 1 && LO < LIMIT) {
      constexpr int M = N / 2;
      OESort<LO, M, OP, LIMIT>::run(x);
      OESort<LO + M, M, OP, LIMIT>::run(x);
      OEMerge<LO, N, 1, OP, LIMIT>::run(x);
    }
  }
};
