// Division by a divisor that the host knows before the launch, as a multiplication (T. Granlund and P. L. Montgomery, "Division
// by Invariant Integers using Multiplication", 1994).  Plain C++ as well: the host's half of the kernels and the tests use it.
#pragma once
#include <stdint.h>

// n / d for 0 <= n < 2^31 and 1 <= d <= 2^31: for d > 1, s = ceil(log2 d), m = floor(2^(31 + s) / d) + 1 fits 32 bits and exceeds
// 2^(31 + s) / d by at most 1 <= 2^s / d, so that n * m / 2^(31 + s) stays below the next integer.  (An integer division costs a
// lone warp 100 - 200 cycles and 20 - 30 instructions, and the first copy of a launch used to wait for five of them.)
struct Div {
  unsigned m;               // 0: d = 1
  int s;                    // s - 1 above
};
static inline Div make_div(long long d) {
  if (d <= 1) return Div{0u, 0};
  int s = 1;
  while ((1LL << s) < d) ++s;
  return Div{(unsigned)((1ull << (31 + s)) / (unsigned long long)d + 1), s - 1};
}
#ifdef __CUDACC__
__host__ __device__ __forceinline__
#else
static inline
#endif
int div_by(int n, Div d) {
#ifdef __CUDA_ARCH__
  const unsigned high = __umulhi((unsigned)n, d.m);
#else
  const unsigned high = (unsigned)(((uint64_t)(unsigned)n * d.m) >> 32);
#endif
  return d.m ? (int)(high >> d.s) : n;
}
