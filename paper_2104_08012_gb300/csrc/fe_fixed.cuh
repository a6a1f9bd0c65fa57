// FP64 values as integers of a common scale, for sums with small integer
// coefficients that are exact and cost two integer instructions per term instead
// of an operation of the FP64 pipe (2 per clock and SM).
#pragma once

#include <cuda_runtime.h>

namespace fe_fixed {

constexpr int kTop = 59;  // top bit of a value: |x| < 2^60 units

__device__ __forceinline__ double pow2(int e) {  // 2^e, -1022 <= e <= 1023
  return __hiloint2double((e + 1023) << 20, 0);
}

struct Pair32 {  // hi 2^30 + lo
  int hi, lo;
};
__device__ __forceinline__ Pair32 operator+(Pair32 a, Pair32 b) { return {a.hi + b.hi, a.lo + b.lo}; }

// A sum of integer coefficients times staged values, exact in 64 bits per word.
struct PairSum {
  long long hi = 0, lo = 0;
  // one 32 x 32 + 64 bit instruction per word (left to itself the compiler turns the small coefficients into sign
  // extensions, shifts and carried additions, three instructions each)
  static __device__ __forceinline__ void mad(long long& a, int k, int v) {
    asm("mad.wide.s32 %0, %1, %2, %0;" : "+l"(a) : "r"(v), "r"(k));
  }
  template <typename... A>
  __device__ __forceinline__ void add(int k, A... v) {  // sums of at most two staged values
    ((mad(hi, k, v.hi), mad(lo, k, v.lo)), ...);
  }
};

// x as hi 2^30 + lo in units of 2^(E - 1023 - kTop), E the largest biased exponent of a tile, both with the sign of x,
// what lies below a unit cut off.  A shift beyond 63 (zeros, far smaller values and, with e > E, values that are not
// finite) gives 0; needs E >= 64.
__device__ __forceinline__ Pair32 fixed_pair(double x, int E) {
  const unsigned int xh = (unsigned int)__double2hiint(x), xl = (unsigned int)__double2loint(x);
  const unsigned int r = min((unsigned int)(E - (int)((xh >> 20) & 0x7FFu)), 63u);
  const unsigned long long m = ((unsigned long long)((xh & 0xFFFFFu) | 0x100000u) << 32) | xl;
  const unsigned long long w = (m << (kTop - 52)) >> r;
  const int sg = 1 | ((int)xh >> 31);
  return {sg * (int)(w >> 30), sg * (int)((unsigned int)w & 0x3FFFFFFFu)};
}
}  // namespace fe_fixed
