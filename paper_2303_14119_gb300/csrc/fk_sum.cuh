// Sums of FP64 values at the memory's rate.  GB300 adds two FP64 values a cycle
// and SM: a plain sum of 67 M values takes its FP64 pipe 112 us, a read of
// them 79 us.  Here kGroup values of a thread are aligned to the largest
// exponent among them and added as 64-bit integers; one conversion and one
// FP64 multiply-add then take the group's sum into the total.
//
// Error: a value loses what lies kGuard bits and more below the last bit of
// the group's largest one (2^-58 of it), the group's sum is rounded once to FP64,
// and the total takes a kGroup-th of the roundings of a plain sum.
#pragma once

#include <cuda_runtime.h>

namespace fk {
namespace {

constexpr int kGroup = 16;  // values aligned together
constexpr int kGuard = 6;   // 53 + 6 bits and 16 values: below 2^63

// total + sum of the group's values
__device__ __forceinline__ double add_group(const double (&x)[kGroup], double total) {
  int top = 0, signs = 0, any = 0;
#pragma unroll
  for (int q = 0; q < kGroup; q++) {
    const int h = __double2hiint(x[q]);
    top = max(top, h & 0x7FFFFFFF);
    signs |= h;
    any |= h | __double2loint(x[q]);
  }
  if (any == 0) return total;
  const int E = top >> 20;  // the largest exponent field
  if (signs < 0 || E >= 2046 || E < 128) {
    // a negative value, an infinity or a NaN, or magnitudes whose alignment
    // would reach the subnormal range: plain additions
#pragma unroll
    for (int q = 0; q < kGroup; q++) total += x[q];
    return total;
  }
  long long acc = 0;
#pragma unroll
  for (int q = 0; q < kGroup; q++) {
    const int h = __double2hiint(x[q]);
    const unsigned long long m =
        ((unsigned long long)(unsigned)((h & 0xFFFFF) | 0x100000) << 32 |
         (unsigned)__double2loint(x[q])) << kGuard;
    acc += (long long)(m >> min(E - (h >> 20), 63));  // zeros and subnormals shift out
  }
  // units of 2^(E - 1075 - kGuard)
  const double unit = __hiloint2double((E - 52 - kGuard) << 20, 0);
  return fma((double)acc, unit, total);
}

}  // namespace
}  // namespace fk
