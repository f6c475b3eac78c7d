// Operations on the bit patterns of doubles, on the integer pipes: FP64 runs at 2 lanes per SM and clock
// on this part. Written on the halves of the pattern: on the whole pattern they are recognised as
// negation and magnitude of a double, which take an addition each on the FP64 pipe.
#pragma once

namespace qcad {

__device__ __forceinline__ unsigned long long abs_bits(double a) {
  return ((unsigned long long)((unsigned)__double2hiint(a) & 0x7fffffffu) << 32) | (unsigned)__double2loint(a);
}
__device__ __forceinline__ double neg_bits(double a) {
  return __hiloint2double(__double2hiint(a) ^ (int)0x80000000u, __double2loint(a));
}
__device__ __forceinline__ bool nonzero_bits(double a) {
  return (((unsigned)__double2hiint(a) << 1) | (unsigned)__double2loint(a)) != 0u;
}
// The key of qcad_internal.cuh's double_key: orders like the doubles.
__device__ __forceinline__ unsigned long long double_key(double a) {
  const int hi = __double2hiint(a), s = hi >> 31;
  return ((unsigned long long)(unsigned)(hi ^ (s | (int)0x80000000u)) << 32) | (unsigned)(__double2loint(a) ^ s);
}
// A double rounded to float (to nearest): the conversion instruction runs on the FP64 pipe.
__device__ __forceinline__ float d2f_bits(double a) {
  const unsigned hi = (unsigned)__double2hiint(a);
  const unsigned e = (hi >> 20) & 0x7FFu;
  if (e < 872u) return __uint_as_float(hi & 0x80000000u);  // below half the smallest float
  if (e < 897u || e > 1149u) return __double2float_rn(a);
  const unsigned long long m = abs_bits(a) - (896ull << 52);
  return __uint_as_float((unsigned)((m + 0x0FFFFFFFull + ((m >> 29) & 1)) >> 29) | (hi & 0x80000000u));
}
// 4 a, by the exponent where a and 4 a are normal numbers.
__device__ __forceinline__ double times4(double a) {
  const int hi = __double2hiint(a);
  const unsigned e = ((unsigned)hi >> 20) & 0x7FFu;
  if (e - 1u < 0x7FCu) return __hiloint2double(hi + (2 << 20), __double2loint(a));
  if (nonzero_bits(a)) {
    asm volatile("");  // keeps the product inside the branch
    a *= 4.0;
  }
  return a;
}

}  // namespace qcad
