// C entry points to the device arithmetic headers, compiled for the host by
// tests/test_device_arithmetic.py with host definitions of the intrinsics they use (CPU only).
#include <cmath>
#include <cstdint>
#include <cstring>

#define __device__
#define __host__
#define __forceinline__ inline
template <class To, class From>
static To pattern(From v) {
  To r;
  static_assert(sizeof(To) == sizeof(From), "same size");
  std::memcpy(&r, &v, sizeof(r));
  return r;
}
static inline int __double2hiint(double a) { return (int)(pattern<uint64_t>(a) >> 32); }
static inline int __double2loint(double a) { return (int)(uint32_t)pattern<uint64_t>(a); }
static inline double __hiloint2double(int hi, int lo) {
  return pattern<double>(((uint64_t)(uint32_t)hi << 32) | (uint32_t)lo);
}
static inline long long __double_as_longlong(double a) { return pattern<long long>(a); }
static inline double __longlong_as_double(long long a) { return pattern<double>(a); }
static inline unsigned __float_as_uint(float a) { return pattern<unsigned>(a); }
static inline float __uint_as_float(unsigned a) { return pattern<float>(a); }
static inline float __double2float_rn(double a) { return (float)a; }

#include "fpbits.cuh"

extern "C" {
void h_times4(int n, const double* a, double* out) {
  for (int i = 0; i < n; ++i) out[i] = qcad::times4(a[i]);
}
void h_d2f(int n, const double* a, float* out) {
  for (int i = 0; i < n; ++i) out[i] = qcad::d2f_bits(a[i]);
}
}
