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

#include "dfloat.cuh"
#include "fpbits.cuh"
#include "launch_rules.h"

using qcad::dfl;
// One step of a double-float sum, product and sum renormalized.
static dfl step(dfl s, dfl a, dfl b) {
  const dfl p = qcad::dfl_prod(a, b);
  return s + qcad::dfl_quick(p.h, p.l);
}

extern "C" {
void h_times4(int n, const double* a, double* out) {
  for (int i = 0; i < n; ++i) out[i] = qcad::times4(a[i]);
}
void h_d2f(int n, const double* a, float* out) {
  for (int i = 0; i < n; ++i) out[i] = qcad::d2f_bits(a[i]);
}
void h_split(int n, const double* a, double* out) {
  for (int i = 0; i < n; ++i) {
    const dfl d = qcad::dfl_from_bits(a[i]);
    out[i] = (double)d.h + (double)d.l;
  }
}
// Sums of 27 products c x (values already double-float exact): by groups of three as the stencil's rows,
// and renormalized at every step.
void h_rows(int n, const double* c, const double* x, double* grouped, double* stepped) {
  for (int i = 0; i < n; ++i) {
    dfl a(0), b(0), cd[27], xd[27];
    for (int q = 0; q < 27; ++q) {
      cd[q] = qcad::dfl_from_bits(c[27 * i + q]);
      xd[q] = qcad::dfl_from_bits(x[27 * i + q]);
    }
    for (int q = 0; q < 27; q += 3) qcad::dfl_mac3(a, cd[q], xd[q], cd[q + 1], xd[q + 1], cd[q + 2], xd[q + 2]);
    for (int q = 0; q < 27; ++q) b = step(b, cd[q], xd[q]);
    grouped[i] = qcad::dfl_to_double(a);
    stepped[i] = qcad::dfl_to_double(b);
  }
}
int h_gram32_flush(int groups) { return qcad::gram32_flush_tiles(groups); }
// once_per_device over a list of devices whose set() fails for the first `fails` calls: the calls of
// set() per launch.
void h_once(int n, const int* devices, int fails, int* calls) {
  qcad::PerDevice state;
  for (int i = 0; i < n; ++i) {
    calls[i] = 0;
    qcad::once_per_device(state, devices[i], [&] {
      ++calls[i];
      return fails-- <= 0;
    });
  }
}
int h_slab_layers(int nx, int ny, int nz) { return qcad::hm_slab_layers(nx, ny, nz); }
// The slabs of an assembly as rows of e0, e1, p0, p1; returns their number (at most max).
int h_slabs(int nz, int slab, int max, int* out) {
  int n = 0;
  for (int p0 = 0; p0 <= nz && n < max; ++n) {
    const qcad::HmSlab b = qcad::hm_next_slab(p0, nz, slab);
    out[4 * n] = b.e0, out[4 * n + 1] = b.e1, out[4 * n + 2] = b.p0, out[4 * n + 3] = b.p1;
    p0 = b.p1;
  }
  return n;
}
}
