// The scalar pieces of the factorisation kernels (csrc/h2_scalar.cuh) compiled
// for the host: the device intrinsics they use are restated here, the FP32
// approximations (rsqrtf, __fdividef) with an error of `seed_ulps` units in the
// last place, so that a test can run them over the range the device allows.
#include <cuda_runtime.h>
#include <math.h>
#include <string.h>

#include <algorithm>

namespace {
int seed_ulps = 0;

template <class To, class From>
To bits(From v) {
  To r;
  memcpy(&r, &v, sizeof r);
  return r;
}
float off(double v) {
  float f = (float)v;
  for (int i = 0; i < abs(seed_ulps); ++i) f = nextafterf(f, seed_ulps > 0 ? INFINITY : -INFINITY);
  return f;
}
int __double2hiint(double v) { return (int)(bits<unsigned long long>(v) >> 32); }
int __double2loint(double v) { return (int)bits<unsigned long long>(v); }
double __hiloint2double(int hi, int lo) {
  return bits<double>((unsigned long long)(unsigned)hi << 32 | (unsigned)lo);
}
float __uint_as_float(unsigned u) { return bits<float>(u); }
unsigned __float_as_uint(float f) { return bits<unsigned>(f); }
float rsqrtf(float x) { return off(1.0 / sqrt((double)x)); }
double rsqrt(double x) { return 1.0 / sqrt(x); }
float __fdividef(float a, float b) { return off((double)a / (double)b); }
double __drcp_rn(double v) { return 1.0 / v; }
using std::max;
using std::min;
}  // namespace

#include "h2_scalar.cuh"

extern "C" {
void set_seed_ulps(int u) { seed_ulps = u; }

// Both lanes of a pair: columns of squared norms na, nb and dot product g
// (as the sum of the two lanes' parts); t[0], t[1] their rotations.
void pair_tan(double na, double nb, float g, float* t) {
  const float d = h2::f32_of_normal(nb - na);
  t[0] = h2::jacobi_tan(g, d, h2::jacobi_threshold(na, nb));
  t[1] = h2::jacobi_tan(g, d, h2::jacobi_threshold(nb, na));
}
float threshold(double na, double nb) { return h2::jacobi_threshold(na, nb); }

void reciprocals(const double* v, int n, double* rsq, double* rec) {
  for (int i = 0; i < n; ++i) {
    rsq[i] = h2::rsqrt_pos(v[i]);
    rec[i] = h2::recip_pos(v[i]);
  }
}
// q = 1 + t^2 and 1 / sqrt(q) of a rotation
void cosines(const float* t, int n, double* q, double* c) {
  for (int i = 0; i < n; ++i) {
    q[i] = fma((double)t[i], (double)t[i], 1.0);
    c[i] = h2::jacobi_cos(q[i], t[i]);
  }
}
}
