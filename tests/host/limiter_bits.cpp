// limiter_bits.cpp -- the FP64 limiters of physics.cuh, which work on the bits, on the host against
// their plain branching forms, value for value; built with the undefined-behaviour checks on.
#include <cuda_runtime.h>
#include <float.h>
#include <math.h>
#include <stdio.h>
#include <string.h>

#define __noinline__ __attribute__((noinline))

// the device functions the header names, as far as the host needs them to compile
inline long long __double_as_longlong(double x) {
  long long b;
  memcpy(&b, &x, sizeof b);
  return b;
}
inline double __longlong_as_double(long long b) {
  double x;
  memcpy(&x, &b, sizeof x);
  return x;
}
float __fdividef(float, float);
float2 __fadd2_rn(float2, float2);
float2 __fmul2_rn(float2, float2);
float2 __ffma2_rn(float2, float2, float2);

#include "../../paper_1204_5849_gb300/csrc/physics.cuh"

static double plain_minmod(double a, double b) {
  if (a > 0.0 && b > 0.0) return a < b ? a : b;
  if (a < 0.0 && b < 0.0) return a > b ? a : b;
  return 0.0;
}

static double plain_half(int lim, double a, double b) {
  if (lim == 0) return 0.5 * plain_minmod(a, b);
  const double ab = a * b;
  return ab > 0.0 ? ab / (a + b) : 0.0;
}

static bool same(double a, double b) {
  return memcmp(&a, &b, sizeof a) == 0 || (a != a && b != b);
}

int main() {
  const double x[] = {0.0, -0.0, DBL_TRUE_MIN, -DBL_TRUE_MIN, 3e-310, -3e-310, DBL_MIN, -DBL_MIN, 1e-170, -1e-170,
                      0.25, -0.25, 1.0, -1.0, 1.0000000000000002, -3.5, 1e200, -1e200, DBL_MAX, -DBL_MAX, INFINITY,
                      -INFINITY, (double)NAN, -(double)NAN};
  int wrong = 0;
  for (double a : x) {
    if (mapgb::positive<double>(a) != (a > 0.0)) {
      printf("positive(%g)\n", a);
      ++wrong;
    }
    for (double b : x) {
      if (!same(mapgb::minmod<double>(a, b), plain_minmod(a, b)) ||
          !same(mapgb::half_limiter<double, 0>(a, b), plain_half(0, a, b)) ||
          !same(mapgb::half_limiter<double, 1>(a, b), plain_half(1, a, b)) ||
          mapgb::positive<double>(a * b) != (a * b > 0.0)) {
        printf("limiter(%g, %g)\n", a, b);
        ++wrong;
      }
    }
  }
  printf("%d wrong\n", wrong);
  return wrong != 0;
}
