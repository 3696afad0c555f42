// dw_from_scaled (dw.cuh) on values of which the scale leaves 2^-60 to 2^-126, on the host.
#include <cmath>
#include <cstdio>
#include <cstring>
#include <random>

static inline long long __double_as_longlong(double x) { long long r; std::memcpy(&r, &x, 8); return r; }
static inline double __longlong_as_double(long long x) { double r; std::memcpy(&r, &x, 8); return r; }
static inline int __float_as_int(float x) { int r; std::memcpy(&r, &x, 4); return r; }
static inline float __int_as_float(int x) { float r; std::memcpy(&r, &x, 4); return r; }
static inline float __uint2float_rn(unsigned x) { return (float)x; }
static inline float __int2float_rn(int x) { return (float)x; }
static inline float __double2float_rn(double x) { return (float)x; }
static inline int __clzll(long long x) { return __builtin_clzll((unsigned long long)x); }
static inline float __shfl_xor_sync(unsigned, float v, int) { return v; }
static inline int max(int a, int b) { return a > b ? a : b; }
static inline int min(int a, int b) { return a < b ? a : b; }
using std::ldexp;
#include "dw.cuh"

int main() {
  std::mt19937_64 g(11);
  std::uniform_real_distribution<double> u(0.0, 1.0);
  long bad = 0;
  for (int t = 0; t < 1000000; ++t) {
    const int e = (int)(u(g) * 1600) - 800;
    double y = std::ldexp(1.0 + u(g), -60 - (int)(u(g) * 67));  // from 2^-126 on
    if (t & 1) y = -y;
    const vp::dw v = vp::dw_from_scaled(std::ldexp(y, e), e);
    const float hi = (float)y, lo = (float)(y - (double)hi);
    if (v.hi != hi || (std::fabs(lo) >= 0x1p-126f ? v.lo != lo : std::fabs(v.lo) > 0x1p-125f)) ++bad;
  }
  std::printf("%ld\n", bad);
  return 0;
}
