// The integer conversions of dw.cuh between FP64 and double words, on the host.
#include <cmath>
#include <cstdint>
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
  std::mt19937_64 g(7);
  std::uniform_real_distribution<double> u(0.0, 1.0);
  long bad_from = 0, bad_to = 0;
  for (int t = 0; t < 2000000; ++t) {
    const int e = (int)(u(g) * 1800) - 900;  // the scale (x stays finite)
    double y = std::ldexp(0.5 + u(g), (int)(u(g) * 100) - 70);  // scaled value
    if (t % 7 == 0) y = std::ldexp(1.0 + std::ldexp(1.0, -(int)(u(g) * 52)), (int)(u(g) * 20));
    if (t & 1) y = -y;
    const double x = std::ldexp(y, e);
    const vp::dw v = vp::dw_from_scaled(x, e);
    const float hi = (float)y, lo = (float)(y - (double)hi);
    // (a low part below 2^-126 may be flushed)
    if (std::fabs(x) > 1e-300 && (v.hi != hi || (v.lo != lo && std::fabs(lo) > 0x1p-125f))) ++bad_from;
    const float h = std::ldexp((float)(0.5 + u(g)), (int)(u(g) * 60) - 30) * (t & 2 ? -1.f : 1.f);
    float l = h * std::ldexp((float)(2 * u(g) - 1), -24 - (int)(u(g) * u(g) * 40));
    if (t % 13 == 0) l = 0.f;
    if (t % 17 == 0) l = h * 0x1p-25f * (t & 4 ? -1.f : 1.f);
    const int ee = (int)(u(g) * 400) - 200;
    if (vp::dw_to_scaled({h, l}, ee) != std::ldexp((double)h + (double)l, ee)) ++bad_to;
  }
  const double inf = HUGE_VAL;
  const bool edges = std::isnan(vp::dw_from_scaled(inf, 3).hi) && std::isnan(vp::dw_from_scaled(-inf, 3).hi) &&
                     std::isnan(vp::dw_from_scaled(std::nan(""), 0).hi) && vp::dw_from_scaled(0.0, 900).hi == 0.f &&
                     vp::dw_from_scaled(-0.0, -900).hi == 0.f && vp::dw_to_scaled({0.f, 0.f}, 5) == 0.0 &&
                     std::isnan(vp::dw_to_scaled({std::nanf(""), 0.f}, 1)) && vp::dw_to_scaled({1.f, 0.f}, 2000) == inf &&
                     vp::dw_to_scaled({1.f, 0.f}, -2000) == 0.0 && vp::dw_to_scaled({0x1p-140f, 0.f}, 0) == 0x1p-140;
  std::printf("%ld %ld %d\n", bad_from, bad_to, edges ? 1 : 0);
  return 0;
}
