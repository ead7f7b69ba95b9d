// The conversions of expansion.cuh between FP64 and sums of FP32 values, on the
// host: widened(x) is x, from_double(x) holds 48 bits of x, and to_double(h + l)
// is the FP64 sum rounded to nearest, powers of two with an l of the other sign
// among them (the last place below a power of two is half as large).  Prints the
// number of violations of each, exits non-zero if there are any.
#include <cmath>
#include <cstdint>
#include <cstdio>
#include <cstring>
#include <cuda_runtime.h>

template <class A, class B>
static A bits_as(B b) {
  A a;
  static_assert(sizeof(a) == sizeof(b), "");
  std::memcpy(&a, &b, sizeof(a));
  return a;
}
static inline float __fadd_rn(float a, float b) { return a + b; }
static inline float __fsub_rn(float a, float b) { return a - b; }
static inline float __fmul_rn(float a, float b) { return a * b; }
static inline float __fmaf_rn(float a, float b, float c) { return std::fma(a, b, c); }
static inline unsigned __float_as_uint(float x) { return bits_as<unsigned>(x); }
static inline float __uint_as_float(unsigned x) { return bits_as<float>(x); }
static inline int __float2int_rn(float x) { return (int)std::nearbyint(x); }
static inline float __int2float_rn(int x) { return (float)x; }
static inline int __double2hiint(double x) { return (int)(bits_as<std::uint64_t>(x) >> 32); }
static inline int __double2loint(double x) { return (int)(bits_as<std::uint64_t>(x) & 0xffffffffu); }
static inline double __hiloint2double(int hi, int lo) {
  return bits_as<double>(((std::uint64_t)(unsigned)hi << 32) | (unsigned)lo);
}
static inline double __longlong_as_double(long long x) { return bits_as<double>(x); }
using std::fma;
#include "expansion.cuh"
using namespace flame;

static std::uint64_t state = 88172645463325252ull;
static std::uint64_t random64() {
  state ^= state << 13;
  state ^= state >> 7;
  return state ^= state << 17;
}
static double uniform() { return (double)(random64() >> 11) * 0x1p-53; }

int main() {
  long bad_widened = 0, bad_from = 0, bad_to = 0, bad_to3 = 0, n = 0;
  for (int i = 0; i < 2000000; ++i) {
    const int e = (int)(random64() % 250) - 124;
    const double sign = random64() & 1 ? -1.0 : 1.0, x = sign * std::ldexp(1.0 + uniform(), e);
    float h = (float)x;
    if (!std::isfinite(h)) continue;
    if (i % 4 == 0) h = (float)(sign * std::ldexp(1.0, e));
    if (widened(h) != (double)h) ++bad_widened;
    const F2 f = from_double(x);
    if (e > -74 && e < 126 && std::fabs(((double)f.h - x) + (double)f.l) > std::fabs(x) * 0x1p-48) ++bad_from;
    // l up to half a unit of h's last place, now and then a few bits that end in a tie
    const double half = std::ldexp(1.0, e - 24);
    float l = (float)((2.0 * uniform() - 1.0) * half);
    if (i % 3 == 0) l = (float)std::ldexp((double)((int)(random64() % 64) - 32), e - 54);
    if (i % 97 == 0) l = (float)(-sign * half);
    // what the sum gives normalised
    const float s = h + l;
    const F2 a{s, (h - s) + l};
    if ((double)a.h + (double)a.l != (double)h + (double)l) continue;  // l below the denormal numbers
    if (to_double(a) != (double)a.h + (double)a.l) ++bad_to;
    const F3 t{a.h, a.l, 0.f};
    if (to_double(t) != (double)a.h + (double)a.l) ++bad_to3;
    ++n;
  }
  if (to_double(F2{1.f, -0x1p-53f}) != 1.0 - 0x1p-53) ++bad_to;
  if (to_double(F2{-1.f, 0x1p-53f}) != 0x1p-53 - 1.0) ++bad_to;
  std::printf("cases %ld widened %ld from_double %ld to_double %ld %ld\n", n, bad_widened, bad_from, bad_to, bad_to3);
  return bad_widened + bad_from + bad_to + bad_to3 != 0;
}
