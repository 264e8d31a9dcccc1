// The kernels' fixed-point reciprocal, exponential and cos/sin (csrc/tami_devmath.cuh) compiled for
// the host and compared with long double, at the places where they can go wrong: the ends of the
// binades and of the tables, arguments next to table points and quadrant boundaries, tiny and huge
// arguments, zeros, infinities and NaNs.  The hardware's reciprocal estimate is replaced by a
// rounded division that is off by RCP_OFF units in the last place.
#include <algorithm>
#include <cmath>
#include <cstdio>
#include <cstring>
#include <limits>
#include <random>
using std::max;
using std::min;
#define __device__
#define __forceinline__ inline
#define __noinline__
#define __align__(n) __attribute__((aligned(n)))
struct ulonglong2 { unsigned long long x, y; };
typedef unsigned long long u64;
template <class A, class B> static A bits_as(B b) { A a; std::memcpy(&a, &b, sizeof a); return a; }
static unsigned __umulhi(unsigned a, unsigned b) { return (unsigned)(((u64)a * b) >> 32); }
static float __uint_as_float(unsigned u) { return bits_as<float>(u); }
static unsigned __float_as_uint(float f) { return bits_as<unsigned>(f); }
static int __float_as_int(float f) { return bits_as<int>(f); }
static long long __double_as_longlong(double d) { return bits_as<long long>(d); }
static double __longlong_as_double(long long d) { return bits_as<double>(d); }
static int __double2hiint(double d) { return (int)(bits_as<u64>(d) >> 32); }
static int __double2loint(double d) { return (int)bits_as<u64>(d); }
static double __hiloint2double(int h, int l) { return bits_as<double>(((u64)(unsigned)h << 32) | (unsigned)l); }
static int __clz(int x) { return x ? __builtin_clz((unsigned)x) : 32; }
static int __clzll(long long x) { return x ? __builtin_clzll((u64)x) : 64; }
static unsigned __funnelshift_l(unsigned lo, unsigned hi, unsigned s) { return s ? (hi << s) | (lo >> (32 - s)) : hi; }
template <class T> static T __ldg(const T* p) { return *p; }
static double __dmul_rn(double a, double b) { return a * b; }
static double __dadd_rn(double a, double b) { return a + b; }
static double __ull2double_rn(u64 a) { return (double)a; }
static int RCP_OFF = 0;
static float host_rcp_estimate(float x) { return __uint_as_float(__float_as_uint((float)(1.0 / (double)x)) + (unsigned)RCP_OFF); }
using std::fabs; using std::fma; using std::fmaf; using std::fmax; using std::fmaxf; using std::fmod; using std::rint;
#include "devmath_host.h"

using namespace tami::dev;
typedef long double L;
static double ulp(double v) { return std::ldexp(1.0, std::ilogb(v) - 52); }
static int failures = 0;
static void check(bool ok, const char* what, double at, double got) {
  if (!ok && failures++ < 20) std::printf("%s at %a: %a\n", what, at, got);
}

static std::mt19937_64 R(7);
static double uniform(double a, double b) { return a + (b - a) * ((R() >> 11) * 0x1p-53); }

static void test_rcp() {
  const double inf = std::numeric_limits<double>::infinity();
  for (RCP_OFF = -1; RCP_OFF <= 1; ++RCP_OFF) {
    auto one = [](double d) {
      const double r = rcp(d);
      const L e = ((L)r * d - 1.0L) / d;                 // r - 1/d, the product exact to 2^-63
      check(std::fabs((double)(e / (L)ulp(r))) <= 0.502, "rcp", d, r);
    };
    for (int i = 0; i < 200000; ++i) {
      one(1.0 + i * 0x1p-52);
      one(2.0 - (i + 1) * 0x1p-53 * 2);
      one(std::ldexp(uniform(1, 2), (int)(R() % 2000) - 1000) * (i & 1 ? -1 : 1));
      one(1.0 + (i & 0x7FFFFF) * 0x1p-23 + (R() & 3) * 0x1p-52);   // next to the estimate's 24 bits
    }
    check(rcp(1.0) == 1.0 && rcp(-4.0) == -0.25 && rcp(0x1p-1022) == 0x1p1022, "rcp exact", 1.0, rcp(1.0));
    for (double d : {0.0, -0.0, 1e-310, inf, -inf, std::nan("")}) check(std::isnan(rcp(d)), "rcp odd", d, rcp(d));
    check(rcp(0x1.8p1022) == 0.0 && std::signbit(rcp(-0x1p1023)), "rcp of a huge value", 0x1.8p1022, rcp(0x1.8p1022));
  }
  RCP_OFF = 0;
}

static void test_exp() {
  const double inf = std::numeric_limits<double>::infinity(), step = std::log(2.0) / 1024;
  auto one = [](double t) {
    double em, unused;
    const double y = exp_neg<true>(t, em), y0 = exp_neg<false>(t, unused);
    check(__double_as_longlong(y) == __double_as_longlong(y0), "exp without e^t - 1", t, y0);
    if (t > -707.0) check(std::fabs((double)(((L)y - std::exp((L)t)) / (L)ulp(y))) <= 0.51, "exp", t, y);
    if (t < -1e-300) check(std::fabs((double)(((L)em - std::expm1((L)t)) / (L)ulp(em))) <= 0.75, "expm1", t, em);
  };
  for (int i = 0; i < 100000; ++i) {
    one(-uniform(0, 1)); one(-uniform(0, 50)); one(-uniform(0, 707)); one(-uniform(0, 4 * step));
    one(-std::pow(10.0, uniform(-299, 2.8)));
    one(-(i % 1030000 / 1.0) * step); one(-i * step * (1 + 0x1p-52)); one(-i * step * (1 - 0x1p-53));
  }
  double em;
  check(exp_neg<true>(0.0, em) == 1.0 && em == 0.0, "exp(0)", 0.0, em);
  check(exp_neg<true>(-1e-320, em) == 1.0 && em == -1e-320, "exp(subnormal)", -1e-320, em);
  for (double t : {-709.0, -745.2, -1023.9, -1024.0, -1e300, -inf})   // below the normal range: 0
    check(exp_neg<true>(t, em) == 0.0 && em == -1.0, "exp underflow", t, em);
  check(std::isnan(exp_neg<true>(std::nan(""), em)) && std::isnan(em), "exp(NaN)", 0.0, em);
}

static void test_trig() {
  const double inf = std::numeric_limits<double>::infinity();
  auto one = [](double k) {
    double s, c;
    cw_sincos(k, s, c);
    check(std::fabs((double)((L)c - std::cos((L)k))) <= 8e-17, "cos", k, c);
    check(std::fabs((double)((L)s - std::sin((L)k))) <= 8e-17, "sin", k, s);
    check(cw_cos(k) == c, "cos alone", k, c);
  };
  for (int i = 0; i < 100000; ++i) {
    one(uniform(-22, 22)); one(uniform(-31.9, 31.9)); one(std::pow(10.0, uniform(-300, 1.5)));
    const double a = (i % 20000 - 10000) * (M_PI / 1024);                 // table points and the middles between
    one(a); one(a * (1 + 0x1p-52)); one(a + uniform(-1e-9, 1e-9));
    const double kx = uniform(-22, 22), ky = uniform(-22, 22);
    double gx, gy;
    const double E = line_energy(kx, ky, 1.0, -0.3, -0.5);
    const L cx = std::cos((L)kx), cy = std::cos((L)ky);
    check(std::fabs((double)((L)E - (-0.5L + 2 * (cx + cy) + 4 * (L)-0.3 * cx * cy))) <= 1.5e-15, "line energy", kx, E);
    check(E == line_energy_grad(kx, ky, 1.0, -0.3, -0.5, gx, gy), "line energy with gradients", kx, E);
    check(std::fabs((double)((L)gx - (2 + 4 * (L)-0.3 * cy) * std::sin((L)kx))) <= 1e-15, "gradient", kx, gx);
  }
  double s, c;
  cw_sincos(0.0, s, c);
  check(s == 0.0 && c == 1.0, "sincos(0)", 0.0, s);
  for (double k : {32.0, -33.5, 100.0, 1e5}) {                             // the out-of-line reduction
    check(std::fabs(cw_cos(k) - std::cos(k)) <= 3e-16 + 1e-20 * k * k, "cos far", k, cw_cos(k));
    check(std::fabs(line_energy(k, 1.0, 1.0, 0.0, 0.0) - 2 * (std::cos(k) + std::cos(1.0))) <= 2e-15, "far line", k, 0.0);
  }
  for (double k : {inf, -inf, std::nan("")})
    check(std::isnan(cw_cos(k)) && std::isnan(line_energy(1.0, k, 1.0, 0.0, 0.0)), "not finite", k, cw_cos(k));
}

int main(int argc, char** argv) {
  const char* what = argc > 1 ? argv[1] : "";
  if (!std::strcmp(what, "rcp")) test_rcp();
  if (!std::strcmp(what, "exp")) test_exp();
  if (!std::strcmp(what, "trig")) test_trig();
  std::printf("%d failures\n", failures);
  return failures != 0;
}
