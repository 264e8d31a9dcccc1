// The relative accuracy of the kernels' fixed-point sine next to its zeros, and of the line gradients
// that are proportional to it, against long double.
#define main fixed_math_main
#include "fixed_math_cases.cpp"
#undef main

// 6e-18 is trig_fixed's stated bound.  sin_near, within 3 pi/1024, rounds the distance from the zero (half
// an ulp of it, one of a sine in the binade below) and the sum (half an ulp); its series and the third
// part of pi add less than 0.02.
static void one(double k, double extra_ulp) {
  double s, c;
  cw_sincos(k, s, c);
  const L ref = std::sin((L)k), err = std::fabs((L)s - ref), u = ulp((double)ref);
  const L from_zero = std::fabs((L)k - (L)M_PIl * std::round((L)k / M_PIl));
  const L bound = from_zero < 0.0092L ? (1.52L + extra_ulp) * u : (0.5L + extra_ulp) * u + 6e-18L;
  check(err <= bound, "sin near a zero", k, s);
  check(std::fabs((double)((L)c - std::cos((L)k))) <= 1.2e-16 * (1 + extra_ulp), "cos near a zero of sin", k, c);
}

int main() {
  for (int i = 0; i < 200000; ++i) {
    const double sign = R() & 1 ? 1.0 : -1.0, pi = M_PI * ((int)(R() % 21) - 10);
    one(sign * std::pow(10.0, uniform(-300, -1)), 0.0);
    one(sign * std::pow(10.0, uniform(-18, -1)), 0.0);
    one(pi + sign * std::pow(10.0, uniform(-16, -1)), 0.0);
    one(pi + uniform(-0.0156, 0.0156), 0.0);                  // the table's side of the boundary and sin_near's
    one(sign * (0x1p-6 + (int)(R() % 2000 - 1000) * 0x1p-58), 0.0);
    one(uniform(-31.99, 31.99), 0.0);
    const double far = M_PI * (11 + (double)(R() % 100000)); // reduced out of line, one more rounding
    one(sign * far * (1 + (int)(R() % 3) * 0x1p-52), 0.6);
    one(far + sign * std::pow(10.0, uniform(-9, -1)), 0.6);
  }
  for (int n = -10; n <= 10; ++n)
    if (n) one(n * M_PI, 0.0);                                // the doubles nearest to the zeros
  for (double k : {1e-3, 1e-5, 1e-9, 1e-15, 1e-18, 1e-300, 5e-324, M_PI, -M_PI, 3 * M_PI}) {
    double gx, gy, s, c;
    line_energy_grad(k, 1.0, 1.0, -0.3, -0.5, gx, gy);
    const L ref = (2 + 4 * (L)-0.3 * std::cos((L)1.0)) * std::sin((L)k);
    check(std::fabs((L)gx - ref) <= 4 * (L)std::max(ulp(gx), 5e-324), "gradient factor near a zero", k, gx);
    cw_sincos(-k, s, c);
    double s1, c1;
    cw_sincos(k, s1, c1);
    check(s == -s1 && c == c1, "odd sine, even cosine", k, s);
  }
  double s, c;
  cw_sincos(0.0, s, c);
  check(s == 0.0 && !std::signbit(s) && c == 1.0, "sin(0)", 0.0, s);
  std::printf("%d failures\n", failures);
  return failures != 0;
}
