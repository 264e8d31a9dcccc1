// The kernels' exponential below the normal range, and a Fermi value there, against long double.
#define main fixed_math_main
#include "fixed_math_cases.cpp"
#undef main

int main() {
  const double inf = std::numeric_limits<double>::infinity();
  auto one = [](double t) {
    double em, em0, unused;
    const double y = exp_neg<kBoseExp>(t, em), y0 = exp_neg<true>(t, em0);
    check(y == exp_neg<kFermiExp>(t, unused), "exp without e^t - 1", t, y);
    check(__double_as_longlong(em) == __double_as_longlong(em0), "e^t - 1 in both forms", t, em);
    if (y0 != 0.0 || t < -1023.0) check(y == y0, "both forms in the normal range", t, y);
    // one rounding of a value within 2^-60 of e^t: half a unit of 2^-1074
    if (t < -708.4 && t > -1023.0) check(std::fabs((double)(((L)y - std::exp((L)t)) / 0x1p-1074L)) <= 0.501, "subnormal exp", t, y);
  };
  for (int i = 0; i < 300000; ++i) {
    one(-uniform(708.0, 746.0)); one(-uniform(744.0, 745.2)); one(-uniform(0.0, 1100.0)); one(-uniform(708.39, 708.4));
  }
  for (double t : {-708.0, -708.3964, -708.3965, -709.0, -745.1, -745.2, -746.0, -1023.9, -1024.0, -1e300, -inf}) one(t);
  double em;
  check(exp_neg<kBoseExp>(-745.2, em) == 0.0 && exp_neg<kBoseExp>(-745.1, em) == 5e-324, "last subnormal", -745.1, em);
  check(std::isnan(exp_neg<kBoseExp>(std::nan(""), em)) && std::isnan(em), "exp(NaN)", 0.0, em);
  const int seg[5] = {0, 1, 0, 2, 2}, fvr[4] = {1, 0, -1, 0};   // g_sigma(x) and g_sigma(-x)
  for (double x : {720.0, -740.0}) {
    double fv[2], bv[2];
    fermi_segment<false, false>(seg, fvr, &x, 1.0, fv, nullptr);
    fermi_segment<true, false>(seg, fvr, &x, 1.0, bv, nullptr);
    const double small = x > 0 ? fv[0] : fv[1], bose = x > 0 ? bv[0] : bv[1];
    check(std::fabs((double)((small - std::exp(-std::fabs((L)x))) / 0x1p-1074L)) <= 1.0, "Fermi tail", x, small);
    check(std::fabs((double)((bose + std::exp(-std::fabs((L)x))) / 0x1p-1074L)) <= 1.0, "Bose tail", x, bose);
  }
  std::printf("%d failures\n", failures);
  return failures != 0;
}
