// Host check of csrc/fixed_math.cuh against long double (64 or more significand bits): prints the
// largest errors of fx_exp2 (units of the last place), fx_log2 and fx_of (units of 2^-52) and fx_rcp (units
// of the last place; the host takes its FP32 seed from a division, and from its neighbours up to two floats away).
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <random>

#include "../paper_2105_12070_gb300/csrc/fixed_math.cuh"

using namespace chemgpu;

static long double ulps(double got, long double want) {
  const double w = (double)want;
  return std::fabs((long double)got - want) / (long double)(std::nextafter(std::fabs(w), INFINITY) - std::fabs(w));
}

int main(int argc, char** argv) {
  const double span = argc > 1 ? std::atof(argv[1]) : 1000.0;  // exponent range of the arguments
  std::mt19937_64 g(7);
  std::uniform_real_distribution<double> U(-1.0, 1.0);
  const long double one = 4503599627370496.0L;
  long double we = 0, wl = 0, wf = 0, wr = 0;
  auto check_exp = [&](fx_t x) { we = std::fmax(we, ulps(fx_exp2(x), std::exp2((long double)x / one))); };
  auto check_log = [&](double x) { wl = std::fmax(wl, std::fabs((long double)fx_log2(x) - std::log2((long double)x) * one)); };
  auto check_rcp = [&](double a) {
    wr = std::fmax(wr, ulps(fx_rcp(a), 1.0L / a));
    uint64_t m = ((uint64_t)fx_bits(a) & 0xfffffffffffffULL) | 0x3ff0000000000000ULL, r;
    float x = 1.0f / (float)std::fmin(fx_from_bits((int64_t)m), 2.0 - std::ldexp(1.0, -23));
    uint32_t rf;
    std::memcpy(&rf, &x, 4);
    // (the floats next to 1/2 from below are half as far apart: one more)
    for (int s = -3; s <= 2; ++s) wr = std::fmax(wr, ulps(fx_rcp_from(a, rf + (uint32_t)s, r), 1.0L / a));
  };
  for (int i = 0; i < 200000; ++i) {
    const double v = span * U(g);
    check_exp(fx_of(v));
    wf = std::fmax(wf, std::fabs((long double)fx_of(v) - (long double)v * one));
    check_log(std::exp2(v));
    check_log(1.0 + 1e-3 * U(g));
    check_rcp(std::exp2(v) * (i & 1 ? 1.0 : -1.0));
  }
  // both sides of every table interval
  for (int n = -2; n <= 2; ++n)
    for (int j = 0; j < 128; ++j)
      for (int s = -1; s <= 1; ++s) check_exp(((fx_t)n << 52) + ((fx_t)j << 45) + s);
  for (int i = 0; i <= 128; ++i) {
    const double x = 1.0 + i / 128.0;
    check_log(x);
    check_log(std::nextafter(x, 0.5 + (i > 0)));
    check_log(std::nextafter(x, 4.0));
    check_rcp(x);
    check_rcp(std::nextafter(x, 0.0));
    check_rcp(x * (1.0 - std::ldexp(1.0, -24)));
    check_rcp(std::ldexp(std::nextafter(x, 4.0), i * 15 - 960));
  }
  // outside the normal range the reciprocal is the division's
  for (double a : {0.0, -0.0, 1e-310, 1e308, (double)INFINITY, -(double)INFINITY})
    if (fx_rcp(a) != 1.0 / a) wr = 1e9;
  if (fx_rcp(NAN) == fx_rcp(NAN)) wr = 1e9;
  std::printf("%.6Lf %.6Lf %.6Lf %.6Lf\n", we, wl, wf, wr);
  return 0;
}
