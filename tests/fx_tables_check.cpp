// Host check of the tables of the fixed-point rate evaluation (csrc/mech_tables.cpp) after changes of ln A: the
// update gives the tables that building all of them gives.  Prints, per change, whether they are equal and the
// lower end of the temperature interval, then the time of a full build over that of an update.
#include <chrono>
#include <cmath>
#include <cstdio>
#include <cstring>

#include "../paper_2105_12070_gb300/csrc/chem_internal.h"

using namespace chemgpu;

template <class T>
static bool same(const std::vector<T>& a, const std::vector<T>& b) {
  return a.size() == b.size() && (a.empty() || std::memcmp(a.data(), b.data(), a.size() * sizeof(T)) == 0);
}

int main(int argc, char** argv) {
  HostMech m;
  std::string err;
  if (argc < 2 || !parse_mechanism(argv[1], m, err)) {
    std::printf("%s\n", err.c_str());
    return 1;
  }
  const HostMech first = m;
  const int R = m.R;
  auto lnA = [&](HostMech& h, int r) -> double& { return h.rxd[(size_t)r * kRxDoubles]; };
  for (int change = 0; change < 7; ++change) {
    for (int r = 0; r < R; ++r) lnA(m, r) = first.rxd[(size_t)r * kRxDoubles];
    if (change == 1)
      for (int r = 0; r < R; ++r) lnA(m, r) += std::sin(1.0 + r);
    if (change == 2) lnA(m, R / 2) = -700.0;
    if (change == 3) lnA(m, 0) = 690.0;
    if (change == 4) lnA(m, R - 1) = 1e6;                               // beyond the fixed-point format
    if (change == 5) {  // an exponent bound that 512 K keeps and 256 K does not, for the highest barrier
      int top = 0;
      for (int r = 0; r < R; ++r)
        if (m.rxd[(size_t)r * kRxDoubles + 2] > m.rxd[(size_t)top * kRxDoubles + 2]) top = r;
      const double* d = &m.rxd[(size_t)top * kRxDoubles];
      lnA(m, top) = (1000.0 - 13.0 * std::fabs(d[1])) / 1.4427 - d[2] / 384.0;
    }
    update_fx_lnA(m);
    HostMech full = m;
    full.fxk.assign(full.fxk.size(), 7);
    full.fx_T = {1.0, 2.0};
    build_fx_tables(full);
    const bool ok = same(m.fxk, full.fxk) && same(m.fx_T, full.fx_T) && same(m.spf, full.spf) && same(m.fxo, full.fxo) &&
                    same(m.rxd_t, full.rxd_t) && same(m.srx, full.srx) && same(m.effx, full.effx);
    std::printf("%d %g\n", ok ? 1 : 0, m.fx_T[0]);
  }
  auto best = [&](auto&& f) {
    double t = 1e9;
    for (int i = 0; i < 20; ++i) {
      const auto t0 = std::chrono::steady_clock::now();
      f();
      t = std::fmin(t, std::chrono::duration<double>(std::chrono::steady_clock::now() - t0).count());
    }
    return t;
  };
  const double tb = best([&] { build_fx_tables(m); }), tu = best([&] { update_fx_lnA(m); });
  std::fprintf(stderr, "build %.1f us, update %.1f us\n", tb * 1e6, tu * 1e6);
  std::printf("%g\n", tb / tu);
  return 0;
}
