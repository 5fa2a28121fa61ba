// Calls a function of chem_jacobian's type from two host threads at once, each with arguments of its own: `calls`
// times from the first and until those are done from the second (at most 100 times as often).  Returns how
// many calls of either failed.
#include <atomic>
#include <cstdint>
#include <thread>

typedef int (*jacobian_fn)(const void* mech, double p, const double* T, const double* Y, int64_t n, double* J,
                           void* stream);
struct Side {
  const void* mech;
  const double *T, *Y;
  int64_t n;
  double* J;
  void* stream;
};

extern "C" int two_threads(jacobian_fn fn, double p, const Side* a, const Side* b, int calls) {
  std::atomic<int> failed{0};
  std::atomic<bool> done{false};
  auto call = [&](const Side* s) { failed += fn(s->mech, p, s->T, s->Y, s->n, s->J, s->stream) != 0; };
  std::thread other([&] {
    for (int64_t i = 0; i < 100 * (int64_t)calls && !done; ++i) call(b);
  });
  for (int i = 0; i < calls; ++i) call(a);
  done = true;
  other.join();
  return failed;
}
