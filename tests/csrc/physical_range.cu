// physical() on the host against rho > 0 and E - |m|^2 / (2 rho) > 0 in long
// double, over states of scales at which neither rho E nor |m|^2 need lie in the
// type's range; pressures within 1e-4 of zero relative to E are left out
// (rounding).  Exit status 0 iff all agree.
#include <cmath>
#include <cstdio>
#include <limits>

#include "dg_common.cuh"
using namespace dgk;

template <class T>
int run(int lo, int hi) {
  unsigned x = 7;
  auto rnd = [&] { return ((x = x * 1664525u + 1013904223u) >> 8) / 16777216.0; };
  int bad = 0, n = 0, phys = 0;
  for (int ex = lo; ex <= hi; ++ex)
    for (int k = 0; k < 200; ++k) {
      const double s = std::pow(10.0, ex), r = s * (0.1 + rnd()), v = 3.0 * (rnd() - 0.5);
      T u[5] = {(T)(rnd() < 0.05 ? -r : r), (T)(r * v), (T)(r * 0.3 * v), (T)(r * 0.1), (T)(s * 2.0 * rnd())};
      const long double q = (long double)u[1] * u[1] + (long double)u[2] * u[2] + (long double)u[3] * u[3];
      const long double p = u[4] - q / (2 * (long double)u[0]);
      if (u[0] > 0 && fabsl(p) < 1e-4L * u[4]) continue;
      const bool want = u[0] > 0 && p > 0, got = physical<3>(u, (T)0.4);
      ++n;
      phys += want;
      if (want != got && bad++ < 5) printf("FP%d scale 1e%d: want %d got %d\n", (int)sizeof(T) * 8, ex, want, got);
    }
  printf("FP%d: %d states, %d physical, %d wrong\n", (int)sizeof(T) * 8, n, phys, bad);
  const T nan = std::numeric_limits<T>::quiet_NaN(), inf = std::numeric_limits<T>::infinity();
  const T odd[][5] = {{nan, 0, 0, 0, 1}, {1, nan, 0, 0, 1}, {1, 0, 0, 0, nan}, {0, 0, 0, 0, 1}, {1, 0, 0, 0, 0},
                      {1, inf, 0, 0, 1}, {1, 0, 0, 0, -1}};
  for (auto& u : odd)
    if (physical<3>(u, (T)0.4)) ++bad, printf("accepted an unphysical state\n");
  return bad;
}

int main() { return run<float>(-33, 33) + run<double>(-250, 250) ? 1 : 0; }
