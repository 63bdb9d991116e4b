// physical() on the host against its definition, rho > 0 and E - |m|^2 / (2 rho) > 0
// in the same type, over states whose scale spans the range in which |m|^2 does
// not overflow (where it underflows the definition takes it as zero; where it
// is denormal neither has more than a few bits of it, and the state is left
// out); pressures within 1e-4 of zero relative to E are left out too
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
      const T q = u[1] * u[1] + u[2] * u[2] + u[3] * u[3], p = u[4] - T(0.5) * q / u[0];
      if (q > 0 && q < std::numeric_limits<T>::min()) continue;
      if (u[0] > 0 && std::fabs(p) < T(1e-4) * std::fabs(u[4])) continue;
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

int main() { return run<float>(-33, 17) + run<double>(-250, 150) ? 1 : 0; }
