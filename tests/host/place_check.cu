// Host-side check of the demodulation's spline position (spline_place, compiled as host
// code) against long double, for sampling intervals from 16 s to 1e-7 s: inside the data the
// interval is the right one, 0 <= f < 1 and i + f is 2 j - phi (2/dt) to the double-floats'
// rounding; outside it, also where the delay is thousands of millions of half-samples, the
// sample is refused.  Prints the worst error in half-samples and "OK".
#include <cmath>
#include <cstdio>
#include <random>

#include "../../paper_1003_0844_gb300/csrc/fs_demod.cuh"

using namespace fs;
using Q = long double;

int main() {
  std::mt19937_64 rng(5);
  std::uniform_real_distribution<double> u01(0.0, 1.0);
  long fails = 0, inside = 0, outside = 0;
  double worst = 0.0;
  const double dts[] = {16.0, 2.0, 0.5, 0.3, 1e-2, 1e-3, 1e-4, 6.1e-5, 2.5e-5, 1e-5, 3e-6, 1e-6, 4e-7, 1e-7};
  const int ns[] = {16, 4097, 43082, 1 << 20};
  for (double dt : dts)
    for (int n : ns) {
      const df32 tod = df_from_double(2.0 / dt);
      const Q scale = (Q)tod.hi + (Q)tod.lo;
      auto one = [&](int j, double phid) {
        const df32 phi = df_from_double(phid);
        const Q u = 2.0L * j - ((Q)phi.hi + (Q)phi.lo) * scale, last = 2.0L * n - 2;
        // v's rounding, and the last bit of f itself
        const Q tol = fabsl(2.0L * j - u) * ldexpl(1.0L, -44) + ldexpl(1.0L, -23);
        unsigned i;
        float f;
        const bool in = spline_place(phi, tod, j, n, &i, &f);
        if (u > tol && u < last - tol) {
          const double err = (double)fabsl((Q)i + (Q)f - u);
          if (!in || !(f >= 0.f && f < 1.f) || i > 2u * (unsigned)n - 2u || !(err <= (double)tol)) {
            if (fails++ < 10) printf("inside: dt %g n %d j %d phi %.17g: i %u f %g want %.9Lf\n", dt, n, j, phid, i, f, u);
          } else {
            worst = std::fmax(worst, err);
          }
          inside++;
        } else if (u < -tol || u > last + tol) {
          if (in && fails++ < 10) printf("outside: dt %g n %d j %d phi %.17g taken as %u\n", dt, n, j, phid, i);
          outside++;
        }
      };
      for (int s = 0; s < 20000; s++) {
        const int j = (int)(u01(rng) * n);
        one(j, 500.0 * (2.0 * u01(rng) - 1.0));                       // any delay
        const double t = (u01(rng) * (n + 1) - 1.0) * dt;             // a source time in the data
        if (std::fabs(j * dt - t) < 500.0) one(j, j * dt - t);
        one(j, (j - std::floor(u01(rng) * 2 * n) * 0.5) * dt);        // on a half-sample, to rounding
        one(j, (s & 1 ? 500.0 : -500.0) * std::exp(-8.0 * u01(rng)));
      }
    }
  printf("inside %ld outside %ld worst %.3e failures %ld\n", inside, outside, worst, fails);
  if (fails || inside < 100000 || outside < 100000) return 1;
  printf("OK\n");
  return 0;
}
