// Host program of test_dense_scalars.py: the integer scalars of the dense
// kernels (fx_scalar.cuh) against extended precision.  Prints "name error",
// the largest relative error in units of 2^-53.
#include <cmath>
#include <cstdio>
#include <cstdlib>

#include "fx_scalar.cuh"

using namespace itp;
typedef long double ld;

static double uniform() { return (rand() + rand() / (RAND_MAX + 1.0)) / (RAND_MAX + 1.0); }
static ld worst[5];
static void note(int which, ld got, ld want) {
  if (fabsl(want) > 1.8e308L && std::isinf((double)got)) return;   // beyond a double
  const ld unit = fmaxl(fabsl(want), 0x1p-1022L);   // (subnormal results: of the smallest normal)
  const ld e = want == 0 ? (got == 0 ? 0 : 1e9L) : fabsl(got - want) / unit * 0x1p53L;
  if (!(e <= worst[which])) worst[which] = e;
}
static void one(double d) {
  note(0, recip(d), 1.0L / d);
  note(1, rsqrt64(d), 1.0L / sqrtl((ld)d));
}
static void reflector(double s2, double x0) {
  double a, b, v;
  fx_reflector(fx_num(s2), x0, &a, &b, &v);
  const ld n = sqrtl((ld)s2), sg = x0 > 0 ? 1 : -1;
  note(2, a, -sg * n);
  note(3, v, x0 + sg * n);
  note(4, b, 1.0L / ((ld)s2 + fabsl((ld)x0) * n));
}

int main() {
  const double edge[] = {1.0, 1.0 + 0x1p-52, 1.0 - 0x1p-53, 2.0 - 0x1p-52, 4.0 - 0x1p-51, 2.0,
                         2.0 + 0x1p-51, 1.5, 3.0, 1.0 + 0x1p-23, 2.0 - 0x1p-23, 4.0 - 0x1p-21};
  for (double d : edge)
    for (int k = -900; k <= 900; k += 75) {
      one(ldexp(d, k));
      if (abs(k) > 800) continue;
      for (double f : {0.0, 1.0, 0.5, 1e-10, 1e-200, 1.0 - 0x1p-53})
        for (double s : {1.0, -1.0}) {
          const double x0 = s * f * (double)sqrtl((ld)ldexp(d, k));
          if (x0 == 0 || fabs(x0) > 0x1p-1000) reflector(ldexp(d, k), x0);
        }
    }
  for (double d : {5e-324, 1e-310, 1e-300, 1e300, 1.7e308}) one(d);
  for (int i = 0; i < 200000; ++i) {
    const double d = ldexp(1.0 + uniform(), rand() % 1800 - 900);
    one(d);
    const double s2 = ldexp(1.0 + uniform(), rand() % 1600 - 800);
    reflector(s2, (2 * uniform() - 1) * (double)sqrtl((ld)s2));
  }
  const char* names[] = {"recip", "rsqrt", "alpha", "v0", "beta"};
  for (int q = 0; q < 5; ++q) printf("%s %.4Lf\n", names[q], worst[q]);
  // sums of 32: error against half a unit of 2^-57 of the largest per addend
  ld bad = 0;
  for (int i = 0; i < 20000; ++i) {
    double v[32];
    ld sum = 0, big = 0;
    int e = 0;
    const int spread = i % 3 == 0 ? 1 : (i % 3 == 1 ? 60 : 700), base = rand() % 500 - 200;
    for (double& x : v) {
      x = ldexp(2 * uniform() - 1, base + rand() % spread);
      if (rand() % 10 == 0) x = 0;
      sum += x;
      big = fmaxl(big, fabsl((ld)x));
      e = fx_max(e, fx_exponent(x));
    }
    if (e < 64) continue;
    long long t = 0;
    for (double x : v) t += fx_addend(x, e);
    const ld got = fx_sum_double(t, e);
    const ld lim = 32 * 0x1p-57L * big + fabsl(sum) * 0x1.01p-53L;
    bad = fmaxl(bad, lim == 0 ? fabsl(got) : fabsl(got - sum) / lim);
  }
  printf("sum %.4Lf\n", bad);
  return 0;
}
