// Host program of test_fixed_point.py: the vector functions of the fixed-point
// FFT arithmetic (fft_fixed.cuh), compiled for the CPU.  For each radix and
// kind of input: real pairs times factors -> DFT -> twiddles -> packed and
// unpacked -> inverse-direction DFT -> factors, against the same chain in
// extended precision; prints "radix kind rms_error" relative to the 2-norm,
// then the special values.
#include <cmath>
#include <cstdio>
#include <cstdlib>

#include "fft_fixed.cuh"

using namespace itp;
typedef long double ld;

static double uniform() { return rand() / (double)RAND_MAX - 0.5; }
static const ld kPi = acosl(-1.0L);

static void entry(ld c, int* h, int* l) {
  const ld t = c * 536870912.0L, r = floorl(t + 0.5L);
  ld q = roundl((t - r) * 4294967296.0L);
  if (q > 2147483647.0L) q = 2147483647.0L;
  if (q < -2147483647.0L) q = -2147483647.0L;
  *h = (int)r;
  *l = (int)q;
}

template <int N>
static void dft_ref(int dir, ld* re, ld* im) {
  ld yr[N], yi[N];
  for (int k = 0; k < N; ++k) {
    yr[k] = yi[k] = 0;
    for (int n = 0; n < N; ++n) {
      const ld c = cosl(2 * kPi * ((n * k) % N) / N), s = dir * sinl(2 * kPi * ((n * k) % N) / N);
      yr[k] += re[n] * c - im[n] * s;
      yi[k] += re[n] * s + im[n] * c;
    }
  }
  for (int k = 0; k < N; ++k) { re[k] = yr[k]; im[k] = yi[k]; }
}

template <int N>
static void chain(int kind) {
  fx_tw tw[256];
  for (int m = 0; m < 256; ++m) {
    entry(cosl(2 * kPi * m / 256), &tw[m].rh, &tw[m].rl);
    entry(-sinl(2 * kPi * m / 256), &tw[m].ih, &tw[m].il);
  }
  ld err = 0, norm = 0;
  for (int rep = 0; rep < 2000; ++rep) {
    double2 p[N], f[N], g[N];
    ld re[N], im[N];
    const double all = kind == 4 ? 1e-140 : (kind == 5 ? 1e140 : 1.0);
    for (int i = 0; i < N; ++i) {
      double s = all;                                     // 0, 4, 5: uniform noise
      if (kind == 1) s = exp(-40 * fabs(uniform()));      // nine orders of magnitude
      if (kind == 2) s = i == rep % N;                    // one nonzero element
      p[i].x = kind == 3 ? 1.0 : s * uniform();           // 3: a constant
      p[i].y = kind == 3 ? 0.7 : s * uniform();
      f[i] = make_double2(exp(uniform()), exp(uniform()));
      g[i] = make_double2(exp(uniform()), exp(uniform()));
      re[i] = (ld)p[i].x * f[i].x;
      im[i] = (ld)p[i].y * f[i].y;
    }
    const int q = rep % 256 / N;
    SVec<cfx, N> a;
    a.template from_pairs<true>(p, f);
    a.template dft<-1>();
    if (rep & 1) fx_twiddle<true>(a, tw, q);
    else fx_twiddle<false>(a, tw, q);
    a.close();
    a.open();
    a.template dft<1>();
    a.mul_pairs(g);
    dft_ref<N>(-1, re, im);
    for (int k = 0; k < N; ++k) {
      const ld c = cosl(2 * kPi * q * k / 256), s = (rep & 1 ? 1 : -1) * sinl(2 * kPi * q * k / 256);
      const ld t = re[k] * c - im[k] * s;
      im[k] = re[k] * s + im[k] * c;
      re[k] = t;
    }
    dft_ref<N>(1, re, im);
    for (int k = 0; k < N; ++k) {
      const ld dx = ldexpl((ld)a.v[k].x, a.e - kFxBias) - re[k] * g[k].x;
      const ld dy = ldexpl((ld)a.v[k].y, a.e - kFxBias) - im[k] * g[k].y;
      err += (dx * dx + dy * dy) / (all * all);
      norm += (re[k] * re[k] * g[k].x * g[k].x + im[k] * im[k] * g[k].y * g[k].y) / (all * all);
    }
  }
  printf("%d %d %.4e\n", N, kind, (double)sqrtl(err / norm));
}

template <int N>
static void special(const char* name, double2 odd) {
  double2 p[N], f[N];
  for (int i = 0; i < N; ++i) {
    p[i] = make_double2(0.0, 0.0);
    f[i] = make_double2(1.5, 1.5);
  }
  p[1] = odd;
  SVec<cfx, N> a;
  a.template from_pairs<true>(p, f);
  a.template dft<-1>();
  a.close();
  a.open();
  a.template dft<1>();
  printf("%s %.17g %.17g\n", name, a.to_double(a.v[1].x) / N, a.to_double_times(a.v[1].y, 2.0) / N);
}

int main() {
  for (int kind = 0; kind < 6; ++kind) {
    chain<2>(kind);
    chain<3>(kind);
    chain<4>(kind);
    chain<6>(kind);
    chain<8>(kind);
    chain<12>(kind);
    chain<16>(kind);
  }
  special<8>("zero", make_double2(0.0, 0.0));
  special<8>("nan", make_double2(NAN, 0.0));
  special<8>("inf", make_double2(0.0, INFINITY));
  special<8>("subnormal", make_double2(4e-320, -4e-320));
  special<8>("large", make_double2(1e300, 1e300));
  special<8>("small", make_double2(1e-300, -1e-300));
  special<8>("one", make_double2(1.0, -2.0));
  return 0;
}
