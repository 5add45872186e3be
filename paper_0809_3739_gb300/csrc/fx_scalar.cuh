// Short chains of FP64 scalars in integer arithmetic, for the dense n x n
// kernels: sums over a warp, reciprocals, inverse square roots and the scalars
// of a Householder reflector.
//
// A dependent FP64 operation costs about 130 cycles on a GB300, an integer
// one about 5.  A warp sum by shuffles is a chain of five FP64 additions, and
// 1 / (|x|^2 + |x_0| |x|) from |x|^2 one of about twenty operations; in
// integers both take the time of one or two.  Values carry 62 bits or more, so
// results are within half a unit in the last place of a double and a little.
#pragma once
#include <math.h>

#include "fft_fixed.cuh"

namespace itp {

// m 2^e, normalised: 2^63 <= m < 2^64.
struct FxNum {
  unsigned long long m;
  int e;
};

ITP_HD unsigned long long fx_mulhi(unsigned long long a, unsigned long long b) {
#ifdef __CUDA_ARCH__
  return __umul64hi(a, b);
#else
  return (unsigned long long)(((unsigned __int128)a * b) >> 64);
#endif
}
ITP_HD int fx_exponent(double d) { return (int)((fx_bits(d) >> 52) & 0x7ff); }
ITP_HD FxNum fx_normal(unsigned long long m, int e) {   // m > 0
  const unsigned h = (unsigned)(m >> 32);
  const int z = h ? fx_clz(h) : 32 + fx_clz((unsigned)m);
  FxNum r;
  r.m = m << z;
  r.e = e - z;
  return r;
}
// |d| for a normal d
ITP_HD FxNum fx_num(double d) {
  FxNum r;
  r.m = ((unsigned long long)fx_bits(d) << 11) | 0x8000000000000000ULL;
  r.e = fx_exponent(d) - 1023 - 63;
  return r;
}
// The nearest double (a normal one), with the sign of s.
ITP_HD double fx_round(FxNum a, long long s) {
  const long long q = (long long)(a.m >> 11) + (long long)((a.m >> 10) & 1ULL);
  const long long r = q + ((long long)(a.e + 63 + 1022) << 52);
  return fx_from_bits(r | (s & (long long)0x8000000000000000ULL));
}

// y as y 2^32, below 2^32 and even: a seed 1/2 <= y <= 1
ITP_HD unsigned fx_seed(float y) {
  y *= 4294967296.0f;
  return y >= 4294967040.0f ? 0xfffffffeu : (unsigned)y;
}
// the float f 2^k of the top 24 bits of m, 1 <= f < 2
ITP_HD float fx_top(unsigned long long m, int k) {
  const unsigned b = ((unsigned)(m >> 40) & 0x7fffffu) | ((127u + (unsigned)k) << 23);
#ifdef __CUDA_ARCH__
  return __uint_as_float(b);
#else
  float f;
  memcpy(&f, &b, 4);
  return f;
#endif
}
// y (1 + s 2^-63) with y = Y 2^-32, as a number scaled 2^64; at least 2^63
ITP_HD FxNum fx_refined(unsigned Y, long long s, int e) {
  const long long c = (long long)((unsigned long long)fx_wideu(Y, fx_lo(s), 0) >> 32);
  const unsigned long long z =
      ((unsigned long long)Y << 31) +
      (unsigned long long)fx_wide(2 * fx_hi(s), (int)(Y >> 1), c);   // scaled 2^63
  FxNum r;
  r.m = z << 1;
  r.e = e;
  if (z >> 63) {   // one
    r.m = 0x8000000000000000ULL;
    r.e = e + 1;
  } else if (!(z >> 62)) {   // a unit below one half
    r.m = 0x8000000000000000ULL;
  }
  return r;
}

// 1 / a: a single-precision seed and one third-order step, residual exact to
// 2^-63 (seed within 2^-22, so the cube of the residual is below that).
ITP_HD FxNum fx_recip(FxNum a) {
#ifdef __CUDA_ARCH__
  const unsigned Y = fx_seed(__frcp_rn(fx_top(a.m, 0)));
#else
  const unsigned Y = fx_seed(1.0f / fx_top(a.m, 0));
#endif
  const unsigned long long lo = (unsigned long long)fx_wideu(fx_lo((long long)a.m), Y, 0) >> 32;
  const unsigned long long t = (unsigned long long)fx_wideu((unsigned)(a.m >> 32), Y, (long long)lo);
  const long long r = (long long)(0x8000000000000000ULL - t);   // (1 - f y) 2^63
  const int h = (int)(r >> 16);
  return fx_refined(Y, r + (fx_wide(h, h, 0) >> 31), -127 - a.e);
}

// 1 / sqrt(a), likewise.  (a = f 2^E with E even and 1 <= f < 4; *F: f 2^62.)
ITP_HD FxNum fx_rsqrt(FxNum a, unsigned long long* F, int* E) {
  const int odd = (a.e + 63) & 1;
  *E = a.e + 63 - odd;
  *F = a.m >> (1 - odd);
#ifdef __CUDA_ARCH__
  const unsigned Y = fx_seed(rsqrtf(fx_top(a.m, odd)));
#else
  const unsigned Y = fx_seed(1.0f / sqrtf(fx_top(a.m, odd)));
#endif
  const unsigned long long t = fx_mulhi(*F, (unsigned long long)fx_wideu(Y, Y, 0));
  const long long r = (long long)(0x4000000000000000ULL - t);   // (1 - f y^2) 2^62
  const int h = (int)(r >> 16);
  // y (1 + r / 2 + 3 r^2 / 8)
  return fx_refined(Y, r + ((3 * fx_wide(h, h, 0)) >> 32), -64 - *E / 2);
}

// 1/d and 1/sqrt(d) for a finite d > 0.
ITP_HD double recip(double d) {
  const int e = fx_exponent(d);
  if (e < 23 || e > 2023) return 1.0 / d;
  return fx_round(fx_recip(fx_num(d)), 0);
}
ITP_HD double rsqrt64(double d) {
  const int e = fx_exponent(d);
  if (e < 23 || e > 2023) return 1.0 / sqrt(d);
  unsigned long long F;
  int E;
  return fx_round(fx_rsqrt(fx_num(d), &F, &E), 0);
}

// The reflector v = x - alpha e_1 of a vector x from s2 = |x|^2 and x_0:
// alpha = -sign(x_0) |x|, v_0 = x_0 - alpha and beta = 2 / v^T v =
// 1 / (|x|^2 + |x_0| |x|).  |x_0| <= |x|; s2 far from the ends of the range.
ITP_HD void fx_reflector(FxNum s2, double x0, double* alpha, double* beta, double* v0) {
  unsigned long long F;
  int E;
  const FxNum z = fx_rsqrt(s2, &F, &E);
  // |x| = f 2^(E/2) / sqrt(f), here N 2^(E/2 - 63)
  unsigned long long N = fx_mulhi(F, z.m);             // scaled 2^62
  if (z.e != -64 - E / 2) N = 0x4000000000000000ULL;   // f = 1
  N = N >> 63 ? ~0ULL : N << 1;
  const int en = E / 2 - 63;
  const FxNum x = fx_num(x0);
  const int down = fx_exponent(x0) == 0 ? 64 : en - x.e;
  const unsigned long long X = down > 63 ? 0 : (down < 0 ? ~0ULL : x.m >> down);
  const unsigned long long D = (F >> 1) + (fx_mulhi(X, N) >> 1);   // scaled 2^61, 2^E
  const long long sx = fx_bits(x0) > 0 ? 0 : -1;                   // the sign of v_0
  FxNum nn;
  nn.m = N;
  nn.e = en;
  *alpha = fx_round(nn, ~sx);
  *v0 = fx_round(fx_normal((X >> 1) + (N >> 1), en + 1), sx);
  *beta = fx_round(fx_recip(fx_normal(D, E - 61)), 0);
}

// ---- sums over lanes ---------------------------------------------------------
// d as an integer of 57 bits at the biased exponent e >= that of d: d =
// result 2^(e - 1079), rounded to nearest; 32 of them add up below 2^62.
ITP_HD long long fx_addend(double d, int e) {
  const long long b = fx_bits(d);
  const int ex = (int)((b >> 52) & 0x7ff);
  long long m = fx_shr(((b & 0xfffffffffffffLL) | 0x10000000000000LL) << 5, e - ex);
  m = ex == 0 ? 0 : (m + 1) >> 1;
  const long long s = b >> 63;
  return (m ^ s) - s;
}
ITP_HD double fx_sum_double(long long t, int e) {   // t 2^(e - 1079)
  if (t == 0) return 0.0;
  const long long s = t >> 63;
  return fx_round(fx_normal((unsigned long long)((t ^ s) - s), e - 1079), s);
}
#ifdef __CUDACC__
// The sum over the 32 lanes as t 2^(e - 1079); false where the exponents are
// near the ends of the range (infinities and NaN too): then there is none.
__device__ __forceinline__ bool fx_warp_sum(double v, long long* t, int* e) {
  const int em = __reduce_max_sync(0xffffffffu, fx_exponent(v));
  *e = em;
  if (em < 64 || em > 1900) return false;
  const long long m = fx_addend(v, em);
  constexpr unsigned kMask = (1u << 27) - 1;
  const unsigned l0 = __reduce_add_sync(0xffffffffu, (unsigned)m & kMask);
  const unsigned l1 = __reduce_add_sync(0xffffffffu, (unsigned)(m >> 27) & kMask);
  const int l2 = __reduce_add_sync(0xffffffffu, (int)(m >> 54));
  *t = (long long)l0 + ((long long)l1 << 27) + ((long long)l2 << 54);
  return true;
}
// The sum over the 32 lanes, to every lane.
__device__ __forceinline__ double warp_sum64(double v) {
  long long t;
  int e;
  if (fx_warp_sum(v, &t, &e)) return fx_sum_double(t, e);
  for (int o = 16; o; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}
#endif

}  // namespace itp
