// 64-bit block fixed point: the arithmetic of the FP64 FFT passes.
//
// A GB300 SM issues one FP64 instruction per sub-partition and about 78
// cycles, but a 64-bit integer add takes 2 cycles and a 32 x 32 + 64-bit
// multiply-add (IMAD.WIDE) 2 in a chain and 3.2 with general operands, a
// shift or a bit operation 2 (measured with chains of independent
// instructions at 8 warps per sub-partition).  The passes are bound by that
// FP64 rate alone, so their transforms run in integers instead: the values
// that one thread transforms together (a vector of up to 16 complex numbers)
// share one exponent and are 58-bit signed integers, additions are exact, a
// twiddle product is twelve IMAD.WIDE, and between stages -- in shared memory
// and in the half spectrum in HBM -- a complex value is 16 bytes as before.
//
// Accuracy.  An element enters a vector rounded to 2^-57 of the vector's
// largest component, i.e. to at least four bits more than the 53 of a double
// of that size, and every product is rounded to an integer whose vector is
// scaled to about 2^59; an FP64 transform rounds each intermediate sum and
// product to 53 bits.  So each small DFT has less error, relative to the
// 2-norm of its inputs, than its FP64 form, and so do the passes.
//
// Packed form of a complex value (x, y), 8 bytes each: the upper 58 bits are
// the signed components, the lower 6 bits of x and of y hold the lower and
// upper half of a 12-bit exponent es; the value is x * 2^(es - kBias), the
// exponent bits counted as part of x (they lie below its precision).  All
// values that one thread stores together carry the same es, chosen so that
// the largest component fills the 64 bits.  es = 4095 marks a vector that a
// NaN or an infinity has reached: it spreads to everything transformed from
// it, as it would in floating point.  The exponent range is wider than that of
// a double (2^-2048 .. 2^2047 around the components' 2^63); below it values
// are zero.
//
// Every unpacking shifts right and so rounds down, which on average takes
// half a unit from each component.  Rounding errors of one sign would add up
// over the passes, so the mean is given back: summed over the inputs of a DFT
// it appears in the output of index 0 alone, and is added there.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>
#include <string.h>

#include "fft_common.cuh"

namespace itp {

constexpr int kFxTop = 4095;           // es of a vector with a NaN or infinity
constexpr int kFxBias = 2048 + 62;     // value = component * 2^(es - kFxBias)
constexpr int kFxDrop = 6;             // exponent bits at the bottom of a component
constexpr int kFxPoison = 1 << 20;     // exponent of a poisoned open vector

ITP_HD int fx_hi(long long v) { return (int)(v >> 32); }
ITP_HD unsigned fx_lo(long long v) { return (unsigned)v; }
// a * b + c as one instruction (the compiler made two or three of the C form:
// FP64 merged pass of 48 states at 128^3 2.15 -> 1.74 ms)
ITP_HD long long fx_wide(int a, int b, long long c) {
#ifdef __CUDA_ARCH__
  long long r;
  asm("mad.wide.s32 %0, %1, %2, %3;" : "=l"(r) : "r"(a), "r"(b), "l"(c));
  return r;
#else
  return (long long)a * b + c;
#endif
}
ITP_HD long long fx_wideu(unsigned a, unsigned b, long long c) {
#ifdef __CUDA_ARCH__
  long long r;
  asm("mad.wide.u32 %0, %1, %2, %3;" : "=l"(r) : "r"(a), "r"(b), "l"(c));
  return r;
#else
  return (long long)((unsigned long long)a * b + (unsigned long long)c);
#endif
}
ITP_HD int fx_clz(unsigned v) {
#ifdef __CUDA_ARCH__
  return __clz((int)v);
#else
  return v ? __builtin_clz(v) : 32;
#endif
}
ITP_HD int fx_max(int a, int b) { return a > b ? a : b; }
ITP_HD int fx_min(int a, int b) { return a < b ? a : b; }
// v >> n, n >= 0 (63 and more: the sign)
ITP_HD long long fx_shr(long long v, int n) {
#ifdef __CUDA_ARCH__
  long long r;   // the instruction clamps the count
  asm("shr.s64 %0, %1, %2;" : "=l"(r) : "l"(v), "r"(n));
  return r;
#else
  return v >> (n > 63 ? 63 : n);
#endif
}
ITP_HD long long fx_shl(long long v, int n) { return (long long)((unsigned long long)v << n); }
// v * p for p = 2^n, n < 32: a left shift on the multiplier, which the passes
// keep less busy than the shifter
ITP_HD long long fx_mulp(long long v, unsigned p) {
  const long long lo = (long long)((unsigned long long)fx_lo(v) * p);
  return lo + ((long long)((unsigned long long)((unsigned)fx_hi(v) * p) << 32));
}
ITP_HD long long fx_bits(double d) {
#ifdef __CUDA_ARCH__
  return __double_as_longlong(d);
#else
  long long v;
  memcpy(&v, &d, 8);
  return v;
#endif
}
ITP_HD double fx_from_bits(long long v) {
#ifdef __CUDA_ARCH__
  return __longlong_as_double(v);
#else
  double d;
  memcpy(&d, &v, 8);
  return d;
#endif
}

// ---- products ----------------------------------------------------------------
// x * c for a constant 0 < c < 1, c = (H + L 2^-32) 2^-31 (|x| < 2^61).
template <int H, int L>
ITP_HD long long fx_mulc(long long x) {
  const int xh = fx_hi(x);
  long long c = fx_wideu(fx_lo(x), (unsigned)H, 1LL << 31);
  c = fx_wide(xh, L, c);
  const long long y = fx_wide(xh, H, c >> 32);   // x c / 2
  return y + y;
}

// The constants of the radix-3 .. radix-16 codelets.
ITP_HD long long fx_cos8(long long x) { return fx_mulc<1984016189, -902489949>(x); }    // cos(pi/8)
ITP_HD long long fx_sin8(long long x) { return fx_mulc<821806413, 1565705635>(x); }     // sin(pi/8)
ITP_HD long long fx_sum8(long long x) { return fx_mulc<658338954, 663215686>(x); }      // cos + sin - 1
ITP_HD long long fx_dif8(long long x) { return fx_mulc<1162209775, 1826771711>(x); }    // cos - sin
ITP_HD long long fx_cos12(long long x) { return fx_mulc<1859775393, 1630710223>(x); }   // sqrt(3)/2
ITP_HD long long fx_sum12(long long x) { return fx_mulc<786033569, 1630710223>(x); }    // (sqrt(3)-1)/2
ITP_HD long long fx_rt2(long long x) { return fx_mulc<1518500250, -51432894>(x); }      // sqrt(1/2)

// a * exp(2 pi i t / 48), t a compile-time multiple of 3 or 4: quarter turns
// for free, 45 degrees with two products, the others with three.
template <int T>
ITP_HD cfx fx_rot(cfx a) {
  constexpr int t = ((T % 48) + 48) % 48, q = t / 12, r = t % 12;
  static_assert(r == 0 || r == 3 || r == 4 || r == 6 || r == 8 || r == 9, "angle");
  cfx b = a;
  if constexpr (r == 6) {
    b.x = fx_rt2(a.x - a.y);
    b.y = fx_rt2(a.x + a.y);
  } else if constexpr (r == 3 || r == 9) {
    const long long s = a.x + a.y;
    const long long k = r == 3 ? fx_cos8(s) : fx_sin8(s);
    b.x = k - a.y - fx_sum8(a.y);
    b.y = r == 3 ? k - fx_dif8(a.x) : k + fx_dif8(a.x);
  } else if constexpr (r == 4 || r == 8) {
    const long long s = a.x + a.y;
    const long long k = r == 4 ? fx_cos12(s) : s >> 1;
    b.x = k - a.y - fx_sum12(a.y);
    b.y = r == 4 ? k - fx_sum12(a.x) : k + fx_sum12(a.x);
  }
  cfx c = b;
  if constexpr (q == 1) { c.x = -b.y; c.y = b.x; }
  if constexpr (q == 2) { c.x = -b.x; c.y = -b.y; }
  if constexpr (q == 3) { c.x = b.y; c.y = -b.x; }
  return c;
}

template <int DIR, int M, int R>
ITP_HD cfx fx_twc(cfx a) { return fx_rot<DIR * ((M % R) * (48 / R))>(a); }

// Specialised by fft_common.cuh's composite DFTs through this overload.
template <int DIR> struct Dft<3, DIR, cfx> {
  static ITP_HD void run(cfx* a) {
    cfx s, d, m, r;
    s.x = a[1].x + a[2].x; s.y = a[1].y + a[2].y;
    d.x = a[1].x - a[2].x; d.y = a[1].y - a[2].y;
    m.x = a[0].x - (s.x >> 1);
    m.y = a[0].y - (s.y >> 1);
    a[0].x += s.x; a[0].y += s.y;
    r.x = -DIR * fx_cos12(d.y);
    r.y = DIR * fx_cos12(d.x);
    a[1].x = m.x + r.x; a[1].y = m.y + r.y;
    a[2].x = m.x - r.x; a[2].y = m.y - r.y;
  }
};

// Table entry of a twiddle w = (re, im): each component c as
// c 2^29 = h + l 2^-32, |l| < 2^31, in the four words (re.h, re.l, im.h, im.l)
// that a 16-byte table slot holds.  a * w / 8 (conj: a * conj(w) / 8), rounded,
// for |a.x|, |a.y| < 2^62.
struct __align__(16) fx_tw { int rh, rl, ih, il; };

template <bool CONJ>
ITP_HD cfx fx_cmul(cfx a, fx_tw w) {
  const int xh = fx_hi(a.x), yh = fx_hi(a.y);
  const int xl = (int)(fx_lo(a.x) >> 1), yl = (int)(fx_lo(a.y) >> 1);
  const int ph = CONJ ? -w.ih : w.ih, pl = CONJ ? -w.il : w.il;
  const int nh = CONJ ? w.ih : -w.ih, nl = CONJ ? w.il : -w.il;
  cfx r;
  long long c = fx_wide(xl, 2 * w.rh, 1LL << 31);
  c = fx_wide(xh, w.rl, c);
  c = fx_wide(yl, 2 * nh, c);
  c = fx_wide(yh, nl, c);
  r.x = fx_wide(yh, nh, fx_wide(xh, w.rh, c >> 32));
  c = fx_wide(xl, 2 * ph, 1LL << 31);
  c = fx_wide(xh, pl, c);
  c = fx_wide(yl, 2 * w.rh, c);
  c = fx_wide(yh, w.rl, c);
  r.y = fx_wide(yh, w.rh, fx_wide(xh, ph, c >> 32));
  return r;
}

// v * m for the mantissa 1 <= m < 2 of the positive double f (|v| < 2^61.5);
// *e receives the exponent of f, 0 (and the product 0) for f = 0 or
// subnormal, and 2047 for infinity or NaN.  The sign of f is ignored: the
// passes' factors are exponentials, |k|^2 and their products.
ITP_HD long long fx_mulf(long long v, double f, int* e) {
  const long long b = fx_bits(f);
  const unsigned bh = (unsigned)(b >> 32), bl = (unsigned)b;
  *e = (int)((bh >> 20) & 0x7ffu);
  const unsigned m30 = (((bh & 0xfffffu) | 0x100000u) << 9) | (bl >> 23);   // m 2^29, integer part
  const int ml = (int)((bl << 8) & 0x7fffffffu);                            // fraction in 2^-31
  const int xh = fx_hi(v);
  long long c = fx_wideu(fx_lo(v), m30, 0);
  c = fx_wide(2 * xh, ml, c);
  const long long y = fx_wide(xh, (int)m30, c >> 32);   // v m / 8, the next 32 bits in c
  const long long r = fx_shl(y, 3) | (long long)((unsigned)c >> 29);
  return *e ? r : 0;
}

// The double nearest to v * 2^(e - kFxBias) (round half up; subnormal results
// are zero), NaN for a poisoned exponent.
ITP_HD double fx_to_double(long long v, int e) {
  const long long s = v >> 63;
  unsigned long long a = (unsigned long long)((v ^ s) - s);
  const unsigned ah = (unsigned)(a >> 32), al = (unsigned)a;
  const int z = ah ? fx_clz(ah) : 32 + fx_clz(al);
  a <<= (z & 63);
  const long long q = (long long)(a >> 11) + (long long)((a >> 10) & 1ull);
  int be = 1023 + 63 - z + e - kFxBias;      // biased exponent before the rounding carry
  const bool zero = v == 0 || be <= 0;
  const bool inf = be >= 2047;
  be = zero || inf ? 1 : be;
  long long r = q + ((long long)(be - 1) << 52);
  if (inf) r = 0x7ff0000000000000LL;
  if (zero) r = 0;
  r |= s & (long long)0x8000000000000000ULL;
  if (e >= kFxPoison) r = 0x7ff8000000000000LL;
  return fx_from_bits(r);
}

// ---- vectors -------------------------------------------------------------------
// The N complex values that one thread works on together.  FP32: just the
// values.  FP64: fixed point with one exponent; `v` holds packed values
// before open() and after close(), and components of value
// v * 2^(e - kFxBias), below 2^57, in between.
template <typename S, int N> struct SVec;

template <int N> struct SVec<float2, N> {
  float2 v[N];
  static constexpr bool fixed = false;
  template <int EXTRA = 0> __device__ __forceinline__ void open() {}
  __device__ __forceinline__ void close() {}
  template <int DIR> __device__ __forceinline__ void dft() { Dft<N, DIR, float2>::run(v); }
};

template <int N> struct SVec<cfx, N> {
  cfx v[N];
  int e;
  static constexpr bool fixed = true;

  // Unpack: align to the largest exponent; EXTRA more bits of headroom.
  template <int EXTRA = 0>
  ITP_HD void open() {
    int em = 0;
    int ei[N];
#pragma unroll
    for (int i = 0; i < N; ++i) {
      ei[i] = (int)((fx_lo(v[i].x) & 63u) + ((fx_lo(v[i].y) & 63u) << 6));
      em = fx_max(em, ei[i]);
    }
    const int top = em + kFxDrop + EXTRA;
#pragma unroll
    for (int i = 0; i < N; ++i) {
      const int s = top - ei[i];
      v[i].x = fx_shr(v[i].x, s);
      v[i].y = fx_shr(v[i].y, s);
    }
    e = em == kFxTop ? kFxPoison : top;
  }

  // Small DFT of freshly opened values: the half units that open() took off
  // each input belong to output 0.
  template <int DIR>
  ITP_HD void dft() {
    Dft<N, DIR, cfx>::run(v);
    v[0].x += N / 2;
    v[0].y += N / 2;
  }

  // Largest components, as a high word: all |v| < (returned + 1) 2^32.
  ITP_HD int top_word() const {
    int mx = 0, mn = -1;
#pragma unroll
    for (int i = 0; i < N; ++i) {
      mx = fx_max(mx, fx_max(fx_hi(v[i].x), fx_hi(v[i].y)));
      mn = fx_min(mn, fx_min(fx_hi(v[i].x), fx_hi(v[i].y)));
    }
    return fx_max(mx, ~mn);
  }

  // Pack: scale up to fill the components, put the exponent at the bottom.
  ITP_HD void close() {
    const int n = fx_clz((unsigned)top_word()) - 1;
    int es = e - n;
    if (e >= kFxTop) es = kFxTop;
    const unsigned p = es < 0 ? 0u : 1u << n;   // zero below the exponent range
    es = fx_max(es, 0);
    const unsigned ex = (unsigned)es & 63u, ey = (unsigned)es >> 6;
#pragma unroll
    for (int i = 0; i < N; ++i) {
      const long long x = fx_mulp(v[i].x, p), y = fx_mulp(v[i].y, p);
      v[i].x = (x & ~63LL) | (long long)ex;
      v[i].y = (y & ~63LL) | (long long)ey;
    }
  }

  // Multiply component pairs by factors f (x by f.x, y by f.y).
  ITP_HD void mul_pairs(const double2 (&f)[N]) {
    int em = 0, ex[N], ey[N];
#pragma unroll
    for (int i = 0; i < N; ++i) {
      v[i].x = fx_mulf(v[i].x, f[i].x, &ex[i]);
      v[i].y = fx_mulf(v[i].y, f[i].y, &ey[i]);
      em = fx_max(em, fx_max(ex[i], ey[i]));
    }
    rescale(em, ex, ey);
  }
  // Multiply value i by the real factor f[i].
  ITP_HD void mul_real(const double (&f)[N]) {
    int em = 0, ei[N];
#pragma unroll
    for (int i = 0; i < N; ++i) {
      v[i].x = fx_mulf(v[i].x, f[i], &ei[i]);
      v[i].y = fx_mulf(v[i].y, f[i], &ei[i]);
      em = fx_max(em, ei[i]);
    }
    rescale(em, ei, ei);
  }

  // From real pairs in FP64 (p = value pairs, times f if HASF), ready for a
  // DFT without open().
  template <bool HASF>
  ITP_HD void from_pairs(const double2 (&p)[N], const double2 (&f)[N]) {
    int em = 0, big = 0, ex[N], ey[N];
#pragma unroll
    for (int i = 0; i < N; ++i) {
      v[i].x = from_double<HASF>(p[i].x, f[i].x, &ex[i], &big);
      v[i].y = from_double<HASF>(p[i].y, f[i].y, &ey[i], &big);
      em = fx_max(em, fx_max(ex[i], ey[i]));
    }
    // components below 2^61 (2^62 after the product): 4 or 5 bits down
    constexpr int kDown = HASF ? 5 : 4;
#pragma unroll
    for (int i = 0; i < N; ++i) {
      v[i].x = fx_shr(v[i].x, em - ex[i] + kDown);
      v[i].y = fx_shr(v[i].y, em - ey[i] + kDown);
    }
    // a double is mant 2^(ex - 1023 - 52), here mant 2^8
    e = em - 1023 - 52 - 8 + kDown + kFxBias + (HASF ? -1023 : 0);
    if (em == 0) e = 0;   // all zero
    if (big == 2047) e = kFxPoison;
  }

  // value component w of element i, times the positive f, as a double
  ITP_HD double to_double_times(long long w, double f) const {
    int ef;
    const long long y = fx_mulf(w, f, &ef);
    return fx_to_double(y, e >= kFxPoison || ef == 2047 ? kFxPoison : e + ef - 1023);
  }
  ITP_HD double to_double(long long w) const { return fx_to_double(w, e); }

 private:
  // Products with factors of exponents ex, ey (the largest em): align them
  // and bring the components below 2^57 again, in one shift.
  ITP_HD void rescale(int em, const int (&ex)[N], const int (&ey)[N]) {
    int mx = 0, mn = -1;
#pragma unroll
    for (int i = 0; i < N; ++i) {
      const int hx = fx_hi(v[i].x) >> fx_min(em - ex[i], 31), hy = fx_hi(v[i].y) >> fx_min(em - ey[i], 31);
      mx = fx_max(mx, fx_max(hx, hy));
      mn = fx_min(mn, fx_min(hx, hy));
    }
    const int r = fx_max(0, 7 - fx_clz((unsigned)fx_max(mx, ~mn)));
#pragma unroll
    for (int i = 0; i < N; ++i) {
      v[i].x = fx_shr(v[i].x, em - ex[i] + r);
      v[i].y = fx_shr(v[i].y, em - ey[i] + r);
    }
    e = e >= kFxPoison || em == 2047 ? kFxPoison : e + em - 1023 + r;
  }
  template <bool HASF>
  static ITP_HD long long from_double(double p, double f, int* e, int* big) {
    const long long b = fx_bits(p);
    const int ep = (int)((b >> 52) & 0x7ff);
    long long m = ((b & 0xfffffffffffffLL) | 0x10000000000000LL) << 8;
    const long long s = b >> 63;
    m = (m ^ s) - s;
    *big = fx_max(*big, ep);
    *e = ep;
    if (ep == 0) m = 0;
    if constexpr (HASF) {
      int ef;
      m = fx_mulf(m, f, &ef);
      *big = fx_max(*big, ef);
      *e = (ep == 0 || ef == 0) ? 0 : ep + ef;
    }
    return m;
  }
};

// a[j] *= w^(q j) (CONJ: w^(-q j)) from the table of roots, all values over 8.
template <bool CONJ, int N>
ITP_HD void fx_twiddle(SVec<cfx, N>& a, const fx_tw* tw, int q) {
#pragma unroll
  for (int j = 1; j < N; ++j) a.v[j] = fx_cmul<CONJ>(a.v[j], tw[q * j]);
  a.v[0].x >>= 3;
  a.v[0].y >>= 3;
  a.e += 3;
}

}  // namespace itp
