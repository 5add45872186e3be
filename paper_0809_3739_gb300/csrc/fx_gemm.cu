// FP64 contractions over the grid: the overlap and the subspace matrix (Gram),
// and the update by an m x m matrix.
//
// The FP64 form of these kernels was bound by the FP64 pipe, one instruction
// per 78 cycles and sub-partition (128 states at 128^3: 65 ms per Gram matrix,
// 58 ms per update, and the Gram computed 128 x 128 products however few the
// states).  So the operands are scaled to integers of 55 or 56 bits.
//
// Up to 32 states they are split into two signed halves v = h 2^28 + l, and a
// product is h h', h l' + l h' and l l', accumulated exactly in 64-bit integers
// over up to 512 terms: a 32 x 32 + 64-bit multiply-add (IMAD.WIDE) issues
// every 3.2 cycles with general operands (every 2 in a chain).  More states have enough products per element to pay
// for splitting it into base-256 digits: the tensor cores multiply those
// exactly (128 states at 64^3, an eighth of those points: 0.76 and 0.81 ms).
#include <cuda_fp16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "fft_fixed.cuh"
#include "itp_kernels.cuh"

namespace itp {

namespace {

constexpr int kMaxM = 256;   // states of the n x n work at most
constexpr int kHalf = 28;    // bits of the lower half

// The double d as an integer of scale 2^(BITS - 1) at the biased exponent e
// (|d| < 2^(e - 1022)): |result| <= 2^BITS, rounded to nearest, 0 for
// subnormal d; to_halves: as halves (h, l) with l in [-2^27, 2^27).
template <int BITS>
__device__ __forceinline__ long long to_integer(double d, int e) {
  const long long b = __double_as_longlong(d);
  const int ex = (int)((b >> 52) & 0x7ff);
  // the 53-bit mantissa, shifted so that one more bit than wanted is left
  constexpr int kUp = BITS + 1 - 53;
  static_assert(kUp >= 1 && kUp <= 9, "54 to 61 bits");
  long long m = fx_shr(((b & 0xfffffffffffffLL) | 0x10000000000000LL) << kUp, fx_max(0, e - ex));
  m = ex == 0 ? 0 : (m + 1) >> 1;   // (the magnitude: no bias towards or from zero)
  const long long sg = b >> 63;
  return (m ^ sg) - sg;
}
template <int BITS>
__device__ __forceinline__ int2 to_halves(double d, int e) {
  const long long m = to_integer<BITS>(d, e);
  int2 r;
  r.x = (int)((m + (1LL << (kHalf - 1))) >> kHalf);
  r.y = (int)((unsigned)m << (32 - kHalf)) >> (32 - kHalf);
  return r;
}
// Biased exponent of |d| (0: zero or subnormal, 2047: not finite).
__device__ __forceinline__ int exponent(double d) {
  return (__double2hiint(d) >> 20) & 0x7ff;
}
// The same of d 2^x: kNone for zero or subnormal d, kNotFinite for infinity
// and NaN.
constexpr int kNone = -(1 << 16), kNotFinite = 1 << 16;
__device__ __forceinline__ int scaled_exponent(double d, int x) {
  const int e = exponent(d);
  return e == 0 ? kNone : (e == 2047 ? kNotFinite : e + x);
}
// 2^k as a double, k clamped to the normal range
__device__ __forceinline__ double pow2(int k) {
  k = fx_max(-1022, fx_min(1023, k));
  return __longlong_as_double((long long)(k + 1023) << 52);
}
// s * 2^k by the exponent field; in two multiplications where that leaves the
// normal range
__device__ __forceinline__ double scale2(double s, int k) {
  const int e = exponent(s) + k;
  if (e > 0 && e < 2047 && exponent(s) != 0)
    return __hiloint2double(__double2hiint(s) + (k << 20), __double2loint(s));
  return s * pow2(k / 2) * pow2(k - k / 2);
}
// N pairs from shared memory, 16 bytes at a time where N is even (p is then
// 16-byte aligned)
template <int N>
__device__ __forceinline__ void load_pairs(const int2* p, int2 (&v)[N]) {
  if constexpr (N % 2 == 0) {
#pragma unroll
    for (int q = 0; q < N; q += 2) {
      const int4 w = *reinterpret_cast<const int4*>(p + q);
      v[q] = make_int2(w.x, w.y);
      v[q + 1] = make_int2(w.z, w.w);
    }
  } else {
#pragma unroll
    for (int q = 0; q < N; ++q) v[q] = p[q];
  }
}

// ---------------------------------------------------------------------------
// Gram partial sums P[c][i][j] = sum over the points p of chunk c of
// A[i][p] B[j][p], up to 16 TT states (one: A and B are the same).  A CTA of
// 16 x 16 threads sums one chunk, TT x TT entries per thread.  A chunk is
// walked in runs of kRun points: the run's largest exponent of every row first
// (the reads bring the run into L2), then tiles of kTile points converted into
// shared memory as halves, [point][row].
//
// Precision: with the row's largest value in the run scaled to 2^54, an
// element is off by at most 2^-55 of it, with random signs, and the products
// are exact, so a sum is off by less than one FP64 rounding of |A_i| |B_j|
// whatever the states' shape.  l l' is part of that: on the diagonal it is a
// square, and without it every squared norm came out too small, by about 2^-55
// of the run's largest square per point (relative error of S_ii 8e-16 for
// oscillator states on 32^3, 4e-15 for one large value per run with 1e-5 beside
// it; with it 7e-17 and 1e-16, below the FP64 sums' 1.2e-16 and equal to them).
constexpr int kRun = 512;
constexpr int kTile = 16;   // (32 points needed more registers for the tile in flight)
constexpr int kGramBits = 54;
// More states than this: the tensor-core form below.  32 states at 64^3 0.184 ms
// here, 0.218 there; at 24^3 0.019 and 0.023; 16 at 64^3 0.066 and 0.206.  With
// this form extended to 64 states (before l l') 57 at 64^3 took 0.50 ms, 0.24
// there; 48 at 128^3 2.30 and 1.68.
constexpr int kGramMmaMin = 32;

template <int TT>
__global__ void __launch_bounds__(256, 3)
    fx_gram_kernel(const double* __restrict__ A, const double* __restrict__ B, int m, long long N,
                   long long chunk, double* __restrict__ partial, int one) {
  constexpr int ROWS = 16 * TT;            // rows of a tile
  constexpr int PITCH = ROWS + 2;          // 16-byte rows of pairs, few bank conflicts
  __shared__ __align__(16) int2 sA[2][kTile][PITCH];   // two tiles: one barrier per tile
  __shared__ __align__(16) int2 sB[2][kTile][PITCH];
  __shared__ int eA[ROWS], eB[ROWS];
  const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4, lane = tid & 31, warp = tid >> 5;
  const long long p_begin = (long long)blockIdx.x * chunk;
  const long long p_end = p_begin + chunk < N ? p_begin + chunk : N;
  double* out = partial + (long long)blockIdx.x * m * m;
  // this CTA's sums stay in its slice of `partial` (L2) between runs
  auto add_sum = [&](int i, int j, double v, bool first) {
    if (i >= m || j >= m) return;
    if (!first) v += out[i * m + j];
    out[i * m + j] = v;
  };
  if (p_begin >= p_end) {
#pragma unroll
    for (int q = 0; q < TT; ++q)
#pragma unroll
      for (int r = 0; r < TT; ++r) add_sum(ty * TT + q, tx * TT + r, 0.0, true);
  }

  // element q of this thread's share of a tile: point tx, row ty + 16 q
  auto load = [&](const double* X, long long p0, long long pe, double (&v)[TT]) {
#pragma unroll
    for (int q = 0; q < TT; ++q) {
      const int i = ty + 16 * q;
      const long long p = p0 + tx;
      v[q] = (i < m && p < pe) ? X[(long long)i * N + p] : 0.0;
    }
  };
  for (long long run = p_begin; run < p_end; run += kRun) {
    const long long re = run + kRun < p_end ? run + kRun : p_end;
    // largest exponents, one warp per row
    for (int op = 0; op < (one ? 1 : 2); ++op) {
      const double* X = op == 0 ? A : B;
      for (int i = warp; i < ROWS; i += 8) {
        int e = 0;
        if (i < m) {
          const double* row = X + (long long)i * N + run;
#pragma unroll 8
          for (int k = lane; k < (int)(re - run); k += 32) e = fx_max(e, exponent(row[k]));
        }
        e = __reduce_max_sync(0xffffffffu, e);
        if (lane == 0) (op == 0 ? eA : eB)[i] = e;
      }
    }
    __syncthreads();
    long long hh[TT][TT], hl[TT][TT], ll[TT][TT];
#pragma unroll
    for (int q = 0; q < TT; ++q)
#pragma unroll
      for (int r = 0; r < TT; ++r) hh[q][r] = hl[q][r] = ll[q][r] = 0;
    double va[TT], vb[TT];
    load(A, run, re, va);
    if (!one) load(B, run, re, vb);
    auto store = [&](int buf) {
#pragma unroll
      for (int q = 0; q < TT; ++q) {
        const int i = ty + 16 * q;
        sA[buf][tx][i] = to_halves<kGramBits>(va[q], eA[i]);
        if (!one) sB[buf][tx][i] = to_halves<kGramBits>(vb[q], eB[i]);
      }
    };
    store(0);
    const int ntile = (int)((re - run + kTile - 1) / kTile);
    for (int t = 0; t < ntile; ++t) {
      const bool more = t + 1 < ntile;
      if (more) {   // the next tile's loads are in flight meanwhile
        const long long p0 = run + (long long)(t + 1) * kTile;
        load(A, p0, re, va);
        if (!one) load(B, p0, re, vb);
      }
      __syncthreads();
      const int2(*tA)[PITCH] = sA[t & 1];
      const int2(*tB)[PITCH] = one ? sA[t & 1] : sB[t & 1];
#pragma unroll 2
      for (int k = 0; k < kTile; ++k) {
        int2 a[TT], b[TT];
        load_pairs(&tA[k][ty * TT], a);
        load_pairs(&tB[k][tx * TT], b);
#pragma unroll
        for (int q = 0; q < TT; ++q)
#pragma unroll
          for (int r = 0; r < TT; ++r)
            hh[q][r] = fx_wide(a[q].x, b[r].x, hh[q][r]);   // <= 512 * 2^52
#pragma unroll
        for (int q = 0; q < TT; ++q)
#pragma unroll
          for (int r = 0; r < TT; ++r)
            hl[q][r] = fx_wide(a[q].x, b[r].y, hl[q][r]);   // <= 256 * 2^54, see below
#pragma unroll
        for (int q = 0; q < TT; ++q)
#pragma unroll
          for (int r = 0; r < TT; ++r) {
            hl[q][r] = fx_wide(a[q].y, b[r].x, hl[q][r]);
            ll[q][r] = fx_wide(a[q].y, b[r].y, ll[q][r]);   // <= 256 * 2^54
          }
      }
      if (more) store((t + 1) & 1);
      if ((t + 1) * kTile == kRun / 2) {   // keep the lower sums within 64 bits
#pragma unroll
        for (int q = 0; q < TT; ++q)
#pragma unroll
          for (int r = 0; r < TT; ++r) {
            hl[q][r] += ll[q][r] >> kHalf;
            ll[q][r] &= (1LL << kHalf) - 1;
            hh[q][r] += hl[q][r] >> kHalf;
            hl[q][r] &= (1LL << kHalf) - 1;
          }
      }
    }
    // the run's sums to FP64: (hh 2^56 + hl 2^28 + ll) 2^(ea + eb - 2 * (1022 + 54))
#pragma unroll
    for (int q = 0; q < TT; ++q) {
      const int ea = eA[ty * TT + q];
#pragma unroll
      for (int r = 0; r < TT; ++r) {
        const int eb = (one ? eA : eB)[tx * TT + r];
        const long long mid = hl[q][r] + (ll[q][r] >> kHalf);
        const double s = fma((double)hh[q][r], (double)(1LL << kHalf), (double)mid);
        double v = scale2(s, ea + eb - 2 * (1022 + kGramBits) + kHalf);
        if (ea == 2047 || eb == 2047) v = __longlong_as_double(0x7ff8000000000000LL);
        add_sum(ty * TT + q, tx * TT + r, v, run == p_begin);
      }
    }
    __syncthreads();   // the exponents are rewritten by the next run
  }
}

// ---------------------------------------------------------------------------
// The same sums for more than kGramMmaMin states on the tensor cores: elements
// as 55-bit integers in seven signed base-256 digits d_0 .. d_6, each exact in
// FP16; the products of digits a and b belong to level a + b, and the levels
// 0 .. 6 (28 digit products per element product) are accumulated apart, in
// FP32: up to 7 * 128 products of at most 2^14 stay below 2^24, so the sums
// over 128 points are exact whatever the rounding.  They are then moved to
// 64-bit integers in shared memory (levels 0-3 and 4-6), and the run's sums to
// FP64.  The levels above 6 left out are about 2^-56 of the two largest values
// per product, with random signs (squares start at level 8), which is below
// the rounding of an FP64 sum: squared norms of 33 and 64 rows off by 4e-16 at
// most for smooth, random and decaying rows (FP64 sums 3e-15 to 1.2e-14), and by
// 3.5e-15 for one large value and 1e-4 beside it (FP64 sums 1.6e-14).
//
// mma.sync reaches 1000 FMAs per clock and SM here, a quarter of tcgen05, but
// its sums are in registers: the seven accumulators of a 128 x 128 tile would
// not fit TMEM, and would have to be read back every 128 points.  A CTA
// of 16 warps sums a 64 x 64 block, 16 x 16 per warp.  (Against the IMAD.WIDE
// form, 3.2 cycles per multiply-add: see kGramMmaMin.)
constexpr int kMmaThreads = 512;
constexpr int kMmaRows = 64;             // rows and columns of a block
constexpr int kMmaTile = 32;             // points per tile
constexpr int kMmaPitch = kMmaTile + 8;  // halves; rows 80 bytes apart: conflict-free ldmatrix
constexpr int kDigits = 7;
constexpr int kMmaBits = 55;
constexpr int kMmaDrain = 128 / kMmaTile;   // tiles between drains
constexpr size_t kMmaOperand = (size_t)kDigits * kMmaRows * kMmaPitch;   // halves
constexpr size_t kMmaSmem = 2 * 2 * kMmaOperand * 2 + (size_t)16 * kMmaThreads * 8;

__device__ __forceinline__ void ldmatrix4(uint32_t (&r)[4], uint32_t addr) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"(addr)
               : "memory");
}
__device__ __forceinline__ void mma_f16(float (&c)[4], const uint32_t (&a)[4], uint32_t b0,
                                        uint32_t b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3},{%4,%5,%6,%7},{%8,%9},"
      "{%0,%1,%2,%3};"
      : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}
// Two FP16 digits from 10-bit fields u = digit + 128 in the halves of x: FP16
// 1024 + u has the bits 0x6400 + u.
__device__ __forceinline__ uint32_t digits_f16(uint32_t x, uint32_t mask) {
  uint32_t r = (x & mask) | 0x64006400u;
  asm("add.f16x2 %0, %0, %1;" : "+r"(r) : "r"(0xe480e480u));   // - 1152
  return r;
}
// The digits of two integers: pair l = (digit l of v0, digit l of v1).
__device__ __forceinline__ void digit_pairs(long long v0, long long v1, uint32_t (&d)[kDigits]) {
  constexpr long long kBias = 0x0080808080808080LL;   // every digit + 128, no borrows
  v0 += kBias;
  v1 += kBias;
  const uint32_t l0 = (uint32_t)v0, h0 = (uint32_t)(v0 >> 32);
  const uint32_t l1 = (uint32_t)v1, h1 = (uint32_t)(v1 >> 32);
  d[0] = digits_f16(__byte_perm(h0, h1, 0x7632), 0x01ff01ffu);
  d[1] = digits_f16(__byte_perm(h0, h1, 0x0501), 0x00ff00ffu);
  d[2] = digits_f16(__byte_perm(h0, h1, 0x0400), 0x00ff00ffu);
  d[3] = digits_f16(__byte_perm(l0, l1, 0x0703), 0x00ff00ffu);
  d[4] = digits_f16(__byte_perm(l0, l1, 0x0602), 0x00ff00ffu);
  d[5] = digits_f16(__byte_perm(l0, l1, 0x0501), 0x00ff00ffu);
  d[6] = digits_f16(__byte_perm(l0, l1, 0x0400), 0x00ff00ffu);
}

// (bi, bj) of the blocks, packed as bi * 256 + bj.
struct GramBlocks {
  int n;
  short ij[64];
};

__global__ void __launch_bounds__(kMmaThreads, 1)
    fx_gram_mma_kernel(const double* __restrict__ A, const double* __restrict__ B, int m,
                       long long N, long long chunk, double* __restrict__ partial,
                       const GramBlocks blocks, int same) {
  extern __shared__ __align__(16) unsigned char smraw[];
  __half* sD = reinterpret_cast<__half*>(smraw);   // [2 buffers][2 operands][digit][row][pitch]
  long long* sacc = reinterpret_cast<long long*>(smraw + 2 * 2 * kMmaOperand * 2);   // [16][tid]
  __shared__ int eA[kMmaRows], eB[kMmaRows];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int bi = blocks.ij[blockIdx.y] >> 8, bj = blocks.ij[blockIdx.y] & 255;
  const bool one = same && bi == bj;       // a diagonal block: one operand
  const int ia = kMmaRows * bi, jb = kMmaRows * bj;
  const long long p_begin = (long long)blockIdx.x * chunk;
  const long long p_end = p_begin + chunk < N ? p_begin + chunk : N;
  double* out = partial + (long long)blockIdx.x * m * m;
  // this warp's 16 x 16 part, and this thread's entry c of its column tile n
  const int wi = 16 * (warp >> 2), wj = 16 * (warp & 3);
  auto row_of = [&](int c) { return wi + (lane >> 2) + 8 * (c >> 1); };
  auto col_of = [&](int n, int c) { return wj + 8 * n + 2 * (lane & 3) + (c & 1); };
  auto add_sum = [&](int i, int j, double v, bool first) {
    if (i >= m || j >= m) return;
    if (!first) v += out[i * m + j];
    out[i * m + j] = v;
    if (same && bi != bj) out[j * m + i] = v;
  };
  if (p_begin >= p_end) {
    for (int q = 0; q < 8; ++q) add_sum(ia + row_of(q & 3), jb + col_of(q >> 2, q & 3), 0.0, true);
    return;
  }
  // ldmatrix addresses: A 16 rows x 16 points, B 16 columns x 16 points
  const uint32_t base = (uint32_t)__cvta_generic_to_shared(sD);
  const uint32_t offA = (uint32_t)(((wi + (lane & 7) + 8 * ((lane >> 3) & 1)) * kMmaPitch +
                                    8 * (lane >> 4)) * 2);
  const uint32_t offB = (uint32_t)(((wj + (lane & 7) + 8 * (lane >> 4)) * kMmaPitch +
                                    8 * ((lane >> 3) & 1)) * 2);
  constexpr uint32_t kSlice = kMmaRows * kMmaPitch * 2, kOp = kMmaOperand * 2;
  const int lr = tid >> 3, lp = 4 * (tid & 7);   // tile load: row, first of four points
  double va[4], vb[4];
  auto load = [&](const double* X, int r0, long long p0, long long pe, double (&v)[4]) {
    const double* src = X + (long long)(r0 + lr) * N + p0 + lp;
#pragma unroll
    for (int q = 0; q < 4; ++q) v[q] = (r0 + lr < m && p0 + lp + q < pe) ? src[q] : 0.0;
  };
  auto store = [&](int buf, int op, const double (&v)[4], int e) {
    uint32_t d0[kDigits], d1[kDigits];
    digit_pairs(to_integer<kMmaBits>(v[0], e), to_integer<kMmaBits>(v[1], e), d0);
    digit_pairs(to_integer<kMmaBits>(v[2], e), to_integer<kMmaBits>(v[3], e), d1);
    __half* dst = sD + (size_t)(buf * 2 + op) * kMmaOperand + lr * kMmaPitch + lp;
#pragma unroll
    for (int l = 0; l < kDigits; ++l)
      *reinterpret_cast<uint2*>(dst + (size_t)l * kMmaRows * kMmaPitch) = make_uint2(d0[l], d1[l]);
  };
  for (long long run = p_begin; run < p_end; run += kRun) {
    const long long re = run + kRun < p_end ? run + kRun : p_end;
    for (int op = 0; op < (one ? 1 : 2); ++op) {   // largest exponents, one warp per row
      const double* X = op == 0 ? A : B;
      const int r0 = op == 0 ? ia : jb;
      for (int i = warp; i < kMmaRows; i += kMmaThreads / 32) {
        int e = 0;
        if (r0 + i < m) {
          const double* row = X + (long long)(r0 + i) * N + run;
#pragma unroll 8
          for (int k = lane; k < (int)(re - run); k += 32) e = fx_max(e, exponent(row[k]));
        }
        e = __reduce_max_sync(0xffffffffu, e);
        if (lane == 0) (op == 0 ? eA : eB)[i] = e;
      }
    }
    load(A, ia, run, re, va);
    if (!one) load(B, jb, run, re, vb);
#pragma unroll
    for (int q = 0; q < 16; ++q) sacc[q * kMmaThreads + tid] = 0;
    __syncthreads();
    store(0, 0, va, eA[lr]);
    if (!one) store(0, 1, vb, eB[lr]);
    float acc[kDigits][2][4];
#pragma unroll
    for (int l = 0; l < kDigits; ++l)
#pragma unroll
      for (int n = 0; n < 2; ++n)
#pragma unroll
        for (int c = 0; c < 4; ++c) acc[l][n][c] = 0.f;
    const int ntile = (int)((re - run + kMmaTile - 1) / kMmaTile);
    for (int t = 0; t < ntile; ++t) {
      const bool more = t + 1 < ntile;
      if (more) {   // the next tile's loads are in flight meanwhile
        const long long p0 = run + (long long)(t + 1) * kMmaTile;
        load(A, ia, p0, re, va);
        if (!one) load(B, jb, p0, re, vb);
      }
      __syncthreads();
      const uint32_t tA = base + (uint32_t)(t & 1) * 2 * kOp + offA;
      const uint32_t tB = base + (uint32_t)(t & 1) * 2 * kOp + (one ? 0 : kOp) + offB;
#pragma unroll 1
      for (int k = 0; k < kMmaTile; k += 16) {
        uint32_t b[kDigits][4];
#pragma unroll
        for (int l = 0; l < kDigits; ++l) ldmatrix4(b[l], tB + l * kSlice + 2 * k);
#pragma unroll
        for (int l = 0; l < kDigits; ++l) {
          uint32_t a[4];
          ldmatrix4(a, tA + l * kSlice + 2 * k);
#pragma unroll
          for (int q = 0; q + l < kDigits; ++q) {
            mma_f16(acc[l + q][0], a, b[q][0], b[q][1]);
            mma_f16(acc[l + q][1], a, b[q][2], b[q][3]);
          }
        }
      }
      if (more) {
        store((t + 1) & 1, 0, va, eA[lr]);
        if (!one) store((t + 1) & 1, 1, vb, eB[lr]);
      }
      if (!more || (t + 1) % kMmaDrain == 0) {
#pragma unroll
        for (int n = 0; n < 2; ++n)
#pragma unroll
          for (int c = 0; c < 4; ++c) {
            int v[kDigits];
#pragma unroll
            for (int l = 0; l < kDigits; ++l) {
              v[l] = __float2int_rn(acc[l][n][c]);
              acc[l][n][c] = 0.f;
            }
            const int q = n * 4 + c;
            long long hi = sacc[q * kMmaThreads + tid], lo = sacc[(8 + q) * kMmaThreads + tid];
            hi += fx_wide(v[0], 1 << 24, fx_wide(v[1], 1 << 16, fx_wide(v[2], 1 << 8, v[3])));
            lo += fx_wide(v[4], 1 << 16, fx_wide(v[5], 1 << 8, v[6]));
            sacc[q * kMmaThreads + tid] = hi;
            sacc[(8 + q) * kMmaThreads + tid] = lo;
          }
      }
    }
    // (hi 2^72 + lo 2^48) 2^(ea + eb - 2 * (1022 + 55))
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      const int i = row_of(q & 3), j = col_of(q >> 2, q & 3);
      const int ea = eA[i], eb = (one ? eA : eB)[j];
      const double sum = fma((double)sacc[q * kMmaThreads + tid], (double)(1 << 24),
                             (double)sacc[(8 + q) * kMmaThreads + tid]);
      double v = scale2(sum, ea + eb - 2 * (1022 + kMmaBits) + 48);
      if (ea == 2047 || eb == 2047) v = __longlong_as_double(0x7ff8000000000000LL);
      add_sum(ia + i, jb + j, v, run == p_begin);
    }
    __syncthreads();   // the exponents and buffers are rewritten by the next run
  }
}

// ---------------------------------------------------------------------------
// Y[i] = sum_k M[i][k] X[k], up to 4 RG states.  Persistent CTAs of 512
// threads over tiles of PT = 1024 / RG points.  State k is scaled by the power
// of two nearest to its norm, from the diagonal of its overlap matrix S (null:
// all states of norm one), and column k of M by the inverse; the rows of that
// M, scaled by their largest entry to 55 bits, stay in shared memory as halves
// [k][i]; a tile of X, each point scaled by its largest value over the states,
// comes as halves [k][point] into one of two buffers while the other one is
// multiplied (one barrier per tile).  A thread holds 4 rows x 2 points.
// lower: M[i][k] = 0 for k > i, so a row group stops there.
//
// Precision: products are exact in 110 bits, so a sum is off by the rounding
// of its operands, 2^-56 of the largest |M_ik| times the point's largest
// |X_k| (both scaled) per term with random signs, and the rounding to a double.
// In the norm of a state that is below an FP64 sum's 2^-53 of the largest
// |M_ik X_k|.  It is not value by value: where a state is in its tail, another
// one is large and their M_ik is small, the FP64 sum's error was as small as
// the tail, this one's is 2^-56 of the other state's size there (and smaller
// values come out as zero).
constexpr int kApplyBits = 55;
constexpr int kApplyThreads = 512;

// hh 2^56 + hl 2^28 + ll as a double, times 2^k (k far below: 0; poison: NaN).
__device__ __forceinline__ double sum_to_double(long long hh, long long hl, long long ll, int k,
                                                bool poison) {
  const long long mid = hl + (ll >> kHalf);
  const long long top = hh + (mid >> kHalf);   // value = (top + low 2^-32) 2^56
  unsigned w2 = (unsigned)(top >> 32), w1 = (unsigned)top, w0 = (unsigned)mid << (32 - kHalf);
  const unsigned s = (unsigned)((int)w2 >> 31);
  w2 ^= s;   // magnitude, to one unit of 2^24
  w1 ^= s;
  w0 ^= s;
  const bool far = w2 == 0;   // cancelled by 2^-32 or more: the lower words
  const int z = __clz(far ? w1 : w2);
  const unsigned hi = __funnelshift_l(far ? w0 : w1, far ? w1 : w2, z);
  const unsigned lo = __funnelshift_l(far ? 0u : w0, far ? w0 : w1, z);
  // hi:lo is normalised (bit 63 set) unless the value is zero
  const unsigned long long m = ((unsigned long long)hi << 32) | lo;
  const long long q = (long long)(m >> 11) + (long long)((m >> 10) & 1ull);
  const int be = 1023 + 56 + 63 - z - (far ? 32 : 0) + k;
  double r = be > 0 && be < 2047 ? __longlong_as_double(q + ((long long)(be - 1) << 52))
                                 : (be >= 2047 ? __longlong_as_double(0x7ff0000000000000LL) : 0.0);
  if (hi == 0) r = 0.0;
  if (poison) r = __longlong_as_double(0x7ff8000000000000LL);
  return s ? -r : r;
}

template <int RG>
__global__ void __launch_bounds__(kApplyThreads)
    fx_apply_kernel(const double* __restrict__ M, int m, int lower, const double* __restrict__ S,
                    const double* __restrict__ X, double* __restrict__ Y, long long N) {
  constexpr int NP = 2;                           // points per thread
  constexpr int ROWS = 4 * RG, TX = kApplyThreads / RG, PT = NP * TX;
  constexpr int MP = ROWS + 2;                    // pitch of sM (16-byte rows)
  constexpr int STEP = kApplyThreads / PT;        // threads per point of a tile load
  constexpr int PER = ROWS / STEP;
  static_assert(PT <= 256 && STEP >= 2, "four row groups at least");
  extern __shared__ __align__(16) unsigned char smraw[];
  int2* sM = reinterpret_cast<int2*>(smraw);      // [ROWS k][MP]
  int2* sX = sM + ROWS * MP;                      // [2][ROWS k][PT]
  int* eM = reinterpret_cast<int*>(sX + 2 * ROWS * PT);   // [ROWS]
  int* xs = eM + ROWS;                            // [ROWS] scales of the states
  int* eX = xs + ROWS;                            // [3][STEP][PT]: tile t in slot t % 3, as
                                                  // slower warps still read tile t - 1's
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int ty = tid / TX, tx = tid - ty * TX;    // row group, point
  for (int k = tid; k < ROWS; k += kApplyThreads) {
    const int e = S && k < m ? exponent(S[(long long)k * (m + 1)]) : 0;
    xs[k] = e > 0 && e < 2047 ? (e - 1023) >> 1 : 0;
  }
  __syncthreads();
  for (int i = warp; i < ROWS; i += kApplyThreads / 32) {
    int e = kNone;
    if (i < m)
      for (int k = lane; k < m; k += 32) e = fx_max(e, scaled_exponent(M[i * m + k], xs[k]));
    e = __reduce_max_sync(0xffffffffu, e);
    if (lane == 0) eM[i] = e;
    for (int k = lane; k < ROWS; k += 32)
      sM[k * MP + i] = i < m && k < m ? to_halves<kApplyBits>(M[i * m + k], e - xs[k])
                                      : make_int2(0, 0);
  }
  const long long ntiles = (N + PT - 1) / PT;
  const int lp = tid & (PT - 1), lk = tid / PT;   // tile load: point, first state
  double v[PER];
  auto load = [&](long long tile) {
    const long long p = tile * PT + lp;
#pragma unroll
    for (int q = 0; q < PER; ++q) {
      const int k = lk + STEP * q;
      v[q] = (tile < ntiles && k < m && p < N) ? X[(long long)k * N + p] : 0.0;
    }
  };
  auto put_exponent = [&](int slot) {
    int e = kNone;
#pragma unroll
    for (int q = 0; q < PER; ++q) e = fx_max(e, scaled_exponent(v[q], -xs[lk + STEP * q]));
    eX[(slot * STEP + lk) * PT + lp] = e;
  };
  auto point_exponent = [&](int slot, int p) {
    int e = kNone;
#pragma unroll
    for (int s = 0; s < STEP; ++s) e = fx_max(e, eX[(slot * STEP + s) * PT + p]);
    return e;
  };
  auto convert = [&](int buf, int slot) {
    const int e = point_exponent(slot, lp);
#pragma unroll
    for (int q = 0; q < PER; ++q)
      sX[(buf * ROWS + lk + STEP * q) * PT + lp] =
          to_halves<kApplyBits>(v[q], e + xs[lk + STEP * q]);
  };
  load(blockIdx.x);
  put_exponent(0);
  __syncthreads();
  convert(0, 0);
  load((long long)blockIdx.x + gridDim.x);
  const int kmax = lower ? fx_min(m, 4 * ty + 4) : m;
  int buf = 0, slot = 0;
  for (long long tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
    const int next = slot == 2 ? 0 : slot + 1;
    put_exponent(next);
    __syncthreads();   // this tile is stored, the other buffer's last reader done
    convert(buf ^ 1, next);
    load(tile + 2LL * gridDim.x);   // in flight meanwhile
    long long hh[4][NP], hl[4][NP], ll[4][NP];
#pragma unroll
    for (int q = 0; q < 4; ++q)
#pragma unroll
      for (int r = 0; r < NP; ++r) hh[q][r] = hl[q][r] = ll[q][r] = 0;
    const int2* xb = sX + buf * ROWS * PT + tx;
#pragma unroll 4
    for (int k = 0; k < kmax; ++k) {
      int2 a[4], b[NP];
      load_pairs(&sM[k * MP + 4 * ty], a);
#pragma unroll
      for (int r = 0; r < NP; ++r) b[r] = xb[k * PT + TX * r];
#pragma unroll
      for (int q = 0; q < 4; ++q)
#pragma unroll
        for (int r = 0; r < NP; ++r) {   // (128 terms would be <= 2^61, 2^62, 2^61)
          hh[q][r] = fx_wide(a[q].x, b[r].x, hh[q][r]);
          hl[q][r] = fx_wide(a[q].x, b[r].y, hl[q][r]);
          ll[q][r] = fx_wide(a[q].y, b[r].y, ll[q][r]);
        }
#pragma unroll
      for (int q = 0; q < 4; ++q)
#pragma unroll
        for (int r = 0; r < NP; ++r) hl[q][r] = fx_wide(a[q].y, b[r].x, hl[q][r]);
    }
#pragma unroll
    for (int r = 0; r < NP; ++r) {
      const long long p = tile * PT + tx + TX * r;
      if (p >= N) continue;
      const int ex = point_exponent(slot, tx + TX * r);
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const int i = 4 * ty + q;
        if (i >= m) continue;
        const int em = eM[i];
        const double d = sum_to_double(hh[q][r], hl[q][r], ll[q][r],
                                       em + ex - 2 * (1022 + kApplyBits),
                                       em == kNotFinite || ex == kNotFinite);
        Y[(long long)i * N + p] = d;
      }
    }
    buf ^= 1;
    slot = next;
  }
}

// ---------------------------------------------------------------------------
// The update for more than kApplyMmaMin states in the digits of the tensor-
// core Gram: a CTA multiplies 64 rows of M (its digits stay in shared memory)
// with up to 128 states, 32 points per tile; a warp holds 16 rows x 8 points
// in eight FP32 accumulators, exact over the 128 states, and turns each sum
// into a double.  lower: the 16-state steps beyond a warp's rows are skipped.
// Scaling and precision as in the integer form.
// (One level more than the Gram, 34 digit products: a sum over few states has
// no averaging over the grid, and without level 7 its error, about 2^-53 of
// the largest product, was that of the FP64 form instead of below it.)
// 57 states at 64^3 0.40 ms in integers, 0.25 here; 128 1.44 and 0.81; 48 at
// 128^3 2.92 and 1.76; but 32 at 64^3 0.142 and 0.203, at 24^3 0.018 either way.
constexpr int kApplyMmaMin = 32;
constexpr int kApplyMmaPts = 32;
constexpr int kApplyLevels = 8;

// (hi 2^72 + lo 2^40) 2^k as a double, |hi|, |lo| < 2^62.
__device__ __forceinline__ double levels_to_double(long long hi, long long lo, int k, bool poison) {
  return sum_to_double(hi + (lo >> 32), (long long)((unsigned)lo >> (32 - kHalf)), 0, k + 16,
                       poison);   // which takes the two in 2^56 and 2^28
}

__device__ __forceinline__ void ldmatrix2(uint32_t (&r)[2], uint32_t addr) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x2.shared.b16 {%0,%1}, [%2];"
               : "=r"(r[0]), "=r"(r[1])
               : "r"(addr)
               : "memory");
}

__global__ void __launch_bounds__(kMmaThreads, 1)
    fx_apply_mma_kernel(const double* __restrict__ M, int m, int lower,
                        const double* __restrict__ S, const double* __restrict__ X,
                        double* __restrict__ Y, long long N, int k0, int nk, int rb0, int add) {
  extern __shared__ __align__(16) unsigned char smraw[];
  __shared__ int eM[kMmaRows], xs[128], eX[kMmaThreads / 32][kApplyMmaPts], sE[kApplyMmaPts];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int r0 = kMmaRows * (rb0 + blockIdx.y), nr = m - r0 < kMmaRows ? m - r0 : kMmaRows;
  const int kk = lower ? fx_min(nk, r0 + kMmaRows - k0) : nk;   // states used, at most 128
  const int KB = (kk + 63) / 64, K = 64 * KB, pitch = K + 8;
  __half* sM = reinterpret_cast<__half*>(smraw);               // [digit][row][pitch]
  __half* sX = sM + (size_t)kDigits * kMmaRows * pitch;         // [digit][point][pitch]
  if (tid < 128) {
    const int e = S && tid < kk ? exponent(S[(long long)(k0 + tid) * (m + 1)]) : 0;
    xs[tid] = e > 0 && e < 2047 ? (e - 1023) >> 1 : 0;
  }
  __syncthreads();
  for (int i = warp; i < kMmaRows; i += kMmaThreads / 32) {   // rows of M
    const double* row = M + (long long)(r0 + i) * m + k0;
    int e = kNone;
    if (i < nr)
      for (int k = lane; k < kk; k += 32) e = fx_max(e, scaled_exponent(row[k], xs[k]));
    e = __reduce_max_sync(0xffffffffu, e);
    if (lane == 0) eM[i] = e;
    for (int k = 2 * lane; k < K; k += 64) {
      const double v0 = i < nr && k < kk ? row[k] : 0.0, v1 = i < nr && k + 1 < kk ? row[k + 1] : 0.0;
      uint32_t d[kDigits];
      digit_pairs(to_integer<kMmaBits>(v0, e - xs[k]), to_integer<kMmaBits>(v1, e - xs[k + 1]), d);
#pragma unroll
      for (int l = 0; l < kDigits; ++l)
        *reinterpret_cast<uint32_t*>(sM + ((size_t)l * kMmaRows + i) * pitch + k) = d[l];
    }
  }
  const long long ntiles = (N + kApplyMmaPts - 1) / kApplyMmaPts;
  // tile load: point = lane, states 4 warp .. + 3 of each 64
  double v[2][4];
  auto load = [&](long long tile) {
    const long long p = tile * kApplyMmaPts + lane;
#pragma unroll
    for (int b = 0; b < 2; ++b)
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const int k = 64 * b + 4 * warp + q;
        v[b][q] = (tile < ntiles && k < kk && p < N) ? X[(long long)(k0 + k) * N + p] : 0.0;
      }
  };
  const int wi = 16 * (warp >> 2), wp = 8 * (warp & 3);
  int steps = (kk + 15) / 16;   // 16-state steps of this warp's rows
  if (lower) steps = fx_max(0, fx_min(steps, (r0 + wi + 16 - k0 + 15) / 16));
  const uint32_t rowM = kMmaRows * pitch * 2, rowX = kApplyMmaPts * pitch * 2;   // digit strides
  const uint32_t adA = (uint32_t)__cvta_generic_to_shared(sM) +
                       (uint32_t)(((wi + (lane & 7) + 8 * ((lane >> 3) & 1)) * pitch +
                                   8 * (lane >> 4)) * 2);
  const uint32_t adB = (uint32_t)__cvta_generic_to_shared(sX) +
                       (uint32_t)(((wp + (lane & 7)) * pitch + 8 * ((lane >> 3) & 1)) * 2);
  load(blockIdx.x);
  for (long long tile = blockIdx.x; tile < ntiles; tile += gridDim.x) {
    int e = kNone;
#pragma unroll
    for (int b = 0; b < 2; ++b)
#pragma unroll
      for (int q = 0; q < 4; ++q)
        e = fx_max(e, scaled_exponent(v[b][q], -xs[64 * b + 4 * warp + q]));
    eX[warp][lane] = e;
    __syncthreads();   // the previous tile is multiplied, the exponents are here
#pragma unroll
    for (int w = 0; w < kMmaThreads / 32; ++w) e = fx_max(e, eX[w][lane]);
    if (warp == 0) sE[lane] = e;
#pragma unroll
    for (int b = 0; b < 2; ++b) {
      if (b < KB) {
        const int k = 64 * b + 4 * warp;
        long long n[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) n[q] = to_integer<kMmaBits>(v[b][q], e + xs[k + q]);
        uint32_t d0[kDigits], d1[kDigits];
        digit_pairs(n[0], n[1], d0);
        digit_pairs(n[2], n[3], d1);
#pragma unroll
        for (int l = 0; l < kDigits; ++l)
          *reinterpret_cast<uint2*>(sX + ((size_t)l * kApplyMmaPts + lane) * pitch + k) =
              make_uint2(d0[l], d1[l]);
      }
    }
    load(tile + gridDim.x);   // in flight meanwhile
    __syncthreads();
    float acc[kApplyLevels][4];
#pragma unroll
    for (int l = 0; l < kApplyLevels; ++l)
#pragma unroll
      for (int c = 0; c < 4; ++c) acc[l][c] = 0.f;
#pragma unroll 1
    for (int s = 0; s < steps; ++s) {
      uint32_t b[kDigits][2];
#pragma unroll
      for (int l = 0; l < kDigits; ++l) ldmatrix2(b[l], adB + l * rowX + 32 * s);
#pragma unroll
      for (int l = 0; l < kDigits; ++l) {
        uint32_t a[4];
        ldmatrix4(a, adA + l * rowM + 32 * s);
#pragma unroll
        for (int q = 0; q < kDigits && q + l < kApplyLevels; ++q)
          mma_f16(acc[l + q], a, b[q][0], b[q][1]);
      }
    }
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      const int i = wi + (lane >> 2) + 8 * (c >> 1), pt = wp + 2 * (lane & 3) + (c & 1);
      const long long p = tile * kApplyMmaPts + pt;
      if (i < nr && p < N) {
        int u[kApplyLevels];
#pragma unroll
        for (int l = 0; l < kApplyLevels; ++l) u[l] = __float2int_rn(acc[l][c]);
        const long long hi =
            fx_wide(u[0], 1 << 24, fx_wide(u[1], 1 << 16, fx_wide(u[2], 1 << 8, u[3])));
        const long long lo =
            fx_wide(u[4], 1 << 24, fx_wide(u[5], 1 << 16, fx_wide(u[6], 1 << 8, u[7])));
        const int em = eM[i], ex = sE[pt];
        const double d = levels_to_double(hi, lo, em + ex - 2 * (1022 + kMmaBits),
                                          em == kNotFinite || ex == kNotFinite);
        double* y = Y + (long long)(r0 + i) * N + p;
        *y = add ? *y + d : d;
      }
    }
  }
}

template <int RG>
cudaError_t apply_launch(const double* M, int m, int lower, const double* S, const double* X,
                         double* Y, long long N, int sms, cudaStream_t st) {
  constexpr int ROWS = 4 * RG, PT = 2 * kApplyThreads / RG, STEP = kApplyThreads / PT;
  const size_t smem = ((size_t)ROWS * (ROWS + 2) + 2 * (size_t)ROWS * PT) * sizeof(int2) +
                      (2 * (size_t)ROWS + 3 * (size_t)STEP * PT) * sizeof(int);
  cudaError_t e = cudaFuncSetAttribute(fx_apply_kernel<RG>,
                                       cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  const long long ntiles = (N + PT - 1) / PT, cap = 2LL * sms;
  const int grid = (int)(ntiles < cap ? ntiles : cap);
  fx_apply_kernel<RG><<<grid, kApplyThreads, smem, st>>>(M, m, lower, S, X, Y, N);
  return cudaGetLastError();
}

}  // namespace

// The tensor-core form has one CTA per SM: as few chunks as fill them, or a
// multiple where each still has four runs of kRun points or more (a chunk pays
// for a ragged last run and for its m x m sums).  Against 304 chunks always: 37
// states at 72 x 48 x 36 2.10 -> 2.06 ms per step, orthonormalisation of a
// 100 x 250047 block 1.65 -> 1.63 ms.
int gram_chunks(int m, bool same, long long n_points, int most, int sms) {
  if (m <= kGramMmaMin) return most;
  const int nb = (m + kMmaRows - 1) / kMmaRows, blocks = same ? nb * (nb + 1) / 2 : nb * nb;
  int c = sms / blocks > 1 ? sms / blocks : 1;
  for (int w = 2; w * sms / blocks <= most && n_points / (w * sms / blocks) >= 4 * kRun; ++w)
    c = w * sms / blocks;
  return c < most ? c : most;
}

cudaError_t launch_gram_partial(const double* A, const double* B, int m, long long n_points,
                                int n_chunks, double* partial, cudaStream_t st) {
  if (m < 1 || m > kMaxM) return cudaErrorInvalidValue;
  long long chunk = (n_points + n_chunks - 1) / n_chunks;
  chunk = (chunk + kTile - 1) / kTile * kTile;
  if (m > kGramMmaMin) {
    // A A^T: the lower blocks, mirrored
    const bool same = A == B;
    GramBlocks blocks{};
    const int nb = (m + kMmaRows - 1) / kMmaRows;
    chunk = (chunk + kMmaTile - 1) / kMmaTile * kMmaTile;
    for (int bi = 0; bi < nb; ++bi)
      for (int bj = 0; bj < nb; ++bj)
        if (!same || bj <= bi) blocks.ij[blocks.n++] = (short)(bi * 256 + bj);
    cudaError_t e = cudaFuncSetAttribute(fx_gram_mma_kernel,
                                         cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)kMmaSmem);
    if (e != cudaSuccess) return e;
    fx_gram_mma_kernel<<<dim3(n_chunks, blocks.n), kMmaThreads, kMmaSmem, st>>>(
        A, B, m, n_points, chunk, partial, blocks, same);
    return cudaGetLastError();
  }
  if (m <= 16)
    fx_gram_kernel<1><<<n_chunks, 256, 0, st>>>(A, B, m, n_points, chunk, partial, A == B);
  else
    fx_gram_kernel<2><<<n_chunks, 256, 0, st>>>(A, B, m, n_points, chunk, partial, A == B);
  return cudaGetLastError();
}

cudaError_t launch_apply_matrix(const double* M, int m, int lower, const double* S,
                                const double* X, double* Y, long long n_points, cudaStream_t st) {
  if (m < 1 || m > kMaxM) return cudaErrorInvalidValue;
  int dev = 0, sms = 152;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (m > kApplyMmaMin) {
    // Y = sum over blocks of 128 states, in stream order; each launch has a CTA
    // row per 64 rows that the block reaches
    const int nb = (m + kMmaRows - 1) / kMmaRows;
    const long long ntiles = (n_points + kApplyMmaPts - 1) / kApplyMmaPts;
    for (int k0 = 0; k0 < m; k0 += 128) {
      const int nk = m - k0 < 128 ? m - k0 : 128, rb0 = lower ? k0 / kMmaRows : 0;
      const int pitch = (nk > 64 ? 128 : 64) + 8;
      const size_t smem = (size_t)kDigits * (kMmaRows + kApplyMmaPts) * pitch * 2;
      cudaError_t e = cudaFuncSetAttribute(fx_apply_mma_kernel,
                                           cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
      if (e != cudaSuccess) return e;
      const int per = sms / (nb - rb0) > 0 ? (sms + nb - rb0 - 1) / (nb - rb0) : 1;
      const int grid = (int)(ntiles < per ? ntiles : per);
      fx_apply_mma_kernel<<<dim3(grid, nb - rb0), kMmaThreads, smem, st>>>(
          M, m, lower, S, X, Y, n_points, k0, nk, rb0, k0 > 0);
      e = cudaGetLastError();
      if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
  }
  if (m <= 16) return apply_launch<4>(M, m, lower, S, X, Y, n_points, sms, st);
  return apply_launch<8>(M, m, lower, S, X, Y, n_points, sms, st);
}

}  // namespace itp
