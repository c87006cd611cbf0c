// fx64_math.h -- 64-bit fixed-point arithmetic of the FP64 transforms
// (fx64.cuh): complex values as two int64, factors of modulus at most one as
// Q62 numbers split into two signed 32-bit halves, and the exact conversions
// from and to FP64.  Plain C++17 on the host too, so the test suite checks it
// against 128-bit integers with g++.
#pragma once
#include <cstdint>
#include <cstring>

#ifdef __CUDACC__
#define GBFFT_HD __host__ __device__ __forceinline__
#define GBFFT_HD_FN __host__ __device__
#else
#define GBFFT_HD inline
#define GBFFT_HD_FN
#endif

namespace gbfft {

struct Fx {   // re, im
  long long x, y;
};
// A real factor c, |c| <= 1: c 2^62 = h 2^32 + l, both signed (l > -2^31).
struct Q62 {
  int h, l;
};
struct Cq62 {   // complex factor
  Q62 r, i;
};

constexpr GBFFT_HD_FN Q62 q62_split(long long q) {
  long long lo = (long long)(int)(unsigned)(unsigned long long)q;
  if (lo == -2147483648LL) ++lo;   // keeps -l representable (2^-62 off)
  return Q62{(int)((q - lo) >> 32), (int)lo};
}
// c 2^62 of an FP64 number
constexpr Q62 q62(double c) { return q62_split((long long)(c * 4611686018427387904.0)); }

// ---- cos and sin of 2 pi m / M to the last bits of Q62 ------------------------
// By the octant symmetries of the unit circle and the Taylor series on
// [0, pi/4] in 64-bit fixed point, for the table entries on the device and for
// constants at compile time.  (FP64 values, right to 2^-54, would be the
// largest error of a transform whose terms are all in phase.)
constexpr GBFFT_HD_FN unsigned long long fx_umulhi(unsigned long long a, unsigned long long b) {
  const unsigned long long al = a & 0xffffffffULL, ah = a >> 32, bl = b & 0xffffffffULL, bh = b >> 32;
  const unsigned long long m1 = al * bh + ((al * bl) >> 32), m2 = ah * bl + (m1 & 0xffffffffULL);
  return ah * bh + (m1 >> 32) + (m2 >> 32);
}
struct FxCosSin {
  long long c, s;   // Q62
};
// 0 <= m < M < 2^29
constexpr GBFFT_HD_FN FxCosSin fx_cossin(long long m, long long M) {
  const long long o = 8 * m / M;
  unsigned long long n = (unsigned long long)(8 * m - o * M), d = (unsigned long long)M;
  if (o & 1) n = d - n;   // odd octants measure from the next multiple of pi/4 downwards
  const unsigned long long pi4 = 0xC90FDAA22168C234ULL;   // pi/4, Q64
  const unsigned long long hi = (n << 32) / d, lo = (((n << 32) % d) << 32) / d;
  const unsigned long long t = n == d ? pi4 : fx_umulhi((hi << 32) | lo, pi4);   // the angle, Q64
  const unsigned long long t2 = fx_umulhi(t, t), one = 1ULL << 63;
  unsigned long long cs = one, sn = one;   // Q63
  for (int k = 12; k >= 1; --k) {
    cs = one - fx_umulhi(t2, cs) / (unsigned long long)((2 * k - 1) * (2 * k));
    sn = one - fx_umulhi(t2, sn) / (unsigned long long)((2 * k) * (2 * k + 1));
  }
  const long long c = (long long)((cs + 1) >> 1), s = (long long)((fx_umulhi(t, sn) + 1) >> 1);
  switch (o) {
    case 0: return FxCosSin{c, s};
    case 1: return FxCosSin{s, c};
    case 2: return FxCosSin{-s, c};
    case 3: return FxCosSin{-c, s};
    case 4: return FxCosSin{-c, -s};
    case 5: return FxCosSin{-s, -c};
    case 6: return FxCosSin{s, -c};
    default: return FxCosSin{c, -s};
  }
}

GBFFT_HD int fx_mulhi(int a, int b) {
#ifdef __CUDA_ARCH__
  return __mulhi(a, b);
#else
  return (int)(((long long)a * (long long)b) >> 32);
#endif
}
GBFFT_HD Fx fx_add(Fx a, Fx b) { return Fx{a.x + b.x, a.y + b.y}; }
GBFFT_HD Fx fx_sub(Fx a, Fx b) { return Fx{a.x - b.x, a.y - b.y}; }

// High half of x = h 2^32 + l with l = (int)x signed.
GBFFT_HD int fx_hi(long long x) { return (int)(x >> 32) + (int)((unsigned)(unsigned long long)x >> 31); }

// x c / 4 (|x| < 2^63, |c| < 2): the 64 x 62-bit product without its lowest 32 x 32
// part.  Each mulhi rounds down by up to one unit; one is added and one
// subtracted, so the errors cancel on average and 0 gives 0.
GBFFT_HD long long fx_mulr(long long x, Q62 c) {
  const int h = fx_hi(x), l = (int)x;
  return (long long)h * c.h + (fx_mulhi(h, c.l) - fx_mulhi(l, -c.h));
}
// a w / 4, the four products of each part rounded the same way
GBFFT_HD Fx fx_cmul(Fx a, Cq62 w) {
  const int rh = fx_hi(a.x), rl = (int)a.x, ih = fx_hi(a.y), il = (int)a.y;
  const int mr = (fx_mulhi(rh, w.r.l) + fx_mulhi(rl, w.r.h)) - (fx_mulhi(ih, w.i.l) + fx_mulhi(il, w.i.h));
  const int mi = (fx_mulhi(rh, w.i.l) + fx_mulhi(rl, w.i.h)) - (fx_mulhi(ih, -w.r.l) + fx_mulhi(il, -w.r.h));
  return Fx{(long long)rh * w.r.h + ((long long)ih * -w.i.h + mr), (long long)rh * w.i.h + ((long long)ih * w.r.h + mi)};
}
// rounded shift right by s >= 1
GBFFT_HD long long fx_shr(long long x, int s) { return (x + (1LL << (s - 1))) >> s; }

// E of a row with the largest high word top of |x|: |x| < 2^(E - 1022).  The
// biased exponent, or less for a row of subnormal numbers.
GBFFT_HD int fx_row_exponent(int top) {
  if (top >= 0x100000) return top >> 20;
#ifdef __CUDA_ARCH__
  return 12 - __clz(top);
#else
  return 12 - (top ? __builtin_clz((unsigned)top) : 32);
#endif
}
// FP64 x (finite) as an integer multiple of 2^(E - 1022 - F), truncated, for a
// row exponent E and 53 <= F <= 61, so that |result| < 2^F.  SUB: subnormal
// inputs count; else they do not reach the result (E > 64).
template <bool SUB>
GBFFT_HD long long fx_from_bits(long long bits, int E, int F) {
  const int hi = (int)(bits >> 32);
  const int e = (hi >> 20) & 0x7ff;
  int mh = (hi & 0xfffff) | 0x100000;
  int d = E - e;
  if (SUB && e == 0) {
    mh = hi & 0xfffff;
    d = E - 1;
  }
  if (d > 63) d = 63;
  int left = F - 53;
  if (SUB && d < 0) {   // a row of subnormal numbers
    left -= d;
    d = 0;
  }
  const unsigned long long m = ((unsigned long long)(unsigned)mh << 32) | (unsigned)(unsigned long long)bits;
  const long long q = (long long)((m << left) >> d);
  const long long s = (long long)(hi >> 31);
  return (q ^ s) - s;
}

// q 2^ex as FP64 bits, rounded to nearest, for |q| < 2^63 and an ex for which
// every such result is normal or zero (fx_normal).  The conversion is one of the
// FP64 pipe's, idle otherwise: 2 a clock and SM, against a leading-zero count, two
// 64-bit shifts and the rounding on the integer units, which bound these kernels
// (4096 points, 2^24 in all: 311 -> 291 us).
constexpr bool fx_normal(int ex) { return ex >= -1022 && ex <= 958; }
GBFFT_HD long long fx_to_bits(long long q, int ex) {
#ifdef __CUDA_ARCH__
  const unsigned long long d = (unsigned long long)__double_as_longlong(__ll2double_rn(q));
#else
  const double f = (double)q;
  unsigned long long d;
  memcpy(&d, &f, 8);
#endif
  const unsigned hi = (unsigned)(d >> 32);
  return (long long)((unsigned long long)(hi ? hi + ((unsigned)ex << 20) : 0u) << 32 | (unsigned)d);
}

// bits of headroom an R-point DFT needs: ceil(log2(R sqrt 2)) (R - 1 additions
// of values whose parts turn into one another)
constexpr int fx_headroom(int r) {
  return r <= 2 ? 2 : r <= 5 ? 3 : r <= 11 ? 4 : 5;
}

// Which transforms fixed point may take.  An input 2^-k of the largest keeps
// about 57 - k bits.  Beside a large input of its own sum that is what FP64 keeps
// of it (the sum rounds it to 53 bits of the larger), but where a whole sum is
// small the result would lose bits that FP64 holds: real and imaginary parts of
// different scale, pulses, combs.  So a transform goes to FP64 arithmetic when the
// real (or the imaginary) inputs of any first-pass butterfly are not all zero
// and all below 2^-fx_plane_bits of its largest input.  Data of one scale stay:
// of Gaussian rows of 4096 points, fewer than 1 in 6,000 (radix 2) to 10^18
// (radix 16) go.
constexpr int fx_plane_bits(int r) { return 4 + (20 + r - 1) / r; }
// Row exponents up to this one hold every subnormal number exactly in fixed
// point (one unit is 2^(E - 1022 - 57)); FP64 products of them would not.
constexpr int kFxSubnormal = 5;

}  // namespace gbfft
