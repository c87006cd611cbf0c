// fx64.cuh -- FP64 (complex128) transforms of any 7-smooth length on the
// integer units: the tile kernel of mixr.cuh (same passes, schedules and
// layouts) over 64-bit fixed-point values with one exponent per transform.
//
// GB300 runs two FP64 operations a clock and SM, which bounds an FP64 FFT far
// above its memory time (4096 points: 32 FP64 operations a point, 1347 us per
// 2^24 points, where the memory takes 79).  It runs about 60 64-bit integer
// additions, 28 high halves of 32-bit products and 14 wide products.  A
// transform is a chain of additions and rotations that never grows by more
// than the radix in a pass, so a block exponent serves it well:
//   * the first pass finds the largest exponent of the transform's inputs and
//     turns them into integers below 2^(62 - headroom of its radix);
//   * every pass records the bits that its outputs use (an OR per thread and
//     one shared-memory atomic), and the next pass shifts so that its largest
//     value uses all the bits that its radix leaves;
//   * a rotation by a table factor (Q62) scales by 1/4 with its product, which
//     is the headroom the next additions need anyway;
//   * the last pass turns integers back into FP64, rounded to nearest.
// The largest value of a transform holds 57 to 62 bits at all times, against
// 53 in FP64, and factors are right to 2^-62, so the error against the norm of a
// row is below that of FP64 sums (4096 points, Gaussian: 5.9e-17 against 2.3e-16).
// Values far below a row's largest have fewer bits, though, where FP64 has 53 at
// any size.  Each transform is therefore looked at as it is read
// (FxTile::wide, fx_plane_bits): those whose inputs are not of one scale, those
// that hold an infinity or a NaN, and those between normal and subnormal numbers
// run in FP64 arithmetic instead, after the tile's other columns
// (fx_mixed_tile; a tile of such transforms alone 1546 us at 4096 points, 2500 at
// 7000).  The choice is a transform's own:
// its neighbours in the tile do not change it.  Results outside FP64's normal
// range take scalbn's rounding to subnormal numbers, zero or infinity.
// Radix 16 with 16 points a thread (128 registers): 16 warps an SM, held by
// latency and instruction fetch; radix 8 at the same 16 points and warps takes
// one pass more (290 against 254 us per 2^24 points at 4096), with 64 registers
// and 32 warps it spills as well (407 against 305, an earlier form).
// Measured per 2^24 points on GB300, against the FP64 kernel: 64 641 -> 151 us,
// 1000 1463 -> 321, 4096 1348 -> 234, 7000 1880 -> 545; two passes: 65536
// 1961 -> 366, 2^20 2485 -> 545.
#pragma once
#include <cuda_runtime.h>

#include <type_traits>

#include "fx64_math.h"
#include "gbfft_internal.h"
#include "mixed_common.cuh"

namespace gbfft {

constexpr double k2m62 = 2.168404344971008868e-19;   // 2^-62

// ---- DFTs ------------------------------------------------------------------------
__device__ __forceinline__ long long fx_shl(long long x, int s) { return (long long)((unsigned long long)x << s); }
__device__ __forceinline__ long long fx_scale4(long long x) { return fx_shl(x, 2); }

// x c for a constant c (Q62, |c| < 1).  Not as 4 (x c / 4), which would scale
// the product's rounding error by 4: four times c fits the 62-bit product when
// |c| < 1/2, and beyond that x c = +-x + x (c -+ 1).
template <long long c>
__device__ __forceinline__ long long fx_mulk(long long x) {
  constexpr long long one = 1LL << 62, half = 1LL << 61;
  constexpr long long m = c < 0 ? -c : c;
  if constexpr (m > half - 16 && m < half + 16) {
    return c < 0 ? (1 - x) >> 1 : (x + 1) >> 1;
  } else if constexpr (m < half) {
    constexpr Q62 k = q62_split(4 * c);
    return fx_mulr(x, k);
  } else if constexpr (c > 0) {
    constexpr Q62 k = q62_split(4 * (c - one));
    return x + fx_mulr(x, k);
  } else {
    constexpr Q62 k = q62_split(4 * (c + one));
    return fx_mulr(x, k) - x;
  }
}

// a W_R^M
template <int R, int M>
__device__ __forceinline__ Fx fx_mulw(Fx a) {
  constexpr int m = M % R;
  if constexpr (m == 0) {
    return a;
  } else if constexpr ((4 * m) % R == 0) {
    constexpr int qt = 4 * m / R;
    if constexpr (qt == 1) return Fx{a.y, -a.x};
    else if constexpr (qt == 2) return Fx{-a.x, -a.y};
    else return Fx{-a.y, a.x};
  } else if constexpr ((8 * m) % R == 0) {
    constexpr int et = 8 * m / R;
    constexpr long long r2 = fx_cossin(1, 8).c;
    if constexpr (et == 1) return Fx{fx_mulk<r2>(a.x + a.y), fx_mulk<r2>(a.y - a.x)};
    else if constexpr (et == 3) return Fx{fx_mulk<r2>(a.y - a.x), fx_mulk<-r2>(a.x + a.y)};
    else if constexpr (et == 5) return Fx{fx_mulk<-r2>(a.x + a.y), fx_mulk<r2>(a.x - a.y)};
    else return Fx{fx_mulk<r2>(a.x - a.y), fx_mulk<r2>(a.x + a.y)};
  } else {
    constexpr long long c = fx_cossin(m, R).c, s = fx_cossin(m, R).s;
    return Fx{fx_mulk<c>(a.x) + fx_mulk<s>(a.y), fx_mulk<c>(a.y) - fx_mulk<s>(a.x)};
  }
}

// The same in FP64, for the transforms that fixed point would shorten.
__device__ __forceinline__ double2 fx_add(double2 a, double2 b) { return gadd(a, b); }
__device__ __forceinline__ double2 fx_sub(double2 a, double2 b) { return gsub(a, b); }
template <int R, int M>
__device__ __forceinline__ double2 fx_mulw(double2 a) {
  constexpr int m = M % R;
  if constexpr (m == 0) {
    return a;
  } else if constexpr ((4 * m) % R == 0) {
    constexpr int qt = 4 * m / R;
    if constexpr (qt == 1) return make_double2(a.y, -a.x);
    else if constexpr (qt == 2) return make_double2(-a.x, -a.y);
    else return make_double2(-a.y, a.x);
  } else if constexpr ((8 * m) % R == 0) {
    constexpr int et = 8 * m / R;
    constexpr double r2 = (double)fx_cossin(1, 8).c * k2m62;
    const double p = r2 * (a.x + a.y), d = r2 * (a.y - a.x);
    if constexpr (et == 1) return make_double2(p, d);
    else if constexpr (et == 3) return make_double2(d, -p);
    else if constexpr (et == 5) return make_double2(-p, -d);
    else return make_double2(-d, p);
  } else {
    constexpr double c = (double)fx_cossin(m, R).c * k2m62, s = (double)fx_cossin(m, R).s * k2m62;
    return gmul(a, make_double2(c, -s));
  }
}

template <typename V>
__device__ __forceinline__ void fx_dft2(V& a, V& b) {
  const V t = a;
  a = fx_add(t, b);
  b = fx_sub(t, b);
}
template <typename V>
__device__ __forceinline__ void fx_dft4(V& x0, V& x1, V& x2, V& x3) {
  const V t0 = fx_add(x0, x2), t1 = fx_sub(x0, x2), t2 = fx_add(x1, x3), d = fx_sub(x1, x3);
  x0 = fx_add(t0, t2);
  x2 = fx_sub(t0, t2);
  x1 = V{t1.x + d.y, t1.y - d.x};
  x3 = V{t1.x - d.y, t1.y + d.x};
}

template <int R, typename V>
__device__ __forceinline__ void fx_dft(V* v);

// odd primes, as dft_odd of mixed_common.cuh
template <int R, int k, int m>
__device__ __forceinline__ void fx_odd_terms(const Fx* t, const Fx* u, Fx& A, Fx& B) {
  constexpr int H = (R - 1) / 2;
  if constexpr (m <= H) {
    constexpr long long c = fx_cossin((m * k) % R, R).c, s = fx_cossin((m * k) % R, R).s;
    A.x += fx_mulk<c>(t[m - 1].x);
    A.y += fx_mulk<c>(t[m - 1].y);
    B.x += fx_mulk<s>(u[m - 1].x);
    B.y += fx_mulk<s>(u[m - 1].y);
    fx_odd_terms<R, k, m + 1>(t, u, A, B);
  }
}
template <int R, int k>
__device__ __forceinline__ void fx_odd_outputs(Fx* out, Fx v0, const Fx* t, const Fx* u) {
  constexpr int H = (R - 1) / 2;
  if constexpr (k <= H) {
    Fx A = v0, B{0, 0};
    fx_odd_terms<R, k, 1>(t, u, A, B);
    out[k] = Fx{A.x + B.y, A.y - B.x};
    out[R - k] = Fx{A.x - B.y, A.y + B.x};
    fx_odd_outputs<R, k + 1>(out, v0, t, u);
  }
}
template <int R>
__device__ __forceinline__ void fx_dft_odd(Fx* v) {
  constexpr int H = (R - 1) / 2;
  Fx t[H], u[H], out[R];
  Fx s = v[0];
#pragma unroll
  for (int m = 1; m <= H; ++m) {
    t[m - 1] = fx_add(v[m], v[R - m]);
    u[m - 1] = fx_sub(v[m], v[R - m]);
    s = fx_add(s, t[m - 1]);
  }
  out[0] = s;
  fx_odd_outputs<R, 1>(out, v[0], t, u);
#pragma unroll
  for (int q = 0; q < R; ++q) v[q] = out[q];
}

template <int R, int B, int n2, int k1, int A, typename V>
__device__ __forceinline__ void fx_inner(V (&x)[B][A]) {
  if constexpr (n2 < B) {
    if constexpr (k1 < A) {
      x[n2][k1] = fx_mulw<R, n2 * k1>(x[n2][k1]);
      fx_inner<R, B, n2, k1 + 1, A>(x);
    } else {
      fx_inner<R, B, n2 + 1, 1, A>(x);
    }
  }
}
// R = A B, as ct_dft_split of mixed_ct.cuh
template <int A, int B, typename V>
__device__ __forceinline__ void fx_dft_split(V* v) {
  constexpr int R = A * B;
  V x[B][A];
#pragma unroll
  for (int n2 = 0; n2 < B; ++n2)
#pragma unroll
    for (int n1 = 0; n1 < A; ++n1) x[n2][n1] = v[B * n1 + n2];
#pragma unroll
  for (int n2 = 0; n2 < B; ++n2) fx_dft<A>(x[n2]);
  fx_inner<R, B, 1, 1, A>(x);
  V y[A][B];
#pragma unroll
  for (int k1 = 0; k1 < A; ++k1)
#pragma unroll
    for (int n2 = 0; n2 < B; ++n2) y[k1][n2] = x[n2][k1];
#pragma unroll
  for (int k1 = 0; k1 < A; ++k1) fx_dft<B>(y[k1]);
#pragma unroll
  for (int k1 = 0; k1 < A; ++k1)
#pragma unroll
    for (int k2 = 0; k2 < B; ++k2) v[k1 + A * k2] = y[k1][k2];
}

template <int R, typename V>
__device__ __forceinline__ void fx_dft(V* v) {
  if constexpr (R == 2) fx_dft2(v[0], v[1]);
  else if constexpr (R == 4) fx_dft4(v[0], v[1], v[2], v[3]);
  else if constexpr ((R == 3 || R == 5 || R == 7) && std::is_same_v<V, double2>) dft_odd<R>(v);
  else if constexpr (R == 3 || R == 5 || R == 7) fx_dft_odd<R>(v);
  else if constexpr (R == 8) fx_dft_split<4, 2>(v);
  else if constexpr (R == 9) fx_dft_split<3, 3>(v);
  else if constexpr (R == 10) fx_dft_split<2, 5>(v);
  else if constexpr (R == 12) fx_dft_split<4, 3>(v);
  else if constexpr (R == 14) fx_dft_split<2, 7>(v);
  else if constexpr (R == 15) fx_dft_split<3, 5>(v);
  else {
    static_assert(R == 16, "radices: 2, 3, 4, 5, 7, 8, 9, 10, 12, 14, 15, 16");
    fx_dft_split<4, 4>(v);
  }
}

// ---- the tile ----------------------------------------------------------------------
__device__ __forceinline__ Cq62 fx_ldw(const int4* p) {
  const int4 w = __ldg(p);   // (r.l, r.h, i.l, i.h)
  return Cq62{Q62{w.y, w.x}, Q62{w.w, w.z}};
}
// The top set bit of h ^ 2h is one above the highest bit that h (the high word
// of a two's complement number) uses beside its sign.
__device__ __forceinline__ int fx_bits(int acc, Fx a) {
  const int x = (int)(a.x >> 32), y = (int)(a.y >> 32);
  return acc | (x ^ (x + x)) | (y ^ (y + y));
}
// Inputs of a transform at the bottom of the exponent range.
static __device__ __noinline__ long long fx_from_any(double x, int E, int F) {
  return fx_from_bits<true>(__double_as_longlong(x), E, F);
}
// Results that may lie outside the normal range.  Out of line: inlined, its
// FP64 instructions would run for every output.
static __device__ __noinline__ double fx_out_any(long long q, int ex) { return scalbn((double)q, ex); }

// a Q62 table factor in FP64
__device__ __forceinline__ double2 fx_factor(const int4* p) {
  const Cq62 w = fx_ldw(p);
  return make_double2(((double)w.r.h * 4294967296.0 + (double)w.r.l) * k2m62,
                      ((double)w.i.h * 4294967296.0 + (double)w.i.l) * k2m62);
}

// points a thread holds in the first and the middle passes: with 20, two
// butterflies of radix 10 and four of radix 5 fit 128 registers (18 before: 1000
// points 469 -> 387 us per 2^24, 4000 610 -> 497)
constexpr int kFxPoints = 20;
template <int R>
struct FxK {
  static constexpr int value = kFxPoints / R > 0 ? kFxPoints / R : 1;
};

template <bool STR, bool LIN>
struct FxTile {
  const FxArgs& a;
  Fx* sm;
  int* slot;       // slot[s * C + c]: s = 0 the largest high word of |inputs|, s > 0 the bits used by pass s - 1
  const double2* gin;
  double2* gout;
  unsigned col0;
  int valid;

  __device__ __forceinline__ void split(int b, int s, int& c, int& j) const {
    if (STR && (s > 0 || !a.in_rows)) {
      c = b & ((1 << a.csh) - 1);
      j = b >> a.csh;
    } else {
      c = (int)fdiv((unsigned)b, a.nb_m[s]);
      j = b - c * (int)a.nb[s];
    }
  }
  __device__ __forceinline__ int at(int c, int n) const {
    if constexpr (STR)
      return (n + (n >> a.pad_sh)) * a.pitch + c;
    else {
      const int i = c * a.N + n;
      return i + (i >> a.pad_sh);
    }
  }
  // tile elements of butterfly (c, j): position j + r NB of the input side,
  // m0 + q Ns of the output side.  LIN: the pad keeps them evenly spaced, so
  // one address and a stride reach them all.
  template <int R>
  __device__ __forceinline__ void load_tile(Fx* v, int s, int c, int j, int NB) const {
    if constexpr (LIN) {
      const Fx* p = sm + at(c, j);
      const int st = a.ld_st[s];
#pragma unroll
      for (int r = 0; r < R; ++r) v[r] = p[r * st];
    } else {
#pragma unroll
      for (int r = 0; r < R; ++r) v[r] = sm[at(c, j + r * NB)];
    }
  }
  __device__ __forceinline__ const double2* in_at(int c, int n) const {
    if constexpr (STR)
      return gin + ((unsigned)c * a.in_cs + (unsigned)n * a.in_ns);
    else
      return gin + (c * a.N + n);
  }
  __device__ __forceinline__ double2* out_at(int c, int k) const {
    if constexpr (STR)
      return gout + ((unsigned)c * a.out_cs + (unsigned)k * a.out_ns);
    else
      return gout + (c * a.N + k);
  }
  // Right shift (left where negative) before the rotations of pass s, whose
  // radix has headroom h: the largest value then uses all the bits it may.
  __device__ __forceinline__ int shift_of(int s, int h, int c) const {
    return 63 - __clz(slot[s * a.C + c]) - (64 - h);
  }
  // exponent of one unit of pass s's input (s = nrad: of the last pass's output)
  __device__ __forceinline__ int exponent(int c) const {
    int e = fx_row_exponent(slot[c]) - 1022 - (62 - a.head[0]);
    for (int s = 1; s < a.nrad; ++s) e += 2 + shift_of(s, a.head[s], c);
    return e;
  }

  // with the largest high words of the real and the imaginary parts
  template <int R>
  __device__ __forceinline__ void load_bits(double2* v, int c, int j, int NB, int& tx, int& ty) const {
    const bool ok = c < valid;
    tx = ty = 0;
#pragma unroll
    for (int r = 0; r < R; ++r) {
      v[r] = ok ? __ldcs(in_at(c, j + r * NB)) : make_double2(0, 0);
      tx = max(tx, __double2hiint(v[r].x) & 0x7fffffff);
      ty = max(ty, __double2hiint(v[r].y) & 0x7fffffff);
    }
  }
  template <int R>
  __device__ __forceinline__ void to_fixed(Fx* f, const double2* v, int E) const {
    constexpr int F = 62 - fx_headroom(R);
    if (E > kFxSubnormal) {
#pragma unroll
      for (int r = 0; r < R; ++r) {
        f[r].x = fx_from_bits<false>(__double_as_longlong(v[r].x), E, F);
        f[r].y = fx_from_bits<false>(__double_as_longlong(v[r].y), E, F);
      }
    } else {
#pragma unroll
      for (int r = 0; r < R; ++r) f[r] = Fx{fx_from_any(v[r].x, E, F), fx_from_any(v[r].y, E, F)};
    }
    if (a.conj_in) {
#pragma unroll
      for (int r = 0; r < R; ++r) f[r].y = -f[r].y;
    }
  }
  template <int R>
  __device__ __forceinline__ void store_tile(const Fx* v, int s, int c, int m0, int Ns) const {
    int bits = 0;
    Fx* p = sm + at(c, m0);
    const int st = a.st_st[s];
#pragma unroll
    for (int q = 0; q < R; ++q) {
      if constexpr (LIN)
        p[q * st] = v[q];
      else
        sm[at(c, m0 + q * Ns)] = v[q];
      bits = fx_bits(bits, v[q]);
    }
    atomicOr(slot + (s + 1) * a.C + c, bits);
  }
  // block shift and rotations
  template <int R>
  __device__ __forceinline__ void rotate(Fx* v, int s, int c, int Ns, int k) const {
    const int sh = shift_of(s, fx_headroom(R), c);
    v[0] = sh > -2 ? Fx{fx_shr(v[0].x, sh + 2), fx_shr(v[0].y, sh + 2)}
                   : Fx{fx_shl(v[0].x, -2 - sh), fx_shl(v[0].y, -2 - sh)};
    if (sh > 0) {
#pragma unroll
      for (int r = 1; r < R; ++r) v[r] = Fx{fx_shr(v[r].x, sh), fx_shr(v[r].y, sh)};
    } else if (sh < 0) {
#pragma unroll
      for (int r = 1; r < R; ++r) v[r] = Fx{fx_shl(v[r].x, -sh), fx_shl(v[r].y, -sh)};
    }
    const int4* t = a.tw + a.tw_off[s] + k;
#pragma unroll
    for (int r = 1; r < R; ++r) v[r] = fx_cmul(v[r], fx_ldw(t + (r - 1) * Ns));
  }
  // outputs k0 + q Ns of column c, in units of 2^ex
  template <int R>
  __device__ __forceinline__ void store_global(Fx* v, int c, int k0, int Ns, int ex) const {
    if (c >= valid) return;
    if constexpr (STR) {
      if (a.ft) {
        const int4* f = a.ft + (size_t)(unsigned)k0 * a.ft_cols + (col0 + c);
        const size_t fs = (size_t)(unsigned)Ns * a.ft_cols;
#pragma unroll
        for (int q = 0; q < R; ++q) v[q] = fx_cmul(v[q], fx_ldw(f + q * fs));
        ex += 2;
      } else if (a.ft_lo) {
        const unsigned col = col0 + (unsigned)c, mask = (1u << a.ft_s) - 1u;
        unsigned e = col * (unsigned)k0;
        const unsigned es = col * (unsigned)Ns;
#pragma unroll
        for (int q = 0; q < R; ++q) {
          const Fx p = fx_cmul(v[q], fx_ldw(a.ft_lo + (e & mask)));
          v[q] = fx_cmul(Fx{fx_scale4(p.x), fx_scale4(p.y)}, fx_ldw(a.ft_hi + (e >> a.ft_s)));
          e += es;
        }
        ex += 2;
      }
    }
    ex += a.scale_ex;
    if (a.scale_q.h) {   // a scale that is no power of two
#pragma unroll
      for (int q = 0; q < R; ++q) v[q] = Fx{v[q].x + fx_mulr(v[q].x, a.scale_q), v[q].y + fx_mulr(v[q].y, a.scale_q)};
    }
    const long long flip = a.conj_out ? (long long)0x8000000000000000ULL : 0;
    if (fx_normal(ex)) {
#pragma unroll
      for (int q = 0; q < R; ++q)
        __stcs(out_at(c, k0 + q * Ns), make_double2(__longlong_as_double(fx_to_bits(v[q].x, ex)),
                                                    __longlong_as_double(fx_to_bits(v[q].y, ex) ^ flip)));
    } else {
#pragma unroll
      for (int q = 0; q < R; ++q)
        *out_at(c, k0 + q * Ns) = make_double2(fx_out_any(v[q].x, ex), fx_out_any(a.conj_out ? -v[q].y : v[q].y, ex));
    }
  }

  // Whether fixed point would shorten a butterfly's inputs beside the row's
  // largest high word top (fx_plane_bits); tx and ty as load_bits gives them.
  template <int R>
  __device__ __forceinline__ bool wide(const double2* v, int tx, int ty, int top) const {
    const int E = fx_row_exponent(top);
    if (E <= 64) return E > kFxSubnormal;
    const int least = top - (fx_plane_bits(R) << 20);
    if (min(tx, ty) >= least) return false;
    if ((tx > 0 && tx < least) || (ty > 0 && ty < least)) return true;
    int low = 0;   // zeros lose nothing, but numbers whose high word is zero would
#pragma unroll
    for (int r = 0; r < R; ++r) {
      low |= __double2hiint(v[r].x) & 0x7fffffff ? 0 : __double2loint(v[r].x);
      low |= __double2hiint(v[r].y) & 0x7fffffff ? 0 : __double2loint(v[r].y);
    }
    return low != 0;
  }
  // The transform of column c is left to FP64 arithmetic.
  __device__ __forceinline__ bool in_fp64(int c) const { return slot[c] >= 0x7ff00000; }

  // True in a thread that met a column for FP64 arithmetic.
  template <int R, int K>
  __device__ __forceinline__ bool first() const {
    const int NB = (int)a.nb[0], total = a.C * NB;
    double2 v[K][R];
    int tx[K], ty[K];
#pragma unroll
    for (int i = 0; i < K; ++i) {
      const int b = threadIdx.x + i * blockDim.x;
      if (b < total) {
        int c, j;
        split(b, 0, c, j);
        load_bits<R>(v[i], c, j, NB, tx[i], ty[i]);
        atomicMax(slot + c, max(tx[i], ty[i]));
      }
    }
    __syncthreads();
    bool any = false;
#pragma unroll
    for (int i = 0; i < K; ++i) {
      const int b = threadIdx.x + i * blockDim.x;
      if (b < total) {
        int c, j;
        split(b, 0, c, j);
        const int top = slot[c];
        if (top >= 0x7ff00000) {
          any = true;
        } else if (wide<R>(v[i], tx[i], ty[i], top)) {
          atomicMax(slot + c, 0x7fffffff);
          any = true;
        }
        Fx f[R];
        to_fixed<R>(f, v[i], fx_row_exponent(top));
        fx_dft<R>(f);
        store_tile<R>(f, 0, c, j * R, 1);
      }
    }
    return any;
  }

  template <int R, int K>
  __device__ __forceinline__ void middle(int s) const {
    const int NB = (int)a.nb[s], Ns = (int)a.ns[s], total = a.C * NB;
    Fx v[K][R];
#pragma unroll
    for (int i = 0; i < K; ++i) {
      const int b = threadIdx.x + i * blockDim.x;
      int c = 0, j = 0;
      if (b < total) split(b, s, c, j);
      // (threads without a butterfly read one too, so that nothing lives across the pass loop)
      load_tile<R>(v[i], s, c, j, NB);
    }
    __syncthreads();
#pragma unroll
    for (int i = 0; i < K; ++i) {
      const int b = threadIdx.x + i * blockDim.x;
      if (b < total) {
        int c, j;
        split(b, s, c, j);
        const int jq = (int)fdiv((unsigned)j, a.ns_m[s]);
        const int k = j - jq * Ns;
        rotate<R>(v[i], s, c, Ns, k);
        fx_dft<R>(v[i]);
        store_tile<R>(v[i], s, c, jq * Ns * R + k, Ns);
      }
    }
  }

  // SKIP: but the columns left to FP64 arithmetic
  template <int R, bool SKIP>
  __device__ __forceinline__ void last(int s) const {
    const int NB = (int)a.nb[s], total = a.C * NB;   // Ns == NB
    for (int b = threadIdx.x; b < total; b += blockDim.x) {
      int c, j;
      split(b, s, c, j);
      if (SKIP && in_fp64(c)) continue;
      Fx v[R];
      load_tile<R>(v, s, c, j, NB);
      rotate<R>(v, s, c, NB, j);
      fx_dft<R>(v);
      store_global<R>(v, c, j, NB, exponent(c));
    }
  }

  // N is a single radix (at most 7): one butterfly a transform, in registers.
  // Radices 2 and 4 add in FP64, exact where the numbers are (180 and 242 us per
  // 2^24 points; the integers take 127 and 124), but rows of subnormal numbers,
  // which the integers hold exactly.
  template <int R>
  __device__ __forceinline__ void only() const {
    for (int c = threadIdx.x; c < a.C; c += blockDim.x) {
      double2 v[R];
      int tx, ty;
      load_bits<R>(v, c, 0, 1, tx, ty);
      const int top = max(tx, ty), E = fx_row_exponent(top);
      bool fp64;
      if constexpr (R == 2 || R == 4) {
        int bits = top;
#pragma unroll
        for (int r = 0; r < R; ++r) bits |= __double2loint(v[r].x) | __double2loint(v[r].y);
        fp64 = E > kFxSubnormal || bits == 0;
      } else {
        fp64 = top >= 0x7ff00000 || wide<R>(v, tx, ty, top);
      }
      if (fp64) {
        if (a.conj_in) {
#pragma unroll
          for (int r = 0; r < R; ++r) v[r].y = -v[r].y;
        }
        fx_dft<R>(v);
#pragma unroll
        for (int q = 0; q < R; ++q) store_double(v[q], c, q);
      } else {
        Fx f[R];
        to_fixed<R>(f, v, E);
        fx_dft<R>(f);
        store_global<R>(f, c, 0, 1, E - 1022 - (62 - fx_headroom(R)));
      }
    }
  }

  // output k of column c in FP64 arithmetic: four-step factor, conjugation, scale
  __device__ __forceinline__ void store_double(double2 y, int c, int k) const {
    if (c >= valid) return;
    if (STR && a.ft) {
      y = gmul(y, fx_factor(a.ft + (size_t)(unsigned)k * a.ft_cols + (col0 + c)));
    } else if (STR && a.ft_lo) {
      const unsigned e = (col0 + (unsigned)c) * (unsigned)k;
      y = gmul(y, gmul(fx_factor(a.ft_lo + (e & ((1u << a.ft_s) - 1u))), fx_factor(a.ft_hi + (e >> a.ft_s))));
    }
    *out_at(c, k) = make_double2(y.x * a.scale, y.y * (a.conj_out ? -a.scale : a.scale));
  }

  // Pass s of the columns left to FP64 arithmetic.
  template <int R, int K>
  __device__ __forceinline__ void double_pass(int s) const {
    const int NB = (int)a.nb[s], Ns = (int)a.ns[s], total = a.C * NB;
    const bool first = s == 0, last = s == a.nrad - 1;
    const int step = NB / Ns;   // W_{Ns R} = W_N^{N / (Ns R)}
    double2* const ds = (double2*)sm;
    // (a middle pass has one round: its inputs are all held before any output is written)
#pragma unroll 1
    for (int base = threadIdx.x; base - (int)threadIdx.x < total; base += K * (int)blockDim.x) {
      double2 v[K][R];
#pragma unroll
      for (int i = 0; i < K; ++i) {
        const int b = base + i * (int)blockDim.x;
        int c = 0, j = 0;
        if (b < total) split(b, s, c, j);
        if (b < total && c < valid && in_fp64(c)) {
#pragma unroll
          for (int r = 0; r < R; ++r) {
            v[i][r] = first ? __ldcs(in_at(c, j + r * NB)) : ds[at(c, j + r * NB)];
            if (first && a.conj_in) v[i][r].y = -v[i][r].y;
          }
        } else {
#pragma unroll
          for (int r = 0; r < R; ++r) v[i][r] = make_double2(0, 0);
        }
      }
      if (!first && !last) __syncthreads();
#pragma unroll
      for (int i = 0; i < K; ++i) {
        const int b = base + i * (int)blockDim.x;
        int c = 0, j = 0;
        if (b < total) split(b, s, c, j);
        if (b < total && c < valid && in_fp64(c)) {
          const int jq = (int)fdiv((unsigned)j, a.ns_m[s]);
          const int k = j - jq * Ns;
          if (!first) {
#pragma unroll
            for (int r = 1; r < R; ++r) v[i][r] = gmul(v[i][r], __ldg(a.wn + r * k * step));
          }
          fx_dft<R>(v[i]);
          const int m0 = jq * Ns * R + k;
#pragma unroll
          for (int q = 0; q < R; ++q) {
            if (last)
              store_double(v[i][q], c, m0 + q * Ns);
            else
              ds[at(c, m0 + q * Ns)] = v[i][q];
          }
        }
      }
    }
  }
};

#define GBFFT_FX_SWITCH(r, CALL) \
  switch (r) {                   \
    case 2: CALL(2); break;      \
    case 3: CALL(3); break;      \
    case 4: CALL(4); break;      \
    case 5: CALL(5); break;      \
    case 7: CALL(7); break;      \
    case 8: CALL(8); break;      \
    case 9: CALL(9); break;      \
    case 10: CALL(10); break;    \
    case 12: CALL(12); break;    \
    case 14: CALL(14); break;    \
    case 15: CALL(15); break;    \
    default: CALL(16); break;    \
  }

template <bool STR, bool LIN>
__device__ __forceinline__ FxTile<STR, LIN> fx_tile(const FxArgs& a, unsigned char* smem) {
  const long long t = a.tile0 + blockIdx.x;
  if constexpr (STR) {
    const long long bt = t / a.tiles_per_batch;
    const long long c0 = (t - bt * a.tiles_per_batch) << a.csh;
    const int valid = (int)(a.ncols - c0 < a.C ? a.ncols - c0 : a.C);
    return FxTile<STR, LIN>{a, (Fx*)smem, (int*)(smem + a.slot_off), a.in + bt * a.in_bs + c0 * a.in_cs,
                            a.out + bt * a.out_bs + c0 * a.out_cs, (unsigned)c0, valid};
  } else {
    const long long c0 = t * a.C;
    const int valid = (int)(a.ncols - c0 < a.C ? a.ncols - c0 : a.C);
    return FxTile<STR, LIN>{a, (Fx*)smem, (int*)(smem + a.slot_off), a.in + c0 * a.N, a.out + c0 * a.N, 0u, valid};
  }
}

// N is a single radix (at most 7).  A kernel of its own: inside fx_kernel these
// branches cost the others 2,268 bytes of spills, 81 local stores and 91 loads a
// thread at 4096 points (294 us per 2^24 points against 230).
template <bool STR, bool LIN>
__global__ void __launch_bounds__(256) fx_only_kernel(const __grid_constant__ FxArgs a) {
  const FxTile<STR, LIN> T = fx_tile<STR, LIN>(a, nullptr);
  switch (a.rad[0]) {
    case 2: T.template only<2>(); break;
    case 3: T.template only<3>(); break;
    case 4: T.template only<4>(); break;
    case 5: T.template only<5>(); break;
    default: T.template only<7>(); break;
  }
}

// The passes in fixed point after the first.
template <bool SKIP, bool STR, bool LIN>
__device__ __forceinline__ void fx_passes(const FxTile<STR, LIN>& T) {
  const int last = T.a.nrad - 1;
  for (int s = 1; s < last; ++s) {
#define CALL(R) T.template middle<R, FxK<R>::value>(s)
    GBFFT_FX_SWITCH(T.a.rad[s], CALL)
#undef CALL
    __syncthreads();
  }
#define CALL(R) T.template last<R, SKIP>(last)
  GBFFT_FX_SWITCH(T.a.rad[last], CALL)
#undef CALL
}

// The rest of a tile with columns that fixed point would shorten: the others,
// then those in FP64 arithmetic, whose inputs are still there when in == out (the
// others' outputs lie elsewhere).  Out of line, with passes of its own: one call
// after the kernel's own passes cost every tile 2 % (registers), and so did a
// second call inside or the tile handed over by reference (4096 points, 2^24 in
// all: 234 us so, 237 to 240 otherwise, 232 without any of it).
template <bool STR>
__device__ __noinline__ void fx_mixed_tile(const FxArgs& a, unsigned char* smem) {
  const FxTile<STR, false> T = fx_tile<STR, false>(a, smem);
  int fixed = 0;
  for (int c = threadIdx.x; c < T.valid; c += blockDim.x) fixed |= !T.in_fp64(c);
  if (__syncthreads_or(fixed)) fx_passes<true>(T);
#pragma unroll 1
  for (int s = 0; s < a.nrad; ++s) {
    __syncthreads();
#define CALL(R) T.template double_pass<R, FxK<R>::value>(s)
    GBFFT_FX_SWITCH(a.rad[s], CALL)
#undef CALL
  }
}

// 128 registers: one CTA of 512 threads per SM, two of 256, four of 128.
template <bool STR, bool LIN>
__global__ void __launch_bounds__(512, 1) fx_kernel(const __grid_constant__ FxArgs a) {
  extern __shared__ __align__(16) unsigned char fx_smem[];
  const FxTile<STR, LIN> T = fx_tile<STR, LIN>(a, fx_smem);
  int* const slot = T.slot;
  for (int i = threadIdx.x; i < a.nrad * a.C; i += blockDim.x) slot[i] = 0;
  __syncthreads();
  int any = 0;
#define CALL(R) any = T.template first<R, FxK<R>::value>()
  GBFFT_FX_SWITCH(a.rad[0], CALL)
#undef CALL
  if (__syncthreads_or(any)) {
    fx_mixed_tile<STR>(a, fx_smem);
    return;
  }
  fx_passes<false>(T);
}

}  // namespace gbfft
