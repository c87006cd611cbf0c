// mixed_common.cuh -- shared by the mixed-radix kernels (mixr.cuh, mixed_ct.cu,
// fx64.cuh): complex arithmetic for FP32 and FP64 elements, the odd-prime 3/5/7
// DFTs, the padded shared-memory index and the reciprocal division.
#pragma once
#include <cuda_runtime.h>

#include "fft_common.cuh"

namespace gbfft {

// ---- complex arithmetic for both element types -----------------------------
template <typename T>
struct Cx;
template <>
struct Cx<float2> {
  using S = float;
  static __device__ __forceinline__ float2 make(float x, float y) { return make_float2(x, y); }
};
template <>
struct Cx<double2> {
  using S = double;
  static __device__ __forceinline__ double2 make(double x, double y) { return make_double2(x, y); }
};
template <typename T>
__device__ __forceinline__ T gadd(T a, T b) { return Cx<T>::make(a.x + b.x, a.y + b.y); }
template <typename T>
__device__ __forceinline__ T gsub(T a, T b) { return Cx<T>::make(a.x - b.x, a.y - b.y); }
template <typename T>
__device__ __forceinline__ T gmul(T a, T b) {
  return Cx<T>::make(fma(a.x, b.x, -a.y * b.y), fma(a.x, b.y, a.y * b.x));
}

// cos(2 pi m / R), sin(2 pi m / R) for the odd prime radices, m = 0..R-1
__device__ __forceinline__ constexpr double mixed_cos(int R, int m) {
  return R == 3 ? (m == 0 ? 1.0 : -0.5)
       : R == 5 ? (m == 0 ? 1.0 : (m == 1 || m == 4) ? 0.30901699437494742410 : -0.80901699437494742410)
       : (m == 0 ? 1.0 : (m == 1 || m == 6) ? 0.62348980185873353053
                       : (m == 2 || m == 5) ? -0.22252093395631440429 : -0.90096886790241912624);
}
__device__ __forceinline__ constexpr double mixed_sin(int R, int m) {
  return R == 3 ? (m == 0 ? 0.0 : m == 1 ? 0.86602540378443864676 : -0.86602540378443864676)
       : R == 5 ? (m == 0 ? 0.0 : m == 1 ? 0.95105651629515357212 : m == 2 ? 0.58778525229247312917
                 : m == 3 ? -0.58778525229247312917 : -0.95105651629515357212)
       : (m == 0 ? 0.0 : m == 1 ? 0.78183148246802980871 : m == 2 ? 0.97492791218182360702
          : m == 3 ? 0.43388373911755812048 : m == 4 ? -0.43388373911755812048 : m == 5 ? -0.97492791218182360702
          : -0.78183148246802980871);
}

// R-point forward DFT for an odd prime R: with t_m = x_m + x_{R-m},
// u_m = x_m - x_{R-m} (m = 1..(R-1)/2),
//   X_k = x_0 + sum_m cos(2 pi mk/R) t_m - i sum_m sin(2 pi mk/R) u_m,
//   X_{R-k} the same with +i.
template <int R, typename T>
__device__ __forceinline__ void dft_odd(T* v) {
  using S = typename Cx<T>::S;
  constexpr int H = (R - 1) / 2;
  T t[H], u[H];
  T s = v[0];
#pragma unroll
  for (int m = 1; m <= H; ++m) {
    t[m - 1] = gadd(v[m], v[R - m]);
    u[m - 1] = gsub(v[m], v[R - m]);
    s = gadd(s, t[m - 1]);
  }
  T out[R];
  out[0] = s;
#pragma unroll
  for (int k = 1; k <= H; ++k) {
    T A = v[0], B = Cx<T>::make(0, 0);
#pragma unroll
    for (int m = 1; m <= H; ++m) {
      const S c = (S)mixed_cos(R, (m * k) % R), sn = (S)mixed_sin(R, (m * k) % R);
      A.x = fma(c, t[m - 1].x, A.x);
      A.y = fma(c, t[m - 1].y, A.y);
      B.x = fma(sn, u[m - 1].x, B.x);
      B.y = fma(sn, u[m - 1].y, B.y);
    }
    out[k] = Cx<T>::make(A.x + B.y, A.y - B.x);
    out[R - k] = Cx<T>::make(A.x - B.y, A.y + B.x);
  }
#pragma unroll
  for (int q = 0; q < R; ++q) v[q] = out[q];
}

// Shared-memory index of tile element n: padded by one entry every 16 when
// PAD (conflict-free strided writes of a leading radix-8/16 pass, chosen per
// plan from a bank model of every pass), identity otherwise.
template <bool PAD>
__device__ __forceinline__ int msidx(int n) { return PAD ? n + (n >> 4) : n; }

// n / d from the reciprocal m = ceil(2^32 / d) (m = 0 stands for d = 1)
__device__ __forceinline__ unsigned fdiv(unsigned n, unsigned m) { return m ? __umulhi(n, m) : n; }

}  // namespace gbfft
