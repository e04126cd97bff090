// Kernel samples of the M2L coupling blocks (Sec. 4.4) between the Chebyshev nodes of a target
// and a source cluster, in FP64 or FP32, and the small complex type they are returned in.
#pragma once

#include <type_traits>

#include "internal.h"
#include "k_common.cuh"

namespace igabem {

template <class T> struct C2 {
  T x, y;
};
template <class T> __device__ inline C2<T> c2(T a, T b) { return {a, b}; }
template <class T> __device__ inline C2<T> add(C2<T> a, C2<T> b) { return {a.x + b.x, a.y + b.y}; }
template <class T> __device__ inline C2<T> mul(C2<T> a, C2<T> b) {
  return {a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x};
}
template <class T> __device__ inline C2<T> fma2(C2<T> a, C2<T> b, C2<T> acc) {  // acc + a b
  return {acc.x + a.x * b.x - a.y * b.y, acc.y + a.x * b.y + a.y * b.x};
}

__device__ inline float2 fma2x(float2 a, float2 b, float2 c) {  // two FP32 multiply-adds, a b + c
  float2 d;
  asm("fma.rn.f32x2 %0, %1, %2, %3;"
      : "=l"(reinterpret_cast<unsigned long long &>(d))
      : "l"(reinterpret_cast<const unsigned long long &>(a)), "l"(reinterpret_cast<const unsigned long long &>(b)),
        "l"(reinterpret_cast<const unsigned long long &>(c)));
  return d;
}

constexpr double TWO_PI = 6.283185307179586476925286766559;

// ---- FP64 arithmetic of the kernel samples -------------------------------------------------------
// The FP64 pipe is what bounds the FP64 product (a warp instruction of it holds a quarter of an SM for
// about 76 cycles; integer, FP32 and shared-memory instructions hide behind it), so these helpers count
// FP64 instructions: 1/sqrt in 5 and exp(i phi) in 9 + 4 (a complex product with the table entry).

// 1/sqrt(x), x a positive normal number: the single-precision estimate of the scaled argument (exponent
// handled by integer instructions), one step of Householder's third-order iteration (relative error of
// the estimate 2^-22, cubed).
__device__ inline double rsqrt64(double x) {
  const int hi = __double2hiint(x), lo = __double2loint(x);
  const int k = ((hi >> 20) - 1023) >> 1;           // x = m 4^k, m in [1, 4)
  const int hm = hi - (k << 21);
  float f;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(f) : "f"(__uint_as_float((unsigned)(hm - (896 << 20)) << 3 | (unsigned)lo >> 29)));
  const unsigned fb = __float_as_uint(f);
  const double y = __hiloint2double((int)(fb >> 3) + (896 << 20) - (k << 20), (int)(fb << 29));
  const double e = fma(-(x * y), y, 1.0);
  return fma(y, e * fma(e, 0.375, 0.5), y);
}

// 1 / x, x a normal number: the single-precision estimate y, one step of Householder's third-order iteration
// y (1 + r + r^2), r = 1 - x y (the relative error of the estimate 2^-23, cubed).
__device__ inline double rcp64(double x) {
  const int hi = __double2hiint(x), lo = __double2loint(x);
  const int e = ((hi >> 20) & 0x7FF) - 1023;       // x = m 2^e, |m| in [1, 2)
  const int hm = hi - (e << 20);
  float f;
  asm("rcp.approx.ftz.f32 %0, %1;"
      : "=f"(f)
      : "f"(__uint_as_float((hi & 0x80000000u) | ((unsigned)((hm & 0x7FFFFFFF) - (896 << 20)) << 3 | (unsigned)lo >> 29))));
  const unsigned fb = __float_as_uint(f);
  const double y = __hiloint2double((int)((fb & 0x80000000u) | (((fb & 0x7FFFFFFFu) >> 3) + (896u << 20))) - (e << 20),
                                    (int)(fb << 29));
  const double r = fma(-x, y, 1.0);
  return fma(y, fma(r, r, r), y);
}

// Table-driven exp(i kappa r) (Tang's method): kappa r = 2 pi (k + u) / CIS_N, |u| <= 1/2, so
// exp(i kappa r) = table[k] (1 + m1 + i s) with m1 + i s = exp(2 pi i u / CIS_N) - 1 by its series.  c0 + c1 is
// kappa CIS_N / (2 pi) in two doubles, so that u is correct to the rounding of r.
__device__ inline void phase64_scale(double kappa, double &c0, double &c1) {
  constexpr double CH = CIS_N / TWO_PI, CL = -CIS_N * 9.839338337591243e-18;  // CIS_N / (2 pi) = CH + CL
  c0 = kappa * CH;
  c1 = fma(kappa, CL, fma(kappa, CH, -c0));
}
struct Phase64 {
  double2 E;
  double m1, s;
};
__device__ inline Phase64 phase64(const double2 *__restrict__ tab, double r, double c0, double c1) {
  constexpr double M = 6755399441055744.0;          // 1.5 2^52: adding it rounds to an integer
  constexpr double T1 = TWO_PI / CIS_N;
  const double tm = fma(r, c0, M);
  const int k = __double2loint(tm) & (CIS_N - 1);
  double u = fma(r, c0, M - tm);
  u = fma(r, c1, u);
  const double u2 = u * u;
  Phase64 p;
  p.s = u * fma(u2, fma(u2, T1 * T1 * T1 * T1 * T1 / 120.0, -T1 * T1 * T1 / 6.0), T1);
  p.m1 = u2 * fma(u2, T1 * T1 * T1 * T1 / 24.0, -T1 * T1 / 2.0);
  p.E = tab[k];
  return p;
}
// p (1 + m1 + i s)
__device__ inline C2<double> phase_mul(double px, double py, const Phase64 &f) {
  return c2(fma(-py, f.s, fma(px, f.m1, px)), fma(px, f.s, fma(py, f.m1, py)));
}

// kappa d + phi0 less whole turns (2 pi in two floats), about [-pi, pi].  The phase rounds once, as much as kappa in FP32
// itself lets it; in turns, with kappa / (2 pi) rounded a second time, the rms error at kappa = 11, d up to 0.3 is
// 1.6e-7 instead of 0.9e-7.
__device__ inline float phase32(float kappa, float d, float phi0) {
  constexpr float M = 12582912.f;  // 1.5 2^23: adding it rounds to an integer
  const float ph = fmaf(kappa, d, phi0), turns = fmaf(ph, 0.15915494309189533577f, M) - M;
  return fmaf(-turns, -1.7484556e-07f, fmaf(-turns, 6.28318548202514648f, ph));
}

// sin(x) and cos(x) - 1, |x| < 1e6: reduced to |y| <= pi/4 about a multiple of pi/2, there the Taylor series (first terms
// left out: 2e-9 and 2e-10 at pi/4); for |x| < pi/4 both are accurate relative to themselves
__device__ inline void sin_cosm1(float x, float &sn, float &cm) {
  const float m = fmaf(x, 0.636619772f, 12582912.f), k = m - 12582912.f;  // 1.5 2^23: rounds to an integer
  const int n = __float_as_int(m);
  const float y = fmaf(-k, -4.37113883e-8f, fmaf(-k, 1.57079637f, x)), z = y * y;
  const float s = fmaf(y * z, fmaf(z, fmaf(z, fmaf(z, 1.f / 362880, -1.f / 5040), 1.f / 120), -1.f / 6), y);
  const float c = z * fmaf(z, fmaf(z, fmaf(z, fmaf(z, -1.f / 3628800, 1.f / 40320), -1.f / 720), 1.f / 24), -0.5f),
              c1 = 1.f + c;
  const float a = n & 1 ? c1 : s, b = n & 1 ? s : c1;
  sn = n & 2 ? -a : a;
  cm = n & 3 ? ((n + 1) & 2 ? -b : b) - 1.f : c;
}

// s + l += v, l the rounding errors of s (Knuth's two-sum)
__device__ inline void two_sum(float &s, float &l, float v) {
  const float t = s + v, b = t - s;
  l += (s - (t - b)) + (v - b);
  s = t;
}

// Sample of one node pair in precision T: returns the kernel value of the requested type.
//   type 0: soft  a_y G'(r)/r (x-y).n~x - i eta a_x a_y G
//   type 1: hard  a_x G'(r)/r (y-x).n~y
//   type 2: hard  G
// x, y: FP64 absolute node positions (FP64 path) or offsets from the cluster centres (FP32 path,
// with the pair constants D, |D|, |D|^2; the pair factor exp(i kappa |D|) is applied by the caller).
template <class T>
__device__ inline C2<T> node_sample(int type, const T *x, const T *nx, T ax, const T *y, const T *ny, T ay,
                                    const T *D, T Dn, T D2, T kappa, T eta) {
  constexpr bool F32 = std::is_same<T, float>::value;
  T d0 = x[0] - y[0], d1 = x[1] - y[1], d2 = x[2] - y[2];
  T r2, ir, r, cph, sph, dn_x, dn_y;
  if constexpr (F32) {
    T Dd = D[0] * d0 + D[1] * d1 + D[2] * d2;
    T dd = d0 * d0 + d1 * d1 + d2 * d2;
    T num = (T)2 * Dd + dd;
    r2 = D2 + num;
    ir = rsqrtf(r2);
    r = r2 * ir;
    T ph = kappa * __fdividef(num, r + Dn);
    T kq = rintf(ph * 0.15915494309189535f);
    ph = fmaf(-kq, 6.28318548202514648f, ph);
    ph = fmaf(-kq, -1.7484556e-07f, ph);
    __sincosf(ph, &sph, &cph);
    dn_x = D[0] * nx[0] + D[1] * nx[1] + D[2] * nx[2] + d0 * nx[0] + d1 * nx[1] + d2 * nx[2];
    dn_y = D[0] * ny[0] + D[1] * ny[1] + D[2] * ny[2] + d0 * ny[0] + d1 * ny[1] + d2 * ny[2];
  } else {
    r2 = d0 * d0 + d1 * d1 + d2 * d2;
    ir = rsqrt(r2);
    r = r2 * ir;
    sincos(kappa * r, &sph, &cph);
    dn_x = d0 * nx[0] + d1 * nx[1] + d2 * nx[2];
    dn_y = d0 * ny[0] + d1 * ny[1] + d2 * ny[2];
  }
  const T f = ir * (T)(0.25 / IGA_PI), kr = kappa * r, g2 = f * ir * ir;
  const C2<T> G = c2(cph * f, sph * f);
  if (type == 2) return G;
  const C2<T> dG = c2((-cph - sph * kr) * g2, (-sph + cph * kr) * g2);
  if (type == 1) {
    T w1 = -ax * dn_y;
    return c2(dG.x * w1, dG.y * w1);
  }
  T w1 = ay * dn_x, w2 = ax * ay * eta;
  return c2(dG.x * w1 + G.y * w2, dG.y * w1 - G.x * w2);
}

}  // namespace igabem
