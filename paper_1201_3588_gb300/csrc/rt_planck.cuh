// rt_planck.cuh -- FP64 Planck integrals over frequency bins and the temperature
// grid of the tables (device functions shared by the table builders).
//
// The Planck function integrated over a frequency bin is evaluated in closed
// form: with x = h nu / k T, the integral of B_nu over [nu0, nu1] equals
// (2 k^4 T^4 / h^3 c^2) [G(x0) - G(x1)], G(x) the integral of t^3/(e^t - 1) from x
// to infinity, summed as sum_k e^{-kx} (x^3/k + 3x^2/k^2 + 6x/k^3 + 6/k^4) for
// x >= 2 and as pi^4/15 minus the Bernoulli series of the integral from 0 to x
// below that.
//
// GB300 retires two FP64 operations per SM and clock, so the number of FP64
// operations is what these tables cost. Both series are polynomials (no division and
// one exponential per edge: the powers of e^{-x} are multiplied up), the split at
// x = 2 bounds them by 17 and 21 terms, and the callers evaluate every bin edge once
// and difference neighbours (planck_between). A form with exp and four divisions per
// term and a split at 1/2 took 1.0 ms for a 1024 x 100 table, this one 0.06 ms; against
// 40-digit quadrature its worst relative error over 200 bins and x = 0.02 .. 100 is
// 2e-14 (the other: 9e-13).
#pragma once

#include <math.h>

namespace rt {
namespace planck {

constexpr double kH = 6.62607015e-27;
constexpr double kK = 1.380649e-16;
constexpr double kC = 2.99792458e10;
constexpr double kPi = 3.14159265358979323846;
constexpr double kPi4Over15 = 6.4939394022668291491;  // pi^4 / 15

constexpr double kSplit = 2.0;  // x below it: the series from 0

// B_{2k+2} / ((2k+2)! (2k+5)), k = 0 .. 16 (B_n the Bernoulli numbers)
static __constant__ double kBernoulli[17] = {
    0.016666666666666666,    -0.0001984126984126984,  3.6743092298647855e-06,
    -7.515632515632516e-08,  1.6059043836821615e-09,  -3.522793425791662e-11,
    7.872080312167458e-13,   -1.784042261222412e-14,  4.088600979179926e-16,
    -9.455950863295921e-18,  2.203601131344092e-19,   -5.1683202540046385e-21,
    1.2188644964239542e-22,  -2.888231428076628e-24,  6.87258318890207e-26,
    -1.641368762534915e-27,  3.9328985827428784e-29};

// 1/k, k = 1 .. 21 (entry 0 unused)
static __constant__ double kInverse[22] = {
    0.0,      1.0,      1.0 / 2,  1.0 / 3,  1.0 / 4,  1.0 / 5,  1.0 / 6,  1.0 / 7,
    1.0 / 8,  1.0 / 9,  1.0 / 10, 1.0 / 11, 1.0 / 12, 1.0 / 13, 1.0 / 14, 1.0 / 15,
    1.0 / 16, 1.0 / 17, 1.0 / 18, 1.0 / 19, 1.0 / 20, 1.0 / 21};

// integral_0^x t^3/(e^t-1) dt for 0 <= x < 2. Below 1/2 eight terms of the series
// reach the last bit, (x / 2 pi)^16 = 2e-18.
static __device__ inline double planck_head(double x) {
  const double x2 = x * x;
  double s;
  if (x < 0.5) {
    s = kBernoulli[7];
#pragma unroll
    for (int k = 6; k >= 0; --k) s = fma(s, x2, kBernoulli[k]);
  } else {
    s = kBernoulli[16];
#pragma unroll
    for (int k = 15; k >= 0; --k) s = fma(s, x2, kBernoulli[k]);
  }
  return x * x2 * (fma(s, x2, -0.125 * x) + 1.0 / 3.0);
}

// integral_x^inf t^3/(e^t-1) dt for x >= 2: terms up to e^{-39} of the first
static __device__ inline double planck_tail(double x) {
  if (!(x < 746.0)) return 0.0;  // e^{-x} underflows
  const double q = exp(-x);
  const int n = min((int)(39.0f / (float)x) + 2, 21);
  const double x2 = x * x, x3 = x2 * x, t2 = 3.0 * x2, t1 = 6.0 * x;
  double e = q, s = 0.0;
  for (int k = 1; k <= n; ++k) {
    const double r = kInverse[k];
    s = fma(e, r * fma(r, fma(r, fma(r, 6.0, t1), t2), x3), s);
    e *= q;
  }
  return s;
}

// one bin edge at x: the integral from 0 below the split, to infinity above it
static __device__ inline double planck_edge(double x) {
  return x < kSplit ? planck_head(x) : planck_tail(x);
}

// integral from x0 to x1 > x0 out of their edge values (>= 0)
static __device__ inline double planck_between(double x0, double e0, double x1, double e1) {
  const double d = x1 < kSplit ? e1 - e0 : (x0 < kSplit ? (kPi4Over15 - e0) - e1 : e0 - e1);
  return d > 0.0 ? d : 0.0;
}

static __device__ inline double planck_factor(double T) {
  const double kT = kK * T;
  return 2.0 * kT * kT * kT * kT / (kH * kH * kH * kC * kC);
}

// integral over [nu0, nu1] of B_nu(T) d nu, erg s^-1 cm^-2 sr^-1
static __device__ inline double planck_bin(double nu0, double nu1, double T) {
  if (!(T > 0.0)) return 0.0;
  const double a = kH / (kK * T);
  const double x0 = a * nu0, x1 = a * nu1;
  return planck_factor(T) * planck_between(x0, planck_edge(x0), x1, planck_edge(x1));
}

// One warp: f(b, integral of B_nu(T) over bin b) for every bin b = 0 .. B-1, each in
// one lane, in chunks of 31 bins (32 edges, one per lane; the upper edge of a lane's
// bin is the next lane's). All lanes of the warp call it with the same arguments.
template <typename F>
static __device__ inline void planck_bins_warp(const double* nu, int B, double T, F f) {
  const int lane = threadIdx.x & 31;
  const double a = T > 0.0 ? kH / (kK * T) : 0.0;
  const double pref = T > 0.0 ? planck_factor(T) : 0.0;
  for (int b0 = 0; b0 < B; b0 += 31) {
    const int b = b0 + lane;
    const double x0 = a * nu[min(b, B)];
    const double e0 = T > 0.0 ? planck_edge(x0) : 0.0;
    const double x1 = __shfl_down_sync(0xffffffffu, x0, 1);
    const double e1 = __shfl_down_sync(0xffffffffu, e0, 1);
    if (lane < 31 && b < B) f(b, T > 0.0 ? pref * planck_between(x0, e0, x1, e1) : 0.0);
  }
}

static __device__ inline double table_T(int i, int n_T, double t_min, double t_max) {
  if (i == 0) return 0.0;
  if (i == n_T - 1) return t_max;
  return t_min * pow(t_max / t_min, (double)(i - 1) / (double)(n_T - 2));
}

}  // namespace planck
}  // namespace rt
