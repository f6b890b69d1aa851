// temperature.cuh -- the radiative-equilibrium temperature of a cell (Sect. 2.1): the T that solves
// Q(T) = 4 pi sum_b kappa_b Bbar_b(T) = q, q the absorbed luminosity per unit mass, in FP64 on the exact
// bin integrals. Host and device code (the temperature kernel; compiled for the host in the tests too).
#pragma once
#include <cmath>

#include "common.cuh"
#include "planck.cuh"

namespace mcrt {

// Q(T) and dQ/dT (erg s^-1 g^-1 and per K) from the bin integrals of Bbar and of T dBbar/dT; the lanes of g take the bins side
// by side (a bin's short edge is its neighbour lane's long one), the result is in all of them.
template <class Group>
__host__ __device__ inline void q_sum_group(const Group& g, const double* __restrict__ lam_e, const double* __restrict__ kabs,
                                            int nlam, double T, double& Q, double& dQ) {
  const double pref = 8.0 * kPi * kKB * kKB * kKB * kKB / (kH * kH * kH * kC * kC);
  const double hx = kH * kC / (1e-4 * kKB * T);
  double s3 = 0.0, s4 = 0.0, g3p = 0.0, g4p = 0.0;  // sums over the bins of kappa dG3, kappa dG4
  for (int b0 = 0; b0 < nlam; b0 += g.size()) {
    const int b = b0 + g.lane();
    double g3 = 0.0, g4 = 0.0;
    if (b < nlam) tails(b + 1 == nlam ? 0.0 : hx / lam_e[b + 1], g3, g4);
    const double a3 = g.below(g3, g3p), a4 = g.below(g4, g4p);
    if (b < nlam) {
      s3 += kabs[b] * (g3 - a3);
      s4 += kabs[b] * (g4 - a4);
    }
    g3p = g.last(g3);
    g4p = g.last(g4);
  }
  const double p3 = pref * T * T * T;
  Q = p3 * T * g.sum(s3);
  dQ = p3 * g.sum(s4);
}
__host__ __device__ inline void q_sum(const double* lam_e, const double* kabs, int nlam, double T, double& Q, double& dQ) {
  q_sum_group(OneLane(), lam_e, kabs, nlam, T, Q, dQ);
}

// The T of the tabulated grid for Q(T) = q > 0 (lQk: log Q(T_k), slQ: d log Q / d log T at T_k, T_k = Tmin exp((k-1)
// dlnT), k >= 1): log T as a cubic Hermite function of log Q between the two grid temperatures that bracket q
// (slopes d log T / d log Q from the table; beyond the grid Q ~ T^4). Within 2e-11 of the root on the grid.
__host__ __device__ inline double temperature_guess(double q, const double* lQk, const double* slQ, int nT, double Tmin,
                                                    double dlnT) {
  const double lq = log(q);
  double Tk;
  if (lq < lQk[1]) {
    Tk = Tmin * exp(0.25 * (lq - lQk[1]));
  } else if (lq >= lQk[nT - 1]) {
    Tk = Tmin * exp((nT - 2) * dlnT) * exp(0.25 * (lq - lQk[nT - 1]));
  } else {
    int lo_k = 1, hi_k = nT - 1;  // lQk[lo_k] <= lq < lQk[hi_k]
    while (hi_k - lo_k > 1) {
      const int mid = (lo_k + hi_k) >> 1;
      if (lQk[mid] <= lq) lo_k = mid; else hi_k = mid;
    }
    const double x0 = lQk[lo_k], x1 = lQk[lo_k + 1], h = x1 - x0;
    const double y0 = (lo_k - 1) * dlnT, y1 = lo_k * dlnT;
    const double m0 = 1.0 / slQ[lo_k], m1 = 1.0 / slQ[lo_k + 1];
    double y = y0;
    if (h > 0) {
      const double t = (lq - x0) / h, t2 = t * t, t3 = t2 * t;
      y = (2 * t3 - 3 * t2 + 1) * y0 + (t3 - 2 * t2 + t) * h * m0 + (-2 * t3 + 3 * t2) * y1 + (t3 - t2) * h * m1;
    }
    Tk = Tmin * exp(y);
  }
  return Tk;
}

// One Newton step of the bracketed search from x, with Q and dQ/dT there (lo, hi: the bracket). True: xn is the root
// to rounding. Q is smooth and increasing in T, so a step of relative size s leaves a relative error of order s^2:
// below 1e-8 the new point is the root (this also ends a guess that is the root already, where f may be 0 and the
// step would not lie strictly inside the bracket).
__host__ __device__ inline bool newton_step(double q, double Q, double dQ, double x, double& lo, double& hi, double& xn) {
  const double f = Q - q;
  if (f > 0) hi = x; else lo = x;
  xn = x - f / dQ;
  if (fabs(xn - x) <= 1e-8 * x) return true;
  if (!(xn > lo && xn < hi)) xn = isinf(hi) ? 2.0 * x : 0.5 * (lo + hi);
  return fabs(xn - x) <= 1e-15 * x;
}

// T with Q(T) = q > 0 by bracketed Newton from x (the tabulated grid's T)
template <class Group>
__host__ __device__ inline double temperature_root(const Group& g, double q, double x, int nlam, const double* __restrict__ lam_e,
                                                   const double* __restrict__ kabs) {
  double lo = 0.0, hi = INFINITY;
  for (int it = 0; it < 100; ++it) {
    double Q, dQ, xn;
    q_sum_group(g, lam_e, kabs, nlam, x, Q, dQ);
    const bool done = newton_step(q, Q, dQ, x, lo, hi, xn);
    x = xn;
    if (done) break;
  }
  return x;
}

// T with Q(T) = q > 0: gray dust in closed form
__host__ __device__ inline double cell_temperature(double q, int gray, double kabs0, int nlam, const double* lam_e,
                                                   const double* kabs, const double* lQk, const double* slQ, int nT,
                                                   double Tmin, double dlnT) {
  if (gray) return pow(q / (4.0 * MCRT_SIGMA * kabs0), 0.25);
  return temperature_root(OneLane(), q, temperature_guess(q, lQk, slQ, nT, Tmin, dlnT), nlam, lam_e, kabs);
}

}  // namespace mcrt
