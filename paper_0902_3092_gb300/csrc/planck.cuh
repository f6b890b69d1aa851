// planck.cuh -- Planck function integrated over wavelength bins, host and device (FP64).
//
// int_bin B_nu(T) dnu = (2 k^4 T^4 / (h^3 c^2)) [F3(x_hi) - F3(x_lo)],  F3(x) = int_0^x t^3/(e^t-1) dt,
// int_bin dB_nu/dT dnu = (2 k^4 T^3 / (h^3 c^2)) [F4(x_hi) - F4(x_lo)], F4(x) = int_0^x t^4 e^t/(e^t-1)^2 dt,
// with x = h nu / (k T). For x <= 2, F3 is the power series of the Bernoulli numbers (Abramowitz & Stegun 27.1.1 for
// n = 3; convergent for x < 2 pi, 17 terms leave 1e-17 at x = 2), and so is F4 = 4 F3 - x^4/(e^x - 1) (by parts); above,
// the complement int_x^inf t^3/(e^t - 1) dt is summed over int t^3 e^{-nt} dt (27.1.2).
// The first bin extends to lambda -> 0 and the last to infinity.
//
// FP64 arithmetic bounds the kernels that use them (1.25 TFLOP/s on this GPU): about 25 operations per edge against
// several hundred for a quadrature with 20 exponentials or a sum with a division per term.
#pragma once
#include <cmath>

#include "lanes.cuh"

namespace mcrt {

constexpr double kH = 6.62607015e-27;
constexpr double kC = 2.99792458e10;
constexpr double kKB = 1.380649e-16;
// 2 pi^5 k^4 / (15 h^3 c^2)
#define MCRT_SIGMA (2.0 * 3.14159265358979323846 * 3.14159265358979323846 * 3.14159265358979323846 * \
                    3.14159265358979323846 * 3.14159265358979323846 * kKB * kKB * kKB * kKB /       \
                    (15.0 * kH * kH * kH * kC * kC))

// Tail integrals from x to infinity, G3 and, with BOTH, G4 (from the same pass).
template <bool BOTH>
__host__ __device__ inline void tails_of(double x, double& g3, double& g4) {
  const double pi4 = 3.14159265358979323846 * 3.14159265358979323846 * 3.14159265358979323846 *
                     3.14159265358979323846;
  if (!(x > 0.0)) {
    g3 = pi4 / 15.0;
    g4 = 4.0 * pi4 / 15.0;
    return;
  }
  if (x > 2.0) {
    const double e1 = exp(-x);
    double e = e1, s = 0.0;
#pragma unroll
    for (int n = 1; n <= 22; ++n) {  // (the terms fall by e^-x < 0.14 each: the 22nd is below 1e-19 of the sum)
      const double X = (double)n * x, q = 1.0 / ((double)n * n * n * n);
      const double t = e * q * (((X + 3.0) * X + 6.0) * X + 6.0);
      s += t;
      if (t <= 1e-18 * s) break;  // (also where exp(-x) underflows to 0)
      e *= e1;
    }
    g3 = s;
    if (BOTH) g4 = 4.0 * s + x * x * x * x * (e1 / (1.0 - e1));  // by parts
    return;
  }
  const double x2 = x * x, x3 = x2 * x;
  double p = 3.9328985827428781132e-29;  // B_2j / ((2j)! (2j + 3)), j = 17 .. 1
  p = p * x2 + -1.6413687625349149844e-27;
  p = p * x2 + 6.8725831889020698797e-26;
  p = p * x2 + -2.8882314280766280163e-24;
  p = p * x2 + 1.2188644964239543006e-22;
  p = p * x2 + -5.1683202540046382743e-21;
  p = p * x2 + 2.2036011313440918061e-19;
  p = p * x2 + -9.4559508632959211871e-18;
  p = p * x2 + 4.0886009791799259829e-16;
  p = p * x2 + -1.7840422612224120352e-14;
  p = p * x2 + 7.8720803121674581370e-13;
  p = p * x2 + -3.5227934257916621232e-11;
  p = p * x2 + 1.6059043836821614599e-9;
  p = p * x2 + -7.5156325156325156325e-8;
  p = p * x2 + 3.6743092298647854203e-6;
  p = p * x2 + -0.00019841269841269841270;
  p = p * x2 + 0.016666666666666666667;
  g3 = pi4 / 15.0 - x3 * (1.0 / 3.0 - 0.125 * x + x2 * p);
  if (!BOTH) return;
  p = -1.2978565323051497773e-27;  // B_2j / (2j)! (1 - 2j) / (2j + 3)
  p = p * x2 + 5.0882431638582364515e-26;
  p = p * x2 + -1.9930491247816002651e-24;
  p = p * x2 + 7.7982248558068956439e-23;
  p = p * x2 + -3.0471612410598857515e-21;
  p = p * x2 + 1.1887136584210668031e-19;
  p = p * x2 + -4.6275623758225927928e-18;
  p = p * x2 + 1.7966306640262250256e-16;
  p = p * x2 + -6.9506216646058741710e-15;
  p = p * x2 + 2.6760633918336180528e-13;
  p = p * x2 + -1.0233704405817695578e-11;
  p = p * x2 + 3.8750727683708283356e-10;
  p = p * x2 + -1.4453139453139453139e-8;
  p = p * x2 + 5.2609427609427609428e-7;
  p = p * x2 + -0.000018371546149323927102;
  p = p * x2 + 0.00059523809523809523810;
  p = p * x2 + -0.016666666666666666667;
  g4 = 4.0 * pi4 / 15.0 - x3 * (1.0 / 3.0 + x2 * p);
}
__host__ __device__ inline void tails(double x, double& g3, double& g4) { tails_of<true>(x, g3, g4); }
__host__ __device__ inline double tail3(double x) {
  double g3, g4;
  tails_of<false>(x, g3, g4);
  return g3;
}

// Bbar_b(T) and dBbar_b/dT for all bins; lam_e in micron (nlam+1 edges). Either output may be null.
__host__ __device__ inline void planck_bins(const double* lam_e, int nlam, double T, double* B, double* dB) {
  if (!(T > 0.0)) {
    for (int b = 0; b < nlam; ++b) {
      if (B) B[b] = 0.0;
      if (dB) dB[b] = 0.0;
    }
    return;
  }
  const double k4 = kKB * kKB * kKB * kKB;
  const double pref3 = 2.0 * k4 * T * T * T * T / (kH * kH * kH * kC * kC);
  const double pref4 = 2.0 * k4 * T * T * T / (kH * kH * kH * kC * kC);
  double g3p = 0.0, g4p = 0.0;  // tails at edge 0 (lambda -> 0, x -> inf)
  for (int b = 0; b < nlam; ++b) {
    double g3, g4;
    if (b + 1 == nlam) {
      tails(0.0, g3, g4);
    } else {
      const double x = kH * kC / (lam_e[b + 1] * 1e-4 * kKB * T);
      tails(x, g3, g4);
    }
    if (B) B[b] = pref3 * (g3 - g3p);
    if (dB) dB[b] = pref4 * (g4 - g4p);
    g3p = g3;
    g4p = g4;
  }
}

// Rosseland mean of chi' = kappa + (1-g) sigma at T (Eq. 3 with Eq. 16), exact bin integrals; the lanes of g take the bins
// side by side (a bin's short edge is its neighbour lane's long one), the result is in all of them.
template <class Group>
__host__ __device__ inline double rosseland_group(const Group& g, const double* __restrict__ lam_e,
                                                  const double* __restrict__ chip, int nlam, double T) {
  const double hx = kH * kC / (1e-4 * kKB * T);
  double s1 = 0.0, s2 = 0.0, g4p = 0.0;  // (the tail at the first bin's short edge, lambda -> 0, is 0)
  for (int b0 = 0; b0 < nlam; b0 += g.size()) {
    const int b = b0 + g.lane();
    double g3, g4 = 0.0;
    if (b < nlam) tails(b + 1 == nlam ? 0.0 : hx / lam_e[b + 1], g3, g4);
    const double a4 = g.below(g4, g4p);
    if (b < nlam) {
      s1 += g4 - a4;
      s2 += (g4 - a4) / chip[b];
    }
    g4p = g.last(g4);
  }
  s1 = g.sum(s1);
  s2 = g.sum(s2);
  return s1 / s2;
}
__host__ __device__ inline double rosseland(const double* lam_e, const double* chip, int nlam, double T) {
  return rosseland_group(OneLane(), lam_e, chip, nlam, T);
}

}  // namespace mcrt
