// Pixel integrals of the rotated Gaussian PSF as polynomials in the two sub-pixel offsets.
//
// The stamps of one wavelength sample share its covariance, so the integral over window pixel
// (m, n) is one function of the stamp's offsets (fx, fy) in its window-centre pixel,
// |fx|, |fy| <= 1/2, and the stamps of a run (slit points with the same window) add up to
//
//   sum_k w_k I_mn(fx_k, fy_k) = sum_ab C_ab(m, n) M_ab,   M_ab = sum_k w_k T_a(2 fx_k) T_b(2 fy_k),
//
// C the Chebyshev coefficients of I_mn, a + b <= kEllDegree.  A stamp costs its kEllTerms moments;
// the K^2 pixels are formed once per run.  Opposite pixels of the window are mirror images,
// I_(K-1-m, K-1-n)(fx, fy) = I_mn(-fx, -fy): the table holds one of each pair, and the terms with
// a + b even (first, kEllEven of them) and odd give the two as a sum and a difference.
//
// C varies with the wavelength only through the widths.  It is tabulated at nodes along the slice
// (every `span` samples, one more beyond either end) and interpolated by the cubic through four
// nodes; the plan takes the span from the widths' slope and curvature so that the interpolation errs
// by less than kEllInterp of a pixel four widths from the centre (and far less of brighter ones).
// Truncated at degree 10 the series is below 4e-8 of I + 1e-4 I(0) at widths 1.2 px, 3e-7 at 1.0 px
// (the window's corners; 1e-9 of the peak).
#pragma once
#include "e2e_device.cuh"

namespace e2e {

constexpr int kEllDegree = 10;
constexpr int kEllTerms = (kEllDegree + 1) * (kEllDegree + 2) / 2;          // 66
constexpr int kEllEven = (kEllDegree / 2 + 1) * (kEllDegree / 2 + 1);       // 36: degrees 0, 2, .. 10
constexpr int kEllRuns = 12;                                                // runs a warp turns into pixels at once
constexpr double kEllMinSigma = 1.0;                                        // narrowest PSF the degree serves (px)
constexpr double kEllInterp = 2e-7;                                         // interpolation error, four widths out
constexpr int kEllMaxSlit = 128;                                            // slit points per item

// Pixel pairs of a K x K window (the centre pairs with itself), and per lane of a warp.
__host__ __device__ constexpr int ell_pairs(int K) { return (K * K + 1) / 2; }
__host__ __device__ constexpr int ell_slots(int K) { return (ell_pairs(K) + 31) / 32; }

// Place of term (a, b): the even degrees first, by degree, then b.
__host__ __device__ constexpr int ell_term(int a, int b) {
  const int t = a + b;
  return (t & 1) ? kEllEven + (t / 2) * (t / 2 + 1) + b : (t / 2) * (t / 2) + b;
}

// Items of one slice and one interval between nodes, rendered by one CTA.
struct EllGroup {
  int32_t first, count;  // items, relative to the launch's
  int32_t interval;      // nodes interval - 1 .. interval + 2 (numbered from -1)
  int32_t pad;
};

}  // namespace e2e
