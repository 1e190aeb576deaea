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
// Truncated at degree 10 the series is below 4e-8 of I + 1e-4 I(0) at widths 1.2 px.
//
// A pixel on the far side of a run's stamps is the small difference of large terms (of e^4 times its
// size at 1.3 px, four widths out along a diagonal), so the large terms are kept to more than FP32:
// the moments are summed with their rounding errors (FastTwoSum), the six of degree <= 2 are handed
// on in two words, and the pixel's terms of those degrees are summed with their errors.  What is left
// in FP32, the coefficients above all, sets kEllMinSigma.  Worst pixel of 3072 single stamps 1.3, 1.4,
// 1.5 and 1.8 px wide, K = 13, in parts of the renderer's bound (1e-6 of the pixel): 0.70, 0.72, 0.53,
// 0.45 (1.88, 1.27, 1.05, 0.66 with every sum in FP32, and 3.5 at 1.3 px for a run of 100 stamps on
// one side of its pixel; stamp by stamp 0.81, 0.87, 0.85, 0.95).
#pragma once
#include "e2e_device.cuh"

namespace e2e {

constexpr int kEllDegree = 10;
constexpr int kEllTerms = (kEllDegree + 1) * (kEllDegree + 2) / 2;          // 66
constexpr int kEllEven = (kEllDegree / 2 + 1) * (kEllDegree / 2 + 1);       // 36: degrees 0, 2, .. 10
constexpr int kEllRuns = 12;                                                // runs a warp turns into pixels at once
constexpr double kEllMinSigma = 1.3;                                        // narrowest PSF served (px)
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

// The terms of degree <= 2 (the first of either parity), whose moments have low words: their rows.
constexpr int kEllLowEven = 4, kEllLowOdd = 2, kEllLow = kEllLowEven + kEllLowOdd;
__host__ __device__ constexpr int ell_low_row(int term) {  // kEllLow: none
  return term < kEllLowEven ? term : term >= kEllEven && term < kEllEven + kEllLowOdd ? kEllLowEven + term - kEllEven : kEllLow;
}

// Items of one slice and one interval between nodes, rendered by one CTA.
struct EllGroup {
  int32_t first, count;  // items, relative to the launch's
  int32_t interval;      // nodes interval - 1 .. interval + 2 (numbered from -1)
  int32_t pad;
};

}  // namespace e2e
