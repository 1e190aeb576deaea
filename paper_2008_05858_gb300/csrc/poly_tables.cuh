// Pixel integrals of the separable Gaussian PSF as polynomials in the sub-pixel offset.
//
// All slit points of one wavelength sample share the sample's widths, so their profiles differ
// only in the offset f of the stamp's centre from its window-centre pixel (|f| <= 1/2).  Window
// pixel m, i = K/2 - m >= 0 pixels left of the centre pixel, integrates the PSF to
// G(i + f), G(x) = Phi((x + 1/2)/sigma) - Phi((x - 1/2)/sigma), its mirror image K-1-m to
// G(i - f).  Per sample, axis and pixel pair the table holds the polynomial of degree
// kPolyDegree of G(i + f) in f, as its even and odd parts
//
//   G(i +- f) ~= E(f^2) +- f O(f^2),   E, O of kPolyTerms coefficients each,
//
// the Taylor series about f = 0 (derivatives of G are differences of Hermite functions at the
// pixel's edges) to degree 17, truncated to kPolyDegree in Chebyshev form on [-1/2, 1/2].  For
// sigma >= kPolyMinSigma the truncation is below 3e-8 of G + 1e-4 G(0) (7e-9 at sigma = 1.2);
// evaluated in FP32, the profile's rms error is 3e-8 to 7e-8, below that of the edge tails
// (phi32.cuh: 1.2e-7), because no tails are subtracted.
#pragma once
#include "e2e_device.cuh"

namespace e2e {

constexpr int kPolyTerms = 5;                   // coefficients of E and of O per pixel pair
constexpr int kPolyDegree = 2 * kPolyTerms - 1;
constexpr double kPolyMinSigma = 1.0;           // narrowest PSF the degree serves (px)

// The K/2 + 1 pixel pairs of an axis (the centre pixel pairs with itself) are dealt to the two
// lanes that evaluate it: lane half h takes pairs h, h + 2, ...
__host__ __device__ constexpr int poly_slots(int K) { return (K / 2 + 2) / 2; }
// float4s of one lane's coefficients: per slot kPolyTerms (E, O) pairs
__host__ __device__ constexpr int poly_role_f4(int K) { return (poly_slots(K) * kPolyTerms * 2 + 3) / 4; }

}  // namespace e2e
