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
//
// Away from the centre G falls by up to e^(i / sigma^2) across a pixel, and on the far side E - f O
// would be the small difference of large numbers: at sigma = 1 the rounding of the sums came to 1.6
// times the renderer's bound (1e-6 of the pixel) four widths out.  From pixel kPolyWing on the table
// therefore holds G without that slope,
//
//   T(f) = G(i + f) 2^(f k_i),   k_i = log2(e) i / sigma^2  (poly_wing_rate),
//
// which varies by a few tens of a percent and needs a term less, and the kernel multiplies
// T(f) = E + f O and T(-f) = E - f O (with the weight) by 2^(-f k_i) and 2^(f k_i).  Worst of 3072
// single stamps, K = 11, in parts of the bound: 1.64, 1.37, 1.02, 1.03 at sigma = 1.0, 1.1, 1.2, 1.3
// as a plain E - f O, 0.64, 0.54, 0.52, 0.44 so (the edge tails 0.64, 0.72, 0.85, 0.84).
#pragma once
#include "e2e_device.cuh"

namespace e2e {

constexpr int kPolyTerms = 5;                   // coefficients of E and of O per pixel pair, at most
constexpr int kPolyDegree = 2 * kPolyTerms - 1;
constexpr double kPolyMinSigma = 1.0;           // narrowest PSF the degree serves (px)
constexpr int kPolyWing = 3;                    // pixels from the centre on that go without their slope

// The K/2 + 1 pixel pairs of an axis (the centre pixel pairs with itself) are dealt to the two
// lanes that evaluate it: lane half h takes pairs h, h + 2, ..., the outermost pair first.
__host__ __device__ constexpr int poly_slots(int K) { return (K / 2 + 2) / 2; }
// Slots whose first (half 0) pixel is a wing pixel, and a slot's terms: one less where both are.
__host__ __device__ constexpr bool poly_wing(int K, int slot) { return K / 2 - 2 * slot >= kPolyWing; }
__host__ __device__ constexpr int poly_terms(int K, int slot) {
  return K / 2 - 1 - 2 * slot >= kPolyWing ? kPolyTerms - 1 : kPolyTerms;
}
// (E, O) pairs before a slot's, and float4s of one lane's coefficients
__host__ __device__ constexpr int poly_at(int K, int slot) {
  int n = 0;
  for (int s = 0; s < slot; ++s) n += poly_terms(K, s);
  return n;
}
__host__ __device__ constexpr int poly_role_f4(int K) { return (poly_at(K, poly_slots(K)) + 1) / 2; }

// k_i in log2 units from g = sqrt(log2 e) / (sqrt 2 sigma), the sample table's FP32 constant: the
// table is built for the rounded value that the kernel forms.
__device__ __forceinline__ float poly_wing_rate(float g, int i) { return __fmul_rn((float)(2 * i), __fmul_rn(g, g)); }

}  // namespace e2e
