// Builds the per-sample polynomial tables of the pixel integrals (poly_tables.cuh), once per
// model and after an update of its coefficients.
//
// One thread per (slice, sample, axis).  The Gaussian at the pixel edges and centres is formed
// in FP64 from one exponential (exp(-m^2 / 8 sigma^2) by a product recurrence: two
// multiplications per half pixel), because its error would scale every coefficient; the Hermite
// recurrences and their differences (pixels near the centre), the Gauss-Legendre sums (wing
// pixels) and the Chebyshev truncation run in FP32, where they add a few 1e-8: the table of a
// 2.04e6-sample model (K = 11) costs 1.4 ms instead of ~10 ms all in FP64.
#include "e2e_kernels.h"
#include "poly_tables.cuh"
#include "quad_coeffs.h"

namespace e2e {

constexpr int kTaylorMax = 17;
constexpr int kWingTaylor = 12;

// Chebyshev truncation on |f| <= 1/2: f^n (n = 10..17) ~= sum over j = n mod 2, +2, ... <= 9 of
// kChebCut[n - 10][j / 2] f^j (the expansion of f^n in T_k(2f), cut after k = 9; exact dyadic
// fractions).
__device__ constexpr float kChebCut[8][kPolyTerms] = {
    {1.9073486328125e-06f, -0.0003814697265625f, 0.01220703125f, -0.13671875f, 0.625f},
    {1.049041748046875e-05f, -0.0008392333984375f, 0.018798828125f, -0.171875f, 0.6875f},
    {1.3113021850585938e-06f, -0.00025177001953125f, 0.0075531005859375f, -0.0751953125f, 0.2578125f},
    {7.748603820800781e-06f, -0.0005950927734375f, 0.0124969482421875f, -0.1015625f, 0.3046875f},
    {5.811452865600586e-07f, -0.00010848045349121094f, 0.003124237060546875f, -0.0291595458984375f, 0.0888671875f},
    {3.632158041000366e-06f, -0.00027120113372802734f, 0.005467414855957031f, -0.041656494140625f,
     0.111083984375f},
    {2.1187588572502136e-07f, -3.8743019104003906e-05f, 0.0010848045349121094f, -0.0097198486328125f,
     0.02777099609375f},
    {1.3853423297405243e-06f, -0.00010132789611816406f, 0.0019860267639160156f, -0.0145263671875f,
     0.03631591796875f}};

// Normalised derivatives h_k = phi_sigma^(k)(x) (-1)^k / k! at x, k = 0..kTaylorMax - 1:
// h_(k+1) = (x h_k - h_(k-1)) / (sigma^2 (k + 1)).
__device__ __forceinline__ void hermite_edge(float phi, float xa2, float a2, float (&h)[kTaylorMax]) {
  h[0] = phi;
  float prev = 0.f;
#pragma unroll
  for (int k = 0; k + 1 < kTaylorMax; ++k) {
    h[k + 1] = fmaf(xa2, h[k], -a2 * prev) * (1.f / (float)(k + 1));
    prev = h[k];
  }
}

// T(f) = G(i + f) e^(i f a + delta f) / phi(i) of a wing pixel (poly_tables.cuh), a = 1 / sigma^2 and
// delta the rounding of the kernel's slope, less the leading term s0 = S(i):
//
//   T = e^(-f^2 a / 2 + delta f) S(i + f),   S(x) = int cosh(x a t) e^(-a t^2 / 2) dt over the pixel.
//
// S's Taylor coefficients are Gauss-Legendre sums of positive terms, so FP32 serves them.
__device__ __forceinline__ void wing_taylor(int i, float a, float s0, float delta, float (&D)[kWingTaylor + 1]) {
#pragma unroll
  for (int n = 1; n <= kWingTaylor; ++n) D[n] = 0.f;
  D[0] = s0;
#pragma unroll 1
  for (int q = kGl12 / 2; q < kGl12; ++q) {
    const float t = (float)kGl12T[q], b = a * t, e = expf((float)i * b);
    float p = (float)kGl12W[q] * expf(-0.5f * b * t);  // two nodes' weight, half a cosh each
    const float ch = e + 1.f / e, sh = e - 1.f / e;
#pragma unroll
    for (int n = 1; n <= kWingTaylor; ++n) {
      p *= b * (1.f / (float)n);
      D[n] = fmaf(p, (n & 1) ? sh : ch, D[n]);
    }
  }
  const float h = -0.5f * a;
#pragma unroll
  for (int n = kWingTaylor; n >= 2; --n) {  // times e^(h f^2)
    float c = 1.f;
#pragma unroll
    for (int k = 1; 2 * k <= n; ++k) {
      c *= h * (1.f / (float)k);
      D[n] = fmaf(c, D[n - 2 * k], D[n]);
    }
  }
#pragma unroll
  for (int n = kWingTaylor; n >= 1; --n) D[n] = fmaf(delta, D[n - 1], D[n]);
}

__global__ void __launch_bounds__(128) k_poly_tables(const DevSlice* __restrict__ slices) {
  const DevSlice& S = slices[blockIdx.y];
  const int K = S.K, H = K / 2;
  const int f4 = poly_role_f4(K);
  const double inv_nl = 1.0 / (double)S.n_lambda;
  const int n = 2 * S.n_lambda;
  for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < n; t += gridDim.x * blockDim.x) {
    const int j = t >> 1, axis = t & 1;
    const double lt = (double)(2 * j + 1 - S.n_lambda) * inv_nl;
    const double* c = axis ? S.sy : S.sx;
    const double a = 1.0 / fma(fma(c[2], lt, c[1]), lt, c[0]);
    // ge = phi_sigma(m / 2): e^(-m^2 a^2 / 8) by ratios w = e^(-(2m + 1) a^2 / 8)
    double g = a * 0.39894228040143267794;
    double w = exp(-0.125 * a * a);
    const double r = w * w;
    const float a2 = (float)(a * a);
    const float4 ge = S.samples[(int64_t)j * (S.degree + 3) + S.degree + 1];
    const float gk = axis ? ge.z : ge.x;  // the kernel's slope constant
    float lo[kTaylorMax], hi[kTaylorMax];  // edges i - 1/2 and i + 1/2
    for (int i = 0; i <= H; ++i) {
      const double gc = g;  // the pixel's centre, m = 2i
      g *= w;
      w *= r;
      if (i < kPolyWing) hermite_edge((float)g, (float)((i + 0.5) * a * a), a2, hi);
      g *= w;
      w *= r;
      if (i == 0) {  // the centre pixel's left edge is the mirror image of its right one
#pragma unroll
        for (int k = 0; k < kTaylorMax; ++k) lo[k] = (k & 1) ? -hi[k] : hi[k];
      }
      // c_0 = G(i) = phi(i) (1 + sum_k h_2k / (phi (2k + 1) 4^k)): the sum is small for the
      // bright pixels, so FP32 serves it
      float s = 0.f;
      {
        const float xa2 = (float)((double)i * a * a);
        float q = 1.f, qp = 0.f, sc = 0.25f;
#pragma unroll
        for (int k = 0; k < 20; ++k) {
          const float qn = fmaf(xa2, q, -a2 * qp) * (1.f / (float)(k + 1));
          qp = q;
          q = qn;
          if (k & 1) {
            s = fmaf(q, sc * (1.f / (float)(k + 2)), s);
            sc *= 0.25f;
          }
        }
      }
      const double c0 = gc * (1.0 + (double)s);
      const int m = H - i, half = m & 1, slot = m >> 1, terms = poly_terms(K, slot);
      float E[kPolyTerms], O[kPolyTerms];
#pragma unroll
      for (int q = 0; q < kPolyTerms; ++q) E[q] = O[q] = 0.f;
      if (i < kPolyWing) {
        // Taylor coefficients of G(i + f) and their truncation to degree kPolyDegree
#pragma unroll
        for (int d = kTaylorMax; d >= 1; --d) {
          const float v = (hi[d - 1] - lo[d - 1]) * ((d & 1) ? 1.f / (float)d : -1.f / (float)d);
          if (d > kPolyDegree) {
#pragma unroll
            for (int q = 0; q < kPolyTerms; ++q) {
              if (d & 1) O[q] = fmaf(v, kChebCut[d - 10][q], O[q]);
              else E[q] = fmaf(v, kChebCut[d - 10][q], E[q]);
            }
          } else if (d & 1) {
            O[d / 2] += v;
          } else {
            E[d / 2] += v;
          }
        }
      } else {
        float D[kWingTaylor + 1];
        const double slope = 0.69314718055994530942 * (double)poly_wing_rate(gk, i) - (double)i * a * a;
        wing_taylor(i, a2, 1.f + s, (float)slope, D);
        const float gf = (float)gc;
#pragma unroll
        for (int d = kWingTaylor; d >= 1; --d) {
          const float v = gf * D[d];
          if (d > kPolyDegree) {
#pragma unroll
            for (int q = 0; q < kPolyTerms; ++q) {
              if (d & 1) O[q] = fmaf(v, kChebCut[d - 10][q], O[q]);
              else E[q] = fmaf(v, kChebCut[d - 10][q], E[q]);
            }
          } else if (d & 1) {
            O[d / 2] += v;
          } else {
            E[d / 2] += v;
          }
        }
        if (terms < kPolyTerms) {  // f^8 and f^9 in their turn, cut to degree 7
          static_assert(kPolyTerms == 5, "the cuts below");
          constexpr float ce[4] = {-3.0517578125e-05f, 0.00390625f, -0.078125f, 0.5f};
          constexpr float co[4] = {-0.0001373291015625f, 0.00732421875f, -0.10546875f, 0.5625f};
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            E[q] = fmaf(E[4], ce[q], E[q]);
            O[q] = fmaf(O[4], co[q], O[q]);
          }
        }
      }
      E[0] = (float)(c0 + (double)E[0]);
      float2* out = reinterpret_cast<float2*>(const_cast<float4*>(S.poly) + ((int64_t)j * 4 + 2 * half + axis) * f4) +
                    poly_at(K, slot);
#pragma unroll
      for (int q = 0; q < kPolyTerms; ++q)
        if (q < terms) out[q] = make_float2(E[q], i == 0 ? 0.f : O[q]);
#pragma unroll
      for (int k = 0; k < kTaylorMax; ++k) lo[k] = hi[k];
    }
  }
}

cudaError_t launch_poly_tables(const DevSlice* slices, int n_slices, int max_lambda, cudaStream_t st) {
  if (n_slices == 0 || max_lambda == 0) return cudaSuccess;
  const int bx = (2 * max_lambda + 127) / 128 < 256 ? (2 * max_lambda + 127) / 128 : 256;
  k_poly_tables<<<dim3(bx, n_slices), 128, 0, st>>>(slices);
  return cudaGetLastError();
}

}  // namespace e2e
