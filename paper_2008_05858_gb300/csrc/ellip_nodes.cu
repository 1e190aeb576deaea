// Builds the elliptical PSF's node tables (ellip_moments.cuh), once per model and after an update.
//
// One CTA per node of a slice, one thread per pixel pair, in FP64.  The Taylor coefficients of the
// pixel integral G(X - fx, Y - fy) at fx = fy = 0 are derivatives of G at the pixel, and those are
//   a, b >= 1:  corner differences of the bivariate normal's derivatives (Hermite recurrence),
//   b = 0:      differences over the pixel's left and right edge of A(x) = int f(x, y) dy over its
//               rows and A's derivatives (A' = -x A / vx + P12/P22 [f] over the rows' ends),
//   a = 0:      the same along y;  a = b = 0: 12-point Gauss-Legendre over A.
// They are then expanded in T_p(2 fx) T_q(2 fy) and cut after p + q = kEllDegree.  FP64 arithmetic
// bounds it (1/64 of the FP32 rate): some 7000 operations a pixel pair, half of them the corners'
// recurrences.  24 slices of 8000 samples, K = 13, a node per 64 samples: 6.5 ms, 0.27 ms a slice,
// of a load of 11 ms (11.2 and 16 ms with the recurrences' divisions as divisions).  An update of the
// coefficients pays it again.
#include "e2e_kernels.h"
#include "ellip_moments.cuh"
#include "mixed_common.cuh"
#include "quad_coeffs.h"

namespace e2e {

constexpr int kEllTaylor = 14;

// (u/2)^a = sum_p kChebOf[a][p] T_p(u)
__device__ constexpr double kChebOf[kEllTaylor + 1][kEllDegree + 1] = {
    {1.0, 0, 0, 0, 0, 0, 0, 0, 0, 0, 0},
    {0, 0.5, 0, 0, 0, 0, 0, 0, 0, 0, 0},
    {0.125, 0, 0.125, 0, 0, 0, 0, 0, 0, 0, 0},
    {0, 0.09375, 0, 0.03125, 0, 0, 0, 0, 0, 0, 0},
    {0.0234375, 0, 0.03125, 0, 0.0078125, 0, 0, 0, 0, 0, 0},
    {0, 0.01953125, 0, 0.009765625, 0, 0.001953125, 0, 0, 0, 0, 0},
    {0.0048828125, 0, 0.00732421875, 0, 0.0029296875, 0, 0.00048828125, 0, 0, 0, 0},
    {0, 0.0042724609375, 0, 0.0025634765625, 0, 0.0008544921875, 0, 0.0001220703125, 0, 0, 0},
    {0.001068115234375, 0, 0.001708984375, 0, 0.0008544921875, 0, 0.000244140625, 0, 3.0517578125e-05, 0, 0},
    {0, 0.0009613037109375, 0, 0.000640869140625, 0, 0.000274658203125, 0, 6.866455078125e-05, 0, 7.62939453125e-06, 0},
    {0.000240325927734375, 0, 0.000400543212890625, 0, 0.0002288818359375, 0, 8.58306884765625e-05, 0, 1.9073486328125e-05, 0, 1.9073486328125e-06},
    {0, 0.00022029876708984375, 0, 0.00015735626220703125, 0, 7.867813110351562e-05, 0, 2.6226043701171875e-05, 0, 5.245208740234375e-06, 0},
    {5.507469177246094e-05, 0, 9.441375732421875e-05, 0, 5.900859832763672e-05, 0, 2.6226043701171875e-05, 0, 7.867813110351562e-06, 0, 1.430511474609375e-06},
    {0, 5.1140785217285156e-05, 0, 3.835558891296387e-05, 0, 2.130866050720215e-05, 0, 8.52346420288086e-06, 0, 2.3245811462402344e-06, 0},
    {1.2785196304321289e-05, 0, 2.2374093532562256e-05, 0, 1.4916062355041504e-05, 0, 7.458031177520752e-06, 0, 2.7120113372802734e-06, 0, 6.780028343200684e-07}};

// 1 / n: an FP64 division is some ten FP64 instructions, and the recurrences divide by their index.
__device__ constexpr double kRecip[kEllTaylor + 2] = {0.0, 1.0, 1.0 / 2, 1.0 / 3, 1.0 / 4, 1.0 / 5, 1.0 / 6, 1.0 / 7, 1.0 / 8,
                                                      1.0 / 9, 1.0 / 10, 1.0 / 11, 1.0 / 12, 1.0 / 13, 1.0 / 14, 1.0 / 15};

// P(a < Z < b) of a standard normal, tails subtracted on one side of the mean.
__device__ __forceinline__ double between(double a, double b) {
  const double r2 = 0.70710678118654752440;
  const double ea = erfc(fabs(a) * r2), eb = erfc(fabs(b) * r2);
  if (a >= 0.0) return 0.5 * (ea - eb);
  if (b <= 0.0) return 0.5 * (eb - ea);
  return 1.0 - 0.5 * (ea + eb);
}

__global__ void __launch_bounds__(128) k_ellip_nodes(const DevSlice* __restrict__ slices) {
  constexpr int N = kEllTaylor;
  const DevSlice& S = slices[blockIdx.y];
  if (!S.enodes) return;  // a slice that renders stamp by stamp
  const int n_int = (S.n_lambda + S.espan - 1) / S.espan;
  const int K = S.K, H = K / 2, NP = ell_pairs(K), NS = ell_slots(K) * 32;
  if ((int)blockIdx.x >= n_int + 3) return;
  const int e = threadIdx.x;
  float* out = const_cast<float*>(S.enodes) + (int64_t)blockIdx.x * kEllTerms * NS + e;
  if (e >= NP) {
    if (e < NS)
      for (int t = 0; t < kEllTerms; ++t) out[t * NS] = 0.f;
    return;
  }
  // node v = blockIdx.x - 1 lies at the boundary before sample v espan
  const double lt = (2.0 * (double)((int)blockIdx.x - 1) * S.espan - S.n_lambda) / (double)S.n_lambda;
  const double sa = fma(fma(S.sx[2], lt, S.sx[1]), lt, S.sx[0]);
  const double sb = fma(fma(S.sy[2], lt, S.sy[1]), lt, S.sy[0]);
  const double cs = S.cos_t, sn = S.sin_t, a2 = sa * sa, b2 = sb * sb;
  const double vx = a2 * cs * cs + b2 * sn * sn, vy = a2 * sn * sn + b2 * cs * cs, cxy = (a2 - b2) * sn * cs;
  const double det = a2 * b2;
  const double P11 = vy / det, P12 = -cxy / det, P22 = vx / det;
  const double bx = cxy / vx, by = cxy / vy, isx = 1.0 / sqrt(vy - bx * cxy), isy = 1.0 / sqrt(vx - by * cxy);
  const double X = (double)(e % K - H), Y = (double)(e / K - H);
  const double rs2pi = 0.39894228040143267794;
  double c[N + 1][N + 1];
#pragma unroll 1
  for (int a = 0; a <= N; ++a)
#pragma unroll 1
    for (int b = 0; b <= N - a; ++b) c[a][b] = 0.0;
  const double inv_det = rs2pi * rs2pi / sqrt(det), ivx = 1.0 / vx, ivy = 1.0 / vy, qx = P12 / P22, qy = P12 / P11;
  // A's and B's derivative sources: differences over the pixel's rows (columns) of h_(a,0) (h_(0,b))
  double fa[2][N + 1], fb[2][N + 1];
#pragma unroll 1
  for (int a = 0; a <= N; ++a) fa[0][a] = fa[1][a] = fb[0][a] = fb[1][a] = 0.0;
#pragma unroll 1
  for (int q = 0; q < 4; ++q) {
    const int ix = q & 1, iy = q >> 1;
    const double x = X + ix - 0.5, y = Y + iy - 0.5, sg = ix == iy ? 1.0 : -1.0;
    const double L1 = P11 * x + P12 * y, L2 = P12 * x + P22 * y;
    double h[N + 1], hp[N + 1];  // rows a and a - 1 of f^(a,b) / (a! b!)
    h[0] = inv_det * exp(-0.5 * (x * L1 + y * L2));
    h[1] = -L2 * h[0];
#pragma unroll 1
    for (int b = 1; b < N; ++b) h[b + 1] = -(L2 * h[b] + P22 * h[b - 1]) * kRecip[b + 1];
#pragma unroll 1
    for (int b = 0; b <= N; ++b) {
      hp[b] = 0.0;
      fb[iy][b] += ix ? h[b] : -h[b];
    }
#pragma unroll 1
    for (int a = 0; a < N; ++a) {
      fa[ix][a] += iy ? h[0] : -h[0];
      const double ra = kRecip[a + 1];
      double left = 0.0;  // row a, column b - 1
#pragma unroll 1
      for (int b = 0; b <= N - a - 1; ++b) {
        const double v = h[b];
        if (b + 1 <= N - a - 1) c[a + 1][b + 1] += sg * v * ra * kRecip[b + 1];
        const double nx = -(L1 * v + P11 * hp[b] + P12 * left) * ra;
        hp[b] = v;
        left = v;
        h[b] = nx;
      }
    }
  }
#pragma unroll 1
  for (int s = 0; s < 2; ++s) {
    const double sg = s ? 1.0 : -1.0;
    const double x = X + s - 0.5, y = Y + s - 0.5;
    double al = rs2pi / sqrt(vx) * exp(-0.5 * x * x / vx) * between((Y - 0.5 - bx * x) * isx, (Y + 0.5 - bx * x) * isx);
    double be = rs2pi / sqrt(vy) * exp(-0.5 * y * y / vy) * between((X - 0.5 - by * y) * isy, (X + 0.5 - by * y) * isy);
    double alp = 0.0, bep = 0.0;
#pragma unroll 1
    for (int a = 1; a <= N; ++a) {
      const double ia = kRecip[a];
      c[a][0] += sg * al * ia;
      c[0][a] += sg * be * ia;
      const double an = (-(x * al + alp) * ivx + qx * fa[s][a - 1]) * ia;
      const double bn = (-(y * be + bep) * ivy + qy * fb[s][a - 1]) * ia;
      alp = al;
      al = an;
      bep = be;
      be = bn;
    }
  }
  double g = 0.0;
#pragma unroll 1
  for (int q = 0; q < kGl12; ++q) {
    const double u = X + kGl12T[q];
    g += kGl12W[q] * exp(-0.5 * u * u * ivx) * between((Y - 0.5 - bx * u) * isx, (Y + 0.5 - bx * u) * isx);
  }
  c[0][0] = g * rs2pi / sqrt(vx);
  // d/dfx = -d/dX: odd a + b change sign; rows then columns into T_p(2 fx) T_q(2 fy)
#pragma unroll 1
  for (int a = 0; a <= N; ++a) {
#pragma unroll 1
    for (int q = 0; q <= min(kEllDegree, N - a); ++q) {
      double v = 0.0;
#pragma unroll 1
      for (int b = q; b <= N - a; b += 2) v += kChebOf[b][q] * ((a + b) & 1 ? -c[a][b] : c[a][b]);
      c[a][q] = v;  // entries below q are final, those above are still Taylor coefficients
    }
  }
#pragma unroll 1
  for (int q = 0; q <= kEllDegree; ++q)
#pragma unroll 1
    for (int p = 0; p + q <= kEllDegree; ++p) {
      double v = 0.0;
#pragma unroll 1
      for (int a = p; a + q <= N; a += 2) v += kChebOf[a][p] * c[a][q];
      out[ell_term(p, q) * NS] = e == NP - 1 && ((p + q) & 1) ? 0.f : (float)v;
    }
}

cudaError_t launch_ellip_nodes(const DevSlice* slices, int n_slices, int max_nodes, cudaStream_t st) {
  if (n_slices == 0) return cudaSuccess;
  k_ellip_nodes<<<dim3(max_nodes, n_slices), 128, 0, st>>>(slices);
  return cudaGetLastError();
}

int64_t ellip_node_floats(int K) { return (int64_t)kEllTerms * ell_slots(K) * 32; }

}  // namespace e2e
