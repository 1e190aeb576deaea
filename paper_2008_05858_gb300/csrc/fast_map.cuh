// Stamp mapping in FP32 about a wavelength sample's own position, deciding exactly as
// map_xy_df / split_coord_df (mixed_common.cuh) do.
//
// A stamp's centre is P_0 + s P_1 + s^2 Q(s).  Only its whole pixel must be exact; the offset
// in the pixel is an FP32 number.  P_0 is cut into its nearest integer and the rest (a pair),
// s P_1 keeps its FMA error term, and s^2 Q (at most 1 px, checked per sample) is plain FP32:
// 10 packed operations and 4 per axis at degree 5 where the double-float Horner takes 65 packed.
// The offset's error stays below 6e-7 px (rms 2e-8), so a stamp whose offset is farther than
// kTieMargin from a pixel edge gets the exact mapping's whole pixel; the few others (one in 1e5),
// and samples outside the bounds, take the exact mapping itself.  Single stamps at the ends of slits bent
// by the 1 px that s^2 Q may reach: worst pixel 0.74 of the renderer's bound at sigma = 1.0 (0.57 by
// the exact mapping), rotated PSF 0.98 at 1.3 px (0.69).
#pragma once
#include "mixed_common.cuh"

namespace e2e {

constexpr float kTieMargin = 4e-6f;

struct FastMap {
  float2 f0h, f0l, p1h, p1l;  // x, y: fraction of P_0 as a pair, P_1
  int ix, iy;                 // nearest integers of P_0
  bool ok;

  __device__ __forceinline__ FastMap(const float4* P, int d) {
    const float4 c0 = P[0];
    const float rx = rintf(c0.x), ry = rintf(c0.y);
    float h, l;
    two_sum(c0.x - rx, c0.z, h, l);
    f0h.x = h;
    f0l.x = l;
    two_sum(c0.y - ry, c0.w, h, l);
    f0h.y = h;
    f0l.y = l;
    float4 c1 = make_float4(0.f, 0.f, 0.f, 0.f);
    if (d >= 1) c1 = P[1];
    p1h = make_float2(c1.x, c1.y);
    p1l = make_float2(c1.z, c1.w);
    float ux = 0.f, uy = 0.f;
    for (int b = 2; b <= d; ++b) {
      const float4 c = P[b];
      ux += fabsf(c.x);
      uy += fabsf(c.y);
    }
    ok = fabsf(c0.x) < 32000.f && fabsf(c0.y) < 32000.f && fabsf(c1.x) <= 64.f && fabsf(c1.y) <= 64.f && ux <= 1.f &&
         uy <= 1.f;
    ix = ok ? (int)rx : 0;
    iy = ok ? (int)ry : 0;
  }

  // Window-centre pixels (kOffFrame as split_coord_df) and offsets of N slit points s = (hi, lo).
  template <int N>
  __device__ __forceinline__ void map(const float4* P, int d, const float2 (&s)[N], int (&ci)[N], float (&fx)[N],
                                      int (&ri)[N], float (&fy)[N]) const {
    constexpr float kMagic = 12582912.f;  // 1.5 * 2^23: adding it rounds to an integer
    float2 q[N];
#pragma unroll
    for (int n = 0; n < N; ++n) q[n] = make_float2(0.f, 0.f);
    if (ok) {
      for (int b = d; b >= 2; --b) {
        const float2 c = *reinterpret_cast<const float2*>(P + b);
#pragma unroll
        for (int n = 0; n < N; ++n) q[n] = __ffma2_rn(q[n], make_float2(s[n].x, s[n].x), c);
      }
    }
#pragma unroll
    for (int n = 0; n < N; ++n) {
      const float2 sh = make_float2(s[n].x, s[n].x), sl = make_float2(s[n].y, s[n].y);
      const float2 u = __fmul2_rn(__fmul2_rn(q[n], sh), sh);
      const float2 ph = __fmul2_rn(p1h, sh);
      float2 pe = __ffma2_rn(p1h, sh, neg2(ph));
      pe = __ffma2_rn(p1l, sh, pe);
      pe = __fadd2_rn(__ffma2_rn(p1h, sl, pe), f0l);
      const float2 b2 = __fadd2_rn(f0h, u);
      const float2 t = __fadd2_rn(__fadd2_rn(ph, b2), make_float2(kMagic, kMagic));
      const float2 c = __fadd2_rn(t, make_float2(-kMagic, -kMagic));
      const float2 f = __fadd2_rn(__fadd2_rn(__fadd2_rn(ph, neg2(c)), b2), pe);
      fx[n] = f.x;
      fy[n] = f.y;
      ci[n] = ix + (__float_as_int(t.x) - 0x4B400000);
      ri[n] = iy + (__float_as_int(t.y) - 0x4B400000);
    }
#pragma unroll
    for (int n = 0; n < N; ++n) {
      if (!ok || fmaxf(fabsf(fx[n]), fabsf(fy[n])) > 0.5f - kTieMargin) {
        float2 hi, lo;
        map_xy_df(P, d, s[n], hi, lo);
        split_coord_df(hi.x, lo.x, ci[n], fx[n]);
        split_coord_df(hi.y, lo.y, ri[n], fy[n]);
      }
    }
  }
};

}  // namespace e2e
