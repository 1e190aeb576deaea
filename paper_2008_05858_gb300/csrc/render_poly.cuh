// The separable-PSF mixed-precision render kernel on polynomial pixel integrals
// (poly_tables.cuh), as a template instantiated by render_poly.cu (production) and
// render_poly_check.cu (debug checks).
//
// Items, boxes and runs are those of k_render_mixed (render_mixed.cuh), which evaluates the
// 2(K + 1) edge tails of every stamp; that was 25 of its 35 warp-instructions per stamp.  Here a
// stamp's 2K pixel integrals are polynomials of degree 9 in its sub-pixel offset whose coefficients
// depend on the wavelength sample only.  A warp takes eight samples, a quad of lanes each, and
// walks all the item's slit points with them, so that a lane loads its coefficients once per
// sample and holds them in registers: lane (axis, half) of the quad evaluates half the pixel pairs
// of one axis of every stamp, at K = 11 some two dozen packed and scalar operations and, for the
// slopes of its two wing pairs, four exponentials (1.5 % of the 9216^2 frame, 3.71 -> 3.77 ms with
// its merge; without them narrow PSFs' wings miss the bound, poly_tables.cuh).  The quad's
// profiles go through shared memory, and each lane adds one quadrant of the tile's outer product.
// The tiles are merged by a kernel of their own: the last CTA of a tile merging it while three
// others hold the SM cost more (0.5 ms of a 9216^2 frame) than the separate launch (0.3 ms).
//
// Measured on the benchmark's 9216^2 frame of 340 slices x 6000 x 64 stamps: 3.76 ms (the edge tails
// with their merge 5.2 ms), 4096^2 frame of 40 x 4000 x 32 with its merge 0.24 ms (0.33).  Per stamp
// 21 warp-instructions; the shared-memory pipe is busy 74 % of the time, the FMA pipe 45 %, issue
// slots 63 %; four CTAs of 128 threads per SM (128 registers) leave the rest to latency.  Five CTAs
// spill.  Windows of 9, 13 and 15 px spill at four already (the wide ones hold four pixel pairs'
// coefficients and a tile quadrant of 7 x 7 pixels) and run three to an SM, with up to 168 registers.
// It is the faster one at every size: 4096^2 frame of 40 traces x 4000 samples, K = 15, 8 / 32 / 64
// slit points 380 / 1250 / 2440 us against 499 / 1631 / 3175 for the edge tails, K = 11, 1 / 4 / 7
// points 143 / 170 / 201 against 155 / 180 / 252.
#pragma once
#include <type_traits>

#include "e2e_device.cuh"
#include "e2e_kernels.h"
#include "fast_map.cuh"
#include "mixed_common.cuh"
#include "phi32.cuh"
#include "poly_tables.cuh"

namespace e2e {

constexpr int kPThreads = 128;
constexpr int kPWarps = kPThreads / 32;
constexpr int kNoStamp = 1 << 30;       // window centre of a stamp that deposits nothing
// fixed_split2_small's bound on the high word, over the largest pixel integral of a PSF of widths
// kPolyMinSigma = 1 (erf(1 / sqrt 8)^2 = 0.1466)
constexpr float kSmallDeposit = 4190000.f / 0.147f;
constexpr int kPQuad = 36;             // floats per quad and stamp of the exchange (4 mod 32: see below)
constexpr int kPBuf = 8 * kPQuad;      // floats per stamp slot of a warp

// A quad's profiles in the exchange: x at 0, y at poly_y_offset, each K values between D zeros on
// either side, so that a lane reads the tile's pixels, zeros outside the window included, from
// D - (the window's offset in the tile) on, and the zeros are written once per CTA.  The y values
// start 2 mod 4 after the x values: the quad's four lanes write four neighbouring pixels' banks,
// the eight quads 4 banks apart, so the stores have no bank conflicts.
__host__ __device__ constexpr int poly_y_offset(int K, int DX, int DY) {
  int a = K + 2 * DX;
  while (((a + DY - DX) & 3) != 2) ++a;
  return a;
}

// Shared-memory layout of one CTA (offsets in bytes), identical on host and device.
struct PolyLayout {
  size_t tabP, tabS, tabW, tabU, stage, org, xch, boxh, boxl, total;
  __host__ __device__ PolyLayout(int J, int NK, int nd, int area) {
    size_t o = 0;
    tabP = o; o += (size_t)J * (nd + 2) * 16;      // the samples' table rows: P_b(lt) of x and y, split_xy pairs, ...
    stage = o; o += (size_t)kPWarps * 16 * 8 * 16;  // mapped stamps: 16 slit points of 8 quads per warp
    xch = o; o += (size_t)kPWarps * 4 * kPBuf * 4;  // profile exchange: two buffers of two stamps
    org = o; o += (size_t)kPWarps * 16 * 8 * 8;     // tile origin of each stamp's run
    tabS = o; o += (size_t)NK * 8;                  // s of each slit point, (hi, lo) floats
    tabU = o; o += (size_t)NK * 8;                  // slit weights, (hi, lo) floats
    tabW = o; o += (size_t)J * 8;                   // flux x bin width per sample, (hi, lo) floats
    boxh = o; o += (size_t)area * 4;                // fixed-point box, high words
    boxl = o; o += (size_t)area * 4;                // low words
    total = o;
  }
};

// The two lane quadrants along an axis of R tile pixels: the first takes [0, quad_span), the
// second the rest.
__host__ __device__ constexpr int quad_span(int R) { return (R + 1) / 2; }

// CHECK: debug build of the same kernel, counting into a.err every deposit the plan did not
// foresee.
// CTAs per SM that a window's registers allow (above).
__host__ __device__ constexpr int poly_ctas(int K) { return K >= 13 || K == 9 ? 3 : 4; }

template <int K, int DX, int DY, bool CHECK>
__global__ void __launch_bounds__(kPThreads, poly_ctas(K)) k_render_poly(const MixedArgs a) {
  constexpr int RX = K + DX, RY = K + DY, H = K / 2;
  constexpr int NS = poly_slots(K), F4 = poly_role_f4(K);
  constexpr int NX = quad_span(RX), NY = quad_span(RY);  // lane quadrant: columns and rows
  constexpr int YO = poly_y_offset(K, DX, DY);
  static_assert(YO + K + 2 * DY <= kPQuad && YO + 2 * NY + DY <= kPQuad, "profiles exceed the exchange row");
  extern __shared__ __align__(16) unsigned char smem[];
  const Item it = a.items[blockIdx.x];
  const DevSlice& S = a.slices[it.slice];
  const int area = it.bw * it.bh;
  const int nd = S.degree + 1;
  const PolyLayout L(32 * a.JB, a.nk_max, a.max_deg + 1, area);
  float4* tabP = reinterpret_cast<float4*>(smem + L.tabP);
  float2* tabS = reinterpret_cast<float2*>(smem + L.tabS);
  float2* tabW = reinterpret_cast<float2*>(smem + L.tabW);
  float2* tabU = reinterpret_cast<float2*>(smem + L.tabU);
  int* boxh = reinterpret_cast<int*>(smem + L.boxh);
  int* boxl = reinterpret_cast<int*>(smem + L.boxl);
  __shared__ double s_w[kPWarps], s_u[kPWarps];

  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  // the item's rows of the per-sample table (one block of memory), copied to shared memory
  // asynchronously while the box is cleared and the weights are built
  for (int e = tid; e < it.nj * (nd + 2); e += kPThreads)
    cp_async16(tabP + e, S.samples + (int64_t)it.j0 * (nd + 2) + e);
  const double* flux = a.flux_tab[S.flux_slot];
  const double* u = a.u_all + S.u_off;
  const double u_first = tid < it.nk ? u[it.k0 + tid] : 0.0;
  const double f_first = tid < it.nj ? flux[it.j0 + tid] : 0.0;
  // the first sample octet's coefficients, in flight while the tables are built
  const int quad = lane >> 2, qi = lane & 3, axis = qi & 1, half = qi >> 1;
  // a warp's eight samples lie njq apart: their tiles share few box pixels (neighbouring samples of
  // a finely sampled trace share most of theirs, and lanes that add to one pixel take turns)
  const int njq = (it.nj + 7) / 8;
  float4 cv[F4];
  auto load_coefs = [&](int task) {
    const float4* src = S.poly + ((int64_t)(it.j0 + min(quad * njq + task, it.nj - 1)) * 4 + qi) * F4;
#pragma unroll
    for (int q = 0; q < F4; ++q) cv[q] = __ldg(src + q);
  };
  load_coefs(warp);
  for (int p = tid; p < area; p += kPThreads) {
    boxh[p] = 0;
    boxl[p] = 0;
  }
  for (int p = tid; p < kPWarps * 4 * kPBuf / 4; p += kPThreads)
    reinterpret_cast<float4*>(smem + L.xch)[p] = make_float4(0.f, 0.f, 0.f, 0.f);
  const double inv_ns = 1.0 / (double)S.n_slit;
  double usum = 0.0;
  for (int kk = tid; kk < it.nk; kk += kPThreads) {
    const double uk = kk == tid ? u_first : u[it.k0 + kk];
    tabS[kk] = split_df(norm_sample_r(it.k0 + kk, S.n_slit, inv_ns));
    tabU[kk] = split_df(uk);
    usum += fabs(uk);
  }
  double wsum = 0.0;
  for (int jj = tid; jj < it.nj; jj += kPThreads) {
    const double wj = (jj == tid ? f_first : flux[it.j0 + jj]) * S.dlam;
    tabW[jj] = split_df(wj);
    wsum += fabs(wj);
  }
  // flux bound of the item: sum over its stamps of |w| (bounds every pixel of its box)
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    wsum += __shfl_xor_sync(0xffffffffu, wsum, o);
    usum += __shfl_xor_sync(0xffffffffu, usum, o);
  }
  if (lane == 0) {
    s_w[warp] = wsum;
    s_u[warp] = usum;
  }
  cp_async_wait_all();  // this thread's table copies; the barrier then publishes all of them
  __syncthreads();
  double wtot = 0.0, utot = 0.0;
#pragma unroll
  for (int q = 0; q < kPWarps; ++q) {
    wtot += s_w[q];
    utot += s_u[q];
  }
  const double total = wtot * utot;
  // scale 2^P with |box sums| <= total < 2^(52-P); clamp so 2^P stays a normal FP32
  int ex = 0;
  frexp(total, &ex);
  const int Psh = total > 0.0 ? max(-100, min(100, 52 - ex)) : 0;
  const float sc = ldexpf(1.f, Psh), sc_hi = ldexpf(1.f, Psh - 22);

  // Lane qi of a quad evaluates axis qi & 1 (x, y), pixel pairs of half qi >> 1; it owns the
  // tile quadrant of columns (qi & 1) NX + [0, NX) and rows (qi >> 1) NY + [0, NY).
  float4* stage = reinterpret_cast<float4*>(smem + L.stage) + warp * 128 + quad;      // [16][8 quads]
  int2* org = reinterpret_cast<int2*>(smem + L.org) + warp * 128 + quad;              // [16][8 quads]
  float* xq = reinterpret_cast<float*>(smem + L.xch) + warp * 4 * kPBuf + quad * kPQuad;
  float* wrow = xq + (axis ? YO + DY : DX) + half;      // where this lane's profile values go
  const float* rx = xq + (qi & 1) * NX;                // the columns and rows it reads back, less
  const float* ry = xq + YO + (qi >> 1) * NY;          // the window's place in the tile
  const int ncol = (qi & 1) ? RX - NX : NX, nrow = (qi >> 1) ? RY - NY : NY;
  const int B = a.B;
  for (int task = warp; task < njq && total > 0.0; task += kPWarps) {
    const int jj = quad * njq + task;
    const bool jvalid = jj < it.nj;  // uniform over the quad
    const int jc = jvalid ? jj : it.nj - 1;
    // this lane's coefficients: NS pixel pairs x kPolyTerms (E, O)
    float2 cf[NS][kPolyTerms];
    if (task != warp) load_coefs(task);
#pragma unroll
    for (int s = 0; s < NS; ++s)
#pragma unroll
      for (int q = 0; q < poly_terms(K, s); ++q) {
        const int e = poly_at(K, s) + q;
        cf[s][q] = (e & 1) ? make_float2(cv[e / 2].z, cv[e / 2].w) : make_float2(cv[e / 2].x, cv[e / 2].y);
      }
    const float2 wj = jvalid ? tabW[jc] : make_float2(0.f, 0.f);
    const float4* Pj = tabP + jc * (nd + 2);
    const FastMap fm(Pj, S.degree);
    float wing[NS];  // slopes of this lane's wing pixels (the other pixel of such a slot has none)
    {
      const float4 ge = Pj[nd];
#pragma unroll
      for (int s = 0; s < NS; ++s) {
        const int i = H - half - 2 * s;
        wing[s] = i >= kPolyWing ? poly_wing_rate(axis ? ge.z : ge.x, i) : 0.f;
      }
    }
    int parity = 0;
    for (int k0 = 0; k0 < it.nk; k0 += 16) {
      const int nk = min(16, it.nk - k0);
      bool small;  // every deposit of these stamps' tiles stays below 2^44 units (fixed_split2_small)
      // map 16 slit points, a quarter per lane; the tile origin of each run of B of them is the
      // least window centre of its on-frame stamps
      {
        int ci[4], ri[4], ox[4], oy[4];
        float fx[4], fy[4], wmax = 0.f;
        float2 sv[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) sv[q] = tabS[k0 + min(qi + 4 * q, nk - 1)];
        fm.map(Pj, S.degree, sv, ci, fx, ri, fy);
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          if (!jvalid || qi + 4 * q >= nk || ci[q] == kOffFrame || ri[q] == kOffFrame) ci[q] = ri[q] = kNoStamp;
          ox[q] = ci[q];
          oy[q] = ri[q];
        }
        if (B >= 2) {
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            ox[q] = min(ox[q], __shfl_xor_sync(0xffffffffu, ox[q], 1));
            oy[q] = min(oy[q], __shfl_xor_sync(0xffffffffu, oy[q], 1));
          }
        }
        if (B >= 4) {
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            ox[q] = min(ox[q], __shfl_xor_sync(0xffffffffu, ox[q], 2));
            oy[q] = min(oy[q], __shfl_xor_sync(0xffffffffu, oy[q], 2));
          }
        }
        if (B >= 8) {
          ox[0] = ox[1] = min(ox[0], ox[1]);
          oy[0] = oy[1] = min(oy[0], oy[1]);
          ox[2] = ox[3] = min(ox[2], ox[3]);
          oy[2] = oy[3] = min(oy[2], oy[3]);
        }
        if (B >= 16) {
          ox[0] = ox[1] = ox[2] = ox[3] = min(ox[0], ox[2]);
          oy[0] = oy[1] = oy[2] = oy[3] = min(oy[0], oy[2]);
        }
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          const int b = qi + 4 * q;
          const bool on = ci[q] != kNoStamp;
          const float2 uk = tabU[k0 + min(b, nk - 1)];
          const float w = on ? fmaf(wj.x, uk.x, fmaf(wj.x, uk.y, wj.y * uk.x)) : 0.f;
          wmax = fmaxf(wmax, fabsf(w));
          int dx = on ? ci[q] - ox[q] : 0, dy = on ? ri[q] - oy[q] : 0;
          if constexpr (CHECK) {
            if (dx > DX || dy > DY) atomicAdd(a.err, 1);  // the run outgrew the planned tile
          }
          dx = min(dx, DX);
          dy = min(dy, DY);
          stage[b * 8] = make_float4(on ? fx[q] : 0.f, on ? fy[q] : 0.f, w, __int_as_float((DX - dx) | ((DY - dy) << 16)));
          org[b * 8] = make_int2(ox[q], oy[q]);
        }
        // a run's tile pixels are at most the sum of its weights times the largest pixel integral
        small = __all_sync(0xffffffffu, wmax * (float)B * sc_hi < kSmallDeposit);
      }
      __syncwarp();
      for (int b0 = 0; b0 < nk; b0 += B) {
        const int2 o2 = org[b0 * 8];
        const int nb = min(B, nk - b0);
        float acc[NY][NX];
#pragma unroll
        for (int r = 0; r < NY; ++r)
#pragma unroll
          for (int c = 0; c < NX; ++c) acc[r][c] = 0.f;
        float4 st[2] = {stage[b0 * 8], stage[min(b0 + 1, 15) * 8]};
        for (int b = b0; b < b0 + nb; b += 2) {  // two stamps per step
          const int off[2] = {__float_as_int(st[0].w), __float_as_int(st[1].w)};
          {
            float2 p[2][NS];
            float mult[2], fw[2], z[2];
#pragma unroll
            for (int e = 0; e < 2; ++e) {
              const float f = axis ? st[e].y : st[e].x;
              // the weight rides on the x profile; with runs of one stamp the second is another run's
              mult[e] = axis ? 1.f : (e == 1 && B == 1 ? 0.f : st[e].z);
              z[e] = f * f;
              fw[e] = f * mult[e];
#pragma unroll
              for (int s = 0; s < NS; ++s) p[e][s] = cf[s][poly_terms(K, s) - 1];
            }
#pragma unroll
            for (int q = kPolyTerms - 2; q >= 0; --q)
#pragma unroll
              for (int e = 0; e < 2; ++e)
#pragma unroll
                for (int s = 0; s < NS; ++s)
                  if (q < poly_terms(K, s) - 1) p[e][s] = __ffma2_rn(p[e][s], make_float2(z[e], z[e]), cf[s][q]);
#pragma unroll
            for (int e = 0; e < 2; ++e) {
              float* row = wrow + (parity + e) * kPBuf;
#pragma unroll
              for (int s = 0; s < NS; ++s) {
                const float Ew = p[e][s].x * mult[e];
                float v0 = fmaf(fw[e], p[e][s].y, Ew), v1 = fmaf(-fw[e], p[e][s].y, Ew);  // G(i + f), G(i - f)
                if (poly_wing(K, s)) {
                  const float t = (axis ? st[e].y : st[e].x) * wing[s];
                  v0 *= ex2_approx(-t);
                  v1 *= ex2_approx(t);
                }
                if (2 * s + 1 <= H || half == 0) {  // half 1 has one pair fewer when H is even
                  row[2 * s] = v0;
                  row[K - 1 - 2 * half - 2 * s] = v1;
                }
              }
            }
          }
          __syncwarp();
          st[0] = stage[min(b + 2, 15) * 8];
          st[1] = stage[min(b + 3, 15) * 8];
#pragma unroll
          for (int e = 0; e < 2; ++e) {
            const float* px = rx + (parity + e) * kPBuf + (off[e] & 0xffff);
            const float* py = ry + (parity + e) * kPBuf + (off[e] >> 16);
            float xv[NX], yv[NY];
#pragma unroll
            for (int c = 0; c < NX; ++c) xv[c] = px[c];
#pragma unroll
            for (int r = 0; r < NY; ++r) yv[r] = py[r];
#pragma unroll
            for (int r = 0; r < NY; ++r) {
              const float2 yy = make_float2(yv[r], yv[r]);
#pragma unroll
              for (int c = 0; c + 1 < NX; c += 2) {
                const float2 v = __ffma2_rn(yy, make_float2(xv[c], xv[c + 1]), make_float2(acc[r][c], acc[r][c + 1]));
                acc[r][c] = v.x;
                acc[r][c + 1] = v.y;
              }
              if constexpr (NX % 2 == 1) acc[r][NX - 1] = fmaf(yv[r], xv[NX - 1], acc[r][NX - 1]);
            }
          }
          parity ^= 2;  // the other buffer: its readers have passed this step's barrier
        }
        // flush this lane's quadrant of the run tile as exact fixed-point increments
        if (o2.x != kNoStamp) {
          const int gx0 = o2.x - H - it.bx0 + (qi & 1) * NX, gy0 = o2.y - H - it.by0 + (qi >> 1) * NY;
          const bool inside = gx0 >= 0 && gx0 + ncol <= it.bw && gy0 >= 0 && gy0 + nrow <= it.bh;
          constexpr int kMinX = RX - NX, kMinY = RY - NY;
          if (inside) {
            int* row0 = boxh + gy0 * it.bw + gx0;
            const int lo = (int)(boxl - boxh);
            auto deposit = [&](auto fast) {
              int* rowh = row0;
#pragma unroll
              for (int r = 0; r < NY; ++r) {
                if (r < kMinY || r < nrow) {
#pragma unroll
                  for (int c = 0; c < NX; c += 2) {
                    const float2 v = make_float2(acc[r][c], c + 1 < NX ? acc[r][c + 1] : 0.f);
                    int2 hw, lw;
                    if (decltype(fast)::value) fixed_split2_small(v, sc, sc_hi, hw, lw);
                    else fixed_split2_s(v, sc, sc_hi, hw, lw);
#pragma unroll
                    for (int h = 0; h < 2 && c + h < NX; ++h) {
                      if (c + h < kMinX || c + h < ncol) {
                        atomicAdd(rowh + c + h, h ? hw.y : hw.x);
                        atomicAdd(rowh + lo + c + h, h ? lw.y : lw.x);
                      }
                    }
                  }
                }
                rowh += it.bw;
              }
            };
            if (small) deposit(std::true_type{});
            else deposit(std::false_type{});  // a sample far above the rest of the item
          } else {  // a tile over the box's edge: the frame ends there
#pragma unroll
            for (int r = 0; r < NY; ++r)
#pragma unroll
              for (int c = 0; c < NX; ++c) {
                const int gx = gx0 + c, gy = gy0 + r;
                if (r >= nrow || c >= ncol) continue;
                if (gy < 0 || gy >= it.bh || gx < 0 || gx >= it.bw) {
                  if constexpr (CHECK) {  // outside the box is legitimate only off the detector
                    const int X = it.bx0 + gx, Y = it.by0 + gy;
                    if (acc[r][c] != 0.f && X >= 0 && X < S.W && Y >= 0 && Y < S.H) atomicAdd(a.err, 1);
                  }
                  continue;
                }
                box_deposit_s(boxh + gy * it.bw + gx, boxl + gy * it.bw + gx, acc[r][c], sc, sc_hi);
              }
          }
        }
      }
      __syncwarp();  // the staging is reused by the next 16 slit points
    }
  }
  __syncthreads();
  // box value = (hi word * 2^22 + lo word) * 2^-P, written as an unevaluated FP32 pair
  float2* out = a.store + it.store_off;
  const float inv = ldexpf(1.f, -Psh);
  for (int p = tid; p < area; p += kPThreads) out[p] = fixed_to_pair_s(boxh[p], boxl[p], inv);
}

template <int K, int DX, int DY, bool CHECK>
static cudaError_t launch_poly_one(const MixedArgs& a, int n_items, size_t smem, cudaStream_t st) {
  auto kern = k_render_poly<K, DX, DY, CHECK>;
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  kern<<<n_items, kPThreads, smem, st>>>(a);
  return cudaGetLastError();
}

cudaError_t launch_render_poly_checked(int K, int DX, int DY, const MixedArgs& a, int n_items, size_t smem,
                                       cudaStream_t st);

// The tile variants (K, DX, DY) of the polynomial kernel: those of k_render_mixed with K >= 3.
#define E2E_POLY_VARIANTS(V)                                                                            \
  V(3, 0, 0) V(5, 0, 0) V(7, 0, 0) V(9, 0, 0) V(11, 0, 0) V(13, 0, 0) V(15, 0, 0)                       \
  V(3, 1, 1) V(5, 1, 1) V(7, 1, 1) V(9, 1, 1) V(11, 1, 1) V(13, 1, 1)                                   \
  V(3, 1, 2) V(5, 1, 2) V(7, 1, 2) V(9, 1, 2) V(11, 1, 2) V(13, 1, 2)                                   \
  V(3, 1, 3) V(5, 1, 3) V(7, 1, 3) V(9, 1, 3) V(11, 1, 3)                                               \
  V(3, 2, 2) V(5, 2, 2) V(7, 2, 2) V(9, 2, 2)

}  // namespace e2e
