// The elliptical-PSF mixed-precision render on the moments of its runs (ellip_moments.cuh).
//
// k_render_ellip (render_ellip.cu) evaluates every stamp's K^2 pixel integrals: 253 warp-
// instructions a stamp at K = 13.  Here a stamp adds its 66 moments to its run's, and a warp turns
// the runs of a wavelength sample into pixels together: 79 warp-instructions a stamp at 128 slit
// points of 8 px (a dozen stamps per run).
//
// One CTA of 12 warps takes the items of one slice between two nodes: their four node tables become
// the cubics' coefficients in shared memory (float4 per term and pixel pair, 101 KB at K = 13).  A
// warp takes one sample and walks its slit points 32 at a time: each lane maps one stamp and forms
// its Chebyshev values; the run boundaries are a ballot; 21 lanes hold the 66 moments as 2 x 2
// blocks of (a, b).  After kEllRuns runs, and at the end of the sample, the warp forms the runs'
// pixels, lane l the pixel pairs l, l + 32, ..., and deposits them into the item's box as exact
// fixed point (the low word 20 bits wide: an item may put 4096 deposits on a pixel).
//
// Measured on 24 slices x 8000 x 128 stamps (K = 13), the whole render: 8.85 ms stamp by stamp, 2.52
// with every sum in plain FP32 (and the far wings of runs on one side of their pixel up to 3.5 times
// the bound off), 3.33 with the errors of the large sums carried (ellip_moments.cuh): 0.2 ms for the
// moments', 0.2 for the pixels', the rest because the sums of twelve runs and their errors take 168
// registers, so 12 warps instead of 16 (at 16 they spill: 3.7 to 4.4 ms; slot by slot without a spill,
// the moments read three times, 3.6).  Issue slots are busy half the time, the shared-memory pipe
// half; one CTA per SM, so its prologue and write-back stand by themselves.
#include "e2e_device.cuh"
#include "e2e_kernels.h"
#include "ellip_moments.cuh"
#include "fast_map.cuh"
#include "mixed_common.cuh"

namespace e2e {

constexpr int kMThreads = 384;
constexpr int kMWarps = kMThreads / 32;
constexpr int kMStage = 16;  // stamps staged at a time
// A staged pair of stamps: 12 float4 {v, v' of the first, v, v' of the second}, (v, v') the values
// u T_2p(2 fx), u T_2p+1(2 fx), p = 0..5 (the last v' is u's leading 12 bits), then T_2p(2 fy),
// T_2p+1(2 fy) (the last v' the rest of u), and 4 floats that spread the pairs over the banks.
constexpr int kMPair = 52;

struct MomentLayout {
  size_t tab, mom, low, stage, tabP, tabS, tabU, tabW, boxh, boxl, total;
  __host__ __device__ MomentLayout(int slots, int NK, int nd, int area) {
    size_t o = 0;
    tab = o; o += (size_t)kEllTerms * slots * 32 * 16;           // cubic coefficients in the interval
    mom = o; o += (size_t)kMWarps * (kEllTerms + 1) * kEllRuns * 4;  // [term][run] moments per warp, a spare row
    low = o; o += (size_t)kMWarps * (kEllLow + 1) * kEllRuns * 4;  // the low words of the first few
    stage = o; o += (size_t)kMWarps * kMStage / 2 * kMPair * 4;
    tabP = o; o += (size_t)32 * (nd + 2) * 16;                   // the item's rows of the sample table
    tabS = o; o += (size_t)NK * 8;
    tabU = o; o += (size_t)NK * 8;
    tabW = o; o += (size_t)32 * 8;
    boxh = o; o += (size_t)area * 4;
    boxl = o; o += (size_t)area * 4;
    total = o;
  }
};

size_t ellip_moment_smem(int K, int area, int nk_max, int nd) {
  return MomentLayout(ell_slots(K), nk_max, nd, area).total;
}

// Fixed-point words of two values, |v sc_hi| < 2^22: multiples of 2^20 (high) and the rest, |rest|
// <= 2^19 (low), rounded by adding 1.5 * 2^23 and read off the mantissas.
__device__ __forceinline__ void split20_pair(float2 v, float sc, float sc_hi, int2& hi, int2& lo) {
  const float2 m = make_float2(12582912.f, 12582912.f);
  const float2 h = __ffma2_rn(v, make_float2(sc_hi, sc_hi), m);
  const float2 l = __fadd2_rn(__ffma2_rn(__fadd2_rn(h, neg2(m)), make_float2(-1048576.f, -1048576.f),
                                         __fmul2_rn(v, make_float2(sc, sc))), m);
  hi = make_int2(__float_as_int(h.x) - 0x4B400000, __float_as_int(h.y) - 0x4B400000);
  lo = make_int2(__float_as_int(l.x) - 0x4B400000, __float_as_int(l.y) - 0x4B400000);
}

// (hi 2^20 + lo) scale as an FP32 pair (fixed_to_pair of the same number in 22-bit words).
__device__ __forceinline__ float2 fixed20_to_pair(int hi, int lo, float scale) {
  hi += lo >> 20;
  lo &= 0xFFFFF;
  return fixed_to_pair(hi >> 2, ((unsigned)(hi & 3) << 20) | (unsigned)lo, scale);
}

// a - b as one packed FMA (no negated copies).
__device__ __forceinline__ float2 sub2(float2 a, float2 b) { return __ffma2_rn(b, make_float2(-1.f, -1.f), a); }

struct MomentArgs {
  MixedArgs a;
  const EllGroup* groups;
};

template <int K>
__global__ void __launch_bounds__(kMThreads, 1) k_ellip_moments(const MomentArgs ma) {
  const MixedArgs& a = ma.a;
  constexpr int H = K / 2, NP = ell_pairs(K), SL = ell_slots(K), NS = SL * 32;
  constexpr int R = kEllRuns;
  extern __shared__ __align__(16) unsigned char smem[];
  const EllGroup grp = ma.groups[blockIdx.x];
  const DevSlice& S = a.slices[a.items[grp.first].slice];
  const int nd = S.degree + 1;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const MomentLayout L(SL, a.nk_max, a.max_deg + 1, 0);
  float4* tab = reinterpret_cast<float4*>(smem + L.tab);
  float* mom = reinterpret_cast<float*>(smem + L.mom) + warp * (kEllTerms + 1) * R;
  float* low = reinterpret_cast<float*>(smem + L.low) + warp * (kEllLow + 1) * R;
  float* stage = reinterpret_cast<float*>(smem + L.stage) + warp * (kMStage / 2) * kMPair;
  float4* tabP = reinterpret_cast<float4*>(smem + L.tabP);
  float2* tabS = reinterpret_cast<float2*>(smem + L.tabS);
  float2* tabU = reinterpret_cast<float2*>(smem + L.tabU);
  float2* tabW = reinterpret_cast<float2*>(smem + L.tabW);
  __shared__ double s_w[kMWarps], s_u[kMWarps];
  {  // the interval's cubics in t = 0..1 between nodes `interval` and `interval` + 1
    constexpr int n = kEllTerms * NS;
    const float* f = S.enodes + (int64_t)grp.interval * n;  // node `interval` - 1
    for (int e = tid; e < n; e += kMThreads) {
      const float fm = f[e], f0 = f[n + e], f1 = f[2 * n + e], f2_ = f[3 * n + e];
      // differences first: the nodes are close
      const float d1 = f1 - f0, dm = f0 - fm, d2 = f2_ - f1;
      const float s2 = d1 - dm;                 // second difference at node 0
      const float s3 = (d2 - d1) - s2;          // third difference
      tab[e] = make_float4(f0, d1 - 0.5f * s2 - s3 * (1.f / 6.f), 0.5f * s2, s3 * (1.f / 6.f));
    }
  }
  // the lane's block of moments: a in {2 pa, 2 pa + 1}, b in {2 pb, 2 pb + 1}, pa + pb <= 5
  int pa = 0, pb = lane;
  while (pb > 5 - pa && pa < 6) {
    pb -= 6 - pa;
    ++pa;
  }
  // and where a run's go in mom and low (past the triangle, or above degree 2: the spare rows).  Two
  // of the other lanes sum the weights themselves, M_00, from their leading 12 bits and the rest,
  // which holds what an FP32 weight leaves out.
  int mrow = 0, lrow = 0;  // a row a byte
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const int ta = 2 * pa + (q >> 1), tb = 2 * pb + (q & 1);
    const int term = pa < 6 && ta + tb <= kEllDegree ? ell_term(ta, tb) : kEllTerms;
    mrow |= term << (8 * q);
    lrow |= ell_low_row(term) << (8 * q);
  }
  const float* sx = stage + 4 * (pa < 6 ? pa : lane == 21 ? 5 : 6);
  const float* sy = stage + 4 * (pa < 6 ? 6 + pb : lane == 21 ? 6 : 11);
  const double* flux = a.flux_tab[S.flux_slot];
  const double* u = a.u_all + S.u_off;
  const double inv_ns = 1.0 / (double)S.n_slit;

  for (int gi = 0; gi < grp.count; ++gi) {
    const Item it = a.items[grp.first + gi];
    const int area = it.bw * it.bh;
    int* boxh = reinterpret_cast<int*>(smem + L.boxh);
    int* boxl = boxh + area;
    for (int e = tid; e < it.nj * (nd + 2); e += kMThreads)
      cp_async16(tabP + e, S.samples + (int64_t)it.j0 * (nd + 2) + e);
    for (int p = tid; p < 2 * area; p += kMThreads) boxh[p] = 0;
    double usum = 0.0, wsum = 0.0;
    if (tid < it.nk) {  // at most kEllMaxSlit
      const double uk = u[it.k0 + tid];
      tabS[tid] = split_df(norm_sample_r(it.k0 + tid, S.n_slit, inv_ns));
      tabU[tid] = split_df(uk);
      usum = fabs(uk);
    }
    if (tid < it.nj) {  // at most 32
      const double wj = flux[it.j0 + tid] * S.dlam;
      tabW[tid] = split_df(wj);
      wsum = fabs(wj);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      wsum += __shfl_xor_sync(0xffffffffu, wsum, o);
      usum += __shfl_xor_sync(0xffffffffu, usum, o);
    }
    if (lane == 0) {
      s_w[warp] = wsum;
      s_u[warp] = usum;
    }
    cp_async_wait_all();
    __syncthreads();
    double wtot = 0.0, utot = 0.0;
#pragma unroll
    for (int q = 0; q < kMWarps; ++q) {
      wtot += s_w[q];
      utot += s_u[q];
    }
    const double total = wtot * utot;
    // every pixel's sum is below 0.148 of the total (widths >= 1 px), so its high word fits 31 bits
    int ex = 0;
    frexp(total, &ex);
    const int Psh = total > 0.0 ? max(-100, min(100, 52 - ex)) : 0;
    const float sc = ldexpf(1.f, Psh), sc_hi = ldexpf(1.f, Psh - 20);
    int off[SL];  // the first pixels of the lane's pairs, in the box from the window's origin
#pragma unroll
    for (int i = 0; i < SL; ++i) {
      const int e = min(lane + 32 * i, NP - 1);
      off[i] = (e / K) * it.bw + e % K;
    }
    const int last = (K - 1) * (it.bw + 1);

    for (int jj = warp; jj < it.nj && total > 0.0; jj += kMWarps) {
      const float4* Pj = tabP + jj * (nd + 2);
      const FastMap fm(Pj, S.degree);
      const float2 wj = tabW[jj];
      const float t = ((float)(it.j0 + jj - grp.interval * S.espan) + 0.5f) / (float)S.espan;
      // moments (2pa, 2pb | 2pb + 1), (2pa + 1, ...), and their sums' rounding errors
      float2 m0 = make_float2(0.f, 0.f), m1 = m0, e0 = m0, e1 = m0;
      int nr = 0;                                  // runs held in mom, the present one not counted
      int cx = kOffFrame, cy = kOffFrame;          // the present run's window centre (uniform)
      int rx = 0, ry = 0;                          // lane r: the window centre of run r

      // the runs' pixels, deposited
      auto apply = [&]() {
        __syncwarp();
        float2 ev[R / 2][SL], od[R / 2][SL];
#pragma unroll
        for (int r = 0; r < R / 2; ++r)
#pragma unroll
          for (int i = 0; i < SL; ++i) ev[r][i] = od[r][i] = make_float2(0.f, 0.f);
        auto term = [&](int q, float2 (&acc)[R / 2][SL]) {
          float c[SL];
#pragma unroll
          for (int i = 0; i < SL; ++i) {
            const float4 k = tab[q * NS + lane + 32 * i];
            c[i] = fmaf(fmaf(fmaf(k.w, t, k.z), t, k.y), t, k.x);
          }
          const float4* mq = reinterpret_cast<const float4*>(mom + q * R);
#pragma unroll
          for (int r4 = 0; r4 < R / 4; ++r4) {
            const float4 m = mq[r4];
#pragma unroll
            for (int i = 0; i < SL; ++i) {
              const float2 cc = make_float2(c[i], c[i]);
              acc[2 * r4][i] = __ffma2_rn(cc, make_float2(m.x, m.y), acc[2 * r4][i]);
              acc[2 * r4 + 1][i] = __ffma2_rn(cc, make_float2(m.z, m.w), acc[2 * r4 + 1][i]);
            }
          }
        };
        // the high degrees first: these sums stay small, and so does their rounding
#pragma unroll 2
        for (int q = kEllTerms - 1; q >= kEllEven + kEllLowOdd; --q) term(q, od);
#pragma unroll 2
        for (int q = kEllEven - 1; q >= kEllLowEven; --q) term(q, ev);
        // then degrees 0 to 2, slot by slot, their sums' errors added to those of the high degrees
        // (FastTwoSum: the lowest degree, the largest, first); ev and od end as the pixels of the pairs
#pragma unroll
        for (int i = 0; i < SL; ++i) {
          float2 se[R / 2], so[R / 2];
#pragma unroll
          for (int r = 0; r < R / 2; ++r) se[r] = so[r] = make_float2(0.f, 0.f);
          auto sure = [&](int q, int lq, float2 (&s)[R / 2], float2 (&acc)[R / 2][SL]) {
            const float4 k = tab[q * NS + lane + 32 * i];
            const float c = fmaf(fmaf(fmaf(k.w, t, k.z), t, k.y), t, k.x);
            const float2 cc = make_float2(c, c);
            const float2* mq = reinterpret_cast<const float2*>(mom + q * R);
            const float2* lw = reinterpret_cast<const float2*>(low + lq * R);
#pragma unroll
            for (int r = 0; r < R / 2; ++r) {
              const float2 m = mq[r], n = __ffma2_rn(cc, m, s[r]);
              float2 e = __ffma2_rn(cc, m, sub2(s[r], n));
              e = __ffma2_rn(cc, lw[r], e);
              acc[r][i] = __fadd2_rn(acc[r][i], e);
              s[r] = n;
            }
          };
#pragma unroll 1
          for (int q = 0; q < kEllLowEven; ++q) sure(q, q, se, ev);
#pragma unroll 1
          for (int q = 0; q < kEllLowOdd; ++q) sure(kEllEven + q, kEllLowEven + q, so, od);
#pragma unroll
          for (int r = 0; r < R / 2; ++r) {  // the sums, then times the sample's flux
            const float2 p = __fadd2_rn(__fadd2_rn(se[r], so[r]), __fadd2_rn(ev[r][i], od[r][i]));
            const float2 n = __fadd2_rn(sub2(se[r], so[r]), sub2(ev[r][i], od[r][i]));
            const float2 wx = make_float2(wj.x, wj.x), wy = make_float2(wj.y, wj.y);
            ev[r][i] = __ffma2_rn(p, wx, __fmul2_rn(p, wy));
            od[r][i] = __ffma2_rn(n, wx, __fmul2_rn(n, wy));
          }
        }
#pragma unroll
        for (int r = 0; r < R; ++r) {
          if (r < nr) {  // uniform
            const int gx0 = __shfl_sync(0xffffffffu, rx, r) - H - it.bx0;
            const int gy0 = __shfl_sync(0xffffffffu, ry, r) - H - it.by0;
            float2 v[SL];
            float mx = 0.f;
#pragma unroll
            for (int i = 0; i < SL; ++i) {
              v[i] = (r & 1) ? make_float2(ev[r / 2][i].y, od[r / 2][i].y) : make_float2(ev[r / 2][i].x, od[r / 2][i].x);
              mx = fmaxf(mx, fmaxf(fabsf(v[i].x), fabsf(v[i].y)));
            }
            const bool small = __all_sync(0xffffffffu, mx * sc_hi < 4190000.f);
            if (small && gx0 >= 0 && gx0 + K <= it.bw && gy0 >= 0 && gy0 + K <= it.bh) {  // uniform
              int* p0 = boxh + gy0 * it.bw + gx0;
#pragma unroll
              for (int i = 0; i < SL; ++i) {
                int2 hi, lo;
                split20_pair(v[i], sc, sc_hi, hi, lo);
                if (32 * (i + 1) <= NP - 1 || lane + 32 * i < NP) {
                  int* p = p0 + off[i];
                  atomicAdd(p, hi.x);
                  atomicAdd(p + area, lo.x);
                }
                if (32 * (i + 1) <= NP - 1 || lane + 32 * i < NP - 1) {  // the centre is its own mirror image
                  int* p = p0 + (last - off[i]);
                  atomicAdd(p, hi.y);
                  atomicAdd(p + area, lo.y);
                }
              }
            } else {
#pragma unroll
              for (int i = 0; i < SL; ++i) {
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                  if (lane + 32 * i >= NP - h) continue;
                  const int e = h ? K * K - 1 - lane - 32 * i : lane + 32 * i;
                  const int gx = gx0 + e % K, gy = gy0 + e / K;
                  const float val = h ? v[i].y : v[i].x;
                  if (gx >= 0 && gx < it.bw && gy >= 0 && gy < it.bh) {
                    int* p = boxh + gy * it.bw + gx;
                    const float hf = rintf(val * sc_hi);
                    atomicAdd(p, __float2int_rz(hf));
                    atomicAdd(p + area, __float2int_rn(fmaf(hf, -1048576.f, val * sc)));
                  } else if (a.err && val != 0.f) {  // outside the box: legitimate only off the detector
                    const int Xd = it.bx0 + gx, Yd = it.by0 + gy;
                    if (Xd >= 0 && Xd < S.W && Yd >= 0 && Yd < S.H) atomicAdd(a.err, 1);
                  }
                }
              }
            }
          }
        }
        nr = 0;
        __syncwarp();
      };
      // the present run's moments into mom
      auto close = [&](bool end) {  // end: the sample's last run, whose pixels the caller forms
        if (cx == kOffFrame) return;
        const float ws = __shfl_sync(0xffffffffu, m1.x, 21);  // M_00: the leading bits and the rest
        const float wr = __shfl_sync(0xffffffffu, e1.x, 21) +
                         (__shfl_sync(0xffffffffu, m0.y, 22) + __shfl_sync(0xffffffffu, e0.y, 22));
        if (lane == 0) {
          m0.x = ws;
          e0.x = wr;
        }
        auto put = [&](int q, float m, float e) {
          const float h = m + e;
          mom[((mrow >> (8 * q)) & 0xff) * R + nr] = h;
          low[((lrow >> (8 * q)) & 0xff) * R + nr] = (m - h) + e;
        };
        put(0, m0.x, e0.x);
        put(1, m0.y, e0.y);
        put(2, m1.x, e1.x);
        put(3, m1.y, e1.y);
        if (lane == nr) {
          rx = cx;
          ry = cy;
        }
        m0 = m1 = e0 = e1 = make_float2(0.f, 0.f);
        if (++nr == R && !end) apply();
      };

      for (int k0 = 0; k0 < it.nk; k0 += 32) {
        const int k = min(k0 + lane, it.nk - 1);
        int ci[1], ri[1];
        float fx[1], fy[1];
        const float2 sv[1] = {tabS[k]};
        fm.map(Pj, S.degree, sv, ci, fx, ri, fy);
        const float2 uk = tabU[k];
        float w = uk.x;
        const float uh = __uint_as_float(__float_as_uint(w) & 0xFFFFF000u);
        float w_lead = uh, w_rest = (w - uh) + uk.y;
        if (k0 + lane >= it.nk || ci[0] == kOffFrame || ri[0] == kOffFrame) ci[0] = ri[0] = kOffFrame;
        const bool on = ci[0] != kOffFrame;
        if (!on) w = w_lead = w_rest = fx[0] = fy[0] = 0.f;
        // a stamp with another window than the one before it begins a run
        int px = __shfl_up_sync(0xffffffffu, ci[0], 1), py = __shfl_up_sync(0xffffffffu, ri[0], 1);
        if (lane == 0) {
          px = cx;
          py = cy;
        }
        const unsigned starts = __ballot_sync(0xffffffffu, ci[0] != px || ri[0] != py);
        const int nk = min(32, it.nk - k0);
        for (int half = 0; half < 2 && half * kMStage < nk; ++half) {
          __syncwarp();  // the staged values of the last half have been read
          {  // lanes 0-15 form the x values of the half's stamps, lanes 16-31 the y values
            const int src = half * kMStage + (lane & 15);
            const float gx = __shfl_sync(0xffffffffu, fx[0], src), gy = __shfl_sync(0xffffffffu, fy[0], src);
            const float gw = __shfl_sync(0xffffffffu, w, src), gl = __shfl_sync(0xffffffffu, w_lead, src);
            const float gr = __shfl_sync(0xffffffffu, w_rest, src);
            const bool isx = lane < 16;
            const float f = isx ? gx : gy, f4 = 4.f * f;
            float t0 = isx ? gw : 1.f, t1 = t0 * (2.f * f);
            float* o = stage + ((lane & 15) >> 1) * kMPair + (isx ? 0 : 24) + 2 * (lane & 1);
#pragma unroll
            for (int q = 0; q < 6; ++q) {
              *reinterpret_cast<float2*>(o + 4 * q) = make_float2(t0, q == 5 ? (isx ? gl : gr) : t1);
              t0 = fmaf(f4, t1, -t0);
              t1 = fmaf(f4, t0, -t1);
            }
          }
          __syncwarp();
          const int ns = min(kMStage, nk - half * kMStage);
          // segments of one run each
          unsigned st = (starts >> (half * kMStage)) & ((1u << ns) - 1u);
          for (int s = 0; s < ns;) {
            if (st & 1u) {  // uniform
              close(false);
              cx = __shfl_sync(0xffffffffu, ci[0], half * kMStage + s);
              cy = __shfl_sync(0xffffffffu, ri[0], half * kMStage + s);
            }
            st >>= 1;
            const int len = st ? __ffs(st) : ns - s;  // this stamp and those up to the next start
            const int end = s + len;
            st >>= len - 1;
            auto add = [&](float xa, float xb, float ya, float yb) {
              auto sum = [](float2 x, float2 y, float2& m, float2& e) {
                const float2 n = __ffma2_rn(x, y, m);
                e = __fadd2_rn(e, __ffma2_rn(x, y, sub2(m, n)));
                m = n;
              };
              const float2 y = make_float2(ya, yb);
              sum(make_float2(xa, xa), y, m0, e0);
              sum(make_float2(xb, xb), y, m1, e1);
            };
            auto one = [&](int q) {
              const int o = (q >> 1) * kMPair + 2 * (q & 1);
              const float2 vx = *reinterpret_cast<const float2*>(sx + o), vy = *reinterpret_cast<const float2*>(sy + o);
              add(vx.x, vx.y, vy.x, vy.y);
            };
            if (s & 1) one(s++);
#pragma unroll 2
            for (; s + 2 <= end; s += 2) {
              const float4 vx = *reinterpret_cast<const float4*>(sx + (s >> 1) * kMPair);
              const float4 vy = *reinterpret_cast<const float4*>(sy + (s >> 1) * kMPair);
              add(vx.x, vx.y, vy.x, vy.y);
              add(vx.z, vx.w, vy.z, vy.w);
            }
            if (s < end) one(s++);
          }
        }
      }
      close(true);
      if (nr > 0) apply();
    }
    __syncthreads();
    float2* out = a.store + it.store_off;
    const float inv = ldexpf(1.f, -Psh);
    for (int p = tid; p < area; p += kMThreads) out[p] = fixed20_to_pair(boxh[p], boxl[p], inv);
    __syncthreads();  // the box and the tables are the next item's
  }
}

template <int K>
static cudaError_t launch_moments_one(const MomentArgs& a, int n_groups, size_t smem, cudaStream_t st) {
  auto kern = k_ellip_moments<K>;
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  kern<<<n_groups, kMThreads, smem, st>>>(a);
  return cudaGetLastError();
}

bool ellip_moments_supported(int K) { return K >= 3 && K <= 13; }

cudaError_t launch_ellip_moments(int K, const DevSlice* slices, const double* const* flux_tab, const double* u_all,
                                 const Item* items, const EllGroup* groups, int n_groups, float2* store, int nk_max,
                                 int max_deg, size_t smem, cudaStream_t st, int* err) {
  if (n_groups == 0) return cudaSuccess;
  const MomentArgs a{MixedArgs{slices, flux_tab, u_all, items, store, 0, 1, nk_max, max_deg, err, 0}, groups};
  switch (K) {
#define E2E_CASE(KK) \
  case KK: return launch_moments_one<KK>(a, n_groups, smem, st);
    E2E_CASE(3) E2E_CASE(5) E2E_CASE(7) E2E_CASE(9) E2E_CASE(11) E2E_CASE(13)
#undef E2E_CASE
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace e2e
