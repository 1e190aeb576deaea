// Tabulated PSF: per-cell phase polynomials of the exact pixel integrals, and the stamp
// renderers that read them.
//
// A slice's PSF is given as maps (Sec. 2.1: the spectrograph unit delivers PSF maps per
// projected fiber image) at field nodes lt_f along the order: map f samples the density at
// offsets ((u - c)/q, (v - c)/q) px from the PSF centre, c = (M - 1)/2, and the density
// between samples is the bilinear interpolant, sum_uv S_uv T(q x - (u - c)) T(q y - (v - c))
// with T the unit tent.  A stamp's pixel value is that density's integral over the pixel for
// the PSF centred at the stamp's position (Sec. 2.2), which factorises:
//
//   I = sum_v sum_u S_uv X_u Y_v / norm,  X_u = (G(q (b - x_u)) - G(q (a - x_u))) / q,
//   G(t) = integral of the tent up to t (0, (1+t)^2/2, 1 - (1-t)^2/2, 1),  norm = sum S / q^2.
//
// As a function of the centre's sub-pixel phase ph (pixel edges at half-integers minus ph),
// X_u is piecewise quadratic, with knots where an edge crosses a knot of a tent: at
// ph = 1/2 - (k + c)/q.  For an integer q these knots are the same for every pixel of the
// window: cells of width 1/q, starting at ph = -1/2 for odd M, half a cell later for even M
// (then the first and last cells are half cells).  Within a cell pair (x, y) the pixel
// integral is therefore exactly a biquadratic in the phase.  At load time k_epsf_build
// evaluates it at the 3 x 3 nodes of every cell (its ends and midpoint per axis) in FP64 and
// stores the biquadratic's coefficients in the centred variable tau in [-1/2, 1/2]:
//
//   f(tau) = T1 + tau (T2 - T0) + tau^2 2 (T0 - 2 T1 + T2)   (per axis; tensor product in 2-D),
//
// in FP64 and FP32.  A stamp evaluates it by Horner in tau_x, tau_y (the terms after the first
// are small, so FP32 keeps a few-ulp error), for the two field nodes around its wavelength (the
// end node beyond the ends), blended linearly in lt: 18 coefficients per pixel, read once for
// all of an item's stamps in a cell, and no interpolation error in the phase.
#include "e2e_device.cuh"
#include "e2e_kernels.h"
#include "mixed_common.cuh"

namespace e2e {

__device__ __forceinline__ double tent_cdf(double t) {
  if (t <= -1.0) return 0.0;
  if (t <= 0.0) return 0.5 * (1.0 + t) * (1.0 + t);
  if (t <= 1.0) return 1.0 - 0.5 * (1.0 - t) * (1.0 - t);
  return 1.0;
}

// One block per (slice, node): the map's norm, sum S / q^2.
__global__ void __launch_bounds__(256) k_map_norm(const TableSlice* __restrict__ ts, const double* __restrict__ maps,
                                                  double* __restrict__ norms) {
  const TableSlice& t = ts[blockIdx.x];
  const int f = blockIdx.y;
  if (f >= t.n_field) return;
  const int M = t.map_size;
  const double* S = maps + t.map_off + (int64_t)f * M * M;
  double sum = 0.0;
  for (int i = threadIdx.x; i < M * M; i += blockDim.x) sum += S[i];
  __shared__ double red[256];
  red[threadIdx.x] = sum;
  __syncthreads();
  for (int o = 128; o > 0; o >>= 1) {
    if ((int)threadIdx.x < o) red[threadIdx.x] += red[threadIdx.x + o];
    __syncthreads();
  }
  if (threadIdx.x == 0) norms[t.field_off + f] = red[0] / ((double)t.q * t.q);
}

// Phase of node a (0, 1, 2: start, midpoint, end) of cell i on one axis: in units of 1/q from
// the cell grid's origin, cell i spans [max(i, h), min(i + 1, q + h)] with h = 1/2 for even
// maps (half cells at both ends), and ph = r / q - 1/2 - h / q.
__device__ __forceinline__ double cell_node_phase(const TableSlice& t, int i, int a) {
  const double h = t.half ? 0.5 : 0.0;
  const double lo = fmax((double)i, h), hi = fmin((double)(i + 1), (double)t.q + h);
  const double r = a == 0 ? lo : (a == 1 ? 0.5 * (lo + hi) : hi);
  return (r - h) / t.q - 0.5;
}

// Pixel integral of map f's normalised density over window pixel (m, n) for the PSF centred
// at phase (phx, phy) from the centre pixel's centre.
__device__ double epsf_pixel(const TableSlice& t, const double* S, double norm, int m, int n, double phx,
                             double phy) {
  const int H = t.K / 2, M = t.map_size;
  const double q = (double)t.q, c = 0.5 * (M - 1);
  const double ax = m - H - 0.5 - phx, bx = ax + 1.0, ay = n - H - 0.5 - phy, by = ay + 1.0;
  // samples whose tents meet [a, b): c + q a - 1 < u < c + q b + 1
  const int u0 = max(0, (int)floor(c + q * ax - 1.0)), u1 = min(M - 1, (int)ceil(c + q * bx + 1.0));
  const int v0 = max(0, (int)floor(c + q * ay - 1.0)), v1 = min(M - 1, (int)ceil(c + q * by + 1.0));
  double sum = 0.0;
  for (int v = v0; v <= v1; ++v) {
    const double yv = (v - c) / q;
    const double wy = (tent_cdf(q * (by - yv)) - tent_cdf(q * (ay - yv))) / q;
    if (wy == 0.0) continue;
    double row = 0.0;
    for (int u = u0; u <= u1; ++u) {
      const double xu = (u - c) / q;
      row += S[(int64_t)v * M + u] * ((tent_cdf(q * (bx - xu)) - tent_cdf(q * (ax - xu))) / q);
    }
    sum += row * wy;
  }
  return sum / norm;
}

// One block per (slice, node, phase cell (cy, cx)): thread (n, m) integrates the map over
// window pixel (m, n) at the cell's 3 x 3 phase nodes and stores the biquadratic's 9
// coefficients C[p][r] (power p of tau_y, r of tau_x) as rows p * 3 + r.
__global__ void __launch_bounds__(128) k_epsf_build(const TableSlice* __restrict__ ts, const double* __restrict__ maps,
                                                    const double* __restrict__ norms, int max_cells,
                                                    double* __restrict__ T64, float* __restrict__ T32) {
  const TableSlice& t = ts[blockIdx.x];
  const int f = blockIdx.y / (max_cells * max_cells);
  const int cell = blockIdx.y - f * max_cells * max_cells;
  const int cyi = cell / max_cells, cxi = cell - cyi * max_cells;
  if (f >= t.n_field || cyi >= t.n_cell || cxi >= t.n_cell) return;
  const int K = t.K, KK = K * K, M = t.map_size;
  const double* S = maps + t.map_off + (int64_t)f * M * M;
  const double norm = norms[t.field_off + f];
  double phx[3], phy[3];
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    phx[a] = cell_node_phase(t, cxi, a);
    phy[a] = cell_node_phase(t, cyi, a);
  }
  const int64_t row0 = (((int64_t)f * t.n_cell + cyi) * t.n_cell + cxi) * 9;
  const int KR = table_row32(K);
  for (int e = threadIdx.x; e < KK; e += blockDim.x) {
    const int n = e / K, m = e - n * K;
    double T[3][3];  // T[y node][x node]
#pragma unroll
    for (int a = 0; a < 3; ++a)
#pragma unroll
      for (int b = 0; b < 3; ++b) T[a][b] = epsf_pixel(t, S, norm, m, n, phx[b], phy[a]);
    // per axis: coefficients of 1, tau, tau^2 from the nodes at tau = -1/2, 0, 1/2
    double R[3][3];  // R[y node][x power]
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      R[a][0] = T[a][1];
      R[a][1] = T[a][2] - T[a][0];
      R[a][2] = 2.0 * (T[a][0] - 2.0 * T[a][1] + T[a][2]);
    }
#pragma unroll
    for (int r = 0; r < 3; ++r) {
      const double c0 = R[1][r], c1 = R[2][r] - R[0][r], c2 = 2.0 * (R[0][r] - 2.0 * R[1][r] + R[2][r]);
      const double cp[3] = {c0, c1, c2};
#pragma unroll
      for (int p = 0; p < 3; ++p) {
        const int64_t row = row0 + p * 3 + r;
        T64[t.tab_off + row * KK + e] = cp[p];
        T32[t.tab_off32 + row * KR + e] = (float)cp[p];
      }
    }
  }
}

cudaError_t launch_epsf_build(const TableSlice* ts, int n_slices, int max_field, int max_cells, const double* maps,
                              double* norms, double* T64, float* T32, cudaStream_t st) {
  if (n_slices == 0) return cudaSuccess;
  k_map_norm<<<dim3(n_slices, max_field), 256, 0, st>>>(ts, maps, norms);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  k_epsf_build<<<dim3(n_slices, max_field * max_cells * max_cells), 128, 0, st>>>(ts, maps, norms, max_cells, T64,
                                                                                    T32);
  return cudaGetLastError();
}

// Cell and centred coordinate tau in [-1/2, 1/2] of sub-pixel phase ph on one axis (FP64: the
// phase is the FP64 mapped coordinate minus its window-centre pixel).
__device__ __forceinline__ void phase_cell(const TableSlice& t, double ph, int& cell, double& tau) {
  const double h = t.half ? 0.5 : 0.0;
  const double r = (ph + 0.5) * t.q + h;
  int i = (int)floor(r);
  i = min(t.n_cell - 1, max(0, i));
  const double lo = fmax((double)i, h), hi = fmin((double)(i + 1), (double)t.q + h);
  cell = i;
  tau = (r - lo) * (hi - lo < 1.0 ? 2.0 : 1.0) - 0.5;  // cells are 1 or 1/2 wide
}

// ------------------------------------------------------------------ mixed precision

// The biquadratic C[p][r] tau_y^p tau_x^r (rows p * 3 + r) of two pixels by Horner in tau_x, then
// tau_y.
__device__ __forceinline__ float2 biquad2(const float2 (&c)[9], float2 tx, float2 ty) {
  const float2 r0 = __ffma2_rn(tx, __ffma2_rn(tx, c[2], c[1]), c[0]);
  const float2 r1 = __ffma2_rn(tx, __ffma2_rn(tx, c[5], c[4]), c[3]);
  const float2 r2 = __ffma2_rn(tx, __ffma2_rn(tx, c[8], c[7]), c[6]);
  return __ffma2_rn(ty, __ffma2_rn(ty, r2, r1), r0);
}

constexpr int kTThreads = 128;
constexpr int kTWarps = kTThreads / 32;

constexpr int kTMaxStage = 512;  // stamps of an item, staged and sorted by phase cell together
constexpr int kTMinStage = 128;  // staged at a time, unsorted, where the box leaves no room

struct TableLayout {
  size_t tabP, tabS, tabW, tabU, tabF, stage, stagew, hist, order, boxh, boxl, total;
  __host__ __device__ TableLayout(int J, int NK, int nd, int area, int cap, int cells) {
    size_t o = 0;
    tabP = o; o += (size_t)J * nd * 16;        // P_b(lt) of x and y, split_xy pairs
    tabS = o; o += (size_t)NK * 8;              // s, (hi, lo) floats
    tabW = o; o += (size_t)J * 8;
    tabU = o; o += (size_t)NK * 8;
    o = (o + 15) & ~(size_t)15;
    tabF = o; o += (size_t)J * 16;              // (f0, f1, weight of f1, -) per sample
    stage = o; o += (size_t)cap * 16;           // per staged stamp: origin, table row offsets
    stagew = o; o += (size_t)cap * 16;          // tau_x, tau_y and the two nodes' weights
    hist = o; o += cap > kTMinStage ? (size_t)cells * 4 : 0;   // stamps per phase cell, then its next place
    order = o; o += cap > kTMinStage ? (size_t)cap * 4 : 0;    // the staged stamps, cell by cell
    boxh = o; o += (size_t)area * 4;
    boxl = o; o += (size_t)area * 4;
    total = o;
  }
};

struct TableArgs {
  MixedArgs m;
  const TableSlice* ts;
  const float* T32;
  const double* field_lt;
  int cap, cells;  // stamps staged at a time; phase cells of the slice that has most
};

// One CTA per work item (<= 32 samples x <= 16 slit points).  The item's stamps are mapped into
// staging and sorted by phase cell, and each warp takes a part of the sorted list: a lane loads
// the coefficients of up to four of the window's pixels (9 at each of the cell's two field nodes,
// in registers, two pixels packed) once per cell and evaluates them for all the cell's stamps --
// five of an item's 512 at 10 samples per pixel, whose 100 cells it visits in any order.  Read
// stamp by stamp the 18 rows were 288 sectors of L2 per stamp, which bounded the kernel (89 % of
// the L2's bandwidth).  A stamp's pixels are deposited one by one as exact fixed point, in whatever
// order: the box does not depend on it.
//
// Measured on 40 slices x 4000 x 32 stamps, K = 11, 10 samples per pixel, 5 field nodes:
// 2.19 -> 1.49 ms of kernel time (2.29 -> 1.59 ms the whole render).
template <int K>
__global__ void __launch_bounds__(kTThreads, 4) k_render_table(const TableArgs ta) {
  const MixedArgs& a = ta.m;
  constexpr int KK = K * K;
  extern __shared__ __align__(16) unsigned char smem[];
  const Item it = a.items[blockIdx.x];
  const DevSlice& S = a.slices[it.slice];
  const TableSlice& TS = ta.ts[it.slice];
  const int area = it.bw * it.bh;
  const int nd = S.degree + 1;
  const TableLayout L(32, a.nk_max, a.max_deg + 1, area, ta.cap, ta.cells);
  float4* tabP = reinterpret_cast<float4*>(smem + L.tabP);
  float2* tabS = reinterpret_cast<float2*>(smem + L.tabS);
  float2* tabW = reinterpret_cast<float2*>(smem + L.tabW);
  float2* tabU = reinterpret_cast<float2*>(smem + L.tabU);
  int4* tabF = reinterpret_cast<int4*>(smem + L.tabF);
  int4* stage = reinterpret_cast<int4*>(smem + L.stage);
  float4* stagew = reinterpret_cast<float4*>(smem + L.stagew);
  int* boxh = reinterpret_cast<int*>(smem + L.boxh);
  int* boxl = reinterpret_cast<int*>(smem + L.boxl);
  __shared__ double s_w[kTWarps], s_u[kTWarps];
  __shared__ int s_sum[kTWarps];

  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  for (int p = tid; p < area; p += kTThreads) {
    boxh[p] = 0;
    boxl[p] = 0;
  }
  const double* flux = a.flux_tab[S.flux_slot];
  const double* u = a.u_all + S.u_off;
  const double inv_ns = 1.0 / (double)S.n_slit;
  double usum = 0.0;
  for (int kk = tid; kk < it.nk; kk += kTThreads) {
    const double uk = u[it.k0 + kk];
    tabS[kk] = split_df(norm_sample_r(it.k0 + kk, S.n_slit, inv_ns));
    tabU[kk] = split_df(uk);
    usum += fabs(uk);
  }
  {  // mapping coefficients and field nodes of the item's samples (per-model tables)
    const int w = nd + 2;
    const float4* rows = S.samples + (int64_t)it.j0 * w;
    for (int e = tid; e < it.nj * w; e += kTThreads) {
      const int jj = e / w, b = e - jj * w;
      if (b < nd) tabP[jj * nd + b] = rows[e];
      else if (b == nd) tabF[jj] = reinterpret_cast<const int4*>(rows)[e];
    }
  }
  double wsum = 0.0;
  for (int jj = tid; jj < it.nj; jj += kTThreads) {
    const double wj = flux[it.j0 + jj] * S.dlam;
    tabW[jj] = split_df(wj);
    wsum += fabs(wj);
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
  __syncthreads();
  double wtot = 0.0, utot = 0.0;
#pragma unroll
  for (int q = 0; q < kTWarps; ++q) {
    wtot += s_w[q];
    utot += s_u[q];
  }
  const double total = wtot * utot;
  int ex = 0;
  frexp(total, &ex);
  const int Psh = total > 0.0 ? max(-100, min(100, 52 - ex)) : 0;
  const float sc = ldexpf(1.f, Psh), sc_hi = ldexpf(1.f, Psh - 22);
  constexpr int KR = table_row32(K);  // floats per table row
  const float* T = ta.T32 + TS.tab_off32;
  // a cell's 9 coefficient rows are consecutive; n_field n_cell^2 <= 65535, so offsets fit 32 bits
  const int cell_stride = 9 * KR;
  const int node_stride = TS.n_cell * TS.n_cell * cell_stride;

  const int nst = it.nj * it.nk;
  int* hist = reinterpret_cast<int*>(smem + L.hist);
  int* order = reinterpret_cast<int*>(smem + L.order);
  const bool sorted = ta.cap > kTMinStage;
  const int cells = TS.n_cell * TS.n_cell;
  constexpr int NI = (KK + 31) / 32;   // pixels per lane: e = lane, lane + 32, ...
  constexpr int GI = NI > 4 ? 4 : NI;  // ... whose coefficients it holds at a time
  constexpr int G2 = (GI + 1) / 2;     // in packed pairs
  for (int base = 0; base < nst && total > 0.0; base += ta.cap) {
    const int ns = min(ta.cap, nst - base);
    __syncthreads();  // the last part's stamps are deposited
    if (sorted) {
      for (int c = tid; c < cells; c += kTThreads) hist[c] = 0;
      __syncthreads();
    }
    int key[kTMaxStage / kTThreads];
#pragma unroll
    for (int q = 0; q < kTMaxStage / kTThreads; ++q) {
      // map a stamp and prepare what a warp needs of it: the window origin, the offsets of its
      // phase cell's coefficient rows at its two field nodes, the cell coordinates tau_x, tau_y
      // and the nodes' weights (linear in wavelength, times the stamp weight)
      key[q] = -1;
      const int i = tid + q * kTThreads;
      if (i < ns) {
        const int idx = base + i;
        const int jj = idx / it.nk;
        const int kk = idx - jj * it.nk;
        float2 mh, ml;  // the centre as double-floats, as the planner maps it
        map_xy_df(tabP + jj * nd, S.degree, tabS[kk], mh, ml);
        int ci, ri;
        float fx, fy;
        split_coord_df(mh.x, ml.x, ci, fx);
        split_coord_df(mh.y, ml.y, ri, fy);
        const float2 wj = tabW[jj], uk = tabU[kk];
        const float w = fmaf(wj.x, uk.x, fmaf(wj.x, uk.y, wj.y * uk.x));
        const int4 fw = tabF[jj];
        int cxi = 0, cyi = 0;
        double tx = 0.0, ty = 0.0;
        if (ci != kOffFrame && ri != kOffFrame) {
          // the phase v - c exactly in FP64 (h - c is exact in FP32, the low word adds exactly)
          phase_cell(TS, (double)(mh.x - (float)ci) + (double)ml.x, cxi, tx);
          phase_cell(TS, (double)(mh.y - (float)ri) + (double)ml.y, cyi, ty);
          key[q] = cyi * TS.n_cell + cxi;
          if (sorted) atomicAdd(hist + key[q], 1);
        }
        const float wf1 = __int_as_float(fw.z);
        const int row = (cyi * TS.n_cell + cxi) * cell_stride;
        stage[i] = make_int4(ci, key[q] < 0 ? kOffFrame : ri, fw.x * node_stride + row, fw.y * node_stride + row);
        stagew[i] = make_float4((float)tx, (float)ty, (1.f - wf1) * w, wf1 * w);
      }
    }
    __syncthreads();
    int n = ns;  // stamps to deposit
    if (sorted) {
      // exclusive sums of the cells' counts: a run of cells per thread, the threads' sums by warp
      const int per = (cells + kTThreads - 1) / kTThreads, c0 = min(tid * per, cells), c1 = min(c0 + per, cells);
      int sum = 0;
      for (int c = c0; c < c1; ++c) sum += hist[c];
      int inc = sum;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int v = __shfl_up_sync(0xffffffffu, inc, o);
        if (lane >= o) inc += v;
      }
      if (lane == 31) s_sum[warp] = inc;
      __syncthreads();
      int at = inc - sum;
      n = 0;
#pragma unroll
      for (int q = 0; q < kTWarps; ++q) {
        if (q < warp) at += s_sum[q];
        n += s_sum[q];
      }
      for (int c = c0; c < c1; ++c) {
        const int v = hist[c];
        hist[c] = at;
        at += v;
      }
      __syncthreads();
#pragma unroll
      for (int q = 0; q < kTMaxStage / kTThreads; ++q)
        if (key[q] >= 0) order[atomicAdd(hist + key[q], 1)] = tid + q * kTThreads;
      __syncthreads();
    }
    // each warp its part of the list, cell by cell
    const int w0 = n * warp / kTWarps, w1 = n * (warp + 1) / kTWarps;
    for (int s0 = w0; s0 < w1;) {
      const int4 st0 = stage[sorted ? order[s0] : s0];
      int s1 = s0 + 1;  // the stamps of this cell and these nodes (uniform)
      while (s1 < w1) {
        const int4 t = stage[sorted ? order[s1] : s1];
        if (t.z != st0.z || t.w != st0.w) break;
        ++s1;
      }
      const float* A = T + st0.z + lane;   // node f0 (rows are padded with zeros to 32 floats)
      const float* Bn = T + st0.w + lane;  // node f1
#pragma unroll
      for (int i0 = 0; i0 < NI; i0 += GI) {
        float2 ca[G2][9], cb[G2][9];
#pragma unroll
        for (int h = 0; h < G2; ++h)
#pragma unroll
          for (int k = 0; k < 9; ++k) {
            const int o = 32 * (i0 + 2 * h) + k * KR;
            const bool two = i0 + 2 * h + 1 < NI;
            if (i0 + 2 * h < NI) {
              ca[h][k] = make_float2(__ldg(A + o), two ? __ldg(A + o + 32) : 0.f);
              cb[h][k] = make_float2(__ldg(Bn + o), two ? __ldg(Bn + o + 32) : 0.f);
            } else {
              ca[h][k] = cb[h][k] = make_float2(0.f, 0.f);
            }
          }
        int off[2 * G2];  // the pixels' places in the box, from the window's first
#pragma unroll
        for (int h = 0; h < 2 * G2; ++h) {
          const int ec = min(lane + 32 * (i0 + h), KK - 1);
          off[h] = (ec / K) * it.bw + ec % K;
        }
        for (int q = s0; q < s1; ++q) {
          const int i = sorted ? order[q] : q;
          const int4 st = stage[i];
          if (st.x == kOffFrame || st.y == kOffFrame) continue;
          const float4 cw = stagew[i];
          const float2 tx = make_float2(cw.x, cw.x), ty = make_float2(cw.y, cw.y);
          float2 v[G2];
#pragma unroll
          for (int h = 0; h < G2; ++h)
            v[h] = __ffma2_rn(make_float2(cw.w, cw.w), biquad2(cb[h], tx, ty),
                              __fmul2_rn(make_float2(cw.z, cw.z), biquad2(ca[h], tx, ty)));
          const int gx = st.x - K / 2 - it.bx0, gy = st.y - K / 2 - it.by0;
          // (a pixel's value is at most the stamp's weight)
          const bool small = (fabsf(cw.z) + fabsf(cw.w)) * sc_hi < 4190000.f;
          if (small && gx >= 0 && gx + K <= it.bw && gy >= 0 && gy + K <= it.bh) {
            int* p = boxh + gy * it.bw + gx;
#pragma unroll
            for (int h = 0; h < G2; ++h) {
              int2 hi, lo;
              fixed_split2_small(v[h], sc, sc_hi, hi, lo);
#pragma unroll
              for (int z = 0; z < 2; ++z) {
                if (i0 + 2 * h + z < NI && (32 * (i0 + 2 * h + z + 1) <= KK || lane + 32 * (i0 + 2 * h + z) < KK)) {
                  int* pz = p + off[2 * h + z];
                  atomicAdd(pz, z ? hi.y : hi.x);
                  atomicAdd(pz + area, z ? lo.y : lo.x);
                }
              }
            }
          } else {
#pragma unroll
            for (int h = 0; h < 2 * G2; ++h) {
              const int e = lane + 32 * (i0 + h);
              if (i0 + h >= NI || e >= KK) continue;
              const int bx = gx + e % K, by = gy + e / K;
              if (bx < 0 || bx >= it.bw || by < 0 || by >= it.bh) {
                if (a.err) {  // outside the box: legitimate only off the detector
                  const int X = it.bx0 + bx, Y = it.by0 + by;
                  if (X >= 0 && X < S.W && Y >= 0 && Y < S.H) atomicAdd(a.err, 1);
                }
                continue;
              }
              box_deposit_s(boxh + by * it.bw + bx, boxl + by * it.bw + bx, (h & 1) ? v[h / 2].y : v[h / 2].x, sc, sc_hi);
            }
          }
        }
      }
      s0 = s1;
    }
  }
  __syncthreads();
  float2* out = a.store + it.store_off;
  const float inv = ldexpf(1.f, -Psh);
  for (int p = tid; p < area; p += kTThreads) out[p] = fixed_to_pair_s(boxh[p], boxl[p], inv);
}

size_t table_smem_bytes(int area, int nk_max, int nd, int cells, size_t limit, int* cap) {
  *cap = kTMaxStage;
  const size_t n = TableLayout(32, nk_max, nd, area, kTMaxStage, cells).total;
  if (n <= limit) return n;
  *cap = kTMinStage;
  return TableLayout(32, nk_max, nd, area, kTMinStage, cells).total;
}

template <int K>
static cudaError_t launch_table_one(const TableArgs& a, int n_items, size_t smem, cudaStream_t st) {
  auto kern = k_render_table<K>;
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  kern<<<n_items, kTThreads, smem, st>>>(a);
  return cudaGetLastError();
}

cudaError_t launch_render_table(int K, const DevSlice* slices, const TableSlice* ts, const float* T32,
                                const double* field_lt, const double* const* flux_tab, const double* u_all,
                                const Item* items, int n_items, float2* store, int nk_max, int max_deg, int cap,
                                int cells, size_t smem, cudaStream_t st, int* err) {
  if (n_items == 0) return cudaSuccess;
  TableArgs a{MixedArgs{slices, flux_tab, u_all, items, store, 0, 1, nk_max, max_deg, err}, ts,
              T32, field_lt, cap, cells};
  switch (K) {
#define E2E_CASE(KK) \
  case KK: return launch_table_one<KK>(a, n_items, smem, st);
    E2E_CASE(1) E2E_CASE(3) E2E_CASE(5) E2E_CASE(7) E2E_CASE(9) E2E_CASE(11) E2E_CASE(13) E2E_CASE(15)
#undef E2E_CASE
    default: return cudaErrorInvalidValue;
  }
}

// ------------------------------------------------------------------ FP64

// One thread per stamp: FP64 mapping, FP64 coefficient tables and evaluation, FP64 atomics.
template <int K>
__global__ void __launch_bounds__(256) k_render_fp64_table(const DevSlice* __restrict__ slices,
                                                           const TableSlice* __restrict__ ts,
                                                           const double* __restrict__ T64,
                                                           const double* __restrict__ field_lt,
                                                           const double* const* __restrict__ flux_tab,
                                                           const double* __restrict__ u_all, double* const* acc,
                                                           const int64_t* __restrict__ pitch) {
  const DevSlice& S = slices[blockIdx.y];
  if (S.K != K) return;
  const TableSlice& TS = ts[blockIdx.y];
  const double* flux = flux_tab[S.flux_slot];
  const double* u = u_all + S.u_off;
  const int64_t n = (int64_t)S.n_lambda * S.n_slit;
  double* frame = acc[S.det];
  const int64_t Pf = pitch[S.det];
  constexpr int KK = K * K, H = K / 2;
  const int64_t node_stride = (int64_t)TS.n_cell * TS.n_cell * 9 * KK;
  for (int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; idx < n; idx += (int64_t)gridDim.x * blockDim.x) {
    const int j = (int)(idx / S.n_slit);
    const int k = (int)(idx - (int64_t)j * S.n_slit);
    const double lt = norm_sample(j, S.n_lambda);
    const double s = norm_sample(k, S.n_slit);
    double x = 0.0, y = 0.0;
    for (int b = S.degree; b >= 0; --b) {
      x = fma(x, s, poly_lt_for_b(S.cx, S.degree, b, lt));
      y = fma(y, s, poly_lt_for_b(S.cy, S.degree, b, lt));
    }
    x = clamp_coord(x);
    y = clamp_coord(y);
    const double ci = floor(x + 0.5), ri = floor(y + 0.5);
    const int i0 = (int)ci - H, r0 = (int)ri - H;
    if (i0 + K <= 0 || i0 >= S.W || r0 + K <= 0 || r0 >= S.H) continue;
    const double w = flux[j] * S.dlam * u[k];
    int f0, f1;
    double wf;
    field_weight(field_lt + TS.field_off, TS.n_field, lt, f0, f1, wf);
    int cxi, cyi;
    double tx, ty;
    phase_cell(TS, x - ci, cxi, tx);
    phase_cell(TS, y - ri, cyi, ty);
    const int64_t row = (int64_t)(cyi * TS.n_cell + cxi) * 9 * KK;
    const double* T0 = T64 + TS.tab_off + (int64_t)f0 * node_stride + row;
    const double* T1 = T64 + TS.tab_off + (int64_t)f1 * node_stride + row;
    for (int nn = 0; nn < K; ++nn) {
      const int r = r0 + nn;
      if (r < 0 || r >= S.H) continue;
      for (int m = 0; m < K; ++m) {
        const int i = i0 + m;
        if (i < 0 || i >= S.W) continue;
        const int e = nn * K + m;
        double v = 0.0;
        for (int side = 0; side < 2; ++side) {
          const double we = side ? wf : 1.0 - wf;
          if (we == 0.0) continue;
          const double* C = (side ? T1 : T0) + e;
          double rp[3];
          for (int p = 0; p < 3; ++p)
            rp[p] = fma(tx, fma(tx, C[(p * 3 + 2) * KK], C[(p * 3 + 1) * KK]), C[(p * 3) * KK]);
          v += we * fma(ty, fma(ty, rp[2], rp[1]), rp[0]);
        }
        atomicAdd(frame + (int64_t)r * Pf + i, w * v);
      }
    }
  }
}

cudaError_t launch_render_fp64_table(int K, int n_slices, int64_t max_stamps, const DevSlice* slices,
                                     const TableSlice* ts, const double* T64, const double* field_lt,
                                     const double* const* flux_tab, const double* u_all, double* const* acc,
                                     const int64_t* pitch, cudaStream_t st) {
  if (n_slices == 0 || max_stamps == 0) return cudaSuccess;
  int64_t bx = (max_stamps + 255) / 256;
  if (bx > 4096) bx = 4096;
  dim3 grid((unsigned)bx, (unsigned)n_slices);
  switch (K) {
#define E2E_CASE(KK) \
  case KK: k_render_fp64_table<KK><<<grid, 256, 0, st>>>(slices, ts, T64, field_lt, flux_tab, u_all, acc, pitch); break;
    E2E_CASE(1) E2E_CASE(3) E2E_CASE(5) E2E_CASE(7) E2E_CASE(9) E2E_CASE(11) E2E_CASE(13) E2E_CASE(15)
#undef E2E_CASE
    default: return cudaErrorInvalidValue;
  }
  return cudaGetLastError();
}

}  // namespace e2e
