// The tile merge of the tiled renderers: the boxes of the items overlapping one 64x32 output
// tile are added per pixel in item order with compensated summation (TwoSum on the FP32
// pairs, Neumaier's correction carried in a second word), converted and written once.  One
// device function serves the standalone merge kernel and the fused merge at the end of the
// edge-tail render kernel (k_render_mixed), so both give the same bits.
//
// Fused merge: every tile counts its finished items.  A render CTA, after writing its box,
// fences, adds one to the count of each tile the box overlaps, and the CTA that brings a
// tile's count to the tile's number of items merges that tile.  Nothing waits: the last
// arrival does the work, and the counts are zeroed before each render.  Tiles that no item
// overlaps are written as zeros by the standalone kernel over the plan's zero-tile list.
#pragma once
#include "e2e_device.cuh"
#include "e2e_kernels.h"
#include "mixed_common.cuh"

namespace e2e {

// A warp merges 32 neighbouring columns x kMergeRows rows at a time.
constexpr int kMergeRows = 8;
constexpr int kMergeBlocks = (kTileW / 32) * (kTileH / kMergeRows);  // such sub-blocks of a tile
// Boxes whose pixels of a sub-block are loaded together: the latency of a load from L2 is paid
// once per kMergeDepth boxes; their pixels are still added one box after the other.
constexpr int kMergeDepth = 2;

// Entry `lane` of tile t's list (zeros beyond its end).
__device__ __forceinline__ TileBox tile_entry(const Tile& t, const TileBox* __restrict__ boxes, int lane) {
  return lane < t.n ? boxes[t.list_off + lane] : TileBox{};
}

// Merge sub-block blk of tile t, by one warp; box reads bypass L1 when CG (the boxes were written
// by other CTAs during this launch).
//
// Of the boxes in a tile's list (6 on the full-detector frame, 24 on a finely sampled 1024 x 256
// tile) only two to four reach a given sub-block.  Following the list item by item (its index, the
// item, then its pixels) cost three loads from L2 per item, one after the other.  Here the lanes
// load 32 list entries at once, which hold the boxes themselves, each lane tests its box against
// the sub-block, and the warp walks the set bits of the ballot.  The boxes are added in list order.
// `first` is this lane's entry of the list's first 32 (any value beyond the list's end).
template <bool CG, typename T>
__device__ __forceinline__ void merge_block(const Tile& t, const TileBox& first, const TileBox* __restrict__ boxes,
                                            const float2* store, T* frame, int64_t P, int H, int W, int blk,
                                            int lane) {
  const int x0 = t.x0 + (blk % (kTileW / 32)) * 32, y0 = t.y0 + (blk / (kTileW / 32)) * kMergeRows;
  if (x0 >= W || y0 >= H) return;
  float sum[kMergeRows], comp[kMergeRows];
#pragma unroll
  for (int q = 0; q < kMergeRows; ++q) sum[q] = comp[q] = 0.f;
  for (int n0 = 0; n0 < t.n; n0 += 32) {
    TileBox b = first;
    bool hit = false;
    if (n0 + lane < t.n) {
      if (n0 > 0) b = boxes[t.list_off + n0 + lane];
      hit = b.bx0 < x0 + 32 && b.bx0 + b.bw > x0 && b.by0 < y0 + kMergeRows && b.by0 + b.bh > y0;
    }
    unsigned m = __ballot_sync(0xffffffffu, hit);
    const int xy = b.bx0 | (b.by0 << 16), wh = b.bw | (b.bh << 16);
    while (m) {
      float2 v[kMergeDepth][kMergeRows];
      const int nd = min(kMergeDepth, __popc(m));
#pragma unroll
      for (int d = 0; d < kMergeDepth; ++d) {
        if (d < nd) {  // uniform over the warp
          const int i = __ffs(m) - 1;
          m &= m - 1;
          const unsigned ixy = __shfl_sync(0xffffffffu, xy, i), iwh = __shfl_sync(0xffffffffu, wh, i);
          const int64_t off = __shfl_sync(0xffffffffu, b.off, i);
          const int bw = iwh & 0xffff, bh = iwh >> 16;
          const int gx = x0 + lane - (int)(ixy & 0xffff), gy = y0 - (int)(ixy >> 16);
          const float2* p = store + off + (int64_t)gy * bw + gx;
          const bool inx = (unsigned)gx < (unsigned)bw;
#pragma unroll
          for (int q = 0; q < kMergeRows; ++q) {
            const bool in = inx && (unsigned)(gy + q) < (unsigned)bh;
            v[d][q] = in ? (CG ? __ldcg(p + q * bw) : p[q * bw]) : make_float2(0.f, 0.f);
          }
        }
      }
#pragma unroll
      for (int d = 0; d < kMergeDepth; ++d) {
        if (d < nd) {
#pragma unroll
          for (int q = 0; q < kMergeRows; ++q) {
            float s, e;
            two_sum(sum[q], v[d][q].x, s, e);
            sum[q] = s;
            comp[q] += e + v[d][q].y;
          }
        }
      }
    }
  }
  const int x = x0 + lane;
  if (x >= W) return;
  T* out = frame + (int64_t)y0 * P + x;
#pragma unroll
  for (int q = 0; q < kMergeRows; ++q)
    if (y0 + q < H) out[q * P] = sizeof(T) == 8 ? (T)((double)sum[q] + (double)comp[q]) : (T)(sum[q] + comp[q]);
}

// Merge tile t with the NT threads (whole warps) of a CTA.
template <int NT, bool CG, typename T>
__device__ __forceinline__ void merge_tile(const Tile& t, const TileBox* __restrict__ boxes, const float2* store,
                                           T* frame, int64_t P, int H, int W, int tid) {
  const int lane = tid & 31;
  const TileBox first = tile_entry(t, boxes, lane);
  for (int blk = tid >> 5; blk < kMergeBlocks; blk += NT / 32)
    merge_block<CG, T>(t, first, boxes, store, frame, P, H, W, blk, lane);
}

// End of a render CTA of NT threads that has written item `it`'s box (every thread's stores
// issued): count the item into its tiles and merge the tiles it completes.
template <int NT>
__device__ void fused_merge_epilogue(const MergeArgs& g, const float2* store, const Item& it, int det) {
  __shared__ int s_tiles[NT];
  __shared__ int s_n;
  __threadfence();  // this thread's box stores are visible device-wide
  __syncthreads();  // ... and every thread's, before any count of this CTA
  const int W = g.dims[2 * det + 1], H = g.dims[2 * det];
  const int ntx_det = (W + kTileW - 1) / kTileW;
  const int tx0 = it.bx0 / kTileW, tx1 = (it.bx0 + it.bw - 1) / kTileW;
  const int ty0 = it.by0 / kTileH, ty1 = (it.by0 + it.bh - 1) / kTileH;
  const int ntx = tx1 - tx0 + 1, n = ntx * (ty1 - ty0 + 1);
  for (int base = 0; base < n; base += NT) {
    if (threadIdx.x == 0) s_n = 0;
    __syncthreads();
    const int i = base + (int)threadIdx.x;
    if (i < n) {
      const int ty = ty0 + i / ntx, tx = tx0 + i % ntx;
      const int tile = g.tile_of[g.grid_off[det] + ty * ntx_det + tx];
      __threadfence();  // release: the CTA's box (ordered before this thread by the barrier)
      if (atomicAdd(&g.count[tile], 1) + 1 == g.tiles[tile].n) {
        __threadfence();  // acquire: the other items' boxes, released before their counts
        s_tiles[atomicAdd(&s_n, 1)] = tile;
      }
    }
    __syncthreads();
    const int m = s_n;
    if (m > 0) {
      __threadfence();  // the other items' boxes, counted before ours, are visible to this CTA
      for (int k = 0; k < m; ++k) {
        const Tile t = g.tiles[s_tiles[k]];
        if (g.dtype == 0)
          merge_tile<NT, true, float>(t, g.boxes, store, static_cast<float*>(g.dst[t.det]), g.pitch[t.det], H, W,
                                      threadIdx.x);
        else
          merge_tile<NT, true, double>(t, g.boxes, store, static_cast<double*>(g.dst[t.det]), g.pitch[t.det], H,
                                       W, threadIdx.x);
      }
    }
    __syncthreads();  // s_tiles and s_n are reused by the next chunk
  }
}

}  // namespace e2e
