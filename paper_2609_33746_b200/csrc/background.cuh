// Background mass of one score row (Eq. 4), shared by the kernels that prepare it: the list sums
// of the scan's segments merged by log-sum-exp, minus the selected tokens' approximate mass.
#pragma once

#include "common.cuh"
#include "scan_common.cuh"

namespace pqhsa {

// Per scan segment of the row's unit: scale of its sums relative to the row's maximum, its
// reference in log2 units (the scan's own product, rounded as there), and the first tile
// (32 tokens of the row) past it.
struct SegTables {
  float scale[kMaxSeg], ref2[kMaxSeg];
  int end[kMaxSeg];
};

struct BgRow {
  float m;                      // max approximate logit of the row; -inf: no background at all
  int nseg;
  const float* sums;            // [segment][n_list][Gc] behind the headers, at this row's head
  const float* head;            // [segment] headers, at this row's head: reference, then Gc on: maximum
  size_t seg_stride;
  size_t lid_base;              // token row of the list ids
  float inv_seg_tiles, tile_off;
  // (for the segment ends)
  ScanSplit sp;
  long long s_u;
  int c_first;
};

// Which scan segments cover the row's unit: depends on seq_lens alone.
__device__ __forceinline__ BgRow bg_row_plan(const Plan& pl, int row, const int32_t* __restrict__ seq_lens,
                                             const float* __restrict__ partials) {
  const int b = row / pl.Hq, h = row % pl.Hq;
  const int kv = h / pl.G, hg = (h % pl.G) / pl.Gc, g = (h % pl.G) % pl.Gc;
  BgRow r;
  r.m = -CUDART_INF_F;
  r.sp = scan_split(seq_lens, pl.B, pl.N_max, pl.upb, pl.scan_ctas);
  long long base = 0;
  for (int bb = 0; bb < b; ++bb) base += (long long)seq_tiles(seq_lens, bb, pl.N_max) * pl.upb;
  const int tb = seq_tiles(seq_lens, b, pl.N_max);
  r.s_u = base + (long long)(kv * pl.n_hg + hg) * tb;
  r.c_first = 0;
  r.nseg = 0;
  if (tb > 0) {
    r.c_first = split_cta_of(r.sp, r.s_u);
    r.nseg = min(kMaxSeg, split_cta_of(r.sp, r.s_u + tb - 1) - r.c_first + 1);
  }
  r.seg_stride = (size_t)pl.Gc * (pl.n_list + 2);
  r.head = partials + (((size_t)b * pl.Hkv + kv) * pl.n_hg + hg) * pl.n_part * r.seg_stride + g;
  r.sums = r.head + 2 * pl.Gc;
  r.lid_base = ((size_t)b * pl.Hkv + kv) * (size_t)pl.N_max;
  r.inv_seg_tiles = r.sp.T > 0 ? (float)r.sp.P_eff / (float)r.sp.T : 0.f;      // segments per tile
  // tiles of segment 0 before this unit
  r.tile_off = r.nseg > 0 ? (float)(r.s_u - split_start(r.sp, r.c_first)) : 0.f;
  return r;
}

// First tile past each segment: depends on seq_lens alone.
__device__ __forceinline__ void bg_segment_ends(const BgRow& r, SegTables& seg, int n_threads) {
  for (int s = threadIdx.x; s < r.nseg; s += n_threads)
    seg.end[s] = s + 1 < r.nseg ? (int)(split_start(r.sp, r.c_first + s + 1) - r.s_u) : 0x7fffffff;
}

// A segment's sums are relative to its reference (exp2(l~ log2 e - ref log2 e)); this re-bases them
// to the row's maximum m.  Rounded the same way wherever it is formed: what is taken out of a list
// and what is put in have to carry the same factor.
__device__ __forceinline__ float bg_seg_scale(float ref, float m) {
  return fast_exp2(fmaf(ref, kLog2e, -__fmul_rn(m, kLog2e)));
}

// Reads the segment headers (after the scan), fills the tables and sets r.m (to the same value by
// every thread).  All threads of the CTA call; ends with the tables complete.
__device__ __forceinline__ void bg_row_begin(const Plan& pl, BgRow& r, SegTables& seg, int n_threads) {
  for (int s = threadIdx.x; s < r.nseg; s += n_threads) {
    seg.scale[s] = r.head[(size_t)s * r.seg_stride + pl.Gc];                  // segment maxima
    seg.ref2[s] = r.head[(size_t)s * r.seg_stride];
  }
  __syncthreads();
  float m = -CUDART_INF_F;
  for (int s = threadIdx.x & 31; s < r.nseg; s += 32) m = fmaxf(m, seg.scale[s]);
  m = warp_max(m);
  __syncthreads();
  r.m = m;
  if (m > -CUDART_INF_F) {
    for (int s = threadIdx.x; s < r.nseg; s += n_threads) {
      const float ref = seg.ref2[s];
      seg.scale[s] = seg.scale[s] > -CUDART_INF_F ? bg_seg_scale(ref, m) : 0.f;
      seg.ref2[s] = __fmul_rn(ref, kLog2e);
    }
  }
  __syncthreads();
}

// Sum over the segments of one list's exp-sums, relative to the row's maximum.
__device__ __forceinline__ float bg_list_sum(const Plan& pl, const BgRow& r, const SegTables& seg, int j) {
  float acc = 0.f;
  for (int s0 = 0; s0 < r.nseg; s0 += 8) {
    float v[8];
#pragma unroll
    for (int u = 0; u < 8; ++u)
      v[u] = s0 + u < r.nseg ? r.sums[(size_t)(s0 + u) * r.seg_stride + (size_t)j * pl.Gc] : 0.f;
#pragma unroll
    for (int u = 0; u < 8; ++u)
      if (s0 + u < r.nseg) acc = fmaf(v[u], seg.scale[s0 + u], acc);
  }
  return acc;
}

// A selected token's approximate mass leaves its list.  It can hold nearly all of its list's mass,
// and what is left after the subtraction is multiplied by the list's mean value, so the term taken
// out is formed exactly as the scan formed the term it put in (the exponent against the reference
// of the token's own segment, the same instructions) and scaled like that segment's sums: what
// remains is the rounding of the additions alone.
__device__ __forceinline__ void bg_take_out(const BgRow& r, const SegTables& seg, int pos, float score,
                                            uint32_t lid, float* __restrict__ mass) {
  // segments are equally long up to one tile: estimate, then settle against the boundaries
  const int tile = pos / kTile;
  int sg = min(r.nseg - 1, max(0, (int)(((float)tile + r.tile_off) * r.inv_seg_tiles)));
  while (sg > 0 && tile < seg.end[sg - 1]) --sg;
  while (tile >= seg.end[sg]) ++sg;                     // (the last entry is INT_MAX)
  const float x = fmaf(score, kLog2e, -seg.ref2[sg]);
  if (x > kScanNegligibleLog2) atomicAdd(&mass[lid], -(fast_exp2(x) * seg.scale[sg]));
}

__device__ __forceinline__ uint32_t bg_lid(const Plan& pl, const BgRow& r,
                                           const uint16_t* __restrict__ lids, int pos) {
  return min((uint32_t)lids[r.lid_base + pos], (uint32_t)(pl.n_list - 1));
}

}  // namespace pqhsa
