// Step 3 of the decode operator, inside the fused call with many rows: exact top-k by one CTA per row (Eq. 3)
// from the largest score of every tile of 32 tokens, which the scan leaves; it also prepares the row's
// background (Eq. 4), as select_cluster.cu does.
//
//   1. the k-th largest maximum is a lower bound of the k-th largest score: as many tiles hold a score at
//      or above it.  It is found to 1/512 (where maxima crowd, 1/2^18) of the maxima's range with a
//      histogram; at a 1 % budget 1.2 k scores of a row in random order reach it;
//   2. only the tiles that reach it are read (a third of them), and what reaches it is listed in shared
//      memory as (key, position);
//   3. a histogram of the listed keys finds the range of the k-th largest, everything above it is taken and
//      the few items inside it are compared with each other (larger score, then lower position: the stable
//      rule).
// A list that is full (scores that crowd in few tiles, or tie) is cut: it keeps the k largest and up to 128 more, what
// it takes from there on has to reach the cut (by position, where too many scores are equal), and the warps go on
// where they were.  The warps start at sixteen places of the row, so that the first cut is near the last one
// also where scores rise along it.  The result is exact for every input; a score that is not a number ranks below -inf.
// (8 x 128K, 2 %, made again from a tighter bound -> cut -> the other top-k, us: scores that crowd in runs of 40
// neighbours 347 -> 315 -> 317, of 300 381 -> 348 -> 350, rising 385 -> 348 -> 346; 1 %, rising 311 -> 295 -> 310, all
// equal 1331 -> 377 -> 1135.)
//
// What bounds it: a chain of short steps around the reads of the tiles, 128 bytes each in random order beside the
// write-back of the scan's lines.  256 rows of 128K: 37 us; of a CTA's 45 to 55 K clocks after the scan, the tiles' maxima
// and the bound take 9 to 12 K, the lists' sums 1 to 3 K, the tiles 17 to 29 K, the range of the k-th 7 to 15 K, writing the
// selection and taking it out of the sums 6 to 9 K.
// Whole decode call, sampled top-k (select.cu) and background kernel -> this one, us: 8 x 128K 299 -> 278 (budget 0.5 %
// 286 -> 260, 2 % 328 -> 319), 16 x 64K 314 -> 297, 8 x 32K 110 -> 97.
#include <cstddef>

#include "background.cuh"
#include "common.cuh"
#include "scan_common.cuh"

namespace pqhsa {

namespace {

constexpr int kTsThreads = 512;
constexpr int kTsWarps = kTsThreads / 32;
constexpr int kTsBins = 512;            // histogram ranges, the largest first
constexpr int kTsTies = 512;            // items ranked one by one
constexpr int kTsSlack = 128;           // items that a cut of the full list may keep beyond the k-th
constexpr uint32_t kNanKey = 1u;        // NaN ranks below -inf: taken only when nothing else is left
constexpr int kTsTiles = 32 * kTsThreads;      // tiles of the longest row (a bit each of a thread's mask)

struct Row {
  const float* rs;
  float* mx;                            // maxima of the tiles
  uint16_t* ids;                        // the tiles that reach the bound
  uint2* list;
  unsigned char* stage;                 // tiles on their way to the list
  uint32_t list_cap;
  int n, n_tiles;                       // scores; tiles, up to a multiple of four
};
struct TsShared {
  alignas(16) uint32_t hist[kTsBins];
  uint2 ties[kTsTies];                  // (key, position)
  uint32_t warp_n[kTsWarps];
  int next[kTsWarps], end[kTsWarps];            // of the listed tiles, those that a warp has still to read
  uint32_t n_list, n_tie, n_emit;
  uint32_t found_bin, found_above, found_count;
  uint32_t min_key, max_key, top_key, m_key;    // finite maxima; all maxima; the scan's segments
  uint32_t cut_key, cut_pos;                    // what the list takes: keys above, or equal and before the position
  int n, k;
  Row row;
  BgRow bg;
  SegTables seg;
};
static_assert(offsetof(TsShared, hist) % 16 == 0 && offsetof(TsShared, ties) % 8 == 0, "read 16 and 8 bytes at a time");
constexpr size_t kTsHead = (sizeof(TsShared) + 127) & ~size_t(127);

// The range of a complete histogram that holds the rank-th largest item (rank from 1): sh.found_*;
// found_count = 0: fewer items than that.  All threads call; ends with the CTA in step.
__device__ __noinline__ void find_range(TsShared& sh, const uint32_t* hist, uint32_t rank) {
  const int tid = threadIdx.x, lane = tid & 31;
  __syncthreads();
  if (tid < 32) {
    constexpr int kPer = kTsBins / 128;
    uint4 v[kPer];
    uint32_t sum[kPer], inc[kPer];
#pragma unroll
    for (int j = 0; j < kPer; ++j) v[j] = *reinterpret_cast<const uint4*>(hist + 4 * (lane + 32 * j));
#pragma unroll
    for (int j = 0; j < kPer; ++j) inc[j] = sum[j] = v[j].x + v[j].y + v[j].z + v[j].w;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
#pragma unroll
      for (int j = 0; j < kPer; ++j) {
        const uint32_t u = __shfl_up_sync(0xffffffffu, inc[j], o);
        if (lane >= o) inc[j] += u;
      }
    }
    if (lane == 0) { sh.found_bin = (uint32_t)kTsBins - 1u; sh.found_above = 0u; sh.found_count = 0u; }
    __syncwarp();
    uint32_t before = 0u;
#pragma unroll
    for (int j = 0; j < kPer; ++j) {
      uint32_t run = before + inc[j] - sum[j];
      before += __shfl_sync(0xffffffffu, inc[j], 31);
      if (run < rank && rank <= run + sum[j]) {
        const uint32_t c[4] = {v[j].x, v[j].y, v[j].z, v[j].w};
#pragma unroll
        for (int t = 0; t < 4; ++t) {
          if (run < rank && rank <= run + c[t]) {
            sh.found_bin = (uint32_t)(4 * (lane + 32 * j) + t);
            sh.found_above = run;
            sh.found_count = c[t];
          }
          run += c[t];
        }
      }
    }
  }
  __syncthreads();
}

// (a bound that is no number's key lets every position through)
__device__ __forceinline__ float floor_of(uint32_t key) { return key > kNanKey ? key_score(key) : -CUDART_INF_F; }
__device__ __forceinline__ uint32_t ranked_key(float x) { return x == x ? score_key(x) : kNanKey; }

// The tiles that reach lo_f, in order of position (a thread looks at neighbouring ones), shared out among the warps;
// empties the list.
__device__ __noinline__ void list_tiles(TsShared& sh, float lo_f) {
  const Row& r = sh.row;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int per = (r.n_tiles / 4 + kTsThreads - 1) / kTsThreads * 4;
  const int first = tid * per;
  uint32_t hit = 0u;
  for (int u = 0; u < per && first + u < r.n_tiles; u += 4) {
    const float4 v = *reinterpret_cast<const float4*>(r.mx + first + u);
    hit |= ((v.x < lo_f ? 0u : 1u) | (v.y < lo_f ? 0u : 2u) | (v.z < lo_f ? 0u : 4u) | (v.w < lo_f ? 0u : 8u)) << u;
  }
  const uint32_t mine = (uint32_t)__popc(hit);
  uint32_t inc = mine;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t u = __shfl_up_sync(0xffffffffu, inc, o);
    if (lane >= o) inc += u;
  }
  if (lane == 31) sh.warp_n[warp] = inc;
  __syncthreads();
  const uint32_t w = lane < kTsWarps ? sh.warp_n[lane] : 0u;
  uint32_t at = __reduce_add_sync(0xffffffffu, lane < warp ? w : 0u) + inc - mine;
  if (warp == 0) {
    const int all = (int)__reduce_add_sync(0xffffffffu, w);
    if (lane < kTsWarps) { sh.next[lane] = all * lane / kTsWarps; sh.end[lane] = all * (lane + 1) / kTsWarps; }
    if (lane == 0) sh.n_list = 0u;
  }
  while (hit) {
    const int u = __ffs(hit) - 1;
    hit &= hit - 1u;
    r.ids[at++] = (uint16_t)(first + u);
  }
  __syncthreads();
}

// The scores of the warp's listed tiles that reach the cut (a larger key, or an equal one before a position), into
// the list.  A warp takes 16 tiles at a time: copied to its 2 KB of shared memory whole lines at a time, then two
// lanes a tile, so that a score costs two instructions (the sign of the difference to the number below the cut,
// into a mask) and what follows is per hit.  (A ballot per score instead: 50 instructions a tile.)
// Ends early when the list is full (n_list beyond its capacity); the warp's next tile is then the first not listed.
// 16-byte chunk c of tile t sits at c ^ (t & 7): the lanes' reads then have no bank conflicts.
constexpr int kBatch = 16;
constexpr int kStageBytes = kTsWarps * kBatch * kTile * 4;
__device__ __noinline__ void gather(TsShared& sh) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const Row& r = sh.row;
  const int n = r.n;
  const uint32_t cap = r.list_cap;
  const float* rs = r.rs;
  const uint16_t* ids = r.ids;
  unsigned char* stage = r.stage + warp * (kBatch * kTile * 4);
  const int t = lane >> 1, half = lane & 1;
  const unsigned char* mine = stage + t * 128;
  const uint32_t cut_key = sh.cut_key, cut_pos = sh.cut_pos;
  const float lo_f = floor_of(cut_key);
  const bool all = !(lo_f > -CUDART_INF_F);             // (at or below -inf: every position counts)
  // the next number below the cut: what reaches the cut is above it, and what is no number is not
  const float under = lo_f == 0.f ? -__uint_as_float(1u) : key_score(score_key(lo_f) - 1u);
  int e0 = sh.next[warp];
  const int e1 = sh.end[warp];
#pragma unroll 1
  for (; e0 < e1; e0 += kBatch) {
    if (__any_sync(0xffffffffu, *const_cast<volatile uint32_t*>(&sh.n_list) > cap)) break;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int tt = 4 * i + (lane >> 3), c = lane & 7;
      const int p = e0 + tt < e1 ? (int)ids[e0 + tt] * kTile + 4 * c : n;
      // (the row stride is a multiple of 4 scores: a partial group of four stays inside the row)
      if (p < n)
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;"
                     ::"r"(smem_u32(stage) + (uint32_t)(tt * 128 + ((c ^ (tt & 7)) << 4))), "l"(rs + p) : "memory");
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
    const int p0 = e0 + t < e1 ? (int)ids[e0 + t] * kTile + 16 * half : n;
    asm volatile("cp.async.wait_group 0;" ::: "memory");
    __syncwarp();
    uint32_t reach = 0u;                                // bit 15 - e: score e of this lane reaches the cut
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const float4 v = *reinterpret_cast<const float4*>(mine + (((4 * half + j) ^ (t & 7)) << 4));
      reach = __funnelshift_l(__float_as_uint(under - v.x), reach, 1);
      reach = __funnelshift_l(__float_as_uint(under - v.y), reach, 1);
      reach = __funnelshift_l(__float_as_uint(under - v.z), reach, 1);
      reach = __funnelshift_l(__float_as_uint(under - v.w), reach, 1);
    }
    auto key_at = [&](int e) {
      return ranked_key(*reinterpret_cast<const float*>(mine + (((4 * half + (e >> 2)) ^ (t & 7)) << 4) + (e & 3) * 4));
    };
    const uint32_t valid = 0xffffu & ~(0xffffu >> min(16, max(0, n - p0)));      // (what was not copied is stale)
    uint32_t hit = (all ? valid : reach & valid) << 16;
    if (all || cut_pos != 0xffffffffu) {                // equal keys count by position
      for (uint32_t left = hit; left;) {
        const int e = __clz(left);
        left ^= 0x80000000u >> e;
        const uint32_t key = key_at(e);
        if (key < cut_key || (key == cut_key && (uint32_t)(p0 + e) >= cut_pos)) hit ^= 0x80000000u >> e;
      }
    }
    const uint32_t cnt = (uint32_t)__popc(hit);
    uint32_t inc = cnt;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t u = __shfl_up_sync(0xffffffffu, inc, o);
      if (lane >= o) inc += u;
    }
    uint32_t slot = 0u;
    if (lane == 31) slot = atomicAdd(&sh.n_list, inc);
    slot = __shfl_sync(0xffffffffu, slot, 31);
    const uint32_t sum = __shfl_sync(0xffffffffu, inc, 31);
    if (slot + sum > cap) {                             // full: these tiles once more after the next cut
      for (uint32_t i = slot + lane; i < cap; i += 32) r.list[i] = make_uint2(0u, 0u);     // (below every key)
      break;
    }
    slot += inc - cnt;
    while (hit) {
      const int e = __clz(hit);
      hit ^= 0x80000000u >> e;
      r.list[slot++] = make_uint2(key_at(e), (uint32_t)(p0 + e));
    }
    __syncwarp();
  }
  if (lane == 0) sh.next[warp] = e0;
}

// The list keeps what is above (lo, cut_pos), which is the cut from here on; of its other tiles a warp keeps those that
// reach it.  Called between barriers; ends with the CTA in step.  (A function of its own: what most rows skip would lie
// between steps that are fetched once per CTA, 1.2 to 2 us of a call: 8 x 32K 102.5 -> 101.1, 8 x 128K 275.0 -> 273.3.)
__device__ __noinline__ void cut_list(TsShared& sh, uint32_t n_mine, uint32_t lo, uint32_t cut_pos) {
  const Row& r = sh.row;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  if (tid == 0) { sh.n_list = 0u; sh.cut_key = lo; sh.cut_pos = cut_pos; }
  constexpr int kMove = 4;
#pragma unroll 1
  for (uint32_t i0 = 0; i0 < n_mine; i0 += kMove * kTsThreads) {
    uint2 it[kMove];
#pragma unroll
    for (int u = 0; u < kMove; ++u) {
      const uint32_t i = i0 + u * kTsThreads + tid;
      it[u] = i < n_mine ? r.list[i] : make_uint2(0u, 0u);
    }
    __syncthreads();                                    // (what is kept lands before what has been read)
#pragma unroll
    for (int u = 0; u < kMove; ++u) {
      const bool keep = it[u].x > lo || (it[u].x == lo && it[u].y < cut_pos);
      const unsigned m = __ballot_sync(0xffffffffu, keep);
      uint32_t at = 0u;
      if (lane == 0 && m) at = atomicAdd(&sh.n_list, (uint32_t)__popc(m));
      at = __shfl_sync(0xffffffffu, at, 0) + __popc(m & ((1u << lane) - 1u));
      if (keep) r.list[at] = it[u];
    }
  }
  const float lo_f = floor_of(lo);
  const int e0 = sh.next[warp], e1 = sh.end[warp];
  int e_end = e0;
#pragma unroll 1
  for (int i0 = e0; i0 < e1; i0 += 32) {
    const uint16_t tile = r.ids[min(i0 + lane, e1 - 1)];
    const bool keep = i0 + lane < e1 && !(r.mx[tile] < lo_f);
    const unsigned m = __ballot_sync(0xffffffffu, keep);
    if (keep) r.ids[e_end + __popc(m & ((1u << lane) - 1u))] = tile;
    e_end += __popc(m);
    __syncwarp();
  }
  __syncwarp();
  if (lane == 0) sh.end[warp] = e_end;
  __syncthreads();
}

// What the re-score wants to know of the top-k (fp16 tables): the listed scores, their bound and number.
struct TsCandidates {
  uint2* cand;
  uint32_t* counters;
  int32_t* rowstate;
};

template <bool kBg>
__global__ void __launch_bounds__(kTsThreads, 2)
select_tiles_kernel(Plan pl, const float* __restrict__ scores, const int32_t* __restrict__ seq_lens,
                    int32_t* __restrict__ sel_idx, int32_t* __restrict__ sel_count, float* __restrict__ kth,
                    int* __restrict__ status, const float* __restrict__ partials, const uint16_t* __restrict__ lids,
                    float* __restrict__ bg_mass, float* __restrict__ bg_max, TsCandidates cand) {
  extern __shared__ __align__(128) unsigned char s_dyn[];
  TsShared& sh = *reinterpret_cast<TsShared*>(s_dyn);
  const int tid = threadIdx.x, lane = tid & 31;
  const int row = (int)blockIdx.x;
  // what depends on the call's inputs only (one thread: the divisions are long sequences)
  if (tid == 0) {
    const int b = row / pl.Hq;
    sh.n = clamp_len(seq_lens[b], pl.N_max);
    sh.k = region_budget(pl, sh.n, b);
    sh.min_key = 0xffffffffu;
    sh.max_key = sh.top_key = sh.m_key = 0u;
    sh.n_tie = sh.n_emit = 0u;
    sh.cut_key = kNanKey;
    sh.cut_pos = 0xffffffffu;
    Row& r = sh.row;
    r.rs = scores + (size_t)row * pl.N_max;
    r.list = reinterpret_cast<uint2*>(s_dyn + kTsHead);
    r.list_cap = (uint32_t)pl.sel_list;
    r.n = sh.n;
    r.n_tiles = (sh.n + 4 * kTile - 1) / (4 * kTile) * 4;
    r.stage = reinterpret_cast<unsigned char*>(r.list + r.list_cap);
    r.mx = reinterpret_cast<float*>(r.stage + kStageBytes);
    r.ids = reinterpret_cast<uint16_t*>(r.mx + pl.n_tile);
  }
  if constexpr (kBg) {
    if (tid == 32) sh.bg = bg_row_plan(pl, row, seq_lens, partials);
  }
  if (tid < kTsBins / 4) reinterpret_cast<uint4*>(sh.hist)[tid] = make_uint4(0u, 0u, 0u, 0u);
  __syncthreads();
  const int n = sh.n, k = sh.k;
  [[maybe_unused]] SegTables& seg = sh.seg;
  [[maybe_unused]] const BgRow& bg = sh.bg;
  const Row& r = sh.row;
  const int n_mx = r.n_tiles;
  if constexpr (kBg) bg_segment_ends(bg, seg, kTsThreads);
  // The steps' instructions are fetched while the scan still runs (a first call costs 1 to 4 thousand clocks
  // more than the next): no tile is listed.
  {
    for (int o = tid; o < n_mx; o += kTsThreads) r.mx[o] = -1.f;
    __syncthreads();
    list_tiles(sh, 0.f);
    gather(sh);
    find_range(sh, sh.hist, 1u);
  }
  pdl_wait();
  pdl_launch_dependents();

  // ---- everything the scan left that is needed soon goes out at once: segment headers, tile maxima, list sums
  [[maybe_unused]] float seg_top = -CUDART_INF_F, seg_ref = 0.f;
  if constexpr (kBg) {
    static_assert(kMaxSeg <= kTsThreads, "a thread per segment");
    if (tid < bg.nseg) {
      seg_top = bg.head[(size_t)tid * bg.seg_stride + pl.Gc];
      seg_ref = bg.head[(size_t)tid * bg.seg_stride];
    }
  }
  const float4* tm = reinterpret_cast<const float4*>(pl.tile_max + (size_t)row * pl.n_tile);
  constexpr int kAtOnce = 2;
  float4 x[kAtOnce];
#pragma unroll
  for (int u = 0; u < kAtOnce; ++u) {
    const int i = u * kTsThreads + tid;
    if (i < n_mx / 4) x[u] = __ldcg(tm + i);
  }
  // The lists' sums: a list's segments are dealt out among 1, 2 or 4 threads, so that
  // what is loaded here is nearly all of them.
  constexpr int kPreLists = 2, kPreSegs = 5;
  [[maybe_unused]] const int tpl = kBg ? (bg.nseg <= kPreSegs ? 0 : bg.nseg <= 2 * kPreSegs ? 1 : 2) : 0;    // (log2)
  [[maybe_unused]] const int sub = tid & ((1 << tpl) - 1);
  [[maybe_unused]] float pre[kPreLists][kPreSegs];
  [[maybe_unused]] auto load_sums = [&](int j0) {
#pragma unroll
    for (int t = 0; t < kPreLists; ++t) {
      const int j = j0 + ((t * kTsThreads + tid) >> tpl);
      const float* at = bg.sums + (size_t)sub * bg.seg_stride + (size_t)j * pl.Gc;
#pragma unroll
      for (int u = 0; u < kPreSegs; ++u) {
        pre[t][u] = j < pl.n_list && sub + (u << tpl) < bg.nseg ? *at : 0.f;
        at += bg.seg_stride << tpl;
      }
    }
  };
  if constexpr (kBg) load_sums(0);
  {
    const int n_real = (n + kTile - 1) / kTile;
    float mn = CUDART_INF_F, mxf = -CUDART_INF_F, top = -CUDART_INF_F;
    for (int i0 = 0; i0 < n_mx / 4; i0 += kAtOnce * kTsThreads) {
#pragma unroll
      for (int u = 0; u < kAtOnce; ++u) {
        const int i = i0 + u * kTsThreads + tid;
        if (i >= n_mx / 4) continue;
        if (i0 > 0) x[u] = __ldcg(tm + i);
        float v[4] = {x[u].x, x[u].y, x[u].z, x[u].w};
#pragma unroll
        for (int t = 0; t < 4; ++t) {
          if (v[t] != v[t] || 4 * i + t >= n_real) v[t] = -CUDART_INF_F;
          top = fmaxf(top, v[t]);
          if (fabsf(v[t]) < CUDART_INF_F) { mn = fminf(mn, v[t]); mxf = fmaxf(mxf, v[t]); }
        }
        reinterpret_cast<float4*>(r.mx)[i] = make_float4(v[0], v[1], v[2], v[3]);
      }
    }
    __syncwarp();
    const uint32_t w_mn = __reduce_min_sync(0xffffffffu, score_key(mn)), w_mx = __reduce_max_sync(0xffffffffu, score_key(mxf));
    const uint32_t w_top = __reduce_max_sync(0xffffffffu, score_key(top));
    [[maybe_unused]] uint32_t w_seg = 0u;
    if constexpr (kBg) w_seg = __reduce_max_sync(0xffffffffu, score_key(seg_top));
    if (lane == 0) {
      atomicMin(&sh.min_key, w_mn);
      atomicMax(&sh.max_key, w_mx);
      atomicMax(&sh.top_key, w_top);
      if constexpr (kBg) atomicMax(&sh.m_key, w_seg);
    }
  }
  __syncthreads();
  [[maybe_unused]] float* const mass = kBg ? bg_mass + (size_t)row * pl.n_list : nullptr;
  [[maybe_unused]] const float bg_m = kBg ? key_score(sh.m_key) : 0.f;      // largest approximate logit; -inf: no background
  [[maybe_unused]] const bool has_bg = kBg && bg_m > -CUDART_INF_F;
  if constexpr (kBg) {
    if (tid < bg.nseg && has_bg) {
      seg.scale[tid] = seg_top > -CUDART_INF_F ? bg_seg_scale(seg_ref, bg_m) : 0.f;
      seg.ref2[tid] = __fmul_rn(seg_ref, kLog2e);
    }
    if (tid == 0) bg_max[row] = bg_m;
    if (k == 0) {
      __syncthreads();
      for (int j = tid; j < pl.n_list; j += kTsThreads) mass[j] = has_bg ? bg_list_sum(pl, bg, seg, j) : 0.f;
    }
  }
  if (k == 0) {
    if (tid == 0) {
      sel_count[row] = 0;
      kth[row] = CUDART_NAN_F;
      if (cand.rowstate != nullptr) cand.rowstate[row * 4 + 2] = 0;
    }
    return;
  }

  // ---- 1. the bound (somewhat lower where the re-score wants the scores around the k-th)
  const uint32_t rank = pl.rescore ? (uint32_t)(k + k / 4 + 64) : (uint32_t)k;
  uint32_t lo_key = kNanKey, hi_key;
  auto next_hist = [&]() {                              // (clear at the start; read by all before the barriers since)
    for (int i = tid; i < kTsBins; i += kTsThreads) sh.hist[i] = 0u;
    __syncthreads();
    return sh.hist;
  };
  uint32_t* hist = sh.hist;
  hi_key = sh.top_key;
  {
    const uint32_t lk = sh.min_key, hk = sh.max_key;
    if (rank <= (uint32_t)((n + kTile - 1) / kTile)) {  // (more: the maxima give no bound)
      const float mn = key_score(lk), range = key_score(hk) - mn;      // (-inf where no maximum is finite)
      // (maxima that span less than 1.5e-36 have no finite scale: like equal ones, they bound by the smallest)
      const float per_range = __fdividef((float)kTsBins, range);
      const bool spread = range > 0.f && range < CUDART_INF_F && per_range < CUDART_INF_F;
      const float scale = spread ? per_range : 0.f, width = spread ? range * (1.f / (float)kTsBins) : 0.f;
      constexpr float kLast = (float)(kTsBins - 1);
      auto bucket = [&](float v) { return fminf(fmaxf(truncf((v - mn) * scale), 0.f), kLast); };
      for (int i = tid; i < n_mx; i += kTsThreads) {
        const float v = r.mx[i];
        if (v > -CUDART_INF_F) atomicAdd(&hist[kTsBins - 1 - (int)bucket(v)], 1u);
      }
      find_range(sh, hist, rank);
      if (sh.found_count > 0u) {                        // (0: fewer finite maxima than that)
        // the range's lower edge, one range or part of it lower for the rounding
        float edge = (float)(kTsBins - 1 - (int)sh.found_bin);
        if (sh.found_count > 64u + rank / 16u && spread) {
          const uint32_t left = rank - sh.found_above;
          hist = next_hist();
          for (int i = tid; i < n_mx; i += kTsThreads) {
            const float v = r.mx[i];
            if (v > -CUDART_INF_F && bucket(v) == edge) {
              const float part = fminf(fmaxf(((v - mn) * scale - edge) * (float)kTsBins, 0.f), kLast);
              atomicAdd(&hist[kTsBins - 1 - (int)part], 1u);
            }
          }
          find_range(sh, hist, left);
          edge += ((float)(kTsBins - 1 - (int)sh.found_bin) - 1.f) / (float)kTsBins;
        } else {
          edge -= 1.f;
        }
        lo_key = max(score_key(edge > 0.f ? fmaf(edge, width, mn) : mn) - 1u, kNanKey);
      }
    }
    lo_key = min(lo_key, hi_key);
  }
  if (tid == 0) sh.cut_key = lo_key;
  list_tiles(sh, floor_of(lo_key));

  // ---- the lists' totals (stored, not added: the selected tokens are taken out with atomics after barriers)
  if constexpr (kBg) {
#pragma unroll 1
    for (int j0 = 0; j0 < pl.n_list; j0 += (kPreLists * kTsThreads) >> tpl) {
      if (j0 != 0) load_sums(j0);
#pragma unroll
      for (int t = 0; t < kPreLists; ++t) {
        const int j = j0 + ((t * kTsThreads + tid) >> tpl);
        float acc = 0.f;
        if (has_bg && j < pl.n_list) {
#pragma unroll
          for (int u = 0; u < kPreSegs; ++u) {
            const int s = sub + (u << tpl);
            if (s < bg.nseg) acc = fmaf(pre[t][u], seg.scale[s], acc);
          }
#pragma unroll 1
          for (int s0 = sub + 4 * kPreSegs; s0 < bg.nseg; s0 += 32) {      // (four threads a list)
            float v[8];
#pragma unroll
            for (int u = 0; u < 8; ++u)
              v[u] = s0 + 4 * u < bg.nseg ? bg.sums[(size_t)(s0 + 4 * u) * bg.seg_stride + (size_t)j * pl.Gc] : 0.f;
#pragma unroll
            for (int u = 0; u < 8; ++u)
              if (s0 + 4 * u < bg.nseg) acc = fmaf(v[u], seg.scale[s0 + 4 * u], acc);
          }
        }
        if (tpl > 0) acc += __shfl_xor_sync(0xffffffffu, acc, 1);
        if (tpl > 1) acc += __shfl_xor_sync(0xffffffffu, acc, 2);
        if (j < pl.n_list && sub == 0) mass[j] = acc;
      }
    }
  }

  int32_t* out = sel_idx + (size_t)row * pl.k_max;
  [[maybe_unused]] auto take_out = [&](int pos, uint32_t key, uint32_t lid) {
    if (has_bg) bg_take_out(bg, seg, pos, key_score(key), min(lid, (uint32_t)(pl.n_list - 1)), mass);
  };
  [[maybe_unused]] const uint16_t* row_lids = lids;
  if constexpr (kBg) row_lids = lids + bg.lid_base;
  constexpr int kPreLids = 4;
  [[maybe_unused]] uint32_t my_lid[kPreLids] = {};      // list ids of this thread's first listed scores

  // ---- 2. what reaches the bound, 3. the range of the k-th largest of what is listed: of keys [lo, hi] and, where
  // too many share one key, of positions [p_lo, p_hi].  A list that is full is cut there and goes on.
  uint32_t lo, hi, p_lo, p_hi, above, inside, n_mine;
  bool first_cut = true;                                // all that reaches the first bound is listed
#pragma unroll 1
  for (;;) {
    gather(sh);
    __syncthreads();
    const bool full = sh.n_list > r.list_cap;
    n_mine = min(sh.n_list, r.list_cap);
    if (n_mine < (uint32_t)k && sh.cut_key != kNanKey) {
      // no bound of the k-th score (no arithmetic above should give one): all scores
      __syncthreads();
      if (tid == 0) { sh.cut_key = kNanKey; sh.cut_pos = 0xffffffffu; }
      list_tiles(sh, -CUDART_INF_F);
      first_cut = false;
      continue;
    }
    if constexpr (kBg) {
      if (!full) {
#pragma unroll
        for (int u = 0; u < kPreLids; ++u)
          if (u * kTsThreads + tid < (int)n_mine) my_lid[u] = (uint32_t)row_lids[r.list[u * kTsThreads + tid].y];
      }
    }
    lo = sh.cut_key, hi = hi_key, p_lo = 0u, p_hi = (uint32_t)n - 1u;
    above = 0u;
    bool by_pos = false;
#pragma unroll 1
    for (;;) {
      const uint32_t span = by_pos ? p_hi - p_lo : hi - lo;
      const int shift = max(0, 32 - __clz(span) - 9);
      hist = next_hist();
#pragma unroll 1
      for (uint32_t i = tid; i < n_mine; i += kTsThreads) {
        const uint2 it = r.list[i];
        if (it.x >= lo && it.x <= hi && it.y >= p_lo && it.y <= p_hi)
          atomicAdd(&hist[(by_pos ? it.y - p_lo : hi - it.x) >> shift], 1u);
      }
      find_range(sh, hist, (uint32_t)k - above);
      above += sh.found_above;
      inside = sh.found_count;
      const uint32_t down = sh.found_bin << shift, width = (1u << shift) - 1u;
      if (by_pos) {
        p_lo += down;
        p_hi = p_lo + min(p_hi - p_lo, width);
      } else {
        hi -= down;
        lo = hi - min(hi - lo, width);
      }
      if (inside <= (uint32_t)(full ? kTsSlack : kTsTies)) break;
      if (lo == hi) by_pos = true;
    }
    if (!full) break;
    cut_list(sh, n_mine, lo, by_pos ? p_hi + 1u : 0xffffffffu);
    first_cut = false;
  }
  if (cand.cand != nullptr) {
    // (the re-score trusts the list only where it reaches down to the first bound: counter 0)
    if (first_cut) {
      uint2* dst = cand.cand + (size_t)row * pl.cand_cap;
      for (uint32_t i = tid; i < n_mine; i += kTsThreads)
        if (i < (uint32_t)pl.cand_cap) dst[i] = r.list[i];
      if (tid == 0) cand.counters[row * 4 + 3] = n_mine;
    } else if (tid == 0) {
      cand.counters[row * 4 + 0] = 1u;
    }
    if (tid == 0) {
      cand.rowstate[row * 4 + 0] = __float_as_int(floor_of(lo_key));
      cand.rowstate[row * 4 + 1] = __float_as_int(CUDART_INF_F);
      cand.rowstate[row * 4 + 2] = k;
      cand.rowstate[row * 4 + 3] = n;
    }
  }

  // ---- everything above the range, and the best of what is inside (larger score, then lower position)
#pragma unroll 1
  for (uint32_t i = tid; i < n_mine; i += kTsThreads) {
    const uint2 it = r.list[i];
    if (it.x >= lo && it.x <= hi && it.y >= p_lo && it.y <= p_hi)
      sh.ties[min(atomicAdd(&sh.n_tie, 1u), (uint32_t)kTsTies - 1u)] = it;
  }
  __syncthreads();
  const uint32_t need = (uint32_t)k - above;
  int u = 0;
#pragma unroll 1
  for (uint32_t i0 = tid & ~31; i0 < n_mine; i0 += kTsThreads, ++u) {
    const uint32_t i = i0 + lane;
    const uint32_t key = i < n_mine ? r.list[i].x : 0u, pos = i < n_mine ? r.list[i].y : 0u;
    bool take = key > hi || (key == lo && pos < p_lo);
    const unsigned m = __ballot_sync(0xffffffffu, take);
    uint32_t at = 0u;
    if (lane == 0 && m) at = atomicAdd(&sh.n_emit, (uint32_t)__popc(m));
    at = __shfl_sync(0xffffffffu, at, 0) + __popc(m & ((1u << lane) - 1u));
    if (take) {
      if (at < (uint32_t)k) out[at] = (int)pos;
    } else if (key >= lo && pos <= p_hi) {
      uint32_t better = 0u;
      for (uint32_t j = 0; j < inside; ++j) {
        const uint2 o = sh.ties[j];
        better += (o.x > key || (o.x == key && o.y < pos)) ? 1u : 0u;
      }
      if (better < need) {
        out[above + better] = (int)pos;
        take = true;
        if (better == need - 1u) {
          sel_count[row] = k;
          kth[row] = key_score(key);
        }
      }
    }
    if constexpr (kBg) {
      if (take) {
        uint32_t lid = u == 0 ? my_lid[0] : u == 1 ? my_lid[1] : u == 2 ? my_lid[2] : my_lid[3];
        if (u >= kPreLids) lid = (uint32_t)row_lids[pos];
        take_out((int)pos, key, lid);
      }
    }
  }
  if (tid == 0 && (need == 0u || inside < need)) {      // (never: the list holds the k largest)
    sel_count[row] = 0;
    kth[row] = CUDART_NAN_F;
    atomicOr(status, kStatusCountMismatch);
  }
}

constexpr size_t kSmemSplits[] = {100 * 1024, 132 * 1024, 164 * 1024, 196 * 1024, 228 * 1024};     // shared, the rest L1
size_t smem_bytes(const Plan& pl) {
  return kTsHead + (size_t)pl.sel_list * 8 + kStageBytes + (size_t)pl.n_tile * 6;
}

template <bool kBg>
cudaError_t launch_t(const Plan& pl, const float* scores, const int32_t* seq_lens, int32_t* sel_idx,
                     int32_t* sel_count, float* kth, int* status, const float* partials, const uint16_t* lids,
                     float* bg_mass, float* bg_max, const TsCandidates& cand, cudaStream_t st) {
  const cudaError_t e = allow_max_smem(select_tiles_kernel<kBg>);
  if (e != cudaSuccess) return e;
  return launch_pdl(select_tiles_kernel<kBg>, dim3(pl.rows), dim3(kTsThreads), smem_bytes(pl), st, pl, scores, seq_lens,
                    sel_idx, sel_count, kth, status, partials, lids, bg_mass, bg_max, cand);
}

}  // namespace

// Where: the maxima have to give a useful bound (no more than three quarters of the tiles selected from), and
// one CTA per row has to fill the GPU (decode call, 128K, others -> this kernel, us: 4 x 32 rows 167 -> 163,
// 3 x 32 rows 137 -> 137, 2 x 32 rows 106 -> 108, 32 rows 63 -> 78; 64 rows of 256K 168 -> 182); rows of 16K
// and less are as fast from shared memory (select_cluster.cu: 16 x 8K 90.4 and 90.3, 32 x 16K 210.7 and 211.1;
// 16 x 32K 191 -> 175).  What one CTA does alone grows with the tokens it selects, on the other path it is shared
// out: up to about 3 K of them (8 x 128K with groups of eight 2.2 % 627 -> 620; 4 x 256K 1 % 289 -> 280, 1.4 % 298 -> 300, with
// groups of eight 525 -> 520 and 558 -> 571; 2 x 512K with groups of eight 0.5 % 486 -> 458, 1 % 524 -> 521, 1.4 % 560 -> 648).
void plan_select_tiles(Plan* pl) {
  pl->sel_tiles = 0;
  pl->n_tile = (pl->N_max + 4 * kTile - 1) / (4 * kTile) * 4;
  // (most that a row selects: the exact set may be rounded up to a multiple; 8 x 128K, multiples of 4096: 883 us in lists
  // sized without it, which no row fitted into, 373 by the sampled top-k)
  long long k = ((long long)pl->N_max * pl->ppm + 999999LL) / 1000000LL + (pl->exact_multiple > 1 ? pl->exact_multiple - 1 : 0);
  if (k > pl->N_max) k = pl->N_max;
  if (4 * (k + (pl->rescore ? k / 4 + 64 : 0)) > 3LL * pl->n_tile) return;
  if (4 * pl->rows < 3 * pl->num_sms || pl->N_max <= 16384 || pl->n_tile > kTsTiles || k > 3072) return;
  pl->sel_tiles = 1;
  // A full list keeps k + 128 scores at most and a warp brings up to 512 at a time.  What the split of the SM's memory
  // that holds these CTAs has left goes to the list too (fewer cuts where scores crowd); a larger split would be
  // taken from L1 (8 x 128K, 1 %: lists of 5.9 K scores 279 us, of 2.8 K 275).
  const long long most = 7 * k / 4 > k + kTsSlack ? 7 * k / 4 : k + kTsSlack;
  pl->sel_list = (int)((most + 32 * 16 + 15) / 16 * 16);
  const size_t need = smem_bytes(*pl) + 1024;           // (1 KB per CTA is the system's)
  const size_t ctas = 2 * need <= kSmemSplits[4] ? 2 : 1;
  for (size_t split : kSmemSplits)
    if (ctas * need <= split) {
      pl->sel_list += (int)((split / ctas - need) / 128 * 16);
      break;
    }
}

cudaError_t launch_select_tiles(const Plan& pl, const WsLayout& L, char* ws, const float* scores, const int32_t* seq_lens,
                                int32_t* sel_idx, int32_t* sel_count, float* kth, int* status, cudaStream_t st) {
  TsCandidates cand = {};
  if (pl.rescore)
    cand = {reinterpret_cast<uint2*>(ws + L.cand), reinterpret_cast<uint32_t*>(ws + L.counters), reinterpret_cast<int32_t*>(ws + L.rowstate)};
  return launch_t<false>(pl, scores, seq_lens, sel_idx, sel_count, kth, status, nullptr, nullptr, nullptr, nullptr, cand, st);
}

cudaError_t launch_select_tiles_bg(const Plan& pl, const float* scores, const int32_t* seq_lens, int32_t* sel_idx,
                                   int32_t* sel_count, float* kth, int* status, const float* partials,
                                   const uint16_t* lids, float* bg_mass, float* bg_max, cudaStream_t st) {
  return launch_t<true>(pl, scores, seq_lens, sel_idx, sel_count, kth, status, partials, lids, bg_mass, bg_max, TsCandidates{}, st);
}

}  // namespace pqhsa
