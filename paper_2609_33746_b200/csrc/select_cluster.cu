// Step 3 of the decode operator for few or short score rows: exact top-k by one thread-block cluster per
// row (Eq. 3); in the fused call it also prepares the row's background (Eq. 4: the scan's list sums
// merged, the selected tokens' approximate mass taken out), so that no kernel of its own has to.
//
// With few or short rows the sampled two-kernel path (select.cu) and the background preparation are
// bound by latency: three launches, each a chain of dependent memory round trips over a few MB.
// Here the CS CTAs of a cluster hold the row in shared memory (one bulk copy per slice) and
// agree through distributed shared memory, so the row is read from L2 once, nothing is sampled
// and no counter lives in global memory:
//   1. every thread takes the maxima of groups of its scores; a cluster-wide histogram of the
//      group maxima over 512 ranges of 1/16 of a power of two below the row's largest score gives a
//      lower bound of the k-th largest score: the k-th largest group maximum is a score with at
//      least k scores at or above it (exact for any data; the groups only decide how tight it is);
//   2. the scores at or above the bound are listed, and a cluster-wide histogram of them over 512
//      equal ranges of keys finds the range of the k-th largest; the range is refined 512-fold until
//      the few items inside fit one CTA (a refinement is needed only when scores pile up), at last
//      over the positions of equal scores;
//   3. everything above the range is emitted to slots from a prefix sum over the cluster; the items
//      inside it are ranked by (score, lower position first) in CTA 0.
// The result is the exact top-k with the stable tie rule for every input; a score that is not a number
// (the token's cached key has one) ranks below -inf.
//
// What bounds it: latency.  A cluster barrier costs 600 to 1000 clocks, and the kernel runs through
// its code once, so that instruction fetches are the largest stall (4.4 warps per issue of 16).
// Hence 512 ranges that every CTA sums by itself (one barrier per histogram, not two), and loops
// and calls that are not unrolled or inlined.  Measured as the whole decode call, sampled top-k and
// background kernel -> this kernel: 36.0 -> 22.0 us (4 rows of 4K), 54 -> 38 (32 x 32K), 81 -> 64
// (32 x 128K), 77 -> 53 (64 rows up to 48K).
#include "background.cuh"
#include "common.cuh"
#include "scan_common.cuh"

namespace pqhsa {

namespace {

constexpr int kClThreads = 512;
constexpr int kClWarps = kClThreads / 32;
constexpr int kClBins = 512;            // histogram ranges, the largest scores first
constexpr int kClTies = 1024;           // items CTA 0 ranks at the end
constexpr int kClList = 3072;           // scores at or above the bound that a CTA lists
constexpr int kClMax = 8;               // largest cluster
constexpr int kOctaveShift = 19;        // step 1: 16 ranges per power of two
constexpr uint32_t kNanKey = 1u;        // NaN ranks below -inf: taken only when nothing else is left

// ---- cluster primitives
__device__ __forceinline__ uint32_t cluster_rank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
__device__ __forceinline__ void cluster_arrive() {
  asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
}
__device__ __forceinline__ void cluster_wait() {
  asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ void cluster_sync() { cluster_arrive(); cluster_wait(); }
// address of this CTA's shared-memory location `p` in CTA `rank` of the cluster
__device__ __forceinline__ uint32_t map_rank(const void* p, uint32_t rank) {
  uint32_t a;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"(smem_u32(p)), "r"(rank));
  return a;
}
__device__ __forceinline__ uint32_t ld_cluster(uint32_t a) {
  uint32_t v;
  asm volatile("ld.shared::cluster.u32 %0, [%1];" : "=r"(v) : "r"(a) : "memory");
  return v;
}
__device__ __forceinline__ uint4 ld_cluster_v4(uint32_t a) {
  uint4 v;
  asm volatile("ld.shared::cluster.v4.u32 {%0, %1, %2, %3}, [%4];"
               : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(a) : "memory");
  return v;
}
__device__ __forceinline__ void st_cluster_v2(uint32_t a, uint32_t x, uint32_t y) {
  asm volatile("st.shared::cluster.v2.u32 [%0], {%1, %2};" ::"r"(a), "r"(x), "r"(y) : "memory");
}

struct ClShared {
  uint32_t hist[2][kClBins];            // used in turn, so that one can be cleared while CTAs read the other
  uint2 list[kClList];                  // this CTA's scores at or above the bound: (key, position)
  uint2 ties[kClTies];                  // CTA 0: (key, position)
  uint32_t warp_a[kClWarps], warp_b[kClWarps];
  uint32_t n_list;                      // scores at or above the bound in this CTA
  uint32_t n_above, n_tie;              // what this CTA will emit / hand to CTA 0
  uint32_t found_bin, found_above, found_count;
  uint32_t kstar;
  uint32_t max_key;
  int n, k;
  BgRow bg;
  SegTables seg;
  uint64_t bar;
};

// After every CTA of the cluster has filled histogram `hist`: the range that holds the rank-th
// largest item (rank counted from 1), the items in the ranges before it and the items in it.
// Every CTA sums all histograms by itself (remote reads cost about 16 clocks per 128 bytes, a
// cluster barrier 600 to 1000: few ranges, and no second exchange).  Results in sh.found_*.
// (Not inlined: the kernel runs through its code once, and instruction fetches are what it waits
// for most.)
__device__ __noinline__ void cluster_find(ClShared& sh, uint32_t* hist, uint32_t rank, uint32_t cs, uint32_t me) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  constexpr int kW = kClBins / 128;                     // warps that take part: 4 ranges per lane
  if (tid == 0) { sh.found_bin = (uint32_t)kClBins - 1u; sh.found_above = 0u; sh.found_count = 0u; }
  if (cs > 1) cluster_sync(); else __syncthreads();     // all histograms complete
  uint4 v = make_uint4(0u, 0u, 0u, 0u);
  uint32_t local = 0u, inc = 0u;
  if (warp < kW) {
    uint32_t* own = hist + 4 * tid;
    v = *reinterpret_cast<const uint4*>(own);
    if (cs > 1) {
      uint4 r[kClMax - 1];
#pragma unroll
      for (int q = 1; q < kClMax; ++q)
        r[q - 1] = q < (int)cs ? ld_cluster_v4(map_rank(own, (me + q) & (cs - 1))) : make_uint4(0u, 0u, 0u, 0u);
#pragma unroll
      for (int q = 0; q < kClMax - 1; ++q) { v.x += r[q].x; v.y += r[q].y; v.z += r[q].z; v.w += r[q].w; }
    }
    local = v.x + v.y + v.z + v.w;
    inc = local;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t u = __shfl_up_sync(0xffffffffu, inc, o);
      if (lane >= o) inc += u;
    }
    if (lane == 31) sh.warp_a[warp] = inc;
  }
  __syncthreads();
  if (warp < kW) {
    uint32_t run = inc - local;
#pragma unroll
    for (int w = 0; w < kW - 1; ++w) run += w < warp ? sh.warp_a[w] : 0u;
    if (run < rank && rank <= run + local) {
      const uint32_t c[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        if (c[j] && run < rank && rank <= run + c[j]) {
          sh.found_bin = (uint32_t)(4 * tid + j);
          sh.found_above = run;
          sh.found_count = c[j];
        }
        run += c[j];
      }
    }
  }
  __syncthreads();
}

// A CTA's part of the row in shared memory.
struct Slice {
  const float4* s;
  int cnt, n4, begin;                   // scores, float4 groups, position of the first one in the row
  __device__ __forceinline__ float4 get(int i4) const {      // -inf past the slice's end
    const float ninf = -CUDART_INF_F;
    if (i4 >= n4) return make_float4(ninf, ninf, ninf, ninf);
    return s[i4];                       // (the last group was padded with -inf)
  }
  // Calls f(key, position, slot) for every score with key >= lo, slot = claim(hits of this lane) +
  // their index.  Hits are marked first, four float4 at a time, so that the divergent part runs
  // once per hit of a lane and not once per float4.  Every lane of a warp calls claim as often.
  template <class C, class F> __device__ __forceinline__ void for_hits(uint32_t lo, C claim, F f) const {
    float lo_f = key_score(lo);
    if (lo_f == 0.f) lo_f = -0.f;                       // (so that -0 - lo_f is not negative)
    const bool all = !(lo_f > -CUDART_INF_F);           // (bound at or below -inf: every position counts)
    for (int w0 = threadIdx.x & ~31; w0 < n4; w0 += 4 * kClThreads) {
      const int i0 = w0 + (threadIdx.x & 31);
      uint32_t miss = 0u;                               // bit 15 - e: score e of this lane is below
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const float4 v = get(i0 + u * kClThreads);
        // (the sign of the difference: two instructions per score)
        miss = __funnelshift_l(__float_as_uint(v.x - lo_f), miss, 1);
        miss = __funnelshift_l(__float_as_uint(v.y - lo_f), miss, 1);
        miss = __funnelshift_l(__float_as_uint(v.z - lo_f), miss, 1);
        miss = __funnelshift_l(__float_as_uint(v.w - lo_f), miss, 1);
      }
      uint32_t hit = ~miss << 16;
      if (all) {
        hit = 0u;
#pragma unroll 1
        for (int u = 0; u < 4; ++u)
          hit |= ((0xf0u >> min(4, max(0, cnt - 4 * (i0 + u * kClThreads)))) & 15u) << (28 - 4 * u);
      }
      uint32_t slot = claim((uint32_t)__popc(hit));
      while (hit) {
        const int e = __clz(hit);
        hit ^= 0x80000000u >> e;
        const int p = 4 * (i0 + (e >> 2) * kClThreads) + (e & 3);
        const float v = reinterpret_cast<const float*>(s)[p];
        f(v == v ? score_key(v) : kNanKey, begin + p, slot++);
      }
    }
  }
  template <class F> __device__ __forceinline__ void for_hits(uint32_t lo, F f) const {
    for_hits(lo, [](uint32_t) { return 0u; }, [&](uint32_t key, int pos, uint32_t) { f(key, pos); });
  }
};

// Range of a key below the row's largest one: kClBins ranges of 1/16 of a power of two.
__device__ __forceinline__ uint32_t octave_bin(uint32_t key, uint32_t hi_key) {
  return min((hi_key >> kOctaveShift) - (key >> kOctaveShift), (uint32_t)kClBins - 1u);
}

// Maxima of groups of 4 U scores (a thread's own loads, 512 float4 apart, so that neighbours of
// the row fall into different groups) into the histogram of step 1.
template <int U> __device__ __forceinline__ void group_hist(const Slice& sl, uint32_t* hist, uint32_t hi_key) {
  for (int i0 = threadIdx.x; i0 < sl.n4; i0 += U * kClThreads) {
    float m = -CUDART_INF_F;
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const float4 v = sl.get(i0 + u * kClThreads);
      m = fmaxf(m, fmaxf(fmaxf(v.x, v.y), fmaxf(v.z, v.w)));
    }
    atomicAdd(&hist[octave_bin(score_key(m), hi_key)], 1u);
  }
}

template <bool kBg, int kPerSm>
__global__ void __launch_bounds__(kClThreads, kPerSm)
select_cluster_kernel(Plan pl, const float* __restrict__ scores, const int32_t* __restrict__ seq_lens,
                      int32_t* __restrict__ sel_idx, int32_t* __restrict__ sel_count,
                      float* __restrict__ kth, int* __restrict__ status,
                      const float* __restrict__ partials, const uint16_t* __restrict__ lids,
                      float* __restrict__ bg_mass, float* __restrict__ bg_max) {
  extern __shared__ __align__(128) unsigned char s_dyn[];
  ClShared& sh = *reinterpret_cast<ClShared*>(s_dyn);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const uint32_t cs = (uint32_t)pl.sel_cluster, me = cluster_rank();
  const int row = (int)(blockIdx.x / cs);
  auto sync_all = [&]() { if (cs > 1) cluster_sync(); else __syncthreads(); };
  // what depends on the call's inputs only (one thread: the divisions are long sequences)
  if (tid == 0) {
    const int b = row / pl.Hq;
    sh.n = clamp_len(seq_lens[b], pl.N_max);
    sh.k = region_budget(pl, sh.n, b);
    sh.max_key = 0u;
    sh.n_list = 0u;
    mbar_init(&sh.bar, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if constexpr (kBg) {
    if (tid == 32) sh.bg = bg_row_plan(pl, row, seq_lens, partials);
  }
  for (int i = tid; i < 2 * kClBins / 4; i += kClThreads)
    reinterpret_cast<uint4*>(sh.hist)[i] = make_uint4(0u, 0u, 0u, 0u);
  __syncthreads();
  const int n = sh.n, k = sh.k;
  const int per = ((n + 4 * (int)cs - 1) / (4 * (int)cs)) * 4;       // scores per CTA, a multiple of 4
  Slice sl;
  sl.begin = min(n, (int)me * per);
  sl.cnt = min(n, sl.begin + per) - sl.begin;
  sl.n4 = (sl.cnt + 3) >> 2;
  float4* const slice = reinterpret_cast<float4*>(s_dyn + ((sizeof(ClShared) + 127) & ~size_t(127)));
  sl.s = slice;
  [[maybe_unused]] SegTables& seg = sh.seg;
  [[maybe_unused]] const BgRow& bg = sh.bg;
  if constexpr (kBg) bg_segment_ends(bg, seg, kClThreads);
  pdl_wait();
  pdl_launch_dependents();
  if (tid == 0 && sl.cnt > 0) {
    // whole 16-byte granules: the row stride is a multiple of 4 scores, so the tail stays inside it
    const uint32_t bytes = (uint32_t)sl.n4 * 16u;
    mbar_expect_tx(&sh.bar, bytes);
    bulk_g2s(slice, scores + (size_t)row * pl.N_max + sl.begin, bytes, &sh.bar);
  }
  [[maybe_unused]] float* const mass = kBg ? bg_mass + (size_t)row * pl.n_list : nullptr;
  // This CTA's share of the lists' sums: four threads per list, a list's segments dealt out among
  // them.  The first loads are issued here and used only after the first exchange.
  [[maybe_unused]] const int jl = kBg ? (int)me * pl.n_list / (int)cs : 0;
  [[maybe_unused]] const int jh = kBg ? (int)(me + 1) * pl.n_list / (int)cs : 0;
  constexpr int kPreLists = 2, kPreSegs = 5;
  [[maybe_unused]] float pre[kPreLists][kPreSegs];
  if constexpr (kBg) {
#pragma unroll
    for (int t = 0; t < kPreLists; ++t) {
      const int j = jl + t * (kClThreads / 4) + (tid >> 2);
#pragma unroll
      for (int u = 0; u < kPreSegs; ++u) {
        const int s = (tid & 3) + 4 * u;
        pre[t][u] = j < jh && s < bg.nseg ? bg.sums[(size_t)s * bg.seg_stride + (size_t)j * pl.Gc] : 0.f;
      }
    }
    bg_row_begin(pl, sh.bg, seg, kClThreads);
    if (me == 0 && tid == 0) bg_max[row] = bg.m;
  }
  if (sl.cnt > 0) {
    if (!mbar_wait(&sh.bar, 0u) && tid == 0) atomicOr(status, kStatusCopyTimeout);
    if (tid < 4 * sl.n4 - sl.cnt) reinterpret_cast<float*>(slice)[sl.cnt + tid] = -CUDART_INF_F;
    __syncthreads();
  }
  if (k == 0) {                                         // uniform over the cluster
    if constexpr (kBg) {
      for (int j = jl + tid; j < jh; j += kClThreads)
        mass[j] = bg.m > -CUDART_INF_F ? bg_list_sum(pl, bg, seg, j) : 0.f;
    }
    if (me == 0 && tid == 0) { sel_count[row] = 0; kth[row] = CUDART_NAN_F; }
    return;
  }

  // ---- 1. lower bound of the k-th largest.  Groups of 4 U scores: about 2 k groups or more, so
  // that the bound lets through at most ~1.4 k scores of a row in random order
  // (the ranges are relative to the row's largest score: with the background it is the maximum of
  // the scan's segments, otherwise one more exchange)
  uint32_t hi_key;
  if constexpr (kBg) {
    hi_key = score_key(bg.m);
  } else {
    float top = -CUDART_INF_F;
    for (int i = tid; i < sl.n4; i += kClThreads) {
      const float4 v = sl.get(i);
      top = fmaxf(top, fmaxf(fmaxf(v.x, v.y), fmaxf(v.z, v.w)));
    }
    const uint32_t key = __reduce_max_sync(0xffffffffu, score_key(top));
    if (lane == 0) atomicMax(&sh.max_key, key);
    sync_all();
    const uint32_t mk = lane < (int)cs ? ld_cluster(map_rank(&sh.max_key, (uint32_t)lane)) : 0u;
    hi_key = __reduce_max_sync(0xffffffffu, mk);
  }
  if (n / 64 >= k) group_hist<8>(sl, sh.hist[0], hi_key);
  else if (n / 32 >= k) group_hist<4>(sl, sh.hist[0], hi_key);
  else if (n / 16 >= k) group_hist<2>(sl, sh.hist[0], hi_key);
  else if (n / 8 >= k) group_hist<1>(sl, sh.hist[0], hi_key);
  else sl.for_hits(1u, [&](uint32_t key, int) { atomicAdd(&sh.hist[0][octave_bin(key, hi_key)], 1u); });
  cluster_find(sh, sh.hist[0], (uint32_t)k, cs, me);
  uint32_t bin = sh.found_bin;
  // The lists' totals are stored, not added: the selected tokens are taken out with atomics, which
  // follow a cluster barrier.
  if constexpr (kBg) {
    const bool any = bg.m > -CUDART_INF_F;
    int t = 0;
#pragma unroll 1
    for (int j0 = jl; j0 < jh; j0 += kClThreads / 4, ++t) {
      const int j = j0 + (tid >> 2);
      float acc = 0.f;
      if (any && j < jh) {
#pragma unroll
        for (int u = 0; u < kPreSegs; ++u) {
          const int s = (tid & 3) + 4 * u;
          float v = t == 0 ? pre[0][u] : pre[1][u];
          if (t >= kPreLists) v = s < bg.nseg ? bg.sums[(size_t)s * bg.seg_stride + (size_t)j * pl.Gc] : 0.f;
          if (s < bg.nseg) acc = fmaf(v, seg.scale[s], acc);
        }
#pragma unroll 1
        for (int s0 = (tid & 3) + 4 * kPreSegs; s0 < bg.nseg; s0 += 32) {
          float v[8];
#pragma unroll
          for (int u = 0; u < 8; ++u)
            v[u] = s0 + 4 * u < bg.nseg ? bg.sums[(size_t)(s0 + 4 * u) * bg.seg_stride + (size_t)j * pl.Gc] : 0.f;
#pragma unroll
          for (int u = 0; u < 8; ++u)
            if (s0 + 4 * u < bg.nseg) acc = fmaf(v[u], seg.scale[s0 + 4 * u], acc);
        }
      }
      acc += __shfl_xor_sync(0xffffffffu, acc, 1);
      acc += __shfl_xor_sync(0xffffffffu, acc, 2);
      if (j < jh && (tid & 3) == 0) mass[j] = acc;
    }
  }
  // scores in play: lo_key <= key <= hi_key (the last range reaches down to the smallest key)
  uint32_t lo_key = bin + 1u < (uint32_t)kClBins ? max(((hi_key >> kOctaveShift) - bin) << kOctaveShift, 1u) : 1u;
  const uint32_t bound = lo_key;

  // ---- 2. the range of keys (then of positions among equal keys) that holds the k-th largest.
  // The first pass also lists the scores at or above the bound; later passes walk that list.
  uint32_t above = 0u;                                  // scores above the current range
  uint32_t m_in = 0u;                                   // scores inside it
  bool by_pos = false, listed = false;
  int p_lo = 0, p_hi = n - 1;                           // positions in play once keys are equal
  uint32_t* hist = sh.hist[1];
#pragma unroll 1
  for (int pass = 0;; ++pass) {
    // 512 equal ranges: width 2^shf, the smallest that covers the span
    const uint32_t span = by_pos ? (uint32_t)(p_hi - p_lo) : hi_key - lo_key;
    const int shf = max(0, 32 - __clz(span) - 9);
    auto count = [&](uint32_t key, int pos) {
      if (!by_pos) {
        if (key >= lo_key && key <= hi_key) atomicAdd(&hist[(hi_key - key) >> shf], 1u);
      } else {                                          // lower positions rank higher
        if (key == lo_key && pos >= p_lo && pos <= p_hi) atomicAdd(&hist[(uint32_t)(pos - p_lo) >> shf], 1u);
      }
    };
    if (pass == 0) {
      sl.for_hits(bound, [&](uint32_t hits) {           // slots: one atomic per warp
        uint32_t inc = hits;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
          const uint32_t u = __shfl_up_sync(0xffffffffu, inc, o);
          if (lane >= o) inc += u;
        }
        uint32_t base = 0u;
        if (lane == 31 && inc) base = atomicAdd(&sh.n_list, inc);
        return __shfl_sync(0xffffffffu, base, 31) + inc - hits;
      }, [&](uint32_t key, int pos, uint32_t i) {
        count(key, pos);
        if (i < (uint32_t)kClList) sh.list[i] = make_uint2(key, (uint32_t)pos);
      });
      __syncthreads();
      listed = sh.n_list <= (uint32_t)kClList;
      if constexpr (kBg) {
        // the list ids of the listed scores are on their way to L1 while the histograms meet
        for (int i = tid; listed && i < (int)sh.n_list; i += kClThreads)
          asm volatile("prefetch.global.L1 [%0];" ::"l"(lids + bg.lid_base + sh.list[i].y));
      }
    } else if (listed) {
      for (int i = tid; i < (int)sh.n_list; i += kClThreads) count(sh.list[i].x, (int)sh.list[i].y);
    } else {
      sl.for_hits(bound, count);
    }
    cluster_find(sh, hist, (uint32_t)k - above, cs, me);
    bin = sh.found_bin;
    above += sh.found_above;
    m_in = sh.found_count;
    if (!by_pos) {
      hi_key -= bin << shf;
      lo_key = hi_key - min(hi_key - lo_key, (1u << shf) - 1u);
    } else {
      p_lo += (int)(bin << shf);
      p_hi = min(p_hi, p_lo + (int)((1u << shf) - 1u));
    }
    if (m_in <= (uint32_t)kClTies) break;
    if (!by_pos && lo_key == hi_key) by_pos = true;
    // the other histogram was last read before the barrier inside cluster_find
    hist = sh.hist[pass & 1];
    for (int i = tid; i < kClBins / 4; i += kClThreads)
      reinterpret_cast<uint4*>(hist)[i] = make_uint4(0u, 0u, 0u, 0u);
    __syncthreads();
  }

  // ---- 3. emission: count, prefix over the cluster, write
  uint32_t n_a = 0u, n_t = 0u;
  auto is_above = [&](uint32_t key, int pos) { return key > hi_key || (by_pos && key == lo_key && pos < p_lo); };
  auto is_in = [&](uint32_t key, int pos) {
    return key >= lo_key && key <= hi_key && (!by_pos || (pos >= p_lo && pos <= p_hi));
  };
  auto tally = [&](uint32_t key, int pos) {
    n_a += is_above(key, pos) ? 1u : 0u;
    n_t += is_in(key, pos) ? 1u : 0u;
  };
  if (listed) {
#pragma unroll 1
    for (int i = tid; i < (int)sh.n_list; i += kClThreads) tally(sh.list[i].x, (int)sh.list[i].y);
  } else {
    sl.for_hits(bound, tally);
  }
  uint32_t inc_a = n_a, inc_t = n_t;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t ua = __shfl_up_sync(0xffffffffu, inc_a, o), ut = __shfl_up_sync(0xffffffffu, inc_t, o);
    if (lane >= o) { inc_a += ua; inc_t += ut; }
  }
  if (lane == 31) { sh.warp_a[warp] = inc_a; sh.warp_b[warp] = inc_t; }
  __syncthreads();
  uint32_t at_a, at_t;                                  // this thread's first slots inside the CTA
  {
    const uint32_t wa = lane < kClWarps ? sh.warp_a[lane] : 0u, wt = lane < kClWarps ? sh.warp_b[lane] : 0u;
    at_a = __reduce_add_sync(0xffffffffu, lane < warp ? wa : 0u) + inc_a - n_a;
    at_t = __reduce_add_sync(0xffffffffu, lane < warp ? wt : 0u) + inc_t - n_t;
    const uint32_t ta = __reduce_add_sync(0xffffffffu, wa), tt = __reduce_add_sync(0xffffffffu, wt);
    if (tid == 0) { sh.n_above = ta; sh.n_tie = tt; }
  }
  sync_all();
  uint32_t sum_a;
  {
    const uint32_t ra = lane < (int)cs ? ld_cluster(map_rank(&sh.n_above, (uint32_t)lane)) : 0u;
    const uint32_t rt = lane < (int)cs ? ld_cluster(map_rank(&sh.n_tie, (uint32_t)lane)) : 0u;
    at_a += __reduce_add_sync(0xffffffffu, lane < (int)me ? ra : 0u);
    at_t += __reduce_add_sync(0xffffffffu, lane < (int)me ? rt : 0u);
    sum_a = __reduce_add_sync(0xffffffffu, ra);
  }
  int32_t* out = sel_idx + (size_t)row * pl.k_max;
  const uint32_t ties0 = map_rank(&sh.ties[0], 0u);
  [[maybe_unused]] auto take_out = [&](int pos, uint32_t key) {
    if (bg.m > -CUDART_INF_F) bg_take_out(bg, seg, pos, key_score(key), bg_lid(pl, bg, lids, pos), mass);
  };
  auto hand_over = [&](uint32_t key, int pos) {         // an item of the range, to CTA 0
    if (is_in(key, pos)) {
      if (at_t < (uint32_t)kClTies) st_cluster_v2(ties0 + 8u * at_t, key, (uint32_t)pos);
      ++at_t;
    }
  };
  auto emit = [&](uint32_t key, int pos) {
    if (is_above(key, pos)) {
      if (at_a < (uint32_t)k) out[at_a] = pos;
      ++at_a;
      if constexpr (kBg) take_out(pos, key);
    }
  };
  // the items of the range first: their barrier completes while the rest is written out
  if (listed) {
#pragma unroll 1
    for (int i = tid; i < (int)sh.n_list; i += kClThreads) hand_over(sh.list[i].x, (int)sh.list[i].y);
  } else {
    sl.for_hits(bound, hand_over);
  }
  cluster_arrive();
  if (listed) {
#pragma unroll 1
    for (int i = tid; i < (int)sh.n_list; i += kClThreads) emit(sh.list[i].x, (int)sh.list[i].y);
  } else {
    sl.for_hits(bound, emit);
  }
  __syncwarp();
  cluster_wait();                                       // CTA 0 holds all items of the range
  if (me != 0) return;
  const uint32_t need = (uint32_t)k - min((uint32_t)k, above);
  const uint32_t m_t = min(m_in, (uint32_t)kClTies);
  if (tid == 0) sh.kstar = 0u;
  __syncthreads();
  for (uint32_t i = tid; i < m_t; i += kClThreads) {
    const uint2 it = sh.ties[i];
    const uint32_t pos = it.y;
    uint32_t rank = 0u;
    for (uint32_t j = 0; j < m_t; ++j) {
      const uint2 o = sh.ties[j];
      rank += (o.x > it.x || (o.x == it.x && o.y < pos)) ? 1u : 0u;
    }
    if (rank < need) {
      if (above + rank < (uint32_t)k) out[above + rank] = (int)pos;
      if constexpr (kBg) take_out((int)pos, it.x);
      if (rank == need - 1u) sh.kstar = it.x;
    }
  }
  __syncthreads();
  if (tid == 0) {
    sel_count[row] = k;
    kth[row] = key_score(sh.kstar);
    if (sum_a != above || need == 0u || m_t < need) atomicOr(status, kStatusCountMismatch);
  }
}

constexpr size_t kClHead = (sizeof(ClShared) + 127) & ~size_t(127);
constexpr int kClSlice = (int)((kMaxDynamicSmem - kClHead) / 16 * 4);       // scores a CTA can hold

int slice_of(const Plan& pl, int cs) { return (pl.N_max + 4 * cs - 1) / (4 * cs) * 4; }
size_t smem_of(const Plan& pl, int cs) { return kClHead + (size_t)slice_of(pl, cs) * 4; }
// (two CTAs, 1 KB of system use each, in an SM's 228 KB)
bool two_per_sm(const Plan& pl, int cs) { return smem_of(pl, cs) <= 113 * 1024; }

template <bool kBg, int kPerSm>
cudaError_t launch_t(const Plan& pl, const float* scores, const int32_t* seq_lens, int32_t* sel_idx,
                     int32_t* sel_count, float* kth, int* status, const float* partials,
                     const uint16_t* lids, float* bg_mass, float* bg_max, cudaStream_t st) {
  const size_t smem = smem_of(pl, pl.sel_cluster);
  auto kernel = select_cluster_kernel<kBg, kPerSm>;
  cudaError_t e = allow_max_smem(kernel);
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(pl.rows * pl.sel_cluster));
  cfg.blockDim = dim3(kClThreads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  attr[1].id = cudaLaunchAttributeClusterDimension;
  attr[1].val.clusterDim.x = (unsigned)pl.sel_cluster;
  attr[1].val.clusterDim.y = 1;
  attr[1].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 2;
  return cudaLaunchKernelEx(&cfg, kernel, pl, scores, seq_lens, sel_idx, sel_count, kth, status,
                            partials, lids, bg_mass, bg_max);
}

}  // namespace

// Cluster size for a shape, or 0 where the sampled path is the better one.  A row is cut while all
// CTAs still run at once and a slice keeps 4096 scores or more, and as often as shared memory
// requires.  Whole decode call, 32 rows per sequence, sampled -> cluster, us:
//   slices that leave room for two CTAs per SM win with any number of rows: 16 x 8K 135 -> 92,
//   32 x 8K 225 -> 165, 32 x 4K 155 -> 136, 16 x 16K 139 -> 127, 32 x 16K 241 -> 229;
//   one CTA per SM and row, several waves: 8 x 20K 92 -> 88, 13 x 20K 123 -> 123; longer slices up to two
//   waves, the last at least half full: 8 x 32K 116 -> 111, 8 x 45K 144 -> 141, but 5 x 32K (1.1 waves)
//   85 -> 89, 6 x 45K (1.3) 114 -> 122, 12 x 45K (2.6) 189 -> 197;
//   several CTAs per row while all run at once: 1 x 92K of 64 heads 91 -> 81, but 3 x 92K 112 -> 124,
//   4 x 92K 136 -> 144.  Of clusters of eight a GPC holds two at most, and 16 rows do not run at once: a row
//   is then cut in four where that is enough (16 rows of 30K 53 -> 45, of 100K 56 -> 45 against eight), in
//   eight while the slices are short and the rows few (16 rows of 200K, sampled -> cluster: 73 -> 66; of
//   256K 117 -> 117, and the top-k alone 28 -> 33; 32 rows of 190K 174 -> 187).
// And only while most of what is selected is listed: passes over the whole slice for every step cost more
// than the sampled path's.  1 x 128K (4 CTAs a row): budget 4 % 0.90 times the sampled path's time, 6 %
// 1.02, 8 % 1.10; 1 x 64K: 12.5 % 0.91, 20 % 1.01; 8 x 32K: 4 % 1.00, 8 % 1.12.  Short slices bear it:
// 1 x 32K: 30 % 1.00, 40 % 0.98; 16 x 8K: 30 % 0.80, 40 % 0.85.  With half of the row or more selected the
// first bound is no bound: 1 x 8K: 40 % 0.76, 50 % 1.12, 70 % 1.38.
constexpr int kClListed = 2048;          // selected scores per CTA that still leave room in its list
constexpr int kClShort = 8192;           // a slice that may be passed over instead
constexpr int kClFill = 24576;           // longest slice whose last wave may be nearly empty
constexpr int kClTurns = 28672;          // longest slice of clusters of eight that take turns
constexpr uint32_t kClMaxPpm = 400000u;
void plan_select_cluster(Plan* pl) {
  pl->sel_cluster = 0;
  if (pl->rescore) return;                 // the re-score reads the sampled path's candidate lists
  int cs = 1;
  const int most = 5 * pl->rows * kClMax <= 4 * pl->num_sms ? kClMax : kClMax / 2;
  while (cs < most && pl->rows * cs * 2 <= pl->num_sms && pl->N_max / cs > 4096) cs *= 2;
  while (cs < kClMax && slice_of(*pl, cs) > kClSlice) cs *= 2;
  if (slice_of(*pl, cs) > (cs > most ? kClTurns : kClSlice)) return;
  if (cs > most && pl->rows * cs > pl->num_sms) return;
  const int waves = (pl->rows * cs + pl->num_sms - 1) / pl->num_sms;
  if (cs > 1 && waves > 1) return;
  if (cs == 1 && waves > 1 && !two_per_sm(*pl, 1)) {
    if (waves > 3) return;
    if (pl->N_max > kClFill && (waves > 2 || 4 * pl->rows < 3 * waves * pl->num_sms)) return;
  }
  if (pl->ppm > kClMaxPpm) return;
  const long long k = ((long long)pl->N_max * pl->ppm + 999999LL) / 1000000LL;
  if (k > (long long)kClListed * cs && slice_of(*pl, cs) > kClShort) return;
  pl->sel_cluster = cs;
}

// (one CTA per SM leaves the compiler 80 registers instead of 64, worth 1 us at 32 rows)
cudaError_t launch_select_cluster(const Plan& pl, const float* scores, const int32_t* seq_lens,
                                  int32_t* sel_idx, int32_t* sel_count, float* kth, int* status,
                                  cudaStream_t st) {
  const bool two = two_per_sm(pl, pl.sel_cluster) && pl.rows * pl.sel_cluster > pl.num_sms;
  return (two ? launch_t<false, 2> : launch_t<false, 1>)(pl, scores, seq_lens, sel_idx, sel_count, kth, status,
                                                         nullptr, nullptr, nullptr, nullptr, st);
}

cudaError_t launch_select_cluster_bg(const Plan& pl, const float* scores, const int32_t* seq_lens,
                                     int32_t* sel_idx, int32_t* sel_count, float* kth, int* status,
                                     const float* partials, const uint16_t* lids, float* bg_mass,
                                     float* bg_max, cudaStream_t st) {
  const bool two = two_per_sm(pl, pl.sel_cluster) && pl.rows * pl.sel_cluster > pl.num_sms;
  return (two ? launch_t<true, 2> : launch_t<true, 1>)(pl, scores, seq_lens, sel_idx, sel_count, kth, status,
                                                       partials, lids, bg_mass, bg_max, st);
}

}  // namespace pqhsa
