// Batched index build (Sec. 3.3, first paragraph; App. C, "Index build"): the k-means problems
// of ALL (sequence, KV head) units are trained together, one launch per step for all of them --
// one coarse problem per unit over its key directions, then one product-quantisation problem
// per (unit, subspace) over the residuals -- instead of thousands of small per-head launches.
// Direction-norm residual IVF-PQ of Sec. 3.1: r_i = |k_i| in fp32 from the cached key,
// u_i = k_i / r_i (0 for a zero key), Lloyd iterations with squared Euclidean distance, a
// centroid is the arithmetic mean of its members (not re-normalised: Eq. 2 uses c_j as is), an
// empty cluster is re-seeded with the point farthest from its centre, ties go to the lower index.
// The random draws of the method (which points seed the centroids and the codewords) are inputs.
//
//   build_prepare_kernel     norms and unit directions U (fp32, workspace) from the paged cache
//   build_seed_kernel        centroids <- U rows at the given positions
//   build_split_kernel       centroids as split fp16 tensor-core tiles (tc.cuh), once per iteration
//   build_assign_kernel      nearest centroid of 256 tokens per CTA on the tensor cores; what comes within
//                            the rounding of the nearest is compared in fp32 (tc.cuh): the lists, and
//                            with them everything that follows, are those of an fp32 search
//   build_hist / _offsets / _scatter   the tokens of a unit grouped by list (counting sort)
//   build_dir_sums_kernel    per-list sums of the member directions (64-bit fixed point, so the
//                            result does not depend on the order of the atomics): a warp sums the
//                            rows of consecutive grouped tokens and adds once per list it meets
//   build_update_centroids_kernel   takes the mean; build_distance_kernel, build_reseed_kernel: empty
//                            lists take the farthest points (rare)
//   build_residual_kernel    U <- U - c_a, in place
//   build_pq_* kernels       the same steps for the residual sub-vectors, also on the tensor cores
//   build_value_* kernels    list value means and member counts from the paged values, in list order
#include "attn_common.cuh"
#include "common.cuh"
#include "tc.cuh"

namespace pqhsa {

namespace {

constexpr int kD = kHeadDim;            // 128
constexpr int kPrepThreads = 256;

// Sums of member vectors are taken in 64-bit fixed point with integer atomics: integer
// addition is associative, so the centroids (and with them the whole index) do not depend on
// the order in which the atomics land -- two builds of the same input are bit-identical.
// Directions and residuals are below 2 in magnitude (scale 2^40, 131,072 members stay below
// 2^58); values are cache-dtype numbers (scale 2^24, exact for bf16 / fp16 inputs up to 2^15).
constexpr float kFixDir = 1099511627776.0f;      // 2^40
constexpr float kFixVal = 16777216.0f;           // 2^24
__device__ __forceinline__ float fix_mean(long long s, int count, float scale) {
  return (float)(((double)s / (double)scale) / (double)count);
}

__device__ __forceinline__ long long kv_row(const Plan& pl, const int32_t* __restrict__ bt, int pos,
                                            int kv, long long sp, long long st, long long sh) {
  const int page = __ldg(bt + pos / pl.page_size);
  return (long long)page * sp + (long long)(pos % pl.page_size) * st + (long long)kv * sh;
}

// ---- norms and directions: a warp per token, a lane holds 4 of the 128 dims
template <typename T>
__global__ void __launch_bounds__(kPrepThreads)
build_prepare_kernel(Plan pl, const T* __restrict__ kc, long long sp, long long st, long long sh,
                     const int32_t* __restrict__ block_table, const int32_t* __restrict__ seq_lens,
                     float* __restrict__ U, float* __restrict__ key_norms) {
  const int kv = blockIdx.y, b = blockIdx.z;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int n = clamp_len(seq_lens[b], pl.N_max);
  const size_t ukv = (size_t)b * pl.Hkv + kv;
  const int32_t* bt = block_table + (size_t)b * pl.max_pages;
  for (int i = blockIdx.x * (kPrepThreads / 32) + warp; i < n; i += gridDim.x * (kPrepThreads / 32)) {
    const T* row = kc + kv_row(pl, bt, i, kv, sp, st, sh);
    float x[4];
    load4<T>(row + 4 * lane, x);
    const float ss = warp_sum(x[0] * x[0] + x[1] * x[1] + x[2] * x[2] + x[3] * x[3]);
    const float r = sqrtf(ss);
    const float inv = r > 0.f ? 1.f / r : 0.f;
    *reinterpret_cast<float4*>(U + (ukv * pl.N_max + i) * kD + 4 * lane) =
        make_float4(x[0] * inv, x[1] * inv, x[2] * inv, x[3] * inv);
    if (lane == 0) key_norms[ukv * pl.N_max + i] = r;
  }
}

// ---- seeds: row j of `dst` [units][n_rows][kD] <- U row at seed_pos[unit][j] (zero if < 0)
__global__ void build_seed_kernel(Plan pl, const float* __restrict__ U,
                                  const int32_t* __restrict__ seed_pos, int n_rows,
                                  float* __restrict__ dst) {
  const size_t unit = blockIdx.y;
  const int j = blockIdx.x * (blockDim.x / 32) + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  if (j >= n_rows) return;
  const int pos = seed_pos[unit * n_rows + j];
  float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
  if (pos >= 0 && pos < pl.N_max) v = *reinterpret_cast<const float4*>(U + (unit * pl.N_max + pos) * kD + 4 * lane);
  *reinterpret_cast<float4*>(dst + (unit * n_rows + j) * kD + 4 * lane) = v;
}

// ---- centroids as tensor-core tiles: 128 rows in the layout of the coarse search, the factor -2 and
// |c|^2 included; rows past n_list are farther than any centroid
constexpr int kAsgTok = 256, kAsgCen = 128, kAsgThreads = 320;
constexpr int kCenTileBytes = kCoarseChunks * kAsgCen * 16;       // 69632
constexpr int kTokTileBytes = kCoarseChunks * 128 * 16;
constexpr int kAsgSmemBytes = 2 * kTokTileBytes + kCenTileBytes;
// A centroid tile arrives in pieces of 4 chunks (8 KB), in the order in which the MMAs want them: the lo
// half (pieces 0-3), the hi half (4-7), the |c|^2 chunks (8).
constexpr int kAsgPieces = 9;
__device__ __forceinline__ constexpr uint32_t piece_chunk(int p) { return p < 4 ? 16 + 4 * p : p < 8 ? 4 * (p - 4) : 32; }

// 8 rows of 128 fp32 into a tile: lane l holds row l & 7 and the chunks (l >> 3) + 4 i, so that loads
// take whole 128-byte lines and stores have no conflicts.  split_rows returns |row|^2 (all lanes of the
// row).
// a whole 32-byte sector in one instruction (two 16-byte loads fetch it twice)
__device__ __forceinline__ void load_sector(const float* p, float (&v)[8]) {
  asm volatile("ld.global.v8.f32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
               : "=f"(v[0]), "=f"(v[1]), "=f"(v[2]), "=f"(v[3]), "=f"(v[4]), "=f"(v[5]), "=f"(v[6]), "=f"(v[7])
               : "l"(p) : "memory");
}
struct RowPart {
  float v[4][8];
};
// (kSectors: rows on 32-byte boundaries, the workspace's; the caller's centroids are on 16)
template <bool kSectors>
__device__ __forceinline__ RowPart load_rows(const float* __restrict__ src, bool real, int lane) {
  RowPart p;
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const float* at = src + 8 * ((lane >> 3) + 4 * i);
    if (real && kSectors) {
      load_sector(at, p.v[i]);
    } else if (real) {
      *reinterpret_cast<float4*>(p.v[i]) = __ldcg(reinterpret_cast<const float4*>(at));
      *reinterpret_cast<float4*>(p.v[i] + 4) = __ldcg(reinterpret_cast<const float4*>(at) + 1);
    } else {
#pragma unroll
      for (int t = 0; t < 8; ++t) p.v[i][t] = 0.f;
    }
  }
  return p;
}
__device__ __forceinline__ float split_rows(const RowPart& p, float scale, unsigned char* dst, int rows, int r, int lane) {
  const int c0 = lane >> 3;
  float n2 = 0.f;
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const float (&v)[8] = p.v[i];
    uint4 hi, lo;
    split_chunk(v, scale, hi, lo);
#pragma unroll
    for (int t = 0; t < 8; ++t) n2 = fmaf(v[t], v[t], n2);
    *reinterpret_cast<uint4*>(dst + ((c0 + 4 * i) * rows + r) * 16) = hi;
    *reinterpret_cast<uint4*>(dst + ((16 + c0 + 4 * i) * rows + r) * 16) = lo;
  }
  n2 += __shfl_xor_sync(0xffffffffu, n2, 8);
  n2 += __shfl_xor_sync(0xffffffffu, n2, 16);
  return n2;
}

__global__ void __launch_bounds__(4 * kAsgCen)
build_split_kernel(Plan pl, const float* __restrict__ centroids, unsigned char* __restrict__ images) {
  const size_t unit = blockIdx.y;
  const int lane = threadIdx.x & 31, r = (threadIdx.x >> 5) * 8 + (lane & 7);
  const int j = blockIdx.x * kAsgCen + r;
  unsigned char* dst = images + (unit * gridDim.x + blockIdx.x) * (size_t)kCenTileBytes;
  const bool real = j < pl.n_list;
  const float n2 = split_rows(load_rows<false>(centroids + (unit * pl.n_list + (real ? j : 0)) * kD, real, lane),
                              -2.f * kTcScale, dst, kAsgCen, r, lane);
  if (lane < 8) *reinterpret_cast<uint4*>(dst + (32 * kAsgCen + r) * 16) = coarse_ext_centre(n2, real);
  else if (lane < 16) *reinterpret_cast<uint4*>(dst + (33 * kAsgCen + r) * 16) = make_uint4(0u, 0u, 0u, 0u);
}

// ---- nearest centroid.  CTA: 256 tokens of one unit as two 128-row tiles that stay in shared memory;
// one centroid tile is resident and is replaced piece by piece: a piece is refilled as soon as its last
// MMA is done, two thirds of a tile's time before the next tile wants it, so that 128 centroids per MMA
// (64 clocks; 64 of them would cost 48) need no second stage.  Warp 8 issues the MMAs, warp 9 the
// copies; warpgroup w reads the accumulators of token tile w (128 columns, double buffered).
// What bounds it: the MMAs.  With all SMs at work they run at 108 clocks, 1.36 of the 1.63 PFLOP/s that a
// cuBLAS GEMM reaches (64 clocks with few SMs busy): 5.4 of the 6.2 thousand clocks per tile; behind them
// the search for the two nearest (2.4 to 3.6 thousand, overlapped) and the token tile at the start (8.1
// thousand, 1 CTA per SM: nothing overlaps it).  1 M tokens x 1024 lists: 1231 us with 64 centroids per
// tile, two stages and an index beside every value, 1000 us so, 940 us with whole sectors loaded, 970 us
// with what fp32 decides.
__global__ void __launch_bounds__(kAsgThreads, 1)
build_assign_kernel(Plan pl, const float* __restrict__ U, const unsigned char* __restrict__ images,
                    const float* __restrict__ centroids, const int32_t* __restrict__ seq_lens,
                    uint16_t* __restrict__ list_ids, float* __restrict__ key_norms) {
  extern __shared__ __align__(128) unsigned char s_asg[];
  unsigned char* s_tok = s_asg;                             // two token tiles
  unsigned char* s_cen = s_asg + 2 * kTokTileBytes;         // the centroid tile
  __shared__ float s_x2[kAsgTok];
  __shared__ uint8_t s_crowd[kAsgTok];                      // tokens that fp32 searches for
  __shared__ int s_n_crowd, s_late;
  __shared__ Found s_found[8][kCrowd];
  __shared__ uint32_t s_tmem;
  __shared__ __align__(8) uint64_t s_full[kAsgPieces], s_used[kAsgPieces], s_done[2], s_free[2], s_end;
  const int kv = blockIdx.y, b = blockIdx.z;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int t0 = blockIdx.x * kAsgTok;
  const size_t ukv = (size_t)b * pl.Hkv + kv;
  // two rounds of rows in flight before anything is waited for (rows past the sequence are not used)
  RowPart part[2];
  auto row_of = [&](int q) { return q * 64 + warp * 8 + (lane & 7); };
  auto load = [&](int q) {
    const int r = row_of(q);
    return load_rows<true>(U + (ukv * pl.N_max + t0 + r) * kD, t0 + r < pl.N_max, lane);
  };
  if (warp < 8) {
    part[0] = load(0);
    part[1] = load(1);
  }
  const int n = clamp_len(seq_lens[b], pl.N_max);
  if (t0 >= n) return;
  const int n_tiles = (pl.n_list + kAsgCen - 1) / kAsgCen;
  const unsigned char* img = images + ukv * (size_t)n_tiles * kCenTileBytes;
  if (tid == 0) { s_n_crowd = 0; s_late = 0; }
  if (warp == 8) tmem_alloc(&s_tmem, 512);
  if (warp == 9) {
    if (lane < kAsgPieces) { mbar_init(&s_full[lane], 1); mbar_init(&s_used[lane], 1); }
    if (lane < 2) { mbar_init(&s_done[lane], 1); mbar_init(&s_free[lane], 8); }
    if (lane == 2) mbar_init(&s_end, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  auto copy = [&](int i, int p) {
    const uint32_t bytes = (p < 8 ? 4u : 2u) * kAsgCen * 16u, at = piece_chunk(p) * kAsgCen * 16u;
    mbar_expect_tx(&s_full[p], bytes);
    bulk_g2s(s_cen + at, img + (size_t)i * kCenTileBytes + at, bytes, &s_full[p]);
  };
  if (warp == 9) {
    __syncwarp();
    if (lane == 0)
      for (int p = 0; p < kAsgPieces; ++p) copy(0, p);
  }
  // the token tiles
  if (warp < 8) {
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int r = row_of(q);
      unsigned char* dst = s_tok + (r >> 7) * kTokTileBytes;
      if (t0 + r >= n) part[q & 1] = load_rows<true>(U, false, lane);         // zeros
      const float x2 = split_rows(part[q & 1], kTcScale, dst, 128, r & 127, lane);
      if (q < 2) part[q & 1] = load(q + 2);
      if (lane < 8) {
        s_x2[r] = x2;
        *reinterpret_cast<uint4*>(dst + (32 * 128 + (r & 127)) * 16) = coarse_ext_row();
      } else if (lane < 16) {
        *reinterpret_cast<uint4*>(dst + (33 * 128 + (r & 127)) * 16) = make_uint4(0u, 0u, 0u, 0u);
      }
    }
    tc_fence_smem();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = s_tmem;
  // A wait that runs out (none does while the GPU works) ends its role's loop, so that nothing in use is
  // overwritten, and is told through s_late: the lists of the CTA's tokens are then not to be trusted.
  bool late = false;
  auto ready = [&](uint64_t* bar, uint32_t parity) {
    if (!late) late = !tc_wait(bar, parity);
    return !late;
  };
  if (warp == 9) {
    if (lane == 0) {
      uint32_t last[kAsgPieces] = {};                       // parity of each piece's last copy
      for (int i = 1; i < n_tiles && !late; ++i) {
#pragma unroll
        for (int p = 0; p < kAsgPieces; ++p) {
          if (!ready(&s_used[p], (uint32_t)(i - 1) & 1u)) break;
          copy(i, p);
          last[p] = (uint32_t)i & 1u;
        }
      }
#pragma unroll
      for (int p = 0; p < kAsgPieces; ++p)                  // (no copy outlives the CTA)
        if (!tc_wait(&s_full[p], last[p])) late = true;
      if (late) s_late = 1;
    }
    __syncwarp();
  } else if (warp == 8) {
    if (lane == 0) {
      const uint64_t a0 = tc_desc(smem_u32(s_tok), 128u * 16u), a1 = tc_desc(smem_u32(s_tok + kTokTileBytes), 128u * 16u);
      const uint64_t bd = tc_desc(smem_u32(s_cen), kAsgCen * 16u);
      for (int i = 0; i < n_tiles; ++i) {
        const uint32_t st = i & 1, ph = st;
        const uint32_t idesc = tc_idesc(pl.n_list - i * kAsgCen <= 64 ? 64u : 128u);
        const uint32_t d0 = tmem + st * 256u, d1 = d0 + 128u;
        if (i >= 2 && !ready(&s_free[st], ((uint32_t)(i >> 1) & 1u) ^ 1u)) break;   // tile i - 2 has been read
        // one piece against 4 chunks of the token tiles (offsets in 16-byte units; all constants)
        auto steps = [&](uint32_t a_chunk, uint32_t b_chunk, bool first) {
#pragma unroll
          for (uint32_t k = 0; k < 4; k += 2) {
            tc_mma(d0, a0 + (a_chunk + k) * 128u, bd + (b_chunk + k) * kAsgCen, idesc, !first || k != 0);
            tc_mma(d1, a1 + (a_chunk + k) * 128u, bd + (b_chunk + k) * kAsgCen, idesc, !first || k != 0);
          }
        };
        // the cross terms first: they are 2^-11 of the rest, so that only nine accumulations round at
        // full magnitude
#pragma unroll
        for (int p = 0; p < 4; ++p) {
          if (!ready(&s_full[p], ph)) break;
          tc_fence_after();
          steps(4 * p, piece_chunk(p), p == 0);
          tc_commit(&s_used[p]);
        }
#pragma unroll
        for (int p = 4; p < 8; ++p) {
          if (!ready(&s_full[p], ph)) break;
          tc_fence_after();
          steps(16 + 4 * (p - 4), piece_chunk(p), false);
        }
        if (late) break;
#pragma unroll
        for (int p = 4; p < 8; ++p) {
          steps(4 * (p - 4), piece_chunk(p), false);
          tc_commit(&s_used[p]);
        }
        if (!ready(&s_full[8], ph)) break;
        tc_fence_after();
        tc_mma(d0, a0 + 32u * 128u, bd + 32u * kAsgCen, idesc, true);
        tc_mma(d1, a1 + 32u * 128u, bd + 32u * kAsgCen, idesc, true);
        tc_commit(&s_used[8]);
        tc_commit(&s_done[st]);
      }
      tc_commit(&s_end);                                    // (nor does an MMA)
      if (!tc_wait(&s_end, 0u)) late = true;
      if (late) s_late = 1;
    }
    __syncwarp();
  } else {
    const int wg = warp >> 2;
    const uint32_t lanes = (uint32_t)((warp & 3) * 32) << 16;
    const int r = wg * 128 + (warp & 3) * 32 + lane;
    const TieLimit lim(s_x2[r]);
    Nearest2 nn;
    nn.clear();
    for (int i = 0; i < n_tiles; ++i) {
      const uint32_t st = i & 1;
      if (__any_sync(0xffffffffu, !ready(&s_done[st], (uint32_t)(i >> 1) & 1u))) { s_late = 1; break; }
      tc_fence_after();
      const int n_cols = min(pl.n_list - i * kAsgCen, kAsgCen);
#pragma unroll 1
      for (int c = 0; c < n_cols; c += 32) {
        float acc[32];
        tmem_ld32(tmem + st * 256u + wg * 128u + c + lanes, acc);
        nn.take(acc, i * (kAsgCen / 32) + (c >> 5), lim);
      }
      tc_fence_before();
      if (lane == 0) asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(&s_free[st])) : "memory");
      __syncwarp();
    }
    // between the centroids of one or two blocks fp32 decides (a few tokens in a hundred), a warp per token
    int near = min(nn.near(), pl.n_list - 1);
    const bool real = t0 + r < n, crowd = real && nn.crowded();
    const int block1 = nn.second_near(lim) ? nn.second_at : nn.best_at;
    unsigned ties = __ballot_sync(0xffffffffu, real && !crowd && nn.tie(lim));
    while (ties) {
      const int src = __ffs(ties) - 1;
      ties &= ties - 1u;
      const int at = nearest_of_blocks<true>(U + (ukv * pl.N_max + t0 + r - lane + src) * kD, centroids + ukv * pl.n_list * (size_t)kD,
                                             pl.n_list, __shfl_sync(0xffffffffu, nn.best_at, src), __shfl_sync(0xffffffffu, block1, src));
      if (lane == src) near = at;
    }
    if (crowd) s_crowd[atomicAdd(&s_n_crowd, 1)] = (uint8_t)r;
    if (real) list_ids[ukv * pl.N_max + t0 + r] = (uint16_t)near;
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 8) { tc_fence_after(); tmem_free(tmem, 512); }
  if (s_late != 0 && t0 + tid < min(n, t0 + kAsgTok)) key_norms[ukv * pl.N_max + t0 + tid] = CUDART_NAN_F;
  // between more of them over all centroids, by eight warps
  const int n_crowd = s_n_crowd;
  const int n_search = n_crowd > kCrowd ? kCrowd : 1;       // for together
#pragma unroll 1
  for (int c = 0; c < n_crowd; c += n_search) {
    const float* rows = U + (ukv * pl.N_max + t0) * kD;
    const float* cen = centroids + ukv * pl.n_list * (size_t)kD;
    if (warp < 8) {
      if (n_search == 1) nearest_of_all<true, 1>(rows, kD, s_crowd, c, n_crowd, cen, pl.n_list, tid, 256, ~0u, s_found[warp]);
      else nearest_of_all<true, kCrowd>(rows, kD, s_crowd, c, n_crowd, cen, pl.n_list, tid, 256, ~0u, s_found[warp]);
    }
    __syncthreads();
    if (tid < n_search && c + tid < n_crowd) {
      Found f = s_found[0][tid];
      for (int w = 1; w < 8; ++w) nearer(f.d, f.at, s_found[w][tid].d, s_found[w][tid].at);
      list_ids[ukv * pl.N_max + t0 + s_crowd[c + tid]] = (uint16_t)f.at;
    }
    __syncthreads();
  }
}

// Squared distance of every token to its list's centroid, in fp32, one chain per sum; only for units with
// an empty list (they take the farthest points), infinite where it is not a number
__global__ void __launch_bounds__(kPrepThreads)
build_distance_kernel(Plan pl, const float* __restrict__ U, const float* __restrict__ centroids,
                      const int32_t* __restrict__ seq_lens, const uint16_t* __restrict__ list_ids,
                      const int32_t* __restrict__ n_empty, float* __restrict__ dmin) {
  const int kv = blockIdx.y, b = blockIdx.z;
  const int n = clamp_len(seq_lens[b], pl.N_max);
  const size_t ukv = (size_t)b * pl.Hkv + kv;
  if (n_empty[ukv] == 0 || n <= pl.n_list) return;
  for (int i = blockIdx.x * kPrepThreads + threadIdx.x; i < n; i += gridDim.x * kPrepThreads) {
    const size_t at = ukv * pl.N_max + i;
    const float d = distance_fp32<true>(U + at * kD, centroids + (ukv * pl.n_list + min((int)list_ids[at], pl.n_list - 1)) * (size_t)kD);
    dmin[at] = d == d ? d : CUDART_INF_F;
  }
}

// ---- tokens grouped by list.  hist: members per list; offsets: exclusive prefix (and a running
// copy); scatter: every token to its list's next slot (the order inside a list does not matter: all
// sums over it are integers).  Only tokens of [lo, hi) take part: the whole sequence for the
// centroids, the indexed region for the value means.
constexpr int kSortThreads = 512;
constexpr int kSortChunk = 4096;         // tokens per CTA
template <bool kRegion> __device__ __forceinline__ Region sort_range(const Plan& pl, int n, int b) {
  if (kRegion) return region_of(pl, n, b);
  return Region{0, n};
}

template <bool kRegion>
__global__ void __launch_bounds__(kSortThreads)
build_hist_kernel(Plan pl, const uint16_t* __restrict__ list_ids, const int32_t* __restrict__ seq_lens,
                  int32_t* __restrict__ counts) {
  extern __shared__ int s_cnt[];                            // [n_list]
  const int kv = blockIdx.y, b = blockIdx.z;
  const int n = clamp_len(seq_lens[b], pl.N_max);
  const Region rg = sort_range<kRegion>(pl, n, b);
  const int lo = rg.r_begin + blockIdx.x * kSortChunk, hi = min(rg.r_end, lo + kSortChunk);
  if (lo >= hi) return;
  const size_t ukv = (size_t)b * pl.Hkv + kv;
  for (int j = threadIdx.x; j < pl.n_list; j += kSortThreads) s_cnt[j] = 0;
  __syncthreads();
  for (int i = lo + threadIdx.x; i < hi; i += kSortThreads)
    atomicAdd(&s_cnt[min((int)list_ids[ukv * pl.N_max + i], pl.n_list - 1)], 1);
  __syncthreads();
  for (int j = threadIdx.x; j < pl.n_list; j += kSortThreads)
    if (s_cnt[j]) atomicAdd(&counts[ukv * pl.n_list + j], s_cnt[j]);
}

__global__ void __launch_bounds__(1024)
build_offsets_kernel(Plan pl, const int32_t* __restrict__ counts, int32_t* __restrict__ cursor,
                     int32_t* __restrict__ n_empty) {
  __shared__ int s_warp[32];
  const size_t unit = blockIdx.x;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  int v[4], local = 0, empty = 0;                           // n_list <= 4096: 4 lists per thread
#pragma unroll
  for (int u = 0; u < 4; ++u) {
    const int j = 4 * tid + u;
    v[u] = j < pl.n_list ? counts[unit * pl.n_list + j] : 0;
    local += v[u];
    empty += j < pl.n_list && v[u] == 0 ? 1 : 0;
  }
  if (empty != 0 && n_empty != nullptr) atomicAdd(&n_empty[unit], empty);
  int inc = local;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int u = __shfl_up_sync(0xffffffffu, inc, o);
    if (lane >= o) inc += u;
  }
  if (lane == 31) s_warp[warp] = inc;
  __syncthreads();
  int run = inc - local;
  for (int w = 0; w < warp; ++w) run += s_warp[w];
#pragma unroll
  for (int u = 0; u < 4; ++u) {
    const int j = 4 * tid + u;
    if (j < pl.n_list) cursor[unit * pl.n_list + j] = run;
    run += v[u];
  }
}

template <bool kRegion>
__global__ void __launch_bounds__(kSortThreads)
build_scatter_kernel(Plan pl, const uint16_t* __restrict__ list_ids, const int32_t* __restrict__ seq_lens,
                     int32_t* __restrict__ cursor, int32_t* __restrict__ order) {
  extern __shared__ int s_cnt[];                            // [n_list] members here, then next slot
  const int kv = blockIdx.y, b = blockIdx.z;
  const int n = clamp_len(seq_lens[b], pl.N_max);
  const Region rg = sort_range<kRegion>(pl, n, b);
  const int lo = rg.r_begin + blockIdx.x * kSortChunk, hi = min(rg.r_end, lo + kSortChunk);
  if (lo >= hi) return;
  const size_t ukv = (size_t)b * pl.Hkv + kv;
  constexpr int kPer = kSortChunk / kSortThreads;
  int lid[kPer], rank[kPer];
  for (int j = threadIdx.x; j < pl.n_list; j += kSortThreads) s_cnt[j] = 0;
  __syncthreads();
#pragma unroll
  for (int u = 0; u < kPer; ++u) {
    const int i = lo + u * kSortThreads + threadIdx.x;
    lid[u] = i < hi ? min((int)list_ids[ukv * pl.N_max + i], pl.n_list - 1) : -1;
    if (lid[u] >= 0) rank[u] = atomicAdd(&s_cnt[lid[u]], 1);
  }
  __syncthreads();
  for (int j = threadIdx.x; j < pl.n_list; j += kSortThreads)
    if (s_cnt[j]) s_cnt[j] = atomicAdd(&cursor[ukv * pl.n_list + j], s_cnt[j]);
  __syncthreads();
#pragma unroll
  for (int u = 0; u < kPer; ++u)
    if (lid[u] >= 0) order[ukv * pl.N_max + s_cnt[lid[u]] + rank[u]] = lo + u * kSortThreads + threadIdx.x;
}

// ---- sums over grouped tokens: a warp takes kRun consecutive entries of `order`, a lane 4 dims; the
// sum goes out when the list changes.  row(i, x) reads token i's 4 dims.
constexpr int kRun = 64, kRunBatch = 8;
// (place: a token's row; asked once per 32 entries, a lane each, and handed round, since the page's
// division and table look-up for every row kept the warps busier than the rows.  1 M rows: values
// 262 -> 156 us, directions 129 -> 115 us)
template <class Place, class Row>
__device__ __forceinline__ void run_sums(const Plan& pl, const uint16_t* __restrict__ lids_u,
                                         const int32_t* __restrict__ order_u, int first, int last,
                                         float scale, long long* __restrict__ sums_u, Place place, Row row) {
  const int lane = threadIdx.x & 31;
  long long acc[4] = {0, 0, 0, 0};
  int cur = -1;
  auto flush = [&]() {
    if (cur < 0) return;
    long long* dst = sums_u + (size_t)cur * kD + 4 * lane;
#pragma unroll
    for (int t = 0; t < 4; ++t) {
      if (acc[t]) atomicAdd(reinterpret_cast<unsigned long long*>(dst + t), (unsigned long long)acc[t]);
      acc[t] = 0;
    }
  };
  for (int base = first; base < last; base += 32) {
    // token and list of 32 entries at once, one per lane
    const int mine = base + lane < last ? order_u[base + lane] : -1;
    const int my_list = mine >= 0 ? min((int)lids_u[mine], pl.n_list - 1) : -1;
    const long long my_place = mine >= 0 ? place(mine) : 0ll;
    const int cnt = min(32, last - base);
    for (int e0 = 0; e0 < cnt; e0 += kRunBatch) {
      float x[kRunBatch][4];
#pragma unroll
      for (int u = 0; u < kRunBatch; ++u) {
        const long long at = __shfl_sync(0xffffffffu, my_place, e0 + u);
        if (e0 + u < cnt) row(at, x[u]);
      }
#pragma unroll
      for (int u = 0; u < kRunBatch; ++u) {
        const int j = __shfl_sync(0xffffffffu, my_list, e0 + u);
        if (j < 0) continue;                               // (warp-uniform)
        if (j != cur) { flush(); cur = j; }
#pragma unroll
        for (int t = 0; t < 4; ++t) acc[t] += __float2ll_rn(x[u][t] * scale);
      }
    }
  }
  flush();
}

__global__ void __launch_bounds__(kPrepThreads)
build_dir_sums_kernel(Plan pl, const float* __restrict__ U, const uint16_t* __restrict__ list_ids,
                      const int32_t* __restrict__ order, const int32_t* __restrict__ seq_lens,
                      long long* __restrict__ sums) {
  const int kv = blockIdx.y, b = blockIdx.z;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int n = clamp_len(seq_lens[b], pl.N_max);
  const size_t ukv = (size_t)b * pl.Hkv + kv;
  const int first = (blockIdx.x * (kPrepThreads / 32) + warp) * kRun, last = min(n, first + kRun);
  if (first >= n) return;
  const float* Ub = U + ukv * pl.N_max * (size_t)kD + 4 * lane;
  run_sums(pl, list_ids + ukv * pl.N_max, order + ukv * pl.N_max, first, last, kFixDir,
           sums + ukv * pl.n_list * (size_t)kD, [&](int i) { return (long long)i * kD; },
           [&](long long at, float (&x)[4]) {
             *reinterpret_cast<float4*>(x) = __ldcg(reinterpret_cast<const float4*>(Ub + at));
           });
}

// c_j <- mean of its members; an empty list keeps its centre; sums are cleared
__global__ void build_update_centroids_kernel(Plan pl, long long* __restrict__ sums,
                                              const int32_t* __restrict__ counts,
                                              float* __restrict__ centroids) {
  const size_t unit = blockIdx.y;
  const int j = blockIdx.x * (blockDim.x / 32) + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  if (j >= pl.n_list) return;
  const size_t at = (unit * pl.n_list + j) * kD + 4 * lane;
  const int c = counts[unit * pl.n_list + j];
  if (c > 0) {
    *reinterpret_cast<float4*>(centroids + at) =
        make_float4(fix_mean(sums[at], c, kFixDir), fix_mean(sums[at + 1], c, kFixDir),
                    fix_mean(sums[at + 2], c, kFixDir), fix_mean(sums[at + 3], c, kFixDir));
  }
#pragma unroll
  for (int t = 0; t < 4; ++t) sums[at + t] = 0;
}

// Empty lists take the farthest points: the e-th empty list (in index order) gets the point
// with the e-th largest distance to its centre (ties: lower position).  One CTA per unit;
// rare, so a plain repeated arg-max over the unit's distances; at most kMaxReseed lists per call.
constexpr int kMaxReseed = 64;
__global__ void __launch_bounds__(1024)
build_reseed_kernel(Plan pl, const float* __restrict__ U, float* __restrict__ dmin,
                    const int32_t* __restrict__ counts, const int32_t* __restrict__ seq_lens,
                    int32_t* __restrict__ n_empty, float* __restrict__ centroids) {
  __shared__ float s_d[32];
  __shared__ int s_i[32];
  __shared__ int s_pick;
  const int unit = blockIdx.x, b = unit / pl.Hkv, tid = threadIdx.x;
  const int n = clamp_len(seq_lens[b], pl.N_max);
  const int ne = n_empty[unit];
  if (ne == 0 || n <= pl.n_list) { if (tid == 0) n_empty[unit] = 0; return; }
  float* d = dmin + (size_t)unit * pl.N_max;
  int j = 0;
  for (int e = 0; e < min(ne, kMaxReseed); ++e) {
    while (j < pl.n_list && counts[(size_t)unit * pl.n_list + j] > 0) ++j;       // uniform
    if (j >= pl.n_list) break;
    float bd = -CUDART_INF_F;
    int bi = 0x7fffffff;
    for (int i = tid; i < n; i += blockDim.x) {
      const float v = d[i];
      if (v > bd || (v == bd && i < bi)) { bd = v; bi = i; }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      const float od = __shfl_xor_sync(0xffffffffu, bd, o);
      const int oi = __shfl_xor_sync(0xffffffffu, bi, o);
      if (od > bd || (od == bd && oi < bi)) { bd = od; bi = oi; }
    }
    if ((tid & 31) == 0) { s_d[tid >> 5] = bd; s_i[tid >> 5] = bi; }
    __syncthreads();
    if (tid < 32) {
      bd = tid < (int)(blockDim.x >> 5) ? s_d[tid] : -CUDART_INF_F;
      bi = tid < (int)(blockDim.x >> 5) ? s_i[tid] : 0x7fffffff;
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        const float od = __shfl_xor_sync(0xffffffffu, bd, o);
        const int oi = __shfl_xor_sync(0xffffffffu, bi, o);
        if (od > bd || (od == bd && oi < bi)) { bd = od; bi = oi; }
      }
      if (tid == 0) {
        s_pick = bi;
        if (bi < n) d[bi] = -CUDART_INF_F;                       // taken: not picked again
      }
    }
    __syncthreads();
    const int pick = s_pick;
    if (pick >= n) break;                                        // (uniform; no distance is a number)
    if (tid < kD) centroids[((size_t)unit * pl.n_list + j) * kD + tid] = U[((size_t)unit * pl.N_max + pick) * kD + tid];
    ++j;
    __syncthreads();
  }
  if (tid == 0) n_empty[unit] = 0;
}

// ---- residuals e_i = u_i - c_{a_i}, in place of the directions
__global__ void __launch_bounds__(kPrepThreads)
build_residual_kernel(Plan pl, float* __restrict__ U, const float* __restrict__ centroids,
                      const uint16_t* __restrict__ list_ids, const int32_t* __restrict__ seq_lens) {
  const int kv = blockIdx.y, b = blockIdx.z;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int n = clamp_len(seq_lens[b], pl.N_max);
  const size_t ukv = (size_t)b * pl.Hkv + kv;
  constexpr int kPer = 4;
  for (int i0 = (blockIdx.x * (kPrepThreads / 32) + warp) * kPer; i0 < n; i0 += gridDim.x * (kPrepThreads / 32) * kPer) {
    float4 u[kPer], c[kPer];
    float4* at = reinterpret_cast<float4*>(U + (ukv * pl.N_max + i0) * kD) + lane;
#pragma unroll
    for (int t = 0; t < kPer; ++t) {
      if (i0 + t >= n) break;
      const uint32_t a = min((uint32_t)list_ids[ukv * pl.N_max + i0 + t], (uint32_t)(pl.n_list - 1));
      u[t] = __ldcg(at + t * (kD / 4));
      c[t] = __ldg(reinterpret_cast<const float4*>(centroids + (ukv * pl.n_list + a) * kD) + lane);
    }
#pragma unroll
    for (int t = 0; t < kPer; ++t) {
      if (i0 + t >= n) break;
      at[t * (kD / 4)] = make_float4(u[t].x - c[t].x, u[t].y - c[t].y, u[t].z - c[t].z, u[t].w - c[t].w);
    }
  }
}

// ---- product quantisation of the residuals E.  Codebooks [unit][M][n_code][dsub].
// Seeds: codeword z of subspace m <- residual sub-vector m of the token at seed_pos[unit][z].
template <int DSUB>
__global__ void build_pq_seed_kernel(Plan pl, const float* __restrict__ E, const int32_t* __restrict__ seed_pos,
                                     float* __restrict__ codebooks) {
  const size_t unit = blockIdx.y;
  const int z = blockIdx.x, d = threadIdx.x;                 // 128 threads: one per dim
  const int pos = seed_pos[unit * pl.n_code + z];
  float e = 0.f;
  if (pos >= 0 && pos < pl.N_max) e = E[(unit * pl.N_max + pos) * kD + d];
  const int m = d / DSUB, t = d % DSUB;
  codebooks[((unit * pl.M + m) * pl.n_code + z) * DSUB + t] = e;
}

// Nearest codeword of every (token, subspace) on the tensor cores.  A CTA keeps the codebooks of
// kMg subspaces (64 bytes of a residual row) as tensor-core tiles and walks a range of tokens, 128 at
// a time per warpgroup: thread = token = accumulator row.  The accumulators give the group of 8
// codewords that holds the minimum, the codeword is decided in fp32 among those 8 (distance =
// (|e|^2 - 2 e.p) + |p|^2, lower index on ties); where a second group comes within the rounding, or two
// of the 8 are equal, all codewords are compared in fp32 (one sub-vector in some thousand).  Training
// accumulates the codewords' sums in 64-bit fixed point: two 32-bit shared-memory limbs of 21 bits and
// the rest (native integer atomics), folded into 64 bits every kFoldSteps steps, before a limb could
// overflow.
// What bounds it: the integer pipe (minima, comparisons, selects) and, with one warp of each group per
// scheduler, the 650 clocks from an MMA's issue to its mbarrier.  1 M tokens x 32 subspaces x 256
// codewords: 1190 us a training pass and 1050 us for the codes with run-time sizes, the codewords decided
// before the next MMA and codes stored byte by byte; 1037 and 914 us so; 1170 and 1034 us with the second
// group kept beside the first.  MMAs of 64 codewords into two accumulators: 1505 and 1395.
template <int DSUB, int NC> struct PqPlan {
  using Tile = PqTile<DSUB>;
  static constexpr int kMg8 = 16 / DSUB;                     // subspaces per CTA, 8-bit codes
  static constexpr int kMg = NC == 16 && kMg8 < 2 ? 2 : kMg8;   // (4-bit codes: whole bytes)
  static constexpr int kWords = kMg * NC;
  static constexpr int kBits = NC == 16 ? 4 : 8, kBytes = kMg * kBits / 8;      // codes of one token
  static constexpr size_t smem(bool train) {
    return (size_t)kWords * (Tile::kChunks * 16 + DSUB * 4) + 4 * Tile::kChunks * 2048 +
           (train ? (size_t)kWords * ((2 * DSUB + 1) * 4 + DSUB * 8) : 0);
  }
};
constexpr int kPqThreads = 512, kPqStep = 512;               // tokens per CTA and step
constexpr int kFoldSteps = 3;                                // 1536 tokens: 2^21 * 1536 < 2^32, 2^20 * 1536 < 2^31
constexpr int kLimbBits = 21;
constexpr float kLimbRange = 7.f;                            // |e|^2 below it: 2^19 |e_t| * 1536 < 2^31
constexpr int kPqCols = 128;                                 // codewords per MMA step
// x * kFixDir to the nearest integer as hi * 2^21 + lo, |lo| <= 2^20, for |x| < 8: rounded by the adder
// (1.5 * 2^23 in, its bits out), the conversion instruction being an eighth as fast
__device__ __forceinline__ void limbs(float x, int& hi, int& lo) {
  constexpr float kMagic = 12582912.f;
  const float y = x * (kFixDir / (float)(1 << kLimbBits)), h = y + kMagic;
  const float l = fmaf(y - (h - kMagic), (float)(1 << kLimbBits), kMagic);
  hi = __float_as_int(h) - __float_as_int(kMagic);
  lo = __float_as_int(l) - __float_as_int(kMagic);
}

// a sub-vector into the sums of codeword z of subspace mm
template <int DSUB, int NC>
__device__ __forceinline__ void add_member(uint32_t* s_limb, int mm, const float (&x)[DSUB], uint32_t z) {
  uint32_t* l = s_limb + mm * (2 * DSUB + 1) * NC + z;
#pragma unroll
  for (int t = 0; t < DSUB; ++t) {
    int hi, lo;
    limbs(x[t], hi, lo);
    atomicAdd(l + (2 * t) * NC, (uint32_t)lo);
    atomicAdd(l + (2 * t + 1) * NC, (uint32_t)hi);
  }
  atomicAdd(l + 2 * DSUB * NC, 1u);
}
// (see settle_codewords; item mm is subspace m0 + mm)
template <int DSUB, int NC, bool kTrain> struct PqSettle {
  const float* rows;                                        // residuals of the warp's tokens, first subspace
  int last;                                                 // last of them inside the range
  const float* s_word;
  uint32_t* s_limb;
  long long* s_sum;
  unsigned long long result;                                // codes of this lane's token
  __device__ __forceinline__ void load(int lane, int mm, float (&x)[DSUB]) const {
    load_sub<DSUB>(rows + (long long)min(lane, last) * kD + mm * DSUB, x);
  }
  __device__ __forceinline__ float distance(int mm, const float (&x)[DSUB], int z) const {
    float w[DSUB], x2 = 0.f, dot = 0.f, p2 = 0.f;
    load_sub<DSUB>(s_word + (mm * NC + z) * DSUB, w);
#pragma unroll
    for (int t = 0; t < DSUB; ++t) { x2 = fmaf(x[t], x[t], x2); dot = fmaf(x[t], w[t], dot); p2 = fmaf(w[t], w[t], p2); }
    return (x2 - 2.0f * dot) + p2;
  }
  __device__ __forceinline__ void done(int mm, const float (&x)[DSUB], int z) {
    if constexpr (kTrain) {
      float x2 = 0.f;
#pragma unroll
      for (int t = 0; t < DSUB; ++t) x2 = fmaf(x[t], x[t], x2);
      if (x2 < kLimbRange) {
        add_member<DSUB, NC>(s_limb, mm, x, (uint32_t)z);
      } else {                                              // (not a number: as the conversion has it)
#pragma unroll
        for (int t = 0; t < DSUB; ++t)
          atomicAdd(reinterpret_cast<unsigned long long*>(s_sum + (mm * DSUB + t) * NC + z), (unsigned long long)__float2ll_rn(x[t] * kFixDir));
        atomicAdd(s_limb + (mm * (2 * DSUB + 1) + 2 * DSUB) * NC + z, 1u);
      }
    } else {
      constexpr int kBits = PqPlan<DSUB, NC>::kBits;
      result = (result & ~((unsigned long long)(NC - 1) << (mm * kBits))) | ((unsigned long long)z << (mm * kBits));
    }
  }
};

template <int DSUB, int NC, bool kTrain>
__global__ void __launch_bounds__(kPqThreads, 1)
build_pq_assign_kernel(Plan pl, const float* __restrict__ E, const float* __restrict__ codebooks,
                       const int32_t* __restrict__ seq_lens, int range, long long* __restrict__ pq_sums,
                       int32_t* __restrict__ pq_counts, uint8_t* __restrict__ codes_out,
                       float* __restrict__ key_norms) {
  using Tile = PqTile<DSUB>;
  using P = PqPlan<DSUB, NC>;
  constexpr int mg = P::kMg, nc = NC, words = P::kWords;
  extern __shared__ __align__(128) unsigned char s_pq[];
  __shared__ uint32_t s_tmem;
  __shared__ __align__(8) uint64_t s_bar[4];
  const int kv = blockIdx.y % pl.Hkv, b = blockIdx.y / pl.Hkv;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int wg = tid >> 7, row = tid & 127;
  const int n = clamp_len(seq_lens[b], pl.N_max);
  const int begin = blockIdx.x * range, end = min(n, begin + range);
  if (begin >= end) return;
  const size_t ukv = (size_t)b * pl.Hkv + kv;
  const int m0 = blockIdx.z * mg;
  // shared memory: codeword tiles, token tiles, fp32 codewords, then the training sums
  unsigned char* s_b = s_pq;                                            // [mg][chunks][nc] x 16 bytes
  unsigned char* s_a = s_b + (size_t)words * Tile::kChunks * 16;        // [4][chunks][128] x 16 bytes
  long long* s_sum = reinterpret_cast<long long*>(s_a + 4 * Tile::kChunks * 2048);   // [mg][DSUB][nc] (training)
  float* s_word = reinterpret_cast<float*>(s_sum + (kTrain ? (size_t)words * DSUB : 0));   // [mg][nc][DSUB]
  uint32_t* s_limb = reinterpret_cast<uint32_t*>(s_word + (size_t)words * DSUB);   // [mg][2 DSUB + 1][nc]
  if (warp == 0) tmem_alloc(&s_tmem, 512);
  if (tid < 4) mbar_init(&s_bar[tid], 1);
  if (tid == 0) asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  const float* cb = codebooks + (ukv * pl.M + m0) * (size_t)nc * DSUB;
  for (int w = tid; w < words; w += kPqThreads) {
    float p[DSUB];
#pragma unroll
    for (int t = 0; t < DSUB; ++t) p[t] = __ldg(cb + (size_t)w * DSUB + t);      // (the caller's: aligned to an element)
    uint4 ch[Tile::kChunks];
    Tile::code_row(p, ch);
    const int mm = w / nc, z = w - mm * nc;
#pragma unroll
    for (int i = 0; i < Tile::kChunks; ++i)
      *reinterpret_cast<uint4*>(s_b + (size_t)((mm * Tile::kChunks + i) * nc + z) * 16) = ch[i];
#pragma unroll
    for (int t = 0; t < DSUB; ++t) s_word[(size_t)w * DSUB + t] = p[t];
    if constexpr (kTrain) {
#pragma unroll
      for (int t = 0; t < DSUB; ++t) s_sum[(size_t)(mm * DSUB + t) * nc + z] = 0;
#pragma unroll
      for (int t = 0; t < 2 * DSUB + 1; ++t) s_limb[(size_t)(mm * (2 * DSUB + 1) + t) * nc + z] = 0u;
    }
  }
  tc_fence_smem();
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t d_tmem = s_tmem + (uint32_t)wg * 128u;
  const uint32_t my_tmem = d_tmem + ((uint32_t)((warp & 3) * 32) << 16);
  unsigned char* pa = s_a + wg * (Tile::kChunks * 2048);
  constexpr int kCols = nc < kPqCols ? nc : kPqCols, per = nc / kCols;   // MMA steps per subspace
  bool late = false;
  // the limbs into 64 bits (every thread its own entries); all threads call
  auto fold = [&]() {
    __syncthreads();
    for (int w = tid; w < words; w += kPqThreads) {
      const int mm = w / nc, z = w - mm * nc;
#pragma unroll
      for (int t = 0; t < DSUB; ++t) {
        uint32_t* l = s_limb + (size_t)(mm * (2 * DSUB + 1) + 2 * t) * nc + z;
        s_sum[(size_t)(mm * DSUB + t) * nc + z] += (long long)(int32_t)l[0] + ((long long)(int32_t)l[nc] << kLimbBits);
        l[0] = 0u;
        l[nc] = 0u;
      }
    }
    __syncthreads();
  };
  // Items: (512 tokens, subspace), subspaces innermost.  The next MMA of a warpgroup is issued as soon as
  // its accumulators have been read: the first of an item therefore before the last item's codewords are
  // decided in fp32, which covers its latency (about 650 clocks from issue to the mbarrier).
  auto put_row = [&](const float (&x)[DSUB]) {
    uint4 ch[Tile::kChunks];
    Tile::token_row(x, ch);
#pragma unroll
    for (int c = 0; c < Tile::kChunks; ++c) *reinterpret_cast<uint4*>(pa + (c * 128 + row) * 16) = ch[c];
    tc_fence_smem();
  };
  // codewords c * kPqCols .. of subspace mm against the group's token tile
  const uint64_t a_desc = tc_desc(smem_u32(pa), 128u * 16u), b_desc = tc_desc(smem_u32(s_b), (uint32_t)nc * 16u);
  constexpr uint32_t idesc = tc_idesc((uint32_t)kCols);
  auto issue = [&](int mm, int c) {
    tc_fence_before();
    group_sync(1 + wg);
    if (row == 0) {
      tc_fence_after();
      const uint64_t bw = b_desc + (uint32_t)(mm * Tile::kChunks * nc + c * kCols);        // (16-byte units)
#pragma unroll
      for (int s = 0; s < Tile::kChunks; s += 2) tc_mma(d_tmem, a_desc + s * 128, bw + (uint32_t)(s * nc), idesc, s != 0);
      tc_commit(&s_bar[wg]);
    }
    __syncwarp();
  };
  auto row_of = [&](int base) {
    return E + (ukv * pl.N_max + min(base + wg * 128 + row, end - 1)) * (size_t)kD + m0 * DSUB;
  };
  constexpr uint32_t kRow = DSUB * 4;                       // bytes of a codeword
  const uint32_t rot = (uint32_t)(lane & 7) * kRow;
  float e[DSUB], e_nxt[DSUB];
  const float* er = row_of(begin);
  load_sub<DSUB>(er, e_nxt);
  put_row(e_nxt);
  issue(0, 0);
  uint32_t parity = 0u;
  int steps = 0;
  for (int base = begin; base < end; base += kPqStep) {
    const bool more = base + kPqStep < end;
    const float* er_next = more ? row_of(base + kPqStep) : er;
    const int i = base + wg * 128 + row;
    const bool real = i < end;
    unsigned long long code = 0ull;
    unsigned ties = 0u;                                     // bit mm: decided after the others
#pragma unroll 1
    for (int mm = 0; mm < mg; ++mm) {
#pragma unroll
      for (int t = 0; t < DSUB; ++t) e[t] = e_nxt[t];
      const bool next = mm + 1 < mg || more;
      load_sub<DSUB>(mm + 1 < mg ? er + (mm + 1) * DSUB : er_next, e_nxt);
      NearestGroup ng;
      ng.clear();
#pragma unroll
      for (int c = 0; c < per; ++c) {
        late |= !tc_wait(&s_bar[wg], parity);
        parity ^= 1u;
        tc_fence_after();
        if (c + 1 == per && next) put_row(e_nxt);           // (the item's last MMA is done)
        if constexpr (nc == 16) {
          float acc[16];
          tmem_ld16(my_tmem, acc);
          ng.take(acc, 0u);
        } else {
#pragma unroll
          for (int h = 0; h < kCols; h += 32) {
            float acc[32];
            tmem_ld32(my_tmem + h, acc);
            ng.take(acc, (uint32_t)(c * kCols + h) / 8u);
          }
        }
        if (c + 1 < per) issue(mm, c + 1);
        else if (next) issue(mm + 1 < mg ? mm + 1 : 0, 0);
      }
      // the winning group in fp32, lower index on ties; the lanes start at different codewords, so that
      // at 16 bytes a codeword the eight lanes of an access hit eight different bank groups
      float en = 0.f, dist[8];
#pragma unroll
      for (int t = 0; t < DSUB; ++t) en = fmaf(e[t], e[t], en);
      const uint32_t at = (uint32_t)(8 * ng.group()) * kRow + rot;
      const unsigned char* s_sub = reinterpret_cast<const unsigned char*>(s_word) + (size_t)mm * nc * kRow;
#pragma unroll
      for (int q = 0; q < 8; ++q) {
        float w[DSUB], dot = 0.f, p2 = 0.f;
        load_sub<DSUB>(reinterpret_cast<const float*>(s_sub + (at ^ (q * kRow))), w);
#pragma unroll
        for (int t = 0; t < DSUB; ++t) { dot = fmaf(e[t], w[t], dot); p2 = fmaf(w[t], w[t], p2); }
        dist[q] = (en - 2.0f * dot) + p2;
      }
      const float dm = min3(min3(dist[0], dist[1], dist[2]), min3(dist[3], dist[4], dist[5]), fminf(dist[6], dist[7]));
      uint32_t above = 0u;                                  // bit 7 - q: codeword q of the lane's order is farther
#pragma unroll
      for (int q = 0; q < 8; ++q) above = __funnelshift_l(__float_as_uint(dm - dist[q]), above, 1);
      const uint32_t equal = ~above << 24;                  // (not a number: all)
      const uint32_t bz = (at ^ ((uint32_t)__clz(equal) * kRow)) / kRow;
      // (equal distances: the lower index; beyond the range of limbs and fp16 terms, as next to a centroid
      // with a member that is not a number: see PqSettle)
      const bool tie = pq_tie(ng, en) || (equal & (equal - 1u)) != 0u || !(en < kLimbRange);
      if (tie) ties |= 1u << mm;
      if constexpr (kTrain) {
        if (real && !tie) add_member<DSUB, NC>(s_limb, mm, e, bz);
      } else {
        code |= (unsigned long long)bz << (mm * P::kBits);
      }
    }
    // where another group may hold a codeword as near: all of them
    if (__any_sync(0xffffffffu, real && ties != 0u)) {
      const PqSettle<DSUB, NC, kTrain> st = {E + (ukv * pl.N_max + i - lane) * (size_t)kD + m0 * DSUB, end - 1 - (i - lane), s_word, s_limb, s_sum, code};
      code = settle_codewords<DSUB, NC>(real ? ties : 0u, mg, st);
    }
    if constexpr (!kTrain) {
      if (real) {
        uint8_t* dst = codes_out + (ukv * pl.N_max + i) * pl.code_bytes + m0 * P::kBits / 8;
        if ((reinterpret_cast<uintptr_t>(dst) & (P::kBytes - 1)) != 0) {      // (the caller's array starts anywhere)
#pragma unroll
          for (int t = 0; t < P::kBytes; ++t) dst[t] = (uint8_t)(code >> (8 * t));
        } else if constexpr (P::kBytes == 8) *reinterpret_cast<unsigned long long*>(dst) = code;
        else if constexpr (P::kBytes == 4) *reinterpret_cast<uint32_t*>(dst) = (uint32_t)code;
        else if constexpr (P::kBytes == 2) *reinterpret_cast<uint16_t*>(dst) = (uint16_t)code;
        else *dst = (uint8_t)code;
      }
    }
    if (late && real) key_norms[ukv * pl.N_max + i] = CUDART_NAN_F;    // a bounded wait ran out
    er = er_next;
    if constexpr (kTrain) {
      if (++steps == kFoldSteps) { fold(); steps = 0; }
    }
  }
  if constexpr (kTrain) {
    fold();
    for (int w = tid; w < words; w += kPqThreads) {
      const int mm = w / nc, z = w - mm * nc;
      const size_t at = (ukv * pl.M + m0 + mm) * nc + z;
      const uint32_t c = s_limb[(size_t)(mm * (2 * DSUB + 1) + 2 * DSUB) * nc + z];
      if (c == 0u) continue;
      atomicAdd(&pq_counts[at], (int32_t)c);
#pragma unroll
      for (int t = 0; t < DSUB; ++t)
        atomicAdd(reinterpret_cast<unsigned long long*>(pq_sums + at * DSUB + t),
                  (unsigned long long)s_sum[(size_t)(mm * DSUB + t) * nc + z]);
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 0) { tc_fence_after(); tmem_free(s_tmem, 512); }
}

// codeword <- mean of its members (kept if it has none); sums and counts cleared
__global__ void build_pq_update_kernel(size_t n_entries, int dsub, long long* __restrict__ pq_sums,
                                       int32_t* __restrict__ pq_counts, float* __restrict__ codebooks) {
  const size_t e = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= n_entries) return;
  const int c = pq_counts[e];
  for (int t = 0; t < dsub; ++t) {
    if (c > 0) codebooks[e * dsub + t] = fix_mean(pq_sums[e * dsub + t], c, kFixDir);
    pq_sums[e * dsub + t] = 0;
  }
  pq_counts[e] = 0;
}

// ---- list value means over the members inside R and member counts (Eq. 4's vbar_j)
template <typename T>
__global__ void __launch_bounds__(kPrepThreads)
build_value_sums_kernel(Plan pl, const T* __restrict__ vc, long long sp, long long st, long long sh,
                        const int32_t* __restrict__ block_table, const int32_t* __restrict__ seq_lens,
                        const uint16_t* __restrict__ list_ids, const int32_t* __restrict__ order,
                        long long* __restrict__ sums) {
  const int kv = blockIdx.y, b = blockIdx.z;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int n = clamp_len(seq_lens[b], pl.N_max);
  const Region rg = region_of(pl, n, b);
  const size_t ukv = (size_t)b * pl.Hkv + kv;
  const int members = rg.r_end - rg.r_begin;
  const int first = (blockIdx.x * (kPrepThreads / 32) + warp) * kRun, last = min(members, first + kRun);
  if (first >= members) return;
  const int32_t* bt = block_table + (size_t)b * pl.max_pages;
  auto sum = [&](auto row) {
    run_sums(pl, list_ids + ukv * pl.N_max, order + ukv * pl.N_max, first, last, kFixVal, sums + ukv * pl.n_list * (size_t)kD,
             [&](int i) { return kv_row(pl, bt, i, kv, sp, st, sh); }, row);
  };
  // (asked once: a question per row kept its loads from being issued together, 156 -> 214 us)
  if (whole_rows(vc)) sum([&](long long at, float (&x)[4]) { to_fp32<T>(load_four<true>(vc + at + 4 * lane), x); });
  else sum([&](long long at, float (&x)[4]) { to_fp32<T>(load_four<false>(vc + at + 4 * lane), x); });
}

__global__ void build_value_means_kernel(Plan pl, long long* __restrict__ sums, const int32_t* __restrict__ counts,
                                         float* __restrict__ vmeans, int32_t* __restrict__ list_counts) {
  const size_t unit = blockIdx.y;
  const int j = blockIdx.x * (blockDim.x / 32) + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  if (j >= pl.n_list) return;
  const size_t at = (unit * pl.n_list + j) * kD + 4 * lane;
  const int c = counts[unit * pl.n_list + j];
  float4 s = make_float4(0.f, 0.f, 0.f, 0.f);
  if (c > 0)
    s = make_float4(fix_mean(sums[at], c, kFixVal), fix_mean(sums[at + 1], c, kFixVal),
                    fix_mean(sums[at + 2], c, kFixVal), fix_mean(sums[at + 3], c, kFixVal));
  *reinterpret_cast<float4*>(vmeans + at) = s;
#pragma unroll
  for (int t = 0; t < 4; ++t) sums[at + t] = 0;
  if (lane == 0) list_counts[unit * pl.n_list + j] = c;
}

struct BuildWs {
  size_t U, dmin, images, order, cursor, sums, counts, n_empty, pq_sums, pq_counts, total;
};
size_t up256(size_t x) { return (x + 255) / 256 * 256; }
BuildWs build_layout(const Plan& pl) {
  BuildWs w;
  size_t o = 0;
  auto take = [&](size_t bytes) { size_t at = o; o = up256(o + bytes); return at; };
  const size_t units = (size_t)pl.B * pl.Hkv;
  w.U = take(units * pl.N_max * kD * 4);
  w.dmin = take(units * pl.N_max * 4);
  w.images = take(units * ((pl.n_list + kAsgCen - 1) / kAsgCen) * (size_t)kCenTileBytes);
  w.order = take(units * pl.N_max * 4);
  w.cursor = take(units * pl.n_list * 4);
  w.sums = take(units * pl.n_list * kD * 8);
  w.counts = take(units * pl.n_list * 4);
  w.n_empty = take(units * 4);
  w.pq_sums = take(units * pl.M * pl.n_code * pl.dsub * 8);
  w.pq_counts = take(units * pl.M * pl.n_code * 4);
  w.total = o;
  return w;
}

#define PQHSA_TRY(x) do { e = (x); if (e != cudaSuccess) return e; } while (0)

// codebooks (pq_iters rounds of k-means from the seeded residuals U), then the codes
template <int DSUB, int NC>
cudaError_t pq_build(const Plan& pl, const float* U, const int32_t* seq_lens, const int32_t* seed_codes, int pq_iters,
                     long long* pq_sums, int32_t* pq_counts, const pqhsa_index_out& ix, cudaStream_t st) {
  using P = PqPlan<DSUB, NC>;
  const int units = pl.B * pl.Hkv;
  if (pl.M % P::kMg != 0) return cudaErrorInvalidValue;
  // about three waves of CTAs, each over a range of tokens that is a multiple of a step; of the splits
  // near that, the one whose last wave is fullest
  const int columns = units * (pl.M / P::kMg), total_steps = (pl.N_max + kPqStep - 1) / kPqStep;
  int steps = total_steps, best_cost = 0x7fffffff;
  for (int s = total_steps; s >= 1; --s) {
    const int ranges = (total_steps + s - 1) / s;
    const long long ctas = (long long)ranges * columns;
    if (ctas > 8LL * pl.num_sms && best_cost != 0x7fffffff) break;
    const int waves = (int)((ctas + pl.num_sms - 1) / pl.num_sms), cost = waves * (s + 2);    // (+ 2: start and end of a CTA)
    if (cost < best_cost) { best_cost = cost; steps = s; }
  }
  const dim3 grid((total_steps + steps - 1) / steps, units, pl.M / P::kMg);
  cudaError_t e;
  const int range = steps * kPqStep, smem_train = (int)P::smem(true), smem_code = (int)P::smem(false);
  PQHSA_TRY(cudaFuncSetAttribute(build_pq_assign_kernel<DSUB, NC, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem_train));
  PQHSA_TRY(cudaFuncSetAttribute(build_pq_assign_kernel<DSUB, NC, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem_code));
  const size_t n_entries = (size_t)units * pl.M * NC;
  build_pq_seed_kernel<DSUB><<<dim3(NC, units), kD, 0, st>>>(pl, U, seed_codes, ix.codebooks);
  for (int it = 0; it < pq_iters; ++it) {
    build_pq_assign_kernel<DSUB, NC, true><<<grid, kPqThreads, smem_train, st>>>(
        pl, U, ix.codebooks, seq_lens, range, pq_sums, pq_counts, nullptr, ix.key_norms);
    build_pq_update_kernel<<<(unsigned)((n_entries + 255) / 256), 256, 0, st>>>(n_entries, DSUB, pq_sums, pq_counts, ix.codebooks);
  }
  build_pq_assign_kernel<DSUB, NC, false><<<grid, kPqThreads, smem_code, st>>>(
      pl, U, ix.codebooks, seq_lens, range, nullptr, nullptr, ix.codes, ix.key_norms);
  return cudaSuccess;
}

template <typename T, int DSUB>
cudaError_t run_build(const Plan& pl, const pqhsa_paged_kv& kv, const int32_t* seq_lens,
                      const int32_t* seed_lists, const int32_t* seed_codes, int coarse_iters,
                      int pq_iters, const pqhsa_index_out& ix, char* ws, cudaStream_t st) {
  const BuildWs w = build_layout(pl);
  float* U = reinterpret_cast<float*>(ws + w.U);
  float* dmin = reinterpret_cast<float*>(ws + w.dmin);
  long long* sums = reinterpret_cast<long long*>(ws + w.sums);
  int32_t* counts = reinterpret_cast<int32_t*>(ws + w.counts);
  int32_t* n_empty = reinterpret_cast<int32_t*>(ws + w.n_empty);
  long long* pq_sums = reinterpret_cast<long long*>(ws + w.pq_sums);
  int32_t* pq_counts = reinterpret_cast<int32_t*>(ws + w.pq_counts);
  const int units = pl.B * pl.Hkv;
  const T* kc = static_cast<const T*>(kv.k_cache);
  const T* vc = static_cast<const T*>(kv.v_cache);
  const long long sp = kv.stride_page, stt = kv.stride_token, sh = kv.stride_head;
  cudaError_t e;
  PQHSA_TRY(cudaMemsetAsync(ws + w.sums, 0, w.total - w.sums, st));
  unsigned char* images = reinterpret_cast<unsigned char*>(ws + w.images);
  int32_t* order = reinterpret_cast<int32_t*>(ws + w.order);
  int32_t* cursor = reinterpret_cast<int32_t*>(ws + w.cursor);
  const int tok_ctas = min(1024, (pl.N_max + 7) / 8);
  build_prepare_kernel<T><<<dim3(tok_ctas, pl.Hkv, pl.B), kPrepThreads, 0, st>>>(
      pl, kc, sp, stt, sh, kv.block_table, seq_lens, U, ix.key_norms);
  build_seed_kernel<<<dim3((pl.n_list + 7) / 8, units), 256, 0, st>>>(pl, U, seed_lists, pl.n_list, ix.centroids);
  PQHSA_TRY(cudaFuncSetAttribute(build_assign_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kAsgSmemBytes));
  const dim3 asg_grid((pl.N_max + kAsgTok - 1) / kAsgTok, pl.Hkv, pl.B);
  const dim3 split_grid((pl.n_list + kAsgCen - 1) / kAsgCen, units);
  const dim3 list_grid((pl.n_list + 7) / 8, units);
  const dim3 sort_grid((pl.N_max + kSortChunk - 1) / kSortChunk, pl.Hkv, pl.B);
  const dim3 run_grid((pl.N_max + kRun * (kPrepThreads / 32) - 1) / (kRun * (kPrepThreads / 32)), pl.Hkv, pl.B);
  const size_t list_smem = (size_t)pl.n_list * 4;
  auto assign = [&]() {
    build_split_kernel<<<split_grid, 4 * kAsgCen, 0, st>>>(pl, ix.centroids, images);
    build_assign_kernel<<<asg_grid, kAsgThreads, kAsgSmemBytes, st>>>(pl, U, images, ix.centroids, seq_lens, ix.list_ids, ix.key_norms);
  };
  for (int it = 0; it < coarse_iters; ++it) {
    assign();
    PQHSA_TRY(cudaMemsetAsync(counts, 0, (size_t)units * pl.n_list * 4, st));
    build_hist_kernel<false><<<sort_grid, kSortThreads, list_smem, st>>>(pl, ix.list_ids, seq_lens, counts);
    build_offsets_kernel<<<units, 1024, 0, st>>>(pl, counts, cursor, n_empty);
    build_distance_kernel<<<dim3(min(64, (pl.N_max + kPrepThreads - 1) / kPrepThreads), pl.Hkv, pl.B), kPrepThreads, 0, st>>>(
        pl, U, ix.centroids, seq_lens, ix.list_ids, n_empty, dmin);
    build_scatter_kernel<false><<<sort_grid, kSortThreads, list_smem, st>>>(pl, ix.list_ids, seq_lens, cursor, order);
    build_dir_sums_kernel<<<run_grid, kPrepThreads, 0, st>>>(pl, U, ix.list_ids, order, seq_lens, sums);
    build_update_centroids_kernel<<<list_grid, 256, 0, st>>>(pl, sums, counts, ix.centroids);
    build_reseed_kernel<<<units, 1024, 0, st>>>(pl, U, dmin, counts, seq_lens, n_empty, ix.centroids);
  }
  assign();
  build_residual_kernel<<<dim3(tok_ctas, pl.Hkv, pl.B), kPrepThreads, 0, st>>>(pl, U, ix.centroids, ix.list_ids, seq_lens);
  const cudaError_t e_pq = pl.n_code == 16 ? pq_build<DSUB, 16>(pl, U, seq_lens, seed_codes, pq_iters, pq_sums, pq_counts, ix, st)
                                           : pq_build<DSUB, 256>(pl, U, seq_lens, seed_codes, pq_iters, pq_sums, pq_counts, ix, st);
  if (e_pq != cudaSuccess) return e_pq;
  // list value means and member counts
  PQHSA_TRY(cudaMemsetAsync(counts, 0, (size_t)units * pl.n_list * 4, st));
  build_hist_kernel<true><<<sort_grid, kSortThreads, list_smem, st>>>(pl, ix.list_ids, seq_lens, counts);
  build_offsets_kernel<<<units, 1024, 0, st>>>(pl, counts, cursor, nullptr);
  build_scatter_kernel<true><<<sort_grid, kSortThreads, list_smem, st>>>(pl, ix.list_ids, seq_lens, cursor, order);
  build_value_sums_kernel<T><<<run_grid, kPrepThreads, 0, st>>>(
      pl, vc, sp, stt, sh, kv.block_table, seq_lens, ix.list_ids, order, sums);
  build_value_means_kernel<<<list_grid, 256, 0, st>>>(pl, sums, counts, ix.list_vmeans, ix.list_counts);
#undef PQHSA_TRY
  return cudaGetLastError();
}

}  // namespace
}  // namespace pqhsa

using namespace pqhsa;

extern "C" {

size_t pqhsa_index_build_workspace_bytes(const pqhsa_params* params) {
  Plan pl;
  if (make_plan(params, &pl) != PQHSA_OK) return 0;
  return build_layout(pl).total;
}

int pqhsa_index_build(const pqhsa_params* params, const pqhsa_paged_kv* kv, const int32_t* seq_lens,
                      const int32_t* seed_lists, const int32_t* seed_codes, int32_t coarse_iters,
                      int32_t pq_iters, const pqhsa_index_out* index, void* ws, size_t ws_bytes,
                      void* stream) {
  Plan pl;
  int rc = make_plan(params, &pl);
  if (rc != PQHSA_OK) return rc;
  if (kv == nullptr || kv->k_cache == nullptr || kv->v_cache == nullptr || kv->block_table == nullptr ||
      seq_lens == nullptr || seed_lists == nullptr || seed_codes == nullptr || index == nullptr ||
      index->centroids == nullptr || index->codebooks == nullptr || index->codes == nullptr ||
      index->list_ids == nullptr || index->key_norms == nullptr || index->list_vmeans == nullptr ||
      index->list_counts == nullptr || coarse_iters < 0 || pq_iters < 0 || ws == nullptr ||
      (reinterpret_cast<uintptr_t>(ws) & 255u) != 0)
    return PQHSA_ERR_INVALID_ARG;
  if (kv->stride_page % 8 || kv->stride_token % 8 || kv->stride_head % 8) return PQHSA_ERR_UNSUPPORTED;
  if (ws_bytes < build_layout(pl).total) return PQHSA_ERR_WORKSPACE;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  char* w = static_cast<char*>(ws);
  cudaError_t e = cudaErrorInvalidValue;
#define PQHSA_BUILD_CASE(DS)                                                                        \
  if (pl.dsub == DS)                                                                                \
    e = pl.dtype == PQHSA_F16                                                                       \
            ? run_build<__half, DS>(pl, *kv, seq_lens, seed_lists, seed_codes, coarse_iters,        \
                                    pq_iters, *index, w, st)                                        \
            : run_build<__nv_bfloat16, DS>(pl, *kv, seq_lens, seed_lists, seed_codes, coarse_iters, \
                                           pq_iters, *index, w, st);
  PQHSA_BUILD_CASE(2) PQHSA_BUILD_CASE(4) PQHSA_BUILD_CASE(8) PQHSA_BUILD_CASE(16)
#undef PQHSA_BUILD_CASE
  return e == cudaSuccess ? PQHSA_OK : PQHSA_ERR_CUDA;
}

}  // extern "C"
