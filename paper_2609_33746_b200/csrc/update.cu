// Index maintenance between decode steps (Sec. 3.3, first paragraph): tokens that leave the
// local window are encoded into the existing lists, without re-clustering, and the list value
// means are refreshed.  Encoding follows Sec. 3.1: r_i = |k_i| (fp32), u_i = k_i / r_i,
// a_i = the list whose centroid is nearest to u_i (squared Euclidean distance, lower index on
// ties), z_im = the codeword nearest to the m-th sub-vector of the residual u_i - c_{a_i}.
//
//   index_encode_kernel         128 new tokens of one (sequence, KV head) per CTA.  Both searches
//       are contractions and run on the tensor cores with split fp16 operands (tc.cuh): tiles of 128
//       centroids, then every warpgroup takes every fourth subspace.  What comes within the rounding of
//       the nearest, and centres too far out for fp16, are compared in fp32: lists and codes are those of
//       an fp32 search.  The codeword is decided in fp32 among the 8 of the winning group.
//   index_encode_few_kernel     the same with fp32 FMAs, 8 tokens per CTA: few tokens against few lists.
//   index_refresh_means_kernel  groups the new tokens by list (first occurrence = leader), sums
//       each group's value rows in token order and sets vbar_j = (n_j vbar_j + sum) / (n_j + new_j),
//       n_j += new_j; a warp per leader.
// What bounds the encoding: latency.  The rows' first loads, the centroids (512 KB at 1024 lists, through
// registers once to be split), then the codes: short steps of store, MMA, wait and search per subspace.
// 8 requests x 8 KV heads x 256 new tokens: 779 us with fp32 FMAs and a serial grouping of the means, 74
// with the split searches alone, 80 with what fp32 decides.
#include "attn_common.cuh"
#include "common.cuh"
#include "tc.cuh"

namespace pqhsa {

namespace {

constexpr int kUpdTok = 128;            // tokens per CTA: rows of the tensor-core tile
constexpr int kUpdGroups = 4;           // warpgroups
constexpr int kUpdThreads = 128 * kUpdGroups;
constexpr int kUpdWarps = kUpdThreads / 32;
constexpr int kUpdCen = 128;            // centroids per tile, 32 columns per warpgroup
constexpr int kUpdWords = 128;          // codewords per tile of a warpgroup
constexpr int kUStride = kHeadDim + 4;  // floats per row of the directions in shared memory
constexpr int kMaxNew = 1024;           // new tokens per sequence and call
constexpr int kMeanTok = 16;            // positions per CTA of the means kernel: one per warp
constexpr int kMeanThreads = 512;

// dynamic shared memory: token tile and two centroid tiles; the residuals and the tiles of the
// codeword search (token rows and codeword rows per warpgroup) take their place afterwards
constexpr int kUpdU = kUpdTok * kUStride * 4;
constexpr int kUpdA = kCoarseChunks * kUpdTok * 16;
constexpr int kUpdB = kCoarseChunks * kUpdCen * 16;
constexpr int kUpdSmem = kUpdA + 2 * kUpdB;
constexpr int kUpdPq = (kUpdSmem - kUpdU) / kUpdGroups;     // codeword search, per warpgroup
static_assert(kUpdU <= kUpdB, "the directions pass through a centroid tile's place");
static_assert(2 * 8 * 128 * 16 <= kUpdPq && kUpdPq % 128 == 0, "codeword tiles of the widest subspace");

// cache row of token `pos` of (sequence b, KV head kv), in elements
__device__ __forceinline__ long long row_offset(const Plan& pl, const int32_t* __restrict__ bt,
                                                int pos, int kv, long long stride_page,
                                                long long stride_token, long long stride_head) {
  const int page = __ldg(bt + pos / pl.page_size);
  return (long long)page * stride_page + (long long)(pos % pl.page_size) * stride_token +
         (long long)kv * stride_head;
}

// |x - word|^2, one chain over the dims
template <int DSUB> __device__ __forceinline__ float word_distance(const float (&x)[DSUB], const float* word) {
  float w[DSUB], dist = 0.f;
  load_sub<DSUB>(word, w);
#pragma unroll
  for (int t = 0; t < DSUB; ++t) dist = fmaf(x[t] - w[t], x[t] - w[t], dist);
  return dist;
}
// (see settle_codewords; item i is subspace wg + 4 i)
template <int DSUB> struct UpdateSettle {
  const float* rows;                                        // residuals of the warp's tokens, first subspace
  const float* words;                                       // its codebook
  size_t item_words;                                        // floats to the next item's
  uint8_t* code;                                            // this lane's
  unsigned long long result;
  __device__ __forceinline__ void load(int lane, int i, float (&x)[DSUB]) const {
    load_sub<DSUB>(rows + lane * kUStride + i * kUpdGroups * DSUB, x);
  }
  __device__ __forceinline__ float distance(int i, const float (&x)[DSUB], int z) const {
    return word_distance<DSUB>(x, words + i * item_words + z * DSUB);
  }
  __device__ __forceinline__ void done(int i, const float (&)[DSUB], int z) { code[i * kUpdGroups] = (uint8_t)z; }
};

template <typename T, int DSUB>
__global__ void __launch_bounds__(kUpdThreads, 1)
index_encode_kernel(Plan pl, const T* __restrict__ kc, long long stride_page, long long stride_token,
                    long long stride_head, const int32_t* __restrict__ block_table,
                    const int32_t* __restrict__ first_pos, const int32_t* __restrict__ n_new,
                    int max_new, const float* __restrict__ centroids,
                    const float* __restrict__ codebooks, uint8_t* __restrict__ codes,
                    uint16_t* __restrict__ list_ids, float* __restrict__ key_norms) {
  extern __shared__ __align__(128) unsigned char s_dyn[];
  unsigned char* s_a = s_dyn;
  unsigned char* s_b = s_a + kUpdA;
  __shared__ float s_best[2][kUpdGroups][kUpdTok];               // the groups' two nearest blocks
  __shared__ uint16_t s_at[2][kUpdGroups][kUpdTok];
  __shared__ uint8_t s_blocks[kUpdGroups][kUpdTok];              // how many within reach, 128: a pair
  __shared__ uint32_t s_seen[kUpdGroups][kUpdTok];               // which of them, a bit per tile
  __shared__ uint16_t s_near[kUpdTok], s_tie[2][kUpdTok];        // the nearest; blocks to search in fp32, or none
  __shared__ float s_x2[kUpdTok];                                // |u|^2
  __shared__ uint8_t s_crowd[kUpdTok];                           // tokens that fp32 searches for
  __shared__ int s_n_crowd, s_wild, s_wild_words[kUpdGroups];
  __shared__ Found s_found[kUpdWarps][kCrowd];
  __shared__ __align__(16) uint8_t s_code[kUpdTok][64];
  __shared__ uint32_t s_tmem;
  __shared__ __align__(8) uint64_t s_bar[2 + kUpdGroups];        // centroid tiles, codeword tiles
  const int kv = blockIdx.y, b = blockIdx.z;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int wg = tid >> 7, row = tid & 127, wq = warp & 3;  // warpgroup, tile row, warp in the group
  const size_t ukv = (size_t)b * pl.Hkv + kv;
  pdl_wait();
  pdl_launch_dependents();
  const int nb = min(max(n_new[b], 0), max_new);
  const int t0 = blockIdx.x * kUpdTok;
  if (t0 >= nb) return;
  const int ntok = min(kUpdTok, nb - t0);
  const int p0 = first_pos[b] + t0;                 // position of this CTA's first token
  const int32_t* bt = block_table + (size_t)b * pl.max_pages;
  // tokens whose position falls outside the index rows are left alone
  auto ok = [&](int t) { return t < ntok && p0 + t >= 0 && p0 + t < pl.N_max; };

  if (warp == 0) tmem_alloc(&s_tmem, 512);
  if (tid < 2 + kUpdGroups) mbar_init(&s_bar[tid], 1);
  if (tid < kUpdGroups) s_wild_words[tid] = -1;
  if (tid == 0) { s_n_crowd = 0; s_wild = 0; }
  if (tid == 0) asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");

  // ---- norms and directions: a warp per token, a lane holds 4 of the 128 dims
  constexpr int kPer = kUpdTok / kUpdWarps;
  uint2 raw[kPer];                                          // (kept for the residuals)
  float inv[kPer];
#pragma unroll
  for (int r = 0; r < kPer; ++r) {
    const int t = r * kUpdWarps + warp;
    raw[r] = make_uint2(0u, 0u);
    if (ok(t))
      raw[r] = load_four(kc + row_offset(pl, bt, p0 + t, kv, stride_page, stride_token, stride_head) + 4 * lane);
  }
  auto direction = [&](int r, float (&x)[4]) {
    float f[8];
    Unpack<T>::run(make_uint4(raw[r].x, raw[r].y, 0u, 0u), f);
#pragma unroll
    for (int i = 0; i < 4; ++i) x[i] = __fmul_rn(f[i], inv[r]);      // (not contracted into what follows)
  };
  {
    float* s_u = reinterpret_cast<float*>(s_b);
#pragma unroll
    for (int r = 0; r < kPer; ++r) {
      const int t = r * kUpdWarps + warp;
      float x[4];
      inv[r] = 1.f;
      direction(r, x);
      const float ss = warp_sum(x[0] * x[0] + x[1] * x[1] + x[2] * x[2] + x[3] * x[3]);
      const float nr = sqrtf(ss);
      inv[r] = nr > 0.f ? 1.f / nr : 0.f;
      direction(r, x);
      *reinterpret_cast<float4*>(s_u + t * kUStride + 4 * lane) = make_float4(x[0], x[1], x[2], x[3]);
      // (|u|^2 = 1; less sure where the squares underflow.  0 and not-a-number stay themselves)
      if (lane == 0) s_x2[t] = nr > 1e-18f ? 1.f : nr > 0.f ? (float)kHeadDim : nr;
      if (lane == 0 && ok(t)) key_norms[ukv * pl.N_max + p0 + t] = nr;
    }
  }
  // A warp splits 8 rows of a centroid tile: lane l holds row l & 7 and the chunks (l >> 3) + 4 i, so
  // that loads take whole 128-byte lines and stores have no conflicts.  Fetched one tile ahead.
  const float* cbase = centroids + ukv * (size_t)pl.n_list * kHeadDim;
  const int br = 8 * warp + (lane & 7), bc = lane >> 3;
  float v[4][8];
  auto fetch = [&](int c0) {
    const bool real = c0 + br < pl.n_list;
    const float4* src = reinterpret_cast<const float4*>(cbase + (size_t)(real ? c0 + br : 0) * kHeadDim);
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      float4 x = make_float4(0.f, 0.f, 0.f, 0.f), y = x;
      if (real) { x = __ldg(src + 2 * (bc + 4 * i)); y = __ldg(src + 2 * (bc + 4 * i) + 1); }
      *reinterpret_cast<float4*>(v[i]) = x;
      *reinterpret_cast<float4*>(v[i] + 4) = y;
    }
  };
  fetch(0);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = s_tmem;
  // ---- token tile: thread = row, a quarter of the dims each
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const int c = 4 * wg + q;
    const float* src = reinterpret_cast<const float*>(s_b) + row * kUStride + 8 * c;
    float x[8];
    *reinterpret_cast<float4*>(x) = *reinterpret_cast<const float4*>(src);
    *reinterpret_cast<float4*>(x + 4) = *reinterpret_cast<const float4*>(src + 4);
    uint4 hi, lo;
    split_chunk(x, kTcScale, hi, lo);
    *reinterpret_cast<uint4*>(s_a + (c * kUpdTok + row) * 16) = hi;
    *reinterpret_cast<uint4*>(s_a + ((16 + c) * kUpdTok + row) * 16) = lo;
  }
  if (wg == 0) *reinterpret_cast<uint4*>(s_a + (32 * kUpdTok + row) * 16) = coarse_ext_row();
  if (wg == 1) *reinterpret_cast<uint4*>(s_a + (33 * kUpdTok + row) * 16) = make_uint4(0u, 0u, 0u, 0u);
  __syncthreads();                                          // the directions have been read

  // ---- nearest centroid: tile i + 1 is split and its MMAs issued before tile i is looked at
  auto put_tile = [&](int c0, unsigned char* dst) {
    float n2 = 0.f;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      uint4 hi, lo;
      split_chunk(v[i], -2.f * kTcScale, hi, lo);
#pragma unroll
      for (int t = 0; t < 8; ++t) n2 = fmaf(v[i][t], v[i][t], n2);
      *reinterpret_cast<uint4*>(dst + ((bc + 4 * i) * kUpdCen + br) * 16) = hi;
      *reinterpret_cast<uint4*>(dst + ((16 + bc + 4 * i) * kUpdCen + br) * 16) = lo;
    }
    n2 += __shfl_xor_sync(0xffffffffu, n2, 8);
    n2 += __shfl_xor_sync(0xffffffffu, n2, 16);
    if (bc == 0) *reinterpret_cast<uint4*>(dst + (32 * kUpdCen + br) * 16) = coarse_ext_centre(n2, c0 + br < pl.n_list);
    if (!(n2 < kTieRange)) s_wild = 1;                      // (the caller's centroids: any numbers)
    if (bc == 1) *reinterpret_cast<uint4*>(dst + (33 * kUpdCen + br) * 16) = make_uint4(0u, 0u, 0u, 0u);
  };
  const uint32_t my_lanes = (uint32_t)(wq * 32) << 16;      // this warp's TMEM lanes
  const int n_tiles = (pl.n_list + kUpdCen - 1) / kUpdCen;
  const TieLimit lim(s_x2[row]);
  Nearest2 nn;
  nn.clear();
  bool late = false;
  for (int i = -1; i < n_tiles; ++i) {
    if (i + 1 < n_tiles) {
      unsigned char* dst = s_b + ((i + 1) & 1) * kUpdB;
      put_tile((i + 1) * kUpdCen, dst);
      if (i + 2 < n_tiles) fetch((i + 2) * kUpdCen);
      tc_fence_smem();
      tc_fence_before();
      __syncthreads();
      if (tid == 0) {
        tc_fence_after();
        tc_coarse_tile<kUpdTok, kUpdCen>(tmem + ((i + 1) & 1) * kUpdCen, smem_u32(s_a), smem_u32(dst));
        tc_commit(&s_bar[(i + 1) & 1]);
      }
      __syncwarp();
    }
    if (i < 0) continue;
    late |= !tc_wait(&s_bar[i & 1], (uint32_t)(i >> 1) & 1u);
    tc_fence_after();
    float acc[32];
    tmem_ld32(tmem + (i & 1) * kUpdCen + 32 * wg + my_lanes, acc);
    nn.take(acc, i * (kUpdCen / 32) + wg, lim);
  }
  s_best[0][wg][row] = nn.best;
  s_best[1][wg][row] = nn.second;
  s_at[0][wg][row] = (uint16_t)nn.best_at;
  s_at[1][wg][row] = (uint16_t)nn.second_at;
  s_seen[wg][row] = nn.seen;
  s_blocks[wg][row] = (uint8_t)(min(nn.blocks, 3) | (nn.pair ? 128 : 0));
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  if (wg == 0) {
#pragma unroll
    for (int g = 1; g < kUpdGroups; ++g) {
      const float b = s_best[0][g][row];
      if (lim(b) <= nn.best) { nn.blocks = 0; nn.pair = false; }      // (as within a group)
      if (b < lim(nn.best)) {
        nn.blocks += s_blocks[g][row] & 127;
        nn.pair |= s_blocks[g][row] >> 7;
      }
      nn.merge(b, s_at[0][g][row]);
      nn.merge(s_best[1][g][row], s_at[1][g][row]);
    }
    const bool crowd = nn.crowded() || s_wild;
    s_near[row] = (uint16_t)min(nn.near(), pl.n_list - 1);
    s_tie[0][row] = (uint16_t)(nn.tie(lim) && !crowd ? nn.best_at : 0xffff);
    s_tie[1][row] = (uint16_t)(nn.second_near(lim) ? nn.second_at : nn.best_at);
    if (ok(row) && crowd) s_crowd[atomicAdd(&s_n_crowd, 1)] = (uint8_t)row;
  }
  __syncthreads();
  // ---- what fp32 decides: a few tokens in a hundred between the centroids of one or two blocks, by the
  // token's warp; hardly any between those of more blocks, by the whole CTA (over all 1024
  // centroids, 512 KB, one such token made an update of 80 us one of 86)
  float* s_u = reinterpret_cast<float*>(s_dyn);             // (the tiles are done)
#pragma unroll
  for (int r = 0; r < kPer; ++r) {
    float x[4];
    direction(r, x);
    *reinterpret_cast<float4*>(s_u + (r * kUpdWarps + warp) * kUStride + 4 * lane) = make_float4(x[0], x[1], x[2], x[3]);
  }
  const int n_crowd = s_n_crowd;
  if (n_crowd != 0) __syncthreads(); else __syncwarp();     // (uniform)
  const int n_search = n_crowd > kCrowd ? kCrowd : 1;       // for together
#pragma unroll 1
  for (int c = 0; c < n_crowd; c += n_search) {
    const uint32_t near_by = s_wild ? ~0u : s_seen[wq][s_crowd[c]];        // (warp w: block w % 4 of a tile)
    if (n_search == 1) nearest_of_all<false, 1>(s_u, kUStride, s_crowd, c, n_crowd, cbase, pl.n_list, tid, kUpdThreads, near_by, s_found[warp]);
    else nearest_of_all<false, kCrowd>(s_u, kUStride, s_crowd, c, n_crowd, cbase, pl.n_list, tid, kUpdThreads, ~0u, s_found[warp]);
    __syncthreads();
    if (tid < n_search && c + tid < n_crowd) {
      Found f = s_found[0][tid];
      for (int w = 1; w < kUpdWarps; ++w) nearer(f.d, f.at, s_found[w][tid].d, s_found[w][tid].at);
      s_near[s_crowd[c + tid]] = (uint16_t)f.at;
    }
    __syncthreads();
  }
  int list[kPer];
#pragma unroll
  for (int r = 0; r < kPer; ++r) {
    const int t = r * kUpdWarps + warp;
    list[r] = s_near[t];
    if (s_tie[0][t] != 0xffff && ok(t))                     // (warp-uniform)
      list[r] = nearest_of_blocks<false>(s_u + t * kUStride, cbase, pl.n_list, s_tie[0][t], s_tie[1][t]);
    if (lane == 0 && ok(t)) list_ids[ukv * pl.N_max + p0 + t] = (uint16_t)list[r];
  }
  __syncthreads();                                          // (the directions have been read)
  // ---- residuals
  {
    float4 c[kPer];
#pragma unroll
    for (int r = 0; r < kPer; ++r)
      c[r] = __ldg(reinterpret_cast<const float4*>(cbase + (size_t)list[r] * kHeadDim) + lane);
#pragma unroll
    for (int r = 0; r < kPer; ++r) {
      float x[4];
      direction(r, x);
      *reinterpret_cast<float4*>(s_u + (r * kUpdWarps + warp) * kUStride + 4 * lane) =
          make_float4(x[0] - c[r].x, x[1] - c[r].y, x[2] - c[r].z, x[3] - c[r].w);
    }
  }
  __syncthreads();

  // ---- codes: group <-> subspaces wg, wg + 4, ..; thread = token, and codeword while a tile is made
  using Tile = PqTile<DSUB>;
  const uint32_t d_tmem = tmem + (uint32_t)wg * 128u;       // this group's accumulator columns
  const uint32_t my_tmem = d_tmem + my_lanes;
  uint32_t parity = 0u;
  unsigned char* pa = s_dyn + kUpdU + wg * kUpdPq;
  unsigned char* pb = pa + Tile::kChunks * 2048;
  // the subspace's codewords in fp32 for the final decision, where they fit
  float* s_word = reinterpret_cast<float*>(pb + Tile::kChunks * 2048);
  const bool staged = 2 * Tile::kChunks * 2048 + pl.n_code * DSUB * 4 <= kUpdPq;
  const int words = min(kUpdWords, pl.n_code);
  float p[DSUB];                                            // this thread's codeword, one tile ahead
  auto fetch_word = [&](int m, int z0) {
    if (row < words && m < pl.M) load_sub<DSUB>(codebooks + ((ukv * pl.M + m) * (size_t)pl.n_code + z0 + row) * DSUB, p);
  };
      unsigned ties = 0u;                                       // bit i: this token's subspace wg + 4 i
  fetch_word(wg, 0);
  for (int m = wg; m < pl.M; m += kUpdGroups) {
    const float* cb = codebooks + (ukv * pl.M + m) * (size_t)pl.n_code * DSUB;
    float e[DSUB];
    load_sub<DSUB>(s_u + row * kUStride + m * DSUB, e);
    uint4 ch[Tile::kChunks];
    Tile::token_row(e, ch);
#pragma unroll
    for (int i = 0; i < Tile::kChunks; ++i) *reinterpret_cast<uint4*>(pa + (i * 128 + row) * 16) = ch[i];
    NearestGroup ng;
    ng.clear();
    for (int z0 = 0; z0 < pl.n_code; z0 += kUpdWords) {
      if (row < words) {
        if (!(Tile::code_row(p, ch) < kTieRange)) s_wild_words[wg] = m;      // (the caller's codebook: any numbers)
        if (staged) {
#pragma unroll
          for (int t = 0; t < DSUB; ++t) s_word[(z0 + row) * DSUB + t] = p[t];
        }
#pragma unroll
        for (int i = 0; i < Tile::kChunks; ++i) *reinterpret_cast<uint4*>(pb + (i * 128 + row) * 16) = ch[i];
      }
      tc_fence_smem();
      tc_fence_before();
      group_sync(1 + wg);
      if (row == 0) {
        tc_fence_after();
        Tile::template mma<128>(d_tmem, smem_u32(pa), smem_u32(pb), (uint32_t)words);
        tc_commit(&s_bar[2 + wg]);
      }
      if (z0 + kUpdWords < pl.n_code) fetch_word(m, z0 + kUpdWords);
      else fetch_word(m + kUpdGroups, 0);
      late |= !tc_wait(&s_bar[2 + wg], parity);
      parity ^= 1u;
      tc_fence_after();
      if (pl.n_code == 16) {
        float acc[16];
        tmem_ld16(my_tmem, acc);
        ng.take(acc, 0u);
      } else {
#pragma unroll
        for (int c = 0; c < kUpdWords; c += 32) {
          float acc[32];
          tmem_ld32(my_tmem + c, acc);
          ng.take(acc, (uint32_t)(z0 + c) / 8u);
        }
      }
    }
    // the winning group's codewords in fp32, first minimum.  The lanes start at different codewords:
    // at 16 bytes a codeword the eight lanes of an access then hit eight different bank groups
    float dm = CUDART_INF_F, e2 = 0.f;
    int bz = 0;
    auto decide = [&](const float* words_of_m) {
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        const int z = 8 * ng.group() + ((i + lane) & 7);
        const float dist = word_distance<DSUB>(e, words_of_m + z * DSUB);
        if (dist < dm || (dist == dm && z < bz)) { dm = dist; bz = z; }
      }
    };
    if (staged) decide(s_word); else decide(cb);
#pragma unroll
    for (int t = 0; t < DSUB; ++t) e2 = fmaf(e[t], e[t], e2);
    if (pq_tie(ng, e2) || !(e2 < kTieRange) || s_wild_words[wg] == m) ties |= 1u << (m / kUpdGroups);
    group_sync(1 + wg);                              // (the codewords are overwritten next)
    s_code[row][m] = (uint8_t)bz;
  }
  // where another group may hold a codeword as near: all of them
  if (__any_sync(0xffffffffu, ok(row) && ties != 0u)) {
    const UpdateSettle<DSUB> st = {s_u + (row & ~31) * kUStride + wg * DSUB,
                                   codebooks + (ukv * pl.M + wg) * (size_t)pl.n_code * DSUB,
                                   (size_t)kUpdGroups * pl.n_code * DSUB, s_code[row] + wg, 0ull};
    const unsigned mine = ok(row) ? ties : 0u;
    if (pl.n_code == 16) settle_codewords<DSUB, 16>(mine, pl.M / kUpdGroups, st);
    else settle_codewords<DSUB, 256>(mine, pl.M / kUpdGroups, st);
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 0) { tc_fence_after(); tmem_free(tmem, 512); }
  // a bounded wait ran out (no status word here): the tokens' norms say so
  if (late && ok(row)) key_norms[ukv * pl.N_max + p0 + row] = CUDART_NAN_F;
  // one byte per code, or two 4-bit codes per byte (subspace 2j in the low nibble of byte j)
  for (int i = tid; i < ntok * pl.code_bytes; i += kUpdThreads) {
    const int t = i / pl.code_bytes, j = i - t * pl.code_bytes;
    const int pos = p0 + t;
    const uint8_t byte = pl.n_code == 16 ? (uint8_t)(s_code[t][2 * j] | (s_code[t][2 * j + 1] << 4))
                                         : s_code[t][j];
    if (pos >= 0 && pos < pl.N_max) codes[(ukv * pl.N_max + pos) * pl.code_bytes + j] = byte;
  }
}

// The same for few tokens against few lists: 8 tokens per CTA, all of it in fp32.  Centroids pass through
// shared memory in tiles of 32 rows (a lane owns a centroid, a warp a token); for the codes a warp owns
// subspaces and a lane codewords, so a codebook row is read once for all 8 tokens.
constexpr int kFewTok = 8;              // tokens per CTA = warps per CTA
constexpr int kFewThreads = 32 * kFewTok;
constexpr int kFewCen = 32;             // centroid rows per tile

template <typename T, int DSUB>
__global__ void __launch_bounds__(kFewThreads)
index_encode_few_kernel(Plan pl, const T* __restrict__ kc, long long stride_page, long long stride_token,
                        long long stride_head, const int32_t* __restrict__ block_table,
                        const int32_t* __restrict__ first_pos, const int32_t* __restrict__ n_new,
                        int max_new, const float* __restrict__ centroids,
                        const float* __restrict__ codebooks, uint8_t* __restrict__ codes,
                        uint16_t* __restrict__ list_ids, float* __restrict__ key_norms) {
  __shared__ float s_u[kFewTok][kHeadDim];                  // direction, later the residual
  __shared__ float s_c[kFewCen][kHeadDim + 1];              // (padded: lane j reads row j without conflicts)
  __shared__ uint8_t s_code[kFewTok][64];
  const int kv = blockIdx.y, b = blockIdx.z;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const size_t ukv = (size_t)b * pl.Hkv + kv;
  pdl_wait();
  pdl_launch_dependents();
  const int nb = min(max(n_new[b], 0), max_new);
  const int t0 = blockIdx.x * kFewTok;
  if (t0 >= nb) return;
  const int ntok = min(kFewTok, nb - t0);
  const int p0 = first_pos[b] + t0;                 // position of this CTA's first token
  const int32_t* bt = block_table + (size_t)b * pl.max_pages;
  // tokens whose position falls outside the index rows are left alone
  const bool mine_ok = warp < ntok && p0 + warp >= 0 && p0 + warp < pl.N_max;
  // ---- norm and direction: warp w <-> token w, a lane holds 4 of the 128 dims
  {
    float x[4] = {0.f, 0.f, 0.f, 0.f};
    if (mine_ok) load4<T>(kc + row_offset(pl, bt, p0 + warp, kv, stride_page, stride_token, stride_head) + 4 * lane, x);
    const float ss = warp_sum(x[0] * x[0] + x[1] * x[1] + x[2] * x[2] + x[3] * x[3]);
    const float r = sqrtf(ss);
    const float inv = r > 0.f ? 1.f / r : 0.f;
#pragma unroll
    for (int i = 0; i < 4; ++i) s_u[warp][4 * lane + i] = x[i] * inv;
    if (mine_ok && lane == 0) key_norms[ukv * pl.N_max + p0 + warp] = r;
  }
  // ---- nearest centroid: |u - c|^2 = |u|^2 - 2 u.c + |c|^2, the first term is common
  float best_d = CUDART_INF_F;
  int best_j = 0;
  const float* cbase = centroids + ukv * (size_t)pl.n_list * kHeadDim;
  for (int c0 = 0; c0 < pl.n_list; c0 += kFewCen) {
    __syncthreads();                                // previous tile consumed, s_u complete
    for (int i = tid; i < kFewCen * (kHeadDim / 4); i += kFewThreads) {
      const int rr = i / (kHeadDim / 4), c4 = i % (kHeadDim / 4);
      float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
      if (c0 + rr < pl.n_list) v = __ldg(reinterpret_cast<const float4*>(cbase + (size_t)(c0 + rr) * kHeadDim) + c4);
      s_c[rr][4 * c4] = v.x; s_c[rr][4 * c4 + 1] = v.y;
      s_c[rr][4 * c4 + 2] = v.z; s_c[rr][4 * c4 + 3] = v.w;
    }
    __syncthreads();
    float dot = 0.f, cn = 0.f;
#pragma unroll 8
    for (int d = 0; d < kHeadDim; ++d) {
      const float c = s_c[lane][d];
      dot = fmaf(s_u[warp][d], c, dot);
      cn = fmaf(c, c, cn);
    }
    const float dist = fmaf(-2.f, dot, cn);
    if (c0 + lane < pl.n_list && dist < best_d) { best_d = dist; best_j = c0 + lane; }
  }
  warp_nearest(best_d, best_j);
  if (mine_ok && lane == 0) list_ids[ukv * pl.N_max + p0 + warp] = (uint16_t)best_j;
  // ---- residual, in place
  {
    const float4 c = __ldg(reinterpret_cast<const float4*>(cbase + (size_t)best_j * kHeadDim) + lane);
    s_u[warp][4 * lane] -= c.x; s_u[warp][4 * lane + 1] -= c.y;
    s_u[warp][4 * lane + 2] -= c.z; s_u[warp][4 * lane + 3] -= c.w;
  }
  __syncthreads();
  // ---- codes: warp <-> subspaces m = warp, warp + 8, ...; lane <-> codewords lane + 32 i
  for (int m = warp; m < pl.M; m += kFewTok) {
    float bd[kFewTok];
    int bz[kFewTok];
#pragma unroll
    for (int t = 0; t < kFewTok; ++t) { bd[t] = CUDART_INF_F; bz[t] = 0; }
    const float* cb = codebooks + (ukv * pl.M + m) * (size_t)pl.n_code * DSUB;
    for (int z0 = 0; z0 < pl.n_code; z0 += 32) {
      const int z = min(z0 + lane, pl.n_code - 1);      // lanes past the codebook repeat its last word
      float p[DSUB];
      if constexpr (DSUB == 2) {
        const float2 v = __ldg(reinterpret_cast<const float2*>(cb + (size_t)z * DSUB));
        p[0] = v.x; p[1] = v.y;
      } else {
#pragma unroll
        for (int c4 = 0; c4 < DSUB / 4; ++c4) {
          const float4 v = __ldg(reinterpret_cast<const float4*>(cb + (size_t)z * DSUB) + c4);
          p[4 * c4] = v.x; p[4 * c4 + 1] = v.y; p[4 * c4 + 2] = v.z; p[4 * c4 + 3] = v.w;
        }
      }
#pragma unroll
      for (int t = 0; t < kFewTok; ++t) {
        float dist = 0.f;
#pragma unroll
        for (int dd = 0; dd < DSUB; ++dd) {
          const float e = s_u[t][m * DSUB + dd] - p[dd];
          dist = fmaf(e, e, dist);
        }
        if (dist < bd[t]) { bd[t] = dist; bz[t] = z; }      // z ascends: first minimum stays
      }
    }
#pragma unroll
    for (int t = 0; t < kFewTok; ++t) {
      warp_nearest(bd[t], bz[t]);
      if (lane == 0) s_code[t][m] = (uint8_t)bz[t];
    }
  }
  __syncthreads();
  for (int i = tid; i < ntok * pl.code_bytes; i += kFewThreads) {
    const int t = i / pl.code_bytes, j = i - t * pl.code_bytes;
    const int pos = p0 + t;
    const uint8_t byte = pl.n_code == 16 ? (uint8_t)(s_code[t][2 * j] | (s_code[t][2 * j + 1] << 4))
                                         : s_code[t][j];
    if (pos >= 0 && pos < pl.N_max) codes[(ukv * pl.N_max + pos) * pl.code_bytes + j] = byte;
  }
}

template <typename T>
__global__ void __launch_bounds__(kMeanThreads)
index_refresh_means_kernel(Plan pl, const T* __restrict__ vc, long long stride_page,
                           long long stride_token, long long stride_head,
                           const int32_t* __restrict__ block_table,
                           const int32_t* __restrict__ first_pos, const int32_t* __restrict__ n_new,
                           int max_new, const uint16_t* __restrict__ list_ids,
                           float* __restrict__ list_vmeans, int32_t* __restrict__ list_counts, int early) {
  extern __shared__ int s_first[];                   // [n_list] first new token of every list
  __shared__ uint16_t s_lid[kMaxNew];
  const int kv = blockIdx.y, b = blockIdx.z;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const size_t ukv = (size_t)b * pl.Hkv + kv;
  for (int j = tid; j < pl.n_list; j += kMeanThreads) s_first[j] = kMaxNew;
  const int p0 = first_pos[b];
  int nb = min(max(n_new[b], 0), max_new);
  if (p0 < 0) nb = 0;
  nb = min(nb, pl.N_max - p0);                       // same positions as the encode kernel
  const int t_begin = blockIdx.x * kMeanTok, t_end = min(nb, t_begin + kMeanTok);
  pdl_wait();                                        // the list ids come from the encode kernel
  // (not beside the small encode kernel of a next call: between these CTAs its own land unevenly, 50 -> 70 us
  // at 256 units x 512 lists)
  if (early) pdl_launch_dependents();
  if (t_begin >= nb) return;
  const int32_t* bt = block_table + (size_t)b * pl.max_pages;
  __syncthreads();
  for (int t = tid; t < nb; t += kMeanThreads) {
    const uint16_t j = (uint16_t)min((int)list_ids[ukv * pl.N_max + p0 + t], pl.n_list - 1);
    s_lid[t] = j;
    atomicMin(&s_first[j], t);
  }
  __syncthreads();
  for (int t1 = t_begin + warp; t1 < t_end; t1 += kMeanThreads / 32) {
    const int j = s_lid[t1];
    if (s_first[j] != t1) continue;                  // not a leader (warp-uniform)
    float4* mean = reinterpret_cast<float4*>(list_vmeans + (ukv * pl.n_list + j) * kHeadDim) + lane;
    float4 v = *mean;
    const int n_old = list_counts[ukv * pl.n_list + j];
    float4 sum = make_float4(0.f, 0.f, 0.f, 0.f);
    int cnt = 0;
    for (int base = t1; base < nb; base += 32) {     // token order: the sum is deterministic
      unsigned hit = __ballot_sync(0xffffffffu, base + lane < nb && s_lid[min(base + lane, nb - 1)] == j);
      while (hit) {
        const int t = base + __ffs(hit) - 1;
        hit &= hit - 1u;
        const T* src = vc + row_offset(pl, bt, p0 + t, kv, stride_page, stride_token, stride_head);
        float x[4];
        load4<T>(src + 4 * lane, x);
        sum.x += x[0]; sum.y += x[1]; sum.z += x[2]; sum.w += x[3];
        ++cnt;
      }
    }
    const float w_old = (float)n_old, inv = 1.f / (float)(n_old + cnt);
    v.x = (w_old * v.x + sum.x) * inv; v.y = (w_old * v.y + sum.y) * inv;
    v.z = (w_old * v.z + sum.z) * inv; v.w = (w_old * v.w + sum.w) * inv;
    *mean = v;
    __syncwarp();
    if (lane == 0) list_counts[ukv * pl.n_list + j] = n_old + cnt;
  }
}

// Which of the two encodes.  Both times fitted, in us of a whole call: a fixed part, the codes, a part that
// grows with the lists, and the CTAs per SM.  Measured, fp32 kernel / tensor cores, 32 one-byte codes: one
// unit, 8 tokens, 16 lists 17 / 37, 128 23 / 38, 384 39 / 45, 512 47 / 47, 1024 78 / 59; 64 units x 32
// tokens, 16 lists 36 / 45, 128 44 / 44, 384 52 / 50.  Eight 4-bit codes: 64 units x 64 tokens, 16 lists
// 23 / 37, 64 27 / 37; 256 units x 16 tokens, 128 lists 36 / 57, 256 52 / 64.
bool few_tokens(const Plan& pl, int max_new) {
  const int units = pl.B * pl.Hkv;
  auto ctas = [&](int tokens) { return units * ((max_new + tokens - 1) / tokens); };
  const bool bytes = pl.n_code == 256;
  const float codes_few = !bytes ? 2.f : pl.M == 8 ? 5.f : pl.M == 16 ? 8.f : pl.M == 32 ? 11.f : 19.f;
  const float codes_tc = !bytes ? 2.f : pl.M == 8 ? 8.f : pl.M == 16 ? 6.f : pl.M == 32 ? 12.f : 31.f;
  const float r = (float)ctas(kFewTok) / (float)pl.num_sms;
  const float few = (8.f + codes_few) * (r > 1.f ? 0.6f + 0.4f * r : 1.f) + 0.061f * pl.n_list * (r > 1.25f ? 0.8f * r : 1.f);
  const int waves = (ctas(kUpdTok) + pl.num_sms - 1) / pl.num_sms;
  return few < (24.f + codes_tc + 0.022f * pl.n_list) * waves;
}

template <typename T>
cudaError_t launch_update_t(const Plan& pl, const pqhsa_index_rw& ix, const pqhsa_paged_kv& kv,
                            const int32_t* first_pos, const int32_t* n_new, int max_new,
                            cudaStream_t st) {
  const T* kc = static_cast<const T*>(kv.k_cache);
  const T* vc = static_cast<const T*>(kv.v_cache);
  const bool few = few_tokens(pl, max_new);
  const int per_cta = few ? kFewTok : kUpdTok;
  const dim3 grid((max_new + per_cta - 1) / per_cta, pl.Hkv, pl.B);
  cudaError_t e;
  auto encode = [&](auto kernel, int threads, size_t smem) {
    return launch_pdl(kernel, grid, dim3(threads), smem, st, pl, kc, (long long)kv.stride_page,
                      (long long)kv.stride_token, (long long)kv.stride_head, kv.block_table, first_pos, n_new,
                      max_new, ix.centroids, ix.codebooks, ix.codes, ix.list_ids, ix.key_norms);
  };
#define PQHSA_UPD_CASE(D)                                                                       \
  case D:                                                                                       \
    if (few) {                                                                                  \
      e = encode(index_encode_few_kernel<T, D>, kFewThreads, 0);                                \
      break;                                                                                    \
    }                                                                                           \
    e = cudaFuncSetAttribute(index_encode_kernel<T, D>,                                         \
                             cudaFuncAttributeMaxDynamicSharedMemorySize, kUpdSmem);            \
    if (e != cudaSuccess) return e;                                                             \
    e = encode(index_encode_kernel<T, D>, kUpdThreads, kUpdSmem);                               \
    break;
  switch (pl.dsub) {
    PQHSA_UPD_CASE(2) PQHSA_UPD_CASE(4) PQHSA_UPD_CASE(8) PQHSA_UPD_CASE(16)
    default: return cudaErrorInvalidValue;
  }
#undef PQHSA_UPD_CASE
  if (e != cudaSuccess) return e;
  return launch_pdl(index_refresh_means_kernel<T>, dim3((max_new + kMeanTok - 1) / kMeanTok, pl.Hkv, pl.B),
                    dim3(kMeanThreads), (size_t)pl.n_list * 4, st, pl, vc,
                    (long long)kv.stride_page, (long long)kv.stride_token,
                    (long long)kv.stride_head, kv.block_table, first_pos, n_new, max_new,
                    static_cast<const uint16_t*>(ix.list_ids), ix.list_vmeans, ix.list_counts, few ? 0 : 1);
}

}  // namespace
}  // namespace pqhsa

using namespace pqhsa;

extern "C" int pqhsa_index_update(const pqhsa_params* params, const pqhsa_index_rw* index,
                                  const pqhsa_paged_kv* kv, const int32_t* first_pos,
                                  const int32_t* n_new, int32_t max_new, void* stream) {
  Plan pl;
  int rc = make_plan(params, &pl);
  if (rc != PQHSA_OK) return rc;
  if (index == nullptr || kv == nullptr || first_pos == nullptr || n_new == nullptr ||
      index->centroids == nullptr || index->codebooks == nullptr || index->codes == nullptr ||
      index->list_ids == nullptr || index->key_norms == nullptr || index->list_vmeans == nullptr ||
      index->list_counts == nullptr || kv->k_cache == nullptr || kv->v_cache == nullptr ||
      kv->block_table == nullptr || max_new < 0 || max_new > kMaxNew)
    return PQHSA_ERR_INVALID_ARG;
  if (kv->stride_page % 8 || kv->stride_token % 8 || kv->stride_head % 8) return PQHSA_ERR_UNSUPPORTED;
  if (max_new == 0) return PQHSA_OK;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  const cudaError_t e =
      pl.dtype == PQHSA_F16
          ? launch_update_t<__half>(pl, *index, *kv, first_pos, n_new, max_new, st)
          : launch_update_t<__nv_bfloat16>(pl, *index, *kv, first_pos, n_new, max_new, st);
  return e == cudaSuccess ? PQHSA_OK : PQHSA_ERR_CUDA;
}
