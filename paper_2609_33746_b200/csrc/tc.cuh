// Fifth-generation tensor core blocks (tcgen05, accumulators in TMEM) for the nearest-centre
// searches of the index: fp16 operands split in two, fp32 accumulation.
//
// A nearest-centre search needs argmin_c (|c|^2 - 2 x.c) with fp32-grade products.  Every fp32
// factor is split as hi + lo in fp16 (22 bits together; scaled by 2^8 so that lo keeps an absolute
// resolution of 2^-32), and x.c is taken as hi.hi + hi.lo + lo.hi, the dropped lo.lo term being
// 2^-22 of the product.  The centre side carries the factor -2, and |c|^2 rides along as three more
// fp16 terms against the constant 256, so the accumulator holds 2^16 (|c|^2 - 2 x.c) itself.
//
// Operand tiles in shared memory use the K-major layout without swizzle: 8 x 16-byte core matrices;
// 8 consecutive k of all R rows form one block ("chunk") of R * 16 bytes, row r at r * 16, so that
// threads that own rows store 16 bytes each without bank conflicts.
#pragma once

#include "common.cuh"
#include "scan_common.cuh"

namespace pqhsa {
namespace {

constexpr float kTcScale = 256.f;              // 2^8 on each side of a product
constexpr float kTcUnscale = 1.f / (kTcScale * kTcScale);
constexpr float kTcFar = 60000.f;              // |c|^2 term of a padding row: farther than any centre

// ---- descriptors (PTX ISA, tcgen05 matrix and instruction descriptors)
// K-major, no swizzle: chunk stride (between core matrices along k) and 8-row stride, in bytes.
__device__ __forceinline__ uint64_t tc_desc(uint32_t saddr, uint32_t chunk_stride) {
  return (uint64_t)((saddr & 0x3ffffu) >> 4) | ((uint64_t)(chunk_stride >> 4) << 16) |
         ((uint64_t)(128u >> 4) << 32) | (1ull << 46);
}
// fp16 x fp16 -> fp32, both K-major, M = 128
__device__ __forceinline__ constexpr uint32_t tc_idesc(uint32_t n) {
  return (1u << 4) | ((n >> 3) << 17) | ((128u >> 4) << 24);
}
// D[tmem] (+)= A B^T for one K = 16 step; one thread
__device__ __forceinline__ void tc_mma(uint32_t d, uint64_t a, uint64_t b, uint32_t idesc, bool accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}"
      ::"r"(d), "l"(a), "l"(b), "r"(idesc), "r"(accumulate ? 1u : 0u) : "memory");
}
// the mbarrier gets one arrival when all MMAs issued by this thread so far are complete
__device__ __forceinline__ void tc_commit(uint64_t* bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];"
               ::"r"(smem_u32(bar)) : "memory");
}
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
// generic shared-memory stores become visible to the tensor core
__device__ __forceinline__ void tc_fence_smem() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }

// one whole warp; the address lands in *slot.  n_cols: power of two, 32 .. 512
__device__ __forceinline__ void tmem_alloc(uint32_t* slot, uint32_t n_cols) {
  asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(slot)), "r"(n_cols) : "memory");
  asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
}
__device__ __forceinline__ void tmem_free(uint32_t addr, uint32_t n_cols) {
  asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(addr), "r"(n_cols));
}
// 32 (16) consecutive columns of this thread's TMEM lane (lane = row of the tile); whole warp
__device__ __forceinline__ void tmem_ld32(uint32_t addr, float (&v)[32]) {
  uint32_t r[32];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
      "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
        "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]),
        "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]),
        "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
      : "r"(addr));
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
  for (int i = 0; i < 32; ++i) v[i] = __uint_as_float(r[i]);
}
__device__ __forceinline__ void tmem_ld16(uint32_t addr, float (&v)[16]) {
  uint32_t r[16];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
        "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
      : "r"(addr));
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
  for (int i = 0; i < 16; ++i) v[i] = __uint_as_float(r[i]);
}
__device__ __forceinline__ void group_sync(int id) {      // the 128 threads of a warpgroup
  asm volatile("bar.sync %0, 128;" ::"r"(id) : "memory");
}

// bounded wait for a commit (see mbar_wait; an MMA takes microseconds at most)
__device__ __forceinline__ bool tc_wait(uint64_t* bar, uint32_t parity) {
  for (int it = 0; it < (1 << 16); ++it) {
    uint32_t done;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(done) : "r"(smem_u32(bar)), "r"(parity) : "memory");
    if (done) return true;
  }
  return false;
}

// ---- fp16 split.  Always two values at a time: the packed conversion runs on the integer pipe, the
// single one on the transcendental unit at an eighth of the rate.
__device__ __forceinline__ uint32_t bits16(__half2 h) { return *reinterpret_cast<const uint32_t*>(&h); }
__device__ __forceinline__ void split2(float a, float b, uint32_t& hi, uint32_t& lo) {
  const __half2 h = __floats2half2_rn(a, b);
  const float2 f = __half22float2(h);
  hi = bits16(h);
  lo = bits16(__floats2half2_rn(a - f.x, b - f.y));
}
// 8 values, scaled, as a chunk of hi and a chunk of lo
__device__ __forceinline__ void split_chunk(const float (&v)[8], float scale, uint4& hi, uint4& lo) {
  split2(scale * v[0], scale * v[1], hi.x, lo.x);
  split2(scale * v[2], scale * v[3], hi.y, lo.y);
  split2(scale * v[4], scale * v[5], hi.z, lo.z);
  split2(scale * v[6], scale * v[7], hi.w, lo.w);
}
// |c|^2 as three fp16 terms (33 bits) against the constant 256 on the other side: the first two in
// one word, the third in the low half of the next
__device__ __forceinline__ void split_norm(float n2, uint32_t& w0, uint32_t& w1) {
  const float v = kTcScale * n2;
  const float r1 = v - __low2float(__floats2half2_rn(v, 0.f));
  const __half2 h = __floats2half2_rn(v, r1);
  w0 = bits16(h);
  w1 = bits16(__floats2half2_rn(r1 - __high2float(h), 0.f));
}

// ---- coarse search: 128-dim rows; chunks 0-15 hi, 16-31 lo, 32 the |c|^2 terms, 33 zero
constexpr int kCoarseChunks = 34;
// The 25 K-steps of one tile (the cross terms first: they are 2^-11 of the rest, so that only nine
// accumulations round at full magnitude).  Unrolled over constant descriptor offsets: an MMA then
// costs its 64 clocks at 128 x 128; with descriptors formed in a loop the issue alone took 148.
template <uint32_t kRowsA, uint32_t kRowsB>
__device__ __forceinline__ void tc_coarse_tile(uint32_t d, uint32_t sa, uint32_t sb) {
  constexpr uint32_t idesc = tc_idesc(kRowsB);
  const uint64_t a = tc_desc(sa, kRowsA * 16u), b = tc_desc(sb, kRowsB * 16u);
#pragma unroll
  for (uint32_t s = 0; s < 16; s += 2) {
    tc_mma(d, a + s * kRowsA, b + (16u + s) * kRowsB, idesc, s != 0);     // (offsets in 16-byte units)
    tc_mma(d, a + (16u + s) * kRowsA, b + s * kRowsB, idesc, true);
  }
#pragma unroll
  for (uint32_t s = 0; s < 16; s += 2) tc_mma(d, a + s * kRowsA, b + s * kRowsB, idesc, true);
  tc_mma(d, a + 32u * kRowsA, b + 32u * kRowsB, idesc, true);
}
__device__ __forceinline__ uint4 coarse_ext_row() {       // the row side of chunk 32
  return make_uint4(bits16(__floats2half2_rn(kTcScale, kTcScale)), bits16(__floats2half2_rn(kTcScale, 0.f)), 0u, 0u);
}
__device__ __forceinline__ uint4 coarse_ext_centre(float n2, bool real) {
  uint32_t w0, w1;
  split_norm(n2, w0, w1);
  return real ? make_uint4(w0, w1, 0u, 0u) : make_uint4(bits16(__floats2half2_rn(kTcFar, 0.f)), 0u, 0u, 0u);
}

// ---- codeword search: DSUB dims; one row is [hi | hi | lo | 256 256 256 | 0 ..] on the token side
// and [hi | lo | hi | |p|^2 terms | 0 ..] on the codeword side, K padded to 16
template <int DSUB> struct PqTile {
  static constexpr int kK = (3 * DSUB + 3 + 15) / 16 * 16;
  static constexpr int kChunks = kK / 8;
  // (DSUB is even, so whole words of two: DSUB / 2 words per copy, the norm's words behind them)
  static __device__ __forceinline__ void token_row(const float (&e)[DSUB], uint4 (&c)[kChunks]) {
    uint32_t w[kK / 2];
#pragma unroll
    for (int i = 0; i < kK / 2; ++i) w[i] = 0u;
#pragma unroll
    for (int t = 0; t < DSUB / 2; ++t) {
      split2(kTcScale * e[2 * t], kTcScale * e[2 * t + 1], w[t], w[DSUB + t]);
      w[DSUB / 2 + t] = w[t];
    }
    w[3 * DSUB / 2] = bits16(__floats2half2_rn(kTcScale, kTcScale));
    w[3 * DSUB / 2 + 1] = bits16(__floats2half2_rn(kTcScale, 0.f));
    pack(w, c);
  }
  // (returns |p|^2)
  static __device__ __forceinline__ float code_row(const float (&p)[DSUB], uint4 (&c)[kChunks]) {
    uint32_t w[kK / 2];
#pragma unroll
    for (int i = 0; i < kK / 2; ++i) w[i] = 0u;
    float n2 = 0.f;
#pragma unroll
    for (int t = 0; t < DSUB / 2; ++t) {
      split2(-2.f * kTcScale * p[2 * t], -2.f * kTcScale * p[2 * t + 1], w[t], w[DSUB / 2 + t]);
      w[DSUB + t] = w[t];
    }
#pragma unroll
    for (int t = 0; t < DSUB; ++t) n2 = fmaf(p[t], p[t], n2);
    split_norm(n2, w[3 * DSUB / 2], w[3 * DSUB / 2 + 1]);
    pack(w, c);
    return n2;
  }
  static __device__ __forceinline__ void pack(const uint32_t (&w)[kK / 2], uint4 (&c)[kChunks]) {
#pragma unroll
    for (int i = 0; i < kChunks; ++i) c[i] = make_uint4(w[4 * i], w[4 * i + 1], w[4 * i + 2], w[4 * i + 3]);
  }
  // 128 tokens x n codewords (chunks of kRowsB rows)
  template <uint32_t kRowsB>
  static __device__ __forceinline__ void mma(uint32_t d, uint32_t sa, uint32_t sb, uint32_t n) {
    const uint64_t a = tc_desc(sa, 128u * 16u), b = tc_desc(sb, kRowsB * 16u);
    const uint32_t idesc = tc_idesc(n);
#pragma unroll
    for (uint32_t s = 0; s < kChunks; s += 2) tc_mma(d, a + s * 128u, b + s * kRowsB, idesc, s != 0);
  }
};

__device__ __forceinline__ float min3(float a, float b, float c) {      // one instruction
  float d;
  asm("min.f32 %0, %1, %2, %3;" : "=f"(d) : "f"(a), "f"(b), "f"(c));
  return d;
}
__device__ __forceinline__ float min32(const float (&v)[32]) {
  float m[11];
#pragma unroll
  for (int i = 0; i < 10; ++i) m[i] = min3(v[3 * i], v[3 * i + 1], v[3 * i + 2]);
  m[10] = fminf(v[30], v[31]);
  const float a = min3(m[0], m[1], m[2]), b = min3(m[3], m[4], m[5]), c = min3(m[6], m[7], m[8]);
  return min3(min3(a, b, c), m[9], m[10]);
}

// ---- When is the smallest accumulator the nearest centre?  The split arithmetic and fp32 each round, so
// a search is trusted only where no other centre comes within the sum of both errors of the smallest;
// everything else is decided in plain fp32, every sum one chain over the dims, lower index on ties.
// The result is then that of an fp32 search over all centres, whatever the split.
//
// For a row x and a centre at distance d, |centre| <= |x| + d: the partial sums are of the size of |x|^2
// and of the accumulated value v = d^2 - |x|^2.  The errors, per unit of those: nine accumulations at
// full magnitude, truncated (4e-6 of the squared distance of unit vectors, the largest error
// seen); the column's bits in the mantissa (2^-18 of |v| for each of the two compared); the fp32 chain.
// kTieFloor: the fp16 terms have an absolute resolution of 2^-32.  Beyond kTieRange (|.|^2 of a row or
// centre) they could overflow: fp32 decides.
constexpr float kTieX2 = 6e-6f, kTieV = 8e-6f;
constexpr float kTieFloor = kTcScale * kTcScale / 536870912.f;      // 2^-29
constexpr float kTieRange = 100.f;
struct TieLimit {
  float k0;
  __device__ __forceinline__ explicit TieLimit(float x2) : k0(fmaf(kTieX2 * kTcScale * kTcScale, x2, kTieFloor)) {}
  // values below this may be as near as the one that gave `low`
  __device__ __forceinline__ float operator()(float low) const { return low + fmaf(kTieV, fabsf(low), k0); }
};

// The nearest centroids of a token, a block of 32 accumulators at a time.  Their column's low 5 bits
// travel in the mantissa, so that a column costs 4 instructions (an index carried beside each value: 7 to
// 8), and only where the 32 hold something near enough to matter.  What is kept: the nearest of the two
// best blocks, and how many blocks hold a centroid within reach of the nearest, or one of them two.
// One or two such blocks are searched in fp32 by the caller, more of them (crowded) mean a search over all.
constexpr uint32_t kColBits = 31u;
struct Nearest2 {
  float low, best, second;                               // exact minimum; with column bits
  int best_at, second_at;                                // which 32 columns
  int blocks;                                            // within reach of `low` (at most so many)
  bool pair;                                             // two in one block
  uint32_t seen;                                         // the blocks counted, a bit for each four (at / 4)
  __device__ __forceinline__ void clear() {
    low = best = second = CUDART_INF_F;
    best_at = second_at = blocks = 0;
    seen = 0u;
    pair = false;
  }
  // (column bits: the value's own, or infinity's zeros)
  __device__ __forceinline__ int near() const { return best_at * 32 + (int)(__float_as_uint(best) & kColBits); }
  __device__ __forceinline__ bool second_near(const TieLimit& lim) const { return second < lim(best); }
  __device__ __forceinline__ bool tie(const TieLimit& lim) const { return pair || second_near(lim); }
  __device__ __forceinline__ bool crowded() const { return blocks > 2; }
  // the best of another block
  __device__ __forceinline__ void merge(float b, int b_at) {
    const bool first = b < best;
    const float other = fmaxf(best, b);
    const int other_at = first ? best_at : b_at;
    if (other < second) { second = other; second_at = other_at; }
    if (first) { best = b; best_at = b_at; }
  }
  __device__ __forceinline__ void take(const float (&acc)[32], int at, const TieLimit& lim) {
    const float m = min32(acc);
    if (m < lim(low)) {
      if (lim(m) <= low) { blocks = 0; pair = false; seen = 0u; }      // all that came before is out of reach
      low = fminf(low, m);
      float b2[16], s2[16];
#pragma unroll
      for (int j = 0; j < 16; ++j) {
        const float x = __uint_as_float((__float_as_uint(acc[2 * j]) & ~kColBits) | (2 * j));
        const float y = __uint_as_float((__float_as_uint(acc[2 * j + 1]) & ~kColBits) | (2 * j + 1));
        b2[j] = fminf(x, y);
        s2[j] = fmaxf(x, y);
      }
#pragma unroll
      for (int o = 8; o > 0; o >>= 1) {
#pragma unroll
        for (int j = 0; j < o; ++j) {
          s2[j] = min3(s2[j], s2[j + o], fmaxf(b2[j], b2[j + o]));
          b2[j] = fminf(b2[j], b2[j + o]);
        }
      }
      ++blocks;
      seen |= 1u << (at >> 2);
      pair |= s2[0] < lim(low);
      merge(b2[0], at);
    }
  }
};

// Squared distances of kT rows and a centroid in fp32, every sum one chain over the dims, up to |x|^2
// where kX2 is false.
template <bool kX2, int kT, class Row>
__device__ __forceinline__ void distances_fp32(Row row, const float* __restrict__ c, float (&d)[kT]) {
  const float4* cp = reinterpret_cast<const float4*>(c);
  float xx[kT], a[kT], n = 0.f;
#pragma unroll
  for (int t = 0; t < kT; ++t) xx[t] = a[t] = 0.f;
#pragma unroll(kT == 1 ? 16 : 8)
  for (int k = 0; k < kHeadDim / 4; ++k) {
    const float4 y = __ldg(cp + k);
    n = fmaf(y.x, y.x, n); n = fmaf(y.y, y.y, n); n = fmaf(y.z, y.z, n); n = fmaf(y.w, y.w, n);
#pragma unroll
    for (int t = 0; t < kT; ++t) {
      const float4 u = reinterpret_cast<const float4*>(row(t))[k];
      a[t] = fmaf(u.x, y.x, a[t]); a[t] = fmaf(u.y, y.y, a[t]); a[t] = fmaf(u.z, y.z, a[t]); a[t] = fmaf(u.w, y.w, a[t]);
      if constexpr (kX2) {
        xx[t] = fmaf(u.x, u.x, xx[t]); xx[t] = fmaf(u.y, u.y, xx[t]); xx[t] = fmaf(u.z, u.z, xx[t]); xx[t] = fmaf(u.w, u.w, xx[t]);
      }
    }
  }
#pragma unroll
  for (int t = 0; t < kT; ++t) d[t] = kX2 ? (xx[t] - 2.0f * a[t]) + n : fmaf(-2.f, a[t], n);
}
template <bool kX2> __device__ __forceinline__ float distance_fp32(const float* x, const float* __restrict__ c) {
  float d[1];
  distances_fp32<kX2, 1>([&](int) { return x; }, c, d);
  return d[0];
}
// the smaller of two (distance, index), the lower index on ties
__device__ __forceinline__ void nearer(float& d, int& at, float od, int oat) {
  if (od < d || (od == d && oat < at)) { d = od; at = oat; }
}
__device__ __forceinline__ void warp_nearest(float& d, int& at) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const float od = __shfl_xor_sync(0xffffffffu, d, o);
    const int oat = __shfl_xor_sync(0xffffffffu, at, o);
    nearer(d, at, od, oat);
  }
}

// The nearest centroid of a row among those of up to two blocks of 32, by a warp.  (A call: rare, and long
// where it would stand.)
template <bool kX2>
__device__ __noinline__ int nearest_of_blocks(const float* x, const float* __restrict__ centroids, int n_list, int block0, int block1) {
  float d = CUDART_INF_F;
  int at = 0;
#pragma unroll 1
  for (int blk = block0;; blk = block1) {
    const int j = 32 * blk + (threadIdx.x & 31);
    if (j < n_list) nearer(d, at, distance_fp32<kX2>(x, centroids + (size_t)j * kHeadDim), j);
    if (blk == block1) break;
  }
  warp_nearest(d, at);
  return at;
}
// ... of kT rows (index[c], index[c + 1], .., at most n of them) among all centroids, by the threads first,
// first + step, .. (step a multiple of 128); leaves each warp's result at found[0 .. kT).  (One row: the
// loads run ahead of the chains; four share every centroid's load, for data where all is equally near.)
// near_by: bit i tells whether the row's block of 32 centroids at the thread's place of every 128 has to be
// looked at in the i-th 128.
struct Found {
  float d;
  int at;
};
template <bool kX2, int kT>
__device__ __noinline__ void nearest_of_all(const float* rows, int stride, const uint8_t* index, int c, int n,
                                            const float* __restrict__ centroids, int n_list, int first, int step, uint32_t near_by,
                                            Found* found) {
  const float* row[kT];
  float d[kT];
  int at[kT];
#pragma unroll
  for (int t = 0; t < kT; ++t) {
    row[t] = rows + (int)index[min(c + t, n - 1)] * stride;
    d[t] = CUDART_INF_F;
    at[t] = 0;
  }
#pragma unroll 1
  for (int j = first; j < n_list; j += step) {
    if (!((near_by >> (j >> 7)) & 1u)) continue;          // (warp-uniform)
    float dist[kT];
    distances_fp32<kX2, kT>([&](int t) { return row[t]; }, centroids + (size_t)j * kHeadDim, dist);
#pragma unroll
    for (int t = 0; t < kT; ++t) nearer(d[t], at[t], dist[t], j);
  }
#pragma unroll
  for (int t = 0; t < kT; ++t) {
    warp_nearest(d[t], at[t]);
    if ((threadIdx.x & 31) == 0) { found[t].d = d[t]; found[t].at = at[t]; }
  }
}
constexpr int kCrowd = 4;                                  // rows searched for together

// ---- codewords: the smallest of every group of 8 accumulators with the group's number (at most 32 of
// them) in the mantissa's low 5 bits, the nearest group and the second's value.  The codeword inside
// the group is found by the caller in fp32; where the second group may hold one as near, the
// caller searches them all.
struct NearestGroup {
  float best, second;
  __device__ __forceinline__ void clear() { best = second = CUDART_INF_F; }
  __device__ __forceinline__ int group() const { return (int)(__float_as_uint(best) & 31u); }
  template <int N> __device__ __forceinline__ void take(const float (&v)[N], uint32_t grp0) {
    float b[N / 8];
#pragma unroll
    for (int g = 0; g < N / 8; ++g) {
      const float* w = v + 8 * g;
      const float m = min3(min3(w[0], w[1], w[2]), min3(w[3], w[4], w[5]), fminf(w[6], w[7]));
      b[g] = __uint_as_float((__float_as_uint(m) & ~31u) | (grp0 + g));
    }
#pragma unroll
    for (int g = 0; g < N / 8; ++g) {
      // (the larger of the two, as their sum without the smaller: the integer pipe, which does minima, is
      // what bounds the search)
      const float sum = best + b[g];
      best = fminf(best, b[g]);
      second = fminf(second, sum - best);
    }
  }
};
// Is the second group within the errors of both arithmetics of the best?  (e2 = |e|^2 of the sub-vector;
// at most four accumulations, the group's bits the larger part: 2^-18 of each value.  Generous: a search
// that was not needed costs less than a hundredth.)
constexpr float kPqTieE2 = 4e-5f, kPqTieV = 1.6e-5f;
__device__ __forceinline__ bool pq_tie(const NearestGroup& g, float e2) {
  const float reach = fmaf(kPqTieE2 * kTcScale * kTcScale, e2, fmaf(kPqTieV, fabsf(g.best), 2.f * kTieFloor));
  return !(g.second >= g.best + reach);
}
template <int DSUB> __device__ __forceinline__ void load_sub(const float* src, float (&x)[DSUB]) {
  if constexpr (DSUB == 2) {
    *reinterpret_cast<float2*>(x) = *reinterpret_cast<const float2*>(src);
  } else {
#pragma unroll
    for (int c4 = 0; c4 < DSUB / 4; ++c4)
      *reinterpret_cast<float4*>(x + 4 * c4) = *reinterpret_cast<const float4*>(src + 4 * c4);
  }
}
// Sub-vectors that have to be compared with all codewords: bit i of `mine` is this lane's i-th.
// s.load(lane, i, x) reads one, s.distance(i, x, z) compares it as the caller does, s.done(i, x, z) takes
// the nearest codeword (lower index on ties) in the lane it belongs to.  One after the other, the warp's
// lanes over the codewords, unless most lanes have one (equal keys, all zeros): then every lane its own.
// That is told for each i: codebooks with a dozen equal words tie for a few lanes at every i, and 8 x 256
// tokens took 281 us with the lanes counted over all i, 103 so.  All lanes call.
// (A call of its own: inlined, it took registers from the search before it, 4 us of an update.)
template <int DSUB, int kCodes, class S>
__device__ __noinline__ unsigned long long settle_codewords(unsigned mine, int n_items, S s) {
  constexpr int kAhead = kCodes < 32 ? 1 : DSUB <= 4 ? 8 : 32 / DSUB;      // codewords in flight (they may be in global memory)
  const int lane = threadIdx.x & 31;
#pragma unroll 1
  for (int i = 0; i < n_items; ++i) {
    const unsigned who = __ballot_sync(0xffffffffu, (mine >> i) & 1u);
    float x[DSUB];
    if (__popc(who) > 16) {
      float d = CUDART_INF_F;
      int at = 0;
      s.load(lane, i, x);
#pragma unroll 2
      for (int z = 0; z < kCodes; ++z) {
        const float dist = s.distance(i, x, z);
        if (dist < d) { d = dist; at = z; }
      }
      if ((who >> lane) & 1u) s.done(i, x, at);
    } else {
#pragma unroll 1
      for (unsigned left = who; left; left &= left - 1u) {
        const int src = __ffs(left) - 1;
        float d = CUDART_INF_F;
        int at = 0;
        s.load(src, i, x);
#pragma unroll 1
        for (int z0 = lane; z0 < kCodes; z0 += 32 * kAhead) {
          float dist[kAhead];
#pragma unroll
          for (int u = 0; u < kAhead; ++u) dist[u] = s.distance(i, x, z0 + 32 * u);
#pragma unroll
          for (int u = 0; u < kAhead; ++u)
            if (dist[u] < d) { d = dist[u]; at = z0 + 32 * u; }
        }
        warp_nearest(d, at);
        if (lane == src) s.done(i, x, at);
      }
    }
  }
  return s.result;
}

}  // namespace
}  // namespace pqhsa
