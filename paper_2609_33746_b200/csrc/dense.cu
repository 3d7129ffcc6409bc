// Dense decode attention over the whole paged KV cache: the comparator of the context-length
// sweep (Eq. 1 with E = every cached token).  Not part of the PQ-HSA path; it exists so that
// the operator's time can be set against a full-KV read on the same GPU and the same cache.
//
// Split-K flash decoding.  grid (splits, KV heads, sequences).  A warp takes windows of 32 tokens and
// serves up to four query heads of the GQA group from one read and one unpacking of each K/V row: 16
// lanes per 256-byte row, online softmax in base 2; groups of more than four heads are shared out
// among the CTA's warps, which walk the same tokens, each from L2.  Rows come through a per-warp ring of
// asynchronous copies, 8 rows (4 KB) a stage and two stages ahead of the one in use; a lane copies
// the 16 bytes that it reads itself, so the ring needs no barrier.  The last CTA of a (sequence, KV
// head) merges the partial (m, Z, N) triples of its G rows (atomic ticket; nobody waits).
// What bounds it: the read of the cache.  8 x 32K tokens, 32 / 8 heads: one warp per head (rows
// unpacked four times) 394 us, four heads per warp with loads into registers 260 us (latency: 3.9
// warps waiting per issue), with the ring 218 us (4.9 TB/s, 0.75 of the copy rate).
#include "attn_common.cuh"
#include "common.cuh"
#include "scan_common.cuh"

namespace pqhsa {

namespace {

constexpr int kDensePart = kPartStride;
constexpr int kDenseThreads = 256, kDenseWarps = kDenseThreads / 32;
constexpr int kMaxDenseHeads = 16;
constexpr int kDenseStages = 3, kStageRows = 8, kStageBytes = kStageRows * 4 * kHeadDim;
constexpr int kDenseSmem = kDenseWarps * kDenseStages * kStageBytes;

__device__ __forceinline__ unsigned long long dup2(float a) {
  unsigned long long r;
  asm("mov.b64 %0, {%1, %1};" : "=l"(r) : "f"(a));
  return r;
}
__device__ __forceinline__ unsigned long long mk2(float a, float b) {
  unsigned long long r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
  return r;
}
__device__ __forceinline__ void un2(unsigned long long v, float& a, float& b) {
  asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(v));
}
__device__ __forceinline__ unsigned long long fma2(unsigned long long a, unsigned long long b, unsigned long long c) {
  unsigned long long r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
  return r;
}
__device__ __forceinline__ unsigned long long mul2(unsigned long long a, unsigned long long b) {
  unsigned long long r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
template <typename T> __device__ __forceinline__ void unpack2(const uint4& u, unsigned long long (&p)[4]) {
  float f[8];
  Unpack<T>::run(u, f);
#pragma unroll
  for (int i = 0; i < 4; ++i) p[i] = mk2(f[2 * i], f[2 * i + 1]);
}

// Sums one value per head over the 16 lanes of a row; lane l of the 16 ends with head head_of(l)'s total.
template <int GH> __device__ __forceinline__ int head_of(int l16) {
  return GH == 4 ? l16 >> 2 : (GH == 2 ? l16 >> 3 : 0);
}
template <int GH> __device__ __forceinline__ float reduce_heads(const float (&d)[GH], int l16) {
  float x;
  if constexpr (GH == 4) {
    const bool up = (l16 & 8) != 0;
    float k0 = up ? d[2] : d[0], k1 = up ? d[3] : d[1];
    k0 += __shfl_xor_sync(0xffffffffu, up ? d[0] : d[2], 8);
    k1 += __shfl_xor_sync(0xffffffffu, up ? d[1] : d[3], 8);
    const bool up4 = (l16 & 4) != 0;
    x = up4 ? k1 : k0;
    x += __shfl_xor_sync(0xffffffffu, up4 ? k0 : k1, 4);
  } else if constexpr (GH == 2) {
    const bool up = (l16 & 8) != 0;
    x = up ? d[1] : d[0];
    x += __shfl_xor_sync(0xffffffffu, up ? d[0] : d[1], 8);
    x += __shfl_xor_sync(0xffffffffu, x, 4);
  } else {
    x = d[0];
    x += __shfl_xor_sync(0xffffffffu, x, 8);
    x += __shfl_xor_sync(0xffffffffu, x, 4);
  }
  x += __shfl_xor_sync(0xffffffffu, x, 2);
  x += __shfl_xor_sync(0xffffffffu, x, 1);
  return x;
}

template <typename T, int GH>
__global__ void __launch_bounds__(kDenseThreads, 2)
dense_decode_kernel(Plan pl, const T* __restrict__ q, const T* __restrict__ kc,
                    const T* __restrict__ vc, long long stride_page, long long stride_token,
                    long long stride_head, const int32_t* __restrict__ block_table,
                    const int32_t* __restrict__ seq_lens, float* __restrict__ part,
                    uint32_t* __restrict__ tickets, T* __restrict__ out) {
  constexpr int U = kStageRows / 2;                         // row pairs per stage
  extern __shared__ __align__(128) unsigned char s_ring[];  // [warp][stage][row][K 256 bytes | V 256 bytes]
  __shared__ int s_last;
  __shared__ float s_m[kDenseWarps][GH], s_Z[kDenseWarps][GH];
  const int split = blockIdx.x, S = gridDim.x, kv = blockIdx.y, b = blockIdx.z;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int half = lane >> 4, l16 = lane & 15;
  const int n_grp = (pl.G + GH - 1) / GH;                   // head groups (1, or up to 4 of four heads)
  const int n_par = kDenseWarps / n_grp;                    // warps that share a head group's tokens
  const int hg = warp / n_par, par = warp - hg * n_par;     // (warps past n_grp * n_par idle)
  const int row0 = b * pl.Hq + kv * pl.G + hg * GH;         // first query head of this warp
  const int n_heads = hg < n_grp ? min(GH, pl.G - hg * GH) : 0;
  pdl_wait();
  pdl_launch_dependents();
  const int n = clamp_len(seq_lens[b], pl.N_max);
  const int tl = (int)((long long)split * n / S), th = n_heads > 0 ? (int)((long long)(split + 1) * n / S) : 0;
  const int32_t* bt = block_table + (size_t)b * pl.max_pages;

  unsigned long long q2[GH][4], acc[GH][4];
#pragma unroll
  for (int g = 0; g < GH; ++g) {
    uint4 w = make_uint4(0u, 0u, 0u, 0u);
    if (g < n_heads) w = load_eight(q + (size_t)(row0 + g) * kHeadDim + 8 * l16);
    unpack2<T>(w, q2[g]);
    const unsigned long long sc = dup2(pl.sm_scale * kLog2e);
#pragma unroll
    for (int t = 0; t < 4; ++t) { q2[g][t] = mul2(q2[g][t], sc); acc[g][t] = 0ull; }
  }
  float m = -CUDART_INF_F, Z = 0.f;                         // of head head_of(l16), this half's rows

  // this warp's windows of 32 tokens: first, first + stride, ..; a stage is a quarter of a window
  const int first = tl + 32 * par, stride = 32 * n_par;
  const int n_steps = first < th ? 4 * ((th - first + stride - 1) / stride) : 0;
  unsigned char* ring = s_ring + warp * (kDenseStages * kStageBytes);
  const uint32_t ring_u32 = smem_u32(ring) + half * 512 + l16 * 16;
  int my_page = (first + lane < th) ? __ldg(bt + (first + lane) / pl.page_size) : 0;
  long long off = 0;                                        // this lane's token of the window being copied
  auto issue = [&](int st) {
    if (st < n_steps) {
      const int base = first + (st >> 2) * stride;
      if ((st & 3) == 0) {
        const int pos = base + lane;
        off = 0;
        if (pos < th)
          off = (long long)my_page * stride_page + (long long)(pos % pl.page_size) * stride_token +
                (long long)kv * stride_head;
        if (pos + stride < th) my_page = __ldg(bt + (pos + stride) / pl.page_size);
      }
      const uint32_t dst = ring_u32 + (uint32_t)(st % kDenseStages) * kStageBytes;
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const int tok = (st & 3) * kStageRows + 2 * u + half;
        const long long o = __shfl_sync(0xffffffffu, off, tok);
        const uint32_t bytes = base + tok < th ? 16u : 0u;  // rows past the slice are zero-filled
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst + u * 1024u),
                     "l"(reinterpret_cast<const uint4*>(kc + o) + l16), "r"(bytes) : "memory");
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst + u * 1024u + 256u),
                     "l"(reinterpret_cast<const uint4*>(vc + o) + l16), "r"(bytes) : "memory");
      }
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  auto row_part = [&](uint32_t addr) {
    uint4 v;
    asm volatile("ld.shared.v4.b32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(addr));
    return v;
  };
#pragma unroll
  for (int st = 0; st < kDenseStages - 1; ++st) issue(st);
#pragma unroll 1
  for (int st = 0; st < n_steps; ++st) {
    issue(st + kDenseStages - 1);
    asm volatile("cp.async.wait_group %0;" ::"n"(kDenseStages - 1) : "memory");
    const uint32_t src = ring_u32 + (uint32_t)(st % kDenseStages) * kStageBytes;
    const int left = th - (first + (st >> 2) * stride + (st & 3) * kStageRows);   // tokens from this stage on
    if (left <= 0) continue;                                // (warp-uniform)
    float sc[U], mx = m;
#pragma unroll
    for (int u = 0; u < U; ++u) {
      unsigned long long k2[4];
      unpack2<T>(row_part(src + u * 1024u), k2);
      float d[GH];
#pragma unroll
      for (int g = 0; g < GH; ++g) {
        unsigned long long a = 0ull;
#pragma unroll
        for (int t = 0; t < 4; ++t) a = fma2(q2[g][t], k2[t], a);
        float x, y;
        un2(a, x, y);
        d[g] = x + y;
      }
      sc[u] = reduce_heads<GH>(d, l16);
      if (2 * u + half >= left) sc[u] = -CUDART_INF_F;
      mx = fmaxf(mx, sc[u]);
    }
    if (__any_sync(0xffffffffu, mx > m)) {                  // some head's maximum grew
      const float a = mx > m && m > -CUDART_INF_F ? fast_exp2(m - mx) : (mx > m ? 0.f : 1.f);
      Z *= a;
      m = mx;
#pragma unroll
      for (int g = 0; g < GH; ++g) {
        const unsigned long long ag = dup2(__shfl_sync(0xffffffffu, a, (lane & 16) + g * (16 / GH)));
#pragma unroll
        for (int t = 0; t < 4; ++t) acc[g][t] = mul2(acc[g][t], ag);
      }
    }
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const float p = sc[u] == -CUDART_INF_F ? 0.f : fast_exp2(sc[u] - m);      // (not a number: shows in the output)
      Z += p;
      unsigned long long v2[4];
      unpack2<T>(row_part(src + u * 1024u + 256u), v2);
#pragma unroll
      for (int g = 0; g < GH; ++g) {
        const unsigned long long pg = dup2(__shfl_sync(0xffffffffu, p, (lane & 16) + g * (16 / GH)));
#pragma unroll
        for (int t = 0; t < 4; ++t) acc[g][t] = fma2(pg, v2[t], acc[g][t]);
      }
    }
  }
  asm volatile("cp.async.wait_group 0;" ::: "memory");
  __syncwarp();                                             // the warp's ring now holds its partial sums
  auto s_N = [&](int w, int g) { return reinterpret_cast<float*>(s_ring + w * (kDenseStages * kStageBytes)) + g * kHeadDim; };
  // the two halves of the warp, then the warps of the head group through shared memory
  {
    const float m_o = __shfl_xor_sync(0xffffffffu, m, 16), Z_o = __shfl_xor_sync(0xffffffffu, Z, 16);
    const float m_n = fmaxf(m, m_o);
    const float a = safe_scale(m, m_n, Z);
    Z = Z * a + Z_o * safe_scale(m_o, m_n, Z_o);
    m = m_n;
#pragma unroll
    for (int g = 0; g < GH; ++g) {
      const float ag = __shfl_sync(0xffffffffu, a, (lane & 16) + g * (16 / GH));
      float f[8];
#pragma unroll
      for (int t = 0; t < 4; ++t) un2(acc[g][t], f[2 * t], f[2 * t + 1]);
#pragma unroll
      for (int t = 0; t < 8; ++t) {
        f[t] *= ag;
        f[t] += __shfl_xor_sync(0xffffffffu, f[t], 16);
      }
      if (half == 0) {
        *reinterpret_cast<float4*>(s_N(warp, g) + 8 * l16) = make_float4(f[0], f[1], f[2], f[3]);
        *reinterpret_cast<float4*>(s_N(warp, g) + 8 * l16 + 4) = make_float4(f[4], f[5], f[6], f[7]);
      }
    }
    if (half == 0 && (l16 & (16 / GH - 1)) == 0) { s_m[warp][head_of<GH>(l16)] = m; s_Z[warp][head_of<GH>(l16)] = Z; }
  }
  __syncthreads();
  const int unit_row0 = b * pl.Hq + kv * pl.G;
  for (int i = tid; i < pl.G * kHeadDim; i += kDenseThreads) {
    const int h = i / kHeadDim, dim = i % kHeadDim, w0 = (h / GH) * n_par, g = h % GH;
    float m_c = -CUDART_INF_F, Z_c = 0.f, N_c = 0.f;
    for (int w = w0; w < w0 + n_par; ++w) if (s_Z[w][g] > 0.f) m_c = fmaxf(m_c, s_m[w][g]);
    for (int w = w0; w < w0 + n_par; ++w) {
      const float a = safe_scale(s_m[w][g], m_c, s_Z[w][g]);
      Z_c = fmaf(s_Z[w][g], a, Z_c);
      N_c = fmaf(s_N(w, g)[dim], a, N_c);
    }
    float* pr = part + ((size_t)(unit_row0 + h) * S + split) * kDensePart;
    pr[4 + dim] = N_c;
    if (dim == 0) { pr[0] = m_c; pr[1] = Z_c; }
  }
  if (!cta_arrived_last(&tickets[b * pl.Hkv + kv], (uint32_t)S, &s_last)) return;
  // last CTA of this (sequence, KV head): a warp merges a row (lane t fetches (m, Z) of partials
  // t, t + 32, ...; then every lane sums its 4 dims over the partials, 8 in flight)
  for (int h = warp; h < pl.G; h += kDenseWarps) {
    const int row = unit_row0 + h;
    const float* rp = part + (size_t)row * S * kDensePart;
    float m_r = -CUDART_INF_F;
    for (int s = lane; s < S; s += 32) {
      const float2 mz = __ldcg(reinterpret_cast<const float2*>(rp + (size_t)s * kDensePart));
      if (mz.y > 0.f) m_r = fmaxf(m_r, mz.x);
    }
    m_r = warp_max(m_r);
    float Z_r = 0.f;
    float4 N_r = make_float4(0.f, 0.f, 0.f, 0.f);
    for (int s0 = 0; s0 < S; s0 += 8) {
      float2 mz[8];
      float4 v[8];
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        mz[u] = make_float2(0.f, 0.f);
        v[u] = make_float4(0.f, 0.f, 0.f, 0.f);
        if (s0 + u < S) {
          mz[u] = __ldcg(reinterpret_cast<const float2*>(rp + (size_t)(s0 + u) * kDensePart));
          v[u] = __ldcg(reinterpret_cast<const float4*>(rp + (size_t)(s0 + u) * kDensePart + 4) + lane);
        }
      }
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        const float a = safe_scale(mz[u].x, m_r, mz[u].y);
        Z_r = fmaf(mz[u].y, a, Z_r);
        N_r.x = fmaf(v[u].x, a, N_r.x); N_r.y = fmaf(v[u].y, a, N_r.y);
        N_r.z = fmaf(v[u].z, a, N_r.z); N_r.w = fmaf(v[u].w, a, N_r.w);
      }
    }
    const float inv = Z_r > 0.f ? 1.f / Z_r : 0.f;
    T* o = out + (size_t)row * kHeadDim + 4 * lane;
    o[0] = Unpack<T>::pack(N_r.x * inv); o[1] = Unpack<T>::pack(N_r.y * inv);
    o[2] = Unpack<T>::pack(N_r.z * inv); o[3] = Unpack<T>::pack(N_r.w * inv);
  }
}

// Splits per (sequence, KV head): whole waves of two CTAs per SM, at least 256 tokens each (more
// pieces even out ragged lengths, but every piece leaves a partial to merge).
int dense_splits(const Plan& pl) {
  const int units = pl.B * pl.Hkv, slots = 2 * pl.num_sms;
  int max_s = pl.N_max / 256 > 0 ? pl.N_max / 256 : 1;
  if (max_s > 256) max_s = 256;
  int best = 1;
  double best_cost = 1e30;
  for (int s = 1; s <= max_s; ++s) {
    const int waves = (units * s + slots - 1) / slots;
    if (waves > 4 && s > 1) break;
    const double cost = (double)waves / s + 0.002 * waves;
    if (cost < best_cost) { best_cost = cost; best = s; }
  }
  return best;
}

template <typename T>
cudaError_t launch_dense_t(const Plan& pl, const void* q, const pqhsa_paged_kv& kv, const int32_t* seq_lens,
                           float* part, uint32_t* tickets, void* out, cudaStream_t st) {
  auto kernel = pl.G == 1 ? dense_decode_kernel<T, 1> : pl.G == 2 ? dense_decode_kernel<T, 2> : dense_decode_kernel<T, 4>;
  const cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kDenseSmem);
  if (e != cudaSuccess) return e;
  return launch_pdl(kernel, dim3(dense_splits(pl), pl.Hkv, pl.B), dim3(kDenseThreads), kDenseSmem, st, pl,
                    static_cast<const T*>(q), static_cast<const T*>(kv.k_cache), static_cast<const T*>(kv.v_cache),
                    (long long)kv.stride_page, (long long)kv.stride_token, (long long)kv.stride_head,
                    kv.block_table, seq_lens, part, tickets, static_cast<T*>(out));
}

size_t align256d(size_t x) { return (x + 255) / 256 * 256; }

// Read-only probe of the gather that the exact part of the attend step performs: the K and V
// rows of the selected tokens, through the block table and the strides, nothing computed (the
// words are xor-ed into a sink that is never written).  A warp takes 32 selected tokens of a
// row at a time: every lane resolves one token's address (position, page) one round ahead,
// then half-warps fetch the K and the V rows, sixteen tokens in flight.  Its time is what the
// memory system charges for these bytes at these addresses: the ceiling the attend kernel is
// measured against.
constexpr int kProbeRows = 16;      // selected tokens per warp in flight (K and V row each)

__global__ void __launch_bounds__(256)
gather_probe_kernel(Plan pl, const unsigned char* __restrict__ kc, const unsigned char* __restrict__ vc,
                    long long stride_page, long long stride_token, long long stride_head,
                    const int32_t* __restrict__ block_table, const int32_t* __restrict__ sel_idx,
                    const int32_t* __restrict__ sel_count, const int32_t* __restrict__ seq_lens,
                    uint4* __restrict__ sink) {
  const int lane = threadIdx.x & 31, half = lane >> 4, l16 = lane & 15;
  const int warp = (int)((blockIdx.x * blockDim.x + threadIdx.x) >> 5);
  const int n_warps = (int)((gridDim.x * blockDim.x) >> 5);
  const int cpr = (pl.k_max + 31) / 32;                  // rounds of 32 tokens per row
  const int rounds = pl.rows * cpr;
  const unsigned char* base = half ? vc : kc;            // lanes 0-15: the K row, 16-31: the V row
  uint4 acc = make_uint4(0u, 0u, 0u, 0u);
  // byte offset of the row of this lane's token in round r, -1 if there is none
  auto resolve = [&](int r) -> long long {
    if (r >= rounds) return -1;
    const int row = r / cpr, t = (r - row * cpr) * 32 + lane;
    const int b = row / pl.Hq, kv = (row % pl.Hq) / pl.G;
    const int cnt = min(max(__ldg(sel_count + row), 0), pl.k_max);
    if (t >= cnt) return -1;
    const int pos = __ldg(sel_idx + (size_t)row * pl.k_max + t);
    if ((unsigned)pos >= (unsigned)clamp_len(seq_lens[b], pl.N_max)) return -1;
    const int page = __ldg(block_table + (size_t)b * pl.max_pages + pos / pl.page_size);
    return 2 * ((long long)page * stride_page + (long long)(pos % pl.page_size) * stride_token +
                (long long)kv * stride_head);             // strides are in 2-byte elements
  };
  long long off = resolve(warp);
  for (int r = warp; r < rounds; r += n_warps) {
    const long long nxt = resolve(r + n_warps);
#pragma unroll
    for (int j0 = 0; j0 < 32; j0 += kProbeRows) {
      uint4 v[kProbeRows];
#pragma unroll
      for (int u = 0; u < kProbeRows; ++u) {
        const long long o = __shfl_sync(0xffffffffu, off, j0 + u);
        v[u] = o >= 0 ? __ldg(reinterpret_cast<const uint4*>(base + o) + l16) : make_uint4(0u, 0u, 0u, 0u);
      }
#pragma unroll
      for (int u = 0; u < kProbeRows; ++u) { acc.x ^= v[u].x; acc.y ^= v[u].y; acc.z ^= v[u].z; acc.w ^= v[u].w; }
    }
    off = nxt;
  }
  // (the store keeps the loads alive; the pattern does not occur)
  if (acc.x == 0x9e3779b9u && acc.y == 0x7f4a7c15u && acc.z == 0xf39cc060u && acc.w == 0x5cedc834u)
    sink[0] = acc;
}

}  // namespace
}  // namespace pqhsa

using namespace pqhsa;

extern "C" {

size_t pqhsa_dense_workspace_bytes(const pqhsa_params* params) {
  Plan pl;
  if (make_plan(params, &pl) != PQHSA_OK) return 0;
  return align256d((size_t)pl.B * pl.Hkv * 4) +
         align256d((size_t)pl.rows * dense_splits(pl) * kDensePart * 4);
}

int pqhsa_dense_decode(const pqhsa_params* params, const void* q, const pqhsa_paged_kv* kv,
                       const int32_t* seq_lens, void* out, void* ws, size_t ws_bytes, void* stream) {
  Plan pl;
  int rc = make_plan(params, &pl);
  if (rc != PQHSA_OK) return rc;
  if (q == nullptr || kv == nullptr || kv->k_cache == nullptr || kv->v_cache == nullptr ||
      kv->block_table == nullptr || seq_lens == nullptr || out == nullptr || ws == nullptr ||
      (reinterpret_cast<uintptr_t>(ws) & 255u) != 0)
    return PQHSA_ERR_INVALID_ARG;
  if (kv->stride_page % 8 || kv->stride_token % 8 || kv->stride_head % 8) return PQHSA_ERR_UNSUPPORTED;
  if (pl.G > kMaxDenseHeads) return PQHSA_ERR_UNSUPPORTED;
  if (ws_bytes < pqhsa_dense_workspace_bytes(params)) return PQHSA_ERR_WORKSPACE;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  char* w = static_cast<char*>(ws);
  const size_t tick_bytes = align256d((size_t)pl.B * pl.Hkv * 4);
  if (cudaMemsetAsync(w, 0, tick_bytes, st) != cudaSuccess) return PQHSA_ERR_CUDA;
  uint32_t* tickets = reinterpret_cast<uint32_t*>(w);
  float* part = reinterpret_cast<float*>(w + tick_bytes);
  const cudaError_t e = pl.dtype == PQHSA_F16
                            ? launch_dense_t<__half>(pl, q, *kv, seq_lens, part, tickets, out, st)
                            : launch_dense_t<__nv_bfloat16>(pl, q, *kv, seq_lens, part, tickets, out, st);
  return e == cudaSuccess ? PQHSA_OK : PQHSA_ERR_CUDA;
}

int pqhsa_gather_probe(const pqhsa_params* params, const pqhsa_paged_kv* kv, const int32_t* sel_idx,
                       const int32_t* sel_count, const int32_t* seq_lens, void* sink16, void* stream) {
  Plan pl;
  int rc = make_plan(params, &pl);
  if (rc != PQHSA_OK) return rc;
  if (kv == nullptr || kv->k_cache == nullptr || kv->v_cache == nullptr || kv->block_table == nullptr ||
      sel_idx == nullptr || sel_count == nullptr || seq_lens == nullptr || sink16 == nullptr ||
      (reinterpret_cast<uintptr_t>(sink16) & 15u) != 0)
    return PQHSA_ERR_INVALID_ARG;
  if (kv->stride_page % 8 || kv->stride_token % 8 || kv->stride_head % 8) return PQHSA_ERR_UNSUPPORTED;
  const cudaError_t e = launch_pdl(
      gather_probe_kernel, dim3(8 * pl.num_sms), dim3(256), 0, static_cast<cudaStream_t>(stream), pl,
      static_cast<const unsigned char*>(kv->k_cache), static_cast<const unsigned char*>(kv->v_cache),
      (long long)kv->stride_page, (long long)kv->stride_token, (long long)kv->stride_head,
      kv->block_table, sel_idx, sel_count, seq_lens, static_cast<uint4*>(sink16));
  return e == cudaSuccess ? PQHSA_OK : PQHSA_ERR_CUDA;
}

}  // extern "C"
