// Step 1 of the decode operator: lookup-table construction (Sec. 3.1, text after Eq. 2).
//
// For every query head h of a (sequence, KV head):  coarse[j] = sm_scale * q_h . c_j  and
// LUT[z][m] = sm_scale * q_h^(m) . p_{m,z}.  Since q = r_q u_q, these are the paper's
// r_q/sqrt(d) * (u_q . c_j) and r_q/sqrt(d) * (u_q^(m) . p_{m,z}).  The tables are written in
// the layout the scan wants to find in shared memory: [z][m][g] with g the head inside its
// head group, so one 16-byte read serves the four heads of a GQA group.
//
// The kernel is bound by instruction issue (many sequences) or latency (few).  So the queries pass
// through registers once per CTA: for the coarse term 8 lanes share a centroid row and keep their 16
// dims of four heads in registers, a warp takes four rows at a time with packed multiply-adds, and
// four shuffles reduce all 16 sums; the number of CTAs per (sequence, KV head) falls as there are
// more of them.  Decode call with a row per warp and 32 CTAs each -> now: 128K x 8
// 314 -> 312 us, 512K 199 -> 190, 4-bit codes 128K x 8 199 -> 193.  In the
// fused decode call it also clears the counters and sums that later kernels need.
#include "common.cuh"

namespace pqhsa {

constexpr int kLutThreads = 256;
constexpr int kLutWarps = kLutThreads / 32;
constexpr int kLutMaxChunks = 32;    // CTAs per (sequence, KV head)
constexpr int kMaxGroup = 16;
constexpr int kBatchRows = kLutWarps * 4;

template <typename T> __device__ __forceinline__ float to_f32(T v);
template <> __device__ __forceinline__ float to_f32<__half>(__half v) { return __half2float(v); }
template <> __device__ __forceinline__ float to_f32<__nv_bfloat16>(__nv_bfloat16 v) {
  return __bfloat162float(v);
}

__device__ __forceinline__ unsigned long long lut_fma2(unsigned long long a, unsigned long long b, unsigned long long c) {
  unsigned long long r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
  return r;
}

template <typename T, int DSUB>
__global__ void __launch_bounds__(kLutThreads)
build_lut_kernel(Plan pl, const T* __restrict__ q, const float* __restrict__ centroids,
                 const float* __restrict__ codebooks, float* __restrict__ lut,
                 float* __restrict__ coarse, uint4* __restrict__ zero_ptr, size_t zero_n16) {
  __shared__ __align__(16) float sq[kMaxGroup][kHeadDim];   // sm_scale * q of the heads, 0-padded
  const int kv = blockIdx.y, b = blockIdx.z;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int G = pl.G, Gc = pl.Gc, n_hg = pl.n_hg;
  const int n_slots = n_hg * Gc;                            // head slots, >= G
  const int gc_shift = Gc == 4 ? 2 : (Gc == 2 ? 1 : 0);     // Gc is 1, 2 or 4
  const int code_shift = 31 - __clz(pl.n_code);             // n_code is 16 or 256
  const size_t ukv = (size_t)b * pl.Hkv + kv;
  pdl_wait();
  pdl_launch_dependents();

  // query (first dependent load of the kernel): 8 elements per thread
  constexpr int kQPer = (kMaxGroup * kHeadDim) / (8 * kLutThreads);      // 1
  static_assert(kQPer == 1, "one load per thread covers the widest group");
  uint4 qw = make_uint4(0u, 0u, 0u, 0u);
  if (8 * tid < G * kHeadDim) qw = load_eight(q + ((size_t)b * pl.Hq + kv * G) * kHeadDim + 8 * tid);

  // ---- prefetch: this lane's part of its first centroid row and the codeword of this thread
  const int rows_per_cta = (pl.n_list + gridDim.x - 1) / gridDim.x;
  const int r0 = blockIdx.x * rows_per_cta;
  const int r1 = min(pl.n_list, r0 + rows_per_cta);
  const int kEntPerM = pl.n_code;
  const int n_ent = pl.M * kEntPerM;
  const int ent_per_cta = (n_ent + gridDim.x - 1) / gridDim.x;
  const int e0 = blockIdx.x * ent_per_cta;
  const int e1 = min(n_ent, e0 + ent_per_cta);

  // lane (r, i) = (lane >> 3, lane & 7): row r of the warp's four, dims 4 (i + 8 t) + 0 .. 3
  const int lr = lane >> 3, li = lane & 7;
  float4 crow[4];
  auto load_row = [&](int jb) {
    const int j = jb + warp * 4 + lr;
#pragma unroll
    for (int t = 0; t < 4; ++t) {
      crow[t] = make_float4(0.f, 0.f, 0.f, 0.f);
      if (j < r1) crow[t] = __ldg(reinterpret_cast<const float4*>(centroids + (ukv * pl.n_list + j) * kHeadDim) + li + 8 * t);
    }
  };
  load_row(r0);
  constexpr int kWordBatch = DSUB <= 4 ? 4 : 16 / DSUB;          // codewords in flight per thread
  float cw[kWordBatch][DSUB];
  auto load_codewords = [&](int eb) {
#pragma unroll
    for (int u = 0; u < kWordBatch; ++u) {
      const int e = eb + u * kLutThreads + tid;
      if (e >= e1) continue;
      const float* p = codebooks + (ukv * (size_t)n_ent + e) * DSUB;
      if constexpr (DSUB == 2) {
        const float2 v = __ldg(reinterpret_cast<const float2*>(p));
        cw[u][0] = v.x; cw[u][1] = v.y;
      } else {
#pragma unroll
        for (int c = 0; c < DSUB / 4; ++c) {
          const float4 v = __ldg(reinterpret_cast<const float4*>(p) + c);
          cw[u][4 * c] = v.x; cw[u][4 * c + 1] = v.y; cw[u][4 * c + 2] = v.z; cw[u][4 * c + 3] = v.w;
        }
      }
    }
  };
  load_codewords(e0);

  // ---- side job: clear a slice of the caller's zero region
  if (zero_ptr != nullptr) {
    const size_t nthreads = (size_t)gridDim.x * gridDim.y * gridDim.z * kLutThreads;
    const size_t gtid = ((size_t)(blockIdx.z * gridDim.y + blockIdx.y) * gridDim.x + blockIdx.x) *
                            kLutThreads + tid;
    for (size_t i = gtid; i < zero_n16; i += nthreads) zero_ptr[i] = make_uint4(0u, 0u, 0u, 0u);
  }

  {
    const T* e = reinterpret_cast<const T*>(&qw);                // (slots past G are zero)
#pragma unroll
    for (int i = 0; i < 8; ++i) (&sq[0][0])[8 * tid + i] = pl.sm_scale * to_f32(e[i]);
  }
  __syncthreads();

  // ---- coarse term, four heads at a time
  for (int hb = 0; hb < n_slots; hb += 4) {
    unsigned long long qq[4][4][2];                              // [head][t][pair]
#pragma unroll
    for (int g = 0; g < 4; ++g)
#pragma unroll
      for (int t = 0; t < 4; ++t) {
        const ulonglong2 v = *reinterpret_cast<const ulonglong2*>(&sq[(hb + g) & (kMaxGroup - 1)][4 * (li + 8 * t)]);
        qq[g][t][0] = v.x;
        qq[g][t][1] = v.y;
      }
    if (hb != 0) load_row(r0);
    for (int jb = r0; jb < r1; jb += kBatchRows) {
      unsigned long long acc[4] = {0ull, 0ull, 0ull, 0ull};
#pragma unroll
      for (int t = 0; t < 4; ++t) {
        const ulonglong2 c = *reinterpret_cast<const ulonglong2*>(&crow[t]);
#pragma unroll
        for (int g = 0; g < 4; ++g) acc[g] = lut_fma2(c.y, qq[g][t][1], lut_fma2(c.x, qq[g][t][0], acc[g]));
      }
      const int j = jb + warp * 4 + lr;
      if (jb + kBatchRows < r1) load_row(jb + kBatchRows);
      float d[4];
#pragma unroll
      for (int g = 0; g < 4; ++g)
        d[g] = __uint_as_float((uint32_t)acc[g]) + __uint_as_float((uint32_t)(acc[g] >> 32));
      // over the 8 lanes of the row; lane i ends with head (i >> 1)
      const bool up4 = (li & 4) != 0, up2 = (li & 2) != 0;
      float k0 = up4 ? d[2] : d[0], k1 = up4 ? d[3] : d[1];
      k0 += __shfl_xor_sync(0xffffffffu, up4 ? d[0] : d[2], 4);
      k1 += __shfl_xor_sync(0xffffffffu, up4 ? d[1] : d[3], 4);
      float tot = up2 ? k1 : k0;
      tot += __shfl_xor_sync(0xffffffffu, up2 ? k0 : k1, 2);
      tot += __shfl_xor_sync(0xffffffffu, tot, 1);
      const int slot = hb + (li >> 1);
      if ((li & 1) == 0 && j < r1 && slot < n_slots)
        coarse[((ukv * n_hg + (slot >> gc_shift)) * (size_t)pl.n_list + j) * Gc + (slot & (Gc - 1))] = tot;
    }
  }

  // ---- PQ table: one thread per (m, z); consecutive threads take consecutive z, so the
  //      subspace m (and with it the query sub-vector) is uniform over a warp
  float* const lut_u = lut + ukv * n_hg * (size_t)pl.n_code * pl.M * Gc;
  for (int eb = e0; eb < e1; eb += kWordBatch * kLutThreads) {
    if (eb != e0) load_codewords(eb);
#pragma unroll
    for (int u = 0; u < kWordBatch; ++u) {
      const int e = eb + u * kLutThreads + tid;
      if (e >= e1) continue;
      const int m = e >> code_shift, z = e & (kEntPerM - 1);
      for (int hg = 0; hg < n_hg; ++hg) {
        float v[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
        for (int g = 0; g < 4; ++g) {
          if (g < Gc) {
            // (the reads are uniform over the warp, 8 or 16 bytes wide)
            const float* qs = &sq[(hg * Gc + g) & (kMaxGroup - 1)][m * DSUB];
            float qv[DSUB];
            if constexpr (DSUB == 2) {
              const float2 t2 = *reinterpret_cast<const float2*>(qs);
              qv[0] = t2.x; qv[1] = t2.y;
            } else {
#pragma unroll
              for (int c = 0; c < DSUB / 4; ++c) {
                const float4 t4 = *reinterpret_cast<const float4*>(qs + 4 * c);
                qv[4 * c] = t4.x; qv[4 * c + 1] = t4.y; qv[4 * c + 2] = t4.z; qv[4 * c + 3] = t4.w;
              }
            }
#pragma unroll
            for (int t = 0; t < DSUB; ++t) v[g] = fmaf(cw[u][t], qv[t], v[g]);
          }
        }
        float* dst = lut_u + (((size_t)hg * pl.n_code + z) * pl.M + m) * Gc;
        if (Gc == 4) *reinterpret_cast<float4*>(dst) = make_float4(v[0], v[1], v[2], v[3]);
        else if (Gc == 2) *reinterpret_cast<float2*>(dst) = make_float2(v[0], v[1]);
        else dst[0] = v[0];
      }
    }
  }
}

template <typename T>
static cudaError_t launch_lut_t(const Plan& pl, const T* q, const pqhsa_index& ix, float* lut,
                                float* coarse, uint4* zp, size_t zn, cudaStream_t st) {
  // one wave of two CTAs per SM: at 64 units (128K x 8) 4 CTAs a unit measured 312 us for the decode
  // call, 8 / 12 / 16 / 32 CTAs 312 / 314 / 315 / 319; at 8 units (512K) 32 are best (190; 4 CTAs 208)
  int chunks = 2 * pl.num_sms / (pl.B * pl.Hkv);
  if (chunks > kLutMaxChunks) chunks = kLutMaxChunks;
  if (chunks < 4) chunks = 4;
  dim3 grid(chunks, pl.Hkv, pl.B);
  switch (pl.dsub) {
    case 2: set_carveout<build_lut_kernel<T, 2>>(kStreamCarveout); return launch_pdl(build_lut_kernel<T, 2>, grid, dim3(kLutThreads), 0, st, pl, q, ix.centroids, ix.codebooks, lut, coarse, zp, zn);
    case 4: set_carveout<build_lut_kernel<T, 4>>(kStreamCarveout); return launch_pdl(build_lut_kernel<T, 4>, grid, dim3(kLutThreads), 0, st, pl, q, ix.centroids, ix.codebooks, lut, coarse, zp, zn);
    case 8: set_carveout<build_lut_kernel<T, 8>>(kStreamCarveout); return launch_pdl(build_lut_kernel<T, 8>, grid, dim3(kLutThreads), 0, st, pl, q, ix.centroids, ix.codebooks, lut, coarse, zp, zn);
    case 16: set_carveout<build_lut_kernel<T, 16>>(kStreamCarveout); return launch_pdl(build_lut_kernel<T, 16>, grid, dim3(kLutThreads), 0, st, pl, q, ix.centroids, ix.codebooks, lut, coarse, zp, zn);
    default: return cudaErrorInvalidValue;
  }
  return cudaGetLastError();
}

cudaError_t launch_build_lut(const Plan& pl, const void* q, const pqhsa_index& ix, float* lut,
                             float* coarse, void* zero_ptr, size_t zero_bytes, cudaStream_t st) {
  uint4* zp = static_cast<uint4*>(zero_ptr);
  const size_t zn = zero_bytes / 16;
  if (pl.dtype == PQHSA_F16)
    return launch_lut_t(pl, static_cast<const __half*>(q), ix, lut, coarse, zp, zn, st);
  return launch_lut_t(pl, static_cast<const __nv_bfloat16*>(q), ix, lut, coarse, zp, zn, st);
}

}  // namespace pqhsa
