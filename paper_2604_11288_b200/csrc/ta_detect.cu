// Embedding-based anchor detector (Section 3.2 "Anchor detection", instantiation 3; Section 5.4): the confidence of a
// token is the largest cosine similarity between its input embedding and a handful of anchor-concept embeddings.
//
// The work is one pass over the embeddings (D bf16 values per token, read once; nothing else is large), so the kernel
// is built around that stream: a block takes 32 tokens at a time, four warps per 16 tokens, each a quarter of the
// dimensions; per 32 dimensions every lane reads 16 contiguous bytes of two token rows straight from global memory (four
// lanes cover 64 contiguous bytes of a row: whole sectors, each fetched once), the dot products with the (at most 8)
// concepts run as m16n8k16 tensor-core products against concept fragments kept in shared memory, and the squared norms of
// the rows are accumulated from the same registers. The quarters meet in shared memory. The order of the dimensions inside a
// product is free as long as both operands use the same one, so a lane's 8 consecutive dimensions serve as its fragment
// columns of two products. The contraction has N = 8: far too small for a tcgen05 tile to pay; the memory stream is what
// bounds it (2*D bytes per token against about 20 instructions per 16 tokens and 16 dimensions). Why quarters: with a warp
// per 16 tokens, 131072 tokens were 1.73 rounds of the resident warps, and the last round ran with a part of them
// (131072 x 2048: 135 us, 4.0 TB/s; now 87 us, 6.2 TB/s).
#include <cuda_bf16.h>

#include "ta_internal.cuh"

namespace {

constexpr int kWarps = 8;
constexpr int kMaxConcepts = 8;
constexpr int kAhead = 4;                            // stretches of 32 dimensions requested ahead
constexpr int kQuarters = 4;                         // warps that share 16 tokens
constexpr int kGroupsPerBlock = kWarps / kQuarters;  // groups of 16 tokens a block handles at a time

__device__ __forceinline__ void mma_bf16_16816(float (&d)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
  asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
               : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
               : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}
__device__ __forceinline__ float sq2(uint32_t w) {  // sum of squares of a bf16 pair
  const float lo = __uint_as_float(w << 16), hi = __uint_as_float(w & 0xffff0000u);
  return fmaf(lo, lo, hi * hi);
}

__global__ void __launch_bounds__(kWarps * 32, 3)
ta_embed_conf_kernel(long long total, const __nv_bfloat16* emb, long long stride, int D, const __nv_bfloat16* concepts, int C,
                     float* __restrict__ conf) {
  extern __shared__ __align__(16) unsigned char smem[];
  const int ld = D + 32;  // padded row: consecutive rows start 64 bytes apart modulo 128 (conflict-free 16-byte loads)
  __nv_bfloat16* s_c = reinterpret_cast<__nv_bfloat16*>(smem);           // [8][D + 32], unused concepts are zero
  float* s_inv = reinterpret_cast<float*>(smem + (size_t)kMaxConcepts * ld * 2);  // 1 / |concept|, 0 for zero vectors
  __shared__ float s_part[kWarps][16][10];  // a warp's products with the 8 concepts and squared norm of its 16 tokens
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  ta_wait_for_prior_grid();
  if ((reinterpret_cast<uintptr_t>(concepts) & 15) == 0) {
    for (int i = tid; i < kMaxConcepts * (ld / 8); i += blockDim.x) {
      const int c = i / (ld / 8), k = i - c * (ld / 8);
      reinterpret_cast<uint4*>(s_c)[i] = (c < C && k * 8 < D) ? reinterpret_cast<const uint4*>(concepts + (size_t)c * D)[k]
                                                              : make_uint4(0u, 0u, 0u, 0u);
    }
  } else {
    for (int i = tid; i < kMaxConcepts * ld; i += blockDim.x) {
      const int c = i / ld, k = i - c * ld;
      s_c[i] = (c < C && k < D) ? concepts[(size_t)c * D + k] : __float2bfloat16(0.0f);
    }
  }
  __syncthreads();
  if (warp < kMaxConcepts) {  // one warp per concept norm
    float acc = 0.0f;
    const uint32_t* row = reinterpret_cast<const uint32_t*>(s_c + (size_t)warp * ld);
    for (int k = lane; k < D / 2; k += 32) acc += sq2(row[k]);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
    if (lane == 0) s_inv[warp] = acc > 0.0f ? rsqrtf(acc) : 0.0f;
  }
  __syncthreads();

  const int r = lane >> 2, q = lane & 3;  // fragment row (and row + 8), column pair
  const int quarter = warp % kQuarters, sub = warp / kQuarters;
  const int chunks = D / 32;
  const int k_lo = chunks * quarter / kQuarters * 32, k_hi = chunks * (quarter + 1) / kQuarters * 32;
  const long long sets = (total + 16 * kGroupsPerBlock - 1) / (16 * kGroupsPerBlock);
  for (long long set = blockIdx.x; set < sets; set += gridDim.x) {
    const long long t0 = (set * kGroupsPerBlock + sub) * 16 + r, t1 = t0 + 8;
    // rows past the end re-read the last token; their results are not written
    const uint4* e0 = reinterpret_cast<const uint4*>(emb + (t0 < total ? t0 : total - 1) * stride) + q;
    const uint4* e1 = reinterpret_cast<const uint4*>(emb + (t1 < total ? t1 : total - 1) * stride) + q;
    const uint4* cb = reinterpret_cast<const uint4*>(s_c + (size_t)r * ld) + q;  // concept r, dimensions 8q .. 8q+7
    // two accumulator sets taken in turn: the tensor core's fp32 accumulation does not round to nearest, and its
    // error grows with the length of one accumulation chain
    float dA[4] = {0.0f, 0.0f, 0.0f, 0.0f}, dB[4] = {0.0f, 0.0f, 0.0f, 0.0f};
    float n0 = 0.0f, n1 = 0.0f;
    auto step = [&](const uint4& v0, const uint4& v1, int k) {  // 32 dimensions = 4 x uint4 per row
      const uint4 vb = cb[k >> 3];
      const uint32_t a0[4] = {v0.x, v1.x, v0.y, v1.y}, a1[4] = {v0.z, v1.z, v0.w, v1.w};
      mma_bf16_16816(dA, a0, vb.x, vb.y);
      mma_bf16_16816(dB, a1, vb.z, vb.w);
      n0 += (sq2(v0.x) + sq2(v0.y)) + (sq2(v0.z) + sq2(v0.w));
      n1 += (sq2(v1.x) + sq2(v1.y)) + (sq2(v1.z) + sq2(v1.w));
    };
    int k = k_lo;
    for (; k + kAhead * 32 <= k_hi; k += kAhead * 32) {  // all loads of a stretch in flight before the first is used
      uint4 v0[kAhead], v1[kAhead];
#pragma unroll
      for (int j = 0; j < kAhead; ++j) {
        v0[j] = ta_ld_stream(e0 + (k >> 3) + 4 * j);
        v1[j] = ta_ld_stream(e1 + (k >> 3) + 4 * j);
      }
#pragma unroll
      for (int j = 0; j < kAhead; ++j) step(v0[j], v1[j], k + 32 * j);
    }
    for (; k < k_hi; k += 32) step(ta_ld_stream(e0 + (k >> 3)), ta_ld_stream(e1 + (k >> 3)), k);
    // the four lanes of a row hold its norm in parts, and its dot products with concepts 2q and 2q + 1
    n0 += __shfl_xor_sync(0xffffffffu, n0, 1);
    n0 += __shfl_xor_sync(0xffffffffu, n0, 2);
    n1 += __shfl_xor_sync(0xffffffffu, n1, 1);
    n1 += __shfl_xor_sync(0xffffffffu, n1, 2);
    __syncthreads();  // the partial results of the previous set have been read
    s_part[warp][r][2 * q] = dA[0] + dB[0];
    s_part[warp][r][2 * q + 1] = dA[1] + dB[1];
    s_part[warp][r + 8][2 * q] = dA[2] + dB[2];
    s_part[warp][r + 8][2 * q + 1] = dA[3] + dB[3];
    if (q == 0) {
      s_part[warp][r][8] = n0;
      s_part[warp][r + 8][8] = n1;
    }
    __syncthreads();
    if (tid < 16 * kGroupsPerBlock) {  // a thread per token
      const int g = tid >> 4, row = tid & 15;
      const long long t = (set * kGroupsPerBlock + g) * 16 + row;
      float d[9];
#pragma unroll
      for (int c = 0; c < 9; ++c) {
        const float* part = &s_part[g * kQuarters][row][c];
        d[c] = (part[0] + part[160]) + (part[320] + part[480]);
      }
      const float inv = d[8] > 0.0f ? rsqrtf(d[8]) : 0.0f;
      // concepts beyond C are zero vectors with similarity 0: they must not win over negative similarities. NaN must survive
      // the maximum (a NaN confidence is "no anchor" downstream): fmaxf drops it, so carry a flag
      float m = -INFINITY;
      bool bad = !(d[8] == d[8]);
#pragma unroll
      for (int c = 0; c < 8; ++c) {
        if (c < C) m = fmaxf(m, d[c] * inv * s_inv[c]);
        bad = bad || !(d[c] == d[c]);
      }
      if (t < total) conf[t] = bad ? NAN : m;
    }
  }
}

}  // namespace

cudaError_t ta_launch_embed_conf(int sm_count, long long total, const void* emb, long long stride, int D,
                                 const void* concepts, int C, float* conf, cudaStream_t stream) {
  if (total == 0) return cudaSuccess;
  const size_t smem = (size_t)kMaxConcepts * (D + 32) * 2 + kMaxConcepts * sizeof(float);
  static bool attr_set[64] = {};
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (!attr_set[dev & 63]) {
    e = cudaFuncSetAttribute(ta_embed_conf_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024);
    if (e != cudaSuccess) return e;
    attr_set[dev & 63] = true;
  }
  const long long sets = (total + 16 * kGroupsPerBlock - 1) / (16 * kGroupsPerBlock);
  // as many blocks as are resident at once (shared memory: the concepts; registers: three blocks), or rather as many as
  // give every block the same number of sets
  const int per_sm = smem > 100 * 1024 ? 1 : smem > 66 * 1024 ? 2 : 3;
  const long long resident = (long long)sm_count * per_sm;
  const long long rounds = (sets + resident - 1) / resident;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)((sets + rounds - 1) / rounds), 1, 1);
  cfg.blockDim = dim3(kWarps * 32, 1, 1);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = stream;
  cudaLaunchAttribute attr[1];
  ta_pdl_attribute(&attr[0]);
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, ta_embed_conf_kernel, total, reinterpret_cast<const __nv_bfloat16*>(emb), stride, D,
                            reinterpret_cast<const __nv_bfloat16*>(concepts), C, conf);
}
