// Step 1 of the retention path: anchor detection, voucher allocation and the attention-free utility
// (Section 3.2; Eq. 2; Eq. 3; Algorithm 1 steps 1-7 without the attention terms).
//
// Kernel ta_mask_kernel works on tiles of the packed token stream. A tile needs no data from other tiles beyond a
// halo of (max span + max pattern length) token ids to its left and (max pattern length) to its right, so the grid
// is embarrassingly parallel and HBM traffic is 4 B read + 5 B written per token.
//   phase a  token ids of tile + halo -> shared memory; per-sequence token histogram via global atomics
//   phase b  warp-parallel multi-pattern match: every lane tests one end position; a 1024-bit filter on the last
//            id of all patterns rejects almost every position before the pattern table is walked; one ballot per 32
//            positions leaves a bitmap of the anchors
//   phase c  span spread: the bitmap's 64 bits before a token, cut off at its sequence's start, name the anchors that can
//            reach it; their vouchers are added nearest anchor first, in fp32 with one rounding per operation (bit-exact by
//            construction)
// What bounds it: latency and instruction issue of blocks that read 4 bytes a token. 524288 tokens with 2048 anchors: 14.2 us
// (17.0 with a segmented max-scan of the anchors' reach in place of the bitmap: five shuffle steps twice and three more barriers).
// Kernel ta_ustatic_kernel then combines recency, anchor flag, frequency and voucher into u_static.
// With a detector's per-token confidences instead of a pattern set (Section 5.1) phase b is a threshold test: the
// anchors are single tokens, all with the same span, and their budget is fixed or proportional to the confidence.
#include "ta_internal.cuh"

namespace {

constexpr int kTile = 512;                                   // tokens per block == threads per block
constexpr int kHaloL = TA_MAX_SPAN + TA_MAX_PATTERN_LEN;     // left halo of token ids
constexpr int kHaloR = TA_MAX_PATTERN_LEN;                   // right halo
constexpr int kExt = kHaloL + kTile + kHaloR;                // ids held in shared memory
constexpr int kWords = (kExt + 31) / 32;                     // of the anchors' bitmap
static_assert(TA_MAX_SPAN == 64 && kHaloL >= 64, "two words of the bitmap before every token of the tile");

__device__ __forceinline__ uint32_t bloom_hash(int32_t x) { return ((uint32_t)x * 2654435761u) >> 22; }

// sequence index of packed token `tok`
__device__ __forceinline__ int seq_of(const ta_seq_desc& s, long long tok) {
  if (!s.cu) return (int)((uint32_t)tok / (uint32_t)s.n_uniform);  // (fewer than 2^31 tokens in all)
  int lo = 0, hi = s.batch;  // cu[lo] <= tok < cu[hi]
  while (hi - lo > 1) {
    const int mid = (lo + hi) >> 1;
    if (s.cu[mid] <= tok) lo = mid; else hi = mid;
  }
  return lo;
}

__device__ __forceinline__ void report(ta_dev_status* st, int code, int where, int d0, int d1) {
  if (atomicCAS(&st->code, 0, code) == 0) {
    st->where = where;
    st->detail0 = d0;
    st->detail1 = d1;
  }
}

// hist = 0. A kernel and not a memset: it can be launched as a programmatic dependent and let its own dependent start.
__global__ void __launch_bounds__(256) ta_clear_kernel(int32_t* __restrict__ hist, long long n) {
  ta_wait_for_prior_grid();
  ta_launch_dependents();
  const long long step = (long long)gridDim.x * blockDim.x, i0 = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  for (long long i = i0; i < n / 4; i += step) reinterpret_cast<int4*>(hist)[i] = make_int4(0, 0, 0, 0);
  for (long long i = n / 4 * 4 + i0; i < n; i += step) hist[i] = 0;
}

struct ConfAnchors {   // anchors from a detector's confidences; conf == nullptr: token-id patterns are matched
  const float* conf;   // [total]
  float threshold;     // anchor iff conf > threshold
  float budget;        // sponsor budget B (rank: B_i = budget * conf_i)
  int span;            // L
  int rank;
};

__global__ void __launch_bounds__(kTile) ta_mask_kernel(ta_seq_desc seq, const int32_t* __restrict__ ids,
                                                        const int32_t* __restrict__ p_ids,
                                                        const int32_t* __restrict__ p_len,
                                                        const float* __restrict__ p_budget,
                                                        const int32_t* __restrict__ p_span,
                                                        const uint32_t* __restrict__ p_bloom, int n_pat,
                                                        int max_len, int max_span, float voucher_decay,
                                                        float budget_decay, int age_steps, int vocab,
                                                        uint8_t* __restrict__ flags, float* __restrict__ voucher,
                                                        int32_t* __restrict__ hist, ta_dev_status* status,
                                                        ConfAnchors ca) {
  __shared__ int32_t s_id[kExt];
  __shared__ int32_t s_start[kExt];     // packed index of the first token of the position's sequence
  __shared__ int16_t s_apat[kExt];      // winning pattern ending here, -1 none
  __shared__ float s_abud[kExt];        // its decayed budget
  __shared__ int32_t s_pid[TA_MAX_PATTERNS * TA_MAX_PATTERN_LEN];
  __shared__ int32_t s_plen[TA_MAX_PATTERNS];
  __shared__ int32_t s_pspan[TA_MAX_PATTERNS];
  __shared__ float s_pbud[TA_MAX_PATTERNS];
  __shared__ uint32_t s_bloom[32];
  __shared__ float s_w[TA_MAX_SPAN + 1];
  __shared__ uint32_t s_bits[kWords + 1];  // bit of every position of the stretch: an anchor ends here

  const int tid = threadIdx.x;
  const long long T0 = (long long)blockIdx.x * kTile;  // first packed token of the tile
  const long long ext0 = T0 - kHaloL;                  // packed token of s_id[0]

  if (ca.conf) {  // one pseudo-pattern of length 1 stands for "the detector fired here"
    if (tid == 0) {
      s_plen[0] = 1;
      s_pspan[0] = ca.span;
      s_pbud[0] = ca.budget;
    }
  } else {
    // the pattern tables: every load is requested before the first is stored (one memory latency for all of them)
    static_assert(TA_MAX_PATTERNS <= kTile && TA_MAX_PATTERNS * TA_MAX_PATTERN_LEN <= 4 * kTile, "slots per thread");
    int32_t r_pid[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int i = tid + q * kTile;
      r_pid[q] = i < n_pat * TA_MAX_PATTERN_LEN ? p_ids[i] : 0;
    }
    const int32_t r_len = tid < n_pat ? p_len[tid] : 0, r_span = tid < n_pat ? p_span[tid] : 0;
    const float r_bud = tid < n_pat ? p_budget[tid] : 0.0f;
    const uint32_t r_bloom = (tid < 32 && n_pat) ? p_bloom[tid] : 0u;
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int i = tid + q * kTile;
      if (i < n_pat * TA_MAX_PATTERN_LEN) s_pid[i] = r_pid[q];
    }
    if (tid < n_pat) {
      s_plen[tid] = r_len;
      s_pspan[tid] = r_span;
      s_pbud[tid] = r_bud;
    }
    if (tid < 32) s_bloom[tid] = r_bloom;
  }
  if (tid <= TA_MAX_SPAN) {  // s_w[k] = decay^k by repeated multiplication (one rounding per step), thread k on its own
    float w = 1.0f;
    for (int k = 0; k < tid; ++k) w = __fmul_rn(w, voucher_decay);
    s_w[tid] = w;
  }

  // Launched as a programmatic dependent of the kernel that clears the histogram, which lets this one start when everything
  // before it is complete: only what follows needs the counters at zero.
  ta_wait_for_prior_grid();
  ta_launch_dependents();
  // phase a: ids + sequence starts for tile and halo; histogram for the tile proper
  for (int i = tid; i < kExt; i += kTile) {
    const long long tok = ext0 + i;
    int32_t id = -1, start = 0;
    if (tok >= 0 && tok < seq.total) {
      id = ids[tok];
      const int b = seq_of(seq, tok);
      start = ta_seq_begin(seq, b);
      if (i >= kHaloL && i < kHaloL + kTile) {
        if (id >= 0 && id < vocab)
          atomicAdd(&hist[(long long)b * vocab + id], 1);
        else
          report(status, TA_ERR_DEVICE_BOUNDS, 1, (int)tok, id);
      }
    }
    s_id[i] = id;
    s_start[i] = start;
  }
  __syncthreads();

  // phase b: which pattern (longest, then lowest index) ends at each position of [T0 - max_span, T0 + kTile + max_len)
  if (tid == 0) s_bits[kWords] = 0u;
  for (int i = tid; i < kWords * 32; i += kTile) {  // (whole warps: one ballot for 32 positions)
    int best = -1, best_len = 0;
    const int32_t x = i < kExt ? s_id[i] : -1;
    float cf = 0.0f;
    if (ca.conf) {
      const long long tok = ext0 + i;
      if (i < kExt && tok >= 0 && tok < seq.total) {
        cf = ca.conf[tok];
        if (cf > ca.threshold) best = 0;  // false for NaN
      }
    } else if (x >= 0 && i >= TA_MAX_PATTERN_LEN) {
      const uint32_t h = bloom_hash(x);
      if (s_bloom[h >> 5] & (1u << (h & 31))) {
        const long long tok = ext0 + i;
        const int avail = (int)min((long long)TA_MAX_PATTERN_LEN, tok - s_start[i] + 1);  // tokens of this sequence up to here
        for (int p = 0; p < n_pat; ++p) {
          const int len = s_plen[p];
          if (len <= best_len || len > avail) continue;
          const int32_t* pid = &s_pid[p * TA_MAX_PATTERN_LEN];
          if (pid[len - 1] != x) continue;
          bool ok = true;
          for (int k = 0; k < len - 1; ++k) ok = ok && (s_id[i - len + 1 + k] == pid[k]);
          if (ok) {
            best = p;
            best_len = len;
          }
        }
      }
    }
    const uint32_t word = __ballot_sync(0xffffffffu, best >= 0);
    if ((tid & 31) == 0) s_bits[i >> 5] = word;
    if (best >= 0) {  // (read only where a bit is set)
      float B = s_pbud[best];
      if (ca.conf && ca.rank) B = __fmul_rn(B, cf);
      for (int t = 0; t < age_steps; ++t) B = __fmul_rn(B, budget_decay);
      s_apat[i] = (int16_t)best;
      s_abud[i] = B;
    }
  }
  __syncthreads();

  // phase c: flags and vouchers for the tile's own tokens
  {
    const int i = kHaloL + tid;  // s_* index
    const long long tok = T0 + tid;
    if (tok < seq.total) {
      const uint32_t* w = s_bits + (i >> 5);
      // S flag: a match ending at e in [tok, tok + max_len) that starts at or before tok
      uint32_t after = __funnelshift_r(w[0], w[1], i & 31);
      const int anchor_end = (int)(after & 1u);
      int anchor_tok = 0;
      for (after &= (1u << max_len) - 1u; after; after &= after - 1u) {
        const int k = __ffs((int)after) - 1;
        if (s_plen[s_apat[i + k]] > k) anchor_tok = 1;
      }
      // bit j: an anchor at position i - 64 + j of the token's own sequence, near enough for the longest span
      unsigned long long before = ((unsigned long long)__funnelshift_r(w[-1], w[0], i & 31) << 32) |
                                  __funnelshift_r(w[-2], w[-1], i & 31);
      const int reach = (int)min((long long)max_span, tok - s_start[i]);
      before = reach <= 0 ? 0ull : before & (~0ull << (64 - min(reach, 64)));
      float V = 0.0f;
      while (before) {
        const int k = __clzll((long long)before) + 1;
        before &= ~(1ull << (64 - k));
        if (k <= s_pspan[s_apat[i - k]]) V = __fadd_rn(V, __fmul_rn(s_abud[i - k], s_w[k]));
      }
      flags[tok] = (uint8_t)((anchor_tok ? TA_FLAG_ANCHOR_TOKEN : 0) | (anchor_end ? TA_FLAG_ANCHOR_END : 0) |
                             (V > 0.0f ? TA_FLAG_SPONSORED : 0));
      voucher[tok] = V;
    }
  }
}

// u_static = ((beta*R + gamma*S) - lambda*F) + V, R = (i0+1)/n, F = count(id)/n  (Eq. 3), one rounding per operation.
__global__ void __launch_bounds__(256) ta_ustatic_kernel(ta_seq_desc seq, const int32_t* __restrict__ ids,
                                                         const uint8_t* flags, const float* voucher,
                                                         const int32_t* hist, int vocab, float beta,
                                                         float gamma, float lambda, float* __restrict__ u_static) {
  ta_wait_for_prior_grid();  // launched as a programmatic dependent of the mask kernel
  const long long tok = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (tok >= seq.total) return;
  const int b = seq_of(seq, tok);
  const int start = ta_seq_begin(seq, b);
  const int n = (seq.cu ? seq.cu[b + 1] : start + seq.n_uniform) - start;
  const int id = ids[tok];
  const int c = (id >= 0 && id < vocab) ? hist[(long long)b * vocab + id] : 0;
  u_static[tok] = ta_static_utility((int)(tok - start), n, c, (flags[tok] & TA_FLAG_ANCHOR_TOKEN) != 0, voucher[tok],
                                    beta, gamma, lambda);
}

}  // namespace

namespace {
template <class Kern, class... Args>
cudaError_t launch_dependent(Kern kern, long long blocks, int threads, cudaStream_t stream, Args... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)blocks, 1, 1);
  cfg.blockDim = dim3((unsigned)threads, 1, 1);
  cfg.stream = stream;
  cudaLaunchAttribute attr[1];
  ta_pdl_attribute(&attr[0]);
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kern, args...);
}

// clears the histogram, runs the mask kernel and (u_static given; otherwise it is left to the forced-set kernel) the
// static-utility kernel
cudaError_t launch_mask_chain(const ta_policy& pol, const ta_seq_desc& seq, const int32_t* ids, const ta_patterns& t,
                              const ConfAnchors& ca, uint8_t* flags, float* voucher, float* u_static, int32_t* hist,
                              ta_dev_status* status, cudaStream_t stream) {
  if (seq.total == 0) return cudaSuccess;
  const long long counters = (long long)seq.batch * pol.vocab_size;
  const long long want = (counters / 4 + 255) / 256;
  cudaError_t e = launch_dependent(ta_clear_kernel, want < 1 ? 1 : want > 1024 ? 1024 : want, 256, stream, hist, counters);
  if (e != cudaSuccess) return e;
  e = launch_dependent(ta_mask_kernel, (seq.total + kTile - 1) / kTile, kTile, stream, seq, ids, (const int32_t*)t.d_ids,
                       (const int32_t*)t.d_len, (const float*)t.d_budget, (const int32_t*)t.d_span,
                       (const uint32_t*)t.d_bloom, t.n_pat, t.max_len, t.max_span, pol.voucher_decay, pol.budget_decay,
                       pol.age_steps, pol.vocab_size, flags, voucher, hist, status, ca);
  if (e != cudaSuccess || !u_static) return e;
  return launch_dependent(ta_ustatic_kernel, (seq.total + 255) / 256, 256, stream, seq, ids, (const uint8_t*)flags,
                          (const float*)voucher, (const int32_t*)hist, pol.vocab_size, pol.beta, pol.gamma, pol.lambda,
                          u_static);
}
}  // namespace

cudaError_t ta_launch_mask_conf(const ta_policy& pol, const ta_seq_desc& seq, const int32_t* ids, const float* conf,
                                float threshold, float budget, int span, int rank, uint8_t* flags, float* voucher,
                                float* u_static, int32_t* hist, ta_dev_status* status, cudaStream_t stream) {
  ta_patterns one = {};  // one pseudo-pattern of length 1 stands for "the detector fired here"
  one.n_pat = 1;
  one.max_len = 1;
  one.max_span = span;
  return launch_mask_chain(pol, seq, ids, one, ConfAnchors{conf, threshold, budget, span, rank}, flags, voucher, u_static,
                           hist, status, stream);
}

cudaError_t ta_launch_mask(const ta_patterns* pats, const ta_policy& pol, const ta_seq_desc& seq, const int32_t* ids,
                           uint8_t* flags, float* voucher, float* u_static, int32_t* hist, ta_dev_status* status,
                           cudaStream_t stream) {
  return launch_mask_chain(pol, seq, ids, *pats, ConfAnchors{nullptr, 0.0f, 0.0f, 0, 0}, flags, voucher, u_static, hist,
                           status, stream);
}
