// Steps 1 and (per-sequence part of) 3 in one kernel, for sequences of up to 16384 tokens: anchor detection, vouchers, the
// attention-free utility (Section 3.2; Eq. 2; Eq. 3; Algorithm 1 steps 1-7 without the attention terms), the forced set of
// Section 3.3 (mandatory tokens and the protected pool) and, in fast mode, the whole selection.
//
// One block of 1024 threads per sequence; token i belongs to thread i mod 1024 in every phase. Everything a phase needs from
// another token sits in shared memory: the ids, the pattern that ends at each position, a bitmap of those positions, and
// the sequence's token histogram (16-bit counters, two per word; in global memory when the vocabulary does not fit).
//   a  ids -> shared memory; counters cleared
//   b  histogram; which pattern (longest, then lowest index) ends at each position, behind a 1024-bit filter on the
//      patterns' last ids; one ballot per 32 positions fills the bitmap
//   c  vouchers: the bitmap's 64 bits before a token name the anchors that can reach it, nearest first; static utility
//   d  forced set (radix select over the vouchers only when there are more sponsored tokens than protected slots)
//   e  fast mode: main pool by utility and the ordered write
// What bounds it: latency (a few barriers, one trip to memory). The same results took a memset and three to five kernels
// (ta_mask.cu, ta_select.cu: still the path for longer sequences, where one block per sequence would be too few), each
// with its own launch, trip to memory and tail: one sequence of 4096 tokens 25.6 -> 11.7 us between events around the stage,
// fast mode with the selection 35.3 -> 12.8 us.
#include <cooperative_groups.h>

#include <atomic>

#include "ta_internal.cuh"

namespace cg = cooperative_groups;

#define TA_SEL_THREADS 1024
#define TA_SEL_NS front1024
#include "ta_select_core.cuh"
#undef TA_SEL_THREADS
#undef TA_SEL_NS

namespace {

using namespace front1024;

constexpr int kPad = TA_MAX_PATTERN_LEN;  // ids before the sequence (never part of a match)
constexpr int kMaxItems = 16;             // tokens per thread
constexpr int kListCap = 256;             // so few sponsored tokens are ranked by comparing them with one another
constexpr int kMaxDynamicSmem = 187 * 1024;  // beside 40 KB of static shared memory (a block may use 227 KB)

struct FrontParams {
  ta_seq_desc seq;
  const int32_t* ids;
  const int32_t* p_ids;
  const int32_t* p_len;
  const float* p_budget;
  const int32_t* p_span;
  const uint32_t* p_bloom;
  int n_pat, max_len, max_span;
  float voucher_decay, budget_decay;
  int age_steps, vocab;
  float beta, gamma, lambda;
  int K, n_sink, n_recent, k_protected;
  int32_t* hist;      // [B][vocab], used when the counters do not fit in shared memory
  uint8_t* forced;    // out (scored)
  float* u_static;    // out (scored)
  int32_t* r_main;    // out (scored)
  int32_t* idx;       // out (fast) [B][K]
  int32_t* count;     // out (fast) [B]
  ta_dev_status* status;
};

// Dynamic shared memory for sequences of up to `items` * 1024 tokens.
struct FrontSmem {
  int ids, apat, bits, hist, end;  // byte offsets
};
__host__ __device__ inline FrontSmem front_smem(int items, int vocab, bool smem_hist) {
  const int n = items * kThreads;
  FrontSmem f;
  f.ids = 0;
  f.bits = f.ids + (kPad + n) * 4;
  f.apat = f.bits + (n / 32 + 4) * 4;  // two words of zeros before and after
  f.hist = f.apat + n * 2;
  f.end = f.hist + (smem_hist ? (vocab + 1) / 2 * 4 : 0);
  return f;
}

template <int ITEMS, bool FAST, bool SMEM_HIST>
__global__ void __launch_bounds__(kThreads, 1) ta_front_kernel(const __grid_constant__ FrontParams p) {
  extern __shared__ __align__(16) unsigned char dyn[];
  __shared__ SelectShared sh;
  __shared__ int32_t s_pid[TA_MAX_PATTERNS * TA_MAX_PATTERN_LEN];
  __shared__ int32_t s_plen[TA_MAX_PATTERNS], s_pspan[TA_MAX_PATTERNS];
  __shared__ float s_pbud[TA_MAX_PATTERNS];
  __shared__ uint32_t s_bloom[32];
  __shared__ float s_w[TA_MAX_SPAN + 1];
  __shared__ uint32_t s_fbits[kMaxItems * kWarps];  // bit of every token: forced
  __shared__ int s_count;
  __shared__ __align__(8) uint2 s_list[kListCap];  // key and position of sponsored, not mandatory tokens
  __shared__ int s_listed;                            // how many there are (also beyond the capacity of the list)
  const FrontSmem L = front_smem(ITEMS, p.vocab, SMEM_HIST);
  int32_t* s_id = reinterpret_cast<int32_t*>(dyn + L.ids) + kPad;       // s_id[-kPad .. n)
  uint32_t* s_bits = reinterpret_cast<uint32_t*>(dyn + L.bits) + 2;     // s_bits[-2 .. n/32 + 2)
  int16_t* s_apat = reinterpret_cast<int16_t*>(dyn + L.apat);
  uint32_t* s_hist = reinterpret_cast<uint32_t*>(dyn + L.hist);

  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int b = blockIdx.x;
  // decay^k by repeated multiplication (one rounding per step), thread k on its own
  if (tid <= TA_MAX_SPAN) {
    float w = 1.0f;
    for (int k = 0; k < tid; ++k) w = __fmul_rn(w, p.voucher_decay);
    s_w[tid] = w;
  }
  if (tid < kPad) s_id[tid - kPad] = -1;
  if (tid < ITEMS * kWarps + 4) s_bits[tid - 2] = 0u;  // also the words of positions behind the sequence
  if (tid == 0) s_count = s_listed = 0;
  if (tid < ITEMS * kWarps) s_fbits[tid] = 0u;
  if (SMEM_HIST)
#pragma unroll 4
    for (int i = tid; i < (p.vocab + 1) / 2; i += kThreads) s_hist[i] = 0u;
  ta_wait_for_prior_grid();
  ta_launch_dependents();

  // ---- a: every load is requested before the first is used
  const SeqInfo s = seq_info(p.seq, b, p.K, p.n_sink, p.n_recent, p.k_protected);
  const int n = s.n;
  int32_t* hist = p.hist + (size_t)b * p.vocab;
  int id[ITEMS];
#pragma unroll
  for (int it = 0; it < ITEMS; ++it) {
    const int i = tid + it * kThreads;
    id[it] = i < n ? p.ids[(long long)s.start + i] : -1;
  }
  int32_t r_pid[2];
#pragma unroll
  for (int q = 0; q < 2; ++q) r_pid[q] = tid + q * kThreads < p.n_pat * TA_MAX_PATTERN_LEN ? p.p_ids[tid + q * kThreads] : 0;
  static_assert(TA_MAX_PATTERNS * TA_MAX_PATTERN_LEN <= 2 * kThreads, "two table entries per thread");
  int32_t r_len = 0, r_span = 0;
  float r_bud = 0.0f;
  if (tid < p.n_pat) {
    r_len = p.p_len[tid];
    r_span = p.p_span[tid];
    r_bud = p.p_budget[tid];
  }
  const uint32_t r_bloom = (tid < 32 && p.n_pat) ? p.p_bloom[tid] : 0u;
#pragma unroll
  for (int q = 0; q < 2; ++q)
    if (tid + q * kThreads < p.n_pat * TA_MAX_PATTERN_LEN) s_pid[tid + q * kThreads] = r_pid[q];
  if (tid < p.n_pat) {
    s_plen[tid] = r_len;
    s_pspan[tid] = r_span;
    for (int t = 0; t < p.age_steps; ++t) r_bud = __fmul_rn(r_bud, p.budget_decay);
    s_pbud[tid] = r_bud;
  }
  if (tid < 32) s_bloom[tid] = r_bloom;
#pragma unroll
  for (int it = 0; it < ITEMS; ++it) {
    const int i = tid + it * kThreads;
    s_id[i] = id[it];
    if (!SMEM_HIST && id[it] >= 0 && id[it] < p.vocab) hist[id[it]] = 0;
  }
  __syncthreads();
  if (s.bad) {
    if (tid == 0) {
      if (atomicCAS(&p.status->code, 0, (int)TA_ERR_DEVICE_BOUNDS) == 0) {
        p.status->where = 3;
        p.status->detail0 = b;
        p.status->detail1 = s.start;
      }
      if (FAST) p.count[b] = 0;
      else p.r_main[b] = -2;  // poisoned: the selection writes an empty result
    }
    if (FAST)
      for (int r = tid; r < p.K; r += kThreads) p.idx[(long long)b * p.K + r] = -1;
    return;
  }

  // The loops over a thread's tokens stay rolled here and in c: one block does the whole sequence, so that the instruction
  // count sets the time (4096 tokens: 11 us unrolled with every key in registers, 9.7 us rolled with a list of the few
  // sponsored tokens).
  // ---- b: histogram and matches
#pragma unroll 1
  for (int it = 0; it * kThreads < n; ++it) {
    const int i = tid + it * kThreads;
    const int x = s_id[i];
    int best = -1;
    bool may_end = false;
    if (i < n) {
      if (x >= 0 && x < p.vocab) {
        if (SMEM_HIST) atomicAdd(&s_hist[x >> 1], (x & 1) ? 0x10000u : 1u);
        else atomicAdd(&hist[x], 1);
      } else if (atomicCAS(&p.status->code, 0, (int)TA_ERR_DEVICE_BOUNDS) == 0) {
        p.status->where = 1;
        p.status->detail0 = s.start + i;
        p.status->detail1 = x;
      }
      const uint32_t h = ((uint32_t)x * 2654435761u) >> 22;
      may_end = x >= 0 && ((s_bloom[h >> 5] >> (h & 31)) & 1u);
    }
    // a position behind the filter is matched by its whole warp, a lane per pattern (one lane with all patterns in turn held
    // the block up: 3.8 K cycles for this phase at 4096 tokens and 8 patterns)
#pragma unroll 1
    for (unsigned left = __ballot_sync(0xffffffffu, may_end); left != 0u; left &= left - 1u) {
      const int src = __ffs((int)left) - 1, end = i - lane + src;
      const int y = __shfl_sync(0xffffffffu, x, src);
      const int avail = min(TA_MAX_PATTERN_LEN, end + 1);  // matches never cross the start of the sequence
      uint32_t mine = 0;                                   // length, then the complement of the index: the largest wins
#pragma unroll 1
      for (int q = lane; q < p.n_pat; q += 32) {
        const int len = s_plen[q];
        const int32_t* pid = &s_pid[q * TA_MAX_PATTERN_LEN];
        if (len > avail || pid[len - 1] != y) continue;
        bool ok = true;
#pragma unroll 1
        for (int k = 0; k < len - 1; ++k) ok = ok && s_id[end - len + 1 + k] == pid[k];
        if (ok) mine = max(mine, ((uint32_t)len << 16) | (uint32_t)(0xffff - q));
      }
      mine = __reduce_max_sync(0xffffffffu, mine);
      if (lane == src && mine != 0u) best = 0xffff - (int)(mine & 0xffffu);
    }
    const unsigned word = __ballot_sync(0xffffffffu, best >= 0);
    if (word) s_apat[i] = (int16_t)best;  // read only where a bit of `word` is set
    if (lane == 0) s_bits[it * kWarps + warp] = word;
  }
  __syncthreads();

  // ---- c: vouchers and static utilities. From here on a thread reads its own ids only: fast mode leaves the utilities in
  // their place.
  float* s_u = reinterpret_cast<float*>(s_id);
  auto mandatory = [&](int i) { return i < s.s_take || i >= s.n - s.r_take; };
  const unsigned long long span_mask = p.max_span >= 64 ? ~0ull : p.max_span <= 0 ? 0ull : ~0ull << (64 - p.max_span);
  // voucher of token i of the warp's word w, nearest anchor first
  auto voucher = [&](const uint32_t* w, int i) {
    // bit j: an anchor at position i - 64 + j
    unsigned long long before = ((unsigned long long)__funnelshift_r(w[-1], w[0], i & 31) << 32) |
                                __funnelshift_r(w[-2], w[-1], i & 31);
    before &= span_mask;
    float V = 0.0f;
#pragma unroll 1
    while (before) {
      const int k = __clzll((long long)before) + 1;
      before &= ~(1ull << (64 - k));
      const int q = s_apat[i - k];
      if (k <= s_pspan[q]) V = __fadd_rn(V, __fmul_rn(s_pbud[q], s_w[k]));
    }
    return V;
  };
#pragma unroll 1
  for (int it = 0; it * kThreads < n; ++it) {
    const int i = tid + it * kThreads;
    const int x = s_id[i];
    const uint32_t* w = s_bits + (i >> 5);  // the same for the whole warp
    float V = 0.0f;
    bool anchor_token = false;
    if ((w[-2] | w[-1] | w[0] | w[1]) != 0u) {  // most warps have no anchor in reach
      V = voucher(w, i);
      // a match that ends at i + k, k < its length, covers this token
      uint32_t after = __funnelshift_r(w[0], w[1], i & 31) & ((1u << p.max_len) - 1u);
#pragma unroll 1
      while (after) {
        const int k = __ffs((int)after) - 1;
        after &= after - 1u;
        anchor_token = anchor_token || s_plen[s_apat[i + k]] > k;
      }
    }
    if (i < n) {
      int c = 0;
      if (x >= 0 && x < p.vocab) {
        if (SMEM_HIST) c = (int)((s_hist[x >> 1] >> ((x & 1) * 16)) & 0xffffu);
        else c = __ldcg(&hist[x]);
      }
      const float u = ta_static_utility(i, n, c, anchor_token, V, p.beta, p.gamma, p.lambda);
      if (FAST) s_u[i] = u;
      else p.u_static[(long long)s.start + i] = u;
      if (V > 0.0f && !mandatory(i)) {
        const int slot = atomicAdd(&s_listed, 1);
        if (slot < kListCap) s_list[slot] = make_uint2(sortable_key(V), (uint32_t)i);
      }
    }
  }
  __syncthreads();

  if (s.K_eff == n) {  // keep everything
    if (FAST) {
      for (int r = tid; r < p.K; r += kThreads) p.idx[(long long)b * p.K + r] = r < n ? r : -1;
      if (tid == 0) p.count[b] = n;
    } else if (tid == 0) {
      p.r_main[b] = -1;
    }
    return;
  }

  // ---- d: the forced set, as bits: the mandatory tokens and the s.p largest vouchers, lower positions first among equals
  KeyCache<ITEMS> kc;
  const int m = s_listed;
  int taken = s.s_take + s.r_take;
  if (m <= kListCap) {
    if (tid < m) {
      const uint2 mine = s_list[tid];
      int before = 0;  // listed tokens that come first
      if (m > s.p)
        for (int j = 0; j < m; ++j) {
          const uint2 o = s_list[j];
          before += o.x > mine.x || (o.x == mine.x && o.y < mine.y);
        }
      if (before < s.p) atomicOr(&s_fbits[mine.y >> 5], 1u << (mine.y & 31));
    }
    taken += min(m, s.p);
  } else {  // many sponsored tokens: radix select over the vouchers, formed again
    uint32_t always = 0;  // the mandatory tokens
    kc.elig = 0;
#pragma unroll
    for (int it = 0; it < ITEMS; ++it) {
      const int i = tid + it * kThreads;
      kc.key[it] = 0u;
      if (i < n) {
        const float V = voucher(s_bits + (i >> 5), i);
        kc.key[it] = sortable_key(V);
        if (mandatory(i)) always |= 1u << it;
        else if (V > 0.0f) kc.elig |= 1u << it;
      }
    }
    const SelectResult r = cached_radix_select<1>(n, n, s.p, kc, sh);
    taken = cached_ordered_emit<1>(n, r, kc, always, [&](int i, int) { atomicOr(&s_fbits[i >> 5], 1u << (i & 31)); }, sh);
  }
  __syncthreads();
  uint32_t fmask = 0;  // bit it: this thread's token of chunk it is forced
#pragma unroll
  for (int it = 0; it < ITEMS; ++it) {
    const int i = tid + it * kThreads;
    const bool f = i < n && (((s_fbits[it * kWarps + warp] >> lane) & 1u) != 0 || mandatory(i));
    if (FAST) fmask |= f ? 1u << it : 0u;
    else if (i < n) p.forced[(long long)s.start + i] = f ? 1 : 0;
  }
  if (!FAST) {
    if (tid == 0) p.r_main[b] = s.K_eff - taken;
    return;
  }

  // ---- e: the main pool by utility among the tokens that are not forced, then all taken positions in order
  int32_t* out = p.idx + (long long)b * p.K;
#pragma unroll
  for (int it = 0; it < ITEMS; ++it) {
    const int i = tid + it * kThreads;
    kc.key[it] = i < n ? sortable_key(s_u[i]) : 0u;
  }
  kc.elig = exist_mask(n) & ~fmask;
  __syncthreads();  // the select state is used a second time
  const SelectResult r2 = cached_radix_select<1>(n, n, s.K_eff - taken, kc, sh);
  const int got = cached_ordered_emit<1>(n, r2, kc, fmask, [&](int i, int rank) {
    if (rank < p.K) out[rank] = i;
  }, sh);
  for (int q = got + tid; q < p.K; q += kThreads) out[q] = -1;
  if (tid == 0) p.count[b] = got;
}

template <int ITEMS, bool FAST>
cudaError_t launch_front(const FrontParams& p, bool smem_hist, cudaStream_t stream) {
  auto kern = smem_hist ? ta_front_kernel<ITEMS, FAST, true> : ta_front_kernel<ITEMS, FAST, false>;
  const int smem = front_smem(ITEMS, p.vocab, smem_hist).end;
  // per device; setting the (sticky) attribute twice from two threads is harmless, the flag only saves the call
  static std::atomic<bool> attr_set[2][64];
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  std::atomic<bool>& set = attr_set[smem_hist ? 1 : 0][dev & 63];
  if (!set.load(std::memory_order_acquire)) {
    e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, kMaxDynamicSmem);
    if (e != cudaSuccess) return e;
    set.store(true, std::memory_order_release);
  }
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)p.seq.batch, 1, 1);
  cfg.blockDim = dim3(kThreads, 1, 1);
  cfg.dynamicSmemBytes = (size_t)smem;
  cfg.stream = stream;
  cudaLaunchAttribute attr[1];
  ta_pdl_attribute(&attr[0]);
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kern, p);
}

}  // namespace

bool ta_front_fits(const ta_seq_desc& seq) { return seq.max_n <= kMaxItems * kThreads; }

cudaError_t ta_launch_front(const ta_patterns* pats, const ta_policy& pol, const ta_select_args& a, const int32_t* ids,
                            int32_t* hist, ta_dev_status* status, cudaStream_t stream) {
  if (a.seq.batch == 0) return cudaSuccess;
  FrontParams p = {};
  p.seq = a.seq;
  p.ids = ids;
  p.p_ids = pats->d_ids;
  p.p_len = pats->d_len;
  p.p_budget = pats->d_budget;
  p.p_span = pats->d_span;
  p.p_bloom = pats->d_bloom;
  p.n_pat = pats->n_pat;
  p.max_len = pats->max_len;
  p.max_span = pats->max_span;
  p.voucher_decay = pol.voucher_decay;
  p.budget_decay = pol.budget_decay;
  p.age_steps = pol.age_steps;
  p.vocab = pol.vocab_size;
  p.beta = pol.beta;
  p.gamma = pol.gamma;
  p.lambda = pol.lambda;
  p.K = a.K;
  p.n_sink = a.n_sink;
  p.n_recent = a.n_recent;
  p.k_protected = a.k_protected;
  p.hist = hist;
  p.forced = a.forced;
  p.u_static = a.static_out;
  p.r_main = a.r_main;
  p.idx = a.idx;
  p.count = a.count;
  p.status = status;
  // the smallest instance that holds the sequences: unused slots cost issue time in every phase
  const int items = a.seq.max_n <= 4 * kThreads ? 4 : a.seq.max_n <= 8 * kThreads ? 8 : 16;
  const bool smem_hist = front_smem(items, pol.vocab_size, true).end <= kMaxDynamicSmem;
  if (a.fast) {
    if (items == 4) return launch_front<4, true>(p, smem_hist, stream);
    if (items == 8) return launch_front<8, true>(p, smem_hist, stream);
    return launch_front<16, true>(p, smem_hist, stream);
  }
  if (items == 4) return launch_front<4, false>(p, smem_hist, stream);
  if (items == 8) return launch_front<8, false>(p, smem_hist, stream);
  return launch_front<16, false>(p, smem_hist, stream);
}
