// Steps 1 and (per-sequence part of) 3 in one kernel, for sequences of up to 262144 tokens: anchor detection, vouchers, the
// attention-free utility (Section 3.2; Eq. 2; Eq. 3; Algorithm 1 steps 1-7 without the attention terms), the forced set of
// Section 3.3 (mandatory tokens and the protected pool) and, in fast mode, the whole selection.
//
// One block of 1024 threads per sequence, or a cluster of them with a slice of the sequence each; token i of a slice belongs to
// thread i mod 1024 in every phase. Everything a phase needs from another token sits in shared memory: the ids (and the ids
// around the slice), the pattern that ends at each position, a bitmap of those positions, and one block's token histogram (16-bit
// counters, two per word; in global memory when the vocabulary does not fit or the sequence is split).
//   a  ids -> shared memory; counters cleared
//   b  histogram; which pattern (longest, then lowest index) ends at each position, behind a 1024-bit filter on the
//      patterns' last ids; one ballot per 32 positions fills the bitmap
//   c  vouchers: the bitmap's 64 bits before a token name the anchors that can reach it, nearest first; static utility
//   d  forced set (radix select over the vouchers only when there are more sponsored tokens than protected slots)
//   e  fast mode: main pool by utility and the ordered write
// What bounds it: latency (a few barriers, one trip to memory). The same results took a memset and three to five kernels
// (ta_mask.cu, ta_select.cu: still the path for longer sequences and for budgets per layer and head), each with its own launch,
// trip to memory and tail: one sequence of 4096 tokens 25.6 -> 11.7 us between events around the stage, fast mode with the
// selection 35.3 -> 12.8 us; four of 131072 tokens 57 -> 35 us a call of one layer with one KV head, 60 of 32768 145 -> 45.
// A slice of 8192 tokens takes 10 K cycles each for the counts with the matches and for the vouchers with the utilities, the search
// among 16 slices 17 K, the rest 16 K. The slices' counts meet in global memory: added up through distributed shared memory (every
// block a share of the vocabulary, the sums handed to all) they took 16 K cycles in place of 5.
#include <cooperative_groups.h>

#include <atomic>

#include "ta_front_rule.h"
#include "ta_internal.cuh"
#include "ta_sm100.cuh"

namespace cg = cooperative_groups;

#define TA_SEL_THREADS 1024
#define TA_SEL_NS front1024
#include "ta_select_core.cuh"
#undef TA_SEL_THREADS
#undef TA_SEL_NS

namespace {

using namespace front1024;

constexpr int kPad = TA_MAX_PATTERN_LEN;  // ids before the sequence (never part of a match)
constexpr int kMaxItems = kFrontMaxItems;
static_assert(kThreads == kFrontThreads, "the rule's block");
constexpr int kListCap = 256;             // so few sponsored tokens are ranked by comparing them with one another
constexpr int kMaxDynamicSmem = 211 * 1024;  // beside at most 16 KB of static shared memory (a block may use 227 KB)
constexpr int kMaxCluster = kFrontMaxCluster;

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
  ta_waits waits;
};

// Dynamic shared memory for sequences of up to `items` * 1024 tokens.
struct FrontSmem {
  int select, ids, apat, bits, hist, end;  // byte offsets
};
__host__ __device__ constexpr int front_halo(int cl) { return cl > 1 ? TA_MAX_SPAN : 0; }
__host__ __device__ inline FrontSmem front_smem(int items, int vocab, bool smem_hist, int cl, size_t select_bytes) {
  const int n = items * kThreads + (cl > 1 ? 32 : 0), halo = front_halo(cl);
  FrontSmem f;
  f.select = 0;
  f.ids = (int)(select_bytes + 15) / 16 * 16;
  f.bits = f.ids + (kPad + halo + n) * 4;
  f.apat = f.bits + (n / 32 + 4) * 4;  // two words of zeros before and after
  f.hist = (f.apat + (halo + n) * 2 + 15) / 16 * 16;
  f.end = f.hist + (smem_hist ? (vocab + 7) / 8 * 16 : 0);
  return f;
}

template <int ITEMS, bool FAST, bool SMEM_HIST, int CL>
__global__ void __launch_bounds__(kThreads, 1) ta_front_kernel(const __grid_constant__ FrontParams p) {
  extern __shared__ __align__(16) unsigned char dyn[];
  __shared__ int32_t s_pid[TA_MAX_PATTERNS * TA_MAX_PATTERN_LEN];
  __shared__ int32_t s_plen[TA_MAX_PATTERNS], s_pspan[TA_MAX_PATTERNS];
  __shared__ float s_pbud[TA_MAX_PATTERNS];
  __shared__ uint32_t s_bloom[32];
  __shared__ float s_w[TA_MAX_SPAN + 1];
  __shared__ uint32_t s_fbits[kMaxItems * kWarps];  // bit of every token: forced
  __shared__ __align__(8) uint2 s_list[kListCap];  // key and position of sponsored, not mandatory tokens
  __shared__ __align__(8) int s_sponsored[CL][2];     // CL > 1: sponsored, not mandatory tokens of every slice
  __shared__ int s_listed;                            // how many there are (also beyond the capacity of the list)
  constexpr int kHalo = front_halo(CL);  // positions before the slice whose matches reach into it
  const FrontSmem L = front_smem(ITEMS, p.vocab, SMEM_HIST, CL, sizeof(SelectShared<CL>));
  SelectShared<CL>& sh = *reinterpret_cast<SelectShared<CL>*>(dyn + L.select);
  int32_t* s_id = reinterpret_cast<int32_t*>(dyn + L.ids) + kPad + kHalo;  // s_id[-kPad - kHalo .. n)
  uint32_t* s_bits = reinterpret_cast<uint32_t*>(dyn + L.bits) + 2;        // s_bits[-2 .. n/32 + 2)
  int16_t* s_apat = reinterpret_cast<int16_t*>(dyn + L.apat) + kHalo;
  uint32_t* s_hist = reinterpret_cast<uint32_t*>(dyn + L.hist);

  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int b = blockIdx.x / CL;
  // decay^k by repeated multiplication (one rounding per step), thread k on its own
  if (tid <= TA_MAX_SPAN) {
    float w = 1.0f;
    for (int k = 0; k < tid; ++k) w = __fmul_rn(w, p.voucher_decay);
    s_w[tid] = w;
  }
  if (CL == 1 && tid < kPad) s_id[tid - kPad] = -1;
  if (tid < ITEMS * kWarps + 4) s_bits[tid - 2] = 0u;  // also the words of positions behind the sequence
  if (tid == 0) s_listed = 0;
  if (tid < ITEMS * kWarps) s_fbits[tid] = 0u;
  if (SMEM_HIST)
#pragma unroll 4
    for (int i = tid; i < (p.vocab + 7) / 8; i += kThreads) reinterpret_cast<uint4*>(s_hist)[i] = make_uint4(0u, 0u, 0u, 0u);
  Exchange<CL> ex{p.waits};
  if constexpr (CL > 1) ex.set_up(sh);
  ta_wait_for_prior_grid();
  ta_launch_dependents();

  // ---- a: every load is requested before the first is used
  const SeqInfo s = seq_info(p.seq, b, p.K, p.n_sink, p.n_recent, p.k_protected);
  const int n = s.n;
  // this CTA's slice: tokens [lo, lo + nl); local index i <-> position lo + i. Whole words of the bitmap.
  const int per = CL == 1 ? n : ((n + CL - 1) / CL + 31) / 32 * 32;
  const int rank = CL == 1 ? 0 : (int)cg::this_cluster().block_rank();
  const int lo = CL == 1 ? 0 : min(n, rank * per), nl = CL == 1 ? n : min(n - lo, per);
  const int nx = CL == 1 ? n : min(nl + TA_MAX_PATTERN_LEN, n - lo);  // with the tokens whose matches can cover the slice's last
  int32_t* hist = p.hist + (size_t)b * p.vocab;
  const int32_t* ids = p.ids + (long long)s.start + lo;
  int id[ITEMS];
#pragma unroll
  for (int it = 0; it < ITEMS; ++it) {
    const int i = tid + it * kThreads;
    id[it] = i < nx ? ids[i] : -1;
  }
  // the tokens before the slice that can match into it, and those behind it that do not fit the threads' slots
  const int i_halo = tid < kPad + kHalo ? tid - kPad - kHalo : ITEMS * kThreads + tid - kPad - kHalo;
  int id_halo = -1;
  if (CL > 1 && tid < kPad + kHalo + kPad && lo + i_halo >= 0 && i_halo < nx) id_halo = ids[i_halo];
  int32_t r_pid[2];
#pragma unroll
  for (int q = 0; q < 2; ++q) r_pid[q] = tid + q * kThreads < p.n_pat * TA_MAX_PATTERN_LEN ? p.p_ids[tid + q * kThreads] : 0;
  static_assert(CL == 1 || !SMEM_HIST, "the counters of one block");
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
    if (CL == 1 && !SMEM_HIST && id[it] >= 0 && id[it] < p.vocab) hist[id[it]] = 0;
  }
  if (CL > 1 && tid < kPad + kHalo + kPad) s_id[i_halo] = id_halo;
  if constexpr (CL > 1) {  // every CTA clears its share of the sequence's counters
    const int share = (p.vocab + CL - 1) / CL, end = min(p.vocab, (rank + 1) * share);
    for (int i = rank * share + tid; i < end; i += kThreads) hist[i] = 0;
    cg::this_cluster().sync();
  } else {
    __syncthreads();
  }
  if (s.bad) {
    if (tid == 0) {
      if (atomicCAS(&p.waits.status->code, 0, (int)TA_ERR_DEVICE_BOUNDS) == 0) {
        p.waits.status->where = 3;
        p.waits.status->detail0 = b;
        p.waits.status->detail1 = s.start;
      }
      if (FAST) p.count[b] = 0;
      else p.r_main[b] = -2;  // poisoned: the selection writes an empty result
    }
    if (FAST && rank == 0)
      for (int r = tid; r < p.K; r += kThreads) p.idx[(long long)b * p.K + r] = -1;
    return;
  }

  // The loops over a thread's tokens stay rolled here and in c: one block does the whole sequence, so that the instruction
  // count sets the time (4096 tokens: 11 us unrolled with every key in registers, 9.7 us rolled with a list of the few
  // sponsored tokens).
  // ---- b: histogram and matches
#pragma unroll 1
  for (int it = CL == 1 ? 0 : -1; it * kThreads < nx; ++it) {  // (chunk -1: the positions before a slice)
    const int i = tid + it * kThreads;
    if (CL > 1 && (i - lane < -kHalo || i - lane >= nx)) continue;  // (whole warps; the words behind the slice are zero)
    const int x = CL == 1 || i < nx ? s_id[i] : -1;
    int best = -1;
    bool may_end = false;
    if (i < nx) {
      if (CL > 1 && (i < 0 || i >= nl)) {
        // another CTA counts it
      } else if (x >= 0 && x < p.vocab) {
        if (SMEM_HIST) atomicAdd(&s_hist[x >> 1], (x & 1) ? 0x10000u : 1u);
        else atomicAdd(&hist[x], 1);
      } else if (atomicCAS(&p.waits.status->code, 0, (int)TA_ERR_DEVICE_BOUNDS) == 0) {
        p.waits.status->where = 1;
        p.waits.status->detail0 = s.start + lo + i;
        p.waits.status->detail1 = x;
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
      const int avail = min(TA_MAX_PATTERN_LEN, lo + end + 1);  // matches never cross the start of the sequence
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
  if constexpr (CL == 1) {
    __syncthreads();
  } else {
    cg::this_cluster().sync();  // the sequence's counts are complete
  }

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
  for (int it = 0; it * kThreads < nl; ++it) {
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
    if (i < nl) {
      int c = 0;
      if (x >= 0 && x < p.vocab) {
        if (SMEM_HIST) c = (int)((s_hist[x >> 1] >> ((x & 1) * 16)) & 0xffffu);
        else c = __ldcg(&hist[x]);
      }
      const float u = ta_static_utility(lo + i, n, c, anchor_token, V, p.beta, p.gamma, p.lambda);
      if (FAST) s_u[i] = u;
      else p.u_static[(long long)s.start + lo + i] = u;
      if (CL > 1 && !FAST) p.forced[(long long)s.start + lo + i] = 0;  // what a wait that runs out leaves: no flags of an earlier call
      if (CL == 1 && V > 0.0f && !mandatory(i)) {
        const int slot = atomicAdd(&s_listed, 1);
        if (slot < kListCap) s_list[slot] = make_uint2(sortable_key(V), (uint32_t)i);
      }
    }
    if (CL > 1) {  // the sponsored, not mandatory tokens as bits: forced if the cluster's fit the protected slots
      const unsigned sponsored = __ballot_sync(0xffffffffu, i < nl && V > 0.0f && !mandatory(lo + i));
      if (lane == 0 && sponsored != 0u) {
        s_fbits[it * kWarps + warp] = sponsored;
        atomicAdd(&s_listed, __popc(sponsored));
      }
    }
  }
  __syncthreads();

  if (s.K_eff == n) {  // keep everything
    if (rank != 0) return;
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
  int m = s_listed;
  int taken = s.s_take + s.r_take;
  if constexpr (CL > 1) {
    if (tid == 0 && rank == 0) {  // what a wait that runs out leaves: an empty result
      if (FAST) p.count[b] = 0;
      else p.r_main[b] = -2;
    }
    if (tid < CL) ex.send2(sh, s_sponsored[rank], tid, (uint32_t)m, 0u);
    ex.wait(sh, CL * 8);
    m = 0;
#pragma unroll
    for (int q = 0; q < CL; ++q) m += s_sponsored[q][0];
  }
  if (CL > 1 && m <= s.p) {
    taken += m;  // (the bits are there)
  } else if (CL == 1 && m <= kListCap) {
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
      if (i < nl) {
        const float V = voucher(s_bits + (i >> 5), i);
        kc.key[it] = sortable_key(V);
        if (mandatory(lo + i)) always |= 1u << it;
        else if (V > 0.0f) kc.elig |= 1u << it;
      }
    }
    if (CL > 1 && tid < ITEMS * kWarps) s_fbits[tid] = 0u;  // (set again below, several barriers later)
    const SelectResult r = cached_radix_select<CL>(nl, n, s.p, kc, sh, ex);
    taken = cached_ordered_emit<CL>(nl, r, kc, always, [&](int i, int) { atomicOr(&s_fbits[i >> 5], 1u << (i & 31)); }, sh, ex);
  }
  __syncthreads();
  uint32_t fmask = 0;  // bit it: this thread's token of chunk it is forced
#pragma unroll
  for (int it = 0; it < ITEMS; ++it) {
    const int i = tid + it * kThreads;
    const bool f = i < nl && (((s_fbits[it * kWarps + warp] >> lane) & 1u) != 0 || mandatory(lo + i));
    if (FAST) fmask |= f ? 1u << it : 0u;
    else if (i < nl) p.forced[(long long)s.start + lo + i] = f ? 1 : 0;
  }
  if (!FAST) {
    if (tid == 0 && rank == 0) p.r_main[b] = s.K_eff - taken;
    return;
  }

  // ---- e: the main pool by utility among the tokens that are not forced, then all taken positions in order
  int32_t* out = p.idx + (long long)b * p.K;
#pragma unroll
  for (int it = 0; it < ITEMS; ++it) {
    const int i = tid + it * kThreads;
    kc.key[it] = i < nl ? sortable_key(s_u[i]) : 0u;
  }
  kc.elig = exist_mask(nl) & ~fmask;
  __syncthreads();  // the select state is used a second time
  const SelectResult r2 = cached_radix_select<CL>(nl, n, s.K_eff - taken, kc, sh, ex);
  const int got = cached_ordered_emit<CL>(nl, r2, kc, fmask, [&](int i, int place) {
    if (place < p.K) out[place] = lo + i;
  }, sh, ex);
  if (rank != 0) return;
  for (int q = got + tid; q < p.K; q += kThreads) out[q] = -1;
  if (tid == 0) p.count[b] = min(got, p.K);
}

// An instance made ready for launching, and how many of its clusters the current device holds at once (0: none).
template <int ITEMS, bool FAST, int CL>
struct FrontInstance {
  bool smem_hist;
  int smem;
  using Kernel = void (*)(const FrontParams);
  Kernel kern;

  explicit FrontInstance(int vocab) {
    smem_hist = CL == 1 && front_smem(ITEMS, vocab, true, CL, sizeof(SelectShared<CL>)).end <= kMaxDynamicSmem;
    kern = smem_hist ? ta_front_kernel<ITEMS, FAST, CL == 1, CL> : ta_front_kernel<ITEMS, FAST, false, CL>;
    smem = front_smem(ITEMS, vocab, smem_hist, CL, sizeof(SelectShared<CL>)).end;
  }
  void configure(cudaLaunchConfig_t* cfg, cudaLaunchAttribute* attr) const {  // room for one attribute
    cfg->blockDim = dim3(kThreads, 1, 1);
    cfg->dynamicSmemBytes = (size_t)smem;
    cfg->attrs = attr;
    cfg->numAttrs = 0;
    if (CL > 1) {
      attr[0].id = cudaLaunchAttributeClusterDimension;
      attr[0].val.clusterDim.x = (unsigned)CL;
      attr[0].val.clusterDim.y = 1;
      attr[0].val.clusterDim.z = 1;
      cfg->numAttrs = 1;
    }
  }
  // per device; doing it twice from two threads is harmless (the attributes are sticky), what is kept only saves the calls
  cudaError_t ready(int* clusters) const {
    static std::atomic<int> known[2][64];  // 1 + clusters
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    std::atomic<int>& k = known[smem_hist ? 1 : 0][dev & 63];
    int have = k.load(std::memory_order_acquire);
    if (have == 0) {
      e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, kMaxDynamicSmem);
      if (e == cudaSuccess && CL > 8) e = cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
      if (e != cudaSuccess) return e;
      int n = 1;
      if (CL > 1) {
        cudaLaunchConfig_t cfg = {};
        cudaLaunchAttribute attr[1];
        configure(&cfg, attr);
        cfg.gridDim = dim3(CL, 1, 1);
        if (cudaOccupancyMaxActiveClusters(&n, kern, &cfg) != cudaSuccess) {
          cudaGetLastError();  // a size that the device does not have
          n = 0;
        }
      }
      have = 1 + n;
      k.store(have, std::memory_order_release);
    }
    *clusters = have - 1;
    return cudaSuccess;
  }
  cudaError_t launch(const FrontParams& p, cudaStream_t stream) const {
    int clusters = 0;
    cudaError_t e = ready(&clusters);
    if (e != cudaSuccess) return e;
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute attr[2];
    configure(&cfg, attr);
    cfg.gridDim = dim3((unsigned)(p.seq.batch * CL), 1, 1);
    cfg.stream = stream;
    ta_pdl_attribute(&attr[cfg.numAttrs++]);
    return cudaLaunchKernelEx(&cfg, kern, p);
  }
};

// f(the smallest instance that holds the slices): unused slots cost issue time in every phase
template <bool FAST, int CL, class F>
cudaError_t with_items(const FrontParams& p, F f) {
  const int items = (p.seq.max_n + CL * kThreads - 1) / (CL * kThreads);
  if (CL != 2 && items <= 4) return f(FrontInstance<CL == 2 ? kMaxItems : 4, FAST, CL>(p.vocab));
  if (CL != 2 && items <= 8) return f(FrontInstance<CL == 2 ? kMaxItems : 8, FAST, CL>(p.vocab));
  return f(FrontInstance<kMaxItems, FAST, CL>(p.vocab));
}
template <bool FAST, class F>
cudaError_t with_instance(const FrontParams& p, int blocks, F f) {
  switch (blocks) {
    case 1: return with_items<FAST, 1>(p, f);
    case 2: return with_items<FAST, 2>(p, f);
    case 4: return with_items<FAST, 4>(p, f);
    case 8: return with_items<FAST, 8>(p, f);
    default: return with_items<FAST, kMaxCluster>(p, f);
  }
}

template <bool FAST>
cudaError_t launch_split(const FrontParams& p, int sms, int score_units, bool* launched, cudaStream_t stream) {
  cudaError_t e = cudaSuccess;
  const int blocks = ta_front_blocks(p.seq.max_n, p.seq.batch, sms, score_units, FAST, [&](int cl) {
    int clusters = 0;
    const cudaError_t r = with_instance<FAST>(p, cl, [&](const auto& inst) { return inst.ready(&clusters); });
    if (r != cudaSuccess) e = r;
    return r == cudaSuccess ? clusters : 0;
  });
  *launched = blocks > 0;
  if (e != cudaSuccess || blocks == 0) return e;
  return with_instance<FAST>(p, blocks, [&](const auto& inst) { return inst.launch(p, stream); });
}

}  // namespace

cudaError_t ta_launch_front(const ta_patterns* pats, const ta_policy& pol, const ta_select_args& a, const int32_t* ids,
                            int32_t* hist, ta_dev_status* status, bool* launched, cudaStream_t stream) {
  *launched = true;
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
  p.waits = {status, ta_wait_limit(a.wait_limit_ns)};
  const int sms = a.sm_count > 0 ? a.sm_count : 148;
  return a.fast ? launch_split<true>(p, sms, 0, launched, stream) : launch_split<false>(p, sms, a.score_units, launched, stream);
}
