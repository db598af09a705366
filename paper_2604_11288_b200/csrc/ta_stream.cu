// Algorithm 1 in the decode loop: one new token per sequence and step, at most K cached tokens per unit afterwards.
// (Section 3.1: a retention policy selects S, |S| <= K, "after each generation step"; Algorithm 1 steps 1-10.)
//
// Per step one kernel runs, ta_stream_step_kernel, a block per unit with its K+1 entries in registers. The block of a sequence's
// first unit works out what the step means for the sequence (pattern match ending at the new token: longest pattern wins, then
// the lowest index; the new token's voucher from the anchors of the last TA_MAX_SPAN positions, Eq. 2 with budgets that decayed
// once per step since detection: a lane per anchor), tells the blocks of the sequence's other units, in two words that each of
// them clears again (a counter of those that have read took 0.8 ns a block), and brings the state that they share (histogram,
// last ids, anchors, tokens seen) up to date: they read none of it but counts of other ids than the new one. Every block appends
// the new token to its unit's position-ordered state, adds this step's attention mass to A, updates the pension average P, forms
// the utility of Eq. 1, applies the budget partition of Section 3.3 to the K+1 cached tokens (exactly one token loses), removes it
// from the ordered state (4-byte entries move; key/value rows never do: the freed cache row is handed to the next token) and
// decays every voucher by budget_decay (Algorithm 1 step 10). A block whose words do not come in time leaves its unit as it is.
// The attention masses go to shared memory by asynchronous copies, which hold no registers and which nothing waits for before the
// block's first barrier (loads that a store to shared memory follows held the loads of the next entry back).
// (A kernel of its own for the sequences, in front of this one, cost its launch and tail. GPU time of a step in us with it / as one
// kernel that loads the masses / now: 8 units of 17 tokens 4.9 / 5.4 / 4.6, of 257 5.5 / 6.0 / 5.0, of 1001 6.4 / 6.7 / 5.9; 1024
// units of 257 7.7 / 7.4 / 6.2, of 1001 19.5 / 17.5 / 16.2; 4096 of 257 19.0 / 17.6 / 16.7.)
// What bounds it: latency at few units, the state's bytes (25 read, 12 to 25 written per cached token, 4 of attention
// mass read) at many. 4096 units of 257 tokens, three states in turn (180 MB: more than L2), where the tokens with a voucher fit
// the protected slots, and where all compete for a quarter of the slots (the extremes of what a generation meets): 31 and 70 us
// with serial scans by one thread in the pool selection, one lane per sequence for the voucher and all entries through shared
// memory; 22 with two entries in 64 registers, of which an SM held 6 blocks; 18.5 and 25.6 with three in 56; 16.5 and 24 now.
// All arithmetic that decides the selection is fp32 with one rounding per operation, in the order the CPU oracle uses.
#include "ta_internal.cuh"

namespace {

__device__ __forceinline__ void report(ta_dev_status* st, int code, int where, int d0, int d1) {
  if (atomicCAS(&st->code, 0, code) == 0) {
    st->where = where;
    st->detail0 = d0;
    st->detail1 = d1;
  }
}

constexpr unsigned long long kPublished = 1ull << 63;

struct PatternTable {
  const int32_t* ids;
  const int32_t* len;
  const float* budget;
  const int32_t* span;
  int n;
};

// What the new token means for its sequence; one warp, the same on every lane.
struct SeqStep {
  int t;          // position of the new token
  int match_len;  // tokens t - match_len + 1 .. t belong to a pattern completed by the new token (0: none)
  float v_new;    // voucher of the new token
  int count;      // earlier occurrences of its id
  int best;       // the pattern that it completes (-1: none)
};
// Everything is requested before the first value is used, by place in the rings and not by distance from the new token: one trip
// to memory (two for the count and for patterns beyond the first 32).
__device__ __forceinline__ SeqStep sequence_step(const ta_stream_dev& st, const PatternTable& pt, int b, int x, int vocab,
                                                 float voucher_decay, float budget_decay) {
  constexpr int kHalves = TA_MAX_SPAN / 32;
  static_assert(TA_MAX_SPAN == 64 && TA_MAX_PATTERN_LEN == 8, "two anchors per lane, eight ids in registers");
  const unsigned all = 0xffffffffu;
  const int lane = threadIdx.x & 31;
  SeqStep r;
  r.t = __ldcg(&st.n_seen[b]);
  int L[kHalves];
  float Bk[kHalves];
#pragma unroll
  for (int h = 0; h < kHalves; ++h) {
    L[h] = __ldcg(&st.anc_L[(size_t)b * TA_MAX_SPAN + 32 * h + lane]);
    Bk[h] = __ldcg(&st.anc_B[(size_t)b * TA_MAX_SPAN + 32 * h + lane]);
  }
  const int last = __ldcg(&st.tok_ring[(size_t)b * TA_MAX_PATTERN_LEN + (lane & 7)]);
  int len = lane < pt.n ? pt.len[lane] : 0;
  const int4 none = make_int4(0, 0, 0, 0);
  int4 p0 = lane < pt.n ? reinterpret_cast<const int4*>(pt.ids)[2 * lane] : none;
  int4 p1 = lane < pt.n ? reinterpret_cast<const int4*>(pt.ids)[2 * lane + 1] : none;
  r.count = x >= 0 && x < vocab ? __ldcg(&st.hist[(size_t)b * vocab + x]) : 0;
  const int t = r.t;
  int ids[TA_MAX_PATTERN_LEN];  // ids[k]: the token k positions before the new one
  ids[0] = x;
#pragma unroll
  for (int k = 1; k < TA_MAX_PATTERN_LEN; ++k) {
    const int id = __shfl_sync(all, last, (t - k) & 7);
    ids[k] = k <= t ? id : -1;
  }
  // patterns ending at t: the longest, of equal lengths the lowest index
  uint32_t mine = 0;
#pragma unroll 1
  for (int p = lane;;) {
    const int pid[TA_MAX_PATTERN_LEN] = {p0.x, p0.y, p0.z, p0.w, p1.x, p1.y, p1.z, p1.w};
    bool ok = len > 0 && len <= t + 1;
#pragma unroll
    for (int m = 0; m < TA_MAX_PATTERN_LEN; ++m) {  // id m of the pattern against the token len - 1 - m positions back
      int id = ids[0];
#pragma unroll
      for (int k = 1; k < TA_MAX_PATTERN_LEN; ++k) id = len - 1 - m == k ? ids[k] : id;
      ok = ok && (m >= len || pid[m] == id);
    }
    if (ok) mine = max(mine, ((uint32_t)len << 16) | (uint32_t)(0xffff - p));
    p += 32;
    if (p - lane >= pt.n) break;
    len = p < pt.n ? pt.len[p] : 0;
    p0 = p < pt.n ? reinterpret_cast<const int4*>(pt.ids)[2 * p] : none;
    p1 = p < pt.n ? reinterpret_cast<const int4*>(pt.ids)[2 * p + 1] : none;
  }
  static_assert(TA_MAX_PATTERNS <= 0xffff, "an index in 16 bits");
  mine = __reduce_max_sync(all, mine);
  r.match_len = (int)(mine >> 16);  // the longest matching pattern covers the tokens of every pattern that ends here
  r.best = mine ? 0xffff - (int)(mine & 0xffffu) : -1;
  // voucher of the new token from the anchors at t-1, t-2, ..: every lane its own terms, summed nearest first
  r.v_new = 0.0f;
  int k[kHalves];  // distance of the lane's anchors; one that does not reach the new token: farther than any
  float term[kHalves];
#pragma unroll
  for (int h = 0; h < kHalves; ++h) {
    k[h] = ((t - (32 * h + lane) - 1) & (TA_MAX_SPAN - 1)) + 1;
    if (!(k[h] <= t && L[h] > 0 && k[h] <= L[h])) k[h] = TA_MAX_SPAN + 1;
    term[h] = 0.0f;
    if (k[h] <= TA_MAX_SPAN) {
      float w = 1.0f;  // decay^k by repeated multiplication (one rounding per step), like the budget's
#pragma unroll 1
      for (int s = 0; s < k[h]; ++s) {
        Bk[h] = __fmul_rn(Bk[h], budget_decay);
        w = __fmul_rn(w, voucher_decay);
      }
      term[h] = __fmul_rn(Bk[h], w);
    }
  }
#pragma unroll 1
  for (;;) {
    const int near = __reduce_min_sync(all, min(k[0], k[1]));
    if (near > TA_MAX_SPAN) break;
    const unsigned in0 = __ballot_sync(all, k[0] == near), in1 = __ballot_sync(all, k[1] == near);
    const float add = in0 ? __shfl_sync(all, term[0], __ffs((int)in0) - 1) : __shfl_sync(all, term[1], __ffs((int)in1) - 1);
    r.v_new = __fadd_rn(r.v_new, add);
#pragma unroll
    for (int h = 0; h < kHalves; ++h)
      if (k[h] == near) k[h] = TA_MAX_SPAN + 1;
  }
  return r;
}
// the two words of a sequence: voucher and match length; position and earlier occurrences
__device__ __forceinline__ ulonglong2 seq_words(const SeqStep& r) {
  return make_ulonglong2(kPublished | ((unsigned long long)r.match_len << 32) | __float_as_uint(r.v_new),
                         kPublished | ((unsigned long long)r.t << 32) | (uint32_t)r.count);
}
__device__ __forceinline__ bool step_gave_up(const ta_dev_status* status) { return *(volatile const int*)&status->step_gave_up != 0; }
// One word, once it is there; 0 if the wait runs out. (The block that writes it has a lower index than every block that waits
// for it.) With one wait that ran out the others of this step end too, and no later step of the context touches its state until
// the host has polled and cleared the words: one that came late must not be taken for the next step's.
__device__ __forceinline__ unsigned long long wait_word(const unsigned long long* word, unsigned long long limit_ns,
                                                        ta_dev_status* status, int u) {
  unsigned long long w, t0 = 0;
  for (int it = 0; ((w = *(volatile const unsigned long long*)word) & kPublished) == 0; ++it) {
    if ((it & 63) != 63) continue;
    if (step_gave_up(status)) return 0ull;
    unsigned long long now;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(now));
    if (t0 == 0) t0 = now;
    if (now - t0 > limit_ns) {
      report(status, TA_ERR_TIMEOUT, 7, u, 0);
      *(volatile int*)&status->step_gave_up = 1;
      return 0ull;
    }
  }
  return w;
}
// The self-test's first units: for longer than the others wait.
__device__ __forceinline__ void hold_words(unsigned long long ns) {
  unsigned long long t0, now;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t0));
  do {
    __nanosleep(1000);
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(now));
  } while (now - t0 < ns);
}

// four bytes to shared memory without a register and without waiting for them
__device__ __forceinline__ void copy_async4(float* to_shared, const float* from) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"((uint32_t)__cvta_generic_to_shared(to_shared)), "l"(from));
}
__device__ __forceinline__ void copy_async_wait() { asm volatile("cp.async.wait_all;" ::: "memory"); }

__device__ __forceinline__ uint32_t sortable_key(float f) {
  uint32_t b = __float_as_uint(f);
  if ((b << 1) == 0u) b = 0u;  // -0 == +0
  return (b & 0x80000000u) ? ~b : (b | 0x80000000u);
}

// The largest block per number of entries in a thread, which at two blocks an SM sets the registers: 56 with three
// entries, 64 with four. The step is bound by how many blocks' loads are in flight, so registers are traded for blocks
// until values spill in the common path (time of 4096 units in us, entries/registers):
//   tokens   2/64   2/40   3/77   3/64   3/56   3/48   4/76   4/64   5/64
//      257   22.0   20.7   21.2   18.3   18.6   20.1   21.8   19.9   21.6
//      513   44.5   37.6   41.5   38.3   35.7   38.9   44.2   37.2   40.8
//     1001   71.6   65.5   80.8   82.8   68.1   74.2   71.9   62.5   77.0
//     1501      -      -      -   94.4   97.8  106.8  101.5  106.9  107.2
//     2041      -      -      -      -      -      -  183.4  123.5  156.1
__host__ __device__ constexpr int step_threads(int e) { return e == 3 ? 576 : e == 4 ? 512 : 480; }
constexpr int step_regs(int e) { return e == 3 ? 56 : 64; }
// warps of the largest block: what the shared arrays are sized for
__host__ __device__ constexpr int step_warps(int e) { return step_threads(e) / 32; }

// Entries per thread for units of C cached tokens: three or four, whichever lets an SM hold more blocks (three when equal:
// fewer spills); nine where a block would have to be larger than those kernels allow: the largest unit, of 4097 tokens, then has
// 480 threads, which leaves them the registers that eight entries in 544 did not have (104 bytes spilled; us with eight / nine:
// 8 units of 2049 tokens 11.3 / 8.1, of 4001 13.0 / 10.9; 1024 units 60.7 / 41.6 and 111 / 79.7).
constexpr int step_block(int C, int e) { return ((C + e - 1) / e + 31) / 32 * 32; }
constexpr int step_resident(int C, int e) {
  return step_block(C, e) <= step_threads(e) ? 65536 / (step_block(C, e) * step_regs(e)) : 0;
}
constexpr int step_items(int C) {
  const int r3 = step_resident(C, 3), r4 = step_resident(C, 4);
  return r3 == 0 && r4 == 0 ? 9 : r3 >= r4 ? 3 : 4;
}
// every block that the rule can choose holds its unit and is no larger than its kernel's arrays and launch bounds
constexpr bool step_shapes_fit() {
  for (int C = 2; C <= TA_MAX_BUDGET + 1; ++C) {
    const int e = step_items(C), nt = step_block(C, e);
    if (nt * e < C || nt > step_threads(e) || nt / 32 > step_warps(e) || nt > 1024) return false;
  }
  return true;
}
static_assert(step_shapes_fit(), "a budget for which the step's block does not fit its kernel");

// the units of one launch: layers l0 .. l0 + nl - 1, sequences b0 .. b0 + nb - 1, KV heads g0 .. g0 + ng - 1
struct StreamPart {
  int l0, nl, b0, nb, g0, ng;
  int update;  // the sequences' last launch
};

// One block per unit; thread tid holds the entries tid, tid + nt, .. (E of them) in registers for the whole step.
// Selection (Section 3.3 on the K+1 cached tokens): mandatory sinks and recents; the protected pool = the sponsored,
// non-mandatory tokens with the largest vouchers (lower position first among equals); exactly one token is then not
// forced and loses: the one with the smallest utility, the latest position among equals. When the sponsored tokens fit the
// protected slots, or are one too many, block-wide minima decide; otherwise a radix select on the voucher keys.
template <int E>
__global__ void __launch_bounds__(step_threads(E), E == 9 ? 1 : 2)
ta_stream_step_kernel(ta_stream_dev st, PatternTable pt, const int32_t* new_ids, const float* attn, ta_stream_sync sync,
                      StreamPart part, int vocab, float voucher_decay, float alpha, float beta, float gamma, float delta,
                      float lambda, float rho, float budget_decay, int n_sink, int n_recent, int k_protected,
                      int32_t* __restrict__ evicted_pos, ta_dev_status* status) {
  extern __shared__ __align__(16) unsigned char smem[];
  // by layer, sequence, head: every sequence's first block comes before those that wait for it
  const int lb = blockIdx.x / part.ng, g = part.g0 + blockIdx.x - lb * part.ng, bi = lb % part.nb, b = part.b0 + bi;
  const int u = ((part.l0 + lb / part.nb) * st.B + b) * st.Hkv + g;
  const bool first = lb < part.nb && g == part.g0;
  const int tid = threadIdx.x, nt = blockDim.x, lane = tid & 31, warp = tid >> 5, n_warps = nt >> 5;
  const int K = st.K, C = K + 1, len = st.len, n = len + 1;
  const size_t base = (size_t)u * C;
  float* s_attn = reinterpret_cast<float*>(smem);  // [C] attention mass by cache row
  __shared__ unsigned long long wfree[32], wmin[32];
  __shared__ int wcand[32];
  __shared__ uint32_t hist[256];
  __shared__ int tie_cnt[E * step_warps(E)];  // [entry][warp]
  __shared__ int sel_bin, sel_above, sel_pop;
  __shared__ ulonglong2 s_seq;
  __shared__ int s_best;

  ta_wait_for_prior_grid();
  // ---- the unit's state (from L2: the step before wrote it) and its attention masses, all requested before the first is used
  const int x = new_ids[b];
  if (first && warp == 0) {  // before everything else: the other blocks wait for it
    const bool gone = step_gave_up(status);
    const SeqStep seq = sequence_step(st, pt, b, x, vocab, voucher_decay, budget_decay);
    if (sync.hold_ns && !gone && part.nl * part.ng > 1) hold_words(sync.hold_ns);
    const ulonglong2 w = gone ? make_ulonglong2(0ull, 0ull) : seq_words(seq);
    for (int q = 1 + lane; q < part.nl * part.ng; q += 32) {
      const int l = q / part.ng;
      ulonglong2* to = sync.words + ((l * part.nb + bi) * part.ng + q - l * part.ng);
      *(volatile unsigned long long*)&to->x = w.x;
      *(volatile unsigned long long*)&to->y = w.y;
    }
    if (lane == 0) {
      s_seq = w;
      s_best = seq.best;
    }
  }
  int pos[E], row[E], id[E], S[E];
  float A[E], P[E], V[E];
#pragma unroll
  for (int e = 0; e < E; ++e) {
    const int r = tid + e * nt;
    const bool old = r < len;
    id[e] = old ? __ldcg(&st.tok[base + r]) : r == len ? x : 0;
    pos[e] = old ? __ldcg(&st.pos[base + r]) : 0;
    row[e] = old ? __ldcg(&st.slot[base + r]) : r == len ? __ldcg(&st.next_slot[u]) : -1;
    A[e] = old ? __ldcg(&st.A[base + r]) : 0.0f;
    P[e] = old ? __ldcg(&st.P[base + r]) : 0.0f;
    V[e] = old ? __ldcg(&st.V[base + r]) : 0.0f;
    S[e] = old ? __ldcg(&st.S[base + r]) : 0;
    if (r < C) copy_async4(&s_attn[r], &attn[base + r]);
  }
  // Two threads wait, each for a word that it alone reads and clears: one that read along could miss the word and wait for good.
  // (The first look at the words: not waited for before the counts are requested.)
  const bool waits = !first && tid < 2;
  unsigned long long* const word = reinterpret_cast<unsigned long long*>(sync.words + blockIdx.x) + (tid & 1);
  unsigned long long said1 = 0;
  bool gone = false;
  if (waits) {
    said1 = *(volatile unsigned long long*)word;
    gone = step_gave_up(status);
  }
  int c[E];  // occurrences of the entry's id; of the new token's, which the sequence's first unit counts up: from the words
#pragma unroll
  for (int e = 0; e < E; ++e) {
    const int r = tid + e * nt;
    const bool counted = r < n && id[e] >= 0 && id[e] < vocab;
    c[e] = counted && id[e] != x ? __ldcg(&st.hist[(size_t)b * vocab + id[e]]) : counted ? -1 : 0;
  }
  if (waits) {
    if (gone) said1 = 0ull;
    else if (!(said1 & kPublished)) said1 = wait_word(word, sync.wait_limit_ns, status, u);
    reinterpret_cast<unsigned long long*>(&s_seq)[tid] = said1;
    if (said1) *word = 0ull;
  }
  copy_async_wait();
  __syncthreads();
  const ulonglong2 said = s_seq;
  if (!(said.x & said.y & kPublished)) return;  // a wait ran out: the unit's state stays as it is
  const int t = (int)(said.y >> 32) & 0x7fffffff, match_len = (int)(said.x >> 32) & 0xff;
  const float v_new = __uint_as_float((uint32_t)said.x);
#pragma unroll
  for (int e = 0; e < E; ++e) {
    if (c[e] < 0) c[e] = (int)(uint32_t)said.y + 1;
    if (tid + e * nt == len) {
      pos[e] = t;
      V[e] = v_new;
    }
  }
  const float nf = (float)(t + 1), rn = __frcp_rn(nf);
  const float omr = __fsub_rn(1.0f, rho);
  // ---- attention update, utility
  uint32_t changed = 0;  // entries whose anchor indicator changed
  uint32_t ku[E];
#pragma unroll
  for (int e = 0; e < E; ++e) {
    const int r = tid + e * nt;
    ku[e] = 0xffffffffu;
    if (r < n) {
      float a = 0.0f;
      if (row[e] >= 0 && row[e] < C) a = s_attn[row[e]];
      else report(status, TA_ERR_DEVICE_BOUNDS, 6, u, row[e]);
      A[e] = __fadd_rn(A[e], a);
      P[e] = __fadd_rn(__fmul_rn(rho, P[e]), __fmul_rn(omr, a));
      if (pos[e] >= t - match_len + 1 && !S[e]) {
        S[e] = 1;
        changed |= 1u << e;
      }
      const float R = ta_div_by((float)(pos[e] + 1), nf, rn);
      const float F = ta_div_by((float)c[e], nf, rn);
      const float t0 = __fadd_rn(__fmul_rn(beta, R), __fmul_rn(gamma, S[e] ? 1.0f : 0.0f));
      const float t1 = __fsub_rn(t0, __fmul_rn(lambda, F));
      const float us = __fadd_rn(t1, V[e]);
      const float ua = __fadd_rn(__fmul_rn(alpha, A[e]), __fmul_rn(delta, P[e]));
      ku[e] = sortable_key(__fadd_rn(ua, us));
    }
  }
  int ev = -1;  // entry to evict
  if (n > K) {
    // ---- budget partition on n = K + 1 tokens
    int p = k_protected < 0 ? K - n_sink - n_recent : k_protected;
    p = max(0, min(p, K));
    const int K_main = K - p;
    const int sinks = min(n_sink, n);
    const int recents = max(0, min(n_recent, n - sinks));
    const int s_take = min(sinks, K_main);
    const int r_take = min(recents, K_main - s_take);
    auto mandatory = [&](int i) { return i < s_take || i >= n - r_take; };
    const uint32_t ones = 0xffffffffu;
    auto warp_min = [&](unsigned long long x) {
      const uint32_t hi = __reduce_min_sync(ones, (uint32_t)(x >> 32));
      const uint32_t lo = __reduce_min_sync(ones, (uint32_t)(x >> 32) == hi ? (uint32_t)x : ones);
      return ((unsigned long long)hi << 32) | lo;
    };
    // candidates of the protected pool; the last of them in line (smallest voucher, latest position), which is the one
    // left out when there is one candidate too many; the loser among the tokens that are no candidates
    auto entry = [](uint32_t key, int r) { return ((unsigned long long)key << 32) | (uint32_t)(~(uint32_t)r); };
    int cand = 0;
    unsigned long long free_min = ~0ull, cand_min = ~0ull;
    uint32_t kv[E];  // key of the voucher, 0: not a candidate
#pragma unroll
    for (int e = 0; e < E; ++e) {
      const int r = tid + e * nt;
      kv[e] = 0u;
      if (r < n && !mandatory(r)) {
        if (V[e] > 0.0f && p > 0) {
          kv[e] = sortable_key(V[e]);
          ++cand;
          cand_min = min(cand_min, entry(kv[e], r));
        } else {
          free_min = min(free_min, entry(ku[e], r));
        }
      }
    }
    free_min = warp_min(free_min);
    cand_min = warp_min(cand_min);
    cand = __reduce_add_sync(ones, cand);
    if (lane == 0) {
      wfree[warp] = free_min;
      wmin[warp] = cand_min;
      wcand[warp] = cand;
    }
    __syncthreads();
    free_min = warp_min(lane < n_warps ? wfree[lane] : ~0ull);
    cand = __reduce_add_sync(ones, lane < n_warps ? wcand[lane] : 0);
    if (cand > p) {
      uint32_t forced = 0;  // bit e: this thread's entry e is in the protected pool
      if (cand == p + 1) {
        // one candidate too many (always so when all slots but the mandatory ones are protected)
        const int out = (int)(~(uint32_t)(warp_min(lane < n_warps ? wmin[lane] : ~0ull) & 0xffffffffull));
#pragma unroll
        for (int e = 0; e < E; ++e) forced |= (kv[e] != 0u && tid + e * nt != out) ? 1u << e : 0u;
      } else {
        // the p largest vouchers: 8 bits at a time from the top; done as soon as the bin is taken as a whole
        uint32_t prefix = 0, mask = 0;
        int remaining = p, pop = 0;
        for (int shift = 24; shift >= 0; shift -= 8) {
          for (int k = tid; k < 256; k += nt) hist[k] = 0;
          __syncthreads();
#pragma unroll
          for (int e = 0; e < E; ++e)
            if (kv[e] != 0u && (kv[e] & mask) == prefix) atomicAdd(&hist[(kv[e] >> shift) & 255u], 1u);
          __syncthreads();
          if (warp == 0) {  // lane l owns bins 8l .. 8l+7; walk down from the top until `remaining` are covered
            int h[8], tot = 0;
#pragma unroll
            for (int k = 0; k < 8; ++k) tot += h[k] = (int)hist[8 * lane + k];
            int run = tot;  // this lane and the lanes above
#pragma unroll
            for (int off = 1; off < 32; off <<= 1) {
              const int o = __shfl_down_sync(ones, run, off);
              if (lane + off < 32) run += o;
            }
            int above = run - tot;
            if (above < remaining && remaining <= run) {
              int k = 7;
              for (; k > 0 && above + h[k] < remaining; --k) above += h[k];
              sel_bin = 8 * lane + k;
              sel_above = above;
              sel_pop = (int)hist[8 * lane + k];
            }
          }
          __syncthreads();
          prefix |= (uint32_t)sel_bin << shift;
          mask |= 255u << shift;
          remaining -= sel_above;
          pop = sel_pop;
          if (pop == remaining) break;
        }
        uint32_t tie = 0;
#pragma unroll
        for (int e = 0; e < E; ++e) {
          const bool in = kv[e] != 0u && (kv[e] & mask) == prefix;
          if (in) tie |= 1u << e;
          if (kv[e] != 0u && ((kv[e] & mask) > prefix || (in && pop == remaining))) forced |= 1u << e;
        }
        if (pop != remaining) {  // equal vouchers: the earliest positions first
#pragma unroll
          for (int e = 0; e < E; ++e) {
            const unsigned word = __ballot_sync(ones, (tie >> e) & 1u);
            if (lane == 0) tie_cnt[e * n_warps + warp] = __popc(word);
          }
          __syncthreads();
#pragma unroll
          for (int e = 0; e < E; ++e) {
            const unsigned word = __ballot_sync(ones, (tie >> e) & 1u);
            int seen = __popc(word & ((1u << lane) - 1u));
            for (int j = 0; j < e * n_warps + warp; ++j) seen += tie_cnt[j];
            if (((tie >> e) & 1u) && seen < remaining) forced |= 1u << e;
          }
        }
      }
      // the loser among the candidates that are left out
      unsigned long long lose = ~0ull;
#pragma unroll
      for (int e = 0; e < E; ++e)
        if (kv[e] != 0u && !((forced >> e) & 1u)) lose = min(lose, entry(ku[e], tid + e * nt));
      lose = warp_min(lose);
      __syncthreads();  // wmin has been read
      if (lane == 0) wmin[warp] = lose;
      __syncthreads();
      free_min = min(free_min, warp_min(lane < n_warps ? wmin[lane] : ~0ull));
    }
    ev = free_min == ~0ull ? K : (int)(~(uint32_t)(free_min & 0xffffffffull));  // (~0: cannot happen, at most K are forced)
  }
  // ---- write the state back without the evicted entry; vouchers decay (Algorithm 1 step 10). Position, row, id and
  // indicator of the entries before the evicted one stay where and what they are.
#pragma unroll
  for (int e = 0; e < E; ++e) {
    const int r = tid + e * nt;
    if (r < n) {
      if (r == ev) {
        st.next_slot[u] = row[e];
        evicted_pos[u] = pos[e];
      } else {
        const bool moved = ev >= 0 && r > ev;
        const size_t d = base + (moved ? r - 1 : r);
        if (moved || r == len) {
          st.pos[d] = pos[e];
          st.slot[d] = row[e];
          st.tok[d] = id[e];
        }
        if (moved || r == len || ((changed >> e) & 1u)) st.S[d] = (uint8_t)S[e];
        st.A[d] = A[e];
        st.P[d] = P[e];
        st.V[d] = __fmul_rn(V[e], budget_decay);
      }
    }
  }
  if (ev < 0 && tid == 0) {
    st.next_slot[u] = n;  // rows fill up in order until the cache is full
    evicted_pos[u] = -1;
  }
  // ---- the first unit: what the sequence's units share goes on by one token
  if (first && part.update && tid == 0) {
    const int x = new_ids[b], t = (int)(s_seq.y >> 32) & 0x7fffffff;
    st.tok_ring[(size_t)b * TA_MAX_PATTERN_LEN + (t & (TA_MAX_PATTERN_LEN - 1))] = x;
    if (x >= 0 && x < vocab) st.hist[(size_t)b * vocab + x] = (int)(uint32_t)s_seq.y + 1;
    else report(status, TA_ERR_DEVICE_BOUNDS, 5, b, x);
    st.anc_B[(size_t)b * TA_MAX_SPAN + (t & (TA_MAX_SPAN - 1))] = s_best >= 0 ? pt.budget[s_best] : 0.0f;
    st.anc_L[(size_t)b * TA_MAX_SPAN + (t & (TA_MAX_SPAN - 1))] = s_best >= 0 ? pt.span[s_best] : 0;
    st.n_seen[b] = t + 1;
  }
}

}  // namespace

cudaError_t ta_launch_stream_step(const ta_stream_dev& st, const ta_patterns* pats, const ta_policy& pol, const int32_t* new_ids,
                                  const float* attn, const ta_stream_sync& sync, int32_t* evicted_pos, ta_dev_status* status,
                                  cudaStream_t stream) {
  const int C = st.K + 1;
  const int items = step_items(C), threads = step_block(C, items);
  const size_t smem = (size_t)C * 4;  // at most 16 KB
  auto kern = items == 3 ? ta_stream_step_kernel<3> : items == 4 ? ta_stream_step_kernel<4> : ta_stream_step_kernel<9>;
  const PatternTable pt = {pats->d_ids, pats->d_len, pats->d_budget, pats->d_span, pats->n_pat};
  cudaLaunchConfig_t cfg = {};
  cfg.blockDim = dim3((unsigned)threads, 1, 1);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = stream;
  cudaLaunchAttribute attr[1];
  ta_pdl_attribute(&attr[0]);
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  cudaError_t e = cudaSuccess;
  // In parts of as many blocks as there are words for, in practice one. The sequences' shared state changes in their last part.
  const int ng = st.Hkv < kStreamWords ? st.Hkv : kStreamWords;
  const int nb = st.B < kStreamWords / ng ? st.B : kStreamWords / ng;
  const int nl = st.n_layers < kStreamWords / (ng * nb) ? st.n_layers : kStreamWords / (ng * nb);
  for (int b0 = 0; b0 < st.B; b0 += nb)
    for (int l0 = 0; l0 < st.n_layers; l0 += nl)
      for (int g0 = 0; g0 < st.Hkv && e == cudaSuccess; g0 += ng) {
        auto rest = [](int all, int from, int n) { return all - from < n ? all - from : n; };
        const StreamPart part = {l0, rest(st.n_layers, l0, nl), b0, rest(st.B, b0, nb), g0, rest(st.Hkv, g0, ng),
                                 l0 + nl >= st.n_layers && g0 + ng >= st.Hkv};
        cfg.gridDim = dim3((unsigned)(part.nl * part.nb * part.ng), 1, 1);
        e = cudaLaunchKernelEx(&cfg, kern, st, pt, new_ids, attn, sync, part, pol.vocab_size, pol.voucher_decay, pol.alpha,
                               pol.beta, pol.gamma, pol.delta, pol.lambda, pol.pension_rho, pol.budget_decay, pol.n_sink,
                               pol.n_recent, pol.k_protected, evicted_pos, status);
      }
  return e;
}
