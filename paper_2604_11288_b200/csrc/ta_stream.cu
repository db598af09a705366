// Algorithm 1 in the decode loop: one new token per sequence and step, at most K cached tokens per unit afterwards.
// (Section 3.1: a retention policy selects S, |S| <= K, "after each generation step"; Algorithm 1 steps 1-10.)
//
// Per step two kernels run:
//   ta_stream_seq_kernel    one warp per sequence: token histogram, pattern match ending at the new token (longest
//                           pattern wins, then the lowest index), the new token's voucher from the anchors of the last
//                           TA_MAX_SPAN positions (Eq. 2 with budgets that decayed once per step since detection; a lane
//                           per distance)
//   ta_stream_step_kernel   one block per unit, its K+1 entries in registers: appends the new token to the position-ordered
//                           state, adds this step's attention mass to A, updates the pension average P, forms the
//                           utility of Eq. 1, applies the budget partition of Section 3.3 to the K+1 cached tokens
//                           (exactly one token loses), removes it from the ordered state (4-byte entries move;
//                           key/value rows never do: the freed cache row is handed to the next token) and decays every
//                           voucher by budget_decay (Algorithm 1 step 10)
// The second kernel runs beside the first: it reads the unit's state and waits for the first only where the new token comes
// in. What bounds it: latency at few units, the state's bytes (25 read, 12 to 25 written per cached token, 4 of attention
// mass read) at many. 4096 units of 257 tokens, three states in turn (180 MB: more than L2), a step of both kernels: where the
// tokens with a voucher fit the protected slots 31 -> 18.5 us, where all compete for a quarter of the slots 70 -> 25.6 us, the
// extremes of what a generation meets (serial scans by one thread in the pool selection, one lane per sequence for the voucher,
// all entries through shared memory before; then 22 us with two entries in 64 registers, of which an SM held 6 blocks).
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

__global__ void __launch_bounds__(32) ta_stream_seq_kernel(ta_stream_dev st, const int32_t* __restrict__ new_ids,
                                                           const int32_t* __restrict__ p_ids,
                                                           const int32_t* __restrict__ p_len,
                                                           const float* __restrict__ p_budget,
                                                           const int32_t* __restrict__ p_span, int n_pat,
                                                           float voucher_decay, float budget_decay, int vocab,
                                                           ta_stream_seq_info* __restrict__ info,
                                                           ta_dev_status* status) {
  constexpr int kHalves = TA_MAX_SPAN / 32;
  static_assert(TA_MAX_SPAN % 32 == 0 && TA_MAX_PATTERN_LEN == 8, "a lane per distance, eight ids in registers");
  const int b = blockIdx.x, lane = threadIdx.x;
  // decay^k by repeated multiplication (one rounding per step) for the distances k = lane + 1, lane + 33, ..
  float w[kHalves];
  {
    float x = 1.0f;
    int done = 0;
#pragma unroll
    for (int h = 0; h < kHalves; ++h) {
      for (; done < 32 * h + lane + 1; ++done) x = __fmul_rn(x, voucher_decay);
      w[h] = x;
    }
  }
  ta_wait_for_prior_grid();
  ta_launch_dependents();
  const int x = new_ids[b];
  const int t = st.n_seen[b];
  int32_t* ring = st.tok_ring + (size_t)b * TA_MAX_PATTERN_LEN;
  float* aB = st.anc_B + (size_t)b * TA_MAX_SPAN;
  int32_t* aL = st.anc_L + (size_t)b * TA_MAX_SPAN;
  // the anchors of the last positions and the last ids, requested together
  int L[kHalves];
  float Bk[kHalves];
#pragma unroll
  for (int h = 0; h < kHalves; ++h) {
    const int k = 32 * h + lane + 1;
    L[h] = k <= t ? aL[(t - k) % TA_MAX_SPAN] : 0;
    Bk[h] = k <= t ? aB[(t - k) % TA_MAX_SPAN] : 0.0f;
  }
  const int last = lane < TA_MAX_PATTERN_LEN - 1 && t - 1 - lane >= 0 ? ring[(t - 1 - lane) % TA_MAX_PATTERN_LEN] : -1;
  int ids[TA_MAX_PATTERN_LEN];  // ids[k]: the token k positions before the new one
  ids[0] = x;
#pragma unroll
  for (int k = 1; k < TA_MAX_PATTERN_LEN; ++k) ids[k] = __shfl_sync(0xffffffffu, last, k - 1);
  if (lane == 0) {
    ring[t % TA_MAX_PATTERN_LEN] = x;
    if (x >= 0 && x < vocab) atomicAdd(&st.hist[(size_t)b * vocab + x], 1);
    else report(status, TA_ERR_DEVICE_BOUNDS, 5, b, x);
  }
  // patterns ending at t
  int best = -1, best_len = 0;
  for (int p = lane; p < n_pat; p += 32) {
    const int len = p_len[p];
    if (len > t + 1 || len <= best_len) continue;  // within a lane p ascends: a later pattern wins only if longer
    const int32_t* pid = p_ids + p * TA_MAX_PATTERN_LEN;
    bool ok = true;
#pragma unroll
    for (int k = 0; k < TA_MAX_PATTERN_LEN; ++k) ok = ok && (k >= len || ids[k] == pid[max(len - 1 - k, 0)]);
    if (ok) {
      best = p;
      best_len = len;
    }
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const int ol = __shfl_xor_sync(0xffffffffu, best_len, o), ob = __shfl_xor_sync(0xffffffffu, best, o);
    if (ol > best_len || (ol == best_len && ob >= 0 && (best < 0 || ob < best))) {
      best_len = ol;
      best = ob;
    }
  }
  // voucher of the new token from the anchors at t-1, t-2, ..: every lane its own term, summed nearest first
  float v = 0.0f;
#pragma unroll
  for (int h = 0; h < kHalves; ++h) {
    const int k = 32 * h + lane + 1;
    const bool reaches = L[h] > 0 && k <= L[h];
    float term = 0.0f;
    if (reaches) {
      for (int s = 0; s < k; ++s) Bk[h] = __fmul_rn(Bk[h], budget_decay);
      term = __fmul_rn(Bk[h], w[h]);
    }
    for (unsigned left = __ballot_sync(0xffffffffu, reaches); left != 0u; left &= left - 1u)
      v = __fadd_rn(v, __shfl_sync(0xffffffffu, term, __ffs((int)left) - 1));
  }
  if (lane == 0) {
    aB[t % TA_MAX_SPAN] = best >= 0 ? p_budget[best] : 0.0f;
    aL[t % TA_MAX_SPAN] = best >= 0 ? p_span[best] : 0;
    st.n_seen[b] = t + 1;
    ta_stream_seq_info si;
    si.t = t;
    si.match_len = best_len;  // the longest matching pattern covers the tokens of every pattern that ends here
    si.v_new = v;
    si.id = x;
    info[b] = si;
  }
}

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
__host__ __device__ constexpr int step_threads(int e) { return e == 3 ? 576 : e == 4 ? 512 : 544; }
constexpr int step_regs(int e) { return e == 3 ? 56 : 64; }
// warps of the largest block: what the shared arrays are sized for
__host__ __device__ constexpr int step_warps(int e) { return step_threads(e) / 32; }

// Entries per thread for units of C cached tokens: three or four, whichever lets an SM hold more blocks (three when equal:
// fewer spills); eight where a block would have to be larger than those kernels allow.
constexpr int step_block(int C, int e) { return ((C + e - 1) / e + 31) / 32 * 32; }
constexpr int step_resident(int C, int e) {
  return step_block(C, e) <= step_threads(e) ? 65536 / (step_block(C, e) * step_regs(e)) : 0;
}
constexpr int step_items(int C) {
  const int r3 = step_resident(C, 3), r4 = step_resident(C, 4);
  return r3 == 0 && r4 == 0 ? 8 : r3 >= r4 ? 3 : 4;
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

// One block per unit; thread tid holds the entries tid, tid + nt, .. (E of them) in registers for the whole step.
// Selection (Section 3.3 on the K+1 cached tokens): mandatory sinks and recents; the protected pool = the sponsored,
// non-mandatory tokens with the largest vouchers (lower position first among equals); exactly one token is then not
// forced and loses: the one with the smallest utility, the latest position among equals. When the sponsored tokens fit the
// protected slots, or are one too many, block-wide minima decide; otherwise a radix select on the voucher keys.
template <int E>
__global__ void __launch_bounds__(step_threads(E), E == 8 ? 1 : 2)
ta_stream_step_kernel(ta_stream_dev st, const ta_stream_seq_info* info, const float* __restrict__ attn,
                      int vocab, float alpha, float beta, float gamma, float delta, float lambda, float rho,
                      float budget_decay, int n_sink, int n_recent, int k_protected, int32_t* __restrict__ evicted_pos,
                      ta_dev_status* status) {
  extern __shared__ __align__(16) unsigned char smem[];
  const int u = blockIdx.x, tid = threadIdx.x, nt = blockDim.x, lane = tid & 31, warp = tid >> 5, n_warps = nt >> 5;
  const int b = (u / st.Hkv) % st.B;
  const int K = st.K, C = K + 1, len = st.len, n = len + 1;
  const size_t base = (size_t)u * C;
  float* s_attn = reinterpret_cast<float*>(smem);  // [C] attention mass by cache row
  __shared__ unsigned long long wfree[32], wmin[32];
  __shared__ int wcand[32];
  __shared__ uint32_t hist[256];
  __shared__ int tie_cnt[E * step_warps(E)];  // [entry][warp]
  __shared__ int sel_bin, sel_above, sel_pop;

  // ---- the unit's state (from L2: other blocks wrote it) and its attention masses, all requested before the first is used.
  // Launched as a programmatic dependent of the per-sequence kernel, which lets this one start when everything before it
  // is complete.
  int pos[E], row[E], id[E], S[E];
  float A[E], P[E], V[E];
#pragma unroll
  for (int e = 0; e < E; ++e) {
    const int r = tid + e * nt;
    const bool old = r < len;
    pos[e] = old ? __ldcg(&st.pos[base + r]) : 0;
    row[e] = old ? __ldcg(&st.slot[base + r]) : r == len ? __ldcg(&st.next_slot[u]) : -1;
    id[e] = old ? __ldcg(&st.tok[base + r]) : 0;
    A[e] = old ? __ldcg(&st.A[base + r]) : 0.0f;
    P[e] = old ? __ldcg(&st.P[base + r]) : 0.0f;
    V[e] = old ? __ldcg(&st.V[base + r]) : 0.0f;
    S[e] = old ? __ldcg(&st.S[base + r]) : 0;
    if (r < C) s_attn[r] = attn[base + r];
  }
  ta_wait_for_prior_grid();
  // (not through a const __restrict__ pointer: such a load counts as invariant and may be moved above the wait)
  static_assert(sizeof(ta_stream_seq_info) == 16, "one 16-byte load");
  const int4 raw = __ldcg(reinterpret_cast<const int4*>(info + b));
  ta_stream_seq_info si;
  si.t = raw.x;
  si.match_len = raw.y;
  si.v_new = __int_as_float(raw.z);
  si.id = raw.w;
  const int t = si.t;
  const float nf = (float)(t + 1), rn = __frcp_rn(nf);
  const float omr = __fsub_rn(1.0f, rho);
  int c[E];
#pragma unroll
  for (int e = 0; e < E; ++e) {
    const int r = tid + e * nt;
    if (r == len) {
      pos[e] = t;
      id[e] = si.id;
      V[e] = si.v_new;
    }
    c[e] = (r < n && id[e] >= 0 && id[e] < vocab) ? __ldcg(&st.hist[(size_t)b * vocab + id[e]]) : 0;
  }
  __syncthreads();
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
      if (pos[e] >= t - si.match_len + 1 && !S[e]) {
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
}

}  // namespace

cudaError_t ta_launch_stream_seq(const ta_stream_dev& st, const ta_patterns* pats, const ta_policy& pol,
                                 const int32_t* new_ids, ta_stream_seq_info* info, ta_dev_status* status,
                                 cudaStream_t stream) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)st.B, 1, 1);
  cfg.blockDim = dim3(32, 1, 1);
  cfg.stream = stream;
  cudaLaunchAttribute attr[1];
  ta_pdl_attribute(&attr[0]);
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, ta_stream_seq_kernel, st, new_ids, (const int32_t*)pats->d_ids,
                            (const int32_t*)pats->d_len, (const float*)pats->d_budget, (const int32_t*)pats->d_span,
                            pats->n_pat, pol.voucher_decay, pol.budget_decay, pol.vocab_size, info, status);
}

cudaError_t ta_launch_stream_step(const ta_stream_dev& st, const ta_policy& pol, const ta_stream_seq_info* info,
                                  const float* attn, int32_t* evicted_pos, ta_dev_status* status,
                                  cudaStream_t stream) {
  const int U = st.n_layers * st.B * st.Hkv, C = st.K + 1;
  const int items = step_items(C), threads = step_block(C, items);
  const size_t smem = (size_t)C * 4;  // at most 16 KB
  auto kern = items == 3 ? ta_stream_step_kernel<3> : items == 4 ? ta_stream_step_kernel<4> : ta_stream_step_kernel<8>;
  // runs beside the kernel before it on the stream (ta_stream_seq_kernel in ta_stream_step)
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)U, 1, 1);
  cfg.blockDim = dim3((unsigned)threads, 1, 1);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = stream;
  cudaLaunchAttribute attr[1];
  ta_pdl_attribute(&attr[0]);
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kern, st, info, attn, pol.vocab_size, pol.alpha, pol.beta, pol.gamma, pol.delta,
                            pol.lambda, pol.pension_rho, pol.budget_decay, pol.n_sink, pol.n_recent, pol.k_protected,
                            evicted_pos, status);
}
