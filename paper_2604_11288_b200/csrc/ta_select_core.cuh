// Core of the budget-K selection (radix select, ordered emit, the two kernels), written against a block size that the
// including file fixes with TA_SEL_THREADS before each inclusion; everything lives in namespace TA_SEL_NS. The
// selection kernels are built for 512 threads (two blocks per SM for short units), for 1024 threads (twice the keys in
// registers for long units, and few short ones) and for 128 and 256 (many short units with small budgets).
namespace TA_SEL_NS {

constexpr int kThreads = TA_SEL_THREADS;
constexpr int kWarps = kThreads / 32;

__device__ __forceinline__ uint32_t sortable_key(float f) {
  uint32_t b = __float_as_uint(f);
  if ((b << 1) == 0u) b = 0u;  // -0 == +0
  return (b & 0x80000000u) ? ~b : (b | 0x80000000u);
}

constexpr int kItemsLong = 32;  // keys per thread of clustered units (up to 8 * kItemsLong * kThreads elements)

struct SelectResult {
  uint32_t thresh;  // key of the last element taken
  int ties;         // how many elements equal to thresh are taken (lowest positions first)
  int all;          // 1: every eligible element is taken (fewer eligible than requested)
  int none;         // 1: nothing is taken
  int all_ties;     // 1: every eligible element equal to thresh is taken (0: not known)
};

constexpr int kCandCap = 2048;  // candidates a split unit finishes locally
constexpr int kCompareCap = 32;  // so few candidates are compared with one another instead of counted by digits

template <int CL>  // CTAs that share a unit
struct SelectShared {
  __align__(16) uint32_t hist[256];
  uint32_t prefix, mask;
  int remaining;
  int done_all;
  int ncand;  // elements in the digit bin the threshold fell into: the candidates of the next pass
  __align__(16) uint32_t warp_cnt[kWarps];  // per warp: definite count (low 16 bits) | tie count (high 16 bits)
  // range of the eligible keys: per warp (smallest, largest, how many), and per CTA of a cluster
  uint32_t wmin[kWarps], wmax[kWarps], wnum[kWarps];
  __align__(16) uint32_t cl_range[CL][4];
  // long sequences are split over the CTAs of a cluster: every CTA's histogram, two counts to a word, as it sent them to all
  // (two buffers alternating by pass), and every CTA's (definite, tie) totals
  __align__(16) uint32_t ghist[CL > 1 ? 2 : 1][CL][CL > 1 ? 128 : 1];
  __align__(8) int totals[2][CL][2];        // (by the exchange's number)
  __align__(8) unsigned long long arrived[2];  // mbarriers of the exchanges between the CTAs, taken in turn
  // ordered write of a unit whose keys sit in registers: bitmaps of the definite and of the tie elements in position
  // order (word e covers positions 32e .. 32e+31 of this CTA's slice)
  // (a row of kWarps words per chunk, padded by one word so that the 32 rows a warp writes fall into 32 banks)
  uint32_t bdef[kItemsLong * (kWarps + 1)], btie[kItemsLong * (kWarps + 1)];
  uint32_t wtot[kWarps];
  uint32_t before[kThreads];  // definite (low 16 bits) and tie elements before every word
  uint32_t total;
  // a unit split over a cluster: once few candidates are left, every CTA sends its own to all and the remaining passes run on
  // that list inside each CTA
  uint32_t cand_n;
  __align__(16) uint32_t cand_keys[kCandCap];
  uint32_t cmp_n, cmp_thresh;  // the same inside one CTA, for at most kCompareCap candidates
  int cmp_above, cmp_equal;
  uint32_t took_part[CL];  // in the exchange of candidates (never read: what counts is that the words arrive)
};
constexpr int kSelectCluster = 8;  // CTAs per unit when a sequence is longer than kItems * kThreads

// Keys of a unit are read once into registers when the unit is short enough (kItems per thread), else they are
// re-read from L2 on every sweep in batches whose loads are all issued before the first use.
constexpr int kItems = 16;
constexpr int kBatch = 8;
static_assert(kItems % 8 == 0 && kItemsLong % 8 == 0, "the cached load works in groups of 8 keys per thread");
template <int ITEMS>
struct KeyCache {
  uint32_t key[ITEMS];
  uint32_t elig;  // bit `it`: element tid + it*kThreads exists and is eligible
};

// Calls body(i, exists, eligible, key) for every element slot in ascending chunks of kThreads; every thread of the
// block makes the same number of calls (the body may hold block-wide barriers).
template <bool CACHED, class KeyFn, class Body, int ITEMS>
__device__ __forceinline__ void sweep(int n, KeyFn key_of, const KeyCache<ITEMS>& kc, Body body) {
  const int tid = threadIdx.x;
  if (CACHED) {
#pragma unroll
    for (int it = 0; it < ITEMS; ++it) {
      if (it * kThreads < n) {
        const int i = tid + it * kThreads;
        body(i, i < n, ((kc.elig >> it) & 1u) != 0, kc.key[it]);
      }
    }
  } else {
    for (int base = 0; base < n; base += kBatch * kThreads) {
      uint32_t k[kBatch];
      uint32_t e = 0;
#pragma unroll
      for (int b = 0; b < kBatch; ++b) {
        const int i = base + b * kThreads + tid;
        k[b] = 0;
        if (i < n && key_of(i, k[b])) e |= 1u << b;
      }
#pragma unroll
      for (int b = 0; b < kBatch; ++b) {
        if (base + b * kThreads < n) {
          const int i = base + b * kThreads + tid;
          body(i, i < n, ((e >> b) & 1u) != 0, k[b]);
        }
      }
    }
  }
}

// Top-`want` of the eligible elements of [0, n) by key. All threads of the block must call it; the result is uniform
// across the block.
template <bool CACHED, int CL, class KeyFn, int ITEMS>
__device__ SelectResult block_radix_select(int n, int want, KeyFn key_of, const KeyCache<ITEMS>& kc, SelectShared<CL>& sh) {
  SelectResult r;
  r.thresh = 0;
  r.ties = 0;
  r.all = 0;
  r.all_ties = 0;
  r.none = (want <= 0);
  if (r.none) return r;
  const int tid = threadIdx.x, lane = tid & 31;
  if (tid == 0) {
    sh.prefix = 0;
    sh.mask = 0;
    sh.remaining = want;
    sh.done_all = 0;
  }
  uint32_t* ghist0 = nullptr;
  if (CL > 1) ghist0 = cg::this_cluster().map_shared_rank(&sh.ghist[0][0][0], 0);
  for (int pass = 0; pass < 4; ++pass) {
    const int shift = 24 - 8 * pass;
    for (int k = tid; k < 256; k += kThreads) {
      sh.hist[k] = 0;
      if (CL > 1) (&sh.ghist[pass & 1][0][0])[k] = 0;  // only rank 0's copy is used; its readers of two passes ago are done
    }
    if (CL > 1) cg::this_cluster().sync();
    else __syncthreads();
    const uint32_t prefix = sh.prefix, mask = sh.mask;
    sweep<CACHED>(n, key_of, kc, [&](int, bool, bool elig, uint32_t key) {
      const int bin = (elig && (key & mask) == prefix) ? (int)((key >> shift) & 255u) : -1;
      // after the first pass most warps hold no candidate at all: a ballot is far cheaper than match.any
      const unsigned have = __ballot_sync(0xffffffffu, bin >= 0);
      if (have == 0u) return;
      if ((have & (have - 1u)) == 0u) {  // a single candidate in the warp
        if (bin >= 0) atomicAdd(&sh.hist[bin], 1u);
        return;
      }
      const unsigned peers = __match_any_sync(0xffffffffu, bin);
      if (bin >= 0 && lane == __ffs(peers) - 1) atomicAdd(&sh.hist[bin], (uint32_t)__popc(peers));
    });
    __syncthreads();
    const uint32_t* hist = sh.hist;
    if (CL > 1) {  // merge the slices' histograms on rank 0, then every CTA takes the same decision from the sum
      uint32_t* gh = ghist0 + (pass & 1) * (CL * 128);
      for (int k = tid; k < 256; k += kThreads)
        if (sh.hist[k]) atomicAdd(&gh[k], sh.hist[k]);
      cg::this_cluster().sync();
      hist = gh;
    }
    if (tid < 32) {
      // lane l owns bins [8l, 8l+8); walk from the top bin down until `remaining` elements are covered
      uint32_t hl[8];
#pragma unroll
      for (int k = 0; k < 8; ++k) hl[k] = hist[8 * lane + k];
      uint32_t tot = 0;
#pragma unroll
      for (int k = 0; k < 8; ++k) tot += hl[k];
      uint32_t above = 0;  // elements in lanes above this one
      {
        uint32_t run = tot;
#pragma unroll
        for (int off = 1; off < 32; off <<= 1) {
          const uint32_t o = __shfl_down_sync(0xffffffffu, run, off);
          if (lane + off < 32) run += o;
        }
        above = run - tot;
      }
      const int remaining = sh.remaining;
      const uint32_t total = __shfl_sync(0xffffffffu, above + tot, 0);
      if (pass == 0 && total < (uint32_t)remaining) {
        if (lane == 0) sh.done_all = 1;
      } else {
        const bool mine = above < (uint32_t)remaining && (uint32_t)remaining <= above + tot;
        if (mine) {
          uint32_t cum = above;
          int k = 7;
#pragma unroll
          for (int kk = 7; kk > 0; --kk) {
            if (k == kk && cum + hl[kk] < (uint32_t)remaining) {
              cum += hl[kk];
              k = kk - 1;
            }
          }
          const int bin = 8 * lane + k;
          sh.remaining = remaining - (int)cum;
          sh.prefix = prefix | ((uint32_t)bin << shift);
          sh.mask = mask | (255u << shift);
        }
      }
    }
    __syncthreads();
    if (sh.done_all) {
      r.all = 1;
      return r;
    }
  }
  r.thresh = sh.prefix;
  r.ties = sh.remaining;
  return r;
}

// A unit split over a cluster, keys in registers: the CTAs exchange what they found with stores that count on the receiver's
// mbarrier when they land. (A cluster barrier of 1024 threads after plain remote stores costs 1.5 to 3 K cycles, most of it the
// release of everything that the threads wrote; a search has five exchanges.) Every CTA sends to all and waits for all, so that
// none can be two exchanges ahead of another: two mbarriers and two buffers, taken in turn, are enough. What is read after an exchange
// is read before the block barrier in front of the next one's sends. A CTA that has been through all exchanges has received all that
// was ever sent to it and may leave. A wait that ran out ends its CTA: what the kernel leaves behind then has to be there before. Its
// peers' next waits run out in turn, and since they may send to it until then it stays until they have all left or given up as well
// (the cluster's barrier counts CTAs that have left. With all CTAs in that barrier 1 x 131072 tokens took 1 us more; with a search
// that returns in place of ending its CTA as much, for registers that it spilled).
template <int CL>
struct Exchange {
  const ta_waits waits;
  int k = 0;  // exchanges begun
  static __device__ __forceinline__ void set_up(SelectShared<CL>& sh) {  // before a barrier of the cluster
    if (threadIdx.x == 0) {
      ta_sm100::mbar_init(ta_sm100::smem_u32(&sh.arrived[0]), 1);
      ta_sm100::mbar_init(ta_sm100::smem_u32(&sh.arrived[1]), 1);
      asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
  }
  // words to the same place in CTA q's shared memory
  __device__ __forceinline__ void send1(SelectShared<CL>& sh, const void* to, int q, uint32_t a) {
    asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.b32 [%0], %1, [%2];" ::"r"(at(to, q)), "r"(a),
                 "r"(at(&sh.arrived[k & 1], q))
                 : "memory");
  }
  __device__ __forceinline__ void send2(SelectShared<CL>& sh, const void* to, int q, uint32_t a, uint32_t b) {
    asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.v2.b32 [%0], {%1, %2}, [%3];" ::"r"(at(to, q)), "r"(a),
                 "r"(b), "r"(at(&sh.arrived[k & 1], q))
                 : "memory");
  }
  __device__ __forceinline__ void send4(SelectShared<CL>& sh, const void* to, int q, uint4 v) {
    asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.v4.b32 [%0], {%1, %2, %3, %4}, [%5];" ::"r"(at(to, q)),
                 "r"(v.x), "r"(v.y), "r"(v.z), "r"(v.w), "r"(at(&sh.arrived[k & 1], q))
                 : "memory");
  }
  // All threads, after the sends: `bytes` have arrived. A barrier of the block. Does not return when they did not come within a limit
  // that CTAs which run together do not reach (reported).
  __device__ __forceinline__ void wait(SelectShared<CL>& sh, uint32_t bytes) {
    const uint32_t bar = ta_sm100::smem_u32(&sh.arrived[k & 1]), parity = (uint32_t)(k >> 1) & 1u;
    if (threadIdx.x == 0) ta_sm100::mbar_expect_tx(bar, bytes);
    ++k;
    bool ok = ta_sm100::mbar_try_wait_cluster(bar, parity);
    if (!ok) ok = wait_slow(bar, parity, waits.limit_ns, waits.status);
    if (__syncthreads_and(ok) == 0) {
      stay();
      asm volatile("exit;");
      __builtin_unreachable();
    }
  }
  // Out of line: with the five waits' loops in a kernel 1 x 60000 tokens of 8 units with their scores took 92.1 us, with this 91.0.
  static __device__ __noinline__ bool wait_slow(uint32_t bar, uint32_t parity, unsigned long long limit_ns, ta_dev_status* status) {
    unsigned long long began = 0;
    for (int tries = 0; !ta_sm100::mbar_try_wait_cluster(bar, parity); ++tries) {
      if ((tries & 63) != 63) continue;
      const unsigned long long now = ta_sm100::globaltimer_ns();
      if (began == 0) began = now;
      if (now - began > limit_ns) {
        if (status && atomicCAS(&status->code, 0, (int)TA_ERR_TIMEOUT) == 0) status->where = 8;
        return false;
      }
    }
    return true;
  }
  static __device__ __forceinline__ void stay() {
    ta_sm100::cluster_arrive();
    ta_sm100::cluster_wait();
    __nanosleep(50000);  // what its peers sent before they arrived has landed
  }

 private:
  static __device__ __forceinline__ uint32_t at(const void* p, int q) {
    return ta_sm100::map_peer(ta_sm100::smem_u32(p), (uint32_t)q);
  }
};
template <>
struct Exchange<1> {
  const ta_waits waits;
  int k = 0;
};

// Shared step of the radix passes: warp 0 walks the 256-bin histogram from the top bin down until `remaining`
// elements are covered and publishes the bin it stops in (sh.prefix gets the digit at `shift`, sh.remaining what is
// still to take inside that bin, sh.ncand the bin's population). Called by all threads of warp 0.
template <int CL>
__device__ __forceinline__ void radix_walk(const uint32_t (&hl)[8], int shift, uint32_t digit_mask, uint32_t prefix,
                                           uint32_t mask, SelectShared<CL>& sh) {
  const int lane = threadIdx.x & 31;  // lane l owns bins [8l, 8l+8): hl
  uint32_t tot = 0;
#pragma unroll
  for (int k = 0; k < 8; ++k) tot += hl[k];
  uint32_t run = tot;  // inclusive sum over this lane and the lanes above it
#pragma unroll
  for (int off = 1; off < 32; off <<= 1) {
    const uint32_t o = __shfl_down_sync(0xffffffffu, run, off);
    if (lane + off < 32) run += o;
  }
  const uint32_t above = run - tot;
  const uint32_t remaining = (uint32_t)sh.remaining;
  if (above < remaining && remaining <= above + tot) {
    uint32_t cum = above;
    int k = 7;
#pragma unroll
    for (int kk = 7; kk > 0; --kk) {
      if (k == kk && cum + hl[kk] < remaining) {
        cum += hl[kk];
        k = kk - 1;
      }
    }
    uint32_t pop = hl[0];
#pragma unroll
    for (int kk = 1; kk < 8; ++kk)
      if (k == kk) pop = hl[kk];
    const int bin = 8 * lane + k;
    sh.remaining = (int)(remaining - cum);
    sh.ncand = (int)pop;
    sh.prefix = prefix | ((uint32_t)bin << shift);
    sh.mask = mask | (digit_mask << shift);
  }
}

template <int CL>
__device__ __forceinline__ void radix_walk(const uint32_t* hist, int shift, uint32_t digit_mask, uint32_t prefix,
                                           uint32_t mask, SelectShared<CL>& sh) {
  uint32_t hl[8];
#pragma unroll
  for (int k = 0; k < 8; ++k) hl[k] = hist[8 * (threadIdx.x & 31) + k];
  radix_walk(hl, shift, digit_mask, prefix, mask, sh);
}

// The remaining radix passes over the m candidate keys in sh.cand_keys (all of them match `prefix` under `mask`),
// with block barriers only. On return prefix/remaining describe the threshold as at the end of the register passes.
template <int CL>
__device__ __forceinline__ void list_radix_finish(int m, int bits, int done, uint32_t& prefix, uint32_t& mask,
                                                  int& remaining, SelectShared<CL>& sh) {
  const int tid = threadIdx.x;
  constexpr int kPer = (kCandCap + kThreads - 1) / kThreads;
  uint32_t lk[kPer];
  uint32_t live = 0;
#pragma unroll
  for (int q = 0; q < kPer; ++q) {
    const int j = tid + q * kThreads;
    lk[q] = j < m ? sh.cand_keys[j] : 0u;
    if (j < m) live |= 1u << q;
  }
  if (tid == 0) sh.remaining = remaining;
  while (done < bits) {
    const int width = min(8, bits - done), shift = bits - done - width;
    const uint32_t digit_mask = (1u << width) - 1u;
    for (int k = tid; k < 256; k += kThreads) sh.hist[k] = 0;
    __syncthreads();
#pragma unroll
    for (int q = 0; q < kPer; ++q) {
      if ((live >> q) & 1u) {
        if ((lk[q] & mask) != prefix) live &= ~(1u << q);
        else atomicAdd(&sh.hist[(lk[q] >> shift) & digit_mask], 1u);
      }
    }
    __syncthreads();
    if (tid < 32) radix_walk(sh.hist, shift, digit_mask, prefix, mask, sh);
    __syncthreads();
    prefix = sh.prefix;
    mask = sh.mask;
    remaining = sh.remaining;
    const int ncand = sh.ncand;
    done += width;
    if (ncand == remaining) break;
  }
}

// The `remaining`-th largest of the m <= kCompareCap keys in sh.cand_keys, by comparing every key with every other: two block
// barriers in place of three for every digit still to resolve. Returns the key; above / equal: how many keys are larger than
// it / equal to it. One warp, a key per lane: beyond 32 keys another digit is cheaper, integer compares run at half rate (256
// keys among 4096: 3.6 K cycles shared out over 32 warps, 1.7 K for a digit and the comparison of what it leaves).
// compare_begin() runs before the barrier that publishes the keys.
template <int CL>
__device__ __forceinline__ void compare_begin(int m, SelectShared<CL>& sh) {
  const int tid = threadIdx.x;
  if (tid >= m && tid < (m + 3) / 4 * 4) sh.cand_keys[tid] = 0u;  // above no key
}
template <int CL>
__device__ __forceinline__ uint32_t compare_finish(int m, int remaining, int& above, int& equal, SelectShared<CL>& sh) {
  const int tid = threadIdx.x;
  static_assert(kCompareCap == 32, "a key per lane");
  if (tid < 32) {
    const uint32_t mine = tid < m ? sh.cand_keys[tid] : 0u;
    const uint4* keys = reinterpret_cast<const uint4*>(sh.cand_keys);
    int gt = 0;
#pragma unroll 2
    for (int j = 0; j < (m + 3) / 4; ++j) {
      const uint4 k = keys[j];
      gt += (k.x > mine) + (k.y > mine) + (k.z > mine) + (k.w > mine);
    }
    // the key with the most keys above it among those with fewer than `remaining`; equal keys have equal counts
    const int best = __reduce_max_sync(0xffffffffu, tid < m && gt < remaining ? gt : -1);
    const unsigned same = __ballot_sync(0xffffffffu, tid < m && gt == best);
    if (tid == __ffs((int)same) - 1) {
      sh.cmp_thresh = mine;
      sh.cmp_above = best;
      sh.cmp_equal = __popc(same);
    }
  }
  __syncthreads();
  above = sh.cmp_above;
  equal = sh.cmp_equal;
  return sh.cmp_thresh;
}

// Top-`want` of the eligible elements when the keys sit in registers. The eligible keys' range is taken first: the
// bits above the highest bit in which two of them differ are common to all and need no pass, so the first 8-bit
// digit already spreads the keys over the whole histogram (utilities of one unit span a few binades: the top byte of
// a float alone would put most of them into two or three bins). The first pass counts every eligible element
// (match.any merges equal digits of a warp into one shared-memory atomic); from then on each thread keeps a bit mask
// of its elements that are still candidates, and the passes touch those only. The passes stop as soon as the
// candidates left are exactly as many as are still to take, or so few that they are compared with one another. FEW (an instance of
// its own: the code costs large budgets 0.6 %): few are wanted. n_unit is the length of the whole unit (n is this CTA's
// slice when CL > 1).
template <int CL, bool FEW = false, int ITEMS>
__device__ SelectResult cached_radix_select(int n, int n_unit, int want, const KeyCache<ITEMS>& kc, SelectShared<CL>& sh,
                                            Exchange<CL>& ex) {
  SelectResult r;
  r.thresh = 0;
  r.ties = 0;
  r.all = 0;
  r.all_ties = 0;
  r.none = (want <= 0);
  if (r.none) return r;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const unsigned lt = (1u << lane) - 1u;
  uint32_t cand = kc.elig;
  uint32_t kmin = 0xffffffffu, kmax = 0u;
#pragma unroll
  for (int it = 0; it < ITEMS; ++it) {
    if ((cand >> it) & 1u) {
      kmin = min(kmin, kc.key[it]);
      kmax = max(kmax, kc.key[it]);
    }
  }
  if (tid == 0) {
    sh.remaining = want;
    sh.cmp_n = 0;
    sh.cand_n = 0;
  }
  static_assert(kWarps <= 32, "one lane per warp in the second reduction step");
  uint32_t num = 0;
  bool bounded = false;
  if constexpr (FEW) {
    static_assert(CL == 1, "one block's threads");
    if (want <= kThreads / 2) {
      // Few are wanted: the want-th largest of the threads' own largest keys is a lower bound of the threshold, and a digit of
      // those (one per thread) costs a fraction of a digit of all keys. Few keys are at or above it.
      const uint32_t mine = kmax;  // (0: no eligible key)
      const uint32_t lo_w = __reduce_min_sync(0xffffffffu, cand != 0u ? mine : 0xffffffffu);
      const uint32_t hi_w = __reduce_max_sync(0xffffffffu, mine);
      const int with = __popc(__ballot_sync(0xffffffffu, cand != 0u));
      if (lane == 0) {
        sh.wmin[warp] = lo_w;
        sh.wmax[warp] = hi_w;
        sh.wnum[warp] = (uint32_t)with;
      }
      for (int k = tid; k < 256; k += kThreads) sh.hist[k] = 0;
      __syncthreads();
      const uint32_t lo = __reduce_min_sync(0xffffffffu, lane < kWarps ? sh.wmin[lane] : 0xffffffffu);
      const uint32_t hi = __reduce_max_sync(0xffffffffu, lane < kWarps ? sh.wmax[lane] : 0u);
      const uint32_t threads_with = __reduce_add_sync(0xffffffffu, lane < kWarps ? sh.wnum[lane] : 0u);
      bounded = threads_with >= (uint32_t)want;
      if (bounded) {
        uint32_t bound = lo;
        if (lo != hi) {
          const int top = 32 - __clz(lo ^ hi), shift = max(top - 8, 0);
          const uint32_t mask = top == 32 ? 0u : (0xffffffffu << top);
          if (cand != 0u) atomicAdd(&sh.hist[(mine >> shift) & 255u & ~(mask >> shift)], 1u);
          __syncthreads();
          if (tid < 32) radix_walk(sh.hist, shift, 255u, hi & mask, mask, sh);
          __syncthreads();
          bound = sh.prefix;
          if (tid == 0) sh.remaining = want;
        }
        uint32_t above = 0;
#pragma unroll
        for (int it = 0; it < ITEMS; ++it) above |= kc.key[it] >= bound ? (1u << it) : 0u;
        cand &= above;
        kmin = bound;
        kmax = hi;
        num = (uint32_t)max(n_unit / 8, kCompareCap + 1);  // (not known; few of n_unit)
      } else {
        __syncthreads();  // wmin, wmax and wnum are written again
      }
    }
  }
  if (!bounded) {
    kmin = __reduce_min_sync(0xffffffffu, kmin);
    kmax = __reduce_max_sync(0xffffffffu, kmax);
    num = __reduce_add_sync(0xffffffffu, (uint32_t)__popc(cand));
    if (lane == 0) {
      sh.wmin[warp] = kmin;
      sh.wmax[warp] = kmax;
      sh.wnum[warp] = num;
    }
    __syncthreads();
    kmin = __reduce_min_sync(0xffffffffu, lane < kWarps ? sh.wmin[lane] : 0xffffffffu);
    kmax = __reduce_max_sync(0xffffffffu, lane < kWarps ? sh.wmax[lane] : 0u);
    num = __reduce_add_sync(0xffffffffu, lane < kWarps ? sh.wnum[lane] : 0u);
  }
  int first = 0;  // CL > 1: how many of the unit's candidates belong to the CTAs before this one, and how many are its own
  int own = 0;
  if constexpr (CL > 1) {
    const int rank = (int)cg::this_cluster().block_rank();
    if (tid < CL) ex.send4(sh, sh.cl_range[rank], tid, make_uint4(kmin, kmax, num, 0u));
    ex.wait(sh, CL * 16);
    kmin = 0xffffffffu;
    kmax = 0u;
    num = 0u;
#pragma unroll
    for (int q = 0; q < CL; ++q) {
      kmin = min(kmin, sh.cl_range[q][0]);
      kmax = max(kmax, sh.cl_range[q][1]);
      if (q < rank) first += (int)sh.cl_range[q][2];
      if (q == rank) own = (int)sh.cl_range[q][2];
      num += sh.cl_range[q][2];
    }
  }
  if (!bounded && num < (uint32_t)want) {  // fewer eligible elements than requested: all of them
    r.all = 1;
    return r;
  }
  const uint32_t diff = kmin ^ kmax;
  if (diff == 0u) {  // all eligible keys are equal
    r.thresh = kmin;
    r.ties = want;
    r.all_ties = !bounded && num == (uint32_t)want;
    return r;
  }
  const int bits = 32 - __clz(diff);  // low bits still to resolve
  uint32_t mask = bits == 32 ? 0u : (0xffffffffu << bits);
  uint32_t prefix = kmax & mask;
  int remaining = want;
  int ncand = (int)num;
  int done = 0, pass = 0;
  while (done < bits) {
    if (CL == 1 && ncand <= kCompareCap) {
      uint32_t mine = 0;
      if (cand != 0u) {
#pragma unroll
        for (int it = 0; it < ITEMS; ++it)
          if (((cand >> it) & 1u) && (kc.key[it] & mask) == prefix) mine |= 1u << it;
      }
      if (__any_sync(0xffffffffu, mine != 0u)) {  // one atomic per warp: neighbours are often candidates together
        const uint32_t cnt = (uint32_t)__popc(mine);
        uint32_t incl = cnt;
#pragma unroll
        for (int off = 1; off < 32; off <<= 1) {
          const uint32_t o = __shfl_up_sync(0xffffffffu, incl, off);
          if (lane >= off) incl += o;
        }
        uint32_t slot = 0;
        if (lane == 31) slot = atomicAdd(&sh.cmp_n, incl);
        slot = __shfl_sync(0xffffffffu, slot, 31) + incl - cnt;
#pragma unroll
        for (int it = 0; it < ITEMS; ++it)
          if ((mine >> it) & 1u) sh.cand_keys[slot++] = kc.key[it];
      }
      compare_begin(ncand, sh);
      __syncthreads();
      int above, equal;
      r.thresh = compare_finish(ncand, remaining, above, equal, sh);
      r.ties = remaining - above;
      r.all_ties = r.ties == equal;
      return r;
    }
    if constexpr (CL > 1) if (ncand <= kCandCap) {
      // Few candidates left (uniform over the cluster: every CTA knows how many each of them has). Every CTA sends its own to
      // the lists of all, behind those of the CTAs before it; when all have arrived every CTA finishes alone. Only the
      // multiset of keys decides the threshold, so that all arrive at the same one. Every CTA also sends a word to all: one
      // that has all the candidates would wait for nobody without it, and its next exchange could reach a CTA that is still
      // in the one before this.
      uint32_t mine = 0;
      if (cand != 0u) {
#pragma unroll
        for (int it = 0; it < ITEMS; ++it)
          if (((cand >> it) & 1u) && (kc.key[it] & mask) == prefix) mine |= 1u << it;
      }
      if (__any_sync(0xffffffffu, mine != 0u)) {
        const uint32_t cnt = (uint32_t)__popc(mine);
        uint32_t incl = cnt;
#pragma unroll
        for (int off = 1; off < 32; off <<= 1) {
          const uint32_t o = __shfl_up_sync(0xffffffffu, incl, off);
          if (lane >= off) incl += o;
        }
        uint32_t slot = 0;
        if (lane == 31) slot = atomicAdd(&sh.cand_n, incl);
        slot = (uint32_t)first + __shfl_sync(0xffffffffu, slot, 31) + incl - cnt;
#pragma unroll
        for (int it = 0; it < ITEMS; ++it)
          if ((mine >> it) & 1u) sh.cand_keys[min(slot++, (uint32_t)kCandCap - 1u)] = kc.key[it];
      }
      __syncthreads();
      const int rank = (int)cg::this_cluster().block_rank();
      if (tid < CL) ex.send1(sh, &sh.took_part[rank], tid, 0u);
      for (int j = tid; j < own * CL; j += kThreads) {
        const int q = j / own, at = min(first + j - q * own, kCandCap - 1);
        if (q != rank) ex.send1(sh, &sh.cand_keys[at], q, sh.cand_keys[at]);
      }
      ex.wait(sh, (uint32_t)(CL + ncand - own) * 4u);
      list_radix_finish(ncand, bits, done, prefix, mask, remaining, sh);
      break;
    }
    const int width = min(8, bits - done), shift = bits - done - width;
    const uint32_t digit_mask = (1u << width) - 1u;
    for (int k = tid; k < 256; k += kThreads) sh.hist[k] = 0;
    __syncthreads();
    if ((pass == 0 && !bounded) || ncand * 4 > n_unit) {  // most elements are candidates (uniform over the unit's CTAs)
#pragma unroll
      for (int it = 0; it < ITEMS; ++it) {
        if (it * kThreads < n) {
          const bool c = ((cand >> it) & 1u) != 0 && (kc.key[it] & mask) == prefix;
          if (!c) cand &= ~(1u << it);
          const int bin = c ? (int)((kc.key[it] >> shift) & digit_mask) : -1;
          const unsigned peers = __match_any_sync(0xffffffffu, bin);
          if (c && (peers & lt) == 0u) atomicAdd(&sh.hist[bin], (uint32_t)__popc(peers));
        }
      }
    } else if (cand != 0u) {
#pragma unroll
      for (int it = 0; it < ITEMS; ++it) {
        if ((cand >> it) & 1u) {
          if ((kc.key[it] & mask) != prefix) cand &= ~(1u << it);
          else atomicAdd(&sh.hist[(kc.key[it] >> shift) & digit_mask], 1u);
        }
      }
    }
    __syncthreads();
    if constexpr (CL > 1) {
      // Every CTA sends its histogram to all and takes the same decision from the sum. (Added up by remote atomics on one CTA
      // and read from there, a search among 16 CTAs took 25 K cycles: distributed shared memory moves some 10 bytes a clock.)
      const int rank = (int)cg::this_cluster().block_rank();
      for (int j = tid; j < 32 * CL; j += kThreads) {
        const int q = j / 32, k = j % 32;  // bins 8k .. 8k + 7 (at most 32768 keys a CTA: 16 bits hold a count)
        const uint4 a = reinterpret_cast<const uint4*>(sh.hist)[2 * k], b = reinterpret_cast<const uint4*>(sh.hist)[2 * k + 1];
        ex.send4(sh, &sh.ghist[pass & 1][rank][4 * k], q,
                 make_uint4(a.x | (a.y << 16), a.z | (a.w << 16), b.x | (b.y << 16), b.z | (b.w << 16)));
      }
      ex.wait(sh, CL * 512);
      if (tid < 32) {
        uint32_t hl[8] = {0u, 0u, 0u, 0u, 0u, 0u, 0u, 0u};
#pragma unroll 4
        for (int q = 0; q < CL; ++q) {
          const uint4 v = reinterpret_cast<const uint4*>(&sh.ghist[pass & 1][q][0])[lane];
          const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
          for (int k = 0; k < 4; ++k) {
            hl[2 * k] += w[k] & 0xffffu;
            hl[2 * k + 1] += w[k] >> 16;
          }
        }
        radix_walk(hl, shift, digit_mask, prefix, mask, sh);
      }
    } else if (tid < 32) {
      radix_walk(sh.hist, shift, digit_mask, prefix, mask, sh);
    }
    __syncthreads();
    prefix = sh.prefix;
    mask = sh.mask;
    remaining = sh.remaining;
    ncand = sh.ncand;
    if constexpr (CL > 1) {  // who has how many of the bin that the threshold fell into
      const int rank = (int)cg::this_cluster().block_rank();
      const uint32_t bin = (prefix >> shift) & digit_mask;
      const uint32_t n_q = lane < CL ? (sh.ghist[pass & 1][lane & (CL - 1)][bin >> 1] >> (16 * (bin & 1))) & 0xffffu : 0u;
      first = (int)__reduce_add_sync(0xffffffffu, lane < rank ? n_q : 0u);
      own = (int)__shfl_sync(0xffffffffu, n_q, rank);
    }
    done += width;
    ++pass;
    if (ncand == remaining) {  // every candidate left is taken: the low bits need no pass
      r.all_ties = 1;
      break;
    }
  }
  r.thresh = prefix;  // with the unresolved low bits zero: candidates above it are definite, equal ones are ties
  r.ties = remaining;
  return r;
}

// Ordered pass over [0, n): classify(i, eligible, key, def, tie) marks element i `definite` (taken for sure) or a
// `tie` (taken while ties last). Calls emit(i, rank) for every taken element with its rank in ascending position
// order. Returns the number taken.
template <bool CACHED, class KeyFn, class ClassFn, class EmitFn, int ITEMS, int CL>
__device__ int block_ordered_emit(int n, int ties_allowed, KeyFn key_of, const KeyCache<ITEMS>& kc, ClassFn classify,
                                  EmitFn emit, SelectShared<CL>& sh, int def_base = 0, int tie_base = 0,
                                  int* def_total_out = nullptr, int* tie_total_out = nullptr) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int def0 = def_base, tie0 = tie_base;
  sweep<CACHED>(n, key_of, kc, [&](int i, bool exists, bool elig, uint32_t key) {
    bool def = false, tie = false;
    if (exists) classify(i, elig, key, def, tie);
    const unsigned bd = __ballot_sync(0xffffffffu, def), bt = __ballot_sync(0xffffffffu, tie);
    const unsigned lt = (1u << lane) - 1u;
    if (lane == 0) sh.warp_cnt[warp] = (uint32_t)__popc(bd) | ((uint32_t)__popc(bt) << 16);
    __syncthreads();
    uint32_t before = 0, total = 0;
    const uint4* wc = reinterpret_cast<const uint4*>(sh.warp_cnt);
#pragma unroll
    for (int q = 0; q < kWarps / 4; ++q) {
      const uint4 c4 = wc[q];
      const uint32_t cs[4] = {c4.x, c4.y, c4.z, c4.w};
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        total += cs[e];
        if (4 * q + e < warp) before += cs[e];
      }
    }
    const int def_before = (int)(before & 0xffffu) + __popc(bd & lt);
    const int ties_seen = tie_base + (int)(before >> 16) + __popc(bt & lt);
    if (def)
      emit(i, def_base + def_before + min(ties_seen, ties_allowed));
    else if (tie && ties_seen < ties_allowed)
      emit(i, def_base + def_before + ties_seen);
    def_base += (int)(total & 0xffffu);
    tie_base += (int)(total >> 16);
    __syncthreads();
  });
  if (def_total_out) *def_total_out = def_base - def0;
  if (tie_total_out) *tie_total_out = tie_base - tie0;
  return def_base + min(tie_base, ties_allowed);
}

// Bit `it` set for every chunk in which this thread's slot (tid + it * kThreads) lies inside [0, n).
__device__ __forceinline__ uint32_t exist_mask(int n) {
  const int tid = threadIdx.x;
  const int cnt = n > tid ? (n - tid + kThreads - 1) / kThreads : 0;
  return cnt >= 32 ? 0xffffffffu : ((1u << cnt) - 1u);
}

// Transpose of a 32 x 32 bit matrix held one row per lane: on return lane i holds, in bit l, what was bit i of lane l.
// Five butterfly steps, each swapping the off-diagonal blocks of size s with the lane s away.
__device__ __forceinline__ uint32_t warp_transpose32(uint32_t x, int lane) {
#pragma unroll
  for (int s = 16; s >= 1; s >>= 1) {
    const uint32_t m = s == 16 ? 0x0000ffffu : s == 8 ? 0x00ff00ffu : s == 4 ? 0x0f0f0f0fu : s == 2 ? 0x33333333u : 0x55555555u;
    const uint32_t y = __shfl_xor_sync(0xffffffffu, x, s);
    x = (lane & s) ? ((x & ~m) | ((y >> s) & m)) : ((x & m) | ((y << s) & ~m));
  }
  return x;
}

// The ordered pass when the keys sit in registers (ITEMS chunks of kThreads elements, element tid + it*kThreads in
// chunk it). One sweep classifies every element (each thread collects its own 32 bits, one in-warp bit transpose turns
// them into what 32 ballots would give) and leaves two bitmaps in shared memory, definite and tie, in position
// order: the bits of warp w in chunk it are word it*kWarps + w and cover positions 32 * word .. + 31.
// From there on thread j owns word j: a block-wide exclusive scan over the words' populations gives it the number
// of definite and of tie elements before its 32 positions, and the taken positions are written from the words alone
// (no key is needed for that). Three or four block barriers (and one exchange of the CTAs' totals). emit may run on another thread than the one that holds the element's key.
template <int CL, class EmitFn, int ITEMS>
__device__ int cached_ordered_emit(int n, const SelectResult& r, const KeyCache<ITEMS>& kc, uint32_t always,
                                   EmitFn emit, SelectShared<CL>& sh, Exchange<CL>& ex) {
  static_assert(ITEMS <= kItemsLong && ITEMS <= 32, "per-thread masks hold one bit per chunk");
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int chunks = (n + kThreads - 1) / kThreads;
  // per thread: bit `it` of mdef / mtie = its element of chunk `it` is definite / a tie. `always` marks the elements
  // taken whatever their key (not eligible for the search); eligible ones are definite above the threshold and ties
  // at it. The elig bits exist only for elements inside the unit.
  const int ties_allowed = r.ties;
  uint32_t mdef = always, mtie = 0;
  if (!r.none) {
    if (r.all) {
      mdef |= kc.elig;
    } else {
      uint32_t above = 0, equal = 0;
#pragma unroll
      for (int it = 0; it < ITEMS; ++it) {
        if (it < chunks) {
          above |= kc.key[it] > r.thresh ? (1u << it) : 0u;
          equal |= kc.key[it] == r.thresh ? (1u << it) : 0u;
        }
      }
      mdef |= kc.elig & above;
      mtie = kc.elig & equal;
      if (r.all_ties) {  // every tie is taken: none are told apart
        mdef |= mtie;
        mtie = 0;
      }
    }
  }
  // the warp's 32 x 32 bits transposed: lane `it` then holds the ballot of chunk `it` (bit l = lane l's element)
  mdef = warp_transpose32(mdef, lane);
  if (!r.all_ties) mtie = warp_transpose32(mtie, lane);
  if (lane < chunks) {
    sh.bdef[lane * (kWarps + 1) + warp] = mdef;
    sh.btie[lane * (kWarps + 1) + warp] = mtie;
  }
  __syncthreads();
  // exclusive scan of the packed populations over the chunks * kWarps words (word tid belongs to thread tid)
  static_assert(kItemsLong * kWarps <= kThreads, "one word per thread");
  const bool owner = tid < chunks * kWarps;
  const int slot = tid + tid / kWarps;  // word tid = (chunk tid / kWarps, warp tid % kWarps) in the padded rows
  const uint32_t wd = owner ? sh.bdef[slot] : 0u, wt = owner ? sh.btie[slot] : 0u;
  const uint32_t mine = (uint32_t)__popc(wd) | ((uint32_t)__popc(wt) << 16);
  uint32_t run = mine;
#pragma unroll
  for (int off = 1; off < 32; off <<= 1) {
    const uint32_t o = __shfl_up_sync(0xffffffffu, run, off);
    if (lane >= off) run += o;
  }
  const uint32_t warp_total = __shfl_sync(0xffffffffu, run, 31);
  const uint32_t warp_most = __reduce_max_sync(0xffffffffu, (uint32_t)__popc(wd | wt));
  if (lane == 0) {
    sh.wtot[warp] = warp_total;
    sh.wmax[warp] = warp_most;
  }
  __syncthreads();
  const int most = (int)__reduce_max_sync(0xffffffffu, lane < kWarps ? sh.wmax[lane] : 0u);  // in one word
  const uint32_t wt_l = lane < kWarps ? sh.wtot[lane] : 0u;  // (no carry between the halves: at most 32768 elements)
  const uint32_t before = __reduce_add_sync(0xffffffffu, lane < warp ? wt_l : 0u);
  const uint32_t all = __reduce_add_sync(0xffffffffu, wt_l);
  const uint32_t upto = before + run - mine;
  int def_base = 0, tie_base = 0;
  const int def_mine = (int)(all & 0xffffu), tie_mine = (int)(all >> 16);
  int def_all = def_mine, tie_all = tie_mine;
  if constexpr (CL > 1) {
    const int rank = (int)cg::this_cluster().block_rank(), turn = ex.k & 1;
    if (tid < CL) ex.send2(sh, sh.totals[turn][rank], tid, (uint32_t)def_all, (uint32_t)tie_all);
    ex.wait(sh, CL * 8);
    def_all = 0;
    tie_all = 0;
#pragma unroll
    for (int r = 0; r < CL; ++r) {
      if (r < rank) {
        def_base += sh.totals[turn][r][0];
        tie_base += sh.totals[turn][r][1];
      }
      def_all += sh.totals[turn][r][0];
      tie_all += sh.totals[turn][r][1];
    }
  }
  int def_before = def_base + (int)(upto & 0xffffu);
  int ties_seen = tie_base + (int)(upto >> 16);
  uint32_t m = wd | wt;
  // Sparse words: every thread walks its own word. Dense ones (recency makes runs of neighbours win together, so that a few
  // words hold most of what is taken): the warps of the block share the words, a lane per position (TA-Fast, 1024 of 4096
  // tokens, with the search above: 58.2 -> 55.8 us a call). A warp meets at most `chunks` words that are not empty that
  // way, a thread up to `most` positions the other way.
  if (most > min(chunks, (def_mine + tie_mine) / kWarps + 1) + 2) {
    sh.before[tid] = upto;
    __syncthreads();
    const unsigned lt = (1u << lane) - 1u;
    const int row = lane * (kWarps + 1) + warp;
    for (unsigned left = __ballot_sync(0xffffffffu, lane < chunks && (sh.bdef[row] | sh.btie[row]) != 0u); left != 0u;
         left &= left - 1u) {
      const int k = __ffs((int)left) - 1;
      const uint32_t d = sh.bdef[k * (kWarps + 1) + warp], t = sh.btie[k * (kWarps + 1) + warp];
      const uint32_t first = sh.before[k * kWarps + warp];
      const int seen = tie_base + (int)(first >> 16) + __popc(t & lt);
      const int rank = def_base + (int)(first & 0xffffu) + __popc(d & lt) + min(seen, ties_allowed);
      if (((d >> lane) & 1u) || (((t >> lane) & 1u) && seen < ties_allowed)) emit(32 * (k * kWarps + warp) + lane, rank);
    }
  } else {
    while (m) {
      const int bit = __ffs((int)m) - 1;
      m &= m - 1u;
      const int i = 32 * tid + bit;
      if ((wd >> bit) & 1u) {
        emit(i, def_before + min(ties_seen, ties_allowed));
        ++def_before;
      } else {
        if (ties_seen < ties_allowed) emit(i, def_before + ties_seen);
        ++ties_seen;
      }
    }
  }
  return def_all + min(tie_all, ties_allowed);
}

// The ordered pass for a unit split over CL CTAs (rank r owns a contiguous, ascending slice): a counting sweep
// gives every CTA its (definite, tie) totals, the totals are exchanged through distributed shared memory, and the
// emitting sweep starts from the sums of the lower ranks. Returns the number taken over the whole unit.
template <bool CACHED, int CL, class KeyFn, class ClassFn, class EmitFn, int ITEMS>
__device__ int cluster_ordered_emit(int n, int ties_allowed, KeyFn key_of, const KeyCache<ITEMS>& kc, ClassFn classify,
                                    EmitFn emit, SelectShared<CL>& sh) {
  static_assert(!CACHED, "keys in registers: call cached_ordered_emit");
  if (CL == 1) return block_ordered_emit<CACHED>(n, ties_allowed, key_of, kc, classify, emit, sh);
  cg::cluster_group cluster = cg::this_cluster();
  const int rank = (int)cluster.block_rank();
  int dt = 0, tt = 0;
  block_ordered_emit<CACHED>(n, 0, key_of, kc, classify, [](int, int) {}, sh, 0, 0, &dt, &tt);
  if (threadIdx.x < CL) {
    int* peer = cluster.map_shared_rank(&sh.totals[0][0][0], threadIdx.x);
    peer[rank * 2 + 0] = dt;
    peer[rank * 2 + 1] = tt;
  }
  cluster.sync();
  int def_base = 0, tie_base = 0, def_all = 0, tie_all = 0;
#pragma unroll
  for (int r = 0; r < CL; ++r) {
    if (r < rank) {
      def_base += sh.totals[0][r][0];
      tie_base += sh.totals[0][r][1];
    }
    def_all += sh.totals[0][r][0];
    tie_all += sh.totals[0][r][1];
  }
  block_ordered_emit<CACHED>(n, ties_allowed, key_of, kc, classify, emit, sh, def_base, tie_base);
  return def_all + min(tie_all, ties_allowed);
}

// Slice [lo, hi) of a unit of n elements owned by this CTA when the unit is split over CL CTAs (whole chunks of
// kThreads elements per CTA so that the slices stay aligned).
template <int CL>
__device__ __forceinline__ void unit_slice(int n, int& lo, int& hi) {
  if (CL == 1) {
    lo = 0;
    hi = n;
    return;
  }
  const int rank = (int)cg::this_cluster().block_rank();
  const int per = ((n + CL - 1) / CL + kThreads - 1) / kThreads * kThreads;
  lo = min(n, rank * per);
  hi = min(n, lo + per);
}

struct SeqInfo {
  int start, n, K_eff, s_take, r_take, p;
  bool bad;  // the sequence does not lie inside the token arrays (cu_seqlens is device data the host cannot check)
};

__device__ __forceinline__ SeqInfo seq_info(const ta_seq_desc& seq, int b, int K, int n_sink, int n_recent,
                                            int k_protected) {
  SeqInfo s;
  s.start = ta_seq_begin(seq, b);
  s.n = (seq.cu ? seq.cu[b + 1] : s.start + seq.n_uniform) - s.start;
  s.bad = s.n < 0 || s.n > seq.max_n || s.start < 0 || (long long)s.start + s.n > seq.total;
  if (s.bad) s.n = 0;
  s.K_eff = min(K, s.n);
  int p = k_protected < 0 ? s.K_eff - n_sink - n_recent : k_protected;
  p = max(0, min(p, s.K_eff));
  s.p = p;
  const int K_main = s.K_eff - p;
  // mandatory list: sinks 0.. then recents n-1, n-2, .. (no duplicates), truncated to K_main entries
  const int sinks = min(n_sink, s.n);
  const int recents = max(0, min(n_recent, s.n - sinks));
  s.s_take = min(sinks, K_main);
  s.r_take = min(recents, K_main - s.s_take);
  return s;
}

template <bool CACHED, int CL, int ITEMS = kItems>
__global__ void __launch_bounds__(kThreads, 1024 / kThreads) ta_forced_kernel(ta_seq_desc seq, int K, int n_sink, int n_recent,
                                                             int k_protected, const float* voucher,
                                                             uint8_t* __restrict__ forced,
                                                             int32_t* __restrict__ r_main, ta_waits waits,
                                                             const int32_t* __restrict__ class_K, ta_static_out so) {
  __shared__ SelectShared<CL> sh;
  ta_launch_dependents();  // its dependent does not start before every block of the kernel before it runs
  ta_wait_for_prior_grid();
  // grid.x = classes * sequences * CL; without budget classes there is one class and K is the argument
  const int b = (blockIdx.x / CL) % seq.batch;
  const int cls = (blockIdx.x / CL) / seq.batch;
  if (class_K) {
    K = class_K[cls];
    forced += (long long)cls * seq.total;
    r_main += cls * seq.batch;
  }
  const SeqInfo s = seq_info(seq, b, K, n_sink, n_recent, k_protected);
  if (so.out && cls == 0) {  // the static utilities of this CTA's slice (a rejected sequence has s.n == 0)
    int slo, shi;
    unit_slice<CL>(s.n, slo, shi);
    // eight tokens per thread and step: their loads (id, then count of that id, flags, voucher) are in flight together
    for (int i0 = slo + (int)threadIdx.x; i0 < shi; i0 += 8 * kThreads) {
      int id[8], c[8];
      uint8_t fl[8];
      float V[8];
#pragma unroll
      for (int q = 0; q < 8; ++q) {
        const int i = i0 + q * kThreads;
        const long long tok = (long long)s.start + i;
        id[q] = i < shi ? so.ids[tok] : -1;
        fl[q] = i < shi ? so.flags[tok] : (uint8_t)0;
        V[q] = i < shi ? voucher[tok] : 0.0f;
      }
#pragma unroll
      for (int q = 0; q < 8; ++q) c[q] = (id[q] >= 0 && id[q] < so.vocab) ? so.hist[(long long)b * so.vocab + id[q]] : 0;
#pragma unroll
      for (int q = 0; q < 8; ++q) {
        const int i = i0 + q * kThreads;
        if (i < shi)
          so.out[(long long)s.start + i] = ta_static_utility(i, s.n, c[q], (fl[q] & TA_FLAG_ANCHOR_TOKEN) != 0, V[q],
                                                             so.beta, so.gamma, so.lambda);
      }
    }
  }
  if (s.bad) {
    if (threadIdx.x == 0) {
      if (atomicCAS(&waits.status->code, 0, (int)TA_ERR_DEVICE_BOUNDS) == 0) {
        waits.status->where = 3;
        waits.status->detail0 = b;
        waits.status->detail1 = s.start;
      }
      r_main[b] = -2;  // poisoned: the select kernel writes an empty result
    }
    return;
  }
  if (s.K_eff == s.n) {
    if (threadIdx.x == 0) r_main[b] = -1;  // keep everything
    return;
  }
  int lo, hi;
  unit_slice<CL>(s.n, lo, hi);
  const float* V = voucher + s.start + lo;  // this CTA's slice; local index il <-> position lo + il
  auto mandatory = [&](int i) { return i < s.s_take || i >= s.n - s.r_take; };
  auto key_of = [&](int il, uint32_t& key) {
    const float v = V[il];
    key = sortable_key(v);
    return v > 0.0f && !mandatory(lo + il);
  };
  KeyCache<ITEMS> kc;
  Exchange<CL> ex{waits};
  if constexpr (CACHED && CL > 1) {
    if (threadIdx.x == 0 && blockIdx.x % CL == 0) r_main[b] = -2;  // what a wait that runs out leaves: an empty result
    ex.set_up(sh);
    cg::this_cluster().barrier_arrive();
  }
  if constexpr (CACHED) {  // loads as selects, never under a branch: nothing keeps them from being in flight together
    float v[ITEMS];
#pragma unroll
    for (int it = 0; it < ITEMS; ++it) {
      const int il = (int)threadIdx.x + it * kThreads;
      v[it] = il < hi - lo ? V[il] : 0.0f;
      if (CL > 1 && il < hi - lo) forced[s.start + lo + il] = 0;  // before a wait can run out: no flags of an earlier call are left
    }
    kc.elig = 0;
#pragma unroll
    for (int it = 0; it < ITEMS; ++it) {
      const int il = (int)threadIdx.x + it * kThreads;
      kc.key[it] = sortable_key(v[it]);
      if (il < hi - lo && v[it] > 0.0f && !mandatory(lo + il)) kc.elig |= 1u << it;
    }
  }
  SelectResult r;
  if constexpr (CACHED && CL > 1) cg::this_cluster().barrier_wait();
  if constexpr (CACHED) r = cached_radix_select<CL>(hi - lo, s.n, s.p, kc, sh, ex);
  else r = block_radix_select<CACHED, CL>(hi - lo, s.p, key_of, kc, sh);
  uint8_t* f = forced + s.start + lo;
  // ordered pass: mandatory tokens and vouchers above the threshold are forced for sure; vouchers equal to the
  // threshold are forced while protected slots last, lowest position first
  auto classify = [&](int il, bool cand, uint32_t key, bool& def, bool& tie) {
    def = mandatory(lo + il) || (cand && !r.none && (r.all || key > r.thresh));
    tie = !def && cand && !r.none && !r.all && key == r.thresh;
    f[il] = 0;  // set by emit when taken (later, after a block barrier; possibly by another thread)
  };
  auto emit = [&](int il, int rank) { f[il] = 1; };
  int taken;
  if constexpr (CACHED) {
    uint32_t always = 0;  // the mandatory tokens; every flag is cleared (here or above) and set by emit after a block barrier
#pragma unroll
    for (int it = 0; it < ITEMS; ++it) {
      const int il = (int)threadIdx.x + it * kThreads;
      if (il < hi - lo) {
        if (CL == 1) f[il] = 0;
        if (mandatory(lo + il)) always |= 1u << it;
      }
    }
    taken = cached_ordered_emit<CL>(hi - lo, r, kc, always, emit, sh, ex);
  } else {
    taken = cluster_ordered_emit<CACHED, CL>(hi - lo, r.ties, key_of, kc, classify, emit, sh);
  }
  if (threadIdx.x == 0 && blockIdx.x % CL == 0) r_main[b] = s.K_eff - taken;
}

struct UnitSrc {  // where a unit's utility comes from
  const float* u;         // fused: [L][Hkv][total]
  const float* A;         // unfused
  const float* P;
  const float* u_static;  // per token
  float alpha, delta;
  ta_waits waits;
};

__device__ __forceinline__ float unit_utility(const UnitSrc& src, long long unit_off, long long tok) {
  const float u0 = src.u_static[tok];
  if (src.u) return __fadd_rn(src.u[unit_off + tok], u0);
  if (!src.A) return u0;
  const float aA = __fmul_rn(src.alpha, src.A[unit_off + tok]);
  const float dP = __fmul_rn(src.delta, src.P ? src.P[unit_off + tok] : 0.0f);
  return __fadd_rn(__fadd_rn(aA, dP), u0);
}

// The block that selected a unit also moves its retained K and V rows (Algorithm 1 step 9): same result as
// ta_compact_kernel (rows at and beyond the retained count, and rows whose index lies outside the sequence, are zero).
// Selection is bound by latency and instruction issue, the copy by HBM: with many units the blocks of one kernel are in
// different phases and the two overlap in part (2048 units of up to 8000 tokens, K = 512: 105 + 175 us as two kernels,
// 210 us as one; starting half of the blocks half a period late changed nothing); with few, a launch is saved.
struct GatherDst {
  ta_bf16_view k, v;
  uint4* k_out;
  uint4* v_out;
};

// Rows are listed in `list` (the first kCandCap of them) and in `out`; all: row r is position r. Of `blocks` blocks that share
// the unit's rows this is number `block`.
__device__ __forceinline__ void gather_unit(const GatherDst& gd, const ta_seq_desc& seq, int unit, int l, int b, int g,
                                            int n, int K, const int32_t* out, int taken, bool all, const uint32_t* list,
                                            int block = 0, int blocks = 1) {
  constexpr int kLanesPerRow = TA_HEAD_DIM * 2 / 16;  // a warp moves the K and the V row of one position at a time
  constexpr int kUnroll = 8;
  static_assert(2 * kLanesPerRow == 32, "one lane per 16-byte piece of a K row and a V row");
  __syncthreads();  // the unit's indices were written by other threads of this block
  const int lane = threadIdx.x & 31, which = lane / kLanesPerRow, piece = lane % kLanesPerRow;
  const ta_bf16_view& src = which ? gd.v : gd.k;
  const long long base = (long long)l * src.stride_l + (long long)g * src.stride_h +
                         (seq.cu ? (long long)seq.cu[b] * src.stride_n : (long long)b * src.stride_b);
  const uint4* from = reinterpret_cast<const uint4*>(reinterpret_cast<const uint16_t*>(src.ptr) + base) + piece;
  uint4* to = (which ? gd.v_out : gd.k_out) + (long long)unit * K * kLanesPerRow + piece;
  const long long row_pieces = src.stride_n / 8;
  const int step = kWarps * blocks;
  for (int r0 = block * kWarps + threadIdx.x / 32; r0 < K; r0 += kUnroll * step) {
    uint4 val[kUnroll];
#pragma unroll
    for (int j = 0; j < kUnroll; ++j) {
      const int r = r0 + j * step;
      int i = all ? r : (int)list[min(r, kCandCap - 1)];
      if (r >= kCandCap && r < taken && !all) i = out[r];
      val[j] = ta_ld_stream_if(from + i * row_pieces, r < taken && i >= 0 && i < n);
    }
#pragma unroll
    for (int j = 0; j < kUnroll; ++j) {
      const int r = r0 + j * step;
      if (r < K) ta_st_stream(to + (long long)r * kLanesPerRow, val[j]);
    }
  }
}

// grid.x = units. scored: unit = (l*B + b)*Hkv + g; fast: unit = b. HELP: the unit has a cluster of blocks, of which the first
// selects and all move rows.
template <bool CACHED, int CL, int ITEMS = kItems, bool GATHER = false, bool FEW = false, bool HELP = false>
__global__ void __launch_bounds__(kThreads, 1024 / kThreads) ta_select_kernel(ta_seq_desc seq, int n_layers, int Hkv, int K, int fast,
                                                             UnitSrc src, const uint8_t* forced,
                                                             const int32_t* r_main,
                                                             int32_t* __restrict__ idx, int32_t* __restrict__ count,
                                                             GatherDst gd, const int32_t* __restrict__ class_of) {
  __shared__ SelectShared<CL> sh;
  ta_wait_for_prior_grid();
  ta_launch_dependents();
  static_assert(!HELP || (GATHER && CL == 1), "helpers move rows and nothing else");
  const int blocks = HELP ? (int)cg::this_cluster().num_blocks() : CL;
  const int unit = blockIdx.x / blocks;
  const bool lead = blockIdx.x % blocks == 0;
  int b, l = 0, g = 0;
  if (fast) {
    b = unit;
  } else {
    g = unit % Hkv;
    b = (unit / Hkv) % seq.batch;
    l = unit / (Hkv * seq.batch);
  }
  if (class_of) {  // budgets per (layer, head): the forced set and the main-pool size of this pair's class
    const int cls = class_of[l * Hkv + g];
    forced += (long long)cls * seq.total;
    r_main += cls * seq.batch;
  }
  const int start = ta_seq_begin(seq, b);
  const int n = (seq.cu ? seq.cu[b + 1] : start + seq.n_uniform) - start;
  int32_t* out = idx + (long long)unit * K;
  const int tid = threadIdx.x;
  const long long unit_off = fast ? 0 : ((long long)l * Hkv + g) * seq.total;
  // the unit's rows, once the selecting block has listed them
  auto gather = [&](int taken, bool all) {
    if constexpr (GATHER && !HELP) gather_unit(gd, seq, unit, l, b, g, n, K, out, taken, all, sh.cand_keys);
    if constexpr (HELP) {
      cg::cluster_group cluster = cg::this_cluster();
      if (lead && tid == 0) {
        sh.totals[0][0][0] = taken;
        sh.totals[0][0][1] = all;
      }
      cluster.sync();
      const int* said = cluster.map_shared_rank(&sh.totals[0][0][0], 0);
      gather_unit(gd, seq, unit, l, b, g, n, K, out, said[0], said[1] != 0, cluster.map_shared_rank(&sh.cand_keys[0], 0),
                  (int)cluster.block_rank(), blocks);
      cluster.sync();  // the selecting block's list has been read
    }
  };
  if (HELP && !lead) {
    gather(0, false);
    return;
  }
  // a sequence that does not lie inside the token arrays (want -2 below) is not read
  const bool inside = n >= 0 && n <= seq.max_n && start >= 0 && (long long)start + n <= seq.total;
  int lo, hi;
  unit_slice<CL>(inside ? n : 0, lo, hi);
  const int nl = hi - lo;
  const float* ap = src.u ? src.u : src.A;
  KeyCache<ITEMS> kc;
  float uu[CACHED ? ITEMS : 1];  // the attention part: from L2 or HBM, requested first (before it is known to be needed)
  if constexpr (CACHED) {
    // loads as selects, never under a branch: nothing then keeps them from being in flight together
    const float* up = ap + unit_off + start + lo;
#pragma unroll
    for (int it = 0; it < ITEMS; ++it) {
      const int i = tid + it * kThreads;
      uu[it] = ap && i < nl ? up[i] : 0.0f;
    }
  }
  const int want = r_main[b];
  // The per-token values, mostly from L2, in groups (registers: a group's loads are in flight together, no more); the first
  // group's before `want` is known.
  constexpr int kGroup = ITEMS < 8 ? ITEMS : ITEMS > 16 ? 4 : 8;
  const uint8_t* f = forced + start + lo;
  const float* sp = src.u_static + start + lo;
  const float* pp = !src.u && src.A && src.P ? src.P + unit_off + start + lo : nullptr;
  float us[CACHED ? kGroup : 1], ps[CACHED ? kGroup : 1];
  uint8_t ff[CACHED ? kGroup : 1];
  auto load_group = [&](int g0) {
#pragma unroll
    for (int q = 0; q < (CACHED ? kGroup : 0); ++q) {
      const int i = tid + (g0 + q) * kThreads;
      us[q] = i < nl ? sp[i] : 0.0f;
      ff[q] = i < nl ? f[i] : (uint8_t)1;
      ps[q] = pp && i < nl ? pp[i] : 0.0f;
    }
  };
  if constexpr (CACHED) load_group(0);
  if (want == -2) {  // sequence rejected by ta_forced_kernel
    if (lead) {
      for (int r = tid; r < K; r += kThreads) out[r] = -1;
      if (tid == 0) count[unit] = 0;
    }
    gather(0, true);
    return;
  }
  if (want == -1) {  // K >= n: keep everything
    if (lead) {
      for (int r = tid; r < K; r += kThreads) out[r] = r < n ? r : -1;
      if (tid == 0) count[unit] = n;
    }
    gather(n, true);
    return;
  }
  Exchange<CL> ex{src.waits};
  auto key_of = [&](int il, uint32_t& key) {
    key = sortable_key(unit_utility(src, unit_off, (long long)start + lo + il));
    return f[il] == 0;
  };
  if constexpr (CACHED) {
    if constexpr (CL > 1) {
      if (lead && tid == 0) count[unit] = 0;  // what a wait that runs out leaves
      ex.set_up(sh);
      cg::this_cluster().barrier_arrive();
    }
    kc.elig = 0;
#pragma unroll
    for (int g0 = 0; g0 < ITEMS; g0 += kGroup) {
      if (g0 > 0) load_group(g0);
#pragma unroll
      for (int q = 0; q < kGroup; ++q) {
        const int it = g0 + q;
        const bool in = tid + it * kThreads < nl;
        // the same roundings as unit_utility()
        float v = us[q];
        if (src.u) v = __fadd_rn(uu[it], v);
        else if (src.A) v = __fadd_rn(__fadd_rn(__fmul_rn(src.alpha, uu[it]), __fmul_rn(src.delta, ps[q])), v);
        kc.key[it] = in ? sortable_key(v) : 0u;
        kc.elig |= (in && ff[q] == 0) ? (1u << it) : 0u;
      }
      asm volatile("" ::: "memory");  // keeps the next group's loads behind this group's use
    }
  }
  SelectResult r;
  if constexpr (CACHED && CL > 1) cg::this_cluster().barrier_wait();
  if constexpr (CACHED) r = cached_radix_select<CL, FEW>(hi - lo, n, want, kc, sh, ex);
  else r = block_radix_select<CACHED, CL>(hi - lo, want, key_of, kc, sh);
  auto classify = [&](int, bool elig, uint32_t key, bool& def, bool& tie) {
    def = !elig || (!r.none && (r.all || key > r.thresh));
    tie = !def && !r.none && !r.all && key == r.thresh;
  };
  auto emit = [&](int il, int rank) {
    if (rank < K) out[rank] = lo + il;
    if (GATHER && rank < min(K, kCandCap)) sh.cand_keys[rank] = (uint32_t)il;  // (the selection is done with the list)
  };
  int taken;
  if constexpr (CACHED)  // forced tokens (not eligible, inside the unit) are taken whatever their key
    taken = cached_ordered_emit<CL>(hi - lo, r, kc, exist_mask(hi - lo) & ~kc.elig, emit, sh, ex);
  else
    taken = cluster_ordered_emit<CACHED, CL>(hi - lo, r.ties, key_of, kc, classify, emit, sh);
  if (!lead) return;
  for (int q = taken + tid; q < K; q += kThreads) out[q] = -1;
  if (tid == 0) count[unit] = CL > 1 ? min(taken, K) : taken;
  gather(min(taken, K), false);
}

}  // namespace TA_SEL_NS
