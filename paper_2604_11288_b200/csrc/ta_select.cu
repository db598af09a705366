// Step 3 of the retention path: budget-K selection with the partition of Section 3.3 (Algorithm 1 step 8).
//
// The retained set is reported in ascending position order, so no sort of the winners is needed: a radix select
// over the order-preserving integer image of the values (8-bit digits, starting below the bits that all keys of the
// unit share) finds the threshold key and how many tokens that tie with it still fit, and one ordered
// stream-compaction pass writes the indices. Order is total and deterministic: larger value first, lower
// position first among equal values.
//
//   ta_forced_kernel   one block per sequence: mandatory sinks/recents and the protected pool (largest vouchers
//                      among sponsored tokens). Independent of layer and head, so it runs once per sequence; on
//                      request it also writes the sequence's static utilities (Eq. 3).
//   ta_select_kernel   one block per unit (layer, sequence, KV head) in scored mode, per sequence in fast mode:
//                      main pool by utility among the tokens not forced, then the ordered write of
//                      forced + chosen positions.
//   ta_broadcast_idx_kernel  fast mode: the per-sequence result is the same for all layers and heads.
//   ta_headsum_kernel, ta_broadcast_heads_kernel  selection shared by the KV heads of a layer: the utilities'
//                      attention parts are summed over the heads, one selection runs per (layer, sequence), and its
//                      result is copied to every head.
#include <cooperative_groups.h>

#include <atomic>

#include "ta_internal.cuh"
#include "ta_sm100.cuh"

namespace cg = cooperative_groups;

#define TA_SEL_THREADS 128
#define TA_SEL_NS sel128
#include "ta_select_core.cuh"
#undef TA_SEL_THREADS
#undef TA_SEL_NS
#define TA_SEL_THREADS 256
#define TA_SEL_NS sel256
#include "ta_select_core.cuh"
#undef TA_SEL_THREADS
#undef TA_SEL_NS
#define TA_SEL_THREADS 512
#define TA_SEL_NS sel512
#include "ta_select_core.cuh"
#undef TA_SEL_THREADS
#undef TA_SEL_NS
#define TA_SEL_THREADS 1024
#define TA_SEL_NS sel1024
#include "ta_select_core.cuh"
#undef TA_SEL_THREADS
#undef TA_SEL_NS

namespace {

using namespace sel512;  // the launchers below name the 512-thread kernels unless they say otherwise

__global__ void ta_broadcast_idx_kernel(int B, int Hkv, int K, int n_layers, const int32_t* __restrict__ idx_seq,
                                        const int32_t* __restrict__ count_seq, int32_t* __restrict__ idx,
                                        int32_t* __restrict__ count) {
  const long long total = (long long)n_layers * B * Hkv * K;
  for (long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x; t < total;
       t += (long long)gridDim.x * blockDim.x) {
    const int r = (int)(t % K);
    const long long unit = t / K;
    const int b = (int)((unit / Hkv) % B);
    idx[t] = idx_seq[(long long)b * K + r];
    if (r == 0) count[unit] = count_seq[b];
  }
}

// u_all[l][tok] = sum over KV heads g (ascending, fp32) of u[l][g][tok]
__global__ void ta_headsum_kernel(int n_layers, int Hkv, long long total, const float* __restrict__ u,
                                  float* __restrict__ u_all) {
  const long long n = (long long)n_layers * total;
  for (long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x; t < n; t += (long long)gridDim.x * blockDim.x) {
    const long long l = t / total, tok = t - l * total;
    const float* src = u + l * Hkv * total + tok;
    float acc = src[0];
    for (int g = 1; g < Hkv; ++g) acc = __fadd_rn(acc, src[(long long)g * total]);
    u_all[t] = acc;
  }
}

// idx[l][b][g][:] = idx_lb[l][b][:], count[l][b][g] = count_lb[l][b]
__global__ void ta_broadcast_heads_kernel(long long units_lb, int Hkv, int K, const int32_t* __restrict__ idx_lb,
                                          const int32_t* __restrict__ count_lb, int32_t* __restrict__ idx,
                                          int32_t* __restrict__ count) {
  const long long total = units_lb * Hkv * K;
  for (long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x; t < total;
       t += (long long)gridDim.x * blockDim.x) {
    const int r = (int)(t % K);
    const long long unit = t / K, lb = unit / Hkv;
    idx[t] = idx_lb[lb * K + r];
    if (r == 0) count[unit] = count_lb[lb];
  }
}

// Two CTAs search 2 x 512 keys together (stop 2: 2 x 2048), and the second stops after what its first `stop` exchanges need: 0
// nothing, 1 and 2 the range of its keys (then candidates or a histogram are missing), 3 also its candidates (then its totals are);
// 4: it stays to the end. *outcome: the keys taken, unless a wait ran out.
__global__ void __launch_bounds__(kThreads) ta_exchange_selftest_kernel(ta_waits waits, int stop, int32_t* outcome) {
  __shared__ SelectShared<2> sh;
  constexpr int kPer = 4, kSent = 8;
  const int tid = threadIdx.x, rank = (int)cg::this_cluster().block_rank();
  const int n = stop == 2 ? kPer * kThreads : kThreads;
  const uint32_t lo = 1u << 20;  // the keys: lo .. lo + 2n - 1, every other one of each CTA
  KeyCache<kPer> kc;
#pragma unroll
  for (int it = 0; it < kPer; ++it) kc.key[it] = lo + 2u * (uint32_t)(tid + it * kThreads) + (uint32_t)rank;
  kc.elig = stop == 2 ? (1u << kPer) - 1u : 1u;
  Exchange<2> ex{waits};
  ex.set_up(sh);
  cg::this_cluster().sync();
  if (rank == 0 || stop >= 4) {
    const SelectResult r = cached_radix_select<2>(n, 2 * n, 100, kc, sh, ex);
    const int taken = cached_ordered_emit<2>(n, r, kc, 0u, [](int, int) {}, sh, ex);
    if (rank == 0 && tid == 0) *outcome = taken;
  } else {
    if (stop >= 1 && tid < 2)
      ex.send4(sh, sh.cl_range[1], tid, make_uint4(lo + 1u, lo + 2u * (uint32_t)n - 1u, stop == 2 ? (uint32_t)n : (uint32_t)kSent, 0u));
    ex.k = 1;
    if (stop >= 3 && tid < 2) ex.send1(sh, &sh.took_part[1], tid, 0u);
    if (stop >= 3 && tid < kSent) ex.send1(sh, &sh.cand_keys[n + tid], 0, lo + 2u * (uint32_t)(n - tid) - 1u);
    ex.stay();  // the first one sends to it
  }
}

}  // namespace

cudaError_t ta_launch_exchange_selftest(ta_dev_status* status, unsigned long long limit_ns, int stop, int32_t* outcome,
                                        cudaStream_t stream) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(2, 1, 1);
  cfg.blockDim = dim3(kThreads, 1, 1);
  cfg.stream = stream;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = 2;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, ta_exchange_selftest_kernel, ta_waits{status, limit_ns}, stop, outcome);
}

// Scratch layout used by the launcher (the caller carves it): forced [total] bytes, r_main [B] ints; fast mode
// additionally idx_seq [B][K] and count_seq [B] (passed through a.idx / a.count by the caller when it wants the
// per-sequence result only).
// Sequences that fit kItems keys per thread run one CTA per unit with the keys in registers; longer ones are split
// over a cluster of kSelectCluster CTAs (keys in registers up to kSelectCluster * 32 * 1024 elements; beyond 65536
// elements the cluster's blocks have 1024 threads).
// Splitting pays only while the clusters of all units fit on the device about at once; with many units one CTA per
// unit (keys re-read in batches when they do not fit in registers) keeps every SM busy without cluster barriers.
bool split_units(int units, int max_n, int sms) {
  if (max_n <= kItems * kThreads) return false;
  return units * kSelectCluster <= 2 * sms;
}

// SM count of the device the launch goes to: the caller's (a context knows its device), else the current device's
int sm_count_of(const ta_select_args& a) {
  if (a.sm_count > 0) return a.sm_count;
  int dev = 0, sms = 0;
  if (cudaGetDevice(&dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || sms < 1)
    sms = 148;
  return sms;
}

// stream_pdl: the stream, and whether the kernel is launched as a programmatic dependent of the kernel before it
struct StreamPdl {
  cudaStream_t stream;
  bool pdl;
};
template <class Kern, class... Args>
cudaError_t launch_threads(int threads, Kern kern, int units, int cl, StreamPdl sp, Args... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(units * cl), 1, 1);
  cfg.blockDim = dim3((unsigned)threads, 1, 1);
  cfg.dynamicSmemBytes = 0;
  cfg.stream = sp.stream;
  cudaLaunchAttribute attr[2];
  int n = 0;
  if (cl > 1) {  // no cluster attribute when no cluster is needed
    attr[n].id = cudaLaunchAttributeClusterDimension;
    attr[n].val.clusterDim.x = (unsigned)cl;
    attr[n].val.clusterDim.y = 1;
    attr[n].val.clusterDim.z = 1;
    ++n;
  }
  if (sp.pdl) ta_pdl_attribute(&attr[n++]);
  cfg.attrs = attr;
  cfg.numAttrs = n;
  return cudaLaunchKernelEx(&cfg, kern, args...);
}
// How many clusters of cl such blocks the current device holds at once; known: what earlier calls found, 1 + clusters per device.
constexpr int kMaxDevices = 64;
template <class Kern>
int clusters_held(Kern kern, int threads, int cl, std::atomic<int>* known) {
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return 0;
  std::atomic<int>& k = known[dev % kMaxDevices];
  const int have = k.load(std::memory_order_relaxed);
  if (have > 0) return have - 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)cl, 1, 1);
  cfg.blockDim = dim3((unsigned)threads, 1, 1);
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = (unsigned)cl;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  int n = 0;
  if (cudaOccupancyMaxActiveClusters(&n, kern, &cfg) != cudaSuccess) {
    cudaGetLastError();  // a size that the device does not have
    n = 0;
  }
  k.store(1 + n, std::memory_order_relaxed);
  return n;
}
template <class Kern, class... Args>
cudaError_t launch_clustered(Kern kern, int units, int cl, StreamPdl sp, Args... args) {
  return launch_threads(kThreads, kern, units, cl, sp, args...);
}

cudaError_t ta_launch_forced(const ta_select_args& a, ta_dev_status* status, cudaStream_t stream_) {
  if (a.seq.batch == 0 || a.n_layers == 0) return cudaSuccess;
  const StreamPdl stream = {stream_, a.pdl_forced != 0};
  const int B = a.seq.batch * (a.n_classes > 0 ? a.n_classes : 1);  // blocks: (class, sequence)
  const int32_t* ck = a.n_classes > 0 ? a.class_K : nullptr;
  const int sms = sm_count_of(a);
  const ta_waits waits = {status, ta_wait_limit(a.wait_limit_ns)};
  ta_static_out so = {};
  so.out = a.static_out;
  so.ids = a.static_ids;
  so.flags = a.flags;
  so.hist = a.static_hist;
  so.vocab = a.static_vocab;
  so.beta = a.beta;
  so.gamma = a.gamma;
  so.lambda = a.lambda;
  if (a.seq.max_n <= kItems * kThreads)
    return launch_clustered(ta_forced_kernel<true, 1>, B, 1, stream, a.seq, a.K, a.n_sink, a.n_recent, a.k_protected,
                            a.voucher, a.forced, a.r_main, waits, ck, so);
  if (!split_units(B, a.seq.max_n, sms) && a.seq.max_n <= kItemsLong * kThreads)
    return launch_clustered(ta_forced_kernel<true, 1, kItemsLong>, B, 1, stream, a.seq, a.K, a.n_sink, a.n_recent,
                            a.k_protected, a.voucher, a.forced, a.r_main, waits, ck, so);
  if (!split_units(B, a.seq.max_n, sms))
    return launch_clustered(ta_forced_kernel<false, 1>, B, 1, stream, a.seq, a.K, a.n_sink, a.n_recent, a.k_protected,
                            a.voucher, a.forced, a.r_main, waits, ck, so);
  if (a.seq.max_n <= kSelectCluster * kItems * kThreads)
    return launch_clustered(ta_forced_kernel<true, kSelectCluster>, B, kSelectCluster, stream, a.seq, a.K, a.n_sink,
                            a.n_recent, a.k_protected, a.voucher, a.forced, a.r_main, waits, ck, so);
  // few very long sequences: the chain of per-thread sweeps and cluster barriers sets the time, so blocks of 1024
  // threads (half the keys per thread) roughly halve it
  if (a.seq.max_n <= kSelectCluster * sel1024::kItems * sel1024::kThreads)
    return launch_threads(sel1024::kThreads, sel1024::ta_forced_kernel<true, kSelectCluster>, B, kSelectCluster,
                          stream, a.seq, a.K, a.n_sink, a.n_recent, a.k_protected, a.voucher, a.forced, a.r_main,
                          waits, ck, so);
  if (a.seq.max_n <= kSelectCluster * sel1024::kItemsLong * sel1024::kThreads)
    return launch_threads(sel1024::kThreads, sel1024::ta_forced_kernel<true, kSelectCluster, sel1024::kItemsLong>, B,
                          kSelectCluster, stream, a.seq, a.K, a.n_sink, a.n_recent, a.k_protected, a.voucher,
                          a.forced, a.r_main, waits, ck, so);
  return launch_clustered(ta_forced_kernel<false, kSelectCluster>, B, kSelectCluster, stream, a.seq, a.K, a.n_sink,
                          a.n_recent, a.k_protected, a.voucher, a.forced, a.r_main, waits, ck, so);
}

// Few short units (at most one block per SM): a launch is then all latency, and blocks of 1024 threads with a quarter of the
// keys per thread take less time than 512 (8 units of 4096 keys with the gather of 16 rows: 9.5 -> 7.1 us).
bool few_short_units(const ta_select_args& a) {
  return !a.fast && a.seq.max_n <= 8 * sel1024::kThreads && a.n_layers * a.seq.batch * a.Hkv <= sm_count_of(a);
}

// Whether the selecting blocks move the rows: keys in registers, one block per unit (see gather_unit).
bool ta_select_gathers(const ta_select_args& a) {
  const int units = a.n_layers * a.seq.batch * a.Hkv;
  return a.gather_k_out && !a.fast && a.seq.max_n <= sel1024::kItemsLong * sel1024::kThreads &&
         !split_units(units, a.seq.max_n, sm_count_of(a));
}

// the same arguments in the types of every block size
template <class Src>
Src unit_src(const ta_select_args& a) {
  Src s;
  s.u = a.fast ? nullptr : a.u;
  s.A = a.fast ? nullptr : a.A;
  s.P = a.fast ? nullptr : a.P;
  s.u_static = a.u_static;
  s.alpha = a.alpha;
  s.delta = a.delta;
  s.waits = {a.status, ta_wait_limit(a.wait_limit_ns)};
  return s;
}
template <class Dst>
Dst gather_dst(const ta_select_args& a, bool gathers) {
  Dst d = {};
  if (gathers) {
    d.k = a.gather_k;
    d.v = a.gather_v;
    d.k_out = reinterpret_cast<uint4*>(a.gather_k_out);
    d.v_out = reinterpret_cast<uint4*>(a.gather_v_out);
  }
  return d;
}

// Threads of a selecting block that also gathers, where small ones pay (0: they do not). A block is a chain of latencies around
// a few barriers, so that more and smaller blocks per SM (eight of 128 threads, four of 256, two of 512) fill one another's gaps
// as long as the gather is small and there are units enough for them; a large gather wants a block's loads together. The budgets
// are those that half a block's threads bound (see cached_radix_select), and a little more where units are short. Time of
// ta_compress_scores in us with 512 / 256 / 128 threads, uniform lengths:
//   2048 units, 4000 tokens: K 16 52 / 36 / 31, K 64 77 / 57 / 53, K 128 88 / 77 / 83, K 192 107 / 105 / 106, K 256 120 / 125 / 128
//   1024 units, 2000 tokens: K 16 27 / 19 / 14, K 64 40 / 29 / 24, K 128 45 / 39 / 39, K 256 61 / 63 / 65
//   400 units, 2000 tokens: K 16 15.8 / 11.9 / 11.0, K 64 21.8 / 16.6 / 16.2, K 128 24.7 / 20.9 / 23.0, K 256 32.7 / 31.7 / 32.6
//   256 units, 4000 tokens: K 16 13.9 / 12.9 / 14.8, K 64 17.5 / 16.9 / 20.0, K 128 19.1 / 19.4 / 27.0
//   2048 units, 8000 tokens: K 16 66 / 49, K 64 101 / 81, K 128 112 / 99, K 192 131 / 135; 256 units: K 64 23.1 / 23.5
int small_threads(const ta_select_args& a, int units, int sms) {
  const int n = a.seq.max_n;
  const bool is_short = n <= 16 * sel256::kThreads;  // also what 128 threads hold
  static_assert(16 * sel256::kThreads == sel128::kItemsLong * sel128::kThreads, "one limit for both");
  if (is_short && units >= 5 * sms && a.K <= sel128::kThreads / 2) return sel128::kThreads;
  if (n <= sel256::kItemsLong * sel256::kThreads &&
      ((units > 2 * sms && a.K <= (is_short ? 192 : sel256::kThreads / 2)) || (is_short && units > sms && a.K <= 64)))
    return sel256::kThreads;
  return 0;
}

cudaError_t ta_launch_select_units(const ta_select_args& a, cudaStream_t stream_) {
  if (a.seq.batch == 0 || a.n_layers == 0) return cudaSuccess;
  const StreamPdl stream = {stream_, a.pdl_units != 0};
  const UnitSrc src = unit_src<UnitSrc>(a);
  const int units = a.fast ? a.seq.batch : a.n_layers * a.seq.batch * a.Hkv;
  const int32_t* co = a.n_classes > 0 ? a.class_of : nullptr;
  const int sms = sm_count_of(a);
  const bool gathers = ta_select_gathers(a);
  const GatherDst gd = gather_dst<GatherDst>(a, gathers);
  const sel1024::UnitSrc src2 = unit_src<sel1024::UnitSrc>(a);
  const sel1024::GatherDst gd2 = gather_dst<sel1024::GatherDst>(a, gathers);
  // The instances that look for few tokens, as long as the budget lets them (see cached_radix_select; us without and with them):
  // 1024 units of 16000 tokens K 128 107 / 90, 250 123 / 109; 2048 units of 4000 tokens K 64 62 / 53; 256 units of 4000 tokens K 256
  // 26.4 / 25.3; 8 units of up to 7000 tokens K 128, 32 calls with their scores 773 / 756. There is none with 4 keys per thread of
  // 1024: 8 units K 16 and 64 take as long with one, K 128, 256, 512 of 4000 tokens 16.7, 18.1, 21.5 without and 15.7, 17.4, 20.7
  // with it, K 256 and 512 of 1000 tokens 14.7 and 17.6 without, 15.0 and 18.0 with it.
  const bool few = gathers && a.K <= kThreads / 2, few1024 = gathers && a.K <= sel1024::kThreads / 2;
  if (few_short_units(a)) {
    // (the instance for few wanted tokens at the one budget that both rules take: 8 units of 5000, 6000, 8000 tokens K 512 22.0, 22.9,
    // 24.1 with it, 22.5, 23.5, 25.2 without)
    const int which = a.seq.max_n <= 4 * sel1024::kThreads ? 0 : few1024 ? 1 : 2;
    auto helped = which == 0   ? sel1024::ta_select_kernel<true, 1, 4, true, false, true>
                  : which == 1 ? sel1024::ta_select_kernel<true, 1, 8, true, true, true>
                               : sel1024::ta_select_kernel<true, 1, 8, true, false, true>;
    static std::atomic<int> held[3][kMaxDevices];
    if (gathers && a.K >= kHelpedBudget && units <= sms / kHelpBlocks &&
        ta_select_helped(a.K, units, clusters_held(helped, sel1024::kThreads, kHelpBlocks, held[which])))
      return launch_threads(sel1024::kThreads, helped, units, kHelpBlocks, stream, a.seq, a.n_layers, a.Hkv, a.K, a.fast, src2,
                            a.forced, a.r_main, a.idx, a.count, gd2, co);
    auto kern = a.seq.max_n <= 4 * sel1024::kThreads
                    ? (gathers ? sel1024::ta_select_kernel<true, 1, 4, true> : sel1024::ta_select_kernel<true, 1, 4, false>)
                    : (few1024   ? sel1024::ta_select_kernel<true, 1, 8, true, true>
                       : gathers ? sel1024::ta_select_kernel<true, 1, 8, true>
                                 : sel1024::ta_select_kernel<true, 1, 8, false>);
    return launch_threads(sel1024::kThreads, kern, units, 1, stream, a.seq, a.n_layers, a.Hkv, a.K, a.fast, src2, a.forced,
                          a.r_main, a.idx, a.count, gd2, co);
  }
  const int small = gathers ? small_threads(a, units, sms) : 0;
  if (small == sel128::kThreads) {
    auto kern = a.seq.max_n <= 16 * sel128::kThreads ? sel128::ta_select_kernel<true, 1, 16, true, true>
                                                     : sel128::ta_select_kernel<true, 1, sel128::kItemsLong, true, true>;
    return launch_threads(small, kern, units, 1, stream, a.seq, a.n_layers, a.Hkv, a.K, a.fast, unit_src<sel128::UnitSrc>(a),
                          a.forced, a.r_main, a.idx, a.count, gather_dst<sel128::GatherDst>(a, true), co);
  }
  if (small == sel256::kThreads) {
    auto kern = a.seq.max_n <= 16 * sel256::kThreads ? sel256::ta_select_kernel<true, 1, 16, true, true>
                                                     : sel256::ta_select_kernel<true, 1, sel256::kItemsLong, true, true>;
    return launch_threads(small, kern, units, 1, stream, a.seq, a.n_layers, a.Hkv, a.K, a.fast, unit_src<sel256::UnitSrc>(a),
                          a.forced, a.r_main, a.idx, a.count, gather_dst<sel256::GatherDst>(a, true), co);
  }
  if (!split_units(units, a.seq.max_n, sms) && a.seq.max_n <= kItemsLong * kThreads) {
    // (the smallest instance that holds the unit: every phase walks over all of a thread's slots)
    auto kern = a.seq.max_n <= 8 * kThreads
                    ? (few       ? ta_select_kernel<true, 1, 8, true, true>
                       : gathers ? ta_select_kernel<true, 1, 8, true>
                                 : ta_select_kernel<true, 1, 8, false>)
                : a.seq.max_n <= kItems * kThreads
                    ? (few       ? ta_select_kernel<true, 1, kItems, true, true>
                       : gathers ? ta_select_kernel<true, 1, kItems, true>
                                 : ta_select_kernel<true, 1, kItems, false>)
                    : (few       ? ta_select_kernel<true, 1, kItemsLong, true, true>
                       : gathers ? ta_select_kernel<true, 1, kItemsLong, true>
                                 : ta_select_kernel<true, 1, kItemsLong, false>);
    return launch_clustered(kern, units, 1, stream, a.seq, a.n_layers, a.Hkv, a.K, a.fast, src, a.forced, a.r_main, a.idx,
                            a.count, gd, co);
  }
  if (!split_units(units, a.seq.max_n, sms) && a.seq.max_n <= sel1024::kItemsLong * sel1024::kThreads) {
    // many long units: blocks of 1024 threads hold a unit of up to 32768 keys in registers (read once instead of
    // once per radix pass and once more for the ordered write)
    auto kern = few1024   ? sel1024::ta_select_kernel<true, 1, sel1024::kItemsLong, true, true>
                : gathers ? sel1024::ta_select_kernel<true, 1, sel1024::kItemsLong, true>
                          : sel1024::ta_select_kernel<true, 1, sel1024::kItemsLong, false>;
    return launch_threads(sel1024::kThreads, kern, units, 1, stream, a.seq, a.n_layers, a.Hkv, a.K, a.fast, src2, a.forced,
                          a.r_main, a.idx, a.count, gd2, co);
  }
  if (!split_units(units, a.seq.max_n, sms))
    return launch_clustered(ta_select_kernel<false, 1>, units, 1, stream, a.seq, a.n_layers, a.Hkv, a.K, a.fast, src,
                            a.forced, a.r_main, a.idx, a.count, gd, co);
  if (a.seq.max_n <= kSelectCluster * kItems * kThreads)
    return launch_clustered(ta_select_kernel<true, kSelectCluster>, units, kSelectCluster, stream, a.seq, a.n_layers,
                            a.Hkv, a.K, a.fast, src, a.forced, a.r_main, a.idx, a.count, gd, co);
  if (a.seq.max_n <= kSelectCluster * sel1024::kItems * sel1024::kThreads)  // as in ta_launch_forced
    return launch_threads(sel1024::kThreads, sel1024::ta_select_kernel<true, kSelectCluster>, units, kSelectCluster,
                          stream, a.seq, a.n_layers, a.Hkv, a.K, a.fast, src2, a.forced, a.r_main, a.idx, a.count, gd2,
                          co);
  if (a.seq.max_n <= kSelectCluster * sel1024::kItemsLong * sel1024::kThreads)
    return launch_threads(sel1024::kThreads, sel1024::ta_select_kernel<true, kSelectCluster, sel1024::kItemsLong>,
                          units, kSelectCluster, stream, a.seq, a.n_layers, a.Hkv, a.K, a.fast, src2, a.forced,
                          a.r_main, a.idx, a.count, gd2, co);
  return launch_clustered(ta_select_kernel<false, kSelectCluster>, units, kSelectCluster, stream, a.seq, a.n_layers,
                          a.Hkv, a.K, a.fast, src, a.forced, a.r_main, a.idx, a.count, gd, co);
}

cudaError_t ta_launch_select(const ta_select_args& a, ta_dev_status* status, cudaStream_t stream) {
  cudaError_t e = ta_launch_forced(a, status, stream);
  if (e != cudaSuccess) return e;
  ta_select_args with_status = a;
  with_status.status = status;
  return ta_launch_select_units(with_status, stream);
}

cudaError_t ta_launch_broadcast_idx(int B, int Hkv, int K, int n_layers, const int32_t* idx_seq,
                                    const int32_t* count_seq, int32_t* idx, int32_t* count, cudaStream_t stream) {
  const long long total = (long long)n_layers * B * Hkv * K;
  if (total == 0) return cudaSuccess;
  const int blocks = (int)((total + 255) / 256 < 4096 ? (total + 255) / 256 : 4096);
  ta_broadcast_idx_kernel<<<blocks, 256, 0, stream>>>(B, Hkv, K, n_layers, idx_seq, count_seq, idx, count);
  return cudaGetLastError();
}

cudaError_t ta_launch_headsum(int n_layers, int Hkv, long long total, const float* u, float* u_all,
                              cudaStream_t stream) {
  const long long n = (long long)n_layers * total;
  if (n == 0) return cudaSuccess;
  const int blocks = (int)((n + 255) / 256 < 8192 ? (n + 255) / 256 : 8192);
  ta_headsum_kernel<<<blocks, 256, 0, stream>>>(n_layers, Hkv, total, u, u_all);
  return cudaGetLastError();
}

cudaError_t ta_launch_broadcast_heads(int n_layers, int B, int Hkv, int K, const int32_t* idx_lb,
                                      const int32_t* count_lb, int32_t* idx, int32_t* count, cudaStream_t stream) {
  const long long total = (long long)n_layers * B * Hkv * K;
  if (total == 0) return cudaSuccess;
  const int blocks = (int)((total + 255) / 256 < 4096 ? (total + 255) / 256 : 4096);
  ta_broadcast_heads_kernel<<<blocks, 256, 0, stream>>>((long long)n_layers * B, Hkv, K, idx_lb, count_lb, idx, count);
  return cudaGetLastError();
}

// ---------------------------------------------------------------------------------------------------------------
// ta_select_topk_static: the selection step for callers that must not allocate device memory.
//
// The regular entry point takes its working memory (one byte per token, a few words per sequence) from a context
// whose creation calls cudaMalloc. This variant keeps that working memory in the array below, which is part of the
// library image: every GPU that loads the library reserves TA_STATIC_SCRATCH_BYTES for it until the process exits.
// The array name is only meaningful to device code; host code must ask the runtime for its device address
// (cudaGetSymbolAddress) once per device, with that device current, and hand that address to the kernels.
#include <mutex>

static __device__ __align__(256) unsigned char g_ta_static_scratch[TA_STATIC_SCRATCH_BYTES];

namespace {
std::mutex g_static_mutex;
unsigned char* g_static_ptr[kMaxDevices] = {};  // device address of g_ta_static_scratch, per device ordinal

size_t static_align(size_t x) { return (x + 255) / 256 * 256; }
}  // namespace

extern "C" ta_status ta_select_topk_static(const ta_policy* policy, const ta_batch* batch, int Hkv, int K,
                                           const uint8_t* flags, const float* voucher, const float* u_static,
                                           const float* A, const float* P, int32_t* idx, int32_t* count,
                                           void* stream_v) {
  if (!policy || !batch || !flags || !voucher || !u_static || !idx || !count) return TA_ERR_INVALID_ARG;
  if (batch->n_layers < 1 || batch->batch < 1 || batch->max_n < 0 || batch->total_tokens < 0 || Hkv < 1 || K < 1)
    return TA_ERR_INVALID_ARG;
  if (!batch->cu_seqlens && (batch->n_uniform < 0 || batch->n_uniform > batch->max_n ||
                             batch->total_tokens != (int64_t)batch->batch * batch->n_uniform))
    return TA_ERR_INVALID_ARG;
  if (policy->mode != TA_MODE_SCORED && policy->mode != TA_MODE_FAST) return TA_ERR_INVALID_ARG;
  if (policy->n_sink < 0 || policy->n_recent < 0) return TA_ERR_INVALID_ARG;
  if (K > TA_MAX_BUDGET || batch->max_n > TA_MAX_SEQ_LEN) return TA_ERR_UNSUPPORTED;
  const bool fast = policy->mode == TA_MODE_FAST;
  if (!fast && !A) return TA_ERR_INVALID_ARG;

  // carve the fixed array: status block, forced flags, per-sequence counters, fast-mode per-sequence result
  const size_t B = (size_t)batch->batch, total = (size_t)batch->total_tokens;
  size_t off = 0;
  const size_t o_status = off; off += static_align(sizeof(ta_dev_status));
  const size_t o_forced = off; off += static_align(total);
  const size_t o_rmain = off;  off += static_align(B * 4);
  const size_t o_idxseq = off; off += static_align(fast ? B * (size_t)K * 4 : 0);
  const size_t o_cntseq = off; off += static_align(fast ? B * 4 : 0);
  if (off > (size_t)TA_STATIC_SCRATCH_BYTES) return TA_ERR_SCRATCH_TOO_SMALL;  // problem larger than the built-in limit

  int dev = -1;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) return TA_ERR_CUDA;
  unsigned char* base = nullptr;
  {
    std::lock_guard<std::mutex> lock(g_static_mutex);
    if (!g_static_ptr[dev]) {  // first call on this device: resolve the array's device address (no allocation)
      void* p = nullptr;
      if (cudaGetSymbolAddress(&p, g_ta_static_scratch) != cudaSuccess || !p) return TA_ERR_CUDA;
      g_static_ptr[dev] = static_cast<unsigned char*>(p);
    }
    base = g_static_ptr[dev];
  }
  cudaStream_t stream = (cudaStream_t)stream_v;
  // the array keeps whatever the previous call left: the status block must start at zero; the other pieces are
  // fully rewritten by the kernels before they are read
  if (cudaMemsetAsync(base + o_status, 0, sizeof(ta_dev_status), stream) != cudaSuccess) return TA_ERR_CUDA;

  ta_select_args a = {};
  a.seq.cu = batch->cu_seqlens;
  a.seq.n_uniform = batch->n_uniform;
  a.seq.batch = batch->batch;
  a.seq.max_n = batch->max_n;
  a.seq.total = batch->total_tokens;
  a.n_layers = batch->n_layers;
  a.Hkv = Hkv;
  a.K = K;
  a.n_sink = policy->n_sink;
  a.n_recent = policy->n_recent;
  a.k_protected = policy->k_protected;
  a.fast = fast;
  a.alpha = policy->alpha;
  a.delta = policy->delta;
  a.flags = flags;
  a.voucher = voucher;
  a.u_static = u_static;
  a.A = A;
  a.P = P;
  a.u = nullptr;
  a.forced = base + o_forced;
  a.r_main = reinterpret_cast<int32_t*>(base + o_rmain);
  int32_t* idx_seq = reinterpret_cast<int32_t*>(base + o_idxseq);
  int32_t* cnt_seq = reinterpret_cast<int32_t*>(base + o_cntseq);
  a.idx = fast ? idx_seq : idx;
  a.count = fast ? cnt_seq : count;
  cudaError_t e = ta_launch_select(a, reinterpret_cast<ta_dev_status*>(base + o_status), stream);
  if (e == cudaSuccess && fast)
    e = ta_launch_broadcast_idx(batch->batch, Hkv, K, batch->n_layers, idx_seq, cnt_seq, idx, count, stream);
  return e == cudaSuccess ? TA_OK : TA_ERR_CUDA;
}
