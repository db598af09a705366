// Step 2 of the retention path: the attention terms of Eq. 1 (A_i, the pension P_i) over the observation window,
// optionally fused with their weights alpha and delta. sm_100a only: TMA tile loads, tcgen05 tensor-core MMAs with the
// accumulators in tensor memory, and a thread-block cluster per unit for the softmax statistics.
//
// For unit (l, b, g) the score matrix is S = Q_obs[heads of g] * K^T, M = G*W rows (<= 256) by n keys. Each row is
// softmax-normalised over the keys it may see and the result is summed over rows per key. The normaliser of a row
// needs every key before any column sum can be finished, so the keys are swept twice:
//   pass 1  S = Q * Ktile^T   (TMEM lane = query row)  -> reference and sum of exponentials per row
//   pass 2  S^T = Ktile * Q^T (TMEM lane = key)        -> sum over rows of exp2(s*c - beta_row) per key
// Both passes use the same shared-memory operand tiles (both K-major, 128-byte swizzle); only the roles in the
// instruction descriptor swap, which puts the reduction axis of each pass along a thread's own registers.
// A unit is handled by a cluster of 1, 2, 4 or 8 CTAs (chosen per launch: one CTA when there are many units, more when there
// are few, 9 to 16 for a handful of units, where all of them fit at once: a cluster stays inside a group of
// SMs, 148 SMs hold 8 clusters of 9 or 10 CTAs and 7 of 11 to 16); each CTA owns a contiguous range of 128-key tiles. Between
// the passes every CTA stores its per-row (reference, sum) pairs into the shared memory of all its peers with stores that count
// on the receiver's mbarrier when they land (reading the peers' pairs over the cluster took 1.9 us of a 15 us kernel, plain
// remote stores with a fence and a signal behind them 0.4 us more than these).
// Pass 2 walks the CTA's tiles backwards so that the tiles read last are re-read first from L2.
// When the caller supplies the rows' log-sum-exp (lse_obs), pass 1 is skipped; the keys of a unit are then independent, and
// a uniform batch is cut into equal shares of tiles, one per CTA (32 layers x 8111 tokens: 256 units on 148 CTAs are 2 rounds
// of whole units but 1.73 rounds of shares; 118 -> 105 us with the rest).
//
// The grid is persistent: as many clusters as the device can hold at once, each walking over its units. Roles, all of them
// whole warps that meet only at mbarriers (no barrier among the softmax warps: each runs on as soon as its own data is
// there):
//   TMA producer        walks the units, publishes each one's description in a small ring, streams query and key tiles
//   MMA issuer          TMEM owner; one elected lane issues, the warp around it is uniform
//   2 statistics warps  one pass only: form the row constants from the log-sum-exps that the caller supplies, a unit ahead
//   16 softmax warps    four groups of four. A "job" is one block of up to 128 score rows of one key tile in one pass; jobs
//                       are dealt round-robin to the four groups and to the four accumulator stages. Two groups at work
//                       keep the special-function unit as busy as it can be (1105 cycles a job against 1095 with three);
//                       the others hide a group's way from one job to the next: its stage's products (some 800 cycles)
//                       and the signals around them. Three groups with a stage to spare took 2 to 5 % longer, two groups
//                       with 16, 32 or 64 columns per load 10 to 15 %. With 129..256 score rows (MB 2) a tile is two
//                       consecutive jobs, one per block of 128 rows; in pass 2 their partial sums meet in a
//                       shared-memory ring. Between the passes the group that ends the first one first merges the row
//                       statistics, exchanges them over the cluster and forms the row constants for pass 2.
// The producer's warpgroup gives registers back (setmaxnreg) at its start and the softmax warps take them.
//
// A call of few units is a chain of latencies (one layer of 4096 tokens: 8 units, 8 CTAs each, four tiles and 26 K cycles per
// CTA, of which the exponentials need 9 K). What the chain waits for is started as early as it can be: the producer requests its
// first tiles before the CTA's set-up is complete (first scores after 4.8 K cycles instead of 7 K), and nothing but the
// barriers that it needs itself precedes them. 21.9 -> 20.5 us a call, 32 calls of 8 shorter units 905 -> 865 us; 19.2 and 788 with
// four groups and the polynomial. Between the passes 4.4 K cycles remain (merge, exchange, merge, constants: code that is executed
// once and fetched for it). Letting the selection's blocks in early, looking at the barriers without suspending and unrolling
// the sends changed nothing or cost time.
//
// What bounds it. With up to 128 rows at full clock (32 layers x 4096 tokens): the softmax warps (two exponentials per score
// element, 16 per clock and SM on the special-function unit, an eighth of them on the FMA pipe) and shared memory, into which
// 32 KB a tile are copied and from which the products read 64 KB a job. A job takes 0.66 us of the steady state (0.70 with three
// groups and all exponentials on one unit); of those 0.70 the parts alone took 0.61 (softmax), 0.43 (products), 0.58 (copies),
// products and copies together 0.67. 256 units on 148 CTAs are two rounds where 1.73 would do. With 256 rows (16 x 32768
// tokens): the special-function unit. Back to back the board's power limit (1000 W) decides: 32 layers x 4096 tokens take 123 mJ
// a call (129 mJ before) at 1687 MHz instead of 1965, 64 ragged sequences of up to 16384 tokens 4.40 J (4.55) at 1342 MHz,
// 16 x 32768 tokens with 256 rows 12.8 J (13.1) at 1560 MHz. The products alone run into it at 1535 TFLOP/s, 5.7 of those
// 12.8 J; products of 256 columns, which read one operand half as often, would reach 1685, but one for both row blocks of a tile
// ties two accumulator stages together and the call takes as long. Equal shares of tiles over unit borders for both passes (a
// cut unit's statistics handed to the next CTA through global memory) save 3 % of a single call and cost 5 % back to back: the
// cut units' keys are read from HBM twice. The scale-and-shift and the running sums are taken two at a time (fma.rn.f32x2,
// add.rn.f32x2: the same roundings as the scalar forms, a third fewer issue slots).
//
// Every wait on an mbarrier is bounded by wall time; when one runs out the CTA records TA_ERR_TIMEOUT, its producer
// and MMA warps stop issuing work, the copies and MMAs in flight are drained, and the other warps leave their loops
// without storing. The only unbounded waits are hardware barriers that every thread reaches on every path.
#include <cuda.h>
#include <string.h>

#include <type_traits>

#include "ta_internal.cuh"
#include "ta_sm100.cuh"

namespace {

using namespace ta_sm100;

constexpr int kTileN = 128;                       // keys per tile
constexpr int kD = TA_HEAD_DIM;                   // 128
constexpr int kHalfBytes = kTileN * 128;          // one 64-column half of a 128-row operand tile: 16 KB
constexpr int kKTileBytes = 2 * kHalfBytes;       // 32 KB
constexpr int kMaxCluster = 16;                   // more than 8 CTAs is a non-portable cluster size; sm_100 allows 16
constexpr int kRankedSeqs = 256;                  // (an index is a byte) sequences of a ragged batch that the kernel itself sorts by length
constexpr int kGroups = 4;                        // softmax warpgroups
constexpr int kSoftWarps = kGroups * 4;
constexpr int kThreads = (kGroups + 1) * 128;     // 640
// Register split after set-up (setmaxnreg); the shares must fit in threads x registers at launch:
// 640 threads x 96 = 61440 = 16*32*104 + 4*32*64
constexpr int kRegsSoftmax = 104;
constexpr int kRegsOther = 64;
constexpr int kRegsNeeded = (kSoftWarps * kRegsSoftmax + 4 * kRegsOther) * 32;

// Of every 16 exponentials, two (they are taken in pairs) run on the FMA pipe in tiles that are not masked, which relieves the
// special-function unit. Back to back the kernel runs into the board's 1000 W limit, and a polynomial costs more energy than
// ex2, so that a larger share does not pay.
// 129 to 256 score rows: a cubic. 8 layers of 16 x 32768 tokens, share 0: 6.22 ms, 2: 6.02 ms, more: the same.
// Up to 128 rows: a polynomial of degree 5, so that a score is as precise as ex2 alone gives it (2-norm error of 4096 tokens
// 8.7e-8 with either). 32 layers of 4096 tokens alone, share 0: 139 us, 2: 134 us, 4: 136 us, 6: 137 us; back to back 120.5,
// 119, 121, 125 us; 2 layers of 16384 tokens 73.0, 70.5, 70.1, 71.9 us.
#ifndef TA_SCORE_POLY_MB2
#define TA_SCORE_POLY_MB2 2
#endif

// how pass 2 turns the exponentials of a key into outputs
constexpr int kOutA = 0;      // A only
constexpr int kOutAP = 3;     // A and P (per-row pension weights), or their weighted sum
constexpr int kOutFused = 4;  // alpha*A + delta*P with the positive row weights folded into the exponent

// Of the eight pairs of a 16-element group, this many run on the FMA pipe; pair q2 (elements 2*q2, 2*q2 + 1) does when
// poly_pair is true (spread evenly). With A and P apart and up to 128 rows none: the registers hold no more.
template <int MB, int PM>
__host__ __device__ constexpr int poly_pairs() {
  return MB == 2 ? TA_SCORE_POLY_MB2 / 2 : PM == kOutAP ? 0 : 1;
}
template <int MB, int PM>
__host__ __device__ constexpr bool poly_pair(int q2) {
  return ((q2 * poly_pairs<MB, PM>()) / 8) != (((q2 + 1) * poly_pairs<MB, PM>()) / 8);
}

struct ScoreParams {
  ta_seq_desc seq;
  int n_layers, Hq, Hkv, G, W;
  int rows;           // G*W
  int cluster;        // CTAs per unit
  int units;          // L * B * Hkv
  // One pass (lse_obs given): the keys of a unit are independent of one another and a unit may be cut anywhere.
  int flat;           // uniform batches: CTA i takes the i-th equal share of all tiles, over unit borders
  int two_pass;       // 0 when lse_obs is given
  int causal;
  float c;            // softmax scale * log2(e)
  float alpha, delta;
  const float* lse_obs;
  const int32_t* order;  // nullable: the clusters walk units order[0], order[1], .. (longest sequences first)
  int by_length;         // the same walk from lengths ranked in the kernel (batches of up to kRankedSeqs sequences)
  int late_wait;         // wait for the kernel before this one at the end instead of at the start (ta_score_args::pdl 2)
  float* A;
  float* P;
  float* u;
  ta_dev_status* status;
  unsigned long long wait_limit_ns;
  float wrow[TA_MAX_WINDOW];  // pension weight of window row t (for W' = W; shorter sequences are handled in-kernel)
};

// ---------------------------------------------------------------------------------------------- shared memory
struct alignas(16) UnitInfo {
  int l, b, g, tok0;       // layer, sequence, KV head, packed index of the first token
  int n, t_begin, T, end;  // tokens, this CTA's first tile and its number of tiles; end: no unit, the walk is over
};
constexpr int kUnitRing = 4;  // unit descriptions in flight between the producer and the other warps
constexpr int kAcc = 4;       // accumulator stages of 128 tensor-memory columns (512 columns in all)
constexpr int kRing = 4;      // MB 2: partial column sums in flight between the groups

template <int MB>
struct alignas(1024) ScoreSmem {
  static constexpr int kQBufs = MB == 1 ? 2 : 1;  // query tiles in flight (next unit's tile loads early)
  static constexpr int kRowsPad = MB * 128;
  static constexpr int kStages = MB == 1 ? 4 : 3;  // ring of key tiles (256 rows: a fourth leaves no room for 16 peers)
  uint8_t q[kQBufs][MB * 2 * kHalfBytes];  // [buffer][half][MB*128 rows][128 B]
  uint8_t k[kStages][kKTileBytes];         // [stage][half][128 rows][128 B]
  // [softmax group][row of its block]: reference and sum of the group's keys (one unit's at a time: a softmax warp waits for
  // the row constants that are formed from them before it goes on to the next unit)
  float part_m[kGroups][128], part_z[kGroups][128];
  float2 peer[kMaxCluster][kRowsPad];           // row statistics (reference, sum) as the CTAs of the cluster sent them
  // [unit parity][row] pass-2 constant of the row; behind them the form that ex2 takes, for rows whose own is the polynomial's
  float tab[2][2 * kRowsPad];
  float wrow[kRowsPad];                    // pension weight per row
  float lv[kRowsPad];                      // log2 of the row's output weight (kOutFused), else 0
  int8_t row_t[kRowsPad];                  // window index t of the row, -1 for padding rows
  float psum[kRing][2][128];               // MB 2: [ring slot][A|P][key] partial sums of row block 0
  UnitInfo unit[kUnitRing];
  unsigned long long full[kStages], empty[kStages], acc_full[kAcc], acc_empty[kAcc];
  unsigned long long q_full[kQBufs], q_empty[kQBufs], ufull[kUnitRing], ufree[kUnitRing];
  unsigned long long stat_full, tab_full[2], tab_free[2], xchg_full, xchg_free, drain;
  unsigned long long pfull[kRing], pfree[kRing];
  uint32_t tmem_base;
  int abort_flag;
  uint8_t by_rank[kRankedSeqs];            // by_length: sequence of every rank, longest first
};

// ---------------------------------------------------------------------------------------------- exponentials
constexpr float kPolyRange = 252.0f;                // width of the clamped argument range [-126, 126]
constexpr float kPolyMagic = 12582912.0f - 126.0f;  // 1.5 * 2^23 - 126: adding it leaves the integer part in the low bits
// minimax cubic for 2^f on [0, 1) in relative error (7.5e-5)
constexpr float kC0 = 0.9999251961708069f, kC1 = 0.6958335638046265f, kC2 = 0.22606715559959412f,
                kC3 = 0.07802452147006989f;

__device__ __forceinline__ float fma_sat(float a, float b, float c) {
  float d;
  asm("fma.rn.sat.f32 %0, %1, %2, %3;" : "=f"(d) : "f"(a), "f"(b), "f"(c));
  return d;
}
// two values of exp2(x), x = s*c - beta clamped to [-126, 126], given c252 = c/252 and bias = (126 - beta)/252
__device__ __forceinline__ void exp2_poly2(float& e0, float& e1, float s0, float s1, float c252, float bias0, float bias1) {
  const float t0 = fma_sat(s0, c252, bias0), t1 = fma_sat(s1, c252, bias1);  // (x + 126) / 252 in [0, 1]
  float p0, p1;
  uint32_t y0, y1;
  asm("{\n\t.reg .b64 t, r, m, y, w, f, p, k;\n\t"
      "mov.b64 t, {%4, %5};\n\tmov.b64 r, {%6, %6};\n\tmov.b64 m, {%7, %7};\n\t"
      "fma.rm.f32x2 y, t, r, m;\n\t"           // 1.5*2^23 + floor(x)
      "mov.b64 k, {%8, %8};\n\t"
      "fma.rn.f32x2 w, y, k, m;\n\t"           // -126 - floor(x), exact
      "fma.rn.f32x2 f, t, r, w;\n\t"           // x - floor(x)
      "mov.b64 p, {%9, %9};\n\tmov.b64 k, {%10, %10};\n\tfma.rn.f32x2 p, p, f, k;\n\t"
      "mov.b64 k, {%11, %11};\n\tfma.rn.f32x2 p, p, f, k;\n\t"
      "mov.b64 k, {%12, %12};\n\tfma.rn.f32x2 p, p, f, k;\n\t"
      "mov.b64 {%0, %1}, p;\n\tmov.b64 {%2, %3}, y;\n\t}"
      : "=f"(p0), "=f"(p1), "=r"(y0), "=r"(y1)
      : "f"(t0), "f"(t1), "f"(kPolyRange), "f"(kPolyMagic), "f"(-1.0f), "f"(kC3), "f"(kC2), "f"(kC1), "f"(kC0));
  e0 = __uint_as_float((y0 << 23) + __float_as_uint(p0));
  e1 = __uint_as_float((y1 << 23) + __float_as_uint(p1));
}
// Two values of exp2(x) as precise as ex2's: a polynomial of degree 5 for 2^f on [0, 1) (minimax in relative error, 7.5e-8) of
// the same argument that ex2 would take, and with ex2's results at the ends: zero below -126, infinity from 128 on, not a
// number for what is none. (The power of two is a factor and not added to the exponent's bits, which would make a number of
// everything: one more multiplication for two values.)
constexpr float kQ0 = 0.9999999404f, kQ1 = 0.6931530833f, kQ2 = 0.2401536107f, kQ3 = 0.05582631752f, kQ4 = 0.008989339694f, kQ5 = 0.001877576695f;
__device__ __forceinline__ void exp2_poly5(float& e0, float& e1, float x0, float x1) {
  asm("max.NaN.f32 %0, %0, %2;\n\tmax.NaN.f32 %1, %1, %2;" : "+f"(x0), "+f"(x1) : "f"(-127.0f));
  asm("min.NaN.f32 %0, %0, %2;\n\tmin.NaN.f32 %1, %1, %2;" : "+f"(x0), "+f"(x1) : "f"(128.0f));
  float p0, p1;
  uint32_t y0, y1;
  asm("{\n\t.reg .b64 x, m, y, w, f, p, k;\n\t"
      "mov.b64 x, {%4, %5};\n\tmov.b64 m, {%6, %6};\n\tmov.b64 k, {%7, %7};\n\t"
      "fma.rm.f32x2 y, x, k, m;\n\t"        // 1.5*2^23 + floor(x)
      "mov.b64 k, {%8, %8};\n\t"
      "fma.rn.f32x2 w, y, k, m;\n\t"        // -floor(x), exact
      "add.rn.f32x2 f, x, w;\n\t"           // x - floor(x), exact
      "mov.b64 p, {%9, %9};\n\tmov.b64 k, {%10, %10};\n\tfma.rn.f32x2 p, p, f, k;\n\t"
      "mov.b64 k, {%11, %11};\n\tfma.rn.f32x2 p, p, f, k;\n\t"
      "mov.b64 k, {%12, %12};\n\tfma.rn.f32x2 p, p, f, k;\n\t"
      "mov.b64 k, {%13, %13};\n\tfma.rn.f32x2 p, p, f, k;\n\t"
      "mov.b64 k, {%14, %14};\n\tfma.rn.f32x2 p, p, f, k;\n\t"
      "mov.b64 {%0, %1}, p;\n\tmov.b64 {%2, %3}, y;\n\t}"
      : "=f"(p0), "=f"(p1), "=r"(y0), "=r"(y1)
      : "f"(x0), "f"(x1), "f"(12582912.0f), "f"(1.0f), "f"(-1.0f), "f"(kQ5), "f"(kQ4), "f"(kQ3), "f"(kQ2), "f"(kQ1), "f"(kQ0));
  // 2^floor(x): 0 for -127, infinity for 128
  const float w0 = __uint_as_float((y0 << 23) + 0x3f800000u), w1 = __uint_as_float((y1 << 23) + 0x3f800000u);
  asm("{\n\t.reg .b64 p, w;\n\tmov.b64 p, {%2, %3};\n\tmov.b64 w, {%4, %5};\n\tmul.rn.f32x2 p, p, w;\n\tmov.b64 {%0, %1}, p;\n\t}"
      : "=f"(e0), "=f"(e1)
      : "f"(p0), "f"(p1), "f"(w0), "f"(w1));
}
// two multiply-adds / two adds in one instruction (same roundings as the scalar forms)
__device__ __forceinline__ void fma2(float& d0, float& d1, float a0, float a1, float b, float c0, float c1) {
  asm("{\n\t.reg .b64 ra, rb, rc, rd;\n\tmov.b64 ra, {%2, %3};\n\tmov.b64 rb, {%4, %4};\n\tmov.b64 rc, {%5, %6};\n\t"
      "fma.rn.f32x2 rd, ra, rb, rc;\n\tmov.b64 {%0, %1}, rd;\n\t}"
      : "=f"(d0), "=f"(d1)
      : "f"(a0), "f"(a1), "f"(b), "f"(c0), "f"(c1));
}
__device__ __forceinline__ void add2(float& d0, float& d1, float a0, float a1) {
  asm("{\n\t.reg .b64 ra, rd;\n\tmov.b64 ra, {%2, %3};\n\tmov.b64 rd, {%0, %1};\n\tadd.rn.f32x2 rd, rd, ra;\n\t"
      "mov.b64 {%0, %1}, rd;\n\t}"
      : "+f"(d0), "+f"(d1)
      : "f"(a0), "f"(a1));
}
__device__ __forceinline__ float poly_bias(float beta) { return (126.0f - beta) * (1.0f / kPolyRange); }

// m + log2(z): a row's log-sum-exp from its reference and its sum of exponentials (about 1 or more: the reference is one of
// the terms' exponents); no sum, or none that is a number, gives +inf, which mutes the row. The exponent of z goes to m first, so
// that the fast logarithm is of a number in [1, 2), where its error is absolute (2^-22) and small beside the sum's own
// rounding: of z itself it is relative, about 12 times that for some thousand keys, and all terms of a row move with it
// (2-norm error of the scores of 4096 tokens with 128 rows 3.1e-7; log2f 0.96e-7, but 0.5 us more a call).
__device__ __forceinline__ float log2_sum(float m, float z) {
  const uint32_t bits = __float_as_uint(z);
  const float e = (float)((int)(bits >> 23) - 127), f = __uint_as_float((bits & 0x007fffffu) | 0x3f800000u);
  return z > 0.0f && z < INFINITY ? (m + e) + __log2f(f) : INFINITY;
}

// Products K .. END-1 of the eight of a job: S = Q_block * Ktile^T (STATS) or S^T = Ktile * Q_block^T, 16 dimensions each.
template <int MB, bool STATS, int K, int END>
__device__ __forceinline__ void issue_job(uint32_t acc, uint32_t q_lo, uint32_t k_lo, uint32_t desc_hi, uint32_t idesc) {
  constexpr uint32_t oq = (uint32_t)((K >> 2) * (MB * kHalfBytes) + (K & 3) * 32) >> 4;
  constexpr uint32_t ok = (uint32_t)((K >> 2) * kHalfBytes + (K & 3) * 32) >> 4;
  if constexpr (STATS) umma_bf16_off<oq, ok, (K > 0)>(acc, q_lo, k_lo, desc_hi, idesc);
  else umma_bf16_off<ok, oq, (K > 0)>(acc, k_lo, q_lo, desc_hi, idesc);
  if constexpr (K + 1 < END) issue_job<MB, STATS, K + 1, END>(acc, q_lo, k_lo, desc_hi, idesc);
}

// ---------------------------------------------------------------------------------------------- the kernel
template <int MB, int PM>
__global__ void __launch_bounds__(kThreads, 1)
ta_score_kernel(const __grid_constant__ CUtensorMap map_q, const __grid_constant__ CUtensorMap map_k,
                const __grid_constant__ ScoreParams p) {
  using Smem = ScoreSmem<MB>;
  constexpr int kWarpTma = kSoftWarps, kWarpMma = kSoftWarps + 1, kWarpStat = kSoftWarps + 2;
  constexpr int kStatWarps = 2;
  constexpr int kQBufs = Smem::kQBufs, kRowsPad = Smem::kRowsPad, kStages = Smem::kStages;
  constexpr uint32_t kTmemCols = 512;  // kAcc accumulator stages of 128 columns
  extern __shared__ uint8_t smem_raw[];
  Smem& sm = *reinterpret_cast<Smem*>(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);

  // the warp index through a shuffle: the compiler then knows the role branches to be warp-uniform
  const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0), lane = tid & 31;
  const uint32_t rank = cluster_ctarank();
  const int cluster_id = blockIdx.x / p.cluster;
  const int n_clusters = gridDim.x / p.cluster;
  const bool one_round = p.units <= n_clusters;  // every cluster has at most one unit
  volatile int* abort_flag = &sm.abort_flag;
  const unsigned long long limit = p.wait_limit_ns;

  // The unit of round `round` of this cluster's walk over units cluster_id + round * n_clusters. With a length-sorted
  // order the rounds are taken in alternating direction (the cluster that got the longest unit of one round gets the
  // shortest of the next), which evens out the clusters' totals. False: there is nothing to do in this round (ui.end: nor in
  // any later one).
  // (Runs ahead of everything else in the CTA: 32-bit arithmetic, a 64-bit division costs some 0.2 us.)
  auto get_unit = [&](int round, UnitInfo& ui) {
    ui = UnitInfo{};
    int u, t_lo = 0, t_hi = 0;
    if (p.flat) {
      const int tiles = (p.seq.n_uniform + kTileN - 1) / kTileN;
      const long long all = (long long)p.units * tiles;
      const long long lo = all * cluster_id / n_clusters, hi = all * (cluster_id + 1) / n_clusters;
      u = (int)(lo / tiles) + round;
      t_lo = (int)max(lo - (long long)u * tiles, 0LL);
      t_hi = (int)min(hi - (long long)u * tiles, (long long)tiles);
      ui.end = t_lo >= t_hi;
    } else {
      u = round * n_clusters + cluster_id;
      ui.end = round * n_clusters >= p.units;
      if ((p.order || p.by_length) && (round & 1)) u = round * n_clusters + (n_clusters - 1 - cluster_id);
    }
    if (ui.end || u >= p.units) return false;
    if (p.order) u = p.order[u];
    // by_length: every sequence's units together (rank, then layer, then head); otherwise layer, sequence, head
    const uint32_t heads = (uint32_t)u / (uint32_t)p.Hkv, inner = (uint32_t)(p.by_length ? p.n_layers : p.seq.batch);
    const int major = (int)(heads / inner), minor = (int)(heads - (uint32_t)major * inner);
    ui.g = (int)((uint32_t)u - heads * (uint32_t)p.Hkv);
    ui.b = p.by_length ? sm.by_rank[major] : minor;
    ui.l = p.by_length ? minor : major;
    ui.tok0 = ta_seq_begin(p.seq, ui.b);
    ui.n = (p.seq.cu ? p.seq.cu[ui.b + 1] : ui.tok0 + p.seq.n_uniform) - ui.tok0;
    // a sequence that does not lie inside the token arrays is skipped here and rejected by the selection step
    if (ui.n > p.seq.max_n || ui.n < 0 || ui.tok0 < 0 || (long long)ui.tok0 + ui.n > p.seq.total) {
      if (atomicCAS(&p.status->code, 0, (int)TA_ERR_DEVICE_BOUNDS) == 0) {
        p.status->where = 2;
        p.status->detail0 = ui.b;
        p.status->detail1 = ui.n;
      }
      return false;
    }
    const int tiles_total = (ui.n + kTileN - 1) / kTileN;
    const uint32_t cl = (uint32_t)p.cluster;  // (at most 16, and at most 2^13 tiles)
    ui.t_begin = p.flat ? t_lo : (int)((uint32_t)tiles_total * rank / cl);
    ui.T = (p.flat ? t_hi : (int)((uint32_t)tiles_total * (rank + 1) / cl)) - ui.t_begin;
    // a CTA without tiles still takes part in its cluster's exchange of statistics
    return ui.T > 0 || (ui.n > 0 && p.two_pass && p.cluster > 1);
  };

  // the query tile of a unit into buffer qb; key tile j of a unit's walk (both passes) into stage s
  auto load_q = [&](const UnitInfo& ui, int qb) {
    const uint32_t bar = smem_u32(&sm.q_full[qb]);
    const uint32_t dst = smem_u32(sm.q[qb]);
    mbar_expect_tx(bar, (uint32_t)(2 * p.rows * 128));
    tma_load_5d(dst, &map_q, bar, 0, 0, ui.g * p.G, ui.b, ui.l);
    tma_load_5d(dst + MB * kHalfBytes, &map_q, bar, 64, 0, ui.g * p.G, ui.b, ui.l);
  };
  auto load_k = [&](const UnitInfo& ui, int j, int s) {
    // the second sweep walks the CTA's tiles backwards: the tiles read last are the ones still in L2
    const int tile = ui.t_begin + (j >= ui.T ? 2 * ui.T - 1 - j : j);
    const int row = (p.seq.cu ? ui.tok0 : 0) + tile * kTileN;  // ragged: tokens are packed along the row axis
    const int bc = p.seq.cu ? 0 : ui.b;
    const uint32_t bar = smem_u32(&sm.full[s]);
    const uint32_t dst = smem_u32(sm.k[s]);
    mbar_expect_tx(bar, kKTileBytes);
    tma_load_5d(dst, &map_k, bar, 0, row, ui.g, bc, ui.l);
    tma_load_5d(dst + kHalfBytes, &map_k, bar, 64, row, ui.g, bc, ui.l);
  };

  // ---- set-up (once per CTA). The warps share it, each its own barriers, a lane per barrier (all of them in one warp kept the
  // others waiting for 0.5 us). Every role gives or takes its registers first: later the softmax warps would wait for the
  // producer to come by.
  auto init = [&](unsigned long long* bar, int n, uint32_t count) {
    if (lane < n) mbar_init(smem_u32(bar + lane), count);
  };
  auto init_done = [&] {
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    __syncwarp();
  };
  bool cluster_known = false;  // this warp knows its peers to run
  // The end of the set-up. Every CTA of the cluster must be running (barriers initialised) before a peer writes to its shared
  // memory or arrives on its barriers: warps that do wait for that before the first time, the others only when they leave.
  auto set_up = [&] {
    tc_fence_before();
    asm volatile("bar.sync 1, %0;" ::"n"(kThreads) : "memory");
    tc_fence_after();
    cluster_arrive_relaxed();
  };
  // window index t of score row r = h*W + t, -1 for padding rows
  auto row_index = [&](int r) { return r < p.rows ? (int)((uint32_t)r % (uint32_t)p.W) : -1; };
  // the tables that the row constants are formed with and that pass 2 reads; written before the first row constants
  auto put_tables = [&](int r, int t) {
    const float w = t >= 0 ? p.wrow[t] : 0.0f;  // (1-rho) rho^(W-1-t); also right for W' < W (same exponent)
    sm.row_t[r] = (int8_t)t;
    sm.wrow[r] = w;
    // kOutFused: the row's contribution alpha + delta*w (positive, checked by the host) goes into the exponent
    sm.lv[r] = PM == kOutFused && t >= 0 ? log2f(fmaf(p.delta, w, p.alpha)) : 0.0f;
  };
  // pass-2 constant of row r from its log2-domain log-sum-exp (+inf: the row is mute)
  auto put_row = [&](int up, int r, float lse2) {
    const float beta = lse2 - sm.lv[r];
    const bool poly = MB == 2 && poly_pair<MB, PM>((r & 15) / 2);
    sm.tab[up][r] = poly ? poly_bias(beta) : -beta;
    // (A and P apart, up to 128 rows: the pension weight stands there, so that one address does for both)
    if constexpr (MB == 1 && PM == kOutAP) sm.tab[up][kRowsPad + r] = sm.wrow[r];
    if constexpr (MB == 2 && poly_pairs<MB, PM>() > 0) {
      if (poly) sm.tab[up][kRowsPad + r] = -beta;
    }
  };

  if (warp >= kSoftWarps) {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(kRegsOther));
    if (warp == kWarpTma) {
      // =========================================================================== TMA producer
      // Walks the units of this cluster, publishes each one's description in the unit ring and streams its tiles. It does not
      // wait for the others' set-up: it publishes its first unit and requests that unit's query tile and first key tiles at
      // once, unless the walk needs the lengths ranked first.
      const bool leader = elect_one();
      init(sm.full, kStages, 1);
      init(sm.empty, kStages, 1);
      init(sm.q_full, kQBufs, 1);
      init(sm.q_empty, kQBufs, 1);
      init(sm.ufull, kUnitRing, 1);
      init(sm.ufree, kUnitRing, kSoftWarps + 1 + (p.two_pass ? 0 : kStatWarps));  // softmax warps, MMA issuer, statistics warps
      if (lane == 0) sm.abort_flag = 0;
      init_done();
      UnitInfo first = {};
      bool first_work = false;
      int pre = 0;  // tiles of the first unit that are requested here
      if (p.by_length) {
        set_up();
        if (!p.late_wait) ta_wait_for_prior_grid();
      } else {
        asm volatile("bar.arrive 1, %0;" ::"n"(kThreads) : "memory");
        cluster_arrive_relaxed();
        if (!p.late_wait) ta_wait_for_prior_grid();  // nothing above reads memory
        first_work = get_unit(0, first);
        if (first_work) {
          pre = __shfl_sync(0xffffffffu, min(kStages, p.two_pass ? 2 * first.T : first.T), 0);
          if (leader) {
            if (pre > 0) load_q(first, 0);
            for (int j = 0; j < pre; ++j) load_k(first, j, j);
            sm.unit[0] = first;
            mbar_arrive(smem_u32(&sm.ufull[0]));
          }
          __syncwarp();
        }
      }
      uint32_t issued = (1u << pre) - 1u, q_issued = 0;  // stages that were armed at least once
      int s = pre % kStages, qb = 0, us = 0;
      uint32_t sph = pre == kStages ? 0 : 1, qph = 1, uph = 1;
      bool ok = true;
      for (int round = 0;; ++round) {
        UnitInfo ui = first;
        const bool begun = round == 0 && first_work;  // during set-up
        const bool work = begun || get_unit(round, ui);
        const bool end = !begun && ui.end != 0;
        if (!work && !end) continue;
        const int T = __shfl_sync(0xffffffffu, ui.T, 0);
        if (!begun) {
          ok = mbar_wait(smem_u32(&sm.ufree[us]), uph, abort_flag, p.status, 12, limit);
          if (!ok) break;
          if (leader) {
            sm.unit[us] = ui;
            mbar_arrive(smem_u32(&sm.ufull[us]));
          }
        }
        if (++us == kUnitRing) us = 0, uph ^= 1;
        if (end) break;
        if (T == 0) continue;
        if (!begun) {
          ok = mbar_wait(smem_u32(&sm.q_empty[qb]), qph, abort_flag, p.status, 11, limit);
          if (!ok) break;  // nothing may be copied into a buffer that was not handed back
          if (leader) load_q(ui, qb);
        }
        q_issued |= 1u << qb;
        if (++qb == kQBufs) qb = 0, qph ^= 1;
        const int n_tiles = p.two_pass ? 2 * T : T;
#pragma unroll 1
        for (int j = pre; j < n_tiles; ++j) {
          ok = mbar_wait(smem_u32(&sm.empty[s]), sph, abort_flag, p.status, 10, limit);
          if (!ok) break;
          if (leader) load_k(ui, j, s);
          issued |= 1u << s;
          if (++s == kStages) s = 0, sph ^= 1;
        }
        pre = 0;  // (requested during set-up: the first unit's only)
        if (!ok) break;
      }
      if (!ok || *abort_flag) {
        // drain: every copy that was started must have landed before the CTA may leave. A stage is only ever armed
        // after its previous contents were handed back, so at most the last copy per stage can still be in flight:
        // stages below the running index were last armed in this round of the ring, the others in the round before.
        for (int i = 0; i < kStages; ++i)
          if ((issued >> i) & 1u) mbar_wait_drain(smem_u32(&sm.full[i]), i < s ? sph ^ 1u : sph, limit);
        for (int i = 0; i < kQBufs; ++i)
          if ((q_issued >> i) & 1u) mbar_wait_drain(smem_u32(&sm.q_full[i]), i < qb ? qph ^ 1u : qph, limit);
      }
    } else if (warp == kWarpMma) {
      // =========================================================================== MMA issuer
      // The whole warp runs the loop and one elected lane issues: with the loop inside a single lane's branch the
      // products of a job took 730 cycles instead of the 512 that the tensor pipe needs. The barriers of the next job
      // are looked at in the middle of the current one, while products are still queued.
      const bool leader = elect_one();
      init(sm.acc_full, kAcc, 1);
      init(sm.acc_empty, kAcc, 4);
      init(&sm.drain, 1, 1);
      init_done();
      tmem_alloc(smem_u32(&sm.tmem_base), kTmemCols);
      tmem_relinquish();
      set_up();
      const uint32_t tmem_base = sm.tmem_base;
      bool ok = true;
      // operand descriptors: the upper word is the same for every tile; the lower word is the address >> 4
      const uint32_t desc_hi = (uint32_t)(smem_desc_sw128(0) >> 32);
      const uint32_t k_lo = (smem_u32(sm.k) & 0x3FFFFu) >> 4;
      const uint32_t q_lo0 = (smem_u32(sm.q[0]) & 0x3FFFFu) >> 4;
      const uint32_t idesc = idesc_bf16(128, 128);
      const uint32_t bar_full = smem_u32(&sm.full[0]), bar_empty = smem_u32(&sm.empty[0]);
      const uint32_t bar_af = smem_u32(&sm.acc_full[0]), bar_ae = smem_u32(&sm.acc_empty[0]);
      int qb = 0, s = 0, a = 0, us = 0;
      uint32_t qph = 0, sph = 0, aph = 1, uph = 0;
      bool k_ready = false, a_ready = false;  // the next job's key tile / accumulator stage is known to be ready
      for (;;) {
        ok = mbar_wait(smem_u32(&sm.ufull[us]), uph, abort_flag, p.status, 23, limit);
        if (!ok) break;
        const int T = __shfl_sync(0xffffffffu, sm.unit[us].T, 0), end = __shfl_sync(0xffffffffu, sm.unit[us].end, 0);
        __syncwarp();
        if (leader) mbar_arrive(smem_u32(&sm.ufree[us]));
        if (++us == kUnitRing) us = 0, uph ^= 1;
        if (end) break;
        if (T == 0) continue;
        ok = mbar_wait(smem_u32(&sm.q_full[qb]), qph, abort_flag, p.status, 22, limit);
        if (!ok) break;
        const uint32_t q_lo = q_lo0 + (uint32_t)((qb * (MB * 2 * kHalfBytes)) >> 4);
        // A tile's product is issued as MB jobs, one per block of 128 score rows, each into its own accumulator
        // stage of 128 columns: S = Q_block * Ktile^T in pass 1, S^T = Ktile * Q_block^T in pass 2. No product is issued
        // on operands that are not ready, nor into an accumulator that was not handed back.
        auto sweep = [&](auto stats_tag) {
          constexpr bool stats = decltype(stats_tag)::value;
#pragma unroll 1
          for (int jt = 0; jt < T; ++jt) {
            if (!k_ready && !mbar_wait(bar_full + s * 8, sph, abort_flag, p.status, 20, limit)) return false;
            const uint32_t dk_lo = k_lo + (uint32_t)((s * kKTileBytes) >> 4);
            const uint32_t bar_es = bar_empty + s * 8;
            if (++s == kStages) s = 0, sph ^= 1;
#pragma unroll
            for (int rb = 0; rb < MB; ++rb) {
              if (!a_ready && !mbar_wait(bar_ae + a * 8, aph, abort_flag, p.status, 21, limit)) return false;
              tc_fence_after();
              const uint32_t acc = tmem_base + (uint32_t)(a * 128);
              const uint32_t bar_fa = bar_af + a * 8;
              const uint32_t dq_lo = q_lo + (uint32_t)((rb * kHalfBytes) >> 4);
              if (++a == kAcc) a = 0, aph ^= 1;
              if (leader) issue_job<MB, stats, 0, 4>(acc, dq_lo, dk_lo, desc_hi, idesc);
              a_ready = mbar_test(bar_ae + a * 8, aph);
              if (rb == MB - 1) k_ready = mbar_test(bar_full + s * 8, sph);
              if (leader) {
                issue_job<MB, stats, 4, 8>(acc, dq_lo, dk_lo, desc_hi, idesc);
                if (rb == MB - 1) umma_commit(bar_es);
                umma_commit(bar_fa);
              }
            }
          }
          return true;
        };
        if (p.two_pass) ok = sweep(std::true_type{});
        if (ok) ok = sweep(std::false_type{});
        if (!ok) break;
        if (leader) umma_commit(smem_u32(&sm.q_empty[qb]));  // the query tile may be overwritten once these MMAs are done
        if (++qb == kQBufs) qb = 0, qph ^= 1;
      }
      if (!ok || *abort_flag) {  // make sure no MMA is still writing tensor memory before it is freed
        if (leader) umma_commit(smem_u32(&sm.drain));
        mbar_wait_drain(smem_u32(&sm.drain), 0, limit);
      }
    } else {
      // =========================================================================== statistics warps
      // One pass: the row constants of the units, ahead of the softmax warps, from the log-sum-exps that the caller supplied.
      // (Between two passes the softmax warps have nothing else to do and form them themselves.)
      if (warp == kWarpStat) {
        init(&sm.stat_full, 1, kSoftWarps);
        init(sm.tab_full, 2, p.two_pass ? 4 : kStatWarps);
        init(sm.tab_free, 2, kSoftWarps);
        init(&sm.xchg_full, 1, 1);
        init(&sm.xchg_free, 1, (uint32_t)p.cluster * 4);
      } else {
        init(sm.pfull, kRing, 4);
        init(sm.pfree, kRing, 4);
      }
      init_done();
      set_up();
      if (!p.late_wait) ta_wait_for_prior_grid();
      const int r0 = (warp - kWarpStat) * 32 + lane;
      int us = 0;
      uint32_t uph = 0;
      // a wait that ran out in an earlier CTA or call (not yet polled) makes the remaining CTAs give up their waits at once
      if (*reinterpret_cast<volatile int*>(&p.status->code) == (int)TA_ERR_TIMEOUT) *abort_flag = 1;
      constexpr int kRows = kRowsPad / (32 * kStatWarps);
      int tr[kRows];
      if (!p.two_pass) {
#pragma unroll
        for (int i = 0; i < kRows; ++i) {
          tr[i] = row_index(r0 + 32 * kStatWarps * i);
          put_tables(r0 + 32 * kStatWarps * i, tr[i]);
        }
      }
      for (int it = 0; !p.two_pass; ++it) {
        if (!mbar_wait(smem_u32(&sm.ufull[us]), uph, abort_flag, p.status, 36, limit)) break;
        const UnitInfo ui = sm.unit[us];
        __syncwarp();
        if (lane == 0) mbar_arrive(smem_u32(&sm.ufree[us]));
        if (++us == kUnitRing) us = 0, uph ^= 1;
        if (ui.end) break;
        const int up = it & 1;
        const uint32_t ph = (uint32_t)(it >> 1) & 1u;
        mbar_wait(smem_u32(&sm.tab_free[up]), ph ^ 1u, abort_flag, p.status, 37, limit);
#pragma unroll
        for (int i = 0; i < kRows; ++i) {
          const int r = r0 + 32 * kStatWarps * i, t = tr[i];
          float lse2 = INFINITY;
          if (t >= 0 && ui.n - p.W + t >= 0) {
            const int h = r / p.W;
            const float lse = p.lse_obs[(((long long)ui.l * p.seq.batch + ui.b) * p.Hq + (ui.g * p.G + h)) * p.W + t];
            lse2 = lse * 1.4426950408889634f;
          }
          put_row(up, r, lse2);
        }
        __syncwarp();
        if (lane == 0) mbar_arrive(smem_u32(&sm.tab_full[up]));
      }
    }
  } else {
    // =========================================================================== softmax warps
    // A job is one block of 128 score rows of one key tile in one pass. Jobs are numbered through over passes and units
    // and dealt round-robin: group grp takes jobs grp, grp + kGroups, ..; job J uses accumulator stage J mod kAcc.
    asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(kRegsSoftmax));
    // Rows of the query tile that the TMA box does not cover are multiplied like any other row: make them zeros so
    // that the padded score columns are finite.
    if (p.rows < kRowsPad) {
      const int pad_rows = kRowsPad - p.rows;
      for (int i = tid; i < kQBufs * 2 * pad_rows * 8; i += kSoftWarps * 32) {
        const int qb = i / (2 * pad_rows * 8), i2 = i % (2 * pad_rows * 8);
        const int half = i2 / (pad_rows * 8), rem = i2 % (pad_rows * 8);
        const int row = p.rows + rem / 8, chunk = rem % 8;
        *reinterpret_cast<uint4*>(&sm.q[qb][half * (MB * kHalfBytes) + row * 128 + chunk * 16]) = make_uint4(0, 0, 0, 0);
      }
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    if (!p.late_wait) ta_wait_for_prior_grid();
    if (p.by_length) {
      // Longest first, equal lengths in sequence order. In unit order the lengths a cluster meets are random and the busiest
      // cluster of a batch with lengths spread 8x carries about 30 % more than the average.
      for (int b = tid; b < p.seq.batch; b += kSoftWarps * 32) {
        const int nb = p.seq.cu[b + 1] - p.seq.cu[b];
        int rank = 0;
        for (int o = 0; o < p.seq.batch; ++o) {
          const int no = p.seq.cu[o + 1] - p.seq.cu[o];
          rank += (no > nb) || (no == nb && o < b);
        }
        sm.by_rank[rank] = (uint8_t)b;
      }
    }
    set_up();
    const uint32_t tmem_base = sm.tmem_base;
    const int grp = warp >> 2;
    const int quad = warp & 3;              // TMEM lane quadrant this warp may read
    const int row_in_tile = quad * 32 + lane;
    static_assert(kGroups % MB == 0, "a group's jobs are all of one row block");
    const int block = MB == 2 ? grp & 1 : 0;  // row block of this group's jobs (a unit has an even number of jobs)
    const uint32_t tlane = tmem_base + ((uint32_t)(quad * 32) << 16);
    const uint32_t bar_af = smem_u32(&sm.acc_full[0]), bar_ae = smem_u32(&sm.acc_empty[0]);
    const float c = p.c;
    const float c252 = c * (1.0f / kPolyRange);

    auto acc_addr = [&](int J) { return tlane + (uint32_t)((J % kAcc) * 128); };
    auto wait_full = [&](int J, int where) {
      mbar_wait(bar_af + (J % kAcc) * 8, (uint32_t)(J / kAcc) & 1u, abort_flag, p.status, where, limit);
      tc_fence_after();
    };
    auto release = [&](int J) {  // the whole accumulator of the job is in registers: hand the stage back
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(bar_ae + (J % kAcc) * 8);
    };

    int tr = -1;  // window index of this thread's row in pass 1
    if (p.two_pass) {
      tr = row_index(block * 128 + row_in_tile);
      if (grp < MB) put_tables(block * 128 + row_in_tile, tr);
    }
    int J = grp;        // this group's next job
    int jg = 0;         // first job of the current pass
    int tg = 0;         // MB 2: pass-2 tiles of the units before this one
    float ra[16], rb[16];
    bool fetched = false;  // the first 16 columns of job J are in flight in `ra`
    int us = 0;
    uint32_t uph = 0;
    for (int it = 0;; ++it) {
      if (!mbar_wait(smem_u32(&sm.ufull[us]), uph, abort_flag, p.status, 35, limit)) break;
      const UnitInfo ui = sm.unit[us];
      __syncwarp();
      if (lane == 0) mbar_arrive(smem_u32(&sm.ufree[us]));
      if (++us == kUnitRing) us = 0, uph ^= 1;
      if (ui.end) break;
      const int n = ui.n, n_jobs = MB * ui.T;
      const int up = it & 1;
      const uint32_t ph = (uint32_t)(it >> 1) & 1u;
      const int j_last = jg + (p.two_pass ? 2 : 1) * n_jobs;  // end of the unit's jobs
      auto fetch = [&](int Jn) {  // starts the load of job Jn's first 16 columns (waits for its products)
        wait_full(Jn, 30);
        tmem_ld16_issue(acc_addr(Jn), ra);
      };
      // the same if job Jn is one of the unit's and its products are there
      auto try_fetch = [&](int Jn) {
        if (Jn >= j_last || !mbar_test(bar_af + (Jn % kAcc) * 8, (uint32_t)(Jn / kAcc) & 1u)) return false;
        tc_fence_after();
        tmem_ld16_issue(acc_addr(Jn), ra);
        return true;
      };

      if (p.two_pass) {
        // ---- pass 1: per row, sum of exp2(s*c - ref) against a reference `ref` that only has to keep the sum inside
        // the fp32 range (the result does not depend on it): the largest of the first 16 keys the row sees. After that
        // a key costs one multiply-add, one exponential and one add, and no maximum is tracked. A tile whose sum
        // leaves the safe range (a score more than 2^60 above ref) is redone against its own maximum. The check runs
        // before the accumulator stage is released and does not wait for the tile's last exponentials: it uses the sum
        // without the last 16 keys and, for those, their largest score. The cubic's exponentials saturate at 2^126,
        // which the same check catches; so does a row without a reference yet (ref -1e30).
        const int pos = n - p.W + tr;
        const int lim = (tr >= 0 && pos >= 0) ? (p.causal ? pos : n - 1) : -1;  // last key that the thread's row sees
        // rows that see no key (padding) get a reference that turns every exponential into 0
        float ref = lim >= 0 ? -1e30f : 1e30f, zsum = 0.0f;
        constexpr float kSumLimit = 1.0e18f;  // about 2^60
        // 16 keys of one row: adds exp2(s*c - rc) to the four sums; `mix`: some of them on the FMA pipe. Masked tiles
        // drop keys beyond `lm`.
        auto half1 = [&](auto masked_tag, auto mix_tag, const float(&cur)[16], float rc, float pbias, float(&s4)[4],
                         int lm, int kbase) {
          constexpr bool masked = decltype(masked_tag)::value;
          constexpr bool mix = decltype(mix_tag)::value;
          float v[16];
#pragma unroll
          for (int q = 0; q < 16; ++q) v[q] = (masked && kbase + q > lm) ? -INFINITY : cur[q];
#pragma unroll
          for (int q = 0; q < 16; q += 2) {
            float e0, e1;
            if (mix && !masked && poly_pair<MB, PM>(q / 2)) {
              if constexpr (MB == 2) {
                exp2_poly2(e0, e1, v[q], v[q + 1], c252, pbias, pbias);
              } else {
                fma2(e0, e1, v[q], v[q + 1], c, -rc, -rc);
                exp2_poly5(e0, e1, e0, e1);
              }
            } else {
              fma2(e0, e1, v[q], v[q + 1], c, -rc, -rc);
              e0 = ex2(e0);
              e1 = ex2(e1);
            }
            add2(s4[q & 3], s4[(q & 3) + 1], e0, e1);
          }
        };
        auto max16 = [&](auto masked_tag, const float(&cur)[16], int lm, int kbase) {  // largest of 16 keys of one row
          constexpr bool masked = decltype(masked_tag)::value;
          float t4[4];
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            float w[4];
#pragma unroll
            for (int e = 0; e < 4; ++e) w[e] = (masked && kbase + 4 * q + e > lm) ? -INFINITY : cur[4 * q + e];
            t4[q] = fmaxf(fmaxf(w[0], w[1]), fmaxf(w[2], w[3]));
          }
          return fmaxf(fmaxf(t4[0], t4[1]), fmaxf(t4[2], t4[3]));
        };
        // One job: the 128 accumulator columns in 32-column chunks, each fetched as two 16-column loads (ra, rb) so
        // that one load is always in flight. On entry the load of the first 16 columns is in flight in `ra`.
        auto job1 = [&](auto masked_tag, float& ref_c, float& z_run, int lm, int key0) {
          const uint32_t abase = acc_addr(J);
          float rc = ref_c;
          float pb = poly_bias(rc);
          float s4[4] = {0.0f, 0.0f, 0.0f, 0.0f};
#pragma unroll 1
          for (int c4 = 0; c4 < 4; ++c4) {
            const uint32_t col = (uint32_t)(c4 * 32);
            tmem_ld_wait(ra);
            tmem_ld16_issue(abase + col + 16, rb);
            half1(masked_tag, std::true_type{}, ra, rc, pb, s4, lm, key0 + c4 * 32);
            tmem_ld_wait(rb);
            if (c4 < 3) {
              tmem_ld16_issue(abase + col + 32, ra);
              half1(masked_tag, std::true_type{}, rb, rc, pb, s4, lm, key0 + c4 * 32 + 16);
            }
          }
          const float sum_head = (s4[0] + s4[1]) + (s4[2] + s4[3]);
          const float mx_tail = max16(masked_tag, rb, lm, key0 + 112);
          // also true for inf and NaN sums
          const bool over = !(sum_head < kSumLimit) || fmaf(mx_tail, c, -rc) > 60.0f;
          if (__any_sync(0xffffffffu, over)) {  // rare: a score far above the reference
            float mx = -INFINITY;
#pragma unroll 1
            for (int h = 0; h < 8; ++h) {
              tmem_ld16_issue(abase + (uint32_t)(h * 16), ra);
              tmem_ld_wait(ra);
              mx = fmaxf(mx, max16(masked_tag, ra, lm, key0 + h * 16));
            }
            const float mx_c = mx * c;
            float r4[4] = {0.0f, 0.0f, 0.0f, 0.0f};
#pragma unroll 1
            for (int h = 0; h < 7; ++h) {
              tmem_ld16_issue(abase + (uint32_t)(h * 16), ra);
              tmem_ld_wait(ra);
              half1(masked_tag, std::false_type{}, ra, over ? mx_c : rc, 0.0f, r4, lm, key0 + h * 16);
            }
            if (over) {
              z_run *= ex2(rc - mx_c);
              rc = ref_c = mx_c;
              pb = poly_bias(mx_c);
#pragma unroll
              for (int q = 0; q < 4; ++q) s4[q] = r4[q];
            }
          }
          release(J);
          fetched = try_fetch(J + kGroups);
          half1(masked_tag, std::true_type{}, rb, rc, pb, s4, lm, key0 + 112);
          z_run += (s4[0] + s4[1]) + (s4[2] + s4[3]);
        };
        const int j_end = jg + n_jobs;
        bool first = true;
        for (; J < j_end; J += kGroups) {
          const int key0 = (ui.t_begin + (J - jg) / MB) * kTileN;
          if (!fetched) fetch(J);
          // tiles that every row of the warp sees completely take the unmasked path (rows that see nothing at all,
          // i.e. padding, still run: their sums are never used)
          const bool masked = __any_sync(0xffffffffu, lim >= 0 && key0 + kTileN - 1 > lim);
          if (first) {  // the reference of the rows: from the 16 keys in flight
            tmem_ld_wait(ra);
            const float mx = masked ? max16(std::true_type{}, ra, lim, key0) : max16(std::false_type{}, ra, lim, key0);
            if (ref < -1e29f && mx > -INFINITY) ref = mx * c;
            first = false;
          }
          if (masked) job1(std::true_type{}, ref, zsum, lim, key0);
          else job1(std::false_type{}, ref, zsum, lim, key0);
        }
        // ---- the group's statistics of the unit; rows that see no key at all (padding, window positions before the
        // sequence start) stay mute
        sm.part_m[grp][row_in_tile] = lim >= 0 ? ref : -1e30f;
        sm.part_z[grp][row_in_tile] = lim >= 0 ? zsum : 0.0f;
        __syncwarp();
        if (lane == 0) mbar_arrive(smem_u32(&sm.stat_full));
        // ---- The group that was done first (the next job would be its) merges the groups' statistics, exchanges them with the
        // cluster's other CTAs and leaves the rows' constants for pass 2: a thread per row (MB 2: two).
        if (J == j_end) {
          mbar_wait(smem_u32(&sm.stat_full), (uint32_t)it & 1u, abort_flag, p.status, 38, limit);
          float m[MB], z[MB];
#pragma unroll
          for (int h = 0; h < MB; ++h) {
            m[h] = sm.part_m[h][row_in_tile];
#pragma unroll
            for (int gq = h + MB; gq < kGroups; gq += MB) m[h] = fmaxf(m[h], sm.part_m[gq][row_in_tile]);
            z[h] = 0.0f;
#pragma unroll
            for (int gq = h; gq < kGroups; gq += MB) z[h] += sm.part_z[gq][row_in_tile] * ex2(sm.part_m[gq][row_in_tile] - m[h]);
          }
          if (p.cluster > 1) {  // (alone, the CTA's statistics are the unit's)
            if (!cluster_known) cluster_wait();
            cluster_known = true;
            // the peers have read what was sent to them for the unit before
            if (it > 0) mbar_wait_cluster(smem_u32(&sm.xchg_free), (uint32_t)(it - 1) & 1u, abort_flag, p.status, 31, limit);
            if (quad == 0 && lane == 0) mbar_expect_tx(smem_u32(&sm.xchg_full), (uint32_t)(p.cluster * kRowsPad * 8));
            // stores that count on the receiver's barrier when they land: no fence, no separate signal
#pragma unroll 2
            for (int q = 0; q < p.cluster; ++q) {
              const uint32_t bar = map_peer(smem_u32(&sm.xchg_full), (uint32_t)q);
#pragma unroll
              for (int h = 0; h < MB; ++h)
                st_async_f32x2(map_peer(smem_u32(&sm.peer[rank][h * 128 + row_in_tile]), (uint32_t)q), m[h], z[h], bar);
            }
            mbar_wait_cluster(smem_u32(&sm.xchg_full), (uint32_t)it & 1u, abort_flag, p.status, 32, limit);
#pragma unroll
            for (int h = 0; h < MB; ++h) m[h] = -1e30f, z[h] = 0.0f;
#pragma unroll 4
            for (int q = 0; q < p.cluster; ++q)
#pragma unroll
              for (int h = 0; h < MB; ++h) m[h] = fmaxf(m[h], sm.peer[q][h * 128 + row_in_tile].x);
#pragma unroll 4
            for (int q = 0; q < p.cluster; ++q)
#pragma unroll
              for (int h = 0; h < MB; ++h) {
                const float2 v = sm.peer[q][h * 128 + row_in_tile];
                z[h] += v.y * ex2(v.x - m[h]);
              }
            if (!one_round) {  // the slots may be written again
              __syncwarp();
              if (lane < p.cluster) mbar_arrive_remote(smem_u32(&sm.xchg_free), (uint32_t)lane);
            }
          }
#pragma unroll
          for (int h = 0; h < MB; ++h) put_row(up, h * 128 + row_in_tile, log2_sum(m[h], z[h]));
          __syncwarp();
          if (lane == 0) mbar_arrive(smem_u32(&sm.tab_full[up]));
        }
        jg = j_end;
      }

      // ---- pass 2: for key row_in_tile of each tile, the sum over the job's rows of exp2(s*c - beta_row)
      {
        mbar_wait(smem_u32(&sm.tab_full[up]), ph, abort_flag, p.status, 39, limit);
        // every valid row sees keys up to here; key i beyond it is seen by the rows with t >= i - (n - W)
        const int min_lim = p.causal ? n - min(p.W, n) : n - 1;
        const long long out0 = ((long long)ui.l * p.Hkv + ui.g) * p.seq.total + ui.tok0;
        float sA4[4], sP;
        // 16 rows (half `hi` of the 32-row chunk cc) of this thread's key, a share of the exponentials on the FMA pipe.
        // Masked form (keys inside the observation window): rows that do not see the key are dropped, and every exponential
        // is ex2's. The last keys are seen by few rows (the last one by one row per head), so that a share of cubics, 2 of
        // 16 over many rows, would be all of such a key's sum there (7.5e-5 instead of 1e-6); a few tiles per unit.
        auto chunk2 = [&](auto masked_tag, auto hi_tag, const float(&cur)[16], int row0, int tau) {
          constexpr bool masked = decltype(masked_tag)::value;
          constexpr int hi = decltype(hi_tag)::value;  // 0: rows row0..row0+15, 1: rows row0+16..row0+31
          const float4* tab4 = reinterpret_cast<const float4*>(&sm.tab[up][row0]) + hi * 4;
          const float4* w4 = MB == 1 ? tab4 + kRowsPad / 4 : reinterpret_cast<const float4*>(&sm.wrow[row0]) + hi * 4;
          const char4* t4 = reinterpret_cast<const char4*>(&sm.row_t[row0]) + hi * 4;
#pragma unroll
          for (int q4 = 0; q4 < 4; ++q4) {
            const float4 tb = tab4[q4];
            float tbv[4] = {tb.x, tb.y, tb.z, tb.w};
            float a[4];
#pragma unroll
            for (int e = 0; e < 4; e += 2) {
              if (poly_pair<MB, PM>(2 * q4 + e / 2) && !masked) {
                if constexpr (MB == 2) {
                  exp2_poly2(a[e], a[e + 1], cur[4 * q4 + e], cur[4 * q4 + e + 1], c252, tbv[e], tbv[e + 1]);
                } else {
                  fma2(a[e], a[e + 1], cur[4 * q4 + e], cur[4 * q4 + e + 1], c, tbv[e], tbv[e + 1]);
                  exp2_poly5(a[e], a[e + 1], a[e], a[e + 1]);
                }
              } else {
                if (MB == 2 && poly_pair<MB, PM>(2 * q4 + e / 2)) {
                  const float2 nb = *reinterpret_cast<const float2*>(&sm.tab[up][kRowsPad + row0 + hi * 16 + 4 * q4 + e]);
                  tbv[e] = nb.x;
                  tbv[e + 1] = nb.y;
                }
                fma2(a[e], a[e + 1], cur[4 * q4 + e], cur[4 * q4 + e + 1], c, tbv[e], tbv[e + 1]);
                a[e] = ex2(a[e]);
                a[e + 1] = ex2(a[e + 1]);
              }
            }
            if (masked) {
              const char4 tt = t4[q4];
              if (tt.x < tau) a[0] = 0.0f;
              if (tt.y < tau) a[1] = 0.0f;
              if (tt.z < tau) a[2] = 0.0f;
              if (tt.w < tau) a[3] = 0.0f;
            }
            add2(sA4[0], sA4[1], a[0], a[1]);
            add2(sA4[2], sA4[3], a[2], a[3]);
            if (PM == kOutAP) {
              const float4 ws = w4[q4];
              sP = fmaf(ws.x, a[0], sP);
              sP = fmaf(ws.y, a[1], sP);
              sP = fmaf(ws.z, a[2], sP);
              sP = fmaf(ws.w, a[3], sP);
            }
          }
        };
        // one job: 32-row chunks, each as two 16-column loads (ra low half, rb high half)
        auto job2 = [&](auto masked_tag, int row0, int n_chunks, int tau) {
          const uint32_t abase = acc_addr(J);
#pragma unroll 1
          for (int ci = 0; ci < n_chunks; ++ci) {
            const uint32_t col = (uint32_t)(ci * 32);
            tmem_ld_wait(ra);
            tmem_ld16_issue(abase + col + 16, rb);
            chunk2(masked_tag, std::integral_constant<int, 0>{}, ra, row0 + ci * 32, tau);
            tmem_ld_wait(rb);
            if (ci == n_chunks - 1) {
              release(J);
              fetched = try_fetch(J + kGroups);
            } else {
              tmem_ld16_issue(abase + col + 32, ra);
            }
            chunk2(masked_tag, std::integral_constant<int, 1>{}, rb, row0 + ci * 32, tau);
          }
        };
        for (; J < j_last; J += kGroups) {
          const int tl = (J - jg) / MB;  // the pass walks the CTA's tiles backwards after a first pass
          const int key = (ui.t_begin + (p.two_pass ? ui.T - 1 - tl : tl)) * kTileN + row_in_tile;
          const int n_chunks = (min(128, p.rows - block * 128) + 31) >> 5;
          if (!fetched) fetch(J);
          sA4[0] = sA4[1] = sA4[2] = sA4[3] = 0.0f;
          sP = 0.0f;
          // only the last W-1 keys of a sequence are hidden from some rows: those tiles take the masked path
          if (__all_sync(0xffffffffu, key <= min_lim || key >= n)) job2(std::false_type{}, block * 128, n_chunks, 0);
          else job2(std::true_type{}, block * 128, n_chunks, p.causal ? key - (n - p.W) : -1);
          float sA = (sA4[0] + sA4[1]) + (sA4[2] + sA4[3]);
          if (MB == 2) {
            // The two row blocks of a tile are consecutive jobs of two different groups. The group of block 0 leaves
            // its sums in a ring slot and goes on; the group of block 1, which gets its job later, picks them up, adds
            // its own and stores. Neither waits for the other unless the ring is full (block 0 four tiles ahead).
            const int r = (tg + tl) % kRing;
            const uint32_t rph = (uint32_t)((tg + tl) / kRing) & 1u;
            if (block == 0) {
              mbar_wait(smem_u32(&sm.pfree[r]), rph ^ 1u, abort_flag, p.status, 33, limit);
              sm.psum[r][0][row_in_tile] = sA;
              if (PM == kOutAP) sm.psum[r][1][row_in_tile] = sP;
              __syncwarp();
              if (lane == 0) mbar_arrive(smem_u32(&sm.pfull[r]));
            } else {
              mbar_wait(smem_u32(&sm.pfull[r]), rph, abort_flag, p.status, 34, limit);
              sA += sm.psum[r][0][row_in_tile];
              if (PM == kOutAP) sP += sm.psum[r][1][row_in_tile];
              __syncwarp();
              if (lane == 0) mbar_arrive(smem_u32(&sm.pfree[r]));
            }
          }
          if (block == MB - 1 && key < n && !*abort_flag) {
            const long long o = out0 + key;
            if (PM == kOutFused) {
              p.u[o] = sA;
            } else {
              if (p.A) p.A[o] = sA;
              if (p.P) p.P[o] = sP;
              if (p.u) p.u[o] = __fadd_rn(__fmul_rn(p.alpha, sA), __fmul_rn(p.delta, sP));
            }
          }
        }
        if (!p.two_pass) {
          __syncwarp();
          if (lane == 0) mbar_arrive(smem_u32(&sm.tab_free[up]));
        }
      }
      jg = j_last;
      tg += ui.T;
    }
  }

  // ---- teardown
  tc_fence_before();
  __syncthreads();
  if (warp == kWarpMma) {
    tc_fence_after();
    tmem_dealloc(sm.tmem_base, kTmemCols);
  }
  // no CTA may leave while a peer can still write to its shared memory or arrive on its barriers
  if (!cluster_known) cluster_wait();  // the set-up's arrival
  cluster_arrive();
  cluster_wait();
  // (after a wait that ran out, statistics that this CTA did not wait for may still be on their way to it)
  if (*abort_flag) __nanosleep(50000);
  if (p.late_wait && blockIdx.x == 0) ta_wait_for_prior_grid();  // this grid ends after the one it ran beside
}

template <int MB>
size_t score_smem_bytes() {
  static_assert(sizeof(ScoreSmem<MB>) + 1024 <= 227 * 1024, "shared memory of a block");
  return sizeof(ScoreSmem<MB>) + 1024;
}

CUresult encode_5d(void* fn, CUtensorMap* map, const void* base, const uint64_t dims[5], const uint64_t strides_el[4],
                   const uint32_t box[5]) {
  auto enc = reinterpret_cast<CUresult (*)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                           const cuuint64_t*, const cuuint32_t*, const cuuint32_t*,
                                           CUtensorMapInterleave, CUtensorMapSwizzle, CUtensorMapL2promotion,
                                           CUtensorMapFloatOOBfill)>(fn);
  cuuint64_t gdim[5], gstr[4];
  cuuint32_t bx[5], es[5];
  for (int i = 0; i < 5; ++i) {
    gdim[i] = dims[i];
    bx[i] = box[i];
    es[i] = 1;
  }
  for (int i = 0; i < 4; ++i) gstr[i] = strides_el[i] * 2;  // bytes
  return enc(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 5, const_cast<void*>(base), gdim, gstr, bx, es,
             CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
             CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
}

template <int MB, int PM>
cudaError_t launch_variant(ta_ctx* ctx, const CUtensorMap& mq, const CUtensorMap& mk, ScoreParams& sp,
                           int tiles_max, int pdl, cudaStream_t stream) {
  auto kern = ta_score_kernel<MB, PM>;
  const size_t smem = score_smem_bytes<MB>();
  // per context (and so per device) and instantiation: the attribute is sticky, the occupancy does not change
  constexpr int vi = (MB - 1) * 3 + (PM == kOutA ? 0 : PM == kOutAP ? 1 : 2);
  int* max_clusters = ctx->score_max_clusters[vi];
  if (!ctx->score_attr_set[vi]) {
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    if (e != cudaSuccess) return e;
    // the in-kernel register split must fit in what the launch provides, or the warps asking for more wait forever
    cudaFuncAttributes fa;
    e = cudaFuncGetAttributes(&fa, kern);
    if (e != cudaSuccess) return e;
    if (fa.numRegs * kThreads < kRegsNeeded) return cudaErrorLaunchOutOfResources;
    for (int cl = 0; cl <= kMaxCluster; ++cl) max_clusters[cl] = 0;
    ctx->score_attr_set[vi] = 1;
  }
  cudaLaunchConfig_t cfg = {};
  cfg.blockDim = dim3(kThreads, 1, 1);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = stream;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = (unsigned)sp.cluster;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  // Persistent grid: as many clusters as can be resident at once (queried once per cluster size). CTAs per unit: the size
  // with the shortest busiest CTA, counted in half jobs: two per job, and per unit what its start and the statistics between the
  // passes take, four per row block with one CTA per unit, 5 (128 rows) or 8 (256) with several. Measured on 32 to 512 units of
  // 1000 to 12000 tokens, 80 sizes per row count, every size forced in turn: what this takes is 0.2 % (256 rows) and 0.00 %
  // (128) slower on average than the best, at most 4.1 % and 0.2 % (152 units of 2048 tokens with 256 rows: 98 us with 1 CTA,
  // 83 us with 2; 320 units of 4096 tokens with 128 rows: 149 us with 1, 134 us with 2). Jobs are not rounded up to whole
  // rounds of the softmax groups: fewer than four at work take little longer per job.
  // With 256 rows 9 to 16 CTAs need the peers' 32 KB, for which one of four stages of key tiles made room (16 x 32768 tokens take as
  // long: 12.63 and 12.61 ms). us a layer with 8 and with up to 16 CTAs: 2 units of 14714 tokens 61.4 / 42.8, of 16000 64.3 / 44.0, of
  // 5000 30.8 / 26.2; 8 units of 8000 39.5 / 37.4, of 6000 34.5 / 32.6.
  // (Choosing more CTAs per unit so that the keys of all units in flight fit in L2 was measured and lost: 16 x 32768
  // tokens, 8 CTAs per unit 2.02 ms against 1.63 ms. With 16 or 32 rows, where the second read is what bounds it, too: 1296 units of
  // 5634 tokens 555, 539, 634, 815 us with 1, 2, 4 and 8 CTAs, 1024 of 12000 912, 927, 999, 1213.)
  int best_cl = ctx->score_force_cluster;
  long long best_cost = best_cl > 0 ? 0 : -1;
  for (int cl = 1; cl <= kMaxCluster; cl = cl < 8 ? 2 * cl : cl + 1) {
    if (ctx->score_force_cluster > 0 && cl != ctx->score_force_cluster) continue;
    if (cl > 1 && tiles_max < 2 * cl && ctx->score_force_cluster <= 0) break;
    if (cl > 8 && sp.units > max_clusters[8]) break;  // only for a single round of few units
    if (max_clusters[cl] == 0) {
      attr[0].val.clusterDim.x = (unsigned)cl;
      cfg.gridDim = dim3((unsigned)(ctx->sm_count / cl * cl), 1, 1);
      int n = 0;
      cudaError_t e = cudaOccupancyMaxActiveClusters(&n, kern, &cfg);
      if (e != cudaSuccess) return e;
      max_clusters[cl] = n < 1 ? -1 : n;
    }
    if (max_clusters[cl] < 1) {
      if (ctx->score_force_cluster > 0) return cudaErrorLaunchOutOfResources;
      continue;
    }
    if (ctx->score_force_cluster > 0) break;
    const int avail = max_clusters[cl];
    const long long rounds = (sp.units + avail - 1) / avail;
    const long long jobs = (long long)((tiles_max + cl - 1) / cl) * MB;
    const long long cost = rounds * (2 * jobs + (cl == 1 ? 4 * MB : MB == 1 ? 5 : 8));
    if (sp.flat) {  // equal shares whatever the number of units: nothing to gain from more CTAs per unit
      best_cl = cl;
      best_cost = 0;
      break;
    }
    if (best_cost < 0 || cost < best_cost) {
      best_cost = cost;
      best_cl = cl;
    }
  }
  if (best_cost < 0) return cudaErrorLaunchOutOfResources;
  sp.cluster = best_cl;
  attr[0].val.clusterDim.x = (unsigned)best_cl;
  int n_clusters = max_clusters[best_cl];
  const long long pieces = sp.flat ? (long long)sp.units * tiles_max : sp.units;
  if (n_clusters > pieces) n_clusters = (int)pieces;
  ctx->score_cluster = sp.cluster;
  ctx->score_clusters = n_clusters;
  cfg.gridDim = dim3((unsigned)(n_clusters * sp.cluster), 1, 1);
  if (pdl) ta_pdl_attribute(&attr[cfg.numAttrs++]);
  return cudaLaunchKernelEx(&cfg, kern, mq, mk, sp);
}

// Ragged batches of more than kRankedSeqs sequences: the order of the units, longest sequences first.
__global__ void ta_unit_order_kernel(ta_seq_desc seq, int n_layers, int Hkv, int32_t* __restrict__ order) {
  const int b = blockIdx.x * blockDim.x + threadIdx.x;
  if (b >= seq.batch) return;
  const int nb = seq.cu[b + 1] - seq.cu[b];
  int rank = 0;
  for (int o = 0; o < seq.batch; ++o) {
    const int no = seq.cu[o + 1] - seq.cu[o];
    rank += (no > nb) || (no == nb && o < b);
  }
  const int per = n_layers * Hkv;
  for (int j = 0; j < per; ++j) {
    const int l = j / Hkv, g = j - l * Hkv;
    order[(long long)rank * per + j] = (l * seq.batch + b) * Hkv + g;
  }
}

// One warp that waits, with the bounded waits of the score kernel, on a barrier nothing ever completes: first the CTA-scope
// form, then (with the abort flag lowered again) the cluster-scope form. Nothing else is in flight.
__global__ void ta_wait_selftest_kernel(ta_dev_status* status, unsigned long long limit_ns, int* outcome) {
  __shared__ unsigned long long bar;
  __shared__ int abort_flag;
  if (threadIdx.x == 0) {
    mbar_init(smem_u32(&bar), 1);
    abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncwarp();
  volatile int* af = &abort_flag;
  const bool a = mbar_wait(smem_u32(&bar), 0, af, status, 90, limit_ns);
  __syncwarp();
  if (threadIdx.x == 0) abort_flag = 0;
  __syncwarp();
  const bool b = mbar_wait_cluster(smem_u32(&bar), 0, af, status, 91, limit_ns);
  if (threadIdx.x == 0 && outcome) *outcome = (a ? 1 : 0) | (b ? 2 : 0) | 4;  // 4: the kernel ran to its end
}

}  // namespace

cudaError_t ta_launch_wait_selftest(ta_dev_status* status, unsigned long long limit_ns, int* outcome,
                                    cudaStream_t stream) {
  ta_wait_selftest_kernel<<<1, 32, 0, stream>>>(status, limit_ns, outcome);
  return cudaGetLastError();
}

// A stride that multiplies a coordinate which is always 0 still has to be a valid tensor-map stride.
static uint64_t safe_stride(int64_t s, uint64_t dim) { return (dim <= 1 || s <= 0) ? 128 : (uint64_t)s; }

cudaError_t ta_launch_score(ta_ctx* ctx, const ta_score_args& a, ta_dev_status* status, cudaStream_t stream,
                            int* launches) {
  const int B = a.seq.batch, L = a.n_layers;
  const int units = L * B * a.Hkv;
  if (units == 0 || a.seq.total == 0) return cudaSuccess;
  const int G = a.Hq / a.Hkv;
  const int rows = G * a.W;
  const int MB = rows <= 128 ? 1 : 2;

  ScoreParams sp = {};
  sp.seq = a.seq;
  sp.n_layers = L;
  sp.Hq = a.Hq;
  sp.Hkv = a.Hkv;
  sp.G = G;
  sp.W = a.W;
  sp.rows = rows;
  sp.two_pass = a.lse_obs ? 0 : 1;
  sp.causal = a.causal;
  sp.flat = a.lse_obs && !a.seq.cu && ctx->score_force_cluster <= 0;
  const float scale = a.scale > 0.0f ? a.scale : 1.0f / sqrtf((float)kD);
  sp.c = scale * 1.4426950408889634f;
  sp.alpha = a.alpha;
  sp.delta = a.delta;
  sp.lse_obs = a.lse_obs;
  sp.A = a.A;
  sp.P = a.P;
  sp.u = a.u;
  sp.status = status;
  sp.wait_limit_ns = ta_wait_limit(ctx->wait_limit_ns);
  if (ctx->wrow_W != a.W || ctx->wrow_rho != a.rho) {  // 32 calls of pow() are a microsecond of host time
    for (int t = 0; t < a.W; ++t)
      ctx->wrow[t] = (float)((1.0 - (double)a.rho) * pow((double)a.rho, (double)(a.W - 1 - t)));
    ctx->wrow_W = a.W;
    ctx->wrow_rho = a.rho;
  }
  memcpy(sp.wrow, ctx->wrow, sizeof(float) * a.W);
  sp.units = units;
  sp.order = nullptr;
  sp.late_wait = a.pdl == 2;
  sp.by_length = a.seq.cu && B > 1 && B <= kRankedSeqs;
  if (a.seq.cu && a.order_scratch && B > kRankedSeqs) {
    ta_unit_order_kernel<<<(B + 127) / 128, 128, 0, stream>>>(a.seq, L, a.Hkv, a.order_scratch);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    sp.order = a.order_scratch;
    if (launches) ++*launches;
    sp.late_wait = 0;  // the order comes from the kernel before this one (which itself follows all before it)
  }
  if (launches) ++*launches;
  const int tiles_max = (a.seq.max_n + kTileN - 1) / kTileN;
  sp.cluster = 1;  // chosen at launch

  // tensor maps: dims (d, position, head, batch, layer)
  CUtensorMap mq, mk;
  {
    const uint64_t dims[5] = {(uint64_t)kD, (uint64_t)a.W, (uint64_t)a.Hq, (uint64_t)B, (uint64_t)L};
    const uint64_t str[4] = {safe_stride(a.q.stride_n, dims[1]), safe_stride(a.q.stride_h, dims[2]),
                             safe_stride(a.q.stride_b, dims[3]), safe_stride(a.q.stride_l, dims[4])};
    const uint32_t box[5] = {64, (uint32_t)a.W, (uint32_t)G, 1, 1};
    if (encode_5d(ctx->encode_tiled, &mq, a.q.ptr, dims, str, box) != CUDA_SUCCESS) return cudaErrorInvalidValue;
  }
  {
    const bool ragged = a.seq.cu != nullptr;
    const uint64_t dims[5] = {(uint64_t)kD, ragged ? (uint64_t)a.seq.total : (uint64_t)a.seq.n_uniform,
                              (uint64_t)a.Hkv, ragged ? 1ull : (uint64_t)B, (uint64_t)L};
    const uint64_t str[4] = {safe_stride(a.k.stride_n, dims[1]), safe_stride(a.k.stride_h, dims[2]),
                             safe_stride(a.k.stride_b, dims[3]), safe_stride(a.k.stride_l, dims[4])};
    const uint32_t box[5] = {64, (uint32_t)kTileN, 1, 1, 1};
    if (encode_5d(ctx->encode_tiled, &mk, a.k.ptr, dims, str, box) != CUDA_SUCCESS) return cudaErrorInvalidValue;
  }
  // Output form of pass 2. With only the weighted sum alpha*A + delta*P wanted and every row weight
  // alpha + delta*w_t positive, the weights go into the exponents and a key costs one sum (kOutFused); otherwise A
  // alone (kOutA) or A and P with per-row weights (kOutAP).
  bool fused = a.u != nullptr && a.A == nullptr && a.P == nullptr;
  for (int t = 0; fused && t < a.W; ++t) fused = a.alpha + a.delta * sp.wrow[t] > 0.0f;
  const bool need_p = a.P != nullptr || (a.u != nullptr && a.delta != 0.0f);
  if (MB == 1) {
    if (fused) return launch_variant<1, kOutFused>(ctx, mq, mk, sp, tiles_max, a.pdl, stream);
    if (need_p) return launch_variant<1, kOutAP>(ctx, mq, mk, sp, tiles_max, a.pdl, stream);
    return launch_variant<1, kOutA>(ctx, mq, mk, sp, tiles_max, a.pdl, stream);
  }
  if (fused) return launch_variant<2, kOutFused>(ctx, mq, mk, sp, tiles_max, a.pdl, stream);
  if (need_p) return launch_variant<2, kOutAP>(ctx, mq, mk, sp, tiles_max, a.pdl, stream);
  return launch_variant<2, kOutA>(ctx, mq, mk, sp, tiles_max, a.pdl, stream);
}
