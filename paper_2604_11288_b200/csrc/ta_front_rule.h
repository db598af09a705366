// How many blocks of the per-sequence kernel (ta_front.cu) share a sequence. Host code only.
#pragma once

constexpr int kFrontThreads = 1024;
constexpr int kFrontMaxItems = 16;    // tokens per thread
constexpr int kFrontMaxCluster = 16;  // blocks per sequence

// fit(cl): how many clusters of cl blocks the device holds at once, 0 when it holds none. score_units: units of the score kernel that
// runs beside, 0 without one. selects: the kernel also searches the main pool (TA-Fast). 0: one kernel per step instead.
// One block holds up to 16384 tokens; more are worth their exchanges where a thread of one block would have more than 12 tokens, or
// has to. Of the sizes that hold the longest sequence the largest of which all sequences' clusters fit at once, else the smallest. How
// many fit depends on the GPU: B200s with 148 SMs hold 7 clusters of 16 blocks, 15 of 8, 33 or 35 of 4, 74 of 2. us per call of
// TA-Fast (one layer, one KV head) with separate kernels for mask, forced set and selection / 2 / 4 / 8 / 16 blocks:
//   1 x 131072 K 64 38.1 / - / - / 41.2 / 29.7; 4 x 131072 K 4096 57.1 / - / - / 46.1 / 35.4; 16 x 131072 109.6 / - / - / 78.5 / 82.6
//   4 x 65536 42.2 / - / 40.5 / 28.5 / 24.5; 8 x 32768 37.7 / 41.4 / 28.5 / 23.6 / 44.0; 60 x 32768 144.6 / 45.4 / 57.9 / 87.5 / 190
// and with one block / 2 / 4 / 8: 1 x 16384 26.3 / 25.7 / 19.3 / 16.9, 8 x 16384 27.5 / 26.8 / 20.5 / 18.2, 60 x 16384 31.7 / 31.1 /
// 41.6 / 66; 4 x 12000 18.5 / 25.6 / 19.4 / 17.6, 1 x 8192 14.7 / 21.7 / 18.0 / 16.6.
// 16 blocks where 8 leave a thread more than 4 tokens (8 / 16 blocks: 4 x 14000 17.7 / 18.2, 7 x 20000 19.8 / 20.4, 7 x 30000 22.3 /
// 23.4, 7 x 70000 31.7 / 25.6; beside a score kernel, 72 sizes of 1 to 7 sequences of 17000 to 32768 tokens, 1 to 112 units: 17 % faster
// to 4 % slower, 3 % faster on average: 4 x 17000, 8 units 41.5 / 46.1, 5 x 24000, 10 units 48.6 / 56.0, 1 x 17000, 8 units 41.2 / 42.9, 3 x
// 32768, 6 units 52.7 / 52.5, 2 x 24000, 16 units 91.3 / 87.4), or where nothing is searched and nothing runs beside (given scores, 8
// units a sequence: 1 x 13000 20.2 / 19.2, 1 x 20000 22.2 / 20.8, 4 x 30000 32.0 / 29.5).
// Beside a score kernel, which hides the one block of up to 16384 tokens, that leaves it the most SMs. Longer ones gain there too: 1
// to 100 sequences, 20000 to 131072 tokens, 1 to 384 units, 205 sizes with separate kernels and with this: 33 % faster to 1.5 % slower
// (4 x 40000, 8 units 73.9 / 66.6; 12 x 131072, 24 units 461.7 / 443.6; 4 layers of 4 x 40000 640 / 634).
// More than 131072 tokens need 16 blocks a sequence. Not worth it: where the last round would hold a single one (separate / 16 blocks:
// 7 x 140000 59.7 / 34.1, 8 x 140000 61.9 / 62.9, 12 x 140000 76.7 / 64.7, 15 x 200000 93.4 / 108.5, 18 x 200000 140.8 / 111.2; three
// rounds and more are always ahead), and where a score kernel of few units, one round of large clusters, does not find room beside those
// of about half the device (on one or the other of three GPUs: 3 x 140000, 24 units 434.7 / 466.2, 12 units 225.5 / 242.8; 4 x 200000,
// 8 units 243.4 / 268.2; with fewer or more sequences or units it is the other way round: 7 x 140000, 14 units 275.4 / 247.6; 4 x
// 140000, 16 units 413.0 / 406.2; 3 x 140000, 6 units 170.8 / 145.6).
template <class Fit>
inline int ta_front_blocks(int n, int batch, int sms, int score_units, bool selects, Fit fit) {
  if (n > kFrontMaxCluster * kFrontMaxItems * kFrontThreads) return 0;
  if (n <= (score_units > 0 ? kFrontMaxItems : 12) * kFrontThreads) return 1;
  int least = 1;
  while (least * kFrontMaxItems * kFrontThreads < n) least *= 2;
  if (least == kFrontMaxCluster) {
    const int at_once = fit(least);
    const bool lone = score_units == 0 && at_once > 1 && (batch == at_once + 1 || batch == 2 * at_once + 1);
    const bool crowded = 2 * batch >= at_once - 1 && 2 * batch <= at_once + 1 && score_units >= 8 && score_units <= (2 * batch < at_once ? 24 : 12);
    return at_once < 1 || lone || crowded ? 0 : least;
  }
  for (int cl = n <= 8 * 4 * kFrontThreads && (selects || score_units > 0) ? 8 : kFrontMaxCluster; cl > 1 && cl >= least; cl /= 2)
    if (batch <= sms / cl && batch <= fit(cl)) return cl;
  for (int cl = least; cl <= kFrontMaxCluster; cl *= 2)
    if (cl == 1 || fit(cl) > 0) return cl;
  return 0;
}
