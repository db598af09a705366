// How many blocks of the per-sequence kernel (ta_front.cu) share a sequence. Host code only.
#pragma once

constexpr int kFrontThreads = 1024;
constexpr int kFrontMaxItems = 16;    // tokens per thread
constexpr int kFrontMaxCluster = 16;  // blocks per sequence

// fit(cl): how many clusters of cl blocks the device holds at once, 0 when it holds none. 0: one kernel per step instead.
// One block holds up to 16384 tokens; more are worth their exchanges where a thread of one block would have more than 12 tokens, or
// has to. Of the sizes that hold the longest sequence the largest of which all sequences' clusters fit at once, else the smallest. How
// many fit depends on the GPU: B200s with 148 SMs hold 7 clusters of 16 blocks, 15 of 8, 33 or 35 of 4, 74 of 2. us per call of
// TA-Fast (one layer, one KV head) with separate kernels for mask, forced set and selection / 2 / 4 / 8 / 16 blocks:
//   1 x 131072 K 64 38.1 / - / - / 41.2 / 29.7; 4 x 131072 K 4096 57.1 / - / - / 46.1 / 35.4; 16 x 131072 109.6 / - / - / 78.5 / 82.6
//   4 x 65536 42.2 / - / 40.5 / 28.5 / 24.5; 8 x 32768 37.7 / 41.4 / 28.5 / 23.6 / 44.0; 60 x 32768 144.6 / 45.4 / 57.9 / 87.5 / 190
// and with one block / 2 / 4 / 8: 1 x 16384 26.3 / 25.7 / 19.3 / 16.9, 8 x 16384 27.5 / 26.8 / 20.5 / 18.2, 60 x 16384 31.7 / 31.1 /
// 41.6 / 66; 4 x 12000 18.5 / 25.6 / 19.4 / 17.6, 1 x 8192 14.7 / 21.7 / 18.0 / 16.6. Beside a score kernel (hidden), which hides it,
// one block leaves it the most SMs.
template <class Fit>
inline int ta_front_blocks(int n, int batch, int sms, bool hidden, Fit fit) {
  if (n > kFrontMaxCluster * kFrontMaxItems * kFrontThreads) return 0;
  if (n <= (hidden ? kFrontMaxItems : 12) * kFrontThreads) return 1;
  int least = 1;
  while (least * kFrontMaxItems * kFrontThreads < n) least *= 2;
  for (int cl = kFrontMaxCluster; cl > 1 && cl >= least; cl /= 2)
    if (batch <= sms / cl && batch <= fit(cl)) return cl;
  for (int cl = least; cl <= kFrontMaxCluster; cl *= 2)
    if (cl == 1 || fit(cl) > 0) return cl;
  return 0;
}
