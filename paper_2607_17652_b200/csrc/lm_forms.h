// Which form of the LM head's product runs (lm_head.cu): one CTA a tile, or a pair of CTAs per two row tiles.
// Plain integer rules, shared by the host, the device and the tests.
#pragma once
#ifdef __CUDACC__
#define FB_HOST_DEVICE __host__ __device__
#else
#define FB_HOST_DEVICE
#endif

namespace fb {

constexpr int kLmBM = 128, kLmBN = 256;      // output tile: rows of x, vocabulary

// Row tiles two by two?  Both forms deal out their tiles in rounds over the SMs, one-CTA tiles `sms` at a time, pairs
// sms / 2, and an odd row tile leaves half of a pair idle.  A round of pairs takes 0.88 to 0.91 of a round of
// single tiles (hidden 1024 to 4096, four row tiles and more), a call with pairs 1.00 at 10 / 9 of the rounds; at hidden
// 768, where the epilogue bounds a tile, 0.96 and 1.03 at 13 / 12.  Calls with pairs over calls without:
//   row tiles                        2    4    6    7    8    9   11   12   13   15   16    rounds at 7, 9, 11, 13
//   hidden 2048, V = 151,552       .92  .90  .91 1.03  .88  .99  .98  .89  .97  .96  .89    8/7  10/9  48/44  56/52
//   hidden 2048, V = 32,000        .92  .89  .89  .99  .88  .97  .97  .91  .97  .96  .90    7/6   9/8  11/10  12/11
//   hidden 2048, V = 16,384        .99  .93  .90  .96  .89 1.03 1.00  .90  .98  .91  .90    4/4   5/4   6/5    7/6
//   hidden 4096, V = 23,296        .91  .88  .88  .90  .89 1.01 1.00  .90 1.00  .91  .90    5/5   7/6   8/7    9/8
//   hidden 768,  V = 151,552       .96  .95  .96 1.09  .97 1.06 1.05  .97 1.03 1.02  .96    as above
FB_HOST_DEVICE inline bool lm_pairs(int m_tiles, int n_tiles, int hidden, int sms) {
  const long long one = ((long long)m_tiles * n_tiles + sms - 1) / sms, per = sms / 2;
  const long long two = ((long long)((m_tiles + 1) / 2) * n_tiles + per - 1) / per;
  return m_tiles >= 2 && 100 * two <= (hidden >= 1024 ? 110 : 103) * one;
}

}  // namespace fb
