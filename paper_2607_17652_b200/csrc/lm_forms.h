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
// 768, where the epilogue bounds a tile, 0.96 and 1.00 at 22 / 21.  Calls with pairs over calls without:
//   row tiles                        2    4    6    7    8    9   11   12   13   15   16    rounds at 7, 9, 11, 13
//   hidden 2048, V = 151,552       .92  .90  .91 1.03  .88  .99  .98  .89  .97  .96  .89    8/7  10/9  48/44  56/52
//   hidden 2048, V = 32,000        .92  .89  .89  .99  .88  .97  .97  .91  .97  .96  .90    7/6   9/8  11/10  12/11
//   hidden 2048, V = 16,384        .99  .93  .90  .96  .89 1.03 1.00  .90  .98  .91  .90    4/4   5/4   6/5    7/6
//   hidden 4096, V = 23,296        .91  .88  .88  .90  .89 1.01 1.00  .90 1.00  .91  .90    5/5   7/6   8/7    9/8
//   hidden 768,  V = 151,552       .96  .95  .96 1.09  .97 1.06 1.05  .97 1.03 1.02  .96    as above
FB_HOST_DEVICE inline bool lm_pairs(int m_tiles, int n_tiles, int hidden, int sms) {
  const long long one = ((long long)m_tiles * n_tiles + sms - 1) / sms, per = sms / 2;
  const long long two = ((long long)((m_tiles + 1) / 2) * n_tiles + per - 1) / per;
  return m_tiles >= 2 && 100 * two <= (hidden >= 1024 ? 110 : 105) * one;
}

// lm_pairs for every count of live row tiles, a bit each; from 64 on all as pairs.  (The rule itself at the start of the
// kernels, two 64-bit divisions, took 1 us of a call.)
FB_HOST_DEVICE inline unsigned long long lm_pairs_mask(int n_tiles, int hidden, int sms) {
  unsigned long long mask = 0;
  for (int m = 0; m < 64; ++m) mask |= (unsigned long long)lm_pairs(m, n_tiles, hidden, sms) << m;
  return mask;
}
FB_HOST_DEVICE inline bool lm_pairs_of(unsigned long long mask, int m_tiles) { return m_tiles >= 64 || (mask >> m_tiles & 1); }

// Launch both forms?  The live rows are only known on the device, so a context that may take pairs launches both forms;
// the one that is turned down costs 0 to 3 us.  A call with pairs saves a tenth (below hidden 1024, where the epilogue
// bounds a tile, 3 to 4 %), so both are launched where the tiles that the context can hold, weighed by what a pair can
// save of them, are enough.  us of both forms against the one-CTA form alone, 24 row tiles of capacity, live 3 / 8 / 12 / 20:
//   hidden 768,  V = 32,000   (3,000 tiles):  +4  +2   +1   -1        not launched
//   hidden 1024, V = 23,296   (2,184 tiles):  +1   0   -2   -5
//   hidden 1024, V = 32,000   (3,000 tiles):  +2  -2   -4   -7
//   hidden 2048, V = 32,000   (3,000 tiles):   0 -11  -12  -21
//   hidden 768,  V = 151,552 (14,208 tiles):  +2  -4   -9  -19
//   hidden 2048, V = 151,552 (14,208 tiles):  +1 -55  -78 -136
FB_HOST_DEVICE inline bool lm_both_forms(int most_tiles, int n_tiles, int hidden, int sms) {
  const long long tiles = (long long)most_tiles * n_tiles;
  return sms >= 2 && most_tiles >= 4 && hidden >= 768 && tiles >= 8ll * sms && tiles * (hidden - 512) >= 1 << 20;
}

}  // namespace fb
