// Which of several kernels, or which split, a call takes: functions of sizes alone, in plain C++.  They decide about speed and never
// about bits, so they may look at the rows of a forward.
#pragma once

namespace ssd {

// The rules that share work out take the machine's size from here; a grid of persistent CTAs asks the device.
constexpr int kSms = 148;

inline int ceil_div(long long a, long long b) { return (int)((a + b - 1) / b); }

// LM head in the dense kernel (256 rows x 256 entries to a pair of SMs, the statistics of a tile under the next tile's main loop)
// instead of the skinny one (row blocks of up to 256 x 128 entries, two CTAs to an SM).  Either works in turns: the dense kernel's
// take the same time whatever the rows, the skinny one's grow with them, and 97 rows are where they meet.  With a single turn
// there is no next tile.  us, skinny / dense, with the kernel that merges the tiles:
//   V 126464, d 4096 (without the merge)   160 rows 223 / 211, 192 246 / 220, 256 287 / 228, 512 497 / 402
//   V 65536 (2 turns against 4)            d 1024: 192 rows 59 / 65, 256 72 / 65, 512 126 / 84;  d 4096: 192 125 / 122, 256 146 / 122
//   V 50304 (2 against 3)                  d 1024: 192 rows 55 / 53, 256 64 / 55;  d 4096: 192 126 / 93, 256 142 / 95
//   V 32000 (1 against 2)                  d 1024: 192 rows 35 / 43, 256 39 / 42;  d 4096: 192 68 / 65, 256 75 / 66
//   V 2048  (1 against 1)                  d 1024: 192 rows 19 / 28, 512 27 / 29;  d 4096: 192 30 / 39, 512 40 / 43
// The smallest heads, whose weights are in the rings before the rows are there, gain by the shorter epilogue: V 2048, d 256: 192 rows
// 15.8 / 15.0, 256 18.7 / 15.0, 512 19.1 / 15.8; d 512: 192 rows 16.7 / 16.3, 256 19.7 / 16.7, 512 20.6 / 17.4.
inline bool lm_head_dense(int V, int K, int R) {
  const int pairs = kSms / 2, blocks = ceil_div(R, 256), block_rows = ceil_div(ceil_div(R, blocks), 16) * 16;
  const long long tiles = (long long)blocks * ceil_div(V, 256), skinny_tiles = (long long)blocks * ceil_div(V, 128);
  if (K <= 512 && 2 * tiles * K <= 256 * pairs) return true;
  const int turns = ceil_div(skinny_tiles, 2 * kSms);
  return turns >= 2 && 97 * ceil_div(tiles, pairs) <= turns * block_rows;
}

}  // namespace ssd
