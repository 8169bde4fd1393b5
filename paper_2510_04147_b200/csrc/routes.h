// Which of several kernels, or which split, a call takes: functions of sizes alone, in plain C++.  They decide about speed and never
// about bits, so they may look at the rows of a forward.
#pragma once

#include <initializer_list>

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

// Evenly shared projections (gemm_wave.cu): the couples of a feature and its partner that make a unit, in as few turns as the width of an
// accumulator allows, one unit for every pair of SMs in each.
struct WaveShare { int turns, couples; };
inline WaveShare wave_share(int N) {
  const int pairs = kSms / 2;
  for (int turns = 1;; ++turns) {
    const int couples = (ceil_div(N / 2, (long long)pairs * turns) + 7) & ~7;
    if (couples <= 256) return {turns, couples < 16 ? 16 : couples};
  }
}

// Gate|up shared out evenly instead of in whole tiles (up to 256 rows): the features an SM has to do, in all turns of either.
// `dense`: the other kernel is the dense one, 256 features to a pair of SMs in a turn; else the skinny one, two tiles of 128 to an SM
// (one, where there are no more tiles than SMs).  One turn pays from a fifth less on, several, which have no other unit's
// main loop over their epilogue, from a ninth.  us, other / even, 192 rows and (dense) 256 rows, d 4096 unless said:
//   features 24576 (256 / 168)   47 / 39, 48 / 41      38912 (512 / 272 and 384 / 272)  88 / 68, 81 / 73
//   28672 (256 / 200)            50 / 47, 54 / 48      49152 (512 / 336, 384 / 336)     96 / 80, 83 / 83;  d 2048 52 / 42, 42 / 45
//   37888 (256 / 256)            57 / 57, 58 / 61      53248 (512 / 368, 384 / 368)     103 / 88, 86 / 90
//   1408, d 256 (128 / 16)       7.6 / 5.3, 6.7 / 5.4  67584 (512 / 464)                115 / 115, 115 / 110 (a forward of four layers 1049 / 1058, 1058 / 1093)
//   65536 (512 / 448)            112 / 105, 115 / 109  75776 (512 / 512)                121 / 121, 117 / 125
//   76800 (768 / 528, 640 / 528) 155 / 125, 146 / 134  90112, d 2048 (768 / 624, 640 / 624)  86 / 73, 67 / 74
inline bool gemm_wave_gains(int N, bool dense) {
  const int tiles = ceil_div(N, 128);
  const int other = dense ? ceil_div(ceil_div(N, 256), kSms / 2) * 128 : tiles <= kSms ? 128 : ceil_div(tiles, 2 * kSms) * 256;
  const WaveShare share = wave_share(N);
  return share.turns == 1 ? 4 * other >= 5 * share.couples : 8LL * other >= 9LL * share.turns * share.couples;
}

// CTAs that share the `parts` of the key tiles of each (query tile, head, sequence) in the tcgen05 attention, `work` of these in all: one
// for each part, one for two, or one for all of them.  An SM has one CTA and a GPC room for few clusters, so clusters take
// turns: in tenths of a us, a turn of CTAs with a part each costs 52 to 74 and 12 to 18 a tile (tiles of 32, 64 and 128 query rows),
// one of CTAs with several 32 to 64, 12 to 20 a tile (128 rows: scores are read twice there) and 15 to 24 where they have something to
// exchange.  Fitted to 730 sizes (4 to 60 heads, 2 to 33 tiles, 32 to 640 rows): the best choice within 3 % in all but 8.  us a launch with one CTA, with half as many as parts and with as many:
//   2 tiles in 2 parts, 128 rows      32 heads 14.3 / - / 11.1       5 tiles in 4 parts  32 heads, 32 rows 12.5 / 11.1 / 9.2
//   17 tiles in 2 parts, 512 rows     40 heads 79.0 / - / 67.5       160 rows            20.0 / 18.7 / 23.7
//   3 tiles in 3 parts, 256 rows      24 heads 17.3 / - / 21.3       17 in 8, 8 heads, 256 rows  43.2 / 23.1 / 28.0
inline int attn_pipe_ctas(int parts, int tiles, long long work, int query_rows) {
  constexpr int kClusters[9] = {0, kSms, kSms / 2, 45, 33, 24, 18, 15, 15};       // of as many CTAs that find an SM each
  const int at = query_rows <= 32 ? 0 : query_rows <= 64 ? 1 : 2;
  constexpr int kTurn[3] = {52, 59, 74}, kTile[3] = {12, 12, 18}, kTurnShared[3] = {32, 33, 64}, kTileShared[3] = {12, 14, 20}, kExchange[3] = {15, 22, 24};
  int ctas = parts;
  long long best = 0;
  for (const int n : {parts, parts / 2, 1}) {
    if (n < 1 || parts % n != 0) continue;
    const long long turns = ceil_div(work, kClusters[n < 8 ? n : 8]), tiles_each = ceil_div(tiles, n);
    const long long cost = n == parts ? 18 + turns * (kTurn[at] + kTile[at] * tiles_each)
                                      : 30 + turns * (kTurnShared[at] + kTileShared[at] * tiles_each + (n > 1 ? kExchange[at] : 0));
    if (best == 0 || cost < best) { best = cost; ctas = n; }
  }
  return ctas;
}

// O and down in the skinny kernel as pairs of tiles, whose clusters are twice as large (2 * splits CTAs).  A pair pays from 8 K
// blocks a split on (below, its set-up and the wider exchange outweigh half of the copies), and only where all clusters find
// room at once: of eight CTAs with an SM each the GPCs take 14 or 15, of CTAs that share an SM (more CTAs than SMs) twice that.
// 32 clusters of these still pay with long splits and blocks of up to 192 rows, the more the longer; with 416 rows they do not
// (57.2 / 60.3), and not where the kernel in front, which is of the same kind (`before` CTAs, two to an SM), fills half of the
// machine in its last turn: one place in every SM is free then, clusters are spread over those, and the last of them have to
// wait.  (Where it leaves most places free, or none, the clusters lie close.)  us, single tiles / pairs (28 tiles: d 3584, and so on), four splits:
//   K blocks each   128 rows       256 rows       288 rows       352 rows
//   8 tiles   4     8.5 / 9.1      12.2 / 13.1    9.2 / 9.8      9.7 / 10.3
//   20 tiles  8     9.9 / 9.9      14.6 / 15.0    15.9 / 15.5    19.7 / 16.7
//   24 tiles 12     11.4 / 11.4    16.2 / 16.4    19.1 / 18.4    23.7 / 20.2
//   24 tiles 32     17.8 / 17.3    24.8 / 24.0    27.3 / 24.9    34.8 / 27.6
//   28 tiles 74     30.0 / 29.1    43.4 / 38.6    47.7 / 42.3    64.8 / 47.1
//   16 tiles  4     8.2 / 8.9      12.4 / 13.0    10.2 / 20.1 (128 CTAs with an SM each: two turns)
//   32 tiles        24.7 / 43.1 (K 12288: 16 clusters)   12 each 19.8 / 20.5; 24 24.8 / 36.6; 32 28.5 / 28.1, 352 rows 36.2 / 29.0;
//                   48 36.0 / 33.2, 47.3 / 35.8; 74 49.4 / 44.9, 68.1 / 50.5.  Last turn 51 % full: 56 39.8 / 44, 384 rows 55 / 72;
//                   59 % (K 24576) 61 / 85, 88 / 105; 62 % (K 15360) 43 / 52, 57 / 71; 38 % (K 22528) 58 / 52, 82 / 71; 84 % (K 17408) 47 / 43, 65 / 54
inline bool residual_pairs(int tiles, int splits, int k_blocks, int row_blocks, int block_rows, int before) {
  const int ctas = tiles * splits * row_blocks, each = k_blocks / splits;
  const bool share = ctas > kSms;
  if (ctas <= (share ? 2 : 1) * 112) return each >= 8;
  const int last_turn = before % (2 * kSms) * 100 / (2 * kSms);        // per cent of the places
  return share && row_blocks > 1 && block_rows <= 192 && each >= 32 && (last_turn < 45 || last_turn >= 75);
}

}  // namespace ssd
