// Where gate+up on bf16 weights runs as one wave of tiles of more than 128 channels (host code, no CUDA headers).
#pragma once

#include <stdint.h>

namespace quasar {

// Channels of a tile for M rows, N channels in all (gate and up) and a contraction of K, or 0: tiles of at most 128, two on an SM.
// One wave of equal tiles loads all SMs alike, which tiles of 128 on 148 SMs do not, and its ring fills all the shared memory while
// the norm in front works; but it starts later and has no second CTA on the SM to work while it finishes its rows.
//
// What a layer of the pass takes against tiles of at most 128, in % (layers of 29 to 213 us; 8 to 24 of them on 1024 positions), at 1
// or 2 / 3 to 5 / 6 or 8 rows; N of 19,072 to 37,888:
//   K          144 channels     160              176              192              208              224              240              256
//   512        +4.9 +3.8 +4.5   +5.2 +4.1 +3.9   +4.4 +4.4 +3.8   +0.7 +0.2 -0.2   -0.8 +0.5 +0.8                    -2.1 -1.5 -1.8   -0.5 -0.8 -1.1
//   768-1280   +1.3 +0.9 +0.1   -0.4 -0.3 -1.2   -1.7 -2.5 -3.1   -1.5 -2.0 -2.2   -1.5 -1.9 -2.3   -1.9 -2.6 -3.4   -1.9 -2.0 -1.7   -0.7 -1.2 -1.9
//   1536-2560  +0.7 +0.1 +0.4   -0.5 -0.1 -0.3   -0.9 -0.3 +0.3   -0.5 +0.4 +0.9   +0.2 +0.7 +0.8   -0.3 -0.1 +0.2   +0.5 +0.6 +0.8   +1.2 +1.4 +1.4
//   3072       -1.0 -1.0 -0.7   -3.6 -1.7 -0.6   -1.9 -0.7 +0.2   -0.5 +0.3 +1.0   +0.5 +0.6 +0.7                    +0.2 +1.0 +1.0   +0.7 +1.0 +1.2
//   3584       -0.3 -0.6 -0.2   -0.3 -0.7 -0.3   -1.1 -0.9 -0.3   -0.6 -0.5 +0.3   -0.9 -0.8 -0.4   -0.8 -0.3 -0.1   -0.8 -0.5 -0.3   +0.5 +0.9 +0.9
//   4096       -3.7 -1.9  0.0   -3.4 -2.9 -0.6   -1.9 -1.2 -0.7   -1.0 -0.5 -0.3   -0.8 -0.6 -0.1   +1.1 +0.8 +1.1   +1.0 +0.8 +0.9   +0.3 +0.5 +0.8
//   4608-5120  -4.2 -3.3 -1.8   -4.7 -3.6 -2.4   -3.3 -2.3 -0.5   -2.0 -1.1 -0.2   -2.6 -2.3 -0.8   -1.0 -0.7 +0.1   +0.3 +0.6 +0.5   +0.7 +0.9 +1.0
//   6144-8192  -1.5 -0.5 -0.6   -2.7 -1.0 -0.3   -1.8 -0.9 +0.4   -1.1 -0.3 +0.3   -0.8 -0.4  0.0    0.0 +0.2 +0.2   -0.2 +0.1 +0.3   +0.1 -0.1 +0.1
// These are means over what stands around the layer (other numbers of kv heads, of layers, other places in memory), and that moves the
// tiles of 128 a lot: 24,576 x 5120 at 4 rows 99.0 -> 99.0 us among 10 kv heads and 8 layers, 102.0 -> 96.2 among 8 and 16.
// One size of them is no ground for a line.  With long contractions the busiest SM's share decides (208 channels instead of 256: a
// fifth less); with short ones the ring holds a good part of the tile before the layer starts, unless there is nearly no tile.
//
// More than 8 rows: 24,576 x 4096, a pass of 36 layers, at 1 row 3094 -> 3000 us, 8 rows 3086 -> 3063, 10 rows 3097 -> 3098, 12 rows
// 3111 -> 3127.
inline int dual_channels(int64_t M, int64_t N, int64_t K) {
  if (M < 1 || M > 8 || K < 768) return 0;
  const int64_t least = K < 3072 ? 160 : 144;
  const int64_t most = K <= 1280 ? 256 : K < 3584 ? 176 : 208;
  const int64_t c = ((N + 147) / 148 + 15) / 16 * 16;   // the narrowest tiles that 148 SMs take at once
  return c >= least && c <= most ? (int)c : 0;
}

}  // namespace quasar
