// Where gate+up on bf16 weights runs as one wave of tiles of more than 128 channels (host code, no CUDA headers).
#pragma once

#include <stdint.h>

namespace quasar {

constexpr int kDualMaxChannels = 208;

// Channels of a tile for M rows, N channels in all (gate and up) and a contraction of K, or 0: tiles of at most 128, two on an SM.
// One wave of equal tiles loads all SMs alike, which tiles of 128 on 148 SMs do not, and its ring fills all the shared memory while
// the norm in front works; but it starts later and has no second CTA on the SM to work while it finishes its rows.  Measured in
// passes of 8 layers on 1024 positions, us a layer against tiles of at most 128 (layers of 57 to 125 us), at 1 / 3 / 5 / 8 rows
// (K of 4096 and 5120: 1 / 2 / 4 / 8); N of 19,072, 22,016, 24,576, 27,648 or 28,672, 34,816, 37,888:
//   K     144 channels         160                  176                 192 or 208          240                  256
//   3072  +.4 +.4 +.5 +.6      -1.0 -.7 -.6 -.2     -.6 -.4 -.2 -.1     -.2 +.2 +.3 +.3     -.4 +.6 +.5 +.7      +.6 +.7 +.8 +1.0
//   3584   0 -.1 -.7 -.5       -1.1 -1.3 -1.0 -.8   -1.1 -1.0 -.8 -.2   -.7 -.5 -.4 0       -.3 -.2 +.2 +.2      +.5 +1.1 +1.0 +1.2
//   4096  -3.6 -3.4 -1.7 0     -3.5 -2.7 -1.6 -.9   -1.1 -1.4 -1.1 -.6  -1.4 -1.6 -1.2 -.5  +1.7 +1.6 +1.9 +1.3   0 +.9 +.5 +.7
//   4608  -1.5 -1.1 -.8 -.7    -3.4 -1.5 -.8 -.6    -4.4 -1.4 -.1 +.3   -2.9 -.7 +.7 +.7    -.1 0 +.3 +.3        +.6 +.7 +.7 +.9
//   5120  -1.8 -2.0 -1.7 -1.6  -2.1 -1.3 -.5 -.3    -1.7 -1.2 0 +1.0    -2.3 -1.5 -.1 +1.3  +.7 +1.3 +1.4 +.7    +.7 +1.2 +1.3 +1.1
// So it is taken where it won: for contractions of some 4096 and up to 208 channels, where the busiest SM has a fifth less to do;
// for longer ones only with few rows to finish.  Below, 2048: +.5 at 144 channels, -.5 at 176, +.8 at 256; only layers whose FFN is
// ten times as wide as their input gained again (K of 768 to 1280, 176 channels and more: up to -1.7).  6144: -3.7 to +2.4 without
// a pattern; 8192: -1.4 at 144 channels, +.6 at 176, of 150.  More than 8 rows: 24,576 x 4096, a pass of 36 layers, at 1 row
// 3094 -> 3000, 8 rows 3086 -> 3063, 10 rows 3097 -> 3098, 12 rows 3111 -> 3127.
inline int dual_channels(int64_t M, int64_t N, int64_t K) {
  if (M < 1 || M > 8 || K < 3584 || K > (M <= 2 ? 5120 : M <= 4 ? 4608 : 4096)) return 0;
  const int64_t c = ((N + 147) / 148 + 15) / 16 * 16;   // the narrowest tiles that 148 SMs take at once
  return c > 128 && c <= kDualMaxChannels ? (int)c : 0;
}

}  // namespace quasar
