// kx columns per block of the FP64 z pass.  Plain C++: a test compiles it for the host and
// compares its choices with measured times.
#pragma once

namespace bfcs {

// Busiest SM's share of the pass in columns, with blocks of T of them: blocks that share an
// SM share its FP64 pipe.
inline long long green_cost(int mx, int ny, int batch, int sms, int T) {
  const long long blocks = (long long)((mx + T - 1) / T) * ny * batch;
  return (blocks + sms - 1) / sms * T;
}

// 4 columns (64 bytes of a row), or 2 where the busiest SM then has less: 32^3 puts 160
// blocks of 4 on 152 SMs, so that 8 of them take two, and 288 blocks of 2 evenly.  A single
// column uses half of every 32-byte sector, so it has to save a fifth.  Whole sweeps in us
// with 4 / 2 / 1 columns (shares):
//   one:  24 x 32 x 128   117.2 / 117.8 / 111.5 (4, 4, 3), 48 x 48 x 24  81.1 / 73.7 / 69.4 (12, 10, 8)
//   two:  32^3  51.5 / 43.3 / 44.0 (8, 4, 4), 96^3  990 / 948 / 1004 (36, 32, 31), 96 x 96 x 48
//         462 / 452 / 505, 256^3  16.41 / 16.06 / 16.17 ms (224, 220, 218), 8 members of 64^3
//         1677 / 1622 / 1744 (124, 116, 112)
//   four: 64^3  241 / 240 / 249 (16, 16, 14), 192 x 48 x 24  211 / 233 / 233 (32, 32, 31)
// Over 37 shapes the rule's choice is 0.5% slower than the fastest width in the mean, 4.5%
// at most; the least share alone chose one column for most lengths (nx / 2 + 1 is odd) and
// was 2.7% slower in the mean, 12% at most.
inline int green_cols_fp64(int mx, int ny, int batch, int sms) {
  const long long c4 = green_cost(mx, ny, batch, sms, 4), c2 = green_cost(mx, ny, batch, sms, 2),
                  c1 = green_cost(mx, ny, batch, sms, 1);
  const long long wide = c2 < c4 ? c2 : c4;
  if (5 * c1 <= 4 * wide) return 1;
  return c2 < c4 ? 2 : 4;
}

}  // namespace bfcs
