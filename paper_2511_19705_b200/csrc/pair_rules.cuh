// Host rules of the dense products on CTA pairs: the width of their tiles, and whether a product runs on them or on the tiled kernel.
#pragma once

namespace cafeq {

// Tile width of a product of M rows: waves of 74 pairs times the width; `least` at least.
inline int t2_width(int M, int N, int b_mn, double* cost, int least = 128) {
  const long long tm = (M + 255) / 256;
  int best = 0;
  double bc = 1e30;
  for (int bn = 256; bn >= least; bn -= b_mn ? 128 : 32) {
    const long long waves = (tm * ((N + bn - 1) / bn) + 73) / 74;
    const double c = (double)waves * (bn + 24);  // (+ the fixed part of a tile: first loads, epilogue)
    if (c < bc) { bc = c; best = bn; }
  }
  if (cost) *cost = bc;
  return best;
}

// Whether CTA pairs are the better choice for a product of the given order (2: three terms, 3: six); cost: t2_width's.
// Six terms always are: one launch over arrays that are loaded once, instead of two.  Three terms are where the contraction is
// long enough for the tile's fixed part (pairs do not overlap an epilogue with the next tile's products), or where the tiled kernel's
// tiles of 128 rows fill the chip badly (waves x width of both, the tiled one's weighted by what it loses to its operand traffic).
// Measured, tiled minus pairs in us, M x N: K 512 / 1024 / 1536 / 2048 / 3584
//   three terms  512 x 512: -2 / -1 / 1 / 5 / 11;  1024 x 1024: -4 / -1 / -4 / 3 / 7;  1024 x 2560: - / 14 / 21 / - / 56
//                2048 x 2048: -12 / -6 / -9 / -4 / 4;  2048 x 3584: -9 / -4 / -4 / 4 / 19;  3584 x 1536: -5 / 3 / 9 / 11 / 28
//                3584 x 3584: -17 / -8 / -8 / 4 / 22;  4608 x 4608: -26 / -14 / -6 / 10 / 43
//   six terms    256 x 256: 4 / 8 / 12 / 16 / 28;  1024 x 1024: 7 / 11 / 14 / 18 / 29;  2048 x 2048: 7 / 9 / 11 / 13 / 28
//                3584 x 3584: 22 / 32 / 40 / 48 / 71
inline bool t2_wanted(int M, int N, int K, int order, double cost) {
  if (order > 2 || K >= 2048) return true;
  if (K < 1024) return false;
  const long long mt = (M + 127) / 128;
  double tiled = 1e30;
  for (int bn : {256, 224, 128, 64}) {
    const long long tiles = mt * ((N + bn - 1) / bn);
    if (bn > 128 && tiles < 96) continue;
    const double c = (double)((tiles + 147) / 148) * ((bn == 64 ? 1.6 : bn == 128 ? 1.4 : 1.25) * bn + 24);
    if (c < tiled) tiled = c;
  }
  return tiled > 1.5 * cost;
}

}  // namespace cafeq
