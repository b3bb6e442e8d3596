// Tile widths of two rotations in one launch (host code without CUDA).
#pragma once
#include <algorithm>

namespace eogp {

// Tiles 0 .. n0 - 1 cost c0 each, the next n1 cost c1; round r of a CTA c of n is tile
// r n + c, in odd rounds r n + n - 1 - c. The cost of the CTA that ends last (n0, n1 >=
// 1). All rounds are full ones of one cost but the round in which the first kind ends
// and the last round; as a function of c the sum only changes where one of these does.
inline long long rotate_last_cta(long long n0, long long c0, long long n1, long long c1, int n) {
  const long long all = n0 + n1, mixed = n0 / n, last = (all - 1) / n;
  const auto at = [&](long long round, int c) {
    const long long t = round * n + (round & 1 ? n - 1 - c : c);
    return t < n0 ? c0 : t < all ? c1 : 0;
  };
  const long long full = mixed * c0 + std::max(0ll, last - mixed - 1) * c1;
  long long most = 0;
  const auto ends_at = [&](long long c) {
    if (c < 0 || c >= n) return;
    const int i = static_cast<int>(c);
    most = std::max(most, full + at(mixed, i) + (last > mixed ? at(last, i) : 0));
  };
  ends_at(0);
  ends_at(n - 1);
  const long long where[3][2] = {{mixed, n0 - mixed * n}, {mixed, all - mixed * n}, {last, all - last * n}};
  for (const auto& w : where)
    for (long long p = w[1] - 1; p <= w[1]; ++p) ends_at(w[0] & 1 ? n - 1 - p : p);
  return most;
}

// Widths bn[2] of the tiles of two sides with `rows` output columns and a reduction
// over K (the longer one first), M rows in tiles of 128: those whose last CTA ends
// first. A K block of a bn-column tile costs 2 bn cycles of the tensor pipe, at least
// ~220 in all.
inline void rotate_both_widths(const int (&rows)[2], const int (&K)[2], int M, int n, int (&bn)[2]) {
  long long best = -1;
  const int widest = std::max(rows[0], rows[1]);
  for (int parts = (widest + 255) / 256; best < 0 || parts <= (widest + 63) / 64; ++parts) {  // tiles of the wider side
    const int w = ((widest + parts - 1) / parts + 15) / 16 * 16;
    int b[2];
    long long cost[2], cnt[2];
    for (int i = 0; i < 2; ++i) {
      const int own = (rows[i] + w - 1) / w;
      b[i] = std::max(16, ((rows[i] + own - 1) / own + 15) / 16 * 16);
      cnt[i] = static_cast<long long>((M + 127) / 128) * ((rows[i] + b[i] - 1) / b[i]);
      cost[i] = static_cast<long long>((K[i] + 63) / 64) * std::max(2 * b[i], 220);
    }
    const long long last = rotate_last_cta(cnt[0], cost[0], cnt[1], cost[1], n) + 12 * w;
    if (best < 0 || last < best) {
      best = last;
      bn[0] = b[0];
      bn[1] = b[1];
    }
  }
}

}  // namespace eogp
