// How the rows of sweeps are split over the CTAs: host arithmetic without CUDA.
#pragma once

#include <algorithm>
#include <cstddef>
#include <vector>

namespace lbm {

// Shared lists of a sweep: the strips of every running case laid end to end and cut
// into one share per CTA slot, shares equal in rows plus the pipeline fill of each
// piece (the smallest such size for which the slots suffice, by bisection).  Item is
// {case, x0, first row, end row}; strips are whole (first row 0).  A piece has
// at least kLeast rows (rs divides them) and starts at a multiple of rs of its strip.  Piece k of share b stands at
// k * shares + b, empty pieces (first row = end row) where a share has fewer.  Returns the
// shares, 0 if the padded list does not fit in cap.
template <typename Item>
int share_out(const std::vector<Item> &strips, int rs, int slots, size_t cap, std::vector<Item> *out) {
  constexpr int kLeast = 8;
  const int fill = 3 * rs + rs * ((6 + rs - 1) / rs);
  long long rows = 0;
  for (const auto &s : strips) rows += s.y1;
  // pieces of each share of `size` rows with their fills
  auto cut = [&](long long size, std::vector<std::vector<Item>> *shares) {
    int used = 0;
    long long left = 0;  // of the current share
    for (const auto &s : strips) {
      int y = 0;
      while (y < s.y1) {
        if (used == 0 || left - fill < std::min(kLeast, s.y1 - y)) {
          ++used;
          left = size;
          if (shares) shares->emplace_back();
        }
        int len = (int)std::min<long long>(s.y1 - y, std::max<long long>(left - fill, kLeast));
        if (len < s.y1 - y) len -= len % rs;
        if (s.y1 - y - len < kLeast) len = s.y1 - y;  // no crumb for the next share
        if (shares) shares->back().push_back({s.case_id, s.x0, y, y + len});
        y += len;
        left -= len + fill;
      }
    }
    return used;
  };
  long long lo = 1, hi = rows + (long long)fill * (long long)strips.size() + fill + kLeast;  // hi: one share
  while (lo < hi) {
    const long long mid = (lo + hi) / 2;
    if (cut(mid, nullptr) <= slots) hi = mid;
    else lo = mid + 1;
  }
  std::vector<std::vector<Item>> shares;
  const int n = cut(hi, &shares);
  size_t deepest = 0;
  for (const auto &s : shares) deepest = std::max(deepest, s.size());
  if (n > slots || deepest * (size_t)n > cap) return 0;
  out->assign(deepest * (size_t)n, Item{0, 0, 0, 0});
  for (int b = 0; b < n; ++b)
    for (size_t k = 0; k < shares[b].size(); ++k) (*out)[k * (size_t)n + b] = shares[b][k];
  return n;
}

}  // namespace lbm
