// How the rows of sweeps are split over the CTAs: host arithmetic without CUDA.
#pragma once

#include <algorithm>
#include <cstddef>
#include <vector>

namespace lbm {

// Segment length for a strip count: the number of segments per strip that
// minimises the rows the slowest CTA sweeps, waves x (segment rows + the
// pipeline fill of fill rows), with the rows of a strip split evenly (a multiple of
// rs each, the last segment the shortest); the fewest segments among equals.  Segments are the
// shorter the more of them a number of waves holds, so one candidate per number of waves
// is enough, up to the waves of which the fills alone cost as much as the best.  Every launch asks
// for it, and lbm_create for up to seven shapes.  With a walk over every number of segments
// lbm_create took 269 us at 2048 x 4096 and 711 us at 1 x 50000, with this one 217 and 53 us (GB300,
// Grace host; 215 and 51 us of it clear the arena).
inline int choose_segment(int ny, int strips, int resident, int rs, int fill) {
  int best_len = ny;
  long long best_cost = -1;
  const long long most = (ny + rs - 1) / rs;  // segments
  for (long long waves = (strips + resident - 1) / resident; best_cost < 0 || waves * (rs + fill) < best_cost; ++waves) {
    const long long nseg = std::min(most, waves * resident / strips);
    int len = (int)((ny + nseg - 1) / nseg);
    len = (len + rs - 1) / rs * rs;
    // (rounding the length up may leave fewer segments, and waves)
    const long long total = (ny + len - 1) / len * (long long)strips;
    const long long cost = (total + resident - 1) / resident * (len + fill);
    if (best_cost < 0 || cost < best_cost) {
      best_cost = cost;
      best_len = len;
    }
    if (nseg == most) break;
  }
  return best_len;
}

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
