// Which widths (cells per thread block) of a cell kernel are worth timing.
#pragma once
#include <algorithm>
#include <array>
#include <cstdint>
#include <utility>
#include <vector>

namespace sipg {

// What a width setting launches on a level: the kernels round it to what they
// lay out (a thread limit, bricks of cells), so several settings are one launch.
struct TileLaunch {
  int cells, threads;   // of a block
  int64_t blocks;       // of the level
  bool operator==(const TileLaunch &o) const {
    return cells == o.cells && threads == o.threads && blocks == o.blocks;
  }
};

// The default width of a level: that of the kernel, lowered on meshes that would
// give fewer blocks than SMs, so that every SM gets cells (GB300 runs two FP64
// FMAs per clock per SM: an FP64 pass over 64 cells in 4 blocks of 16 would use 4
// of the 152 SMs).
inline int default_width(int cb, int64_t ncells, int nsm) {
  if (nsm > 0 && (ncells + cb - 1) / cb < nsm) cb = (int)std::max<int64_t>(1, (ncells + nsm - 1) / nsm);
  return cb;
}

// What a timed choice depends on.  The blocks of axis-aligned cells are cut from
// the mesh's sides (64 x 64 x 1 and 16^3 cells take other bricks), the others
// from the cells in a row.
inline std::array<int64_t, 8> tune_key(int n, bool curved, int precision, int pass, int64_t ncells, const int m[3]) {
  std::array<int64_t, 8> k{n, curved, precision, pass, ncells, 0, 0, 0};
  for (int d = 0; d < 3; ++d) k[5 + d] = curved ? 0 : m[d];
  return k;
}

// The launch of the level's default setting, then up to keep others among the
// settings 1 .. most whose waves of blocks leave the fewest cell slots idle,
// weighted by the share of live lanes in the block's last warp; each launch once,
// named by the cells its blocks take (which as a setting gives it again).
// launch(cb): the TileLaunch of a setting; resident(t): its blocks per SM.
template <typename Launch, typename Resident>
std::vector<int> pick_widths(int standard, int most, int64_t ncells, int nsm, int keep, Launch launch, Resident resident) {
  std::vector<TileLaunch> seen{launch(standard)};
  std::vector<std::pair<double, int>> score;
  for (int cb = 1; cb <= most; ++cb) {
    const TileLaunch t = launch(cb);
    if (std::find(seen.begin(), seen.end(), t) != seen.end()) continue;
    seen.push_back(t);
    const int64_t slots = (int64_t)resident(t) * nsm;
    if (slots <= 0) continue;
    const int64_t waves = (t.blocks + slots - 1) / slots;
    const double lanes = t.threads / (32.0 * ((t.threads + 31) / 32));
    score.push_back({(double)ncells / ((double)waves * slots * t.cells) * lanes, t.cells});
  }
  std::stable_sort(score.begin(), score.end(), [](const auto &x, const auto &y) { return x.first > y.first; });
  std::vector<int> out{seen[0].cells};
  for (size_t i = 0; i < score.size() && (int)i < keep; ++i) out.push_back(score[i].second);
  return out;
}

}  // namespace sipg
