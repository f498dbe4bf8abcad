// The settings that gr_autotune times (host only, no CUDA): the graph's own
// ones first, so that tuning never ends with slower ones than it began with,
// then the rest of the grid.
#pragma once

#include <stdint.h>

#include <algorithm>
#include <vector>

#include "gr.h"

namespace gr {

struct BfsSetting {
  int32_t mode, bps, dir;  // driver, blocks per SM (0: all resident), direction
  float alpha, beta;       // push -> pull and pull -> push thresholds
  bool operator==(const BfsSetting &o) const {
    return mode == o.mode && bps == o.bps && dir == o.dir && alpha == o.alpha && beta == o.beta;
  }
};

struct SsspSetting {
  int32_t mode, bps;
  uint32_t delta;  // bucket width
  float alpha;     // relaxations pull at m / alpha frontier edges (0: never)
  bool operator==(const SsspSetting &o) const {
    return mode == o.mode && bps == o.bps && delta == o.delta && alpha == o.alpha;
  }
};

// `now` first, then `rest` without it.
template <class S>
std::vector<S> with_present_first(const S &now, const std::vector<S> &rest) {
  std::vector<S> out{now};
  for (const S &s : rest)
    if (!(s == now)) out.push_back(s);
  return out;
}

inline std::vector<BfsSetting> bfs_settings(BfsSetting now, bool symmetric) {
  if (now.mode == GR_MODE_AUTO) now.mode = GR_MODE_PERSISTENT;  // what AUTO runs
  std::vector<BfsSetting> all;
  auto add = [&](int32_t dir, float al, float be) {
    for (int32_t bps : {1, 2, 0}) all.push_back({GR_MODE_PERSISTENT, bps, dir, al, be});
    all.push_back({GR_MODE_GRAPH, 0, dir, al, be});
  };
  add(GR_DIR_PUSH, 14.f, 24.f);  // thresholds unused without pull
  if (symmetric)
    for (float al : {4.f, 10.f, 14.f, 40.f})
      for (float be : {8.f, 24.f, 64.f}) add(GR_DIR_AUTO, al, be);
  return with_present_first(now, all);
}

// can_pull: the rows hold the in-edges and their weights, and are not a mesh's;
// the frontier holding half or a sixth of the edges is then tried as the
// threshold.
inline std::vector<SsspSetting> sssp_settings(const SsspSetting &now, double mean_weight,
                                              bool can_pull) {
  const double mw = std::max(1.0, mean_weight);
  std::vector<uint32_t> deltas;
  for (double f : {0.5, 1.0, 2.0, 4.0, 8.0, 32.0, 64.0})
    deltas.push_back((uint32_t)std::max(1.0, std::min(4.0e9, f * mw)));
  deltas.push_back(UINT32_MAX);  // a single bucket
  std::vector<float> alphas = {0.f};
  if (can_pull) alphas.insert(alphas.end(), {2.f, 6.f});
  std::vector<SsspSetting> all;
  for (uint32_t d : deltas)
    for (float al : alphas) {
      all.push_back({GR_MODE_GRAPH, 0, d, al});
      all.push_back({GR_MODE_PERSISTENT, 1, d, al});
      all.push_back({GR_MODE_PERSISTENT, 0, d, al});
    }
  return with_present_first(now, all);
}

}  // namespace gr
