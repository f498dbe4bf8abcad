// The tuner's candidate settings: the graph's own first, none twice, and the
// whole grid whatever the graph's own are.
#include <cstdio>

#include "tune_core.hpp"

using namespace gr;

static int failures = 0;
#define CHECK(x) \
  do { if (!(x)) { std::printf("line %d: %s\n", __LINE__, #x); ++failures; } } while (0)

template <class S>
static bool distinct(const std::vector<S> &v) {
  for (size_t i = 0; i < v.size(); ++i)
    for (size_t j = 0; j < i; ++j)
      if (v[i] == v[j]) return false;
  return true;
}

int main() {
  for (bool symmetric : {false, true})
    for (int32_t bps : {0, 1, 2, 3, 4}) {
      const auto v = bfs_settings({GR_MODE_AUTO, bps, GR_DIR_AUTO, 10.f, 24.f}, symmetric);
      CHECK((v[0] == BfsSetting{GR_MODE_PERSISTENT, bps, GR_DIR_AUTO, 10.f, 24.f}));
      CHECK(distinct(v));
      CHECK(v.size() == (symmetric ? 52u : 4u) + (symmetric && bps < 3 ? 0u : 1u));
      const auto g = bfs_settings({GR_MODE_GRAPH, bps, GR_DIR_PUSH, 14.f, 24.f}, symmetric);
      CHECK(g[0].mode == GR_MODE_GRAPH && distinct(g));
    }
  for (bool can_pull : {false, true})
    for (double factor : {2.0, 6.0, 8.0})
      for (int32_t bps : {0, 1, 3, 4})
        for (float alpha : {0.f, 3.f}) {
          const double mean = 32.5;
          const SsspSetting now{GR_MODE_PERSISTENT, bps, (uint32_t)(factor * mean), alpha};
          const auto v = sssp_settings(now, mean, can_pull);
          const bool known = factor != 6.0 && bps < 2 && alpha == 0.f;
          CHECK(v[0] == now);
          CHECK(distinct(v));
          CHECK(v.size() == (can_pull ? 72u : 24u) + (known ? 0u : 1u));
        }
  CHECK(sssp_settings({GR_MODE_GRAPH, 0, 1, 0.f}, 0.0, false)[1].delta >= 1u);
  if (!failures) std::printf("ok\n");
  return failures ? 1 : 0;
}
