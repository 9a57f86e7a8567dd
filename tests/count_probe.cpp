// A C shim for CPU tests: the load counts of the stream schedule beside the lists they count.
#include <algorithm>
#include <string>
#include <vector>

#include "tree.h"

// out: counted units of the four passes, counted most loads of a node, then the same from the lists;
// 0 on success.
extern "C" int probe_counts(const cfr_game_spec* spec, int pred, int32_t out[10]) {
  pcfr::HostGame g;
  std::string err;
  if (const int rc = pcfr::build_game(*spec, g, err)) return rc;
  int depth = 0, most_actions = 0;
  bool ok = false;
  const std::vector<int32_t> pre = pcfr::dfs_program(g, &depth, &most_actions, &ok);
  pcfr::stream_counts(g, pre, pred != 0, out, &out[4]);
  std::vector<uint32_t> units;
  int unit_off[4], chunk_off[4], chunk_count[4];
  pcfr::stream_tables(g, pre, 12, pred != 0, units, unit_off, &out[5], chunk_off, chunk_count);
  out[9] = 0;
  for (int n : pre)
    for (int p = 0; p < 2; ++p)
      out[9] = std::max(out[9], (int32_t)pcfr::node_loads(g, n, p, true, (uint32_t)g.hstride, pred != 0).size());
  return 0;
}
