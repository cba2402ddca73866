// Column and diagonal paths of a group of pairs on path planes.
#include <algorithm>

#include "agg_planar_shear.cuh"

namespace r2t {

cudaError_t launch_group_shear(PairGroup& g, const Method& mt, cudaStream_t s) {
  const int D = g.p[0].D;
  int64_t chains = 0;
  int wmin = g.p[0].W;
  bool flat = false;
  for (int i = 0; i < g.n; i++) {
    chains += 2 * planar_long_pairs(g.p[i].W, mt.num_paths);
    wmin = std::min(wmin, g.p[i].W);
    flat = flat || g.p[i].W > 2 * g.p[i].H;
  }
  if (planar_shear_dpl(chains, wmin, flat) == 8) {
    const int grid =
        set_prefix(g, [&](const Problem& p) { return planar_long_pairs(p.W, mt.num_paths); });
    return launch_planar_long_t(g, D, grid, mt, s);
  }
  const int grid =
      set_prefix(g, [&](const Problem& p) { return planar_shear_pairs(p.W, p.D, mt.num_paths); });
  return launch_planar_shear_t(g, D, grid, mt, s);
}

}  // namespace r2t
