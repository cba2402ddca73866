// Column and diagonal paths of a group of pairs on path planes (one chain per lane).
#include "agg_planar_shear.cuh"

namespace r2t {

cudaError_t launch_group_shear(PairGroup& g, const Method& mt, cudaStream_t s) {
  const int D = g.p[0].D;
  const int grid = set_prefix(
      g, [&](const Problem& p) { return planar_shear_pairs(p.W, p.D, mt.num_paths, 1); });
  return launch_planar_shear_t<1>(g, D, grid, mt, s);
}

}  // namespace r2t
