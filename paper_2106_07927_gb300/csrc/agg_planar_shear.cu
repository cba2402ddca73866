// Column and diagonal paths of a pair alone on path planes.
#include "agg_planar_shear.cuh"

namespace r2t {

cudaError_t launch_planar_shear(const Problem& pb, const Method& mt, const Tuning& tn,
                                cudaStream_t s) {
  const OnePair one{pb};
  const int cpl = tn.shear_cpl == 2 ? 2 : 1;
  const int grid = planar_shear_pairs(pb.W, pb.D, mt.num_paths, cpl);
  return cpl == 2 ? launch_planar_shear_t<2>(one, pb.D, grid, mt, s)
                  : launch_planar_shear_t<1>(one, pb.D, grid, mt, s);
}

}  // namespace r2t
