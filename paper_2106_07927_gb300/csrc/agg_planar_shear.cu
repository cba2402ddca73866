// Column and diagonal paths of a pair alone on path planes.
#include "agg_planar_shear.cuh"

namespace r2t {

cudaError_t launch_planar_shear(const Problem& pb, const Method& mt, const Tuning& tn,
                                cudaStream_t s) {
  const OnePair one{pb};
  if (tn.shear_dpl == 8 && pb.W >= kRowChunk)
    return launch_planar_long_t(one, pb.D, planar_long_pairs(pb.W, mt.num_paths), mt, s);
  return launch_planar_shear_t(one, pb.D, planar_shear_pairs(pb.W, pb.D, mt.num_paths), mt, s);
}

}  // namespace r2t
