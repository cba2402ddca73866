// Column and diagonal paths on path planes: one instantiation per D / 16 and chains per lane.
#include "launch.h"
#include "planar.cuh"

namespace r2t {

template <int NL, int CPL>
__global__ void __launch_bounds__(kPairThreads) planar_shear_kernel(Problem pb, Method mt) {
  extern __shared__ __align__(16) uint8_t shm[];
  const bool back = threadIdx.x >= 32;
  planar_shear<NL, CPL>(pb, mt, blockIdx.x, back, shm + (back ? planar_shear_smem(CPL) : 0));
  // this kernel starts beside the row kernel (after what precedes that one): it is complete only
  // when both are
  wait_prerequisites();
}

template <int CPL>
static cudaError_t launch_c(const Problem& pb, const Method& mt, cudaStream_t s) {
  const int grid = planar_shear_pairs(pb.W, pb.D, mt.num_paths, CPL);
  switch (pb.D / 16) {
#define R2T_NL(N)                                                                              \
  case N:                                                                                      \
    return launch_agg(planar_shear_kernel<N, CPL>, grid, kPairThreads,                         \
                      2 * planar_shear_smem(CPL), s, true, pb, mt);
    R2T_NL(1) R2T_NL(2) R2T_NL(3) R2T_NL(4) R2T_NL(5) R2T_NL(6) R2T_NL(7) R2T_NL(8)
    R2T_NL(9) R2T_NL(10) R2T_NL(11) R2T_NL(12) R2T_NL(13) R2T_NL(14) R2T_NL(15) R2T_NL(16)
#undef R2T_NL
    default: return cudaErrorInvalidValue;
  }
}

cudaError_t launch_planar_shear(const Problem& pb, const Method& mt, const Tuning& tn,
                                cudaStream_t s) {
  return tn.shear_cpl == 2 ? launch_c<2>(pb, mt, s)
                           : launch_c<1>(pb, mt, s);
}

}  // namespace r2t
