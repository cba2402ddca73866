// Row paths on path planes: one instantiation per words per lane and lane count.
#include "launch.h"
#include "planar.cuh"

namespace r2t {

template <int NW, int LPL, bool FULL>
__global__ void __launch_bounds__(kPairThreads) planar_row_kernel(Problem pb, Method mt) {
  launch_dependents();  // the sheared kernel's blocks follow as soon as every block here runs
  extern __shared__ __align__(16) uint8_t shm[];
  const int y0 = blockIdx.x * (32 / LPL);
  if (threadIdx.x >= 32)
    planar_rows<NW, LPL, FULL, true>(pb, mt, y0, shm + planar_row_smem(NW));
  else
    planar_rows<NW, LPL, FULL, false>(pb, mt, y0, shm);
}

template <int NW, int LPL>
static cudaError_t launch_t(const Problem& pb, const Method& mt, cudaStream_t s) {
  return launch_agg(pb.D == 2 * NW * LPL ? planar_row_kernel<NW, LPL, true>
                                         : planar_row_kernel<NW, LPL, false>,
                    planar_row_warps(pb.H, LPL), kPairThreads, 2 * planar_row_smem(NW), s, false,
                    pb, mt);
}

cudaError_t launch_planar_rows(const Problem& pb, const Method& mt, const Tuning& tn,
                               cudaStream_t s) {
  switch (tn.agg_dpl * 100 + long_lanes(pb.D, tn.agg_dpl)) {
    case 208: return launch_t<1, 8>(pb, mt, s);
    case 216: return launch_t<1, 16>(pb, mt, s);
    case 232: return launch_t<1, 32>(pb, mt, s);
    case 408: return launch_t<2, 8>(pb, mt, s);
    case 416: return launch_t<2, 16>(pb, mt, s);
    case 432: return launch_t<2, 32>(pb, mt, s);
    case 808: return launch_t<4, 8>(pb, mt, s);
    case 816: return launch_t<4, 16>(pb, mt, s);
    case 832: return launch_t<4, 32>(pb, mt, s);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace r2t
