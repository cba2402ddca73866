// Row paths on path planes: one instantiation per words per lane and lane count.
#include "planar.cuh"
#include "planar_group.h"

namespace r2t {

template <int NW, int LPL, bool FULL, class Src>
__global__ void __launch_bounds__(kPairThreads)
    planar_row_kernel(const __grid_constant__ Src src, Method mt) {
  // the sheared kernel's blocks follow as soon as every block here is past this wait, so what precedes
  // this kernel is complete for them too
  wait_prerequisites();
  launch_dependents();
  extern __shared__ __align__(16) uint8_t shm[];
  int item = blockIdx.x;
  const Problem pb = src.locate(item);
  const int y0 = item * (32 / LPL);
  if (threadIdx.x >= 32)
    planar_rows<NW, LPL, FULL, true>(pb, mt, y0, shm + planar_ring_smem(pb.D, LPL));
  else
    planar_rows<NW, LPL, FULL, false>(pb, mt, y0, shm);
}

// One launch of `grid` blocks over pairs with D disparities.
template <int NW, int LPL, class Src>
static cudaError_t launch_t(const Src& src, int D, int grid, const Method& mt, cudaStream_t s) {
  return launch_agg(D == 2 * NW * LPL ? planar_row_kernel<NW, LPL, true, Src>
                                      : planar_row_kernel<NW, LPL, false, Src>,
                    grid, kPairThreads, 2 * planar_ring_smem(D, LPL), s,
                    std::is_same<Src, OnePair>::value, src, mt);
}

template <class Src>
static cudaError_t launch_d(const Src& src, int D, int dpl, int grid, const Method& mt,
                            cudaStream_t s) {
  switch (dpl * 100 + long_lanes(D, dpl)) {
    case 208: return launch_t<1, 8>(src, D, grid, mt, s);
    case 216: return launch_t<1, 16>(src, D, grid, mt, s);
    case 232: return launch_t<1, 32>(src, D, grid, mt, s);
    case 408: return launch_t<2, 8>(src, D, grid, mt, s);
    case 416: return launch_t<2, 16>(src, D, grid, mt, s);
    case 432: return launch_t<2, 32>(src, D, grid, mt, s);
    case 808: return launch_t<4, 8>(src, D, grid, mt, s);
    case 816: return launch_t<4, 16>(src, D, grid, mt, s);
    case 832: return launch_t<4, 32>(src, D, grid, mt, s);
    default: return cudaErrorInvalidValue;
  }
}

cudaError_t launch_planar_rows(const Problem& pb, const Method& mt, const Tuning& tn,
                               cudaStream_t s) {
  const OnePair one{pb};
  return launch_d(one, pb.D, tn.agg_dpl, planar_row_warps(pb.H, long_lanes(pb.D, tn.agg_dpl)), mt,
                  s);
}

cudaError_t launch_group_rows(PairGroup& g, const Method& mt, int row_dpl, cudaStream_t s) {
  const int D = g.p[0].D, lpl = long_lanes(D, row_dpl);
  const int grid = set_prefix(g, [&](const Problem& p) { return planar_row_warps(p.H, lpl); });
  return launch_d(g, D, row_dpl, grid, mt, s);
}

}  // namespace r2t
