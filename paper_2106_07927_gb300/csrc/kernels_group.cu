// The stages of a group of pairs on path planes: one launch per stage, a block's pair found from its
// index.
#include "census_cost.cuh"
#include "planar.cuh"
#include "planar_group.h"
#include "post.cuh"

namespace r2t {

__global__ void __launch_bounds__(256)
    group_census_kernel(const __grid_constant__ PairGroup g, Method mt) {
  __shared__ CensusSmem sm;
  int item = blockIdx.x;
  const Problem pb = g.locate(item);
  census_tile_dispatch(pb, mt, item, sm);
}

__global__ void __launch_bounds__(256)
    group_cost_kernel(const __grid_constant__ PairGroup g, Method mt) {
  __shared__ CostSmem sm;
  int item = blockIdx.x;
  const Problem pb = g.locate(item);
  if (mt.cw == 9)
    cost_tile_planar<true>(pb, item, sm);
  else
    cost_tile_planar<false>(pb, item, sm);
}

template <int R>
__global__ void __launch_bounds__(256)
    group_wta_kernel(const __grid_constant__ PairGroup g, int paths, int T) {
  extern __shared__ __align__(16) uint8_t wsm[];
  int item = blockIdx.x;
  const Problem pb = g.locate(item);
  planar_wta_tile<R>(pb, paths, item, wsm, T);
}

__global__ void __launch_bounds__(256)
    group_median_kernel(const __grid_constant__ PairGroup g, Method mt) {
  __shared__ MedianSmem sm;
  int item = blockIdx.x;
  const Problem pb = g.locate(item);
  lr_median_tile<false, false>(pb, mt, item, sm);
}

template <int R>
static cudaError_t launch_wta(PairGroup& g, int paths, int T, cudaStream_t s) {
  const size_t smem = planar_wta_smem(g.p[0].D, T);
  cudaFuncSetAttribute(group_wta_kernel<R>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  const int grid = set_prefix(g, [&](const Problem& p) { return wta_items(p.W, p.H, T); });
  group_wta_kernel<R><<<grid, 256, smem, s>>>(g, paths, T);
  return cudaGetLastError();
}

cudaError_t run_group(PairGroup& g, const Method& mt, int row_dpl, int wta_px, cudaStream_t s) {
  int grid = set_prefix(g, [](const Problem& p) { return 2 * census_items(p.W, p.H); });
  group_census_kernel<<<grid, 256, 0, s>>>(g, mt);
  grid = set_prefix(g, [](const Problem& p) { return cost_items(p.W, p.H); });
  group_cost_kernel<<<grid, 256, 0, s>>>(g, mt);
  cudaError_t e = cudaGetLastError();
  if (e == cudaSuccess) e = launch_group_rows(g, mt, row_dpl, s);
  if (e == cudaSuccess) e = launch_group_shear(g, mt, s);
  const int T = planar_wta_px(g.p[0].D, wta_px);
  if (e == cudaSuccess) {
    switch (planar_planes(mt)) {
      case 8: e = launch_wta<8>(g, mt.num_paths, T, s); break;
      case 4: e = launch_wta<4>(g, mt.num_paths, T, s); break;
      default: e = launch_wta<2>(g, mt.num_paths, T, s);
    }
  }
  if (e != cudaSuccess) return e;
  grid = set_prefix(g, [](const Problem& p) { return median_items(p.W, p.H); });
  group_median_kernel<<<grid, 256, 0, s>>>(g, mt);
  return cudaGetLastError();
}

}  // namespace r2t
