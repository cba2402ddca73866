// Column and diagonal paths on path planes: one instantiation per lanes of a chain (D / 16), and per
// words per lane where a chain takes a warp, for a pair alone and for groups of pairs.
#pragma once
#include "planar.cuh"
#include "planar_group.h"

namespace r2t {

template <int NL, class Src>
__global__ void __launch_bounds__(kPairThreads, 16)  // 64 registers a thread
    planar_shear_kernel(const __grid_constant__ Src src, Method mt) {
  extern __shared__ __align__(16) uint8_t shm[];
  const bool back = threadIdx.x >= 32;
  int item = blockIdx.x;
  const Problem pb = src.locate(item);
  planar_shear<NL>(pb, mt, item, back, shm + (back ? planar_shear_smem() : 0));
  // this kernel starts beside the row kernel (after what precedes that one): it is complete only
  // when both are
  launch_dependents();
  wait_prerequisites();
}

template <int NW, bool FULL, class Src>
__global__ void __launch_bounds__(kPairThreads)
    planar_long_kernel(const __grid_constant__ Src src, Method mt) {
  extern __shared__ __align__(16) uint8_t shm[];
  const bool back = threadIdx.x >= 32;
  int item = blockIdx.x;
  const Problem pb = src.locate(item);
  planar_long<NW, FULL>(pb, mt, item, back, shm + (back ? planar_ring_smem(pb.D, 32) : 0));
  launch_dependents();
  wait_prerequisites();
}

template <class Src>
static cudaError_t launch_planar_shear_t(const Src& src, int D, int grid, const Method& mt,
                                         cudaStream_t s) {
  switch (D / 16) {
#define R2T_NL(N)                                                             \
  case N:                                                                     \
    return launch_agg(planar_shear_kernel<N, Src>, grid, kPairThreads,        \
                      2 * planar_shear_smem(), s, true, src, mt);
    R2T_NL(1) R2T_NL(2) R2T_NL(3) R2T_NL(4) R2T_NL(5) R2T_NL(6) R2T_NL(7) R2T_NL(8)
    R2T_NL(9) R2T_NL(10) R2T_NL(11) R2T_NL(12) R2T_NL(13) R2T_NL(14) R2T_NL(15) R2T_NL(16)
#undef R2T_NL
    default: return cudaErrorInvalidValue;
  }
}

template <int NW, class Src>
static cudaError_t launch_planar_long_w(const Src& src, int D, int grid, const Method& mt,
                                        cudaStream_t s) {
  return launch_agg(D == 64 * NW ? planar_long_kernel<NW, true, Src>
                                 : planar_long_kernel<NW, false, Src>,
                    grid, kPairThreads, 2 * planar_ring_smem(D, 32), s, true, src, mt);
}
template <class Src>
static cudaError_t launch_planar_long_t(const Src& src, int D, int grid, const Method& mt,
                                        cudaStream_t s) {
  switch (planar_long_words(D)) {
    case 1: return launch_planar_long_w<1>(src, D, grid, mt, s);
    case 2: return launch_planar_long_w<2>(src, D, grid, mt, s);
    default: return launch_planar_long_w<4>(src, D, grid, mt, s);
  }
}

}  // namespace r2t
