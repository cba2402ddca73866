// Column and diagonal paths on path planes: one instantiation per D / 16 and chains per lane, for a
// pair alone and for groups of pairs.
#pragma once
#include "planar.cuh"
#include "planar_group.h"

namespace r2t {

template <int NL, int CPL, class Src>
__global__ void __launch_bounds__(kPairThreads)
    planar_shear_kernel(const __grid_constant__ Src src, Method mt) {
  extern __shared__ __align__(16) uint8_t shm[];
  const bool back = threadIdx.x >= 32;
  int item = blockIdx.x;
  const Problem pb = src.locate(item);
  planar_shear<NL, CPL>(pb, mt, item, back, shm + (back ? planar_shear_smem(CPL) : 0));
  // this kernel starts beside the row kernel (after what precedes that one): it is complete only
  // when both are
  wait_prerequisites();
}

template <int CPL, class Src>
static cudaError_t launch_planar_shear_t(const Src& src, int D, int grid, const Method& mt,
                                         cudaStream_t s) {
  switch (D / 16) {
#define R2T_NL(N)                                                                    \
  case N:                                                                            \
    return launch_agg(planar_shear_kernel<N, CPL, Src>, grid, kPairThreads,          \
                      2 * planar_shear_smem(CPL), s, true, src, mt);
    R2T_NL(1) R2T_NL(2) R2T_NL(3) R2T_NL(4) R2T_NL(5) R2T_NL(6) R2T_NL(7) R2T_NL(8)
    R2T_NL(9) R2T_NL(10) R2T_NL(11) R2T_NL(12) R2T_NL(13) R2T_NL(14) R2T_NL(15) R2T_NL(16)
#undef R2T_NL
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace r2t
