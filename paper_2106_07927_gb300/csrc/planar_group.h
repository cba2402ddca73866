// A group of pairs of one disparity count, run by one launch per stage on path planes. The
// descriptors travel as the kernel's parameter (constant memory), so a batch uploads nothing.
#pragma once
#include <cuda_runtime.h>

#include "common.cuh"
#include "launch.h"

namespace r2t {

constexpr int kGroupPairs = 32;

// A pair alone: its blocks are the items.
struct OnePair {
  Problem p;
  __device__ __forceinline__ const Problem& locate(int&) const { return p; }
};
// Items of pair i are the blocks [prefix[i], prefix[i + 1]).
struct PairGroup {
  int n;
  int prefix[kGroupPairs + 1];
  Problem p[kGroupPairs];
  __device__ __forceinline__ Problem locate(int& item) const {
    int lo = 0, hi = n - 1;  // largest i with prefix[i] <= item
    while (lo < hi) {
      const int mid = (lo + hi + 1) >> 1;
      if (prefix[mid] <= item)
        lo = mid;
      else
        hi = mid - 1;
    }
    item -= prefix[lo];
    return p[lo];
  }
};
static_assert(sizeof(PairGroup) + sizeof(Method) <= 32764, "kernel parameters");

// Launches of a group (the pairs' D, row_dpl and tile are equal); each sets g.prefix for its stage.
cudaError_t launch_group_rows(PairGroup& g, const Method& mt, int row_dpl, cudaStream_t s);
cudaError_t launch_group_shear(PairGroup& g, const Method& mt, cudaStream_t s);
// Census, cost, both aggregation kernels, selection and LR check + median: 6 launches.
cudaError_t run_group(PairGroup& g, const Method& mt, int row_dpl, int wta_px, cudaStream_t s);

// Sets the prefixes to the pairs' items; returns the grid.
template <class F>
inline int set_prefix(PairGroup& g, F items) {
  int total = 0;
  for (int i = 0; i < g.n; i++) {
    g.prefix[i] = total;
    total += items(g.p[i]);
  }
  g.prefix[g.n] = total;
  return total;
}

}  // namespace r2t
