// Prints what the plane kernels' host rules give, for tests/test_planar_schedule.py.
#include <stdio.h>

#include "../paper_2106_07927_gb300/csrc/planar.cuh"

using namespace r2t;

int main() {
  printf("const %d %d %d %d %d\n", kRowStages, kRowChunk, kPlanarRing, kShearGroup, kShearAhead);
  printf("shear_smem %d\n", planar_shear_smem());
  for (int W = 1; W < 60; W++) printf("mid %d %d\n", W, planar_row_mid(W));
  for (int D = 16; D <= 256; D += 16) {
    for (int lpl = 8; lpl <= 32; lpl *= 2) printf("ring %d %d %d\n", D, lpl, planar_ring_smem(D, lpl));
    for (int T = 64; T <= 256; T *= 2)
      printf("tile %d %d %d %zu\n", D, T, planar_wta_px(D, T), planar_wta_smem(D, planar_wta_px(D, T)));
    printf("words %d %d\n", D, planar_long_words(D));
    for (int nw = 1; nw <= 4; nw *= 2)
      for (int lig = 0; lig < 32; lig++)
        printf("at %d %d %d %d\n", D, nw, lig, planar_lane_at(lig, nw, D));
    for (int dpl = 2; dpl <= 8; dpl *= 2)
      if (D / dpl <= 32) printf("lanes %d %d %d\n", D, dpl, long_lanes(D, dpl));
  }
  const int shapes[][3] = {{160, 120, 8}, {320, 240, 8}, {320, 120, 8}, {413, 307, 8},
                           {1000, 375, 4}, {640, 375, 4}, {7, 9, 8}, {8, 9, 8}};
  for (auto& s : shapes)
    printf("shape %d %d %d %d\n", s[0], s[1], s[2],
           planar_shear_dpl(2 * planar_long_pairs(s[0], s[2]), s[0], s[0] > 2 * s[1]));
  return 0;
}
