// Which form a launch takes: the rules on sizes, types and alignment, host
// arithmetic alone in plain C++, so that they can be asked on any machine.
// Every rule states both sides as measured on GB300 (G x T: teams x threads).
#pragma once

#include <cstdint>

namespace rt {

// schedule(auto) 2-D stencil by strips of 64 columns a warp (k_stencil_cols.cu),
// for grids the tensor tiles do not take; the others run in the region kernel.
//   - Strips at least 0.4 full: the lanes beyond a narrow grid's columns idle
//     (608 x 256, region kernel -> strips: 1 x 2,494,174 7.4 -> 138 us, 5 x 355,331
//     6.9 -> 23.1, 11 x 131,295 6.1 -> 10.3, 21 x 20,920 3.2 -> 4.4; from there on
//     30 x 3078 on 52 x 128 4.1 -> 3.2, 33 x 56,391 7.2 -> 6.1, 57 x 89,460 on 313 x 32
//     182 -> 73, 89 x 25,585 8.4 -> 5.9).
//   - Four points a thread on, counted by the lanes in use: below, the region
//     kernel ends in a few rounds of loads (287 x 710 on 62 x 1024 3.1 -> 4.1, 34 x
//     649 on 58 x 128 2.0 -> 2.2, 69 x 11,986 4.3 -> 4.6; 153 x 475 on 50 x 256 2.8 ->
//     2.4).  On grids of 2^18 points with strips nearly full 1.8 are enough (217 x
//     5887 on 1158 x 512 6.8 -> 4.5, 6193 x 82 3.3 -> 2.7; at 1.7 points no difference).
//   - Row numbers and strips count in 32 bits.
constexpr uint32_t kStrip = 64;  // columns a warp
inline bool cols_applies(uint64_t nx, uint64_t ny, uint32_t teams, uint32_t threads) {
  const uint64_t strips = (nx + kStrip - 1) / kStrip;
  if (strips >= (1ull << 31) || ny >= (1ull << 31)) return false;
  const double full = (double)nx / ((double)strips * kStrip);
  const double points = (double)nx * (double)ny * full / ((double)teams * threads);
  const bool large = full >= 0.75 && nx * ny >= (1ull << 18);
  return full >= 0.4 && points >= (large ? 1.8 : 4.0);
}

}  // namespace rt
