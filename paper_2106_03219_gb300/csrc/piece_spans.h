// Which bytes of the grid a lane of the 2-D stencil's piece form fetches
// (k_stencil_pieces.cu): index arithmetic alone, plain C++, so that it can be
// enumerated on the host.
//
// A lane's row is the grid's elements [row, row + RE), row a multiple of RE, of
// which [j0, j1) are its own.  Three spans are fetched in 16-byte units: the
// centre at row, the one above at row - up and the one below at row + down, up
// and down being nx rounded up and down to multiples of 4 (up = nx + sn, down = nx -
// ss).  A unit of the span above is fetched whole: from two columns on it ends inside
// the array.  On grids one column wide it would not, but there every point is on the
// border and copied, and nothing above is fetched.  Unit k4 of a span starts k4
// elements into it, k4 = 0, 4, .. RE; where a span leaves the grid, nothing is fetched
// before its first element or after its last.
#pragma once

#include <cstdint>

#include "host_device.h"

namespace rt {

// The distance up; on grids one column wide beyond any row.  (Bounding each unit above
// instead costs the slab's chain up to 6 % of the time of a launch of few warps.)
RT_HD uint64_t piece_up(uint64_t nx) { return nx == 1 ? 1ull << 62 : (nx + 3) / 4 * 4; }

// How far into each span the grid reaches, in elements, at most RE + 8 (so that
// a byte holds each): the centre's [0, ce), above from ab on, below [0, be).
struct PieceSpans {
  uint32_t ce, ab, be;
};
template <uint32_t RE>
RT_HD PieceSpans piece_spans(uint64_t row, uint64_t n, uint64_t up, uint64_t down) {
  constexpr uint32_t kTop = RE + 8;
  const uint64_t b = row + down;  // row <= n
  PieceSpans s;
  s.ce = n - row < kTop ? (uint32_t)(n - row) : kTop;
  s.ab = row >= up ? 0u : up - row < kTop ? (uint32_t)(up - row) : kTop;
  s.be = b >= n ? 0u : n - b < kTop ? (uint32_t)(n - b) : kTop;
  return s;
}

// Bytes of unit k4 inside the first `end` > k4 elements of its span.
RT_HD uint32_t unit_bytes(uint32_t k4, uint32_t end) {
  const uint32_t b = (end - k4) * 4;
  return b < 16u ? b : 16u;
}
// Whether unit k4 < RE is fetched: where one of the lane's points [j0, j1) reads it
// and the grid reaches into it.  The centre's also holds the points' neighbours west
// and east.  (A test and a length each, not the length alone, and the whole test in
// one place: the copies stay straight-line code with a predicate, 10 % faster than
// branches round them.)
RT_HD bool centre_fetched(uint32_t k4, uint32_t j0, uint32_t j1, uint32_t ce) {
  return j0 < j1 && k4 <= j1 && k4 + 4 >= j0 && k4 < ce;
}
RT_HD bool above_fetched(uint32_t k4, uint32_t j0, uint32_t j1, uint32_t sn, uint32_t ab) {
  return j0 < j1 && k4 < j1 + sn && k4 + 4 > j0 + sn && k4 >= ab;
}
RT_HD bool below_fetched(uint32_t k4, uint32_t j0, uint32_t j1, uint32_t ss, uint32_t be) {
  return j0 < j1 && k4 < j1 + ss && k4 + 4 > j0 + ss && k4 < be;
}
// The same of unit RE, for a lane that has points: their end alone decides.
RT_HD bool centre_edge(uint32_t re, uint32_t j1, uint32_t ce) { return j1 == re && ce > re; }
RT_HD bool above_edge(uint32_t re, uint32_t j1, uint32_t sn, uint32_t ab) {
  return j1 + sn > re && ab <= re;
}
RT_HD bool below_edge(uint32_t re, uint32_t j1, uint32_t ss, uint32_t be) {
  return j1 + ss > re && be > re;
}

}  // namespace rt
