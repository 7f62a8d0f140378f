// schedule(auto) 2-D 5-point stencil on grids the tensor-copied tiles do not
// take: rows that are no whole number of 16-byte units, or arrays that do not
// start on one.
//
// The mapping is free, so a warp walks down a strip of 64 columns, lane l on
// columns l and l + 32: its loads and stores each cover 128 contiguous bytes at
// whatever alignment the grid gives, the rows above, at and below ride in
// registers (each point is loaded once a strip), the points west and east come
// from the neighbouring lanes by shuffle, and only the two columns beside the
// strip are loaded extra.  kAhead rows are on their way at any time.  One strip
// piece a warp, its height chosen so that the launch's warps all have one:
// short enough to fill the chip, as tall as that allows, since every piece
// reads two rows more than it writes.
//
// Before, odd grids ran point by point (five loads and a 64-bit row split a
// point: 62 % issue active).  3001 x 2503, 608 x 256: 24.8 -> 13.8 us (0.65 of the
// copy rate), 4095^2: 54.7 -> 28.7 (0.70).  128 columns and four rows fetched at
// a time, without a standing pipeline: 18.2 and 34.1; every column and row of
// every strip tested: 14.8 and 29.7 (72 % issue active).  What bounds it: issue
// (shuffles, selects), and pieces of 25 rows that start and end cold.
#include "launch_common.cuh"
#include "plan.h"

namespace rt {

struct ColsArgs {
  const float* in;
  float* out;
  uint64_t nx;
  uint32_t ny;
  float c0, c1;
  uint32_t strips;   // of kStrip columns
  uint32_t rows;     // rows a piece
  uint64_t pieces;
};

constexpr uint32_t kAhead = 5;   // rows in flight

// Rows [r0, r1) of the strip at col0.  kFull: the strip and the columns beside it
// are inner columns (all but the first and last strips), so no column is tested.
template <bool kFull>
__device__ __forceinline__ void walk_strip(const ColsArgs& A, uint64_t col0, uint32_t r0,
                                           uint32_t r1) {
  const uint32_t lane = lane_id();
  const uint64_t nx = A.nx;
  const uint32_t rl = r1 < A.ny ? r1 : A.ny - 1;  // the last row it reads
  // this lane's columns inside the grid, whether they are inner ones, and
  // the column it fetches beside the strip (lane 0 the one before it, lane
  // 31 the one after)
  const uint64_t left = nx - col0;
  const bool ok0 = kFull || lane < left, ok1 = kFull || lane + 32 < left;
  const bool in0 = kFull || ((lane || col0) && lane + 1 < left);
  const bool in1 = kFull || lane + 33 < left;
  const bool side = kFull ? lane == 0 || lane == 31
                          : (lane == 0 ? col0 > 0 : lane == 31 && kStrip < left);
  const int64_t beside = lane == 0 ? -1 : 33;
  const float* src = A.in + (uint64_t)r0 * nx + col0 + lane;
  float* out = A.out + (uint64_t)r0 * nx + col0 + lane;
  float u0 = 0.f, u1 = 0.f, d0[kAhead], d1[kAhead], de[kAhead];
  if (r0 > 0) {
    u0 = ok0 ? ld_nc(src - nx) : 0.f;
    u1 = ok1 ? ld_nc(src - nx + 32) : 0.f;
  }
  float c0 = ok0 ? ld_nc(src) : 0.f, c1 = ok1 ? ld_nc(src + 32) : 0.f;
  float edge = side ? ld_nc(src + beside) : 0.f;
  uint32_t q = r0;  // the last row on its way; past rl the last row comes again
  auto fetch = [&](uint32_t k) {
    if (q < rl) {
      src += nx;
      ++q;
    }
    d0[k] = ok0 ? ld_nc(src) : 0.f;
    d1[k] = ok1 ? ld_nc(src + 32) : 0.f;
    de[k] = side ? ld_nc(src + beside) : 0.f;
  };
#pragma unroll
  for (uint32_t k = 0; k < kAhead; ++k) fetch(k);
  auto row = [&](uint32_t k, bool inner) {
    // lane 0 gets lane 31's, lane 31 lane 0's
    const float w0 = __shfl_sync(0xffffffffu, c0, (lane + 31) & 31),
                w1 = __shfl_sync(0xffffffffu, c1, (lane + 31) & 31),
                e0 = __shfl_sync(0xffffffffu, c0, (lane + 1) & 31),
                e1 = __shfl_sync(0xffffffffu, c1, (lane + 1) & 31);
    const float wa = lane == 0 ? edge : w0, ea = lane == 31 ? e1 : e0;
    const float wb = lane == 0 ? w0 : w1, eb = lane == 31 ? edge : e1;
    const float a = __fmaf_rn(A.c1, __fadd_rn(__fadd_rn(u0, d0[k]), __fadd_rn(ea, wa)),
                              __fmul_rn(A.c0, c0));
    const float b = __fmaf_rn(A.c1, __fadd_rn(__fadd_rn(u1, d1[k]), __fadd_rn(eb, wb)),
                              __fmul_rn(A.c0, c1));
    if (ok0) out[0] = inner && in0 ? a : c0;
    if (ok1) out[32] = inner && in1 ? b : c1;
    out += nx;
    u0 = c0;
    u1 = c1;
    c0 = d0[k];
    c1 = d1[k];
    edge = de[k];
    fetch(k);
  };
  uint32_t r = r0;
  for (; r + kAhead <= r1; r += kAhead) {
    const bool mid = r > 0 && r + kAhead < A.ny;  // no boundary row among them
    if (mid) {
#pragma unroll
      for (uint32_t k = 0; k < kAhead; ++k) row(k, true);
    } else {
#pragma unroll
      for (uint32_t k = 0; k < kAhead; ++k) row(k, r + k > 0 && r + k + 1 < A.ny);
    }
  }
#pragma unroll
  for (uint32_t k = 0; k < kAhead; ++k)
    if (r + k < r1) row(k, r + k > 0 && r + k + 1 < A.ny);
}

__global__ void __launch_bounds__(1024) stencil2d_cols_kernel(const ColsArgs A) {
  enter_region_grid();
  const uint64_t warps = (uint64_t)gridDim.x * (blockDim.x / 32);
  for (uint64_t p = (uint64_t)blockIdx.x * (blockDim.x / 32) + warp_id(); p < A.pieces;
       p += warps) {
    const uint64_t col0 = p % A.strips * kStrip;
    const uint32_t r0 = (uint32_t)(p / A.strips) * A.rows;
    const uint32_t r1 = A.ny - r0 < A.rows ? A.ny : r0 + A.rows;
    if (col0 > 0 && A.nx - col0 > kStrip)
      walk_strip<true>(A, col0, r0, r1);
    else
      walk_strip<false>(A, col0, r0, r1);
  }
}

// Returns cudaErrorNotSupported, launching nothing, where the rule (plan.h) leaves
// the grid to the region kernel.
cudaError_t launch_stencil2d_cols(const void* in, float* out, uint64_t nx, uint64_t ny, float c0,
                                  float c1, unsigned teams, unsigned threads, cudaStream_t st) {
  if (!cols_applies(nx, ny, teams, threads)) return cudaErrorNotSupported;
  const uint64_t strips = (nx + kStrip - 1) / kStrip;
  ColsArgs a;
  a.in = (const float*)in;
  a.out = out;
  a.nx = nx;
  a.ny = (uint32_t)ny;
  a.c0 = c0;
  a.c1 = c1;
  a.strips = (uint32_t)strips;
  const uint64_t warps = (uint64_t)teams * (threads / 32);
  const uint64_t bands = warps / strips ? warps / strips : 1;  // row blocks for one piece a warp
  uint64_t rows = (ny + bands - 1) / bands;
  if (rows < 8) rows = 8;
  a.rows = (uint32_t)rows;
  a.pieces = strips * ((ny + rows - 1) / rows);
  return launch_kernel(stencil2d_cols_kernel, dim3(teams), dim3(threads), 0, st, a);
}

}  // namespace rt
