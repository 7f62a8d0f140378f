// 2-D 5-point stencil under static, static(c), dynamic(c) and nonmonotonic
// dynamic, team blocks and rows of any length: lane rows (region_rows.cuh)
// with the rows above and below.
//
// The forms that move whole grid rows or boxes need team blocks of whole rows
// and chunks that divide a row; team counts the runtime picks, odd grids and
// odd chunks give neither.  Here a slab is the next 32 (or 16) points of every
// lane's piece with what they read: those points and one unit on each side,
// and the same span one grid row up and down, each fetched as whole lines with
// 16-byte asynchronous copies.  A grid row that is no whole number of 16-byte
// units puts the rows above and below a fixed number of elements off; they are
// fetched one unit wider and shifted in registers.  Every lane computes its
// own points, four at a time, and the results leave line by line.
#include "launch_common.cuh"
#include "piece_spans.h"

namespace rt {

struct StencilPieceArgs {
  RegionArgs r;       // n, chunk, x, out, c0, c1, nx, ny, dyn_next
  uint32_t sn, ss;    // elements the rows above / below are off: -nx, nx mod 4
  uint64_t up;        // how far up the span above starts (piece_spans.h)
};

__host__ __device__ constexpr uint32_t piece_lane_units(uint32_t nu) { return 3 * nu + 5; }
__host__ __device__ constexpr uint32_t piece_stage_bytes(uint32_t nu) {
  return 32 * 16 * (piece_lane_units(nu) + 1);  // the lanes' rows, one record a lane
}

// elements s .. s + 3 of the eight in a, b (0 <= s < 4, the same for all threads)
__device__ __forceinline__ float4 shift4(const float4& a, const float4& b, uint32_t s) {
  const float4 h = s & 2 ? make_float4(a.z, a.w, b.x, b.y) : a;
  const float l = s & 2 ? b.z : b.x;
  return s & 1 ? make_float4(h.y, h.z, h.w, l) : h;
}

// the first `bytes` of a unit, the rest of it zero
__device__ __forceinline__ void cp_async_if(bool p, uint32_t dst, const char* src,
                                            uint32_t bytes) {
  asm volatile(
      "{ .reg .pred q; setp.ne.u32 q, %2, 0; @q cp.async.cg.shared.global [%0], [%1], 16, %3; }" ::
          "r"(dst),
      "l"(src), "r"((uint32_t)p), "r"(bytes)
      : "memory");
}

// A lane's row in shared memory, in 16-byte units: [0] the unit left of the
// row, [1 .. NU] the row, [NU + 1] the unit right of it; then NU + 1 units of
// the row above and NU + 1 of the row below; one of padding (an odd number
// of units: the lanes of an access phase hit distinct banks).
//
// A lane's record: the row's address, its own points [j0, j1) of it, and how
// far into the three spans the grid reaches (all in elements, one byte each;
// piece_spans.h).
template <uint32_t NU, class Pieces>
__device__ __forceinline__ void run_stencil_pieces(const BodyStencil2D& b,
                                                   const StencilPieceArgs& P, uint64_t bs,
                                                   Pieces& pieces) {
  constexpr uint32_t RE = 4 * NU;  // points a row
  constexpr uint32_t kLane = piece_lane_units(NU) * 16, kN = (NU + 2) * 16,
                     kSo = (2 * NU + 3) * 16;
  constexpr uint32_t kStage = piece_stage_bytes(NU);
  const RegionArgs& a = P.r;
  const uint32_t lane = lane_id(), sn = P.sn, ss = P.ss;
  const uint32_t nx = (uint32_t)a.nx, ny = (uint32_t)a.ny;
  const uint64_t n = a.n, up = P.up, down = a.nx - ss;
  unsigned char* st = nullptr;  // this warp's rows, from its first claim on
  uint64_t pos = 0, end = 0;
  const uint32_t cu = lane % NU, cr = lane / NU, k4 = 4 * cu;
  for (;;) {
    while (!__any_sync(0xffffffffu, pos < end)) {
      if (!pieces.next(pos, end)) return;
      pos += bs;
      end += bs;
    }
    if (!st) {
      uint32_t slot = warp_id();
      if constexpr (Pieces::kAnyWarp) {
        if (lane == 0) slot = atomicAdd(&rt_row_slots, 1u);
        slot = __shfl_sync(0xffffffffu, slot, 0);
      }
      st = rt_dyn_smem + (size_t)slot * kStage;
    }
    uint4* const rec = (uint4*)(st + 32 * kLane);
    {
      const uint64_t row = pos / RE * RE;
      uint32_t j0 = 0, j1 = 0;
      const PieceSpans sp = piece_spans<RE>(row, n, up, down);
      if (pos < end) {
        j0 = (uint32_t)(pos - row);
        j1 = end - row < RE ? (uint32_t)(end - row) : RE;
        pos = row + j1;
      }
      const char* const src = (const char*)(b.in + row);
      rec[lane] = make_uint4((uint32_t)(uintptr_t)src, (uint32_t)((uintptr_t)src >> 32),
                             j0 | j1 << 8, sp.ce | sp.ab << 8 | sp.be << 16);
      if (j0 < j1) {  // the units beyond the row's NU, each fetched by its lane
        const uint32_t mine = smem_addr(st) + lane * kLane;
        cp_async_if(j0 == 0 && row > 0, mine, src - 16, 16);
        cp_async_if(centre_edge(RE, j1, sp.ce), mine + (NU + 1) * 16, src + RE * 4,
                    unit_bytes(RE, sp.ce));
        if (sn | ss) {
          cp_async_if(above_edge(RE, j1, sn, sp.ab), mine + kN + NU * 16,
                      src + RE * 4 - up * 4, 16);
          cp_async_if(below_edge(RE, j1, ss, sp.be), mine + kSo + NU * 16,
                      src + RE * 4 + down * 4, unit_bytes(RE, sp.be));
        }
      }
      __syncwarp();
#pragma unroll
      for (uint32_t q = 0; q < NU; ++q) {
        const uint32_t l = q * (32 / NU) + cr;
        const uint4 m = rec[l];
        const char* const p = (const char*)(((uint64_t)m.y << 32) | m.x) + cu * 16;
        const uint32_t dst = smem_addr(st) + l * kLane + cu * 16;
        const uint32_t i0 = m.z & 255u, i1 = m.z >> 8, ce = m.w & 255u, ab = m.w >> 8 & 255u,
                       be = m.w >> 16;
        cp_async_if(centre_fetched(k4, i0, i1, ce), dst + 16, p, unit_bytes(k4, ce));
        cp_async_if(above_fetched(k4, i0, i1, sn, ab), dst + kN, p - up * 4, 16);
        cp_async_if(below_fetched(k4, i0, i1, ss, be), dst + kSo, p + down * 4,
                    unit_bytes(k4, be));
      }
      cp_async_commit();
    }
    cp_async_wait(0);
    __syncwarp();  // every lane's copies have landed
    const uint4 own = rec[lane];
    const uint32_t j0 = own.z & 255u, j1 = own.z >> 8;
    if (j0 < j1) {
      float4* const mine = (float4*)(st + lane * kLane);
      const float4* const above = (const float4*)(st + lane * kLane + kN);
      const float4* const below = (const float4*)(st + lane * kLane + kSo);
      const uint64_t row = (uint64_t)((const float*)(((uint64_t)own.y << 32) | own.x) - b.in);
      uint32_t r = (uint32_t)b.row_of(row), c = (uint32_t)(row - (uint64_t)r * nx);
      auto points = [&](float4& o, const float4& nn, const float4& so, float w, const float4& cc,
                        float e) {
        o.x = b.point(nn.x, so.x, cc.y, w, cc.x);
        o.y = b.point(nn.y, so.y, cc.z, cc.x, cc.y);
        o.z = b.point(nn.z, so.z, cc.w, cc.y, cc.z);
        o.w = b.point(nn.w, so.w, e, cc.z, cc.w);
      };
      // a unit with another piece's points beside this lane's
      auto part = [&](uint32_t u) {
        const float4 o = mine[u + 1];
        const float v[4] = {o.x, o.y, o.z, o.w};
        float* const dst = b.out + row + 4 * u;
#pragma unroll
        for (uint32_t q = 0; q < 4; ++q)
          if (4 * u + q >= j0 && 4 * u + q < j1) dst[q] = v[q];
      };
      if (c >= 1 && c + RE < nx && r >= 1 && r + 1 < ny) {
        // no boundary point in the whole row: every unit alike (those of
        // other pieces compute on what happens to lie there and stay here)
        float w = mine[0].w;
        float4 cc = mine[1], n0 = above[0], s0 = below[0];
#pragma unroll
        for (uint32_t h = 0; h < NU; h += 2) {
          const float4 c1 = mine[h + 2], c2 = mine[h + 3], n1 = above[h + 1], s1 = below[h + 1],
                       n2 = above[h + 2], s2 = below[h + 2];
          float4 o0, o1;
          points(o0, shift4(n0, n1, sn), shift4(s0, s1, ss), w, cc, c1.x);
          points(o1, shift4(n1, n2, sn), shift4(s1, s2, ss), cc.w, c1, c2.x);
          mine[h + 1] = o0;
          mine[h + 2] = o1;
          w = c1.w;
          cc = c2;
          n0 = n2;
          s0 = s2;
        }
      } else {
        float w = mine[0].w;
        float4 cc = mine[1], n0 = above[0], s0 = below[0];
#pragma unroll 1
        for (uint32_t u = 0; u < NU; ++u) {
          const float4 c1 = mine[u + 2], n1 = above[u + 1], s1 = below[u + 1];
          float4 o;
          points(o, shift4(n0, n1, sn), shift4(s0, s1, ss), w, cc, c1.x);
          float v[4] = {o.x, o.y, o.z, o.w};
          const float p[4] = {cc.x, cc.y, cc.z, cc.w};
#pragma unroll
          for (int q = 0; q < 4; ++q) {  // boundary points are copied
            if (r == 0 || r + 1 >= ny || c == 0 || c + 1 == nx) v[q] = p[q];
            if (++c == nx) {
              c = 0;
              ++r;
            }
          }
          mine[u + 1] = make_float4(v[0], v[1], v[2], v[3]);
          w = cc.w;
          cc = c1;
          n0 = n1;
          s0 = s1;
        }
      }
      if (j0 % 4) part(j0 / 4);
      if (j1 % 4 && (j0 % 4 == 0 || j0 / 4 != j1 / 4)) part(j1 / 4);
    }
    __syncwarp();
#pragma unroll
    for (uint32_t h = 0; h < NU; h += 4) {
      uint4 m[4], v[4];
#pragma unroll
      for (uint32_t q = 0; q < 4; ++q) {
        const uint32_t l = (h + q) * (32 / NU) + cr;
        m[q] = rec[l];
        v[q] = *(const uint4*)(st + l * kLane + 16 + cu * 16);
      }
#pragma unroll
      for (uint32_t q = 0; q < 4; ++q)
        st16_if(k4 >= (m[q].z & 255u) && k4 + 4 <= m[q].z >> 8,
                (char*)b.out + ((const char*)(((uint64_t)m[q].y << 32) | m[q].x) - (const char*)b.in) +
                    cu * 16,
                v[q]);
    }
    __syncwarp();  // the rows have been read: the next slab may land
  }
}

// 1-D 3-point stencil: the same slabs without rows above and below.  A lane's
// row: the unit left of it, its NU units, the unit right of it, one of padding.
template <class Pieces>
__device__ __forceinline__ void run_line_pieces(const BodyStencil1D& b, uint64_t bs,
                                                Pieces& pieces) {
  constexpr uint32_t NU = kLineNu, RE = 4 * NU, kLane = (NU + 3) * 16;
  const uint32_t lane = lane_id();
  const uint64_t n = b.n;
  unsigned char* st = nullptr;  // this warp's rows, from its first claim on
  uint64_t pos = 0, end = 0;
  const uint32_t cu = lane % NU, cr = lane / NU, k4 = 4 * cu;
  for (;;) {
    while (!__any_sync(0xffffffffu, pos < end)) {
      if (!pieces.next(pos, end)) return;
      pos += bs;
      end += bs;
    }
    if (!st) {
      uint32_t slot = warp_id();
      if constexpr (Pieces::kAnyWarp) {
        if (lane == 0) slot = atomicAdd(&rt_row_slots, 1u);
        slot = __shfl_sync(0xffffffffu, slot, 0);
      }
      st = rt_dyn_smem + (size_t)slot * kLineStage;
    }
    uint4* const rec = (uint4*)(st + 32 * kLane);
    const uint64_t row = pos / RE * RE;
    uint32_t j0 = 0, j1 = 0;
    const uint32_t ce = n - row < RE + 8 ? (uint32_t)(n - row) : RE + 8;  // its elements in x
    if (pos < end) {
      j0 = (uint32_t)(pos - row);
      j1 = end - row < RE ? (uint32_t)(end - row) : RE;
      pos = row + j1;
    }
    const char* const src = (const char*)(b.in + row);
    rec[lane] = make_uint4((uint32_t)(uintptr_t)src, (uint32_t)((uintptr_t)src >> 32),
                           j0 | j1 << 8, ce);
    if (j0 < j1) {  // the units beside the row, each fetched by its lane
      const uint32_t mine = smem_addr(st) + lane * kLane;
      cp_async_if(j0 == 0 && row > 0, mine, src - 16, 16);
      cp_async_if(centre_edge(RE, j1, ce), mine + (NU + 1) * 16, src + RE * 4,
                  unit_bytes(RE, ce));
    }
    __syncwarp();
#pragma unroll
    for (uint32_t q = 0; q < NU; ++q) {
      const uint32_t l = q * (32 / NU) + cr;
      const uint4 m = rec[l];
      const uint32_t i0 = m.z & 255u, i1 = m.z >> 8;
      cp_async_if(centre_fetched(k4, i0, i1, m.w), smem_addr(st) + l * kLane + cu * 16 + 16,
                  (const char*)(((uint64_t)m.y << 32) | m.x) + cu * 16, unit_bytes(k4, m.w));
    }
    cp_async_commit();
    cp_async_wait(0);
    __syncwarp();  // every lane's copies have landed
    if (j0 < j1) {
      float4* const mine = (float4*)(st + lane * kLane);
      const bool inner = row >= 1 && row + RE < n;  // no end point in the row
      float w = mine[0].w;
      float4 cc = mine[1];
#pragma unroll
      for (uint32_t u = 0; u < NU; ++u) {
        const float4 nx = mine[u + 2];
        float4 o = make_float4(b.point(w, cc.x, cc.y), b.point(cc.x, cc.y, cc.z),
                               b.point(cc.y, cc.z, cc.w), b.point(cc.z, cc.w, nx.x));
        if (!inner) {
          const uint64_t i = row + 4 * u;
          if (i == 0 || i + 1 == n) o.x = cc.x;
          if (i + 2 == n) o.y = cc.y;
          if (i + 3 == n) o.z = cc.z;
          if (i + 4 == n) o.w = cc.w;
        }
        mine[u + 1] = o;
        w = cc.w;
        cc = nx;
      }
      auto part = [&](uint32_t u) {  // a unit with another piece's points beside this lane's
        const float4 o = mine[u + 1];
        const float v[4] = {o.x, o.y, o.z, o.w};
#pragma unroll
        for (uint32_t q = 0; q < 4; ++q)
          if (4 * u + q >= j0 && 4 * u + q < j1) b.out[row + 4 * u + q] = v[q];
      };
      if (j0 % 4) part(j0 / 4);
      if (j1 % 4 && (j0 % 4 == 0 || j0 / 4 != j1 / 4)) part(j1 / 4);
    }
    __syncwarp();
#pragma unroll
    for (uint32_t h = 0; h < NU; h += 4) {
      uint4 m[4], v[4];
#pragma unroll
      for (uint32_t q = 0; q < 4; ++q) {
        const uint32_t l = (h + q) * (32 / NU) + cr;
        m[q] = rec[l];
        v[q] = *(const uint4*)(st + l * kLane + 16 + cu * 16);
      }
#pragma unroll
      for (uint32_t q = 0; q < 4; ++q)
        st16_if(k4 >= (m[q].z & 255u) && k4 + 4 <= m[q].z >> 8,
                (char*)b.out + ((const char*)(((uint64_t)m[q].y << 32) | m[q].x) - (const char*)b.in) +
                    cu * 16,
                v[q]);
    }
    __syncwarp();  // the rows have been read: the next slab may land
  }
}

constexpr unsigned kPieceThreads = 512;  // largest team in two dimensions
template <int SCHED, uint32_t NU>  // NU 0: the 1-D stencil
__global__ void __launch_bounds__(NU ? kPieceThreads : 1024)
    stencil_pieces_kernel(const StencilPieceArgs P) {
  enter_region_grid();
  const RegionArgs& a = P.r;
  const uint32_t g = blockIdx.x, t = threadIdx.x, T = blockDim.x;
  if (t == 0) rt_row_slots = 0;
  uint64_t bs, bn;
  split_even(a.n, gridDim.x, g, bs, bn);
  auto run = [&](auto pieces) {
    if constexpr (NU == 0)
      run_line_pieces(BodyStencil1D(a), bs, pieces);
    else
      run_stencil_pieces<NU>(BodyStencil2D(a), P, bs, pieces);
  };
  const uint64_t c = a.chunk;
  const uint64_t nch = SCHED != kStatic && bn ? (bn - 1) / c + 1 : 0;
  if constexpr (SCHED == kStatic) {
    uint64_t s, cnt;
    split_even(bn, T, t, s, cnt);
    run(PieceOnce{s, s + cnt, false});
  } else if constexpr (SCHED == kChunked) {
    run(PieceChunks<ClaimStatic>{ClaimStatic{0ull, T, warp_id() * 32u}, nch, c, bn});
  } else if constexpr (SCHED == kDynamic) {
    unsigned long long* const ctr = a.dyn_next + g;
    team_barrier();  // rt_row_slots is set
    run(PieceChunks<ClaimDynamic>{ClaimDynamic{ctr}, nch, c, bn});
    team_barrier();
    if (t == 0) *ctr = 0;  // leave the counter at zero for the next launch
  } else {
    __shared__ unsigned long long nm_next[32], nm_end[32];
    const uint32_t w = warp_id(), W = T / 32;
    if (lane_id() == 0) {
      uint64_t s0, cnt;
      split_even((nch + 31) / 32, W, w, s0, cnt);
      nm_next[w] = s0;
      nm_end[w] = s0 + cnt;
    }
    team_barrier();  // every range is set before any warp steals
    run(PieceChunks<ClaimNonmono>{ClaimNonmono{nm_next, nm_end, W, w, nch}, nch, c, bn});
  }
}

template <int SCHED, uint32_t NU>
static cudaError_t launch_pieces(unsigned teams, unsigned threads, size_t smem, cudaStream_t st,
                                 const StencilPieceArgs& P) {
  auto k = stencil_pieces_kernel<SCHED, NU>;
  static const size_t static_bytes = static_smem_of(k);
  const cudaError_t e = smem_optin(k, smem, static_bytes);
  if (e != cudaSuccess) return e;
  return launch_kernel(k, dim3(teams), dim3(threads), smem, st, P);
}

template <int SCHED>
static cudaError_t launch_pieces_nu(uint32_t nu, unsigned teams, unsigned threads, size_t smem,
                                    cudaStream_t st, const StencilPieceArgs& P) {
  return nu == 8 ? launch_pieces<SCHED, 8>(teams, threads, smem, st, P)
                 : launch_pieces<SCHED, 4>(teams, threads, smem, st, P);
}

// Tried after the block window (k_stencil_window.cu), which takes most of these
// launches where a team's block fits shared memory.  Returns
// cudaErrorNotSupported, launching nothing, where this form does not apply or
// loses to the others (4096^2 and 2048^2, plain or ring forms against this one,
// G x T teams x threads):
//   - pieces of 32 points on in blocks of 16 (dynamic(500), 174 x 122 on 6116 x 128,
//     blocks of four points: 14 us point by point, 22 here); teams of up to 512
//     threads;
//   - odd grids (nx no multiple of 4): always (3001 x 2503, 608 x 256: static
//     98 -> 37 us, static(32) 166 -> 45, static(128) 166 -> 31, static(500) 178
//     -> 41, dynamic(64) 168 -> 34, dynamic(256) 180 -> 46);
//   - other grids: static (608 x 256 68 -> 58, 900 x 128 85 -> 51), static(c) but
//     for the c in [32, 128] of the row ring (static(64) 608 x 256: 65 there, 70
//     here; static(500) 136 -> 55), nonmonotonic (608 x 256 94 -> 62), dynamic(c)
//     with 102 chunks a block of whole 32 points (dynamic(256) 608 x 256 95 -> 64, 900 x
//     128 107 -> 59; dynamic(500), 4096 x 28 on 4 x 64, 58 chunks: 18 -> 48;
//     dynamic(100), 5492 x 1950 on 608 x 256 33 -> 48), or with 48 any in blocks beyond
//     54,000 points, which no window holds (dynamic(1000) 86 x 64 458 -> 255).
// Rows of 16 points under static and short chunks, whose many pieces want many
// warps; of 32 under dynamic and from chunks of 256 on, and where 32 fit.  One
// slab a warp: the same memory as two slabs of half the warps was slower
// everywhere (static(64) 900 x 128: 74 against 131 us).
cudaError_t launch_stencil2d_pieces(int sched, unsigned teams, unsigned threads, int max_smem,
                                    bool row_ring, cudaStream_t st, const RegionArgs& a) {
  const bool whole = sched == kStatic, odd = a.nx % 4 != 0;
  if ((sched != kStatic && sched != kChunked && sched != kDynamic && sched != kNonmono) ||
      threads > kPieceThreads || a.n == 0 || a.nx >= (1ull << 31) || a.ny >= (1ull << 31) ||
      (((uintptr_t)a.x | (uintptr_t)a.out) & 15))
    return cudaErrorNotSupported;
  const uint64_t block = (a.n - 1) / teams + 1;
  if ((whole ? block / threads : a.chunk) < 32 || block < 16) return cudaErrorNotSupported;
  uint32_t warps = threads / 32;  // that can be busy at once
  if (!whole) {
    const uint64_t chunks = (block - 1) / a.chunk + 1;
    if (!odd && chunks < (sched != kDynamic ? 16u : block > 54000 ? 48u : 102u))
      return cudaErrorNotSupported;
    if (!odd && sched == kDynamic && block <= 54000 && a.chunk % 32 != 0)
      return cudaErrorNotSupported;
    if (!odd && sched == kChunked && a.chunk <= 128 && row_ring) return cudaErrorNotSupported;
    if ((chunks + 31) / 32 < warps) warps = (uint32_t)((chunks + 31) / 32);
  }
  const uint64_t room = (uint64_t)max_smem - 1024;
  uint32_t nu = sched == kStatic || (sched == kChunked && a.chunk < 256) ? 4 : 8;
  if ((uint64_t)warps * piece_stage_bytes(nu) > room) nu = 4;
  const size_t smem = (size_t)warps * piece_stage_bytes(nu);
  if (smem > room) return cudaErrorNotSupported;
  const StencilPieceArgs P = {a, (uint32_t)(4 - a.nx % 4) % 4, (uint32_t)(a.nx % 4),
                              piece_up(a.nx)};
  switch (sched) {
    case kStatic: return launch_pieces_nu<kStatic>(nu, teams, threads, smem, st, P);
    case kChunked: return launch_pieces_nu<kChunked>(nu, teams, threads, smem, st, P);
    case kDynamic: return launch_pieces_nu<kDynamic>(nu, teams, threads, smem, st, P);
    default: return launch_pieces_nu<kNonmono>(nu, teams, threads, smem, st, P);
  }
}

// The 1-D stencil.  Returns cudaErrorNotSupported, launching nothing, where the rule
// (plan.h) leaves the launch to the other forms.
cudaError_t launch_stencil1d_pieces(int sched, unsigned teams, unsigned threads, int sm_count,
                                    int max_smem, int smem_per_sm, cudaStream_t st,
                                    const RegionArgs& a) {
  const LinePlan p = line_plan({sm_count, max_smem, smem_per_sm, 0u},
                               (((uintptr_t)a.x | (uintptr_t)a.out) & 15) == 0, a.n, sched, a.chunk,
                               teams, threads);
  if (!p.smem) return cudaErrorNotSupported;
  const size_t smem = p.smem;
  const StencilPieceArgs P = {a, 0u, 0u};
  switch (sched) {
    case kStatic: return launch_pieces<kStatic, 0>(teams, threads, smem, st, P);
    case kChunked: return launch_pieces<kChunked, 0>(teams, threads, smem, st, P);
    case kDynamic: return launch_pieces<kDynamic, 0>(teams, threads, smem, st, P);
    default: return launch_pieces<kNonmono, 0>(teams, threads, smem, st, P);
  }
}

}  // namespace rt
