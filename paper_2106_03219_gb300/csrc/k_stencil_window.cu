// 2-D 5-point stencil under static, static(c), dynamic(c) and nonmonotonic
// dynamic: a team's whole block, with one grid row on each side, in shared
// memory.
//
// In the loop's linear index the points a block reads are one contiguous range,
// whatever the row length: the block, nx elements before it and nx after it.  It
// comes in as a few bulk copies, each with its own barrier, so the first pieces
// start while the rest still arrives; every element is fetched once a team, and
// no row or chunk has to line up with anything.  Every lane then walks its own
// pieces, eight points (one 32-byte sector of the output) at a time, with the
// points west and east carried along; lanes start their piece at different
// points so that a warp's reads spread over the banks.  Where a grid row is no
// whole number of 16-byte units the rows above and below lie a fixed number of
// elements off and are shifted in registers.
//
// Measured (plain, ring or lane-piece forms -> this; G x T teams x threads):
// 4096^2 608 x 256 static 59 -> 38 us, static(64) 65 -> 52, static(8) 122 -> 77,
// dynamic(256) 64 -> 49; 2048^2 608 x 256 static(64) 20.8 -> 13.5, dynamic(256) 30 ->
// 17; 3001 x 2503 608 x 256 static(61) 37 -> 24, dynamic(256) 48 -> 34.  What bounds
// it: on large blocks one or two CTAs an SM, each loading, computing (two-way
// bank conflicts, one sector after another in a lane) and storing in turn.  A
// loop unrolled twice with the stores free to move took 68 to 77 registers and
// was slower (static(64) 52 -> 58 us: fewer CTAs an SM).
#include "launch_common.cuh"

namespace rt {

struct WindowArgs {
  RegionArgs r;     // n, chunk, x, out, c0, c1, nx, ny, dyn_next
  uint32_t sn, ss;  // elements the rows above / below are off: -nx, nx mod 4
  uint32_t lead;    // elements before the block's first sector: nx rounded up to 8, and 8
  uint32_t seg;     // elements a copy (a multiple of 4)
};

constexpr uint32_t kSegs = 8;
static __shared__ __align__(8) uint64_t rt_window_bar[kSegs];

__device__ __forceinline__ float4 window_shift(const float4& a, const float4& b, uint32_t s) {
  const float4 h = s & 2 ? make_float4(a.z, a.w, b.x, b.y) : a;
  const float l = s & 2 ? b.z : b.x;
  return s & 1 ? make_float4(h.y, h.z, h.w, l) : h;
}

// Sectors [d, e) of one lane, in order.  win: element 8 d of the block at
// win[8 d - origin]; the piece is [i0, i1).
template <bool kOdd>
__device__ __forceinline__ void window_run(const BodyStencil2D& b, const WindowArgs& P,
                                           const float* win, int64_t origin, uint64_t d,
                                           uint64_t e, uint64_t i0, uint64_t i1) {
  if (d >= e) return;
  const uint32_t nx = (uint32_t)b.nx, ny = (uint32_t)b.ny;
  uint64_t i = 8 * d;
  uint32_t r = (uint32_t)b.row_of(i), c = (uint32_t)(i - (uint64_t)r * nx);
  const float* p = win + (int64_t)i - origin;
  const float* pn = p - nx - P.sn;
  const float* ps = p + nx - P.ss;
  float w = p[-1];
  float4 c0 = *(const float4*)p;
  float4 n0, s0;
  if constexpr (kOdd) {
    n0 = *(const float4*)pn;
    s0 = *(const float4*)ps;
  }
  for (; d < e; ++d, i += 8, p += 8, pn += 8, ps += 8) {
    const float4 c1 = *(const float4*)(p + 4), c2 = *(const float4*)(p + 8);
    float4 na, nb, sa, sb;
    if constexpr (kOdd) {
      const float4 n1 = *(const float4*)(pn + 4), n2 = *(const float4*)(pn + 8);
      const float4 s1 = *(const float4*)(ps + 4), s2 = *(const float4*)(ps + 8);
      na = window_shift(n0, n1, P.sn);
      nb = window_shift(n1, n2, P.sn);
      sa = window_shift(s0, s1, P.ss);
      sb = window_shift(s1, s2, P.ss);
      n0 = n2;
      s0 = s2;
    } else {
      na = *(const float4*)pn;
      nb = *(const float4*)(pn + 4);
      sa = *(const float4*)ps;
      sb = *(const float4*)(ps + 4);
    }
    float v[8];
    v[0] = b.point(na.x, sa.x, c0.y, w, c0.x);
    v[1] = b.point(na.y, sa.y, c0.z, c0.x, c0.y);
    v[2] = b.point(na.z, sa.z, c0.w, c0.y, c0.z);
    v[3] = b.point(na.w, sa.w, c1.x, c0.z, c0.w);
    v[4] = b.point(nb.x, sb.x, c1.y, c0.w, c1.x);
    v[5] = b.point(nb.y, sb.y, c1.z, c1.x, c1.y);
    v[6] = b.point(nb.z, sb.z, c1.w, c1.y, c1.z);
    v[7] = b.point(nb.w, sb.w, c2.x, c1.z, c1.w);
    if (!(c >= 1 && c + 8 < nx && r >= 1 && r + 1 < ny)) {  // boundary points are copied
      const float q[8] = {c0.x, c0.y, c0.z, c0.w, c1.x, c1.y, c1.z, c1.w};
      uint32_t rr = r, cc = c;
#pragma unroll
      for (int k = 0; k < 8; ++k) {
        if (rr == 0 || rr + 1 >= ny || cc == 0 || cc + 1 == nx) v[k] = q[k];
        if (++cc == nx) {
          cc = 0;
          ++rr;
        }
      }
    }
    float* const out = b.out + i;
    if (i >= i0 && i + 8 <= i1) {
      uint32_t u[8];
#pragma unroll
      for (int k = 0; k < 8; ++k) u[k] = as_u(v[k]);
      st8(out, u);
    } else {  // the piece's ends: another piece's points beside this one's
#pragma unroll
      for (uint32_t k = 0; k < 8; ++k)
        if (i + k >= i0 && i + k < i1) out[k] = v[k];
    }
    w = c1.w;
    c0 = c2;
    for (c += 8; c >= nx; c -= nx) ++r;
  }
}

template <int SCHED, bool kOdd>
__global__ void __launch_bounds__(1024) stencil_window_kernel(const WindowArgs P) {
  enter_region_grid();
  const RegionArgs& a = P.r;
  const uint32_t g = blockIdx.x, t = threadIdx.x, T = blockDim.x, lane = lane_id();
  const BodyStencil2D body(a);
  uint64_t bs, bn;
  split_even(a.n, gridDim.x, g, bs, bn);
  // the window's element 0; what lies outside the grid is neither copied nor used
  const int64_t origin = (int64_t)(bs & ~7ull) - P.lead;
  const uint64_t whole = a.n & ~3ull;
  const uint64_t lo = origin > 0 ? (uint64_t)origin : 0;
  const uint64_t up = bs + bn + a.nx + 8 < a.n ? bs + bn + a.nx + 8 : a.n;
  const uint64_t hi = ((up + 3) & ~3ull) < whole ? (up + 3) & ~3ull : whole;
  float* const win = (float*)rt_dyn_smem;
  if (t == 0) {
    for (uint32_t s = 0; s < kSegs; ++s) mbar_init(smem_addr(&rt_window_bar[s]));
    for (uint32_t s = 0; s < kSegs; ++s) {
      const uint64_t b0 = lo + (uint64_t)s * P.seg;
      if (b0 >= hi || bn == 0) break;
      const uint32_t bytes = (uint32_t)(hi - b0 < P.seg ? hi - b0 : P.seg) * 4;
      mbar_expect_tx(smem_addr(&rt_window_bar[s]), bytes);
      bulk_g2s(win + ((int64_t)b0 - origin), body.in + b0, bytes, smem_addr(&rt_window_bar[s]));
    }
  }
  if (t < a.n - whole && up > whole) win[(int64_t)(whole + t) - origin] = body.in[whole + t];
  team_barrier();  // the barriers and the grid's last odd elements are in place
  uint32_t ready = 0;  // copies known to have landed
  auto run = [&](auto pieces) {
    uint64_t l, h;
    while (pieces.next(l, h)) {
      const uint64_t i0 = bs + l, i1 = bs + h;
      uint32_t need = 0;  // copies the warp's pieces read
      if (l < h) {
        const uint64_t last = i1 + a.nx + 8 < hi ? i1 + a.nx + 8 : hi;
        need = last > lo ? (uint32_t)((last - lo - 1) / P.seg) + 1 : 0;
      }
      need = __reduce_max_sync(0xffffffffu, need);
      bool ok = true;
      for (; ok && ready < need; ++ready)
        ok = mbar_wait(smem_addr(&rt_window_bar[ready]), 0, kStageWaitNs, a.status);
      if (!__all_sync(0xffffffffu, ok)) return;
      if (l < h) {
        const uint64_t d0 = i0 / 8, d1 = (i1 + 7) / 8, nd = d1 - d0;
        const uint64_t turn = (lane - (uint32_t)d0) & 3u, off = turn < nd ? turn : 0;
        window_run<kOdd>(body, P, win, origin, d0 + off, d1, i0, i1);
        window_run<kOdd>(body, P, win, origin, d0, d0 + off, i0, i1);
      }
      __syncwarp();
    }
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
    run(PieceChunks<ClaimDynamic>{ClaimDynamic{ctr}, nch, c, bn});
    team_barrier();
    if (t == 0) *ctr = 0;  // leave the counter at zero for the next launch
  } else {
    __shared__ unsigned long long nm_next[OMPRT_MAX_THREADS / 32], nm_end[OMPRT_MAX_THREADS / 32];
    const uint32_t w = warp_id(), W = T / 32;
    if (lane == 0) {
      uint64_t s0, cnt;
      split_even((nch + 31) / 32, W, w, s0, cnt);
      nm_next[w] = s0;
      nm_end[w] = s0 + cnt;
    }
    team_barrier();  // every range is set before any warp steals
    run(PieceChunks<ClaimNonmono>{ClaimNonmono{nm_next, nm_end, W, w, nch}, nch, c, bn});
  }
  // no copy is in flight when the team ends (a block may need fewer than came)
  if (t == 0 && bn)
    for (uint32_t s = 0; s < kSegs && lo + (uint64_t)s * P.seg < hi; ++s)
      mbar_wait(smem_addr(&rt_window_bar[s]), 0, kStageWaitNs, nullptr);
}

template <int SCHED, bool kOdd>
static cudaError_t launch_window(unsigned teams, unsigned threads, size_t smem, cudaStream_t st,
                                 const WindowArgs& P) {
  auto k = stencil_window_kernel<SCHED, kOdd>;
  static const size_t static_bytes = static_smem_of(k);
  const cudaError_t e = smem_optin(k, smem, static_bytes);
  if (e != cudaSuccess) return e;
  return launch_kernel(k, dim3(teams), dim3(threads), smem, st, P);
}
template <int SCHED>
static cudaError_t launch_window_odd(bool odd, unsigned teams, unsigned threads, size_t smem,
                                     cudaStream_t st, const WindowArgs& P) {
  return odd ? launch_window<SCHED, true>(teams, threads, smem, st, P)
             : launch_window<SCHED, false>(teams, threads, smem, st, P);
}

// Returns cudaErrorNotSupported, launching nothing, where the rule (plan.h) leaves the
// launch to the other forms.
cudaError_t launch_stencil2d_window(int sched, unsigned teams, unsigned threads, int sm_count,
                                    int smem_per_sm, int budget, cudaStream_t st,
                                    const RegionArgs& a) {
  const WindowPlan p =
      window_plan({sm_count, 0, smem_per_sm, 0u}, budget,
                  ((uintptr_t)a.x & 15) == 0 && ((uintptr_t)a.out & 31) == 0, a.nx, a.ny, sched,
                  a.chunk, teams, threads);
  if (!p.smem) return cudaErrorNotSupported;
  const bool odd = a.nx % 4 != 0;
  const size_t smem = p.smem;
  WindowArgs P;
  P.r = a;
  P.sn = (uint32_t)(4 - a.nx % 4) % 4;
  P.ss = (uint32_t)(a.nx % 4);
  P.lead = p.lead;
  P.seg = (uint32_t)((p.floats + kSegs - 1) / kSegs + 3) / 4 * 4;
  switch (sched) {
    case kStatic: return launch_window_odd<kStatic>(odd, teams, threads, smem, st, P);
    case kChunked: return launch_window_odd<kChunked>(odd, teams, threads, smem, st, P);
    case kDynamic: return launch_window_odd<kDynamic>(odd, teams, threads, smem, st, P);
    default: return launch_window_odd<kNonmono>(odd, teams, threads, smem, st, P);
  }
}

}  // namespace rt
