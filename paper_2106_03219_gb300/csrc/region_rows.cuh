// The row form: per-thread contiguous pieces moved through shared memory.
//
// Under static, static(c), dynamic(c), nonmonotonic dynamic and guided every
// thread runs contiguous pieces of the loop.  Read straight from global memory, a
// warp instruction then touches 32 lines, one per lane, and the launch is
// bound by L1 wavefronts (ncu of axpy dynamic(256), 608 x 256, n = 2^26: L1
// 91 % busy, DRAM 52 %, lg_throttle and long scoreboard 170 cycles an issue)
// and by the few bytes 64 registers keep in flight.  Here a warp moves its
// lanes' pieces together: each piece is cut at multiples of 128 (or 64) bytes
// of the array index, and one slab is the next such row of every lane, fetched
// with 16-byte asynchronous copies whose eight neighbouring lanes cover one
// whole line.  Every lane then runs its own row out of shared memory, and a
// written array goes back row by row the same way.  Ownership and each
// thread's pieces are the plain form's.
//
// Two or more stages a warp: the next slabs load while one is computed (608
// x 256: 139 us with two stages and 8 warps an SM, 153 with one and 16).
// Measured, plain -> rows, axpy fp32: dynamic(256) 608 x 256 at n = 2^26 197 ->
// 130-137 us (0.88-0.92 of the copy rate), static 1184 x 256 at n = 50,000,001
// 124 -> 102-105 us (0.85-0.88), static(64) 900 x 128 261 -> 142 us, dynamic(256) 608 x 256 at
// n = 2^22 19.2 -> 12.9 us; where it loses, and stays off: rows_gain in plan.h.  What
// bounds it now: 128-byte accesses that open a
// DRAM page for each row (whole contiguous windows of a warp's range reached
// 0.96 under static, but keep only a few lanes busy and lost everywhere
// else), one-stage teams of 512 and 1024, and the last wave of CTAs.
//
// Pieces may start and end anywhere: copies cover whole 16-byte units, never
// past the array's last whole unit (what is left runs from global memory), and
// a unit that holds another piece's elements is written element by element.
#pragma once

namespace rt {

// Pieces of the calling lane, relative to the team block; next() is reached
// by the whole warp and returns the same answer to all its lanes.  The
// lanes' pieces of one answer are adjacent, in lane order.
struct PieceOnce {  // static without chunk: one piece a thread
  static constexpr bool kAnyWarp = false;
  uint64_t lo, hi;
  bool taken;
  __device__ __forceinline__ bool next(uint64_t& l, uint64_t& h) {
    l = lo;
    h = hi;
    const bool first = !taken;
    taken = true;
    return first;
  }
};
template <class Claim>
struct PieceChunks {  // 32 consecutive chunks of c a claim, lane l running base + l
  static constexpr bool kAnyWarp = !std::is_same<Claim, ClaimStatic>::value;
  Claim claim;
  uint64_t nch, c, bn;
  __device__ __forceinline__ bool next(uint64_t& l, uint64_t& h) {
    const unsigned long long base = claim.next();
    if (base >= nch) return false;
    const uint64_t j = base + lane_id();
    l = h = bn;
    if (j < nch) {
      l = j * c;
      h = bn - l > c ? l + c : bn;
    }
    return true;
  }
};

struct PieceGuided {  // a warp's guided claims
  static constexpr bool kAnyWarp = true;
  uint64_t bn;
  uint32_t* status;
  __device__ __forceinline__ bool next(uint64_t& l, uint64_t& h) {
    const ulonglong2 k = guided_claim(bn, status);
    l = k.x;
    h = k.y;
    return k.x != ~0ull;
  }
};

// Buffers: the host gives a team as many sets of stages as its warps can need
// at once, which for a short block is fewer than its warps (a block of k
// claims keeps k warps busy).  Under a static schedule those are the first
// warps; under a dynamic one a warp takes a set with its first claim.
static __shared__ uint32_t rt_row_slots;

// The elements [r0, r1) of one lane's row (array k at buf + k * arr, element 0
// the loop's element `row`).  Results of whole units stay in the buffer for
// the warp's stores; of a unit that straddles the piece's ends the lane's
// elements go to global memory at once.
template <class Body, class Acc>
__device__ __forceinline__ void run_part_row(const Body& b, unsigned char* buf, uint32_t arr,
                                             uint64_t row, uint32_t r0, uint32_t r1, Acc& acc) {
  constexpr uint32_t A = Body::kStageArrays, EB = Body::kElemBytes, EPU = 16 / EB;
  static_assert(!Body::kStageWrites || EB == 4, "written arrays hold 32-bit elements");
  for (uint32_t u = r0 / EPU; u * EPU < r1; ++u) {
    unsigned char* const p = buf + u * 16;
    uint4 v[A];
#pragma unroll
    for (uint32_t k = 0; k < A; ++k) v[k] = *(const uint4*)(p + k * arr);
    const uint32_t e = u * EPU;
    uint32_t mask = (1u << EPU) - 1u;  // the unit's elements inside the piece
    if (r0 > e) mask &= ~0u << (r0 - e);
    if (r1 < e + EPU) mask &= ~(~0u << (r1 - e));
    b.stage_unit(v, acc, mask);
    if constexpr (Body::kStageWrites) {
      if (mask == (1u << EPU) - 1u) {
        *(uint4*)(p + (A - 1) * arr) = v[A - 1];
      } else {
        const uint32_t w[4] = {v[A - 1].x, v[A - 1].y, v[A - 1].z, v[A - 1].w};
        uint32_t* const dst = (uint32_t*)b.stage_dst() + row + e;
#pragma unroll
        for (uint32_t k = 0; k < EPU; ++k)
          if (mask >> k & 1) dst[k] = w[k];
      }
    }
  }
}

__device__ __forceinline__ void cp_async16_if(bool p, uint32_t dst, const void* src) {
  asm volatile(
      "{ .reg .pred q; setp.ne.u32 q, %2, 0; @q cp.async.cg.shared.global [%0], [%1], 16; }" ::"r"(
          dst),
      "l"(src), "r"((uint32_t)p)
      : "memory");
}
__device__ __forceinline__ void st16_if(bool p, void* dst, uint4 v) {
  asm volatile(
      "{ .reg .pred q; setp.ne.u32 q, %5, 0; @q st.global.v4.b32 [%0], {%1,%2,%3,%4}; }" ::"l"(dst),
      "r"(v.x), "r"(v.y), "r"(v.z), "r"(v.w), "r"((uint32_t)p)
      : "memory");
}
__device__ __forceinline__ void cp_async_commit() {
  asm volatile("cp.async.commit_group;" ::: "memory");
}
// all but the newest `newer` groups of this thread have landed
__device__ __forceinline__ void cp_async_wait(uint32_t newer) {
  switch (newer) {
    case 0: asm volatile("cp.async.wait_group 0;" ::: "memory"); break;
    case 1: asm volatile("cp.async.wait_group 1;" ::: "memory"); break;
    case 2: asm volatile("cp.async.wait_group 2;" ::: "memory"); break;
    default: asm volatile("cp.async.wait_group 3;" ::: "memory"); break;
  }
}

template <uint32_t kRow, class Body, class Acc, class Pieces>
__device__ __forceinline__ void run_rows(const Body& b, const RegionArgs& a, uint64_t bs,
                                         Pieces& pieces, Acc& acc) {
  constexpr uint32_t A = Body::kStageArrays, EB = Body::kElemBytes, EPU = 16 / EB;
  constexpr uint32_t NU = kRow / 16, RE = kRow / EB;  // units and elements a row
  constexpr uint32_t kStride = kRow + 16, kArr = 32 * kStride;
  constexpr uint32_t kStage = row_stage_bytes(A, kRow);
  const uint32_t lane = lane_id(), NS = a.row_stages;
  unsigned char* base = nullptr;  // this warp's stages, from its first claim on
  const uint64_t whole = a.n / EPU * EPU;
  uint64_t pos = 0, end = 0, t0 = 0, t1 = 0;
  bool more = true;
  uint32_t flight = 0, in = 0, out = 0;
  // the unit this lane copies of rows lane / NU, + 32 / NU, ...
  const uint32_t cu = lane % NU, cr = lane / NU;
  for (;;) {
    while (flight < NS) {
      while (more && !__any_sync(0xffffffffu, pos < end)) {
        more = pieces.next(pos, end);
        if (!more) pos = end = 0;
        pos += bs;
        end += bs;
        if (more && end > whole) {
          if (pos < end) {
            t0 = pos > whole ? pos : whole;
            t1 = end;
          }
          end = whole;
        }
      }
      if (!more) break;
      if (!base) {
        uint32_t slot = warp_id();
        if constexpr (Pieces::kAnyWarp) {
          if (lane == 0) slot = atomicAdd(&rt_row_slots, 1u);
          slot = __shfl_sync(0xffffffffu, slot, 0);
        }
        base = rt_dyn_smem + a.stage_off + (size_t)slot * NS * kStage;
      }
      unsigned char* const st = base + in * kStage;
      uint4* const rec = (uint4*)(st + A * kArr);
      const uint64_t row = pos / RE * RE;  // first element of the lane's row
      uint32_t j0 = 0, j1 = 0;             // the lane's elements of it
      if (pos < end) {
        j0 = (uint32_t)(pos - row);
        j1 = end - row < RE ? (uint32_t)(end - row) : RE;
        pos = row + j1;
      }
      rec[lane] = make_uint4((uint32_t)row, (uint32_t)(row >> 32), j0, j1);
      __syncwarp();
      uint4 m[NU];
#pragma unroll
      for (uint32_t q = 0; q < NU; ++q) m[q] = rec[q * (32 / NU) + cr];
#pragma unroll
      for (uint32_t q = 0; q < NU; ++q) {
        const uint32_t r = q * (32 / NU) + cr;
        const uint64_t o = ((((uint64_t)m[q].y << 32) | m[q].x) + cu * EPU) * EB;
        const bool p = cu * EPU < m[q].w && (cu + 1) * EPU > m[q].z;
#pragma unroll
        for (uint32_t k = 0; k < A; ++k)
          cp_async16_if(p, smem_addr(st) + k * kArr + r * kStride + cu * 16,
                        (const char*)b.stage_src(k) + o);
      }
      cp_async_commit();
      in = in + 1 == NS ? 0 : in + 1;
      ++flight;
    }
    if (!flight) break;
    cp_async_wait(flight - 1);
    __syncwarp();  // every lane's copies of the oldest stage have landed
    unsigned char* const st = base + out * kStage;
    uint4* const rec = (uint4*)(st + A * kArr);
    const uint4 own = rec[lane];
    unsigned char* const mine = st + lane * kStride;
    if (own.z == 0 && own.w == RE) {
      constexpr uint32_t kB = 4 / A < NU ? 4 / A : NU;
#pragma unroll
      for (uint32_t q = 0; q < NU; q += kB) {
        uint4 v[kB][A];
#pragma unroll
        for (uint32_t u = 0; u < kB; ++u)
#pragma unroll
          for (uint32_t k = 0; k < A; ++k) v[u][k] = *(const uint4*)(mine + k * kArr + (q + u) * 16);
#pragma unroll
        for (uint32_t u = 0; u < kB; ++u) {
          b.stage_unit(v[u], acc);
          if constexpr (Body::kStageWrites)
            *(uint4*)(mine + (A - 1) * kArr + (q + u) * 16) = v[u][A - 1];
        }
      }
    } else if (own.z < own.w) {
      run_part_row(b, mine, kArr, ((uint64_t)own.y << 32) | own.x, own.z, own.w, acc);
    }
    __syncwarp();
    if constexpr (Body::kStageWrites) {
#pragma unroll
      for (uint32_t h = 0; h < NU; h += 4) {
        uint4 m[4], v[4];
#pragma unroll
        for (uint32_t q = 0; q < 4; ++q) {
          const uint32_t r = (h + q) * (32 / NU) + cr;
          m[q] = rec[r];
          v[q] = *(const uint4*)(st + (A - 1) * kArr + r * kStride + cu * 16);
        }
#pragma unroll
        for (uint32_t q = 0; q < 4; ++q)
          st16_if(cu * EPU >= m[q].z && (cu + 1) * EPU <= m[q].w,
                  (char*)b.stage_dst() + ((((uint64_t)m[q].y << 32) | m[q].x) + cu * EPU) * EB,
                  v[q]);
      }
      __syncwarp();  // the stage has been read: the next slab may land in it
    }
    out = out + 1 == NS ? 0 : out + 1;
    --flight;
  }
  if (t0 < t1) run_scalar(b, t0, 1, t1 - t0, acc);
}

// Whether a body and schedule have a row form.
template <class Body, int SCHED>
constexpr bool rows_for() {
  return Stageable<Body>::value && !StageHalo<Body>::value &&
         (SCHED == kStatic || SCHED == kChunked || SCHED == kDynamic || SCHED == kGuided ||
          SCHED == kNonmono);
}

// The row form's kernel: the region kernel's levels and epilogue around
// run_rows.  A kernel of its own, so that its buffers and registers cost the
// plain forms nothing (with both in one kernel plain dynamic(256) of short
// blocks ran 7-14 % slower).
template <class Body, int SCHED, class Acc>
__global__ void __launch_bounds__(OMPRT_MAX_THREADS) rows_kernel(const RegionArgs a) {
  enter_region_grid();
  const uint32_t g = blockIdx.x, G = gridDim.x, t = threadIdx.x, T = blockDim.x;
  Body body(a);
  Acc acc;
  if (t == 0) {
    if constexpr (Acc::kActive)
      stack_init(a.stack_bytes, g < a.pool_teams ? a.pool + (uint64_t)g * a.pool_bytes : nullptr,
                 a.pool_bytes);
    rt_row_slots = 0;
  }
  uint64_t bs, bn;
  split_even(a.n, G, g, bs, bn);
  auto run = [&](auto pieces) {
    if (a.row_bytes == 128)
      run_rows<128>(body, a, bs, pieces, acc);
    else
      run_rows<64>(body, a, bs, pieces, acc);
  };
  const uint64_t c = a.chunk;
  const uint64_t nch = SCHED != kStatic && SCHED != kGuided && bn ? (bn - 1) / c + 1 : 0;
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
  } else if constexpr (SCHED == kGuided) {
    guided_start(0, c);  // and rt_row_slots is set
    run(PieceGuided{bn, a.status});
  } else {
    __shared__ unsigned long long nm_next[OMPRT_MAX_THREADS / 32], nm_end[OMPRT_MAX_THREADS / 32];
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
  if constexpr (Acc::kActive) reduce_epilogue(acc, a);
}

}  // namespace rt
