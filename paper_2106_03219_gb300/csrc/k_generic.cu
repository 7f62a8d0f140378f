// Generic-mode (non-SPMD) target regions.
//
// The region form is a loop nest whose outer level is sequential per team:
//   #pragma omp target teams distribute        // segments over teams
//   for (s = 0; s < nseg; ++s) {              // run by the team's main thread
//     double v = 0, w = 0;                     // shared with the parallel regions
//     #pragma omp parallel for reduction(+: v) // region 1, run by the whole team
//     for (i = seg[s]; i < seg[s + 1]; ++i) v += x[i] * y[i];
//     float a = (float)v * alpha;              // main thread: uses region 1's result
//     #pragma omp parallel for reduction(+: w) // region 2
//     for (i = seg[s]; i < seg[s + 1]; ++i) { y[i] = a * x[i] + y[i]; w += y[i]; }
//     result[s] = {v, a, w};                   // main thread again
//   }
// (program OMPRT_GENERIC_DOT_AXPY; program OMPRT_GENERIC_REDUCE runs region 1
// alone, its body the descriptor's dot or axpy.)
//
// The runtime side (as in the paper's runtime, Sec. 2.1): thread 0 is the
// main thread and runs the sequential code; the other threads are workers
// waiting in a state machine.  To start a parallel region the main thread
// publishes a work descriptor in team-shared memory (the id of the outlined
// region, its loop bounds and its arguments, among them pointers to the
// variables it shares with the sequential code) and releases the workers;
// every thread reads the descriptor and dispatches on the region id, the
// main thread taking part as thread 0 of the parallel team; a join barrier
// ends the region and the main thread resumes.  The shared variables are
// "globalised" onto the team's shared-memory stack with alloc_shared
// (Sec. 2.1, Listing 1), capacity S from omprt_alloc_shared, overflowing to
// the team's slice of the context's pool; a request that neither holds sets
// OMPRT_DEV_STACK_NOMEM and the team stops.  Every hand-over and every join
// is a team barrier reached by all threads from the same loop, so no thread
// spins; the main thread's code between two regions is one step of its
// program (a small state machine over (segment, phase)).
#include "api_internal.h"

namespace rt {

// Outlined parallel regions a work descriptor can name.
enum : int32_t { kRegionExit = 0, kRegionDot = 1, kRegionAxpy = 2 };

// The hand-over: what the main thread publishes for its workers.
struct WorkDesc {
  int32_t fn;       // outlined region id
  float alpha;      // axpy scale, a value of the sequential code
  uint64_t lo, hi;  // the region's worksharing loop
  double* red;      // globalised reduction variable (on the team stack)
};

struct GenericArgs {
  const int64_t* seg;  // nseg + 1 offsets into x / y
  uint64_t nseg;
  uint64_t n;          // length of x / y (offsets are checked against it)
  int32_t program;     // OMPRT_GENERIC_*
  int32_t body;        // OMPRT_GENERIC_REDUCE: OMPRT_BODY_DOT or OMPRT_BODY_AXPY
  const float* x;
  float* y;
  float alpha;
  uint32_t stack_bytes;   // S of the team stack
  uint32_t pool_bytes;    // fallback pool bytes per team
  uint32_t pool_teams;    // teams with a pool slice
  unsigned char* pool;
  double* result;      // per segment: 1 (REDUCE) or 3 (DOT_AXPY) doubles
  uint32_t* status;
  uint32_t ring_off;   // tiled form: byte offset of the tile ring in dynamic shared memory
  uint32_t tile_log2;  // tiled form: a tile is 2^tile_log2 elements
  uint32_t tiles;      // tiled form: tiles the ring holds
};

// parallel for over [lo, hi) under the default schedule, which OpenMP leaves
// to the implementation: static with a chunk of one 32-byte vector, round
// robin (a warp then covers 1 KB of contiguous memory per access; one
// contiguous piece per thread measured 0.77 of the copy rate for a dot over
// 2^14-element segments).  The iterations before the first 32-byte boundary
// and after the last run as scalars, round robin too.  Returns the thread's
// compensated partial of the reduction.
template <class Body>
__device__ __forceinline__ float2 generic_for(const Body& body, uint64_t lo, uint64_t hi) {
  const uint32_t t = threadIdx.x, T = blockDim.x;
  AccCompF32 acc;
  constexpr uint64_t V = Body::VEC;
  uint64_t vlo = lo, vhi = lo;
  if (body.vec_ok() && hi - lo >= V) {
    vlo = (lo + V - 1) / V * V;
    vhi = hi / V * V;
    if (vhi < vlo) vhi = vlo;
  }
  run_strided(body, lo, vlo - lo, t, T, acc);  // head
  {
    typename Body::Frag f[2];
    uint64_t v = vlo + (uint64_t)t * V;
    for (; v + (uint64_t)T * V < vhi; v += 2ull * T * V) {  // two vectors in flight
      body.load(v, f[0]);
      body.load(v + (uint64_t)T * V, f[1]);
      body.finish(v, f[0], acc);
      body.finish(v + (uint64_t)T * V, f[1], acc);
    }
    if (v < vhi) {
      body.load(v, f[0]);
      body.finish(v, f[0], acc);
    }
  }
  run_strided(body, vhi, hi - vhi, t, T, acc);  // tail
  return acc.part();
}

// ---------------------------------------------------------------------------
// The tiled form: x and y of the segments a team is about to run stream
// through a ring of tiles in shared memory.  A feeder warp beside the team
// issues bulk copies as tiles are freed, across regions and across segments:
// while a segment runs, the next ones already load.  A segment that fits the
// ring is loaded once and stays for its second region; a longer one streams
// through again.  The team's warps move through a region's tiles on their
// own (a full and an empty mbarrier a tile), so a region costs two team
// barriers: one when its last warp is done, one at the next hand-over.
//
// Why: with plain loads a region starts cold, keeps two vectors a thread in
// flight and asks for nothing more until its joins are over.  4096 lognormal
// segments (54.4 M elements, 653 MB), two regions each, 152 teams of 256:
// 434 us plain (DRAM 19 %, barrier and long-scoreboard stalls), 200 us tiled.
// A feeder inside the team, and a team barrier a tile, gained nothing (433 us:
// every tile then waits for the feeding thread).  What bounds it now: the team
// with 1.8 times the mean work, its two warps a scheduler in the latency of the
// compensated adds (0.37 cycles an element and region), and about 3 us of
// sequential code, joins and team reductions a segment.
//
// Tiles start on multiples of 4 elements; the array's last n % 4 elements,
// which no whole 16-byte unit holds, run from global memory.
// ---------------------------------------------------------------------------
static __shared__ __align__(8) uint64_t rt_tile_full[kTilesMax], rt_tile_empty[kTilesMax];
static __shared__ int rt_tile_stop;
constexpr int kAccs = 2;
constexpr uint64_t kTileWaitNs = 1000000000ull;  // 1 s: a tile takes microseconds

// A segment [lo, hi) cut into tiles of the ring.
struct TileSeg {
  uint64_t b0;  // first element of tile 0 (lo rounded down to 4)
  uint64_t e;   // hi, or the array's last whole unit if that is earlier
  uint32_t m;   // tiles
  __device__ __forceinline__ TileSeg(const GenericArgs& A, uint64_t lo, uint64_t hi) {
    const uint64_t whole = A.n & ~3ull;
    b0 = lo & ~3ull;
    e = hi < whole ? hi : whole;
    m = lo < e ? (uint32_t)((e - b0 - 1) >> A.tile_log2) + 1 : 0;
  }
  // its tiles stay in the ring from the first region to the second
  __device__ __forceinline__ bool stays(const GenericArgs& A) const {
    return A.program == OMPRT_GENERIC_DOT_AXPY && m <= A.tiles;
  }
};

// A place in the ring's load sequence: slot and parity of its barriers.
struct TilePos {
  uint32_t slot, parity;
  __device__ __forceinline__ void step(uint32_t tiles) {
    if (++slot == tiles) {
      slot = 0;
      parity ^= 1;
    }
  }
};

// The feeder (one thread): load the tiles of the team's segments in order,
// until the block ends, a segment is invalid (the main thread will report it)
// or the team stops.  Returns with no copy in flight.
__device__ __forceinline__ void feed_tiles(const GenericArgs& A, uint64_t s0, uint64_t scnt) {
  const uint32_t tile = 1u << A.tile_log2;
  TilePos next = {0u, 0u};
  uint32_t filled = 0;  // tiles issued, up to the ring's size
  int64_t lo, hi = scnt ? A.seg[s0] : 0, ahead = scnt ? A.seg[s0 + 1] : 0;
  bool go = true;
  for (uint64_t k = 0; go && k < scnt; ++k) {
    lo = hi;
    hi = ahead;
    if (k + 1 < scnt) ahead = A.seg[s0 + k + 2];  // used a segment later
    if (lo < 0 || lo > hi || (uint64_t)hi > A.n) break;
    const TileSeg sg(A, (uint64_t)lo, (uint64_t)hi);
    const uint64_t up = (sg.e + 3) & ~3ull;
    const int passes = A.program == OMPRT_GENERIC_DOT_AXPY && !sg.stays(A) ? 2 : 1;
    for (int p = 0; go && p < passes; ++p) {
      for (uint32_t j = 0; j < sg.m; ++j) {
        if (filled == A.tiles) {  // until the team's warps have left the slot's last tile
          const uint32_t bar = smem_addr(&rt_tile_empty[next.slot]);
          go = mbar_wait(bar, next.parity ^ 1, kTileWaitNs, A.status, &rt_tile_stop);
          if (!go) break;
        } else {
          ++filled;
        }
        const uint64_t ts = sg.b0 + ((uint64_t)j << A.tile_log2);
        const uint32_t bytes = (uint32_t)(up - ts < tile ? up - ts : tile) * 4;
        unsigned char* const dst = rt_dyn_smem + A.ring_off + (size_t)next.slot * tile * 8;
        const uint32_t bar = smem_addr(&rt_tile_full[next.slot]);
        mbar_expect_tx(bar, 2 * bytes);
        bulk_g2s(dst, A.x + ts, bytes, bar);
        bulk_g2s(dst + (size_t)tile * 4, A.y + ts, bytes, bar);
        next.step(A.tiles);
      }
    }
  }
  for (; filled; --filled) {  // the last loads of every slot, newest first
    if (next.slot == 0) next.parity ^= 1;
    next.slot = next.slot ? next.slot - 1 : A.tiles - 1;
    mbar_wait(smem_addr(&rt_tile_full[next.slot]), next.parity, kTileWaitNs, nullptr);
  }
}

// One tile's share of a parallel for under the default schedule, which OpenMP
// leaves to the implementation: static with a chunk of one 16-byte unit,
// round robin over the team (consecutive lanes, consecutive units: every
// shared-memory access is conflict-free and a warp's stores cover 512 bytes);
// the units that the segment's ends cut go to the first and the last thread.
// [r0, r1): the tile's elements of the segment; element 0 is the loop's t0.
// kAccs accumulators, so that one chain of compensated adds does not hold a
// thread that has few warps beside it.
template <class Body>
__device__ __forceinline__ void tile_for(const Body& b, const unsigned char* buf, uint32_t arr,
                                         uint64_t t0, uint32_t r0, uint32_t r1, uint32_t T,
                                         AccCompF32 (&acc)[kAccs]) {
  constexpr uint32_t kB = 4;  // units a thread keeps in flight
  const uint32_t t = threadIdx.x;
  const uint32_t f0 = (r0 + 3) / 4, f1 = r1 / 4;  // whole units [f0, f1)
  uint32_t* const out = Body::kStageWrites ? (uint32_t*)b.stage_dst() + t0 : nullptr;
  uint32_t u = f0 + t;
  for (; u + (kB - 1) * T < f1; u += kB * T) {
    uint4 v[kB][2];
#pragma unroll
    for (uint32_t q = 0; q < kB; ++q) {
      v[q][0] = *(const uint4*)(buf + (u + q * T) * 16);
      v[q][1] = *(const uint4*)(buf + arr + (u + q * T) * 16);
    }
#pragma unroll
    for (uint32_t q = 0; q < kB; ++q) {
      b.stage_unit(v[q], acc[q % kAccs]);
      if constexpr (Body::kStageWrites) *(uint4*)(out + 4 * (u + q * T)) = v[q][1];
    }
  }
#pragma unroll 1
  for (; u < f1; u += T) {
    uint4 v[2] = {*(const uint4*)(buf + u * 16), *(const uint4*)(buf + arr + u * 16)};
    b.stage_unit(v, acc[0]);
    if constexpr (Body::kStageWrites) *(uint4*)(out + 4 * u) = v[1];
  }
  auto cut = [&](uint32_t c) {  // unit c's elements inside [r0, r1)
    uint32_t mask = 15u;
    if (r0 > 4 * c) mask &= ~0u << (r0 - 4 * c);
    if (r1 < 4 * c + 4) mask &= ~(~0u << (r1 - 4 * c));
    uint4 v[2] = {*(const uint4*)(buf + c * 16), *(const uint4*)(buf + arr + c * 16)};
    b.stage_unit(v, acc[0], mask);
    if constexpr (Body::kStageWrites) {
      const uint32_t w[4] = {v[1].x, v[1].y, v[1].z, v[1].w};
#pragma unroll
      for (uint32_t k = 0; k < 4; ++k)
        if (mask >> k & 1) out[4 * c + k] = w[k];
    }
  };
  if (t == 0 && r0 % 4) cut(r0 / 4);
  if (t == T - 1 && r1 % 4 && (f0 <= f1 || r0 % 4 == 0)) cut(r1 / 4);
}

// The calling thread's share of a parallel for over the segment [lo, hi), from
// place `pos` of the load sequence on; `release`: its tiles are free after
// this region.  False: a copy never came (uniform over the warp).
template <class Body>
__device__ __forceinline__ bool tiles_for(const Body& b, const GenericArgs& A, const TileSeg& sg,
                                          uint64_t lo, uint64_t hi, TilePos pos, bool release,
                                          uint32_t T, AccCompF32 (&acc)[kAccs]) {
  const uint32_t tile = 1u << A.tile_log2;
  for (uint32_t j = 0; j < sg.m; ++j) {
    const bool ok = mbar_wait(smem_addr(&rt_tile_full[pos.slot]), pos.parity, kTileWaitNs, A.status);
    if (!__all_sync(0xffffffffu, ok)) return false;
    const uint64_t t0 = sg.b0 + ((uint64_t)j << A.tile_log2);
    const uint32_t r0 = lo > t0 ? (uint32_t)(lo - t0) : 0u;
    const uint32_t r1 = sg.e - t0 < tile ? (uint32_t)(sg.e - t0) : tile;
    tile_for(b, rt_dyn_smem + A.ring_off + (size_t)pos.slot * tile * 8, tile * 4, t0, r0, r1, T,
             acc);
    if (release) {
      __syncwarp();
      if (lane_id() == 0) mbar_arrive(smem_addr(&rt_tile_empty[pos.slot]));
    }
    pos.step(A.tiles);
  }
  if (hi > sg.e) {  // the array's last n % 4 elements
    const uint64_t from = lo > sg.e ? lo : sg.e;
    run_strided(b, from, hi - from, threadIdx.x, T, acc[0]);
  }
  return true;
}

// The main thread: its sequential code as a small state machine over
// (segment, phase), run up to the next parallel region at each step.
struct MainThread {
  uint64_t s0, scnt;       // the team's block of segments
  uint64_t k;              // segment
  int phase;               // within it
  int64_t lo, hi, next;    // its bounds; the next one's end, read a segment early
  double *v, *w;           // its globalised variables
  float a;
  bool stop;

  __device__ __forceinline__ void start(const GenericArgs& A, uint64_t s, uint64_t n, bool off) {
    s0 = s;
    scnt = n;
    k = 0;
    phase = 0;
    v = w = nullptr;
    a = 0.f;
    stop = off;
    lo = hi = next = 0;
    if (n && !off) {
      hi = A.seg[s];
      next = A.seg[s + 1];
    }
  }
  // the sequential code up to the next parallel region (or the end)
  __device__ __forceinline__ WorkDesc step(const GenericArgs& A) {
    WorkDesc d;
    d.fn = kRegionExit;
    d.alpha = 0.f;
    d.lo = d.hi = 0;
    d.red = nullptr;
    while (!stop && d.fn == kRegionExit) {
      if (phase == 0) {  // a new segment: globalise its shared variables
        if (k == scnt) break;
        lo = hi;
        hi = next;
        if (k + 1 < scnt) next = A.seg[s0 + k + 2];
        if (lo < 0 || lo > hi || (uint64_t)hi > A.n) {
          set_status(A.status, OMPRT_DEV_BAD_ARG);
          stop = true;
          break;
        }
        v = (double*)alloc_shared(sizeof(double), A.status);
        w = A.program == OMPRT_GENERIC_DOT_AXPY ? (double*)alloc_shared(sizeof(double), A.status)
                                                : nullptr;
        if (!v || (A.program == OMPRT_GENERIC_DOT_AXPY && !w)) {  // NOMEM bit already set
          release(A);
          stop = true;
          break;
        }
        *v = 0.0;
        if (w) *w = 0.0;
        d.fn = (A.program == OMPRT_GENERIC_REDUCE && A.body == OMPRT_BODY_AXPY) ? kRegionAxpy
                                                                                : kRegionDot;
        d.alpha = A.alpha;
        d.red = v;
        phase = 1;
      } else if (phase == 1 && A.program == OMPRT_GENERIC_DOT_AXPY) {
        // between the regions: the sequential code reads region 1's result
        a = __fmul_rn((float)*v, A.alpha);
        d.fn = kRegionAxpy;
        d.alpha = a;
        d.red = w;
        phase = 2;
      } else {  // after the segment's last region: results, release, next
        if (A.program == OMPRT_GENERIC_DOT_AXPY) {
          A.result[3 * (s0 + k)] = *v;
          A.result[3 * (s0 + k) + 1] = (double)a;
          A.result[3 * (s0 + k) + 2] = *w;
        } else {
          A.result[s0 + k] = *v;
        }
        release(A);
        ++k;
        phase = 0;
      }
    }
    d.lo = (uint64_t)lo;
    d.hi = (uint64_t)hi;
    return d;
  }
  __device__ __forceinline__ void release(const GenericArgs& A) {
    if (w) free_shared(w, sizeof(double), A.status);
    if (v) free_shared(v, sizeof(double), A.status);
    v = w = nullptr;
  }
};

__global__ void __launch_bounds__(1024) generic_kernel(const GenericArgs A) {
  enter_region_grid();
  __shared__ WorkDesc s_work;  // the team-shared hand-over word
  const uint32_t t = threadIdx.x, g = blockIdx.x, G = gridDim.x;
  if (t == 0)
    stack_init(A.stack_bytes, g < A.pool_teams ? A.pool + (uint64_t)g * A.pool_bytes : nullptr,
               A.pool_bytes);
  // the runtime's team reduction scratch, the bottom block of the team stack
  float2* scratch = (float2*)team_alloc(32 * sizeof(float2), A.status);
  uint64_t s0, scnt;  // teams distribute: a balanced block of segments per team
  split_even(A.nseg, G, g, s0, scnt);
  MainThread main;
  if (t == 0) main.start(A, s0, scnt, scratch == nullptr);
  for (;;) {
    if (t == 0) s_work = main.step(A);
    team_barrier();  // hand-over: workers leave the wait state
    const WorkDesc d = s_work;
    if (d.fn == kRegionExit) break;
    float2 part;
    RegionArgs ra;
    ra.x = A.x;
    ra.y = A.y;
    ra.alpha_f = d.alpha;
    if (d.fn == kRegionDot)  // dispatch on the outlined region's id
      part = generic_for(BodyDotF32(ra), d.lo, d.hi);
    else
      part = generic_for(BodyAxpyF32(ra), d.lo, d.hi);
    const float2 tv = team_reduce<AccCompF32>(part, scratch);
    if (t == 0) *d.red = __dadd_rn(*d.red, __dadd_rn((double)tv.x, (double)tv.y));
    team_barrier();  // join
  }
  if (scratch) team_free(scratch, 32 * sizeof(float2), A.status);
}

// The tiled form's kernel: the team is threads 0 .. T - 1, the feeder a warp
// beside it (T = blockDim.x - 32), and the team's barriers are named ones.  Its
// loops need more than the 64 registers that teams of 1024 leave a thread (98,
// which is four warps in each quarter of an SM).
__global__ void __launch_bounds__(kTiledThreads + 32) generic_tiled_kernel(const GenericArgs A) {
  enter_region_grid();
  __shared__ WorkDesc s_work;  // the team-shared hand-over word
  const uint32_t t = threadIdx.x, T = blockDim.x - 32, g = blockIdx.x;
  if (t == 0) {
    stack_init(A.stack_bytes, g < A.pool_teams ? A.pool + (uint64_t)g * A.pool_bytes : nullptr,
               A.pool_bytes);
    rt_tile_stop = 0;
    for (uint32_t i = 0; i < A.tiles; ++i) {
      mbar_init(smem_addr(&rt_tile_full[i]));
      mbar_init_count(smem_addr(&rt_tile_empty[i]), T / 32);
    }
  }
  // the runtime's team reduction scratch, the bottom block of the team stack;
  // its barriers also publish the ring's
  float2* const scratch = (float2*)team_alloc(32 * sizeof(float2), A.status);
  uint64_t s0, scnt;  // teams distribute: a balanced block of segments per team
  split_even(A.nseg, gridDim.x, g, s0, scnt);
  if (t >= T) {
    if (t == T && scratch) feed_tiles(A, s0, scnt);
  } else {
    MainThread main;
    if (t == 0) main.start(A, s0, scnt, scratch == nullptr);
    TilePos pos = {0u, 0u};  // the current segment's first tile in the load sequence
    for (;;) {
      if (t == 0) s_work = main.step(A);
      named_barrier(1, T);  // hand-over: workers leave the wait state
      const WorkDesc d = s_work;
      if (d.fn == kRegionExit) break;
      RegionArgs ra;
      ra.x = A.x;
      ra.y = A.y;
      ra.alpha_f = d.alpha;
      // the segment's last region frees its tiles; so does every region of a
      // segment that does not fit the ring
      const TileSeg sg(A, d.lo, d.hi);
      const bool again = d.fn == kRegionDot && sg.stays(A);
      AccCompF32 acc[kAccs];
      const bool ok = d.fn == kRegionDot  // dispatch on the outlined region's id
                          ? tiles_for(BodyDotF32(ra), A, sg, d.lo, d.hi, pos, !again, T, acc)
                          : tiles_for(BodyAxpyF32(ra), A, sg, d.lo, d.hi, pos, true, T, acc);
      if (!again) {
        const uint32_t last = pos.slot + sg.m % (2 * A.tiles);  // m places on
        pos.parity ^= last / A.tiles & 1;
        pos.slot = last % A.tiles;
      }
      const float2 part =
          warp_reduce<AccCompF32>(AccCompF32::merge(acc[0].part(), acc[1].part()));
      if (lane_id() == 0) scratch[warp_id()] = part;
      if (named_barrier_or(1, T, !ok)) break;  // join; a team that misses a tile stops
      if (warp_id() == 0) {
        float2 tv = lane_id() < T / 32 ? scratch[lane_id()] : AccCompF32::identity();
        for (uint32_t m = 1; m < T / 32; m *= 2) tv = AccCompF32::merge(tv, AccCompF32::shfl(tv, m));
        if (t == 0) *d.red = __dadd_rn(*d.red, __dadd_rn((double)tv.x, (double)tv.y));
      }
    }
    if (t == 0) {
      main.release(A);
      *(volatile int*)&rt_tile_stop = 1;  // a feeder still waiting for room ends too
    }
  }
  if (scratch) team_free(scratch, 32 * sizeof(float2), A.status);
}

}  // namespace rt

using namespace rt;

extern "C" omprt_status omprt_launch_generic(omprt_ctx* c, const int64_t* seg_dev, int64_t nseg,
                                             const omprt_loop_desc* d, int32_t program,
                                             double* result_dev, int32_t teams, int32_t threads,
                                             void* stream) {
  if (!c) return OMPRT_ERR_NOT_INIT;
  if (!d || nseg < 0 || (nseg && (!seg_dev || !result_dev))) return OMPRT_ERR_INVALID;
  if (program != OMPRT_GENERIC_REDUCE && program != OMPRT_GENERIC_DOT_AXPY)
    return OMPRT_ERR_INVALID;
  if (d->data_type != OMPRT_F32 || d->reserved || d->seq) return OMPRT_ERR_UNSUPPORTED;
  if (program == OMPRT_GENERIC_REDUCE && d->body != OMPRT_BODY_DOT && d->body != OMPRT_BODY_AXPY)
    return OMPRT_ERR_UNSUPPORTED;
  uint64_t n;
  int64_t lb;
  omprt_status st = loop_trip_count(d, &n, &lb);
  if (st) return st;
  if (n && (!d->x || !d->y)) return OMPRT_ERR_INVALID;
  if (threads == 0) threads = 256;
  if (threads < 32 || threads > 1024 || threads % 32) return OMPRT_ERR_INVALID;
  if (teams == 0) teams = c->sm_count;
  if (teams < 1) return OMPRT_ERR_INVALID;
  if (nseg == 0) return OMPRT_OK;
  DeviceGuard guard(c->device);
  OverlapScope overlap(c->launch_overlap, (size_t)c->smem_per_sm);
  GenericArgs a;
  a.seg = seg_dev;
  a.nseg = (uint64_t)nseg;
  a.n = n;
  a.program = program;
  a.body = d->body;
  a.x = (const float*)d->x;
  a.y = (float*)d->y;
  a.alpha = (float)d->alpha;
  a.stack_bytes = c->stack_bytes;
  a.pool_bytes = OMPRT_POOL_BYTES_PER_TEAM;
  a.pool_teams = OMPRT_MAX_RED_TEAMS;
  a.pool = c->pool_dev;
  a.result = result_dev;
  a.status = c->status_dev;
  const uintptr_t xa = (uintptr_t)d->x, ya = (uintptr_t)d->y;
  // Tiles are loaded segments ahead: not where a segment's y is another's x
  // (arrays that overlap without being the same).
  const bool overlap_xy = xa != ya && (xa < ya ? ya - xa : xa - ya) < n * 4;
  const TilePlan p = tile_plan({c->sm_count, c->max_smem_optin, c->smem_per_sm, 0u}, a.stack_bytes,
                               n, a.nseg, program == OMPRT_GENERIC_REDUCE && d->body == OMPRT_BODY_DOT,
                               (uint32_t)teams, (uint32_t)threads);
  a.ring_off = p.ring_off;
  a.tile_log2 = p.tile_log2;
  a.tiles = p.tiles;
  if (!p.tiles || ((xa | ya) & 15) || overlap_xy) {
    static const size_t static_bytes = static_smem_of(generic_kernel);
    if (smem_optin(generic_kernel, a.stack_bytes, static_bytes) != cudaSuccess) {
      cudaGetLastError();
      return OMPRT_ERR_CUDA;
    }
    return launch_kernel(generic_kernel, dim3(teams), dim3(threads), a.stack_bytes,
                         (cudaStream_t)stream, a) == cudaSuccess
               ? OMPRT_OK
               : OMPRT_ERR_CUDA;
  }
  static const size_t static_bytes = static_smem_of(generic_tiled_kernel);
  const size_t smem = a.ring_off + ((size_t)a.tiles << a.tile_log2) * 8;
  if (smem_optin(generic_tiled_kernel, smem, static_bytes) != cudaSuccess) {
    cudaGetLastError();
    return OMPRT_ERR_CUDA;
  }
  return launch_kernel(generic_tiled_kernel, dim3(teams), dim3(threads + 32), smem,
                       (cudaStream_t)stream, a) == cudaSuccess
             ? OMPRT_OK
             : OMPRT_ERR_CUDA;
}
