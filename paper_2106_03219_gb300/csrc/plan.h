// Which form a launch takes: the rules on sizes, types and alignment, host
// arithmetic alone in plain C++, so that they can be asked on any machine.
// Every rule states both sides as measured on GB300 (G x T: teams x threads).
#pragma once

#include <cmath>
#include <cstddef>
#include <cstdint>

#include "host_device.h"

namespace rt {

// Schedules as the kernels are instantiated for them.
enum : int { kStatic = 0, kChunked = 1, kDynamic = 2, kAuto = 3, kDist = 4, kGuided = 5,
             kNonmono = 6 };

// What a rule needs to know of the device and the context.
struct PlanDevice {
  int sm_count, max_smem_optin, smem_per_sm;
  uint32_t stage_bytes;  // omprt_set_stage_bytes
};

// Arrays a body moves per iteration and their element size, for the staged
// form of schedules (0 arrays: the body is not staged); halo: elements its
// input window reaches beyond a pass on each side (the stencils).
struct StageShape {
  uint32_t arrays, elem;
  uint64_t halo;
  bool writes;  // the last array is written back
};
// Staged pass size for a dynamic(c) / static(c) / static launch: the largest
// P <= 32 chunks whose buffers (every warp: P chunks of every array) fit the
// context's per-team staging bytes, or 0 for the plain form.  Measured on
// GB300 (n = 2^26): chunks below 256 bytes are already coalesced in the plain
// form and lose to the per-pass overhead (static(8) axpy 0.94 staged against
// 1.02 plain); without a reduction staging wins from P >= 16 (dynamic(256)
// 0.97 against 0.64, static(64) 1.02 against 0.97) and loses below
// (dynamic(1024): P <= 8); with a (compensated) reduction the per-element
// work needs many warps per SM, and staging wins only with all 32 lanes busy
// on chunks of at most 512 bytes over all arrays (dot dynamic(64) +16%, sum
// +9%; dynamic(256) loses).
struct StagePlan {
  uint32_t chunks;      // P; 0: the plain form
  uint32_t warp_bytes;  // shared memory per warp
};
inline StagePlan stage_plan(const PlanDevice& c, const StageShape& sh, uint64_t chunk,
                            uint32_t threads, size_t smem_base, bool reduction) {
  const StagePlan none = {0u, 0u};
  if (!sh.arrays || c.stage_bytes == 0) return none;
  const uint64_t cb = chunk * sh.elem;
  if (cb % 16 || cb < 256 || cb > c.stage_bytes) return none;
  const uint64_t warps = threads / 32, per_warp = c.stage_bytes / warps;
  uint64_t P;
  if (sh.halo) {
    // window of at most P c + 2 halo + 6 elements (16-byte widened), then P
    // chunks of output.  The halo is re-read from L2 by every pass, so it
    // must stay small against the pass: at most a quarter of it (a 2-D grid
    // of 4096-wide rows needs two 16 KB halo rows per pass, and measured
    // slower staged: 0.21 against 0.25 for dynamic(256)).  A stencil unit
    // costs an owner lane several times an axpy unit, so long chunks walked
    // by one lane lose (1-D, n = 2^26: c = 64 0.94 staged against 0.69,
    // c = 128 0.74 against 0.65, c = 256 0.59 against 0.68): chunks of at
    // most 512 bytes.
    if (reduction || cb > 512) return none;
    const uint64_t fixed = (2 * sh.halo + 8) * sh.elem;
    P = per_warp > fixed ? (per_warp - fixed) / (2 * cb) : 0;
    if (P > 32) P = 32;
    if (P == 0 || 8 * sh.halo * sh.elem > P * cb) return none;
  } else {
    P = per_warp / (sh.arrays * cb);
    if (P > 32) P = 32;
    if (reduction ? (P < 32 || sh.arrays * cb > 512) : P < 16) return none;
  }
  // equal passes: a claim of 32 chunks in ceil(32 / P) passes of (nearly)
  // the same size, not P, P, ..., remainder
  P = (32 + (32 + P - 1) / P - 1) / ((32 + P - 1) / P);
  const uint64_t wb = sh.halo ? ((P * chunk + 2 * sh.halo + 8) * sh.elem + 15) / 16 * 16 + P * cb
                              : P * sh.arrays * cb;
  // leave room for the kernel's static shared memory
  if (smem_base + warps * wb + 2048 > (uint64_t)c.max_smem_optin) return none;
  return {(uint32_t)P, (uint32_t)wb};
}

constexpr uint32_t kRowStagesMax = 4;
// bytes of one stage of one warp: 32 rows of every array, each padded by one
// 16-byte unit (the lanes of a 128-bit access phase, one row apart, then hit
// distinct banks), and one 16-byte record a lane
constexpr RT_HD uint32_t row_stage_bytes(uint32_t arrays, uint32_t row) {
  return 32u * (arrays * (row + 16u) + 16u);
}

// Whether a launch that could take the row form (region_rows.cuh) gains by it.
// Rows cost a trip through shared memory and each warp walks its slabs one after
// another; the plain form has every lane read 32 bytes of its own piece.  The
// plain form loses where that costs most: arrays from DRAM (many open pages),
// pieces whose starts lie a multiple of 128 bytes apart (a warp's 32 lines then
// compete for few sets of L1), two arrays and one written.  Measured plain -> rows
// (us, G x T teams x threads), over 2839 random launches:
//   - Maps, and integer sums with them: rows, but not under static with pieces
//     below 400 bytes (axpy 608 x 256, 304 bytes 37.1 -> 43.3, 500 bytes 45.9 ->
//     43.1), nor where pieces are no multiple of 128 bytes and short (static(50)
//     608 x 256 n = 5.1 M 15.4 -> 23.9, static(100) n = 18 M 51.7 -> 54.9, dynamic(40)
//     1 x 128 616 -> 799; static(200) n = 4.6 M 15.6 -> 12.0), or a warp's share is
//     below 8 KB (nonmonotonic(50) 623 x 128 n = 2.8 M 17.1 -> 27.9).
//   - Reads (sums, max, min, dot), whose plain form has no write-back: from L2 the
//     plain form is faster (max static(4096) 23 x 32 n = 6.6 M 112 -> 176, int64
//     static(50) 6 x 32 180 -> 396, bf16 static 9 x 32 136 -> 262), from DRAM rows
//     are (max static 153 x 64 n = 58 M 138 -> 79, int32 static(1000) 15 x 256 n = 7.8 M
//     100 -> 60).  26 MB of arrays are a fifth of the L2: they are still there from
//     the launch before.  Under dynamic and nonmonotonic, pieces a multiple of 128
//     bytes gain from L2 too with six warps a team (dot dynamic(128) 2 x 512, 492 -> 231).
//   - Compensated sums inside a map: as reads, but always under dynamic schedules.
//   - bf16: only dynamic and static chunks of a multiple of 128 bytes with six warps
//     a team (static(64) 608 x 256 n = 19 M 26.4 -> 19.7; static(256) n = 3.2 M 9.7 ->
//     13.1; nonmonotonic(100) n = 61 M 1259 -> 1562).
// warps: a team's that can be busy; an_sm: of those on an SM at once; row: bytes.
inline bool rows_gain(const StageShape& sh, int sched, uint64_t n, uint64_t chunk, uint64_t block,
                      uint64_t piece, uint32_t warps, double an_sm, uint32_t row, bool comp_sum) {
  const uint64_t bytes = n * sh.elem * sh.arrays, share = block * sh.elem / warps;
  const bool whole = sched == kStatic, guided = sched == kGuided;
  const bool claims = sched == kDynamic || sched == kNonmono;
  const bool even = !whole && chunk * sh.elem % 128 == 0, dram = bytes > 26000000;
  if (sh.writes && !comp_sum) {
    if (whole) return piece >= 400;
    if (guided || even) return true;
    return claims ? share >= 8192 : piece >= 600 || (dram && an_sm <= 4);
  }
  if (sh.elem == 2) return !whole && !guided && even && warps >= 6;
  if (whole) return dram && piece >= 640;
  if (guided) return dram && (comp_sum || an_sm <= 6.3);
  if (sh.writes) return claims || bytes > 40000000 || (even && an_sm > 0.4);
  if (even) return claims ? dram || warps >= 6 : bytes > 40000000;
  if (claims)
    return comp_sum ? bytes > 77000000 : dram && (share >= 24u * 32 * row || piece >= 2000);
  return bytes > 40000000 && piece >= 400 && an_sm <= 8;
}

// The row form of a launch whose threads run contiguous pieces: where it gains
// (above), with
//   - pieces of 128 bytes on under static(c) and dynamic(c) (axpy static(32)
//     608 x 256: 260 -> 150 us; static(16) 232 -> 236);
//   - blocks of 16 chunks on: with fewer, most lanes of the only claim are
//     idle and each walks its chunk slab by slab (7 chunks of 256:
//     11.2 -> 12.6 us; 27 chunks: 19.4 -> 13.4);
//   - not static with a compensated sum: there the adds, not the loads, hold a
//     launch (dot 500 x 512: 101 -> 111 us), unless the pieces are long;
//   - a single stage a warp (teams of 1024) only where the plain form is
//     worst: pieces of 512 bytes on (dynamic(256) 333 x 1024: 261 -> 164 us;
//     static(64) 156 -> 175).
// Shape: rows of 128 bytes where two stages a warp fit, else of 64; 64 also
// for compensated sums, which want more warps (dot dynamic(256): 112 -> 103
// us).  CTAs an SM: the count whose last wave is fullest, among those that
// keep enough in flight (14 stages of 128-byte rows an SM; 608 x 256: one CTA
// with two stages a warp 139 us, two with one 153).  Sized from the device's
// shared memory, whatever the staging bytes; those at zero turn it off.
struct RowPlan {
  uint32_t row_bytes, stages;  // row_bytes 0: not this form
  size_t smem;                 // dynamic shared memory of the buffers
};
inline RowPlan row_plan(const PlanDevice& c, const StageShape& sh, bool aligned16, uint64_t n,
                        int sched, uint64_t chunk, uint32_t teams, uint32_t threads,
                        size_t smem_base, bool comp_sum) {
  RowPlan best = {0u, 0u, 0};
  if (!sh.arrays || sh.halo || c.stage_bytes == 0 || n == 0) return best;
  if (!aligned16) return best;
  const bool whole = sched == kStatic;  // one piece a thread
  const uint64_t block = (n - 1) / teams + 1;
  const uint64_t piece = (whole ? block / threads : chunk) * sh.elem;
  if (piece < (whole ? (comp_sum ? 2048u : 256u) : 128u)) return best;
  uint32_t warps = threads / 32;  // that can be busy at once
  if (!whole) {
    const uint64_t chunks = (block - 1) / chunk + 1;
    if (chunks < 16) return best;
    if ((chunks + 31) / 32 < warps) warps = (uint32_t)((chunks + 31) / 32);
  }
  constexpr uint64_t kStatic_ = 2048;      // the kernels' static shared memory, rounded up
  constexpr uint64_t kReserved = 1024;     // what the hardware keeps of it for each CTA
  const uint32_t most = threads >= 1024 ? 1 : 1024 / threads;  // CTAs an SM, by registers
  double top = 0;
  uint32_t ctas = 1;  // an SM
  for (uint32_t row = comp_sum ? 64 : 128; row >= 64 && !best.row_bytes; row /= 2) {
    const uint64_t set = (uint64_t)warps * row_stage_bytes(sh.arrays, row);
    for (uint32_t k = most; k >= 1; --k) {
      uint64_t room = (uint64_t)c.smem_per_sm / k;
      if (room > (uint64_t)c.max_smem_optin + kReserved) room = (uint64_t)c.max_smem_optin + kReserved;
      const uint64_t fixed = kReserved + kStatic_ + smem_base;
      uint64_t ns = room > fixed ? (room - fixed) / set : 0;
      if (ns > kRowStagesMax) ns = kRowStagesMax;
      if (ns == 0 || (ns == 1 && row == 128)) continue;
      if (ns == 1 && threads >= 1024 && piece < 512) continue;
      const double wave = (double)c.sm_count * k;
      const double full = teams / wave / std::ceil(teams / wave);
      const double flight = (double)(k * warps * ns) * row / (14 * 128), busy = k * warps / 16.0;
      double score = full * std::fmin(flight, 1.0) * (ns > 1 ? 1.0 : 0.92);
      if (comp_sum) score *= std::fmin(busy, 1.0);
      if (score > top * 1.001) {
        top = score;
        ctas = k;
        best = {row, (uint32_t)ns, (size_t)(ns * set)};
      }
    }
  }
  const double an_sm = (double)warps * std::fmin(teams, (double)c.sm_count * ctas) / c.sm_count;
  if (best.row_bytes && !rows_gain(sh, sched, n, chunk, block, piece, warps, an_sm,
                                   best.row_bytes, comp_sum))
    return {0u, 0u, 0};
  return best;
}

// Whether every team's block starts on a 16-byte boundary of the arrays: team
// g's starts at g q + min(g, r), q = n / teams, r = n mod teams.
inline bool blocks_aligned(uint64_t n, uint64_t teams, uint32_t elem) {
  const uint64_t q = n / teams, r = n % teams;
  if (r && (q + 1) * elem % 16) return false;                 // blocks 1 .. r
  return r + 1 >= teams || q * elem % 16 == 0;                // those after
}

// Staged passes, rows, or (neither) the plain form.  aligned16: the arrays
// start on a 16-byte boundary.
struct StreamPlan {
  uint32_t stage_chunks, stage_warp_bytes;  // staged form
  uint64_t stage_chunk;                     // its chunk: the schedule's, or a thread's piece
  uint32_t row_bytes, row_stages;           // row form
  size_t smem;                              // dynamic shared memory beyond smem_base
};
inline StreamPlan stream_plan(const PlanDevice& c, const StageShape& sh, bool stencil2d,
                              bool aligned16, uint64_t n, int sched, uint64_t chunk,
                              uint32_t teams, uint32_t threads, size_t smem_base, bool reduction,
                              bool comp_sum) {
  StreamPlan p = {0u, 0u, 0u, 0u, 0u, 0};
  // the chunk a warp's lanes own (static without chunk: one block of n / (G T)
  // per thread, used only when that division is exact, so every team's block is
  // T of them)
  uint64_t stage_c = 0;
  if (sched == kDynamic || sched == kChunked || sched == kNonmono) stage_c = chunk;
  if (sched == kStatic && n % ((uint64_t)teams * threads) == 0)
    stage_c = n / ((uint64_t)teams * threads);
  // The staged form runs in blocks that start on a 16-byte boundary.  Where not
  // all do, streaming bodies take the row form instead (axpy static(64) at n =
  // 2^26, 900 x 128: 227 -> 139 us); where all do, whatever the remainder of the
  // division, they stay (static(64), n = 2,050,019 on 3 x 64: 261 us staged, 402 in
  // rows; dynamic(32) of int64 values, n = 256,999 on 4 x 64: 52 and 63).
  if (stage_c && (stencil2d || blocks_aligned(n, teams, sh.elem))) {
    const StagePlan sp = stage_plan(c, sh, stage_c, threads, smem_base, reduction);
    if (sp.chunks) {
      p.stage_chunks = sp.chunks;
      p.stage_warp_bytes = sp.warp_bytes;
      p.stage_chunk = stage_c;
      p.smem = (size_t)(threads / 32) * sp.warp_bytes;
      return p;
    }
  }
  if (sched == kStatic || sched == kChunked || sched == kDynamic || sched == kGuided ||
      sched == kNonmono) {
    const RowPlan rp =
        row_plan(c, sh, aligned16, n, sched, chunk, teams, threads, smem_base, comp_sum);
    if (rp.row_bytes) {
      p.row_bytes = rp.row_bytes;
      p.row_stages = rp.stages;
      p.smem = rp.smem;
    }
  }
  return p;
}

// 1-D stencil by lanes' pieces (k_stencil_pieces.cu); smem 0: not this form.
// A warp's slabs follow one another, so it takes data from DRAM or many warps, and
// pieces that fill their rows: whole 32 points, or 80 on (a piece of 40 touches two or
// three rows).  Measured plain -> pieces (us, G x T teams x threads) on 1627 random
// launches; the rule is 5 % and more from the better one in 44 of them:
//   - chunks of 32 points on in blocks of 32 chunks (n = 2^26, 608 x 256: static(64)
//     210 -> 129, dynamic(256) 151 -> 143; n = 2^22 dynamic(256), 27 chunks a block:
//     15.6 -> 16.1), and under static pieces of 64 to 256 points and from 1024 on
//     (608 x 256: 431 points 123 -> 138; 148 x 128, 3542 points 222 -> 181);
//   - static: 26 MB of arrays (a fifth of the L2), teams of 512 threads, or of 256 with
//     80 to 128 points or 1024 on (79 x 256, 95 points 11.9 -> 8.2; 4 x 256, 70 points 6.4 ->
//     7.3);
//   - whole 32 points: 26 MB (under dynamic and nonmonotonic in blocks of 72 chunks or
//     48 MB: 5,700,616 points, dynamic(256) 608 x 256, 37 chunks 17 -> 20), five busy
//     warps a team (dynamic(64), 28 x 128, four, 8 M points 197 -> 158, 50 x 64, two
//     4.9 -> 5.4), or four an SM at once (dynamic(64), 1.2 M points on 595 x 1024, one
//     14.7 -> 17.5);
//   - 80 points on, no multiple of 32: as much data, or more warps, nine under static(c)
//     (static(500) 1 x 256 37 -> 42), twelve else (dynamic(100) 30 x 1024, six, 7.7 -> 9.3;
//     dynamic(1000) 1 x 512, sixteen 404 -> 292);
//   - shorter: 26 MB and sixteen warps an SM (dynamic(40), 608 x 256 180 -> 139, but 133
//     x 32 237 -> 299), from 45 points on also 40 MB or sixteen warps a team (dynamic(50)
//     5 x 1024 96 -> 78, 426 x 1024, six 16.6 -> 19.3).
constexpr uint32_t kLineNu = 8;  // 16-byte units a row
constexpr uint32_t kLineStage = 32 * 16 * (kLineNu + 4);
struct LinePlan {
  size_t smem;
};
inline LinePlan line_plan(const PlanDevice& c, bool aligned16, uint64_t n, int sched,
                          uint64_t chunk, uint32_t teams, uint32_t threads) {
  const LinePlan none = {0};
  const bool whole = sched == kStatic, claims = sched == kDynamic || sched == kNonmono;
  if ((!whole && !claims && sched != kChunked) || n == 0 || !aligned16) return none;
  const uint64_t block = (n - 1) / teams + 1, piece = whole ? block / threads : chunk;
  if (piece < (whole ? 64u : 32u) || (whole && piece > 256 && piece < 1024)) return none;
  uint32_t warps = threads / 32;  // that can be busy at once
  uint64_t chunks = threads;
  if (!whole) {
    chunks = (block - 1) / chunk + 1;
    if (chunks < 32) return none;
    if ((chunks + 31) / 32 < warps) warps = (uint32_t)((chunks + 31) / 32);
  }
  const size_t smem = (size_t)warps * kLineStage;
  if ((int64_t)smem > (int64_t)c.max_smem_optin - 1024) return none;
  // CTAs and busy warps an SM at once
  const double ctas = std::fmin(threads < 1024 ? 1024 / threads : 1,
                                std::floor((double)c.smem_per_sm / (double)(smem + 1024)));
  const double an_sm = warps * std::fmin(teams, c.sm_count * ctas) / c.sm_count;
  const bool dram = n * 8 > 26000000, even = chunk % 32 == 0;
  bool gain;
  if (whole)
    gain = dram || threads >= 512 ||
           (threads >= 256 && (piece >= 1024 || (piece >= 80 && piece <= 128)));
  else if (!even && piece < 80)
    gain = (dram && (an_sm >= 16 || (piece >= 45 && n > 5000000))) || (piece >= 45 && warps >= 16);
  else if (!claims)
    gain = (dram && n > 3400000) || warps >= (even ? 5 : 9) || (even && an_sm > 4);
  else
    gain = (dram && (chunks >= 72 || n > 6000000)) || warps >= (even ? 5 : 12) ||
           (even && an_sm > 4 && chunks >= 44);
  return gain ? LinePlan{smem} : none;
}

// Generic regions by tiles (k_generic.cu); tiles 0: the plain form.
// A tiled CTA is the team and its feeder warp, at 98 registers a thread: an SM holds
// sixteen such warps, one team of 256 threads, three of 128, five of 64.  The ring
// takes what the teams resident on an SM leave each, for at most four: at least
// three tiles, of 8192 elements (64 KB) if they fit, else of 4096, 2048 or 1024.  A
// tile costs a wait and an arrival a warp (4096 uneven segments, one team an SM:
// 206 us with 8192 elements, 250 with 4096).
//
// Measured plain -> tiled (us, G x T teams x threads), 1000 random launches:
//   - one wave of resident teams: tiled (152 x 256, 4096 segments of 13,000 elements
//     434 -> 199; 18 x 32 2068 -> 292), but for single dots shorter than a thread
//     each (152 x 256, 27 segments 4.0 -> 4.4);
//   - more teams than are resident: a second wave starts cold, and teams of 256 run
//     one after another where four plain ones share an SM (161 x 256 31 -> 52, 524 x 256
//     42 -> 133, 2704 x 256 58 -> 184); up to 128 threads it pays from segments of 16
//     elements a thread on (1765 x 32, segments of 13,000 418 -> 101, 960 x 128 of 3500
//     47 -> 30, 3005 x 32 of 100 12 -> 30), and up to two waves where half the teams
//     have none (1020 x 32, 97 segments 6.8 -> 5.3).
constexpr uint32_t kTilesMax = 8;
constexpr uint32_t kTiledThreads = 480;  // largest team, 512 threads with the feeder
struct TilePlan {
  uint32_t tiles, tile_log2, ring_off;  // ring_off: after the team stack
};
inline TilePlan tile_plan(const PlanDevice& c, uint32_t stack_bytes, uint64_t n, uint64_t nseg,
                          bool single_dot, uint32_t teams, uint32_t threads) {
  const TilePlan none = {0u, 0u, 0u};
  if (threads > kTiledThreads || nseg == 0) return none;
  const uint32_t sms = (uint32_t)c.sm_count, fit = 16 / (threads / 32 + 1) < 4
                                                       ? 16 / (threads / 32 + 1) : 4;
  const uint32_t want = (teams - 1) / sms + 1, resident = want < fit ? want : fit;
  int64_t room = c.smem_per_sm / (int64_t)resident - 1024;
  if (room > c.max_smem_optin) room = c.max_smem_optin;
  room -= (int64_t)stack_bytes + 1024;
  TilePlan p = {0u, 13u, (stack_bytes + 127u) & ~127u};
  while (p.tile_log2 > 10 && room < 3 * (8 << p.tile_log2)) --p.tile_log2;
  const int64_t tiles = room > 0 ? room / (8 << p.tile_log2) : 0;
  if (tiles < 2) return none;
  p.tiles = tiles < kTilesMax ? (uint32_t)tiles : kTilesMax;
  const double a_thread = (double)n / (double)nseg / threads;  // a segment's elements
  if (want <= fit) return single_dot && nseg <= teams && a_thread < 1 ? none : p;
  const bool idle = want <= 2 * fit && nseg <= teams / 2 && !(single_dot && a_thread < 1);
  return threads <= 128 && (a_thread >= 16 || idle) ? p : none;
}

// Whether a grid of the region kernel's point-by-point 2-D stencil goes without
// launch overlap.  An overlapped grid's first blocks fill the slots the one before
// leaves free, and SMs that finish early take the rest, so its fullest SM can hold
// more blocks than an even spread gives; bound by instructions, that SM sets the
// time.  It matters where the SMs are nearly evenly filled and have slots for 1.1 to
// 1.8 times the blocks, from four points a thread on, twelve under dist_schedule
// (plain -> overlapped, us: static(8) 1291 x 634, 842 x 128 7.1 -> 8.6; static(1) with
// 47 points a thread, five of eight slots, 18 -> 25; static 2205 wide, six of eight
// 61 -> 77).  Everywhere else the overlap gains its microsecond or costs nothing
// (static 1960 x 21, 161 x 256 2.3 -> 1.9; dist 461 x 145, 577 x 256 3.2 -> 2.8;
// dynamic(8), two of eight slots, 4.7 -> 4.3).
inline bool overlap_uneven(uint64_t n, int sched, uint32_t teams, uint32_t threads, int sm_count) {
  if (teams <= (uint32_t)sm_count) return false;
  const double an_sm = std::ceil((double)teams / sm_count);
  const double slots = threads < 1024 ? 1024 / threads : 1;
  const double full = teams / (sm_count * an_sm), spare = slots / an_sm;
  return full >= 0.7 && spare >= 1.1 && spare < 1.8 &&
         n >= (sched == kDist ? 12ull : 4ull) * teams * threads;
}

// 2-D stencil by block windows (k_stencil_window.cu); smem 0: not this form, either
// because it does not apply (a window beyond `budget` bytes, arrays off 16 and 32
// bytes) or because it loses.  A team loads its block and two grid rows and runs
// it with its own warps only, where the row ring and the streamed ring share rows
// among the teams of a CTA and the plain form has every warp an SM holds.  Measured
// others -> windows (us, G x T teams x threads), 1500 launches:
//   - pieces under 8 points (16 under static) and blocks under 1024 points on grids
//     of whole 16-byte units (700 x 600, static(64), 608 x 256: 6.0 -> 6.7) or with
//     chunks under 32 (293 x 1034, static(8), 1142 x 256: 7.3 -> 8.8): others;
//   - blocks under 16 points: others (dynamic(32), 5 x 1737 on 3378 x 256 13.7 -> 21.4);
//   - pieces under 24 points on grids up to three columns wide (static(8), 3 x 444,749
//     on 864 x 1024 17.0 -> 24.1), and where blocks and rows are whole 32-byte
//     sectors, so that the plain form reads vectors: others (static(8), 4096^2 on
//     8192 x 32 36 -> 88, on 1024 x 32 90 -> 176; static, 16 points a thread, 2048^2 on
//     4096 x 64 12 -> 20; but with halos below 0.4 of a block windows: static(16), 8 x
//     1,741,190 on 9519 x 32 148 -> 53); static(c) of such short pieces also on blocks
//     under 1536 points with four times the halo (static(16), 4096 x 47 on 188 x 1024
//     6.5 -> 9.0);
//   - static(c), c from 32 to 63, where the windows an SM holds at once have at most two
//     warps, in more than one wave: lane pieces on odd grids but for the chunks of whole
//     sectors beyond 32, whose lanes spread over the banks (static(32), 289 x 16,457 on
//     163 x 32 127 -> 180, static(61), 5369 x 3082 on 700 x 32 106 -> 229; static(40), 847 x
//     6781 on 181 x 32 148 -> 102); the row ring up to c = 39 on rows of 2048 to 4999 points
//     (static(32), 2548 x 5652 on 276 x 32 147 -> 250; 192 x 61,956 on 265 x 64 327 -> 127,
//     5536 x 2774 on 897 x 32 193 -> 119, static(44), 5236 x 1843 on 554 x 32 146 -> 77).
//     Of 128 random launches of this kind it is the slower choice in 3;
//   - dynamic on grids of whole units, teams of up to 384 threads: the row ring and
//     the streamed ring with twelve teams an SM on, but for small halos (4096^2,
//     dynamic(100) on 8192 x 32 45 -> 74, on 2048 x 128 44 -> 45; dynamic(256) on 16,000
//     x 32 105 -> 158), and where fewer than 77 lanes an SM get a chunk, but for short
//     blocks of more than a row (dynamic(1000), 16 x 306,391 on 1091 x 64 52 -> 99,
//     2048 x 39 on 39 x 32 14 -> 27; dynamic(256), 2236 x 398 on 525 x 256 20.7 ->
//     14.8);
//   - nonmonotonic with three and more rows a block and many waves: others (4096^2,
//     nonmonotonic(100) on 16,000 x 32 80 -> 111).
struct WindowPlan {
  size_t smem;
  uint64_t floats;  // the window's
  uint32_t lead;    // of them before the block's first sector: nx rounded up to 8, and 8
};
inline bool window_gain(const PlanDevice& c, uint64_t nx, uint64_t n, int sched, uint64_t chunk,
                        uint64_t piece, uint32_t teams, uint32_t threads, size_t smem) {
  const uint64_t block = (n - 1) / teams + 1;
  const bool whole = sched == kStatic, few = piece < 24, odd = nx % 4 != 0;
  if (block < 16 || (few && nx <= 3)) return false;
  // rows of halo a block, resident CTAs an SM, lanes an SM that get a chunk
  const double halo = 2.0 * (double)nx / (double)block;
  if (few && (whole || sched == kChunked) && halo >= 0.4 && nx % 8 == 0 &&
      n % (8ull * teams) == 0 && (!whole || n % (8ull * teams * threads) == 0))
    return false;
  if (few && sched == kChunked && block < 1536 && halo >= 4) return false;
  const double fit = std::fmin(std::fmin(threads < 1024 ? 1024 / threads : 1, 32),
                               std::fmax(1, std::floor((double)c.smem_per_sm / (smem + 1624.0))));
  const double resident = std::fmin(fit, std::ceil((double)teams / c.sm_count));
  if (sched == kNonmono) return halo <= 6 || teams <= 5 * c.sm_count * fit;
  if (sched == kChunked && chunk >= 32 && chunk < 64 && fit * threads <= 64 &&
      teams > c.sm_count * fit &&
      (odd ? chunk % 8 || chunk == 32 : chunk < 40 && nx >= 2048 && nx < 5000))
    return false;
  if (sched != kDynamic || odd || threads > 384) return true;
  if (teams > 12u * (uint32_t)c.sm_count) return threads >= 64 && halo <= 1.5;
  const uint64_t chunks = (block - 1) / chunk + 1;
  const double lanes = resident * std::fmin((double)chunks, threads);
  return lanes > 76 || (block <= 24ull * threads && halo > 0.12);
}
inline WindowPlan window_plan(const PlanDevice& c, int64_t budget, bool aligned, uint64_t nx,
                              uint64_t ny, int sched, uint64_t chunk, uint32_t teams,
                              uint32_t threads) {
  const WindowPlan none = {0, 0, 0u};
  const bool whole = sched == kStatic, odd = nx % 4 != 0;
  const uint64_t n = nx * ny;
  if ((!whole && sched != kChunked && sched != kDynamic && sched != kNonmono) || n == 0 ||
      nx >= (1ull << 24) || ny >= (1ull << 31) || !aligned)
    return none;
  const uint64_t block = (n - 1) / teams + 1, piece = whole ? block / threads : chunk;
  if (piece < (whole ? 16u : 8u) || block > (1ull << 24) ||
      (block < 1024 && (!odd || piece < 32)))
    return none;
  // block, rounded to sectors on both sides, a row and a sector on each side
  WindowPlan p;
  p.lead = (uint32_t)((nx + 7) / 8 * 8 + 8);
  p.floats = block + 16 + 2 * (uint64_t)p.lead + 8;
  p.smem = (size_t)(p.floats + 3) / 4 * 16;
  if ((int64_t)p.smem > budget) return none;
  return window_gain(c, nx, n, sched, chunk, piece, teams, threads, p.smem) ? p : none;
}

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
