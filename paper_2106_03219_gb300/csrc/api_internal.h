// Internal host-side declarations shared by the C-ABI translation units.
#pragma once

#include <atomic>
#include <cstdint>

#include "launch.h"
#include "omprt.h"

struct omprt_ctx {
  int device = 0;
  int sm_count = 0;
  int l2_bytes = 0;
  int max_smem_optin = 0;
  int smem_per_sm = 0;
  uint32_t* status_dev = nullptr;
  unsigned char* slots_dev = nullptr;
  unsigned char* pool_dev = nullptr;
  float* mlp_part_dev = nullptr;   // MLP partial gradients, one a CTA (one CTA an SM)
  uint32_t stack_bytes = 0;
  uint32_t stage_bytes = 32768;    // per-team shared memory for staged dynamic schedules
  uint32_t stencil_stage_bytes = 0;  // per-CTA shared memory for the staged 2-D stencil windows
  uint32_t slab_floats = 0;   // 2-D stencil slabs: floats a line (16 / 32; 0 the default)
  uint32_t slab_buffers = 0;  // and buffers a warp (2 .. 4; 0 the default)
  bool launch_overlap = true;  // executor launches overlap the previous grid's tail
  std::atomic<uint32_t> next_slot{0};
  // learned schedule (host copy of the model)
  bool has_model = false;
  // W1, W2, W3 with the outputs of one input side by side (W[in][out]), so that
  // inference runs over outputs in vector registers; b1, b2, b3 as they are
  float w1t[OMPRT_MLP_IN * OMPRT_MLP_HID], w2t[OMPRT_MLP_HID * OMPRT_MLP_HID],
      w3t[OMPRT_MLP_HID * OMPRT_MLP_OUT];
  float b1[OMPRT_MLP_HID], b2[OMPRT_MLP_HID], b3[OMPRT_MLP_OUT];
  float feat_mean[OMPRT_MLP_IN];
  float feat_std[OMPRT_MLP_IN];
};

// MLP training batch limit, and the floats of one partial gradient (the
// parameters, the loss, padding to 16 bytes).
constexpr int kMlpMaxBatch = 16384;
constexpr int kMlpPartFloats = 6032;

struct DeviceGuard {
  int prev = 0;
  bool changed = false;
  explicit DeviceGuard(int dev);
  ~DeviceGuard();
};

struct ScratchSlot {
  uint32_t* ticket;
  unsigned char* partials;
  unsigned long long* dyn_next;
};
ScratchSlot ctx_next_slot(omprt_ctx* ctx);

omprt_status loop_trip_count(const omprt_loop_desc* d, uint64_t* n, int64_t* wide_lb);

// Teams of a schedule(auto) launch of a one-dimensional body that get an
// iteration: the mapping hands 32-byte vectors to threads in order, grid-stride,
// so with fewer vectors than threads the teams after the last vector run
// nothing.  They are not launched: the others' iterations are the same, and a
// reduction has fewer partials to wait for (10,007 int64 values on 304 x 512: 5
// teams instead of 304, 4.2 -> 4.0 us; one team 4.0 -> 1.9; without allocation,
// 4096 teams by default, 36 -> 8.3).
int32_t auto_teams(int32_t body, int32_t data_type, uintptr_t pointers, uint64_t n, int32_t teams,
                   int32_t threads);

struct LearnedConfig {
  int32_t sched;
  int64_t chunk;
  int32_t teams_per_sm;
  int32_t threads;
};
LearnedConfig learned_config(int k);
