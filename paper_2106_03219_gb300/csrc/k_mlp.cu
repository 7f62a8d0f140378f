// MLP cost model 16 -> 64 -> 64 -> 12 (fp32): forward, loss + gradient, Adam.
//
// The model has 6028 parameters and a batch a few hundred samples, so every
// call is bound by latency: launches, dependent loads, chains of adds.  A CTA
// takes eight samples at a time through the whole model out of shared memory;
// for training it keeps its share of every gradient in registers (each thread
// a 4 x 4 tile of dW2 and its pieces of the rest), adds all its samples to
// them in order, and leaves one partial gradient.  A second kernel adds the
// CTAs' partials in CTA order (deterministic, no atomics).  Both, and the Adam
// step, overlap the launch before them.
// Measured, batch 256 (one sample a warp and one thread a parameter walking the
// batch -> now): under ncu 10.3 + 57.3 -> 8.6 + 4.4 us; a step with Adam through
// the Python binding 43 -> 10 us, what the two host calls take; batch 2048
// 226 -> 19.4, batch 16000 1666 -> 66 us.
#include <cmath>

#include "api_internal.h"

namespace rt {

constexpr int kIn = OMPRT_MLP_IN, kHid = OMPRT_MLP_HID, kOut = OMPRT_MLP_OUT;
constexpr int kOffW1 = 0, kOffB1 = kOffW1 + kHid * kIn, kOffW2 = kOffB1 + kHid,
              kOffB2 = kOffW2 + kHid * kHid, kOffW3 = kOffB2 + kHid,
              kOffB3 = kOffW3 + kOut * kHid, kNParam = kOffB3 + kOut;
static_assert(kNParam == OMPRT_MLP_NPARAM, "parameter layout");

constexpr int kS = 8;          // samples a CTA takes at a time
constexpr int kThreads = 256;  // 64 units x 4 pairs of samples
// Padded strides: rows start 4 banks apart, so that eight lanes reading the
// same 16 bytes of eight rows hit all 32 banks.
constexpr int kP1 = kIn + 4, kP2 = kHid + 4;

struct MlpShared {
  alignas(16) float w1[kHid * kP1];
  alignas(16) float w2[kHid * kP2];
  alignas(16) float w3[kOut * kP2];
  float b1[kHid], b2[kHid], b3[kOut];
  alignas(16) float x[kS][kIn];
  alignas(16) float h1[kS][kP2], h2[kS][kP2], d1[kS][kP2], d2[kS][kP2];
  float dy[kS][kOut], lt[kS][kOut], yt[kS][kOut];
};

// where parameter k lies in shared memory
__device__ __forceinline__ float* param_slot(MlpShared& S, int k) {
  if (k < kOffB1) return S.w1 + k / kIn * kP1 + k % kIn;
  if (k < kOffW2) return S.b1 + (k - kOffB1);
  if (k < kOffB2) return S.w2 + (k - kOffW2) / kHid * kP2 + (k - kOffW2) % kHid;
  if (k < kOffW3) return S.b2 + (k - kOffB2);
  if (k < kOffB3) return S.w3 + (k - kOffW3) / kHid * kP2 + (k - kOffW3) % kHid;
  return S.b3 + (k - kOffB3);
}

__device__ __forceinline__ void load_weights(MlpShared& S, const float* __restrict__ p) {
  if (((uintptr_t)p & 15) == 0) {  // no group of four straddles a row or a layer
    static_assert(kOffB1 % 4 == 0 && kOffW2 % 4 == 0 && kOffB2 % 4 == 0 && kOffW3 % 4 == 0 &&
                      kOffB3 % 4 == 0 && kNParam % 4 == 0,
                  "groups of four");
    constexpr int kN = (kNParam / 4 + kThreads - 1) / kThreads;
    float4 v[kN];
#pragma unroll
    for (int j = 0; j < kN; ++j) {
      const int k = threadIdx.x + j * kThreads;
      if (k < kNParam / 4) v[j] = ((const float4*)p)[k];
    }
#pragma unroll
    for (int j = 0; j < kN; ++j) {
      const int k = threadIdx.x + j * kThreads;
      if (k < kNParam / 4) {
        float* const d = param_slot(S, 4 * k);
        d[0] = v[j].x;
        d[1] = v[j].y;
        d[2] = v[j].z;
        d[3] = v[j].w;
      }
    }
  } else {
    for (int k = threadIdx.x; k < kNParam; k += kThreads) *param_slot(S, k) = p[k];
  }
}

__device__ __forceinline__ float4 ld4(const float* p) { return *(const float4*)p; }
// acc + w . v over four consecutive terms, in order
__device__ __forceinline__ float fma4(float4 w, float4 v, float acc) {
  acc = __fmaf_rn(w.x, v.x, acc);
  acc = __fmaf_rn(w.y, v.y, acc);
  acc = __fmaf_rn(w.z, v.z, acc);
  return __fmaf_rn(w.w, v.w, acc);
}

// kTrain false: write Y; true: add the batch's gradient and loss terms and
// leave this CTA's sums in part[blockIdx.x].
template <bool kTrain>
__global__ void __launch_bounds__(kThreads) mlp_kernel(const float* __restrict__ p,
                                                       const float* __restrict__ X,
                                                       const float* __restrict__ Yt, int B,
                                                       float scale, float* __restrict__ Y,
                                                       float* __restrict__ part) {
  enter_region_grid();
  __shared__ MlpShared S;
  const int t = threadIdx.x;
  load_weights(S, p);
  const int u = t % kHid, s0 = t / kHid * 2;  // this thread's unit and two samples
  const int o4 = t / 16 * 4, i4 = t % 16 * 4;  // its tile of dW2; rows of dW3
  const int o1 = t / 4, i1 = t % 4 * 4;        // its piece of dW1
  float g2[4][4] = {}, g1[4] = {}, g3[4] = {}, gb = 0.f;
  for (int b0 = blockIdx.x * kS; b0 < B; b0 += gridDim.x * kS) {
    const int ns = B - b0 < kS ? B - b0 : kS;
    // Samples beyond the batch run on zeros.  For training their activations are
    // zeros too, so that they add nothing: what the weights make of an input of
    // zeros may be beyond fp32's range where no sample of the batch is.
    const bool real0 = !kTrain || s0 < ns, real1 = !kTrain || s0 + 1 < ns;
    if (t < kS * kIn) S.x[t / kIn][t % kIn] = t < ns * kIn ? X[(size_t)b0 * kIn + t] : 0.f;
    if (kTrain && t >= 128 && t < 128 + kS * kOut) {
      const int q = t - 128;
      S.yt[q / kOut][q % kOut] = q < ns * kOut ? Yt[(size_t)b0 * kOut + q] : 0.f;
    }
    __syncthreads();
    // layer 1
    float a0 = S.b1[u], a1 = a0;
#pragma unroll
    for (int k = 0; k < kIn; k += 4) {
      const float4 w = ld4(S.w1 + u * kP1 + k);
      a0 = fma4(w, ld4(&S.x[s0][k]), a0);
      a1 = fma4(w, ld4(&S.x[s0 + 1][k]), a1);
    }
    const float h1a = real0 ? fmaxf(a0, 0.f) : 0.f, h1b = real1 ? fmaxf(a1, 0.f) : 0.f;
    S.h1[s0][u] = h1a;
    S.h1[s0 + 1][u] = h1b;
    __syncthreads();
    // layer 2
    a0 = a1 = S.b2[u];
#pragma unroll 4
    for (int k = 0; k < kHid; k += 4) {
      const float4 w = ld4(S.w2 + u * kP2 + k);
      a0 = fma4(w, ld4(&S.h1[s0][k]), a0);
      a1 = fma4(w, ld4(&S.h1[s0 + 1][k]), a1);
    }
    const float h2a = real0 ? fmaxf(a0, 0.f) : 0.f, h2b = real1 ? fmaxf(a1, 0.f) : 0.f;
    S.h2[s0][u] = h2a;
    S.h2[s0 + 1][u] = h2b;
    __syncthreads();
    // layer 3: a thread an output
    if (t < kS * kOut) {
      const int s = t / kOut, o = t % kOut;
      float y0 = S.b3[o], y1 = 0.f;  // two chains over halves of the inputs
#pragma unroll 4
      for (int k = 0; k < kHid / 2; k += 4) {
        y0 = fma4(ld4(S.w3 + o * kP2 + k), ld4(&S.h2[s][k]), y0);
        y1 = fma4(ld4(S.w3 + o * kP2 + kHid / 2 + k), ld4(&S.h2[s][kHid / 2 + k]), y1);
      }
      const float y = __fadd_rn(y0, y1);
      if constexpr (!kTrain) {
        if (s < ns) Y[(size_t)b0 * kOut + t] = y;
      } else {
        const float d = s < ns ? __fsub_rn(y, S.yt[s][o]) : 0.f;
        S.lt[s][o] = __fmul_rn(d, d);
        S.dy[s][o] = __fmul_rn(__fmul_rn(2.f, d), scale);
      }
    }
    if constexpr (kTrain) {
      __syncthreads();
      // dh2 = relu'(h2) * W3^T dy
      a0 = a1 = 0.f;
#pragma unroll
      for (int o = 0; o < kOut; ++o) {
        const float w = S.w3[o * kP2 + u];
        a0 = __fmaf_rn(w, S.dy[s0][o], a0);
        a1 = __fmaf_rn(w, S.dy[s0 + 1][o], a1);
      }
      S.d2[s0][u] = h2a > 0.f ? a0 : 0.f;
      S.d2[s0 + 1][u] = h2b > 0.f ? a1 : 0.f;
      __syncthreads();
      // dh1 = relu'(h1) * W2^T dh2
      a0 = a1 = 0.f;
#pragma unroll 4
      for (int k = 0; k < kHid; k += 4) {
        const float4 w = make_float4(S.w2[k * kP2 + u], S.w2[(k + 1) * kP2 + u],
                                     S.w2[(k + 2) * kP2 + u], S.w2[(k + 3) * kP2 + u]);
        a0 = fma4(w, ld4(&S.d2[s0][k]), a0);
        a1 = fma4(w, ld4(&S.d2[s0 + 1][k]), a1);
      }
      S.d1[s0][u] = h1a > 0.f ? a0 : 0.f;
      S.d1[s0 + 1][u] = h1b > 0.f ? a1 : 0.f;
      __syncthreads();
      // this thread's share of the gradients, sample by sample
#pragma unroll
      for (int s = 0; s < kS; ++s) {
        const float4 d = ld4(&S.d2[s][o4]), h = ld4(&S.h1[s][i4]);
        const float dv[4] = {d.x, d.y, d.z, d.w}, hv[4] = {h.x, h.y, h.z, h.w};
#pragma unroll
        for (int r = 0; r < 4; ++r)
#pragma unroll
          for (int c = 0; c < 4; ++c) g2[r][c] = __fmaf_rn(dv[r], hv[c], g2[r][c]);
        const float4 xv = ld4(&S.x[s][i1]);
        const float e = S.d1[s][o1];
        g1[0] = __fmaf_rn(e, xv.x, g1[0]);
        g1[1] = __fmaf_rn(e, xv.y, g1[1]);
        g1[2] = __fmaf_rn(e, xv.z, g1[2]);
        g1[3] = __fmaf_rn(e, xv.w, g1[3]);
        if (t < kOut * 16) {
          const float4 hh = ld4(&S.h2[s][i4]);
          const float f = S.dy[s][t / 16];
          g3[0] = __fmaf_rn(f, hh.x, g3[0]);
          g3[1] = __fmaf_rn(f, hh.y, g3[1]);
          g3[2] = __fmaf_rn(f, hh.z, g3[2]);
          g3[3] = __fmaf_rn(f, hh.w, g3[3]);
        }
      }
      if (t < kHid) {  // biases, and the loss in the last of them
#pragma unroll
        for (int s = 0; s < kS; ++s) gb = __fadd_rn(gb, S.d1[s][t]);
      } else if (t < 2 * kHid) {
#pragma unroll
        for (int s = 0; s < kS; ++s) gb = __fadd_rn(gb, S.d2[s][t - kHid]);
      } else if (t < 2 * kHid + kOut) {
#pragma unroll
        for (int s = 0; s < kS; ++s) gb = __fadd_rn(gb, S.dy[s][t - 2 * kHid]);
      } else if (t == 2 * kHid + kOut) {
        for (int s = 0; s < kS; ++s)
#pragma unroll
          for (int o = 0; o < kOut; ++o) gb = __fadd_rn(gb, S.lt[s][o]);
      }
    }
    __syncthreads();  // the samples' rows are free
  }
  if constexpr (kTrain) {
    float* const g = part + (size_t)blockIdx.x * kMlpPartFloats;
#pragma unroll
    for (int r = 0; r < 4; ++r)
      *(float4*)(g + kOffW2 + (o4 + r) * kHid + i4) =
          make_float4(g2[r][0], g2[r][1], g2[r][2], g2[r][3]);
    *(float4*)(g + kOffW1 + o1 * kIn + i1) = make_float4(g1[0], g1[1], g1[2], g1[3]);
    if (t < kOut * 16)
      *(float4*)(g + kOffW3 + t / 16 * kHid + i4) = make_float4(g3[0], g3[1], g3[2], g3[3]);
    if (t < kHid)
      g[kOffB1 + t] = gb;
    else if (t < 2 * kHid)
      g[kOffB2 + t - kHid] = gb;
    else if (t <= 2 * kHid + kOut)
      g[kOffB3 + t - 2 * kHid] = gb;  // the loss follows the last parameter
  }
}

// Adds the n partial gradients.  A CTA: 32 columns of four parameters x 8
// slices of the partials, each slice in order, then the slices in order.
constexpr int kSlices = 8;
__global__ void __launch_bounds__(32 * kSlices) mlp_combine_kernel(const float* __restrict__ part,
                                                                   int n, float scale,
                                                                   float* __restrict__ grad,
                                                                   float* __restrict__ loss) {
  enter_region_grid();
  __shared__ float4 acc[kSlices][32];
  const int l = threadIdx.x % 32, w = threadIdx.x / 32;
  const int col = blockIdx.x * 32 + l;
  if (col < kMlpPartFloats / 4) {
    const int lo = n * w / kSlices, hi = n * (w + 1) / kSlices;
    float4 s = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll 4
    for (int c = lo; c < hi; ++c) {
      const float4 v = __ldcg((const float4*)(part + (size_t)c * kMlpPartFloats) + col);
      s.x = __fadd_rn(s.x, v.x);
      s.y = __fadd_rn(s.y, v.y);
      s.z = __fadd_rn(s.z, v.z);
      s.w = __fadd_rn(s.w, v.w);
    }
    acc[w][l] = s;
  }
  __syncthreads();
  if (threadIdx.x >= 128) return;
  const int q = blockIdx.x * 128 + threadIdx.x;  // a thread a parameter
  float s = 0.f;
#pragma unroll
  for (int k = 0; k < kSlices; ++k) s = __fadd_rn(s, ((const float*)acc[k])[threadIdx.x]);
  if (q < kNParam)
    grad[q] = s;
  else if (q == kNParam && loss)
    *loss = __fmul_rn(s, scale);
}

__global__ void adam_kernel(float* __restrict__ p, const float* __restrict__ g, float* __restrict__ m,
                            float* __restrict__ v, int n, float lr, float b1, float b2, float eps,
                            float c1, float c2) {
  enter_region_grid();
  const int k = blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= n) return;
  const float gk = g[k];
  const float mk = __fadd_rn(__fmul_rn(b1, m[k]), __fmul_rn(__fsub_rn(1.f, b1), gk));
  const float vk =
      __fadd_rn(__fmul_rn(b2, v[k]), __fmul_rn(__fmul_rn(__fsub_rn(1.f, b2), gk), gk));
  m[k] = mk;
  v[k] = vk;
  const float mh = __fdiv_rn(mk, c1), vh = __fdiv_rn(vk, c2);
  p[k] = __fsub_rn(p[k], __fdiv_rn(__fmul_rn(lr, mh), __fadd_rn(__fsqrt_rn(vh), eps)));
}

}  // namespace rt

using namespace rt;

static_assert(kMlpPartFloats >= kNParam + 1 && kMlpPartFloats % 4 == 0, "partial gradient size");

static int mlp_groups(int B) { return (B + kS - 1) / kS; }

extern "C" {

omprt_status omprt_mlp_forward(omprt_ctx* c, const float* params, const float* x, int32_t B,
                               float* y, void* stream) {
  if (!c) return OMPRT_ERR_NOT_INIT;
  if (!params || B < 0 || (B && (!x || !y))) return OMPRT_ERR_INVALID;
  if (B == 0) return OMPRT_OK;
  DeviceGuard guard(c->device);
  OverlapScope overlap(c->launch_overlap, (size_t)c->smem_per_sm);
  const int groups = mlp_groups(B), most = 4 * c->sm_count;
  return launch_kernel(mlp_kernel<false>, dim3(groups < most ? groups : most), dim3(kThreads), 0,
                       (cudaStream_t)stream, params, x, nullptr, B, 0.f, y,
                       nullptr) == cudaSuccess
             ? OMPRT_OK
             : OMPRT_ERR_CUDA;
}

omprt_status omprt_mlp_loss_grad(omprt_ctx* c, const float* params, const float* x,
                                 const float* target, int32_t B, float* grad, float* loss,
                                 void* stream) {
  if (!c) return OMPRT_ERR_NOT_INIT;
  if (!params || !x || !target || !grad || B < 1 || B > kMlpMaxBatch) return OMPRT_ERR_INVALID;
  DeviceGuard guard(c->device);
  OverlapScope overlap(c->launch_overlap, (size_t)c->smem_per_sm);
  const float scale = 1.0f / ((float)B * kOut);
  cudaStream_t st = (cudaStream_t)stream;
  // one CTA a group of samples, at most one an SM: more would only add
  // partials for the second kernel to read
  const int groups = mlp_groups(B), n = groups < c->sm_count ? groups : c->sm_count;
  if (launch_kernel(mlp_kernel<true>, dim3(n), dim3(kThreads), 0, st, params, x, target, B, scale,
                    nullptr, c->mlp_part_dev) != cudaSuccess)
    return OMPRT_ERR_CUDA;
  return launch_kernel(mlp_combine_kernel, dim3((kNParam + 1 + 127) / 128), dim3(32 * kSlices), 0,
                       st, c->mlp_part_dev, n, scale, grad, loss) == cudaSuccess
             ? OMPRT_OK
             : OMPRT_ERR_CUDA;
}

omprt_status omprt_mlp_adam(omprt_ctx* c, float* params, const float* grad, float* m, float* v,
                            int32_t n, int32_t t, float lr, float beta1, float beta2, float eps,
                            void* stream) {
  if (!c) return OMPRT_ERR_NOT_INIT;
  if (!params || !grad || !m || !v || n < 1 || t < 1) return OMPRT_ERR_INVALID;
  DeviceGuard guard(c->device);
  OverlapScope overlap(c->launch_overlap, (size_t)c->smem_per_sm);
  const float c1 = (float)(1.0 - std::pow((double)beta1, (double)t));
  const float c2 = (float)(1.0 - std::pow((double)beta2, (double)t));
  return launch_kernel(adam_kernel, dim3((n + 127) / 128), dim3(128), 0, (cudaStream_t)stream,
                       params, grad, m, v, n, lr, beta1, beta2, eps, c1, c2) == cudaSuccess
             ? OMPRT_OK
             : OMPRT_ERR_CUDA;
}

}  // extern "C"
