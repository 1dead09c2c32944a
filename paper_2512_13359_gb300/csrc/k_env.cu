// k_env.cu -- CUDA-core kernels of the batched AUV rollout without networks:
// episode reset, action replay, observation and raw Philox words.
// One thread owns one environment for the whole launch; its state lives in
// registers across all T control steps and touches HBM only at the start and
// the end (plus the trajectory rows it writes).
#include "auv_kernels.h"

namespace auv {

// ---------------------------------------------------------------------------
// Reset: env i starts a new episode if mask == NULL or mask[i] != 0.
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(256) k_reset(const Model M, Buffers B, const uint8_t* mask) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= M.n) return;
  if (mask && !mask[i]) return;
  Env e;
  e.ep = B.episode[i];
  reset_env(M, M.id_base + (uint32_t)i, e);
  store_env(M, B.state, B.params, B.t_ep, B.episode, i, e);
}

// ---------------------------------------------------------------------------
// Action replay: T control steps with given actions act[T][8][N].
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(128, 4) k_replay(const Model M, Buffers B,
                                                const float* __restrict__ act, int T,
                                                float* __restrict__ rew, uint8_t* __restrict__ done,
                                                float* __restrict__ trace, Status* st) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= M.n) return;
  const size_t n = (size_t)M.n;
  Env e;
  load_env(M, B.state, B.params, B.t_ep, B.episode, i, e);
  bool bad = false;
  // Step t + 1's actions are loaded while step t integrates, so their DRAM
  // latency is hidden behind a step of arithmetic.
  float a_next[kAct];
#pragma unroll
  for (int k = 0; k < kAct; ++k) a_next[k] = T > 0 ? __ldg(act + (size_t)k * n + i) : 0.0f;
  for (int t = 0; t < T; ++t) {
    float a[kAct];
#pragma unroll
    for (int k = 0; k < kAct; ++k) a[k] = a_next[k];
    if (t + 1 < T) {
#pragma unroll
      for (int k = 0; k < kAct; ++k)
        a_next[k] = __ldg(act + ((size_t)(t + 1) * kAct + k) * n + i);
    }
    bool d;
    const float r = physics_step(M, M.id_base + (uint32_t)i, e, a, &d);
    rew[(size_t)t * n + i] = r;
    done[(size_t)t * n + i] = d ? 1 : 0;
    if (trace) store_state(M, trace + (size_t)t * kStateF * n, i, e);
    bad |= !env_finite(e);
  }
  if (bad) flag_nan(st, i);
  store_env(M, B.state, B.params, B.t_ep, B.episode, i, e);
}

__global__ void __launch_bounds__(256) k_observe(const Model M, Buffers B, float* __restrict__ obs) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= M.n) return;
  Env e;
  load_env(M, B.state, B.params, B.t_ep, B.episode, i, e);
  float o[kObs];
  observe(e, o);
#pragma unroll
  for (int k = 0; k < kObs; ++k) obs[(size_t)k * M.n + i] = o[k];
}

__global__ void __launch_bounds__(256) k_draw_words(const Model M, uint32_t stream_id,
                                                    uint64_t index, int n_blocks,
                                                    uint32_t* __restrict__ out) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= M.n) return;
  const size_t n = (size_t)M.n;
  for (int b = 0; b < n_blocks; ++b) {
    const uint4 r = philox10((uint32_t)index, (uint32_t)(index >> 32), stream_id, (uint32_t)b,
                             M.id_base + (uint32_t)i, M.seed);
    out[(size_t)(4 * b + 0) * n + i] = r.x;
    out[(size_t)(4 * b + 1) * n + i] = r.y;
    out[(size_t)(4 * b + 2) * n + i] = r.z;
    out[(size_t)(4 * b + 3) * n + i] = r.w;
  }
}

// ---------------------------------------------------------------------------
// Host-side launchers (called from the C ABI layer).
// ---------------------------------------------------------------------------
static inline int blocks_for(int n, int b) { return (n + b - 1) / b; }

cudaError_t launch_reset(const Model& M, const Buffers& B, const uint8_t* mask, cudaStream_t s) {
  k_reset<<<blocks_for(M.n, 256), 256, 0, s>>>(M, B, mask);
  return cudaGetLastError();
}

cudaError_t launch_replay(const Model& M, const Buffers& B, const float* act, int T, float* rew,
                          uint8_t* done, float* trace, Status* st, cudaStream_t s) {
  k_replay<<<blocks_for(M.n, 128), 128, 0, s>>>(M, B, act, T, rew, done, trace, st);
  return cudaGetLastError();
}

cudaError_t launch_observe(const Model& M, const Buffers& B, float* obs, cudaStream_t s) {
  k_observe<<<blocks_for(M.n, 256), 256, 0, s>>>(M, B, obs);
  return cudaGetLastError();
}

cudaError_t launch_draw_words(const Model& M, uint32_t stream_id, uint64_t index, int n_blocks,
                              uint32_t* out, cudaStream_t s) {
  k_draw_words<<<blocks_for(M.n, 256), 256, 0, s>>>(M, stream_id, index, n_blocks, out);
  return cudaGetLastError();
}

}  // namespace auv
