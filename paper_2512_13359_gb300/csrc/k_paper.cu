// k_paper.cu -- CUDA-core kernels of the paper's own environment (paper
// §IV-B; device code in paper_device.cuh) without networks: reset, action
// replay and observation.  One thread per env.
#include "auv_kernels.h"
#include "paper_device.cuh"

namespace auv {

namespace {

using paper::kAct;
using paper::kObs;

__global__ void __launch_bounds__(256) k_paper_reset(const Model M, Buffers B,
                                                     const uint8_t* __restrict__ mask) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= M.n) return;
  if (mask && !mask[i]) return;
  paper::Env e;
  e.ep = B.episode[i];
  paper::reset_env(M, M.id_base + (uint32_t)i, e, paper::hist_rows(B.state, M.n, i));
  paper::store_env(M, B.state, B.params, B.t_ep, B.episode, i, e);
}

constexpr int kReplayThreads = 128;

__global__ void __launch_bounds__(kReplayThreads, 4) k_paper_replay(const Model M, Buffers B,
                                                      const float* __restrict__ act, int T,
                                                      float* __restrict__ rew,
                                                      uint8_t* __restrict__ done, float* trace,
                                                      Status* st) {
  // The action history lives in shared memory for the whole launch (one
  // column per thread, copied in and out once): its reads every step are
  // shared-memory loads instead of L2 round trips.
  __shared__ float hist[6 * paper::kHist * kReplayThreads];
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= M.n) return;
  const size_t n = (size_t)M.n;
  const paper::HistS h{hist + threadIdx.x, kReplayThreads};
  for (int r = 0; r < 6 * paper::kHist; ++r) h.st(r, B.state[(13 + r) * n + i]);
  paper::Env e;
  paper::load_env(M, B.state, B.params, B.t_ep, B.episode, i, e);
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
    const float r = paper::physics_step(M, M.id_base + (uint32_t)i, e, a, h, &d);
    rew[(size_t)t * n + i] = r;
    done[(size_t)t * n + i] = d ? 1 : 0;
    if (trace) paper::trace_state(M, h, trace + (size_t)t * paper::kStateF * n, i, e);
    bad |= !paper::env_finite(e);
  }
  if (bad) flag_nan(st, i);
  paper::store_env(M, B.state, B.params, B.t_ep, B.episode, i, e);
  for (int r = 0; r < 6 * paper::kHist; ++r) B.state[(13 + r) * n + i] = h.ld(r);
}

__global__ void __launch_bounds__(256) k_paper_observe(const Model M, Buffers B,
                                                       float* __restrict__ obs) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= M.n) return;
  paper::Env e;
  paper::load_env(M, B.state, B.params, B.t_ep, B.episode, i, e);
  float o[kObs];
  paper::observe(e, o);
#pragma unroll
  for (int k = 0; k < kObs; ++k) obs[(size_t)k * M.n + i] = o[k];
}

inline int blocks_for(int n, int b) { return (n + b - 1) / b; }

}  // namespace

cudaError_t launch_paper_reset(const Model& M, const Buffers& B, const uint8_t* mask,
                               cudaStream_t s) {
  k_paper_reset<<<blocks_for(M.n, 256), 256, 0, s>>>(M, B, mask);
  return cudaGetLastError();
}

cudaError_t launch_paper_replay(const Model& M, const Buffers& B, const float* act, int T,
                                float* rew, uint8_t* done, float* trace, Status* st,
                                cudaStream_t s) {
  k_paper_replay<<<blocks_for(M.n, kReplayThreads), kReplayThreads, 0, s>>>(M, B, act, T, rew,
                                                                             done, trace, st);
  return cudaGetLastError();
}

cudaError_t launch_paper_observe(const Model& M, const Buffers& B, float* obs, cudaStream_t s) {
  k_paper_observe<<<blocks_for(M.n, 256), 256, 0, s>>>(M, B, obs);
  return cudaGetLastError();
}

}  // namespace auv
