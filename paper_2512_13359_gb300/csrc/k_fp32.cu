// k_fp32.cu -- the exact-fp32 networks on CUDA cores: the fused rollouts of
// both models and the network evaluations over given rows (policy, value).
//
// A CTA of 256 threads evaluates both hidden layers and the head of a tile of
// E rows as small register-blocked products, so that one weight read serves
// the whole tile.  Per control step the rollout alternates the networks (all
// eight warps) with the per-env work: the tile's first warp holds one env
// per lane (sampling, physics, next observation) while the second draws the
// next step's normals.
//
//   layer 1   thread = hidden unit; its weights in registers (loaded from the
//             image's transposed W1, coalesced), the rows' inputs broadcast
//             from shared memory
//   layer 2   W2 in 16-column slices, all resident for H = 64, else streamed
//             from L2 through a ring of bulk copies that runs on across layers
//             and steps, so the first slices land during the physics.  A warp
//             owns 32 units of up to 32 rows, a thread RM x RN outputs; even
//             and odd k are the two lanes of packed fp32 FMAs.
//   head      one thread per row and pair of outputs
//
// What bounds it: with one CTA per SM, two warps a scheduler, the latencies of
// FMAs and of the operands' shared-memory reads (a thread's 4 x 8 outputs take 12
// 16-byte reads per 64 packed FMAs): FMA pipe 46 %, shared memory 43 % and issue
// 37 % busy, DRAM and L2 idle (4,096 envs).  Measured per control step of a 32-row tile at width 256, one CTA
// per SM: layer 1 5.9k cycles, layer 2 28k (16.4k of FMA), tanh 1.1k, head 4k,
// physics 3.6k.  4,096 envs x 100 steps of the Fossen model: 56.8 ms with one
// thread per env, 2.1 ms now; 64 envs x 200 steps at width 64: 1.16 ms with a
// 64-thread team per env, 0.43 ms now.
//
// Sums keep one order whatever the tile: layer 1 in k from the bias; layer 2
// even k from the bias plus odd k from zero; the head in k from the bias.
#include <algorithm>
#include <cstring>

#include "auv_bf16.h"
#include "auv_kernels.h"
#include "paper_device.cuh"
#include "tc_ptx.cuh"

namespace auv {

namespace {

constexpr int kThreads = 256;
constexpr int kSlice = 16;          // W2 columns per slice
constexpr int kWs = kSlice + 4;     // padded slice row: 8 consecutive rows in distinct banks

constexpr uint64_t kWaitLimitNs = 2000000000ull;   // 2 s per wait

// Offsets (floats) of one network's arrays in its flat weight vector.
template <int IN, int H>
struct Flat {
  static constexpr int kW1 = 0, kB1 = H * IN, kW2 = kB1 + H, kB2 = kW2 + H * H, kW3 = kB2 + H;
};

// One network's packed image (floats): W2 as kSlice-column slices of H rows
// padded to kWs, as they lie in shared memory, then W1 transposed [IN][H].
template <int IN, int H>
struct Image {
  static constexpr int kSlot = H * kWs, kW1T = H / kSlice * kSlot, kFloats = kW1T + IN * H;
};

// The images of one network or (gridDim.y = 2) both.
template <int IN, int H>
__global__ void k_pack_fp32(const float* __restrict__ w0, float* __restrict__ img0, const float* __restrict__ w1,
                            float* __restrict__ img1) {
  using F = Flat<IN, H>;
  using I = Image<IN, H>;
  const float* const w = blockIdx.y ? w1 : w0;
  float* const img = blockIdx.y ? img1 : img0;
  const int x = blockIdx.x * blockDim.x + threadIdx.x;
  if (x < I::kW1T) {
    const int s = x / I::kSlot, u = x % I::kSlot / kWs, k = x % kWs;
    img[x] = k < kSlice ? w[F::kW2 + u * H + s * kSlice + k] : 0.0f;
  } else if (x < I::kFloats) {
    const int k = (x - I::kW1T) / H, u = (x - I::kW1T) % H;
    img[x] = w[F::kW1 + u * IN + k];
  }
}

// A network's flat weights and its image (16-byte aligned device memory).
struct Net {
  const float* w;
  const float* img;
};

// CTAs that share an SM: two 32-row tiles with a three-slot ring, else one
// (whose threads may use up to 255 registers).
constexpr int ctas_per_sm(int E, int H, int SLOTS) {
  return E == 32 && (H == 64 || SLOTS == 3) ? 2 : 1;
}

// Tile shape: E rows, ring of SLOTS W2 slices (H = 64: every slice of both
// networks resident, SLOTS = 8).
template <int IN, int H, int E, int SLOTS>
struct Tile {
  static_assert(H == 64 || H == 256, "hidden width");
  static constexpr int kSlices = H / kSlice;
  static constexpr bool kResident = H == 64;
  static_assert(!kResident || SLOTS >= 2 * kSlices, "both networks resident");
  static constexpr int kXs = (IN + 3) / 4 * 4, kHs = H + 4;
  static constexpr int kUB = H / 32, kEB = 8 / kUB;     // unit blocks, row blocks over 8 warps
  static constexpr int WE = E / kEB;                    // rows of one warp
  static constexpr int EG = WE >= 16 ? 8 : (WE >= 8 ? 4 : 2), RM = WE / EG;
  static constexpr int UG = 32 / EG, RN = 32 / UG;
  static constexpr int kSlot = H * kWs;                 // floats per ring slot
  // shared memory (floats)
  static constexpr int oW = 0, oH = oW + SLOTS * kSlot, oX = oH + E * kHs, oY = oX + E * kXs,
                       oBar = oY + E * 17 + E % 2,      // oY: head outputs, then the value
                       kNet = oBar + 2 * SLOTS + 2;     // a barrier per slot, the abort flag

  // Running position in the sequence of slices [network 0, network 1]
  // repeated over the launch, and the ring's fill state.
  struct Ring {
    float* sm;
    Net net[2];
    int nets, total;   // networks per step; slices of the whole launch
    int q, slot;       // next slice to use, and its ring slot
    uint32_t phase;    // parity of the slot's fill
    int next, next_slot, next_in_step;   // next slice to fetch (thread 0)

    __device__ __forceinline__ uint64_t* bar(int s) const {
      return reinterpret_cast<uint64_t*>(sm + oBar) + s;
    }
    __device__ __forceinline__ volatile int* abort() const {
      return reinterpret_cast<int*>(sm + oBar + 2 * SLOTS);
    }
    // Thread 0: the next slice of the sequence into the next slot, if any is left.
    __device__ __forceinline__ void fetch() {
      if (next >= total || *abort()) return;
      const float* src = next_in_step < kSlices ? net[0].img + next_in_step * kSlot
                                                : net[1].img + (next_in_step - kSlices) * kSlot;
      tc::mbar_arrive_expect_tx(bar(next_slot), kSlot * 4);
      tc::bulk_g2s(sm + oW + next_slot * kSlot, src, kSlot * 4, bar(next_slot));
      ++next;
      next_slot = next_slot + 1 == SLOTS ? 0 : next_slot + 1;
      next_in_step = next_in_step + 1 == nets * kSlices ? 0 : next_in_step + 1;
    }
    // Every thread: barriers, then the first fills (resident: every slice).
    __device__ __forceinline__ void start(float* sm_, const Net& a, const Net& b, int nets_,
                                          int total_, int tid) {
      sm = sm_;
      net[0] = a;
      net[1] = b;
      nets = nets_;
      total = kResident ? nets * kSlices : total_;
      q = slot = next = next_slot = next_in_step = 0;
      phase = 0u;
      if (tid == 0) {
        for (int s = 0; s < SLOTS; ++s) tc::mbar_init(bar(s), 1);
        *abort() = 0;
        tc::mbar_fence_init();
        for (int s = 0; s < (kResident ? SLOTS : SLOTS - 1); ++s) fetch();
      }
      __syncthreads();
      if (kResident)
        for (int s = 0; s < total; ++s) tc::mbar_wait(bar(s), 0, abort(), kWaitLimitNs);
    }
    // Every thread: the next slice has landed and the slot before it is free
    // again (block-wide barrier); thread 0 refills that one.
    __device__ __forceinline__ const float* advance(int tid) {
      tc::mbar_wait(bar(slot), phase, abort(), kWaitLimitNs);
      __syncthreads();
      if (tid == 0) fetch();
      const float* w = sm + oW + slot * kSlot;
      ++q;
      if (++slot == SLOTS) {
        slot = 0;
        phase ^= 1u;
      }
      return w;
    }
    // Thread 0, at the end: a wait that gave up is latched, after the copies
    // still in flight have landed (each again waited for with the limit).
    __device__ __forceinline__ void finish(Status* st) {
      if (!*abort()) return;
      for (int s = 0; s < SLOTS; ++s) {
        const int fills = next / SLOTS + (s < next % SLOTS ? 1 : 0);
        const uint64_t t0 = tc::global_timer_ns();
        while (fills > 0 && !tc::mbar_test(bar(s), (uint32_t)(fills - 1) & 1u) &&
               tc::global_timer_ns() - t0 < kWaitLimitNs) {
        }
      }
      atomicAdd(&st->timeouts, 1);
      atomicCAS(&st->code, 0, -4);
    }
  };

  // One network over the tile: xs -> out_dim outputs per row at sm[oY + row *
  // 17 + y0 + o].  Begins and ends with a block-wide barrier.
  static __device__ __forceinline__ void run(Ring& ring, int net, int out_dim, int y0, int tid) {
    using F = Flat<IN, H>;
    float* sm = ring.sm;
    const float* wt = net ? ring.net[1].w : ring.net[0].w;
    const float* w1t = (net ? ring.net[1].img : ring.net[0].img) + Image<IN, H>::kW1T;
    float* xs = sm + oX;
    float* hs = sm + oH;
    __syncthreads();
    {   // layer 1
      const int u = tid % H;
      float wr[IN];
#pragma unroll
      for (int k = 0; k < IN; ++k) wr[k] = __ldg(w1t + k * H + u);
      const float b = __ldg(wt + F::kB1 + u);
#pragma unroll 4
      for (int e = tid / H; e < E; e += kThreads / H) {
        float s = b;
#pragma unroll
        for (int k4 = 0; k4 < kXs / 4; ++k4) {
          const float4 x = *reinterpret_cast<const float4*>(xs + e * kXs + 4 * k4);
          const float xv[4] = {x.x, x.y, x.z, x.w};
#pragma unroll
          for (int j = 0; j < 4; ++j)
            if (4 * k4 + j < IN) s = fmaf(wr[4 * k4 + j], xv[j], s);
        }
        hs[e * kHs + u] = tanhf(s);
      }
    }
    const int warp = tid >> 5, lane = tid & 31;
    const int eg = (warp / kUB) * WE + lane % EG, ug = (warp % kUB) * 32 + lane / EG;
    float2 acc[RM][RN];
#pragma unroll
    for (int j = 0; j < RN; ++j) {
      const float b = __ldg(wt + F::kB2 + ug + UG * j);
#pragma unroll
      for (int i = 0; i < RM; ++i) acc[i][j] = make_float2(b, 0.0f);
    }
    if (kResident) __syncthreads();   // h1 complete (the ring's own barrier otherwise)
    for (int s = 0; s < kSlices; ++s) {
      const float* ws = kResident ? sm + oW + (net * kSlices + s) * kSlot : ring.advance(tid);
      const float* a0 = hs + eg * kHs + s * kSlice;
      const float* b0 = ws + ug * kWs;
#pragma unroll
      for (int k4 = 0; k4 < kSlice / 4; ++k4) {
        float4 a[RM];
#pragma unroll
        for (int i = 0; i < RM; ++i) a[i] = *reinterpret_cast<const float4*>(a0 + i * EG * kHs + 4 * k4);
#pragma unroll
        for (int j = 0; j < RN; ++j) {
          const float4 b = *reinterpret_cast<const float4*>(b0 + j * UG * kWs + 4 * k4);
#pragma unroll
          for (int i = 0; i < RM; ++i)
            acc[i][j] = __ffma2_rn(make_float2(b.x, b.y), make_float2(a[i].x, a[i].y), acc[i][j]);
#pragma unroll
          for (int i = 0; i < RM; ++i)
            acc[i][j] = __ffma2_rn(make_float2(b.z, b.w), make_float2(a[i].z, a[i].w), acc[i][j]);
        }
      }
    }
    __syncthreads();   // h1 consumed: h2 takes its place
#pragma unroll
    for (int i = 0; i < RM; ++i)
#pragma unroll
      for (int j = 0; j < RN; ++j)
        hs[(eg + i * EG) * kHs + ug + UG * j] = tanhf(acc[i][j].x + acc[i][j].y);
    __syncthreads();
    // head
    const float* W3 = wt + F::kW3;
    const float* b3 = W3 + out_dim * H;
    for (int it = tid; it < E * ((out_dim + 1) / 2); it += kThreads) {
      const int e = it % E, o = it / E * 2, o2 = o + 1 < out_dim ? o + 1 : o;
      const float4* wa = reinterpret_cast<const float4*>(W3 + o * H);
      const float4* wb = reinterpret_cast<const float4*>(W3 + o2 * H);
      const float4* hr = reinterpret_cast<const float4*>(hs + e * kHs);
      float s = __ldg(b3 + o), s2 = __ldg(b3 + o2);
#pragma unroll (H == 256 ? 16 : 8)
      for (int k4 = 0; k4 < H / 4; ++k4) {
        const float4 a = __ldg(wa + k4), b = __ldg(wb + k4), h = hr[k4];
        s = fmaf(a.x, h.x, s);
        s2 = fmaf(b.x, h.x, s2);
        s = fmaf(a.y, h.y, s);
        s2 = fmaf(b.y, h.y, s2);
        s = fmaf(a.z, h.z, s);
        s2 = fmaf(b.z, h.z, s2);
        s = fmaf(a.w, h.w, s);
        s2 = fmaf(b.w, h.w, s2);
      }
      sm[oY + e * 17 + y0 + o] = s;
      if (o2 != o) sm[oY + e * 17 + y0 + o2] = s2;
    }
    __syncthreads();
  }
};

// The two environment models as the rollout sees them.
struct SimFossen {
  using Env = auv::Env;
  static constexpr int kObs = auv::kObs, kAct = auv::kAct, kHistRows = 0;
  static __device__ __forceinline__ void load(const Model& M, const Buffers& B, int i, Env& e) {
    load_env(M, B.state, B.params, B.t_ep, B.episode, i, e);
  }
  static __device__ __forceinline__ void store(const Model& M, const Buffers& B, int i, const Env& e) {
    store_env(M, B.state, B.params, B.t_ep, B.episode, i, e);
  }
  static __device__ __forceinline__ void obs(const Env& e, float* o) { observe(e, o); }
  static __device__ __forceinline__ bool finite(const Env& e) { return env_finite(e); }
  static __device__ __forceinline__ float step(const Model& M, uint32_t id, Env& e, const float* a,
                                               float*, int, bool* d) {
    return physics_step(M, id, e, a, d);
  }
};

struct SimPaper {
  using Env = paper::Env;
  static constexpr int kObs = paper::kObs, kAct = paper::kAct, kHistRows = 6 * paper::kHist;
  static __device__ __forceinline__ void load(const Model& M, const Buffers& B, int i, Env& e) {
    paper::load_env(M, B.state, B.params, B.t_ep, B.episode, i, e);
  }
  static __device__ __forceinline__ void store(const Model& M, const Buffers& B, int i, const Env& e) {
    paper::store_env(M, B.state, B.params, B.t_ep, B.episode, i, e);
  }
  static __device__ __forceinline__ void obs(const Env& e, float* o) { paper::observe(e, o); }
  static __device__ __forceinline__ bool finite(const Env& e) { return paper::env_finite(e); }
  static __device__ __forceinline__ float step(const Model& M, uint32_t id, Env& e, const float* a,
                                               float* hist, int stride, bool* d) {
    return paper::physics_step(M, id, e, a, paper::HistS{hist, stride}, d);
  }
};

// An env's registers parked in shared memory (word k of lane l at k * E + l)
// while the networks use the register file.
template <int E, class T>
__device__ __forceinline__ void park(float* s, int lane, const T& e) {
  float w[sizeof(T) / 4];
  memcpy(w, &e, sizeof(T));
#pragma unroll
  for (int k = 0; k < (int)(sizeof(T) / 4); ++k) s[k * E + lane] = w[k];
}
template <int E, class T>
__device__ __forceinline__ void unpark(const float* s, int lane, T& e) {
  float w[sizeof(T) / 4];
#pragma unroll
  for (int k = 0; k < (int)(sizeof(T) / 4); ++k) w[k] = s[k * E + lane];
  memcpy(&e, w, sizeof(T));
}

template <class Sim, int H, int E, int SLOTS>
struct RolloutSmem {
  using TL = Tile<Sim::kObs, H, E, SLOTS>;
  static constexpr int oEps = TL::kNet, oEnv = oEps + 2 * E * 8,
                       oHist = oEnv + (int)(sizeof(typename Sim::Env) / 4) * E,
                       kFloats = oHist + Sim::kHistRows * E;
};

template <class Sim, int H, int E, int SLOTS>
__global__ void __launch_bounds__(kThreads, ctas_per_sm(E, H, SLOTS))
k_rollout_fp32(const Model M, Buffers B, Net policy, Net critic, Traj tr, int T, uint64_t t_g0,
               Status* st) {
  using TL = Tile<Sim::kObs, H, E, SLOTS>;
  using L = RolloutSmem<Sim, H, E, SLOTS>;
  constexpr int kO = Sim::kObs, kA = Sim::kAct;
  extern __shared__ __align__(16) float sm[];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int i = blockIdx.x * E + lane;
  const bool mine = lane < E, active = mine && i < M.n;
  const uint32_t id = M.id_base + (uint32_t)i;
  const size_t n = (size_t)M.n;
  const int nets = tr.value ? 2 : 1;
  typename TL::Ring ring;
  ring.start(sm, policy, critic, nets, T * nets * TL::kSlices, tid);
  bool bad = false;
  float* xs = sm + TL::oX;
  float* hist = sm + L::oHist;
  // observation of the env's current state into the tile and the trajectory
  auto show = [&](const typename Sim::Env& e, int t) {
    float o[kO];
    Sim::obs(e, o);
#pragma unroll
    for (int k = 0; k < kO; ++k) xs[lane * TL::kXs + k] = o[k];
    if (tr.obs) {
#pragma unroll
      for (int k = 0; k < kO; ++k) tr.obs[((size_t)t * kO + k) * n + i] = o[k];
    }
  };
  auto draw = [&](int t) {
    float eps[8];
    action_noise(id, M.seed, t_g0 + (uint64_t)t, eps);
#pragma unroll
    for (int k = 0; k < 8; ++k) sm[L::oEps + ((t & 1) * 8 + k) * E + lane] = eps[k];
  };
  if (warp == 0 && mine) {
    if (active) {
      typename Sim::Env e;
      Sim::load(M, B, i, e);
      for (int r = 0; r < Sim::kHistRows; ++r) hist[r * E + lane] = B.state[(13 + r) * n + i];
      show(e, 0);
      park<E>(sm + L::oEnv, lane, e);
    } else {
#pragma unroll
      for (int k = 0; k < kO; ++k) xs[lane * TL::kXs + k] = 0.0f;
    }
  }
  if (warp == 1 && active) draw(0);
  for (int t = 0; t < T; ++t) {
    TL::run(ring, 0, M.policy_out, 0, tid);
    if (nets == 2) TL::run(ring, 1, 1, 16, tid);
    if (warp == 1 && active && t + 1 < T) draw(t + 1);
    if (warp == 0 && active) {
      typename Sim::Env e;
      unpark<E>(sm + L::oEnv, lane, e);
      const float* y = sm + TL::oY + lane * 17;
      float a[kA], lp = 0.0f;
#pragma unroll
      for (int k = 0; k < kA; ++k) {
        const float eps = sm[L::oEps + ((t & 1) * 8 + k) * E + lane];
        float ls = M.logstd_fixed[k];
        if (M.policy_out == 2 * kA) ls = fminf(fmaxf(y[kA + k], M.logstd_min), M.logstd_max);
        a[k] = fmaf(expf(ls), eps, y[k]);
        lp += -0.5f * eps * eps - ls;
      }
      lp -= (float)kA * 0.91893853320467274f;
      const size_t o = (size_t)t * n + i;
      if (tr.value) tr.value[o] = y[16];
      if (tr.act) {
#pragma unroll
        for (int k = 0; k < kA; ++k) tr.act[((size_t)t * kA + k) * n + i] = a[k];
      }
      if (tr.logp) tr.logp[o] = lp;
      bool d;
      const float r = Sim::step(M, id, e, a, hist + lane, E, &d);
      if (tr.rew) tr.rew[o] = r;
      if (tr.done) tr.done[o] = d ? 1 : 0;
      bad |= !Sim::finite(e);
      if (t + 1 < T) {
        show(e, t + 1);
        park<E>(sm + L::oEnv, lane, e);
      } else {
        if (bad) flag_nan(st, i);
        Sim::store(M, B, i, e);
        for (int h = 0; h < Sim::kHistRows; ++h) B.state[(13 + h) * n + i] = hist[h * E + lane];
      }
    }
  }
  if (tid == 0) ring.finish(st);
}

// Networks over rows: row r's input k at obs[((r / ns) * IN + k) * ns + r % ns]
// (ns = 1: row-major; ns = n: a trajectory's observations).  head[r][out_dim]
// if given (policy), value[r] if given.  Each CTA takes every gridDim.x-th
// tile of E rows.
template <int IN, int H, int E, int SLOTS>
__global__ void __launch_bounds__(kThreads, ctas_per_sm(E, H, SLOTS))
k_rows_fp32(Net policy, Net critic, const float* __restrict__ obs, size_t rows, int ns, int out_dim,
            float* __restrict__ head, float* __restrict__ value, Status* st) {
  using TL = Tile<IN, H, E, SLOTS>;
  extern __shared__ __align__(16) float sm[];
  const int tid = threadIdx.x;
  const int nets = head && value ? 2 : 1;
  const size_t tiles = (rows + E - 1) / E;
  const int my = (int)((tiles - blockIdx.x - 1) / gridDim.x + 1);
  typename TL::Ring ring;
  ring.start(sm, head ? policy : critic, critic, nets, my * nets * TL::kSlices, tid);
  for (int m = 0; m < my; ++m) {
    const size_t r0 = (blockIdx.x + (size_t)m * gridDim.x) * E;
    for (int x = tid; x < E * IN; x += kThreads) {
      // row-major input: consecutive threads along a row; trajectory: along rows
      const int e = ns == 1 ? x / IN : x % E, k = ns == 1 ? x % IN : x / E;
      const size_t r = r0 + e;
      float v = 0.0f;
      if (r < rows) {
        const size_t t = r / (size_t)ns, j = r - t * (size_t)ns;
        v = __ldg(obs + (t * IN + k) * (size_t)ns + j);
      }
      sm[TL::oX + e * TL::kXs + k] = v;
    }
    if (head) TL::run(ring, 0, out_dim, 0, tid);
    if (value) TL::run(ring, nets - 1, 1, 16, tid);
    if (head)
      for (int x = tid; x < E * out_dim; x += kThreads) {
        const int e = x / out_dim, o = x - e * out_dim;
        if (r0 + e < rows) head[(r0 + e) * out_dim + o] = sm[TL::oY + e * 17 + o];
      }
    if (value && tid < E && r0 + tid < rows) value[r0 + tid] = sm[TL::oY + tid * 17 + 16];
  }
  if (tid == 0) ring.finish(st);
}

template <class Sim, int H, int E, int SLOTS>
cudaError_t rollout(const Model& M, const Buffers& B, const Net& p, const Net& v, const Traj& tr,
                    int T, uint64_t t_g0, Status* st, cudaStream_t s) {
  constexpr int smem = RolloutSmem<Sim, H, E, SLOTS>::kFloats * 4;
  static_assert(smem <= 226 * 1024 / ctas_per_sm(E, H, SLOTS), "shared memory per CTA");
  auto kern = k_rollout_fp32<Sim, H, E, SLOTS>;
  const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
  if (e != cudaSuccess) return e;
  kern<<<(M.n + E - 1) / E, kThreads, smem, s>>>(M, B, p, v, tr, T, t_g0, st);
  return cudaGetLastError();
}

// Rows per CTA: the fewest that keep one CTA per SM (a step's time grows with
// the tile, 10.4, 14.3 and 21.8 us a step at 8, 16 and 32 rows, width 256, and
// every CTA streams W2 once a step, so more CTAs than SMs gain nothing).
int rows_per_cta(size_t rows) {
  const size_t sms = (size_t)engine_sm_count();
  return rows <= 8 * sms ? 8 : (rows <= 16 * sms ? 16 : 32);
}

// Width 256, 32-row tiles: while every SM has at most one, the kernel compiled
// for one CTA per SM (no register cap at 128, six slots: 1.09 ms for 4,096
// envs x 50 steps against 1.24); above, two CTAs per SM, one's physics under
// the other's products (1.91 ms for 9,728 envs, where one CTA per SM in two
// waves would take 2.2).
bool one_per_sm(size_t rows) { return rows <= 32 * (size_t)engine_sm_count(); }

template <class Sim>
cudaError_t rollout_any(const Model& M, const Buffers& B, const Net& p, const Net& v, const Traj& tr,
                        int T, uint64_t t_g0, Status* st, cudaStream_t s) {
  const int e = rows_per_cta((size_t)M.n);
  if (M.hidden == 64)
    return e == 8 ? rollout<Sim, 64, 8, 8>(M, B, p, v, tr, T, t_g0, st, s)
                  : rollout<Sim, 64, 32, 8>(M, B, p, v, tr, T, t_g0, st, s);
  if (M.hidden == 256)
    return e == 8    ? rollout<Sim, 256, 8, 8>(M, B, p, v, tr, T, t_g0, st, s)
           : e == 16 ? rollout<Sim, 256, 16, 6>(M, B, p, v, tr, T, t_g0, st, s)
           : one_per_sm((size_t)M.n) ? rollout<Sim, 256, 32, 6>(M, B, p, v, tr, T, t_g0, st, s)
                                     : rollout<Sim, 256, 32, 3>(M, B, p, v, tr, T, t_g0, st, s);
  return cudaErrorInvalidValue;
}

template <int IN, int H, int E, int SLOTS>
cudaError_t rows_fp32(const Net& p, const Net& v, const float* obs, size_t rows, int ns, int out_dim,
                      float* head, float* value, Status* st, cudaStream_t s) {
  constexpr int smem = Tile<IN, H, E, SLOTS>::kNet * 4;
  static_assert(smem <= 226 * 1024 / ctas_per_sm(E, H, SLOTS), "shared memory per CTA");
  auto kern = k_rows_fp32<IN, H, E, SLOTS>;
  const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
  if (e != cudaSuccess) return e;
  const size_t tiles = (rows + E - 1) / E, most = (size_t)engine_sm_count() * ctas_per_sm(E, H, SLOTS);
  kern<<<(unsigned)std::min(tiles, most), kThreads, smem, s>>>(p, v, obs, rows, ns, out_dim, head, value,
                                                               st);
  return cudaGetLastError();
}

template <int IN>
cudaError_t rows_any(int H, const Net& p, const Net& v, const float* obs, size_t rows, int ns,
                     int out_dim, float* head, float* value, Status* st, cudaStream_t s) {
  const bool few = rows_per_cta(rows) == 8;
  if (H == 64)
    return few ? rows_fp32<IN, 64, 8, 8>(p, v, obs, rows, ns, out_dim, head, value, st, s)
               : rows_fp32<IN, 64, 32, 8>(p, v, obs, rows, ns, out_dim, head, value, st, s);
  if (H == 256)
    return few ? rows_fp32<IN, 256, 8, 8>(p, v, obs, rows, ns, out_dim, head, value, st, s)
               : rows_fp32<IN, 256, 32, 3>(p, v, obs, rows, ns, out_dim, head, value, st, s);
  return cudaErrorInvalidValue;
}

template <int IN, int H>
cudaError_t pack(const Fp32Nets& w, bool both, cudaStream_t s) {
  auto img = [](const void* p) { return const_cast<float*>(static_cast<const float*>(p)); };
  k_pack_fp32<IN, H><<<dim3((Image<IN, H>::kFloats + 255) / 256, both ? 2 : 1), 256, 0, s>>>(
      w.policy, img(w.policy_img), w.value, img(w.value_img));
  return cudaGetLastError();
}

}  // namespace

size_t fp32_image_bytes(int in_dim, int hidden) {
  return sizeof(float) * ((size_t)hidden / kSlice * hidden * kWs + (size_t)in_dim * hidden);
}

cudaError_t launch_pack_fp32(const Model& M, const Fp32Nets& w, bool both, cudaStream_t s) {
  if (M.model == 1)
    return M.hidden == 64 ? pack<paper::kObs, 64>(w, both, s) : pack<paper::kObs, 256>(w, both, s);
  return M.hidden == 64 ? pack<kObs, 64>(w, both, s) : pack<kObs, 256>(w, both, s);
}

cudaError_t launch_rollout_fp32(const Model& M, const Buffers& B, const Fp32Nets& w, const Traj& tr,
                                int T, uint64_t t_g0, Status* st, cudaStream_t s) {
  const Net p = {w.policy, static_cast<const float*>(w.policy_img)};
  const Net v = {w.value, static_cast<const float*>(w.value_img)};
  return M.model == 1 ? rollout_any<SimPaper>(M, B, p, v, tr, T, t_g0, st, s)
                      : rollout_any<SimFossen>(M, B, p, v, tr, T, t_g0, st, s);
}

cudaError_t launch_rows_fp32(const Model& M, const Fp32Nets& w, const float* obs, size_t rows, int ns,
                             float* head, float* value, Status* st, cudaStream_t s) {
  const Net p = {w.policy, static_cast<const float*>(w.policy_img)};
  const Net v = {w.value, static_cast<const float*>(w.value_img)};
  return M.model == 1
             ? rows_any<paper::kObs>(M.hidden, p, v, obs, rows, ns, M.policy_out, head, value, st, s)
             : rows_any<kObs>(M.hidden, p, v, obs, rows, ns, M.policy_out, head, value, st, s);
}

}  // namespace auv
