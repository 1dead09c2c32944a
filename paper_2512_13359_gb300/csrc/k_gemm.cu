// k_gemm.cu -- the learners' dense products (PPO update and SHAC window,
// paper §III-A) on the library's own kernels.
//
//   C[M][N] = beta * C + sum_k A(m, k) B(n, k)
//
// Tensor cores (bf16 or tf32 operands): one CTA computes a 128 x BN tile of
// C over a range of K.  A producer thread streams 128-byte-swizzled tiles of
// A (128 x BK) and B (BN x BK) into a four-stage shared-memory ring with TMA
// (cp.async.bulk.tensor), one thread issues tcgen05.mma into an fp32
// accumulator in tensor memory, and four warps read the accumulator back
// (tcgen05.ld) and write C, or an fp32 partial when K is split over CTAs.
// BK is 128 bytes of K per row: 64 bf16 or 32 tf32 elements.
//
// Operand tiles in shared memory are the canonical 128-byte-swizzle
// layouts of the tensor-core descriptors:
//  - K-major (row r of the tile, K contiguous): one TMA box of BK x rows;
//    row r at r * 128 bytes, 8-row groups 1024 bytes apart (SBO); an MMA's
//    K-step advances the start address by 32 bytes.
//  - MN-major (K row kk, the M or N index contiguous): boxes of 128 bytes of
//    M/N x BK rows, one per 128 bytes of M/N, BK * 128 bytes apart (LBO);
//    8 K rows form a 1024-byte group (SBO); an MMA's K-step (32 bytes of
//    K) advances the start address by 4096 / element-size bytes.  tf32 reads
//    MN-major operands only with the 128-byte swizzle of 32-byte pieces
//    (4 K rows, 512 bytes, a group): its tensor maps use that swizzle.
//
// fp32 operands without tensor cores (the exact mode): register-blocked CUDA-core
// kernels with the same operand layouts and the same split-K.
//
// Split-K: partial tiles go to ws[z][M_pad][N_pad] (fp32); k_reduce adds
// them in a fixed order (eight interleaved partial sums over z, then those
// eight in order) and applies beta and the output type.
#include <cuda.h>

#include <algorithm>
#include <mutex>

#include "auv_device.cuh"
#include "auv_gemm.h"
#include "auvenv.h"
#include "tc_ptx.cuh"

namespace auv {
namespace gemm {
namespace {

constexpr int kMaxStages = 4;
constexpr int kBM = 128;
constexpr uint64_t kWaitLimitNs = 2000000000ull;

// ---------------------------------------------------------------------------
// device helpers
// ---------------------------------------------------------------------------
__device__ __forceinline__ void tma_load_2d(void* dst, const CUtensorMap* map, int x, int y,
                                            uint64_t* bar) {
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes "
      "[%0], [%1, {%2, %3}], [%4];" ::"r"(tc::smem_u32(dst)),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(x), "r"(y), "r"(tc::smem_u32(bar))
      : "memory");
}

// Shared-memory descriptor with both byte offsets (128-byte swizzle of 16-byte
// pieces, type 2, or of 32-byte pieces, type 1).
__device__ __forceinline__ uint64_t desc_sw128(uint32_t saddr, uint32_t lbo, uint32_t sbo,
                                               uint64_t type = 2) {
  uint64_t d = 0;
  d |= (uint64_t)((saddr & 0x3FFFFu) >> 4);
  d |= (uint64_t)((lbo >> 4) & 0x3FFFu) << 16;
  d |= (uint64_t)((sbo >> 4) & 0x3FFFu) << 32;
  d |= (uint64_t)1u << 46;                       // descriptor version
  d |= type << 61;
  return d;
}

// Instruction descriptor: D fp32, A/B bf16 (kind::f16) or tf32 (kind::tf32),
// major-ness of A (bit 15) and B (bit 16): 1 = MN-major.
__host__ __device__ constexpr uint32_t idesc(bool tf32, bool a_mn, bool b_mn, int M, int N) {
  return (1u << 4) | ((tf32 ? 2u : 1u) << 7) | ((tf32 ? 2u : 1u) << 10) |
         ((a_mn ? 1u : 0u) << 15) | ((b_mn ? 1u : 0u) << 16) | ((uint32_t)(N >> 3) << 17) |
         ((uint32_t)(M >> 4) << 24);
}

template <bool TF32>
__device__ __forceinline__ void mma(uint32_t d, uint64_t a, uint64_t b, uint32_t id, uint32_t acc) {
  if constexpr (TF32) {
    asm volatile(
        "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::tf32 [%0], %1, %2, %3, p;\n\t}" ::"r"(d),
        "l"(a), "l"(b), "r"(id), "r"(acc)
        : "memory");
  } else {
    asm volatile(
        "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(d),
        "l"(a), "l"(b), "r"(id), "r"(acc)
        : "memory");
  }
}

// Wait with the limit whatever the abort flag says (copies or MMAs still in flight
// when a wait has given up: nothing may land after the CTA has left).
__device__ __forceinline__ void wait_landed(uint64_t* b, uint32_t phase) {
  const uint64_t t0 = tc::global_timer_ns();
  while (!tc::mbar_test(b, phase) && tc::global_timer_ns() - t0 < kWaitLimitNs) {
  }
}

struct TcArgs {
  int M, N, K;
  int chunks_per_split;   // K chunks of BK per CTA along z
  void* C;
  int ldc;
  int c_bf16;
  float beta;
  float* ws;              // split partials, or null (write C directly)
  int n_pad, m_pad;
  Status* st;
  int epi;                // EpiKind, on elements written to C with beta = 0
  const void* aux;
  int ld_aux, aux_vec;    // aux_vec: rows of aux start on 32-byte boundaries
  int vec;                // C base and ldc allow 16-byte (1) or 32-byte (2) row segments
  int ws_wide;            // ws 32-byte aligned: partial rows as whole 32-byte sectors
};

// 8 floats to a 32-byte aligned address with one 256-bit store (a whole L2
// sector; a thread writing its own row otherwise fills half a sector per
// access).
__device__ __forceinline__ void st_f32x8(float* p, const uint32_t* v) {
  asm volatile("st.global.v8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(p), "r"(v[0]),
               "r"(v[1]), "r"(v[2]), "r"(v[3]), "r"(v[4]), "r"(v[5]), "r"(v[6]), "r"(v[7])
               : "memory");
}

// (not .nc: a kernel that starts ahead of its predecessor's end may be resident
// while that one writes the array)
__device__ __forceinline__ void ld_f32x8(const float* p, float* v) {
  asm("ld.global.v8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
      : "=f"(v[0]), "=f"(v[1]), "=f"(v[2]), "=f"(v[3]), "=f"(v[4]), "=f"(v[5]), "=f"(v[6]), "=f"(v[7])
      : "l"(p));
}

// One element's epilogue; h: tanh' activation.
__device__ __forceinline__ float epilogue(int epi, float x, float h) {
  return epi == kEpiTanh ? tanhf(x) : (epi == kEpiDtanh ? x * (1.0f - h * h) : x);
}
// aux element (row, col) of C's type.
__device__ __forceinline__ float aux_at(const void* aux, int ld, int c_bf16, size_t row, int col) {
  return c_bf16 ? __uint_as_float((uint32_t)static_cast<const uint16_t*>(aux)[row * ld + col] << 16)
                : static_cast<const float*>(aux)[row * ld + col];
}

// acc += beta C on 32 columns of one row from nb, every read ahead of the first
// sum (and of the stores, which the compiler may not move them across).
__device__ __forceinline__ void add_c32(const TcArgs& a, uint32_t (&acc)[32], size_t row, int nb) {
  float old[32];
  if (a.c_bf16) {
    const uint16_t* c = static_cast<const uint16_t*>(a.C) + row * a.ldc + nb;
#pragma unroll
    for (int q = 0; q < 32; ++q) old[q] = nb + q < a.N ? __uint_as_float((uint32_t)c[q] << 16) : 0.0f;
  } else {
    const float* c = static_cast<const float*>(a.C) + row * a.ldc + nb;
#pragma unroll
    for (int q = 0; q < 32; ++q) old[q] = nb + q < a.N ? c[q] : 0.0f;
  }
#pragma unroll
  for (int q = 0; q < 32; ++q) acc[q] = __float_as_uint(fmaf(a.beta, old[q], __uint_as_float(acc[q])));
}

// 32 columns of C from column nb of one row: beta C + acc, columns below N.
__device__ __forceinline__ void store32(const TcArgs& a, uint32_t (&acc)[32], size_t row, int nb) {
  if (a.beta != 0.0f) add_c32(a, acc, row, nb);
  if (nb + 32 <= a.N && a.vec) {
    // whole 32-column segment, 16-byte aligned rows: vector stores (32-byte
    // aligned rows: whole sectors)
    if (a.c_bf16) {
      uint16_t* crow = static_cast<uint16_t*>(a.C) + row * a.ldc + nb;
      uint32_t w[16];
#pragma unroll
      for (int e = 0; e < 16; ++e)
        w[e] = tc::pack_bf16x2(__uint_as_float(acc[2 * e]), __uint_as_float(acc[2 * e + 1]));
      if (a.vec == 2) {
        st_f32x8(reinterpret_cast<float*>(crow), w);
        st_f32x8(reinterpret_cast<float*>(crow + 16), w + 8);
      } else {
        uint4* dst = reinterpret_cast<uint4*>(crow);
#pragma unroll
        for (int q = 0; q < 4; ++q) dst[q] = make_uint4(w[4 * q], w[4 * q + 1], w[4 * q + 2], w[4 * q + 3]);
      }
    } else if (a.vec == 2) {
      float* crow = static_cast<float*>(a.C) + row * a.ldc + nb;
#pragma unroll
      for (int q = 0; q < 4; ++q) st_f32x8(crow + 8 * q, acc + 8 * q);
    } else {
      uint4* dst = reinterpret_cast<uint4*>(static_cast<float*>(a.C) + row * a.ldc + nb);
#pragma unroll
      for (int q = 0; q < 8; ++q)
        dst[q] = make_uint4(acc[4 * q], acc[4 * q + 1], acc[4 * q + 2], acc[4 * q + 3]);
    }
  } else if (a.c_bf16) {
    uint16_t* crow = static_cast<uint16_t*>(a.C) + row * a.ldc;
#pragma unroll
    for (int q = 0; q < 32; ++q)
      if (nb + q < a.N) crow[nb + q] = (uint16_t)(tc::pack_bf16x2(__uint_as_float(acc[q]), 0.0f) & 0xFFFFu);
  } else {
    float* crow = static_cast<float*>(a.C) + row * a.ldc;
#pragma unroll
    for (int g = 0; g < 4; ++g) {
      const int n = nb + 8 * g;
      if (a.vec == 2 && n + 8 <= a.N) {   // narrow heads: whole sectors
        st_f32x8(crow + n, acc + 8 * g);
        continue;
      }
#pragma unroll
      for (int q = 0; q < 8; ++q)
        if (n + q < a.N) crow[n + q] = __uint_as_float(acc[8 * g + q]);
    }
  }
}

// A warp's 32 rows x 32 columns of C from (row0, nb), lane l holding row l: what
// the vector stores above do not cover (beta, or rows off 16 bytes), turned
// through 4 KB of shared memory so that a row's columns are read and written by
// the warp together (30,011 x 256 x 264 with beta = 1, tf32: into bf16 459 us by
// rows, 48 here; fp32 166 and 28).
__device__ __forceinline__ void store_turned(const TcArgs& a, const uint32_t (&acc)[32], int row0, int nb,
                                             uint8_t* box, int lane) {
#pragma unroll
  for (int q = 0; q < 8; ++q)
    *reinterpret_cast<uint4*>(box + lane * 128 + ((q ^ (lane & 7)) << 4)) =
        make_uint4(acc[4 * q], acc[4 * q + 1], acc[4 * q + 2], acc[4 * q + 3]);
  __syncwarp();
  if (nb + lane < a.N) {
    const size_t at = (size_t)row0 * a.ldc + nb + lane;
#pragma unroll 1
    for (int r0 = 0; r0 < 32 && row0 + r0 < a.M; r0 += 8) {
      const int rows = min(8, a.M - row0 - r0);
      float x[8];
#pragma unroll
      for (int r = 0; r < 8; ++r)
        x[r] = *reinterpret_cast<const float*>(box + (r0 + r) * 128 + ((lane >> 2 ^ ((r0 + r) & 7)) << 4) +
                                               (lane & 3) * 4);
      if (a.c_bf16) {
        uint16_t* c = static_cast<uint16_t*>(a.C) + at + (size_t)r0 * a.ldc;
        if (a.beta != 0.0f) {
          uint32_t old[8];
#pragma unroll
          for (int r = 0; r < 8; ++r) old[r] = r < rows ? c[(size_t)r * a.ldc] : 0u;
#pragma unroll
          for (int r = 0; r < 8; ++r) x[r] = fmaf(a.beta, __uint_as_float(old[r] << 16), x[r]);
        }
#pragma unroll
        for (int r = 0; r < 8; ++r)
          if (r < rows) c[(size_t)r * a.ldc] = (uint16_t)(tc::pack_bf16x2(x[r], 0.0f) & 0xFFFFu);
      } else {
        float* c = static_cast<float*>(a.C) + at + (size_t)r0 * a.ldc;
        if (a.beta != 0.0f) {
          float old[8];
#pragma unroll
          for (int r = 0; r < 8; ++r) old[r] = r < rows ? c[(size_t)r * a.ldc] : 0.0f;
#pragma unroll
          for (int r = 0; r < 8; ++r) x[r] = fmaf(a.beta, old[r], x[r]);
        }
#pragma unroll
        for (int r = 0; r < 8; ++r)
          if (r < rows) c[(size_t)r * a.ldc] = x[r];
      }
    }
  }
  __syncwarp();   // the box is free again
}

// The tanh' activations of one row's 32 columns from nb (0 beyond N), all in
// flight at once.  row includes pdl_enter()'s zero, so that no load comes ahead
// of its wait.
__device__ __forceinline__ void load_aux32(const TcArgs& a, size_t row, int nb, float (&h)[32]) {
  if (a.aux_vec && nb + 32 <= a.N) {
    if (a.c_bf16) {
      const uint16_t* p = static_cast<const uint16_t*>(a.aux) + row * a.ld_aux + nb;
      float w[16];
#pragma unroll
      for (int g = 0; g < 2; ++g) ld_f32x8(reinterpret_cast<const float*>(p + 16 * g), w + 8 * g);
#pragma unroll
      for (int j = 0; j < 32; ++j) {
        const uint32_t u = __float_as_uint(w[j >> 1]);
        h[j] = __uint_as_float(j & 1 ? u & 0xFFFF0000u : u << 16);
      }
    } else {
      const float* p = static_cast<const float*>(a.aux) + row * a.ld_aux + nb;
#pragma unroll
      for (int g = 0; g < 4; ++g) ld_f32x8(p + 8 * g, h + 8 * g);
    }
    return;
  }
#pragma unroll
  for (int j = 0; j < 32; ++j)
    h[j] = nb + j < a.N ? aux_at(a.aux, a.ld_aux, a.c_bf16, row, nb + j) : 0.0f;
}

// 32 accumulator columns of one row.  A bf16 result is rounded before its
// tanh or tanh' too, as when they were passes over the stored product.
__device__ __forceinline__ void epilogue32(const TcArgs& a, uint32_t (&acc)[32], const float (&h)[32]) {
  if (a.c_bf16) {
#pragma unroll
    for (int q = 0; q < 32; ++q)
      acc[q] = tc::pack_bf16x2(__uint_as_float(acc[q]), 0.0f) << 16;
  }
  if (a.epi == kEpiTanh) {
#pragma unroll
    for (int q = 0; q < 32; ++q) acc[q] = __float_as_uint(tanhf(__uint_as_float(acc[q])));
  } else {
#pragma unroll
    for (int q = 0; q < 32; ++q)
      acc[q] = __float_as_uint(__uint_as_float(acc[q]) * (1.0f - h[q] * h[q]));
  }
}

// BN = 320 (for N in (256, 320]: the weight gradients' 264 augmented
// columns) is one N = 256 and one N = 64 MMA per K-step, in a three-stage
// ring; the other widths are one MMA in a four-stage ring.
template <bool TF32, bool A_MN, bool B_MN, int BN>
struct Tile {
  static constexpr int kEs = TF32 ? 4 : 2;
  static constexpr int kBK = 128 / kEs;                 // K elements per stage
  static constexpr int kStages = BN > 256 ? 3 : 4;
  static constexpr uint32_t kABytes = kBM * 128;        // 128 rows (or BK K-rows x 128 B x 128/E)
  static constexpr uint32_t kBBytes = BN * 128;
  static constexpr uint32_t kStage = kABytes + kBBytes;
  static constexpr uint32_t kSmem = kStages * kStage + 256 + 1024;
  static constexpr int kElemsPer128 = 128 / kEs;        // M/N elements per MN-major box
  static constexpr int kBoxRows = BN > 256 ? 64 : BN;   // K-major B: rows per TMA box
  static constexpr uint32_t kTmemCols = BN > 256 ? 512 : BN;
};

struct Bars {
  uint64_t full[kMaxStages];
  uint64_t empty[kMaxStages];
  uint64_t acc_full;
  uint32_t tmem_base;
  int abort;
};

// One CTA: warps 0-3 epilogue (tensor-memory lanes 0..127 = rows), warp 4
// TMA producer, warp 5 MMA issuer and tensor-memory owner.
template <bool TF32, bool A_MN, bool B_MN, int BN>
__global__ void __launch_bounds__(192, 1)
k_gemm_tc(const __grid_constant__ CUtensorMap map_a, const __grid_constant__ CUtensorMap map_b,
          TcArgs args) {
  using TL = Tile<TF32, A_MN, B_MN, BN>;
  constexpr int kProducer = 4, kIssuer = 5;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>(
      (reinterpret_cast<uintptr_t>(smem_raw) + 1023u) & ~(uintptr_t)1023u);
  constexpr int kStages = TL::kStages;
  Bars* bar = reinterpret_cast<Bars*>(smem + kStages * TL::kStage);
  volatile int* abort = &bar->abort;
  const int tid = threadIdx.x, warp = tid >> 5;
  const int m0 = blockIdx.x * kBM, n0 = blockIdx.y * BN;
  const int n_chunks_total = (args.K + TL::kBK - 1) / TL::kBK;
  const int c0 = blockIdx.z * args.chunks_per_split;
  const int c1 = min(n_chunks_total, c0 + args.chunks_per_split);
  const int n_chunks = max(0, c1 - c0);

  if (tid == 0) {
    for (int s = 0; s < kStages; ++s) {
      tc::mbar_init(&bar->full[s], 1);
      tc::mbar_init(&bar->empty[s], 1);
    }
    tc::mbar_init(&bar->acc_full, 1);
    bar->abort = 0;
    tc::mbar_fence_init();
  }
  if (warp == kIssuer) {
    tc::tmem_alloc(&bar->tmem_base, TL::kTmemCols);
    tc::tmem_relinquish();
  }
  tc::tc_fence_before();
  __syncthreads();
  tc::tc_fence_after();
  const int zero = pdl_enter();   // after the allocation: the next kernel's may not come first
  const uint32_t tmem = bar->tmem_base;
  const uint32_t s_base = tc::smem_u32(smem);

  if (warp == kProducer) {
    // ---- producer: TMA tiles of A and B into the ring ----
    if ((tid & 31) == 0) {
      // MN-major blocks of 128 bytes that hold rows or columns of the product
      // (the others' accumulator rows and columns are never read back).  The loops
      // are unrolled over all blocks of a tile: with run-time bounds the one
      // thread's issue of up to ten copies a chunk held the MMAs up (bf16 2,048^3,
      // both MN-major: 31.6 us, 27.6 unrolled; tf32 79 and 68)
      const int na = min(kBM / TL::kElemsPer128, (args.M - m0 + TL::kElemsPer128 - 1) / TL::kElemsPer128);
      const int nb = min(BN / TL::kElemsPer128, (args.N - n0 + TL::kElemsPer128 - 1) / TL::kElemsPer128);
      const uint32_t bytes = (A_MN ? na * (TL::kBK * 128) : TL::kABytes) +
                             (B_MN ? nb * (TL::kBK * 128) : TL::kBBytes);
      int c = 0;
      for (; c < n_chunks; ++c) {
        const int s = c % kStages;
        if (c >= kStages &&
            !tc::mbar_wait(&bar->empty[s], (uint32_t)((c / kStages) - 1) & 1u, abort, kWaitLimitNs))
          break;
        uint8_t* a_dst = smem + s * TL::kStage;
        uint8_t* b_dst = a_dst + TL::kABytes;
        tc::mbar_arrive_expect_tx(&bar->full[s], bytes);
        const int k = (c0 + c) * TL::kBK;
        if (A_MN) {
#pragma unroll
          for (int j = 0; j < kBM / TL::kElemsPer128; ++j)
            if (j < na)
              tma_load_2d(a_dst + j * (TL::kBK * 128), &map_a, m0 + j * TL::kElemsPer128, k, &bar->full[s]);
        } else {
          tma_load_2d(a_dst, &map_a, k, m0, &bar->full[s]);
        }
        if (B_MN) {
#pragma unroll
          for (int j = 0; j < BN / TL::kElemsPer128; ++j)
            if (j < nb)
              tma_load_2d(b_dst + j * (TL::kBK * 128), &map_b, n0 + j * TL::kElemsPer128, k, &bar->full[s]);
        } else {
#pragma unroll
          for (int j = 0; j < BN / TL::kBoxRows; ++j)
            tma_load_2d(b_dst + j * (TL::kBoxRows * 128), &map_b, k, n0 + j * TL::kBoxRows,
                        &bar->full[s]);
        }
      }
      if (*abort)   // the copies still in flight
        for (int s = 0; s < kStages; ++s) {
          const int fills = c / kStages + (s < c % kStages ? 1 : 0);
          if (fills > 0) wait_landed(&bar->full[s], (uint32_t)(fills - 1) & 1u);
        }
    }
    __syncwarp();
  } else if (warp == kIssuer) {
    // ---- MMA issue ----
    if ((tid & 31) == 0) {
      constexpr uint32_t kId = idesc(TF32, A_MN, B_MN, kBM, BN > 256 ? 256 : BN);
      constexpr uint32_t kId2 = idesc(TF32, A_MN, B_MN, kBM, BN > 256 ? BN - 256 : 16);
      // second MMA of a 320-wide tile: B from column 256 (MN-major: the fifth
      // 128-byte block of bf16; K-major: row 256)
      constexpr uint32_t kB2 = B_MN ? (256 / TL::kElemsPer128) * (TL::kBK * 128) : 256 * 128;
      constexpr uint32_t kLbo = TL::kBK * 128;          // MN-major: between 128-byte M/N blocks
      constexpr uint32_t kKStepMn = 4096 / TL::kEs;     // MN-major: bytes per 32 bytes of K
      constexpr uint32_t kSboMn = TF32 ? 512 : 1024;    // and between its K-row groups
      constexpr uint64_t kTypeMn = TF32 ? 1 : 2;
      bool ok = true;
      for (int c = 0; c < n_chunks && ok; ++c) {
        const int s = c % kStages;
        ok = tc::mbar_wait(&bar->full[s], (uint32_t)(c / kStages) & 1u, abort, kWaitLimitNs);
        if (!ok) break;
        tc::tc_fence_after();
        const uint32_t a0 = s_base + s * TL::kStage, b0 = a0 + TL::kABytes;
#pragma unroll
        for (int kk = 0; kk < 4; ++kk) {
          const uint64_t da = A_MN ? desc_sw128(a0 + kk * kKStepMn, kLbo, kSboMn, kTypeMn)
                                   : desc_sw128(a0 + kk * 32, 16, 1024);
          const uint64_t db = B_MN ? desc_sw128(b0 + kk * kKStepMn, kLbo, kSboMn, kTypeMn)
                                   : desc_sw128(b0 + kk * 32, 16, 1024);
          mma<TF32>(tmem, da, db, kId, (c > 0 || kk > 0) ? 1u : 0u);
          if constexpr (BN > 256) {
            const uint64_t db2 = B_MN ? desc_sw128(b0 + kB2 + kk * kKStepMn, kLbo, kSboMn, kTypeMn)
                                      : desc_sw128(b0 + kB2 + kk * 32, 16, 1024);
            mma<TF32>(tmem + 256, da, db2, kId2, (c > 0 || kk > 0) ? 1u : 0u);
          }
        }
        tc::mma_commit(&bar->empty[s]);
      }
      tc::mma_commit(&bar->acc_full);
      wait_landed(&bar->acc_full, 0);   // tensor memory is freed below
    }
    __syncwarp();
  } else {
    // ---- epilogue: one row per thread, BN columns in chunks of 32 ----
    const int row = m0 + tid + zero;
    const bool epi = args.epi != kEpiNone && !args.ws && row < args.M;
    const bool dtanh = epi && args.epi == kEpiDtanh;
    // tanh': a chunk's activations are loaded while the accumulator is still
    // being computed, the next chunk's while this one is stored
    float h[32];
    if (dtanh) load_aux32(args, (size_t)row, n0, h);
    const bool ok = n_chunks > 0 && tc::mbar_wait(&bar->acc_full, 0, abort, kWaitLimitNs);
    tc::tc_fence_after();
    const uint32_t lane_addr = tmem + ((uint32_t)(warp * 32) << 16);
#pragma unroll 1
    for (int j = 0; j < BN / 32; ++j) {
      uint32_t acc[32];
      tc::tmem_ld32(lane_addr + j * 32, acc);
      tc::tmem_ld_wait(acc);
      if (!ok) {
#pragma unroll
        for (int q = 0; q < 32; ++q) acc[q] = 0u;   // no K in range (or a timed-out wait)
      }
      const int nb = n0 + j * 32;
      if (epi) epilogue32(args, acc, h);
      if (dtanh && j + 1 < BN / 32) load_aux32(args, (size_t)row, nb + 32, h);
      if (args.ws) {
        // partials of the rows and 32-column groups the reduction reads
        if (row < args.M && nb < args.N) {
          float* dst = args.ws + ((size_t)blockIdx.z * args.m_pad + row) * args.n_pad + nb;
          if (args.ws_wide) {
#pragma unroll
            for (int q = 0; q < 4; ++q) st_f32x8(dst + 8 * q, acc + 8 * q);
          } else {
            float4* d4 = reinterpret_cast<float4*>(dst);
#pragma unroll
            for (int q = 0; q < 8; ++q)
              d4[q] = make_float4(__uint_as_float(acc[4 * q]), __uint_as_float(acc[4 * q + 1]),
                                  __uint_as_float(acc[4 * q + 2]), __uint_as_float(acc[4 * q + 3]));
          }
        }
      } else if (row < args.M) {
        store32(args, acc, (size_t)row, nb);
      }
    }
  }
  tc::tc_fence_before();
  __syncthreads();
  if (tid == 0 && bar->abort) {
    atomicAdd(&args.st->timeouts, 1);
    atomicCAS(&args.st->code, 0, -4);
  }
  if (warp == kIssuer) {
    tc::tc_fence_after();
    tc::tmem_dealloc(tmem, TL::kTmemCols);
  }
}

// ---------------------------------------------------------------------------
// Products over many rows with a short contraction (a layer's forward product
// or input gradient over a batch: A K-major, at most 9 K-chunks).  They move
// their rows once and reuse one small B, so a CTA keeps its BN columns of B
// resident (147 KB at K = 264 tf32, BN = 128) and walks over row tiles: A
// streams through a ring, two accumulators in tensor memory let a tile's MMAs
// run under the previous tile's epilogue, and 256-column layers are two
// column halves on neighbouring CTAs, which read the same rows at the same
// time (from L2 the second time).  fp32 results with BN = 128 leave as TMA
// boxes of 32 rows x 32 columns (rows of 128 bytes, 16-byte pieces swizzled so
// that a thread per row meets no bank conflicts), and the tanh' operand comes
// in the same way into the same buffer, one per epilogue warp: stores and
// loads of each thread's own row, 32 bytes at a time, took 49 us for a
// 65,536 x 256 input gradient with tanh' (32 us here).
//
// Where the general kernel would have split K in two over CTAs (fewer than
// half as many of its tiles as SMs), chunks from `half` on go to a second
// accumulator and the two are added once: the same sums, bit for bit, without
// the partials' round trip (a closed loop amplifies a changed rounding).
//
// Warps 0-7 (BN = 128) or 0-3: epilogue, warp w on rows 32 (w mod 4) .. + 31
// and column groups w / 4, w / 4 + 2; then the producer and the MMA issuer.
// ---------------------------------------------------------------------------
template <bool TF32, bool B_MN, int BN>
struct RowTile {
  static constexpr int kEs = TF32 ? 4 : 2;
  static constexpr int kBK = 128 / kEs;
  static constexpr int kElemsPer128 = 128 / kEs;
  static constexpr int kMaxChunks = 9, kMaxStages = 8;
  static constexpr uint32_t kStage = kBM * 128;           // A: 128 rows x 128 bytes
  static constexpr uint32_t kBChunk = BN * 128;
  static constexpr bool kBoxes = BN == 128;               // TMA epilogue
  static constexpr int kEpiWarps = kBoxes ? 8 : 4;
  static constexpr int kThreads = 32 * kEpiWarps + 64;
  static constexpr int kCtas = kBoxes ? 1 : 2;            // per SM
  static constexpr uint32_t kBoxBytes = kBoxes ? kEpiWarps * 4096 : 0;
  static constexpr uint32_t kFixed = kBoxBytes + 512 + 1024;   // boxes, barriers, alignment
  static constexpr uint32_t kBudget = (kCtas == 1 ? 227 : 113) * 1024;
  // A stages beside `chunks` resident chunks of B
  static int stages(int chunks) {
    const int n = (int)((kBudget - kFixed - chunks * kBChunk) / kStage);
    return n < kMaxStages ? n : kMaxStages;
  }
  static_assert(kBudget >= kFixed + kMaxChunks * kBChunk + 2 * kStage, "at least two stages");
};

struct RowBars {
  uint64_t full[8], empty[8];      // A stages
  uint64_t b_full;
  uint64_t acc_full[2], acc_empty[2];
  uint64_t aux[8];                 // per epilogue warp: its tanh' box
  uint32_t tmem_base;
  int abort;
};

__device__ __forceinline__ void tma_store_2d(const CUtensorMap* map, const void* src, int x, int y) {
  asm volatile("cp.async.bulk.tensor.2d.global.shared::cta.bulk_group [%0, {%2, %3}], [%1];" ::"l"(
                   reinterpret_cast<uint64_t>(map)),
               "r"(tc::smem_u32(src)), "r"(x), "r"(y)
               : "memory");
}

template <bool TF32, bool B_MN, int BN>
__global__ void __launch_bounds__((RowTile<TF32, B_MN, BN>::kThreads), (RowTile<TF32, B_MN, BN>::kCtas))
k_gemm_rows(const __grid_constant__ CUtensorMap map_a, const __grid_constant__ CUtensorMap map_b,
            const __grid_constant__ CUtensorMap map_c, const __grid_constant__ CUtensorMap map_aux,
            TcArgs args, int tiles_m, int tiles_n, int stages, int half, int boxes) {
  using TL = RowTile<TF32, B_MN, BN>;
  constexpr int kProducer = TL::kEpiWarps, kIssuer = kProducer + 1;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>(
      (reinterpret_cast<uintptr_t>(smem_raw) + 1023u) & ~(uintptr_t)1023u);
  const int n_chunks = (args.K + TL::kBK - 1) / TL::kBK;
  uint8_t* ring = smem + n_chunks * TL::kBChunk;
  uint8_t* box_mem = ring + stages * TL::kStage;
  RowBars* bar = reinterpret_cast<RowBars*>(box_mem + TL::kBoxBytes);
  volatile int* abort = &bar->abort;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  // this CTA's columns, and its row tiles m_first, m_first + m_step, ...
  const int n0 = (int)(blockIdx.x % tiles_n) * BN;
  const int m_first = blockIdx.x / tiles_n, m_step = gridDim.x / tiles_n;

  if (tid == 0) {
    for (int s = 0; s < stages; ++s) {
      tc::mbar_init(&bar->full[s], 1);
      tc::mbar_init(&bar->empty[s], 1);
    }
    tc::mbar_init(&bar->b_full, 1);
    for (int k = 0; k < 2; ++k) {
      tc::mbar_init(&bar->acc_full[k], 1);
      tc::mbar_init(&bar->acc_empty[k], TL::kEpiWarps);
    }
    for (int w = 0; w < TL::kEpiWarps; ++w) tc::mbar_init(&bar->aux[w], 1);
    bar->abort = 0;
    tc::mbar_fence_init();
  }
  if (warp == kIssuer) {
    tc::tmem_alloc(&bar->tmem_base, 4 * BN);   // two tiles x (sum, second half's sum)
    tc::tmem_relinquish();
  }
  tc::tc_fence_before();
  __syncthreads();
  tc::tc_fence_after();
  const int zero = pdl_enter();   // after the allocation: the next kernel's may not come first
  const uint32_t tmem = bar->tmem_base;

  if (warp == kProducer) {
    if (lane == 0) {
      tc::mbar_arrive_expect_tx(&bar->b_full, n_chunks * TL::kBChunk);
      for (int c = 0; c < n_chunks; ++c) {
        uint8_t* dst = smem + c * TL::kBChunk;
        const int k = c * TL::kBK;
        if (B_MN) {
#pragma unroll
          for (int j = 0; j < BN / TL::kElemsPer128; ++j)
            tma_load_2d(dst + j * (TL::kBK * 128), &map_b, n0 + j * TL::kElemsPer128, k, &bar->b_full);
        } else {
          tma_load_2d(dst, &map_b, k, n0, &bar->b_full);
        }
      }
      int s = 0, fill = 0;   // next stage, and how often the ring has gone round
      bool ok = true;
      for (int m = m_first; m < tiles_m && ok; m += m_step) {
        for (int c = 0; c < n_chunks; ++c) {
          ok = fill == 0 || tc::mbar_wait(&bar->empty[s], (uint32_t)(fill - 1) & 1u, abort, kWaitLimitNs);
          if (!ok) break;
          tc::mbar_arrive_expect_tx(&bar->full[s], TL::kStage);
          tma_load_2d(ring + s * TL::kStage, &map_a, c * TL::kBK, m * kBM, &bar->full[s]);
          if (++s == stages) {
            s = 0;
            ++fill;
          }
        }
      }
      if (*abort) {
        wait_landed(&bar->b_full, 0);
        for (int q = 0; q < stages; ++q) {
          const int fills = fill + (q < s ? 1 : 0);
          if (fills > 0) wait_landed(&bar->full[q], (uint32_t)(fills - 1) & 1u);
        }
      }
    }
    __syncwarp();
  } else if (warp == kIssuer) {
    if (lane == 0) {
      constexpr uint32_t kId = idesc(TF32, false, B_MN, kBM, BN);
      constexpr uint32_t kLbo = TL::kBK * 128;
      constexpr uint32_t kKStepMn = 4096 / TL::kEs;
      constexpr uint32_t kSboMn = TF32 ? 512 : 1024;
      constexpr uint64_t kTypeMn = TF32 ? 1 : 2;
      const uint32_t b_base = tc::smem_u32(smem), r_base = tc::smem_u32(ring);
      bool ok = tc::mbar_wait(&bar->b_full, 0, abort, kWaitLimitNs);
      int s = 0, item = 0;
      uint32_t phase = 0;
      for (int m = m_first; m < tiles_m && ok; m += m_step, ++item) {
        const uint32_t d0 = tmem + (item & 1) * 2 * BN;
        ok = item < 2 || tc::mbar_wait(&bar->acc_empty[item & 1], (uint32_t)(item / 2 - 1) & 1u, abort,
                                       kWaitLimitNs);
        for (int c = 0; c < n_chunks && ok; ++c) {
          ok = tc::mbar_wait(&bar->full[s], phase, abort, kWaitLimitNs);
          if (!ok) break;
          tc::tc_fence_after();
          const uint32_t a0 = r_base + s * TL::kStage, b0 = b_base + c * TL::kBChunk;
          const uint32_t d = d0 + (half && c >= half ? BN : 0);
          const bool first = c == 0 || c == half;
#pragma unroll
          for (int kk = 0; kk < 4; ++kk) {
            const uint64_t da = desc_sw128(a0 + kk * 32, 16, 1024);
            const uint64_t db = B_MN ? desc_sw128(b0 + kk * kKStepMn, kLbo, kSboMn, kTypeMn)
                                     : desc_sw128(b0 + kk * 32, 16, 1024);
            mma<TF32>(d, da, db, kId, first && kk == 0 ? 0u : 1u);
          }
          tc::mma_commit(&bar->empty[s]);
          if (++s == stages) {
            s = 0;
            phase ^= 1u;
          }
        }
        if (ok) tc::mma_commit(&bar->acc_full[item & 1]);
      }
      // every MMA has completed before tensor memory is freed (b_full's second phase)
      tc::mma_commit(&bar->b_full);
      wait_landed(&bar->b_full, 1);
    }
    __syncwarp();
  } else {
    const bool box = TL::kBoxes && boxes, box_aux = box && args.epi == kEpiDtanh;
    uint8_t* mine = box_mem + warp * 4096;   // this warp's box: 32 rows of 128 bytes
    const int rw = (warp & 3) * 32;          // its rows of the tile
    const uint32_t lane_addr = tmem + ((uint32_t)rw << 16);
    constexpr int kGroups = BN / 32, kStep = TL::kEpiWarps / 4;
    uint32_t aux_phase = 0;
    bool aux_sent = false, ok = true;
    // lane 0: the tanh' box of row tile m, column group j
    auto fetch_aux = [&](int m, int j) {
      if (lane != 0 || n0 + 32 * j >= args.N) return;
      tc::mbar_arrive_expect_tx(&bar->aux[warp], 4096);
      tma_load_2d(mine, &map_aux, n0 + 32 * j, m * kBM + rw, &bar->aux[warp]);
      aux_sent = true;
    };
    if (box_aux && m_first < tiles_m) fetch_aux(m_first, warp >> 2);
    int item = 0;
    for (int m = m_first; m < tiles_m; m += m_step, ++item) {
      const int row = m * kBM + rw + lane + zero;
      const bool live = row < args.M;
      const bool direct_aux = args.epi == kEpiDtanh && !box_aux && live;
      float h[32];
      if (direct_aux) load_aux32(args, (size_t)row, n0 + (warp >> 2) * 32, h);
      // (a wait that gave up is the whole warp's: what follows is warp-wide)
      ok = __all_sync(0xFFFFFFFFu, tc::mbar_wait(&bar->acc_full[item & 1], (uint32_t)(item / 2) & 1u, abort,
                                                 kWaitLimitNs));
      if (!ok) break;
      tc::tc_fence_after();
#pragma unroll 1
      for (int j = warp >> 2; j < kGroups; j += kStep) {
        const int nb = n0 + j * 32;
        if (nb >= args.N) break;
        uint32_t acc[32];
        tc::tmem_ld32(lane_addr + (item & 1) * 2 * BN + j * 32, acc);
        tc::tmem_ld_wait(acc);
        if (half) {
          uint32_t b[32];
          tc::tmem_ld32(lane_addr + (item & 1) * 2 * BN + BN + j * 32, b);
          tc::tmem_ld_wait(b);
#pragma unroll
          for (int q = 0; q < 32; ++q)
            acc[q] = __float_as_uint(__uint_as_float(acc[q]) + __uint_as_float(b[q]));
        }
        if (box_aux) {
          ok = __all_sync(0xFFFFFFFFu, tc::mbar_wait(&bar->aux[warp], aux_phase, abort, kWaitLimitNs));
          if (!ok) break;
          aux_phase ^= 1u;
          aux_sent = false;
#pragma unroll
          for (int q = 0; q < 8; ++q) {
            const float4 v = *reinterpret_cast<const float4*>(mine + lane * 128 + ((q ^ (lane & 7)) << 4));
            h[4 * q] = v.x;
            h[4 * q + 1] = v.y;
            h[4 * q + 2] = v.z;
            h[4 * q + 3] = v.w;
          }
        }
        if (args.epi != kEpiNone && live) epilogue32(args, acc, h);
        if (direct_aux && j + kStep < kGroups) load_aux32(args, (size_t)row, nb + 32 * kStep, h);
        if (box) {
          if (!box_aux) {   // the warp's previous box has left (tanh': waited for below)
            if (lane == 0) asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");
            __syncwarp();
          }
#pragma unroll
          for (int q = 0; q < 8; ++q)
            *reinterpret_cast<uint4*>(mine + lane * 128 + ((q ^ (lane & 7)) << 4)) =
                make_uint4(acc[4 * q], acc[4 * q + 1], acc[4 * q + 2], acc[4 * q + 3]);
          tc::fence_async_smem();
          __syncwarp();
          if (lane == 0 && m * kBM + rw < args.M) {
            tma_store_2d(&map_c, mine, nb, m * kBM + rw);
            asm volatile("cp.async.bulk.commit_group;" ::: "memory");
          }
          if (box_aux) {   // the next tanh' box, once this one has been read out
            if (lane == 0) asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");
            const bool more = j + kStep < kGroups && nb + 32 * kStep < args.N;
            if (more) fetch_aux(m, j + kStep);
            else if (m + m_step < tiles_m) fetch_aux(m + m_step, warp >> 2);
          }
        } else if (TL::kBoxes && (args.beta != 0.0f || !args.vec)) {
          store_turned(args, acc, m * kBM + rw, nb, mine, lane);
        } else if (live) {
          store32(args, acc, (size_t)row, nb);
        }
      }
      if (!ok) break;
      tc::tc_fence_before();
      __syncwarp();
      if (lane == 0) tc::mbar_arrive(&bar->acc_empty[item & 1]);
    }
    if (box && lane == 0) {
      if (aux_sent) wait_landed(&bar->aux[warp], aux_phase);   // (only after a wait gave up)
      asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");
    }
  }
  tc::tc_fence_before();
  __syncthreads();
  if (tid == 0 && bar->abort) {
    atomicAdd(&args.st->timeouts, 1);
    atomicCAS(&args.st->code, 0, -4);
  }
  if (warp == kIssuer) {
    tc::tc_fence_after();
    tc::tmem_dealloc(tmem, 4 * BN);
  }
}

// ---------------------------------------------------------------------------
// fp32 on the CUDA cores.  Every output is a chain of FMAs in k, or, where K is
// split, such a chain per split, the splits' sums added in order: the same
// bits whichever kernel runs (a closed loop amplifies a changed rounding).
//
// Slices of 16 k are copied to shared memory as they are stored (cp.async, 16
// bytes where rows allow it): K-major operands as [row][16] padded to 20
// floats, read four k at a time, MN-major ones as [k][row], read four rows at
// a time; both without bank conflicts.
// ---------------------------------------------------------------------------
constexpr int kSl = 16, kSlPad = kSl + 4;

struct F32Args {
  int M, N, K;
  const float *A, *B;
  int lda, ldb;
  int seg;                // k per split (a multiple of 8)
  float* C;
  int ldc;
  float beta;
  float* ws;              // split partials, or null (write C)
  int m_pad, n_pad;
  int epi;
  const float* aux;
  int ld_aux;
};

__device__ __forceinline__ void cp_async(float* dst, const float* src, int bytes, bool vec) {
  const uint32_t d = tc::smem_u32(dst);
  if (vec)
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(d), "l"(src), "r"(bytes) : "memory");
  else
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(d), "l"(src), "r"(bytes) : "memory");
}

// Copies of rows r0 .. r0 + ROWS - 1 (below R) of an operand, 16 k at a time
// from k_begin (below k_end), into shared memory by NT threads; absent
// elements become zero.  A thread's addresses are worked out once.
template <int ROWS, bool MN, bool VEC, int NT>
struct F32Loader {
  static constexpr int W = VEC ? 4 : 1, kItems = ROWS * kSl / W, kPer = (kItems + NT - 1) / NT;
  const float* src[kPer];
  int off[kPer], kk[kPer], rows[kPer];   // shared-memory offset, k in the slice, rows below R
  size_t step;
  int k_end;

  __device__ __forceinline__ void init(const float* X, int ld, int r0, int R, int k_begin, int k_end_, int t) {
    k_end = k_end_;
    step = MN ? (size_t)kSl * ld : kSl;
#pragma unroll
    for (int i = 0; i < kPer; ++i) {
      const int e = i * NT + t;
      int r;
      if (MN) {
        kk[i] = e / (ROWS / W);
        r = e % (ROWS / W) * W;
        off[i] = kk[i] * (ROWS + 4) + r;
        rows[i] = min(W, R - r0 - r);
        src[i] = X + (size_t)(k_begin + kk[i]) * ld + r0 + r;
      } else {
        r = e / (kSl / W);
        kk[i] = e % (kSl / W) * W;
        off[i] = r * kSlPad + kk[i];
        rows[i] = r0 + r < R ? W : 0;
        src[i] = X + (size_t)(r0 + r) * ld + k_begin + kk[i];
      }
      if (kItems % NT != 0 && e >= kItems) rows[i] = -W;   // no such item
    }
  }
  // The slice from k kb (the next one on every call); X: any address of the operand.
  __device__ __forceinline__ void fetch(float* dst, const float* X, int kb) {
#pragma unroll
    for (int i = 0; i < kPer; ++i) {
      if (kItems % NT == 0 || rows[i] > -W) {
        int have = rows[i];
        if (kb + kSl > k_end) have = MN ? (kb + kk[i] < k_end ? have : 0) : min(have, k_end - kb - kk[i]);
        have = max(have, 0);
        cp_async(dst + off[i], have ? src[i] : X, 4 * have, VEC);
      }
      src[i] += step;
    }
  }
};

template <int ROWS, bool MN>
constexpr int f32_slice_floats() {
  return MN ? kSl * (ROWS + 4) : ROWS * kSlPad;
}

// Rows of one thread: TM of them (4 per group), thread t of T along the tile.
template <int T, bool MN>
__device__ __forceinline__ int f32_row(int t, int i) {
  return MN ? t * 4 + (i & 3) + (i >> 2) * 4 * T : t + T * i;
}

// acc += over k k0 .. k0 + 7 of a slice (TM x 8 outputs per thread).
template <int BM, int BN, int TM, bool A_MN, bool B_MN>
__device__ __forceinline__ void f32_mac8(const float* As, const float* Bs, int k0, int ty, int tx,
                                         float (&acc)[TM][8]) {
  constexpr int TY = BM / TM, TX = BN / 8;
#pragma unroll
  for (int q = 0; q < 8; q += 4) {
    float a[TM][4];
    if (A_MN) {
#pragma unroll
      for (int kk = 0; kk < 4; ++kk)
#pragma unroll
        for (int g = 0; g < TM / 4; ++g) {
          const float4 v = *reinterpret_cast<const float4*>(As + (k0 + q + kk) * (BM + 4) + ty * 4 + g * 4 * TY);
          a[4 * g][kk] = v.x;
          a[4 * g + 1][kk] = v.y;
          a[4 * g + 2][kk] = v.z;
          a[4 * g + 3][kk] = v.w;
        }
    } else {
#pragma unroll
      for (int i = 0; i < TM; ++i) {
        const float4 v = *reinterpret_cast<const float4*>(As + (ty + TY * i) * kSlPad + k0 + q);
        a[i][0] = v.x;
        a[i][1] = v.y;
        a[i][2] = v.z;
        a[i][3] = v.w;
      }
    }
    if (B_MN) {
#pragma unroll
      for (int kk = 0; kk < 4; ++kk) {
        const float* row = Bs + (k0 + q + kk) * (BN + 4) + tx * 4;
        const float4 u = *reinterpret_cast<const float4*>(row);
        const float4 v = *reinterpret_cast<const float4*>(row + 4 * TX);
        const float b[8] = {u.x, u.y, u.z, u.w, v.x, v.y, v.z, v.w};
#pragma unroll
        for (int i = 0; i < TM; ++i)
#pragma unroll
          for (int j = 0; j < 8; ++j) acc[i][j] = fmaf(a[i][kk], b[j], acc[i][j]);
      }
    } else {
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        const float4 v = *reinterpret_cast<const float4*>(Bs + (tx + TX * j) * kSlPad + k0 + q);
        const float b[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
        for (int kk = 0; kk < 4; ++kk)
#pragma unroll
          for (int i = 0; i < TM; ++i) acc[i][j] = fmaf(a[i][kk], b[kk], acc[i][j]);
      }
    }
  }
}

__device__ __forceinline__ void f32_store(const F32Args& a, int z, int m, int n, float x) {
  if (m >= a.M || n >= a.N) return;
  if (a.ws) {   // partials of the elements the reduction reads
    a.ws[((size_t)z * a.m_pad + m) * a.n_pad + n] = x;
    return;
  }
  float* c = a.C + (size_t)m * a.ldc + n;
  const float h = a.epi == kEpiDtanh ? a.aux[(size_t)m * a.ld_aux + n] : 0.0f;
  *c = a.beta != 0.0f ? fmaf(a.beta, *c, x) : epilogue(a.epi, x, h);
}

template <int BM, int BN>
struct F32Tile {
  static constexpr int TM = BM >= 128 ? 8 : 4;
  static constexpr int kThreads = (BM / TM) * (BN / 8);
  static constexpr int kStages = 3;
  template <bool A_MN, bool B_MN>
  static constexpr int smem_floats() {
    return kStages * (f32_slice_floats<BM, A_MN>() + f32_slice_floats<BN, B_MN>());
  }
};

// A BM x BN tile per CTA, TM x 8 outputs per thread, three slices in flight.
// SEG: every split's chain in turn, its sum added to the total (blockIdx.z is
// 0); else one split per blockIdx.z.  FMA issue and shared-memory reads bound
// them (half to two thirds of the FP32 peak).  64 x 64 tiles, three CTAs an SM,
// serve most shapes: the 8 x 8 outputs of a 128 x 128 tile's thread leave few
// registers, which K-major rows read four k at a time spill, and two CTAs an SM
// finish in coarse waves (launch_fp32_any has the lines).  16- and 32-row tiles
// for the heads' weight gradients.  Against scalar loads through registers:
// 256 x 264 x 30,011 175 -> 113 us, 12 x 264 x 131,072 270 -> 90 us,
// 4,096 x 256 x 264 (five splits) 27 us and a 14 us reduction -> 26 us.
template <int BM, int BN, bool A_MN, bool B_MN, bool VEC, bool SEG>
__global__ void __launch_bounds__((F32Tile<BM, BN>::kThreads), (BM >= 128 ? 2 : 3))
k_gemm_fp32(const F32Args args) {
  using TL = F32Tile<BM, BN>;
  constexpr int TM = TL::TM, TY = BM / TM, TX = BN / 8, NT = TL::kThreads, S = TL::kStages;
  constexpr int kA = f32_slice_floats<BM, A_MN>(), kB = f32_slice_floats<BN, B_MN>();
  extern __shared__ __align__(16) float f32_smem[];
  const int tid = threadIdx.x, tx = tid % TX, ty = tid / TX;
  const int m0 = blockIdx.x * BM, n0 = blockIdx.y * BN;
  const int k_begin = SEG ? 0 : blockIdx.z * args.seg;
  const int k_end = SEG ? args.K : min(args.K, k_begin + args.seg);
  F32Loader<BM, A_MN, VEC, NT> load_a;
  F32Loader<BN, B_MN, VEC, NT> load_b;
  load_a.init(args.A, args.lda, m0, args.M, k_begin, k_end, tid);
  load_b.init(args.B, args.ldb, n0, args.N, k_begin, k_end, tid);
  auto fetch = [&](int kb, int stage) {
    if (kb < k_end) {
      float* d = f32_smem + stage * (kA + kB);
      load_a.fetch(d, args.A, kb);
      load_b.fetch(d + kA, args.B, kb);
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  float acc[TM][8] = {}, total[SEG ? TM : 1][SEG ? 8 : 1];
  int seg_end = args.seg;
  bool first = true;
#pragma unroll
  for (int s = 0; s < S - 1; ++s) fetch(k_begin + s * kSl, s);
  int stage = 0;
  for (int kb = k_begin; kb < k_end; kb += kSl) {
    asm volatile("cp.async.wait_group %0;" ::"n"(S - 2) : "memory");
    __syncthreads();   // this slice has landed for everyone; the one before is consumed
    fetch(kb + (S - 1) * kSl, stage == 0 ? S - 1 : stage - 1);
    const float* As = f32_smem + stage * (kA + kB);
#pragma unroll
    for (int k8 = 0; k8 < kSl; k8 += 8) {
      f32_mac8<BM, BN, TM, A_MN, B_MN>(As, As + kA, k8, ty, tx, acc);
      if (SEG && kb + k8 + 8 == seg_end) {
        seg_end += args.seg;
#pragma unroll
        for (int i = 0; i < TM; ++i)
#pragma unroll
          for (int j = 0; j < 8; ++j) {
            total[SEG ? i : 0][SEG ? j : 0] = first ? acc[i][j] : total[SEG ? i : 0][SEG ? j : 0] + acc[i][j];
            acc[i][j] = 0.0f;
          }
        first = false;
      }
    }
    stage = stage + 1 == S ? 0 : stage + 1;
  }
  const bool tail = SEG && seg_end - args.seg < args.K;   // the last split ends at K, not at its full length
#pragma unroll
  for (int i = 0; i < TM; ++i)
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      float x = acc[i][j];
      if (SEG) x = !tail ? total[SEG ? i : 0][SEG ? j : 0] : (first ? x : total[SEG ? i : 0][SEG ? j : 0] + x);
      f32_store(args, blockIdx.z, m0 + f32_row<TY, A_MN>(ty, i), n0 + f32_row<TX, B_MN>(tx, j), x);
    }
}

// Large products with rows off 16 bytes, which cp.async can only copy float by
// float: a 128 x 128 tile per CTA, 8 x 8 outputs per thread, slices of 8 k
// through registers into two buffers of [k][row] whichever way the operands are
// stored (rows padded by 4 floats: the K-major stores, 8 k of 4 rows per warp,
// land in 32 distinct banks).  30,011 x 1,024 x 1,032 from odd rows: 1.43 to
// 1.47 ms, 1.67 to 1.72 in 64 x 64 tiles.
template <bool A_MN, bool B_MN>
__global__ void __launch_bounds__(256, 2) k_gemm_fp32_regs(const F32Args args) {
  __shared__ __align__(16) float As[2][8][132];
  __shared__ __align__(16) float Bs[2][8][132];
  const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
  const int m0 = blockIdx.x * 128, n0 = blockIdx.y * 128;
  const int k_begin = blockIdx.z * args.seg, k_end = min(args.K, k_begin + args.seg);
  // element e of a 128 x 8 slice, consecutive threads along the stored index
  auto coord = [](int e, bool mn, int& r, int& kk) {
    r = mn ? e % 128 : e >> 3;
    kk = mn ? e / 128 : e & 7;
  };
  auto load = [&](const float* X, int ld, bool mn, int r0, int R, int kb, float (&v)[4]) {
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      int r, kk;
      coord(tid + 256 * q, mn, r, kk);
      const int rr = r0 + r, k = kb + kk;
      v[q] = rr < R && k < k_end ? __ldg(mn ? X + (size_t)k * ld + rr : X + (size_t)rr * ld + k) : 0.0f;
    }
  };
  auto store = [&](float (&S)[8][132], bool mn, const float (&v)[4]) {
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      int r, kk;
      coord(tid + 256 * q, mn, r, kk);
      S[kk][r] = v[q];
    }
  };
  float acc[8][8] = {}, va[4], vb[4];
  load(args.A, args.lda, A_MN, m0, args.M, k_begin, va);
  load(args.B, args.ldb, B_MN, n0, args.N, k_begin, vb);
  store(As[0], A_MN, va);
  store(Bs[0], B_MN, vb);
  __syncthreads();
  int buf = 0;
  for (int kb = k_begin; kb < k_end; kb += 8) {
    const bool more = kb + 8 < k_end;
    if (more) {   // the next slice in flight during this one
      load(args.A, args.lda, A_MN, m0, args.M, kb + 8, va);
      load(args.B, args.ldb, B_MN, n0, args.N, kb + 8, vb);
    }
#pragma unroll
    for (int kk = 0; kk < 8; ++kk) {
      float a[8], b[8];
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const float4 u = *reinterpret_cast<const float4*>(&As[buf][kk][64 * h + ty * 4]);
        const float4 v = *reinterpret_cast<const float4*>(&Bs[buf][kk][64 * h + tx * 4]);
        a[4 * h] = u.x, a[4 * h + 1] = u.y, a[4 * h + 2] = u.z, a[4 * h + 3] = u.w;
        b[4 * h] = v.x, b[4 * h + 1] = v.y, b[4 * h + 2] = v.z, b[4 * h + 3] = v.w;
      }
#pragma unroll
      for (int i = 0; i < 8; ++i)
#pragma unroll
        for (int j = 0; j < 8; ++j) acc[i][j] = fmaf(a[i], b[j], acc[i][j]);
    }
    if (more) {
      store(As[buf ^ 1], A_MN, va);
      store(Bs[buf ^ 1], B_MN, vb);
    }
    __syncthreads();
    buf ^= 1;
  }
#pragma unroll
  for (int i = 0; i < 8; ++i)
#pragma unroll
    for (int j = 0; j < 8; ++j)
      f32_store(args, blockIdx.z, m0 + f32_row<16, true>(ty, i), n0 + f32_row<16, true>(tx, j), acc[i][j]);
}

// Narrow or few tiles: each warp computes a 32 x 32 block over one split with
// slices of its own (no block-wide barrier in the loop).  WS = 8: the CTA's
// warps take the splits (at most eight) of one block and add their sums in
// order; WS = 1 (no split): eight blocks of 32 rows.
constexpr int kWarpSlice = 2 * 32 * kSlPad;   // A and B slice floats of one warp (MN-major B: 16 x 36 fits)
constexpr int kWarpStages = 2;
constexpr int kWarpSmem = 8 * kWarpStages * kWarpSlice * 4;

template <bool B_MN, bool VEC, int WS>
__global__ void __launch_bounds__(256, 2) k_gemm_fp32_warps(const F32Args args) {
  static_assert(f32_slice_floats<32, true>() <= 32 * kSlPad, "slice room");
  extern __shared__ __align__(16) float f32_smem[];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, tx = lane & 3, ty = lane >> 2;
  const int m0 = (blockIdx.x * (8 / WS) + (WS == 1 ? warp : 0)) * 32, n0 = blockIdx.y * 32;
  const int k_begin = WS == 1 ? 0 : warp * args.seg;
  const int k_end = min(args.K, k_begin + args.seg);
  float* mine = f32_smem + warp * kWarpStages * kWarpSlice;
  F32Loader<32, false, VEC, 32> load_a;
  F32Loader<32, B_MN, VEC, 32> load_b;
  load_a.init(args.A, args.lda, m0, args.M, k_begin, k_end, lane);
  load_b.init(args.B, args.ldb, n0, args.N, k_begin, k_end, lane);
  auto fetch = [&](int kb, int stage) {
    if (kb < k_end) {
      float* d = mine + stage * kWarpSlice;
      load_a.fetch(d, args.A, kb);
      load_b.fetch(d + 32 * kSlPad, args.B, kb);
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  float acc[4][8] = {};
  fetch(k_begin, 0);
  int stage = 0;
  for (int kb = k_begin; kb < k_end; kb += kSl) {
    fetch(kb + kSl, stage ^ 1);
    asm volatile("cp.async.wait_group 1;" ::: "memory");
    __syncwarp();
    const float* As = mine + stage * kWarpSlice;
    f32_mac8<32, 32, 4, false, B_MN>(As, As + 32 * kSlPad, 0, ty, tx, acc);
    f32_mac8<32, 32, 4, false, B_MN>(As, As + 32 * kSlPad, 8, ty, tx, acc);
    __syncwarp();   // the slice is read before the next copy overwrites it
    stage ^= 1;
  }
  if (WS == 1) {
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int j = 0; j < 8; ++j)
        f32_store(args, 0, m0 + f32_row<8, false>(ty, i), n0 + f32_row<4, B_MN>(tx, j), acc[i][j]);
    return;
  }
  // the splits' sums through shared memory, 33 floats a row, then in order
  asm volatile("cp.async.wait_group 0;" ::: "memory");
  __syncthreads();
  float* part = f32_smem + warp * 32 * 33;
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < 8; ++j) part[f32_row<8, false>(ty, i) * 33 + f32_row<4, B_MN>(tx, j)] = acc[i][j];
  __syncthreads();
  const int splits = (args.K + args.seg - 1) / args.seg;
#pragma unroll
  for (int e0 = 0; e0 < 4; ++e0) {
    const int r = warp + 8 * e0;
    float x = f32_smem[r * 33 + lane];
    for (int z = 1; z < splits; ++z) x += f32_smem[(z * 32 + r) * 33 + lane];
    f32_store(args, 0, m0 + r, n0 + lane, x);
  }
}

// ---------------------------------------------------------------------------
// A step's weight gradients (bf16, both operands along the samples) in one
// launch of at most one CTA per SM.  The work is cut into units, a 128-row tile
// of an item over one K range of it; the ranges are those of the item's product
// launched alone (group_ranges), so that a gradient has the same bits whatever
// shares its launch.  CTA c takes wide units (more than 192 columns) c, c + G,
// ... and narrow ones from the other end, a wide and a narrow one in turn: each
// kind has its own columns of tensor memory, so one unit's partials are read
// out under the next one's MMAs, and the reads stay even over the SMs.  The
// hidden layers' launch at 65,536 samples of both networks moves 286 MB into the
// SMs in 49 us (cold): DRAM is at 63 %, L2 at 57 % and the tensor pipe at 17 % of
// their peaks.
// 32 PPO steps of 65,536 samples: 9.08 ms with a launch per product, 8.17 here
// (8.00 with longer ranges, fewer partials and a third of the chains, whose
// sums are others).
// ---------------------------------------------------------------------------
struct GroupMaps {
  CUtensorMap a[kMaxGroup], b[kMaxGroup];
};
struct GroupArgs {
  struct Item {
    int M, N, splits, per_split;   // K ranges, K-chunks in each
    int unit0;                     // its first unit of its kind
    float* ws;                     // [splits][M][n_pad]
    int n_pad;
    float* C;
    int ldc;
  } it[kMaxGroup];
  int n, chunks;
  int units[2];                    // wide, narrow
  Status* st;
};

struct GroupTile {
  static constexpr int kBK = 64;
  static constexpr uint32_t kBlock = kBK * 128;          // 64 K-rows of 128 bytes
  static constexpr uint32_t kABytes = 2 * kBlock, kBBytes = 5 * kBlock, kStage = kABytes + kBBytes;
  static constexpr int kStages = 3;
  static constexpr uint32_t kSmem = kStages * kStage + 256 + 1024;
  static constexpr int kNarrow = 192;                    // columns of a narrow unit, at most
  static constexpr uint32_t kNarrowCol = 512 - kNarrow;  // its accumulator's first column
};

struct GroupBars {
  uint64_t full[GroupTile::kStages], empty[GroupTile::kStages];
  uint64_t acc_full[2], acc_empty[2];                    // wide, narrow accumulator
  uint64_t done;
  uint32_t tmem_base;
  int abort;
};

// The j-th unit of this CTA: its kind (j odd: narrow), item, row tile, K range.
struct GroupUnit {
  int kind, q, m0, z, c0, n_chunks;
};
__device__ __forceinline__ bool group_unit(const GroupArgs& args, int j, GroupUnit* u) {
  const int G = (int)gridDim.x;
  u->kind = j & 1;
  const int index = (u->kind ? G - 1 - (int)blockIdx.x : (int)blockIdx.x) + (j >> 1) * G;
  if (index >= args.units[u->kind]) return false;
  u->q = -1;
  for (int k = 0; k < args.n; ++k)
    if ((args.it[k].N <= GroupTile::kNarrow ? 1 : 0) == u->kind && index >= args.it[k].unit0) u->q = k;
  const GroupArgs::Item& it = args.it[u->q];
  const int local = index - it.unit0;
  u->z = local % it.splits;
  u->m0 = local / it.splits * kBM;
  u->c0 = u->z * it.per_split;
  u->n_chunks = min(args.chunks, u->c0 + it.per_split) - u->c0;
  return true;
}
// Units of the CTA that takes most, empty places included.
__device__ __forceinline__ int group_turns(const GroupArgs& args) {
  return 2 * ((max(args.units[0], args.units[1]) + (int)gridDim.x - 1) / (int)gridDim.x);
}

__global__ void __launch_bounds__(192, 1)
k_gemm_group(const __grid_constant__ GroupMaps maps, const __grid_constant__ GroupArgs args) {
  using TL = GroupTile;
  constexpr int kStages = TL::kStages, kProducer = 4, kIssuer = 5;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>(
      (reinterpret_cast<uintptr_t>(smem_raw) + 1023u) & ~(uintptr_t)1023u);
  GroupBars* bar = reinterpret_cast<GroupBars*>(smem + kStages * TL::kStage);
  volatile int* abort = &bar->abort;
  const int tid = threadIdx.x, warp = tid >> 5;
  const int turns = group_turns(args);

  if (tid == 0) {
    for (int s = 0; s < kStages; ++s) {
      tc::mbar_init(&bar->full[s], 1);
      tc::mbar_init(&bar->empty[s], 1);
    }
    for (int k = 0; k < 2; ++k) {
      tc::mbar_init(&bar->acc_full[k], 1);
      tc::mbar_init(&bar->acc_empty[k], 4);
    }
    tc::mbar_init(&bar->done, 1);
    bar->abort = 0;
    tc::mbar_fence_init();
  }
  if (warp == kIssuer) {
    tc::tmem_alloc(&bar->tmem_base, 512);
    tc::tmem_relinquish();
  }
  tc::tc_fence_before();
  __syncthreads();
  tc::tc_fence_after();
  const uint32_t tmem = bar->tmem_base;

  if (warp == kProducer) {
    if ((tid & 31) == 0) {
      int s = 0, fill = 0;   // next stage, and how often the ring has gone round
      bool ok = true;
      GroupUnit u;
      for (int j = 0; j < turns && ok; ++j) {
        if (!group_unit(args, j, &u)) continue;
        const GroupArgs::Item& it = args.it[u.q];
        const int na = min(2, (it.M - u.m0 + 63) / 64), nb = (it.N + 63) / 64;
        for (int c = 0; c < u.n_chunks; ++c) {
          ok = fill == 0 || tc::mbar_wait(&bar->empty[s], (uint32_t)(fill - 1) & 1u, abort, kWaitLimitNs);
          if (!ok) break;
          uint8_t* dst = smem + s * TL::kStage;
          const int k = (u.c0 + c) * TL::kBK;
          tc::mbar_arrive_expect_tx(&bar->full[s], (na + nb) * TL::kBlock);
#pragma unroll
          for (int i = 0; i < 2; ++i)
            if (i < na) tma_load_2d(dst + i * TL::kBlock, &maps.a[u.q], u.m0 + 64 * i, k, &bar->full[s]);
#pragma unroll
          for (int i = 0; i < 5; ++i)
            if (i < nb) tma_load_2d(dst + TL::kABytes + i * TL::kBlock, &maps.b[u.q], 64 * i, k, &bar->full[s]);
          if (++s == kStages) {
            s = 0;
            ++fill;
          }
        }
      }
      if (*abort)   // the copies still in flight
        for (int q = 0; q < kStages; ++q) {
          const int fills = fill + (q < s ? 1 : 0);
          if (fills > 0) wait_landed(&bar->full[q], (uint32_t)(fills - 1) & 1u);
        }
    }
    __syncwarp();
  } else if (warp == kIssuer) {
    if ((tid & 31) == 0) {
      const uint32_t base = tc::smem_u32(smem);
      int s = 0;
      uint32_t phase = 0;
      bool ok = true;
      GroupUnit u;
      for (int j = 0; j < turns && ok; ++j) {
        if (!group_unit(args, j, &u)) continue;
        const int N = args.it[u.q].N, use = j >> 1;   // use: of this kind's accumulator
        // columns in one MMA of up to 256, the rest in a second
        const uint32_t id1 = idesc(false, true, true, kBM, min(256, (N + 15) / 16 * 16));
        const uint32_t id2 = idesc(false, true, true, kBM, max(16, (N - 256 + 15) / 16 * 16));
        const uint32_t d = tmem + (u.kind ? TL::kNarrowCol : 0u);
        ok = use == 0 || tc::mbar_wait(&bar->acc_empty[u.kind], (uint32_t)(use - 1) & 1u, abort, kWaitLimitNs);
        if (ok) tc::tc_fence_after();
        for (int c = 0; c < u.n_chunks && ok; ++c) {
          ok = tc::mbar_wait(&bar->full[s], phase, abort, kWaitLimitNs);
          if (!ok) break;
          tc::tc_fence_after();
          const uint32_t a0 = base + s * TL::kStage, b0 = a0 + TL::kABytes;
#pragma unroll
          for (int kk = 0; kk < 4; ++kk) {
            const uint32_t acc = c > 0 || kk > 0 ? 1u : 0u;
            const uint64_t da = desc_sw128(a0 + kk * 2048, TL::kBlock, 1024);
            mma<false>(d, da, desc_sw128(b0 + kk * 2048, TL::kBlock, 1024), id1, acc);
            if (N > 256)
              mma<false>(d + 256, da, desc_sw128(b0 + 4 * TL::kBlock + kk * 2048, TL::kBlock, 1024), id2, acc);
          }
          tc::mma_commit(&bar->empty[s]);
          if (++s == kStages) {
            s = 0;
            phase ^= 1u;
          }
        }
        if (ok) tc::mma_commit(&bar->acc_full[u.kind]);
      }
      tc::mma_commit(&bar->done);
      wait_landed(&bar->done, 0);   // tensor memory is freed below
    }
    __syncwarp();
  } else {
    const uint32_t lane_addr = tmem + ((uint32_t)(warp * 32) << 16);
    GroupUnit u;
    for (int j = 0; j < turns; ++j) {
      if (!group_unit(args, j, &u)) continue;
      const GroupArgs::Item& it = args.it[u.q];
      const bool ok = tc::mbar_wait(&bar->acc_full[u.kind], (uint32_t)(j >> 1) & 1u, abort, kWaitLimitNs);
      if (!__all_sync(0xFFFFFFFFu, ok)) break;
      tc::tc_fence_after();
      const int row = u.m0 + tid;
      const uint32_t col = u.kind ? TL::kNarrowCol : 0u;
#pragma unroll 1
      for (int nb = 0; nb < it.N; nb += 32) {
        uint32_t acc[32];
        tc::tmem_ld32(lane_addr + col + nb, acc);
        tc::tmem_ld_wait(acc);
        if (row < it.M) {
          float* dst = it.ws + ((size_t)u.z * it.M + row) * it.n_pad + nb;
#pragma unroll
          for (int i = 0; i < 4; ++i) st_f32x8(dst + 8 * i, acc + 8 * i);
        }
      }
      tc::tc_fence_before();
      __syncwarp();
      if ((tid & 31) == 0) tc::mbar_arrive(&bar->acc_empty[u.kind]);
    }
  }
  tc::tc_fence_before();
  __syncthreads();
  if (tid == 0 && bar->abort) {
    atomicAdd(&args.st->timeouts, 1);
    atomicCAS(&args.st->code, 0, -4);
  }
  if (warp == kIssuer) {
    tc::tc_fence_after();
    tc::tmem_dealloc(tmem, 512);
  }
}

// C = beta C + sum_z ws[z], fp32 or bf16 output.  A weight gradient has a
// few tens of thousands of elements and tens of splits, so one thread per
// element summing every split in turn left the kernel bound by load latency
// at under two blocks per SM.  Here a block of 256 threads covers 128
// consecutive elements (32 groups of four, 16-byte loads) for 8 groups of
// splits: thread (g, l) adds the partials z = g, g + 8, g + 16, ... of its
// four elements in increasing z, and the eight group sums are then added in
// the order g = 0..7: a fixed order, the same on every run.
constexpr int kRedGroups = 8;
constexpr int kRedQuads = 32;
__device__ __forceinline__ void reduce_block(long block, int M, int N, int splits,
                                             const float* __restrict__ ws, int m_pad, int n_pad, void* C,
                                             int ldc, int c_bf16, float beta, int epi, const void* aux,
                                             int ld_aux) {
  __shared__ float4 part[kRedGroups][kRedQuads];
  const int lane = threadIdx.x % kRedQuads, grp = threadIdx.x / kRedQuads;
  const int qpr = (N + 3) / 4;   // groups of four per row (n_pad is a multiple of 32)
  const long quad = block * kRedQuads + lane;
  const bool live = quad < (long)M * qpr;
  const int m = live ? (int)(quad / qpr) : 0, n = live ? (int)(quad % qpr) * 4 : 0;
  const size_t zs = (size_t)m_pad * n_pad;
  const float* src = ws + (size_t)m * n_pad + n;
  // 16-byte loads when the workspace is 16-byte aligned (every offset here
  // is a multiple of four floats), four scalar loads otherwise
  const bool vec = (reinterpret_cast<uintptr_t>(ws) & 15u) == 0;
  auto load4 = [&](const float* a) {
    return vec ? __ldcs(reinterpret_cast<const float4*>(a))
               : make_float4(__ldcs(a), __ldcs(a + 1), __ldcs(a + 2), __ldcs(a + 3));
  };
  float4 v = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
  if (live) {
    constexpr int kU = 4;   // loads in flight per thread
    for (int z0 = grp; z0 < splits; z0 += kRedGroups * kU) {
      float4 p[kU];
#pragma unroll
      for (int q = 0; q < kU; ++q) {
        const int z = z0 + q * kRedGroups;
        p[q] = z < splits ? load4(src + (size_t)z * zs) : make_float4(0.0f, 0.0f, 0.0f, 0.0f);
      }
#pragma unroll
      for (int q = 0; q < kU; ++q)
        if (z0 + q * kRedGroups < splits) {
          v.x += p[q].x;
          v.y += p[q].y;
          v.z += p[q].z;
          v.w += p[q].w;
        }
    }
  }
  part[grp][lane] = v;
  __syncthreads();
  if (grp != 0 || !live) return;
  float4 s = part[0][lane];
#pragma unroll
  for (int g = 1; g < kRedGroups; ++g) {
    const float4 u = part[g][lane];
    s.x += u.x;
    s.y += u.y;
    s.z += u.z;
    s.w += u.w;
  }
  const float r[4] = {s.x, s.y, s.z, s.w};
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    if (n + j >= N) break;
    const float h = epi == kEpiDtanh ? aux_at(aux, ld_aux, c_bf16, (size_t)m, n + j) : 0.0f;
    const float v = c_bf16 && epi ? __uint_as_float(tc::pack_bf16x2(r[j], 0.0f) << 16) : r[j];
    float x = epilogue(epi, v, h);
    if (c_bf16) {
      uint16_t* c = static_cast<uint16_t*>(C) + (size_t)m * ldc + n + j;
      if (beta != 0.0f) x = fmaf(beta, __uint_as_float((uint32_t)*c << 16), x);
      *c = (uint16_t)(tc::pack_bf16x2(x, 0.0f) & 0xFFFFu);
    } else {
      float* c = static_cast<float*>(C) + (size_t)m * ldc + n + j;
      *c = beta != 0.0f ? fmaf(beta, *c, x) : x;
    }
  }
}

__global__ void __launch_bounds__(kRedGroups * kRedQuads)
k_reduce(int M, int N, int splits, const float* __restrict__ ws, int m_pad, int n_pad, void* C,
         int ldc, int c_bf16, float beta, int epi, const void* aux, int ld_aux) {
  reduce_block(blockIdx.x + pdl_enter(), M, N, splits, ws, m_pad, n_pad, C, ldc, c_bf16, beta, epi, aux, ld_aux);
}

// Every item of a group (blockIdx.y).
__global__ void __launch_bounds__(kRedGroups * kRedQuads)
k_reduce_group(const __grid_constant__ GroupArgs args) {
  const GroupArgs::Item& it = args.it[blockIdx.y];
  if ((long)blockIdx.x * kRedQuads >= (long)it.M * ((it.N + 3) / 4)) return;
  reduce_block(blockIdx.x, it.M, it.N, it.splits, it.ws, it.M, it.n_pad, it.C, it.ldc, 0, 0.0f, kEpiNone,
               nullptr, 0);
}

// An MN-major fp32 operand (element (r, k) at k * ld + r) copied K-major:
// out[r * ldo + k], 32 x 32 tiles through shared memory, both sides coalesced
// (tf32 operands that TMA cannot read in place: base or rows off 16 bytes).
__global__ void k_transpose(int R, int K, const float* __restrict__ in, int ld, float* out,
                            int ldo) {
  __shared__ float tile[32][33];
  const int r0 = blockIdx.x * 32, k0 = blockIdx.y * 32;
  for (int j = threadIdx.y; j < 32; j += 8) {
    const int k = k0 + j, r = r0 + threadIdx.x;
    tile[j][threadIdx.x] = (k < K && r < R) ? in[(size_t)k * ld + r] : 0.0f;
  }
  __syncthreads();
  for (int j = threadIdx.y; j < 32; j += 8) {
    const int r = r0 + j, k = k0 + threadIdx.x;
    if (r < R && k < ldo) out[(size_t)r * ldo + k] = k < K ? tile[threadIdx.x][j] : 0.0f;
  }
}

// ---------------------------------------------------------------------------
// host side
// ---------------------------------------------------------------------------
using EncodeFn = CUresult (*)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*,
                              const cuuint64_t*, const cuuint64_t*, const cuuint32_t*,
                              const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle,
                              CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

EncodeFn encode_fn() {
  static EncodeFn fn = nullptr;
  static std::once_flag once;
  std::call_once(once, [] {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault,
                                         &q) == cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn = reinterpret_cast<EncodeFn>(p);
    else
      cudaGetLastError();
  });
  return fn;
}

// 2-D map of a stored operand: inner dimension (contiguous) and outer
// dimension, rows ld elements apart; a box of 128 bytes x box_outer rows.
bool make_map(CUtensorMap* map, bool tf32, bool mn, const void* ptr, uint64_t inner, uint64_t outer,
              int ld, uint32_t box_outer) {
  EncodeFn fn = encode_fn();
  if (!fn) return false;
  const int es = tf32 ? 4 : 2;
  const cuuint64_t dims[2] = {inner, outer};
  const cuuint64_t strides[1] = {(cuuint64_t)ld * es};
  const cuuint32_t box[2] = {(cuuint32_t)(128 / es), box_outer};
  const cuuint32_t estr[2] = {1, 1};
  // tf32: the copy rounds each fp32 element to tf32 (nearest), as a tf32
  // GEMM rounds its operands, instead of the MMA dropping the low bits
  return fn(map, tf32 ? CU_TENSOR_MAP_DATA_TYPE_TFLOAT32 : CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2,
            const_cast<void*>(ptr), dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
            tf32 && mn ? CU_TENSOR_MAP_SWIZZLE_128B_ATOM_32B : CU_TENSOR_MAP_SWIZZLE_128B,
            CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// 2-D fp32 map of a row-major array's boxes of 32 columns (128 bytes, 16-byte
// pieces swizzled) x box_rows rows.
bool make_box_map(CUtensorMap* map, const void* ptr, uint64_t cols, uint64_t rows, int ld,
                  uint32_t box_rows) {
  EncodeFn fn = encode_fn();
  if (!fn) return false;
  const cuuint64_t dims[2] = {cols, rows};
  const cuuint64_t strides[1] = {(cuuint64_t)ld * 4};
  const cuuint32_t box[2] = {32, box_rows};
  const cuuint32_t estr[2] = {1, 1};
  return fn(map, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 2, const_cast<void*>(ptr), dims, strides, box, estr,
            CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
            CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

int sm_count_dev() {
  int dev = 0, v = 0;
  if (cudaGetDevice(&dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || v <= 0) {
    cudaGetLastError();
    return 148;
  }
  return v;
}

struct Plan {
  int bm, bn, bk;        // tile and K-chunk sizes
  int tiles_m, tiles_n;
  int chunks, per_split, splits;
  int m_pad, n_pad;
  bool rows;             // many rows, few K-chunks: k_gemm_rows
  int half;              // its first chunk of the second accumulator, or 0
  int fp32;              // Fp32Kernel
  int segments;          // fp32: splits added inside the kernel (1: none)
};

// fp32 kernels: a tile per CTA (partials in the workspace when split), the same
// with the splits in turn, or a warp per 32 x 32 block.
enum Fp32Kernel { kFp32Tiles, kFp32Seg, kFp32Warps };

constexpr int kRowsMaxChunks = RowTile<true, false, 128>::kMaxChunks;

// The narrow tile of k_gemm_rows: one 128-byte block of an MN-major B.
int narrow_bn(Prec prec) { return prec == kTf32 ? 32 : 64; }

Plan plan(Prec prec, int M, int N, int K, bool a_kmajor) {
  Plan p;
  p.rows = false;
  p.half = 0;
  p.fp32 = kFp32Tiles;
  p.segments = 1;
  if (prec == kFp32) {
    p.bm = M <= 32 ? 32 : 128;
    p.bn = 128;
    p.bk = 8;
  } else {
    p.bm = kBM;
    p.bk = prec == kTf32 ? 32 : 64;
    // 320-wide tiles (one CTA over the weight gradients' 264 augmented
    // columns: the other operand read once instead of three times) pay when
    // there are at least two M-tiles (28.1 against 37.9 us for 256 x 264 x
    // 65,536, bf16) or a long contraction: 16 x 264 x K in tf32 takes 21 / 35
    // / 95 us against 27 / 45 / 199 at K = 65,536 / 131,072 / 524,288, but 18
    // against 16 at 16,384.
    p.bn = (N > 128 && N <= 256) ? 256
                                 : ((N > 256 && N <= 320 && (M > kBM || K >= 1024 * p.bk)) ? 320 : 128);
    p.rows = a_kmajor && p.bn <= 256 && M >= 8 * kBM && K <= kRowsMaxChunks * p.bk;
  }
  p.tiles_m = (M + p.bm - 1) / p.bm;
  p.tiles_n = (N + p.bn - 1) / p.bn;
  p.chunks = std::max(1, (K + p.bk - 1) / p.bk);
  const int tiles = p.tiles_m * p.tiles_n;
  // CTAs wanted: one per SM for the tensor-core kernel, two for the
  // CUDA-core one (two 256-thread CTAs resident per SM hide its loads)
  const int sms = sm_count_dev() * (prec == kFp32 ? 2 : 1);
  int want = tiles >= sms / 2 ? 1 : (sms + tiles - 1) / tiles;
  // at least 4 K-chunks per CTA, at most one split per chunk
  want = std::max(1, std::min(want, p.chunks / 4));
  p.per_split = (p.chunks + want - 1) / want;
  p.splits = (p.chunks + p.per_split - 1) / p.per_split;
  if (prec == kFp32 && a_kmajor && p.splits <= 8) {
    // A product over rows: its few splits are added inside the kernel instead
    // of through partials in memory (4,096 x 256 x 264, five splits: 27 us and a
    // 14 us reduction).  A warp per block where the result is narrow or 64 x 64
    // tiles would leave SMs idle; a tile with the splits in turn while their
    // chain is short (4,096 x 256 x 512 41 to 43 us, 45 to 47 as partials; but
    // 4,096 x 512 x 520 103 us, 83, and 1,024^3 76 to 81 us, 69).
    const long small = (long)((M + 63) / 64) * ((N + 63) / 64);
    const bool warps = N <= 32 || (p.splits > 1 && small < sm_count_dev());
    if (warps || p.splits == 1 || K <= 512) {
      p.segments = p.splits;
      p.fp32 = warps ? kFp32Warps : (p.splits > 1 ? kFp32Seg : kFp32Tiles);
      p.splits = 1;
    }
  }
  if (p.rows) {   // nine chunks or fewer: at most two splits
    p.half = p.splits > 1 ? p.per_split : 0;
    p.splits = 1;
    p.bn = N <= narrow_bn(prec) ? narrow_bn(prec) : 128;
    p.tiles_n = (N + p.bn - 1) / p.bn;
  }
  p.m_pad = p.tiles_m * p.bm;
  p.n_pad = p.tiles_n * p.bn;
  return p;
}

template <bool TF32, bool A_MN, bool B_MN, int BN>
cudaError_t launch_tc(const Plan& P, const CUtensorMap& ma, const CUtensorMap& mb,
                      const TcArgs& a, cudaStream_t s) {
  using TL = Tile<TF32, A_MN, B_MN, BN>;
  auto kern = k_gemm_tc<TF32, A_MN, B_MN, BN>;
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, TL::kSmem);
  if (e != cudaSuccess) return e;
  return launch_pdl(kern, dim3(P.tiles_m, P.tiles_n, P.splits), 192, TL::kSmem, s, ma, mb, a);
}

template <bool TF32, int BN>
cudaError_t dispatch_major(bool a_mn, bool b_mn, const Plan& P, const CUtensorMap& ma,
                           const CUtensorMap& mb, const TcArgs& a, cudaStream_t s) {
  if (a_mn && b_mn) return launch_tc<TF32, true, true, BN>(P, ma, mb, a, s);
  if (a_mn) return launch_tc<TF32, true, false, BN>(P, ma, mb, a, s);
  if (b_mn) return launch_tc<TF32, false, true, BN>(P, ma, mb, a, s);
  return launch_tc<TF32, false, false, BN>(P, ma, mb, a, s);
}

template <bool TF32, bool B_MN, int BN>
cudaError_t launch_rows(const Plan& P, const CUtensorMap& ma, const CUtensorMap& mb, const TcArgs& a,
                        cudaStream_t s) {
  using TL = RowTile<TF32, B_MN, BN>;
  auto kern = k_gemm_rows<TF32, B_MN, BN>;
  const int chunks = P.chunks, stages = TL::stages(chunks);
  const uint32_t smem = TL::kFixed + chunks * TL::kBChunk + stages * TL::kStage;
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)TL::kBudget);
  if (e != cudaSuccess) return e;
  // result and tanh' boxes by TMA where the arrays allow it: fp32, 16-byte
  // rows, and whole 16-byte pieces up to column N (a store clips no finer)
  auto box_ok = [](const void* p, int ld) {
    return (reinterpret_cast<uintptr_t>(p) & 15u) == 0 && ld % 4 == 0;
  };
  CUtensorMap mc = ma, mx = ma;
  bool boxes = TL::kBoxes && !a.c_bf16 && a.beta == 0.0f && a.N % 4 == 0 && box_ok(a.C, a.ldc) &&
               (a.epi != kEpiDtanh || box_ok(a.aux, a.ld_aux));
  if (boxes) {
    boxes = make_box_map(&mc, a.C, a.N, a.M, a.ldc, 32) &&
            (a.epi != kEpiDtanh || make_box_map(&mx, a.aux, a.N, a.M, a.ld_aux, 32));
  }
  // every column tile on the same number of CTAs, at most kCtas per SM in all
  const int groups = std::max(1, std::min(P.tiles_m, sm_count_dev() * TL::kCtas / P.tiles_n));
  return launch_pdl(kern, groups * P.tiles_n, TL::kThreads, smem, s, ma, mb, mc, mx, a, P.tiles_m, P.tiles_n,
                    stages, P.half, boxes ? 1 : 0);
}

template <bool TF32>
cudaError_t dispatch_rows(bool b_mn, const Plan& P, const CUtensorMap& ma, const CUtensorMap& mb,
                          const TcArgs& a, cudaStream_t s) {
  constexpr int kNarrow = TF32 ? 32 : 64;
  if (P.bn == 128)
    return b_mn ? launch_rows<TF32, true, 128>(P, ma, mb, a, s) : launch_rows<TF32, false, 128>(P, ma, mb, a, s);
  return b_mn ? launch_rows<TF32, true, kNarrow>(P, ma, mb, a, s)
              : launch_rows<TF32, false, kNarrow>(P, ma, mb, a, s);
}

template <int BM, int BN, bool A_MN, bool B_MN, bool VEC, bool SEG>
cudaError_t launch_fp32_tile(const Plan& P, const F32Args& a, cudaStream_t s) {
  using TL = F32Tile<BM, BN>;
  auto kern = k_gemm_fp32<BM, BN, A_MN, B_MN, VEC, SEG>;
  constexpr int smem = TL::template smem_floats<A_MN, B_MN>() * 4;
  if constexpr (smem > 48 * 1024) {
    const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e != cudaSuccess) return e;
  }
  kern<<<dim3((a.M + BM - 1) / BM, (a.N + BN - 1) / BN, SEG ? 1 : P.splits), TL::kThreads, smem, s>>>(a);
  return cudaGetLastError();
}

template <bool B_MN, bool VEC>
cudaError_t launch_fp32_warps(const Plan& P, const F32Args& a, cudaStream_t s) {
  auto kern = P.segments > 1 ? k_gemm_fp32_warps<B_MN, VEC, 8> : k_gemm_fp32_warps<B_MN, VEC, 1>;
  const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, kWarpSmem);
  if (e != cudaSuccess) return e;
  const int rows = P.segments > 1 ? 32 : 256;
  kern<<<dim3((a.M + rows - 1) / rows, (a.N + 31) / 32), 256, kWarpSmem, s>>>(a);
  return cudaGetLastError();
}

template <bool A_MN, bool B_MN>
cudaError_t launch_fp32_regs(const Plan& P, const F32Args& a, cudaStream_t s) {
  k_gemm_fp32_regs<A_MN, B_MN><<<dim3((a.M + 127) / 128, (a.N + 127) / 128, P.splits), 256, 0, s>>>(a);
  return cudaGetLastError();
}

// 64 x 64 tiles, but
//  - up to 32 rows: tiles of 16 or 32 (24 x 264 x 30,000: 35 us, 62 in 128 rows);
//  - 128 x 128 tiles: an MN-major A in three waves of them or more (30,011 x
//    1,024 x 1,032 1.18 to 1.27 ms, 1.28 to 1.33 in 64 x 64 tiles; but 30,011 x
//    256 x 264, 1.5 waves, 109 to 111 us, 97 to 99, and with a K-major A 122 to
//    140 us, 103 to 105), or just one full wave of whole ones (128 x 128 x
//    128,000 92 to 103 us, 101 to 109);
//  - many rows of 257 to 288 columns: three column tiles of 96 instead of five of
//    64 (30,011 x 264 x 256: 107 to 111 us, 113 to 117);
//  - large products off 16 bytes: through registers (65,536 x 256 x 264 225 to 230
//    us, 249 to 263 in 64 x 64 tiles; below half of that size the tiles are as
//    fast or faster: 30,011 x 129 x 264 117 to 119 us, 95 to 98).
template <bool A_MN, bool B_MN, bool VEC>
cudaError_t launch_fp32_any(const Plan& P, const F32Args& a, cudaStream_t s) {
  if constexpr (!A_MN) {
    if (P.fp32 == kFp32Warps) return launch_fp32_warps<B_MN, VEC>(P, a, s);
    if (P.fp32 == kFp32Seg) return launch_fp32_tile<64, 64, A_MN, B_MN, VEC, true>(P, a, s);
  }
  if (a.M <= 16) return launch_fp32_tile<16, 128, A_MN, B_MN, VEC, false>(P, a, s);
  if (a.M <= 32) return launch_fp32_tile<32, 128, A_MN, B_MN, VEC, false>(P, a, s);
  const int sms = sm_count_dev();
  const long ctas = (long)((a.M + 127) / 128) * ((a.N + 127) / 128) * P.splits;   // of 128 x 128 tiles
  const bool whole = a.M % 128 == 0 && a.N % 128 == 0 && ctas <= 2 * sms && ctas > 2 * sms * 9 / 10;
  if constexpr ((A_MN && B_MN) || (VEC && (A_MN || B_MN))) {
    if (whole || (A_MN && ctas > 6 * sms)) return launch_fp32_tile<128, 128, A_MN, B_MN, VEC, false>(P, a, s);
  }
  if constexpr (VEC) {
    if (a.N > 256 && a.N <= 288 && a.M >= 128 * sms) return launch_fp32_tile<128, 96, A_MN, B_MN, VEC, false>(P, a, s);
  } else if constexpr (!(A_MN && B_MN)) {
    const long tiles = (long)((a.M + 63) / 64) * ((a.N + 63) / 64);
    if (whole || (P.splits == 1 && tiles * a.K >= 500000)) return launch_fp32_regs<A_MN, B_MN>(P, a, s);
  }
  return launch_fp32_tile<64, 64, A_MN, B_MN, VEC, false>(P, a, s);
}

cudaError_t launch_fp32(const Plan& P, const F32Args& a, bool a_mn, bool b_mn, cudaStream_t s) {
  // 16-byte copies where every row of both operands starts on 16 bytes
  const bool vec = ((reinterpret_cast<uintptr_t>(a.A) | reinterpret_cast<uintptr_t>(a.B)) & 15u) == 0 &&
                   a.lda % 4 == 0 && a.ldb % 4 == 0;
  if (a_mn)
    return b_mn ? (vec ? launch_fp32_any<true, true, true>(P, a, s) : launch_fp32_any<true, true, false>(P, a, s))
                : (vec ? launch_fp32_any<true, false, true>(P, a, s) : launch_fp32_any<true, false, false>(P, a, s));
  return b_mn ? (vec ? launch_fp32_any<false, true, true>(P, a, s) : launch_fp32_any<false, true, false>(P, a, s))
              : (vec ? launch_fp32_any<false, false, true>(P, a, s) : launch_fp32_any<false, false, false>(P, a, s));
}

bool tma_ok(const Operand& o, int es) {
  return (reinterpret_cast<uintptr_t>(o.ptr) & 15u) == 0 && ((size_t)o.ld * es) % 16 == 0;
}

}  // namespace

// Room for a K-major copy of an MN-major operand, in 256-byte multiples.
size_t transposed_floats(int rows, int K) {
  return ((size_t)rows * ((K + 3) & ~3) + 63) & ~(size_t)63;
}

size_t workspace_bytes(int M, int N, int K) {
  size_t best = 0;
  for (Prec p : {kFp32, kTf32, kBf16}) {
    const Plan P = plan(p, M, N, K, false);   // (K-major A may need fewer splits, never more)
    best = std::max(best, P.splits > 1 ? (size_t)P.splits * P.m_pad * P.n_pad * sizeof(float) : 0);
  }
  return best;
}

cudaError_t launch(Prec prec, int M, int N, int K, const Operand& A_in, const Operand& B_in,
                   void* C, int ldc, bool c_bf16, float beta, float* ws, size_t ws_bytes,
                   Status* st, cudaStream_t s, const Epilogue& epi) {
  if (M <= 0 || N <= 0) return cudaSuccess;
  if (epi.kind != kEpiNone && beta != 0.0f) return cudaErrorInvalidValue;
  Operand A = A_in, B = B_in;
  if (prec == kTf32 && ((A.mn_major && !tma_ok(A, 4)) || (B.mn_major && !tma_ok(B, 4)))) {
    // transpose the operands that TMA cannot read into the front of the
    // workspace, 256-byte aligned
    const size_t need = (transposed_floats(M, K) + transposed_floats(N, K)) * sizeof(float);
    if (!ws || ws_bytes < need) return cudaErrorInvalidValue;
    float* dst = ws;
    for (Operand* o : {&A, &B}) {
      const int rows = o == &A ? M : N;
      if (o->mn_major && !tma_ok(*o, 4)) {
        const int ldo = (K + 3) & ~3;
        k_transpose<<<dim3((rows + 31) / 32, (ldo + 31) / 32), dim3(32, 8), 0, s>>>(
            rows, K, static_cast<const float*>(o->ptr), o->ld, dst, ldo);
        const cudaError_t e = cudaGetLastError();
        if (e != cudaSuccess) return e;
        *o = {dst, ldo, false};
        dst += transposed_floats(rows, K);
      }
    }
    const size_t used = (size_t)(dst - ws) * sizeof(float);
    ws = dst;
    ws_bytes -= used;
  }
  Plan P = plan(prec, M, N, K, !A.mn_major);
  const size_t need = (size_t)P.splits * P.m_pad * P.n_pad * sizeof(float);
  if (P.splits > 1 && (!ws || ws_bytes < need)) {
    // no room for partials: one CTA per tile over the whole K
    P.per_split = std::max(1, P.chunks);
    P.splits = 1;
  }
  float* part = P.splits > 1 ? ws : nullptr;
  cudaError_t e = cudaSuccess;
  if (prec == kFp32) {
    const F32Args a = {M,   N,       K,        static_cast<const float*>(A.ptr), static_cast<const float*>(B.ptr),
                       A.ld, B.ld,   P.per_split * 8, static_cast<float*>(C), ldc, beta,
                       part, P.m_pad, P.n_pad, (int)epi.kind, static_cast<const float*>(epi.aux), epi.ld_aux};
    e = launch_fp32(P, a, A.mn_major, B.mn_major, s);
  } else {
    const bool tf32 = prec == kTf32;
    const int es = tf32 ? 4 : 2;
    if (!tma_ok(A, es) || !tma_ok(B, es)) return cudaErrorInvalidValue;
    const int bk = P.bk;
    CUtensorMap ma, mb;
    // K-major: inner = K, outer = rows (box: 128 B of K x tile rows);
    // MN-major: inner = rows, outer = K (box: 128 B of rows x BK).
    const bool ok_a = A.mn_major ? make_map(&ma, tf32, true, A.ptr, M, K, A.ld, bk)
                                 : make_map(&ma, tf32, false, A.ptr, K, M, A.ld, kBM);
    const bool ok_b = B.mn_major ? make_map(&mb, tf32, true, B.ptr, N, K, B.ld, bk)
                                 : make_map(&mb, tf32, false, B.ptr, K, N, B.ld, P.bn > 256 ? 64 : P.bn);
    if (!ok_a || !ok_b) return cudaErrorInvalidValue;
    const int ces = c_bf16 ? 2 : 4;
    const int vec = (reinterpret_cast<uintptr_t>(C) % 32 == 0 && ((size_t)ldc * ces) % 32 == 0)
                        ? 2
                        : ((reinterpret_cast<uintptr_t>(C) % 16 == 0 && ((size_t)ldc * ces) % 16 == 0) ? 1 : 0);
    const int ws_wide = reinterpret_cast<uintptr_t>(part) % 32 == 0 ? 1 : 0;
    const int aux_vec = epi.kind == kEpiDtanh && reinterpret_cast<uintptr_t>(epi.aux) % 32 == 0 &&
                        ((size_t)epi.ld_aux * ces) % 32 == 0;
    TcArgs a = {M,    N,    K,       P.per_split, C,  ldc,           c_bf16 ? 1 : 0,
                beta, part, P.n_pad, P.m_pad,     st, (int)epi.kind, epi.aux,
                epi.ld_aux, aux_vec, vec, ws_wide};
    if (P.rows)
      e = tf32 ? dispatch_rows<true>(B.mn_major, P, ma, mb, a, s)
               : dispatch_rows<false>(B.mn_major, P, ma, mb, a, s);
    else if (tf32)
      e = P.bn == 320   ? dispatch_major<true, 320>(A.mn_major, B.mn_major, P, ma, mb, a, s)
          : P.bn == 256 ? dispatch_major<true, 256>(A.mn_major, B.mn_major, P, ma, mb, a, s)
                        : dispatch_major<true, 128>(A.mn_major, B.mn_major, P, ma, mb, a, s);
    else
      e = P.bn == 320   ? dispatch_major<false, 320>(A.mn_major, B.mn_major, P, ma, mb, a, s)
          : P.bn == 256 ? dispatch_major<false, 256>(A.mn_major, B.mn_major, P, ma, mb, a, s)
                        : dispatch_major<false, 128>(A.mn_major, B.mn_major, P, ma, mb, a, s);
  }
  if (e != cudaSuccess || !part) return e;
  const size_t quads = (size_t)M * ((N + 3) / 4);
  return launch_pdl(k_reduce, (unsigned)((quads + kRedQuads - 1) / kRedQuads), kRedGroups * kRedQuads, 0, s, M, N,
                    P.splits, (const float*)part, P.m_pad, P.n_pad, C, ldc, c_bf16 ? 1 : 0, beta, (int)epi.kind,
                    epi.aux, epi.ld_aux);
}

namespace {

// K ranges of one item, as its product alone is split over the SMs: 128-row
// tiles of all columns, but three tiles of 128 columns where a few rows meet
// more than 256, at least four chunks a range.
void group_ranges(const GroupItem& i, int chunks, int* splits, int* per_split) {
  const int sms = sm_count_dev(), tiles = (i.M + kBM - 1) / kBM * (i.M <= kBM && i.N > 256 ? 3 : 1);
  const int want = std::max(1, std::min(tiles >= sms / 2 ? 1 : (sms + tiles - 1) / tiles, chunks / 4));
  *per_split = (chunks + want - 1) / want;
  *splits = (chunks + *per_split - 1) / *per_split;
}

// Units, K ranges and partials (floats of workspace) of a group.
void plan_group(const GroupItem* items, int n, int K, GroupArgs* g, size_t* floats) {
  g->n = n;
  g->chunks = (K + GroupTile::kBK - 1) / GroupTile::kBK;
  g->units[0] = g->units[1] = 0;
  *floats = 0;
  for (int k = 0; k < n; ++k) {
    GroupArgs::Item& it = g->it[k];
    it.M = items[k].M;
    it.N = items[k].N;
    group_ranges(items[k], g->chunks, &it.splits, &it.per_split);
    int& units = g->units[it.N <= GroupTile::kNarrow ? 1 : 0];
    it.unit0 = units;
    units += (it.M + kBM - 1) / kBM * it.splits;
    it.n_pad = (it.N + 31) / 32 * 32;
    it.C = items[k].C;
    it.ldc = items[k].ldc;
    *floats += (size_t)it.splits * it.M * it.n_pad;
  }
}

}  // namespace

size_t group_workspace_bytes(const GroupItem* items, int n, int K) {
  GroupArgs g;
  size_t floats = 0;
  plan_group(items, n, K, &g, &floats);
  return floats * sizeof(float);
}

cudaError_t launch_group(const GroupItem* items, int n, int K, float* ws, size_t ws_bytes, Status* st,
                         cudaStream_t s) {
  if (n < 1 || n > kMaxGroup || K < 1) return cudaErrorInvalidValue;
  GroupArgs g;
  GroupMaps maps;
  size_t floats = 0;
  plan_group(items, n, K, &g, &floats);
  if (!ws || reinterpret_cast<uintptr_t>(ws) % 32 != 0 || ws_bytes < floats * sizeof(float))
    return cudaErrorInvalidValue;
  g.st = st;
  unsigned blocks = 1;
  for (int k = 0; k < n; ++k) {
    const GroupItem& i = items[k];
    if (i.M < 1 || i.N < 1 || i.N > 320 || !i.A.mn_major || !i.B.mn_major || !tma_ok(i.A, 2) ||
        !tma_ok(i.B, 2) || !make_map(&maps.a[k], false, true, i.A.ptr, i.M, K, i.A.ld, GroupTile::kBK) ||
        !make_map(&maps.b[k], false, true, i.B.ptr, i.N, K, i.B.ld, GroupTile::kBK))
      return cudaErrorInvalidValue;
    g.it[k].ws = ws;
    ws += (size_t)g.it[k].splits * i.M * g.it[k].n_pad;
    blocks = std::max(blocks, (unsigned)(((size_t)i.M * ((i.N + 3) / 4) + kRedQuads - 1) / kRedQuads));
  }
  cudaError_t e = cudaFuncSetAttribute(k_gemm_group, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       GroupTile::kSmem);
  if (e != cudaSuccess) return e;
  k_gemm_group<<<std::min(sm_count_dev(), g.units[0] + g.units[1]), 192, GroupTile::kSmem, s>>>(maps, g);
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  k_reduce_group<<<dim3(blocks, n), kRedGroups * kRedQuads, 0, s>>>(g);
  return cudaGetLastError();
}

}  // namespace gemm
}  // namespace auv

// ---------------------------------------------------------------------------
// C ABI (include/auvenv.h): the learners' dense product on its own
// ---------------------------------------------------------------------------
namespace {
// The part of the workspace that holds K-major copies of MN-major tf32
// operands (used for those that TMA cannot read in place).
size_t copies_bytes(int M, int N, int K) {
  return (auv::gemm::transposed_floats(M, K) + auv::gemm::transposed_floats(N, K)) * sizeof(float);
}
}  // namespace

extern "C" size_t auv_gemm_workspace_bytes(int M, int N, int K) {
  return (M > 0 && N > 0 && K > 0) ? auv::gemm::workspace_bytes(M, N, K) + copies_bytes(M, N, K) : 0;
}

extern "C" int auv_gemm(uint32_t precision, int M, int N, int K, const void* A, int lda, int a_mn,
                        const void* B, int ldb, int b_mn, void* C, int ldc, int c_bf16, float beta,
                        void* workspace, size_t workspace_bytes, auv_status* status, void* stream) {
  if (precision > AUV_PPO_BF16 || M < 1 || N < 1 || K < 1 || !A || !B || !C || !status)
    return AUV_ERR_INVALID;
  if ((precision == AUV_PPO_FP32 && c_bf16) || lda < 1 || ldb < 1 || ldc < N ||
      lda < (a_mn ? M : K) || ldb < (b_mn ? N : K))
    return AUV_ERR_INVALID;
  static_assert(sizeof(auv::Status) == sizeof(auv_status), "status block layout");
  // an MN-major tf32 operand needs the copies' room whatever its alignment
  if (precision == AUV_PPO_TF32 && (a_mn || b_mn) && (!workspace || workspace_bytes < copies_bytes(M, N, K)))
    return AUV_ERR_SIZE;
  const auv::gemm::Operand a = {A, lda, a_mn != 0}, b = {B, ldb, b_mn != 0};
  const cudaError_t e = auv::gemm::launch(static_cast<auv::gemm::Prec>(precision), M, N, K, a, b, C,
                                          ldc, c_bf16 != 0, beta, static_cast<float*>(workspace),
                                          workspace ? workspace_bytes : 0,
                                          reinterpret_cast<auv::Status*>(status),
                                          static_cast<cudaStream_t>(stream));
  if (e == cudaErrorInvalidValue) return AUV_ERR_SIZE;
  return e == cudaSuccess ? AUV_OK : AUV_ERR_CUDA;
}
