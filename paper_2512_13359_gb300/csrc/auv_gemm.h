// auv_gemm.h -- dense products of the learners (PPO update, SHAC window) on the
// library's own kernels: tcgen05 tensor-core GEMMs (bf16 or tf32 operands,
// fp32 accumulation in tensor memory) and an fp32 CUDA-core GEMM.
//
//   C[M][N] = beta * C + sum_k A(m, k) B(n, k)            (row-major C, ldc)
//
// Each operand is either K-major (element (r, k) at r * ld + k: a row-major
// activation or weight array whose rows are the M or N index) or MN-major
// (element (r, k) at k * ld + r: a sample-major activation read along the
// batch, as in the weight gradients, whose contraction runs over samples).
// The tensor-core path loads 128-byte-swizzled tiles with TMA; operand
// addresses must be 16-byte aligned and ld * element size a multiple of 16.
// Contractions over the batch are split over CTAs (split-K) into fp32
// partials that a second kernel adds in a fixed order, so results do not
// depend on scheduling.
#pragma once

#include <cstddef>
#include <cstdint>

#include <cuda_runtime.h>

namespace auv {
struct Status;

namespace gemm {

enum Prec { kFp32 = 0, kTf32 = 1, kBf16 = 2 };   // the AUV_PPO_* precisions

struct Operand {
  const void* ptr;   // device memory: fp32 (kFp32, kTf32) or bf16 (kBf16) elements
  int ld;            // elements between consecutive stored rows
  bool mn_major;     // false: (r, k) at r*ld + k; true: (r, k) at k*ld + r
};

// What is done to each element of the product before it is stored (beta = 0
// only): nothing, tanh (a layer's activation), or the product times tanh'
// from the activation h (row r, column c at aux[r * ld_aux + c], of C's
// type): x (1 - h^2).
enum EpiKind { kEpiNone = 0, kEpiTanh = 1, kEpiDtanh = 2 };
struct Epilogue {
  EpiKind kind = kEpiNone;
  const void* aux = nullptr;
  int ld_aux = 0;
};

// Bytes of split-K partials a product of this shape may use (0: none).
size_t workspace_bytes(int M, int N, int K);

// Enqueue C = beta C + A B^T on s.  c_bf16: C holds bf16 (else fp32).
// ws / ws_bytes: scratch for split-K partials (may be null: no split).
// st: status block for device-side wait timeouts (AUV_ERR_TIMEOUT).
// Returns cudaSuccess, cudaErrorInvalidValue for an unsupported layout
// (misaligned operand), or the launch error.
cudaError_t launch(Prec prec, int M, int N, int K, const Operand& A, const Operand& B, void* C,
                   int ldc, bool c_bf16, float beta, float* ws, size_t ws_bytes, Status* st,
                   cudaStream_t s, const Epilogue& epi = Epilogue());

// Weight gradients of one step in one launch: C_i[M][N] = sum_{k < K} A_i(m, k)
// B_i(n, k) for up to kMaxGroup items of bf16 operands stored along their
// samples (MN-major, as TMA reads them), N <= 320, fp32 C.  ws: at least
// group_workspace_bytes.
constexpr int kMaxGroup = 6;
struct GroupItem {
  int M, N;
  Operand A, B;
  float* C;
  int ldc;
};
size_t group_workspace_bytes(const GroupItem* items, int n, int K);
cudaError_t launch_group(const GroupItem* items, int n, int K, float* ws, size_t ws_bytes, Status* st,
                         cudaStream_t s);

}  // namespace gemm
}  // namespace auv
