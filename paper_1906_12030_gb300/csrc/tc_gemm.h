// Tensor-core (tcgen05 / TMEM / TMA) GEMM of the contraction programs.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "plan.h"

namespace mera {

// C[m_dst(m) + n_dst(n)] (+)= alpha * sum_k A[m, k] * B[n, k]
// A: M x K operand matrix with row pitch lda elements (one or more planes),
// B: N x K with pitch ldb.  Operands are TF32 (stored as FP32), BF16, or
// BF16 planes of a split (BF16X3 hi/lo, BF16X6 hi/mid/lo, or the S slices of
// the fixed-point split modes OZ3/OZ4), plane p at p * *_plane_bytes.  FP32
// accumulation in tensor memory.  The destination is either the caller's
// FP64 output (c_final) or the next operand buffer in the same precision
// (c_plane_elems apart for the lower planes); in the fixed-point split modes
// it is the raw hi + lo binary32 pair of the next operand, split afterwards.
struct TcGemmArgs {
  int prec = 0;
  const void* A = nullptr;
  int64_t a_plane_bytes = 0, lda = 0;
  const void* B = nullptr;
  int64_t b_plane_bytes = 0, ldb = 0;
  int64_t M = 0, N = 0, K = 0;
  bool c_final = true;
  void* C = nullptr;
  int64_t c_plane_elems = 0;
  LegMap m_dst, n_dst;
  double alpha = 1.0;
  int accumulate = 0;
  int split = 1;             // K split (from tc_split_k); > 1 needs `partial`
  int bn = 0;                // tile width 16/64/128/256; 0: chosen from N
  float* partial = nullptr;  // FP32 scratch [split][N][M] (a second, lo plane in the fixed-point split modes)
  int64_t partial_plane = 0; // fixed-point split modes: floats from the hi to the lo plane of `partial`
};

// Jobs of one mode and tile width (`bn` or, where that is 0, the same N class).
cudaError_t launch_gemm_tc(const TcGemmArgs* args, int n, cudaStream_t stream);
inline cudaError_t launch_gemm_tc(const TcGemmArgs& args, cudaStream_t stream) {
  return launch_gemm_tc(&args, 1, stream);
}

// The same product in PREC_F64 on the BF16 tensor cores, from the operands'
// digit images and row exponents (x64_split.cu).  alpha must be a power of
// two.  A64 and B64 are the binary64 operands themselves.
struct X64GemmArgs {
  const void* A = nullptr;
  const int* ea = nullptr;
  const double* A64 = nullptr;  // entry (m, k) at A64[m * lda + k]
  int64_t lda = 0;
  const void* B = nullptr;
  const int* eb = nullptr;
  const double* B64 = nullptr;
  int64_t ldb = 0;
  int64_t M = 0, N = 0, K = 0;
  double* C = nullptr;
  LegMap m_dst, n_dst;
  double alpha = 1.0;
  int accumulate = 0;
  int split = 1;             // K split (x64_split_k); > 1 needs `partial`
  float* partial = nullptr;  // hi, mid, lo and magnitude planes [split][N][M]
  int64_t partial_plane = 0; // floats from one plane to the next
  void* mask = nullptr;      // x64_mask_bytes(M, N) of scratch
};

// Jobs that all fit in one block of K per work item, or all do not
// (x64_single).
inline bool x64_single(const X64GemmArgs& a) { return x64_kc((a.K + 15) / 16, a.split) <= kX64BlockSteps; }
cudaError_t launch_gemm_x64(const X64GemmArgs* args, int n, cudaStream_t stream);

// Sets bit MERA_ENOTCONV of the device status word unless the Newton-Schulz
// state state[0] says the iteration converged (used where the host cannot
// look, e.g. inside a captured graph).
cudaError_t launch_report_notconv(const int* state, cudaStream_t stream);

// Device status word (bit MERA_ETIMEOUT set when a bounded wait gave up,
// bit MERA_ENOTCONV when a polar update inside a captured graph did not
// converge).
cudaError_t read_device_status(int* status, bool clear);

}  // namespace mera
