// Tensor-core GEMMs of the first-level products whose tensor TMA cannot stage
// (odd row strides) or whose number format needs a split: binary32 results of
// bfloat16 and binary32 tensors (gemm_tc.cu), binary64 ones (gemm_f64.cu).
#pragma once

#include "plan.cuh"

namespace ttnn {

// C[i][j] = sum_k A(i, k) B(j, k), i < I, j < Jn.
// A(i, k) = A[i * lda + k] (mn = 0) or A[k * lda + i] (mn = 1); B(j, k) =
// B[j * ldb + k].  type (of both): 0 binary64 (C too), 1 binary32, 2 bfloat16
// (C binary32).  Every column up
// to ldc = round_up(Jn, 16) of C is written (zeros beyond Jn).
struct TcGemm {
  int64_t I = 0, Jn = 0, K = 0;
  const void* A = nullptr;
  int64_t lda = 0;
  int mn = 0;
  int type = 1;
  const void* B = nullptr;
  int64_t ldb = 0;
  void* C = nullptr;
  int64_t ldc = 0;
  // B as the kernel reads it (tcg_prepare), if the caller keeps it
  const void* prep = nullptr;
};

bool tcg_supported(const TcGemm& g);
// Bytes of a prepared B operand (a multiple of 256), and its preparation (n <=
// 2 operands, 256-byte aligned) in one launch (binary64: a memset and two).
int64_t tcg_prep_bytes(const TcGemm& g);
ttnn_status tcg_prepare(const TcGemm* g, int n, void* const* dst, cudaStream_t st);
// Runs the n <= 2 products of one type in order on `st`: operands without
// `prep` are prepared first, then one GEMM launch and one sum of its pieces
// each (binary64: per 32 columns).  dry: only *need = workspace bytes.
ttnn_status launch_tcg(const TcGemm* g, int n, int sms, int* err, uint64_t wait_ns, void* ws,
                       int64_t ws_bytes, cudaStream_t st, bool dry, int64_t* need);

// The binary64 parts (gemm_f64.cu).
bool zgemm_supported(const TcGemm& g);
int64_t zgemm_prep_bytes(const TcGemm& g);
int64_t zgemm_piece_bytes(const TcGemm& g, int sms);
ttnn_status zgemm_prepare(const TcGemm* g, int n, void* const* dst, cudaStream_t st);
ttnn_status launch_zgemm(const TcGemm& g, const void* prep, void* pieces, int sms, int* err,
                         uint64_t wait_ns, cudaStream_t st);

}  // namespace ttnn
