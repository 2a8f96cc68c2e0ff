// Tensor-core GEMM of the first-level products whose tensor TMA cannot stage
// (odd row strides) or whose number format needs a split (gemm_tc.cu).
#pragma once

#include "plan.cuh"

namespace ttnn {

// C[i][j] = sum_k A(i, k) B(j, k), i < I, j < Jn, binary32 results.
// A(i, k) = A[i * lda + k] (mn = 0) or A[k * lda + i] (mn = 1); B(j, k) =
// B[j * ldb + k].  type (of both): 1 binary32, 2 bfloat16.  Every column up
// to ldc = round_up(Jn, 16) of C is written (zeros beyond Jn).
struct TcGemm {
  int64_t I = 0, Jn = 0, K = 0;
  const void* A = nullptr;
  int64_t lda = 0;
  int mn = 0;
  int type = 1;
  const void* B = nullptr;
  int64_t ldb = 0;
  float* C = nullptr;
  int64_t ldc = 0;
};

bool tcg_supported(const TcGemm& g);
// Runs the n <= 2 products in order on `st`: one launch prepares both B
// operands, then one GEMM launch (and, with a split reduction, one sum of its
// partials) each.  dry: only *need = workspace bytes.
ttnn_status launch_tcg(const TcGemm* g, int n, int sms, int* err, uint64_t wait_ns, void* ws,
                       int64_t ws_bytes, cudaStream_t st, bool dry, int64_t* need);

}  // namespace ttnn
