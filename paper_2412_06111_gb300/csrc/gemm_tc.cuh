// Tensor-core GEMMs with the large operand loaded by converter warps: the
// first-level products of tensors TMA cannot stage (odd row strides) or whose
// number format needs a split, and the large contractions of the walks.
// binary32 results in gemm_tc.cu, binary64 ones in gemm_f64.cu.
#pragma once

#include "common.cuh"

namespace ttnn {

// Columns [0, n) of a small operand, B(j, k) = p[j * sj + k * sk], or (nkr >
// 0, binary32) the Khatri-Rao product prod_f kr[f][d_f * ki[f] + j * kj[f]] over
// the digits d_f of k in the mixed radix krn (first slowest).
struct TcCols {
  const void* p = nullptr;
  int64_t sj = 0, sk = 0;
  int n = 0, nkr = 0;
  int32_t krn[4] = {0, 0, 0, 0};
  const float* kr[4] = {nullptr, nullptr, nullptr, nullptr};
  int64_t ki[4] = {0, 0, 0, 0}, kj[4] = {0, 0, 0, 0};
};

// C(i, j) = sum_k A(i, k) B(j, k), i < I, j < Jn.
// A(i, k) = A[i * lda + k] (mn = 0) or A[k * lda + i] (mn = 1).  type: 0
// binary64 (B and C too), 1 binary32, 2 bfloat16 (B too), 3 binary64 rounded
// to binary32; C of types 1 to 3 is binary32, B of 1 and 3.  C(i, j) is at
// C[i * ldc + j], with every column up to round_up(Jn, 16) <= ldc written
// (beyond Jn zeros, or NaN in rows with entries that are not finite), or with `trans` (types 1 to 3) at C[j * ldc + i].
struct TcGemm {
  int64_t I = 0, K = 0;
  int Jn = 0;
  const void* A = nullptr;
  int64_t lda = 0;
  int mn = 0, type = 1, trans = 0;
  int chain = 0;         // MMAs (of 16 k) per drain of the accumulators: 2 (types 1, 3), 8 or 16; 0: by size
  TcCols b[2];           // columns of B, one part after the other
  int nb = 1;
  // [round_up(Jn, 16)][2], for an operand of one part and two Khatri-Rao
  // factors that the data decide: the powers of two tcg_prepare takes off the
  // factors of each column, given back to C afterwards (tcg_range_kernel)
  int32_t* shift = nullptr;
  void* C = nullptr;
  int64_t ldc = 0;
  // B as the kernel reads it (tcg_prepare), if the caller keeps it
  const void* prep = nullptr;
};

constexpr int kTcgBatch = 8;   // products of one launch

bool tcg_supported(const TcGemm& g);
// Bytes of a prepared B operand (a multiple of 256) and of the pieces a launch
// needs room for, which grow with the product's columns only.
int64_t tcg_prep_bytes(const TcGemm& g);
int64_t tcg_piece_bytes(const TcGemm& g, int sms);
// Prepares n operands (256-byte aligned) of one type in one launch per
// kTcgBatch (binary64: memsets and two launches).
ttnn_status tcg_prepare(const TcGemm* g, int n, void* const* dst, cudaStream_t st);
// Runs n products with prepared operands: products of one type, majorness and
// width share a launch; each launch is followed by the sum of its pieces.
ttnn_status tcg_run(const TcGemm* g, int n, void* pieces, int sms, int* err, uint64_t wait_ns,
                    cudaStream_t st);
// Both, with the operands lacking `prep` prepared into the workspace.  dry:
// only *need = workspace bytes.
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
