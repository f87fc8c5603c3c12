// gemm64.cuh -- (min,+) products and repeated squaring on 64 x 64 tiles (gemm64.cu).
#pragma once

#include "tgemm.cuh"

namespace apsp {

// Whether an M x N product (K operand words deep) is faster on 64 x 64 tiles (gemm64.cu).
bool gemm64_pays(int64_t M, int64_t N, int64_t K);

// C = min(inf, A (x) B), or min(C, A (x) B) with p.acc, on aligned operands: the arguments of
// launch_tgemm in kModeGemm (p.arith16: packed 16-bit operands, K in words).
int launch_gemm64(bool acc, int dtype, const void *A, int64_t lda, const void *B, int64_t ldb, const TileProblem &p,
                  cudaStream_t s);

// float32, aligned n x n operands: out[i][j] = the first chunk of kArgChunkLen consecutive k that holds
// min_k A[i][k] + B[k][j], or -1 when that minimum is +infinity.
constexpr int kArgChunkLen = 64;
int launch_arg_chunks(const float *A, int64_t lda, const float *B, int64_t ldb, int64_t n, int *out, int64_t ldo,
                      cudaStream_t s);

// Largest n that squaring64 takes (its stages wait on one another inside one launch; beyond it the
// 128 x 128 tiles fill the GPU).
constexpr int64_t kSquaring64MaxN = 4096;
// Scratch of squaring64 beside the product matrix: two sets of packed operands for int32.
size_t squaring64_bytes(int64_t n, int dtype);
// a1, then D <- D (x) D, `iters` times or until nothing changes (D 16-byte aligned, ld % 4 == 0).
// words: the call's 64 zeroed words.  C: n x ldc scratch; packed: squaring64_bytes, or null.
int squaring64(void *d, int64_t n, int64_t ld, int dtype, int inf_i, float inf_f, int iters, int *words, int *C, int64_t ldc,
               void *packed, cudaStream_t s);

}  // namespace apsp
