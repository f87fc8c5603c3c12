// gemm64.cuh -- (min,+) products and repeated squaring on 64 x 64 tiles (gemm64.cu).
#pragma once

#include "tgemm.cuh"

namespace apsp {

// Whether an M x N product (K operand words deep) takes less than percent / 100 of the time on 64 x 64
// tiles that it takes on 128 x 128 ones, by the rounds of tiles of each (gemm64.cu).
bool gemm64_pays(int64_t M, int64_t N, int64_t K, int percent = 85);

// C = min(inf, A (x) B), or min(C, A (x) B) with p.acc, on aligned operands: the arguments of
// launch_tgemm in kModeGemm (p.arith16: packed 16-bit operands, K in words).
int launch_gemm64(bool acc, int dtype, const void *A, int64_t lda, const void *B, int64_t ldb, const TileProblem &p,
                  cudaStream_t s);

// float32, aligned operands, M x K and K x N: out[i][j] = the first chunk of kArgChunkLen consecutive k that
// holds min_k A[i][k] + B[k][j], or -1 when that minimum is +infinity.
constexpr int kArgChunkLen = 64;
int launch_arg_chunks(const float *A, int64_t lda, const float *B, int64_t ldb, int64_t M, int64_t N, int64_t K, int *out,
                      int64_t ldo, cudaStream_t s);

// Repeated squaring, D <- D (x) D `iters` times or until nothing changes, up to kSquaring64MaxN vertices (the
// stages wait on one another inside one launch).  D 16-byte aligned, ld % 4 == 0; words: the call's 64
// zeroed words, words[0] the largest finite weight of an int32 matrix, words[1] zero.
constexpr int64_t kSquaring64MaxN = 4096;
// int32, sentinel above kCap16: a1, then the products on packed 16-bit pairs while the entries allow it.
// packed: squaring64_bytes.  Leaves words[kSquareUnchanged + t] and words[kSquareSkip] set for the 32-bit
// products that may be left: a loop of one launch per product skips product 0 when the latter is set,
// product t + 1 when the former is.
constexpr int kSquareUnchanged = 48, kSquareSkip = 60;
size_t squaring64_bytes(int64_t n, int dtype);
int squaring64_packed(void *d, int64_t n, int64_t ld, int inf_i, int iters, int *words, void *packed, cudaStream_t s);
// The products in 32 bits, on a normalised matrix: all of them, or those squaring64_packed left.
// C: n x ldc scratch.
int squaring64(void *d, int64_t n, int64_t ld, int dtype, int inf_i, int iters, int *words, int *C, int64_t ldc,
               cudaStream_t s);
// Whether they run there rather than in a loop of 128 x 128-tile products: whenever the 64 x 64 tiles are
// not slower on paper by more than the loop's own passes (a commit and two launches per product) cost.
// Measured, whole calls (loop / 64 x 64 tiles, us; tiles' cost on paper): float32 n = 1024 898 / 481
// (0.53), 1200 1067 / 1067 (0.90), 1300 1157 / 1014 (0.95), 1448 1249 / 1282 (1.03), 2048 3319 / 3514 (0.99),
// 2600 6289 / 6653 (1.01), 2896 9321 / 8665 (0.88), 3072 9803 / 10446 (1.01), 3700 20362 / 21460 (0.97), 4096
// 22800 / 24263 (1.00).  After 16-bit products the loop is there only for weights that outgrow them, and its launches
// cost every other call 33 us of returning at once (weights up to 100, n = 2600: 2250 -> 2282): it is taken only
// where that is little.
// int32 beyond the 16-bit products, loop / tiles: 1448 1257 / 1264, 2048 3316 / 3093, 2600 6267 / 6547, 3072
// 9750 / 10275, 4096 22733 / 23171.
constexpr int64_t kSquareLoopAfter16MinN = 2049;
inline bool squaring64_pays(int64_t n, bool after16) {
  return n <= kSquaring64MaxN && (gemm64_pays(n, n, n, 96) || (after16 && n < kSquareLoopAfter16MinN));
}

}  // namespace apsp
