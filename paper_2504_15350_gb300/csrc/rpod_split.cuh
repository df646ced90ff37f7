// FP32 products with a skinny operand (N <= 128 columns) on the bf16 tensor
// cores, every FP32 value as an exact sum of three bf16 parts.
#pragma once
#include "rpod_internal.cuh"

namespace rpod {

// Bytes of the planes of a K x N operand B.
size_t split_plane_bytes(int64_t K, int N);

// Parts of the k range that a product of an M x K and a K x N matrix is
// computed in (each an M x N partial), at most what max_elems floats hold.
int split_count(int64_t M, int64_t K, int N, size_t max_elems);
int split_sm_count();

// D[i di + c dj] = sum_k A(i, k) B[k + c ldb] for i < M, c < N <= 128, with
// A(i, k) = kc ? A[k + i lda] : A[i + k lda]; about as accurate as FP32
// fused multiply-adds.  planes: split_plane_bytes(K, N) of scratch, 16-byte
// aligned; part: part_elems floats for the partial sums (may be null); pct:
// percentage of the default split of the k range, at most 100 (the default
// is the fastest split of an idle GPU); check flags non-finite
// values of A in *status.
int split_gemm(cudaStream_t st, bool kc, int64_t M, int N, int64_t K, const float* A, int64_t lda,
               const float* B, int64_t ldb, float* D, int64_t di, int64_t dj, void* planes, float* part,
               size_t part_elems, int pct, unsigned* status, bool check);

}  // namespace rpod
