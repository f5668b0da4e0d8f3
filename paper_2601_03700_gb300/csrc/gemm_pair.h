// Tile-paired tcgen05 GEMM (gemm_pair.cu): bf16 problems of more than 128 rows.
#pragma once
#include "common.cuh"

namespace adept {
constexpr int PG_MAXG = 32;
// True when the kernel takes the problem with at most max_rows rows.
bool pair_gemm_supported(const GemmProblem& p, int max_rows);
// Enqueues the problems as one launch; the number of kernels launched (1), or -1 when a problem is not taken or its tensor
// maps cannot be encoded (nothing launched).
int pair_gemm(cudaStream_t st, const GemmProblem* probs, int n_probs, const int* max_rows, unsigned* err);
cudaError_t set_wait_limit_pg(long long cycles);
}  // namespace adept
