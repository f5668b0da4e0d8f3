// Weight-streaming tcgen05 GEMM for passes of a few to 128 token rows (gemm_swap.cu).
#pragma once
#include "common.cuh"

namespace adept {

constexpr int SW_MAX_ROWS = 128;   // token rows of a problem (the MMA's N)
constexpr int SW_MAXG = 32;        // problems of a grouped launch

// Whether swap_gemm takes a problem of at most max_rows rows (its tile_stats are ignored: a caller that
// takes this path standardises by a launch of its own).
bool swap_gemm_supported(const GemmProblem& p, int max_rows);

// Enqueues the problems (rows on the device, at most max_rows[i] <= SW_MAX_ROWS each) in one
// launch.  Returns 1, or -1 when a shape is not taken (nothing launched): more than SW_MAX_ROWS
// rows, K not a multiple of 64, unaligned operands, or epilogue kinds that do not
// share a launch (only EPI_QKV and EPI_KV do).
int swap_gemm(cudaStream_t st, const GemmProblem* probs, int n_probs, const int* max_rows, unsigned* err);

cudaError_t set_wait_limit_sw(long long cycles);

}  // namespace adept
