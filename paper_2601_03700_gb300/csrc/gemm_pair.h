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

// What the barrier of ring stage `stage` still lacks when the pair has stopped after n0 and n1 k-blocks' copies (CTA 0's and
// CTA 1's; k-block k goes to stage k % stages), and the parity of the stage's last phase. A CTA refills a stage only once the
// k-block before it there was consumed, for which both had sent theirs: so the counts differ by at most `stages`, and at most
// the last k-block of a stage was sent by one CTA alone.
struct PgLanding {
  // NOTHING: never used. COPIES: both sent, the barrier completes by itself. ARRIVAL: CTA 1 alone; CTA 0's arrival is
  // missing (for one CTA's bytes). BYTES: CTA 0 alone, which announced both CTAs' bytes.
  enum Owe { NOTHING, COPIES, ARRIVAL, BYTES } owe;
  uint32_t parity;
};
__host__ __device__ inline PgLanding pg_landing(uint32_t n0, uint32_t n1, uint32_t stages, uint32_t stage) {
  const uint32_t n = n0 > n1 ? n0 : n1;
  if (stage >= n) return {PgLanding::NOTHING, 0};
  const uint32_t turn = (n - 1 - stage) / stages, last = turn * stages + stage;   // the stage's last k-block
  return {last >= n0 ? PgLanding::ARRIVAL : last >= n1 ? PgLanding::BYTES : PgLanding::COPIES, turn & 1u};
}
}  // namespace adept
