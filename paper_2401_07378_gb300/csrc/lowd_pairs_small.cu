// The one-CTA solves of lowd_pairs.cuh for pairs of at most LOWD_SMALL_CAP
// points per side.
#include "lowd_pairs.cuh"

namespace nnsemd {

int launch_solve_small_cap(const SolveBufs& B, const double* a, const double* b, cudaStream_t st) {
  return solve_small_d<LOWD_SMALL_CAP, LOWD_SMALL_THREADS>(B, a, b, st);
}

int launch_batched_lowd_small(const BatchArgs& A, int grid, cudaStream_t st) {
  return batched_d<LOWD_SMALL_CAP, LOWD_SMALL_THREADS, LOWD_SMALL_PER_SM>(A, grid, st);
}

}  // namespace nnsemd
