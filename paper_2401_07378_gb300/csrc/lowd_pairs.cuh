// Kernels of the one-CTA solves of whole small pairs, d <= 8: a single pair in
// one launch and batches of pairs in one persistent launch, for a capacity of
// CAP points per side and NT threads per pair (lowd_pairs.cu and
// lowd_pairs_small.cu instantiate them).
#pragma once

#include <math_constants.h>

#include "common.cuh"
#include "cta.cuh"
#include "kernels.h"

namespace nnsemd {

// --------------------------------------------------------------------------
// a whole small pair in one launch: load, normalise, every round, the plan,
// R and the leftover mass (no host round trip between rounds)
// --------------------------------------------------------------------------

template <int D, int DP, bool L1, int CAP, int NT>
__global__ void __launch_bounds__(NT, 1) k_solve_small(SolveBufs B, const double* a, const double* b) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  using Sm = LowdSmem<D, DP, L1, CAP, NT>;
  Sm& L = *reinterpret_cast<Sm*>(smem_raw);
  CtaCore<CAP>& S = L.S;
  const int tid = threadIdx.x;
  const int m = (int)B.m, n = (int)B.n;
  if (!cta_load_sides<DP, CAP>(B.x, a, m, B.y, b, n, B.d, L.G.xs, L.G.ys, S, &B.st->err)) return;
  if (tid == 0) {
    S.mt = m;
    S.nt = n;
  }
  __syncthreads();
  cta_compact(S, L.G);  // drop zero weights
  CtaOut O{S.acc, B.plan_i, B.plan_j, B.plan_f, (long long)B.plan_cap, nullptr, nullptr, &B.st->err,
           B.fl_i, B.fl_j, B.fl_f, B.x, B.y, B.d, B.protocol, B.seed, 0};
  unsigned long long nnz = 0;
  long long rounds = 0, pe = 0;
  cta_rounds(S, L.G, B.metric, O, nnz, rounds, pe, (long long)m + n);
  __syncthreads();
  // the leftover mass; then warp 0 rounds it and warp 1 rounds R
  for (int i = tid; i < XS_LIMBS; i += blockDim.x) S.acc2()[i] = 0ULL;
  __syncthreads();
  for (int base = 0; base < S.mt; base += blockDim.x)  // whole warps (xs_add_warp)
    xs_add_warp(S.acc2(), base + tid < S.mt ? S.sres[base + tid] : 0.0);
  for (int base = 0; base < S.nt; base += blockDim.x)
    xs_add_warp(S.acc2(), base + tid < S.nt ? S.cres[base + tid] : 0.0);
  __syncthreads();
  if (tid >= 32 && tid < 64) {
    const double c = xs_round_warp(S.acc);
    if (tid == 32) B.st->cost = c;
  }
  const double left = tid < 32 ? xs_round_warp(S.acc2()) : 0.0;
  if (tid == 0) {
    B.st->leftover = left;
    B.st->nnz = nnz;
    B.st->rounds = rounds;
    B.st->pair_evals = pe;
    B.st->mt = S.mt;
    B.st->nt = S.nt;
  }
}

template <int D, int DP, bool L1, int CAP, int NT>
static int solve_small_t(const SolveBufs& B, const double* a, const double* b, cudaStream_t st) {
  const size_t smem = sizeof(LowdSmem<D, DP, L1, CAP, NT>);
  cudaError_t e =
      cudaFuncSetAttribute(k_solve_small<D, DP, L1, CAP, NT>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return -1;
  k_solve_small<D, DP, L1, CAP, NT><<<1, NT, smem, st>>>(B, a, b);
  return 0;
}

template <int CAP, int NT>
static int solve_small_d(const SolveBufs& B, const double* a, const double* b, cudaStream_t st) {
  const bool l1 = B.metric == METRIC_L1;
#define SMALL_CASE(DD, DPP) \
  case DD:                  \
    return l1 ? solve_small_t<DD, DPP, true, CAP, NT>(B, a, b, st) : solve_small_t<DD, DPP, false, CAP, NT>(B, a, b, st);
  switch (B.d) {
    SMALL_CASE(1, 2) SMALL_CASE(2, 2) SMALL_CASE(3, 4) SMALL_CASE(4, 4)
    SMALL_CASE(5, 8) SMALL_CASE(6, 8) SMALL_CASE(7, 8) SMALL_CASE(8, 8)
    default: return -1;
  }
#undef SMALL_CASE
}

// --------------------------------------------------------------------------
// batched small pairs: one persistent launch, a work queue of pairs, each
// pair solved start to finish by one CTA (Sec. III-D batch processing)
// --------------------------------------------------------------------------

template <int D, int DP, bool L1, int CAP, int NT, int PER_SM>
__global__ void __launch_bounds__(NT, PER_SM) k_batched_lowd(BatchArgs A) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  using Sm = LowdSmem<D, DP, L1, CAP, NT>;
  Sm& L = *reinterpret_cast<Sm*>(smem_raw);
  __shared__ int s_item;
  const int tid = threadIdx.x;
  for (;;) {
    if (tid == 0) s_item = (int)atomicAdd(A.queue, 1u);
    __syncthreads();
    const int item = s_item;
    __syncthreads();
    if (item >= A.num) break;
    const int pr = A.pair_ids[item];
    const int64_t xo = A.x_off[pr], yo = A.n_shared ? 0 : A.y_off[pr];
    const int m = (int)(A.x_off[pr + 1] - xo), n = A.n_shared ? A.n_shared : (int)(A.y_off[pr + 1] - yo);
    if (m > CAP || n > CAP) {  // the host routes only pairs that fit here
      if (tid == 0) atomicOr(A.err, EF_INTERNAL);
      break;
    }
    double cost = 0.0;
    long long rounds = 0, pe = 0;
    const bool ok = cta_solve_pair(L.S, L.G, L.G.xs, L.G.ys, A.x + xo * A.d, A.a + xo, m, A.y + yo * A.d, A.b + yo,
                                   n, A.d, A.metric, A.err, cost, rounds, pe, A.protocol, A.seed);
    if (tid == 0) {
      A.costs[pr] = ok ? cost : CUDART_NAN;
      if (A.rounds) A.rounds[pr] = rounds;
      if (A.pair_evals) A.pair_evals[pr] = pe;
    }
    __syncthreads();
  }
}

template <int D, int DP, bool L1, int CAP, int NT, int PER_SM>
static int batched_t(const BatchArgs& A, int grid, cudaStream_t st) {
  const size_t smem = sizeof(LowdSmem<D, DP, L1, CAP, NT>);
  auto kern = k_batched_lowd<D, DP, L1, CAP, NT, PER_SM>;
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return -1;
  kern<<<grid, NT, smem, st>>>(A);
  return 0;
}

template <int CAP, int NT, int PER_SM>
static int batched_d(const BatchArgs& A, int grid, cudaStream_t st) {
  const bool l1 = A.metric == METRIC_L1;
#define BAT_CASE(DD, DPP) \
  case DD:                \
    return l1 ? batched_t<DD, DPP, true, CAP, NT, PER_SM>(A, grid, st) : batched_t<DD, DPP, false, CAP, NT, PER_SM>(A, grid, st);
  switch (A.d) {
    BAT_CASE(1, 2) BAT_CASE(2, 2) BAT_CASE(3, 4) BAT_CASE(4, 4)
    BAT_CASE(5, 8) BAT_CASE(6, 8) BAT_CASE(7, 8) BAT_CASE(8, 8)
    default: return -1;
  }
#undef BAT_CASE
}

}  // namespace nnsemd
