// High-dimension (d > 8) NNS-EMD kernels for sm_103a, FP32 decisions.
//
// k_nns_f32_tiled -- the NNS operation (Alg. 1, Sec. III-A) for d > 8 on CUDA
//                    cores: each CTA is one 256-thread group that runs 64 x 64
//                    (consumer x supplier) tiles, staging 32 coordinates of
//                    each side at a time in shared memory; every thread
//                    accumulates 4 x 4 pairs over k in order, which reproduces
//                    the FP32 key bit for bit.  CTAs split the suppliers into
//                    chunks and merge through atomicMin on (key, position).
//                    With a consumer list it scans only those consumers (the
//                    fallback of the reduced-precision path).
// k_finish_hd      -- the tail rounds of a large solve in one CTA, coordinates
//                    read from L2 by original index.
// k_batched_hd     -- batches of pairs with up to 2,048 points per side, one
//                    pair per CTA, all rounds on chip (Sec. III-D batching).
#include <math_constants.h>

#include <atomic>

#include "common.cuh"
#include "cta.cuh"
#include "kernels.h"

namespace nnsemd {

template <bool L1>
__global__ void __launch_bounds__(TG_THREADS, 3)
    k_nns_f32_tiled(const float* __restrict__ x, const int* __restrict__ ia, int mt, int chunk,
                    const float* __restrict__ y, const int* __restrict__ ja, const int* __restrict__ cons,
                    const int* __restrict__ ncons_dev, int ncons, int d, unsigned long long* __restrict__ nnkey) {
  __shared__ TileSmem T;
  const int nc_all = ncons_dev ? *ncons_dev : ncons;
  const int c0 = blockIdx.x * TG_M;
  if (c0 >= nc_all) return;
  const int p0 = blockIdx.y * chunk;
  const int p1 = min(p0 + chunk, mt);
  if (p0 >= p1) return;
  unsigned long long out[4];
  group_nns_tile<L1, true>(x, ia, p0, p1, y, ja, cons, c0, min(TG_M, nc_all - c0), d, T, threadIdx.x, 0, out);
  const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
  if (tx == 0) {
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int lq = c0 + ty * 4 + i;
      if (lq < nc_all) atomicMin(nnkey + (cons ? cons[lq] : lq), out[i]);
    }
  }
}

int launch_nns_f32(const SolveBufs& B, int mt, int ncons, const int* cons, const int* ncons_dev, cudaStream_t st) {
  const int gx = (ncons + TG_M - 1) / TG_M;
  const int target = num_sms() * 6;
  int gy = (target + gx - 1) / gx;
  const int tiles = (mt + TG_N - 1) / TG_N;
  if (gy > tiles) gy = tiles;
  const int chunk = ((tiles + gy - 1) / gy) * TG_N;
  gy = (mt + chunk - 1) / chunk;
  dim3 grid(gx, gy);
  const int cur = B.cur;
  if (B.metric == METRIC_L1)
    k_nns_f32_tiled<true><<<grid, TG_THREADS, 0, st>>>(B.x, B.ia[cur], mt, chunk, B.y, B.ja[cur], cons, ncons_dev,
                                                      ncons, B.d, B.nnkey);
  else
    k_nns_f32_tiled<false><<<grid, TG_THREADS, 0, st>>>(B.x, B.ia[cur], mt, chunk, B.y, B.ja[cur], cons, ncons_dev,
                                                       ncons, B.d, B.nnkey);
  return 0;
}

// --------------------------------------------------------------------------
// one-CTA solver, d > 8
// --------------------------------------------------------------------------

template <bool L1>
struct HighdSmem {
  CtaCore<FIN_MAX_HD> S;
  GeoGlobal<L1, FIN_MAX_HD> G;
};

template <bool L1>
__global__ void __launch_bounds__(FIN_THREADS, 1) k_finish_hd(SolveBufs B, long long round_limit) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  HighdSmem<L1>& H = *reinterpret_cast<HighdSmem<L1>*>(smem_raw);
  CtaCore<FIN_MAX_HD>& S = H.S;
  const int tid = threadIdx.x;
  const int mt = B.st->mt, nt = B.st->nt;
  if (mt > FIN_MAX_HD || nt > FIN_MAX_HD) {
    if (tid == 0) atomicOr(&B.st->err, EF_INTERNAL);
    return;
  }
  if (tid == 0) {
    H.G.begin(B.x, B.y, (int)B.m, (int)B.n, B.d, nullptr, 0);
    S.mt = mt;
    S.nt = nt;
  }
  for (int p = tid; p < mt; p += blockDim.x) {
    S.iidx[p] = B.ia[B.cur][p];
    S.sres[p] = B.s[S.iidx[p]];
  }
  for (int q = tid; q < nt; q += blockDim.x) {
    S.jidx[q] = B.ja[B.cur][q];
    S.cres[q] = B.c[S.jidx[q]];
  }
  __syncthreads();
  CtaOut O{nullptr, nullptr, nullptr, nullptr, 0, B.s, B.c, &B.st->err,
           B.fl_i, B.fl_j, B.fl_f, B.x, B.y, B.d, B.protocol, B.seed, B.round0};
  unsigned long long nnz = B.st->nnz;
  long long rounds = B.st->rounds, pe = B.st->pair_evals;
  cta_rounds(S, H.G, B.metric, O, nnz, rounds, pe, round_limit);
  if (tid == 0) {
    B.st->nnz = nnz;
    B.st->rounds = rounds;
    B.st->pair_evals = pe;
    B.st->mt = S.mt;
    B.st->nt = S.nt;
  }
}

template <bool L1>
static int finish_hd_t(const SolveBufs& B, long long round_limit, cudaStream_t st) {
  const size_t smem = sizeof(HighdSmem<L1>);
  cudaError_t e = cudaFuncSetAttribute(k_finish_hd<L1>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return -1;
  k_finish_hd<L1><<<1, FIN_THREADS, smem, st>>>(B, round_limit);
  return 0;
}

int launch_finish_hd(const SolveBufs& B, int64_t round_limit, cudaStream_t st) {
  return B.metric == METRIC_L1 ? finish_hd_t<true>(B, round_limit, st) : finish_hd_t<false>(B, round_limit, st);
}

// --------------------------------------------------------------------------
// the tail on a thread-block cluster, from a key matrix
// --------------------------------------------------------------------------

// The FP32 keys of every active supplier (row) and consumer, one 64 x 64 tile
// per CTA.
template <bool L1>
__global__ void __launch_bounds__(TG_THREADS, 3)
    k_tail_keys(const float* __restrict__ x, const int* __restrict__ ia, int mt, const float* __restrict__ y,
                const int* __restrict__ ja, int nt, int d, float* __restrict__ kmat, int ld) {
  __shared__ TileSmem T;
  const int c0 = blockIdx.x * TG_M, p0 = blockIdx.y * TG_N;
  const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
  group_tiles<L1, true>(x, ia, p0, min(p0 + TG_N, mt), y, ja, nullptr, c0, min(TG_M, nt - c0), d, T, threadIdx.x, 0,
                        [&](int pt, const unsigned long long (&acc)[2][4]) {
                          const int q = c0 + ty * 4;  // four consecutive consumers: one 16-byte store
                          if (q >= nt) return;
#pragma unroll
                          for (int j = 0; j < 4; ++j) {
                            const int p = pt + tx * 4 + j;
                            if (p < mt)
                              *reinterpret_cast<ulonglong2*>(kmat + (size_t)p * ld + q) =
                                  make_ulonglong2(acc[0][j], acc[1][j]);
                          }
                        });
}

constexpr int FIN_HD_CL_THREADS = 512;
constexpr int FIN_HD_CL = 16;  // preferred cluster size (8 where 16 cannot be co-scheduled)

struct MatClusterSmem {
  CtaCore<FIN_MAX_HD> S;
  GeoMatCluster<FIN_MAX_HD, FIN_HD_CL_THREADS> G;
};

// Every remaining round of a d > 8 solve, both active sets at most FIN_MAX_HD
// points: the scheme of k_finish_cl on the key matrix of k_tail_keys.  One CTA
// recomputing the distances of its rounds took 335 us for a 300 x 700 pair at
// d = 128 and could only take over below 2^23 coordinate products a round;
// the multi-CTA rounds before that cost 40 us and more each.
__global__ void __launch_bounds__(FIN_HD_CL_THREADS, 1) k_finish_hd_cl(SolveBufs B, int ld, long long round_limit) {
  namespace cg = cooperative_groups;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  MatClusterSmem& M = *reinterpret_cast<MatClusterSmem*>(smem_raw);
  CtaCore<FIN_MAX_HD>& S = M.S;
  cg::cluster_group cl = cg::this_cluster();
  const bool leader = cl.block_rank() == 0;
  const int tid = threadIdx.x;
  const int mt = B.st->mt, nt = B.st->nt;
  if (mt > FIN_MAX_HD || nt > FIN_MAX_HD || cl.num_blocks() < 8) {  // the same decision in every CTA
    if (tid == 0 && leader) atomicOr(&B.st->err, EF_INTERNAL);
    return;
  }
  for (int p = tid; p < mt; p += FIN_HD_CL_THREADS) {
    M.G.row[p] = p;
    S.iidx[p] = B.ia[B.cur][p];
    S.sres[p] = B.s[S.iidx[p]];
  }
  for (int q = tid; q < nt; q += FIN_HD_CL_THREADS) {
    M.G.col[q] = q;
    S.jidx[q] = B.ja[B.cur][q];
    S.cres[q] = B.c[S.jidx[q]];
  }
  if (tid == 0) {
    M.G.kmat = B.kmat;
    M.G.kld = ld;
    S.mt = mt;
    S.nt = nt;
  }
  M.G.init();
  // the running totals are read before the barrier: the leader writes them back
  // after its rounds, and a solve whose rounds are all local (few points) has
  // no other barrier between that and a late CTA's read
  unsigned long long nnz = B.st->nnz;
  long long rounds = B.st->rounds, pe = B.st->pair_evals;
  // every CTA of the cluster is running before any writes a peer's memory
  cl.sync();
  CtaOut O{nullptr, nullptr, nullptr, nullptr, 0, nullptr, nullptr, &B.st->err,
           nullptr, nullptr, nullptr, B.x, B.y, B.d, B.protocol, B.seed, B.round0, 1};
  if (leader)
    O = CtaOut{nullptr, nullptr, nullptr, nullptr, 0, B.s, B.c, &B.st->err,
               B.fl_i, B.fl_j, B.fl_f, B.x, B.y, B.d, B.protocol, B.seed, B.round0, 0};
  cta_rounds(S, M.G, B.metric, O, nnz, rounds, pe, round_limit);
  if (tid == 0 && leader) {
    B.st->nnz = nnz;
    B.st->rounds = rounds;
    B.st->pair_evals = pe;
    B.st->mt = S.mt;
    B.st->nt = S.nt;
  }
  // no CTA leaves while a peer may still address its shared memory
  cl.sync();
}

static_assert(sizeof(MatClusterSmem) <= 227 * 1024, "cluster tail state exceeds shared memory");

static void finish_hd_cl_config(cudaLaunchConfig_t& cfg, cudaLaunchAttribute* at, int cs) {
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = cs;
  at[0].val.clusterDim.y = 1;
  at[0].val.clusterDim.z = 1;
  cfg.gridDim = dim3(cs);
  cfg.blockDim = dim3(FIN_HD_CL_THREADS);
  cfg.dynamicSmemBytes = sizeof(MatClusterSmem);
  cfg.attrs = at;
  cfg.numAttrs = 1;
}

// Cluster size usable for k_finish_hd_cl on the current device (looked up
// once per device): the preferred size, 8, or 0.
static int finish_hd_cl_size() {
  static std::atomic<int> cache[64];
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return 0;
  const int c = cache[dev].load();
  if (c) return c > 0 ? c : 0;
  int found = -1;
  if (cudaFuncSetAttribute(k_finish_hd_cl, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(MatClusterSmem)) ==
          cudaSuccess &&
      cudaFuncSetAttribute(k_finish_hd_cl, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) == cudaSuccess) {
    for (int cs : {FIN_HD_CL, 8}) {
      cudaLaunchConfig_t cfg = {};
      cudaLaunchAttribute at[1];
      finish_hd_cl_config(cfg, at, cs);
      int n = 0;
      if (cudaOccupancyMaxActiveClusters(&n, k_finish_hd_cl, &cfg) == cudaSuccess && n > 0) {
        found = cs;
        break;
      }
    }
  }
  cudaGetLastError();  // a refused size is an answer, not an error of the solve
  cache[dev].store(found);
  return found > 0 ? found : 0;
}

bool finish_hd_cluster_ready(const SolveBufs& B) { return B.kmat != nullptr && finish_hd_cl_size() > 0; }

int launch_finish_hd_cluster(const SolveBufs& B, int mt, int nt, int64_t round_limit, cudaStream_t st) {
  const int cs = finish_hd_cl_size();
  if (!cs || !B.kmat) return -1;
  const int ld = (int)kmat_ld(nt), cur = B.cur;
  const dim3 grid((nt + TG_M - 1) / TG_M, (mt + TG_N - 1) / TG_N);
  if (B.metric == METRIC_L1)
    k_tail_keys<true><<<grid, TG_THREADS, 0, st>>>(B.x, B.ia[cur], mt, B.y, B.ja[cur], nt, B.d, B.kmat, ld);
  else
    k_tail_keys<false><<<grid, TG_THREADS, 0, st>>>(B.x, B.ia[cur], mt, B.y, B.ja[cur], nt, B.d, B.kmat, ld);
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute at[1];
  finish_hd_cl_config(cfg, at, cs);
  cfg.stream = st;
  return cudaLaunchKernelEx(&cfg, k_finish_hd_cl, B, ld, (long long)round_limit) == cudaSuccess ? 0 : -1;
}

template <bool L1>
__global__ void __launch_bounds__(FIN_THREADS, 1) k_batched_hd(BatchArgs A) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  HighdSmem<L1>& H = *reinterpret_cast<HighdSmem<L1>*>(smem_raw);
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
    if (tid == 0)
      H.G.begin(A.x + xo * A.d, A.y + yo * A.d, m, n, A.d, A.kmat ? A.kmat + blockIdx.x * A.kcap : nullptr, A.kcap);
    __syncthreads();
    double cost = 0.0;
    long long rounds = 0, pe = 0;
    const size_t fo = (size_t)blockIdx.x * A.fl_cap;
    const bool ok = cta_solve_pair(H.S, H.G, nullptr, nullptr, A.x + xo * A.d, A.a + xo, m, A.y + yo * A.d,
                                   A.b + yo, n, A.d, A.metric, A.err, cost, rounds, pe, A.protocol, A.seed,
                                   A.fl_i ? A.fl_i + fo : nullptr, A.fl_i ? A.fl_j + fo : nullptr,
                                   A.fl_i ? A.fl_f + fo : nullptr, A.fl_cap);
    if (tid == 0) {
      A.costs[pr] = ok ? cost : CUDART_NAN;
      if (A.rounds) A.rounds[pr] = rounds;
      if (A.pair_evals) A.pair_evals[pr] = pe;
      if (A.searches) atomicAdd(A.searches, H.G.searches);
    }
    __syncthreads();
  }
}

template <bool L1>
static int batched_hd_t(const BatchArgs& A, int grid, cudaStream_t st) {
  const size_t smem = sizeof(HighdSmem<L1>);
  cudaError_t e = cudaFuncSetAttribute(k_batched_hd<L1>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return -1;
  k_batched_hd<L1><<<grid, FIN_THREADS, smem, st>>>(A);
  return 0;
}

int launch_batched_hd(const BatchArgs& A, int grid, cudaStream_t st) {
  return A.metric == METRIC_L1 ? batched_hd_t<true>(A, grid, st) : batched_hd_t<false>(A, grid, st);
}

// Pairs of at most HD_SMALL_CAP points per side: a 256-thread CTA each, four
// resident per SM, so that four pairs' latency-bound round loops overlap on
// every SM (a 1,024-thread CTA spends most of a small pair's round in its
// barriers: its NNS tile has one 256-thread group's worth of consumers).
template <bool L1>
struct HighdSmallSmem {
  CtaCore<HD_SMALL_CAP> S;
  GeoGlobal<L1, HD_SMALL_CAP, HD_SMALL_THREADS> G;
};

template <bool L1>
__global__ void __launch_bounds__(HD_SMALL_THREADS, 4) k_batched_hd_small(BatchArgs A) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  HighdSmallSmem<L1>& H = *reinterpret_cast<HighdSmallSmem<L1>*>(smem_raw);
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
    if (m > HD_SMALL_CAP || n > HD_SMALL_CAP) {  // the host routes only small pairs here
      if (tid == 0) atomicOr(A.err, EF_INTERNAL);
      break;
    }
    if (tid == 0)
      H.G.begin(A.x + xo * A.d, A.y + yo * A.d, m, n, A.d, A.kmat ? A.kmat + blockIdx.x * A.kcap : nullptr, A.kcap);
    __syncthreads();
    double cost = 0.0;
    long long rounds = 0, pe = 0;
    const size_t fo = (size_t)blockIdx.x * A.fl_cap;
    const bool ok = cta_solve_pair(H.S, H.G, nullptr, nullptr, A.x + xo * A.d, A.a + xo, m, A.y + yo * A.d,
                                   A.b + yo, n, A.d, A.metric, A.err, cost, rounds, pe, A.protocol, A.seed,
                                   A.fl_i ? A.fl_i + fo : nullptr, A.fl_i ? A.fl_j + fo : nullptr,
                                   A.fl_i ? A.fl_f + fo : nullptr, A.fl_cap);
    if (tid == 0) {
      A.costs[pr] = ok ? cost : CUDART_NAN;
      if (A.rounds) A.rounds[pr] = rounds;
      if (A.pair_evals) A.pair_evals[pr] = pe;
      if (A.searches) atomicAdd(A.searches, H.G.searches);
    }
    __syncthreads();
  }
}

template <bool L1>
static int batched_hd_small_t(const BatchArgs& A, int grid, cudaStream_t st) {
  const size_t smem = sizeof(HighdSmallSmem<L1>);
  cudaError_t e =
      cudaFuncSetAttribute(k_batched_hd_small<L1>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return -1;
  k_batched_hd_small<L1><<<grid, HD_SMALL_THREADS, smem, st>>>(A);
  return 0;
}

int launch_batched_hd_small(const BatchArgs& A, int grid, cudaStream_t st) {
  return A.metric == METRIC_L1 ? batched_hd_small_t<true>(A, grid, st) : batched_hd_small_t<false>(A, grid, st);
}

}  // namespace nnsemd
