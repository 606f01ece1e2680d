// The colour-transfer application of NNS-EMD (Sec. IV-D): k-means colour
// quantisation, the barycentric map of a transport plan and the recolouring
// of an image, as C-ABI entry points (declared in nnsemd.h).
//
// Every step is deterministic, so the result does not depend on the order
// in which threads run:
//   k-means   assignment: the nearest centroid by the FP32 squared-distance
//             key of the NNS operation, lowest index on ties (nearest_all);
//             update: each coordinate's sum over a cluster in an exact
//             integer accumulator, centroid = float(correctly rounded sum /
//             count); initial centroids: the points at floor((2c+1) N / 2k);
//   map       y'_j = float(S_j / W_j) with S_j = exact sum of f * x_i over the
//             flows into consumer j (FP64 products) and W_j = exact sum of f;
//   recolour  out[p] = palette[label[p]].
// Coordinates must be finite and non-negative (colours); weights of flows
// are non-negative by construction.
#include <cuda_runtime.h>
#include <math_constants.h>

#include <algorithm>
#include <mutex>
#include <vector>

#include "common.cuh"
#include "ctx.h"
#include "kernels.h"
#include "nnsemd.h"
#include "proposal.h"

using namespace nnsemd;

namespace {

#define CCK(call)                                                                                          \
  do {                                                                                                     \
    cudaError_t e_ = (call);                                                                               \
    if (e_ != cudaSuccess) return ctx_fail(ctx, NNSEMD_ERR_CUDA, "%s: %s", #call, cudaGetErrorString(e_)); \
  } while (0)

// Device scratch of one call, carved out of the context's own buffer for
// these entry points.  Each of them waits for its stream before it returns,
// so no work of an earlier call (on any stream) still uses the buffer.  A
// buffer above SCRATCH_KEEP bytes is given back at the end of its call.
constexpr size_t SCRATCH_KEEP = (size_t)64 << 20;

struct Scratch {
  nnsemd_ctx* ctx;
  size_t off = 0;
  explicit Scratch(nnsemd_ctx* c) : ctx(c) {}
  ~Scratch() {
    if (ctx->cws_bytes > SCRATCH_KEEP) {
      cudaStreamSynchronize(ctx->stream);  // (an early return may have work queued)
      cudaFree(ctx->cws);
      ctx->cws = nullptr;
      ctx->cws_bytes = 0;
    }
  }
  static size_t need(size_t bytes) { return (bytes + 255) & ~(size_t)255; }
  bool reserve(size_t bytes) {
    if (bytes <= ctx->cws_bytes) return true;
    if (ctx->cws) cudaFree(ctx->cws);
    ctx->cws = nullptr;
    ctx->cws_bytes = 0;
    if (cudaMalloc(&ctx->cws, bytes) != cudaSuccess) {
      cudaGetLastError();
      ctx->cws = nullptr;
      return false;
    }
    ctx->cws_bytes = bytes;
    return true;
  }
  template <typename T>
  T* get(size_t count) {
    T* p = reinterpret_cast<T*>(static_cast<char*>(ctx->cws) + off);
    off += need(count * sizeof(T));
    return p;
  }
};

__global__ void k_check_colours(const float* __restrict__ v, int64_t count, unsigned* err) {
  bool bad = false;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < count; i += (int64_t)gridDim.x * blockDim.x)
    bad |= !(isfinite(v[i]) && v[i] >= 0.f);
  if (__syncthreads_or(bad) && threadIdx.x == 0) atomicOr(err, EF_NONFINITE);
}

__global__ void k_init_centroids(const float* __restrict__ pts, int64_t N, int k, int d, float* __restrict__ cent,
                                 const unsigned* __restrict__ err) {
  if (*err) return;
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < k * d; i += gridDim.x * blockDim.x) {
    const int c = i / d, t = i % d;
    const int64_t p = ((2 * (int64_t)c + 1) * N) / (2 * (int64_t)k);
    cent[i] = pts[p * d + t];
  }
}

__global__ void k_km_exact_accum(const float* __restrict__ pts, int64_t N, int d, const int* __restrict__ lab,
                                 unsigned long long* __restrict__ acc, unsigned long long* __restrict__ count,
                                 const unsigned* __restrict__ err) {
  if (*err) return;
  for (int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; p < N; p += (int64_t)gridDim.x * blockDim.x) {
    const int c = lab[p];
    for (int t = 0; t < d; ++t) xs_add(acc + ((size_t)c * d + t) * XS_LIMBS, (double)pts[p * d + t]);
    if (count) atomicAdd(count + c, 1ULL);
  }
}

__global__ void k_km_exact_finish(unsigned long long* __restrict__ acc, const unsigned long long* __restrict__ count,
                                  int k, int d, float* __restrict__ cent, const unsigned* __restrict__ err) {
  if (*err) return;
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < k * d; i += gridDim.x * blockDim.x) {
    const unsigned long long n = count[i / d];
    if (n) cent[i] = __double2float_rn(__ddiv_rn(xs_round(acc + (size_t)i * XS_LIMBS), (double)n));
  }
}

// --------------------------------------------------------------------------
// k-means in low dimension: assignment and update sums in one pass
// --------------------------------------------------------------------------

// Exact sums of non-negative floats, narrow form: a float is M << (e - 1) in
// units of 2^-149 (M < 2^24, e >= 1), split into 16-bit digits.  A block
// adds them into 32-bit shared-memory limbs (at most KM_BLOCK_POINTS values,
// so no limb overflows), then its limbs into 64-bit global ones.
constexpr int KM_LIMBS = 18;
constexpr int KM_THREADS = 256;
constexpr int KM_BLOCK_POINTS = 65536;
constexpr int KM_TILE = 1024;           // centroids staged at a time
constexpr int KM_MAX_KD = 2048;         // k * d whose limbs fit a block's shared memory
constexpr int KM_MAX_COUNTS = 4096;     // k whose sizes are counted in shared memory first

NNS_DEV void km_add(unsigned* acc, float v) {
  const unsigned bits = __float_as_uint(v) & 0x7fffffffu;
  int e = (int)(bits >> 23);
  unsigned long long mant = bits & 0x7fffffu;
  if (e) mant |= 1u << 23;
  else e = 1;
  const int L = (e - 1) >> 4;
  mant <<= (e - 1) & 15;
  const unsigned c0 = (unsigned)mant & 0xffffu, c1 = (unsigned)(mant >> 16) & 0xffffu, c2 = (unsigned)(mant >> 32);
  if (c0) atomicAdd(acc + L, c0);
  if (c1) atomicAdd(acc + L + 1, c1);
  if (c2) atomicAdd(acc + L + 2, c2);
}

// The sum of KM_LIMBS global limbs, correctly rounded to double.
NNS_DEV double km_round(const unsigned long long* __restrict__ acc) {
  constexpr int W = KM_LIMBS / 2 + 2;
  unsigned long long a[W];  // 32-bit digits
  unsigned long long carry = 0;
#pragma unroll
  for (int j = 0; j < W; ++j) {
    const unsigned long long lo = 2 * j < KM_LIMBS ? acc[2 * j] : 0, hi = 2 * j + 1 < KM_LIMBS ? acc[2 * j + 1] : 0;
    const unsigned long long v = lo + (hi << 16) + carry;  // limbs < 2^47
    a[j] = v & 0xffffffffULL;
    carry = v >> 32;
  }
  int w = W - 1;
  while (w > 0 && !a[w]) --w;
  if (w < 2 && (w == 0 || a[1] < (1ULL << 21)))  // below 2^53: exact
    return __dmul_rn((double)(a[0] | (a[1] << 32)), 0x1p-149);
  const int top = 32 * w + 63 - __clzll((long long)a[w]), shift = top - 52;
  const int L = shift >> 5, r = shift & 31;
  auto digit = [&](int i) -> unsigned long long { return i < W ? a[i] : 0ULL; };
  const unsigned long long x0 = digit(L) | (digit(L + 1) << 32), x1 = digit(L + 2);
  unsigned long long mant = (r ? (x0 >> r) | (x1 << (64 - r)) : x0) & ((1ULL << 53) - 1);
  const int rp = shift - 1;
  const bool half = (a[rp >> 5] >> (rp & 31)) & 1ULL;
  bool sticky = (a[rp >> 5] & ((1ULL << (rp & 31)) - 1)) != 0;
  for (int i = 0; i < (rp >> 5); ++i) sticky |= a[i] != 0;
  if (half && (sticky || (mant & 1ULL))) ++mant;  // 2^53 is representable too
  return __dmul_rn(__dmul_rn((double)mant, __hiloint2double((shift + 1023) << 20, 0)), 0x1p-149);
}

// label[p] = the nearest centroid by key32<SQL2> (lowest index on ties),
// the cluster sizes, and with acc the exact coordinate sums of the clusters.
// A thread keeps P points (two per packed FP32x2 register) against centroids
// staged in shared memory, like K1: minima over groups of 8 centroids, and
// the winning group scanned once more for the lowest index.
//
// Bound by the FP32 pipe (2d operations per point and centroid).  The 64 x
// 64 x 32 tiles of the d > 8 search spend 32 coordinates on d = 3, and the
// sums went through global atomics on 68-limb accumulators: 262,144 points,
// k = 256: 161 + 49 us per assignment and update there.
template <int D, int DP, int P>
__global__ void __launch_bounds__(KM_THREADS) k_km_assign(const float* __restrict__ pts, int64_t N, int k,
                                                          const float* __restrict__ cent, int* __restrict__ label,
                                                          unsigned long long* __restrict__ acc,
                                                          unsigned long long* __restrict__ count,
                                                          const unsigned* __restrict__ err) {
  extern __shared__ __align__(16) unsigned char km_smem[];
  if (*err) return;
  const int tile = min(k, KM_TILE), tile_pad = (tile + 7) & ~7;
  float* cs = reinterpret_cast<float*>(km_smem);                      // [tile_pad][DP]
  unsigned* scount = reinterpret_cast<unsigned*>(cs + tile_pad * DP);  // [k]
  unsigned* sacc = scount + k;                                         // [k][D][KM_LIMBS], with acc
  const int tid = threadIdx.x;
  const bool local = k <= KM_MAX_COUNTS;  // (with acc: k <= KM_MAX_KD)
  if (local)
    for (int i = tid; i < (acc ? k * (1 + D * KM_LIMBS) : k); i += KM_THREADS) scount[i] = 0u;
  auto stage = [&](int c0) {
    const int n = min(KM_TILE, k - c0), np = (n + 7) & ~7;
    for (int i = tid; i < np * DP; i += KM_THREADS) {
      const int c = i / DP, t = i % DP;
      cs[i] = c < n ? (t < D ? cent[(size_t)(c0 + c) * D + t] : 0.f) : CUDART_NAN_F;
    }
    return np >> 3;
  };
  int ng = stage(0);
  __syncthreads();
  for (int64_t base = (int64_t)blockIdx.x * KM_THREADS * P; base < N; base += (int64_t)gridDim.x * KM_THREADS * P) {
    unsigned long long yy[P / 2][D];
#pragma unroll
    for (int c = 0; c < P / 2; ++c) {
      const int64_t pa = base + (2 * c) * KM_THREADS + tid, pb = pa + KM_THREADS;
#pragma unroll
      for (int t = 0; t < D; ++t) yy[c][t] = f2_pack(pa < N ? pts[pa * D + t] : 0.f, pb < N ? pts[pb * D + t] : 0.f);
    }
    float best[P];
    int bestg[P];
#pragma unroll
    for (int c = 0; c < P; ++c) { best[c] = CUDART_INF_F; bestg[c] = 0; }
    for (int c0 = 0; c0 < k; c0 += KM_TILE) {
      if (k > KM_TILE) {
        __syncthreads();
        ng = stage(c0);
        __syncthreads();
      }
      for (int g = 0; g < ng; ++g) {
        float gmin[P];
#pragma unroll
        for (int c = 0; c < P; ++c) gmin[c] = CUDART_INF_F;
#pragma unroll
        for (int s = 0; s < 8; s += 2) {
          float x0[DP], x1[DP];
#pragma unroll
          for (int t = 0; t < DP; ++t) {
            x0[t] = cs[(g * 8 + s) * DP + t];
            x1[t] = cs[(g * 8 + s + 1) * DP + t];
          }
#pragma unroll
          for (int c = 0; c < P / 2; ++c) {
            unsigned long long u0 = f2_sub(f2_pack(x0[0], x0[0]), yy[c][0]), u1 = f2_sub(f2_pack(x1[0], x1[0]), yy[c][0]);
            unsigned long long a0 = f2_mul(u0, u0), a1 = f2_mul(u1, u1);
#pragma unroll
            for (int t = 1; t < D; ++t) {
              u0 = f2_sub(f2_pack(x0[t], x0[t]), yy[c][t]);
              u1 = f2_sub(f2_pack(x1[t], x1[t]), yy[c][t]);
              a0 = f2_fma(u0, u0, a0);
              a1 = f2_fma(u1, u1, a1);
            }
            gmin[2 * c] = fmin3(gmin[2 * c], f2_lo(a0), f2_lo(a1));
            gmin[2 * c + 1] = fmin3(gmin[2 * c + 1], f2_hi(a0), f2_hi(a1));
          }
        }
        const int G = (c0 >> 3) + g;
#pragma unroll
        for (int c = 0; c < P; ++c)
          if (gmin[c] < best[c]) { best[c] = gmin[c]; bestg[c] = G; }
      }
    }
#pragma unroll
    for (int c = 0; c < P; ++c) {
      const int64_t p = base + c * KM_THREADS + tid;
      if (p >= N) continue;
      float yv[D];
#pragma unroll
      for (int t = 0; t < D; ++t) yv[t] = (c & 1) ? f2_hi(yy[c >> 1][t]) : f2_lo(yy[c >> 1][t]);
      int lab = bestg[c] * 8;  // (every key infinite: centroid 0)
      for (int s = 0; s < 8 && bestg[c] * 8 + s < k; ++s)
        if (key32<METRIC_SQL2>(k <= KM_TILE ? cs + (bestg[c] * 8 + s) * DP : cent + (size_t)(bestg[c] * 8 + s) * D, yv,
                               D) == best[c]) {
          lab = bestg[c] * 8 + s;
          break;
        }
      label[p] = lab;
      if (local) atomicAdd(scount + lab, 1u);
      else atomicAdd(count + lab, 1ULL);
      if (acc) {
#pragma unroll
        for (int t = 0; t < D; ++t) km_add(sacc + ((size_t)lab * D + t) * KM_LIMBS, yv[t]);
      }
    }
  }
  if (!local) return;
  __syncthreads();
  for (int i = tid; i < k; i += KM_THREADS)
    if (scount[i]) atomicAdd(count + i, (unsigned long long)scount[i]);
  if (!acc) return;
  for (int i = tid; i < k * D * KM_LIMBS; i += KM_THREADS)
    if (sacc[i]) atomicAdd(acc + i, (unsigned long long)sacc[i]);
}

// The centroids from the sums (a cluster without points keeps its own);
// sums and sizes are cleared for the next assignment.
__global__ void k_km_update(unsigned long long* __restrict__ acc, unsigned long long* __restrict__ count, int k, int d,
                            float* __restrict__ cent, const unsigned* __restrict__ err) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (*err || i >= k * d) return;
  unsigned long long* a = acc + (size_t)i * KM_LIMBS;
  const unsigned long long n = count[i / d];
  if (n) cent[i] = __double2float_rn(__ddiv_rn(km_round(a), (double)n));
#pragma unroll
  for (int L = 0; L < KM_LIMBS; ++L) a[L] = 0ULL;
}

template <int D, int DP, int P>
int km_assign_t(const float* pts, int64_t N, int k, const float* cent, int* label, unsigned long long* acc,
                unsigned long long* count, const unsigned* err, cudaStream_t st) {
  const int tile = std::min(k, KM_TILE);
  const size_t smem = sizeof(float) * ((tile + 7) & ~7) * DP +
                      (k <= KM_MAX_COUNTS ? sizeof(unsigned) * k : 0) +
                      (acc ? sizeof(unsigned) * k * (size_t)(D * KM_LIMBS) : 0);
  // The limit belongs to the kernel on the device, not to this call: lowered by
  // another thread, a launch in between would be refused, so it only ever rises.
  // (Set to the 196 KB that the largest k could take, colour transfer with k = 256
  // took 1,405 us instead of 1,390.)
  static std::mutex mu;
  static size_t limit[64] = {};
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return -1;
  {
    std::lock_guard<std::mutex> lock(mu);
    if (smem > limit[dev]) {
      if (cudaFuncSetAttribute(k_km_assign<D, DP, P>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess)
        return -1;
      limit[dev] = smem;
    }
  }
  // one pass per block where the blocks then fit two per SM; never more
  // points in a block than its 32-bit limbs can take
  const int64_t blocks = (N + KM_THREADS * P - 1) / (KM_THREADS * P);
  const int64_t floor_b = (N + KM_BLOCK_POINTS - 1) / KM_BLOCK_POINTS + 1;
  const int grid = (int)std::min<int64_t>(blocks, std::max<int64_t>(2 * num_sms(), floor_b));
  k_km_assign<D, DP, P><<<grid, KM_THREADS, smem, st>>>(pts, N, k, cent, label, acc, count, err);
  return 0;
}

int km_assign(const float* pts, int64_t N, int d, int k, const float* cent, int* label, unsigned long long* acc,
              unsigned long long* count, const unsigned* err, cudaStream_t st) {
  // four points per thread share each centroid load; two where that leaves
  // SMs without a block or the registers are short (d > 4)
  const bool four = N >= (int64_t)num_sms() * KM_THREADS * 4;
#define KM_CASE(DD, DPP, PP)                                                                              \
  case DD:                                                                                                \
    return four ? km_assign_t<DD, DPP, PP>(pts, N, k, cent, label, acc, count, err, st)                   \
                : km_assign_t<DD, DPP, 2>(pts, N, k, cent, label, acc, count, err, st);
  switch (d) {
    KM_CASE(1, 2, 4) KM_CASE(2, 2, 4) KM_CASE(3, 4, 4) KM_CASE(4, 4, 4)
    KM_CASE(5, 8, 2) KM_CASE(6, 8, 2) KM_CASE(7, 8, 2) KM_CASE(8, 8, 2)
    default: return -1;
  }
#undef KM_CASE
}

__global__ void k_count(const int* __restrict__ lab, int64_t N, long long* __restrict__ counts) {
  for (int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; p < N; p += (int64_t)gridDim.x * blockDim.x)
    atomicAdd(reinterpret_cast<unsigned long long*>(counts + lab[p]), 1ULL);
}

__global__ void k_bary_accum(const int32_t* __restrict__ pi, const int32_t* __restrict__ pj,
                             const double* __restrict__ pf, int64_t nnz, const float* __restrict__ x, int d,
                             unsigned long long* __restrict__ acc) {
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < nnz; e += (int64_t)gridDim.x * blockDim.x) {
    const int i = pi[e], j = pj[e];
    const double f = pf[e];
    unsigned long long* a = acc + (size_t)j * (d + 1) * XS_LIMBS;
    for (int t = 0; t < d; ++t) xs_add(a + (size_t)t * XS_LIMBS, __dmul_rn(f, (double)x[(size_t)i * d + t]));
    xs_add(a + (size_t)d * XS_LIMBS, f);
  }
}

// One block per consumer: a warp brings each of its d + 1 accumulators into
// shared memory (coalesced) and one lane rounds it there.  One thread per
// consumer walking 68-limb rows of global memory took 131 us for 256
// consumers.
constexpr int BARY_WARPS = 8;

__global__ void __launch_bounds__(32 * BARY_WARPS) k_bary_finish(const unsigned long long* __restrict__ acc,
                                                                 const float* __restrict__ y, int d,
                                                                 float* __restrict__ out) {
  __shared__ unsigned long long limbs[BARY_WARPS][XS_LIMBS];
  __shared__ double total;
  const int64_t j = blockIdx.x;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nw = blockDim.x >> 5;
  const unsigned long long* a = acc + (size_t)j * (d + 1) * XS_LIMBS;
  double w = 0.0;
  // warp 0 begins with the weight (accumulator d); the others take coordinates
  for (int t0 = 0; t0 <= d; t0 += nw) {
    const int t = t0 + warp == 0 ? d : t0 + warp - 1;
    double v = 0.0;
    if (t0 + warp <= d) {
      for (int L = lane; L < XS_LIMBS; L += 32) limbs[warp][L] = a[(size_t)t * XS_LIMBS + L];
      __syncwarp();
      if (lane == 0) v = xs_round(limbs[warp]);
      __syncwarp();
    }
    if (t0 == 0) {
      if (threadIdx.x == 0) total = v;
      __syncthreads();
      w = total;
    }
    if (t0 + warp <= d && t < d && lane == 0)
      out[j * d + t] = w > 0.0 ? __double2float_rn(__ddiv_rn(v, w)) : y[j * d + t];
  }
}

__global__ void k_recolour(const int* __restrict__ lab, int64_t N, const float* __restrict__ palette, int k, int d,
                           float* __restrict__ out, unsigned* err) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < N * d; i += (int64_t)gridDim.x * blockDim.x) {
    const int c = lab[i / d];
    if (c < 0 || c >= k) {
      atomicOr(err, EF_INTERNAL);
      continue;
    }
    out[i] = palette[(size_t)c * d + (i % d)];
  }
}

int grid_for(int64_t n) { return (int)std::max<int64_t>(1, std::min<int64_t>((n + 255) / 256, num_sms() * 8)); }

int read_err(nnsemd_ctx* ctx, unsigned* err_d, cudaStream_t st) {
  volatile unsigned* hv = reinterpret_cast<volatile unsigned*>(ctx->hmap) + 8;  // pinned
  CCK(cudaMemcpyAsync((void*)hv, err_d, sizeof(unsigned), cudaMemcpyDeviceToHost, st));
  CCK(cudaStreamSynchronize(st));
  const unsigned h = *hv;
  if (h & EF_NONFINITE) return ctx_fail(ctx, NNSEMD_ERR_NONFINITE, "a coordinate is negative or not finite");
  if (h) return ctx_fail(ctx, NNSEMD_ERR_INVALID_ARG, "a label is out of range");
  return NNSEMD_OK;
}

}  // namespace

extern "C" {

int nnsemd_kmeans(nnsemd_ctx* ctx, const float* pts, int64_t N, int32_t d, int32_t k, int32_t iters,
                  float* centroids_out, int32_t* labels_out, int64_t* counts_out) {
  if (!ctx) return NNSEMD_ERR_INVALID_ARG;
  ctx->err.clear();
  if (!pts || !centroids_out || !labels_out || !counts_out || N < 1 || d < 1 || k < 1 || k > N || iters < 0 ||
      N > (1LL << 30) || k > (1 << 20))
    return ctx_fail(ctx, NNSEMD_ERR_INVALID_ARG, "kmeans arguments");
  CCK(cudaSetDevice(ctx->device));
  cudaStream_t st = ctx->stream;
  Scratch S(ctx);
  // d <= 8: assignment and sums in one pass; else the tiled search of the
  // learned proposal's k-means and 68-limb accumulators in global memory
  const bool fused = d <= 8 && (int64_t)k * d <= KM_MAX_KD;
  const bool lowd = d <= 8;
  const size_t limbs = (size_t)k * d * (fused ? KM_LIMBS : XS_LIMBS);
  const size_t niota = lowd ? 0 : (size_t)std::max<int64_t>(N, k);
  if (!S.reserve(S.need(sizeof(unsigned)) + S.need(niota * sizeof(int)) +
                 S.need((lowd ? 0 : N) * sizeof(unsigned long long)) + S.need(limbs * sizeof(unsigned long long)) +
                 S.need(k * sizeof(unsigned long long))))
    return ctx_fail(ctx, NNSEMD_ERR_OOM, "kmeans scratch");
  unsigned* err = S.get<unsigned>(1);
  int* iota = S.get<int>(niota);
  unsigned long long* keys = S.get<unsigned long long>(lowd ? 0 : N);
  unsigned long long* acc = S.get<unsigned long long>(limbs);
  unsigned long long* cnt = S.get<unsigned long long>(k);
  unsigned long long* counts = reinterpret_cast<unsigned long long*>(counts_out);
  CCK(cudaMemsetAsync(err, 0, sizeof(unsigned), st));
  k_check_colours<<<grid_for(N * d), 256, 0, st>>>(pts, N * d, err);
  if (lowd) {
    // (with a coordinate refused, every kernel below leaves at once and the
    // outputs stay as they were)
    k_init_centroids<<<grid_for((int64_t)k * d), 256, 0, st>>>(pts, N, k, d, centroids_out, err);
    if (fused) CCK(cudaMemsetAsync(acc, 0, limbs * sizeof(unsigned long long), st));
    for (int it = 0; it < iters; ++it) {
      CCK(cudaMemsetAsync(cnt, 0, (size_t)k * sizeof(unsigned long long), st));
      if (km_assign(pts, N, d, k, centroids_out, labels_out, fused ? acc : nullptr, cnt, err, st))
        return ctx_fail(ctx, NNSEMD_ERR_CUDA, "assignment launch");
      if (fused) {
        k_km_update<<<(k * d + 127) / 128, 128, 0, st>>>(acc, cnt, k, d, centroids_out, err);
      } else {
        CCK(cudaMemsetAsync(acc, 0, limbs * sizeof(unsigned long long), st));
        k_km_exact_accum<<<grid_for(N), 256, 0, st>>>(pts, N, d, labels_out, acc, nullptr, err);
        k_km_exact_finish<<<grid_for((int64_t)k * d), 256, 0, st>>>(acc, cnt, k, d, centroids_out, err);
      }
    }
    CCK(cudaMemsetAsync(cnt, 0, (size_t)k * sizeof(unsigned long long), st));
    if (km_assign(pts, N, d, k, centroids_out, labels_out, nullptr, cnt, err, st))
      return ctx_fail(ctx, NNSEMD_ERR_CUDA, "assignment launch");
    CCK(cudaGetLastError());
    if (int rc = read_err(ctx, err, st)) return rc;
    CCK(cudaMemcpyAsync(counts, cnt, (size_t)k * sizeof(int64_t), cudaMemcpyDeviceToDevice, st));
    CCK(cudaStreamSynchronize(st));
    return NNSEMD_OK;
  }
  if (int rc = read_err(ctx, err, st)) return rc;
  {
    std::vector<int> h(std::max<int64_t>(N, k));
    for (size_t i = 0; i < h.size(); ++i) h[i] = (int)i;
    CCK(cudaMemcpyAsync(iota, h.data(), h.size() * sizeof(int), cudaMemcpyHostToDevice, st));
    CCK(cudaStreamSynchronize(st));
  }
  k_init_centroids<<<grid_for((int64_t)k * d), 256, 0, st>>>(pts, N, k, d, centroids_out, err);
  if (nearest_all(centroids_out, k, pts, N, d, METRIC_SQL2, iota, keys, labels_out, st))
    return ctx_fail(ctx, NNSEMD_ERR_CUDA, "assignment launch");
  for (int it = 0; it < iters; ++it) {
    CCK(cudaMemsetAsync(acc, 0, (size_t)k * d * XS_LIMBS * sizeof(unsigned long long), st));
    CCK(cudaMemsetAsync(cnt, 0, (size_t)k * sizeof(unsigned long long), st));
    k_km_exact_accum<<<grid_for(N), 256, 0, st>>>(pts, N, d, labels_out, acc, cnt, err);
    k_km_exact_finish<<<grid_for((int64_t)k * d), 256, 0, st>>>(acc, cnt, k, d, centroids_out, err);
    if (nearest_all(centroids_out, k, pts, N, d, METRIC_SQL2, iota, keys, labels_out, st))
      return ctx_fail(ctx, NNSEMD_ERR_CUDA, "assignment launch");
  }
  CCK(cudaMemsetAsync(counts_out, 0, (size_t)k * sizeof(int64_t), st));
  k_count<<<grid_for(N), 256, 0, st>>>(labels_out, N, reinterpret_cast<long long*>(counts_out));
  CCK(cudaGetLastError());
  CCK(cudaStreamSynchronize(st));
  return NNSEMD_OK;
}

int nnsemd_barycentric(nnsemd_ctx* ctx, const nnsemd_plan* plan, const float* x, int64_t m, const float* y,
                       int64_t n, int32_t d, float* y_out) {
  if (!ctx) return NNSEMD_ERR_INVALID_ARG;
  ctx->err.clear();
  if (!plan || !x || !y || !y_out || m < 1 || n < 1 || d < 1 || plan->nnz < 0 || (plan->nnz && (!plan->i || !plan->j || !plan->f)))
    return ctx_fail(ctx, NNSEMD_ERR_INVALID_ARG, "barycentric arguments");
  CCK(cudaSetDevice(ctx->device));
  cudaStream_t st = ctx->stream;
  Scratch S(ctx);
  const size_t limbs = (size_t)n * (d + 1) * XS_LIMBS;
  if (!S.reserve(S.need(sizeof(unsigned)) + S.need(limbs * sizeof(unsigned long long))))
    return ctx_fail(ctx, NNSEMD_ERR_OOM, "barycentric scratch");
  unsigned* err = S.get<unsigned>(1);
  unsigned long long* acc = S.get<unsigned long long>(limbs);
  CCK(cudaMemsetAsync(err, 0, sizeof(unsigned), st));
  k_check_colours<<<grid_for(m * d), 256, 0, st>>>(x, m * d, err);
  if (int rc = read_err(ctx, err, st)) return rc;
  CCK(cudaMemsetAsync(acc, 0, (size_t)n * (d + 1) * XS_LIMBS * sizeof(unsigned long long), st));
  if (plan->nnz) k_bary_accum<<<grid_for(plan->nnz), 256, 0, st>>>(plan->i, plan->j, plan->f, plan->nnz, x, d, acc);
  k_bary_finish<<<(unsigned)n, 32 * std::min(d + 1, BARY_WARPS), 0, st>>>(acc, y, d, y_out);
  CCK(cudaGetLastError());
  CCK(cudaStreamSynchronize(st));
  return NNSEMD_OK;
}

int nnsemd_recolour(nnsemd_ctx* ctx, const int32_t* labels, int64_t N, const float* palette, int32_t k, int32_t d,
                    float* out) {
  if (!ctx) return NNSEMD_ERR_INVALID_ARG;
  ctx->err.clear();
  if (!labels || !palette || !out || N < 1 || k < 1 || d < 1) return ctx_fail(ctx, NNSEMD_ERR_INVALID_ARG, "recolour arguments");
  CCK(cudaSetDevice(ctx->device));
  cudaStream_t st = ctx->stream;
  Scratch S(ctx);
  if (!S.reserve(S.need(sizeof(unsigned)))) return ctx_fail(ctx, NNSEMD_ERR_OOM, "recolour scratch");
  unsigned* err = S.get<unsigned>(1);
  CCK(cudaMemsetAsync(err, 0, sizeof(unsigned), st));
  k_recolour<<<grid_for(N * d), 256, 0, st>>>(labels, N, palette, k, d, out, err);
  return read_err(ctx, err, st);
}

}  // extern "C"
