// The NNS step of a large round for d <= 3 through a spatial order, in place
// of K1's full scan (Alg. 1, Sec. III-A: the same nearest active supplier).
//
//   k_grid_bounds   once per solve: the bounding box of both initial sets;
//   k_grid_count / k_grid_scan / k_grid_scatter
//                   both active sets in the Morton order of a regular grid
//                   over that box (a counting sort; the order inside a cell
//                   does not matter);
//   k_grid_boxes    the bounding boxes of every 32 and every 1,024 suppliers;
//   k_grid_nns      a warp takes 8 consecutive consumers: it looks at the
//                   suppliers around its own place in the order first, then at
//                   every block of 32 suppliers whose box one of them reaches
//                   with its best key so far, one supplier per lane, for those
//                   consumers.
//
// Every key is key32's, and a block is left out only when a lower bound of its
// keys is strictly above the consumer's best, so the result (lowest position among
// the smallest keys) is the full scan's.  The bound: each coordinate gap
// between the consumer and the box, its square and the sum are rounded down, so
// lb <= the exact distance; a key is at least the exact distance times (1 -
// 2^-22) for d <= 3 (subtraction, square and two additions, each within 2^-24)
// as long as no square is subnormal, so lb (1 - 2^-20) > best with lb > 1e-37
// rules out key <= best.
//
// What bounds it: the latency of one block after another in each warp, hence
// few consumers to a warp (more warps).  Boxes are tested for each consumer:
// eight neighbours in the order can lie on both sides of a jump of the curve,
// and tests against the box around them opened most of the grid for those
// warps (131 us for a 65,536-point colour pair; 213 with 32 consumers a warp;
// K1 845).
#include <math_constants.h>

#include <algorithm>

#include "common.cuh"
#include "kernels.h"

namespace nnsemd {

namespace {

constexpr int GB = 32;            // suppliers per block
constexpr int GS = 1024;          // suppliers per super-block
constexpr int GRID_CELLS = 65536; // room for the cells of one side
constexpr int Q_WARPS = 8;        // warps per CTA of the query
constexpr int Q_CONS = 8;         // consumers per warp
constexpr int GRID_TELL = 256;    // a warp adds its visits to the round's total in steps of so many

// cells along one axis: 2^16 in one dimension, 2^8 in two, 2^5 in three
__host__ __device__ constexpr int grid_bits(int D) { return D == 1 ? 16 : (D == 2 ? 8 : 5); }
__host__ __device__ constexpr int grid_cells(int D) { return 1 << (grid_bits(D) * D); }

NNS_DEV float from_ordered(unsigned o) { return __uint_as_float((o & 0x80000000u) ? (o & 0x7fffffffu) : ~o); }
NNS_DEV unsigned to_ordered(float v) {
  const unsigned b = __float_as_uint(v);
  return (b & 0x80000000u) ? ~b : (b | 0x80000000u);
}

struct GridArgs {
  const float* xa;   // packed active suppliers / consumers, DP floats a point
  const float* ya;
  int mt, nt;
  unsigned* box;     // [6]: ordered minima, then ordered maxima, per axis
  int* hist;         // [2][GRID_CELLS]: points in each cell
  int* next;         // [2][GRID_CELLS]: the next sorted place of each cell
  int* start;        // [GRID_CELLS]: first sorted supplier of each cell
  float4* xs;        // sorted suppliers: coordinates, position (bits)
  float4* ys;        // sorted consumers
  float* boxes;      // [blocks][8]: minima (3, pad), maxima (3, pad); then the super-blocks
  unsigned long long* work;  // [0]: sum over the cells of suppliers x consumers; [1]: visits (k_grid_nns)
  unsigned long long* nnkey;
};

template <int D>
NNS_DEV int morton_cell(const float* v, const unsigned* box) {
  constexpr int BITS = grid_bits(D);
  constexpr float G = (float)(1 << BITS);
  unsigned code = 0;
#pragma unroll
  for (int k = 0; k < D; ++k) {
    const float lo = from_ordered(box[k]), hi = from_ordered(box[3 + k]);
    const float u = (v[k] - lo) * (G / (hi - lo));  // (an empty or overflowing range: NaN, cell 0)
    const unsigned c = (unsigned)fminf(fmaxf(u, 0.f), G - 1.f);
#pragma unroll
    for (int b = 0; b < BITS; ++b) code |= ((c >> b) & 1u) << (b * D + k);
  }
  return (int)code;
}

template <int D, int DP>
__global__ void __launch_bounds__(256) k_grid_bounds(GridArgs A) {
  unsigned lo[D], hi[D];
#pragma unroll
  for (int k = 0; k < D; ++k) { lo[k] = 0xffffffffu; hi[k] = 0u; }
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < A.mt + A.nt; i += gridDim.x * blockDim.x) {
    const float* p = i < A.mt ? A.xa + (size_t)i * DP : A.ya + (size_t)(i - A.mt) * DP;
#pragma unroll
    for (int k = 0; k < D; ++k) {
      const unsigned o = to_ordered(p[k]);
      lo[k] = min(lo[k], o);
      hi[k] = max(hi[k], o);
    }
  }
  // over the block before the six atomics
  __shared__ unsigned slo[D][8], shi[D][8];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
#pragma unroll
  for (int k = 0; k < D; ++k) {
    lo[k] = __reduce_min_sync(0xffffffffu, lo[k]);
    hi[k] = __reduce_max_sync(0xffffffffu, hi[k]);
    if (lane == 0) {
      slo[k][w] = lo[k];
      shi[k][w] = hi[k];
    }
  }
  __syncthreads();
  if (threadIdx.x < D) {
    unsigned l = 0xffffffffu, h = 0u;
    for (int u = 0; u < 8; ++u) {
      l = min(l, slo[threadIdx.x][u]);
      h = max(h, shi[threadIdx.x][u]);
    }
    atomicMin(A.box + threadIdx.x, l);
    atomicMax(A.box + 3 + threadIdx.x, h);
  }
}

// The counter of a point's cell before its point.  A warp whose points lie in
// one cell takes it at once (they would queue up at one address).  Every lane
// calls it; those without a point pass a negative counter number.
NNS_DEV int count_cell(int* counters, int c) {
  int same;
  __match_all_sync(0xffffffffu, c, &same);
  if (!same) return c >= 0 ? atomicAdd(counters + c, 1) : 0;
  const int lane = threadIdx.x & 31;
  int at = 0;
  if (c >= 0 && lane == 0) at = atomicAdd(counters + c, 32);
  return __shfl_sync(0xffffffffu, at, 0) + lane;
}

template <int D, int DP>
__global__ void __launch_bounds__(256) k_grid_count(GridArgs A) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  const bool sup = i < A.mt;
  int c = -1;
  if (i < A.mt + A.nt)
    c = (sup ? 0 : GRID_CELLS) + morton_cell<D>(sup ? A.xa + (size_t)i * DP : A.ya + (size_t)(i - A.mt) * DP, A.box);
  count_cell(A.hist, c);
}

// One block per side: exclusive scan of the cell counts (the next place of
// each cell; for the suppliers also start).  A warp owns consecutive cells,
// read and written 16 bytes a lane, all loads in flight at once.  Block 0 sums
// the per-cell products for the rule on the path.
template <int D>
__global__ void __launch_bounds__(1024) k_grid_scan(GridArgs A) {
  constexpr int IT = grid_cells(D) / (32 * 128);  // 128-cell pieces per warp
  __shared__ int wt[32];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int at = w * IT * 32 + lane;  // in vectors; piece k at + 32 k
  const int4* h4 = reinterpret_cast<const int4*>(A.hist + blockIdx.x * GRID_CELLS) + at;
  int4 v[IT];
  int sum = 0;
#pragma unroll
  for (int k = 0; k < IT; ++k) v[k] = h4[32 * k];
#pragma unroll
  for (int k = 0; k < IT; ++k) sum += v[k].x + v[k].y + v[k].z + v[k].w;
  if (blockIdx.x == 0) {
    const int4* o4 = reinterpret_cast<const int4*>(A.hist + GRID_CELLS) + at;
    unsigned long long work = 0;
#pragma unroll
    for (int k = 0; k < IT; ++k) {
      const int4 o = o4[32 * k];
      work += (unsigned long long)v[k].x * (unsigned)o.x + (unsigned long long)v[k].y * (unsigned)o.y +
              (unsigned long long)v[k].z * (unsigned)o.z + (unsigned long long)v[k].w * (unsigned)o.w;
    }
    for (int o = 16; o > 0; o >>= 1) work += __shfl_xor_sync(0xffffffffu, work, o);
    if (lane == 0 && work) atomicAdd(A.work, work);
  }
  sum = __reduce_add_sync(0xffffffffu, sum);
  if (lane == 0) wt[w] = sum;
  __syncthreads();
  int run = __reduce_add_sync(0xffffffffu, lane < w ? wt[lane] : 0);
  int4* n4 = reinterpret_cast<int4*>(A.next + blockIdx.x * GRID_CELLS) + at;
  int4* s4 = reinterpret_cast<int4*>(A.start) + at;
#pragma unroll
  for (int k = 0; k < IT; ++k) {
    const int t = v[k].x + v[k].y + v[k].z + v[k].w;
    int x = t;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int u = __shfl_up_sync(0xffffffffu, x, o);
      if (lane >= o) x += u;
    }
    int4 o;
    o.x = run + x - t;
    o.y = o.x + v[k].x;
    o.z = o.y + v[k].y;
    o.w = o.z + v[k].z;
    n4[32 * k] = o;
    if (blockIdx.x == 0) s4[32 * k] = o;
    run += __shfl_sync(0xffffffffu, x, 31);
  }
}

template <int D, int DP>
__global__ void __launch_bounds__(256) k_grid_scatter(GridArgs A) {
  if (!grid_served(A.work, A.mt, A.nt)) return;
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  const bool sup = i < A.mt, in = i < A.mt + A.nt;
  const int pos = sup ? i : (in ? i - A.mt : 0);
  const float* p = (sup ? A.xa : A.ya) + (size_t)pos * DP;
  const int at = count_cell(A.next, in ? (sup ? 0 : GRID_CELLS) + morton_cell<D>(p, A.box) : -1);
  if (in)
    (sup ? A.xs : A.ys)[at] = make_float4(p[0], D > 1 ? p[D > 1 ? 1 : 0] : 0.f, D > 2 ? p[D > 2 ? 2 : 0] : 0.f,
                                          __uint_as_float((unsigned)pos));
}

// One block of 1,024 threads per super-block, one warp per block.
template <int D>
__global__ void __launch_bounds__(GS) k_grid_boxes(GridArgs A) {
  if (!grid_served(A.work, A.mt, A.nt)) return;
  __shared__ unsigned slo[3][32], shi[3][32];
  const int i = blockIdx.x * GS + threadIdx.x, lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int nb = (A.mt + GB - 1) / GB;
  const bool in = i < A.mt;
  float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
  if (in) v = A.xs[i];
  const float c[3] = {v.x, v.y, v.z};
  const int b = blockIdx.x * (GS / GB) + w;
#pragma unroll
  for (int k = 0; k < D; ++k) {
    const unsigned o = to_ordered(c[k]);
    const unsigned lo = __reduce_min_sync(0xffffffffu, in ? o : 0xffffffffu);
    const unsigned hi = __reduce_max_sync(0xffffffffu, in ? o : 0u);
    if (lane == 0) {
      slo[k][w] = lo;
      shi[k][w] = hi;
      if (b < nb) {
        A.boxes[(size_t)b * 8 + k] = from_ordered(lo);
        A.boxes[(size_t)b * 8 + 4 + k] = from_ordered(hi);
      }
    }
  }
  __syncthreads();
  if (w == 0) {
#pragma unroll
    for (int k = 0; k < D; ++k) {
      const unsigned lo = __reduce_min_sync(0xffffffffu, slo[k][lane]);
      const unsigned hi = __reduce_max_sync(0xffffffffu, shi[k][lane]);
      if (lane == 0) {
        A.boxes[((size_t)nb + blockIdx.x) * 8 + k] = from_ordered(lo);
        A.boxes[((size_t)nb + blockIdx.x) * 8 + 4 + k] = from_ordered(hi);
      }
    }
  }
}

// Lower bound (rounded down) of the distance key between the boxes
// [alo, ahi] and [blo, bhi].
template <int D, bool L1>
NNS_DEV float box_bound(const float* alo, const float* ahi, const float* blo, const float* bhi) {
  float s = 0.f;
#pragma unroll
  for (int k = 0; k < D; ++k) {
    const float g = fmaxf(fmaxf(__fsub_rd(blo[k], ahi[k]), __fsub_rd(alo[k], bhi[k])), 0.f);
    s = L1 ? __fadd_rd(s, g) : __fmaf_rd(g, g, s);
  }
  return s;
}
// Whether every key beyond the bound lb is above best.
NNS_DEV bool beyond(float lb, float best) { return __fmul_rd(lb, 1.f - 0x1p-20f) > best && lb > 1e-37f; }

template <int D, bool L1>
__global__ void __launch_bounds__(32 * Q_WARPS) k_grid_nns(GridArgs A) {
  // (the visits grow meanwhile: a warp leaves as one)
  if (!__all_sync(0xffffffffu, grid_served(A.work, A.mt, A.nt))) return;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int q0 = (blockIdx.x * Q_WARPS + w) * Q_CONS;
  if (q0 >= A.nt) return;
  const int nq = min(Q_CONS, A.nt - q0);
  const unsigned cons = (1u << nq) - 1u;
  // lane c < nq holds consumer c, its best key and position (the other lanes
  // repeat the last consumer's coordinates and take no part)
  const float4 yq = A.ys[q0 + min(lane, nq - 1)];
  const float y[3] = {yq.x, yq.y, yq.z};
  float best = CUDART_INF_F;
  unsigned bpos = 0xffffffffu;
  const int nb = (A.mt + GB - 1) / GB, nsup = (A.mt + GS - 1) / GS;
  const float* sboxes = A.boxes + (size_t)nb * 8;
  // (consumer, block) pairs scanned so far and those added to the round's total;
  // false once the round has too many: K1 serves it
  int visits = 0, told = 0;
  auto go_on = [&]() {
    if (visits - told < GRID_TELL) return true;
    unsigned long long sum = 0;
    if (lane == 0) sum = atomicAdd(A.work + 1, (unsigned long long)(visits - told)) + (unsigned)(visits - told);
    told = visits;
    return __shfl_sync(0xffffffffu, sum, 0) <= grid_most_visits(A.mt, A.nt);
  };
  // supplier of this lane in block b (past the end: a NaN, which no key beats)
  auto fetch = [&](int b) {
    const int i = b * GB + lane;
    return i < A.mt ? A.xs[i] : make_float4(CUDART_NAN_F, CUDART_NAN_F, CUDART_NAN_F, __uint_as_float(0xffffffffu));
  };
  // the suppliers v of a block, one per lane, for the consumers of a mask
  auto scan = [&](const float4& v, unsigned mask) {
    const float x[3] = {v.x, v.y, v.z};
    const unsigned pos = __float_as_uint(v.w);
    visits += __popc(mask);
    for (; mask; mask &= mask - 1) {
      const int c = __ffs(mask) - 1;
      float yc[3] = {0.f, 0.f, 0.f};
#pragma unroll
      for (int k = 0; k < D; ++k) yc[k] = __shfl_sync(0xffffffffu, y[k], c);
      const float cb = __shfl_sync(0xffffffffu, best, c);
      const float key = L1 ? key32<METRIC_L1>(x, yc, D) : key32<METRIC_SQL2>(x, yc, D);
      if (!__any_sync(0xffffffffu, key <= cb)) continue;
      const unsigned kb = key <= cb ? __float_as_uint(key) : 0xffffffffu;  // (keys order like their bits)
      const unsigned m = __reduce_min_sync(0xffffffffu, kb);
      const unsigned mp = __reduce_min_sync(0xffffffffu, kb == m ? pos : 0xffffffffu);
      if (lane == c) {
        bpos = __uint_as_float(m) < best ? mp : min(bpos, mp);
        best = __uint_as_float(m);
      }
    }
  };
  // the blocks around this warp's place in the order
  const int c0 = min(A.start[morton_cell<D>(y, A.box)] / GB, nb - 1);
  const int home = __shfl_sync(0xffffffffu, c0, nq >> 1);
  const int f0 = max(home - 1, 0), f1 = min(home + 1, nb - 1);
  for (int b = f0; b <= f1; ++b) scan(fetch(b), cons);
  // the consumers (a mask) whose best reaches this lane's box
  auto reach = [&](const float* box) {
    const float4 l = *reinterpret_cast<const float4*>(box), h = *reinterpret_cast<const float4*>(box + 4);
    const float lo[3] = {l.x, l.y, l.z}, hi[3] = {h.x, h.y, h.z};
    unsigned m = 0;
    for (int c = 0; c < nq; ++c) {
      float yc[3] = {0.f, 0.f, 0.f};
#pragma unroll
      for (int k = 0; k < D; ++k) yc[k] = __shfl_sync(0xffffffffu, y[k], c);
      const float cb = __shfl_sync(0xffffffffu, best, c);
      m |= (beyond(box_bound<D, L1>(yc, yc, lo, hi), cb) ? 0u : 1u) << c;
    }
    return m;
  };
  // then every other block that may hold a smaller or an equal key
  for (int s0 = 0; s0 < nsup; s0 += 32) {
    const unsigned open = reach(sboxes + (size_t)min(s0 + lane, nsup - 1) * 8);
    for (unsigned sm = __ballot_sync(0xffffffffu, open && s0 + lane < nsup); sm; sm &= sm - 1) {
      const int b = (s0 + __ffs(sm) - 1) * (GS / GB) + lane;
      unsigned need = reach(A.boxes + (size_t)min(b, nb - 1) * 8);
      if (b >= nb || (b >= f0 && b <= f1)) need = 0u;
      for (unsigned bm = __ballot_sync(0xffffffffu, need); bm;) {
        // two blocks in flight
        const int l0 = __ffs(bm) - 1;
        bm &= bm - 1;
        const int l1 = bm ? __ffs(bm) - 1 : l0;
        const float4 v0 = fetch(__shfl_sync(0xffffffffu, b, l0)), v1 = fetch(__shfl_sync(0xffffffffu, b, l1));
        scan(v0, __shfl_sync(0xffffffffu, need, l0));
        if (bm) scan(v1, __shfl_sync(0xffffffffu, need, l1));
        bm &= bm - 1;
      }
      if (!go_on()) return;
    }
  }
  if (lane < nq) A.nnkey[__float_as_uint(yq.w)] = pack_key(best, bpos);
}

template <int D, int DP>
int grid_t(const SolveBufs& B, int mt, int nt, cudaStream_t st) {
  const GridBufs& G = B.grid;
  GridArgs A{B.xa[B.cur], B.ya[B.cur], mt, nt, G.box, G.hist, G.hist + 2 * GRID_CELLS, G.start, (float4*)G.xs, (float4*)G.ys, G.boxes, G.work,
             B.nnkey};
  if (cudaMemsetAsync(G.hist, 0, 2 * GRID_CELLS * sizeof(int), st) != cudaSuccess) return -1;
  if (cudaMemsetAsync(G.work, 0, 2 * sizeof(unsigned long long), st) != cudaSuccess) return -1;
  const int g = (mt + nt + 255) / 256;
  k_grid_count<D, DP><<<g, 256, 0, st>>>(A);
  k_grid_scan<D><<<2, 1024, 0, st>>>(A);
  k_grid_scatter<D, DP><<<g, 256, 0, st>>>(A);
  k_grid_boxes<D><<<(mt + GS - 1) / GS, GS, 0, st>>>(A);
  const int qb = (nt + Q_CONS * Q_WARPS - 1) / (Q_CONS * Q_WARPS);
  if (B.metric == METRIC_L1) k_grid_nns<D, true><<<qb, 32 * Q_WARPS, 0, st>>>(A);
  else k_grid_nns<D, false><<<qb, 32 * Q_WARPS, 0, st>>>(A);
  return 0;
}

}  // namespace

size_t grid_cells_bytes() { return GRID_CELLS * sizeof(int); }
size_t grid_box_floats(int64_t m) { return (size_t)((m + GB - 1) / GB + (m + GS - 1) / GS) * 8; }

int launch_grid_bounds(const SolveBufs& B, int mt, int nt, cudaStream_t st) {
  const GridBufs& G = B.grid;
  if (cudaMemsetAsync(G.box, 0xff, 3 * sizeof(unsigned), st) != cudaSuccess) return -1;
  if (cudaMemsetAsync(G.box + 3, 0, 3 * sizeof(unsigned), st) != cudaSuccess) return -1;
  GridArgs A{};
  A.xa = B.xa[B.cur], A.ya = B.ya[B.cur], A.mt = mt, A.nt = nt, A.box = G.box;
  const int g = num_sms();
  if (B.d == 1) k_grid_bounds<1, 2><<<g, 256, 0, st>>>(A);
  else if (B.d == 2) k_grid_bounds<2, 2><<<g, 256, 0, st>>>(A);
  else k_grid_bounds<3, 4><<<g, 256, 0, st>>>(A);
  return 0;
}

// Large rounds in up to three dimensions, both sides large.
bool grid_nns_wanted(const SolveBufs& B, int mt, int nt) {
  return B.grid.box && B.d <= 3 && std::min(mt, nt) >= GRID_MIN_SIDE;
}

int launch_nns_grid(const SolveBufs& B, int mt, int nt, cudaStream_t st) {
  switch (B.d) {
    case 1: return grid_t<1, 2>(B, mt, nt, st);
    case 2: return grid_t<2, 2>(B, mt, nt, st);
    case 3: return grid_t<3, 4>(B, mt, nt, st);
    default: return -1;
  }
}

}  // namespace nnsemd
