// The one-CTA NNS-EMD solver: every step of a round of Alg. 1 (Sec. III-A)
// for active sets of at most CAP points per side, with all per-point state in
// one CTA's shared memory.  Used for the tail rounds of a large solve, for
// batches of small pairs (one pair per CTA) and by the allocation-free entry
// point.
//
// The coordinates are a policy:
//   GeoSmem   (d <= 8)  coordinates of the active points live in shared
//                       memory and move with the compaction;
//   GeoGlobal (d > 8)   coordinates stay in global memory (L2) and are read
//                       by original index; the NNS step runs 64 x 64 tiles
//                       staged in shared memory by 256-thread groups,
//                       or, for batched pairs, read from a matrix of the
//                       pair's keys computed once;
//   GeoMatCluster (d > 8) the tail of a large solve on a cluster, from a key
//                       matrix;
//   GeoSmemCluster      GeoSmem on every CTA of a thread-block cluster: each
//                       CTA holds the whole state, finds the nearest
//                       supplier of its slice of the consumers and sends the
//                       keys to every CTA through distributed shared memory;
//                       the rest of the round runs, identically, in every
//                       CTA (one of them writes the results).
// Grouping, greedy order, flow and compaction are the same for all.
#pragma once

#include <cooperative_groups.h>
#include <math_constants.h>

#include "common.cuh"
#include "kernels.h"

namespace nnsemd {

constexpr int FIN_THREADS = 1024;

// Exclusive prefix sum over the block; `total` receives the block sum.
NNS_DEV int block_scan_excl(int v, int* wt, int& total) {
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  int x = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    int t = __shfl_up_sync(0xffffffffu, x, o);
    if (lane >= o) x += t;
  }
  if (lane == 31) wt[w] = x;
  __syncthreads();
  if (w == 0) {
    const int nw = blockDim.x >> 5;
    int t = lane < nw ? wt[lane] : 0;
    int y = t;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      int u = __shfl_up_sync(0xffffffffu, y, o);
      if (lane >= o) y += u;
    }
    wt[lane] = y - t;
    if (lane == 31) wt[32] = y;
  }
  __syncthreads();
  total = wt[32];
  const int r = wt[w] + x - v;
  __syncthreads();
  return r;
}

// Per-point state of a pair solved in one CTA (no coordinates).
template <int CAP>
struct CtaCore {
  double sres[CAP];
  double cres[CAP];
  int iidx[CAP];
  int jidx[CAP];
  unsigned long long nnk[CAP];
  unsigned long long mem[CAP];
  unsigned long long mem2[CAP];
  int cnt[CAP + 1];
  int off[CAP + 1];
  unsigned long long acc[XS_LIMBS];
  int wt[33];
  int mt, nt;
  unsigned nflow;
  union {
    double total[2];  // the sides' weight totals (while a pair loads)
    struct {          // running totals handed back by team_rounds
      unsigned long long w_nnz;
      long long w_rounds, w_pe;
    };
  };
  // a second exact sum beside acc, while no round runs
  static_assert(CAP >= XS_LIMBS, "the second accumulator lies in mem2");
  NNS_DEV unsigned long long* acc2() { return mem2; }
};

struct CtaOut {
  unsigned long long* acc;       // exact accumulator for R (shared, nullable)
  int32_t* plan_i;               // plan (nullable)
  int32_t* plan_j;
  double* plan_f;
  long long plan_cap;
  double* s_glob;                // residual write-back by original index (nullable)
  double* c_glob;
  unsigned* err;
  // Deferred costing (fl_i nullable): every flow's original (i, j, f) is
  // recorded in fl_* (global, slot = running flow count) during the rounds,
  // and the cost terms and plan entries of all of them are computed in one
  // pass after the last round from the original coordinates x, y (row
  // stride d).  The FP64 distance chain then costs its latency once per
  // solve instead of once per round.
  int32_t* fl_i;
  int32_t* fl_j;
  double* fl_f;
  const float* x;
  const float* y;
  int d;
  // serving order: greedy (0) or random (1) with the seed and the global
  // index of the loop's first round (the random protocol's keys)
  int protocol;
  unsigned long long seed;
  long long round_base;
  // nonzero: run the rounds without writing any flow, plan entry, cost term
  // or residual out (a CTA of a cluster whose results another CTA writes)
  int quiet;
  long long fl_cap;  // > 0: capacity of fl_* (a flow beyond it raises EF_CAPACITY)
};

// --------------------------------------------------------------------------
// coordinate policies
// --------------------------------------------------------------------------

template <int D, int DP, bool L1, int CAP, int NT = FIN_THREADS>
struct GeoSmem {
  static constexpr int kDP = DP;
  static constexpr int kD = D;
  static constexpr int kThreads = NT;  // threads of the CTA
  float xs[CAP * DP];
  float ys[CAP * DP];
  struct PX { float v[DP]; };

  // FP32 decision key of supplier coordinates xv against consumer
  // coordinates yv (the metric of this policy)
  static NNS_DEV float key_pair(const float* xv, const float* yv) {
    return L1 ? key32<METRIC_L1>(xv, yv, D) : key32<METRIC_SQL2>(xv, yv, D);
  }

  NNS_DEV void load_x(int p, PX& r) const {
#pragma unroll
    for (int k = 0; k < DP; ++k) r.v[k] = xs[p * DP + k];
  }
  NNS_DEV void store_x(int p, const PX& r) {
#pragma unroll
    for (int k = 0; k < DP; ++k) xs[p * DP + k] = r.v[k];
  }
  NNS_DEV void load_y(int q, PX& r) const {
#pragma unroll
    for (int k = 0; k < DP; ++k) r.v[k] = ys[q * DP + k];
  }
  NNS_DEV void store_y(int q, const PX& r) {
#pragma unroll
    for (int k = 0; k < DP; ++k) ys[q * DP + k] = r.v[k];
  }
  template <int C>
  NNS_DEV double dist64(const CtaCore<C>& S, int p, int q, int metric) const {
    return cost_dist64(xs + p * DP, ys + q * DP, D, metric);
  }
  // keys of supplier p against two consumers: coordinates ya, yb, also
  // packed in y2
  NNS_DEV unsigned long long key_two(int p, const unsigned long long* y2, const float* ya, const float* yb) const {
    float xv[D];
#pragma unroll
    for (int k = 0; k < D; ++k) xv[k] = xs[p * DP + k];
    if (L1) return f2_pack(key_pair(xv, ya), key_pair(xv, yb));
    unsigned long long t = f2_sub(f2_pack(xv[0], xv[0]), y2[0]);
    unsigned long long acc = f2_mul(t, t);
#pragma unroll
    for (int k = 1; k < D; ++k) {
      t = f2_sub(f2_pack(xv[k], xv[k]), y2[k]);
      acc = f2_fma(t, t, acc);
    }
    return acc;
  }
  // This lane's consumers qa, qb (those below n; others read as 0) against
  // the suppliers [s0, s1), s0 < s1: the packed (key, first position) of each.
  // All lanes read the same supplier (a broadcast).  Four keys at a time go
  // through minima, and the winning four are looked at once more for the
  // position: the chain of a compare and two selects per supplier, with the
  // load before it, took 60 cycles a supplier for one resident pair.
  NNS_DEV void scan_chunk(int qa, int qb, int n, int s0, int s1, unsigned long long& ka, unsigned long long& kb) const {
    float ya[D], yb[D];
    unsigned long long y2[D];
#pragma unroll
    for (int k = 0; k < D; ++k) {
      ya[k] = qa < n ? ys[qa * DP + k] : 0.f;
      yb[k] = qb < n ? ys[qb * DP + k] : 0.f;
      y2[k] = f2_pack(ya[k], yb[k]);
    }
    float ba = CUDART_INF_F, bb = CUDART_INF_F;
    int pa = s0, pb = s0, p = s0;
    for (; p + 4 <= s1; p += 4) {
      unsigned long long v[4];
#pragma unroll
      for (int e = 0; e < 4; ++e) v[e] = key_two(p + e, y2, ya, yb);
      const float ma = fmin3(fminf(f2_lo(v[0]), f2_lo(v[1])), f2_lo(v[2]), f2_lo(v[3]));
      const float mb = fmin3(fminf(f2_hi(v[0]), f2_hi(v[1])), f2_hi(v[2]), f2_hi(v[3]));
      if (ma < ba) { ba = ma; pa = p; }
      if (mb < bb) { bb = mb; pb = p; }
    }
    for (; p < s1; ++p) {
      const unsigned long long v = key_two(p, y2, ya, yb);
      if (f2_lo(v) < ba) { ba = f2_lo(v); pa = p; }
      if (f2_hi(v) < bb) { bb = f2_hi(v); pb = p; }
    }
    auto first = [&](int g, float best, const float* yv) {
      int r = g;
#pragma unroll
      for (int e = 3; e >= 0; --e)
        if (g + e < s1 && key_pair(xs + (g + e) * DP, yv) == best) r = g + e;
      return r;
    };
    ka = pack_key(ba, (unsigned)first(pa, ba, ya));
    kb = pack_key(bb, (unsigned)first(pb, bb, yb));
  }
  // One consumer by a warp, a supplier per lane, for rounds of few consumers
  // (chunks would meet in the same atomics: 1,000 x 2 points 2,735 us in chunks,
  // 1,570 this way).
  __device__ __noinline__ void scan_one(unsigned long long* nnk, int q, int mt) const {
    const int lane = threadIdx.x & 31;
    float yv[D];
#pragma unroll
    for (int k = 0; k < D; ++k) yv[k] = ys[q * DP + k];
    unsigned best = 0xffffffffu;
    int bp = 0;
#pragma unroll 4
    for (int p = lane; p < mt; p += 32) {
      const unsigned v = __float_as_uint(key_pair(xs + p * DP, yv));  // (keys order like their bits)
      if (v < best) { best = v; bp = p; }
    }
    const unsigned m = __reduce_min_sync(0xffffffffu, best);
    const unsigned mp = __reduce_min_sync(0xffffffffu, best == m ? (unsigned)bp : 0xffffffffu);
    if (lane == 0) nnk[q] = ((unsigned long long)m << 32) | mp;
  }
  // S.nnk[q] = (key32 bits << 32 | p) of the nearest active supplier;
  // returns S.nnk (every NNS policy returns the array holding the keys).  A
  // warp takes 64 consumers and a contiguous chunk of the suppliers; chunks
  // merge by atomicMin on (key, position).
  template <int C>
  NNS_DEV const unsigned long long* nns(CtaCore<C>& S, int mt, int nt, long long = 0) const {
    constexpr int NW = NT / 32;
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (NT > 256 && nt <= NW) {  // (with eight warps the chunks cost no more)
      if (w < nt) scan_one(S.nnk, w, mt);
      __syncthreads();
      return S.nnk;
    }
    const int cg = (nt + 63) >> 6, chunks = max(1, NW / cg);
    if (chunks > 1) {
      for (int q = threadIdx.x; q < nt; q += NT) S.nnk[q] = ~0ULL;
      __syncthreads();
    }
    for (int u = w; u < cg * chunks; u += NW) {
      const int qa = 64 * (u % cg) + lane, qb = qa + 32, ch = u / cg;
      const int s0 = (int)((unsigned)(mt * ch) / (unsigned)chunks);
      const int s1 = (int)((unsigned)(mt * (ch + 1)) / (unsigned)chunks);
      if (s0 >= s1) continue;
      unsigned long long ka, kb;
      scan_chunk(qa, qb, nt, s0, s1, ka, kb);
      if (chunks > 1) {
        if (qa < nt) atomicMin(&S.nnk[qa], ka);
        if (qb < nt) atomicMin(&S.nnk[qb], kb);
      } else {
        if (qa < nt) S.nnk[qa] = ka;
        if (qb < nt) S.nnk[qb] = kb;
      }
    }
    __syncthreads();
    return S.nnk;
  }
  // two consumers of a lane against a chunk (team_rounds)
  static constexpr bool kTeamRounds = true;
  NNS_DEV bool team_ready() const { return true; }
  NNS_DEV void team_count(int) const {}
  template <int C>
  NNS_DEV void team_scan(CtaCore<C>&, int qa, int qb, int nt, int s0, int s1, unsigned long long& ka,
                         unsigned long long& kb) const {
    scan_chunk(qa, qb, nt, s0, s1, ka, kb);
  }
};

// The NNS step of GeoSmem spread over the CTAs of a cluster.  CTA r of R
// (R >= 8) scans the consumers [r nt / R, (r+1) nt / R) against every active
// supplier and stores each key into the receive buffer of every CTA of the
// cluster; one cluster barrier (release / acquire) then makes all nt keys
// visible in every CTA, and the round's later steps read them there.  The
// receive buffer alternates between two halves by round parity: a CTA can
// write round t + 1's keys into a peer while the peer still reads round t's,
// never round t + 2's (that needs the peer at the barrier of round t + 1,
// after its round t).  Every CTA holds identical state, so every later step
// gives identical results in all of them.
//
// Inside a CTA a warp takes 64 consumers of the slice (two per lane, packed
// in FP32x2 registers) and a contiguous chunk of the suppliers; all lanes
// read the same supplier (a shared-memory broadcast), so one load feeds 64
// pairs.  Each lane keeps the first minimum of its chunk (ascending
// positions); the chunks merge through a 64-bit atomicMin on (key bits,
// position), which keeps the lowest-index tie-break.
template <int D, int DP, bool L1, int CAP, int NT>
struct GeoSmemCluster : GeoSmem<D, DP, L1, CAP, NT> {
  static constexpr int kThreads = NT;     // threads of each CTA
  static constexpr int kSlice = CAP / 8;  // consumers per CTA at most (R >= 8)
  unsigned long long xk[2][CAP];          // receive buffers (round parity)
  unsigned long long red[kSlice];         // the slice's keys merged over chunks; all ones between rounds

  // Set red to all ones (before the first round; each round restores it).
  NNS_DEV void init() {
    for (int i = threadIdx.x; i < kSlice; i += blockDim.x) red[i] = ~0ULL;
  }

  template <int C>
  NNS_DEV const unsigned long long* nns(CtaCore<C>& S, int mt, int nt, long long round) {
    // a small round's exchange and cluster barrier cost more than the scan by
    // itself: every CTA then scans it all (the product only shrinks, so the
    // buffers below are not used again).  65,536-point colours, the tail's 41
    // rounds: 911 us with the exchange in every round, 905 us with this line.
    if (mt * nt <= 128 * 128) return GeoSmem<D, DP, L1, CAP, NT>::nns(S, mt, nt);
    namespace cg = cooperative_groups;
    cg::cluster_group cl = cg::this_cluster();
    const unsigned rank = cl.block_rank(), ncl = cl.num_blocks();
    const int h = (int)(round & 1);
    // (32-bit arithmetic: nt, mt <= CAP and R, chunks <= 32)
    const int q0 = (int)((unsigned)nt * rank / ncl), q1 = (int)((unsigned)nt * (rank + 1) / ncl);
    const int tid = threadIdx.x, T = blockDim.x, ns = q1 - q0;
    const int cgroups = (ns + 63) >> 6, nw = T >> 5, w = tid >> 5, lane = tid & 31;
    if (cgroups > 0 && w < nw / cgroups * cgroups) {
      const int chunks = nw / cgroups, ch = w / cgroups;
      const int qa = 64 * (w % cgroups) + lane, qb = qa + 32;  // slice positions
      const int s0 = (int)((unsigned)(mt * ch) / (unsigned)chunks);
      const int s1 = (int)((unsigned)(mt * (ch + 1)) / (unsigned)chunks);
      if (s0 < s1) {
        unsigned long long ka, kb;
        this->scan_chunk(q0 + qa, q0 + qb, q1, s0, s1, ka, kb);
        if (qa < ns) atomicMin(&red[qa], ka);
        if (qb < ns) atomicMin(&red[qb], kb);
      }
    }
    __syncthreads();
    for (int i = tid; i < ns * (int)ncl; i += T) {
      const int r = i / ns, q = i - r * ns;
      cl.map_shared_rank(&xk[h][0], r)[q0 + q] = red[q];
    }
    cl.sync();
    // restore red for the next round (whose atomics follow this round's
    // barriers)
    for (int i = tid; i < ns; i += T) red[i] = ~0ULL;
    return xk[h];
  }
};

// ---- tiled FP32 NNS for d > 8 ---------------------------------------------

constexpr int TG_M = 64;        // consumers per tile
constexpr int TG_N = 64;        // suppliers per tile
constexpr int TG_K = 32;        // coordinates per staged chunk
constexpr int TG_THREADS = 256; // threads per group (4 x 4 pairs each)
constexpr int TG_PAD = 68;

struct __align__(16) TileSmem {
  float Xs[TG_K][TG_PAD];
  float Ys[TG_K][TG_PAD];
};

NNS_DEV void group_sync(int bar) {
  if (bar == 0) __syncthreads();
  else asm volatile("bar.sync %0, %1;" ::"r"(bar), "r"(TG_THREADS) : "memory");
}

// One 256-thread group: the FP32 keys of the consumers cons[c0 .. c0+nc)
// (positions in the list ja, or c0.. directly when cons is null; positions
// are row numbers where ja is null) against the suppliers at positions
// [p0, p1) (likewise through ia), TG_N suppliers at a time.  A thread owns 4
// consumers x 4 suppliers of a tile, the consumers packed two per FP32x2
// register; every pair's key is accumulated over k = 0..d-1 in order (fma
// from +0, which equals the definition's first product), so it is
// bit-identical to key32.  emit(pt, acc) takes each finished tile of
// suppliers pt..: acc[i][j] holds consumers 2i, 2i+1 of this thread against
// its supplier j (suppliers past p1 are NaN, consumers past nc arbitrary).
//
// Bound by the FP32 pipe (2 packed instructions per 2 pairs and coordinate)
// as long as the tiles arrive: rows of whole 16-byte vectors are read 16
// bytes per lane, 4 lanes to a 64-byte piece of one row (a warp touches 8
// rows per load; one row per lane with 4-byte loads cost 32 L1 lookups a load
// and kept the pipe at 0.30: the 16,384-point FP32 solve at d = 64 went from
// 6.87 to 3.55 ms, the 300 x 700 pair at d = 128 from 580 to 430 us).  PRE
// fetches the next 32 coordinates into registers while the current ones are
// used (for kernels with registers to spare).
template <bool L1, bool PRE, class Emit>
NNS_DEV void group_tiles(const float* __restrict__ x, const int* ia, int p0, int p1, const float* __restrict__ y,
                         const int* ja, const int* cons, int c0, int nc, int d, TileSmem& T, int gt, int bar,
                         Emit emit) {
  const int tx = gt & 15, ty = gt >> 4;
  const bool vec = (d & 3) == 0 && ((reinterpret_cast<uintptr_t>(x) | reinterpret_cast<uintptr_t>(y)) & 15) == 0;
  // loader: row lr of the tile, coordinates lk..lk+3 and lk+16..lk+19 of a chunk
  const int lr = gt >> 2, lk = (gt & 3) * 4;
  const float* yrow = nullptr;
  if (lr < nc) {
    const int q = cons ? cons[c0 + lr] : c0 + lr;
    yrow = y + (size_t)(ja ? ja[q] : q) * d;
  }
  const int nch = (d + TG_K - 1) / TG_K;
  const int steps = (p1 - p0 + TG_N - 1) / TG_N * nch;
  float4 rx[2], ry[2];
  auto fetch = [&](const float* row, int k, float pad) -> float4 {
    float4 v = make_float4(pad, pad, pad, pad);
    if (row) {
      if (vec) {
        v = k < d ? *reinterpret_cast<const float4*>(row + k) : make_float4(0.f, 0.f, 0.f, 0.f);
      } else {
        v.x = k < d ? row[k] : 0.f;
        v.y = k + 1 < d ? row[k + 1] : 0.f;
        v.z = k + 2 < d ? row[k + 2] : 0.f;
        v.w = k + 3 < d ? row[k + 3] : 0.f;
      }
    }
    return v;
  };
  int lt = p0, lc = 0;  // supplier tile and chunk of the next fetch
  const float* xrow = nullptr;
  auto load = [&]() {
    if (lc == 0) {
      const int sp = lt + lr;
      xrow = sp < p1 ? x + (size_t)(ia ? ia[sp] : sp) * d : nullptr;
    }
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int k = lc * TG_K + lk + 16 * h;
      rx[h] = fetch(xrow, k, CUDART_NAN_F);
      ry[h] = fetch(yrow, k, 0.f);
    }
    if (++lc == nch) {
      lc = 0;
      lt += TG_N;
    }
  };
  unsigned long long acc[2][4];
#pragma unroll
  for (int i = 0; i < 2; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) acc[i][j] = 0ULL;
  int pt = p0, ch = 0;
  if (PRE && steps > 0) load();
  for (int s = 0; s < steps; ++s) {
    if (!PRE) load();
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int k = lk + 16 * h;
      T.Xs[k][lr] = rx[h].x;
      T.Xs[k + 1][lr] = rx[h].y;
      T.Xs[k + 2][lr] = rx[h].z;
      T.Xs[k + 3][lr] = rx[h].w;
      T.Ys[k][lr] = ry[h].x;
      T.Ys[k + 1][lr] = ry[h].y;
      T.Ys[k + 2][lr] = ry[h].z;
      T.Ys[k + 3][lr] = ry[h].w;
    }
    group_sync(bar);
    if (PRE && s + 1 < steps) load();
    const int kn = min(TG_K, (d - ch * TG_K + 7) & ~7);  // coordinates past d are 0 - 0 on both sides
#pragma unroll 1
    for (int kb = 0; kb < kn; kb += 8)
#pragma unroll
      for (int ku = 0; ku < 8; ++ku) {
        const int k = kb + ku;
        const float4 xv = *reinterpret_cast<const float4*>(&T.Xs[k][tx * 4]);
        const ulonglong2 yv = *reinterpret_cast<const ulonglong2*>(&T.Ys[k][ty * 4]);
        const float xa[4] = {xv.x, xv.y, xv.z, xv.w};
        const unsigned long long ya[2] = {yv.x, yv.y};
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          const unsigned long long xx = f2_pack(xa[j], xa[j]);
#pragma unroll
          for (int i = 0; i < 2; ++i) {
            const unsigned long long t = f2_sub(xx, ya[i]);
            acc[i][j] = L1 ? f2_add(acc[i][j], t & 0x7fffffff7fffffffULL) : f2_fma(t, t, acc[i][j]);
          }
        }
      }
    group_sync(bar);
    if (++ch == nch) {
      ch = 0;
      emit(pt, acc);
      pt += TG_N;
#pragma unroll
      for (int i = 0; i < 2; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j] = 0ULL;
    }
  }
}

// The lowest (key32 bits << 32 | position) over the suppliers [p0, p1) of
// each consumer of group_tiles; returned, in the threads with tx == 0, for
// their 4 consumers (~0 only where p0 == p1).  A thread starts at +inf and its
// own first supplier, so a consumer whose keys all overflow to +inf gets the
// first position, as from a scan in order.  each(pt, acc) sees every tile of
// keys as group_tiles' emit does.
struct NoTile {
  NNS_DEV void operator()(int, const unsigned long long (&)[2][4]) const {}
};
template <bool L1, bool PRE = false, class Each = NoTile>
NNS_DEV void group_nns_tile(const float* __restrict__ x, const int* ia, int p0, int p1, const float* __restrict__ y,
                            const int* ja, const int* cons, int c0, int nc, int d, TileSmem& T, int gt, int bar,
                            unsigned long long out[4], Each each = Each()) {
  const int tx = gt & 15;
  float best[4];
  int bpos[4];
#pragma unroll
  for (int i = 0; i < 4; ++i) { best[i] = CUDART_INF_F; bpos[i] = p0 + tx * 4 < p1 ? p0 + tx * 4 : -1; }
  group_tiles<L1, PRE>(x, ia, p0, p1, y, ja, cons, c0, nc, d, T, gt, bar,
                       [&](int pt, const unsigned long long (&acc)[2][4]) {
#pragma unroll
                         for (int j = 0; j < 4; ++j)
#pragma unroll
                           for (int i = 0; i < 2; ++i) {
                             const float lo = f2_lo(acc[i][j]), hi = f2_hi(acc[i][j]);
                             if (lo < best[2 * i]) { best[2 * i] = lo; bpos[2 * i] = pt + tx * 4 + j; }
                             if (hi < best[2 * i + 1]) { best[2 * i + 1] = hi; bpos[2 * i + 1] = pt + tx * 4 + j; }
                           }
                         each(pt, acc);
                       });
  // reduce over the 16 threads sharing each consumer (adjacent lanes)
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    unsigned long long k = bpos[i] >= 0 ? pack_key(best[i], (unsigned)bpos[i]) : ~0ULL;
#pragma unroll
    for (int o = 1; o < 16; o <<= 1) {
      const unsigned long long other = __shfl_xor_sync(0xffffffffu, k, o);
      k = other < k ? other : k;
    }
    out[i] = k;
  }
}

template <bool L1, int CAP, int NT = FIN_THREADS>
struct GeoGlobal {
  static constexpr int kDP = 0;
  static constexpr int kThreads = NT;  // threads of the CTA (a multiple of TG_THREADS)
  const float* x;  // [m][d] original coordinates (global)
  const float* y;  // [n][d]
  int d;
  // The pair's key matrix (nullable), by original supplier (row, kld floats
  // apart) and consumer: the FP32 keys are computed once in the first round's NNS
  // step; every round is then a minimum over rows of active
  // suppliers instead of m_t n_t d operations (1 x 4,096 documents, d = 300:
  // 11.7 -> 3.09 ms).
  float* kmat;
  int kld, km, kn, kready;
  unsigned long long searches;  // consumer searches of all rounds so far
  TileSmem tiles[NT / TG_THREADS];
  struct PX {};
  NNS_DEV void load_x(int, PX&) const {}
  NNS_DEV void store_x(int, const PX&) {}
  NNS_DEV void load_y(int, PX&) const {}
  NNS_DEV void store_y(int, const PX&) {}
  template <int C>
  NNS_DEV double dist64(const CtaCore<C>& S, int p, int q, int metric) const {
    return cost_dist64(x + (size_t)S.iidx[p] * d, y + (size_t)S.jidx[q] * d, d, metric);
  }
  // Set up a pair (thread 0; the caller's barrier follows): kcap floats at
  // km_ for its key matrix, used where the pair's fits.
  NNS_DEV void begin(const float* x_, const float* y_, int m, int n, int d_, float* km_, long long kcap) {
    x = x_;
    y = y_;
    d = d_;
    kld = (int)kmat_ld(n);
    km = m;
    kn = n;
    kmat = km_ && (long long)m * kld <= kcap ? km_ : nullptr;
    kready = 0;
    searches = 0;
  }
  // The whole key matrix, one 64 x 64 tile per group at a time.
  NNS_DEV void fill() {
    const int g = threadIdx.x / TG_THREADS, gt = threadIdx.x % TG_THREADS;
    const int tx = gt & 15, ty = gt >> 4;
    const int ct = (kn + TG_M - 1) / TG_M, items = ct * ((km + TG_N - 1) / TG_N);
    for (int it = g; it < items; it += NT / TG_THREADS) {
      const int c0 = (it % ct) * TG_M, p0 = (it / ct) * TG_N;
      group_tiles<L1, false>(x, nullptr, p0, min(p0 + TG_N, km), y, nullptr, nullptr, c0, min(TG_M, kn - c0), d,
                             tiles[g], gt, 1 + g, [&](int pt, const unsigned long long (&acc)[2][4]) {
                               const int q = c0 + ty * 4;  // four consecutive consumers: one 16-byte store
                               if (q >= kn) return;
#pragma unroll
                               for (int j = 0; j < 4; ++j) {
                                 const int p = pt + tx * 4 + j;
                                 if (p < km)
                                   *reinterpret_cast<ulonglong2*>(kmat + (size_t)p * kld + q) =
                                       make_ulonglong2(acc[0][j], acc[1][j]);
                               }
                             });
    }
  }
  // The same for a pair of which some points have no weight: the keys of the mt
  // and nt active ones alone (200 pairs of 1,000 points, d = 300, 5 % of the
  // weights not zero: 7.5 ms with every point's keys, 0.43 with these, 1.7
  // without a matrix).
  template <int C>
  __device__ __noinline__ void fill_active(const CtaCore<C>& S, int mt, int nt) {
    const int g = threadIdx.x / TG_THREADS, gt = threadIdx.x % TG_THREADS;
    const int tx = gt & 15, ty = gt >> 4;
    const int ct = (nt + TG_M - 1) / TG_M, items = ct * ((mt + TG_N - 1) / TG_N);
    for (int it = g; it < items; it += NT / TG_THREADS) {
      const int c0 = (it % ct) * TG_M, p0 = (it / ct) * TG_N;
      group_tiles<L1, false>(x, S.iidx, p0, min(p0 + TG_N, mt), y, S.jidx, nullptr, c0, min(TG_M, nt - c0), d, tiles[g],
                             gt, 1 + g, [&](int pt, const unsigned long long (&acc)[2][4]) {
#pragma unroll
                               for (int j = 0; j < 4; ++j) {
                                 const int p = pt + tx * 4 + j;
                                 if (p >= mt) break;
                                 float* row = kmat + (size_t)S.iidx[p] * kld;
#pragma unroll
                                 for (int i = 0; i < 4; ++i) {
                                   const int q = c0 + ty * 4 + i;
                                   if (q < nt) row[S.jidx[q]] = (i & 1) ? f2_hi(acc[i >> 1][j]) : f2_lo(acc[i >> 1][j]);
                                 }
                               }
                             });
    }
  }
  // The NNS step on the key matrix: a warp takes 32 consumers (one per lane)
  // and a contiguous chunk of the active suppliers, eight rows in flight;
  // keys order like their bit patterns (no key is negative or NaN), each
  // lane keeps its first minimum, and chunks merge by atomicMin.
  template <int C>
  NNS_DEV void scan(CtaCore<C>& S, int mt, int nt) const {
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    constexpr int NW = NT / 32;
    const int cg = (nt + 31) >> 5, chunks = max(1, NW / cg);
    if (chunks > 1) {
      for (int q = threadIdx.x; q < nt; q += NT) S.nnk[q] = ~0ULL;
      __syncthreads();
    }
    for (int u = w; u < cg * chunks; u += NW) {
      const int q = 32 * (u % cg) + lane, ch = u / cg;
      const int s0 = (int)((unsigned)(mt * ch) / (unsigned)chunks);
      const int s1 = (int)((unsigned)(mt * (ch + 1)) / (unsigned)chunks);
      const float* col = kmat + S.jidx[q < nt ? q : 0];
      unsigned best = 0xffffffffu;
      int bp = 0;
      for (int p = s0; p < s1; p += 8) {
        unsigned v[8];
#pragma unroll
        for (int e = 0; e < 8; ++e)
          v[e] = p + e < s1 ? __float_as_uint(col[(size_t)S.iidx[p + e] * kld]) : 0xffffffffu;
#pragma unroll
        for (int e = 0; e < 8; ++e)
          if (v[e] < best) { best = v[e]; bp = p + e; }
      }
      const unsigned long long key = ((unsigned long long)best << 32) | (unsigned)bp;
      if (q < nt && s0 < s1) {
        if (chunks > 1) atomicMin(&S.nnk[q], key);
        else S.nnk[q] = key;
      }
    }
    __syncthreads();
  }
  // two consumers of a lane against a chunk (team_rounds)
  static constexpr bool kTeamRounds = true;
  NNS_DEV bool team_ready() const { return kmat != nullptr && kready; }
  NNS_DEV void team_count(int nt) { searches += nt; }
  template <int C>
  NNS_DEV void team_scan(CtaCore<C>& S, int qa, int qb, int nt, int s0, int s1, unsigned long long& ka,
                         unsigned long long& kb) const {
    const float* ca = kmat + S.jidx[qa < nt ? qa : 0];
    const float* cb = kmat + S.jidx[qb < nt ? qb : 0];
    unsigned ba = 0xffffffffu, bb = 0xffffffffu;
    int pa = s0, pb = s0;
    for (int p = s0; p < s1; p += 8) {
      unsigned va[8], vb[8];
#pragma unroll
      for (int e = 0; e < 8; ++e) {
        const size_t row = (size_t)S.iidx[min(p + e, s1 - 1)] * kld;
        va[e] = __float_as_uint(ca[row]);
        vb[e] = __float_as_uint(cb[row]);
      }
#pragma unroll
      for (int e = 0; e < 8; ++e) {  // (repeats of the last supplier never win)
        if (va[e] < ba) { ba = va[e]; pa = p + e; }
        if (vb[e] < bb) { bb = vb[e]; pb = p + e; }
      }
    }
    ka = ((unsigned long long)ba << 32) | (unsigned)pa;
    kb = ((unsigned long long)bb << 32) | (unsigned)pb;
  }
  template <int C>
  NNS_DEV const unsigned long long* nns(CtaCore<C>& S, int mt, int nt, long long = 0) {
    if (threadIdx.x == 0) searches += nt;
    if (kmat) {
      if (!kready) {
        if (mt == km && nt == kn) fill();  // (positions are the original indices)
        else fill_active(S, mt, nt);
        __syncthreads();
        if (threadIdx.x == 0) kready = 1;  // (read again after this step's barriers)
      }
      scan(S, mt, nt);
      return S.nnk;
    }
    const int g = threadIdx.x / TG_THREADS, gt = threadIdx.x % TG_THREADS;
    const int ngroups = blockDim.x / TG_THREADS;
    for (int c0 = g * TG_M; c0 < nt; c0 += ngroups * TG_M) {
      unsigned long long out[4];
      group_nns_tile<L1>(x, S.iidx, 0, mt, y, S.jidx, nullptr, c0, min(TG_M, nt - c0), d, tiles[g], gt, 1 + g,
                         out);
      const int tx = gt & 15, ty = gt >> 4;
      if (tx == 0)
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const int q = c0 + ty * 4 + i;
          if (q < nt) S.nnk[q] = out[i];
        }
    }
    __syncthreads();
    return S.nnk;
  }
};

// The tail of a large d > 8 solve on a thread-block cluster: the key matrix of
// its first round's active points (positions at that time; filled before the
// launch) stays in global memory, every CTA holds the whole per-point state
// with each point's row or column, and the NNS step is split over the CTAs
// and exchanged like GeoSmemCluster's.  A warp takes 32 consumers of the slice
// and a chunk of the active suppliers, 16 rows in flight.
template <int CAP, int NT>
struct GeoMatCluster {
  static constexpr int kDP = 0;
  static constexpr int kThreads = NT;
  static constexpr bool kTeamRounds = true;
  static constexpr int kSlice = CAP / 8;  // consumers per CTA at most (R >= 8)
  const float* kmat;
  int kld;
  int row[CAP];
  int col[CAP];
  unsigned long long xk[2][CAP];   // receive buffers (round parity)
  unsigned long long red[kSlice];  // the slice's keys merged over chunks; all ones between rounds
  struct PX { int v; };
  NNS_DEV void load_x(int p, PX& r) const { r.v = row[p]; }
  NNS_DEV void store_x(int p, const PX& r) { row[p] = r.v; }
  NNS_DEV void load_y(int q, PX& r) const { r.v = col[q]; }
  NNS_DEV void store_y(int q, const PX& r) { col[q] = r.v; }
  template <int C>
  NNS_DEV double dist64(const CtaCore<C>&, int, int, int) const { return 0.0; }  // (flows are costed after the tail)

  // The first minimum of column c (this lane's) over the active suppliers
  // [s0, s1): keys order like their bit patterns (none is negative or NaN).
  NNS_DEV unsigned long long scan_col(int c, int s0, int s1) const {
    constexpr int F = 16;
    unsigned best = 0xffffffffu;
    int bp = s0;
    for (int p = s0; p < s1; p += F) {
      unsigned v[F];
#pragma unroll
      for (int e = 0; e < F; ++e) v[e] = __float_as_uint(kmat[(size_t)row[min(p + e, s1 - 1)] * kld + c]);
#pragma unroll
      for (int e = 0; e < F; ++e)  // (repeats of the last supplier never win)
        if (v[e] < best) { best = v[e]; bp = p + e; }
    }
    return ((unsigned long long)best << 32) | (unsigned)bp;
  }
  NNS_DEV void init() {
    for (int i = threadIdx.x; i < kSlice; i += NT) red[i] = ~0ULL;
  }
  template <int C>
  NNS_DEV const unsigned long long* nns(CtaCore<C>&, int mt, int nt, long long round) {
    namespace cg = cooperative_groups;
    cg::cluster_group cl = cg::this_cluster();
    const unsigned rank = cl.block_rank(), ncl = cl.num_blocks();
    const int h = (int)(round & 1);
    const int q0 = (int)((unsigned)nt * rank / ncl), q1 = (int)((unsigned)nt * (rank + 1) / ncl);
    const int ns = q1 - q0;
    constexpr int NW = NT / 32;
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int cgroups = (ns + 31) >> 5;
    if (cgroups > 0 && w < NW / cgroups * cgroups) {  // (at most NW groups: kSlice / 32)
      const int chunks = NW / cgroups, ch = w / cgroups;
      const int qa = 32 * (w % cgroups) + lane;
      const int s0 = (int)((unsigned)(mt * ch) / (unsigned)chunks);
      const int s1 = (int)((unsigned)(mt * (ch + 1)) / (unsigned)chunks);
      if (s0 < s1) {
        const unsigned long long k = scan_col(col[q0 + min(qa, ns - 1)], s0, s1);
        if (qa < ns) atomicMin(&red[qa], k);
      }
    }
    __syncthreads();
    for (int i = threadIdx.x; i < ns * (int)ncl; i += NT) {
      const int r = i / ns, q = i - r * ns;
      cl.map_shared_rank(&xk[h][0], r)[q0 + q] = red[q];
    }
    cl.sync();
    for (int i = threadIdx.x; i < ns; i += NT) red[i] = ~0ULL;
    return xk[h];
  }
  NNS_DEV bool team_ready() const { return true; }
  NNS_DEV void team_count(int) const {}
  template <int C>
  NNS_DEV void team_scan(CtaCore<C>&, int qa, int qb, int nt, int s0, int s1, unsigned long long& ka,
                         unsigned long long& kb) const {
    ka = scan_col(col[min(qa, nt - 1)], s0, s1);
    kb = scan_col(col[min(qb, nt - 1)], s0, s1);
  }
};

// Note: GeoGlobal passes the CTA's own index arrays (iidx, jidx) as the
// "position -> original index" maps, so positions are CTA-local.

// --------------------------------------------------------------------------
// compaction and rounds
// --------------------------------------------------------------------------

// Stable compaction of both active lists to the points with weight left.
// Warp w owns positions [32 IT w, 32 IT (w + 1)), lane l the positions
// 32 IT w + 32 k + l (coalesced shared-memory accesses); ballots give each
// kept point its rank inside the warp and one block scan the warps' offsets.
// Every kept value is loaded before the scan's barriers and stored after
// them, so the in-place moves never overwrite a value not yet read.
template <int CAP, class Geo>
NNS_DEV void cta_compact(CtaCore<CAP>& S, Geo& G) {
  constexpr int IT = (CAP + Geo::kThreads - 1) / Geo::kThreads;
  const int tid = threadIdx.x, lane = tid & 31;
  const int base = (tid >> 5) * 32 * IT;
  const unsigned lt = (1u << lane) - 1u;
  const int mt = S.mt, nt = S.nt;
  unsigned bs[IT], bc[IT];
  double sv[IT], cv[IT];
  int iv[IT], jv[IT];
  typename Geo::PX px[IT], py[IT];
  int ns = 0, nc = 0;
#pragma unroll
  for (int k = 0; k < IT; ++k) {
    const int p = base + 32 * k + lane;
    bool ks = false, kc = false;
    if (p < mt) {
      sv[k] = S.sres[p];
      ks = residual_positive(sv[k]);
      if (ks) { iv[k] = S.iidx[p]; G.load_x(p, px[k]); }
    }
    if (p < nt) {
      cv[k] = S.cres[p];
      kc = residual_positive(cv[k]);
      if (kc) { jv[k] = S.jidx[p]; G.load_y(p, py[k]); }
    }
    bs[k] = __ballot_sync(0xffffffffu, ks);
    bc[k] = __ballot_sync(0xffffffffu, kc);
    ns += __popc(bs[k]);
    nc += __popc(bc[k]);
  }
  int tot;
  const int ex = __shfl_sync(0xffffffffu, block_scan_excl(lane == 0 ? (ns | (nc << 16)) : 0, S.wt, tot), 0);
  int ps = ex & 0xffff, pc = ex >> 16;
#pragma unroll
  for (int k = 0; k < IT; ++k) {
    if ((bs[k] >> lane) & 1u) {
      const int d = ps + __popc(bs[k] & lt);
      S.sres[d] = sv[k];
      S.iidx[d] = iv[k];
      G.store_x(d, px[k]);
    }
    if ((bc[k] >> lane) & 1u) {
      const int d = pc + __popc(bc[k] & lt);
      S.cres[d] = cv[k];
      S.jidx[d] = jv[k];
      G.store_y(d, py[k]);
    }
    ps += __popc(bs[k]);
    pc += __popc(bc[k]);
  }
  // every thread read the old counts before the scan's barriers
  if (tid == 0) {
    S.mt = tot & 0xffff;
    S.nt = tot >> 16;
  }
  __syncthreads();
}

// Exclusive scan of in[0..n) into out[0..n) (n <= CAP, NT threads), returns
// the total.
template <int CAP, int NT>
NNS_DEV int block_scan_array(const int* in, int* out, int n, int* wt) {
  constexpr int IT = (CAP + NT - 1) / NT;
  int v[IT];
  int s = 0;
#pragma unroll
  for (int k = 0; k < IT; ++k) {
    const int i = threadIdx.x * IT + k;
    v[k] = i < n ? in[i] : 0;
    s += v[k];
  }
  int tot;
  int ex = block_scan_excl(s, wt, tot);
#pragma unroll
  for (int k = 0; k < IT; ++k) {
    const int i = threadIdx.x * IT + k;
    if (i < n) out[i] = ex;
    ex += v[k];
  }
  return tot;
}

// Active sets both at most TEAM_CAP points go to team_rounds.
constexpr int TEAM_CAP = 64;
constexpr int TEAM_WARPS = 4;
NNS_DEV void team_sync() { asm volatile("bar.sync 15, %0;" ::"n"(32 * TEAM_WARPS) : "memory"); }

// The remaining rounds of a pair whose active sets both hold at most TEAM_CAP
// points, run by the CTA's first four warps (policies with kTeamRounds): with
// a few dozen points left, a round of the block-wide steps below is mostly
// barriers of every warp and scans.  The same steps in the same arithmetic as
// cta_rounds, so every result is identical:
//   NNS     each warp scans a quarter of the suppliers for two consumers a
//           lane (the policy's team_scan); quarters merge by atomicMin;
//   order   every consumer's (supplier position, serving key, position) as
//           one 64-bit word and its rank among all of them, one consumer a
//           lane; the members of a group then lie in serving order;
//   flow    lane = supplier, the FP64 residual chain over its group;
//   compact ballots keep the points with residual left, in order, two warps a
//           side.
// (One warp alone took 3,700 cycles a round, 1,900 of them in the NNS and
// 1,700 in the order.  2,048 batched images of some 500 points, GB300: 620 us
// with one warp, 549 us with four; a pair of 256 points 61 and 60 us.)
template <int CAP, class Geo>
NNS_DEV void team_rounds(CtaCore<CAP>& S, Geo& G, int metric, const CtaOut& O, unsigned long long& nnz,
                         long long& rounds, long long& pair_evals, long long round_limit) {
  static_assert(CAP >= 2 * TEAM_CAP && Geo::kThreads >= 32 * TEAM_WARPS, "a round's flows; the team");
  const int t = threadIdx.x, lane = t & 31, w = t >> 5;
  const unsigned lt = (1u << lane) - 1u;
  const bool deferred = O.fl_i != nullptr;
  for (;;) {
    const int mt = S.mt, nt = S.nt;
    if (mt == 0 || nt == 0) break;
    if (rounds >= round_limit) {
      if (t == 0) atomicOr(O.err, EF_ITER);
      break;
    }
    if (t == 0) {
      S.nflow = 0;
      G.team_count(nt);
    }
    if (t < mt) S.cnt[t] = 0;
    if (t >= 64 && t - 64 < nt) S.nnk[t - 64] = ~0ULL;
    team_sync();
    // ---- NNS
    {
      const int s0 = mt * w / TEAM_WARPS, s1 = mt * (w + 1) / TEAM_WARPS;
      if (s0 < s1) {
        unsigned long long ka, kb;
        G.team_scan(S, lane, lane + 32, nt, s0, s1, ka, kb);
        if (lane < nt) atomicMin(&S.nnk[lane], ka);
        if (lane + 32 < nt) atomicMin(&S.nnk[lane + 32], kb);
      }
    }
    team_sync();
    // ---- order: (supplier, serving key, consumer) of every consumer, then
    // its rank among all of them
    unsigned long long mine = ~0ULL;
    if (t < nt) {
      const unsigned long long key = S.nnk[t];
      const unsigned ord = O.protocol == 1 ? rp_key32(O.seed, O.round_base + rounds, S.jidx[t]) : (unsigned)(key >> 32);
      mine = ((key & 0xffffULL) << 40) | ((unsigned long long)ord << 8) | (unsigned)t;
    }
    if (t < ((nt + 3) & ~3)) S.mem[t] = mine;
    team_sync();
    if (t < nt) {
      int rank = 0;
      for (int u = 0; u < nt; u += 4) {
        const ulonglong2 o = *reinterpret_cast<const ulonglong2*>(&S.mem[u]);
        const ulonglong2 v = *reinterpret_cast<const ulonglong2*>(&S.mem[u + 2]);
        rank += (o.x < mine) + (o.y < mine) + (v.x < mine) + (v.y < mine);
      }
      S.mem2[rank] = mine;
    }
    team_sync();
    // group bounds: where the supplier changes along the order
    if (t < nt) {
      const int p = (int)(S.mem2[t] >> 40);
      if (t == 0 || (int)(S.mem2[t - 1] >> 40) != p) S.off[p] = t;
      if (t == nt - 1 || (int)(S.mem2[t + 1] >> 40) != p) S.cnt[p] = t + 1;  // the group's end
    }
    team_sync();
    // ---- flow, one supplier per lane
    if (t < mt && S.cnt[t] > 0) {
      const int p = t, b = S.off[p], en = S.cnt[p];
      double s = S.sres[p];
      for (int r = b; r < en; ++r) {
        if (!residual_positive(s)) break;
        const int q = (int)(S.mem2[r] & 0xffULL);
        double c = S.cres[q];
        const double f = greedy_step(s, c);
        S.cres[q] = c;
        const unsigned k = atomicAdd(&S.nflow, 1u);
        if (O.quiet) {
        } else if (deferred) {
          const unsigned long long slot = nnz + k;
          if (O.fl_cap && (long long)slot >= O.fl_cap) {
            atomicOr(O.err, EF_CAPACITY);
            continue;
          }
          O.fl_i[slot] = S.iidx[p];
          O.fl_j[slot] = S.jidx[q];
          O.fl_f[slot] = f;
          if (O.c_glob) O.c_glob[S.jidx[q]] = c;
        } else {
          // (mem and nnk are free again: the order is in mem2)
          S.mem[k] = ((unsigned long long)p << 32) | (unsigned)q;
          S.nnk[k] = (unsigned long long)__double_as_longlong(f);
        }
      }
      S.sres[p] = s;
      if (O.s_glob) O.s_glob[S.iidx[p]] = s;
    }
    team_sync();
    const unsigned nflow = S.nflow;
    if (!(deferred || O.quiet)) {
      for (unsigned base = 0; base < nflow; base += 32 * TEAM_WARPS) {  // whole warps (xs_add_warp)
        const unsigned k = base + t;
        double term = 0.0;
        if (k < nflow) {
          const unsigned long long pq = S.mem[k];
          const int p = (int)(pq >> 32), q = (int)(pq & 0xffffffffULL);
          const double f = __longlong_as_double((long long)S.nnk[k]);
          term = __dmul_rn(f, G.dist64(S, p, q, metric));
          const unsigned long long slot = nnz + k;
          if (O.plan_i) {
            if ((long long)slot < O.plan_cap) {
              O.plan_i[slot] = S.iidx[p];
              O.plan_j[slot] = S.jidx[q];
              O.plan_f[slot] = f;
            } else {
              atomicOr(O.err, EF_CAPACITY);
            }
          }
          if (O.c_glob) O.c_glob[S.jidx[q]] = S.cres[q];
        }
        if (O.acc) xs_add_warp(O.acc, term);  // one call site for the whole warp
      }
      team_sync();
    }
    nnz += nflow;
    rounds += 1;
    pair_evals += (long long)mt * nt;
    // ---- compaction: warps 0, 1 the suppliers, 2, 3 the consumers; every
    // kept value is read before any is written
    const bool sup = w < 2;
    const int i = t & 63;
    bool keep = false;
    double v = 0.0;
    int id = 0;
    typename Geo::PX px;
    if (i < (sup ? mt : nt)) {
      v = sup ? S.sres[i] : S.cres[i];
      keep = residual_positive(v);
      if (keep) {
        id = sup ? S.iidx[i] : S.jidx[i];
        if (sup) G.load_x(i, px);
        else G.load_y(i, px);
      }
    }
    const unsigned bal = __ballot_sync(0xffffffffu, keep);
    if (lane == 0) S.wt[w] = __popc(bal);
    team_sync();
    if (keep) {
      const int at = ((w & 1) ? S.wt[w - 1] : 0) + __popc(bal & lt);
      (sup ? S.sres : S.cres)[at] = v;
      (sup ? S.iidx : S.jidx)[at] = id;
      if (sup) G.store_x(at, px);
      else G.store_y(at, px);
    }
    if (t == 0) S.mt = S.wt[0] + S.wt[1];
    if (t == 64) S.nt = S.wt[2] + S.wt[3];
    team_sync();
  }
}

// Rounds of Alg. 1 until one active side is empty.  nnz, rounds and
// pair_evals are running totals (identical in every thread on return).
// The rounds after both active sets fit TEAM_CAP run in the first four warps
// (team_rounds) while the others wait.
template <int CAP, class Geo>
NNS_DEV void cta_rounds(CtaCore<CAP>& S, Geo& G, int metric, const CtaOut& O, unsigned long long& nnz,
                        long long& rounds, long long& pair_evals, long long round_limit) {
  const int tid = threadIdx.x;
  const int T = blockDim.x;
  const unsigned long long nnz0 = nnz;
  for (;;) {
    const int mt = S.mt, nt = S.nt;
    if (mt == 0 || nt == 0) break;
    if (rounds >= round_limit) {
      if (tid == 0) atomicOr(O.err, EF_ITER);
      break;
    }
    if constexpr (Geo::kTeamRounds) {
      if (mt <= TEAM_CAP && nt <= TEAM_CAP && G.team_ready()) {
        if (tid < 32 * TEAM_WARPS) {
          team_rounds(S, G, metric, O, nnz, rounds, pair_evals, round_limit);
          if (tid == 0) {
            S.w_nnz = nnz;
            S.w_rounds = rounds;
            S.w_pe = pair_evals;
          }
        }
        __syncthreads();
        nnz = S.w_nnz;
        rounds = S.w_rounds;
        pair_evals = S.w_pe;
        break;
      }
    }
    // group counters of this round (the NNS step ends with a barrier)
    for (int p = tid; p < mt; p += T) S.cnt[p] = 0;
    if (tid == 0) S.nflow = 0;
    // ---- NNS: nearest active supplier of every active consumer
    const unsigned long long* nk = G.nns(S, mt, nt, rounds);
    // ---- group the consumers by their supplier
    for (int q = tid; q < nt; q += T) atomicAdd(&S.cnt[(int)(nk[q] & 0xffffffffULL)], 1);
    __syncthreads();
    {
      const int tot = block_scan_array<CAP, Geo::kThreads>(S.cnt, S.off, mt, S.wt);
      if (tid == 0) S.off[mt] = tot;
    }
    __syncthreads();
    for (int q = tid; q < nt; q += T) {
      const unsigned long long key = nk[q];
      const int p = (int)(key & 0xffffffffULL);
      const int slot = S.off[p] + atomicSub(&S.cnt[p], 1) - 1;
      const unsigned long long order =
          O.protocol == 1 ? ((unsigned long long)rp_key32(O.seed, O.round_base + rounds, S.jidx[q]) << 32)
                          : (key & 0xffffffff00000000ULL);
      S.mem[slot] = order | (unsigned)q;
    }
    __syncthreads();
    // ---- greedy order: rank of each member inside its group
    for (int r = tid; r < nt; r += T) {
      const unsigned long long e = S.mem[r];
      const int q = (int)(e & 0xffffffffULL);
      const int p = (int)(nk[q] & 0xffffffffULL);
      const int b = S.off[p], en = S.off[p + 1];
      int rank = 0;
      for (int u = b; u < en; ++u) rank += S.mem[u] < e;
      S.mem2[b + rank] = e;
    }
    __syncthreads();
    // ---- flow (greedy protocol), one supplier per thread: the residual
    // chain only; each flow is recorded (deferred costing: its original
    // indices and f in O.fl_*; otherwise (p, q) and f in mem / nnk, which are
    // free after the ordering step; every consumer flows at most once)
    const bool deferred = O.fl_i != nullptr;
    for (int p = tid; p < mt; p += T) {
      const int b = S.off[p], en = S.off[p + 1];
      if (b == en) continue;
      double s = S.sres[p];
      for (int r = b; r < en; ++r) {
        if (!residual_positive(s)) break;
        const int q = (int)(S.mem2[r] & 0xffffffffULL);
        double c = S.cres[q];
        const double f = greedy_step(s, c);
        S.cres[q] = c;
        const unsigned k = atomicAdd(&S.nflow, 1u);
        if (O.quiet) {
        } else if (deferred) {
          const unsigned long long slot = nnz + k;
          if (O.fl_cap && (long long)slot >= O.fl_cap) {
            atomicOr(O.err, EF_CAPACITY);
            continue;
          }
          O.fl_i[slot] = S.iidx[p];
          O.fl_j[slot] = S.jidx[q];
          O.fl_f[slot] = f;
          if (O.c_glob) O.c_glob[S.jidx[q]] = c;
        } else {
          S.mem[k] = ((unsigned long long)p << 32) | (unsigned)q;
          S.nnk[k] = (unsigned long long)__double_as_longlong(f);
        }
      }
      S.sres[p] = s;
      if (O.s_glob) O.s_glob[S.iidx[p]] = s;
    }
    __syncthreads();
    // ---- cost terms and plan entries of the round's flows, one per thread
    const unsigned nflow = S.nflow;
    for (unsigned base = (deferred || O.quiet) ? nflow : 0; base < nflow; base += T) {  // whole warps
      const unsigned k = base + tid;
      double term = 0.0;
      if (k < nflow) {
        const unsigned long long pq = S.mem[k];
        const int p = (int)(pq >> 32), q = (int)(pq & 0xffffffffULL);
        const double f = __longlong_as_double((long long)S.nnk[k]);
        term = __dmul_rn(f, G.dist64(S, p, q, metric));
        const unsigned long long slot = nnz + k;
        if (O.plan_i) {
          if ((long long)slot < O.plan_cap) {
            O.plan_i[slot] = S.iidx[p];
            O.plan_j[slot] = S.jidx[q];
            O.plan_f[slot] = f;
          } else {
            atomicOr(O.err, EF_CAPACITY);
          }
        }
        if (O.c_glob) O.c_glob[S.jidx[q]] = S.cres[q];
      }
      if (O.acc) xs_add_warp(O.acc, term);  // one call site for the whole warp
    }
    // (the compaction rewrites what this loop reads; with the loop empty
    // the flow step's barrier suffices)
    if (!(deferred || O.quiet)) __syncthreads();
    nnz += nflow;
    rounds += 1;
    pair_evals += (long long)mt * nt;
    // ---- weights update: retire spent points, compact
    cta_compact(S, G);
  }
  if (O.fl_i && (O.acc || O.plan_i)) {
    // deferred costing: the terms and plan entries of every flow of the loop
    // (a solve whose later pass costs all its flows records them only)
    for (unsigned long long base = nnz0; base < nnz; base += T) {  // whole warps (xs_add_warp)
      const unsigned long long k = base + tid;
      double term = 0.0;
      if (k < nnz) {
        const int i = O.fl_i[k], j = O.fl_j[k];
        const double f = O.fl_f[k];
        term = __dmul_rn(f, cost_dist64(O.x + (size_t)i * O.d, O.y + (size_t)j * O.d, O.d, metric));
        if (O.plan_i) {
          if ((long long)k < O.plan_cap) {
            O.plan_i[k] = i;
            O.plan_j[k] = j;
            O.plan_f[k] = f;
          } else {
            atomicOr(O.err, EF_CAPACITY);
          }
        }
      }
      if (O.acc) xs_add_warp(O.acc, term);  // one call site for the whole warp
    }
    __syncthreads();
  }
}

// Load both sides of a pair (raw rows, weights) into the CTA state, check
// them, and normalise each side's weights by their correctly rounded total.
// With DP > 0 the coordinates are copied (zero-padded to DP) into xs / ys.
// The sides go through every step together (one after the other they took
// twice the latency: 7 us of a 256-point solve).  Clears acc.
template <int DP, int CAP>
NNS_DEV bool cta_load_sides(const float* x, const double* a, int m, const float* y, const double* b, int n, int d,
                            float* xs, float* ys, CtaCore<CAP>& S, unsigned* err) {
  const int tid = threadIdx.x;
  for (int i = tid; i < XS_LIMBS; i += blockDim.x) S.acc[i] = S.acc2()[i] = 0ULL;
  __syncthreads();
  unsigned bad = 0;  // bits 0, 1: a value of x / y not finite; bits 2, 3: a weight of a / b negative
#pragma unroll 1
  for (int base = 0; base < max(m, n); base += blockDim.x) {  // whole warps (xs_add_warp)
    const int p = base + tid;
    double add[2] = {0.0, 0.0};
#pragma unroll
    for (int sd = 0; sd < 2; ++sd) {
      if (p < (sd ? n : m)) {
        const float* pts = sd ? y : x;
        if (DP > 0) {
#pragma unroll
          for (int k = 0; k < (DP > 0 ? DP : 1); ++k) {
            const float v = k < d ? pts[(size_t)p * d + k] : 0.f;
            if (!isfinite(v)) bad |= 1u << sd;
            (sd ? ys : xs)[p * DP + k] = v;
          }
        }
        const double wv = (sd ? b : a)[p];
        if (!isfinite(wv)) bad |= 1u << sd;
        else if (wv < 0.0) bad |= 4u << sd;
        (sd ? S.cres : S.sres)[p] = wv;
        (sd ? S.jidx : S.iidx)[p] = p;
        add[sd] = isfinite(wv) && wv > 0.0 ? wv : 0.0;
      }
    }
    xs_add_warp(S.acc, add[0]);
    xs_add_warp(S.acc2(), add[1]);
  }
  if (DP == 0) {
    // rows checked by the whole CTA, consecutive lanes on consecutive values
#pragma unroll 1
    for (int sd = 0; sd < 2; ++sd) {
      const float* pts = sd ? y : x;
      const int cnt = (sd ? n : m) * d;  // (at most 2,048 rows of 65,536)
      int i0 = 0;
      if ((reinterpret_cast<uintptr_t>(pts) & 15) == 0) {
        // 16 bytes a load, four in flight
        const float4* p4 = reinterpret_cast<const float4*>(pts);
        const int c4 = cnt >> 2;
        bool nf = false;
        for (int i = tid; i < c4; i += 4 * blockDim.x) {
          float4 v[4];
#pragma unroll
          for (int u = 0; u < 4; ++u) v[u] = p4[min(i + u * (int)blockDim.x, c4 - 1)];
#pragma unroll
          for (int u = 0; u < 4; ++u)
            nf |= !(isfinite(v[u].x) && isfinite(v[u].y) && isfinite(v[u].z) && isfinite(v[u].w));
        }
        if (nf) bad |= 1u << sd;
        i0 = c4 << 2;
      }
      for (int i = i0 + tid; i < cnt; i += blockDim.x)
        if (!isfinite(pts[i])) bad |= 1u << sd;
    }
  }
  unsigned all = 0;
#pragma unroll
  for (int k = 0; k < 4; ++k) all |= __syncthreads_or((bad >> k) & 1u) ? 1u << k : 0u;
  if (tid < 64) {
    const double t = xs_round_warp(tid < 32 ? S.acc : S.acc2());
    if ((tid & 31) == 0) S.total[tid >> 5] = t;
  }
  __syncthreads();
  const double ta = S.total[0], tb = S.total[1];
  // the first side's error is reported before the second side's
  const bool ex = (all & 5u) || !(ta > 0.0), ey = (all & 10u) || !(tb > 0.0);
  if (ex || ey) {
    const unsigned e = ex ? all : all >> 1;
    if (tid == 0) atomicOr(err, (e & 1u) ? EF_NONFINITE : ((e & 4u) ? EF_NEGATIVE : EF_ZERO_MASS));
    __syncthreads();
    return false;
  }
  for (int p = tid; p < m; p += blockDim.x) S.sres[p] = __ddiv_rn(S.sres[p], ta);
  for (int p = tid; p < n; p += blockDim.x) S.cres[p] = __ddiv_rn(S.cres[p], tb);
  for (int i = tid; i < XS_LIMBS; i += blockDim.x) S.acc[i] = 0ULL;
  __syncthreads();
  return true;
}

// Shared memory of a one-CTA solver for d <= 8 (coordinates included).
template <int D, int DP, bool L1, int CAP = FIN_MAX, int NT = FIN_THREADS>
struct LowdSmem {
  CtaCore<CAP> S;
  GeoSmem<D, DP, L1, CAP, NT> G;
};

// Whole pair in one CTA: load both sides, drop zero weights, run all rounds,
// return R (correctly rounded) in thread 0.  Returns false on invalid input.
template <int CAP, class Geo>
NNS_DEV bool cta_solve_pair(CtaCore<CAP>& S, Geo& G, float* xs, float* ys, const float* x, const double* a, int m,
                            const float* y, const double* b, int n, int d, int metric, unsigned* err, double& cost,
                            long long& rounds, long long& pe, int protocol = 0, unsigned long long seed = 0,
                            int32_t* fl_i = nullptr, int32_t* fl_j = nullptr, double* fl_f = nullptr,
                            long long fl_cap = 0) {
  if (!cta_load_sides<Geo::kDP, CAP>(x, a, m, y, b, n, d, xs, ys, S, err)) return false;
  if (threadIdx.x == 0) {
    S.mt = m;
    S.nt = n;
  }
  __syncthreads();
  cta_compact(S, G);  // drop zero weights
  CtaOut O{S.acc, nullptr, nullptr, nullptr, 0, nullptr, nullptr, err};
  O.protocol = protocol;
  O.seed = seed;
  if (fl_i) {
    // record the flows and cost them all after the last round (the FP64
    // distance is then computed once per flow with the lanes in parallel,
    // not on every round's critical path)
    O.fl_i = fl_i;
    O.fl_j = fl_j;
    O.fl_f = fl_f;
    O.fl_cap = fl_cap;
    O.x = x;
    O.y = y;
    O.d = d;
  }
  unsigned long long nnz = 0;
  rounds = 0;
  pe = 0;
  cta_rounds(S, G, metric, O, nnz, rounds, pe, (long long)m + n);
  __syncthreads();
  if (threadIdx.x < 32) cost = xs_round_warp(S.acc);  // (thread 0 has it)
  return true;
}

}  // namespace nnsemd
