// Batched reduced-precision NNS-EMD (d > 8): one persistent launch, one pair
// per CTA, all rounds of Alg. 1 (Sec. III-A) on chip (Sec. III-D batch
// processing), with the NNS operation of every round on the tensor cores.
//
// Per round the CTA
//   1. packs its pair's active points (BF16 / FP16 / FP8 with per-row scale)
//      into its own slot of a global scratch area, in the K-major no-swizzle
//      core-matrix layout, with FP32 norms and the certificate's maxima;
//   2. runs a tcgen05 pipeline over (consumer tile of 128) x (supplier tile
//      of BN): warp 0 issues the bulk copies (TMA), warp 1 owns tensor memory
//      and issues the MMAs into two FP32 accumulators, warps 2..5 keep the
//      top-8 approximate suppliers of each consumer; the pipeline's phase
//      counters live for the whole launch;
//   3. re-ranks the 8 candidates of every consumer with the exact FP32 key
//      (all 32 warps) and certifies the best (tc_common.cuh); consumers that
//      cannot be certified are scanned again in FP32 (64 x 64 tiles);
//   4. groups, serves, retires and compacts exactly as the other one-CTA
//      solvers (cta.cuh).
// A pair whose m * n values fit the CTA's distance cache runs 1 and 2 in its
// first round alone and answers every round from candidate lists
// (GeoTC::nns_lists).
// The result equals the FP32 path's.  All waits are bounded (EF_TIMEOUT).
#include <math_constants.h>

#include "common.cuh"
#include "cta.cuh"
#include "kernels.h"
#include "tc_common.cuh"

namespace nnsemd {

// Candidates per consumer in the batched kernel's pass without the distance
// cache (its 1,024 threads have 64 registers each; the multi-CTA kernel keeps
// TC_K = 16).
constexpr int BTC_K = 8;
constexpr int BTC_FILL_WARPS = 16;  // epilogue warps while the distance cache fills (from warp 4 on)

// Per-CTA scratch in global memory.
struct BtcScratch {
  uint8_t* A;       // consumer tiles
  uint8_t* B;       // supplier tiles
  float* nrm_x;
  float* nrm_sx;    // |x| rounded up (0 on padding)
  float* scale_x;
  float* nrm_y;
  float* scale_y;
  float* cand_v;    // [cap][BTC_K]
  int* cand_p;
  // distance cache of a pair that fits kc_cap values (see GeoTC::nns_lists), by
  // the positions j, i of consumer and supplier in the pair's first round:
  // approximate ranking values v' of the tensor-core pass, [j / 32][i / 4][j %
  // 32][i % 4] (a warp of 32 consumers writes four columns as 512 contiguous
  // bytes), and the minimum of each 16 suppliers, [j / 32][i / 16][j % 32]; and
  // those positions by original index, the suppliers' and (from cap on) the
  // consumers' (unset where every point has weight: the original index itself)
  float* vcache;
  float* vmin;
  int* pos;
  // candidate lists by original consumer: (exact key bits << 32 | original
  // supplier) ascending, the next entry to look at | length << 8, and the
  // value a key must stay below to be the nearest (certify_floor)
  unsigned long long* list;
  int* lnext;
  double* lfloor;
  float* ny_o;      // per original consumer: FP32 squared norm, scale, FP64 |y|_2^2 and |y|_1
  float* sy_o;
  double* yl2_o;
  double* yl1_o;
  double* e_o;      // per original consumer: E of the certificate (certify_E); 0: its cache row holds exact keys
};

// Values of a pair's distance cache (rows padded to whole warps, columns to
// whole vectors, at least 16).
__host__ __device__ inline long long btc_cache_values(long long m, long long n) {
  return (kmat_ld(m) < 16 ? 16 : kmat_ld(m)) * ((n + 31) & ~31LL);
}
long long batched_tc_cache_values(long long m, long long n) { return btc_cache_values(m, n); }

__host__ __device__ inline size_t btc_slot_layout(uint8_t* base, int cap, int kb, int bn, BtcScratch* out,
                                                  long long kc_cap = 0) {
  size_t off = 0;
  auto take = [&](size_t bytes) {
    off = (off + 255) & ~(size_t)255;
    uint8_t* p = base ? base + off : nullptr;
    off += bytes;
    return p;
  };
  const int qrows = (cap + TC_BM - 1) / TC_BM * TC_BM;
  const int srows = (cap + bn - 1) / bn * bn;
  BtcScratch s;
  s.A = take((size_t)qrows * kb);
  s.B = take((size_t)srows * kb);
  s.nrm_x = (float*)take(srows * sizeof(float));
  s.nrm_sx = (float*)take(srows * sizeof(float));
  s.scale_x = (float*)take(srows * sizeof(float));
  s.nrm_y = (float*)take(qrows * sizeof(float));
  s.scale_y = (float*)take(qrows * sizeof(float));
  s.cand_v = (float*)take((size_t)cap * BTC_K * sizeof(float));
  s.cand_p = (int*)take((size_t)cap * BTC_K * sizeof(int));
  s.vcache = (float*)take((size_t)kc_cap * sizeof(float));
  s.vmin = (float*)take((size_t)(kc_cap / 8) * sizeof(float));  // (kc_ld / 16 rounded up is at most kc_ld / 8 from 16 columns on)
  s.pos = (int*)take(kc_cap ? 2 * (size_t)cap * sizeof(int) : 0);
  s.list = (unsigned long long*)take(kc_cap ? (size_t)cap * BTC_K * sizeof(unsigned long long) : 0);
  s.lnext = (int*)take(kc_cap ? (size_t)cap * sizeof(int) : 0);
  s.lfloor = (double*)take(kc_cap ? (size_t)cap * sizeof(double) : 0);
  s.ny_o = (float*)take(kc_cap ? (size_t)cap * sizeof(float) : 0);
  s.sy_o = (float*)take(kc_cap ? (size_t)cap * sizeof(float) : 0);
  s.yl2_o = (double*)take(kc_cap ? (size_t)cap * sizeof(double) : 0);
  s.yl1_o = (double*)take(kc_cap ? (size_t)cap * sizeof(double) : 0);
  s.e_o = (double*)take(kc_cap ? (size_t)cap * sizeof(double) : 0);
  if (out) *out = s;
  return (off + 255) & ~(size_t)255;
}

size_t batched_tc_slot_bytes(int cap, int kb, int bn, long long kc_cap) {
  return btc_slot_layout(nullptr, cap, kb, bn, nullptr, kc_cap);
}

struct BtcArgs {
  BatchArgs base;
  uint8_t* scratch;          // grid x slot_bytes
  size_t slot_bytes;
  int kb, bn, nstage, fmt;
  unsigned long long* certified;
  unsigned long long* fallbacks;
  unsigned long long* near_ties;
  int rk;                    // candidates re-ranked per consumer (1 .. BTC_K)
  long long kc_cap;          // distance-cache entries per CTA (0: no cache)
};

// The NNS policy of the batched tensor-core solver (coordinates in global
// memory, index-only active lists, like GeoGlobal).
template <bool KIND8, int CAP>
struct GeoTC {
  static constexpr int kDP = 0;
  static constexpr int kThreads = FIN_THREADS;
  // (a list is a warp's work of 20 us and more: the last rounds of a pair make
  // theirs in 32 warps rather than in team_rounds' four)
  static constexpr bool kTeamRounds = false;
  static constexpr int SEL_BUF = 128;  // words a warp's selection collects at most
  struct PX {};
  const float* x;  // this pair's coordinates
  const float* y;
  int d;
  BtcScratch scr;
  int kb, bn, nstage, fmt, rk;
  uint32_t tmem_base;
  unsigned* err;
  uint64_t bar_full[8];
  uint64_t bar_empty[8];
  uint64_t bar_acc_full[2];
  uint64_t bar_acc_empty[2];
  // the same for passes that fill the distance cache (BTC_FILL_WARPS
  // epilogue warps, one arrival each)
  uint64_t bar_accf_full[2];
  uint64_t bar_accf_empty[2];
  uint64_t bar_a_full;
  uint64_t bar_a_empty;
  // pipeline counters: prod_* only by the producer thread, mma_* only by the
  // MMA thread; epi_acc is read by the epilogue threads at the start of a
  // phase and advanced by one thread after it
  unsigned prod_a, prod_b, mma_a, mma_b, mma_acc, epi_acc, mma_accf, epi_accf;
  unsigned stat_rx, stat_rx1, stat_sx;  // certificate maxima of this round (float bits)
  int nfb, nscan;
  unsigned long long ncert, nfall, nnear;
  // distance cache of the current pair: on (m * n fits), filled (after the
  // pair's first round), the active suppliers of that round and its row length,
  // whether every point was active then (positions are original indices)
  int kc_on, kc_ready, kc_m, kc_ld, kc_dense;
  int pair_m, pair_n;  // the pair's points
  double kc_gam;  // gamma_d of the certificate
  int fb[CAP];
  // staging: tensor-core operand tiles or FP32 fallback tiles (never both at
  // once); the launch reserves max(sizeof(tiles), A + stages * B) bytes
  union __align__(128) Stage {
    TileSmem tiles[FIN_THREADS / TG_THREADS];
    unsigned long long sel[FIN_THREADS / 32 * SEL_BUF];  // make_lists
    uint8_t bytes[16];
  } U;

  NNS_DEV void load_x(int, PX&) const {}
  NNS_DEV void store_x(int, const PX&) {}
  NNS_DEV void load_y(int, PX&) const {}
  NNS_DEV void store_y(int, const PX&) {}
  template <int C>
  NNS_DEV double dist64(const CtaCore<C>& S, int p, int q, int metric) const {
    return cost_dist64(x + (size_t)S.iidx[p] * d, y + (size_t)S.jidx[q] * d, d, metric);
  }

  // The NNS step of a round from the pair's distance cache (the tensor-core
  // pass of its first round filled every v').  Active suppliers only ever
  // leave, so a consumer keeps a list of the rk active suppliers with the
  // smallest v' at the time it was made, ordered by exact FP32 key, and walks
  // it from round to round: its first entry that is still active is the
  // nearest active supplier as long as its key is below the list's
  // certificate bound (every supplier outside the list has v' >= tau, the
  // list's largest).  A consumer whose list runs out, or whose next entry the
  // bound does not certify, makes a new one from the suppliers active now
  // (a warp makes up to four at a time):
  //   1. the rk smallest v' (ties by position), their exact FP32 keys, one
  //      per lane in the definition's sequential order, ordered by (key,
  //      original index: positions keep that order);
  //   2. the certificate of the first against tau, with the first round's
  //      supplier maxima (a superset of every later round's); with no other
  //      active supplier every entry is the answer in its turn;
  //   3. not certified: the FP32 tiles over every active supplier, for all
  //      such consumers of the round together.  Their exact keys take the place
  //      of v' in the cache (E = 0 says so), where a later selection by (key,
  //      position) needs no certificate.
  // A consumer takes about two searches, so 8 entries serve it; 32 cost more
  // in exact keys (each lane walks its own row) than they saved.  1,000
  // retrieval pairs (256..2,048 points, d = 128, FP16): 43.5 ms with the
  // candidates selected anew in every round, 16.1 ms so.
  //
  // S.off holds, by original index, the position of each active supplier
  // (free until the round's grouping); a stale entry fails its check.
  template <int C>
  NNS_DEV void map_positions(CtaCore<C>& S, int mt, int first, int step) const {
    for (int p = first; p < mt; p += step) S.off[S.iidx[p]] = p;
  }
  // One consumer from its list: true and its packed key, or false.
  template <int C>
  NNS_DEV bool serve(const CtaCore<C>& S, int mt, int j, unsigned long long& key) const {
    const int st = scr.lnext[j], end = st >> 8;
    const unsigned long long* l = scr.list + (size_t)j * BTC_K;
    for (int t = st & 0xff; t < end; ++t) {
      const unsigned long long e = l[t];
      const int i = (int)(unsigned)e, p = S.off[i];
      if ((unsigned)p >= (unsigned)mt || S.iidx[p] != i) continue;  // retired
      if (!((double)__uint_as_float((unsigned)(e >> 32)) < scr.lfloor[j])) return false;
      scr.lnext[j] = (st & ~0xff) | t;
      key = (e & 0xffffffff00000000ULL) | (unsigned)p;
      return true;
    }
    return false;
  }
  // cache row of an original consumer, column of an original supplier
  NNS_DEV int row_of(int j) const { return kc_dense ? j : scr.pos[CAP + j]; }
  NNS_DEV int col_of(int i) const { return kc_dense ? i : scr.pos[i]; }
  NNS_DEV size_t v_at(int j, int i) const {
    return ((((size_t)(j >> 5) * (kc_ld >> 2)) + (i >> 2)) * 32 + (j & 31)) * 4 + (i & 3);
  }
  // The 8 smallest of the warp's words v (four a lane, ~0 for none), in order
  // in lanes 0..7 with their ids: eight minima over the warp, each by one
  // reduction; equal words in the order of v[0] of every lane, v[1], ...
  NNS_DEV void extract8(unsigned (&v)[4], const int (&id)[4], unsigned& rv, int& rid) const {
    const int lane = threadIdx.x & 31;
    rv = 0xffffffffu;
    rid = 0;
#pragma unroll 1
    for (int k = 0; k < 8; ++k) {
      const unsigned mine = min(min(v[0], v[1]), min(v[2], v[3]));
      const unsigned w = __reduce_min_sync(0xffffffffu, mine);
      if (w == 0xffffffffu) break;
      const unsigned u = v[0] == w ? 0u : (v[1] == w ? 1u : (v[2] == w ? 2u : 3u));
      const int src = (int)(__reduce_min_sync(0xffffffffu, mine == w ? 32 * u + lane : 0xffffffffu) & 31u);
      int my = u == 0 ? id[0] : (u == 1 ? id[1] : (u == 2 ? id[2] : id[3]));
      my = __shfl_sync(0xffffffffu, my, src);
      if (lane == src) {
        if (u == 0) v[0] = 0xffffffffu;
        else if (u == 1) v[1] = 0xffffffffu;
        else if (u == 2) v[2] = 0xffffffffu;
        else v[3] = 0xffffffffu;
      }
      if (lane == k) {
        rv = w;
        rid = my;
      }
    }
  }
  // The 8 smallest value(p), p < mt, as extract8 gives them (ids: original
  // indices).  The 8th smallest of the lanes' minima bounds the 8th smallest
  // of all; a second pass collects what does not exceed it (a few more than 8
  // values; where the buffer would overflow the 8 best so far stay).
  template <class C, class Value>
  NNS_DEV void scan8(const C& S, int mt, unsigned long long* buf, unsigned& rv, int& rid, Value value) const {
    const int lane = threadIdx.x & 31;
    const unsigned lt = (1u << lane) - 1u;
    unsigned mn = 0xffffffffu;
#pragma unroll 4
    for (int p = lane; p < mt; p += 32) mn = min(mn, value(p));
    unsigned v[4] = {mn, 0xffffffffu, 0xffffffffu, 0xffffffffu};
    int id[4] = {0, 0, 0, 0};
    extract8(v, id, rv, rid);
    const unsigned thr = __shfl_sync(0xffffffffu, rv, 7);
    int cnt = 0;
    auto take = [&]() {  // the best 8 of the collected ones
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const unsigned long long w = 32 * u + lane < cnt ? buf[32 * u + lane] : ~0ULL;
        v[u] = (unsigned)(w >> 32);
        id[u] = (int)(unsigned)w;
      }
      extract8(v, id, rv, rid);
      __syncwarp();
    };
#pragma unroll 1
    for (int p0 = 0; p0 < mt; p0 += 96) {  // three loads a lane in flight
      unsigned w[3], bal[3];
#pragma unroll
      for (int u = 0; u < 3; ++u) {
        const int p = p0 + 32 * u + lane;
        w[u] = p < mt ? value(p) : 0xffffffffu;
      }
#pragma unroll
      for (int u = 0; u < 3; ++u) bal[u] = __ballot_sync(0xffffffffu, p0 + 32 * u + lane < mt && w[u] <= thr);
      const int add = __popc(bal[0]) + __popc(bal[1]) + __popc(bal[2]);
      if (!add) continue;
      if (cnt + add > SEL_BUF) {
        take();
        cnt = 8;
        if (lane < 8) buf[lane] = ((unsigned long long)rv << 32) | (unsigned)rid;
        __syncwarp();
      }
#pragma unroll
      for (int u = 0; u < 3; ++u) {
        if ((bal[u] >> lane) & 1u)
          buf[cnt + __popc(bal[u] & lt)] = ((unsigned long long)w[u] << 32) | (unsigned)S.iidx[p0 + 32 * u + lane];
        cnt += __popc(bal[u]);
      }
      __syncwarp();
    }
    take();
  }
  // The same for v' of cache row j while every supplier of the first round is
  // active (ids: positions): each of the 8 smallest lies in one of the 8 groups of
  // 16 with the smallest minima.
  NNS_DEV void groups8(int j, unsigned& rv, int& rid) const {
    const int lane = threadIdx.x & 31;
    const int nb = (kc_ld + 15) >> 4;  // at most 128
    const float* mrow = scr.vmin + (size_t)(j >> 5) * nb * 32 + (j & 31);
    unsigned v[4];
    int id[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int b = 32 * u + lane;
      v[u] = b < nb ? ordered_bits(mrow[(size_t)b * 32]) : 0xffffffffu;
      id[u] = b;
    }
    extract8(v, id, rv, rid);
    // four lanes a group, four values a lane
    const int b = __shfl_sync(0xffffffffu, rid, lane >> 2);
    const bool on = __shfl_sync(0xffffffffu, rv, lane >> 2) != 0xffffffffu;
    const int i0 = 16 * b + 4 * (lane & 3);
    float4 f = make_float4(0.f, 0.f, 0.f, 0.f);
    if (on && i0 < kc_ld) f = *reinterpret_cast<const float4*>(scr.vcache + v_at(j, i0));
    const float e[4] = {f.x, f.y, f.z, f.w};
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      id[u] = i0 + u;
      v[u] = on && i0 + u < kc_m ? ordered_bits(e[u]) : 0xffffffffu;
    }
    extract8(v, id, rv, rid);
  }
  // Key of original supplier i against consumer row yrow (16 bytes at a time
  // where the rows allow it: the same chain).
  NNS_DEV float exact_key(int i, const float* yrow, bool vec) const {
    return vec ? key32_sql2_v4(x + (size_t)i * d, yrow, d) : key32<METRIC_SQL2>(x + (size_t)i * d, yrow, d);
  }
  // New lists for up to four consumers (one warp; cnt of them, positions
  // qs(0..cnt)): eight lanes a consumer.  Stores their packed keys in S.nnk.
  template <int C, class Qs>
  NNS_DEV void make_lists(CtaCore<C>& S, int mt, int cnt, Qs qs) {
    const int lane = threadIdx.x & 31, g = lane >> 3, sub = lane & 7;
    unsigned long long* buf = U.sel + (threadIdx.x >> 5) * SEL_BUF;
    const bool vec = (d & 3) == 0 && ((reinterpret_cast<uintptr_t>(x) | reinterpret_cast<uintptr_t>(y)) & 15) == 0;
    const int len = min(rk, mt);
    // 1.
    unsigned cv = 0xffffffffu;  // this lane's candidate: v' and original index
    int i = 0;
#pragma unroll 1
    for (int h = 0; h < cnt; ++h) {
      const int jj = row_of(S.jidx[qs(h)]);
      unsigned rv;
      int rid;
      if (mt == kc_m && scr.e_o[S.jidx[qs(h)]] != 0.0) {
        groups8(jj, rv, rid);
        rid = S.iidx[rid];
      } else {
        scan8(S, mt, buf, rv, rid, [&](int p) { return ordered_bits(scr.vcache[v_at(jj, col_of(S.iidx[p]))]); });
      }
      rv = __shfl_sync(0xffffffffu, rv, sub);
      rid = __shfl_sync(0xffffffffu, rid, sub);
      if (g == h) {
        cv = rv;
        i = rid;
      }
    }
    const int q = qs(min(g, cnt - 1)), j = S.jidx[q];
    const float* yrow = y + (size_t)j * d;
    // (a supplier whose norm overflows has v' = NaN, which orders like the word
    // for none: it may be missing here, so its consumers go to 3.)
    const bool wanted = g < cnt && sub < len, on = wanted && cv != 0xffffffffu;
    if (!on) i = 0;
    const unsigned long long e = on ? pack_key(exact_key(i, yrow, vec), (unsigned)i) : ~0ULL;
    const int first = __shfl_sync(0xffffffffu, i, lane & 24);  // the approximate choice
    int rank = 0;
    unsigned long long best = ~0ULL;
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      const unsigned long long o = __shfl_sync(0xffffffffu, e, (lane & 24) + u);
      rank += o < e;
      best = o < best ? o : best;
    }
    // 2.
    const unsigned tb = __shfl_sync(0xffffffffu, cv, (lane & 24) + len - 1);
    double fl = CUDART_INF;
    bool bad = ((__ballot_sync(0xffffffffu, wanted && !on) >> (lane & 24)) & 0xffu) != 0;
    if (g < cnt && mt > len && scr.e_o[j] != 0.0) {
      const float tau = __uint_as_float((tb & 0x80000000u) ? (tb & 0x7fffffffu) : ~tb);
      fl = certify_floor_from_E(scr.ny_o[j], tau, scr.e_o[j], kc_gam);
      bad |= !((double)__uint_as_float((unsigned)(best >> 32)) < fl);
    }
    if (on && !bad) scr.list[(size_t)j * BTC_K + rank] = e;
    if (g < cnt && sub == 0 && !bad) {
      scr.lnext[j] = len << 8;
      scr.lfloor[j] = fl;
      S.nnk[q] = (best & 0xffffffff00000000ULL) | (unsigned)S.off[(int)(unsigned)best];
      atomicAdd(&ncert, 1ULL);
      if ((int)(unsigned)best != first) atomicAdd(&nnear, 1ULL);
    }
    // 3. left to the FP32 tiles
    if (g < cnt && sub == 0 && bad) {
      scr.lnext[j] = 0;
      const int k = atomicAdd(&nscan, 1);
      scan_list(S)[k] = q;
      scan_first(S)[k] = first;
    }
    __syncwarp();
  }
  // Consumers for the FP32 tiles and their approximate choices (S.mem and
  // S.mem2 are free during the NNS step).
  template <int C>
  NNS_DEV int* scan_list(CtaCore<C>& S) const { return reinterpret_cast<int*>(S.mem); }
  template <int C>
  NNS_DEV int* scan_first(CtaCore<C>& S) const { return reinterpret_cast<int*>(S.mem2); }
  // The FP32 tiles over every active supplier for n consumers of a list; KEEP:
  // their keys replace v' in the cache.  Up to 128 consumers leave groups
  // without a tile: those share the suppliers, and the parts merge by atomicMin.
  template <bool KEEP, int C>
  __device__ __noinline__ void scan_exact(CtaCore<C>& S, int mt, const int* list, int n) {
    const int g = threadIdx.x / TG_THREADS, gt = threadIdx.x % TG_THREADS;
    const int tx = gt & 15, ty = gt >> 4;
    constexpr int ngroups = kThreads / TG_THREADS;
    const int ct = (n + TG_M - 1) / TG_M, parts = max(1, ngroups / ct);
    if (parts > 1) {
      for (int k = threadIdx.x; k < n; k += kThreads) S.nnk[list[k]] = ~0ULL;
      __syncthreads();
    }
    for (int it = g; it < ct * parts; it += ngroups) {
      const int c0 = (it % ct) * TG_M, part = it / ct;
      const int p0 = mt * part / parts, p1 = mt * (part + 1) / parts;
      unsigned long long out[4];
      group_nns_tile<false>(x, S.iidx, p0, p1, y, S.jidx, list, c0, min(TG_M, n - c0), d, U.tiles[g], gt, 1 + g, out,
                            [&](int pt, const unsigned long long (&acc)[2][4]) {
                              if (!KEEP) return;
#pragma unroll 1
                              for (int i = 0; i < 4 && c0 + ty * 4 + i < n; ++i) {
                                const int r = row_of(S.jidx[list[c0 + ty * 4 + i]]);
#pragma unroll
                                for (int j = 0; j < 4; ++j) {
                                  const unsigned long long a = i < 2 ? acc[0][j] : acc[1][j];
                                  const int p = pt + tx * 4 + j;
                                  if (p < p1) scr.vcache[v_at(r, col_of(S.iidx[p]))] = (i & 1) ? f2_hi(a) : f2_lo(a);
                                }
                              }
                            });
      if (tx == 0)
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const int lq = c0 + ty * 4 + i;
          if (lq >= n) break;
          if (parts > 1) atomicMin(&S.nnk[list[lq]], out[i]);
          else S.nnk[list[lq]] = out[i];
        }
    }
  }
  template <int C>
  NNS_DEV const unsigned long long* nns_lists(CtaCore<C>& S, int mt, int nt) {
    const int tid = threadIdx.x;
    map_positions(S, mt, tid, kThreads);
    if (tid == 0) nfb = nscan = 0;
    __syncthreads();
    int cert = 0;
    for (int q = tid; q < nt; q += kThreads) {
      unsigned long long key;
      if (serve(S, mt, S.jidx[q], key)) {
        S.nnk[q] = key;
        ++cert;
      } else {
        fb[atomicAdd(&nfb, 1)] = q;
      }
    }
    __syncwarp();
    cert = __reduce_add_sync(0xffffffffu, cert);
    if ((tid & 31) == 0 && cert) atomicAdd(&ncert, (unsigned long long)cert);
    __syncthreads();
    const int n = nfb;
    // (a warp makes its lists one after the other: as few each as the warps allow)
    const int per = min(4, (n + kThreads / 32 - 1) / (kThreads / 32));
#pragma unroll 1
    for (int k = per * (tid >> 5); k < n; k += per * (kThreads / 32))
      make_lists(S, mt, min(per, n - k), [&](int h) { return fb[k + h]; });
    __syncthreads();
    const int ns = nscan;
    if (ns > 0) {
      scan_exact<true>(S, mt, scan_list(S), ns);
      __syncthreads();
      for (int k = tid; k < ns; k += kThreads) {
        const int q = scan_list(S)[k], j = S.jidx[q];
        if (S.iidx[(int)(unsigned)S.nnk[q]] != scan_first(S)[k]) atomicAdd(&nnear, 1ULL);
        scr.ny_o[j] = 0.f;  // |x - y|^2 itself is in the cache
        scr.e_o[j] = 0.0;
      }
      if (tid == 0) nfall += ns;
      __syncthreads();
    }
    return S.nnk;
  }
  template <int C>
  NNS_DEV const unsigned long long* nns(CtaCore<C>& S, int mt, int nt, long long = 0) {
    if (kc_on && kc_ready) return nns_lists(S, mt, nt);
    // with the cache on, this is the pair's first round: the tensor-core
    // pass fills the cache (every v' of the pair) instead of keeping top-K
    const bool fill = kc_on != 0;
    const int tid = threadIdx.x, T = blockDim.x;
    const int warp = tid >> 5, lane = tid & 31;
    const int qtiles = (nt + TC_BM - 1) / TC_BM;
    const int stiles = (mt + bn - 1) / bn;
    const int nblk = kb / 16;
    // ---- 1. pack both sides
    if (tid == 0) {
      stat_rx = stat_rx1 = stat_sx = 0u;
      nfb = 0;
    }
    if (fill) {
      // the cache's rows and columns are this round's positions
      const bool dense = mt == pair_m && nt == pair_n;
      if (tid == 0) {
        kc_m = mt;
        kc_ld = mt < 16 ? 16 : (int)kmat_ld(mt);
        kc_dense = dense;
      }
      for (int q = tid; q < nt; q += T) scr.lnext[S.jidx[q]] = 0;  // no lists yet
      if (!dense) {
        for (int p = tid; p < mt; p += T) scr.pos[S.iidx[p]] = p;
        for (int q = tid; q < nt; q += T) scr.pos[CAP + S.jidx[q]] = q;
      }
    }
    __syncthreads();
    {
      // one warp per row: the lanes take the row's coordinates and 16-byte
      // blocks (coalesced loads, all in flight at once), and the scale and
      // norms are warp reductions.  Any summation order keeps the FP32
      // squared norm within gamma_d |v|^2, the bound the certificate uses.
      const int srows = stiles * bn, qrows = qtiles * TC_BM;
      const int total = srows + qrows;
      // two rows of a warp at once (their loads overlap)
#pragma unroll 1
      for (int row0 = 2 * warp; row0 < total; row0 += 2 * (T / 32)) {
        const float* rows2[2];
        float mx[2] = {0.f, 0.f}, a2f[2] = {0.f, 0.f}, a1f[2] = {0.f, 0.f};
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const int row_id = row0 + h;
          const bool sup = row_id < srows;
          const int p = sup ? row_id : row_id - srows;
          rows2[h] = nullptr;
          if (row_id < total && p < (sup ? mt : nt)) rows2[h] = (sup ? x : y) + (size_t)(sup ? S.iidx[p] : S.jidx[p]) * d;
        }
        for (int k = lane; k < d; k += 32) {
          float v[2];
#pragma unroll
          for (int h = 0; h < 2; ++h) v[h] = rows2[h] ? rows2[h][k] : 0.f;
#pragma unroll
          for (int h = 0; h < 2; ++h) {
            mx[h] = fmaxf(mx[h], fabsf(v[h]));
            a2f[h] = __fmaf_rn(v[h], v[h], a2f[h]);
            a1f[h] = __fadd_rn(a1f[h], fabsf(v[h]));
          }
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1)
#pragma unroll
          for (int h = 0; h < 2; ++h) {
            mx[h] = fmaxf(mx[h], __shfl_xor_sync(0xffffffffu, mx[h], o));
            a2f[h] = __fadd_rn(a2f[h], __shfl_xor_sync(0xffffffffu, a2f[h], o));
            a1f[h] = __fadd_rn(a1f[h], __shfl_xor_sync(0xffffffffu, a1f[h], o));
          }
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const int row_id = row0 + h;
          if (row_id >= total) break;
          const bool sup = row_id < srows;
          const int p = sup ? row_id : row_id - srows;
          const float* row = rows2[h];
          const float s = row ? scale_of_max(mx[h], fmt) : 1.f;
          const int rows = sup ? bn : TC_BM;
          uint8_t* tile = (sup ? scr.B : scr.A) + (size_t)(p / rows) * rows * kb;
          for (int c = lane; c < nblk; c += 32) pack_block(row, d, c, s, fmt, tile, rows, p % rows, sup);
          if (lane == 0) {
            float* nrm = sup ? scr.nrm_x : scr.nrm_y;
            float* scl = sup ? scr.scale_x : scr.scale_y;
            if (row) {
              const float l2sq = a2f[h], l1 = a1f[h];
              nrm[p] = l2sq;
              scl[p] = s;
              if (sup) {
                scr.nrm_sx[p] = norm_up(l2sq);
                atomicMax(&stat_rx, __float_as_uint(norm_up(l2sq)));
                atomicMax(&stat_rx1, __float_as_uint(l1 * (1.f + 1e-4f)));
                atomicMax(&stat_sx, __float_as_uint(s));
              } else if (fill) {
                // what the certificate needs of this consumer in every round
                const int j = S.jidx[p];
                scr.ny_o[j] = l2sq;
                scr.sy_o[j] = s;
              }
            } else {
              nrm[p] = CUDART_INF_F;
              scl[p] = 1.f;
              if (sup) scr.nrm_sx[p] = 0.f;
            }
          }
        }
      }
    }
    fence_proxy_async_global();                                   // packed tiles -> later bulk copies
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");  // last round's FP32 tiles -> bulk writes
    __syncthreads();
    // ---- 2. tensor-core pipeline
    const uint32_t a_bytes = TC_BM * kb, b_bytes = bn * kb;
    uint8_t* sA = U.bytes;
    uint8_t* sB = U.bytes + a_bytes;
    bool ok = true;
    if (warp == 0) {
      if (lane == 0) {
        for (int qt = 0; qt < qtiles && ok; ++qt) {
          ok = mbar_wait_bounded(&bar_a_empty, (prod_a & 1) ^ 1);
          if (!ok) break;
          mbar_expect_tx(&bar_a_full, a_bytes);
          tma_load_1d(sA, scr.A + (size_t)qt * a_bytes, a_bytes, &bar_a_full);
          ++prod_a;
          for (int st = 0; st < stiles && ok; ++st) {
            const unsigned s = prod_b % nstage, u = prod_b / nstage;
            ok = mbar_wait_bounded(&bar_empty[s], (u & 1) ^ 1);
            if (!ok) break;
            mbar_expect_tx(&bar_full[s], b_bytes);
            tma_load_1d(sB + (size_t)s * b_bytes, scr.B + (size_t)st * b_bytes, b_bytes, &bar_full[s]);
            ++prod_b;
          }
        }
      }
    } else if (warp == 1) {
      if (lane == 0) {
        const uint32_t idesc = make_idesc(fmt_is_bf16(fmt) ? 1 : 0, TC_BM, bn);
        const int ksteps = kb / 32;
        const uint32_t a0 = smem_u32(sA);
        for (int qt = 0; qt < qtiles && ok; ++qt) {
          ok = mbar_wait_bounded(&bar_a_full, mma_a & 1);
          if (!ok) break;
          for (int st = 0; st < stiles && ok; ++st) {
            const unsigned s = mma_b % nstage, u = mma_b / nstage;
            unsigned& na = fill ? mma_accf : mma_acc;
            const unsigned b = na & 1, v = na >> 1;
            ok = mbar_wait_bounded(&bar_full[s], u & 1);
            if (ok) ok = mbar_wait_bounded(fill ? &bar_accf_empty[b] : &bar_acc_empty[b], (v & 1) ^ 1);
            if (!ok) break;
            tc_fence_after();
            const uint32_t b0 = smem_u32(sB + (size_t)s * b_bytes);
            const uint32_t tmem_d = tmem_base + b * (uint32_t)bn;
            for (int k = 0; k < ksteps; ++k) {
              const uint64_t ad = make_desc(a0 + k * 2 * TC_BM * 16, TC_BM * 16, 128);
              const uint64_t bd = make_desc(b0 + k * 2 * bn * 16, bn * 16, 128);
              mma_issue<KIND8 ? FMT_E4M3 : FMT_BF16>(tmem_d, ad, bd, idesc, k > 0 ? 1u : 0u);
            }
            mma_commit(&bar_empty[s]);
            mma_commit(fill ? &bar_accf_full[b] : &bar_acc_full[b]);
            ++mma_b;
            ++na;
          }
          mma_commit(&bar_a_empty);  // A may be overwritten once these MMAs are done
          ++mma_a;
        }
      }
    } else if (fill) {
      // Cache fill: four warps per TMEM lane quarter, each a share of the
      // tile's columns; a thread holds one consumer's 16 columns and writes
      // them as four 16-byte stores, contiguous over the warp, and their
      // minimum.  (Four warps, each value stored by itself: 39,000 cycles a
      // tile of 128 x 128.)  Meanwhile the other warps, and these when they are
      // done, sum the consumers' FP64 norms for the certificate (an FP64 instruction
      // takes 16 cycles a warp: beside the packing's loads they were half of the
      // packing).
      if (warp >= 4 && warp < 4 + BTC_FILL_WARPS) {
        const int quarter = warp & 3, part = (warp - 4) >> 2;
        const int row = quarter * 32 + lane;
        unsigned ea = epi_accf;
        for (int qt = 0; qt < qtiles; ++qt) {
          const int q = qt * TC_BM + row;
          const float sy = q < nt ? scr.scale_y[q] : 1.f;
          const float cy = quant_coeff(fmt, q < nt ? scr.nrm_y[q] : 0.f);
          float4* vrow = reinterpret_cast<float4*>(scr.vcache + v_at(q, 0));  // column group c at vrow[32 c]
          float* mrow = scr.vmin + (size_t)(q >> 5) * ((kc_ld + 15) >> 4) * 32 + (q & 31);
          const bool live = (q & ~31) < nt;  // (a warp's 32 rows are written whole)
          for (int st = 0; st < stiles; ++st, ++ea) {
            const unsigned b = ea & 1, v = ea >> 1;
            if (ok) ok = mbar_wait_bounded(&bar_accf_full[b], v & 1);
            ok = __all_sync(0xffffffffu, ok);  // warp-uniform: the loads below are warp-wide
            tc_fence_after();
            if (ok)
              for (int c0 = 16 * part; c0 < bn; c0 += 64) {
                uint32_t r[16];
                tmem_ld16(tmem_base + ((uint32_t)(quarter * 32) << 16) + b * (uint32_t)bn + (uint32_t)c0, r);
                const size_t at = (size_t)st * bn + c0;
                float mn = CUDART_INF_F;
#pragma unroll
                for (int e = 0; e < 16; e += 4) {
                  const float4 nx = *reinterpret_cast<const float4*>(scr.nrm_x + at + e);
                  const float4 nsx = *reinterpret_cast<const float4*>(scr.nrm_sx + at + e);
                  float4 w = make_float4(-2.f, -2.f, -2.f, -2.f);
                  if (!fmt_is_bf16(fmt)) {
                    const float4 sx = *reinterpret_cast<const float4*>(scr.scale_x + at + e);
                    w = make_float4(-2.f * sy * sx.x, -2.f * sy * sx.y, -2.f * sy * sx.z, -2.f * sy * sx.w);
                  }
                  float4 o;
                  o.x = __fmaf_rn(-cy, nsx.x, __fmaf_rn(w.x, __uint_as_float(r[e]), nx.x));
                  o.y = __fmaf_rn(-cy, nsx.y, __fmaf_rn(w.y, __uint_as_float(r[e + 1]), nx.y));
                  o.z = __fmaf_rn(-cy, nsx.z, __fmaf_rn(w.z, __uint_as_float(r[e + 2]), nx.z));
                  o.w = __fmaf_rn(-cy, nsx.w, __fmaf_rn(w.w, __uint_as_float(r[e + 3]), nx.w));
                  // (kc_ld is a multiple of 4: the last vector of a row stays inside it)
                  if (live && (int)at + e < kc_ld) vrow[(at + e) * 8] = o;
                  mn = fminf(fminf(mn, o.x), fminf(fminf(o.y, o.z), o.w));
                }
                if (live && (int)at < kc_ld) mrow[(at >> 4) * 32] = mn;
              }
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(&bar_accf_empty[b]);
          }
        }
      }
      // two rows at a time; their four sums share the steps over the lanes
      for (;;) {
        int q = 0;
        if (lane == 0) q = atomicAdd(&nfb, 2);  // (its next use starts from 0)
        q = __shfl_sync(0xffffffffu, q, 0);
        if (q >= nt) break;
        const float* yrow[2];
        double a2[2] = {0.0, 0.0}, a1[2] = {0.0, 0.0};
#pragma unroll
        for (int h = 0; h < 2; ++h) yrow[h] = y + (size_t)S.jidx[min(q + h, nt - 1)] * d;
        for (int k = lane; k < d; k += 32)
#pragma unroll
          for (int h = 0; h < 2; ++h) {
            const double v = yrow[h][k];
            a2[h] += v * v;
            a1[h] += fabs(v);
          }
        // lanes 0..15 take the first row's sums, the others the second's; then
        // the lower eight of each |y|_2^2, the upper |y|_1
        const bool up = (lane & 16) != 0, l1 = (lane & 8) != 0;
        const double s2 = (up ? a2[1] : a2[0]) + __shfl_xor_sync(0xffffffffu, up ? a2[0] : a2[1], 16);
        const double s1 = (up ? a1[1] : a1[0]) + __shfl_xor_sync(0xffffffffu, up ? a1[0] : a1[1], 16);
        double sum = (l1 ? s1 : s2) + __shfl_xor_sync(0xffffffffu, l1 ? s2 : s1, 8);
        for (int o = 4; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
        if ((lane & 7) == 0 && q + (lane >> 4) < nt) {
          const int j = S.jidx[q + (lane >> 4)];
          (l1 ? scr.yl1_o : scr.yl2_o)[j] = sum;
        }
      }
    } else if (warp < 6) {
      const int quarter = warp & 3;
      const int row = quarter * 32 + lane;
      unsigned ea = epi_acc;
      for (int qt = 0; qt < qtiles; ++qt) {
        const int q = qt * TC_BM + row;
        const float sy = q < nt ? scr.scale_y[q] : 1.f;
        const float cy = quant_coeff(fmt, q < nt ? scr.nrm_y[q] : 0.f);
        float tv[BTC_K];
        int tp[BTC_K];
#pragma unroll
        for (int k = 0; k < BTC_K; ++k) { tv[k] = CUDART_INF_F; tp[k] = -1; }
        for (int st = 0; st < stiles; ++st, ++ea) {
          const unsigned b = ea & 1, v = ea >> 1;
          if (ok) ok = mbar_wait_bounded(&bar_acc_full[b], v & 1);
          ok = __all_sync(0xffffffffu, ok);  // warp-uniform: the loads below are warp-wide
          tc_fence_after();
          if (ok) {
            const float* nx = scr.nrm_x + (size_t)st * bn;
            const float* nsx = scr.nrm_sx + (size_t)st * bn;
            const float* sx = scr.scale_x + (size_t)st * bn;
            for (int c0 = 0; c0 < bn; c0 += 16) {
              uint32_t r[16];
              tmem_ld16(tmem_base + ((uint32_t)(quarter * 32) << 16) + b * (uint32_t)bn + (uint32_t)c0, r);
#pragma unroll
              for (int e = 0; e < 16; ++e) {
                const float w = fmt_is_bf16(fmt) ? -2.f : -2.f * sy * sx[c0 + e];
                const float val = __fmaf_rn(-cy, nsx[c0 + e], __fmaf_rn(w, __uint_as_float(r[e]), nx[c0 + e]));
                topk_insert(tv, tp, val, st * bn + c0 + e);
              }
            }
          }
          tc_fence_before();
          mbar_arrive(&bar_acc_empty[b]);
        }
        if (q < nt) {
#pragma unroll
          for (int k = 0; k < BTC_K; ++k) {
            scr.cand_v[(size_t)q * BTC_K + k] = tv[k];
            scr.cand_p[(size_t)q * BTC_K + k] = tp[k];
          }
        }
      }
    }
    if (!ok) atomicOr(err, EF_TIMEOUT);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (tid == 64) (fill ? epi_accf : epi_acc) += (unsigned)(qtiles * stiles);
    if (fill) {
      // the cache holds every v' of the pair; this and every later round
      // are answered from it.  The certificate's E of every consumer, once:
      // the supplier maxima of this first round bound every later round's.
      const double rx = __uint_as_float(stat_rx), rx1 = __uint_as_float(stat_rx1);
      const double sxm = __uint_as_float(stat_sx);
      for (int q = tid; q < nt; q += T) {
        const int j = S.jidx[q];
        scr.e_o[j] = certify_E(fmt, d, scr.ny_o[j], sqrt(scr.yl2_o[j]) * (1 + 1e-12), scr.yl1_o[j], scr.sy_o[j], rx, rx1,
                                sxm);
      }
      if (tid == 0) {
        kc_gam = certify_gamma(d);
        kc_ready = 1;
      }
      __syncthreads();
      return nns_lists(S, mt, nt);
    }
    // ---- 3. exact re-rank + certificate (a warp per consumer)
    const double rx = __uint_as_float(stat_rx), rx1 = __uint_as_float(stat_rx1), sxm = __uint_as_float(stat_sx);
    for (int q = warp; q < nt; q += T / 32) {
      const float* yrow = y + (size_t)S.jidx[q] * d;
      unsigned long long best = ~0ULL;
      int have = 0;  // candidates: all active suppliers where the list is not full, or some are lost to overflow
      if (lane < rk) {
        const int p = scr.cand_p[(size_t)q * BTC_K + lane];
        have = p >= 0;
        if (p >= 0) best = pack_key(key32<METRIC_SQL2>(x + (size_t)S.iidx[p] * d, yrow, d), (unsigned)p);
      }
      have = __reduce_add_sync(0xffffffffu, have);
      double yl2 = 0.0, yl1 = 0.0;
      for (int k = lane; k < d; k += 32) {
        yl2 += (double)yrow[k] * yrow[k];
        yl1 += fabs((double)yrow[k]);
      }
      for (int o = 16; o > 0; o >>= 1) {
        const unsigned long long ob = __shfl_xor_sync(0xffffffffu, best, o);
        best = ob < best ? ob : best;
        yl2 += __shfl_xor_sync(0xffffffffu, yl2, o);
        yl1 += __shfl_xor_sync(0xffffffffu, yl1, o);
      }
      if (lane == 0) {
        // tau: the rk-th approximate value; the first candidate is the
        // approximate best, and an exact best elsewhere is a near-tie
        const float tau = scr.cand_v[(size_t)q * BTC_K + rk - 1];
        if (best != ~0ULL && (int)(unsigned)best != scr.cand_p[(size_t)q * BTC_K]) atomicAdd(&nnear, 1ULL);
        const bool cert = best != ~0ULL && (tau <= 3.402823466e38f || have == mt) &&
                          certify(fmt, d, scr.nrm_y[q], sqrt(yl2) * (1 + 1e-12), yl1, scr.scale_y[q], rx, rx1, sxm, tau,
                                  __uint_as_float((unsigned)(best >> 32)));
        if (cert) {
          S.nnk[q] = best;
          atomicAdd(&ncert, 1ULL);
        } else {
          fb[atomicAdd(&nfb, 1)] = q;
          atomicAdd(&nfall, 1ULL);
        }
      }
    }
    __syncthreads();
    // ---- 4. FP32 rescan of the consumers that were not certified
    if (nfb > 0) scan_exact<false>(S, mt, fb, nfb);
    __syncthreads();
    return S.nnk;
  }
};

template <bool KIND8, int CAP>
struct BtcSmem {
  CtaCore<CAP> S;
  GeoTC<KIND8, CAP> G;  // its staging union is last and may extend past sizeof()
};

template <bool KIND8, int CAP>
size_t btc_smem_bytes(int kb, int bn, int nstage) {
  using M = BtcSmem<KIND8, CAP>;
  const size_t stage = (size_t)TC_BM * kb + (size_t)nstage * bn * kb;
  const size_t have = sizeof(typename GeoTC<KIND8, CAP>::Stage);
  return sizeof(M) + (stage > have ? stage - have : 0);
}

template <bool KIND8, int CAP>
__global__ void __launch_bounds__(FIN_THREADS, 1) k_batched_tc(BtcArgs A) {
  extern __shared__ __align__(1024) unsigned char smem_raw[];
  BtcSmem<KIND8, CAP>& M = *reinterpret_cast<BtcSmem<KIND8, CAP>*>(smem_raw);
  CtaCore<CAP>& S = M.S;
  GeoTC<KIND8, CAP>& G = M.G;
  __shared__ int s_item;
  __shared__ uint32_t tmem_slot;
  const int tid = threadIdx.x, warp = tid >> 5;
  const uint32_t ncols = 2u * (uint32_t)A.bn;
  if (tid == 0) {
    for (int s = 0; s < A.nstage; ++s) {
      mbar_init(&G.bar_full[s], 1);
      mbar_init(&G.bar_empty[s], 1);
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(&G.bar_acc_full[b], 1);
      mbar_init(&G.bar_acc_empty[b], 4 * 32);
      mbar_init(&G.bar_accf_full[b], 1);
      mbar_init(&G.bar_accf_empty[b], BTC_FILL_WARPS);
    }
    mbar_init(&G.bar_a_full, 1);
    mbar_init(&G.bar_a_empty, 1);
    mbar_fence_init();
    G.prod_a = G.prod_b = G.mma_a = G.mma_b = G.mma_acc = G.epi_acc = G.mma_accf = G.epi_accf = 0u;
    G.ncert = G.nfall = G.nnear = 0ULL;
    G.rk = A.rk;
    G.kb = A.kb;
    G.bn = A.bn;
    G.nstage = A.nstage;
    G.fmt = A.fmt;
    G.err = A.base.err;
    btc_slot_layout(A.scratch + (size_t)blockIdx.x * A.slot_bytes, CAP, A.kb, A.bn, &G.scr, A.kc_cap);
  }
  if (warp == 1) tmem_alloc(&tmem_slot, ncols);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  if (tid == 0) G.tmem_base = tmem_slot;
  __syncthreads();
  const BatchArgs& B = A.base;
  for (;;) {
    if (tid == 0) s_item = (int)atomicAdd(B.queue, 1u);
    __syncthreads();
    const int item = s_item;
    __syncthreads();
    if (item >= B.num) break;
    const int pr = B.pair_ids[item];
    const int64_t xo = B.x_off[pr], yo = B.n_shared ? 0 : B.y_off[pr];
    const int m = (int)(B.x_off[pr + 1] - xo), n = B.n_shared ? B.n_shared : (int)(B.y_off[pr + 1] - yo);
    if (tid == 0) {
      G.x = B.x + xo * B.d;
      G.y = B.y + yo * B.d;
      G.d = B.d;
      G.kc_on = btc_cache_values(m, n) <= A.kc_cap ? 1 : 0;
      G.kc_ready = 0;
      G.pair_m = m;
      G.pair_n = n;
    }
    __syncthreads();
    double cost = 0.0;
    long long rounds = 0, pe = 0;
    const size_t fo = (size_t)blockIdx.x * B.fl_cap;
    const bool ok = cta_solve_pair(S, G, nullptr, nullptr, B.x + xo * B.d, B.a + xo, m, B.y + yo * B.d, B.b + yo, n,
                                   B.d, B.metric, B.err, cost, rounds, pe, B.protocol, B.seed,
                                   B.fl_i ? B.fl_i + fo : nullptr, B.fl_i ? B.fl_j + fo : nullptr,
                                   B.fl_i ? B.fl_f + fo : nullptr, B.fl_cap);
    if (tid == 0) {
      B.costs[pr] = ok ? cost : CUDART_NAN;
      if (B.rounds) B.rounds[pr] = rounds;
      if (B.pair_evals) B.pair_evals[pr] = pe;
    }
    __syncthreads();
  }
  if (tid == 0) {
    atomicAdd(A.certified, G.ncert);
    atomicAdd(A.fallbacks, G.nfall);
    atomicAdd(A.near_ties, G.nnear);
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  if (warp == 1) tmem_dealloc(G.tmem_base, ncols);
}

template <bool KIND8, int CAP>
static int batched_tc_t(const BtcArgs& A, int grid, cudaStream_t st) {
  const size_t smem = btc_smem_bytes<KIND8, CAP>(A.kb, A.bn, A.nstage);
  if (smem > 227 * 1024) return -2;
  // (what nearly every launch stays below, whatever this one takes: the limit
  // belongs to the kernel on the device, and another thread's launch may need
  // more)
  constexpr size_t all = 225 * 1024;  // (the static words are padded to the alignment of the dynamic part)
  cudaError_t e = cudaFuncSetAttribute(k_batched_tc<KIND8, CAP>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)(smem > all ? smem : all));
  if (e != cudaSuccess) return -1;
  k_batched_tc<KIND8, CAP><<<grid, FIN_THREADS, smem, st>>>(A);
  return 0;
}

// Largest number of pipeline stages that fits the shared-memory budget.
int batched_tc_max_stages(int cap, int kb, int bn, int precision) {
  for (int ns = 4; ns >= 1; --ns) {
    size_t b;
    if (precision == 3)
      b = cap <= HD_SMALL_CAP ? btc_smem_bytes<true, HD_SMALL_CAP>(kb, bn, ns) : btc_smem_bytes<true, FIN_MAX_HD>(kb, bn, ns);
    else
      b = cap <= HD_SMALL_CAP ? btc_smem_bytes<false, HD_SMALL_CAP>(kb, bn, ns) : btc_smem_bytes<false, FIN_MAX_HD>(kb, bn, ns);
    if (b <= 227 * 1024) return ns;
  }
  return 0;
}

int launch_batched_tc(const BatchArgs& base, int precision, int cap, int kb, int bn, int nstage, uint8_t* scratch,
                      size_t slot_bytes, unsigned long long* certified, unsigned long long* fallbacks,
                      unsigned long long* near_ties, int rerank_k, long long kc_cap, int grid, cudaStream_t st) {
  const int rk = rerank_k >= 1 && rerank_k <= BTC_K ? rerank_k : BTC_K;
  BtcArgs A{base, scratch, slot_bytes, kb, bn, nstage, fmt_of_precision(precision), certified, fallbacks,
            near_ties, rk, kc_cap};
  if (cap != FIN_MAX_HD) return -2;
  return precision == 3 ? batched_tc_t<true, FIN_MAX_HD>(A, grid, st) : batched_tc_t<false, FIN_MAX_HD>(A, grid, st);
}

}  // namespace nnsemd
