// Reduced-precision NNS for d > 8 on the 5th-generation tensor cores
// (tcgen05, sm_103a), followed by an exact FP32 re-rank with a certificate.
//
//   approx(i, j) = |y_j|^2 + |x_i|^2 - 2 <x~_i, y~_j>
//
// where x~, y~ are BF16 / FP16 / FP8-E4M3 copies of the points (FP16 and FP8
// with a per-row power-of-two scale) and the dot products accumulate in FP32
// in tensor memory.  For every active consumer the kernel keeps the K
// suppliers with the smallest approximate distance.  The re-rank then
// computes the exact FP32 key (the same definition as every other path) of
// those candidates, takes the smallest (lowest position on ties), and
// certifies it (tc_common.cuh): no supplier outside the candidates can reach
// or beat it.  Consumers that cannot be certified are scanned again in FP32
// (k_nns_f32_tiled).  The result is therefore identical to the FP32 path.
//
// K2 k_nns_tc: a CTA owns 128 consumers (the MMA's M) and streams supplier
// tiles of BN rows.  Warp 0 issues 1-D bulk copies (TMA) of the packed tiles
// into a ring of shared-memory stages; warp 1 allocates tensor memory and
// one elected thread issues tcgen05.mma for each tile into a ring of
// TC_NACC FP32 accumulators (BN columns each); warp 2 copies each tile's
// column norms into a ring of its own; the warps from 3 on read each
// accumulator row back with tcgen05.ld (one consumer per thread, two or four
// warps per row, a share of the columns each) and update its top-K.  Every
// wait on an mbarrier is bounded and raises EF_TIMEOUT instead of hanging.
#include <algorithm>
#include <climits>
#include <cmath>

#include "common.cuh"
#include "kernels.h"
#include "tc_common.cuh"

namespace nnsemd {

// warp 0 operand copies, warp 1 MMA, warp 2 column-norm copies, then the
// epilogue warps (EW / 4 per TMEM lane quarter, each a share of the columns).
// Sixteen epilogue warps (more latency hidden) where their registers fit:
// BF16 operands (no per-column scale) and lists of 8.
__host__ __device__ constexpr int tc_epi_warps(int fmt, int kl) { return fmt_is_bf16(fmt) && kl <= 8 ? 16 : 8; }
__host__ __device__ constexpr int tc_threads(int fmt, int kl) { return 32 * (3 + tc_epi_warps(fmt, kl)); }
// A tile + one B stage must fit in this much dynamic shared memory (what
// every instantiation has left beside its static arrays); more stages use
// what the instantiation actually has left.
constexpr int TC_SMEM_BUDGET = 150 * 1024;
constexpr int TC_SMEM_MAX = 227 * 1024;  // per block, static + dynamic
// The epilogue warps work in groups on alternate tiles: a warp's visit to a tile
// is a chain of waits and loads, and with every warp on every tile that chain
// (1,830 cycles), not the MMAs (768 at K = 192) or the shared memory, set the
// pace.
constexpr int TC_GROUPS = 2;
// The consumer tile (A) of the 16-bit formats lies in tensor memory: a 128 x
// 128 x 16 step reads as many bytes of A as of B from shared memory otherwise,
// and shared-memory bandwidth is what bounds K2 (at 32,768 points a tile of K =
// 192 took 3,046 cycles: 768 of operand reads, 384 of copies and some 1,450
// of epilogue accesses).
__host__ __device__ constexpr bool tc_a_in_tmem(int fmt) { return fmt != FMT_E4M3; }
// FP32 accumulators in tensor memory (a ring of tiles in flight); beside three
// of 128 columns A has 128 columns, 512 bytes a row.
__host__ __device__ constexpr int tc_nacc(int fmt, int bn) { return tc_a_in_tmem(fmt) && bn == 128 ? 3 : 4; }
constexpr int TC_NNRM = 4;                  // column-norm slots (a ring of its own, loaded ahead)

// Packs rows in groups of PACK_ROWS: a warp reads its rows (coalesced) into
// shared memory and sums their norms on the way, then each lane takes one row
// of the group and each warp a share of its 16-byte blocks, so that a warp
// writes 512 contiguous bytes of a block column.  (One thread per row, walking
// its own row three times 4 bytes at a time, took 137 us for 131,072 rows of
// d = 64; the bytes read and written take 13.)  Also writes, per point, the
// FP32 squared norm (any order of summation keeps it within gamma_d |v|^2, the
// bound the certificate uses), the per-row scale and, in `stats`, the maxima
// of |v|_2, |v|_1 and the scale over the points (as float bits; all values >=
// 0).  Row p holds the point idx[sel ? sel[p] : p] for p < cnt (cnt read from
// cnt_dev when given; the rest is padding).
constexpr int PACK_ROWS = 32;
constexpr int PACK_THREADS = 256;
constexpr int PACK_SMEM_MAX = 200 * 1024;  // rows of 1,600 coordinates; tc_supported ends at 800

__global__ void __launch_bounds__(PACK_THREADS)
    k_pack_tc(const float* __restrict__ pts, const int* __restrict__ idx, const int* __restrict__ sel,
              const int* __restrict__ cnt_dev, int cnt, int rows_pad, int d, int kb, int fmt, int tile_rows,
              uint8_t* __restrict__ out, float* __restrict__ nrm, float* __restrict__ nrm_s,
              float* __restrict__ scale, unsigned* __restrict__ stats) {
  extern __shared__ float prow[];  // [PACK_ROWS][d rounded up to odd]
  __shared__ float s_scale[PACK_ROWS];
  const int nblk = kb / 16, ld = d | 1;
  const int count = cnt_dev ? min(*cnt_dev, cnt) : cnt;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  constexpr int NW = PACK_THREADS / 32, PER = PACK_ROWS / NW;
  unsigned m0 = 0u, m1 = 0u, m2 = 0u;  // this thread's maxima (float bits of values >= 0)
  for (int p0 = blockIdx.x * PACK_ROWS; p0 < rows_pad; p0 += gridDim.x * PACK_ROWS) {
    const float* row[PER];
    float mx[PER], a2[PER], a1[PER];
#pragma unroll
    for (int h = 0; h < PER; ++h) {
      const int p = p0 + warp * PER + h;
      row[h] = p < count ? pts + (size_t)idx[sel ? sel[p] : p] * d : nullptr;
      mx[h] = a2[h] = a1[h] = 0.f;
    }
    for (int k = lane; k < d; k += 32) {
      float v[PER];
#pragma unroll
      for (int h = 0; h < PER; ++h) v[h] = row[h] ? row[h][k] : 0.f;
#pragma unroll
      for (int h = 0; h < PER; ++h) {
        prow[(warp * PER + h) * ld + k] = v[h];
        mx[h] = fmaxf(mx[h], fabsf(v[h]));
        a2[h] = __fmaf_rn(v[h], v[h], a2[h]);
        a1[h] = __fadd_rn(a1[h], fabsf(v[h]));
      }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
#pragma unroll
      for (int h = 0; h < PER; ++h) {
        mx[h] = fmaxf(mx[h], __shfl_xor_sync(0xffffffffu, mx[h], o));
        a2[h] = __fadd_rn(a2[h], __shfl_xor_sync(0xffffffffu, a2[h], o));
        a1[h] = __fadd_rn(a1[h], __shfl_xor_sync(0xffffffffu, a1[h], o));
      }
    if (lane == 0) {
#pragma unroll
      for (int h = 0; h < PER; ++h) {
        const int p = p0 + warp * PER + h;
        const float s = row[h] ? scale_of_max(mx[h], fmt) : 1.f;
        s_scale[warp * PER + h] = s;
        if (p < rows_pad) {
          nrm[p] = row[h] ? a2[h] : CUDART_INF_F;
          if (nrm_s) nrm_s[p] = row[h] ? norm_up(a2[h]) : 0.f;
          scale[p] = s;
        }
        if (row[h]) {
          m0 = max(m0, __float_as_uint(norm_up(a2[h])));
          m1 = max(m1, __float_as_uint(a1[h] * (1.f + 1e-4f)));
          m2 = max(m2, __float_as_uint(s));
        }
      }
    }
    __syncthreads();
    const int p = p0 + lane;
    if (p < rows_pad) {
      const int t = p / tile_rows, r = p % tile_rows;
      const float* mine = p < count ? prow + lane * ld : nullptr;
      for (int c = warp; c < nblk; c += NW)
        pack_block(mine, d, c, s_scale[lane], fmt, out + (size_t)t * tile_rows * kb, tile_rows, r, nrm_s != nullptr);
    }
    __syncthreads();
  }
  // the maxima: over the warp first, then one atomic per warp (every
  // thread of the block reaches this point: the loop above has no exit)
  m0 = __reduce_max_sync(0xffffffffu, m0);
  m1 = __reduce_max_sync(0xffffffffu, m1);
  m2 = __reduce_max_sync(0xffffffffu, m2);
  if ((threadIdx.x & 31) == 0 && (m0 | m1 | m2)) {
    atomicMax(stats + 0, m0);
    atomicMax(stats + 1, m1);
    atomicMax(stats + 2, m2);
  }
}

// --------------------------------------------------------------------------
// K2
// --------------------------------------------------------------------------

struct TcArgs {
  const uint8_t* A;        // packed consumer tiles (TC_BM rows each)
  const uint8_t* B;        // packed supplier tiles (bn rows each)
  const float* nrm_x;      // [supplier tiles * bn] squared norms (+inf on padding)
  const float* nrm_sx;     // [supplier tiles * bn] norms rounded up (0 on padding)
  const float* nrm_y;      // per-consumer squared norm
  const float* scale_x;    // per-supplier scale
  const float* scale_y;    // per-consumer scale
  int nt;                  // active consumers
  int mt;                  // active suppliers
  int kb;                  // bytes per packed row
  int bn;                  // suppliers per tile
  int nstage;
  int tiles_per_chunk;
  int num_tiles;           // supplier tiles in total
  int nt_pad;              // consumer count rounded up to TC_BM
  float* cand_v;           // [chunks][nt_pad][KL] approximate values (v = |x|^2 - 2 <x~,y~>)
  int* cand_p;             // [chunks][nt_pad][KL] supplier positions
  unsigned* err;
  const int* nq_dev;       // packed consumer rows in use (nullable: nt); tiles past it exit
};

// KL: the length of each consumer's list (TC_K, or TC_K / 2 when at most
// that many candidates are re-ranked: half the insertion work)
template <int FMT, int BN, int KL>
__global__ void __launch_bounds__(tc_threads(FMT, KL), 1) k_nns_tc(TcArgs P) {
  constexpr int EW = tc_epi_warps(FMT, KL);
  constexpr bool ATM = tc_a_in_tmem(FMT);
  constexpr int TC_NACC = tc_nacc(FMT, BN);
  constexpr int PARTS = EW / 4;               // epilogue warps per TMEM lane quarter, lists per row
  constexpr int GW = EW / TC_GROUPS;          // epilogue warps that take a tile
  constexpr int CPART = BN * TC_GROUPS / PARTS;  // columns of a tile per epilogue warp
  static_assert(CPART % 32 == 0, "whole pairs of 16-column blocks per epilogue warp");
  extern __shared__ __align__(1024) uint8_t smem[];
  __shared__ __align__(8) uint64_t bar_full[8];
  __shared__ __align__(8) uint64_t bar_empty[8];
  // an accumulator's barriers alternate between two sets, so that a barrier
  // belongs to tiles of one group and its phases are waited for one by one
  constexpr int NABAR = TC_GROUPS * TC_NACC;
  __shared__ __align__(8) uint64_t bar_acc_full[NABAR];
  __shared__ __align__(8) uint64_t bar_acc_empty[NABAR];
  __shared__ __align__(8) uint64_t bar_nrm_full[TC_NNRM];
  __shared__ __align__(8) uint64_t bar_nrm_empty[TC_NNRM];
  __shared__ __align__(8) uint64_t bar_a;
  __shared__ uint32_t tmem_slot;
  __shared__ __align__(16) float nrm_buf[TC_NNRM][3][BN];  // per tile in flight: |x|^2, |x| rounded up, scale
  // per epilogue thread: one 16-column block (at the end: the lists of
  // parts 1.. of each row, merged into part 0's)
  __shared__ __align__(16) float stage[16][EW * 32];
  __shared__ int tag_pos[TagList<KL>::NTAG][EW * 32];  // per epilogue thread: tag -> position
  __shared__ float seen[PARTS][TC_BM];  // per row and part: its KL / PARTS-th smallest value so far (rounded up)
  static_assert(2 * (PARTS - 1) * KL * TC_BM <= 16 * EW * 32, "the merge lists fit in the staging area");
  float* const merge_v = &stage[0][0];                                              // [PARTS-1][KL][TC_BM]
  int* const merge_p = reinterpret_cast<int*>(&stage[0][0]) + (PARTS - 1) * KL * TC_BM;  // same shape

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int qtile = blockIdx.x;
  const int t0 = blockIdx.y * P.tiles_per_chunk;
  const int t1 = min(t0 + P.tiles_per_chunk, P.num_tiles);
  const int ntiles = t1 - t0;
  if (ntiles <= 0) return;
  if (P.nq_dev && qtile * TC_BM >= *P.nq_dev) return;  // the whole CTA leaves before any set-up
  const int kb = P.kb;
  const uint32_t a_bytes = TC_BM * kb;
  const uint32_t b_bytes = BN * kb;
  uint8_t* sA = smem;
  uint8_t* sB = ATM ? smem : smem + a_bytes;
  const int NST = P.nstage;
  constexpr uint32_t NCOLS = TC_NACC * BN;  // the accumulator ring
  constexpr uint32_t TMEM_ALLOC = ATM ? 512 : NCOLS;  // (A from column NCOLS on: kb / 4 columns)
  static_assert(NCOLS <= 512 && (ATM || (NCOLS & (NCOLS - 1)) == 0), "tensor memory holds 512 columns");
  constexpr uint32_t NRM_BYTES = 3 * BN * sizeof(float);

  if (threadIdx.x == 0) {
    for (int s = 0; s < NST; ++s) {
      mbar_init(&bar_full[s], 1);
      mbar_init(&bar_empty[s], 1);
    }
    for (int b = 0; b < NABAR; ++b) {
      mbar_init(&bar_acc_full[b], 1);
      mbar_init(&bar_acc_empty[b], GW);  // one arrival per epilogue warp of the group
    }
    for (int n = 0; n < TC_NNRM; ++n) {
      mbar_init(&bar_nrm_full[n], 1);
      mbar_init(&bar_nrm_empty[n], GW);
    }
    mbar_init(&bar_a, 1);
    mbar_fence_init();
  }
  if (warp == 1) tmem_alloc(&tmem_slot, TMEM_ALLOC);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = tmem_slot;
  bool ok = true;
  if (ATM) {
    // four warps bring A into tensor memory, a quarter of its rows each
    if (warp >= 4 && warp < 8) {
      const int quarter = warp & 3;
      const uint4* src = reinterpret_cast<const uint4*>(P.A + (size_t)qtile * a_bytes) + quarter * 32 + lane;
      const uint32_t dst = tmem_base + ((uint32_t)(quarter * 32) << 16) + NCOLS;
      for (int c = 0; c < kb / 16; c += 2) {  // (kb is a multiple of 32)
        const uint4 u = src[(size_t)c * TC_BM], v = src[(size_t)(c + 1) * TC_BM];
        tmem_st4(dst + 4 * c, u);
        tmem_st4(dst + 4 * c + 4, v);
      }
      tmem_st_wait();
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
  }

  if (warp == 0) {
    // ---------------- producer: TMA bulk copies of the operand tiles ----------------
    if (lane == 0) {
      if (!ATM) {
        mbar_expect_tx(&bar_a, a_bytes);
        tma_load_1d(sA, P.A + (size_t)qtile * a_bytes, a_bytes, &bar_a);
      }
      for (int t = 0; t < ntiles && ok; ++t) {
        const int s = t % NST, u = t / NST;
        ok = mbar_wait_sleep(&bar_empty[s], (u & 1) ^ 1);
        if (!ok) break;
        mbar_expect_tx(&bar_full[s], b_bytes);
        tma_load_1d(sB + (size_t)s * b_bytes, P.B + (size_t)(t0 + t) * b_bytes, b_bytes, &bar_full[s]);
      }
    }
  } else if (warp == 1) {
    // ---------------- MMA issuer ----------------
    if (lane == 0) {
      constexpr int AB = fmt_is_bf16(FMT) ? 1 : 0;
      const uint32_t idesc = make_idesc(AB, TC_BM, BN);
      const int ksteps = kb / 32;
      if (!ATM) ok = mbar_wait_bounded(&bar_a, 0);
      const uint32_t a0 = smem_u32(sA);
      for (int t = 0; t < ntiles && ok; ++t) {
        const int s = t % NST, u = t / NST;
        const int b = t % TC_NACC, f = t - TC_NACC;  // f: the tile that had this accumulator
        ok = mbar_wait_sleep(&bar_full[s], u & 1);
        if (ok && f >= 0) ok = mbar_wait_sleep(&bar_acc_empty[f % NABAR], (f / NABAR) & 1);
        if (!ok) break;
        tc_fence_after();
        const uint32_t b0 = smem_u32(sB + (size_t)s * b_bytes);
        const uint32_t tmem_d = tmem_base + (uint32_t)(b * BN);
        for (int k = 0; k < ksteps; ++k) {
          const uint64_t bd = make_desc(b0 + k * 2 * BN * 16, BN * 16, 128);
          if constexpr (ATM) {
            mma_issue_atm(tmem_d, tmem_base + NCOLS + 8 * k, bd, idesc, k > 0 ? 1u : 0u);
          } else {
            const uint64_t ad = make_desc(a0 + k * 2 * TC_BM * 16, TC_BM * 16, 128);
            mma_issue<FMT>(tmem_d, ad, bd, idesc, k > 0 ? 1u : 0u);
          }
        }
        mma_commit(&bar_empty[s]);
        mma_commit(&bar_acc_full[t % NABAR]);
      }
    }
  } else if (warp == 2) {
    // ---------------- producer: the column norms of each tile, a ring of their own ----------------
    if (lane == 0) {
      for (int t = 0; t < ntiles && ok; ++t) {
        const int n = t % TC_NNRM, w = t / TC_NNRM;
        ok = mbar_wait_sleep(&bar_nrm_empty[n], (w & 1) ^ 1);
        if (!ok) break;
        const size_t col = (size_t)(t0 + t) * BN;
        mbar_expect_tx(&bar_nrm_full[n], NRM_BYTES);
        tma_load_1d(nrm_buf[n][0], P.nrm_x + col, BN * sizeof(float), &bar_nrm_full[n]);
        tma_load_1d(nrm_buf[n][1], P.nrm_sx + col, BN * sizeof(float), &bar_nrm_full[n]);
        tma_load_1d(nrm_buf[n][2], P.scale_x + col, BN * sizeof(float), &bar_nrm_full[n]);
      }
    }
  } else {
    // ---------------- epilogue: TMEM -> top-K per consumer ----------------
    // PARTS warps per TMEM lane quarter; each takes CPART of the tile's
    // columns and keeps its own top-K, and the parts merge at the end.
    const int e = warp - 3;
    const int etid = e * 32 + lane;
    const int quarter = warp & 3;  // TMEM lanes 32*quarter .. +31
    const int part = e >> 2;                              // this warp's list of its rows
    const int group = part / (PARTS / TC_GROUPS), cpart = part % (PARTS / TC_GROUPS);
    const int row = quarter * 32 + lane;
    const int q = qtile * TC_BM + row;
    const float sy = (q < P.nt) ? P.scale_y[q] : 1.f;
    const float cy = quant_coeff(FMT, (q < P.nt) ? P.nrm_y[q] : 0.f);
    // the list: tagged values (tc_common.cuh), ascending, +inf while not full
    float tv[KL];
    unsigned used = 0u;  // tags held by entries of the list
#pragma unroll
    for (int k = 0; k < KL; ++k) tv[k] = CUDART_INF_F;
    // The row's parts hold KL / PARTS values each at or below the largest of
    // their `seen`, so nothing above that can be among the row's KL smallest:
    // it filters with a row's own list of all columns, not of a part's (about
    // a third of the insertions).  A stale value of another part is larger.
    constexpr int SEEN = KL / PARTS - 1;
    volatile float* const mine = &seen[part][row];
    *mine = CUDART_INF_F;
    asm volatile("bar.sync 1, %0;" ::"r"(EW * 32) : "memory");
    float lim = CUDART_INF_F;
    int* const table = &tag_pos[0][etid];
    constexpr int TSTRIDE = EW * 32;
    static_assert(TC_NNRM % TC_GROUPS == 0, "a norm slot belongs to tiles of one group");
    for (int t = group; t < ntiles; t += TC_GROUPS) {
      const int b = t % TC_NACC, a = t % NABAR, v = t / NABAR;
      const int n = t % TC_NNRM, w = t / TC_NNRM;
      if (ok) ok = mbar_wait_sleep(&bar_acc_full[a], v & 1, 200u);
      if (ok) ok = mbar_wait_sleep(&bar_nrm_full[n], w & 1, 200u);
      tc_fence_after();
      if (ok) {
        const int tile = t0 + t;
        const float* nx = nrm_buf[n][0];
        const float* ns = nrm_buf[n][1];
        const float* sx = nrm_buf[n][2];
        // 32 of this warp's columns of the accumulator at once (one wait for
        // two loads in flight), then two columns per packed FP32x2 step
        constexpr int NB = 2;
        const unsigned long long mcy2 = f2_pack(-cy, -cy);
        const unsigned long long w2c = f2_pack(-2.f, -2.f);
        const unsigned long long wsy2 = f2_pack(-2.f * sy, -2.f * sy);
#pragma unroll 1
        for (int cc = cpart * CPART; cc < (cpart + 1) * CPART; cc += 16 * NB) {
          uint32_t rr[NB][16];
#pragma unroll
          for (int bb = 0; bb < NB; ++bb)
            tmem_ld16_async(tmem_base + ((uint32_t)(quarter * 32) << 16) + (uint32_t)(b * BN + cc + 16 * bb), rr[bb]);
          tmem_ld_wait(rr);
#pragma unroll
          for (int bb = 0; bb < NB; ++bb) {
            const int c0 = cc + 16 * bb;
            const uint32_t(&r)[16] = rr[bb];
            float val[16];
#pragma unroll
            for (int k = 0; k < 16; k += 4) {
              const float4 vx = *reinterpret_cast<const float4*>(nx + c0 + k);
              const float4 vs = *reinterpret_cast<const float4*>(ns + c0 + k);
              unsigned long long w01 = w2c, w23 = w2c;
              if (!fmt_is_bf16(FMT)) {
                // w = (-2 sy) sx: both powers of two, so the product is exact
                const float4 vc = *reinterpret_cast<const float4*>(sx + c0 + k);
                w01 = f2_mul(wsy2, f2_pack(vc.x, vc.y));
                w23 = f2_mul(wsy2, f2_pack(vc.z, vc.w));
              }
              const unsigned long long a01 = f2_pack(__uint_as_float(r[k]), __uint_as_float(r[k + 1]));
              const unsigned long long a23 = f2_pack(__uint_as_float(r[k + 2]), __uint_as_float(r[k + 3]));
              const unsigned long long v01 = f2_fma(mcy2, f2_pack(vs.x, vs.y), f2_fma(w01, a01, f2_pack(vx.x, vx.y)));
              const unsigned long long v23 = f2_fma(mcy2, f2_pack(vs.z, vs.w), f2_fma(w23, a23, f2_pack(vx.z, vx.w)));
              val[k] = f2_lo(v01);
              val[k + 1] = f2_hi(v01);
              val[k + 2] = f2_lo(v23);
              val[k + 3] = f2_hi(v23);
            }
            // the block's minimum as a tree of three-input minima (8 for 16)
            const float mn =
                fminf(fmin3(fmin3(val[0], val[1], val[2]), fmin3(val[3], val[4], val[5]), fmin3(val[6], val[7], val[8])),
                      fmin3(fmin3(val[9], val[10], val[11]), fmin3(val[12], val[13], val[14]), val[15]));
            if (mn < lim) {
              // the few columns that beat the current K-th entry: park the
              // block's values, then one (rolled) insertion per such column
              // that still beats it
              const float thr = lim;
              unsigned msk = 0;
#pragma unroll
              for (int k = 0; k < 16; ++k) {
                msk |= (val[k] < thr ? 1u : 0u) << k;
                stage[k][etid] = val[k];
              }
#pragma unroll 1
              while (msk) {
                const int k = __ffs(msk) - 1;
                msk &= msk - 1;
                const float vk = stage[k][etid];
                if (vk < lim) {
                  tag_insert<KL>(tv, used, table, TSTRIDE, vk, tile * BN + c0 + k);
                  lim = fminf(lim, tv[KL - 1]);
                }
              }
              if (tv[SEEN] < CUDART_INF_F) *mine = tag_ceil(tv[SEEN], TagList<KL>::MASK);
            }
          }
        }
      }
      float m = *const_cast<volatile float*>(&seen[0][row]);
#pragma unroll
      for (int u = 1; u < PARTS; ++u) m = fmaxf(m, *const_cast<volatile float*>(&seen[u][row]));
      lim = fminf(tv[KL - 1], m);
      tc_fence_before();
      __syncwarp();
      if (lane == 0) {
        mbar_arrive(&bar_acc_empty[a]);
        mbar_arrive(&bar_nrm_empty[n]);
      }
    }
    // untag: positions from the table, values floored to lower bounds of
    // the exact approximate values (every bound taken from a list is then
    // at most the value it stands for)
    int tp[KL];
#pragma unroll
    for (int k = 0; k < KL; ++k) {
      const bool real = tv[k] != CUDART_INF_F;
      tp[k] = real ? table[(__float_as_uint(tv[k]) & TagList<KL>::MASK) * TSTRIDE] : -1;
      if (real) tv[k] = tag_floor(tv[k], TagList<KL>::MASK);
    }
    // merge: parts 1.. hand their lists to part 0 (through the staging
    // area, once every epilogue warp has left it)
    asm volatile("bar.sync 1, %0;" ::"r"(EW * 32) : "memory");
    if (part > 0) {
      const int o = (part - 1) * KL * TC_BM;
#pragma unroll
      for (int k = 0; k < KL; ++k) {
        merge_v[o + k * TC_BM + row] = tv[k];
        merge_p[o + k * TC_BM + row] = tp[k];
      }
    }
    asm volatile("bar.sync 1, %0;" ::"r"(EW * 32) : "memory");
    if (part == 0) {
      for (int pp = 0; pp < PARTS - 1; ++pp) {
        const int o = pp * KL * TC_BM;
#pragma unroll
        for (int k = 0; k < KL; ++k) topk_insert(tv, tp, merge_v[o + k * TC_BM + row], merge_p[o + k * TC_BM + row]);
      }
      if (q < P.nt) {
        const size_t o = ((size_t)blockIdx.y * P.nt_pad + q) * KL;
#pragma unroll
        for (int k = 0; k < KL; ++k) {
          P.cand_v[o + k] = tv[k];
          P.cand_p[o + k] = tp[k];
        }
      }
    }
  }
  if (!ok) atomicOr(P.err, EF_TIMEOUT);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  if (warp == 1) tmem_dealloc(tmem_base, TMEM_ALLOC);
}

// --------------------------------------------------------------------------
// exact re-rank + certificate
// --------------------------------------------------------------------------

struct RerankArgs {
  const float* x;       // original coordinates
  const float* y;
  const int* ia;        // active supplier position -> original index
  const int* ja;
  int d, nt, nt_pad, chunks, fmt;
  const float* cand_v;
  const int* cand_p;
  const float* nrm_y;   // FP32 squared norm of each active consumer
  const float* scale_y;
  const unsigned* stats_x;  // max |x|_2, max |x|_1, max scale over active suppliers (float bits)
  unsigned long long* nnkey;
  int* fallback;        // consumer positions to rescan in FP32
  int* nfallback;
  unsigned long long* ncertified;
  unsigned long long* nfallback_total;
  unsigned long long* nnear;  // consumers whose exact best differs from the approximate best
  const int* sel;       // packed row -> consumer position (nullable: identity)
  const int* nq_dev;    // rows in use (nullable: nt)
  TcLists lists;        // candidate lists to make (list == nullptr: none)
  int mt;               // active suppliers
  int rk;               // candidates of each chunk re-ranked (1 .. kl)
  int kl;               // list length of each chunk (the stride of cand_v / cand_p)
};

// RR_ROWS (8 or 32) packed consumer rows per block, G lanes a row (8 where the rows'
// candidates are that few, else a warp).  The first rk candidates of every
// chunk are re-ranked; tau is the smallest rk-th approximate value over the
// chunks (every supplier outside them lies at or above it).  A consumer whose
// exact best differs from the candidate the approximate values ranked first
// (over all chunks, lowest position on ties) is counted as a near-tie of the
// operand precision.
//
// The certificate is about fifty FP64 operations a row, and an FP64
// instruction holds its pipe as long for one active lane as for 32: the last
// step takes one row per lane of a warp; the FP64 norms before it are sums over
// a row's lanes.  (One warp per row, its certificate in one lane and its counters
// updated one by one took 725 us for 131,072 rows, against 100 of candidate rows
// read.)
// Where a block of 32 rows would leave SMs idle (few consumers, many chunks of
// candidates: a few thousand consumers of a learned round took 300 us), RR_ROWS
// is 8, one row a warp.
constexpr int RR_THREADS = 256;

template <int G, int RR_ROWS>
__global__ void __launch_bounds__(RR_THREADS) k_rerank_certify(RerankArgs R) {
  __shared__ unsigned long long s_best[RR_ROWS], s_abest[RR_ROWS];
  __shared__ float s_tau[RR_ROWS];
  __shared__ double s_l2[RR_ROWS], s_l1[RR_ROWS];  // |y|_2^2 and |y|_1
  __shared__ unsigned s_drop[RR_ROWS];  // the smallest key (bits) a list leaves out
  __shared__ int s_len[RR_ROWS], s_have[RR_ROWS];
  const int nq = R.nq_dev ? min(*R.nq_dev, R.nt) : R.nt;
  const int r0 = blockIdx.x * RR_ROWS;
  if (r0 >= nq) return;
  const int sub = threadIdx.x % G;
  const int rk = R.rk;
  const int ncand = R.chunks * rk;
  // rows read 16 bytes at a time where d and both bases allow it
  const bool vec = (R.d & 3) == 0 && ((reinterpret_cast<uintptr_t>(R.x) | reinterpret_cast<uintptr_t>(R.y)) & 15) == 0;
  for (int k0 = threadIdx.x / G; k0 < RR_ROWS; k0 += RR_THREADS / G) {  // (whole warps: RR_ROWS is a multiple)
    const int r = r0 + k0;
    unsigned long long best = ~0ULL, abest = ~0ULL;
    float tau = CUDART_INF_F;  // smallest chunk threshold (rk-th value of each chunk)
    // this lane's two smallest keys by original index, and the smallest other
    unsigned long long e1 = ~0ULL, e2 = ~0ULL;
    unsigned drop = 0xffffffffu;
    int j = 0, have = 0;
    double l2 = 0.0, l1 = 0.0;
    if (r < nq) {
      const int q = R.sel ? R.sel[r] : r;
      j = R.ja[q];
      const float* yrow = R.y + (size_t)j * R.d;
      for (int c = sub; c < ncand; c += G) {
        const int chunk = c / rk, k = c % rk;
        const size_t o = ((size_t)chunk * R.nt_pad + r) * R.kl + k;
        const int p = R.cand_p[o];
        if (k == rk - 1) tau = fminf(tau, R.cand_v[o]);
        if (p < 0) continue;
        ++have;
        if (k == 0) {
          const unsigned long long ak = ((unsigned long long)ordered_bits(R.cand_v[o]) << 32) | (unsigned)p;
          abest = ak < abest ? ak : abest;
        }
        // squared-Euclidean FP32 key (the contraction has no L1 form)
        const int i = R.ia[p];
        const float* xr = R.x + (size_t)i * R.d;
        const float acc = vec ? key32_sql2_v4(xr, yrow, R.d) : key32<METRIC_SQL2>(xr, yrow, R.d);
        const unsigned long long key = pack_key(acc, (unsigned)p);
        best = key < best ? key : best;
        const unsigned long long e = pack_key(acc, (unsigned)i);
        if (e < e2) {
          drop = min(drop, (unsigned)(e2 >> 32));
          e2 = e < e1 ? e1 : e;
          e1 = e < e1 ? e : e1;
        } else {
          drop = min(drop, (unsigned)(e >> 32));
        }
      }
      for (int k = sub; k < R.d; k += G) {
        const double v = yrow[k];
        l2 += v * v;
        l1 += fabs(v);
      }
    }
    if (R.lists.list) {
      // the TCL smallest keys, in order
      if (G == 8) {  // at most one key a lane
        int rank = 0, len = 0;
#pragma unroll
        for (int u = 0; u < 8; ++u) {
          const unsigned long long o = __shfl_sync(0xffffffffu, e1, (threadIdx.x & 24) + u);
          rank += o < e1;
          len += o != ~0ULL;
        }
        if (e1 != ~0ULL) R.lists.list[(size_t)j * TCL + rank] = e1;
        if (sub == 0) {
          s_len[k0] = len;
          s_drop[k0] = 0xffffffffu;
        }
      } else {
        const int lane = threadIdx.x & 31;
        unsigned long long mine = ~0ULL;
        int len = 0;
#pragma unroll 1
        for (; len < TCL; ++len) {
          const unsigned hi = __reduce_min_sync(0xffffffffu, (unsigned)(e1 >> 32));
          if (hi == 0xffffffffu) break;
          const unsigned lo = __reduce_min_sync(0xffffffffu, (unsigned)(e1 >> 32) == hi ? (unsigned)e1 : 0xffffffffu);
          const unsigned long long w = ((unsigned long long)hi << 32) | lo;
          if (e1 == w) {
            e1 = e2;
            e2 = ~0ULL;
          }
          if (lane == len) mine = w;
        }
        if (lane < len) R.lists.list[(size_t)j * TCL + lane] = mine;
        // (a lane's third key and beyond are above its two kept ones, but may
        // be below another lane's that the list took; kept keys that the list
        // left out come after all of its own)
        drop = __reduce_min_sync(0xffffffffu, drop);
        if (sub == 0) {
          s_len[k0] = len;
          s_drop[k0] = drop;
        }
      }
    }
#pragma unroll
    for (int o = G / 2; o > 0; o >>= 1) {
      const unsigned long long ob = __shfl_xor_sync(0xffffffffu, best, o);
      best = ob < best ? ob : best;
      const unsigned long long oa = __shfl_xor_sync(0xffffffffu, abest, o);
      abest = oa < abest ? oa : abest;
      tau = fminf(tau, __shfl_xor_sync(0xffffffffu, tau, o));
      have += __shfl_xor_sync(0xffffffffu, have, o);
      // (FP64: the first step leaves l2 to the lower lanes and l1 to the upper)
      const bool up = (sub & (G / 2)) != 0;
      const double send = o == G / 2 ? (up ? l2 : l1) : l2;
      l2 = (o == G / 2 && up ? l1 : l2) + __shfl_xor_sync(0xffffffffu, send, o);
    }
    if (sub == 0) {
      s_have[k0] = have;
      s_best[k0] = best;
      s_abest[k0] = abest;
      s_tau[k0] = tau;
      s_l2[k0] = l2;
    }
    if (sub == G / 2) s_l1[k0] = l2;
  }
  __syncthreads();
  if (threadIdx.x >= 32) return;
  const int lane = threadIdx.x, r = r0 + lane;
  const bool live = lane < RR_ROWS && r < nq;
  const int q = live ? (R.sel ? R.sel[r] : r) : 0;
  const unsigned long long best = live ? s_best[lane] : ~0ULL;
  bool certified = false;
  if (live && best != ~0ULL) {
    const float ny = R.nrm_y[r];
    const double yl2 = sqrt(s_l2[lane]) * (1 + 1e-12);
    const float tau = s_tau[lane], key = __uint_as_float((unsigned)(best >> 32));
    // (as certify; the bound itself serves the list too.  tau = +inf: no list
    // is full, so every supplier is a candidate, unless its value was lost to
    // an overflowing norm)
    double fl = CUDART_INF;
    if (tau <= 3.402823466e38f)
      fl = certify_floor(R.fmt, R.d, ny, yl2, s_l1[lane], R.scale_y[r],
                         __uint_as_float(R.stats_x[0]), __uint_as_float(R.stats_x[1]), __uint_as_float(R.stats_x[2]),
                         tau);
    certified = tau <= 3.402823466e38f ? (double)key < fl : s_have[lane] == R.mt;
    if (R.lists.list) {
      const unsigned drop = s_drop[lane];
      if (drop != 0xffffffffu) fl = fmin(fl, (double)__uint_as_float(drop));
      const int j = R.ja[q];
      R.lists.next[j] = certified ? s_len[lane] << 8 : 0;
      R.lists.floor[j] = fl;
    }
  } else if (live && R.lists.list) {
    R.lists.next[R.ja[q]] = 0;
  }
  if (certified) R.nnkey[q] = best;
  const unsigned ok = __ballot_sync(0xffffffffu, certified), bad = __ballot_sync(0xffffffffu, live && !certified);
  const unsigned near =
      __ballot_sync(0xffffffffu, live && best != ~0ULL && (unsigned)best != (unsigned)s_abest[lane]);
  int base = 0;
  if (lane == 0) {
    if (near) atomicAdd(R.nnear, (unsigned long long)__popc(near));
    if (ok) atomicAdd(R.ncertified, (unsigned long long)__popc(ok));
    if (bad) {
      atomicAdd(R.nfallback_total, (unsigned long long)__popc(bad));
      base = atomicAdd(R.nfallback, __popc(bad));
    }
  }
  base = __shfl_sync(0xffffffffu, base, 0);
  if ((bad >> lane) & 1u) R.fallback[base + __popc(bad & ((1u << lane) - 1u))] = q;
}

// --------------------------------------------------------------------------
// host side
// --------------------------------------------------------------------------

size_t tc_kb(int d, int precision) {
  const int esize = precision == 3 ? 1 : 2;
  const int64_t values = (int64_t)d * fmt_parts(fmt_of_precision(precision));
  return (size_t)((values * esize + 31) / 32 * 32);
}

int tc_bn(size_t kb) { return kb <= 384 ? 128 : 64; }

bool tc_supported(int d, int precision) {
  const size_t kb = tc_kb(d, precision);
  const size_t a_bytes = (size_t)TC_BM * kb, b_bytes = (size_t)tc_bn(kb) * kb;
  return a_bytes + b_bytes <= (size_t)TC_SMEM_BUDGET;
}

// B stages (up to 4) in what the instantiation leaves beside its static
// shared memory; the first launch of each instantiation sets the attribute.
template <int FMT, int BN, int KL>
static int launch_tc_t(TcArgs P, dim3 grid, size_t a_bytes, size_t b_bytes, cudaStream_t st) {
  static const int static_smem = [] {
    cudaFuncAttributes fa{};
    if (cudaFuncGetAttributes(&fa, k_nns_tc<FMT, BN, KL>) != cudaSuccess) return -1;
    if (cudaFuncSetAttribute(k_nns_tc<FMT, BN, KL>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             TC_SMEM_MAX - 1024 - (int)fa.sharedSizeBytes) != cudaSuccess)
      return -1;
    return (int)fa.sharedSizeBytes;
  }();
  if (static_smem < 0) return -1;
  const size_t avail = (size_t)(TC_SMEM_MAX - 1024 - static_smem);
  if (tc_a_in_tmem(FMT)) {
    if (tc_nacc(FMT, BN) * BN + a_bytes / TC_BM / 4 > 512) return -2;  // (tc_supported keeps rows below 1,024 bytes)
    a_bytes = 0;
  }
  if (a_bytes + b_bytes > avail) return -2;
  P.nstage = (int)std::min<size_t>(4, (avail - a_bytes) / b_bytes);
  const size_t smem = a_bytes + (size_t)P.nstage * b_bytes;
  k_nns_tc<FMT, BN, KL><<<grid, tc_threads(FMT, KL), smem, st>>>(P);
  return 0;
}

template <int FMT>
static int launch_tc_f(const TcArgs& P, int bn, int kl, dim3 grid, size_t a, size_t b, cudaStream_t st) {
  if (bn == 128) return kl == TC_K ? launch_tc_t<FMT, 128, TC_K>(P, grid, a, b, st)
                                   : launch_tc_t<FMT, 128, TC_K / 2>(P, grid, a, b, st);
  return kl == TC_K ? launch_tc_t<FMT, 64, TC_K>(P, grid, a, b, st) : launch_tc_t<FMT, 64, TC_K / 2>(P, grid, a, b, st);
}

// --------------------------------------------------------------------------
// later rounds from the candidate lists
//
// Active suppliers only ever leave.  A consumer's list holds the smallest exact
// keys of the suppliers active when it was made, and every other one of them
// lay at or above `floor`, so its first entry that is still active is the
// nearest active supplier as long as its key is below floor.  Rounds after the
// first then run the contraction for the consumers whose list is used up or
// does not decide, and those get new lists.  Measured on 131,072 points at d =
// 64 (BF16X3, eight candidates): 19.9 -> 14.0 ms.
// --------------------------------------------------------------------------

__global__ void k_map_positions(const int* __restrict__ ia, int mt, int* __restrict__ pos, int* __restrict__ nsel) {
  const int p = blockIdx.x * blockDim.x + threadIdx.x;
  if (p == 0) *nsel = 0;
  if (p < mt) pos[ia[p]] = p;
}

__global__ void __launch_bounds__(256) k_serve_lists(TcLists T, const int* __restrict__ ia, int mt,
                                                     const int* __restrict__ ja, int nt,
                                                     unsigned long long* __restrict__ nnkey,
                                                     unsigned long long* __restrict__ ncertified) {
  const int q = blockIdx.x * blockDim.x + threadIdx.x, lane = threadIdx.x & 31;
  bool served = false;
  if (q < nt) {
    const int j = ja[q], st = T.next[j], end = st >> 8;
    for (int t = st & 0xff; t < end; ++t) {
      const unsigned long long e = T.list[(size_t)j * TCL + t];
      const int i = (int)(unsigned)e, p = T.pos[i];
      if ((unsigned)p >= (unsigned)mt || ia[p] != i) continue;  // retired
      served = (double)__uint_as_float((unsigned)(e >> 32)) < T.floor[j];
      if (served) {
        nnkey[q] = (e & 0xffffffff00000000ULL) | (unsigned)p;
        T.next[j] = (st & ~0xff) | t;
      }
      break;
    }
  }
  const unsigned ok = __ballot_sync(0xffffffffu, served), left = __ballot_sync(0xffffffffu, q < nt && !served);
  int base = 0;
  if (lane == 0) {
    if (ok) atomicAdd(ncertified, (unsigned long long)__popc(ok));
    if (left) base = atomicAdd(T.nsel, __popc(left));
  }
  base = __shfl_sync(0xffffffffu, base, 0);
  if ((left >> lane) & 1u) T.sel[base + __popc(left & ((1u << lane) - 1u))] = q;
}

__global__ void k_add_count(unsigned long long* ctr, unsigned long long v) { *ctr += v; }

void launch_add_count(unsigned long long* ctr, unsigned long long v, cudaStream_t st) {
  k_add_count<<<1, 1, 0, st>>>(ctr, v);
}

int launch_serve_lists(const SolveBufs& B, int mt, int nt, cudaStream_t st) {
  const TcLists& T = B.lists;
  k_map_positions<<<(mt + 255) / 256, 256, 0, st>>>(B.ia[B.cur], mt, T.pos, T.nsel);
  k_serve_lists<<<(nt + 255) / 256, 256, 0, st>>>(T, B.ia[B.cur], mt, B.ja[B.cur], nt, B.nnkey, &B.st->certified);
  return cudaGetLastError() == cudaSuccess ? 0 : -1;
}

// With sel / nsel_dev the consumers are the positions sel[0 .. *nsel_dev)
// (at most nt of them), e.g. those a learned proposal could not certify.
int launch_nns_tc(const SolveBufs& B, const TcBufs& T, int mt, int nt, int precision, cudaStream_t st,
                  const int* sel, const int* nsel_dev) {
  const int fmt = fmt_of_precision(precision);
  const int kb = (int)tc_kb(B.d, precision);
  const int bn = tc_bn(kb);
  const int qtiles = (nt + TC_BM - 1) / TC_BM;
  const int stiles = (mt + bn - 1) / bn;
  // pack both sides
  if (cudaMemsetAsync(T.stats, 0, 8 * sizeof(unsigned), st) != cudaSuccess) return -1;
  {
    const size_t smem = (size_t)PACK_ROWS * (B.d | 1) * sizeof(float);
    // (one limit for every row length: it belongs to the kernel on the device,
    // and another thread's shorter rows must not lower it under this launch)
    if (smem > PACK_SMEM_MAX) return -2;
    if (smem > 48 * 1024 &&
        cudaFuncSetAttribute(k_pack_tc, cudaFuncAttributeMaxDynamicSharedMemorySize, PACK_SMEM_MAX) != cudaSuccess)
      return -1;
    auto grid = [](int64_t rows) { return (int)std::min<int64_t>((rows + PACK_ROWS - 1) / PACK_ROWS, num_sms() * 16); };
    k_pack_tc<<<grid((int64_t)qtiles * TC_BM), PACK_THREADS, smem, st>>>(
        B.y, B.ja[B.cur], sel, nsel_dev, nt, qtiles * TC_BM, B.d, kb, fmt, TC_BM, T.A, T.nrm_y, nullptr, T.scale_y,
        T.stats + 4);
    k_pack_tc<<<grid((int64_t)stiles * bn), PACK_THREADS, smem, st>>>(B.x, B.ia[B.cur], nullptr, nullptr, mt, stiles * bn,
                                                                  B.d, kb, fmt, bn, T.B, T.nrm_x, T.nrm_sx, T.scale_x,
                                                                  T.stats);
  }
  // candidates re-ranked per chunk; the scan keeps half the lists when that suffices
  const int rk = T.rerank_k >= 1 && T.rerank_k <= TC_K ? T.rerank_k : TC_K;
  const int kl = rk <= TC_K / 2 ? TC_K / 2 : TC_K;
  // Chunks of supplier tiles: waves of CTAs (one per SM) x (tiles of a CTA +
  // what a CTA costs beside its tiles, about six of them), smallest first.
  // Aiming at four CTAs per SM alone left a fifth, nearly empty wave (49
  // consumer tiles x 13 chunks = 637 CTAs).  More chunks also mean more
  // candidates to re-rank: another count has to save 3 %.
  int chunks = 1;
  {
    // (what the candidate buffers hold: layout_solve)
    const int most = std::min(std::min(stiles, T.max_chunks), (tc_target_ctas() + qtiles) * TC_K / kl / qtiles);
    double best = 1e30;
    for (int c = 1; c <= most; ++c) {
      const int tiles = (stiles + c - 1) / c;
      const int64_t ctas = (int64_t)qtiles * ((stiles + tiles - 1) / tiles);
      const double t = (double)((ctas + num_sms() - 1) / num_sms()) * (tiles + 6);
      if (t < 0.97 * best) {
        best = t;
        chunks = c;
      }
    }
  }
  const int per = (stiles + chunks - 1) / chunks;
  chunks = (stiles + per - 1) / per;
  const size_t a_bytes = (size_t)TC_BM * kb, b_bytes = (size_t)bn * kb;
  const int nt_pad = qtiles * TC_BM;
  TcArgs P{T.A,      T.B,      T.nrm_x,    T.nrm_sx, T.nrm_y,  T.scale_x,  T.scale_y, nt, mt,
           kb,       bn,       0,          per,      stiles,   nt_pad,     T.cand_v,  T.cand_p, &B.st->err,
           nsel_dev};
  dim3 grid(qtiles, chunks);
  int rc;
  if (T.ev0) cudaEventRecord(T.ev0, st);
  if (fmt == FMT_BF16)
    rc = launch_tc_f<FMT_BF16>(P, bn, kl, grid, a_bytes, b_bytes, st);
  else if (fmt == FMT_BF16X3)
    rc = launch_tc_f<FMT_BF16X3>(P, bn, kl, grid, a_bytes, b_bytes, st);
  else if (fmt == FMT_F16)
    rc = launch_tc_f<FMT_F16>(P, bn, kl, grid, a_bytes, b_bytes, st);
  else
    rc = launch_tc_f<FMT_E4M3>(P, bn, kl, grid, a_bytes, b_bytes, st);
  if (rc) return rc;
  if (T.ev1) cudaEventRecord(T.ev1, st);
  // exact re-rank and certificate
  if (cudaMemsetAsync(T.nfallback, 0, sizeof(int), st) != cudaSuccess) return -1;
  RerankArgs R{B.x,      B.y,        B.ia[B.cur], B.ja[B.cur], B.d,       nt,          nt_pad,
               chunks,   fmt,        T.cand_v,    T.cand_p,    T.nrm_y,   T.scale_y,   T.stats,
               B.nnkey,  T.fallback, T.nfallback, &B.st->certified, &B.st->fallbacks, &B.st->near_ties,
               sel,      nsel_dev,   B.lists,     mt,          rk,          kl};
  const bool wide = chunks * rk > 8, few = nt < 32 * 4 * num_sms();
  if (!wide) k_rerank_certify<8, 32><<<(nt + 31) / 32, RR_THREADS, 0, st>>>(R);
  else if (few) k_rerank_certify<32, 8><<<(nt + 7) / 8, RR_THREADS, 0, st>>>(R);
  else k_rerank_certify<32, 32><<<(nt + 31) / 32, RR_THREADS, 0, st>>>(R);
  // FP32 scan of the consumers that were not certified
  launch_nns_f32(B, mt, nt, T.fallback, T.nfallback, st);
  return 0;
}

// --------------------------------------------------------------------------
// A plain BF16 contraction on the tensor cores, S = X W^T with FP32
// accumulation (rows of X against rows of W), for the learned proposal's
// per-solve passes.  Both operands are packed like K2's (K-major, no
// swizzle, tiles of 128 rows).  The epilogue either stores S + b (a linear
// layer), keeps each row's largest S + b (an assignment), or turns S into a
// lower bound of a squared distance (below).
// --------------------------------------------------------------------------

constexpr int LIN_TILE = 128;  // rows of X and of W per tile
constexpr int LIN_MAX_K = 256; // packed values per row

enum LinMode : int { LIN_STORE = 0, LIN_ARGMAX = 1, LIN_LOWER = 2, LIN_PACK_RELU = 3 };

struct LinArgs {
  const uint8_t* X;
  const uint8_t* W;
  int K;                     // packed values per row
  int rows, N;
  const float* bias;         // STORE / ARGMAX: [N]
  float* Z;                  // STORE / LOWER: [rows][N]
  uint8_t* P;                // PACK_RELU: relu(S + b) packed in BF16 as the next layer's X (N values a row)
  unsigned long long* part;  // ARGMAX: [rows], all zero before the launch
  // LOWER: the rows and columns as points; X and W hold BF16X3 copies
  const float* row_sq_lo;    // [rows] |y|^2 rounded down
  const float* row_nrm_up;   // [rows] |y| rounded up
  const float* col_sq_lo;    // [N] |mu|^2 rounded down
  const float* col_nrm_up;   // [N] |mu| rounded up
  const float* col_radius;   // [N] r_c (rounded up when formed)
  float err_coeff;           // |S - <y, mu>| <= err_coeff |y| |mu| + 1e-30
  unsigned* err;
};

// Rows [0, rows) of src [rows][d] packed in tiles of LIN_TILE rows (padding
// rows zero): BF16 copies (fmt FMT_BF16), or BF16X3 splits (FMT_BF16X3;
// `supplier` picks the segment order) of 3d values per row.  One thread per
// 16-byte block of a row; consecutive threads write consecutive rows of one
// block column.
__global__ void k_pack_rows(const float* __restrict__ src, int rows, int rows_pad, int d, int fmt, bool supplier,
                            uint8_t* __restrict__ out) {
  const int kb = 2 * d * fmt_parts(fmt);
  const int64_t total = (int64_t)rows_pad * (kb / 16);
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < total; i += (int64_t)gridDim.x * blockDim.x) {
    const int c = (int)(i / rows_pad), p = (int)(i % rows_pad);
    const float* row = p < rows ? src + (size_t)p * d : nullptr;
    const int t = p / LIN_TILE, r = p % LIN_TILE;
    pack_block(row, d, c, 1.f, fmt, out + (size_t)t * LIN_TILE * kb, LIN_TILE, r, supplier);
  }
}

// 128 x 128 blocks of S, a contiguous range of them (columns fastest) per
// CTA.  One thread loads and multiplies: the W tile of the next block arrives
// by a bulk copy while this one's K / 16 MMAs run into one of two 128-column
// accumulators (the X tile stays until the range reaches the next row of
// blocks), and eight epilogue warps (lane quadrant x column half) take the
// other accumulator's values through the mode's epilogue: columns >= N and
// rows >= rows are skipped; ARGMAX keeps each row's largest S + b, lowest
// column on ties, as a packed key over the CTA's blocks and merges it into
// part[row].
//
// LOWER: with S~ the computed <y~, mu~> of the BF16X3 copies, |S~ - <y, mu>|
// <= err_coeff |y| |mu| (+ 1e-30 for the subnormal floors), so
//   |y - mu|^2 >= |y|^2_lo + |mu|^2_lo - 2 (S~ + err_coeff |y|_up |mu|_up),
// and the bound on the squared distance to any point of cell `col` is
// max(0, sqrt(that) - r_col)^2, every step rounded toward the bound.
//
// Bound by the epilogue: some 14 instructions and a 4-byte store per value.
// Stores go out through a warp's staging rows as 64 contiguous bytes of eight
// rows (16 bytes of 32 rows per store cost 32 L1 lookups each).  One block
// per CTA, load, multiply and epilogue one after the other, took 52.7 us
// (LOWER) and 40.3 us (STORE) for 4,096 rows x 4,096 columns at 64 and 256
// coordinates; now 32.7 and 24.3 us.
constexpr int LIN_EPI = 8;                        // epilogue warps
constexpr int LIN_THREADS = 32 * (LIN_EPI + 1);
constexpr int LIN_STAGE = 20;                     // floats per staged row (16 and a pad: no bank conflicts)
constexpr int LIN_SMEM = 3 * LIN_TILE * 2 * LIN_MAX_K + LIN_EPI * 32 * LIN_STAGE * 4;

template <int MODE>
__global__ void __launch_bounds__(LIN_THREADS, 1) k_linear_tc(LinArgs A, int tiles, int ncol) {
  extern __shared__ __align__(1024) uint8_t smem[];
  __shared__ __align__(8) uint64_t bar_full[2], bar_mma[2], bar_free[2];
  __shared__ uint32_t tslot;
  __shared__ __align__(16) float s_col[LIN_EPI][3][64];  // a block's per-column terms, each warp its own copy
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t tile_bytes = LIN_TILE * 2 * A.K;
  uint8_t* sX = smem;
  uint8_t* sW = smem + tile_bytes;  // two buffers
  const int t0 = (int)((int64_t)tiles * blockIdx.x / gridDim.x);
  const int nt = (int)((int64_t)tiles * (blockIdx.x + 1) / gridDim.x) - t0;
  if (threadIdx.x == 0) {
#pragma unroll
    for (int i = 0; i < 2; ++i) {
      mbar_init(&bar_full[i], 1);
      mbar_init(&bar_mma[i], 1);
      mbar_init(&bar_free[i], LIN_EPI);
    }
    mbar_fence_init();
  }
  if (warp == LIN_EPI) tmem_alloc(&tslot, 2 * LIN_TILE);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = tslot;
  if (warp == LIN_EPI) {
    if (lane == 0) {
      auto load = [&](int i, bool with_x) {
        const int t = t0 + i, b = i & 1;
        mbar_expect_tx(&bar_full[b], (with_x ? 2 : 1) * tile_bytes);
        if (with_x) tma_load_1d(sX, A.X + (size_t)(t / ncol) * tile_bytes, tile_bytes, &bar_full[b]);
        tma_load_1d(sW + b * tile_bytes, A.W + (size_t)(t % ncol) * tile_bytes, tile_bytes, &bar_full[b]);
      };
      const uint32_t idesc = make_idesc(1, LIN_TILE, LIN_TILE);
      const uint32_t x0 = smem_u32(sX);
      bool ok = true;
      int loaded = 0, arrived = 0, issued = 0;
      if (nt > 0) {
        load(0, true);
        loaded = 1;
      }
      for (int i = 0; i < nt; ++i) {
        const int b = i & 1;
        const unsigned ph = (unsigned)(i >> 1) & 1u;
        const bool next = i + 1 < nt, new_row = next && (t0 + i + 1) % ncol == 0;
        if (next && !new_row) {  // the buffer of block i - 1
          if (i > 0 && !(ok = mbar_wait_bounded(&bar_mma[b ^ 1], (unsigned)((i - 1) >> 1) & 1u))) break;
          load(i + 1, false);
          loaded = i + 2;
        }
        if (!(ok = mbar_wait_bounded(&bar_full[b], ph))) break;
        arrived = i + 1;
        if (i > 1 && !(ok = mbar_wait_bounded(&bar_free[b], ph ^ 1u))) break;  // block i - 2 is read
        tc_fence_after();
        const uint32_t w0 = smem_u32(sW + b * tile_bytes);
        for (int k = 0; k < A.K / 16; ++k)
          mma_issue<FMT_BF16>(tmem + (uint32_t)(b * LIN_TILE),
                              make_desc(x0 + k * 2 * LIN_TILE * 16, LIN_TILE * 16, 128),
                              make_desc(w0 + k * 2 * LIN_TILE * 16, LIN_TILE * 16, 128), idesc, k > 0 ? 1u : 0u);
        mma_commit(&bar_mma[b]);
        issued = i + 1;
        if (new_row) {  // X may go once its last MMAs are done
          if (!(ok = mbar_wait_bounded(&bar_mma[b], ph))) break;
          load(i + 1, true);
          loaded = i + 2;
        }
      }
      if (!ok) {  // leave no copy and no MMA in flight
        for (int i = arrived; i < loaded; ++i) mbar_wait_bounded(&bar_full[i & 1], (unsigned)(i >> 1) & 1u);
        if (issued > 0) mbar_wait_bounded(&bar_mma[(issued - 1) & 1], (unsigned)((issued - 1) >> 1) & 1u);
        atomicOr(A.err, EF_TIMEOUT);
      }
    }
    __syncwarp();
  } else {
    const int quad = warp & 3, half = warp >> 2;
    float* stage = reinterpret_cast<float*>(smem + 3 * tile_bytes) + warp * 32 * LIN_STAGE;
    float(*col)[64] = s_col[warp];
    unsigned long long best = 0ULL;
    for (int i = 0; i < nt; ++i) {
      const int t = t0 + i, b = i & 1;
      const int row = t / ncol * LIN_TILE + quad * 32 + lane;
      const int n0 = t % ncol * LIN_TILE + half * 64;
      const bool live = row < A.rows;
      __syncwarp();  // the previous block's reads of col
#pragma unroll
      for (int u = lane; u < 64; u += 32) {
        const int n = n0 + u;
        const bool in = n < A.N;
        if (MODE == LIN_LOWER) {
          col[0][u] = in ? A.col_sq_lo[n] : 0.f;
          col[1][u] = in ? A.col_nrm_up[n] : 0.f;
          col[2][u] = in ? A.col_radius[n] : 0.f;
        } else {
          col[0][u] = in ? A.bias[n] : 0.f;
        }
      }
      float ysq = 0.f, ynr = 0.f;
      if (MODE == LIN_LOWER && live) {
        ysq = A.row_sq_lo[row];
        ynr = A.row_nrm_up[row];
      }
      // (every lane of a warp agrees before the aligned loads)
      if (!__all_sync(0xffffffffu, mbar_wait_bounded(&bar_mma[b], (unsigned)(i >> 1) & 1u))) {
        if (lane == 0) atomicOr(A.err, EF_TIMEOUT);
        break;
      }
      tc_fence_after();
      uint32_t rr[4][16];
#pragma unroll
      for (int g = 0; g < 4; ++g)
        tmem_ld16_async(tmem + ((uint32_t)(quad * 32) << 16) + (uint32_t)(b * LIN_TILE + half * 64 + 16 * g), rr[g]);
      tmem_ld_wait(rr);
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(&bar_free[b]);
#pragma unroll
      for (int g = 0; g < 4; ++g) {
        const int nb = n0 + 16 * g;
        if (nb >= A.N) continue;
        if constexpr (MODE == LIN_PACK_RELU) {
          // 16 columns = two 16-byte blocks of the next layer's packed row
          // (zeros for padding rows, so the next tile holds no garbage)
          const int kb = 2 * A.N;
          uint8_t* base = A.P + (size_t)(row / LIN_TILE) * LIN_TILE * kb + (size_t)(row % LIN_TILE) * 16;
          uint32_t w[8];
#pragma unroll
          for (int e = 0; e < 8; ++e) {
            const float lo = live ? fmaxf(__uint_as_float(rr[g][2 * e]) + col[0][16 * g + 2 * e], 0.f) : 0.f;
            const float hi = live ? fmaxf(__uint_as_float(rr[g][2 * e + 1]) + col[0][16 * g + 2 * e + 1], 0.f) : 0.f;
            w[e] = (uint32_t)__bfloat16_as_ushort(__float2bfloat16_rn(lo)) |
                   ((uint32_t)__bfloat16_as_ushort(__float2bfloat16_rn(hi)) << 16);
          }
          *reinterpret_cast<uint4*>(base + (size_t)(nb / 8) * LIN_TILE * 16) = make_uint4(w[0], w[1], w[2], w[3]);
          *reinterpret_cast<uint4*>(base + (size_t)(nb / 8 + 1) * LIN_TILE * 16) = make_uint4(w[4], w[5], w[6], w[7]);
        } else if constexpr (MODE == LIN_ARGMAX) {
#pragma unroll
          for (int e = 0; e < 16; ++e) {
            const int n = nb + e;
            const unsigned long long key =
                ((unsigned long long)ordered_bits(__uint_as_float(rr[g][e]) + col[0][16 * g + e]) << 32) |
                (0xffffffffu - (unsigned)n);
            if (n < A.N && key > best) best = key;
          }
        } else {
#pragma unroll
          for (int e = 0; e < 16; e += 4) {
            const float4 c0 = *reinterpret_cast<const float4*>(&col[0][16 * g + e]);
            const float ca[4] = {c0.x, c0.y, c0.z, c0.w};
            float out[4];
            if (MODE == LIN_STORE) {
#pragma unroll
              for (int f = 0; f < 4; ++f) out[f] = __uint_as_float(rr[g][e + f]) + ca[f];
            } else {
              const float4 c1 = *reinterpret_cast<const float4*>(&col[1][16 * g + e]);
              const float4 c2 = *reinterpret_cast<const float4*>(&col[2][16 * g + e]);
              const float cn[4] = {c1.x, c1.y, c1.z, c1.w}, cr[4] = {c2.x, c2.y, c2.z, c2.w};
#pragma unroll
              for (int f = 0; f < 4; ++f) {
                const float sv = __uint_as_float(rr[g][e + f]);
                const float eb = __fmaf_ru(A.err_coeff, __fmul_ru(ynr, cn[f]), 1e-30f);
                const float d2 = __fsub_rd(__fadd_rd(ysq, ca[f]), __fmul_ru(2.f, __fadd_ru(sv, eb)));
                // sqrt from below: x * rsqrtf(x) is within 2^-22 of sqrt(x)
                // (rsqrtf is documented to 2 ulp), and the factor 1 - 2^-20
                // takes it under; tiny or non-positive x gives 0
                const float dist = d2 > 1e-30f ? __fmul_rd(__fmul_rd(d2, rsqrtf(d2)), 0.99999905f) : 0.f;
                const float gap = __fsub_rd(dist, cr[f]);
                out[f] = gap > 0.f ? __fmul_rd(gap, gap) : 0.f;
              }
            }
            *reinterpret_cast<float4*>(stage + lane * LIN_STAGE + e) = make_float4(out[0], out[1], out[2], out[3]);
          }
          __syncwarp();
          // eight rows of 64 bytes at a time
          const int n = nb + 4 * (lane & 3);
#pragma unroll
          for (int h = 0; h < 4; ++h) {
            const int r = 8 * h + (lane >> 2);
            const int gr = row - lane + r;
            const float4 v = *reinterpret_cast<const float4*>(stage + r * LIN_STAGE + 4 * (lane & 3));
            if (gr < A.rows) {
              float* zr = A.Z + (size_t)gr * A.N;
              if ((A.N & 3) == 0) {
                if (n < A.N) *reinterpret_cast<float4*>(zr + n) = v;
              } else {
                const float o[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
                for (int f = 0; f < 4; ++f)
                  if (n + f < A.N) zr[n + f] = o[f];
              }
            }
          }
          __syncwarp();
        }
      }
      if (MODE == LIN_ARGMAX && (i + 1 == nt || (t + 1) % ncol == 0)) {
        if (live) atomicMax(A.part + row, best);
        best = 0ULL;
      }
    }
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  if (warp == LIN_EPI) tmem_dealloc(tmem, 2 * LIN_TILE);
}

// out[row] = the column of the row's largest key
__global__ void k_argmax_parts(const unsigned long long* __restrict__ part, int rows, int* __restrict__ out) {
  const int r = blockIdx.x * blockDim.x + threadIdx.x;
  if (r < rows) out[r] = (int)(0xffffffffu - (unsigned)(part[r] & 0xffffffffu));
}

// Per point: |p|^2 (relative error <= gamma_d in any order of summation)
// rounded down and |p| rounded up.  Eight lanes a point: one lane walking a row
// left the GPU idle at 4,096 rows (12.4 us).
__global__ void k_point_norms(const float* __restrict__ pts, int n, int d, float* __restrict__ sq_lo,
                              float* __restrict__ nrm_up) {
  const int i = (blockIdx.x * blockDim.x + threadIdx.x) >> 3, sub = threadIdx.x & 7;
  float s = 0.f;
  if (i < n)
    for (int k = sub; k < d; k += 8) s = __fmaf_rn(pts[(size_t)i * d + k], pts[(size_t)i * d + k], s);
#pragma unroll
  for (int o = 4; o > 0; o >>= 1) s = __fadd_rn(s, __shfl_xor_sync(0xffffffffu, s, o));
  if (i >= n || sub != 0) return;
  const double g = certify_gamma(d);
  sq_lo[i] = __fmul_rd(s, __double2float_rd(1.0 - g));
  nrm_up[i] = __fsqrt_ru(__fmul_ru(s, __double2float_ru(1.0 + g / (1.0 - g))));
}

bool linear_tc_supported(int K) { return K >= 16 && K <= LIN_MAX_K && K % 16 == 0; }

size_t linear_tc_packed_bytes(int rows, int K) {
  return (size_t)(rows + LIN_TILE - 1) / LIN_TILE * LIN_TILE * 2 * K;
}

static int pack_rows(const float* src, int rows, int d, int fmt, bool supplier, uint8_t* out, cudaStream_t st) {
  const int rows_pad = (rows + LIN_TILE - 1) / LIN_TILE * LIN_TILE;
  const int64_t work = (int64_t)rows_pad * (2 * d * fmt_parts(fmt) / 16);
  const int g = (int)std::max<int64_t>(1, std::min<int64_t>((work + 255) / 256, num_sms() * 16));
  k_pack_rows<<<g, 256, 0, st>>>(src, rows, rows_pad, d, fmt, supplier, out);
  return cudaGetLastError() == cudaSuccess ? 0 : -1;
}

int pack_rows_bf16(const float* src, int rows, int K, uint8_t* out, cudaStream_t st) {
  return pack_rows(src, rows, K, FMT_BF16, false, out, st);
}

template <int MODE>
static int launch_linear_tc(const LinArgs& A, cudaStream_t st) {
  if (!linear_tc_supported(A.K) || A.rows <= 0 || A.N <= 0) return -2;
  static const bool attr =
      cudaFuncSetAttribute(k_linear_tc<MODE>, cudaFuncAttributeMaxDynamicSharedMemorySize, LIN_SMEM) == cudaSuccess;
  if (!attr) return -1;
  const int ncol = (A.N + LIN_TILE - 1) / LIN_TILE;
  const int64_t tiles = (int64_t)ncol * ((A.rows + LIN_TILE - 1) / LIN_TILE);
  if (tiles > INT_MAX) return -2;
  const int smem = 3 * LIN_TILE * 2 * A.K + LIN_EPI * 32 * LIN_STAGE * 4;
  k_linear_tc<MODE><<<(int)std::min<int64_t>(tiles, num_sms()), LIN_THREADS, smem, st>>>(A, (int)tiles, ncol);
  return cudaGetLastError() == cudaSuccess ? 0 : -1;
}

int linear_tc(const uint8_t* X, int rows, int K, const uint8_t* W, const float* bias, int N, float* Z, unsigned* err,
              cudaStream_t st) {
  LinArgs A{};
  A.X = X, A.W = W, A.K = K, A.rows = rows, A.N = N, A.bias = bias, A.Z = Z, A.err = err;
  return launch_linear_tc<LIN_STORE>(A, st);
}

int linear_tc_pack_relu(const uint8_t* X, int rows, int K, const uint8_t* W, const float* bias, int N, uint8_t* out,
                        unsigned* err, cudaStream_t st) {
  if (N % 16) return -2;
  LinArgs A{};
  A.X = X, A.W = W, A.K = K, A.rows = rows, A.N = N, A.bias = bias, A.P = out, A.err = err;
  return launch_linear_tc<LIN_PACK_RELU>(A, st);
}

int linear_tc_argmax(const uint8_t* X, int rows, int K, const uint8_t* W, const float* bias, int N,
                     unsigned long long* part, int* out, unsigned* err, cudaStream_t st) {
  LinArgs A{};
  A.X = X, A.W = W, A.K = K, A.rows = rows, A.N = N, A.bias = bias, A.part = part, A.err = err;
  if (rows > 0 && cudaMemsetAsync(part, 0, (size_t)rows * sizeof(unsigned long long), st) != cudaSuccess) return -1;
  const int rc = launch_linear_tc<LIN_ARGMAX>(A, st);
  if (rc) return rc;
  k_argmax_parts<<<(rows + 255) / 256, 256, 0, st>>>(part, rows, out);
  return cudaGetLastError() == cudaSuccess ? 0 : -1;
}

bool cell_bounds_tc_supported(int d) { return d % 16 == 0 && linear_tc_supported(3 * d); }

int cell_bounds_tc_cells(const float* mu, int cells, int d, uint8_t* packed, float* sq_lo, float* nrm_up,
                         cudaStream_t st) {
  k_point_norms<<<(cells + 31) / 32, 256, 0, st>>>(mu, cells, d, sq_lo, nrm_up);
  return pack_rows(mu, cells, d, FMT_BF16X3, true, packed, st);
}

int cell_bounds_tc(const float* y, int rows, int d, uint8_t* packed_y, float* y_sq_lo, float* y_nrm_up,
                   const uint8_t* packed_mu, const float* mu_sq_lo, const float* mu_nrm_up, const float* radius,
                   int cells, float* out, unsigned* err, cudaStream_t st) {
  k_point_norms<<<(rows + 31) / 32, 256, 0, st>>>(y, rows, d, y_sq_lo, y_nrm_up);
  if (pack_rows(y, rows, d, FMT_BF16X3, false, packed_y, st)) return -1;
  // |<y~, mu~> - <y, mu>| <= (Q + K 2^-22 nf^2) |y| |mu| for the BF16X3
  // copies (the certificate's quantisation and accumulation terms, K = 3d
  // packed values), with a little slack for this single-precision use
  const int K = 3 * d;
  const double nf = quant_norm_factor(FMT_BF16X3);
  const double c = (quant_err(FMT_BF16X3) + K * 0x1p-22 * nf * nf) * (1.0 + 1e-3);
  LinArgs A{};
  A.X = packed_y, A.W = packed_mu, A.K = K, A.rows = rows, A.N = cells, A.Z = out, A.err = err;
  A.row_sq_lo = y_sq_lo, A.row_nrm_up = y_nrm_up, A.col_sq_lo = mu_sq_lo, A.col_nrm_up = mu_nrm_up;
  A.col_radius = radius;
  float cf = (float)c;
  if ((double)cf < c) cf = std::nextafter(cf, 2.f * cf);  // rounded up
  A.err_coeff = cf;
  return launch_linear_tc<LIN_LOWER>(A, st);
}

}  // namespace nnsemd
