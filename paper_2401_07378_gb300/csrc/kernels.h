// Host-side launchers of the NNS-EMD kernels (internal to the library).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "common.cuh"

namespace nnsemd {

// Supplier tile staged in shared memory by K1, and the granularity every
// packed active list is padded to (with NaN coordinates) so that a tile
// never reads past its buffer.
constexpr int K1_TS = 256;
// Streaming multiprocessors of the current device (the device attribute
// cudaDevAttrMultiProcessorCount, looked up once per device); grids are
// sized in multiples of it.
int num_sms();
// K2's candidate buffers hold this many (consumer tile, supplier chunk) pairs:
// four CTAs per SM (launch_nns_tc chooses the chunks).
inline int tc_target_ctas() { return 4 * num_sms(); }
constexpr int PAD_POINTS = K1_TS;
// Largest active set the single-CTA solver keeps in shared memory (d <= 8:
// with coordinates; d > 8: per-point state only, coordinates stay in L2).
constexpr int FIN_MAX = 1024;
constexpr int FIN_MAX_HD = 2048;
// Point capacity per side of the cluster tail (d <= 8): its whole state,
// the coordinates at DP floats per point and the key exchange buffers fit
// one CTA's shared memory up to 2048 points for DP <= 4, 1024 for DP = 8.
constexpr int FIN_CL_MAX = 2048;
__host__ __device__ constexpr int fin_cl_cap(int dp) { return dp <= 4 ? FIN_CL_MAX : 1024; }

// Row length of a key matrix over n consumers (rows start on 16 bytes).
__host__ __device__ inline long long kmat_ld(long long n) { return (n + 3) & ~3LL; }

__host__ __device__ inline int padded_dim(int d) { return d <= 2 ? 2 : (d <= 4 ? 4 : 8); }
__host__ __device__ inline int64_t pad_points(int64_t n) { return (n + PAD_POINTS - 1) / PAD_POINTS * PAD_POINTS; }

// Buffers of the reduced-precision NNS step (tc.cu).
struct TcBufs {
  uint8_t* A;                  // packed consumer tiles
  uint8_t* B;                  // packed supplier tiles
  float* nrm_x;                // per supplier position (padded), +inf on padding
  float* nrm_sx;               // per supplier position: |x| rounded up, 0 on padding
  float* nrm_y;                // per consumer position
  float* scale_x;
  float* scale_y;
  unsigned* stats;             // [8]: supplier max |x|_2, |x|_1, scale; consumer the same at +4
  float* cand_v;               // [chunks][nt_pad][8]
  int* cand_p;
  int* fallback;               // consumer positions to rescan
  int* nfallback;              // device counter (this round)
  int max_chunks;
  int rerank_k;                // candidates per chunk re-ranked in FP32 (1..16; other values: 16)
  cudaEvent_t ev0, ev1;        // optional: recorded around the tensor-core kernel
};

// Candidate lists kept over the rounds of a reduced-precision solve (tc.cu), by
// original consumer: up to TCL exact keys (key32 bits << 32 | original
// supplier) ascending, the next entry to look at | length << 8, and the value a
// key must stay below to be the nearest active supplier's.
constexpr int TCL = 8;
struct TcLists {
  unsigned long long* list;  // [n][TCL]; null: no lists
  int* next;                 // [n]
  double* floor;             // [n]
  int* pos;                  // [m] position of each active supplier by original index (others: stale)
  int* sel;                  // [n] consumer positions the lists do not answer
  int* nsel;
};

// Buffers of the spatially ordered NNS step (lowd_grid.cu, d <= 3).
struct GridBufs {
  unsigned* box;             // [6] bounding box of both sets (ordered bits); null: not laid out
  int* hist;
  int* start;
  float* xs;                 // sorted suppliers / consumers, 4 floats a point
  float* ys;
  float* boxes;
  unsigned long long* work;  // [2] what the round's cells hold in common and its visits (grid_served)
};

// Buffers of one single-pair solve (device pointers inside the workspace).
struct SolveBufs {
  int precision;   // nnsemd_precision of the NNS step (0 = FP32)
  int protocol;    // nnsemd_protocol (0 greedy, 1 random)
  unsigned long long seed;  // random protocol seed
  long long round0;         // rounds run before the one-CTA tail (random-protocol keys)
  TcBufs tc;       // used when precision != 0
  TcLists lists;   // used when precision != 0 and no proposal
  GridBufs grid;   // d <= 3
  const float* x;  // original coordinates [m][d]
  const float* y;  // [n][d]
  int64_t m, n;
  int d, dp, metric;
  double* s;       // residual supplier weights [m] (original index)
  double* c;       // residual consumer weights [n]
  float* xa[2];    // packed active supplier coordinates [pad(m)][dp]
  int* ia[2];      // their original indices
  float* ya[2];
  int* ja[2];
  int cur;         // which of the double buffers is current
  unsigned long long* nnkey;  // [n] per active consumer: key32 bits << 32 | supplier position
  int* cnt;        // [m] consumers per supplier position
  int2* seg;       // [m] (offset, length) of each supplier's group
  int* seglist;    // [m] non-empty groups
  int* biglist;    // [m] groups longer than a warp
  int* medlist;    // [m] groups of 9..32 consumers
  unsigned long long* member;  // [n] group members: key32 bits << 32 | consumer position
  int32_t* fl_i;   // [m+n] flow record of the one-CTA rounds (deferred costing)
  int32_t* fl_j;
  double* fl_f;
  float* kmat;     // d > 8 (nullable): key matrix of the cluster tail
  int* blockcounts;            // compaction scratch
  unsigned long long* xs_acc;  // 4 exact-sum accumulators of XS_LIMBS limbs
  // Early notification of the active counts (nullable): the compaction's
  // count kernel writes {seq, m_t, n_t, error bits} of the round here (host
  // memory mapped into the device) as soon as the counts are known, before
  // the scatter that moves the points has run.
  volatile int* notify;
  int notify_seq;
  DevState* st;
  // caller's plan arrays (nullable) and capacity
  int32_t* plan_i;
  int32_t* plan_j;
  double* plan_f;
  int64_t plan_cap;
};

// rounds.cu ---------------------------------------------------------------
// After the last round: the cost terms and plan entries of every recorded
// flow, R into st->cost and the leftover mass into st->leftover.
void launch_leftover(const SolveBufs& B, cudaStream_t st);
// Exact totals of a and b and their normalisation into B.s / B.c (two
// launches; B.xs_acc cleared by the caller).
void launch_setup_sums(const SolveBufs& B, const double* a, const double* b, cudaStream_t st);
// Initial packing of both sides: active = positive weight, coordinates checked.
int launch_initial_pack(SolveBufs& B, cudaStream_t st);
// One multi-CTA round on the current active lists (mt, nt known on the host).
int launch_big_round(SolveBufs& B, int mt, int nt, long long round, cudaStream_t st);

// lowd.cu ------------------------------------------------------------------
// `grid_work` (nullable): skip the scan where the grid step before it served
// the round (grid_served), else say so in *refused (host memory mapped into the
// device).
int launch_nns_lowd(const SolveBufs& B, int mt, int nt, cudaStream_t st, const unsigned long long* grid_work = nullptr,
                    int* refused = nullptr);

// lowd_grid.cu -------------------------------------------------------------
// Points of the smaller side from which a round takes the grid.  Its four small
// launches and the query take some 50 us and the gaps between them 10 where K1
// takes 82 (just below 16,384 x 16,384 points, d = 3) and 48 (some 13,000 a side),
// and the query's time per warp grows with the larger side alone: few consumers, or few suppliers to sort many consumers for, leave
// it behind K1 (whole solves with the grid from 2^26 pairs on, without and with
// it: 8,192 x 8,192 uniform points d = 2 495 and 527 us, 300,000 x 300 101 and
// 156 ms, 200,000 x 3,000 12.3 and 18.9 ms; 32,768 x 32,768 d = 3 1,170 and 954
// us).
constexpr int64_t GRID_MIN_SIDE = 7 << 11;
size_t grid_cells_bytes();
size_t grid_box_floats(int64_t m);
// The box of the initial active sets (once per solve, before the first grid
// step).
int launch_grid_bounds(const SolveBufs& B, int mt, int nt, cudaStream_t st);
bool grid_nns_wanted(const SolveBufs& B, int mt, int nt);
// Nearest active supplier of every active consumer into B.nnkey, unless the rule
// below sends the round to K1 (launch_nns_lowd with B.grid.work, behind it).
int launch_nns_grid(const SolveBufs& B, int mt, int nt, cudaStream_t st);
// The rule, on the device (what it reads is only known there).  work[0]: points
// that share few cells lie in no order, so every block has to be looked at; known
// before the sort.  work[1]: the (consumer, block) pairs the query has scanned,
// which the cells do not tell (suppliers on a circle around the consumers, two
// sets in different places).  All of them cost about four times K1's scan
// (65,536 points on a circle, d = 2: 5.4 ms with K1, 20.3 with every block
// visited), so a query that is past a sixteenth stops; the keys it has stored
// stay (K1 merges by minima).
NNS_DEV unsigned long long grid_most_visits(int mt, int nt) { return (unsigned long long)mt * (unsigned)nt / (32 * 16); }
NNS_DEV bool grid_served(const unsigned long long* work, int mt, int nt) {
  const ulonglong2 w = __ldcg(reinterpret_cast<const ulonglong2*>(work));
  return w.x <= (unsigned long long)mt * (unsigned)nt / 32 && w.y <= grid_most_visits(mt, nt);
}
// Run all remaining rounds of the current active lists in one CTA.
int launch_finish(const SolveBufs& B, int64_t round_limit, cudaStream_t st);
// The same on a thread-block cluster (k_finish_cl), for active sets of at
// most finish_cluster_cap(d) points per side.  finish_cluster_cap returns 0
// when this device cannot co-schedule the cluster (the one-CTA tail serves).
int finish_cluster_cap(int d, int metric);
int launch_finish_cluster(const SolveBufs& B, int64_t round_limit, cudaStream_t st);
// A whole pair with m, n <= FIN_MAX and d <= 8 in one launch (writes st->cost,
// nnz, rounds, pair_evals, leftover and the plan).
int launch_solve_small(const SolveBufs& B, const double* a, const double* b, cudaStream_t st);

// Batched small pairs (all in one persistent launch), low d.
struct BatchArgs {
  const float* x; const double* a; const int64_t* x_off;
  const float* y; const double* b; const int64_t* y_off;
  const int* pair_ids;   // pairs handled by the CTA solver
  int num;               // number of entries in pair_ids
  int d, metric;
  double* costs;         // [P]
  long long* rounds;     // [P] rounds per pair (nullable)
  long long* pair_evals; // [P] (nullable)
  unsigned* queue;       // work-queue counter (device, zeroed)
  unsigned* err;
  int protocol;          // nnsemd_protocol
  unsigned long long seed;
  int n_shared;          // > 0: every pair's consumers are rows 0..n_shared-1 of y (y_off unused)
  // flow records (nullable): CTA b records a pair's flows in entries
  // [b fl_cap, (b + 1) fl_cap) and costs them once after the pair's last
  // round (d > 8 solvers)
  int32_t* fl_i;
  int32_t* fl_j;
  double* fl_f;
  long long fl_cap;
  // key matrices (nullable; d > 8, FP32): kcap floats per CTA, a multiple of
  // 4, used by the pairs whose matrix (m rows of kmat_ld(n) floats) fits
  float* kmat;
  long long kcap;
  unsigned long long* searches;  // nullable: the consumer searches of all rounds are added here (d > 8, FP32)
};
int launch_batched_lowd(const BatchArgs& A, int grid, cudaStream_t st);
// The same two for pairs of at most LOWD_SMALL_CAP points per side
// (lowd_pairs_small.cu): fewer threads per pair, several pairs per SM.  A
// round of such a pair is barrier and memory latency, which more resident
// pairs hide and more threads lengthen: 2,048 image pairs of 80..400 points
// took 2.01 ms with one 1,024-thread CTA per SM, 881 us with two of 512
// threads, 610 us with four of 256 and 607 us with six of 128; a single
// 256-point pair 84 us at 1,024 threads, 58 at 512, 62 at 256 and at 128.  (The
// single pair takes the batches' 256 threads too: a class of 512 would be sixteen
// instantiations more for 4 us.)
constexpr int LOWD_SMALL_CAP = 512;
constexpr int LOWD_SMALL_THREADS = 256;
constexpr int LOWD_SMALL_PER_SM = 4;
int launch_solve_small_cap(const SolveBufs& B, const double* a, const double* b, cudaStream_t st);
int launch_batched_lowd_small(const BatchArgs& A, int grid, cudaStream_t st);

// highd.cu (d > 8) ---------------------------------------------------------
// FP32 NNS over all active suppliers for the first `ncons` active consumers,
// or, with `cons`, for the consumer positions listed there (count in
// ncons_dev when given, else ncons).  Merges into B.nnkey with atomicMin.
int launch_nns_f32(const SolveBufs& B, int mt, int ncons, const int* cons, const int* ncons_dev, cudaStream_t st);
int launch_finish_hd(const SolveBufs& B, int64_t round_limit, cudaStream_t st);
// All remaining rounds on a thread-block cluster (two launches), for active
// sets of at most FIN_MAX_HD points per side, where finish_hd_cluster_ready
// (the key matrix is laid out and the device co-schedules the cluster).
bool finish_hd_cluster_ready(const SolveBufs& B);
int launch_finish_hd_cluster(const SolveBufs& B, int mt, int nt, int64_t round_limit, cudaStream_t st);
int launch_batched_hd(const BatchArgs& A, int grid, cudaStream_t st);
// Batched FP32 solver for pairs of at most HD_SMALL_CAP points per side
// (d > 8), HD_SMALL_THREADS threads per pair, several pairs per SM.
constexpr int HD_SMALL_CAP = 512;
constexpr int HD_SMALL_THREADS = 256;
int launch_batched_hd_small(const BatchArgs& A, int grid, cudaStream_t st);
// All d coordinates of both sides finite (else EF_NONFINITE).
void launch_check_finite(const float* v, int64_t count, unsigned* err, cudaStream_t st);

// tc.cu (reduced precision, d > 8, squared-Euclidean order) ----------------
size_t tc_kb(int d, int precision);  // packed bytes per row
int tc_bn(size_t kb);                // supplier rows per tile
bool tc_supported(int d, int precision);  // the operand tiles of K2 fit its shared memory

// A BF16 linear layer on the tensor cores (tc.cu): Z [rows][N] = X W^T + b
// with FP32 accumulation, X [rows][K] and W [N][K] packed by
// pack_rows_bf16 into linear_tc_packed_bytes(rows, K) bytes each; K a
// multiple of 16 up to 256 (linear_tc_supported).  A wait that gives up
// sets EF_TIMEOUT in *err.
bool linear_tc_supported(int K);
size_t linear_tc_packed_bytes(int rows, int K);
int pack_rows_bf16(const float* src, int rows, int K, uint8_t* out, cudaStream_t st);
int linear_tc(const uint8_t* X, int rows, int K, const uint8_t* W, const float* bias, int N, float* Z, unsigned* err,
              cudaStream_t st);
// The same layer with ReLU, written as the next layer's packed X (BF16,
// tiles of 128 rows, padding rows zero; N a multiple of 16).
int linear_tc_pack_relu(const uint8_t* X, int rows, int K, const uint8_t* W, const float* bias, int N, uint8_t* out,
                        unsigned* err, cudaStream_t st);
// The same layer reduced per row: out[row] = the column of the row's largest
// value of X W^T + b (lowest column on ties); part holds rows x
// ceil(N / 128) partial keys.
int linear_tc_argmax(const uint8_t* X, int rows, int K, const uint8_t* W, const float* bias, int N,
                     unsigned long long* part, int* out, unsigned* err, cudaStream_t st);
// Lower bounds of the squared distance from each row y of [rows][d] to any
// point of each cell (centre mu_c, radius r_c): out[row][c] =
// max(0, |y - mu_c| - r_c)^2 with |y - mu_c| bounded from below through a
// BF16X3 contraction and its error bound, rounded toward the bound.  The
// cells are packed once (cell_bounds_tc_cells: packed into
// linear_tc_packed_bytes(cells, 3d) bytes, |mu|^2 down and |mu| up); the
// rows use scratch of linear_tc_packed_bytes(rows, 3d) bytes and 2 x rows
// floats.  d a multiple of 16 with 3d <= 256 (cell_bounds_tc_supported).
bool cell_bounds_tc_supported(int d);
int cell_bounds_tc_cells(const float* mu, int cells, int d, uint8_t* packed, float* sq_lo, float* nrm_up,
                         cudaStream_t st);
int cell_bounds_tc(const float* y, int rows, int d, uint8_t* packed_y, float* y_sq_lo, float* y_nrm_up,
                   const uint8_t* packed_mu, const float* mu_sq_lo, const float* mu_nrm_up, const float* radius,
                   int cells, float* out, unsigned* err, cudaStream_t st);
// NNS of every active consumer: tensor-core candidates, exact FP32 re-rank,
// certificate, FP32 rescan of the rest.  Writes B.nnkey (must be all ones).
int launch_nns_tc(const SolveBufs& B, const TcBufs& T, int mt, int nt, int precision, cudaStream_t st,
                  const int* sel = nullptr, const int* nsel_dev = nullptr);
// Answers what it can of a round from B.lists (two launches); the other
// consumers' positions go to B.lists.sel, their number to *B.lists.nsel.
int launch_serve_lists(const SolveBufs& B, int mt, int nt, cudaStream_t st);
// Consumers at or below which a full scan runs in FP32 rather than on the
// tensor cores (packing every active supplier costs more).
constexpr int TC_SCAN_MIN = 256;
void launch_add_count(unsigned long long* ctr, unsigned long long v, cudaStream_t st);

// batched_tc.cu: batches of pairs with up to `cap` points per side (FIN_MAX_HD;
// batched_tc_max_stages also answers for HD_SMALL_CAP, 0: rows too long),
// reduced-precision NNS inside each pair's CTA.
// kc_cap: values of each CTA's distance cache (pairs whose
// batched_tc_cache_values fit are answered from it after their first round; 0
// turns it off).
long long batched_tc_cache_values(long long m, long long n);
size_t batched_tc_slot_bytes(int cap, int kb, int bn, long long kc_cap);
int batched_tc_max_stages(int cap, int kb, int bn, int precision);
// rerank_k: candidates re-ranked per consumer (1..8; other values: 8);
// certified / fallbacks / near_ties: device counters the launch adds to.
int launch_batched_tc(const BatchArgs& base, int precision, int cap, int kb, int bn, int nstage, uint8_t* scratch,
                      size_t slot_bytes, unsigned long long* certified, unsigned long long* fallbacks,
                      unsigned long long* near_ties, int rerank_k, long long kc_cap, int grid, cudaStream_t st);

}  // namespace nnsemd
