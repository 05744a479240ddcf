// Internal host-side interfaces between the translation units of the library.
#pragma once

#include <cstdint>
#include <cuda_runtime.h>

#include "kk_spgemm.h"

namespace kk {

// Per-kernel CUDA-event timer (enabled by options.timing).
struct KernelTimer;
void timer_begin(KernelTimer* t, cudaStream_t s, const char* name);
void timer_end(KernelTimer* t, cudaStream_t s);

// Bit vectors of wide-tier rows kept by the symbolic phase for the numeric
// phase of the same arrays: rows whose nnz(C(i,:)) exceeds min_cnt get a slot
// of `stride` u32 (the bits, then the chunk table) when one is left.  With
// tasks (sorted B) the numeric phase computes them chunk by chunk
// (k_num_chunk); without, the wide kernel loads their bits.
struct WideKeep {
  uint32_t* bits;     // max_slots slots
  int32_t* slot;      // per row: slot or -1
  int32_t* next;      // [0] slots, [1] tasks, [2] tasks claimed by the numeric phase, [3] indexed rows of B
  int2* tasks;        // (row, chunk), max_tasks of them; null: no tasks
  int* kept;          // += rows kept with tasks
  const int32_t* bidx;  // index slot of every row of B (-1: none)
  const int32_t* btab;  // tab_stride positions per slot
  int32_t tab_stride;
  int32_t shift;        // chunks end at multiples of 2^shift columns
  int32_t max_slots;  // 0: nothing kept / nothing to use
  int32_t min_cnt;
  int32_t stride;
  int32_t max_chunks;  // chunk table entries of a slot
  int32_t max_tasks;
};

// Compressed B (the paper's B_C): row j of B as (column >> 5, 32-bit column
// mask) pairs in column order, stored at B's own row offsets
// bc[B.rowptr[j] .. B.rowptr[j] + len[j]).  Built only for sorted B.
struct BComp {
  const int2* bc;
  const int32_t* len;
};

struct LaunchCtx {
  cudaStream_t stream;
  KernelTimer* timer;  // may be null
  int* status;         // device status word
  int num_sms;
  int max_smem_optin;
  const int32_t* row_lo;  // first column of each row's span window (window tier)
  const long long* flop;  // flop bound of each row (wide tier)
  WideKeep keep;          // kept wide-tier bit vectors (wide tier)
  int debug_checks;       // options.debug_checks
  int stage_long_rows;    // options.stage_long_rows (wide symbolic: bulk-copy staging)
  // structure fingerprints of the index arrays at the symbolic call ([0]) and
  // at this numeric call ([1]); null when the kept structure is not in use
  const unsigned long long* fingerprint;
  // 1: the window and rank tiers' rows run in float64 whatever the call's
  // arithmetic (options.arith = AUTO: on GB300 native float64 measured faster
  // there, 1.91 ms against 2.42 for the 27-point value pass)
  int kept_f64;
  BComp bcomp;  // compressed B, when the call has it (wide symbolic)
};

struct CsrView {
  int32_t m, n, nnz;
  const int32_t* rowptr;
  const int32_t* colind;
  const double* vals;
  // Jacobi-fused numeric phase (null otherwise): row i of A enters the product
  // as jac_s[i] * A(i,:) plus 1 at entry jac_p[i] (the row's first diagonal
  // entry), i.e. as row i of I - omega D^-1 A, without a scaled copy of A.  The
  // thread tier forms s_i and that position from the row itself with
  // jac_omega; the other tiers' rows get them from a row-scale kernel.
  const double* jac_s;
  const int32_t* jac_p;
  double jac_omega;
};

#ifdef __CUDACC__
// Row i's Jacobi scaling (loaded once per row): on = false for the plain product.
struct ARowScale {
  double s;
  int p;
  bool on;
};
__device__ __forceinline__ ARowScale a_row_scale(const CsrView& A, int i) {
  ARowScale r{1.0, -1, A.jac_s != nullptr};
  if (r.on) {
    r.s = A.jac_s[i];
    r.p = A.jac_p[i];
  }
  return r;
}
// Value of A's entry p as the numeric phase multiplies it: the stored value v,
// or for the Jacobi-fused product s_i * v (+ 1 at the row's first diagonal
// entry), formed once per A entry as it is loaded.
__device__ __forceinline__ double a_scaled(const ARowScale& r, int p, double v) {
  return r.on ? (p == r.p ? fma(r.s, v, 1.0) : r.s * v) : v;
}
__device__ __forceinline__ double a_value(const CsrView& A, int i, int p) {
  return a_scaled(a_row_scale(A, i), p, A.vals[p]);
}
#endif

// Accumulator tiers.  In statistics the thread tier counts as the team tier, the
// rank tier as the window tier.
enum Tier : int32_t { kTierTeam = 0, kTierCta = 1, kTierDense = 2, kTierWindow = 3, kTierThread = 4, kTierRank = 5 };
__host__ __device__ constexpr int32_t stat_tier(int32_t t) {
  return t == kTierThread ? kTierTeam : t == kTierRank ? kTierWindow : t;
}

// Thread tier (kk_thread.cu): one thread per row, accumulator in registers.
constexpr int kThreadSymMax = 16;     // symbolic rows: flop bound <= this
constexpr int kThreadNumMax = 8;      // numeric rows: nnz(C(i,:)) <= this ...
constexpr int kThreadNumMaxFlop = 64; // ... and flop bound <= this
// Small products (kk_small.cu): one launch per phase, a thread per row, for A
// with at most options.small_max_rows rows (at most kSmallMaxRowsCap), C rows
// of at most kSmallN columns, tried when A's rows average at most
// kSmallMaxMeanFlop products.
constexpr int kSmallThreads = 256;     // symbolic CTA
constexpr int kSmallNumThreads = 64;   // numeric CTA (more CTAs for a few thousand rows)
constexpr int kSmallMaxRowsCap = 8192;
constexpr int kSmallN = 16;
constexpr int kSmallMaxMeanFlop = 32;

// Window tier: a row whose columns of C all lie in [row_lo, row_lo + W) gets a
// dense bit vector of W bits (plus per-word ranks in the numeric phase).
constexpr int kNumWindowClasses = 5;
constexpr int32_t kWindowBits[kNumWindowClasses] = {4096, 12288, 24576, 40960, 65536};
__host__ __device__ constexpr int32_t window_bits(int w) {
  return w == 0 ? 4096 : w == 1 ? 12288 : w == 2 ? 24576 : w == 3 ? 40960 : 65536;
}
constexpr int32_t kWindowMaxNnz = 256;   // numeric window rows: nnz(C(i,:)) <= this
constexpr int32_t kWindowFlopRatio = 128;  // window used only when W <= ratio * flop
// Symbolic rows of a narrow B (k <= 65,536) with more than kWindowMaxFlop products
// leave the window tier, because the wide tier's chunks serve their numeric phase
// (60,000 random rows of 4,900 products: 2.9 ms, 7.9 without) - but for rows with
// few columns, whose numeric phase is the kept rows' or the rank tier's either way:
// those of a span up to kWindowFreeSpan, and those whose B rows hold kWindowDense
// columns or more to a word, while the pairs that the window's warp walks are no
// more than kWindowMaxFlop.  (Rows of small dense blocks, 81 x 81: 6,561 products,
// 283 pairs.  59,940 of them, both phases: 1.50 ms in the window, 4.43 in the wide
// tier without kept structure.)  Power-law rows have 2 to 5 columns to a word: all
// of them by their pairs took the scale-15 R-MAT square from 1.98 to 2.62 ms, those
// of 4 or more to 2.09.
constexpr long long kWindowMaxFlop = 4096;
constexpr int32_t kWindowFreeSpan = 1024;
constexpr int kWindowDense = 6;

// Rank tier (kk_rank.cu): numeric rows without kept structure, nnz(C(i,:)) at
// most kRankNnz[2], span at most kRankBits of the bin; symbolic rows of an
// unsorted B (span: B's columns).
constexpr int kNumRankBits = 5, kNumRankNnz = 3;
constexpr int32_t kRankBits[kNumRankBits] = {4096, 8192, 16384, 32768, 65536};
constexpr int32_t kRankNnz[kNumRankNnz] = {256, 512, 1024};
// Rank tier used only when W <= kRankFlopRatio * flop, and for rows of at most
// kRankMinNnz columns when W <= kWindowFlopRatio * flop: short rows share a warp
// in the thread and team tiers (262,144 rows of 7 columns over 8,200: 130 us in
// the team tier, 400 in the rank tier).
constexpr int32_t kRankFlopRatio = 512;
constexpr int32_t kRankMinNnz = 32;
// ... and (automatic tiers) only for rows of more columns (numeric) or products
// (symbolic) than these, where the window is wider than the first class and than
// kRankShortBits: fewer are done sooner by hash.  300,000 rows, hash and rank: 36
// columns in 8,192 580 and 465 us, in 16,384 595 and 501; 63 columns in 32,768 650 and
// 798; 9-point rows of a 1,080 x 614 grid, 25 columns of 81 products in 4,325, 837 and
// 1,054; symbolic 36 products of an unsorted B 225 and 305, 49 products 275 and 280,
// 100 products 357 and 265.
constexpr int32_t kRankShortBits = 16384, kRankWideMinNnz = 64, kRankMinFlop = 56;
// Symbolic rank rows: flop bound <= this, the line of the window tier for a B as
// narrow; heavier rows are too many products for one warp and stay where they were.
constexpr long long kRankMaxFlop = 4096;
static_assert(kWindowFreeSpan <= kRankNnz[kNumRankNnz - 1], "their numeric phase is the rank tier's or the kept rows'");
constexpr int kMaxWindowBins = kNumWindowClasses + kNumRankBits * kNumRankNnz;

// Per-row structure kept by the symbolic window kernel for the numeric phase
// of the same A and B: the row's non-empty window words (index relative to
// the word of row_lo, at most kCacheWords) and their bits; n[i] = number of
// words, -1 if the row has no kept structure.
constexpr int kCacheWords = 64;
struct WinCache {
  uint16_t* w;
  uint32_t* m;
  int32_t* n;
  unsigned long long* kept;  // += rows whose structure was kept
};
struct WinCacheView {
  const uint16_t* w;
  const uint32_t* m;
  const int32_t* n;
};
// One bin of rows: its tier and the accumulator geometry.
struct BinSpec {
  int32_t tier;
  int32_t team;   // lanes per row (team tier); threads per CTA otherwise
  int32_t slots;  // hash slots (team / CTA tiers); chunk width in columns (dense)
  int32_t flat;   // 1: lanes walk the flattened (A entry, B entry) products
  int64_t lo, hi; // bin range of the binning quantity (flop or nnz), inclusive
};

// Sparse matrix addition (kk_spadd.cu): symbolic counts, and what the numeric phase
// goes by: per row its kind, and (in apos and bpos) its bits or its entries' slots in C
// (long_rows: a list of up to m rows, its count in the first element, zeroed by the
// caller; kinds: whether there are rows for teams, warps and CTAs, on the device, zeroed
// by the caller); numeric writes C's columns and values (kinds: on the
// host).
cudaError_t launch_spadd_symbolic(const LaunchCtx& ctx, const CsrView& A, const CsrView& B, int32_t* cnt,
                                  int32_t* apos, int32_t* bpos, uint8_t* kind, int32_t* long_rows, int32_t* kinds);
cudaError_t launch_spadd_numeric(const LaunchCtx& ctx, const CsrView& A, const CsrView& B, double alpha,
                                 double beta, const int64_t* c_rowptr, const int32_t* apos,
                                 const int32_t* bpos, const uint8_t* kind, const int32_t* long_rows,
                                 const int32_t* kinds, int32_t* c_colind, double* c_vals);

// Numeric phase of window rows with kept structure (kk_kept.cu).
cudaError_t launch_num_kept(const LaunchCtx& ctx, const CsrView& A, const CsrView& B,
                            const WinCacheView& cache, const float2* b_split, const int32_t* b_range_bad,
                            int32_t arith, const int64_t* c_rowptr, const int32_t* rows, int32_t nrows,
                            int32_t* c_colind, double* c_vals);

// Symbolic phase of the rank tier's rows (unsorted B): window of bin.slots columns.
cudaError_t launch_sym_rank(const LaunchCtx& ctx, const BinSpec& bin, const CsrView& A, const CsrView& B,
                            const int32_t* rows, int32_t nrows, int32_t* cnt);

// Numeric phase of the rank tier's rows (kk_rank.cu): window of bin.slots
// columns, at most bin.hi columns of C per row.
cudaError_t launch_num_rank(const LaunchCtx& ctx, const BinSpec& bin, const CsrView& A, const CsrView& B,
                            int32_t b_sorted, const BComp& bcomp, const float2* b_split,
                            const int32_t* b_range_bad, int32_t arith, const int64_t* c_rowptr,
                            const int32_t* rows, int32_t nrows, int32_t* c_colind, double* c_vals);

// Analysis kernels: rows of more than kLongRow entries, listed for a second
// launch with a warp per row (rows null: no list).
constexpr int kLongRow = 512;
struct LongRows {
  int32_t* rows;
  int32_t* count;
  int32_t most;
};

// Analysis of B (kk_analyze.cu): clears *sorted_flag unless every row is
// strictly ascending, sets KK_ERR_BAD_INDEX on out-of-range structure, and,
// when bc is non-null, writes the compressed rows (pairs counted into *pairs).
cudaError_t launch_analyze_b(const LaunchCtx& ctx, const CsrView& B, int32_t* sorted_flag,
                             int2* bc, int32_t* len, unsigned long long* pairs, const LongRows& lr);

// Arithmetic mode for the numeric kernels.
enum ArithMode : int32_t { kArithF64 = 1, kArithDF32 = 2 };

// Column chunks only where B has at most this many columns: R-MAT square of scale 19
// (2^19 columns) 91.0 ms with them, 102.1 with one CTA per row; of scale 20 296.5 and
// 273.0 (chunks also end every 65,536 columns, so a wide B has more of them per row,
// and each walks all of the row's entries of A).
constexpr int32_t kChunkMaxCols = 1 << 19;
// Defaults of options.sym_team_max_flop and options.num_team_max_nnz: with these the
// lines to the chunks are the library's, any other value holds as it was given.
constexpr int32_t kSymTeamMaxFlop = 3072, kNumTeamMaxNnz = 1024;
// Sorted B: symbolic rows of more than kKeepEarlyFlop products that the wide tier
// would keep (wide_keep_min_flop) leave the team tier for it, because its chunks
// serve their numeric phase.
constexpr long long kKeepEarlyFlop = 512;
// Products from which k_sym_wide keeps a row's bits for chunk tasks: fewer leave
// most words empty, and it walks a summary instead.  Measured with the line above,
// R-MAT squares of scale 18 and 19: words / 4 and 768 30.4 and 92.6 ms, words / 11
// and 768 28.7 and 91.7, words / 16 and 512 28.5 and 91.0, words / 24 and 384 28.4
// and 90.8 (hardly less, for more rows to hold).  A row has a chunk for every 2,048
// words at least, and each walks all of its entries of A: beyond five of them (k >
// 327,680) spread rows of words / 16 products are the hash kernels' (both phases of
// random rows, hash and chunks: k = 520,000, 1,089 products 55.4 and 71.1 ms, 1,600
// products 72.5 and 74.6, 2,116 products 84.3 and 77.8; k = 400,000, 1,296 products
// 45.3 and 48.7, 1,764 products 57.1 and 51.2; k = 300,000, 900 products 39.5 and
// 25.4), so the line is words / 8 there.
__host__ __device__ inline int wide_keep_min_flop(int words) { return words <= 10240 ? words / 16 : words / 8; }
// Rows whose products outnumber the pairs of their B rows (by 9 to 4, of few pairs
// by 7 to 4) stay in the team tier up to kSymTeamMaxFlop products: runs of
// neighbouring columns mostly meet in few columns of C, too few for chunks (27-point
// rows of a 200 x 200 x 3 grid, 567 products in 75 columns, 2.45 to 2.8 products to
// a pair: symbolic phase 0.43 ms by hash, 0.52 in the wide tier; 250 x 250 x 4 0.60
// and 1.13; 1.8 products to a pair in at most 405 pairs where a grid's lines put the
// runs across words). Power-law rows of 513 to 3,072 products have 1.2 to 2.1 to a
// pair, those of at most 384 pairs under 1.7.
constexpr int kKeepFewPairs = 416;
__host__ __device__ inline bool wide_spread_row(long long flop, long long pairs) {
  return flop * 4 < pairs * (pairs <= kKeepFewPairs ? 7 : 9);
}

// Symbolic launch: rows[0..nrows) of A (a device array) get cnt[i] = nnz(C(i,:)).
cudaError_t launch_symbolic_bin(const LaunchCtx& ctx, const BinSpec& bin, const CsrView& A,
                                const CsrView& B, int32_t b_sorted, const int32_t* rows,
                                int32_t nrows, int32_t* cnt);

// Numeric launch.  b_split: B's values pre-split into DF32 pairs (float2), used
// when arith == kArithDF32 and *b_range_bad == 0 (read on the device).
cudaError_t launch_numeric_bin(const LaunchCtx& ctx, const BinSpec& bin, const CsrView& A,
                               const CsrView& B, int32_t b_sorted, const float2* b_split,
                               const int32_t* b_range_bad, int32_t arith,
                               const int64_t* c_rowptr, const int32_t* rows, int32_t nrows,
                               int32_t* c_colind, double* c_vals, int32_t debug_checks);

// Wide tier (kk_wide.cu): CTA-per-row bit vector over all k columns, used for
// the CTA and dense bins when it fits in shared memory.
bool wide_symbolic_fits(const LaunchCtx& ctx, int32_t k);
int32_t wide_word_count(int32_t k);                           // words of a k-bit vector
int32_t wide_keep_min_cnt(const LaunchCtx& ctx, int32_t k);  // rows above this go to C by atomics
bool wide_numeric_fits(const LaunchCtx& ctx, int32_t k);
cudaError_t launch_symbolic_wide(const LaunchCtx& ctx, const CsrView& A, const CsrView& B,
                                 const long long* flop, const int32_t* rows, int32_t nrows,
                                 int32_t* cnt, bool light);
cudaError_t launch_numeric_wide(const LaunchCtx& ctx, const CsrView& A, const CsrView& B,
                                const int64_t* c_rowptr, const int32_t* rows, int32_t nrows,
                                int32_t* c_colind, double* c_vals, long long max_nnz);
// The rows kept with tasks by the symbolic phase (ctx.keep), and the index of B's
// longer rows that their numeric phase uses.
int32_t wide_chunk_shift(int32_t k);
int32_t wide_max_chunks(int32_t k);                                       // of a row of k columns
long long wide_slot_tasks(int32_t k);                    // tasks that a row needs whatever its columns
long long wide_column_tasks(int32_t k, long long flops);  // further tasks of rows with `flops` products together
int32_t wide_index_stride(int32_t k);
int32_t wide_index_rows(const CsrView& B);  // rows of B worth an index, at most
cudaError_t launch_chunk_index(const LaunchCtx& ctx, const CsrView& B, int32_t max_rows, int32_t* slot, int32_t* row,
                               int32_t* tab);
// (fp: structure fingerprints of the symbolic call and of this one).
cudaError_t launch_num_chunk(const LaunchCtx& ctx, const CsrView& A, const CsrView& B, const unsigned long long* fp,
                             const int64_t* c_rowptr, int32_t* c_colind, double* c_vals);

cudaError_t launch_symbolic_thread(const LaunchCtx& ctx, const CsrView& A, const CsrView& B,
                                   const int32_t* rows, int32_t nrows, int32_t* cnt, long long max_flop);
cudaError_t launch_small_symbolic(const LaunchCtx& ctx, const CsrView& A, const CsrView& B, int64_t* c_rowptr,
                                  int32_t* cnt, int32_t* flags, long long* out);
cudaError_t launch_small_numeric(const LaunchCtx& ctx, const CsrView& A, const CsrView& B,
                                 const int64_t* c_rowptr, int32_t* c_colind, double* c_vals);
cudaError_t launch_numeric_thread(const LaunchCtx& ctx, const CsrView& A, const CsrView& B,
                                  const int64_t* c_rowptr, const int32_t* rows, int32_t nrows,
                                  int32_t* c_colind, double* c_vals, long long max_nnz);

// Window-tier launches (kk_window.cu).
cudaError_t launch_symbolic_window(const LaunchCtx& ctx, const BinSpec& bin, const CsrView& A,
                                   const CsrView& B, const BComp& bcomp, const int32_t* rows,
                                   int32_t nrows, int32_t* cnt, const WinCache& cache);
// Speculative one-pass (learned form) over rows whose predicted table is
// 2^log2s slots (log2s in 5..9); see k_num_warp_vec<LOG2S, true>.
cudaError_t launch_onepass(const LaunchCtx& ctx, int32_t log2s, const CsrView& A, const CsrView& B,
                           const float2* b_split, const int32_t* b_range_bad, int32_t arith,
                           const int64_t* soff, const int32_t* rows, int32_t nrows, int32_t* scol,
                           double* sval, int32_t* cnt_out);

// Learned form (kk_learned.cu).  Rows predicted to need at most
// 16 << (kOnepassClasses - 1) entries take the speculative one-pass.
constexpr int kOnepassClasses = 5;
// Learned bins: [0, kOnepassClasses) hash one-pass by capacity class,
// [kOnepassClasses, kLearnedHeavy) window one-pass by window class,
// kLearnedHeavy = plain path.
constexpr int kLearnedHeavy = kOnepassClasses + kNumWindowClasses;
// Speculative one-pass for window rows through a word table (kk_onepass.cu).
cudaError_t launch_onepass_table(const LaunchCtx& ctx, const CsrView& A, const CsrView& B,
                                 const BComp& bcomp, const float2* b_split,
                                 const int32_t* b_range_bad, int32_t arith, const int64_t* soff,
                                 const int32_t* cap, const int32_t* rows, int32_t nrows,
                                 int32_t* scol, double* sval, int32_t* cnt_out);
cudaError_t launch_learned_classify(const LaunchCtx& ctx, const CsrView& A, int32_t bn,
                                    const int32_t* b_sorted, int32_t use_window, int32_t window_onepass,
                                    const float* params,
                                    float quantile, int32_t use_pred, const long long* flop,
                                    const int32_t* row_span, const int2* stat, uint8_t* lbin, int32_t* cap);
cudaError_t launch_learned_leftover(const LaunchCtx& ctx, int32_t m, const uint8_t* lbin,
                                    const int32_t* cnt, uint8_t* plain, const uint8_t* sbin_all,
                                    uint8_t* sbin);
cudaError_t launch_mask_bins(const LaunchCtx& ctx, int32_t m, const uint8_t* plain,
                             const uint8_t* nbin, uint8_t* out);
cudaError_t launch_copy_staged(const LaunchCtx& ctx, int32_t m, const uint8_t* lbin,
                               const uint8_t* plain, const int64_t* soff, const int64_t* rowptr,
                               const int32_t* scol, const double* sval, int32_t* ccol,
                               double* cval);

// Batched form (kk_batched.cu).
struct PairDesc {
  CsrView A, B;
  long long row_base;    // first global row of this pair
  long long split_base;  // first DF32 pair of B's values in the split buffer
  int32_t b_sorted;      // set on the device
  int32_t range_bad;     // set on the device (values outside the DF32 window)
};
constexpr int kMaxBBins = 24;
struct BBinTable {
  int32_t nb;
  int32_t kind[kMaxBBins];   // 0 warp, 1 CTA
  int32_t log2s[kMaxBBins];
  int32_t flat[kMaxBBins];
  long long hi[kMaxBBins];
};
void batched_bin_tables(BBinTable& sym, BBinTable& num, int sym_load_pct, int num_load_pct);
// Packed batch (block-diagonal A and B for the plain kernels); base holds per
// pair the A rows, A entries, B rows and B entries that precede it.
cudaError_t launch_b_pack(cudaStream_t s, int32_t count, const PairDesc* d,
                          const long long* base, bool vals_only, int32_t* pa_rp, int32_t* pa_ci,
                          double* pa_v, int32_t* pb_rp, int32_t* pb_ci, double* pb_v, long long RA,
                          long long NA, long long RB, long long NB);
cudaError_t launch_b_prepare(cudaStream_t s, int num_sms, int32_t count, PairDesc* d, long long R,
                             int32_t* row_pair, int* status);
cudaError_t launch_b_analyze_a(cudaStream_t s, int num_sms, long long R, const PairDesc* d,
                               const int32_t* row_pair, const BBinTable& tab, int32_t vec_min_len,
                               long long* flop, uint8_t* bin, unsigned long long* total_flop, int* status);
cudaError_t launch_b_nclassify(cudaStream_t s, int num_sms, long long R, const PairDesc* d,
                               const int32_t* row_pair, const int64_t* rowptr, const long long* flop,
                               const BBinTable& tab, int32_t vec_min_len, uint8_t* bin, int* status);
cudaError_t launch_b_symbolic(const LaunchCtx& ctx, const PairDesc* d, const int32_t* row_pair,
                              const int32_t* rows, const int32_t* bin_start, int32_t* tile_prefix,
                              const BBinTable& tab, int* queue, int32_t* cnt);
cudaError_t launch_b_numeric(const LaunchCtx& ctx, int32_t count, PairDesc* d, const int32_t* row_pair,
                             const int32_t* rows, const int32_t* bin_start, int32_t* tile_prefix,
                             const BBinTable& tab, int* queue, int32_t arith, float2* split,
                             const int64_t* rowptr, int32_t* ccol, double* cval);
cudaError_t launch_b_offsets(cudaStream_t s, int32_t count, const PairDesc* d, long long R,
                             const int64_t* rowptr, int64_t* off);

// Row features (kk_mlp.cu); mm is scratch int2[B.m].
cudaError_t launch_row_features(cudaStream_t s, const CsrView& A, const CsrView& B, int2* mm,
                                float* feat, int num_sms);

// Shared-memory bytes a bin's kernel needs per CTA (0 if it does not fit).
size_t symbolic_smem_bytes(const BinSpec& bin);
size_t numeric_smem_bytes(const BinSpec& bin);

}  // namespace kk
