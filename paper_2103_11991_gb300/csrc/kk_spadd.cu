// Sparse matrix addition C = alpha A + beta B (Kokkos Kernels paper, Sec.
// "SpAdd"), symbolic and numeric phases.
//
// Rows that are strictly ascending in both matrices, of up to kAddWarpMax combined
// entries, are merged by binary search of each entry in the other row.  While both rows
// fit a team of 8, 16 or 32 lanes the search goes through shuffles and nothing is kept
// between the phases: the symbolic phase counts the shared columns, the numeric phase
// searches again, which costs less than writing and reading a slot per entry.  Longer
// rows are staged in shared memory by a warp, and their merged order is kept as bits:
// which slots of C's row hold an entry of A, and which of A's entries share their
// column with one of B; the numeric phase reads each entry once, in C's order.
// What bounds it: the latency of a row's two dependent loads, so each kind of row has a
// numeric kernel of its own with registers for 64 warps on an SM, and the float64 pipe
// (two multiplications a row; sums are left to L2).  Two matrices of 500,000 rows of 30,
// both phases: 546 us with a slot per entry for every row (and C zeroed and added to by
// atomics), 337 when one kernel with registers for 40 warps took all kinds, 305 now.
// The numeric phase alone was slower than by slots there; slots, one kernel, now:
// 27-point rows of 512,000 plus themselves 142, 194, 151 us; 400,000 rows of 20 plus
// rows of 2 128, 146, 132; 50,000 rows of 100 94, 114, 84; 100 rows of 3,000 (a CTA
// each now) 60, 107, 26.
//
// Other rows: the entries of A and B become 64-bit keys
// (column << 32 | source bit (B) << 31 | index within the source row) in
// shared memory and are sorted by a bitonic network; equal columns are then
// adjacent, so a scan of "first of its column" flags gives nnz(C(i,:)) and, for
// every entry of A and of B, its slot in the row of C (the paper's Apos and
// Bpos; kAddLater marks all but the first entry of a column).  When both rows
// are sorted (repeats allowed) the keys are laid out as A ascending, then padding,
// then B descending: a bitonic sequence, so only the final merge stage runs (the
// paper's sorted-input method); otherwise the full sort runs (its unsorted-input
// method).  Rows of up to kAddWarpMax combined entries take one warp, rows of up to
// kAddCtaMax one CTA of 1024 threads; longer rows are reported as KK_ERR_CAPACITY.
// Their numeric phase stores the first entry of every column with its value and adds
// the others to it (float64 atomics: repeated columns are added in no fixed order).
#include "kk_internal.h"
#include "kk_device.cuh"

namespace kk {
namespace {

using u64 = unsigned long long;
constexpr unsigned kFull = 0xffffffffu;
constexpr int kAddWarpMax = 256;
constexpr int kAddCtaMax = 8192;
constexpr int kAddCtaThreads = 1024;
constexpr u64 kAddPad = ~0ull;
constexpr int kAddLater = (int)0x80000000u, kAddSlot = 0x7fffffff;
// How the numeric phase takes a row: through slots by a warp or (kAddByCta) a CTA,
// merged by a team (kAddSame: the same columns in both matrices), or through bits (kept
// in the place of the row's slots) by a warp.
constexpr uint8_t kAddBySlots = 0, kAddByTeam = 1, kAddByBits = 2, kAddByCta = 3, kAddSame = 4;

__device__ __forceinline__ int next_pow2(int x) {
  int n = 32;
  while (n < x) n <<= 1;
  return n;
}

// Exclusive scan of v over the CTA (blockDim.x a multiple of 32, at most 1024);
// *total receives the sum.  scratch: 33 ints of shared memory.
__device__ __forceinline__ int add_block_scan(int v, int* scratch, int* total) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int nw = blockDim.x >> 5;
  const int incl = team_inclusive_scan<32>(v, lane, kFull);
  if (lane == 31) scratch[warp] = incl;
  __syncthreads();
  if (warp == 0) {
    const int w = lane < nw ? scratch[lane] : 0;
    const int wi = team_inclusive_scan<32>(w, lane, kFull);
    if (lane < nw) scratch[lane] = wi - w;
    if (lane == 31) scratch[32] = wi;
  }
  __syncthreads();
  const int r = scratch[warp] + incl - v;
  *total = scratch[32];
  __syncthreads();
  return r;
}

// Bitonic sort (merge_only: the final merge of an already bitonic sequence) of
// key[0, n), n a power of two, by NT cooperating threads (32: one warp, else the
// whole CTA).
template <int NT>
__device__ __forceinline__ void add_sort(u64* key, int n, int tid, bool merge_only) {
  for (int k = merge_only ? n : 2; k <= n; k <<= 1) {
    for (int j = k >> 1; j > 0; j >>= 1) {
      for (int t = tid; t < n; t += NT) {
        const int l = t ^ j;
        if (l > t) {
          const u64 a = key[t], b = key[l];
          const bool up = (t & k) == 0;
          if ((a > b) == up) {
            key[t] = b;
            key[l] = a;
          }
        }
      }
      if (NT == 32) __syncwarp();
      else __syncthreads();
    }
  }
}

// Keys of row r into key[0, n): A at [0, la), padding, B reversed at [n - lb, n).
// Returns (by reference) whether both rows are non-decreasing and whether a
// column lies outside [0, ncols).
template <int NT>
__device__ __forceinline__ void add_load(const CsrView& A, const CsrView& B, int pa, int la, int pb,
                                         int lb, int n, u64* key, int tid, int& unsorted, int& bad) {
  for (int t = tid; t < n; t += NT) key[t] = kAddPad;
  if (NT == 32) __syncwarp();
  else __syncthreads();
  for (int t = tid; t < la; t += NT) {
    const int c = A.colind[pa + t];
    if ((unsigned)c >= (unsigned)A.n) bad = 1;
    if (t > 0 && A.colind[pa + t - 1] > c) unsorted = 1;
    key[t] = ((u64)(uint32_t)c << 32) | (u64)t;
  }
  for (int t = tid; t < lb; t += NT) {
    const int c = B.colind[pb + t];
    if ((unsigned)c >= (unsigned)B.n) bad = 1;
    if (t > 0 && B.colind[pb + t - 1] > c) unsorted = 1;
    key[n - 1 - t] = ((u64)(uint32_t)c << 32) | (1ull << 31) | (u64)t;
  }
}

// First index in the sorted row x[0, len) whose column is >= c.
__device__ __forceinline__ int add_lower_bound(const int32_t* x, int len, int c) {
  int lo = 0, hi = len;
  while (lo < hi) {
    const int mid = (lo + hi) >> 1;
    if (x[mid] < c) lo = mid + 1;
    else hi = mid;
  }
  return lo;
}

struct AddRow {
  int pa, la, pb, lb;
};

// The coefficients.  One that is 1 skips the float64 multiply, and whether it is 1 is
// found once: a float64 instruction, a comparison too, occupies its pipe for about 19
// cycles whatever the lanes that take part.
struct AddCoef {
  double alpha, beta;
  bool alpha1, beta1;
};
__device__ __forceinline__ AddCoef add_coef(double alpha, double beta) {
  return AddCoef{alpha, beta, alpha == 1.0, beta == 1.0};
}
// coefficient * value, rounded once.  Products and sums are the rounded intrinsics: the
// compiler may contract plain ones into one fma, and a row's values would then depend
// on which of the paths below it takes.
__device__ __forceinline__ double add_alpha(const AddCoef& k, double v) { return k.alpha1 ? v : __dmul_rn(k.alpha, v); }
__device__ __forceinline__ double add_beta(const AddCoef& k, double v) { return k.beta1 ? v : __dmul_rn(k.beta, v); }

// A row by a warp: its columns go to col (A's la, then B's lb); *strict: both
// rows strictly ascending.
__device__ __forceinline__ void add_stage(const CsrView& A, const CsrView& B, const AddRow& r, int32_t* col,
                                          int lane, bool* strict, int* bad) {
  __syncwarp();
  for (int t = lane; t < r.la; t += 32) col[t] = A.colind[r.pa + t];
  for (int t = lane; t < r.lb; t += 32) col[r.la + t] = B.colind[r.pb + t];
  __syncwarp();
  bool off = false;
  for (int t = lane; t < r.la + r.lb; t += 32) {
    const int c = col[t];
    if ((unsigned)c >= (unsigned)A.n) *bad = 1;  // (A and B have the same columns)
    off |= t > 0 && t != r.la && col[t - 1] >= c;
  }
  *strict = !__any_sync(kFull, off);
}

// The bits of a row: words of A's slots in C's row, then of A's shared entries, in the
// place of the slots of the longer of its two rows (which has as many).
template <class Int>
__device__ __forceinline__ Int* add_bits(const AddRow& r, Int* apos, Int* bpos) {
  return r.la >= r.lb ? apos + r.pa : bpos + r.pb;
}

// Strictly ascending staged rows, by a warp: their bits to out; returns the length of
// C's row.  Entry t of A lands at t + #{B < its column} - #{shared columns before it}.
// word: 16 words of shared memory.
__device__ __forceinline__ int add_merge_bits(const AddRow& r, const int32_t* col, uint32_t* word,
                                              int32_t* __restrict__ out, int lane) {
  uint32_t* shared = word + kAddWarpMax / 32;
  if (lane < 2 * kAddWarpMax / 32) word[lane] = 0u;
  __syncwarp();
  int common = 0;
  for (int t0 = 0; t0 < r.la; t0 += 32) {
    const int t = t0 + lane;
    bool found = false;
    int k = 0;
    if (t < r.la) {
      const int c = col[t];
      k = add_lower_bound(col + r.la, r.lb, c);
      found = k < r.lb && col[r.la + k] == c;
    }
    const unsigned f = __ballot_sync(kFull, found);
    const int s = t + k - common - __popc(f & ((1u << lane) - 1u));
    if (t < r.la) atomicOr(&word[s >> 5], 1u << (s & 31));
    if (lane == 0) shared[t0 >> 5] = f;
    common += __popc(f);
  }
  __syncwarp();
  const int n = r.la + r.lb - common, na = (n + 31) >> 5, nf = (r.la + 31) >> 5;
  if (lane < na) out[lane] = (int32_t)word[lane];
  if (lane < nf) out[na + lane] = (int32_t)shared[lane];
  return n;
}

// Numeric of a row through its bits, by a warp.  False: they are not this row's.
__device__ __forceinline__ bool add_by_bits(const CsrView& A, const CsrView& B, const AddCoef& k,
                                            const AddRow& r, const int32_t* __restrict__ words, int64_t off, int n,
                                            int32_t* __restrict__ c_colind, double* __restrict__ c_vals, int lane) {
  if (n < 0 || r.la + r.lb > kAddWarpMax || n > r.la + r.lb) return false;
  const int na = (n + 31) >> 5, nf = (r.la + 31) >> 5;  // (8 words each at most)
  const uint32_t aw = lane < na ? (uint32_t)words[lane] : 0u, fw = lane < nf ? (uint32_t)words[na + lane] : 0u;
  const int mine = __popc(aw) | (__popc(fw) << 16);
  const int incl = team_inclusive_scan<32>(mine, lane, kFull), before = incl - mine;
  const int total = __shfl_sync(kFull, incl, 31);
  if ((total & 0xffff) != r.la || r.la + r.lb - (total >> 16) != n) return false;
  for (int s0 = 0; s0 < n; s0 += 32) {
    const int s = s0 + lane, w = s0 >> 5;
    const uint32_t m = __shfl_sync(kFull, aw, w);
    const int ia = (__shfl_sync(kFull, before, w) & 0xffff) + __popc(m & ((1u << lane) - 1u));
    const uint32_t f = __shfl_sync(kFull, fw, ia >> 5);
    const int ib = s - ia + (__shfl_sync(kFull, before, ia >> 5) >> 16) + __popc(f & ((1u << (ia & 31)) - 1u));
    if (s < n) {
      const bool a = (m >> lane & 1u) != 0u, both = a && (f >> (ia & 31) & 1u) != 0u;
      const double v = a ? A.vals[r.pa + ia] : B.vals[r.pb + ib], w = both ? B.vals[r.pb + ib] : 0.0;
      c_colind[off + s] = a ? A.colind[r.pa + ia] : B.colind[r.pb + ib];
      c_vals[off + s] = (a ? k.alpha1 : k.beta1) ? v : __dmul_rn(a ? k.alpha : k.beta, v);
      if (both) atomicAdd(&c_vals[off + s], add_beta(k, w));
    }
  }
  return true;
}

// Rows of up to T entries in each matrix: a lane holds one entry of each, and the
// search goes through shuffles.
// Whether the team's rows, one entry of each in a lane (INT_MAX past their ends),
// are strictly ascending.
template <int T>
__device__ __forceinline__ bool add_strict(int ca, int cb, const AddRow& r, int ncols, int tl, unsigned team,
                                           int* bad) {
  if ((tl < r.la && (unsigned)ca >= (unsigned)ncols) || (tl < r.lb && (unsigned)cb >= (unsigned)ncols)) *bad = 1;
  const int ua = __shfl_up_sync(kFull, ca, 1, T), ub = __shfl_up_sync(kFull, cb, 1, T);
  const bool off = tl > 0 && ((tl < r.la && ua >= ca) || (tl < r.lb && ub >= cb));
  return (__ballot_sync(kFull, off) & team) == 0u;
}
// Columns below c in the team's sorted x (padded with INT_MAX); *at: x holds c there.
template <int T>
__device__ __forceinline__ int add_search(int x, int c, bool* at) {
  int pos = 0;
#pragma unroll
  for (int st = T / 2; st > 0; st >>= 1)
    if (__shfl_sync(kFull, x, pos + st - 1, T) < c) pos += st;
  const int v = __shfl_sync(kFull, x, pos, T);
  *at = v == c;
  return pos + (v < c ? 1 : 0);
}

// Slots of a row that is not strictly ascending, sorted by one warp; returns
// nnz(C(i,:)).
__device__ __forceinline__ int add_sort_row(const CsrView& A, const CsrView& B, const AddRow& r, u64* key,
                                            int32_t* __restrict__ apos, int32_t* __restrict__ bpos, int lane,
                                            int& bad) {
  const int L = r.la + r.lb, n = next_pow2(L);
  int unsorted = 0;
  add_load<32>(A, B, r.pa, r.la, r.pb, r.lb, n, key, lane, unsorted, bad);
  unsorted = __any_sync(kFull, unsorted);
  __syncwarp();
  add_sort<32>(key, n, lane, !unsorted);
  // slots: scan of "first of its column" flags over the L sorted keys
  int run = 0;
  for (int t0 = 0; t0 < L; t0 += 32) {
    const int t = t0 + lane;
    u64 k = 0;
    int first = 0;
    if (t < L) {
      k = key[t];
      first = (t == 0 || (key[t - 1] >> 32) != (k >> 32)) ? 1 : 0;
    }
    const int incl = team_inclusive_scan<32>(first, lane, kFull);
    if (t < L) {
      const int slot = (run + incl - 1) | (first ? 0 : kAddLater);
      const int idx = (int)(k & 0x7fffffffull);
      if (k & (1ull << 31)) bpos[r.pb + idx] = slot;
      else apos[r.pa + idx] = slot;
    }
    run += __shfl_sync(kFull, incl, 31);
  }
  __syncwarp();
  return run;
}

// Symbolic, T lanes per row: rows that do not fit the team, or are not strictly
// ascending, are taken by the whole warp afterwards; rows of more than
// kAddWarpMax entries go to long_rows (count first).
constexpr int kAddRowWarps = 8;
template <int T>
__global__ void __launch_bounds__(kAddRowWarps * 32)
k_spadd_count(CsrView A, CsrView B, int32_t* __restrict__ cnt, int32_t* __restrict__ apos,
              int32_t* __restrict__ bpos, uint8_t* __restrict__ kind, int32_t* __restrict__ long_rows,
              int32_t* __restrict__ kinds, int* status) {
  __shared__ u64 keys[kAddRowWarps][kAddWarpMax];
  __shared__ unsigned cta_kinds;
  if (threadIdx.x == 0) cta_kinds = 0u;
  __syncthreads();
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, tl = lane % T, tm = lane / T;
  const unsigned team = team_mask<T>();
  const long long stride = (long long)gridDim.x * kAddRowWarps * (32 / T);
  int bad = 0;
  bool by_team = false, by_warp = false, by_cta = false;
  auto bounds = [&](long long row) -> AddRow {
    AddRow r{0, 0, 0, 0};
    if (row < A.m) {
      r.pa = A.rowptr[row];
      r.la = A.rowptr[row + 1] - r.pa;
      r.pb = B.rowptr[row];
      r.lb = B.rowptr[row + 1] - r.pb;
      if (r.la < 0 || r.lb < 0) {
        bad = 1;
        r.la = r.lb = 0;
      }
    }
    return r;
  };
  const long long first = ((long long)blockIdx.x * kAddRowWarps + warp) * (32 / T);
  for (long long r0 = first; r0 < A.m; r0 += stride) {
    const long long row = r0 + tm;
    const AddRow all = bounds(row);
    AddRow r = all;
    const int L = r.la + r.lb;
    const bool big = r.la > T || r.lb > T;
    if (big) r.la = r.lb = 0;
    const int ca = tl < r.la ? A.colind[r.pa + tl] : 0x7fffffff;
    const int cb = tl < r.lb ? B.colind[r.pb + tl] : 0x7fffffff;
    const bool ok = add_strict<T>(ca, cb, r, A.n, tl, team, &bad);
    bool found;
    add_search<T>(cb, ca, &found);
    const int common = __popc(__ballot_sync(kFull, found && tl < r.la) & team);
    if (row < A.m && !big && ok && tl == 0) {
      by_team = true;
      cnt[row] = L - common;
      kind[row] = common == r.la && r.la == r.lb ? kAddSame : kAddByTeam;
    }
    for (unsigned m = __ballot_sync(kFull, (big || !ok) && tl == 0); m; m &= m - 1) {
      const int src = __ffs(m) - 1;
      const AddRow w{__shfl_sync(kFull, all.pa, src), __shfl_sync(kFull, all.la, src),
                     __shfl_sync(kFull, all.pb, src), __shfl_sync(kFull, all.lb, src)};
      const long long wrow = r0 + src / T;
      if (w.la + w.lb > kAddWarpMax) {
        if (lane == 0) {
          long_rows[1 + atomicAdd(long_rows, 1)] = (int32_t)wrow;
          kind[wrow] = kAddByCta;
        }
        by_cta = true;
        continue;
      }
      by_warp = true;
      bool strict = false;
      int32_t* col = reinterpret_cast<int32_t*>(keys[warp]);
      if (__shfl_sync(kFull, (int)big, src)) add_stage(A, B, w, col, lane, &strict, &bad);
      const int n = strict ? add_merge_bits(w, col, reinterpret_cast<uint32_t*>(col) + kAddWarpMax,
                                            add_bits(w, apos, bpos), lane)
                           : add_sort_row(A, B, w, keys[warp], apos, bpos, lane, bad);
      if (lane == 0) {
        cnt[wrow] = n;
        kind[wrow] = strict ? kAddByBits : kAddBySlots;
      }
      __syncwarp();
    }
  }
  if (bad) set_status(status, KK_ERR_BAD_INDEX);
  // (one store per CTA, and only until it is seen: stores of every warp to one address
  // take turns, 70 us for 26,738 rows)
  const unsigned seen = (by_team ? 1u : 0u) | (by_warp ? 2u : 0u) | (by_cta ? 4u : 0u);
  const unsigned mine = __reduce_or_sync(kFull, seen);
  if (lane == 0 && mine) atomicOr(&cta_kinds, mine);
  __syncthreads();
  if (threadIdx.x < 3 && (cta_kinds >> threadIdx.x & 1u)) {
    volatile int32_t* flag = kinds + threadIdx.x;
    if (*flag == 0) *flag = 1;
  }
}

// One CTA of kAddCtaThreads per long row (dynamic shared memory kAddCtaMax keys).
__global__ void __launch_bounds__(kAddCtaThreads)
k_spadd_sym_cta(CsrView A, CsrView B, int32_t* __restrict__ cnt, int32_t* __restrict__ apos,
                int32_t* __restrict__ bpos, const int32_t* __restrict__ long_rows, int* status) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  u64* key = reinterpret_cast<u64*>(smem_raw);
  __shared__ int scratch[33];
  __shared__ int flags[2];
  const int tid = threadIdx.x;
  const int nrows = long_rows[0];
  for (int q = blockIdx.x; q < nrows; q += gridDim.x) {
    const int r = long_rows[1 + q];
    const int pa = A.rowptr[r], la = A.rowptr[r + 1] - pa;
    const int pb = B.rowptr[r], lb = B.rowptr[r + 1] - pb;
    const int L = la + lb;
    if (L > kAddCtaMax) {
      if (tid == 0) set_status(status, KK_ERR_CAPACITY);
      continue;
    }
    if (tid == 0) {
      flags[0] = 0;
      flags[1] = 0;
    }
    int n = 32;
    while (n < L) n <<= 1;
    int unsorted = 0, bad = 0;
    add_load<kAddCtaThreads>(A, B, pa, la, pb, lb, n, key, tid, unsorted, bad);
    if (unsorted) flags[0] = 1;
    if (bad) flags[1] = 1;
    __syncthreads();
    const bool merge_only = flags[0] == 0;
    if (tid == 0 && flags[1]) set_status(status, KK_ERR_BAD_INDEX);
    add_sort<kAddCtaThreads>(key, n, tid, merge_only);
    int run = 0;
    for (int t0 = 0; t0 < L; t0 += kAddCtaThreads) {
      const int t = t0 + tid;
      u64 k = 0;
      int first = 0;
      if (t < L) {
        k = key[t];
        first = (t == 0 || (key[t - 1] >> 32) != (k >> 32)) ? 1 : 0;
      }
      int tot;
      const int ex = add_block_scan(first, scratch, &tot);
      if (t < L) {
        const int slot = (run + ex + first - 1) | (first ? 0 : kAddLater);
        const int idx = (int)(k & 0x7fffffffull);
        if (k & (1ull << 31)) bpos[pb + idx] = slot;
        else apos[pa + idx] = slot;
      }
      run += tot;
    }
    if (tid == 0) cnt[r] = run;
    __syncthreads();
  }
}

// Numeric of a row through its slots, by NT threads: the first entry of every column is
// stored, then the others are added to it.
template <int NT>
__device__ __forceinline__ void add_scatter(const CsrView& A, const CsrView& B, const AddCoef& k,
                                            const AddRow& r, const int32_t* __restrict__ apos,
                                            const int32_t* __restrict__ bpos, int64_t off, int n,
                                            int32_t* __restrict__ c_colind, double* __restrict__ c_vals, int tid,
                                            int& mismatch) {
  auto any = [](bool p) -> bool {
    if constexpr (NT == 32) {
      __syncwarp();
      return __any_sync(kFull, p);
    } else {
      return __syncthreads_or(p) != 0;
    }
  };
  bool again_a = false, again_b = false;
  for (int t = tid; t < max(r.la, r.lb); t += NT) {
    const bool a = t < r.la, b = t < r.lb;
    int sa = 0, sb = 0, ca = 0, cb = 0;
    double va = 0.0, vb = 0.0;
    if (a) sa = apos[r.pa + t];
    if (b) sb = bpos[r.pb + t];
    if (a) ca = A.colind[r.pa + t];
    if (b) cb = B.colind[r.pb + t];
    if (a) va = A.vals[r.pa + t];
    if (b) vb = B.vals[r.pb + t];
    const int at = sa & kAddSlot, bt = sb & kAddSlot;
    if ((a && at >= n) || (b && bt >= n)) {
      mismatch = 1;
      continue;
    }
    again_a |= a && sa < 0;
    again_b |= b && sb < 0;
    if (a && sa >= 0) {
      c_colind[off + at] = ca;
      c_vals[off + at] = add_alpha(k, va);
    }
    if (b && sb >= 0) {
      c_colind[off + bt] = cb;
      c_vals[off + bt] = add_beta(k, vb);
    }
  }
  if (any(again_a)) {
    for (int t = tid; t < r.la; t += NT) {
      const int s = apos[r.pa + t], at = s & kAddSlot;
      if (s < 0 && at < n) atomicAdd(&c_vals[off + at], add_alpha(k, A.vals[r.pa + t]));
    }
  }
  if (any(again_b)) {
    for (int t = tid; t < r.lb; t += NT) {
      const int s = bpos[r.pb + t], at = s & kAddSlot;
      if (s < 0 && at < n) atomicAdd(&c_vals[off + at], add_beta(k, B.vals[r.pb + t]));
    }
  }
}

// Numeric of the rows of kind kAddByTeam, T lanes per row: a lane holds one entry of each
// matrix and writes both.  A's entry of a shared column is stored, then B's is added to
// it (in L2: an addition here would occupy the float64 pipe).  The other
// kinds have kernels of their own: together they need registers that cost these rows,
// a chain of two loads, 2 of 5 warps in flight.
template <int T>
__global__ void __launch_bounds__(kAddRowWarps * 32, 8)
k_spadd_team(CsrView A, CsrView B, double alpha, double beta, const int64_t* __restrict__ c_rowptr,
             const uint8_t* __restrict__ kind, int32_t* __restrict__ c_colind, double* __restrict__ c_vals,
             int* status) {
  const int lane = threadIdx.x & 31, tl = lane % T;
  const unsigned team = team_mask<T>(), before = (1u << lane) - 1u;
  const long long per = 32 / T, stride = (long long)gridDim.x * kAddRowWarps * per;
  const AddCoef k = add_coef(alpha, beta);
  int mismatch = 0;
  for (long long r0 = ((long long)blockIdx.x * kAddRowWarps + (threadIdx.x >> 5)) * per; r0 < A.m; r0 += stride) {
    const long long row = r0 + lane / T;
    AddRow r{0, 0, 0, 0};
    int64_t off = 0;
    int n = 0, how = kAddByTeam;
    if (row < A.m) {
      how = kind[row];
      r.pa = A.rowptr[row];
      r.la = A.rowptr[row + 1] - r.pa;
      r.pb = B.rowptr[row];
      r.lb = B.rowptr[row + 1] - r.pb;
      off = c_rowptr[row];
      n = (int)(c_rowptr[row + 1] - off);
    }
    const bool same = how == kAddSame, here = same || how == kAddByTeam;
    if (!here || r.la > T || r.lb > T || (same && r.la != r.lb)) {
      if (here) mismatch = 1;  // not the rows of the symbolic call
      r.la = r.lb = n = 0;
    }
    const int ca = tl < r.la ? A.colind[r.pa + tl] : 0x7fffffff;
    const double va = tl < r.la ? A.vals[r.pa + tl] : 0.0, vb = tl < r.lb ? B.vals[r.pb + tl] : 0.0;
    if (!__any_sync(kFull, how == kAddByTeam)) {  // the same columns: entry t of each is in slot t
      if (r.la != n) mismatch = 1;
      if (tl < r.la && tl < n) {
        c_colind[off + tl] = ca;
        c_vals[off + tl] = add_alpha(k, va);
        atomicAdd(&c_vals[off + tl], add_beta(k, vb));
      }
      continue;
    }
    const int cb = tl < r.lb ? B.colind[r.pb + tl] : 0x7fffffff;
    bool fa, fb;
    const int ka = add_search<T>(cb, ca, &fa), kb = add_search<T>(ca, cb, &fb);
    const unsigned ma = __ballot_sync(kFull, fa && tl < r.la) & team, mb = __ballot_sync(kFull, fb && tl < r.lb) & team;
    if (r.la + r.lb - __popc(ma) != n) mismatch = 1;
    const int sa = tl + ka - __popc(ma & before);
    const double wa = add_alpha(k, va), wb = add_beta(k, vb);
    if (tl < r.la && sa < n) {
      c_colind[off + sa] = ca;
      c_vals[off + sa] = wa;
    }
    __syncwarp();
    // (a shared column's slot counts the shared columns before it, as A's does)
    const int sb = tl + kb - __popc(mb & before);
    if (tl < r.lb && sb < n) {
      if (mb >> lane & 1u) {
        atomicAdd(&c_vals[off + sb], wb);
      } else {
        c_colind[off + sb] = cb;
        c_vals[off + sb] = wb;
      }
    }
  }
  if (mismatch) set_status(status, KK_ERR_STRUCTURE_MISMATCH);
}

// Numeric of the rows of kinds kAddBySlots and kAddByBits, a warp each: a warp reads the bounds of `group` rows at a
// time (at most 32, fewer where there are not warps enough otherwise) and takes those
// of its kinds.
__global__ void __launch_bounds__(kAddRowWarps * 32)
k_spadd_warp(CsrView A, CsrView B, double alpha, double beta, const int64_t* __restrict__ c_rowptr,
             const int32_t* __restrict__ apos, const int32_t* __restrict__ bpos, const uint8_t* __restrict__ kind,
             int32_t group, int32_t* __restrict__ c_colind, double* __restrict__ c_vals, int* status) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const long long stride = (long long)gridDim.x * kAddRowWarps * group;
  const AddCoef k = add_coef(alpha, beta);
  int mismatch = 0;
  for (long long r0 = ((long long)blockIdx.x * kAddRowWarps + warp) * group; r0 < A.m; r0 += stride) {
    const long long row = r0 + lane;
    const bool on = lane < group && row < A.m;
    const int how = on ? kind[row] : kAddByTeam;
    AddRow r{0, 0, 0, 0};
    int64_t off = 0;
    int n = 0;
    if (how == kAddBySlots || how == kAddByBits) {
      r.pa = A.rowptr[row];
      r.la = A.rowptr[row + 1] - r.pa;
      r.pb = B.rowptr[row];
      r.lb = B.rowptr[row + 1] - r.pb;
      off = c_rowptr[row];
      n = (int)(c_rowptr[row + 1] - off);
    }
    for (unsigned m = __ballot_sync(kFull, how == kAddBySlots || how == kAddByBits); m; m &= m - 1) {
      const int src = __ffs(m) - 1;
      const AddRow w{__shfl_sync(kFull, r.pa, src), __shfl_sync(kFull, r.la, src), __shfl_sync(kFull, r.pb, src),
                     __shfl_sync(kFull, r.lb, src)};
      const int64_t woff = __shfl_sync(kFull, (long long)off, src);
      const int wn = __shfl_sync(kFull, n, src);
      if (__shfl_sync(kFull, how, src) == kAddBySlots)
        add_scatter<32>(A, B, k, w, apos, bpos, woff, wn, c_colind, c_vals, lane, mismatch);
      else if (w.la < 0 || w.lb < 0 ||
               !add_by_bits(A, B, k, w, add_bits(w, apos, bpos), woff, wn, c_colind, c_vals, lane))
        mismatch = 1;
    }
  }
  if (mismatch) set_status(status, KK_ERR_STRUCTURE_MISMATCH);
}

// Numeric of the long rows, a CTA each.
__global__ void __launch_bounds__(256)
k_spadd_long(CsrView A, CsrView B, double alpha, double beta, const int64_t* __restrict__ c_rowptr,
             const int32_t* __restrict__ apos, const int32_t* __restrict__ bpos,
             const int32_t* __restrict__ long_rows, int32_t* __restrict__ c_colind, double* __restrict__ c_vals,
             int* status) {
  const AddCoef k = add_coef(alpha, beta);
  const int nrows = long_rows[0];
  int mismatch = 0;
  for (int q = blockIdx.x; q < nrows; q += gridDim.x) {
    const int row = long_rows[1 + q];
    AddRow r;
    r.pa = A.rowptr[row];
    r.la = A.rowptr[row + 1] - r.pa;
    r.pb = B.rowptr[row];
    r.lb = B.rowptr[row + 1] - r.pb;
    const int64_t off = c_rowptr[row];
    add_scatter<256>(A, B, k, r, apos, bpos, off, (int)(c_rowptr[row + 1] - off), c_colind, c_vals, threadIdx.x,
                     mismatch);
  }
  if (mismatch) set_status(status, KK_ERR_STRUCTURE_MISMATCH);
}

// Lanes per row: enough for the typical row of either matrix.
int add_team(const CsrView& A, const CsrView& B) {
  const long long avg = (A.nnz > B.nnz ? A.nnz : B.nnz) / A.m;
  return avg <= 7 ? 8 : avg <= 14 ? 16 : 32;
}

int add_grid(const LaunchCtx& ctx, int m, int rows_per_cta) {
  long long blocks = ((long long)m + rows_per_cta - 1) / rows_per_cta;
  const long long cap = (long long)ctx.num_sms * 32;
  return (int)(blocks > cap ? cap : blocks);
}

}  // namespace

cudaError_t launch_spadd_symbolic(const LaunchCtx& ctx, const CsrView& A, const CsrView& B, int32_t* cnt,
                                  int32_t* apos, int32_t* bpos, uint8_t* kind, int32_t* long_rows,
                                  int32_t* kinds) {
  if (A.m <= 0) return cudaSuccess;
  const int T = add_team(A, B), grid = add_grid(ctx, A.m, kAddRowWarps * 32 / T);
  auto kern = T == 8 ? k_spadd_count<8> : T == 16 ? k_spadd_count<16> : k_spadd_count<32>;
  kern<<<grid, kAddRowWarps * 32, 0, ctx.stream>>>(A, B, cnt, apos, bpos, kind, long_rows, kinds, ctx.status);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  // the list's length is on the device: one wave of CTAs strides over it
  const size_t smem = (size_t)kAddCtaMax * 8;
  e = cudaFuncSetAttribute(k_spadd_sym_cta, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  k_spadd_sym_cta<<<ctx.num_sms * 2, kAddCtaThreads, smem, ctx.stream>>>(A, B, cnt, apos, bpos, long_rows,
                                                                         ctx.status);
  return cudaGetLastError();
}

cudaError_t launch_spadd_numeric(const LaunchCtx& ctx, const CsrView& A, const CsrView& B, double alpha,
                                 double beta, const int64_t* c_rowptr, const int32_t* apos,
                                 const int32_t* bpos, const uint8_t* kind, const int32_t* long_rows,
                                 const int32_t* kinds, int32_t* c_colind, double* c_vals) {
  if (A.m <= 0) return cudaSuccess;
  if (kinds[0]) {
    const int T = add_team(A, B), grid = add_grid(ctx, A.m, kAddRowWarps * 32 / T);
    auto kern = T == 8 ? k_spadd_team<8> : T == 16 ? k_spadd_team<16> : k_spadd_team<32>;
    kern<<<grid, kAddRowWarps * 32, 0, ctx.stream>>>(A, B, alpha, beta, c_rowptr, kind, c_colind, c_vals, ctx.status);
  }
  if (kinds[1]) {
    const int per = A.m / (ctx.num_sms * kAddRowWarps * 32), group = per < 1 ? 1 : per > 8 ? 8 : per;
    k_spadd_warp<<<add_grid(ctx, A.m, kAddRowWarps * group), kAddRowWarps * 32, 0, ctx.stream>>>(
        A, B, alpha, beta, c_rowptr, apos, bpos, kind, group, c_colind, c_vals, ctx.status);
  }
  if (kinds[2])  // (their number is on the device)
    k_spadd_long<<<A.m < ctx.num_sms * 8 ? A.m : ctx.num_sms * 8, 256, 0, ctx.stream>>>(
        A, B, alpha, beta, c_rowptr, apos, bpos, long_rows, c_colind, c_vals, ctx.status);
  return cudaGetLastError();
}

}  // namespace kk
