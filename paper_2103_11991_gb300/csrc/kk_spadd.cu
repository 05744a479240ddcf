// Sparse matrix addition C = alpha A + beta B (Kokkos Kernels paper, Sec.
// "SpAdd"), symbolic and numeric phases.
//
// Rows that are strictly ascending in both matrices, of up to kAddWarpMax combined
// entries, are merged by binary search of each entry in the other row: through
// shuffles in teams of 8, 16 or 32 lanes while both rows fit the team, staged in
// shared memory by a warp otherwise.  The symbolic phase counts the shared columns,
// the numeric phase merges again and writes the row of C in one go.  Nothing is
// kept between the phases for them: reading both rows' columns again, which C's
// columns need anyway, costs less than writing and reading a slot per entry, adding
// into C with atomics and zeroing it first (two matrices of 500,000 rows of 30: 286
// us symbolic and 217 numeric that way, 116 and 180 now, both phases with their
// scan 546 -> 337).  Bound by issue and by the latency of a row's loads; prefetching
// the next row's costs a third of the warps in flight and gave nothing.
//
// Other rows: the entries of A and B become 64-bit keys
// (column << 32 | source bit (B) << 31 | index within the source row) in
// shared memory and are sorted by a bitonic network; equal columns are then
// adjacent, so a scan of "first of its column" flags gives nnz(C(i,:)) and, for
// every entry of A and of B, its slot in the row of C (the paper's Apos and
// Bpos; the sign bit marks all but the first entry of a column).  When both rows
// are sorted (repeats allowed) the keys are laid out as A ascending, then padding,
// then B descending: a bitonic sequence, so only the final merge stage runs (the
// paper's sorted-input method); otherwise the full sort runs (its unsorted-input
// method).  Rows of up to kAddWarpMax combined entries take one warp, rows of up to
// kAddCtaMax one CTA of 1024 threads; longer rows are reported as KK_ERR_CAPACITY.
// Their numeric phase stores the first entry of every column with its value, then
// adds the others (float64 atomics: repeated columns are added in no fixed order).
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

// coefficient * value, rounded once.  A coefficient of 1 skips the float64 multiply
// (FP64 is the scarce pipe; the branch is uniform over the grid).  Products and sums
// are the rounded intrinsics: the compiler may contract plain ones into one fma, and
// a row's values would then depend on which of the paths below it takes.
__device__ __forceinline__ double add_scaled(double coefficient, double v) {
  return coefficient == 1.0 ? v : __dmul_rn(coefficient, v);
}

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

// Columns that strictly ascending staged rows share.
__device__ __forceinline__ int add_common(const AddRow& r, const int32_t* col, int lane) {
  int common = 0;
  for (int t0 = 0; t0 < r.la; t0 += 32) {
    const int t = t0 + lane;
    bool found = false;
    if (t < r.la) {
      const int c = col[t], k = add_lower_bound(col + r.la, r.lb, c);
      found = k < r.lb && col[r.la + k] == c;
    }
    common += __popc(__ballot_sync(kFull, found));
  }
  return common;
}

// Strictly ascending staged rows into row off .. off + n of C; returns the merged
// length.  Entry k of a row lands at k + #{other < its column} - #{shared columns
// before it}; a shared column is summed by A's entry.
__device__ __forceinline__ int add_merge(const CsrView& A, const CsrView& B, double alpha, double beta,
                                         const AddRow& r, const int32_t* col, int64_t off, int n,
                                         int32_t* __restrict__ c_colind, double* __restrict__ c_vals, int lane) {
  const unsigned before = (1u << lane) - 1u;
  const int32_t* ca = col;
  const int32_t* cb = col + r.la;
  int common = 0, seen = 0;
  for (int t0 = 0; t0 < r.la; t0 += 32) {
    const int t = t0 + lane;
    bool found = false;
    int c = 0, k = 0;
    double v = 0.0;
    if (t < r.la) {
      v = A.vals[r.pa + t];
      c = ca[t];
      k = add_lower_bound(cb, r.lb, c);
      found = k < r.lb && cb[k] == c;
    }
    v = add_scaled(alpha, v);
    if (found) v = __dadd_rn(v, add_scaled(beta, B.vals[r.pb + k]));
    const unsigned f = __ballot_sync(kFull, found);
    const int s = t + k - common - __popc(f & before);
    if (t < r.la && s < n) {
      c_colind[off + s] = c;
      c_vals[off + s] = v;
    }
    common += __popc(f);
  }
  for (int t0 = 0; t0 < r.lb; t0 += 32) {
    const int t = t0 + lane;
    bool found = false;
    int c = 0, k = 0;
    double v = 0.0;
    if (t < r.lb) {
      v = B.vals[r.pb + t];
      c = cb[t];
      k = add_lower_bound(ca, r.la, c);
      found = k < r.la && ca[k] == c;
    }
    v = add_scaled(beta, v);
    const unsigned f = __ballot_sync(kFull, found);
    const int s = t + k - seen - __popc(f & before);
    if (t < r.lb && !found && s < n) {
      c_colind[off + s] = c;
      c_vals[off + s] = v;
    }
    seen += __popc(f);
  }
  return r.la + r.lb - common;
}

// Rows of up to T entries in each matrix: a lane holds one entry of each, and the
// searches go through shuffles (110 instructions a row instead of 330 through
// shared memory).
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
      const int slot = (run + incl - 1) | (first ? 0 : (int)0x80000000u);
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
// kAddWarpMax entries go to long_rows (count first).  kind: 1 for a row that the
// numeric phase merges, 0 for one with slots.
constexpr int kAddRowWarps = 8;
template <int T>
__global__ void __launch_bounds__(kAddRowWarps * 32)
k_spadd_count(CsrView A, CsrView B, int32_t* __restrict__ cnt, int32_t* __restrict__ apos,
              int32_t* __restrict__ bpos, uint8_t* __restrict__ kind, int32_t* __restrict__ long_rows,
              int* status) {
  __shared__ u64 keys[kAddRowWarps][kAddWarpMax];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, tl = lane % T, tm = lane / T;
  const unsigned team = team_mask<T>();
  const long long stride = (long long)gridDim.x * kAddRowWarps * (32 / T);
  int bad = 0;
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
      cnt[row] = L - common;
      kind[row] = 1;
    }
    for (unsigned m = __ballot_sync(kFull, (big || !ok) && tl == 0); m; m &= m - 1) {
      const int src = __ffs(m) - 1;
      const AddRow w{__shfl_sync(kFull, all.pa, src), __shfl_sync(kFull, all.la, src),
                     __shfl_sync(kFull, all.pb, src), __shfl_sync(kFull, all.lb, src)};
      const long long wrow = r0 + src / T;
      if (w.la + w.lb > kAddWarpMax) {
        if (lane == 0) {
          long_rows[1 + atomicAdd(long_rows, 1)] = (int32_t)wrow;
          kind[wrow] = 0;
        }
        continue;
      }
      bool strict = false;
      int32_t* col = reinterpret_cast<int32_t*>(keys[warp]);
      if (__shfl_sync(kFull, (int)big, src)) add_stage(A, B, w, col, lane, &strict, &bad);
      const int n = strict ? w.la + w.lb - add_common(w, col, lane)
                           : add_sort_row(A, B, w, keys[warp], apos, bpos, lane, bad);
      if (lane == 0) {
        cnt[wrow] = n;
        kind[wrow] = strict ? 1 : 0;
      }
      __syncwarp();
    }
  }
  if (bad) set_status(status, KK_ERR_BAD_INDEX);
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
        const int slot = (run + ex + first - 1) | (first ? 0 : (int)0x80000000u);
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

// Numeric of a row through its slots, by one warp: the first entry of every
// column is stored, the others are added to it.
__device__ __forceinline__ void add_scatter(const CsrView& A, const CsrView& B, double alpha, double beta,
                                            const AddRow& r, const int32_t* __restrict__ apos,
                                            const int32_t* __restrict__ bpos, int64_t off, int n,
                                            int32_t* __restrict__ c_colind, double* __restrict__ c_vals, int lane,
                                            int& mismatch) {
  bool more = false;
  auto put = [&](int s, int c, double v) {
    const int at = s & 0x7fffffff;
    if (at >= n) {
      mismatch = 1;
    } else if (s < 0) {
      more = true;
    } else {
      c_colind[off + at] = c;
      c_vals[off + at] = v;
    }
  };
  for (int t = lane; t < max(r.la, r.lb); t += 32) {
    const bool a = t < r.la, b = t < r.lb;
    const int sa = a ? apos[r.pa + t] : 0, sb = b ? bpos[r.pb + t] : 0;
    const int ca = a ? A.colind[r.pa + t] : 0, cb = b ? B.colind[r.pb + t] : 0;
    const double va = a ? add_scaled(alpha, A.vals[r.pa + t]) : 0.0, vb = b ? add_scaled(beta, B.vals[r.pb + t]) : 0.0;
    if (a) put(sa, ca, va);
    if (b) put(sb, cb, vb);
  }
  __syncwarp();
  if (!__any_sync(kFull, more)) return;
  auto add = [&](int s, double v) {
    const int at = s & 0x7fffffff;
    if (s < 0 && at < n) atomicAdd(&c_vals[off + at], v);
  };
  for (int t = lane; t < r.la; t += 32) add(apos[r.pa + t], add_scaled(alpha, A.vals[r.pa + t]));
  for (int t = lane; t < r.lb; t += 32) add(bpos[r.pb + t], add_scaled(beta, B.vals[r.pb + t]));
}

// Numeric, T lanes per row as in k_spadd_count.
template <int T>
__global__ void __launch_bounds__(kAddRowWarps * 32)
k_spadd_num(CsrView A, CsrView B, double alpha, double beta, const int64_t* __restrict__ c_rowptr,
            const int32_t* __restrict__ apos, const int32_t* __restrict__ bpos, const uint8_t* __restrict__ kind,
            int32_t* __restrict__ c_colind, double* __restrict__ c_vals, int* status) {
  __shared__ int32_t cols[kAddRowWarps][kAddWarpMax];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, tl = lane % T, tm = lane / T;
  const unsigned team = team_mask<T>(), before = (1u << lane) - 1u;
  const long long stride = (long long)gridDim.x * kAddRowWarps * (32 / T);
  int bad = 0, mismatch = 0;
  struct Row {
    AddRow r;
    int n;        // the row's length in C
    int64_t off;  // ... and its start
    bool fits, merge;
  };
  auto bounds = [&](long long row) -> Row {
    Row x{{0, 0, 0, 0}, 0, 0, true, true};
    if (row < A.m) {
      x.r.pa = A.rowptr[row];
      x.r.la = A.rowptr[row + 1] - x.r.pa;
      x.r.pb = B.rowptr[row];
      x.r.lb = B.rowptr[row + 1] - x.r.pb;
      x.off = c_rowptr[row];
      x.n = (int)(c_rowptr[row + 1] - x.off);
      x.merge = kind[row] != 0;
      if (x.r.la < 0 || x.r.lb < 0) {
        mismatch = 1;
        x.r.la = x.r.lb = 0;
      }
      x.fits = x.r.la <= T && x.r.lb <= T && x.merge;
    }
    return x;
  };
  const long long first = ((long long)blockIdx.x * kAddRowWarps + warp) * (32 / T);
  for (long long r0 = first; r0 < A.m; r0 += stride) {
    const long long row = r0 + tm;
    const Row cur = bounds(row);
    AddRow r = cur.r;
    if (!cur.fits) r.la = r.lb = 0;
    const int64_t off = cur.off;
    const int n = cur.n;
    const int ca = tl < r.la ? A.colind[r.pa + tl] : 0x7fffffff;
    const int cb = tl < r.lb ? B.colind[r.pb + tl] : 0x7fffffff;
    double va = tl < r.la ? A.vals[r.pa + tl] : 0.0, vb = tl < r.lb ? B.vals[r.pb + tl] : 0.0;
    if (__any_sync(kFull, cur.fits)) {
      const bool strict = add_strict<T>(ca, cb, r, A.n, tl, team, &bad);
      if (!strict) mismatch = 1;  // not the rows of the symbolic call
      va = add_scaled(alpha, va);
      vb = add_scaled(beta, vb);
      bool fa, fb;
      const int ka = add_search<T>(cb, ca, &fa), kb = add_search<T>(ca, cb, &fb);
      fa = fa && tl < r.la;
      fb = fb && tl < r.lb;
      const unsigned ma = __ballot_sync(kFull, fa) & team, mb = __ballot_sync(kFull, fb) & team;
      if (__any_sync(kFull, fa)) {  // shared columns: A's entry takes the sum
        const double w = __shfl_sync(kFull, vb, min(ka, T - 1), T);
        if (fa) va = __dadd_rn(va, w);
      }
      if (cur.fits) {
        if (row < A.m && r.la + r.lb - __popc(ma) != n) mismatch = 1;
        const int sa = tl + ka - __popc(ma & before), sb = tl + kb - __popc(mb & before);
        if (tl < r.la && sa < n) {
          c_colind[off + sa] = ca;
          c_vals[off + sa] = va;
        }
        if (tl < r.lb && !fb && sb < n) {
          c_colind[off + sb] = cb;
          c_vals[off + sb] = vb;
        }
      }
    }
    for (unsigned m = __ballot_sync(kFull, !cur.fits && tl == 0); m; m &= m - 1) {
      const int src = __ffs(m) - 1;
      const AddRow w{__shfl_sync(kFull, cur.r.pa, src), __shfl_sync(kFull, cur.r.la, src),
                     __shfl_sync(kFull, cur.r.pb, src), __shfl_sync(kFull, cur.r.lb, src)};
      const int64_t woff = __shfl_sync(kFull, (long long)off, src);
      const int wn = __shfl_sync(kFull, n, src);
      if (!__shfl_sync(kFull, (int)cur.merge, src)) {
        add_scatter(A, B, alpha, beta, w, apos, bpos, woff, wn, c_colind, c_vals, lane, mismatch);
      } else if (w.la + w.lb > kAddWarpMax) {
        mismatch = 1;
      } else {
        bool ok;
        add_stage(A, B, w, cols[warp], lane, &ok, &bad);
        if (!ok || add_merge(A, B, alpha, beta, w, cols[warp], woff, wn, c_colind, c_vals, lane) != wn) mismatch = 1;
      }
    }
  }
  if (mismatch || bad) set_status(status, KK_ERR_STRUCTURE_MISMATCH);
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
                                  int32_t* apos, int32_t* bpos, uint8_t* kind, int32_t* long_rows) {
  if (A.m <= 0) return cudaSuccess;
  const int T = add_team(A, B), grid = add_grid(ctx, A.m, kAddRowWarps * 32 / T);
  auto kern = T == 8 ? k_spadd_count<8> : T == 16 ? k_spadd_count<16> : k_spadd_count<32>;
  kern<<<grid, kAddRowWarps * 32, 0, ctx.stream>>>(A, B, cnt, apos, bpos, kind, long_rows, ctx.status);
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
                                 const int32_t* bpos, const uint8_t* kind, int32_t* c_colind, double* c_vals) {
  if (A.m <= 0) return cudaSuccess;
  const int T = add_team(A, B), grid = add_grid(ctx, A.m, kAddRowWarps * 32 / T);
  auto kern = T == 8 ? k_spadd_num<8> : T == 16 ? k_spadd_num<16> : k_spadd_num<32>;
  kern<<<grid, kAddRowWarps * 32, 0, ctx.stream>>>(A, B, alpha, beta, c_rowptr, apos, bpos, kind, c_colind, c_vals,
                                                   ctx.status);
  return cudaGetLastError();
}

}  // namespace kk
