// Thread tier: rows with very few products (the smallest bins), one thread
// per row, the row's accumulator in registers.
//
// The paper's method A (Sec. "Standard SpGEMM Kernel": one row per thread,
// B rows walked sequentially) for rows whose product count is so small that
// any shared-memory table, its clearing and its sort cost more than the
// products: the symbolic phase keeps the distinct columns seen so far in a
// register array (at most kThreadSymMax), the numeric phase keeps up to
// kThreadNumMax (column, value) pairs in the order of their first product and
// writes each at its rank.  Values are float64 in storage order (fma(a, b, v)
// from v = 0), the oracle's order, so the thread tier is bit-exact.  Thirty-two
// rows per warp keep many independent load chains in flight.
// What bounds it: issue.  Every product goes through all slots with compares and
// selects, so the kernels come for rows of up to half as many columns too, and
// nothing is kept sorted: the 128^3 Laplacian times its prolongator (4 columns a
// row) took 139 us with 8 sorted slots (1,242 instructions per 32 rows, an
// insertion shifting them all), its symbolic phase 80 with 16.
#include "kk_internal.h"
#include "kk_device.cuh"

namespace kk {
namespace {

constexpr int kThreadBlock = 256;

// A entries whose loads (column, B row bounds, first B entry) are issued together:
// a row's chain of dependent loads is then as long as one entry's.
constexpr int kThreadBatch = 4;

template <int N>
__global__ void __launch_bounds__(kThreadBlock)
k_sym_thread(CsrView A, CsrView B, const int32_t* __restrict__ rows, int32_t nrows,
             int32_t* __restrict__ cnt, int* status) {
  int over = 0;
  for (long long r = (long long)blockIdx.x * blockDim.x + threadIdx.x; r < nrows;
       r += (long long)gridDim.x * blockDim.x) {
    const int i = rows[r];
    const int pa = A.rowptr[i], pe = A.rowptr[i + 1];
    int key[N];
#pragma unroll
    for (int k = 0; k < N; ++k) key[k] = -1;
    int n = 0;
    auto insert = [&](int c) {
      bool found = false;
#pragma unroll
      for (int k = 0; k < N; ++k) found |= key[k] == c;
      if (!found) {
#pragma unroll
        for (int k = 0; k < N; ++k) key[k] = k == n ? c : key[k];
        ++n;
      }
    };
    for (int p0 = pa; p0 < pe; p0 += kThreadBatch) {
      int j[kThreadBatch], q[kThreadBatch], e[kThreadBatch], c[kThreadBatch];
#pragma unroll
      for (int u = 0; u < kThreadBatch; ++u) j[u] = p0 + u < pe ? A.colind[p0 + u] : -1;
#pragma unroll
      for (int u = 0; u < kThreadBatch; ++u) {
        q[u] = e[u] = 0;
        if (j[u] >= 0) {
          q[u] = B.rowptr[j[u]];
          e[u] = B.rowptr[j[u] + 1];
        }
      }
#pragma unroll
      for (int u = 0; u < kThreadBatch; ++u) c[u] = q[u] < e[u] ? B.colind[q[u]] : -1;
#pragma unroll
      for (int u = 0; u < kThreadBatch; ++u) {
        if (q[u] < e[u]) insert(c[u]);
        for (int t = q[u] + 1; t < e[u]; ++t) insert(B.colind[t]);
      }
    }
    cnt[i] = n;
    if (n > N) over = 1;
  }
  if (over) set_status(status, KK_ERR_CAPACITY);
}

template <int N, bool JAC>
__global__ void __launch_bounds__(kThreadBlock)
k_num_thread(CsrView A, CsrView B, const int64_t* __restrict__ c_rowptr,
             const int32_t* __restrict__ rows, int32_t nrows, int32_t* __restrict__ c_colind,
             double* __restrict__ c_vals, int* status) {
  int over = 0, mismatch = 0, bad = 0;
  for (long long r = (long long)blockIdx.x * blockDim.x + threadIdx.x; r < nrows;
       r += (long long)gridDim.x * blockDim.x) {
    const int i = rows[r];
    const int pa = A.rowptr[i], pe = A.rowptr[i + 1];
    const int64_t off = c_rowptr[i];
    const int cnt = (int)(c_rowptr[i + 1] - off);
    int key[N];
    double val[N];
#pragma unroll
    for (int k = 0; k < N; ++k) {
      key[k] = -1;
      val[k] = 0.0;
    }
    int n = 0;
    // JAC (a template switch: the plain kernel keeps its registers): the
    // Jacobi-fused product, A(i,:) taken as s_i A(i,:) plus 1 at the row's first
    // diagonal entry, s_i = -omega / D(i) with D(i) the sum of the row's stored
    // diagonal entries in storage order.  The row is short, so a first pass over
    // it finds D(i); the second pass below reads it again from L1.
    ARowScale ars{1.0, -1, JAC};
    if (JAC) {
      double d = 0.0;
      int first = -1;
      for (int p = pa; p < pe; ++p) {
        if (A.colind[p] == i) {
          d = first < 0 ? A.vals[p] : d + A.vals[p];
          first = first < 0 ? p : first;
        }
      }
      if (first < 0 || (__double_as_longlong(d) << 1) == 0) {
        bad = 1;
        ars.s = 0.0;
      } else {
        ars.s = -A.jac_omega * jacobi_recip(d);
      }
      ars.p = first;
    }
    // One product: into the slot that holds c, else the next free one.  One fma
    // per product on a value picked by selects: the float64 pipe is the scarce
    // one on this part, and a product under each slot's predicate occupies it
    // once per slot.
    auto add = [&](double a, int c, double b) {
      bool at[N], found = false;
#pragma unroll
      for (int k = 0; k < N; ++k) {
        at[k] = key[k] == c;
        found |= at[k];
      }
      double cur = 0.0;
#pragma unroll
      for (int k = 0; k < N; ++k) {
        at[k] |= !found && k == n;
        cur = at[k] ? val[k] : cur;
      }
      n += found ? 0 : 1;
      const double t = fma(a, b, cur);
#pragma unroll
      for (int k = 0; k < N; ++k) {
        key[k] = at[k] ? c : key[k];
        val[k] = at[k] ? t : val[k];
      }
    };
    // the loads run ahead: the column of entry p + 3, the B row bounds of entry
    // p + 2 and the first B entry of entry p + 1 while entry p's products are added
    auto column = [&](int p) -> int { return p < pe ? A.colind[p] : -1; };
    auto bounds = [&](int p, int j, int& q, int& e, double& a) {
      q = e = 0;
      a = 0.0;
      if (j >= 0) {
        q = B.rowptr[j];
        e = B.rowptr[j + 1];
        a = A.vals[p];
      }
    };
    auto first = [&](int q, int e, int& c, double& b) {
      c = 0;
      b = 0.0;
      if (q < e) {
        c = B.colind[q];
        b = B.vals[q];
      }
    };
    int j2 = column(pa + 2), q0, e0, q1, e1, c0;
    double a0, a1, b0;
    bounds(pa, column(pa), q0, e0, a0);
    bounds(pa + 1, column(pa + 1), q1, e1, a1);
    first(q0, e0, c0, b0);
    for (int p = pa; p < pe; ++p) {
      const int j3 = column(p + 3);
      int q2, e2, c1;
      double a2, b1;
      bounds(p + 2, j2, q2, e2, a2);
      first(q1, e1, c1, b1);
      const double av = JAC ? a_scaled(ars, p, a0) : a0;
      for (int t = q0; t < e0; ++t) {
        add(av, c0, b0);
        if (t + 1 < e0) {
          c0 = B.colind[t + 1];
          b0 = B.vals[t + 1];
        }
      }
      j2 = j3;
      q0 = q1, e0 = e1, a0 = a1, c0 = c1, b0 = b1;
      q1 = q2, e1 = e2, a1 = a2;
    }
    if (n != cnt) mismatch = 1;
    if (n > N) over = 1;
#pragma unroll
    for (int k = 0; k < N; ++k) {
      int rank = 0;
#pragma unroll
      for (int l = 0; l < N; ++l) rank += (unsigned)key[l] < (unsigned)key[k] ? 1 : 0;  // free slots are last
      if (k < n && rank < cnt) {
        c_colind[off + rank] = key[k];
        c_vals[off + rank] = val[k];
      }
    }
  }
  if (over) set_status(status, KK_ERR_CAPACITY);
  if (mismatch) set_status(status, KK_ERR_STRUCTURE_MISMATCH);
  // a row without a stored diagonal, or whose diagonal sums to 0
  if (JAC && bad) set_status(status, KK_ERR_INVALID_ARG);
}

int thread_grid(const LaunchCtx& ctx, int nrows) {
  long long g = ((long long)nrows + kThreadBlock - 1) / kThreadBlock;
  const long long cap = (long long)ctx.num_sms * 16;
  if (g > cap) g = cap;
  return (int)(g < 1 ? 1 : g);
}

}  // namespace

cudaError_t launch_symbolic_thread(const LaunchCtx& ctx, const CsrView& A, const CsrView& B,
                                   const int32_t* rows, int32_t nrows, int32_t* cnt, long long max_flop) {
  if (nrows <= 0) return cudaSuccess;
  timer_begin(ctx.timer, ctx.stream, "sym_thread");
  auto kern = max_flop <= kThreadSymMax / 2 ? k_sym_thread<kThreadSymMax / 2> : k_sym_thread<kThreadSymMax>;
  kern<<<thread_grid(ctx, nrows), kThreadBlock, 0, ctx.stream>>>(A, B, rows, nrows, cnt, ctx.status);
  timer_end(ctx.timer, ctx.stream);
  return cudaGetLastError();
}

cudaError_t launch_numeric_thread(const LaunchCtx& ctx, const CsrView& A, const CsrView& B,
                                  const int64_t* c_rowptr, const int32_t* rows, int32_t nrows,
                                  int32_t* c_colind, double* c_vals, long long max_nnz) {
  if (nrows <= 0) return cudaSuccess;
  timer_begin(ctx.timer, ctx.stream, "num_thread");
  const bool jac = A.jac_s != nullptr;
  auto kern = max_nnz <= kThreadNumMax / 2
                  ? (jac ? k_num_thread<kThreadNumMax / 2, true> : k_num_thread<kThreadNumMax / 2, false>)
                  : (jac ? k_num_thread<kThreadNumMax, true> : k_num_thread<kThreadNumMax, false>);
  kern<<<thread_grid(ctx, nrows), kThreadBlock, 0, ctx.stream>>>(
      A, B, c_rowptr, rows, nrows, c_colind, c_vals, ctx.status);
  timer_end(ctx.timer, ctx.stream);
  return cudaGetLastError();
}

}  // namespace kk
