// Rank tier: numeric rows of up to 1,024 columns whose span fits a bit vector of at
// most 65,536 columns, one or two warps per row; symbolic rows of an unsorted B.
//
// The paper's dense accumulator (Sec. "Standard SpGEMM Kernel": bit vector and
// scalar array) over the row's span: the row's column bits are set, one pass
// over the words gives every 64-column group its prefix count, and a product's
// slot is its column's rank: prefix + popcount of the group's bits below it.
// The slots are C's row in column order, so there is no probing and no sort.
//
// What bounds it: issue and shared-memory accesses.  Rows here have up to a few
// hundred products spread over a wide span (random x random rows), so the
// pass over the words is done the cheap way for a warp: every lane takes a
// 16-byte piece of 128 columns, two pieces per warp scan (their counts packed
// into one register), about 25 instructions per 8,192 columns.  A list of the
// non-empty words costs more than that (summary bits, ordered list, a scan and
// an expansion per word; with a CTA of four warps per row and three barriers the
// window rows of a 256-pair batch took 8.9 ms and its hash rows 4.6, together 5.2
// here).  90,666 rows of about 500 columns of an unsorted B take 592 us: 1,250 with
// an entry of A at a time, 905 flattened, 800 without branches, then two warps per
// row where a row's shared memory leaves few of them on an SM.  C's columns come
// from the products themselves (each writes its column's offset beside its value),
// not from expanding the bits; a slot that no product wrote means that B is not the
// one whose compressed rows gave the bits.
//
// The row's products are walked flattened, 32 per step whatever the lengths of
// the B rows (an entry at a time left lanes idle and, for B rows of more than
// 32 entries, one load in flight), kRankBatch steps at a time: their loads,
// then their slots, then their additions are issued together.  Additions are
// plain (no atomics): the batch's products first write an id into a tag byte of
// their slot; those that share a slot find another's id there and are added
// afterwards one step at a time, in lane order.  Contributions to an entry are
// therefore added in A-row storage order (the oracle's order, bit-exact in
// float64), for sorted and unsorted B alike.
#include "kk_internal.h"
#include "kk_rowops.cuh"

namespace kk {
namespace {

constexpr unsigned kFull = 0xffffffffu;
constexpr int kRankThreads = 64;  // two rows of a warp each, or one row of two warps
// rows whose shared memory is larger than this take two warps (below it the SM
// holds as many one-warp rows as its registers allow)
constexpr uint32_t kRankPairBytes = 8 * 1024;
constexpr int kRankBatch = 4;  // steps of 32 products whose loads are issued together

__host__ __device__ constexpr size_t al16(size_t x) { return (x + 15) / 16 * 16; }

// Shared memory of a row of nw warps for a window of `words` 32-column words (a multiple
// of 128 nw) and vmax slots: bits u32[words] | word prefixes u16[words]
// | values u64[vmax + 2] (the last ones: spare slot) | A entries int4[nw][32]
// | columns u16[vmax + 2] | tags u8[vmax + 16]
struct RankGeom {
  int words, vmax;
  uint32_t pre_off, val_off, info_off, col_off, tag_off, bytes;
};
constexpr RankGeom rank_geom(int bits, int vmax, int nw) {
  RankGeom g{};
  // the window may start anywhere inside its first word
  const int unit = 128 * nw;
  g.words = (int)((((long long)bits + 31) / 32 + 1 + unit - 1) / unit * unit);
  g.vmax = vmax;
  g.pre_off = (uint32_t)g.words * 4;
  g.val_off = g.pre_off + (uint32_t)g.words * 2;
  g.info_off = g.val_off + (uint32_t)al16((size_t)(vmax + 2) * 8);
  g.col_off = g.info_off + (uint32_t)nw * 32 * 16;
  g.tag_off = g.col_off + (uint32_t)al16((size_t)(vmax + 2) * 2);
  g.bytes = g.tag_off + (uint32_t)al16((size_t)vmax + 16);
  return g;
}

// Every launch fits the 48 KB that need no function attribute: one set to each
// launch's own size could be lowered by another thread's launch in between.
constexpr size_t kRankPlainSmem = 48 * 1024 - 1024;
static_assert(rank_geom(kRankBits[kNumRankBits - 1], kRankNnz[kNumRankNnz - 1], 2).bytes <= kRankPlainSmem &&
                  kRankPairBytes * 2 <= kRankPlainSmem,
              "k_num_rank's shared memory");

struct RankArgs {
  CsrView A, B;
  BComp bcomp;                 // compressed B (sorted B only)
  const int32_t* row_lo;
  const float2* bspl;
  const int32_t* b_range_bad;
  const int64_t* c_rowptr;
  const int32_t* rows;
  int32_t nrows;
  int32_t* c_colind;
  double* c_vals;
  int* status;
  const u64* fp;  // structure fingerprints of the symbolic call and of this one (may be null)
};

// The products of up to 32 rows of entries, flattened: lane t's row holds len
// entries; the non-empty rows are numbered in lane order.
struct FlatRows {
  int start;  // this lane's row: flattened index of its first entry
  int k;      // ... and its number among the non-empty ones
  int total;
};
__device__ __forceinline__ FlatRows flat_rows(int len, int lane) {
  FlatRows f;
  const int incl = team_inclusive_scan<32>(len, lane, kFull);
  f.start = len > 0 ? incl - len : -1;
  f.total = __shfl_sync(kFull, incl, 31);
  f.k = __popc(__ballot_sync(kFull, len > 0) & ((1u << lane) - 1u));
  return f;
}
// Rows that start before flattened entry f0.
__device__ __forceinline__ int flat_seen(const FlatRows& f, int f0) {
  return __popc(__ballot_sync(kFull, f.start >= 0 && f.start < f0));
}
// Number of the row that holds flattened entry f0 + lane; seen = rows that start
// before f0 (updated).  The rows that start in the step are found by one warp
// reduction, so there is no search.
__device__ __forceinline__ int flat_owner(const FlatRows& f, int f0, int lane, int& seen) {
  const unsigned at = (unsigned)(f.start - f0);
  const unsigned starts = __reduce_or_sync(kFull, f.start >= 0 && at < 32u ? 1u << at : 0u);
  const int own = seen + __popc(starts & (0xffffffffu >> (31 - lane))) - 1;
  seen += __popc(starts);
  return own;
}

// vals[rank] += a * b, in DF32 or float64.
template <bool DFM>
__device__ __forceinline__ u64 rank_add(u64 v, bool df, int2 a, float2 b) {
  if (DFM && df) {
    DF av, bv, s = df_unpack(v);
    av.hi = __int_as_float(a.x);
    av.lo = __int_as_float(a.y);
    bv.hi = b.x;
    bv.lo = b.y;
    df_fma(s, av, bv);
    return df_pack(s);
  }
  const double x = __hiloint2double(a.y, a.x);
  const double y = __hiloint2double(__float_as_int(b.y), __float_as_int(b.x));
  return (u64)__double_as_longlong(fma(x, y, __longlong_as_double((long long)v)));
}

// Symbolic phase of rows of an unsorted B: the row's column bits as in k_num_rank,
// counted as they are set (those that an OR finds clear), one warp per row.  A hash
// set takes a chain of probes for every product; here the products of four steps
// are loaded together and each costs one OR (90,666 rows of 510 products in 60,013
// columns: 657 us by hash, 123 so; bound by the ORs and the load latency).
constexpr int kSymRankWarps = 4;
static_assert((size_t)kSymRankWarps * rank_geom(kRankBits[kNumRankBits - 1], 0, 1).words * 4 <= kRankPlainSmem,
              "k_sym_rank's shared memory");
__global__ void __launch_bounds__(kSymRankWarps * 32)
k_sym_rank(CsrView A, CsrView B, const int32_t* __restrict__ rows, int32_t nrows, int32_t nwords,
           int32_t* __restrict__ cnt, int* status) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ int qbase[kSymRankWarps][32];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  uint32_t* bits = reinterpret_cast<uint32_t*>(smem_raw) + (size_t)warp * nwords;
  uint4* bits4 = reinterpret_cast<uint4*>(bits);
  int* qb = qbase[warp];
  const uint32_t words = (uint32_t)nwords;
  int bad = 0;
  for (int r = blockIdx.x * kSymRankWarps + warp; r < nrows; r += gridDim.x * kSymRankWarps) {
    const int i = rows[r];
    const int pa = A.rowptr[i], pe = A.rowptr[i + 1];
    for (int q = lane; q < nwords / 4; q += 32) bits4[q] = make_uint4(0u, 0u, 0u, 0u);
    int c = 0;
    for (int p0 = pa; p0 < pe; p0 += 32) {
      int xs = 0, ys = 0;
      if (p0 + lane < pe) {
        const int j = A.colind[p0 + lane];
        xs = B.rowptr[j];
        ys = B.rowptr[j + 1] - xs;
      }
      const FlatRows f = flat_rows(ys, lane);
      __syncwarp();
      if (ys > 0) qb[f.k] = xs - f.start;
      __syncwarp();
      int seen = 0;
      for (int f0 = 0; f0 < f.total; f0 += 32 * kRankBatch) {
        int v[kRankBatch];
#pragma unroll
        for (int u = 0; u < kRankBatch; ++u) {
          const int fl = min(f0 + u * 32 + lane, f.total - 1);
          v[u] = B.colind[qb[flat_owner(f, f0 + u * 32, lane, seen)] + fl];
        }
#pragma unroll
        for (int u = 0; u < kRankBatch; ++u) {
          const uint32_t w = (uint32_t)v[u] >> 5, bit = 1u << (v[u] & 31);
          bad |= w >= words;
          if (w < words) c += !(atomicOr(&bits[w], bit) & bit);
        }
      }
    }
    c = team_sum<32>(c, kFull);
    if (lane == 0) cnt[i] = c;
    __syncwarp();
  }
  if (bad) set_status(status, KK_ERR_CAPACITY);
}

// SORTED: B's rows strictly ascending; the bits come from the compressed B and
// a product outside them means that B's structure is not the one they were
// built from (KK_ERR_STRUCTURE_MISMATCH).  Otherwise the bits come from B's
// columns and the window starts at column 0.  DFM: the call asks for DF32
// (rows outside its bounds run in float64 all the same).
// NW: warps per row (they split the words and the products of a batch).
template <int NW, bool SORTED, bool DFM>
__global__ void __launch_bounds__(kRankThreads, 14) k_num_rank(RankArgs g, RankGeom geo) {
  constexpr int RPC = kRankThreads / 32 / NW;  // rows per CTA
  constexpr int NT = NW * 32;                  // threads per row
  constexpr int BATCH = NT * kRankBatch;       // products per batch (ids fit the tag byte)
  static_assert(BATCH <= 256, "tag ids are bytes");
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ int part_total[NW];
  const int lane = threadIdx.x & 31, part = NW == 1 ? 0 : threadIdx.x >> 5;
  const int slot = NW == 1 ? threadIdx.x >> 5 : 0, tid = part * 32 + lane;
  unsigned char* base = smem_raw + (size_t)slot * geo.bytes;
  uint32_t* bits = reinterpret_cast<uint32_t*>(base);
  uint4* bits4 = reinterpret_cast<uint4*>(base);
  const uint16_t* pre = reinterpret_cast<const uint16_t*>(base + geo.pre_off);
  uint2* pre4 = reinterpret_cast<uint2*>(base + geo.pre_off);
  u64* vals = reinterpret_cast<u64*>(base + geo.val_off);
  int4* ainfo = reinterpret_cast<int4*>(base + geo.info_off) + part * 32;
  uint16_t* cols = reinterpret_cast<uint16_t*>(base + geo.col_off);
  uint8_t* tag = base + geo.tag_off;
  const int vmax = geo.vmax, n4 = geo.words >> 2, n4p = n4 / NW;  // 16-byte pieces, per warp
  const uint32_t words = (uint32_t)geo.words, half = words / 2;
  auto sync = [&]() {
    if constexpr (NW == 1) __syncwarp();
    else __syncthreads();
  };
  auto any = [&](bool p) -> bool {
    if constexpr (NW == 1) return __any_sync(kFull, p);
    else return __syncthreads_or(p) != 0;
  };
  const int32_t* __restrict__ acol = g.A.colind;
  const int32_t* __restrict__ brp = g.B.rowptr;
  const int32_t* __restrict__ bcol = g.B.colind;
  const double* __restrict__ bval = g.B.vals;
  const bool df_all = DFM && *g.b_range_bad == 0;
  if (g.fp && blockIdx.x == 0 && threadIdx.x == 0 && g.fp[0] != g.fp[1])
    set_status(g.status, KK_ERR_STRUCTURE_MISMATCH);
  for (int q = tid; q < n4; q += NT) bits4[q] = make_uint4(0u, 0u, 0u, 0u);
  sync();
  const int nw = gridDim.x * RPC;  // rows dealt round-robin over the grid
  int r = blockIdx.x * RPC + slot;
  // the next row's id, bounds and first chunk of A entries are loaded while a
  // row is processed (the chain of dependent loads is otherwise exposed)
  int i = 0, pa = 0, pe = 0, lo = 0, x = 0, y = 0, z = 0, i_n = -1;
  if (r < g.nrows) {
    i = g.rows[r];
    pa = g.A.rowptr[i];
    pe = g.A.rowptr[i + 1];
    lo = g.row_lo[i];
    if (pa + lane < pe) {
      const int j = acol[pa + lane];
      x = brp[j];
      y = brp[j + 1] - x;
      z = SORTED ? g.bcomp.len[j] : y;
    }
    if (r + nw < g.nrows) i_n = g.rows[r + nw];
  }
  for (; r < g.nrows; r += nw) {
    const int64_t off = g.c_rowptr[i];
    const int cnt = (int)(g.c_rowptr[i + 1] - off);
    double a = pa + lane < pe ? a_value(g.A, i, pa + lane) : 0.0;
    int pa_n = 0, pe_n = 0, lo_n = 0;
    if (i_n >= 0) {
      pa_n = g.A.rowptr[i_n];
      pe_n = g.A.rowptr[i_n + 1];
      lo_n = g.row_lo[i_n];
    }
    const int i_nn = r + 2 * nw < g.nrows ? g.rows[r + 2 * nw] : -1;
    const int lo_w = SORTED ? lo >> 5 : 0;
    const int lo_c = lo_w * 32;
    int bad = 0;
    // the row's column bits: the (word, mask) pairs of the compressed rows, or
    // the columns themselves
    for (int p0 = pa; p0 < pe; p0 += 32) {
      int xs = x, ys = z;
      if (p0 != pa) {
        xs = ys = 0;
        if (p0 + lane < pe) {
          const int j = acol[p0 + lane];
          xs = brp[j];
          ys = SORTED ? g.bcomp.len[j] : brp[j + 1] - xs;
        }
      }
      const FlatRows f = flat_rows(ys, lane);
      int* qb = reinterpret_cast<int*>(ainfo);
      if (ys > 0) qb[f.k] = xs - f.start;
      __syncwarp();
      for (int f0 = part * (BATCH / NW); f0 < f.total; f0 += BATCH) {
        int seen = flat_seen(f, f0);
        int2 v[kRankBatch];
#pragma unroll
        for (int u = 0; u < kRankBatch; ++u) {
          // lanes past the end repeat the last entry (its bits are set twice)
          const int fl = min(f0 + u * 32 + lane, f.total - 1);
          const int q = qb[flat_owner(f, f0 + u * 32, lane, seen)] + fl;
          if (SORTED) {
            v[u] = g.bcomp.bc[q];
          } else {
            const int c = bcol[q];
            v[u] = make_int2(c >> 5, (int)(1u << (c & 31)));
          }
        }
#pragma unroll
        for (int u = 0; u < kRankBatch; ++u) {
          const uint32_t w = (uint32_t)(v[u].x - lo_w);
          bad |= w >= words;
          atomicOr(&bits[min(w, words - 1)], w < words ? (uint32_t)v[u].y : 0u);
        }
      }
      __syncwarp();
    }
    const int nout = min(cnt, vmax);
    // a slot's column comes from its products: offset 0 stands for none yet (the
    // offsets ascend; that of a sorted B's slot 0 is 0, so 1 stands for it there)
    for (int e = tid; e < nout; e += NT) {
      vals[e] = 0ull;
      cols[e] = SORTED && e == 0 ? 1 : 0;
    }
    if (NW > 1) sync();
    int j_n = -1;
    if (i_n >= 0 && pa_n + lane < pe_n) j_n = acol[pa_n + lane];
    // prefix count of every word within the warp's part: pieces of 128 columns,
    // two per scan
    int run = 0;
    for (int k = 0; k < n4p; k += 64) {
      const bool two = k + 32 < n4p;
      const int q0 = part * n4p + k + lane;
      const uint4 v0 = bits4[q0];
      const uint4 v1 = two ? bits4[q0 + 32] : make_uint4(0u, 0u, 0u, 0u);
      const int p1 = __popc(v0.x), p2 = p1 + __popc(v0.y), p3 = p2 + __popc(v0.z), c0 = p3 + __popc(v0.w);
      const int q1 = __popc(v1.x), q2 = q1 + __popc(v1.y), q3 = q2 + __popc(v1.z), c1 = q3 + __popc(v1.w);
      const int incl = team_inclusive_scan<32>(c0 | (c1 << 16), lane, kFull);
      const int tot = __shfl_sync(kFull, incl, 31);
      // (a count beyond 16 bits belongs to a row reported below)
      const unsigned b0 = (unsigned)(run + (incl & 0xffff) - c0) & 0xffffu;
      pre4[q0] = make_uint2(b0 | ((b0 + p1) << 16), ((b0 + p2) & 0xffffu) | ((b0 + p3) << 16));
      run += tot & 0xffff;
      if (two) {
        const unsigned b1 = (unsigned)(run + (int)((unsigned)incl >> 16) - c1) & 0xffffu;
        pre4[q0 + 32] = make_uint2(b1 | ((b1 + q1) << 16), ((b1 + q2) & 0xffffu) | ((b1 + q3) << 16));
        run += (int)((unsigned)tot >> 16);
      }
    }
    int low = 0;  // columns in the first warp's part
    if (NW > 1) {
      if (lane == 0) part_total[part] = run;
      sync();
      low = part_total[0];
      run = part_total[0] + part_total[NW - 1];
    }
    if (run != cnt) bad = 1;
    // arithmetic of this row: float64 unless DF32 is asked for and its bound holds
    const bool df = df_all && df_row_terms_ok(pa, pe) && row_df_ok<32>(g.A.vals, pa, pe, lane, kFull);
    // values and columns
    for (int p0 = pa; p0 < pe; p0 += 32) {
      int xs = x, ys = y;
      if (p0 != pa) {
        xs = ys = 0;
        a = 0.0;
        if (p0 + lane < pe) {
          const int j = acol[p0 + lane];
          xs = brp[j];
          ys = brp[j + 1] - xs;
          a = a_value(g.A, i, p0 + lane);
        }
      }
      const FlatRows f = flat_rows(ys, lane);
      int2 az = make_int2(__double2loint(a), __double2hiint(a));
      if (DFM && df) {
        DF ad;
        df_split(a, ad);
        az = make_int2(__float_as_int(ad.hi), __float_as_int(ad.lo));
      }
      if (ys > 0) ainfo[f.k] = make_int4(xs - f.start, 0, az.x, az.y);
      __syncwarp();
      for (int f0 = 0; f0 < f.total; f0 += BATCH) {
        const int fp = f0 + part * (BATCH / NW);
        int seen = flat_seen(f, fp);
        int s[kRankBatch];
        int2 av[kRankBatch];
        float2 b[kRankBatch];
        {
          int c[kRankBatch];
#pragma unroll
          for (int u = 0; u < kRankBatch; ++u) {
            // lanes past the end take the last product to a slot that is not read
            const int fl = min(fp + u * 32 + lane, f.total - 1);
            const int4 in = ainfo[min(flat_owner(f, fp + u * 32, lane, seen), 31)];
            const int q = in.x + fl;
            av[u] = make_int2(in.z, in.w);
            c[u] = bcol[q];
            if (DFM && df) {
              b[u] = g.bspl[q];
            } else {
              const double bb = bval[q];
              b[u] = make_float2(__int_as_float(__double2loint(bb)), __int_as_float(__double2hiint(bb)));
            }
          }
          // slots: the column's rank (vmax, never read, outside the bits)
#pragma unroll
          for (int u = 0; u < kRankBatch; ++u) {
            const uint32_t o = (uint32_t)(c[u] - lo_c), w = min(o >> 5, words - 1);
            const uint32_t m = bits[w], bit = 1u << (o & 31);
            const bool member = (o >> 5) == w && (m & bit) != 0u;
            bad |= !member;
            int rank = (int)pre[w] + __popc(m & (bit - 1u));
            if (NW > 1) rank += w >= half ? low : 0;
            s[u] = member ? min(rank, vmax) : vmax;
            if (fp + u * 32 + lane >= f.total) s[u] = vmax + 1;
            cols[s[u]] = (uint16_t)(c[u] - lo);
            tag[s[u]] = (uint8_t)(tid + u * NT);
          }
        }
        sync();
        unsigned lost = 0u;  // bit u: the product of step u shares its slot
#pragma unroll
        for (int u = 0; u < kRankBatch; ++u)
          lost |= s[u] <= vmax && tag[s[u]] != (uint8_t)(tid + u * NT) ? 1u << u : 0u;
        const bool clash = any(lost != 0u);
        if (clash) {
          // those that lost write their id again, so that the one whose id was
          // there finds out too
#pragma unroll
          for (int u = 0; u < kRankBatch; ++u)
            if (lost >> u & 1u) tag[s[u]] = (uint8_t)(tid + u * NT);
          sync();
#pragma unroll
          for (int u = 0; u < kRankBatch; ++u)
            lost |= s[u] <= vmax && tag[s[u]] != (uint8_t)(tid + u * NT) ? 1u << u : 0u;
        }
        {
          u64 v[kRankBatch];
#pragma unroll
          for (int u = 0; u < kRankBatch; ++u) v[u] = vals[s[u]];
#pragma unroll
          for (int u = 0; u < kRankBatch; ++u)
            if (!(lost >> u & 1u)) vals[s[u]] = rank_add<DFM>(v[u], df, av[u], b[u]);
        }
        if (clash) {
          // products that share a slot, in order: warps, steps, lanes
#pragma unroll
          for (int w = 0; w < NW; ++w) {
            __syncwarp();
            if (part == w) {
#pragma unroll
              for (int u = 0; u < kRankBatch; ++u) {
                const bool mine = (lost >> u & 1u) != 0u;
                const unsigned m = __ballot_sync(kFull, mine);
                if (m == 0u) continue;
                int turn = 0, last = 0;
                if (m & (m - 1u)) {
                  const unsigned peers = __match_any_sync(kFull, mine ? s[u] : -1 - lane);
                  turn = mine ? __popc(peers & ((1u << lane) - 1u)) : 0;
                  last = (int)__reduce_max_sync(kFull, (unsigned)turn);
                }
                for (int t = 0; t <= last; ++t) {
                  if (mine && turn == t) vals[s[u]] = rank_add<DFM>(vals[s[u]], df, av[u], b[u]);
                  __syncwarp();
                }
              }
            }
            if (NW > 1) sync();
          }
        }
        sync();
      }
    }
    int x_n = 0, y_n = 0, z_n = 0;
    if (j_n >= 0) {
      x_n = brp[j_n];
      y_n = brp[j_n + 1] - x_n;
      z_n = SORTED ? g.bcomp.len[j_n] : y_n;
    }
    for (int e = tid; e < nout; e += NT) {
      const int o = (int)cols[e];
      bad |= SORTED && (e == 0) != (o == 0);  // a column of the bits without a product
      g.c_colind[off + e] = lo + (SORTED && e == 0 ? 0 : o);
      g.c_vals[off + e] = out_value(vals[e], DFM && df);
    }
    if (bad) set_status(g.status, KK_ERR_STRUCTURE_MISMATCH);
    for (int q = tid; q < n4; q += NT) bits4[q] = make_uint4(0u, 0u, 0u, 0u);
    sync();
    i = i_n;
    pa = pa_n;
    pe = pe_n;
    lo = lo_n;
    x = x_n;
    y = y_n;
    z = z_n;
    i_n = i_nn;
  }
}

}  // namespace

cudaError_t launch_sym_rank(const LaunchCtx& ctx, const BinSpec& bin, const CsrView& A, const CsrView& B,
                            const int32_t* rows, int32_t nrows, int32_t* cnt) {
  if (nrows <= 0) return cudaSuccess;
  const int nwords = rank_geom(B.n < bin.slots ? B.n : bin.slots, 0, 1).words;
  const size_t smem = (size_t)kSymRankWarps * nwords * 4;
  int per_sm = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_sym_rank, kSymRankWarps * 32, smem) != cudaSuccess ||
      per_sm < 1) {
    (void)cudaGetLastError();
    per_sm = 1;
  }
  long long blocks = ((long long)nrows + kSymRankWarps - 1) / kSymRankWarps;
  if (blocks > (long long)ctx.num_sms * per_sm) blocks = (long long)ctx.num_sms * per_sm;
  timer_begin(ctx.timer, ctx.stream, "sym_rank");
  k_sym_rank<<<(int)blocks, kSymRankWarps * 32, smem, ctx.stream>>>(A, B, rows, nrows, nwords, cnt, ctx.status);
  timer_end(ctx.timer, ctx.stream);
  return cudaGetLastError();
}

cudaError_t launch_num_rank(const LaunchCtx& ctx, const BinSpec& bin, const CsrView& A, const CsrView& B,
                            int32_t b_sorted, const BComp& bcomp, const float2* b_split,
                            const int32_t* b_range_bad, int32_t arith, const int64_t* c_rowptr,
                            const int32_t* rows, int32_t nrows, int32_t* c_colind, double* c_vals) {
  if (nrows <= 0) return cudaSuccess;
  const bool df = arith == kArithDF32 && !ctx.kept_f64;
  const int bits = B.n < bin.slots ? B.n : bin.slots;  // no wider than B
  const int nw = rank_geom(bits, (int)bin.hi, 1).bytes > kRankPairBytes ? 2 : 1;
  const RankGeom geo = rank_geom(bits, (int)bin.hi, nw);
  auto kern = nw == 2 ? (b_sorted ? (df ? k_num_rank<2, true, true> : k_num_rank<2, true, false>)
                                  : (df ? k_num_rank<2, false, true> : k_num_rank<2, false, false>))
                      : (b_sorted ? (df ? k_num_rank<1, true, true> : k_num_rank<1, true, false>)
                                  : (df ? k_num_rank<1, false, true> : k_num_rank<1, false, false>));
  const int rpc = kRankThreads / 32 / nw;  // rows per CTA
  const size_t smem = (size_t)rpc * geo.bytes;
  // one resident wave: neighbouring rows are in flight together and share B rows in L2
  int per_sm = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, kRankThreads, smem) != cudaSuccess ||
      per_sm < 1) {
    (void)cudaGetLastError();
    per_sm = 1;
  }
  long long blocks = ((long long)nrows + rpc - 1) / rpc;
  if (blocks > (long long)ctx.num_sms * per_sm) blocks = (long long)ctx.num_sms * per_sm;
  timer_begin(ctx.timer, ctx.stream, "num_rank");
  const RankArgs g{A, B, bcomp, ctx.row_lo, b_split, b_range_bad, c_rowptr, rows, nrows, c_colind, c_vals,
                   ctx.status, ctx.fingerprint};
  kern<<<(int)blocks, kRankThreads, smem, ctx.stream>>>(g, geo);
  timer_end(ctx.timer, ctx.stream);
  return cudaGetLastError();
}

}  // namespace kk
