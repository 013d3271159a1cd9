// Heavy rows: rows with too many products for the one-warp workspaces.  One
// CTA owns one row, or one window of a row's output (the shard pattern of
// Sec. 4), so every output segment is written by one CTA and no CTA waits on
// another.
//
// Dense rows (kClsRcd): the row's column range is at most 65,536 columns and
// it has at most kRcdMaxA stored A entries (typically hub rows: few stored A
// entries whose B rows are long).
//   symbolic: every product stores 1 into the flag byte of its column (plain
//             byte stores, no atomics: the store is idempotent, the sparse
//             byte-map workspace); the flags are then packed into a bitmap that
//             stays in the plan, and nnz of the row is its population count.
//   numeric:  the row's output is cut into windows of consecutive entries
//             (ranks), each an item of its own; a CTA reads the row's bitmap
//             back, ranks its words, writes the window's columns from it and
//             adds a * b at the rank of every product that falls into the
//             window (at its column if a window covers them all).  The CTA takes one long B row at a time: its columns are
//             distinct, so the adds need no atomics.
//
// Wide rows (kClsWb): column range up to 2^20 columns.  A bitmap over the
// whole range (one bit per column) is the workspace:
//   symbolic: atomicOr every product column, count the bits that were 0; the
//             bitmap stays in the plan if there is room.
//   numeric:  read the bitmap back (or set the bits again), rank it in 128-bit
//             chunks, write C's column indices in order straight from it, zero
//             C's values, and let every product add its value at the rank of its
//             column in C (global atomic add).  The products of a row of more
//             than kWbPart are cut into parts, an item each.
#include <climits>
#include <cstddef>

#include "ws_internal.cuh"

namespace wsk {

namespace {

constexpr int kRcdThreads = 512;
constexpr int kWbThreads = 1024;  // one CTA per SM (its 128 KB bitmap), so 32 warps hide the gathers
constexpr int kWbBatch = 4;  // stored A entries a lane group has in flight in the wide-bitmap numeric pass

// ---------------------------------------------------------------- dense rows

constexpr int kRcdCacheA = 1024;  // stored A entries handled at a time
constexpr int kRcdWords = kMaxBitmapSpan / 32;
constexpr long long kRcdBigProducts = 32768;  // rows with more products are taken first
static_assert(kRcdWords == 4 * kRcdThreads, "four bitmap words per thread");
static_assert(kRcdCacheA == 2 * kRcdThreads, "two cached entries per thread");

// The parts of B rows a CTA walks next: those of up to kRcdCacheA stored A
// entries.  Parts of more than SHORT entries are cut into pieces of PIECE;
// first[j] counts the pieces before entry j.
struct RcdParts {
  long long b0[kRcdCacheA];   // first position of the part in B
  int len[kRcdCacheA];
  int first[kRcdCacheA + 2];
};

// Exclusive scan of the piece counts of the cached entries 0..n-1 (two
// consecutive ones per thread).  Every thread calls it; returns the total.
template <int PIECE, int SHORT>
__device__ __forceinline__ int rcd_scan_pieces(RcdParts& e, int n, int* s_scan) {
  const int j = threadIdx.x * 2;
  auto pieces = [&](int i) { return i < n && e.len[i] > SHORT ? (e.len[i] + PIECE - 1) / PIECE : 0; };
  const int p0 = pieces(j), p1 = pieces(j + 1);
  int total;
  const int before = block_exclusive_scan(p0 + p1, s_scan, &total);
  e.first[j] = before;
  e.first[j + 1] = before + p0;
  if (threadIdx.x == 0) e.first[kRcdCacheA] = total;
  __syncthreads();
  return total;
}

// Symbolic pass.  The warps share the row's B rows in pieces of kSymPiece
// entries, so a row of a few long B rows keeps every warp busy: 610 us on
// R-MAT 2^16 squared, a warp per B row 906 us.  Bound by the shared-memory
// pipe (60% of its peak) and the barriers of a row.
constexpr int kSymPiece = 256;
constexpr int kSymShort = 32;  // B rows up to this length: a group of kSymLanes lanes, one round of loads
constexpr int kSymLanes = 8;
static_assert(kSymLanes * 4 >= kSymShort, "a short B row takes one round of loads");

struct RcdSymbolic {
  alignas(16) uint8_t flags[kMaxBitmapSpan];  // read in 16-byte words
  RcdParts e;
};

// AGAIN: the numeric pass makes the bitmaps once more; a column outside the
// row's range (the input changed since) is left out and reported.
template <typename T, bool AGAIN>
__global__ void __launch_bounds__(kRcdThreads, 2) rcd_symbolic_kernel(const RowPlan<T> p) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  RcdSymbolic& s = *reinterpret_cast<RcdSymbolic*>(smem_raw);
  RcdParts& e = s.e;
  __shared__ int s_scan[32];
  __shared__ long long s_sums[32];
  __shared__ int s_row;
  constexpr int kWarps = kRcdThreads / 32;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  uint4* flags4 = reinterpret_cast<uint4*>(s.flags);
  for (int i = threadIdx.x; i < kMaxBitmapSpan / 16; i += kRcdThreads) flags4[i] = make_uint4(0u, 0u, 0u, 0u);
  bool bad = false;
  for (int64_t guard = 0; guard <= p.seg_len; ++guard) {
    if (threadIdx.x == 0) s_row = atomicAdd(&p.rcd_ctr[kRcdNextRow], 1);
    __syncthreads();
    const int r = s_row;
    if (r >= p.seg_len) break;
    const int32_t row = p.perm[p.seg_begin + r];
    const int lo = p.lo[row];
    const int span = p.hi[row] - lo + 1;
    const int64_t ra = p.A.rowptr[row], re = p.A.rowptr[row + 1];
    auto flag = [&](int c) {
      if constexpr (AGAIN) {
        uint32_t off;
        if (column_place(c, lo, span, &off)) {
          s.flags[off] = 1;
        } else {
          bad |= c >= 0;
        }
      } else {
        if (c >= 0) s.flags[c - lo] = 1;
      }
    };
    long long products = 0;
    for (int64_t e0 = ra; e0 < re; e0 += kRcdCacheA) {
      const int n = static_cast<int>(min(static_cast<int64_t>(kRcdCacheA), re - e0));
      for (int j = threadIdx.x; j < n; j += kRcdThreads) {
        const int k = p.A.colidx[e0 + j];
        const int64_t b0 = p.B.rowptr[k];
        e.b0[j] = b0;
        e.len[j] = static_cast<int>(p.B.rowptr[k + 1] - b0);
        products += e.len[j];
      }
      __syncthreads();
      const int npieces = rcd_scan_pieces<kSymPiece, kSymShort>(e, n, s_scan);
      // Long B rows: the warp's pieces are consecutive, so it finds its first
      // entry by a binary search and then only moves on.
      const int pc1 = static_cast<int>(static_cast<long long>(npieces) * (warp + 1) / kWarps);
      int pc = static_cast<int>(static_cast<long long>(npieces) * warp / kWarps);
      int jl = 0, jh = n - 1;  // the last entry whose first piece is <= pc
      while (pc < pc1 && jl < jh) {
        const int mid = (jl + jh + 1) >> 1;
        if (e.first[mid] <= pc) {
          jl = mid;
        } else {
          jh = mid - 1;
        }
      }
      for (; pc < pc1; ++pc) {
        while (jl + 1 < n && e.first[jl + 1] <= pc) ++jl;
        const int t0 = (pc - e.first[jl]) * kSymPiece + lane, end = e.len[jl];
        const int32_t* cols = p.B.colidx + e.b0[jl];
        int c[kSymPiece / 32];
#pragma unroll
        for (int u = 0; u < kSymPiece / 32; ++u) c[u] = t0 + u * 32 < end ? cols[t0 + u * 32] : -1;
#pragma unroll
        for (int u = 0; u < kSymPiece / 32; ++u) flag(c[u]);
      }
      for (int j = warp * (32 / kSymLanes) + lane / kSymLanes; j < n; j += kWarps * (32 / kSymLanes)) {
        const int len = e.len[j];
        if (len > kSymShort) continue;
        const int32_t* cols = p.B.colidx + e.b0[j];
        int c[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) c[u] = lane % kSymLanes + u * kSymLanes < len ? cols[lane % kSymLanes + u * kSymLanes] : -1;
#pragma unroll
        for (int u = 0; u < 4; ++u) flag(c[u]);
      }
      __syncthreads();
    }
    // Packs 16 flag bytes into 16 bits of the plan's bitmap, counts and clears them.
    uint16_t* bits16 = reinterpret_cast<uint16_t*>(p.rcd_bits + static_cast<int64_t>(r) * p.rcd_words);
    int cnt = 0;
    for (int i = threadIdx.x; i < p.rcd_words * 2; i += kRcdThreads) {
      uint32_t m = 0;
      if (i * 16 < span) {
        const uint4 v = flags4[i];
        flags4[i] = make_uint4(0u, 0u, 0u, 0u);
        // byte k of a word (0 or 1) to bit 24 + k of the product
        m = ((v.x * 0x01020408u) >> 24 & 15u) | ((v.y * 0x01020408u) >> 24 & 15u) << 4 |
            ((v.z * 0x01020408u) >> 24 & 15u) << 8 | ((v.w * 0x01020408u) >> 24 & 15u) << 12;
      }
      bits16[i] = static_cast<uint16_t>(m);
      cnt += __popc(m);
    }
    // products in the high half, entries in the low half of one sum
    long long sums;
    block_exclusive_scan((products << 32) | cnt, s_sums, &sums);
    if (threadIdx.x == 0) {
      const int total = static_cast<int>(sums & 0xffffffffll);
      const bool big = (sums >> 32) > kRcdBigProducts;
      if (!AGAIN) p.c_rowptr[row + 1] = total;
      const int nw = (total + p.rcd_width - 1) / p.rcd_width;
      const long long cap = static_cast<long long>(p.seg_len) * p.rcd_slices;
      if (big) {
        const int at = atomicAdd(&p.rcd_ctr[kRcdBigItems], nw);
        for (int w = 0; w < nw; ++w) p.rcd_items[at + w] = static_cast<long long>(r) * p.rcd_slices + w;
      } else {
        const int at = atomicAdd(&p.rcd_ctr[kRcdItems], nw);
        for (int w = 0; w < nw; ++w) p.rcd_items[cap - 1 - at - w] = static_cast<long long>(r) * p.rcd_slices + w;
      }
    }
  }
  if (AGAIN && bad) atomicOr(p.status, kErrCount);
}

// Numeric pass: one item (row, window of p.rcd_width output ranks) per CTA at a
// time, the items of rows with many products first.
//
// A B row part of more than kNumShort entries is taken by the whole CTA, in
// rounds of kNumThreads * PER entries: its columns are distinct, so the window is
// updated with a load, one multiply-add and a store, and a barrier separates
// it from the next part.  Shared-memory fp64 adds by compare-and-swap were
// what bound this pass: this GPU issues an fp64 instruction over about 16
// cycles of the SM, a swap loop that loses its slot repeats it, and a multiply
// followed by the built-in atomic add pays it twice.  Measured on R-MAT 2^16
// (edge factor 16, fp64) squared, 372 million products in these rows: 2.6 ms;
// the built-in adds over column slices 3.6 ms; pieces spread over the warps
// with a fused multiply-add in a swap loop 9.2 ms.  The multiply-adds alone
// keep the fp64 pipe busy for 0.8 ms; the rest is the latency of an item's
// other steps, which three CTAs per SM overlap (windows of 64 KB with two CTAs
// per SM: 3.9 ms against 3.3 ms).  Columns and values are loaded kAhead rounds
// before they are added and ranked one round before.  Parts of up to 96 entries
// go to a warp each and are added atomically (R-MAT 2^16 and 2^14 squared: 3.46
// and 0.405 ms in all; groups of 16 lanes for up to 64 entries 3.51 and 0.429; a
// warp for up to 256 entries 3.53 and 0.421).
// Parts of up to 16 entries take four lanes each: hub rows over short B rows
// are bound by the latency of the parts in flight, and a warp per part had the
// fewest (4000 rows of 2000 entries times rows of 3 over 4000 columns, fp32: 1.31
// ms in all with a warp, 0.69 with four lanes, 0.75 with eight; of 8 over
// 60,000 1.28, 0.76 and 0.80; of 16 over 30,000 0.52, 0.40 and 0.39; the column
// slices before the windows 0.93, 1.17 and 0.67).
constexpr int kNumThreads = 256;
constexpr int kNumCacheA = kNumThreads;       // stored A entries handled at a time
constexpr int kNumDesc = 128;                 // rounds described at a time
constexpr int kNumWords = kRcdWords / kNumThreads;  // bitmap words per thread
constexpr int kNumShort = kRcdLongB;  // a warp each, three entries per lane
constexpr int kNumTiny = 16;    // a group of kNumTinyLanes lanes each
constexpr int kNumTinyLanes = 4;
constexpr int kAhead = 3;
static_assert(kNumShort % 32 == 0, "whole entries per lane");
static_assert(kNumWords == 8, "two 16-byte words of the bitmap per thread");

// One round: entries [b, b + n) of B, times a stored A entry (cached entry j).
struct alignas(16) RcdRound {
  long long b;
  int n;
  int j;
};

template <typename T>
struct RcdNumeric {
  static constexpr int kWidth = kRcdWidthBytes / static_cast<int>(sizeof(T));
  alignas(16) T win[kWidth];          // accessed in 16-byte words too
  RcdRound round[kNumDesc];
  alignas(16) uint2 rk[kRcdWords];    // bitmap word and the rank, in the window, of its first column
  long long b0[kNumCacheA];           // parts of B rows: first position,
  T a[kNumCacheA];                    //   the A value,
  int len[kNumCacheA];                //   length,
  int first[kNumCacheA];              //   rounds before the part
};

// Start and end of the part of the sorted cols[0..n) inside [c0, c1]: two
// searches in 4-way steps whose six loads are in flight together.
__device__ __forceinline__ void part_bounds(const int32_t* cols, int n, int c0, int c1, int* start, int* end) {
  int l[2] = {0, 0}, h[2] = {n, n};
  const int limit[2] = {c0, c1};  // first column >= c0, first column > c1
  auto before = [&](int i, int v) { return i == 0 ? v < limit[0] : v <= limit[1]; };
  while (h[0] - l[0] >= 4 || h[1] - l[1] >= 4) {
    int v[2][3];
#pragma unroll
    for (int i = 0; i < 2; ++i) {
      const int q = (h[i] - l[i]) >> 2;
#pragma unroll
      for (int t = 0; t < 3; ++t) v[i][t] = h[i] - l[i] >= 4 ? cols[l[i] + (t + 1) * q] : 0;
    }
#pragma unroll
    for (int i = 0; i < 2; ++i) {
      const int q = (h[i] - l[i]) >> 2, m = l[i];
      if (h[i] - m < 4) continue;
      if (before(i, v[i][1])) {
        l[i] = before(i, v[i][2]) ? m + 3 * q + 1 : m + 2 * q + 1;
        h[i] = before(i, v[i][2]) ? h[i] : m + 3 * q;
      } else {
        l[i] = before(i, v[i][0]) ? m + q + 1 : m;
        h[i] = before(i, v[i][0]) ? m + 2 * q : m + q;
      }
    }
  }
#pragma unroll
  for (int i = 0; i < 2; ++i) {  // at most three columns are left: their count before the limit
    int below = 0;
#pragma unroll
    for (int t = 0; t < 3; ++t) below += l[i] + t < h[i] && before(i, cols[l[i] + t]);
    (i == 0 ? *start : *end) = l[i] + below;
  }
}

// DIRECT: B has no more columns than a window has places, which then hold a
// value per column of the row's range instead of one per entry: a product needs
// no look-up of its rank (2000 rows of 280 entries times rows of 280 over 2000
// columns: 0.61 against 0.72 ms in fp32, 0.70 against 0.87 in fp64; the column
// slices before the windows 0.66 and 1.25).  Only where B's rows are longer than
// kNumShort on average: 10,000 rows of 40 entries times rows of 60 over 4000
// columns took 0.49 ms by column and 0.45 by rank in fp32 (more to clear, and the
// short parts are added atomically either way).
// PER: entries per thread and round.  Direct fp32 rounds are so short that B rows
// of more than 512 entries on average take 1024 at a time (2000 rows of 590
// entries times rows of 590 over 2000 columns 1.89 ms with two per thread, 1.62
// with four; fp64 2.27 and 2.11, but 5.00 and 5.10 with rows of 1000, and rows of
// 280 entries 0.61 and 0.75 in fp32).
template <typename T, bool DIRECT, int PER>
__global__ void __launch_bounds__(kNumThreads, 3) rcd_numeric_kernel(const RowPlan<T> p) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  using S = RcdNumeric<T>;
  S& s = *reinterpret_cast<S*>(smem_raw);
  constexpr int kWidth = S::kWidth;  // p.rcd_width is at most this
  constexpr int kNumPer = PER;       // entries per thread and round
  constexpr int kNumPiece = kNumThreads * kNumPer;
  constexpr int kWarps = kNumThreads / 32;
  __shared__ int s_scan[32];
  __shared__ int s_item, s_c0, s_c1;
  const int tid = static_cast<int>(threadIdx.x), lane = tid & 31, warp = tid >> 5;
  const int nbig = p.rcd_ctr[kRcdBigItems], nitems = nbig + p.rcd_ctr[kRcdItems];
  const long long cap = static_cast<long long>(p.seg_len) * p.rcd_slices;
  bool bad = false;
  for (int guard = 0; guard <= nitems; ++guard) {
    __syncthreads();  // the previous item is done with the shared state
    if (tid == 0) s_item = atomicAdd(&p.rcd_ctr[kRcdNextItem], 1);
    __syncthreads();
    const int it = s_item;
    if (it >= nitems) break;
    const long long item = it < nbig ? p.rcd_items[it] : p.rcd_items[cap - 1 - (it - nbig)];
    const int64_t r = item / p.rcd_slices;
    const int q0 = static_cast<int>(item % p.rcd_slices) * p.rcd_width;  // first rank of the window
    const int32_t row = p.perm[p.seg_begin + r];
    const int lo = p.lo[row];
    const int64_t cbase = p.c_rowptr[row] + q0;
    const long long want = p.c_rowptr[row + 1] - cbase;  // entries of the row from this window on
    // 1. the row's bitmap and the rank of every word
    uint32_t wv[kNumWords];
    int cnt = 0;
#pragma unroll
    for (int h = 0; h < kNumWords / 4; ++h) {
      const int i = tid * (kNumWords / 4) + h;  // 16-byte word
      uint4 v = make_uint4(0u, 0u, 0u, 0u);
      if (i * 4 < p.rcd_words) v = reinterpret_cast<const uint4*>(p.rcd_bits + r * p.rcd_words)[i];
      wv[4 * h] = v.x;
      wv[4 * h + 1] = v.y;
      wv[4 * h + 2] = v.z;
      wv[4 * h + 3] = v.w;
      cnt += __popc(v.x) + __popc(v.y) + __popc(v.z) + __popc(v.w);
    }
    int total;
    int run = block_exclusive_scan(cnt, s_scan, &total);
#pragma unroll
    for (int q = 0; q < kNumWords; ++q) {
      s.rk[tid * kNumWords + q] = make_uint2(wv[q], static_cast<uint32_t>(run - q0));
      run += __popc(wv[q]);
    }
    if (total - q0 != want) bad = true;
    const int in_win = min(p.rcd_width, total - q0);  // ranks in the window, at least 1
    const int n_out = static_cast<int>(max(0ll, min(static_cast<long long>(in_win), want)));
    __syncthreads();
    // 2. the window's columns, placed in the (still unused) window memory:
    // every thread takes as many consecutive ranks (an odd number, so the
    // lanes' stores fall into different banks) and walks the set bits from the
    // word that holds its first one.  With a thread or a warp per word the
    // densest words set the time (2.0 of 8.0 million cycles per CTA on R-MAT
    // 2^16 squared).
    int* cols = reinterpret_cast<int*>(s.win);
    const int per = ((in_win + kNumThreads - 1) / kNumThreads) | 1;
    const int t0 = tid * per, t1 = min(t0 + per, in_win);
    if (t0 < t1) {
      int w = 0, wh = kRcdWords - 1;  // the last word whose first rank is <= t0
      while (w < wh) {
        const int mid = (w + wh + 1) >> 1;
        if (static_cast<int>(s.rk[mid].y) <= t0) {
          w = mid;
        } else {
          wh = mid - 1;
        }
      }
      uint32_t m = s.rk[w].x;
      for (int skip = t0 - static_cast<int>(s.rk[w].y); skip > 0; --skip) m &= m - 1u;
      for (int at = t0; at < t1; ++at, m &= m - 1u) {
        while (m == 0u && w + 1 < kRcdWords) m = s.rk[++w].x;
        const int c = lo + (w << 5) + __ffs(m) - 1;
        cols[at] = c;
        if (at == 0) s_c0 = c;
        if (at == in_win - 1) s_c1 = c;
      }
    }
    __syncthreads();
#pragma unroll 4
    for (int i = tid; i < n_out; i += kNumThreads) p.c_colidx[cbase + i] = cols[i];
    __syncthreads();
    const int used = DIRECT ? min(p.hi[row] - lo + 1, kWidth) : in_win;
    for (int i = tid; i < (used * static_cast<int>(sizeof(T)) + 15) / 16; i += kNumThreads)
      reinterpret_cast<uint4*>(s.win)[i] = make_uint4(0u, 0u, 0u, 0u);
    const int c0 = s_c0, c1 = s_c1;
    const bool whole = DIRECT || total <= p.rcd_width;
    // Place of column c in the window; kWidth (and an error) if it has none,
    // which only an input changed since the symbolic pass can cause.
    auto rank_of = [&](int c) {
      const uint32_t off = static_cast<uint32_t>(c - lo);
      if constexpr (DIRECT) return off < static_cast<uint32_t>(kWidth) ? static_cast<int>(off) : kWidth;
      const uint2 rk = s.rk[(off >> 5) & (kRcdWords - 1)];
      const uint32_t at = rk.y + __popc(rk.x & ((1u << (off & 31u)) - 1u));
      return at < static_cast<uint32_t>(kWidth) ? static_cast<int>(at) : kWidth;
    };
    // One product, none if c < 0.  Only a warp with a product multiplies: an
    // fp64 multiplication of empty slots cost parts of 39 entries 8%.
    auto add = [&](int c, T a, T b) {
      if (c >= 0) {
        const int q = rank_of(c);
        if (q < kWidth) {
          atomicAdd(s.win + q, a * b);
        } else {
          bad = true;
        }
      }
    };
    const int64_t ra = p.A.rowptr[row], re = p.A.rowptr[row + 1];
    for (int64_t e0 = ra; e0 < re; e0 += kNumCacheA) {
      const int n = static_cast<int>(min(static_cast<int64_t>(kNumCacheA), re - e0));
      // 3. the part of every entry's B row inside the window's columns, and the
      // rounds of the long parts (with the number of shortest parts above them)
      constexpr int kTinyShift = 20;
      static_assert(static_cast<long long>(kNumCacheA) * kMaxBitmapSpan / kNumPiece < 1 << kTinyShift, "all rounds fit below");
      int rounds = 0;
      if (tid < n) {
        const int k = p.A.colidx[e0 + tid];
        s.a[tid] = p.A.vals[e0 + tid];
        const long long b0 = p.B.rowptr[k];
        int start = 0, end = static_cast<int>(p.B.rowptr[k + 1] - b0);
        if (!whole) part_bounds(p.B.colidx + b0, end, c0, c1, &start, &end);
        s.b0[tid] = b0 + start;
        s.len[tid] = end - start;
        rounds = end - start > kNumShort  ? (end - start + kNumPiece - 1) / kNumPiece
                 : end - start > kNumTiny ? 0
                                          : 1 << kTinyShift;
      }
      int nrounds;
      s.first[tid] = block_exclusive_scan(rounds, s_scan, &nrounds) & ((1 << kTinyShift) - 1);
      const int ntiny = nrounds >> kTinyShift;
      nrounds &= (1 << kTinyShift) - 1;
      __syncthreads();
      // 4a. long parts, round by round
      for (int p0 = 0; p0 < nrounds; p0 += kNumDesc) {
        const int np = min(kNumDesc, nrounds - p0);
        if (tid < np) {
          int jl = 0, jh = n - 1;  // the last entry whose first round is <= p0 + tid
          while (jl < jh) {
            const int mid = (jl + jh + 1) >> 1;
            if (s.first[mid] <= p0 + tid) {
              jl = mid;
            } else {
              jh = mid - 1;
            }
          }
          const int t0 = (p0 + tid - s.first[jl]) * kNumPiece;
          s.round[tid] = RcdRound{s.b0[jl] + t0, min(kNumPiece, s.len[jl] - t0), jl};
        }
        __syncthreads();
        // Round i sits in registers i % kAhead: its columns and values, and its
        // stored A entry.  The loads of shared memory a round needs (window,
        // A value, the next round's ranks, the descriptor of the round to load)
        // are issued together, ahead of the multiply-adds.
        int col[kAhead][kNumPer], ent[kAhead];
        T val[kAhead][kNumPer];
        int at[kNumPer];
        auto load = [&](const RcdRound& d, int u) {
          ent[u] = d.j;
          const int32_t* bc = p.B.colidx + d.b + tid;
          const T* bv = p.B.vals + d.b + tid;
#pragma unroll
          for (int h = 0; h < kNumPer; ++h) {
            col[u][h] = -1;
            if (tid + h * kNumThreads < d.n) {
              col[u][h] = bc[h * kNumThreads];
              val[u][h] = bv[h * kNumThreads];
            }
          }
        };
        const RcdRound none{0, 0, -1};
#pragma unroll
        for (int u = 0; u < kAhead; ++u) load(u < np ? s.round[u] : none, u);
#pragma unroll
        for (int h = 0; h < kNumPer; ++h) at[h] = col[0][h] >= 0 ? rank_of(col[0][h]) : -1;
        for (int i0 = 0; i0 < np; i0 += kAhead) {
#pragma unroll
          for (int u = 0; u < kAhead; ++u) {
            const int v = (u + 1) % kAhead;
            if (i0 + u < np) {
              const RcdRound d = i0 + u + kAhead < np ? s.round[i0 + u + kAhead] : none;
              const int j = ent[u];
              const T a = s.a[j];
              T w[kNumPer], x[kNumPer];
              int next[kNumPer];
#pragma unroll
              for (int h = 0; h < kNumPer; ++h) {
                w[h] = at[h] >= 0 && at[h] < kWidth ? s.win[at[h]] : T(0);
                x[h] = val[u][h];
              }
#pragma unroll
              for (int h = 0; h < kNumPer; ++h) next[h] = col[v][h] >= 0 ? rank_of(col[v][h]) : -1;
              load(d, u);
#pragma unroll
              for (int h = 0; h < kNumPer; ++h) {
                if (at[h] >= 0) {
                  if (at[h] < kWidth) {
                    s.win[at[h]] = fma(a, x[h], w[h]);
                  } else {
                    bad = true;
                  }
                }
                at[h] = next[h];
              }
              if (ent[v] != j) __syncthreads();  // the same in every thread
            }
          }
        }
        __syncthreads();
      }
      // 4b. the shortest parts
      constexpr int kTinyPer = kNumTiny / kNumTinyLanes;
      const int tl = lane % kNumTinyLanes;
#pragma unroll 2
      for (int j = tid / kNumTinyLanes; ntiny > 0 && j < n; j += kNumThreads / kNumTinyLanes) {
        const int len = s.len[j];
        if (len > kNumTiny) continue;
        const T a = s.a[j];
        const long long b0 = s.b0[j];
        int c[kTinyPer];
        T bv[kTinyPer];
#pragma unroll
        for (int u = 0; u < kTinyPer; ++u) {
          const int t = tl + u * kNumTinyLanes;
          c[u] = t < len ? p.B.colidx[b0 + t] : -1;
          bv[u] = t < len ? p.B.vals[b0 + t] : T(0);
        }
#pragma unroll
        for (int u = 0; u < kTinyPer; ++u) add(c[u], a, bv[u]);
      }
      // 4c. short parts
      constexpr int kPerLane = kNumShort / 32;
#pragma unroll 2
      for (int j = warp; j < n; j += kWarps) {
        const int len = s.len[j];
        if (len > kNumShort || len <= kNumTiny) continue;
        const T a = s.a[j];
        const long long b0 = s.b0[j];
        int c[kPerLane];
        T bv[kPerLane];
#pragma unroll
        for (int u = 0; u < kPerLane; ++u) {
          const int t = lane + u * 32;
          c[u] = t < len ? p.B.colidx[b0 + t] : -1;
          bv[u] = t < len ? p.B.vals[b0 + t] : T(0);
        }
#pragma unroll
        for (int u = 0; u < kPerLane; ++u) add(c[u], a, bv[u]);
      }
      __syncthreads();
    }
    // 5. the window's values
#pragma unroll 4
    for (int i = tid; i < n_out; i += kNumThreads) {
      const int q = DIRECT ? min(max(p.c_colidx[cbase + i] - lo, 0), kWidth - 1) : i;  // written above by this CTA
      p.c_vals[cbase + i] = s.win[q];
    }
  }
  if (bad) atomicOr(p.status, kErrCount);
}

// ----------------------------------------------------------------- wide rows

// Measured on R-MAT 2^20 (edge factor 8, fp64) times rows of 4 entries, 1,048
// such rows of 12,500 products on average and 93,000 at most: symbolic 86 us,
// numeric 186 us and 7 us for the zeroes.  A CTA per row that also set the bits
// again in the numeric pass, one thread writing the columns of 8 consecutive
// chunks, took 87 and 361 us, bound by its longest row.  Bound by the latency
// of a round's three dependent loads: with four instead of eight entries in
// flight the symbolic pass, which also stores 137 MB of bitmaps, takes 95 us.
// 20 rows of 8 entries times rows of 30,000 take 0.69 ms in all; with one load
// of each of eight B rows in flight at any length they took 1.28.

// Calls f(column, value of B, value of A) for the products of the stored A
// entries [ra, re).  A group of lanes takes BATCH entries per round, so
// their row-pointer loads and then their columns and values are in flight
// together (a hub row has tens of thousands of entries).
template <typename T, bool VALUES, int BATCH, typename F>
__device__ __forceinline__ void wb_products(const RowPlan<T>& p, int64_t ra, int64_t re, F&& f) {
  const int lg = p.log2_group;
  const int gsize = 1 << lg;
  const int grp = threadIdx.x >> lg;
  const int gl = threadIdx.x & (gsize - 1);
  const int ngrp = kWbThreads >> lg;
  for (int64_t pa0 = ra + grp; pa0 < re; pa0 += static_cast<int64_t>(BATCH) * ngrp) {
    int64_t qb[BATCH];
    int len[BATCH], most = 0;
    T av[BATCH];
#pragma unroll
    for (int u = 0; u < BATCH; ++u) {
      const int64_t pa = pa0 + static_cast<int64_t>(u) * ngrp;
      qb[u] = 0;
      len[u] = 0;
      av[u] = T(0);
      if (pa < re) {
        const int k = p.A.colidx[pa];
        if constexpr (VALUES) av[u] = p.A.vals[pa];
        qb[u] = p.B.rowptr[k];
        len[u] = static_cast<int>(p.B.rowptr[k + 1] - qb[u]);
      }
    }
#pragma unroll
    for (int u = 0; u < BATCH; ++u) most = max(most, len[u]);
    if (most > 4 * gsize) {  // long B rows: one at a time, kWbBatch steps in flight
#pragma unroll 1
      for (int u = 0; u < BATCH; ++u) {
        const int64_t pa = pa0 + static_cast<int64_t>(u) * ngrp;
        if (pa >= re) break;
        const int k = p.A.colidx[pa];
        const T a = VALUES ? p.A.vals[pa] : T(0);
        const int64_t b0 = p.B.rowptr[k];
        const int n = static_cast<int>(p.B.rowptr[k + 1] - b0);
        for (int t = gl; t < n; t += kWbBatch * gsize) {
          int c[kWbBatch];
          T bv[kWbBatch];
#pragma unroll
          for (int v = 0; v < kWbBatch; ++v) {
            const int i = t + v * gsize;
            c[v] = i < n ? p.B.colidx[b0 + i] : -1;
            bv[v] = VALUES && i < n ? p.B.vals[b0 + i] : T(0);
          }
#pragma unroll
          for (int v = 0; v < kWbBatch; ++v) {
            if (c[v] >= 0) f(c[v], bv[v], a);
          }
        }
      }
      continue;
    }
    for (int t = gl; t < most; t += gsize) {
      int c[BATCH];
      T bv[BATCH];
#pragma unroll
      for (int u = 0; u < BATCH; ++u) {
        c[u] = t < len[u] ? p.B.colidx[qb[u] + t] : -1;
        bv[u] = VALUES && t < len[u] ? p.B.vals[qb[u] + t] : T(0);
      }
#pragma unroll
      for (int u = 0; u < BATCH; ++u) {
        if (c[u] >= 0) f(c[u], bv[u], av[u]);
      }
    }
  }
}

template <typename T>
__global__ void __launch_bounds__(kWbThreads, 1) wb_symbolic_kernel(const RowPlan<T> p) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  uint32_t* bm = reinterpret_cast<uint32_t*>(smem_raw);  // kWbMaxSpan / 32 words
  uint4* bm4 = reinterpret_cast<uint4*>(smem_raw);
  __shared__ long long s_scan[32];
  constexpr int kShift = 24;
  static_assert(kWbMaxSpan < 1 << kShift, "a row's entries fit below its products");
  for (int i = threadIdx.x; i < kWbMaxSpan / 128; i += kWbThreads) bm4[i] = make_uint4(0u, 0u, 0u, 0u);
  __syncthreads();
  for (int64_t r = blockIdx.x; r < p.seg_len; r += gridDim.x) {
    const int32_t row = p.perm[p.seg_begin + r];
    const int lo = p.lo[row];
    const int nchunks = (p.hi[row] - lo + 128) >> 7;
    long long sums = 0;  // entries in the low bits, products above them
    wb_products<T, false, 2 * kWbBatch>(p, p.A.rowptr[row], p.A.rowptr[row + 1], [&](int c, T, T) {
      const uint32_t off = static_cast<uint32_t>(c - lo);
      const uint32_t bit = 1u << (off & 31u);
      sums += (1ll << kShift) + ((atomicOr(bm + (off >> 5), bit) & bit) == 0u);
    });
    __syncthreads();
    long long total;
    block_exclusive_scan(sums, s_scan, &total);
    if (threadIdx.x == 0) {
      p.c_rowptr[row + 1] = total & ((1ll << kShift) - 1);
      const long long products = total >> kShift;
      const long long most = min(static_cast<long long>(kWbMaxParts), static_cast<long long>(p.A.rowptr[row + 1] - p.A.rowptr[row]));
      const int parts = !p.wb_bits ? 1 : static_cast<int>(min((products + p.wb_part - 1) / p.wb_part, most));
      const int at = atomicAdd(&p.wb_ctr[parts > 1 ? kWbBigItems : kWbItems], parts);
      for (int q = 0; q < parts; ++q) {
        p.wb_items[parts > 1 ? at + q : p.wb_cap - 1 - at - q] = r << 32 | static_cast<long long>(q) << 16 | parts;
      }
    }
    uint4* bits = reinterpret_cast<uint4*>(p.wb_bits ? p.wb_bits + r * p.wb_words : nullptr);
    for (int i = threadIdx.x; i < nchunks; i += kWbThreads) {
      if (bits) bits[i] = bm4[i];
      bm4[i] = make_uint4(0u, 0u, 0u, 0u);
    }
    __syncthreads();
  }
}

// Zeroes the values of the rows that several items add to.
template <typename T>
__global__ void __launch_bounds__(256) wb_zero_kernel(const RowPlan<T> p) {
  const int nbig = p.wb_ctr[kWbBigItems];
  for (int it = blockIdx.x; it < nbig; it += gridDim.x) {
    const long long item = p.wb_items[it];
    const int32_t row = p.perm[p.seg_begin + (item >> 32)];
    const long long q = item >> 16 & 0xffff, parts = item & 0xffff;
    const int64_t c0 = p.c_rowptr[row], n = p.c_rowptr[row + 1] - c0;
    for (int64_t i = n * q / parts + threadIdx.x; i < n * (q + 1) / parts; i += 256) p.c_vals[c0 + i] = T(0);
  }
}

template <typename T>
__global__ void __launch_bounds__(kWbThreads, 1) wb_numeric_kernel(const RowPlan<T> p) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  uint32_t* bm = reinterpret_cast<uint32_t*>(smem_raw);          // kWbMaxSpan / 32 words
  uint4* bm4 = reinterpret_cast<uint4*>(smem_raw);
  uint32_t* pre = bm + kWbMaxSpan / 32;                           // one prefix per 128-bit chunk
  __shared__ long long s_scan[32];
  __shared__ int s_item;
  const int lane = static_cast<int>(threadIdx.x) & 31, warp = static_cast<int>(threadIdx.x) >> 5;
  const int nbig = p.wb_ctr[kWbBigItems], nitems = nbig + p.wb_ctr[kWbItems];
  bool bad = false;
  for (int guard = 0; guard <= nitems; ++guard) {
    __syncthreads();  // the previous item is done with the shared state
    if (threadIdx.x == 0) s_item = atomicAdd(&p.wb_ctr[kWbNextItem], 1);
    __syncthreads();
    const int it = s_item;
    if (it >= nitems) break;
    const long long item = it < nbig ? p.wb_items[it] : p.wb_items[p.wb_cap - 1 - (it - nbig)];
    const int64_t r = item >> 32, part = item >> 16 & 0xffff, parts = item & 0xffff;
    const int32_t row = p.perm[p.seg_begin + r];
    const int lo = p.lo[row];
    const int nchunks = (p.hi[row] - lo + 128) >> 7;
    const int64_t ra = p.A.rowptr[row], na = p.A.rowptr[row + 1] - ra;
    const int64_t cbase = p.c_rowptr[row], cend = p.c_rowptr[row + 1];
    if (parts == 1) {
      for (int64_t i = cbase + threadIdx.x; i < cend; i += kWbThreads) p.c_vals[i] = T(0);
    }
    // 1. the row's bitmap: from the plan, or made again
    const uint4* bits = reinterpret_cast<const uint4*>(p.wb_bits ? p.wb_bits + r * p.wb_words : nullptr);
#pragma unroll 4
    for (int i = threadIdx.x; i < nchunks; i += kWbThreads) bm4[i] = bits ? bits[i] : make_uint4(0u, 0u, 0u, 0u);
    __syncthreads();
    if (!bits) {
      wb_products<T, false, 2 * kWbBatch>(p, ra, ra + na, [&](int c, T, T) {
        uint32_t off;
        if (column_place(c, lo, nchunks << 7, &off)) {
          atomicOr(bm + (off >> 5), 1u << (off & 31u));
        } else {
          bad = true;
        }
      });
      __syncthreads();
    }
    // 2. the chunks' ranks.  A warp owns consecutive chunks, 32 at a time.
    const int per = (nchunks + kWbThreads - 1) / kWbThreads;
    const int first = warp * per * 32 + lane;
    int mine = 0;
    for (int j = 0; j < per; ++j) {
      const int i = first + j * 32;
      if (i < nchunks) {
        const uint4 v = bm4[i];
        mine += __popc(v.x) + __popc(v.y) + __popc(v.z) + __popc(v.w);
      }
    }
    long long total;
    long long run = block_exclusive_scan(static_cast<long long>(mine), s_scan, &total);
    run = __shfl_sync(0xffffffffu, run, 0);  // entries before the warp's chunks
    bad |= total != cend - cbase;
    // The part's share of the columns is written on the way.
    const int e0 = static_cast<int>(nchunks * part / parts), e1 = static_cast<int>(nchunks * (part + 1) / parts);
    for (int j = 0; j < per; ++j) {
      const int i = first + j * 32;
      const uint4 v = i < nchunks ? bm4[i] : make_uint4(0u, 0u, 0u, 0u);
      const int n = __popc(v.x) + __popc(v.y) + __popc(v.z) + __popc(v.w);
      int upto = n;
#pragma unroll
      for (int d = 1; d < 32; d <<= 1) {
        const int x = __shfl_up_sync(0xffffffffu, upto, d);
        if (lane >= d) upto += x;
      }
      int64_t pos = cbase + run + upto - n;
      if (i < nchunks) pre[i] = static_cast<uint32_t>(pos - cbase);
      if (i >= e0 && i < e1) {
        const uint32_t wv[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          for (uint32_t x = wv[q]; x; x &= x - 1u, ++pos) {
            if (pos < cend) p.c_colidx[pos] = lo + (i << 7) + (q << 5) + __ffs(x) - 1;
          }
        }
      }
      run += __shfl_sync(0xffffffffu, upto, 31);
    }
    __syncthreads();  // prefixes and the zeroed values are visible to the CTA
    // 3. the part's products
    wb_products<T, true, kWbBatch>(p, ra + na * part / parts, ra + na * (part + 1) / parts, [&](int c, T b, T a) {
      uint32_t off;
      if (!column_place(c, lo, nchunks << 7, &off)) {
        bad = true;
        return;
      }
      const uint32_t i = off >> 7;
      const uint4 v = bm4[i];
      const uint32_t wq = (off >> 5) & 3u;
      const uint32_t wd = wq == 0 ? v.x : wq == 1 ? v.y : wq == 2 ? v.z : v.w;
      const int64_t pos = cbase + pre[i] + (wq > 0 ? __popc(v.x) : 0) + (wq > 1 ? __popc(v.y) : 0) +
                          (wq > 2 ? __popc(v.z) : 0) + __popc(wd & ((1u << (off & 31u)) - 1u));
      if (pos < cend) {
        atomicAdd(p.c_vals + pos, a * b);
      } else {
        bad = true;
      }
    });
  }
  if (bad) atomicOr(p.status, kErrCount);
}

template <typename K>
int occupancy(K kern, int threads, size_t smem) {
  cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(smem));
  int n = 0;
  cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, kern, threads, smem);
  return n > 0 ? n : 1;
}

int grid_of(int64_t rows, int num_sms, int per_sm) {
  int64_t g = rows;
  const int64_t cap = static_cast<int64_t>(num_sms) * per_sm;
  if (g > cap) g = cap;
  if (g < 1) g = 1;
  return static_cast<int>(g);
}

}  // namespace

template <typename T>
void launch_rcd(const RowPlan<T>& p, bool numeric, int num_sms, cudaStream_t s, int* launches) {
  if (!numeric) {
    const size_t smem = sizeof(RcdSymbolic);
    auto kern = p.rcd_again ? rcd_symbolic_kernel<T, true> : rcd_symbolic_kernel<T, false>;
    static int per_sm[2] = {0, 0};
    if (per_sm[p.rcd_again] == 0) per_sm[p.rcd_again] = occupancy(kern, kRcdThreads, smem);
    kern<<<grid_of(p.seg_len, num_sms, per_sm[p.rcd_again]), kRcdThreads, smem, s>>>(p);
  } else {
    const size_t smem = sizeof(RcdNumeric<T>);
    static int per_sm[3] = {0, 0, 0};
    const int v = !p.rcd_direct ? 0 : sizeof(T) == 4 && p.rcd_long_b ? 2 : 1;
    auto kern = v == 0 ? rcd_numeric_kernel<T, false, 2> : rcd_numeric_kernel<T, true, 2>;
    if constexpr (sizeof(T) == 4) {
      if (v == 2) kern = rcd_numeric_kernel<T, true, 4>;
    }
    if (per_sm[v] == 0) per_sm[v] = occupancy(kern, kNumThreads, smem);
    kern<<<grid_of(p.seg_len * p.rcd_slices, num_sms, per_sm[v]), kNumThreads, smem, s>>>(p);
  }
  *launches += 1;
}

template <typename T>
void launch_wb(const RowPlan<T>& p, bool numeric, int num_sms, cudaStream_t s, int* launches) {
  if (!numeric) {
    const size_t smem = kWbMaxSpan / 8;
    static int per_sm = 0;
    if (per_sm == 0) per_sm = occupancy(wb_symbolic_kernel<T>, kWbThreads, smem);
    wb_symbolic_kernel<T><<<grid_of(p.seg_len, num_sms, per_sm), kWbThreads, smem, s>>>(p);
    *launches += 1;
  } else {
    const size_t smem = kWbMaxSpan / 8 + (kWbMaxSpan / 128) * 4;
    static int per_sm = 0;
    if (per_sm == 0) per_sm = occupancy(wb_numeric_kernel<T>, kWbThreads, smem);
    if (p.wb_bits) {
      wb_zero_kernel<T><<<grid_of(p.wb_cap, num_sms, 8), 256, 0, s>>>(p);
      *launches += 1;
    }
    wb_numeric_kernel<T><<<grid_of(p.wb_cap, num_sms, per_sm), kWbThreads, smem, s>>>(p);
    *launches += 1;
  }
}

template void launch_rcd<float>(const RowPlan<float>&, bool, int, cudaStream_t, int*);
template void launch_rcd<double>(const RowPlan<double>&, bool, int, cudaStream_t, int*);
template void launch_wb<float>(const RowPlan<float>&, bool, int, cudaStream_t, int*);
template void launch_wb<double>(const RowPlan<double>&, bool, int, cudaStream_t, int*);

}  // namespace wsk
