// Row analysis and binning (first step of the symbolic pass), plus CSR validation.
//
// For every row i of C = A*B:
//   nnzA_i = A.rowptr[i+1] - A.rowptr[i]
//   ub_i   = sum over stored A[i,k] of (B.rowptr[k+1] - B.rowptr[k])   (products of the row)
//   lo_i   = min over those k of the first column of B[k,:]
//   hi_i   = max over those k of the last column of B[k,:]
// (B's rows are sorted, so every product of the row lands in [lo_i, hi_i].)
// The row's class follows from (nnzA_i, ub_i); the counts per class go to
// DevSummary so the host can size the per-class launches.  The work per row
// is not known before this pass (Sec. 1, irregular compute balance); the
// binning replaces the static/dynamic loop schedules of Sec. 4 with a
// partition of rows by their work.
#include <climits>

#include "ws_internal.cuh"

namespace wsk {

namespace {

__device__ __forceinline__ int ceil_log2_ll(long long x) {  // x >= 1
  return x <= 1 ? 0 : 64 - __clzll(x - 1);
}

// Class of a row from its stored-entry count, product count, column range and
// the shape of its B rows.
// Regular rows (at most kBmrMaxA entries whose B rows fit one lane group) with
// a range that fits a bitmap not much larger than their products (at most 8
// words per product plus 64) take the register bitmap bins (the bitmap bins
// if those are disabled).  The other rows of at most hash_max products take the
// hash bins unless
// - their products crowd a range of less than kCrowded columns per product:
//   most products repeat a column there, and the hash buckets fill up;
// - one of their B rows is longer than kShortB: such rows (hub rows of a
//   power-law matrix) tend to be dense at one end, which fills some buckets;
// - the row has more than 16 entries and its B rows have lumps (three of four
//   of those of more than three columns among the first kLooks, at least
//   kLeastLooks): runs of neighbouring columns, as of a box stencil or of blocks,
//   fill a bucket each (with one look as the least, 26 of 128,000 rows of
//   scattered columns went to bins of their own, whose launches cost 20 us); or
// - a bitmap is cheaper although the columns spread: above kLargeHash products
//   of B rows of kLongB columns and more (the windows of the dense rows), and in
//   the bin of kSmallTo products and 16,384 columns when the B rows are of about the
//   same length, of kSmallB columns and more, so that the lane groups are full
//   (that hash bin holds as much as twice the products for the same time; a few
//   rows of 150 entries and B rows of 2 took 10 us more in a bitmap).
// Those take the bitmap bins, and the dense rows above them.  Measured (24
// million products, fp32, bitmap or dense rows against hash bins, ms): rows of
// 0-40 entries and B rows of 0-20 over 16,000 columns 0.86 against 0.59; 40 of 20
// 0.81 against 0.57, 24 of 12 0.48 against 0.63, 42 of 12 0.47 against 0.53 (over
// 32,000 columns 24 of 12 0.68 against 0.60); 60 of 60 over 16,000 0.41 against
// 0.57, 150 of 16 0.49 against 0.65, 300 of 10 0.67 against 0.65; 60 of 60 over 250
// 0.32 against 1.26.  27-point stencil of 64^3 squared 3.9 against 16.4, 9-point
// stencil of 3 x 3 blocks on 128^2 0.91 against 3.4.  R-MAT 2^16 squared with and
// without the second exception 3.5 and 4.3.
// Rows with more products go to the dense rows (range up to 65,536 columns), the
// 8192-entry bitmap bin, the wide bitmap (range up to 2^20) and finally the
// column-sliced dense window.
constexpr long long kCrowded = 2;
constexpr int kShortB = 64;
constexpr int kLooks = 8, kLeastLooks = 5;
constexpr long long kLargeHash = 2048, kLongB = 16;
constexpr long long kSmallB = 8, kSmallFrom = bitmap_cap(0), kSmallTo = bitmap_cap(1), kSmallSpan = 32ll << bitmap_log_words(1);
constexpr int kBatch = 4;  // stored A entries of a long row that a thread has in flight

// What a row's class depends on, gathered over its stored A entries.
struct RowShape {
  long long ub = 0;  // products
  int lo = INT_MAX, hi = -1, maxlen = 0;
  int looked = 0, lumps = 0;  // B rows whose columns were looked at, and those of them with lumps

  // B row [bs, be).
  __device__ __forceinline__ void add(const int32_t* colidx, int64_t bs, int64_t be) {
    if (be > bs) {
      ub += be - bs;
      maxlen = max(maxlen, static_cast<int>(min(be - bs, static_cast<int64_t>(INT_MAX))));
      lo = min(lo, colidx[bs]);
      hi = max(hi, colidx[be - 1]);
    }
  }
  // The B rows of the stored A entries q0, q0 + step, ... before e, BATCH at a
  // time, so that each of the three dependent loads is in flight for all of
  // them.  A B row of an entry before look_end has lumps if its first three
  // columns lie within a quarter of its average distance between two columns
  // (one of 38 rows of columns drawn at random does).
  template <typename T, int BATCH>
  __device__ __forceinline__ void gather(const RowPlan<T>& p, int64_t q0, int64_t e, int step, int64_t look_end) {
    for (; q0 < e; q0 += static_cast<int64_t>(BATCH) * step) {
      int64_t bs[BATCH], be[BATCH];
      int k[BATCH], first[BATCH], last[BATCH], third = 0;
#pragma unroll
      for (int u = 0; u < BATCH; ++u) {
        const int64_t q = q0 + static_cast<int64_t>(u) * step;
        k[u] = q < e ? p.A.colidx[q] : -1;
      }
#pragma unroll
      for (int u = 0; u < BATCH; ++u) {
        bs[u] = k[u] >= 0 ? p.B.rowptr[k[u]] : 0;
        be[u] = k[u] >= 0 ? p.B.rowptr[k[u] + 1] : 0;
      }
      const bool look = q0 < look_end && be[0] - bs[0] > 3;
#pragma unroll
      for (int u = 0; u < BATCH; ++u) {
        first[u] = be[u] > bs[u] ? p.B.colidx[bs[u]] : INT_MAX;
        last[u] = be[u] > bs[u] ? p.B.colidx[be[u] - 1] : -1;
      }
      if (look) third = p.B.colidx[bs[0] + 2];
#pragma unroll
      for (int u = 0; u < BATCH; ++u) {
        const int64_t n = be[u] - bs[u];
        ub += n;
        maxlen = max(maxlen, static_cast<int>(min(n, static_cast<int64_t>(INT_MAX))));
        lo = min(lo, first[u]);
        hi = max(hi, last[u]);
      }
      looked += look;
      lumps += look && 4 * (static_cast<int64_t>(third) - first[0]) * (be[0] - bs[0] - 1) <= static_cast<int64_t>(last[0]) - first[0];
    }
  }
  __device__ __forceinline__ bool lumpy() const { return looked >= kLeastLooks && 4 * lumps >= 3 * looked; }

  __device__ __forceinline__ void merge(const RowShape& o) {
    ub += o.ub;
    lo = min(lo, o.lo);
    hi = max(hi, o.hi);
    maxlen = max(maxlen, o.maxlen);
    looked += o.looked;
    lumps += o.lumps;
  }
  // Over the lanes of a warp.
  __device__ __forceinline__ void warp_merge() {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) ub += __shfl_xor_sync(0xffffffffu, ub, o);
    lo = __reduce_min_sync(0xffffffffu, lo);
    hi = __reduce_max_sync(0xffffffffu, hi);
    maxlen = __reduce_max_sync(0xffffffffu, maxlen);
    const int both = __reduce_add_sync(0xffffffffu, looked << 16 | lumps);
    looked = both >> 16;
    lumps = both & 0xffff;
  }
};

__device__ __forceinline__ uint8_t classify(long long nnza, const RowShape& r, const AnalyzeParams& ap) {
  const long long ub = r.ub;
  const int lo = r.lo, hi = r.hi, maxlen = r.maxlen;
  if (ub == 0) return kClsEmpty;
  if (nnza == 1) return kClsDirect;
  const long long span = static_cast<long long>(hi) - lo + 1;
  const long long est = ub < span ? ub : span;  // entries of the row are at most this
  const bool bitmap_ok = span <= ap.bitmap_span && ((span + 31) >> 5) <= 8 * ub + 64;
  const bool regular = nnza <= kBmrMaxA && maxlen <= ap.group;
  const bool spread = span >= kCrowded * ub && maxlen <= kShortB && !r.lumpy();
  const bool bitmap_cheaper = (ub > kLargeHash && ub >= kLongB * nnza) ||
                              (ub > kSmallFrom && ub <= kSmallTo && span <= kSmallSpan && ub >= kSmallB * nnza &&
                               4 * ub >= 3 * nnza * maxlen);
  const bool hashed = ub <= ap.hash_max && (!bitmap_ok || (!regular && spread && !bitmap_cheaper));
  if (bitmap_ok && !hashed) {
    if (regular && nnza <= ap.bmr_max_a) {
#pragma unroll
      for (int b = 0; b < kNumBmrBins; ++b) {
        if (span <= (32ll << bmr_log_words(b))) return static_cast<uint8_t>(kClsBmr0 + b);
      }
    }
#pragma unroll
    for (int b = 0; b < kNumBitmapBins - 1; ++b) {
      if (span <= (32ll << bitmap_log_words(b)) && est <= bitmap_cap(b)) return static_cast<uint8_t>(kClsBitmap0 + b);
    }
  }
  const bool heavy = !hashed && (ub > 4096 || (bitmap_ok && est > bitmap_cap(kNumBitmapBins - 2)));
  if (heavy && span <= kMaxBitmapSpan && nnza <= ap.rcd_max_a) return kClsRcd;
  if (bitmap_ok && !hashed && span <= (32ll << bitmap_log_words(kNumBitmapBins - 1)) && est <= bitmap_cap(kNumBitmapBins - 1))
    return static_cast<uint8_t>(kClsBitmap0 + kNumBitmapBins - 1);
  if (ub <= ap.hash_max) {
    int b = ceil_log2_ll(ub) - kMinHashLog;
    b = b < 0 ? 0 : b;
    return static_cast<uint8_t>(kClsHash0 + b);
  }
  if (span <= ap.wb_span) return kClsWb;
  return kClsDense;
}

__device__ __forceinline__ int segment_of(uint8_t cls) {
  if (cls == kClsDirect) return kSegDirect;
  if (cls == kClsDense) return kSegDense;
  if (cls == kClsBmrWide) return kSegBmrWide;
  if (cls == kClsRcd) return kSegRcd;
  if (cls == kClsWb) return kSegWb;
  if (cls < kClsBitmap0) return kSegBmr0 + (cls - kClsBmr0);      // register bitmap bins
  if (cls < kClsHash0) return kSegBitmap0 + (cls - kClsBitmap0);  // bitmap bins
  return kSegHash0 + (cls - kClsHash0);                            // hash bins
}

// Stores the class and column range of row i (and its count if it is known
// already) and returns the class.
template <typename T>
__device__ __forceinline__ uint8_t store_row(const RowPlan<T>& p, const AnalyzeParams& ap, int64_t i, long long nnza,
                                             const RowShape& r, long long* s_slices, long long* s_wb) {
  const uint8_t c = classify(nnza, r, ap);
  p.cls[i] = c;
  // Direct rows know their count already; the others start at 0 and are
  // filled by the hash / dense-window symbolic kernels.
  p.c_rowptr[i + 1] = (c == kClsDirect) ? r.ub : 0;
  if (c != kClsEmpty) {
    p.lo[i] = r.lo;
    p.hi[i] = r.hi;
    if (c == kClsDense) {
      const long long span = static_cast<long long>(r.hi) - r.lo + 1;
      atomicAdd(reinterpret_cast<unsigned long long*>(s_slices),
                static_cast<unsigned long long>((span + ap.dense_width - 1) / ap.dense_width));
    }
    if (c == kClsWb) atomicAdd(reinterpret_cast<unsigned long long*>(s_wb), static_cast<unsigned long long>(r.ub));
  }
  return c;
}

// store_row for one row analysed by a single thread, with its counts added
// to the CTA's counters.
template <typename T>
__device__ __forceinline__ void record_row(const RowPlan<T>& p, const AnalyzeParams& ap, int64_t i, long long nnza,
                                           const RowShape& r, int* s_seg, long long* s_prod, long long* s_slices,
                                           long long* s_wb, int* s_empty) {
  const uint8_t c = store_row(p, ap, i, nnza, r, s_slices, s_wb);
  if (c == kClsEmpty) {
    atomicAdd(s_empty, 1);
  } else {
    atomicAdd(&s_seg[segment_of(c)], 1);
  }
  atomicAdd(reinterpret_cast<unsigned long long*>(s_prod), static_cast<unsigned long long>(r.ub));
}

template <typename T>
__device__ __forceinline__ void flush_counts(const RowPlan<T>& p, int* s_seg, long long* s_prod,
                                             long long* s_slices, long long* s_wb, int* s_empty) {
  if (threadIdx.x < kNumSegs && s_seg[threadIdx.x]) atomicAdd(&p.sum->seg_count[threadIdx.x], s_seg[threadIdx.x]);
  if (threadIdx.x == 0) {
    if (*s_prod) atomicAdd(reinterpret_cast<unsigned long long*>(&p.sum->products),
                           static_cast<unsigned long long>(*s_prod));
    if (*s_slices) atomicAdd(reinterpret_cast<unsigned long long*>(&p.sum->dense_slices),
                             static_cast<unsigned long long>(*s_slices));
    if (*s_wb) atomicAdd(reinterpret_cast<unsigned long long*>(&p.sum->wb_products), static_cast<unsigned long long>(*s_wb));
    if (*s_empty) atomicAdd(&p.sum->n_empty, *s_empty);
  }
}

// Longest row a warp analyses; longer rows take a whole CTA.
constexpr int64_t kMidRowMax = 2048;

// One thread per row for rows with at most long_threshold stored entries;
// longer rows are queued in long_rows for analyze_long_kernel: rows up to
// kMidRowMax entries from the front (a warp per row), the others from the back
// (a CTA per row).
template <typename T>
__global__ void __launch_bounds__(256) analyze_kernel(const RowPlan<T> p, const AnalyzeParams ap,
                                                      int32_t* long_rows, const int32_t* rows) {
  __shared__ int s_seg[kNumSegs];
  __shared__ long long s_prod, s_slices, s_wb;
  __shared__ int s_empty;
  if (threadIdx.x < kNumSegs) s_seg[threadIdx.x] = 0;
  if (threadIdx.x == 0) {
    s_prod = 0;
    s_slices = 0;
    s_wb = 0;
    s_empty = 0;
  }
  __syncthreads();
  const int64_t nrows = rows ? static_cast<int64_t>(*reinterpret_cast<volatile int*>(&p.sum->n_pending)) : ap.m;
  // Whole warps walk the rows (lane l takes row t0 + l), so that the counts
  // per class can be added once per warp and class: every row adding to the
  // same few CTA counters serialised on the shared-memory atomics.
  const int lane = threadIdx.x & 31;
  unsigned long long prod = 0;
  for (int64_t t0 = static_cast<int64_t>(blockIdx.x) * blockDim.x + (threadIdx.x & ~31); t0 < nrows;
       t0 += static_cast<int64_t>(gridDim.x) * blockDim.x) {
    const int64_t t = t0 + lane;
    int seg = -2;  // no row, or a long row (queued)
    if (t < nrows) {
      const int64_t i = rows ? rows[t] : t;
      const int64_t s = p.A.rowptr[i], e = p.A.rowptr[i + 1];
      if (e - s > ap.long_threshold) {
        if (e - s <= kMidRowMax) {
          long_rows[atomicAdd(&p.sum->n_mid, 1)] = static_cast<int32_t>(i);
        } else {
          long_rows[ap.m - 1 - atomicAdd(&p.sum->n_long, 1)] = static_cast<int32_t>(i);
        }
      } else {
        RowShape r;
#pragma unroll 4
        for (int64_t q = s; q < e; ++q) {
          const int k = p.A.colidx[q];
          r.add(p.B.colidx, p.B.rowptr[k], p.B.rowptr[k + 1]);
        }
        const uint8_t c = store_row(p, ap, i, e - s, r, &s_slices, &s_wb);
        seg = c == kClsEmpty ? -1 : segment_of(c);
        prod += static_cast<unsigned long long>(r.ub);
      }
    }
    const unsigned peers = __match_any_sync(0xffffffffu, seg);
    if (seg >= -1 && lane == __ffs(peers) - 1) {
      if (seg < 0) {
        atomicAdd(&s_empty, __popc(peers));
      } else {
        atomicAdd(&s_seg[seg], __popc(peers));
      }
    }
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) prod += __shfl_xor_sync(0xffffffffu, prod, o);
  if (lane == 0 && prod) atomicAdd(reinterpret_cast<unsigned long long*>(&s_prod), prod);
  __syncthreads();
  flush_counts(p, s_seg, &s_prod, &s_slices, &s_wb, &s_empty);
}

// Rows queued by analyze_kernel.  First one CTA per long row (a power-law
// row can hold tens of thousands of entries, and its three dependent loads
// per entry are a latency chain), then one warp per row of long_threshold + 1
// .. kMidRowMax entries (the lanes stride over the entries, kBatch in flight
// each, and warp reductions give the row's shape).  For a long row the threads
// stride over the row's stored entries, kBatch in flight each, and the CTA
// reduces its shape.  Five CTAs per SM with four entries in flight: 57 registers
// (four CTAs) cost rows of 17-24 entries 1%; an unrolled loop over conditional loads
// took 15 us more on R-MAT 2^20 than these batches.
template <typename T>
__global__ void __launch_bounds__(256, 5) analyze_long_kernel(const RowPlan<T> p, const AnalyzeParams ap,
                                                           const int32_t* long_rows, DevSummary* host) {
  const int nlong = *reinterpret_cast<volatile int*>(&p.sum->n_long);
  const int nmid = *reinterpret_cast<volatile int*>(&p.sum->n_mid);
  if (nlong == 0 && nmid == 0) {  // no long rows: nothing changes the summary any more
    if (host && blockIdx.x == 0) publish_summary(p.sum, host, false);
    return;
  }
  __shared__ int s_last;
  __shared__ int s_seg[kNumSegs];
  __shared__ long long s_prod, s_slices, s_wb;
  __shared__ int s_empty;
  __shared__ RowShape s_shape[8];
  if (threadIdx.x < kNumSegs) s_seg[threadIdx.x] = 0;
  if (threadIdx.x == 0) {
    s_prod = 0;
    s_slices = 0;
    s_wb = 0;
    s_empty = 0;
  }
  __syncthreads();
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  for (int64_t w = blockIdx.x; w < nlong; w += gridDim.x) {
    const int64_t i = long_rows[ap.m - 1 - w];  // long rows fill the list from the back
    const int64_t s = p.A.rowptr[i], e = p.A.rowptr[i + 1];
    RowShape r;
    r.gather<T, kBatch>(p, s + threadIdx.x, e, blockDim.x, s + kLooks);
    r.warp_merge();
    if (lane == 0) s_shape[warp] = r;
    __syncthreads();
    if (threadIdx.x == 0) {
      for (int w2 = 1; w2 < static_cast<int>(blockDim.x >> 5); ++w2) r.merge(s_shape[w2]);
      record_row(p, ap, i, e - s, r, s_seg, &s_prod, &s_slices, &s_wb, &s_empty);
    }
    __syncthreads();  // s_shape is reused by the next row
  }
  const int64_t gw = (static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x) >> 5;
  const int64_t nw = (static_cast<int64_t>(gridDim.x) * blockDim.x) >> 5;
  for (int64_t w = gw; w < nmid; w += nw) {
    const int64_t i = long_rows[w];
    const int64_t s = p.A.rowptr[i], e = p.A.rowptr[i + 1];
    RowShape r;
    if (e - s <= 32) {
      r.gather<T, 1>(p, s + lane, e, 32, s + kLooks);
    } else {
      r.gather<T, kBatch>(p, s + lane, e, 32, s + kLooks);
    }
    r.warp_merge();
    if (lane == 0) record_row(p, ap, i, e - s, r, s_seg, &s_prod, &s_slices, &s_wb, &s_empty);
  }
  __syncthreads();
  flush_counts(p, s_seg, &s_prod, &s_slices, &s_wb, &s_empty);
  if (host) {  // the last CTA to get here copies the summary for the host
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) s_last = atomicAdd(&p.sum->n_done, 1) == static_cast<int>(gridDim.x) - 1;
    __syncthreads();
    if (s_last) {
      __threadfence();
      publish_summary(p.sum, host, false);
    }
  }
}

struct SegOffsets {
  long long off[kNumSegs];
};

// Groups non-empty rows by segment: perm[seg_offset[s] .. + seg_count[s]).
// Rows of one block keep their relative order inside each segment.
template <typename T>
__global__ void __launch_bounds__(256) scatter_kernel(const RowPlan<T> p, int64_t m, const SegOffsets so) {
  __shared__ int s_cnt[kNumSegs];
  __shared__ int s_base[kNumSegs];
  for (int64_t tile = static_cast<int64_t>(blockIdx.x) * blockDim.x; tile < m;
       tile += static_cast<int64_t>(gridDim.x) * blockDim.x) {
    if (threadIdx.x < kNumSegs) s_cnt[threadIdx.x] = 0;
    __syncthreads();
    const int64_t i = tile + threadIdx.x;
    int seg = -1, rank = 0;
    if (i < m) {
      const uint8_t c = p.cls[i];
      if (c != kClsEmpty) {
        seg = segment_of(c);
        rank = atomicAdd(&s_cnt[seg], 1);
      }
    }
    __syncthreads();
    if (threadIdx.x < kNumSegs && s_cnt[threadIdx.x])
      s_base[threadIdx.x] = atomicAdd(&p.sum->seg_cursor[threadIdx.x], s_cnt[threadIdx.x]);
    __syncthreads();
    if (seg >= 0) p.perm[so.off[seg] + s_base[seg] + rank] = static_cast<int32_t>(i);
    __syncthreads();
  }
}

// Expands every dense-window row into its column slices.
template <typename T>
__global__ void __launch_bounds__(256) dense_slices_kernel(const RowPlan<T> p, int32_t* slice_row,
                                                           int32_t* slice_idx, int32_t* slice_first) {
  for (int64_t r = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x; r < p.seg_len;
       r += static_cast<int64_t>(gridDim.x) * blockDim.x) {
    const int32_t row = p.perm[p.seg_begin + r];
    const long long span = static_cast<long long>(p.hi[row]) - p.lo[row] + 1;
    const long long ns = (span + p.dense_width - 1) / p.dense_width;
    const long long first =
        static_cast<long long>(atomicAdd(reinterpret_cast<unsigned long long*>(&p.sum->slice_cursor),
                                         static_cast<unsigned long long>(ns)));
    for (long long s = 0; s < ns; ++s) {
      slice_row[first + s] = row;
      slice_idx[first + s] = static_cast<int32_t>(s);
      slice_first[first + s] = static_cast<int32_t>(first);
    }
  }
}

// Checks the CSR invariants of one matrix; records the smallest offending row
// in `sum` (pinned host memory, written only for a broken matrix).
__global__ void __launch_bounds__(256) validate_kernel(const int64_t* rowptr, const int32_t* colidx, int64_t nrows,
                                                       int64_t ncols, int64_t nnz, DevSummary* sum) {
  int worst = INT_MAX;  // first bad row this thread saw
  for (int64_t i = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x; i < nrows;
       i += static_cast<int64_t>(gridDim.x) * blockDim.x) {
    const int64_t s = rowptr[i], e = rowptr[i + 1];
    bool bad = s < 0 || e < s || e > nnz || (i == 0 && s != 0) || (i == nrows - 1 && e != nnz);
    if (!bad) {
      int prev = -1;
      for (int64_t q = s; q < e; ++q) {
        const int c = colidx[q];
        if (c <= prev || c >= ncols) {
          bad = true;
          break;
        }
        prev = c;
      }
    }
    if (bad) worst = min(worst, static_cast<int>(i < INT_MAX ? i : INT_MAX - 1));
  }
  worst = __reduce_min_sync(0xffffffffu, worst);
  if ((threadIdx.x & 31) == 0 && worst < INT_MAX) {
    atomicOr(&sum->status, kErrInvalidCsr);
    atomicMin(&sum->bad_row, worst);
  }
}

int grid_for(int64_t work, int per_block, int num_sms, int blocks_per_sm) {
  int64_t g = (work + per_block - 1) / per_block;
  const int64_t cap = static_cast<int64_t>(num_sms) * blocks_per_sm;
  if (g > cap) g = cap;
  if (g < 1) g = 1;
  return static_cast<int>(g);
}

}  // namespace

template <typename T>
void launch_analyze(const RowPlan<T>& p, const AnalyzeParams& ap, int32_t* long_rows, const int32_t* rows,
                    DevSummary* host, int num_sms, cudaStream_t s, int* launches) {
  analyze_kernel<T><<<grid_for(ap.m, 256, num_sms, 8), 256, 0, s>>>(p, ap, long_rows, rows);
  // a warp per long row: A's entries bound their number (a full grid of CTAs
  // without work takes 7 us)
  analyze_long_kernel<T><<<grid_for(ap.nnz / (ap.long_threshold + 1), 8, num_sms, 8), 256, 0, s>>>(p, ap, long_rows, host);
  *launches += 2;
}

template <typename T>
void launch_scatter(const RowPlan<T>& p, int64_t m, const int64_t* seg_offset, int num_sms, cudaStream_t s,
                    int* launches) {
  SegOffsets so;
  for (int i = 0; i < kNumSegs; ++i) so.off[i] = seg_offset[i];
  scatter_kernel<T><<<grid_for(m, 256, num_sms, 8), 256, 0, s>>>(p, m, so);
  *launches += 1;
}

template <typename T>
void launch_dense_slices(const RowPlan<T>& p, int32_t* slice_row, int32_t* slice_idx, int32_t* slice_first,
                         int num_sms, cudaStream_t s, int* launches) {
  dense_slices_kernel<T><<<grid_for(p.seg_len, 256, num_sms, 4), 256, 0, s>>>(p, slice_row, slice_idx,
                                                                              slice_first);
  *launches += 1;
}

void launch_validate(const int64_t* rowptr, const int32_t* colidx, int64_t nrows, int64_t ncols, int64_t nnz,
                     DevSummary* sum, int num_sms, cudaStream_t s) {
  validate_kernel<<<grid_for(nrows, 256, num_sms, 8), 256, 0, s>>>(rowptr, colidx, nrows, ncols, nnz, sum);
}

#define WS_INST(T)                                                                                          \
  template void launch_analyze<T>(const RowPlan<T>&, const AnalyzeParams&, int32_t*, const int32_t*,           \
                                  DevSummary*, int, cudaStream_t, int*);                                                       \
  template void launch_scatter<T>(const RowPlan<T>&, int64_t, const int64_t*, int, cudaStream_t, int*);      \
  template void launch_dense_slices<T>(const RowPlan<T>&, int32_t*, int32_t*, int32_t*, int, cudaStream_t, int*);
WS_INST(float)
WS_INST(double)
#undef WS_INST

}  // namespace wsk
