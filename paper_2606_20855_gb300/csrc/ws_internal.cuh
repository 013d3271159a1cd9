// Internal declarations shared by the CUDA translation units of the SpGEMM library.
//
// Row classes.  The symbolic pass sorts every output row i of C = A*B into one
// class by its product count ub_i = sum over stored A[i,k] of |B[k,:]| (the
// work of the row, which is data dependent and unknown before the pass --
// the load-balance problem of Sec. 1):
//   empty         ub_i = 0                       -> no output
//   direct        exactly one stored A[i,k]      -> C[i,:] = A[i,k] * B[k,:]
//   bitmap bin b  column range of the row at most 32 << log_words(b) columns and
//                 min(ub_i, range) <= cap(b)     -> bitmap + rank workspace
//   register      at most 16 stored A entries whose B rows fit a lane group
//   bitmap bin b                                 -> bitmap ranked by one warp, ranks kept
//   hash bin b    ub_i <= 32 << b (b = 0..7)     -> products in registers, ranked through
//                                                  32 << b monotone-hash buckets
//   dense heavy   range up to 65,536 columns     -> flag bytes and a kept bitmap, then windows
//                                                  of consecutive output entries
//   wide heavy    range up to 2^20 columns       -> kept bitmap, then parts of the row's
//                                                  products added to C
//   dense window  rows above the others' limits  -> column slices of the row, each a
//                                                  dense bitmap + value workspace
// (analyze.cu says which rows take which).  Each class is a different
// realisation of the per-row workspace w of Gustavson's algorithm (Sec. 5.1).
// Every row, or window or slice of a row, is written by exactly one thread team,
// so C's segments are disjoint (the shard pattern, Sec. 4); only the parts of a
// wide heavy row add to the same segment (the atomic level).
#pragma once

#include <cstdint>
#include <cuda_runtime.h>

namespace wsk {

constexpr int kNumHashBins = 8;
constexpr int kMinHashLog = 5;  // bin b holds rows of at most 1 << (kMinHashLog + b) products
// Most products of a hash bucket that are compared with one another: what the 6 bits
// of its counter hold; fuller buckets sort the row.  Lower limits of 48, 32 and 16
// measured against 63: 27-point stencil over a range wider than 65,536 columns,
// squared, 17.5, 17.3 and 17.3 ms against 26.6; R-MAT 2^17 (edge factor 8) squared
// 19.24, 19.47 and 19.86 against 19.40; R-MAT 2^20 (edge factor 2) squared 56.2, 56.6
// and 56.7 against 56.0.
constexpr int kMaxHashBucket = 63;
constexpr int kMaxHashProducts = 32 << (kNumHashBins - 1);  // 4096

// Bitmap bins: bitmap of 1 << log_words 32-bit words (the row's column range
// is at most 32 << log_words columns) and a staging array of cap entries.
struct BitmapBin {
  int log_words;
  int cap;
};
constexpr int kNumBitmapBins = 5;
constexpr BitmapBin kBitmapBins[kNumBitmapBins] = {{6, 256}, {9, 512}, {11, 512}, {11, 1024}, {11, 8192}};
constexpr int kMaxBitmapSpan = 32 << 11;  // 65,536 columns
__host__ __device__ constexpr int bitmap_log_words(int b) {
  return b == 0 ? kBitmapBins[0].log_words : b == 1 ? kBitmapBins[1].log_words : b == 2 ? kBitmapBins[2].log_words
       : b == 3 ? kBitmapBins[3].log_words : kBitmapBins[4].log_words;
}
__host__ __device__ constexpr int bitmap_cap(int b) {
  return b == 0 ? kBitmapBins[0].cap : b == 1 ? kBitmapBins[1].cap : b == 2 ? kBitmapBins[2].cap
       : b == 3 ? kBitmapBins[3].cap : kBitmapBins[4].cap;
}

// Register bitmap bins: rows with at most kBmrMaxA stored A entries whose B
// rows fit one lane group; bitmap of 1 << bmr_log_words(b) words (column
// ranges of at most 4096, 16,384 and 65,536 columns).
constexpr int kNumBmrBins = 3;
constexpr int kBmrPlannedBin = kNumBmrBins;  // launch_bmr: numeric pass of the rows ranked by the planning pass
constexpr int kBmrMaxA = 16;
constexpr int kBmrCap = 512;  // >= kBmrMaxA * 32 products
constexpr int kBmrSlots = 512;  // rank slots per register bitmap row (one per possible product)
__host__ __device__ constexpr int bmr_log_words(int b) { return b == 0 ? 7 : b == 1 ? 9 : 11; }
// Sparsest row the planning pass takes: its sweep and clear cost the same for
// every row of a launch (the whole bitmap), so rows with fewer products go to
// the hash bins, whose cost follows the product count.  At 16 words per
// product a 65,536-column bitmap takes rows of 124 products and more.
constexpr long long kPlanWordsPerProduct = 16;
// Smallest register bitmap bin whose bitmap covers `span` columns (span <= kMaxBitmapSpan).
__host__ __device__ constexpr int bmr_bin_for_span(long long span) {
  return span <= (32ll << bmr_log_words(0)) ? 0 : span <= (32ll << bmr_log_words(1)) ? 1 : 2;
}

// Row class codes stored per row (uint8).
constexpr uint8_t kClsEmpty = 0;
constexpr uint8_t kClsDirect = 1;
constexpr uint8_t kClsBmr0 = 2;                            // .. + kNumBmrBins - 1
constexpr uint8_t kClsBitmap0 = kClsBmr0 + kNumBmrBins;    // .. + kNumBitmapBins - 1
constexpr uint8_t kClsHash0 = kClsBitmap0 + kNumBitmapBins;  // .. + kNumHashBins - 1
constexpr uint8_t kClsDense = kClsHash0 + kNumHashBins;
constexpr uint8_t kClsBmrWide = kClsDense + 1;  // register bitmap rows counted by the planning pass
constexpr uint8_t kClsRcd = kClsBmrWide + 1;    // dense heavy rows
constexpr uint8_t kClsWb = kClsRcd + 1;         // wide heavy rows (wide bitmap)

// Dense heavy rows.
constexpr int kRcdMaxA = 8192;            // stored A entries a row may have
constexpr int kRcdDefaultMaxA = 8192;     // default limit used by the classification
constexpr int kRcdWidthBytes = 49152;     // value window of a numeric item, at most
constexpr int kRcdLeastWidth = 512;       // entries of a window, at least
constexpr int kRcdLongB = 96;             // longest part of a B row that a warp takes; B is long above it on average
// Counters: items of rows with many products, other items, next row of the
// symbolic pass, next item of the numeric pass.
constexpr int kRcdBigItems = 0, kRcdItems = 1, kRcdNextRow = 2, kRcdNextItem = 3, kRcdCounters = 4;
// Wide heavy rows.
constexpr int kWbMaxSpan = 1 << 20;       // widest column range
constexpr int kWbPart = 16384;            // products of a numeric item, at least
constexpr int kWbMaxParts = 1024;         // items of a row, at most
// Counters: items of rows of several items, other items, next item of the numeric pass.
constexpr int kWbBigItems = 0, kWbItems = 1, kWbNextItem = 2, kWbCounters = 3;

// Segments of the row permutation: direct rows, register bitmap bins, bitmap
// bins, hash bins, dense-window rows.
constexpr int kSegDirect = 0;
constexpr int kSegBmr0 = 1;
constexpr int kSegBitmap0 = kSegBmr0 + kNumBmrBins;
constexpr int kSegHash0 = kSegBitmap0 + kNumBitmapBins;
constexpr int kSegDense = kSegHash0 + kNumHashBins;
constexpr int kSegBmrWide = kSegDense + 1;
constexpr int kSegRcd = kSegBmrWide + 1;
constexpr int kSegWb = kSegRcd + 1;
constexpr int kNumSegs = kSegWb + 1;

// Device error flags (OR-ed into DevSummary::status).
enum DevError : int {
  kErrCount = 4,       // the numeric pass found a different entry count than the symbolic pass
  kErrInvalidCsr = 8,  // validation found broken CSR invariants
};

// Counters shared between the kernels of one product and read back by the host.
struct DevSummary {
  long long nnz;       // nnz(C), written by the scan
  long long products;  // sum of ub_i
  long long dense_slices;
  long long wb_products;  // products of the wide-bitmap rows
  long long slice_cursor;
  int status;   // validation only; the passes use the status word of their plan
  int n_done;   // CTAs of analyze_long_kernel that have added their counts
  int n_sort;  // hash rows ranked by a sort
  int n_long;   // rows analysed by a CTA each (queued from the back of the long-row list)
  int n_mid;    // rows analysed by a warp each (queued from the front)
  int n_empty;
  int bad_row;
  int n_pending;  // rows the planning pass left to the analysis kernel
  int seg_count[kNumSegs];
  int seg_cursor[kNumSegs];
};

// Pinned host side of a plan: the copy of the summary, and two status words
// that kernels write errors to directly.  Passes of one handle alternate
// between the words, so a late error of an earlier pass cannot mark the next.
struct HostSummary : DevSummary {
  int slot[2];
};

// Copies the summary to its host copy and, with `reset`, clears it.  Called by
// a whole CTA after a barrier that follows the last change of the summary.
__device__ __forceinline__ void publish_summary(DevSummary* sum, DevSummary* host, bool reset) {
  static_assert(sizeof(DevSummary) % sizeof(int) == 0, "copied as ints");
  volatile int* d = reinterpret_cast<volatile int*>(sum);
  volatile int* h = reinterpret_cast<volatile int*>(host);
  for (int w = threadIdx.x; w < static_cast<int>(sizeof(DevSummary) / sizeof(int)); w += blockDim.x) {
    h[w] = d[w];
    if (reset) d[w] = 0;
  }
}

// Whether column c lies in a workspace that covers the `span` columns from lo
// on, and its offset there.  A numeric pass asks before it touches a workspace
// laid out for the columns that the symbolic pass saw; a negative c is outside.
__host__ __device__ __forceinline__ bool column_place(int c, int lo, int span, uint32_t* off) {
  *off = static_cast<uint32_t>(c) - static_cast<uint32_t>(lo);
  return *off < static_cast<uint32_t>(span);
}

// Read-only view of an input CSR matrix.
template <typename T>
struct CsrView {
  const int64_t* rowptr;
  const int32_t* colidx;
  const T* vals;
};

// Everything the row kernels need about one product.
template <typename T>
struct RowPlan {
  CsrView<T> A;
  CsrView<T> B;
  int64_t* c_rowptr;   // C.rowptr; symbolic writes counts to [i + 1] then scans in place
  int32_t* c_colidx;   // numeric only
  T* c_vals;           // numeric only
  int32_t* perm;       // rows grouped by segment
  uint8_t* cls;        // row class per row
  int32_t* lo;         // smallest column any product of the row can hit
  int32_t* hi;         // largest such column
  const int32_t* slice_row;    // dense-window slices: row, slice index, first slice of the row
  const int32_t* slice_idx;
  const int32_t* slice_first;
  int32_t* slice_cnt;          // entries per dense-window slice
  uint16_t* ranks;             // register bitmap rows: output position of every product, kBmrSlots per row
  uint16_t* hash_ranks;        // hash bin: output position of every product, 32 << bin per row of the segment
                               // (nullptr: the plan has no room, the numeric pass ranks again)
  uint32_t* rcd_bits;          // dense heavy rows: bitmap of the row's columns from lo on, rcd_words words per row
  int rcd_words;               // a multiple of 4, enough for min(columns of B, kMaxBitmapSpan)
  int rcd_width;               // entries of a value window
  bool rcd_direct;             // a window covers all columns of B, whose rows are long on average
  bool rcd_long_b;             // B's rows have more than 512 entries on average
  int rcd_slices;              // value windows of a row at most
  long long* rcd_items;        // their numeric work items (row * rcd_slices + window): rows with many products
                               // from the front, the others from the back of seg_len * rcd_slices places
  bool rcd_again;              // their bitmaps and items are wanted once more, the counts stand
  int32_t* rcd_ctr;            // counters kRcdBigItems .. kRcdNextItem
  uint32_t* wb_bits;           // wide-bitmap rows: the row's bitmap, wb_words words per row (nullptr: no room)
  int wb_words;                // a multiple of 4, enough for min(columns of B, kWbMaxSpan)
  long long* wb_items;         // numeric items (row << 32 | part << 16 | parts of the row): rows of several parts
  long long wb_cap;            // from the front, the others from the back of wb_cap places
  int32_t* wb_ctr;             // counters kWbBigItems .. kWbNextItem
  int64_t wb_part;             // products per numeric item
  DevSummary* sum;
  int* status;         // error flags (pinned host memory)
  int64_t seg_begin;   // first position in perm of the segment a kernel processes
  int64_t seg_len;     // rows in that segment
  int log2_group;      // lanes per stored A entry when walking B rows (1 << log2_group)
  int run_limit;       // most products a bucket of a hash row may hold (more: the row is sorted)
  int dense_width;     // dense-window slice width in columns
};

// Elementwise operations C = A op B on CSR matrices of one shape.
constexpr int kEwiseAdd = 1;  // SpAdd: pattern union, values added
constexpr int kEwiseMul = 2;  // Hadamard product: pattern intersection, values multiplied
constexpr int kEwTileItems = 2040;  // items of a tile: merged entries and row ends

template <typename T>
struct EwisePlan {
  CsrView<T> A;
  CsrView<T> B;
  int64_t m;
  int64_t* c_rowptr;
  int32_t* c_colidx;   // numeric only
  T* c_vals;           // numeric only
  int64_t ntiles;      // tiles of kEwTileItems items; enough for m rows and the entries of A and B
  int32_t* tile_row;   // [ntiles + 1]: first item of every tile: its row
  int64_t* tile_a;     // [ntiles + 1]:   and positions in A's
  int64_t* tile_b;     // [ntiles + 1]:   and B's arrays
  int64_t* tile_off;   // [ntiles + 1]: equal pairs before every tile (counts, then scanned in place)
  int64_t* partials;   // scan scratch for ntiles entries
  DevSummary* sum;
  int* status;         // error flags (pinned host memory)
  DevSummary* host;    // pinned: receives nnz
  int op;              // kEwiseAdd or kEwiseMul
};
template <typename T>
void launch_ewise_symbolic(const EwisePlan<T>& p, int num_sms, cudaStream_t s, int* launches);
template <typename T>
void launch_ewise_numeric(const EwisePlan<T>& p, int num_sms, cudaStream_t s, int* launches);

// Sparse matrix - sparse vector product y = A x, A given by columns (At = A^T in CSR).
template <typename T>
struct SpmspvPlan {
  CsrView<T> At;         // n x m: row j holds column j of A
  int64_t n;             // columns of A (rows of At)
  int64_t m;             // rows of A = length of y
  int64_t nnz_a;
  int64_t nx;            // stored entries of x
  const int32_t* x_idx;  // strictly increasing in [0, n)
  const T* x_vals;
  int64_t* off;          // [nx + 1]: products per x entry, then scanned in place
  int64_t* first;        // [nx]: first entry of each x entry's column in At
  T* acc;                // [m]: dense accumulator
  uint8_t* mark;         // [tiles * 4096]: 1 at the positions of y hit
  int64_t* cnt;          // [tiles + 1]: set bits per compaction tile, then scanned in place
  int64_t* partials;     // scan scratch for max(nx, tiles) entries
  DevSummary* sum;
  int* status;           // error flags (pinned host memory)
  DevSummary* host;      // host copy of the summary
  int32_t* y_idx;        // [cap]
  T* y_vals;             // [cap]
  int64_t cap;           // capacity of y (m)
};
int64_t spmspv_tiles(int64_t m);
template <typename T>
void launch_spmspv(const SpmspvPlan<T>& p, int num_sms, cudaStream_t s, int* launches);

// Submatrix S = A[r0:r1, c0:c1]: per-row counts into s_rowptr[1..rows], then the copy.
void launch_submatrix_count(const int64_t* rowptr, const int32_t* colidx, int64_t r0, int64_t rows, int64_t c0,
                            int64_t c1, int64_t* s_rowptr, int num_sms, cudaStream_t s, int* launches);
template <typename T>
void launch_submatrix_copy(const int64_t* rowptr, const int32_t* colidx, const T* vals, int64_t r0, int64_t rows,
                           int64_t c0, const int64_t* s_rowptr, int32_t* s_colidx, T* s_vals, int* status,
                           int num_sms, cudaStream_t s, int* launches);

// Host-side launchers (one translation unit each).
struct AnalyzeParams {
  int64_t m;
  int64_t hash_max;    // largest ub that uses a hash bin
  int64_t bitmap_span; // largest column range that uses a bitmap bin (0: none)
  int group;           // lanes per stored A entry in the register bitmap kernels
  int bmr_max_a;       // most stored A entries of a register bitmap row (0: none)
  int rcd_max_a;       // most stored A entries of a dense heavy row (0: no dense heavy rows)
  int64_t wb_span;     // widest column range of a wide-bitmap heavy row (0: none)
  int dense_width;
  int long_threshold;
  int64_t nnz;         // stored entries of A; an estimate, which sizes a grid only
};
// rows == nullptr: every row of A; otherwise the first sum->n_pending entries of rows.
// host != nullptr: the summary is copied there at the end.
template <typename T>
void launch_analyze(const RowPlan<T>& p, const AnalyzeParams& ap, int32_t* long_rows, const int32_t* rows,
                    DevSummary* host, int num_sms, cudaStream_t s, int* launches);
template <typename T>
void launch_bmr_plan(const RowPlan<T>& p, const AnalyzeParams& ap, int64_t ncols, int32_t* pending, int num_sms,
                     cudaStream_t s, int* launches);
template <typename T>
void launch_scatter(const RowPlan<T>& p, int64_t m, const int64_t* seg_offset, int num_sms, cudaStream_t s,
                    int* launches);
template <typename T>
void launch_dense_slices(const RowPlan<T>& p, int32_t* slice_row, int32_t* slice_idx, int32_t* slice_first,
                         int num_sms, cudaStream_t s, int* launches);
template <typename T>
void launch_hash(const RowPlan<T>& p, int bin, bool numeric, int num_sms, cudaStream_t s, int* launches);
template <typename T>
void launch_bmr(const RowPlan<T>& p, int bin, bool numeric, int num_sms, cudaStream_t s, int* launches);
template <typename T>
void launch_bitmap(const RowPlan<T>& p, int bin, bool numeric, int num_sms, cudaStream_t s, int* launches);
template <typename T>
void launch_rcd(const RowPlan<T>& p, bool numeric, int num_sms, cudaStream_t s, int* launches);
template <typename T>
void launch_wb(const RowPlan<T>& p, bool numeric, int num_sms, cudaStream_t s, int* launches);
template <typename T>
void launch_dense(const RowPlan<T>& p, int64_t nslices, bool numeric, int num_sms, cudaStream_t s,
                  int* launches);
template <typename T>
void launch_direct(const RowPlan<T>& p, int num_sms, cudaStream_t s, int* launches);

// Writes rowptr[0] = 0 too (not when m = 0: nothing is launched then).
// skip != nullptr: the scan does nothing when *skip != 0 (read on the device).
// host != nullptr: the summary block is copied there at the end, and cleared
// on the device unless the scan was skipped.
void launch_scan(int64_t* rowptr, int64_t m, int64_t* partials, DevSummary* sum, cudaStream_t s, int* launches,
                 const int* skip = nullptr, DevSummary* host = nullptr);
int64_t scan_partials_needed(int64_t m);

void launch_validate(const int64_t* rowptr, const int32_t* colidx, int64_t nrows, int64_t ncols, int64_t nnz,
                     DevSummary* sum, int num_sms, cudaStream_t s);

// Dynamic shared memory needed by the dense-window kernel.
size_t dense_smem_bytes(int width, size_t value_bytes, bool numeric);

// Exclusive prefix sum over the threads of a CTA of blockDim.x threads
// (a multiple of 32, at most 1024).  `scratch` holds 32 values; returns this
// thread's exclusive prefix and stores the CTA total in *total.  Every thread
// of the CTA must call it.
template <typename V>
__device__ __forceinline__ V block_exclusive_scan(V x, V* scratch, V* total) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarps = blockDim.x >> 5;
  V incl = x;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const V y = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += y;
  }
  if (lane == 31) scratch[warp] = incl;
  __syncthreads();
  if (warp == 0) {
    V w = lane < nwarps ? scratch[lane] : V(0);
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const V y = __shfl_up_sync(0xffffffffu, w, o);
      if (lane >= o) w += y;
    }
    if (lane < nwarps) scratch[lane] = w;  // inclusive scan of warp totals
  }
  __syncthreads();
  const V warp_prefix = warp > 0 ? scratch[warp - 1] : V(0);
  *total = scratch[nwarps - 1];
  __syncthreads();
  return warp_prefix + incl - x;
}

}  // namespace wsk
