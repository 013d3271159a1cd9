// Device-wide prefix sum that turns per-row entry counts into C's row
// pointer (the monotone position array of the compressed format, Sec. 1 and
// Sec. 3.1): on entry rowptr[i + 1] holds nnz(C[i,:]); on exit rowptr[0] = 0
// and rowptr[i + 1] = sum_{r <= i} nnz(C[r,:]).
//
// Reduce-then-scan: tile sums, then every CTA scans its tile from the sum of
// the tiles before it, which it adds up itself (two launches; above
// kDirectPartials tiles one more launch scans the tile sums first).  Arrays of
// at most kSmallScan entries are scanned by one CTA in one launch.  No CTA
// waits on another, so the scan cannot stall however the CTAs are scheduled.
// Tiles go through shared memory, so that global loads and stores are
// coalesced (a thread reading its 16 consecutive entries from global memory
// took 12.5 us for 2^20 rows, 3 of 21 us being the launch for the tile sums).
// With a `skip` flag the kernels do nothing when *skip != 0 (a scan queued
// before the host knows whether every count is in place).
//
// With `host` the CTA that ends the scan also copies the summary block to that
// (pinned) host address, which saves a copy of its own, and, unless the scan is
// skipped, clears the block for the next pass.
#include "ws_internal.cuh"

namespace wsk {

namespace {

constexpr int kScanThreads = 256;
constexpr int kScanItems = 16;
constexpr int kTile = kScanThreads * kScanItems;
constexpr int64_t kDirectPartials = 4096;
constexpr int kSmallThreads = 1024;
constexpr int kSmallItems = 4;
constexpr int64_t kSmallScan = static_cast<int64_t>(kSmallThreads) * kSmallItems;

__global__ void __launch_bounds__(kScanThreads) scan_reduce_kernel(const int64_t* x, int64_t n, int64_t* partial,
                                                                    const int* skip) {
  if (skip && *skip) return;
  __shared__ long long scratch[32];
  const int64_t tile0 = static_cast<int64_t>(blockIdx.x) * kTile;
  long long s = 0;
#pragma unroll
  for (int j = 0; j < kScanItems; ++j) {
    const int64_t i = tile0 + static_cast<int64_t>(j) * kScanThreads + threadIdx.x;
    if (i < n) s += x[i];
  }
  long long total;
  block_exclusive_scan(s, scratch, &total);
  if (threadIdx.x == 0) partial[blockIdx.x] = total;
}

// Exclusive scan of the tile sums, in place, by one CTA of 1024 threads.
__global__ void __launch_bounds__(1024) scan_partials_kernel(int64_t* partial, int64_t nb, const int* skip) {
  if (skip && *skip) return;
  __shared__ long long scratch[32];
  long long carry = 0;
  for (int64_t b0 = 0; b0 < nb; b0 += blockDim.x) {
    const int64_t b = b0 + threadIdx.x;
    const long long v = b < nb ? partial[b] : 0;
    long long total;
    const long long ex = block_exclusive_scan(v, scratch, &total);
    if (b < nb) partial[b] = carry + ex;
    carry += total;
  }
}

// Inclusive scan of one tile of x in place, continuing from `before`; returns
// the tile's sum.  buf holds THREADS * (ITEMS + 1) values: entry i sits at
// i + i / ITEMS, so a thread's ITEMS consecutive entries and the coalesced
// accesses both fall into different banks.
template <int THREADS, int ITEMS>
__device__ __forceinline__ long long scan_tile(int64_t* x, int64_t n, int64_t tile0, long long before, long long* buf,
                                               long long* scratch) {
  const int t = threadIdx.x;
#pragma unroll
  for (int j = 0; j < ITEMS; ++j) {
    const int k = j * THREADS + t;
    buf[k + k / ITEMS] = tile0 + k < n ? x[tile0 + k] : 0;
  }
  __syncthreads();
  long long v[ITEMS], s = 0;
#pragma unroll
  for (int j = 0; j < ITEMS; ++j) {
    v[j] = buf[t * (ITEMS + 1) + j];
    s += v[j];
  }
  long long total;
  long long run = block_exclusive_scan(s, scratch, &total) + before;
#pragma unroll
  for (int j = 0; j < ITEMS; ++j) {
    run += v[j];
    buf[t * (ITEMS + 1) + j] = run;
  }
  __syncthreads();
#pragma unroll
  for (int j = 0; j < ITEMS; ++j) {
    const int k = j * THREADS + t;
    if (tile0 + k < n) x[tile0 + k] = buf[k + k / ITEMS];
  }
  return total;
}

// The end of a scan: C.rowptr[0], nnz, and the summary for the host.
__device__ __forceinline__ void finish_scan(int64_t* x, long long nnz, DevSummary* sum, DevSummary* host, bool skipped) {
  if (threadIdx.x == 0 && !skipped) {
    x[-1] = 0;
    sum->nnz = nnz;
  }
  if (host) {
    __syncthreads();
    publish_summary(sum, host, !skipped);
  }
}

__global__ void __launch_bounds__(kScanThreads) scan_apply_kernel(int64_t* x, int64_t n, const int64_t* partial,
                                                                   bool scanned, DevSummary* sum, const int* skip,
                                                                   DevSummary* host) {
  const bool last = blockIdx.x + 1 == gridDim.x;
  if (skip && *skip) {
    if (last) finish_scan(x, 0, sum, host, true);
    return;
  }
  __shared__ long long buf[kScanThreads * (kScanItems + 1)];
  __shared__ long long scratch[32];
  long long before = 0;
  if (scanned) {
    before = partial[blockIdx.x];
  } else {
    long long s = 0;
    for (int64_t b = threadIdx.x; b < blockIdx.x; b += kScanThreads) s += partial[b];
    block_exclusive_scan(s, scratch, &before);
  }
  const long long total = scan_tile<kScanThreads, kScanItems>(x, n, static_cast<int64_t>(blockIdx.x) * kTile, before, buf, scratch);
  if (last) finish_scan(x, before + total, sum, host, false);
}

__global__ void __launch_bounds__(kSmallThreads) scan_small_kernel(int64_t* x, int64_t n, DevSummary* sum,
                                                                   const int* skip, DevSummary* host) {
  if (skip && *skip) {
    finish_scan(x, 0, sum, host, true);
    return;
  }
  __shared__ long long buf[kSmallThreads * (kSmallItems + 1)];
  __shared__ long long scratch[32];
  const long long total = scan_tile<kSmallThreads, kSmallItems>(x, n, 0, 0, buf, scratch);
  finish_scan(x, total, sum, host, false);
}

}  // namespace

int64_t scan_partials_needed(int64_t m) { return (m + kTile - 1) / kTile; }

void launch_scan(int64_t* rowptr, int64_t m, int64_t* partials, DevSummary* sum, cudaStream_t s, int* launches,
                 const int* skip, DevSummary* host) {
  if (m <= 0) return;
  if (m <= kSmallScan) {
    scan_small_kernel<<<1, kSmallThreads, 0, s>>>(rowptr + 1, m, sum, skip, host);
    *launches += 1;
    return;
  }
  const int64_t nb = scan_partials_needed(m);
  const bool scanned = nb > kDirectPartials;
  scan_reduce_kernel<<<static_cast<int>(nb), kScanThreads, 0, s>>>(rowptr + 1, m, partials, skip);
  if (scanned) scan_partials_kernel<<<1, 1024, 0, s>>>(partials, nb, skip);
  scan_apply_kernel<<<static_cast<int>(nb), kScanThreads, 0, s>>>(rowptr + 1, m, partials, scanned, sum, skip, host);
  *launches += scanned ? 3 : 2;
}

}  // namespace wsk
