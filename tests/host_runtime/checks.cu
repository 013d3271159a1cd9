// Checks of the library's host code on a fake CUDA runtime: checks <name>.
#include <climits>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <vector>

#include "fake_launchers.cuh"
#include "ws_spgemm.h"

namespace {

#define CHECK(cond)                                                              \
  do {                                                                           \
    if (!(cond)) {                                                               \
      std::printf("%s:%d: %s (%s)\n", __func__, __LINE__, #cond, ws_last_error()); \
      std::exit(1);                                                              \
    }                                                                            \
  } while (0)

// An m x n handle with `nnz` stored entries, whose arrays nothing reads.
ws_csr_t matrix(int64_t m, int64_t n, int64_t nnz) {
  ws_csr_t h = nullptr;
  auto* rowptr = static_cast<int64_t*>(std::calloc(static_cast<size_t>(m + 1), 8));
  CHECK(ws_csr_create(&h, m, n, nnz, rowptr, static_cast<int32_t*>(std::calloc(static_cast<size_t>(nnz + 1), 4)),
                      std::calloc(static_cast<size_t>(nnz + 1), 8), WS_F64, 0, nullptr) == WS_OK);
  return h;
}

ws_status_t failing_spmspv(ws_csr_t At) {
  int32_t idx[8] = {};
  double val[8] = {};
  int64_t n = 0;
  fake::launch_status = wsk::kErrCount;
  const ws_status_t st = ws_spmspv(At, 1, idx, val, idx, val, &n, nullptr);
  fake::launch_status = 0;
  return st;
}

// A device error of a destroyed handle does not come up in another caller's
// operation that takes over its plan.
void error_stays_with_its_handle() {
  ws_csr_t A = matrix(8, 8, 8), B = matrix(8, 8, 8), C = matrix(8, 8, 0), X = matrix(8, 8, 8);
  int64_t nnz = 0;
  CHECK(ws_spgemm_outer_symbolic(A, B, C, 3, &nnz, nullptr) == WS_OK);
  CHECK(failing_spmspv(X) == WS_ERR_DEVICE);
  CHECK(ws_csr_destroy(X) == WS_OK);
  CHECK(ws_spgemm_outer_symbolic(A, B, C, 3, &nnz, nullptr) == WS_OK);
}

// A handle destroyed while another device is current waits for its own device
// before its scratch goes to the next handle, and leaves the current device.
void destroy_waits_for_the_handles_device() {
  fake::device = 1;
  ws_csr_t X = matrix(8, 8, 8);
  int64_t nnz = 0;
  ws_csr_t S = matrix(8, 8, 0);
  CHECK(ws_csr_submatrix_symbolic(X, 0, 8, 0, 8, S, &nnz, nullptr) == WS_OK);
  fake::device = 0;
  CHECK(ws_csr_destroy(S) == WS_OK);
  CHECK(fake::synced_devices == std::vector<int>{1});
  CHECK(fake::device == 0);
}

// Side streams and their events are made on the device of the operation.
void side_streams_belong_to_the_handles_device() {
  fake::device = 1;
  ws_csr_t A = matrix(1 << 17, 1 << 17, 64), B = matrix(1 << 17, 1 << 17, 64), C = matrix(1 << 17, 1 << 17, 0);
  fake::device = 0;
  for (int b = 0; b < 4; ++b) fake::summary.seg_count[wsk::kSegHash0 + b] = 1;
  int64_t nnz = 0;
  CUstream_st stream{1, 0};
  CHECK(ws_spgemm_symbolic(A, B, C, &nnz, &stream) == WS_OK);
  CHECK(!fake::streams.empty() && !fake::events.empty());
  for (const CUstream_st* s : fake::streams) CHECK(s->device == 1);
  for (const CUevent_st* e : fake::events) CHECK(e->device == 1);
  CHECK(fake::device == 0);
}

// A product with a row in each of `kinds` hash bins, through both passes, on `stream`.
void hash_product(int kinds, cudaStream_t stream) {
  const int64_t m = 1 << 17;  // above 65,536 columns: no planning pass
  ws_csr_t A = matrix(m, m, 64), B = matrix(m, m, 64), C = matrix(m, m, 0);
  fake::summary = wsk::DevSummary{};
  for (int b = 0; b < kinds; ++b) fake::summary.seg_count[wsk::kSegHash0 + b] = 1;
  fake::summary.nnz = 64;
  fake::row_kernels.clear();
  int64_t nnz = 0;
  CHECK(ws_spgemm_symbolic(A, B, C, &nnz, stream) == WS_OK);
  CHECK(ws_spgemm_numeric(A, B, C, static_cast<int32_t*>(std::malloc(64 * 4)), std::malloc(64 * 8), stream) == WS_OK);
  CHECK(fake::row_kernels.size() == 2u * static_cast<unsigned>(kinds));
}

// Every row kernel runs at the priority of the caller's stream.
void side_streams_keep_the_callers_priority() {
  CUstream_st plain{0, 0}, high{0, -5};
  for (CUstream_st* s : {&plain, &high, &plain, &high}) {
    hash_product(4, s);
    int others = 0;
    for (cudaStream_t q : fake::row_kernels) {
      CHECK(q->priority == s->priority);
      others += q != s;
    }
    CHECK(others > 0);
  }
  CHECK(fake::streams.size() == 6);  // a set for each priority, used again
}

// A stream confined to a part of the GPU keeps all row kernels; side streams
// made in one context are not used in another.
void side_streams_stay_where_the_caller_is() {
  CUstream_st confined{0, 0, true}, plain{0, 0};
  hash_product(4, &confined);
  for (cudaStream_t q : fake::row_kernels) CHECK(q == &confined);
  CHECK(fake::streams.empty());
  for (unsigned long long context : {1, 2, 1}) {
    fake::context = context;
    hash_product(4, &plain);
    for (cudaStream_t q : fake::row_kernels) CHECK(q == &plain || q->context == context);
  }
  CHECK(fake::streams.size() == 6);  // a set for each context, used again
}

// The outer product's blocks use the same scratch one after another.
void outer_blocks_share_scratch() {
  const int64_t m = 1 << 17;
  ws_csr_t A = matrix(m, m, 64), B = matrix(m, m, 64), C = matrix(m, m, 0);
  const size_t rows = 20000, ranks = rows * 2 * wsk::kMaxHashProducts;
  fake::summary.seg_count[wsk::kSegHash0 + wsk::kNumHashBins - 1] = rows;
  fake::summary.nnz = 64;
  int64_t nnz = 0;
  CHECK(ws_spgemm_outer_symbolic(A, B, C, 8, &nnz, nullptr) == WS_OK);
  CHECK(fake::peak > ranks && fake::peak < 2 * ranks);
  CHECK(ws_spgemm_outer_numeric(A, B, C, static_cast<int32_t*>(std::malloc(64 * 4)), std::malloc(64 * 8), nullptr) == WS_OK);
  CHECK(fake::bytes < ranks / 2);  // the last block's goes with its partial product
  CHECK(ws_spgemm_wait(C, nullptr) == WS_OK);
}

// When a block of the outer product finds no memory, the status words of the
// blocks before it are given back after the kernels that may write to them.
void failed_outer_product_waits_for_its_kernels() {
  const int64_t m = 1 << 17;
  ws_csr_t A = matrix(m, m, 64), B = matrix(m, m, 64), C = matrix(m, m, 0);
  fake::summary.seg_count[wsk::kSegHash0] = 1;
  fake::summary.nnz = 64;
  int64_t nnz = 0;
  int failed = 0;
  for (int k = 0; k < 40; ++k) {  // some allocations the call can do without
    fake::fail_in = k;
    failed += ws_spgemm_outer_symbolic(A, B, C, 5, &nnz, nullptr) == WS_ERR_ALLOC;
    CHECK(fake::pending.empty());
  }
  CHECK(failed > 20);
}

// A column has a place in a row's workspace only inside the row's range.
void columns_outside_have_no_place() {
  const int lows[] = {0, 1, 65535, 1 << 20, INT_MAX - (1 << 20)}, spans[] = {1, 31, 128, 65536, 1 << 20};
  for (int lo : lows) {
    for (int span : spans) {
      const long long end = static_cast<long long>(lo) + span;
      for (long long c : {-1ll, 0ll, lo - 1ll, static_cast<long long>(lo), end - 1, end, end + 1, static_cast<long long>(INT_MAX)}) {
        if (c > INT_MAX) continue;
        uint32_t off = 0;
        const bool in = wsk::column_place(static_cast<int>(c), lo, span, &off);
        CHECK(in == (c >= lo && c < end));
        CHECK(!in || off == c - lo);
      }
    }
  }
}

// Wide rows share few large items when there are many of them (the fake GPU
// has 4 SMs).
void wide_rows_are_cut_as_far_as_the_gpu_needs() {
  const int64_t m = 1 << 17;
  const struct {
    int rows;
    int64_t products, part;
  } cases[] = {{1, 5000, 16384}, {7, 7 * 18000, 16384}, {8, 8 * 18000, 32768}, {100, 100 * 18000, 100 * 18000 / 16}};
  for (const auto& c : cases) {
    ws_csr_t A = matrix(m, m, 64), B = matrix(m, m, 64), C = matrix(m, m, 0);
    fake::summary = wsk::DevSummary{};
    fake::summary.seg_count[wsk::kSegWb] = c.rows;
    fake::summary.products = fake::summary.wb_products = c.products;
    int64_t nnz = 0;
    CHECK(ws_spgemm_symbolic(A, B, C, &nnz, nullptr) == WS_OK);
    CHECK(fake::wb_part == c.part);
  }
}

// The bitmap bin of 65,536 columns is ahead of the side streams if it has rows
// enough, and shares them otherwise.
void many_wide_bitmap_rows_run_by_themselves() {
  const int64_t m = 1 << 17;
  CUstream_st stream{0, 0};
  for (int rows : {16384, 16385}) {
    ws_csr_t A = matrix(m, m, 64), B = matrix(m, m, 64), C = matrix(m, m, 0);
    fake::summary = wsk::DevSummary{};
    fake::summary.seg_count[wsk::kSegBitmap0 + 2] = rows;
    for (int b = 0; b < 4; ++b) fake::summary.seg_count[wsk::kSegHash0 + b] = 1;
    fake::summary.nnz = 64;
    int64_t nnz = 0;
    fake::row_kernels.clear();
    fake::bitmap_after.clear();
    CHECK(ws_spgemm_symbolic(A, B, C, &nnz, &stream) == WS_OK);
    CHECK(ws_spgemm_numeric(A, B, C, static_cast<int32_t*>(std::malloc(64 * 4)), std::malloc(64 * 8), &stream) == WS_OK);
    CHECK(fake::row_kernels.size() == 10u && fake::bitmap_after.size() == 2u);
    // kernels queued before it, the same in both passes
    CHECK(fake::bitmap_after[0] == (rows > 16384 ? 0u : 4u) && fake::bitmap_after[1] == fake::bitmap_after[0] + 5u);
    if (rows > 16384) CHECK(fake::row_kernels[0] == &stream && fake::row_kernels[5] == &stream);
  }
}

// Dense rows are cut into value windows for three CTAs per SM (of 4) if they
// would not keep every SM busy and B's rows have more than 96 entries on average.
void few_dense_rows_take_small_windows() {
  const int widest = wsk::kRcdWidthBytes / 8;
  const struct {
    int rows;
    int64_t ncols, b_row;
    int width;
  } cases[] = {{1, 3000, 97, 512},      {3, 3000, 97, 1024},     {4, 3000, 97, widest}, {1, 60000, 97, widest},
               {1, 20000, 97, widest}, {1, 18000, 97, 1536}, {1, 3000, 96, widest}};
  for (const auto& c : cases) {
    ws_csr_t A = matrix(100, 1 << 10, 64), B = matrix(1 << 10, c.ncols, c.b_row << 10), C = matrix(100, c.ncols, 0);
    fake::summary = wsk::DevSummary{};
    fake::summary.n_pending = 1;
    fake::summary.seg_count[wsk::kSegRcd] = c.rows;
    int64_t nnz = 0;
    CHECK(ws_spgemm_symbolic(A, B, C, &nnz, nullptr) == WS_OK);
    CHECK(fake::rcd_width == c.width);
    CHECK(fake::rcd_slices == (c.ncols + c.width - 1) / c.width);
  }
}

// Ranks and bitmaps kept between the passes take at most 4 GiB of each kind, as
// allocated, and a little more with the items and the rows' arrays.
void kept_scratch_is_bounded() {
  const struct {
    int seg;
    int64_t ncols, rows;
  } cases[] = {{wsk::kSegHash0 + wsk::kNumHashBins - 1, 1 << 17, 500000}, {wsk::kSegRcd, 60000, 560000}, {wsk::kSegWb, 1 << 21, 32000}};
  for (const auto& c : cases) {
    ws_csr_t A = matrix(c.rows, 1 << 17, 64), B = matrix(1 << 17, c.ncols, 64), C = matrix(c.rows, c.ncols, 0);
    fake::summary = wsk::DevSummary{};
    fake::summary.n_pending = 1;
    fake::summary.seg_count[c.seg] = static_cast<int>(c.rows);
    fake::peak = fake::bytes;
    const size_t before = fake::bytes;
    int64_t nnz = 0;
    CHECK(ws_spgemm_symbolic(A, B, C, &nnz, nullptr) == WS_OK);
    CHECK(fake::peak - before < (size_t{4} << 30) + 100 * static_cast<size_t>(c.rows) + (size_t{64} << 20));
    CHECK(ws_csr_destroy(C) == WS_OK);
  }
}

// Buckets of more than 63 products are sorted, whatever limit is asked for.
void bucket_limit_is_what_the_kernel_can_hold() {
  hash_product(1, nullptr);
  CHECK(fake::run_limit == 63);
  for (int64_t limit : {4096, 64, 63, 62, 1}) {
    CHECK(ws_set_tuning(2, limit) == WS_OK);
    hash_product(1, nullptr);
    CHECK(fake::run_limit == (limit < 63 ? limit : 63));
  }
  CHECK(ws_set_tuning(2, 4097) == WS_ERR_INVALID_ARG);
}

struct {
  const char* name;
  void (*run)();
} const kChecks[] = {
    {"error_stays_with_its_handle", error_stays_with_its_handle},
    {"destroy_waits_for_the_handles_device", destroy_waits_for_the_handles_device},
    {"side_streams_belong_to_the_handles_device", side_streams_belong_to_the_handles_device},
    {"side_streams_keep_the_callers_priority", side_streams_keep_the_callers_priority},
    {"side_streams_stay_where_the_caller_is", side_streams_stay_where_the_caller_is},
    {"outer_blocks_share_scratch", outer_blocks_share_scratch},
    {"wide_rows_are_cut_as_far_as_the_gpu_needs", wide_rows_are_cut_as_far_as_the_gpu_needs},
    {"many_wide_bitmap_rows_run_by_themselves", many_wide_bitmap_rows_run_by_themselves},
    {"few_dense_rows_take_small_windows", few_dense_rows_take_small_windows},
    {"kept_scratch_is_bounded", kept_scratch_is_bounded},
    {"bucket_limit_is_what_the_kernel_can_hold", bucket_limit_is_what_the_kernel_can_hold},
    {"columns_outside_have_no_place", columns_outside_have_no_place},
    {"failed_outer_product_waits_for_its_kernels", failed_outer_product_waits_for_its_kernels},
};

}  // namespace

int main(int argc, char** argv) {
  if (argc < 2) {
    for (const auto& c : kChecks) std::puts(c.name);
    return 0;
  }
  for (const auto& c : kChecks) {
    if (std::strcmp(c.name, argv[1]) == 0) {
      c.run();
      return 0;
    }
  }
  std::puts("no such check");
  return 2;
}
