// C ABI of the SpGEMM library (declared in include/ws_spgemm.h).
//
// Symbolic pass (ws_spgemm_symbolic):
//   1. plan      regular rows counted in the first read of A, where
//                columns and averages allow                         (1 launch and a scan)
//      analyze   per-row product count, column range, class         (2 launches)
//   -- the class counts reach the host (written by the last kernel, stream sync);
//      if the planning pass took every row, this is the end
//   2. scatter   group rows by class                                (1 launch)
//   3. rows      count the distinct columns, per class and bin      (1 launch each, 2 for dense windows)
//   4. scan      counts -> C.rowptr                                 (1, 2 or 3 launches)
//   -- nnz(C) and the status word reach the host (written by the scan, stream sync)
// Numeric pass (ws_spgemm_numeric), no sync: one launch per non-empty class and
// bin; one more that zeroes the wide rows cut into parts; dense heavy rows without
// room for all bitmaps go in batches of two.
// The row kernels of both passes are spread over the caller's stream and up to
// three side streams (class Fork), everything else stays on the caller's stream.
#include <cuda.h>

#include <cstdarg>
#include <cstddef>
#include <cstdio>
#include <cstring>
#include <mutex>
#include <new>
#include <string>
#include <utility>
#include <vector>

#include "ws_internal.cuh"
#include "ws_spgemm.h"

using namespace wsk;

namespace {

thread_local std::string g_last_error;

// Process-wide tuning (ws_set_tuning).
int64_t g_hash_max = kMaxHashProducts;
int64_t g_bitmap_span = kMaxBitmapSpan;
int g_bmr_max_a = kBmrMaxA;
int g_rcd_max_a = kRcdDefaultMaxA;
int64_t g_wb_span = kWbMaxSpan;
int g_run_limit = kMaxHashBucket;
int g_dense_width = 0;  // 0 = default per value type
constexpr int kLongRowThreshold = 16;  // rows with more stored entries are analysed by a warp or a CTA

ws_status_t fail(ws_status_t st, const char* fmt, ...) __attribute__((format(printf, 2, 3)));
ws_status_t fail(ws_status_t st, const char* fmt, ...) {
  char buf[512];
  va_list ap;
  va_start(ap, fmt);
  vsnprintf(buf, sizeof(buf), fmt, ap);
  va_end(ap);
  g_last_error = buf;
  return st;
}

ws_status_t cuda_fail(cudaError_t e, const char* what) {
  return fail(WS_ERR_CUDA, "%s: %s", what, cudaGetErrorString(e));
}

#define WS_CUDA(call, what)                     \
  do {                                          \
    cudaError_t e_ = (call);                    \
    if (e_ != cudaSuccess) return cuda_fail(e_, what); \
  } while (0)

size_t align_up(size_t x, size_t a) { return (x + a - 1) / a * a; }

// Makes `device` the current device for its own lifetime.
class DeviceGuard {
 public:
  explicit DeviceGuard(int device) {
    if (cudaGetDevice(&before_) != cudaSuccess) return;
    ok_ = before_ == device || cudaSetDevice(device) == cudaSuccess;
    changed_ = ok_ && before_ != device;
    if (!ok_) cudaGetLastError();
  }
  DeviceGuard(const DeviceGuard&) = delete;
  DeviceGuard& operator=(const DeviceGuard&) = delete;
  ~DeviceGuard() {
    if (changed_) cudaSetDevice(before_);
  }
  bool ok() const { return ok_; }

 private:
  int before_ = 0;
  bool ok_ = false, changed_ = false;
};

// Grow-only stream-ordered device buffer.
struct DevBuf {
  void* ptr = nullptr;
  size_t bytes = 0;
  uint64_t gen = 0;  // changes with every allocation (0: none yet)
  static size_t allocated(size_t need) { return need + need / 8; }
  ws_status_t reserve(size_t need, cudaStream_t s) {
    if (need <= bytes) return WS_OK;
    if (ptr) {
      cudaError_t e = cudaFreeAsync(ptr, s);
      ptr = nullptr;
      bytes = 0;
      if (e != cudaSuccess) return cuda_fail(e, "cudaFreeAsync");
    }
    const size_t want = allocated(need);
    cudaError_t e = cudaMallocAsync(&ptr, want, s);
    if (e != cudaSuccess) {
      ptr = nullptr;
      return fail(WS_ERR_ALLOC, "cudaMallocAsync(%zu bytes): %s", want, cudaGetErrorString(e));
    }
    bytes = want;
    ++gen;
    return WS_OK;
  }
  // Returns the memory to the stream-ordered pool (callers synchronise the
  // device first, so no queued work still uses it).
  void release() {
    if (ptr) cudaFreeAsync(ptr, nullptr);
    ptr = nullptr;
    bytes = 0;
  }
};

// Pinned host copies of the summary block, recycled across handles: a
// cudaMallocHost / cudaFreeHost pair per handle costs more than a small
// product.  Blocks are allocated 64 at a time and kept until the process
// exits.
std::mutex g_host_sum_mutex;
std::vector<HostSummary*> g_host_sum_free;

HostSummary* acquire_host_sum() {
  std::lock_guard<std::mutex> lock(g_host_sum_mutex);
  if (g_host_sum_free.empty()) {
    constexpr int kBlocks = 64;
    const size_t each = (sizeof(HostSummary) + 255) / 256 * 256;
    char* base = nullptr;
    if (cudaMallocHost(reinterpret_cast<void**>(&base), each * kBlocks) != cudaSuccess) return nullptr;
    for (int i = kBlocks - 1; i >= 0; --i) g_host_sum_free.push_back(reinterpret_cast<HostSummary*>(base + i * each));
  }
  HostSummary* h = g_host_sum_free.back();
  g_host_sum_free.pop_back();
  h->slot[0] = h->slot[1] = 0;
  return h;
}

void release_host_sum(HostSummary* h) {
  if (!h) return;
  std::lock_guard<std::mutex> lock(g_host_sum_mutex);
  g_host_sum_free.push_back(h);
}

// Once per device: let the default stream-ordered pool keep freed memory
// (its default releases it to the system at every synchronisation, so the
// next handle's scratch would be allocated from scratch again).  This is a
// setting of this process's pool, not of the GPU.
void keep_pool_memory(int dev) {
  static std::mutex m;
  static bool done[64] = {};
  std::lock_guard<std::mutex> lock(m);
  if (dev < 0 || dev >= 64 || done[dev]) return;
  cudaMemPool_t pool;
  if (cudaDeviceGetDefaultMemPool(&pool, dev) == cudaSuccess) {
    uint64_t keep = UINT64_MAX;
    cudaMemPoolSetAttribute(pool, cudaMemPoolAttrReleaseThreshold, &keep);
  }
  done[dev] = true;
}

// A driver function by name (nullptr if the driver has none of that name).
template <typename F>
F driver_function(const char* name, unsigned version) {
  void* f = nullptr;
  cudaDriverEntryPointQueryResult found = cudaDriverEntryPointSymbolNotFound;
  if (cudaGetDriverEntryPointByVersion(name, &f, version, cudaEnableDefault, &found) != cudaSuccess ||
      found != cudaDriverEntryPointSuccess) {
    cudaGetLastError();
    return nullptr;
  }
  return reinterpret_cast<F>(f);
}

// The number of the current context, and whether `s` is confined to a part of
// the GPU (a stream of a green context).  False if the driver cannot tell.
bool stream_place(cudaStream_t s, unsigned long long* context, bool* confined) {
  static const auto get_current = driver_function<CUresult(CUDAAPI*)(CUcontext*)>("cuCtxGetCurrent", 4000);
  static const auto get_id = driver_function<CUresult(CUDAAPI*)(CUcontext, unsigned long long*)>("cuCtxGetId", 12000);
  static const auto get_green = driver_function<CUresult(CUDAAPI*)(CUstream, CUgreenCtx*)>("cuStreamGetGreenCtx", 12040);
  CUcontext ctx = nullptr;
  CUgreenCtx green = nullptr;
  if (!get_current || !get_id || !get_green || get_current(&ctx) != CUDA_SUCCESS || !ctx ||
      get_id(ctx, context) != CUDA_SUCCESS || get_green(s, &green) != CUDA_SUCCESS)
    return false;
  *confined = green != nullptr;
  return true;
}

// Side streams for the independent row kernels of one pass: the classes of
// rows touch different rows of C, so their kernels may overlap, and a class of
// few long rows then does not leave the GPU to one CTA per row.  They have the
// priority of the caller's stream.  Sets are checked out for the duration of one call, recycled across handles and
// threads, and at most kMaxSets are kept.
struct SideStreams {
  static constexpr int kStreams = 3;
  int device = 0;
  int priority = 0;
  unsigned long long context = 0;  // streams serve the context they were made in only
  cudaStream_t st[kStreams] = {};
  cudaEvent_t fork = nullptr, join[kStreams] = {};
};
constexpr size_t kMaxSets = 8;
std::mutex g_side_mutex;
std::vector<SideStreams*> g_side_free;

void destroy_side(SideStreams* x) {
  for (int i = 0; i < SideStreams::kStreams; ++i) {
    if (x->st[i]) cudaStreamDestroy(x->st[i]);
    if (x->join[i]) cudaEventDestroy(x->join[i]);
  }
  if (x->fork) cudaEventDestroy(x->fork);
  delete x;
}

SideStreams* acquire_side(int device, int priority, unsigned long long context) {
  {
    std::lock_guard<std::mutex> lock(g_side_mutex);
    for (size_t i = 0; i < g_side_free.size(); ++i) {
      SideStreams* x = g_side_free[i];
      if (x->device == device && x->priority == priority && x->context == context) {
        g_side_free.erase(g_side_free.begin() + static_cast<std::ptrdiff_t>(i));
        return x;
      }
    }
  }
  SideStreams* x = new (std::nothrow) SideStreams;
  if (!x) return nullptr;
  x->device = device;
  x->priority = priority;
  x->context = context;
  bool ok = cudaEventCreateWithFlags(&x->fork, cudaEventDisableTiming) == cudaSuccess;
  for (int i = 0; i < SideStreams::kStreams && ok; ++i) {
    ok = cudaStreamCreateWithPriority(&x->st[i], cudaStreamNonBlocking, priority) == cudaSuccess &&
         cudaEventCreateWithFlags(&x->join[i], cudaEventDisableTiming) == cudaSuccess;
  }
  if (!ok) {
    cudaGetLastError();  // the caller goes on without side streams
    destroy_side(x);
    return nullptr;
  }
  return x;
}

void release_side(SideStreams* x) {
  {
    std::lock_guard<std::mutex> lock(g_side_mutex);
    if (g_side_free.size() < kMaxSets) {
      try {
        g_side_free.push_back(x);
        return;
      } catch (...) {
      }
    }
  }
  destroy_side(x);  // pending work completes first
}

// Spreads `kernels` independent launches over the caller's stream and a set
// of side streams, everything ordered after what the caller's stream holds;
// join() orders the caller's stream after all of them, so outside the call
// the work looks as if it had been queued on that stream alone.  Fewer than
// kMinKernels launches, streams that are being captured (a recycled stream
// must not stay in a capture) and streams confined to a part of the GPU use the
// caller's stream only.
class Fork {
 public:
  static constexpr int kMinKernels = 3;
  Fork(cudaStream_t main, int device, int kernels) : main_(main) {
    if (kernels < kMinKernels) return;
    const DeviceGuard guard(device);
    if (!guard.ok()) return;
    cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
    if (cudaStreamIsCapturing(main, &cap) != cudaSuccess || cap != cudaStreamCaptureStatusNone) {
      cudaGetLastError();
      return;
    }
    unsigned long long context = 0;
    bool confined = false;
    if (!stream_place(main, &context, &confined) || confined) return;
    int priority = 0;
    if (cudaStreamGetPriority(main, &priority) != cudaSuccess) {
      cudaGetLastError();
      return;
    }
    side_ = acquire_side(device, priority, context);
    if (side_ && cudaEventRecord(side_->fork, main_) != cudaSuccess) {
      cudaGetLastError();
      release_side(side_);
      side_ = nullptr;
    }
  }
  Fork(const Fork&) = delete;
  Fork& operator=(const Fork&) = delete;
  ~Fork() { join(); }
  // Stream of the next launch.
  cudaStream_t next() {
    if (!side_) return main_;
    const int i = turn_++ % (SideStreams::kStreams + 1) - 1;
    if (i < 0) return main_;
    if (!used_[i]) {
      if (cudaStreamWaitEvent(side_->st[i], side_->fork, 0) != cudaSuccess) {
        cudaGetLastError();
        return main_;
      }
      used_[i] = true;
    }
    return side_->st[i];
  }
  cudaError_t join() {
    if (!side_) return cudaSuccess;
    cudaError_t e = cudaSuccess;
    for (int i = 0; i < SideStreams::kStreams; ++i) {
      if (!used_[i]) continue;
      cudaError_t x = cudaEventRecord(side_->join[i], side_->st[i]);
      if (x == cudaSuccess) x = cudaStreamWaitEvent(main_, side_->join[i], 0);
      if (x != cudaSuccess) {
        cudaStreamSynchronize(side_->st[i]);  // keeps the order all the same
        e = x;
      }
    }
    release_side(side_);
    side_ = nullptr;
    return e;
  }

 private:
  cudaStream_t main_;
  SideStreams* side_ = nullptr;
  bool used_[SideStreams::kStreams] = {};
  int turn_ = 0;
};

enum PlanKind { kPlanNone = 0, kPlanSpgemm = 1, kPlanEwise = 2, kPlanSub = 3 };

struct Plan {
  DevBuf rows;    // per-row arrays + summary + scan partials
  DevBuf slices;  // dense-window slice arrays
  DevBuf ranks;   // register bitmap rows: kBmrSlots uint16 ranks per row of A
  DevBuf ew;      // elementwise operations: summary, chunk arrays, scan partials
  DevBuf sv;      // sparse matrix - sparse vector product (in A^T's handle): accumulator, byte-map, offsets
  DevBuf hranks;  // hash rows: uint16 ranks of their products, one block per bin
  DevBuf rcd;     // dense heavy rows: work counters, numeric items, the rows' bitmaps
  DevBuf wb;      // wide-bitmap rows: work counters, numeric items, the rows' bitmaps
  int kind = kPlanNone;  // which symbolic pass filled this plan
  // elementwise plan (kPlanEwise)
  int ew_op = 0;
  int64_t ew_ntiles = 0;
  int32_t* ew_tile_row = nullptr;
  int64_t* ew_tile_a = nullptr;
  int64_t* ew_tile_b = nullptr;
  int64_t* ew_tile_off = nullptr;
  int64_t* ew_partials = nullptr;
  int32_t* rcd_ctr = nullptr;
  long long* rcd_items = nullptr;
  uint32_t* rcd_bits = nullptr;
  int rcd_words = 0;
  int rcd_width = 0, rcd_slices = 0;
  int32_t* wb_ctr = nullptr;
  long long* wb_items = nullptr;
  uint32_t* wb_bits = nullptr;
  int wb_words = 0;
  int64_t wb_cap = 0;
  int64_t wb_part = 0;
  int64_t wb_products = 0;
  int64_t rcd_batch = 0;  // dense heavy rows that rcd_items and rcd_bits have room for
  // submatrix plan (kPlanSub): the block the symbolic pass counted
  int64_t sub_r0 = 0, sub_r1 = 0, sub_c0 = 0, sub_c1 = 0;
  HostSummary* host_sum = nullptr;  // pinned
  int slot = 0;                     // status word of the current pass in it
  const DevBuf* clean_buf = nullptr;  // buffer whose summary block the last pass left cleared,
  uint64_t clean_gen = 0;             // in this allocation of it
  // carved pointers
  DevSummary* dsum = nullptr;
  int32_t* perm = nullptr;
  uint8_t* cls = nullptr;
  int32_t* lo = nullptr;
  int32_t* hi = nullptr;
  int32_t* long_rows = nullptr;
  int32_t* pending = nullptr;
  int64_t* partials = nullptr;
  int32_t* slice_row = nullptr;
  int32_t* slice_idx = nullptr;
  int32_t* slice_first = nullptr;
  int32_t* slice_cnt = nullptr;
  // results of the last symbolic pass
  bool ready = false;
  const void* A = nullptr;
  const void* B = nullptr;
  int64_t a_nnz = -1, b_nnz = -1;
  int64_t seg_count[kNumSegs] = {};
  int64_t seg_offset[kNumSegs + 1] = {};
  int64_t n_sort = 0, n_empty = 0, dense_slices = 0, products = 0;
  int log2_group = 5;
  bool all_planned = false;  // the planning pass took every row: its segment is rows 0..m-1 in order
  int dense_width = 0;
  int run_limit = kMaxHashBucket;
  bool hash_ranked = false;  // hranks holds the hash rows' ranks
  int sym_launches = 0, num_launches = 0;
  struct OuterState* outer = nullptr;  // outer-product SpGEMM between its two passes
  int device = 0;

  size_t scratch_bytes() const {
    size_t n = 0;
    for (const DevBuf* b : {&rows, &slices, &ranks, &ew, &sv, &hranks, &rcd, &wb}) n += b->bytes;
    return n;
  }
  // Back to a new plan that owns the same scratch and pinned block, whose
  // status words start clear like those of a new one.
  void recycle() {
    host_sum->slot[0] = host_sum->slot[1] = 0;
    Plan fresh;
    fresh.rows = rows;
    fresh.slices = slices;
    fresh.ranks = ranks;
    fresh.ew = ew;
    fresh.sv = sv;
    fresh.hranks = hranks;
    fresh.rcd = rcd;
    fresh.wb = wb;
    fresh.host_sum = host_sum;
    fresh.slot = slot;
    fresh.clean_buf = clean_buf;  // points into this object, whose address stays
    fresh.clean_gen = clean_gen;
    fresh.device = device;
    *this = fresh;
  }
};

// Plans of destroyed handles, for the next handles of their device: a one-shot
// call otherwise spends as long on allocating and freeing its scratch as on a
// small product.  A plan gets here after its device has finished all work, so
// it may serve any stream.  At most kMaxPlans of at most kMaxPlanBytes scratch
// each are kept; larger scratch goes back to the stream-ordered pool.
constexpr size_t kMaxPlans = 8;
constexpr size_t kMaxPlanBytes = size_t{32} << 20;
std::mutex g_plan_mutex;
std::vector<Plan*> g_plan_free;

Plan* recycled_plan(int device) {
  std::lock_guard<std::mutex> lock(g_plan_mutex);
  for (size_t i = g_plan_free.size(); i-- > 0;) {
    if (g_plan_free[i]->device == device) {
      Plan* pl = g_plan_free[i];
      g_plan_free.erase(g_plan_free.begin() + static_cast<std::ptrdiff_t>(i));
      return pl;
    }
  }
  return nullptr;
}

bool keep_plan(Plan* pl) {
  if (!pl->host_sum || pl->scratch_bytes() > kMaxPlanBytes) return false;
  std::lock_guard<std::mutex> lock(g_plan_mutex);
  if (g_plan_free.size() >= kMaxPlans) return false;
  try {
    g_plan_free.reserve(kMaxPlans);
  } catch (...) {
    return false;
  }
  pl->recycle();
  g_plan_free.push_back(pl);
  return true;
}

}  // namespace

struct ws_csr_s {
  int64_t nrows = 0, ncols = 0, nnz = 0;
  int64_t* rowptr = nullptr;
  int32_t* colidx = nullptr;
  void* vals = nullptr;
  ws_dtype_t dtype = WS_F64;
  int device = 0;
  Plan* plan = nullptr;
};

namespace {

int num_sms_of(int device) {
  static int cached_dev = -1, cached = 0;
  if (cached_dev != device) {
    int n = 0;
    if (cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, device) != cudaSuccess || n <= 0) n = 1;
    cached = n;
    cached_dev = device;
  }
  return cached;
}

int log2_group_for(const ws_csr_s* B) {
  const double avg = B->nrows > 0 ? static_cast<double>(B->nnz) / static_cast<double>(B->nrows) : 0.0;
  if (avg <= 4.0) return 2;
  if (avg <= 8.0) return 3;
  if (avg <= 16.0) return 4;
  return 5;
}

// A fresh status word for the next pass.
void next_status(Plan* pl) {
  pl->slot ^= 1;
  pl->host_sum->slot[pl->slot] = 0;
}

// Start of a symbolic pass whose summary block heads `buf`: a fresh status
// word, and the block cleared unless the last pass left it so.
ws_status_t begin_pass(Plan* pl, const DevBuf& buf, cudaStream_t s) {
  next_status(pl);
  const bool clean = pl->clean_buf == &buf && pl->clean_gen == buf.gen;
  pl->clean_buf = nullptr;
  if (!clean) WS_CUDA(cudaMemsetAsync(pl->dsum, 0, sizeof(DevSummary), s), "cudaMemsetAsync(summary)");
  return WS_OK;
}

// The pass ended with a scan that cleared the block.
void end_pass(Plan* pl, const DevBuf& buf) {
  pl->clean_buf = &buf;
  pl->clean_gen = buf.gen;
}

int* status_word(const Plan* pl) { return &pl->host_sum->slot[pl->slot]; }

// Waits for a summary that the stream's last kernels publish.
ws_status_t wait_summary(cudaStream_t s) {
  WS_CUDA(cudaStreamSynchronize(s), "cudaStreamSynchronize");
  return WS_OK;
}

// Status of the plan's current pass, whose queued work has completed.
ws_status_t device_status(const Plan* pl) {
  const int st = *static_cast<volatile const int*>(status_word(pl));
  if (st == 0) return WS_OK;
  return fail(WS_ERR_DEVICE, "device status 0x%x (count=%d)", st, !!(st & kErrCount));
}

template <typename T>
RowPlan<T> make_rowplan(const ws_csr_s* A, const ws_csr_s* B, ws_csr_s* C, Plan* pl) {
  RowPlan<T> p{};
  p.A = {A->rowptr, A->colidx, static_cast<const T*>(A->vals)};
  p.B = {B->rowptr, B->colidx, static_cast<const T*>(B->vals)};
  p.c_rowptr = C->rowptr;
  p.c_colidx = C->colidx;
  p.c_vals = static_cast<T*>(C->vals);
  p.perm = pl->perm;
  p.cls = pl->cls;
  p.lo = pl->lo;
  p.hi = pl->hi;
  p.slice_row = pl->slice_row;
  p.slice_idx = pl->slice_idx;
  p.slice_first = pl->slice_first;
  p.slice_cnt = pl->slice_cnt;
  p.ranks = static_cast<uint16_t*>(pl->ranks.ptr);
  p.rcd_ctr = pl->rcd_ctr;
  p.rcd_items = pl->rcd_items;
  p.rcd_bits = pl->rcd_bits;
  p.rcd_words = pl->rcd_words;
  p.rcd_width = pl->rcd_width;
  p.rcd_direct = B->ncols <= pl->rcd_width && B->nnz > kRcdLongB * B->nrows;
  p.rcd_long_b = B->nnz > 512 * B->nrows;
  p.rcd_slices = pl->rcd_slices;
  p.wb_ctr = pl->wb_ctr;
  p.wb_items = pl->wb_items;
  p.wb_bits = pl->wb_bits;
  p.wb_words = pl->wb_words;
  p.wb_cap = pl->wb_cap;
  p.wb_part = pl->wb_part;
  p.sum = pl->dsum;
  p.status = status_word(pl);
  p.log2_group = pl->log2_group;
  p.run_limit = pl->run_limit;
  p.dense_width = pl->dense_width;
  return p;
}

ws_status_t carve_rows(Plan* pl, int64_t m, cudaStream_t s) {
  const int64_t nb = scan_partials_needed(m);
  size_t off = 0;
  const size_t o_sum = off; off = align_up(off + sizeof(DevSummary), 256);
  const size_t o_perm = off; off = align_up(off + 4 * static_cast<size_t>(m), 256);
  const size_t o_lo = off; off = align_up(off + 4 * static_cast<size_t>(m), 256);
  const size_t o_hi = off; off = align_up(off + 4 * static_cast<size_t>(m), 256);
  const size_t o_long = off; off = align_up(off + 4 * static_cast<size_t>(m), 256);
  const size_t o_pend = off; off = align_up(off + 4 * static_cast<size_t>(m), 256);
  const size_t o_part = off; off = align_up(off + 8 * static_cast<size_t>(nb + 1), 256);
  const size_t o_cls = off; off = align_up(off + static_cast<size_t>(m), 256);
  ws_status_t st = pl->rows.reserve(off, s);
  if (st != WS_OK) return st;
  char* b = static_cast<char*>(pl->rows.ptr);
  pl->dsum = reinterpret_cast<DevSummary*>(b + o_sum);
  pl->perm = reinterpret_cast<int32_t*>(b + o_perm);
  pl->lo = reinterpret_cast<int32_t*>(b + o_lo);
  pl->hi = reinterpret_cast<int32_t*>(b + o_hi);
  pl->long_rows = reinterpret_cast<int32_t*>(b + o_long);
  pl->pending = reinterpret_cast<int32_t*>(b + o_pend);
  pl->partials = reinterpret_cast<int64_t*>(b + o_part);
  pl->cls = reinterpret_cast<uint8_t*>(b + o_cls);
  return WS_OK;
}

ws_status_t carve_slices(Plan* pl, int64_t nslices, cudaStream_t s) {
  const size_t n = static_cast<size_t>(nslices > 0 ? nslices : 1);
  const size_t each = align_up(4 * n, 256);
  ws_status_t st = pl->slices.reserve(4 * each, s);
  if (st != WS_OK) return st;
  char* b = static_cast<char*>(pl->slices.ptr);
  pl->slice_row = reinterpret_cast<int32_t*>(b);
  pl->slice_idx = reinterpret_cast<int32_t*>(b + each);
  pl->slice_first = reinterpret_cast<int32_t*>(b + 2 * each);
  pl->slice_cnt = reinterpret_cast<int32_t*>(b + 3 * each);
  return WS_OK;
}

// The ranks of hash bin b's products in the plan (nullptr if it has no room).
uint16_t* hash_ranks_of(const Plan* pl, int b) {
  if (!pl->hash_ranked) return nullptr;
  size_t off = 0;
  for (int i = 0; i < b; ++i) off += static_cast<size_t>(pl->seg_count[kSegHash0 + i]) << (kMinHashLog + i);
  return static_cast<uint16_t*>(pl->hranks.ptr) + off;
}

// Most memory that ranks or bitmaps of rows may take between the two passes.
// They spare the numeric pass a repetition of the symbolic one, but the caller
// still has to find room for C.  Each of the three (hash ranks, bitmaps of the
// dense and of the wide rows) takes 4 GiB at most: the ranks of 466,000 rows of
// 4096 products, or the bitmaps of 466,000 rows of 65,536 columns.
constexpr size_t kMaxKeptBytes = size_t{4} << 30;
size_t g_kept_bytes = kMaxKeptBytes;  // ws_set_tuning can lower it

// Room for the ranks of the hash rows.  They are an aid, not a need: if the
// memory is not to be had the numeric pass works them out again.
void reserve_hash_ranks(Plan* pl, cudaStream_t s) {
  size_t n = 0;
  for (int b = 0; b < kNumHashBins; ++b) n += static_cast<size_t>(pl->seg_count[kSegHash0 + b]) << (kMinHashLog + b);
  pl->hash_ranked = n > 0 && DevBuf::allocated(n * sizeof(uint16_t)) <= g_kept_bytes && pl->hranks.reserve(n * sizeof(uint16_t), s) == WS_OK;
  if (n > 0 && !pl->hash_ranked) {
    cudaGetLastError();  // the failed allocation is not an error of this call
    g_last_error.clear();
  }
}

// Room for the bitmaps and numeric items of the dense heavy rows: of all of
// them, or else of as many as can be had.  The rows are then taken in batches,
// and the numeric pass makes the bitmaps again.  The value windows are as large
// as shared memory allows, unless B's rows are long and there would be fewer
// windows than one per SM: an item is one CTA's work, and three fit an SM.  Every
// item walks all stored entries of its row, so short B rows gain from it only
// where rows are very few (fp32: 100 rows of 2800 entries times rows of 90 over 12,000
// columns 0.39 whole and 0.46 split, 40 of 6600 times rows of 10 over 5000 0.26
// and 0.28, 10 of 6600 times rows of 60 over 30,000 0.68 and 0.48).  30 rows of 2000 entries times rows of
// 1460 over 3000 columns: 0.83 ms (fp64) and 0.76 (fp32), 1.98 and 1.58 with a window
// each; 300 rows of 500 entries times rows of 460, two windows a row instead of
// one: 0.52 and 0.46 against 0.35 and 0.27.
template <typename T>
ws_status_t carve_rcd(Plan* pl, int64_t ncols, bool long_b, int sms, cudaStream_t s) {
  constexpr int64_t kMinBatch = 1024;
  constexpr int64_t kWidest = kRcdWidthBytes / sizeof(T);
  const int64_t nr = pl->seg_count[kSegRcd], span = ncols < kMaxBitmapSpan ? ncols : kMaxBitmapSpan;
  int64_t width = kWidest;
  if (long_b && nr * ((span + kWidest - 1) / kWidest) < sms) width = align_up(static_cast<size_t>(span * nr / (3 * sms) + 1), kRcdLeastWidth);
  pl->rcd_width = static_cast<int>(width < kWidest ? width : kWidest);
  pl->rcd_slices = static_cast<int>((span + pl->rcd_width - 1) / pl->rcd_width);
  pl->rcd_words = static_cast<int>(align_up((span + 31) / 32, 4));
  const size_t row_bytes = static_cast<size_t>(pl->rcd_words) * 4;
  const int64_t fit = static_cast<int64_t>(g_kept_bytes / DevBuf::allocated(row_bytes)), most = fit > kMinBatch ? fit : kMinBatch;
  const size_t o_items = align_up(4 * kRcdCounters, 256);
  for (int64_t n = nr < most ? nr : most;; n = n / 2 < kMinBatch ? kMinBatch : n / 2) {
    const size_t o_bits = align_up(o_items + 8 * static_cast<size_t>(n) * pl->rcd_slices, 256);
    ws_status_t st = pl->rcd.reserve(o_bits + static_cast<size_t>(n) * pl->rcd_words * 4, s);
    if (st == WS_OK) {
      char* b = static_cast<char*>(pl->rcd.ptr);
      pl->rcd_ctr = reinterpret_cast<int32_t*>(b);
      pl->rcd_items = reinterpret_cast<long long*>(b + o_items);
      pl->rcd_bits = reinterpret_cast<uint32_t*>(b + o_bits);
      pl->rcd_batch = n;
      return WS_OK;
    }
    if (st != WS_ERR_ALLOC || n <= kMinBatch) return st;
    cudaGetLastError();  // the failed allocation is not an error of this call
    g_last_error.clear();
  }
}

// Room for the numeric items of the wide-bitmap rows and, if it can be had,
// for their bitmaps.  A row of several items has its bitmap read and ranked
// once per item, so the items are larger when there are rows, or products,
// enough to keep the GPU busy.  Rows of 300 entries times rows of 60 over 10^6
// columns, fp64, cut into items of 16,384 products and whole: 2000 rows 0.94 and
// 0.74 ms, 400 rows 0.28 and 0.23, 60 rows 0.12 and 0.13; 400 rows of 2000 entries
// 0.98 in eight items each, 0.83 in two, 1.07 whole.
ws_status_t carve_wb(Plan* pl, int64_t ncols, int sms, cudaStream_t s) {
  const int64_t nr = pl->seg_count[kSegWb];
  pl->wb_words = static_cast<int>(align_up(((ncols < kWbMaxSpan ? ncols : kWbMaxSpan) + 31) / 32, 4));
  const int64_t least = nr >= 2 * sms ? 2 * kWbPart : kWbPart, fair = pl->wb_products / (4 * sms);
  pl->wb_part = fair > least ? fair : least;
  pl->wb_cap = nr + pl->wb_products / pl->wb_part;
  const size_t o_items = align_up(4 * kWbCounters, 256);
  const size_t o_bits = align_up(o_items + 8 * static_cast<size_t>(pl->wb_cap), 256);
  const size_t bits = static_cast<size_t>(nr) * pl->wb_words * 4;
  bool kept = DevBuf::allocated(bits) <= g_kept_bytes && pl->wb.reserve(o_bits + bits, s) == WS_OK;
  if (!kept) {
    cudaGetLastError();  // the failed allocation is not an error of this call
    g_last_error.clear();
    ws_status_t st = pl->wb.reserve(o_bits, s);
    if (st != WS_OK) return st;
  }
  char* b = static_cast<char*>(pl->wb.ptr);
  pl->wb_ctr = reinterpret_cast<int32_t*>(b);
  pl->wb_items = reinterpret_cast<long long*>(b + o_items);
  pl->wb_bits = kept ? reinterpret_cast<uint32_t*>(b + o_bits) : nullptr;
  WS_CUDA(cudaMemsetAsync(pl->wb_ctr, 0, kWbCounters * sizeof(int32_t), s), "cudaMemsetAsync(wide row counters)");
  return WS_OK;
}

// A pass over the dense heavy rows, on stream s.
template <typename T>
ws_status_t run_rcd(Plan* pl, RowPlan<T> p, bool numeric, int sms, cudaStream_t s, int* launches) {
  const int64_t begin = pl->seg_offset[kSegRcd], nr = pl->seg_count[kSegRcd];
  const bool whole = pl->rcd_batch >= nr;
  for (int64_t r = 0; r < nr; r += pl->rcd_batch) {
    p.seg_begin = begin + r;
    p.seg_len = nr - r < pl->rcd_batch ? nr - r : pl->rcd_batch;
    if (!numeric || !whole) {
      p.rcd_again = numeric;
      WS_CUDA(cudaMemsetAsync(pl->rcd_ctr, 0, kRcdCounters * sizeof(int32_t), s), "cudaMemsetAsync(rcd counters)");
      launch_rcd<T>(p, false, sms, s, launches);
    } else {
      WS_CUDA(cudaMemsetAsync(pl->rcd_ctr + kRcdNextItem, 0, sizeof(int32_t), s), "cudaMemsetAsync(rcd work counter)");
    }
    if (numeric) launch_rcd<T>(p, true, sms, s, launches);
  }
  return WS_OK;
}

// Segments whose kernels run by themselves, ahead of the side streams: the
// bitmap bin of 512 entries over 65,536 columns when its rows fill the GPU
// several times over.  Its CTAs take most of an SM's shared memory, and next
// to CTAs that want the memory as L1 cache both run at a fraction of their
// occupancy.  Rows of 0-10 entries times rows of 0-80 over 32,000 columns (24
// million products, fp32): 0.70 ms, 0.97 overlapped, 0.77 without side streams.
// Other bins gained nothing or lost by it (rows of 0-80 entries times rows of 0-40
// over 1000 columns, in the bin of 1024 entries: 1.04 against 0.99), and with few
// rows the overlap is worth more (R-MAT 2^14: 0.58 without, 0.40 with).
constexpr int64_t kAloneRows = 16384;
bool runs_alone(const Plan* pl, int g) { return g == kSegBitmap0 + 2 && pl->seg_count[g] > kAloneRows; }

// Row kernels of a pass next to them (the symbolic pass has none for direct
// and planned rows).
int bin_launches(const Plan* pl, bool numeric) {
  int n = 0;
  for (int g = 0; g < kNumSegs; ++g)
    n += pl->seg_count[g] > 0 && (numeric || (g != kSegDirect && g != kSegBmrWide)) && !runs_alone(pl, g);
  return n;
}

template <typename T>
void launch_alone(const Plan* pl, RowPlan<T> p, bool numeric, int sms, cudaStream_t s, int* launches) {
  for (int b = 0; b < kNumBitmapBins; ++b) {
    const int g = kSegBitmap0 + b;
    if (!runs_alone(pl, g)) continue;
    p.seg_begin = pl->seg_offset[g];
    p.seg_len = pl->seg_count[g];
    launch_bitmap<T>(p, b, numeric, sms, s, launches);
  }
}

// Second half of the symbolic pass when some rows were not ranked by the
// planning pass: group the rows by segment, run the per-bin symbolic kernels,
// scan the counts into C's row pointer and read the summary back.
template <typename T>
ws_status_t symbolic_bins(const ws_csr_s* A, const ws_csr_s* B, ws_csr_s* C, Plan* pl, RowPlan<T> p, int64_t off,
                          int sms, cudaStream_t s) {
  const int64_t m = A->nrows;
  ws_status_t st = WS_OK;
  if (off > 0) {
    launch_scatter<T>(p, m, pl->seg_offset, sms, s, &pl->sym_launches);
  }
  // All scratch and counters first, on the caller's stream.
  int64_t bmr_rows = 0;
  for (int b = 0; b < kNumBmrBins; ++b) bmr_rows += pl->seg_count[kSegBmr0 + b];
  if (bmr_rows > 0) {
    st = pl->ranks.reserve(static_cast<size_t>(m) * kBmrSlots * sizeof(uint16_t), s);
    if (st != WS_OK) return st;
  }
  if (pl->seg_count[kSegDense] > 0) {
    st = carve_slices(pl, pl->dense_slices, s);
    if (st != WS_OK) return st;
  }
  if (pl->seg_count[kSegRcd] > 0) {
    st = carve_rcd<T>(pl, B->ncols, B->nnz > kRcdLongB * B->nrows, sms, s);
    if (st != WS_OK) return st;
  }
  if (pl->seg_count[kSegWb] > 0) {
    st = carve_wb(pl, B->ncols, sms, s);
    if (st != WS_OK) return st;
  }
  reserve_hash_ranks(pl, s);
  p = make_rowplan<T>(A, B, C, pl);
  launch_alone<T>(pl, p, false, sms, s, &pl->sym_launches);
  Fork fork(s, C->device, bin_launches(pl, false));
  auto segment = [&](int g) {
    p.seg_begin = pl->seg_offset[g];
    p.seg_len = pl->seg_count[g];
    return p.seg_len > 0;
  };
  if (segment(kSegRcd)) {
    st = run_rcd<T>(pl, p, false, sms, fork.next(), &pl->sym_launches);
    if (st != WS_OK) return st;
  }
  if (segment(kSegWb)) launch_wb<T>(p, false, sms, fork.next(), &pl->sym_launches);
  if (segment(kSegDense)) {
    const cudaStream_t q = fork.next();
    launch_dense_slices<T>(p, pl->slice_row, pl->slice_idx, pl->slice_first, sms, q, &pl->sym_launches);
    launch_dense<T>(p, pl->dense_slices, false, sms, q, &pl->sym_launches);
  }
  for (int b = kNumHashBins - 1; b >= 0; --b) {
    p.hash_ranks = hash_ranks_of(pl, b);
    if (segment(kSegHash0 + b)) launch_hash<T>(p, b, false, sms, fork.next(), &pl->sym_launches);
  }
  for (int b = kNumBitmapBins - 1; b >= 0; --b) {
    if (segment(kSegBitmap0 + b) && !runs_alone(pl, kSegBitmap0 + b)) launch_bitmap<T>(p, b, false, sms, fork.next(), &pl->sym_launches);
  }
  for (int b = kNumBmrBins - 1; b >= 0; --b) {
    if (segment(kSegBmr0 + b)) launch_bmr<T>(p, b, false, sms, fork.next(), &pl->sym_launches);
  }
  WS_CUDA(fork.join(), "joining the side streams");
  launch_scan(C->rowptr, m, pl->partials, pl->dsum, s, &pl->sym_launches, nullptr, pl->host_sum);
  WS_CUDA(cudaGetLastError(), "symbolic launches");
  return wait_summary(s);
}

template <typename T>
ws_status_t symbolic_impl(const ws_csr_s* A, const ws_csr_s* B, ws_csr_s* C, Plan* pl, cudaStream_t s,
                          int64_t* nnz_out) {
  const int64_t m = A->nrows;
  const int dev = C->device;
  const int sms = num_sms_of(dev);
  pl->ready = false;
  pl->kind = kPlanSpgemm;
  pl->sym_launches = 0;
  pl->num_launches = 0;
  pl->log2_group = log2_group_for(B);
  pl->run_limit = g_run_limit;
  pl->dense_width = g_dense_width > 0 ? g_dense_width : (sizeof(T) == 8 ? 8192 : 16384);

  ws_status_t st = carve_rows(pl, m, s);
  if (st != WS_OK) return st;
  st = begin_pass(pl, pl->rows, s);
  if (st != WS_OK) return st;

  RowPlan<T> p = make_rowplan<T>(A, B, C, pl);
  if (m == 0) {
    WS_CUDA(cudaMemsetAsync(C->rowptr, 0, sizeof(int64_t), s), "cudaMemsetAsync(rowptr[0])");
    static_cast<DevSummary&>(*pl->host_sum) = DevSummary{};
  } else {
    AnalyzeParams ap{m,           g_hash_max, g_bitmap_span,   1 << pl->log2_group, g_bmr_max_a,
                     g_rcd_max_a, g_wb_span,  pl->dense_width, kLongRowThreshold,   A->nnz};
    // When every row of C fits the widest register bitmap (B has at most
    // 65,536 columns), the planning pass counts the eligible rows in its first
    // read of A and only the remaining rows go through the analysis kernel.
    // It is left out when the average row of A has more entries than it takes,
    // or fewer products than it takes for that many columns: reading A for the
    // few rows that differ took longer (100,000 rows of 20 entries times rows
    // of 6 over 16,000 columns: 0.39 ms with it, 0.31 without).
    const double avg_a = static_cast<double>(A->nnz) / static_cast<double>(m);
    const double avg_products = avg_a * static_cast<double>(B->nnz) / static_cast<double>(B->nrows > 0 ? B->nrows : 1);
    const bool plan_pass = g_bmr_max_a > 0 && B->ncols > 0 && B->ncols <= kMaxBitmapSpan && g_bitmap_span >= B->ncols &&
                           avg_a <= kBmrMaxA &&
                           static_cast<double>((B->ncols + 31) / 32) <= kPlanWordsPerProduct * avg_products + 64;
    if (plan_pass) {
      st = pl->ranks.reserve(static_cast<size_t>(m) * kBmrSlots * sizeof(uint16_t), s);
      if (st != WS_OK) return st;
      p.ranks = static_cast<uint16_t*>(pl->ranks.ptr);
      launch_bmr_plan<T>(p, ap, B->ncols, pl->pending, sms, s, &pl->sym_launches);
      launch_analyze<T>(p, ap, pl->long_rows, pl->pending, nullptr, sms, s, &pl->sym_launches);
      // If the planning pass took every row, all counts are in place now: a
      // scan queued here (a no-op otherwise) saves the second read-back.
      launch_scan(C->rowptr, m, pl->partials, pl->dsum, s, &pl->sym_launches, &pl->dsum->n_pending, pl->host_sum);
    } else {
      launch_analyze<T>(p, ap, pl->long_rows, nullptr, pl->host_sum, sms, s, &pl->sym_launches);
    }
    WS_CUDA(cudaGetLastError(), "analyze launch");
  }
  st = wait_summary(s);
  if (st != WS_OK) return st;
  const DevSummary& hs = *pl->host_sum;
  int64_t off = 0;
  for (int g = 0; g < kNumSegs; ++g) {
    pl->seg_count[g] = hs.seg_count[g];
    pl->seg_offset[g] = off;
    off += hs.seg_count[g];
  }
  pl->seg_offset[kNumSegs] = off;
  pl->n_empty = hs.n_empty;
  pl->products = hs.products;
  pl->dense_slices = hs.dense_slices;
  pl->wb_products = hs.wb_products;
  if (pl->dense_slices > INT32_MAX) return fail(WS_ERR_OVERFLOW, "too many dense-window slices (%lld)", (long long)pl->dense_slices);
  pl->all_planned = m > 0 && hs.n_pending == 0 && pl->seg_count[kSegBmrWide] == m;
  if (m > 0 && !pl->all_planned) {
    st = symbolic_bins<T>(A, B, C, pl, p, off, sms, s);
    if (st != WS_OK) return st;
  }
  if (m > 0) end_pass(pl, pl->rows);
  st = device_status(pl);
  if (st != WS_OK) return st;
  pl->n_sort = pl->host_sum->n_sort;
  C->nnz = m > 0 ? pl->host_sum->nnz : 0;
  pl->A = A;
  pl->B = B;
  pl->a_nnz = A->nnz;
  pl->b_nnz = B->nnz;
  pl->ready = true;
  *nnz_out = C->nnz;
  return WS_OK;
}

template <typename T>
ws_status_t numeric_impl(const ws_csr_s* A, const ws_csr_s* B, ws_csr_s* C, Plan* pl, cudaStream_t s) {
  const int sms = num_sms_of(C->device);
  pl->num_launches = 0;
  RowPlan<T> p = make_rowplan<T>(A, B, C, pl);
  if (pl->seg_count[kSegWb] > 0)
    WS_CUDA(cudaMemsetAsync(pl->wb_ctr + kWbNextItem, 0, sizeof(int32_t), s), "cudaMemsetAsync(wide row counter)");
  launch_alone<T>(pl, p, true, sms, s, &pl->num_launches);
  Fork fork(s, C->device, bin_launches(pl, true));
  auto segment = [&](int g) {
    p.seg_begin = pl->seg_offset[g];
    p.seg_len = pl->seg_count[g];
    return p.seg_len > 0;
  };
  if (segment(kSegRcd)) {
    const ws_status_t st = run_rcd<T>(pl, p, true, sms, fork.next(), &pl->num_launches);
    if (st != WS_OK) return st;
  }
  if (segment(kSegWb)) launch_wb<T>(p, true, sms, fork.next(), &pl->num_launches);
  if (segment(kSegDense)) launch_dense<T>(p, pl->dense_slices, true, sms, fork.next(), &pl->num_launches);
  if (segment(kSegBmrWide)) {
    if (pl->all_planned) p.perm = nullptr;  // rows in order, no permutation was built
    launch_bmr<T>(p, kBmrPlannedBin, true, sms, fork.next(), &pl->num_launches);
    p.perm = pl->perm;
  }
  for (int b = kNumHashBins - 1; b >= 0; --b) {
    p.hash_ranks = hash_ranks_of(pl, b);
    if (segment(kSegHash0 + b)) launch_hash<T>(p, b, true, sms, fork.next(), &pl->num_launches);
  }
  for (int b = kNumBitmapBins - 1; b >= 0; --b) {
    if (segment(kSegBitmap0 + b) && !runs_alone(pl, kSegBitmap0 + b)) launch_bitmap<T>(p, b, true, sms, fork.next(), &pl->num_launches);
  }
  for (int b = kNumBmrBins - 1; b >= 0; --b) {
    if (segment(kSegBmr0 + b)) launch_bmr<T>(p, b, true, sms, fork.next(), &pl->num_launches);
  }
  if (segment(kSegDirect)) launch_direct<T>(p, sms, fork.next(), &pl->num_launches);
  WS_CUDA(fork.join(), "joining the side streams");
  WS_CUDA(cudaGetLastError(), "numeric launches");
  return WS_OK;
}

// ----------------------------------------------------- elementwise operations

ws_status_t carve_ewise(Plan* pl, int64_t ntiles, cudaStream_t s) {
  const size_t n = static_cast<size_t>(ntiles) + 1;
  size_t off = 0;
  const size_t o_sum = off; off = align_up(off + sizeof(DevSummary), 256);
  const size_t o_row = off; off = align_up(off + 4 * n, 256);
  const size_t o_a = off; off = align_up(off + 8 * n, 256);
  const size_t o_b = off; off = align_up(off + 8 * n, 256);
  const size_t o_off = off; off = align_up(off + 8 * n, 256);
  const size_t o_part = off; off = align_up(off + 8 * static_cast<size_t>(scan_partials_needed(ntiles) + 1), 256);
  ws_status_t st = pl->ew.reserve(off, s);
  if (st != WS_OK) return st;
  char* b = static_cast<char*>(pl->ew.ptr);
  pl->dsum = reinterpret_cast<DevSummary*>(b + o_sum);
  pl->ew_tile_row = reinterpret_cast<int32_t*>(b + o_row);
  pl->ew_tile_a = reinterpret_cast<int64_t*>(b + o_a);
  pl->ew_tile_b = reinterpret_cast<int64_t*>(b + o_b);
  pl->ew_tile_off = reinterpret_cast<int64_t*>(b + o_off);
  pl->ew_partials = reinterpret_cast<int64_t*>(b + o_part);
  return WS_OK;
}

template <typename T>
EwisePlan<T> make_ewise(const ws_csr_s* A, const ws_csr_s* B, ws_csr_s* C, const Plan* pl) {
  EwisePlan<T> p{};
  p.A = {A->rowptr, A->colidx, static_cast<const T*>(A->vals)};
  p.B = {B->rowptr, B->colidx, static_cast<const T*>(B->vals)};
  p.m = A->nrows;
  p.c_rowptr = C->rowptr;
  p.c_colidx = C->colidx;
  p.c_vals = static_cast<T*>(C->vals);
  p.ntiles = pl->ew_ntiles;
  p.tile_row = pl->ew_tile_row;
  p.tile_a = pl->ew_tile_a;
  p.tile_b = pl->ew_tile_b;
  p.tile_off = pl->ew_tile_off;
  p.partials = pl->ew_partials;
  p.sum = pl->dsum;
  p.status = status_word(pl);
  p.host = pl->host_sum;
  p.op = pl->ew_op;
  return p;
}

template <typename T>
ws_status_t ewise_symbolic_impl(const ws_csr_s* A, const ws_csr_s* B, ws_csr_s* C, Plan* pl, int op,
                                cudaStream_t s, int64_t* nnz_out) {
  const int64_t m = A->nrows;
  pl->ready = false;
  pl->kind = kPlanEwise;
  pl->sym_launches = 0;
  pl->num_launches = 0;
  pl->ew_op = op;
  const int64_t merged = A->nnz + B->nnz;
  pl->ew_ntiles = (merged + m + kEwTileItems - 1) / kEwTileItems;
  ws_status_t st = carve_ewise(pl, pl->ew_ntiles, s);
  if (st != WS_OK) return st;
  next_status(pl);  // the summary block only takes the scan's total: it need not be cleared
  pl->clean_buf = nullptr;
  if (m > 0) {
    launch_ewise_symbolic<T>(make_ewise<T>(A, B, C, pl), num_sms_of(C->device), s, &pl->sym_launches);
    WS_CUDA(cudaGetLastError(), "elementwise symbolic launches");
  } else {
    WS_CUDA(cudaMemsetAsync(C->rowptr, 0, sizeof(int64_t), s), "cudaMemsetAsync(rowptr[0])");
  }
  st = wait_summary(s);
  if (st != WS_OK) return st;
  st = device_status(pl);
  if (st != WS_OK) return st;
  C->nnz = m > 0 ? pl->host_sum->nnz : 0;
  pl->products = merged;
  pl->A = A;
  pl->B = B;
  pl->a_nnz = A->nnz;
  pl->b_nnz = B->nnz;
  pl->ready = true;
  *nnz_out = C->nnz;
  return WS_OK;
}

// ------------------------------------------ sparse matrix - sparse vector

// Creates a handle's plan and its pinned summary if missing.
ws_status_t ensure_plan(ws_csr_s* h) {
  if (!h->plan) h->plan = recycled_plan(h->device);
  if (!h->plan) {
    h->plan = new (std::nothrow) Plan;
    if (!h->plan) return fail(WS_ERR_ALLOC, "host allocation failed");
    h->plan->device = h->device;
  }
  if (!h->plan->host_sum) {
    keep_pool_memory(h->device);
    h->plan->host_sum = acquire_host_sum();
    if (!h->plan->host_sum) return fail(WS_ERR_ALLOC, "cudaMallocHost failed");
  }
  return WS_OK;
}

template <typename T>
ws_status_t spmspv_impl(ws_csr_s* At, int64_t nx, const int32_t* x_idx, const void* x_vals, int32_t* y_idx,
                        void* y_vals, int64_t* nnz_y, cudaStream_t s) {
  Plan* pl = At->plan;
  const int64_t m = At->ncols, n = At->nrows;
  const int64_t tiles = spmspv_tiles(m);
  const int64_t mark_bytes = tiles * 4096;  // the byte-map, padded to whole compaction tiles
  const int64_t nb = scan_partials_needed(nx > tiles ? nx : tiles);
  size_t off = 0;
  const size_t o_sum = off; off = align_up(off + sizeof(DevSummary), 256);
  const size_t o_acc = off; off = align_up(off + sizeof(T) * static_cast<size_t>(m), 256);  // whole 16-byte words
  const size_t o_mark = off; off = align_up(off + static_cast<size_t>(mark_bytes), 256);
  const size_t o_off = off; off = align_up(off + 8 * static_cast<size_t>(nx + 1), 256);
  const size_t o_first = off; off = align_up(off + 8 * static_cast<size_t>(nx), 256);
  const size_t o_cnt = off; off = align_up(off + 8 * static_cast<size_t>(tiles + 1), 256);
  const size_t o_part = off; off = align_up(off + 8 * static_cast<size_t>(nb + 1), 256);
  ws_status_t st = pl->sv.reserve(off, s);
  if (st != WS_OK) return st;
  char* b = static_cast<char*>(pl->sv.ptr);
  SpmspvPlan<T> p{};
  p.At = {At->rowptr, At->colidx, static_cast<const T*>(At->vals)};
  p.n = n;
  p.m = m;
  p.nnz_a = At->nnz;
  p.nx = nx;
  p.x_idx = x_idx;
  p.x_vals = static_cast<const T*>(x_vals);
  p.sum = reinterpret_cast<DevSummary*>(b + o_sum);
  p.acc = reinterpret_cast<T*>(b + o_acc);
  p.mark = reinterpret_cast<uint8_t*>(b + o_mark);
  p.off = reinterpret_cast<int64_t*>(b + o_off);
  p.first = reinterpret_cast<int64_t*>(b + o_first);
  p.cnt = reinterpret_cast<int64_t*>(b + o_cnt);
  p.partials = reinterpret_cast<int64_t*>(b + o_part);
  p.y_idx = y_idx;
  p.y_vals = static_cast<T*>(y_vals);
  p.cap = m;
  pl->dsum = p.sum;
  next_status(pl);
  p.status = status_word(pl);
  p.host = pl->host_sum;
  pl->sym_launches = 0;
  pl->num_launches = 0;
  // the summary block only takes the scans' totals: it need not be cleared
  if (m > 0) {
    launch_spmspv<T>(p, num_sms_of(At->device), s, &pl->num_launches);
    WS_CUDA(cudaGetLastError(), "spmspv launches");
  }
  st = wait_summary(s);
  if (st != WS_OK) return st;
  st = device_status(pl);
  if (st != WS_OK) return st;
  *nnz_y = m > 0 ? pl->host_sum->nnz : 0;
  return WS_OK;
}

// Shared checks of the operand and output handles; creates C's plan.
ws_status_t prepare_output(const ws_csr_s* A, const ws_csr_s* B, ws_csr_s* C) {
  if (C == A || C == B) return fail(WS_ERR_INVALID_ARG, "C must be a separate output handle");
  if (A->dtype != B->dtype || C->dtype != A->dtype) return fail(WS_ERR_DTYPE, "A, B and C dtypes differ");
  return ensure_plan(C);
}

ws_status_t check_handle(const ws_csr_s* h, const char* name) {
  if (!h) return fail(WS_ERR_INVALID_ARG, "%s is NULL", name);
  return WS_OK;
}

// ------------------------------------------------------ outer-product SpGEMM
//
// C = A*B with the k loop split over P workers (Sec. 5.1, Fig. "SpGEMM
// implemented in WingSpan", outer product): worker p multiplies the column
// block A[:, K_p] by the row block B[K_p, :] into its own copy of C, and a
// merge level coalesces the copies (Sec. 4, coalesce).  On one GPU every
// block's product already fills the device, so the blocks run one after
// another on the caller's stream:
//   - B[K_p, :] is a view of B's rows (no copy);
//   - A[:, K_p] is extracted (count, scan, copy) into one library buffer of
//     nnz(A) entries that every block reuses, so its size needs no read-back;
//   - the partial product is the row-wise product of the two blocks;
//   - the partial products are merged pairwise by sparse additions (a sum of
//     exactly 0.0 is kept, so C's structure equals the row-wise product's).
// The symbolic call runs everything but the value pass of the last merge,
// whose structure pass writes C.rowptr; the numeric call runs that value pass.

// A CSR matrix whose arrays the library owns (stream-ordered allocations).
struct Owned {
  ws_csr_s h;
  void* rp_mem = nullptr;  // row pointer
  void* cv_mem = nullptr;  // column indices and values
};

struct OuterState {
  int parts = 1;
  const ws_csr_s* A = nullptr;
  const ws_csr_s* B = nullptr;
  int64_t a_nnz = 0, b_nnz = 0;
  Owned* x = nullptr;  // operands of the last merge (parts >= 2)
  Owned* y = nullptr;
};

// Frees a plan's scratch stream-ordered on s (no device synchronisation).
void release_plan_async(Plan* pl, cudaStream_t s);

void release_owned(Owned* o, cudaStream_t s) {
  if (!o) return;
  release_plan_async(o->h.plan, s);
  o->h.plan = nullptr;
  if (o->rp_mem) cudaFreeAsync(o->rp_mem, s);
  if (o->cv_mem) cudaFreeAsync(o->cv_mem, s);
  delete o;
}

void release_outer(Plan* pl, cudaStream_t s) {
  if (!pl || !pl->outer) return;
  release_owned(pl->outer->x, s);
  release_owned(pl->outer->y, s);
  delete pl->outer;
  pl->outer = nullptr;
}

// The scratch of `from`, whose last pass is queued on a stream, for passes of
// `to` on the same stream (and the scratch of `to`, if it has some, for `from`).
// So the blocks of an outer product use the scratch of one.  Freeing it after
// every block instead left the stream-ordered pool with other free ranges than
// the next partial product and merge ask for, and a product of 65,539 rows
// of 16 entries times rows of 32 in four blocks took 2.71 instead of 2.06 ms.
void hand_over_scratch(Plan* from, Plan* to) {
  DevBuf* a[] = {&from->rows, &from->slices, &from->ranks, &from->ew, &from->sv, &from->hranks, &from->rcd, &from->wb};
  DevBuf* b[] = {&to->rows, &to->slices, &to->ranks, &to->ew, &to->sv, &to->hranks, &to->rcd, &to->wb};
  for (size_t i = 0; i < sizeof(a) / sizeof(a[0]); ++i) std::swap(*a[i], *b[i]);
  // a summary block that the last pass left cleared goes with its buffer
  to->clean_buf = from->clean_buf == &from->rows ? &to->rows : nullptr;
  to->clean_gen = from->clean_gen;
  from->clean_buf = nullptr;
  from->ready = false;
}

void release_plan_async(Plan* pl, cudaStream_t s) {
  if (!pl) return;
  release_outer(pl, s);
  DevBuf* bufs[] = {&pl->rows, &pl->slices, &pl->ranks, &pl->ew, &pl->sv, &pl->hranks, &pl->rcd, &pl->wb};
  for (DevBuf* b : bufs) {
    if (b->ptr) cudaFreeAsync(b->ptr, s);
    b->ptr = nullptr;
    b->bytes = 0;
  }
  release_host_sum(pl->host_sum);
  delete pl;
}

// An owned m x n matrix with its row pointer allocated; entries come later.
ws_status_t new_owned(int64_t m, int64_t n, ws_dtype_t dt, int dev, cudaStream_t s, Owned** out) {
  *out = nullptr;
  Owned* o = new (std::nothrow) Owned;
  if (!o) return fail(WS_ERR_ALLOC, "host allocation failed");
  o->h.nrows = m;
  o->h.ncols = n;
  o->h.nnz = 0;
  o->h.dtype = dt;
  o->h.device = dev;
  const cudaError_t e = cudaMallocAsync(&o->rp_mem, 8 * static_cast<size_t>(m + 1), s);
  if (e != cudaSuccess) {
    delete o;
    return fail(WS_ERR_ALLOC, "cudaMallocAsync(row pointer): %s", cudaGetErrorString(e));
  }
  o->h.rowptr = static_cast<int64_t*>(o->rp_mem);
  ws_status_t st = ensure_plan(&o->h);
  if (st != WS_OK) {
    release_owned(o, s);
    return st;
  }
  *out = o;
  return WS_OK;
}

// Room for cap entries (column indices and values) of an owned matrix.
ws_status_t owned_entries(Owned* o, int64_t cap, cudaStream_t s) {
  const size_t vs = o->h.dtype == WS_F64 ? 8 : 4;
  const size_t o_val = align_up(4 * static_cast<size_t>(cap > 0 ? cap : 1), 256);
  const cudaError_t e = cudaMallocAsync(&o->cv_mem, o_val + vs * static_cast<size_t>(cap > 0 ? cap : 1), s);
  if (e != cudaSuccess) return fail(WS_ERR_ALLOC, "cudaMallocAsync(%lld entries): %s", (long long)cap, cudaGetErrorString(e));
  o->h.colidx = static_cast<int32_t*>(o->cv_mem);
  o->h.vals = static_cast<char*>(o->cv_mem) + o_val;
  return WS_OK;
}

// Status of a partial product or merge whose queued work has completed.
ws_status_t plan_status(const Plan* pl) {
  const int st = *static_cast<volatile const int*>(status_word(pl));
  if (st != 0) return fail(WS_ERR_DEVICE, "device status 0x%x in an outer-product step", st);
  return WS_OK;
}

template <typename T>
ws_status_t outer_symbolic_impl(const ws_csr_s* A, const ws_csr_s* B, ws_csr_s* C, int parts, cudaStream_t s,
                                int64_t* nnz_out) {
  Plan* pl = C->plan;
  release_outer(pl, s);
  const int64_t m = A->nrows, K = A->ncols, n = B->ncols;
  const int P = static_cast<int>(parts < 1 ? 1 : (parts > K ? (K > 0 ? K : 1) : parts));
  OuterState* os = new (std::nothrow) OuterState;
  if (!os) return fail(WS_ERR_ALLOC, "host allocation failed");
  os->parts = P;
  os->A = A;
  os->B = B;
  os->a_nnz = A->nnz;
  os->b_nnz = B->nnz;
  if (P == 1) {  // one block: the row-wise product itself
    ws_status_t st = symbolic_impl<T>(A, B, C, pl, s, nnz_out);
    if (st != WS_OK) {
      delete os;
      return st;
    }
    pl->outer = os;
    return WS_OK;
  }
  const int sms = num_sms_of(C->device);
  int launches = 0;
  std::vector<Owned*> partial;
  Owned* ab = nullptr;  // the current column block of A
  void* ex_mem = nullptr;  // the extraction's summary and scan partials
  ws_status_t st = WS_OK;
  auto cleanup = [&]() {
    // Queued kernels may still write to the status words that the plans give
    // back to the pool here.
    if (cudaStreamSynchronize(s) != cudaSuccess) cudaGetLastError();
    for (Owned* o : partial) release_owned(o, s);
    release_owned(ab, s);
    if (ex_mem) cudaFreeAsync(ex_mem, s);
    delete os;
  };
  const size_t o_part = align_up(sizeof(DevSummary), 256);
  cudaError_t e = cudaMallocAsync(&ex_mem, o_part + 8 * static_cast<size_t>(scan_partials_needed(m) + 1), s);
  if (e != cudaSuccess) {
    ex_mem = nullptr;
    cleanup();
    return fail(WS_ERR_ALLOC, "cudaMallocAsync(extraction scratch): %s", cudaGetErrorString(e));
  }
  DevSummary* ex_sum = static_cast<DevSummary*>(ex_mem);
  int64_t* ex_part = reinterpret_cast<int64_t*>(static_cast<char*>(ex_mem) + o_part);
  if ((st = new_owned(m, 1, A->dtype, C->device, s, &ab)) != WS_OK || (st = owned_entries(ab, A->nnz, s)) != WS_OK) {
    cleanup();
    return st;
  }
  for (int p = 0; p < P && st == WS_OK; ++p) {
    const int64_t k0 = K * p / P, k1 = K * (p + 1) / P;
    // A[:, k0:k1], columns shifted by -k0
    ab->h.ncols = k1 - k0;
    if (m == 0 && cudaMemsetAsync(ab->h.rowptr, 0, sizeof(int64_t), s) != cudaSuccess) {
      st = fail(WS_ERR_CUDA, "cudaMemsetAsync(block row pointer)");
      break;
    }
    if (m > 0) {
      launch_submatrix_count(A->rowptr, A->colidx, 0, m, k0, k1, ab->h.rowptr, sms, s, &launches);
      launch_scan(ab->h.rowptr, m, ex_part, ex_sum, s, &launches);
      launch_submatrix_copy<T>(A->rowptr, A->colidx, static_cast<const T*>(A->vals), 0, m, k0, ab->h.rowptr,
                               ab->h.colidx, static_cast<T*>(ab->h.vals), status_word(ab->h.plan), sms, s, &launches);
    }
    // B[k0:k1, :]: a view of B's rows (positions stay absolute in B's arrays)
    ws_csr_s bp = *B;
    bp.plan = nullptr;
    bp.nrows = k1 - k0;
    bp.rowptr = B->rowptr + k0;
    // estimates: only the choice of lane groups, of the planning pass and of grid sizes reads them
    bp.nnz = K > 0 ? B->nnz * (k1 - k0) / K : 0;
    ab->h.nnz = K > 0 ? A->nnz * (k1 - k0) / K : 0;
    // the worker's partial product
    Owned* cp = nullptr;
    if ((st = new_owned(m, n, A->dtype, C->device, s, &cp)) != WS_OK) break;
    partial.push_back(cp);
    if (partial.size() > 1) hand_over_scratch(partial[partial.size() - 2]->h.plan, cp->h.plan);
    int64_t nnz_p = 0;
    if ((st = symbolic_impl<T>(&ab->h, &bp, &cp->h, cp->h.plan, s, &nnz_p)) != WS_OK) break;
    cp->h.nnz = nnz_p;
    if ((st = owned_entries(cp, nnz_p, s)) != WS_OK) break;
    if ((st = numeric_impl<T>(&ab->h, &bp, &cp->h, cp->h.plan, s)) != WS_OK) break;
    launches += cp->h.plan->sym_launches + cp->h.plan->num_launches;
  }
  // every extraction has completed (each block's structure pass synchronised)
  if (st == WS_OK) st = plan_status(ab->h.plan);
  release_owned(ab, s);
  ab = nullptr;
  // merge levels: pairwise sparse additions until two copies are left
  while (st == WS_OK && partial.size() > 2) {
    std::vector<Owned*> next;
    size_t i = 0;
    for (; i + 1 < partial.size() && st == WS_OK; i += 2) {
      Owned* x = partial[i];
      Owned* y = partial[i + 1];
      Owned* z = nullptr;
      if ((st = new_owned(m, n, A->dtype, C->device, s, &z)) != WS_OK) break;
      next.push_back(z);
      int64_t nz = 0;
      if ((st = ewise_symbolic_impl<T>(&x->h, &y->h, &z->h, z->h.plan, kEwiseAdd, s, &nz)) != WS_OK) break;
      if ((st = plan_status(x->h.plan)) != WS_OK || (st = plan_status(y->h.plan)) != WS_OK) break;
      z->h.nnz = nz;
      if ((st = owned_entries(z, nz, s)) != WS_OK) break;
      if (nz > 0) launch_ewise_numeric<T>(make_ewise<T>(&x->h, &y->h, &z->h, z->h.plan), sms, s, &launches);
      launches += z->h.plan->sym_launches;
      release_owned(x, s);  // stream-ordered: the value pass above still reads them
      release_owned(y, s);
      partial[i] = partial[i + 1] = nullptr;
    }
    for (; i < partial.size(); ++i) {
      if (partial[i]) next.push_back(partial[i]);
      partial[i] = nullptr;
    }
    for (Owned* o : partial) release_owned(o, s);
    partial.swap(next);
  }
  if (st == WS_OK) {  // the last merge's structure pass writes C.rowptr
    st = ewise_symbolic_impl<T>(&partial[0]->h, &partial[1]->h, C, pl, kEwiseAdd, s, nnz_out);
    if (st == WS_OK && (st = plan_status(partial[0]->h.plan)) == WS_OK) st = plan_status(partial[1]->h.plan);
  }
  cudaFreeAsync(ex_mem, s);
  ex_mem = nullptr;
  if (st != WS_OK) {
    cleanup();
    return st;
  }
  os->x = partial[0];
  os->y = partial[1];
  partial.clear();
  pl->outer = os;
  pl->sym_launches += launches;
  return WS_OK;
}

template <typename T>
ws_status_t outer_numeric_impl(ws_csr_s* C, cudaStream_t s) {
  Plan* pl = C->plan;
  OuterState* os = pl->outer;
  if (os->parts == 1) return numeric_impl<T>(os->A, os->B, C, pl, s);
  pl->num_launches = 0;
  if (C->nnz > 0)
    launch_ewise_numeric<T>(make_ewise<T>(&os->x->h, &os->y->h, C, pl), num_sms_of(C->device), s, &pl->num_launches);
  WS_CUDA(cudaGetLastError(), "outer-product merge launch");
  release_outer(pl, s);  // stream-ordered: the copies stay valid for the pass just queued
  return WS_OK;
}

}  // namespace

extern "C" {

ws_status_t ws_csr_create(ws_csr_t* out, int64_t nrows, int64_t ncols, int64_t nnz, int64_t* rowptr,
                          int32_t* colidx, void* vals, ws_dtype_t dtype, int validate, ws_stream_t stream) {
  g_last_error.clear();
  if (!out) return fail(WS_ERR_INVALID_ARG, "out is NULL");
  *out = nullptr;
  if (nrows < 0 || ncols < 0 || nnz < 0) return fail(WS_ERR_INVALID_ARG, "negative size");
  if (nrows > INT32_MAX - 1 || ncols > INT32_MAX)
    return fail(WS_ERR_OVERFLOW, "nrows/ncols exceed the int32 index range");
  if (dtype != WS_F32 && dtype != WS_F64) return fail(WS_ERR_INVALID_ARG, "unknown dtype %d", (int)dtype);
  if (!rowptr) return fail(WS_ERR_INVALID_ARG, "rowptr is NULL");
  if (nnz > 0 && (!colidx || !vals)) return fail(WS_ERR_INVALID_ARG, "colidx/vals NULL with nnz > 0");
  int dev = 0;
  WS_CUDA(cudaGetDevice(&dev), "cudaGetDevice");
  if (validate) {
    cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
    if (nrows == 0) {
      int64_t r0 = -1;
      WS_CUDA(cudaMemcpyAsync(&r0, rowptr, sizeof(r0), cudaMemcpyDeviceToHost, s), "cudaMemcpyAsync(rowptr[0])");
      WS_CUDA(cudaStreamSynchronize(s), "cudaStreamSynchronize");
      if (r0 != 0 || nnz != 0) return fail(WS_ERR_INVALID_CSR, "empty matrix needs rowptr[0] = 0 and nnz = 0");
    } else {
      // the kernel writes what it finds to a pinned block: nothing for a valid matrix
      HostSummary* h = acquire_host_sum();
      if (!h) return fail(WS_ERR_ALLOC, "cudaMallocHost failed");
      h->status = 0;
      h->bad_row = INT32_MAX;
      launch_validate(rowptr, colidx, nrows, ncols, nnz, h, num_sms_of(dev), s);
      cudaError_t e = cudaGetLastError();
      if (e == cudaSuccess) e = cudaStreamSynchronize(s);
      const volatile HostSummary* v = h;
      const int status = v->status, bad_row = v->bad_row;
      if (e != cudaSuccess) return cuda_fail(e, "validation");  // the block is not reused: the kernel may still run
      release_host_sum(h);
      if (status & kErrInvalidCsr) return fail(WS_ERR_INVALID_CSR, "CSR invariants violated (first bad row %d)", bad_row);
    }
  }
  ws_csr_s* hnd = new (std::nothrow) ws_csr_s;
  if (!hnd) return fail(WS_ERR_ALLOC, "host allocation failed");
  hnd->nrows = nrows;
  hnd->ncols = ncols;
  hnd->nnz = nnz;
  hnd->rowptr = rowptr;
  hnd->colidx = colidx;
  hnd->vals = vals;
  hnd->dtype = dtype;
  hnd->device = dev;
  *out = hnd;
  return WS_OK;
}

ws_status_t ws_spgemm_symbolic(ws_csr_t A, ws_csr_t B, ws_csr_t C, int64_t* nnz_out, ws_stream_t stream) {
  g_last_error.clear();
  ws_status_t st;
  if ((st = check_handle(A, "A")) != WS_OK || (st = check_handle(B, "B")) != WS_OK ||
      (st = check_handle(C, "C")) != WS_OK)
    return st;
  if (!nnz_out) return fail(WS_ERR_INVALID_ARG, "nnz_out is NULL");
  if (C == A || C == B) return fail(WS_ERR_INVALID_ARG, "C must be a separate output handle");
  if (A->ncols != B->nrows)
    return fail(WS_ERR_SHAPE, "A is %lldx%lld but B is %lldx%lld", (long long)A->nrows, (long long)A->ncols,
                (long long)B->nrows, (long long)B->ncols);
  if (C->nrows != A->nrows || C->ncols != B->ncols)
    return fail(WS_ERR_SHAPE, "C is %lldx%lld, expected %lldx%lld", (long long)C->nrows, (long long)C->ncols,
                (long long)A->nrows, (long long)B->ncols);
  if (A->dtype != B->dtype || C->dtype != A->dtype) return fail(WS_ERR_DTYPE, "A, B and C dtypes differ");
  if (A->nnz > 0 && B->nrows == 0) return fail(WS_ERR_INVALID_CSR, "A has entries but B has no rows");
  if ((st = prepare_output(A, B, C)) != WS_OK) return st;
  Plan* pl = C->plan;
  cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
  release_outer(pl, s);
  C->nnz = -1;
  if (A->dtype == WS_F64) return symbolic_impl<double>(A, B, C, pl, s, nnz_out);
  return symbolic_impl<float>(A, B, C, pl, s, nnz_out);
}

ws_status_t ws_spgemm_numeric(ws_csr_t A, ws_csr_t B, ws_csr_t C, int32_t* c_colidx, void* c_vals,
                              ws_stream_t stream) {
  g_last_error.clear();
  ws_status_t st;
  if ((st = check_handle(A, "A")) != WS_OK || (st = check_handle(B, "B")) != WS_OK ||
      (st = check_handle(C, "C")) != WS_OK)
    return st;
  Plan* pl = C->plan;
  if (!pl || !pl->ready || pl->kind != kPlanSpgemm)
    return fail(WS_ERR_STATE, "numeric called before a successful SpGEMM symbolic pass");
  if (pl->A != A || pl->B != B || pl->a_nnz != A->nnz || pl->b_nnz != B->nnz)
    return fail(WS_ERR_STATE, "numeric called with other operands than the symbolic pass");
  if (C->nnz > 0 && (!c_colidx || !c_vals)) return fail(WS_ERR_INVALID_ARG, "c_colidx/c_vals NULL with nnz(C) > 0");
  C->colidx = c_colidx;
  C->vals = c_vals;
  cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
  if (A->dtype == WS_F64) return numeric_impl<double>(A, B, C, pl, s);
  return numeric_impl<float>(A, B, C, pl, s);
}

ws_status_t ws_spgemm_outer_symbolic(ws_csr_t A, ws_csr_t B, ws_csr_t C, int parts, int64_t* nnz_out,
                                     ws_stream_t stream) {
  g_last_error.clear();
  ws_status_t st;
  if ((st = check_handle(A, "A")) != WS_OK || (st = check_handle(B, "B")) != WS_OK ||
      (st = check_handle(C, "C")) != WS_OK)
    return st;
  if (!nnz_out) return fail(WS_ERR_INVALID_ARG, "nnz_out is NULL");
  if (parts < 1) return fail(WS_ERR_INVALID_ARG, "parts must be at least 1, got %d", parts);
  if (C == A || C == B) return fail(WS_ERR_INVALID_ARG, "C must be a separate output handle");
  if (A->ncols != B->nrows)
    return fail(WS_ERR_SHAPE, "A is %lldx%lld but B is %lldx%lld", (long long)A->nrows, (long long)A->ncols,
                (long long)B->nrows, (long long)B->ncols);
  if (C->nrows != A->nrows || C->ncols != B->ncols)
    return fail(WS_ERR_SHAPE, "C is %lldx%lld, expected %lldx%lld", (long long)C->nrows, (long long)C->ncols,
                (long long)A->nrows, (long long)B->ncols);
  if (A->dtype != B->dtype || C->dtype != A->dtype) return fail(WS_ERR_DTYPE, "A, B and C dtypes differ");
  if (A->nnz > 0 && B->nrows == 0) return fail(WS_ERR_INVALID_CSR, "A has entries but B has no rows");
  if ((st = prepare_output(A, B, C)) != WS_OK) return st;
  cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
  C->nnz = -1;
  if (A->dtype == WS_F64) return outer_symbolic_impl<double>(A, B, C, parts, s, nnz_out);
  return outer_symbolic_impl<float>(A, B, C, parts, s, nnz_out);
}

ws_status_t ws_spgemm_outer_numeric(ws_csr_t A, ws_csr_t B, ws_csr_t C, int32_t* c_colidx, void* c_vals,
                                    ws_stream_t stream) {
  g_last_error.clear();
  ws_status_t st;
  if ((st = check_handle(A, "A")) != WS_OK || (st = check_handle(B, "B")) != WS_OK ||
      (st = check_handle(C, "C")) != WS_OK)
    return st;
  Plan* pl = C->plan;
  if (!pl || !pl->ready || !pl->outer)
    return fail(WS_ERR_STATE, "numeric called before a successful outer-product symbolic pass");
  const OuterState* os = pl->outer;
  if (os->A != A || os->B != B || os->a_nnz != A->nnz || os->b_nnz != B->nnz)
    return fail(WS_ERR_STATE, "numeric called with other operands than the symbolic pass");
  if (C->nnz > 0 && (!c_colidx || !c_vals)) return fail(WS_ERR_INVALID_ARG, "c_colidx/c_vals NULL with nnz(C) > 0");
  C->colidx = c_colidx;
  C->vals = c_vals;
  cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
  if (A->dtype == WS_F64) return outer_numeric_impl<double>(C, s);
  return outer_numeric_impl<float>(C, s);
}

ws_status_t ws_ewise_symbolic(ws_csr_t A, ws_csr_t B, ws_csr_t C, int op, int64_t* nnz_out, ws_stream_t stream) {
  g_last_error.clear();
  ws_status_t st;
  if ((st = check_handle(A, "A")) != WS_OK || (st = check_handle(B, "B")) != WS_OK ||
      (st = check_handle(C, "C")) != WS_OK)
    return st;
  if (!nnz_out) return fail(WS_ERR_INVALID_ARG, "nnz_out is NULL");
  if (op != WS_EWISE_ADD && op != WS_EWISE_MUL) return fail(WS_ERR_INVALID_ARG, "unknown elementwise op %d", op);
  if (A->nrows != B->nrows || A->ncols != B->ncols)
    return fail(WS_ERR_SHAPE, "A is %lldx%lld but B is %lldx%lld", (long long)A->nrows, (long long)A->ncols,
                (long long)B->nrows, (long long)B->ncols);
  if (C->nrows != A->nrows || C->ncols != A->ncols)
    return fail(WS_ERR_SHAPE, "C is %lldx%lld, expected %lldx%lld", (long long)C->nrows, (long long)C->ncols,
                (long long)A->nrows, (long long)A->ncols);
  if ((st = prepare_output(A, B, C)) != WS_OK) return st;
  cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
  release_outer(C->plan, s);
  C->nnz = -1;
  const int kop = op == WS_EWISE_ADD ? kEwiseAdd : kEwiseMul;
  if (A->dtype == WS_F64) return ewise_symbolic_impl<double>(A, B, C, C->plan, kop, s, nnz_out);
  return ewise_symbolic_impl<float>(A, B, C, C->plan, kop, s, nnz_out);
}

ws_status_t ws_ewise_numeric(ws_csr_t A, ws_csr_t B, ws_csr_t C, int32_t* c_colidx, void* c_vals,
                             ws_stream_t stream) {
  g_last_error.clear();
  ws_status_t st;
  if ((st = check_handle(A, "A")) != WS_OK || (st = check_handle(B, "B")) != WS_OK ||
      (st = check_handle(C, "C")) != WS_OK)
    return st;
  Plan* pl = C->plan;
  if (!pl || !pl->ready || pl->kind != kPlanEwise)
    return fail(WS_ERR_STATE, "numeric called before a successful elementwise symbolic pass");
  if (pl->A != A || pl->B != B || pl->a_nnz != A->nnz || pl->b_nnz != B->nnz)
    return fail(WS_ERR_STATE, "numeric called with other operands than the symbolic pass");
  if (C->nnz > 0 && (!c_colidx || !c_vals)) return fail(WS_ERR_INVALID_ARG, "c_colidx/c_vals NULL with nnz(C) > 0");
  C->colidx = c_colidx;
  C->vals = c_vals;
  pl->num_launches = 0;
  if (C->nnz == 0) return WS_OK;
  cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
  const int sms = num_sms_of(C->device);
  if (A->dtype == WS_F64) {
    launch_ewise_numeric<double>(make_ewise<double>(A, B, C, pl), sms, s, &pl->num_launches);
  } else {
    launch_ewise_numeric<float>(make_ewise<float>(A, B, C, pl), sms, s, &pl->num_launches);
  }
  WS_CUDA(cudaGetLastError(), "elementwise numeric launch");
  return WS_OK;
}

ws_status_t ws_spmspv(ws_csr_t At, int64_t nnz_x, const int32_t* x_idx, const void* x_vals, int32_t* y_idx,
                      void* y_vals, int64_t* nnz_y, ws_stream_t stream) {
  g_last_error.clear();
  ws_status_t st;
  if ((st = check_handle(At, "At")) != WS_OK) return st;
  if (!nnz_y) return fail(WS_ERR_INVALID_ARG, "nnz_y is NULL");
  if (nnz_x < 0 || nnz_x > At->nrows) return fail(WS_ERR_INVALID_ARG, "nnz_x must be in [0, %lld]", (long long)At->nrows);
  if (nnz_x > 0 && (!x_idx || !x_vals)) return fail(WS_ERR_INVALID_ARG, "x_idx/x_vals NULL with nnz_x > 0");
  if (At->ncols > 0 && (!y_idx || !y_vals)) return fail(WS_ERR_INVALID_ARG, "y_idx/y_vals NULL");
  if ((st = ensure_plan(At)) != WS_OK) return st;
  cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
  if (At->dtype == WS_F64) return spmspv_impl<double>(At, nnz_x, x_idx, x_vals, y_idx, y_vals, nnz_y, s);
  return spmspv_impl<float>(At, nnz_x, x_idx, x_vals, y_idx, y_vals, nnz_y, s);
}

ws_status_t ws_csr_submatrix_symbolic(ws_csr_t A, int64_t r0, int64_t r1, int64_t c0, int64_t c1, ws_csr_t S,
                                      int64_t* nnz_out, ws_stream_t stream) {
  g_last_error.clear();
  ws_status_t st;
  if ((st = check_handle(A, "A")) != WS_OK || (st = check_handle(S, "S")) != WS_OK) return st;
  if (!nnz_out) return fail(WS_ERR_INVALID_ARG, "nnz_out is NULL");
  if (S == A) return fail(WS_ERR_INVALID_ARG, "S must be a separate output handle");
  if (r0 < 0 || r0 > r1 || r1 > A->nrows || c0 < 0 || c0 > c1 || c1 > A->ncols)
    return fail(WS_ERR_INVALID_ARG, "block [%lld:%lld, %lld:%lld] outside the %lldx%lld matrix", (long long)r0,
                (long long)r1, (long long)c0, (long long)c1, (long long)A->nrows, (long long)A->ncols);
  if (S->nrows != r1 - r0 || S->ncols != c1 - c0)
    return fail(WS_ERR_SHAPE, "S is %lldx%lld, expected %lldx%lld", (long long)S->nrows, (long long)S->ncols,
                (long long)(r1 - r0), (long long)(c1 - c0));
  if (S->dtype != A->dtype) return fail(WS_ERR_DTYPE, "A and S dtypes differ");
  if ((st = ensure_plan(S)) != WS_OK) return st;
  Plan* pl = S->plan;
  cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
  const int64_t rows = r1 - r0;
  const int64_t nb = scan_partials_needed(rows);
  const size_t o_part = align_up(sizeof(DevSummary), 256);
  if ((st = pl->ew.reserve(o_part + 8 * static_cast<size_t>(nb + 1), s)) != WS_OK) return st;
  char* b = static_cast<char*>(pl->ew.ptr);
  pl->dsum = reinterpret_cast<DevSummary*>(b);
  int64_t* partials = reinterpret_cast<int64_t*>(b + o_part);
  pl->ready = false;
  pl->kind = kPlanSub;
  pl->sym_launches = 0;
  pl->num_launches = 0;
  S->nnz = -1;
  if ((st = begin_pass(pl, pl->ew, s)) != WS_OK) return st;
  if (rows == 0) {
    WS_CUDA(cudaMemsetAsync(S->rowptr, 0, sizeof(int64_t), s), "cudaMemsetAsync(rowptr[0])");
  } else {
    const int sms = num_sms_of(S->device);
    launch_submatrix_count(A->rowptr, A->colidx, r0, rows, c0, c1, S->rowptr, sms, s, &pl->sym_launches);
    launch_scan(S->rowptr, rows, partials, pl->dsum, s, &pl->sym_launches, nullptr, pl->host_sum);
    WS_CUDA(cudaGetLastError(), "submatrix symbolic launches");
  }
  if ((st = wait_summary(s)) != WS_OK) return st;
  if (rows > 0) end_pass(pl, pl->ew);
  S->nnz = rows > 0 ? pl->host_sum->nnz : 0;
  pl->A = A;
  pl->B = nullptr;
  pl->a_nnz = A->nnz;
  pl->sub_r0 = r0;
  pl->sub_r1 = r1;
  pl->sub_c0 = c0;
  pl->sub_c1 = c1;
  pl->ready = true;
  *nnz_out = S->nnz;
  return WS_OK;
}

ws_status_t ws_csr_submatrix_numeric(ws_csr_t A, ws_csr_t S, int32_t* s_colidx, void* s_vals, ws_stream_t stream) {
  g_last_error.clear();
  ws_status_t st;
  if ((st = check_handle(A, "A")) != WS_OK || (st = check_handle(S, "S")) != WS_OK) return st;
  Plan* pl = S->plan;
  if (!pl || !pl->ready || pl->kind != kPlanSub)
    return fail(WS_ERR_STATE, "numeric called before a successful submatrix symbolic pass");
  if (pl->A != A || pl->a_nnz != A->nnz)
    return fail(WS_ERR_STATE, "numeric called with another matrix than the symbolic pass");
  if (S->nnz > 0 && (!s_colidx || !s_vals)) return fail(WS_ERR_INVALID_ARG, "s_colidx/s_vals NULL with nnz(S) > 0");
  S->colidx = s_colidx;
  S->vals = s_vals;
  pl->num_launches = 0;
  if (S->nnz == 0) return WS_OK;
  cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
  const int sms = num_sms_of(S->device);
  const int64_t rows = pl->sub_r1 - pl->sub_r0;
  if (A->dtype == WS_F64) {
    launch_submatrix_copy<double>(A->rowptr, A->colidx, static_cast<const double*>(A->vals), pl->sub_r0, rows,
                                  pl->sub_c0, S->rowptr, s_colidx, static_cast<double*>(s_vals), status_word(pl), sms, s,
                                  &pl->num_launches);
  } else {
    launch_submatrix_copy<float>(A->rowptr, A->colidx, static_cast<const float*>(A->vals), pl->sub_r0, rows,
                                 pl->sub_c0, S->rowptr, s_colidx, static_cast<float*>(s_vals), status_word(pl), sms, s,
                                 &pl->num_launches);
  }
  WS_CUDA(cudaGetLastError(), "submatrix numeric launch");
  return WS_OK;
}

ws_status_t ws_spgemm_wait(ws_csr_t C, ws_stream_t stream) {
  g_last_error.clear();
  if (!C) return fail(WS_ERR_INVALID_ARG, "C is NULL");
  Plan* pl = C->plan;
  cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
  WS_CUDA(cudaStreamSynchronize(s), "cudaStreamSynchronize");
  if (!pl || !pl->host_sum || !pl->dsum) return WS_OK;
  return device_status(pl);
}

ws_status_t ws_csr_destroy(ws_csr_t h) {
  if (!h) return WS_OK;
  if (Plan* pl = h->plan) {
    const DeviceGuard guard(h->device);  // the scratch is that device's, whichever is current
    bool idle = guard.ok();
    if (pl->scratch_bytes() > 0 || pl->outer) idle = cudaDeviceSynchronize() == cudaSuccess && idle;
    release_outer(pl, nullptr);
    if (!idle || !keep_plan(pl)) {
      for (DevBuf* b : {&pl->rows, &pl->slices, &pl->ranks, &pl->ew, &pl->sv, &pl->hranks, &pl->rcd, &pl->wb}) b->release();
      release_host_sum(pl->host_sum);
      delete pl;
    }
  }
  delete h;
  return WS_OK;
}

const char* ws_status_string(ws_status_t st) {
  switch (st) {
    case WS_OK: return "ok";
    case WS_ERR_INVALID_ARG: return "invalid argument";
    case WS_ERR_INVALID_CSR: return "invalid CSR matrix";
    case WS_ERR_SHAPE: return "shape mismatch";
    case WS_ERR_DTYPE: return "dtype mismatch";
    case WS_ERR_OVERFLOW: return "size overflow";
    case WS_ERR_ALLOC: return "allocation failed";
    case WS_ERR_CUDA: return "CUDA error";
    case WS_ERR_DEVICE: return "device-side failure";
    case WS_ERR_STATE: return "calls out of order";
  }
  return "unknown status";
}

const char* ws_last_error(void) { return g_last_error.c_str(); }

ws_status_t ws_csr_nnz(ws_csr_t h, int64_t* nnz_out) {
  if (!h || !nnz_out) return fail(WS_ERR_INVALID_ARG, "NULL argument");
  *nnz_out = h->nnz;
  return WS_OK;
}

ws_status_t ws_spgemm_plan_info(ws_csr_t C, int64_t* info, int n) {
  if (!C || !info || n < 0) return fail(WS_ERR_INVALID_ARG, "NULL argument");
  const Plan* pl = C->plan;
  int64_t v[12] = {0, 0, 0, 0, 0, 0, 0, 0, 0, 0, 0, 0};
  if (pl) {
    int64_t hash_rows = 0, bitmap_rows = 0;
    for (int b = 0; b < kNumHashBins; ++b) hash_rows += pl->seg_count[kSegHash0 + b];
    for (int b = 0; b < kNumBitmapBins; ++b) bitmap_rows += pl->seg_count[kSegBitmap0 + b];
    for (int b = 0; b < kNumBmrBins; ++b) bitmap_rows += pl->seg_count[kSegBmr0 + b];
    bitmap_rows += pl->seg_count[kSegBmrWide];
    v[0] = pl->n_empty;
    v[1] = pl->seg_count[kSegDirect];
    v[2] = hash_rows;
    v[3] = pl->n_sort;
    v[4] = pl->seg_count[kSegDense];
    v[5] = pl->dense_slices;
    v[6] = pl->products;
    v[7] = pl->sym_launches;
    v[8] = pl->num_launches;
    v[9] = bitmap_rows;
    v[10] = pl->seg_count[kSegRcd];
    v[11] = pl->seg_count[kSegWb];
  }
  for (int i = 0; i < n && i < 12; ++i) info[i] = v[i];
  return WS_OK;
}

ws_status_t ws_set_tuning(int key, int64_t value) {
  switch (key) {
    case 1:
      if (value < 0 || value > kMaxHashProducts) return fail(WS_ERR_INVALID_ARG, "hash limit out of range");
      g_hash_max = value;
      return WS_OK;
    case 2:
      if (value < 1 || value > 4096) return fail(WS_ERR_INVALID_ARG, "run limit out of range");
      g_run_limit = value < kMaxHashBucket ? static_cast<int>(value) : kMaxHashBucket;
      return WS_OK;
    case 3:
      if (value != 0 && (value < 1024 || value > 16384 || value % 1024 != 0))
        return fail(WS_ERR_INVALID_ARG, "dense width must be 0 or a multiple of 1024 in [1024, 16384]");
      g_dense_width = static_cast<int>(value);
      return WS_OK;
    case 4:
      if (value < 0 || value > kMaxBitmapSpan) return fail(WS_ERR_INVALID_ARG, "bitmap span out of range");
      g_bitmap_span = value;
      return WS_OK;
    case 5:
      if (value < 0 || value > kBmrMaxA) return fail(WS_ERR_INVALID_ARG, "register-row entry limit out of range");
      g_bmr_max_a = static_cast<int>(value);
      return WS_OK;
    case 6:
      if (value < 0 || value > kRcdMaxA) return fail(WS_ERR_INVALID_ARG, "dense-row entry limit out of range");
      g_rcd_max_a = static_cast<int>(value);
      return WS_OK;
    case 7:
      if (value < 0 || value > kWbMaxSpan) return fail(WS_ERR_INVALID_ARG, "wide-bitmap span out of range");
      g_wb_span = value;
      return WS_OK;
    case 8:  // accepted, without effect: the elementwise operations have one path
      if (value < -1 || value > 64 || (value > 2 && (value & (value - 1)) != 0))
        return fail(WS_ERR_INVALID_ARG, "elementwise lanes per chunk must be -1, 0, 1, 2, 4, 8, 16, 32 or 64");
      return WS_OK;
    case 9:  // likewise
      if (value < 2 || value > (int64_t{1} << 20)) return fail(WS_ERR_INVALID_ARG, "elementwise chunk length out of range");
      return WS_OK;
    case 10:
      if (value < 0 || value > static_cast<int64_t>(kMaxKeptBytes)) return fail(WS_ERR_INVALID_ARG, "kept bytes out of range");
      g_kept_bytes = static_cast<size_t>(value);
      return WS_OK;
  }
  return fail(WS_ERR_INVALID_ARG, "unknown tuning key %d", key);
}

}  // extern "C"
