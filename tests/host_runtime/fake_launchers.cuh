// Kernel launchers that do no work; those that end a pass hand the host the
// summary a check prepared.  Linked with api.cu instead of the kernel files.
#pragma once
#include <cstring>

#include "fake_state.h"
#include "ws_internal.cuh"

namespace fake {

inline wsk::DevSummary summary{};             // what a pass hands to the host
inline std::vector<size_t> bitmap_after;      // row kernels queued before every bitmap kernel
inline int run_limit = 0;                    // products of a hash bucket that are compared
inline int rcd_width = 0, rcd_slices = 0;     // value windows of the dense rows
inline int64_t wb_part = 0;  // products per item that the wide rows' kernels were given
inline int launch_status = 0;                 // error flags that SpMSpV's kernels find
inline std::vector<cudaStream_t> row_kernels; // stream of every row kernel launched

}  // namespace fake

namespace wsk {

int64_t scan_partials_needed(int64_t m) { return (m + 4095) / 4096; }
int64_t spmspv_tiles(int64_t m) { return (m + 4095) / 4096; }

void launch_scan(int64_t*, int64_t, int64_t*, DevSummary*, cudaStream_t, int*, const int*, DevSummary* host) {
  if (host) std::memcpy(static_cast<void*>(host), &fake::summary, sizeof(DevSummary));
}
void launch_validate(const int64_t*, const int32_t*, int64_t, int64_t, int64_t, DevSummary*, int, cudaStream_t) {}
void launch_submatrix_count(const int64_t*, const int32_t*, int64_t, int64_t, int64_t, int64_t, int64_t*, int,
                            cudaStream_t, int*) {}
template <typename T>
void launch_submatrix_copy(const int64_t*, const int32_t*, const T*, int64_t, int64_t, int64_t, const int64_t*, int32_t*,
                           T*, int*, int, cudaStream_t, int*) {}
template <typename T>
void launch_analyze(const RowPlan<T>&, const AnalyzeParams&, int32_t*, const int32_t*, DevSummary* host, int,
                    cudaStream_t, int*) {
  if (host) std::memcpy(static_cast<void*>(host), &fake::summary, sizeof(DevSummary));
}
template <typename T>
void launch_bmr_plan(const RowPlan<T>&, const AnalyzeParams&, int64_t, int32_t*, int, cudaStream_t, int*) {}
template <typename T>
void launch_scatter(const RowPlan<T>&, int64_t, const int64_t*, int, cudaStream_t, int*) {}
template <typename T>
void launch_dense_slices(const RowPlan<T>&, int32_t*, int32_t*, int32_t*, int, cudaStream_t, int*) {}
template <typename T>
void launch_hash(const RowPlan<T>& p, int, bool, int, cudaStream_t s, int*) {
  fake::row_kernels.push_back(s);
  fake::pending[p.status] = s;
  fake::run_limit = p.run_limit;
}
template <typename T>
void launch_bmr(const RowPlan<T>&, int, bool, int, cudaStream_t s, int*) { fake::row_kernels.push_back(s); }
template <typename T>
void launch_bitmap(const RowPlan<T>&, int, bool, int, cudaStream_t s, int*) {
  fake::bitmap_after.push_back(fake::row_kernels.size());
  fake::row_kernels.push_back(s);
}
template <typename T>
void launch_rcd(const RowPlan<T>& p, bool, int, cudaStream_t s, int*) {
  fake::row_kernels.push_back(s);
  fake::rcd_width = p.rcd_width;
  fake::rcd_slices = p.rcd_slices;
}
template <typename T>
void launch_wb(const RowPlan<T>& p, bool, int, cudaStream_t s, int*) {
  fake::row_kernels.push_back(s);
  fake::wb_part = p.wb_part;
}
template <typename T>
void launch_dense(const RowPlan<T>&, int64_t, bool, int, cudaStream_t s, int*) { fake::row_kernels.push_back(s); }
template <typename T>
void launch_direct(const RowPlan<T>&, int, cudaStream_t s, int*) { fake::row_kernels.push_back(s); }
template <typename T>
void launch_ewise_symbolic(const EwisePlan<T>& p, int, cudaStream_t, int*) { p.host->nnz = fake::summary.nnz; }
template <typename T>
void launch_ewise_numeric(const EwisePlan<T>&, int, cudaStream_t, int*) {}
template <typename T>
void launch_spmspv(const SpmspvPlan<T>& p, int, cudaStream_t, int*) {
  *p.status |= fake::launch_status;
  p.host->nnz = 0;
}

#define FAKE_INST(T)                                                                                                  \
  template void launch_submatrix_copy<T>(const int64_t*, const int32_t*, const T*, int64_t, int64_t, int64_t,         \
                                         const int64_t*, int32_t*, T*, int*, int, cudaStream_t, int*);                \
  template void launch_analyze<T>(const RowPlan<T>&, const AnalyzeParams&, int32_t*, const int32_t*, DevSummary*, int, \
                                  cudaStream_t, int*);                                                                \
  template void launch_bmr_plan<T>(const RowPlan<T>&, const AnalyzeParams&, int64_t, int32_t*, int, cudaStream_t,      \
                                   int*);                                                                             \
  template void launch_scatter<T>(const RowPlan<T>&, int64_t, const int64_t*, int, cudaStream_t, int*);               \
  template void launch_dense_slices<T>(const RowPlan<T>&, int32_t*, int32_t*, int32_t*, int, cudaStream_t, int*);     \
  template void launch_hash<T>(const RowPlan<T>&, int, bool, int, cudaStream_t, int*);                                \
  template void launch_bmr<T>(const RowPlan<T>&, int, bool, int, cudaStream_t, int*);                                 \
  template void launch_bitmap<T>(const RowPlan<T>&, int, bool, int, cudaStream_t, int*);                              \
  template void launch_rcd<T>(const RowPlan<T>&, bool, int, cudaStream_t, int*);                                      \
  template void launch_wb<T>(const RowPlan<T>&, bool, int, cudaStream_t, int*);                                       \
  template void launch_dense<T>(const RowPlan<T>&, int64_t, bool, int, cudaStream_t, int*);                           \
  template void launch_direct<T>(const RowPlan<T>&, int, cudaStream_t, int*);                                         \
  template void launch_ewise_symbolic<T>(const EwisePlan<T>&, int, cudaStream_t, int*);                               \
  template void launch_ewise_numeric<T>(const EwisePlan<T>&, int, cudaStream_t, int*);                                \
  template void launch_spmspv<T>(const SpmspvPlan<T>&, int, cudaStream_t, int*);
FAKE_INST(float)
FAKE_INST(double)

}  // namespace wsk
