// State of the fake CUDA runtime (fake_runtime.cpp) that checks look at.
#pragma once
#include <cuda.h>
#include <cuda_runtime_api.h>

#include <map>
#include <vector>

// A stream of the fake runtime.
struct CUstream_st {
  int device = 0, priority = 0;
  bool confined = false;  // belongs to a green context
  unsigned long long context = 0;
};
struct CUevent_st {
  int device = 0;
};

namespace fake {

inline int device = 0;                        // current device
inline unsigned long long context = 1;        // number of the current context
inline std::map<void*, size_t> live;          // device memory
inline size_t bytes = 0, peak = 0;            // in use now, and at most
inline long long fail_in = -1;                // the allocation with this number from now on fails (-1: none)
inline std::vector<int> synced_devices;       // device of every cudaDeviceSynchronize
inline std::map<int*, cudaStream_t> pending;  // status words that queued hash kernels may write to, and their stream
inline std::vector<CUstream_st*> streams;     // streams created by the library
inline std::vector<CUevent_st*> events;


}  // namespace fake
