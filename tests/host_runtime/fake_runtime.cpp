// The part of the CUDA runtime that the library's host code calls, on the CPU:
// several devices, memory that is counted, streams and events that remember
// where they were made, a record of the synchronisations.
#include <cstdlib>
#include <cstring>
#include <iterator>

#include "fake_state.h"

extern "C" {
cudaError_t cudaGetDevice(int* d) { *d = fake::device; return cudaSuccess; }
cudaError_t cudaSetDevice(int d) { fake::device = d; return cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int* v, cudaDeviceAttr, int) { *v = 4; return cudaSuccess; }
cudaError_t cudaDeviceGetDefaultMemPool(cudaMemPool_t* p, int) { *p = nullptr; return cudaSuccess; }
cudaError_t cudaMemPoolSetAttribute(cudaMemPool_t, cudaMemPoolAttr, void*) { return cudaSuccess; }
cudaError_t cudaGetLastError() { return cudaSuccess; }
const char* cudaGetErrorString(cudaError_t e) { return e == cudaSuccess ? "no error" : "error"; }
cudaError_t cudaDeviceSynchronize() { fake::synced_devices.push_back(fake::device); return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t s) {
  for (auto it = fake::pending.begin(); it != fake::pending.end();) it = it->second == s ? fake::pending.erase(it) : std::next(it);
  return cudaSuccess;
}
cudaError_t cudaMallocAsync(void** p, size_t n, cudaStream_t) {
  if (fake::fail_in == 0) {
    fake::fail_in = -1;
    *p = nullptr;
    return cudaErrorMemoryAllocation;
  }
  if (fake::fail_in > 0) --fake::fail_in;
  *p = std::malloc(n);
  fake::live[*p] = n;
  fake::bytes += n;
  fake::peak = fake::bytes > fake::peak ? fake::bytes : fake::peak;
  return cudaSuccess;
}
cudaError_t cudaFreeAsync(void* p, cudaStream_t) {
  fake::bytes -= fake::live.at(p);
  fake::live.erase(p);
  std::free(p);
  return cudaSuccess;
}
cudaError_t cudaMallocHost(void** p, size_t n) { *p = std::calloc(1, n); return cudaSuccess; }
cudaError_t cudaMemsetAsync(void* p, int v, size_t n, cudaStream_t) { std::memset(p, v, n); return cudaSuccess; }
cudaError_t cudaMemcpyAsync(void* d, const void* s, size_t n, cudaMemcpyKind, cudaStream_t) { std::memcpy(d, s, n); return cudaSuccess; }
cudaError_t cudaStreamCreateWithFlags(cudaStream_t* s, unsigned) {
  fake::streams.push_back(*s = new CUstream_st{fake::device, 0, false, fake::context});
  return cudaSuccess;
}
cudaError_t cudaStreamCreateWithPriority(cudaStream_t* s, unsigned, int priority) {
  fake::streams.push_back(*s = new CUstream_st{fake::device, priority, false, fake::context});
  return cudaSuccess;
}
cudaError_t cudaStreamGetPriority(cudaStream_t s, int* priority) { *priority = s ? s->priority : 0; return cudaSuccess; }
cudaError_t cudaStreamDestroy(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamIsCapturing(cudaStream_t, cudaStreamCaptureStatus* c) { *c = cudaStreamCaptureStatusNone; return cudaSuccess; }
cudaError_t cudaStreamWaitEvent(cudaStream_t, cudaEvent_t, unsigned) { return cudaSuccess; }
cudaError_t cudaEventCreateWithFlags(cudaEvent_t* e, unsigned) {
  fake::events.push_back(*e = new CUevent_st{fake::device});
  return cudaSuccess;
}
cudaError_t cudaEventDestroy(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return cudaSuccess; }
// the driver
static CUresult current_context(CUcontext* c) { *c = reinterpret_cast<CUcontext>(&fake::context); return CUDA_SUCCESS; }
static CUresult context_id(CUcontext c, unsigned long long* id) { *id = *reinterpret_cast<unsigned long long*>(c); return CUDA_SUCCESS; }
static CUresult green_context(CUstream s, CUgreenCtx* g) {
  *g = s && s->confined ? reinterpret_cast<CUgreenCtx>(s) : nullptr;
  return CUDA_SUCCESS;
}
cudaError_t cudaGetDriverEntryPointByVersion(const char* name, void** f, unsigned, unsigned long long,
                                             cudaDriverEntryPointQueryResult* found) {
  *f = std::strcmp(name, "cuCtxGetCurrent") == 0       ? reinterpret_cast<void*>(current_context)
       : std::strcmp(name, "cuCtxGetId") == 0          ? reinterpret_cast<void*>(context_id)
       : std::strcmp(name, "cuStreamGetGreenCtx") == 0 ? reinterpret_cast<void*>(green_context)
                                                       : nullptr;
  *found = *f ? cudaDriverEntryPointSuccess : cudaDriverEntryPointSymbolNotFound;
  return cudaSuccess;
}
// nvcc's registration of (no) kernels
void** __cudaRegisterFatBinary(void*) { return nullptr; }
void __cudaRegisterFatBinaryEnd(void**) {}
void __cudaUnregisterFatBinary(void**) {}
}
