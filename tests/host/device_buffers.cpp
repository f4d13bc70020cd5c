// device_buffers.cpp -- the buffers a network keeps between calls
// (csrc/devbuf.h) over a fake of the four CUDA calls it makes.  Test
// infrastructure.
#include <cstdlib>
#include <set>

#include "../../paper_2312_02836_gb300/csrc/devbuf.h"

static std::set<void*> live;
static bool capturing, refuse;

extern "C" cudaError_t cudaMalloc(void** p, size_t n) {
  if (refuse) return cudaErrorMemoryAllocation;
  live.insert(*p = std::malloc(n));
  return cudaSuccess;
}
extern "C" cudaError_t cudaFree(void* p) {
  live.erase(p);
  std::free(p);
  return cudaSuccess;
}
extern "C" cudaError_t cudaStreamIsCapturing(cudaStream_t, cudaStreamCaptureStatus* s) {
  *s = capturing ? cudaStreamCaptureStatusActive : cudaStreamCaptureStatusNone;
  return cudaSuccess;
}
extern "C" cudaError_t cudaGetLastError() { return cudaSuccess; }

static nb::DevBuf<double> buf;
static std::vector<void*> kept;

// the buffer's address after a call that needs `need` bytes, null: refused
extern "C" void* buf_call(size_t need, int in_capture, int no_memory) {
  capturing = in_capture;
  refuse = no_memory;
  return nb::ensure(buf, kept, need, nullptr) == NB_OK ? buf.p : nullptr;
}
extern "C" int buf_live(void* p) { return (int)live.count(p); }
extern "C" int buf_count() { return (int)live.size(); }
