// devbuf.h -- device buffers a network keeps between calls.
#pragma once
#include <cuda_runtime_api.h>

#include <cstddef>
#include <vector>

#include "../../include/netburn.h"

namespace nb {

template <class T>
struct DevBuf {
  T* p = nullptr;
  size_t bytes = 0;
  bool in_graph = false;   // a captured launch holds its address
};

// whether work on stream st is being captured into a graph
inline bool capturing(cudaStream_t st) {
  cudaStreamCaptureStatus s = cudaStreamCaptureStatusNone;
  if (cudaStreamIsCapturing(st, &s) != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  return s != cudaStreamCaptureStatusNone;
}

// Make buffer b at least `need` bytes for work on stream st.  A graph keeps
// the addresses of its capture and may be replayed after any later call, so a
// buffer that a capture has used is not freed when it has to grow: it goes to
// `kept`, which is freed with the network (at most one buffer of each kind a
// capture).
template <class T>
inline int ensure(DevBuf<T>& b, std::vector<void*>& kept, size_t need, cudaStream_t st) {
  if (!b.p || b.bytes < need) {
    if (b.p && b.in_graph) kept.push_back(b.p);
    else if (b.p) cudaFree(b.p);
    b = DevBuf<T>();
    void* p = nullptr;
    if (cudaMalloc(&p, need) != cudaSuccess) return NB_E_NOMEM;
    b.p = static_cast<T*>(p);
    b.bytes = need;
  }
  if (capturing(st)) b.in_graph = true;
  return NB_OK;
}

}  // namespace nb
