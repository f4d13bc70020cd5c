// host.h -- host-side objects behind the C ABI handles (not part of the ABI).
#pragma once
#include <cuda_runtime.h>

#include <algorithm>
#include <mutex>
#include <string>
#include <vector>

#include "blob.h"
#include "devbuf.h"
#include "device.cuh"
#include "../../include/netburn.h"

struct nb_net_s {
  nb::BlobHeader h;
  std::vector<uint8_t> blob;
  unsigned char* d_blob = nullptr;
  int device = 0;
  int sm_count = 0;
  size_t smem_optin = 0;
  nb::DevBuf<double> ws;
  unsigned long long* queue = nullptr;
  // staging for the host-pointer entry point
  nb::DevBuf<unsigned char> stage;
  nb::DevBuf<double> ws_adj;              // adjoint per-lane workspace
  nb::DevBuf<unsigned char> sched;        // claim-order keys, indices, sort scratch
  nb::DevBuf<unsigned char> sched_adj;    // the adjoint's claim order and sort scratch
  std::vector<void*> kept;                // outgrown buffers that captured graphs use
  // network-specialised kernels by storage variant (1..3) and, from
  // kSpecTeam on, by lanes per zone (4, 8, 16, 32): 0 not built, 1 loaded,
  // -1 failed (log kept)
  static constexpr int kSpecTeam = 4;
  struct Spec {
    int state = 0;
    cudaLibrary_t lib = nullptr;
    cudaKernel_t kern = nullptr;
    std::string log;
  } spec[kSpecTeam + 4];
  int last_spec = 0;   // variant the last burn ran (0 generic)
  std::mutex mu;
};

struct nb_tape_s {
  nb_net net;
  long long Z;
  int cap;
  nb::TapeDev dev{};
  long long recZ = 0;       // zones of the recorded burn
  double* lnm = nullptr;   // copy of the multipliers of the recorded burn
  int lnm_per_zone = 0;
  int has_lnm = 0;
  double t_end = 0, rtol = 0, atol = 0;
  int recorded = 0;
  // arithmetic of the recording burn: NB_KERNEL_PERSISTENT for the
  // one-zone-per-lane kernels (which share their bits), NB_KERNEL_COOP for
  // one zone per warp; a checkpointed block is recomputed in the same one
  int family = 0;
  unsigned magic = 0x7a9e5eedu;
};

// device buffers of a tape (each may be null)
inline void tape_release(nb_tape_s* tp) {
  cudaFree(tp->dev.sched); cudaFree(tp->dev.ord); cudaFree(tp->dev.states);
  cudaFree(tp->dev.steps); cudaFree(tp->dev.zstat); cudaFree(tp->dev.rho);
  cudaFree(tp->dev.T9f); cudaFree(tp->dev.scr); cudaFree(tp->lnm);
}

#define CK(call)                                                   \
  do {                                                             \
    cudaError_t e_ = (call);                                       \
    if (e_ != cudaSuccess) return NB_E_CUDA;                       \
  } while (0)


namespace nb {
// Let a kernel be launched with any dynamic shared memory a block may have
// (smem_optin; the kernels here have no other).  The limit belongs to the
// kernel, not to a launch: set to one launch's size, another thread's call for
// a smaller network could lower it before that launch, which would fail.
inline cudaError_t allow_shared(const void* fn, size_t smem_optin) {
  return cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem_optin);
}

// Blocks of `teams` zones that hold the zones of `blocks` blocks of `warps`
// (0: four) warps with a zone each, the shape an option asks for.
inline int team_blocks(int blocks, int warps, int teams) {
  const long long zones = (long long)blocks * (warps > 0 ? warps : 4);
  return (int)std::min<long long>((zones + teams - 1) / teams, 64);
}

// doubles per lane of a start-up pass (k_burn_start)
__host__ __device__ constexpr int start_doubles(int n, int R) { return 5 * n + 2 * R + 2; }
// its lanes, one zone each at a time: what four blocks per SM hold (one block
// of 128 lanes for all zones took 0.9 s for 262,144 zones of the 48-species
// network), and their workspace
inline long long prepass_lanes(nb_net net, long long Z) {
  return std::min<long long>((Z + 127) / 128 * 128, (long long)net->sm_count * 512);
}
inline size_t prepass_bytes(nb_net net, long long Z) {
  return (size_t)prepass_lanes(net, Z) * start_doubles(net->h.n, net->h.R) * sizeof(double);
}

// Longest-first claim order: h0 of every zone (a start-up pass in the
// workspace already allocated), then a radix sort of (h0, zone).  Sets
// P.order.  (burn.cu)
int schedule_longest_first(nb_net net, BurnParams& P, cudaStream_t st);
// The cooperative launch (coop.cu).  Caller holds net->mu.
int launch_coop(nb_net net, BurnParams& P, const nb_options& o, cudaStream_t st);
// A persistent burn by teams with the lane kernel's bits; false when the
// network is too large for it (coop.cu).  Caller holds net->mu.
bool launch_lane_teams(nb_net net, BurnParams& P, const nb_options& o, cudaStream_t st, int* rc);
}  // namespace nb
