// coop_kernel.cuh -- the persistent kernel that gives a zone to a team of
// threads (coop.cuh), instantiated in coop.cu and coop_forms.cu.
#pragma once
#include "coop.cuh"

namespace nb {

// One zone per team of P threads (coop.cuh), sums of pattern S.  MEM 0: the
// team's arrays in the global workspace; 1: its Newton-loop arrays in shared
// memory, f0 and the history in the workspace.  B.smem_warps holds the doubles
// between one team's arrays and the next in shared memory.
template <int P, int S, int MEM, int TPB, int MINB>
__global__ void __launch_bounds__(TPB, MINB) k_burn_coop(const __grid_constant__ BurnParams B, const __grid_constant__ BlobHeader H) {
  extern __shared__ __align__(16) unsigned char sm[];
  const unsigned char* blob = B.blob;
  if (B.blob_in_smem) {
    const int4* src = reinterpret_cast<const int4*>(B.blob);
    int4* dst = reinterpret_cast<int4*>(sm);
    for (int i = threadIdx.x; i < B.blob_bytes / 16; i += blockDim.x) dst[i] = src[i];
    __syncthreads();
    blob = sm;
  }
  unsigned char* rest = sm + (B.blob_in_smem ? B.blob_bytes : 0);
  const TNet<P, S> t(BlobDims(blob, H), reinterpret_cast<unsigned long long*>(rest));
  double* smd = reinterpret_cast<double*>(rest + team_scratch_bytes(P));
  const int tib = threadIdx.x / P;
  const long long team = (long long)blockIdx.x * (blockDim.x / P) + tib;
  const int thot = H.thot, tcold = H.tcold;
  CWS w;
  if constexpr (MEM == 1) {
    w = make_cws(H, smd + (size_t)tib * B.smem_warps, B.ws + team * tcold);
  } else {
    double* hot = B.ws + team * (thot + tcold);
    w = make_cws(H, hot, hot + thot);
  }
  coop_claim_loop(t, w, B);
}

// One built form of the kernel.
struct TeamKernel {
  int P, S, mem;
  void (*fn)(const BurnParams, const BlobHeader);
};
#define NB_TEAM(P, S, MEM, TPB, MINB) {P, S, MEM, nb::k_burn_coop<P, S, MEM, TPB, MINB>}

// the forms of coop_forms.cu
constexpr int kOtherTeams = 8;
extern const TeamKernel kOtherTeamKernels[kOtherTeams];

}  // namespace nb
