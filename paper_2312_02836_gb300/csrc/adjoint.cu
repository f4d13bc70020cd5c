// adjoint.cu -- discrete adjoint of a recorded burn.
//
// The rate sensitivity the paper explores by re-running the detonation with
// changed networks (arXiv:2312.02836 Sec. 1 and Sec. 3) is computed here as
// the exact gradient of the discrete map the forward burn applied, with the
// step schedule (t_n, h_n, k_n) frozen and every Newton solution treated as
// exact.  Forward step s solves
//     G_s = alpha_0 x_s + sum_{j=1..k} alpha_j x_{s-j} - h f(x_s; p) = 0,
//     E_s = (h edot(x_s; p) - sum_j alpha_j E_{s-j}) / alpha_0,
// so, walking s = S..1 with cotangents lam_s (of x_s) and e_s (of E_s):
//     lam_s += e_s h / alpha_0 * d edot / dx,   e_{s-j} -= e_s alpha_j / alpha_0
//     (alpha_0 I - h J(x_s))^T mu = lam_s
//     lam_{s-j} -= alpha_j mu
//     dL/dp_r += R_r(x_s) (h c_r^T mu + e_s h / alpha_0 Q_r)
// (plus mu_T Q_r / c_v in c_r^T mu under self-heating, and the temperature
// derivative through g_r = d ln lambda_r / dT9 when T9 is a parameter).
// The tape keeps states only at checkpoints: the reverse sweep takes the steps
// in blocks of the tape's stride, last block first, recomputes each block's
// states forward from its checkpointed history window with the forward's
// own step computation (attempt_solve, so the same bits), then reverses it.
// One lane per zone (k_adjoint), or a team of threads per zone
// (k_adjoint_coop: the same per-zone code with the network spread over the
// team, coop.cuh); K cotangent sets share each LU factorisation.
#include <cuda_runtime.h>
#include <cub/device/device_radix_sort.cuh>

#include <algorithm>
#include <cstring>

#include "blob.h"
#include "adjoint.cuh"
#include "codegen.h"
#include "coop_adjoint.cuh"
#include "device.cuh"
#include "host.h"
#include "../../include/netburn.h"

using namespace nb;

namespace {

__global__ void __launch_bounds__(128) k_adjoint(AdjParams A) {
  extern __shared__ __align__(16) unsigned char sm[];
  const unsigned char* blob = A.blob;
  if (A.blob_in_smem) {
    const int4* src = reinterpret_cast<const int4*>(A.blob);
    int4* dst = reinterpret_cast<int4*>(sm);
    for (int i = threadIdx.x; i < A.blob_bytes / 16; i += blockDim.x) dst[i] = src[i];
    __syncthreads();
    blob = sm;
  }
  const Net t = make_net(blob);
  const int lane = threadIdx.x & 31;
  const long long warp = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  double* lane_base = A.ws + warp * A.lane_doubles * WS_LANES + lane;
  const WS w = make_ws(t, lane_base);
  const AWS a = make_aws(A, lane_base);
  AdjZone Zs;
  Zs.z = -1;
  Zs.s = -1;
  Zs.rs = 1;
  Zs.re = 0;
  Zs.lo = 1;
  Zs.fail = false;
  bool active = false, retired = false, fresh = false;
  for (;;) {
    const unsigned need = __ballot_sync(0xffffffffu, !active && !retired);
    if (need) {
      const int leader = __ffs(need) - 1;
      unsigned long long base = 0;
      if (lane == leader) base = atomicAdd(A.queue, (unsigned long long)__popc(need));
      base = __shfl_sync(0xffffffffu, base, leader);
      if (!active && !retired) {
        const unsigned long long z = base + __popc(need & ((1u << lane) - 1u));
        if (z < (unsigned long long)A.Z) {
          Zs.z = A.order ? (long long)A.order[z] : (long long)z;
          active = true;
          fresh = true;
        } else {
          retired = true;
        }
      }
    }
    if (__all_sync(0xffffffffu, retired)) break;
    if (active) {
      bool done;
      if (fresh) {
        done = adj_init(t, Zs, w, a, A);
        fresh = false;
      } else if (Zs.rs <= Zs.re) {
        done = adj_replay(t, Zs, w, a, A);
      } else {
        done = adj_step(t, Zs, w, a, A);
      }
      if (done) {
        adj_finish(t, Zs, a, A);
        active = false;
      }
    }
  }
}

// One zone per team of P threads.  With C.smem the team's Newton-loop arrays
// and its adjoint arrays sit in shared memory after the (optional) blob copy,
// C.stride doubles per team; else everything is in the workspace.
struct CoopAdj {
  int smem;
  long long stride;
  TeamAdj a;
};

template <int P, int S, int TPB, int MINB>
__global__ void __launch_bounds__(TPB, MINB)
    k_adjoint_coop(const __grid_constant__ AdjParams A, const __grid_constant__ CoopAdj C,
                   const __grid_constant__ BlobHeader H) {
  extern __shared__ __align__(16) unsigned char sm[];
  const unsigned char* blob = A.blob;
  if (A.blob_in_smem) {
    const int4* src = reinterpret_cast<const int4*>(A.blob);
    int4* dst = reinterpret_cast<int4*>(sm);
    for (int i = threadIdx.x; i < A.blob_bytes / 16; i += blockDim.x) dst[i] = src[i];
    __syncthreads();
    blob = sm;
  }
  unsigned char* rest = sm + (A.blob_in_smem ? A.blob_bytes : 0);
  const TNet<P, S> t(BlobDims(blob, H), reinterpret_cast<unsigned long long*>(rest));
  const int tib = threadIdx.x / P;
  const long long team = (long long)blockIdx.x * (blockDim.x / P) + tib;
  const int thot = H.thot, tcold = H.tcold;
  double *hot, *cold;
  if (C.smem) {
    hot = reinterpret_cast<double*>(rest + team_scratch_bytes(P)) + (size_t)tib * C.stride;
    cold = A.ws + team * tcold;
  } else {
    hot = A.ws + team * (C.stride + tcold);
    cold = hot + C.stride;
  }
  CWS w = make_cws(H, hot, cold);
  const TAWS a = make_taws(C.a, hot + thot);
  AdjZone Zs;
  bool active = false;
  for (;;) {
    bool done;
    if (!active) {
      unsigned long long c = 0;
      if (t.lane == 0) c = atomicAdd(A.queue, 1ull);
      c = t.bcast(c);
      if (c >= (unsigned long long)A.Z) break;
      Zs.z = A.order ? (long long)A.order[c] : (long long)c;
      Zs.rs = 1;
      Zs.re = 0;
      Zs.lo = 1;
      done = adj_init(t, Zs, w, a, A);
    } else if (Zs.rs <= Zs.re) {
      done = adj_replay(t, Zs, w, a, A);
    } else {
      done = adj_step(t, Zs, w, a, A);
    }
    active = !done;
    if (done) {
      adj_finish(t, Zs, a, A);
      t.sync();
    }
  }
}

__global__ void k_zone_index(int32_t* idx, long long Z) {
  const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < Z) idx[i] = (int32_t)i;
}

}  // namespace

extern "C" int nb_burn_adjoint(nb_net net, void* tape, int32_t K, const double* gY,
                               const double* gE, const double* gT9, double* d_ln_mult,
                               double* dY0, double* dT0, void* stream) {
  return nb_burn_adjoint_ex(net, tape, K, gY, gE, gT9, d_ln_mult, dY0, dT0, nullptr, stream);
}

extern "C" int nb_burn_adjoint_ex(nb_net net, void* tape, int32_t K, const double* gY,
                                  const double* gE, const double* gT9, double* d_ln_mult,
                                  double* dY0, double* dT0, const nb_options* opt,
                                  void* stream) {
  if (!net || !tape || K < 1 || K > 64 || !gY || !d_ln_mult) return NB_E_ARG;
  nb_tape_s* tp = (nb_tape_s*)tape;
  if (tp->magic != 0x7a9e5eedu || tp->net != net || !tp->recorded) return NB_E_TAPE;
  const BlobHeader& h = net->h;
  const long long Z = tp->recZ;
  if (Z == 0) return NB_OK;
  AdjParams A;
  std::memset(&A, 0, sizeof(A));
  A.blob = net->d_blob;
  A.blob_bytes = h.bytes;
  A.Z = Z;
  A.K = K;
  A.tape = tp->dev;
  A.rtol = tp->rtol;
  A.atol = tp->atol;
  A.lnm = tp->has_lnm ? tp->lnm : nullptr;
  A.lnm_per_zone = tp->lnm_per_zone;
  A.gY = gY; A.gE = gE; A.gT9 = gT9;
  A.dl = d_ln_mult; A.dY0 = dY0; A.dT0 = dT0;
  const int n = h.n;
  long long off = h.lane_doubles;
  A.o_lam = (int)off; off += (long long)HMAX * K * n;
  A.o_ee = (int)off; off += (long long)HMAX * K;
  A.o_gr = (int)off; off += (long long)K * h.R;
  A.o_gt = (int)off; off += K;
  A.o_mu = (int)off; off += n;
  A.o_de = (int)off; off += n;
  A.o_seg = (int)off; off += (long long)tp->dev.stride * n;
  A.lane_doubles = off;
  nb_options o;
  nb_default_options(&o);
  if (opt) o = *opt;
  // the kernel: as asked; else, when blocks are recomputed (stride > 1), the
  // arithmetic of the recording burn, so that the recomputed states are the
  // forward's bits; else one warp per zone from 24 state entries on
  int kernel = o.kernel;
  const bool recompute = tp->dev.stride > 1;
  const bool family_ok = tp->family == NB_KERNEL_COOP || tp->family == NB_KERNEL_PERSISTENT;
  if (!opt || kernel == NB_KERNEL_AUTO) {
    if (recompute && !family_ok) return NB_E_TAPE;   // recorded by teams of warps
    kernel = recompute ? tp->family : (n >= 24 ? NB_KERNEL_COOP : NB_KERNEL_PERSISTENT);
  }
  if (kernel != NB_KERNEL_COOP && kernel != NB_KERNEL_PERSISTENT) return NB_E_ARG;
  if (recompute && kernel != tp->family) return NB_E_TAPE;
  cudaStream_t st = (cudaStream_t)stream;
  std::lock_guard<std::mutex> lk(net->mu);
  const size_t blob_b = (size_t)h.bytes;
  int tpb = 0, in_smem = 0;
  size_t dyn = 0;
  long long blocks = 0;
  CoopAdj C;
  std::memset(&C, 0, sizeof(C));
  const size_t scratch = team_scratch_bytes(64);
  auto team_fn = &k_adjoint_coop<64, 32, 64, 4>;
  size_t per_unit;   // global workspace per lane (lane kernel) or team (coop)
  // A lane-recorded tape by teams in the lane order, the lane kernel's bits.
  // One lane takes 540 ms for its longest zone's reverse sweep whatever the
  // number of zones up to an SM's lanes (self-heating chain, K = 1); with 8,
  // 16, 32 lanes a zone 256 zones take 158, 130, 67 ms; 1,024 (7 an SM) 127,
  // 96, 79; 4,096 (27) 156, 150, 233; 12,000 (79) 241, 354, 605. A large
  // network's zone keeps two warps busy (48 species, 96 zones, K = 2: 6,971
  // ms by lanes, 175 ms). A launch shape asked for is the lane kernel's.
  int lane_team = 0;
  if (kernel == NB_KERNEL_PERSISTENT && o.threads_per_block <= 0 && o.blocks_per_sm <= 0) {
    const long long sm = net->sm_count;
    lane_team = n >= 24 ? 64 : Z <= 12 * sm ? 32 : Z <= 24 * sm ? 16 : Z <= 160 * sm ? 8 : 0;
  }
  int teams = 1;   // zones of a block of teams
  if (lane_team) {
    team_layout(h, K, tp->dev.stride, 0, &C.a);
    C.stride = (h.thot + C.a.total + 7) / 16 * 16 + 8;
    const size_t team_b = (size_t)C.stride * sizeof(double);
    const long long per_sm = (Z + net->sm_count - 1) / net->sm_count;
    // a team of several warps is a block of its own (its barrier and its
    // broadcasts are the block's)
    tpb = lane_team > 32 ? lane_team
                         : (int)std::min<long long>(128, (per_sm * lane_team + 31) / 32 * 32);
    in_smem = blob_b <= 32 * 1024;
    const size_t fixed = (in_smem ? blob_b : 0) + scratch;
    while (lane_team <= 32 && tpb > 32 && fixed + tpb / lane_team * team_b > net->smem_optin) tpb -= 32;
    teams = tpb / lane_team;
    C.smem = fixed + teams * team_b <= net->smem_optin;
    dyn = fixed + (C.smem ? teams * team_b : 0);
    team_fn = lane_team == 8    ? &k_adjoint_coop<8, 0, 128, 2>
              : lane_team == 16 ? &k_adjoint_coop<16, 0, 128, 2>
              : lane_team == 32 ? &k_adjoint_coop<32, 0, 128, 2>
                                : &k_adjoint_coop<64, 0, 64, 4>;
    CK(nb::allow_shared((const void*)team_fn, net->smem_optin));
    int occ = 0;
    CK(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, (const void*)team_fn, tpb, dyn));
    // The lane kernel holds all of an SM's zones at once; teams take them by
    // turns, and the more K and the tape's stride fill their arrays the fewer
    // at a time.  Its time over that of one turn of the teams (self-heating
    // chain, 120 to 160 zones an SM): K = 1, strides 16, 64, 256: 7.4 (32
    // resident: 368 and 550 ms), 6.5 (16: 435 and 380), 5.7 (4: 1,577 and
    // 296); K = 6: 15; K = 16: 23, 17; in global memory, where 32 are
    // resident, 3.7 (K = 1, stride 1,400: 267 and 261 ms), 6, 10 for K = 1,
    // 16, 64.  Networks past the chains (349 statements) more: 16 species
    // (1,462) 20 to 26, 19 species (1,772) and up 51 and more.  A large
    // network's lane takes 20 to 80 times its team's time.
    const long long size = straight_line_size(h), twice = size < 1000 ? 2 : size < 1600 ? 5 : 10;
    const long long turns = (C.smem ? 5 + K : 3 + K / 8) * twice / 2;
    if (occ < 1 || (lane_team <= 32 && per_sm > turns * occ * teams)) {
      lane_team = 0;
    } else {
      blocks = std::min((long long)occ * net->sm_count, (Z + teams - 1) / teams);
      per_unit = (size_t)(h.tcold + (C.smem ? 0 : C.stride)) * 8;
      int rc = nb::ensure(net->ws_adj, net->kept,
                          std::max<size_t>((size_t)blocks * teams * per_unit, 256), st);
      if (rc) return rc;
    }
  }
  if (kernel == NB_KERNEL_COOP) {
    // per team in shared memory: the forward hot arrays and the adjoint's
    const int S = 32;
    team_layout(h, K, tp->dev.stride, S, &C.a);
    C.stride = h.thot + C.a.total;
    const size_t team_b = (size_t)C.stride * sizeof(double);
    // an explicit block of several zones has to fit with one zone per warp
    const int warps = o.threads_per_block / 32;
    if (o.threads_per_block % 32 != 0 || warps > 8) return NB_E_ARG;
    const size_t warp_b = ((size_t)h.hot_doubles + A.lane_doubles - h.lane_doubles) * sizeof(double);
    if (warps > 0 && o.ws_in_shared != 0 && warp_b <= net->smem_optin &&
        warps * warp_b > net->smem_optin)
      return NB_E_TOO_LARGE;
    C.smem = o.ws_in_shared != 0 && team_b + scratch <= net->smem_optin;
    // Threads of a team: a large network's four warps while the longest zone
    // sets the time (up to 8 zones an SM: 1,024 zones of the 48-species
    // network take 226, 220, 184 ms with 1, 2, 4 warps), else two (K = 6, 60
    // zones an SM: 324, 297, 403 ms; K = 1: 201, 210, 361); where two zones'
    // arrays don't fit an SM's shared memory, eight.  Networks with a
    // generated kernel (up to 6,000 statements) past 8 zones an SM one, of
    // which an SM holds eight, and with one or two cotangents always: 28
    // species (4,784 statements), K = 1 and 6, 8 zones an SM 129 and 149 ms
    // (four warps 129 and 141; at stride 1, K = 1, 61 and 79), 30 zones 170
    // and 193 (two 249 and 374).  Below 3,000 statements always (24 species,
    // 2,596 statements, 8 zones an SM 58, 64, 83 ms; the self-heating chain
    // 82, 126, 221).
    const long long size = straight_line_size(h), sm = net->sm_count;
    const int P = C.smem && 2 * (team_b + 1024) > net->smem_optin                     ? 256
                  : size < 3000 || (specialize_auto_ok(h) && (Z > 8 * sm || K < 3)) ? 32
                  : C.smem && Z <= 8 * sm                                             ? 128
                                                                                      : 64;
    tpb = P;
    if (P == 32) {   // several teams a block
      tpb = (int)std::min(128LL, 32 * ((Z + sm - 1) / sm));
      while (C.smem && tpb > 32 && scratch + tpb / 32 * team_b > net->smem_optin) tpb -= 32;
    }
    teams = tpb / P;
    team_fn = P == 256   ? &k_adjoint_coop<256, 32, 256, 1>
              : P == 128 ? &k_adjoint_coop<128, 32, 128, 2>
              : P == 64  ? &k_adjoint_coop<64, 32, 64, 4>
                         : &k_adjoint_coop<32, 32, 128, 2>;
    const size_t arrays_b = C.smem ? teams * team_b : 0;
    in_smem = o.blob_in_shared != 0 && blob_b <= 96 * 1024 &&
              blob_b + scratch + arrays_b <= net->smem_optin;
    dyn = (in_smem ? blob_b : 0) + scratch + arrays_b;
    CK(nb::allow_shared((const void*)team_fn, net->smem_optin));
    int occ = 0;
    CK(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, (const void*)team_fn, tpb, dyn));
    if (occ < 1) return NB_E_TOO_LARGE;
    const int bps = o.blocks_per_sm > 0 ? nb::team_blocks(o.blocks_per_sm, warps, teams) : occ;
    blocks = std::min(std::min(bps, occ) * sm, (Z + teams - 1) / teams);
    per_unit = (size_t)(h.tcold + (C.smem ? 0 : C.stride)) * 8;
    int rc = nb::ensure(net->ws_adj, net->kept,
                        std::max<size_t>((size_t)blocks * teams * per_unit, 256), st);
    if (rc) return rc;
  } else if (!lane_team) {
    // one zone per lane; smaller blocks when there are few zones per SM
    const long long per_sm = (Z + net->sm_count - 1) / net->sm_count;
    tpb = o.threads_per_block > 0 ? o.threads_per_block
                                  : (per_sm >= 128 ? 128 : (int)std::max(32LL, per_sm / 32 * 32));
    if (tpb % 32 != 0 || tpb > 128) return NB_E_ARG;
    in_smem = blob_b <= 96 * 1024 ? 1 : 0;
    dyn = in_smem ? blob_b : 0;
    if (dyn > 48 * 1024)
      CK(nb::allow_shared((const void*)k_adjoint, net->smem_optin));
    int occ = 0;
    CK(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, k_adjoint, tpb, dyn));
    blocks = (long long)std::max(1, std::min(o.blocks_per_sm > 0 ? o.blocks_per_sm : 2, occ)) *
             net->sm_count;
    const long long needed = (Z + tpb - 1) / tpb;
    if (blocks > needed) blocks = needed;
    per_unit = (size_t)A.lane_doubles * sizeof(double);
    int rc = nb::ensure(net->ws_adj, net->kept, (size_t)blocks * tpb * per_unit, st);
    if (rc) return rc;
  }
  int rc = NB_OK;
  A.ws = net->ws_adj.p;
  A.queue = net->queue + 1;   // a second counter in the same allocation
  A.blob_in_smem = in_smem;
  // Claim order: the tape holds every zone's step count, the exact length of
  // its reverse sweep, so zones are claimed longest first and the last lanes
  // to finish run short zones (one lane per zone otherwise waits on the
  // longest zone).
  if (Z > 1 && Z <= 0x7fffffffLL) {
    size_t temp = 0;
    CK(cub::DeviceRadixSort::SortPairsDescending(nullptr, temp, (const int32_t*)nullptr,
                                                 (int32_t*)nullptr, (const int32_t*)nullptr,
                                                 (int32_t*)nullptr, (int)Z, 0, 32, st));
    auto al = [](size_t b) { return (b + 255) & ~size_t(255); };
    const size_t ib = al((size_t)Z * 4);
    rc = nb::ensure(net->sched_adj, net->kept, 3 * ib + al(temp), st);
    if (rc) return rc;
    int32_t* k_out = (int32_t*)net->sched_adj.p;
    int32_t* i_in = (int32_t*)(net->sched_adj.p + ib);
    int32_t* i_out = (int32_t*)(net->sched_adj.p + 2 * ib);
    k_zone_index<<<(unsigned)((Z + 255) / 256), 256, 0, st>>>(i_in, Z);
    CK(cudaGetLastError());
    CK(cub::DeviceRadixSort::SortPairsDescending(net->sched_adj.p + 3 * ib, temp, tp->dev.steps,
                                                 k_out, i_in, i_out, (int)Z, 0, 32, st));
    A.order = i_out;
  }
  CK(cudaMemsetAsync(A.queue, 0, sizeof(unsigned long long), st));
  if (kernel == NB_KERNEL_COOP || lane_team)
    team_fn<<<(unsigned)blocks, tpb, dyn, st>>>(A, C, h);
  else
    k_adjoint<<<(unsigned)blocks, tpb, dyn, st>>>(A);
  CK(cudaGetLastError());
  return NB_OK;
}
