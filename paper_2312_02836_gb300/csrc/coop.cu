// coop.cu -- the persistent kernels that give a zone to a team of threads
// (coop.cuh), and their launches.
#include <cuda_runtime.h>

#include <algorithm>

#include "blob.h"
#include "codegen.h"
#include "coop_kernel.cuh"
#include "host.h"
#include "../../include/netburn.h"

using namespace nb;

namespace {

// All forms take the registers they want (254): a 168-register form for
// three blocks of four warps per SM, which the earlier kernel gained from,
// spills and ran 1030 ms where this one, with two blocks, takes 936 ms (48
// species, 65,536 zones).
const TeamKernel kTeamKernels[] = {
    NB_TEAM(32, 32, 0, 256, 1),
    NB_TEAM(32, 32, 1, 256, 1),
    NB_TEAM(64, 32, 1, 64, 4),
    NB_TEAM(128, 32, 1, 128, 2),
};

const TeamKernel& team_kernel(int P, int S, int mem) {
  const TeamKernel* hit = kTeamKernels;
  for (const TeamKernel& k : kTeamKernels)
    if (k.P == P && k.S == S && k.mem == mem) hit = &k;
  for (int i = 0; i < nb::kOtherTeams; ++i) {
    const TeamKernel& k = nb::kOtherTeamKernels[i];
    if (k.P == P && k.S == S && k.mem == mem) hit = &k;
  }
  return *hit;
}

// Launch kernel k with `threads` per block (a multiple of its P), at most
// `bps` blocks per SM (0: as many as fit).
int launch_team(nb_net net, BurnParams& P, const nb_options& o, const TeamKernel& k, int threads,
                int bps, int in_smem, cudaStream_t st) {
  const int teams = threads / k.P;
  const size_t blob_b = in_smem ? (size_t)net->h.bytes : 0;
  const int stride = k.mem == 0 ? 0 : net->h.thot;
  const size_t dyn = blob_b + team_scratch_bytes(k.P) + (size_t)teams * stride * sizeof(double);
  if (dyn > net->smem_optin) return NB_E_TOO_LARGE;
  CK(nb::allow_shared((const void*)k.fn, net->smem_optin));
  int occ = 0;
  CK(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, (const void*)k.fn, threads, dyn));
  if (occ < 1) return NB_E_TOO_LARGE;
  long long blocks = (long long)std::max(1, std::min(bps > 0 ? bps : occ, occ)) * net->sm_count;
  blocks = std::min(blocks, (P.Z + teams - 1) / teams);
  const size_t per_team =
      8 * ((size_t)(k.mem == 0 ? net->h.thot : 0) + net->h.tcold);
  size_t need = std::max<size_t>((size_t)blocks * teams * per_team, 256);
  if (o.schedule == 1) need = std::max(need, nb::prepass_bytes(net, P.Z));
  int rc = nb::ensure(net->ws, net->kept, need, st);
  if (rc) return rc;
  P.ws = net->ws.p;
  P.queue = net->queue;
  P.blob_in_smem = in_smem;
  P.smem_warps = stride;
  P.order = nullptr;
  if (o.schedule == 1 && P.Z > 1) {
    rc = nb::schedule_longest_first(net, P, st);
    if (rc) return rc;
  }
  CK(cudaMemsetAsync(net->queue, 0, sizeof(unsigned long long), st));
  k.fn<<<(unsigned)blocks, threads, dyn, st>>>(P, net->h);
  CK(cudaGetLastError());
  return NB_OK;
}

// Whether the options' shape fits: a zone's Newton-loop arrays as the lane
// kernels lay them out, `warps` such zones a block (0: as few as one) or one
// with the partial sums of wpz warps, and the blob when it is asked for (left
// to the library it stays out where it doesn't fit).  Teams keep a little more
// a zone; where that alone is too much, the arrays go to the workspace.
bool coop_shape_fits(nb_net net, const nb_options& o, int wpz, int warps) {
  const size_t zone_b = (size_t)net->h.hot_doubles * sizeof(double);
  const size_t blob_b = o.blob_in_shared > 0 ? (size_t)net->h.bytes : 0;
  const size_t red = wpz > 1 ? (2 * wpz + 1) * sizeof(double) : 0;
  const bool hot = o.ws_in_shared != 0 && zone_b + red <= net->smem_optin;
  return blob_b + red + (hot ? std::max(warps, 1) * zone_b : 0) <= net->smem_optin;
}

}  // namespace

// Sums in team order of S = 32 x warps_per_zone partial sums.
// threads_per_block (default: the warps whose Newton-loop arrays fit in
// shared memory, at most 4 of them) and blocks_per_sm bound the zones in
// flight; ws_in_shared 0 keeps all arrays in global memory, otherwise
// (default) in shared memory when they fit; blob_in_shared as for the
// persistent kernel.  The threads P of a team follow the work and the zones:
//  * a large network (1,000 and more update pairs a pivot, 128 species:
//    1,763) keeps eight warps busy whatever the number of zones: 300 zones
//    take 492 ms with two warps, 296 ms with eight (128 species, S = 64);
//    one warp and four (S = 32): 247 and 123 ms.  Two teams of eight warps
//    don't fit an SM's registers, so with S = 32, for which a zone has one
//    of several warps of a block's, it is four;
//  * else (48 species: 238 pairs) one warp a zone does the most zones per
//    second (16,384 zones 237 ms, two warps 560 ms), but with few zones per
//    SM the longest zone sets the time, and two or four warps shorten it:
//    16 zones 100, 84, 77 ms with 1, 2, 4 warps; 912 zones 100, 84, 82 ms;
//    2,048 zones 108, 83, 83 ms; 4,096 zones 110, 167, 168 ms;
//  * below 2,000 statements (the chains, 16 species: 1,462) a zone has little
//    to give a second warp, and an SM holds two teams of four warps or four
//    of two against eight warps: always one (self-heating chain, zones an
//    SM: 1: 45, 45, 47 ms with 1, 2, 4 warps, 6: 52, 86, 138; 16 species at
//    6: 79, 93, 135; 22 species, 2,737 statements, at 1: 38, 35, 35).
// threads_per_block and blocks_per_sm count a warp a zone, however many
// threads share one here.
int nb::launch_coop(nb_net net, BurnParams& P, const nb_options& o, cudaStream_t st) {
  const size_t blob_b = (size_t)net->h.bytes;
  const size_t hot_team = (size_t)net->h.thot * sizeof(double);
  const int wpz = o.warps_per_zone <= 1 ? 1 : o.warps_per_zone;
  if (o.warps_per_zone < 0 || (wpz != 1 && wpz != 2 && wpz != 4)) return NB_E_ARG;
  if (wpz == 1 && o.threads_per_block > 0 &&
      (o.threads_per_block % 32 != 0 || o.threads_per_block > 256))
    return NB_E_ARG;
  const int warps_asked = wpz == 1 && o.threads_per_block > 0 ? o.threads_per_block / 32 : 0;
  if (!coop_shape_fits(net, o, wpz, warps_asked)) return NB_E_TOO_LARGE;
  const size_t scratch = team_scratch_bytes(64);
  // a blob asked for in shared memory goes first
  const size_t blob_asked = o.blob_in_shared > 0 ? blob_b : 0;
  const bool hot_smem =
      o.ws_in_shared != 0 && blob_asked + hot_team + scratch <= net->smem_optin;
  int in_smem = o.blob_in_shared;
  if (in_smem < 0)
    in_smem = blob_b <= 96 * 1024 && blob_b + (hot_smem ? hot_team : 0) + scratch <= net->smem_optin;
  const size_t fixed = (in_smem ? blob_b : 0) + scratch;
  const int S = 32 * wpz;
  const bool large = net->h.nD >= 1024 * net->h.n;
  int T = S;
  if (hot_smem) {
    if (large) T = wpz == 1 ? 128 : 256;
    else if (wpz == 1 && straight_line_size(net->h) >= 2000)
      T = P.Z <= 6LL * net->sm_count ? 128 : P.Z <= 16LL * net->sm_count ? 64 : 32;
  }
  int threads = T;
  if (T == 32) {
    int warps = warps_asked > 0 ? warps_asked : 4;
    if (hot_smem)
      while (warps > 1 && fixed + (size_t)warps * hot_team > net->smem_optin) --warps;
    threads = 32 * warps;
  }
  int bps = o.blocks_per_sm;
  if (bps > 0 && wpz == 1) bps = nb::team_blocks(bps, warps_asked, threads / T);
  return launch_team(net, P, o, team_kernel(T, S, hot_smem ? 1 : 0), threads, bps, in_smem, st);
}

// A persistent burn of a large network without a generated kernel by teams in
// the lane order, the generic lane kernel's bits: one lane takes 2.7 ms a
// step attempt of the 48-species network and its lanes' arrays leave L2
// (16,384 zones 3,940 ms, 328 ms by teams).  False when a zone's arrays don't
// fit in shared memory.
bool nb::launch_lane_teams(nb_net net, BurnParams& P, const nb_options& o, cudaStream_t st, int* rc) {
  const size_t hot_team = (size_t)net->h.thot * sizeof(double);
  const size_t scratch = team_scratch_bytes(64);
  if (hot_team + scratch > net->smem_optin) return false;
  const bool wide = net->h.nD >= 1024 * net->h.n || P.Z <= 6LL * net->sm_count;
  int threads = 128;
  if (!wide)
    while (threads > 32 && scratch + threads / 32 * hot_team > net->smem_optin) threads -= 32;
  *rc = launch_team(net, P, o, team_kernel(wide ? 128 : 32, 0, 1), threads, 0, 0, st);
  return true;
}
