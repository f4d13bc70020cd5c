// multi.cu -- several networks burned in one launch.
//
// The paper's study burns the same hydro zones with different networks
// (aprox13-like, subch_simple, He-C-Fe; arXiv:2312.02836 Sec. 3 and 4) to see
// which nuclear physics matters.  nb_burn_multi takes up to
// NB_MULTI_MAX_SETS (network, zones) sets and runs them in one persistent
// launch (two when many zones of small networks come with a large one): all
// lanes of the GPU claim from one device queue that spans every set's zones,
// so a set of few expensive zones and a set of many cheap ones keep the same
// warps busy.  Each lane (or, with few zones or a large network, each team of
// lanes) reads the compiled network of the zone it claimed and runs the
// generic integrator, so every zone gives the same bits as a single-network
// burn.
#include <cuda_runtime.h>
#include <cub/device/device_segmented_radix_sort.cuh>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <mutex>
#include <vector>

#include "blob.h"
#include "coop.cuh"
#include "device.cuh"
#include "host.h"
#include "../../include/netburn.h"

using namespace nb;

namespace {

struct MultiParams {
  int n;                                  // sets, in claim order
  long long off[NB_MULTI_MAX_SETS + 1];   // first claim index of each set
  BurnParams p[NB_MULTI_MAX_SETS];
  double* ws;                             // per-lane workspace, max lane_doubles
  int lane_doubles;
  unsigned long long* queue;
  unsigned long long budget_ns;
  const int32_t* order;                   // claim position -> claim index, or null
};
// passed by value as the kernel's parameter block (the classic 4 KB limit)
static_assert(sizeof(MultiParams) <= 4000, "MultiParams exceeds the kernel parameter space");

__global__ void __launch_bounds__(128, 1) k_burn_multi(const __grid_constant__ MultiParams M) {
  const int lane = threadIdx.x & 31;
  const long long warp = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  double* lane_base = M.ws + warp * (long long)M.lane_doubles * WS_LANES + lane;
  const long long total = M.off[M.n];
  Zone s;
  s.z = -1;
  int m = 0;
  bool active = false, retired = false, fresh = false;
  const unsigned long long t_start = M.budget_ns ? gpu_ns() : 0ull;
  for (;;) {
    const unsigned need = __ballot_sync(0xffffffffu, !active && !retired);
    if (need) {
      const int leader = __ffs(need) - 1;
      unsigned long long base = 0;
      if (lane == leader) base = atomicAdd(M.queue, (unsigned long long)__popc(need));
      base = __shfl_sync(0xffffffffu, base, leader);
      if (!active && !retired) {
        const unsigned long long c = base + __popc(need & ((1u << lane) - 1u));
        if (c < (unsigned long long)total) {
          // the order keeps every position within its own set's range
          const long long ci = M.order ? (long long)M.order[c] : (long long)c;
          m = 0;
          while (m + 1 < M.n && ci >= M.off[m + 1]) ++m;
          s.z = ci - M.off[m];
          active = true;
          fresh = true;
        } else {
          retired = true;
        }
      }
    }
    if (__all_sync(0xffffffffu, retired)) break;
    if (active) {
      const BurnParams& P = M.p[m];
      const Net t = make_net(P.blob);
      WS w = make_ws(t, lane_base);
      const bool expired = M.budget_ns && gpu_ns() - t_start > M.budget_ns;
      bool done;
      if (expired && fresh) {
        zone_timeout_unstarted(t, s.z, P);
        fresh = false;
        active = false;
        continue;
      }
      if (expired) {
        s.status = NB_Z_TIMEOUT;
        done = true;
      } else if (fresh) {
        done = zone_init(t, s, w, P);
        fresh = false;
      } else {
        done = zone_attempt(t, s, w, P);
      }
      if (done) {
        zone_finish(t, s, w, P);
        active = false;
      }
    }
  }
}

// The same queue served by teams of P threads in the lane order (coop.cuh),
// which gives the same bits.  A team's arrays are in shared memory, sized for
// the largest network (f0 and the history too when cold_smem); the compiled
// networks are copied there when they all fit.
struct MultiTeams {
  MultiParams M;
  BlobHeader H[NB_MULTI_MAX_SETS];
  int blob_at[NB_MULTI_MAX_SETS];   // byte offset in shared memory, or -1
  int blob_bytes;                   // of all the copies
  int stride;                       // doubles from one team's arrays to the next
  int cold_smem, cold_doubles;
};

template <int P>
__global__ void __launch_bounds__(128, 2) k_multi_team(const __grid_constant__ MultiTeams T) {
  extern __shared__ __align__(16) unsigned char sm[];
  const MultiParams& M = T.M;
  for (int m = 0; m < M.n; ++m) {
    if (T.blob_at[m] < 0) continue;
    const int4* src = reinterpret_cast<const int4*>(M.p[m].blob);
    int4* dst = reinterpret_cast<int4*>(sm + T.blob_at[m]);
    for (int i = threadIdx.x; i < T.H[m].bytes / 16; i += blockDim.x) dst[i] = src[i];
  }
  __syncthreads();
  const int tib = threadIdx.x / P;
  const long long team = (long long)blockIdx.x * (blockDim.x / P) + tib;
  double* hot = reinterpret_cast<double*>(sm + T.blob_bytes) + (size_t)tib * T.stride;
  double* cold = M.ws + team * T.cold_doubles;
  const unsigned long long total = (unsigned long long)M.off[M.n];
  const bool lead = threadIdx.x % P == 0;
  const unsigned mask =
      P >= 32 ? 0xffffffffu : ((1u << (P & 31)) - 1u) << (threadIdx.x & 31 & ~(P - 1));
  // the team's watchdog starts at thread 0's clock and reads it: threads that
  // each read their own could decide apart, and part at a shuffle
  unsigned long long t_start = 0ull;
  if (M.budget_ns) t_start = __shfl_sync(mask, lead ? gpu_ns() : 0ull, 0, P);
  Zone s;
  int m = 0;
  bool active = false;
  for (;;) {
    if (!active) {
      unsigned long long c = 0;
      if (lead) c = atomicAdd(M.queue, 1ull);
      c = __shfl_sync(mask, c, 0, P);
      if (c >= total) break;
      // the order keeps every position within its own set's range
      const long long ci = M.order ? (long long)M.order[c] : (long long)c;
      m = 0;
      while (m + 1 < M.n && ci >= M.off[m + 1]) ++m;
      s.z = ci - M.off[m];
    }
    const BurnParams& B = M.p[m];
    const BlobHeader& H = T.H[m];
    const TNet<P, 0> t(BlobDims(T.blob_at[m] < 0 ? B.blob : sm + T.blob_at[m], H), nullptr);
    CWS w = make_cws(H, hot, T.cold_smem ? hot + H.thot : cold);
    bool expired = false;
    if (M.budget_ns) expired = t.bcast(lead ? gpu_ns() : 0ull) - t_start > M.budget_ns;
    bool done;
    if (expired) {
      if (!active) {
        zone_timeout_unstarted(t, s.z, B);
        continue;
      }
      s.status = NB_Z_TIMEOUT;
      done = true;
    } else {
      done = active ? zone_attempt(t, s, w, B) : zone_init(t, s, w, B);
    }
    active = !done;
    if (done) {
      zone_finish(t, s, w, B);
      t.sync();
    }
  }
}

// Scheduling pre-pass: every zone's starting step h0 (the integrator's own
// start-up) as the key of its claim index; zones that finish in start-up go
// last.  Sorted within each set, the keys give each set's zones longest
// first, so a warp's lanes get zones of alike length.
__global__ void __launch_bounds__(128, 1) k_multi_estimate(const __grid_constant__ MultiParams M,
                                                          double* key, int32_t* idx) {
  const int lane = threadIdx.x & 31;
  const long long warp = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  double* lane_base = M.ws + warp * (long long)M.lane_doubles * WS_LANES + lane;
  const long long total = M.off[M.n];
  const long long stride = (long long)gridDim.x * blockDim.x;
  for (long long c = (long long)blockIdx.x * blockDim.x + threadIdx.x; c < total; c += stride) {
    int m = 0;
    while (m + 1 < M.n && c >= M.off[m + 1]) ++m;
    const BurnParams& P = M.p[m];
    const Net t = make_net(P.blob);
    WS w = make_ws(t, lane_base);
    Zone s;
    s.z = c - M.off[m];
    const bool done = zone_init(t, s, w, P);
    key[c] = done ? 1e300 : s.h;
    idx[c] = (int32_t)c;
  }
}

// a cost proxy per zone of a network: sets with larger networks are claimed
// first, so their long zones start early
long long set_cost(const nb_net net) {
  const BlobHeader& h = net->h;
  return (long long)h.nnz * 4 + (long long)h.nd + (long long)h.R * 8;
}

// Where the teams' arrays of the sets ord[0..n) go, P threads a zone: T's
// header, the threads of a block and its shared memory.  False when a zone's
// arrays don't fit.
bool team_layout(const nb_burn_set* sets, const int* ord, int n, long long total, int P,
                 MultiTeams* T, int* threads, size_t* dyn) {
  const nb_net_s& host = *sets[ord[0]].net;
  std::memset(T, 0, sizeof(*T));
  int hot = 0, all = 0, cold = 0, bytes = 0;
  for (int k = 0; k < n; ++k) {
    const BlobHeader& h = sets[ord[k]].net->h;
    T->H[k] = h;
    hot = std::max(hot, h.thot);
    cold = std::max(cold, h.tcold);
    all = std::max(all, h.thot + h.tcold);
    T->blob_at[k] = bytes;
    bytes += h.bytes;
  }
  const bool copy = bytes <= 48 * 1024;
  for (int k = 0; k < n && !copy; ++k) T->blob_at[k] = -1;
  T->blob_bytes = copy ? bytes : 0;
  T->cold_smem = all <= 1024;
  T->cold_doubles = T->cold_smem ? 0 : cold;
  T->stride = ((T->cold_smem ? all : hot) + 7) / 16 * 16 + 8;
  const size_t team_b = (size_t)T->stride * sizeof(double);
  const long long per_sm = (total + host.sm_count - 1) / host.sm_count;
  *threads = (int)std::min<long long>(128, (per_sm * P + 31) / 32 * 32);
  while (*threads > 32 && T->blob_bytes + *threads / P * team_b > host.smem_optin) *threads -= 32;
  *dyn = T->blob_bytes + *threads / P * team_b;
  return *dyn <= host.smem_optin;
}

// One launch over the sets ord[0..n), P threads a zone (0, or when a zone's
// arrays don't fit: the lane kernel).  `host` lends its workspace and queue
// counter; the caller holds its lock.
int launch_sets(nb_net host, const nb_burn_set* sets, const int* ord, int n, double t_end,
                double rtol, double atol, const nb_options& o, int P, cudaStream_t st) {
  const int tpb = o.threads_per_block > 0 ? o.threads_per_block : 128;
  MultiParams M;
  std::memset(&M, 0, sizeof(M));
  M.n = n;
  M.budget_ns = o.time_budget_s > 0.0 ? (unsigned long long)(o.time_budget_s * 1e9) + 1ull : 0ull;
  long long total = 0;
  int lane_doubles = 1;
  for (int k = 0; k < n; ++k) {
    const nb_burn_set& b = sets[ord[k]];
    BurnParams& p = M.p[k];
    M.off[k] = total;
    total += b.Z;
    lane_doubles = std::max(lane_doubles, (int)b.net->h.lane_doubles);
    p.blob = b.net->d_blob;
    p.blob_bytes = b.net->h.bytes;
    p.Z = b.Z;
    p.Y0 = b.Y0; p.T9_0 = b.T9_0; p.rho = b.rho;
    p.t_end = t_end; p.rtol = rtol; p.atol = atol;
    p.lnm = b.ln_mult; p.lnm_per_zone = b.ln_mult_per_zone ? 1 : 0;
    p.Y = b.Y; p.T9 = b.T9; p.E = b.E; p.counters = b.counters; p.status = b.status;
    p.max_attempts = o.max_attempts;
    p.t_end_zone = b.t_end_zone;
    p.zeta_zone = b.zeta_zone;
  }
  M.off[n] = total;
  M.lane_doubles = lane_doubles;
  const long long sm = host->sm_count;
  int occ = 0;
  CK(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, k_burn_multi, tpb, 0));
  if (occ < 1) return NB_E_TOO_LARGE;
  const int bps = std::max(1, std::min(o.blocks_per_sm > 0 ? o.blocks_per_sm : 1, occ));
  const long long blocks = std::min(bps * sm, (total + tpb - 1) / tpb);
  MultiTeams T;
  int t_threads = 0;
  long long t_blocks = 0;
  size_t t_dyn = 0, t_ws = 0;
  auto t_fn = P == 8 ? &k_multi_team<8> : P == 16 ? &k_multi_team<16> : &k_multi_team<32>;
  if (P && !team_layout(sets, ord, n, total, P, &T, &t_threads, &t_dyn)) P = 0;
  if (P) {
    int t_occ = 0;
    CK(nb::allow_shared((const void*)t_fn, host->smem_optin));
    CK(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&t_occ, (const void*)t_fn, t_threads, t_dyn));
    if (t_occ < 1) {
      P = 0;
    } else {
      const int teams = t_threads / P;
      t_blocks = std::min(t_occ * sm, (total + teams - 1) / teams);
      t_ws = (size_t)t_blocks * teams * T.cold_doubles * sizeof(double);
    }
  }
  const size_t need =
      std::max(t_ws, (size_t)blocks * tpb * lane_doubles * sizeof(double));
  int rc = nb::ensure(host->ws, host->kept, need, st);
  if (rc) return rc;
  M.ws = host->ws.p;
  M.queue = host->queue;
  M.order = nullptr;
  if (o.schedule == 1 && total > 1 && total <= 0x7fffffffLL) {
    // longest first within each set (segments at the sets' claim offsets)
    int seg[NB_MULTI_MAX_SETS + 1];
    for (int k = 0; k <= n; ++k) seg[k] = (int)M.off[k];
    size_t temp = 0;
    CK(cub::DeviceSegmentedRadixSort::SortPairs(
        nullptr, temp, (const double*)nullptr, (double*)nullptr, (const int32_t*)nullptr,
        (int32_t*)nullptr, (int)total, n, seg, seg + 1, 0, 64, st));
    auto al = [](size_t b) { return (b + 255) & ~size_t(255); };
    const size_t kb = al((size_t)total * 8), ib = al((size_t)total * 4);
    const size_t sb = al(sizeof(seg));
    rc = nb::ensure(host->sched, host->kept, 2 * kb + 2 * ib + sb + al(temp), st);
    if (rc) return rc;
    unsigned char* base = host->sched.p;
    double* k_in = (double*)base;
    double* k_out = (double*)(base + kb);
    int32_t* i_in = (int32_t*)(base + 2 * kb);
    int32_t* i_out = (int32_t*)(base + 2 * kb + ib);
    int* d_seg = (int*)(base + 2 * kb + 2 * ib);
    void* tmp = base + 2 * kb + 2 * ib + sb;
    CK(cudaMemcpyAsync(d_seg, seg, sizeof(seg), cudaMemcpyHostToDevice, st));
    k_multi_estimate<<<(unsigned)blocks, tpb, 0, st>>>(M, k_in, i_in);
    CK(cudaGetLastError());
    CK(cub::DeviceSegmentedRadixSort::SortPairs(tmp, temp, k_in, k_out, i_in, i_out, (int)total,
                                                n, d_seg, d_seg + 1, 0, 64, st));
    M.order = i_out;
  }
  CK(cudaMemsetAsync(host->queue, 0, sizeof(unsigned long long), st));
  if (P) {
    T.M = M;
    t_fn<<<(unsigned)t_blocks, t_threads, t_dyn, st>>>(T);
  } else {
    k_burn_multi<<<(unsigned)blocks, tpb, 0, st>>>(M);
  }
  CK(cudaGetLastError());
  return NB_OK;
}

}  // namespace

extern "C" int nb_burn_multi(int32_t n_sets, const nb_burn_set* sets, double t_end,
                             double rtol, double atol, const nb_options* opt, void* stream) {
  if (n_sets < 1 || n_sets > NB_MULTI_MAX_SETS || !sets) return NB_E_ARG;
  if (!(rtol > 0.0) || !(atol > 0.0) || !(t_end >= 0.0) || !std::isfinite(t_end)) return NB_E_ARG;
  nb_options o;
  nb_default_options(&o);
  if (opt) o = *opt;
  if (o.max_attempts <= 0 || !(o.time_budget_s >= 0.0)) return NB_E_ARG;
  const int tpb = o.threads_per_block > 0 ? o.threads_per_block : 128;
  if (tpb % 32 != 0 || tpb > 128) return NB_E_ARG;
  int dev = 0;
  CK(cudaGetDevice(&dev));
  long long total = 0, large = 0;   // zones; those of large networks
  for (int i = 0; i < n_sets; ++i) {
    const nb_burn_set& b = sets[i];
    if (!b.net || b.Z < 0 || b.net->device != dev) return NB_E_ARG;
    if (b.Z > 0 && (!b.Y0 || !b.T9_0 || !b.rho || !b.Y || !b.T9 || !b.status)) return NB_E_ARG;
    total += b.Z;
    if (b.net->h.n >= 24) large += b.Z;
  }
  if (total == 0) return NB_OK;
  // claim order: larger networks first
  int ord[NB_MULTI_MAX_SETS];
  for (int i = 0; i < n_sets; ++i) ord[i] = i;
  auto by_cost = [&](int a, int b) { return set_cost(sets[a].net) > set_cost(sets[b].net); };
  std::stable_sort(ord, ord + n_sets, by_cost);
  // the first set's network lends its workspace and queue counter
  nb_net host = sets[0].net;
  cudaStream_t st = (cudaStream_t)stream;
  std::lock_guard<std::mutex> lk(host->mu);
  // Lanes per zone, 0 for the lane kernel above, which takes 236 to 260 ms for
  // three chain networks of any 64 to 4,000 zones each (its longest zone):
  // 3 x 64 zones take 44 ms with 32 lanes, 3 x 500 (10 an SM) 59 ms with 16;
  // with 8 lanes an SM does a zone in 2 ms, so the two meet near 100 an SM.
  // A launch shape asked for is the lane kernel's.
  const long long sm = host->sm_count, small = total - large;
  const bool shaped = o.threads_per_block > 0 || o.blocks_per_sm > 0;
  auto lanes = [&](long long zones) {
    return shaped ? 0 : zones <= 5 * sm ? 32 : zones <= 12 * sm ? 16 : zones <= 100 * sm ? 8 : 0;
  };
  if (shaped || large == 0)
    return launch_sets(host, sets, ord, n_sets, t_end, rtol, atol, o, lanes(total), st);
  // With a large network a warp per zone: one lane takes 2.4 s for a zone of
  // 48 species (4,096 chain and 512 such zones 2,750 ms, by teams 168 ms).  A
  // warp is too much for a small network's zone, though, once there are many:
  // 34 us a chain's zone, and the lane kernel takes no longer for 16,384 with
  // 16 of 48 species (570 ms) and half as long for 32,768 (581 and 1,140 ms).
  // So past 40 small zones an SM the large networks go first, by teams, and
  // the others follow in a launch of their own: 512 zones of 48 species and
  // 27, 40, 108, 215 chain zones an SM take 169, 235, 590, 1,150 ms together,
  // 190, 224, 325, 484 ms one after the other.  (With a watchdog, whose
  // budget is the call's, or arrays that don't fit teams: one launch of
  // lanes.)
  if (small <= 40 * sm)
    return launch_sets(host, sets, ord, n_sets, t_end, rtol, atol, o, 32, st);
  const int n_large = (int)(std::stable_partition(ord, ord + n_sets, [&](int i) {
                              return sets[i].net->h.n >= 24;
                            }) - ord);
  MultiTeams T;
  int threads = 0;
  size_t dyn = 0;
  if (o.time_budget_s > 0.0 || !team_layout(sets, ord, n_large, large, 32, &T, &threads, &dyn)) {
    std::stable_sort(ord, ord + n_sets, by_cost);
    return launch_sets(host, sets, ord, n_sets, t_end, rtol, atol, o, 0, st);
  }
  const int rc = launch_sets(host, sets, ord, n_large, t_end, rtol, atol, o, 32, st);
  return rc ? rc : launch_sets(host, sets, ord + n_large, n_sets - n_large, t_end, rtol, atol, o,
                               lanes(small), st);
}
