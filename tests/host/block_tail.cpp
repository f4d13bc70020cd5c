// block_tail.cpp -- the end of a block of the generated lane kernel
// (block_done: the barrier of every turn, the packing of the last zones) run
// on the host, one fibre per thread of the block.  Test infrastructure: the
// fibres switch only at barriers and ballots, and at each switch the runnable
// thread of the first warp in a given order goes on, so a warp may run ahead
// of the others as far as the barriers let it.  A barrier that threads reach
// at different places, a thread that never gets past one, and a zone that is
// lost, run twice or run with another zone's arrays are reported.
#include <ucontext.h>

#include <cmath>
#include <cstdint>
#include <cstring>
#include <vector>

#define NB_HD
#define NB_EMULATED_BLOCK
#define __host__
#define __device__
#define __forceinline__ inline
#define __shared__ static
#define __syncthreads() barrier(__LINE__, false)
#define __syncthreads_or(p) barrier(__LINE__, p)

namespace {

constexpr int MAXT = 256;
constexpr size_t STACK = 64 << 10;

struct Fibre {
  ucontext_t ctx;
  std::vector<char> stack;
  int site = 0;          // barrier (line) or ballot (-1) it waits at, 0 running
  bool pred = false, done = false;
};

struct Dim { int x; } threadIdx, blockDim;
Fibre fib[MAXT];
ucontext_t sched;
int cur;
unsigned warp_bits[MAXT / 32];
unsigned long long shfl_val[MAXT];
bool block_or;

void wait_at(int site, bool pred) {
  fib[cur].site = site;
  fib[cur].pred = pred;
  const int me = cur;
  swapcontext(&fib[me].ctx, &sched);
}
bool barrier(int line, bool pred) {
  wait_at(line, pred);
  return block_or;
}
unsigned __ballot_sync(unsigned, bool pred) {
  wait_at(-1, pred);
  return warp_bits[threadIdx.x >> 5];
}
bool __all_sync(unsigned, bool pred) { return __ballot_sync(~0u, pred) == ~0u; }
unsigned long long __shfl_sync(unsigned, unsigned long long v, int src) {
  shfl_val[threadIdx.x] = v;
  __ballot_sync(~0u, false);
  const unsigned long long r = shfl_val[(threadIdx.x & ~31) + src];
  __ballot_sync(~0u, false);
  return r;
}
unsigned long long atomicAdd(unsigned long long* p, unsigned long long v) {
  const unsigned long long o = *p;
  *p += v;
  return o;
}
int __popc(unsigned x) { return __builtin_popcount(x); }
int __ffs(unsigned x) { return __builtin_ffs((int)x); }

}  // namespace

#include "../../paper_2312_02836_gb300/csrc/integrator.cuh"

// A network whose zones take a given number of turns: the first starts a
// zone, the others attempt a step.
namespace nb {

struct TurnNet {
  static constexpr bool in_step = true;
  static constexpr int lane_doubles = 3;
};
std::vector<long long> held;   // the zone whose history an array holds
struct TurnWS {
  long long at;   // this lane's arrays
  void take(long long d) { held[at] = held[at + d]; }
};

const int* turns;        // turns zone z needs
std::vector<int> ran;    // turns it got
std::vector<int> ended;
int error;

bool turn(Zone& s, TurnWS& w) {
  if (held[w.at] != s.z) error |= 4;
  return ++ran[s.z] >= turns[s.z];
}
bool zone_init(const TurnNet&, Zone& s, TurnWS& w, const BurnParams&) {
  held[w.at] = s.z;
  return turn(s, w);
}
bool zone_attempt(const TurnNet&, Zone& s, TurnWS& w, const BurnParams&) { return turn(s, w); }
void zone_finish(const TurnNet&, const Zone& s, const TurnWS&, const BurnParams&) { ++ended[s.z]; }
void zone_timeout_unstarted(const TurnNet&, long long, const BurnParams&) { error |= 8; }

}  // namespace nb

namespace {

nb::BurnParams params;

void entry() {
  const nb::TurnNet t;
  nb::TurnWS w{(long long)(threadIdx.x >> 5) * t.lane_doubles * nb::WS_LANES + (threadIdx.x & 31)};
  nb::burn_claim_loop(t, w, params);
  fib[cur].done = true;
  swapcontext(&fib[cur].ctx, &sched);
}

}  // namespace

// 0: every zone ran its turns.  Bits: 1 threads at different barriers, 2 no
// thread can run, 4 another zone's arrays, 8 a zone's turns are wrong, 16 too
// long.  warp_order: the warp that goes on first, ..., last.
extern "C" int run_block(int threads, long long zones, const int* zone_turns,
                         const int* warp_order) {
  unsigned long long queue = 0;
  std::memset(&params, 0, sizeof params);
  params.Z = zones;
  params.queue = &queue;
  nb::turns = zone_turns;
  nb::error = 0;
  nb::ran.assign(zones, 0);
  nb::ended.assign(zones, 0);
  nb::held.assign((size_t)(threads / 32) * nb::TurnNet::lane_doubles * nb::WS_LANES, -1);
  blockDim.x = threads;
  for (int i = 0; i < threads; ++i) {
    Fibre& f = fib[i];
    f.site = 0;
    f.done = false;
    f.stack.resize(STACK);
    getcontext(&f.ctx);
    f.ctx.uc_stack.ss_sp = f.stack.data();
    f.ctx.uc_stack.ss_size = STACK;
    f.ctx.uc_link = nullptr;
    makecontext(&f.ctx, entry, 0);
  }
  const int nw = threads / 32;
  for (long long step = 0; step < 50000000; ++step) {
    // the first warp that can go on: a runnable thread, or a ballot that all
    // its threads have reached
    int pick = -1;
    bool all_done = true;
    for (int o = 0; o < nw && pick < 0; ++o) {
      const int v = warp_order[o];
      bool full = true;
      unsigned bits = 0;
      for (int l = 0; l < 32 && pick < 0; ++l) {
        const Fibre& f = fib[v * 32 + l];
        if (!f.done && f.site == 0) pick = v * 32 + l;
        full = full && !f.done && f.site == -1;
        if (f.pred) bits |= 1u << l;
      }
      if (pick < 0 && full) {
        warp_bits[v] = bits;
        for (int l = 0; l < 32; ++l) fib[v * 32 + l].site = 0;
        pick = v * 32;
      }
    }
    if (pick >= 0) {
      cur = pick;
      threadIdx.x = pick;
      swapcontext(&sched, &fib[pick].ctx);
      continue;
    }
    // nobody can: the block's barrier
    int site = 0;
    bool any = false, full = true;
    for (int i = 0; i < threads; ++i) {
      if (fib[i].done) continue;
      all_done = false;
      if (fib[i].site <= 0) { full = false; continue; }
      if (site && site != fib[i].site) return nb::error | 1;
      site = fib[i].site;
      any = any || fib[i].pred;
    }
    if (all_done) {
      for (long long z = 0; z < zones; ++z)
        if (nb::ran[z] != nb::turns[z] || nb::ended[z] != 1) nb::error |= 8;
      return nb::error;
    }
    if (!full) return nb::error | 2;
    for (int i = 0; i < threads; ++i)
      if (fib[i].done) return nb::error | 1;   // a thread left before this barrier
    block_or = any;
    for (int i = 0; i < threads; ++i) fib[i].site = 0;
  }
  return nb::error | 16;
}
