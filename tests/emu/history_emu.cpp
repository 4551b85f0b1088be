// Host emulation of the history decoder's device code (test infrastructure).
//
// Every lane of a CTA is a fiber; it runs until it reaches a warp collective or a
// block barrier and goes on when all lanes of its warp or block have arrived.  The
// next lane to run is drawn from a seed, so a program that depends on the order of
// lanes between two synchronisations gives different outcomes for different
// seeds, and a collective that some lanes of the warp never reach is reported
// instead of hanging.
#include <cuda_runtime.h>
#include <stdint.h>
#include <stdlib.h>
#include <string.h>
#include <ucontext.h>

#include <algorithm>
#include <memory>
#include <vector>

using std::max;
using std::min;

namespace emu {

enum Op { kNone, kExchange, kOr, kAnd, kAdd, kXor, kBallot, kWarp, kBlock };

struct Lane {
  ucontext_t ctx;
  std::unique_ptr<uint8_t[]> stack;
  int op = kNone;      // collective it waits at
  uint64_t in = 0;     // its value
  uint64_t out = 0;    // the result for it
  int src = 0;         // kExchange: lane it reads
  bool done = false;
};

constexpr size_t kStack = 128 * 1024;
std::vector<Lane> lanes;
ucontext_t scheduler;
int current;

uint64_t wait(int op, uint64_t in, int src = 0) {
  Lane& l = lanes[current];
  l.op = op;
  l.in = in;
  l.src = src;
  swapcontext(&l.ctx, &scheduler);
  return lanes[current].out;
}

// Completes a collective of lanes lo .. hi - 1 if all of them are at it; false if
// they can never be (different collectives, or some have left).
bool complete(int lo, int hi, bool block, std::vector<int>& ready) {
  bool any = false, all = true;
  int op = kNone;
  for (int i = lo; i < hi; ++i) {
    const Lane& l = lanes[i];
    const bool here = !l.done && l.op != kNone && (l.op == kBlock) == block;
    any |= here;
    all &= here;
    if (here) op = l.op;
  }
  if (!any) return true;
  if (!all) {
    for (int i = lo; i < hi; ++i)
      if (lanes[i].done) return false;
    return true;  // the others may still come
  }
  for (int i = lo; i < hi; ++i)
    if (lanes[i].op != op) return false;
  uint64_t r = op == kAnd ? ~0ull : 0;
  for (int i = lo; i < hi; ++i) {
    const uint64_t v = lanes[i].in;
    if (op == kOr || op == kBlock) r |= v;
    if (op == kAnd) r &= v;
    if (op == kAdd) r += v;
    if (op == kXor) r ^= v;
    if (op == kBallot && v) r |= 1ull << (i - lo);
  }
  for (int i = lo; i < hi; ++i) {
    Lane& l = lanes[i];
    l.out = op == kExchange ? lanes[lo + (l.src & 31)].in : r;
    ready.push_back(i);
  }
  for (int i = lo; i < hi; ++i) lanes[i].op = kNone;
  return true;
}

void (*entry)(int);
void trampoline() {
  entry(current);
  lanes[current].done = true;
  swapcontext(&lanes[current].ctx, &scheduler);
}

// Runs body(tid) on n lanes; false if lanes of a warp or block went apart.
bool run(int n, uint64_t seed, void (*body)(int)) {
  entry = body;
  if ((int)lanes.size() < n) lanes.resize(n);
  std::vector<int> ready(n);
  for (int i = 0; i < n; ++i) {
    Lane& l = lanes[i];
    if (!l.stack) l.stack.reset(new uint8_t[kStack]);
    getcontext(&l.ctx);
    l.ctx.uc_stack.ss_sp = l.stack.get();
    l.ctx.uc_stack.ss_size = kStack;
    l.ctx.uc_link = nullptr;
    l.op = kNone;
    l.done = false;
    makecontext(&l.ctx, trampoline, 0);
    ready[i] = i;
  }
  uint64_t rng = seed * 2 + 1;
  for (;;) {
    if (ready.empty()) {
      bool all = true;
      for (int i = 0; i < n; ++i) all &= lanes[i].done;
      return all;
    }
    rng = rng * 6364136223846793005ull + 1442695040888963407ull;
    const size_t q = (size_t)((rng >> 33) % ready.size());
    current = ready[q];
    ready[q] = ready.back();
    ready.pop_back();
    swapcontext(&scheduler, &lanes[current].ctx);
    const int w = current & ~31;
    const bool block = lanes[current].op == kBlock || lanes[current].done;
    if (!complete(w, min(w + 32, n), false, ready)) return false;
    if (block && !complete(0, n, true, ready)) return false;
  }
}

}  // namespace emu

// ------------------------------------------------------ the device's builtins
static inline void __syncwarp(unsigned = 0xffffffffu) { emu::wait(emu::kWarp, 0); }
static inline void __syncthreads() { emu::wait(emu::kBlock, 0); }
static inline int __syncthreads_or(int p) { return emu::wait(emu::kBlock, p != 0) != 0; }
template <class T>
static inline T exchange(T v, int src) {
  uint64_t b = 0;
  memcpy(&b, &v, sizeof v);
  b = emu::wait(emu::kExchange, b, src);
  memcpy(&v, &b, sizeof v);
  return v;
}
template <class T>
static inline T __shfl_sync(unsigned, T v, int src) { return exchange(v, src); }
template <class T>
static inline T __shfl_up_sync(unsigned, T v, int o) {
  const int lane = emu::current & 31;
  return exchange(v, lane >= o ? lane - o : lane);
}
static inline unsigned __reduce_or_sync(unsigned, unsigned v) { return emu::wait(emu::kOr, v); }
static inline int __reduce_add_sync(unsigned, int v) { return (int)emu::wait(emu::kAdd, (unsigned)v); }
static inline unsigned __reduce_xor_sync(unsigned, unsigned v) { return emu::wait(emu::kXor, v); }
static inline unsigned __ballot_sync(unsigned, int p) { return emu::wait(emu::kBallot, p != 0); }
static inline int __all_sync(unsigned, int p) { return emu::wait(emu::kAnd, p != 0) != 0; }
static inline int __any_sync(unsigned, int p) { return emu::wait(emu::kOr, p != 0) != 0; }
template <class T>
static inline T atomicAdd(T* p, T v) { T o = *p; *p = o + v; return o; }
template <class T>
static inline T atomicOr(T* p, T v) { T o = *p; *p = o | v; return o; }
template <class T>
static inline T atomicXor(T* p, T v) { T o = *p; *p = o ^ v; return o; }
template <class T>
static inline T atomicCAS(T* p, T c, T v) { T o = *p; if (o == c) *p = v; return o; }
template <class T>
static inline T __ldcg(const T* p) { return *p; }
template <class T>
static inline T __ldcs(const T* p) { return *p; }
template <class T>
static inline void __stcs(T* p, T v) { *p = v; }
static inline int __popc(unsigned v) { return __builtin_popcount(v); }
static inline int __ffs(int v) { return __builtin_ffs(v); }
static inline unsigned __funnelshift_r(unsigned lo, unsigned hi, unsigned s) {
  s &= 31;
  return s ? (lo >> s) | (hi << (32 - s)) : lo;
}
static inline unsigned __funnelshift_lc(unsigned lo, unsigned hi, unsigned s) {
  if (s >= 32) return lo;
  return s ? (hi << s) | (lo >> (32 - s)) : hi;
}
#undef __noinline__
#define __noinline__
#undef __forceinline__
#define __forceinline__ inline

#include "qca_history.cuh"

using namespace qca;
using namespace qca::hist;

namespace {

DecodeArgs g_args;
Geom g_geom;
uint32_t* g_sm;
int g_threads;

template <int NT, bool PLAIN, bool OPEN>
void lane_body(int tid) {
  Decoder<NT, false, PLAIN, OPEN> d{g_args, g_geom};
  d.ring = g_sm;
  d.C = g_sm + g_geom.o_C;
  d.F = g_sm + g_geom.o_F;
  d.list = g_sm + g_geom.o_list;
  d.table = g_sm + g_geom.o_table;
  d.snap = g_sm + g_geom.o_snap;
  d.few = reinterpret_cast<uint16_t*>(g_sm + g_geom.o_few);
  d.misc = reinterpret_cast<int*>(g_sm + g_geom.o_misc);
  d.nset = reinterpret_cast<uint16_t*>(g_sm + g_geom.o_misc + 8);
  d.place = d.nset + kSteps;
  d.shot = 0;
  d.tid = tid;
  d.lane = tid & 31;
  d.warp = tid >> 5;
  d.run();
  d.sync();
}

}  // namespace

// Decodes `shots` shots (noise, or anyon indicators) of size L <= 256 one after
// the other.  `fill`: byte that the correction and the shared memory hold before;
// `skew`: bytes by which the arrays start off a 16-byte boundary; `order`: seed of
// the lanes' order; `threads`: per shot, 0 for those of a large batch.  A shot left
// pending has steps -1.  Returns 0, -1 (no geometry), -2 (lanes went apart) or -3 (a
// write next to an array).
extern "C" int emu_history(const uint8_t* in, int L, int shots, int max_steps, int m_max,
                           uint64_t move_thr, uint64_t seed, int tie, int bal, int from_sigma,
                           int open, int all, int fill, int skew, uint64_t order, int threads,
                           uint8_t* out_C, int32_t* out_steps, uint8_t* out_flag) {
  size_t smem, slot_words;
  if (L > 256 || !make_hist_geom(L, m_max, g_geom, g_threads, smem, slot_words, all != 0)) return -1;
  if (threads) g_threads = threads;
  DecodeArgs& a = g_args;
  memset(&a, 0, sizeof(a));
  a.L = L;
  a.shots = 1;
  a.max_steps = max_steps;
  a.v = 3;
  a.m_max = m_max;
  a.move_thr = move_thr;
  a.move_key = splitmix64(seed ^ kTagMove);
  a.balance_key = splitmix64(seed ^ kTagBalance);
  a.tie_order = tie;
  a.balance_rule = bal;
  a.from_sigma = from_sigma;
  const size_t ib = (size_t)(from_sigma ? 1 : 2) * L * L, ob = 2 * (size_t)L * L;
  constexpr size_t kGuard = 256;
  std::vector<uint8_t> ibuf(ib + kGuard + 16), obuf(ob + 2 * kGuard + 16);
  std::vector<uint8_t> sbuf(smem + 2 * kGuard + 16);
  auto align16 = [](uint8_t* p) { return p + ((16 - ((uintptr_t)p & 15)) & 15); };
  uint8_t* ip = align16(ibuf.data()) + skew;
  uint8_t* op = align16(obuf.data() + kGuard) + skew;
  uint8_t* sp = align16(sbuf.data() + kGuard);
  const bool plain = !move_thr && !tie && !bal;
  if (open && !plain) return -1;
  void (*body)(int) = nullptr;
  if (g_threads == 32)
    body = open ? lane_body<32, true, true> : (plain ? lane_body<32, true, false> : lane_body<32, false, false>);
  else if (open ? g_threads > 128 : g_threads == 256 || g_threads == 512)
    body = open ? nullptr
                : (g_threads == 256 ? (plain ? lane_body<256, true, false> : lane_body<256, false, false>)
                                    : (plain ? lane_body<512, true, false> : lane_body<512, false, false>));
  else
    body = open ? lane_body<128, true, true> : (plain ? lane_body<128, true, false> : lane_body<128, false, false>);
  if (!body) return -1;
  for (int s = 0; s < shots; ++s) {
    std::fill(obuf.begin(), obuf.end(), (uint8_t)fill);
    std::fill(sbuf.begin(), sbuf.end(), (uint8_t)fill);
    memcpy(ip, in + (size_t)s * ib, ib);
    int32_t steps = -7;
    uint8_t flag = 9, cut[2] = {9, 9}, exhausted = 9;
    a.in = ip;
    a.out_C = op;
    a.out_steps = &steps;
    a.out_flag = &flag;
    a.out_cut = cut;
    a.out_exhausted = &exhausted;
    a.shot_offset = s;
    g_sm = reinterpret_cast<uint32_t*>(sp);
    if (!emu::run(g_threads, order + s, body)) return -2;
    for (uint8_t* q = obuf.data(); q < op; ++q)
      if (*q != (uint8_t)fill) return -3;
    for (uint8_t* q = op + ob; q < obuf.data() + obuf.size(); ++q)
      if (*q != (uint8_t)fill) return -3;
    for (uint8_t* q = sbuf.data(); q < sp; ++q)
      if (*q != (uint8_t)fill) return -3;
    for (uint8_t* q = sp + smem; q < sbuf.data() + sbuf.size(); ++q)
      if (*q != (uint8_t)fill) return -3;
    memcpy(out_C + (size_t)s * ob, op, ob);
    out_steps[s] = steps;
    out_flag[s] = from_sigma ? exhausted : flag;
  }
  return 0;
}
