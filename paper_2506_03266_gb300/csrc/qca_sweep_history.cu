// Host side and kernels of the history sweep (qca_history.cuh).
//
// Up to L = 256 the last 4 to 8 syndrome bitmaps and the anyon list are in the
// shared memory of the shot's CTA; older syndromes go to the shot's own
// correction block, which is not written before the shot ends, as bitmaps while
// the anyons are many and as lists of sites afterwards, so that shots of random
// noise keep all 85 syndromes a message can come from (none was left up to p = 0.2
// with 8 shots per size and rate, L = 20 to 256).  A shot that has
// too many large old ones (a syndrome with a part that stays dense for dozens of
// steps and a part that is sparse) is left pending, and the sweep with message
// planes decodes it in a second launch, which otherwise only looks for pending
// shots.  Above L = 256 the bitmaps live in a slot of a cached workspace that
// holds all 85.
//
// What bounds it: latency at 19 to 24 warps per SM (L = 256: 172 thousand warp
// instructions per shot, issued in 48 % of the schedulers' cycles; warps wait for their
// own last instruction, for link maps and correction in L2 and at barriers about
// equally); instruction fetch for the small sizes, whose warps are all at different
// places of the code.  L = 256, p = 0.05, 20 000 shots: 4.85 ms, against 55 ms for the
// sweep over message planes; floor by bytes 0.77 ms.
#include <stdint.h>
#include <string.h>

#include <algorithm>
#include <atomic>
#include <mutex>

#include "qca_history.cuh"

namespace qca {

namespace {

using namespace hist;

template <int NT, bool LARGE, bool PLAIN, bool OPEN>
__global__ void __launch_bounds__(NT, NT == 32 ? 24 : (LARGE ? 1024 / NT : 768 / NT))
    history_kernel(const __grid_constant__ DecodeArgs a, const __grid_constant__ Geom g,
                   uint32_t* ws, size_t slot_words, int64_t first) {
  extern __shared__ __align__(16) uint32_t sm[];
  uint32_t* base = LARGE ? ws + (size_t)blockIdx.x * slot_words : sm;
  auto decode = [&](int64_t k) {
    Decoder<NT, LARGE, PLAIN, OPEN> d{a, g};
    d.ring = base;
    d.C = base + g.o_C;
    d.F = base + g.o_F;
    d.list = sm + g.o_list;
    d.table = sm + g.o_table;
    d.snap = sm + g.o_snap;
    d.few = reinterpret_cast<typename Decoder<NT, LARGE, PLAIN, OPEN>::Ent*>(sm + g.o_few);
    d.misc = reinterpret_cast<int*>(sm + g.o_misc);
    d.nset = reinterpret_cast<uint16_t*>(sm + g.o_misc + 8);
    d.place = d.nset + kSteps;
    d.shot = a.shot_list ? (int64_t)a.shot_list[k] : k;
    d.tid = threadIdx.x;
    d.lane = threadIdx.x & 31;
    d.warp = threadIdx.x >> 5;
    d.run();
    if (NT > 32) d.sync();  // the next shot reuses the state
  };
  if (NT > 32) {
    for (int64_t k = blockIdx.x; k < a.shots; k += gridDim.x) decode(k);
  } else {
    // one shot per CTA: a loop over shots costs the one-warp form 150 bytes of spills
    // (20 000 shots, p = 0.05, with it / without: L = 24 467 / 456 us, L = 48 641 / 622);
    // the forms of several warps spill without it
    decode(first + blockIdx.x);
  }
}

// Shots of several sizes: CTA b takes the b-th shot from the end of the list,
// which is grouped by increasing size, so that the large shots start first.
struct MixArgs {
  DecodeArgs a;
  int nsizes;
  int64_t first[kHistoryMixSizes];  // list index of each size's first shot
  int64_t end;
  Geom geom[kHistoryMixSizes];
};

template <int NT, bool PLAIN>
__global__ void __launch_bounds__(NT, NT == 32 ? 24 : 768 / NT)
    history_mixed_kernel(const __grid_constant__ MixArgs m) {
  extern __shared__ __align__(16) uint32_t sm[];
  const int64_t k = m.end - 1 - blockIdx.x;
  int c = 0;
  while (c + 1 < m.nsizes && k >= m.first[c + 1]) ++c;
  const Geom& g = m.geom[c];
  Decoder<NT, false, PLAIN> d{m.a, g};
  d.ring = sm;
  d.C = sm + g.o_C;
  d.F = nullptr;
  d.list = sm + g.o_list;
  d.table = sm + g.o_table;
  d.snap = sm + g.o_snap;
  d.few = reinterpret_cast<uint16_t*>(sm + g.o_few);
  d.misc = reinterpret_cast<int*>(sm + g.o_misc);
  d.nset = reinterpret_cast<uint16_t*>(sm + g.o_misc + 8);
  d.place = d.nset + kSteps;
  d.shot = m.a.shot_list[k];
  d.tid = threadIdx.x;
  d.lane = threadIdx.x & 31;
  d.warp = threadIdx.x >> 5;
  d.run();
}

// Shared-memory allowance of one kernel, raised once per device.
template <class K>
int allow_smem(K kern, size_t smem, std::atomic<int> (&have)[64], int dev) {
  if (smem <= 48 * 1024 || have[dev].load() >= (int)smem) return QCA_OK;
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       227 * 1024);
  if (e != cudaSuccess) return cuda_fail(e, "history sweep smem attribute");
  have[dev].store(227 * 1024);
  return QCA_OK;
}

struct HistWorkspace {
  uint32_t* ptr = nullptr;
  size_t bytes = 0;
  size_t refused = SIZE_MAX;  // smallest size that could not be allocated since the last release
  cudaEvent_t done = nullptr;
};
std::mutex g_hws_mu;
HistWorkspace g_hws[64];

// The default rules have a kernel of their own.
bool plain_rules(const DecodeArgs& a) {
  return a.move_thr == 0 && a.tie_order == QCA_TIE_LEX && a.balance_rule == QCA_BALANCE_STAY;
}

template <int NT, bool PLAIN, bool OPEN = false>
int launch_small(const DecodeArgs& a, const Geom& g, size_t smem, int dev, cudaStream_t stream) {
  static std::atomic<int> have[64];
  auto kern = history_kernel<NT, false, PLAIN, OPEN>;
  if (int rc = allow_smem(kern, smem, have, dev)) return rc;
  // a CTA per shot: the hardware hands out shots as CTAs retire
  int64_t first = 0;
  do {
    const int64_t grid = std::min<int64_t>(a.shots - first, 1 << 30);
    kern<<<(unsigned)grid, NT, smem, stream>>>(a, g, nullptr, 0, first);
    first += grid;
  } while (NT == 32 && first < a.shots);
  return cuda_fail(cudaGetLastError(), "history sweep launch");
}

template <int NT, bool PLAIN>
int launch_mix(const MixArgs& m, size_t smem, int64_t shots, int dev, cudaStream_t stream) {
  static std::atomic<int> have[64];
  auto kern = history_mixed_kernel<NT, PLAIN>;
  if (int rc = allow_smem(kern, smem, have, dev)) return rc;
  kern<<<(unsigned)shots, NT, smem, stream>>>(m);
  return cuda_fail(cudaGetLastError(), "history sweep launch (mixed sizes)");
}

template <int NT, bool PLAIN>
int launch_large(const DecodeArgs& a, const Geom& g, size_t smem, size_t slot_words, int dev,
                 cudaStream_t stream) {
  static std::atomic<int> have[64];
  auto kern = history_kernel<NT, true, PLAIN, false>;
  if (int rc = allow_smem(kern, smem, have, dev)) return rc;
  int sms = 0, per_sm = 0;
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, NT, smem);
  if (e != cudaSuccess) return cuda_fail(e, "history sweep occupancy");
  // slots for the resident CTAs, at most 2 GiB
  int64_t slots = std::min<int64_t>((int64_t)std::max(per_sm, 1) * sms,
                                    (int64_t)((size_t(2) << 30) / (4 * slot_words)));
  slots = std::max<int64_t>(1, std::min<int64_t>(slots, a.shots));
  const size_t slot = 4 * slot_words, need = slot * (size_t)slots;
  std::lock_guard<std::mutex> lk(g_hws_mu);
  HistWorkspace& w = g_hws[dev];
  if (w.bytes < need && (need < w.refused || w.bytes < slot)) {
    if (w.ptr) {
      // the previous workspace may still be in use by queued work on any stream
      e = cudaDeviceSynchronize();
      if (e != cudaSuccess) return cuda_fail(e, "synchronise before workspace growth");
      cudaFree(w.ptr);
      w.ptr = nullptr;
      w.bytes = 0;
    }
    // where memory is short, fewer shots at a time (L = 1024: 12 MB each)
    size_t n = (size_t)slots;
    while ((e = cudaMalloc(&w.ptr, slot * n)) == cudaErrorMemoryAllocation) {
      cudaGetLastError();
      w.ptr = nullptr;
      w.refused = std::min(w.refused, slot * n);
      if (n == 1) break;
      n = (n + 1) / 2;
    }
    if (e != cudaSuccess) return cuda_fail(e, "history workspace allocation");
    w.bytes = slot * n;
  }
  slots = std::min<int64_t>(slots, (int64_t)(w.bytes / slot));
  if (!w.done) {
    e = cudaEventCreateWithFlags(&w.done, cudaEventDisableTiming);
    if (e != cudaSuccess) return cuda_fail(e, "event creation");
  }
  // launches on different streams share the workspace: order them
  e = cudaStreamWaitEvent(stream, w.done, 0);
  if (e != cudaSuccess) return cuda_fail(e, "stream wait");
  kern<<<(unsigned)slots, NT, smem, stream>>>(a, g, w.ptr, slot_words, 0);
  e = cudaGetLastError();
  if (e != cudaSuccess) return cuda_fail(e, "history sweep launch");
  return cuda_fail(cudaEventRecord(w.done, stream), "event record");
}

}  // namespace

bool history_takes(int L, int v) { return v == 3 && L >= 8 && L <= QCA_MAX_L; }

bool history_may_leave_pending(int L, int64_t shots) { return L <= 256 && !all_slots(L, shots); }

int launch_history(const DecodeArgs& a, cudaStream_t stream) {
  Geom g;
  int threads;
  size_t smem, slot_words;
  if (a.v != 3 || !make_hist_geom(a.L, a.m_max, g, threads, smem, slot_words,
                                  all_slots(a.L, a.shots))) {
    set_error("no history sweep for L=%d v=%d", a.L, a.v);
    return QCA_ERR_UNSUPPORTED;
  }
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return cuda_fail(e, "cudaGetDevice");
  if (dev < 0 || dev >= 64) {
    set_error("device index %d out of range", dev);
    return QCA_ERR_UNSUPPORTED;
  }
  const bool plain = plain_rules(a);
  // Threads per shot where the batch is too small to fill the SMs with the fewest
  // (threads_for): a shot's steps then take as long as one warp or four need for
  // them.  us per call, 32 / 128 threads: L = 64, p = 0.05, 32 shots 87 / 76, 912
  // shots 122 / 116, 2000 shots 321 / 347.  128 / 256 / 512 threads: L = 256, p =
  // 0.05, 32 shots 224 / 178 / 159, 304 shots 260 / 215 / 307, 912 shots 356 / 406 /
  // 709; p = 0.3 (anyons stay dense), 32 shots 2343 / 1687 / 1197 (sweep over message
  // planes: 1173).  L = 128, p = 0.08, 304 shots 758 / 740 / 940, 912 shots 846 / 1139.
  int sms = 0;
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (threads == 32 && a.shots <= 6 * sms)
    threads = 128;
  else if (threads == 128 && a.L > 128 && a.shots <= sms)
    threads = 512;
  else if (threads == 128 && a.shots <= (a.L > 128 ? 3 : 2) * sms)
    threads = 256;
  switch (threads) {
    case 256:
      return plain ? launch_small<256, true>(a, g, smem, dev, stream)
                   : launch_small<256, false>(a, g, smem, dev, stream);
    case 512:
      return plain ? launch_small<512, true>(a, g, smem, dev, stream)
                   : launch_small<512, false>(a, g, smem, dev, stream);
    case 32:
      return plain ? launch_small<32, true>(a, g, smem, dev, stream)
                   : launch_small<32, false>(a, g, smem, dev, stream);
    case 128:
      return plain ? launch_small<128, true>(a, g, smem, dev, stream)
                   : launch_small<128, false>(a, g, smem, dev, stream);
    default: {
      // two CTAs of 512 threads per SM where there are shots for them and their
      // workspace stays small (1000 shots, p = 0.05: L = 384 1.51 -> 1.27 ms, L =
      // 512 2.14 -> 1.83 ms; at L = 1024 the same for 512 shots, and 1.23 -> 1.71 ms
      // for 100)
      if (a.L <= 512 && a.shots > sms)
        return plain ? launch_large<512, true>(a, g, smem, slot_words, dev, stream)
                     : launch_large<512, false>(a, g, smem, slot_words, dev, stream);
      return plain ? launch_large<1024, true>(a, g, smem, slot_words, dev, stream)
                   : launch_large<1024, false>(a, g, smem, slot_words, dev, stream);
    }
  }
}

int launch_history_open(const DecodeArgs& a, cudaStream_t stream) {
  Geom g;
  int threads;
  size_t smem, slot_words;
  if (a.v != 3 || a.L > 256 || !make_hist_geom(a.L, a.m_max, g, threads, smem, slot_words)) {
    set_error("no open-boundary history sweep for L=%d v=%d", a.L, a.v);
    return QCA_ERR_UNSUPPORTED;
  }
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return cuda_fail(e, "cudaGetDevice");
  if (dev < 0 || dev >= 64) {
    set_error("device index %d out of range", dev);
    return QCA_ERR_UNSUPPORTED;
  }
  return threads == 32 ? launch_small<32, true, true>(a, g, smem, dev, stream)
                       : launch_small<128, true, true>(a, g, smem, dev, stream);
}

int history_threads(int L) { return L >= 8 && L <= 256 ? threads_for(L) : 0; }

int launch_history_mixed(const DecodeArgs& a, const int* sizes, const int64_t* start, int nsizes,
                         cudaStream_t stream) {
  const int64_t shots = nsizes > 0 ? start[nsizes] - start[0] : 0;
  if (shots == 0) return QCA_OK;
  if (nsizes > kHistoryMixSizes || shots >= (int64_t)1 << 31) {
    set_error("history sweep: %d sizes, %lld shots in one launch", nsizes, (long long)shots);
    return QCA_ERR_UNSUPPORTED;
  }
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return cuda_fail(e, "cudaGetDevice");
  if (dev < 0 || dev >= 64) {
    set_error("device index %d out of range", dev);
    return QCA_ERR_UNSUPPORTED;
  }
  MixArgs m;
  memset(&m, 0, sizeof(m));
  m.a = a;
  m.nsizes = nsizes;
  m.end = start[nsizes];
  size_t smem = 0;
  int threads = 0;
  for (int c = 0; c < nsizes; ++c) {
    size_t s, slot;
    m.first[c] = start[c];
    if (!make_hist_geom(sizes[c], a.m_max, m.geom[c], threads, s, slot) ||
        threads != history_threads(sizes[0])) {
      set_error("no mixed history sweep for L=%d", sizes[c]);
      return QCA_ERR_UNSUPPORTED;
    }
    smem = std::max(smem, s);
  }
  const bool plain = plain_rules(a);
  if (threads == 32)
    return plain ? launch_mix<32, true>(m, smem, shots, dev, stream)
                 : launch_mix<32, false>(m, smem, shots, dev, stream);
  return plain ? launch_mix<128, true>(m, smem, shots, dev, stream)
               : launch_mix<128, false>(m, smem, shots, dev, stream);
}

int history_workspace_release() {
  std::lock_guard<std::mutex> lk(g_hws_mu);
  int dev = 0;
  cudaGetDevice(&dev);
  if (dev < 0 || dev >= 64) return QCA_OK;
  g_hws[dev].refused = SIZE_MAX;
  if (!g_hws[dev].ptr) return QCA_OK;
  cudaError_t e = cudaFree(g_hws[dev].ptr);
  g_hws[dev].ptr = nullptr;
  g_hws[dev].bytes = 0;
  return cuda_fail(e, "history workspace free");
}

}  // namespace qca
