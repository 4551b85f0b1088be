// Host side and kernels of the history sweep (qca_history.cuh).
//
// Up to L = 256 everything a shot needs is in one CTA's shared memory: the last
// 4 to 8 syndrome bitmaps, the correction, the flipped-link maps and the anyon
// list; older syndromes go to the shot's own correction block, which is not
// written before the shot ends (16 bitmaps of L^2 / 8 bytes fit its 2 L^2).  A
// shot that needs a still older one (all anyons of a region far apart while
// others elsewhere linger) is
// left pending, and the sweep with message planes decodes it in a second
// launch, which otherwise only looks for pending shots.  Above L = 256 the
// bitmaps live in a slot of a cached workspace that holds all 85 syndromes a
// message can come from.
#include <algorithm>
#include <atomic>
#include <mutex>

#include "qca_history.cuh"

namespace qca {

namespace {

using namespace hist;

template <int NT, bool LARGE>
__global__ void __launch_bounds__(NT, NT == 32 ? 24 : (NT == 1024 ? 1 : 768 / NT))
    history_kernel(const __grid_constant__ DecodeArgs a, const __grid_constant__ Geom g,
                   uint32_t* ws, size_t slot_words) {
  extern __shared__ __align__(16) uint32_t sm[];
  uint32_t* base = LARGE ? ws + (size_t)blockIdx.x * slot_words : sm;
  for (int64_t k = blockIdx.x; k < a.shots; k += gridDim.x) {
    Decoder<NT, LARGE> d{a, g};
    d.ring = base;
    d.C = base + g.o_C;
    d.F = base + g.o_F;
    d.list = sm + g.o_list;
    d.few = reinterpret_cast<typename Decoder<NT, LARGE>::Ent*>(sm + g.o_few);
    d.misc = reinterpret_cast<int*>(sm + g.o_misc);
    d.shot = a.shot_list ? (int64_t)a.shot_list[k] : k;
    d.tid = threadIdx.x;
    d.lane = threadIdx.x & 31;
    d.warp = threadIdx.x >> 5;
    d.run();
    d.sync();  // the next shot reuses the state
  }
}

// Threads per shot: a warp up to L = 64 (no block barriers), then about eight
// bitmap words per thread.
int threads_for(int L) { return L <= 64 ? 32 : (L <= 128 ? 128 : (L <= 256 ? 256 : 1024)); }

bool make_hist_geom(int L, int m_max, Geom& g, int& threads, size_t& smem, size_t& slot_words) {
  if (L < 8 || L > QCA_MAX_L) return false;
  const bool large = L > 256;
  threads = threads_for(L);
  g.L = L;
  const int wpr = (L + 31) / 32;
  g.lws = 0;
  while ((1 << g.lws) < wpr) ++g.lws;
  g.nws = L << g.lws;
  g.kmax = (m_max - 1) / 3;
  const int K = L <= 128 ? 8 : 4;
  g.kmask = K - 1;
  g.spill = g.kmax > K - 2 ? 16 : 0;
  // the dense pass costs about as much as searching half an anyon per word
  g.sparse_max = std::max(kFew, std::min(4 * threads, g.nws / 2));
  g.list_cap = std::max(g.nws / 2, g.sparse_max) + 64;
  if (large) g.list_cap = std::min(g.list_cap, 8192);
  const int few = large ? kFewWords<true> : kFewWords<false>;
  if (large) {
    g.o_C = kLargeRing * g.nws;
    g.o_F = g.o_C + 2 * g.nws;
    slot_words = (size_t)g.o_F + 2 * g.nws;
    g.o_few = 0;
    g.o_list = few;
    g.o_misc = g.o_list + g.list_cap;
  } else {
    // the few-anyon mode's sets take the link maps' place
    g.o_C = K * g.nws;
    g.o_F = (g.o_C + 2 * g.nws + 3) & ~3;
    g.o_few = g.o_F;
    g.o_list = g.o_F + std::max(2 * g.nws, few);
    g.o_misc = g.o_list + g.list_cap;
    slot_words = 0;
  }
  smem = (size_t)(g.o_misc + 8) * 4;
  return true;
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
  cudaEvent_t done = nullptr;
};
std::mutex g_hws_mu;
HistWorkspace g_hws[64];

template <int NT>
int launch_small(const DecodeArgs& a, const Geom& g, size_t smem, int dev, cudaStream_t stream) {
  static std::atomic<int> have[64];
  auto kern = history_kernel<NT, false>;
  if (int rc = allow_smem(kern, smem, have, dev)) return rc;
  // a CTA per shot: the hardware hands out shots as CTAs retire
  const int64_t grid = std::min<int64_t>(a.shots, 1 << 30);
  kern<<<(unsigned)grid, NT, smem, stream>>>(a, g, nullptr, 0);
  return cuda_fail(cudaGetLastError(), "history sweep launch");
}

int launch_large(const DecodeArgs& a, const Geom& g, size_t smem, size_t slot_words, int dev,
                 cudaStream_t stream) {
  constexpr int NT = 1024;
  static std::atomic<int> have[64];
  auto kern = history_kernel<NT, true>;
  if (int rc = allow_smem(kern, smem, have, dev)) return rc;
  int sms = 0, per_sm = 0;
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, NT, smem);
  if (e != cudaSuccess) return cuda_fail(e, "history sweep occupancy");
  // slots for the resident CTAs, at most 2 GiB
  int64_t slots = std::min<int64_t>((int64_t)std::max(per_sm, 1) * sms,
                                    (int64_t)((size_t(2) << 30) / (4 * slot_words)));
  slots = std::max<int64_t>(1, std::min<int64_t>(slots, a.shots));
  const size_t need = 4 * slot_words * (size_t)slots;
  std::lock_guard<std::mutex> lk(g_hws_mu);
  HistWorkspace& w = g_hws[dev];
  if (w.bytes < need) {
    if (w.ptr) {
      // the previous workspace may still be in use by queued work on any stream
      e = cudaDeviceSynchronize();
      if (e != cudaSuccess) return cuda_fail(e, "synchronise before workspace growth");
      cudaFree(w.ptr);
      w.ptr = nullptr;
      w.bytes = 0;
    }
    e = cudaMalloc(&w.ptr, need);
    if (e != cudaSuccess) return cuda_fail(e, "history workspace allocation");
    w.bytes = need;
  }
  if (!w.done) {
    e = cudaEventCreateWithFlags(&w.done, cudaEventDisableTiming);
    if (e != cudaSuccess) return cuda_fail(e, "event creation");
  }
  // launches on different streams share the workspace: order them
  e = cudaStreamWaitEvent(stream, w.done, 0);
  if (e != cudaSuccess) return cuda_fail(e, "stream wait");
  kern<<<(unsigned)slots, NT, smem, stream>>>(a, g, w.ptr, slot_words);
  e = cudaGetLastError();
  if (e != cudaSuccess) return cuda_fail(e, "history sweep launch");
  return cuda_fail(cudaEventRecord(w.done, stream), "event record");
}

}  // namespace

bool history_takes(int L, int v) { return v == 3 && L >= 8 && L <= QCA_MAX_L; }

bool history_may_leave_pending(int L) { return L <= 256; }

int launch_history(const DecodeArgs& a, cudaStream_t stream) {
  Geom g;
  int threads;
  size_t smem, slot_words;
  if (a.v != 3 || !make_hist_geom(a.L, a.m_max, g, threads, smem, slot_words)) {
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
  switch (threads) {
    case 32: return launch_small<32>(a, g, smem, dev, stream);
    case 128: return launch_small<128>(a, g, smem, dev, stream);
    case 256: return launch_small<256>(a, g, smem, dev, stream);
    default: return launch_large(a, g, smem, slot_words, dev, stream);
  }
}

int history_workspace_release() {
  std::lock_guard<std::mutex> lk(g_hws_mu);
  int dev = 0;
  cudaGetDevice(&dev);
  if (dev < 0 || dev >= 64 || !g_hws[dev].ptr) return QCA_OK;
  cudaError_t e = cudaFree(g_hws[dev].ptr);
  g_hws[dev].ptr = nullptr;
  g_hws[dev].bytes = 0;
  return cuda_fail(e, "history workspace free");
}

}  // namespace qca
