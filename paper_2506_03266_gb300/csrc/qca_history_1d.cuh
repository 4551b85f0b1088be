// The ring automaton (repetition code) decoded from its syndrome history, device
// side.  As on the torus (qca_history.cuh), a field is the distance to the
// nearest anyon of the past light cone:
//   m^{s}_r = min { d <= m_max : sigma_{t - floor((d - 1) / v)} has an anyon at r - s d },
// and an anyon moves toward the nearer of its two sides (not at all when both are
// equally far).  A thread owns 32 sites as one word, so one distance is two
// shifted reads of an old syndrome for all of them; the state of a ring is its
// history in shared memory and a few registers.  Once a warp has few undecided
// anyons left they are searched one by one, a lane per slice.
//
// Bound by instruction issue: about thirty instructions per slice and warp, and
// as many per random draw.  L = 1024, p = 0.3, 10 % random moves, 20 000 rings:
// 590 us, against 3450 us for the sweep that keeps the two fields as bytes.
#pragma once

#include "qca_history.cuh"

namespace qca {

struct Args1D {
  const uint8_t* in;
  int L;
  int64_t shots;
  int max_steps;
  int v;
  int m_max;
  uint64_t move_thr;
  uint64_t move_key;
  int64_t shot_offset;
  uint8_t* out_C;
  int32_t* out_steps;
  uint8_t* out_flag;
  uint8_t* out_maj;
};

namespace hist {

constexpr int kRingFew = 6;  // undecided anyons of a warp searched one by one

template <int NT>
struct RingDecoder {
  const Args1D& a;
  int W;            // words per ring
  int depth;        // syndromes kept: (m_max - 1) / v + 2
  uint32_t* ring;   // [depth][W]
  uint32_t* xch;    // [2][W] words passed to neighbours
  int* misc;        // 0 weight of the noise
  int tid, lane;

  __device__ __forceinline__ bool sync_or(bool p) const {
    if (NT == 32) {
      const bool any = __any_sync(kFull, p);
      __syncwarp();
      return any;
    }
    return __syncthreads_or(p);
  }
  __device__ __forceinline__ void sync() const {
    if (NT == 32) {
      __syncwarp();
    } else {
      __syncthreads();
    }
  }
  // 32 sites from site c (mod L, 0 <= c < L); L >= 64
  __device__ __forceinline__ uint32_t window(const uint32_t* w, int c) const {
    const int i = c >> 5;
    uint32_t v = __funnelshift_r(w[i], i + 1 < W ? w[i + 1] : 0u, c & 31);
    if (c + 32 > a.L) v |= w[0] << (a.L - c);  // 1 .. 31
    return v;
  }
  __device__ __forceinline__ bool bit(const uint32_t* w, int c) const {
    return (w[c >> 5] >> (c & 31)) & 1u;
  }
  __device__ __forceinline__ int wrap(int c) const {  // |c| < L + 256, L >= 64
#pragma unroll 1
    while (c < 0) c += a.L;
#pragma unroll 1
    while (c >= a.L) c -= a.L;
    return c;
  }

  __device__ __forceinline__ void run(int64_t shot) {
    const int L = a.L, v = a.v, lastb = (L - 1) & 31;
    const int kmax = (a.m_max - 1) / v;
    const bool on = tid < W, last = tid == W - 1;
    const uint32_t valid = !on ? 0u : (last ? kFull >> (31 - lastb) : kFull);
    const uint8_t* N = a.in + shot * L;
    // ---- sigma_0 and the weight of the noise
    if (on) xch[tid] = 0;
    if (tid == 0) misc[0] = 0;
    sync();
    load_flat(N, 1, L, 9, xch, false, tid, NT);
    sync();
    uint32_t s = 0;
    uint32_t first = 0;  // N[0]
    {
      const uint32_t b = on ? xch[tid] : 0u;
      const uint32_t before = on ? (tid ? xch[tid - 1] >> 31 : (xch[W - 1] >> lastb) & 1u) : 0u;
      s = (b ^ ((b << 1) | before)) & valid;
      first = xch[0] & 1u;
      const int n = __reduce_add_sync(kFull, __popc(b));
      if (lane == 0 && n) atomicAdd(&misc[0], n);
    }
    uint32_t C = 0;
    int t = 0, flag = 0, cur = 0, still = 0;
    if (on) ring[tid] = s;
    bool any = sync_or(s != 0);
    const uint64_t k1 = a.move_thr ? splitmix64(a.move_key ^ (uint64_t)(a.shot_offset + shot)) : 0;
    const int c0 = tid << 5;
#pragma unroll 1
    while (any) {
      if (t >= a.max_steps || still > kmax) {
        flag = 2;
        t = a.max_steps;
        break;
      }
      uint32_t left = 0, right = 0, u = s;
      if (a.move_thr) {
        const uint64_t key = splitmix64(k1 ^ (uint64_t)(uint32_t)t);
#pragma unroll 1
        for (uint32_t b = s; b; b &= b - 1) {
          const int q = __ffs(b) - 1;
          const uint64_t r = splitmix64(key ^ (uint64_t)(c0 + q));
          if (r < a.move_thr) {
            u &= ~(1u << q);
            if (splitmix64(r) >> 63) left |= 1u << q;
            else right |= 1u << q;
          }
        }
      }
      // ---- nearest anyon of the past on either side
      const int lastk = min(t, kmax);
      int slot = cur;
#pragma unroll 1
      for (int k = 0; k <= lastk; ++k) {
        const uint32_t* w = ring + slot * W;
        slot = slot == 0 ? depth - 1 : slot - 1;
        if (u) {
          const int end = min(v * (k + 1), a.m_max);
#pragma unroll 1
          for (int d = v * k + 1; d <= end; ++d) {
            const uint32_t p = window(w, wrap(c0 - d)) & u;  // from the left: m^+
            const uint32_t m = window(w, wrap(c0 + d)) & u;
            left |= p & ~m;
            right |= m & ~p;
            u &= ~(p | m);
          }
        }
        const uint32_t open = __ballot_sync(kFull, u != 0);
        if (!open) break;
        if (k >= 2 && k < lastk && __popc(open) <= kRingFew) {
          if (__reduce_add_sync(kFull, __popc(u)) <= kRingFew) {
            one_by_one(u, left, right, k + 1, lastk, cur);
            break;
          }
        }
      }
      // ---- feedback: link <r, r + 1> flips iff r moves right or r + 1 moves left
      uint32_t F, Fb;
      if (NT == 32) {
        const uint32_t nb = __shfl_sync(kFull, left, last ? 0 : lane + 1) & 1u;
        F = (right | (left >> 1) | (nb << (last ? lastb : 31))) & valid;
        Fb = __shfl_sync(kFull, F, lane ? lane - 1 : W - 1);
        Fb = lane ? Fb >> 31 : (Fb >> lastb) & 1u;
      } else {
        if (on) xch[tid] = left;
        sync();
        const uint32_t nb = on ? xch[last ? 0 : tid + 1] & 1u : 0u;
        F = (right | (left >> 1) | (nb << (last ? lastb : 31))) & valid;
        if (on) xch[W + tid] = F;
        sync();
        Fb = on ? (tid ? xch[W + tid - 1] >> 31 : (xch[W + W - 1] >> lastb) & 1u) : 0u;
      }
      C ^= F;
      s = (s ^ F ^ ((F << 1) | Fb)) & valid;
      cur = cur + 1 == depth ? 0 : cur + 1;
      if (on) ring[cur * W + tid] = s;
      // without random moves a ring that has not moved for kmax + 1 steps never
      // moves again
      if (!a.move_thr) still = sync_or(F != 0) ? 0 : still + 1;
      any = sync_or(s != 0);
      ++t;
    }
    // ---- outputs
    if (on) xch[tid] = C;
    sync();
    int lw = 0;
    while ((1 << lw) < W) ++lw;
    store_flat(a.out_C + shot * L, 1, L, lw, xch, tid, NT);
    if (tid == 0) {
      const int value = (int)((first ^ C) & 1u);
      const int majority = 2 * misc[0] > L ? 1 : 0;
      a.out_steps[shot] = t;
      a.out_flag[shot] = (uint8_t)(flag == 2 ? 2 : value);
      if (a.out_maj) a.out_maj[shot] = (uint8_t)(flag == 2 ? 2 : (value != majority));
    }
  }

  // The warp's undecided anyons one after the other, slices k0 .. lastk, a lane
  // per slice.
  __device__ __forceinline__ void one_by_one(uint32_t& u, uint32_t& left, uint32_t& right, int k0,
                                             int lastk, int cur) const {
    uint32_t open = __ballot_sync(kFull, u != 0);
#pragma unroll 1
    while (open) {
      const int src = __ffs(open) - 1;
      const uint32_t us = __shfl_sync(kFull, u, src);
      const int q = __ffs(us) - 1;
      const int r = ((tid - lane + src) << 5) + q;
      int side = 0;
#pragma unroll 1
      for (int kb = k0; kb <= lastk; kb += 32) {
        const int k = kb + lane;
        int got = 0;
        if (k <= lastk) {
          int slot = cur - k;
          if (slot < 0) slot += depth;
          const uint32_t* w = ring + slot * W;
          const int end = min(a.v * (k + 1), a.m_max);
#pragma unroll 1
          for (int d = a.v * k + 1; d <= end && !got; ++d)
            got = (bit(w, wrap(r - d)) ? 1 : 0) | (bit(w, wrap(r + d)) ? 2 : 0);
        }
        const uint32_t hit = __ballot_sync(kFull, got != 0);
        if (hit) {
          side = __shfl_sync(kFull, got, __ffs(hit) - 1);
          break;
        }
      }
      if (lane == src) {
        if (side == 1) left |= 1u << q;
        if (side == 2) right |= 1u << q;
        u &= u - 1;
      }
      open = __ballot_sync(kFull, u != 0);
    }
  }
};

}  // namespace hist
}  // namespace qca
