// The ring automaton (repetition code) decoded from its syndrome history, device
// side.  As on the torus (qca_history.cuh), a field is the distance to the
// nearest anyon of the past light cone:
//   m^{s}_r = min { d <= m_max : sigma_{t - floor((d - 1) / v)} has an anyon at r - s d },
// and an anyon moves toward the nearer of its two sides (not at all when both are
// equally far).  A thread owns 32 sites as one word, so one distance is two
// shifted reads of an old syndrome for all of them; the state of a ring is its
// history in shared memory and a few registers.  Once a warp has few undecided
// anyons left they are searched one by one, a lane per slice (not with 8 or 16
// copies, which get through the distances faster than that).
//
// A ring of at most 512 sites needs at most half a warp's lanes for its words.  The
// warp then holds it 2 to 16 times over, and each copy looks at a distance of its
// own; the copies before it say which sites are decided already.  With one copy
// the lanes left over idle, and a step took as long as its distances are many, longer
// than with the two fields as bytes.  us, one copy / several / byte fields: 20 000
// rings with 10 % random moves, p = 0.3, L = 64 1604 / 501 / 713, L = 128 308 / 155 /
// 368, L = 512 413 / 325 / 1644; 2000 rings, p = 0.4, L = 128 1367 / 693 / 619.
//
// Bound by instruction issue: about thirty instructions per slice and warp, and
// as many per random draw.  L = 1024, p = 0.3, 10 % random moves, 20 000 rings:
// 570 us, against 3450 us for the sweep that keeps the two fields as bytes.
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
  int stride;       // lanes of a copy of the ring (NT == 32: a power of two >= W)
  int copies;       // 32 / stride; 1 for the larger forms
  int j, copy;      // word and copy of this thread
  // first distance of this copy, less one, over v and modulo v, the same of the step
  // from one distance to the next, and the first sites at it on either side
  int k0, r0, dk, dr, lo0, hi0;

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
  // OR of the copies' values for a word, to all copies.
  __device__ __forceinline__ uint32_t across(uint32_t v) const {
    if (NT == 32) {
#pragma unroll 1
      for (int o = stride; o < 32; o <<= 1) v |= __shfl_xor_sync(kFull, v, o);
    }
    return v;
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
    stride = 1;
    while (NT == 32 && stride < W) stride *= 2;
    copies = NT == 32 ? 32 / stride : 1;
    j = NT == 32 ? lane & (stride - 1) : tid;
    copy = NT == 32 ? lane / stride : 0;
    const bool on = j < W, last = j == W - 1, keeps = on && copy == 0;
    const uint32_t valid = !on ? 0u : (last ? kFull >> (31 - lastb) : kFull);
    const uint8_t* N = a.in + shot * L;
    // ---- sigma_0 and the weight of the noise
    if (keeps) xch[j] = 0;
    if (tid == 0) misc[0] = 0;
    sync();
    load_flat(N, 1, L, 9, xch, false, tid, NT);
    sync();
    uint32_t s = 0;
    uint32_t first = 0;  // N[0]
    {
      const uint32_t b = on ? xch[j] : 0u;
      const uint32_t before = on ? (j ? xch[j - 1] >> 31 : (xch[W - 1] >> lastb) & 1u) : 0u;
      s = (b ^ ((b << 1) | before)) & valid;
      first = xch[0] & 1u;
      const int n = __reduce_add_sync(kFull, copy == 0 ? __popc(b) : 0);
      if (lane == 0 && n) atomicAdd(&misc[0], n);
    }
    uint32_t C = 0;
    int t = 0, flag = 0, cur = 0, still = 0;
    if (keeps) ring[j] = s;
    bool any = sync_or(s != 0);
    const uint64_t k1 = a.move_thr ? splitmix64(a.move_key ^ (uint64_t)(a.shot_offset + shot)) : 0;
    const int c0 = j << 5;
    k0 = copy / v;
    r0 = copy - k0 * v;
    dk = copies / v;
    dr = copies - dk * v;
    lo0 = wrap(c0 - 1 - copy);
    hi0 = wrap(c0 + 1 + copy);
    // sites whose draws this copy makes
    const uint32_t share = copies == 1 ? kFull : (kFull / ((1u << copies) - 1u)) << copy;
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
        for (uint32_t b = s & share; b; b &= b - 1) {
          const int q = __ffs(b) - 1;
          const uint64_t r = splitmix64(key ^ (uint64_t)(c0 + q));
          if (r < a.move_thr) {
            if (splitmix64(r) >> 63) left |= 1u << q;
            else right |= 1u << q;
          }
        }
        left = across(left);
        right = across(right);
        u &= ~(left | right);
      }
      // ---- nearest anyon of the past on either side
      const int lastk = min(t, kmax);
      int slot = cur;
      if (NT == 32 && copies > 1) search_copies(u, left, right, lastk, cur);
#pragma unroll 1
      for (int k = 0; k <= lastk && copies == 1; ++k) {
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
        const uint32_t nb = __shfl_sync(kFull, left, last ? lane - j : lane + 1) & 1u;
        F = (right | (left >> 1) | (nb << (last ? lastb : 31))) & valid;
        Fb = __shfl_sync(kFull, F, j ? lane - 1 : lane + W - 1);
        Fb = j ? Fb >> 31 : (Fb >> lastb) & 1u;
      } else {
        if (on) xch[j] = left;
        sync();
        const uint32_t nb = on ? xch[last ? 0 : j + 1] & 1u : 0u;
        F = (right | (left >> 1) | (nb << (last ? lastb : 31))) & valid;
        if (on) xch[W + j] = F;
        sync();
        Fb = on ? (j ? xch[W + j - 1] >> 31 : (xch[W + W - 1] >> lastb) & 1u) : 0u;
      }
      C ^= F;
      s = (s ^ F ^ ((F << 1) | Fb)) & valid;
      cur = cur + 1 == depth ? 0 : cur + 1;
      if (keeps) ring[cur * W + j] = s;
      // without random moves a ring that has not moved for kmax + 1 steps never
      // moves again
      if (!a.move_thr) still = sync_or(F != 0) ? 0 : still + 1;
      any = sync_or(s != 0);
      ++t;
    }
    // ---- outputs
    if (keeps) xch[j] = C;
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

  // The nearest anyons of the past for the undecided sites u (the same in all copies):
  // copy i looks at distance i + 1 of each `copies` distances, and decides the sites
  // that no copy before it has decided.
  __device__ __forceinline__ void search_copies(uint32_t u, uint32_t& left, uint32_t& right,
                                                int lastk, int cur) const {
    const int v = a.v, L = a.L, dmax = min(v * (lastk + 1), a.m_max);
    int slot = cur - k0, rest = r0, lo = lo0, hi = hi0;
    if (slot < 0) slot += depth;
#pragma unroll 1
    for (int base = 0; __any_sync(kFull, u != 0);) {
      uint32_t p = 0, m = 0;
      if (u && base + copy < dmax) {
        const uint32_t* w = ring + slot * W;
        p = window(w, lo) & u;  // from the left: m^+
        m = window(w, hi) & u;
      }
      uint32_t hit = p | m;
      if (__any_sync(kFull, hit != 0)) {
        const uint32_t own_l = p & ~m, own_r = m & ~p;
#pragma unroll 1
        for (int o = stride; o < 32; o <<= 1) {
          const uint32_t h = __shfl_up_sync(kFull, hit, o);
          if (lane >= o) hit |= h;
        }
        uint32_t before = __shfl_up_sync(kFull, hit, stride);
        if (copy == 0) before = 0;
        left |= own_l & ~before;
        right |= own_r & ~before;
        u &= ~__shfl_sync(kFull, hit, 32 - stride + j);
      }
      base += copies;
      if (base >= dmax) break;
      if (copies <= 4 && base >= 3 * v) {
        uint32_t mine = copy == 0 ? u : 0u;
        if (__reduce_add_sync(kFull, __popc(mine)) <= kRingFew) {
          one_by_one(mine, left, right, base / v, lastk, cur);
          break;
        }
      }
      // the next distance of this copy
      slot -= dk;
      rest += dr;
      if (rest >= v) {
        rest -= v;
        --slot;
      }
      if (slot < 0) slot += depth;
      lo -= copies;
      if (lo < 0) lo += L;
      hi += copies;
      if (hi >= L) hi -= L;
    }
    left = across(left);
    right = across(right);
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
