// Synchronous decoding from the syndrome history (v = 3), device side.
//
// Unrolling the update rule of A^(D) (Def. Dd_msg_passing) gives every message
// field in closed form: after step t,
//   m^{s a}_r = min { d : 1 <= d <= m_max, sigma_{t - floor((d - 1) / v)} has an
//                     anyon at r - s d a^ + j b^ for some |j| <= d },
// because a message started in the sub-step d - 1 sub-steps ago has moved d
// sites along its axis and up to d sites across it, and the nearest start wins.
// Forces are needed at anyon sites only (reading R2), and of an anyon's four
// fields only the smallest distance matters and which directions attain it
// (with QCA_TIE_LITERAL also which attain the next one).  So no message plane
// is kept: the state is the site bitmaps of the last syndromes, and a step
// looks outward from each anyon, three distances ("slice" k: distances 3k + 1
// .. 3k + 3, all read from sigma_{t-k}) at a time, until one finds an anyon.
// Anyons thin out quickly and see each other at short range (L = 256, p =
// 0.05: 11 230, 3811, 1478, 641, 300, 160, 93, ... anyons per step, mean
// distance 1.0, 1.2, 1.4, 1.6, 2.0, 2.4, 2.6, ...), so a shot costs some 18
// thousand short searches instead of 18 sweeps over 4 x 65 536 fields.
//
// One CTA of NT threads decodes one shot.  A step runs in one of three modes:
//   dense   many anyons: distance 1 of all anyons 32 sites per bitmap word, the
//           undecided ones (a few per cent) listed and searched one by one;
//   listed  at most sparse_max anyons, one thread per anyon for slice 0, a
//           whole warp per anyon beyond it;
//   few     at most 8 anyons: one warp runs all remaining steps by itself, one
//           lane per (anyon, slice), from a ring of the last anyon sets.
// Flipped links are marked in a map, so that a link crossed from both ends
// flips once (the OR of Eq. ddfeedback).
#pragma once

#include <type_traits>

#include "qca_internal.cuh"

namespace qca {
namespace hist {

constexpr int kFew = 8;        // most anyons of the few-anyon mode
constexpr int kFewRing = 128;  // steps of anyon sets it keeps (more than 85)
constexpr int kLargeRing = 88; // syndromes kept per shot above L = 256 (more than 85)
constexpr uint32_t kFull = 0xffffffffu;

struct Geom {
  int L;
  int lws;         // log2 of the 32-bit words per bitmap row
  int nws;         // words of one site bitmap (L << lws)
  int kmask;       // syndromes kept in shared memory, less one (a power of two less one)
  int spill;       // most older syndromes kept in the correction block (0: none needed)
  int kmax;        // oldest slice a message can come from: (m_max - 1) / 3
  int sparse_max;  // most anyons of the listed mode
  int list_cap;    // entries of the anyon list
  // word offsets in the CTA's shared memory (L <= 256) or its global slot
  int o_C, o_F, o_list, o_few, o_misc;
};

__device__ __forceinline__ int wrap_lo(int i, int L) { return i < 0 ? i + L : i; }
__device__ __forceinline__ int wrap_hi(int i, int L) { return i >= L ? i - L : i; }

// Bits c, c + 1, ..., c + n - 1 (mod L) of a bitmap row; n <= 32, n <= L, 0 <= c < L.
__device__ __forceinline__ uint32_t row_bits_wrapped(const uint32_t* row, int wpr, int L, int c,
                                                     int n) {
  const int w = c >> 5, sh = c & 31;
  const uint32_t lo = row[w];
  const uint32_t hi = w + 1 < wpr ? row[w + 1] : 0u;
  uint32_t v = __funnelshift_r(lo, hi, sh);  // the bits past column L - 1 are 0
  if (c + n > L) v |= row[0] << (L - c);     // L - c < n <= 32
  return n >= 32 ? v : v & ((1u << n) - 1u);
}

// Any anyon within `reach` columns of x in a bitmap row.
__device__ __forceinline__ uint32_t row_any(const uint32_t* row, int wpr, int L, int x,
                                            int reach) {
  uint32_t any = 0;
  if (2 * reach + 1 >= L) {
    for (int w = 0; w < wpr; ++w) any |= row[w];
  } else {
    int c = wrap_lo(x - reach, L);
    for (int left = 2 * reach + 1; left > 0; left -= 32) {
      any |= row_bits_wrapped(row, wpr, L, c, left < 32 ? left : 32);
      c = wrap_hi(c + 32, L);
      if (c >= L) c %= L;  // L < 32
    }
  }
  return any != 0;
}

// Hits of one slice as 12 bits: bit 4 (d - 1) + f is set when the anyon hears
// field f (0 +x, 1 -x, 2 +y, 3 -y) at distance 3k + d.  m_max cuts the last slice.
__device__ __forceinline__ uint32_t slice_limit(int m_max, int k) {
  const int n = m_max - 3 * k;
  return n >= 3 ? 0xFFFu : (n == 2 ? 0xFFu : (n == 1 ? 0xFu : 0u));
}

// Slice 0 of the anyon at (x, y), by one thread: a 7 x 7 neighbourhood.
__device__ __forceinline__ uint32_t slice0(const uint32_t* sig, int lws, int L, int x, int y) {
  const int wpr = 1 << lws;
  const int s = wrap_lo(x - 3, L);
  const int w0 = s >> 5, sh = s & 31;
  const int w1 = min(w0 + 1, wpr - 1);
  const int sl = w0 < wpr - 1 ? 32 - sh : 32;  // 1 .. 32
  const int n0 = s + 7 > L ? L - s : 0;        // columns before the wrap, if any
  uint32_t r[7];  // bit i: column x - 3 + i of row y - 3 + j
#pragma unroll
  for (int j = 0; j < 7; ++j) {
    const int yy = wrap_hi(wrap_lo(y + j - 3, L), L);
    const uint32_t* row = sig + (yy << lws);
    uint32_t v = (row[w0] >> sh) | __funnelshift_lc(0u, row[w1], sl);
    if (n0) v |= row[0] << n0;  // the bits past column L - 1 are 0
    r[j] = v & 0x7Fu;
  }
  const uint32_t v1 = r[2] | r[3] | r[4];
  const uint32_t v2 = v1 | r[1] | r[5];
  const uint32_t v3 = v2 | r[0] | r[6];
  // +x comes from column x - d, -x from x + d, +y from row y - d, -y from y + d
  uint32_t m = ((v1 >> 2) & 1u) | ((v1 >> 3) & 2u);
  m |= ((v2 << 3) & 0x10u) | (v2 & 0x20u);
  m |= ((v3 << 8) & 0x100u) | ((v3 << 3) & 0x200u);
  m |= (r[2] & 0x1Cu) ? 0x4u : 0u;
  m |= (r[4] & 0x1Cu) ? 0x8u : 0u;
  m |= (r[1] & 0x3Eu) ? 0x40u : 0u;
  m |= (r[5] & 0x3Eu) ? 0x80u : 0u;
  m |= r[0] ? 0x400u : 0u;
  m |= r[6] ? 0x800u : 0u;
  return m;
}

// Slice k >= 1 of the anyon at (x, y) by a whole warp, from the bitmap of
// sigma_{t-k}: a lane per row for the x fields (three columns on either side),
// six lanes for the y fields' rows.
__device__ __forceinline__ uint32_t slice_warp(const uint32_t* sig, int lws, int L, int x, int y,
                                               int k, int lane) {
  const int wpr = 1 << lws;
  const int r = 3 * k + 3;
  const int nrows = min(2 * r + 1, L);
  const int half = nrows == L ? (L - 1) >> 1 : r;
  const int cl = wrap_lo(x - r % L, L);              // columns x - 3k - 3 ..
  const int cr = wrap_hi(x + (3 * k + 1) % L, L);    // columns x + 3k + 1 ..
  uint32_t m = 0;
  for (int i = lane; i < nrows; i += 32) {
    const int j = i - half;
    const uint32_t* row = sig + (wrap_hi(wrap_lo(y + j, L), L) << lws);
    const uint32_t l = row_bits_wrapped(row, wpr, L, cl, 3);  // d = 3, 2, 1
    const uint32_t q = row_bits_wrapped(row, wpr, L, cr, 3);  // d = 1, 2, 3
    uint32_t h = ((l >> 2) & 1u) | ((q << 1) & 2u) | ((l << 3) & 0x10u) | ((q << 4) & 0x20u) |
                 ((l << 8) & 0x100u) | ((q << 7) & 0x200u);
    const int aj = (j < 0 ? -j : j) - 3 * k;  // |j| <= 3k + d
    if (aj > 1) h &= aj > 2 ? 0xF00u : 0xFF0u;
    m |= h;
  }
  if (lane < 6) {
    const int d = lane < 3 ? lane + 1 : lane - 2;
    const int reach = 3 * k + d, dr = reach % L;
    const int yy = lane < 3 ? wrap_lo(y - dr, L) : wrap_hi(y + dr, L);
    m |= row_any(sig + (yy << lws), wpr, L, x, reach) << (4 * (d - 1) + (lane < 3 ? 2 : 3));
  }
  return __reduce_or_sync(kFull, m);
}

// Slice k of the anyon at (xa, ya) against one anyon (xb, yb) of sigma_{t-k};
// c = (3k + 1) mod L.
__device__ __forceinline__ uint32_t slice_pair(int xa, int ya, int xb, int yb, int L, int k,
                                               int c) {
  const int dx = wrap_lo(xa - xb, L), dy = wrap_lo(ya - yb, L);
  const int ax = min(dx, L - dx), ay = min(dy, L - dy);
  // e: distance less 3k + 1 of the first distance from 3k + 1 on that is
  // congruent to the offset along the field's direction
  auto first = [&](int off) { return wrap_lo(off - c, L); };
  const int epx = first(dx), emx = first(dx ? L - dx : 0);
  const int epy = first(dy), emy = first(dy ? L - dy : 0);
  uint32_t m = 0;
  if (epx < 3 && ay <= 3 * k + 1 + epx) m |= 1u << (4 * epx);
  if (emx < 3 && ay <= 3 * k + 1 + emx) m |= 2u << (4 * emx);
  if (epy < 3 && ax <= 3 * k + 1 + epy) m |= 4u << (4 * epy);
  if (emy < 3 && ax <= 3 * k + 1 + emy) m |= 8u << (4 * emy);
  return m;
}

// Direction from the fields heard at the smallest distance (h0, never 0) and,
// for QCA_TIE_LITERAL, at the next one (h1): 1 +x, 2 -x, 3 +y, 4 -y, 5 / 6 a
// balanced x / y axis.  Lexicographic order: -y, -x, +x, +y.  Literal key
// 3m + s a: -y, -x at the smallest distance, then -y at the next, +x, -x at the
// next, +y (equal keys go to the larger m).
__device__ __forceinline__ int direction(uint32_t h0, uint32_t h1, int tie_order) {
  if (h0 & 8u) return (h0 & 4u) ? 6 : 3;
  if (tie_order == QCA_TIE_LITERAL) {
    if (h0 & 2u) return (h0 & 1u) ? 5 : 1;
    if (h1 & 8u) return (h0 & 4u) ? 4 : ((h1 & 4u) ? 6 : 3);
    if (h0 & 1u) return 2;
    if (h1 & 2u) return (h1 & 1u) ? 5 : 1;
    return 4;
  }
  if (h0 & 3u) return (h0 & 3u) == 3u ? 5 : ((h0 & 1u) ? 2 : 1);
  return 4;
}

// Whether the next distance's hits are needed beside h0 (literal ties).
__device__ __forceinline__ bool needs_next(uint32_t h0, int tie_order) {
  return tie_order == QCA_TIE_LITERAL && !(h0 & 10u);
}

// 16 bytes of 0 / 1 -> 16 bits; ANY: of zero / nonzero.
template <bool ANY>
__device__ __forceinline__ uint32_t pack4(uint32_t w) {
  if (ANY) w = ((((w & 0x7F7F7F7Fu) + 0x7F7F7F7Fu) | w) & 0x80808080u) >> 7;
  return (w * 0x01020408u) >> 24;
}
template <bool ANY>
__device__ __forceinline__ uint32_t pack16(uint4 v) {
  return pack4<ANY>(v.x) | (pack4<ANY>(v.y) << 4) | (pack4<ANY>(v.z) << 8) |
         (pack4<ANY>(v.w) << 12);
}
// 4 bits -> 4 bytes of 0 / 1.
__device__ __forceinline__ uint32_t unpack4(uint32_t nib) {
  return (nib * 0x00204081u) & 0x01010101u;
}

// rows x L bytes at src -> bitmap rows (2^lws words each, padding bits 0).
template <int NT, bool ANY>
__device__ __forceinline__ void load_bits(const uint8_t* src, int rows, int L, int lws,
                                          uint32_t* dst, int tid) {
  if ((L & 15) == 0 && (reinterpret_cast<uintptr_t>(src) & 15) == 0) {
    // 16 bytes per lane and access: a warp reads 512 contiguous bytes
    const int vpr = L >> 4, n = rows * vpr;
    const uint4* s16 = reinterpret_cast<const uint4*>(src);
    uint16_t* d16 = reinterpret_cast<uint16_t*>(dst);
    const int dr = NT / vpr, dc = NT - dr * vpr;
    int r = tid / vpr, c = tid - r * vpr;
#pragma unroll 8
    for (int i = tid; i < n; i += NT) {
      const uint4 v = __ldcs(s16 + i);
      d16[(r << (lws + 1)) + c] = (uint16_t)pack16<ANY>(v);
      r += dr;
      c += dc;
      if (c >= vpr) {
        c -= vpr;
        ++r;
      }
    }
    return;
  }
  // any size and alignment: a bitmap word per thread from aligned 32-bit
  // loads, single bytes at the two ends of the block
  const uint8_t* end = src + (size_t)rows * L;
  const int wpr = 1 << lws;
  for (int i = tid; i < rows << lws; i += NT) {
    const int r = i >> lws, x0 = (i & (wpr - 1)) << 5;
    if (x0 >= L) continue;
    const int n = min(32, L - x0);
    const uint8_t* p = src + (size_t)r * L + x0;
    const int mis = (int)(reinterpret_cast<uintptr_t>(p) & 3);
    const uint8_t* q = p - mis;
    uint64_t acc = 0;
    const int nw = (mis + n + 3) >> 2;
    for (int w = 0; w < nw; ++w, q += 4) {
      uint32_t v = 0;
      if (q >= src && q + 4 <= end) {
        v = *reinterpret_cast<const uint32_t*>(q);
      } else {
        for (int b = 0; b < 4; ++b)
          if (q + b >= src && q + b < end) v |= (uint32_t)q[b] << (8 * b);
      }
      acc |= (uint64_t)(pack4<ANY>(v) & 0xFu) << (4 * w);
    }
    const uint32_t bits = (uint32_t)(acc >> mis);
    dst[i] = n == 32 ? bits : bits & ((1u << n) - 1u);
  }
}

// Bitmap rows -> rows x L bytes of 0 / 1 at out.
template <int NT>
__device__ __forceinline__ void store_bits(uint8_t* out, int rows, int L, int lws,
                                           const uint32_t* src, int tid) {
  if ((L & 15) == 0 && (reinterpret_cast<uintptr_t>(out) & 15) == 0) {
    const int vpr = L >> 4, n = rows * vpr;
    uint4* o16 = reinterpret_cast<uint4*>(out);
    const uint16_t* s16 = reinterpret_cast<const uint16_t*>(src);
    const int dr = NT / vpr, dc = NT - dr * vpr;
    int r = tid / vpr, c = tid - r * vpr;
#pragma unroll 4
    for (int i = tid; i < n; i += NT) {
      const uint32_t b = s16[(r << (lws + 1)) + c];
      __stcs(o16 + i, make_uint4(unpack4(b & 15u), unpack4((b >> 4) & 15u),
                                 unpack4((b >> 8) & 15u), unpack4(b >> 12)));
      r += dr;
      c += dc;
      if (c >= vpr) {
        c -= vpr;
        ++r;
      }
    }
    return;
  }
  // any size and alignment: aligned groups of four bytes, single bytes at the ends
  const int total = rows * L;
  const int head = (int)((4 - (reinterpret_cast<uintptr_t>(out) & 3)) & 3);
  for (int i = tid; 4 * i - 4 + head < total; i += NT) {
    const int f0 = 4 * i - 4 + head;  // group 0 holds the bytes before the first boundary
    const int fs = max(f0, 0);
    int r = fs / L, x = fs - r * L;
    uint32_t v = 0;
    for (int b = fs - f0; b < 4; ++b) {
      if (f0 + b >= total) break;
      v |= ((src[(r << lws) + (x >> 5)] >> (x & 31)) & 1u) << (8 * b);
      if (++x == L) {
        x = 0;
        ++r;
      }
    }
    if (f0 >= 0 && f0 + 4 <= total) {
      *reinterpret_cast<uint32_t*>(out + f0) = v;
    } else {
      for (int b = 0; b < 4; ++b)
        if (f0 + b >= 0 && f0 + b < total) out[f0 + b] = (uint8_t)(v >> (8 * b));
    }
  }
}

// Words of the few-anyon mode: the ring of anyon sets and one snapshot of it
// (orbit detection); entries are 16 bits up to L = 256, 32 bits above.
template <bool LARGE>
constexpr int kFewWords = 2 * kFewRing * kFew / (LARGE ? 1 : 2);

template <int NT, bool LARGE>
struct Decoder {
  using Ent = typename std::conditional<LARGE, uint32_t, uint16_t>::type;

  const DecodeArgs& a;
  const Geom& g;
  uint32_t* ring;    // [kmask + 1][nws] (LARGE: [kLargeRing][nws])
  uint32_t* C;       // [2][nws] correction
  uint32_t* F;       // [2][nws] links flipped this step
  uint32_t* list;    // [list_cap] anyons (y << 16 | x)
  Ent* few;          // [kFewRing][kFew], then the snapshot
  int* misc;         // 0-2 rotating counters, 3 miss, 4 steps, 5 flag, 6-7 cuts
  uint32_t* spill;   // [nspill][nws] in the correction block
  int nspill;
  int64_t shot;
  int tid, lane, warp;
  int ph;            // rotating counter in use
  int tb;            // step of the newest bitmap

  __device__ __forceinline__ void sync() const {
    if (NT == 32) {
      __syncwarp();
    } else {
      __syncthreads();
    }
  }

  // bitmap of sigma_s for a step s <= tb + 1 (tb + 1: the next one, being made)
  __device__ __forceinline__ uint32_t* slot(int s) const {
    if (LARGE) return ring + (size_t)(s % kLargeRing) * g.nws;
    return ring + (s & g.kmask) * g.nws;
  }
  // bitmap of the older sigma_s, or null when it is no longer kept
  __device__ __forceinline__ const uint32_t* past(int s) const {
    if (LARGE) return slot(s);
    const int oldest = tb - g.kmask + 1;  // the slot of tb + 1 is already reused
    if (s >= oldest) return slot(s);
    if (s < oldest - nspill) return nullptr;
    return spill + (s % nspill) * g.nws;
  }

  // Sum of n over the CTA through rotating counter ph; ends with a barrier.
  __device__ __forceinline__ int total(int n) {
    n = __reduce_add_sync(kFull, n);
    if (NT == 32) {
      __syncwarp();
      return n;
    }
    if (lane == 0 && n) atomicAdd(&misc[ph], n);
    return next_counter();
  }
  // Barrier, value of counter ph, and on to the next one (the one after it is cleared).
  __device__ __forceinline__ int next_counter() {
    sync();
    const int v = misc[ph];
    const int p2 = ph == 0 ? 2 : ph - 1;
    if (tid == 0) misc[p2] = 0;
    ph = ph == 2 ? 0 : ph + 1;
    return v;
  }

  // Makes sigma_s (in its slot) the newest bitmap: moves the oldest one out of
  // the slot of s + 1, copies sigma_s there (the listed mode flips bits in it)
  // and, if asked, lists the anyons.  Returns their number; ends with a barrier.
  __device__ __forceinline__ int advance(int s, bool do_list) {
    const uint32_t* cur = slot(s);
    uint32_t* nxt = slot(s + 1);
    const int old = s + 1 - (g.kmask + 1);
    uint32_t* sp = (!LARGE && nspill && old >= 0) ? spill + (old % nspill) * g.nws : nullptr;
    const int wsm = (1 << g.lws) - 1;
    int n = 0;
    for (int w = tid; w < g.nws; w += NT) {
      const uint32_t v = cur[w];
      if (sp) sp[w] = nxt[w];
      nxt[w] = v;
      n += __popc(v);
    }
    tb = s;
    if (do_list) {
      int incl = n;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int v = __shfl_up_sync(kFull, incl, o);
        if (lane >= o) incl += v;
      }
      int base = 0;
      if (lane == 31 && incl) base = atomicAdd(&misc[ph], incl);
      base = __shfl_sync(kFull, base, 31);
      int pos = base + incl - n;
      if (n) {
        for (int w = tid; w < g.nws; w += NT) {
          uint32_t b = cur[w];
          const uint32_t yx = ((uint32_t)(w >> g.lws) << 16) | ((w & wsm) << 5);
          while (b) {
            const int q = __ffs(b) - 1;
            b &= b - 1;
            if (pos < g.list_cap) list[pos] = yx + q;
            ++pos;
          }
        }
      }
      return next_counter();
    }
    sync();
    return 0;
  }

  __device__ __forceinline__ uint32_t site(int x, int y) const { return (uint32_t)(y * g.L + x); }

  // Slices 1 .. of the anyon at (x, y) by the whole warp; returns the first
  // slice's hits (0: nothing heard) and its index in k.
  __device__ __forceinline__ uint32_t search_far(int x, int y, int t, int& k) const {
    const int last = min(t, g.kmax);
    for (; k <= last; ++k) {
      const uint32_t* sig = past(t - k);
      if (!sig) {
        misc[3] = 1;  // the shot needs a syndrome that is no longer kept
        return 0;
      }
      const uint32_t m = slice_warp(sig, g.lws, g.L, x, y, k, lane) & slice_limit(a.m_max, k);
      if (m) return m;
    }
    return 0;
  }

  struct Keys {
    uint64_t move, bal;
  };
  __device__ __forceinline__ Keys keys_of(int t) const {
    Keys q{0, 0};
    if (a.move_thr) q.move = move_step_key(a.move_key, a.shot_offset + shot, t);
    if (a.balance_rule) q.bal = move_step_key(a.balance_key, a.shot_offset + shot, t);
    return q;
  }
  // Random move of the anyon at site r, or 0.
  __device__ __forceinline__ int drawn_move(const Keys& q, uint32_t r) const {
    if (!a.move_thr) return 0;
    const uint64_t u = splitmix64(q.move ^ (uint64_t)r);
    return u < a.move_thr ? 1 + (int)(splitmix64(u) >> 62) : 0;
  }
  __device__ __forceinline__ int resolve(int dir, const Keys& q, uint32_t r) const {
    if (dir >= 5) dir = a.balance_rule ? balance_resolve(dir, q.bal, r) : 0;
    return dir;
  }

  // Lower end of the link an anyon at (x, y) crosses when it moves: word of the
  // link maps and bit.
  __device__ __forceinline__ int link_of(int x, int y, int dir, uint32_t& bit) const {
    const int lx = dir == 2 ? wrap_lo(x - 1, g.L) : x;
    const int ly = dir == 4 ? wrap_lo(y - 1, g.L) : y;
    bit = 1u << (lx & 31);
    return (dir >= 3 ? g.nws : 0) + (ly << g.lws) + (lx >> 5);
  }

  // Decides and marks the moves of the n listed anyons at step t.  LISTED: the
  // correction and the copy of sigma in the next slot are flipped at once and
  // the marked words are returned in mark[] (4 per thread at most); else only
  // the link map is marked.
  template <bool LISTED>
  __device__ __forceinline__ void move_listed(int n, int t, int (&mark)[4]) {
    constexpr int NW = NT / 32;
    const uint32_t* sig = slot(t);
    uint32_t* sn = slot(t + 1);
    const Keys key = keys_of(t);
    const uint32_t lim0 = slice_limit(a.m_max, 0);
    const bool far = t > 0 && g.kmax > 0;
    auto one = [&](int it, int& mk) {
      // consecutive list entries go to different warps
      const int i = it * NT + lane * NW + warp;
      const bool act = i < n;
      int x = 0, y = 0, dir = 0, k = 0;
      uint32_t m = 0;
      bool need = false, edge = false;
      if (act) {
        const uint32_t e = list[i];
        x = e & 0xFFFFu;
        y = e >> 16;
        dir = drawn_move(key, site(x, y));
        if (!dir) {
          m = slice0(sig, g.lws, g.L, x, y) & lim0;
          need = far && m == 0;
        }
      }
      uint32_t todo = __ballot_sync(kFull, need);
      while (todo) {
        const int src = __ffs(todo) - 1;
        todo &= todo - 1;
        int kk = 1;
        const uint32_t mm = search_far(__shfl_sync(kFull, x, src), __shfl_sync(kFull, y, src), t,
                                       kk);
        if (lane == src) {
          m = mm;
          k = kk;
        }
      }
      uint32_t h0 = 0, h1 = 0;
      if (m) {
        const int d4 = (__ffs(m) - 1) & ~3;
        h0 = (m >> d4) & 15u;
        h1 = (m >> (d4 + 4)) & 15u;  // 0 past the slice's third distance
        edge = d4 == 8 && needs_next(h0, a.tie_order) && k < min(t, g.kmax);
      }
      todo = __ballot_sync(kFull, edge);
      while (todo) {
        // the next distance is the first one of the next slice
        const int src = __ffs(todo) - 1;
        todo &= todo - 1;
        const int ks = __shfl_sync(kFull, k, src) + 1;
        const uint32_t* ps = past(t - ks);
        uint32_t mm = 0;
        if (ps) {
          mm = slice_warp(ps, g.lws, g.L, __shfl_sync(kFull, x, src), __shfl_sync(kFull, y, src),
                          ks, lane) & slice_limit(a.m_max, ks);
        } else {
          misc[3] = 1;
        }
        if (lane == src) h1 = mm & 15u;
      }
      if (h0) dir = resolve(direction(h0, h1, a.tie_order), key, site(x, y));
      if (dir) {
        uint32_t bit;
        const int w = link_of(x, y, dir, bit);
        if (LISTED) {
          mk = w;
          if (!(atomicOr(&F[w], bit) & bit)) {
            const int nx = dir == 1 ? wrap_hi(x + 1, g.L) : (dir == 2 ? wrap_lo(x - 1, g.L) : x);
            const int ny = dir == 3 ? wrap_hi(y + 1, g.L) : (dir == 4 ? wrap_lo(y - 1, g.L) : y);
            atomicXor(&C[w], bit);
            atomicXor(&sn[(y << g.lws) + (x >> 5)], 1u << (x & 31));
            atomicXor(&sn[(ny << g.lws) + (nx >> 5)], 1u << (nx & 31));
          }
        } else {
          atomicOr(&F[w], bit);
        }
      }
    };
    if (LISTED) {
#pragma unroll
      for (int it = 0; it < 4; ++it) {
        mark[it] = -1;
        if (it * NT < n) one(it, mark[it]);
      }
    } else {
      int unused;
      for (int it = 0; it * NT < n; ++it) one(it, unused);
    }
  }

  // One anyon decided by one thread alone, all slices (the list is full).
  // A static function on a copy, so that the kernel's own state stays in registers.
  static __device__ __noinline__ int decide_alone(const Decoder self, int x, int y, int t,
                                                  const Keys key) {
    return self.decide(x, y, t, key);
  }
  __device__ __forceinline__ int decide(int x, int y, int t, const Keys& key) const {
    int dir = drawn_move(key, site(x, y));
    if (dir) return dir;
    const int last = min(t, g.kmax);
    uint32_t h0 = 0;
    for (int k = 0; k <= last; ++k) {
      const uint32_t* sig = past(t - k);
      if (!sig) {
        misc[3] = 1;
        return 0;
      }
      uint32_t m = 0;
      if (k == 0) {
        m = slice0(sig, g.lws, g.L, x, y);
      } else {
        for (int d = 1; d <= 3; ++d) {
          const int reach = 3 * k + d, dr = reach % g.L, wpr = 1 << g.lws;
          const int xl = wrap_lo(x - dr, g.L), xr = wrap_hi(x + dr, g.L);
          const int half = min(reach, g.L >> 1);
          uint32_t h = 0;
          for (int j = -half; j <= half; ++j) {
            const uint32_t* row = sig + (wrap_hi(wrap_lo(y + j, g.L), g.L) << g.lws);
            h |= ((row[xl >> 5] >> (xl & 31)) & 1u) | (((row[xr >> 5] >> (xr & 31)) & 1u) << 1);
          }
          h |= row_any(sig + (wrap_lo(y - dr, g.L) << g.lws), wpr, g.L, x, reach) << 2;
          h |= row_any(sig + (wrap_hi(y + dr, g.L) << g.lws), wpr, g.L, x, reach) << 3;
          m |= h << (4 * (d - 1));
        }
      }
      m &= slice_limit(a.m_max, k);
      if (h0) return resolve(direction(h0, m & 15u, a.tie_order), key, site(x, y));
      if (m) {
        const int d4 = (__ffs(m) - 1) & ~3;
        h0 = (m >> d4) & 15u;
        if (d4 < 8 || !needs_next(h0, a.tie_order))
          return resolve(direction(h0, (m >> (d4 + 4)) & 15u, a.tie_order), key, site(x, y));
      }
    }
    return h0 ? resolve(direction(h0, 0, a.tie_order), key, site(x, y)) : 0;
  }

  // Dense step t: distance 1 of every anyon 32 sites at a time, the others
  // listed.  Marks the crossed links; returns the number listed (ends with a
  // barrier).
  __device__ __forceinline__ int mark_dense(int t) {
    const uint32_t* sig = slot(t);
    const int L = g.L, lws = g.lws, wsm = (1 << lws) - 1;
    const int lastw = (L - 1) >> 5, lastb = (L - 1) & 31;
    const Keys key = keys_of(t);
    const bool lit = a.tie_order == QCA_TIE_LITERAL;
    for (int w = tid; w < g.nws; w += NT) {
      const uint32_t c = sig[w];
      if (!c) continue;
      const int y = w >> lws, j = w & wsm;
      const int yu = y == 0 ? L - 1 : y - 1, yd = y == L - 1 ? 0 : y + 1;
      const int jl = j == 0 ? lastw : j - 1, jr = j == lastw ? 0 : j + 1;
      const int sl = j == 0 ? lastb : 31, top = j == lastw ? lastb : 31;
      uint32_t todo;
      if (a.move_thr) {
        todo = c;  // any anyon may be drawn to move: one by one
      } else {
        const uint32_t *ru = sig + (yu << lws), *r0 = sig + (y << lws), *rd = sig + (yd << lws);
        const uint32_t u = ru[j], d = rd[j];
        const uint32_t ul = (ru[jl] >> sl) & 1u, cl = (r0[jl] >> sl) & 1u, dl = (rd[jl] >> sl) & 1u;
        const uint32_t ur = (ru[jr] & 1u) << top, cr = (r0[jr] & 1u) << top,
                       dr = (rd[jr] & 1u) << top;
        const uint32_t v = u | c | d;
        const uint32_t px = (v << 1) | ul | cl | dl;  // anyon in column x - 1
        const uint32_t mx = (v >> 1) | ur | cr | dr;  // in column x + 1
        const uint32_t py = u | (u << 1) | ul | (u >> 1) | ur;
        const uint32_t my = d | (d << 1) | dl | (d >> 1) | dr;
        uint32_t mpx, mmx, mpy, mmy, bx, by;  // moves +x, -x, +y, -y; balanced axes
        todo = c & ~(px | mx | py | my);
        mpy = c & my & ~py;
        by = c & my & py;
        uint32_t xs = c & ~my & (px | mx);
        mmy = c & py & ~(my | px | mx);
        if (lit) {
          // +x or +y alone at distance 1 may lose to -y or -x at distance 2
          todo |= c & ~(my | mx) & (px | py);
          xs &= mx;
          mmy = 0;
        }
        mpx = xs & mx & ~px;
        mmx = xs & px & ~mx;
        bx = xs & px & mx;
        if (a.balance_rule) {
          for (uint32_t b = bx; b; b &= b - 1) {
            const int q = __ffs(b) - 1;
            if (balance_resolve(5, key.bal, site((j << 5) + q, y)) == 1) mpx |= 1u << q;
            else mmx |= 1u << q;
          }
          for (uint32_t b = by; b; b &= b - 1) {
            const int q = __ffs(b) - 1;
            if (balance_resolve(6, key.bal, site((j << 5) + q, y)) == 3) mpy |= 1u << q;
            else mmy |= 1u << q;
          }
        }
        const uint32_t fx = mpx | (mmx >> 1);
        if (fx) atomicOr(&F[w], fx);
        if (mmx & 1u) atomicOr(&F[(y << lws) + jl], 1u << sl);
        if (mpy) atomicOr(&F[g.nws + w], mpy);
        if (mmy) atomicOr(&F[g.nws + (yu << lws) + j], mmy);
      }
      if (todo) {
        int pos = atomicAdd(&misc[ph], __popc(todo));
        while (todo) {
          const int q = __ffs(todo) - 1;
          todo &= todo - 1;
          if (pos < g.list_cap) {
            list[pos] = ((uint32_t)y << 16) | ((j << 5) + q);
          } else {
            const int x = (j << 5) + q;
            const int dir = decide_alone(*this, x, y, t, key);
            if (dir) {
              uint32_t bit;
              const int lw = link_of(x, y, dir, bit);
              atomicOr(&F[lw], bit);
            }
          }
          ++pos;
        }
      }
    }
    return min(next_counter(), g.list_cap);
  }

  // sigma_{t+1} and the correction from the marked links; the anyons left (ends
  // with a barrier).
  __device__ __forceinline__ int apply_dense(int t) {
    const uint32_t* sig = slot(t);
    uint32_t* sn = slot(t + 1);
    const int L = g.L, lws = g.lws, wsm = (1 << lws) - 1;
    const int lastw = (L - 1) >> 5, lastb = (L - 1) & 31;
    int n = 0;
    for (int w = tid; w < g.nws; w += NT) {
      const int y = w >> lws, j = w & wsm;
      if (j > lastw) continue;  // padding word (stays 0)
      const int yu = y == 0 ? L - 1 : y - 1;
      const uint32_t fx = F[w], fy = F[g.nws + w], fu = F[g.nws + (yu << lws) + j];
      const uint32_t carry =
          j ? F[w - 1] >> 31 : (F[(y << lws) + lastw] >> lastb) & 1u;
      const uint32_t valid = j == lastw ? kFull >> (31 - lastb) : kFull;
      const uint32_t s = sig[w] ^ ((fx ^ ((fx << 1) | carry) ^ fy ^ fu) & valid);
      sn[w] = s;
      n += __popc(s);
      if (fx) C[w] ^= fx;
      if (fy) C[g.nws + w] ^= fy;
    }
    return total(n);
  }

  // --------------------------------------------------------- few anyons
  __device__ __forceinline__ Ent enc(uint32_t p) const {
    return LARGE ? (Ent)p : (Ent)(((p >> 16) << 8) | (p & 0xFFu));
  }
  __device__ __forceinline__ uint32_t dec(Ent e) const {
    return LARGE ? (uint32_t)e : (((uint32_t)e >> 8) << 16) | ((uint32_t)e & 0xFFu);
  }
  // Hits of slice k against the anyon set of step s (a set shorter than 8
  // entries is filled with its first one).
  __device__ __forceinline__ uint32_t slice_set(int s, int x, int y, int k) const {
    const uint4* p = reinterpret_cast<const uint4*>(few + (s & (kFewRing - 1)) * kFew);
    uint32_t e[kFew];
    const uint4 v = p[0];
    if constexpr (LARGE) {
      const uint4 u = p[1];
      e[0] = v.x, e[1] = v.y, e[2] = v.z, e[3] = v.w;
      e[4] = u.x, e[5] = u.y, e[6] = u.z, e[7] = u.w;
    } else {
      e[0] = v.x & 0xFFFFu, e[1] = v.x >> 16, e[2] = v.y & 0xFFFFu, e[3] = v.y >> 16;
      e[4] = v.z & 0xFFFFu, e[5] = v.z >> 16, e[6] = v.w & 0xFFFFu, e[7] = v.w >> 16;
    }
    int c = 3 * k + 1;
    if (c >= g.L) c %= g.L;
    uint32_t m = 0;
#pragma unroll
    for (int q = 0; q < kFew; ++q) {
      if (q > 0 && e[q] == e[0]) break;
      const uint32_t b = dec((Ent)e[q]);
      m |= slice_pair(x, y, (int)(b & 0xFFFFu), (int)(b >> 16), g.L, k, c);
    }
    return m & slice_limit(a.m_max, k);
  }
  // Slice k of one anyon at step t by the whole warp, from the set or the bitmap.
  __device__ __forceinline__ uint32_t slice_any(int x, int y, int t, int k, int tf) const {
    if (t - k >= tf) return slice_set(t - k, x, y, k);
    const uint32_t* sig = past(t - k);
    if (!sig) {
      misc[3] = 1;
      return 0;
    }
    return slice_warp(sig, g.lws, g.L, x, y, k, lane) & slice_limit(a.m_max, k);
  }

  // All steps from t on, with n <= 8 anyons in the list, by one warp.  Leaves
  // the step count in misc[4] and the budget flag in misc[5].
  //
  // Periodic orbits: with the deterministic rules a step is a function of the
  // last kmax + 1 anyon sets, so once those equal the ones of P steps before,
  // the shot never ends, its anyons at max_steps are those of any step
  // congruent to it modulo P, and the correction, which gains the same flips
  // every period, repeats with period 2P.  The sets are compared with a
  // snapshot that is renewed at doubling intervals (Brent's cycle search), and
  // the shot stops at the first step whose outcome is the budget's.
  __device__ __forceinline__ void few_steps(int t, int n) {
    const int L = g.L, tf = t;
    const bool lit = a.tie_order == QCA_TIE_LITERAL;
    const bool watch = a.move_thr == 0 && a.balance_rule == QCA_BALANCE_STAY;
    Ent* snap = few + kFewRing * kFew;
    int t_snap = -1, t_renew = tf + g.kmax + 1, interval = 64, t_stop = -1;
    int flag = 0;
    uint32_t pos = lane < n ? list[lane] : 0;
    {  // sorted set of the first step
      int rank = 0;
      for (int q = 0; q < n; ++q) rank += __shfl_sync(kFull, pos, q) < pos;
      if (lane < n) few[(t & (kFewRing - 1)) * kFew + rank] = enc(pos);
      __syncwarp();
      Ent* row = few + (t & (kFewRing - 1)) * kFew;
      if (lane >= n && lane < kFew) row[lane] = row[0];
      __syncwarp();
      pos = lane < n ? dec(row[lane]) : 0;
    }
    while (n) {
      if (t >= a.max_steps || t == t_stop) {
        flag = 2;
        t = a.max_steps;
        break;
      }
      if (watch && t_stop < 0) {
        if (t_snap >= 0 && t > t_snap) {
          const Ent* now = few + (t & (kFewRing - 1)) * kFew;
          const Ent* then = snap + (t_snap & (kFewRing - 1)) * kFew;
          bool same = lane >= kFew || now[lane] == then[lane];
          if (__all_sync(kFull, same)) {
            for (int i = lane; i <= g.kmax && same; i += 32) {
              const Ent* p = few + ((t - i) & (kFewRing - 1)) * kFew;
              const Ent* q = snap + ((t_snap - i) & (kFewRing - 1)) * kFew;
#pragma unroll
              for (int b = 0; b < kFew; ++b) same = same && p[b] == q[b];
            }
            if (__all_sync(kFull, same)) {
              const int P = t - t_snap, R = a.max_steps - t, per = R / P;
              t_stop = t + (R - per * P) + ((per & 1) ? P : 0);
              if (t_stop == t) continue;
            }
          }
        }
        if (t_stop < 0 && t >= t_renew) {
          // (kFewRing entries cover the kmax + 1 <= 85 sets ending at t)
          for (int i = lane; i < kFewRing * kFew; i += 32) snap[i] = few[i];
          t_snap = t;
          t_renew = t + interval;
          interval <<= 1;
          __syncwarp();
        }
      }
      const Keys key = keys_of(t);
      const int last = min(t, g.kmax), lastl = min(last, t - tf);
      // lanes = (anyon, slice)
      const int lgS = n <= 2 ? 4 : (n <= 4 ? 3 : 2), S = 1 << lgS;
      const int ai = lane >> lgS, kk = lane & (S - 1);
      const uint32_t pa = __shfl_sync(kFull, pos, ai);
      const int xa = pa & 0xFFFFu, ya = pa >> 16;
      uint32_t h0 = 0, h1 = 0;
      int kf = 0;
      bool done = ai >= n, edge = false;
      for (int kb = 0; kb <= lastl; kb += S) {
        uint32_t m = 0;
        if (!done && kb + kk <= lastl) m = slice_set(t - kb - kk, xa, ya, kb + kk);
        const uint32_t seg = (__ballot_sync(kFull, m != 0) >> (ai << lgS)) & ((1u << S) - 1u);
        const int src = (ai << lgS) + (seg ? __ffs(seg) - 1 : 0);
        const uint32_t hm = __shfl_sync(kFull, m, src);
        if (!done && seg) {
          const int d4 = (__ffs(hm) - 1) & ~3;
          h0 = (hm >> d4) & 15u;
          h1 = (hm >> (d4 + 4)) & 15u;
          kf = kb + src - (ai << lgS);
          edge = d4 == 8 && needs_next(h0, a.tie_order) && kf < last;
          done = true;
        }
        if (__all_sync(kFull, done)) break;
      }
      // anyons that hear nothing from the sets: the bitmaps before them
      uint32_t todo = __ballot_sync(kFull, kk == 0 && ai < n && h0 == 0 && lastl < last);
      while (todo) {
        const int src = __ffs(todo) - 1;
        todo &= todo - 1;
        int k = lastl + 1;
        const uint32_t mm = search_far(__shfl_sync(kFull, xa, src), __shfl_sync(kFull, ya, src), t,
                                       k);
        if (lane == src && mm) {
          const int d4 = (__ffs(mm) - 1) & ~3;
          h0 = (mm >> d4) & 15u;
          h1 = (mm >> (d4 + 4)) & 15u;
          kf = k;
          edge = d4 == 8 && needs_next(h0, a.tie_order) && k < last;
        }
      }
      if (lit) {
        todo = __ballot_sync(kFull, kk == 0 && edge);
        while (todo) {
          const int src = __ffs(todo) - 1;
          todo &= todo - 1;
          const uint32_t mm =
              slice_any(__shfl_sync(kFull, xa, src), __shfl_sync(kFull, ya, src), t,
                        __shfl_sync(kFull, kf, src) + 1, tf);
          if (lane == src) h1 = mm & 15u;
        }
      }
      __syncwarp();
      if (!LARGE && *(volatile int*)&misc[3]) return;
      // the moves, anyon i on lane i
      h0 = __shfl_sync(kFull, h0, (lane << lgS) & 31);
      h1 = __shfl_sync(kFull, h1, (lane << lgS) & 31);
      const int x = pos & 0xFFFFu, y = pos >> 16;
      int dir = 0;
      if (lane < n) {
        dir = drawn_move(key, site(x, y));
        if (!dir && h0) dir = resolve(direction(h0, h1, a.tie_order), key, site(x, y));
      }
      uint32_t np = pos, bit = 0;
      int lw = 0;
      if (dir) {
        lw = link_of(x, y, dir, bit);
        const int nx = dir == 1 ? wrap_hi(x + 1, L) : (dir == 2 ? wrap_lo(x - 1, L) : x);
        const int ny = dir == 3 ? wrap_hi(y + 1, L) : (dir == 4 ? wrap_lo(y - 1, L) : y);
        np = ((uint32_t)ny << 16) | nx;
      }
      // a link crossed from both ends flips once and takes both anyons;
      // otherwise the anyons are where an odd number of them end
      int crossed = 0, first_cross = 1;
      for (int q = 0; q < n; ++q) {
        const uint32_t bq = __shfl_sync(kFull, bit, q);
        const int wq = __shfl_sync(kFull, lw, q);
        const bool eq = dir && bq == bit && wq == lw;
        crossed += eq;
        if (eq && q < lane) first_cross = 0;
      }
      if (dir && first_cross) atomicXor(&C[lw], bit);
      const bool stays = lane < n && crossed < 2;
      if (!stays) np = 0x80000000u | lane;
      int same = 0, lower = 0;
      for (int q = 0; q < n; ++q) {
        const uint32_t v = __shfl_sync(kFull, np, q);
        same += v == np;
        lower += v == np && q < lane;
      }
      const bool alive = stays && (same & 1) && lower == 0;
      const uint32_t am = __ballot_sync(kFull, alive);
      int rank = 0;
      for (int q = 0; q < n; ++q) {
        const uint32_t v = __shfl_sync(kFull, np, q);
        rank += ((am >> q) & 1u) && v < np;
      }
      ++t;
      n = __popc(am);
      Ent* row = few + (t & (kFewRing - 1)) * kFew;
      if (alive) row[rank] = enc(np);
      __syncwarp();
      if (lane >= n && lane < kFew) row[lane] = row[0];
      __syncwarp();
      pos = lane < n ? dec(row[lane]) : 0;
    }
    if (lane == 0) {
      misc[4] = t;
      misc[5] = flag;
    }
  }

  // ------------------------------------------------------------ one shot
  __device__ __forceinline__ void run() {
    const int L = g.L, LL = L * L, lws = g.lws;
    const int lastw = (L - 1) >> 5, lastb = (L - 1) & 31;
    const uint8_t* N = a.in + shot_offset_of(a, shot);
    uint8_t* outC = a.out_C + correction_offset_of(a, shot);
    spill = reinterpret_cast<uint32_t*>(
        (reinterpret_cast<uintptr_t>(outC) + 3) & ~(uintptr_t)3);
    nspill = min(g.spill, (2 * LL - (int)(reinterpret_cast<uint8_t*>(spill) - outC)) / (4 * g.nws));
    if (tid < 8) misc[tid] = 0;
    ph = 0;
    tb = 0;
    // ---- sigma_0 (Def. synch_ccqs) and the cut parities of N
    int wx = 0, wy = 0, n = 0;
    uint32_t* s0 = slot(0);
    if (a.from_sigma) {
      for (int w = tid; w < g.nws; w += NT) s0[w] = 0;
      sync();
      load_bits<NT, true>(N, L, L, lws, s0, tid);
      for (int w = tid; w < 2 * g.nws; w += NT) C[w] = 0;
      for (int w = tid; w < 2 * g.nws; w += NT) F[w] = 0;
      sync();
      for (int w = tid; w < g.nws; w += NT) n += __popc(s0[w]);
    } else {
      // the link bits, in the correction's place
      if (L & 31) {
        for (int w = tid; w < 2 * g.nws; w += NT) C[w] = 0;
        sync();
      }
      load_bits<NT, false>(N, 2 * L, L, lws, C, tid);
      for (int w = tid; w < 2 * g.nws; w += NT) F[w] = 0;
      sync();
      const int wsm = (1 << lws) - 1;
      for (int w = tid; w < g.nws; w += NT) {
        const int y = w >> lws, j = w & wsm;
        uint32_t s = 0;
        if (j <= lastw) {
          const int yu = y == 0 ? L - 1 : y - 1;
          const uint32_t bx = C[w], by = C[g.nws + w], bu = C[g.nws + (yu << lws) + j];
          const uint32_t carry = j ? C[w - 1] >> 31 : (C[(y << lws) + lastw] >> lastb) & 1u;
          s = (bx ^ ((bx << 1) | carry) ^ by ^ bu) &
              (j == lastw ? kFull >> (31 - lastb) : kFull);
          if (j == 0) wx ^= (int)(bx & 1u);
          if (y == 0) wy ^= __popc(by) & 1;
        }
        s0[w] = s;
        n += __popc(s);
      }
      sync();
      for (int w = tid; w < 2 * g.nws; w += NT) C[w] = 0;
    }
    n = total(n);
    int t = 0, flag = 0;
    if (n) advance(0, n <= g.sparse_max);
    // ---- steps
    while (n) {
      if (t >= a.max_steps) {
        flag = 2;
        break;
      }
      if (n <= kFew) {
        if (warp == 0) few_steps(t, n);
        sync();
        if (!LARGE && misc[3]) break;
        t = misc[4];
        flag = misc[5];
        break;
      }
      int mark[4];
      if (n <= g.sparse_max) {
        move_listed<true>(n, t, mark);
        sync();
        if (!LARGE && misc[3]) break;
#pragma unroll
        for (int q = 0; q < 4; ++q)
          if (mark[q] >= 0) F[mark[q]] = 0;
        n = advance(t + 1, true);
      } else {
        const int nl = mark_dense(t);
        if (nl) {
          move_listed<false>(nl, t, mark);
          sync();
        }
        if (!LARGE && misc[3]) break;
        n = apply_dense(t);
        for (int w = tid; w < 2 * g.nws; w += NT) F[w] = 0;
        if (n) advance(t + 1, n <= g.sparse_max);
      }
      ++t;
    }
    if (!LARGE && misc[3]) {
      // the whole CTA leaves together (misc[3] was read behind a barrier); the
      // banded or generic sweep decodes the shot afterwards
      if (tid == 0) a.out_steps[shot] = kStepsPending;
      return;
    }
    // ---- correction, homology, steps, flag
    for (int y = tid; y < L; y += NT) wx ^= (int)(C[y << lws] & 1u);
    for (int j = tid; j <= lastw; j += NT) wy ^= __popc(C[g.nws + j]) & 1;
    wx = __reduce_xor_sync(kFull, wx);
    wy = __reduce_xor_sync(kFull, wy);
    if (NT > 32) {
      if (lane == 0 && wx) atomicXor(&misc[6], 1);
      if (lane == 0 && wy) atomicXor(&misc[7], 1);
      sync();
      wx = misc[6];
      wy = misc[7];
    }
    store_bits<NT>(outC, 2 * L, L, lws, C, tid);
    if (tid == 0) {
      a.out_steps[shot] = t;
      if (a.from_sigma) {
        a.out_cut[2 * shot] = (uint8_t)wx;
        a.out_cut[2 * shot + 1] = (uint8_t)wy;
        if (a.out_exhausted) a.out_exhausted[shot] = (uint8_t)(flag == 2);
      } else {
        a.out_flag[shot] = (uint8_t)(flag == 2 ? 2 : ((wx | wy) ? 1 : 0));
      }
    }
  }
};

}  // namespace hist
}  // namespace qca
