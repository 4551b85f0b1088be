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
//   listed  at most sparse_max anyons, one thread per anyon for slices 0 to 4
//           (a (6k + 7)^2 neighbourhood), a whole warp per anyon beyond them;
//   few     at most 8 anyons: one warp runs all remaining steps by itself, one
//           lane per (anyon, slice), from a ring of the last anyon sets.
// Flipped links are marked in a map, so that a link crossed from both ends
// flips once (the OR of Eq. ddfeedback).
#pragma once

#include <algorithm>
#include <type_traits>

#include "qca_internal.cuh"

namespace qca {
namespace hist {

constexpr int kFew = 8;        // most anyons of the few-anyon mode
constexpr int kFewRing = 128;  // steps of anyon sets it keeps (more than 85)
constexpr int kSteps = 128;    // steps whose place in the archive is known (more than 85)
// what the archive holds of a step, if not a list of so many anyons
constexpr uint16_t kNotKept = 0xFFFF, kBitmap = 0xFFFE;
constexpr int kLargeRing = 88; // syndromes kept per shot above L = 256 (more than 85)
constexpr uint32_t kFull = 0xffffffffu;

struct Geom {
  int L;
  int lws;         // log2 of the 32-bit words per bitmap row
  int nws;         // words of one site bitmap (L << lws)
  int nslot;       // words of a bitmap's place in shared memory (a multiple of 4)
  int kmask;       // syndromes kept in shared memory, less one (a power of two less one)
  int spill;       // whether syndromes older than those are needed at all
  int kthread;     // oldest slice a single thread can search: min(4, (L - 7) / 6)
  int c_global;    // the correction is kept in the correction block
  int f_global;    // and so are the dense steps' link maps
  int kmax;        // oldest slice a message can come from: (m_max - 1) / 3
  int sparse_max;  // most anyons of the listed mode
  int list_cap;    // entries of the anyon list
  // word offsets in the CTA's shared memory (L <= 256) or its global slot
  int o_C, o_F, o_list, o_table, o_few, o_snap, o_misc;  // (o_F: LARGE only)
  int tmask;       // entries of the crossing table, less one
};

// Words of the few-anyon mode's ring of anyon sets, and of each of the two
// snapshots of it (orbit detection); entries are 16 bits up to L = 256, 32 bits
// above.
template <bool LARGE>
constexpr int kFewWords = kFewRing * kFew / (LARGE ? 1 : 2);

// ---------------------------------------------------------------- host: geometry
// Threads per shot: a warp up to L = 64 (no block barriers).  Above, four warps:
// the steps with few anyons leave most of a larger CTA idle, so more and smaller
// CTAs per SM are better (L = 256: 256 threads 5.4 ms per 20 000 shots at three
// CTAs per SM, 128 threads at the same three 6.3 ms, at six 4.8 ms).  What lets
// six fit at L = 256 is keeping the correction and the dense steps' link maps in
// the shot's (L2-resident) correction block instead of shared memory.
inline int threads_for(int L) { return L <= 64 ? 32 : (L <= 256 ? 128 : 1024); }

// Whether a small batch of small lattices keeps all 85 syndromes in shared memory
// (128 slots, 21 KB at L = 32): the shots are all resident anyway, and the call
// then has no second launch for pending shots (64 shots of L = 16: 30.7 -> 26.7 us
// per call on the device).
constexpr int kAllSlotsL = 32, kAllSlotsShots = 1024;
inline bool all_slots(int L, int64_t shots) { return L <= kAllSlotsL && shots <= kAllSlotsShots; }

inline bool make_hist_geom(int L, int m_max, Geom& g, int& threads, size_t& smem,
                           size_t& slot_words, bool all = false) {
  if (L < 8 || L > QCA_MAX_L) return false;
  const bool large = L > 256;
  threads = threads_for(L);
  g.L = L;
  const int wpr = (L + 31) / 32;
  g.lws = 0;
  while ((1 << g.lws) < wpr) ++g.lws;
  g.nws = L << g.lws;
  g.nslot = (g.nws + 3) & ~3;
  g.kmax = (m_max - 1) / 3;
  g.kthread = std::min(4, (L - 7) / 6);
  const int K = all ? 128 : (L <= 128 ? 8 : 4);
  g.kmask = K - 1;
  // (up to L = 176 six CTAs per SM fit with the correction in shared memory too)
  g.c_global = !large && L > 176;
  g.f_global = !large && L > 128;
  // a listed step t gives up one slot, for sigma_{t+1}, and keeps slices 0 to K - 2;
  // a dense one whose link maps are in slots gives up two more
  g.spill = g.kmax > (g.f_global ? K - 2 : K - 4);
  // a dense pass costs about as much as searching half an anyon per word (L = 32,
  // p = 0.06: 0.80 ms per 20 000 shots, 0.87 at a quarter); above L = 128 the
  // smaller list and crossing table let one more CTA fit (L = 256: 4.8 against
  // 5.8 ms)
  g.sparse_max = std::max(kFew, L <= 128 ? g.nws / 2 : g.nws / 4);
  if (large) g.sparse_max = std::min(g.sparse_max, 4096);
  g.list_cap = g.sparse_max;
  int tsize = 1;
  while (tsize < g.sparse_max) tsize *= 2;
  g.tmask = tsize - 1;
  const int few = large ? kFewWords<true> : kFewWords<false>;
  // the crossing table and the few-anyon mode's sets are never in use at once
  int o = 0, region = std::max(few, tsize);
  if (large) {
    g.o_C = kLargeRing * g.nws;
    g.o_F = g.o_C + 2 * g.nws;
    slot_words = (size_t)g.o_F + 2 * g.nws;
  } else {
    o = K * g.nslot;
    g.o_list = o;
    // the snapshots are taken when the bitmaps and the list are no longer needed (a
    // place of their own let 19 instead of 24 CTAs fit at L = 48: 20 000 shots, p = 0.05,
    // 742 -> 641 us)
    g.o_snap = 0;
    o = std::max((o + g.list_cap + 3) & ~3, 2 * few);
    g.o_C = g.o_F = 0;
    if (!g.c_global) {
      g.o_C = o;
      o = (o + 2 * g.nws + 3) & ~3;
    }
    slot_words = 0;
  }
  g.o_table = g.o_few = o;
  o += (region + 3) & ~3;
  if (large) {
    g.o_snap = o;
    o += 2 * few;
    g.o_list = o;
    o += g.list_cap;
  }
  g.o_misc = o;
  smem = (size_t)(o + 8 + kSteps) * 4;  // counters; archived sets' sizes and places
  return true;
}

// Syndromes that have left shared memory, in the part of the shot's correction
// block (2 L^2 bytes, not written before the shot ends) that the correction and
// the link maps leave.  It is a ring of 4-byte words: a listed set is written to
// it as a list of 16-bit sites when it is made, one that was never listed as a
// bitmap (rows without padding) when it leaves its slot, each right after the one
// before, over whatever is oldest.  Lists take what they need: of L = 144, p = 0.08,
// whose sets have 5300, 2600, 1500, 850, 490, 310, 210, 170, 130, ... anyons, six
// bitmaps and all lists since fit (24 of the 32 KB).  With a place of fixed size for
// each of 86 lists, three quarters of such shots asked for a set that was gone.
// A word of the ring always holds the last thing written to it, and whatever a new
// entry covers is marked as not kept, so a search finds a set whole or not at all.
struct Archive {
  uint32_t* words;
  int size;  // words of the ring
  int head;  // next free word
  int next;  // syndromes that have left their slot
  bool round;  // the ring has been filled once: new entries cover old ones
  uint32_t listed;  // bit i: the (i + 1)-th last step was archived as a list
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

// The same without wrap: columns below 0 or from L on are 0 (0 - n < c < L).
__device__ __forceinline__ uint32_t row_bits_clipped(const uint32_t* row, int wpr, int L, int c,
                                                     int n) {
  const int s = max(c, 0), w = s >> 5;
  uint32_t v = 0;
  if (s < L) {
    v = __funnelshift_r(row[w], w + 1 < wpr ? row[w + 1] : 0u, s & 31);
    if (c < 0) v <<= -c;
  }
  return n >= 32 ? v : v & ((1u << n) - 1u);
}

// Any anyon within `reach` columns of x in a bitmap row; OPEN: a row that does
// not wrap.
template <bool OPEN>
__device__ __forceinline__ uint32_t row_any(const uint32_t* row, int wpr, int L, int x,
                                            int reach) {
  uint32_t any = 0;
  if (OPEN) {
    const int hi = min(x + reach, L - 1);
#pragma unroll 1
    for (int c = max(x - reach, 0); c <= hi; c += 32)
      any |= row_bits_clipped(row, wpr, L, c, min(32, hi - c + 1));
  } else if (2 * reach + 1 >= L) {
#pragma unroll 1
    for (int w = 0; w < wpr; ++w) any |= row[w];
  } else {
    int c = wrap_lo(x - reach, L);
#pragma unroll 1
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

// Slice k of the anyon at (x, y) by one thread, from the bitmap of sigma_{t-k}:
// the (6k + 7) x (6k + 7) neighbourhood, a row window per row; needs 6k + 7 <=
// 31 and <= L.  OPEN: rows and columns outside the lattice are empty.  ROWS: rows
// whose loads are in flight together (1 in shared memory, where short code is
// worth more; 6 in global memory, whose latency it would otherwise pay per row).
template <bool OPEN, int ROWS>
__device__ __forceinline__ uint32_t slice_thread(const uint32_t* sig, int lws, int L, int x, int y,
                                                 int k) {
  const int wpr = 1 << lws;
  const int r = 3 * k + 3, n = 2 * r + 1;
  const int s = OPEN ? max(x - r, 0) : wrap_lo(x - r, L);
  const int w0 = s >> 5, sh = s & 31;
  const int w1 = min(w0 + 1, wpr - 1);
  const int sl = w0 < wpr - 1 ? 32 - sh : 32;  // 1 .. 32
  // columns before the wrap, if any; OPEN: columns left of the lattice
  const int n0 = OPEN ? s - (x - r) : (s + n > L ? L - s : 0);
  const uint32_t mask = (1u << n) - 1u;
  int yy = OPEN ? y - r : wrap_lo(y - r, L);
  auto next = [&]() {  // bit i: column x - r + i of the next row
    if (OPEN && (unsigned)yy >= (unsigned)L) {
      ++yy;
      return 0u;
    }
    const uint32_t* row = sig + (yy << lws);
    uint32_t v = (row[w0] >> sh) | __funnelshift_lc(0u, row[w1], sl);
    if (OPEN)
      v <<= n0;
    else if (n0)
      v |= row[0] << n0;  // the bits past column L - 1 are 0
    ++yy;
    if (!OPEN && yy == L) yy = 0;
    return v & mask;
  };
  // rows y - r .. y + r; the distances' cone sections across the rows are
  // |j| <= 3k + 1, 3k + 2, 3k + 3
  const uint32_t u3 = next(), u2 = next(), u1 = next();
  uint32_t v1 = u1;
  int i = n - 6;  // 1 + 6k
  if (ROWS > 1) {
#pragma unroll 1
    for (; i >= ROWS; i -= ROWS) {
      uint32_t v[ROWS];
#pragma unroll
      for (int q = 0; q < ROWS; ++q) v[q] = next();
#pragma unroll
      for (int q = 0; q < ROWS; ++q) v1 |= v[q];
    }
  }
#pragma unroll 1
  for (; i > 0; --i) v1 |= next();
  const uint32_t d1 = next(), d2 = next(), d3 = next();
  v1 |= d1;
  const uint32_t v2 = v1 | u2 | d2, v3 = v2 | u3 | d3;
  // +x comes from column x - d, -x from x + d, +y from row y - d, -y from y + d
  uint32_t m = ((v1 >> 2) & 1u) | (((v1 >> (n - 3)) & 1u) << 1);
  m |= ((v2 << 3) & 0x10u) | (((v2 >> (n - 2)) & 1u) << 5);
  m |= ((v3 << 8) & 0x100u) | ((v3 >> (n - 1)) << 9);
  const uint32_t m1 = (mask >> 4) << 2, m2 = (mask >> 2) << 1;
  if (u1 & m1) m |= 0x4u;
  if (d1 & m1) m |= 0x8u;
  if (u2 & m2) m |= 0x40u;
  if (d2 & m2) m |= 0x80u;
  if (u3) m |= 0x400u;
  if (d3) m |= 0x800u;
  return m;
}

// Any slice of the anyon at (x, y) by a whole warp, from a bitmap of wpr words per
// row: a lane per row for the x
// fields (three columns on either side), six lanes for the y fields' rows.  For
// the far slices, which few anyons reach: a function of its own, since the
// kernel is bound by instruction fetch when every use is a copy.
template <bool OPEN>
static __device__ __noinline__ uint32_t slice_warp(const uint32_t* sig, int wpr, int L, int x, int y,
                                               int k, int lane) {
  const int r = 3 * k + 3;
  const int nrows = OPEN ? 2 * r + 1 : min(2 * r + 1, L);
  const int half = nrows == 2 * r + 1 ? r : (L - 1) >> 1;
  const int cl = OPEN ? x - r : wrap_lo(x - r % L, L);                  // columns x - 3k - 3 ..
  const int cr = OPEN ? x + r - 2 : wrap_hi(x + (3 * k + 1) % L, L);    // columns x + 3k + 1 ..
  uint32_t m = 0;
#pragma unroll 1
  for (int i = lane; i < nrows; i += 32) {
    const int j = i - half;
    if (OPEN && (unsigned)(y + j) >= (unsigned)L) continue;
    const uint32_t* row = sig + wrap_hi(wrap_lo(y + j, L), L) * wpr;
    // d = 3, 2, 1 and d = 1, 2, 3
    const uint32_t l = OPEN ? (cl > -3 ? row_bits_clipped(row, wpr, L, cl, 3) : 0u)
                            : row_bits_wrapped(row, wpr, L, cl, 3);
    const uint32_t q = OPEN ? row_bits_clipped(row, wpr, L, cr, 3)
                            : row_bits_wrapped(row, wpr, L, cr, 3);
    uint32_t h = ((l >> 2) & 1u) | ((q << 1) & 2u) | ((l << 3) & 0x10u) | ((q << 4) & 0x20u) |
                 ((l << 8) & 0x100u) | ((q << 7) & 0x200u);
    const int aj = (j < 0 ? -j : j) - 3 * k;  // |j| <= 3k + d
    if (aj > 1) h &= aj > 2 ? 0xF00u : 0xFF0u;
    m |= h;
  }
  if (lane < 6) {
    const int d = lane < 3 ? lane + 1 : lane - 2;
    const int reach = 3 * k + d, dr = OPEN ? reach : reach % L;
    int yy = lane < 3 ? y - dr : y + dr;
    if (!OPEN) yy = wrap_hi(wrap_lo(yy, L), L);
    if (!OPEN || (unsigned)yy < (unsigned)L)
      m |= row_any<OPEN>(sig + yy * wpr, wpr, L, x, reach) << (4 * (d - 1) + (lane < 3 ? 2 : 3));
  }
  return __reduce_or_sync(kFull, m);
}

// Slice k of the anyon at (xa, ya) against one anyon (xb, yb) of sigma_{t-k}, for
// slices within half the torus (3k + 3 <= (L - 1) / 2; OPEN: any slice): the
// larger of the two coordinate distances decides.
template <bool OPEN>
__device__ __forceinline__ uint32_t slice_near(int xa, int ya, int xb, int yb, int L, int k) {
  const int half = L >> 1;
  int sx = xa - xb, sy = ya - yb;
  if (!OPEN) {
    if (sx > half) sx -= L;
    if (sx < -half) sx += L;
    if (sy > half) sy -= L;
    if (sy < -half) sy += L;
  }
  const int ax = abs(sx), ay = abs(sy), d = max(ax, ay), e = d - 3 * k - 1;
  if ((unsigned)e >= 3u) return 0;
  return ((ax == d ? (sx > 0 ? 1u : 2u) : 0u) | (ay == d ? (sy > 0 ? 4u : 8u) : 0u)) << (4 * e);
}
// The same for any slice; c = (3k + 1) mod L.
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

// The same against all n anyons of an archived set, by a whole warp.
template <bool OPEN>
static __device__ __noinline__ uint32_t slice_list(const uint16_t* set, int n, int L, int x, int y,
                                                   int k, int lane) {
  const int c = (3 * k + 1) % L;
  uint32_t m = 0;
#pragma unroll 1
  for (int i = lane; i < n; i += 32) {
    const uint32_t e = set[i];
    m |= OPEN ? slice_near<true>(x, y, (int)(e & 0xFFu), (int)(e >> 8), L, k)
              : slice_pair(x, y, (int)(e & 0xFFu), (int)(e >> 8), L, k, c);
  }
  return __reduce_or_sync(kFull, m);
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

// The counter draws, out of line: options that most calls leave off.
static __device__ __noinline__ uint64_t key_of(uint64_t key, int64_t shot, int t) {
  return move_step_key(key, shot, t);
}
// Random move of the anyon at site r, or 0.
static __device__ __noinline__ int draw_move(uint64_t key, uint64_t thr, uint32_t r) {
  const uint64_t u = splitmix64(key ^ (uint64_t)r);
  return u < thr ? 1 + (int)(splitmix64(u) >> 62) : 0;
}
static __device__ __noinline__ int draw_balance(int code, uint64_t key, uint32_t r) {
  return balance_resolve(code, key, r);
}

// 16 bytes -> 16 bits: bit 0 of each byte, or (any) whether it is not 0.
__device__ __forceinline__ uint32_t pack4(uint32_t w) { return (w * 0x01020408u) >> 24; }
__device__ __forceinline__ uint32_t nonzero4(uint32_t w) {
  return ((((w & 0x7F7F7F7Fu) + 0x7F7F7F7Fu) | w) & 0x80808080u) >> 7;
}
__device__ __forceinline__ uint32_t pack16(uint4 v, bool any) {
  if (any) v = make_uint4(nonzero4(v.x), nonzero4(v.y), nonzero4(v.z), nonzero4(v.w));
  return pack4(v.x) | (pack4(v.y) << 4) | (pack4(v.z) << 8) | (pack4(v.w) << 12);
}
// 4 bits -> 4 bytes of 0 / 1.
__device__ __forceinline__ uint32_t unpack4(uint32_t nib) {
  return (nib * 0x00204081u) & 0x01010101u;
}
__device__ __forceinline__ uint4 unpack16(uint32_t b) {
  return make_uint4(unpack4(b & 15u), unpack4((b >> 4) & 15u), unpack4((b >> 8) & 15u),
                    unpack4((b >> 12) & 15u));
}

// rows x L bytes at src -> bitmap rows (2^lws words each), any size and
// alignment: 16-byte groups of the flat block (single bytes at its two ends),
// whose bits go to the two or three rows they belong to.  dst is zeroed before.
static __device__ __noinline__ void load_flat(const uint8_t* src, int rows, int L, int lws,
                                              uint32_t* dst, bool any, int tid, int nt) {
  const int total = rows * L;
  const int skew = (int)(reinterpret_cast<uintptr_t>(src) & 15);
#pragma unroll 2
  for (int i = tid; 16 * i < total + skew; i += nt) {
    int f = 16 * i - skew;
    uint32_t b = 0;
    if (f >= 0 && f + 16 <= total) {
      b = pack16(*reinterpret_cast<const uint4*>(src + f), any);
    } else {
#pragma unroll 1
      for (int q = 0; q < 16; ++q)
        if (f + q >= 0 && f + q < total && (any ? src[f + q] != 0 : src[f + q] & 1)) b |= 1u << q;
      if (f < 0) {
        b >>= -f;
        f = 0;
      }
    }
    int r = f / L, x = f - r * L;
    while (b) {
      const uint32_t v = L - x < 16 ? b & ((1u << (L - x)) - 1u) : b;
      uint32_t* row = dst + (r << lws);
      const int sh = x & 31;
      if (v << sh) atomicOr(&row[x >> 5], v << sh);
      if (sh > 16 && v >> (32 - sh)) atomicOr(&row[(x >> 5) + 1], v >> (32 - sh));
      b = L - x < 16 ? b >> (L - x) : 0;
      x = 0;
      ++r;
    }
  }
}

// Bitmap rows -> rows x L bytes of 0 / 1 at out, any size and alignment.
static __device__ __noinline__ void store_flat(uint8_t* out, int rows, int L, int lws,
                                               const uint32_t* src, int tid, int nt) {
  const int total = rows * L, wpr = 1 << lws;
  const int skew = (int)(reinterpret_cast<uintptr_t>(out) & 15);
#pragma unroll 1
  for (int i = tid; 16 * i < total + skew; i += nt) {
    const int f0 = 16 * i - skew, f = max(f0, 0);
    int r = f / L, x = f - r * L;
    uint32_t b = 0;
    for (int have = f - f0; have < 16 && r < rows; ++r) {
      const uint32_t* row = src + (r << lws);
      const int w = x >> 5;
      uint32_t v = __funnelshift_r(row[w], w + 1 < wpr ? row[w + 1] : 0u, x & 31);
      if (L - x < 16) v &= (1u << (L - x)) - 1u;
      b |= (v & 0xFFFFu) << have;
      have += L - x;
      x = 0;
    }
    if (f0 >= 0 && f0 + 16 <= total) {
      __stcs(reinterpret_cast<uint4*>(out + f0), unpack16(b));
    } else {
#pragma unroll 1
      for (int q = 0; q < 16; ++q)
        if (f0 + q >= 0 && f0 + q < total) out[f0 + q] = (uint8_t)((b >> q) & 1u);
    }
  }
}

// The same for rows of whole 16-byte groups on a 16-byte boundary: a warp
// moves 512 contiguous bytes at a time.
template <int NT>
__device__ __forceinline__ void load_rows(const uint8_t* src, int rows, int L, int lws,
                                          uint32_t* dst, bool any, int tid) {
  const int vpr = L >> 4, n = rows * vpr;
  const uint4* s16 = reinterpret_cast<const uint4*>(src);
  uint16_t* d16 = reinterpret_cast<uint16_t*>(dst);
  const int dr = NT / vpr, dc = NT - dr * vpr;
  int r = tid / vpr, c = tid - r * vpr;
#pragma unroll 4
  for (int i = tid; i < n; i += NT) {
    d16[(r << (lws + 1)) + c] = (uint16_t)pack16(__ldcs(s16 + i), any);
    r += dr;
    c += dc;
    if (c >= vpr) {
      c -= vpr;
      ++r;
    }
  }
}
template <int NT>
__device__ __forceinline__ void store_rows(uint8_t* out, int rows, int L, int lws,
                                           const uint32_t* src, int tid) {
  const int vpr = L >> 4, n = rows * vpr;
  uint4* o16 = reinterpret_cast<uint4*>(out);
  const uint16_t* s16 = reinterpret_cast<const uint16_t*>(src);
  const int dr = NT / vpr, dc = NT - dr * vpr;
  int r = tid / vpr, c = tid - r * vpr;
#pragma unroll 2
  for (int i = tid; i < n; i += NT) {
    __stcs(o16 + i, unpack16(s16[(r << (lws + 1)) + c]));
    r += dr;
    c += dc;
    if (c >= vpr) {
      c -= vpr;
      ++r;
    }
  }
}

// Whether the kmax + 1 anyon sets up to step t equal those up to step t_snap
// of the snapshot; `words` 32-bit words per set.  By one warp.
static __device__ __noinline__ bool sets_repeat(const uint32_t* now, const uint32_t* snap, int t,
                                                int t_snap, int kmax, int words, int lane) {
  bool same = true;
#pragma unroll 1
  for (int i = lane; i <= kmax && same; i += 32) {
    const uint32_t* p = now + ((t - i) & (kFewRing - 1)) * words;
    const uint32_t* q = snap + ((t_snap - i) & (kFewRing - 1)) * words;
#pragma unroll 1
    for (int b = 0; b < words; ++b) same = same && p[b] == q[b];
  }
  return __all_sync(kFull, same);
}

// First step from t on whose outcome is that of step max_steps of an orbit of
// period P (the correction repeats with period 2P).
static __device__ __noinline__ int orbit_stop(int t, int P, int max_steps) {
  const int R = max_steps - t, per = R / P;
  return t + (R - per * P) + ((per & 1) ? P : 0);
}

// PLAIN: lexicographic ties, a balanced axis stays, no random moves (the
// default rules); the other forms read the rules from the arguments.
// OPEN (with PLAIN only): the lattice with open boundaries (Def. "message passing
// automaton with open boundaries"): no wrap; the columns x = 0 and x = L - 1 hold
// no anyons and no messages, send m^{+x} and m^{-x} into the bulk in every
// sub-step and absorb anyons; only the links between bulk sites and those to the
// two columns exist.
template <int NT, bool LARGE, bool PLAIN, bool OPEN = false>
struct Decoder {
  using Ent = typename std::conditional<LARGE, uint32_t, uint16_t>::type;
  // crossing table: bits of a link (word of the link maps and bit), steps it
  // tells apart
  static constexpr int kIdBits = LARGE ? 21 : 17;
  static constexpr int kEpochs = LARGE ? 1023 : 16383;
  static constexpr int kRowsAhead = LARGE ? 4 : 2;  // rows of a strip in flight

  const DecodeArgs& a;
  const Geom& g;
  uint32_t* ring;    // [kmask + 1][nws] (LARGE: [kLargeRing][nws])
  uint32_t* C;       // [2][nws] correction
  uint32_t* F;       // LARGE or f_global: [2][nws] links flipped in a dense step
  uint32_t* list;    // [list_cap] anyons (y << 16 | x)
  uint32_t* table;   // [tmask + 1] links crossed toward an anyon in a listed step
  Ent* few;          // [kFewRing][kFew]
  uint32_t* snap;    // [2][kFewWords] snapshots of it
  int* misc;         // 0-2 rotating counters, 3 miss, 4 steps, 5 flag, 6-7 cuts
  uint16_t* nset;    // [kSteps] anyons in the archived list of a step, kBitmap or kNotKept
  uint16_t* place;   // [kSteps] and its first word in the ring
                     // (entry i of both is written by thread i mod NT alone)
  Archive ar;
  int64_t shot;
  int tid, lane, warp;
  int ph;            // rotating counter in use
  int tb;            // step of the newest bitmap

  __device__ __forceinline__ bool literal() const {
    return !PLAIN && a.tie_order == QCA_TIE_LITERAL;
  }
  __device__ __forceinline__ bool moves_random() const { return !PLAIN && a.move_thr != 0; }
  __device__ __forceinline__ bool balance_random() const { return !PLAIN && a.balance_rule != 0; }

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
    return ring + (s & g.kmask) * g.nslot;
  }
  // oldest syndrome whose bitmap is in its slot
  __device__ __forceinline__ int oldest() const { return LARGE ? 0 : ar.next; }
  // x- / y-link map of dense step t: their own place, or the two slots with the
  // oldest syndromes
  __device__ __forceinline__ bool maps_in_slots() const { return !LARGE && !g.f_global; }
  __device__ __forceinline__ uint32_t* map_x(int t) const {
    return maps_in_slots() ? slot(t + 2) : F;
  }
  __device__ __forceinline__ uint32_t* map_y(int t) const {
    return maps_in_slots() ? slot(t + 3) : F + g.nws;
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
  // Barrier with the OR of p over the CTA.
  __device__ __forceinline__ bool sync_or(bool p) const {
    if (NT == 32) {
      const bool any = __any_sync(kFull, p);
      __syncwarp();
      return any;
    }
    return __syncthreads_or(p);
  }
  // Sum of n over the CTA; ends with a barrier.
  __device__ __forceinline__ int total(int n) {
    n = __reduce_add_sync(kFull, n);
    if (NT == 32) {
      __syncwarp();
      return n;
    }
    if (lane == 0 && n) atomicAdd(&misc[ph], n);
    return next_counter();
  }
  // Place of this thread's n entries in a list of all threads' entries.
  __device__ __forceinline__ int places(int n) {
    int incl = n;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int v = __shfl_up_sync(kFull, incl, o);
      if (lane >= o) incl += v;
    }
    int base = 0;
    if (lane == 31 && incl) base = atomicAdd(&misc[ph], incl);
    return __shfl_sync(kFull, base, 31) + incl - n;
  }

  // Words of an archived bitmap, and of the ring's entry i.
  __device__ __forceinline__ int bitmap_words() const { return g.L * ((g.L + 31) >> 5); }
  __device__ __forceinline__ int entry_words(int i) const {
    return nset[i] == kBitmap ? bitmap_words() : (nset[i] + 1) >> 1;
  }
  // First word of a new entry of at most n words (the ring has more); marks the
  // entries that it covers.
  __device__ __forceinline__ int reserve(int n) {
    const bool back = ar.head + n > ar.size;
    const int at = back ? 0 : ar.head;
    ar.round |= back;
#pragma unroll 1
    for (int i = ar.round ? tid : kSteps; i < kSteps; i += NT)
      if (nset[i] != kNotKept && place[i] < at + n && place[i] + entry_words(i) > at)
        nset[i] = kNotKept;
    return at;
  }
  // (by every thread: the one that owns the entry writes it)
  __device__ __forceinline__ void record(int s, uint16_t what, int at) {
    if (tid != (s & (kSteps - 1)) % NT) return;
    nset[s & (kSteps - 1)] = what;
    place[s & (kSteps - 1)] = (uint16_t)at;
  }

  // Makes sigma_s (in its slot), of at most n anyons, the newest bitmap, and moves
  // the syndrome in the slot of s + 1 to the archive, in a dense step perhaps also
  // those in the slots of s + 2 and s + 3, which become the link maps.  listed:
  // copies sigma_s to the slot of s + 1, where the moves will flip bits, and lists
  // the anyons; returns their number.  Ends with a barrier.
  __device__ __forceinline__ int advance(int s, bool listed, int n) {
    const uint4* cur = reinterpret_cast<const uint4*>(slot(s));
    uint4* nxt = reinterpret_cast<uint4*>(slot(s + 1));
    const int n4 = g.nslot >> 2;
    if (!LARGE) {
      const int end = (listed || !maps_in_slots() ? s + 1 : s + 3) - g.kmask;
      bool any = false;
#pragma unroll 1
      for (; ar.next < end; ++ar.next) {
        const int old = ar.next;
        if (!g.spill || (ar.listed >> (s - 1 - old)) & 1u) continue;
        const int at = reserve(bitmap_words());
        uint32_t* to = ar.words + at;
        const uint32_t* from = slot(old);
        const int wpr = (g.L + 31) >> 5, wsm = (1 << g.lws) - 1;
#pragma unroll 2
        for (int w = tid; w < g.nws; w += NT)
          if ((w & wsm) < wpr) to[(w >> g.lws) * wpr + (w & wsm)] = from[w];
        record(old, kBitmap, at);
        ar.head = at + bitmap_words();
        any = true;
      }
      if (any) sync();
    }
    tb = s;
    // a list where it is no longer than the bitmap
    const bool keep = !LARGE && listed && g.spill && n <= 2 * bitmap_words();
    if (!LARGE) ar.listed = ar.listed << 1 | (keep ? 1u : 0u);
    if (!listed) {
      if (!LARGE) record(s, kNotKept, 0);
      sync();
      return 0;
    }
    const int at = keep ? reserve((n + 1) >> 1) : 0;
    n = 0;
    uint32_t some = 0;  // which of this thread's groups hold anyons (at most 32 of them)
#pragma unroll 4
    for (int i = tid, q = 0; i < n4; i += NT, ++q) {
      const uint4 v = cur[i];
      nxt[i] = v;
      if (v.x | v.y | v.z | v.w) some |= 1u << q;
      n += __popc(v.x) + __popc(v.y) + __popc(v.z) + __popc(v.w);
    }
    int pos = places(n);
    if (n) {
      uint16_t* set = reinterpret_cast<uint16_t*>(ar.words + at);
      const int wsm = (1 << g.lws) - 1;
#pragma unroll 1
      for (; some; some &= some - 1) {
        const int i = tid + (__ffs(some) - 1) * NT;
        const uint4 v = cur[i];
        const uint32_t q4[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          uint32_t b = q4[q];
          const int w = 4 * i + q;
          const uint32_t yx = ((uint32_t)(w >> g.lws) << 16) | ((w & wsm) << 5);
          while (b) {
            const uint32_t e = yx + __ffs(b) - 1;
            b &= b - 1;
            list[pos] = e;
            if (keep) set[pos] = (uint16_t)((e >> 8) | (e & 0xFFu));
            ++pos;
          }
        }
      }
    }
    const int all = next_counter();
    if (!LARGE) {
      // (read from the next step on)
      record(s, keep ? (uint16_t)all : kNotKept, at);
      if (keep) ar.head = at + ((all + 1) >> 1);
    }
    return all;
  }

  __device__ __forceinline__ uint32_t site(int x, int y) const { return (uint32_t)(y * g.L + x); }

  // OPEN: hits of slice k from the two rough columns.
  __device__ __forceinline__ uint32_t edges(int x, int k) const {
    if (!OPEN) return 0u;
    const int l = x - 3 * k - 1, r = g.L - 2 - x - 3 * k;
    return ((unsigned)l < 3u ? 1u << (4 * l) : 0u) | ((unsigned)r < 3u ? 2u << (4 * r) : 0u);
  }
  // OPEN: whether column x can hold anyons.
  __device__ __forceinline__ bool bulk(int x) const {
    return !OPEN || (x > 0 && x < g.L - 1);
  }

  // One slice of the anyon at (x, y) by the whole warp, wherever the syndrome is.
  __device__ __forceinline__ uint32_t far_slice(int x, int y, int t, int k) const {
    const int s = t - k;
    const uint32_t* sig = nullptr;
    int wpr = 1 << g.lws;
    uint32_t m = 0;
    if (LARGE || s >= oldest()) {
      sig = slot(s);
    } else {
      const int n = nset[s & (kSteps - 1)];
      const uint32_t* at = ar.words + place[s & (kSteps - 1)];
      if (n == kNotKept) {
        misc[3] = 1;
      } else if (n == kBitmap) {
        sig = at;
        wpr = (g.L + 31) >> 5;
      } else {
        m = slice_list<OPEN>(reinterpret_cast<const uint16_t*>(at), n, g.L, x, y, k, lane);
      }
    }
    if (sig) m = slice_warp<OPEN>(sig, wpr, g.L, x, y, k, lane);
    return (m | edges(x, k)) & slice_limit(a.m_max, k);
  }
  // Slices from k on by the whole warp; returns the first slice's hits (0:
  // nothing heard) and its index in k.
  __device__ __forceinline__ uint32_t search_far(int x, int y, int t, int& k) const {
    const int last = min(t, g.kmax);
    uint32_t m = 0;
#pragma unroll 1
    for (; k <= last; ++k) {
      m = far_slice(x, y, t, k);
      // (other warps set the flag at any time: one vote, so that the warp stays together)
      if (m || (!LARGE && __any_sync(kFull, *(volatile int*)&misc[3]))) break;
    }
    return m;
  }

  __device__ __forceinline__ uint64_t move_key_of(int t) const {
    return moves_random() ? key_of(a.move_key, a.shot_offset + shot, t) : 0;
  }
  // A balanced axis (5 x, 6 y) of the anyon at (x, y) at step t, resolved.
  __device__ __forceinline__ int balanced(int code, int x, int y, int t) const {
    if (!balance_random()) return 0;
    return draw_balance(code, key_of(a.balance_key, a.shot_offset + shot, t), site(x, y));
  }
  // The move of the anyon at (x, y) that hears h0 (and h1 at the next distance).
  __device__ __forceinline__ int move_of(uint64_t move_key, int x, int y, int t, uint32_t h0,
                                         uint32_t h1) const {
    int dir = h0 ? direction(h0, h1, PLAIN ? QCA_TIE_LEX : a.tie_order) : 0;
    if (moves_random()) {
      const int d = draw_move(move_key, a.move_thr, site(x, y));
      if (d) return d;
    }
    if (dir >= 5) dir = balanced(dir, x, y, t);
    return dir;
  }
  // Hits at the smallest distance of a slice's hits, and at the next one (0
  // past the slice's third distance).
  __device__ __forceinline__ void nearest(uint32_t m, uint32_t& h0, uint32_t& h1) const {
    const int d4 = (__ffs(m) - 1) & ~3;
    h0 = (m >> d4) & 15u;
    h1 = (m >> (d4 + 4)) & 15u;
  }

  // Lower end of the link an anyon at (x, y) crosses when it moves: word of the
  // link maps and bit.
  __device__ __forceinline__ int link_of(int x, int y, int dir, uint32_t& bit) const {
    const int lx = dir == 2 ? wrap_lo(x - 1, g.L) : x;
    const int ly = dir == 4 ? wrap_lo(y - 1, g.L) : y;
    bit = 1u << (lx & 31);
    return (dir >= 3 ? g.nws : 0) + (ly << g.lws) + (lx >> 5);
  }
  __device__ __forceinline__ uint32_t site_after(int x, int y, int dir) const {
    if (dir == 1) x = wrap_hi(x + 1, g.L);
    if (dir == 2) x = wrap_lo(x - 1, g.L);
    if (dir == 3) y = wrap_hi(y + 1, g.L);
    if (dir == 4) y = wrap_lo(y - 1, g.L);
    return ((uint32_t)y << 16) | x;
  }

  // Whether this is the first crossing of a link (id) in step t: the anyons that
  // cross it toward one another both ask.  Entries carry the step, so the table
  // is cleared only once in kEpochs + 1 steps.
  __device__ __forceinline__ bool first_crossing(uint32_t id, int t) const {
    const uint32_t key = ((uint32_t)(t & kEpochs) + 1u) << kIdBits | id;
    uint32_t h = (id * 0x9E3779B1u) >> 16;
#pragma unroll 1
    for (;; ++h) {
      uint32_t* e = &table[h & g.tmask];
      uint32_t old = *(volatile uint32_t*)e;
      while ((old >> kIdBits) != (key >> kIdBits)) {  // free in this step
        const uint32_t was = atomicCAS(e, old, key);
        if (was == old) return true;
        old = was;
      }
      if (old == key) return false;
    }
  }

  // Decides and marks the moves of the n listed anyons at step t, a thread per
  // anyon.  listed: the correction and the copy of sigma in the next slot are
  // flipped at once; else (dense step) only the link map is marked.  Returns
  // whether this thread's anyons moved.
  __device__ __forceinline__ bool move_listed(int n, int t, bool listed) {
    bool moved = false;
    const uint32_t* sig = slot(t);
    uint32_t* sn = slot(t + 1);
    const uint64_t key = move_key_of(t);
    const int last = min(t, g.kmax);
    const int lastt = min(min(last, g.kthread), t - oldest());
#pragma unroll 1
    for (int i0 = 0; i0 < n; i0 += NT) {
      // a warp searches its far anyons one after the other: few anyons are spread
      // over the warps (L = 256, p = 0.08: 6.8 -> 5.6 ms per 2000 shots), many are
      // packed, so that fewer warps run the near slices (L = 256, p = 0.05: 4.9 ->
      // 4.8 ms per 20 000 shots)
      const bool spread = LARGE || n <= NT / 2;
      const int i = i0 + (spread ? lane * (NT / 32) + warp : tid);
      if (i0 + (spread ? warp : tid - lane) >= n) break;
      const bool act = i < n;
      int x = 0, y = 0, k = 0;
      uint32_t m = 0;
      if (act) {
        const uint32_t e = list[i];
        x = e & 0xFFFFu;
        y = e >> 16;
#pragma unroll 1
        for (;; ++k) {
          m = slice_thread<OPEN, LARGE ? 6 : 1>(slot(t - k), g.lws, g.L, x, y, k) | edges(x, k);
          m &= slice_limit(a.m_max, k);
          if (m || k >= lastt) break;
        }
      }
      uint32_t todo = __ballot_sync(kFull, act && m == 0 && lastt < last);
#pragma unroll 1
      while (todo) {
        const int src = __ffs(todo) - 1;
        todo &= todo - 1;
        int kk = lastt + 1;
        const uint32_t mm = search_far(__shfl_sync(kFull, x, src), __shfl_sync(kFull, y, src), t,
                                       kk);
        if (lane == src) {
          m = mm;
          k = kk;
        }
      }
      uint32_t h0 = 0, h1 = 0;
      if (m) nearest(m, h0, h1);
      if (literal()) {
        // the next distance may be the first one of the next slice
        todo = __ballot_sync(kFull, h0 && !(m & 0xFFu) && !(h0 & 10u) && k < last);
#pragma unroll 1
        while (todo) {
          const int src = __ffs(todo) - 1;
          todo &= todo - 1;
          const uint32_t mm = far_slice(__shfl_sync(kFull, x, src), __shfl_sync(kFull, y, src), t,
                                        __shfl_sync(kFull, k, src) + 1);
          if (lane == src) h1 = mm & 15u;
        }
      }
      const int dir = act ? move_of(key, x, y, t, h0, h1) : 0;
      if (dir) {
        moved = true;
        uint32_t bit;
        const int w = link_of(x, y, dir, bit);
        if (!listed) {
          atomicOr(w < g.nws ? map_x(t) + w : map_y(t) + (w - g.nws), bit);
        } else {
          const uint32_t to = site_after(x, y, dir);
          const int nx = to & 0xFFFFu, ny = to >> 16;
          const int wn = (ny << g.lws) + (nx >> 5);
          // two anyons that swap sites cross one link, which flips once
          if (!((sig[wn] >> (nx & 31)) & 1u) ||
              first_crossing((uint32_t)w << 5 | (__ffs(bit) - 1), t)) {
            atomicXor(&C[w], bit);
            atomicXor(&sn[(y << g.lws) + (x >> 5)], 1u << (x & 31));
            if (bulk(nx)) atomicXor(&sn[wn], 1u << (nx & 31));
          }
        }
      }
    }
    return moved;
  }

  // Dense steps go through the bitmaps in strips of rows: lane group of 2^lws
  // lanes = the words of a row, each group a strip of consecutive rows, so that
  // a row is read once and its neighbours in the row come by shuffles.
  struct Strip {
    int j;              // word of the row
    int jl, jr;         // lanes of the words to the left and to the right
    int sl, top;        // bit of the left word that is column x - 1 of this word's first
                        // column, bit of this word that is its last column
    uint32_t valid;     // this word's columns that can hold anyons
    bool on;            // not a padding word
    int y0, y1;         // rows
  };
  __device__ __forceinline__ Strip strip() const {
    const int lws = g.lws, wpr = 1 << lws, lastw = (g.L - 1) >> 5, lastb = (g.L - 1) & 31;
    const int H = (g.L + (NT >> lws) - 1) / (NT >> lws);
    Strip p;
    p.j = lane & (wpr - 1);
    const int base = lane - p.j;
    p.jl = base + (p.j == 0 ? lastw : p.j - 1);
    p.jr = base + (p.j >= lastw ? 0 : p.j + 1);
    p.sl = p.j == 0 ? lastb : 31;
    p.top = p.j == lastw ? lastb : 31;
    p.valid = p.j < lastw ? kFull : (p.j == lastw ? kFull >> (31 - lastb) : 0u);
    if (OPEN && p.j == 0) p.valid &= ~1u;
    if (OPEN && p.j == lastw) p.valid &= ~(1u << lastb);
    p.on = p.j <= lastw;
    p.y0 = min((tid >> lws) * H, g.L);
    p.y1 = min(p.y0 + H, g.L);
    return p;
  }
  __device__ __forceinline__ int strip_rows() const {
    return (g.L + (NT >> g.lws) - 1) / (NT >> g.lws);
  }
  // v shifted by one column: bit x = column x - 1 / x + 1 of the row
  __device__ __forceinline__ uint32_t from_left(uint32_t v, const Strip& p) const {
    return (v << 1) | ((__shfl_sync(kFull, v, p.jl) >> p.sl) & 1u);
  }
  __device__ __forceinline__ uint32_t from_right(uint32_t v, const Strip& p) const {
    return (v >> 1) | ((__shfl_sync(kFull, v, p.jr) & 1u) << p.top);
  }

  // Dense step t: distance 1 of every anyon, 32 sites per word.  Writes the link
  // map, and the undecided anyons as a bitmap to the next slot; returns this
  // thread's number of them.
  __device__ __forceinline__ int mark_dense(int t, const Strip& p) {
    const uint32_t* sig = slot(t) + p.j;
    uint32_t* open = slot(t + 1) + p.j;
    uint32_t *fxp = map_x(t) + p.j, *fyp = map_y(t) + p.j;
    const int L = g.L, lws = g.lws, H = strip_rows();
    const bool on = p.on && p.y0 < L;
    const uint64_t key = move_key_of(t);
    int n = 0, y = p.y0;
    auto row = [&](int r) {
      if (OPEN && (unsigned)r >= (unsigned)L) return 0u;
      return on ? sig[wrap_hi(wrap_lo(r, L), L) << lws] : 0u;
    };
    // OPEN: bits of the columns next to the rough ones (which hold no anyons, so
    // the shifts need no clipping)
    const uint32_t first = OPEN && p.j == 0 ? 2u : 0u;
    const uint32_t last = OPEN && (L - 2) >> 5 == p.j ? 1u << ((L - 2) & 31) : 0u;
    // rows y - 1 (u), y (c), y + 1 (d), each with its shifted copies
    uint32_t u = row(y - 1), c = row(y);
    uint32_t ul = from_left(u, p), ur = from_right(u, p);
    uint32_t cl = from_left(c, p), cr = from_right(c, p);
    uint32_t up = 0;  // +y moves of the row before
    uint32_t ahead = row(y + 1);
    // one row more than the strip has: its -y moves cross the last row's links
#pragma unroll 1
    for (int i = 0; i <= H; ++i, ++y) {
      const uint32_t d = ahead;
      if (i < H) ahead = row(y + 2);  // (loaded a row early)
      const uint32_t dl = from_left(d, p), dr = from_right(d, p);
      const uint32_t px = ul | cl | dl | first;  // anyon in column x - 1
      const uint32_t mx = ur | cr | dr | last;   // in column x + 1
      const uint32_t py = u | ul | ur, my = d | dl | dr;
      uint32_t todo = c & ~(px | mx | py | my);
      uint32_t mpy = c & my & ~py;  // moves +y
      uint32_t xs = c & ~my & (px | mx);
      uint32_t mmy = c & py & ~(my | px | mx);
      if (literal()) {
        // +x or +y alone at distance 1 may lose to -y or -x at distance 2
        todo |= c & ~(my | mx) & (px | py);
        xs &= mx;
        mmy = 0;
      }
      uint32_t mpx = xs & mx & ~px, mmx = xs & px & ~mx;
      if (balance_random()) {
#pragma unroll 1
        for (uint32_t b = xs & px & mx; b; b &= b - 1) {
          const int q = __ffs(b) - 1;
          if (balanced(5, (p.j << 5) + q, wrap_hi(y, L), t) == 1) mpx |= 1u << q;
          else mmx |= 1u << q;
        }
#pragma unroll 1
        for (uint32_t b = c & my & py; b; b &= b - 1) {
          const int q = __ffs(b) - 1;
          if (balanced(6, (p.j << 5) + q, wrap_hi(y, L), t) == 3) mpy |= 1u << q;
          else mmy |= 1u << q;
        }
      }
      if (moves_random()) {
        // a decided anyon may be drawn to move another way (an undecided one draws
        // when it is searched; searching all of them took L = 256, p = 0.05, 16 shots
        // 650 us instead of 358)
#pragma unroll 1
        for (uint32_t b = c & ~todo; b; b &= b - 1) {
          const int q = __ffs(b) - 1;
          const int d = draw_move(key, a.move_thr, site((p.j << 5) + q, wrap_hi(y, L)));
          if (d == 0) continue;
          const uint32_t bit = 1u << q;
          mpx = d == 1 ? mpx | bit : mpx & ~bit;
          mmx = d == 2 ? mmx | bit : mmx & ~bit;
          mpy = d == 3 ? mpy | bit : mpy & ~bit;
          mmy = d == 4 ? mmy | bit : mmy & ~bit;
        }
      }
      const uint32_t fx = mpx | from_right(mmx, p);
      if (on) {
        if (i > 0 && y <= p.y1) fyp[(y - 1) << lws] = up | mmy;
        if (y < p.y1) {
          fxp[y << lws] = fx;
          open[y << lws] = todo;
          n += __popc(todo);
        }
      }
      up = mpy;
      u = c, ul = cl, ur = cr;
      c = d, cl = dl, cr = dr;
    }
    return n;
  }

  // Anyons r0 .. r0 + list_cap - 1 of the undecided ones to the list (this
  // thread's n start at place pos).
  __device__ __forceinline__ void list_open(int t, const Strip& p, int n, int pos, int r0) {
    if (n == 0 || pos >= r0 + g.list_cap || pos + n <= r0) return;
    const uint32_t* open = slot(t + 1) + p.j;
#pragma unroll 1
    for (int y = p.y0; y < p.y1; ++y) {
      uint32_t b = open[y << g.lws];
      while (b) {
        const uint32_t e = ((uint32_t)y << 16) | ((p.j << 5) + __ffs(b) - 1);
        b &= b - 1;
        if (pos >= r0 && pos < r0 + g.list_cap) list[pos - r0] = e;
        ++pos;
      }
    }
  }

  // sigma_{t+1} and the correction from the marked links; the anyons left (ends
  // with a barrier).  moved: whether a link of this thread's flipped.
  __device__ __forceinline__ int apply_dense(int t, const Strip& p, bool& moved) {
    const uint32_t* sig = slot(t) + p.j;
    uint32_t* sn = slot(t + 1) + p.j;
    const uint32_t *fxp = map_x(t) + p.j, *fyp = map_y(t) + p.j;
    uint32_t *cx = C + p.j, *cy = C + g.nws + p.j;
    const int lws = g.lws, H = strip_rows();
    const bool on = p.on && p.y0 < g.L;
    int n = 0;
    if (!on && p.y0 < g.L) {  // padding words stay 0
#pragma unroll 1
      for (int y = p.y0; y < p.y1; ++y) sn[y << lws] = 0;
    }
    uint32_t fu = on ? fyp[wrap_lo(p.y0 - 1, g.L) << lws] : 0u;
#pragma unroll kRowsAhead
    for (int y = p.y0; y < p.y0 + H; ++y) {
      const bool in = on && y < p.y1;
      const int o = y << lws;
      const uint32_t fx = in ? fxp[o] : 0u;
      const uint32_t fxl = from_left(fx, p);
      if (in) {
        const uint32_t fy = fyp[o];
        const uint32_t s = sig[o] ^ ((fx ^ fxl ^ fy ^ fu) & p.valid);
        sn[o] = s;
        n += __popc(s);
        fu = fy;
        moved |= (fx | fy) != 0;
        if (t == 0) {
          cx[o] = fx;
          cy[o] = fy;
        } else if (!LARGE && !g.c_global) {
          cx[o] ^= fx;
          cy[o] ^= fy;
        } else {
          // (no value comes back, so a correction in global memory costs no wait)
          if (fx) atomicXor(&cx[o], fx);
          if (fy) atomicXor(&cy[o], fy);
        }
      }
    }
    return total(n);
  }

  // --------------------------------------------------------- few anyons
  __device__ __forceinline__ Ent enc(uint32_t p) const {
    return LARGE ? (Ent)p : (Ent)((p >> 8) | (p & 0xFFu));
  }
  __device__ __forceinline__ uint32_t dec(Ent e) const {
    return LARGE ? (uint32_t)e : (((uint32_t)e & 0xFF00u) << 8) | ((uint32_t)e & 0xFFu);
  }
  __device__ __forceinline__ Ent* set_of(int s) const {
    return few + (s & (kFewRing - 1)) * kFew;
  }
  // Hits of slice k against the anyon set of step s (a set shorter than 8
  // entries is filled with its first one); near: slice_near serves.
  __device__ __forceinline__ uint32_t slice_set(int s, int x, int y, int k, bool near) const {
    const Ent* e = set_of(s);
    const Ent first = e[0];
    Ent b = first;
    uint32_t m = 0;
    int q = 0;
    if (OPEN || near) {
#pragma unroll 1
      do {
        const uint32_t yx = dec(b);
        m |= slice_near<OPEN>(x, y, (int)(yx & 0xFFFFu), (int)(yx >> 16), g.L, k);
        if (++q == kFew) break;
        b = e[q];
      } while (b != first);
    } else {
      int c = 3 * k + 1;
      if (c >= g.L) c %= g.L;
#pragma unroll 1
      do {
        const uint32_t yx = dec(b);
        m |= slice_pair(x, y, (int)(yx & 0xFFFFu), (int)(yx >> 16), g.L, k, c);
        if (++q == kFew) break;
        b = e[q];
      } while (b != first);
    }
    return (m | edges(x, k)) & slice_limit(a.m_max, k);
  }
  // Writes the anyons with alive set (np on lanes 0 .. n - 1) as the set of step
  // t, sorted; returns the anyon of lane i < number in pos.
  __device__ __forceinline__ uint32_t write_set(int t, uint32_t alive, uint32_t np, int n) {
    int rank = 0;
#pragma unroll 1
    for (int q = 0; q < n; ++q) {
      const uint32_t v = __shfl_sync(kFull, np, q);
      rank += ((alive >> q) & 1u) && v < np;
    }
    Ent* row = set_of(t);
    const int left = __popc(alive);
    if ((alive >> lane) & 1u) row[rank] = enc(np);
    __syncwarp();
    if (lane >= left && lane < kFew) row[lane] = row[0];
    __syncwarp();
    return lane < left ? dec(row[lane]) : 0u;
  }

  // Steps of two anyons from t on, for as long as they hear one another's (or
  // their own) sites of the steps since t_pair: a loop
  // short enough for the nearest instruction cache, since a pair that never
  // meets runs it alone for hundreds of steps.  Stops before step t_event, before
  // a step at which a snapshot's last set comes back (watched), and before a step
  // it cannot decide; returns that step.  n becomes 0 when the pair meets.
  __device__ __forceinline__ int pair_steps(int t, int t_pair, uint32_t& pos, int& n, int near,
                                            bool watched, int t_kept, int t_moving,
                                            int t_event) const {
    constexpr int kWords = kFew * (int)sizeof(Ent) / 4;
    const uint32_t* now = reinterpret_cast<const uint32_t*>(few);
    uint32_t p0 = __shfl_sync(kFull, pos, 0), p1 = __shfl_sync(kFull, pos, 1);
    const uint32_t none = LARGE ? kFull : 0u;  // no set begins with this word
    uint32_t e1 = none, e2 = none;
    if (watched && t_kept >= 0) e1 = snap[(t_kept & (kFewRing - 1)) * kWords];
    if (watched && t_moving >= 0)
      e2 = snap[kFewRing * kWords + (t_moving & (kFewRing - 1)) * kWords];
    const int kk = lane & 15;
    const int klim = min(near, a.m_max / 3) - 1;  // slices that m_max does not cut
    const bool second = lane >= 16;
#pragma unroll 1
    for (const int t0 = t; t < t_event;) {
      const uint32_t e = now[(t & (kFewRing - 1)) * kWords];
      if ((e == e1 || e == e2) && t > t0) break;
      const uint32_t pa = second ? p1 : p0;
      const int xa = pa & 0xFFFFu, ya = pa >> 16;
      const int lim = min(klim, t - t_pair);
      uint32_t hm = 0, hn = 0;  // hits of the first slice with any, of the one after it
      bool next = false;        // hn is known
#pragma unroll 1
      for (int k = kk; k - kk <= lim; k += 16) {
        uint32_t m = 0;
        if (k <= lim) {
          const Ent* set = set_of(t - k);
          const uint32_t b0 = dec(set[0]), b1 = dec(set[1]);
          m = slice_near<false>(xa, ya, (int)(b0 & 0xFFFFu), (int)(b0 >> 16), g.L, k) |
              slice_near<false>(xa, ya, (int)(b1 & 0xFFFFu), (int)(b1 >> 16), g.L, k);
        }
        const uint32_t seg = (__ballot_sync(kFull, m != 0) >> (lane & 16)) & 0xFFFFu;
        const int f = (__ffs(seg) - 1) & 15;
        const uint32_t mm = __shfl_sync(kFull, m, (lane & 16) | f);
        if (!PLAIN) {
          const uint32_t mn = __shfl_sync(kFull, m, (lane & 16) | ((f + 1) & 15));
          if (!hm && seg && f < 15 && k - kk + f < lim) {
            hn = mn;
            next = true;
          }
        }
        if (!hm && seg) hm = mm;
        if (__all_sync(kFull, hm != 0)) break;
      }
      if (lim == klim && !__all_sync(kFull, hm != 0)) {
        // beyond half the torus
        const int lim2 = min((a.m_max / 3) - 1, t - t_pair);
#pragma unroll 1
        for (int k = lim + 1 + kk; k - kk <= lim2; k += 16) {
          uint32_t m = 0;
          if (k <= lim2) m = slice_set(t - k, xa, ya, k, false);
          const uint32_t seg = (__ballot_sync(kFull, m != 0) >> (lane & 16)) & 0xFFFFu;
          const uint32_t mm = __shfl_sync(kFull, m, (lane & 16) | ((__ffs(seg) - 1) & 15));
          if (!hm && seg) hm = mm;
          if (__all_sync(kFull, hm != 0)) break;
        }
      }
      uint32_t h0 = 0, h1 = 0;
      if (hm) nearest(hm, h0, h1);
      // (literal ties may ask for a distance of the next slice)
      if (literal() && !(hm & 0xFFu) && !(h0 & 10u)) {
        h1 = hn & 15u;
        if (!next) hm = 0;
      }
      if (!__all_sync(kFull, hm != 0)) break;
      int dir = direction(h0, h1, PLAIN ? QCA_TIE_LEX : a.tie_order);
      if (dir >= 5) dir = 0;
      const uint32_t np = dir ? site_after(xa, ya, dir) : pa;
      const uint32_t q0 = __shfl_sync(kFull, np, 0), q1 = __shfl_sync(kFull, np, 16);
      const bool swap = q0 == p1 && q1 == p0;
      if (kk == 0 && dir && !(swap && second)) {
        uint32_t bit;
        const int w = link_of(xa, ya, dir, bit);
        atomicXor(&C[w], bit);
      }
      ++t;
      if (swap || q0 == q1) {
        n = 0;
        return t;
      }
      p0 = min(q0, q1);
      p1 = max(q0, q1);
      if (lane < kFew) set_of(t)[lane] = enc(lane == 1 ? p1 : p0);
      __syncwarp();
    }
    pos = lane == 0 ? p0 : (lane == 1 ? p1 : 0u);
    return t;
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
    constexpr int kWords = kFew * (int)sizeof(Ent) / 4;
    const int tf = t;
    uint32_t* const now = reinterpret_cast<uint32_t*>(few);
    const bool watch = !moves_random() && !balance_random();
    // the two snapshots' steps (-1: none), when the next ones are due
    int t_kept = -1, t_moving = -1, due_kept = 0, due_moving = 0, interval = 0;
    int n_before = 0, t_stop = -1, flag = 0;
    const int near = OPEN ? 1 << 20 : (g.L - 1) / 6;  // slices within half the torus
    int t_pair = 1 << 30;            // first step with two anyons
    uint32_t pos = lane < n ? list[lane] : 0u;
    pos = write_set(t, (1u << n) - 1u, pos, n);
#pragma unroll 1
    while (n) {
      if (t >= a.max_steps || t == t_stop) {
        flag = 2;
        t = a.max_steps;
        break;
      }
      if (n == 2 && t_pair > t) t_pair = t;
      if (watch && t_stop < 0) {
        if (n != n_before) {
          // the number of anyons changed: a new orbit, if it is one
          n_before = n;
          t_kept = t_moving = -1;
          due_moving = max(t, tf) + g.kmax + 1;
          due_kept = due_moving + g.kmax + 1;
          interval = 64;
        }
        const uint32_t e = now[(t & (kFewRing - 1)) * kWords];
        if (t_kept >= 0 && e == snap[(t_kept & (kFewRing - 1)) * kWords] &&
            sets_repeat(now, snap, t, t_kept, g.kmax, kWords, lane))
          t_stop = orbit_stop(t, t - t_kept, a.max_steps);
        uint32_t* const snap2 = snap + kFewRing * kWords;
        if (t_stop < 0 && t_moving >= 0 && e == snap2[(t_moving & (kFewRing - 1)) * kWords] &&
            sets_repeat(now, snap2, t, t_moving, g.kmax, kWords, lane))
          t_stop = orbit_stop(t, t - t_moving, a.max_steps);
        if (t_stop >= 0) continue;
        const bool keep = t_kept < 0 && t >= due_kept;
        if (keep || t >= due_moving) {
          // (kFewRing entries cover the kmax + 1 <= 85 sets ending at t)
          __syncwarp();  // every lane has compared with the snapshot it replaces
#pragma unroll 1
          for (int i = lane; i < kFewRing * kWords; i += 32) {
            if (keep) snap[i] = now[i];
            else snap2[i] = now[i];
          }
          if (keep) {
            t_kept = t;
          } else {
            t_moving = t;
            due_moving = t + interval;
            interval <<= 1;
          }
          __syncwarp();
        }
      }
      if (!OPEN && watch && n == 2 && t > t_pair) {
        const int t1 = pair_steps(
            t, t_pair, pos, n, near, t_stop < 0, t_kept, t_moving,
            min(a.max_steps,
                t_stop >= 0 ? t_stop : (t_kept < 0 ? min(due_kept, due_moving) : due_moving)));
        if (t1 != t) {
          t = t1;
          continue;
        }
      }
      const int last = min(t, g.kmax), lastl = min(last, t - tf);
      // lanes = (anyon, slice)
      const int lgS = n <= 2 ? 4 : (n <= 4 ? 3 : 2), S = 1 << lgS;
      const int ai = lane >> lgS, kk = lane & (S - 1);
      const uint32_t pa = __shfl_sync(kFull, pos, ai);
      const int xa = pa & 0xFFFFu, ya = pa >> 16;
      uint32_t hm = 0;  // hits of the first slice with any
      int kf = 0;       // that slice
#pragma unroll 1
      for (int kb = 0; kb <= lastl;) {
        const bool nr = kb < near;
        const int lim = nr ? min(lastl, near - 1) : lastl;
        uint32_t m = 0;
        if (ai < n && !hm && kb + kk <= lim) m = slice_set(t - kb - kk, xa, ya, kb + kk, nr);
        const uint32_t seg = (__ballot_sync(kFull, m != 0) >> (ai << lgS)) & ((1u << S) - 1u);
        const int f = seg ? __ffs(seg) - 1 : 0;
        const uint32_t mm = __shfl_sync(kFull, m, (ai << lgS) + f);
        if (!hm && seg) {
          hm = mm;
          kf = kb + f;
        }
        if (__all_sync(kFull, ai >= n || hm)) break;
        kb = min(kb + S, lim + 1);
      }
      // anyons that hear nothing from the sets: the bitmaps before them, two
      // slices at a time on two lanes of each anyon, the far ones by the warp
      if (lastl < last) {
        const int lastt = min(last, min(g.kthread, t - oldest()));
        int kb = lastl + 1;
        uint32_t open = __ballot_sync(kFull, ai < n && !hm);
#pragma unroll 1
        for (; kb <= lastt && open; kb += 2) {
          uint32_t m = 0;
          const int k = kb + kk;
          if (kk < 2 && k <= lastt && ai < n && !hm)
            m = (slice_thread<OPEN, LARGE ? 6 : 1>(slot(t - k), g.lws, g.L, xa, ya, k) | edges(xa, k)) &
                slice_limit(a.m_max, k);
          const uint32_t m0 = __shfl_sync(kFull, m, ai << lgS);
          const uint32_t m1 = __shfl_sync(kFull, m, (ai << lgS) + 1);
          if (!hm && (m0 | m1)) {
            hm = m0 ? m0 : m1;
            kf = m0 ? kb : kb + 1;
          }
          open = __ballot_sync(kFull, ai < n && !hm);
        }
        if (lastt < last) {
          open = __ballot_sync(kFull, kk == 0 && ai < n && !hm);
#pragma unroll 1
          while (open) {
            const int src = __ffs(open) - 1;
            open &= open - 1;
            int k = max(lastl, lastt) + 1;
            const uint32_t mm =
                search_far(__shfl_sync(kFull, xa, src), __shfl_sync(kFull, ya, src), t, k);
            if (lane == src) {
              hm = mm;
              kf = k;
            }
          }
        }
      }
      uint32_t h0 = 0, h1 = 0;
      if (hm) nearest(hm, h0, h1);
      if (literal()) {
        uint32_t todo = __ballot_sync(
            kFull, kk == 0 && h0 && !(hm & 0xFFu) && !(h0 & 10u) && kf < last);
#pragma unroll 1
        while (todo) {
          const int src = __ffs(todo) - 1;
          todo &= todo - 1;
          const int xs = __shfl_sync(kFull, xa, src), ys = __shfl_sync(kFull, ya, src);
          const int ks = __shfl_sync(kFull, kf, src) + 1;
          const uint32_t mm =
              t - ks >= tf ? slice_set(t - ks, xs, ys, ks, false) : far_slice(xs, ys, t, ks);
          if (lane == src) h1 = mm & 15u;
        }
      }
      __syncwarp();
      if (!LARGE && *(volatile int*)&misc[3]) return;
      // the moves, anyon i on lane i
      h0 = __shfl_sync(kFull, h0, (lane << lgS) & 31);
      h1 = __shfl_sync(kFull, h1, (lane << lgS) & 31);
      const int x = pos & 0xFFFFu, y = pos >> 16;
      const uint64_t key = move_key_of(t);
      const int dir = lane < n ? move_of(key, x, y, t, h0, h1) : 0;
      uint32_t np = pos, bit = 0;
      int lw = 0;
      if (dir) {
        lw = link_of(x, y, dir, bit);
        np = site_after(x, y, dir);
      }
      // a link crossed from both ends (the two anyons swap sites) flips once and
      // takes both; otherwise the anyons are where an odd number of them end
      bool swap = false, first = true;
#pragma unroll 1
      for (int q = 0; q < n; ++q) {
        const uint32_t to = __shfl_sync(kFull, np, q), from = __shfl_sync(kFull, pos, q);
        if (dir && to == pos && from == np) {
          swap = true;
          first = q > lane;
        }
      }
      if (dir && first) atomicXor(&C[lw], bit);
      const bool stays = lane < n && !swap && bulk(np & 0xFFFFu);
      if (!stays) np = 0x80000000u | lane;
      int same = 0, lower = 0;
#pragma unroll 1
      for (int q = 0; q < n; ++q) {
        const uint32_t v = __shfl_sync(kFull, np, q);
        same += v == np;
        lower += v == np && q < lane;
      }
      const uint32_t am = __ballot_sync(kFull, stays && (same & 1) && lower == 0);
      ++t;
      pos = write_set(t, am, np, n);
      n = __popc(am);
    }
    if (lane == 0) {
      misc[4] = t;
      misc[5] = flag;
    }
  }

  // ------------------------------------------------------------ one shot
  __device__ __forceinline__ void zero(uint32_t* p, int words) const {
#pragma unroll 2
    for (int w = tid; w < words; w += NT) p[w] = 0;
  }
  __device__ __forceinline__ void load(const uint8_t* src, int rows, uint32_t* dst, bool any) {
    const int L = g.L;
    if ((L & 15) == 0 && (reinterpret_cast<uintptr_t>(src) & 15) == 0) {
      if (L & 31) {
        zero(dst, rows << g.lws);
        sync();
      }
      load_rows<NT>(src, rows, L, g.lws, dst, any, tid);
    } else {
      zero(dst, rows << g.lws);
      sync();
      load_flat(src, rows, L, g.lws, dst, any, tid, NT);
    }
  }

  __device__ __forceinline__ void run() {
    const int L = g.L, LL = L * L, lws = g.lws;
    const int lastw = (L - 1) >> 5, lastb = (L - 1) & 31;
    const uint8_t* N = a.in + shot_offset_of(a, shot);
    uint8_t* outC = a.out_C + correction_offset_of(a, shot);
    if (!LARGE) {
      uint8_t* room = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(outC) + 3) &
                                                 ~(uintptr_t)3);
      if (g.c_global) {
        C = reinterpret_cast<uint32_t*>(room);
        room += 8 * g.nws;
      }
      if (g.f_global) {
        F = reinterpret_cast<uint32_t*>(room);
        room += 8 * g.nws;
      }
      ar.words = reinterpret_cast<uint32_t*>(room);
      ar.size = (2 * LL - (int)(room - outC)) >> 2;
      ar.head = ar.next = 0;
      ar.listed = 0;
      ar.round = false;
    }
    if (tid < 8) misc[tid] = 0;
    ph = 0;
    tb = 0;
    // ---- sigma_0 (Def. synch_ccqs) and the cut parities of N
    int wx = 0, wy = 0, n = 0;
    uint32_t* s0 = slot(0);
    if (a.from_sigma) {
      if (lastw < (1 << lws) - 1) {
        zero(s0, g.nws);  // the padding words, which no row of bytes covers
        sync();
      }
      load(N, L, s0, true);
      sync();
#pragma unroll 1
      for (int w = tid; w < g.nws; w += NT) n += __popc(s0[w]);
    } else {
      // the link bits, in slots not yet in use
      uint32_t* B = LARGE ? C : ring + 2 * g.nslot;
      load(N, 2 * L, B, false);
      sync();
      const int wsm = (1 << lws) - 1;
#pragma unroll 2
      for (int w = tid; w < g.nws; w += NT) {
        const int y = w >> lws, j = w & wsm;
        uint32_t s = 0;
        if (j <= lastw) {
          const int yu = y == 0 ? L - 1 : y - 1;
          uint32_t bx = B[w], by = B[g.nws + w], bu = B[g.nws + (yu << lws) + j];
          uint32_t carry = j ? B[w - 1] >> 31 : (B[(y << lws) + lastw] >> lastb) & 1u;
          uint32_t cols = j == lastw ? kFull >> (31 - lastb) : kFull;
          if (OPEN) {
            // links that do not exist count for nothing; the rough columns hold no
            // anyons
            if (j == 0) carry = 0;
            if (j == lastw) bx &= ~(1u << lastb), cols &= ~(1u << lastb);
            if (j == 0) cols &= ~1u;
            if (y == L - 1) by = 0;
            if (y == 0) bu = 0;
          }
          s = (bx ^ ((bx << 1) | carry) ^ by ^ bu) & cols;
          if (j == 0) wx ^= (int)(bx & 1u);
          if (y == 0) wy ^= __popc(by) & 1;
        }
        s0[w] = s;
        n += __popc(s);
      }
    }
    n = total(n);
    if (!LARGE && g.nws < g.nslot) {  // the slots' last words
#pragma unroll 1
      for (int i = tid; i < 4 * (g.kmask + 1); i += NT)
        if (g.nws + (i & 3) < g.nslot) ring[(i >> 2) * g.nslot + g.nws + (i & 3)] = 0;
    }
    int t = 0, flag = 0;
    bool listed = n <= g.sparse_max;
    if (listed || a.max_steps == 0) {  // else the first dense step writes it
      zero(C, 2 * g.nws);
      if (listed) zero(table, g.tmask + 1);
      sync();
    }
    // ---- steps.  With the deterministic rules a shot whose anyons have not
    // moved for kmax + 1 steps never moves again.
    const bool watch = !moves_random() && !balance_random();
    int still = 0;
#pragma unroll 1
    while (n) {
      const int nl = advance(t, listed, n);
      if (listed) n = nl;
      if (n == 0) break;
      if (t >= a.max_steps || still > g.kmax) {
        flag = 2;
        t = a.max_steps;
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
      Strip p;
      int mine = 0, pos = 0, todo = n, r0 = 0;
      if (!listed) {
        p = strip();
        mine = mark_dense(t, p);
        pos = places(mine);
        todo = next_counter();
      }
      bool moved = false;
#pragma unroll 1
      for (; r0 < todo; r0 += g.list_cap) {
        if (!listed) {
          list_open(t, p, mine, pos, r0);
          sync();
        }
        moved = sync_or(move_listed(min(todo - r0, g.list_cap), t, listed));
      }
      if (!LARGE && misc[3]) break;
      if (listed) {
        if ((t & kEpochs) == kEpochs) {
          zero(table, g.tmask + 1);
          sync();
        }
      } else {
        moved = false;
        const int left = apply_dense(t, p, moved);
        if (left == n) moved = sync_or(moved);
        else moved = true;
        n = left;
        listed = n <= g.sparse_max;
        if (listed) zero(table, g.tmask + 1);
      }
      still = watch && !moved ? still + 1 : 0;
      ++t;
    }
    if (!LARGE && misc[3]) {
      // the whole CTA leaves together (misc[3] was read behind a barrier); the
      // banded or generic sweep decodes the shot afterwards
      if (tid == 0) {
        a.out_steps[shot] = kStepsPending;
        if (a.pending) atomicAdd(a.pending, 1u);
      }
      return;
    }
    // ---- correction, homology, steps, flag
    if (!LARGE && g.c_global) {
      // the bytes will take the place of the correction's words
#pragma unroll 2
      for (int w = tid; w < 2 * g.nws; w += NT) ring[w] = __ldcg(C + w);
      C = ring;
      sync();
    }
#pragma unroll 1
    for (int y = tid; y < L; y += NT) wx ^= (int)(C[y << lws] & 1u);
#pragma unroll 1
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
    if ((L & 15) == 0 && (reinterpret_cast<uintptr_t>(outC) & 15) == 0)
      store_rows<NT>(outC, 2 * L, L, lws, C, tid);
    else
      store_flat(outC, 2 * L, L, lws, C, tid, NT);
    if (tid == 0) {
      a.out_steps[shot] = t;
      if (a.from_sigma) {
        a.out_cut[2 * shot] = (uint8_t)wx;
        a.out_cut[2 * shot + 1] = (uint8_t)wy;
        if (a.out_exhausted) a.out_exhausted[shot] = (uint8_t)(flag == 2);
      } else {
        // (the open lattice has one cut, between columns 0 and 1)
        a.out_flag[shot] = (uint8_t)(flag == 2 ? 2 : ((OPEN ? wx : wx | wy) ? 1 : 0));
      }
    }
  }
};

}  // namespace hist
}  // namespace qca
