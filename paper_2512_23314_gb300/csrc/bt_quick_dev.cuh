// bt_quick_dev.cuh -- the steps of the level pass by first occurrences
// (bt_quick.cu says what they do), written for any span of threads: the
// kernels of bt_quick.cu run them over a grid, the batched kernel over a CTA or cluster
// (which writes and reads the same arrays in one launch: no __restrict__ here).
#pragma once

#include "bt_bytes.cuh"
#include "bt_internal.cuh"
#include "bt_kr.cuh"
#include "bt_quick.cuh"

namespace bt {

// The threads that share a step: this one's index and their number.
struct Span {
  uint64_t tid, n;
};

constexpr uint32_t kGramLen = 16;
constexpr uint32_t kSubs = kGramLen - 3;       // 4-byte substrings of a gram
constexpr uint32_t kNoDist = 0xFFFFFFFFu;      // no selected gram in the range
constexpr uint32_t kSubMul = 0x9E3779B1u;
constexpr uint32_t kSegBytes = 1024;           // positions per entry of seg1; 64 of those per entry of seg2
// Bytes per comparison item: on the levels of the longest blocks few pieces,
// since nearly all of them are looked at only to find nothing to compare.
__host__ __device__ inline uint64_t q_piece(uint64_t b) { return b >= (64u << 10) ? 32u << 10 : 4u << 10; }

// The 12 words of T[x0, x0 + 48) (zeros past the text's end).
__device__ __forceinline__ void load48(const uint8_t* T, uint64_t n, uint64_t x0, bool aligned, uint32_t* w) {
  if (aligned && x0 + 48 <= n) {
    const uint4* p = (const uint4*)(T + x0);
#pragma unroll
    for (int q = 0; q < 3; q++) {
      const uint4 v = p[q];
      w[4 * q] = v.x, w[4 * q + 1] = v.y, w[4 * q + 2] = v.z, w[4 * q + 3] = v.w;
    }
  } else {
#pragma unroll
    for (int q = 0; q < 12; q++) {
      w[q] = 0;
#pragma unroll
      for (int t = 0; t < 4; t++)
        if (x0 + 4 * q + t < n) w[q] |= (uint32_t)T[x0 + 4 * q + t] << (8 * t);
    }
  }
}

// Which of the 16 grams from x0 (a multiple of 16) on are selected.  T is
// 16-byte aligned and followed by at least 48 readable bytes.
__device__ __forceinline__ uint32_t half_mask(const uint8_t* T, uint64_t n, uint64_t x0) {
  const uint4 v0 = *(const uint4*)(T + x0), v1 = *(const uint4*)(T + x0 + 16);
  const uint32_t w[8] = {v0.x, v0.y, v0.z, v0.w, v1.x, v1.y, v1.z, v1.w};
  uint32_t m[28], c[21];
#pragma unroll
  for (int i = 0; i < 28; i++) m[i] = __funnelshift_r(w[i >> 2], w[(i >> 2) + 1], 8 * (i & 3)) * kSubMul;
#pragma unroll
  for (int i = 0; i < 21; i++)
    c[i] = min(min(min(m[i], m[i + 1]), min(m[i + 2], m[i + 3])), min(min(m[i + 4], m[i + 5]), min(m[i + 6], m[i + 7])));
  uint32_t bits = 0;
#pragma unroll
  for (int i = 0; i < 16; i++) {
    const uint32_t least = min(c[i], c[i + 5]);
    if (m[i] == least || m[i + kSubs - 1] == least) bits |= 1u << i;
  }
  return bits;
}

__device__ __forceinline__ uint32_t gram_cell(uint32_t w0, uint32_t w1, uint32_t w2, uint32_t w3, uint32_t cmask) {
  uint32_t h = w0 * 0x9E3779B1u;
  uint32_t t = w1 * 0x85EBCA77u;
  h ^= __funnelshift_l(t, t, 13);
  t = w2 * 0xC2B2AE3Du;
  h ^= __funnelshift_l(t, t, 7);
  t = w3 * 0x27D4EB2Fu;
  h ^= __funnelshift_l(t, t, 19);
  h ^= h >> 16;
  h *= 0x7FEB352Du;
  h ^= h >> 15;
  h *= 0x846CA68Bu;
  h ^= h >> 16;
  return h & cmask;
}

struct QGeo {
  const uint8_t* T;
  uint64_t n, c, b;
  const uint64_t* st;
};

__device__ __forceinline__ uint64_t qblen(const QGeo& g, uint64_t k) {
  const uint64_t s = g.st[k];
  return g.n - s < g.b ? g.n - s : g.b;
}

// Min over the list entries e in [e0, e1), taken by lane gl of G.
__device__ __forceinline__ uint32_t min_entries(const uint32_t* D, uint32_t e0, uint32_t e1, unsigned gl,
                                                unsigned G, uint32_t d) {
  uint32_t e = e0 + gl;
  for (; e + 3 * G < e1; e += 4 * G) {
    const uint32_t d0 = D[e], d1 = D[e + G], d2 = D[e + 2 * G], d3 = D[e + 3 * G];
    d = min(min(d, min(d0, d1)), min(d2, d3));
  }
  for (; e < e1; e += G) d = min(d, D[e]);
  return d;
}

__device__ __forceinline__ uint32_t list_at(const QList& Q, uint64_t w) { return Q.idx[w < Q.nw ? w : Q.nw]; }

// A[k]: min D over the grams inside block k; X[k]: over the grams that start
// in block k and reach into block k+1 (inside the pair).  A group of G lanes
// per block; a block's inside is read at the coarsest grain that fits it (64
// KiB, 1 KiB, list entries), so that the upper levels cost next to nothing.
__device__ __forceinline__ void quick_min(const QGeo& g, const QList& Q, unsigned G, uint32_t* A,
                                          uint32_t* X, uint32_t* flags, Span w) {
  const unsigned lane = threadIdx.x & 31, grp = lane / G, gl = lane % G, gpw = 32 / G;
  const uint64_t warps = w.n / 32;
  for (uint64_t base = w.tid / 32 * gpw; base < g.c; base += warps * gpw) {
    const uint64_t k = base + grp;
    uint32_t a = kNoDist, xm = kNoDist;
    if (k < g.c) {
      const uint64_t s = g.st[k], len = g.n - s < g.b ? g.n - s : g.b;
      // Gram starts inside the block: [s, aend); inside the pair: [s, pend), pend <= s + len.
      const uint64_t aend = len >= kGramLen ? s + len - kGramLen + 1 : s;
      uint64_t pend = aend;
      if (k + 1 < g.c && g.st[k + 1] == s + len) {
        const uint64_t len2 = g.n - s - len < g.b ? g.n - s - len : g.b;
        if (len + len2 >= kGramLen) {
          pend = s + len + len2 - kGramLen + 1;
          if (pend > s + len) pend = s + len;
        }
      }
      const uint64_t w0 = (s + 31) / 32, w1 = aend / 32;
      uint64_t rest = s;  // first position not covered by whole words
      if (w1 > w0) {
        if (s & 31) {
          for (uint32_t e = list_at(Q, s / 32) + gl, e1 = list_at(Q, w0); e < e1; e += G)
            if (Q.x[e] >= s) a = min(a, Q.D[e]);
        }
        const uint64_t j0 = (w0 + 31) / 32, j1 = w1 / 32;  // 1 KiB segments inside
        if (j1 > j0 + 2) {
          a = min_entries(Q.D, list_at(Q, w0), list_at(Q, 32 * j0), gl, G, a);
          const uint64_t i0 = (j0 + 63) / 64, i1 = j1 / 64;
          if (i1 > i0) {
            a = min_entries(Q.seg1, (uint32_t)j0, (uint32_t)(64 * i0), gl, G, a);
            a = min_entries(Q.seg2, (uint32_t)i0, (uint32_t)i1, gl, G, a);
            a = min_entries(Q.seg1, (uint32_t)(64 * i1), (uint32_t)j1, gl, G, a);
          } else {
            a = min_entries(Q.seg1, (uint32_t)j0, (uint32_t)j1, gl, G, a);
          }
          a = min_entries(Q.D, list_at(Q, 32 * j1), list_at(Q, w1), gl, G, a);
        } else {
          a = min_entries(Q.D, list_at(Q, w0), list_at(Q, w1), gl, G, a);
        }
        rest = 32 * w1;
      }
      for (uint32_t e = list_at(Q, rest / 32) + gl, e1 = list_at(Q, (pend + 31) / 32); e < e1; e += G) {
        const uint64_t p = Q.x[e];
        if (p < s || p >= pend) continue;
        if (p < aend) a = min(a, Q.D[e]);
        else xm = min(xm, Q.D[e]);
      }
    }
    for (unsigned o = G / 2; o; o >>= 1) {
      a = min(a, __shfl_xor_sync(0xFFFFFFFFu, a, o));
      xm = min(xm, __shfl_xor_sync(0xFFFFFFFFu, xm, o));
    }
    if (k < g.c && gl == 0) {
      A[k] = a;
      X[k] = xm;
      flags[k] = 0;
    }
  }
}

// min D over the pair (k, k+1).
__device__ __forceinline__ uint32_t pair_dist(const uint32_t* A, const uint32_t* X, uint64_t k,
                                              uint64_t len2) {
  const uint32_t d = min(A[k], X[k]);
  return len2 >= kGramLen ? min(d, A[k + 1]) : d;
}

constexpr uint32_t kBlkDiffers = 1, kPairDiffers = 2;

// Compare every block and pair with the bytes at its bound s - min D (at 0
// when the bound is negative): flags[k] says which differ.  A group of L lanes
// per piece of the pair; the block's comparison is the first half of the
// pair's when both have the same bound.  Bound: instruction issue (nearly every
// block is looked at, few bytes each), so a lane takes about four 16-byte
// units rather than one -- the item's bookkeeping is then shared by more
// lanes' worth of text -- and positions are 32 bits.  With one unit per lane
// and 64-bit positions: 836 us on the 256 MiB text and 6.4 ms on 2 GiB of DNA
// copies (55-70 % of the issue slots, 10-13 % of DRAM).
__device__ __forceinline__ void quick_compare(const QGeo& g, const uint32_t* A,
                                              const uint32_t* X, uint32_t* flags,
                                              uint32_t ppk, unsigned L, Span w) {
  const unsigned lane = threadIdx.x & 31, grp = lane / L, gl = lane % L, gpw = 32 / L;
  const unsigned gmask = (L == 32 ? 0xFFFFFFFFu : ((1u << L) - 1u)) << (grp * L);
  const bool aligned16 = (((uintptr_t)g.T) & 15) == 0;
  const uint32_t c = (uint32_t)g.c, n = (uint32_t)g.n, bl = (uint32_t)(g.b < g.n ? g.b : g.n);
  const uint32_t warps = (uint32_t)(w.n / 32), total = c * ppk, piece = (uint32_t)q_piece(g.b);
  // Warp-uniform loop: every lane reaches the ballots of every iteration.
  for (uint32_t base = (uint32_t)(w.tid / 32) * gpw; base < total; base += warps * gpw) {
    const uint32_t u = base + grp;
    bool db = false, dp = false;
    uint32_t k = 0;
    if (u < total) {
      k = ppk == 1 ? u : u / ppk;
      const uint32_t off = ppk == 1 ? 0 : (u - k * ppk) * piece;
      const uint32_t s = (uint32_t)g.st[k], dk = A[k], xk = X[k];
      const bool more = k + 1 < c;
      const uint32_t s1 = more ? (uint32_t)g.st[k + 1] : 0, d1 = more ? A[k + 1] : 0;
      const uint32_t f = ppk > 1 ? *(volatile uint32_t*)&flags[k] : 0u;  // (another piece may have settled it)
      const uint32_t len = n - s < bl ? n - s : bl;
      const bool blk = dk != 0 && dk != kNoDist && s != 0 && off < len && !(f & kBlkDiffers);
      bool pair = false;
      uint32_t d2 = 0, plen = 0;
      if (more && s != 0 && s1 == s + len) {
        const uint32_t len2 = n - s1 < bl ? n - s1 : bl;
        plen = len + len2;
        d2 = min(dk, xk);
        if (len2 >= kGramLen) d2 = min(d2, d1);
        pair = d2 != 0 && d2 != kNoDist && off < plen && !(f & kPairDiffers);
      }
      if (blk || pair) {
        const uint32_t pk = dk > s ? 0 : s - dk, pp = d2 > s ? 0 : s - d2;
        const uint32_t bend = min(off + piece, len), pend = min(off + piece, plen);
        const bool one = blk && pair && pk == pp;
        if (aligned16 && ((s | len | off) & 15) == 0 && (!pair || (plen & 15) == 0)) {
          // One bound for both: the block's bytes are the pair's first half.
          if (blk) {
            const Shift16 sh(pk);
            for (uint32_t y = off + 16 * gl; y < (one ? pend : bend); y += 32 * L) {
              const uint32_t y2 = y + 16 * L < (one ? pend : bend) ? y + 16 * L : y;
              const Unit16 a = load_units(g.T, pk + y, s + y), b = load_units(g.T, pk + y2, s + y2);
              const bool da = sh.differ(a), dc = sh.differ(b);
              if (one) dp |= da | dc;
              db |= (da && y < len) || (dc && y2 < len);
            }
          }
          if (pair && !one) {
            const Shift16 sh(pp);
            for (uint32_t y = off + 16 * gl; y < pend; y += 32 * L) {
              const uint32_t y2 = y + 16 * L < pend ? y + 16 * L : y;
              const Unit16 a = load_units(g.T, pp + y, s + y), b = load_units(g.T, pp + y2, s + y2);
              dp |= sh.differ(a) | sh.differ(b);
            }
          }
        } else {
          if (blk) {
            db = differs(g.T, g.n, aligned16, pk, s, off, bend, gl, L);
            if (one) dp = db;
          }
          if (pair) {
            const uint32_t from = one ? max(off, bend) : off;
            if (from < pend) dp |= differs(g.T, g.n, aligned16, pp, s, from, pend, gl, L);
          }
        }
      }
    }
    const unsigned bb = __ballot_sync(0xFFFFFFFFu, db), bp = __ballot_sync(0xFFFFFFFFu, dp);
    const uint32_t set = (bb & gmask ? kBlkDiffers : 0u) | (bp & gmask ? kPairDiffers : 0u);
    if (u < total && gl == 0 && set) atomicOr(&flags[k], set);
  }
}

__device__ __forceinline__ uint64_t warp_sum64(uint64_t v) {
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xFFFFFFFFu, v, o);
  return v;
}

constexpr uint8_t kIsPair = 1, kLeftmost = 2;  // state of the pair (k, k+1)

// What the comparisons say about the pair (k, k+1).
__device__ __forceinline__ uint8_t pair_state(const QGeo& g, const uint32_t* A, const uint32_t* X,
                                              const uint32_t* flags, uint64_t k, uint32_t* dist, uint64_t* plen,
                                              bool* open) {
  *open = false;
  if (k + 1 >= g.c) return 0;
  const uint64_t s = g.st[k], len = g.n - s < g.b ? g.n - s : g.b;
  if (g.st[k + 1] != s + len) return 0;
  const uint64_t len2 = g.n - s - len < g.b ? g.n - s - len : g.b;
  const uint32_t d = pair_dist(A, X, k, len2);
  *dist = d;
  *plen = len + len2;
  if (s == 0 || d == 0) return kIsPair | kLeftmost;
  *open = d == kNoDist || (flags[k] & kPairDiffers);
  return kIsPair;
}

// ---------------------------------------------------------------------------
// The open keys: every occurrence of an open key has the key's newest gram at
// the key's offset.  (gram, offset) pairs go to a table, each once; the list
// scan proposes p = x - offset wherever one of the grams occurs before the
// last start of a key with that pair, and a proposed window's fingerprint is
// looked up among the open blocks (and, joined with the one at p + b, among
// the open pairs).  A gram is named by its first position F.
//
// Where few grams make up the text (records from few values, words in any order,
// two letters), many keys have the same newest gram, each at an offset of its
// own, and a window is proposed once for every gram it holds: up to hundreds of
// windows per text position.  Two other ways are tried then.  The keys go by their
// *first* gram: of any 12 consecutive grams one is selected, so its offset is at
// most 11, and the first gram of a window is the list's next entry, so an entry at
// x proposes only windows after the entry before it, each window once.  That is
// little where keys start at few places of the grams (records), and a window per
// position where they start anywhere; then every window is scanned.
// ---------------------------------------------------------------------------
struct __align__(32) CSlot {  // a block fingerprint: leftmost window, last start of an open pair beginning with it
  unsigned long long key, lo, maxpst, pad;
};
struct __align__(16) CPair {  // (slot, slot): leftmost window
  unsigned long long key, lo;
};
struct __align__(16) CGram {  // F << 32 | offset; windows from `bound` on are of no use
  unsigned long long key, bound;
};

// When a search is given up.  Its work is counted in steps of a warp's walk over
// the gram table (about 0.45 ns each with the whole GPU), and six for testing 32
// windows (2.9 ns); the scan of every window costs about n / 26 of these (4.6 ms on
// 256 MiB).  With a list long enough for two parts the first sixteenth is a
// sample: above n / 700 there (versions and copies stay below n / 800), or given up
// at n / 64, first grams are tried on the same sixteenth, and the better way takes
// the rest unless both are above n / 256.  No search goes on beyond n / 32.
// Giving up has a price of its own, so no bound but the sample's comparisons is below
// a fixed one.  On the grid 2^21 steps: with bounds of n / 32 + 4096 two-letter runs of
// 256 KiB took 3.11 ms and random bits of 1 MiB 2.09, now 1.66 and 1.70 (1.65 and 1.68
// without bounds); such runs of 512 KiB by 2^16, 2^18, 2^20: 3.24, 2.21, 2.08.  For one
// CTA it is 2^17 on documents below 96 KiB and 2^12 on longer ones: 256 documents of
// two-letter runs by 2^12 and 2^15, 32 KiB 5.6 and 4.7 ms, 128 KiB 9.8 and 14.7.  The
// registration is given up too: keys that share a gram stand in one run of slots,
// which each passes (80 ns a slot: 4 M keys of two-letter text took 30 ms).
enum ChaseState : uint32_t {
  kSearchDone = 0,
  kCompare = 1,   // the sample is done, and much work
  kTryFirst = 2,  // registration or sample given up
  kGiveUp = 3,
};
constexpr uint32_t kWalkWork = 1, kTestWork = 6;
__host__ __device__ inline uint64_t work_sample(uint64_t n) { return n / 700; }
__host__ __device__ inline uint64_t work_few(uint64_t n) { return n / 256 + 4096; }
__host__ __device__ inline uint64_t work_most(uint64_t n, bool sample, uint64_t least) {
  const uint64_t most = sample ? n / 64 : n / 32;
  return most > least ? most : least;
}
constexpr uint64_t kLeastWork = 1u << 21;
__host__ __device__ inline uint64_t least_work_cta(uint64_t n) { return n < (96u << 10) ? 1u << 17 : 1u << 12; }
constexpr uint32_t kLongProbe = 64;  // slots; a walk counts from there on
__host__ __device__ inline uint64_t probes_most(uint64_t nitems) { return 4 * nitems + (1u << 16); }

struct Chase {
  bool first;              // keys go by their first gram (otherwise by their newest)
  uint64_t probes;         // most slots passed by long walks before the registration is given up
  QGeo g;
  QList Q;
  const uint32_t* A;
  const uint32_t* X;
  const uint32_t* items;
  uint32_t nitems;
  uint64_t Bb, Br, r;  // B^b, B^r; length of the short last block (0: none)
  CSlot* bt;
  CPair* pt;
  CGram* gt;
  uint32_t bmask, pmask, gmask;
  uint32_t* bitmap;
  uint32_t bshift;         // bitmap bit = (F * odd) >> bshift
  uint32_t* islot;         // per item: its slot in bt or pt
  uint32_t* igram;         // per item: its slot in gt
  unsigned long long* bound2;
  uint32_t* differ;        // per item: the verification found a difference
  uint32_t* susp;          // items whose fingerprint match was false
  unsigned long long* exlo;
  QuickStatus* qs;
  Status* status;
  uint64_t* lo;
  uint8_t* ps;
};

constexpr uint32_t kTailItem = 0xFFFFFFFEu;  // islot of a key that ends in the short last block

template <class S>
__device__ __forceinline__ uint32_t c_insert(S* t, uint32_t mask, unsigned long long key) {
  uint32_t h = (uint32_t)mix64(key) & mask;
  for (uint32_t it = 0; it <= mask; it++) {
    unsigned long long old = *(volatile unsigned long long*)&t[h].key;
    if (old == kNone) old = atomicCAS(&t[h].key, (unsigned long long)kNone, key);
    if (old == kNone || old == key) return h;
    h = (h + 1) & mask;
  }
  return kNoSlot;
}
template <class S>
__device__ __forceinline__ uint32_t c_find(const S* t, uint32_t mask, unsigned long long key) {
  uint32_t h = (uint32_t)mix64(key) & mask;
  for (uint32_t it = 0; it <= mask; it++) {
    const unsigned long long k = t[h].key;
    if (k == key) return h;
    if (k == kNone) return kNoSlot;
    h = (h + 1) & mask;
  }
  return kNoSlot;
}
// Grams probe from a place that depends on F alone, so that all offsets of a
// gram are met on one walk to the next empty slot.
__device__ __forceinline__ uint32_t c_gram_home(uint32_t F, uint32_t mask) {
  uint32_t h = F * 0x9E3779B1u;
  h ^= h >> 15;
  h *= 0x85EBCA77u;
  h ^= h >> 13;
  return h & mask;
}
__device__ __forceinline__ uint32_t c_bit(const Chase& C, uint32_t F) { return (F * 0xC2B2AE3Du) >> C.bshift; }

__device__ __forceinline__ void c_min(unsigned long long* a, uint64_t p) {
  if (*(volatile unsigned long long*)a > p) atomicMin(a, (unsigned long long)p);
}

// `again`: the gram table alone (the keys' tables and what was found stay).
__device__ __forceinline__ void chase_init(const Chase& C, uint32_t bwords, bool again, Span w) {
  uint64_t top = (uint64_t)C.bmask + 1;
  top = top > (uint64_t)C.pmask + 1 ? top : (uint64_t)C.pmask + 1;
  top = top > (uint64_t)C.gmask + 1 ? top : (uint64_t)C.gmask + 1;
  top = top > bwords ? top : bwords;
  for (uint64_t i = w.tid; i < top; i += w.n) {
    if (i <= C.bmask && !again) C.bt[i] = CSlot{kNone, kNone, 0, 0};
    if (i <= C.pmask && !again) C.pt[i] = CPair{kNone, kNone};
    if (i <= C.gmask) {
      C.gt[i] = CGram{kNone, 0};
      C.bound2[i] = 0;
    }
    if (i < bwords) C.bitmap[i] = 0;
    if (i < C.nitems) {
      C.differ[i] = 0;
      C.igram[i] = C.islot[i] = kNoSlot;  // (a registration that is given up leaves some)
    }
    if (i == 0) {
      C.qs->tail_F = C.qs->tail_off = 0xFFFFFFFFu;
      C.qs->redo = kSearchDone;
      C.qs->probes = 0;
    }
    if (i == 0 && !again) {
      C.qs->fp_tail = C.qs->lo_tail = C.qs->lo_tailpair = kNone;
      C.qs->pretail = kNoSlot;
      C.qs->cands = C.qs->hits = C.qs->work = 0;
    }
  }
}

// G lanes per open key (one when blocks are short, else a warp): the list entry
// with the key's min D (or its first entry), then (one lane) the tables.  A pair
// enters both of its blocks.
template <class M, unsigned G>
__device__ __forceinline__ void chase_keys(const M& m, const PrefixAt<M>& H, const Chase& C, Span w) {
  const unsigned gl = threadIdx.x % G;
  const QGeo& g = C.g;
  for (uint64_t i = w.tid / G; i < C.nitems; i += w.n / G) {
    const uint32_t it = C.items[i];
    const bool given_up = *(volatile unsigned int*)&C.qs->redo != kSearchDone;
    if (G == 1 ? given_up : __any_sync(0xFFFFFFFFu, given_up)) return;  // (a warp's lanes together: they vote below)
    const uint64_t k = it >> 1;
    const bool pair = it & 1;
    const uint64_t s = g.st[k], len = g.n - s < g.b ? g.n - s : g.b;
    const uint64_t len2 = pair ? (g.n - s - len < g.b ? g.n - s - len : g.b) : 0;
    const uint32_t d = pair ? pair_dist(C.A, C.X, k, len2) : C.A[k];
    const uint64_t end = s + len + len2 - kGramLen + 1;  // gram starts [s, end) when the key has a gram at all
    uint32_t F = 0, off = 0;
    bool found = false;
    if (d != kNoDist) {
      const uint32_t e1 = list_at(C.Q, (end + 31) / 32);
      for (uint32_t e0 = list_at(C.Q, s / 32); e0 < e1 && !found; e0 += G) {
        const uint32_t e = e0 + gl;
        const uint32_t x = e < e1 ? C.Q.x[e] : 0, D = e < e1 ? C.Q.D[e] : 0;
        const bool hit = e < e1 && x >= s && x < end && (C.first || D == d);
        if (G == 1) {
          found = hit;
          if (hit) F = x - D, off = (uint32_t)(x - s);
        } else {
          const unsigned bal = __ballot_sync(0xFFFFFFFFu, hit);
          found = bal != 0;
          if (found) {
            const uint32_t fx = __shfl_sync(0xFFFFFFFFu, x, __ffs(bal) - 1);
            F = fx - __shfl_sync(0xFFFFFFFFu, D, __ffs(bal) - 1), off = (uint32_t)(fx - s);
          }
        }
      }
    }
    if (gl) continue;
    const bool tail = !pair && len != g.b;
    if (found && !tail) {
      uint32_t h = c_gram_home(F, C.gmask);
      const unsigned long long key = ((unsigned long long)F << 32) | off;
      bool placed = false;
      for (uint32_t q = 0; q <= C.gmask && !placed; q++) {
        unsigned long long old = *(volatile unsigned long long*)&C.gt[h].key;
        if (old == kNone) old = atomicCAS(&C.gt[h].key, (unsigned long long)kNone, key);
        if (old == kNone || old == key) placed = true;
        else h = (h + 1) & C.gmask;
        if (q % kLongProbe == kLongProbe - 1 && !placed &&
            atomicAdd(&C.qs->probes, (unsigned long long)kLongProbe) >= C.probes) {
          C.qs->redo = kTryFirst;
          break;
        }
      }
      if (placed) {
        atomicMax(&C.gt[h].bound, (unsigned long long)s);
        C.igram[i] = h;
      } else if (!C.qs->redo) {
        atomicExch(&C.status->error, 21ull);
      }
    }
    if (found) {
      const uint32_t bit = c_bit(C, F);
      atomicOr(&C.bitmap[bit >> 5], 1u << (bit & 31));
    } else if (!tail) {
      atomicExch(&C.status->error, 22ull);  // a key of 27 bytes or more has a selected gram
    }
    const uint64_t h0 = H.at(m, s), h1 = H.at(m, s + len);
    if (tail) {
      C.qs->fp_tail = m.sub(h1, m.mul(h0, C.Br));
      c_min(&C.qs->lo_tail, s);
      if (found) {
        C.qs->tail_F = F;
        C.qs->tail_off = off;
      }
      C.islot[i] = kTailItem;
      continue;
    }
    const uint32_t slot = c_insert(C.bt, C.bmask, m.sub(h1, m.mul(h0, C.Bb)));
    if (slot == kNoSlot) {
      atomicExch(&C.status->error, 23ull);
      continue;
    }
    c_min(&C.bt[slot].lo, s);
    if (!pair) {
      C.islot[i] = slot;
      continue;
    }
    atomicMax(&C.bt[slot].maxpst, (unsigned long long)s);
    const uint64_t h2 = H.at(m, s + len + len2);
    if (len2 != g.b) {  // the pair that ends in the short last block
      C.qs->pretail = slot;
      C.qs->fp_tail = m.sub(h2, m.mul(h1, C.Br));
      c_min(&C.qs->lo_tailpair, s);
      C.islot[i] = kTailItem;
      continue;
    }
    const uint32_t slot2 = c_insert(C.bt, C.bmask, m.sub(h2, m.mul(h1, C.Bb)));
    const uint32_t sp = slot2 == kNoSlot ? kNoSlot : c_insert(C.pt, C.pmask, ((unsigned long long)slot << 32) | slot2);
    if (sp == kNoSlot) {
      atomicExch(&C.status->error, 24ull);
      continue;
    }
    c_min(&C.pt[sp].lo, s);
    C.islot[i] = sp;
  }
}

// The window at p: its fingerprint among the open blocks, joined with the
// window at p + b among the open pairs.
template <class M>
__device__ __forceinline__ void chase_test(const M& m, const PrefixAt<M>& H, const Chase& C, uint64_t p, uint32_t pretail,
                                        uint64_t fp_tail, uint32_t& nhit) {
  const QGeo& g = C.g;
  if (p + g.b > g.n) return;
  const uint64_t h0 = H.at(m, p), h1 = H.at(m, p + g.b);
  const uint32_t sl = c_find(C.bt, C.bmask, m.sub(h1, m.mul(h0, C.Bb)));
  if (sl == kNoSlot) return;
  nhit++;
  c_min(&C.bt[sl].lo, p);
  if (p > C.bt[sl].maxpst) return;
  if (p + 2 * g.b <= g.n) {
    const uint32_t s2 = c_find(C.bt, C.bmask, m.sub(H.at(m, p + 2 * g.b), m.mul(h1, C.Bb)));
    if (s2 != kNoSlot) {
      const uint32_t sp = c_find(C.pt, C.pmask, ((unsigned long long)sl << 32) | s2);
      if (sp != kNoSlot) c_min(&C.pt[sp].lo, p);
    }
  }
  if (C.r && sl == pretail && p + g.b + C.r <= g.n &&
      m.sub(H.at(m, p + g.b + C.r), m.mul(h1, C.Br)) == fp_tail)
    c_min(&C.qs->lo_tailpair, p);
}

// List entries [e0, e1): the bitmap test, then per warp a queue of gram hits
// in shared memory, the gram table's walk, a queue of proposed windows and
// their tests, by full warps and without a barrier.  Neither
// queue can overflow: a batch is taken out as soon as there are 32 entries.
// Bound: the list's stream, one bitmap test per entry, and the chains of
// dependent reads of the hits (table, prefix values and text, block table).  A
// warp that walked 32 hits until the longest walk ended took 14.0 ms on 2 GiB of
// DNA copies and 1.37 on 256 MiB of text; lanes that take the next hit when
// theirs has ended, across tiles, 9.2 and 1.23.
constexpr uint32_t kChaseTile = 256;                 // entries per warp and step, eight per lane
constexpr uint32_t kHitQ = kChaseTile + 32, kCandQ = 64;
constexpr uint32_t kChaseBitWords = 4096;            // bitmap kept in shared memory up to 16 KiB
// Work of a warp before it adds it to the level's: often enough that what all warps
// do meanwhile is no more than the limit, or 64.
constexpr uint32_t kChaseReport = 256, kChaseReportOften = 64;

// hq, cq: the warp's queues; gq: for first grams, the distance of each hit to
// the entry before it; bits: the bitmap (shared or global memory).  Above a work of
// `limit` on the level in all it stops and leaves `verdict` in C.qs->redo.  first:
// as C.first, or that value as a type.
template <class M, class FIRST>
__device__ __forceinline__ void chase_scan(const M& m, const PrefixAt<M>& H, const Chase& C, FIRST first, uint32_t e0, uint32_t e1,
                                           const uint32_t* bits, uint2* hq, uint8_t* gq, uint32_t* cq,
                                           const unsigned long long* bound2, unsigned long long limit,
                                           ChaseState verdict, Span w) {
  const unsigned lane = threadIdx.x & 31, lt = (1u << lane) - 1u;
  uint32_t hn = 0, cn = 0;  // warp-uniform
  const uint32_t tail_F = C.qs->tail_F, tail_off = C.qs->tail_off, pretail = C.qs->pretail;
  const uint64_t fp_tail = C.qs->fp_tail;
  const uint32_t given_up = *(volatile unsigned int*)&C.qs->redo;  // (before, or just now: looked at with the first tile)
  uint32_t ncand = 0, nhit = 0, work = 0;  // ncand, work (since the last report): warp-uniform
  const uint32_t every = limit >= kChaseReport * (w.n / 32) ? kChaseReport : kChaseReportOften;
  bool stop = false;
  auto report = [&]() {
    unsigned long long all = 0;
    if (lane == 0) all = atomicAdd(&C.qs->work, (unsigned long long)work) + work;
    work = 0;
    stop = __shfl_sync(0xFFFFFFFFu, all > limit, 0);
    if (stop && lane == 0) C.qs->redo = verdict;
  };
  // 32 proposed windows (fewer at the end).
  auto take_cands = [&]() {
    const uint32_t n = cn < 32 ? cn : 32;
    __syncwarp();
    if (lane < n) chase_test(m, H, C, cq[cn - n + lane], pretail, fp_tail, nhit);
    cn -= n;
    __syncwarp();
  };
  // One step of the lanes' walks: a lane whose walk has ended takes the next
  // gram hit, every lane looks at one slot of the table, and a slot that holds
  // its gram proposes a window.  (Walks end: half the slots are empty.)
  bool live = false;
  uint2 hit = make_uint2(0, 0);
  uint32_t s = 0, gap = 0xFFFFFFFFu;
  auto walk = [&]() {
    __syncwarp();
    const unsigned idle = __ballot_sync(0xFFFFFFFFu, !live);
    const uint32_t k = __popc(idle & lt), free = __popc(idle);
    if (!live && k < hn) {
      hit = hq[hn - 1 - k];
      if (first) gap = gq[hn - 1 - k];
      s = c_gram_home(hit.y, C.gmask);
      live = true;
      if (hit.y == tail_F && tail_off <= hit.x) {
        const uint64_t p = hit.x - tail_off;
        if (p + C.r < C.g.n && p < *(volatile unsigned long long*)&C.qs->lo_tail &&
            m.sub(H.at(m, p + C.r), m.mul(H.at(m, p), C.Br)) == fp_tail)
          c_min(&C.qs->lo_tail, p);
      }
    }
    hn -= free < hn ? free : hn;
    bool want = false;
    uint32_t p = 0;
    if (live) {
      const ulonglong2 en = *(const ulonglong2*)&C.gt[s];
      if (en.x == kNone) {
        live = false;
      } else if ((uint32_t)(en.x >> 32) == hit.y) {
        const uint32_t off = (uint32_t)en.x;
        p = hit.x - off;
        want = off <= hit.x && (!first || off < gap) && p < (bound2 ? bound2[s] : en.y);
      }
      s = (s + 1) & C.gmask;
    }
    const unsigned bal = __ballot_sync(0xFFFFFFFFu, want);
    if (bal) {
      if (want) cq[cn + __popc(bal & lt)] = p;
      cn += __popc(bal);
      ncand += __popc(bal);
      if (cn >= 32) {
        take_cands();
        work += kTestWork;
      }
    }
    work += kWalkWork;
    if (work >= every) {
      report();
      if (stop) live = false, hn = cn = 0;
    }
  };
  // (A short list is dealt out one entry a lane: eight would leave most warps
  // without and the others with eight times the steps one after the other.)
  const uint32_t per = e1 - e0 <= w.n ? 1 : kChaseTile / 32;
  for (uint64_t t0 = e0 + w.tid / 32 * (32 * per); t0 < e1 && !stop; t0 += w.n / 32 * (32 * per)) {
    uint32_t x[8], F[8];
    uint32_t pass = 0;
    const uint64_t e = t0 + (uint64_t)per * lane;
    if (per == 8 && e + 8 <= e1) {
#pragma unroll
      for (int q = 0; q < 2; q++) {
        const uint4 a = ((const uint4*)(C.Q.x + e))[q], d = ((const uint4*)(C.Q.D + e))[q];
        x[4 * q] = a.x, x[4 * q + 1] = a.y, x[4 * q + 2] = a.z, x[4 * q + 3] = a.w;
        F[4 * q] = a.x - d.x, F[4 * q + 1] = a.y - d.y, F[4 * q + 2] = a.z - d.z, F[4 * q + 3] = a.w - d.w;
      }
#pragma unroll
      for (int u = 0; u < 8; u++) {
        const uint32_t bit = c_bit(C, F[u]);
        pass |= ((bits[bit >> 5] >> (bit & 31)) & 1u) << u;
      }
    } else {
#pragma unroll
      for (int u = 0; u < 8; u++) {
        x[u] = F[u] = 0;
        if (u >= (int)per || e + u >= e1) continue;
        x[u] = C.Q.x[e + u];
        F[u] = x[u] - C.Q.D[e + u];
        const uint32_t bit = c_bit(C, F[u]);
        pass |= ((bits[bit >> 5] >> (bit & 31)) & 1u) << u;
      }
    }
    if (__any_sync(0xFFFFFFFFu, given_up)) break;
#pragma unroll
    for (int u = 0; u < 8; u++) {
      const bool ok = (pass >> u) & 1u;
      const unsigned bal = __ballot_sync(0xFFFFFFFFu, ok);
      if (ok) {
        const uint32_t at = hn + __popc(bal & lt);
        hq[at] = make_uint2(x[u], F[u]);
        // (The text's first entry proposes every window before it: 255 is more than any offset of a first gram.)
        if (first) gq[at] = e + u ? (uint8_t)min(x[u] - (u ? x[u ? u - 1 : 0] : C.Q.x[e - 1]), 255u) : (uint8_t)255;
      }
      hn += __popc(bal);
    }
    while (hn >= 32) walk();  // (unfinished walks go on with the next tile's)
  }
  while (hn || __any_sync(0xFFFFFFFFu, live)) walk();
  while (cn) take_cands();
  nhit = __reduce_add_sync(0xFFFFFFFFu, nhit);
  if (lane == 0 && work) atomicAdd(&C.qs->work, (unsigned long long)work);
  if (lane == 0 && ncand) atomicAdd(&C.qs->cands, (unsigned long long)ncand);
  if (lane == 0 && nhit) atomicAdd(&C.qs->hits, (unsigned long long)nhit);
}

// Between the two halves of the scan: a (gram, offset) pair's windows are of
// use up to the largest leftmost window found so far among its keys.
__device__ __forceinline__ void chase_bound(const Chase& C, Span w) {
  for (uint64_t i = w.tid; i < C.nitems; i += w.n) {
    const uint32_t h = C.igram[i], sl = C.islot[i];
    if (h == kNoSlot || sl == kNoSlot) continue;
    const bool pair = C.items[i] & 1;
    const unsigned long long lo = sl == kTailItem ? C.qs->lo_tailpair : pair ? C.pt[sl].lo : C.bt[sl].lo;
    atomicMax(&C.bound2[h], lo);
  }
}

// After chase_bound, into a cleared bitmap: the grams that entries from `split` on
// can still propose a window for.  The copies' content is settled by then, and
// its grams, most of the list's hits, are left out (the search on 2 GiB of DNA
// copies: 16.3 ms without, 14.0 with).
__device__ __forceinline__ void chase_live(const Chase& C, uint32_t split, Span w) {
  const uint32_t xs = C.Q.x[split];
  auto set = [&](uint32_t F) {
    const uint32_t bit = c_bit(C, F), one = 1u << (bit & 31);
    if (!(*(volatile uint32_t*)&C.bitmap[bit >> 5] & one)) atomicOr(&C.bitmap[bit >> 5], one);
  };
  for (uint64_t i = w.tid; i <= C.gmask; i += w.n) {
    const unsigned long long key = C.gt[i].key;
    if (key != kNone && C.bound2[i] + (uint32_t)key > xs) set((uint32_t)(key >> 32));
  }
  if (w.tid == 0 && C.qs->tail_F != 0xFFFFFFFFu) set(C.qs->tail_F);
}

// The short last block when it has no selected gram (at most 26 bytes): every
// position before it, 16 per thread, filtered by its first bytes.
__device__ __forceinline__ void chase_tail(const Chase& C, Span w) {
  if (C.qs->lo_tail == kNone || C.qs->tail_F != 0xFFFFFFFFu) return;  // not open, or found through its gram
  const QGeo& g = C.g;
  const uint64_t s = g.st[g.c - 1], r = C.r;
  const uint32_t f = (uint32_t)(r < 4 ? r : 4);
  uint32_t want = 0;
  for (uint32_t t = 0; t < f; t++) want |= (uint32_t)g.T[s + t] << (8 * t);
  const uint32_t fm = f == 4 ? 0xFFFFFFFFu : (1u << (8 * f)) - 1u;
  const bool aligned = (((uintptr_t)g.T) & 15) == 0;
  for (uint64_t p0 = 16ull * w.tid; p0 < s; p0 += 16ull * w.n) {
    if (p0 >= *(volatile unsigned long long*)&C.qs->lo_tail) return;
    uint32_t w[5];
    if (aligned && p0 + 20 <= g.n) {
      const uint4 v = *(const uint4*)(g.T + p0);
      w[0] = v.x, w[1] = v.y, w[2] = v.z, w[3] = v.w;
      w[4] = *(const uint32_t*)(g.T + p0 + 16);
    } else {
#pragma unroll
      for (int q = 0; q < 5; q++) {
        w[q] = 0;
        for (int t = 0; t < 4; t++)
          if (p0 + 4 * q + t < g.n) w[q] |= (uint32_t)g.T[p0 + 4 * q + t] << (8 * t);
      }
    }
#pragma unroll
    for (uint32_t i = 0; i < 16; i++) {
      if ((__funnelshift_r(w[i >> 2], w[(i >> 2) + 1], 8 * (i & 3)) & fm) != want) continue;
      const uint64_t p = p0 + i;
      if (p >= s) break;
      bool eq = true;
      for (uint64_t t = f; t < r && eq; t++) eq = g.T[p + t] == g.T[s + t];
      if (eq) {
        c_min(&C.qs->lo_tail, p);
        break;
      }
    }
  }
}

// An open key's leftmost fingerprint match.
__device__ __forceinline__ uint64_t item_lo(const Chase& C, uint64_t i, uint64_t* k, uint64_t* s, uint64_t* len) {
  const QGeo& g = C.g;
  const uint32_t it = C.items[i], sl = C.islot[i];
  const bool pair = it & 1;
  *k = it >> 1;
  *s = g.st[*k];
  *len = g.n - *s < g.b ? g.n - *s : g.b;
  if (pair) *len += g.n - *s - *len < g.b ? g.n - *s - *len : g.b;
  if (sl == kNoSlot) return *s;
  return sl == kTailItem ? (pair ? C.qs->lo_tailpair : C.qs->lo_tail) : pair ? C.pt[sl].lo : C.bt[sl].lo;
}

__device__ __forceinline__ void chase_verify(const Chase& C, uint64_t ppk, unsigned L, Span w) {
  const QGeo& g = C.g;
  const unsigned lane = threadIdx.x & 31, grp = lane / L, gl = lane % L, gpw = 32 / L;
  const unsigned gmask = (L == 32 ? 0xFFFFFFFFu : ((1u << L) - 1u)) << (grp * L);
  const bool aligned16 = (((uintptr_t)g.T) & 15) == 0;
  const uint64_t warps = w.n / 32, total = C.nitems * ppk, piece = q_piece(g.b);
  for (uint64_t base = w.tid / 32 * gpw; base < total; base += warps * gpw) {
    const uint64_t u = base + grp;
    bool d = false;
    uint64_t i = 0;
    if (u < total) {
      i = u / ppk;
      const uint64_t off = (u - i * ppk) * piece;
      uint64_t k, s, len;
      const uint64_t p = item_lo(C, i, &k, &s, &len);
      if (p < s && off < len)
        d = differs(g.T, g.n, aligned16, p, s, off, off + piece < len ? off + piece : len, gl, L);
    }
    const unsigned bal = __ballot_sync(0xFFFFFFFFu, d);
    if (u < total && gl == 0 && (bal & gmask)) C.differ[i] = 1;
  }
}

__device__ __forceinline__ void chase_apply(const Chase& C, Span w) {
  uint64_t vb = 0;
  for (uint64_t i = w.tid; i < C.nitems; i += w.n) {
    uint64_t k, s, len;
    const uint64_t p = item_lo(C, i, &k, &s, &len);
    const bool pair = C.items[i] & 1;
    if (p > s) {
      atomicExch(&C.status->error, 25ull);
      continue;
    }
    if (p < s) vb += 2 * len;
    if (p < s && C.differ[i]) {  // a fingerprint collision: resolved exactly
      atomicAdd(&C.status->collisions, 1ull);
      const unsigned long long q = atomicAdd(&C.qs->nsusp, 1ull);
      C.susp[q] = (uint32_t)i;
      C.exlo[q] = s;
    } else if (pair) {
      C.ps[k] = kIsPair | (p == s ? kLeftmost : 0);
    } else {
      C.lo[k] = p;
    }
  }
  vb = warp_sum64(vb);
  if ((threadIdx.x & 31) == 0 && vb) atomicAdd(&C.status->verify_bytes, (unsigned long long)vb);
}

// Exact leftmost occurrence of the keys whose match was false: every earlier
// position, byte by byte (a test modulus makes this frequent; with 2^61 - 1 it
// does not happen).
__device__ __forceinline__ void chase_exact(const Chase& C, uint64_t q0, uint64_t qstep, uint64_t nsusp, Span w) {
  for (uint64_t q = q0; q < nsusp; q += qstep) {
    uint64_t k, s, len;
    item_lo(C, C.susp[q], &k, &s, &len);
    for (uint64_t p = w.tid; p < s; p += w.n) {
      bool eq = true;
      for (uint64_t t = 0; t < len && eq; t++) eq = C.g.T[p + t] == C.g.T[s + t];
      if (eq) c_min(&C.exlo[q], p);
    }
  }
}

__device__ __forceinline__ void chase_exact_apply(const Chase& C, uint64_t nsusp, Span w) {
  for (uint64_t q = w.tid; q < nsusp; q += w.n) {
    uint64_t k, s, len;
    item_lo(C, C.susp[q], &k, &s, &len);
    if (C.items[C.susp[q]] & 1) C.ps[k] = kIsPair | (C.exlo[q] == s ? kLeftmost : 0);
    else C.lo[k] = C.exlo[q];
  }
}

}  // namespace bt
