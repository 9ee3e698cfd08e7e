// bt_batch.cu -- batched construction: a persistent, level-synchronous kernel
// with a per-document work queue.
//
// Each CTA (or, for few long documents, each cluster of CTAs) of k_batch
// repeatedly takes the next document of the batch from a device work queue (an
// atomic counter; the documents come in decreasing expected work, length times
// levels) and builds its whole block tree by itself:
//
//   1. alphabet (byte histogram -> dense symbol map, sigma check);
//   2. Karp-Rabin prefix fingerprints H(32 j) (section 2, the all-prefix form of
//      section 4.1) and the list of selected grams with the distances to their
//      first occurrences (bt_quick.cu);
//   3. for every level (section 3) of blocks of 27 bytes or more the steps of
//      bt_quick.cu over the CTA: bounds from the list, byte comparisons, and a
//      search of the list for the keys left open; for shorter blocks block and
//      pair fingerprints in open-addressing tables and a scan of every window
//      (section 3.1), byte verification of every accepted minimum with an
//      exact rescan of a key whose fingerprint collided.  Then marks (a pair is
//      marked when its leftmost occurrence is its own start, a block in no pair
//      is marked), back-pointers (ptr, off), and the tau-way split of marked
//      blocks into the next level;
//   4. the pruning post-pass (section 3.1, "Optional Pruning"), with the same
//      four conditions and the same right-to-left rule as the standard path,
//      resolved by frontier rounds over the candidates;
//   5. the rank/select counters, level-1 prefix counts and leaf text, written
//      with the tree's arrays into a region of the batch's output pool taken
//      with one atomic add.
//
// Between steps the CTA (or cluster) meets at a barrier; nothing waits on
// another document's CTAs, on another launch or on the host.  The tree of every document is the one
// bt_build_ex builds for it alone: the same readings of the paper, the same
// sizing, marking, pointer and pruning rules, every match verified.
#include <algorithm>
#include <atomic>
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <functional>
#include <memory>
#include <mutex>
#include <queue>
#include <thread>
#include <vector>

#include <chrono>

#include "bt_batch.cuh"
#include "bt_prune_dev.cuh"
#include "bt_quick_dev.cuh"

namespace bt {

int plan_sizes(uint64_t n, uint32_t tau, uint32_t leaf, const bt_opts& o, std::vector<uint64_t>& b);
uint64_t base_for(uint64_t seed, uint64_t q);
unsigned device_sm_count();

namespace {

constexpr uint32_t kBTailPair = 0xFFFFFFFEu;
constexpr uint32_t kMaxBThreads = 1024;
// 32-bit words of dynamic shared memory: the open keys' queues and bitmap, the
// window filter, the counters' histograms (1024 words a warp) and tiles, one
// after the other.
constexpr uint32_t dyn_words_of(uint32_t threads) { return 32 * threads; }

struct __align__(32) BSlot {
  unsigned long long key, lo, maxpst, pad;
};
struct __align__(16) PSlot {
  unsigned long long key, lo;
};
struct BJob {
  uint64_t a, b, len, idx;
};


constexpr uint32_t kMaxGroup = 16;  // CTAs of a cluster that share a document

// State that all CTAs of a group change.
struct Common {
  uint32_t doc;
  int err;
  uint32_t seen[8];                 // which bytes occur
  uint64_t part[kMaxGroup];         // one value per CTA (sums over its part of the text)
  unsigned long long fp_tail, lo_tail, lo_tailpair;
  uint32_t pretail;
  unsigned int npairs, njobs, nsusp;
  QuickStatus qs;
  Status status;
  unsigned long long verify_bytes, collisions;
  unsigned long long lastk;
  PruneShared prune;
  unsigned long long out_off;
};

static_assert(sizeof(Common) <= kCommonBytes, "a cluster's common state fits its place in the scratch");

// Where it is: in shared memory for one CTA, at the start of a cluster's scratch
// otherwise (64-bit minima and maxima are no native operations on another CTA's
// shared memory).
template <class GRP>
struct CommonOf;
template <>
struct CommonOf<One> {
  Common own;
  __device__ Common& common() { return own; }
};
template <>
struct CommonOf<Cluster> {
  Common* g;
  __device__ Common& common() { return *g; }
};

// State of a CTA; what is not scratch of its own is the same in all CTAs of the
// group, which each compute it from the same arrays.
template <class GRP>
struct Cta : CommonOf<GRP> {
  GRP grp;
  int bad;
  uint64_t n;
  uint32_t S, L;
  int16_t sym[256];
  unsigned int hist[256];
  ScratchLayout sl;
  uint64_t c[kBMaxLevels];
  uint64_t nmarked[kBMaxLevels];
  uint32_t arity[kBMaxLevels];
  uint64_t stats[kBMaxLevels][BT_ST_FIELDS];
  uint64_t last_start;
  // current level
  uint64_t r, Bb, Br;
  uint32_t bshift;
  uint32_t nsel;                      // entries of the list of selected grams
  int expanded;                       // H holds every position (the list is gone)
  QList list;
  Chase chase;
  // scans
  uint32_t wtot[kScanWords];
  uint64_t wsum[32];
  uint64_t carry;
  // output
  uint64_t out_off, out_bytes;
  // phase timing (SM cycles)
  unsigned long long cyc[6];
  long long t_mark;
};

// Adds the cycles since the last mark to phase `ph` (thread 0; call right
// after a barrier).
template <class GRP>
__device__ __forceinline__ void tmark(Cta<GRP>& C, int ph) {
  if (threadIdx.x == 0) {
    const long long t = clock64();
    C.cyc[ph] += (unsigned long long)(t - C.t_mark);
    C.t_mark = t;
  }
}

template <class GRP>
__device__ __forceinline__ void fail(Cta<GRP>& C, int code) { atomicCAS(&C.common().err, 0, code); }
// Barrier of the group; has a step failed?  (Two barriers in a cluster: no
// later step's failure may be seen by some of its CTAs only.)
template <class GRP>
__device__ __forceinline__ bool failed(Cta<GRP>& C) {
  if (!GRP::many) return __syncthreads_or(C.common().err != 0) != 0;
  gsync(C.grp);
  const int e = *(volatile int*)&C.common().err;
  gsync(C.grp);
  return e != 0;
}

__device__ __forceinline__ void min_pos(unsigned long long* a, uint64_t p) {
  if (*(volatile unsigned long long*)a > p) atomicMin(a, (unsigned long long)p);
}
// The same without the read: an atomic whose result is not used (a reduction
// the thread does not wait for), for the scan's frequent hits.
__device__ __forceinline__ void red_min(unsigned long long* a, uint64_t p) { atomicMin(a, (unsigned long long)p); }

template <class M>
__device__ __forceinline__ uint64_t phi(const M& m, const uint64_t* __restrict__ H, uint64_t BL, uint64_t p,
                                        uint64_t len) {
  return m.sub(H[p + len], m.mul(H[p], BL));
}

template <class Slot>
__device__ __forceinline__ uint32_t t_insert(Slot* t, uint64_t mask, uint64_t key) {
  uint64_t h = mix64(key) & mask;
  for (uint64_t it = 0; it <= mask; it++) {
    unsigned long long old = *(volatile unsigned long long*)&t[h].key;
    if (old == kNone) old = atomicCAS(&t[h].key, (unsigned long long)kNone, (unsigned long long)key);
    if (old == kNone || old == key) return (uint32_t)h;
    h = (h + 1) & mask;
  }
  return kNoSlot;
}

template <class Slot>
__device__ __forceinline__ uint32_t t_find(const Slot* t, uint64_t mask, uint64_t key) {
  uint64_t h = mix64(key) & mask;
  for (uint64_t it = 0; it <= mask; it++) {
    const uint64_t k = t[h].key;
    if (k == key) return (uint32_t)h;
    if (k == kNone) return kNoSlot;
    h = (h + 1) & mask;
  }
  return kNoSlot;
}

// ---------------------------------------------------------------------------
// Level geometry.
// ---------------------------------------------------------------------------
struct LV {
  const uint8_t* T;
  uint64_t n, c, b;
  uint64_t* st;
};

__device__ __forceinline__ uint64_t blen(const LV& g, uint64_t k) {
  const uint64_t s = g.st[k];
  return g.n - s < g.b ? g.n - s : g.b;
}

// End of block k and of up to two following blocks consecutive with it.
__device__ __forceinline__ uint64_t avail_end(const LV& g, uint64_t k) {
  uint64_t e = g.st[k] + blen(g, k);
  if (k + 1 < g.c && g.st[k + 1] == e) {
    e += blen(g, k + 1);
    if (k + 2 < g.c && g.st[k + 2] == e) e += blen(g, k + 2);
  }
  return e;
}

// 16 bytes of T starting at any x, from the two aligned 16-byte units that
// cover them (the text buffer is padded, so the second unit is readable).
__device__ __forceinline__ uint4 load16u(const uint8_t* __restrict__ T, uint64_t x) {
  const uint64_t x0 = x & ~15ull;
  const uint32_t d = (uint32_t)(x & 15);
  const uint4 u0 = *(const uint4*)(T + x0);
  if (d == 0) return u0;
  const uint4 u1 = *(const uint4*)(T + x0 + 16);
  const uint32_t q = d >> 2, sh = 8 * (d & 3);
  const uint32_t w[8] = {u0.x, u0.y, u0.z, u0.w, u1.x, u1.y, u1.z, u1.w};
  uint32_t o[5];
#pragma unroll
  for (int i = 0; i < 5; i++) o[i] = w[(q + i) & 7];
  return make_uint4(__funnelshift_r(o[0], o[1], sh), __funnelshift_r(o[1], o[2], sh),
                    __funnelshift_r(o[2], o[3], sh), __funnelshift_r(o[3], o[4], sh));
}

// Do T[a, a+len) and T[b, b+len) differ?  G lanes (lane gl of them) compare
// 16 bytes each per step.
__device__ __forceinline__ bool differs(const uint8_t* __restrict__ T, uint64_t a, uint64_t b, uint64_t len,
                                        unsigned gl, unsigned G) {
  bool diff = false;
  for (uint64_t y = 16ull * gl; y < len; y += 16ull * G) {
    const uint4 va = load16u(T, a + y), vb = load16u(T, b + y);
    const uint64_t cnt = len - y < 16 ? len - y : 16;
    const uint32_t xa[4] = {va.x ^ vb.x, va.y ^ vb.y, va.z ^ vb.z, va.w ^ vb.w};
#pragma unroll
    for (int q = 0; q < 4; q++) {
      const uint64_t lo = 4ull * q;
      if (lo >= cnt) break;
      const uint32_t mk = cnt - lo >= 4 ? kFull : ((1u << (8 * (cnt - lo))) - 1u);
      diff |= (xa[q] & mk) != 0;
    }
  }
  return diff;
}

// Verify jobs[0, nj): mismatch[i] = 1 when the two ranges differ.  Groups of
// G lanes (about len/16, a power of two up to 32) take one job each.
template <class GRP>
__device__ void verify_jobs(const uint8_t* __restrict__ T, const BJob* jobs, uint32_t nj, uint64_t maxlen,
                            unsigned int* mismatch, const GRP& grp_) {
  unsigned G = 1;
  while (G < 32 && 16ull * G < maxlen) G <<= 1;
  const unsigned lane = threadIdx.x & 31, grp = lane / G, gl = lane % G, gpw = 32 / G;
  const unsigned gmask = (G == 32 ? kFull : ((1u << G) - 1u)) << (grp * G);
  const unsigned nw = grp_.threads() >> 5, warp = grp_.tid() >> 5;
  // Warp-uniform loop: every lane reaches every ballot.
  for (uint64_t base = (uint64_t)warp * gpw; base < nj; base += (uint64_t)nw * gpw) {
    const uint64_t j = base + grp;
    bool diff = false;
    if (j < nj) {
      const BJob J = jobs[j];
      diff = differs(T, J.a, J.b, J.len, gl, G);
    }
    const unsigned bal = __ballot_sync(kFull, diff);
    if (j < nj && gl == 0) mismatch[j] = (bal & gmask) ? 1u : 0u;
  }
}

// ---------------------------------------------------------------------------
// Document set-up: alphabet and prefix fingerprints.
// ---------------------------------------------------------------------------
// (Only which bytes occur matters: after a document's first lines every mark
// is set, and looking costs no atomics and no conflicts on frequent bytes.)
template <class GRP>
__device__ void alphabet(const uint8_t* __restrict__ T, uint64_t n, uint32_t sigma, Cta<GRP>& C) {
  volatile unsigned int* seen = C.hist;
  const unsigned tid = C.grp.tid(), nt = C.grp.threads(), t = threadIdx.x;
  for (uint32_t i = t; i < 256; i += blockDim.x) seen[i] = 0;
  __syncthreads();
  const uint64_t nv = n / 16;
  for (uint64_t i = tid; i < nv; i += nt) {
    const uint4 q = ((const uint4*)T)[i];
    const uint32_t w[4] = {q.x, q.y, q.z, q.w};
    uint32_t f[16];
#pragma unroll
    for (int a = 0; a < 16; a++) f[a] = seen[(w[a >> 2] >> (8 * (a & 3))) & 0xFF];
#pragma unroll
    for (int a = 0; a < 16; a++)
      if (!f[a]) seen[(w[a >> 2] >> (8 * (a & 3))) & 0xFF] = 1;
  }
  for (uint64_t i = nv * 16 + tid; i < n; i += nt) seen[T[i]] = 1;
  __syncthreads();
  if (t < 256) {
    const uint32_t bits = __ballot_sync(kFull, seen[t] != 0);
    if ((t & 31) == 0 && bits) atomicOr(&C.common().seen[t >> 5], bits);
  }
  gsync(C.grp);
  if (t < 256) {
    uint32_t before = 0, all = 0, mine = 0;
    for (uint32_t w = 0; w < 8; w++) {
      const uint32_t bits = *(volatile uint32_t*)&C.common().seen[w];
      if (w < t >> 5) before += __popc(bits);
      if (w == t >> 5) mine = bits;
      all += __popc(bits);
    }
    C.sym[t] = (mine >> (t & 31)) & 1u ? (int16_t)(before + __popc(mine & ((1u << (t & 31)) - 1u))) : (int16_t)-1;
    if (t == 0) {
      C.S = all;
      if (all > sigma) fail(C, BT_EINVAL);
    }
  }
}

// Hs[j] = H(32 j) for j <= n / 32: four chunks of 32 bytes per thread, their
// byte dot products scanned over the CTA (as the prefix kernels of bt_scan.cu).
// A CTA takes the chunks [j0, j1) after the ones whose fingerprint is `carry`;
// returns (in C.carry) the fingerprint up to j1, a multiple of four chunks on,
// or, with `store`, writes Hs.
template <class M, class GRP>
__device__ void prefix_range(const M& m, const PrefixConst<M>& PC, const KrPow& pw, const uint8_t* T, uint64_t nchunks,
                             uint64_t r0, uint64_t r1, uint64_t carry0, bool store, uint64_t* Hs, Cta<GRP>& C) {
  if (threadIdx.x == 0) C.carry = carry0;
  __syncthreads();
  const uint64_t xl = kr_lane_pow(m, pw);
  for (uint64_t t0 = r0; t0 < r1; t0 += 4ull * blockDim.x) {
    const uint64_t j0 = t0 + 4ull * threadIdx.x;
    const unsigned last = (unsigned)((r1 - t0 < 4ull * blockDim.x ? r1 - t0 : 4ull * blockDim.x) + 3) / 4 - 1;
    uint64_t c[4];
#pragma unroll
    for (int i = 0; i < 4; i++) {
      uint32_t w[8];
      load_chunk(T, nchunks, j0 + i, true, w);
      c[i] = PC.hash(m, w);
    }
    uint64_t h = c[0];
#pragma unroll
    for (int i = 1; i < 4; i++) h = m.add(m.mul(h, PC.B32), c[i]);
    const uint64_t carry = C.carry;
    if (threadIdx.x == 0) h = m.add(m.mul(carry, pw.x[0]), h);
    const uint64_t incl = cta_kr_scan(m, h, pw, xl, C.wsum);
    uint64_t up = __shfl_up_sync(kFull, incl, 1);
    if ((threadIdx.x & 31) == 31) C.wsum[threadIdx.x >> 5] = incl;
    if (threadIdx.x == last) C.carry = incl;
    __syncthreads();
    if (store) {
      if ((threadIdx.x & 31) == 0) up = threadIdx.x ? C.wsum[(threadIdx.x >> 5) - 1] : carry;
#pragma unroll
      for (int i = 0; i < 4; i++) {
        if (j0 + i < r1) Hs[j0 + i] = up;
        up = m.add(m.mul(up, PC.B32), c[i]);
      }
    }
    __syncthreads();
  }
}

// In a cluster each CTA takes an equal part of the text: its fingerprint, then
// the parts before it, then its values.
template <class M, class GRP>
__device__ void prefix_pass(const M& m, const PrefixConst<M>& PC, const KrPow& pw, const uint8_t* T, uint64_t n,
                            uint64_t* Hs, Cta<GRP>& C) {
  const uint64_t nchunks = n / 32, all = nchunks + 1;
  if constexpr (!GRP::many) {
    prefix_range(m, PC, pw, T, nchunks, 0, all, 0, true, Hs, C);
  } else {
    const uint64_t per = (all + 4 * C.grp.size - 1) / (4 * C.grp.size) * 4;
    const uint64_t r0 = per * C.grp.rank < all ? per * C.grp.rank : all, r1 = r0 + per < all ? r0 + per : all;
    prefix_range(m, PC, pw, T, nchunks, r0, r1, 0, false, Hs, C);
    if (threadIdx.x == 0) C.common().part[C.grp.rank] = C.carry;
    gsync(C.grp);
    uint64_t carry = 0;
    if (threadIdx.x == 0) {
      const uint64_t x = pow_mod(m, PC.B32, per);
      for (uint32_t k = 0; k < C.grp.rank; k++) carry = m.add(m.mul(carry, x), *(volatile uint64_t*)&C.common().part[k]);
    }
    prefix_range(m, PC, pw, T, nchunks, r0, r1, carry, true, Hs, C);
    gsync(C.grp);
  }
}

// H[p] for every p in [0, n] (levels of blocks too short for the list).
template <class M, class GRP>
__device__ void expand_pass(const M& m, const uint8_t* T, uint64_t n, uint64_t B, const uint64_t* Hs, uint64_t* H,
                            const GRP& grp) {
  for (uint64_t j = grp.tid(); j <= n / 32; j += grp.threads()) {
    uint64_t h = Hs[j];
    for (uint64_t p = 32 * j; p < 32 * j + 32 && p <= n; p++) {
      H[p] = h;
      if (p < n) h = m.add(m.mul(h, B), (uint64_t)T[p] + 1);
    }
  }
  gsync(grp);
}

// Exclusive sum of one value per thread over the CTA; *total = the sum.
template <class GRP>
__device__ uint32_t cta_excl_u32(uint32_t v, Cta<GRP>& C, uint32_t* total) {
  const unsigned lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  uint32_t x = v;
#pragma unroll
  for (int d = 1; d < 32; d <<= 1) {
    const uint32_t o = __shfl_up_sync(kFull, x, d);
    if ((int)lane >= d) x += o;
  }
  if (lane == 31) C.wtot[warp] = x;
  __syncthreads();
  if (warp == 0) {
    uint32_t w = lane < nw ? C.wtot[lane] : 0u;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      const uint32_t o = __shfl_up_sync(kFull, w, d);
      if ((int)lane >= d) w += o;
    }
    C.wtot[lane] = w;
  }
  __syncthreads();
  const uint32_t r = (warp ? C.wtot[warp - 1] : 0u) + x - v;
  *total = C.wtot[nw - 1];
  __syncthreads();
  return r;
}

// The list of selected grams (bt_quick.cu): a thread takes 32 positions of a
// tile, the entries' places come from a CTA scan, then the first-occurrence
// table, the distances and the segment minima.  In a cluster each CTA takes an
// equal part of the text: it marks and counts its entries first (the marks wait
// in the first-occurrence table's place).
template <class GRP>
__device__ void list_pass(const uint8_t* T, uint64_t n, char* scr, Cta<GRP>& C) {
  const unsigned tid = C.grp.tid(), nt = C.grp.threads(), lane = tid & 31;
  const uint64_t nw = n < kGramLen ? 0 : (n - kGramLen + 1 + 31) / 32, ns = (n + kSegBytes - 1) / kSegBytes,
                 ns2 = (ns + 63) / 64;
  uint32_t* idx = (uint32_t*)(scr + C.sl.idx);
  uint32_t* x = (uint32_t*)(scr + C.sl.big);
  uint32_t* D = x + ((n + 63) & ~63ull);
  uint32_t* first = (uint32_t*)(scr + C.sl.first);
  uint32_t* seg1 = (uint32_t*)(scr + C.sl.seg1);
  uint32_t* seg2 = (uint32_t*)(scr + C.sl.seg2);
  const uint32_t cmask = (uint32_t)(C.sl.cells - 1);
  auto mask = [&](uint64_t j) {
    uint32_t bits = half_mask(T, n, 32 * j) | half_mask(T, n, 32 * j + 16) << 16;
    const uint64_t left = n - kGramLen + 1 - 32 * j;
    if (left < 32) bits &= (1u << left) - 1u;
    return bits;
  };
  constexpr bool multi = GRP::many;
  const uint64_t per = (nw + C.grp.size - 1) / C.grp.size, a0 = per * C.grp.rank < nw ? per * C.grp.rank : nw,
                 a1 = a0 + per < nw ? a0 + per : nw;
  uint32_t total = 0, all = 0;
  if constexpr (multi) {
    uint32_t mine = 0, sum;
    for (uint64_t j = a0 + threadIdx.x; j < a1; j += blockDim.x) {
      const uint32_t bits = mask(j);
      first[j] = bits;
      mine += __popc(bits);
    }
    cta_excl_u32(mine, C, &sum);
    if (threadIdx.x == 0) C.common().part[C.grp.rank] = sum;
    gsync(C.grp);
    for (uint32_t k = 0; k < C.grp.size; k++) {
      const uint32_t x = (uint32_t)*(volatile uint64_t*)&C.common().part[k];
      if (k < C.grp.rank) total += x;
      all += x;
    }
  } else {
    for (uint64_t i = tid; i < C.sl.cells; i += nt) first[i] = 0xFFFFFFFFu;
  }
  for (uint64_t j0 = a0; j0 < a1; j0 += blockDim.x) {
    const uint64_t j = j0 + threadIdx.x;
    uint32_t bits = j < a1 ? (multi ? first[j] : mask(j)) : 0u;
    uint32_t sum;
    uint32_t o = total + cta_excl_u32(__popc(bits), C, &sum);
    if (j < a1) idx[j] = o;
    for (; bits; bits &= bits - 1, o++) {
      const uint32_t p = (uint32_t)(32 * j) + __ffs(bits) - 1, sh = 8 * (p & 3);
      const uint32_t* w = (const uint32_t*)(T + (p & ~3u));
      const uint32_t w0 = w[0], w1 = w[1], w2 = w[2], w3 = w[3], w4 = w[4];
      x[o] = p;
      D[o] = gram_cell(__funnelshift_r(w0, w1, sh), __funnelshift_r(w1, w2, sh), __funnelshift_r(w2, w3, sh),
                       __funnelshift_r(w3, w4, sh), cmask);
    }
    total += sum;
  }
  if (multi) {
    gsync(C.grp);
    for (uint64_t i = tid; i < C.sl.cells; i += nt) first[i] = 0xFFFFFFFFu;
    total = all;
  }
  if (tid == 0) idx[nw] = total;
  if (threadIdx.x == 0) {
    C.nsel = total;
    C.list = QList{idx, x, D, seg1, seg2, nw};
  }
  gsync(C.grp);
  for (uint32_t e = tid; e < total; e += 4 * nt) {
    uint32_t c[4], f[4];
#pragma unroll
    for (uint32_t u = 0; u < 4; u++) c[u] = e + u * nt < total ? D[e + u * nt] : 0;
#pragma unroll
    for (uint32_t u = 0; u < 4; u++) f[u] = *(volatile uint32_t*)&first[c[u]];
#pragma unroll
    for (uint32_t u = 0; u < 4; u++)
      if (e + u * nt < total && f[u] > x[e + u * nt]) atomicMin(&first[c[u]], x[e + u * nt]);
  }
  gsync(C.grp);
  for (uint32_t e = tid; e < total; e += 4 * nt) {
    uint32_t f[4];
#pragma unroll
    for (uint32_t u = 0; u < 4; u++) f[u] = e + u * nt < total ? *(volatile uint32_t*)&first[D[e + u * nt]] : 0;
#pragma unroll
    for (uint32_t u = 0; u < 4; u++)
      if (e + u * nt < total) D[e + u * nt] = x[e + u * nt] - f[u];
  }
  gsync(C.grp);
  for (uint64_t j = tid / 32; j < ns; j += nt / 32) {
    const uint64_t w0 = j * (kSegBytes / 32), w1 = w0 + kSegBytes / 32 < nw ? w0 + kSegBytes / 32 : nw;
    const uint32_t d = __reduce_min_sync(kFull, min_entries(D, idx[w0 < nw ? w0 : nw], idx[w1], lane, 32, kNoDist));
    if (lane == 0) seg1[j] = d;
  }
  gsync(C.grp);
  for (uint64_t j = tid; j < ns2; j += nt) {
    uint32_t d = kNoDist;
    for (uint64_t i = 64 * j; i < 64 * j + 64 && i < ns; i++) d = min(d, seg1[i]);
    seg2[j] = d;
  }
  gsync(C.grp);
}

struct Work {
  uint64_t *fpB, *job_of, *susp, *exBL;
  unsigned long long* exlo;
  uint32_t *slotB, *slotP, *wpop;
  unsigned int* mismatch;
  uint8_t* pm;
  BJob* jobs;
  BSlot* bt;
  PSlot* pt;
};

__device__ Work carve_level(char* temp, uint64_t c, uint64_t bcap, uint64_t pcap) {
  Work W;
  char* p = temp;
  W.fpB = (uint64_t*)carve(p, c * 8 + 8);
  W.exBL = (uint64_t*)carve(p, c * 8 + 8);  // (the unused pair-lo slot of the layout)
  W.job_of = (uint64_t*)carve(p, c * 8 + 8);
  W.susp = (uint64_t*)carve(p, c * 8 + 8);
  W.exlo = (unsigned long long*)carve(p, c * 8 + 8);
  W.slotB = (uint32_t*)carve(p, c * 4 + 4);
  W.slotP = (uint32_t*)carve(p, c * 4 + 4);
  W.mismatch = (unsigned int*)carve(p, c * 4 + 4);
  W.wpop = (uint32_t*)carve(p, c * 4 + 4);
  W.pm = (uint8_t*)carve(p, c + 8);
  W.jobs = (BJob*)carve(p, c * 32 + 32);
  carve(p, c * 8 + 8);
  W.bt = (BSlot*)carve(p, bcap * 32);
  W.pt = (PSlot*)carve(p, pcap * 16);
  return W;
}

// Exact leftmost occurrence of every suspect key (a fingerprint collision
// was found by verification): every window before the key's start, inside a
// run, whose fingerprint equals the key's is compared byte by byte.
template <class M, class GRP>
__device__ void exact_pass(const M& m, const LV& g, const uint64_t* H, const Work& W, int pair, uint64_t B,
                           Cta<GRP>& C) {
  const uint32_t ns = C.common().nsusp;
  // Key fingerprint, length and B^length of each suspect (in the job array).
  for (uint32_t i = C.grp.tid(); i < ns; i += C.grp.threads()) {
    const uint64_t k = W.susp[i];
    uint64_t klen = blen(g, k), kfp = W.fpB[k];
    if (pair) {
      const uint64_t l2 = blen(g, k + 1);
      kfp = m.add(m.mul(kfp, pow_mod(m, B, l2)), W.fpB[k + 1]);
      klen += l2;
    }
    W.jobs[i] = BJob{kfp, pow_mod(m, B, klen), klen, g.st[k]};
  }
  gsync(C.grp);
  const uint64_t per = g.c * g.b;
  for (uint64_t w = C.grp.tid(); w < (uint64_t)ns * per; w += C.grp.threads()) {
    const uint64_t i = w / per, rest = w - i * per;
    const uint64_t k = rest / g.b, j = rest - k * g.b;
    if (j >= blen(g, k)) continue;
    const BJob J = W.jobs[i];
    const uint64_t p = g.st[k] + j;
    if (p >= J.idx) continue;
    if (p + J.len > avail_end(g, k)) continue;
    if (phi(m, H, J.b, p, J.len) != J.a) continue;
    bool eq = true;
    for (uint64_t x = 0; x < J.len && eq; x++) eq = g.T[p + x] == g.T[J.idx + x];
    if (eq) min_pos(&W.exlo[i], p);
  }
  gsync(C.grp);
}

// A window of the scan whose fingerprint passed the filter: the block-table
// probe; for a match, the slot minimum, the pair that ends in the short tail,
// and the pair joined at p + b.  Out of line: matches are few, and the scan
// loop keeps its registers for the loads in flight.
struct ScanArgs {
  const uint64_t* H;
  BSlot* bt;
  PSlot* pt;
  uint64_t bmask, pmask, b, r, Bb, Br, fp_tail;
  uint32_t pretail;
  unsigned long long* lo_tailpair;
};

template <class M>
__device__ __forceinline__ void window_hit(const M& m, const ScanArgs& A, uint64_t p, uint64_t av, uint64_t x,
                                        uint64_t hb) {
  const uint32_t sl = t_find(A.bt, A.bmask, x);
  if (sl == kNoSlot) return;
  red_min(&A.bt[sl].lo, p);
  if (A.r && sl == A.pretail && p + A.b + A.r <= av && m.sub(A.H[p + A.b + A.r], m.mul(hb, A.Br)) == A.fp_tail)
    min_pos(A.lo_tailpair, p);
  if (p <= A.bt[sl].maxpst && p + 2 * A.b <= av) {
    const uint64_t fp2 = m.sub(A.H[p + 2 * A.b], m.mul(hb, A.Bb));
    const uint32_t s2 = t_find(A.bt, A.bmask, fp2);
    if (s2 != kNoSlot) {
      const uint32_t ps = t_find(A.pt, A.pmask, ((uint64_t)sl << 32) | s2);
      if (ps != kNoSlot) red_min(&A.pt[ps].lo, p);
    }
  }
}

// Marks and leftmost occurrences of a level of short blocks (fewer than
// kQuickMinB bytes), or of one whose search by grams was given up: fingerprint
// tables and a scan of every window.
template <class M, class GRP>
__device__ void scan_keys(const M& m, const BParams& P, const BDoc& D, Cta<GRP>& C, const LV& g, char* scr, uint32_t l,
                          uint32_t* filt, uint32_t filt_words_max) {
  const uint64_t n = C.n, c = g.c, b = g.b;
  const unsigned tid = C.grp.tid(), nt = C.grp.threads();
  uint64_t* lo = (uint64_t*)(scr + C.sl.lo[l]);
  uint32_t* mw = (uint32_t*)(scr + C.sl.mw[l]);
  uint32_t* mr = (uint32_t*)(scr + C.sl.mr[l]);
  uint64_t* H = (uint64_t*)(scr + C.sl.big);
  if (!C.expanded) {
    expand_pass(m, D.T, n, P.B, (const uint64_t*)(scr + C.sl.Hs), H, C.grp);
    if (threadIdx.x == 0) C.expanded = 1;
  }
  const uint64_t bcap = pow2_ge(2 * c), pcap = pow2_ge(2 * c);
  const Work W = carve_level(scr + C.sl.temp, c, bcap, pcap);
  if (tid == 0) C.common().npairs = 0;  // (a search that was given up counted them)
  for (uint64_t i = tid; i < bcap; i += nt) W.bt[i] = BSlot{kNone, kNone, 0, 0};
  for (uint64_t i = tid; i < pcap; i += nt) W.pt[i] = PSlot{kNone, kNone};
  for (uint64_t i = tid; i < c; i += nt) W.mismatch[i] = 0;
  gsync(C.grp);
  tmark(C, 3);
  const uint64_t r = C.r, Bb = C.Bb, Br = C.Br, bmask = bcap - 1, pmask = pcap - 1;

  // Block fingerprints; full-length blocks into the block table (the slot's
  // leftmost window starts at the block's own start).
  for (uint64_t k = tid; k < c; k += nt) {
    const uint64_t s = g.st[k], len = blen(g, k);
    const uint64_t fp = phi(m, H, len == b ? Bb : Br, s, len);
    W.fpB[k] = fp;
    if (len == b) {
      const uint32_t slot = t_insert(W.bt, bmask, fp);
      W.slotB[k] = slot;
      if (slot == kNoSlot) {
        fail(C, BT_EINTERNAL);
        continue;
      }
      min_pos(&W.bt[slot].lo, s);
    } else {
      W.slotB[k] = kNoSlot;
      C.common().fp_tail = fp;
      atomicMin(&C.common().lo_tail, (unsigned long long)s);
    }
  }
  if (failed(C)) return;
  // Pairs of consecutive blocks: one pair-table slot per (slot, slot); the
  // pair ending in the short tail is kept in the CTA's scalars.
  for (uint64_t k = tid; k + 1 < c; k += nt) {
    W.slotP[k] = kNoSlot;
    if (g.st[k + 1] != g.st[k] + b) continue;
    atomicAdd(&C.common().npairs, 1u);
    const uint32_t sk = W.slotB[k];
    if (sk == kNoSlot) {
      fail(C, BT_EINTERNAL);
      continue;
    }
    if (*(volatile unsigned long long*)&W.bt[sk].maxpst < g.st[k])
      atomicMax(&W.bt[sk].maxpst, (unsigned long long)g.st[k]);
    if (W.slotB[k + 1] == kNoSlot) {
      W.slotP[k] = kBTailPair;
      C.common().pretail = sk;
      atomicMin(&C.common().lo_tailpair, (unsigned long long)g.st[k]);
    } else {
      const uint32_t sp = t_insert(W.pt, pmask, ((uint64_t)sk << 32) | W.slotB[k + 1]);
      W.slotP[k] = sp;
      if (sp == kNoSlot) {
        fail(C, BT_EINTERNAL);
        continue;
      }
      min_pos(&W.pt[sp].lo, g.st[k]);
    }
  }
  if (failed(C)) return;
  uint32_t fwords = 32;
  while (fwords < c && fwords < filt_words_max) fwords <<= 1;
  // A bitmap of the full-length block fingerprints in shared memory (about
  // 32 bits per key): a window whose fingerprint's bit is clear matches no
  // key, so only the few that pass probe the table in global memory.
  const uint64_t fmask = (uint64_t)fwords * 32 - 1;
  // (every CTA has its own)
  for (uint32_t i = threadIdx.x; i < fwords; i += blockDim.x) filt[i] = 0;
  __syncthreads();
  for (uint64_t k = threadIdx.x; k < c; k += blockDim.x)
    if (W.slotB[k] != kNoSlot) {
      const uint64_t bit = W.fpB[k] & fmask;
      atomicOr(&filt[bit >> 5], 1u << (bit & 31));
    }
  gsync(C.grp);
  tmark(C, 1);

  // The window scan: every window [p, p+b) inside a run (and [p, p+r) for the
  // short tail); the few whose fingerprint's bit is set probe the table.
  {
    const uint32_t pretail = C.common().pretail, bshift = C.bshift;
    const uint64_t fp_tail = C.common().fp_tail;
    const ScanArgs A{H, W.bt, W.pt, bmask, pmask, b, r, Bb, Br, fp_tail, pretail, &C.common().lo_tailpair};
    for (uint64_t w = tid; w < c * b; w += nt) {
      const uint64_t k = bshift != 0xFFu ? w >> bshift : w / b;
      const uint64_t j = w - k * b;
      if (j >= blen(g, k)) continue;
      const uint64_t p = g.st[k] + j, av = avail_end(g, k);
      if (p + b <= av) {
        const uint64_t hb = H[p + b];
        const uint64_t x = m.sub(hb, m.mul(H[p], Bb));
        const uint64_t bit = x & fmask;
        if ((filt[bit >> 5] >> (bit & 31)) & 1u) window_hit(m, A, p, av, x, hb);
      }
      if (r && p + r <= av && phi(m, H, Br, p, r) == fp_tail) min_pos(&C.common().lo_tail, p);
    }
  }
  gsync(C.grp);
  tmark(C, 2);

  // Pairs: leftmost when the minimum is the pair's own start; otherwise the
  // earlier occurrence is verified.
  for (uint64_t k = tid; k + 1 < c; k += nt) {
    W.pm[k] = 0;
    W.job_of[k] = kNone;
    const uint32_t sp = W.slotP[k];
    if (sp == kNoSlot) continue;
    const uint64_t lp = sp == kBTailPair ? C.common().lo_tailpair : W.pt[sp].lo;
    const uint64_t s = g.st[k];
    if (lp == s) {
      W.pm[k] = 1;
    } else if (lp < s) {
      const uint64_t len = b + blen(g, k + 1);
      const uint32_t id = atomicAdd(&C.common().njobs, 1u);
      W.jobs[id] = BJob{lp, s, len, k};
      W.job_of[k] = id;
      atomicAdd(&C.common().verify_bytes, 2ull * len);
    } else {
      fail(C, BT_EINTERNAL);  // the pair's own window was not seen
    }
  }
  if (failed(C)) return;
  verify_jobs(g.T, W.jobs, C.common().njobs, 2 * b, W.mismatch, C.grp);
  gsync(C.grp);
  for (uint64_t k = tid; k + 1 < c; k += nt) {
    const uint64_t id = W.job_of[k];
    if (id == kNone || !W.mismatch[id]) continue;
    atomicAdd(&C.common().collisions, 1ull);
    const uint32_t i = atomicAdd(&C.common().nsusp, 1u);
    W.susp[i] = k;
    W.exlo[i] = g.st[k];
  }
  gsync(C.grp);
  if (C.common().nsusp) {
    exact_pass(m, g, H, W, 1, P.B, C);
    for (uint32_t i = tid; i < C.common().nsusp; i += nt) W.pm[W.susp[i]] = W.exlo[i] == g.st[W.susp[i]];
    gsync(C.grp);
  }

  // Marks: a block in a leftmost pair, or in no pair.
  const uint64_t words = (c + 31) / 32;
  {
    const unsigned lane = tid & 31, nw = nt >> 5;
    for (uint64_t wb = tid >> 5; wb < words; wb += nw) {
      const uint64_t k = wb * 32 + lane;
      bool mk = false;
      if (k < c) {
        const bool left = k > 0 && W.slotP[k - 1] != kNoSlot;
        const bool right = k + 1 < c && W.slotP[k] != kNoSlot;
        mk = (left && W.pm[k - 1]) || (right && W.pm[k]) || (!left && !right);
      }
      const uint32_t bits = __ballot_sync(kFull, mk);
      if (lane == 0) {
        mw[wb] = bits;
        W.wpop[wb] = __popc(bits);
      }
    }
  }
  gsync(C.grp);
  if (C.grp.rank == 0) cta_scan_u32(W.wpop, mr, words, C.wtot);
  if (GRP::many) gsync(C.grp);

  // Leftmost occurrence of every block that becomes a pointer (of every
  // block when pruning needs it), verified.
  if (tid == 0) {
    C.common().njobs = 0;
    C.common().nsusp = 0;
  }
  for (uint64_t i = tid; i < c; i += nt) W.mismatch[i] = 0;
  gsync(C.grp);
  for (uint64_t k = tid; k < c; k += nt) {
    W.job_of[k] = kNone;
    lo[k] = kNone;
    if (!P.prune && marked(mw, k)) continue;
    const uint64_t s = g.st[k], len = blen(g, k);
    const uint64_t p = W.slotB[k] == kNoSlot ? C.common().lo_tail : W.bt[W.slotB[k]].lo;
    lo[k] = p;
    if (p < s) {
      const uint32_t id = atomicAdd(&C.common().njobs, 1u);
      W.jobs[id] = BJob{p, s, len, k};
      W.job_of[k] = id;
      atomicAdd(&C.common().verify_bytes, 2ull * len);
    } else if (p > s) {
      fail(C, BT_EINTERNAL);
    }
  }
  if (failed(C)) return;
  verify_jobs(g.T, W.jobs, C.common().njobs, b, W.mismatch, C.grp);
  gsync(C.grp);
  for (uint64_t k = tid; k < c; k += nt) {
    const uint64_t id = W.job_of[k];
    if (id == kNone || !W.mismatch[id]) continue;
    atomicAdd(&C.common().collisions, 1ull);
    const uint32_t i = atomicAdd(&C.common().nsusp, 1u);
    W.susp[i] = k;
    W.exlo[i] = g.st[k];
  }
  gsync(C.grp);
  if (C.common().nsusp) {
    exact_pass(m, g, H, W, 0, P.B, C);
    for (uint32_t i = tid; i < C.common().nsusp; i += nt) lo[W.susp[i]] = W.exlo[i];
    gsync(C.grp);
  }
}

// Marks and leftmost occurrences of a level by first occurrences: the steps of
// bt_quick.cu over one CTA.  Measured on 1024 versioned documents of 4 KiB - 4
// MiB (0.65 GB): with fingerprint tables and a scan of every window (anchored
// on levels of 1 KiB blocks and more) the kernel took 50 ms, the longest
// document 51; now 15 and 15.
// False, the same for all threads: given up, the level goes by scan_keys.
template <class M, class GRP>
__device__ bool quick_keys(const M& m, const PrefixConst<M>& PC, Cta<GRP>& C, const LV& g, char* scr, uint32_t l,
                           uint32_t* dyn, uint32_t dyn_words) {
  const uint64_t n = C.n, c = g.c, b = g.b, words = (c + 31) / 32;
  const unsigned tid = C.grp.tid(), nt = C.grp.threads(), lane = tid & 31, warp = threadIdx.x >> 5,
                 nwarps = blockDim.x >> 5;
  uint64_t* lo = (uint64_t*)(scr + C.sl.lo[l]);
  uint32_t* mw = (uint32_t*)(scr + C.sl.mw[l]);
  uint32_t* mr = (uint32_t*)(scr + C.sl.mr[l]);
  char* p = scr + C.sl.temp;
  uint32_t* A = (uint32_t*)carve(p, c * 4 + 4);
  uint32_t* X = (uint32_t*)carve(p, c * 4 + 4);
  uint32_t* flags = (uint32_t*)carve(p, c * 4 + 4);
  uint32_t* wpop = (uint32_t*)carve(p, c * 4 + 4);
  uint32_t* items = (uint32_t*)carve(p, c * 8 + 8);
  uint8_t* ps = (uint8_t*)carve(p, c + 8);
  const QGeo q{g.T, n, c, b, g.st};
  const Span w{tid, nt};
  unsigned G = 1;
  while (G < 32 && 64ull * 2 * G <= b) G <<= 1;
  quick_min(q, C.list, G, A, X, flags, w);
  gsync(C.grp);
  tmark(C, 1);
  const uint64_t bl = b < n ? b : n;
  const uint32_t ppk = (uint32_t)((2 * bl + q_piece(b) - 1) / q_piece(b));
  const unsigned L = b >= 1024 ? 32u : b >= 512 ? 16u : b >= 256 ? 8u : b >= 128 ? 4u : b >= 64 ? 2u : 1u;
  quick_compare(q, A, X, flags, ppk, L, w);
  gsync(C.grp);
  tmark(C, 3);
  uint64_t vb = 0;
  uint32_t np = 0, nob = 0, nop = 0;
  for (uint64_t k = tid; k < c; k += nt) {
    const uint64_t s = g.st[k], len = blen(g, k);
    const uint32_t d = A[k];
    uint64_t at = s;
    bool open = false;
    if (s != 0 && d != 0) {
      open = d == kNoDist || (flags[k] & kBlkDiffers);
      at = open ? kNone : (d > s ? 0 : s - d);
      if (d != kNoDist) vb += 2 * len;
    }
    lo[k] = at;
    if (open) {
      items[atomicAdd(&C.common().qs.nitems, 1ull)] = (uint32_t)(2 * k);
      nob++;
    }
    uint32_t d2 = 0;
    uint64_t plen = 0;
    const uint8_t st = pair_state(q, A, X, flags, k, &d2, &plen, &open);
    ps[k] = st;
    np += st & kIsPair;
    if (st == kIsPair && d2 != kNoDist) vb += 2 * plen;
    if (open) {
      items[atomicAdd(&C.common().qs.nitems, 1ull)] = (uint32_t)(2 * k + 1);
      nop++;
    }
  }
  vb = warp_sum64(vb);
  np = __reduce_add_sync(kFull, np);
  nob = __reduce_add_sync(kFull, nob);
  nop = __reduce_add_sync(kFull, nop);
  if (lane == 0) {
    if (vb) atomicAdd(&C.common().status.verify_bytes, (unsigned long long)vb);
    if (np) atomicAdd(&C.common().npairs, np);
    if (nob) atomicAdd(&C.common().qs.nopen[0], (unsigned long long)nob);
    if (nop) atomicAdd(&C.common().qs.nopen[1], (unsigned long long)nop);
  }
  gsync(C.grp);
  tmark(C, 3);
  const uint64_t ni = C.common().qs.nitems;
  if (ni) {
    const uint64_t nb = C.common().qs.nopen[0] + 2 * C.common().qs.nopen[1];
    const uint64_t bcap = pow2_ge(2 * (nb < c ? nb : c)), pcap = pow2_ge(2 * C.common().qs.nopen[1]), gcap = pow2_ge(2 * ni);
    uint32_t fbits = 12;
    while ((1ull << fbits) < 16 * ni && fbits < 30) fbits++;
    const uint32_t bwords = 1u << (fbits - 5);
    if (threadIdx.x == 0) {
      Chase& K = C.chase;
      K.first = false;
      K.probes = probes_most(ni);
      K.g = q;
      K.Q = C.list;
      K.A = A;
      K.X = X;
      K.items = items;
      K.nitems = (uint32_t)ni;
      K.Bb = C.Bb;
      K.Br = C.Br;
      K.r = C.r;
      K.bt = (CSlot*)carve(p, bcap * 32);
      K.pt = (CPair*)carve(p, pcap * 16);
      K.gt = (CGram*)carve(p, gcap * 16);
      K.bound2 = (unsigned long long*)carve(p, gcap * 8);
      K.bitmap = (uint32_t*)carve(p, bwords * 4ull);
      K.islot = (uint32_t*)carve(p, ni * 4);
      K.igram = (uint32_t*)carve(p, ni * 4);
      K.differ = (uint32_t*)carve(p, ni * 4);
      K.susp = (uint32_t*)carve(p, ni * 4);
      K.exlo = (unsigned long long*)carve(p, ni * 8);
      K.bmask = (uint32_t)(bcap - 1);
      K.pmask = (uint32_t)(pcap - 1);
      K.gmask = (uint32_t)(gcap - 1);
      K.bshift = 32 - fbits;
      K.qs = &C.common().qs;
      K.status = &C.common().status;
      K.lo = lo;
      K.ps = ps;
    }
    __syncthreads();
    const Chase& K = C.chase;
    const PrefixAt<M> H(PC, g.T, n, (const uint64_t*)(scr + C.sl.Hs));
    // Shared memory: the warps' queues, then the bitmap while it fits.
    uint2* hq = (uint2*)dyn + warp * kHitQ;
    uint32_t* queues = (uint32_t*)((uint2*)dyn + nwarps * kHitQ);
    uint32_t* cq = queues + warp * kCandQ;
    uint8_t* gq = (uint8_t*)(queues + nwarps * kCandQ) + warp * kHitQ;
    uint32_t* bits_s = queues + nwarps * (kCandQ + kHitQ / 4);
    const bool fits = bwords <= dyn_words - nwarps * (2 * kHitQ + kCandQ + kHitQ / 4);
    const uint32_t* bits = fits ? bits_s : K.bitmap;
    // As for a single text (bt_quick.cu): the sample by newest grams, perhaps by
    // first grams too, then the rest by one of them, or every window.
    enum { kBySample, kByBoth, kByRest };
    const uint32_t total = C.nsel, split = total > (1u << 16) ? (total / 16) & ~(8 * kChaseTile - 1) : 0;
    // (The scan of every window costs a CTA more of these steps than it does the
    // whole GPU, so each bound is four times as high.  256 documents of 512 KiB, with
    // the bounds 1, 2, 4, 8 times as high and with none: 100 words 26, 19, 16, 16, 17
    // ms, random bits 22, 13, 13, 13, 14, two-letter runs 31, 32, 33, 54, 67, ten words
    // 45, 47, 56, 44, 45.)
    const uint64_t wn = 4 * n, least = least_work_cta(n), few = split ? work_few(wn) : work_most(wn, false, least);
    uint64_t limit = work_most(wn, split != 0, least), newest = 0, before = 0;
    uint32_t step = kBySample;
    bool enter = true;
    for (bool again = false;; again = true) {
      const bool rest = step == kByRest;
      if (enter) {
        chase_init(K, bwords, again, w);
        gsync(C.grp);
        if (b <= 256) chase_keys<M, 1>(m, H, K, w);
        else chase_keys<M, 32>(m, H, K, w);
        gsync(C.grp);
      }
      if (rest) {
        chase_bound(K, w);
        for (uint32_t i = tid; i < bwords; i += nt) K.bitmap[i] = 0;
        gsync(C.grp);
        chase_live(K, split, w);
        gsync(C.grp);
      }
      if (fits)
        for (uint32_t i = threadIdx.x; i < bwords; i += blockDim.x) bits_s[i] = K.bitmap[i];
      __syncthreads();
      chase_scan(m, H, K, K.first, rest ? split : 0, rest || !split ? total : split, bits, hq, gq, cq, rest ? K.bound2 : nullptr, limit,
                 kGiveUp, w);
      gsync(C.grp);
      const bool over = *(volatile unsigned int*)&K.qs->redo != kSearchDone;
      const uint64_t seen = *(volatile unsigned long long*)&K.qs->work;
      bool first = K.first;
      gsync(C.grp);
      if (step == kBySample && !over && (!split || seen <= work_sample(wn))) {
        if (!split) break;
        step = kByRest;
        enter = false;
      } else if (step == kBySample) {
        step = kByBoth;
        newest = over ? ~0ull : seen;
        first = enter = true;
      } else if (step == kByBoth) {
        const uint64_t by_first = over ? ~0ull : seen - before;
        if ((newest < by_first ? newest : by_first) > few) return false;
        if (!split) break;
        step = kByRest;
        enter = newest < by_first;
        first = !enter;
      } else {
        if (over) return false;
        break;
      }
      before = seen;
      limit = seen + (step == kByBoth ? few : work_most(wn, false, least));
      if (threadIdx.x == 0) {
        C.chase.first = first;
        C.chase.probes = ~0ull;
      }
      __syncthreads();
    }
    if (C.r && C.r < kQuickMinB) chase_tail(K, w);
    gsync(C.grp);
    tmark(C, 2);
    const unsigned Lv = b >= 256 ? 32u : b >= 128 ? 16u : b >= 64 ? 8u : 4u;
    chase_verify(K, (2 * b + q_piece(b) - 1) / q_piece(b), Lv, w);
    gsync(C.grp);
    chase_apply(K, w);
    gsync(C.grp);
    const uint64_t nsusp = C.common().qs.nsusp;
    if (nsusp) {
      chase_exact(K, 0, 1, nsusp, w);
      gsync(C.grp);
      chase_exact_apply(K, nsusp, w);
      gsync(C.grp);
    }
  }
  if (tid == 0 && C.common().status.error) fail(C, BT_EINTERNAL);  // (the level goes on; the caller looks at the end)
  for (uint64_t wb = tid >> 5; wb < words; wb += nt >> 5) {
    const uint64_t k = wb * 32 + lane;
    bool mk = false;
    if (k < c) {
      const uint8_t left = k ? ps[k - 1] : 0, r = ps[k];
      mk = (left & kLeftmost) || (r & kLeftmost) || !((left | r) & kIsPair);
    }
    const uint32_t bits = __ballot_sync(kFull, mk);
    if (lane == 0) {
      mw[wb] = bits;
      wpop[wb] = __popc(bits);
    }
  }
  gsync(C.grp);
  if (C.grp.rank == 0) cta_scan_u32(wpop, mr, words, C.wtot);
  if (GRP::many) gsync(C.grp);
  return true;
}

template <class M, class GRP>
__device__ void level_pass(const M& m, const PrefixConst<M>& PC, const BParams& P, const BDoc& D, Cta<GRP>& C, char* scr,
                           uint32_t l, uint32_t* dyn, uint32_t dyn_words) {
  const uint64_t* bsz = P.sizes + D.lv_off;
  const uint64_t n = C.n, c = C.c[l], b = bsz[l];
  const bool last = l + 1 == C.L;
  const unsigned tid = C.grp.tid(), nt = C.grp.threads();
  LV g{D.T, n, c, b, (uint64_t*)(scr + C.sl.st[l])};
  uint64_t* lo = (uint64_t*)(scr + C.sl.lo[l]);
  uint64_t* off = (uint64_t*)(scr + C.sl.off[l]);
  uint32_t* ptr = (uint32_t*)(scr + C.sl.ptr[l]);
  uint32_t* mw = (uint32_t*)(scr + C.sl.mw[l]);
  uint32_t* mr = (uint32_t*)(scr + C.sl.mr[l]);
  const uint64_t words = (c + 31) / 32;
  if (threadIdx.x == 0) {
    const uint64_t len_last = n - C.last_start;
    C.r = len_last < b ? len_last : 0;
    C.Bb = pow_mod(m, P.B, b);
    C.Br = C.r ? pow_mod(m, P.B, C.r) : 0;
    C.bshift = (b & (b - 1)) == 0 ? (uint32_t)(__ffsll((long long)b) - 1) : 0xFFu;
  }
  if (tid == 0) {
    Common& G = C.common();
    G.fp_tail = kNone;
    G.lo_tail = kNone;
    G.lo_tailpair = kNone;
    G.pretail = kNoSlot;
    G.npairs = 0;
    G.njobs = 0;
    G.nsusp = 0;
    G.verify_bytes = 0;
    G.collisions = 0;
    G.lastk = 0;
    G.qs.nopen[0] = G.qs.nopen[1] = G.qs.nitems = G.qs.npairs = G.qs.nsusp = 0;
    G.status.error = G.status.verify_bytes = G.status.collisions = 0;
  }
  gsync(C.grp);
  // (The scan's H takes the place of the list.)
  bool quick = b >= kQuickMinB && !C.expanded;
  if (quick) quick = quick_keys(m, PC, C, g, scr, l, dyn, dyn_words);
  if (!quick) {
    scan_keys(m, P, D, C, g, scr, l, dyn, dyn_words);
    if (failed(C)) return;
  }

  // Pointers of unmarked blocks: the block holding the leftmost occurrence
  // and the offset into it.
  for (uint64_t k = tid; k < c; k += nt) {
    if (marked(mw, k)) {
      ptr[k] = 0;
      off[k] = 0;
      continue;
    }
    const uint64_t p = lo[k], len = blen(g, k);
    uint64_t a = 0, z = c;
    while (a < z) {
      const uint64_t mid = (a + z) / 2;
      if (g.st[mid] <= p) a = mid + 1;
      else z = mid;
    }
    bool ok = a > 0;
    const uint64_t j = a - 1;
    if (ok) ok = p < g.st[j] + blen(g, j) && marked(mw, j) && p + len <= g.st[k];
    if (ok && p + len > g.st[j] + blen(g, j))
      ok = j + 1 < c && g.st[j + 1] == g.st[j] + blen(g, j) && marked(mw, j + 1);
    if (!ok) {
      fail(C, BT_EINTERNAL);
      continue;
    }
    ptr[k] = (uint32_t)j;
    off[k] = p - g.st[j];
  }
  if (failed(C)) return;

  const uint64_t nm = mr[words];
  if (threadIdx.x == 0) {
    C.nmarked[l] = nm;
    uint64_t* S = C.stats[l];
    S[BT_ST_NBLOCKS] = c;
    S[BT_ST_B] = b;
    S[BT_ST_COV] = (c - 1) * b + blen(g, c - 1);
    S[BT_ST_NMARKED] = nm;
    S[BT_ST_NPAIRS] = C.common().npairs;
    S[BT_ST_VERIFY_BYTES] = quick ? C.common().status.verify_bytes : C.common().verify_bytes;
    S[BT_ST_COLLISIONS] = quick ? C.common().status.collisions : C.common().collisions;
    S[BT_ST_FINAL_BLOCKS] = c;
    S[BT_ST_CANDIDATES] = quick && C.common().qs.nitems ? C.common().qs.cands : 0;
    S[BT_ST_HITS] = quick && C.common().qs.nitems ? C.common().qs.hits : 0;
  }
  if (last) {
    if (threadIdx.x == 0) C.arity[l] = 0;
    gsync(C.grp);
    tmark(C, 3);
    return;
  }
  // Children of marked blocks: rank r puts its children at r*arity + i.
  const uint64_t bn = bsz[l + 1];
  const uint32_t arity = (uint32_t)(b / bn);
  uint64_t* nst = (uint64_t*)(scr + C.sl.st[l + 1]);
  for (uint64_t wb = tid; wb < words; wb += nt)
    if (mw[wb]) atomicMax(&C.common().lastk, (unsigned long long)(wb * 32 + 31 - __clz(mw[wb])));
  gsync(C.grp);
  if (threadIdx.x == 0) {
    C.arity[l] = arity;
    const uint64_t lk = C.common().lastk;
    C.bad = nm == 0;
    if (nm != 0) {
      const uint64_t nch = (blen(g, lk) + bn - 1) / bn;
      const uint64_t nc = (nm - 1) * arity + nch;
      C.bad = nc > (n + bn - 1) / bn;
      C.c[l + 1] = nc;
      C.last_start = g.st[lk] + (nch - 1) * bn;
    }
    if (C.bad) fail(C, BT_EINTERNAL);
  }
  __syncthreads();
  if (C.bad) {  // (so in every CTA of the group)
    gsync(C.grp);
    return;
  }
  for (uint64_t w = tid; w < c * arity; w += nt) {
    const uint64_t k = w / arity, i = w - k * arity;
    if (!marked(mw, k)) continue;
    const uint64_t s = g.st[k] + i * bn;
    if (s >= g.st[k] + blen(g, k)) continue;
    nst[mrank(mw, mr, k) * arity + i] = s;
  }
  gsync(C.grp);
  tmark(C, 3);
}

template <class GRP>
__device__ PLv plevel(const Cta<GRP>& C, char* scr, const uint64_t* bsz, uint32_t l) {
  return PLv{C.n, C.c[l], bsz[l], (uint64_t*)(scr + C.sl.st[l]), (uint32_t*)(scr + C.sl.mw[l]),
             (uint32_t*)(scr + C.sl.mr[l]), (uint32_t*)(scr + C.sl.ptr[l]), (uint64_t*)(scr + C.sl.off[l]),
             (uint64_t*)(scr + C.sl.lo[l])};
}

// Levels with this few blocks are pruned by the leading CTA alone: some thirty
// barriers of the cluster cost more than its help.
constexpr uint64_t kLeaderPrune = 8192;

template <class GRP>
__device__ void prune_pass(const BParams& P, const BDoc& D, Cta<GRP>& C, char* scr) {
  const uint64_t* bsz = P.sizes + D.lv_off;
  for (int l = (int)C.L - 2; l >= 0; l--) {
    const PLv v = plevel(C, scr, bsz, (uint32_t)l), w = plevel(C, scr, bsz, (uint32_t)l + 1);
    const bool alone = v.c + w.c <= kLeaderPrune;
    uint64_t c2 = 0;
    const bool w_last = l + 1 == (int)C.L - 1;
    char* temp = scr + C.sl.temp;
    if (!GRP::many || (alone && C.grp.rank == 0))
      c2 = prune_level(v, w, w_last, C.arity[l], temp, P.max_rounds, C.common().prune, C.wtot, One{});
    else if (!alone)
      c2 = prune_level(v, w, w_last, C.arity[l], temp, P.max_rounds, C.common().prune, C.wtot, C.grp);
    if (GRP::many && alone) {
      if (C.grp.tid() == 0) C.common().part[0] = c2;
      gsync(C.grp);
      c2 = *(volatile uint64_t*)&C.common().part[0];
      gsync(C.grp);
    }
    if (c2 == kNone) {  // (so in every CTA of the group)
      if (C.grp.tid() == 0) fail(C, BT_EINTERNAL);
      gsync(C.grp);
      return;
    }
    if (threadIdx.x == 0) {
      C.c[l + 1] = c2;
      C.stats[l + 1][BT_ST_FINAL_BLOCKS] = c2;
    }
    __syncthreads();
  }
}

// ---------------------------------------------------------------------------
// Output: the tree's arrays, counters, level-1 prefix counts and leaf text in
// the pool; the device view that the query kernels read.
// ---------------------------------------------------------------------------
// Counters of a level, symbol-major (cp entries per symbol).  mode 0: symbol
// counts of each block (marked blocks of a non-last level are filled from their
// children afterwards); mode 1: counts of T[st[ptr], st[ptr] + off) of each
// unmarked block.  A warp takes BLOCKS consecutive blocks at a time, 16 bytes per
// lane and block in flight together, each with its own histogram (hist: 1024
// words per warp).  Four of them write the four counters of a symbol at once
// (zeros where a block is not counted; nothing when none of the four is); one, on
// levels with too few blocks to give every warp four, writes single counters.
template <uint32_t BLOCKS, class GRP>
__device__ void count_rows(const uint8_t* __restrict__ T, const Cta<GRP>& C, const PLv& v, int mode, bool last,
                           void* out, uint32_t cw, uint64_t cp, unsigned int* hist) {
  constexpr uint32_t IN_FLIGHT = BLOCKS < 2 ? BLOCKS : 2;
  const uint32_t S = C.S;
  const unsigned lane = threadIdx.x & 31, nw = C.grp.threads() >> 5;
  unsigned int* h = hist + (threadIdx.x >> 5) * 1024;
  for (uint64_t g = C.grp.tid() >> 5; BLOCKS * g < v.c; g += nw) {
    uint64_t s0[BLOCKS];
    uint32_t len[BLOCKS], top = 0;
    bool any = false;
#pragma unroll
    for (uint32_t q = 0; q < BLOCKS; q++) {
      const uint64_t k = BLOCKS * g + q;
      s0[q] = 0;
      len[q] = 0;
      if (k >= v.c) continue;
      const bool mk = marked(v.mw, k);
      any |= mode == 0 ? last || !mk : !mk;
      if (mode == 0 && (last || !mk)) {
        s0[q] = v.st[k];
        len[q] = (uint32_t)plen(v, k);
      } else if (mode == 1 && !mk) {
        s0[q] = v.st[v.ptr[k]];
        len[q] = (uint32_t)v.off[k];
      }
      top = top > len[q] ? top : len[q];
    }
    if (!any) continue;
    for (uint32_t i = lane; i < S; i += 32) {
#pragma unroll
      for (uint32_t q = 0; q < BLOCKS; q++) h[256 * q + i] = 0;
    }
    __syncwarp();
    for (uint32_t x = 16 * lane; x < top; x += 512) {
#pragma unroll
      for (uint32_t q0 = 0; q0 < BLOCKS; q0 += IN_FLIGHT) {
        uint4 t[IN_FLIGHT];
#pragma unroll
        for (uint32_t q = 0; q < IN_FLIGHT; q++)
          if (x < len[q0 + q]) t[q] = load16u(T, s0[q0 + q] + x);
#pragma unroll
        for (uint32_t q = 0; q < IN_FLIGHT; q++) {
          if (x >= len[q0 + q]) continue;
          const uint32_t w[4] = {t[q].x, t[q].y, t[q].z, t[q].w};
          const uint32_t have = len[q0 + q] - x;
#pragma unroll
          for (uint32_t i = 0; i < 16; i++)
            if (i < have) atomicAdd(&h[256 * (q0 + q) + C.sym[(w[i >> 2] >> (8 * (i & 3))) & 0xFF]], 1u);
        }
      }
    }
    __syncwarp();
    for (uint32_t i = lane; i < S; i += 32) {
      const uint64_t at = i * cp + BLOCKS * g;
      if constexpr (BLOCKS == 1) {
        cput(out, cw, at, h[i]);
      } else {
        const uint32_t a = h[i], b = h[256 + i], c = h[512 + i], d = h[768 + i];
        if (cw == 1) *(uint32_t*)((uint8_t*)out + at) = a | (b << 8) | (c << 16) | (d << 24);
        else if (cw == 2) *(uint2*)((uint16_t*)out + at) = make_uint2(a | (b << 16), c | (d << 16));
        else *(uint4*)((uint32_t*)out + at) = make_uint4(a, b, c, d);
      }
    }
    __syncwarp();
  }
}

// One-byte counters: a thread per block into a tile [S][TB] in shared memory
// (as k_count_small of bt_query.cu: warp w takes the columns that put its
// lanes in different banks), rows leave as runs.
template <class GRP>
__device__ void count_small(const uint8_t* __restrict__ T, const Cta<GRP>& C, const PLv& v, int mode, bool last, uint8_t* out,
                            uint64_t cp, uint8_t* tile, uint32_t tile_words) {
  const uint32_t S = C.S, tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  // As wide as the level, while the tile has room: at 128 blocks of 256 symbols
  // a tile of 512 was cleared and written mostly for nothing.
  uint32_t shift = 31 - __clz(blockDim.x);
  while (((uint64_t)S << shift) > tile_words * 4ull) shift--;
  while (shift > 7 && (1ull << (shift - 1)) >= v.c) shift--;
  const uint32_t TB = 1u << shift;
  const uint32_t col = 4 * (lane + 32 * (warp >> 2)) + (warp & 3);
  for (uint64_t k0 = (uint64_t)C.grp.rank * TB; k0 < v.c; k0 += (uint64_t)C.grp.size * TB) {
    __syncthreads();
    for (uint32_t i = tid; i < S * (TB / 4); i += blockDim.x) ((uint32_t*)tile)[i] = 0;
    __syncthreads();
    const uint64_t k = k0 + col;
    if (col < TB && k < v.c) {
      const bool mk = marked(v.mw, k);
      uint64_t s0 = 0;
      uint32_t len = 0;
      if (mode == 0 && (last || !mk)) {
        s0 = v.st[k];
        len = (uint32_t)plen(v, k);
      } else if (mode == 1 && !mk) {
        s0 = v.st[v.ptr[k]];
        len = (uint32_t)v.off[k];
      }
      uint8_t* my = tile + col;
      for (uint32_t x = 0; x < len; x += 16) {
        const uint4 q = load16u(T, s0 + x);
        const uint32_t w[4] = {q.x, q.y, q.z, q.w};
        const uint32_t have = len - x;
#pragma unroll
        for (uint32_t i = 0; i < 16; i++)
          if (i < have) my[TB * (uint32_t)C.sym[(w[i >> 2] >> (8 * (i & 3))) & 0xFF]]++;
      }
    }
    __syncthreads();
    for (uint32_t i = tid; i < S * (TB / 4); i += blockDim.x) {
      const uint32_t row = i >> (shift - 2), w = i & (TB / 4 - 1);
      const uint64_t at = k0 + 4 * w;
      if (at < cp) *(uint32_t*)(out + row * cp + at) = ((const uint32_t*)tile)[i];
    }
  }
  __syncthreads();
}

template <class GRP>
__device__ void write_output(const BParams& P, const BDoc& D, Cta<GRP>& C, char* scr, unsigned int* hist) {
  const uint64_t* bsz = P.sizes + D.lv_off;
  const unsigned tid = C.grp.tid(), nt = C.grp.threads(), lane = tid & 31, warp = tid >> 5, nw = nt >> 5;
  const uint32_t L = C.L, S = C.S;
  __shared__ OutLevel s_ol[kBMaxLevels];
  __shared__ uint32_t s_cw[kBMaxLevels];
  __shared__ uint64_t s_view, s_pre, s_leaf, s_sym;
  __shared__ uint32_t s_base;
  if (threadIdx.x == 0) {
    for (uint32_t l = 0; l < L; l++) s_cw[l] = counter_width(bsz[l]);
    const uint64_t words = (C.c[L - 1] + 31) / 32;
    const uint32_t* mrl = (const uint32_t*)(scr + C.sl.mr[L - 1]);
    const uint64_t nm = mrl[words];
    const uint64_t leaf_alloc = nm * bsz[L - 1];
    s_base = out_base(L, C.c, bsz, C.n, S);
    const uint64_t need = out_layout(L, s_base, C.c, s_cw, S, leaf_alloc, s_ol, &s_view, &s_pre, &s_leaf, &s_sym);
    C.out_bytes = need;
    if (tid == 0) {
      const unsigned long long o = atomicAdd(P.pool_used, (unsigned long long)need);
      C.common().out_off = C.out_off = o;
      if (o + need > P.pool_cap) fail(C, BT_ENOMEM);
    }
  }
  if (failed(C)) return;
  char* out = P.pool + C.common().out_off;
  const uint32_t bl = s_base;
  // Level arrays.
  for (uint32_t l = 0; l < L; l++) {
    const PLv v = plevel(C, scr, bsz, l);
    const uint64_t words = (v.c + 31) / 32;
    uint32_t* mw = (uint32_t*)(out + s_ol[l].mw);
    uint32_t* mr = (uint32_t*)(out + s_ol[l].mr);
    uint2* rec = (uint2*)(out + s_ol[l].rec);
    for (uint64_t k = tid; k < v.c; k += nt)
      rec[k] = marked(v.mw, k) ? make_uint2(kMarkedRec, (uint32_t)mrank(v.mw, v.mr, k))
                               : make_uint2(v.ptr[k], (uint32_t)v.off[k]);
    for (uint64_t i = tid; i <= words; i += nt) {
      if (i < words) mw[i] = v.mw[i];
      mr[i] = v.mr[i];
    }
  }
  gsync(C.grp);
  // Counters, last level first (marked blocks sum their children's).
  for (int l = (int)L - 1; l >= (int)bl; l--) {
    const PLv v = plevel(C, scr, bsz, (uint32_t)l);
    const bool last = l + 1 == (int)L;
    void* cnt = out + s_ol[l].cnt;
    void* pc = out + s_ol[l].pc;
    const uint32_t cw = s_cw[l];
    const uint64_t cp = counter_stride(v.c);
    if (cw == 1) {
      count_small(D.T, C, v, 0, last, (uint8_t*)cnt, cp, (uint8_t*)hist, P.dyn_words);
      count_small(D.T, C, v, 1, last, (uint8_t*)pc, cp, (uint8_t*)hist, P.dyn_words);
    } else {
      for (int mode = 0; mode < 2; mode++) {
        if (v.c >= 4 * nw) count_rows<4>(D.T, C, v, mode, last, mode ? pc : cnt, cw, cp, hist);
        else count_rows<1>(D.T, C, v, mode, last, mode ? pc : cnt, cw, cp, hist);
      }
    }
    gsync(C.grp);
    if (!last) {
      const void* ccnt = out + s_ol[l + 1].cnt;
      const uint32_t ccw = s_cw[l + 1];
      const uint64_t bn = bsz[l + 1], ccp = counter_stride(C.c[l + 1]);
      const uint32_t arity = C.arity[l];
      // A warp takes 32 blocks and a part of the symbols -- a quarter, or fewer
      // where the level has too few blocks for all warps, down to four (with
      // quarters a document of 4 KiB and 256 symbols took 160 thousand cycles
      // here, a third of its build); four symbols' children are read together.
      const uint32_t chunks = (uint32_t)((v.c + 31) / 32);
      uint32_t parts = 4;
      while (parts * chunks < nw && 4 * parts < S) parts *= 2;
      for (uint32_t it = warp; it < parts * chunks; it += nw) {
        const uint32_t part = it & (parts - 1);
        const uint64_t k = (uint64_t)(it / parts) * 32 + lane;
        if (k >= v.c || !marked(v.mw, k)) continue;
        const uint32_t s0 = S * part / parts, s1 = S * (part + 1) / parts;
        const uint64_t first = mrank(v.mw, v.mr, k) * arity;
        const uint32_t nch = (uint32_t)((plen(v, k) + bn - 1) / bn);
        for (uint32_t s = s0; s < s1; s += 4) {
          uint32_t x[4];
          if (ccw == 1 && nch == 4 && arity == 4) {
#pragma unroll
            for (uint32_t u = 0; u < 4; u++)
              x[u] = s + u < s1 ? *(const uint32_t*)((const uint8_t*)ccnt + (s + u) * ccp + first) : 0u;
#pragma unroll
            for (uint32_t u = 0; u < 4; u++) x[u] = __dp4a(x[u], 0x01010101u, 0u);
          } else if (nch == 2) {
            uint32_t y[4];
#pragma unroll
            for (uint32_t u = 0; u < 4; u++) {
              const uint64_t at = (s + u < s1 ? s + u : s) * ccp + first;
              x[u] = cget(ccnt, ccw, at);
              y[u] = cget(ccnt, ccw, at + 1);
            }
#pragma unroll
            for (uint32_t u = 0; u < 4; u++) x[u] += y[u];
          } else {
#pragma unroll
            for (uint32_t u = 0; u < 4; u++) x[u] = s + u < s1 ? sum_run(ccnt, ccw, (s + u) * ccp + first, nch) : 0u;
          }
#pragma unroll
          for (uint32_t u = 0; u < 4; u++)
            if (s + u < s1) cput(cnt, cw, (s + u) * cp + k, x[u]);
        }
      }
      gsync(C.grp);
    }
  }
  // Prefix counts of the base level, a warp per symbol.
  {
    const uint64_t c0 = C.c[bl], cp = counter_stride(c0);
    uint32_t* pre = (uint32_t*)(out + s_pre);
    const void* cnt = out + s_ol[bl].cnt;
    for (uint32_t s = warp; s < S; s += nw) {
      uint32_t carry = 0;
      for (uint64_t base = 0; base < c0; base += 32) {
        const uint64_t k = base + lane;
        const uint32_t x = k < c0 ? cget(cnt, s_cw[bl], s * cp + k) : 0u;
        uint32_t y = x;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
          const uint32_t o = __shfl_up_sync(kFull, y, d);
          if ((int)lane >= d) y += o;
        }
        if (k < c0) pre[s * (c0 + 1) + k] = carry + y - x;
        carry += __shfl_sync(kFull, y, 31);
      }
      if (lane == 0) pre[s * (c0 + 1) + c0] = carry;
    }
  }
  // Leaf text of the marked last-level blocks: rank r at r * b_L.
  {
    const PLv v = plevel(C, scr, bsz, L - 1);
    uint8_t* leaf = (uint8_t*)(out + s_leaf);
    // (16 bytes per thread when blocks are whole units.)
    const uint32_t unit = v.b % 16 == 0 ? 16 : 1;
    const uint64_t per = v.b / unit;
    for (uint64_t w = tid; w < v.c * per; w += nt) {
      const uint64_t k = w / per, i = (w - k * per) * unit;
      if (!marked(v.mw, k) || v.st[k] + i >= C.n) continue;
      uint8_t* to = leaf + mrank(v.mw, v.mr, k) * v.b + i;
      const uint64_t x = v.st[k] + i;
      if (unit == 16) {  // (a last unit past the text's end copies its padding)
        *(uint4*)to = *(const uint4*)(D.T + x);
      } else {
        *to = D.T[x];
      }
    }
    if (tid == 0) {
      const uint64_t words = (v.c + 31) / 32;
      const uint64_t nm = v.mr[words];
      uint64_t lb = nm * v.b;
      if (nm && marked(v.mw, v.c - 1) && C.n - v.st[v.c - 1] < v.b) lb -= v.b - (C.n - v.st[v.c - 1]);
      P.res[D.index].leaf_bytes = lb;
    }
  }
  int16_t* sym = (int16_t*)(out + s_sym);
  for (uint32_t i = tid; i < 256; i += nt) sym[i] = C.sym[i];
  if (tid == 0) {
    TreeView* tv = (TreeView*)(out + s_view);
    tv->n = C.n;
    tv->L = L;
    tv->S = S;
    tv->base = bl;
    for (uint32_t l = 0; l < L; l++) {
      const uint64_t words = (C.c[l] + 31) / 32;
      LevelView& lv = tv->lv[l];
      lv.c = (uint32_t)C.c[l];
      lv.b = view_len(bsz[l]);
      lv.arity = C.arity[l];
      lv.bshift = block_shift(view_len(bsz[l]));
      const PLv v = plevel(C, scr, bsz, l);
      lv.last_len = (uint32_t)plen(v, v.c - 1);
      lv.rec = (const uint2*)(out + s_ol[l].rec);
      lv.cnt = l >= bl ? out + s_ol[l].cnt : nullptr;
      lv.pc = l >= bl ? out + s_ol[l].pc : nullptr;
      lv.cw = s_cw[l];
      lv.cp = (uint32_t)counter_stride(C.c[l]);
      const uint32_t* mrl = (const uint32_t*)(scr + C.sl.mr[l]);
      C.nmarked[l] = mrl[words];
    }
    tv->pre = (const uint32_t*)(out + s_pre);
    tv->leaf = (const uint8_t*)(out + s_leaf);
    tv->sym = (const int16_t*)(out + s_sym);
  }
  gsync(C.grp);
}

template <class M, class GRP>
__device__ void build_doc(const M& m, const PrefixConst<M>& PC, const KrPow& pw, const BParams& P, uint32_t d, Cta<GRP>& C, char* scr, unsigned int* hist,
                          uint32_t dyn_words) {
  const BDoc D = P.docs[d];
  const uint64_t* bsz = P.sizes + D.lv_off;
  if (threadIdx.x == 0) {
    C.n = D.n;
    C.L = D.L;
    C.bad = D.L == 0 || D.L > kBMaxLevels || scratch_layout(D.n, D.L, bsz, &C.sl) > P.scratch_per_cta;
    if (C.grp.rank == 0) {
      C.common().err = C.bad ? BT_EINTERNAL : 0;
      for (uint32_t& x : C.common().seen) x = 0;
    }
    C.out_off = 0;
    C.out_bytes = 0;
    for (int i = 0; i < 6; i++) C.cyc[i] = 0;
    C.t_mark = clock64();
  }
  gsync(C.grp);
  if (!C.bad) alphabet(D.T, D.n, D.sigma, C);
  if (!failed(C)) {
    prefix_pass(m, PC, pw, D.T, D.n, (uint64_t*)(scr + C.sl.Hs), C);
    if (threadIdx.x == 0) C.expanded = 0;
    if (bsz[0] >= kQuickMinB) list_pass(D.T, D.n, scr, C);
    // Level 1: blocks k b_1.
    uint64_t* st0 = (uint64_t*)(scr + C.sl.st[0]);
    const uint64_t c0 = (D.n + bsz[0] - 1) / bsz[0];
    for (uint64_t k = C.grp.tid(); k < c0; k += C.grp.threads()) st0[k] = k * bsz[0];
    if (threadIdx.x == 0) {
      C.c[0] = c0;
      C.last_start = (c0 - 1) * bsz[0];
    }
    gsync(C.grp);
    tmark(C, 0);
    for (uint32_t l = 0; l < D.L; l++) {
      level_pass(m, PC, P, D, C, scr, l, (uint32_t*)hist, dyn_words);
      if (failed(C)) break;
    }
  }
  if (!failed(C) && P.prune) {
    prune_pass(P, D, C, scr);
    tmark(C, 4);
  }
  if (!failed(C)) write_output(P, D, C, scr, hist);
  gsync(C.grp);
  tmark(C, 5);
  // Results, from the leading CTA.
  if (C.grp.rank != 0) return;
  if (threadIdx.x == 0) {
    BRes& R = P.res[D.index];
    R.status = C.common().err;
    R.S = C.S;
    R.out_off = C.out_off;
    R.out_bytes = C.out_bytes;
    for (int i = 0; i < 6; i++) R.cycles[i] = C.cyc[i];
  }
  if (C.common().err == 0) {
    for (uint32_t l = threadIdx.x; l < D.L; l += blockDim.x) {
      BLevelRes& Lr = P.lres[D.lv_off + l];
      Lr.c = C.c[l];
      Lr.b = bsz[l];
      Lr.nmarked = C.nmarked[l];
      Lr.arity = C.arity[l];
      Lr.cw = counter_width(bsz[l]);
      for (int f = 0; f < BT_ST_FIELDS; f++) Lr.stats[f] = C.stats[l][f];
    }
  }
  __syncthreads();
}

// 64 registers per thread: one CTA of 1024 threads per SM, or several narrower
// ones (launch_shape).  A document belongs to a CTA, or to a cluster of them.
// Compiled apart for the two: one kernel for both spilled 2000 bytes of stores and
// 4160 of loads (-Xptxas -v, modulus 2^61 - 1), these 344 and 780 (one CTA) and 972
// and 2524 (cluster); with the bounded search of the open keys 712 and 1500, 932 and
// 2244.
template <class M, class GRP>
__global__ void __launch_bounds__(kMaxBThreads, 1) k_batch(const __grid_constant__ BParams P, M m,
                                                           const __grid_constant__ PrefixConst<M> PC,
                                                           const __grid_constant__ KrPow pw) {
  // Dynamic shared memory: the open keys' queues and bitmap of a level (or its
  // window filter), then (during the output) the symbol counters.
  extern __shared__ unsigned int s_hist[];
  __shared__ Cta<GRP> C;
  GRP grp;
  if constexpr (GRP::many) grp = this_cluster();
  char* scr = P.scratch + (uint64_t)(blockIdx.x / grp.size) * P.scratch_per_cta;
  if constexpr (GRP::many) {
    if (threadIdx.x == 0) {
      C.grp = grp;
      C.g = (Common*)scr;
    }
    __syncthreads();
  }
  for (;;) {
    if (grp.tid() == 0) C.common().doc = atomicAdd(P.next, 1u);
    gsync(grp);
    const uint32_t d = *(volatile uint32_t*)&C.common().doc;
    gsync(grp);
    if (d >= P.ndocs) return;
    build_doc(m, PC, pw, P, d, C, scr, s_hist, P.dyn_words);
  }
}

// ---------------------------------------------------------------------------
// Host driver.
// ---------------------------------------------------------------------------
// What the last batched build did (bt_batch_report).
struct Report {
  uint64_t kernel_docs, worker_docs, launches, retried, threads, ctas_per_sm, pool_bytes, scratch_bytes,
      max_grid, upload_us, kernel_us;
};
std::mutex g_report_mu;
Report g_report{};

struct DocPlan {
  uint64_t i;              // caller index
  uint64_t n;
  uint32_t sigma, L;
  uint64_t need;           // CTA scratch bytes
  uint64_t size_off;       // first block size in the batch's size array
};

// Opt the kernels in to their dynamic shared memory and to clusters of sixteen
// CTAs, once per device; the largest cluster the device can hold.
template <class M>
int prepare_batch_kernel(int bytes, uint32_t* max_group) {
  static std::atomic<uint32_t> most[64] = {};
  int dev = 0;
  BT_CUDA(cudaGetDevice(&dev));
  uint32_t g = most[dev & 63].load(std::memory_order_acquire);
  if (!g) {
    BT_CUDA(cudaFuncSetAttribute(k_batch<M, One>, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes));
    BT_CUDA(cudaFuncSetAttribute(k_batch<M, Cluster>, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes));
    g = 8;
    if (cudaFuncSetAttribute(k_batch<M, Cluster>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) == cudaSuccess) g = 16;
    for (; g > 1; g /= 2) {
      cudaLaunchConfig_t cfg{};
      cfg.gridDim = dim3(g);
      cfg.blockDim = dim3(kMaxBThreads);
      cfg.dynamicSmemBytes = bytes;
      cudaLaunchAttribute at{};
      at.id = cudaLaunchAttributeClusterDimension;
      at.val.clusterDim.x = g;
      at.val.clusterDim.y = at.val.clusterDim.z = 1;
      cfg.attrs = &at;
      cfg.numAttrs = 1;
      int n = 0;
      if (cudaOccupancyMaxActiveClusters(&n, k_batch<M, Cluster>, &cfg) == cudaSuccess && n > 0) break;
    }
    cudaGetLastError();
    most[dev & 63].store(g, std::memory_order_release);
  }
  *max_group = g;
  return BT_OK;
}

// `groups` clusters of `group` CTAs, per_group bytes of scratch each.
template <class M>
int launch_docs(const M& m, const BParams& base, uint32_t first, uint32_t count, unsigned groups, uint32_t group,
                uint64_t per_group, char* scratch, unsigned int* next, uint32_t threads, cudaStream_t s) {
  BParams P = base;
  P.docs = base.docs + first;
  P.ndocs = count;
  P.next = next;
  P.scratch = scratch;
  P.scratch_per_cta = per_group;
  P.dyn_words = dyn_words_of(threads);
  const int smem = (int)(P.dyn_words * sizeof(unsigned int));
  uint32_t most;
  BT_TRY(prepare_batch_kernel<M>((int)(dyn_words_of(kMaxBThreads) * sizeof(unsigned int)), &most));
  if (group > most) group = most;
  const PrefixConst<M> PC(m, P.B);
  const KrPow pw = kr_pow(m, pow_mod(m, P.B, 128));  // a thread of the prefix pass takes four 32-byte chunks
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(groups * group);
  cfg.blockDim = dim3(threads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute at{};
  at.id = cudaLaunchAttributeClusterDimension;
  at.val.clusterDim.x = group;
  at.val.clusterDim.y = at.val.clusterDim.z = 1;
  cfg.attrs = &at;
  cfg.numAttrs = group > 1 ? 1 : 0;
  if (group > 1) BT_LAUNCH(BT_CUDA(cudaLaunchKernelEx(&cfg, k_batch<M, Cluster>, P, m, PC, pw)));
  else BT_LAUNCH(BT_CUDA(cudaLaunchKernelEx(&cfg, k_batch<M, One>, P, m, PC, pw)));
  return BT_OK;
}

// Points a tree at the arrays that the kernel wrote to its pool.
void tree_from(bt_tree* t, uint64_t n, uint32_t tau, uint32_t leaf_len, uint32_t L, const bt_opts& o, int device,
               const BRes& R, const BLevelRes* lres, const std::shared_ptr<void>& pool) {
  t->n = n;
  t->tau = tau;
  t->leaf_len = leaf_len;
  t->L = L;
  t->prune = o.prune ? 1 : 0;
  t->seed = o.seed;
  t->q = o.modulus ? o.modulus : Mersenne61::Q;
  t->B = base_for(o.seed, t->q);
  t->device = device;
  t->S = R.S;
  t->leaf_bytes = R.leaf_bytes;
  t->slab = pool;
  t->lv.resize(L);
  uint64_t c[kBMaxLevels], bs[kBMaxLevels], o_view, o_pre, o_leaf, o_sym;
  uint32_t cw[kBMaxLevels];
  OutLevel ol[kBMaxLevels];
  for (uint32_t l = 0; l < L; l++) {
    c[l] = lres[l].c;
    bs[l] = lres[l].b;
    cw[l] = lres[l].cw;
  }
  const BLevelRes& last = lres[L - 1];
  t->base = out_base(L, c, bs, n, R.S);
  out_layout(L, t->base, c, cw, R.S, last.nmarked * last.b, ol, &o_view, &o_pre, &o_leaf, &o_sym);
  char* base = (char*)pool.get() + R.out_off;
  for (uint32_t l = 0; l < L; l++) {
    Level& v = t->lv[l];
    v.c = lres[l].c;
    v.b = lres[l].b;
    v.arity = lres[l].arity;
    v.nmarked = lres[l].nmarked;
    v.cw = lres[l].cw;
    v.mw = (uint32_t*)(base + ol[l].mw);
    v.mr = (uint32_t*)(base + ol[l].mr);
    v.rec = (uint2*)(base + ol[l].rec);
    v.cnt = l >= t->base ? base + ol[l].cnt : nullptr;
    v.pc = l >= t->base ? base + ol[l].pc : nullptr;
    memcpy(v.stats, lres[l].stats, sizeof(v.stats));
  }
  t->view = (TreeView*)(base + o_view);
  t->pre = (uint32_t*)(base + o_pre);
  t->leaf = (uint8_t*)(base + o_leaf);
  t->sym = (int16_t*)(base + o_sym);
  t->dev_bytes = R.out_bytes;
}

// A pool for finished trees, `cap` bytes.  It outlives the call: the memory
// goes back to the device's stream-ordered pool when the last tree is freed (on
// the freeing thread's stream; a tree is never freed while queries on it run).
int make_pool(uint64_t cap, cudaStream_t s, std::shared_ptr<void>& out) {
  void* p = nullptr;
  if (!alloc_allowed(cap)) return BT_ENOMEM;
  cudaError_t e = cudaMallocAsync(&p, cap, s);
  if (e != cudaSuccess) {
    cudaGetLastError();
    return e == cudaErrorMemoryAllocation ? BT_ENOMEM : BT_ECUDA;
  }
  out = std::shared_ptr<void>(p, [](void* x) {
    cudaFreeAsync(x, cudaStreamPerThread);
    cudaStreamSynchronize(cudaStreamPerThread);
  });
  return BT_OK;
}

// Device memory of one batched call, stream-ordered on the call's stream (no
// device-wide synchronisation, so calls on several host threads overlap).
struct DevFree {
  cudaStream_t s = nullptr;
  std::vector<void*> p;
  ~DevFree() {
    for (void* q : p) cudaFreeAsync(q, s);
  }
  template <class T>
  int alloc(T** out, uint64_t count) {
    void* q = nullptr;
    if (!alloc_allowed((count ? count : 1) * sizeof(T))) return BT_ENOMEM;
    cudaError_t e = cudaMallocAsync(&q, (count ? count : 1) * sizeof(T), s);
    if (e != cudaSuccess) {
      note_cuda_error(e, "cudaMallocAsync", __FILE__, __LINE__);
      cudaGetLastError();
      return e == cudaErrorMemoryAllocation ? BT_ENOMEM : BT_ECUDA;
    }
    p.push_back(q);
    *out = (T*)q;
    return BT_OK;
  }
};

// Threads of a CTA and CTAs per SM.  A short document leaves most of 1024 threads
// idle between barriers that wait for all of them, so several narrow CTAs share
// an SM where the documents are short enough and enough to fill them.  Kernel
// time of versioned texts (DNA copies, random bytes), us, with 1 x 1024, 2 x 512
// and 4 x 256 threads per SM:
//    64 of   4 KiB   152  124  123   (193  170  155;   163   163   199)
//   512 of   4 KiB   475  244  160   (643  332  213;   459   287   244)
//  2048 of  32 KiB  3414 1890 1401  (4529 2830 2478;  2951  1870  1666)
//   512 of  64 KiB  1260  750  574  (1563 1080 1104;  1014   734  1104)
//  1024 of 128 KiB  5050 4094 4319  (5355 4489 5074;  2952  2295  2562)
//   256 of 512 KiB  4923 4273 5822  (3830 3424 5191;  2710  3726  6470)
// A document much longer than the others would outlast them in a narrow CTA; a
// caller's bound on the CTAs counts whole SMs.
struct Shape {
  unsigned threads, ctas_per_sm;
};
Shape launch_shape(uint64_t docs, uint64_t mean, uint64_t longest, bool bounded) {
  const unsigned nsm = device_sm_count();
  if (bounded) return Shape{kMaxBThreads, 1};
  if (docs > nsm && mean <= (32u << 10) && longest <= (128u << 10)) return Shape{256, 4};
  if (docs > 2 * nsm && mean <= (128u << 10) && longest <= (512u << 10)) return Shape{512, 2};
  if (docs <= nsm && longest <= (8u << 10)) return Shape{512, 1};
  return Shape{kMaxBThreads, 1};
}

template <class M>
int run_batch(const M& m, const uint8_t* const* texts, const uint32_t* taus, const uint32_t* leaf_lens,
              const bt_opts& o, std::vector<DocPlan>& plans, const std::vector<uint64_t>& sizes,
              bt_tree** outs, cudaStream_t s) {
  const uint64_t nd = plans.size();
  if (nd == 0) return BT_OK;
  uint64_t bytes_all = 0, longest = 0;
  for (const DocPlan& d : plans) bytes_all += d.n, longest = std::max(longest, d.n);
  const Shape shape = launch_shape(nd, bytes_all / nd, longest, o.batch_ctas != 0);
  const unsigned threads = shape.threads, ctas_per_sm = shape.ctas_per_sm;
  int device = 0;
  BT_CUDA(cudaGetDevice(&device));
  const uint64_t q = o.modulus ? o.modulus : Mersenne61::Q;
  const uint64_t B = base_for(o.seed, q);
  // Longest documents first: the work queue hands them out first.
  std::vector<const DocPlan*> order(nd);
  for (uint64_t k = 0; k < nd; k++) order[k] = &plans[k];
  // Longest expected work first (text length times levels: each level
  // scans up to the whole text), so that the last CTAs to finish hold short
  // documents.
  std::stable_sort(order.begin(), order.end(), [](const DocPlan* a, const DocPlan* b) {
    return a->n * a->L > b->n * b->L;
  });
  DevFree mem;
  mem.s = s;
  // Texts, each at a 16-byte aligned offset and followed by at least 48 bytes
  // of padding (16-byte loads past a text's end stay in the buffer).
  std::vector<uint64_t> toff(nd);
  uint64_t ttotal = 0;
  for (uint64_t k = 0; k < nd; k++) {
    toff[k] = ttotal;
    ttotal += (plans[k].n + 63) & ~15ull;
  }
  uint8_t* d_text;
  BT_TRY(mem.alloc(&d_text, ttotal + 64));
  const auto t_up = std::chrono::steady_clock::now();
  for (uint64_t k = 0; k < nd; k++)
    BT_CUDA(cudaMemcpyAsync(d_text + toff[k], texts[plans[k].i], plans[k].n, cudaMemcpyDefault, s));
  const uint64_t upload_us = (uint64_t)std::chrono::duration_cast<std::chrono::microseconds>(
                                 std::chrono::steady_clock::now() - t_up).count();
  // Documents in processing order, block sizes, results.
  std::vector<BDoc> hd(nd);
  uint64_t nlv = 0;
  for (uint64_t k = 0; k < nd; k++) nlv += plans[k].L;
  std::vector<uint64_t> hsz(nlv);
  std::vector<uint32_t> lv_off(nd);
  {
    uint64_t o2 = 0;
    for (uint64_t k = 0; k < nd; k++) {
      lv_off[k] = (uint32_t)o2;
      for (uint32_t l = 0; l < plans[k].L; l++) hsz[o2 + l] = sizes[plans[k].size_off + l];
      o2 += plans[k].L;
    }
  }
  for (uint64_t r = 0; r < nd; r++) {
    const uint64_t k = (uint64_t)(order[r] - plans.data());
    hd[r] = BDoc{d_text + toff[k], plans[k].n, plans[k].sigma, plans[k].L, (uint32_t)k, lv_off[k]};
  }
  BDoc* d_docs;
  uint64_t* d_sizes;
  BRes* d_res;
  BLevelRes* d_lres;
  unsigned int* d_next;
  BT_TRY(mem.alloc(&d_docs, nd));
  BT_TRY(mem.alloc(&d_sizes, nlv));
  BT_TRY(mem.alloc(&d_res, nd));
  BT_TRY(mem.alloc(&d_lres, nlv));
  BT_TRY(mem.alloc(&d_next, 64));
  BT_CUDA(cudaMemcpyAsync(d_docs, hd.data(), nd * sizeof(BDoc), cudaMemcpyHostToDevice, s));
  BT_CUDA(cudaMemcpyAsync(d_sizes, hsz.data(), nlv * sizeof(uint64_t), cudaMemcpyHostToDevice, s));
  BT_CUDA(cudaMemsetAsync(d_res, 0, nd * sizeof(BRes), s));
  // Output pool: three bytes per text byte plus a fixed part per document;
  // a document that does not fit is built again into a pool of exactly the
  // size it reported.
  uint64_t pool_cap = 0;
  for (uint64_t k = 0; k < nd; k++) pool_cap += 3 * plans[k].n + (32u << 10);
  std::shared_ptr<void> pool;
  BT_TRY(make_pool(pool_cap, s, pool));
  unsigned long long* d_used;
  BT_TRY(mem.alloc(&d_used, 1));
  BT_CUDA(cudaMemsetAsync(d_used, 0, sizeof(unsigned long long), s));

  BParams P{};
  P.docs = d_docs;
  P.sizes = d_sizes;
  P.res = d_res;
  P.lres = d_lres;
  P.pool = (char*)pool.get();
  P.pool_used = d_used;
  P.pool_cap = pool_cap;
  P.B = B;
  P.prune = o.prune ? 1 : 0;
  P.max_rounds = o.max_rounds ? o.max_rounds : 4096;

  // Size classes: consecutive documents (in decreasing scratch need) whose
  // need is within 4x of the class's first; one launch per class, with as
  // many CTAs as memory allows, up to ctas_per_sm per SM.
  size_t free_b = 0, total_b = 0;
  BT_CUDA(cudaMemGetInfo(&free_b, &total_b));
  const uint64_t budget = (uint64_t)(free_b * 0.6);
  const unsigned nsm = device_sm_count();
  struct Cls {
    uint32_t first, count;
    uint64_t per_cta;
    unsigned grid;   // documents at a time
    uint32_t group;  // CTAs for each
  };
  std::vector<Cls> cls;
  uint64_t scratch_max = 0;
  for (uint32_t r = 0; r < nd;) {
    // One launch for every remaining document when the scratch of a full
    // grid sized for the largest of them fits; otherwise a class of the
    // documents within 4x of the largest, with as many CTAs as fit.
    uint64_t top = 0;
    for (uint32_t q2 = r; q2 < nd; q2++) top = std::max<uint64_t>(top, out_align(order[q2]->need));
    const uint64_t full = std::min<uint64_t>((uint64_t)(nd - r), (uint64_t)nsm * ctas_per_sm);
    uint32_t e = r;
    uint64_t grid;
    const uint64_t cap = o.batch_ctas ? o.batch_ctas : ~0ull;
    if (std::min<uint64_t>(full, cap) * top <= budget) {
      e = (uint32_t)nd;
      grid = std::min<uint64_t>(full, cap);
    } else {
      // The class: the documents of the order whose need is within 4x of the
      // first one's, with a grid sized for the largest of them.
      const uint64_t first = out_align(order[r]->need);
      top = first;
      while (e < nd && order[e]->need * 4 >= first && order[e]->need <= first * 4) {
        top = std::max<uint64_t>(top, out_align(order[e]->need));
        e++;
      }
      grid = std::min<uint64_t>({(uint64_t)(e - r), budget / top, cap});
      if (grid == 0) grid = 1;
    }
    // Fewer documents than SMs: a cluster of CTAs for each (not with a bound
    // on the CTAs, which leaves SMs to other work).  One document of DNA copies,
    // tau 2, leaf 32, by 1 and 16 CTAs: 130 KiB 1357 and 1355 us, 256 KiB 1539 and
    // 1165, 1 MiB 4513 and 2163 -- from 128 KiB a document on.
    uint64_t bytes = 0;
    for (uint32_t q2 = r; q2 < e; q2++) bytes += order[q2]->n;
    uint32_t group = 1;
    while (!o.batch_ctas && bytes >= (e - r) * (128ull << 10) && group < kMaxGroup && grid * group * 2 <= nsm) group *= 2;
    cls.push_back(Cls{r, e - r, top, (unsigned)grid, group});
    scratch_max = std::max<uint64_t>(scratch_max, grid * top);
    r = e;
  }
  char* d_scratch;
  BT_TRY(mem.alloc(&d_scratch, scratch_max));
  // The launches' device time (measurement hook), between two events.
  cudaEvent_t ev[2] = {nullptr, nullptr};
  const bool timed = cudaEventCreate(&ev[0]) == cudaSuccess && cudaEventCreate(&ev[1]) == cudaSuccess;
  if (timed) cudaEventRecord(ev[0], s);
  int lrc = BT_OK;
  for (size_t ci = 0; ci < cls.size() && lrc == BT_OK; ci++) {
    unsigned int* next = d_next + (ci % 64);
    lrc = cudaMemsetAsync(next, 0, sizeof(unsigned int), s) == cudaSuccess ? BT_OK : BT_ECUDA;
    if (lrc == BT_OK)
      lrc = launch_docs(m, P, cls[ci].first, cls[ci].count, cls[ci].grid, cls[ci].group, cls[ci].per_cta, d_scratch, next, threads, s);
  }
  if (timed) cudaEventRecord(ev[1], s);
  std::vector<BRes> res(nd);
  std::vector<BLevelRes> lres(nlv);
  if (lrc == BT_OK) {
    lrc = cudaMemcpyAsync(res.data(), d_res, nd * sizeof(BRes), cudaMemcpyDeviceToHost, s) == cudaSuccess &&
                  cudaMemcpyAsync(lres.data(), d_lres, nlv * sizeof(BLevelRes), cudaMemcpyDeviceToHost, s) ==
                      cudaSuccess && cudaStreamSynchronize(s) == cudaSuccess
              ? BT_OK
              : BT_ECUDA;
  }
  float kernel_ms = 0;
  if (timed && lrc == BT_OK) cudaEventElapsedTime(&kernel_ms, ev[0], ev[1]);
  for (cudaEvent_t e : ev)
    if (e) cudaEventDestroy(e);
  BT_TRY(lrc);

  // Documents whose tree did not fit in the pool: once more, into a pool of
  // the size they reported.
  std::vector<std::shared_ptr<void>> pool_of(nd, pool);
  uint64_t retried = 0;
  {
    std::vector<uint32_t> again;
    uint64_t cap2 = 0;
    for (uint64_t k = 0; k < nd; k++)
      if (res[k].status == BT_ENOMEM) {
        again.push_back((uint32_t)k);
        cap2 += out_align(res[k].out_bytes);
      }
    if (!again.empty()) {
      std::shared_ptr<void> pool2;
      BT_TRY(make_pool(cap2, s, pool2));
      std::vector<BDoc> hd2;
      uint64_t top = 0;
      for (uint32_t k : again) {
        for (uint64_t r = 0; r < nd; r++)
          if (hd[r].index == k) hd2.push_back(hd[r]);
        top = std::max<uint64_t>(top, out_align(plans[k].need));
      }
      BDoc* d_docs2;
      BT_TRY(mem.alloc(&d_docs2, hd2.size()));
      BT_CUDA(cudaMemcpyAsync(d_docs2, hd2.data(), hd2.size() * sizeof(BDoc), cudaMemcpyHostToDevice, s));
      BT_CUDA(cudaMemsetAsync(d_used, 0, sizeof(unsigned long long), s));
      BParams P2 = P;
      P2.docs = d_docs2;
      P2.pool = (char*)pool2.get();
      P2.pool_cap = cap2;
      const unsigned grid = (unsigned)std::max<uint64_t>(
          1, std::min<uint64_t>({(uint64_t)hd2.size(), (uint64_t)nsm * ctas_per_sm, scratch_max / top,
                                 o.batch_ctas ? (uint64_t)o.batch_ctas : ~0ull}));
      BT_CUDA(cudaMemsetAsync(d_next, 0, sizeof(unsigned int), s));
      BT_TRY(launch_docs(m, P2, 0, (uint32_t)hd2.size(), grid, 1, top, d_scratch, d_next, threads, s));
      BT_CUDA(cudaMemcpyAsync(res.data(), d_res, nd * sizeof(BRes), cudaMemcpyDeviceToHost, s));
      BT_CUDA(cudaMemcpyAsync(lres.data(), d_lres, nlv * sizeof(BLevelRes), cudaMemcpyDeviceToHost, s));
      BT_CUDA(cudaStreamSynchronize(s));
      for (uint32_t k : again) pool_of[k] = pool2;
      retried = again.size();
    }
  }

  // Trees.
  for (uint64_t k = 0; k < nd; k++) {
    const BRes& R = res[k];
    if (R.status != BT_OK) return R.status;
  }
  for (uint64_t k = 0; k < nd; k++) {
    const BRes& R = res[k];
    const DocPlan& D = plans[k];
    bt_tree* t = new (std::nothrow) bt_tree();
    if (!t) return BT_ENOMEM;
    outs[D.i] = t;
    tree_from(t, D.n, taus[D.i], leaf_lens[D.i], D.L, o, device, R, &lres[lv_off[k]], pool_of[k]);
    for (int i = 0; i < 6; i++) t->batch_cycles[i] = R.cycles[i];
  }
  {
    std::lock_guard<std::mutex> g(g_report_mu);
    g_report.kernel_docs = nd;
    g_report.upload_us = upload_us;
    g_report.kernel_us = (uint64_t)(kernel_ms * 1000.0f);
    g_report.launches = cls.size();
    g_report.retried = retried;
    g_report.threads = threads;
    g_report.ctas_per_sm = ctas_per_sm;
    g_report.pool_bytes = pool_cap;
    g_report.scratch_bytes = scratch_max;
    g_report.max_grid = 0;
    for (const Cls& c2 : cls) g_report.max_grid = std::max<uint64_t>(g_report.max_grid, (uint64_t)c2.grid * c2.group);
  }
  return BT_OK;
}

// Texts up to this long are built by one CTA in one launch: at 4 KiB and four
// levels it takes 160 us, some fifty launches and four round trips 350 us.  The
// line lies where one CTA is too slow for the counters of many symbols: random
// bytes take about as long both ways at 16 KiB (DNA copies still half at 64 KiB).
constexpr uint64_t kSoloText = 16u << 10;
constexpr uint64_t kSoloOut = 64u << 20;  // most room for its tree

// What a single build sends (to the start of its scratch) and receives (in the
// thread's pinned page, written by the kernel).
struct SoloHead {
  BDoc doc;
  uint64_t sizes[kBMaxLevels];
  unsigned long long used;
  unsigned int next;
};
struct SoloPage {
  SoloHead head;
  BRes res;
  BLevelRes lres[kBMaxLevels];
};
static_assert(sizeof(SoloPage) <= kPageBytes - kPageSolo, "a document fits its place in the pinned page");

// Moves a finished tree to memory of its own: the arrays as they are, the view's
// pointers moved along.
__global__ void __launch_bounds__(256) k_move_tree(const char* from, char* to, uint64_t bytes) {
  for (uint64_t i = 16 * (blockIdx.x * 256ull + threadIdx.x); i < bytes; i += 16 * 256ull * gridDim.x) {
    if (i >= sizeof(TreeView)) *(uint4*)(to + i) = *(const uint4*)(from + i);
  }
  if (blockIdx.x) return;
  // (The view, one thread per level: the rest of its 16-byte unit is padding.)
  const TreeView* a = (const TreeView*)from;
  TreeView* b = (TreeView*)to;
  auto moved = [&](const void* p) { return p ? to + ((const char*)p - from) : nullptr; };
  const uint32_t l = threadIdx.x;
  if (l < a->L) {
    LevelView v = a->lv[l];
    v.rec = (const uint2*)moved(v.rec);
    v.cnt = moved(v.cnt);
    v.pc = moved(v.pc);
    b->lv[l] = v;
  }
  if (l == 255) {
    b->n = a->n;
    b->L = a->L;
    b->S = a->S;
    b->base = a->base;
    b->pre = (const uint32_t*)moved(a->pre);
    b->leaf = (const uint8_t*)moved(a->leaf);
    b->sym = (const int16_t*)moved(a->sym);
  }
}

// The most a text's tree can take (no level pruned, all symbols).
uint64_t most_out(uint64_t n, uint32_t sigma, const std::vector<uint64_t>& b) {
  const uint32_t L = (uint32_t)b.size();
  uint64_t c[kBMaxLevels], x;
  uint32_t cw[kBMaxLevels];
  OutLevel ol[kBMaxLevels];
  for (uint32_t l = 0; l < L; l++) {
    c[l] = (n + b[l] - 1) / b[l];
    cw[l] = counter_width(b[l]);
  }
  const uint32_t S = (uint32_t)std::min<uint64_t>(std::min<uint64_t>(sigma, 256), n);
  // The prefix table is the largest at the level with the most blocks.
  return out_layout(L, 0, c, cw, S, c[L - 1] * b[L - 1], ol, &x, &x, &x, &x) + (c[L - 1] + 1) * (uint64_t)S * 4;
}

template <class M>
int run_solo(const M& m, const uint8_t* text, uint64_t n, uint32_t sigma, uint32_t tau, uint32_t leaf_len,
             const bt_opts& o, const std::vector<uint64_t>& sizes, cudaStream_t s, bt_tree* t) {
  char* page = pinned_page();
  if (!page) return BT_ENOMEM;
  SoloPage* S = (SoloPage*)(page + kPageSolo);
  const uint32_t L = (uint32_t)sizes.size();
  int device = 0;
  BT_CUDA(cudaGetDevice(&device));
  ScratchLayout sl;
  const uint64_t need = scratch_layout(n, L, sizes.data(), &sl), head = out_align(sizeof(SoloHead)),
                 room = out_align(n + 64), cap = out_align(most_out(n, sigma, sizes));
  DevFree mem;
  mem.s = s;
  char* d;
  BT_TRY(mem.alloc(&d, head + room + need + cap));
  SoloHead* dh = (SoloHead*)d;
  char* out = d + head + room + need;
  BT_CUDA(cudaMemcpyAsync(d + head, text, n, cudaMemcpyDefault, s));
  S->head.doc = BDoc{(const uint8_t*)(d + head), n, sigma, L, 0, 0};
  for (uint32_t l = 0; l < L; l++) S->head.sizes[l] = sizes[l];
  S->head.used = 0;
  S->head.next = 0;
  S->res.status = BT_ECUDA;
  BT_CUDA(cudaMemcpyAsync(dh, &S->head, sizeof(SoloHead), cudaMemcpyHostToDevice, s));
  BParams P{};
  P.docs = &dh->doc;
  P.sizes = dh->sizes;
  P.res = &S->res;
  P.lres = S->lres;
  P.pool = out;
  P.pool_used = &dh->used;
  P.pool_cap = cap;
  P.B = base_for(o.seed, o.modulus ? o.modulus : Mersenne61::Q);
  P.prune = o.prune ? 1 : 0;
  P.max_rounds = o.max_rounds ? o.max_rounds : 4096;
  BT_TRY(launch_docs(m, P, 0, 1, 1, 1, need, d + head + room, &dh->next, kMaxBThreads, s));
  BT_CUDA(cudaStreamSynchronize(s));
  const int rc = *(volatile int*)&S->res.status;
  if (rc == BT_ENOMEM) return BT_EINTERNAL;  // (the room was the most it can take)
  if (rc != BT_OK) return rc;
  std::shared_ptr<void> own;
  const uint64_t bytes = out_align16(S->res.out_bytes);
  BT_TRY(make_pool(bytes, s, own));
  BT_LAUNCH(k_move_tree<<<(unsigned)std::min<uint64_t>(152, bytes / 4096 + 1), 256, 0, s>>>(out, (char*)own.get(), bytes));
  BT_CUDA(cudaGetLastError());
  BT_CUDA(cudaStreamSynchronize(s));
  tree_from(t, n, tau, leaf_len, L, o, device, S->res, S->lres, own);
  return BT_OK;
}

}  // namespace

// One short text by one CTA.  BT_ENOMEM leaves the tree untouched: the caller's
// other path needs no memory in one piece.
int solo_build(const uint8_t* text, uint64_t n, uint32_t sigma, uint32_t tau, uint32_t leaf_len, const bt_opts& o,
               const std::vector<uint64_t>& sizes, cudaStream_t s, bt_tree* t) {
  if (!o.modulus) return run_solo(Mersenne61{}, text, n, sigma, tau, leaf_len, o, sizes, s, t);
  return run_solo(SmallMod{o.modulus}, text, n, sigma, tau, leaf_len, o, sizes, s, t);
}

bool solo_takes(uint64_t n, uint32_t sigma, const std::vector<uint64_t>& sizes) {
  return n <= kSoloText && sizes.size() <= kBMaxLevels && most_out(n, sigma, sizes) <= kSoloOut;
}

// Builds, with the persistent kernel, every document it can take (at most
// kBMaxText bytes and kBMaxLevels levels): routed[d] = 1 and outs[d] holds
// its tree.  Documents it cannot take keep routed[d] = 0 and are left to the
// caller.  Arguments are validated as bt_build_ex does.  Returns the first
// failure's status; trees already made stay in outs for the caller to free.
int batch_kernel_build(const uint8_t* const* texts, const uint64_t* ns, const uint32_t* sigmas,
                       const uint32_t* taus, const uint32_t* leaf_lens, uint64_t ndocs, const bt_opts& o,
                       std::vector<char>& routed, bt_tree** outs, cudaStream_t s, const std::vector<char>* eligible) {
  if (o.modulus && (o.modulus < 300 || o.modulus >= (1ull << 32))) return BT_EINVAL;
  std::vector<DocPlan> plans;
  std::vector<uint64_t> sizes;
  routed.assign(ndocs, 0);
  for (uint64_t d = 0; d < ndocs; d++) {
    const uint64_t n = ns[d];
    if (!texts[d] || n == 0 || n >= (1ull << 32) || taus[d] < 2 || taus[d] > 64 || leaf_lens[d] == 0 ||
        sigmas[d] == 0)
      return BT_EINVAL;
    std::vector<uint64_t> b;
    BT_TRY(plan_sizes(n, taus[d], leaf_lens[d], o, b));
    if (n > kBMaxText || b.size() > kBMaxLevels) continue;
    if (eligible && !(*eligible)[d]) continue;
    DocPlan pl;
    pl.i = d;
    pl.n = n;
    pl.sigma = sigmas[d];
    pl.L = (uint32_t)b.size();
    ScratchLayout sl;
    pl.need = scratch_layout(n, pl.L, b.data(), &sl);
    pl.size_off = sizes.size();
    sizes.insert(sizes.end(), b.begin(), b.end());
    plans.push_back(pl);
    routed[d] = 1;
  }
  if (o.modulus)
    return run_batch(SmallMod{o.modulus}, texts, taus, leaf_lens, o, plans, sizes, outs, s);
  return run_batch(Mersenne61{}, texts, taus, leaf_lens, o, plans, sizes, outs, s);
}

void batch_report_workers(uint64_t docs) {
  std::lock_guard<std::mutex> g(g_report_mu);
  g_report.worker_docs = docs;
}

void batch_report_reset() {
  std::lock_guard<std::mutex> g(g_report_mu);
  g_report = Report{};
}

// Long documents are built by the level kernels of the single-text path on
// host workers, at the same time as the batched kernel builds the others: a
// document longer than the batch's share per CTA would outlast the batch in
// its one CTA, and the single-text path gets more out of a
// long text than one CTA does.  A document is long at kSplitMin bytes or more
// and at least half the batch's bytes per CTA (so a batch large enough to
// balance its CTAs is not split).  The batched kernel then leaves the workers
// a share of the SMs in proportion to the long documents' bytes (at least 8
// SMs, at most half).  Returns the kernel's CTA cap (0: no split) and clears
// eligible[d] for the long documents.
constexpr uint64_t kSplitMin = 8ull << 20;

uint32_t batch_split(const uint64_t* ns, const uint32_t* taus, const uint32_t* leaf_lens, uint64_t ndocs,
                     const bt_opts& o, std::vector<char>& eligible) {
  (void)taus;
  (void)leaf_lens;
  eligible.assign(ndocs, 1);
  if (ndocs < 64 || o.batch_ctas) return 0;
  const unsigned nsm = device_sm_count();
  double total = 0, heavy = 0;
  for (uint64_t d = 0; d < ndocs; d++) total += (double)ns[d];
  const double share = total / (double)nsm;
  const double lim = std::max((double)kSplitMin, 0.5 * share);
  for (uint64_t d = 0; d < ndocs; d++)
    if ((double)ns[d] >= lim) {
      eligible[d] = 0;
      heavy += (double)ns[d];
    }
  if (heavy == 0 || heavy == total) {
    eligible.assign(ndocs, 1);
    return 0;
  }
  uint32_t reserve = (uint32_t)((double)nsm * heavy / total + 0.5);
  reserve = std::max<uint32_t>(8, std::min<uint32_t>(reserve, nsm / 2));
  return nsm - reserve;
}

}  // namespace bt

extern "C" int bt_batch_report(uint64_t* out, uint32_t cap) {
  using namespace bt;
  if (!out || cap < 13) return BT_EINVAL;
  std::lock_guard<std::mutex> g(g_report_mu);
  const uint64_t v[13] = {g_report.kernel_docs, g_report.worker_docs, g_report.launches, g_report.retried,
                          g_report.threads, g_report.ctas_per_sm, g_report.pool_bytes, g_report.scratch_bytes,
                          g_report.max_grid, 0, 0, g_report.upload_us,
                          g_report.kernel_us};
  memcpy(out, v, sizeof(v));
  return BT_OK;
}

extern "C" int bt_batch_cycles(const bt_tree* t, uint64_t* out, uint32_t cap) {
  if (!t || !out || cap < 6) return BT_EINVAL;
  memcpy(out, t->batch_cycles, 6 * sizeof(uint64_t));
  return BT_OK;
}
