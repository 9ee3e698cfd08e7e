// bt_quick.cu -- the level pass by first occurrences of selected grams.
//
// Section 3.1 finds the leftmost occurrence LO(x) of every block and pair
// with a scan of the level's windows.  Most of those windows can be ruled out
// without looking at them.  Select 16-byte grams by content alone (below) and
// let F(g) be the first position of a selected gram g in T.  If a string x
// holds g at offset a, then every occurrence p of x has g at p + a, so
//     LO(x) >= F(g) - a        for every selected gram of x,
// and with D = (g's own position) - F(g), a string at s has
//     LO(x) >= s - min D       over its selected grams.
// - min D = 0: the string holds a gram that occurs nowhere before it: LO = s.
// - otherwise p = s - min D is the earliest place x can occur at.  The bytes
//   there are compared with x: if they are equal, LO = p, proven.
// - otherwise x is left open ("active") and its occurrences are looked for:
//   every occurrence p of x has x's newest gram (the one with min D) at the
//   same offset, so only the occurrences of that one gram propose windows.
// Versioned and copied texts settle 90-100 % of the keys in the first two
// steps: an edit makes grams that occur nowhere before, and a block without
// an edit lies where its newest gram was first seen.  The scan of the other
// keys reads the list of selected grams, tests a bitmap of the active keys'
// grams and proposes a window only where an active key's newest gram occurs,
// instead of every place where any key's first gram occurs.  Windows tested
// by the levels of a build: 256 MiB of versioned text 41.3 M before (14.5 M of
// them matched a key), 7.3 M now; 2 GiB of DNA copies 469 M before, 37.5 M now.
// The builds: 16.2 -> 6.7 ms and 178 -> 42 ms (export included).
//
// Selection.  A gram is selected when the least of the 13 hashes of its
// 4-byte substrings is the first or the last of them (a closed syncmer,
// Edgar 2021).  Unlike a sliding minimum this depends on the gram alone, so
// all occurrences of a gram are selected or none; unlike a hash threshold it
// leaves no gap: of any 12 consecutive grams at least one is selected (density
// about 2/13).  So every string of 27 bytes or more has a selected gram, and
// every changed byte in the middle of a block changes a selected gram.
//
// F is a direct-mapped table indexed by the gram's hash that holds the least
// position seen: two grams that share a cell get the smaller of their first
// positions, which is still a lower bound (fewer keys settled, never a wrong
// one).  Everything is decided by byte comparisons or, for the active keys,
// by fingerprints whose matches are verified by byte comparison.
#include <algorithm>
#include <atomic>
#include <cstdio>
#include <type_traits>

#include "bt_quick_dev.cuh"

namespace bt {

namespace {

constexpr unsigned kT = 256;

__device__ __forceinline__ Span grid_span() {
  return Span{blockIdx.x * (uint64_t)kT + threadIdx.x, (uint64_t)gridDim.x * kT};
}

// ---------------------------------------------------------------------------
// The list of selected grams.
// ---------------------------------------------------------------------------

// mask[j]: the selected grams that start in [32 j, 32 j + 32); cnt[j] their
// number.  A thread takes one word of 32 positions: 44 substring hashes in
// registers, the minimum over 13 of them in four steps (2, 4, 8, then 8 + 8
// overlapping).  About 10 instructions per byte: issue-bound (256 MiB).
__global__ void __launch_bounds__(kT) k_list_mask(const uint8_t* __restrict__ T, uint64_t n, uint64_t nw,
                                                  uint32_t* __restrict__ mask, uint32_t* __restrict__ cnt) {
  const bool aligned = (((uintptr_t)T) & 15) == 0;
  for (uint64_t j = blockIdx.x * (uint64_t)kT + threadIdx.x; j < nw; j += (uint64_t)gridDim.x * kT) {
    uint32_t w[12], m[44];
    load48(T, n, 32 * j, aligned, w);
#pragma unroll
    for (int i = 0; i < 44; i++) m[i] = __funnelshift_r(w[i >> 2], w[(i >> 2) + 1 < 12 ? (i >> 2) + 1 : 11], 8 * (i & 3)) * kSubMul;
    uint32_t bits = 0;
    uint32_t a[43], b[41], c[37];
#pragma unroll
    for (int i = 0; i < 43; i++) a[i] = min(m[i], m[i + 1]);
#pragma unroll
    for (int i = 0; i < 41; i++) b[i] = min(a[i], a[i + 2]);
#pragma unroll
    for (int i = 0; i < 37; i++) c[i] = min(b[i], b[i + 4]);
#pragma unroll
    for (int i = 0; i < 32; i++) {
      const uint32_t least = min(c[i], c[i + 5]);
      if (m[i] == least || m[i + kSubs - 1] == least) bits |= 1u << i;
    }
    const uint64_t left = n - kGramLen + 1 - 32 * j;  // gram positions from 32 j on (nw covers at least one)
    if (left < 32) bits &= (1u << left) - 1u;
    mask[j] = bits;
    cnt[j] = __popc(bits);
  }
}

// The list entries: position x[e], and the cell of the gram in cell[e].  A CTA
// takes 256 words: its text and the positions of its grams are staged in
// shared memory, so that entries, not words, are dealt to the threads and
// leave in order.
__global__ void __launch_bounds__(kT) k_list_write(const uint8_t* __restrict__ T, uint64_t n, uint64_t nw,
                                                   const uint32_t* __restrict__ mask, const uint32_t* __restrict__ idx,
                                                   uint32_t* __restrict__ x, uint32_t* __restrict__ cell, uint32_t cmask) {
  constexpr uint32_t kBytes = 32 * kT;
  __shared__ __align__(16) uint32_t text[kBytes / 4 + 8];
  __shared__ uint16_t at[kBytes];
  const bool aligned = (((uintptr_t)T) & 15) == 0;
  for (uint64_t j0 = (uint64_t)blockIdx.x * kT; j0 < nw; j0 += (uint64_t)gridDim.x * kT) {
    const uint64_t p0 = 32 * j0;
    __syncthreads();
    for (uint32_t u = threadIdx.x; u < kBytes / 16 + 2; u += kT) {
      const uint64_t p = p0 + 16ull * u;
      uint4 v = make_uint4(0, 0, 0, 0);
      if (aligned && p + 16 <= n) {
        v = *(const uint4*)(T + p);
      } else if (p < n) {
        uint32_t b[4] = {0, 0, 0, 0};
        for (uint32_t t = 0; t < 16 && p + t < n; t++) b[t >> 2] |= (uint32_t)T[p + t] << (8 * (t & 3));
        v = make_uint4(b[0], b[1], b[2], b[3]);
      }
      ((uint4*)text)[u] = v;
    }
    const uint64_t j = j0 + threadIdx.x;
    const uint32_t e0 = idx[j0];
    const uint64_t jend = j0 + kT < nw ? j0 + kT : nw;
    const uint32_t ne = idx[jend] - e0;
    if (j < nw) {
      uint32_t o = idx[j] - e0;
      for (uint32_t b = mask[j]; b; b &= b - 1) at[o++] = (uint16_t)(32 * threadIdx.x + __ffs(b) - 1);
    }
    __syncthreads();
    for (uint32_t i = threadIdx.x; i < ne; i += kT) {
      const uint32_t a = at[i], q = a >> 2, sh = 8 * (a & 3);
      uint32_t w[5];
#pragma unroll
      for (int u = 0; u < 5; u++) w[u] = text[q + u];
      x[e0 + i] = (uint32_t)(p0 + a);
      cell[e0 + i] = gram_cell(__funnelshift_r(w[0], w[1], sh), __funnelshift_r(w[1], w[2], sh),
                               __funnelshift_r(w[2], w[3], sh), __funnelshift_r(w[3], w[4], sh), cmask);
    }
  }
}

// The list's leading part, whose first occurrences are found before the rest:
// in a repetitive text most later entries meet a cell that has one of those,
// which is final, so one read of the table settles them.  In one part, DNA 2
// GiB took 5.0 + 4.9 ms for the two passes; now 0.4 + 5.6 + 0.3.  Lists of up to
// 2^22 entries stay whole: the third launch costs what the second read does
// (text 20 MB: 1.63 and 1.66 ms).
constexpr uint32_t kWholeList = 1u << 22;
__host__ __device__ inline uint64_t list_split(uint32_t total) {
  return total > kWholeList ? (total / 16) & ~127ull : total;
}

// first[cell] = the least position of a leading entry with that cell (read first:
// after a gram's first copies have been seen nobody writes).  A pass of its
// own: inside k_list_write, between that kernel's barriers, the same random
// reads took 400 us of a 256 MiB build instead of 180.
__global__ void __launch_bounds__(kT) k_list_first(const uint32_t* __restrict__ total_p, const uint32_t* __restrict__ x,
                                                   const uint32_t* __restrict__ cell, uint32_t* first) {
  const uint64_t total = list_split(*total_p);
  for (uint64_t i = blockIdx.x * (uint64_t)kT + threadIdx.x; 4 * i < total; i += (uint64_t)gridDim.x * kT) {
    if (4 * i + 4 <= total) {
      const uint4 X = ((const uint4*)x)[i], C = ((const uint4*)cell)[i];
      const uint32_t f0 = *(volatile uint32_t*)&first[C.x], f1 = *(volatile uint32_t*)&first[C.y],
                     f2 = *(volatile uint32_t*)&first[C.z], f3 = *(volatile uint32_t*)&first[C.w];
      if (f0 > X.x) atomicMin(&first[C.x], X.x);
      if (f1 > X.y) atomicMin(&first[C.y], X.y);
      if (f2 > X.z) atomicMin(&first[C.z], X.z);
      if (f3 > X.w) atomicMin(&first[C.w], X.w);
    } else {
      for (uint64_t e = 4 * i; e < total; e++) atomicMin(&first[cell[e]], x[e]);
    }
  }
}

// D[e] = x[e] - F in place of the cell, four entries per thread (their random
// reads are in flight together), for the entries whose cell has a position of the leading part; the
// others lower their cell and are marked in `open` (a bit per entry, from the
// split on).
__global__ void __launch_bounds__(kT) k_list_dist(const uint32_t* __restrict__ total_p, const uint32_t* __restrict__ x,
                                                  uint32_t* __restrict__ D, uint32_t* first, uint32_t* __restrict__ open) {
  const uint64_t total = *total_p, split = list_split((uint32_t)total);
  const uint32_t xs = split < total ? x[split] : 0xFFFFFFFFu;
  // Whole warps: eight threads put their bits together.
  for (uint64_t i = blockIdx.x * (uint64_t)kT + threadIdx.x; 4 * (i & ~31ull) < total; i += (uint64_t)gridDim.x * kT) {
    uint32_t bits = 0;
    if (4 * i + 4 <= total) {
      const uint4 X = ((const uint4*)x)[i];
      uint4 C = ((const uint4*)D)[i];
      const uint32_t f0 = *(volatile uint32_t*)&first[C.x], f1 = *(volatile uint32_t*)&first[C.y],
                     f2 = *(volatile uint32_t*)&first[C.z], f3 = *(volatile uint32_t*)&first[C.w];
      auto one = [&](uint32_t p, uint32_t& c, uint32_t f, uint32_t bit) {
        if (f < xs) {
          c = p - f;
        } else {
          if (f > p) atomicMin(&first[c], p);
          bits |= bit;
        }
      };
      one(X.x, C.x, f0, 1);
      one(X.y, C.y, f1, 2);
      one(X.z, C.z, f2, 4);
      one(X.w, C.w, f3, 8);
      ((uint4*)D)[i] = C;
    } else {
      for (uint64_t e = 4 * i; e < total; e++) {
        const uint32_t c = D[e], f = *(volatile uint32_t*)&first[c];
        if (f < xs) {
          D[e] = x[e] - f;
        } else {
          atomicMin(&first[c], x[e]);
          bits |= 1u << (e & 3);
        }
      }
    }
    if (split == total) continue;
    bits <<= 4 * (threadIdx.x & 7);
#pragma unroll
    for (int o = 1; o < 8; o <<= 1) bits |= __shfl_xor_sync(0xFFFFFFFFu, bits, o);
    if ((threadIdx.x & 7) == 0 && 4 * i < total) open[i / 8] = bits;
  }
}

// The marked entries' distances, a warp per 32.
__global__ void __launch_bounds__(kT) k_list_rest(const uint32_t* __restrict__ total_p, const uint32_t* __restrict__ x,
                                                  uint32_t* __restrict__ D, const uint32_t* __restrict__ first,
                                                  const uint32_t* __restrict__ open) {
  const uint64_t total = *total_p, split = list_split((uint32_t)total), words = (total + 31) / 32;
  if (split == total) return;
  const unsigned lane = threadIdx.x & 31;
  for (uint64_t w0 = split / 32 + (blockIdx.x * (uint64_t)kT + threadIdx.x) / 32 * 32; w0 < words;
       w0 += (uint64_t)gridDim.x * kT) {
    const uint32_t mine = w0 + lane < words ? open[w0 + lane] : 0u;
    for (unsigned left = __ballot_sync(0xFFFFFFFFu, mine != 0); left; left &= left - 1) {
      const unsigned src = __ffs(left) - 1;
      const uint64_t e = 32 * (w0 + src) + lane;
      if ((__shfl_sync(0xFFFFFFFFu, mine, src) >> lane) & 1u) D[e] = x[e] - first[D[e]];
    }
  }
}

// seg1[j]: min D over the grams that start in [1024 j, 1024 j + 1024).
__global__ void __launch_bounds__(kT) k_list_seg1(uint64_t nw, const uint32_t* __restrict__ idx,
                                                  const uint32_t* __restrict__ D, uint64_t ns, uint32_t* __restrict__ seg1) {
  const unsigned lane = threadIdx.x & 31;
  for (uint64_t j = (blockIdx.x * (uint64_t)kT + threadIdx.x) / 32; j < ns; j += (uint64_t)gridDim.x * (kT / 32)) {
    const uint64_t w0 = j * (kSegBytes / 32), w1 = w0 + kSegBytes / 32 < nw ? w0 + kSegBytes / 32 : nw;
    uint32_t d = kNoDist;
    const uint32_t e1 = idx[w1];
    for (uint32_t e = idx[w0] + lane; e < e1; e += 32) d = min(d, D[e]);
    d = __reduce_min_sync(0xFFFFFFFFu, d);
    if (lane == 0) seg1[j] = d;
  }
}
// seg2[j]: min over 64 entries of seg1.
__global__ void __launch_bounds__(kT) k_list_seg2(uint64_t ns, const uint32_t* __restrict__ seg1, uint64_t ns2,
                                                  uint32_t* __restrict__ seg2) {
  for (uint64_t j = blockIdx.x * (uint64_t)kT + threadIdx.x; j < ns2; j += (uint64_t)gridDim.x * kT) {
    uint32_t d = kNoDist;
    for (uint64_t i = 64 * j; i < 64 * j + 64 && i < ns; i++) d = min(d, seg1[i]);
    seg2[j] = d;
  }
}

// ---------------------------------------------------------------------------
// One level.
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(kT) k_quick_min(QGeo g, QList Q, unsigned G, uint32_t* __restrict__ A,
                                                  uint32_t* __restrict__ X, uint32_t* __restrict__ flags,
                                                  QuickStatus* qs) {
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    qs->nopen[0] = qs->nopen[1] = qs->npairs = qs->nsusp = qs->nitems = 0;
    qs->redo = kSearchDone;
    qs->total = Q.idx[Q.nw];
  }
  quick_min(g, Q, G, A, X, flags, grid_span());
}

__global__ void __launch_bounds__(kT) k_quick_compare(QGeo g, const uint32_t* __restrict__ A, const uint32_t* __restrict__ X,
                                                      uint32_t* __restrict__ flags, uint32_t ppk, unsigned L) {
  quick_compare(g, A, X, flags, ppk, L, grid_span());
}

__global__ void __launch_bounds__(kT) k_chase_init(Chase C, uint32_t bwords, bool again) { chase_init(C, bwords, again, grid_span()); }

template <class M, unsigned G>
__global__ void __launch_bounds__(kT) k_chase_keys(M m, const __grid_constant__ PrefixConst<M> P, const uint64_t* Hs, Chase C) {
  chase_keys<M, G>(m, PrefixAt<M>(P, C.g.T, C.g.n, Hs), C, grid_span());
}

template <class M, class FIRST>
__global__ void __launch_bounds__(kT, 4) k_chase_scan(M m, const __grid_constant__ PrefixConst<M> P, const uint64_t* Hs,
                                                      const __grid_constant__ Chase C, uint32_t e0, uint32_t e1,
                                                      uint32_t smem_words, const unsigned long long* __restrict__ bound2,
                                                      unsigned long long limit, ChaseState verdict) {
  extern __shared__ uint32_t bits_s[];
  __shared__ uint2 hit_q[kT / 32][kHitQ];
  __shared__ uint8_t gap_q[FIRST::value ? kT / 32 : 1][kHitQ];
  __shared__ uint32_t cand_q[kT / 32][kCandQ];
  for (uint32_t i = threadIdx.x; i < smem_words; i += kT) bits_s[i] = C.bitmap[i];
  __syncthreads();
  const unsigned warp = threadIdx.x >> 5;
  chase_scan(m, PrefixAt<M>(P, C.g.T, C.g.n, Hs), C, FIRST{}, e0, e1, smem_words ? bits_s : C.bitmap, hit_q[warp],
             gap_q[FIRST::value ? warp : 0], cand_q[warp], bound2, limit, verdict, grid_span());
}

// (After the sample: too much work in it?)
__global__ void __launch_bounds__(kT) k_chase_bound(Chase C, unsigned long long most) {
  const uint64_t work = C.qs->work;
  const uint32_t redo = C.qs->redo;
  chase_bound(C, grid_span());
  if (blockIdx.x == 0 && threadIdx.x == 0 && redo == kSearchDone && work > most) C.qs->redo = kCompare;
}

__global__ void __launch_bounds__(kT) k_chase_live(Chase C, uint32_t split) { chase_live(C, split, grid_span()); }

__global__ void __launch_bounds__(kT) k_chase_tail(Chase C) { chase_tail(C, grid_span()); }

__global__ void __launch_bounds__(kT) k_chase_verify(Chase C, uint64_t ppk, unsigned L) { chase_verify(C, ppk, L, grid_span()); }

// (What a search that was given up has found is not the answer.)
__global__ void __launch_bounds__(kT) k_chase_apply(Chase C) {
  if (C.qs->redo == kSearchDone) chase_apply(C, grid_span());
}

__global__ void __launch_bounds__(kT) k_chase_exact(Chase C, uint64_t nsusp) {
  chase_exact(C, blockIdx.y, gridDim.y, nsusp, grid_span());
}

__global__ void __launch_bounds__(kT) k_chase_exact_apply(Chase C, uint64_t nsusp) { chase_exact_apply(C, nsusp, grid_span()); }

// Settled blocks get their leftmost occurrence, open keys go to the item list
// (2 k: block k, 2 k + 1: the pair that starts with it), and the marks follow
// from the settled pairs (again later if some were open).
__global__ void __launch_bounds__(kT) k_quick_settle(QGeo g, const uint32_t* __restrict__ A, const uint32_t* __restrict__ X,
                                                     const uint32_t* __restrict__ flags, uint64_t* __restrict__ lo,
                                                     uint8_t* __restrict__ ps, uint32_t* __restrict__ items,
                                                     uint32_t* __restrict__ mw, uint32_t* __restrict__ wpop,
                                                     QuickStatus* qs, Status* status) {
  // One atomic per counter and CTA, and one per 256 blocks that hold an open
  // key: with one per warp and counter their queue on five addresses was the
  // whole time (121 and 191 us on the two lowest levels of the 256 MiB text).
  __shared__ uint32_t s_cnt[kT / 32];
  __shared__ unsigned long long s_at, s_sum[kT / 32][4];
  const unsigned lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const uint64_t tiles = (g.c + kT - 1) / kT;
  uint64_t sum_vb = 0;
  uint32_t sum_np = 0, sum_b = 0, sum_p = 0;
  for (uint64_t tile = blockIdx.x; tile < tiles; tile += gridDim.x) {
    const uint64_t base = tile * kT + warp * 32, k = base + lane;
    bool ob = false, op = false;
    uint8_t st = 0;
    uint64_t vb = 0;
    if (k < g.c) {
      const uint64_t s = g.st[k], len = g.n - s < g.b ? g.n - s : g.b;
      const uint32_t d = A[k];
      uint64_t p = s;
      if (s != 0 && d != 0) {
        ob = d == kNoDist || (flags[k] & kBlkDiffers);
        p = ob ? kNone : (d > s ? 0 : s - d);
        if (d != kNoDist) vb += 2 * len;
      }
      lo[k] = p;
      uint32_t d2 = 0;
      uint64_t plen = 0;
      st = pair_state(g, A, X, flags, k, &d2, &plen, &op);
      ps[k] = st;
      if (st == kIsPair && d2 != kNoDist) vb += 2 * plen;
    }
    uint32_t left = __shfl_up_sync(0xFFFFFFFFu, (uint32_t)st, 1);
    if (lane == 0) {
      left = 0;
      if (k > 0 && k <= g.c) {
        uint32_t d2;
        uint64_t plen;
        bool o;
        left = pair_state(g, A, X, flags, k - 1, &d2, &plen, &o);
      }
    }
    const bool mk = k < g.c && ((left & kLeftmost) || (st & kLeftmost) || !((left | st) & kIsPair));
    const uint32_t bits = __ballot_sync(0xFFFFFFFFu, mk);
    const uint32_t bb = __ballot_sync(0xFFFFFFFFu, ob), bp = __ballot_sync(0xFFFFFFFFu, op);
    sum_np += __popc(__ballot_sync(0xFFFFFFFFu, st & kIsPair));
    sum_b += __popc(bb);
    sum_p += __popc(bp);
    sum_vb += vb;
    if (lane == 0 && base < g.c) {
      mw[base / 32] = bits;
      wpop[base / 32] = __popc(bits);
    }
    const uint32_t mine = __popc(bb) + __popc(bp);
    if (lane == 0) s_cnt[warp] = mine;
    if (__syncthreads_or(mine != 0)) {
      if (threadIdx.x == 0) {
        uint32_t n = 0;
        for (unsigned w = 0; w < kT / 32; w++) {
          const uint32_t v = s_cnt[w];
          s_cnt[w] = n;
          n += v;
        }
        s_at = atomicAdd(&qs->nitems, (unsigned long long)n);
      }
      __syncthreads();
      const uint64_t at = s_at + s_cnt[warp];
      const uint32_t lt = (1u << lane) - 1u;
      if (ob) items[at + __popc(bb & lt)] = (uint32_t)(2 * k);
      if (op) items[at + __popc(bb) + __popc(bp & lt)] = (uint32_t)(2 * k + 1);
    }
    __syncthreads();
  }
  sum_vb = warp_sum64(sum_vb);
  if (lane == 0) {
    s_sum[warp][0] = sum_b;
    s_sum[warp][1] = sum_p;
    s_sum[warp][2] = sum_np;
    s_sum[warp][3] = sum_vb;
  }
  __syncthreads();
  if (threadIdx.x < 4) {
    unsigned long long v = 0;
    for (unsigned w = 0; w < kT / 32; w++) v += s_sum[w][threadIdx.x];
    unsigned long long* to = threadIdx.x == 0   ? &qs->nopen[0]
                             : threadIdx.x == 1 ? &qs->nopen[1]
                             : threadIdx.x == 2 ? &qs->npairs
                                                : &status->verify_bytes;
    if (v) atomicAdd(to, v);
  }
}

// The marks again, from the pair states the open keys' search completed.
__global__ void __launch_bounds__(kT) k_quick_remark(uint64_t c, const uint8_t* __restrict__ ps, uint32_t* __restrict__ mw,
                                                     uint32_t* __restrict__ wpop) {
  const uint64_t words = (c + 31) / 32;
  for (uint64_t base = (blockIdx.x * (uint64_t)kT + threadIdx.x) & ~31ull; base < words * 32;
       base += (uint64_t)gridDim.x * kT) {
    const uint64_t k = base + (threadIdx.x & 31);
    bool mk = false;
    if (k < c) {
      const uint8_t l = k ? ps[k - 1] : 0, r = ps[k];
      mk = (l & kLeftmost) || (r & kLeftmost) || !((l | r) & kIsPair);
    }
    const uint32_t bits = __ballot_sync(0xFFFFFFFFu, mk);
    if ((threadIdx.x & 31) == 0) {
      mw[base / 32] = bits;
      wpop[base / 32] = __popc(bits);
    }
  }
}

// Size of the next level and the start of its last block (one thread).
__device__ void level_end(const QGeo& g, const uint32_t* mw, const uint32_t* mr, uint64_t words, uint64_t nmarked,
                          uint32_t arity, uint64_t bn, Status* status, QuickStatus* qs) {
  qs->nmarked = nmarked;
  status->next_c = 0;
  status->last_start = 0;
  if (arity == 0 || nmarked == 0) return;
  const uint64_t w = last_marked_word(mw, mr, words, nmarked);
  const uint64_t last = w * 32 + 31 - __clz(mw[w]);
  const uint64_t len = qblen(g, last), nch = (len + bn - 1) / bn;
  status->next_c = (nmarked - 1) * arity + nch;
  status->last_start = g.st[last] + (nch - 1) * bn;
}

// Rank prefix of a level of at most kRankWords mark words and the level's end,
// by one CTA (eight words per thread and step).
constexpr uint64_t kRankWords = 16384;
__global__ void __launch_bounds__(1024) k_quick_rank(QGeo g, const uint32_t* __restrict__ mw, const uint32_t* __restrict__ wpop,
                                                     uint32_t* mr, uint32_t arity, uint64_t bn, Status* status,
                                                     QuickStatus* qs) {
  __shared__ uint32_t sm[32];
  const uint64_t words = (g.c + 31) / 32;
  const unsigned lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  uint32_t carry = 0;
  for (uint64_t base = 0; base < words; base += 8192) {
    const uint64_t i = base + 8ull * threadIdx.x;
    uint32_t v[8], sum = 0;
#pragma unroll
    for (int u = 0; u < 8; u++) {
      v[u] = i + u < words ? wpop[i + u] : 0;
      sum += v[u];
    }
    uint32_t x = sum;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      const uint32_t o = __shfl_up_sync(0xFFFFFFFFu, x, d);
      if (lane >= (unsigned)d) x += o;
    }
    if (lane == 31) sm[warp] = x;
    __syncthreads();
    if (warp == 0) {
      uint32_t w = sm[lane];
#pragma unroll
      for (int d = 1; d < 32; d <<= 1) {
        const uint32_t o = __shfl_up_sync(0xFFFFFFFFu, w, d);
        if (lane >= (unsigned)d) w += o;
      }
      sm[lane] = w;
    }
    __syncthreads();
    uint32_t at = carry + (warp ? sm[warp - 1] : 0) + x - sum;
#pragma unroll
    for (int u = 0; u < 8; u++) {
      if (i + u < words) mr[i + u] = at;
      at += v[u];
    }
    carry += sm[31];
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    mr[words] = carry;
    level_end(g, mw, mr, words, carry, arity, bn, status, qs);
  }
}
__global__ void k_quick_end(QGeo g, const uint32_t* mw, const uint32_t* mr, uint32_t arity, uint64_t bn, Status* status,
                            QuickStatus* qs) {
  const uint64_t words = (g.c + 31) / 32;
  level_end(g, mw, mr, words, mr[words], arity, bn, status, qs);
}

__device__ __forceinline__ bool qmark(const uint32_t* __restrict__ mw, uint64_t k) { return (mw[k >> 5] >> (k & 31)) & 1u; }

// Back-pointers of the unmarked blocks (the block that holds the leftmost
// occurrence and the offset into it; the copied window must lie in one or two
// marked blocks and end before the block) and the children of the marked
// ones: the block of mark rank r puts its children at r arity + i.  The host
// reads the status one step later, after the next level or the pruning has run
// on these pointers: a block whose occurrence fails the check still gets one that
// lies in the level.
__global__ void __launch_bounds__(kT) k_quick_points(QGeo g, const uint32_t* __restrict__ mw, const uint32_t* __restrict__ mr,
                                                     const uint64_t* __restrict__ lo, uint32_t* __restrict__ ptr,
                                                     uint64_t* __restrict__ off, uint32_t arity, uint64_t bn,
                                                     uint64_t* __restrict__ next_st, Status* status) {
  const bool all_present = g.c == (g.n + g.b - 1) / g.b;
  for (uint64_t k = blockIdx.x * (uint64_t)kT + threadIdx.x; k < g.c; k += (uint64_t)gridDim.x * kT) {
    const uint64_t s = g.st[k], len = g.n - s < g.b ? g.n - s : g.b;
    if (qmark(mw, k)) {
      ptr[k] = 0;
      off[k] = 0;
      if (next_st) {
        const uint64_t r = mr[k >> 5] + __popc(mw[k >> 5] & ((1u << (k & 31)) - 1u));
        for (uint64_t i = 0; i * bn < len; i++) next_st[r * arity + i] = s + i * bn;
      }
      continue;
    }
    const uint64_t p = lo[k];
    uint64_t j;
    bool ok = p < s && len <= s - p;
    if (all_present) {
      j = ok ? p / g.b : 0;
    } else {
      uint64_t a = 0, z = k;  // first index with st > p; p < s
      while (a < z) {
        const uint64_t mid = (a + z) / 2;
        if (g.st[mid] <= p) a = mid + 1;
        else z = mid;
      }
      ok = ok && a > 0;
      j = a ? a - 1 : 0;
    }
    if (ok) ok = p < g.st[j] + qblen(g, j) && qmark(mw, j);
    if (ok && p + len > g.st[j] + qblen(g, j))
      ok = j + 1 < g.c && g.st[j + 1] == g.st[j] + qblen(g, j) && qmark(mw, j + 1);
    if (!ok) {
      atomicExch(&status->error, 5ull);
      ptr[k] = 0;
      off[k] = 0;
      continue;
    }
    ptr[k] = (uint32_t)j;
    off[k] = p - g.st[j];
  }
}

// Opt a kernel in to more than 48 KiB of shared memory, once per device.
template <auto FN>
int allow_smem(int bytes) {
  static std::atomic<uint64_t> done{0};
  int dev = 0;
  BT_CUDA(cudaGetDevice(&dev));
  const uint64_t bit = 1ull << (dev & 63);
  if (done.load(std::memory_order_acquire) & bit) return BT_OK;
  BT_CUDA(cudaFuncSetAttribute(FN, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes));
  done.fetch_or(bit, std::memory_order_acq_rel);
  return BT_OK;
}

uint64_t pow2_from(uint64_t x) {
  uint64_t p = 64;
  while (p < x) p <<= 1;
  return p;
}

}  // namespace

int quick_list(BuildCtx& ctx, QuickBuild& qb) {
  const uint64_t n = ctx.t->n;
  cudaStream_t s = ctx.s;
  const uint64_t nw = n < kGramLen ? 0 : (n - kGramLen + 1 + 31) / 32;  // words of 32 gram positions
  const uint64_t ns = (n + kSegBytes - 1) / kSegBytes, ns2 = (ns + 63) / 64;
  // Cells of the first-occurrence table: one per eight positions (there is
  // about one list entry per six, most of them repeats), at most 256 MiB:
  // random reads run at 300 G/s from L2-sized tables, 80-90 from 256 MiB, 47
  // from 1 GiB (GB300), and a shared cell only loosens a bound.  Builds with
  // one cell per 8, 16 and 32 positions of the 256 MiB text: 8.69, 8.74 and
  // 9.12 ms; with at most 2^24 .. 2^27 cells for 2 GiB of DNA: 71.3, 57.2, 58.1
  // and 59.2 ms.
  uint64_t cells = 1024;
  while (cells < n / 8 && cells < (1ull << 26)) cells <<= 1;
  uint32_t *mask, *first, *agg;
  Scratch tmp(s);
  BT_TRY(tmp.alloc(&mask, nw));
  BT_TRY(tmp.alloc(&agg, scan_scratch_words(nw)));
  BT_TRY(qb.mem.alloc(&qb.idx, nw + 1));
  BT_TRY(tmp.alloc(&first, cells));
  BT_TRY(qb.mem.alloc(&qb.seg1, ns));
  BT_TRY(qb.mem.alloc(&qb.seg2, ns2));
  ProfScope ps("gram_list", s, n);
  if (nw) BT_LAUNCH(k_list_mask<<<grid_for(nw, kT), kT, 0, s>>>(ctx.T, n, nw, mask, qb.idx));
  BT_TRY(scan_u32(qb.idx, qb.idx, nw, s, agg));
  // Room for the entries: all positions of a short text (no round trip), the
  // number found otherwise.
  uint64_t cap = n;
  if (n > (4ull << 20)) {
    uint32_t total = 0;
    BT_CUDA(cudaMemcpyAsync(&total, qb.idx + nw, sizeof(uint32_t), cudaMemcpyDeviceToHost, s));
    BT_CUDA(cudaStreamSynchronize(s));
    cap = total;
  }
  cap = (cap + 63) & ~63ull;
  uint32_t* xd;
  BT_TRY(qb.mem.alloc(&xd, 2 * (cap ? cap : 64)));
  qb.x = xd;
  qb.D = xd + (cap ? cap : 64);
  BT_CUDA(cudaMemsetAsync(first, 0xFF, cells * sizeof(uint32_t), s));
  if (nw)
    BT_LAUNCH(k_list_write<<<(unsigned)std::min<uint64_t>((nw + kT - 1) / kT, 152 * 16), kT, 0, s>>>(
        ctx.T, n, nw, mask, qb.idx, qb.x, qb.D, (uint32_t)(cells - 1)));
  BT_LAUNCH(k_list_first<<<grid_for(cap / 4 + 1, kT, 152 * 16), kT, 0, s>>>(qb.idx + nw, qb.x, qb.D, first));
  uint32_t* open = mask;  // (not read any more, and as long: a list has no more entries than grams)
  const bool parts = cap > kWholeList;
  BT_LAUNCH(k_list_dist<<<grid_for(cap / 4 + 1, kT, 152 * 16), kT, 0, s>>>(qb.idx + nw, qb.x, qb.D, first, open));
  if (parts)
    BT_LAUNCH(k_list_rest<<<grid_for(cap / 32 + 1, kT, 152 * 8), kT, 0, s>>>(qb.idx + nw, qb.x, qb.D, first, open));
  BT_LAUNCH(k_list_seg1<<<grid_for(ns * 32, kT), kT, 0, s>>>(nw, qb.idx, qb.D, ns, qb.seg1));
  BT_LAUNCH(k_list_seg2<<<grid_for(ns2, kT), kT, 0, s>>>(ns, qb.seg1, ns2, qb.seg2));
  BT_CUDA(cudaGetLastError());
  qb.list = QList{qb.idx, qb.x, qb.D, qb.seg1, qb.seg2, nw};
  qb.ready = true;
  BT_TRY(qb.mem.alloc(&qb.qs, 1));
  qb.qs_host = (QuickStatus*)(pinned_page() + kPageQuick);  // (the build made sure of the page)
  return BT_OK;
}

// The search of a level's open keys: its tables, the list's two parts (the first
// sixteenth, then the rest against the bounds it lowered: most copies' content is
// first seen early; short lists have one part), and the launches of its steps.
struct SearchRun {
  Chase C;
  uint64_t ni, gcap, top;
  uint32_t bwords, total, split;
};

template <class M>
struct Search {
  const M& m;
  BuildCtx& ctx;
  QuickBuild& qb;
  SearchRun& R;
  const PrefixConst<M> P;
  cudaStream_t s;
  const uint64_t n;
  Search(const M& m_, BuildCtx& ctx_, QuickBuild& qb_, SearchRun& R_)
      : m(m_), ctx(ctx_), qb(qb_), R(R_), P(m_, ctx_.t->B), s(ctx_.s), n(ctx_.t->n) {}

  static constexpr unsigned long long kAny = ~0ull;

  int keys(bool first, bool again, unsigned long long probes = kAny) {
    R.C.first = first;
    R.C.probes = probes;
    BT_LAUNCH(k_chase_init<<<grid_for(R.top, kT), kT, 0, s>>>(R.C, R.bwords, again));
    if (R.C.g.b <= 256) BT_LAUNCH(k_chase_keys<M, 1><<<grid_for(R.ni, kT), kT, 0, s>>>(m, P, ctx.Hs, R.C));
    else BT_LAUNCH(k_chase_keys<M, 32><<<grid_for(R.ni * 32, kT), kT, 0, s>>>(m, P, ctx.Hs, R.C));
    return BT_OK;
  }
  int scan(uint32_t e0, uint32_t e1, bool bounded, unsigned long long limit, ChaseState verdict) {
    if (e1 <= e0) return BT_OK;
    const uint32_t sw = R.bwords <= kChaseBitWords ? R.bwords : 0;
    const unsigned grid = (unsigned)std::min<uint64_t>((e1 - e0 + 8ull * kChaseTile - 1) / (8 * kChaseTile), 152 * 4);
    auto launch = [&](auto kernel) {
      BT_LAUNCH(kernel<<<grid, kT, sw * 4, s>>>(m, P, ctx.Hs, R.C, e0, e1, sw, bounded ? R.C.bound2 : nullptr, limit, verdict));
    };
    if (R.C.first) launch(k_chase_scan<M, std::true_type>);
    else launch(k_chase_scan<M, std::false_type>);
    return BT_OK;
  }
  // The second part against the bounds of what was found so far, unless that
  // was more work than `most`.
  int rest(unsigned long long most, unsigned long long limit) {
    BT_LAUNCH(k_chase_bound<<<grid_for(R.ni, kT), kT, 0, s>>>(R.C, most));
    BT_CUDA(cudaMemsetAsync(R.C.bitmap, 0, R.bwords * 4, s));
    BT_LAUNCH(k_chase_live<<<grid_for(R.gcap, kT), kT, 0, s>>>(R.C, R.split));
    return scan(R.split, R.total, true, limit, kGiveUp);
  }
  int finish() {
    const QGeo& g = R.C.g;
    if (R.C.r && R.C.r < kQuickMinB) BT_LAUNCH(k_chase_tail<<<grid_for(n / 16 + 1, kT, 152 * 8), kT, 0, s>>>(R.C));
    const uint64_t ppk = (2 * g.b + q_piece(g.b) - 1) / q_piece(g.b);
    const unsigned L = g.b >= 256 ? 32u : g.b >= 128 ? 16u : g.b >= 64 ? 8u : 4u;
    BT_LAUNCH(k_chase_verify<<<grid_for(R.ni * ppk * L, kT), kT, 0, s>>>(R.C, ppk, L));
    BT_LAUNCH(k_chase_apply<<<grid_for(R.ni, kT, 152 * 4), kT, 0, s>>>(R.C));
    BT_CUDA(cudaGetLastError());
    return BT_OK;
  }
  int wait() {
    BT_CUDA(cudaGetLastError());
    BT_CUDA(cudaMemcpyAsync(qb.qs_host, qb.qs, sizeof(QuickStatus), cudaMemcpyDeviceToHost, s));
    BT_CUDA(cudaStreamSynchronize(s));
    return BT_OK;
  }

  // By newest grams, all steps without a look at the host.
  int newest() {
    BT_TRY((allow_smem<k_chase_scan<M, std::false_type>>(kChaseBitWords * 4)));
    BT_TRY((allow_smem<k_chase_scan<M, std::true_type>>(kChaseBitWords * 4)));
    BT_TRY(keys(false, false, probes_most(R.ni)));
    {
      ProfScope prof("window_scan", s, 0);  // (the level's bytes are counted by its first part)
      BT_TRY(scan(0, R.split ? R.split : R.total, false, work_most(n, R.split != 0, kLeastWork), kTryFirst));
      if (R.split) BT_TRY(rest(work_sample(n), work_most(n, false, kLeastWork)));
    }
    return finish();
  }
  // What the host does when the status says that the search is not done;
  // kEveryWindow: that is the better way.
  int others() {
    const QuickStatus* q = qb.qs_host;
    if (q->redo == kGiveUp) return kEveryWindow;
    ProfScope prof("window_scan", s, 0);
    const unsigned long long few = R.split ? work_few(n) : work_most(n, false, kLeastWork);
    const unsigned long long by_newest = q->redo == kCompare ? q->work : kAny, before = q->work;
    BT_TRY(keys(true, true));
    BT_TRY(scan(0, R.split ? R.split : R.total, false, before + few, kGiveUp));
    BT_TRY(wait());
    const unsigned long long by_first = q->redo ? kAny : q->work - before;
    if (std::min(by_newest, by_first) > few) return kEveryWindow;
    if (R.split) {
      if (by_newest < by_first) BT_TRY(keys(false, true));
      BT_TRY(rest(kAny, q->work + work_most(n, false, kLeastWork)));
      BT_TRY(wait());
      if (q->redo) return kEveryWindow;
    }
    return finish();
  }
  // Without memory for the scan of every window: whatever it takes.
  int all() {
    BT_TRY(keys(false, true));
    BT_TRY(scan(0, R.total, false, kAny, kGiveUp));
    return finish();
  }
};

static int search_tables(BuildCtx& ctx, QuickBuild& qb, const QGeo& g, uint64_t last_start, const uint32_t* A,
                         const uint32_t* X, const uint32_t* items, uint64_t* lo, uint8_t* ps, SearchRun& R) {
  bt_tree* t = ctx.t;
  const uint64_t nb = qb.qs_host->nopen[0], np = qb.qs_host->nopen[1], ni = nb + np;
  const uint64_t len_last = g.n - last_start;
  Chase& C = R.C;
  C.g = g;
  C.Q = qb.list;
  C.A = A;
  C.X = X;
  C.items = items;
  C.nitems = (uint32_t)ni;
  C.r = len_last < g.b ? len_last : 0;
  auto power = [&](uint64_t e) { return t->q == Mersenne61::Q ? pow_mod(Mersenne61{}, t->B, e) : pow_mod(SmallMod{t->q}, t->B, e); };
  C.Bb = power(g.b);
  C.Br = C.r ? power(C.r) : 0;
  // (No more blocks are open, or halves of open pairs, than there are.)
  const uint64_t bcap = pow2_from(2 * std::min(nb + 2 * np, g.c)), pcap = pow2_from(2 * np), gcap = pow2_from(4 * ni);  // (2 ni: DNA 2 GiB 41.5 ms, not 40.8)
  uint32_t fbits = 12;
  while ((1ull << fbits) < 16 * ni && fbits < 30) fbits++;
  R.bwords = 1u << (fbits - 5);
  C.bmask = (uint32_t)(bcap - 1);
  C.pmask = (uint32_t)(pcap - 1);
  C.gmask = (uint32_t)(gcap - 1);
  C.bshift = 32 - fbits;
  C.qs = qb.qs;
  C.status = ctx.st;
  C.lo = lo;
  C.ps = ps;
  Arena& A2 = qb.open;
  auto carve = [&]() {
    C.bt = A2.take<CSlot>(bcap);
    C.pt = A2.take<CPair>(pcap);
    C.gt = A2.take<CGram>(gcap);
    C.bound2 = A2.take<unsigned long long>(gcap);
    C.bitmap = A2.take<uint32_t>(R.bwords);
    C.islot = A2.take<uint32_t>(ni);
    C.igram = A2.take<uint32_t>(ni);
    C.differ = A2.take<uint32_t>(ni);
    C.susp = A2.take<uint32_t>(ni);
    C.exlo = A2.take<unsigned long long>(ni);
  };
  A2.begin_dry();
  carve();
  BT_TRY(A2.reserve());
  carve();
  R.ni = ni;
  R.gcap = gcap;
  R.top = std::max<uint64_t>(std::max(bcap, pcap), std::max<uint64_t>(gcap, R.bwords));
  R.total = qb.qs_host->total;
  // (From 2^20 on, 8 MiB: ten words 7.0 ms, not 5.2, DNA copies 2.0, not 1.8; two-letter runs of 2 MiB 5.7, not 4.5.)
  R.split = R.total > (1u << 21) ? (R.total / 16) & ~(8 * kChaseTile - 1) : 0;
  return BT_OK;
}

enum class How { kNewest, kOthers, kAll };

template <class M>
static int search_as(const M& m, BuildCtx& ctx, QuickBuild& qb, SearchRun& R, How how) {
  Search<M> S(m, ctx, qb, R);
  return how == How::kNewest ? S.newest() : how == How::kOthers ? S.others() : S.all();
}

static int search_open(BuildCtx& ctx, QuickBuild& qb, SearchRun& R, How how) {
  const uint64_t q = ctx.t->q;
  return q == Mersenne61::Q ? search_as(Mersenne61{}, ctx, qb, R, how) : search_as(SmallMod{q}, ctx, qb, R, how);
}

// Exact leftmost occurrences of the keys whose fingerprint match was false.
static int search_exact(BuildCtx& ctx, const SearchRun& R, uint64_t nsusp) {
  const dim3 grid(grid_for(R.C.g.n, kT, 1024), (unsigned)std::min<uint64_t>(nsusp, 1024));
  BT_LAUNCH(k_chase_exact<<<grid, kT, 0, ctx.s>>>(R.C, nsusp));
  BT_LAUNCH(k_chase_exact_apply<<<grid_for(nsusp, kT), kT, 0, ctx.s>>>(R.C, nsusp));
  BT_CUDA(cudaGetLastError());
  return BT_OK;
}

// One level: marks, leftmost occurrences, pointers, the next level's blocks.
int quick_level(BuildCtx& ctx, QuickBuild& qb, uint32_t l, uint64_t last_start) {
  bt_tree* t = ctx.t;
  Level& v = t->lv[l];
  cudaStream_t s = ctx.s;
  const uint64_t c = v.c, b = v.b, n = t->n, words = (c + 31) / 32;
  const bool last_level = l + 1 == t->L;
  const uint64_t bn = last_level ? 0 : t->lv[l + 1].b;
  v.arity = last_level ? 0 : (uint32_t)(b / bn);
  const QGeo g{ctx.T, n, c, b, v.st};
  BT_TRY(alloc_level_arrays(v, words, s));
  uint32_t *A, *X, *flags, *items, *wpop, *sagg;
  uint8_t* ps;
  Arena& R = ctx.arena;
  auto carve = [&]() {
    A = R.take<uint32_t>(c);
    X = R.take<uint32_t>(c);
    flags = R.take<uint32_t>(c);
    items = R.take<uint32_t>(2 * c);
    ps = R.take<uint8_t>(c);
    wpop = R.take<uint32_t>(words);
    sagg = R.take<uint32_t>(scan_scratch_words(words));
  };
  R.begin_dry();
  carve();
  BT_TRY(R.reserve());
  carve();
  const unsigned gc = grid_for(c, kT);
  unsigned G = 1;
  while (G < 32 && 64ull * 2 * G <= b) G <<= 1;
  {
  ProfScope prof("window_scan", s, (c - 1) * b + (n - last_start < b ? n - last_start : b));
  BT_LAUNCH(k_quick_min<<<grid_for(c * G, kT), kT, 0, s>>>(g, qb.list, G, A, X, flags, qb.qs));
  // (A block is at most n long, so c ppk < 2^32.)
  const uint64_t bl = b < n ? b : n;
  const uint32_t ppk = (uint32_t)((2 * bl + q_piece(b) - 1) / q_piece(b));
  const unsigned L = b >= 1024 ? 32u : b >= 512 ? 16u : b >= 256 ? 8u : b >= 128 ? 4u : b >= 64 ? 2u : 1u;
  BT_LAUNCH(k_quick_compare<<<grid_for(c * ppk * L, kT), kT, 0, s>>>(g, A, X, flags, ppk, L));
  BT_LAUNCH(k_quick_settle<<<grid_for(c, kT, 152 * 8), kT, 0, s>>>(g, A, X, flags, v.lo, ps, items, v.mw, wpop, qb.qs, ctx.st));
  }
  auto rank_and_wait = [&]() -> int {
    if (words <= kRankWords) {
      BT_LAUNCH(k_quick_rank<<<1, 1024, 0, s>>>(g, v.mw, wpop, v.mr, v.arity, bn, ctx.st, qb.qs));
    } else {
      BT_TRY(scan_u32(wpop, v.mr, words, s, sagg));
      BT_LAUNCH(k_quick_end<<<1, 1, 0, s>>>(g, v.mw, v.mr, v.arity, bn, ctx.st, qb.qs));
    }
    BT_CUDA(cudaGetLastError());
    BT_CUDA(cudaMemcpyAsync(qb.qs_host, qb.qs, sizeof(QuickStatus), cudaMemcpyDeviceToHost, s));
    return sync_status(ctx);
  };
  BT_TRY(rank_and_wait());
  const QuickStatus q0 = *qb.qs_host;
  if (q0.nitems) {
    SearchRun run;
    BT_TRY(search_tables(ctx, qb, g, last_start, A, X, items, v.lo, ps, run));
    auto remark = [&]() -> int {
      BT_LAUNCH(k_quick_remark<<<grid_for(words * 32, kT), kT, 0, s>>>(c, ps, v.mw, wpop));
      return rank_and_wait();
    };
    BT_TRY(search_open(ctx, qb, run, How::kNewest));
    BT_TRY(remark());
    if (qb.qs_host->redo) {
      int rc = search_open(ctx, qb, run, How::kOthers);
      if (rc == kEveryWindow) {
        rc = qb.expand();
        if (rc == BT_OK) {
          qb.open.release();  // (room for the scan's tables)
          return kEveryWindow;
        }
        if (rc != BT_ENOMEM) return rc;
        cudaGetLastError();
        rc = search_open(ctx, qb, run, How::kAll);
      }
      BT_TRY(rc);
      BT_TRY(remark());
    }
    if (qb.qs_host->nsusp) {
      BT_TRY(search_exact(ctx, run, qb.qs_host->nsusp));
      BT_TRY(remark());
    }
  }
  uint64_t* next_st = nullptr;
  if (!last_level) {
    Level& nx = t->lv[l + 1];
    nx.c = ctx.st_host->next_c;
    if (nx.c == 0) return BT_EINTERNAL;
    BT_CUDA(cudaMallocAsync(&nx.st, nx.c * sizeof(uint64_t), s));
    nx.owned.push_back(nx.st);
    next_st = nx.st;
  }
  // Wide nodes (explicit block sizes) leave their children to a kernel that
  // deals them to the threads.
  const bool wide = v.arity > 64;
  BT_LAUNCH(k_quick_points<<<gc, kT, 0, s>>>(g, v.mw, v.mr, v.lo, v.ptr, v.off, v.arity, bn, wide ? nullptr : next_st,
                                             ctx.st));
  if (next_st && wide) BT_TRY(launch_children(ctx, l, bn, next_st));
  BT_CUDA(cudaGetLastError());
  v.nmarked = qb.qs_host->nmarked;
  v.stats[BT_ST_NBLOCKS] = c;
  v.stats[BT_ST_B] = b;
  v.stats[BT_ST_COV] = (c - 1) * b + (n - last_start < b ? n - last_start : b);
  v.stats[BT_ST_NMARKED] = v.nmarked;
  v.stats[BT_ST_NPAIRS] = q0.npairs;
  v.stats[BT_ST_VERIFY_BYTES] = ctx.st_host->verify_bytes - ctx.verify_bytes;
  v.stats[BT_ST_COLLISIONS] = ctx.st_host->collisions - ctx.collisions;
  v.stats[BT_ST_CANDIDATES] = q0.nitems ? qb.qs_host->cands : 0;
  v.stats[BT_ST_HITS] = q0.nitems ? qb.qs_host->hits : 0;
  ctx.prev_cands = v.stats[BT_ST_CANDIDATES];  // (a level of short blocks sizes its queue by it)
  ctx.verify_bytes = ctx.st_host->verify_bytes;
  ctx.collisions = ctx.st_host->collisions;
  if (ctx.st_host->error) {
    if (getenv("BT_VERBOSE"))
      fprintf(stderr, "bt: level %u (b=%llu, c=%llu): device check %llu failed\n", l, (unsigned long long)b,
              (unsigned long long)c, (unsigned long long)ctx.st_host->error);
    return BT_EINTERNAL;
  }
  return BT_OK;
}

}  // namespace bt
