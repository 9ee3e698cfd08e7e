// bt_prune_dev.cuh -- one level of the pruning pass by one CTA or a cluster of
// CTAs, for the batched kernel (bt_batch.cu) and the small levels of a single
// text (bt_prune.cu).
#pragma once

#include <cooperative_groups.h>

#include "bt_internal.cuh"

namespace bt {

// The CTAs that share a document: one (One), or a thread-block cluster (Cluster).
// Every thread of the group reaches every gsync.  Which of the two is known when
// the code is compiled: with the choice made at every barrier, and the shared
// state reached through a pointer that could lead to shared or global memory, a
// short document took 1.4 times as long in one CTA.
struct One {
  static constexpr bool many = false;
  static constexpr uint32_t rank = 0, size = 1;
  __device__ unsigned tid() const { return threadIdx.x; }
  __device__ unsigned threads() const { return blockDim.x; }
};
struct Cluster {
  static constexpr bool many = true;
  uint32_t rank, size;
  __device__ unsigned tid() const { return rank * blockDim.x + threadIdx.x; }
  __device__ unsigned threads() const { return size * blockDim.x; }
};

__device__ __forceinline__ Cluster this_cluster() {
  const cooperative_groups::cluster_group c = cooperative_groups::this_cluster();
  Cluster g;
  g.rank = c.block_rank();
  g.size = c.num_blocks();
  return g;
}

// Barrier of the group; what its threads wrote before is seen by all after.
__device__ __forceinline__ void gsync(const One&) { __syncthreads(); }
__device__ __forceinline__ void gsync(const Cluster&) { cooperative_groups::this_cluster().sync(); }

enum : uint32_t { P_UNDEC = 0, P_PRUNED = 1, P_KEPT = 2, P_NOTCAND = 3 };
constexpr uint32_t kFull = 0xFFFFFFFFu;

__device__ __forceinline__ bool marked(const uint32_t* mw, uint64_t k) { return (mw[k >> 5] >> (k & 31)) & 1u; }
__device__ __forceinline__ uint64_t mrank(const uint32_t* mw, const uint32_t* mr, uint64_t k) {
  return mr[k >> 5] + __popc(mw[k >> 5] & ((1u << (k & 31)) - 1u));
}

__device__ __forceinline__ char* carve(char*& p, uint64_t bytes) {
  char* q = p;
  p += (bytes + 255) & ~255ull;
  return q;
}

// Exclusive prefix sum of in[0, n) into out[0, n]; out[n] = total.  in and
// out may be the same array.  Four elements per thread and round.
__device__ inline void cta_scan_u32(const uint32_t* in, uint32_t* out, uint64_t n, uint32_t* wtot) {
  const unsigned lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  uint32_t carry = 0;
  for (uint64_t base = 0; base < n; base += 4 * blockDim.x) {
    const uint64_t i = base + 4 * threadIdx.x;
    uint32_t v[4];
#pragma unroll
    for (int u = 0; u < 4; u++) v[u] = i + u < n ? in[i + u] : 0u;
    const uint32_t sum = v[0] + v[1] + v[2] + v[3];
    uint32_t x = sum;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      const uint32_t o = __shfl_up_sync(0xFFFFFFFFu, x, d);
      if ((int)lane >= d) x += o;
    }
    if (lane == 31) wtot[warp] = x;
    __syncthreads();
    if (warp == 0) {
      uint32_t w = lane < nw ? wtot[lane] : 0u;
#pragma unroll
      for (int d = 1; d < 32; d <<= 1) {
        const uint32_t o = __shfl_up_sync(0xFFFFFFFFu, w, d);
        if ((int)lane >= d) w += o;
      }
      wtot[lane] = w;
    }
    __syncthreads();
    uint32_t o = carry + (warp ? wtot[warp - 1] : 0u) + x - sum;
#pragma unroll
    for (int u = 0; u < 4; u++) {
      if (i + u < n) out[i + u] = o;
      o += v[u];
    }
    carry += wtot[nw - 1];
    __syncthreads();
  }
  if (threadIdx.x == 0) out[n] = carry;
  __syncthreads();
}

// ---------------------------------------------------------------------------
// Pruning (section 3.1, "Optional Pruning"): for l = L-2 down to 0, a marked
// block k of level l becomes a pointer and loses its children when (i) none
// of its children has children, (ii) no pointer of level l (original, or made
// by pruning a block to its right) has a target window overlapping k, (iii)
// no pointer of level l+1 targets a child of k, and (iv) LO(S(k)) + |k| <=
// start(k).  Conditions (i), (iii), (iv) and the original pointers of (ii)
// leave a candidate set; a candidate is pruned iff no pruned candidate to its
// right targets it, resolved by frontier rounds (then right to left for what
// the round bound leaves).
// ---------------------------------------------------------------------------
// Shared-memory words of one CTA's scans.
constexpr uint32_t kScanWords = 32;

struct PrW {
  uint8_t *hit_v, *hit2, *tgt_w, *gone, *mk2;
  uint32_t *state, *indeg, *fq0, *fq1, *nidx, *wpop, *ptr2;
  uint64_t *t1, *t2, *st2, *off2, *lo2;
};

__device__ inline PrW carve_prune(char* temp, uint64_t cv, uint64_t cw) {
  PrW R;
  char* p = temp;
  R.hit_v = (uint8_t*)carve(p, cv + 8);
  R.hit2 = (uint8_t*)carve(p, cv + 8);
  R.tgt_w = (uint8_t*)carve(p, cw + 8);
  R.gone = (uint8_t*)carve(p, cw + 8);
  R.mk2 = (uint8_t*)carve(p, cw + 8);
  R.state = (uint32_t*)carve(p, cv * 4 + 4);
  R.indeg = (uint32_t*)carve(p, cv * 4 + 4);
  R.fq0 = (uint32_t*)carve(p, cv * 4 + 4);
  R.fq1 = (uint32_t*)carve(p, cv * 4 + 4);
  R.nidx = (uint32_t*)carve(p, cw * 4 + 4);
  R.wpop = (uint32_t*)carve(p, (cv > cw ? cv : cw) * 4 + 4);  // mark words of either level
  R.ptr2 = (uint32_t*)carve(p, cw * 4 + 4);
  R.t1 = (uint64_t*)carve(p, cv * 8 + 8);
  R.t2 = (uint64_t*)carve(p, cv * 8 + 8);
  R.st2 = (uint64_t*)carve(p, cw * 8 + 8);
  R.off2 = (uint64_t*)carve(p, cw * 8 + 8);
  R.lo2 = (uint64_t*)carve(p, cw * 8 + 8);
  return R;
}

struct PLv {
  uint64_t n, c, b;
  uint64_t* st;
  uint32_t* mw;
  uint32_t* mr;
  uint32_t* ptr;
  uint64_t* off;
  uint64_t* lo;
};

__device__ __forceinline__ uint64_t plen(const PLv& v, uint64_t k) {
  const uint64_t s = v.st[k];
  return v.n - s < v.b ? v.n - s : v.b;
}

// Shared state of a group that prunes (a CTA's in shared memory, a cluster's
// in global memory).
struct PruneShared {
  unsigned int wl[3];  // lengths of the rounds' worklists
  unsigned long long undecided;
  int err;
};

template <class GRP>
__device__ inline void flag_targets(const PLv& v, uint8_t* flag, const GRP& G) {
  for (uint64_t u = G.tid(); u < v.c; u += G.threads()) {
    if (marked(v.mw, u)) continue;
    const uint64_t j = v.ptr[u];
    flag[j] = 1;
    if (v.off[u] + plen(v, u) > plen(v, j)) flag[j + 1] = 1;
  }
}

// Level l = v, its children w; returns the blocks of w that stay (kNone: a
// device check failed).  v's marks, ranks, pointers and offsets are updated, w
// is compacted in place.
template <class GRP>
__device__ inline uint64_t prune_level(const PLv& v, const PLv& w, bool w_last, uint32_t arity, char* temp,
                                       uint64_t max_rounds, PruneShared& Z, uint32_t* wtot, const GRP& G) {
  const unsigned tid = G.tid(), nt = G.threads(), lane = tid & 31, nw = nt >> 5;
  // A check that failed anywhere: everyone's to know before anyone goes on.
  auto failed = [&]() {
    gsync(G);
    const int e = *(volatile int*)&Z.err;
    gsync(G);
    return e != 0;
  };
  const PrW R = carve_prune(temp, v.c, w.c);
  for (uint64_t i = tid; i <= v.c; i += nt) {
    R.hit_v[i] = 0;
    R.hit2[i] = 0;
    if (i < v.c) R.indeg[i] = 0;
  }
  for (uint64_t i = tid; i <= w.c; i += nt) {
    R.tgt_w[i] = 0;
    R.gone[i] = 0;
  }
  if (tid == 0) {
    Z.wl[0] = Z.wl[1] = Z.wl[2] = 0;
    Z.undecided = 0;
    Z.err = 0;
  }
  gsync(G);
  flag_targets(v, R.hit_v, G);
  flag_targets(w, R.tgt_w, G);
  gsync(G);
  // Candidates and their target blocks.
  for (uint64_t k = tid; k < v.c; k += nt) {
    R.state[k] = P_NOTCAND;
    if (!marked(v.mw, k) || R.hit_v[k]) continue;
    const uint64_t s = v.st[k], len = plen(v, k), lo = v.lo[k];
    if (lo == kNone) {
      Z.err = 1;
      continue;
    }
    if (lo + len > s) continue;  // (iv)
    const uint64_t first = mrank(v.mw, v.mr, k) * arity, nch = (len + w.b - 1) / w.b;
    bool ok = true;
    for (uint64_t i = 0; i < nch && ok; i++) {
      const uint64_t ch = first + i;
      if (!w_last && marked(w.mw, ch)) ok = false;  // (i)
      if (R.tgt_w[ch]) ok = false;                  // (iii)
    }
    if (!ok) continue;
    uint64_t a = 0, z = v.c;
    while (a < z) {
      const uint64_t mid = (a + z) / 2;
      if (v.st[mid] <= lo) a = mid + 1;
      else z = mid;
    }
    const uint64_t j = a - 1;
    R.t1[k] = j;
    R.t2[k] = (lo + len > v.st[j] + plen(v, j)) ? j + 1 : kNone;
    R.state[k] = P_UNDEC;
  }
  if (failed()) return kNone;
  for (uint64_t k = tid; k < v.c; k += nt) {
    if (R.state[k] != P_UNDEC) continue;
    if (R.state[R.t1[k]] != P_NOTCAND) atomicAdd(&R.indeg[R.t1[k]], 1u);
    if (R.t2[k] != kNone && R.state[R.t2[k]] != P_NOTCAND) atomicAdd(&R.indeg[R.t2[k]], 1u);
  }
  gsync(G);
  // Round 0: candidates nothing targets are pruned.
  for (uint64_t k = tid; k < v.c; k += nt)
    if (R.state[k] == P_UNDEC && R.indeg[k] == 0) {
      R.state[k] = P_PRUNED;
      R.fq0[atomicAdd(&Z.wl[0], 1u)] = (uint32_t)k;
    }
  gsync(G);
  // Rounds: the candidates decided in the previous round inform their
  // targets (a pruned attacker keeps its target; the last kept attacker of
  // a target prunes it).
  uint64_t r = 1;
  for (; r < max_rounds; r++) {
    const uint32_t m = *(volatile uint32_t*)&Z.wl[(r - 1) % 3];
    if (m == 0) break;
    if (tid == 0) Z.wl[r % 3] = 0;
    gsync(G);
    const uint32_t* qin = (r - 1) & 1 ? R.fq1 : R.fq0;
    uint32_t* qout = r & 1 ? R.fq1 : R.fq0;
    for (uint32_t i = tid; i < m; i += nt) {
      const uint64_t k = qin[i];
      const uint32_t sk = R.state[k];
      for (int e = 0; e < 2; e++) {
        const uint64_t t = e == 0 ? R.t1[k] : R.t2[k];
        if (t == kNone || R.state[t] == P_NOTCAND) continue;
        uint32_t target = 0;
        if (sk == P_PRUNED) target = P_KEPT;
        else if (atomicSub(&R.indeg[t], 1u) == 1u) target = P_PRUNED;
        if (target && atomicCAS(&R.state[t], (uint32_t)P_UNDEC, target) == P_UNDEC)
          qout[atomicAdd(&Z.wl[r % 3], 1u)] = (uint32_t)t;
      }
    }
    gsync(G);
  }
  // Right-to-left finish of the candidates the round bound left undecided.
  for (uint64_t k = tid; k < v.c; k += nt)
    if (R.state[k] == P_UNDEC) atomicAdd(&Z.undecided, 1ull);
  gsync(G);
  if (tid == 0 && Z.undecided) {
    for (uint64_t k = v.c; k-- > 0;) {
      uint32_t s = R.state[k];
      if (s == P_UNDEC) {
        s = R.hit2[k] ? P_KEPT : P_PRUNED;
        R.state[k] = s;
      }
      if (s == P_PRUNED) {
        R.hit2[R.t1[k]] = 1;
        if (R.t2[k] != kNone) R.hit2[R.t2[k]] = 1;
      }
    }
  }
  gsync(G);
  // Apply: pruned blocks lose their children and become pointers.
  for (uint64_t k = tid; k < v.c; k += nt) {
    if (R.state[k] != P_PRUNED) continue;
    const uint64_t first = mrank(v.mw, v.mr, k) * arity, nch = (plen(v, k) + w.b - 1) / w.b;
    for (uint64_t i = 0; i < nch; i++) R.gone[first + i] = 1;
    v.ptr[k] = (uint32_t)R.t1[k];
    v.off[k] = v.lo[k] - v.st[R.t1[k]];
  }
  gsync(G);
  const uint64_t words = (v.c + 31) / 32;
  for (uint64_t wb = tid >> 5; wb < words; wb += nw) {
    const uint64_t k = wb * 32 + lane;
    const bool mk = k < v.c && marked(v.mw, k) && R.state[k] != P_PRUNED;
    const uint32_t bits = __ballot_sync(kFull, mk);
    if (lane == 0) R.wpop[wb] = __popc(bits);
    __syncwarp();
    if (lane == 0) v.mw[wb] = bits;
  }
  gsync(G);
  if (G.rank == 0) cta_scan_u32(R.wpop, v.mr, words, wtot);
  // Compact level l+1 without the deleted children.
  for (uint64_t k = tid; k < w.c; k += nt) R.nidx[k] = R.gone[k] ? 0u : 1u;
  gsync(G);
  if (G.rank == 0) cta_scan_u32(R.nidx, R.nidx, w.c, wtot);
  if (GRP::many) gsync(G);
  for (uint64_t k = tid; k < w.c; k += nt) {
    if (R.gone[k]) continue;
    const uint64_t i = R.nidx[k];
    R.st2[i] = w.st[k];
    const bool mk = marked(w.mw, k);
    R.mk2[i] = mk;
    R.off2[i] = w.off[k];
    R.lo2[i] = w.lo[k];
    if (mk) {
      R.ptr2[i] = 0;
    } else {
      const uint32_t j = w.ptr[k];
      if (R.gone[j]) Z.err = 1;
      R.ptr2[i] = R.nidx[j];
    }
  }
  if (failed()) return kNone;
  const uint64_t c2 = R.nidx[w.c];
  const uint64_t words2 = (c2 + 31) / 32;
  for (uint64_t i = tid; i < c2; i += nt) {
    w.st[i] = R.st2[i];
    w.off[i] = R.off2[i];
    w.lo[i] = R.lo2[i];
    w.ptr[i] = R.ptr2[i];
  }
  for (uint64_t wb = tid >> 5; wb < words2; wb += nw) {
    const uint64_t k = wb * 32 + lane;
    const uint32_t bits = __ballot_sync(kFull, k < c2 && R.mk2[k]);
    if (lane == 0) {
      w.mw[wb] = bits;
      R.wpop[wb] = __popc(bits);
    }
  }
  gsync(G);
  if (G.rank == 0) cta_scan_u32(R.wpop, w.mr, words2, wtot);
  if (GRP::many) gsync(G);
  return c2;
}

}  // namespace bt
