// bt_query.cu -- alphabet map, rank/select counters, leaf text and queries.
//
// access, rank and select are the queries of section 1; the paper's
// implementation stores one bit vector per level plus pointers and offsets
// (section 4.4) and names the rank/select auxiliary data as future work
// (section 6).  The counters used here:
//   cnt[s][k]  occurrences of symbol s in block k (from the base level on),
//   pc[s][u]   occurrences of s in T[st[ptr], st[ptr] + off) for an unmarked
//              block u (the part of its target before the copied window),
//   pre[s][k]  occurrences of s before block k of the base level.
// rank_c(i) descends from the base-level block holding i: inside a marked block
// it adds the counts of the children left of the one holding i; at an
// unmarked block it continues in its target (ptr or ptr+1) and subtracts
// pc.  select mirrors it.  One thread answers one query.
#include <atomic>
#include <cstdlib>

#include "bt_internal.cuh"

namespace bt {

namespace {

// Which bytes occur (seen[0, 256), all zero at first), and by the last CTA to
// finish (seen[256] counts them) the dense symbol map.  Only presence matters:
// after a CTA's first lines every mark is set, and looking costs no atomics and
// no conflicts on frequent bytes.  Bound: the text's stream and a lookup per
// byte; 256 MiB of text in 64 us (107 with a word per symbol).
__global__ void __launch_bounds__(256) k_alphabet(const uint8_t* __restrict__ T, uint64_t n, uint32_t* seen,
                                                  int16_t* __restrict__ sym, Status* status) {
  __shared__ volatile uint8_t h[256];  // (a text's letters share a few words, which are broadcast)
  __shared__ uint32_t s_last, count[8];
  const unsigned tid = threadIdx.x;
  h[tid] = 0;
  __syncthreads();
  const uint64_t stride = (uint64_t)gridDim.x * 256, t0 = blockIdx.x * 256ull + tid;
  if (((uintptr_t)T & 15) == 0) {
    const uint4* V = (const uint4*)T;
    const uint64_t units = n / 16;
    for (uint64_t i = t0; i < units; i += 2 * stride) {
      const uint4 q[2] = {V[i], V[i + stride < units ? i + stride : i]};
#pragma unroll
      for (int u = 0; u < 2; u++) {
        const uint32_t w[4] = {q[u].x, q[u].y, q[u].z, q[u].w};
        uint32_t f = 1;
#pragma unroll
        for (int a = 0; a < 16; a++) f &= h[(w[a >> 2] >> (8 * (a & 3))) & 0xFF];
        if (f) continue;
#pragma unroll
        for (int a = 0; a < 16; a++) h[(w[a >> 2] >> (8 * (a & 3))) & 0xFF] = 1;
      }
    }
    for (uint64_t i = n / 16 * 16 + t0; i < n; i += stride) h[T[i]] = 1;
  } else {
    for (uint64_t i = t0; i < n; i += stride) h[T[i]] = 1;
  }
  __syncthreads();
  if (h[tid]) atomicExch(&seen[tid], 1u);
  __threadfence();
  __syncthreads();
  if (tid == 0) s_last = atomicAdd(&seen[256], 1u) == gridDim.x - 1;
  __syncthreads();
  if (!s_last) return;
  __threadfence();
  const bool mine = *(volatile uint32_t*)&seen[tid] != 0;
  // Rank among the bytes that occur.
  const unsigned bal = __ballot_sync(0xFFFFFFFFu, mine);
  if ((tid & 31) == 0) count[tid >> 5] = __popc(bal);
  __syncthreads();
  uint32_t before = 0, all = 0;
  for (uint32_t w = 0; w < 8; w++) {
    if (w < tid >> 5) before += count[w];
    all += count[w];
  }
  sym[tid] = mine ? (int16_t)(before + __popc(bal & ((1u << (tid & 31)) - 1u))) : (int16_t)-1;
  if (tid == 0) status->symbols = all;
}

// Up to four counters of one symbol as read, and how many of them count:
// their sum is taken when it is needed.
struct Run4 {
  uint32_t v[4];
  uint32_t m;
};
__device__ __forceinline__ void read_run(Run4& r, const void* cnt, uint32_t w, uint64_t i, uint32_t m) {
  r.m = m;
  if (w == 1) {
    r.v[0] = *(const uint32_t*)((const uint8_t*)cnt + i);
  } else if (w == 2) {
    const uint2 q = *(const uint2*)((const uint16_t*)cnt + i);
    r.v[0] = q.x, r.v[1] = q.y;
  } else {
    const uint4 q = *(const uint4*)((const uint32_t*)cnt + i);
    r.v[0] = q.x, r.v[1] = q.y, r.v[2] = q.z, r.v[3] = q.w;
  }
}
// What a level's counters are counted from.
struct CountLevel {
  const uint64_t* st;   // block starts of the level
  const uint32_t* ptr;  // targets and offsets of the unmarked blocks
  const uint64_t* off;
  const uint32_t* mw;
  uint64_t c, b, n, cp;
  void* cnt;            // symbol-major, cw bytes each
  void* pc;
  uint32_t cw;
  int only_unmarked;    // cnt of the marked blocks is summed from their children later
};

// The text counted for entry k of cnt (which = 0) or pc (1): [s0, s0 + len),
// perhaps empty; false for an entry that is not counted.
__device__ __forceinline__ bool count_range(const CountLevel& J, int which, uint64_t k, uint64_t* s0, uint32_t* len) {
  const bool mk = (J.mw[k >> 5] >> (k & 31)) & 1u;
  *s0 = 0;
  *len = 0;
  if (which == 0) {
    if (J.only_unmarked && mk) return false;
    *s0 = J.st[k];
    *len = (uint32_t)(J.n - *s0 < J.b ? J.n - *s0 : J.b);
    return true;
  }
  if (mk) return false;
  *s0 = J.st[J.ptr[k]];
  *len = (uint32_t)J.off[k];
  return true;
}

// One-byte counters (b <= 255): a thread per block.  The CTA's counters are a
// tile [S][128] in shared memory; thread t has the column 4 (t mod 32) + t/32,
// so that the lanes of a warp update 32 different banks, and rows leave as
// 128-byte lines.  blockIdx.y: cnt or pc.  Entries that are not counted are
// written as zeros; k_sum_children overwrites its own.  Bound: the counters'
// writes (S bytes per block).  Measured on the two lowest levels of the
// 256 MiB text: 670 us with block-major rows (zeroed byte by byte, four-way
// bank conflicts), 190 now.
constexpr uint32_t kSmallCountThreads = 128;

__global__ void __launch_bounds__(kSmallCountThreads) k_count_small(CountLevel J, const int16_t* __restrict__ sym_g,
                                                                    const uint8_t* __restrict__ T, uint32_t S) {
  extern __shared__ uint8_t tile[];  // [S][128], then the symbol map (one byte each)
  uint8_t* sym = tile + kSmallCountThreads * S;
  const uint32_t t = threadIdx.x, col = 4 * (t & 31) + (t >> 5);
  for (uint32_t i = t; i < 256; i += kSmallCountThreads) sym[i] = (uint8_t)sym_g[i];
  for (uint32_t i = t; i < 32 * S; i += kSmallCountThreads) ((uint32_t*)tile)[i] = 0;
  __syncthreads();
  const int which = blockIdx.y;
  uint8_t* out = (uint8_t*)(which ? J.pc : J.cnt);
  const uint64_t k0 = (uint64_t)blockIdx.x * kSmallCountThreads, k = k0 + col;
  if (k < J.c) {
    uint64_t s0;
    uint32_t len;
    count_range(J, which, k, &s0, &len);
    uint8_t* my = tile + col;
    uint32_t x = 0;
    if ((((uintptr_t)(T + s0)) & 15) == 0) {
      for (; x < len && s0 + x + 16 <= J.n; x += 16) {
        const uint4 v = *(const uint4*)(T + s0 + x);
        const uint32_t w[4] = {v.x, v.y, v.z, v.w};
        const uint32_t have = len - x;
#pragma unroll
        for (uint32_t i = 0; i < 16; i++)
          if (i < have) my[kSmallCountThreads * sym[(w[i >> 2] >> (8 * (i & 3))) & 0xFF]]++;
      }
    }
    for (; x < len; x++) my[kSmallCountThreads * sym[T[s0 + x]]]++;
  }
  __syncthreads();
  for (uint32_t i = t; i < 32 * S; i += kSmallCountThreads) {
    const uint64_t at = k0 + 4 * (i & 31);
    if (at < J.cp) *(uint32_t*)(out + (uint64_t)(i >> 5) * J.cp + at) = ((const uint32_t*)tile)[i];
  }
}

// Two-byte counters (blocks of 256 bytes to 64 KiB): a CTA takes a tile of
// consecutive blocks and writes its counters of a symbol as one run.  Bound by
// the chain of dependent reads before a block's text (mark, target, start): the
// lanes of a warp walk it for all the warp's blocks at once, and the texts of
// the next blocks are in flight while the current ones are counted.  Few
// symbols (DNA) are counted by comparing words with each symbol, a group of
// lanes per block, without memory; more go to four copies of a histogram in
// shared memory (lanes take different copies: a frequent symbol's updates meet
// less often), two blocks at a time.  blockIdx.y: cnt or pc.
constexpr uint32_t kFewSymbols = 8;
constexpr uint32_t kTileFew = 128, kTileMany = 64;  // blocks per tile
constexpr uint64_t kCountPiece = 1 << 16;

// 16 text bytes from x of a range (zeros past it); bytes outside are not read.
__device__ __forceinline__ uint4 range16(const uint8_t* __restrict__ T, uint64_t s0, uint32_t len, uint32_t x, bool al) {
  if (x >= len) return make_uint4(0, 0, 0, 0);
  if (al && x + 16 <= len) return *(const uint4*)(T + s0 + x);
  uint32_t w[4] = {0, 0, 0, 0};
#pragma unroll
  for (uint32_t q = 0; q < 16; q++)
    if (x + q < len) w[q >> 2] |= (uint32_t)T[s0 + x + q] << (8 * (q & 3));
  return make_uint4(w[0], w[1], w[2], w[3]);
}

template <bool FEW>
__global__ void __launch_bounds__(256) k_count_tile(CountLevel J, const int16_t* __restrict__ sym_g,
                                                    const uint8_t* __restrict__ T, uint32_t S) {
  constexpr uint32_t TB = FEW ? kTileFew : kTileMany, PW = TB / 8;  // blocks per tile and per warp
  extern __shared__ uint32_t hist[];  // per warp two [S][4] (not FEW), then [S][TB] of two bytes, then the symbol map
  __shared__ uint8_t byte_of[kFewSymbols];
  const unsigned lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  uint32_t* h = hist + warp * 8 * S;
  uint16_t* rows = (uint16_t*)(hist + (FEW ? 0 : 8 * 8 * S));
  uint8_t* sym = (uint8_t*)(rows + S * TB);
  for (uint32_t i = threadIdx.x; i < 256; i += 256) {
    const int v = sym_g[i];
    sym[i] = (uint8_t)v;
    if (FEW && v >= 0) byte_of[v] = (uint8_t)i;
  }
  const int which = blockIdx.y;
  uint16_t* out = (uint16_t*)(which ? J.pc : J.cnt);
  const uint64_t tiles = (J.c + TB - 1) / TB;
  // Lanes per block of the comparing kernel: one 16-byte unit each at first.
  unsigned L = 32;
  while (L > 1 && 16ull * (L / 2) >= J.b) L >>= 1;
  for (uint64_t tl = blockIdx.x; tl < tiles; tl += gridDim.x) {
    __syncthreads();
    bool any = false;
    uint64_t rs = 0;
    uint32_t rl = 0;
    if (lane < PW) {
      const uint64_t k = tl * TB + warp * PW + lane;
      if (k < J.c) any = count_range(J, which, k, &rs, &rl);
    }
    if (FEW) {
      const unsigned gl = lane % L, grp = lane / L, gpw = 32 / L;
      for (uint32_t i0 = 0; i0 < PW; i0 += 2 * gpw) {
        uint32_t acc[2][kFewSymbols] = {};
        uint64_t s0[2];
        uint32_t len[2];
        bool al[2];
#pragma unroll
        for (int u = 0; u < 2; u++) {
          const uint32_t i = i0 + u * gpw + grp;
          s0[u] = __shfl_sync(0xFFFFFFFFu, rs, i & 31);
          len[u] = __shfl_sync(0xFFFFFFFFu, rl, i & 31);
          if (i >= PW) len[u] = 0;
          al[u] = (((uintptr_t)(T + s0[u])) & 15) == 0;
        }
        const uint32_t top = len[0] > len[1] ? len[0] : len[1];
        for (uint32_t x = 16 * gl; x < top; x += 16 * L) {
          uint4 v[2];
#pragma unroll
          for (int u = 0; u < 2; u++) v[u] = range16(T, s0[u], len[u], x, al[u]);
#pragma unroll
          for (int u = 0; u < 2; u++) {
            if (x >= len[u]) continue;
            const uint32_t have = len[u] - x;  // bytes of the unit that count
            const uint32_t w[4] = {v[u].x, v[u].y, v[u].z, v[u].w};
            uint32_t keep[4];
#pragma unroll
            for (uint32_t q = 0; q < 4; q++)
              keep[q] = have >= 4 * q + 4 ? 0xFFFFFFFFu : have <= 4 * q ? 0u : (1u << (8 * (have - 4 * q))) - 1u;
#pragma unroll
            for (uint32_t s = 0; s < kFewSymbols; s++) {
              if (s >= S) break;
              const uint32_t cc = byte_of[s] * 0x01010101u;
#pragma unroll
              for (uint32_t q = 0; q < 4; q++) acc[u][s] += __popc(__vcmpeq4(w[q], cc) & keep[q]);
            }
          }
        }
#pragma unroll
        for (int u = 0; u < 2; u++) {
          const uint32_t i = i0 + u * gpw + grp;
#pragma unroll
          for (uint32_t s = 0; s < kFewSymbols; s++) {
            if (s >= S) break;
            uint32_t v = acc[u][s];
            for (unsigned o = L / 2; o; o >>= 1) v += __shfl_xor_sync(0xFFFFFFFFu, v, o);
            if (gl == 0 && i < PW) rows[s * TB + warp * PW + i] = (uint16_t)(v >> 3);
          }
        }
      }
    } else {
      const uint32_t cpy = lane & 3;
      uint4 next[2];  // the first 512 bytes of the next two blocks
#pragma unroll
      for (int u = 0; u < 2; u++) {
        const uint64_t s0 = __shfl_sync(0xFFFFFFFFu, rs, u);
        const uint32_t len = __shfl_sync(0xFFFFFFFFu, rl, u);
        next[u] = range16(T, s0, len, 16 * lane, (((uintptr_t)(T + s0)) & 15) == 0);
      }
      for (uint32_t i = 0; i < PW; i += 2) {
        for (uint32_t z = lane; z < 2 * S; z += 32) ((uint4*)h)[z] = make_uint4(0, 0, 0, 0);
        uint4 cur[2] = {next[0], next[1]};
        if (i + 2 < PW) {
#pragma unroll
          for (int u = 0; u < 2; u++) {
            const uint64_t s0 = __shfl_sync(0xFFFFFFFFu, rs, i + 2 + u);
            const uint32_t len = __shfl_sync(0xFFFFFFFFu, rl, i + 2 + u);
            next[u] = range16(T, s0, len, 16 * lane, (((uintptr_t)(T + s0)) & 15) == 0);
          }
        }
        __syncwarp();
#pragma unroll
        for (int u = 0; u < 2; u++) {
          const uint64_t s0 = __shfl_sync(0xFFFFFFFFu, rs, i + u);
          const uint32_t len = __shfl_sync(0xFFFFFFFFu, rl, i + u);
          uint32_t* hu = h + 4 * S * u + cpy;
          const bool al = (((uintptr_t)(T + s0)) & 15) == 0;
          for (uint32_t x = 16 * lane; x < len; x += 512) {
            const uint4 v = x < 512 ? cur[u] : range16(T, s0, len, x, al);
            const uint32_t w[4] = {v.x, v.y, v.z, v.w};
            const uint32_t have = len - x;
#pragma unroll
            for (uint32_t q = 0; q < 16; q++)
              if (q < have) atomicAdd(&hu[4 * sym[(w[q >> 2] >> (8 * (q & 3))) & 0xFF]], 1u);
          }
        }
        __syncwarp();
        for (uint32_t s = lane; s < S; s += 32) {
          const uint4 a = ((const uint4*)h)[s], b = ((const uint4*)h)[S + s];
          *(uint32_t*)(rows + s * TB + warp * PW + i) = (a.x + a.y + a.z + a.w) | ((b.x + b.y + b.z + b.w) << 16);
        }
        __syncwarp();
      }
    }
    // (A tile without counted entries needs no write: those of marked blocks
    // are summed from the children or never read.)
    if (!__syncthreads_or(any)) continue;
    const uint64_t have = (J.cp - tl * TB) / 2;  // words of the row from the tile on
    for (uint32_t i = threadIdx.x; i < S * (TB / 2); i += 256) {
      const uint32_t s = i / (TB / 2), w = i % (TB / 2);
      if (w >= have) continue;
      ((uint32_t*)(out + (uint64_t)s * J.cp + tl * TB))[w] = ((const uint32_t*)rows)[i];
    }
  }
}

// Blocks longer than a piece: one warp per (block, piece of 64 KiB), added to
// four-byte counters that start at zero.  blockIdx.y: cnt or pc.
__global__ void __launch_bounds__(256) k_count_long(CountLevel J, const int16_t* __restrict__ sym,
                                                    const uint8_t* __restrict__ T, uint32_t S, uint64_t ppb) {
  extern __shared__ uint32_t hist[];  // 8 warps x S
  const unsigned lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  uint32_t* h = hist + wid * S;
  uint32_t* out = (uint32_t*)(blockIdx.y ? J.pc : J.cnt);
  const uint64_t warps = (uint64_t)gridDim.x * (blockDim.x / 32);
  for (uint64_t w = (blockIdx.x * (uint64_t)blockDim.x + threadIdx.x) / 32; w < J.c * ppb; w += warps) {
    const uint64_t k = w / ppb, a = (w - k * ppb) * kCountPiece;
    uint64_t s0;
    uint32_t len;
    count_range(J, blockIdx.y, k, &s0, &len);
    if (a >= len) continue;
    const uint64_t e = a + kCountPiece < len ? a + kCountPiece : len;
    for (uint32_t i = lane; i < S; i += 32) h[i] = 0;
    __syncwarp();
    for (uint64_t x = a + lane; x < e; x += 32) atomicAdd(&h[sym[T[s0 + x]]], 1u);
    __syncwarp();
    for (uint32_t i = lane; i < S; i += 32)
      if (h[i]) atomicAdd(&out[(uint64_t)i * J.cp + k], h[i]);
    __syncwarp();
  }
}

// Marked blocks of a non-last level: sums of their children's counters.  A
// thread per block and group of symbols (blockIdx.y): neighbouring marked
// blocks read neighbouring children.  Four symbols at a time, so that their
// reads are in flight together: bound by latency, 278 us with one at a time on
// 0.88 M blocks of 96 symbols.
template <uint32_t CW, uint32_t CCW>
__global__ void __launch_bounds__(256) k_sum_children(CountLevel J, const uint32_t* __restrict__ mr, uint32_t arity,
                                                      uint64_t bn, const void* __restrict__ child_cnt, uint64_t child_cp,
                                                      uint32_t S) {
  const uint32_t s0 = (uint32_t)((uint64_t)S * blockIdx.y / gridDim.y), s1 = (uint32_t)((uint64_t)S * (blockIdx.y + 1) / gridDim.y);
  for (uint64_t k = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; k < J.c; k += (uint64_t)gridDim.x * blockDim.x) {
    const uint32_t word = J.mw[k >> 5];
    if (!((word >> (k & 31)) & 1u)) continue;
    const uint64_t len = J.n - J.st[k] < J.b ? J.n - J.st[k] : J.b;
    const uint64_t first = (mr[k >> 5] + __popc(word & ((1u << (k & 31)) - 1u))) * (uint64_t)arity;
    const uint32_t nch = (uint32_t)((len + bn - 1) / bn);
    uint32_t s = s0;
    if (nch == 4 && arity == 4) {  // one read per symbol
      for (; s + 4 <= s1; s += 4) {
        Run4 v[4];
#pragma unroll
        for (uint32_t u = 0; u < 4; u++) read_run(v[u], child_cnt, CCW, (uint64_t)(s + u) * child_cp + first, 4);
#pragma unroll
        for (uint32_t u = 0; u < 4; u++) {
          const uint32_t x = CCW == 1   ? __dp4a(v[u].v[0], 0x01010101u, 0u)
                             : CCW == 2 ? (v[u].v[0] & 0xFFFFu) + (v[u].v[0] >> 16) + (v[u].v[1] & 0xFFFFu) + (v[u].v[1] >> 16)
                                        : v[u].v[0] + v[u].v[1] + v[u].v[2] + v[u].v[3];
          cput(J.cnt, CW, (uint64_t)(s + u) * J.cp + k, x);
        }
      }
    }
    for (; s < s1; s++)
      cput(J.cnt, CW, (uint64_t)s * J.cp + k, sum_run(child_cnt, CCW, (uint64_t)s * child_cp + first, nch));
  }
}

// pre[s][k]: exclusive prefix sums of the base level's counters, a CTA per
// symbol, eight counters per thread and step: the base level grows with the text
// (16 M blocks for 2 GiB of four random letters), and with one counter a step 2 M
// blocks took 461 us, now 318.
__global__ void __launch_bounds__(1024) k_base_prefix(uint64_t c, const void* __restrict__ cnt, uint32_t cw, uint64_t cp,
                                                      uint32_t* __restrict__ pre) {
  __shared__ uint32_t sm[32];
  const unsigned lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  const uint64_t s = blockIdx.x;
  uint32_t carry = 0;
  for (uint64_t base = 0; base < c; base += 8ull * blockDim.x) {
    const uint64_t k = base + 8ull * threadIdx.x;
    uint32_t v[8], sum = 0;
#pragma unroll
    for (int u = 0; u < 8; u++) {
      v[u] = k + u < c ? cget(cnt, cw, s * cp + k + u) : 0u;
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
      uint32_t w = lane < nw ? sm[lane] : 0;
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
      if (k + u < c) pre[s * (c + 1) + k + u] = at;
      at += v[u];
    }
    carry += sm[nw - 1];
    __syncthreads();
  }
  if (threadIdx.x == 0) pre[s * (c + 1) + c] = carry;
}

// Text of the marked last-level blocks, block of rank r at r b.  VEC: b, and
// so every start, is a multiple of 16 and the text aligned: 16 bytes per thread.
template <bool VEC>
__global__ void __launch_bounds__(256) k_leaf_text(uint64_t c, uint64_t b, uint64_t n, const uint64_t* __restrict__ st,
                                                   const uint32_t* __restrict__ mw, const uint32_t* __restrict__ mr,
                                                   const uint8_t* __restrict__ T, uint8_t* __restrict__ leaf) {
  const uint32_t unit = VEC ? 16 : 1;
  const uint64_t per = b / unit;
  const uint32_t shift = (per & (per - 1)) == 0 ? 63 - __clzll(per) : 64;
  for (uint64_t w = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; w < c * per;
       w += (uint64_t)gridDim.x * blockDim.x) {
    const uint64_t k = shift < 64 ? w >> shift : w / per, i = (w - k * per) * unit;
    const uint32_t word = mw[k >> 5];
    if (!((word >> (k & 31)) & 1u)) continue;
    const uint64_t x = st[k] + i;
    if (x >= n) continue;
    uint8_t* to = leaf + (uint64_t)(mr[k >> 5] + __popc(word & ((1u << (k & 31)) - 1u))) * b + i;
    if (VEC && x + 16 <= n) {
      *(uint4*)to = *(const uint4*)(T + x);
    } else {
      for (uint32_t q = 0; q < unit && x + q < n; q++) to[q] = T[x + q];
    }
  }
}

// ---------------------------------------------------------------------------
// Queries.
// ---------------------------------------------------------------------------
__device__ __forceinline__ uint32_t qlen(const LevelView& v, uint32_t k) { return k + 1 == v.c ? v.last_len : v.b; }

// x / b for the block length of a level (a shift when b is a power of two).
__device__ __forceinline__ uint32_t div_b(uint32_t x, const LevelView& v) {
  return v.bshift != 0xFFu ? x >> v.bshift : x / v.b;
}

// The bytes of one aligned 16-byte unit that equal c, 0xFF each, those before
// byte `from` and from byte `to` on cleared.
struct Eq16 {
  uint32_t e[4];
};
__device__ __forceinline__ Eq16 unit_equals(const uint8_t* p, uint32_t cc, uint32_t from, uint32_t to) {
  const uint4 v = *(const uint4*)p;
  const uint32_t w[4] = {v.x, v.y, v.z, v.w};
  Eq16 r;
#pragma unroll
  for (uint32_t q = 0; q < 4; q++) {
    r.e[q] = __vcmpeq4(w[q], cc);
    if (from > 4 * q) r.e[q] = from >= 4 * q + 4 ? 0u : r.e[q] & (0xFFFFFFFFu << (8 * (from - 4 * q)));
    if (to < 4 * q + 4) r.e[q] = to <= 4 * q ? 0u : r.e[q] & ((1u << (8 * (to - 4 * q))) - 1u);
  }
  return r;
}
__device__ __forceinline__ uint32_t matches(const Eq16& r) {
  return (__popc(r.e[0]) + __popc(r.e[1]) + __popc(r.e[2]) + __popc(r.e[3])) >> 3;
}

// Occurrences of byte c in p[0, o): aligned 16-byte units whatever p's alignment,
// four in flight on long stretches.  (The leaf text starts at such a unit and is
// followed by 16 bytes, so the first and the last one are readable.)  When only
// aligned starts took whole units, the lanes of a warp did both loops one after the
// other: 300 k ranks on DNA copies with leaves of 200 bytes and no stored leaf
// counters took 343 us, now 117.
__device__ __forceinline__ uint32_t leaf_count(const uint8_t* p, uint32_t o, uint32_t c) {
  if (o == 0) return 0;
  const uint32_t d = (uint32_t)((uintptr_t)p & 15), end = d + o, cc = c * 0x01010101u;
  const uint8_t* u = p - d;
  uint32_t acc = matches(unit_equals(u, cc, d, end)), y = 16;
  for (; y + 64 <= end; y += 64) {
    const uint4* q = (const uint4*)(u + y);
    const uint4 v[4] = {q[0], q[1], q[2], q[3]};
    uint32_t a = 0;
#pragma unroll
    for (int i = 0; i < 4; i++)
      a += __popc(__vcmpeq4(v[i].x, cc)) + __popc(__vcmpeq4(v[i].y, cc)) + __popc(__vcmpeq4(v[i].z, cc)) +
           __popc(__vcmpeq4(v[i].w, cc));
    acc += a >> 3;
  }
  for (; y < end; y += 16) acc += matches(unit_equals(u + y, cc, 0, end - y));
  return acc;
}

// Position of the j-th occurrence (j >= 1) of byte c in p[0, len), or kNoSlot.
__device__ __forceinline__ uint32_t leaf_find(const uint8_t* p, uint32_t len, uint32_t c, uint32_t j) {
  const uint32_t d = (uint32_t)((uintptr_t)p & 15), end = d + len, cc = c * 0x01010101u;
  const uint8_t* u = p - d;
  for (uint32_t y = 0; y < end; y += 16) {
    const uint4 v = *(const uint4*)(u + y);
    Eq16 r{{__vcmpeq4(v.x, cc), __vcmpeq4(v.y, cc), __vcmpeq4(v.z, cc), __vcmpeq4(v.w, cc)}};
    if (y < d) r = unit_equals(u, cc, d, 16);  // (the bytes before p)
    const uint32_t k = matches(r);
    if (k < j) {
      j -= k;
      continue;
    }
#pragma unroll
    for (uint32_t q = 0; q < 4; q++) {
      const uint32_t kq = __popc(r.e[q]) >> 3;
      if (j > kq) {
        j -= kq;
        continue;
      }
      uint32_t m = r.e[q] & 0x01010101u;
      for (; j > 1; j--) m &= m - 1;
      const uint32_t at = y + 4 * q + (__ffs(m) - 1) / 8 - d;
      return at < len ? at : kNoSlot;
    }
  }
  return kNoSlot;
}

// Space-efficient counters (BT_FLAG_LEAF_COUNTS): the last level stores no
// symbol counters; they are counted in the leaf text when a query needs them.
// A marked last-level block's text is its leaf text; an unmarked one copies a
// window of at most two marked blocks (its target and the next one), whose
// text is in the leaf text too.
__device__ __noinline__ uint32_t leaf_block_count(const uint8_t* leaf, const LevelView& v, uint32_t k, uint32_t c) {
  const uint32_t len = qlen(v, k);
  const uint2 r = v.rec[k];
  // The two blocks have ranks r and r + 1, so that their text is one stretch of the
  // leaf text, and the lanes of a warp, some at marked blocks and some at copies,
  // count together: 1 M ranks on 64 MiB of DNA copies, leaves of 64 bytes, 336 us with
  // up to three stretches, 250 now.
  const uint8_t* p = leaf + (uint64_t)r.y * v.b;
  if (r.x != kMarkedRec) p = leaf + (uint64_t)v.rec[r.x].y * v.b + r.y;
  return leaf_count(p, len, c);
}

// Counts of byte c in the target of an unmarked last-level block before the window.
__device__ __noinline__ uint32_t leaf_prefix_count(const uint8_t* leaf, const LevelView& v, uint2 r, uint32_t c) {
  return leaf_count(leaf + (uint64_t)v.rec[r.x].y * v.b, r.y, c);
}

// Counter of symbol s (byte c) of block k: stored, or counted in the leaf text.
__device__ __forceinline__ uint32_t blk_cnt(const uint8_t* leaf, const LevelView& v, uint32_t k, uint32_t s, uint32_t c) {
  return v.cnt ? cget(v.cnt, v.cw, (uint64_t)s * v.cp + k) : leaf_block_count(leaf, v, k, c);
}
__device__ __forceinline__ uint32_t blk_pc(const uint8_t* leaf, const LevelView& v, uint32_t k, uint2 r, uint32_t s,
                                           uint32_t c) {
  return v.pc ? cget(v.pc, v.cw, (uint64_t)s * v.cp + k) : leaf_prefix_count(leaf, v, r, c);
}

// What a descent needs of the tree besides the level table.
struct QTree {
  uint64_t n;
  uint32_t L;           // levels from the base on (the level table starts there)
  const uint32_t* pre;
  const uint8_t* leaf;
  const int16_t* sym;
};

// A descent keeps the offset o inside the current block instead of a text
// position, so no block starts are read: one 8-byte record per step.
__device__ __forceinline__ uint64_t q_access(const QTree& t, const LevelView* __restrict__ lv, uint64_t i) {
  if (i >= t.n) return kNone;
  uint32_t l = 0, k = div_b((uint32_t)i, lv[0]), o = (uint32_t)i - k * lv[0].b;
  for (uint32_t step = 0; step < 4 * t.L + 4; step++) {
    const LevelView& v = lv[l];
    const uint2 r = v.rec[k];
    if (r.x == kMarkedRec) {
      if (l + 1 == t.L) return t.leaf[(uint64_t)r.y * v.b + o];
      l++;
      const uint32_t j = div_b(o, lv[l]);
      k = r.y * v.arity + j;
      o -= j * lv[l].b;
    } else {
      const uint32_t lp = qlen(v, r.x), x = r.y + o;
      k = r.x + (x >= lp);
      o = x >= lp ? x - lp : x;
    }
  }
  return kNone;
}

__device__ __forceinline__ uint32_t run_sum(const Run4& r, uint32_t w) {  // of the first m <= 3
  if (r.m == 0) return 0;
  if (w == 1) return __dp4a(r.v[0] & ((1u << (8 * r.m)) - 1u), 0x01010101u, 0u);
  if (w == 2) return (r.v[0] & 0xFFFFu) + (r.m > 1 ? r.v[0] >> 16 : 0) + (r.m > 2 ? r.v[1] & 0xFFFFu : 0);
  return r.v[0] + (r.m > 1 ? r.v[1] : 0) + (r.m > 2 ? r.v[2] : 0);
}

// rank descends likewise.  Its counters are off the chain of dependent reads:
// they are added one step later, when the next record has been read too.
__device__ __forceinline__ uint64_t q_rank(const QTree& t, const LevelView* __restrict__ lv, uint32_t c, uint64_t i) {
  if (i > t.n) return kNone;
  const int s = t.sym[c];
  if (s < 0) return 0;
  const uint32_t* pre = t.pre + (uint64_t)s * (lv[0].c + 1);
  if (i == t.n) return pre[lv[0].c];
  uint32_t l = 0, k = div_b((uint32_t)i, lv[0]), o = (uint32_t)i - k * lv[0].b;
  uint32_t acc = pre[k];  // (sums may pass below zero on the way: modulo 2^32, the answer is at most n)
  Run4 run;
  run.m = 0;
  uint32_t rw = 1, p0 = 0, m0 = 0;  // counters in flight: a run of width rw and p0 to add, m0 to subtract
  for (uint32_t step = 0; step < 4 * t.L + 4; step++) {
    const LevelView& v = lv[l];
    if (o == 0) return acc + run_sum(run, rw) + p0 - m0;
    if (o == qlen(v, k)) return acc + run_sum(run, rw) + p0 - m0 + blk_cnt(t.leaf, v, k, s, c);
    const uint2 r = v.rec[k];
    acc += run_sum(run, rw) + p0 - m0;
    run.m = p0 = m0 = 0;
    if (r.x == kMarkedRec) {
      if (l + 1 == t.L) return acc + leaf_count(t.leaf + (uint64_t)r.y * v.b, o, c);
      const uint32_t f = r.y * v.arity, ar = v.arity;
      const LevelView& w = lv[++l];
      const uint32_t j = div_b(o, w);
      o -= j * w.b;
      k = f + j;
      if (w.cnt) {
        uint64_t at = (uint64_t)s * w.cp + f;
        uint32_t left = j;
        if ((ar & 3) == 0) {
          if (left >= 4) {
            acc += sum_run(w.cnt, w.cw, at, left & ~3u);
            at += left & ~3u;
            left &= 3u;
          }
          if (left) read_run(run, w.cnt, rw = w.cw, at, left);
        } else {
          acc += sum_run(w.cnt, w.cw, at, left);
        }
      } else {
        for (uint32_t x = 0; x < j; x++) acc += leaf_block_count(t.leaf, w, f + x, c);
      }
    } else {
      m0 = blk_pc(t.leaf, v, k, r, s, c);
      const uint32_t lp = qlen(v, r.x), x = r.y + o;
      if (x <= lp) {
        k = r.x;
        o = x;
      } else {
        p0 = blk_cnt(t.leaf, v, r.x, s, c);
        k = r.x + 1;
        o = x - lp;
      }
    }
  }
  return kNone;
}

// select needs the counters to find its way: those of up to three children
// are read together, and an unmarked block's prefix counter with its record.
__device__ __forceinline__ uint64_t q_select(const QTree& t, const LevelView* __restrict__ lv, uint32_t c, uint64_t jq) {
  const int s = t.sym[c];
  if (s < 0 || jq == 0) return kNone;
  const LevelView& top = lv[0];
  const uint32_t* pre = t.pre + (uint64_t)s * (top.c + 1);
  if (jq > pre[top.c]) return kNone;
  uint32_t a = 0, z = top.c;  // last k with pre[k] < j: four parts per step, their bounds read together
  const uint32_t jw = (uint32_t)jq;
  while (z - a > 1) {
    const uint32_t d = z - a, q1 = a + ((d + 3) >> 2), q2 = a + ((d + 1) >> 1), q3 = a + d - (d >> 2);
    const uint32_t v1 = pre[q1], v2 = pre[q2], v3 = pre[q3 < z ? q3 : z - 1];
    if (v2 < jw) {
      a = q2;
      if (q3 < z && q3 > q2) {
        if (v3 < jw) a = q3;
        else z = q3;
      }
    } else {
      z = q2;
      if (q1 < q2) {
        if (v1 < jw) a = q1;
        else z = q1;
      }
    }
  }
  uint32_t k = a, l = 0;
  uint32_t j = jw - pre[k];
  int64_t res = (int64_t)k * top.b;
  for (uint32_t step = 0; step < 4 * t.L + 4; step++) {
    const LevelView& v = lv[l];
    const uint2 r = v.rec[k];
    const uint32_t pck = v.pc ? cget(v.pc, v.cw, (uint64_t)s * v.cp + k) : 0;
    if (r.x == kMarkedRec) {
      if (l + 1 == t.L) {
        const uint32_t x = leaf_find(t.leaf + (uint64_t)r.y * v.b, qlen(v, k), c, j);
        return x == kNoSlot ? kNone : (uint64_t)(res + x);
      }
      const uint32_t f = r.y * v.arity, ar = v.arity;
      const LevelView& w = lv[++l];
      uint32_t i = 0;
      bool found = false;
      if (w.cnt) {
        const uint64_t at = (uint64_t)s * w.cp + f;
        // (A short last block has fewer children: the entries behind them are
        // the row's padding or not counted; the j-th symbol lies before them.)
        const uint32_t have = w.c - f < ar ? w.c - f : ar;
        while (i < have && !found) {
          uint32_t cc[4];
          if ((ar & 3) == 0) {
            Run4 run;
            read_run(run, w.cnt, w.cw, at + i, 4);
            if (w.cw == 1) {
#pragma unroll
              for (uint32_t u = 0; u < 4; u++) cc[u] = (run.v[0] >> (8 * u)) & 0xFFu;
            } else if (w.cw == 2) {
              cc[0] = run.v[0] & 0xFFFFu, cc[1] = run.v[0] >> 16, cc[2] = run.v[1] & 0xFFFFu, cc[3] = run.v[1] >> 16;
            } else {
#pragma unroll
              for (uint32_t u = 0; u < 4; u++) cc[u] = run.v[u];
            }
          } else {
#pragma unroll
            for (uint32_t u = 0; u < 4; u++) cc[u] = i + u < have ? cget(w.cnt, w.cw, at + i + u) : 0;
          }
#pragma unroll
          for (uint32_t u = 0; u < 4; u++) {
            if (found || i + u >= have) continue;
            if (cc[u] >= j) {
              found = true;
              i += u;
              break;
            }
            j -= cc[u];
          }
          if (!found) i += 4;
        }
      } else {
        for (; i < ar && !found; i++) {
          const uint32_t cc = leaf_block_count(t.leaf, w, f + i, c);
          if (cc >= j) {
            found = true;
            break;
          }
          j -= cc;
        }
      }
      if (!found) return kNone;
      res += (int64_t)i * w.b;
      k = f + i;
    } else {
      const uint32_t cp = blk_cnt(t.leaf, v, r.x, s, c);
      const uint32_t jj = j + (v.pc ? pck : leaf_prefix_count(t.leaf, v, r, c));
      if (jj <= cp) {
        res -= (int64_t)r.y;
        k = r.x;
        j = jj;
      } else {
        res += (int64_t)qlen(v, r.x) - r.y;
        j = jj - cp;
        k = r.x + 1;
      }
    }
  }
  return kNone;
}

template <int KIND>
__device__ __forceinline__ uint64_t q_answer(const QTree& t, const LevelView* __restrict__ lv, uint64_t a0, uint64_t a1) {
  if (KIND == BT_Q_ACCESS) return q_access(t, lv, a0);
  if (a0 > 255) return kNone;
  return KIND == BT_Q_RANK ? q_rank(t, lv, (uint32_t)a0, a1) : q_select(t, lv, (uint32_t)a0, a1);
}

// The batched query kernel: one thread answers a query.  Bound: the chain of
// dependent reads (a record per level and pointer hop, L2 or DRAM) times the
// threads in flight.  The level table is in shared memory; the records of the
// upper levels stay in L1.  Measured on 4 M queries of each kind on the tree of
// the 256 MiB text: 3.68 ms when a step read block starts, marks, ranks,
// pointers and offsets from five arrays (and every CTA copied the top levels
// into shared memory), 2.82 ms with one record, 1.69 with symbol-major counters
// and the base level; 1000 queries of each kind 79, 42 and 35 us.
template <int KIND, int NT, int MINB>
__global__ void __launch_bounds__(NT, MINB) k_queries(const TreeView* __restrict__ tv, const uint64_t* __restrict__ args,
                                                      uint64_t m, uint64_t* __restrict__ out) {
  __shared__ __align__(16) LevelView lv[kMaxLevels];
  const QTree t{tv->n, tv->L - tv->base, tv->pre, tv->leaf, tv->sym};
  const uint32_t* from = (const uint32_t*)(tv->lv + tv->base);
  for (uint32_t i = threadIdx.x; i < t.L * (sizeof(LevelView) / 4); i += NT) ((uint32_t*)lv)[i] = from[i];
  __syncthreads();
  for (uint64_t q = blockIdx.x * (uint64_t)NT + threadIdx.x; q < m; q += (uint64_t)gridDim.x * NT) {
    if (KIND == BT_Q_ACCESS) {
      out[q] = q_answer<KIND>(t, lv, args[q], 0);
    } else if ((((uintptr_t)args) & 15) == 0) {
      const ulonglong2 a = ((const ulonglong2*)args)[q];
      out[q] = q_answer<KIND>(t, lv, a.x, a.y);
    } else {
      out[q] = q_answer<KIND>(t, lv, args[2 * q], args[2 * q + 1]);
    }
  }
}

// One query, its arguments in the launch and its answer written to `out`
// (pinned host memory): 38 us a call with copies around it, 22 now.
__global__ void k_query_one(const TreeView* __restrict__ tv, int kind, uint64_t a0, uint64_t a1, uint64_t* out) {
  const QTree t{tv->n, tv->L - tv->base, tv->pre, tv->leaf, tv->sym};
  const LevelView* lv = tv->lv + tv->base;
  if (kind == BT_Q_ACCESS) *out = q_answer<BT_Q_ACCESS>(t, lv, a0, a1);
  else if (kind == BT_Q_RANK) *out = q_answer<BT_Q_RANK>(t, lv, a0, a1);
  else *out = q_answer<BT_Q_SELECT>(t, lv, a0, a1);
}

// The records of all levels (blockIdx.y) and their mark words, from the
// arrays of the construction, and the tree's device view (filled in here with
// the lengths of the levels' last blocks).
struct PackLevel {
  uint64_t c, b;
  const uint64_t* st;
  const uint32_t* mw;
  const uint32_t* mr;
  const uint32_t* ptr;
  const uint64_t* off;
  uint2* rec;
  uint32_t* mw2;
  uint32_t* mr2;
};
struct PackArgs {
  PackLevel lv[kMaxLevels];
  TreeView view;
};
__global__ void __launch_bounds__(256) k_pack_records(const __grid_constant__ PackArgs P, TreeView* __restrict__ view) {
  const PackLevel& v = P.lv[blockIdx.y];
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    if (blockIdx.y == 0) {
      view->n = P.view.n;
      view->L = P.view.L;
      view->S = P.view.S;
      view->base = P.view.base;
      view->pre = P.view.pre;
      view->leaf = P.view.leaf;
      view->sym = P.view.sym;
    }
    LevelView lv = P.view.lv[blockIdx.y];
    const uint64_t last = P.view.n - v.st[v.c - 1];
    lv.last_len = (uint32_t)(last < v.b ? last : v.b);
    view->lv[blockIdx.y] = lv;
  }
  const uint64_t words = (v.c + 31) / 32, stride = (uint64_t)gridDim.x * blockDim.x;
  for (uint64_t k = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; k < v.c; k += stride) {
    const uint32_t w = v.mw[k >> 5], bit = (uint32_t)k & 31u;
    if ((w >> bit) & 1u) v.rec[k] = make_uint2(kMarkedRec, v.mr[k >> 5] + __popc(w & ((1u << bit) - 1u)));
    else v.rec[k] = make_uint2(v.ptr[k], (uint32_t)v.off[k]);
  }
  for (uint64_t i = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; i <= words; i += stride) {
    if (i < words) v.mw2[i] = v.mw[i];
    v.mr2[i] = v.mr[i];
  }
}

}  // namespace

int alphabet(const uint8_t* T, uint64_t n, uint32_t* seen, bt_tree* t, Status* st, cudaStream_t s) {
  BT_CUDA(cudaMallocAsync((void**)&t->sym, 256 * sizeof(int16_t), s));
  BT_LAUNCH(k_alphabet<<<grid_for(n / 16 + 1, 256, 152 * 8), 256, 0, s>>>(T, n, seen, t->sym, st));
  BT_CUDA(cudaGetLastError());
  return BT_OK;
}

// The level queries start at: the lowest one with all blocks of the text
// (every block above it is marked), while its prefix table, 4 bytes per block
// and symbol, stays within an eighth of the text (or 64 KiB).  A descent of the
// 256 MiB text's tree then starts at level 8 of 12, and the levels above need
// no counters.
static uint32_t base_level(const bt_tree* t, uint32_t last) {
  uint32_t base = 0;
  for (uint32_t l = 1; l <= last; l++) {
    const Level& v = t->lv[l];
    if (v.c != (t->n + v.b - 1) / v.b || v.b > 0xFFFFFFFFull) break;
    const uint64_t bytes = (v.c + 1) * t->S * 4;
    if (bytes <= t->n / 8 || bytes <= (64u << 10)) base = l;
  }
  return base;
}

// The tile counter of 256 symbols needs 96.25 KiB of shared memory:
// opted in once per device.
static int allow_count_smem() {
  static std::atomic<uint64_t> done{0};
  int dev = 0;
  BT_CUDA(cudaGetDevice(&dev));
  const uint64_t bit = 1ull << (dev & 63);
  if (done.load(std::memory_order_acquire) & bit) return BT_OK;
  BT_CUDA(cudaFuncSetAttribute(k_count_tile<false>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                               256 * kTileMany * 2 + 256 + 8 * 8 * 256 * 4));
  done.fetch_or(bit, std::memory_order_acq_rel);
  return BT_OK;
}

int build_counters(BuildCtx& ctx) {
  bt_tree* t = ctx.t;
  cudaStream_t s = ctx.s;
  const uint32_t S = t->S;
  const unsigned T = 256;
  // Space-efficient counters: the last level keeps none (queries count its
  // blocks in the leaf text), and the marked blocks of the level above are
  // counted in the text instead of summed from children.
  const bool leaf_counts = ctx.leaf_counts && t->L >= 2;
  t->base = base_level(t, leaf_counts ? t->L - 2 : t->L - 1);
  for (int l = (int)t->L - 1; l >= (int)t->base; l--) {
    Level& v = t->lv[l];
    v.cw = counter_width(v.b);
    if (leaf_counts && l + 1 == (int)t->L) {
      v.cnt = v.pc = nullptr;
      continue;
    }
    const uint64_t cp = counter_stride(v.c), half = (S * cp * v.cw + 255) & ~255ull;
    char* mem;
    BT_CUDA(cudaMallocAsync((void**)&mem, 2 * half, s));
    v.owned.push_back(mem);
    v.cnt = mem;
    v.pc = mem + half;
    const bool last = l + 1 == (int)t->L;
    const bool children_counted = !last && !(leaf_counts && l + 2 == (int)t->L);
    const CountLevel J{v.st, v.ptr, v.off, v.mw, v.c, v.b, t->n, cp, v.cnt, v.pc, v.cw, children_counted};
    if (v.cw == 1) {
      const size_t sm = (size_t)kSmallCountThreads * S + 256;
      BT_LAUNCH(k_count_small<<<dim3((unsigned)((v.c + kSmallCountThreads - 1) / kSmallCountThreads), 2),
                                kSmallCountThreads, sm, s>>>(J, t->sym, ctx.T, S));
    } else if (v.cw == 2) {
      const dim3 grid(grid_for(v.c, S <= kFewSymbols ? kTileFew : kTileMany, 152 * 16), 2);
      const size_t rows = (size_t)S * (S <= kFewSymbols ? kTileFew : kTileMany) * 2 + 256, hists = 8ull * 8 * S * 4;
      if (S <= kFewSymbols) {
        BT_LAUNCH(k_count_tile<true><<<grid, 256, rows, s>>>(J, t->sym, ctx.T, S));
      } else {
        BT_TRY(allow_count_smem());
        BT_LAUNCH(k_count_tile<false><<<grid, 256, rows + hists, s>>>(J, t->sym, ctx.T, S));
      }
    } else {
      BT_CUDA(cudaMemsetAsync(mem, 0, 2 * half, s));
      const uint64_t ppb = (v.b + kCountPiece - 1) / kCountPiece;
      BT_LAUNCH(k_count_long<<<dim3(grid_for(v.c * ppb * 32, T), 2), T, 8 * S * sizeof(uint32_t), s>>>(J, t->sym, ctx.T, S,
                                                                                                    ppb));
    }
    if (children_counted) {
      const Level& w = t->lv[l + 1];
      const dim3 grid(grid_for(v.c, T), S < 8 ? 1 : 8);
      auto sum = [&](auto kernel) {
        BT_LAUNCH(kernel<<<grid, T, 0, s>>>(J, v.mr, v.arity, w.b, w.cnt, counter_stride(w.c), S));
      };
      if (v.cw == 1) sum(k_sum_children<1, 1>);
      else if (v.cw == 2) w.cw == 1 ? sum(k_sum_children<2, 1>) : sum(k_sum_children<2, 2>);
      else if (w.cw == 1) sum(k_sum_children<4, 1>);
      else w.cw == 2 ? sum(k_sum_children<4, 2>) : sum(k_sum_children<4, 4>);
    }
    BT_CUDA(cudaGetLastError());
  }
  const Level& r = t->lv[t->base];
  BT_CUDA(cudaMallocAsync((void**)&t->pre, (r.c + 1) * S * sizeof(uint32_t), s));
  BT_LAUNCH(k_base_prefix<<<S, r.c > 512 ? 1024 : 128, 0, s>>>(r.c, r.cnt, r.cw, counter_stride(r.c), t->pre));
  // Leaf text of the marked last-level blocks.
  const Level& z = t->lv[t->L - 1];
  t->leaf_bytes = z.nmarked * z.b;
  BT_CUDA(cudaMallocAsync(&t->leaf, t->leaf_bytes + 16, s));
  if (z.b % 16 == 0 && ((uintptr_t)ctx.T & 15) == 0)
    BT_LAUNCH(k_leaf_text<true><<<grid_for(z.c * (z.b / 16), T), T, 0, s>>>(z.c, z.b, t->n, z.st, z.mw, z.mr, ctx.T, t->leaf));
  else
    BT_LAUNCH(k_leaf_text<false><<<grid_for(z.c * z.b, T), T, 0, s>>>(z.c, z.b, t->n, z.st, z.mw, z.mr, ctx.T, t->leaf));
  BT_CUDA(cudaGetLastError());
  t->leaf_bytes -= ctx.st_host->leaf_short;  // the text's last block may be short
  return BT_OK;
}

// The finished tree keeps records instead of the construction's arrays, which
// are given back: 8 bytes per block instead of 20, in one allocation.
int pack_records(BuildCtx& ctx) {
  bt_tree* t = ctx.t;
  cudaStream_t s = ctx.s;
  auto al = [](uint64_t x) { return (x + 255) & ~255ull; };
  uint64_t total = 0, cmax = 1;
  for (const Level& v : t->lv) {
    const uint64_t words = (v.c + 31) / 32;
    total += al(v.c * 8) + al(words * 4) + al((words + 1) * 4);
    cmax = v.c > cmax ? v.c : cmax;
  }
  char* mem;
  BT_CUDA(cudaMallocAsync((void**)&mem, total, s));
  t->recs = mem;
  BT_CUDA(cudaMallocAsync((void**)&t->view, sizeof(TreeView), s));
  PackArgs P;
  P.view.n = t->n;
  P.view.L = t->L;
  P.view.S = t->S;
  P.view.base = t->base;
  P.view.pre = t->pre;
  P.view.leaf = t->leaf;
  P.view.sym = t->sym;
  for (uint32_t l = 0; l < t->L; l++) {
    Level& v = t->lv[l];
    const uint64_t words = (v.c + 31) / 32;
    PackLevel& p = P.lv[l];
    p = PackLevel{v.c, v.b, v.st, v.mw, v.mr, v.ptr, v.off, (uint2*)mem, nullptr, nullptr};
    P.view.lv[l] = LevelView{(uint32_t)v.c, view_len(v.b), v.arity, block_shift(view_len(v.b)), 0, v.cw,
                             (uint32_t)counter_stride(v.c), 0, p.rec, v.cnt, v.pc};
    mem += al(v.c * 8);
    p.mw2 = (uint32_t*)mem;
    mem += al(words * 4);
    p.mr2 = (uint32_t*)mem;
    mem += al((words + 1) * 4);
  }
  BT_LAUNCH(k_pack_records<<<dim3(grid_for(cmax, 256, 2048), t->L), 256, 0, s>>>(P, t->view));
  BT_CUDA(cudaGetLastError());
  for (uint32_t l = 0; l < t->L; l++) {
    Level& v = t->lv[l];
    v.rec = P.lv[l].rec;
    v.mw = P.lv[l].mw2;
    v.mr = P.lv[l].mr2;
    v.st = v.off = v.lo = nullptr;
    v.ptr = nullptr;
    std::vector<void*> keep;
    for (void* a : v.owned) {
      if (a == v.cnt) keep.push_back(a);
      else cudaFreeAsync(a, s);
    }
    v.owned.swap(keep);
  }
  return BT_OK;
}

int run_query_one(const bt_tree* t, int kind, uint64_t a0, uint64_t a1, uint64_t* out, cudaStream_t s) {
  BT_LAUNCH(k_query_one<<<1, 1, 0, s>>>(t->view, kind, a0, a1, out));
  BT_CUDA(cudaGetLastError());
  return BT_OK;
}

int run_queries(const bt_tree* t, int kind, const uint64_t* d_args, uint64_t m, uint64_t* d_out,
                cudaStream_t s) {
  if (m == 0) return BT_OK;
  // CTAs of 128 threads: small batches spread over more SMs; 64 registers, so
  // that 1024 threads fit on an SM.
  const unsigned g = grid_for(m, 128, 152 * 64);
  if (kind == BT_Q_ACCESS) BT_LAUNCH(k_queries<BT_Q_ACCESS, 128, 16><<<g, 128, 0, s>>>(t->view, d_args, m, d_out));
  else if (kind == BT_Q_RANK) BT_LAUNCH(k_queries<BT_Q_RANK, 128, 8><<<g, 128, 0, s>>>(t->view, d_args, m, d_out));
  else BT_LAUNCH(k_queries<BT_Q_SELECT, 128, 8><<<g, 128, 0, s>>>(t->view, d_args, m, d_out));
  BT_CUDA(cudaGetLastError());
  return BT_OK;
}

}  // namespace bt
