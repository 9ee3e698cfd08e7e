// bt_scan.cu -- device-wide prefix operations.
//
//  * scan_u32 / scan_u64: exclusive prefix sums (rank support of the mark
//    bit vectors, job offsets).
//    Three passes: a CTA-local scan of 1024 items, a single-CTA scan of the
//    CTA aggregates, and a pass that adds each CTA's prefix to its items.
//  * prefix_fingerprints: the Karp-Rabin prefix H(32 j) of the whole text
//    (section 2 defines phi; Lemmas 7 and 8 of section 4.1 compute all
//    fingerprints with an all-prefix operation).  The 32-byte chunks are
//    hashed and combined with the associative operator
//    (h1, P1) (x) (h2, P2) = (h1 * P2 + h2, P1 * P2) of the all-prefix lemma
//    (Lemma 1); every chunk has the same length, so P is a power of
//    B^32 determined by the number of chunks combined: a tree or a scan needs
//    only its squares.  Tile totals, a single-CTA scan of them, then a pass
//    that computes every chunk's prefix from its tile's.
#include <cstdio>
#include <algorithm>
#include <mutex>

#include "bt_internal.cuh"
#include "bt_kr.cuh"

namespace bt {

namespace {

constexpr int kTile = 1024;  // items per CTA (one per thread)

template <class T>
__device__ T cta_exclusive_sum(T v, T* sm, T* total) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  T x = v;
  for (int d = 1; d < 32; d <<= 1) {
    T o = __shfl_up_sync(0xFFFFFFFFu, x, d);
    if (lane >= d) x += o;
  }
  if (lane == 31) sm[warp] = x;
  __syncthreads();
  if (warp == 0) {
    T w = sm[lane];
    for (int d = 1; d < 32; d <<= 1) {
      T o = __shfl_up_sync(0xFFFFFFFFu, w, d);
      if (lane >= d) w += o;
    }
    sm[lane] = w;
  }
  __syncthreads();
  T incl = x + (warp > 0 ? sm[warp - 1] : T(0));
  *total = sm[31];
  __syncthreads();
  return incl - v;
}

template <class T>
__global__ void __launch_bounds__(kTile) k_sum_local(const T* __restrict__ in, T* __restrict__ out,
                                                     uint64_t n, T* __restrict__ agg) {
  __shared__ T sm[32];
  uint64_t i = (uint64_t)blockIdx.x * kTile + threadIdx.x;
  T v = i < n ? in[i] : T(0);
  T tot;
  T e = cta_exclusive_sum(v, sm, &tot);
  if (i < n) out[i] = e;
  if (threadIdx.x == 0) agg[blockIdx.x] = tot;
}

// Exclusive scan of the aggregates by one CTA; agg[na] receives the total.
template <class T>
__global__ void __launch_bounds__(kTile) k_sum_aggs(T* agg, uint64_t na) {
  __shared__ T sm[32];
  T carry = 0;
  for (uint64_t base = 0; base < na; base += kTile) {
    uint64_t i = base + threadIdx.x;
    T v = i < na ? agg[i] : T(0);
    T tot;
    T e = cta_exclusive_sum(v, sm, &tot);
    if (i < na) agg[i] = carry + e;
    carry += tot;
  }
  if (threadIdx.x == 0) agg[na] = carry;
}

template <class T>
__global__ void __launch_bounds__(kTile) k_sum_add(T* out, uint64_t n, const T* __restrict__ agg) {
  uint64_t i = (uint64_t)blockIdx.x * kTile + threadIdx.x;
  if (i < n) out[i] += agg[blockIdx.x];
  if (i == 0) {
    uint64_t na = (n + kTile - 1) / kTile;
    out[n] = agg[na];
  }
}

template <class T>
int scan_sum(const T* in, T* out, uint64_t n, cudaStream_t s) {
  if (n == 0) {
    BT_CUDA(cudaMemsetAsync(out, 0, sizeof(T), s));
    return BT_OK;
  }
  uint64_t na = (n + kTile - 1) / kTile;
  if (na > (1ull << 31)) return BT_EINVAL;
  Scratch sc(s);
  T* agg;
  BT_TRY(sc.alloc(&agg, na + 1));
  BT_LAUNCH(k_sum_local<T><<<(unsigned)na, kTile, 0, s>>>(in, out, n, agg));
  BT_LAUNCH(k_sum_aggs<T><<<1, kTile, 0, s>>>(agg, na));
  BT_LAUNCH(k_sum_add<T><<<(unsigned)na, kTile, 0, s>>>(out, n, agg));
  BT_CUDA(cudaGetLastError());
  return BT_OK;
}

// ---------------------------------------------------------------------------
// Karp-Rabin all-prefix.
//
// Bound: the text read and n/4 bytes written once (60 us on 256 MiB); in fact
// the issue of the first pass's integer instructions.  A Horner step is a 61-bit
// product (about 20 instructions) per byte; instead a 32-byte chunk is the dot
// product of its bytes with the powers B^31 .. B^0, whose eight 8-bit limbs are
// constants: two 4-way byte products (__dp4a) per byte and one reduction per
// chunk.  A thread takes eight chunks, so that the scan's products (about seven
// per thread) are shared by 256 bytes, and leaves values local to its chunks,
// which the last pass moves along by one product each: it reads and writes the
// n/4 bytes once more, mostly in the L2, where a second pass over the text for
// final values took twice the first one's instructions.
// Measured on 256 MiB + 77, the whole call: 548 us with a Horner pass, 169 with
// dot products in two passes over the text, 110 now
// (68, 9 and 27).
// ---------------------------------------------------------------------------
constexpr int kKrThreads = 256;    // threads of a tile
constexpr int kKrChunks = 8;       // chunks per thread
constexpr int kKrTile = kKrThreads * kKrChunks;

// X^(lane + 1) for a thread's shift X, by lane.
struct KrLane {
  uint64_t x[32];
};

// First pass, a tile of kKrTile chunks per CTA, kKrChunks per thread: of a
// thread's chunks j0 .. the fingerprint of the tile's chunks before j0 goes to
// Hs[j0], that of chunks j0 .. j - 1 to Hs[j] (j <= nchunks), and every tile's but the
// last to agg.
template <class M>
__global__ void __launch_bounds__(kKrThreads) k_kr_local(M m, const uint8_t* __restrict__ T, uint64_t nchunks,
                                                         const __grid_constant__ ChunkHash<M> hash, uint64_t P,
                                                         const __grid_constant__ KrPow pw,
                                                         const __grid_constant__ KrLane xl, uint64_t* __restrict__ agg,
                                                         uint64_t* __restrict__ Hs) {
  __shared__ uint64_t sm[kKrThreads / 32];
  __shared__ uint64_t val[kKrTile + kKrTile / kKrChunks];  // (one word more per thread: no bank conflicts)
  const bool aligned = (((uintptr_t)T) & 15) == 0;
  const uint64_t tile0 = (uint64_t)blockIdx.x * kKrTile;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  // Chunks in the order of the threads (coalesced), then each thread its own.
#pragma unroll
  for (int q = 0; q < kKrChunks; q += 4) {
    uint32_t w[4][8];
#pragma unroll
    for (int i = 0; i < 4; i++) load_chunk(T, nchunks, tile0 + (q + i) * kKrThreads + threadIdx.x, aligned, w[i]);
#pragma unroll
    for (int i = 0; i < 4; i++) {
      const uint32_t at = (q + i) * kKrThreads + threadIdx.x;
      val[at + at / kKrChunks] = hash(m, w[i]);
    }
  }
  __syncthreads();
  uint64_t* mine = val + threadIdx.x * (kKrChunks + 1);
  uint64_t o[kKrChunks], h = mine[0];
#pragma unroll
  for (int i = 1; i < kKrChunks; i++) {
    o[i] = h;
    h = m.add(m.mul(h, P), mine[i]);
  }
#pragma unroll
  for (int i = 0; i < 5; i++) {
    const uint64_t u = __shfl_up_sync(0xFFFFFFFFu, h, 1 << i);
    if (lane >= (1 << i)) h = m.add(m.mul(u, pw.x[i]), h);
  }
  if (lane == 31) sm[warp] = h;
  __syncthreads();
  uint64_t before = 0;  // the warps before this one
  for (int k = 0; k < warp; k++) before = k ? m.add(m.mul(before, pw.w[0]), sm[k]) : sm[0];
  const uint64_t up = __shfl_up_sync(0xFFFFFFFFu, h, 1);
  if (threadIdx.x == kKrThreads - 1 && blockIdx.x + 1 < gridDim.x) agg[blockIdx.x] = m.add(m.mul(before, pw.w[0]), h);
  mine[0] = lane ? m.add(m.mul(before, xl.x[lane - 1]), up) : before;
#pragma unroll
  for (int i = 1; i < kKrChunks; i++) mine[i] = o[i];
  __syncthreads();
#pragma unroll
  for (int i = 0; i < kKrChunks; i++) {
    const uint32_t at = i * kKrThreads + threadIdx.x;
    if (tile0 + at <= nchunks) Hs[tile0 + at] = val[at + at / kKrChunks];
  }
}

// agg[i] = fingerprint of tiles 0 .. i, by one CTA: a thread folds `per`
// consecutive tiles (all loads first, eight at a time), then the threads are
// scanned.  Y: the shift of a tile; pw: the shift of a thread's tiles.
constexpr int kAggThreads = 512;

template <class M>
__global__ void __launch_bounds__(kAggThreads) k_kr_aggs(M m, uint64_t* __restrict__ agg, uint64_t na, uint64_t per,
                                                   uint64_t Y, KrPow pw) {
  __shared__ uint64_t sm[32];
  const uint64_t i0 = threadIdx.x * per;
  uint64_t h = 0;
  for (uint64_t i = 0; i < per; i += 8) {
    uint64_t v[8];
#pragma unroll
    for (int u = 0; u < 8; u++) v[u] = i + u < per && i0 + i + u < na ? agg[i0 + i + u] : 0;
#pragma unroll
    for (int u = 0; u < 8; u++)
      if (i + u < per) h = m.add(m.mul(h, Y), v[u]);
  }
  const uint64_t incl = cta_kr_scan(m, h, pw, kr_lane_pow(m, pw), sm);
  uint64_t up = __shfl_up_sync(0xFFFFFFFFu, incl, 1);
  if ((threadIdx.x & 31) == 31) sm[threadIdx.x >> 5] = incl;
  __syncthreads();
  if ((threadIdx.x & 31) == 0) up = threadIdx.x ? sm[(threadIdx.x >> 5) - 1] : 0;
  for (uint64_t i = 0; i < per; i += 8) {
    uint64_t v[8];
#pragma unroll
    for (int u = 0; u < 8; u++) v[u] = i + u < per && i0 + i + u < na ? agg[i0 + i + u] : 0;
#pragma unroll
    for (int u = 0; u < 8; u++)
      if (i + u < per && i0 + i + u < na) {
        up = m.add(m.mul(up, Y), v[u]);
        agg[i0 + i + u] = up;
      }
  }
}

// Last pass: with c = the text before a thread's chunks (the tiles before, the
// tile's chunks before them), Hs[j0] = c and Hs[j] = c P^(j - j0) + Hs[j].  The last
// tiles first: what the first pass wrote last is in the L2.  pw: the shift of a
// thread's chunks.
struct KrShift {
  uint64_t p[kKrChunks];  // P^i
};
constexpr int kShiftThreads = 256, kShiftPairs = kKrTile / 2 / kShiftThreads;  // pairs of values per thread
template <class M>
__global__ void __launch_bounds__(kShiftThreads) k_kr_shift(M m, uint64_t nchunks, uint64_t tiles,
                                                            const __grid_constant__ KrShift S,
                                                            const __grid_constant__ KrPow pw,
                                                            const uint64_t* __restrict__ agg, uint64_t* __restrict__ Hs) {
  constexpr int kPer = kKrChunks / 2;  // threads that hold a first-pass thread's values
  const unsigned t = threadIdx.x, r = 2 * (t % kPer);
  uint64_t x[kShiftPairs] = {1};  // the shift of the tile's chunks before the values' first-pass thread
#pragma unroll
  for (int i = 0; i < 6; i++)
    if ((t / kPer >> i) & 1u) x[0] = m.mul(x[0], i < 5 ? pw.x[i] : pw.w[0]);
#pragma unroll
  for (int u = 1; u < kShiftPairs; u++) x[u] = m.mul(x[u - 1], pw.w[1]);
  const uint64_t p0 = S.p[r], p1 = S.p[r + 1];
  const bool aligned = (((uintptr_t)Hs) & 15) == 0;
  for (uint64_t tile = tiles - 1 - blockIdx.x; tile < tiles; tile -= gridDim.x) {
    const uint64_t carry = tile ? agg[tile - 1] : 0;
    ulonglong2 v[kShiftPairs];
#pragma unroll
    for (int u = 0; u < kShiftPairs; u++) {
      const uint64_t j = tile * kKrTile + 2 * (t + u * kShiftThreads);
      if (aligned && j + 1 <= nchunks) v[u] = *(const ulonglong2*)(Hs + j);
      else v[u] = make_ulonglong2(j <= nchunks ? Hs[j] : 0, j + 1 <= nchunks ? Hs[j + 1] : 0);
    }
#pragma unroll
    for (int u = 0; u < kShiftPairs; u++) {
      const uint64_t j = tile * kKrTile + 2 * (t + u * kShiftThreads);
      const uint64_t c = m.add(m.mul(carry, x[u]), __shfl_sync(0xFFFFFFFFu, v[u].x, (t & 31) & ~(kPer - 1)));
      const uint64_t a = r ? m.add(m.mul(c, p0), v[u].x) : c, b = m.add(m.mul(c, p1), v[u].y);
      if (aligned && j + 1 <= nchunks) {
        *(ulonglong2*)(Hs + j) = make_ulonglong2(a, b);
      } else {
        if (j <= nchunks) Hs[j] = a;
        if (j + 1 <= nchunks) Hs[j + 1] = b;
      }
    }
  }
}
static_assert(kShiftThreads / (kKrChunks / 2) == 64, "a round of pairs is those of 64 first-pass threads");

// The three launches; agg holds nchunks / kKrTile entries.
template <class M>
int kr_launch(const M& m, const uint8_t* T, uint64_t n, uint64_t B, uint64_t* Hs, uint64_t* agg, cudaStream_t s) {
  const uint64_t nchunks = n / kPrefixStride;
  const uint64_t tiles = nchunks / kKrTile + 1, na = tiles - 1;  // the last tile writes Hs[nchunks]
  const uint64_t P = pow_mod(m, B, kPrefixStride);
  const uint64_t X = pow_mod(m, P, kKrChunks);
  const KrPow pw = kr_pow(m, X);
  const ChunkHash<M> hash(m, B);
  KrLane xl;
  KrShift S;
  for (int i = 0; i < 32; i++) xl.x[i] = i ? m.mul(xl.x[i - 1], X) : X;
  for (int i = 0; i < kKrChunks; i++) S.p[i] = i ? m.mul(S.p[i - 1], P) : 1;
  BT_LAUNCH(k_kr_local<M><<<(unsigned)tiles, kKrThreads, 0, s>>>(m, T, nchunks, hash, P, pw, xl, agg, Hs));
  if (na) {
    const uint64_t per = (na + kAggThreads - 1) / kAggThreads, Y = pow_mod(m, P, kKrTile);
    BT_LAUNCH(k_kr_aggs<M><<<1, kAggThreads, 0, s>>>(m, agg, na, per, Y, kr_pow(m, pow_mod(m, Y, per))));
  }
  BT_LAUNCH(k_kr_shift<M><<<(unsigned)std::min<uint64_t>(tiles, 152 * 8), kShiftThreads, 0, s>>>(m, nchunks, tiles, S, pw, agg, Hs));
  BT_CUDA(cudaGetLastError());
  return BT_OK;
}

template <class M>
int kr_prefix(const M& m, const uint8_t* T, uint64_t n, uint64_t B, uint64_t* Hs, cudaStream_t s) {
  const uint64_t nchunks = n / kPrefixStride;
  if (nchunks == 0) {
    BT_CUDA(cudaMemsetAsync(Hs, 0, sizeof(uint64_t), s));
    return BT_OK;
  }
  Scratch sc(s);
  uint64_t* agg = nullptr;
  if (nchunks >= kKrTile) BT_TRY(sc.alloc(&agg, nchunks / kKrTile));
  ProfScope ps("prefix_fingerprint", s, n);
  return kr_launch(m, T, n, B, Hs, agg, s);
}

// H[p] at every position from the stride-32 values: the lane of chunk j
// extends Hs[j] by Horner over the chunk's bytes (section 2), keeping the 32
// prefixes in a shared-memory tile; the warp then writes the tile row by row
// so that each store covers 32 consecutive positions.
constexpr uint32_t kExpandWarps = 4;

template <class M>
__global__ void __launch_bounds__(32 * kExpandWarps) k_kr_expand(M m, const uint8_t* __restrict__ T,
                                                                uint64_t n, uint64_t B,
                                                                const uint64_t* __restrict__ Hs,
                                                                uint64_t* __restrict__ H) {
  __shared__ uint64_t tile[kExpandWarps][32][33];
  const unsigned lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const uint64_t nchunks = n / kPrefixStride + 1;  // the last one may be partial
  const uint64_t j0 = ((uint64_t)blockIdx.x * kExpandWarps + warp) * 32;
  const uint64_t j = j0 + lane;
  if (j < nchunks) {
    uint64_t h = Hs[j];
    const uint64_t p0 = j * kPrefixStride;
    if (p0 + kPrefixStride <= n && (((uintptr_t)(T + p0)) & 15) == 0) {
      // A full chunk: its 32 bytes are loaded before the multiply chain.
      const uint4 v0 = ((const uint4*)(T + p0))[0], v1 = ((const uint4*)(T + p0))[1];
      const uint32_t wv[8] = {v0.x, v0.y, v0.z, v0.w, v1.x, v1.y, v1.z, v1.w};
#pragma unroll
      for (uint32_t i = 0; i < kPrefixStride; i++) {
        tile[warp][lane][i] = h;
        h = m.add(m.mul(h, B), (uint64_t)((wv[i >> 2] >> (8 * (i & 3))) & 0xFFu) + 1);
      }
    } else {
#pragma unroll 4
      for (uint32_t i = 0; i < kPrefixStride; i++) {
        tile[warp][lane][i] = h;
        if (p0 + i < n) h = m.add(m.mul(h, B), (uint64_t)T[p0 + i] + 1);
      }
    }
  }
  __syncwarp();
  for (uint32_t r = 0; r < 32 && j0 + r < nchunks; r++) {
    const uint64_t p = (j0 + r) * kPrefixStride + lane;
    if (p <= n) H[p] = tile[warp][r][lane];
  }
}

template <class M>
int kr_expand(const M& m, const uint8_t* T, uint64_t n, uint64_t B, const uint64_t* Hs, uint64_t* H,
              cudaStream_t s) {
  const uint64_t nchunks = n / kPrefixStride + 1;
  const uint64_t per_cta = 32ull * kExpandWarps;
  ProfScope ps("prefix_expand", s, n);
  BT_LAUNCH(k_kr_expand<M><<<(unsigned)((nchunks + per_cta - 1) / per_cta), 32 * kExpandWarps, 0, s>>>(
      m, T, n, B, Hs, H));
  BT_CUDA(cudaGetLastError());
  return BT_OK;
}

}  // namespace

int scan_u32(const uint32_t* in, uint32_t* out, uint64_t n, cudaStream_t s) {
  return scan_sum<uint32_t>(in, out, n, s);
}
int scan_u32(const uint32_t* in, uint32_t* out, uint64_t n, cudaStream_t s, uint32_t* agg) {
  if (n == 0) {
    BT_CUDA(cudaMemsetAsync(out, 0, sizeof(uint32_t), s));
    return BT_OK;
  }
  const uint64_t na = (n + kTile - 1) / kTile;
  BT_LAUNCH(k_sum_local<uint32_t><<<(unsigned)na, kTile, 0, s>>>(in, out, n, agg));
  BT_LAUNCH(k_sum_aggs<uint32_t><<<1, kTile, 0, s>>>(agg, na));
  BT_LAUNCH(k_sum_add<uint32_t><<<(unsigned)na, kTile, 0, s>>>(out, n, agg));
  BT_CUDA(cudaGetLastError());
  return BT_OK;
}
int scan_u64(const uint64_t* in, uint64_t* out, uint64_t n, cudaStream_t s) {
  return scan_sum<uint64_t>(in, out, n, s);
}

int prefix_fingerprints(const uint8_t* T, uint64_t n, uint64_t B, uint64_t q, uint64_t* Hs,
                        cudaStream_t s) {
  if (q == Mersenne61::Q) return kr_prefix(Mersenne61{}, T, n, B, Hs, s);
  return kr_prefix(SmallMod{q}, T, n, B, Hs, s);
}

int expand_prefix(const uint8_t* T, uint64_t n, uint64_t B, uint64_t q, const uint64_t* Hs, uint64_t* H,
                  cudaStream_t s) {
  if (q == Mersenne61::Q) return kr_expand(Mersenne61{}, T, n, B, Hs, H, s);
  return kr_expand(SmallMod{q}, T, n, B, Hs, H, s);
}

// ---------------------------------------------------------------------------
// Prefix fingerprints without allocation (bt_prefix_fingerprints_noalloc).
//
// Some callers cannot allocate device memory.  For example, a host runtime may
// reserve all device memory for its own allocator up front and forbid the
// libraries it loads to call cudaMalloc.  Code on a latency-critical path may
// also be unable to risk an allocation's implicit synchronisation or failure.
// This variant of the prefix-fingerprint pass takes its scratch (the per-tile
// totals) from a fixed array in device memory instead of cudaMallocAsync.  Every GPU that loads the library holds the
// array until the process exits.
// ---------------------------------------------------------------------------
namespace {

constexpr uint64_t kNoAllocMaxN = 1ull << 31;  // largest text accepted (2 GiB)
constexpr uint64_t kNoAllocAggs = (kNoAllocMaxN / kPrefixStride + kKrTile - 1) / kKrTile;
constexpr uint64_t kNoAllocWords = kNoAllocAggs;  // 32768 u64, 256 KiB
constexpr int kNoAllocDevices = 64;
// The array holds exactly the tile totals of the largest text.
static_assert(kNoAllocAggs == 32768, "one aggregate per 2048 chunks of 32 bytes of a 2 GiB text");

static __device__ __align__(256) uint64_t g_noalloc_scratch[kNoAllocWords];

std::mutex g_noalloc_mu;
uint64_t* g_noalloc_addr[kNoAllocDevices] = {};

// Device address of the scratch array on the current device.  In host code
// the array's name stands for a host-side shadow, not device memory, so the
// address is looked up once per device (the first call on a device does it)
// and cached.
int noalloc_scratch(uint64_t** out) {
  int dev = 0;
  BT_CUDA(cudaGetDevice(&dev));
  if (dev < 0 || dev >= kNoAllocDevices) return BT_EINVAL;
  std::lock_guard<std::mutex> g(g_noalloc_mu);
  if (!g_noalloc_addr[dev]) {
    void* p = nullptr;
    cudaError_t e = cudaGetSymbolAddress(&p, g_noalloc_scratch);
    if (e != cudaSuccess) {
      note_cuda_error(e, "cudaGetSymbolAddress", __FILE__, __LINE__);
      return BT_ECUDA;
    }
    g_noalloc_addr[dev] = (uint64_t*)p;
  }
  *out = g_noalloc_addr[dev];
  return BT_OK;
}

template <class M>
int kr_prefix_noalloc(const M& m, const uint8_t* T, uint64_t n, uint64_t B, uint64_t* Hs,
                      uint64_t* scratch, cudaStream_t s) {
  if (n / kPrefixStride == 0) {
    BT_CUDA(cudaMemsetAsync(Hs, 0, sizeof(uint64_t), s));
    return BT_OK;
  }
  return kr_launch(m, T, n, B, Hs, scratch, s);
}

}  // namespace

}  // namespace bt

extern "C" int bt_prefix_fingerprints_noalloc(const uint8_t* d_text, uint64_t n, uint64_t seed,
                                              uint64_t modulus, uint32_t stride, uint64_t* d_out,
                                              void* stream) {
  using namespace bt;
  if (n > kNoAllocMaxN) return BT_ERANGE;  // before every other check
  if (!d_text || !d_out || stride != kPrefixStride) return BT_EINVAL;
  if (modulus && (modulus < 300 || modulus >= (1ull << 32))) return BT_EINVAL;
  uint64_t* scratch = nullptr;
  BT_TRY(noalloc_scratch(&scratch));
  const uint64_t q = modulus ? modulus : Mersenne61::Q;
  const uint64_t B = bt_fingerprint_base(seed, modulus);
  cudaStream_t s = stream ? (cudaStream_t)stream : cudaStreamPerThread;
  if (q == Mersenne61::Q) return kr_prefix_noalloc(Mersenne61{}, d_text, n, B, d_out, scratch, s);
  return kr_prefix_noalloc(SmallMod{q}, d_text, n, B, d_out, scratch, s);
}

namespace bt {
namespace {

// Integer-pipe microbenchmark: kMulChains independent chains of the 61-bit
// modular multiply the fingerprints use, `iters` steps each, per thread.  The
// base arrives at run time and every chain's result is stored, so nothing
// folds away.
constexpr int kMulChains = 8;

__global__ void __launch_bounds__(256) k_mulmod_bench(uint64_t B, uint32_t iters, uint64_t* __restrict__ out) {
  const Mersenne61 m;
  const uint64_t t = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x;
  uint64_t a[kMulChains];
#pragma unroll
  for (int u = 0; u < kMulChains; u++) a[u] = (t * kMulChains + u) % (Mersenne61::Q - 1) + 1;
  for (uint32_t i = 0; i < iters; i++) {
#pragma unroll
    for (int u = 0; u < kMulChains; u++) a[u] = m.mul(a[u], B);
  }
  uint64_t x = 0;
#pragma unroll
  for (int u = 0; u < kMulChains; u++) x ^= a[u];
  out[t] = x;
}

}  // namespace
}  // namespace bt

extern "C" int bt_mulmod_bench(uint32_t blocks, uint32_t iters, uint64_t seed, uint64_t* d_out, void* stream,
                               uint64_t* mulmods) {
  using namespace bt;
  if (!d_out || !mulmods || blocks == 0 || iters == 0) return BT_EINVAL;
  cudaStream_t s = stream ? (cudaStream_t)stream : cudaStreamPerThread;
  BT_LAUNCH(k_mulmod_bench<<<blocks, 256, 0, s>>>(bt_fingerprint_base(seed, 0), iters, d_out));
  BT_CUDA(cudaGetLastError());
  *mulmods = (uint64_t)blocks * 256 * iters * kMulChains;
  return BT_OK;
}
