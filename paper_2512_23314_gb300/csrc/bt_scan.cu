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
// Bound: the text once per pass (twice in all) and n/4 bytes written.  A
// Horner step is a 61-bit product (about 20 instructions) per byte; instead a
// 32-byte chunk is the dot product of its bytes with the powers B^31 .. B^0,
// whose eight 8-bit limbs are constants: two 4-way byte products (__dp4a)
// per byte and one reduction per chunk.  A thread takes four chunks, so that
// the scan's products (about eight per thread) are shared by 128 bytes.  The
// CTA totals come from a pass of their own and the text is read again: the
// pass that writes then writes final values, instead of local ones that a
// third pass reads, corrects and writes once more.  The second pass takes
// the tiles from the last to the first, so that it starts with the text the
// first pass left in L2.
// Measured on 256 MiB + 77, the whole call: 548 us with a Horner pass that
// wrote local values (454), their totals (33) and a correcting pass (32); 169
// us now.
// ---------------------------------------------------------------------------
constexpr int kKrThreads = 256;    // threads of a tile of kTile chunks
constexpr int kKrChunks = 4;       // chunks per thread
static_assert(kKrThreads * kKrChunks == kTile, "a tile is kTile chunks");

// agg[i] = fingerprint of tile i (kTile chunks); the last tile is not needed.
// pw: the shift of a thread's four chunks, P = B^32 the shift of one.
template <class M>
__global__ void __launch_bounds__(kKrThreads) k_kr_totals(M m, const uint8_t* __restrict__ T, uint64_t nchunks,
                                                          const ChunkHash<M> hash, uint64_t P, KrPow pw,
                                                          uint64_t* __restrict__ agg) {
  __shared__ uint64_t sm[kKrThreads / 32];
  const bool aligned = (((uintptr_t)T) & 15) == 0;
  const uint64_t j0 = (uint64_t)blockIdx.x * kTile + (uint64_t)threadIdx.x * kKrChunks;
  uint32_t w[kKrChunks][8];
#pragma unroll
  for (int i = 0; i < kKrChunks; i++) load_chunk(T, nchunks, j0 + i, aligned, w[i]);
  uint64_t h = hash(m, w[0]);
#pragma unroll
  for (int i = 1; i < kKrChunks; i++) h = m.add(m.mul(h, P), hash(m, w[i]));
  // Ordered tree over the warp, then over the warps.
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
  for (int i = 0; i < 5; i++) h = m.add(m.mul(h, pw.x[i]), __shfl_down_sync(0xFFFFFFFFu, h, 1 << i));
  if (lane == 0) sm[warp] = h;
  __syncthreads();
  if (threadIdx.x == 0) {
    h = sm[0];
#pragma unroll
    for (int i = 1; i < kKrThreads / 32; i++) h = m.add(m.mul(h, pw.w[0]), sm[i]);
    agg[blockIdx.x] = h;
  }
}

// agg[i] = fingerprint of tiles 0 .. i, by one CTA: a thread folds `per`
// consecutive tiles (all loads first, eight at a time), then the threads are
// scanned.  Y: the shift of a tile; pw: the shift of a thread's tiles.
template <class M>
__global__ void __launch_bounds__(kTile) k_kr_aggs(M m, uint64_t* __restrict__ agg, uint64_t na, uint64_t per,
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
  for (uint64_t i = 0; i < per && i0 + i < na; i++) {
    up = m.add(m.mul(up, Y), agg[i0 + i]);
    agg[i0 + i] = up;
  }
}

// Hs[j] = H(32 j) for j <= nchunks: every thread's four chunks again, scanned
// over the tile with the tile's prefix as the first item's carry-in.
template <class M>
__global__ void __launch_bounds__(kKrThreads) k_kr_write(M m, const uint8_t* __restrict__ T, uint64_t nchunks,
                                                         const ChunkHash<M> hash, uint64_t P, KrPow pw,
                                                         const uint64_t* __restrict__ agg, uint64_t* __restrict__ Hs) {
  __shared__ uint64_t sm[32];
  const bool aligned = (((uintptr_t)T) & 15) == 0;
  const uint64_t tile = gridDim.x - 1 - blockIdx.x;
  const uint64_t j0 = tile * kTile + (uint64_t)threadIdx.x * kKrChunks;
  uint64_t c[kKrChunks];
  {
    uint32_t w[kKrChunks][8];
#pragma unroll
    for (int i = 0; i < kKrChunks; i++) load_chunk(T, nchunks, j0 + i, aligned, w[i]);
#pragma unroll
    for (int i = 0; i < kKrChunks; i++) c[i] = hash(m, w[i]);
  }
  uint64_t h = c[0];
#pragma unroll
  for (int i = 1; i < kKrChunks; i++) h = m.add(m.mul(h, P), c[i]);
  const uint64_t carry = threadIdx.x == 0 && tile ? agg[tile - 1] : 0;
  if (threadIdx.x == 0) h = m.add(m.mul(carry, pw.x[0]), h);
  const uint64_t incl = cta_kr_scan(m, h, pw, kr_lane_pow(m, pw), sm);
  uint64_t up = __shfl_up_sync(0xFFFFFFFFu, incl, 1);
  if ((threadIdx.x & 31) == 31) sm[threadIdx.x >> 5] = incl;
  __syncthreads();
  if ((threadIdx.x & 31) == 0) up = threadIdx.x ? sm[(threadIdx.x >> 5) - 1] : carry;
  // up = H(32 j0); the four values are one aligned 32-byte sector.
  uint64_t o[kKrChunks];
#pragma unroll
  for (int i = 0; i < kKrChunks; i++) {
    o[i] = up;
    up = m.add(m.mul(up, P), c[i]);
  }
  if (j0 + kKrChunks - 1 <= nchunks && (((uintptr_t)Hs) & 15) == 0) {
    ((ulonglong2*)(Hs + j0))[0] = make_ulonglong2(o[0], o[1]);
    ((ulonglong2*)(Hs + j0))[1] = make_ulonglong2(o[2], o[3]);
  } else {
#pragma unroll
    for (int i = 0; i < kKrChunks; i++)
      if (j0 + i <= nchunks) Hs[j0 + i] = o[i];
  }
}

// The three launches; agg holds nchunks / kTile entries.
template <class M>
int kr_launch(const M& m, const uint8_t* T, uint64_t n, uint64_t B, uint64_t* Hs, uint64_t* agg, cudaStream_t s) {
  const uint64_t nchunks = n / kPrefixStride;
  const uint64_t tiles = nchunks / kTile + 1, na = tiles - 1;  // the last tile writes Hs[nchunks]
  const uint64_t P = pow_mod(m, B, kPrefixStride);
  const KrPow pw = kr_pow(m, pow_mod(m, P, kKrChunks));
  const ChunkHash<M> hash(m, B);
  if (na) {
    BT_LAUNCH(k_kr_totals<M><<<(unsigned)na, kKrThreads, 0, s>>>(m, T, nchunks, hash, P, pw, agg));
    const uint64_t per = (na + kTile - 1) / kTile, Y = pow_mod(m, P, kTile);
    BT_LAUNCH(k_kr_aggs<M><<<1, kTile, 0, s>>>(m, agg, na, per, Y, kr_pow(m, pow_mod(m, Y, per))));
  }
  BT_LAUNCH(k_kr_write<M><<<(unsigned)tiles, kKrThreads, 0, s>>>(m, T, nchunks, hash, P, pw, agg, Hs));
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
  if (nchunks >= kTile) BT_TRY(sc.alloc(&agg, nchunks / kTile));
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
constexpr uint64_t kNoAllocAggs = (kNoAllocMaxN / kPrefixStride + kTile - 1) / kTile;
constexpr uint64_t kNoAllocWords = kNoAllocAggs;  // 65536 u64, 512 KiB
constexpr int kNoAllocDevices = 64;
// The array holds exactly the tile totals of the largest text.
static_assert(kNoAllocAggs == 65536, "one aggregate per 1024 chunks of 32 bytes of a 2 GiB text");

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
