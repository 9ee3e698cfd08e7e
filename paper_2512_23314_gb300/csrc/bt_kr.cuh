// bt_kr.cuh -- Karp-Rabin fingerprints of 32-byte chunks and of single
// positions, shared by the prefix kernels (bt_scan.cu) and the level pass
// that reads the stride-32 prefix values (bt_quick.cu).
#pragma once

#include "bt_internal.cuh"

namespace bt {

// Fingerprint of a 32-byte chunk (eight little-endian words).
template <class M>
struct ChunkHash;
// A modulus below 2^32: the symbols' dot product with the powers stays below
// 2^45, so one division ends it.  (A Horner step divides for every byte; with
// eight chunks to a thread 1 MiB took 64 us that way, 45 with one chunk.)
template <>
struct ChunkHash<SmallMod> {
  uint32_t power[kPrefixStride];  // B^31 .. B^0
  ChunkHash() = default;
  ChunkHash(const SmallMod& m, uint64_t B) {
    uint64_t p = 1 % m.Q;
    for (int i = (int)kPrefixStride - 1; i >= 0; i--) {
      power[i] = (uint32_t)p;
      p = m.mul(p, B % m.Q);
    }
  }
  __device__ __forceinline__ uint64_t operator()(const SmallMod& m, const uint32_t* w) const {
    uint64_t h = 0;
#pragma unroll
    for (int i = 0; i < (int)kPrefixStride; i++)
      h += (uint64_t)(((w[i >> 2] >> (8 * (i & 3))) & 0xFFu) + 1) * power[i];
    return h % m.Q;
  }
};
template <>
struct ChunkHash<Mersenne61> {
  uint32_t limb[8][8];  // [word][l]: bits 8l..8l+7 of the powers of the word's four bytes
  uint64_t ones;        // the sum of the powers: every symbol is its byte + 1
  ChunkHash() = default;
  ChunkHash(const Mersenne61& m, uint64_t B) {
    uint64_t p = 1;
    ones = 0;
    for (int i = 31; i >= 0; i--) {
      for (int l = 0; l < 8; l++) {
        if ((i & 3) == 3) limb[i >> 2][l] = 0;
        limb[i >> 2][l] |= (uint32_t)((p >> (8 * l)) & 0xFF) << (8 * (i & 3));
      }
      ones = m.add(ones, p);
      p = m.mul(p, B);
    }
  }
  // sum of byte i times B^(31 - i), without the symbols' + 1
  __device__ __forceinline__ uint64_t dot(const uint32_t* w) const {
    uint32_t s[8];  // each at most 32 * 255^2 < 2^21
#pragma unroll
    for (int l = 0; l < 8; l++) {
      s[l] = 0;
#pragma unroll
      for (int q = 0; q < 8; q++) s[l] = __dp4a(w[q], limb[q][l], s[l]);
    }
    const uint64_t lo = (uint64_t)s[0] + ((uint64_t)s[1] << 8) + ((uint64_t)s[2] << 16) + ((uint64_t)s[3] << 24);
    const uint64_t hi = (uint64_t)s[4] + ((uint64_t)s[5] << 8) + ((uint64_t)s[6] << 16) + ((uint64_t)s[7] << 24);
    // lo + hi 2^32 with hi = a 2^29 + r: a 2^61 + r 2^32 = a + r 2^32; < 2^62.
    uint64_t x = lo + (hi >> 29) + ((hi & ((1u << 29) - 1)) << 32);
    x = (x & Mersenne61::Q) + (x >> 61);
    return x >= Mersenne61::Q ? x - Mersenne61::Q : x;
  }
  __device__ __forceinline__ uint64_t operator()(const Mersenne61& m, const uint32_t* w) const {
    return m.add(dot(w), ones);
  }
};

// Powers of the shift X of one scan item: X^1,2,4,8,16 within a warp and
// X^32,64,..,512 across the warps.
struct KrPow {
  uint64_t x[5], w[5];
};
template <class M>
KrPow kr_pow(const M& m, uint64_t X) {
  KrPow p;
  for (int i = 0; i < 5; i++) {
    p.x[i] = X;
    X = m.mul(X, X);
  }
  for (int i = 0; i < 5; i++) {
    p.w[i] = X;
    X = m.mul(X, X);
  }
  return p;
}

// Inclusive scan of the items' fingerprints over a CTA of at most 1024
// threads (sm: 32 words).
template <class M>
__device__ __forceinline__ uint64_t cta_kr_scan(const M& m, uint64_t h, const KrPow& pw, uint64_t xl, uint64_t* sm) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
#pragma unroll
  for (int i = 0; i < 5; i++) {
    const uint64_t o = __shfl_up_sync(0xFFFFFFFFu, h, 1 << i);
    if (lane >= (1 << i)) h = m.add(m.mul(o, pw.x[i]), h);
  }
  if (lane == 31) sm[warp] = h;
  __syncthreads();
  if (warp == 0) {
    uint64_t w = lane < nw ? sm[lane] : 0;
#pragma unroll
    for (int i = 0; i < 5; i++) {
      const uint64_t o = __shfl_up_sync(0xFFFFFFFFu, w, 1 << i);
      if (lane >= (1 << i)) w = m.add(m.mul(o, pw.w[i]), w);
    }
    sm[lane] = w;
  }
  __syncthreads();
  if (warp > 0) h = m.add(m.mul(sm[warp - 1], xl), h);
  __syncthreads();
  return h;
}

// X^(lane + 1) from the squares: the shift of a warp's carry-in.
template <class M>
__device__ __forceinline__ uint64_t kr_lane_pow(const M& m, const KrPow& pw) {
  const unsigned e = (threadIdx.x & 31) + 1;
  uint64_t r = 1;
#pragma unroll
  for (int i = 0; i < 5; i++)
    if ((e >> i) & 1u) r = m.mul(r, pw.x[i]);
  return e == 32 ? pw.w[0] : r;
}

// The words of chunk j, or zeros for a chunk the text does not hold.
__device__ __forceinline__ void load_chunk(const uint8_t* __restrict__ T, uint64_t nchunks, uint64_t j, bool aligned,
                                           uint32_t* w) {
  if (j >= nchunks) {
#pragma unroll
    for (int i = 0; i < 8; i++) w[i] = 0;
    return;
  }
  const uint8_t* p = T + j * kPrefixStride;
  if (aligned) {
    const uint4 v0 = ((const uint4*)p)[0], v1 = ((const uint4*)p)[1];
    w[0] = v0.x, w[1] = v0.y, w[2] = v0.z, w[3] = v0.w;
    w[4] = v1.x, w[5] = v1.y, w[6] = v1.z, w[7] = v1.w;
  } else {
#pragma unroll
    for (int i = 0; i < 8; i++)
      w[i] = (uint32_t)p[4 * i] | ((uint32_t)p[4 * i + 1] << 8) | ((uint32_t)p[4 * i + 2] << 16) |
             ((uint32_t)p[4 * i + 3] << 24);
  }
}

// H(p) at any position from the stride-32 prefix values and the text.  With
// j = p / 32 and r = p mod 32, H(p) B^(32-r) = H(32 j) B^32 + the chunk's
// first r symbols times B^31, B^30, ..: the same constants for every r (bytes
// past r masked off), then one product with B^-(32-r) (the modulus is prime).
// A value costs two sectors (one of the values, one of the text) where the
// expanded array H(0), H(1), .. cost one, but that array is 8 bytes per
// text byte: this form neither writes it (445 us of a 256 MiB build) nor
// needs its memory.
template <class M>
struct PrefixConst {  // any modulus: Horner
  uint64_t B, B32;
  ChunkHash<M> hash;
  PrefixConst(const M& m, uint64_t B_) : B(B_), B32(pow_mod(m, B_, 32)), hash(m, B_) {}
  __device__ __forceinline__ uint64_t at(const M& m, const uint8_t* T, uint64_t, const uint64_t* Hs, bool,
                                         uint64_t p) const {
    uint64_t h = Hs[p / kPrefixStride];
    for (uint64_t x = p & ~(uint64_t)(kPrefixStride - 1); x < p; x++) h = m.add(m.mul(h, B), (uint64_t)T[x] + 1);
    return h;
  }
};
template <>
struct PrefixConst<Mersenne61> {
  uint64_t B, B32;
  ChunkHash<Mersenne61> hash;
  uint64_t ones[32], inv[32];  // [r]: the sum of B^31 .. B^(32-r); B^-(32-r)
  // (One inverse and products: a build makes this once per level, and again where
  // a search is given up; 32 inverses took 10 us of host time.)
  PrefixConst(const Mersenne61& m, uint64_t B_) : B(B_), B32(pow_mod(m, B_, 32)), hash(m, B_) {
    uint64_t power[32];
    power[0] = 1;
    for (int i = 1; i < 32; i++) power[i] = m.mul(power[i - 1], B);
    ones[0] = 0;
    for (int r = 1; r < 32; r++) ones[r] = m.add(ones[r - 1], power[32 - r]);
    const uint64_t step = pow_mod(m, B, Mersenne61::Q - 2);
    inv[31] = step;
    for (int r = 30; r >= 0; r--) inv[r] = m.mul(inv[r + 1], step);
  }
  __device__ __forceinline__ uint64_t at(const Mersenne61& m, const uint8_t* T, uint64_t n, const uint64_t* Hs,
                                         bool aligned, uint64_t p) const {
    const uint64_t j = p >> 5;
    const uint32_t r = (uint32_t)p & 31u;
    const uint64_t h = Hs[j];
    if (r == 0) return h;
    uint32_t w[8];
    if (aligned && 32 * j + 32 <= n) {
      const uint4 v0 = ((const uint4*)(T + 32 * j))[0], v1 = ((const uint4*)(T + 32 * j))[1];
      w[0] = v0.x, w[1] = v0.y, w[2] = v0.z, w[3] = v0.w;
      w[4] = v1.x, w[5] = v1.y, w[6] = v1.z, w[7] = v1.w;
    } else {
#pragma unroll
      for (uint32_t q = 0; q < 8; q++) {
        w[q] = 0;
#pragma unroll
        for (uint32_t t = 0; t < 4; t++)
          if (4 * q + t < r) w[q] |= (uint32_t)T[32 * j + 4 * q + t] << (8 * t);
      }
    }
#pragma unroll
    for (int q = 0; q < 8; q++) {
      const int keep = (int)r - 4 * q;  // bytes of word q below r
      w[q] = keep >= 4 ? w[q] : keep <= 0 ? 0u : w[q] & ((1u << (8 * keep)) - 1u);
    }
    const uint64_t u = m.add(m.mul(h, B32), m.add(hash.dot(w), ones[r]));
    return m.mul(u, inv[r]);
  }
};

// The prefix values of one text.
template <class M>
struct PrefixAt {
  const PrefixConst<M>& c;
  const uint8_t* T;
  const uint64_t* Hs;
  uint64_t n;
  bool aligned;
  __device__ __forceinline__ PrefixAt(const PrefixConst<M>& c_, const uint8_t* T_, uint64_t n_, const uint64_t* Hs_)
      : c(c_), T(T_), Hs(Hs_), n(n_), aligned((((uintptr_t)T_) & 15) == 0) {}
  __device__ __forceinline__ uint64_t at(const M& m, uint64_t p) const { return c.at(m, T, n, Hs, aligned, p); }
};

}  // namespace bt
