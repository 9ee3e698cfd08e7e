// bt_kr.cuh -- Karp-Rabin fingerprints of 32-byte chunks and of single
// positions, shared by the prefix kernels (bt_scan.cu) and the level pass
// that reads the stride-32 prefix values (bt_quick.cu).
#pragma once

#include "bt_internal.cuh"

namespace bt {

// Fingerprint of a 32-byte chunk (eight little-endian words).
template <class M>
struct ChunkHash {  // any modulus: Horner
  uint64_t B;
  ChunkHash() = default;
  ChunkHash(const M&, uint64_t base) : B(base) {}
  __device__ __forceinline__ uint64_t operator()(const M& m, const uint32_t* w) const {
    uint64_t h = 0;
#pragma unroll
    for (int i = 0; i < (int)kPrefixStride; i++)
      h = m.add(m.mul(h, B), (uint64_t)((w[i >> 2] >> (8 * (i & 3))) & 0xFFu) + 1);
    return h;
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

// H(p) at any position from the stride-32 prefix values and the text.  With
// j = p / 32 and r = p mod 32, H(p) B^(32-r) = H(32 j) B^32 + the chunk's
// first r symbols times B^31, B^30, ..: the same constants for every r (bytes
// past r masked off), then one product with B^-(32-r) (the modulus is prime).
// A value costs two sectors (one of the values, one of the text) where the
// expanded array H(0), H(1), .. cost one, but that array is 8 bytes per
// text byte: this form neither writes it (445 us of a 256 MiB build) nor
// needs its memory.
template <class M>
struct PrefixAt {  // any modulus: Horner
  const uint8_t* T;
  const uint64_t* Hs;
  uint64_t n, B;
  PrefixAt(const M&, const uint8_t* T_, uint64_t n_, const uint64_t* Hs_, uint64_t B_) : T(T_), Hs(Hs_), n(n_), B(B_) {}
  __device__ __forceinline__ uint64_t at(const M& m, uint64_t p) const {
    uint64_t h = Hs[p / kPrefixStride];
    for (uint64_t x = p & ~(uint64_t)(kPrefixStride - 1); x < p; x++) h = m.add(m.mul(h, B), (uint64_t)T[x] + 1);
    return h;
  }
};
template <>
struct PrefixAt<Mersenne61> {
  const uint8_t* T;
  const uint64_t* Hs;
  uint64_t n, B32;
  bool aligned;
  ChunkHash<Mersenne61> hash;
  uint64_t ones[32], inv[32];  // [r]: the sum of B^31 .. B^(32-r); B^-(32-r)
  PrefixAt(const Mersenne61& m, const uint8_t* T_, uint64_t n_, const uint64_t* Hs_, uint64_t B)
      : T(T_), Hs(Hs_), n(n_), B32(pow_mod(m, B, 32)), aligned((((uintptr_t)T_) & 15) == 0), hash(m, B) {
    ones[0] = 0;
    for (int r = 1; r < 32; r++) ones[r] = m.add(ones[r - 1], pow_mod(m, B, 32 - r));
    for (int r = 0; r < 32; r++) inv[r] = pow_mod(m, pow_mod(m, B, 32 - r), Mersenne61::Q - 2);
  }
  __device__ __forceinline__ uint64_t at(const Mersenne61& m, uint64_t p) const {
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

}  // namespace bt
