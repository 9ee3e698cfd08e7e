// bt_bytes.cuh -- byte comparison of two text ranges by a group of lanes.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

namespace bt {

// The 16 bytes T[A, A+16) from the aligned units at A & ~15 (u0, u1).
__device__ __forceinline__ uint4 unaligned16(uint4 u0, uint4 u1, uint32_t d) {
  const uint32_t q = d >> 2, sh = 8 * (d & 3);
  const uint32_t w0 = q == 0 ? u0.x : q == 1 ? u0.y : q == 2 ? u0.z : u0.w;
  const uint32_t w1 = q == 0 ? u0.y : q == 1 ? u0.z : q == 2 ? u0.w : u1.x;
  const uint32_t w2 = q == 0 ? u0.z : q == 1 ? u0.w : q == 2 ? u1.x : u1.y;
  const uint32_t w3 = q == 0 ? u0.w : q == 1 ? u1.x : q == 2 ? u1.y : u1.z;
  const uint32_t w4 = q == 0 ? u1.x : q == 1 ? u1.y : q == 2 ? u1.z : u1.w;
  return make_uint4(__funnelshift_r(w0, w1, sh), __funnelshift_r(w1, w2, sh), __funnelshift_r(w2, w3, sh),
                    __funnelshift_r(w3, w4, sh));
}

// The 16 bytes at b (16-byte aligned) and the two aligned units that hold the
// 16 bytes at a < b (T aligned).  The second unit ends at b + 16 or before.
struct Unit16 {
  uint4 b, u0, u1;
};
__device__ __forceinline__ Unit16 load_units(const uint8_t* __restrict__ T, uint32_t a, uint32_t b) {
  const uint4* p = (const uint4*)(T + (a & ~15u));
  return Unit16{*(const uint4*)(T + b), p[0], p[1]};
}
// Realignment by a mod 16, the same for all units of a comparison.
struct Shift16 {
  bool w2, w1;
  uint32_t sh;
  __device__ __forceinline__ explicit Shift16(uint32_t a) : w2(a & 8), w1(a & 4), sh(8 * (a & 3)) {}
  __device__ __forceinline__ bool differ(const Unit16& v) const {
    uint32_t a[8] = {v.u0.x, v.u0.y, v.u0.z, v.u0.w, v.u1.x, v.u1.y, v.u1.z, v.u1.w};
#pragma unroll
    for (int i = 0; i < 6; i++) a[i] = w2 ? a[i + 2] : a[i];
#pragma unroll
    for (int i = 0; i < 5; i++) a[i] = w1 ? a[i + 1] : a[i];
    return ((__funnelshift_r(a[0], a[1], sh) ^ v.b.x) | (__funnelshift_r(a[1], a[2], sh) ^ v.b.y) |
            (__funnelshift_r(a[2], a[3], sh) ^ v.b.z) | (__funnelshift_r(a[3], a[4], sh) ^ v.b.w)) != 0;
  }
};

// Compare T[a + x] and T[b + x] for x in [off, end) by L lanes: bytes up to
// the first 16-byte unit of the side at b, then 16 bytes per lane and step,
// the other side realigned from two aligned loads; bytes for the ragged end.
__device__ __forceinline__ bool differs(const uint8_t* __restrict__ T, uint64_t n, bool aligned16, uint64_t a,
                                        uint64_t b, uint64_t off, uint64_t end, unsigned lane, unsigned L) {
  bool diff = false;
  uint64_t x = off;
  if (aligned16 && end - off >= 16) {
    const uint64_t first = off + ((16 - ((b + off) & 15)) & 15);
    for (uint64_t y = off + lane; y < first; y += L) diff |= T[a + y] != T[b + y];
    const uint64_t full = first + ((end - first) & ~15ull);
    for (uint64_t y = first + 16ull * lane; y < full; y += 16ull * L) {
      const uint4 vb = *(const uint4*)(T + b + y);
      const uint64_t A = a + y, A0 = A & ~15ull;
      const uint32_t d = (uint32_t)(A & 15);
      const uint4 u0 = *(const uint4*)(T + A0);
      uint4 va;
      if (d == 0) {
        va = u0;
      } else if (A0 + 32 <= n) {
        va = unaligned16(u0, *(const uint4*)(T + A0 + 16), d);
      } else {  // the unit past the text's end is not read
        uint32_t v[4] = {0, 0, 0, 0};
        for (uint32_t t = 0; t < 16; t++) v[t >> 2] |= (uint32_t)T[A + t] << (8 * (t & 3));
        va = make_uint4(v[0], v[1], v[2], v[3]);
      }
      diff |= va.x != vb.x || va.y != vb.y || va.z != vb.z || va.w != vb.w;
    }
    x = full;
  }
  for (x += lane; x < end; x += L) diff |= T[a + x] != T[b + x];
  return diff;
}

}  // namespace bt
