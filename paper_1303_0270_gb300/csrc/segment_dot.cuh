// segment_dot.cuh -- the dot product of a segment (32 consecutive fields of a
// row, at any bit offset) with 32 entries of x held as bytes, shared by the
// batched and the ragged matvec: the x byte order, the loads of a staged
// segment, the byte-dot decodes (dp4a / dp2a) and the division that turns a
// segment number into a row.
#pragma once

#include "ccm_device.cuh"

namespace ccm {
namespace seg {

// Unsigned 32-bit division by a run-time invariant d >= 1 with one high
// multiply, after Granlund and Montgomery, "Division by invariant integers
// using multiplication" (1994), Fig. 4.1: with l = ceil(log2 d) and
// m = floor(2^32 (2^l - d) / d) + 1, q = (t + ((v - t) >> min(l, 1))) >>
// max(l - 1, 0) where t = mulhi(m, v), for every 32-bit v.
struct DivSeg {
  uint32_t m, s1, s2;
  static DivSeg make(uint32_t d) {
    int l = 0;
    while (l < 32 && (1ull << l) < d) ++l;
    const uint64_t m = (((1ull << l) - d) << 32) / d + 1;
    return {(uint32_t)m, (uint32_t)(l < 1 ? l : 1), (uint32_t)(l > 1 ? l - 1 : 0)};
  }
};

__device__ __forceinline__ uint32_t div_seg(uint32_t v, uint32_t dm, uint32_t ds1, uint32_t ds2) {
  const uint32_t t = __umulhi(v, dm);
  return (t + ((v - t) >> ds1)) >> ds2;
}

// Position of field f of a segment in its 32-byte x image on the fast path:
// the order in which the width-b decode pairs fields with x bytes (natural,
// except for b = 1, 2, 4, where byte p of the k-th shifted copy of word i
// holds field i (32/b) + p (8/b) + k).
__device__ __forceinline__ uint32_t xbyte_pos(uint32_t f, int b) {
  if (b == 1 || b == 2 || b == 4) {
    const uint32_t per = 32u / b, r = 8u / b;
    const uint32_t i = f / per, q = f % per;
    return 4u * (i * r + q % r) + q / r;
  }
  return f;
}

// ---------------------------------------------------------------------------
// Dot product of one segment (32 fields in f[0..B-1], f[B] spare)
// ---------------------------------------------------------------------------
__device__ __forceinline__ int dp4a_us(uint32_t a, int b, int c) {
  int d;
  asm("dp4a.u32.s32 %0, %1, %2, %3;" : "=r"(d) : "r"(a), "r"(b), "r"(c));
  return d;
}
__device__ __forceinline__ int dp2a_lo_us(uint32_t a, int b, int c) {
  int d;
  asm("dp2a.lo.u32.s32 %0, %1, %2, %3;" : "=r"(d) : "r"(a), "r"(b), "r"(c));
  return d;
}
__device__ __forceinline__ int dp2a_hi_us(uint32_t a, int b, int c) {
  int d;
  asm("dp2a.hi.u32.s32 %0, %1, %2, %3;" : "=r"(d) : "r"(a), "r"(b), "r"(c));
  return d;
}
// Byte k of w sign-extended to 32 bits (prmt with the sign-replicate bit
// set in the selectors of bytes 1..3).
__device__ __forceinline__ int sbyte(uint32_t w, int k) {
  const uint32_t sel = (uint32_t)k | ((uint32_t)(k | 8) * 0x1110u);
  int d;
  asm("prmt.b32 %0, %1, 0, %2;" : "=r"(d) : "r"(w), "r"(sel));
  return d;
}

__host__ __device__ constexpr uint32_t low_bits(int b) { return b >= 32 ? 0xffffffffu : ((1u << b) - 1u); }


// Signed fields of at most 16 bits are taken in offset binary: their sign bits
// flipped before the dot product, which subtracts 2^(B-1) times the sum of x.
// (Wider ones flip theirs inside.)
template <int B, bool SGN>
__device__ __forceinline__ void flip_signs(uint32_t (&f)[B + 1]) {
  if constexpr (SGN && B <= 16) {
#pragma unroll
    for (int i = 0; i < B; ++i) f[i] ^= group_sign_bits(B, i);
  }
}

// Sum over the segment's fields (after flip_signs) of a_f x_f with x bytes
// xw[0..7] in the order of xbyte_pos; `xs` is the segment's sum of x.
template <int B, bool SGN>
__device__ __forceinline__ int64_t seg_dot_fast(const uint32_t (&f)[B + 1], const int (&xw)[8], int xs) {
  if constexpr (B <= 16) {
    int acc0 = 0, acc1 = 0;
    if constexpr (B == 1 || B == 2 || B == 4) {
      constexpr int R = 8 / B;
      constexpr uint32_t m = low_bits(B) * 0x01010101u;
#pragma unroll
      for (int i = 0; i < B; ++i)
#pragma unroll
        for (int k = 0; k < R; ++k) {
          const uint32_t v = (f[i] >> (B * k)) & m;
          if ((i * R + k) & 1)
            acc1 = dp4a_us(v, xw[i * R + k], acc1);
          else
            acc0 = dp4a_us(v, xw[i * R + k], acc0);
        }
    } else if constexpr (B == 8) {
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        if (i & 1)
          acc1 = dp4a_us(f[i], xw[i], acc1);
        else
          acc0 = dp4a_us(f[i], xw[i], acc0);
      }
    } else if constexpr (B < 8) {
      // four fields (4B bits) -> two 16-bit halves of two fields -> four bytes
      constexpr uint32_t m2 = low_bits(2 * B), m1 = low_bits(B) * 0x00010001u;
#pragma unroll
      for (int c = 0; c < 8; ++c) {
        constexpr int kB4 = 4 * B;
        const int bit = kB4 * c, wi = bit >> 5, sh = bit & 31;
        const uint32_t x4 = (sh + kB4 <= 32) ? (f[wi] >> sh) : __funnelshift_r(f[wi], f[wi + 1], sh);
        const uint32_t u = (x4 & m2) | ((x4 << (16 - 2 * B)) & (m2 << 16));
        const uint32_t v = (u & m1) | ((u << (8 - B)) & (m1 << 8));
        if (c & 1)
          acc1 = dp4a_us(v, xw[c], acc1);
        else
          acc0 = dp4a_us(v, xw[c], acc0);
      }
    } else if constexpr (B == 16) {
#pragma unroll
      for (int c = 0; c < 16; ++c) {
        if (c & 1)
          acc1 = dp2a_hi_us(f[c], xw[c >> 1], acc1);
        else
          acc0 = dp2a_lo_us(f[c], xw[c >> 1], acc0);
      }
    } else {
      // two fields (2B bits) -> two 16-bit halves
      constexpr uint32_t mb = low_bits(B);
#pragma unroll
      for (int c = 0; c < 16; ++c) {
        constexpr int kB2 = 2 * B;
        const int bit = kB2 * c, wi = bit >> 5, sh = bit & 31;
        const uint32_t x2 = (sh + kB2 <= 32) ? (f[wi] >> sh) : __funnelshift_r(f[wi], f[wi + 1], sh);
        const uint32_t v = (x2 & mb) | ((x2 << (16 - B)) & (mb << 16));
        if (c & 1)
          acc1 = dp2a_hi_us(v, xw[c >> 1], acc1);
        else
          acc0 = dp2a_lo_us(v, xw[c >> 1], acc0);
      }
    }
    int acc = acc0 + acc1;
    if constexpr (SGN) acc -= xs * (1 << (B - 1));
    return acc;
  } else {
    // B = 17..32: a field is its low 16 bits plus 2^16 times its high B - 16
    // bits.  Per four fields: the low halves of two fields in one register
    // (prmt) against two x bytes (dp2a); the high parts, of at most 8 bits all
    // four in the bytes of one register against the four x bytes (dp4a), else
    // as the low halves.  Signed fields: the sign bit flipped (offset binary).
    constexpr uint32_t mh = B <= 24 ? low_bits(B - 16) * 0x01010101u : low_bits(B - 16) * 0x00010001u;
    constexpr uint32_t sflip =
        !SGN ? 0u : B <= 24 ? (1u << (B - 17)) * 0x01010101u : (1u << (B - 17)) * 0x00010001u;
    int lo0 = 0, lo1 = 0, hi = 0;
#pragma unroll
    for (int c = 0; c < 8; ++c) {
      uint32_t t[4];
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        const int bit = B * (4 * c + k), wi = bit >> 5, sh = bit & 31;
        t[k] = (sh + B <= 32) ? (f[wi] >> sh) : __funnelshift_r(f[wi], f[wi + 1], sh);
      }
      const uint32_t l01 = __byte_perm(t[0], t[1], 0x5410), l23 = __byte_perm(t[2], t[3], 0x5410);
      lo0 = dp2a_lo_us(l01, xw[c], lo0);
      lo1 = dp2a_hi_us(l23, xw[c], lo1);
      if constexpr (B <= 24) {
        const uint32_t h01 = __byte_perm(t[0], t[1], 0x0062), h23 = __byte_perm(t[2], t[3], 0x0062);
        const uint32_t h = (__byte_perm(h01, h23, 0x5410) & mh) ^ sflip;
        hi = dp4a_us(h, xw[c], hi);
      } else {
        const uint32_t h01 = (__byte_perm(t[0], t[1], 0x7632) & mh) ^ sflip;
        const uint32_t h23 = (__byte_perm(t[2], t[3], 0x7632) & mh) ^ sflip;
        hi = dp2a_hi_us(h23, xw[c], dp2a_lo_us(h01, xw[c], hi));
      }
    }
    int64_t acc = (int64_t)(lo0 + lo1) + (int64_t)hi * 65536;
    if constexpr (SGN) acc -= (int64_t)xs * (1ll << (B - 1));
    return acc;
  }
}

// The staged words of a segment: b + 1 words from word `wo` of the slot
// (a generic pointer into shared memory: the loads take immediate offsets).
template <int B>
__device__ __forceinline__ void load_segment(uint32_t sp, uint32_t wo, uint32_t sh,
                                             uint32_t (&f)[B + 1]) {
  const uint32_t* w = reinterpret_cast<const uint32_t*>(__cvta_shared_to_generic(sp)) + wo;
#pragma unroll
  for (int j = 0; j <= B; ++j) f[j] = w[j];
#pragma unroll
  for (int j = 0; j < B; ++j) f[j] = __funnelshift_r(f[j], f[j + 1], sh);
}

}  // namespace seg
}  // namespace ccm
