// cta_pack.cuh -- a short vector of int64 values (up to 65,536) packed by a
// small grid in one launch: every CTA reads all the values for the width
// statistics (a few hundred KB of L2 reads at most), stages only its own
// groups of 32 fields in shared memory and packs them; CTA 0 writes the
// header and the pad words.  No CTA waits for another (k_pack_vec's y,
// k_pack_small's small dense input).
#pragma once

#include <type_traits>

#include "ccm_device.cuh"

namespace ccm {

constexpr uint32_t kVecGroupsPerCta = 16;  // 32-field groups a CTA packs
constexpr int kVecThreads = 512;

// CTAs for m values.
__host__ __device__ constexpr uint32_t vec_pack_ctas(uint64_t m) {
  return (uint32_t)(((m + 31) / 32 + kVecGroupsPerCta - 1) / kVecGroupsPerCta);
}

// Shared state of one CTA: its groups' fields (33 slots per group, so the 32
// lanes that fill a group hit 32 different banks) and the statistics.
struct VecPackSmem {
  uint64_t ys[kVecGroupsPerCta * 33];
  uint64_t s_or[kVecThreads / 32];
  uint32_t s_neg[kVecThreads / 32];
};

// 16 bytes of values.
template <typename T>
struct alignas(16) VecOf {
  T v[16 / sizeof(T)];
};

// Adds one value to the running statistics: o collects the folded values
// (32 bits of them for int32), ng the signs in its top bit.
__device__ __forceinline__ void add_stats(int64_t v, uint64_t& o, uint32_t& ng) {
  o |= fold(v);
  ng |= (uint32_t)(v >> 32);
}
__device__ __forceinline__ void add_stats(int32_t v, uint32_t& o, uint32_t& ng) {
  o |= (uint32_t)(v ^ (v >> 31));
  ng |= (uint32_t)v;
}

// The fields of groups [g0, g0 + kVecGroupsPerCta) of the mm values at src into
// sm.ys, and the statistics of all of them (OR of the folded values, any
// negative), reduced to every thread.  The statistics are what takes the time of
// a long vector: 16-byte loads, eight of them in flight per thread (an input
// aligned only to its entries is read one by one).  Measured on GB300 (packs of
// 65,536 entries, calls queued back to back; one entry per load before): int32
// 12.4 -> 6.2 us, int64 12.4 -> 8.3; 16,384 entries 6.2 -> 4.2 and 6.2.
template <typename T>
__device__ __forceinline__ void vec_stats_stage(const T* __restrict__ src, uint32_t mm,
                                                uint32_t g0, VecPackSmem& sm, uint64_t& orv,
                                                uint32_t& neg) {
  constexpr uint32_t kPer = 16 / sizeof(T);
  using Acc = typename std::conditional<sizeof(T) == 8, uint64_t, uint32_t>::type;
  static_assert(kVecGroupsPerCta * 32 == kVecThreads, "a thread stages one field");
  const uint32_t own = g0 * 32 + threadIdx.x;
  const int64_t mine = own < mm ? (int64_t)src[own] : 0;
  Acc o = 0;
  uint32_t ng = 0;
  const bool aligned = reinterpret_cast<uintptr_t>(src) % 16 == 0;
  const uint32_t nv = aligned ? mm / kPer : 0;  // whole vectors
  const VecOf<T>* vs = reinterpret_cast<const VecOf<T>*>(src);
  for (uint32_t base = threadIdx.x; base < nv; base += 8 * kVecThreads) {
    VecOf<T> x[8];
#pragma unroll
    for (int j = 0; j < 8; ++j)  // (past the end: the first vector again)
      x[j] = vs[base + j * kVecThreads < nv ? base + j * kVecThreads : 0];
#pragma unroll
    for (int j = 0; j < 8; ++j)
#pragma unroll
      for (uint32_t k = 0; k < kPer; ++k) add_stats(x[j].v[k], o, ng);
  }
  for (uint32_t base = nv * kPer + threadIdx.x; base < mm; base += 8 * kVecThreads) {
    T x[8];
#pragma unroll
    for (int j = 0; j < 8; ++j)
      x[j] = src[base + j * kVecThreads < mm ? base + j * kVecThreads : 0];
#pragma unroll
    for (int j = 0; j < 8; ++j) add_stats(x[j], o, ng);
  }
  sm.ys[(threadIdx.x >> 5) * 33 + (threadIdx.x & 31)] = (uint64_t)mine;
  const uint64_t o64 = warp_or64((uint64_t)o);
  ng = __reduce_or_sync(0xffffffffu, ng) >> 31;
  const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
  if (lane == 0) {
    sm.s_or[warp] = o64;
    sm.s_neg[warp] = ng;
  }
  __syncthreads();
  orv = 0;
  neg = 0;
  for (int w = 0; w < kVecThreads / 32; ++w) {
    orv |= sm.s_or[w];
    neg |= sm.s_neg[w];
  }
}

// Packs the staged groups [g0, g0 + kVecGroupsPerCta) of the mm fields at
// width b.  A group is b whole words; lane i of the warp that takes the group
// assembles its words i and i + 32 from the fields that overlap them (no
// word is written twice).  CTA 0 also zeroes the pad words from dw to nw.
__device__ __forceinline__ void vec_pack_groups(const VecPackSmem& sm, uint32_t mm, uint32_t g0,
                                                int b, uint32_t* words, uint64_t dw,
                                                uint64_t nw) {
  const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
  const uint64_t mask = field_mask(b);
  const uint32_t g1 = umin((mm + 31) / 32, g0 + kVecGroupsPerCta);
  int flo[2], fhi[2];  // fields overlapping word i (and i + 32) of a group
  for (int h = 0; h < 2; ++h) {
    const int wi = lane + 32 * h;
    flo[h] = wi * 32 / b;
    fhi[h] = (wi * 32 + 31) / b;
  }
  for (uint32_t g = g0 + warp; g < g1; g += kVecThreads / 32) {
    const uint32_t nf = umin(32, mm - g * 32);
    const uint32_t nwg = (uint32_t)((nf * (uint64_t)b + 31) / 32);  // words of this group
    const uint64_t* src = sm.ys + (g - g0) * 33;
    for (int h = 0; h < 2; ++h) {
      const uint32_t wi = lane + 32 * h;
      if (wi >= nwg) continue;
      uint32_t acc = 0;
      const int fe = fhi[h] < (int)nf - 1 ? fhi[h] : (int)nf - 1;
      for (int f = flo[h]; f <= fe; ++f) {
        const int o = f * b - (int)wi * 32;  // field start relative to the word
        const uint64_t pat = src[f] & mask;
        acc |= o >= 0 ? (uint32_t)(pat << o) : (uint32_t)(pat >> (-o));
      }
      words[(uint64_t)g * b + wi] = acc;
    }
  }
  if (blockIdx.x == 0)
    for (uint64_t W = dw + threadIdx.x; W < nw; W += kVecThreads) words[W] = 0;
}

}  // namespace ccm
