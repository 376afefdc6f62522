// segment_range.cuh -- the products of a run of segments of one matrix with x,
// by one warp: the common core of the segment matvec (matvec_ragged.cu) and of
// the batched matvec (batch.cu).
//
// Row i of an m x n matrix is cut into nsr = ceil(n / 32) segments of 32 fields,
// numbered row-major.  The warp streams its segments through a ring of slots in
// shared memory (one 1-D cp.async.bulk per stage on the slot's mbarrier, bounded
// waits).  Lane l takes segment 32 p + l of a stage: the b + 1 words that cover
// it, funnel-shifted once to its first bit, then a dot product with x held as
// bytes (dp4a / dp2a, segment_dot.cuh).  x past the end of a row is zero, so the
// last segment needs no mask, and x of 9 to 14 bits is two balanced byte digits
// (two dot products per segment).
//
// Widths of 16 and 32 bits would have the lanes' segments in one or two banks,
// and x of more than 14 bits has no byte images; they take a field per lane
// instead: a segment is b whole words, so along a row a lane's shift is fixed
// and its word advances by b, and each field is one 64-bit multiply-add with x
// as int32 (field_range).  On rows of a few segments a lane has a segment again,
// every lane at another field of its own, so that neither the words nor x meet
// in a bank (lane_range).
//
// Row sums.  Rows of 32 segments or more: the lanes add to a running sum of the
// warp's current row, reduced (redux.sync on 26-bit parts) and added to y with
// one atomic when the warp leaves the row.  Shorter rows: every lane adds its
// segment's sum with an atomic of its own (a prefix sum over the lanes, which
// would leave one per row, holds the warp up for as long: 10,000 matrices 899
// against 891 us, 100000 x 128 35 against 32 us).
#pragma once

#include "async_copy.cuh"
#include "segment_dot.cuh"

namespace ccm {
namespace seg {

constexpr int kMaxX = 31;            // widest x
constexpr int kMaxByteX = 14;        // widest x as byte digits, signed or not
constexpr int kMaxLaneSegs = 8;      // segments per lane of a stage
constexpr int kMaxSlots = 4;         // ring depth limit

// Segments per lane of a stage of about stage_bytes at width b (a sub-step of
// 32 segments holds 128 b bytes of A).
__host__ __device__ constexpr uint32_t lane_segments(uint32_t stage_bytes, int b) {
  const uint32_t p = stage_bytes / (128u * (uint32_t)b);
  return p < 1 ? 1u : (p > (uint32_t)kMaxLaneSegs ? (uint32_t)kMaxLaneSegs : p);
}

// Bytes of a slot for widths up to bmax: the widest stage, the 12 bytes that
// the copy may start before it, and the b + 1 words that a lane reads from its
// segment's first word on, also where the segment is the short last one of a
// row: the highest word read is at most 32 P b + 4 + b words into the slot.
__host__ __device__ constexpr uint32_t slot_bytes(uint32_t stage_bytes, int bmax) {
  uint32_t m = 0;
  for (int b = 1; b <= bmax; ++b) {
    const uint32_t v = lane_segments(stage_bytes, b) * 128u * (uint32_t)b + 4u * (uint32_t)b;
    m = v > m ? v : m;
  }
  return (m + 64u + 127u) & ~127u;
}

// ---------------------------------------------------------------------------
// The x image: per byte digit [2][nsr][16] bytes (half h holds image bytes 16 h
// .. 16 h + 15 of every segment) and the nsr sums of x; or x as int32.
// ---------------------------------------------------------------------------
__host__ __device__ constexpr uint64_t digit_bytes(uint32_t nsr) {
  return (36ull * nsr + 15) & ~15ull;
}

enum XMode : uint32_t { kOneDigit = 0, kTwoDigits = 1, kFields = 2 };

// (Rows under 8 segments stay with byte digits at 16 and 32 bits: reducing every
// row costs more than the bank conflicts.)
__device__ __forceinline__ XMode x_mode(int b, int bx, int sx, uint32_t nsr) {
  if (bx > kMaxByteX || ((b == 16 || b == 32) && nsr >= 8)) return kFields;
  return (sx ? bx <= 8 : bx <= 7) ? kOneDigit : kTwoDigits;
}

// Lane `lane` of the warp that takes segment s writes entry 32 s + lane.
__device__ __forceinline__ void write_x(uint8_t* img, uint32_t nsr, uint32_t s, uint32_t lane,
                                        int v, int b, XMode mode) {
  if (mode == kFields) {
    reinterpret_cast<int*>(img)[32ull * s + lane] = v;
    return;
  }
  const uint32_t pos = xbyte_pos(lane, b);
  for (int d = mode; d >= 0; --d, img += digit_bytes(nsr)) {
    const int lo = d ? (int)(int8_t)v : v;  // balanced digit, then the rest
    v = (v - lo) >> 8;
    img[(pos / 16) * 16ull * nsr + 16ull * s + pos % 16] = (uint8_t)lo;
    const int sum = __reduce_add_sync(0xffffffffu, lo);
    if (lane == 0) reinterpret_cast<int*>(img + 32ull * nsr)[s] = sum;
  }
}

// ---------------------------------------------------------------------------
// One matrix, and the ring of one warp
// ---------------------------------------------------------------------------
struct MatView {
  const uint32_t* wa;
  const uint8_t* ximg;
  int64_t* y;
  uint32_t n, nsr;
  uint32_t dm, ds1, ds2;  // division by nsr

  __device__ __forceinline__ uint32_t row_of(uint32_t g) const { return div_seg(g, dm, ds1, ds2); }
  __device__ __forceinline__ uint64_t bit_of(uint32_t q, uint32_t s, int b) const {
    return ((uint64_t)q * n + 32u * s) * (uint32_t)b;
  }
};

// Slots used in turn; all are empty between two ranges, so the cursor of the
// waits is also where the next range's copies begin.
struct Ring {
  uint8_t* mem;
  uint64_t* bar;
  uint32_t slot_bytes, depth, stage_bytes;
  uint32_t slot, phase;  // of the next stage to wait for

  __device__ __forceinline__ void init(int lane) {
    slot = phase = 0;
    if (lane == 0) {
      for (uint32_t s = 0; s < depth; ++s) ax::mbar_init(&bar[s], 1);
      ax::mbar_init_fence();
    }
    __syncwarp();
  }
  // Segments [g0, g1) of A into slot `at`.
  __device__ __forceinline__ void issue(const MatView& M, int b, uint32_t g0, uint32_t g1,
                                        uint32_t at) const {
    const uint32_t q0 = M.row_of(g0), ql = M.row_of(g1 - 1), sl = g1 - 1 - ql * M.nsr;
    const uint64_t eb = ((uint64_t)ql * M.n + min(M.n, 32u * sl + 32u)) * (uint32_t)b;
    const uint64_t w_lo = (M.bit_of(q0, g0 - q0 * M.nsr, b) >> 5) & ~3ull;
    const uint64_t w_hi = (((eb + 31) >> 5) + 3) & ~3ull;  // (the words are padded to four)
    const uint32_t bytes = (uint32_t)((w_hi - w_lo) * 4);
    if (threadIdx.x % 32 == 0) {
      ax::mbar_expect_tx(&bar[at], bytes);
      ax::bulk_g2s(mem + at * slot_bytes, M.wa + w_lo, bytes, &bar[at]);
    }
  }
  // The first stages of [r0, r1), ss segments each.
  __device__ __forceinline__ void start(const MatView& M, int b, uint32_t r0, uint32_t r1,
                                        uint32_t ss) const {
    uint32_t at = slot;
    for (uint32_t k = 0; k < depth && r0 + k * ss < r1; ++k) {
      issue(M, b, r0 + k * ss, min(r0 + (k + 1) * ss, r1), at);
      if (++at == depth) at = 0;
    }
  }
  __device__ __forceinline__ bool wait() const { return ax::mbar_wait(&bar[slot], phase); }
  // The stage from g0 on has been read: its slot takes the stage `depth` on.
  __device__ __forceinline__ void release(const MatView& M, int b, uint32_t g0, uint32_t r1,
                                          uint32_t ss) {
    __syncwarp();
    ax::fence_proxy_async_smem();
    const uint32_t g = g0 + depth * ss;
    if (g < r1) issue(M, b, g, min(g + ss, r1), slot);
    if (++slot == depth) {
      slot = 0;
      phase ^= 1;
    }
  }
  // After a wait that gave up on the stage from g0 on: the copies still in
  // flight land before shared memory goes away (bounded).
  __device__ __forceinline__ void drain(uint32_t g0, uint32_t r1, uint32_t ss) {
    for (uint32_t k = 1; k < depth && g0 + k * ss < r1; ++k) {
      if (++slot == depth) {
        slot = 0;
        phase ^= 1;
      }
      wait();
    }
  }
};

__device__ __forceinline__ void add_y(int64_t* y, uint32_t row, int64_t v) {
  if (v) atomicAdd(reinterpret_cast<unsigned long long*>(y + row), (unsigned long long)v);
}

// The sum over the lanes (of 26-bit parts: none leaves 32 bits).
__device__ __forceinline__ int64_t warp_sum(int64_t v) {
  constexpr uint32_t kPart = (1u << 26) - 1;
  const uint32_t lo = __reduce_add_sync(0xffffffffu, (uint32_t)v & kPart);
  const uint32_t mid = __reduce_add_sync(0xffffffffu, (uint32_t)(v >> 26) & kPart);
  const int hi = __reduce_add_sync(0xffffffffu, (int)(v >> 52));
  return ((int64_t)hi << 52) + ((int64_t)mid << 26) + lo;
}

// Segments [r0, r1) at width B.  `started` is called once the first copies are
// under way: what it waits for, they hide.
template <int B, bool SGN, class F>
__device__ __forceinline__ bool segment_range(const MatView& M, Ring& ring, uint32_t r0,
                                              uint32_t r1, XMode mode, F& started) {
  const int lane = threadIdx.x % 32;
  const uint32_t nsr = M.nsr, ss = 32 * lane_segments(ring.stage_bytes, B);
  const int4* xb = reinterpret_cast<const int4*>(M.ximg);
  const int* xsum = reinterpret_cast<const int*>(M.ximg + 32ull * nsr);
  const bool long_rows = nsr >= 32;
  ring.start(M, B, r0, r1, ss);
  started();
  int64_t racc = 0;
  uint32_t rrow = M.row_of(r0);  // (long rows: the warp's row)
  for (uint32_t g0 = r0; g0 < r1; g0 += ss) {
    if (!ring.wait()) {
      ring.drain(g0, r1, ss);
      return false;
    }
    const uint32_t sp = ax::smem_u32(ring.mem + ring.slot * ring.slot_bytes);
    const uint32_t g1 = min(g0 + ss, r1);
    const uint32_t q0 = M.row_of(g0), s0 = g0 - q0 * nsr;
    const uint32_t bit0 = (uint32_t)M.bit_of(q0, s0, B) & 127u;
#pragma unroll 1
    for (uint32_t base = g0; base < g1; base += 32) {
      const uint32_t g = base + lane;
      const bool live = g < g1;
      const uint32_t gg = live ? g : base;  // a dead lane decodes a live segment, then drops it
      const uint32_t q = M.row_of(gg), s = gg - q * nsr;
      const int4 x0 = __ldg(xb + s), x1 = __ldg(xb + nsr + s);
      const int xs = SGN ? __ldg(xsum + s) : 0;
      const uint32_t bit = bit0 + ((q - q0) * M.n + 32u * s - 32u * s0) * (uint32_t)B;
      uint32_t f[B + 1];
      load_segment<B>(sp, bit >> 5, bit & 31u, f);
      flip_signs<B, SGN>(f);
      const int xw[8] = {x0.x, x0.y, x0.z, x0.w, x1.x, x1.y, x1.z, x1.w};
      int64_t acc = seg_dot_fast<B, SGN>(f, xw, xs);
      if (mode == kTwoDigits) {
        const uint8_t* img = M.ximg + digit_bytes(nsr);
        const int4* p = reinterpret_cast<const int4*>(img) + s;
        const int4 h0 = __ldg(p), h1 = __ldg(p + nsr);
        const int xh[8] = {h0.x, h0.y, h0.z, h0.w, h1.x, h1.y, h1.z, h1.w};
        const int xhs = SGN ? __ldg(reinterpret_cast<const int*>(img + 32ull * nsr) + s) : 0;
        acc += seg_dot_fast<B, SGN>(f, xh, xhs) * 256;
      }
      if (!live) acc = 0;
      const int top = (int)min(31u, g1 - 1 - base);
      if (long_rows) {
        // at most two rows meet in a step
        const bool cur = q == rrow;
        if (cur) racc += acc;
        const uint32_t qn = __shfl_sync(0xffffffffu, q, top);
        if (qn != rrow) {  // (uniform)
          const int64_t t = warp_sum(racc);
          if (lane == 0) add_y(M.y, rrow, t);
          rrow = qn;
          racc = cur ? 0 : acc;
        }
      } else {
        add_y(M.y, q, acc);
      }
    }
    ring.release(M, B, g0, r1, ss);
  }
  if (long_rows) {
    const int64_t t = warp_sum(racc);
    if (lane == 0) add_y(M.y, rrow, t);
  }
  return true;
}

// Segments [r0, r1), a field per lane, at run-time width.  V: the type a field
// is taken as (int where it fits: one 32 x 32 -> 64-bit multiply-add).
template <bool SGN, typename V, class F>
__device__ __forceinline__ bool field_range(const MatView& M, Ring& ring, uint32_t r0, uint32_t r1,
                                            int b, F& started) {
  const int lane = threadIdx.x % 32, sh = 32 - b;
  const uint32_t nsr = M.nsr, ss = 32 * lane_segments(ring.stage_bytes, b);
  const int* xi = reinterpret_cast<const int*>(M.ximg) + lane;
  ring.start(M, b, r0, r1, ss);
  started();
  int64_t racc = 0;
  uint32_t q = M.row_of(r0), s = r0 - q * nsr;
  for (uint32_t g0 = r0; g0 < r1; g0 += ss) {
    if (!ring.wait()) {
      ring.drain(g0, r1, ss);
      return false;
    }
    const uint32_t* words = reinterpret_cast<const uint32_t*>(ring.mem + ring.slot * ring.slot_bytes);
    uint32_t g = g0;
    const uint32_t g1 = min(g0 + ss, r1);
    const uint64_t w_lo = (M.bit_of(q, s, b) >> 5) & ~3ull;
    while (g < g1) {
      // the segments of row q in this stage: this lane's field moves b words on
      const uint32_t cnt = min(nsr - s, g1 - g);
      const uint32_t bit = (uint32_t)(M.bit_of(q, s, b) - w_lo * 32) + lane * b;
      const uint32_t* w = words + (bit >> 5);
      const uint32_t at = bit & 31u;
      const int* x = xi + 32 * s;
#pragma unroll 8
      for (uint32_t c = 0; c < cnt; ++c, w += b, x += 32) {
        const uint32_t t = __funnelshift_r(w[0], w[1], at) << sh;
        const V v = SGN ? (V)((int)t >> sh) : (V)(t >> sh);
        racc += (long long)v * __ldg(x);
      }
      g += cnt;
      s += cnt;
      if (s == nsr) {
        const int64_t t = warp_sum(racc);
        if (lane == 0) add_y(M.y, q, t);
        racc = 0;
        s = 0;
        ++q;
      }
    }
    ring.release(M, b, g0, r1, ss);
  }
  if (s) {
    const int64_t t = warp_sum(racc);
    if (lane == 0) add_y(M.y, q, t);
  }
  return true;
}

// Segments [r0, r1), a segment per lane and its fields two by two, at run-time
// width (V as above).  Lane l begins with pair `turn` of its segment and goes
// round its end: where all begin at pair l, up to 11 lanes' words lie in one bank
// at some widths (30 bits; by counting); with this turn 2.4 on average over widths
// and row lengths, at most 3.5.  For rows of fewer than kShortRow segments (the
// caller's): field_range sums every row over the warp, which on such rows takes
// longer than the products.  Bound by the integer pipe (about 10 instructions per
// field).  Measured on GB300 (2,500 matrices at
// 12 bits, x of 16 bits, us per batch; field_range / this): 5714 x 7 2025 / 595,
// 2500 x 16 900 / 252, 625 x 64 303 / 130, 200 x 200 218 / 139, 156 x 256 141 /
// 126, 100 x 400 180 / 170, 83 x 480 (15 segments) 171 / 162; at 16 segments
// field_range takes 121.  (Fields one by one, 14 instructions each: 154 at 625 x
// 64, 154 at 200 x 200.)  A function of its own: inlined, it had k_batch_mv spill
// registers on the other paths (2 to 4 %).  The copies of the first stages are
// under way when it is called; it returns the ring's slot and phase, or kGaveUp.
constexpr uint32_t kGaveUp = 0xffffffffu;

// (A pointer into shared memory that comes as an argument is a generic one.)
__device__ __forceinline__ uint32_t ld_shared(uint32_t addr) {
  uint32_t v;
  asm volatile("ld.shared.u32 %0, [%1];\n" : "=r"(v) : "r"(addr) : "memory");
  return v;
}

template <bool SHORT, bool SGN, typename V>
__device__ __noinline__ uint32_t lane_range(MatView M, Ring ring, uint32_t r0, uint32_t r1, int b) {
  const uint32_t lane = threadIdx.x % 32, sh = 32 - b;
  const uint32_t nsr = M.nsr, ss = 32 * lane_segments(ring.stage_bytes, b);
  const int* xi = reinterpret_cast<const int*>(M.ximg);
  // pairs of a segment (of the only one of a row, rounded up to a power of two: x
  // is zero past the end)
  const uint32_t pairs = !SHORT ? 16u : M.n <= 2 ? 1u : 1u << (31 - __clz((int)M.n - 1));
  const uint32_t turn = 11 * (lane + (lane >> 4));  // (lane l's first pair)
  for (uint32_t g0 = r0; g0 < r1; g0 += ss) {
    if (!ring.wait()) {
      ring.drain(g0, r1, ss);
      return kGaveUp;
    }
    const uint32_t words = ax::smem_u32(ring.mem + ring.slot * ring.slot_bytes);
    const uint32_t g1 = min(g0 + ss, r1);
    const uint32_t q0 = M.row_of(g0), s0 = g0 - q0 * nsr;
    const uint32_t bit0 = (uint32_t)M.bit_of(q0, s0, b) & 127u;
#pragma unroll 1
    for (uint32_t g = g0 + lane; g < g1; g += 32) {
      const uint32_t q = M.row_of(g), s = g - q * nsr;
      const uint32_t bit = bit0 + ((q - q0) * M.n + 32u * s - 32u * s0) * (uint32_t)b;
      const int* x = xi + 32 * s;
      int64_t acc = 0;
#pragma unroll 4
      for (uint32_t j = 0; j < pairs; ++j) {
        const uint32_t e = 2 * ((j + turn) & (pairs - 1)), at = bit + e * (uint32_t)b;
        const uint32_t w = words + (at >> 5) * 4;
        const uint32_t w0 = ld_shared(w), w1 = ld_shared(w + 4), w2 = ld_shared(w + 8);
        const uint32_t lo = __funnelshift_r(w0, w1, at), hi = __funnelshift_r(w1, w2, at);
        const uint32_t t0 = lo << sh, t1 = __funnelshift_rc(lo, hi, b) << sh;
        const int2 xv = __ldg(reinterpret_cast<const int2*>(x + e));
        acc += (long long)(SGN ? (V)((int)t0 >> sh) : (V)(t0 >> sh)) * xv.x;
        acc += (long long)(SGN ? (V)((int)t1 >> sh) : (V)(t1 >> sh)) * xv.y;
      }
      add_y(M.y, q, acc);
    }
    ring.release(M, b, g0, r1, ss);
  }
  return ring.slot | ring.phase << 8;
}

// Segments [r0, r1) of a matrix of fields of b bits (1 .. 32): false when a
// wait gave up.
template <uint32_t kShortRow, class F>
__device__ __forceinline__ bool matrix_range(const MatView& M, Ring& ring, uint32_t r0, uint32_t r1,
                                             int b, bool sgn, XMode mode, F started) {
  if (mode == kFields && M.nsr < kShortRow) {
    ring.start(M, b, r0, r1, 32 * lane_segments(ring.stage_bytes, b));
    started();
    const uint32_t at =
        M.n < 32 ? (sgn ? lane_range<true, true, int>(M, ring, r0, r1, b)
                        : lane_range<true, false, long long>(M, ring, r0, r1, b))
                 : (sgn ? lane_range<false, true, int>(M, ring, r0, r1, b)
                        : b < 32 ? lane_range<false, false, int>(M, ring, r0, r1, b)
                                 : lane_range<false, false, long long>(M, ring, r0, r1, b));
    if (at == kGaveUp) return false;
    ring.slot = at & 255u;
    ring.phase = at >> 8;
    return true;
  }
  if (mode == kFields)
    return sgn ? field_range<true, int>(M, ring, r0, r1, b, started)
               : b < 32 ? field_range<false, int>(M, ring, r0, r1, b, started)
                        : field_range<false, long long>(M, ring, r0, r1, b, started);
  switch (2 * b + (sgn ? 1 : 0)) {
#define CCM_SEG(B)                                                              \
  case 2 * B: return segment_range<B, false>(M, ring, r0, r1, mode, started); \
  case 2 * B + 1: return segment_range<B, true>(M, ring, r0, r1, mode, started);
    CCM_SEG(1) CCM_SEG(2) CCM_SEG(3) CCM_SEG(4) CCM_SEG(5) CCM_SEG(6) CCM_SEG(7) CCM_SEG(8)
    CCM_SEG(9) CCM_SEG(10) CCM_SEG(11) CCM_SEG(12) CCM_SEG(13) CCM_SEG(14) CCM_SEG(15) CCM_SEG(16)
    CCM_SEG(17) CCM_SEG(18) CCM_SEG(19) CCM_SEG(20) CCM_SEG(21) CCM_SEG(22) CCM_SEG(23)
    CCM_SEG(24) CCM_SEG(25) CCM_SEG(26) CCM_SEG(27) CCM_SEG(28) CCM_SEG(29) CCM_SEG(30)
    CCM_SEG(31) CCM_SEG(32)
#undef CCM_SEG
    default: return true;
  }
}

}  // namespace seg
}  // namespace ccm
