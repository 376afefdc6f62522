// matvec_ragged.cu -- y = A x for rows that begin anywhere in a word (any
// number of columns, fields of at most 32 bits, x of at most 31).
//
// Row i is cut into ceil(n / 32) segments of 32 fields, numbered row-major.
// A persistent grid gives every warp a contiguous run of segments, streamed
// through a ring of two slots in shared memory (one 1-D cp.async.bulk per
// stage on the slot's mbarrier, bounded waits).  Lane l takes segment 32 p + l
// of a stage: the b + 1 words that cover it, funnel-shifted once to its first
// bit, then a dot product with x held as bytes (dp4a / dp2a, segment_dot.cuh).
// x past the end of a row is zero, so the last segment needs no mask, and x of
// 9 to 14 bits is two balanced byte digits (two dot products per segment).
//
// Widths of 16 and 32 bits would have the lanes' segments in one or two banks, and x of more than 14 bits has no byte images; they take a field per
// lane instead: a segment is b whole words, so along a row a lane's shift is
// fixed and its word advances by b, and each field is one 64-bit multiply-add
// with x as int32.
//
// Row sums: lanes add to a running sum of the warp's current row; when the
// warp leaves the row the sums of the lanes are reduced (redux.sync on 26-bit
// parts) and added to y with one atomic.  Rows of fewer
// than 32 segments change several times per step; there every lane adds its
// own sum when its row changes.
//
// Bound by the integer pipe (about 4 instructions per field: words, funnel
// shifts, masks, dot) beside the stream of A.  Measured on GB300 (whole call,
// 20011 x 5003, x of 8 bits; one field per lane and step from global memory
// before): 14 bits 392 -> 47 us (3.7 TB/s), 16 bits 335 -> 62, 32 bits 76 us
// (5.3 TB/s).
#include "async_copy.cuh"
#include "kernels.h"
#include "pack_engine.cuh"
#include "segment_dot.cuh"

namespace ccm {
namespace mvr {

using namespace seg;

constexpr int kThreads = 256;
constexpr int kWarps = kThreads / 32;
constexpr int kCtas = 3;             // per SM
constexpr int kSlots = 2;            // (a third costs more L1, which holds x, than it hides)
constexpr uint32_t kStageBytes = 4096;
constexpr int kMaxX = 31;            // widest x
constexpr int kMaxByteX = 14;        // widest x as byte digits, signed or not

// Segments per lane of a stage at width b (a sub-step of 32 segments holds
// 128 b bytes of A).
__host__ __device__ constexpr uint32_t lane_segs(int b) {
  const uint32_t p = kStageBytes / (128u * (uint32_t)b);
  return p < 1 ? 1 : p > 8 ? 8 : p;
}

// Bytes of a slot for widths up to bmax: the widest stage, the 12 bytes that
// the copy may start before it, and the b + 1 words that a lane reads from its
// segment's first word on, also where the segment is the short last one.
__host__ __device__ constexpr uint32_t slot_bytes(int bmax) {
  uint32_t m = 0;
  for (int b = 1; b <= bmax; ++b) {
    const uint32_t v = lane_segs(b) * 128u * (uint32_t)b + 4u * (uint32_t)b;
    m = v > m ? v : m;
  }
  return (m + 64u + 127u) & ~127u;
}

struct Args {
  ccm_header* out;
  const ccm_header* ha;
  const uint32_t* wa;
  uint64_t a_cap;
  const ccm_header* hx;
  const uint32_t* wx;
  uint64_t x_cap;
  uint64_t m, n;
  uint32_t nsr;       // segments per row
  uint32_t nseg;      // m * nsr
  DivSeg div;         // by nsr
  uint8_t* ximg;      // per digit: bytes [2][nsr][16], then the nsr sums of x; or x as int32
  int64_t* y;
  uint32_t slot;      // bytes of a ring slot
  int fresh;          // initialise y's header and sums (0: a further product term)
};

// Bytes of one digit's image.
__host__ __device__ constexpr uint64_t digit_bytes(uint32_t nsr) {
  return (36ull * nsr + 15) & ~15ull;
}

__device__ __forceinline__ int x_digits(int bx, int sx) { return (sx ? bx <= 8 : bx <= 7) ? 1 : 2; }

// A field per lane rather than a segment.  (Rows of a few segments stay with a
// segment per lane: reducing every row costs more than the bank conflicts.)
__device__ __forceinline__ bool field_lanes(int b, int bx, uint32_t nsr) {
  return bx > kMaxByteX || ((b == 16 || b == 32) && nsr >= 8);
}

// Validates A and x, initialises y's header and sums, decodes x into the byte
// images (a warp per segment).
__global__ void __launch_bounds__(256) k_rag_init(const __grid_constant__ Args a) {
  ax::grid_dep_launch();
  const HeaderView ha = load_header(a.ha), hx = load_header(a.hx);
  int st = check_header(ha, a.m, a.n, a.a_cap);
  if (st == CCM_OK) st = check_header(hx, a.n, 1, a.x_cap);
  if (a.fresh) {
    if (blockIdx.x == 0 && threadIdx.x == 0) {
      ccm_header* o = a.out;
      o->magic = CCM_MAGIC;
      o->width = 0;
      o->is_signed = 0;
      o->status = st;
      o->rows = a.m;
      o->cols = 1;
      o->nwords = 0;
      o->stat_or = 0;
      o->stat_neg = 0;
      o->reserved0 = 0;
      o->reserved1 = 0;
    }
    for (uint64_t i = (uint64_t)blockIdx.x * 256 + threadIdx.x; i < a.m;
         i += (uint64_t)gridDim.x * 256)
      a.y[i] = 0;
  }
  if (st != CCM_OK) return;
  const int b = ha.width, bx = hx.width, sx = hx.is_signed, nd = x_digits(bx, sx);
  const uint32_t lane = threadIdx.x % 32;
  const uint32_t pos = xbyte_pos(lane, b);
  for (uint32_t s = blockIdx.x * 8 + threadIdx.x / 32; s < a.nsr; s += gridDim.x * 8) {
    const uint64_t j = 32ull * s + lane;
    int v = j < a.n ? (int)decode_field(a.wx, j, bx, sx) : 0;
    if (field_lanes(b, bx, a.nsr)) {
      reinterpret_cast<int*>(a.ximg)[j] = v;
      continue;
    }
    for (int d = 0; d < nd; ++d) {
      const int lo = d + 1 < nd ? (int)(int8_t)v : v;  // balanced digit, then the rest
      v = (v - lo) >> 8;
      uint8_t* img = a.ximg + d * digit_bytes(a.nsr);
      img[(pos / 16) * 16 * a.nsr + 16 * s + pos % 16] = (uint8_t)lo;
      const int sum = __reduce_add_sync(0xffffffffu, lo);
      if (lane == 0) reinterpret_cast<int*>(img + 32ull * a.nsr)[s] = sum;
    }
  }
}

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

// The ring of one warp over segments [r0, r1) of A at width b: stage k holds
// segments r0 + k SS .. (SS = 32 lane_segs(b)) and, in front of them, up to
// 127 bits of 16-byte rounding.
struct Ring {
  const Args& a;
  uint8_t* mem;
  uint64_t* bar;
  uint32_t r0, r1, ss, stages;
  int b;
  __device__ __forceinline__ uint32_t row_of(uint32_t g) const {
    return div_seg(g, a.div.m, a.div.s1, a.div.s2);
  }
  __device__ __forceinline__ uint64_t bit_of(uint32_t q, uint32_t s) const {
    return ((uint64_t)q * (uint32_t)a.n + 32u * s) * (uint32_t)b;
  }
  __device__ __forceinline__ void issue(uint32_t k) const {
    const uint32_t g0 = r0 + k * ss, g1 = min(g0 + ss, r1);
    const uint32_t q0 = row_of(g0), ql = row_of(g1 - 1), sl = g1 - 1 - ql * a.nsr;
    const uint64_t eb = ((uint64_t)ql * (uint32_t)a.n + min((uint32_t)a.n, 32u * sl + 32u)) * (uint32_t)b;
    const uint64_t w_lo = (bit_of(q0, g0 - q0 * a.nsr) >> 5) & ~3ull;
    const uint64_t w_hi = (((eb + 31) >> 5) + 3) & ~3ull;  // (the words are padded to four)
    const uint32_t bytes = (uint32_t)((w_hi - w_lo) * 4), slot = k % kSlots;
    if (threadIdx.x % 32 == 0) {
      ax::mbar_expect_tx(&bar[slot], bytes);
      ax::bulk_g2s(mem + slot * a.slot, a.wa + w_lo, bytes, &bar[slot]);
    }
  }
  __device__ __forceinline__ void start() const {
    for (uint32_t k = 0; k < kSlots && k < stages; ++k) issue(k);
  }
  __device__ __forceinline__ bool wait(uint32_t k) const {
    return ax::mbar_wait(&bar[k % kSlots], (k / kSlots) & 1);
  }
  // Stage k has been read: its slot takes stage k + kSlots.
  __device__ __forceinline__ void release(uint32_t k) const {
    __syncwarp();
    ax::fence_proxy_async_smem();
    if (k + kSlots < stages) issue(k + kSlots);
  }
  // After a wait that gave up on stage k: the copies still in flight land
  // before shared memory goes away (bounded).
  __device__ __forceinline__ void drain(uint32_t k) const {
    for (uint32_t j = k + 1; j < stages && j < k + kSlots; ++j) wait(j);
  }
};

// Segments [r0, r1) of A at width B by one warp.
template <int B, bool SGN>
__device__ __forceinline__ bool rag_range(const Args& a, uint8_t* mem, uint64_t* bar, uint32_t r0,
                                          uint32_t r1, int nd) {
  const int lane = threadIdx.x % 32;
  const uint32_t n = (uint32_t)a.n, nsr = a.nsr;
  constexpr uint32_t kSs = 32 * lane_segs(B);
  const Ring ring{a, mem, bar, r0, r1, kSs, (r1 - r0 + kSs - 1) / kSs, B};
  const int4* xb = reinterpret_cast<const int4*>(a.ximg);
  const int* xsum = reinterpret_cast<const int*>(a.ximg + 32ull * nsr);
  const bool long_rows = nsr >= 32;
  ring.start();
  int64_t racc = 0;
  uint32_t rrow = ring.row_of(r0);  // (long rows: the warp's row)
  bool ok = true;
  for (uint32_t k = 0; k < ring.stages; ++k) {
    if (!ring.wait(k)) {
      ring.drain(k);
      ok = false;
      break;
    }
    const uint32_t sp = ax::smem_u32(mem + k % kSlots * a.slot);
    const uint32_t g0 = r0 + k * ring.ss, g1 = min(g0 + ring.ss, r1);
    const uint32_t q0 = ring.row_of(g0), s0 = g0 - q0 * nsr;
    const uint32_t bit0 = (uint32_t)ring.bit_of(q0, s0) & 127u;
#pragma unroll 1
    for (uint32_t base = g0; base < g1; base += 32) {
      const uint32_t g = base + lane;
      const bool live = g < g1;
      const uint32_t gg = live ? g : base;  // a dead lane decodes a live segment, then drops it
      const uint32_t q = ring.row_of(gg), s = gg - q * nsr;
      const int4 x0 = __ldg(xb + s), x1 = __ldg(xb + nsr + s);
      const int xs = SGN ? __ldg(xsum + s) : 0;
      const uint32_t bit = bit0 + ((q - q0) * n + 32u * s - 32u * s0) * (uint32_t)B;
      uint32_t f[B + 1];
      load_segment<B>(sp, bit >> 5, bit & 31u, f);
      flip_signs<B, SGN>(f);
      const int xw[8] = {x0.x, x0.y, x0.z, x0.w, x1.x, x1.y, x1.z, x1.w};
      int64_t acc = seg_dot_fast<B, SGN>(f, xw, xs);
      if (nd > 1) {
        const uint8_t* img = a.ximg + digit_bytes(nsr);
        const int4* p = reinterpret_cast<const int4*>(img) + s;
        const int4 h0 = __ldg(p), h1 = __ldg(p + nsr);
        const int xh[8] = {h0.x, h0.y, h0.z, h0.w, h1.x, h1.y, h1.z, h1.w};
        const int xhs = SGN ? __ldg(reinterpret_cast<const int*>(img + 32ull * nsr) + s) : 0;
        acc += seg_dot_fast<B, SGN>(f, xh, xhs) * 256;
      }
      if (!live) acc = 0;
      if (long_rows) {
        // at most two rows meet in a step
        const bool cur = q == rrow;
        if (cur) racc += acc;
        const uint32_t qn = __shfl_sync(0xffffffffu, q, min(31u, g1 - 1 - base));
        if (qn != rrow) {  // (uniform)
          const int64_t t = warp_sum(racc);
          if (lane == 0) add_y(a.y, rrow, t);
          rrow = qn;
          racc = cur ? 0 : acc;
        }
      } else if (live) {
        if (q != rrow) {
          add_y(a.y, rrow, racc);
          rrow = q;
          racc = acc;
        } else {
          racc += acc;
        }
      }
    }
    ring.release(k);
  }
  if (long_rows) {
    const int64_t t = warp_sum(racc);
    if (lane == 0) add_y(a.y, rrow, t);
  } else {
    add_y(a.y, rrow, racc);
  }
  return ok;
}

// Segments [r0, r1) of A, a field per lane, at run-time width.  V: the type a
// field is taken as (int where it fits: one 32 x 32 -> 64-bit multiply-add).
template <bool SGN, typename V>
__device__ __forceinline__ bool field_range(const Args& a, uint8_t* mem, uint64_t* bar, uint32_t r0,
                                            uint32_t r1) {
  const int lane = threadIdx.x % 32, b = a.ha->width, sh = 32 - b;
  const uint32_t nsr = a.nsr;
  const uint32_t ss = 32 * lane_segs(b);
  const Ring ring{a, mem, bar, r0, r1, ss, (r1 - r0 + ss - 1) / ss, b};
  const int* xi = reinterpret_cast<const int*>(a.ximg) + lane;
  ring.start();
  int64_t racc = 0;
  uint32_t q = ring.row_of(r0), s = r0 - q * nsr;
  for (uint32_t k = 0; k < ring.stages; ++k) {
    if (!ring.wait(k)) {
      ring.drain(k);
      return false;
    }
    const uint32_t* slot = reinterpret_cast<const uint32_t*>(mem + k % kSlots * a.slot);
    uint32_t g = r0 + k * ring.ss;
    const uint32_t g1 = min(g + ring.ss, r1);
    const uint64_t w_lo = (ring.bit_of(q, s) >> 5) & ~3ull;
    while (g < g1) {
      // the segments of row q in this stage: this lane's field moves b words on
      const uint32_t cnt = min(nsr - s, g1 - g);
      const uint32_t bit = (uint32_t)(ring.bit_of(q, s) - w_lo * 32) + lane * b;
      const uint32_t* w = slot + (bit >> 5);
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
        if (lane == 0) add_y(a.y, q, t);
        racc = 0;
        s = 0;
        ++q;
      }
    }
    ring.release(k);
  }
  if (s) {
    const int64_t t = warp_sum(racc);
    if (lane == 0) add_y(a.y, q, t);
  }
  return true;
}

__global__ void __launch_bounds__(kThreads, kCtas) k_rag(const __grid_constant__ Args a) {
  extern __shared__ __align__(128) uint8_t s_ring[];
  __shared__ __align__(8) uint64_t s_bar[kWarps][kSlots];
  const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
  uint64_t* bar = s_bar[warp];
  if (lane == 0) {
    for (int s = 0; s < kSlots; ++s) ax::mbar_init(&bar[s], 1);
    ax::mbar_init_fence();
  }
  __syncwarp();
  ax::grid_dep_launch();
  ax::grid_dep_wait();
  if (a.out->status != CCM_OK) return;
  const uint64_t w = (uint64_t)blockIdx.x * kWarps + warp, W = (uint64_t)gridDim.x * kWarps;
  const uint32_t r0 = (uint32_t)(a.nseg * w / W), r1 = (uint32_t)(a.nseg * (w + 1) / W);
  if (r0 >= r1) return;
  uint8_t* ring = s_ring + (size_t)warp * kSlots * a.slot;
  const int nd = x_digits(a.hx->width, a.hx->is_signed);
  bool ok = true;
  if (field_lanes(a.ha->width, a.hx->width, a.nsr)) {
    const bool sgn = a.ha->is_signed;
    ok = sgn ? field_range<true, int>(a, ring, bar, r0, r1)
             : a.ha->width < 32 ? field_range<false, int>(a, ring, bar, r0, r1)
                                : field_range<false, long long>(a, ring, bar, r0, r1);
    if (!ok && lane == 0) set_status(a.out, CCM_E_TIMEOUT);
    return;
  }
  switch (2 * a.ha->width + (a.ha->is_signed ? 1 : 0)) {
#define CCM_RAG(B)                                                            \
  case 2 * B: ok = rag_range<B, false>(a, ring, bar, r0, r1, nd); break;      \
  case 2 * B + 1: ok = rag_range<B, true>(a, ring, bar, r0, r1, nd); break;
    CCM_RAG(1) CCM_RAG(2) CCM_RAG(3) CCM_RAG(4) CCM_RAG(5) CCM_RAG(6) CCM_RAG(7) CCM_RAG(8)
    CCM_RAG(9) CCM_RAG(10) CCM_RAG(11) CCM_RAG(12) CCM_RAG(13) CCM_RAG(14) CCM_RAG(15) CCM_RAG(16)
    CCM_RAG(17) CCM_RAG(18) CCM_RAG(19) CCM_RAG(20) CCM_RAG(21) CCM_RAG(22) CCM_RAG(23)
    CCM_RAG(24) CCM_RAG(25) CCM_RAG(26) CCM_RAG(27) CCM_RAG(28) CCM_RAG(29) CCM_RAG(30)
    CCM_RAG(31) CCM_RAG(32)
#undef CCM_RAG
    default: break;
  }
  if (!ok && lane == 0) set_status(a.out, CCM_E_TIMEOUT);
}

bool ragged_applies(uint64_t m, uint64_t n, int bmax_a, int bmax_x) {
  if (!m || !n || bmax_a > 32 || bmax_x > kMaxX) return false;
  return n < (1ull << 31) && m * ((n + 31) / 32) < (1ull << 31);
}

// `fresh`: y's header and sums are initialised here, else this is a further
// term added to the sums of a header already initialised.
void run_ragged(const ccm_matrix& a, const ccm_matrix& x, const ccm_matrix& y, void* ximg,
                int64_t* yv, bool fresh, cudaStream_t st) {
  const uint32_t nsr = (uint32_t)((a.cols + 31) / 32);
  const int bmax = width_bound(a.capacity, a.rows * a.cols);
  Args g{y.hdr, a.hdr, a.words, a.capacity, x.hdr, x.words, x.capacity, a.rows, a.cols, nsr,
         (uint32_t)(a.rows * nsr), DivSeg::make(nsr), (uint8_t*)ximg, yv, slot_bytes(bmax),
         fresh ? 1 : 0};
  const size_t smem = (size_t)kWarps * kSlots * g.slot;
  cudaFuncSetAttribute(k_rag, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  const unsigned gi = (unsigned)umin(umax((nsr + 7) / 8, fresh ? (a.rows + 2047) / 2048 : 1),
                                     (uint64_t)num_sms() * 2);
  k_rag_init<<<gi, 256, 0, st>>>(g);
  const bool pdl = !profile_armed();
  // whole sub-steps of 32 segments per warp
  const unsigned grid = (unsigned)umax(1, umin((uint64_t)num_sms() * kCtas,
                                               (g.nseg + 32 * kWarps - 1) / (32 * kWarps)));
  profile_begin(st);
  if (pdl)
    ax::launch_pdl(k_rag, dim3(grid), dim3(kThreads), smem, st, g);
  else
    k_rag<<<grid, kThreads, smem, st>>>(g);
  profile_end(st);
  note_launch(2);
}

}  // namespace mvr
}  // namespace ccm
