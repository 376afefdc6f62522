// matvec_ragged.cu -- y = A x for rows that begin anywhere in a word (any
// number of columns, fields of at most 32 bits, x of at most 31).
//
// A persistent grid gives every warp a contiguous run of the matrix's segments
// (segment_range.cuh): streamed through a ring of two slots per warp, 32 fields
// per lane, products with byte digits of x, one atomic per row and warp.
//
// Bound by the integer pipe (about 4 instructions per field: words, funnel
// shifts, masks, dot) beside the stream of A.  Measured on GB300 (whole call,
// 20011 x 5003, x of 8 bits; one field per lane and step from global memory
// before): 14 bits 392 -> 47 us (3.7 TB/s), 16 bits 335 -> 62, 32 bits 76 us
// (5.3 TB/s).
#include "async_copy.cuh"
#include "host_cache.h"
#include "kernels.h"
#include "pack_engine.cuh"
#include "segment_range.cuh"

namespace ccm {
namespace mvr {

using namespace seg;

constexpr int kThreads = 256;
constexpr int kWarps = kThreads / 32;
constexpr int kCtas = 3;             // per SM
constexpr int kSlots = 2;            // (a third costs more L1, which holds x, than it hides)
constexpr uint32_t kStageBytes = 4096;
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
  uint8_t* ximg;      // x image (segment_range.cuh)
  int64_t* y;
  uint32_t slot;      // bytes of a ring slot
  int fresh;          // initialise y's header and sums (0: a further product term)
};

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
  const int b = ha.width, bx = hx.width, sx = hx.is_signed;
  const XMode mode = x_mode(b, bx, sx, a.nsr);
  const uint32_t lane = threadIdx.x % 32;
  for (uint32_t s = blockIdx.x * 8 + threadIdx.x / 32; s < a.nsr; s += gridDim.x * 8) {
    const uint64_t j = 32ull * s + lane;
    write_x(a.ximg, a.nsr, s, lane, j < a.n ? (int)decode_field(a.wx, j, bx, sx) : 0, b, mode);
  }
}

__global__ void __launch_bounds__(kThreads, kCtas) k_rag(const __grid_constant__ Args a) {
  extern __shared__ __align__(128) uint8_t s_ring[];
  __shared__ __align__(8) uint64_t s_bar[kWarps][kSlots];
  const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
  Ring ring{s_ring + (size_t)warp * kSlots * a.slot, s_bar[warp], a.slot, kSlots, kStageBytes, 0, 0};
  ring.init(lane);
  ax::grid_dep_launch();
  ax::grid_dep_wait();
  if (a.out->status != CCM_OK) return;
  const uint64_t w = (uint64_t)blockIdx.x * kWarps + warp, W = (uint64_t)gridDim.x * kWarps;
  const uint32_t r0 = (uint32_t)(a.nseg * w / W), r1 = (uint32_t)(a.nseg * (w + 1) / W);
  if (r0 >= r1) return;
  const int b = a.ha->width;
  const MatView M{a.wa, a.ximg, a.y, (uint32_t)a.n, a.nsr, a.div.m, a.div.s1, a.div.s2};
  const XMode mode = x_mode(b, a.hx->width, a.hx->is_signed, a.nsr);
  // (without lane_range, whose call takes 8 registers from the other paths; taken
  // field by field it gave 45 -> 31 us at 235294 x 17 and x of 16 bits, and 16.4 ->
  // 17.4 at 20000 x 200)
  if (!matrix_range<0>(M, ring, r0, r1, b, a.ha->is_signed != 0, mode, [] {}) &&
      lane == 0)
    set_status(a.out, CCM_E_TIMEOUT);
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
         (uint32_t)(a.rows * nsr), DivSeg::make(nsr), (uint8_t*)ximg, yv, slot_bytes(kStageBytes, bmax),
         fresh ? 1 : 0};
  const size_t smem = (size_t)kWarps * kSlots * g.slot;
  static DeviceCache attr;  // (the attribute is the device's)
  int dev = 0;
  cudaGetDevice(&dev);
  attr.get(dev, 0, [] {  // (an error is the call's: CCM_E_CUDA)
    return cudaFuncSetAttribute(k_rag, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                kWarps * kSlots * (int)slot_bytes(kStageBytes, 32)) == cudaSuccess;
  });
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
