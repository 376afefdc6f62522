// batch.cu -- y_i = A_i x_i for thousands of packed matrices of uneven
// shapes and widths in one persistent launch.
//
// Row i of an m x n matrix is cut into ceil(n / 32) segments of up to 32
// fields; segments are numbered row-major within a matrix, and a work unit is
// a run of consecutive segments of one matrix (the plan's unit list).  Every
// warp of the persistent kernel takes units from an atomic ticket of its own
// (no CTA barrier: the warps of a CTA are independent) and runs each through
// its ring of D slots with the width-specialised segment code
// (segment_range.cuh).  The next unit's ticket, record and matrix are fetched
// while the first copies of the unit at hand are under way, so a unit begins
// with its copies.
//
// The tickets hand out the units in the order of their matrices' codes
// (width, sign, form of x): after the initialisation a kernel sorts them by
// counting.  So at any time the warps of an SM decode one or two widths, and
// the code of one width-specialised decode stays in the instruction cache.
//
// The warp that completes the last unit of a matrix (per-matrix counter)
// re-packs that matrix's y at its exact width (width rule of Eq. 1 with the
// two's complement reading) and writes y's header.  The launches can be
// captured in a CUDA graph.
#include <cstring>
#include <vector>

#include "async_copy.cuh"
#include "ccm_device.cuh"
#include "kernels.h"
#include "segment_range.cuh"

namespace ccm {
namespace bt {

using namespace seg;

constexpr int kThreads = 256;
constexpr int kWarps = kThreads / 32;
constexpr int kMaxCols = 8192;       // x of at most 8192 entries per matrix
constexpr uint32_t kDefaultStageBytes = 3072;
constexpr uint32_t kShortRow = 16;   // segments of a row from which field_range is ahead of lane_range

struct Mat {
  const ccm_header* ha;
  const uint32_t* wa;
  const ccm_header* hx;
  const uint32_t* wx;
  ccm_header* hy;
  uint32_t* wy;
  uint64_t a_cap, x_cap, y_cap;
  uint32_t m, n;
  uint64_t y_off;      // offset of this matrix's rows in the int64 y scratch
  uint32_t units;      // work units of this matrix
  uint64_t x_off;      // offset of this matrix's x image (ints; a multiple of 32)
  uint32_t nseg_row;   // segments per row, ceil(n / 32)
  uint32_t dm, ds1, ds2;  // v / nseg_row as a multiply and shifts (DivSeg)
  uint32_t unit0;      // index of the matrix's first unit in the unit list
};

struct Unit {
  uint32_t mat;
  uint32_t seg0;   // first segment (row-major numbering within the matrix)
  uint32_t nseg;   // number of segments
  uint32_t pad;
};

// Per-matrix run-time code, written by k_batch_init from the headers: 0 for
// an entry that is skipped (its y header holds the error), else
// width | sign << 7 | (2 - form of x) << 8: a field per lane, the slowest form,
// sorts first, so that the last units are not the longest.
__device__ __forceinline__ uint32_t make_code(int b, int sgn, XMode mode) {
  return (uint32_t)b | (sgn ? 1u << 7 : 0u) | ((2u - (uint32_t)mode) << 8);
}
__device__ __forceinline__ int code_width(uint32_t c) { return (int)(c & 127u); }
__device__ __forceinline__ bool code_signed(uint32_t c) { return (c >> 7) & 1u; }
__device__ __forceinline__ XMode code_mode(uint32_t c) { return (XMode)(2u - (c >> 8)); }

struct Args {
  const Mat* mats;
  const Unit* units;
  uint32_t nmats, nunits;
  int64_t* yscratch;
  uint32_t* ticket;     // unit dispenser
  uint32_t* done;       // per-matrix completed units
  uint32_t* codes;      // per-matrix run-time code
  uint32_t* order;      // unit indices in code order; order[nunits] = their count
  int* ximage;          // x image of every matrix (Mat::x_off)
  uint32_t slot_bytes;  // bytes of one ring slot
  uint32_t stage_bytes; // target bytes of A per stage
  uint32_t slots;       // ring depth D (2..4)
  uint32_t bmax;        // widest A the slots hold
};

// ---------------------------------------------------------------------------
// Initialisation: validate inputs, write y headers and codes, clear counters
// and the y scratch, decode x into its image.
// ---------------------------------------------------------------------------
constexpr int kInitThreads = 128;
__global__ void __launch_bounds__(kInitThreads) k_batch_init(const __grid_constant__ Args a) {
  const uint32_t i = blockIdx.x;  // one block per matrix
  const Mat& M = a.mats[i];
  // (every thread reads the headers: one round trip, no barrier)
  const HeaderView ha = load_header(M.ha), hx = load_header(M.hx);
  int st = check_header(ha, M.m, M.n, M.a_cap);
  if (st == CCM_OK) st = check_header(hx, M.n, 1, M.x_cap);
  // widths the kernel handles, and sums that provably fit int64
  if (st == CCM_OK && (ha.width > (int)a.bmax || hx.width > kMaxX ||
                       ha.width + hx.width + bitlen64(M.n) > 63))
    st = CCM_E_WIDTH;
  const uint32_t nsr = M.nseg_row;
  const int bx = hx.width, sx = hx.is_signed;
  const XMode mode = x_mode(ha.width, bx, sx, nsr);
  if (threadIdx.x == 0) {
    ccm_header* y = M.hy;
    y->magic = CCM_MAGIC;
    y->width = 0;
    y->is_signed = 0;
    y->status = st;
    y->rows = M.m;
    y->cols = 1;
    y->nwords = 0;
    y->stat_or = 0;
    y->stat_neg = 0;
    a.done[i] = 0;
    if (i == 0) *a.ticket = 0;
    a.codes[i] = st == CCM_OK ? make_code(ha.width, ha.is_signed, mode) : 0;
  }
  for (uint32_t r = threadIdx.x; r < M.m; r += kInitThreads) a.yscratch[M.y_off + r] = 0;
  if (st != CCM_OK) return;
  uint8_t* img = reinterpret_cast<uint8_t*>(a.ximage + M.x_off);
  const uint32_t lane = threadIdx.x % 32;
#pragma unroll 2
  for (uint32_t s = threadIdx.x / 32; s < nsr; s += kInitThreads / 32) {
    const uint32_t j = 32 * s + lane;
    write_x(img, nsr, s, lane, j < M.n ? (int)decode_field(M.wx, j, bx, sx) : 0, ha.width, mode);
  }
}

// ---------------------------------------------------------------------------
// Unit order: a counting sort of the valid entries' units by code.  Each CTA
// counts all the entries (4 bytes of code and one sector of the record each: 360 KB
// from L2 for 10,000) and those before its own slice, so it knows where its slice's units of every code go
// without waiting for another CTA; then a warp writes an entry's units.  (By
// one CTA, with one thread per entry: 105 us for 10,000 matrices.)
// ---------------------------------------------------------------------------
constexpr int kOrderThreads = 512;
constexpr int kCodes = 1024;  // codes: width, sign, form of x

__global__ void __launch_bounds__(kOrderThreads) k_batch_order(const __grid_constant__ Args a) {
  __shared__ uint32_t s_cnt[kCodes];   // units of every code, then where they begin
  __shared__ uint32_t s_mine[kCodes];  // units of the entries before this slice
  __shared__ uint32_t s_warp[kOrderThreads / 32];
  const int tid = threadIdx.x, lane = tid % 32, warp = tid / 32;
  for (int c = tid; c < kCodes; c += kOrderThreads) s_cnt[c] = s_mine[c] = 0;
  __syncthreads();
  const uint32_t i0 = (uint32_t)((uint64_t)a.nmats * blockIdx.x / gridDim.x);
  const uint32_t i1 = (uint32_t)((uint64_t)a.nmats * (blockIdx.x + 1) / gridDim.x);
#pragma unroll 4
  for (uint32_t i = tid; i < a.nmats; i += kOrderThreads) {
    const uint32_t code = a.codes[i], units = a.mats[i].units;
    if (!code) continue;
    atomicAdd(&s_cnt[code & (kCodes - 1)], units);
    if (i < i0) atomicAdd(&s_mine[code & (kCodes - 1)], units);
  }
  __syncthreads();
  {
    // exclusive scan of the counts, kCodes / kOrderThreads per thread
    constexpr int kPer = kCodes / kOrderThreads;
    uint32_t v[kPer], sum = 0;
#pragma unroll
    for (int k = 0; k < kPer; ++k) {
      v[k] = s_cnt[tid * kPer + k];
      sum += v[k];
    }
    uint32_t incl = sum;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      const uint32_t o = __shfl_up_sync(0xffffffffu, incl, d);
      if (lane >= d) incl += o;
    }
    if (lane == 31) s_warp[warp] = incl;
    __syncthreads();
    uint32_t run = incl - sum;
    for (int w = 0; w < warp; ++w) run += s_warp[w];
    if (blockIdx.x == 0 && tid == kOrderThreads - 1) a.order[a.nunits] = run + sum;  // to hand out
#pragma unroll
    for (int k = 0; k < kPer; ++k) {
      s_mine[tid * kPer + k] += run;
      run += v[k];
    }
  }
  __syncthreads();
  for (uint32_t i = i0 + warp; i < i1; i += kOrderThreads / 32) {
    const uint32_t code = a.codes[i];
    if (!code) continue;
    const uint32_t units = a.mats[i].units, unit0 = a.mats[i].unit0;
    uint32_t at = 0;
    if (lane == 0) at = atomicAdd(&s_mine[code & (kCodes - 1)], units);
    at = __shfl_sync(0xffffffffu, at, 0);
    for (uint32_t k = lane; k < units; k += 32) a.order[at + k] = unit0 + k;
  }
}

// Re-pack y of one matrix at its exact width; the whole warp takes part
// (lane l assembles the b words of the 32-field groups l, l + 32, ...).
__device__ void pack_y_warp(const Mat& M, const int64_t* __restrict__ ys, int lane) {
  const uint32_t m = M.m;
  uint64_t orv = 0;
  uint32_t neg = 0;
  for (uint32_t i = lane; i < m; i += 32) {
    const int64_t v = __ldcg(ys + i);
    orv |= fold(v);
    neg |= (uint32_t)(v < 0);
  }
  orv = warp_or64(orv);
  neg = __reduce_or_sync(0xffffffffu, neg);
  const int b = width_from_stats(orv, neg);
  const uint64_t nw = words_for(m, b);
  const bool fits = nw <= M.y_cap;
  if (lane == 0) {
    ccm_header* h = M.hy;
    h->stat_or = orv;
    h->stat_neg = neg;
    h->width = b;
    h->is_signed = neg ? 1 : 0;
    h->nwords = nw;
    if (!fits) h->status = CCM_E_CAPACITY;
  }
  if (!fits) return;
  const uint64_t mask = field_mask(b);
  const uint32_t groups = (m + 31) / 32;
  for (uint32_t g = lane; g < groups; g += 32) {
    uint64_t w = (uint64_t)g * b;  // first word of the group
    unsigned __int128 buf = 0;     // bits not yet written
    int fill = 0;
    for (int e = 0; e < 32; ++e) {
      const uint64_t i = (uint64_t)g * 32 + e;
      const uint64_t pat = i < m ? ((uint64_t)__ldcg(ys + i) & mask) : 0;
      buf |= (unsigned __int128)pat << fill;
      fill += b;
      while (fill >= 32) {
        if (w < nw) M.wy[w] = (uint32_t)buf;
        ++w;
        buf >>= 32;
        fill -= 32;
      }
    }
  }
  // words past the last group's (the 16-byte padding)
  for (uint64_t w = (uint64_t)groups * b + lane; w < nw; w += 32) M.wy[w] = 0;
}

// ---------------------------------------------------------------------------
// The persistent kernel
// ---------------------------------------------------------------------------
// A unit with its matrix, as lane 0 fetches it for its warp.
struct alignas(16) Job {
  MatView view;
  uint32_t seg0, nseg, code, mat;
  uint32_t units;  // of the matrix; 0: no unit left
};

// Dynamic shared memory: each warp's D ring slots.
__global__ void __launch_bounds__(kThreads, 3) k_batch_mv(const __grid_constant__ Args a) {
  extern __shared__ __align__(128) uint8_t s_ring[];
  __shared__ __align__(8) uint64_t s_bar[kWarps][kMaxSlots];
  __shared__ Job s_job[kWarps];
  const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
  Ring ring{s_ring + (size_t)warp * a.slots * a.slot_bytes, s_bar[warp], a.slot_bytes, a.slots,
            a.stage_bytes, 0, 0};
  ring.init(lane);
  const uint32_t count = a.order[a.nunits];  // units to hand out (the valid entries')
  uint32_t ticket = 0;                       // lane 0: the next unit's
  if (lane == 0) ticket = atomicAdd(a.ticket, 1u);
  // Lane 0: the unit of `ticket` into the warp's job.
  auto fetch = [&] {
    if (lane == 0) {
      Job j{};
      if (ticket < count) {
        const Unit u = a.units[a.order[ticket]];
        const Mat& M = a.mats[u.mat];
        j.view = MatView{M.wa, reinterpret_cast<const uint8_t*>(a.ximage + M.x_off),
                         a.yscratch + M.y_off, M.n, M.nseg_row, M.dm, M.ds1, M.ds2};
        j.seg0 = u.seg0;
        j.nseg = u.nseg;
        j.code = a.codes[u.mat];
        j.mat = u.mat;
        j.units = M.units;
      }
      s_job[warp] = j;
    }
  };
  fetch();
  __syncwarp();
  Job job = s_job[warp];
  while (job.units) {
    auto next = [&] {
      if (lane == 0) ticket = atomicAdd(a.ticket, 1u);
      fetch();
    };
    bool ok = true;
    if (job.nseg)
      ok = matrix_range<kShortRow>(job.view, ring, job.seg0, job.seg0 + job.nseg, code_width(job.code),
                        code_signed(job.code), code_mode(job.code), next);
    else
      next();
    if (!ok) {
      // a wait gave up: mark the entries whose units this warp holds
      if (lane == 0) {
        set_status(a.mats[job.mat].hy, CCM_E_TIMEOUT);
        if (s_job[warp].units) set_status(a.mats[s_job[warp].mat].hy, CCM_E_TIMEOUT);
      }
      break;
    }
    // the unit is complete; the warp completing a matrix packs its y
    __threadfence();
    __syncwarp();
    uint32_t fin = 0;
    if (lane == 0) fin = atomicAdd(a.done + job.mat, 1u) + 1 == job.units;
    fin = __shfl_sync(0xffffffffu, fin, 0);
    if (fin) {
      __threadfence();
      pack_y_warp(a.mats[job.mat], job.view.y, lane);
    }
    __syncwarp();
    job = s_job[warp];
    __syncwarp();
  }
}

}  // namespace bt
}  // namespace ccm

// ---------------------------------------------------------------------------
// Host side
// ---------------------------------------------------------------------------
namespace ccm {
namespace bt {

size_t align256(size_t v) { return (v + 255) & ~(size_t)255; }

// x image of an n-column matrix: whole 32-field segments.
uint64_t x_image_ints(uint64_t cols) { return (cols + 31) / 32 * 32; }

// Workspace: int64 y scratch, per-matrix done counters, per-matrix codes,
// the ticket, x images.
size_t ws_done(uint64_t yrows) { return align256(yrows * 8); }
size_t ws_codes(uint64_t yrows, uint32_t count) {
  return ws_done(yrows) + align256((size_t)count * 4);
}
size_t ws_ticket(uint64_t yrows, uint32_t count) {
  return ws_codes(yrows, count) + align256((size_t)count * 4);
}
size_t ws_order(uint64_t yrows, uint32_t count) { return ws_ticket(yrows, count) + 256; }
size_t ws_ximage(uint64_t yrows, uint32_t count, uint64_t units) {
  return ws_order(yrows, count) + align256((units + 1) * 4);
}
size_t ws_bytes(uint64_t yrows, uint32_t count, uint64_t xints, uint64_t units) {
  return ws_ximage(yrows, count, units) + align256(xints * 4);
}

struct Layout {
  uint32_t nmats = 0, nunits = 0;
  uint64_t yrows = 0;
  size_t mats_off = 0, units_off = 0, bytes = 0;
};

uint64_t segments_of(const ccm_batch_entry& e) { return e.a.rows * ((e.a.cols + 31) / 32); }

int validate(const ccm_batch_entry& e) {
  const ccm_matrix &a = e.a, &x = e.x, &y = e.y;
  if (!a.hdr || !x.hdr || !y.hdr) return CCM_E_INVAL;
  if (x.rows != a.cols || x.cols != 1 || y.rows != a.rows || y.cols != 1) return CCM_E_SHAPE;
  if (a.cols > (uint64_t)kMaxCols || a.rows >= (1ull << 31)) return CCM_E_SHAPE;
  const uint64_t n = a.rows * a.cols;
  if (y.capacity < words_for(y.rows, 1)) return CCM_E_CAPACITY;
  auto al = [](const void* p) { return reinterpret_cast<uintptr_t>(p) % 16 == 0; };
  if (!al(a.hdr) || !al(x.hdr) || !al(y.hdr) || !al(a.words) || !al(x.words) || !al(y.words))
    return CCM_E_INVAL;
  if ((n && !a.words) || (a.cols && !x.words) || (y.capacity && !y.words)) return CCM_E_INVAL;
  return CCM_OK;
}

Layout layout(const ccm_batch_entry* e, int count, uint32_t unit_segs) {
  Layout L;
  L.nmats = (uint32_t)count;
  uint64_t units = 0;
  for (int i = 0; i < count; ++i) {
    const uint64_t s = segments_of(e[i]);
    units += s ? (s + unit_segs - 1) / unit_segs : 1;
    L.yrows += e[i].a.rows;
  }
  L.nunits = (uint32_t)units;
  L.mats_off = align256(sizeof(ccm_batch_info));
  L.units_off = L.mats_off + align256(sizeof(Mat) * (size_t)count);
  L.bytes = L.units_off + align256(sizeof(Unit) * (size_t)units);
  return L;
}

}  // namespace bt
}  // namespace ccm

extern "C" {

size_t ccm_batch_plan_bytes(const ccm_batch_entry* entries, int count, uint32_t unit_segments) {
  if (!entries || count <= 0 || unit_segments == 0) return 0;
  return ccm::bt::layout(entries, count, unit_segments).bytes;
}

size_t ccm_batch_workspace_bytes(const ccm_batch_entry* entries, int count) {
  if (!entries || count <= 0) return 0;
  uint64_t yrows = 0, xints = 0, units = 0;
  for (int i = 0; i < count; ++i) {
    yrows += entries[i].a.rows;
    xints += ccm::bt::x_image_ints(entries[i].a.cols);
    // the most units any plan cuts this entry into (unit_segments >= 32)
    units += ccm::umax(1, (ccm::bt::segments_of(entries[i]) + 31) / 32);
  }
  return ccm::bt::ws_bytes(yrows, (uint32_t)count, xints, units);
}

ccm_status ccm_batch_plan(const ccm_batch_entry* entries, int count, uint32_t unit_segments,
                          void* plan, size_t plan_bytes, ccm_batch_info* info) {
  using namespace ccm::bt;
  if (!entries || count <= 0 || !plan || !info || unit_segments == 0) return CCM_E_INVAL;
  if (unit_segments % 32) return CCM_E_INVAL;
  for (int i = 0; i < count; ++i) {
    int st = validate(entries[i]);
    if (st != CCM_OK) return (ccm_status)st;
  }
  Layout L = layout(entries, count, unit_segments);
  if (plan_bytes < L.bytes || reinterpret_cast<uintptr_t>(plan) % 256) return CCM_E_CAPACITY;
  std::vector<uint8_t> host(L.bytes, 0);
  Mat* mats = reinterpret_cast<Mat*>(host.data() + L.mats_off);
  Unit* units = reinterpret_cast<Unit*>(host.data() + L.units_off);
  uint64_t yoff = 0, xoff = 0, u = 0;
  for (int i = 0; i < count; ++i) {
    const ccm_batch_entry& e = entries[i];
    Mat& M = mats[i];
    M.ha = e.a.hdr;
    M.wa = e.a.words;
    M.hx = e.x.hdr;
    M.wx = e.x.words;
    M.hy = e.y.hdr;
    M.wy = e.y.words;
    M.a_cap = e.a.capacity;
    M.x_cap = e.x.capacity;
    M.y_cap = e.y.capacity;
    M.m = (uint32_t)e.a.rows;
    M.n = (uint32_t)e.a.cols;
    M.nseg_row = (uint32_t)((e.a.cols + 31) / 32);
    const DivSeg dv = DivSeg::make(M.nseg_row ? M.nseg_row : 1);
    M.dm = dv.m;
    M.ds1 = dv.s1;
    M.ds2 = dv.s2;
    M.y_off = yoff;
    yoff += e.a.rows;
    M.x_off = xoff;
    xoff += x_image_ints(e.a.cols);
    const uint64_t s = segments_of(e);
    const uint64_t nu = s ? (s + unit_segments - 1) / unit_segments : 1;
    M.units = (uint32_t)nu;
    M.unit0 = (uint32_t)u;
    for (uint64_t k = 0; k < nu; ++k, ++u) {
      units[u].mat = (uint32_t)i;
      units[u].seg0 = (uint32_t)(k * unit_segments);
      units[u].nseg = (uint32_t)(s ? ccm::umin(unit_segments, s - k * unit_segments) : 0);
    }
  }
  uint64_t maxcols = 0, maxw = 1;
  for (int i = 0; i < count; ++i) {
    maxcols = ccm::umax(maxcols, entries[i].a.cols);
    // the widest A the capacity admits (a valid header's width is at most this)
    const uint64_t n = entries[i].a.rows * entries[i].a.cols;
    if (n) maxw = ccm::umax(maxw, ccm::umin(entries[i].a.capacity * 32 / n, 32));
  }
  info->count = (uint32_t)count;
  info->max_cols = (uint32_t)maxcols;
  info->max_width = (uint32_t)maxw;
  info->slots = 0;
  info->stage_bytes = 0;
  info->reserved = 0;
  info->x_ints = xoff;
  info->units = L.nunits;
  info->y_rows = L.yrows;
  info->unit_segments = unit_segments;
  info->plan_bytes = L.bytes;
  std::memcpy(host.data(), info, sizeof(ccm_batch_info));
  if (cudaMemcpy(plan, host.data(), L.bytes, cudaMemcpyHostToDevice) != cudaSuccess)
    return CCM_E_CUDA;
  return CCM_OK;
}

ccm_status ccm_batch_matvec(const void* plan, const ccm_batch_info* info, void* ws,
                            size_t ws_bytes, int grid, ccm_stream_t stream) {
  using namespace ccm::bt;
  if (!plan || !info || !ws || info->count == 0) return CCM_E_INVAL;
  if (reinterpret_cast<uintptr_t>(ws) % 256) return CCM_E_INVAL;
  if (ws_bytes < ccm::bt::ws_bytes(info->y_rows, info->count, info->x_ints, info->units))
    return CCM_E_CAPACITY;
  Layout L;
  L.mats_off = align256(sizeof(ccm_batch_info));
  L.units_off = L.mats_off + align256(sizeof(Mat) * (size_t)info->count);
  Args a;
  a.mats = reinterpret_cast<const Mat*>((const uint8_t*)plan + L.mats_off);
  a.units = reinterpret_cast<const Unit*>((const uint8_t*)plan + L.units_off);
  a.nmats = info->count;
  a.nunits = info->units;
  a.yscratch = (int64_t*)ws;
  a.done = (uint32_t*)((uint8_t*)ws + ws_done(info->y_rows));
  a.codes = (uint32_t*)((uint8_t*)ws + ws_codes(info->y_rows, info->count));
  a.ticket = (uint32_t*)((uint8_t*)ws + ws_ticket(info->y_rows, info->count));
  a.order = (uint32_t*)((uint8_t*)ws + ws_order(info->y_rows, info->count));
  a.ximage = (int*)((uint8_t*)ws + ws_ximage(info->y_rows, info->count, info->units));
  // the warps' ring slots, sized for the widest A
  if (info->max_width < 1 || info->max_width > 32 || info->max_cols > (uint32_t)kMaxCols)
    return CCM_E_INVAL;
  a.bmax = info->max_width;
  if (info->slots != 0 && (info->slots < 2 || info->slots > (uint32_t)kMaxSlots))
    return CCM_E_INVAL;
  a.slots = info->slots ? info->slots : 3;
  if (info->stage_bytes != 0 && (info->stage_bytes < 128 || info->stage_bytes > 16384))
    return CCM_E_INVAL;
  a.stage_bytes = info->stage_bytes ? info->stage_bytes : kDefaultStageBytes;
  a.slot_bytes = ccm::seg::slot_bytes(a.stage_bytes, (int)a.bmax);
  // warps per CTA: 8, or 4 when that keeps more warps resident per SM (the
  // rings are per warp, so a smaller CTA packs the shared memory tighter)
  static size_t attr = 0;
  const size_t smem_max = (size_t)kWarps * a.slots * a.slot_bytes;
  if (smem_max > (size_t)ccm::max_smem_optin()) return CCM_E_INVAL;
  if (smem_max > attr) {
    if (cudaFuncSetAttribute(k_batch_mv, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)smem_max) != cudaSuccess)
      return CCM_E_CUDA;
    attr = smem_max;
  }
  static uint64_t occ_key = 0;  // (slots, slot bytes) of the cached choice
  static int occ_warps = kWarps, occ_per = 1;
  const uint64_t key = ((uint64_t)a.slots << 32) | a.slot_bytes;
  if (key != occ_key) {
    int best = 0;
    occ_warps = kWarps;
    occ_per = 1;
    for (int w = kWarps; w >= 4; w /= 2) {
      int p = 0;
      const size_t sm = (size_t)w * a.slots * a.slot_bytes;
      if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&p, k_batch_mv, 32 * w, sm) !=
          cudaSuccess)
        p = 0;
      if (p * w > best) best = p * w, occ_warps = w, occ_per = p;
    }
    if (best == 0) occ_per = 1;
    occ_key = key;
  }
  const int warps = occ_warps, per = occ_per;
  const size_t smem = (size_t)warps * a.slots * a.slot_bytes;
  if (grid <= 0) grid = ccm::num_sms() * per;  // one resident wave
  cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
  k_batch_init<<<info->count, kInitThreads, 0, st>>>(a);
  // (a slice of at least 64 entries per CTA)
  const unsigned order_grid =
      (unsigned)ccm::umax(1, ccm::umin((info->count + 63) / 64, (uint64_t)ccm::num_sms()));
  k_batch_order<<<order_grid, kOrderThreads, 0, st>>>(a);
  ccm::profile_begin(st);
  k_batch_mv<<<grid, 32 * warps, smem, st>>>(a);
  ccm::profile_end(st);
  ccm::note_launch(3);
  return cudaGetLastError() == cudaSuccess ? CCM_OK : CCM_E_CUDA;
}

}  // extern "C"
