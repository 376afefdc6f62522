// pack.cu -- SM compression and decompression kernels (Methods, Method 1):
// width selection + pack of dense int32/int64 matrices, unpack, element
// access, and the elementwise operations whose results are re-packed by the
// same engine (add, scale).
#include "ew_kernels.cuh"
#include "async_copy.cuh"
#include "cta_pack.cuh"
#include "kernels.h"
#include "pack_engine.cuh"

namespace ccm {

int width_bound(uint64_t capacity, uint64_t n) {
  if (n == 0) return 64;
  return (int)umin(capacity * 32 / n, 64);
}

int bitlen_host(uint64_t v) {
  int l = 0;
  for (; v; v >>= 1) ++l;
  return l;
}

namespace {

// Width class of the group-engine kernels for a width bound (0: none, use
// the run-time-width kernels).
int ew_class(int bmax) { return bmax <= 8 ? 8 : bmax <= 16 ? 16 : bmax <= 32 ? 32 : 0; }

void launch_ew(int cls, const ge::EwCall& c, cudaStream_t st) {
  int launched;
  switch (cls) {
    case 8: launched = ge::launch_ew_class<8>(c, st); break;
    case 16: launched = ge::launch_ew_class<16>(c, st); break;
    default: launched = ge::launch_ew_class<32>(c, st); break;
  }
  note_launch(launched);
}

}  // namespace

int num_sms() {
  int dev = 0;
  cudaGetDevice(&dev);
  static DeviceCache sms;
  return sms.get(dev, 1, [&] {
    int v = 0;
    cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, dev);
    return v;
  });
}

int max_smem_optin() {
  int dev = 0;
  cudaGetDevice(&dev);
  static DeviceCache bytes;
  return bytes.get(dev, 48 * 1024, [&] {
    int v = 0;
    cudaDeviceGetAttribute(&v, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    return v;
  });
}

__global__ void k_init(InitArgs a) {
  ax::grid_dep_launch();  // a programmatically launched successor may start now
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    int st = CCM_OK;
    if (a.in0) st = check_input(a.in0, a.in0_rows, a.in0_cols, a.in0_capacity);
    if (st == CCM_OK && a.in1) st = check_input(a.in1, a.in1_rows, a.in1_cols, a.in1_capacity);
    ccm_header* o = a.out;
    o->magic = CCM_MAGIC;
    o->width = 0;
    o->is_signed = 0;
    o->status = st;
    o->rows = a.out_rows;
    o->cols = a.out_cols;
    o->nwords = 0;
    o->stat_or = 0;
    o->stat_neg = 0;
    o->reserved0 = 0;
    o->reserved1 = 0;
  }
  if (a.zero_ptr) {
    uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
    for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < a.zero_count; i += stride)
      a.zero_ptr[i] = 0;
  }
}

// Validates one more pair of inputs against an already initialised output:
// the first invalid header's status goes to the output header.
__global__ void k_check(InitArgs a) {
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    int st = CCM_OK;
    if (a.in0) st = check_input(a.in0, a.in0_rows, a.in0_cols, a.in0_capacity);
    if (st == CCM_OK && a.in1) st = check_input(a.in1, a.in1_rows, a.in1_cols, a.in1_capacity);
    if (st != CCM_OK) set_status(a.out, st);
  }
}

void launch_check(const ccm_matrix& p, const ccm_matrix& q, ccm_header* out, cudaStream_t st) {
  InitArgs ia{};
  ia.out = out;
  ia.in0 = p.hdr;
  ia.in0_rows = p.rows;
  ia.in0_cols = p.cols;
  ia.in0_capacity = p.capacity;
  ia.in1 = q.hdr;
  ia.in1_rows = q.rows;
  ia.in1_cols = q.cols;
  ia.in1_capacity = q.capacity;
  k_check<<<1, 32, 0, st>>>(ia);
  note_launch();
}

void launch_init(const InitArgs& a, cudaStream_t st) {
  int grid = 1;
  if (a.zero_ptr && a.zero_count > 256)
    grid = (int)umin((a.zero_count + 255) / 256, (uint64_t)num_sms() * 4);
  k_init<<<grid, 256, 0, st>>>(a);
  note_launch();
}

// ---------------------------------------------------------------------------
// pack / measure
// ---------------------------------------------------------------------------
// Finalises the header of a measure-only call (no words): width, sign, nwords.
__global__ void k_measure_finish(ccm_header* out, uint64_t n) {
  if (out->status != CCM_OK) return;
  int b = width_from_stats(out->stat_or, out->stat_neg);
  out->width = b;
  out->is_signed = out->stat_neg ? 1 : 0;
  out->nwords = words_for(n, b);
}

void run_measure(const void* dense, int dtype, uint64_t rows, uint64_t cols, ccm_header* hdr,
                 cudaStream_t st) {
  InitArgs ia{};
  ia.out = hdr;
  ia.out_rows = rows;
  ia.out_cols = cols;
  launch_init(ia, st);
  uint64_t n = rows * cols;
  if (n) {
    profile_begin(st);
    if (dtype == CCM_I64)
      launch_stats(ProdDenseI64{(const int64_t*)dense}, hdr, n, st);
    else
      launch_stats(ProdDenseI32{(const int32_t*)dense}, hdr, n, st);
    profile_end(st);
  }
  k_measure_finish<<<1, 1, 0, st>>>(hdr, n);
  note_launch();
}

size_t pack_workspace(uint64_t rows, uint64_t cols, uint64_t capacity) {
  const uint64_t n = rows * cols;
  const int cls = ew_class(width_bound(capacity, n));
  return (cls && n) ? ge::pack_ws_bytes(n, cls) : 0;
}

// A small dense input (n <= kSmallPack entries) packed in one launch by
// vec_pack_ctas(n) CTAs (cta_pack.cuh): each reads all the entries for the
// width statistics (Eq. 1) and packs its own 16 groups of 32 fields; CTA 0
// writes the whole header.  Up to 65,536 entries the general path's three
// launches (header, tiles, re-code) cost as much or more: 8.0 to 8.5 us per call
// queued back to back from 20,000 entries on (20.6 past 32 bits) against 6.2
// here, 8.3 at 65,536 int64 entries; a call that the host waits for has two
// launches less on top.
constexpr uint64_t kSmallPack = 65536;

template <typename T>
__global__ void __launch_bounds__(kVecThreads) k_pack_small(const T* __restrict__ src,
                                                            uint64_t rows, uint64_t cols,
                                                            ccm_header* out, uint32_t* words,
                                                            uint64_t capacity) {
  __shared__ VecPackSmem sm;
  const uint32_t mm = (uint32_t)(rows * cols);  // 1 .. kSmallPack
  const uint32_t g0 = blockIdx.x * kVecGroupsPerCta;
  uint64_t orv;
  uint32_t neg;
  vec_stats_stage(src, mm, g0, sm, orv, neg);
  const int b = width_from_stats(orv, neg);
  const uint64_t nw = words_for(mm, b), dw = data_words(mm, b);
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    out->magic = CCM_MAGIC;
    out->width = b;
    out->is_signed = neg ? 1 : 0;
    out->status = nw > capacity ? CCM_E_CAPACITY : CCM_OK;
    out->rows = rows;
    out->cols = cols;
    out->nwords = nw;
    out->stat_or = orv;
    out->stat_neg = neg;
    out->reserved0 = 0;
    out->reserved1 = 0;
  }
  if (nw > capacity) return;
  vec_pack_groups(sm, mm, g0, b, words, dw, nw);
}

void run_pack(const void* dense, int dtype, uint64_t rows, uint64_t cols, const ccm_matrix& out,
              void* ws, size_t ws_bytes, cudaStream_t st) {
  uint64_t n = rows * cols;
  if (n && n <= kSmallPack) {
    const uint32_t g = vec_pack_ctas(n);
    profile_begin(st);
    if (dtype == CCM_I64)
      k_pack_small<int64_t><<<g, kVecThreads, 0, st>>>((const int64_t*)dense, rows, cols,
                                                      out.hdr, out.words, out.capacity);
    else
      k_pack_small<int32_t><<<g, kVecThreads, 0, st>>>((const int32_t*)dense, rows, cols,
                                                      out.hdr, out.words, out.capacity);
    profile_end(st);
    note_launch();
    return;
  }
  InitArgs ia{};
  ia.out = out.hdr;
  ia.out_rows = rows;
  ia.out_cols = cols;
  launch_init(ia, st);
  const int cls = ew_class(width_bound(out.capacity, n));
  // (the single pass stages the dense tiles with 16-byte copies: it needs a
  // 16-byte aligned input; an input aligned only to its element size takes
  // the two-pass path below, which reads it element by element)
  const bool aligned16 = reinterpret_cast<uintptr_t>(dense) % 16 == 0;
  if (cls && n && ws && ws_bytes >= ge::pack_ws_bytes(n, cls) && aligned16) {
    // single pass over the dense input: local-width tiles, then re-code
    ge::EwCall c{};
    c.kind = dtype == CCM_I64 ? ge::EwKind::LocalI64 : ge::EwKind::LocalI32;
    c.dense = dense;
    c.out = out.hdr;
    c.words = out.words;
    c.capacity = out.capacity;
    c.rows = rows;
    c.cols = cols;
    c.ws = ws;
    c.slot_class = cls;
    // the widest width the output's capacity holds: the speculative width
    c.spec = width_bound(out.capacity, n);
    if (c.spec > cls) c.spec = 0;
    // (starts while the header is initialised, unless this call is timed)
    c.pdl = profile_armed() ? 0 : 1;
    profile_begin(st);
    launch_ew(cls, c, st);
    profile_end(st);
    c.kind = ge::EwKind::Repack;
    launch_ew(cls, c, st);
    return;
  }
  if (cls && n) {
    if (dtype == CCM_I64)
      launch_stats(ProdDenseI64{(const int64_t*)dense}, out.hdr, n, st);
    else
      launch_stats(ProdDenseI32{(const int32_t*)dense}, out.hdr, n, st);
    ge::EwCall c{};
    c.kind = dtype == CCM_I64 ? ge::EwKind::PackI64 : ge::EwKind::PackI32;
    c.dense = dense;
    c.out = out.hdr;
    c.words = out.words;
    c.capacity = out.capacity;
    c.rows = rows;
    c.cols = cols;
    profile_begin(st);
    launch_ew(cls, c, st);
    profile_end(st);
  } else if (dtype == CCM_I64) {
    ProdDenseI64 p{(const int64_t*)dense};
    if (n) launch_stats(p, out.hdr, n, st);
    profile_begin(st);
    launch_pack(p, out.hdr, out.words, out.capacity, n, st);
    profile_end(st);
  } else {
    ProdDenseI32 p{(const int32_t*)dense};
    if (n) launch_stats(p, out.hdr, n, st);
    profile_begin(st);
    launch_pack(p, out.hdr, out.words, out.capacity, n, st);
    profile_end(st);
  }
}

// ---------------------------------------------------------------------------
// unpack: every field, sign/zero extended, to int64 or int32.
// ---------------------------------------------------------------------------
template <typename T>
__global__ void __launch_bounds__(256) k_unpack(const ccm_header* h, const uint32_t* __restrict__ w,
                                                uint64_t rows, uint64_t cols, uint64_t capacity,
                                                T* __restrict__ out, int32_t* err) {
  int st = check_input(h, rows, cols, capacity);
  const int b = h->width, sgn = h->is_signed;
  if (st == CCM_OK && sizeof(T) == 4 && (sgn ? b > 32 : b > 31)) st = CCM_E_WIDTH;
  if (st != CCM_OK) {
    if (err && blockIdx.x == 0 && threadIdx.x == 0) *err = st;
    return;
  }
  if (err && blockIdx.x == 0 && threadIdx.x == 0) *err = CCM_OK;
  const uint64_t n = rows * cols;
  const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
  for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += stride)
    out[i] = (T)decode_field(w, i, b, sgn);
}

// Fields of at most 32 bits to a dense matrix.  A warp unpacks runs of 512 fields (16 b whole words): lane l takes
// the pairs 2 l + 64 j, so a lane's shift is fixed and its words lie 2 b apart,
// every load is one of 24 issued together, and each warp store writes 64
// consecutive entries (as pairs where the destination is aligned to them).  A
// full run may read up to two words of the next one, which exist (the words
// are padded to four).  Bound by HBM (b/8 bytes in, the entry out).  Measured
// on GB300 (8192^2 at 12 bits to int64; before: a group of 32 fields per lane
// through shared memory, 8 warps per SM): 122 -> 103 us (6.2 TB/s).
constexpr int kUnpackPairs = 8;                      // per lane and run
constexpr int kUnpackRun = 64 * kUnpackPairs;        // fields

template <typename T>
struct Pair;
template <>
struct Pair<int64_t> { using type = longlong2; };
template <>
struct Pair<int32_t> { using type = int2; };

template <typename T>
__global__ void __launch_bounds__(256) k_unpack_pairs(const ccm_header* h,
                                                      const uint32_t* __restrict__ w, uint64_t rows,
                                                      uint64_t cols, uint64_t capacity,
                                                      T* __restrict__ out, int32_t* err) {
  const HeaderView hv = load_header(h);
  int st = check_header(hv, rows, cols, capacity);
  const int b = hv.width, sgn = hv.is_signed;
  if (st == CCM_OK && sizeof(T) == 4 && (sgn ? b > 32 : b > 31)) st = CCM_E_WIDTH;
  if (st == CCM_OK && b > 32) st = CCM_E_INPUT;  // (the capacity bounds b by 32)
  if (err && blockIdx.x == 0 && threadIdx.x == 0) *err = st;
  if (st != CCM_OK) return;
  using V = typename Pair<T>::type;
  const uint64_t n = rows * cols, dw = data_words(n, b);
  const int lane = threadIdx.x % 32, sh = 32 - b;
  const uint32_t bit = 2 * lane * b, at = bit & 31;
  const uint64_t runs = (n + kUnpackRun - 1) / kUnpackRun, warps = (uint64_t)gridDim.x * 8;
  const bool pairs = reinterpret_cast<uintptr_t>(out) % sizeof(V) == 0;
  auto low = [&](uint32_t x) {  // the low b bits as an entry
    const uint32_t t = x << sh;
    return sgn ? (T)((int)t >> sh) : (T)(t >> sh);
  };
  for (uint64_t r = (uint64_t)blockIdx.x * 8 + threadIdx.x / 32; r < runs; r += warps) {
    const uint64_t w0 = r * (uint64_t)(16 * b) + (bit >> 5);
    const uint64_t e0 = r * kUnpackRun + 2 * lane;
    if (r + 1 < runs) {
      const uint32_t* p = w + w0;
      uint32_t x[kUnpackPairs][3];
#pragma unroll
      for (int j = 0; j < kUnpackPairs; ++j, p += 2 * b)
#pragma unroll
        for (int q = 0; q < 3; ++q) x[j][q] = __ldg(p + q);
#pragma unroll
      for (int j = 0; j < kUnpackPairs; ++j) {
        const uint32_t lo = __funnelshift_r(x[j][0], x[j][1], at);
        const uint32_t hi = __funnelshift_r(x[j][1], x[j][2], at);
        V v;
        v.x = low(lo);
        v.y = low(__funnelshift_rc(lo, hi, b));
        if (pairs) {
          __stcs(reinterpret_cast<V*>(out + e0) + 32 * j, v);
        } else {
          out[e0 + 64 * j] = v.x;
          out[e0 + 64 * j + 1] = v.y;
        }
      }
    } else {
      // the last run: no word past the data, no entry past the end
      for (int j = 0; j < kUnpackPairs; ++j) {
        const uint64_t wj = w0 + (uint64_t)(2 * b) * j, e = e0 + 64 * j;
        uint32_t x[3];
#pragma unroll
        for (int q = 0; q < 3; ++q) x[q] = wj + q < dw ? __ldg(w + wj + q) : 0u;
        const uint32_t lo = __funnelshift_r(x[0], x[1], at), hi = __funnelshift_r(x[1], x[2], at);
        if (e < n) out[e] = low(lo);
        if (e + 1 < n) out[e + 1] = low(__funnelshift_rc(lo, hi, b));
      }
    }
  }
}

void run_unpack(const ccm_matrix& a, void* dense, int dtype, int32_t* err, cudaStream_t st) {
  const uint64_t n = a.rows * a.cols;
  profile_begin(st);
  if (n && width_bound(a.capacity, n) <= 32) {
    const uint64_t runs = (n + kUnpackRun - 1) / kUnpackRun;
    const int grid = (int)umin((runs + 7) / 8, (uint64_t)num_sms() * 16);
    if (dtype == CCM_I64)
      k_unpack_pairs<int64_t><<<grid, 256, 0, st>>>(a.hdr, a.words, a.rows, a.cols, a.capacity,
                                                    (int64_t*)dense, err);
    else
      k_unpack_pairs<int32_t><<<grid, 256, 0, st>>>(a.hdr, a.words, a.rows, a.cols, a.capacity,
                                                    (int32_t*)dense, err);
  } else {
    const int grid = (int)umin(umax((n + 255) / 256, 1), (uint64_t)num_sms() * 16);
    if (dtype == CCM_I64)
      k_unpack<int64_t><<<grid, 256, 0, st>>>(a.hdr, a.words, a.rows, a.cols, a.capacity,
                                              (int64_t*)dense, err);
    else
      k_unpack<int32_t><<<grid, 256, 0, st>>>(a.hdr, a.words, a.rows, a.cols, a.capacity,
                                              (int32_t*)dense, err);
  }
  profile_end(st);
  note_launch();
}

// ---------------------------------------------------------------------------
// get: element access by flat row-major index.
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(256) k_get(const ccm_header* h, const uint32_t* __restrict__ w,
                                             uint64_t rows, uint64_t cols, uint64_t capacity,
                                             const uint64_t* __restrict__ idx, uint64_t count,
                                             int64_t* __restrict__ out, int32_t* err) {
  int st = check_input(h, rows, cols, capacity);
  if (err && blockIdx.x == 0 && threadIdx.x == 0 && st != CCM_OK) *err = st;
  if (st != CCM_OK) return;
  const int b = h->width, sgn = h->is_signed;
  const uint64_t n = rows * cols;
  const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
  int bad = 0;
  for (uint64_t k = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; k < count; k += stride) {
    uint64_t e = idx[k];
    if (e < n) {
      out[k] = decode_field(w, e, b, sgn);
    } else {
      out[k] = 0;
      bad = 1;
    }
  }
  if (err && bad) atomicCAS(err, CCM_OK, CCM_E_RANGE);
}

// The same for up to kGetSmall indices by one CTA, which also writes `err`
// (for more, a launch before k_get clears it).
constexpr uint64_t kGetSmall = 4096;
__global__ void __launch_bounds__(1024) k_get_small(const ccm_header* h,
                                                    const uint32_t* __restrict__ w, uint64_t rows,
                                                    uint64_t cols, uint64_t capacity,
                                                    const uint64_t* __restrict__ idx,
                                                    uint32_t count, int64_t* __restrict__ out,
                                                    int32_t* err) {
  const HeaderView hv = load_header(h);
  const int st = check_header(hv, rows, cols, capacity);
  int bad = 0;
  if (st == CCM_OK) {
    const uint64_t n = rows * cols;
    for (uint32_t k = threadIdx.x; k < count; k += 1024) {
      const uint64_t e = idx[k];
      bad |= e >= n;
      out[k] = e < n ? decode_field(w, e, hv.width, hv.is_signed) : 0;
    }
  }
  bad = __syncthreads_or(bad);
  if (err && threadIdx.x == 0) *err = st != CCM_OK ? st : bad ? CCM_E_RANGE : CCM_OK;
}

__global__ void k_set_i32(int32_t* p, int32_t v) { *p = v; }

void run_get(const ccm_matrix& a, const uint64_t* idx, uint64_t count, int64_t* out, int32_t* err,
             cudaStream_t st) {
  if (count && count <= kGetSmall) {
    profile_begin(st);
    k_get_small<<<1, 1024, 0, st>>>(a.hdr, a.words, a.rows, a.cols, a.capacity, idx,
                                    (uint32_t)count, out, err);
    profile_end(st);
    note_launch();
    return;
  }
  if (err) {
    k_set_i32<<<1, 1, 0, st>>>(err, CCM_OK);
    note_launch();
  }
  if (!count) return;
  int grid = (int)umin((count + 255) / 256, (uint64_t)num_sms() * 8);
  profile_begin(st);
  k_get<<<grid, 256, 0, st>>>(a.hdr, a.words, a.rows, a.cols, a.capacity, idx, count, out,
                              err);
  profile_end(st);
  note_launch();
}

// ---------------------------------------------------------------------------
// add / scale
// ---------------------------------------------------------------------------
void run_add(const ccm_matrix& a, const ccm_matrix& b, const ccm_matrix& c, void* /*ws*/,
             size_t /*ws_bytes*/, cudaStream_t st) {
  InitArgs ia{};
  ia.out = c.hdr;
  ia.in0 = a.hdr;
  ia.in1 = b.hdr;
  ia.in0_rows = a.rows;
  ia.in0_cols = a.cols;
  ia.in0_capacity = a.capacity;
  ia.in1_rows = b.rows;
  ia.in1_cols = b.cols;
  ia.in1_capacity = b.capacity;
  ia.out_rows = c.rows;
  ia.out_cols = c.cols;
  launch_init(ia, st);
  uint64_t n = c.rows * c.cols;
  const int cls = ew_class(max(max(width_bound(a.capacity, n), width_bound(b.capacity, n)),
                               width_bound(c.capacity, n)));
  if (cls && n) {
    ge::EwCall e{};
    e.ha = a.hdr;
    e.wa = a.words;
    e.hb = b.hdr;
    e.wb = b.words;
    e.out = c.hdr;
    e.words = c.words;
    e.capacity = c.capacity;
    e.rows = c.rows;
    e.cols = c.cols;
    // one pass at the width the input ranges give, then the finish (a second
    // pass only when the exact width is smaller)
    e.kind = ge::EwKind::AddSpec;
    profile_begin(st);
    launch_ew(cls, e, st);
    e.kind = ge::EwKind::AddPack;
    e.spec = 1;
    launch_ew(cls, e, st);
    profile_end(st);
    return;
  }
  // No width class holds the output bound.  With inputs of at most 32 bits
  // the lane pass may still write the sum (up to 33 bits) first; the
  // run-time passes then return at once.
  ProdAdd p{{a.hdr, a.words, 0, 0}, {b.hdr, b.words, 0, 0}};
  const int in_bound = max(width_bound(a.capacity, n), width_bound(b.capacity, n));
  const int lanes = n && in_bound <= 32;
  profile_begin(st);
  if (lanes) {
    const ge::OpAdd op{ge::PackedIn{a.hdr, a.words, 0, 0, 0}, ge::PackedIn{b.hdr, b.words, 0, 0, 0}};
    ge::launch_lanes_add(op, c.hdr, c.words, c.capacity, n, in_bound, st);
    note_launch();
  }
  if (n) launch_stats(p, c.hdr, n, st, lanes);
  launch_pack(p, c.hdr, c.words, c.capacity, n, st, lanes);
  profile_end(st);
}

void run_scale(const ccm_matrix& a, int64_t s, const ccm_matrix& c, void* /*ws*/,
               size_t /*ws_bytes*/, cudaStream_t st) {
  InitArgs ia{};
  ia.out = c.hdr;
  ia.in0 = a.hdr;
  ia.in0_rows = a.rows;
  ia.in0_cols = a.cols;
  ia.in0_capacity = a.capacity;
  ia.out_rows = c.rows;
  ia.out_cols = c.cols;
  launch_init(ia, st);
  uint64_t n = c.rows * c.cols;
  const int cls = ew_class(max(width_bound(a.capacity, n), width_bound(c.capacity, n)));
  if (cls && n) {
    ge::EwCall e{};
    e.ha = a.hdr;
    e.wa = a.words;
    e.s = s;
    e.out = c.hdr;
    e.words = c.words;
    e.capacity = c.capacity;
    e.rows = c.rows;
    e.cols = c.cols;
    e.kind = ge::EwKind::ScaleSpec;
    profile_begin(st);
    launch_ew(cls, e, st);
    e.kind = ge::EwKind::ScalePack;
    e.spec = 1;
    launch_ew(cls, e, st);
    profile_end(st);
    return;
  }
  // No width class holds the output bound: the lane pass may still write
  // s A (up to 36 bits) first for 1 <= |s| < 2^5; the run-time passes then
  // return at once.
  ProdScale p{{a.hdr, a.words, 0, 0}, s};
  const int in_bound = width_bound(a.capacity, n);
  const int lanes = n && in_bound <= 32 && s != 0 && s > -32 && s < 32;
  profile_begin(st);
  if (lanes) {
    const ge::OpScale<true> op{ge::PackedIn{a.hdr, a.words, 0, 0, 0}, s};
    ge::launch_lanes_scale(op, c.hdr, c.words, c.capacity, n, in_bound, st);
    note_launch();
  }
  if (n) launch_stats(p, c.hdr, n, st, lanes);
  launch_pack(p, c.hdr, c.words, c.capacity, n, st, lanes);
  profile_end(st);
}

void run_pack_scratch32(const int32_t* vals, const ccm_matrix& out, cudaStream_t st) {
  const uint64_t n = out.rows * out.cols;
  const int cls = ew_class(width_bound(out.capacity, n));
  if (cls && n && reinterpret_cast<uintptr_t>(vals) % 16 == 0) {
    // the producer merged the statistics: one pass at the exact width (the
    // staged single-pass kernel, spec < 0: minus the widest width), then the header
    ge::EwCall c{};
    c.kind = ge::EwKind::LocalI32;
    c.dense = vals;
    c.out = out.hdr;
    c.words = out.words;
    c.capacity = out.capacity;
    c.rows = out.rows;
    c.cols = out.cols;
    c.slot_class = cls;
    c.spec = -width_bound(out.capacity, n);
    launch_ew(cls, c, st);
    c.kind = ge::EwKind::Repack;
    launch_ew(cls, c, st);
    return;
  }
  launch_pack(ProdDenseI32{vals}, out.hdr, out.words, out.capacity, n, st);
}

// Width, header and words of a vector of int64 values (y of a matvec) in one
// launch of vec_pack_ctas(n) CTAs: each reads all the values for the
// statistics (from L2) and packs its own 16 groups of 32 fields (cta_pack.cuh);
// CTA 0 writes the header.
__global__ void __launch_bounds__(kVecThreads) k_pack_vec(ccm_header* out, uint32_t* words,
                                                          uint64_t capacity,
                                                          const int64_t* __restrict__ y,
                                                          uint64_t m) {
  __shared__ VecPackSmem sm;
  ax::grid_dep_wait();  // every sum is in place
  if (out->status != CCM_OK) return;
  const uint32_t mm = (uint32_t)m;  // <= kVecMax
  const uint32_t g0 = blockIdx.x * kVecGroupsPerCta;
  uint64_t orv;
  uint32_t neg;
  vec_stats_stage(y, mm, g0, sm, orv, neg);
  const int b = width_from_stats(orv, neg);
  const uint64_t nw = words_for(m, b), dw = data_words(m, b);
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    out->stat_or = orv;
    out->stat_neg = neg;
    out->width = b;
    out->is_signed = neg ? 1 : 0;
    out->nwords = nw;
    out->magic = CCM_MAGIC;
    if (nw > capacity) out->status = CCM_E_CAPACITY;
  }
  if (nw > capacity) return;
  vec_pack_groups(sm, mm, g0, b, words, dw, nw);
}

// Longest vector of the one-launch pack: every CTA reads all of it (512 KB at
// this length), which up to here beats a statistics pass and a pack pass
// (whole products of 64 columns, 65,536 rows 16.7 us, 66,000 rows 22.6).
constexpr uint64_t kVecMax = 65536;

// Pack an int64 result held in device scratch (matvec / matmul epilogue).
// `pdl`: may start while the kernel that writes `vals` still runs (it waits
// for it).
void run_pack_scratch(const int64_t* vals, const ccm_matrix& out, cudaStream_t st,
                      bool stats_done, bool pdl) {
  ProdDenseI64 p{vals};
  uint64_t n = out.rows * out.cols;
  if (n && n <= kVecMax && !stats_done) {
    const uint32_t g = vec_pack_ctas(n);
    if (pdl)
      ax::launch_pdl(k_pack_vec, dim3(g), dim3(kVecThreads), 0, st, out.hdr, out.words,
                     out.capacity, vals, n);
    else
      k_pack_vec<<<g, kVecThreads, 0, st>>>(out.hdr, out.words, out.capacity, vals, n);
    note_launch();
    return;
  }
  const int cls = ew_class(width_bound(out.capacity, n));
  if (cls && n) {
    if (!stats_done) launch_stats(p, out.hdr, n, st);
    ge::EwCall c{};
    c.kind = ge::EwKind::PackI64;
    c.dense = vals;
    c.out = out.hdr;
    c.words = out.words;
    c.capacity = out.capacity;
    c.rows = out.rows;
    c.cols = out.cols;
    launch_ew(cls, c, st);
    return;
  }
  if (n && !stats_done) launch_stats(p, out.hdr, n, st);
  launch_pack(p, out.hdr, out.words, out.capacity, n, st);
}

}  // namespace ccm
