// matmul_tc.cu -- exact integer C = A B on the tcgen05 tensor cores.
//
// GB300 (sm_103a) has no integer tensor-core MMA (tcgen05.mma .kind::i8 is
// rejected by ptxas for this target), so the product runs on fp16 operands
// whose values are integers, accumulated in fp32:
//
//   a = sum_l d_l 2^(w l),   l = 0 .. d-1,   |d_l| <= 2^(w-1)   (balanced digits)
//   C = sum_{l, m} 2^(w_a l + w_b m) (A_l B_m)
//
// With e the width of a field as a two's complement number (b for signed
// matrices, b + 1 for unsigned ones), d digits need w = ceil(e / d) bits.
// fp16 holds every integer up to 2^11, so a digit may have up to 12 bits and
// fields of up to 12 bits are one digit.  Products of magnitudes 2^p and 2^q
// are integers; a sum of 2^(24 - p - q) of them is at most 2^24, so every
// partial sum of such a run of k is an integer that fp32 holds exactly in
// whatever order it is formed.  The product of every digit pair is therefore
// accumulated in tensor memory over runs of k of at most that length (at
// least kMinRun), and the epilogue warps add each run to integer accumulators
// in registers while the next run is being multiplied.
//
// Why fp16 and not e4m3: fp8 runs at twice the rate but holds 4 significant
// bits, so an 8 x 8-bit product takes 4 fp8 MMAs (2 units of fp16 time) where
// one fp16 MMA does, a 12 x 12-bit one 9 (4.5 units) instead of 2, a
// 16 x 16-bit one 16 (8 units) instead of 4.
//
// Measured on GB300 (whole call; before: e4m3 digits in one-CTA tiles, or the
// CUDA cores above 16 bits): 4096^3 at 4 / 8 / 12 / 16 signed bits 0.21 / 0.39 /
// 0.92 / 1.31 -> 0.14 / 0.14 / 0.36 / 0.51 ms; 3001 x 2503 x 3500 at 20 x 18
// bits 8.30 -> 0.33 ms.  What bounds it, by the times over tile widths: the L2,
// which feeds the stages about 46 bytes per clock and SM.
//
// Kernels:
//   k_planes  packed A and B -> fp16 digit planes, K-major (B transposed)
//   k_mm      persistent pairs of CTAs (one tcgen05 cta_group::2 tile of
//             256 x BN outputs per pair): warp 0 TMA producer, warp 1 MMA
//             issuer (leader CTA), warps 4-11 epilogue
//
// Every wait on an mbarrier is bounded; a wait that gives up records
// CCM_E_TIMEOUT in C's header and the CTAs free their tensor memory and exit.
#include <cuda.h>
#include <cuda_fp16.h>
#include <cudaTypedefs.h>

#include <type_traits>

#include "async_copy.cuh"
#include "ccm_device.cuh"
#include "host_cache.h"
#include "kernels.h"
#include "matmul_tc.h"
#include "matmul_tile.h"

namespace ccm {
namespace tc {

using ax::mbar_init;
using ax::smem_u32;

constexpr int kBK = 64;           // fp16 elements of a block of k (a 128-byte swizzled row)
constexpr uint32_t kGroupM = 4;   // tile rows per raster group
constexpr int kMaxDigits = 3;
constexpr int kMaxMag = 11;       // fp16 integers are exact up to 2^11
constexpr int kMinRun = 256;      // shortest run of k between two flushes

// Digit counts and widths of one product.
struct Split {
  uint8_t da, wa, db, wb;
  // k elements whose products stay exact in fp32 (a multiple of kBK)
  __host__ __device__ int run() const { return 1 << (26 - wa - wb); }
};

// The cheapest split for operands of e_a and e_b bits (two's complement),
// 1 .. kMaxE each: fewest digit pairs, then the longest run.  da = 0: none
// fits.  A table, because every CTA asks for it once it knows the widths.
constexpr int kMaxE = 32;
struct SplitTable {
  Split at[kMaxE + 1][kMaxE + 1];
};
constexpr SplitTable make_splits() {
  SplitTable t{};
  for (int ea = 1; ea <= kMaxE; ++ea)
    for (int eb = 1; eb <= kMaxE; ++eb) {
      int best = 1 << 30;
      for (int da = 1; da <= kMaxDigits; ++da)
        for (int db = 1; db <= kMaxDigits; ++db) {
          const int wa = (ea + da - 1) / da, wb = (eb + db - 1) / db;
          const int mags = wa + wb - 2;
          if (wa - 1 > kMaxMag || wb - 1 > kMaxMag || mags > 16 ||
              (kMinRun << mags) > (1 << 24))
            continue;
          const int score = da * db * 64 + mags;
          if (score < best) {
            best = score;
            t.at[ea][eb].da = (uint8_t)da;
            t.at[ea][eb].wa = (uint8_t)wa;
            t.at[ea][eb].db = (uint8_t)db;
            t.at[ea][eb].wb = (uint8_t)wb;
          }
        }
    }
  return t;
}
constexpr SplitTable kSplits = make_splits();
__constant__ SplitTable c_splits = make_splits();

// The split of the two headers' widths (the host has bounded both by 31).
__device__ __forceinline__ Split split_of(const ccm_header* ha, const ccm_header* hb) {
  const int ea = ha->width + !ha->is_signed, eb = hb->width + !hb->is_signed;
  if (ea > kMaxE || eb > kMaxE) return Split{0, 0, 0, 0};
  return c_splits.at[ea][eb];
}

__host__ __device__ inline uint64_t round_up(uint64_t v, uint64_t m) { return (v + m - 1) / m * m; }

// ---------------------------------------------------------------------------
// Digit planes
// ---------------------------------------------------------------------------
// Eight consecutive fields of B bits of a packed stream from field e0 on
// (`cnt` of them; the others read as zero): all their words loaded at once (no
// word past the last field), moved to a common start, and cut with shifts
// fixed at compile time.
template <int B>
__device__ __forceinline__ void decode8(const uint32_t* __restrict__ words, uint64_t e0, int cnt,
                                        int sgn, int (&v)[8]) {
  constexpr int kX = (8 * B + 31) / 32;  // aligned words
  const uint64_t p = e0 * (uint64_t)B;
  const uint32_t* q = words + (p >> 5);
  const uint32_t s = (uint32_t)p & 31;
  const int need = (int)(s + max(cnt, 0) * B + 31) >> 5;
  uint32_t w[kX + 1], x[kX];
#pragma unroll
  for (int j = 0; j <= kX; ++j) w[j] = j < need && cnt > 0 ? __ldg(q + j) : 0u;
#pragma unroll
  for (int j = 0; j < kX; ++j) x[j] = __funnelshift_r(w[j], w[j + 1], s);
#pragma unroll
  for (int j = 0; j < 8; ++j) {
    const int bit = j * B, wi = bit >> 5, sh = bit & 31;
    uint32_t t;  // the field at the top of the word
    if (sh + B <= 32)
      t = x[wi] << (32 - B - sh);
    else
      t = __funnelshift_r(x[wi], x[wi + 1 < kX ? wi + 1 : wi], sh) << (32 - B);
    v[j] = sgn ? (int)t >> (32 - B) : (int)(t >> (32 - B));
  }
  if (cnt < 8) {
#pragma unroll
    for (int j = 0; j < 8; ++j)
      if (j >= cnt) v[j] = 0;
  }
}

// Splits off the low balanced digit of w bits: v becomes the rest.
__device__ __forceinline__ int take_digit(int& v, int w) {
  const int d = (int)((uint32_t)v << (32 - w)) >> (32 - w);
  v = (v >> w) + ((v >> (w - 1)) & 1);
  return d;
}

// Two integers as halves.  Magnitudes of at most 256 (`small`): 0x6600 is
// 1536 = 1.5 * 2^10, whose ulp is 1, so adding the integer to its bits adds it
// to its value, and the subtraction is exact (the conversion instruction runs
// at a fraction of that rate).
__device__ __forceinline__ uint32_t half2_bits(int x, int y, bool small) {
  __half2 h;
  if (small) {
    const uint32_t u = (uint32_t)x + ((uint32_t)y << 16) + 0x66006600u, base = 0x66006600u;
    h = __hsub2(*reinterpret_cast<const __half2*>(&u), *reinterpret_cast<const __half2*>(&base));
  } else {
    h = __halves2half2(__int2half_rn(x), __int2half_rn(y));
  }
  return *reinterpret_cast<const uint32_t*>(&h);
}

struct PlaneArgs {
  const ccm_header *out, *ha, *hb;
  const uint32_t *wa, *wb;
  uint64_t row0, col0;   // the strips begin at A's row row0 and B's column col0
  uint64_t m, k, n, kp;  // rows of A's strip, columns of B's; kp: k rounded up to 64 (a row of a plane)
  uint64_t ldb;          // columns of B
  __half *pa, *pb;       // [da][m][kp], [db][n][kp]
  uint32_t row_runs;     // A: warp-runs (32 groups of 8 fields) per row
  uint32_t blocks_a;     // CTAs [0, blocks_a) write A's planes, the rest B's
  uint32_t tiles_k;      // B: 64 x 64 tiles along k
};

// A's planes: 8 fields of a row per lane, one 16-byte store per digit.
template <int B>
__device__ __forceinline__ void planes_a(const PlaneArgs& a, const Split& sp) {
  const int sgn = a.ha->is_signed, lane = threadIdx.x % 32;
  const bool small = sp.wa <= 9;
  const uint64_t items = a.m * a.row_runs;
  for (uint64_t it = (uint64_t)blockIdx.x * 8 + threadIdx.x / 32; it < items;
       it += (uint64_t)a.blocks_a * 8) {
    const uint64_t i = items >> 32 ? it / a.row_runs : (uint32_t)it / a.row_runs;
    const uint64_t kk = 8 * ((it - i * a.row_runs) * 32 + lane);
    if (kk >= a.kp) continue;
    int v[8];
    decode8<B>(a.wa, (a.row0 + i) * a.k + kk, kk < a.k ? (int)umin(8, a.k - kk) : 0, sgn, v);
    __half* dst = a.pa + i * a.kp + kk;
    for (int l = 0; l < sp.da; ++l, dst += a.m * a.kp) {
      int d[8];
#pragma unroll
      for (int j = 0; j < 8; ++j) d[j] = l + 1 < sp.da ? take_digit(v[j], sp.wa) : v[j];
      *reinterpret_cast<uint4*>(dst) =
          make_uint4(half2_bits(d[0], d[1], small), half2_bits(d[2], d[3], small),
                     half2_bits(d[4], d[5], small), half2_bits(d[6], d[7], small));
    }
  }
}

// B's planes: a 64 (k) x 64 (n) tile per CTA; a thread decodes 8 fields of two
// rows of B and writes them as (k, k + 1) pairs into a transposed shared tile,
// whose rows (64 k of one column) leave as 16-byte stores.
template <int B>
__device__ __forceinline__ void planes_b(const PlaneArgs& a, const Split& sp,
                                         uint32_t (*tile)[33]) {
  const int sgn = a.hb->is_signed, tid = threadIdx.x;
  const bool small = sp.wb <= 9;
  const uint32_t t = blockIdx.x - a.blocks_a;
  const uint64_t k0 = (uint64_t)(t % a.tiles_k) * 64, j0 = (uint64_t)(t / a.tiles_k) * 64;
  const int cols = (int)umin(64, a.n - j0);
  const int g8 = 8 * (tid % 8), kpair = tid / 8, cnt = min(8, cols - g8);
  const uint64_t row = k0 + 2 * kpair;
  int v0[8], v1[8];
  const uint64_t e0 = row * a.ldb + a.col0 + j0 + g8;
  decode8<B>(a.wb, e0, row < a.k ? cnt : 0, sgn, v0);
  decode8<B>(a.wb, e0 + a.ldb, row + 1 < a.k ? cnt : 0, sgn, v1);
  const int col = tid / 4, q = tid % 4;
  __half* dst = a.pb + (j0 + col) * a.kp + k0 + 16 * q;
  for (int l = 0; l < sp.db; ++l, dst += a.n * a.kp) {
    const bool last = l + 1 == sp.db;
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      const int x = last ? v0[j] : take_digit(v0[j], sp.wb);
      const int y = last ? v1[j] : take_digit(v1[j], sp.wb);
      tile[g8 + j][kpair] = half2_bits(x, y, small);
    }
    __syncthreads();
    if (col < cols) {
      const uint32_t* src = &tile[col][8 * q];
      reinterpret_cast<uint4*>(dst)[0] = make_uint4(src[0], src[1], src[2], src[3]);
      reinterpret_cast<uint4*>(dst)[1] = make_uint4(src[4], src[5], src[6], src[7]);
    }
    __syncthreads();
  }
}

#define CCM_TC_WIDTHS(M)                                                                       \
  M(1) M(2) M(3) M(4) M(5) M(6) M(7) M(8) M(9) M(10) M(11) M(12) M(13) M(14) M(15) M(16) M(17) \
  M(18) M(19) M(20) M(21) M(22) M(23) M(24) M(25) M(26) M(27) M(28) M(29) M(30) M(31)

// The planes of a strip of A and of one of B (or of one of the two) in one launch.  The bytes are b/8 in and 2 d out per
// field; what is left beside them is the cutting of the fields, so the widths
// are compile-time bodies chosen from the headers.
__global__ void __launch_bounds__(256) k_planes(const __grid_constant__ PlaneArgs a) {
  __shared__ uint32_t tile[64][33];
  ax::grid_dep_launch();
  ax::grid_dep_wait();
  if (a.out->status != CCM_OK) return;
  const Split sp = split_of(a.ha, a.hb);
  if (blockIdx.x < a.blocks_a) {
    switch (a.ha->width) {
#define CCM_TC_A(B) \
  case B: planes_a<B>(a, sp); break;
      CCM_TC_WIDTHS(CCM_TC_A)
#undef CCM_TC_A
      default: break;
    }
  } else {
    switch (a.hb->width) {
#define CCM_TC_B(B) \
  case B: planes_b<B>(a, sp, tile); break;
      CCM_TC_WIDTHS(CCM_TC_B)
#undef CCM_TC_B
      default: break;
    }
  }
}

// ---------------------------------------------------------------------------
// PTX wrappers (tcgen05 with CTA pairs, TMA, cluster mbarriers)
// ---------------------------------------------------------------------------
__device__ __forceinline__ uint32_t cluster_rank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %cluster_ctarank;\n" : "=r"(r));
  return r;
}

// One lane of the (converged) warp.
__device__ __forceinline__ bool elect_one() {
  uint32_t p;
  asm volatile("{\n.reg .pred p;\nelect.sync _|p, 0xffffffff;\nselp.u32 %0, 1, 0, p;\n}\n"
               : "=r"(p));
  return p != 0;
}

__device__ __forceinline__ void cluster_sync() {
  asm volatile("barrier.cluster.arrive.release.aligned;\nbarrier.cluster.wait.acquire.aligned;\n" ::
                   : "memory");
}

// The shared::cluster address of `p` in CTA `rank` of the cluster.
__device__ __forceinline__ uint32_t map_rank(const void* p, uint32_t rank) {
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;\n" : "=r"(r) : "r"(smem_u32(p)), "r"(rank));
  return r;
}

// (At its default scope: what it orders are tensor-memory reads, fenced before
// it; a release at cluster scope is a memory barrier, which made a flush of an
// accumulator take some 4000 cycles: 4096^3 at 12 bits 431 us, now 255.)
__device__ __forceinline__ void arrive_remote(uint32_t cluster_addr) {
  asm volatile("mbarrier.arrive.shared::cluster.b64 _, [%0];\n" ::"r"(cluster_addr) : "memory");
}

__device__ __forceinline__ uint32_t ld_remote(uint32_t cluster_addr) {
  uint32_t v;
  asm volatile("ld.shared::cluster.u32 %0, [%1];\n" : "=r"(v) : "r"(cluster_addr) : "memory");
  return v;
}

// kSub blocks of k from block x on, rows from y on, of plane z; the bytes are
// counted on the leader's barrier.
__device__ __forceinline__ void tma_load_pair(uint32_t dst, const CUtensorMap* map, uint32_t bar,
                                              int x, int y, int z) {
  asm volatile(
      "cp.async.bulk.tensor.4d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes"
      " [%0], [%1, {%3, %4, %5, %6}], [%2];\n" ::"r"(dst),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(bar), "r"(0), "r"(y), "r"(x), "r"(z)
      : "memory");
}

// Shared-memory matrix descriptor: K-major operand, rows of 128 bytes in the
// 128-byte swizzle pattern, 8-row groups 1024 bytes apart.
__device__ __forceinline__ uint64_t smem_desc_sw128(uint32_t saddr) {
  uint64_t d = 0;
  d |= (uint64_t)((saddr >> 4) & 0x3FFFu);  // start address
  d |= (uint64_t)1 << 16;                    // leading byte offset (unused for this layout)
  d |= (uint64_t)(1024 >> 4) << 32;          // stride byte offset: 8 rows x 128 B
  d |= (uint64_t)1 << 46;                    // descriptor version (sm_100 family)
  d |= (uint64_t)2 << 61;                    // swizzle: 128 bytes
  return d;
}

// Instruction descriptor: kind::f16, A = B = f16, D = f32, both K-major.
__host__ __device__ constexpr uint32_t idesc_f16_f32(int m, int n) {
  return (1u << 4) | ((uint32_t)(n >> 3) << 17) | ((uint32_t)(m >> 4) << 24);
}

__device__ __forceinline__ void mma_f16_pair(uint32_t tmem_d, uint64_t adesc, uint64_t bdesc,
                                             uint32_t idesc, uint32_t accumulate) {
  asm volatile(
      "{\n.reg .pred p;\nsetp.ne.b32 p, %4, 0;\n"
      "tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(tmem_d),
      "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate));
}

// Arrives on `bar` (same offset) in both CTAs of the pair when the MMAs
// issued so far have completed.
__device__ __forceinline__ void mma_commit_pair(uint64_t* bar) {
  asm volatile(
      "tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64"
      " [%0], %1;\n" ::"r"(smem_u32(bar)),
      "h"((uint16_t)3)
      : "memory");
}

__device__ __forceinline__ void tmem_ld16(uint32_t taddr, uint32_t (&r)[16]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 "
      "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];\n"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
        "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]),
        "=r"(r[14]), "=r"(r[15])
      : "r"(taddr));
}
__device__ __forceinline__ void tmem_ld_wait() {
  asm volatile("tcgen05.wait::ld.sync.aligned;\n" ::: "memory");
}
__device__ __forceinline__ void tmem_fence_before() {
  asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
}
__device__ __forceinline__ void tmem_fence_after() {
  asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
}

// ---------------------------------------------------------------------------
// The product kernel
// ---------------------------------------------------------------------------
struct MmArgs {
  ccm_header* out;  // C header: status, width statistics
  const ccm_header *ha, *hb;
  void* c;          // the strip of C: m x n, rows ldc apart, int64 or int32
  uint64_t m, n, ldc;
  uint32_t k_blocks;
  uint32_t tiles_m, tiles_n;
  int c32;          // 1: C is stored as int32 (the output capacity bounds its width by 31)
};

constexpr int kEpiWarps = 8;
constexpr int kThreads = 32 * (4 + kEpiWarps);  // (two warps idle: registers are granted per four warps)

// Geometry of one instance.  Acc64: C needs more than 32 bits, so a thread
// holds 64-bit accumulators and the tile is at most 128 columns wide.
template <int BN, bool kAcc64>
struct Geo {
  static constexpr int kHalf = BN / 2;                 // columns per epilogue half
  static constexpr int kCCols = !kAcc64 && kHalf % 32 == 0 ? 32 : 16;  // columns stored at a time
  // blocks of k per stage: a stage costs about 380 cycles of barrier round
  // trips in the producer and the issuer, a block BN * 2 cycles of MMA
  static constexpr int kSub = BN > 128 ? 1 : 2;
  static constexpr uint32_t kATile = 128 * kBK * 2;    // bytes per CTA and block of k
  static constexpr uint32_t kBTile = (BN / 2) * kBK * 2;
  static constexpr uint32_t kBOff = kSub * kATile;     // B's blocks behind A's
  static constexpr uint32_t kStage = kSub * (kATile + kBTile);
  static constexpr uint32_t kCStage = 32 * (kCCols + 1) * (kAcc64 ? 8 : 4);  // per epilogue warp
  static constexpr int kBufs = BN > 128 ? 2 : 4;       // accumulators in tensor memory
  static constexpr uint32_t kBufCols = 512 / kBufs;
  static constexpr int kStages = (int)((224 * 1024 - kEpiWarps * kCStage) / kStage) > 8
                                     ? 8
                                     : (int)((224 * 1024 - kEpiWarps * kCStage) / kStage);
  static constexpr size_t kSmem = 1024 + (size_t)kStages * kStage + kEpiWarps * kCStage;
};

// Output tile t (grouped raster): consecutive tiles sweep the tile columns
// of a group of kGroupM tile rows before the next group.
__device__ __forceinline__ void tile_coords(uint32_t t, uint32_t tiles_m, uint32_t tiles_n,
                                            uint32_t& tm, uint32_t& tn) {
  const uint32_t per_group = kGroupM * tiles_n, group = t / per_group;
  const uint32_t first_m = group * kGroupM;
  const uint32_t gm = tiles_m - first_m < kGroupM ? tiles_m - first_m : kGroupM;
  const uint32_t in_group = t - group * per_group;
  tm = first_m + in_group % gm;
  tn = in_group / gm;
}

// acc += run << shift for 16 columns: the run's sums are integers of at most
// 2^24, so the conversion is exact.
__device__ __forceinline__ void add_run(const uint32_t (&r)[16], int shift, uint32_t* acc) {
#pragma unroll
  for (int j = 0; j < 16; ++j) acc[j] += (uint32_t)__float2int_rn(__uint_as_float(r[j])) << shift;
}
__device__ __forceinline__ void add_run(const uint32_t (&r)[16], int shift,
                                        unsigned long long* acc) {
  if (shift <= 30) {  // one 32 x 32 -> 64-bit multiply-add per column
    const int mul = 1 << shift;
#pragma unroll
    for (int j = 0; j < 16; ++j)
      acc[j] += (unsigned long long)((long long)__float2int_rn(__uint_as_float(r[j])) * mul);
  } else {
#pragma unroll
    for (int j = 0; j < 16; ++j)
      acc[j] += (unsigned long long)((long long)__float2int_rn(__uint_as_float(r[j]))) << shift;
  }
}

// One warp's 32 rows x kHalf columns of C, from one row per lane to rows of
// consecutive lanes: through a transposing tile, kCCols columns at a time.
template <int BN, bool kAcc64, typename T, typename UAcc, typename Acc>
__device__ __forceinline__ void store_tile(const UAcc (&acc)[BN / 2], Acc* st, int lane, T* c,
                                           uint64_t row0, uint64_t col0, uint64_t m, uint64_t n,
                                           uint64_t ldc) {
  constexpr int W = Geo<BN, kAcc64>::kCCols, kRows = 32 / W;
  const int r0 = lane / W, cl = lane % W;
  const int rows = row0 < m ? (int)umin(32, m - row0) : 0;
#pragma unroll
  for (int c0 = 0; c0 < BN / 2; c0 += W) {
#pragma unroll
    for (int j = 0; j < W; ++j) st[lane * (W + 1) + j] = (Acc)acc[c0 + j];
    __syncwarp();
    const uint64_t col = col0 + c0 + cl;
    if (col < n) {
      T* dst = c + (row0 + r0) * ldc + col;
      const Acc* src = st + r0 * (W + 1) + cl;
#pragma unroll 8
      for (int r = 0; r < 32; r += kRows) {
        if (r + r0 < rows) *dst = (T)src[r * (W + 1)];
        dst += kRows * ldc;
      }
    }
    __syncwarp();
  }
}

template <int BN, bool kAcc64>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(kThreads, 1)
    k_mm(const __grid_constant__ CUtensorMap map_a, const __grid_constant__ CUtensorMap map_b,
         const __grid_constant__ MmArgs args) {
  using G = Geo<BN, kAcc64>;
  using Acc = typename std::conditional<kAcc64, long long, int>::type;
  using UAcc = typename std::make_unsigned<Acc>::type;  // (sums wrap: only the total must fit)
  constexpr int S = G::kStages;
  extern __shared__ __align__(1024) uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) &
                                             ~(uintptr_t)1023);
  __shared__ uint64_t full_bar[S], empty_bar[S], acc_full[G::kBufs], acc_empty[G::kBufs];
  __shared__ uint32_t tmem_base_s;
  __shared__ __align__(4) Split split_s;
  __shared__ volatile int abort_s;
  __shared__ uint32_t issued_s;  // stages whose loads this CTA issued

  const int warp = __shfl_sync(0xffffffffu, threadIdx.x / 32, 0), lane = threadIdx.x % 32;
  const uint32_t rank = cluster_rank();
  if (threadIdx.x == 0) {
    for (int s = 0; s < S; ++s) {
      mbar_init(&full_bar[s], 1);
      mbar_init(&empty_bar[s], 1);
    }
    for (int a = 0; a < G::kBufs; ++a) {
      mbar_init(&acc_full[a], 1);
      mbar_init(&acc_empty[a], 2 * kEpiWarps);  // the epilogue warps of both CTAs
    }
    abort_s = 0;
    issued_s = 0;
    ax::mbar_init_fence();
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;\n" ::"r"(
                     smem_u32(&tmem_base_s)),
                 "r"(512u));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;\n");
  }
  ax::grid_dep_launch();
  ax::grid_dep_wait();
  // the leader's reading of the status and the widths decides for the pair
  // (another CTA may set the status meanwhile)
  if (rank == 0 && threadIdx.x == 0) {
    split_s = split_of(args.ha, args.hb);
    if (args.out->status != CCM_OK) split_s.da = 0;
  }
  tmem_fence_before();
  cluster_sync();
  tmem_fence_after();
  const uint32_t tmem = tmem_base_s;
  const uint32_t sw = ld_remote(map_rank(&split_s, 0));
  const Split sp{(uint8_t)sw, (uint8_t)(sw >> 8), (uint8_t)(sw >> 16), (uint8_t)(sw >> 24)};
  const uint32_t tiles = sp.da ? args.tiles_m * args.tiles_n : 0;
  const uint32_t nk = (args.k_blocks + G::kSub - 1) / G::kSub;  // stages along k
  const uint32_t pairs = sp.da * sp.db;
  const uint32_t run = min((uint32_t)(sp.run() / (kBK * G::kSub)), nk);  // stages per flush
  const uint32_t first = blockIdx.x / 2, step = gridDim.x / 2;

  // Producer and issuer run as whole warps, one elected lane issuing, so that
  // addresses and descriptors stay in uniform registers, and nothing but the
  // stage's barrier is touched per k block: every further access to shared
  // memory costs a hundred cycles or so of a loop that has 512 (at BN = 256).
  // Issued from a single-lane branch with an abort flag read per k block, a
  // k block took 730-780 cycles whatever BN was.
  if (warp == 0) {
    const uint32_t full0 = __shfl_sync(0xffffffffu, map_rank(&full_bar[0], 0), 0);
    const uint32_t smem0 = __shfl_sync(0xffffffffu, smem_u32(smem), 0);
    uint32_t s = 0, parity = 1, issued = 0;
    bool ok = true;
    for (uint32_t t = first; t < tiles && ok; t += step) {
      uint32_t tm, tn;
      tile_coords(t, args.tiles_m, args.tiles_n, tm, tn);
      const int ya = tm * kBM + rank * 128, yb = tn * BN + rank * (BN / 2);
      for (uint32_t p = 0; p < pairs && ok; ++p) {
        const int l = p / sp.db, q = p % sp.db;
        if (abort_s) ok = false;
        for (uint32_t kb = 0; kb < nk && ok; ++kb) {
          if (!__all_sync(0xffffffffu, ax::mbar_wait_suspended(&empty_bar[s], parity))) {
            ok = false;
            break;
          }
          if (elect_one()) {
            if (rank == 0) ax::mbar_expect_tx(&full_bar[s], 2 * G::kStage);
            tma_load_pair(smem0 + s * G::kStage, &map_a, full0 + 8 * s, G::kSub * kb, ya, l);
            tma_load_pair(smem0 + s * G::kStage + G::kBOff, &map_b, full0 + 8 * s, G::kSub * kb, yb, q);
          }
          __syncwarp();
          ++issued;
          if (++s == (uint32_t)S) {
            s = 0;
            parity ^= 1;
          }
        }
      }
    }
    if (lane == 0) issued_s = issued;
    // the leader's commits still on their way to this CTA's barriers
    for (uint32_t x = issued > (uint32_t)S ? issued - S : 0; x < issued && ok; ++x)
      ok = __all_sync(0xffffffffu, ax::mbar_wait_suspended(&empty_bar[x % S], (x / S) & 1));
    if (!ok) abort_s = 1;
  } else if (warp == 1) {
    if (rank == 0) {
      constexpr uint32_t idesc = idesc_f16_f32(kBM, BN);
      const uint32_t smem0 = __shfl_sync(0xffffffffu, smem_u32(smem), 0);
      const uint32_t tmem0 = __shfl_sync(0xffffffffu, tmem, 0);
      uint32_t s = 0, parity = 0, f = 0;  // stage and its phase; runs
      bool ok = true;
      for (uint32_t t = first; t < tiles && ok; t += step) {
        for (uint32_t p = 0; p < pairs && ok; ++p) {
          for (uint32_t k0 = 0; k0 < nk && ok; k0 += run, ++f) {
            const uint32_t buf = f % G::kBufs;
            if (abort_s || !__all_sync(0xffffffffu,
                                       ax::mbar_wait_suspended(&acc_empty[buf], ((f / G::kBufs) & 1) ^ 1))) {
              ok = false;
              break;
            }
            tmem_fence_after();
            const uint32_t acc = tmem0 + buf * G::kBufCols;
            const uint32_t k1 = k0 + run < nk ? k0 + run : nk;
            for (uint32_t kb = k0; kb < k1; ++kb) {
              if (!__all_sync(0xffffffffu, ax::mbar_wait_suspended(&full_bar[s], parity))) {
                ok = false;
                break;
              }
              tmem_fence_after();
              const uint64_t da = smem_desc_sw128(smem0 + s * G::kStage);
              const uint64_t db = smem_desc_sw128(smem0 + s * G::kStage + G::kBOff);
              if (elect_one()) {
#pragma unroll
                for (int kk = 0; kk < 4 * G::kSub; ++kk) {
                  // 32 bytes further along k; the second block is a tile on
                  const uint32_t in = 2 * (kk % 4), blk = kk / 4;
                  mma_f16_pair(acc, da + in + blk * (G::kATile / 16), db + in + blk * (G::kBTile / 16),
                               idesc, (kb > k0 || kk > 0) ? 1u : 0u);
                }
                mma_commit_pair(&empty_bar[s]);  // frees the stage in both CTAs
              }
              __syncwarp();
              if (++s == (uint32_t)S) {
                s = 0;
                parity ^= 1;
              }
            }
            if (elect_one())
              mma_commit_pair(&acc_full[buf]);  // (also when giving up: what was issued completes)
            __syncwarp();
          }
        }
      }
      if (!ok) abort_s = 1;
    }
  } else if (warp >= 4) {
    // epilogue: tensor-memory lane quadrant q, column half h of every tile
    const int ew = warp - 4, q = warp % 4, h = ew / 4;
    const uint32_t lane_base = (uint32_t)(q * 32) << 16;
    uint8_t* cst = smem + S * G::kStage + ew * G::kCStage;
    UAcc orv = 0, sgn = 0;
    uint32_t f = 0;
    bool ok = true;
    for (uint32_t t = first; t < tiles && ok; t += step) {
      UAcc acc[G::kHalf];
#pragma unroll
      for (int j = 0; j < G::kHalf; ++j) acc[j] = 0;
      for (uint32_t p = 0; p < pairs && ok; ++p) {
        const int shift = sp.wa * (int)(p / sp.db) + sp.wb * (int)(p % sp.db);
        for (uint32_t k0 = 0; k0 < nk; k0 += run, ++f) {
          const uint32_t buf = f % G::kBufs;
          // (one decision for the whole warp: the tensor-memory loads are warp-wide)
          if (!__all_sync(0xffffffffu, ax::mbar_wait_suspended(&acc_full[buf], (f / G::kBufs) & 1)) ||
              __any_sync(0xffffffffu, abort_s != 0)) {
            ok = false;
            break;
          }
          tmem_fence_after();
          const uint32_t src = tmem + lane_base + buf * G::kBufCols + h * G::kHalf;
#pragma unroll
          for (int c = 0; c < G::kHalf; c += 16) {
            uint32_t r[16];
            tmem_ld16(src + c, r);
            tmem_ld_wait();
            add_run(r, shift, &acc[c]);
          }
          // this accumulator has been read: the run after next may start
          tmem_fence_before();
          __syncwarp();
          if (lane == 0) arrive_remote(map_rank(&acc_empty[buf], 0));
        }
      }
      if (!ok) {
        abort_s = 1;
        break;
      }
      uint32_t tm, tn;
      tile_coords(t, args.tiles_m, args.tiles_n, tm, tn);
      const uint64_t row0 = (uint64_t)tm * kBM + rank * 128 + q * 32;
      const uint64_t col0 = (uint64_t)tn * BN + h * G::kHalf;
      // (rows and columns outside C are products of zero fill: they add nothing)
#pragma unroll
      for (int j = 0; j < G::kHalf; ++j) {
        orv |= (UAcc)((Acc)acc[j] ^ ((Acc)acc[j] >> (sizeof(Acc) * 8 - 1)));
        sgn |= acc[j];
      }
      if (args.c32)
        store_tile<BN, kAcc64, int32_t>(acc, reinterpret_cast<Acc*>(cst), lane,
                                        reinterpret_cast<int32_t*>(args.c), row0, col0, args.m,
                                        args.n, args.ldc);
      else
        store_tile<BN, kAcc64, int64_t>(acc, reinterpret_cast<Acc*>(cst), lane,
                                        reinterpret_cast<int64_t*>(args.c), row0, col0, args.m,
                                        args.n, args.ldc);
    }
    const uint64_t orv64 = warp_or64((uint64_t)orv);
    const uint32_t neg = __any_sync(0xffffffffu, (Acc)sgn < 0);
    if (lane == 0) {
      if (orv64) atomicOr(reinterpret_cast<unsigned long long*>(&args.out->stat_or),
                          (unsigned long long)orv64);
      if (neg) atomicOr(&args.out->stat_neg, 1u);
    }
  }
  __syncwarp();
  tmem_fence_before();
  __syncthreads();
  if (threadIdx.x == 0) {
    // the copies of both CTAs land on the leader's barriers: all of them have
    // (at once) unless a wait gave up, and then this waits for them (bounded)
    // before shared memory is released
    if (rank == 0) {
      const uint32_t issued = issued_s;
      for (uint32_t g = issued > (uint32_t)S ? issued - S : 0; g < issued; ++g)
        if (!ax::mbar_wait_suspended(&full_bar[g % S], (g / S) & 1)) break;
    }
    if (abort_s) set_status(args.out, CCM_E_TIMEOUT);
  }
  cluster_sync();
  tmem_fence_after();
  if (warp == 1) {
    asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;\n" ::"r"(tmem), "r"(512u));
  }
}

// ---------------------------------------------------------------------------
// Host side
// ---------------------------------------------------------------------------
PFN_cuTensorMapEncodeTiled_v12000 encode_fn() {
  static PFN_cuTensorMapEncodeTiled_v12000 fn = []() -> PFN_cuTensorMapEncodeTiled_v12000 {
    cudaDriverEntryPointQueryResult q;
    void* p = nullptr;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault,
                                         &q) == cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      return reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(p);
    return nullptr;
  }();
  return fn;
}

// Planes [d][rows][kp], as blocks of 64 along k; rows past the end and an odd
// last block are read as zero.
bool make_map(CUtensorMap* map, void* base, uint64_t kp, uint64_t rows, int d, uint32_t box_rows,
              uint32_t box_blocks) {
  auto fn = encode_fn();
  if (!fn) return false;
  cuuint64_t dims[4] = {64, rows, kp / 64, (cuuint64_t)d};
  cuuint64_t strides[3] = {kp * 2, 128, rows * kp * 2};
  cuuint32_t box[4] = {64, box_rows, box_blocks, 1};
  cuuint32_t estr[4] = {1, 1, 1, 1};
  return fn(map, CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 4, base, dims, strides, box, estr,
            CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
            CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// Most digits per operand over every pair of widths up to (ba, bb) and both
// sign modes (the widths and signs themselves are only known on the GPU);
// {0, 0} when some of them has no split.
struct DigitBound {
  uint8_t da, db;
};
DigitBound digit_bound(int ba, int bb) {
  DigitBound d{0, 0};
  if (ba < 1 || bb < 1 || ba + 1 > kMaxE || bb + 1 > kMaxE) return d;
  for (int ea = 1; ea <= ba + 1; ++ea)
    for (int eb = 1; eb <= bb + 1; ++eb) {
      const Split& s = kSplits.at[ea][eb];
      if (!s.da) return DigitBound{0, 0};
      d.da = max(d.da, s.da);
      d.db = max(d.db, s.db);
    }
  return d;
}

struct Bounds {
  int ba, bb;
  DigitBound d;
};
Bounds bounds_of(const ccm_matrix& a, const ccm_matrix& b) {
  Bounds r;
  r.ba = width_bound(a.capacity, a.rows * a.cols);
  r.bb = width_bound(b.capacity, b.rows * b.cols);
  r.d = digit_bound(r.ba, r.bb);
  return r;
}

size_t plane_bytes(uint64_t m, uint64_t k, uint64_t n, int da, int db) {
  const uint64_t kp = round_up(k, 64);
  return round_up(2 * (uint64_t)da * m * kp, 256) + round_up(2 * (uint64_t)db * n * kp, 256);
}

}  // namespace tc

bool matmul_c32(const ccm_matrix& c) { return width_bound(c.capacity, c.rows * c.cols) <= 31; }

// The product runs on the tensor cores when every width the capacities allow
// has a split and every sum stays inside int64.
bool matmul_tc_applies(const ccm_matrix& a, const ccm_matrix& b) {
  const uint64_t m = a.rows, k = a.cols, n = b.cols;
  if (!m || !n || !k || m >= (1ull << 31) || n >= (1ull << 31) || k >= (1ull << 31)) return false;
  const tc::Bounds r = tc::bounds_of(a, b);
  if (!r.d.da || r.ba + r.bb + bitlen_host(k) > 62) return false;
  return tc::encode_fn() != nullptr;
}

// All of C where the planes of both operands fit.  Else the fewest strips (then
// the fewest plane elements written: B's are written again for every strip of
// A) whose planes fit, in steps of 32 rows and columns.  Up to kMaxParts of each:
// the least workspace that ccm_matmul accepts for the explicit tensor path
// never needs more, and with less room than about a quarter of the planes the
// CUDA cores take the product.  4096^3 in the least workspace (in brackets: with
// room for all): 4 bits 199 us (139), 12 bits 460 (362), 16 bits 564 (507); on
// the CUDA cores 33 to 107 times as long.
Strips matmul_tc_strips(const ccm_matrix& a, const ccm_matrix& b, size_t room) {
  constexpr uint64_t kMaxParts = 4;
  const uint64_t m = a.rows, k = a.cols, n = b.cols;
  const tc::Bounds r = tc::bounds_of(a, b);
  if (tc::plane_bytes(m, k, n, r.d.da, r.d.db) <= room) return Strips{m, n};
  Strips best{0, 0};
  uint64_t best_parts = 0, best_written = 0;
  for (uint64_t pm = 1; pm <= kMaxParts; ++pm)
    for (uint64_t pn = 1; pn <= kMaxParts; ++pn) {
      const Strips s{umin(m, tc::round_up((m + pm - 1) / pm, 32)),
                     umin(n, tc::round_up((n + pn - 1) / pn, 32))};
      if (tc::plane_bytes(s.rows, k, s.cols, r.d.da, r.d.db) > room) continue;
      const uint64_t written = r.d.da * m + r.d.db * n * (pn > 1 ? pm : 1);
      if (!best_parts || pm * pn < best_parts ||
          (pm * pn == best_parts && written < best_written)) {
        best = s;
        best_parts = pm * pn;
        best_written = written;
      }
    }
  return best;
}

size_t matmul_tc_bytes_upper(uint64_t m, uint64_t k, uint64_t n) {
  if (!m || !n || !k) return 0;
  return tc::plane_bytes(m, k, n, tc::kMaxDigits, tc::kMaxDigits);
}

namespace {

template <int BN, bool kAcc64>
cudaError_t launch_mm(const CUtensorMap& ta, const CUtensorMap& tb, const tc::MmArgs& args,
                      unsigned pairs, bool pdl, cudaStream_t st) {
  using G = tc::Geo<BN, kAcc64>;
  static DeviceCache attr;  // (the attribute is the device's)
  int dev = 0;
  cudaGetDevice(&dev);
  cudaError_t e = cudaSuccess;
  attr.get(dev, 0, [&] {
    e = cudaFuncSetAttribute(tc::k_mm<BN, kAcc64>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)G::kSmem);
    return e == cudaSuccess;
  });
  if (e != cudaSuccess) return e;
  if (pdl)
    return ax::launch_pdl(tc::k_mm<BN, kAcc64>, dim3(2 * pairs), dim3(tc::kThreads), G::kSmem, st,
                          ta, tb, args);
  tc::k_mm<BN, kAcc64><<<2 * pairs, tc::kThreads, G::kSmem, st>>>(ta, tb, args);
  return cudaGetLastError();
}

}  // namespace

namespace {

// C's strip of `rows` x `cols` from row0, col0 on: the planes that are not in
// place yet, then their product.
struct StripCall {
  const ccm_matrix &a, &b, &c;
  void* c_scratch;
  __half *pa, *pb;
  tc::Bounds r;
  uint64_t row0, col0, rows, cols;
  bool planes_a, planes_b;
  bool pdl;
};

int run_strip(const StripCall& s, cudaStream_t st) {
  const ccm_matrix &a = s.a, &b = s.b, &c = s.c;
  const tc::Bounds& r = s.r;
  const uint64_t m = s.rows, k = a.cols, n = s.cols, kp = tc::round_up(k, 64);
  const bool pdl = s.pdl;
  {
    tc::PlaneArgs p{c.hdr, a.hdr, b.hdr, a.words, b.words, s.row0, s.col0, m, k, n, kp, b.cols,
                    s.pa, s.pb, 0, 0, 0};
    p.row_runs = (uint32_t)((kp / 8 + 31) / 32);
    p.blocks_a =
        s.planes_a ? (uint32_t)umin((m * p.row_runs + 7) / 8, (uint64_t)num_sms() * 32) : 0;
    p.tiles_k = (uint32_t)(kp / 64);
    const uint64_t tiles_b = s.planes_b ? p.tiles_k * ((n + 63) / 64) : 0;
    const unsigned grid = (unsigned)(p.blocks_a + tiles_b);
    if (pdl)
      ax::launch_pdl(tc::k_planes, dim3(grid), dim3(256), 0, st, p);
    else
      tc::k_planes<<<grid, 256, 0, st>>>(p);
    note_launch();
  }
  // 32-bit accumulators when no result can leave int32.
  const bool acc32 = r.ba + r.bb + bitlen_host(k) <= 31;
  const uint64_t tiles_m = (m + tc::kBM - 1) / tc::kBM, pairs = (uint64_t)num_sms() / 2;
  const int bn = tc::tile_columns(m, n, acc32, pairs);
  const uint32_t sub = bn > 128 ? 1 : 2;
  CUtensorMap ta, tb;
  if (!tc::make_map(&ta, s.pa, kp, m, r.d.da, 128, sub) ||
      !tc::make_map(&tb, s.pb, kp, n, r.d.db, (uint32_t)bn / 2, sub))
    return CCM_E_CUDA;
  const bool c32 = matmul_c32(c);
  const uint64_t at = s.row0 * b.cols + s.col0;
  void* cs = c32 ? (void*)((int32_t*)s.c_scratch + at) : (void*)((int64_t*)s.c_scratch + at);
  tc::MmArgs args{c.hdr, a.hdr, b.hdr, cs, m, n, b.cols, (uint32_t)((k + tc::kBK - 1) / tc::kBK),
                  (uint32_t)tiles_m, (uint32_t)((n + bn - 1) / bn), c32 ? 1 : 0};
  const unsigned grid = (unsigned)umin((uint64_t)args.tiles_m * args.tiles_n, pairs);
  cudaError_t e = cudaErrorInvalidValue;
  profile_begin(st);  // (of the first strip's product; run_matmul_tc ends it)
  if (acc32) {
    switch (bn) {
      case 256: e = launch_mm<256, false>(ta, tb, args, grid, pdl, st); break;
      case 224: e = launch_mm<224, false>(ta, tb, args, grid, pdl, st); break;
      case 192: e = launch_mm<192, false>(ta, tb, args, grid, pdl, st); break;
      case 128: e = launch_mm<128, false>(ta, tb, args, grid, pdl, st); break;
      default: e = launch_mm<64, false>(ta, tb, args, grid, pdl, st); break;
    }
  } else {
    switch (bn) {
      case 128: e = launch_mm<128, true>(ta, tb, args, grid, pdl, st); break;
      default: e = launch_mm<64, true>(ta, tb, args, grid, pdl, st); break;
    }
  }
  note_launch();
  return e == cudaSuccess ? CCM_OK : CCM_E_CUDA;
}

}  // namespace

int run_matmul_tc(const ccm_matrix& a, const ccm_matrix& b, const ccm_matrix& c, void* c_scratch,
                  void* ws, const Strips& s, cudaStream_t st) {
  const tc::Bounds r = tc::bounds_of(a, b);
  const uint64_t kp = tc::round_up(a.cols, 64);
  __half* pa = (__half*)ws;
  __half* pb = (__half*)((char*)ws + tc::round_up(2 * (uint64_t)r.d.da * s.rows * kp, 256));
  const bool pdl = !profile_armed();
  int rc = CCM_OK;
  for (uint64_t i = 0; i < a.rows && rc == CCM_OK; i += s.rows)
    for (uint64_t j = 0; j < b.cols && rc == CCM_OK; j += s.cols)
      rc = run_strip({a, b, c, c_scratch, pa, pb, r, i, j, umin(s.rows, a.rows - i),
                      umin(s.cols, b.cols - j), j == 0, i == 0 || s.cols < b.cols, pdl},
                     st);
  profile_end(st);
  return rc;
}

}  // namespace ccm
