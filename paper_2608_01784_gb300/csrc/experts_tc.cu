// experts_tc.cu — grouped SwiGLU expert GEMMs over ragged per-expert row
// ranges on the 5th-generation tensor cores (tcgen05.mma, accumulators in
// TMEM, operands staged by TMA), for the sparse execution of Eq. 2 (REFLEX
// Sec. 3.2).  Routed-expert work is 6 * d * inter FLOPs per selected pair
// (Eq. 10), two thirds in the gate/up GEMM and one third in the down GEMM.
//
// Problem.  Rows of the pair-ordered input A are grouped by expert
// (rows [offsets[e], offsets[e+1]) belong to expert e).  For each group:
//   SwiGLU mode: out[r, c] = silu(A_r . Wg[e, c]) * (A_r . Wu[e, c])
//   Down mode:   out[r, n] = A_r . Wd[e, n]
// with every operand K-major bf16 and fp32 accumulation; out is bf16.
//
// Tiles.  An output tile is 128 rows (one m-tile of a group; rows past the
// group's end are computed from the next rows or TMA zero fill and never
// stored) by BN columns.  In SwiGLU mode the BN-row weight tile is the
// BN/2 gate rows followed by the matching BN/2 up rows, loaded by two TMA
// boxes, so one MMA chain yields gate and up side by side in TMEM and the
// epilogue emits BN/2 activations.  Tiles are numbered expert-major, then
// n-tile, then m-tile, so CTAs running at the same time share weight tiles
// in L2.
//
// Kernel.  Persistent: one CTA per SM walks tiles blockIdx.x, +gridDim.x, ...
//   warp 0     TMA producer: 192 KB ring of (A 128x64, B BNx64) bf16 stages
//              (4 for BN 256, 6 for 128, 8 for 64), 128-byte swizzle,
//              completion on a per-stage mbarrier;
//   warp 1     allocates 2*BN TMEM columns (two accumulators) and issues
//              tcgen05.mma (M=128, N=BN, K=16) from one thread; each stage
//              is released with tcgen05.commit when its MMAs have read it;
//   warps 2-5  epilogue: tcgen05.ld 32x32b of their TMEM lane quarter,
//              SwiGLU or conversion, 16-byte stores; the accumulator is
//              handed back through an mbarrier, so the epilogue of tile i
//              overlaps the main loop of tile i+1.
// A tile number maps to (expert, n-tile, rows) through the per-expert tile
// prefix, copied into shared memory once per CTA (TileIndex).  Every wait is
// bounded (2 s); on expiry the CTA records the timeout in the error word,
// drains its outstanding TMA loads and MMAs, frees TMEM and exits.  The
// 2-SM (CTA pair) variant further down has its own description.
#include "common.cuh"
#include "internal.h"

namespace rx {
namespace {

constexpr int BM = kTileM;   // 128
constexpr int BK = 64;       // 64 bf16 = 128 bytes = one swizzle row
constexpr int UMMA_K = 16;
constexpr int kThreads = 192;
// scores mode: four more warps (6-9) that sum the squares of each A row from
// the shared-memory stages while the MMAs read them (token norms for the
// router screen's interval)
constexpr int kThreadsScores = 320;
constexpr int kRingBytes = 192 * 1024;  // TMA ring budget per CTA
constexpr uint64_t kWaitNs = 2000000000ull;
constexpr uint64_t kDrainNs = 1000000000ull;

enum { kModeSwiGLU = 0, kModeDown = 1, kModeScores = 2 };

template <int BN>
struct Cfg {
  static constexpr int kABytes = BM * BK * 2;
  static constexpr int kBBytes = BN * BK * 2;
  static constexpr int kStageBytes = kABytes + kBBytes;
  static constexpr int kStages = kRingBytes / kStageBytes;  // 4 (BN 256), 6 (BN 128)
  static constexpr int kTmemCols = 2 * BN;
  static constexpr int kBarBytes = 256;
  static constexpr int kIndexInts = 2 * 1025;  // both prefix arrays, E <= 1024
  static constexpr int kSmemBytes = kStages * kStageBytes + kBarBytes + kIndexInts * 4 + 1024;
  static_assert(kStages >= 2 && kStages <= 8, "ring depth");
};

struct KParams {
  int K;
  int n_tiles;           // column tiles per group
  int b_rows_per_group;
  int b_up_offset;
  GroupRows g;
  const int32_t* mt_prefix;  // [E+1] prefix of tile counts (grouped mode)
  int max_mtiles;            // host upper bound of m-tiles
  int tile_rows;             // rows per tile: 128 (1-SM) or 256 (CTA pair)
  __nv_bfloat16* out;
  int ldo;
  uint32_t* err;
  // scores mode (dense, fp32 out): K is cut into k_splits slices; slice ks of
  // tile (m, n) writes out_f32 + ks * split_stride; columns >= n_valid dropped
  int k_splits;
  float* out_f32;
  int64_t split_stride;
  int n_valid;
  // 1: launched right behind a kernel that writes none of this kernel's
  // inputs or outputs; start at once and wait for it only before exiting
  int defer_wait;
  // SwiGLU: map_b is the 3D {K, inter, 2 groups} map of tc_gate_up_3d
  int b3d;
  // scores mode, k_splits == 1: sum of squares of every A row (fp32), nullable
  float* norm_out;
  // 1-SM kernel: a dense problem carried by the same launch (the shared
  // expert): its sh_tiles tiles come first, sh_rows rows, n_tiles2 column
  // tiles, reduction length K2, operands through map_a2 / map_b2
  int sh_tiles;
  int sh_rows;
  int n_tiles2;
  int K2;
  __nv_bfloat16* out2;
  int ldo2;
  // 1: the first ring stages' weights are requested before the dependency
  // wait (early_tile)
  int early_b;
  // SwiGLU on CTA pairs: A rows gathered from the token rows (TcGemmArgs)
  const int32_t* gather_perm;
  const __nv_bfloat16* gather_x;
  int gather_kmax;
  int gather_tokens;
};

// ---- PTX wrappers ---------------------------------------------------------
__device__ __forceinline__ void mbar_expect_tx(uint32_t bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar),
               "r"(bytes)
               : "memory");
}
// Announces bytes on a phase whose arrival comes later (another expect_tx).
__device__ __forceinline__ void mbar_expect_tx_only(uint32_t bar, uint32_t bytes) {
  asm volatile("mbarrier.expect_tx.relaxed.cta.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(bytes)
               : "memory");
}
__device__ __forceinline__ void mbar_arrive1(uint32_t bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void tma_load_2d(uint32_t dst, const CUtensorMap* map,
                                            int c0, int c1, uint32_t bar) {
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes"
      " [%0], [%1, {%2, %3}], [%4];" ::"r"(dst),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(c0), "r"(c1), "r"(bar)
      : "memory");
}
// L2 eviction priority for TMA loads.  A weight tile of a group that fits in
// one m-tile is read by exactly one CTA, so it is loaded evict-first and the
// weight stream does not push the group rows, activations and outputs out of
// L2 (LLaDA-MoE layer: gate/up GEMM 102 -> 97 us).  Every other load is a
// plain load: evict-first on weights that several m-tiles read makes the
// second reader miss, and an explicit evict-normal hint measured slower than
// no hint (2-5% at 4096-16384 tokens).
constexpr int kPolFirst = 0;
__device__ __forceinline__ uint64_t l2_policy(int) {
  uint64_t pol;
  asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(pol));
  return pol;
}
__device__ __forceinline__ void tma_load_2d_hint(uint32_t dst, const CUtensorMap* map, int c0,
                                                 int c1, uint32_t bar, uint64_t pol) {
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes"
      ".L2::cache_hint [%0], [%1, {%2, %3}], [%4], %5;" ::"r"(dst),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(c0), "r"(c1), "r"(bar), "l"(pol)
      : "memory");
}
// 3D boxes: the gate and up blocks of one weight tile in one copy (the map's
// dims are {K, rows per half, halves}: halves 2e and 2e + 1 of expert e)
__device__ __forceinline__ void tma_load_3d(uint32_t dst, const CUtensorMap* map, int c0,
                                            int c1, int c2, uint32_t bar) {
  asm volatile(
      "cp.async.bulk.tensor.3d.shared::cluster.global.tile.mbarrier::complete_tx::bytes"
      " [%0], [%1, {%2, %3, %4}], [%5];" ::"r"(dst),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(c0), "r"(c1), "r"(c2), "r"(bar)
      : "memory");
}
__device__ __forceinline__ void tma_load_3d_hint(uint32_t dst, const CUtensorMap* map, int c0,
                                                 int c1, int c2, uint32_t bar, uint64_t pol) {
  asm volatile(
      "cp.async.bulk.tensor.3d.shared::cluster.global.tile.mbarrier::complete_tx::bytes"
      ".L2::cache_hint [%0], [%1, {%2, %3, %4}], [%5], %6;" ::"r"(dst),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(c0), "r"(c1), "r"(c2), "r"(bar), "l"(pol)
      : "memory");
}
__device__ __forceinline__ void prefetch_map(const CUtensorMap* map) {
  asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(map))
               : "memory");
}
// Shared-memory matrix descriptor: K-major tile with 128-byte swizzle, rows
// of 128 bytes, 8-row groups 1024 bytes apart.
__device__ __forceinline__ uint64_t desc_sw128(uint32_t saddr) {
  uint64_t desc = static_cast<uint64_t>((saddr >> 4) & 0x3FFFu);  // start
  desc |= static_cast<uint64_t>(1) << 16;            // leading offset (unused)
  desc |= static_cast<uint64_t>(1024 >> 4) << 32;    // stride offset
  desc |= static_cast<uint64_t>(1) << 46;            // descriptor version
  desc |= static_cast<uint64_t>(2) << 61;            // 128-byte swizzle
  return desc;
}
// Instruction descriptor of kind::f16: bf16 A and B, fp32 accumulator,
// both K-major, M = 128, N = n.
__host__ __device__ constexpr uint32_t idesc_bf16(int n) {
  return (1u << 4) | (1u << 7) | (1u << 10) |
         (static_cast<uint32_t>(n >> 3) << 17) |
         (static_cast<uint32_t>(BM >> 4) << 24);
}
__device__ __forceinline__ void mma_bf16(uint32_t tmem_d, uint64_t da,
                                         uint64_t db, uint32_t idesc,
                                         uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}\n" ::"r"(tmem_d),
      "l"(da), "l"(db), "r"(idesc), "r"(accumulate)
      : "memory");
}
__device__ __forceinline__ void mma_commit(uint32_t bar) {
  asm volatile(
      "tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar)
      : "memory");
}
__device__ __forceinline__ void tc_fence_before() {
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
}
__device__ __forceinline__ void tc_fence_after() {
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
}
__device__ __forceinline__ void tmem_alloc(uint32_t slot, uint32_t ncols) {
  asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(slot),
               "r"(ncols)
               : "memory");
  asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_dealloc(uint32_t taddr, uint32_t ncols) {
  asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr),
               "r"(ncols)
               : "memory");
}
// 32 TMEM lanes x 32 consecutive fp32 columns: one column per register.
__device__ __forceinline__ void tmem_ld32(uint32_t taddr, uint32_t (&r)[32]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
      "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
      "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, "
      "[%32];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]),
        "=r"(r[6]), "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]),
        "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]), "=r"(r[16]),
        "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]),
        "=r"(r[22]), "=r"(r[23]), "=r"(r[24]), "=r"(r[25]), "=r"(r[26]),
        "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
      : "r"(taddr));
}
__device__ __forceinline__ void tmem_ld_wait() {
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
}

// ---- tile numbering -------------------------------------------------------
struct Tile {
  int e, n, row0, rows;
  int mtiles;  // m-tiles of the tile's group (readers of each weight tile)
  int ks;      // K slice (scores mode; 0 otherwise)
  bool sh;     // tile of the dense problem that the launch carries along
};

// The group prefix arrays a tile lookup reads: copies in shared memory where
// they fit, else the global arrays.  Looking a tile up takes a binary search
// over the experts; from global memory that is a chain of about log2(E) + 2
// dependent L2 loads (about 3 us), longer than the ring's lead over the MMAs
// at each tile start, so the copies are made once per CTA.
struct TileIndex {
  const int32_t* pref;  // [E+1] tile-count prefix (p.mt_prefix)
  const int32_t* offs;  // [E+1] row offsets (p.g.offsets)
};
// Every thread of the CTA calls this (it synchronises the CTA) after the
// kernel's dependency wait; cache holds cap ints.
__device__ __forceinline__ TileIndex load_tile_index(const KParams& p, int32_t* cache,
                                                     int cap) {
  TileIndex ix{p.mt_prefix, p.g.offsets};
  if (p.g.offsets == nullptr) return ix;
  const int n = p.g.E + 1;
  const bool both = 2 * n <= cap, pref_only = !both && n <= cap;
  if (both || pref_only) {
    for (int i = threadIdx.x; i < n; i += blockDim.x) {
      cache[i] = p.mt_prefix[i];
      if (both) cache[n + i] = p.g.offsets[i];
    }
    __syncthreads();
    ix.pref = cache;
    if (both) ix.offs = cache + n;
  }
  return ix;
}

template <bool SH>
__device__ __forceinline__ int total_tiles(const KParams& p, const TileIndex& ix) {
  int mt;
  if (p.g.offsets == nullptr) {
    mt = (p.g.dense_rows + p.tile_rows - 1) / p.tile_rows * p.k_splits;
  } else {
    mt = ix.pref[p.g.E];
    if (mt < 0) mt = 0;
    if (mt > p.max_mtiles) mt = p.max_mtiles;
  }
  return mt * p.n_tiles + (SH ? p.sh_tiles : 0);
}

// Tile t -> (expert, n-tile, rows); false when the workspace is inconsistent.
// SH: the launch carries a dense problem, whose tiles come first.
template <bool SH>
__device__ __forceinline__ bool decode_tile(const KParams& p, const TileIndex& ix, int t,
                                            Tile& o) {
  o.sh = SH && t < p.sh_tiles;
  if (o.sh) {
    const int mt = (p.sh_rows + p.tile_rows - 1) / p.tile_rows;
    o.ks = 0;
    o.e = 0;
    o.n = t / mt;
    o.row0 = (t % mt) * p.tile_rows;
    o.rows = min(p.tile_rows, p.sh_rows - o.row0);
    o.mtiles = mt;
    return true;
  }
  if (SH) t -= p.sh_tiles;
  if (p.g.offsets == nullptr) {
    const int mt = (p.g.dense_rows + p.tile_rows - 1) / p.tile_rows;
    const int per = mt * p.n_tiles;
    o.ks = t / per;
    t -= o.ks * per;
    o.e = 0;
    o.n = t / mt;
    o.row0 = (t % mt) * p.tile_rows;
    o.rows = min(p.tile_rows, p.g.dense_rows - o.row0);
    o.mtiles = mt;
    return o.ks < p.k_splits;
  }
  o.ks = 0;
  int lo = 0, hi = p.g.E;  // n_tiles*prefix[lo] <= t < n_tiles*prefix[hi]
  while (hi - lo > 1) {
    const int mid = (lo + hi) >> 1;
    if (p.n_tiles * ix.pref[mid] <= t) lo = mid; else hi = mid;
  }
  // an inconsistent workspace can hold any values; in unsigned arithmetic
  // whatever wraps fails one of the comparisons
  const uint32_t first = ix.pref[lo], last = ix.pref[lo + 1];
  const uint32_t row_lo = ix.offs[lo], row_hi = ix.offs[lo + 1];
  const uint32_t mt_e = last - first, most = p.max_mtiles;
  if (mt_e - 1u >= most) return false;
  const uint32_t l = t - p.n_tiles * first, n = l / mt_e;
  const uint32_t row0 = row_lo + (l - n * mt_e) * p.tile_rows;
  o.e = lo;
  o.mtiles = mt_e;
  o.n = n;
  o.row0 = row0;
  o.rows = min(static_cast<uint32_t>(p.tile_rows), row_hi - row0);
  // row_hi <= cap < 2^31 and (l mod mt_e) tile_rows < cap + E tile_rows, so
  // row0 cannot wrap past row_lo while row_lo <= row_hi
  return n < static_cast<uint32_t>(p.n_tiles) && row_lo <= row0 && row0 < row_hi &&
         row_hi <= static_cast<uint32_t>(p.g.cap_rows);
}

// Expert, n-tile and m-tile count of tile t, read before the kernel's
// dependency wait, by a whole warp (a 32-ary search: one or two rounds of L2
// loads).  The host asks for it (early_b) only where the kernel in front of
// this one in the stream waited for the dispatch itself before it let this
// one launch, so the prefix is complete; the operand that the kernel in front
// writes (A) is not touched.  False: no such tile.
template <bool SH>
__device__ __forceinline__ bool early_tile(const KParams& p, int t, Tile& o) {
  o.sh = SH && t < p.sh_tiles;
  if (o.sh) {
    const int mt = (p.sh_rows + p.tile_rows - 1) / p.tile_rows;
    o.e = 0;
    o.n = t / mt;
    o.mtiles = mt;
    return true;
  }
  if (SH) t -= p.sh_tiles;
  if (p.g.offsets == nullptr) {
    const int mt = (p.g.dense_rows + p.tile_rows - 1) / p.tile_rows;
    o.e = 0;
    o.n = t / mt;
    o.mtiles = mt;
    return o.n < p.n_tiles;
  }
  const int lane = threadIdx.x & 31;
  int lo = 0, n = p.g.E;
  while (n > 1) {
    const int step = (n + 31) / 32;
    const bool below = lane * step < n && p.n_tiles * __ldcg(p.mt_prefix + lo + lane * step) <= t;
    const int hit = 31 - __clz(__ballot_sync(0xffffffffu, below) | 1u);
    lo += hit * step;
    n = min(step, n - hit * step);
  }
  const int first = __ldcg(p.mt_prefix + lo), mt = __ldcg(p.mt_prefix + lo + 1) - first;
  if (mt <= 0 || t < p.n_tiles * first) return false;
  o.e = lo;
  o.n = (t - p.n_tiles * first) / mt;
  o.mtiles = mt;
  return o.n < p.n_tiles;
}

template <int BN, int MODE, bool SH>
__global__ void __launch_bounds__(MODE == kModeScores ? kThreadsScores : kThreads, 1)
    grouped_gemm_kernel(const __grid_constant__ CUtensorMap map_a,
                        const __grid_constant__ CUtensorMap map_b,
                        const __grid_constant__ CUtensorMap map_a2,
                        const __grid_constant__ CUtensorMap map_b2, const KParams p) {
  using C = Cfg<BN>;
  constexpr int kStages = C::kStages;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>(
      (reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~static_cast<uintptr_t>(1023));
  uint8_t* sa = smem;
  uint8_t* sb = smem + kStages * C::kABytes;
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem + kStages * C::kStageBytes);
  uint64_t* full = bars;
  uint64_t* empty = bars + kStages;
  uint64_t* acc_full = bars + 2 * kStages;
  uint64_t* acc_empty = bars + 2 * kStages + 2;
  uint64_t* drain = bars + 2 * kStages + 4;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + 2 * kStages + 5);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);

  const int warp = threadIdx.x >> 5;
  const int lane = threadIdx.x & 31;

  const bool norms = MODE == kModeScores && p.norm_out != nullptr;
  if (threadIdx.x == 0) {
    for (int s = 0; s < kStages; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], norms ? 5 : 1);  // the MMA commit (+ 4 norm warps)
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(&acc_full[b], 1);
      mbar_init(&acc_empty[b], 4);  // one arrival per epilogue warp
    }
    mbar_init(drain, 1);
    *abort_flag = 0;
    fence_mbar_init();
    prefetch_map(&map_a);
    prefetch_map(&map_b);
    if (SH) {
      prefetch_map(&map_a2);
      prefetch_map(&map_b2);
    }
  }
  const int nk_main = p.K / BK / p.k_splits, nk_sh = p.K2 / BK;  // k-blocks per tile
  auto nk_of = [&](int t) { return SH && t < p.sh_tiles ? nk_sh : nk_main; };
  const uint64_t pol_once = l2_policy(kPolFirst);
  // the weight tile of k-block kb of tile tl into stage s
  auto load_weights = [&](const Tile& tl, bool once, int kb, int s, int nk) {
    const uint32_t fb = smem_addr(&full[s]);
    const uint32_t b_dst = smem_addr(sb + s * C::kBBytes);
    const CUtensorMap* mb = SH && tl.sh ? &map_b2 : &map_b;
    const int k0 = (tl.ks * nk + kb) * BK;
    const int wr = tl.e * p.b_rows_per_group + tl.n * (MODE == kModeSwiGLU ? BN / 2 : BN);
    auto load_b = [&](uint32_t dst, int row) {
      if (once) tma_load_2d_hint(dst, mb, k0, row, fb, pol_once);
      else tma_load_2d(dst, mb, k0, row, fb);
    };
    if (MODE == kModeSwiGLU && p.b3d) {
      // gate rows then up rows of the tile, one copy
      if (once) tma_load_3d_hint(b_dst, mb, k0, tl.n * (BN / 2), 2 * tl.e, fb, pol_once);
      else tma_load_3d(b_dst, mb, k0, tl.n * (BN / 2), 2 * tl.e, fb);
    } else {
      load_b(b_dst, wr);
      if (MODE == kModeSwiGLU) load_b(b_dst + (BN / 2) * BK * 2, wr + p.b_up_offset);
    }
  };
  // The ring's first weights while the kernel in front still runs: the
  // stream starts a ring earlier (32 tokens of the LLaDA-MoE shape 162 -> 158
  // us, 16 of the LLaDA2.0-mini shape 143 -> 137, 1024 337 -> 330)
  int early = 0;  // stages whose weights are on their way (warp 0)
  if (MODE != kModeScores && p.early_b && warp == 0) {
    __syncwarp();
    Tile tl;
    if (early_tile<SH>(p, blockIdx.x, tl)) {
      tl.ks = 0;
      const int nk = nk_of(blockIdx.x);
      early = nk < kStages ? nk : kStages;
      const bool once = p.g.offsets != nullptr && tl.mtiles == 1;
      if (lane == 0) {
        for (int s = 0; s < early; ++s) {
          mbar_expect_tx_only(smem_addr(&full[s]), C::kBBytes);
          load_weights(tl, once, s, s, nk);
        }
      }
    }
  }
  if (warp == 1) tmem_alloc(smem_addr(tmem_slot), C::kTmemCols);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;
  // the tile count and every operand come from earlier kernels
  if (!p.defer_wait) grid_dep_wait();
  grid_dep_launch();
  const TileIndex ix = load_tile_index(
      p, reinterpret_cast<int32_t*>(smem + kStages * C::kStageBytes + C::kBarBytes),
      C::kIndexInts);
  const int ntiles = total_tiles<SH>(p, ix);

  if (warp == 0 && lane == 0) {
    // ---------------- TMA producer ----------------
    int stage = 0;
    uint32_t phase = 0;
    uint32_t issued_mask = 0, issued_phase = 0;
    bool ok = true;
    const bool grouped = p.g.offsets != nullptr;
    for (int t = blockIdx.x; t < ntiles && ok; t += gridDim.x) {
      Tile tl;
      if (!decode_tile<SH>(p, ix, t, tl)) {
        set_err(p.err, kErrIndex);
        *abort_flag = 1;
        break;
      }
      const bool once = grouped && tl.mtiles == 1;  // one reader per weight tile
      const int nk = nk_of(t);
      const CUtensorMap* ma = SH && tl.sh ? &map_a2 : &map_a;
      for (int kb = 0; kb < nk; ++kb) {
        if (!mbar_wait(&empty[stage], phase ^ 1u, abort_flag, kWaitNs)) {
          ok = false;
          break;
        }
        const uint32_t fb = smem_addr(&full[stage]);
        const int k0 = (tl.ks * nk + kb) * BK;
        const bool ahead = early > 0;  // the weights are already on their way
        mbar_expect_tx(fb, ahead ? C::kABytes : C::kStageBytes);
        tma_load_2d(smem_addr(sa + stage * C::kABytes), ma, k0, tl.row0, fb);
        if (ahead) --early;
        else load_weights(tl, once, kb, stage, nk);
        issued_mask |= 1u << stage;
        issued_phase = (issued_phase & ~(1u << stage)) | (phase << stage);
        if (++stage == kStages) {
          stage = 0;
          phase ^= 1u;
        }
      }
    }
    if (!ok) {
      set_err(p.err, kErrTimeout);
      *abort_flag = 1;
    }
    // weights requested early for stages that never got their rows (no tile,
    // or an error): the phase completes with the arrival that is missing
    const int unused = early;
    for (int s = 0; s < unused; ++s) {
      const int st = (stage + s) % kStages;
      mbar_arrive1(smem_addr(&full[st]));
      mbar_wait(&full[st], 0, nullptr, kDrainNs);
    }
    if (*abort_flag) {
      // every issued load must land before the CTA may exit
      for (int s = 0; s < kStages; ++s)
        if (issued_mask & (1u << s))
          mbar_wait(&full[s], (issued_phase >> s) & 1u, nullptr, kDrainNs);
    }
  } else if (warp == 1 && lane == 0) {
    // ---------------- MMA issuer ----------------
    constexpr uint32_t idesc = idesc_bf16(BN);
    int stage = 0;
    uint32_t phase = 0;
    int lt = 0;
    bool ok = true, issued_any = false;
    for (int t = blockIdx.x; t < ntiles && ok; t += gridDim.x, ++lt) {
      const int ab = lt & 1;
      const uint32_t acc_phase = (lt >> 1) & 1;
      if (!mbar_wait(&acc_empty[ab], acc_phase ^ 1u, abort_flag, kWaitNs)) {
        ok = false;
        break;
      }
      tc_fence_after();
      const uint32_t d_tmem = tmem_base + static_cast<uint32_t>(ab * BN);
      const int nk = nk_of(t);
      for (int kb = 0; kb < nk; ++kb) {
        if (!mbar_wait(&full[stage], phase, abort_flag, kWaitNs)) {
          ok = false;
          break;
        }
        tc_fence_after();
        const uint32_t a0 = smem_addr(sa + stage * C::kABytes);
        const uint32_t b0 = smem_addr(sb + stage * C::kBBytes);
#pragma unroll
        for (int k = 0; k < BK / UMMA_K; ++k) {
          mma_bf16(d_tmem, desc_sw128(a0 + k * UMMA_K * 2),
                   desc_sw128(b0 + k * UMMA_K * 2), idesc,
                   (kb > 0 || k > 0) ? 1u : 0u);
        }
        issued_any = true;
        mma_commit(smem_addr(&empty[stage]));
        if (++stage == kStages) {
          stage = 0;
          phase ^= 1u;
        }
      }
      if (!ok) break;
      mma_commit(smem_addr(&acc_full[ab]));
    }
    if (!ok) {
      set_err(p.err, kErrTimeout);
      *abort_flag = 1;
    }
    if (*abort_flag && issued_any) {
      // MMAs in flight must finish before TMEM is freed
      mma_commit(smem_addr(drain));
      mbar_wait(drain, 0, nullptr, kDrainNs);
    }
  } else if (MODE == kModeScores && warp >= 6) {
    // ---------------- row norms (scores mode) ----------------
    // warp 6 + q sums the squares of A rows 32 q .. 32 q + 31 of every tile,
    // one row per lane, reading each stage as the MMAs do and releasing it
    // on the stage's "empty" barrier next to the MMA commit
    if (norms) {
      const int r = (warp - 6) * 32 + lane;
      int stage = 0;
      uint32_t phase = 0;
      bool ok = true;
      for (int t = blockIdx.x; t < ntiles && ok; t += gridDim.x) {
        Tile tl;
        const bool tile_ok = decode_tile<SH>(p, ix, t, tl);
        float ss = 0.f;
        for (int kb = 0; kb < nk_main; ++kb) {
          // every lane observes the stage's completion before reading it
          const bool w = __all_sync(0xffffffffu,
                                    mbar_wait(&full[stage], phase, abort_flag, kWaitNs));
          if (!w) {
            ok = false;
            break;
          }
          // row r of the 128-byte-swizzled A stage: 16-byte chunk c at
          // r * 128 + ((c ^ (r & 7)) << 4)
          const uint8_t* rowp = sa + stage * C::kABytes + r * 128;
#pragma unroll
          for (int c = 0; c < 8; ++c) {
            const uint4 q = *reinterpret_cast<const uint4*>(rowp + ((c ^ (r & 7)) << 4));
            const uint32_t wd[4] = {q.x, q.y, q.z, q.w};
#pragma unroll
            for (int i = 0; i < 4; ++i) {
              const float lo = __uint_as_float(wd[i] << 16);
              const float hi = __uint_as_float(wd[i] & 0xffff0000u);
              ss = fmaf(lo, lo, ss);
              ss = fmaf(hi, hi, ss);
            }
          }
          fence_proxy_async_smem();  // the reads above, before the next TMA fill
          __syncwarp();
          if (lane == 0) mbar_arrive1(smem_addr(&empty[stage]));
          if (++stage == kStages) {
            stage = 0;
            phase ^= 1u;
          }
        }
        if (ok && tile_ok && r < tl.rows) p.norm_out[tl.row0 + r] = ss;
      }
      if (!ok && lane == 0) {
        if (!*abort_flag) set_err(p.err, kErrTimeout);
        *abort_flag = 1;
      }
    }
  } else if (warp >= 2) {
    // ---------------- epilogue ----------------
    const int quarter = warp & 3;  // TMEM lanes 32*quarter .. +31
    const int row = quarter * 32 + lane;
    int lt = 0;
    for (int t = blockIdx.x; t < ntiles; t += gridDim.x, ++lt) {
      Tile tl;
      const bool tile_ok = decode_tile<SH>(p, ix, t, tl);
      const int ab = lt & 1;
      const uint32_t acc_phase = (lt >> 1) & 1;
      int ok = 1;
      if (lane == 0) ok = mbar_wait(&acc_full[ab], acc_phase, abort_flag, kWaitNs) ? 1 : 0;
      ok = __shfl_sync(0xffffffffu, ok, 0);
      if (!ok) {
        if (lane == 0) {
          if (!*abort_flag) set_err(p.err, kErrTimeout);
          *abort_flag = 1;
        }
        break;
      }
      tc_fence_after();
      const uint32_t tbase = tmem_base + (static_cast<uint32_t>(quarter * 32) << 16) +
                             static_cast<uint32_t>(ab * BN);
      const bool store = tile_ok && row < tl.rows;
      __nv_bfloat16* orow = (SH && tl.sh ? p.out2 : p.out) +
                            static_cast<int64_t>(tl.row0 + (store ? row : 0)) *
                                (SH && tl.sh ? p.ldo2 : p.ldo);
      if (MODE == kModeScores) {
        float* srow = p.out_f32 + tl.ks * p.split_stride +
                      static_cast<int64_t>(tl.row0 + (store ? row : 0)) * p.ldo;
#pragma unroll 1
        for (int c = 0; c < BN; c += 32) {
          uint32_t v32[32];
          tmem_ld32(tbase + c, v32);
          tmem_ld_wait();
          const int col0 = tl.n * BN + c;
          if (store) {
            if (col0 + 32 <= p.n_valid && (p.ldo & 3) == 0) {
              float4* dst = reinterpret_cast<float4*>(srow + col0);
#pragma unroll
              for (int v = 0; v < 8; ++v)
                dst[v] = make_float4(__uint_as_float(v32[4 * v]), __uint_as_float(v32[4 * v + 1]),
                                     __uint_as_float(v32[4 * v + 2]),
                                     __uint_as_float(v32[4 * v + 3]));
            } else {
#pragma unroll
              for (int i = 0; i < 32; ++i)
                if (col0 + i < p.n_valid) srow[col0 + i] = __uint_as_float(v32[i]);
            }
          }
        }
      } else if (MODE == kModeSwiGLU) {
#pragma unroll 1
        for (int c = 0; c < BN / 2; c += 32) {
          uint32_t g[32], u[32];
          tmem_ld32(tbase + c, g);
          tmem_ld32(tbase + BN / 2 + c, u);
          tmem_ld_wait();
          if (store) {
            uint32_t packed[16];
#pragma unroll
            for (int i = 0; i < 16; ++i) {
              const float g0 = __uint_as_float(g[2 * i]), g1 = __uint_as_float(g[2 * i + 1]);
              const float u0 = __uint_as_float(u[2 * i]), u1 = __uint_as_float(u[2 * i + 1]);
              const float a0 = g0 / (1.0f + __expf(-g0)) * u0;
              const float a1 = g1 / (1.0f + __expf(-g1)) * u1;
              __nv_bfloat162 h2 = __floats2bfloat162_rn(a0, a1);
              packed[i] = *reinterpret_cast<uint32_t*>(&h2);
            }
            uint4* dst = reinterpret_cast<uint4*>(orow + tl.n * (BN / 2) + c);
#pragma unroll
            for (int v = 0; v < 4; ++v)
              dst[v] = make_uint4(packed[4 * v], packed[4 * v + 1], packed[4 * v + 2],
                                  packed[4 * v + 3]);
          }
        }
      } else {
#pragma unroll 1
        for (int c = 0; c < BN; c += 32) {
          uint32_t v32[32];
          tmem_ld32(tbase + c, v32);
          tmem_ld_wait();
          if (store) {
            uint32_t packed[16];
#pragma unroll
            for (int i = 0; i < 16; ++i) {
              __nv_bfloat162 h2 = __floats2bfloat162_rn(__uint_as_float(v32[2 * i]),
                                                        __uint_as_float(v32[2 * i + 1]));
              packed[i] = *reinterpret_cast<uint32_t*>(&h2);
            }
            uint4* dst = reinterpret_cast<uint4*>(orow + tl.n * BN + c);
#pragma unroll
            for (int v = 0; v < 4; ++v)
              dst[v] = make_uint4(packed[4 * v], packed[4 * v + 1], packed[4 * v + 2],
                                  packed[4 * v + 3]);
          }
        }
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive1(smem_addr(&acc_empty[ab]));
    }
  }

  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  if (warp == 1) {
    __syncwarp();
    tmem_dealloc(tmem_base, C::kTmemCols);
  }
  if (p.defer_wait) grid_dep_wait();
}

// The tiles of a dense problem (nullptr: none) that a 1-SM launch carries
// along: `cols` output columns per tile.
void set_shared_problem(KParams& p, const TcGemmArgs* sh, int cols) {
  p.sh_rows = sh != nullptr ? sh->g.dense_rows : 0;
  p.n_tiles2 = sh != nullptr ? sh->n_total / cols : 0;
  p.K2 = sh != nullptr ? sh->K : 0;
  p.out2 = sh != nullptr ? static_cast<__nv_bfloat16*>(sh->out) : nullptr;
  p.ldo2 = sh != nullptr ? sh->ldo : 0;
  p.sh_tiles = (p.sh_rows + p.tile_rows - 1) / p.tile_rows * p.n_tiles2;
}

template <int BN, int MODE, bool SH>
cudaError_t launch_impl(const TcGemmArgs& a, cudaStream_t stream) {
  using C = Cfg<BN>;
  auto kernel = grouped_gemm_kernel<BN, MODE, SH>;
  cudaError_t e = cudaFuncSetAttribute(
      kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, C::kSmemBytes);
  if (e != cudaSuccess) return e;
  KParams p;
  p.K = a.K;
  p.n_tiles = MODE == kModeSwiGLU ? a.n_total / (BN / 2) : a.n_total / BN;
  p.b_rows_per_group = a.b_rows_per_group;
  p.b_up_offset = a.b_up_offset;
  p.g = a.g;
  p.max_mtiles = a.g.offsets ? (a.g.cap_rows + BM - 1) / BM + a.g.E
                             : (a.g.dense_rows + BM - 1) / BM;
  p.out = static_cast<__nv_bfloat16*>(a.out);
  p.ldo = a.ldo;
  p.err = a.err;
  p.mt_prefix = a.g.mt_prefix;
  p.tile_rows = BM;
  p.k_splits = 1;
  p.out_f32 = nullptr;
  p.split_stride = 0;
  p.n_valid = 0;
  p.defer_wait = 0;
  p.early_b = a.early_b ? 1 : 0;
  p.b3d = MODE == kModeSwiGLU && a.b_gate_up_3d ? 1 : 0;
  p.norm_out = nullptr;
  p.gather_perm = nullptr;
  p.gather_x = nullptr;
  p.gather_kmax = 1;
  p.gather_tokens = 0;
  set_shared_problem(p, SH ? a.shared : nullptr, MODE == kModeSwiGLU ? BN / 2 : BN);
  const int64_t max_tiles = static_cast<int64_t>(p.n_tiles) * p.max_mtiles + p.sh_tiles;
  if (max_tiles == 0) return cudaSuccess;
  const int grid = static_cast<int>(max_tiles < a.num_sms ? max_tiles : a.num_sms);
  const TcGemmArgs& sh = SH ? *a.shared : a;
  return launch_pdl(kernel, dim3(grid), dim3(kThreads), C::kSmemBytes, stream, *a.map_a,
                    *a.map_b, *sh.map_a, *sh.map_b, p);
}

// ===========================================================================
// 2-SM variant (cta_group::2) for groups of many rows.
//
// A cluster of two CTAs on one TPC computes a tile of 256 weight rows x up to
// 256 token rows.  The weights are the M operand (M = 256, 128 rows per CTA)
// and the token rows the N operand (each CTA holds half of them), so a tile
// that ends inside its group computes and loads its own rows rounded up to
// 32, not 256: with about 330 rows per expert a third of all MMA work had
// been padding rows (LLaDA-MoE shape, 3270 tokens: gate/up 179 -> 153 us, down
// 88 -> 84; 32768 tokens: gate/up 812 -> 780; LLaDA2.0-mini shape, 65536: 1293
// -> 1255, its K = 512 down GEMM 742 -> 757).
// SwiGLU: CTA rank r holds 64 gate rows and the matching 64 up rows, 16 gate
// then 16 up rows in turn (one box of a 5D map), so gate and up of one output
// meet in one warp's TMEM lanes, 16 apart.  Down: rows n*256 + 128 r of
// W_down.  A 192 KB ring holds 3 stages of two consecutive 64-k blocks, at
// most 32 KB per SM and block.  With gathered rows (SwiGLU,
// TcGemmArgs::gather_perm) four more warps copy the rows straight from the
// token rows (cp.async, the tokens looked up through the pair permutation);
// the rows, tiles and MMA order are those of the copied rows, so the outputs
// are the same bits.  Their two stages in flight do not cover the L2 latency
// (32768 tokens x 64 experts: gate/up 0.78 -> 1.53 ms), so it is opt-in;
// four-row TMA gathers before them took 3.08 ms.  One thread of the leader CTA (rank 0) issues
// tcgen05.mma.cta_group::2; each CTA's TMEM receives its 128 weight rows x
// the tile's token columns (two buffers of 256 columns, allocated
// collectively by one warp per CTA).
// Barriers: both producers arrive (with their byte counts) on the leader's
// "full" barrier and their TMA loads complete on it; MMA completion is
// multicast to both CTAs' "empty" and "accumulator full" barriers; both
// CTAs' epilogue warps arrive on the leader's "accumulator empty" barrier.
// Every barrier wait is bounded, as in the 1-SM kernel.
// ===========================================================================
// warps: 0 TMA producer, 1 MMA issuer (leader), 2-9 epilogue (two warps per
// TMEM lane quarter, each draining half of the accumulator's columns)
constexpr int kThreads2 = 320;
constexpr int kEpiWarps2 = 8;
// SwiGLU: four more warps (10-13) that gather the token rows
constexpr int kGatherWarps = 4;
constexpr int kThreads2Up = kThreads2 + 32 * kGatherWarps;

__device__ __forceinline__ uint32_t cluster_rank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
__device__ __forceinline__ void cluster_sync_all() {
  asm volatile("barrier.cluster.arrive.release.aligned;\n\t"
               "barrier.cluster.wait.acquire.aligned;" ::: "memory");
}
// shared::cta address -> the same variable's shared::cluster address in CTA `rank`
__device__ __forceinline__ uint32_t map_to_rank(uint32_t addr, uint32_t rank) {
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
  return r;
}
// Byte-count announcement on the leader's barrier from the peer CTA: no
// release needed (the bytes themselves arrive by TMA complete_tx).
__device__ __forceinline__ void mbar_expect_tx_cluster(uint32_t cl_bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.relaxed.cluster.shared::cluster.b64 _, [%0], %1;" ::"r"(cl_bar),
               "r"(bytes)
               : "memory");
}
__device__ __forceinline__ void mbar_expect_tx_only_cluster(uint32_t cl_bar, uint32_t bytes) {
  asm volatile("mbarrier.expect_tx.relaxed.cluster.shared::cluster.b64 [%0], %1;" ::"r"(cl_bar),
               "r"(bytes)
               : "memory");
}
// Arrival that orders nothing but the arriving thread's own progress: used to
// hand a TMEM accumulator back once its last tcgen05.ld has completed
// (tcgen05.wait::ld); the epilogue's global stores need not be visible to
// the MMA issuer, so no release fence makes them drain first.
__device__ __forceinline__ void mbar_arrive_cluster_relaxed(uint32_t cl_bar) {
  asm volatile("mbarrier.arrive.relaxed.cluster.shared::cluster.b64 _, [%0];" ::"r"(cl_bar)
               : "memory");
}
// TMA tile load whose completion is counted on a barrier in either CTA of the pair.
__device__ __forceinline__ void tma_load_2d_pair(uint32_t dst, const CUtensorMap* map, int c0,
                                                 int c1, uint32_t cl_bar) {
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes.cta_group::2"
      " [%0], [%1, {%2, %3}], [%4];" ::"r"(dst),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(c0), "r"(c1), "r"(cl_bar)
      : "memory");
}
__device__ __forceinline__ void tma_load_5d_pair(uint32_t dst, const CUtensorMap* map, int c0,
                                                 int c3, int c4, uint32_t cl_bar) {
  asm volatile(
      "cp.async.bulk.tensor.5d.shared::cluster.global.tile.mbarrier::complete_tx::bytes.cta_group::2"
      " [%0], [%1, {%2, %3, %3, %4, %5}], [%6];" ::"r"(dst),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(c0), "r"(0), "r"(c3), "r"(c4), "r"(cl_bar)
      : "memory");
}
__device__ __forceinline__ void tma_load_2d_pair_hint(uint32_t dst, const CUtensorMap* map,
                                                      int c0, int c1, uint32_t cl_bar,
                                                      uint64_t pol) {
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes.cta_group::2"
      ".L2::cache_hint [%0], [%1, {%2, %3}], [%4], %5;" ::"r"(dst),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(c0), "r"(c1), "r"(cl_bar), "l"(pol)
      : "memory");
}
__device__ __forceinline__ void tma_load_5d_pair_hint(uint32_t dst, const CUtensorMap* map,
                                                      int c0, int c3, int c4, uint32_t cl_bar,
                                                      uint64_t pol) {
  asm volatile(
      "cp.async.bulk.tensor.5d.shared::cluster.global.tile.mbarrier::complete_tx::bytes.cta_group::2"
      ".L2::cache_hint [%0], [%1, {%2, %3, %3, %4, %5}], [%6], %7;" ::"r"(dst),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(c0), "r"(0), "r"(c3), "r"(c4), "r"(cl_bar),
      "l"(pol)
      : "memory");
}
// 16 bytes of a gathered row into shared memory, and the hand-over of a stage
// whose rows came that way: the copies have landed (wait_group), are visible
// to the tensor core's reads (proxy fence), and count as one arrival on the
// leader's barrier.
__device__ __forceinline__ void cp_async_row(uint32_t dst, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async_commit_group() {
  asm volatile("cp.async.commit_group;" ::: "memory");
}
template <int N>
__device__ __forceinline__ void cp_async_wait_but() {
  asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}
// mbar_wait that also acquires what the other CTA's warps released
__device__ __forceinline__ bool mbar_wait_cluster(uint64_t* bar, uint32_t parity,
                                                  const volatile int* abort, uint64_t limit_ns) {
  uint64_t t0 = 0;
  for (;;) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}\n"
        : "=r"(ok)
        : "r"(smem_addr(bar)), "r"(parity)
        : "memory");
    if (ok) return true;
    if (abort != nullptr && *abort) return false;
    const uint64_t now = global_ns();
    if (t0 == 0) t0 = now;
    if (now - t0 > limit_ns) return false;
  }
}
__device__ __forceinline__ void mbar_arrive_cluster(uint32_t cl_bar) {
  asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(cl_bar)
               : "memory");
}
__device__ __forceinline__ void mma_bf16_pair(uint32_t tmem_d, uint64_t da, uint64_t db,
                                              uint32_t idesc, uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\n\t}\n" ::"r"(tmem_d),
      "l"(da), "l"(db), "r"(idesc), "r"(accumulate)
      : "memory");
}
// Arrive on the barrier at this shared-memory offset in both CTAs of the pair
// once all prior MMAs of this thread have completed.
__device__ __forceinline__ void mma_commit_pair(uint32_t bar) {
  asm volatile(
      "tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64"
      " [%0], %1;" ::"r"(bar),
      "h"(static_cast<uint16_t>(0x3))
      : "memory");
}
__device__ __forceinline__ void tmem_alloc_pair(uint32_t slot, uint32_t ncols) {
  asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(slot),
               "r"(ncols)
               : "memory");
  asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_dealloc_pair(uint32_t taddr, uint32_t ncols) {
  asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ncols)
               : "memory");
}

struct Cfg2 {
  static constexpr int BN = 256;                 // most token rows of a tile
  static constexpr int KS = 2;                   // 64-k blocks per stage
  static constexpr int kSubBytes = BM * BK * 2;  // 16 KB: one 128-row x 64-k box
  static constexpr int kWBytes = KS * kSubBytes; // this CTA's 128 weight rows
  static constexpr int kXBytes = KS * kSubBytes; // this CTA's half of the token rows, at most
  static constexpr int kStageBytes = kWBytes + kXBytes;
  static constexpr int kStages = kRingBytes / kStageBytes;  // 3
  static constexpr int kTmemCols = 2 * BN;       // two accumulators
  static constexpr int kStagingBytes = 32 * 128; // per epilogue warp: 32 rows x 128 B
  static constexpr int kIndexInts = 384;         // both prefix arrays to E = 191, the first to 383
  static constexpr int kSmemBytes =
      kStages * kStageBytes + 256 + kEpiWarps2 * kStagingBytes + kIndexInts * 4 + 1024;
  static_assert(kSmemBytes <= 227 * 1024, "shared memory of one CTA");
};

// TMA tile store of a shared-memory box (bulk-group completion) and its waits.
__device__ __forceinline__ void tma_store_2d(const CUtensorMap* map, uint32_t src, int c0,
                                             int c1) {
  asm volatile("cp.async.bulk.tensor.2d.global.shared::cta.bulk_group [%0, {%2, %3}], [%1];"
               ::"l"(reinterpret_cast<uint64_t>(map)), "r"(src), "r"(c0), "r"(c1)
               : "memory");
}
__device__ __forceinline__ void bulk_commit() {
  asm volatile("cp.async.bulk.commit_group;" ::: "memory");
}
// all stores but the latest N have read their shared-memory source
template <int N>
__device__ __forceinline__ void bulk_wait_read() {
  asm volatile("cp.async.bulk.wait_group.read %0;" ::"n"(N) : "memory");
}
// ... and completed
__device__ __forceinline__ void bulk_wait_all() {
  asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");
}

// The epilogue's bf16 outputs reach global memory through staging tiles of 32
// token rows x 64 output columns (128 bytes a row, 16-byte chunk j at
// position j ^ (row & 7), the 128-byte swizzle of a TMA box).  The TMEM lanes
// hold output columns, so the tile is transposed on the way: 16x256b loads
// give a thread two neighbouring tokens of a column, the fragment that
// stmatrix stores transposed, 16-byte row segments without bank conflicts
// (packing across lanes with shuffles took a quarter of the shared-memory
// pipe of a K = 512 tile).  Several warps fill one staging tile; a whole tile
// leaves by one TMA store, a partial one by lane stores of whole 128-byte row
// segments.
// 16 TMEM lanes x 32 fp32 columns: r[4 j + i] of thread t is lane t / 4 (+ 8
// for i >= 2), column 8 j + 2 (t mod 4) + (i mod 2).
__device__ __forceinline__ void tmem_ld_frag(uint32_t taddr, uint32_t (&r)[16]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.16x256b.x4.b32 "
      "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
        "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]),
        "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
      : "r"(taddr));
}
// Four 8 x 8 matrices (columns x tokens in the registers) stored transposed:
// thread t gives the address of row t mod 8 of matrix t / 8.
__device__ __forceinline__ void stmatrix_trans(uint32_t addr, uint32_t a, uint32_t b, uint32_t c,
                                               uint32_t d) {
  asm volatile("stmatrix.sync.aligned.m8n8.x4.trans.shared.b16 [%0], {%1, %2, %3, %4};" ::"r"(addr),
               "r"(a), "r"(b), "r"(c), "r"(d)
               : "memory");
}
// address of 16-byte chunk j of row `row` of a staging tile
__device__ __forceinline__ uint32_t stage_addr(uint32_t stg, int row, int j) {
  return stg + static_cast<uint32_t>(row * 128 + ((j ^ (row & 7)) << 4));
}
__device__ __forceinline__ uint32_t pack_bf16(float lo, float hi) {
  __nv_bfloat162 h2 = __floats2bfloat162_rn(lo, hi);
  return *reinterpret_cast<uint32_t*>(&h2);
}
__device__ __forceinline__ uint32_t pack_bf16(uint32_t lo, uint32_t hi) {
  return pack_bf16(__uint_as_float(lo), __uint_as_float(hi));
}
// named barrier of `threads` threads; the second form returns whether v held
// in every one of them
__device__ __forceinline__ void group_sync(int id, int threads) {
  asm volatile("barrier.cta.sync %0, %1;" ::"r"(id), "r"(threads) : "memory");
}
__device__ __forceinline__ bool group_all(int id, int threads, bool v) {
  uint32_t r;
  asm volatile(
      "{\n\t.reg .pred p, q;\n\t"
      "setp.ne.u32 q, %1, 0;\n\t"
      "barrier.cta.red.and.pred p, %2, %3, q;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(r)
      : "r"(v ? 1u : 0u), "r"(id), "r"(threads)
      : "memory");
  return r != 0;
}
// rows [0, nrows) of the staging tile to out rows row_base + r, columns
// col0 .. col0 + 63 (bf16), row stride ldo
__device__ __forceinline__ void flush_staging(const uint8_t* stg, int lane,
                                              __nv_bfloat16* out, int64_t row_base, int ldo,
                                              int col0, int nrows) {
  __syncwarp();
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const int r = 4 * i + (lane >> 3), c = lane & 7;
    const uint4 v = *reinterpret_cast<const uint4*>(stg + r * 128 + ((c ^ (r & 7)) << 4));
    if (r < nrows)
      *reinterpret_cast<uint4*>(out + (row_base + r) * ldo + col0 + 8 * c) = v;
  }
  __syncwarp();
}

// Token columns of a tile of `rows` token rows: the MMA's N, a multiple of 32
// (16 rows per CTA).
__device__ __forceinline__ int tile_cols(int rows) { return (rows + 31) & ~31; }

// ONCE: a weight tile of a group of one m-tile (one reader) is loaded
// evict-first, as in the 1-SM kernel, so that the weight stream leaves the
// gathered rows, activations and outputs in L2 while they fit there (LLaDA-MoE
// shape: 1500 tokens 217 -> 205 us, 1024 tokens 192 -> 182; with 220 MB of
// rows no gain, and the larger code cost 65536 tokens 0.6%).
template <int MODE, bool ONCE>
__global__ void __launch_bounds__(MODE == kModeSwiGLU ? kThreads2Up : kThreads2, 1)
    grouped_gemm_pair_kernel(const __grid_constant__ CUtensorMap map_w,
                             const __grid_constant__ CUtensorMap map_x32,
                             const __grid_constant__ CUtensorMap map_x64,
                             const __grid_constant__ CUtensorMap map_x96,
                             const __grid_constant__ CUtensorMap map_x128,
                             const __grid_constant__ CUtensorMap map_out, const KParams p) {
  using C = Cfg2;
  constexpr int kStages = C::kStages;
  constexpr int BN = C::BN;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>(
      (reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~static_cast<uintptr_t>(1023));
  uint8_t* sw = smem;                         // weight rows
  uint8_t* sx = smem + kStages * C::kWBytes;  // token rows
  // after the ring: the epilogue's staging tiles (1024-byte aligned, the
  // 128-byte swizzle of the output map), the barriers, the tile index
  uint8_t* staging = smem + kStages * C::kStageBytes;
  uint64_t* bars = reinterpret_cast<uint64_t*>(staging + kEpiWarps2 * C::kStagingBytes);
  uint64_t* full = bars;                        // leader's is the one used
  uint64_t* empty = bars + kStages;             // per CTA
  uint64_t* acc_full = bars + 2 * kStages;      // per CTA
  uint64_t* acc_empty = bars + 2 * kStages + 2; // leader's is the one used
  uint64_t* drain = bars + 2 * kStages + 4;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + 2 * kStages + 5);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);

  const int warp = threadIdx.x >> 5;
  const int lane = threadIdx.x & 31;
  const uint32_t rank = cluster_rank();
  const bool leader = rank == 0;
  const int pair = blockIdx.x >> 1;
  const int npairs = gridDim.x >> 1;

  const bool gather = MODE == kModeSwiGLU && p.gather_perm != nullptr;
  if (threadIdx.x == 0) {
    for (int s = 0; s < kStages; ++s) {
      // one expect_tx arrival per CTA of the pair (+ one per gather warp)
      mbar_init(&full[s], gather ? 2 + 2 * kGatherWarps : 2);
      mbar_init(&empty[s], 1);
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(&acc_full[b], 1);
      mbar_init(&acc_empty[b], 2 * kEpiWarps2);  // every epilogue warp of both CTAs
    }
    mbar_init(drain, 1);
    *abort_flag = 0;
    fence_mbar_init();
    prefetch_map(&map_w);
    prefetch_map(&map_x128);
    prefetch_map(&map_out);
  }
  cluster_sync_all();  // barriers of both CTAs initialised; the peer is running
  const int nk = p.K / (BK * C::KS);  // stages per tile
  // this CTA's weight rows of k-block k0 of tile (e, n), counted on fb
  const uint64_t pol_once = ONCE ? l2_policy(kPolFirst) : 0;
  auto load_weights = [&](const Tile& tl, uint32_t dst, int k0, uint32_t fb) {
    if (MODE == kModeSwiGLU) {  // groups of 16 features: 4 per CTA, 8 per tile
      const int blk = tl.n * 8 + static_cast<int>(rank) * 4;
      if (ONCE && tl.mtiles == 1)
        tma_load_5d_pair_hint(dst, &map_w, k0, blk, tl.e, fb, pol_once);
      else
        tma_load_5d_pair(dst, &map_w, k0, blk, tl.e, fb);
    } else {
      const int row = tl.e * p.b_rows_per_group + tl.n * 256 + static_cast<int>(rank) * BM;
      if (ONCE && tl.mtiles == 1)
        tma_load_2d_pair_hint(dst, &map_w, k0, row, fb, pol_once);
      else
        tma_load_2d_pair(dst, &map_w, k0, row, fb);
    }
  };
  // the ring's first weights while the kernel in front still runs, as in the
  // 1-SM kernel; both CTAs' bytes count on the leader's barriers
  int early = 0;  // stages whose weights are on their way (warp 0)
  if (p.early_b && warp == 0) {
    Tile tl;
    if (early_tile<false>(p, pair, tl)) {
      early = nk < kStages ? nk : kStages;
      if (lane == 0) {
        for (int s = 0; s < early; ++s) {
          const uint32_t fb = map_to_rank(smem_addr(&full[s]), 0);
          if (leader) mbar_expect_tx_only(smem_addr(&full[s]), C::kWBytes);
          else mbar_expect_tx_only_cluster(fb, C::kWBytes);
          for (int u = 0; u < C::KS; ++u)
            load_weights(tl, smem_addr(sw + s * C::kWBytes + u * C::kSubBytes),
                         (s * C::KS + u) * BK, fb);
        }
      }
    }
  }
  if (warp == 1) tmem_alloc_pair(smem_addr(tmem_slot), C::kTmemCols);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;
  grid_dep_wait();
  grid_dep_launch();
  const TileIndex ix =
      load_tile_index(p, reinterpret_cast<int32_t*>(reinterpret_cast<uint8_t*>(bars) + 256),
                      C::kIndexInts);
  // tiles are 256 weight rows x up to 256 token rows (both CTAs); mt_prefix
  // counts 256-row tiles
  const int ntiles = total_tiles<false>(p, ix);

  if (warp == 0 && lane == 0) {
    // ---------------- TMA producer (each CTA: its weight rows, its token rows)
    int stage = 0;
    uint32_t phase = 0;
    uint32_t issued_mask = 0, issued_phase = 0;
    bool ok = true;
    for (int t = pair; t < ntiles && ok; t += npairs) {
      Tile tl;
      if (!decode_tile<false>(p, ix, t, tl)) {
        set_err(p.err, kErrIndex);
        *abort_flag = 1;
        break;
      }
      const int half_rows = tile_cols(tl.rows) / 2;  // token rows per CTA, a multiple of 16
      const int xrow = tl.row0 + static_cast<int>(rank) * half_rows;
      // the smallest box that holds them; rows past the tile's end are
      // computed from the next rows or TMA zero fill and never stored
      const int bx = (half_rows + 31) / 32;
      const CUtensorMap* mx = bx == 1 ? &map_x32 : bx == 2 ? &map_x64 : bx == 3 ? &map_x96
                                                                             : &map_x128;
      const uint32_t xbytes = gather ? 0u : static_cast<uint32_t>(C::KS * bx * 32 * 128);
      for (int kb = 0; kb < nk; ++kb) {
        if (!mbar_wait(&empty[stage], phase ^ 1u, abort_flag, kWaitNs)) {
          ok = false;
          break;
        }
        const uint32_t fb = map_to_rank(smem_addr(&full[stage]), 0);
        const bool ahead = early > 0;  // the weights are already on their way
        if (ahead) --early;
        const uint32_t bytes = (ahead ? 0u : static_cast<uint32_t>(C::kWBytes)) + xbytes;
        if (leader)
          mbar_expect_tx(smem_addr(&full[stage]), bytes);
        else
          mbar_expect_tx_cluster(fb, bytes);
        // consecutive k blocks of the same rows back to back
#pragma unroll
        for (int u = 0; u < C::KS; ++u) {
          const int k0 = (kb * C::KS + u) * BK;
          if (!gather)
            tma_load_2d_pair(smem_addr(sx + stage * C::kXBytes + u * C::kSubBytes), mx, k0, xrow,
                             fb);
          if (!ahead)
            load_weights(tl, smem_addr(sw + stage * C::kWBytes + u * C::kSubBytes), k0, fb);
        }
        issued_mask |= 1u << stage;
        issued_phase = (issued_phase & ~(1u << stage)) | (phase << stage);
        if (++stage == kStages) {
          stage = 0;
          phase ^= 1u;
        }
      }
    }
    if (!ok) {
      set_err(p.err, kErrTimeout);
      *abort_flag = 1;
    }
    // early weights of stages that never got their rows: the arrivals that
    // are missing come from both CTAs, and the leader sees the bytes land
    for (int s = 0; s < early; ++s) {
      const int st = (stage + s) % kStages;
      for (int n = 0; n < (gather ? 1 + kGatherWarps : 1); ++n) {
        if (leader) mbar_arrive1(smem_addr(&full[st]));
        else mbar_arrive_cluster_relaxed(map_to_rank(smem_addr(&full[st]), 0));
      }
      if (leader) mbar_wait(&full[st], 0, nullptr, kDrainNs);
    }
    if (*abort_flag && leader) {
      for (int s = 0; s < kStages; ++s)
        if (issued_mask & (1u << s))
          mbar_wait(&full[s], (issued_phase >> s) & 1u, nullptr, kDrainNs);
    }
  } else if (warp == 1 && lane == 0 && leader) {
    // ---------------- MMA issuer (leader CTA only) ----------------
    int stage = 0;
    uint32_t phase = 0;
    int lt = 0;
    bool ok = true, issued_any = false;
    for (int t = pair; t < ntiles && ok; t += npairs, ++lt) {
      const int ab = lt & 1;
      const uint32_t acc_phase = (lt >> 1) & 1;
      Tile tl;
      const int cols = decode_tile<false>(p, ix, t, tl) ? tile_cols(tl.rows) : BN;
      const uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) |
                             (static_cast<uint32_t>(cols >> 3) << 17) |
                             (static_cast<uint32_t>((2 * BM) >> 4) << 24);
      if (!mbar_wait(&acc_empty[ab], acc_phase ^ 1u, abort_flag, kWaitNs)) {
        ok = false;
        break;
      }
      tc_fence_after();
      const uint32_t d_tmem = tmem_base + static_cast<uint32_t>(ab * BN);
      for (int kb = 0; kb < nk; ++kb) {
        if (!(gather ? mbar_wait_cluster(&full[stage], phase, abort_flag, kWaitNs)
                     : mbar_wait(&full[stage], phase, abort_flag, kWaitNs))) {
          ok = false;
          break;
        }
        tc_fence_after();
        const uint32_t w0 = smem_addr(sw + stage * C::kWBytes);
        const uint32_t x0 = smem_addr(sx + stage * C::kXBytes);
#pragma unroll
        for (int u = 0; u < C::KS; ++u)
#pragma unroll
          for (int k = 0; k < BK / UMMA_K; ++k)
            mma_bf16_pair(d_tmem, desc_sw128(w0 + u * C::kSubBytes + k * UMMA_K * 2),
                          desc_sw128(x0 + u * C::kSubBytes + k * UMMA_K * 2), idesc,
                          (kb > 0 || u > 0 || k > 0) ? 1u : 0u);
        issued_any = true;
        mma_commit_pair(smem_addr(&empty[stage]));
        if (++stage == kStages) {
          stage = 0;
          phase ^= 1u;
        }
      }
      if (!ok) break;
      mma_commit_pair(smem_addr(&acc_full[ab]));
    }
    if (!ok) {
      set_err(p.err, kErrTimeout);
      *abort_flag = 1;
    }
    if (*abort_flag && issued_any) {
      mma_commit_pair(smem_addr(drain));
      mbar_wait(drain, 0, nullptr, kDrainNs);
    }
  } else if (MODE == kModeSwiGLU && warp >= 2 + kEpiWarps2) {
    // ---------------- row gather (each CTA: its half of the tile's rows) -------
    // Warp g copies rows 32 g .. +31 of the half, eight lanes per row segment
    // of 128 bytes, into the swizzled stage; lane l handles rows 4 i + l / 8.
    // A stage is handed over once the next one's copies are on their way, so
    // two stages are in flight; the next tile's rows are looked up a tile
    // ahead.
    if (gather) {
      const int g0 = (warp - 2 - kEpiWarps2) * 32 + (lane >> 3);
      const int ch = lane & 7;
      int tok[8], next[8], half_rows = 0, next_half = 0;
      auto look_up = [&](int t, int (&tk)[8], int& hr) {
        Tile tl;
        hr = 0;
        if (t >= ntiles || !decode_tile<false>(p, ix, t, tl)) return;
        hr = tile_cols(tl.rows) / 2;
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          // rows past the tile's end repeat its last row (never stored)
          const int r = min(static_cast<int>(rank) * hr + min(g0 + 4 * i, hr - 1), tl.rows - 1);
          tk[i] = p.gather_perm[tl.row0 + r];
        }
      };
      int stage = 0, prev = -1;
      uint32_t phase = 0;
      bool ok = true;
      auto hand_over = [&](int st) {
        fence_proxy_async_smem();  // this lane's landed copies, before the MMAs read them
        __syncwarp();
        if (lane == 0) mbar_arrive_cluster(map_to_rank(smem_addr(&full[st]), 0));
      };
      look_up(pair, next, next_half);
      for (int t = pair; t < ntiles && ok; t += npairs) {
        half_rows = next_half;
        const __nv_bfloat16* src[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          tok[i] = next[i] >= 0 ? next[i] / p.gather_kmax : -1;
          if (half_rows > 0 && (tok[i] < 0 || tok[i] >= p.gather_tokens)) {
            set_err(p.err, kErrIndex);
            tok[i] = 0;
          }
          src[i] = p.gather_x + static_cast<int64_t>(half_rows > 0 ? tok[i] : 0) * p.K + ch * 8;
        }
        look_up(t + npairs, next, next_half);
        if (half_rows == 0) break;  // inconsistent workspace: the producer aborts
        for (int kb = 0; kb < nk; ++kb) {
          if (!__all_sync(0xffffffffu,
                          mbar_wait(&empty[stage], phase ^ 1u, abort_flag, kWaitNs))) {
            ok = false;
            break;
          }
#pragma unroll
          for (int u = 0; u < C::KS; ++u) {
            const uint32_t dst = smem_addr(sx + stage * C::kXBytes + u * C::kSubBytes);
            const int k0 = (kb * C::KS + u) * BK;
#pragma unroll
            for (int i = 0; i < 8; ++i) {
              const int r = g0 + 4 * i;
              if (r < half_rows)
                cp_async_row(dst + r * 128 + ((ch ^ (r & 7)) << 4), src[i] + k0);
            }
          }
          cp_async_commit_group();
          if (prev >= 0) {
            cp_async_wait_but<1>();
            hand_over(prev);
          }
          prev = stage;
          if (++stage == kStages) {
            stage = 0;
            phase ^= 1u;
          }
        }
      }
      cp_async_wait_but<0>();  // every copy lands before the CTA exits
      if (ok && prev >= 0) hand_over(prev);
    }
  } else if (warp >= 2) {
    // ---------------- epilogue (each CTA: its 128 weight rows) ----------------
    // Warp w drains TMEM lanes 32 (w % 4) .. +31; warps 2-5 take the tile's
    // even 32-column (token) chunks, 6-9 the odd ones.  The warps that fill
    // one staging tile (64 output columns) are a group: SwiGLU all four of a
    // half (16 columns each), down two (32 columns each).  Once a warp's last
    // chunk is in registers it hands the accumulator back (relaxed arrive),
    // and the conversion and stores overlap the next tile's MMAs.
    const int quarter = warp & 3;
    const int half = (warp - 2) >> 2;
    constexpr bool kUp = MODE == kModeSwiGLU;
    constexpr int kGroup = kUp ? 128 : 64;     // threads of a group
    constexpr int kBufs = kUp ? 4 : 2;         // staging tiles of a group
    const int box = kUp ? 0 : quarter >> 1;    // 64-column box of the CTA's columns
    const int bar_id = 1 + (kUp ? half : half * 2 + box);
    const bool lead = kUp ? quarter == 0 : (quarter & 1) == 0;  // the warp that stores
    uint8_t* stg0 = staging + (kUp ? half * 4 : half * 4 + box * 2) * C::kStagingBytes;
    const uint32_t acc_empty_leader0 = map_to_rank(smem_addr(&acc_empty[0]), 0);
    const uint32_t acc_empty_leader1 = map_to_rank(smem_addr(&acc_empty[1]), 0);
    int lt = 0, nbuf = 0;
    for (int t = pair; t < ntiles; t += npairs, ++lt) {
      Tile tl;
      const bool tile_ok = decode_tile<false>(p, ix, t, tl);
      const int ab = lt & 1;
      const uint32_t acc_phase = (lt >> 1) & 1;
      int ok = 1;
      if (lane == 0) ok = mbar_wait(&acc_full[ab], acc_phase, abort_flag, kWaitNs) ? 1 : 0;
      ok = __shfl_sync(0xffffffffu, ok, 0);
      // one decision for the whole group: its barriers below have no limit
      if (!group_all(bar_id, kGroup, ok != 0)) {
        if (lane == 0) {
          if (!*abort_flag) set_err(p.err, kErrTimeout);
          *abort_flag = 1;
        }
        break;
      }
      tc_fence_after();
      const uint32_t tbase = tmem_base + (static_cast<uint32_t>(quarter * 32) << 16) +
                             static_cast<uint32_t>(ab * BN);
      const uint32_t release_bar = ab ? acc_empty_leader1 : acc_empty_leader0;
      auto hand_back = [&]() {
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive_cluster_relaxed(release_bar);
      };
      const int nchunks = tile_ok ? tile_cols(tl.rows) / 32 : 0;
      // first output column of the group's staging tile
      const int col0 = kUp ? tl.n * 128 + static_cast<int>(rank) * 64
                           : tl.n * 256 + static_cast<int>(rank) * BM + box * 64;
      if (half >= nchunks) hand_back();
      for (int c = half; c < nchunks; c += 2) {
        // SwiGLU: gate rows (lanes 0-15) and the matching up rows (16-31) of
        // the same columns and tokens; down: the first and the last 16 columns
        uint32_t v0[16], v1[16];
        tmem_ld_frag(tbase + 32 * c, v0);
        tmem_ld_frag(tbase + (16u << 16) + 32 * c, v1);
        tmem_ld_wait();
        if (c + 2 >= nchunks) hand_back();
        uint8_t* stg = stg0 + (nbuf % kBufs) * C::kStagingBytes;
        const uint32_t stg_s = smem_addr(stg);
        // the store that last used this staging tile has read it
        if (lead && lane == 0) bulk_wait_read<kBufs - 1>();
        group_sync(bar_id, kGroup);
        const int mrow = lane & 7, mat = lane >> 3;  // of the row this thread addresses
        if (kUp) {
          uint32_t w[8];  // [8-token group][8-column block]
#pragma unroll
          for (int i = 0; i < 8; ++i) {
            float act[2];
#pragma unroll
            for (int h = 0; h < 2; ++h) {
              const float gt = __uint_as_float(v0[2 * i + h]), up = __uint_as_float(v1[2 * i + h]);
              act[h] = gt / (1.0f + __expf(-gt)) * up;
            }
            w[i] = pack_bf16(act[0], act[1]);
          }
          // matrices: token groups 2 m and 2 m + 1, column blocks 0 and 1 of each
#pragma unroll
          for (int m = 0; m < 2; ++m)
            stmatrix_trans(stage_addr(stg_s, 8 * (2 * m + (mat >> 1)) + mrow,
                                      quarter * 2 + (mat & 1)),
                           w[4 * m], w[4 * m + 1], w[4 * m + 2], w[4 * m + 3]);
        } else {
          // one token group per store, its four column blocks
#pragma unroll
          for (int j = 0; j < 4; ++j)
            stmatrix_trans(stage_addr(stg_s, 8 * j + mrow, (quarter & 1) * 4 + mat),
                           pack_bf16(v0[4 * j], v0[4 * j + 1]),
                           pack_bf16(v0[4 * j + 2], v0[4 * j + 3]),
                           pack_bf16(v1[4 * j], v1[4 * j + 1]),
                           pack_bf16(v1[4 * j + 2], v1[4 * j + 3]));
        }
        fence_proxy_async_smem();  // the staging writes, before the store reads them
        group_sync(bar_id, kGroup);
        if (lead) {
          const int nrows = min(32, tl.rows - 32 * c);
          if (nrows == 32) {
            if (lane == 0)
              tma_store_2d(&map_out, smem_addr(stg), col0, tl.row0 + 32 * c);
          } else {
            flush_staging(stg, lane, p.out, static_cast<int64_t>(tl.row0) + 32 * c, p.ldo, col0,
                          nrows);
          }
          if (lane == 0) bulk_commit();  // a group per chunk, empty for lane stores
        }
        ++nbuf;
      }
    }
    if (lead && lane == 0) bulk_wait_all();  // every store written before exit
  }

  tc_fence_before();
  __syncthreads();
  cluster_sync_all();  // the pair's MMAs and TMEM reads are done in both CTAs
  tc_fence_after();
  if (warp == 1) {
    __syncwarp();
    tmem_dealloc_pair(tmem_base, C::kTmemCols);
  }
}

template <int MODE, bool ONCE>
cudaError_t launch_pair_impl(const TcGemmArgs& a, cudaStream_t stream) {
  using C = Cfg2;
  auto kernel = grouped_gemm_pair_kernel<MODE, ONCE>;
  cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       C::kSmemBytes);
  if (e != cudaSuccess) return e;
  if (a.K % (BK * C::KS) != 0) return cudaErrorInvalidValue;  // whole stages
  if (a.map_x == nullptr || a.map_out == nullptr) return cudaErrorInvalidValue;
  KParams p;
  p.K = a.K;
  p.n_tiles = MODE == kModeSwiGLU ? a.n_total / 128 : a.n_total / 256;
  p.b_rows_per_group = a.b_rows_per_group;
  p.b_up_offset = a.b_up_offset;
  p.g = a.g;
  p.mt_prefix = a.g.mt2_prefix;
  p.tile_rows = 2 * BM;
  p.max_mtiles = a.g.offsets ? (a.g.cap_rows + p.tile_rows - 1) / p.tile_rows + a.g.E
                             : (a.g.dense_rows + p.tile_rows - 1) / p.tile_rows;
  p.out = static_cast<__nv_bfloat16*>(a.out);
  p.ldo = a.ldo;
  p.err = a.err;
  set_shared_problem(p, nullptr, C::BN);
  p.k_splits = 1;
  p.out_f32 = nullptr;
  p.split_stride = 0;
  p.n_valid = 0;
  p.defer_wait = 0;
  p.early_b = a.early_b ? 1 : 0;
  p.b3d = 0;
  p.norm_out = nullptr;
  p.gather_perm = MODE == kModeSwiGLU ? a.gather_perm : nullptr;
  p.gather_x = static_cast<const __nv_bfloat16*>(a.gather_x);
  p.gather_kmax = a.gather_kmax;
  p.gather_tokens = a.gather_tokens;
  if (p.gather_perm != nullptr && (p.gather_x == nullptr || p.gather_kmax < 1 || p.gather_tokens < 1))
    return cudaErrorInvalidValue;
  const int64_t max_tiles = static_cast<int64_t>(p.n_tiles) * p.max_mtiles;
  if (max_tiles == 0) return cudaSuccess;
  int pairs = a.num_sms / 2;
  if (pairs > max_tiles) pairs = static_cast<int>(max_tiles);
  if (pairs < 1) pairs = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(2 * pairs);
  cfg.blockDim = dim3(MODE == kModeSwiGLU ? kThreads2Up : kThreads2);
  cfg.dynamicSmemBytes = C::kSmemBytes;
  cfg.stream = stream;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = 2;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 2;
  return cudaLaunchKernelEx(&cfg, kernel, *a.map_b, a.map_x[0], a.map_x[1], a.map_x[2],
                            a.map_x[3], *a.map_out, p);
}

}  // namespace

template <int MODE>
cudaError_t launch_any(const TcGemmArgs& a, int bn, cudaStream_t stream) {
  if (a.shared != nullptr)
    return bn == 128 ? launch_impl<128, MODE, true>(a, stream)
                     : launch_impl<256, MODE, true>(a, stream);
  return bn == 128 ? launch_impl<128, MODE, false>(a, stream)
                   : launch_impl<256, MODE, false>(a, stream);
}
cudaError_t launch_swiglu_tc(const TcGemmArgs& a, int bn, cudaStream_t stream) {
  return launch_any<kModeSwiGLU>(a, bn, stream);
}
cudaError_t launch_down_tc(const TcGemmArgs& a, int bn, cudaStream_t stream) {
  return launch_any<kModeDown>(a, bn, stream);
}
template <int BN>
cudaError_t launch_scores_impl(const TcGemmArgs& a, int k_splits, float* out,
                               int64_t split_stride, int n_valid, bool defer_wait,
                               float* row_norms, cudaStream_t stream) {
  using C = Cfg<BN>;
  auto kernel = grouped_gemm_kernel<BN, kModeScores, false>;
  if (a.g.offsets != nullptr || k_splits < 1 || (a.K / BK) % k_splits != 0 ||
      a.K % BK != 0 || n_valid < 1 || (row_norms != nullptr && k_splits != 1))
    return cudaErrorInvalidValue;
  cudaError_t e = cudaFuncSetAttribute(
      kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, C::kSmemBytes);
  if (e != cudaSuccess) return e;
  KParams p{};
  p.K = a.K;
  p.n_tiles = (n_valid + BN - 1) / BN;
  p.b_rows_per_group = 0;
  p.b_up_offset = 0;
  p.g = a.g;
  p.max_mtiles = (a.g.dense_rows + BM - 1) / BM;
  p.out = nullptr;
  p.ldo = a.ldo;
  p.err = a.err;
  p.mt_prefix = nullptr;
  p.tile_rows = BM;
  p.k_splits = k_splits;
  p.out_f32 = out;
  p.split_stride = split_stride;
  p.n_valid = n_valid;
  p.defer_wait = defer_wait ? 1 : 0;
  p.b3d = 0;
  p.norm_out = row_norms;
  const int64_t max_tiles = static_cast<int64_t>(p.n_tiles) * p.max_mtiles * k_splits;
  if (max_tiles == 0) return cudaSuccess;
  const int grid = static_cast<int>(max_tiles < a.num_sms ? max_tiles : a.num_sms);
  return launch_pdl(kernel, dim3(grid), dim3(kThreadsScores), C::kSmemBytes, stream,
                    *a.map_a, *a.map_b, *a.map_a, *a.map_b, p);
}

// SwiGLU loads gate and up halves as two boxes of bn/2 rows; down loads one
// box of bn rows.
int tc_b_box_rows(bool swiglu, int bn) { return swiglu ? bn / 2 : bn; }

cudaError_t launch_scores_tc(const TcGemmArgs& a, int bn, int k_splits, float* out,
                             int64_t split_stride, int n_valid, bool defer_wait,
                             cudaStream_t stream, float* row_norms) {
  if (bn == 64)
    return launch_scores_impl<64>(a, k_splits, out, split_stride, n_valid, defer_wait,
                                  row_norms, stream);
  if (bn == 128)
    return launch_scores_impl<128>(a, k_splits, out, split_stride, n_valid, defer_wait,
                                   row_norms, stream);
  if (bn == 256)
    return launch_scores_impl<256>(a, k_splits, out, split_stride, n_valid, defer_wait,
                                   row_norms, stream);
  return cudaErrorInvalidValue;
}

cudaError_t launch_swiglu_tc_pair(const TcGemmArgs& a, cudaStream_t stream) {
  return a.once ? launch_pair_impl<kModeSwiGLU, true>(a, stream)
                : launch_pair_impl<kModeSwiGLU, false>(a, stream);
}
cudaError_t launch_down_tc_pair(const TcGemmArgs& a, cudaStream_t stream) {
  return a.once ? launch_pair_impl<kModeDown, true>(a, stream)
                : launch_pair_impl<kModeDown, false>(a, stream);
}
// Output columns of one tile.
int tc_n_granule(bool swiglu, int bn) { return swiglu ? bn / 2 : bn; }

// Tile width: 256 when there are enough tiles to fill every SM several
// times over (large M per expert: fewer re-reads of the A rows per output),
// else 128 so that the persistent CTAs get more, smaller tiles and the last
// partial wave is short (small M: the GEMM is a weight stream).
int tc_pick_bn(bool swiglu, int n_total, int64_t mtiles_est, int num_sms) {
  const int g256 = tc_n_granule(swiglu, 256);
  const int g128 = tc_n_granule(swiglu, 128);
  if (n_total % g256 != 0) return (n_total % g128 == 0) ? 128 : 0;
  const int64_t tiles256 = static_cast<int64_t>(n_total / g256) * mtiles_est;
  return tiles256 >= 8LL * num_sms ? 256 : 128;
}

}  // namespace rx
