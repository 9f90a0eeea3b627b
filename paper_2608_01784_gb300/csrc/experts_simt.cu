// experts_simt.cu — SwiGLU expert GEMMs over ragged per-expert row groups on
// the SIMT pipes (fp32 path, and a bf16 cross-check of the tensor-core path).
//
// For the pair rows of expert e (rows [offsets[e], offsets[e+1]) of the
// gathered input), Eq. 2's expert E_e is
//   act[r, c] = silu(x_r . Wg[e, c]) * (x_r . Wu[e, c])      c < inter
//   y[r, n]   = act_r . Wd[e, n]                              n < d
//
// Bound: the fp32 FMA pipe (6 d inter FLOPs per pair at about 75 TFLOP/s).
// One warp per output row and column, lanes over k, re-read both operands
// from L1 / L2 for every product and ran at 6 TFLOP/s (about 2000 pairs, d =
// 1024, inter = 512: gate/up 650 us, down 514 us; now 138 and 76 us, of which
// a third is the last of two waves of 64 x 128 tiles); here a CTA computes a
// BM x BN tile with register tiles of TM x TN outputs per thread, so a k step
// costs TM + TN shared-memory values for TM TN fmas.  SK groups of 128
// threads each take 1 / SK of every k block (tiles of short batches get more
// warps).  No fp32 chain is longer than 8 or 16 products: a running sum then
// joins the total, and the rounding of that addition is carried into the next
// running sum (Kahan's compensation), so the result rounds no more than 32
// lanes' partial sums did.
#include "common.cuh"
#include "internal.h"

namespace rx {
namespace {

constexpr int kGroupThreads = 128;  // 8 row x 16 column threads

template <int TM_, int TN_, int SK_, int BK_, int RUN_>
struct Tile {
  static constexpr int TM = TM_, TN = TN_, SK = SK_, BK = BK_;
  static constexpr int BM = 8 * TM, BN = 16 * TN, NT = SK * kGroupThreads;
  static constexpr int KG = BK / SK;  // k of a block that one group takes
  static constexpr int kRun = RUN_;   // products per running sum
  static constexpr int kStage = (BM + BN) * BK;  // floats
  static constexpr int kTiles = 2 * kStage;
  static constexpr int kReduce = (SK - 1) * kGroupThreads * TM * TN;
  static constexpr int kSmemFloats = kTiles > kReduce ? kTiles : kReduce;
  static constexpr int kALoads = BM * BK / 4 / NT > 0 ? BM * BK / 4 / NT : 1;
  static constexpr int kBLoads = BN * BK / 4 / NT;
  static_assert(BK % 16 == 0 && KG % kRun == 0 && KG % 4 == 0 && BN * BK / 4 % NT == 0, "tile shape");
  static_assert(kSmemFloats * 4 <= 48 * 1024, "static shared memory");
  static_assert(kTileM % BM == 0, "whole tiles in a 128-row group tile");
};
using TileLarge = Tile<8, 8, 2, 32, 16>;  // 64 x 128 outputs, 256 threads
using TileSmall = Tile<2, 4, 4, 64, 8>;  // 16 x 64 outputs, 512 threads

template <int V>
struct Int {
  static constexpr int value = V;
};

// 4 consecutive elements, widened to fp32
__device__ __forceinline__ float4 ld4(const float* p) {
  return __ldg(reinterpret_cast<const float4*>(p));
}
__device__ __forceinline__ float4 ld4(const __nv_bfloat16* p) {
  const uint2 v = __ldg(reinterpret_cast<const uint2*>(p));
  return make_float4(__uint_as_float(v.x << 16), __uint_as_float(v.x & 0xffff0000u),
                     __uint_as_float(v.y << 16), __uint_as_float(v.y & 0xffff0000u));
}
// N consecutive outputs (N = 2 or 4)
template <int N>
__device__ __forceinline__ void st(float* p, const float* v) {
  if constexpr (N == 4)
    *reinterpret_cast<float4*>(p) = make_float4(v[0], v[1], v[2], v[3]);
  else
    *reinterpret_cast<float2*>(p) = make_float2(v[0], v[1]);
}
template <int N>
__device__ __forceinline__ void st(__nv_bfloat16* p, const float* v) {
#pragma unroll
  for (int i = 0; i < N; i += 2)
    *reinterpret_cast<__nv_bfloat162*>(p + i) = __floats2bfloat162_rn(v[i], v[i + 1]);
}
template <int N>
__device__ __forceinline__ void lds(const float* p, float* v) {
  if constexpr (N == 4) {
    const float4 q = *reinterpret_cast<const float4*>(p);
    v[0] = q.x; v[1] = q.y; v[2] = q.z; v[3] = q.w;
  } else {
    const float2 q = *reinterpret_cast<const float2*>(p);
    v[0] = q.x; v[1] = q.y;
  }
}

// Two fp32 values in one 64-bit register: packed fma and add round each
// half as the scalar operation does and take half the issue slots.
using f32x2 = unsigned long long;
__device__ __forceinline__ f32x2 pack2(float lo, float hi) {
  f32x2 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
  return r;
}
__device__ __forceinline__ void unpack2(f32x2 v, float& lo, float& hi) {
  asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v));
}
__device__ __forceinline__ f32x2 fma2(f32x2 a, f32x2 b, f32x2 c) {
  f32x2 r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
  return r;
}
__device__ __forceinline__ f32x2 add2(f32x2 a, f32x2 b) {
  f32x2 r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}

__device__ __forceinline__ f32x2 sub2(f32x2 a, f32x2 b) {  // a - b: -1 * b is exact
  return fma2(b, pack2(-1.0f, -1.0f), a);
}

// Sums without the carry, for outputs that came out NaN.  By whole warps, for
// each lane with `need` in turn: x . w over K, or (w == nullptr) a NaN if x
// holds one, else 0; the lanes split k, so that their loads are whole lines.
// (1024 tokens, 16 experts of 512, d = 1024, 346 us: a NaN in every row 4920 ->
// 348 us, an infinity in one 545 -> 392, in a gate row of every expert 2256 ->
// 1264, against sums by the threads that hold the outputs.)
template <typename Te>
__device__ __noinline__ float dot_again(const Te* x, const Te* w, int K, bool need) {
  const int lane = threadIdx.x & 31;
  float mine = 0.f;
  for (uint32_t left = __ballot_sync(0xffffffffu, need); left != 0u; left &= left - 1u) {
    const int src = __ffs(left) - 1;
    const Te* xs = reinterpret_cast<const Te*>(
        __shfl_sync(0xffffffffu, reinterpret_cast<unsigned long long>(x), src));
    const Te* ws = reinterpret_cast<const Te*>(
        __shfl_sync(0xffffffffu, reinterpret_cast<unsigned long long>(w), src));
    float s = 0.f;
    for (int k = 4 * lane; k < K; k += 128) {
      const float4 a = ld4(xs + k);
      if (ws == nullptr) {
        if (a.x != a.x || a.y != a.y || a.z != a.z || a.w != a.w) s = a.x + a.y + a.z + a.w;
        continue;
      }
      const float4 b = ld4(ws + k);
      s = __fmaf_rn(a.w, b.w, __fmaf_rn(a.z, b.z, __fmaf_rn(a.y, b.y, __fmaf_rn(a.x, b.x, s))));
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (lane == src) mine = s;
  }
  return mine;
}

// The same by one thread, for tiles of 8 outputs a thread: the warps' sums cost
// the loop of those tiles, short of registers, 1 to 2%.  A partial sum that is
// a NaN stays one (300 tokens, 189 us: a NaN in every row 1358 -> 159 us, an
// infinity in one 290 -> 316).
template <typename Te>
__device__ __noinline__ float dot_again_alone(const Te* x, const Te* w, int K) {
  float s = 0.f;
  for (int k = 0; k < K && s == s; k += 4) {
    const float4 a = ld4(x + k), b = ld4(w + k);
    s = __fmaf_rn(a.w, b.w, __fmaf_rn(a.z, b.z, __fmaf_rn(a.y, b.y, __fmaf_rn(a.x, b.x, s))));
  }
  return s;
}

// Group of 128-row tile mt: the expert whose tile prefix holds it (a 32-ary
// search, every warp for itself); -1 when there is none.
__device__ __forceinline__ int group_of_tile(const GroupRows& g, int mt) {
  const int lane = threadIdx.x & 31;
  int lo = 0, n = g.E;
  while (n > 1) {
    const int step = (n + 31) / 32;
    const int i = lo + lane * step;
    const bool below = lane * step < n && g.mt_prefix[i] <= mt;
    const int hit = 31 - __clz(__ballot_sync(0xffffffffu, below) | 1u);
    lo += hit * step;
    n = min(step, n - hit * step);
  }
  return g.mt_prefix[lo] <= mt && mt < g.mt_prefix[lo + 1] ? lo : -1;
}

// MODE 0: act = silu(x Wg^T) * (x Wu^T), BN / 2 columns per tile (the first
// half of the B tile holds gate rows, the second the matching up rows);
// MODE 1: y = x W^T, BN columns per tile.  x [rows, K], w rows of length K.
// PER_SM: CTAs per SM that the registers allow.
template <typename Te, typename C, int MODE, int PER_SM>
__global__ void __launch_bounds__(C::NT, PER_SM)
    gemm_simt_kernel(const Te* __restrict__ x, const Te* __restrict__ w, int K, int n_total,
                     GroupRows g, Te* __restrict__ out) {
  constexpr int TM = C::TM, TN = C::TN, BM = C::BM, BN = C::BN, BK = C::BK, HN = TN / 2;
  constexpr int kCols = MODE == 0 ? BN / 2 : BN;  // output columns of a tile
  __shared__ __align__(16) float smem[C::kSmemFloats];
  grid_dep_wait();
  grid_dep_launch();
  constexpr int kSub = kTileM / BM;
  const int mt = blockIdx.x / kSub, sub = blockIdx.x % kSub;
  const int n0 = blockIdx.y * kCols;
  int e = 0, row0, rows;
  if (g.offsets != nullptr) {
    e = group_of_tile(g, mt);
    if (e < 0) return;
    const int first = g.offsets[e], last = g.offsets[e + 1];
    // values of an inconsistent workspace can be any: no row outside [0, cap)
    const int64_t at = static_cast<int64_t>(first) +
                       (static_cast<int64_t>(mt) - g.mt_prefix[e]) * kTileM + sub * BM;
    if (first < 0 || last > g.cap_rows || at >= last) return;
    row0 = static_cast<int>(at);
    rows = min(BM, last - row0);
  } else {
    row0 = mt * kTileM + sub * BM;
    rows = min(BM, g.dense_rows - row0);
  }
  if (rows <= 0) return;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int grp = tid / kGroupThreads, gw = warp & 3;  // k group, warp within it
  const int ty = (gw & 1) * 4 + (lane >> 3), tx = (gw >> 1) * 8 + (lane & 7);
  const int64_t wrows = MODE == 0 ? 2 * static_cast<int64_t>(n_total) : n_total;
  const Te* we = w + static_cast<int64_t>(e) * wrows * K;
  const Te* xe = x + static_cast<int64_t>(row0) * K;

  // Shared tiles are k-major: row k holds BM (BN) values, value m at m ^ (8 q)
  // with q = k / 4 mod 4 (mod 2 for 16-row tiles): a warp's transposing store
  // (8 rows x 4 vectors of 4 k) then spreads over the banks, and groups of 8
  // stay whole for the vector reads.
  constexpr int kAMask = BM >= 32 ? 3 : 1;
  // vector v of a tile: 8 rows x 4 vectors per warp
  auto place = [](int v, int nrow, int& r, int& kv) {
    const int u = v >> 5, l = v & 31, rb = nrow / 8;
    r = (u % rb) * 8 + (l >> 2);
    kv = (u / rb) * 4 + (l & 3);
  };
  float4 ra[2][C::kALoads], rb[2][C::kBLoads];  // the next two blocks' loads
  auto load = [&](int k0, auto set_c) {
    constexpr int set = decltype(set_c)::value;
#pragma unroll
    for (int i = 0; i < C::kALoads; ++i) {
      int r, kv;
      const int v = tid + i * C::NT;
      place(v, BM, r, kv);
      ra[set][i] = v < BM * BK / 4 && r < rows
                  ? ld4(xe + static_cast<int64_t>(r) * K + k0 + 4 * kv)
                  : make_float4(0.f, 0.f, 0.f, 0.f);
    }
#pragma unroll
    for (int i = 0; i < C::kBLoads; ++i) {
      int r, kv;
      place(tid + i * C::NT, BN, r, kv);
      // weight row of B-tile row r (columns past n_total: zero)
      const int col = MODE == 0 ? n0 + r % (BN / 2) : n0 + r;
      const int wr = MODE == 0 && r >= BN / 2 ? n_total + col : col;
      rb[set][i] = col < n_total ? ld4(we + static_cast<int64_t>(wr) * K + k0 + 4 * kv)
                            : make_float4(0.f, 0.f, 0.f, 0.f);
    }
  };
  auto store = [&](auto set_c) {  // block kb sits in register set and buffer kb mod 2
    constexpr int set = decltype(set_c)::value;
    float* a = smem + set * C::kStage;
    float* b = a + BM * BK;
#pragma unroll
    for (int i = 0; i < C::kALoads; ++i) {
      int r, kv;
      const int v = tid + i * C::NT;
      place(v, BM, r, kv);
      if (v < BM * BK / 4) {
        const int m = r ^ (8 * (kv & kAMask));
        a[(4 * kv) * BM + m] = ra[set][i].x;
        a[(4 * kv + 1) * BM + m] = ra[set][i].y;
        a[(4 * kv + 2) * BM + m] = ra[set][i].z;
        a[(4 * kv + 3) * BM + m] = ra[set][i].w;
      }
    }
#pragma unroll
    for (int i = 0; i < C::kBLoads; ++i) {
      int r, kv;
      place(tid + i * C::NT, BN, r, kv);
      const int n = r ^ (8 * (kv & 3));
      b[(4 * kv) * BN + n] = rb[set][i].x;
      b[(4 * kv + 1) * BN + n] = rb[set][i].y;
      b[(4 * kv + 2) * BN + n] = rb[set][i].z;
      b[(4 * kv + 3) * BN + n] = rb[set][i].w;
    }
  };

  f32x2 acc2[TM][HN], run[TM][HN];  // pairs of adjacent columns: total, running sum
  const int nkb = K / BK;
  // Block kb: its loads were issued two blocks ago (one block's fmas do not
  // cover an L2 miss), the next block's values go to the other buffer, which
  // was last read in block kb - 1, before its barrier.
  auto block = [&](int kb, auto set_c) {
    constexpr int set = decltype(set_c)::value;
    using Other = Int<1 - set>;
    if (kb + 2 < nkb) load((kb + 2) * BK, set_c);
    const float* a = smem + set * C::kStage;
    const float* b = a + BM * BK;
#pragma unroll
    for (int kk = 0; kk < C::KG; ++kk) {
      const int k = grp * C::KG + kk;
      const int q = grp * (C::KG / 4) + kk / 4;  // k / 4
      float av[TM], bv[TN];
      const float* ar = a + k * BM + ((ty * TM) ^ (8 * (q & kAMask)));
      if constexpr (TM == 8) {
        lds<4>(ar, av);
        lds<4>(ar + 4, av + 4);
      } else {
        lds<TM>(ar, av);
      }
      lds<HN>(b + k * BN + ((tx * HN) ^ (8 * (q & 3))), bv);
      lds<HN>(b + k * BN + ((BN / 2 + tx * HN) ^ (8 * (q & 3))), bv + HN);
      f32x2 b2[HN];
#pragma unroll
      for (int j = 0; j < HN; ++j) b2[j] = pack2(bv[2 * j], bv[2 * j + 1]);
#pragma unroll
      for (int i = 0; i < TM; ++i) {
        const f32x2 a2 = pack2(av[i], av[i]);
#pragma unroll
        for (int j = 0; j < HN; ++j)
          run[i][j] = fma2(a2, b2[j], run[i][j]);
      }
      // the running sum joins the total; what that addition rounds off
      // starts the next running sum
      if ((kk + 1) % C::kRun == 0) {
#pragma unroll
        for (int i = 0; i < TM; ++i)
#pragma unroll
          for (int j = 0; j < HN; ++j) {
            const f32x2 s = add2(acc2[i][j], run[i][j]);
            run[i][j] = sub2(run[i][j], sub2(s, acc2[i][j]));
            acc2[i][j] = s;
          }
      }
    }
    if (kb + 1 < nkb) store(Other{});
    __syncthreads();
  };
#pragma unroll
  for (int i = 0; i < TM; ++i)
#pragma unroll
    for (int j = 0; j < HN; ++j) acc2[i][j] = run[i][j] = 0ull;
  load(0, Int<0>{});
  if (nkb > 1) load(BK, Int<1>{});
  store(Int<0>{});
  __syncthreads();
  for (int kb = 0; kb < nkb; kb += 2) {
    block(kb, Int<0>{});
    if (kb + 1 < nkb) block(kb + 1, Int<1>{});
  }
  float acc[TM][TN];
#pragma unroll
  for (int i = 0; i < TM; ++i)
#pragma unroll
    for (int j = 0; j < HN; ++j) unpack2(acc2[i][j], acc[i][2 * j], acc[i][2 * j + 1]);
  // the groups' sums, in group order
  float* red = smem;
  if (grp > 0) {
    float* my = red + ((grp - 1) * kGroupThreads + (tid % kGroupThreads));
#pragma unroll
    for (int i = 0; i < TM; ++i)
#pragma unroll
      for (int j = 0; j < TN; ++j)
        my[(i * TN + j) * (C::SK - 1) * kGroupThreads] = acc[i][j];
  }
  __syncthreads();
  if (grp > 0) return;
#pragma unroll
  for (int i = 0; i < TM; ++i)
#pragma unroll
    for (int j = 0; j < TN; ++j)
#pragma unroll
      for (int s = 0; s < C::SK - 1; ++s)
        acc[i][j] += red[(i * TN + j) * (C::SK - 1) * kGroupThreads + s * kGroupThreads + tid];
#pragma unroll
  for (int i = 0; i < TM; ++i) {
    const int r = ty * TM + i;
    // what rounds off an infinite sum is a NaN, so a NaN may stand for an
    // infinity: such an output is summed again without the carry
    if constexpr (TM * TN > 8) {
      bool again = false;
#pragma unroll
      for (int j = 0; j < TN; ++j) again |= acc[i][j] != acc[i][j];
      again &= r < rows;
      if (__any_sync(0xffffffffu, again)) {
        const Te* xr = xe + static_cast<int64_t>(r) * K;
        const float has = dot_again<Te>(xr, nullptr, K, again && (lane & 7) == 0);
        again &= __shfl_sync(0xffffffffu, has, lane & 24) == 0.f;  // no NaN in the row
#pragma unroll
        for (int j = 0; j < TN; ++j) {
          const int c = n0 + tx * HN + (j % HN) + (MODE == 1 && j >= HN ? BN / 2 : 0);
          const int64_t wr = MODE == 0 && j >= HN ? static_cast<int64_t>(n_total) + c : c;
          const bool need = again && acc[i][j] != acc[i][j] && c < n_total;
          const float v = dot_again<Te>(xr, we + wr * K, K, need);
          if (need) acc[i][j] = v;
        }
      }
    } else if (r < rows) {
#pragma unroll
      for (int j = 0; j < TN; ++j) {
        const int c = n0 + tx * HN + (j % HN) + (MODE == 1 && j >= HN ? BN / 2 : 0);
        const int64_t wr = MODE == 0 && j >= HN ? static_cast<int64_t>(n_total) + c : c;
        if (acc[i][j] != acc[i][j] && c < n_total)
          acc[i][j] = dot_again_alone(xe + static_cast<int64_t>(r) * K, we + wr * K, K);
      }
    }
    if (r >= rows) continue;
    Te* orow = out + static_cast<int64_t>(row0 + r) * n_total;
    if (MODE == 0) {
      float v[HN];
#pragma unroll
      for (int j = 0; j < HN; ++j) {
        const float s = acc[i][j] / (1.0f + expf(-acc[i][j]));
        v[j] = s * acc[i][HN + j];
      }
      if (n0 + tx * HN < n_total) st<HN>(orow + n0 + tx * HN, v);
    } else {
      const int c0 = n0 + tx * HN, c1 = c0 + BN / 2;
      if (c0 < n_total) st<HN>(orow + c0, acc[i]);
      if (c1 < n_total) st<HN>(orow + c1, acc[i] + HN);
    }
  }
}

// A few rows per expert: the weights are the work, each row of them read for
// these rows, and one warp per output row and column streams them best.
// The warp's lanes split the reduction index in 8-element vectors and a
// butterfly adds the 32 partials.
constexpr int kDotRows = 8;   // one warp per row
constexpr int kDotCols = 16;  // columns per CTA (loop inside the warp)

__device__ __forceinline__ int group_of(const GroupRows& g, int r) {
  if (g.offsets == nullptr) return 0;
  int lo = 0, hi = g.E;  // offsets[lo] <= r < offsets[hi]
  while (hi - lo > 1) {
    const int mid = (lo + hi) >> 1;
    if (g.offsets[mid] <= r) lo = mid; else hi = mid;
  }
  return lo;
}

__device__ __forceinline__ int rows_of(const GroupRows& g) {
  if (g.offsets == nullptr) return g.dense_rows;
  const int n = g.totals[0];
  return n < g.cap_rows ? n : g.cap_rows;
}

__device__ __forceinline__ float warp_sum(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

template <typename Te>
__global__ void __launch_bounds__(kDotRows * 32)
    swiglu_dot_kernel(const Te* __restrict__ x, const Te* __restrict__ wgu,
                       int d, int inter, GroupRows g, Te* __restrict__ act) {
  grid_dep_wait();
  grid_dep_launch();
  const int lane = threadIdx.x & 31;
  const int r = blockIdx.x * kDotRows + (threadIdx.x >> 5);
  if (r >= rows_of(g)) return;
  const int e = group_of(g, r);
  const Te* xr = x + static_cast<int64_t>(r) * d;
  const Te* wg_e = wgu + static_cast<int64_t>(e) * 2 * inter * d;
  for (int cc = 0; cc < kDotCols; ++cc) {
    const int c = blockIdx.y * kDotCols + cc;
    if (c >= inter) break;
    const Te* wg = wg_e + static_cast<int64_t>(c) * d;
    const Te* wu = wg_e + static_cast<int64_t>(inter + c) * d;
    float ga = 0.f, ua = 0.f;
    for (int k = lane * 8; k < d; k += 256) {
      float xv[8], gv[8], uv[8];
      load8(xr + k, xv);
      load8(wg + k, gv);
      load8(wu + k, uv);
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        ga = __fmaf_rn(xv[i], gv[i], ga);
        ua = __fmaf_rn(xv[i], uv[i], ua);
      }
    }
    ga = warp_sum(ga);
    ua = warp_sum(ua);
    if (lane == 0) {
      const float s = ga / (1.0f + expf(-ga));
      act[static_cast<int64_t>(r) * inter + c] = from_f32<Te>(s * ua);
    }
  }
}

template <typename Te>
__global__ void __launch_bounds__(kDotRows * 32)
    down_dot_kernel(const Te* __restrict__ act, const Te* __restrict__ wd,
                     int d, int inter, GroupRows g, Te* __restrict__ y) {
  grid_dep_wait();
  grid_dep_launch();
  const int lane = threadIdx.x & 31;
  const int r = blockIdx.x * kDotRows + (threadIdx.x >> 5);
  if (r >= rows_of(g)) return;
  const int e = group_of(g, r);
  const Te* ar = act + static_cast<int64_t>(r) * inter;
  const Te* wd_e = wd + static_cast<int64_t>(e) * d * inter;
  for (int nn = 0; nn < kDotCols; ++nn) {
    const int n = blockIdx.y * kDotCols + nn;
    if (n >= d) break;
    const Te* wrow = wd_e + static_cast<int64_t>(n) * inter;
    float acc = 0.f;
    for (int c = lane * 8; c < inter; c += 256) {
      float av[8], wv[8];
      load8(ar + c, av);
      load8(wrow + c, wv);
#pragma unroll
      for (int i = 0; i < 8; ++i) acc = __fmaf_rn(av[i], wv[i], acc);
    }
    acc = warp_sum(acc);
    if (lane == 0) y[static_cast<int64_t>(r) * d + n] = from_f32<Te>(acc);
  }
}

template <typename Te, typename C, int MODE, int PER_SM>
cudaError_t launch_tile(const Te* x, const Te* w, int K, int n_total, const GroupRows& g,
                        Te* out, cudaStream_t stream) {
  const int cols = MODE == 0 ? C::BN / 2 : C::BN;
  const int64_t mt = g.offsets != nullptr
                         ? (static_cast<int64_t>(g.cap_rows) + kTileM - 1) / kTileM + g.E
                         : (static_cast<int64_t>(g.dense_rows) + kTileM - 1) / kTileM;
  const dim3 grid(static_cast<unsigned>(mt * (kTileM / C::BM)), (n_total + cols - 1) / cols);
  return launch_pdl(gemm_simt_kernel<Te, C, MODE, PER_SM>, grid, dim3(C::NT), 0, stream, x, w, K,
                    n_total, g, out);
}

template <typename Te, int MODE>
cudaError_t launch_mode(const void* x, const void* w, int K, int n_total, const GroupRows& g,
                        void* out, int num_sms, cudaStream_t stream) {
  // Large tiles once the expected pairs (half of the row capacity) fill half
  // of one per group and the SMs with them; below that the small tiles' extra
  // CTAs and fewer padding rows win (48 tokens, 32 experts of 512, d = 1024:
  // 247 us with large tiles, 155 with small).  Small tiles run two CTAs per
  // SM when there are more than the SMs take at a time (200 tokens, 16 experts
  // of 512, d = 1024: 180 -> 151 us), else one with twice the registers (tiny
  // layer 35 -> 30 us).
  const int64_t groups = g.offsets != nullptr ? g.E : 1;
  const int64_t rows = (g.offsets != nullptr ? g.cap_rows / 2 : g.dense_rows) / groups;
  auto tiles = [&](int bm, int cols) {
    return groups * ((rows + bm - 1) / bm > 0 ? (rows + bm - 1) / bm : 1) *
           ((n_total + cols - 1) / cols);
  };
  constexpr int kDiv = MODE == 0 ? 2 : 1;  // output columns of a tile: BN / kDiv
  const Te* xt = static_cast<const Te*>(x);
  const Te* wt = static_cast<const Te*>(w);
  Te* ot = static_cast<Te*>(out);
  // A few expected rows per group of enough weights: the dot kernels.  fp32 below
  // two rows, where the small tiles are more than the SMs; bf16, half of whose
  // weight bytes make the dots that much cheaper while the tiles' cost stays, up
  // to six, from 2^20 weights of a projection on.  Layer, dot kernels against
  // tiles, mean over 24 to 40 shapes (4 to 128 experts, d 256 to 2048, 128 to
  // 512 wide), with as many rows as expected and with twice as many:
  //   fp32, many tiles   1.5 rows -22%, -13%   2 -18, -3   2.5 -13, +9   3 -6, +26
  //   bf16, many tiles   4 rows -32%, -4%   5 -27, +9   6 -15, +26   8 -3, +25
  //   bf16, few tiles    4 rows -7, -1   5 -3, +3 (2^19 weights +5, 2^18 +22)   6 -1, +8
  // (at two rows the fp32 tiles' error against 64 bits is 3% smaller).
  const bool dots = sizeof(Te) == 2
                        ? g.cap_rows <= 12 * groups &&
                              groups * n_total * static_cast<int64_t>(K) >= (1 << 20)
                        : g.cap_rows < 4 * groups &&
                              tiles(TileSmall::BM, TileSmall::BN / kDiv) > num_sms;
  if (g.offsets != nullptr && dots) {
    const dim3 grid((g.cap_rows + kDotRows - 1) / kDotRows, (n_total + kDotCols - 1) / kDotCols);
    if constexpr (MODE == 0)
      return launch_pdl(swiglu_dot_kernel<Te>, grid, dim3(kDotRows * 32), 0, stream, xt, wt, K,
                        n_total, g, ot);
    else
      return launch_pdl(down_dot_kernel<Te>, grid, dim3(kDotRows * 32), 0, stream, xt, wt, n_total,
                        K, g, ot);
  }
  if (rows >= TileLarge::BM / 2 && tiles(TileLarge::BM, TileLarge::BN / kDiv) >= num_sms)
    return launch_tile<Te, TileLarge, MODE, 1>(xt, wt, K, n_total, g, ot, stream);
  if (tiles(TileSmall::BM, TileSmall::BN / kDiv) > num_sms)
    return launch_tile<Te, TileSmall, MODE, 2>(xt, wt, K, n_total, g, ot, stream);
  return launch_tile<Te, TileSmall, MODE, 1>(xt, wt, K, n_total, g, ot, stream);
}

int max_rows(const GroupRows& g) {
  return g.offsets == nullptr ? g.dense_rows : g.cap_rows;
}

}  // namespace

cudaError_t launch_swiglu_simt(int dtype, const void* x, const void* w_gate_up,
                               int d, int inter, const GroupRows& g, void* act,
                               int num_sms, cudaStream_t stream) {
  if (max_rows(g) == 0) return cudaSuccess;
  if (dtype == 0)
    return launch_mode<float, 0>(x, w_gate_up, d, inter, g, act, num_sms, stream);
  return launch_mode<__nv_bfloat16, 0>(x, w_gate_up, d, inter, g, act, num_sms, stream);
}

cudaError_t launch_down_simt(int dtype, const void* act, const void* w_down,
                             int d, int inter, const GroupRows& g, void* y,
                             int num_sms, cudaStream_t stream) {
  if (max_rows(g) == 0) return cudaSuccess;
  if (dtype == 0)
    return launch_mode<float, 1>(act, w_down, inter, d, g, y, num_sms, stream);
  return launch_mode<__nv_bfloat16, 1>(act, w_down, inter, d, g, y, num_sms, stream);
}

}  // namespace rx
