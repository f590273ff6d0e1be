// fp32 on the bf16 tensor cores (tcgen05 + TMEM + TMA), sm_100a: every operand as three bf16 planes hi + mid + lo whose sum
// is the fp32 value, every product as the six plane products above 2^-24 of it.
//
// The two contractions of Eqs. 6-7 cost six times their bf16 form, which is a tenth of what the FFMA pipes could do at
// best (8192 against 128 multiply-adds per clock and SM).  What keeps the result as close to 64 bits as the FFMA kernels of
// simt.cu: planes are rounded to nearest (what the six products leave out is some 2^-27 of a product).  The accumulators of
// the tensor cores cut off towards zero instead of rounding, at every step of 16 terms: so the five small products come
// first, a chain of large ones is two steps (four in MMA1), the chains are added up in 32-bit registers, and the mean of what
// a chain loses (kCut) is put back.  z', D' and the division are 32-bit arithmetic on the unsplit values.  Output against 64
// bits, in the 2-norm, where the FFMA kernels are 8-10e-8 off: 6-8e-8; without kCut 11e-8; in chains of eight 15e-8; all six
// products a step, one step after the other: some 60e-8.
//
// k_f32_planes (haar.cu): Q, K -> T_f(Q), T_f(K) and V as planes
// k_tcx_kside      : S' = ReLU(K_F W)^T V, z' per sequence chunk and group of 128 features
// k_tcx_qside      : O = ReLU(Q_F W) S' / (ReLU(Q_F W) z' + eps'); with two groups each leaves N'_g and D'_g
// k_tcx_combine    : O = sum_g N'_g / (sum_g D'_g + eps')
// k_tcx_bwd_prep   : dO as planes; 1 / D, -dO.O (per token) and sum dD
// k_tcx_kside again: dS' = ReLU(Q_F W)^T (dO / D), dz' = sum of ReLU(Q_F W) dD
// k_tcx_bwd        : dQ_F, or dK_F and dV; a launch per group of 128 features
//
// The tensor-core kernels: 512 threads, 128 registers each.  Warp 0 copies, warp 1 issues the projections (MMA1), warp 2
// the contractions (MMA2), warps 4-11 two groups that take the tiles in turn: accumulator -> ReLU -> planes back into
// TMEM; warps 12-15 drain.  TMEM: two buffers of 192 columns (128 of D1, replaced in place by the hi and mid planes, 64 of
// the lo plane), two accumulators of 64 (k_tcx_bwd has its own).  Every wait is bounded, as in tc_fwd.cu.
// 2 x 8 x 4096, d = 64, m = 256: planes 19 us, key side 28, query side 29, combining 7; the forward 235 -> 96 us.  Alone and on a
// cold L2 the key side takes 49 k cycles for the eight tiles of a CTA, the query side 47 k, with the tensor pipe active 43
// and 46 % of them.
#include "common.cuh"
#include "tc_common.cuh"
#include "tc_maps.cuh"

namespace wersa {
using namespace tc;

namespace {

constexpr int kTile = 128;
constexpr uint32_t kTileBytes = kTile * kD * 2;   // one plane of a tile: 128 x 64 bf16
constexpr uint32_t kTileStep = kTileBytes >> 4;   // in descriptor units
constexpr int kXFeatures = 128;                   // features of a CTA at most
// Features of a CTA in kernels of NF; planes of an argument of type T (a bf16 value is its own first plane, and the products
// with the other two are left out).
template <typename T> constexpr bool kExact = sizeof(T) == 2;
template <typename T> constexpr uint32_t kPlanes = kExact<T> ? 1 : 3;
__device__ __forceinline__ float arg(float x) { return x; }
__device__ __forceinline__ float arg(__nv_bfloat16 x) { return __bfloat162float(x); }
constexpr int kXThreads = 512;
constexpr uint32_t kBufCols = 192, kLoCol = 128, kAccCol = 384;   // TMEM columns
constexpr uint32_t kIdesc2 = make_idesc_bf16(128, 64, false, true);     // B = V or S', N-major
enum { kErrXCopy = 31, kErrXMma = 32, kErrXElem = 33, kErrXDrain = 34 };
enum { kBarZ = 1, kBarDrain = 2 };

// Mean relative loss of a value cut off at 24 bits: half a unit of 2^-23, over the mantissas 1 .. 2 of a value without a
// scale of its own (density 1 / (x ln 2)): 2^-24 / (2 ln 2).
constexpr float kCut = 4.2996e-8f;
__device__ __forceinline__ float put_back(float x) { return fmaf(x, kCut, x); }

// Plane products in the order they are added.
__device__ constexpr int kPa[6] = {2, 0, 1, 1, 0, 0}, kPb[6] = {0, 2, 1, 0, 1, 0};
// (with kExactA / kExactB only those of the operand's first plane)
template <bool kExactA, bool kExactB> __device__ constexpr bool product_on(int q) { return (!kExactA || kPa[q] == 0) && (!kExactB || kPb[q] == 0); }
template <bool kExactA, bool kExactB> __device__ constexpr int first_product() { return product_on<kExactA, kExactB>(0) ? 0 : 1; }

struct alignas(8) XBars {
  uint64_t x_full[2], x_empty[2], v_full, v_empty, d1_full[2], phi_ready[2], d1_free[2], acc_full[2], acc_free[2], den_free[2];
  uint32_t tmem_base;
  int abort_flag;
};
template <typename T> struct KxSmem {
  static constexpr uint32_t wt = 0;                          // planes of W^T (128 features x 64)
  static constexpr uint32_t x = wt + kPlanes<T> * kTileBytes;   // two stages of K_F planes
  static constexpr uint32_t v = x + 6 * kTileBytes;          // planes of V
  static constexpr uint32_t sum = v + kPlanes<T> * kTileBytes;        // S' of the chunk so far: 64 x 128 floats, features side by side
  static constexpr uint32_t zx = sum + 2 * kTileBytes;       // 128 floats
  static constexpr uint32_t bars = zx + 512;
  static constexpr uint32_t total = bars + 256 + 1024;       // + alignment slack
};
template <typename T> struct QxSmem {
  static constexpr uint32_t wt = 0;
  static constexpr uint32_t s = wt + kPlanes<T> * kTileBytes;   // planes of S' (128 features x 64)
  static constexpr uint32_t x = s + 3 * kTileBytes;          // two stages of Q_F planes
  static constexpr uint32_t out = x + 6 * kTileBytes;        // result tile: two boxes of 128 rows x 32 floats
  static constexpr uint32_t out16 = out + 2 * kTileBytes;    // the same as bf16
  static constexpr uint32_t zs = out16 + (kExact<T> ? kTileBytes : 0);       // z' of the group
  static constexpr uint32_t den = zs + 512;                  // denominators of two tiles
  static constexpr uint32_t bars = den + 2 * 512;
  static constexpr uint32_t total = bars + 256 + 1024;
};
static_assert(QxSmem<float>::total <= 232448 && KxSmem<float>::total <= 232448 && sizeof(XBars) <= 256, "shared memory of an SM");

// Tokens of a slab in the per-token arrays of the backward: whole tiles, since they are read past n and in pairs (a slab has
// to begin on an 8-byte boundary where n is odd).
__host__ __device__ __forceinline__ int padded_tokens(int n) { return (n + kTile - 1) / kTile * kTile; }

// Two floats -> one packed pair per plane.  kLarge: values above the largest bf16 keep a finite first plane (see
// bf16_range); features go without, since what a feature of that size adds to is beyond 32 bits with anything above 1.
template <bool kLarge = false>
__device__ __forceinline__ void split3(float a, float b, uint32_t& hi, uint32_t& mid, uint32_t& lo) {
  hi = kLarge ? pack_bf16x2(bf16_range(a), bf16_range(b)) : pack_bf16x2(a, b);
  a -= __uint_as_float(hi << 16);
  b -= __uint_as_float(hi & 0xFFFF0000u);
  mid = pack_bf16x2(a, b);
  a -= __uint_as_float(mid << 16);
  b -= __uint_as_float(mid & 0xFFFF0000u);
  lo = pack_bf16x2(a, b);
}
// Eight floats -> planes.  Is one of them not finite (or above the largest bf16)?
__device__ __forceinline__ bool split8(const float (&v)[8], uint32_t (&p)[3][4]) {
  uint32_t top = 0;
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    split3(v[2 * i], v[2 * i + 1], p[0][i], p[1][i], p[2][i]);
    top |= full_exponents(p[0][i]);
  }
  if (top != 0) {
#pragma unroll
    for (int i = 0; i < 4; ++i) split3<true>(v[2 * i], v[2 * i + 1], p[0][i], p[1][i], p[2][i]);
  }
  return top != 0;
}
// The same -> 16-byte chunk `chunk` of row `row` of the three plane tiles at `tile`.
__device__ __forceinline__ bool put_planes8(uint8_t* tile, int row, int chunk, const float (&v)[8]) {
  uint32_t p[3][4];
  const bool bad = split8(v, p);
#pragma unroll
  for (int s = 0; s < 3; ++s)
    *reinterpret_cast<uint4*>(tile + s * kTileBytes + swz128(row, chunk)) = make_uint4(p[s][0], p[s][1], p[s][2], p[s][3]);
  return bad;
}
// W (d x m, row-major) -> planes of rows f0 .. f0 + 127 of W^T, zero past column d and row m.  512 threads.  The answer is split8's.
template <typename T>
__device__ __forceinline__ bool load_w_planes(const T* __restrict__ W, int d, int m, int f0, uint8_t* wt) {
  const int f = threadIdx.x & 127, part = threadIdx.x >> 7;   // 16 columns
  bool bad = false;
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    float v[8];
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      const int c = 16 * part + 8 * h + j;
      v[j] = c < d && f0 + f < m ? arg(W[(size_t)c * m + f0 + f]) : 0.f;
    }
    if constexpr (kExact<T>) {
      uint32_t u[4], top = 0;
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        u[i] = pack_bf16x2(v[2 * i], v[2 * i + 1]);
        top |= full_exponents(u[i]);
      }
      bad |= top != 0;
      *reinterpret_cast<uint4*>(wt + swz128(f, 2 * part + h)) = make_uint4(u[0], u[1], u[2], u[3]);
    } else {
      bad |= put_planes8(wt, f, 2 * part + h, v);
    }
  }
  return bad;
}
// S' or dS' of a slab's features f0 .. f0 + 127 (64 columns) -> planes, and the group's z' or dz' -> zs: results of the kernel
// in front (see launch_after).  512 threads.
template <int NF>
__device__ __forceinline__ void load_s_planes(const float* S, const float* zg, size_t row0, uint8_t* tile, float* zs) {
  const int f = threadIdx.x >> 2, part = threadIdx.x & 3;   // 16 columns of a feature's row
  const float* src = S + (row0 + f) * kD + 16 * part;
  if (NF == kXFeatures || f < NF) {
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const float4 a = __ldcg(reinterpret_cast<const float4*>(src + 8 * h)), b = __ldcg(reinterpret_cast<const float4*>(src + 8 * h + 4));
      const float v[8] = {a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w};
      put_planes8(tile, f, 2 * part + h, v);
    }
  }
  if (threadIdx.x < NF) zs[threadIdx.x] = __ldcg(zg + row0 + threadIdx.x);
}

// The planes of an infinite value are infinity, NaN and NaN: what the tensor cores make of a dot product that meets one is NaN,
// and a ReLU would drop it.  In 32 bits it is infinite, or NaN where infinities cancel: such elements are formed again, from
// the planes' sums and W.  (Only their class matters: a NaN came from an operand that is not finite.)  The kernels look for
// them where W holds one (which they see as they read it) or the projected tensor does (k_f32_planes leaves word); looking
// every time cost 1 us in each of the kernels of 2 x 4 x 4096, d = 32, m = 128 (a training step 107 -> 110).
template <typename T> struct Operands {
  const __nv_bfloat16* x3;   // first plane: slabs x n rows of d values
  const T* W;                // d x m
  int slab, slabs, n, d, m;
  bool look;                 // is there anything that is not finite?
};
// Are there NaN among 32 columns of the warp?  (False alarms, such as opposite infinities, cost time only.)
__device__ __forceinline__ bool warp_meets_nan(const uint32_t (&r)[32]) {
  f32x2 t[4];
#pragma unroll
  for (int j = 0; j < 4; ++j) t[j] = pk2u(r[2 * j], r[2 * j + 1]);
#pragma unroll
  for (int j = 4; j < 16; ++j) t[j & 3] = add2(t[j & 3], pk2u(r[2 * j], r[2 * j + 1]));
  const float s = sum2(add2(add2(t[0], t[1]), add2(t[2], t[3])));
  return __any_sync(0xffffffffu, s != s);
}
// The NaN among the 32 columns at taddr again.  Column j of a lane is token tok + j * dtok, feature feat + j * dfeat.
template <typename T>
__device__ __noinline__ void form_again(uint32_t taddr, const Operands<T> op, int tok, int dtok, int feat, int dfeat) {
  const size_t plane = (size_t)op.slabs * op.n * op.d;
  for (int j = 0; j < 32; ++j, tok += dtok, feat += dfeat) {
    uint32_t r;
    tmem_ld1(taddr + j, r);
    tmem_ld_wait();
    float a = __uint_as_float(r);
    if (a != a && tok < op.n) {   // (rows past n are zeros: NaN against an infinite W, and no feature either way)
      const __nv_bfloat16* x = op.x3 + ((size_t)op.slab * op.n + tok) * op.d;
      a = 0.f;
      for (int c = 0; c < op.d && a == a; ++c) {
        float v = __bfloat162float(__ldcg(x + c));
        if (fabsf(v) < INFINITY) v = (v + __bfloat162float(__ldcg(x + plane + c))) + __bfloat162float(__ldcg(x + 2 * plane + c));
        a = fmaf(v, arg(op.W[(size_t)c * op.m + feat]), a);
      }
      r = __float_as_uint(a);
    }
    __syncwarp();
    tmem_st1(taddr + j, r);
  }
  tmem_st_wait();
}
// 32 columns of pre-activations.
template <typename T>
__device__ __forceinline__ void load_projected(uint32_t taddr, uint32_t (&r)[32], const Operands<T>& op, int tok, int dtok, int feat,
                                               int dfeat) {
  tmem_ld32(taddr, r);
  tmem_ld_wait();
  reg_fence32(r);
  if (op.look && warp_meets_nan(r)) {
    form_again(taddr, op, tok, dtok, feat, dfeat);
    tmem_ld32(taddr, r);
    tmem_ld_wait();
    reg_fence32(r);
  }
}

// One D1 buffer: 128 fp32 columns -> ReLU -> planes.  32 columns hold 16 hi and 16 mid pairs of their features, the lo pairs
// go to the columns behind them.  Returns the sum of the row's values, kWeighted: each times w[column], in chains of
// eight, as few additions in a row as the FFMA kernels have (two chains of 64: D' 8e-8 off, more than all else together).
// kScaled: the values are multiplied by s[column] first, and the sum is of those times w[column]; both arrays in global
// memory, on an 8-byte boundary, and may hold anything where the value is zero.
// kTokens: the columns are tokens from tok on and the lane is feature feat, else the other way round.
// NC: columns / 32.
template <int NC, bool kTokens, bool kWeighted, bool kScaled = false, typename T>
__device__ __forceinline__ float relu_planes(uint32_t taddr, const Operands<T>& op, int tok, int feat, const float* w,
                                             const float* s = nullptr) {
  uint32_t r[32];
  float total = 0.f;
#pragma unroll 1
  for (int c = 0; c < NC; ++c) {
    load_projected(taddr + 32 * c, r, op, tok + (kTokens ? 32 * c : 0), kTokens, feat + (kTokens ? 0 : 32 * c), !kTokens);
    uint32_t hi[16], mid[16], lo[16];
    float e[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
    for (int j = 0; j < 16; ++j) {
      float a = fmaxf(put_back(__uint_as_float(r[2 * j])), 0.f), b = fmaxf(put_back(__uint_as_float(r[2 * j + 1])), 0.f);
      const int k = 2 * (j & 1);
      if constexpr (kScaled) {
        const float2 z = __ldg(reinterpret_cast<const float2*>(w + 32 * c + 2 * j));
        const float2 f = __ldg(reinterpret_cast<const float2*>(s + 32 * c + 2 * j));
        const bool on_a = a > 0.f, on_b = b > 0.f;
        a = on_a ? a * f.x : 0.f;
        b = on_b ? b * f.y : 0.f;
        e[k] += on_a ? a * z.x : 0.f;
        e[k + 1] += on_b ? b * z.y : 0.f;
      } else if constexpr (kWeighted) {
        const float2 z = *reinterpret_cast<const float2*>(w + 32 * c + 2 * j);
        e[k] = fmaf(a, z.x, e[k]);
        e[k + 1] = fmaf(b, z.y, e[k + 1]);
      } else {
        e[k] += a;
        e[k + 1] += b;
      }
      split3(a, b, hi[j], mid[j], lo[j]);
    }
    total += (e[0] + e[1]) + (e[2] + e[3]);
    tmem_st16(taddr + 32 * c, hi);
    tmem_st16(taddr + 32 * c + 16, mid);
    tmem_st16(taddr + kLoCol + 16 * c, lo);
  }
  tmem_st_wait();
  return total;
}
// TMEM column (inside a buffer) of the eight columns that hold plane `pl` of the 16 values of MMA step k.
__device__ __forceinline__ constexpr uint32_t phi_col(int pl, int k) {
  return pl == 2 ? kLoCol + 8u * k : 32u * (k >> 1) + 16u * pl + 8u * (k & 1);
}

__device__ __forceinline__ void init_bars(XBars* b) {
  for (int i = 0; i < 2; ++i) {
    mbar_init(&b->x_full[i], 1);
    mbar_init(&b->x_empty[i], 1);
    mbar_init(&b->d1_full[i], 1);
    mbar_init(&b->phi_ready[i], 4);
    mbar_init(&b->d1_free[i], 1);
    mbar_init(&b->acc_full[i], 1);
    mbar_init(&b->acc_free[i], 4);
    mbar_init(&b->den_free[i], 4);
  }
  mbar_init(&b->v_full, 1);
  mbar_init(&b->v_empty, 1);
  b->abort_flag = 0;
  fence_mbar_init();
}

// The planes of one tile.
template <uint32_t kN = 3>
__device__ __forceinline__ void load_planes(uint8_t* dst, const CUtensorMap* map, int row0, int slab, int slabs, uint64_t* bar) {
  mbar_arrive_expect_tx(bar, kN * kTileBytes);
#pragma unroll
  for (uint32_t pl = 0; pl < kN; ++pl) tma_load_3d(dst + pl * kTileBytes, map, 0, row0, pl * slabs + slab, bar);
}

// D[128 x N] = A B^T over the head dimension in steps of 16 columns, both operands as planes of up to 128 rows x 64 columns.
// kParts: the steps from the third on go to a second accumulator, kPartCol columns behind the first.
constexpr uint32_t kPartCol = 64;
template <int N, bool kExactA, bool kExactB, bool kParts = false>
__device__ __forceinline__ void issue_planes(uint32_t dst, uint32_t a_lo, uint32_t b_lo, int ksteps, uint32_t hi) {
  constexpr uint32_t kIdesc1 = make_idesc_bf16(128, N, false, false);   // both operands K-major
#pragma unroll
  for (int q = 0; q < 6; ++q)
    if (product_on<kExactA, kExactB>(q))
#pragma unroll
      for (int k = 0; k < 4; ++k)
        if (k < ksteps)
          mma_ss(dst + (kParts && k >= 2 ? kPartCol : 0), smem_desc_join(a_lo + kPa[q] * kTileStep + 2 * k, hi),
                 smem_desc_join(b_lo + kPb[q] * kTileStep + 2 * k, hi), kIdesc1,
                 (q > first_product<kExactA, kExactB>() || (kParts ? k & 1 : k) > 0) ? 1u : 0u);
}
// MMA1 of every tile.  kXIsA: the tile is A (query side: tokens x NF features), else W^T is (key side: features x tokens).
template <bool kXIsA, int NF, bool kExactW>
__device__ __forceinline__ void issue_mma1(XBars* bars, uint8_t* x, uint8_t* wt, uint32_t tmem, int nt, int d,
                                           volatile int* abort_flag, int* status) {
  const uint32_t hi = smem_desc_hi(1024);
  const uint32_t wt_lo = smem_desc_lo(smem_u32(wt), 16), x_lo0 = smem_desc_lo(smem_u32(x), 16);
  const int ksteps = (d + 15) >> 4;   // the rest of a narrow head is zeros
  for (int t = 0; t < nt; ++t) {
    const int b = t & 1;
    if (!mbar_wait(&bars->x_full[b], (t >> 1) & 1, abort_flag, status, kErrXMma)) break;
    if (t >= 2 && !mbar_wait(&bars->d1_free[b], ((t >> 1) - 1) & 1, abort_flag, status, kErrXMma)) break;
    tc_fence_after_sync();
    const uint32_t x_lo = x_lo0 + b * 3 * kTileStep;
    issue_planes<kXIsA ? NF : 128, !kXIsA && kExactW, kXIsA && kExactW>(tmem + b * kBufCols, kXIsA ? x_lo : wt_lo,
                                                                        kXIsA ? wt_lo : x_lo, ksteps, hi);
    mma_commit(&bars->d1_full[b]);
    mma_commit(&bars->x_empty[b]);
  }
}
// The t-th contraction of a CTA, a part (32 of the 32 NC values of K) at a time: accumulator u % 2 (64 columns each, from
// `acc` on) = Phi (planes in the buffer at `buf`) * B (planes of 64 columns at b_lo), u = NC t + part.
template <int NC, bool kExactB, typename Bars>
__device__ __forceinline__ bool issue_mma2(Bars* bars, uint32_t acc, uint32_t buf, int t, uint32_t b_lo, uint32_t hi,
                                           volatile int* abort_flag, int* status) {
#pragma unroll
  for (int c = 0; c < NC; ++c) {
    const int u = NC * t + c, r = c & 1;
    if (u >= 2 && !mbar_wait(&bars->acc_free[r], ((u >> 1) - 1) & 1, abort_flag, status, kErrXMma)) return false;
    tc_fence_after_sync();
#pragma unroll
    for (int q = 0; q < 6; ++q)
      if (product_on<false, kExactB>(q))
#pragma unroll
        for (int k = 2 * c; k < 2 * c + 2; ++k)
          mma_ts(acc + 64 * r, buf + phi_col(kPa[q], k), smem_desc_join(b_lo + kPb[q] * kTileStep + 128 * k, hi), kIdesc2,
                 (q > 0 || k > 2 * c) ? 1u : 0u);
    mma_commit(&bars->acc_full[r]);
  }
  return true;
}
// s[0 .. 63] += the parts of the t-th contraction.  One warp's share (32 lanes); taddr: its lanes, first accumulator.
template <int NC, typename Bars>
__device__ __forceinline__ bool drain_tile(Bars* bars, uint32_t taddr, int t, float (&s)[64], volatile int* abort_flag, int* status) {
#pragma unroll 1
  for (int u = NC * t; u < NC * t + NC; ++u) {
    const int r = u & 1;
    if (!__all_sync(0xffffffffu, mbar_wait(&bars->acc_full[r], (u >> 1) & 1, abort_flag, status, kErrXDrain))) return false;
    tc_fence_after_sync();
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      uint32_t v[32];
      tmem_ld32(taddr + 64 * r + 32 * h, v);
      tmem_ld_wait();
      reg_fence32(v);
#pragma unroll
      for (int j = 0; j < 32; ++j) s[32 * h + j] += __uint_as_float(v[j]);
    }
    tc_fence_before_sync();
    warp_arrive(&bars->acc_free[r]);
  }
  return true;
}

// ---- key side.  grid (chunks, slabs, feature groups) ---------------------------------------------
// kScaled: the query side of the backward, with Q_F and dO in the place of K_F and V.  Feature values are divided by their
// token's D (scale, slabs of padded_tokens(n)), the sums weighted by c = -dO.O on top: dS' and dz'.
// NF = 64: the rows of the tile past them hold nothing (their warps keep step, and D1's zeros there are nobody's operand).
template <bool kScaled, typename T, int NF>
__global__ void __launch_bounds__(kXThreads, 1)
k_tcx_kside(const __grid_constant__ CUtensorMap map_k, const __grid_constant__ CUtensorMap map_v, const T* __restrict__ W,
            float* __restrict__ spart, float* __restrict__ zpart, int n, int d, int m, int chunk_tiles, int* __restrict__ status,
            const __nv_bfloat16* x3, const int* seen, const float* __restrict__ scale, const float* __restrict__ weight) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = align_smem(smem_raw);
  using SL = KxSmem<T>;
  XBars* bars = reinterpret_cast<XBars*>(smem + SL::bars);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int chunk = blockIdx.x, slab = blockIdx.y, slabs = gridDim.y, f0 = blockIdx.z * NF;
  const int t0 = chunk * chunk_tiles, nt = min(chunk_tiles, (n + kTile - 1) / kTile - t0);
  if (threadIdx.x == 0) init_bars(bars);
  if (warp == 1) {
    tmem_alloc(&bars->tmem_base, 512);
    tmem_relinquish();
  }
  const bool bad_w = load_w_planes(W, d, m, f0, smem + SL::wt);
  fence_proxy_async_smem();
  tc_fence_before_sync();
  const bool look_w = __syncthreads_or(bad_w);
  tc_fence_after_sync();
  wait_for_stream_predecessor();   // (launched as a programmatic dependent: the planes come from the kernel before)
  let_stream_successor_start();
  const uint32_t tmem = bars->tmem_base;
  volatile int* abort_flag = &bars->abort_flag;
  if (warp == 0 && lane == 0) {
    // K_F two tiles ahead of MMA1, V behind it: a stage of K_F is free long before the buffer of V
    int xs = 0, vs = 0;
    bool ok = true;
    auto load_x = [&](int t) {
      const int s = t & 1;
      if (t >= 2) ok = mbar_wait(&bars->x_empty[s], ((t >> 1) - 1) & 1, abort_flag, status, kErrXCopy);
      if (!ok) return;
      load_planes(smem + SL::x + s * 3 * kTileBytes, &map_k, (t0 + t) * kTile, slab, slabs, &bars->x_full[s]);
      ++xs;
    };
    load_x(0);
    if (nt > 1) load_x(1);
    for (int t = 0; t < nt && ok; ++t) {
      if (t > 0) ok = mbar_wait(&bars->v_empty, (t - 1) & 1, abort_flag, status, kErrXCopy);
      if (!ok) break;
      load_planes<kPlanes<T>>(smem + SL::v, &map_v, (t0 + t) * kTile, slab, slabs, &bars->v_full);
      ++vs;
      if (t + 2 < nt) load_x(t + 2);
    }
    if (*abort_flag != 0) {   // let copies in flight land before the CTA's shared memory goes away
      for (int t = max(0, xs - 2); t < xs; ++t) mbar_wait_drain(&bars->x_full[t & 1], (t >> 1) & 1);
      if (vs > 0) mbar_wait_drain(&bars->v_full, (vs - 1) & 1);
    }
  } else if (warp == 1 && lane == 0) {
    issue_mma1<false, NF, kExact<T>>(bars, smem + SL::x, smem + SL::wt, tmem, nt, d, abort_flag, status);
  } else if (warp == 2 && lane == 0) {
    const uint32_t hi = smem_desc_hi(1024), v_lo = smem_desc_lo(smem_u32(smem + SL::v), 1024);
    for (int t = 0; t < nt; ++t) {
      if (!mbar_wait(&bars->v_full, t & 1, abort_flag, status, kErrXMma)) break;
      if (!mbar_wait(&bars->phi_ready[t & 1], (t >> 1) & 1, abort_flag, status, kErrXMma)) break;
      if (!issue_mma2<4, kExact<T>>(bars, tmem + kAccCol, tmem + (t & 1) * kBufCols, t, v_lo, hi, abort_flag, status)) break;
      mma_commit(&bars->d1_free[t & 1]);
      mma_commit(&bars->v_empty);
    }
  } else if (warp >= 4 && warp < 12) {
    const int g = (warp - 4) >> 2;
    const uint32_t row = 32u * (warp & 3) + lane;   // feature of the group = TMEM lane
    const uint32_t taddr = tmem + ((32u * (warp & 3)) << 16) + g * kBufCols;
    float* zx = reinterpret_cast<float*>(smem + SL::zx);
    const Operands<T> op = {x3, W, slab, slabs, n, d, m, look_w || __ldcg(seen) != 0};
    float z = 0.f;
    bool ok = true;
    for (int t = g; t < nt && ok; t += 2) {
      ok = __all_sync(0xffffffffu, mbar_wait(&bars->d1_full[g], (t >> 1) & 1, abort_flag, status, kErrXElem));
      if (!ok) break;
      tc_fence_after_sync();
      if (row >= NF) {   // (whole warps)
      } else if constexpr (kScaled) {
        const size_t tok = (size_t)slab * padded_tokens(n) + (size_t)(t0 + t) * kTile;
        z += relu_planes<4, true, true, true>(taddr, op, (t0 + t) * kTile, f0 + row, weight + tok, scale + tok);
      } else {
        z += relu_planes<4, true, false>(taddr, op, (t0 + t) * kTile, f0 + row, nullptr);
      }
      tc_fence_before_sync();
      warp_arrive(&bars->phi_ready[g]);
    }
    if (g == 1) zx[row] = z;
    named_bar_sync(kBarZ, 256);
    if (g == 0 && ok && row < NF) zpart[((size_t)slab * gridDim.x + chunk) * m + f0 + row] = z + zx[row];
  } else if (warp >= 12) {
    const uint32_t row = 32u * (warp & 3) + lane;
    const uint32_t taddr = tmem + ((32u * (warp & 3)) << 16) + kAccCol;
    // (a tile's quarters first, then the chunk: the chunk's sum is added to once a tile)
    float* sum = reinterpret_cast<float*>(smem + SL::sum) + row;
    bool ok = true;
    for (int t = 0; t < nt && ok; ++t) {
      float s[64];
#pragma unroll
      for (int j = 0; j < 64; ++j) s[j] = 0.f;
      ok = drain_tile<4>(bars, taddr, t, s, abort_flag, status);
      if (!ok) break;
#pragma unroll
      for (int j = 0; j < 64; ++j) sum[j * kXFeatures] = t > 0 ? sum[j * kXFeatures] + s[j] : s[j];
    }
    if (ok && row < NF) {
      float* dst = spart + (((size_t)slab * gridDim.x + chunk) * m + f0 + row) * kD;
#pragma unroll
      for (int j = 0; j < 64; j += 4)
        *reinterpret_cast<float4*>(dst + j) =
            make_float4(put_back(sum[j * kXFeatures]), put_back(sum[(j + 1) * kXFeatures]), put_back(sum[(j + 2) * kXFeatures]),
                        put_back(sum[(j + 3) * kXFeatures]));
    }
  }
  tc_fence_before_sync();
  __syncthreads();
  if (warp == 1) {
    tc_fence_after_sync();
    tmem_dealloc(tmem, 512);
  }
}

// ---- query side.  grid (chunks, slabs, feature groups) -------------------------------------------
// One group: O, divided, and with keep (for a backward) once more into map_keep.  Several: N'_g into map_o (group-major
// slabs).  den_out, where given: D'_g at [(group * slabs + slab) * n + token].
template <typename T, int NF>
__global__ void __launch_bounds__(kXThreads, 1)
k_tcx_qside(const __grid_constant__ CUtensorMap map_q, const __grid_constant__ CUtensorMap map_o, const T* __restrict__ W,
            const float* __restrict__ S, const float* __restrict__ zg, const float* __restrict__ beta, float eps, float bw_floor,
            float* __restrict__ den_out, const __grid_constant__ CUtensorMap map_keep, int keep, int n, int d, int m, int chunk_tiles,
            int* __restrict__ status, const __nv_bfloat16* x3,
            const int* seen) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = align_smem(smem_raw);
  using SL = QxSmem<T>;
  XBars* bars = reinterpret_cast<XBars*>(smem + SL::bars);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int chunk = blockIdx.x, slab = blockIdx.y, slabs = gridDim.y, f0 = blockIdx.z * NF;
  const int t0 = chunk * chunk_tiles, nt = min(chunk_tiles, (n + kTile - 1) / kTile - t0);
  float* zs = reinterpret_cast<float*>(smem + SL::zs);
  float* den = reinterpret_cast<float*>(smem + SL::den);
  if (threadIdx.x == 0) {
    init_bars(bars);
    // (launched as a programmatic dependent: the planes are older than the reduction in front of this kernel)
    for (int t = 0; t < min(nt, 2); ++t)
      load_planes(smem + SL::x + t * 3 * kTileBytes, &map_q, (t0 + t) * kTile, slab, slabs, &bars->x_full[t]);
  }
  if (warp == 1) {
    tmem_alloc(&bars->tmem_base, 512);
    tmem_relinquish();
  }
  const bool bad_w = load_w_planes(W, d, m, f0, smem + SL::wt);
  wait_for_stream_predecessor();
  load_s_planes<NF>(S, zg, (size_t)slab * m + f0, smem + SL::s, zs);
  fence_proxy_async_smem();
  tc_fence_before_sync();
  const bool look_w = __syncthreads_or(bad_w);
  tc_fence_after_sync();
  const uint32_t tmem = bars->tmem_base;
  volatile int* abort_flag = &bars->abort_flag;
  if (warp == 0 && lane == 0) {
    int xs = min(nt, 2);
    for (int t = 2; t < nt; ++t) {
      const int s = t & 1;
      if (!mbar_wait(&bars->x_empty[s], ((t >> 1) - 1) & 1, abort_flag, status, kErrXCopy)) break;
      load_planes(smem + SL::x + s * 3 * kTileBytes, &map_q, (t0 + t) * kTile, slab, slabs, &bars->x_full[s]);
      ++xs;
    }
    if (*abort_flag != 0)   // let copies in flight land before the CTA's shared memory goes away
      for (int t = max(0, xs - 2); t < xs; ++t) mbar_wait_drain(&bars->x_full[t & 1], (t >> 1) & 1);
  } else if (warp == 1 && lane == 0) {
    issue_mma1<true, NF, kExact<T>>(bars, smem + SL::x, smem + SL::wt, tmem, nt, d, abort_flag, status);
  } else if (warp == 2 && lane == 0) {
    const uint32_t hi = smem_desc_hi(1024), s_lo = smem_desc_lo(smem_u32(smem + SL::s), 1024);
    for (int t = 0; t < nt; ++t) {
      if (!mbar_wait(&bars->phi_ready[t & 1], (t >> 1) & 1, abort_flag, status, kErrXMma)) break;
      if (!issue_mma2<NF / 32, false>(bars, tmem + kAccCol, tmem + (t & 1) * kBufCols, t, s_lo, hi, abort_flag, status)) break;
      mma_commit(&bars->d1_free[t & 1]);
    }
  } else if (warp >= 4 && warp < 12) {
    const int g = (warp - 4) >> 2;
    const uint32_t row = 32u * (warp & 3) + lane;   // token of the tile = TMEM lane
    const uint32_t taddr = tmem + ((32u * (warp & 3)) << 16) + g * kBufCols;
    const Operands<T> op = {x3, W, slab, slabs, n, d, m, look_w || __ldcg(seen) != 0};
    bool ok = true;
    for (int t = g; t < nt && ok; t += 2) {
      ok = __all_sync(0xffffffffu, mbar_wait(&bars->d1_full[g], (t >> 1) & 1, abort_flag, status, kErrXElem));
      if (!ok) break;
      tc_fence_after_sync();
      const float sum = relu_planes<NF / 32, false, true>(taddr, op, (t0 + t) * kTile + row, f0, zs);
      if (t >= 2) {   // the drain has read the denominators of tile t - 2
        ok = __all_sync(0xffffffffu, mbar_wait(&bars->den_free[g], ((t >> 1) - 1) & 1, abort_flag, status, kErrXElem));
        if (!ok) break;
      }
      den[g * kTile + row] = sum;
      tc_fence_before_sync();
      warp_arrive(&bars->phi_ready[g]);
    }
  } else if (warp >= 12) {
    const int et = threadIdx.x - 384;               // token of the tile = TMEM lane
    const uint32_t taddr = tmem + ((32u * (warp & 3)) << 16) + kAccCol;
    const float bw = fmaxf(beta[0], bw_floor);
    const float epsp = eps * (float)m * bw * bw;
    const bool divide = gridDim.z == 1;
    const int out_slab = blockIdx.z * slabs + slab;
    uint8_t* out = smem + SL::out;
    bool ok = true;
    for (int t = 0; t < nt; ++t) {
      const int b = t & 1, row0 = (t0 + t) * kTile;
      float s[64], scale = 1.f;
#pragma unroll
      for (int j = 0; j < 64; ++j) s[j] = 0.f;
      if (ok) ok = drain_tile<NF / 32>(bars, taddr, t, s, abort_flag, status);
      if (ok) {   // (the tile's denominators are older than its first accumulator)
        const float dn = den[b * kTile + et];
        if (divide) scale = put_back(1.f / (dn + epsp));
        if (den_out != nullptr && row0 + et < n) den_out[(size_t)out_slab * n + row0 + et] = dn;
        warp_arrive(&bars->den_free[b]);
      }
      if (et == 0) bulk_wait_group_read0();   // the tile before has left the staging boxes
      named_bar_sync(kBarDrain, 128);
      if (ok) {
        if constexpr (kExact<T>) {
#pragma unroll
          for (int j = 0; j < 8; ++j)
            *reinterpret_cast<uint4*>(smem + SL::out16 + swz128(et, j)) =
                make_uint4(pack_bf16x2(s[8 * j] * scale, s[8 * j + 1] * scale), pack_bf16x2(s[8 * j + 2] * scale, s[8 * j + 3] * scale),
                           pack_bf16x2(s[8 * j + 4] * scale, s[8 * j + 5] * scale), pack_bf16x2(s[8 * j + 6] * scale, s[8 * j + 7] * scale));
        }
        if (!kExact<T> || keep)
#pragma unroll
        for (int j = 0; j < 16; ++j)
          *reinterpret_cast<float4*>(out + (j >> 3) * kTileBytes + swz128(et, j & 7)) =
              make_float4(s[4 * j] * scale, s[4 * j + 1] * scale, s[4 * j + 2] * scale, s[4 * j + 3] * scale);
        fence_proxy_async_smem();
      }
      named_bar_sync(kBarDrain, 128);
      if (et == 0 && ok) {   // rows past n and columns past d are clipped
        if constexpr (kExact<T>) {
          tma_store_3d(&map_o, smem + SL::out16, 0, row0, out_slab);
        } else {
          tma_store_3d(&map_o, out, 0, row0, out_slab);
          if (d > 32) tma_store_3d(&map_o, out + kTileBytes, 32, row0, out_slab);
        }
        if (keep) {
          tma_store_3d(&map_keep, out, 0, row0, out_slab);
          if (d > 32) tma_store_3d(&map_keep, out + kTileBytes, 32, row0, out_slab);
        }
        bulk_commit_group();
      }
    }
    if (et == 0) bulk_wait_group0();
  }
  tc_fence_before_sync();
  __syncthreads();
  if (warp == 1) {
    tc_fence_after_sync();
    tmem_dealloc(tmem, 512);
  }
}

// O = (N'_0 + N'_1) / (D'_0 + D'_1 + eps'), one thread per four columns; with keep (for a backward) there too.
__global__ void __launch_bounds__(256) k_tcx_combine(const float* __restrict__ N, const float* __restrict__ den,
                                                     const float* __restrict__ beta, float eps, float bw_floor, int m,
                                                     float* __restrict__ O, float* __restrict__ keep, size_t tokens, int d) {
  wait_for_stream_predecessor();   // (launched as a programmatic dependent: see launch_after)
  const size_t idx = (size_t)blockIdx.x * 256 + threadIdx.x;
  const int per = d >> 2;
  const size_t tok = idx / per;
  if (tok >= tokens) return;
  const float bw = fmaxf(beta[0], bw_floor);
  const float inv = put_back(1.f / ((load_after_wait(den + tok) + load_after_wait(den + tokens + tok)) + eps * (float)m * bw * bw));
  const float4 a = load4_after_wait(N + idx * 4), b = load4_after_wait(N + tokens * d + idx * 4);
  const float4 o = make_float4((a.x + b.x) * inv, (a.y + b.y) * inv, (a.z + b.z) * inv, (a.w + b.w) * inv);
  *reinterpret_cast<float4*>(O + idx * 4) = o;
  if (keep != nullptr) *reinterpret_cast<float4*>(keep + idx * 4) = o;
}

// ---- backward ------------------------------------------------------------------------------------
// Per token: planes of dO, 1 / D (D = sum_g D'_g + eps'), c = -dO.O; sum of dD = c / D per CTA.  tpt threads (a power of
// two >= d / 8) on a token, eight columns each.  Bound by memory (2 x 8 x 4096, d = 64: 59 MB).
// (bf16 gradients are their own plane: dO3 stays unwritten)
template <typename T>
__global__ void __launch_bounds__(256, 6)
k_tcx_bwd_prep(const T* __restrict__ dO, const float* __restrict__ O, const float* __restrict__ den, int groups,
               const float* __restrict__ beta, float eps, float bw_floor, int m, int d, int tpt, size_t tokens, int n,
               __nv_bfloat16* __restrict__ dO3, float* __restrict__ inv, float* __restrict__ c, float* __restrict__ sumdD) {
  __shared__ float sums[8];
  wait_for_stream_predecessor();   // (launched as a programmatic dependent: see launch_after)
  let_stream_successor_start();
  const float bw = fmaxf(beta[0], bw_floor);
  const float epsp = eps * (float)m * bw * bw;
  const size_t total = tokens * tpt, plane = tokens * d;
  const size_t warp_first = (size_t)blockIdx.x * 256 + (threadIdx.x & ~31u);
  float dd = 0.f;
  for (size_t w0 = warp_first; w0 < total; w0 += (size_t)gridDim.x * 256) {   // whole warps: the shuffles want all lanes
    const size_t i = w0 + (threadIdx.x & 31), tok = i / tpt;
    const int c0 = 8 * (int)(i % tpt);
    float dot = 0.f;
    if (tok < tokens && c0 < d) {
      float g[8];
      load8(dO + tok * d + c0, g);
      const float4 oa = load4_after_wait(O + tok * d + c0), ob = load4_after_wait(O + tok * d + c0 + 4);
      const float o[8] = {oa.x, oa.y, oa.z, oa.w, ob.x, ob.y, ob.z, ob.w};
#pragma unroll
      for (int j = 0; j < 8; ++j) dot = fmaf(g[j], o[j], dot);
      if constexpr (!kExact<T>) {
        uint32_t pl[3][4];
        split8(g, pl);
#pragma unroll
        for (int s = 0; s < 3; ++s)
          *reinterpret_cast<uint4*>(dO3 + s * plane + tok * d + c0) = make_uint4(pl[s][0], pl[s][1], pl[s][2], pl[s][3]);
      }
    }
    for (int o = tpt >> 1; o > 0; o >>= 1) dot += __shfl_xor_sync(0xffffffffu, dot, o);
    if (tok < tokens && c0 == 0) {
      float D = 0.f;
      for (int g = 0; g < groups; ++g) D += load_after_wait(den + g * tokens + tok);
      const float iv = 1.f / (D + epsp);
      const size_t slab = tok / n, at = slab * padded_tokens(n) + (tok - slab * n);
      inv[at] = iv;
      c[at] = -dot;
      dd = fmaf(-dot, iv, dd);
    }
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) dd += __shfl_xor_sync(0xffffffffu, dd, o);
  if ((threadIdx.x & 31) == 0) sums[threadIdx.x >> 5] = dd;
  __syncthreads();
  if (threadIdx.x == 0) {
    float s = 0.f;
#pragma unroll
    for (int i = 0; i < 8; ++i) s += sums[i];
    sumdD[blockIdx.x] = s;
  }
}

struct alignas(8) YBars {
  uint64_t x_full, x_empty, y_full, y_empty, a_full, a_done, g_full, g_done, a_ready, g_ready, acc_full[2], acc_free[2];
  uint32_t tmem_base;
  int abort_flag;
};
template <typename T> struct YSmem {
  static constexpr uint32_t wt = 0;                          // planes of W^T (128 features x 64)
  static constexpr uint32_t s = wt + kPlanes<T> * kTileBytes;   // planes of S' or dS'
  static constexpr uint32_t x = s + 3 * kTileBytes;          // planes of Q_F or K_F
  static constexpr uint32_t y = x + 3 * kTileBytes;          // planes of dO or V
  static constexpr uint32_t out = y + kPlanes<T> * kTileBytes;        // result tile: two boxes of 128 rows x 32 floats
  static constexpr uint32_t zs = out + 2 * kTileBytes;       // z' or dz' of the group
  static constexpr uint32_t bars = zs + 512;
  static constexpr uint32_t total = bars + 256 + 1024;
};
static_assert(YSmem<float>::total <= 232448 && sizeof(YBars) <= 256, "shared memory of an SM");

// Chunk `chunk` (32 of 128 values) of a row -> planes, laid out as relu_planes leaves them.
__device__ __forceinline__ void store_chunk_planes(uint32_t buf, int chunk, const float (&v)[32]) {
  uint32_t hi[16], mid[16], lo[16];
#pragma unroll
  for (int j = 0; j < 16; ++j) split3(v[2 * j], v[2 * j + 1], hi[j], mid[j], lo[j]);
  tmem_st16(buf + 32 * chunk, hi);
  tmem_st16(buf + 32 * chunk + 16, mid);
  tmem_st16(buf + kLoCol + 16 * chunk, lo);
}

// Per 128-token tile and group: A = X W (which features are on) and G = Y S^T, then
// queries (X = Q_F, Y = dO, S = S'):  dQ_F = [(G + c z') / D where on] W^T
// keys    (X = K_F, Y = V, S = dS'):  dK_F = [(G + dz') where on] W^T,  dV = ReLU(A) dS'
// Both accumulators of a tile wait for the groups of warps 4-7 and 8-11, half the features each; dQ_F, dK_F and dV of a second
// group of features are added by the copy engine (the launches follow one another).
// Bound by latency: a tile is one chain copy -> MMA1 -> ReLU -> MMA2 -> drain with nothing of the next tile beside it but its
// copies.  2 x 4 x 4096, d = 32, m = 128 (two tiles a CTA): queries 15 us, keys some 22; the backward of 8 x 4 x 1024 92 -> 65 us.
// TMEM: keys: A and its planes 192, G and its planes 192; queries: A 128, G 192; then two accumulators of 64.
// With 64 features G has room for two accumulators of its own, of 32 columns of Y each: chains of two steps, as long as those of
// O and dS', lose the same in the mean.  phi . (G + c z') is zero for every token, the two terms being of opposite signs, and so is the
// sum of phi (G + dz') over all keys and features: the gate's gradients, which are sums of such terms by bands, hold the
// difference of the two losses many times over.  dgate_w, domega against 64 bits, medians of 20 seeds, with one chain of four, two of
// two, FFMA, in 1e-6: bf16 60 x 2 x 900 2.6 5.1, 1.2 1.2, 0.6 0.9; 300 x 260 2.7 2.8, 1.1 1.2, 0.7 0.6; 1 x 2 x 20001 0.8 1.1, 0.7 0.7, 0.6
// 0.6; fp32 300 x 260 3.3 3.5, 1.4 1.3, 0.6 0.7.  (Another constant than kCut for G: worse on either side.)  Training steps
// 14 x 21903, bf16 447.3 -> 449.1 us, 53 x 4 x 355 204.0 -> 206.1.
// TG: type of dV.
template <bool kKeys, typename T, typename TG, int NF>
__global__ void __launch_bounds__(kXThreads, 1)
k_tcx_bwd(const __grid_constant__ CUtensorMap map_x, const __grid_constant__ CUtensorMap map_y, const T* __restrict__ W,
          const float* __restrict__ S, const float* __restrict__ zg, const float* __restrict__ tok_inv,
          const float* __restrict__ tok_c, const __grid_constant__ CUtensorMap map_dx, const __grid_constant__ CUtensorMap map_dv,
          int add, int n, int d, int m, int f0, int chunk_tiles, int* __restrict__ status, const __nv_bfloat16* x3,
            const int* seen) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = align_smem(smem_raw);
  using SL = YSmem<T>;
  constexpr uint32_t kG = kKeys ? kBufCols : 128, kAcc = kG + kBufCols;
  constexpr int kPer = kKeys ? 2 : 1;   // contractions of a tile
  constexpr int kHalf = NF / 2, kH = NF / 64;   // features of a group of warps, and 32 at a time
  constexpr bool kParts = NF <= (int)kPartCol;
  YBars* bars = reinterpret_cast<YBars*>(smem + SL::bars);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int chunk = blockIdx.x, slab = blockIdx.y, slabs = gridDim.y;
  const int t0 = chunk * chunk_tiles, nt = min(chunk_tiles, (n + kTile - 1) / kTile - t0);
  float* zs = reinterpret_cast<float*>(smem + SL::zs);
  if (threadIdx.x == 0) {
    mbar_init(&bars->x_full, 1);
    mbar_init(&bars->x_empty, 1);
    mbar_init(&bars->y_full, 1);
    mbar_init(&bars->y_empty, 1);
    mbar_init(&bars->a_full, 1);
    mbar_init(&bars->a_done, kKeys ? 1 : 8);   // keys: MMA2 has read the planes; queries: the warps have read A
    mbar_init(&bars->g_full, 1);
    mbar_init(&bars->g_done, 1);
    mbar_init(&bars->a_ready, 8);
    mbar_init(&bars->g_ready, 8);
    for (int i = 0; i < 2; ++i) {
      mbar_init(&bars->acc_full[i], 1);
      mbar_init(&bars->acc_free[i], 4);
    }
    bars->abort_flag = 0;
    fence_mbar_init();
  }
  if (warp == 1) {
    tmem_alloc(&bars->tmem_base, 512);
    tmem_relinquish();
  }
  const bool bad_w = load_w_planes(W, d, m, f0, smem + SL::wt);
  wait_for_stream_predecessor();   // (launched as a programmatic dependent: see launch_after)
  // (behind the key side come kernels that start with reads of what it writes and that lost time placed early)
  if constexpr (!kKeys) let_stream_successor_start();
  load_s_planes<NF>(S, zg, (size_t)slab * m + f0, smem + SL::s, zs);
  fence_proxy_async_smem();
  tc_fence_before_sync();
  const bool look_w = __syncthreads_or(bad_w);
  tc_fence_after_sync();
  const uint32_t tmem = bars->tmem_base;
  volatile int* abort_flag = &bars->abort_flag;
  const uint32_t hi = smem_desc_hi(1024);
  if (warp == 0 && lane == 0) {
    int xs = 0, ys = 0;
    for (int t = 0; t < nt; ++t) {
      if (t > 0 && !mbar_wait(&bars->x_empty, (t - 1) & 1, abort_flag, status, kErrXCopy)) break;
      load_planes(smem + SL::x, &map_x, (t0 + t) * kTile, slab, slabs, &bars->x_full);
      ++xs;
      if (t > 0 && !mbar_wait(&bars->y_empty, (t - 1) & 1, abort_flag, status, kErrXCopy)) break;
      load_planes<kPlanes<T>>(smem + SL::y, &map_y, (t0 + t) * kTile, slab, slabs, &bars->y_full);
      ++ys;
    }
    if (*abort_flag != 0) {   // let copies in flight land before the CTA's shared memory goes away
      if (xs > 0) mbar_wait_drain(&bars->x_full, (xs - 1) & 1);
      if (ys > 0) mbar_wait_drain(&bars->y_full, (ys - 1) & 1);
    }
  } else if (warp == 1 && lane == 0) {
    const uint32_t x_lo = smem_desc_lo(smem_u32(smem + SL::x), 16), y_lo = smem_desc_lo(smem_u32(smem + SL::y), 16);
    const uint32_t wt_lo = smem_desc_lo(smem_u32(smem + SL::wt), 16), s_lo = smem_desc_lo(smem_u32(smem + SL::s), 16);
    const int ksteps = (d + 15) >> 4;
    for (int t = 0; t < nt; ++t) {
      if (!mbar_wait(&bars->x_full, t & 1, abort_flag, status, kErrXMma)) break;
      if (t > 0 && !mbar_wait(&bars->a_done, (t - 1) & 1, abort_flag, status, kErrXMma)) break;
      tc_fence_after_sync();
      issue_planes<NF, false, kExact<T>>(tmem, x_lo, wt_lo, ksteps, hi);
      mma_commit(&bars->a_full);
      mma_commit(&bars->x_empty);
      if (!mbar_wait(&bars->y_full, t & 1, abort_flag, status, kErrXMma)) break;
      if (t > 0 && !mbar_wait(&bars->g_done, (t - 1) & 1, abort_flag, status, kErrXMma)) break;
      tc_fence_after_sync();
      issue_planes<NF, kExact<T>, false, kParts>(tmem + kG, y_lo, s_lo, ksteps, hi);
      mma_commit(&bars->g_full);
      mma_commit(&bars->y_empty);
    }
  } else if (warp == 2 && lane == 0) {
    const uint32_t s_lo = smem_desc_lo(smem_u32(smem + SL::s), 1024), wt_lo = smem_desc_lo(smem_u32(smem + SL::wt), 1024);
    for (int t = 0; t < nt; ++t) {
      if constexpr (kKeys) {
        if (!mbar_wait(&bars->a_ready, t & 1, abort_flag, status, kErrXMma)) break;
        if (!issue_mma2<NF / 32, false>(bars, tmem + kAcc, tmem, 2 * t, s_lo, hi, abort_flag, status)) break;
        mma_commit(&bars->a_done);
      }
      if (!mbar_wait(&bars->g_ready, t & 1, abort_flag, status, kErrXMma)) break;
      if (!issue_mma2<NF / 32, kExact<T>>(bars, tmem + kAcc, tmem + kG, kPer * t + kPer - 1, wt_lo, hi, abort_flag, status)) break;
      mma_commit(&bars->g_done);
    }
  } else if (warp >= 4 && warp < 12) {
    const int g = (warp - 4) >> 2;                        // features kHalf g .. + kHalf - 1
    const uint32_t row = 32u * (warp & 3) + lane;         // token of the tile = TMEM lane
    const uint32_t lanes = tmem + ((32u * (warp & 3)) << 16);
    const Operands<T> op = {x3, W, slab, slabs, n, d, m, look_w || __ldcg(seen) != 0};
    bool ok = true;
    for (int t = 0; t < nt && ok; ++t) {
      float inv = 0.f, c = 0.f;
      if constexpr (!kKeys) {
        const int tok = (t0 + t) * kTile + row;
        if (tok < n) {
          inv = __ldcg(tok_inv + (size_t)slab * padded_tokens(n) + tok);
          c = __ldcg(tok_c + (size_t)slab * padded_tokens(n) + tok);
        }
      }
      ok = __all_sync(0xffffffffu, mbar_wait(&bars->a_full, t & 1, abort_flag, status, kErrXElem));
      if (!ok) break;
      tc_fence_after_sync();
      uint32_t on[kH];
      uint32_t r[32];
#pragma unroll
      for (int h = 0; h < kH; ++h) {
        load_projected(lanes + kHalf * g + 32 * h, r, op, (t0 + t) * kTile + row, 0, f0 + kHalf * g + 32 * h, 1);
        on[h] = 0;
        float v[32];
#pragma unroll
        for (int j = 0; j < 32; ++j) {
          const float x = __uint_as_float(r[j]);
          on[h] |= (x > 0.f ? 1u : 0u) << j;
          v[j] = fmaxf(put_back(x), 0.f);
        }
        if constexpr (kKeys) store_chunk_planes(lanes, kH * g + h, v);
      }
      if constexpr (kKeys) tmem_st_wait();
      tc_fence_before_sync();
      warp_arrive(kKeys ? &bars->a_ready : &bars->a_done);
      ok = __all_sync(0xffffffffu, mbar_wait(&bars->g_full, t & 1, abort_flag, status, kErrXElem));
      if (!ok) break;
      tc_fence_after_sync();
#pragma unroll
      for (int h = 0; h < kH; ++h) {
        tmem_ld32(lanes + kG + kHalf * g + 32 * h, r);
        tmem_ld_wait();
        reg_fence32(r);
        float v[32];
#pragma unroll
        for (int j = 0; j < 32; ++j) v[j] = put_back(__uint_as_float(r[j]));
        if (kParts && d > 32) {
          tmem_ld32(lanes + kG + kPartCol + kHalf * g + 32 * h, r);
          tmem_ld_wait();
          reg_fence32(r);
#pragma unroll
          for (int j = 0; j < 32; ++j) v[j] += put_back(__uint_as_float(r[j]));
        }
        const float* z = zs + kHalf * g + 32 * h;
#pragma unroll
        for (int j = 0; j < 32; ++j) {
          const float x = v[j];
          const float y = kKeys ? x + z[j] : fmaf(c, z[j], x) * inv;
          v[j] = ((on[h] >> j) & 1u) ? y : 0.f;
        }
        store_chunk_planes(lanes + kG, kH * g + h, v);
      }
      tmem_st_wait();
      tc_fence_before_sync();
      warp_arrive(&bars->g_ready);
    }
  } else if (warp >= 12) {
    const int et = threadIdx.x - 384;               // token of the tile = TMEM lane
    const uint32_t taddr = tmem + ((32u * (warp & 3)) << 16) + kAcc;
    uint8_t* out = smem + SL::out;
    bool ok = true;
    for (int v = 0; v < kPer * nt; ++v) {
      const int row0 = (t0 + v / kPer) * kTile;
      float s[64];
#pragma unroll
      for (int j = 0; j < 64; ++j) s[j] = 0.f;
      if (ok) ok = drain_tile<NF / 32>(bars, taddr, v, s, abort_flag, status);
      if (et == 0) bulk_wait_group_read0();   // the tile before has left the staging boxes
      named_bar_sync(kBarDrain, 128);
      const bool values = kKeys && (v & 1) == 0;   // dV
      if (ok && sizeof(TG) == 2 && values) {
#pragma unroll
        for (int j = 0; j < 8; ++j)
          *reinterpret_cast<uint4*>(out + swz128(et, j)) =
              make_uint4(pack_bf16x2(put_back(s[8 * j]), put_back(s[8 * j + 1])), pack_bf16x2(put_back(s[8 * j + 2]), put_back(s[8 * j + 3])),
                         pack_bf16x2(put_back(s[8 * j + 4]), put_back(s[8 * j + 5])), pack_bf16x2(put_back(s[8 * j + 6]), put_back(s[8 * j + 7])));
        fence_proxy_async_smem();
      } else if (ok) {
#pragma unroll
        for (int j = 0; j < 16; ++j)
          *reinterpret_cast<float4*>(out + (j >> 3) * kTileBytes + swz128(et, j & 7)) =
              make_float4(put_back(s[4 * j]), put_back(s[4 * j + 1]), put_back(s[4 * j + 2]), put_back(s[4 * j + 3]));
        fence_proxy_async_smem();
      }
      named_bar_sync(kBarDrain, 128);
      if (et == 0 && ok) {   // rows past n and columns past d are clipped
        const CUtensorMap* map = values ? &map_dv : &map_dx;
        for (int c = 0; c < (d > 32 && !(sizeof(TG) == 2 && values) ? 2 : 1); ++c) {
          if (add)
            tma_reduce_add_3d(map, out + c * kTileBytes, 32 * c, row0, slab);
          else
            tma_store_3d(map, out + c * kTileBytes, 32 * c, row0, slab);
        }
        bulk_commit_group();
      }
    }
    if (et == 0) bulk_wait_group0();
  }
  tc_fence_before_sync();
  __syncthreads();
  if (warp == 1) {
    tc_fence_after_sync();
    tmem_dealloc(tmem, 512);
  }
}

// Runs body(T(), NF) with the type of the arguments and the features of a CTA as constants: fp32, or bf16 with 64 features
// (wider bf16 maps: tc_fwd.cu, tc_bwd.cu).
template <int V> struct Int { static constexpr int value = V; };
template <typename F> cudaError_t with_args(const Plan& p, F&& body) {
  if (p.bf16) return p.cfg.features == 64 ? body(__nv_bfloat16(), Int<64>()) : cudaErrorInvalidValue;
  return p.cfg.features == 64 ? body(float(), Int<64>()) : body(float(), Int<128>());
}
int groups_of(const Plan& p) { return p.cfg.features <= kXFeatures ? 1 : p.cfg.features / kXFeatures; }

// S' and z' (or dS' and dz') per chunk from planes of X (the projected operand) and Y (bf16: the tensor itself).
template <bool kScaled>
cudaError_t launch_summary(const Plan& p, const Ws& w, const __nv_bfloat16* x3, const void* y3, const void* W, const float* scale,
                           const float* weight, cudaStream_t st, int* launches) {
  return with_args(p, [&](auto tag, auto nf) {
    using T = decltype(tag);
    constexpr int NF = decltype(nf)::value;
    auto kernel = k_tcx_kside<kScaled, T, NF>;
    CUtensorMap map_x, map_y;
    cudaError_t err;
    if ((err = make_tile_map(x3, 3 * p.slabs, p.cfg.seq_len, &map_x, p.cfg.head_dim)) != cudaSuccess) return err;
    if ((err = make_tile_map(y3, kPlanes<T> * p.slabs, p.cfg.seq_len, &map_y, p.cfg.head_dim)) != cudaSuccess) return err;
    if ((err = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, KxSmem<T>::total)) != cudaSuccess) return err;
    *launches += 1;
    return launch_after(kernel, dim3(p.xchunks, p.slabs, groups_of(p)), dim3(kXThreads), KxSmem<T>::total, st, map_x, map_y,
                        (const T*)W, w.spart, w.zpart, p.cfg.seq_len, p.cfg.head_dim, p.cfg.features, p.xchunk_tiles, w.status,
                        x3, (const int*)(x3 == w.KF3 ? w.seen + 1 : w.seen), scale, weight);
  });
}

template <bool kKeys>
cudaError_t launch_bwd(const Plan& p, const Ws& w, const __nv_bfloat16* x3, const void* y3, const void* W, const float* S,
                       const float* z, float* dx, void* dv, cudaStream_t st, int* launches) {
  return with_args(p, [&](auto tag, auto nf) {
    using T = decltype(tag);
    constexpr int NF = decltype(nf)::value;
    const int n = p.cfg.seq_len, d = p.cfg.head_dim;
    const bool half = kKeys && p.grad_bf16;
    auto kernel = kExact<T> && half ? k_tcx_bwd<kKeys, T, T, NF> : k_tcx_bwd<kKeys, T, float, NF>;   // (bf16 gradients: of bf16 tensors)
    CUtensorMap map_x, map_y, map_dx, map_dv;
    cudaError_t err;
    if (half && !kExact<T>) return cudaErrorInvalidValue;
    if ((err = make_tile_map(x3, 3 * p.slabs, n, &map_x, d)) != cudaSuccess) return err;
    if ((err = make_tile_map(y3, kPlanes<T> * p.slabs, n, &map_y, d)) != cudaSuccess) return err;
    if ((err = make_out_map(dx, p.slabs, n, d, false, &map_dx)) != cudaSuccess) return err;
    if ((err = make_out_map(dv, p.slabs, n, d, half, &map_dv)) != cudaSuccess) return err;
    if ((err = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, YSmem<T>::total)) != cudaSuccess) return err;
    for (int f0 = 0; f0 < p.cfg.features; f0 += NF) {
      *launches += 1;
      err = launch_after(kernel, dim3(p.xbchunks, p.slabs), dim3(kXThreads), YSmem<T>::total, st, map_x, map_y, (const T*)W, S, z,
                         (const float*)w.xinv, (const float*)w.xc, map_dx, map_dv, f0 > 0 ? 1 : 0, n, d, p.cfg.features, f0,
                         p.xbchunk_tiles, w.status, x3, (const int*)(kKeys ? w.seen + 1 : w.seen));
      if (err != cudaSuccess) return err;
    }
    return cudaSuccess;
  });
}

}  // namespace

cudaError_t launch_tcx_kside(const Plan& p, const Ws& w, const void* V, const void* W, cudaStream_t st, int* launches) {
  return launch_summary<false>(p, w, w.KF3, p.bf16 ? V : w.V3, W, nullptr, nullptr, st, launches);
}

cudaError_t launch_tcx_qside(const Plan& p, const Ws& w, const void* W, const float* beta, void* O, cudaStream_t st, int* launches) {
  const int groups = groups_of(p), n = p.cfg.seq_len, d = p.cfg.head_dim;
  const size_t tokens = (size_t)p.slabs * n;
  // Several groups leave their shares where the planes of K_F and V were (which the key side has read), unless a backward
  // reads those again.
  float* share = p.use_xb ? w.xshare : reinterpret_cast<float*>(w.KF3);
  float* den = p.use_xb ? w.xden : groups > 1 ? share + groups * tokens * d : nullptr;
  float* keep = p.use_xb ? w.xO : nullptr;
  void* out = groups == 1 ? O : share;
  const cudaError_t err = with_args(p, [&](auto tag, auto nf) {
    using T = decltype(tag);
    constexpr int NF = decltype(nf)::value;
    auto kernel = k_tcx_qside<T, NF>;
    CUtensorMap map_q, map_o, map_keep;
    cudaError_t e;
    if ((e = make_tile_map(w.QF3, 3 * p.slabs, n, &map_q, d)) != cudaSuccess) return e;
    if ((e = make_out_map(out, groups * p.slabs, n, d, kExact<T>, &map_o)) != cudaSuccess) return e;
    if ((e = make_out_map(keep != nullptr ? keep : out, p.slabs, n, d, keep == nullptr && kExact<T>, &map_keep)) != cudaSuccess) return e;
    if ((e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, QxSmem<T>::total)) != cudaSuccess) return e;
    *launches += 1;
    return launch_after(kernel, dim3(p.xchunks, p.slabs, groups), dim3(kXThreads), QxSmem<T>::total, st, map_q, map_o, (const T*)W,
                        (const float*)w.S, (const float*)w.z, beta, p.cfg.eps, p.cfg.bw_floor, den, map_keep,
                        keep != nullptr && groups == 1 ? 1 : 0, n, d, p.cfg.features, p.xchunk_tiles, w.status,
                        (const __nv_bfloat16*)w.QF3, (const int*)w.seen);
  });
  if (err != cudaSuccess || groups == 1) return err;
  *launches += 1;
  return launch_after(k_tcx_combine, dim3((unsigned)((tokens * (d >> 2) + 255) / 256)), dim3(256), 0, st, (const float*)share,
                      (const float*)den, beta, p.cfg.eps, p.cfg.bw_floor, p.cfg.features, (float*)O, keep, tokens, d);
}

cudaError_t launch_tcx_bwd_prep(const Plan& p, const Ws& w, const void* dO, const float* beta, cudaStream_t st, int* launches) {
  int tpt = 1;
  while (tpt * 8 < p.cfg.head_dim) tpt *= 2;
  *launches += 1;
  auto go = [&](auto kernel, auto* g) {
    return launch_after(kernel, dim3(p.xprep), dim3(256), 0, st, g, (const float*)w.xO, (const float*)w.xden, groups_of(p), beta,
                        p.cfg.eps, p.cfg.bw_floor, p.cfg.features, p.cfg.head_dim, tpt, (size_t)p.slabs * p.cfg.seq_len,
                        p.cfg.seq_len, w.dO3, w.xinv, w.xc, w.sumdD);
  };
  return p.bf16 ? go(k_tcx_bwd_prep<__nv_bfloat16>, (const __nv_bfloat16*)dO) : go(k_tcx_bwd_prep<float>, (const float*)dO);
}

cudaError_t launch_tcx_bwd_qside(const Plan& p, const Ws& w, const void* W, const void* dO, cudaStream_t st, int* launches) {
  const void* y = p.bf16 ? dO : w.dO3;
  const cudaError_t err = launch_bwd<false>(p, w, w.QF3, y, W, w.S, w.z, w.dQF, w.dQF, st, launches);
  if (err != cudaSuccess) return err;
  return launch_summary<true>(p, w, w.QF3, y, W, w.xinv, w.xc, st, launches);
}

cudaError_t launch_tcx_bwd_kside(const Plan& p, const Ws& w, const void* V, const void* W, void* dV, cudaStream_t st, int* launches) {
  return launch_bwd<true>(p, w, w.KF3, p.bf16 ? V : w.V3, W, w.dS, w.dz, w.dKF, dV, st, launches);
}

}  // namespace wersa
