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
//
// Both tensor-core kernels: 512 threads, 128 registers each.  Warp 0 copies, warp 1 issues the projections (MMA1), warp 2
// the contractions (MMA2), warps 4-11 two groups that take the tiles in turn: accumulator -> ReLU -> planes back into
// TMEM; warps 12-15 drain.  TMEM: two buffers of 192 columns (128 of D1, replaced in place by the hi and mid planes, 64 of
// the lo plane), two accumulators of 64.  Every wait is bounded, as in tc_fwd.cu.
// 2 x 8 x 4096, d = 64, m = 256: planes 19 us, key side 28, query side 29, combining 7; the forward 235 -> 95 us.  A tile and
// group takes some 5 k cycles of tensor pipe (MMA1 reads both operands of its 24 instructions from shared memory, 105-115
// cycles each instead of 64; the 48 of MMA2 45 each), 60 % of the time.
#include "common.cuh"
#include "tc_common.cuh"
#include "tc_maps.cuh"

namespace wersa {
using namespace tc;

namespace {

constexpr int kTile = 128;
constexpr uint32_t kTileBytes = kTile * kD * 2;   // one plane of a tile: 128 x 64 bf16
constexpr uint32_t kTileStep = kTileBytes >> 4;   // in descriptor units
constexpr int kXFeatures = 128;                   // features of a CTA
constexpr int kXThreads = 512;
constexpr uint32_t kBufCols = 192, kLoCol = 128, kAccCol = 384;   // TMEM columns
constexpr uint32_t kIdesc1 = make_idesc_bf16(128, 128, false, false);   // both operands K-major
constexpr uint32_t kIdesc2 = make_idesc_bf16(128, 64, false, true);     // B = V or S', N-major
enum { kErrXCopy = 31, kErrXMma = 32, kErrXElem = 33, kErrXDrain = 34 };
enum { kBarZ = 1, kBarDrain = 2 };

// Mean relative loss of a value cut off at 24 bits: half a unit of 2^-23, over the mantissas 1 .. 2 of a value without a
// scale of its own (density 1 / (x ln 2)): 2^-24 / (2 ln 2).
constexpr float kCut = 4.2996e-8f;
__device__ __forceinline__ float put_back(float x) { return fmaf(x, kCut, x); }

// Plane products in the order they are added.
__device__ constexpr int kPa[6] = {2, 0, 1, 1, 0, 0}, kPb[6] = {0, 2, 1, 0, 1, 0};

struct alignas(8) XBars {
  uint64_t x_full[2], x_empty[2], v_full, v_empty, d1_full[2], phi_ready[2], d1_free[2], acc_full[2], acc_free[2], den_free[2];
  uint32_t tmem_base;
  int abort_flag;
};
struct KxSmem {
  static constexpr uint32_t wt = 0;                          // planes of W^T (128 features x 64)
  static constexpr uint32_t x = wt + 3 * kTileBytes;         // two stages of K_F planes
  static constexpr uint32_t v = x + 6 * kTileBytes;          // planes of V
  static constexpr uint32_t sum = v + 3 * kTileBytes;        // S' of the chunk so far: 64 x 128 floats, features side by side
  static constexpr uint32_t zx = sum + 2 * kTileBytes;       // 128 floats
  static constexpr uint32_t bars = zx + 512;
  static constexpr uint32_t total = bars + 256 + 1024;       // + alignment slack
};
struct QxSmem {
  static constexpr uint32_t wt = 0;
  static constexpr uint32_t s = wt + 3 * kTileBytes;         // planes of S' (128 features x 64)
  static constexpr uint32_t x = s + 3 * kTileBytes;          // two stages of Q_F planes
  static constexpr uint32_t out = x + 6 * kTileBytes;        // result tile: two boxes of 128 rows x 32 floats
  static constexpr uint32_t zs = out + 2 * kTileBytes;       // z' of the group
  static constexpr uint32_t den = zs + 512;                  // denominators of two tiles
  static constexpr uint32_t bars = den + 2 * 512;
  static constexpr uint32_t total = bars + 256 + 1024;
};
static_assert(QxSmem::total <= 232448 && KxSmem::total <= 232448 && sizeof(XBars) <= 256, "shared memory of an SM");

// Two floats -> one packed pair per plane.
__device__ __forceinline__ void split3(float a, float b, uint32_t& hi, uint32_t& mid, uint32_t& lo) {
  hi = pack_bf16x2(a, b);
  a -= __uint_as_float(hi << 16);
  b -= __uint_as_float(hi & 0xFFFF0000u);
  mid = pack_bf16x2(a, b);
  a -= __uint_as_float(mid << 16);
  b -= __uint_as_float(mid & 0xFFFF0000u);
  lo = pack_bf16x2(a, b);
}
// Eight floats -> 16-byte chunk `chunk` of row `row` of the three plane tiles at `tile`.
__device__ __forceinline__ void put_planes8(uint8_t* tile, int row, int chunk, const float (&v)[8]) {
  uint32_t p[3][4];
#pragma unroll
  for (int i = 0; i < 4; ++i) split3(v[2 * i], v[2 * i + 1], p[0][i], p[1][i], p[2][i]);
#pragma unroll
  for (int s = 0; s < 3; ++s)
    *reinterpret_cast<uint4*>(tile + s * kTileBytes + swz128(row, chunk)) = make_uint4(p[s][0], p[s][1], p[s][2], p[s][3]);
}
// W (d x m, row-major) -> planes of rows f0 .. f0 + 127 of W^T, zero past column d.  512 threads.
__device__ __forceinline__ void load_w_planes(const float* __restrict__ W, int d, int m, int f0, uint8_t* wt) {
  const int f = threadIdx.x & 127, part = threadIdx.x >> 7;   // 16 columns
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    float v[8];
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      const int c = 16 * part + 8 * h + j;
      v[j] = c < d ? W[(size_t)c * m + f0 + f] : 0.f;
    }
    put_planes8(wt, f, 2 * part + h, v);
  }
}
// S' or dS' of a slab's features f0 .. f0 + 127 (64 columns) -> planes, and the group's z' or dz' -> zs: results of the kernel
// in front (see launch_after).  512 threads.
__device__ __forceinline__ void load_s_planes(const float* S, const float* zg, size_t row0, uint8_t* tile, float* zs) {
  const int f = threadIdx.x >> 2, part = threadIdx.x & 3;   // 16 columns of a feature's row
  const float* src = S + (row0 + f) * kD + 16 * part;
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    const float4 a = __ldcg(reinterpret_cast<const float4*>(src + 8 * h)), b = __ldcg(reinterpret_cast<const float4*>(src + 8 * h + 4));
    const float v[8] = {a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w};
    put_planes8(tile, f, 2 * part + h, v);
  }
  if (threadIdx.x < kXFeatures) zs[threadIdx.x] = __ldcg(zg + row0 + threadIdx.x);
}

// One D1 buffer: 128 fp32 columns -> ReLU -> planes.  32 columns hold 16 hi and 16 mid pairs of their features, the lo pairs
// go to the columns behind them.  Returns the sum of the row's values, kWeighted: each times w[column], in chains of
// eight, as few additions in a row as the FFMA kernels have (two chains of 64: D' 8e-8 off, more than all else together).
template <bool kWeighted>
__device__ __forceinline__ float relu_planes(uint32_t taddr, const float* w) {
  uint32_t r[32];
  float total = 0.f;
#pragma unroll 1
  for (int c = 0; c < 4; ++c) {
    tmem_ld32(taddr + 32 * c, r);
    tmem_ld_wait();
    reg_fence32(r);
    uint32_t hi[16], mid[16], lo[16];
    float e[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
    for (int j = 0; j < 16; ++j) {
      float a = fmaxf(put_back(__uint_as_float(r[2 * j])), 0.f), b = fmaxf(put_back(__uint_as_float(r[2 * j + 1])), 0.f);
      const int k = 2 * (j & 1);
      if constexpr (kWeighted) {
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

// Three planes of one tile.
__device__ __forceinline__ void load_planes(uint8_t* dst, const CUtensorMap* map, int row0, int slab, int slabs, uint64_t* bar) {
  mbar_arrive_expect_tx(bar, 3 * kTileBytes);
#pragma unroll
  for (int pl = 0; pl < 3; ++pl) tma_load_3d(dst + pl * kTileBytes, map, 0, row0, pl * slabs + slab, bar);
}

// D[128 x 128] = A B^T over the head dimension in steps of 16 columns, both operands as planes of 128 rows x 64 columns.
__device__ __forceinline__ void issue_planes(uint32_t dst, uint32_t a_lo, uint32_t b_lo, int ksteps, uint32_t hi) {
#pragma unroll
  for (int q = 0; q < 6; ++q)
#pragma unroll
    for (int k = 0; k < 4; ++k)
      if (k < ksteps)
        mma_ss(dst, smem_desc_join(a_lo + kPa[q] * kTileStep + 2 * k, hi), smem_desc_join(b_lo + kPb[q] * kTileStep + 2 * k, hi),
               kIdesc1, (q > 0 || k > 0) ? 1u : 0u);
}
// MMA1 of every tile.  kXIsA: the tile is A (query side: tokens x features), else W^T is (key side: features x tokens).
template <bool kXIsA>
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
    issue_planes(tmem + b * kBufCols, kXIsA ? x_lo : wt_lo, kXIsA ? wt_lo : x_lo, ksteps, hi);
    mma_commit(&bars->d1_full[b]);
    mma_commit(&bars->x_empty[b]);
  }
}
// The t-th contraction of a CTA, a quarter (32 of the 128 values of K) at a time: accumulator u % 2 (64 columns each, from
// `acc` on) = Phi (planes in the buffer at `buf`) * B (planes of 128 rows x 64 columns at b_lo), u = 4 t + quarter.
template <typename Bars>
__device__ __forceinline__ bool issue_mma2(Bars* bars, uint32_t acc, uint32_t buf, int t, uint32_t b_lo, uint32_t hi,
                                           volatile int* abort_flag, int* status) {
#pragma unroll
  for (int c = 0; c < 4; ++c) {
    const int u = 4 * t + c, r = c & 1;
    if (u >= 2 && !mbar_wait(&bars->acc_free[r], ((u >> 1) - 1) & 1, abort_flag, status, kErrXMma)) return false;
    tc_fence_after_sync();
#pragma unroll
    for (int q = 0; q < 6; ++q)
#pragma unroll
      for (int k = 2 * c; k < 2 * c + 2; ++k)
        mma_ts(acc + 64 * r, buf + phi_col(kPa[q], k), smem_desc_join(b_lo + kPb[q] * kTileStep + 128 * k, hi), kIdesc2,
               (q > 0 || k > 2 * c) ? 1u : 0u);
    mma_commit(&bars->acc_full[r]);
  }
  return true;
}
// s[0 .. 63] += the four quarters of the t-th contraction.  One warp's share (32 lanes); taddr: its lanes, first accumulator.
template <typename Bars>
__device__ __forceinline__ bool drain_tile(Bars* bars, uint32_t taddr, int t, float (&s)[64], volatile int* abort_flag, int* status) {
#pragma unroll 1
  for (int u = 4 * t; u < 4 * t + 4; ++u) {
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
__global__ void __launch_bounds__(kXThreads, 1)
k_tcx_kside(const __grid_constant__ CUtensorMap map_k, const __grid_constant__ CUtensorMap map_v, const float* __restrict__ W,
            float* __restrict__ spart, float* __restrict__ zpart, int n, int d, int m, int chunk_tiles, int* __restrict__ status) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = align_smem(smem_raw);
  using SL = KxSmem;
  XBars* bars = reinterpret_cast<XBars*>(smem + SL::bars);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int chunk = blockIdx.x, slab = blockIdx.y, slabs = gridDim.y, f0 = blockIdx.z * kXFeatures;
  const int t0 = chunk * chunk_tiles, nt = min(chunk_tiles, (n + kTile - 1) / kTile - t0);
  if (threadIdx.x == 0) init_bars(bars);
  if (warp == 1) {
    tmem_alloc(&bars->tmem_base, 512);
    tmem_relinquish();
  }
  load_w_planes(W, d, m, f0, smem + SL::wt);
  fence_proxy_async_smem();
  tc_fence_before_sync();
  __syncthreads();
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
      load_planes(smem + SL::v, &map_v, (t0 + t) * kTile, slab, slabs, &bars->v_full);
      ++vs;
      if (t + 2 < nt) load_x(t + 2);
    }
    if (*abort_flag != 0) {   // let copies in flight land before the CTA's shared memory goes away
      for (int t = max(0, xs - 2); t < xs; ++t) mbar_wait_drain(&bars->x_full[t & 1], (t >> 1) & 1);
      if (vs > 0) mbar_wait_drain(&bars->v_full, (vs - 1) & 1);
    }
  } else if (warp == 1 && lane == 0) {
    issue_mma1<false>(bars, smem + SL::x, smem + SL::wt, tmem, nt, d, abort_flag, status);
  } else if (warp == 2 && lane == 0) {
    const uint32_t hi = smem_desc_hi(1024), v_lo = smem_desc_lo(smem_u32(smem + SL::v), 1024);
    for (int t = 0; t < nt; ++t) {
      if (!mbar_wait(&bars->v_full, t & 1, abort_flag, status, kErrXMma)) break;
      if (!mbar_wait(&bars->phi_ready[t & 1], (t >> 1) & 1, abort_flag, status, kErrXMma)) break;
      if (!issue_mma2(bars, tmem + kAccCol, tmem + (t & 1) * kBufCols, t, v_lo, hi, abort_flag, status)) break;
      mma_commit(&bars->d1_free[t & 1]);
      mma_commit(&bars->v_empty);
    }
  } else if (warp >= 4 && warp < 12) {
    const int g = (warp - 4) >> 2;
    const uint32_t row = 32u * (warp & 3) + lane;   // feature of the group = TMEM lane
    const uint32_t taddr = tmem + ((32u * (warp & 3)) << 16) + g * kBufCols;
    float* zx = reinterpret_cast<float*>(smem + SL::zx);
    float z = 0.f;
    bool ok = true;
    for (int t = g; t < nt && ok; t += 2) {
      ok = __all_sync(0xffffffffu, mbar_wait(&bars->d1_full[g], (t >> 1) & 1, abort_flag, status, kErrXElem));
      if (!ok) break;
      tc_fence_after_sync();
      z += relu_planes<false>(taddr, nullptr);
      tc_fence_before_sync();
      warp_arrive(&bars->phi_ready[g]);
    }
    if (g == 1) zx[row] = z;
    named_bar_sync(kBarZ, 256);
    if (g == 0 && ok) zpart[((size_t)slab * gridDim.x + chunk) * m + f0 + row] = z + zx[row];
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
      ok = drain_tile(bars, taddr, t, s, abort_flag, status);
      if (!ok) break;
#pragma unroll
      for (int j = 0; j < 64; ++j) sum[j * kXFeatures] = t > 0 ? sum[j * kXFeatures] + s[j] : s[j];
    }
    if (ok) {
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
// One group: O, divided.  Several: N'_g into map_o (group-major slabs) and D'_g into den_out[(group * slabs + slab) * n + token].
__global__ void __launch_bounds__(kXThreads, 1)
k_tcx_qside(const __grid_constant__ CUtensorMap map_q, const __grid_constant__ CUtensorMap map_o, const float* __restrict__ W,
            const float* __restrict__ S, const float* __restrict__ zg, const float* __restrict__ beta, float eps, float bw_floor,
            float* __restrict__ den_out, int n, int d, int m, int chunk_tiles, int* __restrict__ status) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = align_smem(smem_raw);
  using SL = QxSmem;
  XBars* bars = reinterpret_cast<XBars*>(smem + SL::bars);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int chunk = blockIdx.x, slab = blockIdx.y, slabs = gridDim.y, f0 = blockIdx.z * kXFeatures;
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
  load_w_planes(W, d, m, f0, smem + SL::wt);
  wait_for_stream_predecessor();
  load_s_planes(S, zg, (size_t)slab * m + f0, smem + SL::s, zs);
  fence_proxy_async_smem();
  tc_fence_before_sync();
  __syncthreads();
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
    issue_mma1<true>(bars, smem + SL::x, smem + SL::wt, tmem, nt, d, abort_flag, status);
  } else if (warp == 2 && lane == 0) {
    const uint32_t hi = smem_desc_hi(1024), s_lo = smem_desc_lo(smem_u32(smem + SL::s), 1024);
    for (int t = 0; t < nt; ++t) {
      if (!mbar_wait(&bars->phi_ready[t & 1], (t >> 1) & 1, abort_flag, status, kErrXMma)) break;
      if (!issue_mma2(bars, tmem + kAccCol, tmem + (t & 1) * kBufCols, t, s_lo, hi, abort_flag, status)) break;
      mma_commit(&bars->d1_free[t & 1]);
    }
  } else if (warp >= 4 && warp < 12) {
    const int g = (warp - 4) >> 2;
    const uint32_t row = 32u * (warp & 3) + lane;   // token of the tile = TMEM lane
    const uint32_t taddr = tmem + ((32u * (warp & 3)) << 16) + g * kBufCols;
    bool ok = true;
    for (int t = g; t < nt && ok; t += 2) {
      ok = __all_sync(0xffffffffu, mbar_wait(&bars->d1_full[g], (t >> 1) & 1, abort_flag, status, kErrXElem));
      if (!ok) break;
      tc_fence_after_sync();
      const float sum = relu_planes<true>(taddr, zs);
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
      if (ok) ok = drain_tile(bars, taddr, t, s, abort_flag, status);
      if (ok) {   // (the tile's denominators are older than its first accumulator)
        const float dn = den[b * kTile + et];
        if (divide) scale = put_back(1.f / (dn + epsp));
        if (den_out != nullptr && row0 + et < n) den_out[(size_t)out_slab * n + row0 + et] = dn;
        warp_arrive(&bars->den_free[b]);
      }
      if (et == 0) bulk_wait_group_read0();   // the tile before has left the staging boxes
      named_bar_sync(kBarDrain, 128);
      if (ok) {
#pragma unroll
        for (int j = 0; j < 16; ++j)
          *reinterpret_cast<float4*>(out + (j >> 3) * kTileBytes + swz128(et, j & 7)) =
              make_float4(s[4 * j] * scale, s[4 * j + 1] * scale, s[4 * j + 2] * scale, s[4 * j + 3] * scale);
        fence_proxy_async_smem();
      }
      named_bar_sync(kBarDrain, 128);
      if (et == 0 && ok) {   // rows past n and columns past d are clipped
        tma_store_3d(&map_o, out, 0, row0, out_slab);
        if (d > 32) tma_store_3d(&map_o, out + kTileBytes, 32, row0, out_slab);
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

// O = (N'_0 + N'_1) / (D'_0 + D'_1 + eps'), one thread per four columns.
__global__ void __launch_bounds__(256) k_tcx_combine(const float* __restrict__ N, const float* __restrict__ den,
                                                     const float* __restrict__ beta, float eps, float bw_floor, int m,
                                                     float* __restrict__ O, size_t tokens, int d) {
  wait_for_stream_predecessor();   // (launched as a programmatic dependent: see launch_after)
  const size_t idx = (size_t)blockIdx.x * 256 + threadIdx.x;
  const int per = d >> 2;
  const size_t tok = idx / per;
  if (tok >= tokens) return;
  const float bw = fmaxf(beta[0], bw_floor);
  const float inv = put_back(1.f / ((load_after_wait(den + tok) + load_after_wait(den + tokens + tok)) + eps * (float)m * bw * bw));
  const float4 a = load4_after_wait(N + idx * 4), b = load4_after_wait(N + tokens * d + idx * 4);
  *reinterpret_cast<float4*>(O + idx * 4) =
      make_float4((a.x + b.x) * inv, (a.y + b.y) * inv, (a.z + b.z) * inv, (a.w + b.w) * inv);
}

}  // namespace

cudaError_t launch_tcx_kside(const Plan& p, const Ws& w, const void* W, cudaStream_t st, int* launches) {
  CUtensorMap map_k, map_v;
  cudaError_t err;
  if ((err = make_tile_map(w.KF3, 3 * p.slabs, p.cfg.seq_len, &map_k, p.cfg.head_dim)) != cudaSuccess) return err;
  if ((err = make_tile_map(w.V3, 3 * p.slabs, p.cfg.seq_len, &map_v, p.cfg.head_dim)) != cudaSuccess) return err;
  if ((err = cudaFuncSetAttribute(k_tcx_kside, cudaFuncAttributeMaxDynamicSharedMemorySize, KxSmem::total)) != cudaSuccess) return err;
  *launches += 1;
  return launch_after(k_tcx_kside, dim3(p.xchunks, p.slabs, p.cfg.features / kXFeatures), dim3(kXThreads), KxSmem::total, st, map_k,
                      map_v, (const float*)W, w.spart, w.zpart, p.cfg.seq_len, p.cfg.head_dim, p.cfg.features, p.xchunk_tiles,
                      w.status);
}

cudaError_t launch_tcx_qside(const Plan& p, const Ws& w, const void* W, const float* beta, void* O, cudaStream_t st, int* launches) {
  const int groups = p.cfg.features / kXFeatures, n = p.cfg.seq_len, d = p.cfg.head_dim;
  const size_t tokens = (size_t)p.slabs * n;
  // several groups leave their shares where the planes of K_F and V were (which the key side has read)
  float* share = groups > 1 ? reinterpret_cast<float*>(w.KF3) : static_cast<float*>(O);
  float* den = groups > 1 ? share + groups * tokens * d : nullptr;
  CUtensorMap map_q, map_o;
  cudaError_t err;
  if ((err = make_tile_map(w.QF3, 3 * p.slabs, n, &map_q, d)) != cudaSuccess) return err;
  if ((err = make_out_map(share, groups * p.slabs, n, d, false, &map_o)) != cudaSuccess) return err;
  if ((err = cudaFuncSetAttribute(k_tcx_qside, cudaFuncAttributeMaxDynamicSharedMemorySize, QxSmem::total)) != cudaSuccess) return err;
  *launches += 1;
  err = launch_after(k_tcx_qside, dim3(p.xchunks, p.slabs, groups), dim3(kXThreads), QxSmem::total, st, map_q, map_o, (const float*)W,
                     w.S, w.z, beta, p.cfg.eps, p.cfg.bw_floor, den, n, d, p.cfg.features, p.xchunk_tiles, w.status);
  if (err != cudaSuccess || groups == 1) return err;
  *launches += 1;
  return launch_after(k_tcx_combine, dim3((unsigned)((tokens * (d >> 2) + 255) / 256)), dim3(256), 0, st, share, den, beta, p.cfg.eps,
                      p.cfg.bw_floor, p.cfg.features, (float*)O, tokens, d);
}

}  // namespace wersa
