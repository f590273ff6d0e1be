// Multi-level Haar analysis -> per-scale gating -> synthesis along the sequence, as one on-chip
// pass over tiles of 256 tokens (Sec. 3.1 steps 3, 5, 6 and Algorithm 2 of the WERSA paper).
//
// Because the Haar detail projector of level l equals blockmean_{2^(l-1)} - blockmean_{2^l} and
// the approximation projector of level L equals blockmean_{2^L}, the filtered signal is
//   T_f x = f_0 x + sum_{i=1..L} (f_i - f_{i-1}) * blockmean_{2^i}(x),
// so one pass needs only the aligned block sums of 2, 4, ..., 2^L rows.  A thread holds 8 consecutive rows of a few
// columns in registers (levels 1-3), partner lanes (a warp covers 32 rows) give levels 4-5 through shuffles, and the
// eight warps exchange their 32-row sums through shared memory around one barrier (levels 6-8, only when L > 5).
// (With the 8-row sums in a pyramid that one thread per column summed up, three barriers and a serial chain stood
// between a tile's loads and its stores; B=4 H=8 n=16384: inner products of Q 55 -> 47 us, dK with products 69 -> 61 us.)
// Rows past the end of the sequence read as zero, which is the zero padding of Algorithm 2.
#include "common.cuh"
#include "gate_backward.cuh"

namespace wersa {
namespace {

struct LevelCoef {
  float f0;
  float k[kMaxLevels + 1];   // k[i] = (f_i - f_{i-1}) / 2^i for 1 <= i <= L, else 0
};

// kOrdered: f is the result of the kernel in front (see launch_after).
template <bool kOrdered = false> __device__ __forceinline__ LevelCoef level_coef(const float* __restrict__ f, int L) {
  float v[kMaxLevels + 1];   // (no load depends on another one or on a branch)
#pragma unroll
  for (int i = 0; i <= kMaxLevels; ++i) {
    const float* p = f + (i <= L ? i : L);
    v[i] = kOrdered ? load_after_wait(p) : *p;
  }
  LevelCoef c;
  c.f0 = v[0];
  float scale = 0.5f;
#pragma unroll
  for (int i = 1; i <= kMaxLevels; ++i) {
    c.k[i] = (i <= L) ? (v[i] - v[i - 1]) * scale : 0.f;
    scale *= 0.5f;
  }
  c.k[0] = 0.f;
  return c;
}

constexpr int kHalfD = kD / 2;
// (kStream: with the evict-first hint, for data that is not read again)
template <bool kStream = false> __device__ __forceinline__ void load4(const float* p, float (&v)[4]) {
  const float4* q = reinterpret_cast<const float4*>(p);
  const float4 a = kStream ? __ldcs(q) : *q;
  v[0] = a.x; v[1] = a.y; v[2] = a.z; v[3] = a.w;
}
template <bool kStream = false> __device__ __forceinline__ void load4(const __nv_bfloat16* p, float (&v)[4]) {
  const uint2* q = reinterpret_cast<const uint2*>(p);
  const uint2 raw = kStream ? __ldcs(q) : *q;
  v[0] = __uint_as_float(raw.x << 16);
  v[1] = __uint_as_float(raw.x & 0xFFFF0000u);
  v[2] = __uint_as_float(raw.y << 16);
  v[3] = __uint_as_float(raw.y & 0xFFFF0000u);
}
__device__ __forceinline__ void store4(float* p, const float (&v)[4]) {
  *reinterpret_cast<float4*>(p) = make_float4(v[0], v[1], v[2], v[3]);
}
__device__ __forceinline__ void store4(__nv_bfloat16* p, const float (&v)[4]) {
  const __nv_bfloat162 a = __floats2bfloat162_rn(v[0], v[1]), b2 = __floats2bfloat162_rn(v[2], v[3]);
  uint2 raw;
  raw.x = *reinterpret_cast<const uint32_t*>(&a);
  raw.y = *reinterpret_cast<const uint32_t*>(&b2);
  *reinterpret_cast<uint2*>(p) = raw;
}


// The transform acts on every column separately, so a CTA of COLS virtual columns (32 or 64) works on
//  * head dimensions of at least COLS: a block of COLS columns of one 256-row tile (d = 64, COLS = 32: two CTAs
//    per tile; columns past d idle), or
//  * narrower heads: COLS / d whole tiles side by side (d = 16, COLS = 32: rows 0-255 in virtual columns 0-15,
//    rows 256-511 in 16-31).
// The kernels take the head dimension 64 as a constant (kFull): with a run-time pitch the row addresses and the
// column map cost registers the 8-row tiles need (k_haar_backward with its output on B=4 H=8 n=16384: 88 against
// 68 us; the pass that writes dQ 49 against 43).
template <int COLS> struct ColMap {
  int row0, col;   // first row of this thread's tile, column in the tensor
  bool on;
  // bx: block index inside the slab, c: the thread's virtual column
  __device__ __forceinline__ ColMap(int bx, int c, int d) {
    if (d >= COLS) {
      const int parts = (d + COLS - 1) / COLS;
      row0 = (bx / parts) * kHaarTile;
      col = (bx % parts) * COLS + c;
      on = col < d;
    } else {
      const int subs = COLS / d, sub = c / d;
      row0 = (bx * subs + sub) * kHaarTile;
      col = c - sub * d;
      on = sub < subs;
    }
  }
};
template <int COLS> int col_blocks(int htiles, int d) {   // blocks per slab
  return d >= COLS ? htiles * ((d + COLS - 1) / COLS) : (htiles + COLS / d - 1) / (COLS / d);
}

// Sum of a value over the 16- and 32-row blocks that contain this thread's 8 rows (lane = 8 (rg & 3) + column group).
__device__ __forceinline__ float sum16(float s3) { return s3 + __shfl_xor_sync(0xffffffffu, s3, 8); }
__device__ __forceinline__ float sum32(float s4) { return s4 + __shfl_xor_sync(0xffffffffu, s4, 16); }
// Weight of warp w's 32-row sum in the levels 6-8 term of warp `own`.
__device__ __forceinline__ float coarse_weight(const LevelCoef& k, int w, int own) {
  return k.k[8] + ((w >> 2) == (own >> 2) ? k.k[7] : 0.f) + ((w >> 1) == (own >> 1) ? k.k[6] : 0.f);
}
// hi[c] += levels 6-8 for columns 4 cg .. + 3 of the exchange rows ex[8][W].
template <int W>
__device__ __forceinline__ void add_coarse4(const float (*ex)[W], const LevelCoef& k, int warp, int col, float* hi) {
#pragma unroll
  for (int w = 0; w < 8; ++w) {
    const float kw = coarse_weight(k, w, warp);
    const float4 v = *reinterpret_cast<const float4*>(&ex[w][col]);
    hi[0] = fmaf(kw, v.x, hi[0]);
    hi[1] = fmaf(kw, v.y, hi[1]);
    hi[2] = fmaf(kw, v.z, hi[2]);
    hi[3] = fmaf(kw, v.w, hi[3]);
  }
}

// Stand-alone filter pass, XF = T_f(X).  The transform acts on every column separately, so one CTA takes
// 256 rows x 32 columns (half of the head dimension), 8 rows x 4 columns per thread: a register tile of
// 32 values lets several CTAs share an SM, so that the loads of one overlap the arithmetic and stores of
// the others (the pass is bound by memory bandwidth).
// With kAddVec every output row of slab s also gets vec[s][:] * vec_scale added (the mean-pool term of dQ); that pass
// goes through the blocks backwards, since the end of its input is what k_haar_backward has left in the L2.
// inputs_ready: X and X2 were complete before the kernel in front of this one passed its wait (see launch_after), and are
// fetched ahead of this one's.  That holds for dQ_F too, and the rows of the pass that writes dQ are on their way while the
// gate backward is still at work.
// place_next: the kernel behind this one may be placed early (see launch_haar_filter).
// grid (col_blocks<32>, slabs, 1 or 2 tensors: X -> XF, X2 -> XF2); block 256.
template <bool kFull, typename Tin, typename Tout, bool kAddVec>
__global__ void __launch_bounds__(256, 4) k_haar_filter(const Tin* __restrict__ X, const float* __restrict__ f,
                                                     Tout* __restrict__ XF, const Tin* __restrict__ X2,
                                                     Tout* __restrict__ XF2, int n, int d_arg, int L,
                                                     const float* __restrict__ vec, float vec_scale, bool inputs_ready,
                                                     bool place_next) {
  // (launched as a programmatic dependent: see launch_after)
  if (!kAddVec && !inputs_ready) wait_for_stream_predecessor();
  const int d = kFull ? kD : d_arg;
  __shared__ __align__(16) float ex[8][kHalfD];   // 32-row sums of the warps
  const int bx = kAddVec ? gridDim.x - 1 - blockIdx.x : blockIdx.x, slab = kAddVec ? gridDim.y - 1 - blockIdx.y : blockIdx.y;
  const int warp = threadIdx.x >> 5, cg = threadIdx.x & 7, rg = threadIdx.x >> 3;
  const ColMap<32> at(bx, cg * 4, d);
  const int row0 = at.row0 + rg * 8;
  const int col0 = at.col;   // first of this thread's four columns
  const int rows = at.on ? n - row0 : 0;   // rows of this thread inside the sequence
  float x[8][4];
  {
    const Tin* xp = (blockIdx.z == 0 ? X : X2) + ((size_t)slab * n + row0) * d + col0;
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      if (j < rows) {
        load4<kAddVec>(xp + (size_t)j * d, x[j]);
      } else {
#pragma unroll
        for (int c = 0; c < 4; ++c) x[j][c] = 0.f;
      }
    }
  }
  if constexpr (!kAddVec) {   // (with the row vector it is the last kernel of its pass, and f is the forward's)
    wait_for_stream_predecessor();
    if (place_next) let_stream_successor_start();
  }
  const LevelCoef k = level_coef<!kAddVec>(f + (size_t)slab * (L + 1), L);
  float hi[4], s5[4];
#pragma unroll
  for (int c = 0; c < 4; ++c) {
    const float s3 = ((x[0][c] + x[1][c]) + (x[2][c] + x[3][c])) + ((x[4][c] + x[5][c]) + (x[6][c] + x[7][c]));
    const float s4 = sum16(s3);
    s5[c] = sum32(s4);
    hi[c] = fmaf(k.k[3], s3, fmaf(k.k[4], s4, k.k[5] * s5[c]));
  }
  if constexpr (kAddVec) {
    wait_for_stream_predecessor();   // the row vector is the gate backward's result
    if (at.on) {
      const float4 v = load4_after_wait(vec + (size_t)slab * kD + col0);
      hi[0] = fmaf(v.x, vec_scale, hi[0]);
      hi[1] = fmaf(v.y, vec_scale, hi[1]);
      hi[2] = fmaf(v.z, vec_scale, hi[2]);
      hi[3] = fmaf(v.w, vec_scale, hi[3]);
    }
  }
  if (L > 5) {
    if ((threadIdx.x & 24) == 0) *reinterpret_cast<float4*>(&ex[warp][cg * 4]) = make_float4(s5[0], s5[1], s5[2], s5[3]);
    __syncthreads();
    add_coarse4(ex, k, warp, cg * 4, hi);
  }
  Tout* dst = (blockIdx.z == 0 ? XF : XF2) + ((size_t)slab * n + row0) * d + col0;
#pragma unroll
  for (int j = 0; j < 8; j += 4) {   // four rows (one level-2 block) at a time
    float y[4][4];
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      const float a0 = x[j][c] + x[j + 1][c], a1 = x[j + 2][c] + x[j + 3][c];
      const float c2 = fmaf(k.k[2], a0 + a1, hi[c]);
      const float c10 = fmaf(k.k[1], a0, c2), c11 = fmaf(k.k[1], a1, c2);
      y[0][c] = fmaf(k.f0, x[j][c], c10);
      y[1][c] = fmaf(k.f0, x[j + 1][c], c10);
      y[2][c] = fmaf(k.f0, x[j + 2][c], c11);
      y[3][c] = fmaf(k.f0, x[j + 3][c], c11);
    }
#pragma unroll
    for (int jj = 0; jj < 4; ++jj)
      if (j + jj < rows) store4(dst + (size_t)(j + jj) * d, y[jj]);
  }
}

// The last pass of a backward with gate weights: dQ = T_f(dQ_F) + d q-bar / n on every row, as k_haar_filter with a row vector, which
// is worked out here: every CTA of a slab takes df (16 numbers), du and the slab's d q-bar (64) for itself while its rows are on
// their way, and the first H + 2 CTAs do what k_gate_backward does for the parameters.  The three launches before were latency from
// end to end, as most of this one is: behind the pass over K and Q 8.4 us and now 5.7 on 5 x 3 x 1777, 7.2 and 5.9 on 2 x 4 x 4096, d = 32,
// 16.5 and 11.9 on 16 x 12 x 1024 (25 MB of dQ_F in, half of it out); and the host has two launches less, 2 us each: training step of 2 x 2 x
// 256, d = 16, m = 256 56.1 -> 53 us.
// kSum: df from the partials of `blocks` CTAs per slab and tensor, else from the reduction's result.
// grid: H + 2 + slabs * blocks.
template <bool kFull, typename Tout, bool kSum>
__global__ void __launch_bounds__(256, 4) k_haar_dq(const float* __restrict__ G, const float* __restrict__ f, Tout* __restrict__ dQ,
                                                    int n, int d_arg, int L, int slabs, int blocks, float inv_n,
                                                    const float* __restrict__ df_in, const float* __restrict__ sg,
                                                    const float* __restrict__ qbar, const float* __restrict__ gate_w,
                                                    const float* __restrict__ omega, const float* __restrict__ sumdD, int n_sumdD,
                                                    const float* __restrict__ beta, float eps, float bw_floor, int m, int B, int H,
                                                    int per_head, float* __restrict__ dbeta, float* __restrict__ dgate_w,
                                                    float* __restrict__ dgate_b, float* __restrict__ domega) {
  // (launched as a programmatic dependent: see launch_after)
  if ((int)blockIdx.x < H + 2) {
    auto wait = []() { wait_for_stream_predecessor(); };
    const GateBwdArgs args = {sg, qbar, gate_w, omega, sumdD, beta, n_sumdD, eps, bw_floor, m, B, H, kFull ? kD : d_arg, L + 1, per_head,
                              dbeta, dgate_w, dgate_b, domega, nullptr};
    if constexpr (kSum) gate_backward_cta<4>(blockIdx.x, SummedDf{df_in, slabs, blocks, L}, args, wait);
    else gate_backward_cta<4>(blockIdx.x, GivenDf{df_in}, args, wait);
    return;
  }
  const int d = kFull ? kD : d_arg;
  __shared__ __align__(16) float ex[8][kHalfD];   // 32-row sums of the warps
  __shared__ float gws[kMaxLevels + 1][kD], red[16][kBandVals + 1], dus[kMaxLevels + 1];
  __shared__ __align__(16) float vec[kD];
  const int at_block = gridDim.x - 1 - blockIdx.x;   // (backwards: see k_haar_filter)
  const int slab = at_block / blocks, bx = at_block - slab * blocks;
  const int tid = threadIdx.x, warp = tid >> 5, cg = tid & 7, rg = tid >> 3;
  const ColMap<32> at(bx, cg * 4, d);
  const int row0 = at.row0 + rg * 8;
  const int col0 = at.col;   // first of this thread's four columns
  const int rows = at.on ? n - row0 : 0;   // rows of this thread inside the sequence
  float x[8][4];
  {
    const float* xp = G + ((size_t)slab * n + row0) * d + col0;
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      if (j < rows) {
        load4<true>(xp + (size_t)j * d, x[j]);
      } else {
#pragma unroll
        for (int c = 0; c < 4; ++c) x[j][c] = 0.f;
      }
    }
  }
  // (gate weights are arguments, f and the sigmoids the forward's)
  const int h = slab % H;
  for (int e = tid; e < d * (L + 1); e += 256) {
    const int c = e / (L + 1);
    gws[e - c * (L + 1)][c] = gate_w[(size_t)h * d * (L + 1) + e];
  }
  float slope = 0.f;
  if (tid <= L) {
    const float sgm = sg[(size_t)slab * (L + 1) + tid];
    slope = omega[tid] * sgm * (1.f - sgm) * inv_n;
  }
  const LevelCoef k = level_coef(f + (size_t)slab * (L + 1), L);
  float hi[4], s5[4];
#pragma unroll
  for (int c = 0; c < 4; ++c) {
    const float s3 = ((x[0][c] + x[1][c]) + (x[2][c] + x[3][c])) + ((x[4][c] + x[5][c]) + (x[6][c] + x[7][c]));
    const float s4 = sum16(s3);
    s5[c] = sum32(s4);
    hi[c] = fmaf(k.k[3], s3, fmaf(k.k[4], s4, k.k[5] * s5[c]));
  }
  if (L > 5 && (tid & 24) == 0) *reinterpret_cast<float4*>(&ex[warp][cg * 4]) = make_float4(s5[0], s5[1], s5[2], s5[3]);
  wait_for_stream_predecessor();
  {
    // df: slot j by sixteen threads; the gate of a batch element sums over its heads
    const int j = tid & (kBandVals - 1), pt = tid >> 4;
    const int first = per_head ? slab : slab - h, count = per_head ? 1 : H;
    float s = 0.f;
    if (j <= L) {
      if constexpr (kSum) {
        const float* src = df_in + (j < L ? j : 8 + L - 1);
        const int all = count * blocks;   // of one tensor: the partials of neighbouring slabs lie side by side
        for (int t = pt; t < all; t += 48) {   // (three at a time: see haar_dq_sums_bands)
          float v[6];
#pragma unroll
          for (int e = 0; e < 3; ++e) {
            const float* q = src + ((size_t)first * blocks + min(t + 16 * e, all - 1)) * kBandVals;
            v[2 * e] = __ldcg(q);
            v[2 * e + 1] = __ldcg(q + (size_t)slabs * blocks * kBandVals);
          }
#pragma unroll
          for (int e = 0; e < 3; ++e) s += t + 16 * e < all ? v[2 * e] + v[2 * e + 1] : 0.f;
        }
      } else {
        for (int t = pt; t < count; t += 16) s += __ldcg(df_in + (size_t)(first + t) * kBandVals + j);
      }
    }
    red[pt][j] = s;
    __syncthreads();
    if (tid <= L) {
      float df = 0.f;
#pragma unroll
      for (int q = 0; q < 16; ++q) df += red[q][tid];
      dus[tid] = df * slope;
    }
    __syncthreads();
    if (tid < d) {
      float v = 0.f;
      for (int i = 0; i <= L; ++i) v = fmaf(gws[i][tid], dus[i], v);
      vec[tid] = v;
    }
    __syncthreads();
  }
  if (at.on) {
    const float4 v = *reinterpret_cast<const float4*>(&vec[col0]);
    hi[0] += v.x;
    hi[1] += v.y;
    hi[2] += v.z;
    hi[3] += v.w;
  }
  if (L > 5) add_coarse4(ex, k, warp, cg * 4, hi);
  Tout* dst = dQ + ((size_t)slab * n + row0) * d + col0;
#pragma unroll
  for (int j = 0; j < 8; j += 4) {   // four rows (one level-2 block) at a time
    float y[4][4];
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      const float a0 = x[j][c] + x[j + 1][c], a1 = x[j + 2][c] + x[j + 3][c];
      const float c2 = fmaf(k.k[2], a0 + a1, hi[c]);
      const float c10 = fmaf(k.k[1], a0, c2), c11 = fmaf(k.k[1], a1, c2);
      y[0][c] = fmaf(k.f0, x[j][c], c10);
      y[1][c] = fmaf(k.f0, x[j + 1][c], c10);
      y[2][c] = fmaf(k.f0, x[j + 2][c], c11);
      y[3][c] = fmaf(k.f0, x[j + 3][c], c11);
    }
#pragma unroll
    for (int jj = 0; jj < 4; ++jj)
      if (j + jj < rows) store4(dst + (size_t)(j + jj) * d, y[jj]);
  }
}

// What the fp32 kernels of the tensor cores read: T_f(Q), T_f(K) and V as three bf16 planes hi, mid, lo each (their sum
// carries the fp32 value; see k_haar_filter_split3), and for a backward that will want them T_f(Q) and T_f(K) themselves.
// Tiles and arithmetic are those of k_haar_filter; all three tensors are arguments and fetched ahead of the wait.  Bound by
// memory: 640 bytes a row of 64 columns and tensor, 2 x 8 x 4096 19 us, 6.6 TB/s.
// grid (col_blocks<32>, slabs, 3; of bf16 tensors 2: V is its own plane), block 256.
template <bool kFull, bool kKeep, typename Tin>
__global__ void __launch_bounds__(256, 3) k_f32_planes(const Tin* __restrict__ Q, const Tin* __restrict__ K,
                                                       const Tin* __restrict__ V, const float* __restrict__ f,
                                                       __nv_bfloat16* __restrict__ Q3, __nv_bfloat16* __restrict__ K3,
                                                       __nv_bfloat16* __restrict__ V3, float* __restrict__ QF,
                                                       float* __restrict__ KF, size_t plane, int n, int d_arg, int L,
                                                       int* __restrict__ seen) {
  const int d = kFull ? kD : d_arg;
  __shared__ __align__(16) float ex[8][kHalfD];   // 32-row sums of the warps
  const int slab = blockIdx.y, warp = threadIdx.x >> 5, cg = threadIdx.x & 7, rg = threadIdx.x >> 3;
  const ColMap<32> at(blockIdx.x, cg * 4, d);
  const int row0 = at.row0 + rg * 8;
  const int rows = at.on ? n - row0 : 0;   // rows of this thread inside the sequence
  const size_t first = ((size_t)slab * n + row0) * d + at.col;
  const bool filtered = blockIdx.z < 2;
  const Tin* __restrict__ X = blockIdx.z == 0 ? Q : blockIdx.z == 1 ? K : V;
  float x[8][4];
#pragma unroll
  for (int j = 0; j < 8; ++j) {
    if (j < rows) {
      load4<true>(X + first + (size_t)j * d, x[j]);
    } else {
#pragma unroll
      for (int c = 0; c < 4; ++c) x[j][c] = 0.f;
    }
  }
  wait_for_stream_predecessor();   // (launched as a programmatic dependent, see launch_after: f is the gate kernel's)
  let_stream_successor_start();
  if (filtered) {
    const LevelCoef k = level_coef<true>(f + (size_t)slab * (L + 1), L);
    float hi[4], s5[4];
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      const float s3 = ((x[0][c] + x[1][c]) + (x[2][c] + x[3][c])) + ((x[4][c] + x[5][c]) + (x[6][c] + x[7][c]));
      const float s4 = sum16(s3);
      s5[c] = sum32(s4);
      hi[c] = fmaf(k.k[3], s3, fmaf(k.k[4], s4, k.k[5] * s5[c]));
    }
    if (L > 5) {
      if ((threadIdx.x & 24) == 0) *reinterpret_cast<float4*>(&ex[warp][cg * 4]) = make_float4(s5[0], s5[1], s5[2], s5[3]);
      __syncthreads();
      add_coarse4(ex, k, warp, cg * 4, hi);
    }
#pragma unroll
    for (int j = 0; j < 8; j += 4) {   // four rows (one level-2 block) at a time
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        const float a0 = x[j][c] + x[j + 1][c], a1 = x[j + 2][c] + x[j + 3][c];
        const float c2 = fmaf(k.k[2], a0 + a1, hi[c]);
        const float c10 = fmaf(k.k[1], a0, c2), c11 = fmaf(k.k[1], a1, c2);
        x[j][c] = fmaf(k.f0, x[j][c], c10);
        x[j + 1][c] = fmaf(k.f0, x[j + 1][c], c10);
        x[j + 2][c] = fmaf(k.f0, x[j + 2][c], c11);
        x[j + 3][c] = fmaf(k.f0, x[j + 3][c], c11);
      }
    }
  }
  __nv_bfloat16* dst = (blockIdx.z == 0 ? Q3 : blockIdx.z == 1 ? K3 : V3) + first;
  float* keep = blockIdx.z == 0 ? QF : KF;
  uint32_t top = 0;   // not 0: a value that is not finite, or above the largest bf16
#pragma unroll
  for (int j = 0; j < 8; ++j) {
    if (j >= rows) break;
    if (kKeep && filtered) store4(keep + first + (size_t)j * d, x[j]);
#pragma unroll
    for (int pl = 0; pl < 3; ++pl) {   // what a plane leaves is the next one's input
      auto plane_of = [](float x0, float x1, float x2, float x3) {
        const __nv_bfloat162 a = __floats2bfloat162_rn(x0, x1), b = __floats2bfloat162_rn(x2, x3);
        return make_uint2(*reinterpret_cast<const uint32_t*>(&a), *reinterpret_cast<const uint32_t*>(&b));
      };
      uint2 w = plane_of(x[j][0], x[j][1], x[j][2], x[j][3]);
      if (pl == 0) {
        const uint32_t t = full_exponents(w.x) | full_exponents(w.y);
        if (t != 0) w = plane_of(bf16_range(x[j][0]), bf16_range(x[j][1]), bf16_range(x[j][2]), bf16_range(x[j][3]));
        top |= t;
      }
      *reinterpret_cast<uint2*>(dst + (size_t)pl * plane + (size_t)j * d) = w;
      x[j][0] -= __uint_as_float(w.x << 16);
      x[j][1] -= __uint_as_float(w.x & 0xFFFF0000u);
      x[j][2] -= __uint_as_float(w.y << 16);
      x[j][3] -= __uint_as_float(w.y & 0xFFFF0000u);
    }
  }
  if (filtered && top != 0) seen[blockIdx.z] = 1;   // (who multiplies by W wants to know: see Operands)
}

// The same pass for bf16 input: a thread keeps its 8 rows x 8 columns as the 32 packed words it loaded
// (16-byte loads; unpacked where they are used, twice), so that three CTAs of 256 rows x 64 columns share an
// SM with 16-byte accesses in flight.  grid (htiles, slabs), block 256.
__device__ __forceinline__ float bf_lo(uint32_t u) { return __uint_as_float(u << 16); }
__device__ __forceinline__ float bf_hi(uint32_t u) { return __uint_as_float(u & 0xFFFF0000u); }

// Keeps the compiler from carrying unpacked rows from one use to the next (64 registers).
__device__ __forceinline__ void rows_fence(uint32_t (&u)[8][4]) {
#pragma unroll
  for (int q = 0; q < 8; ++q) asm volatile("" : "+r"(u[q][0]), "+r"(u[q][1]), "+r"(u[q][2]), "+r"(u[q][3]));
}
// Coarse part of a thread's 8 rows x 8 columns (packed rows u): hi[c] = sum_{l=3..8} k_l s_l.
__device__ __forceinline__ void packed_coarse(const uint32_t (&u)[8][4], const LevelCoef& k, int L, float (*ex)[kD],
                                              float (&hi)[8]) {
  const int warp = threadIdx.x >> 5, cg = threadIdx.x & 7;
  float s5[8];
#pragma unroll
  for (int c = 0; c < 8; ++c) {
    float s3 = 0.f;
#pragma unroll
    for (int j = 0; j < 8; j += 2)   // pairs first, as the other kernels add them
      s3 += (c & 1) ? bf_hi(u[j][c >> 1]) + bf_hi(u[j + 1][c >> 1]) : bf_lo(u[j][c >> 1]) + bf_lo(u[j + 1][c >> 1]);
    const float s4 = sum16(s3);
    s5[c] = sum32(s4);
    hi[c] = fmaf(k.k[3], s3, fmaf(k.k[4], s4, k.k[5] * s5[c]));
  }
  if (L <= 5) return;
  if ((threadIdx.x & 24) == 0) {
    *reinterpret_cast<float4*>(&ex[warp][cg * 8]) = make_float4(s5[0], s5[1], s5[2], s5[3]);
    *reinterpret_cast<float4*>(&ex[warp][cg * 8 + 4]) = make_float4(s5[4], s5[5], s5[6], s5[7]);
  }
  __syncthreads();
  add_coarse4(ex, k, warp, cg * 8, hi);
  add_coarse4(ex, k, warp, cg * 8 + 4, hi + 4);
}

template <bool kFull, typename Tout>
__global__ void __launch_bounds__(256, 3) k_haar_filter_bf16(const __nv_bfloat16* __restrict__ X,
                                                             const float* __restrict__ f, Tout* __restrict__ XF,
                                                             const __nv_bfloat16* __restrict__ X2,
                                                             Tout* __restrict__ XF2, int n, int d_arg, int L,
                                                             bool inputs_ready, bool place_next) {
  if (!inputs_ready) wait_for_stream_predecessor();   // (launched as a programmatic dependent: see launch_after)
  const int d = kFull ? kD : d_arg;
  __shared__ __align__(16) float ex[8][kD];   // 32-row sums of the warps
  const int slab = blockIdx.y;
  const int cg = threadIdx.x & 7, rg = threadIdx.x >> 3;
  const ColMap<64> at(blockIdx.x, cg * 8, d);
  const int row0 = at.row0 + rg * 8;
  const int rows = at.on ? n - row0 : 0;   // rows of this thread inside the sequence
  uint32_t u[8][4];
  {
    const __nv_bfloat16* xp = (blockIdx.z == 0 ? X : X2) + ((size_t)slab * n + row0) * d + at.col;
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      uint4 raw = make_uint4(0u, 0u, 0u, 0u);
      if (j < rows) raw = *reinterpret_cast<const uint4*>(xp + (size_t)j * d);
      u[j][0] = raw.x; u[j][1] = raw.y; u[j][2] = raw.z; u[j][3] = raw.w;
    }
  }
  wait_for_stream_predecessor();   // f may be the gate kernel's result
  if (place_next) let_stream_successor_start();
  const LevelCoef k = level_coef<true>(f + (size_t)slab * (L + 1), L);
  float hi[8];
  packed_coarse(u, k, L, ex, hi);
  rows_fence(u);
  Tout* dst = (blockIdx.z == 0 ? XF : XF2) + ((size_t)slab * n + row0) * d + at.col;
  if constexpr (sizeof(Tout) == 2) {
    // bf16 out: the results replace the packed inputs column pair by column pair, rows are stored whole
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const float h0 = hi[2 * i], h1 = hi[2 * i + 1];
#pragma unroll
      for (int j = 0; j < 8; j += 4) {
        float y[4][2];
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const float x0 = h ? bf_hi(u[j][i]) : bf_lo(u[j][i]), x1 = h ? bf_hi(u[j + 1][i]) : bf_lo(u[j + 1][i]);
          const float x2 = h ? bf_hi(u[j + 2][i]) : bf_lo(u[j + 2][i]), x3 = h ? bf_hi(u[j + 3][i]) : bf_lo(u[j + 3][i]);
          const float a0 = x0 + x1, a1 = x2 + x3;
          const float c2 = fmaf(k.k[2], a0 + a1, h ? h1 : h0);
          const float c10 = fmaf(k.k[1], a0, c2), c11 = fmaf(k.k[1], a1, c2);
          y[0][h] = fmaf(k.f0, x0, c10);
          y[1][h] = fmaf(k.f0, x1, c10);
          y[2][h] = fmaf(k.f0, x2, c11);
          y[3][h] = fmaf(k.f0, x3, c11);
        }
#pragma unroll
        for (int jj = 0; jj < 4; ++jj) {
          const __nv_bfloat162 pk = __floats2bfloat162_rn(y[jj][0], y[jj][1]);
          u[j + jj][i] = *reinterpret_cast<const uint32_t*>(&pk);
        }
      }
    }
#pragma unroll
    for (int j = 0; j < 8; ++j)
      if (j < rows)
        *reinterpret_cast<uint4*>(dst + (size_t)j * d) = make_uint4(u[j][0], u[j][1], u[j][2], u[j][3]);
  } else {
#pragma unroll
    for (int j = 0; j < 8; j += 4) {   // four rows (one level-2 block) at a time
      float y[4][8];
#pragma unroll
      for (int i = 0; i < 4; ++i) {
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const int c = 2 * i + h;
          const float x0 = h ? bf_hi(u[j][i]) : bf_lo(u[j][i]), x1 = h ? bf_hi(u[j + 1][i]) : bf_lo(u[j + 1][i]);
          const float x2 = h ? bf_hi(u[j + 2][i]) : bf_lo(u[j + 2][i]), x3 = h ? bf_hi(u[j + 3][i]) : bf_lo(u[j + 3][i]);
          const float a0 = x0 + x1, a1 = x2 + x3;
          const float c2 = fmaf(k.k[2], a0 + a1, hi[c]);
          const float c10 = fmaf(k.k[1], a0, c2), c11 = fmaf(k.k[1], a1, c2);
          y[0][c] = fmaf(k.f0, x0, c10);
          y[1][c] = fmaf(k.f0, x1, c10);
          y[2][c] = fmaf(k.f0, x2, c11);
          y[3][c] = fmaf(k.f0, x3, c11);
        }
      }
#pragma unroll
      for (int jj = 0; jj < 4; ++jj)
        if (j + jj < rows) store8(dst + (size_t)(j + jj) * d, y[jj]);
    }
  }
}

// The same filter with the result written as three bf16 planes hi + mid + lo (each slabs x n x d):
// hi = bf16(x), mid = bf16(x - hi), lo = bf16(x - hi - mid), so that their sum carries the fp32
// value (24 mantissa bits) into bf16 tensor-core products.  The backward kernels need that: the
// ReLU mask 1[a > 0] of a = X_F W must not flip through the rounding of X_F.
// The rows stay the packed words they were loaded as (three CTAs per SM; with the unpacked 8 x 8 tile in registers two:
// B=4 H=8 n=16384, both tensors 120 -> 90 us, 6.0 TB/s).  With S one more layer of the grid leaves the low-order image of
// S' that the query side takes beside bf16(S').  grid (col_blocks<64>, slabs, 1 or 2 tensors [+ 1]), block 256.
template <bool kFull>
__global__ void __launch_bounds__(256, 3) k_haar_filter_split3(const __nv_bfloat16* __restrict__ X,
                                                               const float* __restrict__ f,
                                                               __nv_bfloat16* __restrict__ XF3,
                                                               const __nv_bfloat16* __restrict__ X2,
                                                               __nv_bfloat16* __restrict__ XF3_2, size_t plane, int n,
                                                               int d_arg, int L, const float* __restrict__ S,
                                                               const __nv_bfloat16* __restrict__ Sbf,
                                                               __nv_bfloat16* __restrict__ Slo, int features, int groups) {
  wait_for_stream_predecessor();   // (launched as a programmatic dependent: see launch_after)
  let_stream_successor_start();
  if (S != nullptr && blockIdx.z == gridDim.z - 1) {   // the last layer of the grid: Slo = bf16(S - Sbf)
    const int per = features * kD;   // of one group (S has a slab's features together, Sbf and Slo a group's slabs)
    for (int i = (blockIdx.x * 256 + threadIdx.x) * 4; i < per * groups; i += gridDim.x * 1024) {
      const int g = i / per;
      const size_t o = ((size_t)g * gridDim.y + blockIdx.y) * per + (i - g * per);
      const float4 v = *reinterpret_cast<const float4*>(S + (size_t)blockIdx.y * per * groups + i);
      const uint2 h = *reinterpret_cast<const uint2*>(Sbf + o);
      const __nv_bfloat162 a = __floats2bfloat162_rn(v.x - bf_lo(h.x), v.y - bf_hi(h.x));
      const __nv_bfloat162 b = __floats2bfloat162_rn(v.z - bf_lo(h.y), v.w - bf_hi(h.y));
      *reinterpret_cast<uint2*>(Slo + o) =
          make_uint2(*reinterpret_cast<const uint32_t*>(&a), *reinterpret_cast<const uint32_t*>(&b));
    }
    return;
  }
  const int d = kFull ? kD : d_arg;
  __shared__ __align__(16) float ex[8][kD];   // 32-row sums of the warps
  const int slab = blockIdx.y;
  const int cg = threadIdx.x & 7, rg = threadIdx.x >> 3;
  const ColMap<64> at(blockIdx.x, cg * 8, d);
  const int row0 = at.row0 + rg * 8;
  const int rows = at.on ? n - row0 : 0;   // rows of this thread inside the sequence
  const LevelCoef k = level_coef(f + (size_t)slab * (L + 1), L);
  uint32_t u[8][4];
  {
    const __nv_bfloat16* xp = (blockIdx.z == 0 ? X : X2) + ((size_t)slab * n + row0) * d + at.col;
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      uint4 raw = make_uint4(0u, 0u, 0u, 0u);
      if (j < rows) raw = *reinterpret_cast<const uint4*>(xp + (size_t)j * d);
      u[j][0] = raw.x; u[j][1] = raw.y; u[j][2] = raw.z; u[j][3] = raw.w;
    }
  }
  float hi[8];
  packed_coarse(u, k, L, ex, hi);
  __nv_bfloat16* dst = (blockIdx.z == 0 ? XF3 : XF3_2) + ((size_t)slab * n + row0) * d + at.col;
#pragma unroll
  for (int j = 0; j < 8; ++j) {   // a row at a time; what a plane leaves is the next one's input
    rows_fence(u);
    float y[8];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int p = j & ~1, o = p ^ 2;   // the row's pair and the other pair of its block of four
        const float xj = h ? bf_hi(u[j][i]) : bf_lo(u[j][i]);
        const float a0 = (h ? bf_hi(u[p][i]) : bf_lo(u[p][i])) + (h ? bf_hi(u[p + 1][i]) : bf_lo(u[p + 1][i]));
        const float a1 = (h ? bf_hi(u[o][i]) : bf_lo(u[o][i])) + (h ? bf_hi(u[o + 1][i]) : bf_lo(u[o + 1][i]));
        y[2 * i + h] = k.f0 * xj + k.k[1] * a0 + k.k[2] * (a0 + a1) + hi[2 * i + h];
      }
    }
    if (j >= rows) continue;
    __nv_bfloat16* row = dst + (size_t)j * d;
#pragma unroll
    for (int pl = 0; pl < 3; ++pl) {
      uint32_t w[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const __nv_bfloat162 pk = __floats2bfloat162_rn(y[2 * i], y[2 * i + 1]);
        w[i] = *reinterpret_cast<const uint32_t*>(&pk);
        y[2 * i] -= bf_lo(w[i]);
        y[2 * i + 1] -= bf_hi(w[i]);
      }
      *reinterpret_cast<uint4*>(row + (size_t)pl * plane) = make_uint4(w[0], w[1], w[2], w[3]);
    }
  }
}

// Backward of the filter for one tile: dX = T_f(G) (the operator is symmetric) and the band
// inner products of (G, X) that give df:
//   slot l-1 (l = 1..8): sum over blocks of Delta_l(G) * Delta_l(X) / 2^l, the product of the
//                        level-l detail coefficients (Delta_l = left half sum - right half sum);
//   slot 8+l-1:          sum over blocks of s_l(G) * s_l(X) / 2^l, the product of the level-l
//                        approximation coefficients.
// The transform acts on every column separately, so one CTA takes 256 rows x 32 columns (half of the
// head dimension): 8 rows x 4 columns per thread, a small register tile (several CTAs per SM keep loads,
// arithmetic and stores of different tiles overlapped).  G and X are loaded together, X, which nobody reads again, with
// the streaming hint (16 x 12 x 1024: 46.6 -> 44.5 us, and G of the second tensor stays in the L2 for the dQ pass).
// Levels 1-3 come from the register tiles, 4-5 from shuffles (every lane of a block adds its equal share of the product), 6-8 from the warps'
// 32-row sums: the lanes of warp 0, one per column, add the products, every thread the coarse part of its output rows.
// grid (col_blocks<32>, slabs, 1 or 2 tensors: X, G -> dX, bands `which`; X2, G2 -> dX2, the other half of the bands); one
// band partial per CTA.  A null dX is not written (only the band inner products are wanted); kWrite = false says so for
// all of the launch and takes half the registers.
template <bool kFull, typename Tin, typename Tout, bool kWrite>
__global__ void __launch_bounds__(256, kWrite ? 2 : 4)
k_haar_backward(const Tin* __restrict__ X1, const float* __restrict__ G1, Tout* __restrict__ dX1,
                const Tin* __restrict__ X2, const float* __restrict__ G2, Tout* __restrict__ dX2,
                const float* __restrict__ f, float* __restrict__ bands, int which, int n, int d_arg, int L) {
  wait_for_stream_predecessor();   // (launched as a programmatic dependent: see launch_after)
  let_stream_successor_start();
  const bool second = blockIdx.z != 0;
  const Tin* __restrict__ X = second ? X2 : X1;
  const float* __restrict__ G = second ? G2 : G1;
  Tout* __restrict__ dX = second ? dX2 : dX1;
  const int d = kFull ? kD : d_arg;
  __shared__ __align__(16) float ex[2][8][kHalfD];   // 32-row sums of the warps: [0] = G, [1] = X
  __shared__ float red[8][kBandVals];
  const int slab = blockIdx.y;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int cg = threadIdx.x & 7, rg = threadIdx.x >> 3;
  const ColMap<32> at(blockIdx.x, cg * 4, d);
  const int row0 = at.row0 + rg * 8;
  const int rows = at.on ? n - row0 : 0;   // rows of this thread inside the sequence
  float acc[kBandVals];
#pragma unroll
  for (int i = 0; i < kBandVals; ++i) acc[i] = 0.f;
  float g[8][4], gs[4], hi[4];
  {
    float x[8][4];
    const float* gp = G + ((size_t)slab * n + row0) * d + at.col;
    const Tin* xp = X + ((size_t)slab * n + row0) * d + at.col;
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      if (j < rows) {
        load4(gp + (size_t)j * d, g[j]);
        load4<true>(xp + (size_t)j * d, x[j]);
      } else {
#pragma unroll
        for (int c = 0; c < 4; ++c) g[j][c] = x[j][c] = 0.f;
      }
    }
    const LevelCoef k = level_coef(f + (size_t)slab * (L + 1), L);
    float xs[4];
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      float g1[4], x1[4];
#pragma unroll
      for (int p = 0; p < 4; ++p) {
        g1[p] = g[2 * p][c] + g[2 * p + 1][c];
        x1[p] = x[2 * p][c] + x[2 * p + 1][c];
        acc[0] += (g[2 * p][c] - g[2 * p + 1][c]) * (x[2 * p][c] - x[2 * p + 1][c]);
        acc[8] += g1[p] * x1[p];
      }
      const float g20 = g1[0] + g1[1], g21 = g1[2] + g1[3], x20 = x1[0] + x1[1], x21 = x1[2] + x1[3];
      acc[1] += (g1[0] - g1[1]) * (x1[0] - x1[1]) + (g1[2] - g1[3]) * (x1[2] - x1[3]);
      acc[9] += g20 * x20 + g21 * x21;
      const float g3 = g20 + g21, x3 = x20 + x21;
      acc[2] += (g20 - g21) * (x20 - x21);
      acc[10] += g3 * x3;
      const float g3o = __shfl_xor_sync(0xffffffffu, g3, 8), x3o = __shfl_xor_sync(0xffffffffu, x3, 8);
      const float g4 = g3 + g3o, x4 = x3 + x3o;
      acc[3] += 0.5f * (g3 - g3o) * (x3 - x3o);
      acc[11] += 0.5f * g4 * x4;
      const float g4o = __shfl_xor_sync(0xffffffffu, g4, 16), x4o = __shfl_xor_sync(0xffffffffu, x4, 16);
      gs[c] = g4 + g4o;
      xs[c] = x4 + x4o;
      acc[4] += 0.25f * (g4 - g4o) * (x4 - x4o);
      acc[12] += 0.25f * gs[c] * xs[c];
      if constexpr (kWrite) hi[c] = fmaf(k.k[3], g3, fmaf(k.k[4], g4, k.k[5] * gs[c]));
    }
    if (L > 5) {
      if (lane < 8) {
        *reinterpret_cast<float4*>(&ex[0][warp][cg * 4]) = make_float4(gs[0], gs[1], gs[2], gs[3]);
        *reinterpret_cast<float4*>(&ex[1][warp][cg * 4]) = make_float4(xs[0], xs[1], xs[2], xs[3]);
      }
      __syncthreads();
      if (warp == 0) {   // lane = column
        float a[8], b[8];
#pragma unroll
        for (int w = 0; w < 8; ++w) {
          a[w] = ex[0][w][lane];
          b[w] = ex[1][w][lane];
        }
#pragma unroll
        for (int l = 5; l < 8; ++l) {   // levels 6, 7, 8: pairs of what is left
#pragma unroll
          for (int w = 0; w < (128 >> l); ++w) {
            acc[l] += (a[2 * w] - a[2 * w + 1]) * (b[2 * w] - b[2 * w + 1]);
            a[w] = a[2 * w] + a[2 * w + 1];
            b[w] = b[2 * w] + b[2 * w + 1];
            acc[8 + l] += a[w] * b[w];
          }
        }
      }
      if constexpr (kWrite) add_coarse4(ex[0], k, warp, cg * 4, hi);
    }
    if (kWrite && dX != nullptr) {
      Tout* dst = dX + ((size_t)slab * n + row0) * d + at.col;
#pragma unroll
      for (int j = 0; j < 8; j += 4) {   // four rows (one level-2 block) at a time
        float y[4][4];
#pragma unroll
        for (int c = 0; c < 4; ++c) {
          const float a0 = g[j][c] + g[j + 1][c], a1 = g[j + 2][c] + g[j + 3][c];
          const float c2 = fmaf(k.k[2], a0 + a1, hi[c]);
          const float c10 = fmaf(k.k[1], a0, c2), c11 = fmaf(k.k[1], a1, c2);
          y[0][c] = fmaf(k.f0, g[j][c], c10);
          y[1][c] = fmaf(k.f0, g[j + 1][c], c10);
          y[2][c] = fmaf(k.f0, g[j + 2][c], c11);
          y[3][c] = fmaf(k.f0, g[j + 3][c], c11);
        }
#pragma unroll
        for (int jj = 0; jj < 4; ++jj)
          if (j + jj < rows) store4(dst + (size_t)(j + jj) * d, y[jj]);
      }
    }
  }
  // Sums over the warp: in four steps a lane passes on half of the values it still holds, so that each ends up with
  // one of the sixteen; the 1 / 2^l normalisation rides on the last one.
#pragma unroll
  for (int s = 8, o = 16; s >= 1; s >>= 1, o >>= 1) {
    const bool up = (lane & o) != 0;
#pragma unroll
    for (int i = 0; i < s; ++i) {
      const float keep = up ? acc[i + s] : acc[i], send = up ? acc[i] : acc[i + s];
      acc[i] = keep + __shfl_xor_sync(0xffffffffu, send, o);
    }
  }
  const int slot = lane >> 1;   // bits 16, 8, 4, 2 of the lane chose 8, 4, 2, 1
  const float v = acc[0] + __shfl_xor_sync(0xffffffffu, acc[0], 1);
  if ((lane & 1) == 0) red[warp][slot] = v * (1.f / (float)(2 << (slot & 7)));
  __syncthreads();
  if (threadIdx.x < kBandVals) {
    float tot = 0.f;
#pragma unroll
    for (int wi = 0; wi < 8; ++wi) tot += red[wi][threadIdx.x];
    bands[(((size_t)(second ? 1 - which : which) * gridDim.y + slab) * gridDim.x + blockIdx.x) * kBandVals + threadIdx.x] = tot;
  }
}

}  // namespace

int haar_band_blocks(const Plan& p, int d) { return col_blocks<32>(p.htiles, d); }

// Runs the statements with kFull = (d == 64) as a constant.
#define WERSA_FULL(...)                                    \
  if (d == kD) { constexpr bool kFull = true; __VA_ARGS__ } \
  else { constexpr bool kFull = false; __VA_ARGS__ }

// The FFMA key side behind a filter: not placed early where several of its small tiles' CTAs come to share an SM and the
// filter's grid covers more than a third of the SMs: they gather on the others.  Forwards, placed early and not: 80 x 130, d = 32, m = 64
// 38.3 and 31.0 us; 40 x 200 30.0 and 27.2; 4 x 1024, d = 64 28.9 and 25.2; 10 x 1344 49.6 and 41.9; 16 x 500, m = 128 47.7 and
// 42.7; 30 x 130, d = 16 24.6 and 22.0.  One CTA an SM, full tiles or a small grid of the filter: 1 x 1024, m = 64 21.1 and
// 22.5; 64 x 1024 87.8 and 89.7; 4 x 700, m = 256 38.4 and 39.6; 12 x 256, d = 32, m = 128 (24 CTAs here) 23.5 and 24.6; 20 x
// 200, m = 64 (40) 21.6 and 21.7.
bool place_key_side_early(const Plan& p, unsigned ctas) {
  return !(p.simt_small && p.cfg.features < 256 && (long long)p.schunks * p.slabs > p.sms && 3 * ctas > (unsigned)p.sms);
}

// X2 / XF2: a second tensor of the same shape in the same launch (or null).
cudaError_t launch_haar_filter(const Plan& p, const void* X, int in_kind, const float* f, void* XF, const void* X2,
                               void* XF2, int out_kind, int d, bool inputs_ready, cudaStream_t st, int* launches) {
  const unsigned z = X2 != nullptr ? 2 : 1;
  const dim3 grid(col_blocks<32>(p.htiles, d), p.slabs, z), grid_bf(col_blocks<64>(p.htiles, d), p.slabs, z);
  const int n = p.cfg.seq_len, L = p.cfg.levels;
  using bf = __nv_bfloat16;
  const unsigned ctas = in_kind == 1 ? grid_bf.x * grid_bf.y * z : grid.x * grid.y * z;
  // (without inputs_ready it is a pass of its own: 1 x 8 x 131072, bf16, call after call 51.1 us before it let the next one be
  // placed early, 48.2 to 48.8 since)
  const bool place_next = !inputs_ready || place_key_side_early(p, ctas);
  cudaError_t err;
  WERSA_FULL({
    if (in_kind == 1 && out_kind == 1)
      err = launch_after(k_haar_filter_bf16<kFull, bf>, grid_bf, dim3(256), 0, st, (const bf*)X, f, (bf*)XF, (const bf*)X2, (bf*)XF2, n, d, L,
                         inputs_ready, place_next);
    else if (in_kind == 1 && out_kind == 0)
      err = launch_after(k_haar_filter_bf16<kFull, float>, grid_bf, dim3(256), 0, st, (const bf*)X, f, (float*)XF, (const bf*)X2,
                         (float*)XF2, n, d, L, inputs_ready, place_next);
    else
      err = launch_after(k_haar_filter<kFull, float, float, false>, grid, dim3(256), 0, st, (const float*)X, f, (float*)XF,
                         (const float*)X2, (float*)XF2, n, d, L, nullptr, 0.f, inputs_ready, place_next);
  })
  *launches += 1;
  return err != cudaSuccess ? err : cudaGetLastError();
}

cudaError_t launch_f32_planes(const Plan& p, const Ws& w, const void* Q, const void* K, const void* V, bool keep,
                              cudaStream_t st, int* launches) {
  const int n = p.cfg.seq_len, L = p.cfg.levels, d = p.cfg.head_dim;
  const dim3 grid(col_blocks<32>(p.htiles, d), p.slabs, p.bf16 ? 2 : 3);
  const size_t plane = (size_t)p.slabs * n * d;
  cudaError_t err;
  auto go = [&](auto kernel, auto* q) {
    using P = decltype(q);
    return launch_after(kernel, grid, dim3(256), 0, st, q, (P)K, (P)V, (const float*)w.f, w.QF3, w.KF3, w.V3, w.QF, w.KF, plane, n, d, L, w.seen);
  };
  using bf = __nv_bfloat16;
  WERSA_FULL({
    if (p.bf16) err = keep ? go(k_f32_planes<kFull, true, bf>, (const bf*)Q) : go(k_f32_planes<kFull, false, bf>, (const bf*)Q);
    else err = keep ? go(k_f32_planes<kFull, true, float>, (const float*)Q) : go(k_f32_planes<kFull, false, float>, (const float*)Q);
  })
  *launches += 1;
  return err != cudaSuccess ? err : cudaGetLastError();
}

cudaError_t launch_haar_filter_addvec(const Plan& p, const float* G, const float* f, const float* vec,
                                      float vec_scale, void* dX, int out_kind, int d, cudaStream_t st, int* launches) {
  const dim3 grid(col_blocks<32>(p.htiles, d), p.slabs);
  const int n = p.cfg.seq_len, L = p.cfg.levels;
  using bf = __nv_bfloat16;
  cudaError_t err;
  WERSA_FULL({
    if (out_kind == 0)
      err = launch_after(k_haar_filter<kFull, float, float, true>, grid, dim3(256), 0, st, G, f, (float*)dX, nullptr, nullptr, n, d, L, vec, vec_scale, true, false);
    else
      err = launch_after(k_haar_filter<kFull, float, bf, true>, grid, dim3(256), 0, st, G, f, (bf*)dX, nullptr, nullptr, n, d, L, vec, vec_scale, true, false);
  })
  *launches += 1;
  return err != cudaSuccess ? err : cudaGetLastError();
}

// The gate's CTAs here have 256 threads: one round of 28 batch elements, and sixteen slabs a thread of d omega.  Beyond that
// k_gate_backward with its 1024 threads is the faster one (88 x 372, m = 256 a training step 103.6 us, 107.4 with four rounds
// here; 85 x 12 x 202, the gate of a batch element 432 and 458).  df is summed in place while a CTA reads at most some 40 partials a
// slot for its own slab (or batch element) and the one of d omega 2048 for all of them.
bool haar_dq_takes_gate(const Plan& p) { return p.cfg.batch <= 28 && p.slabs <= 256; }
bool haar_dq_sums_bands(const Plan& p) {
  const long long blocks = haar_band_blocks(p, p.cfg.head_dim);
  return blocks * (p.cfg.gate_per_head ? 1 : p.cfg.heads) <= 48 && blocks * p.slabs <= 2048;
}
cudaError_t launch_haar_dq(const Plan& p, const Ws& w, const GateBwdArgs& args, void* dQ, int out_kind, cudaStream_t st, int* launches) {
  const int n = p.cfg.seq_len, L = p.cfg.levels, d = p.cfg.head_dim, blocks = col_blocks<32>(p.htiles, d);
  const dim3 grid((unsigned)(p.cfg.heads + 2 + p.slabs * blocks));
  const float* df = haar_dq_sums_bands(p) ? w.bands : w.dqbar + (size_t)p.slabs * kD;
  using bf = __nv_bfloat16;
  auto go = [&](auto kernel, auto* out) {
    return launch_after(kernel, grid, dim3(256), 0, st, (const float*)w.dQF, (const float*)w.f, out, n, d, L, p.slabs, blocks,
                        1.f / (float)n, df, args.sg, args.qbar, args.gate_w, args.omega, args.sumdD, args.n_sumdD, args.beta, args.eps,
                        args.bw_floor, args.m, args.B, args.H, args.per_head, args.dbeta, args.dgate_w, args.dgate_b, args.domega);
  };
  cudaError_t err;
  const bool sum = haar_dq_sums_bands(p);
  WERSA_FULL({
    if (out_kind == 0) err = sum ? go(k_haar_dq<kFull, float, true>, (float*)dQ) : go(k_haar_dq<kFull, float, false>, (float*)dQ);
    else err = sum ? go(k_haar_dq<kFull, bf, true>, (bf*)dQ) : go(k_haar_dq<kFull, bf, false>, (bf*)dQ);
  })
  *launches += 1;
  return err != cudaSuccess ? err : cudaGetLastError();
}

cudaError_t launch_haar_filter_split3(const Plan& p, const Ws& w, const void* X, __nv_bfloat16* XF3, const void* X2,
                                      __nv_bfloat16* XF3_2, bool split_S, cudaStream_t st, int* launches) {
  const int n = p.cfg.seq_len, L = p.cfg.levels, d = p.cfg.head_dim;
  const dim3 grid(col_blocks<64>(p.htiles, d), p.slabs, (X2 != nullptr ? 2 : 1) + (split_S ? 1 : 0));
  const size_t plane = (size_t)p.slabs * n * d;
  using bf = __nv_bfloat16;
  cudaError_t err;
  WERSA_FULL({
    err = launch_after(k_haar_filter_split3<kFull>, grid, dim3(256), 0, st, (const bf*)X, w.f, XF3, (const bf*)X2, XF3_2, plane, n, d, L,
                       split_S ? w.S : nullptr, w.Sbf, w.Slo, p.cfg.features / p.groups, p.groups);
  })
  *launches += 1;
  return err != cudaSuccess ? err : cudaGetLastError();
}

cudaError_t launch_haar_backward(const Plan& p, const Ws& w, int which, const void* X, const float* G, void* dX,
                                 const void* X2, const float* G2, void* dX2, int in_kind, int out_kind, int d,
                                 cudaStream_t st, int* launches) {
  const dim3 grid(haar_band_blocks(p, d), p.slabs, X2 != nullptr ? 2 : 1);
  const int n = p.cfg.seq_len, L = p.cfg.levels;
  using bf = __nv_bfloat16;
  cudaError_t err;
  auto go = [&](auto kernel, auto* x, auto* out) {
    return launch_after(kernel, grid, dim3(256), 0, st, x, G, out, static_cast<decltype(x)>(X2), G2,
                        static_cast<decltype(out)>(dX2), w.f, w.bands, which, n, d, L);
  };
  WERSA_FULL({
    if (dX == nullptr && dX2 == nullptr) {   // band inner products only (sequence shards, whose tensors are bf16)
      err = go(k_haar_backward<kFull, bf, float, false>, (const bf*)X, (float*)nullptr);
    } else if (in_kind == 1 && out_kind == 1) {
      err = go(k_haar_backward<kFull, bf, bf, true>, (const bf*)X, (bf*)dX);
    } else if (in_kind == 1 && out_kind == 0) {
      err = go(k_haar_backward<kFull, bf, float, true>, (const bf*)X, (float*)dX);
    } else if (in_kind == 0 && out_kind == 0) {
      err = go(k_haar_backward<kFull, float, float, true>, (const float*)X, (float*)dX);
    } else {
      err = go(k_haar_backward<kFull, float, bf, true>, (const float*)X, (bf*)dX);
    }
  })
  *launches += 1;
  return err != cudaSuccess ? err : cudaGetLastError();
}

}  // namespace wersa
