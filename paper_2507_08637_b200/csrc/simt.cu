// fp32 FFMA kernels of the WERSA attention path (Eqs. 6-7 of the paper and their backward):
// random projection + ReLU, key summary S' = ReLU(K_F W)^T V and z' = ReLU(K_F W)^T 1 over
// sequence chunks, output O = ReLU(Q_F W) S' / (ReLU(Q_F W) z' + eps'), and the gradient kernels.
//
// The feature-map factor c = 1/(bw sqrt(m)) is folded away: ReLU is positively homogeneous, so
// phi = c ReLU(X_F W) and O = N'/(D' + eps/c^2) with the unscaled N', D'; eps' = eps m bw^2.
//
// These kernels serve the fp32 configuration (a 1e-4 tolerance rules out 10-bit-mantissa tensor
// core inputs) and give every other path a second opinion.  They are bound by the FFMA pipes, so
// everything is arranged for operand reuse in registers: a group of 64 threads (8 x 8) owns 8 TI
// tokens x 64 features, a thread TI tokens (ty + 8 i) x 8 features (tx + 8 j), and every small GEMM
// is a loop that loads TI + 8 float4 from shared memory for 32 TI FFMAs (TI = 8: 16 loads for 256).
// A CTA is M / 64 feature groups times TG token groups; M / 64 * TG = 4 groups (256 threads, about 200
// registers each, one CTA per SM) fill the four FFMA pipes of an SM.  With one token per lane
// and four features per step (one load for four FFMAs) the same passes were bound by shared-memory
// loads.  B=2 H=8 n=4096 d=64 m=256: key + query side 449 -> 231 us (19 -> 37 TFLOP/s of the 74 the pipes
// have at 1.965 GHz; the FFMA pipe is then busy half of the time: a chunk's set-up and last, partly filled
// tile, and dispatch stalls between FFMAs are the rest); training step at B=2 H=4 n=4096 d=32 m=128
// 462 -> 156 us.  The products with S' (or W^T) rows and the token sums then went to packed fma, two columns per
// instruction against a doubled scalar: half the issue slots for the same pipe time, 231 -> 222 us and 152 -> 146 us.
// The projection stays scalar: its packed form pairs even and odd k, takes twice the sums, hence two passes over the
// tokens, and cost the query side 10 us of 115.
//
// Tiles in shared memory hold rows of DP floats (the head dimension rounded up to 16, 32 or 64,
// columns past it are zero) without padding; a row's 16-byte chunks are permuted (swz) so that eight
// consecutive rows can be read at one chunk index without bank conflicts.
#include <type_traits>

#include "common.cuh"

namespace wersa {
namespace {

template <int M, int DP, int TI, int TG_, bool kB, bool kG> struct Cfg {
  static constexpr int TG = TG_;                    // token groups
  static constexpr int FG = M / 64;                 // feature groups
  static constexpr int kThreads = 64 * FG * TG;
  static constexpr int TT = 8 * TI, CT = TT * TG;   // tokens per group / per CTA
  // shared memory, in floats
  static constexpr int wt = 0;                          // W^T [M][DP]
  static constexpr int b = wt + M * DP;                 // S' or dS' [M][DP]
  static constexpr int x = b + (kB ? M * DP : 0);       // filtered tile [CT][DP]
  static constexpr int g = x + CT * DP;                 // V or dO tile [CT][DP]
  static constexpr int r = g + (kG ? CT * DP : 0);      // per group: features or gradients [TT][64], partial results
  static constexpr int zs = r + FG * TG * TT * 64;      // z' or dz' [M]
  static constexpr int st = zs + M;                     // row sums per feature group [FG][CT][2]
  static constexpr int total = st + FG * CT * 2;
};

template <int DP> __device__ __forceinline__ int swz(int row, int chunk) {
  return DP >= 32 ? (chunk ^ (row & 7)) : (chunk ^ ((row >> 1) & 3));
}

__device__ __forceinline__ void cp_async16(float* dst, const float* src, bool valid) {
  const uint32_t d = static_cast<uint32_t>(__cvta_generic_to_shared(dst));
  const int bytes = valid ? 16 : 0;   // 0: zero fill, the source is not read
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(d), "l"(src), "r"(bytes) : "memory");
}
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_all;" ::: "memory"); }
__device__ __forceinline__ void group_sync(int gid) { asm volatile("bar.sync %0, 64;" ::"r"(gid + 1) : "memory"); }

// Rows [row0, row0 + ROWS) of an (n x d) slab -> dst[ROWS][DP], rows past n and columns past d as zeros.
// fp32 goes through cp.async (the caller waits), bf16 (kind 1) is converted on the way.
template <int DP, int ROWS, int THREADS>
__device__ __forceinline__ void load_rows(const void* __restrict__ src, int kind, int d, int n, int row0, float* dst) {
  constexpr int NC = DP / 4;
  for (int i = threadIdx.x; i < ROWS * NC; i += THREADS) {
    const int r = i / NC, c = i - r * NC;
    const bool valid = row0 + r < n && c * 4 < d;
    float* p = dst + r * DP + 4 * swz<DP>(r, c);
    const size_t off = valid ? (size_t)(row0 + r) * d + c * 4 : 0;
    if (kind == 0) {
      cp_async16(p, static_cast<const float*>(src) + off, valid);
    } else {
      uint2 raw = make_uint2(0u, 0u);
      if (valid) raw = *reinterpret_cast<const uint2*>(static_cast<const __nv_bfloat16*>(src) + off);
      *reinterpret_cast<float4*>(p) =
          make_float4(__uint_as_float(raw.x << 16), __uint_as_float(raw.x & 0xFFFF0000u), __uint_as_float(raw.y << 16),
                      __uint_as_float(raw.y & 0xFFFF0000u));
    }
  }
}
// W (d x M, row-major) -> WT[M][DP].
template <int M, int DP, int THREADS>
__device__ __forceinline__ void load_wt(const void* __restrict__ W, int kind, int d, float* WT) {
  constexpr int kBatch = 16;   // loads in flight
#pragma unroll 1
  for (int i0 = threadIdx.x; i0 < M * DP; i0 += kBatch * THREADS) {
    float v[kBatch];
#pragma unroll
    for (int q = 0; q < kBatch; ++q) {
      const int i = i0 + q * THREADS, c = i / M, f = i - c * M;   // consecutive threads: consecutive features
      v[q] = 0.f;
      if (i < M * DP && c < d)
        v[q] = kind == 0 ? static_cast<const float*>(W)[(size_t)c * M + f]
                         : __bfloat162float(static_cast<const __nv_bfloat16*>(W)[(size_t)c * M + f]);
    }
#pragma unroll
    for (int q = 0; q < kBatch; ++q) {
      const int i = i0 + q * THREADS, c = i / M, f = i - c * M;
      if (i < M * DP) WT[f * DP + 4 * swz<DP>(f, c >> 2) + (c & 3)] = v[q];
    }
  }
}
// S' or dS' of a slab ([M][64] in the workspace) -> B[M][DP].
template <int M, int DP, int THREADS>
__device__ __forceinline__ void load_b(const float* __restrict__ S, float* B) {
  constexpr int NC = DP / 4;
  for (int i = threadIdx.x; i < M * NC; i += THREADS) {
    const int f = i / NC, c = i - f * NC;
    cp_async16(B + f * DP + 4 * swz<DP>(f, c), S + (size_t)f * kD + c * 4, true);
  }
}

// acc[i][j] = sum_k X[ty + 8 i][k] B[tx + 8 j][k], X and B the first rows of this group's tokens / features.
template <int DP, int TI>
__device__ __forceinline__ void gemm_nt(const float* __restrict__ X, const float* __restrict__ B, int tx, int ty,
                                        float (&acc)[TI][8]) {
#pragma unroll
  for (int i = 0; i < TI; ++i)
#pragma unroll
    for (int j = 0; j < 8; ++j) acc[i][j] = 0.f;
#pragma unroll 2
  for (int k = 0; k < DP / 4; ++k) {
    const float* xp = X + ty * DP + 4 * swz<DP>(ty, k);   // rows 8 apart share the permutation
    const float* bp = B + tx * DP + 4 * swz<DP>(tx, k);
    float4 x[TI];
#pragma unroll
    for (int i = 0; i < TI; ++i) x[i] = *reinterpret_cast<const float4*>(xp + i * 8 * DP);
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      const float4 w = *reinterpret_cast<const float4*>(bp + j * 8 * DP);
#pragma unroll
      for (int i = 0; i < TI; ++i) {
        acc[i][j] = fmaf(x[i].x, w.x, acc[i][j]);
        acc[i][j] = fmaf(x[i].y, w.y, acc[i][j]);
        acc[i][j] = fmaf(x[i].z, w.z, acc[i][j]);
        acc[i][j] = fmaf(x[i].w, w.w, acc[i][j]);
      }
    }
  }
}

// Element (token ty + 8 i, feature tx + 8 j) of a group's [TT][64] tile R: chunk c of row t sits at c ^ 2 (t & 3),
// so that the four rows a warp writes at once fall into different banks.
__device__ __forceinline__ int r_index(int tx, int ty, int i, int j) {
  return (ty + 8 * i) * 64 + ((8 * j) ^ ((ty & 3) << 3)) + tx;
}

// CW consecutive-in-pairs columns of a DP-wide row: DP = 64: 4 tx .. + 3 and 32 + 4 tx .. + 3; DP = 32: 4 tx .. + 3;
// DP = 16: 2 tx, 2 tx + 1.
template <int DP> __device__ __forceinline__ void load_cols(const float* __restrict__ row, int r, int tx, f32x2 (&v)[DP / 16]) {
  if constexpr (DP == 16) {
    v[0] = *reinterpret_cast<const f32x2*>(row + 4 * swz<DP>(r, tx >> 1) + 2 * (tx & 1));
  } else {
    const float* p = row + 4 * swz<DP>(r, tx);
    const ulonglong2 a = *reinterpret_cast<const ulonglong2*>(p);
    v[0] = a.x; v[1] = a.y;
    if constexpr (DP == 64) {
      const ulonglong2 b = *reinterpret_cast<const ulonglong2*>(p + 32);
      v[2] = b.x; v[3] = b.y;
    }
  }
}

// acc[i][c] = sum over the group's 64 features f of R[ty + 8 i][f] B[f][column c of tx].
template <int DP, int TI>
__device__ __forceinline__ void gemm_contract(const float* __restrict__ R, const float* __restrict__ B, int tx, int ty,
                                              f32x2 (&acc)[TI][DP / 16]) {
#pragma unroll
  for (int i = 0; i < TI; ++i)
#pragma unroll
    for (int c = 0; c < DP / 16; ++c) acc[i][c] = 0ull;
#pragma unroll 2
  for (int f4 = 0; f4 < 16; ++f4) {
    float4 r[TI];
    const float* rp = R + ty * 64 + 4 * (f4 ^ ((ty & 3) << 1));
#pragma unroll
    for (int i = 0; i < TI; ++i) r[i] = *reinterpret_cast<const float4*>(rp + i * 512);
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int f = 4 * f4 + q;
      f32x2 b[DP / 16];
      load_cols<DP>(B + f * DP, f, tx, b);
#pragma unroll
      for (int i = 0; i < TI; ++i) {
        const float rv = q == 0 ? r[i].x : q == 1 ? r[i].y : q == 2 ? r[i].z : r[i].w;
        const f32x2 r2 = pk2(rv, rv);
#pragma unroll
        for (int c = 0; c < DP / 16; ++c) acc[i][c] = fma2(r2, b[c], acc[i][c]);
      }
    }
  }
}

// acc[v][c] += sum over the group's TT tokens t of R[t][feature v of tx] G[t][column c of ty], features 4 tx .. + 3
// and 32 + 4 tx .. + 3 of the group.
template <int DP, int TI>
__device__ __forceinline__ void gemm_tokens(const float* __restrict__ R, const float* __restrict__ G, int tx, int ty,
                                            f32x2 (&acc)[8][DP / 16]) {
#pragma unroll 4
  for (int t = 0; t < 8 * TI; ++t) {
    const float* rp = R + t * 64 + 4 * (tx ^ ((t & 3) << 1));
    const float4 a = *reinterpret_cast<const float4*>(rp), b = *reinterpret_cast<const float4*>(rp + 32);
    const float rv[8] = {a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w};
    f32x2 g[DP / 16];
    load_cols<DP>(G + t * DP, t, ty, g);
#pragma unroll
    for (int v = 0; v < 8; ++v) {
      const f32x2 r2 = pk2(rv[v], rv[v]);
#pragma unroll
      for (int c = 0; c < DP / 16; ++c) acc[v][c] = fma2(r2, g[c], acc[v][c]);
    }
  }
}

// A group's (TT x DP) partial product -> its own R region, rows of DP floats.
template <int DP, int TI>
__device__ __forceinline__ void put_partial(float* R, int tx, int ty, const f32x2 (&acc)[TI][DP / 16]) {
#pragma unroll
  for (int i = 0; i < TI; ++i) {
    float* p = R + (ty + 8 * i) * DP;
    if constexpr (DP == 16) {
      *reinterpret_cast<f32x2*>(p + 2 * tx) = acc[i][0];
    } else {
      *reinterpret_cast<ulonglong2*>(p + 4 * tx) = make_ulonglong2(acc[i][0], acc[i][1]);
      if constexpr (DP == 64) *reinterpret_cast<ulonglong2*>(p + 32 + 4 * tx) = make_ulonglong2(acc[i][2], acc[i][3]);
    }
  }
}

__device__ __forceinline__ void store_chunk(void* base, int kind, size_t off, float4 v) {
  if (kind == 0) {
    *reinterpret_cast<float4*>(static_cast<float*>(base) + off) = v;
  } else {
    const __nv_bfloat162 a = __floats2bfloat162_rn(v.x, v.y), b = __floats2bfloat162_rn(v.z, v.w);
    uint2 raw;
    raw.x = *reinterpret_cast<const uint32_t*>(&a);
    raw.y = *reinterpret_cast<const uint32_t*>(&b);
    *reinterpret_cast<uint2*>(static_cast<__nv_bfloat16*>(base) + off) = raw;
  }
}

// Sum of the feature groups' partials (in group order), times 1 / (den + epsp) with kScale, -> the tile's rows
// [row0, min(row0 + TG TT, n)) of a slab of d columns (TT = 8 TI: see for_tiles; the groups' regions stay C::TT apart).
template <typename C, int DP, int TT, bool kScale>
__device__ __forceinline__ void combine_rows(const float* __restrict__ R, const float* __restrict__ st, float epsp,
                                             void* __restrict__ out, int kind, int d, int n, int row0) {
  constexpr int NC = DP / 4;
  for (int i = threadIdx.x; i < C::TG * TT * NC; i += C::kThreads) {
    const int t = i / NC, c = i - t * NC;
    if (row0 + t >= n || c * 4 >= d) continue;
    const float* p = R + (t / TT) * C::FG * C::TT * 64 + (t % TT) * DP + c * 4;
    float4 v = *reinterpret_cast<const float4*>(p);
#pragma unroll
    for (int fg = 1; fg < C::FG; ++fg) {
      const float4 u = *reinterpret_cast<const float4*>(p + fg * C::TT * 64);
      v.x += u.x; v.y += u.y; v.z += u.z; v.w += u.w;
    }
    if constexpr (kScale) {
      float den = st[2 * t];
#pragma unroll
      for (int fg = 1; fg < C::FG; ++fg) den += st[2 * (fg * C::CT + t)];
      const float inv = 1.f / (den + epsp);
      v.x *= inv; v.y *= inv; v.z *= inv; v.w *= inv;
    }
    store_chunk(out, kind, (size_t)(row0 + t) * d + c * 4, v);
  }
}

// The CTA's sums over its chunk -> one partial of S' (or dS') and z' (or dz'), [M][64] and [M]: the token groups'
// shares are added through their R regions in group order, columns past DP are zero.
template <typename C, int M, int DP>
__device__ __forceinline__ void store_partials(float* R, const f32x2 (&acc2)[8][DP / 16], const float (&zacc)[8], int fg,
                                               int tg, int tx, int ty, float* __restrict__ sp, float* __restrict__ zp) {
  float acc[8][DP / 8];
#pragma unroll
  for (int v = 0; v < 8; ++v)
#pragma unroll
    for (int c = 0; c < DP / 16; ++c) upk2(acc2[v][c], acc[v][2 * c], acc[v][2 * c + 1]);
  constexpr int TG = C::CT / C::TT;
  __syncthreads();   // R is free
  if constexpr (TG > 1) {
    static_assert(C::TT == 64, "a region holds 64 x 64 sums");
    float* reg = R + (tg * C::FG + fg) * C::TT * 64;
#pragma unroll
    for (int v = 0; v < 8; ++v)
#pragma unroll
      for (int c = 0; c < DP / 8; ++c) reg[(v * (DP / 8) + c) * 64 + ty * 8 + tx] = acc[v][c];
    __syncthreads();
  }
  if (tg == 0) {
#pragma unroll
    for (int v = 0; v < 8; ++v) {
      const int f = fg * 64 + (v < 4 ? 4 * tx + v : 32 + 4 * tx + v - 4);
      float s[DP / 8];
#pragma unroll
      for (int c = 0; c < DP / 8; ++c) {
        s[c] = acc[v][c];
        if constexpr (TG > 1) {
#pragma unroll
          for (int q = 1; q < TG; ++q) s[c] += R[(q * C::FG + fg) * C::TT * 64 + (v * (DP / 8) + c) * 64 + ty * 8 + tx];
        }
      }
      float* dst = sp + (size_t)f * kD;
      if constexpr (DP == 16) {
        *reinterpret_cast<float2*>(dst + 2 * ty) = make_float2(s[0], s[1]);
        *reinterpret_cast<float2*>(dst + 16 + 2 * ty) = make_float2(0.f, 0.f);
        *reinterpret_cast<float4*>(dst + 32 + 4 * ty) = make_float4(0.f, 0.f, 0.f, 0.f);
      } else {
        *reinterpret_cast<float4*>(dst + 4 * ty) = make_float4(s[0], s[1], s[2], s[3]);
        if constexpr (DP == 64)
          *reinterpret_cast<float4*>(dst + 32 + 4 * ty) = make_float4(s[4], s[5], s[6], s[7]);
        else
          *reinterpret_cast<float4*>(dst + 32 + 4 * ty) = make_float4(0.f, 0.f, 0.f, 0.f);
      }
    }
  }
  // z: thread (tx, ty) of a group holds the sums of features tx + 8 j over its own tokens
  __syncthreads();
#pragma unroll
  for (int j = 0; j < 8; ++j) R[(tg * C::FG + fg) * 512 + ty * 64 + tx + 8 * j] = zacc[j];
  __syncthreads();
  for (int f = threadIdx.x; f < M; f += C::kThreads) {
    float s = 0.f;
#pragma unroll
    for (int q = 0; q < TG; ++q)
#pragma unroll
      for (int y = 0; y < 8; ++y) s += R[(q * C::FG + (f >> 6)) * 512 + y * 64 + (f & 63)];
    zp[f] = s;
  }
}

// Runs body(integral constant TI, row0) over the tiles of rows [first, last): full tiles of C::CT rows, and what is
// left as one tile of TI = 2 (16 rows per token group) where that is enough, so that a chunk need not be a
// multiple of the full tile.
template <int V> struct Int { static constexpr int value = V; };
template <typename C, typename F> __device__ __forceinline__ void for_tiles(int first, int last, F&& body) {
  for (int row0 = first; row0 < last; row0 += C::CT) {
    if (C::TT > 16 && last - row0 <= 16 * C::TG) body(Int<2>(), row0);
    else body(Int<C::TT / 8>(), row0);
  }
}

// Thread coordinates.
template <typename C> struct Who {
  int gid, fg, tg, tx, ty;
  __device__ __forceinline__ Who() {
    gid = threadIdx.x >> 6;
    fg = gid % C::FG;
    tg = gid / C::FG;
    tx = threadIdx.x & 7;
    ty = (threadIdx.x >> 3) & 7;
  }
};

// ---- forward, key side: partial S', z' of one sequence chunk.  grid (chunks, slabs) ------------------------
// Per tile: features from K_F (its buffer is refilled for the next tile while the token sum runs), then
// S'[64 features x DP] += R^T V per group, held in registers for the whole chunk.
template <int M, int DP, int TI, int TG>
__global__ void __launch_bounds__(M * TG, 1)
k_simt_kside(const float* __restrict__ KF, const void* __restrict__ V, const void* __restrict__ W, int kind,
             float* __restrict__ spart, float* __restrict__ zpart, int n, int d, int chunk_rows) {
  using C = Cfg<M, DP, TI, TG, false, true>;
  extern __shared__ __align__(16) float sm[];
  const Who<C> me;
  const int chunk = blockIdx.x, slab = blockIdx.y;
  const float* kf = KF + (size_t)slab * n * d;
  const void* v = kind == 0 ? (const void*)(static_cast<const float*>(V) + (size_t)slab * n * d)
                            : (const void*)(static_cast<const __nv_bfloat16*>(V) + (size_t)slab * n * d);
  const int first = chunk * chunk_rows, last = min(n, first + chunk_rows);
  // (launched as a programmatic dependent, see launch_after: V and W are arguments, K_F comes from the kernel before)
  load_rows<DP, C::CT, C::kThreads>(v, kind, d, last, first, sm + C::g);
  load_wt<M, DP, C::kThreads>(W, kind, d, sm + C::wt);
  wait_for_stream_predecessor();
  if constexpr (TI == 2) let_stream_successor_start();   // (with full tiles: 2 x 4 x 4096, d = 32, m = 128 146 instead of 141 us)
  load_rows<DP, C::CT, C::kThreads>(kf, 0, d, last, first, sm + C::x);
  f32x2 acc[8][DP / 16];
  float zacc[8];
#pragma unroll
  for (int q = 0; q < 8; ++q) {
    zacc[q] = 0.f;
#pragma unroll
    for (int c = 0; c < DP / 16; ++c) acc[q][c] = 0ull;
  }
  float* R = sm + C::r + me.gid * C::TT * 64;
  cp_async_wait_all();
  __syncthreads();
  for_tiles<C>(first, last, [&](auto ti, int row0) {
    constexpr int T = decltype(ti)::value, TT = 8 * T;   // tokens per thread / per group of this tile
    {
      float a[T][8];
      gemm_nt<DP, T>(sm + C::x + me.tg * TT * DP, sm + C::wt + me.fg * 64 * DP, me.tx, me.ty, a);
#pragma unroll
      for (int i = 0; i < T; ++i)
#pragma unroll
        for (int j = 0; j < 8; ++j) {
          const float p = fmaxf(a[i][j], 0.f);
          zacc[j] += p;
          R[r_index(me.tx, me.ty, i, j)] = p;
        }
    }
    cp_async_wait_all();   // V of this tile
    __syncthreads();
    if (row0 + C::CT < last) load_rows<DP, C::CT, C::kThreads>(kf, 0, d, last, row0 + C::CT, sm + C::x);
    gemm_tokens<DP, T>(R, sm + C::g + me.tg * TT * DP, me.tx, me.ty, acc);
    cp_async_wait_all();   // K_F of the next tile
    __syncthreads();
    if (row0 + C::CT < last) load_rows<DP, C::CT, C::kThreads>(v, kind, d, last, row0 + C::CT, sm + C::g);
  });
  const size_t pidx = (size_t)slab * gridDim.x + chunk;
  store_partials<C, M, DP>(sm + C::r, acc, zacc, me.fg, me.tg, me.tx, me.ty, spart + pidx * M * kD, zpart + pidx * M);
}

// ---- forward, query side.  grid (chunks, slabs) -------------------------------------------------------------
template <int M, int DP, int TI, int TG>
__global__ void __launch_bounds__(M * TG, 1)
k_simt_qside(const float* __restrict__ QF, const void* __restrict__ W, int kind, const float* __restrict__ Sg,
             const float* __restrict__ zg, const float* __restrict__ beta, float eps, float bw_floor,
             void* __restrict__ O, int n, int d, int chunk_rows) {
  using C = Cfg<M, DP, TI, TG, true, false>;
  extern __shared__ __align__(16) float sm[];
  const Who<C> me;
  const int chunk = blockIdx.x, slab = blockIdx.y;
  const float* qf = QF + (size_t)slab * n * d;
  void* o = kind == 0 ? (void*)(static_cast<float*>(O) + (size_t)slab * n * d)
                      : (void*)(static_cast<__nv_bfloat16*>(O) + (size_t)slab * n * d);
  const int first = chunk * chunk_rows, last = min(n, first + chunk_rows);
  // (launched as a programmatic dependent, see launch_after: Q_F is older than the reduction, which leaves S' and z')
  load_rows<DP, C::CT, C::kThreads>(qf, 0, d, last, first, sm + C::x);
  load_wt<M, DP, C::kThreads>(W, kind, d, sm + C::wt);
  wait_for_stream_predecessor();
  load_b<M, DP, C::kThreads>(Sg + (size_t)slab * M * kD, sm + C::b);
  for (int i = threadIdx.x; i < M; i += C::kThreads) sm[C::zs + i] = __ldcg(zg + (size_t)slab * M + i);
  const float bw = fmaxf(beta[0], bw_floor);
  const float epsp = eps * (float)M * bw * bw;
  float* R = sm + C::r + me.gid * C::TT * 64;
  const float* zs = sm + C::zs + me.fg * 64 + me.tx;
  cp_async_wait_all();
  __syncthreads();
  for_tiles<C>(first, last, [&](auto ti, int row0) {
    constexpr int T = decltype(ti)::value, TT = 8 * T;   // tokens per thread / per group of this tile
    {
      float a[T][8];
      gemm_nt<DP, T>(sm + C::x + me.tg * TT * DP, sm + C::wt + me.fg * 64 * DP, me.tx, me.ty, a);
      __syncthreads();   // everybody has read the previous tile's partials; this tile's X is free
      if (row0 + C::CT < last) load_rows<DP, C::CT, C::kThreads>(qf, 0, d, last, row0 + C::CT, sm + C::x);
#pragma unroll
      for (int i = 0; i < T; ++i) {
        float den = 0.f;
#pragma unroll
        for (int j = 0; j < 8; ++j) {
          const float p = fmaxf(a[i][j], 0.f);
          den = fmaf(p, zs[8 * j], den);
          R[r_index(me.tx, me.ty, i, j)] = p;
        }
#pragma unroll
        for (int s = 1; s < 8; s <<= 1) den += __shfl_xor_sync(0xffffffffu, den, s);
        if (me.tx == 0) sm[C::st + 2 * (me.fg * C::CT + me.tg * TT + me.ty + 8 * i)] = den;
      }
    }
    group_sync(me.gid);
    {
      f32x2 num[T][DP / 16];
      gemm_contract<DP, T>(R, sm + C::b + me.fg * 64 * DP, me.tx, me.ty, num);
      group_sync(me.gid);
      put_partial<DP, T>(R, me.tx, me.ty, num);
    }
    cp_async_wait_all();
    __syncthreads();
    combine_rows<C, DP, TT, true>(sm + C::r, sm + C::st, epsp, o, kind, d, last, row0);
  });
}

// ---- backward, query side.  grid (chunks, slabs) ------------------------------------------------------------
// Per tile, with R = ReLU(Q_F W), G = dO S'^T (both tokens x features) and D = R z' + eps':
//   dO . O = sum_f R G / D, so N' is never formed;  dD = -(dO . O) / D =: c / D;
//   dS' += (R / D)^T dO;  dz' += (R / D)^T c;  dA = (G + c z') / D where R > 0;  dQ_F = dA W^T.
template <int M, int DP, int TI, int TG>
__global__ void __launch_bounds__(M * TG, 1)
k_simt_bwd_qside(const float* __restrict__ QF, const void* __restrict__ W, int kind, const float* __restrict__ Sg,
                 const float* __restrict__ zg, const float* __restrict__ beta, float eps, float bw_floor,
                 const void* __restrict__ dO, float* __restrict__ dQF, float* __restrict__ dspart,
                 float* __restrict__ dzpart, float* __restrict__ sumdD, int n, int d, int chunk_rows) {
  wait_for_stream_predecessor();   // (launched as a programmatic dependent: see launch_after)
  if constexpr (TI == 2) let_stream_successor_start();   // (with full tiles: 2 x 4 x 4096, d = 32, m = 128 146 instead of 141 us)
  using C = Cfg<M, DP, TI, TG, true, true>;
  extern __shared__ __align__(16) float sm[];
  const Who<C> me;
  const int chunk = blockIdx.x, slab = blockIdx.y;
  const float* qf = QF + (size_t)slab * n * d;
  const void* go = kind == 0 ? (const void*)(static_cast<const float*>(dO) + (size_t)slab * n * d)
                             : (const void*)(static_cast<const __nv_bfloat16*>(dO) + (size_t)slab * n * d);
  float* dqf = dQF + (size_t)slab * n * d;
  const int first = chunk * chunk_rows, last = min(n, first + chunk_rows);
  load_rows<DP, C::CT, C::kThreads>(qf, 0, d, last, first, sm + C::x);
  load_rows<DP, C::CT, C::kThreads>(go, kind, d, last, first, sm + C::g);
  load_b<M, DP, C::kThreads>(Sg + (size_t)slab * M * kD, sm + C::b);
  load_wt<M, DP, C::kThreads>(W, kind, d, sm + C::wt);
  for (int i = threadIdx.x; i < M; i += C::kThreads) sm[C::zs + i] = __ldcg(zg + (size_t)slab * M + i);
  const float bw = fmaxf(beta[0], bw_floor);
  const float epsp = eps * (float)M * bw * bw;
  f32x2 acc[8][DP / 16];
  float zacc[8];
#pragma unroll
  for (int q = 0; q < 8; ++q) {
    zacc[q] = 0.f;
#pragma unroll
    for (int c = 0; c < DP / 16; ++c) acc[q][c] = 0ull;
  }
  float sum_dd = 0.f;   // first feature group, tx = 0: sum of dD over this thread's tokens
  float* R = sm + C::r + me.gid * C::TT * 64;
  float* st = sm + C::st;
  const float* zs = sm + C::zs + me.fg * 64 + me.tx;
  cp_async_wait_all();
  __syncthreads();
  for_tiles<C>(first, last, [&](auto ti, int row0) {
    constexpr int T = decltype(ti)::value, TT = 8 * T;   // tokens per thread / per group of this tile
    const int tok0 = me.tg * TT + me.ty;   // first token of this thread inside the CTA tile
    float a[T][8];
    gemm_nt<DP, T>(sm + C::x + me.tg * TT * DP, sm + C::wt + me.fg * 64 * DP, me.tx, me.ty, a);
    __syncthreads();   // everybody has read the previous tile's partials; this tile's X is free
    if (row0 + C::CT < last) load_rows<DP, C::CT, C::kThreads>(qf, 0, d, last, row0 + C::CT, sm + C::x);
#pragma unroll
    for (int i = 0; i < T; ++i) {
      float den = 0.f;
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        const float p = fmaxf(a[i][j], 0.f);
        den = fmaf(p, zs[8 * j], den);
        R[r_index(me.tx, me.ty, i, j)] = p;
      }
#pragma unroll
      for (int s = 1; s < 8; s <<= 1) den += __shfl_xor_sync(0xffffffffu, den, s);
      if (me.tx == 0) st[2 * (me.fg * C::CT + tok0 + 8 * i)] = den;
    }
    gemm_nt<DP, T>(sm + C::g + me.tg * TT * DP, sm + C::b + me.fg * 64 * DP, me.tx, me.ty, a);   // G
#pragma unroll
    for (int i = 0; i < T; ++i) {
      float num = 0.f;
#pragma unroll
      for (int j = 0; j < 8; ++j) num = fmaf(R[r_index(me.tx, me.ty, i, j)], a[i][j], num);   // (own elements)
#pragma unroll
      for (int s = 1; s < 8; s <<= 1) num += __shfl_xor_sync(0xffffffffu, num, s);
      if (me.tx == 0) st[2 * (me.fg * C::CT + tok0 + 8 * i) + 1] = num;
    }
    __syncthreads();
#pragma unroll
    for (int i = 0; i < T; ++i) {
      float den = epsp, num = 0.f;
#pragma unroll
      for (int fg = 0; fg < C::FG; ++fg) {
        const float2 s = *reinterpret_cast<const float2*>(st + 2 * (fg * C::CT + tok0 + 8 * i));
        den += s.x;
        num += s.y;
      }
      const bool live = row0 + tok0 + 8 * i < last;   // rows past the end contribute nothing
      const float inv = live ? 1.f / den : 0.f;
      const float c = -num * inv;
      if (me.fg == 0 && me.tx == 0) sum_dd += c * inv;
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        float* rp = R + r_index(me.tx, me.ty, i, j);
        const float p = *rp;
        a[i][j] = p > 0.f ? fmaf(c, zs[8 * j], a[i][j]) * inv : 0.f;   // dA
        const float ps = p * inv;
        zacc[j] = fmaf(ps, c, zacc[j]);
        *rp = ps;
      }
    }
    group_sync(me.gid);
    gemm_tokens<DP, T>(R, sm + C::g + me.tg * TT * DP, me.tx, me.ty, acc);
    __syncthreads();   // this tile's dO is free, every group has read its R
    if (row0 + C::CT < last) load_rows<DP, C::CT, C::kThreads>(go, kind, d, last, row0 + C::CT, sm + C::g);
#pragma unroll
    for (int i = 0; i < T; ++i)
#pragma unroll
      for (int j = 0; j < 8; ++j) R[r_index(me.tx, me.ty, i, j)] = a[i][j];
    group_sync(me.gid);
    {
      f32x2 gx[T][DP / 16];
      gemm_contract<DP, T>(R, sm + C::wt + me.fg * 64 * DP, me.tx, me.ty, gx);
      group_sync(me.gid);
      put_partial<DP, T>(R, me.tx, me.ty, gx);
    }
    cp_async_wait_all();
    __syncthreads();
    combine_rows<C, DP, TT, false>(sm + C::r, nullptr, 0.f, dqf, 0, d, last, row0);
  });
  const size_t pidx = (size_t)slab * gridDim.x + chunk;
  store_partials<C, M, DP>(sm + C::r, acc, zacc, me.fg, me.tg, me.tx, me.ty, dspart + pidx * M * kD, dzpart + pidx * M);
  __syncthreads();
  if (me.fg == 0 && me.tx == 0) sm[C::st + me.tg * 8 + me.ty] = sum_dd;
  __syncthreads();
  if (threadIdx.x == 0) {
    float s = 0.f;
    for (int i = 0; i < 8 * TG; ++i) s += sm[C::st + i];
    sumdD[pidx] = s;
  }
}

// ---- backward, key side.  grid (chunks, slabs) --------------------------------------------------------------
// Per tile: R = ReLU(K_F W); dV = R dS'; dB = (V dS'^T + 1 dz'^T) (.) 1[R > 0]; dK_F = dB W^T.
template <int M, int DP, int TI, int TG>
__global__ void __launch_bounds__(M * TG, 1)
k_simt_bwd_kside(const float* __restrict__ KF, const void* __restrict__ V, const void* __restrict__ W, int kind,
                 const float* __restrict__ dSg, const float* __restrict__ dzg, void* __restrict__ dV, int gkind,
                 float* __restrict__ dKF, int n, int d, int chunk_rows) {
  using C = Cfg<M, DP, TI, TG, true, true>;
  extern __shared__ __align__(16) float sm[];
  const Who<C> me;
  const int chunk = blockIdx.x, slab = blockIdx.y;
  const float* kf = KF + (size_t)slab * n * d;
  const void* v = kind == 0 ? (const void*)(static_cast<const float*>(V) + (size_t)slab * n * d)
                            : (const void*)(static_cast<const __nv_bfloat16*>(V) + (size_t)slab * n * d);
  void* dv = gkind == 0 ? (void*)(static_cast<float*>(dV) + (size_t)slab * n * d)
                        : (void*)(static_cast<__nv_bfloat16*>(dV) + (size_t)slab * n * d);
  float* dkf = dKF + (size_t)slab * n * d;
  const int first = chunk * chunk_rows, last = min(n, first + chunk_rows);
  // (launched as a programmatic dependent, see launch_after: K_F is the forward's, the reduction leaves dS' and dz')
  load_rows<DP, C::CT, C::kThreads>(kf, 0, d, last, first, sm + C::x);
  load_rows<DP, C::CT, C::kThreads>(v, kind, d, last, first, sm + C::g);
  load_wt<M, DP, C::kThreads>(W, kind, d, sm + C::wt);
  wait_for_stream_predecessor();
  load_b<M, DP, C::kThreads>(dSg + (size_t)slab * M * kD, sm + C::b);
  for (int i = threadIdx.x; i < M; i += C::kThreads) sm[C::zs + i] = __ldcg(dzg + (size_t)slab * M + i);
  float* R = sm + C::r + me.gid * C::TT * 64;
  const float* zs = sm + C::zs + me.fg * 64 + me.tx;
  cp_async_wait_all();
  __syncthreads();
  for_tiles<C>(first, last, [&](auto ti, int row0) {
    constexpr int T = decltype(ti)::value, TT = 8 * T;   // tokens per thread / per group of this tile
    uint32_t mask[2] = {0u, 0u};   // bit (i & 3) * 8 + j of word i >> 2: R > 0
    {
      float a[T][8];
      gemm_nt<DP, T>(sm + C::x + me.tg * TT * DP, sm + C::wt + me.fg * 64 * DP, me.tx, me.ty, a);
      __syncthreads();   // everybody has read the previous tile's partials; this tile's X is free
      if (row0 + C::CT < last) load_rows<DP, C::CT, C::kThreads>(kf, 0, d, last, row0 + C::CT, sm + C::x);
#pragma unroll
      for (int i = 0; i < T; ++i)
#pragma unroll
        for (int j = 0; j < 8; ++j) {
          mask[i >> 2] |= (a[i][j] > 0.f ? 1u : 0u) << ((i & 3) * 8 + j);
          R[r_index(me.tx, me.ty, i, j)] = fmaxf(a[i][j], 0.f);
        }
    }
    group_sync(me.gid);
    {
      f32x2 out[T][DP / 16];
      gemm_contract<DP, T>(R, sm + C::b + me.fg * 64 * DP, me.tx, me.ty, out);
      group_sync(me.gid);
      put_partial<DP, T>(R, me.tx, me.ty, out);
    }
    __syncthreads();
    combine_rows<C, DP, TT, false>(sm + C::r, nullptr, 0.f, dv, gkind, d, last, row0);
    {
      float a[T][8];
      gemm_nt<DP, T>(sm + C::g + me.tg * TT * DP, sm + C::b + me.fg * 64 * DP, me.tx, me.ty, a);
      __syncthreads();   // dV has been read out of R; this tile's V is free
      if (row0 + C::CT < last) load_rows<DP, C::CT, C::kThreads>(v, kind, d, last, row0 + C::CT, sm + C::g);
#pragma unroll
      for (int i = 0; i < T; ++i)
#pragma unroll
        for (int j = 0; j < 8; ++j)
          R[r_index(me.tx, me.ty, i, j)] = (mask[i >> 2] >> ((i & 3) * 8 + j)) & 1u ? a[i][j] + zs[8 * j] : 0.f;
    }
    group_sync(me.gid);
    {
      f32x2 out[T][DP / 16];
      gemm_contract<DP, T>(R, sm + C::wt + me.fg * 64 * DP, me.tx, me.ty, out);
      group_sync(me.gid);
      put_partial<DP, T>(R, me.tx, me.ty, out);
    }
    cp_async_wait_all();
    __syncthreads();
    combine_rows<C, DP, TT, false>(sm + C::r, nullptr, 0.f, dkf, 0, d, last, row0);
  });
}

// S[slab][i] = sum over chunks of part[slab][chunk][i], always in the same order: four running sums
// take the chunks k = 0, 1, 2, 3 (mod 4) in increasing k (several loads in flight instead of one) and are
// added as (a0 + a1) + (a2 + a3).  T = float or float4.
__device__ __forceinline__ void add_to(float& a, float b) { a += b; }
__device__ __forceinline__ void add_to(float4& a, const float4& b) {
  a.x += b.x;
  a.y += b.y;
  a.z += b.z;
  a.w += b.w;
}
template <typename T, int U = sizeof(T) == 4 ? 16 : 8>
__device__ __forceinline__ T sum_chunks4(const T* __restrict__ p, size_t stride, int chunks) {
  T a[4] = {};
  for (int k = 0; k < chunks; k += U) {   // U loads in flight
    T v[U];
    if (k + U <= chunks) {
#pragma unroll
      for (int q = 0; q < U; ++q) v[q] = p[(size_t)(k + q) * stride];
#pragma unroll
      for (int q = 0; q < U; ++q) add_to(a[q & 3], v[q]);
    } else {
#pragma unroll
      for (int q = 0; q < U - 1; ++q)
        if (k + q < chunks) v[q] = p[(size_t)(k + q) * stride];
#pragma unroll
      for (int q = 0; q < U - 1; ++q)
        if (k + q < chunks) add_to(a[q & 3], v[q]);
    }
  }
  add_to(a[0], a[1]);
  add_to(a[2], a[3]);
  add_to(a[0], a[2]);
  return a[0];
}

// grid (m / (8 J), slabs, feature groups), block 512 / V + 32: one CTA adds the partials of J times eight consecutive features (512
// elements of S', V = 1 or 4 per thread, and by the last warp their eight entries of z') in chunk order.  With Sbf it also leaves the bf16
// copy of S', with Simg the operand image of the query-side kernel (see simg_offset): eight consecutive features
// are one 16-byte chunk of an image row, so the 80 rows of the CTA's part go out as one 16-byte store each.
// ctas > 0: the partials are the segments of the tensor-core backward instead of `chunks` per slab.
// What bounds it is the number of bytes in flight: with one element per thread most of a large grid's time went into
// waves of threads that live for two or three loads, with four a small grid leaves the SMs with too few threads
// (32 x 128 CTAs with 2 or 3 partials, as fp32 S' and bf16: 21 us with V = 1, 14 with 4; 24 x 192: 16 and 12 us;
// 32 x 8 CTAs with 18 partials: a whole forward of 1 x 8 x 131072 201 us with V = 1, 203 with 4).  From 16 such CTAs per SM
// on, four parts in one CTA (J = 4), whose loads go out together where there are up to three partials, as many slabs have:
// 1023 slabs, m = 128 38 -> 26 us of a training step of 271, 192 slabs 16.5 -> 15.6.
template <int V, int J>
__global__ void __launch_bounds__(512 / V + 32) k_reduce_partials(const float* __restrict__ spart,
                                                         const float* __restrict__ zpart, int chunks, int tps, int ctas,
                                                         int m, float* __restrict__ S, float* __restrict__ z,
                                                         __nv_bfloat16* __restrict__ Sbf, uint8_t* __restrict__ Simg) {
  // Programmatic dependent launch: the kernel after this one may be staged now (it waits for this grid
  // before it reads S, z, Sbf, Simg), and this kernel may itself have been staged early: the partials are
  // complete once the kernel before it has finished.
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  asm volatile("griddepcontrol.wait;" ::: "memory");
  __shared__ __align__(16) __nv_bfloat16 tile[J][kSimgRows][8];   // [part][image row][feature of the part]
  // slab counts through the slabs of one group after the other; S and z have a slab's features together
  const int slab = blockIdx.z * gridDim.y + blockIdx.y, f0 = blockIdx.x * 8 * J;
  const size_t out = blockIdx.y * gridDim.z + blockIdx.z;
  const int ns = m * kD;
  size_t slot = (size_t)slab * chunks;          // first partial of this slab
  if (ctas > 0) {   // segments: CTA c has tiles [all c / ctas, all (c + 1) / ctas) of the list of all tiles
    const long long all = (long long)tps * gridDim.y, t0 = (long long)tps * slab;
    const int c0 = (int)(((t0 + 1) * ctas - 1) / all), c1 = (int)(((t0 + tps) * ctas - 1) / all);
    slot = (size_t)c0 + slab;
    chunks = c1 - c0 + 1;
  }
  constexpr int kMain = 512 / V, kThreads = kMain + 32;
  using T = typename std::conditional<V == 4, float4, float>::type;
  if (threadIdx.x < kMain) {
    const int e = V * threadIdx.x;                // first element of the thread in each 8 x 64 part
    const int i = f0 * kD + e;                    // element of S' (feature i / 64, column i % 64) in the first part
    const T* src = reinterpret_cast<const T*>(spart + slot * ns + i);
    T s[J];
    if (J > 1 && chunks <= 3) {   // (the sums of sum_chunks4)
#pragma unroll
      for (int j = 0; j < J; ++j) s[j] = src[j * kMain];
      for (int k = 1; k < chunks; ++k) {
        T v[J];
#pragma unroll
        for (int j = 0; j < J; ++j) v[j] = src[(size_t)k * (ns / V) + j * kMain];
#pragma unroll
        for (int j = 0; j < J; ++j) add_to(s[j], v[j]);
      }
    } else {
#pragma unroll
      for (int j = 0; j < J; ++j) s[j] = sum_chunks4(src + j * kMain, ns / V, chunks);
    }
#pragma unroll
    for (int j = 0; j < J; ++j) {
      *reinterpret_cast<T*>(S + out * ns + i + 512 * j) = s[j];
      union {
        __nv_bfloat16 b[V];
        typename std::conditional<V == 4, uint2, uint16_t>::type all;
      } r;
#pragma unroll
      for (int q = 0; q < V; ++q) {
        r.b[q] = __float2bfloat16_rn(reinterpret_cast<const float*>(&s[j])[q]);
        tile[j][(e & (kD - 1)) + q][e >> 6] = r.b[q];
      }
      if (Sbf != nullptr) *reinterpret_cast<decltype(r.all)*>(Sbf + (size_t)slab * ns + i + 512 * j) = r.all;
    }
  } else {
    const int q = threadIdx.x - kMain;
    if (q < 8 * J) {
      const int r = f0 + q;
      const float zr = sum_chunks4(zpart + slot * m + r, m, chunks);
      z[out * m + r] = zr;
      tile[q >> 3][kD][q & 7] = __float2bfloat16_rn(zr);   // z' is row 64 of the image
    }
    for (int e = q; e < J * (kSimgRows - kD - 1); e += 32)   // rows 65-79 are zero
      *reinterpret_cast<uint4*>(&tile[e / (kSimgRows - kD - 1)][kD + 1 + e % (kSimgRows - kD - 1)][0]) = make_uint4(0u, 0u, 0u, 0u);
  }
  if (Simg == nullptr) return;
  __syncthreads();
  for (int e = threadIdx.x; e < J * kSimgRows; e += kThreads) {
    const int j = e / kSimgRows, row = e - j * kSimgRows;
    *reinterpret_cast<uint4*>(Simg + (size_t)slab * simg_bytes(m) + simg_offset(f0 + 8 * j, row)) =
        *reinterpret_cast<const uint4*>(&tile[j][row][0]);
  }
}

template <typename K>
cudaError_t set_smem(K kernel, size_t bytes) {
  return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
}

// Runs `body` with M, DP, TI, TG as constants: DP = head dimension rounded up to 16, 32 or 64; the tile of four
// groups x 64 tokens, or (p.simt_small: where those would leave SMs idle or with an uneven load, see make_plan)
// one token group of 16 tokens, of which several CTAs share an SM.  One head of 1024 tokens, m = 64: key / query side 12.6 / 12.3 us with the small
// tile, 14.4 / 14.3 with the large one; with tiles for all SMs the small one has a quarter of the operand reuse.
#define WERSA_SIMT_TILE(MM, DD, ...)                                                        \
  if (p.simt_small) { constexpr int M = MM, DP = DD, TI = 2, TG = 1; __VA_ARGS__; }          \
  else { constexpr int M = MM, DP = DD, TI = 8, TG = 256 / MM; __VA_ARGS__; }
#define WERSA_SIMT_DP(MM, ...)                                          \
  if (p.cfg.head_dim > 32) { WERSA_SIMT_TILE(MM, 64, __VA_ARGS__) }      \
  else if (p.cfg.head_dim > 16) { WERSA_SIMT_TILE(MM, 32, __VA_ARGS__) } \
  else { WERSA_SIMT_TILE(MM, 16, __VA_ARGS__) }
#define WERSA_SIMT(...)                                     \
  switch (p.cfg.features) {                                  \
    case 64: { WERSA_SIMT_DP(64, __VA_ARGS__) } break;       \
    case 128: { WERSA_SIMT_DP(128, __VA_ARGS__) } break;     \
    case 256: { WERSA_SIMT_DP(256, __VA_ARGS__) } break;     \
    default: return cudaErrorInvalidValue;                  \
  }

}  // namespace

cudaError_t launch_simt_kside(const Plan& p, const Ws& w, const void* V, const void* W, cudaStream_t st,
                              int* launches) {
  const dim3 grid(p.schunks, p.slabs);
  const int kind = p.bf16 ? 1 : 0;
  cudaError_t err = cudaSuccess;
  WERSA_SIMT({
    using C = Cfg<M, DP, TI, TG, false, true>;
    auto k = k_simt_kside<M, DP, TI, TG>;
    if ((err = set_smem(k, sizeof(float) * C::total)) != cudaSuccess) return err;
    err = launch_after(k, grid, dim3(C::kThreads), sizeof(float) * C::total, st, w.KF, V, W, kind, w.spart, w.zpart,
                       p.cfg.seq_len, p.cfg.head_dim, p.schunk_rows);
  })
  *launches += 1;
  return err != cudaSuccess ? err : cudaGetLastError();
}

static cudaError_t launch_reduce(const Plan& p, int groups, const float* spart, const float* zpart, int chunks, int tps, int ctas,
                                 float* S, float* z, __nv_bfloat16* Sbf, uint8_t* Simg, cudaStream_t st, int* launches,
                                 bool first = false) {
  const int m = p.cfg.features;
  const dim3 grid(m / 8, p.slabs, groups);
  // (four CTAs per SM: see k_reduce_partials; a sequence shard's caller may hand in sums that lie at any float, such as a
  // view into the buffer of a larger all-reduce, and those are read one by one)
  const bool aligned = (reinterpret_cast<uintptr_t>(spart) & 15u) == 0;
  const unsigned ctas8 = grid.x * grid.y * grid.z;
  auto go = [&](auto kernel, dim3 g, int threads) {
    return launch_behind(!first, kernel, g, dim3(threads), 0, st, spart, zpart, chunks, tps, ctas, m, S, z, Sbf, Simg);
  };
  const cudaError_t err = !aligned || ctas8 <= 4u * p.sms ? go(k_reduce_partials<1, 1>, grid, 544)
                          : ctas8 <= 16u * p.sms          ? go(k_reduce_partials<4, 1>, grid, 160)
                                                          : go(k_reduce_partials<4, 4>, dim3(m / 32, grid.y, grid.z), 160);
  *launches += 1;
  return err != cudaSuccess ? err : cudaGetLastError();
}
cudaError_t launch_reduce_partials(const Plan& p, const float* spart, const float* zpart, int chunks, float* S,
                                   float* z, __nv_bfloat16* Sbf, uint8_t* Simg, cudaStream_t st, int* launches, bool first) {
  return launch_reduce(p, p.groups, spart, zpart, chunks, 0, 0, S, z, Sbf, Simg, st, launches, first);
}
cudaError_t launch_reduce_segments(const Plan& p, const Ws& w, cudaStream_t st, int* launches) {
  return launch_reduce(p, 1, w.spart, w.zpart, 0, (p.cfg.seq_len + 127) / 128, p.bctas, w.dS, w.dz, w.dSbf, nullptr, st, launches);
}

cudaError_t launch_simt_qside(const Plan& p, const Ws& w, const void* W, const float* beta, void* O,
                              cudaStream_t st, int* launches) {
  const dim3 grid(p.schunks, p.slabs);
  const int kind = p.bf16 ? 1 : 0;
  cudaError_t err = cudaSuccess;
  WERSA_SIMT({
    using C = Cfg<M, DP, TI, TG, true, false>;
    auto k = k_simt_qside<M, DP, TI, TG>;
    if ((err = set_smem(k, sizeof(float) * C::total)) != cudaSuccess) return err;
    err = launch_after(k, grid, dim3(C::kThreads), sizeof(float) * C::total, st, w.QF, W, kind, w.S, w.z, beta,
                       p.cfg.eps, p.cfg.bw_floor, O, p.cfg.seq_len, p.cfg.head_dim, p.schunk_rows);
  })
  *launches += 1;
  return err != cudaSuccess ? err : cudaGetLastError();
}

cudaError_t launch_simt_bwd_qside(const Plan& p, const Ws& w, const void* W, const float* beta, const void* dO,
                                  cudaStream_t st, int* launches) {
  const dim3 grid(p.schunks, p.slabs);
  const int kind = p.bf16 ? 1 : 0;
  cudaError_t err = cudaSuccess;
  WERSA_SIMT({
    using C = Cfg<M, DP, TI, TG, true, true>;
    auto k = k_simt_bwd_qside<M, DP, TI, TG>;
    if ((err = set_smem(k, sizeof(float) * C::total)) != cudaSuccess) return err;
    err = launch_after(k, grid, dim3(C::kThreads), sizeof(float) * C::total, st, w.QF, W, kind, w.S, w.z, beta,
                       p.cfg.eps, p.cfg.bw_floor, dO, w.dQF, w.spart, w.zpart, w.sumdD, p.cfg.seq_len, p.cfg.head_dim,
                       p.schunk_rows);
  })
  *launches += 1;
  return err != cudaSuccess ? err : cudaGetLastError();
}

cudaError_t launch_simt_bwd_kside(const Plan& p, const Ws& w, const void* V, const void* W, void* dV,
                                  cudaStream_t st, int* launches) {
  const dim3 grid(p.schunks, p.slabs);
  const int kind = p.bf16 ? 1 : 0, gkind = p.grad_bf16 ? 1 : 0;
  cudaError_t err = cudaSuccess;
  WERSA_SIMT({
    using C = Cfg<M, DP, TI, TG, true, true>;
    auto k = k_simt_bwd_kside<M, DP, TI, TG>;
    if ((err = set_smem(k, sizeof(float) * C::total)) != cudaSuccess) return err;
    err = launch_after(k, grid, dim3(C::kThreads), sizeof(float) * C::total, st, w.KF, V, W, kind, w.dS, w.dz, dV,
                       gkind, w.dKF, p.cfg.seq_len, p.cfg.head_dim, p.schunk_rows);
  })
  *launches += 1;
  return err != cudaSuccess ? err : cudaGetLastError();
}

}  // namespace wersa
