// bf16 forward of short slabs in one launch: a slab (and group of at most 256 features) is one cluster of thread blocks, each of
// which holds T consecutive tokens of Q, K and V on chip, so that the mean pool, the gate, the filter, the key summary and the
// output need no pass over memory in between; every sum over the slab (column sums of Q, block sums of the levels above T, S',
// z') goes through the cluster's shared memory.
//
// Why: below some 8,000 tokens the three to five launches of the general path are chains of latencies, 3-5 us each, whatever is
// in them.  Forwards, general path and this one, us: 4 x 1000, m = 128 16.3 -> 10.5; 3 x 130, m = 256 18.9 -> 13; 2 x 300, d = 16,
// m = 128 16.8 -> 8.5; 8 x 64, m = 1024 (with the combination of the groups) 30 -> 15.  What bounds it is latency again: of the 18 k
// cycles of 4 x 1000 the first loads take 3 k, each of the three exchanges 2-3 k, the products 4-5 k, the rest is the gate, the
// filter and code that is fetched for one pass.
//
// Precision is that of tc_fwd.cu: filtered rows, features, S' and z' enter the products as bf16 and every sum is fp32; here
// z' is added up in fp32 and enters D' as two bf16 (hi + lo), and the filter is fp32 until its one rounding.
//
// The products go through warp-level MMAs: they are short (a block has 16 to 128 rows) and their accumulators are the next
// one's operand in the registers, where tcgen05.mma would want its set-up and a way through TMEM for each.  A warp of the key side
// owns 16 features, whose values (accumulators of the projection) are the A operand of S' += Phi^T V; one of the query side 16
// tokens and T features, likewise.
#include "cluster.cuh"
#include "common.cuh"
#include "tc_common.cuh"

namespace wersa {
namespace {
using tc::pack_bf16x2;
using tc::relu_pack_bf16x2;

// Two neighbouring columns of a row (bf16: packed as they were loaded until they are used).
template <typename T> struct Pair { using type = float2; };
template <> struct Pair<__nv_bfloat16> { using type = uint32_t; };
__device__ __forceinline__ float2 pair(float2 v) { return v; }
__device__ __forceinline__ float2 pair(uint32_t u) { return make_float2(__uint_as_float(u << 16), __uint_as_float(u & 0xFFFF0000u)); }

struct GateArgs {
  const float *gate_w, *gate_b, *omega;
  float *qbar, *sg, *f;   // the slab's results, written by one block of the cluster
  int per_head_row;       // row of gate_b: the head, or 0 for the gate of a batch element (of one head)
  int h, L, n, d;
};
// Sums of the eight-row segments of this block, and of all rows of every block, per tensor (0 = Q, 1 = K) and column.
template <int T> struct alignas(16) FilterSmem {
  float seg[2][T / 8][kD];
  float total[kMaxCluster][2][kD];
};

// Mean pool, gate and filter of the block's T tokens of Q and K: put(tensor, token, lane, y0, y1) takes T_f of columns
// 2 lane, 2 lane + 1 (zeros past n and past d), every one of the 32 NW threads calls it for 8-row segments.
// A warp holds segments of eight rows, a lane two columns of them; levels 1-3 are sums of its own rows, the levels up to T come
// from the segments of the block, those above from the blocks' totals, which are the partial sums of the mean pool too.
// Every warp works out the gate for itself: no more barriers.  `late` runs while the other blocks' totals are
// on their way.  Returns f_0.
template <int T, int NW, typename Tin, typename Late, typename Put>
__device__ __forceinline__ float pool_gate_filter(const Tin* __restrict__ Q, const Tin* __restrict__ K, const GateArgs& a, int row0,
                                                 uint32_t rank, uint32_t blocks, FilterSmem<T>& sm, Late&& late, Put&& put) {
  constexpr int kSegs = T / 8, kTasks = 2 * kSegs, kPer = (kTasks + NW - 1) / NW;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, c0 = 2 * lane;
  const int L1 = a.L + 1;
  using Raw = typename Pair<Tin>::type;
  Raw raw[kPer][8];
#pragma unroll
  for (int i = 0; i < kPer; ++i) {
    const int task = warp + i * NW, first = row0 + 8 * (task % kSegs);
    const Tin* src = (task < kSegs ? Q : K) + (size_t)first * a.d + c0;
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      raw[i][j] = Raw();
      if (task < kTasks && c0 < a.d && first + j < a.n) raw[i][j] = *reinterpret_cast<const Raw*>(src + (size_t)j * a.d);
    }
  }
  // (what the gate needs of its weights: the two columns of this lane, fetched ahead of the sums)
  float gw[2][kMaxLevels + 1];
#pragma unroll
  for (int i = 0; i <= kMaxLevels; ++i)
#pragma unroll
    for (int c = 0; c < 2; ++c)
      gw[c][i] = a.gate_w != nullptr && i < L1 && c0 < a.d ? a.gate_w[((size_t)a.h * a.d + c0 + c) * L1 + i] : 0.f;
  const int slot = lane >> 1;   // the level whose logit ends up in this lane
  const float gb = a.gate_b != nullptr && slot < L1 ? a.gate_b[a.per_head_row * L1 + slot] : 0.f;
  const float om = slot < L1 ? a.omega[slot] : 0.f;
#pragma unroll
  for (int i = 0; i < kPer; ++i) {
    const int task = warp + i * NW;
    float2 s = make_float2(0.f, 0.f);
#pragma unroll
    for (int j = 0; j < 8; j += 4) {
      const float2 x0 = pair(raw[i][j]), x1 = pair(raw[i][j + 1]), x2 = pair(raw[i][j + 2]), x3 = pair(raw[i][j + 3]);
      s.x += (x0.x + x1.x) + (x2.x + x3.x);
      s.y += (x0.y + x1.y) + (x2.y + x3.y);
    }
    if (task < kTasks) *reinterpret_cast<float2*>(&sm.seg[task / kSegs][task % kSegs][c0]) = s;
  }
  __syncthreads();
  // this block's totals, to every block: warp w serves tensor w & 1 and the blocks w / 2, w / 2 + NW / 2, ...
  {
    const int tensor = warp & 1;
    float2 s = make_float2(0.f, 0.f);
#pragma unroll
    for (int q = 0; q < kSegs; ++q) {
      const float2 v = *reinterpret_cast<const float2*>(&sm.seg[tensor][q][c0]);
      s.x += v.x;
      s.y += v.y;
    }
    const uint32_t at = shared_addr(&sm.total[rank][tensor][c0]);
    if (blocks > 1) cluster_wait();   // (every block has begun: the caller has arrived)
    for (uint32_t r = warp >> 1; r < blocks; r += NW / 2) peer_store2(peer_addr(at, r), s);
  }
  if (blocks > 1) cluster_release();
  late();
  if (blocks > 1) cluster_acquire();
  else __syncthreads();
  // ---- q-bar (Eq. 1) and the gate (Eqs. 2-3)
  float2 qb = make_float2(0.f, 0.f);
#pragma unroll 4
  for (uint32_t r = 0; r < blocks; ++r) {
    const float2 v = *reinterpret_cast<const float2*>(&sm.total[r][0][c0]);
    qb.x += v.x;
    qb.y += v.y;
  }
  qb.x /= (float)a.n;
  qb.y /= (float)a.n;
  float u[16];
#pragma unroll
  for (int i = 0; i < 16; ++i) u[i] = i <= kMaxLevels && a.gate_w != nullptr && c0 < a.d ? gw[0][i < 9 ? i : 0] * qb.x + gw[1][i < 9 ? i : 0] * qb.y : 0.f;
  // sums over the warp: in four steps a lane passes on half of the values it still holds
#pragma unroll
  for (int s = 8, o = 16; s >= 1; s >>= 1, o >>= 1) {
    const bool up = (lane & o) != 0;
#pragma unroll
    for (int i = 0; i < s; ++i) {
      const float keep = up ? u[i + s] : u[i], send = up ? u[i] : u[i + s];
      u[i] = keep + __shfl_xor_sync(0xffffffffu, send, o);
    }
  }
  const float logit = u[0] + __shfl_xor_sync(0xffffffffu, u[0], 1) + gb;
  const float sgm = 1.f / (1.f + expf(-logit));
  const float fv = sgm * om;
  if (rank == 0 && warp == 0 && a.qbar != nullptr) {
    *reinterpret_cast<float2*>(a.qbar + c0) = qb;
    if ((lane & 1) == 0 && slot < L1) {
      a.sg[slot] = sgm;
      a.f[slot] = fv;
    }
  }
  float k[kMaxLevels + 1];   // k[i] = (f_i - f_{i-1}) / 2^i
  const float f0 = __shfl_sync(0xffffffffu, fv, 0);
  {
    float before = f0, scale = 0.5f;
#pragma unroll
    for (int i = 1; i <= kMaxLevels; ++i) {
      const float fi = __shfl_sync(0xffffffffu, fv, 2 * i);
      k[i] = i < L1 ? (fi - before) * scale : 0.f;
      before = fi;
      scale *= 0.5f;
    }
  }
  // ---- the filter
  constexpr int kTopLevel = T == 16 ? 4 : T == 32 ? 5 : T == 64 ? 6 : 7;   // the block's own levels
  static_assert(1 << kTopLevel == T, "T is a power of two");
#pragma unroll
  for (int i = 0; i < kPer; ++i) {
    const int task = warp + i * NW;
    if (task >= kTasks) break;
    const int tensor = task / kSegs, seg = task % kSegs;
    float2 hi = make_float2(0.f, 0.f);
    const int own = min(a.L, kTopLevel) - 3;   // segments of the block's coarsest level: 2^own
    if (own > 0) {
#pragma unroll
      for (int q = 0; q < kSegs; ++q) {
        if ((q >> own) != (seg >> own)) continue;   // (no other rows, not even with a weight of zero: they may be infinite)
        float w = 0.f;
#pragma unroll
        for (int l = 4; l <= kTopLevel; ++l) w += (q >> (l - 3)) == (seg >> (l - 3)) ? k[l] : 0.f;
        const float2 v = *reinterpret_cast<const float2*>(&sm.seg[tensor][q][c0]);
        hi.x = fmaf(w, v.x, hi.x);
        hi.y = fmaf(w, v.y, hi.y);
      }
    }
    if (a.L > kTopLevel) {   // blocks of 2T rows and more: whole thread blocks of the cluster
      const uint32_t first = rank & ~((1u << (a.L - kTopLevel)) - 1u), last = min(first + (1u << (a.L - kTopLevel)), blocks);
#pragma unroll 1
      for (uint32_t r = first; r < last; ++r) {
        float w = 0.f;
#pragma unroll
        for (int l = kTopLevel + 1; l <= kMaxLevels; ++l) w += (r >> (l - kTopLevel)) == (rank >> (l - kTopLevel)) ? k[l] : 0.f;
        const float2 v = *reinterpret_cast<const float2*>(&sm.total[r][tensor][c0]);
        hi.x = fmaf(w, v.x, hi.x);
        hi.y = fmaf(w, v.y, hi.y);
      }
    }
    float2 x[8], a2[2], s3;
#pragma unroll
    for (int j = 0; j < 8; ++j) x[j] = pair(raw[i][j]);
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      a2[q].x = (x[4 * q].x + x[4 * q + 1].x) + (x[4 * q + 2].x + x[4 * q + 3].x);
      a2[q].y = (x[4 * q].y + x[4 * q + 1].y) + (x[4 * q + 2].y + x[4 * q + 3].y);
    }
    s3.x = a2[0].x + a2[1].x;
    s3.y = a2[0].y + a2[1].y;
    hi.x = fmaf(k[3], s3.x, hi.x);
    hi.y = fmaf(k[3], s3.y, hi.y);
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      const int p = j & ~1;
      const float2 own = x[j], pair = make_float2(x[p].x + x[p + 1].x, x[p].y + x[p + 1].y);
      float y0 = fmaf(f0, own.x, fmaf(k[1], pair.x, fmaf(k[2], a2[j >> 2].x, hi.x)));
      float y1 = fmaf(f0, own.y, fmaf(k[1], pair.y, fmaf(k[2], a2[j >> 2].y, hi.y)));
      const int t = 8 * seg + j;
      const bool on = row0 + t < a.n && c0 < a.d;   // (rows past the end: the trim of Algorithm 2)
      put(tensor, t, lane, on ? y0 : 0.f, on ? y1 : 0.f);
    }
  }
  return f0;
}

constexpr int kPitch = 72;   // elements of a 64-column row in shared memory: rows 8 apart start in different banks

// M features of a group, T tokens of a block, KS steps of 16 columns (the others of a narrow head are zeros).
template <int M, int T, int KS> struct SmallSmem {
  static constexpr int kWarps = M / 16, kThreads = 32 * kWarps;
  static constexpr int kWPitch = M + 8;
  static constexpr int kSumPitch = 16 * KS + 4;   // floats of a row of S' with z' behind it
  static constexpr uint32_t kRowBytes = kSumPitch * 4;
  static constexpr int kTokGroups = T / 16, kSlices = kWarps / kTokGroups;   // of the query side: 16 tokens x T features
  static constexpr uint32_t w_bytes = 16 * KS * kWPitch * 2, s_bytes = M * kPitch * 2;
  static constexpr uint32_t w = 0;                                      // W, 64 x M bf16; later the slab's [S' | z' hi, lo | 0], bf16
  static constexpr uint32_t s = 0;
  static constexpr uint32_t x = w_bytes > s_bytes ? w_bytes : s_bytes;  // T_f(Q), T_f(K)
  static constexpr uint32_t v = x + 2 * T * kPitch * 2;                 // V
  static constexpr uint32_t stage = v + T * kPitch * 2;                 // this block's S' (fp32; column 64: z'); later the slices' [N' | D']
  static constexpr uint32_t recv = stage + M * kRowBytes;               // the other blocks' share of the rows that this one adds up
  static constexpr uint32_t filt = recv + (M + kMaxCluster) * kRowBytes;
  static constexpr uint32_t bars = filt + sizeof(FilterSmem<T>);
  static constexpr uint32_t total = bars + 32;
  static_assert(kSlices * 16 * kTokGroups == M && kSlices >= 1 && total <= 232448, "a warp's share; shared memory of an SM");
};
struct alignas(8) SmallBars {
  uint64_t sums, image;   // the other blocks' sums, their rows of the image
  int abort_flag;
};
enum { kErrSmall = 41 };

__device__ __forceinline__ void cp_async16(uint32_t dst, const void* src, bool valid) {
  const int bytes = valid ? 16 : 0;   // 0: zero fill, the source is not read
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(bytes) : "memory");
}
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_all;" ::: "memory"); }
__device__ __forceinline__ void ldsm4(uint32_t addr, uint32_t (&r)[4]) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0, %1, %2, %3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr) : "memory");
}
__device__ __forceinline__ void ldsm4t(uint32_t addr, uint32_t (&r)[4]) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0, %1, %2, %3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr) : "memory");
}
__device__ __forceinline__ void ldsm2t(uint32_t addr, uint32_t (&r)[2]) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x2.trans.shared.b16 {%0, %1}, [%2];" : "=r"(r[0]), "=r"(r[1]) : "r"(addr) : "memory");
}
// c += a b, 16 x 8 x 16
__device__ __forceinline__ void mma(float (&c)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
  asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};"
               : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
               : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}
// The accumulators of two neighbouring tiles of eight columns, after the ReLU, as the A operand of 16 values of K.
__device__ __forceinline__ void features(const float (&c0)[4], const float (&c1)[4], uint32_t (&a)[4]) {
  a[0] = relu_pack_bf16x2(c0[0], c0[1]);
  a[1] = relu_pack_bf16x2(c0[2], c0[3]);
  a[2] = relu_pack_bf16x2(c1[0], c1[1]);
  a[3] = relu_pack_bf16x2(c1[2], c1[3]);
}
__device__ __forceinline__ float bf_sum(uint32_t u) { return __uint_as_float(u << 16) + __uint_as_float(u & 0xFFFF0000u); }

// grid (blocks, slabs, feature groups), clusters of `blocks`.  m: features of the whole map.  Sbf, Wt: for a backward, or null.
// den: with several groups, every token's denominator times r = bf16(f_0) / f_0 as tc_fwd.cu leaves it, and O is the group's.
// A block whose wait runs out sends and stores nothing from there on; it leaves through the barrier that every block of the cluster
// passes, and not before the copies on their way to it have landed (or had their time).
// kLoss: for the self-test of that, waits are short and block 1 keeps its shares of the sums (1) or its rows of the image (2) to itself.
template <int M, int T, int KS, int kLoss = 0>
__global__ void __launch_bounds__(SmallSmem<M, T, KS>::kThreads, 1)
k_small_forward(const __nv_bfloat16* __restrict__ Q, const __nv_bfloat16* __restrict__ K, const __nv_bfloat16* __restrict__ V,
                const __nv_bfloat16* __restrict__ W, const float* __restrict__ beta, const float* __restrict__ gate_w,
                const float* __restrict__ gate_b, const float* __restrict__ omega, float eps, float bw_floor, int n, int d, int L,
                int H, int per_head, int m, __nv_bfloat16* __restrict__ O, float* __restrict__ den, float* __restrict__ qbar,
                float* __restrict__ sg, float* __restrict__ f, float* __restrict__ S, float* __restrict__ z,
                __nv_bfloat16* __restrict__ Sbf, __nv_bfloat16* __restrict__ Wt, int* __restrict__ status) {
  extern __shared__ __align__(128) uint8_t smem[];
  using SL = SmallSmem<M, T, KS>;
  constexpr int NT = SL::kThreads, kSumPitch = SL::kSumPitch, kTiles = 2 * KS;   // tiles of eight columns
  constexpr uint32_t kRowBytes = SL::kRowBytes;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const uint32_t rank = cluster_rank(), blocks = gridDim.x;
  const int slab = blockIdx.y, group = blockIdx.z, f0g = group * M, row0 = (int)rank * T;
  const int per = (M + (int)blocks - 1) / (int)blocks;   // rows of S' that a block adds up
  constexpr unsigned long long kLimitNs = kLoss == 0 ? tc::kWaitLimitNs : 1000 * 1000;
  const uint32_t base = shared_addr(smem);
  const int count = max(0, min(per, M - (int)rank * per));   // (none for the last block or two where blocks are many)
  SmallBars* bars = reinterpret_cast<SmallBars*>(smem + SL::bars);
  if (tid == 0) {
    tc::mbar_init(&bars->sums, 1);
    tc::mbar_init(&bars->image, 1);
    bars->abort_flag = 0;
    tc::fence_mbar_init();
    tc::mbar_arrive_expect_tx(&bars->sums, blocks * count * kRowBytes);
    tc::mbar_arrive_expect_tx(&bars->image, (M - count) * kPitch * 2);
  }
  if (blocks > 1) cluster_arrive();
  wait_for_stream_predecessor();   // (launched as a programmatic dependent; the first kernel of its pass: see launch_behind)
  let_stream_successor_start();
  const size_t slab_off = (size_t)slab * n * d;
  const GateArgs gate = {gate_w, gate_b, omega, group == 0 ? qbar + (size_t)slab * kD : nullptr, sg + (size_t)slab * (L + 1),
                         f + (size_t)slab * (L + 1), per_head ? slab % H : 0, slab % H, L, n, d};
  const float f0 = pool_gate_filter<T, SL::kWarps>(
      Q + slab_off, K + slab_off, gate, row0, rank, blocks, *reinterpret_cast<FilterSmem<T>*>(smem + SL::filt),
      [&]() {
        constexpr int kWChunks = M / 8;
#pragma unroll 4
        for (int i = tid; i < 16 * KS * kWChunks; i += NT) {
          const int c = i / kWChunks, q = i - c * kWChunks;
          cp_async16(base + SL::w + (c * SL::kWPitch + 8 * q) * 2, W + (c < d ? (size_t)c * m + f0g + 8 * q : 0), c < d);
        }
#pragma unroll 2
        for (int i = tid; i < T * kTiles; i += NT) {
          const int t = i / kTiles, q = i - t * kTiles;
          const bool on = row0 + t < n && 8 * q < d;
          cp_async16(base + SL::v + (t * kPitch + 8 * q) * 2, V + (on ? slab_off + (size_t)(row0 + t) * d + 8 * q : 0), on);
        }
      },
      [&](int tensor, int t, int at, float y0, float y1) {
        *reinterpret_cast<uint32_t*>(smem + SL::x + ((tensor * T + t) * kPitch + 2 * at) * 2) = pack_bf16x2(y0, y1);
      });
  const float bw = fmaxf(beta[0], bw_floor);
  cp_async_wait_all();
  __syncthreads();
  const int r8 = lane & 7, q8 = lane >> 3, g = lane >> 2, q = lane & 3;
  // ---- key side: this warp's 16 features over the block's tokens
  {
    uint32_t wa[KS][4];   // W^T: rows = features
#pragma unroll
    for (int k = 0; k < KS; ++k)
      ldsm4t(base + SL::w + ((16 * k + 8 * (q8 >> 1) + r8) * SL::kWPitch + 16 * warp + 8 * (q8 & 1)) * 2, wa[k]);
    float acc[kTiles][4], z0 = 0.f, z1 = 0.f;
#pragma unroll
    for (int c = 0; c < kTiles; ++c)
#pragma unroll
      for (int j = 0; j < 4; ++j) acc[c][j] = 0.f;
#pragma unroll 2
    for (int t = 0; t < T; t += 16) {
      float p0[4] = {0.f, 0.f, 0.f, 0.f}, p1[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
      for (int k = 0; k < KS; ++k) {
        uint32_t b[4];
        ldsm4(base + SL::x + ((T + t + 8 * (q8 >> 1) + r8) * kPitch + 16 * k + 8 * (q8 & 1)) * 2, b);
        mma(p0, wa[k], b[0], b[1]);
        mma(p1, wa[k], b[2], b[3]);
      }
      uint32_t a[4];
      features(p0, p1, a);
      z0 += bf_sum(a[0]) + bf_sum(a[2]);
      z1 += bf_sum(a[1]) + bf_sum(a[3]);
#pragma unroll
      for (int c = 0; c < KS; ++c) {
        uint32_t b[4];
        ldsm4t(base + SL::v + ((t + 8 * (q8 & 1) + r8) * kPitch + 16 * c + 8 * (q8 >> 1)) * 2, b);
        mma(acc[2 * c], a, b[0], b[1]);
        mma(acc[2 * c + 1], a, b[2], b[3]);
      }
    }
#pragma unroll
    for (int o = 1; o < 4; o <<= 1) {
      z0 += __shfl_xor_sync(0xffffffffu, z0, o);
      z1 += __shfl_xor_sync(0xffffffffu, z1, o);
    }
    float* stage = reinterpret_cast<float*>(smem + SL::stage);
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      float* row = stage + (16 * warp + 8 * h + g) * kSumPitch;
#pragma unroll
      for (int c = 0; c < kTiles; ++c) *reinterpret_cast<float2*>(row + 8 * c + 2 * q) = make_float2(acc[c][2 * h], acc[c][2 * h + 1]);
      if (q == 0) row[8 * kTiles] = h == 0 ? z0 : z1;
    }
  }
  // ---- query side, the features of 16 tokens x T features of this warp
  const int tok = 16 * (warp % SL::kTokGroups), slice = warp / SL::kTokGroups;
  uint32_t phi[T / 16][4];
  {
    uint32_t xa[KS][4];
#pragma unroll
    for (int k = 0; k < KS; ++k)
      ldsm4(base + SL::x + ((tok + 8 * (q8 & 1) + r8) * kPitch + 16 * k + 8 * (q8 >> 1)) * 2, xa[k]);
#pragma unroll
    for (int i = 0; i < T / 16; ++i) {
      const int ft = slice * T + 16 * i;
      float p0[4] = {0.f, 0.f, 0.f, 0.f}, p1[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
      for (int k = 0; k < KS; ++k) {
        uint32_t b[4];
        ldsm4t(base + SL::w + ((16 * k + 8 * (q8 & 1) + r8) * SL::kWPitch + ft + 8 * (q8 >> 1)) * 2, b);
        mma(p0, xa[k], b[0], b[1]);
        mma(p1, xa[k], b[2], b[3]);
      }
      features(p0, p1, phi[i]);
    }
  }
  if (Wt != nullptr && slab == 0) {   // W^T for the backward: rows of 64
    for (int i = tid; i < per * 8; i += NT) {
      const int row = rank * per + i % per, c0 = i / per * 8;
      if (row >= M) continue;
      uint32_t u[4];
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const uint16_t* p = reinterpret_cast<const uint16_t*>(smem + SL::w) + (c0 + 2 * j) * SL::kWPitch + row;
        u[j] = c0 < 16 * KS ? p[0] | (uint32_t)p[SL::kWPitch] << 16 : 0u;
      }
      *reinterpret_cast<uint4*>(Wt + (size_t)(f0g + row) * kD + c0) = make_uint4(u[0], u[1], u[2], u[3]);
    }
  }
  tc::fence_proxy_async_smem();
  __syncthreads();   // (the image may be written over W, by the other blocks too once they have this one's sums)
  if (lane == 0 && !(kLoss == 1 && rank == 1)) {   // their rows to the blocks that add them up, this one among them
    for (uint32_t r = warp; r < blocks; r += SL::kWarps) {
      const int rows = min(per, M - (int)r * per);
      if (rows > 0)
        peer_copy(peer_addr(base + SL::recv + rank * per * kRowBytes, r), base + SL::stage + r * per * kRowBytes, rows * kRowBytes,
                  peer_addr(shared_addr(&bars->sums), r));
    }
  }
  __syncwarp();
  // (one answer per warp until the barriers that stand here anyway; to ask at all takes 0.1 of 10.4 us, 1 x 4 x 1000, m = 128)
  bool ok = __all_sync(0xffffffffu, tc::mbar_wait(&bars->sums, 0, &bars->abort_flag, status, kErrSmall, kLimitNs));
  // ---- S', z' of this block's rows -> the place of the first block's share, and the image's rows
  float* sums = reinterpret_cast<float*>(smem + SL::recv);
  for (int i = ok ? tid : count * (2 * kTiles + 1); i < count * (2 * kTiles + 1); i += NT) {
    const int c = i / count, r = i - c * count;   // pieces of four columns, then z' and what lies behind it
    float4 s = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll 1
    for (uint32_t b0 = 0; b0 < blocks; b0 += 4) {
      float4 v[4];   // (no branch between the loads: one after the other they cost 110 cycles each)
#pragma unroll
      for (uint32_t j = 0; j < 4; ++j) v[j] = *reinterpret_cast<const float4*>(sums + (min(b0 + j, blocks - 1) * per + r) * kSumPitch + 4 * c);
#pragma unroll
      for (uint32_t j = 0; j < 4; ++j) {
        const bool on = b0 + j < blocks;
        s.x += on ? v[j].x : 0.f;
        s.y += on ? v[j].y : 0.f;
        s.z += on ? v[j].z : 0.f;
        s.w += on ? v[j].w : 0.f;
      }
    }
    *reinterpret_cast<float4*>(sums + r * kSumPitch + 4 * c) = s;
    uint8_t* img = smem + SL::s + ((rank * per + r) * kPitch + (c < 2 * kTiles ? 4 * c : 64)) * 2;
    if (c < 2 * kTiles) {
      *reinterpret_cast<uint2*>(img) = make_uint2(pack_bf16x2(s.x, s.y), pack_bf16x2(s.z, s.w));
    } else {
      const float top = __bfloat162float(__float2bfloat16_rn(s.x));
      const float low = fabsf(top) < INFINITY ? s.x - top : 0.f;   // (behind an infinite z' infinity again, or NaN: D' is infinite)
      *reinterpret_cast<uint4*>(img) = make_uint4(pack_bf16x2(top, low), 0u, 0u, 0u);
    }
  }
  if (blocks > 1) tc::fence_proxy_async_smem();
  ok = __syncthreads_and(ok);
  if (blocks > 1 && ok) {
    if (lane == 0 && count > 0 && !(kLoss == 2 && rank == 1))
      for (uint32_t r = warp; r < blocks; r += SL::kWarps) {
        const uint32_t at = base + SL::s + rank * per * kPitch * 2;
        if (r != rank) peer_copy(peer_addr(at, r), at, count * kPitch * 2, peer_addr(shared_addr(&bars->image), r));
      }
    __syncwarp();
    ok = __all_sync(0xffffffffu, tc::mbar_wait(&bars->image, 0, &bars->abort_flag, status, kErrSmall, kLimitNs));
  }
  if (!ok) {
    tc::mbar_wait_drain(&bars->sums, 0, kLimitNs);
    tc::mbar_wait_drain(&bars->image, 0, kLimitNs);
    __syncwarp();
  }
  if (blocks > 1) cluster_arrive();   // (this block has what the others had for it)
  // ---- query side, the contraction
  if (ok) {
    float acc[kTiles + 1][4];   // N', and D' from z' (hi, lo) behind it
#pragma unroll
    for (int c = 0; c < kTiles + 1; ++c)
#pragma unroll
      for (int j = 0; j < 4; ++j) acc[c][j] = 0.f;
#pragma unroll
    for (int i = 0; i < T / 16; ++i) {
      const uint32_t srow = base + SL::s + (slice * T + 16 * i + 8 * (q8 & 1) + r8) * kPitch * 2;
#pragma unroll
      for (int c = 0; c < KS; ++c) {
        uint32_t b[4];
        ldsm4t(srow + (16 * c + 8 * (q8 >> 1)) * 2, b);
        mma(acc[2 * c], phi[i], b[0], b[1]);
        mma(acc[2 * c + 1], phi[i], b[2], b[3]);
      }
      uint32_t b[2];
      ldsm2t(srow + 64 * 2, b);   // (the addresses of lanes 0-15)
      mma(acc[kTiles], phi[i], b[0], b[1]);
    }
    float* red = reinterpret_cast<float*>(smem + SL::stage) + (size_t)slice * T * kSumPitch;
#pragma unroll
    for (int c = 0; c < kTiles + 1; ++c)
      if (c < kTiles || q == 0) {
        *reinterpret_cast<float2*>(red + (tok + g) * kSumPitch + 8 * c + 2 * q) = make_float2(acc[c][0], acc[c][1]);
        *reinterpret_cast<float2*>(red + (tok + g + 8) * kSumPitch + 8 * c + 2 * q) = make_float2(acc[c][2], acc[c][3]);
      }
  }
  if (!__syncthreads_and(ok)) {
    if (blocks > 1) cluster_wait();
    return;
  }
  const float epsp = eps * (float)M * bw * bw;   // (of the group)
  const float* red = reinterpret_cast<const float*>(smem + SL::stage);
  for (int i = tid; i < T * kTiles; i += NT) {
    const int t = i / kTiles, c = i - t * kTiles;
    if (row0 + t >= n || 8 * c >= d) continue;
    float num[8], dn = 0.f;
#pragma unroll
    for (int j = 0; j < 8; ++j) num[j] = 0.f;
#pragma unroll
    for (int s = 0; s < SL::kSlices; ++s) {
      const float* p = red + (s * T + t) * kSumPitch;
      const float4 u = *reinterpret_cast<const float4*>(p + 8 * c), v = *reinterpret_cast<const float4*>(p + 8 * c + 4);
      const float2 zz = *reinterpret_cast<const float2*>(p + 8 * kTiles);
      num[0] += u.x; num[1] += u.y; num[2] += u.z; num[3] += u.w;
      num[4] += v.x; num[5] += v.y; num[6] += v.z; num[7] += v.w;
      dn += zz.x + zz.y;
    }
    dn += epsp;
    const float inv = 1.f / dn;
#pragma unroll
    for (int j = 0; j < 8; ++j) num[j] *= inv;
    store8(O + ((size_t)group * gridDim.y + slab) * n * d + (size_t)(row0 + t) * d + 8 * c, num);
    if (den != nullptr && c == 0) {
      const float fb = __bfloat162float(__float2bfloat16_rn(f0));
      den[((size_t)group * gridDim.y + slab) * n + row0 + t] = f0 != 0.f ? dn * (fb / f0) : dn;
    }
  }
  // S', z' (and for a backward bf16(S')), in rows of 64 columns
  for (int i = tid; i < count * 16; i += NT) {
    const int r = i >> 4, c = i & 15, row = rank * per + r;
    const float4 v = c < 2 * kTiles ? *reinterpret_cast<const float4*>(sums + r * kSumPitch + 4 * c) : make_float4(0.f, 0.f, 0.f, 0.f);
    *reinterpret_cast<float4*>(S + ((size_t)slab * m + f0g + row) * kD + 4 * c) = v;
    if (Sbf != nullptr)
      *reinterpret_cast<uint2*>(Sbf + (((size_t)group * gridDim.y + slab) * M + row) * kD + 4 * c) =
          make_uint2(pack_bf16x2(v.x, v.y), pack_bf16x2(v.z, v.w));
    if (c == 0) z[(size_t)slab * m + f0g + row] = sums[r * kSumPitch + 8 * kTiles];
  }
  if (blocks > 1) cluster_wait();   // (the others have what this block had for them)
}

// Mean pool, gate and filter alone, in front of the FFMA kernels (which follow as they are: with them in the same launch one head of
// 1024 tokens, m = 64, fp32 went from 20.5 to 19.5 us, two thirds of it FFMA passes on 16 SMs).  One launch in the place of
// k_qmean_gate and k_haar_filter, and Q is read once; bound by latency.  Forwards, us, before and now: fp32, d = 64, m = 64 1 x 1000
// 20.7 -> 17.9, 4 x 200 18.7 -> 16.1; d = 16, m = 128 16 x 60 17.2 -> 15.2; bf16, m = 64 1 x 1000 22.5 -> 19.7.
// grid (blocks, slabs), clusters of `blocks`.  place_next: see launch_haar_filter.
constexpr int kFilterWarps = 8;
template <int T, typename Tin>
__global__ void __launch_bounds__(32 * kFilterWarps)
k_small_filter(const Tin* __restrict__ Q, const Tin* __restrict__ K, const float* __restrict__ gate_w, const float* __restrict__ gate_b,
               const float* __restrict__ omega, int n, int d, int L, int H, int per_head, float* __restrict__ qbar,
               float* __restrict__ sg, float* __restrict__ f, float* __restrict__ QF, float* __restrict__ KF, bool place_next) {
  __shared__ FilterSmem<T> sm;
  const uint32_t rank = cluster_rank(), blocks = gridDim.x;
  if (blocks > 1) cluster_arrive();
  wait_for_stream_predecessor();   // (launched as a programmatic dependent; the first kernel of its pass: see launch_behind)
  if (place_next) let_stream_successor_start();
  const int slab = blockIdx.y, row0 = (int)rank * T;
  const size_t slab_off = (size_t)slab * n * d;
  const GateArgs gate = {gate_w, gate_b, omega, qbar + (size_t)slab * kD, sg + (size_t)slab * (L + 1), f + (size_t)slab * (L + 1),
                         per_head ? slab % H : 0, slab % H, L, n, d};
  pool_gate_filter<T, kFilterWarps>(Q + slab_off, K + slab_off, gate, row0, rank, blocks, sm, []() {},
                                    [&](int tensor, int t, int at, float y0, float y1) {
                                      if (row0 + t < n && 2 * at < d)
                                        *reinterpret_cast<float2*>((tensor == 0 ? QF : KF) + slab_off + (size_t)(row0 + t) * d + 2 * at) =
                                            make_float2(y0, y1);
                                    });
}

template <int V> struct Int { static constexpr int value = V; };

// Runs body(kernel, threads, shared memory) with the kernel of p's tile, if there is one.
template <typename F> bool with_small(const Plan& p, F&& body) {
  auto one = [&](auto m, auto t, auto ks) {
    using SL = SmallSmem<decltype(m)::value, decltype(t)::value, decltype(ks)::value>;
    body(k_small_forward<decltype(m)::value, decltype(t)::value, decltype(ks)::value>, (int)SL::kThreads, (size_t)SL::total);
    return true;
  };
  auto width = [&](auto m, auto t) {
    return p.cfg.head_dim <= 16 ? one(m, t, Int<1>()) : p.cfg.head_dim <= 32 ? one(m, t, Int<2>()) : one(m, t, Int<4>());
  };
  const bool wide = p.cfg.features / p.groups == 256;
  switch (p.small_tokens) {
    case 16: return wide ? width(Int<256>(), Int<16>()) : width(Int<128>(), Int<16>());
    case 32: return wide ? width(Int<256>(), Int<32>()) : width(Int<128>(), Int<32>());
    case 64: return wide ? width(Int<256>(), Int<64>()) : width(Int<128>(), Int<64>());
    case 128: return wide ? false : width(Int<128>(), Int<128>());   // (256 features: more than the shared memory)
    default: return false;
  }
}

}  // namespace

template <typename Kernel>
static cudaError_t launch_small(Kernel kernel, int threads, size_t bytes, const Plan& p, const Ws& w, const void* Q, const void* K,
                                const void* V, const void* W, const float* beta, const float* gate_w, const float* gate_b,
                                const float* omega, void* O, cudaStream_t st) {
  using bf = __nv_bfloat16;
  return launch_cluster(kernel, dim3(p.small_blocks, p.slabs, p.groups), dim3(threads), bytes, st, (const bf*)Q, (const bf*)K,
                        (const bf*)V, (const bf*)W, beta, gate_w, gate_b, omega, p.cfg.eps, p.cfg.bw_floor, p.cfg.seq_len,
                        p.cfg.head_dim, p.cfg.levels, p.cfg.heads, p.cfg.gate_per_head, p.cfg.features,
                        p.groups > 1 ? (bf*)w.Og : (bf*)O, p.groups > 1 ? w.den : nullptr, w.qbar, w.sg, w.f, w.S, w.z,
                        p.with_backward ? w.Sbf : nullptr, p.with_backward ? w.Wt : nullptr, w.status);
}

cudaError_t launch_small_forward(const Plan& p, const Ws& w, const void* Q, const void* K, const void* V, const void* W,
                                 const float* beta, const float* gate_w, const float* gate_b, const float* omega, void* O,
                                 cudaStream_t st, int* launches) {
  *launches += 1;
  cudaError_t err = cudaErrorInvalidValue;
  with_small(p, [&](auto kernel, int threads, size_t bytes) {
    err = launch_small(kernel, threads, bytes, p, w, Q, K, V, W, beta, gate_w, gate_b, omega, O, st);
  });
  return err;
}

// The same with block 1 of every cluster keeping its shares of the sums (loss = 1) or its rows of the image (2) to itself.
bool selftest_small_supported(const Plan& p) {
  return p.small_tokens == 16 && p.small_blocks > 1 && p.cfg.features == 128 && p.cfg.head_dim <= 16;
}
cudaError_t launch_selftest_small(const Plan& p, const Ws& w, int loss, const void* Q, const void* K, const void* V, const void* W,
                                  const float* beta, const float* omega, void* O, cudaStream_t st) {
  using SL = SmallSmem<128, 16, 1>;
  auto kernel = loss == 1 ? k_small_forward<128, 16, 1, 1> : k_small_forward<128, 16, 1, 2>;
  const cudaError_t err = prepare_cluster(kernel, SL::total, p.small_blocks);
  return err != cudaSuccess ? err : launch_small(kernel, SL::kThreads, SL::total, p, w, Q, K, V, W, beta, nullptr, nullptr, omega, O, st);
}

// Runs body(kernel) with the kernel of p's tensors and tile.
template <typename F> void with_filter(const Plan& p, F&& body) {
  using bf = __nv_bfloat16;
  if (p.bf16) {
    if (p.filter_tokens == 32) body(k_small_filter<32, bf>, (const bf*)nullptr);
    else body(k_small_filter<64, bf>, (const bf*)nullptr);
  } else {
    if (p.filter_tokens == 32) body(k_small_filter<32, float>, (const float*)nullptr);
    else body(k_small_filter<64, float>, (const float*)nullptr);
  }
}
static int filter_blocks(const Plan& p) { return (p.cfg.seq_len + p.filter_tokens - 1) / p.filter_tokens; }

cudaError_t launch_small_filter(const Plan& p, const Ws& w, const void* Q, const void* K, const float* gate_w, const float* gate_b,
                                const float* omega, cudaStream_t st, int* launches) {
  const int blocks = filter_blocks(p);
  const bool place_next = place_key_side_early(p, (unsigned)(p.slabs * blocks));
  cudaError_t err = cudaErrorInvalidDeviceFunction;
  with_filter(p, [&](auto kernel, auto* type) {
    using P = decltype(type);
    err = launch_cluster(kernel, dim3(blocks, p.slabs), dim3(32 * kFilterWarps), 0, st, (P)Q, (P)K, gate_w, gate_b, omega, p.cfg.seq_len,
                         p.cfg.head_dim, p.cfg.levels, p.cfg.heads, p.cfg.gate_per_head, w.qbar, w.sg, w.f, w.QF, w.KF, place_next);
    *launches += 1;
  });
  return err;
}

// Clusters of p's tile that the device holds at once, and the shared memory of a block.  (The query also prepares the kernel for its
// launches: clusters_at_once.)
static int small_clusters(const Plan& p, size_t* bytes) {
  constexpr int kDevices = 16;
  static KnownClusters known[kDevices][4][2][3][kMaxCluster + 1];
  int clusters = 0;
  with_small(p, [&](auto kernel, int threads, size_t b) {
    *bytes = b;
    const int d = p.cfg.head_dim, t = p.small_tokens;
    auto ask = [&]() { return clusters_at_once(kernel, threads, b, p.small_blocks); };
    clusters = p.cfg.device >= kDevices ? ask()
                                        : known[p.cfg.device][t == 16 ? 0 : t == 32 ? 1 : t == 64 ? 2 : 3]
                                               [p.cfg.features == 128 ? 0 : 1][d <= 16 ? 0 : d <= 32 ? 1 : 2][p.small_blocks].get(ask);
  });
  return clusters;
}

// Likewise of p's filter kernel.
static int filter_clusters(const Plan& p) {
  constexpr int kDevices = 16;
  static KnownClusters known[kDevices][2][2][kMaxCluster + 1];
  const int blocks = filter_blocks(p);
  int clusters = 0;
  auto ask = [&]() {
    with_filter(p, [&](auto kernel, auto*) { clusters = clusters_at_once(kernel, 32 * kFilterWarps, 0, blocks); });
    return clusters;
  };
  return p.cfg.device >= kDevices ? ask() : known[p.cfg.device][p.bf16][p.filter_tokens == 32][blocks].get(ask);
}

// Mean pool, gate and filter of the FFMA forward in one launch: slabs of up to 1024 tokens, in blocks of 32 tokens, 64 where 32
// are too many for a cluster, and as long as the clusters are few.  Forwards, us, by two launches and by one: m = 64, d = 16 16 x 500 (256
// blocks) 17.3 and 15.4, 40 x 200 (280) 18.7 and 18.1, 80 x 200 (560) 22.1 and 24.2; blocks of 64 4 x 1000 (64) 18.2 and
// 16.7, m = 128 16 x 1000 (256) 24.1 and 24.7; of 128 (not built) 1 x 2000 17.7 and 20.1.  With 256 features and more the key side's
// blocks are large and wait behind these: 4 x 200 (28) 17.5 and 15.9, 16 x 60 (32) 19.9 and 18.3, 4 x 500 (64) 19.9 and 21.9.
// Contexts with a backward: see choose_small_forward.
static void choose_small_filter(Plan* p) {
  if (p->use_x || (p->cfg.flags & WERSA_FLAG_SIMT_ONLY) || p->cfg.seq_len > 64 * kMaxCluster) return;
  p->filter_tokens = p->cfg.seq_len <= 32 * kMaxCluster ? 32 : 64;
  const long long clusters = p->slabs, blocks = clusters * filter_blocks(*p);
  const long long most = p->cfg.features >= 256 ? 32 : p->filter_tokens == 32 ? 2 * p->sms : 64;
  if (blocks > most || filter_clusters(*p) <= 0) p->filter_tokens = 0;
}

// The one-launch forward where all slabs and groups fit the device at once, a block an SM: then it was faster than the general
// path in each of 190 shapes (1 to 148 slabs of 64 to 2000 tokens, d = 16, 32, 64, m = 128, 256, 1024; by 1 to 15 us), and a second
// wave of clusters loses (8 x 1000, m = 128: blocks of 64 tokens 20.5 us, of 128 14.1, general 16.6; 16 x 1000 27 and 18.8).  The
// tokens of a block: as few as fit, since a block's time grows with them (m = 128, d = 64 8.4, 9.0, 10.5 and 14.2 us for 16, 32, 64
// and 128), unless that makes blocks share SMs (32 x 64, m = 128: 16 tokens 10.6, 32 9.3).  The gate of a batch element of several
// heads is a sum over slabs, which the clusters do not exchange.  A context with a backward and one feature group takes this launch
// or k_small_filter up to 512 tokens.  They would pay beyond that too; such contexts have kept the bits of a launch per step, and
// nothing else holds the line there.  Forwards of contexts with a backward, us, by steps and by one launch: 1 x 4 x 600, m = 128 20.1
// and 10.3; 1 x 4 x 1000 15.7 and 11.0, m = 256 17.3 and 16.0; 3 x 700, d = 32, m = 256 17.7 and 10.8; 1 x 4 x 2000 16.2 and 14.5; fp32,
// m = 64 1 x 1000 21.0 and 18.2.  (The steps of a sequence shard are launches of their own in every context, and give what
// wersa_forward does up to rounding.)
void choose_small_forward(Plan* p) {
  p->small_tokens = p->small_blocks = p->filter_tokens = 0;
  if ((p->cfg.flags & WERSA_FLAG_STEPWISE) || !(p->cfg.gate_per_head || p->cfg.heads == 1)) return;
  if (p->with_backward && p->groups == 1 && p->cfg.seq_len > 512) return;
  if (!p->use_tc) {
    choose_small_filter(p);
    return;
  }
  constexpr int kTokens[4] = {16, 32, 64, 128};
  constexpr double kCost[4] = {8.4, 9, 10.5, 14};
  Plan best = *p;
  double least = 0;
  for (int i = 0; i < 4; ++i) {
    Plan q = *p;
    q.small_tokens = kTokens[i];
    q.small_blocks = (p->cfg.seq_len + kTokens[i] - 1) / kTokens[i];
    const long long clusters = (long long)p->slabs * p->groups, blocks = clusters * q.small_blocks;
    if (q.small_blocks > kMaxCluster || blocks > p->sms) continue;
    size_t bytes = 0;
    if (small_clusters(q, &bytes) < clusters) continue;
    const bool share = 2 * (bytes + 1024) <= 228 * 1024 && 4 * blocks > 3 * p->sms;
    const double cost = kCost[i] * (share ? 1.5 : 1);
    if (best.small_tokens == 0 || cost < least) {
      best = q;
      least = cost;
    }
  }
  *p = best;
}

}  // namespace wersa
