// bf16 tensor-core (tcgen05 + TMEM + TMA) backward kernels of the WERSA attention path, sm_100a.
// The paper does not write the backward pass; these are the chain rule through Eq. 6 / Eq. 7 with
// dReLU(a)/da = 1[a > 0], on the same unscaled quantities the forward kernels use.
//
// The filtered tensors come as three bf16 planes hi + mid + lo that add up to the fp32 values, so that the mask
// 1[a > 0] of a = X_F W does not flip through rounding; gradients that are rounded to bf16 on their way into a
// further product (dA, dB, and S' in G) enter it as hi + lo pairs.  Both kernels run one CTA per SM over even shares
// of the list of all 128-token tiles, with copies, MMAs, elementwise work and stores in warps of their own.  Every
// mbarrier wait is bounded; a role whose wait expires keeps its control flow (so that group barriers stay balanced)
// but skips all further work, and the host sees the status word.
#include "common.cuh"
#include "tc_common.cuh"
#include "tc_maps.cuh"

namespace wersa {
using namespace tc;

namespace {

constexpr int kTile = 128;
constexpr uint32_t kTileBytes = kTile * kD * 2;   // 128 x 64 bf16
constexpr uint32_t kIdescP = make_idesc_bf16(128, 128, false, false);  // projections: both operands K-major
constexpr uint32_t kIdescC = make_idesc_bf16(128, 64, false, true);    // contractions over features: B N-major
enum { kErrBwdCopy = 21, kErrBwdMma = 22 };

// A 128 x 64 result tile leaves through shared memory and a TMA store: written straight from the
// registers (one token row per lane) every store instruction of a warp would touch 32 different
// 128-byte lines, and the load/store unit stays busy with them for about 2,000 cycles per tile, during
// which the barrier polls and MMA issues of the next step queue behind them.
// stage_row32: columns 32 wg .. 32 wg + 31 of row tl into the staging image, in the 128-byte-swizzled
// layout the store's tensor map describes: fp32 = two boxes of 128 rows x 32 columns (16 KB each, box
// wg), bf16 = one box of 128 rows x 64 columns (16-byte chunks 4 wg .. 4 wg + 3 of the row).
template <typename TG>
__device__ __forceinline__ void stage_row32(uint8_t* stage, int tl, int wg, const uint32_t (&r)[32]);
template <> __device__ __forceinline__ void stage_row32<float>(uint8_t* stage, int tl, int wg, const uint32_t (&r)[32]) {
  uint8_t* box = stage + wg * kTileBytes;
#pragma unroll
  for (int j = 0; j < 8; ++j)
    *reinterpret_cast<uint4*>(box + swz128(tl, j)) = make_uint4(r[4 * j], r[4 * j + 1], r[4 * j + 2], r[4 * j + 3]);
}
template <>
__device__ __forceinline__ void stage_row32<__nv_bfloat16>(uint8_t* stage, int tl, int wg, const uint32_t (&r)[32]) {
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    uint4 v;
    v.x = pack_bf16x2(__uint_as_float(r[8 * j]), __uint_as_float(r[8 * j + 1]));
    v.y = pack_bf16x2(__uint_as_float(r[8 * j + 2]), __uint_as_float(r[8 * j + 3]));
    v.z = pack_bf16x2(__uint_as_float(r[8 * j + 4]), __uint_as_float(r[8 * j + 5]));
    v.w = pack_bf16x2(__uint_as_float(r[8 * j + 6]), __uint_as_float(r[8 * j + 7]));
    *reinterpret_cast<uint4*>(stage + swz128(tl, 4 * wg + j)) = v;
  }
}
// Issued by one thread after the CTA barrier that follows the staging writes (each writer has fenced its
// writes for the async proxy).  Rows past the end of the slab are clipped by the tensor map.
// kAdd: the tile is added to what the tensor holds (feature groups after the first accumulate their share).
// d: columns of the tensor; the second fp32 box (columns 32 ..) only exists for d > 32.
template <typename TG, bool kAdd = false>
__device__ __forceinline__ void store_tile(const CUtensorMap* map, const uint8_t* stage, int row0, int slab, int d) {
  if constexpr (kAdd) {
    tma_reduce_add_3d(map, stage, 0, row0, slab);
    if (sizeof(TG) == 4 && d > 32) tma_reduce_add_3d(map, stage + kTileBytes, 32, row0, slab);
  } else {
    tma_store_3d(map, stage, 0, row0, slab);
    if (sizeof(TG) == 4 && d > 32) tma_store_3d(map, stage + kTileBytes, 32, row0, slab);
  }
  bulk_commit_group();
}

// ---- key side -----------------------------------------------------------------------------------
constexpr int kKElemWarps = 16;   // elementwise warps
constexpr int kKEpiWarp0 = 4 + kKElemWarps;
constexpr int kKThreads = 32 * (kKEpiWarp0 + 4);
constexpr int kKRegsCtl = 40, kKRegsElem = 88, kKRegsEpi = 88, kKRegsLaunch = 80;   // 768 threads: 80 registers each at launch
static_assert(4 * kKRegsCtl + kKElemWarps * kKRegsElem + 4 * kKRegsEpi <= (kKThreads / 32) * kKRegsLaunch,
              "roles may not claim more registers than the CTA was launched with");
constexpr int kKBufs = 3;   // accumulators of 128 TMEM columns

struct alignas(8) BwdKBars {
  uint64_t w_full, x_full[2], v_full[2], s_full[2], s_empty[2];
  uint64_t d_full[kKBufs], d_ready[kKBufs], d_free[kKBufs], dv_full, dv_free, dk_full, dk_free, dv_staged[2], dk_staged[2];
  uint32_t tmem_base;
  int abort_flag;
};
template <int NH> struct BwdKSmem {
  static constexpr int imgs = 2;                                   // dS' images: this slab's and the next one's
  static constexpr uint32_t wt = 0;                                // W^T image, NH x (128 x 64) bf16
  static constexpr uint32_t ds = wt + NH * kTileBytes;             // dS' images, same shape
  // 2 stages of three K_F planes and V; the results of a tile leave through its own stage: dV through planes 0 and 1
  // (dead once B has been formed), dK_F through plane 2 and V (dead once G has)
  static constexpr uint32_t x = ds + imgs * NH * kTileBytes;
  static constexpr uint32_t stage_bytes = 4 * kTileBytes;
  static constexpr uint32_t bars = x + 2 * stage_bytes;
  static constexpr uint32_t total = bars + 512 + 1024;             // + alignment slack
};
static_assert(BwdKSmem<2>::total <= 232448 && BwdKSmem<1>::total <= 232448, "shared memory of an SM");

// One CTA per SM walks an even share of the list of all tiles (slab-major): a tile of this side depends on no other
// tile, only on the dS' image and dz' of its slab.  A tile is 2 NH units of 128 features, B_0 .. G_0 .., each in one
// of three rotating accumulators:
//   unit B_h:  MMA K_F W_h (three planes)   threads: Phi = ReLU -> bf16 pairs in place (kept in registers: the mask)
//              MMA dV += Phi_h dS'_h
//   unit G_h:  MMA V dS'_h^T                threads: dB = (G + dz') 1[Phi > 0] -> hi + lo pairs in place
//              MMA dK_F += dB_h W_h^T
// Warp 0: TMA copies; warp 1: the MMAs that fill units; warp 2: those of dV; warp 3: those of dK_F; warps 4-19
// elementwise (thread = token tl, features 32 wq .. + 31 of the unit); warps 20-23 drain dV and dK_F to shared memory,
// from where warp 0 stores them before it refills the stage.  The tensor pipe takes 4.2 k cycles a tile with m = 256 (1.5 B, 0.5 G, 0.7 dV,
// 1.4 dK_F), 49 % of the time: three accumulators do not hide all of the hand-offs (B=4 H=8 n=16384: 132 us).
template <int NH, typename TG, bool kAdd = false>
__global__ void __launch_bounds__(kKThreads, 1)
k_tc_bwd_kside(const __grid_constant__ CUtensorMap map_kf, const __grid_constant__ CUtensorMap map_v,
               const __grid_constant__ CUtensorMap map_w, const __grid_constant__ CUtensorMap map_ds,
               const float* __restrict__ dzg, const __grid_constant__ CUtensorMap map_dv,
               const __grid_constant__ CUtensorMap map_dkf, int n, int d, int slabs, int* __restrict__ status) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = align_smem(smem_raw);
  using SL = BwdKSmem<NH>;
  BwdKBars* bars = reinterpret_cast<BwdKBars*>(smem + SL::bars);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  constexpr int m = NH * 128;
  constexpr uint32_t kCols = 512, kAccV = 384, kAccK = 448;   // TMEM: three accumulators at 0, dV, dK_F
  const int tps = (n + kTile - 1) / kTile;                    // tiles per slab
  const long long tiles_all = (long long)tps * slabs;
  const int g0 = (int)(tiles_all * blockIdx.x / gridDim.x), nt = (int)(tiles_all * (blockIdx.x + 1) / gridDim.x) - g0;

  if (threadIdx.x == 0) {
    uint64_t* one[] = {&bars->w_full, &bars->dv_full, &bars->dk_full};
#pragma unroll
    for (int i = 0; i < 3; ++i) mbar_init(one[i], 1);
    for (int i = 0; i < 2; ++i) {
      mbar_init(&bars->x_full[i], 1);
      mbar_init(&bars->v_full[i], 1);
      mbar_init(&bars->dv_staged[i], 4);
      mbar_init(&bars->dk_staged[i], 4);
      mbar_init(&bars->s_full[i], 1);
      mbar_init(&bars->s_empty[i], 2);   // G's and dV's last reads
    }
    for (int i = 0; i < kKBufs; ++i) {
      mbar_init(&bars->d_full[i], 1);
      mbar_init(&bars->d_ready[i], kKElemWarps);
      mbar_init(&bars->d_free[i], 1);
    }
    mbar_init(&bars->dv_free, 4);
    mbar_init(&bars->dk_free, 4);
    bars->abort_flag = 0;
    fence_mbar_init();
  }
  if (warp == 1) {
    tmem_alloc(&bars->tmem_base, kCols);
    tmem_relinquish();
  }
  tc_fence_before_sync();
  __syncthreads();
  tc_fence_after_sync();
  const uint32_t tmem = bars->tmem_base;
  volatile int* abort_flag = &bars->abort_flag;
  constexpr uint32_t kTileStep = kTileBytes >> 4;
  const uint32_t hi = smem_desc_hi(1024);

  if (warp < 4) {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(kKRegsCtl));
    if (warp == 0 && lane == 0) {
      // ---- copies
      mbar_arrive_expect_tx(&bars->w_full, NH * kTileBytes);
#pragma unroll
      for (int h = 0; h < NH; ++h) tma_load_3d(smem + SL::wt + h * kTileBytes, &map_w, 0, h * kTile, 0, &bars->w_full);
      griddep_wait();   // (W^T is the forward's; nothing else is read or written before: see launch_after)
      int sent = 0, seg = 0, slab_now = -1;
      bool ok = true;
      auto store_results = [&](int it) {   // of tile `it`, from its stage
        const int slab = (g0 + it) / tps, r0 = (g0 + it - slab * tps) * kTile, s = it & 1;
        const uint8_t* st = smem + SL::x + s * SL::stage_bytes;
        ok = mbar_wait(&bars->dv_staged[s], (it >> 1) & 1, abort_flag, status, kErrBwdMma);
        if (!ok) return;
        store_tile<TG, kAdd>(&map_dv, st, r0, slab, d);
        ok = mbar_wait(&bars->dk_staged[s], (it >> 1) & 1, abort_flag, status, kErrBwdMma);
        if (!ok) return;
        store_tile<float, kAdd>(&map_dkf, st + 2 * kTileBytes, r0, slab, d);
      };
      for (int it = 0; it < nt; ++it) {
        const int slab = (g0 + it) / tps, r0 = (g0 + it - slab * tps) * kTile, s = it & 1;
        if (it >= 2) {
          store_results(it - 2);
          if (!ok) break;
          bulk_wait_group_read0();
        }
        uint8_t* st = smem + SL::x + s * SL::stage_bytes;
        mbar_arrive_expect_tx(&bars->x_full[s], 3 * kTileBytes);
#pragma unroll
        for (int pl = 0; pl < 3; ++pl) tma_load_3d(st + pl * kTileBytes, &map_kf, 0, r0, pl * slabs + slab, &bars->x_full[s]);
        mbar_arrive_expect_tx(&bars->v_full[s], kTileBytes);
        tma_load_3d(st + 3 * kTileBytes, &map_v, 0, r0, slab, &bars->v_full[s]);
        ++sent;
        if (slab != slab_now) {   // the first tile of a slab: its dS' image
          slab_now = slab;
          const int i = seg % SL::imgs;
          ok = mbar_wait(&bars->s_empty[i], ((seg / SL::imgs) & 1) ^ 1, abort_flag, status, kErrBwdCopy);
          if (!ok) break;
          mbar_arrive_expect_tx(&bars->s_full[i], NH * kTileBytes);
#pragma unroll
          for (int h = 0; h < NH; ++h)
            tma_load_3d(smem + SL::ds + (i * NH + h) * kTileBytes, &map_ds, 0, h * kTile, slab, &bars->s_full[i]);
          ++seg;
        }
      }
      for (int it = max(0, nt - 2); it < nt && ok; ++it) store_results(it);
      if (*abort_flag != 0) {   // let copies in flight land before the CTA's shared memory goes away
        mbar_wait_drain(&bars->w_full, 0);
        for (int t = max(0, sent - 2); t < sent; ++t) {
          mbar_wait_drain(&bars->x_full[t & 1], (t >> 1) & 1);
          mbar_wait_drain(&bars->v_full[t & 1], (t >> 1) & 1);
        }
        for (int t = max(0, seg - SL::imgs); t < seg; ++t)
          mbar_wait_drain(&bars->s_full[t % SL::imgs], (t / SL::imgs) & 1);
      }
      bulk_wait_group0();   // the stores read this CTA's shared memory
    } else if (warp == 1 && lane == 0) {
      // ---- MMAs that fill the units
      const int ksteps = (d + 15) >> 4;   // 16 columns of the head dimension each; the others are zeros
      uint32_t wt_k = smem_desc_lo(smem_u32(smem + SL::wt), 16);
      const uint32_t ds_k = smem_desc_lo(smem_u32(smem + SL::ds), 16);
      const uint32_t x_k = smem_desc_lo(smem_u32(smem + SL::x), 16);
      constexpr uint32_t kStageStep = SL::stage_bytes >> 4;
      uint32_t b = 0, round = 0;   // accumulator of the next unit, uses of accumulator 0 so far
      int seg = -1, slab_now = -1;
      bool ok = mbar_wait(&bars->w_full, 0, abort_flag, status, kErrBwdCopy);
      auto next_buf = [&]() {   // the MMA that read this accumulator three units ago must have completed
        if (round > 0) {
          ok = mbar_wait(&bars->d_free[b], (round - 1) & 1, abort_flag, status, kErrBwdMma);
          if (ok) tc_fence_after_sync();
        }
        return ok;
      };
      auto step_buf = [&]() {
        mma_commit(&bars->d_full[b]);
        b = b == kKBufs - 1 ? 0 : b + 1;
        round += b == 0;
      };
      for (int it = 0; it < nt && ok; ++it) {
        const int slab = (g0 + it) / tps, s = it & 1;
        ok = mbar_wait(&bars->x_full[s], (it >> 1) & 1, abort_flag, status, kErrBwdCopy);
        if (!ok) break;
        tc_fence_after_sync();
        asm volatile("" : "+r"(wt_k));   // (opaque: descriptors are recomputed instead of kept in registers)
#pragma unroll 1
        for (int h = 0; h < NH; ++h) {
          if (!next_buf()) break;
          const uint32_t a_lo = x_k + s * kStageStep, b_lo = wt_k + h * kTileStep;
#pragma unroll
          for (int pl = 0; pl < 3; ++pl)
#pragma unroll
            for (int k = 0; k < 4; ++k)
              if (k < ksteps)
                mma_ss(tmem + b * 128, smem_desc_join(a_lo + pl * kTileStep + 2 * k, hi), smem_desc_join(b_lo + 2 * k, hi),
                       kIdescP, (pl > 0 || k > 0) ? 1u : 0u);
          step_buf();
        }
        if (!ok) break;
        if (slab != slab_now) {
          slab_now = slab;
          ++seg;
          ok = mbar_wait(&bars->s_full[seg % SL::imgs], (seg / SL::imgs) & 1, abort_flag, status, kErrBwdCopy);
        }
        ok = ok && mbar_wait(&bars->v_full[s], (it >> 1) & 1, abort_flag, status, kErrBwdCopy);
        if (!ok) break;
        tc_fence_after_sync();
#pragma unroll 1
        for (int h = 0; h < NH; ++h) {
          if (!next_buf()) break;
          const uint32_t a_lo = x_k + s * kStageStep + 3 * kTileStep, b_lo = ds_k + ((seg % SL::imgs) * NH + h) * kTileStep;
#pragma unroll
          for (int k = 0; k < 4; ++k)
            if (k < ksteps)
              mma_ss(tmem + b * 128, smem_desc_join(a_lo + 2 * k, hi), smem_desc_join(b_lo + 2 * k, hi), kIdescP, k > 0);
          step_buf();
        }
        if (!ok) break;
        if ((g0 + it + 1) / tps != slab) mma_commit(&bars->s_empty[seg % SL::imgs]);
      }
    } else if (warp == 2 && lane == 0) {
      // ---- dV
      const uint32_t ds_n = smem_desc_lo(smem_u32(smem + SL::ds), 1024);
      int seg = -1, slab_now = -1;
      bool ok = true;
      for (int it = 0; it < nt && ok; ++it) {
        const int slab = (g0 + it) / tps;
        if (slab != slab_now) {
          slab_now = slab;
          ++seg;
          ok = mbar_wait(&bars->s_full[seg % SL::imgs], (seg / SL::imgs) & 1, abort_flag, status, kErrBwdCopy);
        }
        if (ok && it > 0) ok = mbar_wait(&bars->dv_free, (it - 1) & 1, abort_flag, status, kErrBwdMma);
#pragma unroll 1
        for (int h = 0; h < NH && ok; ++h) {
          const int u = 2 * NH * it + h, b = u % kKBufs;
          ok = mbar_wait(&bars->d_ready[b], (u / kKBufs) & 1, abort_flag, status, kErrBwdMma);
          if (!ok) break;
          tc_fence_after_sync();
          const uint32_t b_lo = ds_n + ((seg % SL::imgs) * NH + h) * kTileStep;
#pragma unroll
          for (int k = 0; k < 8; ++k)   // 32 columns hold the 16 pairs of 32 features
            mma_ts(tmem + kAccV, tmem + b * 128 + 32 * (k >> 1) + 8 * (k & 1), smem_desc_join(b_lo + 128 * k, hi), kIdescC,
                   (h > 0 || k > 0) ? 1u : 0u);
          mma_commit(&bars->d_free[b]);
        }
        if (!ok) break;
        mma_commit(&bars->dv_full);
        if ((g0 + it + 1) / tps != slab) mma_commit(&bars->s_empty[seg % SL::imgs]);
      }
    } else if (warp == 3 && lane == 0) {
      // ---- dK_F
      const uint32_t wt_n = smem_desc_lo(smem_u32(smem + SL::wt), 1024);
      bool ok = mbar_wait(&bars->w_full, 0, abort_flag, status, kErrBwdCopy);
      for (int it = 0; it < nt && ok; ++it) {
        if (it > 0) ok = mbar_wait(&bars->dk_free, (it - 1) & 1, abort_flag, status, kErrBwdMma);
#pragma unroll 1
        for (int h = 0; h < NH && ok; ++h) {
          const int u = 2 * NH * it + NH + h, b = u % kKBufs;
          ok = mbar_wait(&bars->d_ready[b], (u / kKBufs) & 1, abort_flag, status, kErrBwdMma);
          if (!ok) break;
          tc_fence_after_sync();
          const uint32_t b_lo = wt_n + h * kTileStep;
#pragma unroll
          for (int k = 0; k < 8; ++k)
#pragma unroll
            for (int part = 0; part < 2; ++part)   // 16 columns per 16 features: 8 of hi pairs, 8 of lo pairs
              mma_ts(tmem + kAccK, tmem + b * 128 + 16 * k + 8 * part, smem_desc_join(b_lo + 128 * k, hi), kIdescC,
                     (h > 0 || k > 0 || part > 0) ? 1u : 0u);
          mma_commit(&bars->d_free[b]);
        }
        if (!ok) break;
        mma_commit(&bars->dk_full);
      }
    }
  } else if (warp < kKEpiWarp0) {
    asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(kKRegsElem));
    griddep_wait();   // (and no let_stream_successor_start: see there)
    const int wq = (warp - 4) >> 2;
    const uint32_t trow = tmem + ((32u * (warp & 3)) << 16) + 32 * wq;   // this warp's lane quarter and columns
    uint32_t b = 0, par = 0;   // accumulator and phase of the next unit
    bool ok = true;
    auto wait_unit = [&]() {   // one warp of a lane quarter polls
      ok = group_wait(&bars->d_full[b], par, wq == 0, ok, 2 + (warp & 3), 128, abort_flag, status, kErrBwdMma);
      if (ok) tc_fence_after_sync();
    };
    auto done_unit = [&]() {
      if (ok) {
        tmem_st_wait();
        tc_fence_before_sync();
        warp_arrive(&bars->d_ready[b]);
      }
      b = b == kKBufs - 1 ? 0 : b + 1;
      par ^= b == 0;
    };
    for (int it = 0; it < nt; ++it) {
      const int slab = (g0 + it) / tps;
      uint32_t rp[NH][16];
#pragma unroll
      for (int h = 0; h < NH; ++h) {
        wait_unit();
        if (ok) {
          const uint32_t col = trow + b * 128;
          uint32_t r[32];
          tmem_ld32(col, r);
          tmem_ld_wait();
          reg_fence32(r);
#pragma unroll
          for (int j = 0; j < 16; ++j) rp[h][j] = relu_pack_bf16x2(__uint_as_float(r[2 * j]), __uint_as_float(r[2 * j + 1]));
          tmem_st16(col, rp[h]);
        }
        done_unit();
      }
#pragma unroll
      for (int h = 0; h < NH; ++h) {
        const float* z = dzg + (size_t)slab * m + h * 128 + 32 * wq;
        wait_unit();
        if (ok) {
          const uint32_t col = trow + b * 128;
          const f32x2 minus1 = pk2(-1.f, -1.f), one = pk2(1.f, 1.f);
          uint32_t a[2][16];
          tmem_ld16(col, a[0]);
#pragma unroll
          for (int q = 0; q < 2; ++q) {
            uint32_t(&g)[16] = a[q];
            tmem_ld_wait();
            reg_fence16(g);
            if (q == 0) tmem_ld16(col + 16, a[1]);
            uint32_t ph[8], pl[8];
#pragma unroll
            for (int j = 0; j < 8; j += 2) {
              const float4 zz = load4_after_wait(z + 16 * q + 2 * j);
              const f32x2 zp[2] = {pk2(zz.x, zz.y), pk2(zz.z, zz.w)};
#pragma unroll
              for (int i = 0; i < 2; ++i) {
                const f32x2 val = fma2(one, zp[i], pk2u(g[2 * (j + i)], g[2 * (j + i) + 1]));
                const uint32_t mk = positive_mask_bf16x2(rp[h][8 * q + j + i]);
                const uint32_t hv = pack2_bf16(val);
                pl[j + i] = pack2_bf16(fma2(minus1, unpack2_bf16(hv), val)) & mk;
                ph[j + i] = hv & mk;
              }
            }
            tmem_st8(col + 16 * q, ph);
            tmem_st8(col + 16 * q + 8, pl);
          }
        }
        done_unit();
      }
    }
  } else {
    asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(kKRegsEpi));
    const int et = threadIdx.x - 32 * kKEpiWarp0;              // token = TMEM lane
    const uint32_t trow = tmem + ((32u * (warp & 3)) << 16);
    bool ok = true;
    // 64 accumulator columns -> the staging image at `out` (see stage_row32)
    auto drain = [&](uint64_t* full, uint64_t* free_, uint64_t* staged, uint32_t col, uint32_t par, auto tag, uint8_t* out) {
      using T = decltype(tag);
      if (ok) ok = __all_sync(0xffffffffu, mbar_wait(full, par, abort_flag, status, kErrBwdMma));
      if (!ok) return;
      tc_fence_after_sync();
      uint32_t r[32];
      tmem_ld32(trow + col, r);
      tmem_ld_wait();
      reg_fence32(r);
      stage_row32<T>(out, et, 0, r);
      tmem_ld32(trow + col + 32, r);
      tmem_ld_wait();
      reg_fence32(r);
      tc_fence_before_sync();
      warp_arrive(free_);
      stage_row32<T>(out, et, 1, r);
      fence_proxy_async_smem();
      warp_arrive(staged);
    };
    for (int it = 0; it < nt; ++it) {
      uint8_t* st = smem + SL::x + (it & 1) * SL::stage_bytes;
      drain(&bars->dv_full, &bars->dv_free, &bars->dv_staged[it & 1], kAccV, it & 1, TG(), st);
      drain(&bars->dk_full, &bars->dk_free, &bars->dk_staged[it & 1], kAccK, it & 1, float(), st + 2 * kTileBytes);
    }
  }
  tc_fence_before_sync();
  __syncthreads();
  if (warp == 1) {
    tc_fence_after_sync();
    tmem_dealloc(tmem, kCols);
  }
}

// ---- query side ---------------------------------------------------------------------------------
constexpr int kQElemWarps = 16, kQElem = 32 * kQElemWarps;   // elementwise threads
constexpr int kQThreads = 128 + kQElem;
constexpr int kQRegsCtl = 40, kQRegsElem = 104, kQRegsLaunch = 96;   // 640 threads: 96 registers each at launch
static_assert(4 * kQRegsCtl + kQElemWarps * kQRegsElem <= (kQThreads / 32) * kQRegsLaunch,
              "roles may not claim more registers than the CTA was launched with");

struct alignas(8) BwdQBars {
  uint64_t w_full, x_full, x_empty, do_full[2], do_empty[2], s_full, s_free, a_full, a_read, g_full, da_ready[4], dq_full, staged, p_free;
  uint32_t tmem_base;
  int abort_flag;
};
template <int NH> struct BwdQSmem {
  static constexpr uint32_t wt = 0;                          // W^T image
  static constexpr uint32_t shi = wt + NH * kTileBytes;      // S' image, bf16(S')
  static constexpr uint32_t slo = shi + NH * kTileBytes;     // bf16(S' - bf16(S'))
  static constexpr uint32_t p = slo + NH * kTileBytes;       // R / D, 2 NH blocks of 128 tokens x 64 features; result staging
  static constexpr uint32_t scratch = p + 2 * kTileBytes;    // (dz' sums at the end of a segment: R / D is dead then)
  static constexpr uint32_t x = p + 4 * kTileBytes;          // three Q_F planes
  static constexpr int dos = NH == 1 ? 2 : 1;                // buffers of dO
  static constexpr uint32_t g = x + 3 * kTileBytes;          // dO
  static constexpr uint32_t zs = g + dos * kTileBytes;       // NH x 128 floats
  static constexpr uint32_t cs = zs + NH * 512;              // 128 floats
  static constexpr uint32_t bars = cs + 512;
  static constexpr uint32_t total = bars + 256 + 1024;       // + alignment slack
};
static_assert(BwdQSmem<2>::total <= 232448, "shared memory of an SM");
constexpr uint32_t kIdescT = make_idesc_bf16(128, 64, true, true);   // contraction over tokens: both operands MN-major

// One CTA per SM walks an even share of the list of all tiles (slab-major); where the share crosses into the next
// slab it leaves the partial dS', dz' of the slab behind (slot blockIdx.x + slab of the partial buffers: along the
// list either index steps, so slots are distinct and those of one slab are consecutive) and takes up the next one.
// Warp 0: TMA copies.  Warp 1: every MMA.  Warp 2: dQ_F stores.  Warps 4-19: elementwise, thread = token tl (TMEM lane) and features
// 128 h + 32 wq .. + 31 of every half h.  Per tile, all in the accumulator X (m columns of TMEM):
//   MMA:  X = A (three planes)             threads: R = ReLU(A), D' = R . z', summed over the four threads of a token
//                                          (through spare TMEM columns), R / D -> bf16 pairs in registers
//   MMA:  X = G = dO S'^T (S' as hi + lo)  threads: num / D = (R / D) . G, summed likewise, c = - num / D, then half by
//                                          half R / D -> shared memory, dA D = (G + c z') 1[R > 0] -> X as hi + lo pairs
//   MMA, half by half: dS'_h += (R / D)_h^T dO,  dQ_F D += dA_h D W_h^T;  then X = A of the next tile
//   threads meanwhile: dz' += (R / D)^T c from shared memory, then dQ_F (row scaled by 1 / D) -> staging
// dO . O = num / D, so N' is never formed, and dO enters both contractions as it is (bf16, exact).  R / D is rounded from the
// 32-bit R while G is formed: of the weights of dS' and dz' one rounding and no more, and nothing left to pack in the last
// pass (B=4 H=8 n=16384 m=256 202 us; 205 with R rounded first).  What bounds a tile (m = 256): 4.8 k cycles of tensor
// pipe (1.5 A, 1.0 G, 0.8 dS', 1.4 dQ_F; 35 % of the time) plus num and the first half of dA, during which the pipe has
// nothing to do (X is the only accumulator that fits).
// With m = 128 X is double: A of the next tile is formed beside G and the last MMAs of this one, and taken before dz' and dQ_F
// (16 x 12 x 1024 55.4 -> 53.5 us).
// kGroup: the launch handles one group of 256 features of a wider feature map.  The denominator of Eq. 7 and
// dD' then belong to the whole map and come from den_ext / dd_ext (one float per token), and with kAdd the
// group's share of dQ_F is added to what the groups before it left.
template <int NH, bool kGroup = false, bool kAdd = false>
__global__ void __launch_bounds__(kQThreads, 1)
k_tc_bwd_qside(const __grid_constant__ CUtensorMap map_qf, const __grid_constant__ CUtensorMap map_do,
               const __grid_constant__ CUtensorMap map_w, const __grid_constant__ CUtensorMap map_shi,
               const __grid_constant__ CUtensorMap map_slo, const float* __restrict__ zg, int z_stride,
               const float* __restrict__ beta, float eps, float bw_floor,
               const __grid_constant__ CUtensorMap map_dqf, float* __restrict__ dspart, float* __restrict__ dzpart,
               float* __restrict__ sumdD, int n, int d, int slabs, int* __restrict__ status,
               const float* __restrict__ den_ext, const float* __restrict__ dd_ext) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = align_smem(smem_raw);
  using SL = BwdQSmem<NH>;
  BwdQBars* bars = reinterpret_cast<BwdQBars*>(smem + SL::bars);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  constexpr int m = NH * 128;
  constexpr uint32_t kCols = 512, kAccS = 256, kAccQ = 384, kStat = 448;   // TMEM: X at 0, dS'_h, dQ_F, row sums
  const int tps = (n + kTile - 1) / kTile;   // tiles per slab
  const long long tiles_all = (long long)tps * slabs;
  const int g0 = (int)(tiles_all * blockIdx.x / gridDim.x), g1 = (int)(tiles_all * (blockIdx.x + 1) / gridDim.x);

  if (threadIdx.x == 0) {
    uint64_t* one[] = {&bars->w_full, &bars->x_full, &bars->x_empty, &bars->s_full, &bars->s_free, &bars->a_full, &bars->g_full,
                       &bars->dq_full, &bars->p_free};
#pragma unroll
    for (int i = 0; i < 9; ++i) mbar_init(one[i], 1);
    for (int i = 0; i < 2; ++i) {
      mbar_init(&bars->do_full[i], 1);
      mbar_init(&bars->do_empty[i], 1);
    }
    mbar_init(&bars->a_read, kQElemWarps);
    for (int i = 0; i < 4; ++i) mbar_init(&bars->da_ready[i], kQElemWarps);
    mbar_init(&bars->staged, kQElemWarps);
    bars->abort_flag = 0;
    fence_mbar_init();
  }
  if (warp == 1) {
    tmem_alloc(&bars->tmem_base, kCols);
    tmem_relinquish();
  }
  tc_fence_before_sync();
  __syncthreads();
  tc_fence_after_sync();
  const uint32_t tmem = bars->tmem_base;
  volatile int* abort_flag = &bars->abort_flag;

  if (warp < 4) {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(kQRegsCtl));
    if (warp == 0 && lane == 0) {
      // ---- copies.  The planes of the next tile are fetched as soon as A has been formed, dO as soon as dS' has taken it (one
      // buffer; two where the next tile's G is wanted before that), both before they are needed.
      mbar_arrive_expect_tx(&bars->w_full, NH * kTileBytes);
#pragma unroll
      for (int h = 0; h < NH; ++h) tma_load_3d(smem + SL::wt + h * kTileBytes, &map_w, 0, h * kTile, 0, &bars->w_full);
      griddep_wait();   // (W^T is the forward's; nothing else is read or written before: see launch_after)
      int it = 0, seg = -1, slab_now = -1, x_sent = 0, do_sent = 0, s_sent = 0;
      bool ok = true;
      for (int gt = g0; gt < g1; ++gt, ++it) {
        const int slab = gt / tps, r0 = (gt - slab * tps) * kTile;
        if (it > 0) ok = mbar_wait(&bars->x_empty, (it - 1) & 1, abort_flag, status, kErrBwdCopy);
        if (!ok) break;
        mbar_arrive_expect_tx(&bars->x_full, 3 * kTileBytes);
#pragma unroll
        for (int pl = 0; pl < 3; ++pl)
          tma_load_3d(smem + SL::x + pl * kTileBytes, &map_qf, 0, r0, pl * slabs + slab, &bars->x_full);
        ++x_sent;
        const int gb = it % SL::dos;
        if (it >= SL::dos) ok = mbar_wait(&bars->do_empty[gb], (it / SL::dos - 1) & 1, abort_flag, status, kErrBwdCopy);
        if (!ok) break;
        mbar_arrive_expect_tx(&bars->do_full[gb], kTileBytes);
        tma_load_3d(smem + SL::g + gb * kTileBytes, &map_do, 0, r0, slab, &bars->do_full[gb]);
        ++do_sent;
        if (slab != slab_now) {   // a segment begins: the images of S' of its slab
          slab_now = slab;
          ++seg;
          if (seg > 0) ok = mbar_wait(&bars->s_free, (seg - 1) & 1, abort_flag, status, kErrBwdCopy);
          if (!ok) break;
          mbar_arrive_expect_tx(&bars->s_full, 2 * NH * kTileBytes);
#pragma unroll
          for (int h = 0; h < NH; ++h) {
            tma_load_3d(smem + SL::shi + h * kTileBytes, &map_shi, 0, h * kTile, slab, &bars->s_full);
            tma_load_3d(smem + SL::slo + h * kTileBytes, &map_slo, 0, h * kTile, slab, &bars->s_full);
          }
          ++s_sent;
        }
      }
      if (*abort_flag != 0) {   // let copies in flight land before the CTA's shared memory goes away
        mbar_wait_drain(&bars->w_full, 0);
        if (x_sent > 0) mbar_wait_drain(&bars->x_full, (x_sent - 1) & 1);
        for (int t = max(0, do_sent - SL::dos); t < do_sent; ++t) mbar_wait_drain(&bars->do_full[t % SL::dos], (t / SL::dos) & 1);
        if (s_sent > 0) mbar_wait_drain(&bars->s_full, (s_sent - 1) & 1);
      }
    } else if (warp == 1 && lane == 0) {
      // ---- MMAs
      const int ksteps = (d + 15) >> 4;   // 16 columns of the head dimension each; the others are zeros
      const uint32_t hi = smem_desc_hi(1024);
      uint32_t wt_k = smem_desc_lo(smem_u32(smem + SL::wt), 16), wt_n = smem_desc_lo(smem_u32(smem + SL::wt), 1024);
      uint32_t s_k = smem_desc_lo(smem_u32(smem + SL::shi), 16);
      uint32_t x_k = smem_desc_lo(smem_u32(smem + SL::x), 16);
      uint32_t do_k = smem_desc_lo(smem_u32(smem + SL::g), 16), do_n = smem_desc_lo(smem_u32(smem + SL::g), 1024);
      uint32_t p_m = smem_desc_lo(smem_u32(smem + SL::p), kTileBytes);   // 64-feature blocks one tile apart
      constexpr uint32_t kTileStep = kTileBytes >> 4;
      // A and G take all features in one instruction: with N = 256 an instruction reads 12 KB of operands in its 128
      // cycles, with N = 128 8 KB in 64, all the bandwidth shared memory has (measured: 105-115 cycles instead of 64; A in halves,
      // the first of them as soon as dQ_F was done with that half of X, made 4 x 8 x 16384 2 % slower, m = 1024 3 %)
      constexpr uint32_t kIdescX = make_idesc_bf16(128, m, false, false);
      auto issue_a = [&](uint32_t dst) {
        asm volatile("" : "+r"(x_k), "+r"(wt_k));
#pragma unroll
        for (int pl = 0; pl < 3; ++pl)
#pragma unroll
          for (int k = 0; k < 4; ++k)
            if (k < ksteps)
              mma_ss(dst, smem_desc_join(x_k + pl * kTileStep + 2 * k, hi), smem_desc_join(wt_k + 2 * k, hi), kIdescX,
                     (pl > 0 || k > 0) ? 1u : 0u);
        mma_commit(&bars->a_full);
        mma_commit(&bars->x_empty);
      };
      const int nt = g1 - g0;
      int seg = 0, slab_now = -1;
      bool ok = mbar_wait(&bars->w_full, 0, abort_flag, status, kErrBwdCopy) &&
                mbar_wait(&bars->x_full, 0, abort_flag, status, kErrBwdCopy);
      if (ok) {
        tc_fence_after_sync();
        issue_a(tmem);
      }
      for (int it = 0; it < nt && ok; ++it) {
        const uint32_t par = it & 1;
        const uint32_t x = tmem + (NH == 1 ? 128 * par : 0);   // this tile's X
        const bool more = it + 1 < nt;
        // (the empty asm statements: the compiler would keep every descriptor of the unrolled loops in registers)
        const int slab = (g0 + it) / tps, gb = it % SL::dos;
        const bool fresh = slab != slab_now;   // first tile of a segment: dS' starts over
        if (fresh) {
          slab_now = slab;
          ok = mbar_wait(&bars->s_full, seg & 1, abort_flag, status, kErrBwdCopy);
          ++seg;
        }
        ok = ok && mbar_wait(&bars->do_full[gb], (it / SL::dos) & 1, abort_flag, status, kErrBwdCopy) &&
             mbar_wait(&bars->a_read, par, abort_flag, status, kErrBwdMma);
        if (!ok) break;
        tc_fence_after_sync();
        asm volatile("" : "+r"(s_k), "+r"(do_k));
#pragma unroll
        for (int part = 0; part < 2; ++part)
#pragma unroll
          for (int k = 0; k < 4; ++k)
            if (k < ksteps)
              mma_ss(x, smem_desc_join(do_k + gb * kTileStep + 2 * k, hi), smem_desc_join(s_k + part * NH * kTileStep + 2 * k, hi),
                     kIdescX, (part > 0 || k > 0) ? 1u : 0u);
        mma_commit(&bars->g_full);
        if (NH == 1 && more) {   // A of the next tile, in the other X, where the tile before had its dA
          ok = (it == 0 || mbar_wait(&bars->dq_full, par ^ 1, abort_flag, status, kErrBwdMma)) &&
               mbar_wait(&bars->x_full, par ^ 1, abort_flag, status, kErrBwdCopy);
          if (!ok) break;
          tc_fence_after_sync();
          issue_a(tmem + 128 * (par ^ 1));
        }
#pragma unroll 1
        for (int h = 0; h < NH && ok; ++h) {
#pragma unroll 1
          for (int q = 0; q < 2; ++q) {   // features 32 i + 16 q .. + 15 of the half
            ok = mbar_wait(&bars->da_ready[2 * h + q], par, abort_flag, status, kErrBwdMma);
            if (!ok) break;
            tc_fence_after_sync();
            if (q == 1) {
              asm volatile("" : "+r"(p_m), "+r"(do_n));
#pragma unroll
              for (int k = 0; k < 8; ++k)
                mma_ss(tmem + kAccS + h * 64, smem_desc_join(p_m + 2 * h * kTileStep + 128 * k, hi),
                       smem_desc_join(do_n + gb * kTileStep + 128 * k, hi), kIdescT, (!fresh || k > 0) ? 1u : 0u);
              if (h == NH - 1) mma_commit(&bars->do_empty[gb]);
            }
            asm volatile("" : "+r"(wt_n));
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
              for (int part = 0; part < 2; ++part)   // 16 columns per 16 features: 8 of hi pairs, 8 of lo pairs
                mma_ts(tmem + kAccQ, x + h * 128 + 32 * i + 16 * q + 8 * part,
                       smem_desc_join(wt_n + h * kTileStep + 128 * (2 * i + q), hi), kIdescC,
                       (h > 0 || q > 0 || i > 0 || part > 0) ? 1u : 0u);
          }
          if (ok && h == NH - 1) mma_commit(&bars->dq_full);   // (every MMA of the tile)
        }
        if (NH == 2 && ok && more) {   // A of the next tile overwrites X once the MMAs that read dA there have completed
          // (instructions with different shapes and accumulators are not ordered by being issued one after the other)
          ok = mbar_wait(&bars->dq_full, par, abort_flag, status, kErrBwdMma) &&
               mbar_wait(&bars->x_full, par ^ 1, abort_flag, status, kErrBwdCopy);
          if (!ok) break;
          tc_fence_after_sync();
          issue_a(tmem);
        }
      }
    } else if (warp == 2 && lane == 0) {
      // ---- dQ_F stores: the wait for the copy to have read the staging tile (some 1.4 k cycles) holds nobody up
      bool ok = true;
      for (int it = 0; it < g1 - g0; ++it) {
        const int slab = (g0 + it) / tps, row0 = (g0 + it - slab * tps) * kTile;
        ok = mbar_wait(&bars->staged, it & 1, abort_flag, status, kErrBwdMma);
        if (!ok) break;
        store_tile<float, kAdd>(&map_dqf, smem + SL::p, row0, slab, d);
        bulk_wait_group_read0();
        mbar_arrive(&bars->p_free);   // R / D of the next tile may be written
      }
      bulk_wait_group0();   // the stores read this CTA's shared memory
    }
  } else {
    asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(kQRegsElem));
    const int et = threadIdx.x - 128, wq = (warp - 4) >> 2;
    const int tl = 32 * (warp & 3) + lane;                     // token = TMEM lane
    const uint32_t trow = tmem + ((32u * (warp & 3)) << 16);   // this warp's lane quarter
    griddep_wait();
    griddep_launch();
    float* zs = reinterpret_cast<float*>(smem + SL::zs);
    float* cs = reinterpret_cast<float*>(smem + SL::cs);
    float* scratch = reinterpret_cast<float*>(smem + SL::scratch);
    uint8_t* pt = smem + SL::p;
    const float bw = fmaxf(beta[0], bw_floor);
    const float epsp = eps * (float)m * bw * bw;
    // the dz' pass: 16-byte chunk and first token of this thread, tokens per thread
    constexpr int kChunks = m / 8, kDzTok = kTile * kChunks / kQElem;
    const int dz_ch = et % kChunks, dz_t0 = (et / kChunks) * kDzTok;
    bool ok = true;
    float sum_dd = 0.f;   // wq = 0: sum of dD' over this thread's tokens
    // One of the four warps of a lane quarter polls the barrier; the quarter goes on as one or not at all.
    auto wait_all = [&](uint64_t* bar, uint32_t par) {
      ok = group_wait(bar, par, wq == 0, ok, 2 + (warp & 3), 128, abort_flag, status, kErrBwdMma);
      if (ok) tc_fence_after_sync();
    };
    const int nt = g1 - g0;
    // The tile whose A is taken next.  (Stepped along: a division by the tiles of a slab in every thread and tile cost 1 k cycles a tile.)
    int slab = g0 / tps, row0 = (g0 - slab * tps) * kTile;
    uint32_t kept[NH][16];              // NH = 1: R / D of the tile whose A was read last
    float inv = 0.f, c = 0.f;           // 1 / D of the tile whose A was read last (0 past the end: such rows contribute nothing); with kGroup c
    // kGroup: D and dD' of the next tile's token, a tile ahead of their use (with the division above 183 -> 168 us a group of 32 x 4 x
    // 4096, d = 32)
    float ext_d = 1.f, ext_dd = 0.f;
    const float* zr = zs + 32 * wq;
    auto fetch_ext = [&]() {
      const size_t tok = (size_t)slab * n + min(row0 + tl, n - 1);
      ext_d = load_after_wait(den_ext + tok);   // (in this place, not where the values are used)
      ext_dd = load_after_wait(dd_ext + tok);
    };
    if (kGroup && nt > 0) fetch_ext();
    // row sums over the four threads of a token, through spare TMEM columns (four for D', four for num / D)
    auto row_total = [&](int it, uint32_t col, float share) {
      tmem_st1(trow + kStat + col + wq, __float_as_uint(share));
      tmem_st_wait();
      tc_fence_before_sync();
      if (it > 0 && col > 0) wait_all(&bars->p_free, (it & 1) ^ 1);   // (long past, as a rule)
      else named_bar_sync(2 + (warp & 3), 128);
      tc_fence_after_sync();
      uint32_t st[4];
      tmem_ld4(trow + kStat + col, st);
      tmem_ld_wait();
      reg_fence4(st);
      return (__uint_as_float(st[0]) + __uint_as_float(st[1])) + (__uint_as_float(st[2]) + __uint_as_float(st[3]));
    };
    // ---- D', and R / D, rounded to bf16 once from R in 32 bits
    auto take_a = [&](int it, uint32_t (&pp)[NH][16]) {
      const uint32_t xrow = trow + (NH == 1 ? 128u * (it & 1) : 0u);
      const bool on = row0 + tl < n;
      if (it == 0 || row0 == 0) {   // a segment begins (every thread is past its last use of z')
        if (et < m) zs[et] = zg[(size_t)slab * z_stride + et];
        named_bar_sync(1, kQElem);
      }
      row0 += kTile;
      if (row0 >= n) {
        row0 = 0;
        ++slab;
      }
      inv = 0.f;
      if constexpr (kGroup) {
        inv = on ? 1.f / ext_d : 0.f;
        c = on ? ext_dd * ext_d : 0.f;
        if (it + 1 < nt) fetch_ext();
      }
      uint32_t r[NH][32];
      wait_all(&bars->a_full, it & 1);
      if (!ok) return;   // (every wait has one answer for the lane quarter: its barriers may stand inside)
#pragma unroll
      for (int h = 0; h < NH; ++h) tmem_ld32(xrow + h * 128 + 32 * wq, r[h]);
      tmem_ld_wait();
#pragma unroll
      for (int h = 0; h < NH; ++h) reg_fence32(r[h]);
      tc_fence_before_sync();
      warp_arrive(&bars->a_read);   // X may become G
      if constexpr (!kGroup) {
        float den = 0.f, den2 = 0.f;
#pragma unroll
        for (int h = 0; h < NH; ++h) {
#pragma unroll
          for (int j = 0; j < 32; j += 4) {
            if ((j & 7) == 0) asm volatile("" ::: "memory");   // (z' is read as it is used, not kept in registers)
            const float4 z = *reinterpret_cast<const float4*>(zr + h * 128 + j);
            den = fmaf(fmaxf(__uint_as_float(r[h][j]), 0.f), z.x, den);
            den2 = fmaf(fmaxf(__uint_as_float(r[h][j + 1]), 0.f), z.y, den2);
            den = fmaf(fmaxf(__uint_as_float(r[h][j + 2]), 0.f), z.z, den);
            den2 = fmaf(fmaxf(__uint_as_float(r[h][j + 3]), 0.f), z.w, den2);
          }
        }
        const float total = row_total(it, 0, den + den2);
        if (on) inv = 1.f / (epsp + total);
      }
#pragma unroll
      for (int h = 0; h < NH; ++h)
#pragma unroll
        for (int j = 0; j < 16; ++j)
          pp[h][j] = relu_pack_bf16x2(__uint_as_float(r[h][2 * j]) * inv, __uint_as_float(r[h][2 * j + 1]) * inv);
    };
    float dz[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) dz[i] = 0.f;
    // With one half of features X is double, and a tile's A is taken while the MMAs of the tile before it still run.
#pragma unroll 1
    for (int it = NH == 1 ? -1 : 0; it < nt; ++it) {   // (left where a barrier of all threads has given them one answer)
      const uint32_t par = it & 1;
      const uint32_t xrow = trow + (NH == 1 ? 128u * par : 0u);
      uint32_t own[NH][16];   // (of the iteration alone: what was kept would have to be, up to a wait that runs out)
      uint32_t(&pp)[NH][16] = NH == 1 ? kept : own;
      if constexpr (NH == 2) take_a(it, pp);
      const bool last = row0 == 0 || it + 1 == nt;   // the tile ends its segment (its A has been taken, the next one's has not)
      const int now = row0 == 0 ? slab - 1 : slab;   // its slab
      float scale = 0.f;   // of this tile's dQ_F
      if (it >= 0) {
        // ---- num / D = (R / D) . G
        wait_all(&bars->g_full, par);
        if (ok && last && it + 1 < nt && et == 0) mbar_arrive(&bars->s_free);   // (G was the last to read the images of S')
        if constexpr (!kGroup) {
          if (ok) {
            f32x2 num = pk2(0.f, 0.f);
            uint32_t a[16], b[16];
            tmem_ld16(xrow + 32 * wq, a);
#pragma unroll
            for (int h = 0; h < NH; ++h) {
              reg_fence16(pp[h]);   // (R / D is unpacked again in every pass, not kept unpacked)
              tmem_ld_wait();
              reg_fence16(a);
              tmem_ld16(xrow + h * 128 + 32 * wq + 16, b);
#pragma unroll
              for (int j = 0; j < 8; ++j) num = fma2(unpack2_bf16(pp[h][j]), pk2u(a[2 * j], a[2 * j + 1]), num);
              tmem_ld_wait();
              reg_fence16(b);
              if (h + 1 < NH) tmem_ld16(xrow + (h + 1) * 128 + 32 * wq, a);
#pragma unroll
              for (int j = 0; j < 8; ++j) num = fma2(unpack2_bf16(pp[h][8 + j]), pk2u(b[2 * j], b[2 * j + 1]), num);
            }
            c = -row_total(it, 4, sum2(num));
          }
        } else if (it > 0) {
          wait_all(&bars->p_free, par ^ 1);
        }
        if (ok) {
          if (wq == 0) {
            cs[tl] = c;
            sum_dd += c * inv;
          }
          // (with eps = 0 a token without an active feature has D = 0; its dA is zero, and so is its dQ_F)
          scale = inv <= 3.402823466e38f ? inv : 0.f;
          // ---- dA D (hi + lo, in place) and R / D to shared memory, 16 features at a time
          // (the mask 1[R > 0], taken from R / D, cuts the packed pairs: a factor would have to be 1 for the smallest R
          // too, and would let an infinity or NaN of a feature that is off through)
          const f32x2 c2 = pk2(c, c), minus1 = pk2(-1.f, -1.f);
          uint32_t a[2][16];
          tmem_ld16(xrow + 32 * wq, a[0]);
#pragma unroll
          for (int h = 0; h < NH; ++h) reg_fence16(pp[h]);
#pragma unroll
          for (int s = 0; s < 2 * NH; ++s) {
            const int h = s >> 1, q = s & 1;
            const uint32_t col = xrow + h * 128 + 32 * wq + 16 * q;
            uint32_t(&g)[16] = a[s & 1];
            tmem_ld_wait();
            reg_fence16(g);
            if (s + 1 < 2 * NH) tmem_ld16(xrow + ((s + 1) >> 1) * 128 + 32 * wq + 16 * ((s + 1) & 1), a[(s + 1) & 1]);
            const float* z = zr + h * 128 + 16 * q;
            uint32_t ph[8], pl[8];
#pragma unroll
            for (int j = 0; j < 8; ++j) {
              if ((j & 1) == 0) asm volatile("" ::: "memory");
              const float2 zz = *reinterpret_cast<const float2*>(z + 2 * j);
              const uint32_t mk = positive_mask_bf16x2(pp[h][8 * q + j]);
              const f32x2 val = fma2(c2, pk2(zz.x, zz.y), pk2u(g[2 * j], g[2 * j + 1]));
              const uint32_t hv = pack2_bf16(val);
              ph[j] = hv & mk;
              pl[j] = pack2_bf16(fma2(minus1, unpack2_bf16(hv), val)) & mk;
            }
            tmem_st8(col, ph);
            tmem_st8(col + 8, pl);
            uint8_t* blk = pt + (2 * h + (wq >> 1)) * kTileBytes;
            const uint32_t ch = 4 * (wq & 1) + 2 * q;
            const uint32_t* pq = pp[h] + 8 * q;
            *reinterpret_cast<uint4*>(blk + swz128(tl, ch)) = make_uint4(pq[0], pq[1], pq[2], pq[3]);
            *reinterpret_cast<uint4*>(blk + swz128(tl, ch + 1)) = make_uint4(pq[4], pq[5], pq[6], pq[7]);
            tmem_st_wait();
            if (q == 1) fence_proxy_async_smem();   // R / D of the half, for the MMA of dS'
            else asm volatile("" ::: "memory");
            tc_fence_before_sync();
            warp_arrive(&bars->da_ready[s]);
          }
        }
        ok = named_bar_all(1, kQElem, ok);
        if (!ok) break;   // (all quarters together)
      }
      if constexpr (NH == 1) {
        if (it + 1 < nt) take_a(it + 1, pp);
        if (it < 0) continue;
      }
      // ---- dz' += (R / D)^T c: thread = eight features (a 16-byte chunk) x kDzTok tokens.  (As warp-level MMAs the
      // same sums waited for the tensor pipe, which is busy here: 2.9 k cycles.)
      {
        const uint8_t* blk = pt + (dz_ch >> 3) * kTileBytes;
#pragma unroll
        for (int t = 0; t < kDzTok; t += 4) {
          const float4 cv = *reinterpret_cast<const float4*>(cs + dz_t0 + t);
          const float cc[4] = {cv.x, cv.y, cv.z, cv.w};
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            const uint4 w = *reinterpret_cast<const uint4*>(blk + swz128(dz_t0 + t + i, dz_ch & 7));
            const uint32_t u[4] = {w.x, w.y, w.z, w.w};
#pragma unroll
            for (int k = 0; k < 4; ++k) {
              dz[2 * k] = fmaf(__uint_as_float(u[k] << 16), cc[i], dz[2 * k]);
              dz[2 * k + 1] = fmaf(__uint_as_float(u[k] & 0xFFFF0000u), cc[i], dz[2 * k + 1]);
            }
          }
        }
      }
      // ---- dQ_F: 16 columns per thread, times 1 / D, to the staging boxes and out
      wait_all(&bars->dq_full, par);
      uint32_t r[16];
      if (ok) {
        tmem_ld16(trow + kAccQ + 16 * wq, r);
        tmem_ld_wait();
        reg_fence16(r);
        tc_fence_before_sync();
      }
      ok = named_bar_all(1, kQElem, ok);   // the dz' pass has read R / D (and dS' has: its MMAs precede dq_full)
      if (!ok) break;
      {
        uint8_t* box = pt + (wq >> 1) * kTileBytes;
#pragma unroll
        for (int q = 0; q < 4; ++q)
          *reinterpret_cast<float4*>(box + swz128(tl, 4 * (wq & 1) + q)) =
              make_float4(__uint_as_float(r[4 * q]) * scale, __uint_as_float(r[4 * q + 1]) * scale,
                          __uint_as_float(r[4 * q + 2]) * scale, __uint_as_float(r[4 * q + 3]) * scale);
        fence_proxy_async_smem();
      }
      warp_arrive(&bars->staged);
      if (!last) continue;
      // ---- end of the segment: partial dS', dz' (every MMA of the segment has completed)
      {
        float* dst = scratch + (et / kChunks) * m + 8 * dz_ch;
        *reinterpret_cast<float4*>(dst) = make_float4(dz[0], dz[1], dz[2], dz[3]);
        *reinterpret_cast<float4*>(dst + 4) = make_float4(dz[4], dz[5], dz[6], dz[7]);
#pragma unroll
        for (int i = 0; i < 8; ++i) dz[i] = 0.f;
      }
      named_bar_sync(1, kQElem);
      const size_t pidx = (size_t)blockIdx.x + now;
      tc_fence_after_sync();
      if (et < m) {
        float s = 0.f;
#pragma unroll
        for (int q = 0; q < kQElem / kChunks; ++q) s += scratch[q * m + et];
        dzpart[pidx * m + et] = s;
      }
#pragma unroll
      for (int ii = 0; ii < NH; ++ii) {
        const int i = wq * NH + ii, h = i >> 2, cc = i & 3;   // 16 columns of one half
        uint32_t r16[16];
        tmem_ld16(trow + kAccS + h * 64 + 16 * cc, r16);
        tmem_ld_wait();
        reg_fence16(r16);
        float* dst = dspart + (pidx * m + h * 128 + tl) * kD + 16 * cc;
#pragma unroll
        for (int q = 0; q < 4; ++q)
          *reinterpret_cast<uint4*>(dst + 4 * q) = make_uint4(r16[4 * q], r16[4 * q + 1], r16[4 * q + 2], r16[4 * q + 3]);
      }
      tc_fence_before_sync();
      named_bar_sync(1, kQElem);   // the scratch and z' may be written again
    }
    // sum of dD' of this CTA (zero if it gave up)
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) sum_dd += __shfl_xor_sync(0xffffffffu, sum_dd, o);
    if (wq == 0 && lane == 0) scratch[warp - 4] = ok ? sum_dd : 0.f;
    named_bar_sync(1, kQElem);
    if (et == 0) sumdD[blockIdx.x] = (scratch[0] + scratch[1]) + (scratch[2] + scratch[3]);
  }
  tc_fence_before_sync();
  __syncthreads();
  if (warp == 1) {
    tc_fence_after_sync();
    tmem_dealloc(tmem, kCols);
  }
}

// ---- host side ----------------------------------------------------------------------------------
template <int NH, typename TG, bool kAdd = false>
cudaError_t launch_kside(const Plan& p, const Ws& w, const CUtensorMap& map_kf, const CUtensorMap& map_v, void* dV,
                         cudaStream_t st) {
  CUtensorMap map_w, map_ds, map_dv, map_dkf;
  cudaError_t err;
  if ((err = make_tile_map(w.Wt, 1, p.cfg.features, &map_w)) != cudaSuccess) return err;
  if ((err = make_tile_map(w.dSbf, p.slabs, p.cfg.features, &map_ds)) != cudaSuccess) return err;
  if ((err = make_out_map(dV, p.slabs, p.cfg.seq_len, p.cfg.head_dim, sizeof(TG) == 2, &map_dv)) != cudaSuccess) return err;
  if ((err = make_out_map(w.dKF, p.slabs, p.cfg.seq_len, p.cfg.head_dim, false, &map_dkf)) != cudaSuccess) return err;
  auto k = k_tc_bwd_kside<NH, TG, kAdd>;
  if ((err = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, BwdKSmem<NH>::total)) != cudaSuccess)
    return err;
  return launch_after(k, dim3(p.bctas), dim3(kKThreads), BwdKSmem<NH>::total, st, map_kf, map_v, map_w, map_ds, w.dz,
                      map_dv, map_dkf, p.cfg.seq_len, p.cfg.head_dim, p.slabs, w.status);
}

template <int NH, bool kGroup = false, bool kAdd = false>
cudaError_t launch_qside(const Plan& p, const Ws& w, const CUtensorMap& map_qf, const CUtensorMap& map_do,
                         const float* beta, cudaStream_t st, const float* den_ext = nullptr,
                         const float* dd_ext = nullptr) {
  CUtensorMap map_w, map_shi, map_slo, map_dqf;
  cudaError_t err;
  if ((err = make_tile_map(w.Wt, 1, p.cfg.features, &map_w)) != cudaSuccess) return err;
  if ((err = make_tile_map(w.Sbf, p.slabs, p.cfg.features, &map_shi)) != cudaSuccess) return err;
  if ((err = make_tile_map(w.Slo, p.slabs, p.cfg.features, &map_slo)) != cudaSuccess) return err;
  if ((err = make_out_map(w.dQF, p.slabs, p.cfg.seq_len, p.cfg.head_dim, false, &map_dqf)) != cudaSuccess) return err;
  auto k = k_tc_bwd_qside<NH, kGroup, kAdd>;
  if ((err = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, BwdQSmem<NH>::total)) != cudaSuccess)
    return err;
  return launch_after(k, dim3(p.bctas), dim3(kQThreads), BwdQSmem<NH>::total, st, map_qf, map_do, map_w, map_shi, map_slo,
                      w.z, p.cfg.features * p.groups, beta, p.cfg.eps, p.cfg.bw_floor, map_dqf, w.spart, w.zpart, w.sumdD, p.cfg.seq_len,
                      p.cfg.head_dim, p.slabs, w.status, den_ext, dd_ext);
}

}  // namespace

cudaError_t launch_tc_bwd_qside(const Plan& p, const Ws& w, const void* QF3, const float* beta, const void* dO,
                                const float* den_ext, const float* dd_ext, bool add, cudaStream_t st, int* launches) {
  CUtensorMap map_qf, map_do;
  cudaError_t err;
  if ((err = make_tile_map(QF3, 3 * p.slabs, p.cfg.seq_len, &map_qf, p.cfg.head_dim)) != cudaSuccess) return err;
  if ((err = make_tile_map(dO, p.slabs, p.cfg.seq_len, &map_do, p.cfg.head_dim)) != cudaSuccess) return err;
  *launches += 1;
  if (den_ext != nullptr) {   // one group of 256 features of a wider map
    if (p.cfg.features != 256 || dd_ext == nullptr) return cudaErrorInvalidValue;
    return add ? launch_qside<2, true, true>(p, w, map_qf, map_do, beta, st, den_ext, dd_ext)
               : launch_qside<2, true, false>(p, w, map_qf, map_do, beta, st, den_ext, dd_ext);
  }
  return p.cfg.features == 256 ? launch_qside<2>(p, w, map_qf, map_do, beta, st)
                               : launch_qside<1>(p, w, map_qf, map_do, beta, st);
}

cudaError_t launch_tc_bwd_kside(const Plan& p, const Ws& w, const void* KF3, const void* V, void* dV, bool add,
                                cudaStream_t st, int* launches) {
  CUtensorMap map_kf, map_v;
  cudaError_t err;
  if ((err = make_tile_map(KF3, 3 * p.slabs, p.cfg.seq_len, &map_kf, p.cfg.head_dim)) != cudaSuccess) return err;
  if ((err = make_tile_map(V, p.slabs, p.cfg.seq_len, &map_v, p.cfg.head_dim)) != cudaSuccess) return err;
  *launches += 1;
  if (add) {   // a feature group after the first: dV and dK_F accumulate
    if (p.cfg.features != 256) return cudaErrorInvalidValue;
    return p.grad_bf16 ? launch_kside<2, __nv_bfloat16, true>(p, w, map_kf, map_v, dV, st)
                       : launch_kside<2, float, true>(p, w, map_kf, map_v, dV, st);
  }
  if (p.cfg.features == 256)
    return p.grad_bf16 ? launch_kside<2, __nv_bfloat16>(p, w, map_kf, map_v, dV, st)
                       : launch_kside<2, float>(p, w, map_kf, map_v, dV, st);
  return p.grad_bf16 ? launch_kside<1, __nv_bfloat16>(p, w, map_kf, map_v, dV, st)
                     : launch_kside<1, float>(p, w, map_kf, map_v, dV, st);
}

}  // namespace wersa
