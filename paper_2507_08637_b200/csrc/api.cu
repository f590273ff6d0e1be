// C-ABI layer of the WERSA library: configuration checks, workspace planning and the launch
// sequences of the forward and backward passes.  All arithmetic lives in the kernels.
#include <new>

#include "common.cuh"

namespace wersa {

bool tc_supported(const wersa_config& cfg);   // tc_fwd.cu

namespace {

size_t align_up(size_t x, size_t a) { return (x + a - 1) / a * a; }
constexpr long long kXUnits = 64;   // (see make_plan)
constexpr double kXBytes = 64. * (1 << 30);
int ceil_div(int a, int b) { return (a + b - 1) / b; }
int next_pow2(int n) {
  int p = 1;
  while (p < n) p <<= 1;
  return p;
}
// Streaming multiprocessors of the device the plan is made for: the chunk counts below aim at whole
// waves of CTAs.  Without a device (host-only sizing queries) the count of a B200 is assumed.
int device_sm_count(int device) {
  int sms = 0;
  if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, device) != cudaSuccess || sms < 1) {
    cudaGetLastError();   // a failed query leaves no sticky error behind
    sms = 148;
  }
  return sms;
}

}  // namespace

// The checks of a configuration and the split of the mean pool: all of a plan that wersa_gate_static needs, which makes
// one on every call (with the search for the fp32 kernels' tiles behind it 1.2 to 5.8 us of host time, without 0.4).
static wersa_status make_pool_plan(const wersa_config& c, Plan* p) {
  if (c.batch < 1 || c.heads < 1 || c.seq_len < 2 || c.head_dim < 1 || c.levels < 1 || c.features < 1)
    return WERSA_ERR_INVALID_ARG;
  if (c.dtype != WERSA_F32 && c.dtype != WERSA_BF16) return WERSA_ERR_INVALID_ARG;
  if (c.grad_dtype != WERSA_F32 && c.grad_dtype != WERSA_BF16) return WERSA_ERR_INVALID_ARG;
  if (!(c.eps >= 0.f) || !(c.bw_floor > 0.f)) return WERSA_ERR_INVALID_ARG;
  if (c.device < 0) return WERSA_ERR_INVALID_ARG;
  if (c.levels <= 30 && (1LL << c.levels) > (long long)next_pow2(c.seq_len)) return WERSA_ERR_INVALID_ARG;
  // head dimensions 8, 16, ... 64
  if (c.head_dim > kD || c.head_dim < 8 || c.head_dim % 8 != 0) return WERSA_ERR_UNSUPPORTED;
  if (c.levels > kMaxLevels) return WERSA_ERR_UNSUPPORTED;
  // feature maps of 64, 128 or 256, and (bf16 tensor-core path) 512, 768, 1024 in groups of 256
  const bool grouped = c.features > kGroupFeatures;
  if (grouped) {
    if (c.features % kGroupFeatures != 0 || c.features > 4 * kGroupFeatures) return WERSA_ERR_UNSUPPORTED;
    if (c.dtype != WERSA_BF16 || (c.flags & WERSA_FLAG_SIMT_ONLY)) return WERSA_ERR_UNSUPPORTED;
  } else if (c.features != 64 && c.features != 128 && c.features != 256) {
    return WERSA_ERR_UNSUPPORTED;
  }
  if ((long long)c.batch * c.heads > 65535) return WERSA_ERR_UNSUPPORTED;   // gridDim.y

  *p = Plan();   // (what is not decided here or in make_plan, or not on this device, is 0)
  p->cfg = c;
  p->slabs = c.batch * c.heads;
  p->L1 = c.levels + 1;
  p->bf16 = c.dtype == WERSA_BF16;
  p->grad_bf16 = c.grad_dtype == WERSA_BF16;
  p->with_backward = !(c.flags & WERSA_FLAG_FORWARD_ONLY);
  p->dpad = c.head_dim < kD;
  p->groups = grouped ? c.features / kGroupFeatures : 1;
  p->use_tc = p->bf16 && !(c.flags & WERSA_FLAG_SIMT_ONLY) && tc_supported(c);
  const int n = c.seq_len;
  p->sms = device_sm_count(c.device);

  p->qchunks = ceil_div(4 * p->sms, p->slabs);
  if (p->qchunks > ceil_div(n, 128)) p->qchunks = ceil_div(n, 128);
  if (p->qchunks < 1) p->qchunks = 1;
  // In a context the chunks of a slab are one cluster (of at most 16) where that still covers most of the SMs and a chunk is not long: training
  // steps of 2 x 4 x 4096, d = 32, fp32 104.6 -> 103.3 us, of 4 x 8 x 16384 710.7 -> 703.9; forwards of 2 x 8 x 4096, fp32 96.6 -> 95.7.
  // With fewer slabs up to 1 MB of Q a slab (2 MB where the tensor-core key side has its first copies under way meanwhile): what
  // the counters take is then more than the longer chunks do.  Forwards, us, more chunks and 16: bf16 2 x 3994, d = 32, m = 512 22.1
  // and 20.3, 1 x 16000, d = 16, m = 128 21.9 and 19.0, d = 64, m = 256 22.8 and 21.8; m = 64 1 x 8000 25.1 and 24.0, 2 x 16000 (2 MB) 34.5
  // and 35.4; fp32 1 x 3994, m = 256 28.3 and 27.7, 1 x 11000 (2.8 MB) 37.5 and 38.6.
  // At the end of the range of lengths, forwards of 7, 8 and 12 slabs of d = 64, m = 256, bf16: 16384 tokens 40.5, 41.1, 52.2 and 39.7, 40.2,
  // 50.9; beyond it 16 chunks would give 16500 41.4, 42.2, 52.2 and 40.9, 41.7, 51.5, 20000 42.1, 45.9, 57.5 and 42.7, 46.0, 57.1, 32768
  // 56.8, 59.5, 77.8 and 59.5, 62.7, 79.6; fp32, m = 128 7 x 16384 103.3 and 103.7, 7 x 20000 119.5 and 121.1.  (Narrow heads would
  // gain further on, 1 x 17000, d = 16 23.6 and 20.5, and are cut as before.)
  // qchunks are those of launches that keep arrival counters: wersa_gate_static (8 slabs of 16384, fp32 14.5 us, with 16 chunks 16.6; but
  // 32 slabs of 4096, bf16 12.2 and 10.4), and where a cluster finds no room.
  const long long slab_bytes = (long long)n * c.head_dim * (p->bf16 ? 2 : 4);
  const bool few = slab_bytes <= (p->use_tc ? 2 << 20 : 1 << 20);
  int pool = p->qchunks;
  if (pool > 16 && (few || 16 * p->slabs * 4 >= 3 * p->sms) && n <= 16 * 1024) pool = 16;
  p->qcluster_rows = ceil_div(ceil_div(n, pool), 32) * 32;
  p->qcluster = ceil_div(n, p->qcluster_rows);
  if (p->qcluster > 16) p->qcluster = 0;
  p->qchunk_rows = ceil_div(ceil_div(n, p->qchunks), 32) * 32;
  p->qchunks = ceil_div(n, p->qchunk_rows);
  return WERSA_OK;
}

wersa_status make_plan(const wersa_config& c, Plan* p) {
  const wersa_status s = make_pool_plan(c, p);
  if (s != WERSA_OK) return s;
  const int n = c.seq_len, m = c.features;
  const bool grouped = p->groups > 1;
  p->htiles = ceil_div(n, kHaarTile);

  // fp32 FFMA kernels: a CTA tile is 64 tokens x (256 / m) token groups, one CTA per SM, or 16 tokens, of which m = 64
  // lets four and m = 128 two CTAs share an SM; a chunk is a whole number of quarter tiles.  Tile and chunk count minimise
  // an estimate of a training step's four kernels and two reductions in us, fitted to d = 64: a full tile 105, 93 or 88
  // (m = 64, 128, 256; a last quarter 0.4 of it) and 7 for a CTA's start; a small one 22.7, 25.5 or 31, a fifth (m = 128: a
  // quarter) more for every further CTA that an SM holds at once, all of it again for those it does not, and 4 (m = 256: 8)
  // for a CTA's start.
  // Training steps, small against full tiles: 10 slabs of 1344, m = 64 108 us (two tiles a chunk; 181 with six) and 127;
  // 16 of 500, m = 128 108 and 120; 4 of 700, m = 256 107 and 127; but 64 of 1024, m = 64 333 and 275; 8 of 4096, d = 32,
  // m = 128 193 and 138; 40 of 600, m = 128 261 (304 with one tile a chunk) and 235.  One slab of 20000, m = 256, forward: 148 chunks 92 us, 64 (the earlier limit) 159 us.
  p->simt_small = false;
  p->schunks = 1;
  p->schunk_rows = n;
  double ffma_cost = 0;
  if (!p->use_tc) {
    const int mt = m < 256 ? m : 256;
    const int big = 64 * (256 / mt), share = 256 / mt;
    const double t_big = mt == 64 ? 105 : mt == 128 ? 93 : 88, t_small = mt == 64 ? 22.7 : mt == 128 ? 25.5 : 31;
    const double more = mt == 64 ? 0.2 : 0.26;
    double best = -1;
    int rows_best = 0;
    for (int small = 0; small < 2; ++small) {
      const int tile = small ? 16 : big, unit = small ? 16 : big / 4;
      int rows_before = 0;
      for (int ch = 1; ch <= ceil_div(n, unit) && ch <= 256; ++ch) {
        const int rows = ceil_div(ceil_div(n, ch), unit) * unit, left = rows % tile, chunks = ceil_div(n, rows);
        if (rows == rows_before) continue;
        rows_before = rows;
        const int ctas = ceil_div(p->slabs * chunks, p->sms);   // of one SM
        const double tiles = rows / tile + (left == 0 ? 0.0 : left <= unit ? 0.4 : 1.0);
        const int rest = ctas % share;
        const double rounds = ctas / share * (1 + more * (share - 1)) + (rest > 0 ? 1 + more * (rest - 1) : 0);
        const double cost = 0.07 * chunks + (small ? t_small * tiles * rounds + (share == 1 ? 8 : 4) * ctas : ctas * (t_big * tiles + 7));
        if (best < 0 || cost < best) {
          best = cost;
          rows_best = rows;
          p->simt_small = small != 0;
        }
      }
    }
    p->schunk_rows = rows_best;
    p->schunks = ceil_div(n, rows_best);
    ffma_cost = best;
  }

  // fp32 arithmetic on the tensor cores, of fp32 tensors and of bf16 ones with m = 64: one CTA per SM and group, in chunks that minimise waves x (tiles + 3), 3 tiles being about what
  // a CTA spends before its first and after its last one, and a 64th of a tile for a chunk's partial in the reduction.  Up to
  // a chunk per SM: one slab of 131072, m = 128 in 64 chunks against 147, forward d = 16 121 -> 83 us (FFMA 101), d = 64 165 ->
  // 124; training step d = 16 368 -> 239 (294), d = 64 500 -> 348.
  // Planes multiply tiles of 128 tokens and 64 columns whatever is in them, the FFMA kernels 16 tokens and 16, 32 or 64 columns:
  // short slabs and narrow heads are theirs.  The line lies where two estimates in us meet, fitted to 435 shapes of 1 to
  // 1023 slabs, 16 to 131072 tokens, d = 8 to 64, m = 128 and 256 (rms 4 % off for planes, 10 % for FFMA; 10 of the 435 choices
  // cost more than 5 %).  Per unit of the FFMA plan's cost, with full and small tiles.  FFMA and planes, us:
  //   forward  1 x 8192, d = 16, m = 128 37 27;  1 x 16384 29 34;   300 x 128 56 64;    148 x 256 38 37;    1023 x 16 60 153
  //            512 x 64, d = 32, m = 128 77 89;  256 x 64 54 49;    300 x 128 77 65;    100 x 200 62 34
  //            512 x 32, d = 64, m = 256 164 156; 148 x 40 50 52;   1023 x 16 192 314;  200 x 50, m = 128 76 50
  //   backward 300 x 128, d = 16, m = 128 109 123; 8 x 8192 111 97; 512 x 64, d = 32 146 178; 300 x 128 155 136
  // With m = 128, 256 from kXUnits tiles x groups of 128 features on, the backward from one tile per SM on (below these lines
  // planes have not been chosen, whatever the estimates say).
  // Their operands as planes take more memory than the FFMA kernels' fp32 ones (see the layout below): a problem that asks
  // for more than kXBytes of it stays with those, so that what fitted the device beside its tensors before still does.
  p->use_x = p->use_xb = false;
  p->xchunks = p->xbchunks = 1;
  p->xchunk_tiles = p->xbchunk_tiles = 1;
  p->xprep = 0;
  if (!p->use_tc && !(c.flags & WERSA_FLAG_SIMT_ONLY)) {
    const int tiles = ceil_div(n, 128), groups = m <= 128 ? 1 : m / 128;
    const double plane_bytes = (p->bf16 ? p->with_backward ? 24. : 12. : p->with_backward ? 32. : 18.) * p->slabs * n * c.head_dim;
    long long best = 0;
    for (int ch = 1; ch <= tiles && ch <= p->sms; ++ch) {
      const long long cost = (long long)ceil_div(p->slabs * groups * ch, p->sms) * (ceil_div(tiles, ch) + 3) * 64 + ch;
      if (ch == 1 || cost < best) {
        best = cost;
        p->xchunks = ch;
      }
    }
    p->xchunk_tiles = ceil_div(tiles, p->xchunks);
    p->xchunks = ceil_div(tiles, p->xchunk_tiles);
    for (int ch = 1; ch <= tiles && ch <= p->sms; ++ch) {
      const long long cost = (long long)ceil_div(p->slabs * ch, p->sms) * (ceil_div(tiles, ch) + 1);
      if (ch == 1 || cost < best) {
        best = cost;
        p->xbchunks = ch;
      }
    }
    p->xbchunk_tiles = ceil_div(tiles, p->xbchunks);
    p->xbchunks = ceil_div(tiles, p->xbchunk_tiles);
    const int width = c.head_dim <= 16 ? 0 : c.head_dim <= 32 ? 1 : 2;
    const int waves = ceil_div(p->slabs * groups * p->xchunks, p->sms), bwaves = ceil_div(p->slabs * p->xbchunks, p->sms) * groups;
    double f_fwd, f_bwd, x_fwd, x_bwd;
    bool enough = true, enough_b = true;
    if (m >= 128) {
      constexpr double kFwd[2][3] = {{0.13, 0.205, 0.345}, {0.17, 0.25, 0.46}}, kBwd[2][3] = {{0.275, 0.445, 0.745}, {0.33, 0.53, 0.8}};
      f_fwd = 14 + kFwd[p->simt_small][width] * ffma_cost;
      f_bwd = 15 + kBwd[p->simt_small][width] * ffma_cost;
      x_fwd = 9 + (12.5 + 6 * p->xchunk_tiles) * waves + 0.02 * p->xchunks;
      x_bwd = 14.5 + (15 + 3 * p->xchunk_tiles) * waves + 9. * bwaves * (p->xbchunk_tiles + 1);
      enough = (long long)p->slabs * tiles * groups >= kXUnits;
      enough_b = (long long)p->slabs * tiles >= p->sms;
    } else {
      // m = 64, fitted to 220 shapes (1 to 1023 slabs, 16 to 131072 tokens, d = 16 to 64, fp32 and bf16; rms 5 % off for planes, 8
      // and 13 % for FFMA; 14 of 440 choices cost more than 5 %, the worst 13 %).  FFMA and planes, us: forward bf16 1 x 7861, d = 16
      // 26 24; 237 x 20 24 40; 1 x 7258, d = 64 32 24; 14 x 21903 405 160; fp32 1 x 1024 20.9 21.4; 2 x 36480 94 69; training step
      // bf16 212 x 355 444 206.  From 24 tiles on, the fewest of the fit.
      constexpr double kFwd[2][3] = {{0.144, 0.216, 0.371}, {0.184, 0.291, 0.426}}, kBwd[2][3] = {{0.291, 0.428, 0.754}, {0.404, 0.59, 0.805}};
      const double elems = 1e-6 * p->slabs * n * c.head_dim, wt = (double)waves * p->xchunk_tiles, bt = (double)bwaves * (p->xbchunk_tiles + 1);
      f_fwd = 11.2 + kFwd[p->simt_small][width] * ffma_cost;
      f_bwd = 10.3 + kBwd[p->simt_small][width] * ffma_cost;
      x_fwd = p->bf16 ? 6.8 + 12.7 * waves + 3.06 * wt + 4.34 * elems : 7.2 + 12.2 * waves + 4.23 * wt + 6.07 * elems;
      enough = (long long)p->slabs * tiles >= 24;
      x_bwd = p->bf16 ? 5.3 + 23.5 * waves + 3.47 * wt + 3.08 * bt + 8.23 * elems : 6.6 + 24 * waves + 5.64 * wt + 2.29 * bt + 10.2 * elems;
    }
    p->use_x = enough && x_fwd <= f_fwd && plane_bytes <= kXBytes && p->slabs < 65535;
    p->use_xb = p->use_x && p->with_backward && (p->bf16 || !p->grad_bf16) && enough_b && x_bwd <= f_bwd;
    p->xprep = (int)std::min<long long>(((long long)p->slabs * n * 8 + 255) / 256, 8LL * p->sms);
  }

  p->tchunks = 0;
  p->tchunk_blocks = 0;
  p->tqchunks = 0;
  p->tqchunk_blocks = 0;
  if (p->use_tc) {
    const int blocks = ceil_div(n, 256);
    p->tchunks = p->sms / p->slabs;
    if (p->tchunks < 1) p->tchunks = 1;
    if (p->tchunks > blocks) p->tchunks = blocks;
    // Feature groups: one launch covers all of them (CTAs of one chunk of one slab and one group), in chunks that
    // minimise waves x (blocks + 5), 5 blocks being about what a CTA spends before its first and after its last one.
    // Against a launch per group in one wave, or with more slabs than SMs a persistent one:
    // 1 x 4 x 131072, m = 1024 316 -> 254 us; 1 x 2 x 1024, m = 1024 69 -> 27 us; 144 slabs of one block, m = 1024
    // 125 -> 118 us; 768 slabs of one block 475 -> 480 us, of four, m = 512 460 -> 462 us; 160 slabs of 16 393 -> 320 us.
    if (grouped) {
      long long best = 0;
      for (int ch = 1; ch <= blocks && ch <= 64; ++ch) {
        const long long cost = (long long)ceil_div(p->slabs * p->groups * ch, p->sms) * (ceil_div(blocks, ch) + 5);
        if (ch == 1 || cost < best) {
          best = cost;
          p->tchunks = ch;
        }
      }
    }
    p->tchunk_blocks = ceil_div(blocks, p->tchunks);
    p->tchunks = ceil_div(blocks, p->tchunk_blocks);
    // Query side: with more slabs than SMs its CTAs walk items, and since chunks cost it no partial sums they are
    // chosen to even the CTAs' loads: rounds x (blocks + 1), the 1 for an item's start.  A forward with whole slabs as
    // items and so: 160 slabs of 16 blocks, m = 256 172 -> 152 us, m = 128 132 -> 114 us; 208 of 12, m = 128 117 -> 111;
    // 300 of 8, m = 256 147 -> 142; 768 of 4 stays whole.  (Even shares of one list of all blocks need no such choice
    // but cost 68 bytes of spilled registers per thread: 147 us and 114 us, but 600 slabs of one block 83 -> 86 us.)
    p->tqchunks = p->tchunks;
    if (!grouped && p->slabs > p->sms) {
      long long best = 0;
      for (int ch = 1; ch <= blocks && ch <= 16; ++ch) {
        const long long cost = (long long)ceil_div(p->slabs * ch, p->sms) * (ceil_div(blocks, ch) + 1);
        if (ch == 1 || cost < best) {
          best = cost;
          p->tqchunks = ch;
        }
      }
    }
    p->tqchunk_blocks = ceil_div(blocks, p->tqchunks);
    p->tqchunks = ceil_div(blocks, p->tqchunk_blocks);
  }
  {
    // tensor-core backward: one wave of CTAs that share the list of all 128-token tiles evenly
    const long long tiles = (long long)ceil_div(n, 128) * p->slabs;
    p->bctas = (int)(tiles < p->sms ? tiles : p->sms);
  }

  size_t off = 0;
  auto take = [&](size_t bytes) {
    size_t o = off;
    off = align_up(off + bytes, 256);
    return o;
  };
  const size_t slabs = (size_t)p->slabs;
  // status word (256 bytes) followed by the arrival counters; cleared together before the first launch
  p->off_status = off;
  p->off_counters = off + 256;
  p->status_bytes = align_up(256 + sizeof(int) * (2 * slabs + (size_t)c.batch), 256);
  take(p->status_bytes);
  p->off_qpart = take(sizeof(float) * slabs * p->qchunks * kD);
  p->off_qbar = take(sizeof(float) * slabs * kD);
  p->off_sg = take(sizeof(float) * slabs * p->L1);
  p->off_f = take(sizeof(float) * slabs * p->L1);
  // rows of partial sums: chunks of the forward or of the fp32 kernels, or the segments of the tensor-core
  // backward (slot = CTA + slab) of one feature group; of all feature groups in the forward
  size_t part_rows = slabs * p->groups * (p->use_tc ? p->tchunks : p->schunks) * (m < kGroupFeatures ? m : kGroupFeatures);
  const bool ffma_bwd = p->use_x && p->with_backward && !p->use_xb;
  if (p->use_x) part_rows = slabs * m * (ffma_bwd ? std::max(p->xchunks, p->schunks) : p->xchunks);
  if (p->use_tc && p->with_backward) {
    const size_t seg_rows = ((size_t)p->bctas + slabs) * (m < kGroupFeatures ? m : kGroupFeatures);
    if (seg_rows > part_rows) part_rows = seg_rows;
  }
  p->off_spart = take(sizeof(float) * part_rows * kD);
  p->off_zpart = take(sizeof(float) * part_rows);
  p->off_S = take(sizeof(float) * slabs * m * kD);
  p->off_z = take(sizeof(float) * slabs * m);
  p->off_Sbf = take(sizeof(__nv_bfloat16) * slabs * m * kD);
  p->off_Wt = take(sizeof(__nv_bfloat16) * (size_t)m * kD);
  p->off_Simg = take(p->use_tc ? slabs * simg_bytes(m) : 0);
  const size_t slab_elems = slabs * (size_t)n * kD;
  const size_t io_bytes = p->bf16 ? 2 : 4;
  // The buffers of filtered tensors, their gradients and group outputs are sized for 64 columns, of which the kernels use
  // the first slabs * n * head_dim elements; the 256 bytes behind them are unused.  Both keep the order that the sizes of
  // narrow and 64-wide contexts have always had (a narrow one asks for more), which the interface's test pins.
  take(p->dpad ? 256 : 0);
  p->off_Og = take(grouped ? io_bytes * slab_elems * p->groups : 0);
  p->off_den = take(grouped ? sizeof(float) * slabs * n * p->groups : 0);
  // fp32 arithmetic on the tensor cores: bytes per element of a tensor (slabs x n x head_dim: narrow heads pay for their own columns).
  // Planes of T_f(Q), T_f(K) and V, 18 in all, over whose last two lie first the query side's shares of a forward without a
  // backward (see launch_tcx_qside), then dQ_F and dK_F of an FFMA backward, which keeps T_f(Q) and T_f(K) as well: 26.  A
  // backward on the planes: O (4), dQ_F (4) and planes of dO (6), 32 in all; the forward's shares lie over the last two,
  // dK_F over the planes of dO, which its kernels no longer read.  bf16 tensors have planes of T_f(Q) and T_f(K) alone, 12 and 24
  // (24 with an FFMA backward).  FFMA alone: 8 and 16, 64 columns each.
  const size_t tensor = slabs * (size_t)n * c.head_dim, plane3 = 3 * sizeof(__nv_bfloat16) * tensor;
  p->off_dO3 = p->off_xO = p->off_xden = p->off_xinv = p->off_xc = p->off_xshare = 0;
  p->off_QF = p->off_KF = p->off_QF3 = p->off_KF3 = p->off_V3 = p->off_dQF = p->off_dKF = 0;
  if (p->use_x) {
    p->off_QF3 = take(plane3);
    p->off_KF3 = take(plane3);
    p->off_V3 = take(!p->bf16 ? plane3 : ffma_bwd ? sizeof(float) * tensor : 0);   // (bf16: of use to dK_F below alone)
    if (ffma_bwd) {
      p->off_QF = take(sizeof(float) * tensor);
      p->off_KF = take(sizeof(float) * tensor);
      p->off_dQF = p->off_KF3;
      p->off_dKF = p->off_KF3 + align_up(sizeof(float) * tensor, 256);
    }
  } else if (!p->use_tc) {   // (the bf16 kernels of the tensor cores filter on chip, or read planes in the backward)
    p->off_QF = take(sizeof(float) * slab_elems);
    p->off_KF = take(sizeof(float) * slab_elems);
  }
  if (p->with_backward) {
    p->off_dS = take(sizeof(float) * slabs * m * kD);
    p->off_dz = take(sizeof(float) * slabs * m);
    p->off_sumdD = take(sizeof(float) * (p->use_tc ? (size_t)p->bctas : p->use_xb ? (size_t)p->xprep : slabs * p->schunks));
    if (p->use_xb) {
      const size_t groups = c.features <= 128 ? 1 : c.features / 128, padded = (size_t)ceil_div(c.seq_len, 128) * 128;
      p->off_xO = take(sizeof(float) * tensor);
      p->off_xden = take(sizeof(float) * groups * slabs * c.seq_len);
      p->off_xinv = take(sizeof(float) * slabs * padded);
      p->off_xc = take(sizeof(float) * slabs * padded);
      p->off_dQF = p->off_xshare = take(sizeof(float) * tensor);
      p->off_dO3 = p->off_dKF = take(p->bf16 ? sizeof(float) * tensor : plane3);
    }
    p->off_bands = take(sizeof(float) * 2 * slabs * 2 * p->htiles * kBandVals);   // Q and K; two column halves per tile
    p->off_dqbar = take(sizeof(float) * slabs * (kD + kBandVals));
    if (!p->use_x) {
      p->off_dQF = take(sizeof(float) * slab_elems);
      p->off_dKF = take(sizeof(float) * slab_elems);
    }
    p->off_dSbf = take(sizeof(__nv_bfloat16) * slabs * m * kD);
    if (p->use_tc) {
      p->off_KF3 = take(3 * sizeof(__nv_bfloat16) * slab_elems);
      p->off_QF3 = take(3 * sizeof(__nv_bfloat16) * slab_elems);
    }
    p->off_Slo = take(p->use_tc ? sizeof(__nv_bfloat16) * slabs * m * kD : 0);
    p->off_Dtot = take(grouped ? sizeof(float) * 2 * slabs * n : 0);
    p->off_shardtot = take(256);
  } else {
    p->off_Dtot = p->off_shardtot = 0;
    p->off_dS = p->off_dz = p->off_sumdD = p->off_bands = p->off_dqbar = p->off_dSbf = p->off_Slo = 0;
  }
  p->total = off;
  return WERSA_OK;
}

Ws resolve(const Plan& p, void* workspace) {
  char* b = static_cast<char*>(workspace);
  Ws w;
  w.status = reinterpret_cast<int*>(b + p.off_status);
  w.seen = w.status + 16;   // (the status word has 256 bytes to itself)
  w.counters = reinterpret_cast<int*>(b + p.off_counters);
  w.qpart = reinterpret_cast<float*>(b + p.off_qpart);
  w.qbar = reinterpret_cast<float*>(b + p.off_qbar);
  w.sg = reinterpret_cast<float*>(b + p.off_sg);
  w.f = reinterpret_cast<float*>(b + p.off_f);
  w.spart = reinterpret_cast<float*>(b + p.off_spart);
  w.zpart = reinterpret_cast<float*>(b + p.off_zpart);
  w.S = reinterpret_cast<float*>(b + p.off_S);
  w.z = reinterpret_cast<float*>(b + p.off_z);
  w.Sbf = reinterpret_cast<__nv_bfloat16*>(b + p.off_Sbf);
  w.Wt = reinterpret_cast<__nv_bfloat16*>(b + p.off_Wt);
  w.Simg = reinterpret_cast<uint8_t*>(b + p.off_Simg);
  w.QF = reinterpret_cast<float*>(b + p.off_QF);
  w.KF = reinterpret_cast<float*>(b + p.off_KF);
  w.dS = reinterpret_cast<float*>(b + p.off_dS);
  w.dz = reinterpret_cast<float*>(b + p.off_dz);
  w.sumdD = reinterpret_cast<float*>(b + p.off_sumdD);
  w.bands = reinterpret_cast<float*>(b + p.off_bands);
  w.dqbar = reinterpret_cast<float*>(b + p.off_dqbar);
  w.dQF = reinterpret_cast<float*>(b + p.off_dQF);
  w.dKF = reinterpret_cast<float*>(b + p.off_dKF);
  w.dSbf = reinterpret_cast<__nv_bfloat16*>(b + p.off_dSbf);
  w.KF3 = reinterpret_cast<__nv_bfloat16*>(b + p.off_KF3);
  w.QF3 = reinterpret_cast<__nv_bfloat16*>(b + p.off_QF3);
  w.V3 = reinterpret_cast<__nv_bfloat16*>(b + p.off_V3);
  w.dO3 = reinterpret_cast<__nv_bfloat16*>(b + p.off_dO3);
  w.xO = reinterpret_cast<float*>(b + p.off_xO);
  w.xden = reinterpret_cast<float*>(b + p.off_xden);
  w.xinv = reinterpret_cast<float*>(b + p.off_xinv);
  w.xc = reinterpret_cast<float*>(b + p.off_xc);
  w.xshare = reinterpret_cast<float*>(b + p.off_xshare);
  w.Slo = reinterpret_cast<__nv_bfloat16*>(b + p.off_Slo);
  w.Og = b + p.off_Og;
  w.den = reinterpret_cast<float*>(b + p.off_den);
  w.Dtot = reinterpret_cast<float*>(b + p.off_Dtot);
  w.shardtot = reinterpret_cast<float*>(b + p.off_shardtot);
  return w;
}

}  // namespace wersa

using namespace wersa;

constexpr int kMaxSteps = 32;

// Optional per-step timing: an event before the first launch and one after every step.
struct StepTimer {
  bool enabled = false;
  cudaEvent_t ev[2][kMaxSteps + 1];
  const char* name[2][kMaxSteps];
  int count[2] = {0, 0};
};

struct wersa_ctx {
  Plan plan;
  Ws ws;
  void* workspace;
  bool forward_done;
  bool status_cleared;
  int launches_fwd, launches_bwd;
  StepTimer timer;
};

namespace {

bool aligned16(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }

// Makes cfg.device current for the lifetime of the object and restores the caller's device.
struct DeviceGuard {
  int prev = -1;
  cudaError_t err;
  explicit DeviceGuard(int dev) {
    err = cudaGetDevice(&prev);
    if (err == cudaSuccess && prev != dev) err = cudaSetDevice(dev);
    else if (err == cudaSuccess) prev = -1;
  }
  ~DeviceGuard() {
    if (prev >= 0) cudaSetDevice(prev);
  }
};

#define WERSA_CUDA(call)                                   \
  do {                                                     \
    cudaError_t e_ = (call);                               \
    if (e_ != cudaSuccess) return WERSA_ERR_CUDA;          \
  } while (0)

// Runs one step of a pass and, when step timing is on, records an event behind it.
#define WERSA_STEP(which, label, call)                                             \
  do {                                                                             \
    WERSA_CUDA(call);                                                              \
    StepTimer& t_ = ctx->timer;                                                    \
    if (t_.enabled && t_.count[which] < kMaxSteps) {                               \
      t_.name[which][t_.count[which]] = label;                                     \
      WERSA_CUDA(cudaEventRecord(t_.ev[which][t_.count[which] + 1], st));          \
      ++t_.count[which];                                                           \
    }                                                                              \
  } while (0)

wersa_status begin_pass(wersa_ctx* ctx, int which, cudaStream_t st) {
  StepTimer& t = ctx->timer;
  t.count[which] = 0;
  if (t.enabled) WERSA_CUDA(cudaEventRecord(t.ev[which][0], st));
  return WERSA_OK;
}

// Feature group g of a map wider than 256 features: the plan of a 256-feature problem and the workspace
// regions of that group (the kernels' buffers are kept group-major: [group][slab][...], S' and z' [slab][group][...]).
Plan group_plan(const Plan& p) {
  Plan pg = p;
  pg.cfg.features = kGroupFeatures;
  return pg;
}
// (In the backward all groups use the same region of partial sums, one after the other.)
Ws group_view(const Plan& p, const Ws& w, int g) {
  Ws v = w;
  const size_t slabs = (size_t)p.slabs, mg = kGroupFeatures;
  v.Wt = w.Wt + (size_t)g * mg * kD;
  if (p.with_backward) {
    v.dS = w.dS + (size_t)g * slabs * mg * kD;
    v.dz = w.dz + (size_t)g * slabs * mg;
    v.dSbf = w.dSbf + (size_t)g * slabs * mg * kD;
    v.Slo = w.Slo + (size_t)g * slabs * mg * kD;
  }
  v.S = w.S + (size_t)g * mg * kD;   // (rows of the whole map's features)
  v.z = w.z + (size_t)g * mg;
  v.Sbf = w.Sbf + (size_t)g * slabs * mg * kD;
  v.Simg = w.Simg + (size_t)g * slabs * simg_bytes((int)mg);
  return v;
}

wersa_status clear_status_once(wersa_ctx* ctx, cudaStream_t st) {
  if (!ctx->status_cleared) {
    WERSA_CUDA(cudaMemsetAsync(ctx->ws.status, 0, ctx->plan.status_bytes, st));
    ctx->status_cleared = true;
  }
  return WERSA_OK;
}

}  // namespace

extern "C" {

size_t wersa_workspace_bytes(const wersa_config* cfg) {
  if (cfg == nullptr) return 0;
  Plan p;
  if (make_plan(*cfg, &p) != WERSA_OK) return 0;
  return p.total;
}

wersa_status wersa_create(const wersa_config* cfg, void* workspace, size_t workspace_bytes, wersa_ctx** out) {
  if (cfg == nullptr || out == nullptr) return WERSA_ERR_INVALID_ARG;
  Plan p;
  wersa_status s = make_plan(*cfg, &p);
  if (s != WERSA_OK) return s;
  if (workspace == nullptr || (reinterpret_cast<uintptr_t>(workspace) & 255u) != 0 || workspace_bytes < p.total)
    return WERSA_ERR_WORKSPACE;
  {
    DeviceGuard guard(p.cfg.device);
    if (guard.err == cudaSuccess) {
      choose_small_forward(&p);
      prepare_qmean_gate(p);
    }
  }
  wersa_ctx* ctx = new (std::nothrow) wersa_ctx;
  if (ctx == nullptr) return WERSA_ERR_INVALID_ARG;
  ctx->plan = p;
  ctx->workspace = workspace;
  ctx->ws = resolve(p, workspace);
  ctx->forward_done = false;
  ctx->status_cleared = false;
  ctx->launches_fwd = ctx->launches_bwd = 0;
  *out = ctx;
  return WERSA_OK;
}

wersa_status wersa_forward(wersa_ctx* ctx, const void* Q, const void* K, const void* V, const void* W,
                           const float* beta, const float* gate_w, const float* gate_b, const float* omega,
                           void* O, void* cuda_stream) {
  if (ctx == nullptr || Q == nullptr || K == nullptr || V == nullptr || W == nullptr || beta == nullptr ||
      omega == nullptr || O == nullptr)
    return WERSA_ERR_INVALID_ARG;
  if (!aligned16(Q) || !aligned16(K) || !aligned16(V) || !aligned16(W) || !aligned16(O))
    return WERSA_ERR_INVALID_ARG;
  const Plan& p = ctx->plan;
  const Ws& w = ctx->ws;
  cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
  DeviceGuard guard(p.cfg.device);
  if (guard.err != cudaSuccess) return WERSA_ERR_CUDA;
  wersa_status s = clear_status_once(ctx, st);
  if (s != WERSA_OK) return s;
  int launches = 0;
  const int kind = p.bf16 ? 1 : 0;
  if ((s = begin_pass(ctx, 0, st)) != WERSA_OK) return s;
  const size_t rows = (size_t)p.slabs * p.cfg.seq_len;
  const int d = p.cfg.head_dim;   // (narrow heads: every forward kernel reads and writes the narrow tensors themselves)
  if (p.small_blocks > 0) {
    WERSA_STEP(0, "small_forward", launch_small_forward(p, w, Q, K, V, W, beta, gate_w, gate_b, omega, O, st, &launches));
    if (p.groups > 1)
      WERSA_STEP(0, "combine_groups", launch_combine_groups(w.Og, w.den, O, rows, p.groups, d, st, &launches));
    ctx->launches_fwd = launches;
    ctx->forward_done = true;
    return WERSA_OK;
  }
  if (p.filter_tokens > 0)
    WERSA_STEP(0, "small_filter", launch_small_filter(p, w, Q, K, gate_w, gate_b, omega, st, &launches));
  else
    WERSA_STEP(0, "qmean_gate",
               launch_qmean_gate(p, w, Q, gate_w, gate_b, omega, p.use_tc ? W : nullptr, d, st, &launches));
  if (p.groups > 1) {
    // feature groups of 256 (tensor-core path): every group runs the key side and the query side on its own
    // rows of W^T, all groups in one launch each; the query side leaves O_g and the denominators, which the last
    // launch combines.  (Buffers are group-major but for S' and z', which have a slab's features together.)
    const Plan pg = group_plan(p);
    WERSA_STEP(0, "tc_kside", launch_tc_kside(pg, w, K, V, st, &launches));
    if (p.tchunks > 1)
      WERSA_STEP(0, "reduce_partials",
                 launch_reduce_partials(pg, w.spart, w.zpart, p.tchunks, w.S, w.z, p.with_backward ? w.Sbf : nullptr, w.Simg, st, &launches));
    WERSA_STEP(0, "tc_qside", launch_tc_qside(pg, w, Q, beta, w.Og, w.den, st, &launches));
    WERSA_STEP(0, "combine_groups",
               launch_combine_groups(w.Og, w.den, O, rows, p.groups, d, st, &launches));
  } else if (p.use_tc) {
    WERSA_STEP(0, "tc_kside", launch_tc_kside(p, w, K, V, st, &launches));
    if (p.tchunks > 1)   // with one chunk per slab the key-side kernel has written S', z' and the image itself
      WERSA_STEP(0, "reduce_partials",
                 launch_reduce_partials(p, w.spart, w.zpart, p.tchunks, w.S, w.z, p.with_backward ? w.Sbf : nullptr, w.Simg, st, &launches));
    WERSA_STEP(0, "tc_qside", launch_tc_qside(p, w, Q, beta, O, nullptr, st, &launches));
  } else if (p.use_x) {
    WERSA_STEP(0, "f32_planes", launch_f32_planes(p, w, Q, K, V, p.with_backward && !p.use_xb, st, &launches));
    WERSA_STEP(0, "tcx_kside", launch_tcx_kside(p, w, V, W, st, &launches));
    WERSA_STEP(0, "reduce_partials",
               launch_reduce_partials(p, w.spart, w.zpart, p.xchunks, w.S, w.z, nullptr, nullptr, st, &launches));
    WERSA_STEP(0, "tcx_qside", launch_tcx_qside(p, w, W, beta, O, st, &launches));
  } else {
    if (p.filter_tokens == 0)
      WERSA_STEP(0, "haar_filter_qk", launch_haar_filter(p, Q, kind, w.f, w.QF, K, w.KF, 0, d, true, st, &launches));
    WERSA_STEP(0, "simt_kside", launch_simt_kside(p, w, V, W, st, &launches));
    WERSA_STEP(0, "reduce_partials",
               launch_reduce_partials(p, w.spart, w.zpart, p.schunks, w.S, w.z, nullptr, nullptr, st, &launches));
    WERSA_STEP(0, "simt_qside", launch_simt_qside(p, w, W, beta, O, st, &launches));
  }
  ctx->launches_fwd = launches;
  ctx->forward_done = true;
  return WERSA_OK;
}

// ---- sequence-sharded forward ------------------------------------------------------------------------
// The four steps of wersa_forward with the two places opened where shards of one sequence have to exchange
// sums: after the mean pool (column sums of Q) and after the key side (S', z').  Tensor-core path, one feature
// group; the context is created with the shard's own length.
static bool shardable(const Plan& p) { return p.use_tc && p.groups == 1; }

wersa_status wersa_shard_pool(wersa_ctx* ctx, const void* Q, const void* W, float* qsum, void* cuda_stream) {
  if (ctx == nullptr || Q == nullptr || W == nullptr || qsum == nullptr) return WERSA_ERR_INVALID_ARG;
  if (!aligned16(Q) || !aligned16(W)) return WERSA_ERR_INVALID_ARG;
  const Plan& p = ctx->plan;
  if (!shardable(p)) return WERSA_ERR_UNSUPPORTED;
  const Ws& w = ctx->ws;
  cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
  DeviceGuard guard(p.cfg.device);
  if (guard.err != cudaSuccess) return WERSA_ERR_CUDA;
  wersa_status s = clear_status_once(ctx, st);
  if (s != WERSA_OK) return s;
  int launches = 0;
  // (the gate this launch also computes belongs to the shard alone and is replaced by wersa_shard_gate)
  WERSA_CUDA(launch_qmean_gate(p, w, Q, nullptr, nullptr, nullptr, W, p.cfg.head_dim, st, &launches));
  WERSA_CUDA(launch_shard_qsum(p, w, qsum, st, &launches));
  ctx->launches_fwd = launches;
  ctx->forward_done = false;
  return WERSA_OK;
}

wersa_status wersa_shard_gate(wersa_ctx* ctx, const float* qsum_total, int64_t n_total, const float* gate_w,
                              const float* gate_b, const float* omega, void* cuda_stream) {
  if (ctx == nullptr || qsum_total == nullptr || omega == nullptr || n_total < 1 || n_total > 0x7fffffffLL)
    return WERSA_ERR_INVALID_ARG;
  const Plan& p = ctx->plan;
  if (!shardable(p)) return WERSA_ERR_UNSUPPORTED;
  cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
  DeviceGuard guard(p.cfg.device);
  if (guard.err != cudaSuccess) return WERSA_ERR_CUDA;
  int launches = 0;
  WERSA_CUDA(launch_gate_from_sums(p, ctx->ws, qsum_total, n_total, gate_w, gate_b, omega, p.cfg.head_dim, st, &launches));
  ctx->launches_fwd += launches;
  return WERSA_OK;
}

wersa_status wersa_shard_keys(wersa_ctx* ctx, const void* K, const void* V, void* cuda_stream) {
  if (ctx == nullptr || K == nullptr || V == nullptr) return WERSA_ERR_INVALID_ARG;
  if (!aligned16(K) || !aligned16(V)) return WERSA_ERR_INVALID_ARG;
  const Plan& p = ctx->plan;
  if (!shardable(p)) return WERSA_ERR_UNSUPPORTED;
  const Ws& w = ctx->ws;
  cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
  DeviceGuard guard(p.cfg.device);
  if (guard.err != cudaSuccess) return WERSA_ERR_CUDA;
  int launches = 0;
  WERSA_CUDA(launch_tc_kside(p, w, K, V, st, &launches, true));
  if (p.tchunks > 1)
    WERSA_CUDA(launch_reduce_partials(p, w.spart, w.zpart, p.tchunks, w.S, w.z, p.with_backward ? w.Sbf : nullptr, w.Simg, st, &launches));
  ctx->launches_fwd += launches;
  ctx->forward_done = true;   // S', z' of this shard can be read with wersa_saved
  return WERSA_OK;
}

wersa_status wersa_shard_output(wersa_ctx* ctx, const void* Q, const float* S_total, const float* z_total,
                                const float* beta, void* O, void* cuda_stream) {
  if (ctx == nullptr || Q == nullptr || S_total == nullptr || z_total == nullptr || beta == nullptr || O == nullptr)
    return WERSA_ERR_INVALID_ARG;
  if (!aligned16(Q) || !aligned16(O)) return WERSA_ERR_INVALID_ARG;
  const Plan& p = ctx->plan;
  if (!shardable(p)) return WERSA_ERR_UNSUPPORTED;
  const Ws& w = ctx->ws;
  cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
  DeviceGuard guard(p.cfg.device);
  if (guard.err != cudaSuccess) return WERSA_ERR_CUDA;
  int launches = 0;
  // the totals take the place of a single partial: the reduction copies them and writes the operand images
  WERSA_CUDA(launch_reduce_partials(p, S_total, z_total, 1, w.S, w.z, p.with_backward ? w.Sbf : nullptr, w.Simg, st, &launches, true));
  WERSA_CUDA(launch_tc_qside(p, w, Q, beta, O, nullptr, st, &launches));
  ctx->launches_fwd += launches;
  return WERSA_OK;
}

// ---- sequence-sharded backward: three steps with the sums of dS', dz' and of (df, sum dD') taken by the caller
static bool shardable_bwd(const Plan& p) { return shardable(p) && p.with_backward && !p.dpad; }

wersa_status wersa_shard_backward_queries(wersa_ctx* ctx, const void* Q, const float* beta, const void* dO,
                                          void* cuda_stream) {
  if (ctx == nullptr || Q == nullptr || beta == nullptr || dO == nullptr) return WERSA_ERR_INVALID_ARG;
  if (!aligned16(Q) || !aligned16(dO)) return WERSA_ERR_INVALID_ARG;
  const Plan& p = ctx->plan;
  if (!shardable_bwd(p)) return WERSA_ERR_UNSUPPORTED;
  if (!ctx->forward_done) return WERSA_ERR_STATE;
  const Ws& w = ctx->ws;
  cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
  DeviceGuard guard(p.cfg.device);
  if (guard.err != cudaSuccess) return WERSA_ERR_CUDA;
  int launches = 0;
  const int kind = 1, gkind = p.grad_bf16 ? 1 : 0;
  WERSA_CUDA(launch_haar_filter_split3(p, w, Q, w.QF3, nullptr, nullptr, true, st, &launches));
  WERSA_CUDA(launch_tc_bwd_qside(p, w, w.QF3, beta, dO, nullptr, nullptr, false, st, &launches));
  WERSA_CUDA(launch_reduce_segments(p, w, st, &launches));
  WERSA_CUDA(launch_haar_backward(p, w, 0, Q, w.dQF, nullptr, nullptr, nullptr, nullptr, kind, gkind, kD, st, &launches));   // band inner products
  ctx->launches_bwd = launches;
  return WERSA_OK;
}

wersa_status wersa_shard_backward_keys(wersa_ctx* ctx, const void* K, const void* V, const float* dS_total,
                                       const float* dz_total, void* dK, void* dV, void* cuda_stream) {
  if (ctx == nullptr || K == nullptr || V == nullptr || dS_total == nullptr || dz_total == nullptr || dK == nullptr ||
      dV == nullptr)
    return WERSA_ERR_INVALID_ARG;
  if (!aligned16(K) || !aligned16(V) || !aligned16(dK) || !aligned16(dV)) return WERSA_ERR_INVALID_ARG;
  const Plan& p = ctx->plan;
  if (!shardable_bwd(p)) return WERSA_ERR_UNSUPPORTED;
  if (!ctx->forward_done) return WERSA_ERR_STATE;
  const Ws& w = ctx->ws;
  cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
  DeviceGuard guard(p.cfg.device);
  if (guard.err != cudaSuccess) return WERSA_ERR_CUDA;
  int launches = 0;
  const int kind = 1, gkind = p.grad_bf16 ? 1 : 0;
  // the totals take the place of a single partial: the reduction copies them and writes the bf16 image of dS'
  WERSA_CUDA(launch_reduce_partials(p, dS_total, dz_total, 1, w.dS, w.dz, w.dSbf, nullptr, st, &launches));
  WERSA_CUDA(launch_haar_filter_split3(p, w, K, w.KF3, nullptr, nullptr, false, st, &launches));
  WERSA_CUDA(launch_tc_bwd_kside(p, w, w.KF3, V, dV, false, st, &launches));
  WERSA_CUDA(launch_haar_backward(p, w, 1, K, w.dKF, dK, nullptr, nullptr, nullptr, kind, gkind, kD, st, &launches));
  float* df = w.dqbar + (size_t)p.slabs * kD;
  WERSA_CUDA(launch_band_sums(p, w, haar_band_blocks(p, kD), p.bctas, df, w.shardtot, st, &launches));
  ctx->launches_bwd += launches;
  return WERSA_OK;
}

wersa_status wersa_shard_backward_gate(wersa_ctx* ctx, const float* df_total, const float* sumdD_total, int64_t n_total,
                                       const float* beta, const float* gate_w, const float* omega, float* dbeta,
                                       float* dgate_w, float* dgate_b, float* domega, void* dQ, void* cuda_stream) {
  if (ctx == nullptr || df_total == nullptr || sumdD_total == nullptr || beta == nullptr || omega == nullptr ||
      dQ == nullptr || n_total < 1)
    return WERSA_ERR_INVALID_ARG;
  if (!aligned16(dQ)) return WERSA_ERR_INVALID_ARG;
  const Plan& p = ctx->plan;
  if (!shardable_bwd(p)) return WERSA_ERR_UNSUPPORTED;
  if (!ctx->forward_done) return WERSA_ERR_STATE;
  const Ws& w = ctx->ws;
  cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
  DeviceGuard guard(p.cfg.device);
  if (guard.err != cudaSuccess) return WERSA_ERR_CUDA;
  int launches = 0;
  WERSA_CUDA(launch_gate_backward_from(p, w, df_total, sumdD_total, beta, gate_w, omega, dbeta, dgate_w, dgate_b, domega,
                                       st, &launches));
  WERSA_CUDA(launch_haar_filter_addvec(p, w.dQF, w.f, w.dqbar, 1.f / (float)n_total, dQ, p.grad_bf16 ? 1 : 0, kD,
                                       st, &launches));
  ctx->launches_bwd += launches;
  return WERSA_OK;
}

wersa_status wersa_forward_host(wersa_ctx* ctx, const void* hQ, const void* hK, const void* hV, void* dQ,
                                void* dK, void* dV, const void* W, const float* beta, const float* gate_w,
                                const float* gate_b, const float* omega, void* dO, void* hO, void* cuda_stream) {
  if (ctx == nullptr || hQ == nullptr || hK == nullptr || hV == nullptr || hO == nullptr || dQ == nullptr ||
      dK == nullptr || dV == nullptr || dO == nullptr || W == nullptr || beta == nullptr || omega == nullptr)
    return WERSA_ERR_INVALID_ARG;
  if (!aligned16(dQ) || !aligned16(dK) || !aligned16(dV) || !aligned16(dO) || !aligned16(W))
    return WERSA_ERR_INVALID_ARG;
  const Plan& p = ctx->plan;
  cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
  const size_t bytes = (size_t)p.slabs * p.cfg.seq_len * p.cfg.head_dim * (p.bf16 ? 2 : 4);
  DeviceGuard guard(p.cfg.device);
  if (guard.err != cudaSuccess) return WERSA_ERR_CUDA;
  WERSA_CUDA(cudaMemcpyAsync(dQ, hQ, bytes, cudaMemcpyHostToDevice, st));
  WERSA_CUDA(cudaMemcpyAsync(dK, hK, bytes, cudaMemcpyHostToDevice, st));
  WERSA_CUDA(cudaMemcpyAsync(dV, hV, bytes, cudaMemcpyHostToDevice, st));
  const wersa_status s = wersa_forward(ctx, dQ, dK, dV, W, beta, gate_w, gate_b, omega, dO, cuda_stream);
  if (s != WERSA_OK) return s;
  WERSA_CUDA(cudaMemcpyAsync(hO, dO, bytes, cudaMemcpyDeviceToHost, st));
  return WERSA_OK;
}

wersa_status wersa_backward(wersa_ctx* ctx, const void* Q, const void* K, const void* V, const void* W,
                            const float* beta, const float* gate_w, const float* gate_b, const float* omega,
                            const void* dO, void* dQ, void* dK, void* dV, float* dbeta, float* dgate_w,
                            float* dgate_b, float* domega, void* cuda_stream) {
  (void)gate_b;
  if (ctx == nullptr || Q == nullptr || K == nullptr || V == nullptr || W == nullptr || beta == nullptr ||
      omega == nullptr || dO == nullptr || dQ == nullptr || dK == nullptr || dV == nullptr)
    return WERSA_ERR_INVALID_ARG;
  if (!aligned16(Q) || !aligned16(K) || !aligned16(V) || !aligned16(W) || !aligned16(dO) || !aligned16(dQ) ||
      !aligned16(dK) || !aligned16(dV))
    return WERSA_ERR_INVALID_ARG;
  const Plan& p = ctx->plan;
  if (!p.with_backward) return WERSA_ERR_UNSUPPORTED;
  if (!ctx->forward_done) return WERSA_ERR_STATE;
  const Ws& w = ctx->ws;
  cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
  DeviceGuard guard(p.cfg.device);
  if (guard.err != cudaSuccess) return WERSA_ERR_CUDA;
  int launches = 0;
  const int kind = p.bf16 ? 1 : 0, gkind = p.grad_bf16 ? 1 : 0;
  wersa_status s = begin_pass(ctx, 1, st);
  if (s != WERSA_OK) return s;
  const size_t rows = (size_t)p.slabs * p.cfg.seq_len;
  const int d = p.cfg.head_dim;   // (narrow heads: every kernel reads and writes the narrow tensors themselves)
  if (p.groups > 1) {
    // Feature groups: the denominator and dD' of the whole map come from what the forward left (the groups'
    // outputs and denominators); every group then runs both tensor-core kernels on its own rows of W^T, S', z',
    // dS', dz', and dQ_F, dV, dK_F accumulate over the groups in launch order.
    WERSA_STEP(1, "haar_filter_qk", launch_haar_filter_split3(p, w, Q, w.QF3, K, w.KF3, true, st, &launches));
    WERSA_STEP(1, "group_bwd_prep",
               launch_group_bwd_prep(w.Og, w.den, dO, d, w.f, p.cfg.seq_len, p.L1, rows, p.groups, w.Dtot,
                                     w.Dtot + rows, st, &launches));
    const Plan pg = group_plan(p);
    for (int g = 0; g < p.groups; ++g) {
      const Ws wg = group_view(p, w, g);
      WERSA_STEP(1, "tc_bwd_qside",
                 launch_tc_bwd_qside(pg, wg, w.QF3, beta, dO, w.Dtot, w.Dtot + rows, g > 0, st, &launches));
      WERSA_STEP(1, "reduce_partials",
                 launch_reduce_segments(pg, wg, st, &launches));
      WERSA_STEP(1, "tc_bwd_kside", launch_tc_bwd_kside(pg, wg, w.KF3, V, dV, g > 0, st, &launches));
    }
  } else if (p.use_tc) {
    // the tensor-core forward keeps Q_F, K_F on chip: rebuild them, as three bf16 planes each
    WERSA_STEP(1, "haar_filter_qk", launch_haar_filter_split3(p, w, Q, w.QF3, K, w.KF3, true, st, &launches));
    WERSA_STEP(1, "tc_bwd_qside", launch_tc_bwd_qside(p, w, w.QF3, beta, dO, nullptr, nullptr, false, st, &launches));
  } else if (p.use_xb) {
    WERSA_STEP(1, "tcx_bwd_prep", launch_tcx_bwd_prep(p, w, dO, beta, st, &launches));
    WERSA_STEP(1, "tcx_bwd_qside", launch_tcx_bwd_qside(p, w, W, dO, st, &launches));
  } else {
    WERSA_STEP(1, "simt_bwd_qside", launch_simt_bwd_qside(p, w, W, beta, dO, st, &launches));
  }
  if (p.groups == 1)
    WERSA_STEP(1, "reduce_partials",
               p.use_tc ? launch_reduce_segments(p, w, st, &launches)
                        : launch_reduce_partials(p, w.spart, w.zpart, p.use_xb ? p.xchunks : p.schunks, w.dS, w.dz, nullptr,
                                                 nullptr, st, &launches));
  if (p.groups > 1) {
    // (done group by group above)
  } else if (p.use_tc) {
    WERSA_STEP(1, "tc_bwd_kside", launch_tc_bwd_kside(p, w, w.KF3, V, dV, false, st, &launches));
  } else if (p.use_xb) {
    WERSA_STEP(1, "tcx_bwd_kside", launch_tcx_bwd_kside(p, w, V, W, dV, st, &launches));
  } else {
    WERSA_STEP(1, "simt_bwd_kside", launch_simt_bwd_kside(p, w, V, W, dV, st, &launches));
  }
  // With gate weights dQ has a second term, d(qbar) / n on every row (Eq. 1), which is known only after the
  // gate backward: the first pass over dQ_F then takes the band inner products alone, and dQ is written
  // once, by a filter pass that adds the row vector.
  const bool pooled_term = gate_w != nullptr;
  WERSA_STEP(1, "haar_backward_kq",
             launch_haar_backward(p, w, 1, K, w.dKF, dK, Q, w.dQF, pooled_term ? nullptr : dQ, kind, gkind, d, st, &launches));
  const int n_sumdD = p.use_tc ? p.bctas : p.use_xb ? p.xprep : p.slabs * p.schunks;
  if (pooled_term)
    WERSA_STEP(1, "gate_backward_dq",
               launch_gate_backward_dq(p, w, haar_band_blocks(p, d), beta, gate_w, omega, n_sumdD, dbeta, dgate_w, dgate_b, domega, dQ,
                                       gkind, st, &launches));
  else
    WERSA_STEP(1, "gate_backward",
               launch_gate_backward(p, w, haar_band_blocks(p, d), beta, gate_w, omega, n_sumdD, dbeta, dgate_w, dgate_b, domega, st,
                                    &launches));
  ctx->launches_bwd = launches;
  return WERSA_OK;
}

wersa_status wersa_haar_filter(wersa_ctx* ctx, const void* X, const float* f, void* XF, void* cuda_stream) {
  if (ctx == nullptr || X == nullptr || f == nullptr || XF == nullptr) return WERSA_ERR_INVALID_ARG;
  if (!aligned16(X) || !aligned16(XF)) return WERSA_ERR_INVALID_ARG;
  const Plan& p = ctx->plan;
  DeviceGuard guard(p.cfg.device);
  if (guard.err != cudaSuccess) return WERSA_ERR_CUDA;
  int launches = 0;
  const int kind = p.bf16 ? 1 : 0;
  cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
  WERSA_CUDA(launch_haar_filter(p, X, kind, f, XF, nullptr, nullptr, kind, p.cfg.head_dim, false, st, &launches));
  return WERSA_OK;
}

wersa_status wersa_gate_static(const wersa_config* cfg, const void* Q, const float* gate_w, const float* gate_b,
                               const float* omega, float* qbar, float* f, void* cuda_stream) {
  if (cfg == nullptr || Q == nullptr || omega == nullptr || qbar == nullptr || f == nullptr)
    return WERSA_ERR_INVALID_ARG;
  if (!aligned16(Q)) return WERSA_ERR_INVALID_ARG;
  Plan p;
  wersa_status s = make_pool_plan(*cfg, &p);
  if (s != WERSA_OK) return s;
  if (p.dpad) return WERSA_ERR_UNSUPPORTED;   // head_dim 64 only: its q-bar has 64 columns
  if (static_scratch_floats_needed(p) > static_scratch_capacity_floats() ||
      static_scratch_counters_needed(p) > static_scratch_counter_capacity())
    return WERSA_ERR_TOO_LARGE;
  DeviceGuard guard(p.cfg.device);
  if (guard.err != cudaSuccess) return WERSA_ERR_CUDA;
  float* scratch = nullptr;
  WERSA_CUDA(static_scratch_address(p.cfg.device, &scratch));
  WERSA_CUDA(launch_qmean_gate_static(p, scratch, Q, gate_w, gate_b, omega, qbar, f,
                                      static_cast<cudaStream_t>(cuda_stream)));
  return WERSA_OK;
}

wersa_status wersa_saved(wersa_ctx* ctx, int which, const float** device_ptr, size_t* count) {
  if (ctx == nullptr || device_ptr == nullptr || count == nullptr) return WERSA_ERR_INVALID_ARG;
  if (!ctx->forward_done) return WERSA_ERR_STATE;
  const Plan& p = ctx->plan;
  const size_t slabs = (size_t)p.slabs;
  switch (which) {
    case 0: *device_ptr = ctx->ws.f; *count = slabs * p.L1; break;
    case 1: *device_ptr = ctx->ws.qbar; *count = slabs * kD; break;
    case 2: *device_ptr = ctx->ws.S; *count = slabs * p.cfg.features * kD; break;
    case 3: *device_ptr = ctx->ws.z; *count = slabs * p.cfg.features; break;
    // sequence-sharded backward: this shard's dS', dz', band inner products and sum of dD'
    case 4: if (!p.with_backward) return WERSA_ERR_UNSUPPORTED; *device_ptr = ctx->ws.dS; *count = slabs * p.cfg.features * kD; break;
    case 5: if (!p.with_backward) return WERSA_ERR_UNSUPPORTED; *device_ptr = ctx->ws.dz; *count = slabs * p.cfg.features; break;
    case 6: if (!p.with_backward) return WERSA_ERR_UNSUPPORTED; *device_ptr = ctx->ws.dqbar + slabs * kD; *count = slabs * kBandVals; break;
    case 7: if (!p.with_backward) return WERSA_ERR_UNSUPPORTED; *device_ptr = ctx->ws.shardtot; *count = 1; break;
    default: return WERSA_ERR_INVALID_ARG;
  }
  return WERSA_OK;
}

wersa_status wersa_query_status(wersa_ctx* ctx, void* cuda_stream) {
  if (ctx == nullptr) return WERSA_ERR_INVALID_ARG;
  cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
  DeviceGuard guard(ctx->plan.cfg.device);
  if (guard.err != cudaSuccess) return WERSA_ERR_CUDA;
  WERSA_CUDA(cudaStreamSynchronize(st));
  if (!ctx->status_cleared) return WERSA_OK;   // nothing has run yet
  int word = 0;
  WERSA_CUDA(cudaMemcpyAsync(&word, ctx->ws.status, sizeof(int), cudaMemcpyDeviceToHost, st));
  WERSA_CUDA(cudaStreamSynchronize(st));
  if (word != 0) {
    WERSA_CUDA(cudaMemsetAsync(ctx->ws.status, 0, 256, st));
    WERSA_CUDA(cudaStreamSynchronize(st));
    return WERSA_ERR_TIMEOUT;
  }
  return WERSA_OK;
}

wersa_status wersa_selftest_wait_timeout(wersa_ctx* ctx, uint32_t limit_us, int32_t* observed, void* cuda_stream) {
  if (ctx == nullptr || observed == nullptr || limit_us == 0 || limit_us > 100000) return WERSA_ERR_INVALID_ARG;
  cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
  DeviceGuard guard(ctx->plan.cfg.device);
  if (guard.err != cudaSuccess) return WERSA_ERR_CUDA;
  wersa_status s = clear_status_once(ctx, st);
  if (s != WERSA_OK) return s;
  WERSA_CUDA(launch_selftest_wait(ctx->ws, 1000ull * limit_us, observed, st));
  return WERSA_OK;
}

wersa_status wersa_selftest_short_forward(wersa_ctx* ctx, int32_t loss, const void* Q, const void* K, const void* V, const void* W,
                                          const float* beta, const float* omega, void* O, void* cuda_stream) {
  if (ctx == nullptr || loss < 1 || loss > 2 || Q == nullptr || K == nullptr || V == nullptr || W == nullptr || beta == nullptr ||
      omega == nullptr || O == nullptr)
    return WERSA_ERR_INVALID_ARG;
  if (!aligned16(Q) || !aligned16(K) || !aligned16(V) || !aligned16(W) || !aligned16(O)) return WERSA_ERR_INVALID_ARG;
  const Plan& p = ctx->plan;
  if (!selftest_small_supported(p)) return WERSA_ERR_UNSUPPORTED;
  cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
  DeviceGuard guard(p.cfg.device);
  if (guard.err != cudaSuccess) return WERSA_ERR_CUDA;
  wersa_status s = clear_status_once(ctx, st);
  if (s != WERSA_OK) return s;
  WERSA_CUDA(launch_selftest_small(p, ctx->ws, loss, Q, K, V, W, beta, omega, O, st));
  return WERSA_OK;
}

wersa_status wersa_set_step_timing(wersa_ctx* ctx, int enable) {
  if (ctx == nullptr) return WERSA_ERR_INVALID_ARG;
  StepTimer& t = ctx->timer;
  if ((enable != 0) == t.enabled) return WERSA_OK;
  DeviceGuard guard(ctx->plan.cfg.device);
  if (guard.err != cudaSuccess) return WERSA_ERR_CUDA;
  if (enable) {
    for (int wch = 0; wch < 2; ++wch)
      for (int i = 0; i <= kMaxSteps; ++i) WERSA_CUDA(cudaEventCreate(&t.ev[wch][i]));
    t.count[0] = t.count[1] = 0;
    t.enabled = true;
  } else {
    t.enabled = false;
    for (int wch = 0; wch < 2; ++wch)
      for (int i = 0; i <= kMaxSteps; ++i) cudaEventDestroy(t.ev[wch][i]);
  }
  return WERSA_OK;
}

wersa_status wersa_step_times(wersa_ctx* ctx, int which, int capacity, float* ms, const char** names,
                              int* count) {
  if (ctx == nullptr || count == nullptr || which < 0 || which > 1) return WERSA_ERR_INVALID_ARG;
  StepTimer& t = ctx->timer;
  if (!t.enabled) return WERSA_ERR_STATE;
  DeviceGuard guard(ctx->plan.cfg.device);
  if (guard.err != cudaSuccess) return WERSA_ERR_CUDA;
  const int n = t.count[which];
  *count = n;
  if (n == 0) return WERSA_OK;
  WERSA_CUDA(cudaEventSynchronize(t.ev[which][n]));
  for (int i = 0; i < n && i < capacity; ++i) {
    if (ms != nullptr) WERSA_CUDA(cudaEventElapsedTime(&ms[i], t.ev[which][i], t.ev[which][i + 1]));
    if (names != nullptr) names[i] = t.name[which][i];
  }
  return WERSA_OK;
}

wersa_status wersa_destroy(wersa_ctx* ctx) {
  if (ctx != nullptr && ctx->timer.enabled) wersa_set_step_timing(ctx, 0);
  delete ctx;
  return WERSA_OK;
}

const char* wersa_status_string(wersa_status status) {
  switch (status) {
    case WERSA_OK: return "ok";
    case WERSA_ERR_INVALID_ARG: return "invalid argument";
    case WERSA_ERR_UNSUPPORTED: return "unsupported configuration";
    case WERSA_ERR_WORKSPACE: return "workspace missing, misaligned or too small";
    case WERSA_ERR_CUDA: return "CUDA runtime error";
    case WERSA_ERR_TIMEOUT: return "bounded device wait expired";
    case WERSA_ERR_STATE: return "backward or saved-tensor query without a preceding forward";
    case WERSA_ERR_TOO_LARGE: return "problem exceeds the fixed scratch of wersa_gate_static (253952 floats + 8192 counters)";
  }
  return "unknown status";
}

int32_t wersa_uses_tensor_cores(const wersa_ctx* ctx) { return ctx != nullptr && ctx->plan.use_tc ? 1 : 0; }

int32_t wersa_launch_count(const wersa_ctx* ctx, int which) {
  if (ctx == nullptr) return 0;
  return which == 0 ? ctx->launches_fwd : ctx->launches_bwd;
}

}  // extern "C"
