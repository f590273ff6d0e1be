// Kernels around the at most 256-feature kernels:
//  * feature maps wider than 256 run as groups of 256 features.  With N'_g, D'_g the numerator and
//    denominator of group g (Eq. 7 restricted to the group's features) and eps' shared out evenly,
//    O = sum_g N'_g / sum_g (D'_g + eps'/G) = sum_g O_g den_g / sum_g den_g, where O_g = N'_g / den_g is what
//    the query-side kernel writes for the group and den_g = D'_g + eps'/G is the denominator it leaves beside it.
#include "common.cuh"

namespace wersa {
namespace {

// O[tok][:] = sum_g Og[g][tok][:] * den[g][tok] / sum_g den[g][tok], groups in a fixed order.  Og and O have `cols`
// columns.  One thread per 8 columns of a token; tokens = slabs * n.  Bound by memory: with the groups' outputs as
// wide as the head instead of 64 columns, 4 groups, 512k tokens: d = 16 58 -> 18 us, d = 32 61 -> 33 us.
__global__ void __launch_bounds__(256) k_combine_groups(const __nv_bfloat16* __restrict__ Og, const float* __restrict__ den,
                                                        __nv_bfloat16* __restrict__ O, size_t tokens, int groups, int cols) {
  wait_for_stream_predecessor();   // (launched as a programmatic dependent: see launch_after)
  const size_t idx = (size_t)blockIdx.x * 256 + threadIdx.x;
  const int per = cols >> 3;
  const size_t tok = idx / per;
  if (tok >= tokens) return;
  float acc[8], dsum = 0.f;
#pragma unroll
  for (int j = 0; j < 8; ++j) acc[j] = 0.f;
#pragma unroll 4
  for (int g = 0; g < groups; ++g) {
    const float dg = den[(size_t)g * tokens + tok];
    float v[8];
    load8(Og + ((size_t)g * tokens * per + idx) * 8, v);
#pragma unroll
    for (int j = 0; j < 8; ++j) acc[j] = fmaf(v[j], dg, acc[j]);
    dsum += dg;
  }
  const float inv = 1.f / dsum;
#pragma unroll
  for (int j = 0; j < 8; ++j) acc[j] *= inv;
  store8(O + idx * 8, acc);
}

// O = sum_g Og den_g / sum_g den_g, D = sum_g den_g / r, dD' = -(dO . O) / D, `tpt` threads (a power of two, at least
// d / 8) per token with 8 columns each.  The forward's denominators carry the factor r = bf16(f_0) / f_0 of its filter
// stage, which the backward's filtered planes do not.  (4 groups, 512k tokens, d = 32, Og of d instead of 64 columns:
// 78 -> 45 us.)
__global__ void __launch_bounds__(256) k_group_bwd_prep(const __nv_bfloat16* __restrict__ Og, const float* __restrict__ den,
                                                        const __nv_bfloat16* __restrict__ dO, int d, int tpt, const float* __restrict__ f,
                                                        int n, int L1, size_t tokens, int groups,
                                                        float* __restrict__ Dtot, float* __restrict__ dDtot) {
  wait_for_stream_predecessor();   // (launched as a programmatic dependent: see launch_after)
  let_stream_successor_start();
  const size_t idx = (size_t)blockIdx.x * 256 + threadIdx.x;
  const size_t tok = idx / tpt;
  const int c0 = (int)(idx & (tpt - 1)) * 8;
  const bool live = tok < tokens && c0 < d;
  float dsum = 0.f, dot = 0.f;
  if (live) {
    float acc[8], g8[8];
    load8(dO + tok * d + c0, g8);
#pragma unroll
    for (int j = 0; j < 8; ++j) acc[j] = 0.f;
#pragma unroll 4
    for (int g = 0; g < groups; ++g) {
      const float dg = den[(size_t)g * tokens + tok];
      float v[8];
      load8(Og + ((size_t)g * tokens + tok) * d + c0, v);
#pragma unroll
      for (int j = 0; j < 8; ++j) acc[j] = fmaf(v[j], dg, acc[j]);
      dsum += dg;
    }
#pragma unroll
    for (int j = 0; j < 8; ++j) dot = fmaf(g8[j], acc[j], dot);
  }
  for (int o = tpt >> 1; o > 0; o >>= 1) dot += __shfl_xor_sync(0xffffffffu, dot, o);   // the threads of a token
  if (live && c0 == 0) {
    const float f0 = f[(tok / n) * L1];
    const float f0b = __bfloat162float(__float2bfloat16_rn(f0));
    const float r = f0 != 0.f ? f0b / f0 : 1.f;
    const float D = dsum / r;
    // dot = sum_c dO_c (sum_g Og_c den_g); O = that / dsum
    Dtot[tok] = D;
    dDtot[tok] = -(dot / dsum) / D;
  }
}

unsigned blocks_for(size_t threads) { return (unsigned)((threads + 255) / 256); }

}  // namespace

cudaError_t launch_combine_groups(const void* Og, const float* den, void* O, size_t tokens, int groups, int cols,
                                  cudaStream_t st, int* launches) {
  using bf = __nv_bfloat16;
  *launches += 1;
  return launch_after(k_combine_groups, dim3(blocks_for(tokens * (cols >> 3))), dim3(256), 0, st, (const bf*)Og, den, (bf*)O,
                      tokens, groups, cols);
}

cudaError_t launch_group_bwd_prep(const void* Og, const float* den, const void* dO, int d, const float* f, int n, int L1,
                                  size_t tokens, int groups, float* Dtot, float* dDtot, cudaStream_t st, int* launches) {
  using bf = __nv_bfloat16;
  int tpt = 1;
  while (8 * tpt < d) tpt <<= 1;
  *launches += 1;
  return launch_after(k_group_bwd_prep, dim3(blocks_for(tokens * tpt)), dim3(256), 0, st, (const bf*)Og, den, (const bf*)dO, d,
                      tpt, f, n, L1, tokens, groups, Dtot, dDtot);
}

}  // namespace wersa
