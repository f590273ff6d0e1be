// Backward of the gate, for the kernel of its own (gate.cu) and for the pass that writes dQ (haar.cu).
#pragma once
#include "common.cuh"

namespace wersa {

// df of one slab: given (slabs x kBandVals), or added up where it is wanted from the band inner products of `blocks` CTAs per slab
// and tensor.  i < L: the detail band of level i + 1, i = L: the approximation band of level L.
struct GivenDf {
  const float* df;
  __device__ __forceinline__ float operator()(int slab, int i) const { return __ldcg(df + (size_t)slab * kBandVals + i); }
};
struct SummedDf {
  const float* bands;
  int slabs, blocks, L;
  __device__ __forceinline__ float operator()(int slab, int i) const {
    float s = 0.f;
    const float* src = bands + (size_t)slab * blocks * kBandVals + (i < L ? i : 8 + L - 1);
    const size_t other = (size_t)slabs * blocks * kBandVals;
    // (the addresses depend on nothing: as many loads in flight as registers allow, those past the end of the last one's place)
    for (int t = 0; t < blocks; t += 8) {
      float v[16];
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        const int u = min(t + j, blocks - 1) * kBandVals;
        v[j] = __ldcg(src + u);
        v[8 + j] = __ldcg(src + other + u);
      }
#pragma unroll
      for (int j = 0; j < 8; ++j) s += t + j < blocks ? v[j] + v[8 + j] : 0.f;
    }
    return s;
  }
};

// Chain rule through f = sigmoid(u) * omega, u = gate(qbar): domega, dgate_b, dgate_w, dqbar; and the
// bandwidth gradient dbeta = 2 eps m bw * sum_t dDh_t (ReLU is positively homogeneous, so beta only
// acts through eps).  Grid H + 2, 256 threads: CTA h < H handles head h, CTA H sums domega, CTA H + 1 sums dbeta; every
// sum has a fixed order.  In CTA h the 256 threads work out du of 28 batch elements x 9 levels at a time, one each, while
// q-bar is on its way; then thread (c = column of q-bar, q) takes the batch elements q, q + 4, ... of the round.  All of
// it is latency: with the reduction before it 36 us at B=32 H=4 with a barrier and a dependent load per batch element,
// 20 us with every thread working out du itself (with the gate shared by the heads nine loads after one another:
// 19 us at B=5 H=3), 11 now (9 at B=5 H=3).
template <typename Df> __device__ __forceinline__ float gate_df(const Df& df, int b, int h, int H, int per_head, int i) {
  if (per_head) return df(b * H + h, i);
  float s = 0.f;
#pragma unroll 4
  for (int hh = 0; hh < H; ++hh) s += df(b * H + hh, i);
  return s;
}
// kParts = 4 parts of 64 threads, 16 where the batch is more than one round of four: at B=341 H=3 13 rounds of two
// latencies each, and 22 for domega, took 37 us of a training step of 291, with 16 parts 16 (the step 271).
// Sum of the parts' values in pairs of pairs.
template <int kParts, typename F>
__device__ __forceinline__ float sum_parts(F value) {
  float s = (value(0) + value(1)) + (value(2) + value(3));
#pragma unroll
  for (int a = 4; a < kParts; a += 4) s += (value(a) + value(a + 1)) + (value(a + 2) + value(a + 3));
  return s;
}
// (Kernels take these as parameters of their own: pointers out of a structure are generic ones, 2 of 10 us.)
struct GateBwdArgs {
  const float *sg, *qbar, *gate_w, *omega, *sumdD, *beta;
  int n_sumdD;
  float eps, bw_floor;
  int m, B, H, dcols, L1, per_head;
  float *dbeta, *dgate_w, *dgate_b, *domega, *dqbar;   // dqbar may be null
};
// What CTA `cta` of H + 2 does, with 64 kParts threads.  Behind `wait` everything of the kernels in front may be read; gate
// weights are read ahead of it.
template <int kParts, typename Df, typename Wait>
__device__ __forceinline__ void gate_backward_cta(int cta, const Df& df, const GateBwdArgs& a, Wait&& wait) {
  const float *__restrict__ sg = a.sg, *__restrict__ qbar = a.qbar, *__restrict__ gate_w = a.gate_w, *__restrict__ omega = a.omega;
  float *__restrict__ dqbar = a.dqbar, *__restrict__ dgate_w = a.dgate_w, *__restrict__ dgate_b = a.dgate_b;
  const int B = a.B, H = a.H, dcols = a.dcols, L1 = a.L1, per_head = a.per_head;
  constexpr int kThreads = 64 * kParts;
  constexpr int kGateRound = 7 * kParts;   // batch elements of a round: seven a part, 7 x 9 values for its 64 threads
  static_assert(kGateRound * (kMaxLevels + 1) <= kThreads, "a value of a round per thread");
  __shared__ float part[kParts][kMaxLevels + 1][kD];
  __shared__ float gbs[kParts][kMaxLevels + 1];
  __shared__ float dus[kGateRound][kMaxLevels + 1];
  float* flat = &part[0][0][0];
  const int tid = threadIdx.x;
  if (cta < H) {
    const int h = cta, c = tid & (kD - 1), q = tid >> 6;
    float gw[kMaxLevels + 1], gw_acc[kMaxLevels + 1], gb_acc[kMaxLevels + 1];
#pragma unroll
    for (int i = 0; i <= kMaxLevels; ++i) {
      gw_acc[i] = gb_acc[i] = 0.f;
      gw[i] = i < L1 && gate_w != nullptr && c < dcols ? gate_w[((size_t)h * dcols + c) * L1 + i] : 0.f;
    }
    wait();
    const int db = tid / (kMaxLevels + 1), di = tid - db * (kMaxLevels + 1);   // this thread's du of a round
    for (int b0 = 0; b0 < B; b0 += kGateRound) {
      float qb[kGateRound / kParts];
#pragma unroll
      for (int r = 0; r < kGateRound / kParts; ++r) {
        const int b = b0 + q + kParts * r;
        qb[r] = b < B ? qbar[((size_t)b * H + h) * kD + c] : 0.f;
      }
      if (b0 > 0) __syncthreads();   // the round before has been read
      if (db < kGateRound) {
        float du = 0.f;
        if (di < L1 && b0 + db < B) {
          const float s = sg[((size_t)(b0 + db) * H + h) * L1 + di];
          du = gate_df(df, b0 + db, h, H, per_head, di) * omega[di] * s * (1.f - s);
        }
        dus[db][di] = du;
      }
      __syncthreads();
#pragma unroll
      for (int r = 0; r < kGateRound / kParts; ++r) {
        const int b = b0 + q + kParts * r;
        if (b >= B) break;
        float dq = 0.f;
#pragma unroll
        for (int i = 0; i <= kMaxLevels; ++i)
          if (i < L1) {
            const float du = dus[q + kParts * r][i];
            gw_acc[i] += qb[r] * du;
            gb_acc[i] += du;
            if (gate_w != nullptr) dq += gw[i] * du;   // (none without weights, whatever du is)
          }
        if (dqbar != nullptr) dqbar[((size_t)b * H + h) * kD + c] = dq;
      }
    }
#pragma unroll
    for (int i = 0; i <= kMaxLevels; ++i) {
      part[q][i][c] = gw_acc[i];
      if (c == 0) gbs[q][i] = gb_acc[i];
    }
    __syncthreads();
    for (int e = tid; e < dcols * L1; e += kThreads) {   // (columns past the head dimension are padding of qbar)
      const int cc = e / L1, i = e - cc * L1;
      if (dgate_w != nullptr)
        dgate_w[(size_t)h * dcols * L1 + e] = sum_parts<kParts>([&](int a) { return part[a][i][cc]; });
    }
    if (dgate_b != nullptr && tid < L1)
      dgate_b[h * L1 + tid] = per_head || h == 0 ? sum_parts<kParts>([&](int a) { return gbs[a][tid]; }) : 0.f;
  } else if (cta == H) {
    // domega[i] = sum over slabs of df_i * sigmoid(u_i) (one sigmoid for the heads of a batch element where they share the gate):
    // thread (i = tid & 15, q = tid >> 4) takes every (4 kParts)th slab, then the parts are added in order
    const int i = tid & 15, q = tid >> 4;
    float acc = 0.f;
    wait();
    if (a.domega != nullptr && i < L1) {
#pragma unroll 4
      for (int slab = q; slab < B * H; slab += 4 * kParts) acc += df(slab, i) * sg[(size_t)slab * L1 + i];
    }
    flat[tid] = acc;
    __syncthreads();
    if (a.domega != nullptr && tid < L1) {
      float s = 0.f;
#pragma unroll
      for (int r = 0; r < 4 * kParts; ++r) s += flat[16 * r + tid];
      a.domega[tid] = s;
    }
  } else {
    wait();
    float tot = 0.f;
#pragma unroll 4
    for (int i = tid; i < a.n_sumdD; i += kThreads) tot += __ldcg(a.sumdD + i);
    flat[tid] = tot;
    __syncthreads();
    for (int o = kThreads / 2; o > 0; o >>= 1) {
      if (tid < o) flat[tid] += flat[tid + o];
      __syncthreads();
    }
    if (a.dbeta != nullptr && tid == 0) {
      const float bt = a.beta[0];
      const float bw = fmaxf(bt, a.bw_floor);
      a.dbeta[0] = bt > a.bw_floor ? 2.f * a.eps * (float)a.m * bw * flat[0] : 0.f;
    }
  }
}

}  // namespace wersa
