// Mean-pooled query, content-adaptive gate (Eqs. 1-3 of the WERSA paper) and its backward pass.
#include <mutex>

#include "cluster.cuh"
#include "common.cuh"
#include "gate_backward.cuh"

namespace wersa {
namespace {

// Scratch of wersa_gate_static: lives in the library image of every GPU that loads it.  The last
// kStaticCounterInts elements are reserved for the arrival counters, at a place that does not depend on
// the problem, so that no float of any call's layout can ever land on them.
constexpr size_t kStaticScratchFloats = 262144;   // 1 MiB
constexpr size_t kStaticCounterInts = 8192;       // slab counters, then batch counters
static __device__ __align__(256) float g_static_scratch[kStaticScratchFloats];
constexpr int kMaxDevices = 64;
float* g_static_scratch_addr[kMaxDevices] = {nullptr};
std::mutex g_static_scratch_mutex;

// Finish of one slab by one CTA (256 threads): qbar = sum of the chunk partials load(chunk, column) in chunk order / n (Eq. 1), the head's logits u = gate_w[h]^T qbar (Eq. 2) and, for the
// per-head gate, sigmoid(u + gate_b[h]) and f = sigmoid * omega (Eq. 3).  For the batch-wide gate the
// bias-free logits are parked in f for batch_gate.
template <typename Load>
__device__ __forceinline__ void slab_gate(Load&& load, int qchunks, int slab, int H, int n, int L1,
                                          int per_head, const float* __restrict__ gate_w,
                                          const float* __restrict__ gate_b, const float* __restrict__ omega,
                                          float* __restrict__ qbar, float* __restrict__ sg, float* __restrict__ f,
                                          float (*red)[kD], float* qs, int dcols) {
  const int h = slab % H;
  const int c = threadIdx.x & (kD - 1), part = threadIdx.x >> 6;   // 4 interleaved partial sums per column
  // logits: 16 lanes per band, four of the 64 terms each; what they need of the gate is fetched ahead of the sums
  const int i = threadIdx.x >> 4, seg = threadIdx.x & 15;
  float gw[4], gb = 0.f, om = 1.f;
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    const int kk = seg * 4 + j;   // gate_w is (heads, dcols, L1); columns >= dcols of qbar are zero padding
    gw[j] = gate_w != nullptr && i < L1 && kk < dcols ? gate_w[((size_t)h * dcols + kk) * L1 + i] : 0.f;
  }
  if (i < L1 && per_head) {
    if (gate_b != nullptr) gb = gate_b[h * L1 + i];
    if (omega != nullptr) om = omega[i];
  }
  float s = 0.f;
  int k = part;
  for (; k + 12 < qchunks; k += 16) {
    const float v0 = load(k, c), v1 = load(k + 4, c), v2 = load(k + 8, c), v3 = load(k + 12, c);
    s += (v0 + v1) + (v2 + v3);
  }
  {
    float v[3];   // at most three left
#pragma unroll
    for (int j = 0; j < 3; ++j) v[j] = k + 4 * j < qchunks ? load(k + 4 * j, c) : 0.f;
#pragma unroll
    for (int j = 0; j < 3; ++j) s += v[j];
  }
  red[part][c] = s;
  __syncthreads();
  if (threadIdx.x < kD) {
    const float q = ((red[0][c] + red[1][c]) + (red[2][c] + red[3][c])) / (float)n;
    qbar[(size_t)slab * kD + c] = q;
    qs[c] = q;
  }
  __syncthreads();
  float u = 0.f;   // (then a fixed-order butterfly)
  if (gate_w != nullptr) {   // without weights the logits are the bias alone, whatever q-bar is (0 * inf)
#pragma unroll
    for (int j = 0; j < 4; ++j) u += gw[j] * qs[seg * 4 + j];
  }
#pragma unroll
  for (int o = 8; o > 0; o >>= 1) u += __shfl_xor_sync(0xffffffffu, u, o);
  if (i < L1 && seg == 0) {
    if (per_head) {
      u += gb;
      const float sgm = 1.f / (1.f + expf(-u));
      sg[(size_t)slab * L1 + i] = sgm;
      f[(size_t)slab * L1 + i] = sgm * om;
    } else {
      f[(size_t)slab * L1 + i] = u;
    }
  }
}

// Batch-wide gate (Algorithm 1, W_filter), by the last slab of a batch element to finish:
// u[b] = sum_h u[b,h] + gate_b[0], one sigmoid per batch element shared by its heads.
__device__ __forceinline__ void batch_gate(int b, int H, int L1, const float* __restrict__ gate_b,
                                           const float* __restrict__ omega, float* __restrict__ sg,
                                           float* __restrict__ f) {
  const int i = threadIdx.x;
  if (i >= L1) return;
  float u = gate_b != nullptr ? gate_b[i] : 0.f;
  for (int h = 0; h < H; ++h) u += __ldcg(f + ((size_t)b * H + h) * L1 + i);
  const float sgm = 1.f / (1.f + expf(-u));
  for (int h = 0; h < H; ++h) {
    sg[((size_t)b * H + h) * L1 + i] = sgm;
    f[((size_t)b * H + h) * L1 + i] = sgm * (omega != nullptr ? omega[i] : 1.f);
  }
}

// Mean pool and gate in one launch.  grid (qcluster or qchunks, slabs [+ 1]), block 256.
// Rows y < slabs: partial column sums of one row chunk of one slab of Q -- thread (cg = tid & 7,
// rl = tid >> 3) owns 8 consecutive columns and every 32nd row, loads 16 bytes (bf16) / 32 bytes
// (fp32) per row, four rows in flight, with the streaming cache hint (Q is read once here).  kCluster: the chunks of a slab are a
// cluster, whose first block gets the others' sums into its shared memory and runs slab_gate.  Otherwise the CTA that finds it is
// the last of its slab to finish (a counter per slab) does, which takes two fences, an atomic and two more trips to the L2 (1 x 1024
// fp32 4.3 us of a forward, 3.2 as a cluster; 5 x 3 x 1777 9.5 and 8.2; 8 x 8 x 4096 12.2 and 10.6).  For the batch-wide gate the last
// slab of a batch element (a counter per batch element) runs batch_gate; sums are taken in a fixed order, so the result does not
// depend on which CTA comes last.  The counters start at zero and are left at zero.
// Row y == slabs (only of bf16 tensors, with W or seen): bf16 transpose Wt (m x 64) of W (64 x m) for the tensor-core kernels;
// seen is cleared there.
// kFull = false: Q has dcols < 64 columns (a multiple of 8), gate_w dcols rows per head and W dcols rows;
// dcols / 8 threads share a row, 256 / (dcols / 8) rows are in flight per pass, and the partial sums, q-bar
// and W^T come out 64 wide with zeros in the columns past dcols.  fp32 tensors keep the 64-wide assignment
// (eight threads a row, those past dcols idle): their sums have the bits of the zero-padded problem.
template <typename T, bool kFull, bool kCluster>
__global__ void __launch_bounds__(256) k_qmean_gate(const T* __restrict__ Q, float* __restrict__ qpart, int n,
                                                    int chunk_rows, int slabs, int H, int L1, int per_head,
                                                    const float* __restrict__ gate_w, const float* __restrict__ gate_b,
                                                    const float* __restrict__ omega, float* __restrict__ qbar,
                                                    float* __restrict__ sg, float* __restrict__ f,
                                                    int* __restrict__ slab_count, int* __restrict__ batch_count,
                                                    const __nv_bfloat16* __restrict__ W, __nv_bfloat16* __restrict__ Wt,
                                                    int m, int dcols_arg, int* __restrict__ seen) {
  const int dcols = kFull ? kD : dcols_arg;
  // This grid may have been placed while the work before it in the stream was still running: nothing is
  // read or written before that work has completed.  After that the key-side kernel may be staged
  // (programmatic dependent launch; it waits for this grid before it reads W^T or the gate).
  asm volatile("griddepcontrol.wait;" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  if constexpr (sizeof(T) == 4) {   // (in the bf16 kernels, which have no use for it, four registers and a CTA per SM)
    if (seen != nullptr && blockIdx.x + blockIdx.y == 0 && threadIdx.x < 2) seen[threadIdx.x] = 0;   // see k_f32_planes
  }
  if ((int)blockIdx.y == slabs) {
    if (sizeof(T) == 2 && seen != nullptr && blockIdx.x == 0 && threadIdx.x < 2) seen[threadIdx.x] = 0;   // see k_f32_planes
    if (W == nullptr) return;
    // A thread takes eight columns of W^T's row r: neighbouring threads read neighbouring features and store 16 bytes.  (An
    // element a thread reads 2 bytes out of 32 different sectors a warp, and the grid's other CTAs wait for nothing else:
    // with two chunks a slab and m = 1024 this row took as long as all of the mean pool, 24.9 us; now 12.4.)
    for (int i = blockIdx.x * 256 + threadIdx.x; i < m * (kD / 8); i += gridDim.x * 256) {
      const int c0 = i / m * 8, r = i - c0 / 8 * m;
      union {
        __nv_bfloat16 v[8];
        uint4 all;
      } w;
      w.all = make_uint4(0u, 0u, 0u, 0u);
      if (c0 < dcols) {
#pragma unroll
        for (int j = 0; j < 8; ++j) w.v[j] = W[(size_t)(c0 + j) * m + r];
      }
      *reinterpret_cast<uint4*>(Wt + (size_t)r * kD + c0) = w.all;
    }
    return;
  }
  if constexpr (kCluster) cluster_arrive();
  const int chunk = blockIdx.x, slab = blockIdx.y;
  const int cgs = kFull || sizeof(T) == 4 ? 8 : dcols >> 3;   // threads across a row
  const int rp = kFull ? 32 : 256 / cgs;       // rows per pass
  const int cg = kFull ? (threadIdx.x & 7) : (int)threadIdx.x % cgs;
  const int rl = kFull ? (threadIdx.x >> 3) : (int)threadIdx.x / cgs;
  const bool on = kFull || (rl < rp && cg * 8 < dcols);   // (256 need not be a multiple of cgs)
  const int r0 = chunk * chunk_rows;
  const int r1 = min(n, r0 + chunk_rows);
  const T* base = Q + (size_t)slab * n * dcols + cg * 8;
  float acc[8];
#pragma unroll
  for (int j = 0; j < 8; ++j) acc[j] = 0.f;
  int r = on ? r0 + rl : r1;
  for (; r + 3 * rp < r1; r += 4 * rp) {
    float v0[8], v1[8], v2[8], v3[8];
    load8_stream(base + (size_t)r * dcols, v0);
    load8_stream(base + (size_t)(r + rp) * dcols, v1);
    load8_stream(base + (size_t)(r + 2 * rp) * dcols, v2);
    load8_stream(base + (size_t)(r + 3 * rp) * dcols, v3);
#pragma unroll
    for (int j = 0; j < 8; ++j) acc[j] += (v0[j] + v1[j]) + (v2[j] + v3[j]);
  }
  for (; r < r1; r += rp) {
    float v0[8];
    load8_stream(base + (size_t)r * dcols, v0);
#pragma unroll
    for (int j = 0; j < 8; ++j) acc[j] += v0[j];
  }
  __shared__ float red[kFull ? 32 * (kD + 1) : 256 * 9];   // rp rows of dcols + 1 floats
  __shared__ float red4[4][kD];
  __shared__ float qs[kD];
  __shared__ int s_last;
  if (on) {
#pragma unroll
    for (int j = 0; j < 8; ++j) red[rl * (dcols + 1) + cg * 8 + j] = acc[j];
  }
  __syncthreads();
  float total = 0.f;   // kCluster
  if (threadIdx.x < kD) {
    float s = 0.f;
    if ((int)threadIdx.x < dcols) {
#pragma unroll 8
      for (int i = 0; i < rp; ++i) s += red[i * (dcols + 1) + threadIdx.x];   // fixed order
    }
    if constexpr (!kCluster) {
      qpart[((size_t)slab * gridDim.x + chunk) * kD + threadIdx.x] = s;
      __threadfence();
    } else {
      total = s;
    }
  }
  if constexpr (kCluster) {
    __shared__ float shares[kMaxCluster][kD];
    cluster_wait();   // (the first block has begun)
    if (threadIdx.x < kD) peer_store(peer_addr(shared_addr(&shares[chunk][threadIdx.x]), 0), total);
    cluster_release();
    cluster_acquire();
    if (chunk != 0) return;
    slab_gate([&](int k, int c) { return shares[k][c]; }, gridDim.x, slab, H, n, L1, per_head, gate_w, gate_b, omega, qbar, sg, f, red4,
              qs, dcols);
  } else {
    __syncthreads();
    if (threadIdx.x == 0) s_last = atomicAdd(&slab_count[slab], 1) == (int)gridDim.x - 1;
    __syncthreads();
    if (!s_last) return;
    __threadfence();
    const float* src = qpart + (size_t)slab * gridDim.x * kD;
    slab_gate([&](int k, int c) { return __ldcg(src + (size_t)k * kD + c); }, gridDim.x, slab, H, n, L1, per_head, gate_w, gate_b, omega,
              qbar, sg, f, red4, qs, dcols);
    if (threadIdx.x == 0) slab_count[slab] = 0;
  }
  if (per_head) return;
  __threadfence();
  __syncthreads();
  const int b = slab / H;
  if (threadIdx.x == 0) s_last = atomicAdd(&batch_count[b], 1) == H - 1;
  __syncthreads();
  if (!s_last) return;
  __threadfence();
  batch_gate(b, H, L1, gate_b, omega, sg, f);
  if (threadIdx.x == 0) batch_count[b] = 0;
}

// Gate from column sums that are already complete (sequence shards: the sums of all shards were added by the
// caller): one CTA of 256 threads per slab runs slab_gate on a single "partial" with the whole sequence's
// length, then, for the batch-wide gate, a second launch runs batch_gate per batch element.
// qbar_scale: q-bar of a shard times its length gives the shard's column sums back.
__global__ void __launch_bounds__(256) k_scale_qbar(const float* __restrict__ qbar, float scale,
                                                    float* __restrict__ qsum, int count) {
  wait_for_stream_predecessor();   // (launched as a programmatic dependent: see launch_after)
  const int i = blockIdx.x * 256 + threadIdx.x;
  if (i < count) qsum[i] = qbar[i] * scale;
}
__global__ void __launch_bounds__(256) k_gate_from_sums(const float* __restrict__ qsum, int H, int n_total, int L1,
                                                        int per_head, const float* __restrict__ gate_w,
                                                        const float* __restrict__ gate_b,
                                                        const float* __restrict__ omega, float* __restrict__ qbar,
                                                        float* __restrict__ sg, float* __restrict__ f, int dcols) {
  wait_for_stream_predecessor();   // (launched as a programmatic dependent: see launch_after)
  __shared__ float red4[4][kD];
  __shared__ float qs[kD];
  const float* src = qsum + (size_t)blockIdx.x * kD;
  slab_gate([&](int, int c) { return __ldcg(src + c); }, 1, blockIdx.x, H, n_total, L1, per_head, gate_w, gate_b, omega, qbar, sg, f, red4, qs, dcols);
}
__global__ void __launch_bounds__(32) k_batch_gate(int H, int L1, const float* __restrict__ gate_b,
                                                   const float* __restrict__ omega, float* __restrict__ sg,
                                                   float* __restrict__ f) {
  wait_for_stream_predecessor();   // (launched as a programmatic dependent: see launch_after)
  batch_gate(blockIdx.x, H, L1, gate_b, omega, sg, f);
}

// Sum the per-tile band inner products of both filtered tensors and turn them into df[slab][i]: i < L takes
// the detail-band product of level i+1, i = L the approximation product of level L.  One CTA of 256 threads
// per slab: thread (j = tid & 15, part = tid >> 4) adds every 16th partial of band slot j in tile order
// (four loads in flight), the 16 parts are added in a fixed order: the result repeats bit for bit.
__global__ void __launch_bounds__(256) k_band_reduce(const float* __restrict__ bands, int slabs, int htiles,
                                                     int L, float* __restrict__ df) {
  // (launched as a programmatic dependent: see launch_after; the gate backward, which may be placed ahead of this kernel's
  // wait, reads nothing of the passes over dK_F and dQ_F but what this kernel leaves it)
  let_stream_successor_start();
  wait_for_stream_predecessor();
  __shared__ float part[16][kBandVals];
  const int slab = blockIdx.x, j = threadIdx.x & (kBandVals - 1), pt = threadIdx.x >> 4;
  float s = 0.f;
  for (int which = 0; which < 2; ++which) {
    const float* src = bands + (((size_t)which * slabs + slab) * htiles) * kBandVals + j;
    int t = pt;
    for (; t + 48 < htiles; t += 64) {
      const float v0 = __ldcg(src + (size_t)t * kBandVals), v1 = __ldcg(src + (size_t)(t + 16) * kBandVals);
      const float v2 = __ldcg(src + (size_t)(t + 32) * kBandVals), v3 = __ldcg(src + (size_t)(t + 48) * kBandVals);
      s += (v0 + v1) + (v2 + v3);
    }
    for (; t < htiles; t += 16) s += __ldcg(src + (size_t)t * kBandVals);
  }
  part[pt][j] = s;
  __syncthreads();
  if (threadIdx.x < kBandVals) {
    float tot = 0.f;
#pragma unroll
    for (int q = 0; q < 16; ++q) tot += part[q][j];
    // slots 0..7: detail products of levels 1..8; slots 8..15: approximation products of levels 1..8
    if (j < L) df[(size_t)slab * kBandVals + j] = tot;
    if (j == 8 + L - 1) df[(size_t)slab * kBandVals + L] = tot;
  }
}

// out[0] = sum of x[0..n) in a fixed order (64 threads, strided partial sums, then a tree).
__global__ void __launch_bounds__(kD) k_sum_floats(const float* __restrict__ x, int n, float* __restrict__ out) {
  wait_for_stream_predecessor();   // (launched as a programmatic dependent: see launch_after)
  __shared__ float part[kD];
  const int c = threadIdx.x;
  float tot = 0.f;
  for (int i = c; i < n; i += kD) tot += x[i];
  part[c] = tot;
  __syncthreads();
  for (int o = kD / 2; o > 0; o >>= 1) {
    if (c < o) part[c] += part[c + o];
    __syncthreads();
  }
  if (c == 0) out[0] = part[0];
}

// (launched as a programmatic dependent: see launch_after; the pass that writes dQ may be placed ahead of this kernel's wait, and
// unless it is the first one of its pass the gate weights are fetched ahead of it)
template <int kParts>
__global__ void __launch_bounds__(64 * kParts) k_gate_backward(
    const float* __restrict__ df, const float* __restrict__ sg, const float* __restrict__ qbar, const float* __restrict__ gate_w,
    const float* __restrict__ omega, const float* __restrict__ sumdD, int n_sumdD, const float* __restrict__ beta, float eps,
    float bw_floor, int m, int B, int H, int dcols, int L1, int per_head, float* __restrict__ dbeta, float* __restrict__ dgate_w,
    float* __restrict__ dgate_b, float* __restrict__ domega, float* __restrict__ dqbar, bool first) {
  if (first) wait_for_stream_predecessor();
  let_stream_successor_start();
  const GateBwdArgs args = {sg, qbar, gate_w, omega, sumdD, beta, n_sumdD, eps, bw_floor, m, B, H, dcols, L1, per_head,
                            dbeta, dgate_w, dgate_b, domega, dqbar};
  gate_backward_cta<kParts>(blockIdx.x, GivenDf{df}, args, []() { wait_for_stream_predecessor(); });
}

}  // namespace

// The launch shared by the workspace and the static-scratch variants.
static cudaError_t launch_qmean_gate_impl(const Plan& p, const void* Q, float* qpart, const float* gate_w,
                                          const float* gate_b, const float* omega, float* qbar, float* sg, float* f,
                                          int* counters, const void* W, __nv_bfloat16* Wt, int cols,
                                          int* seen, bool cluster, cudaStream_t st) {
  const int rows = p.slabs + (W != nullptr || (p.bf16 && seen != nullptr) ? 1 : 0);
  int* slab_count = counters;
  int* batch_count = counters + p.slabs;
  cudaError_t launch_err = cudaSuccess;
  // Launched as a programmatic dependent of whatever precedes it in the stream: the kernel's first instruction waits for that
  // work to complete, so ordering and visibility are those of a plain launch, but its CTAs are already placed when the wait
  // ends (2 us per forward in a sequence of steps).
  auto launch = [&](auto kernel, auto clustered, auto* q) {
    auto go = [&](int chunk_rows, auto start) {
      launch_err = start(q, qpart, p.cfg.seq_len, chunk_rows, p.slabs, p.cfg.heads, p.L1, p.cfg.gate_per_head, gate_w, gate_b, omega,
                         qbar, sg, f, slab_count, batch_count, (const __nv_bfloat16*)W, Wt, p.cfg.features, cols, seen);
    };
    if (cluster) {
      go(p.qcluster_rows, [&](auto... args) { return launch_cluster(clustered, dim3(p.qcluster, rows), dim3(256), 0, st, args...); });
      if (launch_err == cudaSuccess) return;
      cudaGetLastError();   // (a part of a GPU may have no room for a cluster of more than eight)
    }
    go(p.qchunk_rows, [&](auto... args) { return launch_after(kernel, dim3(p.qchunks, rows), dim3(256), 0, st, args...); });
  };
  using bf = __nv_bfloat16;
  if (p.bf16) {
    if (cols == kD) launch(k_qmean_gate<bf, true, false>, k_qmean_gate<bf, true, true>, (const bf*)Q);
    else launch(k_qmean_gate<bf, false, false>, k_qmean_gate<bf, false, true>, (const bf*)Q);
  } else {
    if (cols == kD) launch(k_qmean_gate<float, true, false>, k_qmean_gate<float, true, true>, (const float*)Q);
    else launch(k_qmean_gate<float, false, false>, k_qmean_gate<float, false, true>, (const float*)Q);
  }
  return launch_err != cudaSuccess ? launch_err : cudaGetLastError();
}

cudaError_t launch_qmean_gate(const Plan& p, const Ws& w, const void* Q, const float* gate_w,
                              const float* gate_b, const float* omega, const void* W, int cols, cudaStream_t st,
                              int* launches) {
  *launches += 1;
  return launch_qmean_gate_impl(p, Q, w.qpart, gate_w, gate_b, omega, w.qbar, w.sg, w.f, w.counters, W, w.Wt, cols,
                                p.use_x ? w.seen : nullptr, p.qcluster > 0, st);
}

void prepare_qmean_gate(const Plan& p) {
  using bf = __nv_bfloat16;
  const bool full = p.cfg.head_dim == kD;
  if (p.qcluster == 0) return;
  auto go = [&](auto kernel) {
    if (prepare_cluster(kernel, 0, p.qcluster) != cudaSuccess) cudaGetLastError();   // (the launch then falls back)
  };
  if (p.bf16) full ? go(k_qmean_gate<bf, true, true>) : go(k_qmean_gate<bf, false, true>);
  else full ? go(k_qmean_gate<float, true, true>) : go(k_qmean_gate<float, false, true>);
}

cudaError_t launch_shard_qsum(const Plan& p, const Ws& w, float* qsum, cudaStream_t st, int* launches) {
  const int count = p.slabs * kD;
  launch_after(k_scale_qbar, dim3((count + 255) / 256), dim3(256), 0, st, w.qbar, (float)p.cfg.seq_len, qsum, count);
  *launches += 1;
  return cudaGetLastError();
}

cudaError_t launch_gate_from_sums(const Plan& p, const Ws& w, const float* qsum, long long n_total,
                                  const float* gate_w, const float* gate_b, const float* omega, int cols,
                                  cudaStream_t st, int* launches) {
  launch_after(k_gate_from_sums, dim3(p.slabs), dim3(256), 0, st, qsum, p.cfg.heads, (int)n_total, p.L1, p.cfg.gate_per_head, gate_w, gate_b,
                                           omega, w.qbar, w.sg, w.f, cols);
  *launches += 1;
  if (!p.cfg.gate_per_head) {
    launch_after(k_batch_gate, dim3(p.cfg.batch), dim3(32), 0, st, p.cfg.heads, p.L1, gate_b, omega, w.sg, w.f);
    *launches += 1;
  }
  return cudaGetLastError();
}

// Device address of the static scratch array on the current device, resolved once per device.
// In host code the array's name is only a handle: the kernels need the address this returns.
cudaError_t static_scratch_address(int device, float** out) {
  if (device < 0 || device >= kMaxDevices) return cudaErrorInvalidDevice;
  std::lock_guard<std::mutex> lock(g_static_scratch_mutex);
  if (g_static_scratch_addr[device] == nullptr) {
    void* ptr = nullptr;
    cudaError_t err = cudaGetSymbolAddress(&ptr, g_static_scratch);
    if (err != cudaSuccess) return err;
    g_static_scratch_addr[device] = static_cast<float*>(ptr);
  }
  *out = g_static_scratch_addr[device];
  return cudaSuccess;
}

size_t static_scratch_capacity_floats() { return kStaticScratchFloats - kStaticCounterInts; }
size_t static_scratch_counter_capacity() { return kStaticCounterInts; }

cudaError_t launch_qmean_gate_static(const Plan& p, float* scratch, const void* Q, const float* gate_w,
                                     const float* gate_b, const float* omega, float* qbar, float* f,
                                     cudaStream_t st) {
  // scratch = [ partial column sums: slabs x qchunks x 64 | sigmoid(u): slabs x (L+1) | unused ...
  //             | arrival counters in the last kStaticCounterInts elements: slabs, then batch ints ]
  // The counters this call uses are cleared on the stream first (a memset allocates nothing): a call
  // then starts from zero whatever an earlier call of another shape, or one that failed half way, left.
  float* qpart = scratch;
  float* sg = scratch + (size_t)p.slabs * p.qchunks * kD;
  int* counters = reinterpret_cast<int*>(scratch + (kStaticScratchFloats - kStaticCounterInts));
  cudaError_t err = cudaMemsetAsync(counters, 0, sizeof(int) * ((size_t)p.slabs + (size_t)p.cfg.batch), st);
  if (err != cudaSuccess) return err;
  return launch_qmean_gate_impl(p, Q, qpart, gate_w, gate_b, omega, qbar, sg, f, counters, nullptr, nullptr, kD, nullptr, false, st);
}

size_t static_scratch_floats_needed(const Plan& p) {
  return (size_t)p.slabs * p.qchunks * kD + (size_t)p.slabs * p.L1;
}
size_t static_scratch_counters_needed(const Plan& p) { return (size_t)p.slabs + (size_t)p.cfg.batch; }

static GateBwdArgs gate_args(const Plan& p, const Ws& w, const float* beta, const float* gate_w, const float* omega, const float* sumdD,
                             int n_sumdD, float* dbeta, float* dgate_w, float* dgate_b, float* domega, float* dqbar) {
  return {w.sg, w.qbar, gate_w, omega, sumdD, beta, n_sumdD, p.cfg.eps, p.cfg.bw_floor, p.cfg.features, p.cfg.batch, p.cfg.heads,
          p.cfg.head_dim, p.L1, p.cfg.gate_per_head, dbeta, dgate_w, dgate_b, domega, dqbar};
}
static void gate_backward_kernel(const Plan& p, const float* df, const GateBwdArgs& args, bool first, cudaStream_t st) {
  auto go = [&](auto kernel, int threads) {
    launch_after(kernel, dim3(p.cfg.heads + 2), dim3(threads), 0, st, df, args.sg, args.qbar, args.gate_w, args.omega, args.sumdD,
                 args.n_sumdD, args.beta, args.eps, args.bw_floor, args.m, args.B, args.H, args.dcols, args.L1, args.per_head,
                 args.dbeta, args.dgate_w, args.dgate_b, args.domega, args.dqbar, first);
  };
  if (p.cfg.batch <= 28) go(k_gate_backward<4>, 256);
  else go(k_gate_backward<16>, 1024);
}

// The two halves of launch_gate_backward, for sequence shards: this shard's band inner products (df, slabs x 16)
// and its sum of dD'; then, from the sums over all shards, the parameter gradients and d(qbar).
cudaError_t launch_band_sums(const Plan& p, const Ws& w, int band_blocks, int n_sumdD, float* df, float* sumdD_total,
                             cudaStream_t st, int* launches) {
  launch_after(k_band_reduce, dim3(p.slabs), dim3(256), 0, st, w.bands, p.slabs, band_blocks, p.cfg.levels, df);
  launch_after(k_sum_floats, dim3(1), dim3(kD), 0, st, w.sumdD, n_sumdD, sumdD_total);
  *launches += 2;
  return cudaGetLastError();
}
cudaError_t launch_gate_backward_from(const Plan& p, const Ws& w, const float* df, const float* sumdD_total,
                                      const float* beta, const float* gate_w, const float* omega, float* dbeta,
                                      float* dgate_w, float* dgate_b, float* domega, cudaStream_t st, int* launches) {
  gate_backward_kernel(p, df, gate_args(p, w, beta, gate_w, omega, sumdD_total, 1, dbeta, dgate_w, dgate_b, domega, w.dqbar), true, st);
  *launches += 1;
  return cudaGetLastError();
}

cudaError_t launch_gate_backward(const Plan& p, const Ws& w, int band_blocks, const float* beta, const float* gate_w,
                                 const float* omega, int n_sumdD, float* dbeta, float* dgate_w, float* dgate_b,
                                 float* domega, cudaStream_t st, int* launches) {
  float* df = w.dqbar + (size_t)p.slabs * kD;   // df lives behind dqbar in the same region
  launch_after(k_band_reduce, dim3(p.slabs), dim3(256), 0, st, w.bands, p.slabs, band_blocks, p.cfg.levels, df);
  gate_backward_kernel(p, df, gate_args(p, w, beta, gate_w, omega, w.sumdD, n_sumdD, dbeta, dgate_w, dgate_b, domega, w.dqbar), false, st);
  *launches += 2;
  return cudaGetLastError();
}

cudaError_t launch_gate_backward_dq(const Plan& p, const Ws& w, int band_blocks, const float* beta, const float* gate_w,
                                    const float* omega, int n_sumdD, float* dbeta, float* dgate_w, float* dgate_b, float* domega,
                                    void* dQ, int out_kind, cudaStream_t st, int* launches) {
  if (!haar_dq_takes_gate(p)) {
    const cudaError_t err = launch_gate_backward(p, w, band_blocks, beta, gate_w, omega, n_sumdD, dbeta, dgate_w, dgate_b, domega, st, launches);
    return err != cudaSuccess ? err
                              : launch_haar_filter_addvec(p, w.dQF, w.f, w.dqbar, 1.f / (float)p.cfg.seq_len, dQ, out_kind,
                                                          p.cfg.head_dim, st, launches);
  }
  if (!haar_dq_sums_bands(p)) {
    launch_after(k_band_reduce, dim3(p.slabs), dim3(256), 0, st, w.bands, p.slabs, band_blocks, p.cfg.levels, w.dqbar + (size_t)p.slabs * kD);
    *launches += 1;
  }
  return launch_haar_dq(p, w, gate_args(p, w, beta, gate_w, omega, w.sumdD, n_sumdD, dbeta, dgate_w, dgate_b, domega, nullptr), dQ, out_kind,
                        st, launches);
}

}  // namespace wersa
