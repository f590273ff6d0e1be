// Shared declarations of the WERSA CUDA library: the host-side plan, the workspace layout and
// the launch functions each translation unit exports to the C-ABI layer (api.cu).
#pragma once
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stddef.h>
#include <stdint.h>

#include "../../include/wersa.h"

namespace wersa {

constexpr int kD = 64;           // widest head; S', z' images, partial sums and q-bar of narrower ones have zero columns up to it
constexpr int kGroupFeatures = 256;   // widest feature map of one kernel launch; wider maps run in groups
constexpr int kMaxLevels = 8;    // Haar levels supported: block of 2^8 = 256 tokens
constexpr int kHaarTile = 256;   // tokens per Haar tile (>= 2^kMaxLevels)
constexpr int kBandVals = 16;    // per-tile band inner products kept by the Haar backward

// Host-side plan: problem sizes, chunking and byte offsets into the caller's workspace.
struct Plan {
  wersa_config cfg;
  int slabs;          // B*H
  int sms;            // streaming multiprocessors of cfg.device
  int L1;             // levels + 1
  bool bf16;          // storage type of Q,K,V,W,O,dO
  bool grad_bf16;     // storage type of dQ,dK,dV
  bool use_tc;        // bf16 tcgen05 forward kernels
  bool with_backward;
  bool dpad;          // cfg.head_dim < 64
  int groups;         // feature groups of kGroupFeatures (1 when cfg.features <= 256)
  // mean pool
  int qchunks, qchunk_rows;
  int qcluster, qcluster_rows;   // the same where the chunks of a slab are one cluster; 0: they are not
  // haar tiles
  int htiles;
  // fp32 FFMA key-side / backward query-side split of the sequence
  int schunks, schunk_rows;    // chunks per slab, tokens per chunk
  bool simt_small;             // the 16-token tile (see make_plan and WERSA_SIMT_TILE)
  // tcgen05 key-side split
  int tchunks, tchunk_blocks;  // chunks per slab, 256-token blocks per chunk
  int tqchunks, tqchunk_blocks;  // the same for the query side of the forward
  bool use_x;         // fp32 forward on the tensor cores (tc_f32.cu)
  int xchunks, xchunk_tiles;   // its chunks per slab, 128-token tiles per chunk
  bool use_xb;        // fp32 backward on them too: chunks and tiles of its gradient kernels, CTAs of its first pass
  int xbchunks, xbchunk_tiles, xprep;
  int small_tokens, small_blocks;   // bf16 forward in one launch (small.cu): tokens of a thread block, blocks of a slab; 0: not
  int filter_tokens;  // FFMA forward: mean pool, gate and filter in one launch (small.cu): tokens of a thread block; 0: in two
  int bctas;          // tcgen05 backward: CTAs that share the list of all 128-token tiles
  // workspace offsets (bytes)
  size_t off_status, off_counters, status_bytes, off_qpart, off_qbar, off_sg, off_f, off_spart, off_zpart, off_S, off_z,
      off_Sbf, off_Wt, off_dS, off_dz, off_sumdD, off_bands, off_dqbar, off_QF, off_KF, off_dQF,
      off_dKF, off_dSbf, off_KF3, off_QF3, off_Slo, off_Simg, off_Og, off_den, off_Dtot, off_shardtot, off_V3, off_dO3, off_xO, off_xden, off_xinv, off_xc, off_xshare, total;
};

// Fills `p` from `cfg`; returns WERSA_OK, WERSA_ERR_INVALID_ARG or WERSA_ERR_UNSUPPORTED.
wersa_status make_plan(const wersa_config& cfg, Plan* p);

struct Ws {   // resolved workspace pointers
  int* status;
  int* seen;       // fp32 on the tensor cores: not 0 where T_f(Q) [0], T_f(K) [1] hold a value that is not finite
  int* counters;   // arrival counters (slabs + batch + slabs ints), zero between launches
  float *qpart, *qbar, *sg, *f, *spart, *zpart, *S, *z, *dS, *dz, *sumdD, *bands, *dqbar;
  float *xO, *xden, *xinv, *xc, *xshare;   // fp32 on the tensor cores: O and D'_g for the backward, 1 / D and -dO.O per token, shares of N'
  __nv_bfloat16 *Sbf, *Wt, *dSbf, *KF3, *QF3, *V3, *dO3, *Slo;   // Slo = bf16(S' - bf16(S')), built by the backward
  uint8_t* Simg;   // [S' | z' | 0]^T operand images of the query-side kernel, one per slab (see simg_offset)
  float *QF, *KF, *dQF, *dKF;
  // features > 256: per-group outputs and denominators
  void* Og;
  float* den;
  float* shardtot;   // sequence shards, backward: this shard's sum of dD' (one float)
  float* Dtot;   // backward with feature groups: the whole map's denominator per token, then dD' per token
};
Ws resolve(const Plan& p, void* workspace);

// ---- gate.cu -------------------------------------------------------------------------------
// What k_qmean_gate's launches as clusters need, once for a context (on its device).
void prepare_qmean_gate(const Plan& p);
// Partial column sums of Q over row chunks, then qbar, sigmoid(u) and f per slab (Eqs. 1-3).
// With W != nullptr the second launch also leaves the bf16 transpose of W (m x 64) in w.Wt.
// cols: columns of Q as stored (64, or the head dimension when Q comes unpadded; then gate_w has cols rows
// per head and W cols rows).
cudaError_t launch_qmean_gate(const Plan& p, const Ws& w, const void* Q, const float* gate_w,
                              const float* gate_b, const float* omega, const void* W, int cols, cudaStream_t st,
                              int* launches);
// Sequence shards: column sums of this shard's Q (q-bar times the shard's length), and the gate from the
// sums of all shards and the whole sequence's length (writes w.qbar, w.sg, w.f).
cudaError_t launch_shard_qsum(const Plan& p, const Ws& w, float* qsum, cudaStream_t st, int* launches);
cudaError_t launch_gate_from_sums(const Plan& p, const Ws& w, const float* qsum, long long n_total,
                                  const float* gate_w, const float* gate_b, const float* omega, int cols,
                                  cudaStream_t st, int* launches);
// band_blocks: partials per slab and tensor in w.bands (haar_band_blocks).
cudaError_t launch_band_sums(const Plan& p, const Ws& w, int band_blocks, int n_sumdD, float* df, float* sumdD_total,
                             cudaStream_t st, int* launches);
cudaError_t launch_gate_backward_from(const Plan& p, const Ws& w, const float* df, const float* sumdD_total,
                                      const float* beta, const float* gate_w, const float* omega, float* dbeta,
                                      float* dgate_w, float* dgate_b, float* domega, cudaStream_t st, int* launches);
// Gate backward: band inner products -> df -> domega, dgate_b, dgate_w, dqbar; dbeta.
cudaError_t launch_gate_backward(const Plan& p, const Ws& w, int band_blocks, const float* beta, const float* gate_w,
                                 const float* omega, int n_sumdD, float* dbeta, float* dgate_w, float* dgate_b,
                                 float* domega, cudaStream_t st, int* launches);

// Gate backward and dQ, in one launch or up to three (see launch_haar_dq).
cudaError_t launch_gate_backward_dq(const Plan& p, const Ws& w, int band_blocks, const float* beta, const float* gate_w,
                                    const float* omega, int n_sumdD, float* dbeta, float* dgate_w, float* dgate_b, float* domega,
                                    void* dQ, int out_kind, cudaStream_t st, int* launches);

// Mean pool + gate with their scratch in a file-scope device array (no caller workspace).
cudaError_t static_scratch_address(int device, float** out);
size_t static_scratch_capacity_floats();      // floats available to the partial sums and sigmoids
size_t static_scratch_counter_capacity();     // ints reserved for the arrival counters
size_t static_scratch_floats_needed(const Plan& p);
size_t static_scratch_counters_needed(const Plan& p);
cudaError_t launch_qmean_gate_static(const Plan& p, float* scratch, const void* Q, const float* gate_w,
                                     const float* gate_b, const float* omega, float* qbar, float* f,
                                     cudaStream_t st);

// ---- haar.cu -------------------------------------------------------------------------------
// d: columns of the tensors as stored (a multiple of 8, at most 64).  in_kind/out_kind: 0 = float, 1 = bf16 (float input: float output).
// Whether the FFMA key side may be placed early behind a filter of `ctas` CTAs.
bool place_key_side_early(const Plan& p, unsigned ctas);
// XF = T_f(X), and with X2 also XF2 = T_f(X2) in the same launch.
cudaError_t launch_haar_filter(const Plan& p, const void* X, int in_kind, const float* f, void* XF, const void* X2,
                               void* XF2, int out_kind, int d, bool inputs_ready, cudaStream_t st, int* launches);
// XF3 = T_f(X) (X bf16) as three bf16 planes hi, mid, lo (each slabs x n x head_dim) whose sum is the fp32 result;
// with X2 also XF3_2 from X2 in the same launch, with split_S also w.Slo = bf16(w.S - w.Sbf).
cudaError_t launch_haar_filter_split3(const Plan& p, const Ws& w, const void* X, __nv_bfloat16* XF3, const void* X2,
                                      __nv_bfloat16* XF3_2, bool split_S, cudaStream_t st, int* launches);
// w.QF3 = T_f(Q), w.KF3 = T_f(K) and, of fp32 tensors, w.V3 = V as planes; with keep also w.QF and w.KF.
cudaError_t launch_f32_planes(const Plan& p, const Ws& w, const void* Q, const void* K, const void* V, bool keep,
                              cudaStream_t st, int* launches);
// dX = T_f(G) + vec[slab] * vec_scale on every row (G fp32, vec = slabs x 64 floats).
cudaError_t launch_haar_filter_addvec(const Plan& p, const float* G, const float* f, const float* vec,
                                      float vec_scale, void* dX, int out_kind, int d, cudaStream_t st, int* launches);
// The same with the row vector d q-bar / n worked out in the pass, and with the gradients of the gate's parameters and of beta: where
// haar_dq_takes_gate; from the partial band inner products themselves where haar_dq_sums_bands, else behind launch_band_reduce.
struct GateBwdArgs;
bool haar_dq_takes_gate(const Plan& p);
bool haar_dq_sums_bands(const Plan& p);
cudaError_t launch_haar_dq(const Plan& p, const Ws& w, const GateBwdArgs& args, void* dQ, int out_kind, cudaStream_t st, int* launches);
// dX = T_f(G) (G fp32) and the band inner products of (G, X), one partial for each of haar_band_blocks(p, d)
// CTAs per slab, into bands[which]; dX == nullptr: only the band inner products.  X2 / G2 / dX2: the other tensor
// (bands[1 - which]) in the same launch, after the first, or null.
int haar_band_blocks(const Plan& p, int d);
cudaError_t launch_haar_backward(const Plan& p, const Ws& w, int which, const void* X, const float* G, void* dX,
                                 const void* X2, const float* G2, void* dX2, int in_kind, int out_kind, int d,
                                 cudaStream_t st, int* launches);

// ---- simt.cu -------------------------------------------------------------------------------
cudaError_t launch_simt_kside(const Plan& p, const Ws& w, const void* V, const void* W,
                              cudaStream_t st, int* launches);
// S = sum_chunks spart, z = sum_chunks zpart in chunk order (also used for dS, dz).  first: the first kernel of its pass, and
// the next one fetches arguments ahead of its wait (see launch_behind).
cudaError_t launch_reduce_partials(const Plan& p, const float* spart, const float* zpart, int chunks,
                                   float* S, float* z, __nv_bfloat16* Sbf, uint8_t* Simg, cudaStream_t st,
                                   int* launches, bool first = false);
// The same for the segments the tensor-core backward leaves (slot CTA + slab for every CTA that has tiles of the
// slab): dS, dz and the bf16 image of dS.
cudaError_t launch_reduce_segments(const Plan& p, const Ws& w, cudaStream_t st, int* launches);
cudaError_t launch_simt_qside(const Plan& p, const Ws& w, const void* W, const float* beta, void* O,
                              cudaStream_t st, int* launches);
cudaError_t launch_simt_bwd_qside(const Plan& p, const Ws& w, const void* W, const float* beta,
                                  const void* dO, cudaStream_t st, int* launches);
cudaError_t launch_simt_bwd_kside(const Plan& p, const Ws& w, const void* V, const void* W, void* dV,
                                  cudaStream_t st, int* launches);

// ---- tc_f32.cu -----------------------------------------------------------------------------
// fp32 on the tensor cores.  Forward: partial S', z' (p.xchunks per slab) from w.KF3 and w.V3; O from w.QF3, w.S and w.z,
// with a backward also w.xO and w.xden.  Backward: dO as planes and what the division leaves per token; dQ_F, partial dS',
// dz'; dK_F and dV.
cudaError_t launch_tcx_kside(const Plan& p, const Ws& w, const void* V, const void* W, cudaStream_t st, int* launches);
cudaError_t launch_tcx_qside(const Plan& p, const Ws& w, const void* W, const float* beta, void* O, cudaStream_t st, int* launches);

cudaError_t launch_tcx_bwd_prep(const Plan& p, const Ws& w, const void* dO, const float* beta, cudaStream_t st, int* launches);
cudaError_t launch_tcx_bwd_qside(const Plan& p, const Ws& w, const void* W, const void* dO, cudaStream_t st, int* launches);
cudaError_t launch_tcx_bwd_kside(const Plan& p, const Ws& w, const void* V, const void* W, void* dV, cudaStream_t st, int* launches);

// ---- tc_fwd.cu -----------------------------------------------------------------------------
// Both read the raw bf16 tensors and apply the Haar filter (coefficients from w.f) on chip.  first: the first kernel of its
// pass (see launch_behind).
cudaError_t launch_tc_kside(const Plan& p, const Ws& w, const void* K, const void* V, cudaStream_t st, int* launches,
                            bool first = false);
// den != nullptr (features == 256 only): also leaves every token's denominator in den[slab * n + token].
cudaError_t launch_tc_qside(const Plan& p, const Ws& w, const void* Q, const float* beta, void* O, float* den,
                            cudaStream_t st, int* launches);

// ---- small.cu ------------------------------------------------------------------------------
// The whole forward of slabs of p.small_blocks * p.small_tokens tokens in one launch: O (with several feature groups w.Og and
// w.den), f, q-bar, S', z', and what a backward reads beside them.
cudaError_t launch_small_forward(const Plan& p, const Ws& w, const void* Q, const void* K, const void* V, const void* W,
                                 const float* beta, const float* gate_w, const float* gate_b, const float* omega, void* O,
                                 cudaStream_t st, int* launches);
// Self-test of its waits that run out.
bool selftest_small_supported(const Plan& p);
cudaError_t launch_selftest_small(const Plan& p, const Ws& w, int loss, const void* Q, const void* K, const void* V, const void* W,
                                  const float* beta, const float* omega, void* O, cudaStream_t st);
// Mean pool, gate, and w.QF = T_f(Q), w.KF = T_f(K), in one launch (p.filter_tokens).
cudaError_t launch_small_filter(const Plan& p, const Ws& w, const void* Q, const void* K, const float* gate_w, const float* gate_b,
                                const float* omega, cudaStream_t st, int* launches);
// Decides p->small_tokens, p->small_blocks and p->filter_tokens (asks the device, which is current).
void choose_small_forward(Plan* p);

// ---- tc_bwd.cu -----------------------------------------------------------------------------
// Key-side backward on the tensor cores: dV and dK_F from K_F as three bf16 planes, V, the bf16 dS' image
// (w.dSbf), dz' (w.dz) and the bf16 W^T image (w.Wt).
// Query-side backward on the tensor cores: dQ_F, the partials of dS', dz' (w.spart, w.zpart: see
// launch_reduce_segments) and p.bctas partial sums of dD' (w.sumdD), from Q_F as three bf16 planes, dO, the bf16 S'
// image (w.Sbf) and its low-order part, z' (w.z) and the bf16 W^T image.
// Feature groups (p.cfg.features == 256 as one group of a wider map): den_ext / dd_ext hold the whole map's
// denominator and dD' per token (slabs x n floats each), `add` makes dQ_F (dV, dK_F) accumulate.
cudaError_t launch_tc_bwd_qside(const Plan& p, const Ws& w, const void* QF3, const float* beta, const void* dO,
                                const float* den_ext, const float* dd_ext, bool add, cudaStream_t st, int* launches);
cudaError_t launch_tc_bwd_kside(const Plan& p, const Ws& w, const void* KF3, const void* V, void* dV, bool add,
                                cudaStream_t st, int* launches);


// ---- glue.cu -------------------------------------------------------------------------------
// O = sum_g Og[g] * den[g] / sum_g den[g] per token (Og: groups x tokens x cols, den: groups x tokens; bf16).
cudaError_t launch_combine_groups(const void* Og, const float* den, void* O, size_t tokens, int groups, int cols,
                                  cudaStream_t st, int* launches);
// Backward of the combination: per token the whole map's denominator D = sum_g den_g / r (r = the filter
// stage's factor carried by the forward's denominators, from f) and dD' = -(dO . O) / D with
// O = sum_g Og den_g / sum_g den_g.  Og and dO have d columns.
cudaError_t launch_group_bwd_prep(const void* Og, const float* den, const void* dO, int d, const float* f, int n, int L1,
                                  size_t tokens, int groups, float* Dtot, float* dDtot, cudaStream_t st,
                                  int* launches);

// ---- selftest.cu ---------------------------------------------------------------------------
// One CTA whose bounded wait runs out after limit_ns: sets the status word; observed[0] = abort flag,
// observed[1], observed[2] = whether the two roles' waits succeeded (both must read 0).
cudaError_t launch_selftest_wait(const Ws& w, unsigned long long limit_ns, int* observed, cudaStream_t st);

// ---- operand image of the query-side second contraction --------------------------------------
// The query-side kernel multiplies the features by [S' | z' | 0] (m x 80) as a K-major bf16 operand: per
// slab, m / 64 blocks of 80 rows x 128 bytes -- rows 0-63 are the columns of S', row 64 is z', rows 65-79
// are zero, and a row holds 64 consecutive features in the 128-byte swizzle the tensor core reads (16-byte
// chunk j of row r sits at chunk j ^ (r & 7)).  Whoever produces S' and z' leaves this image in global
// memory in exactly that byte order, so that the kernel fetches it with one bulk copy.
constexpr int kSimgRows = 80;
constexpr size_t kSimgBlockBytes = kSimgRows * 128;
__host__ __device__ inline size_t simg_bytes(int m) { return (size_t)(m / 64) * kSimgBlockBytes; }
// byte offset of (feature f, row r) inside a slab's image
__device__ __forceinline__ size_t simg_offset(int f, int r) {
  return (size_t)(f >> 6) * kSimgBlockBytes + (size_t)r * 128 + (size_t)((((f & 63) >> 3) ^ (r & 7)) << 4) + (f & 7) * 2;
}

// Two fp32 values in one 64-bit register: the packed add / multiply / fma of sm_100 issue one
// instruction for both halves.
typedef unsigned long long f32x2;
__device__ __forceinline__ f32x2 pk2(float lo, float hi) {
  f32x2 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
  return r;
}
__device__ __forceinline__ void upk2(f32x2 v, float& lo, float& hi) {
  asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v));
}
__device__ __forceinline__ f32x2 mul2(f32x2 a, f32x2 b) {
  f32x2 r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ f32x2 fma2(f32x2 a, f32x2 b, f32x2 c) {
  f32x2 r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
  return r;
}
__device__ __forceinline__ f32x2 add2(f32x2 a, f32x2 b) {
  f32x2 r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ float sum2(f32x2 v) {
  float lo, hi;
  upk2(v, lo, hi);
  return lo + hi;
}

// Launch as a programmatic dependent of the work before it in the stream.  Ordering and visibility are those of a plain
// launch, since the kernel writes nothing and reads nothing of that work before wait_for_stream_predecessor(); only the
// placement of its CTAs, and what they set up or fetch ahead of the wait, overlaps the end of that work.
// What may be fetched ahead of the wait: what a kernel wrote behind which, and in front of this one, there is a kernel of the
// same pass that lets its successor start only after its own wait, or at its end (call it closed).  Not every kernel is:
// k_reduce_partials, k_band_reduce and k_gate_backward (unless first) let the next one start at once, and that one then runs
// beside the kernel in front of THEM.  So the arguments of a call may be fetched ahead behind the first closed kernel of the
// pass (k_qmean_gate in the forward, whatever comes first in a backward; dQ_F by the last pass of a backward: k_haar_backward is
// closed), and the first kernel of a pass fetches nothing: what stands in front of it may be the end of another pass, such
// as a gate backward beside a k_haar_backward that still writes dQ.  Kernels that fetch arguments ahead and may be the first
// of a pass, or stand behind a first one that is not closed, are told: overlap = false is a plain launch.
// Where work stands ahead of the wait, results of the kernel in front are read with load_after_wait (or __ldcg where the L1
// has no use for them), not through a const __restrict__ pointer: such a load counts as free of order with anything, and the
// compiler did move the row vector of dQ above the wait.
template <typename... KArgs, typename... Args>
inline cudaError_t launch_behind(bool overlap, void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t st,
                                 Args&&... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = overlap ? 1 : 0;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kernel, KArgs(args)...);
}
template <typename... KArgs, typename... Args>
inline cudaError_t launch_after(void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, Args&&... args) {
  return launch_behind(true, kernel, grid, block, smem, st, args...);
}
__device__ __forceinline__ void wait_for_stream_predecessor() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ float load_after_wait(const float* p) {
  float v;
  asm volatile("ld.global.f32 %0, [%1];" : "=f"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ float4 load4_after_wait(const float* p) {
  float4 v;
  asm volatile("ld.global.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "l"(p) : "memory");
  return v;
}
// The kernel behind this one may be placed once every CTA of this grid has got here (or has ended).  Not where that kernel
// is bound by memory and several of its CTAs share an SM: placed as the SMs fall free, they gather on some and all start at
// once, and the passes of the first ones stay in step (the mean pool behind the query side of 1 x 8 x 131072: 16 us more a
// forward; k_haar_backward behind the key side of 4 x 8 x 16384: 160 instead of 105 us).
__device__ __forceinline__ void let_stream_successor_start() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

// ---- device helpers ------------------------------------------------------------------------
__device__ __forceinline__ float to_f32(float x) { return x; }
__device__ __forceinline__ float to_f32(__nv_bfloat16 x) { return __bfloat162float(x); }
template <typename T> __device__ __forceinline__ T from_f32(float x);
template <> __device__ __forceinline__ float from_f32<float>(float x) { return x; }
template <> __device__ __forceinline__ __nv_bfloat16 from_f32<__nv_bfloat16>(float x) {
  return __float2bfloat16_rn(x);
}

// A finite value inside the range of bf16, whose largest is 2^128 - 2^120 (what is above it rounds to infinity); infinities and
// NaN as they are.
__device__ __forceinline__ float bf16_range(float x) {
  const float most = __uint_as_float(0x7F7F0000u);
  return fabsf(x) < INFINITY ? fminf(fmaxf(x, -most), most) : x;
}
// Not 0 where one of two packed bf16 has an exponent of all ones: infinity, NaN, or what rounded to infinity.
__device__ __forceinline__ uint32_t full_exponents(uint32_t w) { return ((w & 0x7F807F80u) + 0x00800080u) & 0x80008000u; }

// Loads 8 consecutive elements (16-byte aligned for bf16, 32-byte for float) as floats.
__device__ __forceinline__ void load8(const float* p, float (&v)[8]) {
  float4 a = *reinterpret_cast<const float4*>(p);
  float4 b = *reinterpret_cast<const float4*>(p + 4);
  v[0] = a.x; v[1] = a.y; v[2] = a.z; v[3] = a.w;
  v[4] = b.x; v[5] = b.y; v[6] = b.z; v[7] = b.w;
}
__device__ __forceinline__ void load8(const __nv_bfloat16* p, float (&v)[8]) {
  uint4 raw = *reinterpret_cast<const uint4*>(p);
  const uint32_t u[4] = {raw.x, raw.y, raw.z, raw.w};
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    v[2 * i] = __uint_as_float(u[i] << 16);
    v[2 * i + 1] = __uint_as_float(u[i] & 0xFFFF0000u);
  }
}
// The same loads with the streaming (evict-first) cache hint, for data that is read once: the lines make room
// for themselves in L2 instead of pushing out what other kernels left there (dirty output lines of the step
// before are then written back later, under kernels that do not need the DRAM bandwidth).
__device__ __forceinline__ void load8_stream(const float* p, float (&v)[8]) {
  const float4 a = __ldcs(reinterpret_cast<const float4*>(p));
  const float4 b = __ldcs(reinterpret_cast<const float4*>(p + 4));
  v[0] = a.x; v[1] = a.y; v[2] = a.z; v[3] = a.w;
  v[4] = b.x; v[5] = b.y; v[6] = b.z; v[7] = b.w;
}
__device__ __forceinline__ void load8_stream(const __nv_bfloat16* p, float (&v)[8]) {
  const uint4 raw = __ldcs(reinterpret_cast<const uint4*>(p));
  const uint32_t u[4] = {raw.x, raw.y, raw.z, raw.w};
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    v[2 * i] = __uint_as_float(u[i] << 16);
    v[2 * i + 1] = __uint_as_float(u[i] & 0xFFFF0000u);
  }
}
__device__ __forceinline__ void store8(float* p, const float (&v)[8]) {
  *reinterpret_cast<float4*>(p) = make_float4(v[0], v[1], v[2], v[3]);
  *reinterpret_cast<float4*>(p + 4) = make_float4(v[4], v[5], v[6], v[7]);
}
__device__ __forceinline__ void store8(__nv_bfloat16* p, const float (&v)[8]) {
  uint4 raw;
  uint32_t* u = reinterpret_cast<uint32_t*>(&raw);
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    __nv_bfloat162 h = __floats2bfloat162_rn(v[2 * i], v[2 * i + 1]);
    u[i] = *reinterpret_cast<uint32_t*>(&h);
  }
  *reinterpret_cast<uint4*>(p) = raw;
}

}  // namespace wersa
