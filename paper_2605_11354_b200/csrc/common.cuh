// Shared host/device helpers of the lite3r library (internal; the public surface is include/lite3r.h).
#pragma once

#include <cuda.h>
#include <cuda_runtime.h>
#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <cuda_fp8.h>
#include <stdint.h>

#include "lite3r.h"

namespace lite3r {

constexpr int kHeadDim = 64;
// One row of per-key-block linear-branch summaries: (H_j W)^T as [e][d] (4096 values) followed by z_j[d] (64).
constexpr int kSummaryRow = kHeadDim * kHeadDim + kHeadDim;

// Records a CUDA error for lite3r_last_cuda_error(); returns LITE3R_ERR_CUDA if err != cudaSuccess.
lite3r_status record_cuda(cudaError_t err);
// Counts one enqueued kernel launch and returns the launch's error state as a status.
lite3r_status after_launch();

// Benchmark stage timing: records event `idx` (0..7; stage s runs from event 2s to 2s+1) on `stream` when
// profiling is enabled.
void profile_mark(int idx, cudaStream_t stream);
bool profile_enabled();

// Number of SMs of the current device (looked up once per device).
lite3r_status sm_count(int* count);
// LITE3R_OK when the current device is a compute-capability 10.x part (the kernels are sm_100a code), else
// LITE3R_ERR_UNSUPPORTED (looked up once per device).
lite3r_status check_device();

// Sets a kernel's dynamic shared-memory limit, but only when this launch needs more than any earlier launch of that
// kernel on that device asked for (the limits already set are remembered per kernel and device; guarded by a mutex so
// that concurrent callers cannot leave a smaller limit behind).
lite3r_status ensure_smem_limit(const void* kernel, int bytes);
template <typename K>
lite3r_status ensure_dynamic_smem(K* kernel, int bytes) {
  return ensure_smem_limit(reinterpret_cast<const void*>(kernel), bytes);
}

// Enqueues a kernel as a programmatic dependent of the launch before it in the stream: it may start while that one is
// still running, and waits (griddepcontrol.wait) before it touches anything that one reads or writes.  Every kernel of
// the library that is launched this way lets its own successor start early as soon as its set-up is done.
// This holds wherever the launch stands: behind an event wait or a copy the stream orders it as an ordinary launch, and
// captured, the edges from every kernel that it follows, those of a join among them, become programmatic and its wait
// covers all of them.
// cluster: CTAs per thread-block cluster.
template <typename... Params, typename... Args>
lite3r_status launch_dependent_cluster(void (*kernel)(Params...), dim3 grid, int block, int smem_bytes, int cluster,
                                       cudaStream_t stream, const Args&... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = dim3(static_cast<unsigned>(block));
  cfg.dynamicSmemBytes = static_cast<size_t>(smem_bytes);
  cfg.stream = stream;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  attr[1].id = cudaLaunchAttributeClusterDimension;
  attr[1].val.clusterDim.x = static_cast<unsigned>(cluster);
  attr[1].val.clusterDim.y = attr[1].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = cluster > 1 ? 2 : 1;
  const lite3r_status st = record_cuda(cudaLaunchKernelEx(&cfg, kernel, static_cast<Params>(args)...));
  return st == LITE3R_OK ? after_launch() : st;
}
template <typename... Params, typename... Args>
lite3r_status launch_dependent(void (*kernel)(Params...), dim3 grid, int block, int smem_bytes, cudaStream_t stream,
                               const Args&... args) {
  return launch_dependent_cluster(kernel, grid, block, smem_bytes, 1, stream, args...);
}

inline int ceil_div(int a, int b) { return (a + b - 1) / b; }

struct Counts {
  int k_crit, k_marg, k_neg;
};
Counts class_counts(int nb, double crit, double neg);

// Value of an e4m3 code in units of 2^-9 (an exact integer, |v| <= 448 * 512).
__device__ __forceinline__ int e4m3_units(uint32_t code) {
  const int e = (code >> 3) & 0xF;
  const int m = code & 0x7;
  const int mag = e ? ((8 | m) << (e - 1)) : m;
  return (code & 0x80) ? -mag : mag;
}

// Decodes four packed e4m3 codes to fp32 (exact).
__device__ __forceinline__ void e4m3x4_to_float(uint32_t packed, float out[4]) {
  const __half2_raw lo = __nv_cvt_fp8x2_to_halfraw2(static_cast<__nv_fp8x2_storage_t>(packed & 0xFFFFu), __NV_E4M3);
  const __half2_raw hi = __nv_cvt_fp8x2_to_halfraw2(static_cast<__nv_fp8x2_storage_t>(packed >> 16), __NV_E4M3);
  const float2 a = __half22float2(__half2(lo));
  const float2 b = __half22float2(__half2(hi));
  out[0] = a.x;
  out[1] = a.y;
  out[2] = b.x;
  out[3] = b.y;
}

// Scale of a tile or row with this largest magnitude.
__device__ __forceinline__ float e4m3_scale(float amax) { return __fdiv_rn(__fadd_rn(amax, 1e-8f), 448.0f); }

// The e4m3 codes of x / scale, where x / scale is the correctly rounded fp32 quotient (so that codes equal those of a plain
// fp32 program bit for bit), saturated at +-448 and rounded to nearest even.  The quotient comes from the correctly
// rounded reciprocal r and corrections q + (x - q s) r, whose residual a fused multiply-add gives exactly (scales are at
// least 1e-8 / 448, so for every x whose code is not zero).  Two corrections make it correctly rounded: the first brings the
// product x r to within one ulp, after which the second is (P. Markstein, "Computation of elementary functions on the IBM
// RISC System/6000 processor", IBM J. Res. Dev. 34, 1990).  One is enough for the code, except for rare scales:
//   After one correction q = RN(x / s + h) with |h| <= 2^-47 |x / s|, so q and the quotient differ only when x / s lies within
//   h of the middle M of two neighbouring fp32 values, and their codes only when one of those two is a rounding boundary of
//   e4m3.  A boundary has at most 5 significant bits, so M as an integer of 25 (at a power of two 26) bits is
//   m 2^20 +- 1.  With x and s as integers X and S of 24 bits, |X 2^k - M S| (k >= 24) would be below 8.  It is not zero (M is
//   odd and longer than X), and modulo 2^20 it is +-S: the low 20 bits of S would lie within 8 of 0.  (When they are all
//   zero, S = t 2^20, |X 2^(k-20) - M t| would be below 1, so zero, which it cannot be.)
// close says that the scale is one of those (with a margin): the caller then takes the codes with two corrections.  Three
// packed multiply-adds per pair instead of five.
// Everything is computed for -x / scale, which keeps the sign of a zero through the corrections; flip undoes it.
struct E4m3Quotient {
  unsigned long long neg_r2, s2;
  bool close;
  static constexpr uint32_t kFlip = 0x80808080u;
  __device__ __forceinline__ explicit E4m3Quotient(float scale) {
    const float r = -__frcp_rn(scale);
    const uint32_t low = __float_as_uint(scale) & 0xFFFFFu;
    close = low != 0 && ((low + 16u) & 0xFFFFFu) <= 32u;
    asm("mov.b64 %0, {%1, %1};" : "=l"(neg_r2) : "f"(r));
    asm("mov.b64 %0, {%1, %1};" : "=l"(s2) : "f"(scale));
  }
  // two codes (low byte first), sign bits inverted
  template <bool kTwice>
  __device__ __forceinline__ uint32_t pair(unsigned long long x2) const {
    unsigned long long q, e;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(q) : "l"(x2), "l"(neg_r2));
#pragma unroll
    for (int i = 0; i < (kTwice ? 2 : 1); ++i) {
      asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(e) : "l"(q), "l"(s2), "l"(x2));
      asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(q) : "l"(e), "l"(neg_r2), "l"(q));
    }
    float2 y;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(y.x), "=f"(y.y) : "l"(q));
    return __nv_cvt_float2_to_fp8x2(y, __NV_SATFINITE, __NV_E4M3);
  }
  // four codes of two pairs; kTwice where close
  template <bool kTwice>
  __device__ __forceinline__ uint32_t four(unsigned long long a, unsigned long long b) const {
    return (pair<kTwice>(a) | (pair<kTwice>(b) << 16)) ^ kFlip;
  }
};

__device__ __forceinline__ float warp_max(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(0xFFFFFFFFu, v, o));
  return v;
}
// The same for values that are not negative (and not NaN), whose bits are ordered like they are: one instruction.
__device__ __forceinline__ float warp_max_abs(float v) {
  return __uint_as_float(__reduce_max_sync(0xFFFFFFFFu, __float_as_uint(v)));
}
__device__ __forceinline__ float warp_sum(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xFFFFFFFFu, v, o);
  return v;
}

// Kernel launchers (one per translation unit).  All enqueue on `stream` and return a status.
// One launch quantises `count` (1..3) source tensors of the same shape and dtype.
lite3r_status launch_quantize(const lite3r_tensor* const* x, const lite3r_fp8* out, int count, const lite3r_shape& s,
                              cudaStream_t stream);
void set_plan_variant(int variant);  // test hook, see lite3r_plan_variant
// beside_prior: the launch before it in the stream was the summary kernel of the same step, beside which it may run.
lite3r_status launch_plan(const lite3r_fp8& q, const lite3r_fp8& k, const lite3r_shape& s, const Counts& c,
                          const lite3r_plan& plan, bool beside_prior, cudaStream_t stream);

struct ForwardArgs {
  lite3r_fp8 q, k, v;
  const float* proj;
  long long proj_head_stride;
  lite3r_shape s;
  int phi;
  lite3r_plan plan;
  void* out;
  int out_dtype;
  long long out_stride_b, out_stride_h, out_stride_n;
  int linear_only;      // 1: the sparse branch is left out (the output is the linear branch through proj alone)
  int plan_inside;      // 1: the plan is built in the workspace from q/k column sums and the fractions below
  double crit, neg;
  void* workspace;
  size_t workspace_bytes;
  int* device_status;
};
struct AttentionLaunch {
  lite3r_shape shape;
  const uint8_t* q_codes;
  const uint8_t* k_codes;
  const float* q_scales;
  const float* k_scales;
  const float* v_scales;
  const float* k_norms;       // [tiles] largest norm of a key block's rows in units of the codes; NULL: not known
  const __half* v16;          // [tiles*Bs][64] dequantised V as fp16
  const __nv_bfloat16* g16;   // [tiles][64][64] aggregated projected summaries, [e][d]
  const float* zeta;          // [tiles][64]
  const int* crit_idx;
  int k_crit, k_marg, phi;
  void* out;
  int out_dtype;  // lite3r_dtype of the output
  long long out_stride_b, out_stride_h, out_stride_n;
  int* device_status;
  bool overlap_prior;  // the preceding launch in the stream produced only g16 and zeta: start before it has finished
};
lite3r_status launch_attention(const AttentionLaunch& a, cudaStream_t stream);
void set_attention_plain_stores(int on);  // test hook, see lite3r_attention_plain_stores

// Per-key-block summaries ((H_j W)^T | z_j) in bf16, one kSummaryRow-wide row per (b, h, key block).
// Clears *device_status.
lite3r_status launch_summary(const lite3r_fp8& k, const lite3r_fp8& v, const float* proj, long long proj_head_stride,
                             const lite3r_shape& s, int phi, __nv_bfloat16* hws, __half* v16, float* k_norms, int* device_status,
                             cudaStream_t stream);

// Marginal aggregation G_i = sum over marginal j of the summary rows, as a 0/1-mask GEMM on tensor cores.
// attention_ctas, steps: CTAs of the attention kernel that runs beside it and the steps each makes before it needs the sums
// (0: it does not run beside).
lite3r_status launch_aggregate(const __nv_bfloat16* hws, const signed char* cls, const lite3r_shape& s, int nb,
                               int attention_ctas, int steps, __nv_bfloat16* g16, float* zeta, int* device_status,
                               cudaStream_t stream);
constexpr int kAttentionCtasPerSm = 3;

// TMA descriptor of a row-major 2-D tensor [rows][inner] (row pitch in bytes, 0: inner * elem_bytes; a multiple of 16)
// with a box of box_inner x box_rows elements.  The make_tensor_map functions keep what they have encoded (a few hundred
// descriptors per calling thread): descriptors depend on their arguments only, and a caller that runs the same buffers
// again, or those of many layers in turn, gets a copy.
lite3r_status make_tensor_map_2d(CUtensorMap* map, CUtensorMapDataType type, int elem_bytes, const void* base, uint64_t inner,
                                      uint64_t rows, uint32_t box_inner, uint32_t box_rows, CUtensorMapSwizzle swizzle,
                                      uint64_t pitch_bytes = 0);
// The same for a 3-D tensor [planes][rows][inner] with a box of box_inner x box_rows x 1 (rows past the end of a plane
// are zero-filled, so a tile never runs into the next plane).
lite3r_status make_tensor_map_3d(CUtensorMap* map, CUtensorMapDataType type, int elem_bytes, const void* base, uint64_t inner,
                                      uint64_t rows, uint64_t planes, uint32_t box_inner, uint32_t box_rows,
                                      CUtensorMapSwizzle swizzle);
// Rank 4, extents dims[0..3], byte strides of dimensions 1..3 (multiples of 16), box of box[0..3] elements.
lite3r_status make_tensor_map_4d(CUtensorMap* map, CUtensorMapDataType type, const void* base, const uint64_t dims[4],
                                      const uint64_t strides_bytes[3], const uint32_t box[4], CUtensorMapSwizzle swizzle);

// The FP8 linear layer in front of the attention (linear.cu).
lite3r_status launch_rowquant(const void* x, int dtype, long long row_stride, int rows, int cols, uint8_t* codes,
                              float* scales, cudaStream_t stream);
lite3r_status launch_linear_fp8(const uint8_t* x_codes, const float* x_scales, const uint8_t* w_codes,
                                const float* w_scales, const float* bias, int rows, int d_in, int d_out, void* y,
                                int y_dtype, long long y_stride, int* device_status, cudaStream_t stream);
lite3r_status launch_qkv_project(const uint8_t* x_codes, const float* x_scales, const uint8_t* w_codes,
                                 const float* w_scales, const float* bias, const lite3r_shape& s, int d_model,
                                 const lite3r_fp8* out, int* device_status, cudaStream_t stream);

// Training side of the linear-branch projection (train.cu).
size_t train_workspace_bytes(const lite3r_shape& s);
lite3r_status launch_mse_distill(const void* student, const void* teacher, int dtype, size_t count, __nv_bfloat16* grad,
                                 double* loss, double* partials, cudaStream_t stream);
lite3r_status launch_proj_lin_backward(const __nv_bfloat16* o_lin, const __nv_bfloat16* d_out, const lite3r_shape& s,
                                       float* d_w, float* partials, int* device_status, cudaStream_t stream);

lite3r_status launch_wait_expiry_probe(int* status, unsigned long long limit_ns, cudaStream_t stream);
size_t forward_workspace_bytes(const lite3r_shape& s, const Counts& c, bool plan_inside = false);
// byte offsets of the workspace's parts: summaries, aggregates, zeta, fp16 V, class bytes, critical lists
void forward_workspace_offsets(const lite3r_shape& s, const Counts& c, bool plan_inside, size_t* offsets);
// phases: 1 = the plan-independent first part, 2 = the rest, 3 = the whole forward
lite3r_status launch_forward(const ForwardArgs& a, int phases, cudaStream_t stream);

}  // namespace lite3r
