// The FP8 linear layer in front of the attention (Algorithm 2 "FP8 fake-quantised linear" in its deployed form; Eq. 2):
//   quantise_rows   per-token (activations) / per-output-row (weights) scaled e4m3 quantiser
//   linear_fp8      y = x_q W_q^T + b on tcgen05 (e4m3 x e4m3, fp32 accumulation in TMEM), scales applied in the epilogue
//   qkv_project     the same product for the qkv projection, with the block quantiser of the attention path fused into
//                   its epilogue: Q, K and V leave the kernel as e4m3 codes + per-(b, h, token-block) scales + column
//                   sums in the library's own layout, so the separate quantiser pass over Q, K, V disappears.
//
// GEMM kernel: persistent CTAs (one per SM) over 128 x 256 output tiles (128 tokens x 256 output columns = four heads
// of the projection), or pairs of CTAs over tiles of 256 x 256 (cta_group::2 products that read half of the weights from
// either CTA).  The operand bytes from L2 bound the product: 43968 x 1024 x 1024 took 54.5 us by single CTAs and takes 50 us
// by pairs, with the tensor pipe busy for 46 % of it (in a long run of whole layers, under the power cap at 1.69 GHz, 51 us).  Warp 0 = TMA producer (A = activation codes, B = weight codes, both
// K-major rows of 128 bytes, 128B swizzle, ring of three or four stages), warp 1 = MMA issuer (four kind::f8f6f4 products
// of K = 32 per stage into one of two accumulators), warps 4-19 = four epilogue warpgroups, one per 64 columns of the tile
// (thread = token row = TMEM lane; two passes over the accumulator so that a row of 64 values never has to stay in
// registers: the first scales, adds the bias, takes the maximum and writes the values back, the second makes the codes).
// The products of the next tile run under the epilogue of this one.  With the block quantiser the epilogue is what bounds
// the kernel: 10992 x 1024 x 3072 in 45 us (49 us while both passes scaled the products and a quotient took two
// corrections).
// Every mbarrier wait is bounded; on expiry the CTA sets *device_status and its roles leave their loops.
#include <algorithm>
#include <type_traits>

#include "common.cuh"
#include "sm100.cuh"

namespace lite3r {

namespace {

using namespace sm100;

// ------------------------------------------------------------------------------------------------ row quantiser
// Eight values as they lie in memory, their conversion to fp32 and the running maximum of their magnitudes (for bf16 on
// packed pairs: the maximum of bf16 values is one of them).
template <typename SrcT>
struct Eight;
template <>
struct Eight<__nv_bfloat16> {
  uint4 w;
  using Max = __nv_bfloat162;
  __device__ __forceinline__ void load(const __nv_bfloat16* p) { w = __ldg(reinterpret_cast<const uint4*>(p)); }
  __device__ __forceinline__ void clear() { w = make_uint4(0u, 0u, 0u, 0u); }
  static __device__ __forceinline__ Max zero() { return __float2bfloat162_rn(0.f); }
  __device__ __forceinline__ Max max_with(Max m) const {
    const uint32_t x[4] = {w.x, w.y, w.z, w.w};
#pragma unroll
    for (int i = 0; i < 4; ++i) m = __hmax2(m, __habs2(*reinterpret_cast<const __nv_bfloat162*>(&x[i])));
    return m;
  }
  static __device__ __forceinline__ float top(Max m) { return fmaxf(__low2float(m), __high2float(m)); }
  __device__ __forceinline__ void values(float v[8]) const {
    const uint32_t x[4] = {w.x, w.y, w.z, w.w};
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      v[2 * i] = __uint_as_float(x[i] << 16);
      v[2 * i + 1] = __uint_as_float(x[i] & 0xFFFF0000u);
    }
  }
};
template <>
struct Eight<float> {
  float4 a, b;
  using Max = float;
  __device__ __forceinline__ void load(const float* p) {
    a = __ldg(reinterpret_cast<const float4*>(p));
    b = __ldg(reinterpret_cast<const float4*>(p + 4));
  }
  __device__ __forceinline__ void clear() { a = b = make_float4(0.f, 0.f, 0.f, 0.f); }
  static __device__ __forceinline__ Max zero() { return 0.f; }
  __device__ __forceinline__ Max max_with(Max m) const {
    m = fmaxf(fmaxf(m, fabsf(a.x)), fmaxf(fabsf(a.y), fmaxf(fabsf(a.z), fabsf(a.w))));
    return fmaxf(fmaxf(m, fabsf(b.x)), fmaxf(fabsf(b.y), fmaxf(fabsf(b.z), fabsf(b.w))));
  }
  static __device__ __forceinline__ float top(Max m) { return m; }
  __device__ __forceinline__ void values(float v[8]) const {
    v[0] = a.x; v[1] = a.y; v[2] = a.z; v[3] = a.w;
    v[4] = b.x; v[5] = b.y; v[6] = b.z; v[7] = b.w;
  }
};

// Scale of a row and the codes of eight of its values.
struct RowScale {
  float scale;
  E4m3Quotient quotient;
  __device__ __forceinline__ explicit RowScale(float amax)
      : scale(e4m3_scale(amax)), quotient(scale) {}
  template <bool kTwice>
  __device__ __forceinline__ uint2 eight(const float v[8]) const {
    return make_uint2(quotient.four<kTwice>(pack_f32x2(v[0], v[1]), pack_f32x2(v[2], v[3])),
                      quotient.four<kTwice>(pack_f32x2(v[4], v[5]), pack_f32x2(v[6], v[7])));
  }
  __device__ __forceinline__ uint2 codes(const float v[8]) const { return quotient.close ? eight<true>(v) : eight<false>(v); }
};

// One warp per row.  Rows of up to 256 kSegs values stay in registers as they lie in memory (all requested before the
// first is used), and bf16 rows of that length are requested one row ahead, so that a warp's loads run under the
// arithmetic of the row before; longer rows are read twice (maximum, then codes; the second read comes from L1 / L2).
// Bound by HBM: 43968 x 1024 bf16 values (135 MB) in 18.7 us with the input partly in L2 (21.5 us with two corrections per
// quotient, 31 us while a third of the groups of 256 values went through a division), 29 us after L2 has been flushed, and
// 32 us, 4.2 TB/s, in a run of layers whose GEMM leaves its 90 MB result in L2.
template <typename SrcT, int kSegs>
__global__ void __launch_bounds__(256) rowquant_kernel(const SrcT* __restrict__ x, long long row_stride, int rows, int cols,
                                                       uint8_t* __restrict__ codes, float* __restrict__ scales) {
  wait_for_prior_grid();
  launch_dependents();
  const int lane = threadIdx.x & 31;
  const int warps = (gridDim.x * blockDim.x) >> 5;
  const int segs = cols >> 3;
  int row = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  if constexpr (kSegs > 0) {
    constexpr bool kAhead = sizeof(SrcT) == 2;
    Eight<SrcT> next[kSegs];
    auto fetch = [&](int r) {
      const SrcT* src = x + static_cast<long long>(r) * row_stride + lane * 8;
#pragma unroll
      for (int q = 0; q < kSegs; ++q) {
        if (lane + 32 * q < segs) next[q].load(src + 256 * q);
        else next[q].clear();
      }
    };
    if (row < rows) fetch(row);
    for (; row < rows; row += warps) {
      if (!kAhead) fetch(row);
      Eight<SrcT> cur[kSegs];
      typename Eight<SrcT>::Max m = Eight<SrcT>::zero();
#pragma unroll
      for (int q = 0; q < kSegs; ++q) {
        cur[q] = next[q];
        m = cur[q].max_with(m);
      }
      if (kAhead && row + warps < rows) fetch(row + warps);
      const RowScale rs(warp_max_abs(Eight<SrcT>::top(m)));
      if (lane == 0) scales[row] = rs.scale;
      uint8_t* dst = codes + static_cast<size_t>(row) * cols + lane * 8;
#pragma unroll
      for (int q = 0; q < kSegs; ++q) {
        if (lane + 32 * q >= segs) continue;
        float v[8];
        cur[q].values(v);
        *reinterpret_cast<uint2*>(dst + 256 * q) = rs.codes(v);
      }
    }
  } else {
    for (; row < rows; row += warps) {
      const SrcT* src = x + static_cast<long long>(row) * row_stride;
      typename Eight<SrcT>::Max m = Eight<SrcT>::zero();
      Eight<SrcT> e;
      for (int s = lane; s < segs; s += 32) {
        e.load(src + s * 8);
        m = e.max_with(m);
      }
      const RowScale rs(warp_max_abs(Eight<SrcT>::top(m)));
      if (lane == 0) scales[row] = rs.scale;
      uint8_t* dst = codes + static_cast<size_t>(row) * cols;
      for (int s = lane; s < segs; s += 32) {
        float v[8];
        e.load(src + s * 8);
        e.values(v);
        *reinterpret_cast<uint2*>(dst + s * 8) = rs.codes(v);
      }
    }
  }
}

// ------------------------------------------------------------------------------------------------ GEMM
constexpr int kTileM = 128, kTileN = 256, kTileK = 128;  // rows and columns of a CTA's accumulator; K in bytes = e4m3 elements
constexpr int kEpiGroups = kTileN / 64;                   // epilogue warpgroups, one per 64 columns (one head) of the tile
constexpr int kThreads = 128 + kEpiGroups * 128;          // 4 control warps + the epilogue warpgroups
constexpr uint32_t kAccCols = kTileN;           // one accumulator (128 x 256 fp32)
constexpr uint32_t kTmemCols = 2 * kAccCols;    // two of them (all of tensor memory): the products of the next tile run
                                                // under this tile's epilogue
// kPair: two CTAs work on one tile of 256 x 256.  Each loads its own 128 rows of A and one half of B's rows, 32 KB instead
// of 48 KB per K step and accumulator, since the pair's products read both halves of B from where they lie.
template <bool kPair>
struct Layout {
  static constexpr int kStages = kPair ? 4 : 3;
  static constexpr int kLoadN = kPair ? kTileN / 2 : kTileN;  // rows of B this CTA loads
  static constexpr uint32_t kStageBytes = kTileM * kTileK + kLoadN * kTileK;
  static constexpr uint32_t kOffB = kTileM * kTileK;
  static constexpr uint32_t kOffOut = kStages * kStageBytes;  // staged output, 16 KB per epilogue warpgroup (4 KB per warp)
  static constexpr uint32_t kOffMisc = kOffOut + kEpiGroups * 16384;  // column scales and bias (two tiles each), reduction
                                                                      // slots, column sums
  static constexpr uint32_t kOffBar = kOffMisc + 4096 + 64 + 2048;
  static constexpr uint32_t kSmemBytes = kOffBar + 256;  // one CTA per SM
};

struct Bars {
  uint64_t full[4], empty[4];
  uint64_t acc_full[2], acc_empty[2];  // accumulator written (issuer -> epilogue) / read out (epilogue -> issuer)
  uint32_t tmem_base;
  int abort;
};

struct LinearParams {
  const float* x_scales;  // [rows]
  const float* w_scales;  // [d_out]
  const float* bias;      // [d_out] or null
  int rows, d_in, d_out;
  int col_tiles, tiles;   // output tiles per row of tiles, and in all
  // plain output
  void* y;
  long long y_stride;  // elements
  int y_dtype;
  // fused qkv output: rows = batch * tokens, d_out = 3 * heads * 64
  int fused, batch, tokens, heads, block, nb;
  uint8_t* codes[3];
  float* scales[3];
  int* colsum[3];
  int* status;
};

// Tensor maps of the output: y in boxes of 32 rows x 128 bytes (128B swizzle), or the codes of q, k and v in boxes of 64
// rows x 64 bytes (64B swizzle).
struct OutMaps {
  CUtensorMap m[3];
};

__device__ __forceinline__ void named_barrier_sync(int id, int threads) {
  asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(threads) : "memory");
}

// Persistent CTAs (one per SM) walk the output tiles blockIdx.x, blockIdx.x + gridDim.x, ... (tiles of one row of
// tiles are neighbours, so the CTAs running at any time share their activation rows in L2).  The operand ring and the
// two accumulators are never re-initialised: ring stages and barrier parities continue on a running count of K steps,
// the accumulators alternate with the CTA's tile count.  The producer and the issuer run ahead into the next tile
// while the epilogue warps drain the previous accumulator: with one tile per CTA the operand loads stopped during
// every epilogue and the kernel was bound by the latency of its loads, not by the tensor pipe or the epilogue.
template <bool kPair>
__global__ void __launch_bounds__(kThreads, 1)
linear_fp8_kernel(const __grid_constant__ CUtensorMap map_x, const __grid_constant__ CUtensorMap map_w,
                  const __grid_constant__ OutMaps maps, const LinearParams p) {
  using L = Layout<kPair>;
  constexpr int kStages = L::kStages;
  constexpr uint32_t kStageBytes = L::kStageBytes, kOffB = L::kOffB, kOffOut = L::kOffOut, kOffMisc = L::kOffMisc;
  extern __shared__ __align__(1024) uint8_t smem[];
  Bars* bars = reinterpret_cast<Bars*>(smem + L::kOffBar);
  volatile int* abort_flag = &bars->abort;
  if ((smem_u32(smem) & 1023u) != 0) {  // the same in both CTAs of a pair
    if (threadIdx.x == 0 && p.status != nullptr) atomicCAS(p.status, 0, 900);
    return;
  }

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  // row tiles never run through a batch boundary in the fused form (a tile belongs to one sequence)
  constexpr int kCtas = kPair ? 2 : 1;
  const int tiles_per_seq = ((p.fused ? p.tokens : p.rows) + kCtas * kTileM - 1) / (kCtas * kTileM);
  const int rank = kPair ? static_cast<int>(cluster_rank()) : 0;
  const int first_tile = blockIdx.x / kCtas, tile_step = gridDim.x / kCtas;
  const int k_steps = p.d_in / kTileK;
  struct TileAt {
    int seq, tile_in_seq, row0, rows_valid, col0;
  };
  auto tile_at = [&](int tile_id) {
    TileAt t;
    const int row_tile = tile_id / p.col_tiles;
    t.col0 = (tile_id - row_tile * p.col_tiles) * kTileN;
    t.seq = row_tile / tiles_per_seq;
    t.tile_in_seq = kCtas * (row_tile - t.seq * tiles_per_seq) + rank;  // of 128 rows
    t.row0 = (p.fused ? t.seq * p.tokens : 0) + t.tile_in_seq * kTileM;
    t.rows_valid = min(kTileM, (p.fused ? p.tokens : p.rows) - t.tile_in_seq * kTileM);
    return t;
  };

  float* const s_wscale = reinterpret_cast<float*>(smem + kOffMisc);  // [2][256] column scales, [2][256] bias
  float* const s_red = s_wscale + 4 * kTileN;  // 4 floats per epilogue warpgroup
  int* const s_colsum = reinterpret_cast<int*>(s_red + 4 * kEpiGroups);  // 128 ints per epilogue warpgroup

  if (threadIdx.x == 0) {
    for (int s = 0; s < kStages; ++s) {
      mbar_init(&bars->full[s], 1);
      mbar_init(&bars->empty[s], 1);
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(&bars->acc_full[b], 1);
      mbar_init(&bars->acc_empty[b], kCtas * kEpiGroups * 4);  // one arrival per epilogue warp
    }
    bars->abort = 0;
    mbar_fence_init();
  }
  if (warp == 1) {
    if constexpr (kPair) {
      tmem_alloc_pair(&bars->tmem_base, kTmemCols);
      tmem_relinquish_pair();
    } else {
      tmem_alloc(&bars->tmem_base, kTmemCols);
      tmem_relinquish();
    }
  }
  tc_fence_before();
  if constexpr (kPair) cluster_sync();  // barriers and tensor memory of both CTAs are there
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = bars->tmem_base;
  wait_for_prior_grid();
  launch_dependents();
  if (blockIdx.x == 0 && threadIdx.x == 0 && p.status != nullptr) *p.status = 0;

  if (warp == 0) {
    if (lane == 0) {
      tma_prefetch_desc(&map_x);
      tma_prefetch_desc(&map_w);
      bool ok = true;
      int kc = 0;  // K steps issued so far, through all tiles
      for (int tile_id = first_tile; ok && tile_id < p.tiles; tile_id += tile_step) {
        const TileAt t = tile_at(tile_id);
        for (int k = 0; ok && k < k_steps; ++k, ++kc) {
          const int st = kc % kStages;
          if (kc >= kStages)
            ok = mbar_wait_clearing(&bars->empty[st], ((kc - kStages) / kStages) & 1, abort_flag, p.status, 601, 32);
          if (!ok) break;
          if (rank == 0) mbar_arrive_expect_tx(&bars->full[st], kCtas * kStageBytes);
          if constexpr (kPair) {  // both CTAs' loads count on the leader's barrier
            const uint32_t full = cluster_u32(&bars->full[st], 0);
            tma_load_2d_pair(smem + st * kStageBytes, &map_x, full, k * kTileK, t.row0);
            tma_load_2d_pair(smem + st * kStageBytes + kOffB, &map_w, full, k * kTileK, t.col0 + rank * L::kLoadN);
          } else {
            tma_load_2d(smem + st * kStageBytes, &map_x, &bars->full[st], k * kTileK, t.row0);
            tma_load_2d(smem + st * kStageBytes + kOffB, &map_w, &bars->full[st], k * kTileK, t.col0);
          }
        }
      }
    }
  } else if (warp == 1) {
    if (lane == 0 && rank == 0) {
      constexpr uint32_t idesc = instr_desc(0, kCtas * kTileM, kTileN, 0, 0);  // e4m3 x e4m3, both K-major
      const uint64_t a_desc0 = smem_desc(smem_u32(smem), 16, 1024, kSwizzle128);
      const uint64_t b_desc0 = smem_desc(smem_u32(smem) + kOffB, 16, 1024, kSwizzle128);
      bool ok = true;
      int kc = 0, it = 0;
      for (int tile_id = first_tile; ok && tile_id < p.tiles; tile_id += tile_step, ++it) {
        const int ab = it & 1;
        // the accumulator was last used two tiles ago: wait until the epilogue warps have read it out
        if (it >= 2) ok = mbar_wait_clearing(&bars->acc_empty[ab], ((it - 2) >> 1) & 1, abort_flag, p.status, 604);
        tc_fence_after();
        for (int k = 0; ok && k < k_steps; ++k, ++kc) {
          const int st = kc % kStages;
          ok = mbar_wait_clearing(&bars->full[st], (kc / kStages) & 1, abort_flag, p.status, 602);
          if (!ok) break;
          tc_fence_after();
          const uint64_t off = static_cast<uint64_t>((st * kStageBytes) >> 4);
#pragma unroll
          for (int kk = 0; kk < 4; ++kk) {
            const uint64_t a_desc = a_desc0 + off + ((kk * 32) >> 4), b_desc = b_desc0 + off + ((kk * 32) >> 4);
            const uint32_t accumulate = (k > 0 || kk > 0) ? 1u : 0u;
            if constexpr (kPair) mma_f8_pair(tmem + ab * kAccCols, a_desc, b_desc, idesc, accumulate);
            else mma_f8(tmem + ab * kAccCols, a_desc, b_desc, idesc, accumulate);
          }
          if constexpr (kPair) mma_commit_pair(&bars->empty[st]);
          else mma_commit(&bars->empty[st]);
        }
        if (ok) {
          if constexpr (kPair) mma_commit_pair(&bars->acc_full[ab]);
          else mma_commit(&bars->acc_full[ab]);
        }
      }
    }
  } else if (warp >= 4) {
    // ------------------------------------------------------------------------------------------ epilogue
    const int quarter = warp & 3;
    const int hh = (warp - 4) >> 2;     // which 64 columns of the tile this warpgroup owns
    const int r = quarter * 32 + lane;  // row of the tile = TMEM lane
    const int tid = threadIdx.x - (4 + hh * 4) * 32;  // thread of the warpgroup
    uint8_t* const staged = smem + kOffOut + hh * 16384;  // this warpgroup's output on its way to memory
    const int bar_id = 1 + hh;
    auto acc_read_out = [&](int ab) {  // the issuer waits in the leader
      tc_fence_before();
      __syncwarp();
      if (lane == 0) {
        if constexpr (kPair) mbar_arrive_cluster(cluster_u32(&bars->acc_empty[ab], 0));
        else mbar_arrive(&bars->acc_empty[ab]);
      }
    };
    bool ok = true;
    int it = 0;
    for (int tile_id = first_tile; ok && tile_id < p.tiles; tile_id += tile_step, ++it) {
    const TileAt ta = tile_at(tile_id);
    const int row0 = ta.row0, rows_valid = ta.rows_valid, seq = ta.seq, tile_in_seq = ta.tile_in_seq;
    const int ab = it & 1;
    const bool row_ok = r < rows_valid;
    const uint32_t acc_addr = tmem + ((static_cast<uint32_t>(quarter) * 32u) << 16) + ab * kAccCols + hh * 64;
    const float sx = row_ok ? __ldg(p.x_scales + row0 + r) : 0.f;
    const int col = ta.col0 + hh * 64;
    // this warpgroup's 64 column scales and biases: two sets by turns, so that this barrier is also what separates the
    // last reads of a set from its next writes
    float* const wsc = s_wscale + ab * kTileN + hh * 64;
    float* const bia = wsc + 2 * kTileN;
    if (tid < 64) {
      wsc[tid] = col + tid < p.d_out ? __ldg(p.w_scales + col + tid) : 0.f;
      bia[tid] = (p.bias != nullptr && col + tid < p.d_out) ? __ldg(p.bias + col + tid) : 0.f;
    }
    named_barrier_sync(bar_id, 128);
    ok = mbar_wait_clearing(&bars->acc_full[ab], (it >> 1) & 1, abort_flag, p.status, 603);
    tc_fence_after();
    ok = __all_sync(0xFFFFFFFFu, ok);
    if (!ok) break;
    if (col < p.d_out && !p.fused) {
      // y = acc * (sx * sw) + b.  The warp stages its 32 rows, 128 bytes at a time, in the layout the store engine reads
      // (128B swizzle); rows and columns past the output are clipped by the engine.
      const bool wide = p.y_dtype == LITE3R_F32;
      uint8_t* const warp_tile = staged + quarter * 4096;
      const uint32_t my_row = smem_u32(warp_tile) + lane * 128;
      const int swz = lane & 7;
#pragma unroll 1
      for (int cb = 0; cb < 64; cb += 32) {
        uint32_t v[32];
        tmem_ld32(acc_addr + cb, v);
        if (wide || cb == 0) {  // what was staged here before has been read by the store engine
          if (lane == 0) bulk_wait_group_read0();
          __syncwarp();
        }
        tmem_wait_ld();
        if (cb == 32) {  // the accumulator is in registers: the issuer may reuse it
          acc_read_out(ab);
        }
#pragma unroll
        for (int c = 0; c < 32; c += 4) {
          const float4 sw4 = *reinterpret_cast<const float4*>(wsc + cb + c);
          const float4 b4 = *reinterpret_cast<const float4*>(bia + cb + c);
          v[c] = __float_as_uint(fmaf(__uint_as_float(v[c]), sx * sw4.x, b4.x));
          v[c + 1] = __float_as_uint(fmaf(__uint_as_float(v[c + 1]), sx * sw4.y, b4.y));
          v[c + 2] = __float_as_uint(fmaf(__uint_as_float(v[c + 2]), sx * sw4.z, b4.z));
          v[c + 3] = __float_as_uint(fmaf(__uint_as_float(v[c + 3]), sx * sw4.w, b4.w));
        }
        if (wide) {
#pragma unroll
          for (int c = 0; c < 8; ++c) sts128(my_row + ((c ^ swz) << 4), v[4 * c], v[4 * c + 1], v[4 * c + 2], v[4 * c + 3]);
        } else {
#pragma unroll
          for (int c = 0; c < 4; ++c) {
            uint32_t w[4];
#pragma unroll
            for (int q = 0; q < 4; ++q) {
              const float y0 = __uint_as_float(v[8 * c + 2 * q]), y1 = __uint_as_float(v[8 * c + 2 * q + 1]);
              if (p.y_dtype == LITE3R_BF16) {
                __nv_bfloat162 h = __floats2bfloat162_rn(y0, y1);
                w[q] = *reinterpret_cast<uint32_t*>(&h);
              } else {
                __half2 h = __floats2half2_rn(y0, y1);
                w[q] = *reinterpret_cast<uint32_t*>(&h);
              }
            }
            sts128(my_row + (((cb / 8 + c) ^ swz) << 4), w[0], w[1], w[2], w[3]);
          }
        }
        if (wide || cb == 32) {
          fence_proxy_async_smem();
          __syncwarp();
          if (lane == 0) {
            tma_store_2d(&maps.m[0], warp_tile, col + (wide ? cb : 0), row0 + quarter * 32);
            bulk_commit_group();
          }
        }
      }
    } else if (col < p.d_out) {
      // Fused block quantiser: this warpgroup's 64 columns are one head; each (head, token block) sub-tile gets its
      // maximum, scale, codes and column sums exactly as the stand-alone quantiser computes them from fp32 values.
      const int hd = p.heads * kHeadDim;
      const int part = col / hd, head = (col - part * hd) / kHeadDim;  // 0 q, 1 k, 2 v
      const int blocks_in_tile = kTileM / p.block;            // 2 at block 64, 1 at block 128
      const int my_block = r / p.block;                       // token block of the tile this row is in
      const int block_first_warp = my_block * (p.block / 32);  // first warp (0..3) of that block in the warpgroup
      float* const red = s_red + hh * 4;
      int* const cs = s_colsum + hh * 128;  // column sums [token block of the tile][64]
      cs[tid] = 0;
      if (tid == 0) bulk_wait_group_read0();  // the codes of the tile before have left their place
      // pass 1: the row's largest magnitude, then the block's
      // (two columns per instruction: sx * sw and acc * (sx sw) + b as packed fp32 pairs, each lane rounded exactly
      // as the scalar expression would be)
      const uint64_t sx2 = pack_f32x2(sx, sx), neg0 = pack_f32x2(-0.f, -0.f);
      float amax = 0.f;
#pragma unroll 1
      for (int cb = 0; cb < 64; cb += 32) {
        uint32_t v[32];
        tmem_ld32(acc_addr + cb, v);
        tmem_wait_ld();
#pragma unroll
        for (int c = 0; c < 32; c += 4) {
          const ulonglong2 sw4 = *reinterpret_cast<const ulonglong2*>(wsc + cb + c);
          const ulonglong2 b4 = *reinterpret_cast<const ulonglong2*>(bia + cb + c);
          float y0, y1, y2, y3;
          unpack_f32x2(fma_f32x2(pack_f32x2(__uint_as_float(v[c]), __uint_as_float(v[c + 1])), fma_f32x2(sx2, sw4.x, neg0), b4.x), y0, y1);
          unpack_f32x2(fma_f32x2(pack_f32x2(__uint_as_float(v[c + 2]), __uint_as_float(v[c + 3])), fma_f32x2(sx2, sw4.y, neg0), b4.y), y2, y3);
          v[c] = __float_as_uint(y0);
          v[c + 1] = __float_as_uint(y1);
          v[c + 2] = __float_as_uint(y2);
          v[c + 3] = __float_as_uint(y3);
          amax = fmaxf(amax, fmaxf(fmaxf(fabsf(y0), fabsf(y1)), fmaxf(fabsf(y2), fabsf(y3))));
        }
        tmem_st32(acc_addr + cb, v);  // the finished values take the products' place
      }
      amax = warp_max_abs(row_ok ? amax : 0.f);
      if (lane == 0) red[quarter] = amax;
      named_barrier_sync(bar_id, 128);
      amax = 0.f;
      for (int wq = 0; wq < p.block / 32; ++wq) amax = fmaxf(amax, red[block_first_warp + wq]);
      const float scale = e4m3_scale(amax);
      const int token_block = tile_in_seq * blocks_in_tile + my_block;
      const bool block_ok = token_block < p.nb;
      const size_t tile_out = (static_cast<size_t>(seq) * p.heads + head) * p.nb + token_block;
      if (block_ok && (r % p.block) == 0) p.scales[part][tile_out] = scale;
      // pass 2: codes
      const E4m3Quotient quotient(scale);
      tmem_wait_st();
      const bool want_colsum = p.colsum[part] != nullptr;
      const uint32_t my_row = smem_u32(staged) + r * 64;
      const int swz = (r >> 1) & 3;
#pragma unroll 1
      for (int cb = 0; cb < 64; cb += 32) {
        uint32_t v[32], packed[8];
        tmem_ld32(acc_addr + cb, v);
        tmem_wait_ld();
        if (cb == 32) {  // the accumulator is in registers: the issuer may reuse it
          acc_read_out(ab);
        }
        auto codes_of = [&](auto twice) {
#pragma unroll
          for (int c = 0; c < 32; c += 4)
            packed[c >> 2] = quotient.four<decltype(twice)::value>(pack_f32x2(__uint_as_float(v[c]), __uint_as_float(v[c + 1])),
                                                                   pack_f32x2(__uint_as_float(v[c + 2]), __uint_as_float(v[c + 3])));
        };
        if (quotient.close) codes_of(std::true_type());
        else codes_of(std::false_type());
        if (!row_ok) {
#pragma unroll
          for (int c = 0; c < 8; ++c) packed[c] = 0u;
        }
        // rows past the sequence end inside an existing block are written as zeros
        sts128(my_row + (((cb / 16) ^ swz) << 4), packed[0], packed[1], packed[2], packed[3]);
        sts128(my_row + (((cb / 16 + 1) ^ swz) << 4), packed[4], packed[5], packed[6], packed[7]);
      }
      fence_proxy_async_smem();
      named_barrier_sync(bar_id, 128);
      if (tid == 0) {  // two boxes of 64 rows, as far as their blocks exist
        const int first_row = static_cast<int>((static_cast<size_t>(seq) * p.heads + head) * p.nb * p.block) + tile_in_seq * kTileM;
        for (int x = 0; x < 2; ++x)
          if (tile_in_seq * kTileM + x * 64 < p.nb * p.block) tma_store_2d(&maps.m[part], staged + x * 4096, 0, first_row + x * 64);
        bulk_commit_group();
      }
      if (want_colsum) {
        // Column sums of the code values (exact integers in units of 2^-9) from the staged codes: a thread adds four columns
        // over every eighth row in fp32 (exact: at most 8 x 448 in steps of 2^-9), 64 rows at a time, the row groups meet
        // in shared memory.
        const int cg = tid & 15;
#pragma unroll 1
        for (int x = 0; x < 2; ++x) {
          float a0 = 0.f, a1 = 0.f, a2 = 0.f, a3 = 0.f;
#pragma unroll
          for (int rr = 0; rr < 8; ++rr) {
            const int row = x * 64 + rr * 8 + (tid >> 4);
            const uint32_t w4 = *reinterpret_cast<const uint32_t*>(staged + row * 64 + (((cg >> 2) ^ ((row >> 1) & 3)) << 4) + (cg & 3) * 4);
            const __half2_raw lo = __nv_cvt_fp8x2_to_halfraw2(static_cast<__nv_fp8x2_storage_t>(w4 & 0xFFFFu), __NV_E4M3);
            const __half2_raw hi = __nv_cvt_fp8x2_to_halfraw2(static_cast<__nv_fp8x2_storage_t>(w4 >> 16), __NV_E4M3);
            const float2 f01 = __half22float2(__half2(lo)), f23 = __half22float2(__half2(hi));
            a0 += f01.x;
            a1 += f01.y;
            a2 += f23.x;
            a3 += f23.y;
          }
          int* dst = cs + (p.block == 64 ? x * 64 : 0) + cg * 4;
          atomicAdd(dst, __float2int_rn(a0 * 512.f));
          atomicAdd(dst + 1, __float2int_rn(a1 * 512.f));
          atomicAdd(dst + 2, __float2int_rn(a2 * 512.f));
          atomicAdd(dst + 3, __float2int_rn(a3 * 512.f));
        }
        named_barrier_sync(bar_id, 128);
        if (tid < blocks_in_tile * 64) {
          const int blk = tid >> 6, cc = tid & 63;
          const int tb = tile_in_seq * blocks_in_tile + blk;
          if (tb < p.nb)
            p.colsum[part][((static_cast<size_t>(seq) * p.heads + head) * p.nb + tb) * kHeadDim + cc] = cs[tid];
        }
      }
    } else {
      acc_read_out(ab);  // nothing to do for columns past the output
    }
    }  // tiles
    bulk_wait_group_read0();  // what is staged stays in place until it has been read
  }

  tc_fence_before();
  __syncthreads();
  linger_after_abort(abort_flag);
  if constexpr (kPair) cluster_sync();  // neither CTA leaves while the other one's loads, products or arrivals may reach it
  if (warp == 1) {
    tc_fence_after();
    if constexpr (kPair) tmem_dealloc_pair(tmem, kTmemCols);
    else tmem_dealloc(tmem, kTmemCols);
  }
}

int row_tiles(const LinearParams& p, int rows) {
  return p.fused ? p.batch * ceil_div(p.tokens, rows) : ceil_div(p.rows, rows);
}

template <bool kPair>
lite3r_status launch_tiles(const uint8_t* x_codes, const uint8_t* w_codes, const OutMaps& maps, const LinearParams& p, int sms,
                           cudaStream_t stream) {
  using L = Layout<kPair>;
  constexpr int kCtas = kPair ? 2 : 1;
  CUtensorMap map_x, map_w;
  lite3r_status st;
  if ((st = make_tensor_map_2d(&map_x, CU_TENSOR_MAP_DATA_TYPE_UINT8, 1, x_codes, p.d_in, p.rows, kTileK, kTileM,
                               CU_TENSOR_MAP_SWIZZLE_128B)) != LITE3R_OK) return st;
  if ((st = make_tensor_map_2d(&map_w, CU_TENSOR_MAP_DATA_TYPE_UINT8, 1, w_codes, p.d_in, p.d_out, kTileK, L::kLoadN,
                               CU_TENSOR_MAP_SWIZZLE_128B)) != LITE3R_OK) return st;
  if ((st = ensure_dynamic_smem(linear_fp8_kernel<kPair>, static_cast<int>(L::kSmemBytes))) != LITE3R_OK) return st;
  LinearParams q = p;
  q.col_tiles = ceil_div(p.d_out, kTileN);
  q.tiles = q.col_tiles * row_tiles(p, kCtas * kTileM);
  const int grid = kCtas * std::min(q.tiles, sms / kCtas);
  return launch_dependent_cluster(linear_fp8_kernel<kPair>, dim3(static_cast<unsigned>(grid)), kThreads,
                                  static_cast<int>(L::kSmemBytes), kCtas, stream, map_x, map_w, maps, q);
}

// Pairs of CTAs when there is more than one tile of 128 x 256 per SM: a tile's operand bytes, which bound the kernel, are a
// third fewer.  Up to one tile per SM nothing overlaps and the pair's two hand-shakes are in the way (one frame of the qkv
// projection, 132 tiles: 13.3 us by single CTAs, 13.8 by pairs).
lite3r_status launch_gemm(const uint8_t* x_codes, const uint8_t* w_codes, const OutMaps& maps, const LinearParams& p,
                          cudaStream_t stream) {
  int sms = 0;
  const lite3r_status st = sm_count(&sms);
  if (st != LITE3R_OK) return st;
  return static_cast<long long>(ceil_div(p.d_out, kTileN)) * row_tiles(p, kTileM) > sms
             ? launch_tiles<true>(x_codes, w_codes, maps, p, sms, stream)
             : launch_tiles<false>(x_codes, w_codes, maps, p, sms, stream);
}

template <typename SrcT>
lite3r_status launch_rowquant_typed(const SrcT* x, long long row_stride, int rows, int cols, uint8_t* codes, float* scales,
                                    cudaStream_t stream) {
  int sms = 0;
  lite3r_status st = sm_count(&sms);
  if (st != LITE3R_OK) return st;
  // rows in registers up to 1024 values (512 with half the registers); four or eight resident CTAs per SM walk the rows
  const int segs = ceil_div(cols, 256);
  auto* kernel = segs <= 2 ? rowquant_kernel<SrcT, 2> : segs <= 4 ? rowquant_kernel<SrcT, 4> : rowquant_kernel<SrcT, 0>;
  const int blocks = std::min(ceil_div(rows, 8), sms * 4);
  return launch_dependent(kernel, dim3(static_cast<unsigned>(blocks)), 256, 0, stream, x, row_stride, rows, cols, codes, scales);
}

}  // namespace

lite3r_status launch_rowquant(const void* x, int dtype, long long row_stride, int rows, int cols, uint8_t* codes,
                              float* scales, cudaStream_t stream) {
  return dtype == LITE3R_BF16
             ? launch_rowquant_typed(static_cast<const __nv_bfloat16*>(x), row_stride, rows, cols, codes, scales, stream)
             : launch_rowquant_typed(static_cast<const float*>(x), row_stride, rows, cols, codes, scales, stream);
}

lite3r_status launch_linear_fp8(const uint8_t* x_codes, const float* x_scales, const uint8_t* w_codes,
                                const float* w_scales, const float* bias, int rows, int d_in, int d_out, void* y,
                                int y_dtype, long long y_stride, int* device_status, cudaStream_t stream) {
  LinearParams p = {};
  p.x_scales = x_scales;
  p.w_scales = w_scales;
  p.bias = bias;
  p.rows = rows;
  p.d_in = d_in;
  p.d_out = d_out;
  p.y = y;
  p.y_stride = y_stride;
  p.y_dtype = y_dtype;
  p.fused = 0;
  p.status = device_status;
  const int elem = y_dtype == LITE3R_F32 ? 4 : 2;
  OutMaps maps;
  const lite3r_status st = make_tensor_map_2d(&maps.m[0],
                                              y_dtype == LITE3R_F32    ? CU_TENSOR_MAP_DATA_TYPE_FLOAT32
                                              : y_dtype == LITE3R_BF16 ? CU_TENSOR_MAP_DATA_TYPE_BFLOAT16
                                                                       : CU_TENSOR_MAP_DATA_TYPE_FLOAT16,
                                              elem, y, d_out, rows, 128 / elem, 32, CU_TENSOR_MAP_SWIZZLE_128B,
                                              static_cast<uint64_t>(y_stride) * elem);
  if (st != LITE3R_OK) return st;
  maps.m[1] = maps.m[2] = maps.m[0];
  return launch_gemm(x_codes, w_codes, maps, p, stream);
}

lite3r_status launch_qkv_project(const uint8_t* x_codes, const float* x_scales, const uint8_t* w_codes,
                                 const float* w_scales, const float* bias, const lite3r_shape& s, int d_model,
                                 const lite3r_fp8* out, int* device_status, cudaStream_t stream) {
  LinearParams p = {};
  p.x_scales = x_scales;
  p.w_scales = w_scales;
  p.bias = bias;
  p.rows = s.batch * s.tokens;
  p.d_in = d_model;
  p.d_out = 3 * s.heads * kHeadDim;
  p.fused = 1;
  p.batch = s.batch;
  p.tokens = s.tokens;
  p.heads = s.heads;
  p.block = s.block;
  p.nb = ceil_div(s.tokens, s.block);
  for (int i = 0; i < 3; ++i) {
    p.codes[i] = out[i].codes;
    p.scales[i] = out[i].scales;
    p.colsum[i] = out[i].colsum;
  }
  p.status = device_status;
  OutMaps maps;
  lite3r_status st;
  for (int i = 0; i < 3; ++i)
    if ((st = make_tensor_map_2d(&maps.m[i], CU_TENSOR_MAP_DATA_TYPE_UINT8, 1, out[i].codes, kHeadDim,
                                 static_cast<uint64_t>(s.batch) * s.heads * p.nb * s.block, 64, 64, CU_TENSOR_MAP_SWIZZLE_64B)) != LITE3R_OK)
      return st;
  return launch_gemm(x_codes, w_codes, maps, p, stream);
}

}  // namespace lite3r
