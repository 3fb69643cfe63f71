// K4: critical-block softmax attention + linear branch + add (Algorithm 1's sparse branch, linear output, projection
// and sum) on tcgen05 / TMEM / TMA.
//
// One CTA owns 128 query rows of one (b, h): at block 64 a PAIR of query blocks (two M=64 problems interleaved in the
// two 16-lane halves of every TMEM sub-partition, each with its own list of critical key blocks), at block 128 one
// query block (M=128).  Work advances in steps of 64 keys.  Per step t:
//   TMA      K tile(s) (e4m3, 64-byte rows, 64B swizzle) and V tile(s) (dequantised fp16, 128B swizzle) -> rings of two
//   tcgen05  S = Q K^T             kind::f8f6f4, fp32 accumulators in TMEM (64 columns)
//   softmax  one thread per query row (TMEM lane = thread): the 64 scores are read into registers and S is released at
//            once (Q K^T of step t+1 runs under the exponentials of step t); exp2, row sum; the probabilities go back
//            to TMEM as packed fp16 (P, 32 columns)
//   tcgen05  O += P V              kind::f16 with the A operand read from TMEM, V as MN-major B operand from shared
//                                  memory, one fp32 accumulator in TMEM (64 columns), under the exponentials of step t+1
// so the softmax warps never wait for a product in the steady state.  The largest unit is the exponential one: 16 per clock
// and SM, 448 clocks per step with an eighth of the exponentials on the multiply-add pipe; the products of a step take 384
// clocks of tensor pipe at block 64 (M = 64 runs at half rate) and 192 at block 128.  A warp alone needs some 1100 clocks
// for its 32 x 64 scores (loads, stores and barriers included), so two warps per scheduler are the least that can keep
// the unit busy: S, P and O take 160 TMEM columns, 74 KB of shared memory and 80 registers per thread, and THREE CTAs fit
// on an SM (two CTAs with two softmax warpgroups each on alternate steps of one tile: 757 clocks per step and SM at 10 % of
// 2147 key blocks, three CTAs 654 with a maximum in every step).  No unit is saturated; what the softmax warps issue decides
// (see kHeadroom).
// A CTA takes tile after tile: it asks the hardware's work scheduler for a CTA that has not been launched yet and computes
// that one's tile itself (taken only where the grid is larger than the chip holds and a tile has products).  The next tile's Q, K and V tiles and
// its first scores are then under way while the softmax warps write this tile's output, and what lies between two tiles
// of a CTA (5.5 k clocks of 13 k: launch, barriers, TMEM allocation, first loads) is paid once.  Barriers are never
// re-initialised: rings and parities run on a count through all tiles.
// The code (50 KB) is kept below the instruction cache's limit (at 62 KB the same kernel is 8 % slower): waits with their
// rare part out of line, loops not unrolled, warp-uniform values made known to the compiler.
// P is carried in fp16 (not e4m3): one e4m3 term has a 2.6 % rounding error per probability, which alone is ten
// times the output tolerance.  V travels as the dequantised value in fp16 (2^-12 relative rounding).
// Tail: phi(Q) (bf16) times the aggregated, projected summaries G_i (bf16) as one more MMA, divided by
// phi(Q) . zeta_i, added to the normalised softmax output and stored.
//
// Warp roles (256 threads): warp 0 = TMA producer, warp 1 = Q K^T issuer, warp 2 = P V issuer (and the linear product)
// (all lanes run the loops, one elected lane issues; all waits block on mbarriers in the order in which the events
// occur), warp 3 fetches the tensor maps, warps 4-7 = softmax.  The control warps give registers back (setmaxnreg) so that a softmax
// thread can hold a whole row of scores next to its probabilities.
// Every wait is bounded (1 s); on expiry the CTA sets *device_status and all roles leave their loops.
#include <atomic>
#include <type_traits>
#include <utility>

#include "common.cuh"
#include "sm100.cuh"

namespace lite3r {

namespace {

using namespace sm100;

constexpr int kCtrlWarps = 4;
constexpr int kSoftmaxWarps = 4;
constexpr int kThreads = (kCtrlWarps + kSoftmaxWarps) * 32;
constexpr int kCtasPerSm = kAttentionCtasPerSm;
constexpr int kCtrlRegs = 48, kSoftmaxRegs = 112;  // 128 * 48 + 128 * 112 = 256 * 80, the launch allocation
constexpr int kStepKeys = 64;
constexpr int kStages = 2;  // K ring and V ring
// TMEM: 64 columns of scores (later the product of the linear branch), 64 of O, 32 of probabilities (packed fp16), each an
// allocation of its own, the smallest first: three CTAs then fit in whatever order they come and beside whatever an earlier
// kernel's last CTAs still hold.  (With one allocation of 128 columns and one of 32, a 32 left in the middle by such a
// start kept the third CTA out of an SM for the whole grid: 6 % at 16 heads of 137400 tokens.)
constexpr uint32_t kColsS = 64, kColsO = 64, kColsP = 32;
constexpr float kLog2e = 1.4426950408889634f;
constexpr float kRescaleThreshold = 8.0f;  // lazy rescale: keep the old reference until it is beaten by 2^8
// A step in which no score of the row can beat the reference by more than 2^15 needs no maximum: probabilities of up to 2^15
// are fp16 numbers of full precision (the largest is 2^16 - 32).  The kernel is bound by what the softmax warps issue (copies
// that leave out the exponentials, the maxima or the sums of a step are 13-20, 7-10 and 3 % faster, one with a quarter of the
// P V products 1-3 %).  16 heads of 10992 / 43968 tokens, 4 x 16 of 21984 in blocks of 128, 4 of 137400: 92.5 / 518 / 826 /
// 2292 us with a maximum in every step, 86.4 / 486 / 778 / 2166 us with it only where this bound does not do.
constexpr float kHeadroom = 15.0f;
constexpr float kNoMax = -1.0e30f;    // reference maximum of a row that has seen no valid key yet
constexpr int kScalSlots = 64;

// shared-memory map (bytes from a 1024-aligned base); a step's tiles take half a stage at block 128 (one key block's)
constexpr uint32_t kStageK = 8192, kStageV = 16384;
constexpr uint32_t kOffQ = 0;                           // 8 KB
constexpr uint32_t kOffK = kOffQ + 8192;
constexpr uint32_t kOffV = kOffK + kStages * kStageK;
constexpr uint32_t kOffPhi = kOffV + kStages * kStageV;  // phi(Q) as bf16 A operand of the linear product (16 KB); after
                                                         // that product the output rows, each warp in its own rows' place
constexpr uint32_t kOffZeta = kOffPhi + 16384;           // zeta_i of the linear branch (256 B per query block), two tiles
constexpr uint32_t kOffScal = kOffZeta + 1024;           // per ring entry and query block: {exponent factor, bound and valid keys}
constexpr uint32_t kOffNext = kOffScal + kScalSlots * 16;  // answer of the work scheduler (16 B), tile numbers (4 x 4 B)
constexpr uint32_t kOffBar = kOffNext + 32;
constexpr uint32_t kSmemBytes = kOffBar + 256;           // three CTAs per SM: 3 * (76064 + 1024 reserved) <= 233472
constexpr int kTileSlots = 4;

struct Bars {
  uint64_t q_full, phi_full, next_full;
  uint64_t tile_full[kTileSlots];             // tile number of the CTA's next tile known
  uint64_t k_full[kStages], v_full[kStages];  // TMA -> issuer
  uint64_t s_full[kStages];                   // Q K^T number n complete (n % 2) -> softmax, producer (K stage free)
  uint64_t v_done[kStages];                   // product number n of the V ring complete (n % 2) -> softmax (P free, O or
                                              // the linear product valid), producer (V stage free)
  uint64_t s_free, p_full;                    // softmax -> issuers: score columns read / probabilities stored
  uint32_t tmem_s, tmem_o, tmem_p;
  int abort;
};
static_assert(sizeof(Bars) <= 256, "barrier block");

struct AttnParams {
  const float* q_scales;
  const float* k_scales;
  const float* k_norms;  // largest norm of a key block's rows, in units of the codes (NULL: not known)
  const int* crit_idx;  // [B*H*Nb][k_crit]
  const float* zeta;    // [B*H*Nb][64]
  void* out;
  long long out_stride_b, out_stride_h, out_stride_n;
  int heads, tokens, nb, tiles_per_head, k_crit, phi, out_dtype;
  // output through TMA stores (map_o): position of the token / head / batch dimension among the map's dimensions
  // 1..3 (they are ordered by stride); tma_out = 0: plain stores
  int tma_out, dim_token, dim_head, dim_batch;
  // The preceding launch must have completed before anything is read.  0: it is the aggregation, which writes G and zeta
  // only; codes, scales, v16 and crit_idx come from launches before it and are read ahead of this kernel's wait on the
  // word of the aggregation's (sm100.cuh, "reading ahead of the own wait").
  int wait_first;
  int steal;  // more tiles than CTAs fit on the chip: CTAs take over the tiles of CTAs not yet launched (see launch)
  int* status;
};

__device__ __forceinline__ uint32_t pack_half2(float a, float b) {
  __half2 h = __floats2half2_rn(a, b);
  return *reinterpret_cast<uint32_t*>(&h);
}
__device__ __forceinline__ float max3(float a, float b, float c) {
  float r;
  asm("max.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(b), "f"(c));
  return r;
}
__device__ __forceinline__ uint32_t pack_bf162(float a, float b) {
  __nv_bfloat162 h = __floats2bfloat162_rn(a, b);
  return *reinterpret_cast<uint32_t*>(&h);
}
// D[tmem] (+)= A[tmem] * B[smem], kind::f16: the A operand (M x 16 halves per instruction = 8 columns of packed
// pairs, row = TMEM lane) is read from tensor memory.
__device__ __forceinline__ void mma_f16_ts(uint32_t d_tmem, uint32_t a_tmem, uint64_t b_desc, uint32_t idesc,
                                           uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n\t}"
      ::"r"(d_tmem), "r"(a_tmem), "l"(b_desc), "r"(idesc), "r"(accumulate)
      : "memory");
}
__device__ __forceinline__ uint2 lds_volatile_v2(uint32_t addr) {
  uint2 v;
  asm volatile("ld.volatile.shared.v2.u32 {%0, %1}, [%2];" : "=r"(v.x), "=r"(v.y) : "r"(addr) : "memory");
  return v;
}
__device__ __forceinline__ void sts_volatile_v2(uint32_t addr, uint32_t x, uint32_t y) {
  asm volatile("st.volatile.shared.v2.u32 [%0], {%1, %2};" ::"r"(addr), "r"(x), "r"(y) : "memory");
}
// Hides where a value comes from: what is derived from it is then computed where it is used instead of being kept in
// registers (dozens of them) around the loop over the tiles.
__device__ __forceinline__ void opaque(uint32_t& v) { asm volatile("" : "+r"(v)); }
__device__ __forceinline__ void mbar_expect_tx(uint64_t* bar, uint32_t bytes) {
  asm volatile("mbarrier.expect_tx.relaxed.cta.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes) : "memory");
}

// Scales the 64 accumulator columns of this thread's TMEM lane by alpha (rare).
static __device__ __noinline__ void rescale_accumulator(uint32_t o_addr, float alpha) {
#pragma unroll 1
  for (int part = 0; part < 4; ++part) {
    uint32_t o[16];
    tmem_ld16(o_addr + part * 16, o);
    tmem_wait_ld();
#pragma unroll
    for (int k = 0; k < 16; ++k) o[k] = __float_as_uint(__uint_as_float(o[k]) * alpha);
    tmem_st16(o_addr + part * 16, o);
  }
  tmem_wait_st();
}

// 2^a for a pair of arguments on the fused-multiply-add units: a = n + f with n = round(a) (adding 1.5 * 2^23 leaves n in
// the low mantissa bits) and |f| <= 1/2, 2^f by a degree-5 polynomial (minimax in the relative error by a Remez
// exchange; 2.1e-7 in fp32 arithmetic over all of [-1/2, 1/2], the size of the hardware approximation's own error),
// n added to the exponent field.  Arguments are at most 15 (kHeadroom) and a rounding; from below they are clamped to stay
// inside the exponent range (a value that small is zero as a probability).
__device__ __forceinline__ void exp2_pair_fma(uint64_t a2, float& p0, float& p1) {
  float a0, a1;
  unpack_f32x2(a2, a0, a1);
  a2 = pack_f32x2(fmaxf(a0, -125.f), fmaxf(a1, -125.f));
  auto both = [](float v) { return pack_f32x2(v, v); };
  const uint64_t t2 = add_f32x2(a2, both(12582912.f));
  const uint64_t f2 = fma_f32x2(add_f32x2(t2, both(-12582912.f)), both(-1.f), a2);
  uint64_t q = fma_f32x2(both(0.0013276472454890609f), f2, both(0.009675540961325169f));
  q = fma_f32x2(q, f2, both(0.05550713092088699f));
  q = fma_f32x2(q, f2, both(0.24022120237350464f));
  q = fma_f32x2(q, f2, both(0.6931469440460205f));
  q = fma_f32x2(q, f2, both(1.0000001192092896f));
  float t0, t1, q0, q1;
  unpack_f32x2(t2, t0, t1);
  unpack_f32x2(q, q0, q1);
  p0 = __uint_as_float(__float_as_uint(q0) + (__float_as_uint(t0) << 23));
  p1 = __uint_as_float(__float_as_uint(q1) + (__float_as_uint(t1) << 23));
}

// exp2 of 32 scaled scores, packed to fp16 pairs; adds them to two running pairs of sums.  Arguments and sums run on
// pairs of columns (packed fp32x2 fma / add).  Every eighth pair goes to the multiply-add units at block 64, every fifth at
// block 128, where the products leave the tensor pipe idle for longer (16 heads of 43968 tokens in blocks of 64: none 514 us,
// every 16th 494, eighth 486, fifth 500, fourth 500; 4 x 16 of 21984 in blocks of 128: 811, 789, 776, 764, 764).
template <int kPolyEvery>
__device__ __forceinline__ void exp_half_row(const uint32_t (&x)[32], uint64_t c2, uint64_t shift2, uint32_t* packed,
                                             uint64_t (&sum2)[2]) {
#pragma unroll
  for (int k = 0; k < 32; k += 2) {
    const uint64_t a2 = fma_f32x2(pack_f32x2(__uint_as_float(x[k]), __uint_as_float(x[k + 1])), c2, shift2);
    float p0, p1;
    if ((k >> 1) % kPolyEvery == kPolyEvery - 1) {
      exp2_pair_fma(a2, p0, p1);
    } else {
      float a0, a1;
      unpack_f32x2(a2, a0, a1);
      p0 = ex2(a0);
      p1 = ex2(a1);
    }
    sum2[(k >> 1) & 1] = add_f32x2(sum2[(k >> 1) & 1], pack_f32x2(p0, p1));
    packed[k >> 1] = pack_half2(p0, p1);
  }
}

// Work stealing: asks for the cancellation of a CTA of this grid that has not been launched yet (the answer arrives in
// shared memory and is counted on `bar`); taken_cta returns the number of the cancelled CTA, whose tile the asking CTA then
// computes itself, or -1 when none was left.
__device__ __forceinline__ void request_next_cta(uint32_t answer, uint64_t* bar) {
  asm volatile("clusterlaunchcontrol.try_cancel.async.shared::cta.mbarrier::complete_tx::bytes.b128 [%0], [%1];"
               ::"r"(answer), "r"(smem_u32(bar)) : "memory");
}
__device__ __forceinline__ int taken_cta(uint32_t answer) {
  uint32_t x, ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t.reg .b128 r;\n\t"
      "ld.shared.b128 r, [%2];\n\t"
      "clusterlaunchcontrol.query_cancel.is_canceled.pred.b128 p, r;\n\t"
      "selp.u32 %1, 1, 0, p;\n\tmov.u32 %0, 0;\n\t"
      "@p clusterlaunchcontrol.query_cancel.get_first_ctaid::x.b32.b128 %0, r;\n\t}"
      : "=r"(x), "=r"(ok) : "r"(answer) : "memory");
  return ok != 0 ? static_cast<int>(x) : -1;
}

// kLinear: there are marginal blocks, and with them phi(Q), G, zeta and the norms of the key blocks.  An instance of its own without
// them (39 KB of code instead of 47 to 50): tiles of one or two steps, which one instance for both had made 2 to 5 % longer when the
// norm bound came in, 64 x 16 (b, h) of two blocks 42.4 -> 41.1 us a pass, 32 x 16 of 301 tokens 49.2 -> 47.7; dense rows 734 -> 727.
template <int BS, bool kLinear>
__global__ void __launch_bounds__(kThreads, kCtasPerSm)
attention_kernel(const __grid_constant__ CUtensorMap map_q, const __grid_constant__ CUtensorMap map_k,
                 const __grid_constant__ CUtensorMap map_v, const __grid_constant__ CUtensorMap map_g,
                 const __grid_constant__ CUtensorMap map_o, const AttnParams p) {
  constexpr bool kPair = (BS == 64);
  constexpr int kHalves = kPair ? 2 : 1;             // independent M=64 problems per CTA
  constexpr int kStepsPerBlock = BS / kStepKeys;     // 1 or 2
  constexpr int kM = kPair ? 64 : 128;
  constexpr int kPolyEvery = kPair ? 8 : 5;  // pairs of exponentials per one on the multiply-add units (see exp_half_row)
  constexpr uint32_t kTxK = kHalves * 4096, kTxV = kHalves * 8192;  // bytes of a step's tiles

  extern __shared__ __align__(1024) uint8_t smem[];
  Bars* bars = reinterpret_cast<Bars*>(smem + kOffBar);
  volatile int* abort_flag = &bars->abort;
  // The swizzled operand tiles need a 1024-byte aligned base; refuse to run on anything else.
  if ((smem_u32(smem) & 1023u) != 0) {
    if (threadIdx.x == 0 && p.status != nullptr) atomicCAS(p.status, 0, 900);
    return;
  }

  // (a shuffle from lane 0 tells the compiler that a value is the same in all lanes)
  const int warp = __shfl_sync(0xFFFFFFFFu, threadIdx.x >> 5, 0), lane = threadIdx.x & 31;
  const int steps = p.k_crit * kStepsPerBlock;
  const int v_steps = steps + (kLinear ? 1 : 0);  // V-ring entries of a tile: the steps' V tiles, then G
  // a tile's (b, h) and its query blocks (the second of an odd pair is a copy that is not stored)
  struct Tile {
    int bh, i_q[2];
  };
  auto tile_at = [&](int id) {
    Tile t;
    t.bh = id / p.tiles_per_head;
    const int i = id - t.bh * p.tiles_per_head;
    t.i_q[0] = kPair ? 2 * i : i;
    t.i_q[1] = kPair ? min(2 * i + 1, p.nb - 1) : i;
    return t;
  };

  if (threadIdx.x == 0) {
    mbar_init(&bars->q_full, 1);
    mbar_init(&bars->phi_full, kSoftmaxWarps);
    mbar_init(&bars->next_full, 1);
    mbar_init(&bars->s_free, kSoftmaxWarps);
    mbar_init(&bars->p_full, kSoftmaxWarps);
    for (int s = 0; s < kTileSlots; ++s) mbar_init(&bars->tile_full[s], 1);
    for (int s = 0; s < kStages; ++s) {
      mbar_init(&bars->k_full[s], 1);
      mbar_init(&bars->v_full[s], 1);
      mbar_init(&bars->s_full[s], 1);
      mbar_init(&bars->v_done[s], 1);
    }
    bars->abort = 0;
    mbar_fence_init();
  }
  if (warp == 3 && lane == 0) {  // fetched while barriers and tensor memory are set up
    tma_prefetch_desc(&map_q);
    tma_prefetch_desc(&map_k);
    tma_prefetch_desc(&map_v);
    tma_prefetch_desc(&map_g);
    tma_prefetch_desc(&map_o);
  }
  if (warp == 1) {
    tmem_alloc(&bars->tmem_p, kColsP);
    tmem_alloc(&bars->tmem_s, kColsS);
    tmem_alloc(&bars->tmem_o, kColsO);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_s = __shfl_sync(0xFFFFFFFFu, bars->tmem_s, 0), tmem_o = __shfl_sync(0xFFFFFFFFu, bars->tmem_o, 0);
  const uint32_t tmem_p = __shfl_sync(0xFFFFFFFFu, bars->tmem_p, 0);
  if (p.wait_first) wait_for_prior_grid();
  volatile int* const tile_ids = reinterpret_cast<volatile int*>(smem + kOffNext + 16);
  // number of the CTA's tile after `it` tiles (-1: none is left, -2: a wait has expired), from the producer
  auto next_tile = [&](int it, int code, auto role) {
    if (!mbar_wait_far<decltype(role)::value>(&bars->tile_full[it % kTileSlots], (it / kTileSlots) & 1, abort_flag, p.status, code)) return -2;
    return __shfl_sync(0xFFFFFFFFu, tile_ids[it % kTileSlots], 0);
  };
  // each branch below starts by giving registers back (control warps) or taking them (softmax warps)

  if (warp < kCtrlWarps) {
  setmaxnreg_dec<kCtrlRegs>();
  if (warp == 0) {
    // ------------------------------------------------------------------------------------------ TMA producer
    // All 32 lanes run the loop and the waits, so that control flow, step counters and addresses are the same in every
    // lane (the compiler can then keep them in the warp's uniform registers, which is where TMA and tcgen05
    // instructions take their operands from); one elected lane issues.
    const bool leader = elect_one();
    const uint32_t answer = smem_u32(smem + kOffNext);
    // Key blocks are fetched 32 steps at a time, lane l holding those of step 32 c + l, and handed to the issuing lane by a
    // shuffle; the scalars made from their scales go to the softmax threads through shared memory: no global load sits in the
    // per-step path.
    int jl[2] = {0, 0};
    // The K cursor runs one step ahead of the V cursor (Q K^T of step t+1 is issued under the exponentials of step t, before
    // P V of step t): the events the two wait for alternate in time in exactly this order, so blocking waits lose nothing.
    bool ok = true;
    int kc = 0, vc = 0;  // ring entries so far, through all tiles
    auto wait_all = [&](uint64_t* bar, uint32_t parity, int code) {
      return __all_sync(0xFFFFFFFFu, mbar_wait_far<1>(bar, parity, abort_flag, p.status, code));
    };
    auto wait_v_stage = [&]() {
      return vc < kStages || wait_all(&bars->v_done[vc % kStages], (vc / kStages - 1) & 1, 102);
    };
    int id = blockIdx.x;
#pragma unroll 1
    for (int it = 0; id >= 0; ++it) {
      const Tile tile = tile_at(id);
      const size_t bh_rows = static_cast<size_t>(tile.bh) * p.nb;
      // tile row (in the code tensors) of a step in key block j
      auto tile_row = [&](int t, int j) {
        if (kPair) return static_cast<int>((bh_rows + j) * 64);
        return static_cast<int>((bh_rows + j) * 128 + (t & 1) * 64);
      };
      if (it > 0) {  // the previous tile's last Q K^T and phi(Q) have read the Q tile
        if (steps > 0) ok = wait_all(&bars->s_full[(kc - 1) % kStages], ((kc - 1) / kStages) & 1, 104);
        if (kLinear) ok = ok && wait_all(&bars->phi_full, (it - 1) & 1, 105);
        if (!ok) break;
      }
      if (leader && v_steps > 0) {  // (a tile without products has no reader of Q: the copy could outlive the CTA)
        mbar_arrive_expect_tx(&bars->q_full, 8192);
        for (int x = 0; x < 2; ++x)
          tma_load_2d(smem + kOffQ + x * 4096, &map_q, &bars->q_full, 0,
                      static_cast<int>(kPair ? (bh_rows + tile.i_q[x]) * 64 : (bh_rows + tile.i_q[0]) * 128 + x * 64));
      }
      int jv[2] = {0, 0};  // key blocks of the V cursor's step
#pragma unroll 1
      for (int t = 0; t <= steps; ++t) {
        // The next tile is asked for two steps before the loads of this one end, which covers the answer's latency, and not
        // earlier: asked for at a tile's start, the tiles left over from the first wave all went to the CTAs that were
        // first to start, three to an SM, while other SMs ran dry (688 tiles of 69 steps: 248 us per step of two heads of 43968 tokens,
        // 225 us asked for here).
        if (t == max(steps - 1, 0) && leader && p.steal) {
          mbar_arrive_expect_tx(&bars->next_full, 16);
          request_next_cta(answer, &bars->next_full);
        }
        int jk[2] = {0, 0};
        if (t < steps) {
          const bool refill = (t & 31) == 0;
          if (refill) {
            const int tt = min(t + lane, steps - 1);
            for (int hf = 0; hf < kHalves; ++hf)
              jl[hf] = ldg_pinned(p.crit_idx + (bh_rows + tile.i_q[hf]) * p.k_crit + (kPair ? tt : tt / 2));
          }
          const int st = kc % kStages;
          if (kc >= kStages) ok = wait_all(&bars->s_full[st], (kc / kStages - 1) & 1, 101);
          if (!ok) break;
          for (int hf = 0; hf < kHalves; ++hf) jk[hf] = __shfl_sync(0xFFFFFFFFu, jl[hf], t & 31);
          if (leader) {
            mbar_expect_tx(&bars->k_full[st], kTxK);
            for (int hf = 0; hf < kHalves; ++hf)
              tma_load_2d(smem + kOffK + st * kStageK + hf * 4096, &map_k, &bars->k_full[st], 0, tile_row(t, jk[hf]));
          }
          // The steps' scalars for the softmax threads, made when their key blocks are fetched, lane l those of the l-th step,
          // while the tiles travel.  Slots are those of the ring entries: the 32 written here are at most entries kc .. kc + 31,
          // and those that may still be read kc - 2 and kc - 1.
          if (refill) {
            for (int hf = 0; hf < kHalves; ++hf) {
              const float sk = ldg_pinned(p.k_scales + bh_rows + jl[hf]);
              const float c = ldg_pinned(p.q_scales + bh_rows + tile.i_q[hf]) * (kLog2e * 0.125f) * sk;  // raw score -> base-2 exponent
              int valid = p.tokens - jl[hf] * BS - (kPair ? 0 : ((t + lane) & 1) * kStepKeys);
              valid = max(0, min(kStepKeys, valid));
              // second word: the factor times the largest norm, raised by 2^7 steps of the last place or more to a multiple of
              // that many (infinity where it is not known), and in these seven bits the number of valid keys.  With u = 2^-24 the
              // norms may be 9.5 u (query: 17 roundings under the root, and the root's) and 6 u (key: 10) too small, this
              // product 1 u, and a score 64 u too large; what is added is 128 u or more.
              const float reach = p.k_norms != nullptr ? c * ldg_pinned(p.k_norms + bh_rows + jl[hf]) : INFINITY;
              const uint32_t reach_bits = reach < 1.0e30f ? (__float_as_uint(reach) + 0xFFu) & ~0x7Fu : 0x7F800000u;
              if (t + lane < steps)
                sts_volatile_v2(smem_u32(smem + kOffScal) + ((kc + lane) % kScalSlots) * 16 + hf * 8, __float_as_uint(c),
                                reach_bits | static_cast<uint32_t>(valid));
            }
            __syncwarp();
          }
          if (leader) mbar_arrive(&bars->k_full[st]);
          ++kc;
        }
        if (t > 0) {
          const int st = vc % kStages;
          if (!(ok = wait_v_stage())) break;
          if (leader) {
            mbar_arrive_expect_tx(&bars->v_full[st], kTxV);
            for (int hf = 0; hf < kHalves; ++hf)
              tma_load_2d(smem + kOffV + st * kStageV + hf * 8192, &map_v, &bars->v_full[st], 0, tile_row(t - 1, jv[hf]));
          }
          ++vc;
        }
        for (int hf = 0; hf < kHalves; ++hf) jv[hf] = jk[hf];
      }
      if (ok && kLinear) {
        // The aggregated summaries follow the last V tile through its ring.  G and zeta come from the kernel enqueued
        // just before this one, which may still be running when this kernel was launched to overlap with it: everything
        // above reads older results only.
        const int st = vc % kStages;
        ok = wait_v_stage();
        if (it == 0) wait_for_prior_grid();
        if (ok && leader) {
          mbar_arrive_expect_tx(&bars->v_full[st], kHalves * (256 + 8192));
          for (int hf = 0; hf < kHalves; ++hf) {
            bulk_load(smem + kOffZeta + (it & 1) * 512 + hf * 256, p.zeta + (bh_rows + tile.i_q[hf]) * kHeadDim, 256, &bars->v_full[st]);
            tma_load_2d(smem + kOffV + st * kStageV + hf * 8192, &map_g, &bars->v_full[st], 0,
                        static_cast<int>((bh_rows + tile.i_q[hf]) * 64));
          }
        }
        ++vc;
      }
      if (!ok) break;
      id = -1;
      if (p.steal) {
        if (!(ok = wait_all(&bars->next_full, it & 1, 106))) break;
        id = __shfl_sync(0xFFFFFFFFu, taken_cta(answer), 0);
      }
      fence_proxy_async_smem();  // the answer has been read before the next one may be written
      __syncwarp();
      if (leader) {
        tile_ids[it % kTileSlots] = id;
        mbar_arrive(&bars->tile_full[it % kTileSlots]);
      }
    }
  } else if (warp == 1) {
    // ------------------------------------------------------------------------------------------ Q K^T issuer
    const bool leader = elect_one();
    constexpr uint32_t idesc_qk = instr_desc(0, kM, 64, 0, 0);  // e4m3 x e4m3, both K-major
    const uint64_t q_desc = smem_desc(smem_u32(smem + kOffQ), 16, 512, kSwizzle64);
    const uint64_t k_desc0 = smem_desc(smem_u32(smem + kOffK), 16, 512, kSwizzle64);
    bool ok = true;
    int kc = 0, sc = 0;  // products issued, releases of the score columns waited for, through all tiles
#pragma unroll 1
    for (int it = 0, id = 0; id >= 0 && steps > 0; id = next_tile(it, 210, std::integral_constant<int, 1>{}), ++it) {
      ok = mbar_wait_far<1>(&bars->q_full, it & 1, abort_flag, p.status, 201);
#pragma unroll 1
      for (int t = 0; t < steps; ++t, ++kc) {
        const int st = kc % kStages;
        ok = ok && mbar_wait_far<1>(&bars->k_full[st], (kc / kStages) & 1, abort_flag, p.status, 202);
        if (t > 0 || it > 0) {  // the scores of the step before (in a tile's first step: the linear product) have been read
          ok = ok && mbar_wait_far<1>(&bars->s_free, sc & 1, abort_flag, p.status, 203);
          ++sc;
        }
        ok = __all_sync(0xFFFFFFFFu, ok);
        if (!ok) break;
        const uint64_t k_desc = k_desc0 + static_cast<uint64_t>((st * kStageK) >> 4);
        tc_fence_after();
        if (leader) {
#pragma unroll
          for (int kk = 0; kk < 2; ++kk) {
#pragma unroll
            for (int hf = 0; hf < kHalves; ++hf)
              mma_f8(tmem_s + ((hf * 16u) << 16), q_desc + ((hf * 4096 + kk * 32) >> 4), k_desc + ((hf * 4096 + kk * 32) >> 4),
                     idesc_qk, kk);
          }
          mma_commit(&bars->s_full[st]);
        }
      }
      if (!ok) break;
      if (kLinear) {  // the release of the last scores, which the linear product takes up, passes by here
        ok = __all_sync(0xFFFFFFFFu, mbar_wait_far<1>(&bars->s_free, sc & 1, abort_flag, p.status, 208));
        ++sc;
        if (!ok) break;
      }
    }
  } else if (warp == 2) {
    // ------------------------------------------------------------------------------------------ P V issuer
    const bool leader = elect_one();
    constexpr uint32_t idesc_pv = instr_desc(0, kM, 64, 0, 1);   // f16 x f16, P from TMEM, V MN-major
    constexpr uint32_t idesc_lin = instr_desc(1, kM, 64, 0, 0);  // bf16 x bf16, both K-major
    const uint64_t v_desc0 = smem_desc(smem_u32(smem + kOffV), 8192, 1024, kSwizzle128);
    bool ok = true;
    int vc = 0, pc = 0;  // V-ring entries, probability tiles, through all tiles
#pragma unroll 1
    for (int it = 0, id = 0; id >= 0; id = next_tile(it, 211, std::integral_constant<int, 1>{}), ++it) {
#pragma unroll 1
      for (int t = 0; t < steps; ++t, ++vc, ++pc) {  // O += P V(t)
        const int st = vc % kStages;
        ok = mbar_wait_far<1>(&bars->v_full[st], (vc / kStages) & 1, abort_flag, p.status, 205) &&
             mbar_wait_far<1>(&bars->p_full, pc & 1, abort_flag, p.status, 204);
        ok = __all_sync(0xFFFFFFFFu, ok);
        if (!ok) break;
        const uint64_t v_desc = v_desc0 + static_cast<uint64_t>((st * kStageV) >> 4);
        tc_fence_after();
        if (leader) {
#pragma unroll
          for (int kk = 0; kk < 4; ++kk) {
#pragma unroll
            for (int hf = 0; hf < kHalves; ++hf)
              mma_f16_ts(tmem_o + ((hf * 16u) << 16), tmem_p + ((hf * 16u) << 16) + kk * 8,
                         v_desc + ((hf * 8192 + kk * 2048) >> 4), idesc_pv, (t > 0 || kk > 0) ? 1u : 0u);
          }
          mma_commit(&bars->v_done[st]);
        }
      }
      if (!ok) break;
      if (kLinear) {
        // phi(Q) G into the score columns (released by the softmax threads: this step's probabilities, waited for above,
        // were made from the last scores)
        const int st = vc % kStages;
        ok = mbar_wait_far<1>(&bars->phi_full, it & 1, abort_flag, p.status, 207) &&
             mbar_wait_far<1>(&bars->v_full[st], (vc / kStages) & 1, abort_flag, p.status, 206);
        ok = __all_sync(0xFFFFFFFFu, ok);
        if (!ok) break;
        tc_fence_after();
        if (leader) {
          const uint64_t a0 = smem_desc(smem_u32(smem + kOffPhi), 16, 1024, kSwizzle128);
          const uint64_t b0 = smem_desc(smem_u32(smem + kOffV) + st * kStageV, 16, 1024, kSwizzle128);
#pragma unroll
          for (int kk = 0; kk < 4; ++kk) {
#pragma unroll
            for (int hf = 0; hf < kHalves; ++hf)
              mma_f16(tmem_s + ((hf * 16u) << 16), a0 + ((hf * 8192 + kk * 32) >> 4), b0 + ((hf * 8192 + kk * 32) >> 4), idesc_lin, kk);
          }
          mma_commit(&bars->v_done[st]);
        }
        ++vc;
      }
    }
  }
  } else {
    // ------------------------------------------------------------------------------------------ softmax + epilogue
    setmaxnreg_inc<kSoftmaxRegs>();
    const int quarter = warp & 3;                       // TMEM sub-partition this warp may touch
    const int hf = kPair ? (lane >> 4) : 0;             // which query block of the pair this thread serves
    const int row_in_block = kPair ? quarter * 16 + (lane & 15) : quarter * 32 + lane;
    const int p_row = kPair ? hf * 64 + row_in_block : row_in_block;  // row inside the 128-row tile
    const uint32_t lane_off = (static_cast<uint32_t>(quarter) * 32u) << 16;
    const uint32_t s_addr = tmem_s + lane_off, o_addr = tmem_o + lane_off, p_addr = tmem_p + lane_off;
    const uint32_t scal_slot = smem_u32(smem + kOffScal) + hf * 8;
    const int swz = p_row & 7;
    // hands the probabilities of the step just finished to the P V issuer
    auto publish = [&]() {
      tmem_wait_st();
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(&bars->p_full);
    };
    bool ok = true;
    int kc = 0, vc = 0;  // Q K^T products and V-ring products so far, through all tiles
#pragma unroll 1
    for (int it = 0, id = blockIdx.x; id >= 0; id = next_tile(it, 310, std::integral_constant<int, 0>{}), ++it) {
    // shared-memory addresses of this thread's row: phi(q) / staged output, and the query
    uint32_t phi_row = smem_u32(smem + kOffPhi) + p_row * 128, q_row = smem_u32(smem + kOffQ) + p_row * 64;
    opaque(phi_row);
    opaque(q_row);
    const Tile tile = tile_at(id);
    const int iq = tile.i_q[hf];
    const size_t bh_rows = static_cast<size_t>(tile.bh) * p.nb;

    // linear branch, first part: phi(q) as bf16 A operand of the linear product.  It needs the Q tile only, so it is
    // computed while the first key tiles are on their way and the softmax threads would be idle; the denominators
    // phi(q) . zeta_i follow in the epilogue, from the operand's own rounded values.
    // The query row comes from the Q tile in shared memory (64-byte rows, 64B swizzle: 16-byte chunk c of row r sits at
    // chunk c ^ ((r >> 1) & 3)).  The loops over chunks are not unrolled: the kernel's code has to stay within the
    // instruction cache.
    float q_norm = INFINITY;  // norm of the query row in units of the codes (not known without a linear branch)
    if (kLinear) {
      const float sq = __ldg(p.q_scales + bh_rows + iq);
      if (!(ok = mbar_wait_far(&bars->q_full, it & 1, abort_flag, p.status, 307))) break;
      // the previous tile's output rows, staged where this warp's rows of phi(q) go, must have been read
      if (lane == 0) bulk_wait_group_read0();
      __syncwarp();
      const int qswz = (p_row >> 1) & 3;
      // phi = softmax over the components: any common shift of the exponents cancels in the ratio numerator /
      // denominator.  448 * scale bounds every component of the block, so it serves as the shift without a pass over
      // the row; only when exponents could then leave the fp32 range (block magnitudes in the hundreds) is the row's
      // own maximum looked up.
      const bool phi_softmax = p.phi == LITE3R_PHI_SOFTMAX;
      const float cq = sq * kLog2e;
      float shift = 448.f * cq;
      if (phi_softmax && 896.f * cq > 100.f) {
        float mxq = -INFINITY;
#pragma unroll 1
        for (int c4 = 0; c4 < 4; ++c4) {
          const uint4 raw = lds128(q_row + ((c4 ^ qswz) << 4));
          const uint32_t words[4] = {raw.x, raw.y, raw.z, raw.w};
#pragma unroll
          for (int xw = 0; xw < 4; ++xw) {
            float fv[4];
            e4m3x4_to_float(words[xw], fv);
            mxq = fmaxf(max3(mxq, fv[0], fv[1]), fmaxf(fv[2], fv[3]));
          }
        }
        shift = mxq * cq;  // sq > 0 commutes with max
      }
      uint64_t squares[2] = {0ull, 0ull};  // bit pattern of (0.f, 0.f)
#pragma unroll 1
      for (int c4 = 0; c4 < 4; ++c4) {
        const uint4 raw = lds128(q_row + ((c4 ^ qswz) << 4));
        const uint32_t words[4] = {raw.x, raw.y, raw.z, raw.w};
        uint32_t pk8[8];
#pragma unroll
        for (int xw = 0; xw < 4; ++xw) {
          float fv[4];
          e4m3x4_to_float(words[xw], fv);
#pragma unroll
          for (int y = 0; y < 4; y += 2) {
            float e0, e1;
            const uint64_t pair = pack_f32x2(fv[y], fv[y + 1]);
            squares[y >> 1] = fma_f32x2(pair, pair, squares[y >> 1]);
            if (phi_softmax) {  // the softmax normaliser cancels in the ratio
              unpack_f32x2(fma_f32x2(pair, pack_f32x2(cq, cq), pack_f32x2(-shift, -shift)), e0, e1);
              e0 = ex2(e0);
              e1 = ex2(e1);
            } else {
              e0 = fv[y] > 0.f ? fmaf(fv[y], sq, 1.f) : ex2(fv[y] * cq);
              e1 = fv[y + 1] > 0.f ? fmaf(fv[y + 1], sq, 1.f) : ex2(fv[y + 1] * cq);
            }
            pk8[xw * 2 + (y >> 1)] = pack_bf162(e0, e1);
          }
        }
        sts128(phi_row + (((c4 * 2) ^ swz) << 4), pk8[0], pk8[1], pk8[2], pk8[3]);
        sts128(phi_row + (((c4 * 2 + 1) ^ swz) << 4), pk8[4], pk8[5], pk8[6], pk8[7]);
      }
      float sq0, sq1;
      unpack_f32x2(add_f32x2(squares[0], squares[1]), sq0, sq1);
      q_norm = sqrtf(sq0 + sq1);
      fence_proxy_async_smem();
      __syncwarp();
      if (lane == 0) mbar_arrive(&bars->phi_full);
    }

    float m_ref = kNoMax, l = 0.f;  // the row's reference, and its sum relative to it
#pragma unroll 1
    for (int t = 0; t < steps; ++t, ++kc) {
      if (!(ok = mbar_wait_far(&bars->s_full[kc % kStages], (kc / kStages) & 1, abort_flag, p.status, 301))) break;
      tc_fence_after();
      uint32_t xa[32], xb[32];
      tmem_ld32(s_addr, xa);
      tmem_ld32(s_addr + 32, xb);
      if (t > 0) publish();  // the store of step t-1 has had this step's wait and loads to complete under
      // the step's scalars, left by the producer before it completed the K stage
      const uint2 scal = lds_volatile_v2(scal_slot + (kc % kScalSlots) * 16);
      const float c = __uint_as_float(scal.x);
      const int valid = static_cast<int>(scal.y & 0x7Fu);
      tmem_wait_ld();
      // the whole row of scores is in registers: the issuer may overwrite S with step t+1 right away
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(&bars->s_free);
      if (valid < kStepKeys) {
#pragma unroll
        for (int k = 0; k < 32; ++k) {
          if (k >= valid) xa[k] = 0xFF800000u;  // -inf
          if (32 + k >= valid) xb[k] = 0xFF800000u;
        }
      }
      // |q . k| <= |q| |k| bounds the step's scores, also as computed: the second word allows for the roundings before, and the
      // product and the sum here are rounded to the safe side (references beyond 2^24 are further apart than what 2^15 leaves
      // to the largest fp16 number).
      // Queries and keys of ordinary size pass it in most steps after a tile's first, which has no reference yet (92 % of those at 22
      // key blocks, six steps to a tile, 99.7 % at 687, 34 steps); they go without the maximum, its vote and the wait for both.
      if (!kLinear || !__all_sync(0xFFFFFFFFu, __fmul_ru(q_norm, __uint_as_float(scal.y)) <= __fadd_rd(m_ref, kHeadroom))) {
        // row maximum of the raw scores (c > 0 commutes with max), eight independent chains; a step without any valid key
        // (second half of a short last block) leaves the reference where it is
        float mx[8];
#pragma unroll
        for (int q = 0; q < 8; ++q) mx[q] = fmaxf(__uint_as_float(xa[q]), __uint_as_float(xb[q]));
#pragma unroll
        for (int k = 8; k < 32; k += 8) {
#pragma unroll
          for (int q = 0; q < 8; ++q) mx[q] = max3(mx[q], __uint_as_float(xa[k + q]), __uint_as_float(xb[k + q]));
        }
        const float top = fmaxf(max3(max3(mx[0], mx[1], mx[2]), max3(mx[3], mx[4], mx[5]), fmaxf(mx[6], mx[7])) * c, kNoMax);
        // lazy rescale: the reference of a row moves only when it is beaten by 2^8 (and in the first step)
        if (__any_sync(0xFFFFFFFFu, top > m_ref + kRescaleThreshold)) {
          const float m_new = top > m_ref + kRescaleThreshold ? top : m_ref;
          const float alpha = ex2(m_ref - m_new);
          l *= alpha;
          m_ref = m_new;
          if (t > 0) {
            // O is being accumulated into by the P V product of step t-1: wait for it first
            const int u = vc + t - 1;
            if (!(ok = mbar_wait_far(&bars->v_done[u % kStages], (u / kStages) & 1, abort_flag, p.status, 303))) break;
            tc_fence_after();
            rescale_accumulator(o_addr, alpha);
          }
        }
      }
      uint32_t packed[32];
      {
        const uint64_t c2 = pack_f32x2(c, c), shift2 = pack_f32x2(-m_ref, -m_ref);
        uint64_t sum2[2] = {0ull, 0ull};  // bit pattern of (0.f, 0.f)
        exp_half_row<kPolyEvery>(xa, c2, shift2, packed, sum2);
        exp_half_row<kPolyEvery>(xb, c2, shift2, packed + 16, sum2);
        float s0, s1;
        unpack_f32x2(add_f32x2(sum2[0], sum2[1]), s0, s1);
        l += s0 + s1;
      }
      // P is free once the P V product of step t-1 has completed (long ago in the steady state)
      if (t > 0) {
        const int u = vc + t - 1;
        if (!(ok = mbar_wait_far(&bars->v_done[u % kStages], (u / kStages) & 1, abort_flag, p.status, 302))) break;
        tc_fence_after();
      }
      tmem_st32(p_addr, packed);
    }
    if (!ok) break;
    if (steps > 0) publish();

    // linear branch, second part: the denominator phi(q) . zeta_i, with the same rounded values as the numerator's operand;
    // zeta_i arrives with the aggregated summaries behind the last V tile
    const int v_last = vc + v_steps - 1;  // the tile's last product
    float den = 0.f;
    if (kLinear) {
      if (!(ok = mbar_wait_far(&bars->v_full[v_last % kStages], (v_last / kStages) & 1, abort_flag, p.status, 308))) break;
      const uint32_t zeta = smem_u32(smem + kOffZeta) + (it & 1) * 512 + hf * 256;
      uint64_t den2[2] = {0ull, 0ull};  // bit pattern of (0.f, 0.f)
#pragma unroll 1
      for (int c8 = 0; c8 < 8; ++c8) {  // 16-byte chunks of eight components
        const uint4 rw = lds128(phi_row + ((c8 ^ swz) << 4));
        const uint32_t words[4] = {rw.x, rw.y, rw.z, rw.w};
#pragma unroll
        for (int half = 0; half < 2; ++half) {
          const uint4 z = lds128(zeta + c8 * 32 + half * 16);
          den2[0] = fma_f32x2(pack_f32x2(__uint_as_float(words[2 * half] << 16), __uint_as_float(words[2 * half] & 0xFFFF0000u)),
                              pack_f32x2(__uint_as_float(z.x), __uint_as_float(z.y)), den2[0]);
          den2[1] = fma_f32x2(pack_f32x2(__uint_as_float(words[2 * half + 1] << 16), __uint_as_float(words[2 * half + 1] & 0xFFFF0000u)),
                              pack_f32x2(__uint_as_float(z.z), __uint_as_float(z.w)), den2[1]);
        }
      }
      float d0, d1, d2, d3;
      unpack_f32x2(den2[0], d0, d1);
      unpack_f32x2(den2[1], d2, d3);
      den = (d0 + d1) + (d2 + d3);
      // (the last P V product is the one before)
      if (steps > 0 && !(ok = mbar_wait_far(&bars->v_done[(v_last - 1) % kStages], ((v_last - 1) / kStages) & 1, abort_flag, p.status, 304))) break;
    }
    if (v_steps > 0 && !(ok = mbar_wait_far(&bars->v_done[v_last % kStages], (v_last / kStages) & 1, abort_flag, p.status, 305))) break;
    vc += v_steps;
    tc_fence_after();

    // Output, 128 bytes of a row at a time (32 fp32 columns or 64 of a 16-bit type).  The warp stages its rows where it
    // kept its rows of phi(q) (the linear product has read them) in the layout the store engine reads: 128-byte rows with the
    // 128B swizzle.
    const int bb = tile.bh / p.heads, h = tile.bh - bb * p.heads;
    const float inv_l = steps > 0 ? 1.f / l : 0.f;
    const float l_scale = kLinear ? 1.f / den : 0.f;
    const bool wide = p.out_dtype == LITE3R_F32;
    const bool to_bf16 = p.out_dtype == LITE3R_BF16;
    if (!kLinear) {  // the previous tile's rows must have been read (next to a linear branch phi(q) has waited for that)
      if (lane == 0) bulk_wait_group_read0();
      __syncwarp();
    }
#pragma unroll 1
    for (int half = 0; half < 2; ++half) {  // 32 columns
      uint32_t v[32], u[32];
      tmem_ld32(o_addr + half * 32, v);
      tmem_ld32(s_addr + half * 32, u);
      if (wide && half == 1) {  // the first half's rows have been read by the store engine (or by the lanes that stored them)
        if (lane == 0) bulk_wait_group_read0();
        __syncwarp();
      }
      tmem_wait_ld();
      if (kLinear && half == 1) {  // the linear product has been read: the score columns are free for the next tile
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(&bars->s_free);
      }
      if (steps == 0 || !kLinear) {  // without a critical block O, without a linear branch its product was never written
#pragma unroll
        for (int k = 0; k < 32; ++k) {
          if (steps == 0) v[k] = 0u;
          if (!kLinear) u[k] = 0u;
        }
      }
      const uint64_t inv2 = pack_f32x2(inv_l, inv_l), lin2 = pack_f32x2(l_scale, l_scale);
#pragma unroll
      for (int k = 0; k < 32; k += 2) {
        const uint64_t o = mul_f32x2(pack_f32x2(__uint_as_float(v[k]), __uint_as_float(v[k + 1])), inv2);
        float y0, y1;
        unpack_f32x2(fma_f32x2(pack_f32x2(__uint_as_float(u[k]), __uint_as_float(u[k + 1])), lin2, o), y0, y1);
        v[k] = __float_as_uint(y0);
        v[k + 1] = __float_as_uint(y1);
      }
      if (wide) {
#pragma unroll
        for (int ch = 0; ch < 8; ++ch)
          sts128(phi_row + ((ch ^ swz) << 4), v[4 * ch], v[4 * ch + 1], v[4 * ch + 2], v[4 * ch + 3]);
      } else {
#pragma unroll
        for (int ch = 0; ch < 4; ++ch) {
          uint32_t pk[4];
#pragma unroll
          for (int y = 0; y < 4; ++y)
            pk[y] = to_bf16 ? pack_bf162(__uint_as_float(v[8 * ch + 2 * y]), __uint_as_float(v[8 * ch + 2 * y + 1]))
                            : pack_half2(__uint_as_float(v[8 * ch + 2 * y]), __uint_as_float(v[8 * ch + 2 * y + 1]));
          sts128(phi_row + (((half * 4 + ch) ^ swz) << 4), pk[0], pk[1], pk[2], pk[3]);
        }
        if (half == 0) continue;
      }
      if (p.tma_out != 0) {
        // boxes of 16 tokens x 128 bytes: lanes 0-15 and 16-31 hold 16 consecutive tokens each (of the two query blocks
        // of a pair, or of the two halves of the warp's 32 rows); rows past the end of the sequence are clipped by the
        // store engine, the copy of the last block in an odd pair is not stored at all
        fence_proxy_async_smem();
        __syncwarp();
        if (lane == 0) {
#pragma unroll
          for (int g2 = 0; g2 < 2; ++g2) {
            const int token0 = kPair ? tile.i_q[g2] * BS + quarter * 16 : tile.i_q[0] * BS + quarter * 32 + 16 * g2;
            if (token0 >= p.tokens || (kPair && g2 == 1 && tile.i_q[1] == tile.i_q[0])) continue;
            int c[4] = {0, 0, 0, 0};
            c[p.dim_token] = token0;
            c[p.dim_head] = h;
            c[p.dim_batch] = bb;
            const int row0 = kPair ? g2 * 64 + quarter * 16 : quarter * 32 + g2 * 16;
            tma_store_4d(&map_o, smem + kOffPhi + row0 * 128, wide ? half * 32 : 0, c[1], c[2], c[3]);
          }
          bulk_commit_group();
        }
      } else {
        __syncwarp();
        const int ch = lane & 7;
        const uint32_t elem = wide ? 4u : 2u;
        uint8_t* const out_bh = static_cast<uint8_t*>(p.out) +
                                (static_cast<long long>(bb) * p.out_stride_b + static_cast<long long>(h) * p.out_stride_h) * elem +
                                (wide ? half * 128 : 0) + ch * 16;
        const long long row_pitch = p.out_stride_n * static_cast<long long>(elem);
        const bool second_block_is_copy = kPair && tile.i_q[1] == tile.i_q[0];
#pragma unroll 1
        for (int r = lane >> 3; r < 32; r += 4) {  // row of this warp's block: thread r computed it
          const int r_hf = kPair ? (r >> 4) : 0;
          const int r_in_block = kPair ? quarter * 16 + (r & 15) : quarter * 32 + r;
          const int r_p = kPair ? r_hf * 64 + r_in_block : r_in_block;
          const int r_token = tile.i_q[r_hf] * BS + r_in_block;
          const uint4 val = *reinterpret_cast<const uint4*>(smem + kOffPhi + r_p * 128 + ((ch ^ (r_p & 7)) << 4));
          if (r_token < p.tokens && !(second_block_is_copy && r_hf == 1))
            *reinterpret_cast<uint4*>(out_bh + r_token * row_pitch) = val;
        }
        __syncwarp();
      }
    }
    tc_fence_before();  // O and the linear product have been read (ordered before the next tile's arrivals)
    }  // tiles
    if (lane == 0) bulk_wait_group_read0();  // the staged rows must stay in place until the engine has read them
  }

  tc_fence_before();
  __syncthreads();
  linger_after_abort(abort_flag);
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc(tmem_p, kColsP);
    tmem_dealloc(tmem_s, kColsS);
    tmem_dealloc(tmem_o, kColsO);
  }
}

// ------------------------------------------------------------------------------------------------ host side
// Test hook: non-zero makes the kernel write its output with plain stores even where a TMA map exists.
std::atomic<int> g_plain_stores{0};

template <int BS>
lite3r_status launch(const AttentionLaunch& a, cudaStream_t stream) {
  const lite3r_shape& s = a.shape;
  const int nb = ceil_div(s.tokens, BS);
  const uint64_t tiles = static_cast<uint64_t>(s.batch) * s.heads * nb;
  lite3r_status st;
  CUtensorMap map_q, map_k, map_v, map_g, map_o;
  if ((st = make_tensor_map_2d(&map_q, CU_TENSOR_MAP_DATA_TYPE_UINT8, 1, a.q_codes, 64, tiles * BS, 64, 64, CU_TENSOR_MAP_SWIZZLE_64B)) != LITE3R_OK) return st;
  if ((st = make_tensor_map_2d(&map_k, CU_TENSOR_MAP_DATA_TYPE_UINT8, 1, a.k_codes, 64, tiles * BS, 64, 64, CU_TENSOR_MAP_SWIZZLE_64B)) != LITE3R_OK) return st;
  if ((st = make_tensor_map_2d(&map_v, CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 2, a.v16, 64, tiles * BS, 64, 64, CU_TENSOR_MAP_SWIZZLE_128B)) != LITE3R_OK) return st;
  if ((st = make_tensor_map_2d(&map_g, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, a.g16, 64, tiles * 64, 64, 64, CU_TENSOR_MAP_SWIZZLE_128B)) != LITE3R_OK) return st;
  AttnParams p;
  // The output goes through TMA stores when a tiled map can describe it: the token, head and batch dimensions ordered
  // by stride (dimensions of extent 1 last), 16 tokens x 128 bytes per box.  If the driver refuses the map the kernel
  // falls back to plain stores.
  const int elem = a.out_dtype == LITE3R_F32 ? 4 : 2;
  struct Dim {
    long long stride;
    int extent, which;  // which: 0 token, 1 head, 2 batch
  } dm[3] = {{a.out_stride_n, s.tokens, 0}, {a.out_stride_h, s.heads, 1}, {a.out_stride_b, s.batch, 2}};
  // order: extents above 1 by ascending stride, then the extent-1 dimensions (whose stride does not matter)
  auto before = [](const Dim& x, const Dim& y) {
    if ((x.extent > 1) != (y.extent > 1)) return x.extent > 1;
    if (x.extent > 1 && x.stride != y.stride) return x.stride < y.stride;
    return x.which < y.which;
  };
  for (int i = 0; i < 3; ++i)
    for (int j = i + 1; j < 3; ++j)
      if (before(dm[j], dm[i])) std::swap(dm[i], dm[j]);
  uint64_t dims[4] = {kHeadDim, 0, 0, 0}, strides[3];
  uint32_t box[4] = {128u / elem, 1, 1, 1};  // 128 bytes of a row
  uint64_t packed = static_cast<uint64_t>(kHeadDim) * elem;  // stride a dimension would have if packed after the previous ones
  bool describable = (reinterpret_cast<uintptr_t>(a.out) & 15u) == 0;
  for (int i = 0; i < 3; ++i) {
    dims[i + 1] = static_cast<uint64_t>(dm[i].extent);
    strides[i] = dm[i].extent > 1 ? static_cast<uint64_t>(dm[i].stride) * elem : packed;
    describable = describable && strides[i] > 0 && (strides[i] & 15u) == 0;
    packed = strides[i] * dims[i + 1];
    if (dm[i].which == 0) {
      box[i + 1] = 16;
      p.dim_token = i + 1;
    } else if (dm[i].which == 1) {
      p.dim_head = i + 1;
    } else {
      p.dim_batch = i + 1;
    }
  }
  p.tma_out = 0;
  if (describable && g_plain_stores.load(std::memory_order_relaxed) == 0)
    p.tma_out = make_tensor_map_4d(&map_o,
                                   a.out_dtype == LITE3R_F32    ? CU_TENSOR_MAP_DATA_TYPE_FLOAT32
                                   : a.out_dtype == LITE3R_BF16 ? CU_TENSOR_MAP_DATA_TYPE_BFLOAT16
                                                                : CU_TENSOR_MAP_DATA_TYPE_FLOAT16,
                                   a.out, dims, strides, box, CU_TENSOR_MAP_SWIZZLE_128B) == LITE3R_OK
                    ? 1 : 0;
  if (p.tma_out == 0) map_o = map_q;  // any valid map when it is not used
  p.q_scales = a.q_scales;
  p.k_scales = a.k_scales;
  p.k_norms = a.k_norms;
  p.crit_idx = a.crit_idx;
  p.zeta = a.zeta;
  p.out = a.out;
  p.out_stride_b = a.out_stride_b;
  p.out_stride_h = a.out_stride_h;
  p.out_stride_n = a.out_stride_n;
  p.heads = s.heads;
  p.tokens = s.tokens;
  p.nb = nb;
  p.tiles_per_head = BS == 64 ? (nb + 1) / 2 : nb;
  p.k_crit = a.k_crit;
  p.phi = a.phi;
  p.out_dtype = a.out_dtype;
  p.status = a.device_status;
  auto* const kernel = a.k_marg > 0 ? attention_kernel<BS, true> : attention_kernel<BS, false>;
  st = ensure_dynamic_smem(kernel, static_cast<int>(kSmemBytes));
  if (st != LITE3R_OK) return st;
  const int ctas = s.batch * s.heads * p.tiles_per_head;
  int sms = 0;
  if ((st = sm_count(&sms)) != LITE3R_OK) return st;
  // What keeps the producer from running ahead of the softmax warps are the waits for products that read what it loaded.
  // Without critical and without marginal blocks a tile has none: the output is zeros, every CTA writes its own tile's, and
  // nothing is taken over (the producer would lap the four slots for tile numbers).
  p.steal = ctas > sms * kCtasPerSm && (a.k_crit > 0 || a.k_marg > 0) ? 1 : 0;
  // With a linear branch the launch before this one is the aggregation, whose results are needed only at a tile's end: the
  // kernel then runs beside it and waits for its completion itself.  Otherwise it waits before it reads anything.
  p.wait_first = a.overlap_prior ? 0 : 1;
  return launch_dependent(kernel, dim3(static_cast<unsigned>(ctas)), kThreads, static_cast<int>(kSmemBytes), stream,
                          map_q, map_k, map_v, map_g, map_o, p);
}

}  // namespace

void set_attention_plain_stores(int on) { g_plain_stores.store(on, std::memory_order_relaxed); }

lite3r_status launch_attention(const AttentionLaunch& a, cudaStream_t stream) {
  return a.shape.block == 64 ? launch<64>(a, stream) : launch<128>(a, stream);
}

}  // namespace lite3r
