// K3b: marginal aggregation as a mask-GEMM on tcgen05 tensor cores.
//
// For one (b, h):  G[i, n] = sum_j M[i, j] * S[j, n],  M[i, j] = 1 if key block j is marginal for query block i, else 0,
// S[j, :] = the 4160-wide bf16 summary row of key block j ((H_j W)^T | z_j).  0/1 is exact in bf16 and the
// accumulation is fp32 in TMEM, so this equals the gather-and-add of the summaries while reading each summary once per
// 128 query blocks instead of once per query block.
//
// A tile is 128 (rows) x 256 (summary columns; the last column tile is the 64 of zeta); the reduction runs over key blocks
// in chunks of 64.  Rows and keys are numbered through all (b, h).  Tiles either stay inside one (b, h), or, for short
// sequences, run through the (b, h) boundaries so that several small problems share a tile (the mask is then
// block-diagonal); the launcher takes the cheaper tiling.
//
// Persistent CTAs, one per SM, walk the tiles (the column tiles of a row tile are neighbours, so that the CTAs running at any
// time share class rows and summaries in L2).  The ring of four chunks runs on through the tiles and the two accumulators
// alternate, so that loads, mask tiles and products of the next tile run under the stores of this one.  Warp 0 brings the
// 64 x 256 slab of summaries by TMA (MN-major B operand, four 64-column boxes, 128B swizzle); warp 1 issues four
// 128x256x16 MMAs per chunk; two warpgroups, each taking every other chunk, expand the class bytes into the bf16 0/1 A tile
// (K-major, 128B swizzle), eight lanes to a row; two more, one per accumulator, read their rows from TMEM, turn them around
// in shared memory so that stores write whole 128-byte segments, and store the first 4096 columns as bf16 (the attention
// kernel's B operand) and the last 64 (zeta) as fp32.
// Bound by shared memory: a chunk's products read 48 KB of operands in 512 clocks of tensor pipe, TMA writes 32 KB and the
// masks 16 KB beside them.  Where a CTA has one tile it is a chain instead: masks, products, stores (see kOne).  Against two CTAs per SM of one tile each, which set up, filled their ring and drained one
// after the other: 512 (b, h) of 22 / 86 blocks 49.6 / 177 -> 41.4 / 119 us, 64 of 172 62 -> 43.5 us, 16 of 172 / 687 / 2147
// blocks 20.8 / 92 / 551 -> 18.8 / 80 / 548 us (4 of 2147, 7.8 tiles per SM: 140 -> 148 us).
#include <algorithm>

#include "common.cuh"
#include "sm100.cuh"

namespace lite3r {

namespace {

using namespace sm100;

constexpr int kStages = 4;
constexpr int kTileM = 128, kTileN = 256, kChunk = 64;
constexpr int kColTiles = (kSummaryRow + kTileN - 1) / kTileN;
constexpr int kBuilders = 2;    // warpgroups that expand masks (warps 4-11)
constexpr int kDrainers = 2;    // warpgroups that store results, one per accumulator (warps 12-19)
constexpr int kThreads = 128 + (kBuilders + kDrainers) * 128;
constexpr uint32_t kABytes = kTileM * kChunk * 2;   // 16 KB
constexpr uint32_t kBBytes = kChunk * kTileN * 2;   // 32 KB
constexpr uint32_t kOffA = 0;
constexpr uint32_t kOffB = kStages * kABytes;
constexpr uint32_t kOffOut = kOffB + kStages * kBBytes;  // 4 KB per storing warp
constexpr uint32_t kOffBar = kOffOut + kDrainers * 4 * 4096;
constexpr uint32_t kSmemBytes = kOffBar + 192;
constexpr uint32_t kTmemCols = 2 * kTileN;

struct Bars {
  uint64_t a_full[kStages], b_full[kStages], empty[kStages];
  uint64_t acc_full[2], acc_empty[2];
  uint32_t tmem_base;
  int abort;
};
static_assert(sizeof(Bars) <= 192, "barrier block");

struct AggregateParams {
  const signed char* cls;
  int nb, total_rows;
  int row_tiles;  // of one (b, h), or (flat) of all rows
  float inverse;  // of row_tiles, or (flat) of nb
  int tiles;      // row tiles times column tiles, of all (b, h)
  int cols;       // (masks at once) column tiles of a CTA
  __nv_bfloat16* g16;
  float* zeta;
  int* status;
};

// Rows and keys are numbered through all (b, h): row R = (b h) Nb + i, key (b h) Nb + j, the row numbers of the class
// matrix, the summaries and the outputs.  A tile is 128 consecutive rows and reduces over the keys of the (b, h) it
// touches.
struct Tile {
  int col, row0, row_limit, key0, chunks;
};
// n / d for n / d below 2^22 (a float quotient is then off by at most one).
__device__ __forceinline__ int divide(int n, int d, float inverse) {
  int q = static_cast<int>(static_cast<float>(n) * inverse);
  const int rest = n - q * d;
  q += rest >= d ? 1 : 0;
  return rest < 0 ? q - 1 : q;
}
template <bool kFlat>
__device__ __forceinline__ Tile tile_at(const AggregateParams& p, int id) {
  Tile t;
  const int rt = id / kColTiles;
  t.col = id - rt * kColTiles;
  int key_end;
  if (kFlat) {
    t.row0 = rt * kTileM;
    t.row_limit = p.total_rows;
    t.key0 = divide(t.row0, p.nb, p.inverse) * p.nb;
    key_end = divide(min(t.row0 + kTileM, p.total_rows) - 1, p.nb, p.inverse) * p.nb + p.nb;
  } else {
    const int bh = divide(rt, p.row_tiles, p.inverse);
    t.key0 = bh * p.nb;
    key_end = t.key0 + p.nb;
    t.row0 = t.key0 + (rt - bh * p.row_tiles) * kTileM;
    t.row_limit = key_end;
  }
  t.chunks = (key_end - t.key0 + kChunk - 1) / kChunk;
  return t;
}

// kOne: every CTA has one tile (masks at once: one or two), and what counts is how soon its products can start.
//   Inside a (b, h) the mask warpgroups then share every chunk's rows instead of taking every other chunk, which pays each
//   chunk's waits twice (16 heads of 687 blocks, eleven tiles to a CTA, 80 -> 99 us alone).
//   Through the boundaries, where a tile's keys fit into the ring, all its masks are made at once: operand tiles zeroed ahead
//   of the wait for the plan, then a one written for every marginal entry of the tile's 128 Nb class bytes, which lie one after
//   the other, four to a thread and turn.  Kernel alone, chunk by chunk / at once in us: 20 (b, h) of 15 blocks 8.3 / 6.2, 64 of
//   8 7.6 / 5.7, 64 of 15 9.1 / 6.6, 32 of 22 8.6 / 6.3 (the last mask was ready 5100 clocks after the plan, products and stores
//   take 4000 more); a whole pass of 4 x 5 (b, h) of 900 tokens 25.0 -> 21.6 us, of 2 x 16 of 1374 40.0 -> 37.5.  A CTA can
//   take two neighbouring column tiles of a row tile with the same masks, one per accumulator: where one each would be more than
//   one per SM (64 (b, h) of 22 blocks, 187 tiles: 17.5 -> 8.2 us from the end of the plan, a pass 71.5 -> 64.1), and where the SMs
//   left over are worth more to the attention kernel.
template <bool kFlat, bool kOne>
__global__ void __launch_bounds__(kThreads, 1)
aggregate_mma_kernel(const __grid_constant__ CUtensorMap map_s, const AggregateParams p) {
  extern __shared__ __align__(1024) uint8_t smem[];
  Bars* bars = reinterpret_cast<Bars*>(smem + kOffBar);
  volatile int* abort_flag = &bars->abort;
  if ((smem_u32(smem) & 1023u) != 0) {
    if (threadIdx.x == 0 && p.status != nullptr) atomicCAS(p.status, 0, 901);
    return;
  }
  const int warp = __shfl_sync(0xFFFFFFFFu, threadIdx.x >> 5, 0), lane = threadIdx.x & 31;
  constexpr bool kAtOnce = kFlat && kOne, kShare = !kFlat && kOne;
  // The CTA's tiles: first_id(), first_id() + step, ... below last_tile.  (first_id() reads the block's number in the roles themselves: from
  // a copy made ahead of them the compiler no longer sees that it is not negative, 1.8 KB of code and 0.3 us more.)
  const int groups = kAtOnce ? (kColTiles + p.cols - 1) / p.cols : 1, row_tile = blockIdx.x / groups;
  const int first_at_once = row_tile * kColTiles + (blockIdx.x - row_tile * groups) * p.cols;
  auto first_id = [&]() -> int { return kAtOnce ? first_at_once : blockIdx.x; };
  const int last_tile = kAtOnce ? min(first_at_once + p.cols, (row_tile + 1) * kColTiles) : p.tiles;
  const int step = kAtOnce ? 1 : static_cast<int>(gridDim.x);
  constexpr int kAtOnceThreads = (kBuilders + kDrainers) * 128;  // (the storing warps have nothing else to do yet)

  if (threadIdx.x == 0) {
    for (int s = 0; s < kStages; ++s) {
      mbar_init(&bars->a_full[s], kAtOnce ? kAtOnceThreads / 32 : kShare ? 4 * kBuilders : 4);  // one arrival per warp
      mbar_init(&bars->b_full[s], 1);
      mbar_init(&bars->empty[s], 1);
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(&bars->acc_full[b], 1);
      mbar_init(&bars->acc_empty[b], 4);
    }
    bars->abort = 0;
    mbar_fence_init();
  }
  if (warp == 1) {
    tmem_alloc(&bars->tmem_base, kTmemCols);
    tmem_relinquish();
  }
  if (kAtOnce && warp >= 4) {
    const uint32_t bytes = tile_at<kFlat>(p, first_id()).chunks * kABytes;
    for (uint32_t at = (threadIdx.x - 128) * 16; at < bytes; at += kAtOnceThreads * 16) sts128(smem_u32(smem + kOffA) + at, 0u, 0u, 0u, 0u);
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = bars->tmem_base;
  wait_for_prior_grid();
  // The attention kernel that follows needs this kernel's results only at the end of a tile: it may be scheduled as soon
  // as every CTA of this grid has its tensor memory and knows the summaries complete (it waits for this grid's completion
  // itself before it reads G and zeta).
  sm100::launch_dependents();

  if (kAtOnce && warp >= 4) {
    // The class bytes of the tile's rows, in the aligned words that hold them, two words to a thread and turn.
    const Tile t = tile_at<kFlat>(p, first_id());
    const char* const first = reinterpret_cast<const char*>(p.cls) + static_cast<long long>(t.row0) * p.nb;
    const int ahead = static_cast<int>(reinterpret_cast<intptr_t>(first) & 3);  // bytes of the first word before the tile's
    const int bytes = (min(t.row0 + kTileM, t.row_limit) - t.row0) * p.nb;
    const int words = (ahead + bytes + 3) >> 2;
    const int* const src = reinterpret_cast<const int*>(first - ahead);
    const int own0 = t.row0 - t.key0;  // row 0 of the tile inside its (b, h)
    for (int w = threadIdx.x - 128; w < words; w += 2 * kAtOnceThreads) {
      uint32_t four[2];
#pragma unroll
      for (int k = 0; k < 2; ++k) four[k] = w + k * kAtOnceThreads < words ? static_cast<uint32_t>(ldg_pinned(src + w + k * kAtOnceThreads)) : 0u;
#pragma unroll
      for (int k = 0; k < 2; ++k) {
        const int e0 = 4 * (w + k * kAtOnceThreads) - ahead;  // entry of the word's first byte
        int row = divide(max(e0, 0), p.nb, p.inverse), col = e0 - row * p.nb;
        int own = divide(own0 + row, p.nb, p.inverse) * p.nb;  // first key of the row's (b, h), from the tile's
#pragma unroll
        for (int b = 0; b < 4; ++b) {
          if (((four[k] >> (8 * b)) & 0xFFu) == 1u && e0 + b >= 0 && e0 + b < bytes) {
            const int key = own + col;
            sts16(smem_u32(smem + kOffA) + (key >> 6) * kABytes + row * 128 + ((((key >> 3) & 7) ^ (row & 7)) << 4) + (key & 7) * 2, 0x3F80u);
          }
          if (++col == p.nb) {
            col = 0;
            ++row;
            own += own0 + row == own + p.nb ? p.nb : 0;
          }
        }
      }
    }
    fence_proxy_async_smem();
    __syncwarp();
    if (lane == 0) mbar_arrive(&bars->a_full[0]);
  }
  if (warp == 0) {
    if (lane == 0) {
      tma_prefetch_desc(&map_s);
      bool ok = true;
      int kc = 0;  // chunks so far, through all tiles
      for (int id = first_id(); ok && id < last_tile; id += step) {
        const Tile t = tile_at<kFlat>(p, id);
        const int boxes = t.col == kColTiles - 1 ? 1 : kTileN / 64;
        for (int c = 0; c < t.chunks; ++c, ++kc) {
          const int st = kc % kStages;
          if (!(ok = mbar_wait(&bars->empty[st], ((kc / kStages) & 1) ^ 1, abort_flag, p.status, 401))) break;
          mbar_arrive_expect_tx(&bars->b_full[st], boxes * 8192);
          for (int q = 0; q < boxes; ++q)  // rows past the tensor are zero-filled by TMA
            tma_load_2d(smem + kOffB + st * kBBytes + q * 8192, &map_s, &bars->b_full[st], t.col * kTileN + q * 64, t.key0 + c * kChunk);
        }
      }
    }
  } else if (warp == 1) {
    if (lane == 0) {
      constexpr uint32_t idesc_all = instr_desc(1, kTileM, kTileN, 0, 1);  // bf16, A K-major, B MN-major
      constexpr uint32_t idesc_zeta = instr_desc(1, kTileM, 64, 0, 1);
      const uint32_t a_addr = smem_u32(smem + kOffA), b_addr = smem_u32(smem + kOffB);
      bool ok = true;
      int kc = 0, it = 0;
      for (int id = first_id(); ok && id < last_tile; id += step, ++it) {
        const Tile t = tile_at<kFlat>(p, id);
        const uint32_t idesc = t.col == kColTiles - 1 ? idesc_zeta : idesc_all;
        const uint32_t acc = tmem + (it & 1) * kTileN;
        if (!(ok = mbar_wait(&bars->acc_empty[it & 1], ((it >> 1) & 1) ^ 1, abort_flag, p.status, 406))) break;
        tc_fence_after();
        for (int c = 0; c < t.chunks; ++c, ++kc) {
          const int st = kc % kStages;
          const uint32_t par = (kc / kStages) & 1;
          ok = mbar_wait(&bars->b_full[st], par, abort_flag, p.status, 403) &&
               mbar_wait(&bars->a_full[kAtOnce ? 0 : st], kAtOnce ? 0 : par, abort_flag, p.status, 402);
          if (!ok) break;
          tc_fence_after();
          for (int kk = 0; kk < 4; ++kk) {
            const uint64_t a = smem_desc(a_addr + (kAtOnce ? c : st) * kABytes + kk * 32, 16, 1024, kSwizzle128);
            const uint64_t b = smem_desc(b_addr + st * kBBytes + kk * 2048, 8192, 1024, kSwizzle128);
            mma_f16(acc, a, b, idesc, (c > 0 || kk > 0) ? 1u : 0u);
          }
          mma_commit(&bars->empty[st]);
        }
        if (ok) mma_commit(&bars->acc_full[it & 1]);
      }
    }
  } else if (!kAtOnce && warp >= 4 && warp < 4 + 4 * kBuilders) {
    // Eight lanes take the eight groups of eight keys of one row, a warp four rows at a time, eight times (sharing: four
    // times).  The class bytes of a group travel as the three aligned words that hold them (rows start at any byte), requested a chunk of
    // the warpgroup's ahead, so that the latency hides behind the wait for the stage and the expansion: loads read whole
    // 64-byte rows, stores write whole 128-byte operand rows.
    constexpr int kRows = kShare ? kTileM / (16 * kBuilders) : kTileM / 16;  // of a lane
    constexpr int kStride = kShare ? 1 : kBuilders;                           // chunks from one of the warpgroup's to its next
    const int group = (warp - 4) >> 2, quarter = warp & 3;
    const int first = ((kShare ? group * 4 : 0) + quarter) * 4 * kRows + (lane >> 3);  // rows first, first + 4, ... of the tile
    const int kg = lane & 7;
    // the warpgroup's position: tile, its chunk, chunks so far
    struct At {
      Tile t;
      int id, c, kc, own;  // own (flat): first key of the (b, h) of row `first`
    };
    auto enter = [&](At& at) {
      at.t = tile_at<kFlat>(p, at.id);
      at.own = kFlat ? divide(min(at.t.row0 + first, p.total_rows - 1), p.nb, p.inverse) * p.nb : at.t.key0;
    };
    auto settle = [&](At& at) {  // carries a chunk number past the tile's end over to the next tiles
      while (at.id < p.tiles && at.c >= at.t.chunks) {
        at.c -= at.t.chunks;
        at.id += step;
        if (at.id < p.tiles) enter(at);
      }
    };
    // Calls fn(i, row, own) for the lane's rows: row (clamped to the tile's last) and first key of its (b, h).
    auto each_row = [&](const At& at, auto fn) {
      int own = at.own;
#pragma unroll
      for (int i = 0; i < kRows; ++i) {
        const int row = min(at.t.row0 + first + 4 * i, at.t.row_limit - 1);
        if constexpr (kFlat) {
          if (p.nb >= 4)
            own += row - own >= p.nb ? p.nb : 0;
          else
            own = divide(row, p.nb, p.inverse) * p.nb;
        }
        fn(i, row, own);
      }
    };
    // Whether every position of the chunk is a key of every row, and of none its last (a word behind it is then still
    // inside the class matrix).
    auto whole = [&](const At& at) { return !kFlat && (at.c + 1) * kChunk < p.nb; };
    const intptr_t cls0 = reinterpret_cast<intptr_t>(p.cls);
    auto fetch = [&](const At& at, uint32_t (&w)[kRows][3]) {
      if (at.id >= p.tiles) return;
      const int key = at.t.key0 + at.c * kChunk + 8 * kg;  // the group's first
      if (whole(at)) {
        each_row(at, [&](int i, int row, int own) {
          const uint32_t* const wp = reinterpret_cast<const uint32_t*>((cls0 + static_cast<long long>(row) * p.nb + (key - own)) & ~intptr_t(3));
#pragma unroll
          for (int k = 0; k < 3; ++k) w[i][k] = static_cast<uint32_t>(ldg_pinned(reinterpret_cast<const int*>(wp + k)));
        });
      } else {
        each_row(at, [&](int i, int row, int own) {
          const intptr_t addr = cls0 + static_cast<long long>(row) * p.nb + (key - own);
          const uint32_t* const wp = reinterpret_cast<const uint32_t*>(addr & ~intptr_t(3));
          const int at0 = key - own - static_cast<int>(addr & 3);  // key number in its row of the first word's first byte
#pragma unroll
          for (int k = 0; k < 3; ++k)  // words without a byte of the row are not read
            w[i][k] = at0 + 4 * k + 3 >= 0 && at0 + 4 * k < p.nb ? static_cast<uint32_t>(ldg_pinned(reinterpret_cast<const int*>(wp + k))) : 0u;
        });
      }
    };
    // A class byte (0 negligible, 1 marginal, 2 critical) picks the two bytes of its bf16 mask entry (0x3F80 for 1) from a
    // table: b0 + 256 b1 times 0x11 are the four nibbles b0, b0, b1, b1 of a byte permutation's selector.
    auto expand = [&](uint32_t bytes, uint32_t& o0, uint32_t& o1) {
      const uint32_t sel = bytes * 0x11u + 0x40404040u;
      o0 = __byte_perm(0x00008000u, 0x00003F00u, sel);
      o1 = __byte_perm(0x00008000u, 0x00003F00u, sel >> 16);
    };
    // the group's eight class bytes of each row; zero outside the row's keys, where the words hold other rows' bytes
    auto realign = [&](const At& at, const uint32_t (&w)[kRows][3], uint32_t (&m)[kRows][2]) {
      const int key = at.t.key0 + at.c * kChunk + 8 * kg;
      const bool all = whole(at);
      each_row(at, [&](int i, int row, int own) {
        const uint32_t shift = (static_cast<uint32_t>(cls0) + static_cast<uint32_t>(row) * static_cast<uint32_t>(p.nb) + static_cast<uint32_t>(key - own)) * 8u;
        m[i][0] = __funnelshift_r(w[i][0], w[i][1], shift);  // (of the shift the lower five bits count)
        m[i][1] = __funnelshift_r(w[i][1], w[i][2], shift);
        if (!all) {
          const int j = key - own;
          const int from = min(max(-j, 0), 8), to = min(max(p.nb - j, 0), 8);  // bytes from .. to - 1 stay
          const uint64_t keep = from < to ? (~0ull >> (64 - 8 * to)) & (~0ull << (8 * from)) : 0ull;
          m[i][0] &= static_cast<uint32_t>(keep);
          m[i][1] &= static_cast<uint32_t>(keep >> 32);
        }
      });
    };
    At at;
    at.id = blockIdx.x;
    at.c = at.kc = kShare ? 0 : group;
    if (at.id < p.tiles) enter(at);
    settle(at);
    uint32_t w[kRows][3];
    fetch(at, w);
    while (at.id < p.tiles) {
      uint32_t m[kRows][2];
      realign(at, w, m);
      const int st = at.kc % kStages;
      const uint32_t parity = ((at.kc / kStages) & 1) ^ 1;
      at.c += kStride;
      at.kc += kStride;
      settle(at);
      fetch(at, w);  // the warpgroup's next chunk
      if (!mbar_wait(&bars->empty[st], parity, abort_flag, p.status, 404)) break;
      const uint32_t base = smem_u32(smem + kOffA) + st * kABytes + first * 128;
#pragma unroll
      for (int i = 0; i < kRows; ++i) {
        uint32_t o[4];
        expand(m[i][0], o[0], o[1]);
        expand(m[i][1], o[2], o[3]);
        sts128(base + i * 512 + ((kg ^ ((first + 4 * i) & 7)) << 4), o[0], o[1], o[2], o[3]);
      }
      fence_proxy_async_smem();
      __syncwarp();
      if (lane == 0) mbar_arrive(&bars->a_full[st]);
    }
  } else if (warp >= 4 + 4 * kBuilders) {
    const int which = (warp - 4 - 4 * kBuilders) >> 2;  // accumulator
    const int quarter = warp & 3;
    const uint32_t lane_addr = tmem + which * kTileN + ((static_cast<uint32_t>(quarter) * 32u) << 16);
    // A thread owns one accumulator row, so direct stores would touch 32 different lines per instruction.  Each
    // warp turns its 32 rows x 128 bytes (64 bf16 columns) around in shared memory and stores whole 128-byte row
    // segments, four rows per instruction.
    uint8_t* const stage = smem + kOffOut + (warp - 4 - 4 * kBuilders) * 4096;
    int n = 0;  // tiles of this accumulator so far
    for (int id = first_id() + which * step; id < last_tile; id += 2 * step, ++n) {
      const Tile t = tile_at<kFlat>(p, id);
      if (!mbar_wait(&bars->acc_full[which], n & 1, abort_flag, p.status, 405)) break;
      tc_fence_after();
      const int row_w = t.row0 + quarter * 32;  // the warp's first row
      if (t.col < kColTiles - 1) {
#pragma unroll 1
        for (int pp = 0; pp < kTileN / 64; ++pp) {
          uint32_t pk[32];
          {
            uint32_t v0[32], v1[32];
            tmem_ld32(lane_addr + pp * 64, v0);
            tmem_ld32(lane_addr + pp * 64 + 32, v1);
            tmem_wait_ld();
#pragma unroll
            for (int x = 0; x < 16; ++x) {
              __nv_bfloat162 h = __floats2bfloat162_rn(__uint_as_float(v0[2 * x]), __uint_as_float(v0[2 * x + 1]));
              pk[x] = *reinterpret_cast<uint32_t*>(&h);
              h = __floats2bfloat162_rn(__uint_as_float(v1[2 * x]), __uint_as_float(v1[2 * x + 1]));
              pk[16 + x] = *reinterpret_cast<uint32_t*>(&h);
            }
          }
          if (pp == kTileN / 64 - 1) {  // the accumulator has been read
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(&bars->acc_empty[which]);
          }
#pragma unroll
          for (int ch = 0; ch < 8; ++ch)
            *reinterpret_cast<uint4*>(stage + lane * 128 + ((ch ^ (lane & 7)) << 4)) =
                make_uint4(pk[4 * ch], pk[4 * ch + 1], pk[4 * ch + 2], pk[4 * ch + 3]);
          __syncwarp();
          const int ch = lane & 7;
          __nv_bfloat16* const dst = p.g16 + static_cast<size_t>(row_w) * (kHeadDim * kHeadDim) + t.col * kTileN + pp * 64 + ch * 8;
#pragma unroll
          for (int k = 0; k < 8; ++k) {
            const int rr = 4 * k + (lane >> 3);
            const uint4 val = *reinterpret_cast<const uint4*>(stage + rr * 128 + ((ch ^ (rr & 7)) << 4));
            if (row_w + rr < t.row_limit) *reinterpret_cast<uint4*>(dst + static_cast<size_t>(rr) * (kHeadDim * kHeadDim)) = val;
          }
          __syncwarp();
        }
      } else {
        uint32_t v0[32], v1[32];
        tmem_ld32(lane_addr, v0);
        tmem_ld32(lane_addr + 32, v1);
        tmem_wait_ld();
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(&bars->acc_empty[which]);
        if (row_w + lane < t.row_limit) {
          float4* dst = reinterpret_cast<float4*>(p.zeta + static_cast<size_t>(row_w + lane) * kHeadDim);
#pragma unroll
          for (int q = 0; q < 8; ++q) {
            dst[q] = make_float4(__uint_as_float(v0[4 * q]), __uint_as_float(v0[4 * q + 1]), __uint_as_float(v0[4 * q + 2]),
                                 __uint_as_float(v0[4 * q + 3]));
            dst[8 + q] = make_float4(__uint_as_float(v1[4 * q]), __uint_as_float(v1[4 * q + 1]), __uint_as_float(v1[4 * q + 2]),
                                     __uint_as_float(v1[4 * q + 3]));
          }
        }
      }
    }
  }

  tc_fence_before();
  __syncthreads();
  linger_after_abort(abort_flag);
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc(tmem, kTmemCols);
  }
}

}  // namespace

lite3r_status launch_aggregate(const __nv_bfloat16* hws, const signed char* cls, const lite3r_shape& s, int nb,
                               int attention_ctas, int steps, __nv_bfloat16* g16, float* zeta, int* device_status,
                               cudaStream_t stream) {
  const uint64_t rows = static_cast<uint64_t>(s.batch) * s.heads * nb;
  CUtensorMap map_s;
  lite3r_status st = make_tensor_map_2d(&map_s, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, hws, kSummaryRow, rows, 64, 64,
                                        CU_TENSOR_MAP_SWIZZLE_128B);
  if (st != LITE3R_OK) return st;
  if (rows > 0x7FFFFFFFull - kTileM) return LITE3R_ERR_UNSUPPORTED;
  const int total_rows = static_cast<int>(rows), bh = s.batch * s.heads;
  int sms = 0;
  if ((st = sm_count(&sms)) != LITE3R_OK) return st;
  // Tiles through the (b, h) boundaries pay with a longer reduction (the keys of every (b, h) a tile touches) and with masks
  // that have to be cut to every row's own keys, tiles inside one (b, h) with padding when Nb is not a multiple of 128.
  // Estimate of either, in half microseconds: rounds of one tile per SM times the cost of a tile, 1.6 + one per chunk of 64
  // keys inside a (b, h), 2.8 + 1.5 per chunk through the boundaries and 1.2 per chunk once for the first masks; where the masks are
  // made at once, 1.2 + 1.4 per chunk + one per 32 blocks of a row (its class bytes) + 3 for a second column tile.  Measured, inside / flat in us: 16 (b, h) of 172 blocks
  // 14.5 / 21.7, of 687 80 / 121; 64 of 64 blocks 18.9 / 20.9, of 172 43.5 / 57.8; 512 of 22 blocks 71 / 37, of 64 97 / 97, of 86
  // 119 / 154; with the masks at once 4 (b, h) of 22 blocks 4.7 / 5.6, 10 of 15 5.6 / 6.2, 15 of 64 6.5 / 6.9, 16 of 22 6.3 / 6.2,
  // 12 of 32 6.2 / 5.9, 20 of 15 7.3 / 6.2, 32 of 22 8.5 / 6.3, 64 of 8 12.8 / 5.7.
  const long long row_tiles = ceil_div(total_rows, kTileM);
  const long long tiles_inside = static_cast<long long>(kColTiles) * bh * ceil_div(nb, kTileM), tiles_flat = kColTiles * row_tiles;
  if (tiles_inside > 0x7FFFFFFFll - 2 * sms || tiles_flat > 0x7FFFFFFFll - 2 * sms) return LITE3R_ERR_UNSUPPORTED;
  // chunks of a flat tile: one (b, h) when it starts and ends in the same one, else every (b, h) it touches
  double flat_chunks = 0.0;
  int most_chunks = 0;
  const long long probe = std::min<long long>(row_tiles, 4096);  // the pattern repeats; a prefix is representative
  for (long long t = 0; t < probe; ++t) {
    const int r0 = static_cast<int>(t) * kTileM;
    const int k0 = r0 / nb * nb, k1 = (std::min(r0 + kTileM, total_rows) - 1) / nb * nb + nb;
    flat_chunks += ceil_div(k1 - k0, kChunk);
    most_chunks = std::max(most_chunks, ceil_div(k1 - k0, kChunk));
  }
  flat_chunks /= static_cast<double>(probe);
  auto rounds = [](long long tiles, long long ctas) { return static_cast<double>((tiles + ctas - 1) / ctas); };
  // A CTA of this kernel fills its SM.  Where the whole attention grid finds room on the SMs that are left, it runs beside this
  // one up to the end of its critical blocks, and what counts is the longer of the two instead of their sum; where a part of it
  // does, 0.7 of that share of the shorter one is saved.  That part of the attention kernel takes 4.5 half microseconds (launch, set-up,
  // phi(Q)) and 1.4 / 1.65 / 2 per step with one / two / three of its CTAs on an SM.  All forms are tried on all SMs, and those of any
  // grid also on the SMs that three attention CTAs to an SM leave (taken when that is a microsecond shorter).  A whole pass in
  // us: 15 (b, h) of 3001 tokens in blocks of 128 on all SMs 43.6, on 28 40.6; tiles inside the (b, h) / as chosen here: 16 heads of
  // 1374 tokens 33.3 / 26.0, 8 of 629 22.6 / 20.5, of 1374 28.4 / 22.6, of 3000 28.0 / 24.9, 16 of 832 24.9 / 21.9, with room for a part
  // 12 of 4748 in blocks of 128 46.3 / 43.2, 16 of 4122 53.4 / 51.2.
  struct Choice {
    bool flat;
    int cols;  // masks at once: column tiles to a CTA; else 0
    long long grid;
    double own, both;
  };
  auto choice = [&](bool flat, int cols, long long ctas) {
    Choice c{flat, cols, 0, 0.0, 0.0};
    if (cols > 0) {
      c.grid = row_tiles * ceil_div(kColTiles, cols);
      c.own = c.grid <= ctas && most_chunks <= kStages ? 1.2 + 1.4 * most_chunks + nb / 32.0 + 3.0 * (cols - 1) : 1e30;
    } else {
      c.grid = std::min(ctas, flat ? tiles_flat : tiles_inside);
      c.own = flat ? rounds(tiles_flat, ctas) * (2.8 + 1.5 * flat_chunks) + 1.2 * flat_chunks : rounds(tiles_inside, ctas) * (1.6 + ceil_div(nb, kChunk));
    }
    const long long left = sms - c.grid;
    const bool beside = left * kAttentionCtasPerSm >= attention_ctas;
    const long long per_sm = beside ? (attention_ctas + left - 1) / left : kAttentionCtasPerSm;
    const double other = steps == 0 ? 0.0 : 4.5 + steps * (per_sm <= 1 ? 1.4 : per_sm == 2 ? 1.65 : 2.0);
    c.both = beside ? std::max(c.own, other) : c.own + other - 0.7 * std::min(c.own, other) * std::max(left, 0ll) / sms;
    return c;
  };
  Choice best = choice(false, 0, sms);
  for (const Choice& c : {choice(true, 0, sms), choice(true, 1, sms), choice(true, 2, sms)})
    if (c.both < best.both || (c.both == best.both && c.own < best.own)) best = c;
  const long long spare = sms - ceil_div(attention_ctas, kAttentionCtasPerSm);
  if (steps > 0 && spare > 0) {
    for (const Choice& c : {choice(false, 0, spare), choice(true, 0, spare)})
      if (c.both + 2.0 < best.both) best = c;
  }
  const bool flat = best.flat;
  AggregateParams p;
  p.cls = cls;
  p.nb = nb;
  p.total_rows = total_rows;
  p.row_tiles = flat ? static_cast<int>(row_tiles) : ceil_div(nb, kTileM);
  p.inverse = 1.f / static_cast<float>(flat ? nb : p.row_tiles);
  p.tiles = static_cast<int>(flat ? tiles_flat : tiles_inside);
  p.g16 = g16;
  p.zeta = zeta;
  p.status = device_status;
  p.cols = best.cols;
  auto* const kernel = flat ? (best.cols > 0 ? aggregate_mma_kernel<true, true> : aggregate_mma_kernel<true, false>)
                            : (p.tiles == best.grid ? aggregate_mma_kernel<false, true> : aggregate_mma_kernel<false, false>);
  st = ensure_dynamic_smem(kernel, static_cast<int>(kSmemBytes));
  if (st != LITE3R_OK) return st;
  return launch_dependent(kernel, dim3(static_cast<unsigned>(best.grid)), kThreads, static_cast<int>(kSmemBytes), stream,
                          map_s, p);
}

}  // namespace lite3r
