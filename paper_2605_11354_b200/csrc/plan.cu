// K2: pooled scores and row-wise top-k block classification (the score and TopKMask steps of Algorithm 1 on block means).
//
// The pooled mean of block i is colsum_i * 2^-9 * scale_i / valid_i with colsum an exact integer vector, so
//   s_ij = (colsum^Q_i . colsum^K_j) * [scale^K_j / valid_j] * [scale^Q_i / (valid_i * 8 * 2^18)].
// The last bracket is a positive constant of row i and cannot change the ranking inside the row, so the
// kernel ranks t_ij = (integer dot product, exact in fp64 below 2^53) * scale^K_j / valid_j.  Two fp64
// roundings separate t_ij from the exact value; the ranking is therefore the exact one except between
// scores that agree to ~1e-15 relative.  Ranking order: score descending, then key-block index ascending.
//
// plan_kernel: one CTA of R warps handles R consecutive query blocks (rows) of one (b, h); R = 8 for rows of up to 80
// blocks, R = 1 for those too long for plan_compact_kernel.
//   Phase A (whole CTA): the scores of the R rows against all key blocks, kept in shared memory as order-preserving
//     64-bit keys.  R = 8: fp64 tensor-core products (m8n8k4) fed with the int32 column sums straight from global
//     memory, no staging and no barrier.  R = 1: 32 key blocks at a time staged in shared memory as doubles, one to a lane.
//   Phase B (one warp per row): "the k best of the row".  A histogram over 256 buckets that are linear in the score
//     places the k-th best in a bucket of usually a handful of keys; those are listed by index and a
//     most-significant-digit-first radix select over their 64-bit keys (8-bit digits placed at the highest bit on
//     which the remaining candidates differ, per-warp histogram in shared memory) decides between them: it yields a
//     key prefix such that every entry above it is selected, and of the entries equal to it the first `take` in
//     index order are.  That is exactly the total order (score descending, index ascending), at O(Nb) work per
//     row.  Two selections give the classes: the best k_crit are critical, the best Nb - k_neg are
//     critical-or-marginal.
//   Phase C (same warp): class row and ascending index lists, written with ballot prefix sums.
//
// late_wait: the launch before this one in the stream (the summaries) neither writes what this kernel reads nor touches
// what it writes, and has itself waited for everything that does: the two run side by side, and this kernel waits for the
// other one's completion only before it ends, so that its own completion stands for both.  Until that wait it reads the
// column sums and scales on the word of the summaries' wait (sm100.cuh, "reading ahead of the own wait"): it may
// not read anything that the launch before it writes.
#include <atomic>
#include <type_traits>

#include "common.cuh"
#include "sm100.cuh"

namespace lite3r {

namespace {

constexpr int kStaged = 32;           // key blocks staged per pass (R = 1)
constexpr int kLongestRow = 24316;    // blocks; longer sequences are refused
constexpr int kPitch = kHeadDim + 4;  // staged row pitch in doubles: 16-byte aligned rows; 8-byte reads of four consecutive
                                      // values from four (eight) rows and 16-byte reads of eight rows fall on different banks

// Maps a double to an unsigned key with the same order (larger double -> larger key).
__device__ __forceinline__ unsigned long long order_key(double v) {
  const unsigned long long u = static_cast<unsigned long long>(__double_as_longlong(v));
  return (u >> 63) ? ~u : (u | 0x8000000000000000ull);
}

struct Selection {
  // An entry is selected when its bucket is above `bucket`; inside that bucket when (key & mask) > prefix, and of the
  // entries with (key & mask) == prefix the first `take` in index order.
  unsigned long long prefix, mask;
  int take, bucket;
};

constexpr int kBuckets = 256;
constexpr int kRankMax = 64;     // rows of up to this many blocks are ranked by comparing all pairs of entries
constexpr int kMaxListed = 128;  // candidates of a threshold bucket kept as an index list; fuller buckets are re-scanned

// Position of rank `remaining` (1-based, counted from the top bin down) in a 256-bin histogram: the bin holding it, the
// entries in the bins above and the size of that bin.  Warp-collective; lane L owns bins 255-8L .. 248-8L.
struct Located {
  int bin, above, size;
};
__device__ __forceinline__ Located locate(const unsigned int* hist, int remaining, int lane) {
  int cnt[8], tot = 0;
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    cnt[i] = static_cast<int>(hist[255 - 8 * lane - i]);
    tot += cnt[i];
  }
  int incl = tot;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int up = __shfl_up_sync(0xFFFFFFFFu, incl, o);
    if (lane >= o) incl += up;
  }
  const int excl = incl - tot;
  const bool mine = excl < remaining && remaining <= incl;
  Located r = {0, 0, 0};
  if (mine) {
    int run = excl;
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      if (r.size == 0 && run + cnt[i] >= remaining) {
        r.bin = 255 - 8 * lane - i;
        r.above = run;
        r.size = cnt[i];
      }
      run += cnt[i];
    }
  }
  const int src = __ffs(__ballot_sync(0xFFFFFFFFu, mine)) - 1;
  r.bin = __shfl_sync(0xFFFFFFFFu, r.bin, src);
  r.above = __shfl_sync(0xFFFFFFFFu, r.above, src);
  r.size = __shfl_sync(0xFFFFFFFFu, r.size, src);
  return r;
}

// The k best (largest key, then lowest position) of the m candidates cand(0) .. cand(m - 1), 0 < k < m as far as the
// valid ones go: cand(c, key) says whether candidate c takes part and gives its key.  Most-significant-digit-first
// radix select over the 64-bit keys, 8-bit digits placed at the highest bit on which the remaining candidates still
// differ (keys of one row share their sign and leading exponent bits, so fixed digit positions would spend whole
// passes on digits that are equal for everyone).  Warp-collective; hist is this warp's 256 counters.
template <class Cand>
__device__ void radix_select(Cand cand, int m, int k, unsigned int* hist, int lane, Selection& s) {
  unsigned long long prefix = 0ull, mask = 0ull;
  int remaining = k;
  while (true) {
    unsigned long long all_and = ~0ull, all_or = 0ull;
    for (int c = lane; c < m; c += 32) {
      unsigned long long key;
      if (cand(c, key) && (key & mask) == prefix) {
        all_and &= key;
        all_or |= key;
      }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      all_and &= __shfl_xor_sync(0xFFFFFFFFu, all_and, o);
      all_or |= __shfl_xor_sync(0xFFFFFFFFu, all_or, o);
    }
    const unsigned long long diff = all_and ^ all_or;
    if (diff == 0ull) {  // all candidates are equal: the first `remaining` of them by index are selected
      prefix = all_and;
      mask = ~0ull;
      break;
    }
    const int hb = 63 - __clzll(static_cast<long long>(diff));      // highest differing bit
    const int shift = hb >= 7 ? hb - 7 : 0;                          // digit = bits shift .. shift+7
    const unsigned long long above_hb = hb == 63 ? 0ull : ~((2ull << hb) - 1ull);
    prefix |= all_and & above_hb & ~mask;                            // the common leading bits join the prefix
    mask |= above_hb;
#pragma unroll
    for (int b = 0; b < 8; ++b) hist[lane + 32 * b] = 0u;
    __syncwarp();
    for (int c = lane; c < m; c += 32) {
      unsigned long long key;
      if (cand(c, key) && (key & mask) == prefix) atomicAdd(&hist[static_cast<unsigned int>(key >> shift) & 255u], 1u);
    }
    __syncwarp();
    const Located at = locate(hist, remaining, lane);
    remaining -= at.above;
    const unsigned long long field = 0xFFull << shift;
    prefix = (prefix & ~field) | (static_cast<unsigned long long>(at.bin) << shift);
    mask |= field;
    __syncwarp();
    if (at.size == remaining || shift == 0) break;  // the whole bin is selected, or every bit has been decided
  }
  s.prefix = prefix;
  s.mask = mask;
  s.take = remaining;
}

// The same for at most 64 candidates, all of which take part: every candidate is compared with all others (one or two per
// lane, the others by shuffle), and the key of the one with exactly k - 1 better ones is the threshold.  A threshold
// bucket usually holds a dozen candidates; the radix select spends some 250 instructions on every digit, and two to
// four digits, whatever their number.
template <int kPerLane, class Key>
__device__ void rank_select_n(Key key_of, int m, int k, int lane, Selection& s) {
  unsigned long long key[kPerLane];
  int rank[kPerLane];
#pragma unroll
  for (int x = 0; x < kPerLane; ++x) {
    key[x] = lane + 32 * x < m ? key_of(lane + 32 * x) : 0ull;
    rank[x] = 0;
  }
#pragma unroll
  for (int y = 0; y < kPerLane; ++y) {
    const int end = min(m - 32 * y, 32);
#pragma unroll 1
    for (int o = 0; o < end; ++o) {
      const unsigned long long other = __shfl_sync(0xFFFFFFFFu, key[y], o);
      // an equal key goes first when its candidate does: other >= key, that is other > key - 1 (keys are never 0)
#pragma unroll
      for (int x = 0; x < kPerLane; ++x) rank[x] += other > key[x] - (o + 32 * y < lane + 32 * x ? 1 : 0) ? 1 : 0;
    }
  }
  unsigned long long threshold = 0ull;
#pragma unroll
  for (int x = 0; x < kPerLane; ++x) {
    const unsigned hit = __ballot_sync(0xFFFFFFFFu, lane + 32 * x < m && rank[x] == k - 1);
    if (hit != 0u) threshold = __shfl_sync(0xFFFFFFFFu, key[x], __ffs(hit) - 1);
  }
  int above = 0;
#pragma unroll
  for (int x = 0; x < kPerLane; ++x) above += __popc(__ballot_sync(0xFFFFFFFFu, lane + 32 * x < m && key[x] > threshold));
  s.prefix = threshold;
  s.mask = ~0ull;
  s.take = k - above;
}
template <class Key>
__device__ void rank_select(Key key_of, int m, int k, int lane, Selection& s) {
  if (m <= 32)
    rank_select_n<1>(key_of, m, k, lane, s);
  else
    rank_select_n<2>(key_of, m, k, lane, s);
}

// The k best (largest key, then lowest index) of keys[0..n).  First a histogram over 256 buckets that are linear in
// the score (bucket(j), any monotone map of the score to 0..255, computed from a single-precision copy): it places
// the k-th best in one bucket with usually a handful of entries, listed by index (idx, at most kMaxListed) for the
// radix select that decides between them.  hist must hold the bucket counts of the row on entry.  Warp-collective.
template <class Bucket>
__device__ Selection select_top(const unsigned long long* keys, Bucket bucket, int n, int k, unsigned int* hist,
                                const unsigned int* bucket_hist, unsigned short* idx, int lane) {
  Selection s;
  s.prefix = 0ull;
  s.mask = 0ull;
  s.take = 0;
  if (k <= 0) {  // nothing selected
    s.bucket = kBuckets;
    return s;
  }
  if (k >= n) {  // everything selected
    s.bucket = -1;
    return s;
  }
  const Located at = locate(bucket_hist, k, lane);
  s.bucket = at.bin;
  const int remaining = k - at.above;
  if (remaining == at.size) {  // the whole bucket is selected
    s.take = at.size;
    return s;
  }
  if (at.size <= kMaxListed) {
    const unsigned below = (1u << lane) - 1u;
    int listed = 0;
    for (int j0 = 0; j0 < n; j0 += 32) {
      const int j = j0 + lane;
      const bool is = j < n && bucket(j) == at.bin;
      const unsigned b = __ballot_sync(0xFFFFFFFFu, is);
      if (is) idx[listed + __popc(b & below)] = static_cast<unsigned short>(j);
      listed += __popc(b);
    }
    __syncwarp();
    if (at.size <= 64) {
      rank_select([&](int c) { return keys[idx[c]]; }, at.size, remaining, lane, s);
    } else {
      radix_select([&](int c, unsigned long long& key) {
        key = keys[idx[c]];
        return true;
      }, at.size, remaining, hist, lane, s);
    }
  } else {
    radix_select([&](int c, unsigned long long& key) {
      key = keys[c];
      return bucket(c) == at.bin;
    }, n, remaining, hist, lane, s);
  }
  return s;
}

template <int R>
__global__ void __launch_bounds__(R * 32) plan_kernel(const int* __restrict__ q_colsum, const int* __restrict__ k_colsum,
                                                       const float* __restrict__ k_scales, int tokens, int block,
                                                       int nb, int k_crit, int k_marg, int k_neg, int late_wait,
                                                       signed char* __restrict__ cls, int* __restrict__ crit_idx,
                                                       int* __restrict__ marg_idx) {
  constexpr int kThreads = R * 32;
  constexpr bool kDirect = R >= 8;                // column sums straight from global memory into the fp64 MMA
  constexpr int kTiles = kDirect ? R / 8 : 1;     // 8-row MMA tiles per warp
  static_assert(kDirect || R == 1, "one row per CTA, or whole 8-row tiles");

  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int pitch = (nb + 1) & ~1;  // key-row pitch: keeps everything behind the keys 16-byte aligned
  unsigned long long* s_key = reinterpret_cast<unsigned long long*>(smem_raw);        // [R][pitch]
  unsigned int* s_hist = reinterpret_cast<unsigned int*>(s_key + static_cast<size_t>(R) * pitch);  // [R][2][256]
  unsigned short* s_idx = reinterpret_cast<unsigned short*>(s_hist + R * 2 * kBuckets);            // [R][2][kMaxListed]
  float2* s_range = reinterpret_cast<float2*>(s_idx + R * 2 * kMaxListed);                         // [R][R]     (direct)
  unsigned char* s_bkt = reinterpret_cast<unsigned char*>(s_range + R * R);                        // [R][pitch] (direct)

  const int row_tiles = (nb + R - 1) / R;
  const int bh = blockIdx.x / row_tiles;
  const int i0 = (blockIdx.x % row_tiles) * R;
  const int warp = threadIdx.x >> 5;
  const int lane = threadIdx.x & 31;
  const size_t bh_rows = static_cast<size_t>(bh) * nb;

  if (!late_wait) sm100::wait_for_prior_grid();
  sm100::launch_dependents();
  if constexpr (kDirect) {
    // Phase A, R rows x 8 key blocks per warp and step as fp64 tensor-core products (m8n8k4, 16 k-steps over the 64
    // columns, one 8-row tile after the other against the same B values): the integer products and sums stay below
    // 2^53, so the result is the exact dot product whatever the order.  The product does not care which column sits
    // at which k index as long as A and B agree, so lane (g, t) supplies columns 16 t .. 16 t + 15 of its row (q
    // row g of each tile for A, key block g of the warp's eight for B): 64 contiguous bytes of the int32 column
    // sums, read straight from global memory (L2) one step ahead, with no staging and no barrier.  Every CTA
    // streams all column sums of its (b, h) once, which is what bounds this phase: hence as many rows per CTA as
    // shared memory allows.  int32 -> fp64 is exact and takes one xor and one subtraction: the double with high
    // word 0x43300000 and low word v ^ 2^31 is 2^52 + 2^31 + v.
    const int g = lane >> 2, t4 = lane & 3;
    auto widen = [](int v) {
      return __hiloint2double(0x43300000, v ^ static_cast<int>(0x80000000u)) - 4503601774854144.0;
    };
    // `local` is a block index inside the (b, h); past the end the last block is read instead (its products land
    // in rows or columns that are never stored), which keeps the loads free of predicates and zero fills
    auto load16 = [&](const int* base, int local, int4 dst[4]) {
      const int4* src = reinterpret_cast<const int4*>(base + (bh_rows + min(local, nb - 1)) * kHeadDim + 16 * t4);
#pragma unroll
      for (int q = 0; q < 4; ++q) dst[q] = __ldg(src + q);
    };
    double q_frag[kTiles][16];
#pragma unroll
    for (int m = 0; m < kTiles; ++m) {
      int4 qv[4];
      load16(q_colsum, i0 + 8 * m + g, qv);
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        q_frag[m][4 * q] = widen(qv[q].x);
        q_frag[m][4 * q + 1] = widen(qv[q].y);
        q_frag[m][4 * q + 2] = widen(qv[q].z);
        q_frag[m][4 * q + 3] = widen(qv[q].w);
      }
    }
    // the scales of the two key blocks whose scores the lane ends up with travel with the column sums
    auto load_scales = [&](int j, float dst[2]) {
#pragma unroll
      for (int x = 0; x < 2; ++x) dst[x] = __ldg(k_scales + bh_rows + min(j + x, nb - 1));
    };
    int4 nxt[4];
    float nxt_ks[2];
    load16(k_colsum, warp * 8 + g, nxt);
    load_scales(warp * 8 + 2 * t4, nxt_ks);
    float lo[kTiles], hi[kTiles];  // range of the scores of row 8 m + g, as far as this lane sees them
#pragma unroll
    for (int m = 0; m < kTiles; ++m) {
      lo[m] = INFINITY;
      hi[m] = -INFINITY;
    }
    const bool block_pow2 = (block & (block - 1)) == 0;
    const double inv_block = 1.0 / static_cast<double>(block);
    for (int j0 = warp * 8; j0 < nb; j0 += 8 * R) {
      int4 cur[4];
#pragma unroll
      for (int q = 0; q < 4; ++q) cur[q] = nxt[q];
      const float cur_ks[2] = {nxt_ks[0], nxt_ks[1]};
      if (j0 + 8 * R < nb) {
        load16(k_colsum, j0 + 8 * R + g, nxt);
        load_scales(j0 + 8 * R + 2 * t4, nxt_ks);
      }
      // per tile two accumulation chains (even / odd k-steps), which hide the MMA latency; four were slower
      constexpr int kChains = 2;
      double c[kTiles][kChains][2];
#pragma unroll
      for (int m = 0; m < kTiles; ++m) {
#pragma unroll
        for (int n = 0; n < kChains; ++n) c[m][n][0] = c[m][n][1] = 0.0;
      }
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const int vals[4] = {cur[q].x, cur[q].y, cur[q].z, cur[q].w};
#pragma unroll
        for (int y = 0; y < 4; ++y) {
          const int st = 4 * q + y;
          const double bv = widen(vals[y]);
#pragma unroll
          for (int m = 0; m < kTiles; ++m) {
            asm volatile("mma.sync.aligned.m8n8k4.row.col.f64.f64.f64.f64 {%0, %1}, {%2}, {%3}, {%0, %1};"
                         : "+d"(c[m][st % kChains][0]), "+d"(c[m][st % kChains][1])
                         : "d"(q_frag[m][st]), "d"(bv));
          }
        }
      }
      // the lane ends with the scores of rows 8 m + g against key blocks 2 t and 2 t + 1 of the warp's eight
#pragma unroll
      for (int x = 0; x < 2; ++x) {
        const int j = j0 + 2 * t4 + x;
        if (j < nb) {
          const int valid = min(block, tokens - j * block);
          const double ks = static_cast<double>(cur_ks[x]);
          const bool full = valid == block && block_pow2;
#pragma unroll
          for (int m = 0; m < kTiles; ++m) {
            // a full block of 2^n tokens divides exactly by a multiplication; only the last block can be shorter
            const double num = (c[m][0][x] + c[m][1][x]) * ks;
            const double tt = (full ? num * inv_block : num / static_cast<double>(valid)) + 0.0;
            s_key[static_cast<size_t>(8 * m + g) * pitch + j] = order_key(tt);
            // range of the row in single precision, for the bucket histogram of the selection
            const float tf = static_cast<float>(tt);
            lo[m] = fminf(lo[m], tf);
            hi[m] = fmaxf(hi[m], tf);
          }
        }
      }
    }
#pragma unroll
    for (int m = 0; m < kTiles; ++m) {
#pragma unroll
      for (int o = 1; o <= 2; o <<= 1) {
        lo[m] = fminf(lo[m], __shfl_xor_sync(0xFFFFFFFFu, lo[m], o));
        hi[m] = fmaxf(hi[m], __shfl_xor_sync(0xFFFFFFFFu, hi[m], o));
      }
      if (t4 == 0) s_range[warp * R + 8 * m + g] = make_float2(lo[m], hi[m]);
    }
  } else {
    // Phase A for one very long row: the column sums of 32 key blocks at a time are staged in shared memory as doubles
    // (fetched with 16-byte loads one pass ahead), and a lane takes one of them.  The pitch of 68 doubles keeps the
    // 16-byte reads of eight staged rows on different banks.
    double* s_q = reinterpret_cast<double*>(s_idx + R * 2 * kMaxListed);  // [kPitch]
    double* s_k = s_q + kPitch;                                           // [kStaged][kPitch]
    for (int d = lane; d < kHeadDim; d += 32) s_q[d] = static_cast<double>(q_colsum[(bh_rows + i0) * kHeadDim + d]);
    constexpr int kLoads = kStaged * (kHeadDim / 4) / kThreads;  // int4 loads per thread and pass
    int4 pre[kLoads];
    auto prefetch = [&](int j0) {
      const int4* src = reinterpret_cast<const int4*>(k_colsum + (bh_rows + j0) * kHeadDim);
      const int n4 = min(kStaged, nb - j0) * (kHeadDim / 4);
#pragma unroll
      for (int q = 0; q < kLoads; ++q) {
        const int v = lane + q * kThreads;
        pre[q] = v < n4 ? __ldg(src + v) : make_int4(0, 0, 0, 0);
      }
    };
    prefetch(0);
    for (int j0 = 0; j0 < nb; j0 += kStaged) {
      __syncthreads();
#pragma unroll
      for (int q = 0; q < kLoads; ++q) {
        const int v = lane + q * kThreads;
        double* dst = s_k + (v / (kHeadDim / 4)) * kPitch + (v % (kHeadDim / 4)) * 4;
        *reinterpret_cast<double2*>(dst) = make_double2(static_cast<double>(pre[q].x), static_cast<double>(pre[q].y));
        *reinterpret_cast<double2*>(dst + 2) = make_double2(static_cast<double>(pre[q].z), static_cast<double>(pre[q].w));
      }
      if (j0 + kStaged < nb) prefetch(j0 + kStaged);
      __syncthreads();
      const int j = j0 + lane;
      if (j < nb) {
        const double2* kr = reinterpret_cast<const double2*>(s_k + lane * kPitch);
        const double2* qr = reinterpret_cast<const double2*>(s_q);
        double acc = 0.0;
#pragma unroll 8
        for (int d2 = 0; d2 < kHeadDim / 2; ++d2) {
          const double2 kv = kr[d2], qv = qr[d2];
          acc = fma(qv.x, kv.x, acc);
          acc = fma(qv.y, kv.y, acc);
        }
        const int valid = min(block, tokens - j * block);
        const double t = acc * static_cast<double>(k_scales[bh_rows + j]) / static_cast<double>(valid) + 0.0;
        s_key[j] = order_key(t);
      }
    }
  }
  __syncthreads();
  const int i = i0 + warp;
  if (i >= nb) return;

  const unsigned long long* keys = s_key + static_cast<size_t>(warp) * pitch;
  if (kDirect && nb <= kRankMax) {
    // Short rows: the rank of every entry by comparing it with all others (one or two entries per lane, the others read
    // as broadcasts).  At 22 blocks that is a tenth of what the histogram and the radix select below cost, whose 256
    // counters alone take longer to clear and scan than the row has entries.
    unsigned long long key[2];
    int rank[2] = {0, 0};
#pragma unroll
    for (int x = 0; x < 2; ++x) key[x] = lane + 32 * x < nb ? keys[lane + 32 * x] : 0ull;
    for (int o = 0; o < nb; ++o) {
      const unsigned long long other = keys[o];
#pragma unroll
      for (int x = 0; x < 2; ++x) rank[x] += (other > key[x] || (other == key[x] && o < lane + 32 * x)) ? 1 : 0;
    }
    const size_t row = bh_rows + i;
    int n_crit = 0, n_marg = 0;
    const unsigned below = (1u << lane) - 1u;
#pragma unroll
    for (int x = 0; x < 2; ++x) {
      const int j = lane + 32 * x;
      const int c = j >= nb ? -1 : (rank[x] < k_crit ? 2 : (rank[x] < nb - k_neg ? 1 : 0));
      if (j < nb) cls[row * nb + j] = static_cast<signed char>(c);
      const unsigned m_crit = __ballot_sync(0xFFFFFFFFu, c == 2), m_marg = __ballot_sync(0xFFFFFFFFu, c == 1);
      if (c == 2) crit_idx[row * k_crit + n_crit + __popc(m_crit & below)] = j;
      if (c == 1 && marg_idx != nullptr) marg_idx[row * k_marg + n_marg + __popc(m_marg & below)] = j;
      n_crit += __popc(m_crit);
      n_marg += __popc(m_marg);
    }
    if (late_wait) sm100::wait_for_prior_grid();
    return;
  }

  // Phase B
  unsigned int* hist = s_hist + warp * 2 * kBuckets;  // radix digits; the second half holds the bucket counts
  unsigned int* bucket_hist = hist + kBuckets;
  // Buckets linear in the score between the row's extremes; with one row per CTA (very long sequences) there are no bucket
  // bytes and every key falls into bucket 0, which leaves the whole selection to the radix select.
  float lo = 0.f, scale = 0.f;
  unsigned char* bkt = s_bkt + static_cast<size_t>(warp) * pitch;
  if constexpr (kDirect) {
    float2 range = lane < R ? s_range[lane * R + warp] : make_float2(INFINITY, -INFINITY);
#pragma unroll
    for (int o = 1; o < R; o <<= 1) {
      range.x = fminf(range.x, __shfl_xor_sync(0xFFFFFFFFu, range.x, o));
      range.y = fmaxf(range.y, __shfl_xor_sync(0xFFFFFFFFu, range.y, o));
    }
    range.x = __shfl_sync(0xFFFFFFFFu, range.x, 0);
    range.y = __shfl_sync(0xFFFFFFFFu, range.y, 0);
    lo = range.x;
    scale = range.y > range.x ? 255.5f / (range.y - range.x) : 0.f;
  }
  auto bucket = [&](int j) -> int {
    if constexpr (!kDirect) return 0;
    return bkt[j];
  };
#pragma unroll
  for (int b = 0; b < 8; ++b) bucket_hist[lane + 32 * b] = 0u;
  __syncwarp();
  for (int j = lane; j < nb; j += 32) {
    int b = 0;
    if constexpr (kDirect) {
      // key -> double -> float: every step keeps the order (weakly), which is all the buckets need
      const unsigned long long key = keys[j];
      const unsigned long long u = (key >> 63) ? (key & 0x7FFFFFFFFFFFFFFFull) : ~key;
      const float tf = static_cast<float>(__longlong_as_double(static_cast<long long>(u)));
      b = min(kBuckets - 1, max(0, __float2int_rz((tf - lo) * scale)));
      bkt[j] = static_cast<unsigned char>(b);
    }
    atomicAdd(&bucket_hist[b], 1u);
  }
  __syncwarp();
  unsigned short* idx = s_idx + warp * 2 * kMaxListed;
  const Selection sc = select_top(keys, bucket, nb, k_crit, hist, bucket_hist, idx, lane);
  const Selection sm = select_top(keys, bucket, nb, nb - k_neg, hist, bucket_hist, idx + kMaxListed, lane);

  // Phase C
  const size_t row = bh_rows + i;
  signed char* out_cls = cls + row * nb;
  int* crit_row = crit_idx + row * k_crit;  // where the row's lists go on
  int* marg_row = marg_idx != nullptr ? marg_idx + row * k_marg : nullptr;
  int tie_c = 0, tie_m = 0;
  const unsigned below = (1u << lane) - 1u;
#pragma unroll 2
  for (int j0 = 0; j0 < nb; j0 += 32) {
    const int j = j0 + lane;
    const bool in = j < nb;
    const int bk = in ? bucket(j) : -2;
    bool sel_c = in && bk > sc.bucket, sel_m = in && bk > sm.bucket;
    // the 64-bit keys only matter for entries inside one of the two threshold buckets: most groups of 32 have none
    if (__any_sync(0xFFFFFFFFu, bk == sc.bucket || bk == sm.bucket)) {
      const unsigned long long key = in ? keys[j] : 0ull;
      const unsigned long long kc = key & sc.mask, km = key & sm.mask;
      const bool eq_c = bk == sc.bucket && kc == sc.prefix, eq_m = bk == sm.bucket && km == sm.prefix;
      const unsigned b_eq_c = __ballot_sync(0xFFFFFFFFu, eq_c), b_eq_m = __ballot_sync(0xFFFFFFFFu, eq_m);
      sel_c = sel_c || (bk == sc.bucket && kc > sc.prefix) || (eq_c && tie_c + __popc(b_eq_c & below) < sc.take);
      sel_m = sel_m || (bk == sm.bucket && km > sm.prefix) || (eq_m && tie_m + __popc(b_eq_m & below) < sm.take);
      tie_c += __popc(b_eq_c);
      tie_m += __popc(b_eq_m);
    }
    const int c = !in ? -1 : (sel_c ? 2 : (sel_m ? 1 : 0));
    if (in) out_cls[j] = static_cast<signed char>(c);
    const unsigned m_crit = __ballot_sync(0xFFFFFFFFu, c == 2);
    const unsigned m_marg = __ballot_sync(0xFFFFFFFFu, c == 1);
    if (c == 2) crit_row[__popc(m_crit & below)] = j;
    crit_row += __popc(m_crit);
    if (marg_row != nullptr) {
      if (c == 1) marg_row[__popc(m_marg & below)] = j;
      marg_row += __popc(m_marg);
    }
  }
  if (late_wait) sm100::wait_for_prior_grid();
}

// Two neighbouring column sums times 2^-10 as fp16 pairs hi + lo (22 bits between them).
__device__ __forceinline__ void split_pair(int v0, int v1, uint32_t& hi, uint32_t& lo) {
  const float f0 = __int2float_rn(v0) * 0x1p-10f, f1 = __int2float_rn(v1) * 0x1p-10f;
  const __half2 h = __floats2half2_rn(f0, f1);
  const float2 back = __half22float2(h);
  const __half2 l = __floats2half2_rn(f0 - back.x, f1 - back.y);
  hi = *reinterpret_cast<const uint32_t*>(&h);
  lo = *reinterpret_cast<const uint32_t*>(&l);
}
__device__ __forceinline__ __half2 as_half2(uint32_t v) { return *reinterpret_cast<const __half2*>(&v); }
__device__ __forceinline__ uint32_t as_word(__half2 v) { return *reinterpret_cast<const uint32_t*>(&v); }
// Two neighbouring column sums times `mult` (together below 449 * 2^16) as fp16 pairs hi + mid in units of 2^16: hi the
// nearest integer, mid the next eight bits, what is left out at most 2^-9.  Integer bits are put under the exponent of a
// power of two (1024 + n is exact in fp16 for n < 1024) and the offset is taken off again: no conversion instruction.
__device__ __forceinline__ void digits_pair(int v0, int v1, int mult, uint32_t& hi, uint32_t& mid) {
  constexpr uint32_t kBias = (0x6600u << 16) + 0x8080u;  // 1536.0 over the upper half; 128.5 steps of mid
  const uint32_t w0 = static_cast<uint32_t>(v0 * mult) + kBias, w1 = static_cast<uint32_t>(v1 * mult) + kBias;
  const uint32_t m = (__byte_perm(w0, w1, 0x5511) & 0x00FF00FFu) | 0x64006400u;  // 1024 + (0..255)
  hi = as_word(__hadd2(as_half2(__byte_perm(w0, w1, 0x7632)), as_half2(0xE600E600u)));          // - 1536
  mid = as_word(__hfma2(as_half2(m), as_half2(0x1C001C00u), as_half2(0xC480C480u)));            // / 256 - 4.5
}
__device__ __forceinline__ void mma_m16n8k16(float (&c)[4], const uint4& a, uint32_t b0, uint32_t b1) {
  asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};"
               : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
               : "r"(a.x), "r"(a.y), "r"(a.z), "r"(a.w), "r"(b0), "r"(b1));
}

// Places: what a score becomes in shared memory, two bytes instead of an eight-byte key.  The row's scores lie within
// +-448 S max_j scale^K_j with S = sum_d |colsum^Q_d| 2^-10; this interval is mapped linearly to the integers
// kPlaceLow .. kPlaceHigh.  Where up to kLarge key blocks have more than twice the scale that is usual in the row, the
// interval is that of the others; their own places, the interval's ends where they lie outside it, come from exact scores, as
// approximate ones are as much less exact as their scales are larger.  All of them are bit patterns of normal, finite fp16 numbers, which are ordered like the
// integers, so one instruction compares two of them; an entry past the row's end holds a NaN, which fails every comparison.
constexpr int kPlaceMid = 16024, kPlaceSpan = 14990, kPlaceLow = 1024, kPlaceHigh = 31030;
constexpr int kNever = 0x7C00, kTopPlace = 0x7BFF;  // above every place; place of an entry found to be critical
constexpr int kListed = 32;                         // entries of a threshold range that are decided from a list (64: up to 60 against 35 us, figures as below)
constexpr int kLarge = 32;                          // key blocks of large scale (one per lane)
constexpr int kPicked = 256;                        // indices of undecided entries at a time (eight per lane)
constexpr int kFewListed = 14;                      // with more than this in its bucket the range is narrowed first
constexpr int kFinest = 0x7F7F;                     // finer places: their top 128 stay free, as 0xFFFF is what lies past a row's end

__device__ __forceinline__ long long dot4(const int4& a, const int4& b) {
  return static_cast<long long>(a.x) * b.x + static_cast<long long>(a.y) * b.y + static_cast<long long>(a.z) * b.z +
         static_cast<long long>(a.w) * b.w;
}

// Place of a key block of large scale from its exact score.
__device__ __forceinline__ int place_of(const int4* q4, const int* k_colsum, const float* k_scale, int valid, float unit) {
  long long dot = 0;
#pragma unroll 4
  for (int d = 0; d < kHeadDim / 4; ++d) dot += dot4(q4[d], __ldg(reinterpret_cast<const int4*>(k_colsum) + d));
  const double score = static_cast<double>(dot) * static_cast<double>(__ldg(k_scale)) / static_cast<double>(valid);
  return min(max(__double2int_rn(fma(score, static_cast<double>(unit) * 0x1p-19, static_cast<double>(kPlaceMid))), kPlaceLow), kPlaceHigh);
}

// Pitch of a row of places: 16-byte aligned, and eight rows on different banks for 4-byte accesses (an odd multiple of 16
// bytes).
__host__ __device__ constexpr int place_pitch(int nb) { return (((nb + 7) >> 3) | 1) << 3; }

// Bits 0..7: which of the eight halves of four mask words (0xFFFF or 0 each) are set.
__device__ __forceinline__ uint32_t mask_bits(uint32_t m0, uint32_t m1, uint32_t m2, uint32_t m3) {
  const uint32_t x = (m0 & 0x00020001u) | (m1 & 0x00080004u) | (m2 & 0x00200010u) | (m3 & 0x00800040u);
  return (x | (x >> 16)) & 0xFFu;
}

// Without a branch: counts one in shared memory where flag holds; *dst++ = v where flag != 0.
__device__ __forceinline__ void count_if(uint32_t counter, bool flag) {
  asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.u32 p, %1, 0;\n\t@p red.shared.add.u32 [%0], 1;\n\t}" ::"r"(counter), "r"(flag ? 1u : 0u) : "memory");
}
__device__ __forceinline__ void append_if(int*& dst, int v, uint32_t flag) {
  asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.u32 p, %2, 0;\n\t@p st.global.u32 [%0], %1;\n\t@p add.s64 %0, %0, 4;\n\t}"
               : "+l"(dst) : "r"(v), "r"(flag) : "memory");
}

// The same plan for rows of more than kRankMax blocks: approximate scores as 16-bit places in shared memory, exact keys
// only for the few entries that the approximation leaves undecided at a selection threshold.
//   Phase A (whole CTA, R = 16 or 8 rows): fp16 tensor products (m16n8k16) of the query sums split in two (hi + lo, 22 bits)
//     and the key sums' upper 18 bits as two digits (hi + mid): hi hi + hi mid + lo hi.  A key block of `valid` tokens
//     has |colsum| <= 448 512 valid, so colsum * mult with mult = floor(128 / valid) fills the digits' range in short
//     last blocks too.  What is left out, per unit of S (khat up to 448): the key digits' rest 2^-9, lo mid 2^-12,
//     the query's rest 448 2^-22, twelve fp32 accumulations 12 * 448 * 2^-22, the scalings 448 3 2^-24: together below
//     0.004, and at most twice that in a last block whose sums reach only half the range.  In places: 0.004 *
//     14990 / 448 = 0.14 (0.27), plus 0.5 for the rounding to an integer.  Places of two entries that differ by two or
//     more are therefore in the order of the exact scores, and the k-th largest place is within 0.77 of that of the
//     k-th largest score: an entry two places above the k-th largest place is selected, one two below is not, and only
//     those within one place (`margin`) need their exact 64-bit keys, recomputed from the integer column sums (an
//     int64 dot product, equal to the fp64 tensor-core value as long as that is exact, i.e. below 2^53).
//     Rows without such an interval (all sums zero, a scale that is not finite) leave everything undecided.
//   Phase B (one warp per row): the bucket of a 256-bucket histogram between the row's extremes that holds the k-th
//     largest place; when it is too full, a second histogram inside that bucket, one counter per place; then the entries of
//     the bucket and a margin on both sides as a list (up to kListed, in any order), ranked by comparing all pairs, first
//     by place, then, inside the margin, by exact key and index.  Longer lists get finer places from exact scores, and what
//     is equal then too (ties, rows without places) goes to the radix select, which recomputes keys pass by pass.  What was
//     decided is written back over the places, so that the class of every entry is a comparison with two thresholds.
//   Phase C (same warp): eight entries per lane and turn: class bytes (stored as aligned 8-byte words, shifted over from the
//     neighbouring lane where the row's address is not a multiple of eight) and the ascending lists, whose positions
//     come from one warp scan of the lanes' counts.
// Bound by instruction issue: 9.0 k instructions per row of 2147 blocks, half of the issue slots or more taken.  Single-precision
// scores read four bytes at a time, with ballots for every 32 entries, took 17 k and, at four bytes an entry, room for one
// CTA per SM instead of two: 16 heads of 2147 blocks 1005 -> 460 us, of 687 blocks (with 64-bit keys before) 108 -> 61 us.
template <int R>
__global__ void __launch_bounds__(R * 32, 32 / R) plan_compact_kernel(const int* __restrict__ q_colsum, const int* __restrict__ k_colsum,
                                                                       const float* __restrict__ k_scales, int tokens, int block,
                                                                       int nb, int k_crit, int k_marg, int k_neg, int late_wait, int mult_last, float factor_last,
                                                                       signed char* __restrict__ cls, int* __restrict__ crit_idx,
                                                                       int* __restrict__ marg_idx) {
  static_assert(R == 8 || R == 16, "rows of one tensor product");
  static_assert(kBuckets * 4 >= 2 * kListed * 8 && kPicked * 2 >= 2 * kListed * 4 && R * kBuckets * 4 >= 4096, "undecided entries and query operands take the histograms' place");
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int pitch = place_pitch(nb);
  unsigned short* s_place = reinterpret_cast<unsigned short*>(smem_raw);                              // [R][pitch]
  unsigned int* s_hist = reinterpret_cast<unsigned int*>(s_place + static_cast<size_t>(R) * pitch);   // [R][kBuckets]
  uint4* s_a = reinterpret_cast<uint4*>(s_hist);  // [2][4][32] query operands (hi, lo) of phase A, ahead of the histograms
  unsigned int* s_list = s_hist + R * kBuckets;                                                          // [R][2][kListed], or [R][kPicked] halves
  int* s_q = reinterpret_cast<int*>(s_list + R * kPicked / 2);                                         // [R][64]
  unsigned int* s_range = reinterpret_cast<unsigned int*>(s_q + R * kHeadDim);                        // [R][R] lowest | highest << 16
  __shared__ float s_sum[R];
  __shared__ unsigned s_kmax[R];
  __shared__ float s_top;
  __shared__ int s_large_count;
  __shared__ unsigned short s_large[kLarge];

  const int row_tiles = (nb + R - 1) / R;
  const int bh = blockIdx.x / row_tiles;
  const int i0 = (blockIdx.x % row_tiles) * R;
  const int warp = __shfl_sync(0xFFFFFFFFu, threadIdx.x >> 5, 0);  // (known to be the same in all lanes)
  const int lane = threadIdx.x & 31;
  const size_t bh_rows = static_cast<size_t>(bh) * nb;
  const int g = lane >> 2, t4 = lane & 3;

  if (!late_wait) sm100::wait_for_prior_grid();
  sm100::launch_dependents();

  // ---- Phase A
  // Lane (g, t) supplies columns 16 t .. 16 t + 15 of its rows (rows g and g + 8 for A, key block g of the warp's eight for
  // B), one and the same assignment of columns to k indices on both sides.  Key sums come straight from global memory
  // (L2) one step ahead; past the end the last block is read instead.
  int4 nxt[4];
  float nxt_ks[2];
  auto load_keys = [&](int j0) {
    const int4* src = reinterpret_cast<const int4*>(k_colsum + (bh_rows + min(j0 + g, nb - 1)) * kHeadDim + 16 * t4);
#pragma unroll
    for (int q = 0; q < 4; ++q) nxt[q] = __ldg(src + q);
#pragma unroll
    for (int x = 0; x < 2; ++x) nxt_ks[x] = __ldg(k_scales + bh_rows + min(j0 + 2 * t4 + x, nb - 1));
  };
  load_keys(warp * 8);
  {
    const int2 qv = __ldg(reinterpret_cast<const int2*>(q_colsum + (bh_rows + min(i0 + warp, nb - 1)) * kHeadDim) + lane);
    *reinterpret_cast<int2*>(s_q + warp * kHeadDim + 2 * lane) = qv;
    const unsigned sum_q = __reduce_add_sync(0xFFFFFFFFu, static_cast<unsigned>(abs(qv.x)) + static_cast<unsigned>(abs(qv.y)));
    // bits of the largest scale and sum of the upper bits: scales are not negative, and what is not a number counts as the largest
    unsigned kmax = 0u, ksum = 0u;
    for (int j = warp * 32; j < nb; j += R * 32) {
      const unsigned bits = j + lane < nb ? __float_as_uint(__ldg(k_scales + bh_rows + j + lane)) : 0u;
      kmax = max(kmax, bits);
      ksum += bits >> 14;
    }
    kmax = __reduce_max_sync(0xFFFFFFFFu, kmax);
    ksum = __reduce_add_sync(0xFFFFFFFFu, ksum);
    if (lane == 0) {
      s_sum[warp] = static_cast<float>(sum_q) * 0x1p-10f;
      s_kmax[warp] = kmax;
      s_list[warp] = ksum;
    }
    if (threadIdx.x == 0) s_large_count = 0;
    if (warp < 4) {  // operands of k-step `warp`
      uint4 hi = make_uint4(0u, 0u, 0u, 0u), lo = hi;
      auto load_row = [&](int r) {
        return __ldg(reinterpret_cast<const int4*>(q_colsum + (bh_rows + min(i0 + r, nb - 1)) * kHeadDim + 16 * t4) + warp);
      };
      const int4 v = load_row(g);
      split_pair(v.x, v.y, hi.x, lo.x);
      split_pair(v.z, v.w, hi.z, lo.z);
      if constexpr (R == 16) {
        const int4 v8 = load_row(g + 8);
        split_pair(v8.x, v8.y, hi.y, lo.y);
        split_pair(v8.z, v8.w, hi.w, lo.w);
      }
      s_a[warp * 32 + lane] = hi;
      s_a[(4 + warp) * 32 + lane] = lo;
    }
  }
  __syncthreads();
  float k_top = __uint_as_float(__reduce_max_sync(0xFFFFFFFFu, lane < R ? s_kmax[lane] : 0u));
  {
    // Twice the value whose bits are the mean of the scales' bits, about twice their geometric mean, tells large ones.  Costs 0.3 us at
    // 16 heads of 172 blocks, 0.8 at 687; with one token of Gaussian keys 30 times larger 35 -> 18.5 and 180 -> 102 us.
    const unsigned ksum = __reduce_add_sync(0xFFFFFFFFu, lane < R ? s_list[lane] : 0u);
    const float most = __uint_as_float(static_cast<unsigned>(static_cast<float>(ksum) * __fdividef(16384.f, static_cast<float>(nb))) + 0x00800000u);
    if (k_top > most && k_top < INFINITY) {  // (the same for the whole CTA; next to an infinite scale the row has no places)
      for (int j = threadIdx.x; j < nb; j += R * 32) {
        if (__ldg(k_scales + bh_rows + j) > most) {
          const int at = atomicAdd(&s_large_count, 1);
          if (at < kLarge) s_large[at] = static_cast<unsigned short>(j);
        }
      }
      __syncthreads();
      if (s_large_count <= kLarge) k_top = most;
    }
  }
  // places per unit of a row's score; 0: the row has no places
  auto places_per_unit = [&](int r, float top) {
    const float reach = 448.f * s_sum[r] * top;
    return reach > 0.f && reach < 0x1p126f ? __fdividef(static_cast<float>(kPlaceSpan), reach) : 0.f;
  };
  {
    constexpr int kHalves = R / 8;
    float unit[kHalves];
    uint32_t lo2[kHalves], hi2[kHalves];
#pragma unroll
    for (int r = 0; r < kHalves; ++r) {
      unit[r] = places_per_unit(8 * r + g, k_top);
      lo2[r] = 0x7BFF7BFFu;
      hi2[r] = 0u;
    }
    const int mult_full = 128 / block;
    // one step of eight key blocks; `edge`: the last block or what lies behind it is among them
    auto step = [&](int j0, auto edge) {
      constexpr bool kEdge = decltype(edge)::value;
      const int mult = kEdge && j0 + g >= nb - 1 ? mult_last : mult_full;
      uint32_t b_hi[8], b_mid[8];
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        digits_pair(nxt[q].x, nxt[q].y, mult, b_hi[2 * q], b_mid[2 * q]);
        digits_pair(nxt[q].z, nxt[q].w, mult, b_hi[2 * q + 1], b_mid[2 * q + 1]);
      }
      const int j = j0 + 2 * t4;
      float factor[2] = {nxt_ks[0], nxt_ks[1]};
      if constexpr (kEdge) {
        if (j >= nb - 1) factor[0] *= factor_last;
        if (j + 1 >= nb - 1) factor[1] *= factor_last;
      } else {
        if (j0 + 8 * R < nb) load_keys(j0 + 8 * R);
      }
      float c[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
      for (int st = 0; st < 4; ++st) {
        const uint4 a_hi = s_a[st * 32 + lane], a_lo = s_a[(4 + st) * 32 + lane];
        mma_m16n8k16(c, a_hi, b_hi[2 * st], b_hi[2 * st + 1]);
        mma_m16n8k16(c, a_hi, b_mid[2 * st], b_mid[2 * st + 1]);
        mma_m16n8k16(c, a_lo, b_hi[2 * st], b_hi[2 * st + 1]);
      }
#pragma unroll
      for (int r = 0; r < kHalves; ++r) {
        // 1.5 * 2^23 leaves the rounded place in the low mantissa bits
        const float at0 = fmaf(c[2 * r], factor[0] * unit[r], 12582912.f + kPlaceMid);
        const float at1 = fmaf(c[2 * r + 1], factor[1] * unit[r], 12582912.f + kPlaceMid);
        uint32_t both = __byte_perm(__float_as_uint(at0), __float_as_uint(at1), 0x5410);
        // (sums that no quantiser has written could lead anywhere: every place has to be one)
        both = as_word(__hmin2(__hmax2(as_half2(both), as_half2(kPlaceLow * 0x10001u)), as_half2(kPlaceHigh * 0x10001u)));
        if constexpr (kEdge) {
          if (j + 1 >= nb) both |= j >= nb ? 0xFFFFFFFFu : 0xFFFF0000u;
        }
        *reinterpret_cast<uint32_t*>(s_place + static_cast<size_t>(8 * r + g) * pitch + j) = both;
        lo2[r] = as_word(__hmin2(as_half2(lo2[r]), as_half2(both)));
        hi2[r] = as_word(__hmax2(as_half2(hi2[r]), as_half2(both)));
      }
    };
    int j0 = warp * 8;
    for (; j0 + 8 < nb; j0 += 8 * R) step(j0, std::false_type{});
    if (j0 < nb) step(j0, std::true_type{});
#pragma unroll
    for (int r = 0; r < kHalves; ++r) {
#pragma unroll
      for (int o = 1; o <= 2; o <<= 1) {
        lo2[r] = as_word(__hmin2(as_half2(lo2[r]), as_half2(__shfl_xor_sync(0xFFFFFFFFu, lo2[r], o))));
        hi2[r] = as_word(__hmax2(as_half2(hi2[r]), as_half2(__shfl_xor_sync(0xFFFFFFFFu, hi2[r], o))));
      }
      if (t4 == 0) s_range[warp * R + 8 * r + g] = min(lo2[r] & 0xFFFFu, lo2[r] >> 16) | (max(hi2[r] & 0xFFFFu, hi2[r] >> 16) << 16);
    }
  }
  const bool no_places = places_per_unit(warp, k_top) == 0.f;
  const int large = s_large_count;
  if (threadIdx.x == 0) s_top = k_top;
  __syncthreads();
  const int i = i0 + warp;
  if (i >= nb) return;

  // ---- Phase B
  unsigned short* const row = s_place + static_cast<size_t>(warp) * pitch;
  const uint4* const row8 = reinterpret_cast<const uint4*>(row);  // eight places
  const int chunks = (nb + 7) >> 3;
  unsigned int* const hist = s_hist + warp * kBuckets;
  unsigned int* const list_c = s_list + warp * kPicked / 2;  // index | place << 16 | selected << 31
  unsigned int* const list_m = list_c + kListed;
  const int4* const q4 = reinterpret_cast<const int4*>(s_q + warp * kHeadDim);
  const int margin = no_places ? 0x7FFF : 1;
  const double inv_block = 1.0 / static_cast<double>(block);
  const unsigned below = (1u << lane) - 1u;
  const unsigned range = lane < R ? s_range[lane * R + warp] : 0x0000FFFFu;
  int low = static_cast<int>(__reduce_min_sync(0xFFFFFFFFu, range & 0xFFFFu)), high = static_cast<int>(__reduce_max_sync(0xFFFFFFFFu, range >> 16));

  // the ranking score from an exact dot product (same expression as in plan_kernel)
  auto exact_score = [&](long long dot, int j) -> double {
    const int valid = min(block, tokens - j * block);
    const double num = static_cast<double>(dot) * static_cast<double>(__ldg(k_scales + bh_rows + j));
    return (valid == block ? num * inv_block : num / static_cast<double>(valid)) + 0.0;  // block is a power of two
  };
  auto exact_order_key = [&](long long dot, int j) -> unsigned long long { return order_key(exact_score(dot, j)); };
  auto exact_key = [&](int j) -> unsigned long long {  // of entry j, by one lane
    const int4* const k4 = reinterpret_cast<const int4*>(k_colsum + (bh_rows + j) * kHeadDim);
    long long dot = 0;
#pragma unroll 4
    for (int d = 0; d < kHeadDim / 4; ++d) dot += dot4(q4[d], __ldg(k4 + d));
    return exact_order_key(dot, j);
  };
  if (large > 0 && large <= kLarge) {  // places of the key blocks of large scale, from their exact scores
    const int j = s_large[min(lane, large - 1)];
    const int place = place_of(q4, k_colsum + (bh_rows + j) * kHeadDim, k_scales + bh_rows + j, min(block, tokens - j * block), places_per_unit(warp, s_top));
    row[j] = static_cast<unsigned short>(place);
    low = min(low, __reduce_min_sync(0xFFFFFFFFu, place));
    high = max(high, __reduce_max_sync(0xFFFFFFFFu, place));
    __syncwarp();
  }

  auto half_of = [](const uint4& v, int x) -> int {
    const uint32_t w = x < 2 ? v.x : (x < 4 ? v.y : (x < 6 ? v.z : v.w));
    return static_cast<int>((x & 1) ? w >> 16 : w & 0xFFFFu);
  };
  // The passes over a row are loops of the whole warp (a lane past the end has eight entries that fail every comparison):
  // lanes that leave a loop early, or take a branch of their own, would run what follows separately.
  auto chunk = [&](int c) -> uint4 { return c < chunks ? row8[c] : make_uint4(~0u, ~0u, ~0u, ~0u); };
  auto clear_hist = [&]() {
    __syncwarp();
#pragma unroll
    for (int x = 0; x < 2; ++x) reinterpret_cast<uint4*>(hist)[lane + 32 * x] = make_uint4(0u, 0u, 0u, 0u);
    __syncwarp();
  };
  // The eight neighbouring counters of a lane and how many entries the lanes before it have (in its group of `width` lanes).
  auto levels_of = [&](int width, int (&count)[8], int& before, int& after) {
    const uint4 a = reinterpret_cast<const uint4*>(hist)[2 * lane], b = reinterpret_cast<const uint4*>(hist)[2 * lane + 1];
    count[0] = a.x, count[1] = a.y, count[2] = a.z, count[3] = a.w;
    count[4] = b.x, count[5] = b.y, count[6] = b.z, count[7] = b.w;
    int total = 0;
#pragma unroll
    for (int x = 0; x < 8; ++x) total += count[x];
    after = total;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int up = __shfl_up_sync(0xFFFFFFFFu, after, o, width);
      if (o < width && (lane & (width - 1)) >= o) after += up;
    }
    before = after - total;
  };
  // If the k-th entry is in one of the lane's counters: entries before that counter, its size and its number among the
  // lane's, packed (rows have fewer than 2^14 entries).
  auto level_at = [](const int (&count)[8], int before, int k) -> unsigned {
    unsigned found = 0u;
#pragma unroll
    for (int x = 0; x < 8; ++x) {
      if (before < k) found = static_cast<unsigned>(before) << 17 | static_cast<unsigned>(count[x]) << 3 | static_cast<unsigned>(x);
      before += count[x];
    }
    return found;
  };
  // first histogram: 256 buckets of 2^shift places, from the highest place down (the places span less than 2^15: shift <= 7)
  const int shift = max(24 - __clz(high - low), 0);
  const uint32_t counters = sm100::smem_u32(hist);
  clear_hist();
  for (int c0 = 0; c0 < chunks; c0 += 32) {
    const uint4 v = chunk(c0 + lane);
    if (8 * c0 + 256 <= nb) {
#pragma unroll
      for (int x = 0; x < 8; ++x) atomicAdd(&hist[(high - half_of(v, x)) >> shift], 1u);
    } else {  // (what lies past the end is above the highest place)
#pragma unroll
      for (int x = 0; x < 8; ++x)
        count_if(counters + (((high - half_of(v, x)) >> shift) << 2), half_of(v, x) <= high);
    }
  }
  __syncwarp();

  // A selection: entries whose place is above t_hi are selected, those in [t_lo, t_hi] are decided one by one (from a list
  // or, `recompute`, by their finer places), the rest are not.
  struct Chosen {
    int k, t_lo, t_hi;
    int above, bucket_hi;  // entries with a place above bucket_hi
    bool open, recompute;  // something is to be decided; too many entries for a list
  };
  auto begin = [&](int k) -> Chosen {
    Chosen r;
    r.k = k;
    r.open = k > 0 && k < nb;
    r.recompute = false;
    r.above = r.bucket_hi = 0;
    r.t_lo = k <= 0 ? kNever : 0;  // an empty interval above or below all places
    r.t_hi = r.t_lo - 1;
    return r;
  };
  Chosen cc = begin(k_crit), cm = begin(nb - k_neg);
  {
    int count[8], before, after, size_c = 0, size_m = 0;
    levels_of(32, count, before, after);
    auto find = [&](Chosen& r) -> int {
      const int src = __ffs(static_cast<int>(__ballot_sync(0xFFFFFFFFu, before < r.k && r.k <= after))) - 1;
      const unsigned found = __shfl_sync(0xFFFFFFFFu, level_at(count, before, r.k), src);
      r.t_hi = high - ((8 * src + static_cast<int>(found & 7u)) << shift);
      r.t_lo = r.t_hi - (1 << shift) + 1;
      r.above = static_cast<int>(found >> 17);
      return static_cast<int>((found >> 3) & 0x3FFFu);
    };
    if (cc.open) size_c = find(cc);
    if (cm.open) size_m = find(cm);
    // Too many entries: a second histogram inside the two buckets, a counter for each of their (at most 128) places.
    if (shift > 0 && max(size_c, size_m) > kFewListed) {
      const int width = 1 << shift;
      const int top_c = cc.open ? cc.t_hi : -1, top_m = cm.open ? cm.t_hi : -1;  // (no place is within `width` below -1)
      clear_hist();
      for (int c0 = 0; c0 < chunks; c0 += 32) {
        const uint4 v = chunk(c0 + lane);
#pragma unroll
        for (int x = 0; x < 8; ++x) {
          const int p = half_of(v, x);
          const unsigned at_c = static_cast<unsigned>(top_c - p), at_m = static_cast<unsigned>(top_m - p);
          count_if(counters + (at_c << 2), at_c < static_cast<unsigned>(width));
          count_if(counters + 512 + (at_m << 2), at_m < static_cast<unsigned>(width));
        }
      }
      __syncwarp();
      int count2[8], before2, after2;
      levels_of(16, count2, before2, after2);  // lanes 0-15: the first selection's counters, 16-31 the second's
      const int k = lane < 16 ? cc.k - cc.above : cm.k - cm.above;
      const unsigned found = level_at(count2, before2, k);
      const unsigned where = __ballot_sync(0xFFFFFFFFu, before2 < k && k <= after2);
      auto enter = [&](Chosen& r, int base) {
        if (!r.open) return;
        const int src = __ffs(static_cast<int>((where >> base) & 0xFFFFu)) - 1;
        const unsigned f = __shfl_sync(0xFFFFFFFFu, found, base + src);
        r.t_hi -= 8 * src + static_cast<int>(f & 7u);
        r.t_lo = r.t_hi;
        r.above += static_cast<int>(f >> 17);
      };
      enter(cc, 0);
      enter(cm, 16);
    }
  }
  __syncwarp();
  for (Chosen* r : {&cc, &cm}) {
    if (!r->open) continue;
    r->bucket_hi = r->t_hi;
    r->t_lo = max(r->t_lo - margin, 1);
    r->t_hi = min(r->t_hi + margin, kTopPlace - 1);
    if (no_places) {
      r->above = 0;
      r->bucket_hi = r->t_hi;
    }
  }

  if (cc.open || cm.open) {  // the entries of the two ranges, in any order
    if (lane < 2) hist[lane] = 0u;
    __syncwarp();
    auto twice = [](int place) { return as_half2(static_cast<uint32_t>(place) * 0x10001u); };
    const __half2 lo_c = twice(cc.t_lo), end_c = twice(cc.t_hi + 1), lo_m = twice(cm.t_lo), end_m = twice(cm.t_hi + 1);
    for (int c0 = 0; c0 < chunks; c0 += 32) {
      const uint4 v = chunk(c0 + lane);
      const uint32_t words[4] = {v.x, v.y, v.z, v.w};
      uint32_t in_c[4], in_m[4];
#pragma unroll
      for (int w = 0; w < 4; ++w) {
        in_c[w] = __hge2_mask(as_half2(words[w]), lo_c) & ~__hge2_mask(as_half2(words[w]), end_c);
        in_m[w] = __hge2_mask(as_half2(words[w]), lo_m) & ~__hge2_mask(as_half2(words[w]), end_m);
      }
      uint32_t bits = mask_bits(in_c[0], in_c[1], in_c[2], in_c[3]) | mask_bits(in_m[0], in_m[1], in_m[2], in_m[3]) << 8;
      while (__any_sync(0xFFFFFFFFu, bits != 0u)) {
        if (bits != 0u) {
          const int b = __ffs(static_cast<int>(bits)) - 1, j = 8 * (c0 + lane) + (b & 7), which = b >> 3;
          bits &= bits - 1u;
          const unsigned at = atomicAdd(hist + which, 1u);
          if (at < static_cast<unsigned>(kListed)) list_c[which * kListed + at] = (static_cast<unsigned>(row[j]) << 16) | static_cast<unsigned>(j);
        }
        __syncwarp();
      }
    }
    __syncwarp();
  }
  const int n_c = cc.open ? static_cast<int>(hist[0]) : 0, n_m = cm.open ? static_cast<int>(hist[1]) : 0;
  __syncwarp();
  cc.recompute = n_c > kListed;
  cm.recompute = n_m > kListed;

  // Decides the listed entries of both selections side by side, kPer entries per lane: first those of the critical list,
  // then those of the other.  The selected ones are marked (bit 31).
  unsigned long long* const u_key = reinterpret_cast<unsigned long long*>(hist);        // [2 kListed], over the histogram
  const int m_c = cc.recompute || cm.recompute ? 0 : n_c, m_m = cc.recompute || cm.recompute ? 0 : n_m;
  auto decide = [&](auto per) {
    constexpr int kPer = decltype(per)::value;
    // the lists are read four entries at a time, the shorter one as far as the longer one goes
    const int end = (max(m_c, m_m) + 3) & ~3;
    for (int o = 0; o < end; o += 32) {
      const int at = o + lane;
      if (at >= m_c && at < end) list_c[at] = 0u;
      if (at >= m_m && at < end) list_m[at] = 0u;
    }
    __syncwarp();
    unsigned e[kPer];
    int place[kPer], rank[kPer];
    bool in[kPer], of_m[kPer];
    const unsigned int* own[kPer];
    struct Two {
      int c, m;
    };
    auto tally = [&](const bool (&flag)[kPer]) {  // how many entries of either list have the flag
      Two n = {0, 0};
#pragma unroll
      for (int x = 0; x < kPer; ++x) {
        n.c += __popc(__ballot_sync(0xFFFFFFFFu, flag[x] && !of_m[x]));
        n.m += __popc(__ballot_sync(0xFFFFFFFFu, flag[x] && of_m[x]));
      }
      return n;
    };
    bool flag[kPer];
#pragma unroll
    for (int x = 0; x < kPer; ++x) {
      const int at = lane + 32 * x;
      of_m[x] = at >= m_c;
      in[x] = at < m_c + m_m;
      own[x] = of_m[x] ? list_m : list_c;
      e[x] = in[x] ? own[x][of_m[x] ? at - m_c : at] : 0u;
      place[x] = static_cast<int>(e[x] >> 16);
      rank[x] = 0;
      flag[x] = in[x] && place[x] > (of_m[x] ? cm.bucket_hi : cc.bucket_hi);
    }
    // how many of the listed are selected: the margin took in some that are counted as above the bucket
    Two need = tally(flag);
    need.c += cc.k - cc.above;
    need.m += cm.k - cm.above;
    for (int o = 0; o < end; o += 4) {
#pragma unroll
      for (int x = 0; x < kPer; ++x) {
        const uint4 v = *reinterpret_cast<const uint4*>(own[x] + o);
        rank[x] += (v.x > e[x] ? 1 : 0) + (v.y > e[x] ? 1 : 0) + (v.z > e[x] ? 1 : 0) + (v.w > e[x] ? 1 : 0);
      }
    }
    Two kth = {0, 0};
#pragma unroll
    for (int x = 0; x < kPer; ++x) {
      const int hit = in[x] && rank[x] == (of_m[x] ? need.m : need.c) - 1 ? place[x] : 0;
      kth.c = max(kth.c, of_m[x] ? 0 : hit);
      kth.m = max(kth.m, of_m[x] ? hit : 0);
    }
    kth.c = __reduce_max_sync(0xFFFFFFFFu, kth.c);
    kth.m = __reduce_max_sync(0xFFFFFFFFu, kth.m);
    bool sel[kPer], und[kPer];
#pragma unroll
    for (int x = 0; x < kPer; ++x) {
      const int d = place[x] - (of_m[x] ? kth.m : kth.c);
      sel[x] = in[x] && d > margin;
      und[x] = in[x] && d >= -margin && !sel[x];
    }
    const Two sure = tally(sel), open = tally(und);
    need.c -= sure.c;
    need.m -= sure.m;
    const bool exact_c = need.c != open.c, exact_m = need.m != open.m;  // else all that are open are selected
    if (exact_c || exact_m) {
      // exact keys of the open entries, eight lanes to an entry (its 256 bytes of column sums read whole)
      const int l8 = lane & 7;
#pragma unroll
      for (int x = 0; x < kPer; ++x) {
        unsigned todo = __ballot_sync(0xFFFFFFFFu, und[x] && (of_m[x] ? exact_m : exact_c));
        while (todo != 0u) {
          // the first four of those left, one for each group of eight lanes
          const unsigned t1 = todo & (todo - 1u), t2 = t1 & (t1 - 1u), t3 = t2 & (t2 - 1u);
          const unsigned mine = lane < 8 ? todo : (lane < 16 ? t1 : (lane < 24 ? t2 : t3));
          const int src = __ffs(static_cast<int>(mine != 0u ? mine : todo)) - 1;
          const int j = static_cast<int>(__shfl_sync(0xFFFFFFFFu, e[x], src) & 0xFFFFu);
          const int4* const k4 = reinterpret_cast<const int4*>(k_colsum + (bh_rows + j) * kHeadDim);
          long long dot = dot4(q4[l8], __ldg(k4 + l8)) + dot4(q4[l8 + 8], __ldg(k4 + l8 + 8));
#pragma unroll
          for (int o = 1; o < 8; o <<= 1) dot += __shfl_xor_sync(0xFFFFFFFFu, dot, o);
          if (l8 == 0) u_key[32 * x + src] = exact_order_key(dot, j);
          todo = t3 & (t3 - 1u);
        }
      }
      __syncwarp();
#pragma unroll
      for (int x = 0; x < kPer; ++x) {
        const bool exact = und[x] && (of_m[x] ? exact_m : exact_c);
        const unsigned long long key = exact ? u_key[32 * x + lane] : 0ull;
        int better = 0;
#pragma unroll
        for (int y = 0; y < kPer; ++y) {
          unsigned others = __ballot_sync(0xFFFFFFFFu, und[y] && (of_m[y] ? exact_m : exact_c));
          const unsigned theirs = __ballot_sync(0xFFFFFFFFu, of_m[y]);
          for (; others != 0u; others &= others - 1u) {
            const int src = __ffs(static_cast<int>(others)) - 1;
            const unsigned j = __shfl_sync(0xFFFFFFFFu, e[y], src) & 0xFFFFu;
            const unsigned long long other = u_key[32 * y + src];
            if (((theirs >> src) & 1u) == (of_m[x] ? 1u : 0u) && (other > key || (other == key && j < (e[x] & 0xFFFFu)))) ++better;
          }
        }
        if (und[x]) sel[x] = !exact || better < (of_m[x] ? need.m : need.c);
      }
    } else {
#pragma unroll
      for (int x = 0; x < kPer; ++x) sel[x] = sel[x] || und[x];
    }
#pragma unroll
    for (int x = 0; x < kPer; ++x) {
      const int at = of_m[x] ? kListed + lane + 32 * x - m_c : lane + 32 * x;
      if (sel[x]) list_c[at] = e[x] | 0x80000000u;
    }
    __syncwarp();
  };
  __syncwarp();
  if (m_c + m_m > 32)
    decide(std::integral_constant<int, 2>{});
  else if (m_c + m_m > 0)
    decide(std::integral_constant<int, 1>{});

  // Thresholds of the class pass: place >= thr_c is critical, else place >= thr_m marginal.  What was decided is written
  // over the places: kTopPlace for critical, `mark` = thr_c - 1 for marginal, 0 for negligible.  No other entry holds
  // `mark`: as the upper end of the critical range its entries have all been decided.
  const int thr_c = cc.t_hi + 1, mark = max(thr_c - 1, 0), thr_m = min(cm.t_hi + 1, mark);
  if (cc.recompute || cm.recompute) {
    // Ranges too full for a list (one key block of a much larger scale than the others, scores that differ by little): every
    // entry of a range gets its exact score once, eight lanes to an entry, and with it a finer place inside the range, 0 ..
    // kFinest, kept in place of the coarse one under bit 15.  The rounding is the same function of every exact score, so only
    // equal finer places are undecided; two histograms find the one at the threshold, and where it is not selected or left
    // as a whole, the radix select its share.  Ranges that overlap are treated as one.  With lists of 64 and longer ones left to
    // the radix select, which recomputed the keys in each of its passes, one lane to a key: 16 heads of 687 blocks of Gaussian
    // keys with one token 30 times larger 1095 -> 179 us, of 172 blocks 83 -> 35, 10 times larger (clustered keys) 312 -> 112 and 28 -> 27,
    // keys and queries within 2 % of one value 248 -> 130 and 25 -> 25; of 2147 blocks clustered keys as they are 1063 -> 770
    // (one large key in a row no longer leads here).
    const int l8 = lane & 7, group = lane >> 3;
    const bool apart = cc.open && cm.open && cm.t_hi < cc.t_lo;
    unsigned short* const picked = reinterpret_cast<unsigned short*>(list_c);  // [kPicked], over both lists
    for (int turn = 0; turn < 2; ++turn) {
      const bool has_c = turn == 0 && cc.open, has_m = cm.open && apart == (turn == 1);
      if (!has_c && !has_m) continue;
      const int lo = has_m ? cm.t_lo : cc.t_lo, hi = has_c ? cc.t_hi : cm.t_hi;
      const double per_place = static_cast<double>(kFinest) / static_cast<double>(hi - lo + 2);
      const double slope = static_cast<double>(places_per_unit(warp, s_top)) * 0x1p-19 * per_place;  // (a place is score * unit * 2^-19)
      const double offset = static_cast<double>(kPlaceMid - lo + 1) * per_place;
      const __half2 from = as_half2(static_cast<uint32_t>(lo) * 0x10001u), end = as_half2(static_cast<uint32_t>(hi + 1) * 0x10001u);
      clear_hist();
      int above = 0;
      for (int c0 = 0; c0 < chunks; c0 += 32) {
        const uint4 v = chunk(c0 + lane);
        const uint32_t words[4] = {v.x, v.y, v.z, v.w};
        uint32_t ge[4], gt[4];
#pragma unroll
        for (int w = 0; w < 4; ++w) {
          gt[w] = __hge2_mask(as_half2(words[w]), end);
          ge[w] = __hge2_mask(as_half2(words[w]), from) & ~gt[w];
        }
        above += __popc(mask_bits(gt[0], gt[1], gt[2], gt[3]));
        uint32_t bits = mask_bits(ge[0], ge[1], ge[2], ge[3]);
        int at = __popc(bits);
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
          const int up = __shfl_up_sync(0xFFFFFFFFu, at, o);
          if (lane >= o) at += up;
        }
        const int total = __shfl_sync(0xFFFFFFFFu, at, 31);
        at -= __popc(bits);
        for (; bits != 0u; bits &= bits - 1u) picked[at++] = static_cast<unsigned short>(8 * (c0 + lane) + __ffs(static_cast<int>(bits)) - 1);
        __syncwarp();
        for (int e0 = 0; e0 < total; e0 += 32) {
          long long dot = 0;  // of entry e0 + 4 l8 + group
#pragma unroll 2
          for (int t = 0; t < 8 && e0 + 4 * t < total; ++t) {
            const int j = picked[min(e0 + 4 * t + group, total - 1)];
            const int4* const k4 = reinterpret_cast<const int4*>(k_colsum + (bh_rows + j) * kHeadDim);
            long long part = dot4(q4[l8], __ldg(k4 + l8)) + dot4(q4[l8 + 8], __ldg(k4 + l8 + 8));
#pragma unroll
            for (int o = 1; o < 8; o <<= 1) part += __shfl_xor_sync(0xFFFFFFFFu, part, o);
            if (l8 == t) dot = part;
          }
          const int own = e0 + 4 * l8 + group;
          if (own < total) {
            const int j = picked[own];
            const int fine = no_places ? 0 : min(max(__double2int_rd(fma(exact_score(dot, j), slope, offset)), 0), kFinest);
            row[j] = static_cast<unsigned short>(0x8000 | fine);
            atomicAdd(&hist[255 - (fine >> 7)], 1u);
          }
          __syncwarp();
        }
      }
      above = __reduce_add_sync(0xFFFFFFFFu, above);
      __syncwarp();
      // finer places above at_c are critical, else above at_m marginal; equal to one that is open: `take` of them are
      int at_c = has_c ? 0 : 0x8000, at_m = has_m ? 0 : -1, take_c = cc.k - above, take_m = cm.k - above;
      {
        int count[8], before, after;
        levels_of(32, count, before, after);
        auto find = [&](int& at, int& take) {  // the highest finer place of the counter
          const int src = __ffs(static_cast<int>(__ballot_sync(0xFFFFFFFFu, before < take && take <= after))) - 1;
          const unsigned found = __shfl_sync(0xFFFFFFFFu, level_at(count, before, take), src);
          at = ((255 - 8 * src - static_cast<int>(found & 7u)) << 7) + 127;
          take -= static_cast<int>(found >> 17);
        };
        if (has_c) find(at_c, take_c);
        if (has_m) find(at_m, take_m);
      }
      clear_hist();
      for (int c0 = 0; c0 < chunks; c0 += 32) {
        const uint4 v = chunk(c0 + lane);
#pragma unroll
        for (int x = 0; x < 8; ++x) {  // (neither a coarse place nor what lies past the end is within 128 below a counter's highest)
          const int fine = half_of(v, x) ^ 0x8000;
          const unsigned d_c = static_cast<unsigned>(at_c - fine), d_m = static_cast<unsigned>(at_m - fine);
          count_if(counters + (d_c << 2), has_c && d_c < 128u);
          count_if(counters + 512 + (d_m << 2), has_m && d_m < 128u);
        }
      }
      __syncwarp();
      bool open_c = false, open_m = false;
      {
        int count[8], before, after;
        levels_of(16, count, before, after);  // lanes 0-15: the first selection's counters, 16-31 the second's
        const int k = lane < 16 ? take_c : take_m;
        const unsigned found = level_at(count, before, k);
        const unsigned where = __ballot_sync(0xFFFFFFFFu, before < k && k <= after);
        auto enter = [&](int& at, int& take, int base) -> bool {
          const int src = __ffs(static_cast<int>((where >> base) & 0xFFFFu)) - 1;
          const unsigned f = __shfl_sync(0xFFFFFFFFu, found, base + src);
          at -= 8 * src + static_cast<int>(f & 7u);
          take -= static_cast<int>(f >> 17);
          if (take < static_cast<int>((f >> 3) & 0x3FFFu)) return true;
          --at;  // all of them
          return false;
        };
        if (has_c) open_c = enter(at_c, take_c, 0);
        if (has_m) open_m = enter(at_m, take_m, 16);
      }
      __syncwarp();
      if (open_c || open_m) {
        Selection sel[2] = {};
        for (int w = 0; w < 2; ++w) {
          if (!(w == 0 ? open_c : open_m)) continue;
          const int code = 0x8000 | (w == 0 ? at_c : at_m);
          radix_select([&](int c, unsigned long long& key) {
            if (row[c] != code) return false;
            key = exact_key(c);
            return true;
          }, nb, w == 0 ? take_c : take_m, hist, lane, sel[w]);
        }
        int tie_c = 0, tie_m = 0;
        for (int j0 = 0; j0 < nb; j0 += 32) {
          const int j = j0 + lane;
          const int fine = j < nb ? row[j] ^ 0x8000 : -1;
          const bool of_c = open_c && fine == at_c, of_m = open_m && fine == at_m;
          if (!__any_sync(0xFFFFFFFFu, of_c || of_m)) continue;
          const unsigned long long key = of_c || of_m ? exact_key(j) : 0ull;
          const unsigned long long kc = key & sel[0].mask, km = key & sel[1].mask;
          const bool eq_c = of_c && kc == sel[0].prefix, eq_m = of_m && km == sel[1].prefix;
          const unsigned b_eq_c = __ballot_sync(0xFFFFFFFFu, eq_c), b_eq_m = __ballot_sync(0xFFFFFFFFu, eq_m);
          const bool sel_c = of_c && (kc > sel[0].prefix || (eq_c && tie_c + __popc(b_eq_c & below) < sel[0].take));
          const bool sel_m = of_m && (km > sel[1].prefix || (eq_m && tie_m + __popc(b_eq_m & below) < sel[1].take));
          tie_c += __popc(b_eq_c);
          tie_m += __popc(b_eq_m);
          if (of_c || of_m) row[j] = static_cast<unsigned short>(sel_c ? kTopPlace : (sel_m || !of_m ? mark : 0));
        }
        __syncwarp();
      }
      for (int c0 = 0; c0 < chunks; c0 += 32) {
        const uint4 v = chunk(c0 + lane);
        uint32_t words[4] = {v.x, v.y, v.z, v.w};
        auto settled = [&](uint32_t p) -> uint32_t {
          const int fine = static_cast<int>(p) - 0x8000;
          return fine < 0 || p == 0xFFFFu ? p : (fine > at_c ? kTopPlace : (fine > at_m ? mark : 0));
        };
#pragma unroll
        for (int w = 0; w < 4; ++w) words[w] = settled(words[w] & 0xFFFFu) | settled(words[w] >> 16) << 16;
        if (c0 + lane < chunks) reinterpret_cast<uint4*>(row)[c0 + lane] = make_uint4(words[0], words[1], words[2], words[3]);
      }
      __syncwarp();
    }
  }
  // the marginal list first: an entry of both lists that is not critical keeps what that one says
  for (int o = 0; o < m_m; o += 32) {
    const unsigned e = o + lane < m_m ? list_m[o + lane] : 0u;
    if (o + lane < m_m && row[e & 0xFFFFu] != kTopPlace) row[e & 0xFFFFu] = static_cast<unsigned short>((e >> 31) != 0u ? mark : 0);
  }
  __syncwarp();
  for (int o = 0; o < m_c; o += 32) {
    const unsigned e = o + lane < m_c ? list_c[o + lane] : 0u;
    const bool top = (e >> 31) != 0u;
    if (top || (o + lane < m_c && static_cast<int>(e >> 16) > cm.t_hi)) row[e & 0xFFFFu] = static_cast<unsigned short>(top ? kTopPlace : mark);
  }
  __syncwarp();

  // ---- Phase C
  const size_t out_row = bh_rows + i;
  signed char* const out_cls = cls + out_row * nb;
  const int ahead = static_cast<int>(reinterpret_cast<uintptr_t>(out_cls) & 7u);  // bytes of the first word that are not ours
  int* crit_row = crit_idx + out_row * k_crit;
  int* marg_row = marg_idx != nullptr ? marg_idx + out_row * k_marg : nullptr;
  const __half2 thr_c2 = as_half2(static_cast<uint32_t>(thr_c) * 0x10001u), thr_m2 = as_half2(static_cast<uint32_t>(thr_m) * 0x10001u);
  const int words = (nb + ahead + 7) >> 3;
  uint2 saved = make_uint2(0u, 0u);
  for (int c0 = 0; c0 < words; c0 += 32) {
    const int c = c0 + lane;
    const uint4 v = chunk(c);
    const uint32_t pairs[4] = {v.x, v.y, v.z, v.w};
    uint32_t top[4], mid[4], two[4];
#pragma unroll
    for (int w = 0; w < 4; ++w) {
      top[w] = __hge2_mask(as_half2(pairs[w]), thr_c2);
      mid[w] = __hge2_mask(as_half2(pairs[w]), thr_m2) & ~top[w];
      two[w] = (top[w] & 0x00020002u) | (mid[w] & 0x00010001u);
    }
    const uint2 own = make_uint2(__byte_perm(two[0], two[1], 0x6420), __byte_perm(two[2], two[3], 0x6420));
    // word c of the row's 8-byte words: the last `ahead` bytes of the entries before, the first of the lane's own
    const uint2 left = make_uint2(__shfl_sync(0xFFFFFFFFu, own.x, lane - 1), __shfl_sync(0xFFFFFFFFu, own.y, lane - 1));
    const uint2 prev = lane == 0 ? saved : left;
    saved = left;
    const int from = 8 - ahead;
    const uint32_t x0 = from >= 8 ? own.x : (from >= 4 ? prev.y : prev.x);
    const uint32_t x1 = from >= 8 ? own.y : (from >= 4 ? own.x : prev.y);
    const uint32_t x2 = from >= 4 ? own.y : own.x;
    const uint2 word = make_uint2(__funnelshift_r(x0, x1, 8 * (from & 3)), __funnelshift_r(x1, x2, 8 * (from & 3)));
    const int j = 8 * c - ahead;  // entry of the word's first byte
    const bool whole = j >= 0 && j + 8 <= nb;
    if (whole) *reinterpret_cast<uint2*>(out_cls + j) = word;
    for (unsigned part = __ballot_sync(0xFFFFFFFFu, !whole && c < words); part != 0u; part &= part - 1u) {  // first and last word of the row
      const int src = __ffs(static_cast<int>(part)) - 1, jb = 8 * (c0 + src) - ahead + lane;
      const uint32_t w0 = __shfl_sync(0xFFFFFFFFu, word.x, src), w1 = __shfl_sync(0xFFFFFFFFu, word.y, src);
      if (lane < 8 && jb >= 0 && jb < nb) out_cls[jb] = static_cast<signed char>((lane < 4 ? w0 : w1) >> (8 * (lane & 3)));
    }
    const uint32_t bits_c = mask_bits(top[0], top[1], top[2], top[3]), bits_m = mask_bits(mid[0], mid[1], mid[2], mid[3]);
    const int count = __popc(bits_c) | (__popc(bits_m) << 16);
    int incl = count;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int up = __shfl_up_sync(0xFFFFFFFFu, incl, o);
      if (lane >= o) incl += up;
    }
    const int total = __shfl_sync(0xFFFFFFFFu, incl, 31);
    const int excl = incl - count;
    int* dst = crit_row + (excl & 0xFFFF);
#pragma unroll
    for (int x = 0; x < 8; ++x)
      append_if(dst, 8 * c + x, bits_c & (1u << x));
    crit_row += total & 0xFFFF;
    if (marg_row != nullptr) {
      dst = marg_row + (excl >> 16);
#pragma unroll
      for (int x = 0; x < 8; ++x)
        append_if(dst, 8 * c + x, bits_m & (1u << x));
      marg_row += total >> 16;
    }
  }
  if (late_wait) sm100::wait_for_prior_grid();
}

constexpr size_t kSmemLimit = 227 * 1024, kCompactLimit = kSmemLimit - 256;  // (the kernel from places has static shared memory, too)
constexpr size_t plan_compact_smem_bytes(int nb, int rows) {
  return static_cast<size_t>(rows) * (place_pitch(nb) * 2 + kBuckets * 4 + kPicked * 2 + kHeadDim * 4 + rows * 4);
}
static_assert(plan_compact_smem_bytes(1 << 14, 8) > kCompactLimit, "counts are packed into 14 bits");

template <int R>
lite3r_status launch_compact(const lite3r_fp8& q, const lite3r_fp8& k, const lite3r_shape& s, const Counts& c,
                             const lite3r_plan& plan, int nb, int late_wait, cudaStream_t stream) {
  const size_t smem = plan_compact_smem_bytes(nb, R);
  lite3r_status st = ensure_dynamic_smem(plan_compact_kernel<R>, static_cast<int>(smem));
  if (st != LITE3R_OK) return st;
  const int row_tiles = ceil_div(nb, R);
  const int valid_last = s.tokens - (nb - 1) * s.block, mult_last = 128 / valid_last;
  const float factor_last = 128.f / static_cast<float>(valid_last * mult_last);
  return launch_dependent(plan_compact_kernel<R>, dim3(static_cast<unsigned>(s.batch * s.heads * row_tiles)), R * 32,
                          static_cast<int>(smem), stream, q.colsum, k.colsum, k.scales, s.tokens, s.block, nb, c.k_crit, c.k_marg,
                          c.k_neg, late_wait, mult_last, factor_last, plan.cls, plan.crit_idx, plan.marg_idx);
}

size_t plan_smem_bytes(int nb, int rows) {
  const size_t pitch = static_cast<size_t>((nb + 1) & ~1);
  const size_t common = rows * pitch * 8 + static_cast<size_t>(rows) * 2 * kBuckets * 4 +
                        static_cast<size_t>(rows) * 2 * kMaxListed * 2;  // keys, two histograms, two index lists
  // eight rows: score ranges and one bucket byte per key (the column sums come straight from global memory); one row: the
  // staged column sums as doubles
  if (rows == 8) return common + static_cast<size_t>(rows) * rows * sizeof(float2) + rows * pitch;
  return common + (1 + kStaged) * static_cast<size_t>(kPitch) * 8;
}

template <int R>
lite3r_status launch_rows(const lite3r_fp8& q, const lite3r_fp8& k, const lite3r_shape& s, const Counts& c,
                          const lite3r_plan& plan, int nb, int late_wait, cudaStream_t stream) {
  const size_t smem = plan_smem_bytes(nb, R);
  lite3r_status st = ensure_dynamic_smem(plan_kernel<R>, static_cast<int>(smem));
  if (st != LITE3R_OK) return st;
  const int row_tiles = ceil_div(nb, R);
  return launch_dependent(plan_kernel<R>, dim3(static_cast<unsigned>(s.batch * s.heads * row_tiles)), R * 32,
                          static_cast<int>(smem), stream, q.colsum, k.colsum, k.scales, s.tokens, s.block, nb, c.k_crit, c.k_marg,
                          c.k_neg, late_wait, plan.cls, plan.crit_idx, plan.marg_idx);
}

}  // namespace

// Test hook: which kernel launch_plan takes (0 = by size, as described there).
static std::atomic<int> g_plan_variant{0};
void set_plan_variant(int variant) { g_plan_variant.store(variant, std::memory_order_relaxed); }

lite3r_status launch_plan(const lite3r_fp8& q, const lite3r_fp8& k, const lite3r_shape& s, const Counts& c,
                          const lite3r_plan& plan, bool beside_prior, cudaStream_t stream) {
  const int late_wait = beside_prior ? 1 : 0;
  const int nb = ceil_div(s.tokens, s.block);
  switch (g_plan_variant.load(std::memory_order_relaxed)) {  // forced by a test; sizes that do not fit are refused
    case 1: return plan_smem_bytes(nb, 8) <= kSmemLimit ? launch_rows<8>(q, k, s, c, plan, nb, late_wait, stream) : LITE3R_ERR_UNSUPPORTED;
    case 2: return plan_compact_smem_bytes(nb, 8) <= kCompactLimit ? launch_compact<8>(q, k, s, c, plan, nb, late_wait, stream) : LITE3R_ERR_UNSUPPORTED;
    case 3: return plan_compact_smem_bytes(nb, 16) <= kCompactLimit ? launch_compact<16>(q, k, s, c, plan, nb, late_wait, stream) : LITE3R_ERR_UNSUPPORTED;
    case 4: return nb <= kLongestRow ? launch_rows<1>(q, k, s, c, plan, nb, late_wait, stream) : LITE3R_ERR_UNSUPPORTED;
    default: break;
  }
  // Rows of more than 80 blocks: approximate scores as 16-bit places.  Its fixed part is larger than that of the 64-bit keys
  // (16 heads of 65 blocks: 9.1 against 8.3 us), the share of every entry smaller: 512 heads of 86 blocks 92.5 against 97.0
  // us, 64 of 172 28 against 38.6, 16 of 687 61 against 108.  Eight rows per CTA where that is at most one CTA per SM: such a
  // CTA is done sooner (alone 1 head of 313 blocks 10.3 against 11.6 us, 5 of 129 7.6 against 8.1, 8 of 129 7.6 against 8.2) and, with half
  // the registers, starts beside the CTAs of the summaries instead of behind them (a pass of 5 heads of 129 blocks 44.8 against 47.9 us, of
  // 2 of 313 53.6 against 58.9).  Else sixteen where they fit (some 6300 blocks; 8 heads of 172 blocks 8.8 against 9.7 us, two of
  // 2147 71 against 102), else eight.
  constexpr int kShortRow = 80;
  if (nb > kShortRow) {
    int sms = 0;
    const lite3r_status st = sm_count(&sms);
    if (st != LITE3R_OK) return st;
    const bool sixteen = static_cast<long long>(s.batch) * s.heads * ceil_div(nb, 8) > sms;
    if (sixteen && plan_compact_smem_bytes(nb, 16) <= kCompactLimit) return launch_compact<16>(q, k, s, c, plan, nb, late_wait, stream);
    if (plan_compact_smem_bytes(nb, 8) <= kCompactLimit) return launch_compact<8>(q, k, s, c, plan, nb, late_wait, stream);
  }
  if (nb <= kShortRow) return launch_rows<8>(q, k, s, c, plan, nb, late_wait, stream);
  if (nb <= kLongestRow) return launch_rows<1>(q, k, s, c, plan, nb, late_wait, stream);  // (from some 13600 blocks on)
  return LITE3R_ERR_UNSUPPORTED;
}

}  // namespace lite3r
