// Token partition (Sec. 2.2, Eq. 3; App. B "dynamic token selection", Eq. 7)
// and the per-iteration active set (Sec. 2.2 modular rule, Sec. 2.3, Sec. 2.5
// caching window).
//
// Partition = a stable rank of the statistic.  Each fp32 value is mapped to an
// unsigned key whose integer order is the float order (-0 folded onto +0); the
// rank of a token is its position in the (key, token) order, which is the tie
// rule, and rank r maps to its group.  Three paths give the same groups:
//   N <= 4864     one launch ranks every token by counting the pairs before it;
//   N <= 360448   one launch of a cluster of 8 CTAs (keys spread over their
//                 shared memory) finds the pair at each group boundary and
//                 compares every token with those pairs;
//   larger N      a least-significant-digit radix sort of the (key, token)
//                 pairs: four passes of 8 bits, each a per-tile histogram, one
//                 exclusive scan of the (digit, tile) counts in digit-major
//                 order, and a stable scatter (the pairs start in token order,
//                 so equal keys stay in token order), then rank -> group.
//
// The active set needs no workspace: the CTAs of clusters count what comes
// before their tokens and compact (see active_set_kernel).
#include <cooperative_groups.h>

#include <algorithm>
#include <atomic>

#include "hsa_internal.cuh"

namespace hsa {
namespace {

constexpr int kSortThreads = 256;
constexpr int kTileThreads = 1024;
constexpr int kItems = 4;                               // per thread per tile
constexpr int kTile = kTileThreads * kItems;            // 4096 tokens
constexpr int kTileWarps = kTileThreads / 32;
constexpr int kWarpItems = kTile / kTileWarps;          // 128 consecutive tokens
constexpr int kScanCtas = 8;
constexpr int kMaxGroups = 32;

struct GroupStarts {
  int start[kMaxGroups];   // first rank of group k (ranks ascend with the statistic)
  int count[kMaxGroups];
};

constexpr size_t align256(size_t b) { return (b + 255) & ~(size_t)255; }

struct SortLayout {
  size_t keys0, keys1, vals0, vals1, hist, total;
  int tiles;
};

// Workspace layout of the radix-sort path; constexpr so that the fixed
// scratch array of hsa_partition_static is sized by this same formula.
constexpr SortLayout sort_layout(int N) {
  SortLayout L{};
  L.tiles = (int)(((long long)N + kTile - 1) / kTile);
  const size_t a = align256((size_t)N * 4);
  L.keys0 = 0;
  L.keys1 = a;
  L.vals0 = 2 * a;
  L.vals1 = 3 * a;
  L.hist = 4 * a;
  L.total = L.hist + align256((size_t)256 * L.tiles * 4);
  return L;
}

__device__ __forceinline__ uint32_t order_key(float f) {
  uint32_t u = __float_as_uint(f);
  if (u == 0x80000000u) u = 0u;                          // -0 ranks with +0
  return (u & 0x80000000u) ? ~u : (u | 0x80000000u);     // float order as uint order
}

// The sort's kernels are short (a few microseconds each at 524288 tokens, whose
// keys and tokens stay in L2), so each lets the next one launch at once and
// what bounds them is latency: every thread issues all its loads before it
// uses the first, and a tile is shared by 32 warps.  GPU time of a whole
// partition of 524288 tokens: 281 -> 48 us.
__global__ void __launch_bounds__(kSortThreads)
radix_key_kernel(const float *__restrict__ stat, int N, uint32_t *__restrict__ keys,
                 unsigned *err) {
  pdl_wait();
  pdl_trigger();
  const bool vec = (reinterpret_cast<uintptr_t>(stat) & 15) == 0;
  const int n4 = (int)(((unsigned)N + 3u) >> 2);
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n4; i += gridDim.x * blockDim.x) {
    float f[4];
    if (vec && 4 * i + 3 < N) {
      const float4 v = __ldg(reinterpret_cast<const float4 *>(stat) + i);
      f[0] = v.x, f[1] = v.y, f[2] = v.z, f[3] = v.w;
    } else {
#pragma unroll
      for (int e = 0; e < 4; ++e) f[e] = 4 * i + e < N ? __ldg(stat + 4 * i + e) : 0.f;
    }
    if (!(isfinite(f[0]) && isfinite(f[1]) && isfinite(f[2]) && isfinite(f[3])))
      set_error(err, kErrNonfinite);
    // the buffer holds whole 256-byte blocks, so the last vector may pass N
    reinterpret_cast<uint4 *>(keys)[i] =
        make_uint4(order_key(f[0]), order_key(f[1]), order_key(f[2]), order_key(f[3]));
  }
}

__global__ void __launch_bounds__(kTileThreads)
radix_hist_kernel(const uint32_t *__restrict__ keys, int N, int shift, uint32_t *__restrict__ hist,
                  int tiles) {
  pdl_wait();
  pdl_trigger();
  // four histograms, so that the warps of a concentrated digit (the exponent
  // bits of most statistics) contend less
  __shared__ uint32_t h[4][256];
  const int base = blockIdx.x * kTile + 4 * threadIdx.x;
  uint4 k = make_uint4(0u, 0u, 0u, 0u);
  if (base < N) k = *reinterpret_cast<const uint4 *>(keys + base);
  (&h[0][0])[threadIdx.x] = 0;
  __syncthreads();
  uint32_t *mine = h[(threadIdx.x >> 5) & 3];
  const uint32_t kk[4] = {k.x, k.y, k.z, k.w};
#pragma unroll
  for (int e = 0; e < 4; ++e)
    if (base + e < N) atomicAdd(&mine[(kk[e] >> shift) & 255u], 1u);
  __syncthreads();
  if (threadIdx.x < 256)
    hist[threadIdx.x * tiles + blockIdx.x] =
        h[0][threadIdx.x] + h[1][threadIdx.x] + h[2][threadIdx.x] + h[3][threadIdx.x];
}

// Exclusive scan, in place, of the 256*tiles counts in digit-major order, by
// one cluster: CTA c owns a contiguous share, sums it, learns the shares
// before it through distributed shared memory, then scans its share 4096
// counts (one 16-byte vector per thread) at a time.  One cluster instead of one
// block that gave each thread a contiguous (uncoalesced) run: at 524288 tokens
// 55 us -> about 4.
__global__ void __launch_bounds__(1024) radix_scan_kernel(uint32_t *__restrict__ hist, int total) {
  pdl_wait();
  pdl_trigger();
  namespace cg = cooperative_groups;
  cg::cluster_group cl = cg::this_cluster();
  __shared__ uint32_t warp_sum[32];
  __shared__ uint32_t share[kScanCtas];                  // every CTA's total
  cl.barrier_arrive();                                   // this CTA has started
  const int cta = (int)cl.block_rank(), ctas = (int)cl.num_blocks();
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  uint4 *h4 = reinterpret_cast<uint4 *>(hist);
  const int n4 = total / 4;                              // total is a multiple of 256
  const int lo = (int)((long long)n4 * cta / ctas), hi = (int)((long long)n4 * (cta + 1) / ctas);
  uint32_t s = 0;
#pragma unroll 4
  for (int i = lo + threadIdx.x; i < hi; i += 1024) {
    const uint4 v = h4[i];
    s += v.x + v.y + v.z + v.w;
  }
  s = __reduce_add_sync(0xffffffffu, s);
  if (lane == 0) warp_sum[w] = s;
  cl.barrier_wait();                                     // every CTA has, so its memory exists
  __syncthreads();
  if (w == 0) {
    const uint32_t t = __reduce_add_sync(0xffffffffu, warp_sum[lane]);
    if (lane < ctas) *cl.map_shared_rank(&share[cta], lane) = t;
  }
  cl.sync();                                             // every share has arrived
  uint32_t run = 0;
  for (int c = 0; c < cta; ++c) run += share[c];
  for (int b = lo; b < hi; b += 1024) {
    const int i = b + threadIdx.x;
    uint4 v = make_uint4(0u, 0u, 0u, 0u);
    if (i < hi) v = h4[i];
    const uint32_t sum = v.x + v.y + v.z + v.w;
    uint32_t incl = sum;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t t = __shfl_up_sync(0xffffffffu, incl, o);
      if (lane >= o) incl += t;
    }
    __syncthreads();                                     // warp_sum is free
    if (lane == 31) warp_sum[w] = incl;
    __syncthreads();
    const uint32_t ws = warp_sum[lane];
    const uint32_t before = __reduce_add_sync(0xffffffffu, lane < w ? ws : 0u);
    const uint32_t all = __reduce_add_sync(0xffffffffu, ws);
    const uint32_t x = run + before + incl - sum;
    if (i < hi) h4[i] = make_uint4(x, x + v.x, x + v.x + v.y, x + v.x + v.y + v.z);
    run += all;
  }
}

// Stable scatter of one tile.  Warp w owns tokens [w*128, w*128+128) of the
// tile and walks them 32 at a time in order; lanes holding the same digit find
// each other, so a token's rank among equal digits in the tile is (earlier warps'
// count) + (this warp's running count) + (earlier lanes of this step).  They do so
// by eight ballots, one per bit: __match_any_sync takes longer the more digits a
// warp holds, up to 32 on the low digits (9.7 us a pass at 524288 tokens against
// 7.9); on the last pass, the exponent bits, they are few and it is the faster
// (5.6 against 6.8).  The tile is first sorted in shared memory, so that
// neighbouring threads store neighbouring elements of a digit's run (16 on
// average): stored from where they stood, each 4-byte element cost a 32-byte
// sector, 12.7 us a pass.  vin NULL: the pairs are
// still in token order.  kout NULL: the last pass, whose keys nothing reads.
__global__ void __launch_bounds__(kTileThreads)
radix_scatter_kernel(const uint32_t *__restrict__ kin, const int32_t *__restrict__ vin,
                     uint32_t *__restrict__ kout, int32_t *__restrict__ vout, int N, int shift,
                     const uint32_t *__restrict__ offsets, int tiles) {
  pdl_wait();
  pdl_trigger();
  // the warps' digit counts, then the sorted tile (kTile keys, kTile tokens)
  __shared__ __align__(16) uint32_t cnt[kTileWarps][256];
  static_assert(sizeof(cnt) == 2 * kTile * sizeof(uint32_t), "the sorted tile reuses the counts");
  __shared__ uint32_t base_of[256];                      // digit's first place in the tile
  __shared__ uint32_t dst_of[256];                       // its first place in the output
  __shared__ uint32_t warp_sum[8];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int tile0 = blockIdx.x * kTile;
  const int base = tile0 + w * kWarpItems;
  uint32_t key[kItems];
  int32_t val[kItems];
  uint32_t local[kItems];
#pragma unroll
  for (int it = 0; it < kItems; ++it) {
    const int n = base + it * 32 + lane;
    key[it] = n < N ? kin[n] : 0u;
    val[it] = n < N && vin ? vin[n] : n;
  }
  if (threadIdx.x < 256) dst_of[threadIdx.x] = offsets[threadIdx.x * tiles + blockIdx.x];
  uint4 *c4 = reinterpret_cast<uint4 *>(&cnt[w][0]);
  c4[lane] = make_uint4(0u, 0u, 0u, 0u);                 // this warp's 256 counts
  c4[lane + 32] = make_uint4(0u, 0u, 0u, 0u);
  __syncwarp();
  const unsigned lt_mask = (1u << lane) - 1u;
#pragma unroll
  for (int it = 0; it < kItems; ++it) {
    const bool valid = base + it * 32 + lane < N;
    const uint32_t d = (key[it] >> shift) & 255u;
    unsigned peers;
    if (kout) {
      peers = __ballot_sync(0xffffffffu, valid);
#pragma unroll
      for (int b = 0; b < 8; ++b) {
        const bool bit = d >> b & 1u;
        const unsigned bal = __ballot_sync(0xffffffffu, bit);
        peers &= bit ? bal : ~bal;
      }
    } else {
      peers = __match_any_sync(0xffffffffu, valid ? d : 256u + lane);
    }
    const uint32_t before = valid ? cnt[w][d] : 0u;
    local[it] = before + __popc(peers & lt_mask);
    __syncwarp();
    if (valid && lane == __ffs(peers) - 1) cnt[w][d] = before + __popc(peers);
    __syncwarp();
  }
  __syncthreads();
  // exclusive prefix over warps: four neighbouring threads share a digit, each
  // eight warps of it
  {
    const int d = threadIdx.x >> 2, part = threadIdx.x & 3;
    constexpr int kPer = kTileWarps / 4;
    uint32_t c[kPer], sum = 0;
#pragma unroll
    for (int i = 0; i < kPer; ++i) {
      c[i] = cnt[part * kPer + i][d];
      sum += c[i];
    }
    uint32_t incl = sum;
#pragma unroll
    for (int o = 1; o < 4; o <<= 1) {
      const uint32_t t = __shfl_up_sync(0xffffffffu, incl, o, 4);
      if (part >= o) incl += t;
    }
    uint32_t run = incl - sum;
#pragma unroll
    for (int i = 0; i < kPer; ++i) {
      cnt[part * kPer + i][d] = run;
      run += c[i];
    }
    if (part == 3) base_of[d] = run;                     // tokens of the digit in the tile
  }
  __syncthreads();
  // exclusive prefix over digits
  uint32_t count = 0, incl = 0;
  if (threadIdx.x < 256) {
    count = incl = base_of[threadIdx.x];
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t t = __shfl_up_sync(0xffffffffu, incl, o);
      if (lane >= o) incl += t;
    }
    if (lane == 31) warp_sum[w] = incl;
  }
  __syncthreads();
  if (threadIdx.x < 256) {
    const uint32_t ws = lane < w ? warp_sum[lane & 7] : 0u;   // w < 8: earlier warps only
    base_of[threadIdx.x] = __reduce_add_sync(0xffffffffu, ws) + incl - count;
  }
  __syncthreads();
#pragma unroll
  for (int it = 0; it < kItems; ++it) {
    const uint32_t d = (key[it] >> shift) & 255u;
    local[it] += base_of[d] + cnt[w][d];
  }
  __syncthreads();                                       // the counts have been read
  uint32_t *skey = &cnt[0][0];
  int32_t *sval = reinterpret_cast<int32_t *>(skey + kTile);
#pragma unroll
  for (int it = 0; it < kItems; ++it) {
    if (base + it * 32 + lane < N) {
      skey[local[it]] = key[it];
      sval[local[it]] = val[it];
    }
  }
  __syncthreads();
  const int n_tile = min(kTile, N - tile0);
#pragma unroll
  for (int it = 0; it < kItems; ++it) {
    const int i = it * kTileThreads + threadIdx.x;
    if (i < n_tile) {
      const uint32_t k = skey[i];
      const uint32_t d = (k >> shift) & 255u;
      const uint32_t q = dst_of[d] + (i - base_of[d]);
      if (kout) kout[q] = k;
      vout[q] = sval[i];
    }
  }
}

// ------------------------------------------------ small layers: rank by count
//
// For N <= kRankMaxN every block holds all N keys in shared memory, and a
// token's rank is the number of tokens ordered before it by (key, index):
// exactly the ranks of the stable sort, in one launch instead of fourteen.
// A block takes 32 tokens (its lanes) and splits the key range over its
// warps; the partial counts are summed in shared memory.
// Issue-bound: N^2 / 32 comparisons.  Tokens of earlier blocks are all before
// this block's in index, later ones all behind, so outside the block's own 32
// tokens the pair order is one unsigned comparison of keys, against kn + 1
// (ties count) before them and kn (ties do not) behind them: two instructions
// per key and a quarter of a 16-byte broadcast load, instead of the five of
// the general pair test on single words.  Calls in a row (GPU time of a graph
// of 20): N = 3000 8.2 -> 3.8 us.
constexpr int kRankThreads = 512;
constexpr int kRankWarps = kRankThreads / 32;
constexpr int kRankTokens = 32;
// The keys (dynamic, whole 16-byte vectors) and the partial counts (static)
// stay within the 48 KB a block gets without opting in to more shared memory.
// One block per SM is the limit: 4500 tokens 4.9 us against 7.5 for the select
// below, 6144 tokens (a second block on some SMs) 8.9 against 8.0.
constexpr int kRankMaxN = 152 * kRankTokens;           // 4864
static_assert(kRankMaxN % 4 == 0 && kRankMaxN * 4 + kRankTokens * 4 <= 48 * 1024,
              "rank partition shared memory");

__global__ void __launch_bounds__(kRankThreads)
rank_partition_kernel(const float *__restrict__ stat, int N, int K, GroupStarts gs,
                      int32_t *__restrict__ group_of, unsigned *err) {
  pdl_wait();
  pdl_trigger();
  extern __shared__ uint4 skey4[];                       // N keys, padded with the largest key
  uint32_t *skey = reinterpret_cast<uint32_t *>(skey4);
  __shared__ int total[kRankTokens];
  const int n4 = (N + 3) >> 2;
  const bool vec = (reinterpret_cast<uintptr_t>(stat) & 15) == 0;
  for (int i = threadIdx.x; i < n4; i += kRankThreads) {
    float f[4];
    if (vec && 4 * i + 3 < N) {
      const float4 v = __ldg(reinterpret_cast<const float4 *>(stat) + i);
      f[0] = v.x, f[1] = v.y, f[2] = v.z, f[3] = v.w;
    } else {
#pragma unroll
      for (int e = 0; e < 4; ++e) f[e] = 4 * i + e < N ? __ldg(stat + 4 * i + e) : 0.f;
    }
    if (blockIdx.x == 0 &&
        !(isfinite(f[0]) && isfinite(f[1]) && isfinite(f[2]) && isfinite(f[3])))
      set_error(err, kErrNonfinite);
    uint32_t k[4];
#pragma unroll
    for (int e = 0; e < 4; ++e) k[e] = 4 * i + e < N ? order_key(f[e]) : 0xffffffffu;
    skey4[i] = make_uint4(k[0], k[1], k[2], k[3]);
  }
  if (threadIdx.x < kRankTokens) total[threadIdx.x] = 0;
  __syncthreads();
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int n = blockIdx.x * kRankTokens + lane;
  const uint32_t kn = n < N ? skey[n] : 0u;
  // 16-byte vectors [0, own0) hold earlier tokens, [own1, n4) later ones
  const int own0 = blockIdx.x * (kRankTokens / 4), own1 = min(n4, own0 + kRankTokens / 4);
  const int per = (n4 + kRankWarps - 1) / kRankWarps;
  const int v0 = min(n4, w * per), v1 = min(n4, v0 + per);
  int r = 0;
  auto count = [&](int lo, int hi, uint32_t bound) {     // keys below bound in vectors [lo, hi)
#pragma unroll 4
    for (int v = lo; v < hi; ++v) {
      const uint4 k = skey4[v];                          // the same vector for every lane
      r += k.x < bound;
      r += k.y < bound;
      r += k.z < bound;
      r += k.w < bound;
    }
  };
  count(v0, min(v1, own0), kn + 1u);                     // a finite key is below 2^32 - 1
  for (int v = max(v0, own0); v < min(v1, own1); ++v) {
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      const int m = 4 * v + e;
      r += (skey[m] < kn) + ((skey[m] == kn) & (m < n));
    }
  }
  count(max(v0, own1), v1, kn);
  atomicAdd(&total[lane], r);
  __syncthreads();
  if (w == 0 && n < N) {
    const int rank = total[lane];
    int g = 0;
    for (int k = 0; k < K; ++k)
      if (rank >= gs.start[k] && rank < gs.start[k] + gs.count[k]) g = k;
    group_of[n] = g;
  }
}

// ------------------------------------------------ larger layers: select
//
// A token's group depends only on which group boundaries its rank passes:
// rank >= start[k] for k = 0 .. K-2 (group K-1 holds the lowest ranks), and
// rank >= b holds exactly when (key, token) >= the pair of rank b in the
// (key, token) order.  So it is enough to find the pair of each boundary rank
// and to compare every token with those pairs: one launch instead of a sort's
// fourteen, and the same ranks as the stable sort.
//
// It runs on one thread-block cluster.  CTA c holds the keys of tokens
// [c*chunk, (c+1)*chunk) in its shared memory.
//   1. The cluster's smallest and largest key.
//   2. A histogram of 2048 or 4096 bins over that range (2^s keys each); every
//      CTA sums the cluster's through distributed shared memory and finds each
//      boundary's bin (identical integer work on identical data, so no broadcast
//      is needed).  The bins follow the values at hand, so they hold few keys
//      (a lognormal statistic of 75600 tokens: about 120 at a quartile) and
//      their counters seldom collide.
//   3. The keys of a boundary's bin, with their tokens, go to the list of the
//      CTA that owns the boundary (boundary j: CTA j mod 8), which finds the
//      pair with the right number of smaller pairs and writes it to every CTA.
// A bin with more than kCsList keys is split further first, 256 ways per pass,
// until it holds fewer or a single key value; a value that more tokens share is
// resolved by counting it in token order (CTA order is token order).
// Cluster barriers are hardware barriers that every thread of every CTA
// reaches, so none can wait forever.  Latency-bound (8 SMs, four cluster
// barriers): 12033 tokens 26.8 -> 8.3 us, 75600 43 -> 13.8, 360448
// 110 -> 37, against four fixed 8-bit digit passes with two barriers each and bins
// that most keys shared.  Of the 75600 tokens' 12 us in the kernel, reading the
// eight histograms takes 2, the two sweeps and the lists 5.
constexpr int kMaxBounds = kMaxGroups - 1;
constexpr int kCsCtas = 8;
constexpr int kCsThreads = 1024;
constexpr int kCsMaxChunk = 44 * 1024;                 // keys per CTA: 176 KB
constexpr int kCsMaxN = kCsCtas * kCsMaxChunk;         // 360448 tokens
constexpr int kCsFineN = 98304;                        // above: 4096 bins
constexpr int kCsList = 512;                           // pairs a boundary's list holds
constexpr int kCsLists = (kMaxBounds + kCsCtas - 1) / kCsCtas;   // boundaries a CTA owns
constexpr int kCsHist = kMaxBounds * 256;              // counters, 4096 in the first histogram
static_assert(kCsList * 2 == kCsThreads && kCsHist >= 4 * kCsThreads, "select layout");
constexpr int kCsFixedBytes = kCsHist * 4 + kCsLists * kCsList * 8;   // besides the keys

// kPer: bins per thread of the first histogram.
template <int kPer>
__global__ void __cluster_dims__(kCsCtas, 1, 1) __launch_bounds__(kCsThreads, 1)
cluster_select_kernel(const float *__restrict__ stat, int N, int chunk, int K, GroupStarts gs,
                      int32_t *__restrict__ group_of, unsigned *err) {
  pdl_wait();
  pdl_trigger();
  namespace cg = cooperative_groups;
  cg::cluster_group cl = cg::this_cluster();
  extern __shared__ uint4 cs_smem[];
  unsigned long long *list = reinterpret_cast<unsigned long long *>(cs_smem);
  uint32_t *hist = reinterpret_cast<uint32_t *>(list + kCsLists * kCsList);
  uint4 *ckey4 = reinterpret_cast<uint4 *>(hist + kCsHist);   // this CTA's keys
  uint32_t *skey = reinterpret_cast<uint32_t *>(ckey4);
  __shared__ uint2 range[kCsCtas];                     // every CTA's smallest, largest key
  __shared__ uint32_t low[kMaxBounds];                 // boundary j's keys: [low, low + 2^sh)
  __shared__ int sh[kMaxBounds];
  __shared__ int below[kMaxBounds];                    // keys below low
  __shared__ int count[kMaxBounds];                    // keys in the range
  __shared__ int fill[kMaxBounds];                     // place of this CTA's next pair of them
  __shared__ int slot[kMaxBounds];                     // first boundary with the same range
  __shared__ int target[kMaxBounds];                   // boundary's rank; -1: 0 or N
  __shared__ int split;                                // whether a range holds too many keys
  __shared__ int whole;                                // whether a pass left one's keys together
  __shared__ uint32_t kmn[kMaxBounds], kmx[kMaxBounds];   // such a range's keys in this CTA
  __shared__ unsigned long long thr[kMaxBounds];       // boundary pair (key << 32 | token)
  __shared__ int eqc[kMaxBounds];                      // local keys equal to a boundary key
  __shared__ int warp_tot[kCsThreads / 32];
  __shared__ uint32_t warp_min[kCsThreads / 32], warp_max[kCsThreads / 32];
  cl.barrier_arrive();                                 // this CTA has started
  const int cta = (int)cl.block_rank();
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int nb = K - 1;
  const int lo = min(N, cta * chunk), hi = min(N, lo + chunk);
  const int n_loc = hi - lo;
  const int n4 = (n_loc + 3) >> 2;
  // keys of [lo, hi); chunk is a multiple of 4, so a 16-byte aligned stat
  // gives 16-byte aligned rows
  const bool vec = (reinterpret_cast<uintptr_t>(stat) & 15) == 0;
  uint32_t kmin = 0xffffffffu, kmax = 0u;
#pragma unroll 4
  for (int i = threadIdx.x; i < n4; i += kCsThreads) {
    float f[4];
    if (vec && 4 * i + 3 < n_loc) {
      const float4 v = __ldg(reinterpret_cast<const float4 *>(stat + lo) + i);
      f[0] = v.x, f[1] = v.y, f[2] = v.z, f[3] = v.w;
    } else {
#pragma unroll
      for (int e = 0; e < 4; ++e)                      // past the end: the last key again
        f[e] = __ldg(stat + lo + min(4 * i + e, n_loc - 1));
    }
    if (!(isfinite(f[0]) && isfinite(f[1]) && isfinite(f[2]) && isfinite(f[3])))
      set_error(err, kErrNonfinite);
    const uint4 k = make_uint4(order_key(f[0]), order_key(f[1]), order_key(f[2]), order_key(f[3]));
    kmin = min(kmin, min(min(k.x, k.y), min(k.z, k.w)));
    kmax = max(kmax, max(max(k.x, k.y), max(k.z, k.w)));
    ckey4[i] = k;
  }
#pragma unroll
  for (int i = 0; i < kPer; ++i) hist[i * kCsThreads + threadIdx.x] = 0u;
  if (threadIdx.x < nb) {
    const int r = gs.start[threadIdx.x];
    target[threadIdx.x] = r > 0 && r < N ? r : -1;
    thr[threadIdx.x] = r <= 0 ? 0ull : ~0ull;
    eqc[threadIdx.x] = 0;
    count[threadIdx.x] = 0;
    fill[threadIdx.x] = kCsList;
  }
  if (threadIdx.x == 0) split = whole = 0;
  kmin = __reduce_min_sync(0xffffffffu, kmin);
  kmax = __reduce_max_sync(0xffffffffu, kmax);
  if (lane == 0) {
    warp_min[w] = kmin;
    warp_max[w] = kmax;
  }
  cl.barrier_wait();                                   // every CTA has, so its memory exists
  __syncthreads();
  if (w == 0) {
    kmin = __reduce_min_sync(0xffffffffu, warp_min[lane]);
    kmax = __reduce_max_sync(0xffffffffu, warp_max[lane]);
    if (lane < kCsCtas) *cl.map_shared_rank(&range[cta], lane) = make_uint2(kmin, kmax);
  }
  cl.sync();                                           // every CTA's range has arrived
#pragma unroll
  for (int r = 0; r < kCsCtas; ++r) {
    kmin = r ? min(kmin, range[r].x) : range[0].x;
    kmax = r ? max(kmax, range[r].y) : range[0].y;
  }
  // bins of 2^s keys: (kmax - kmin) >> s < 1024 * kPer
  int s = max(0, (kPer == 4 ? 20 : 21) - __clz(kmax - kmin));
  for (int i = threadIdx.x; i < n4; i += kCsThreads) {
    const uint4 k4 = ckey4[i];
    const uint32_t kk[4] = {k4.x, k4.y, k4.z, k4.w};
#pragma unroll
    for (int e = 0; e < 4; ++e)
      if (4 * i + e < n_loc) atomicAdd(&hist[(kk[e] - kmin) >> s], 1u);
  }
  cl.sync();                                           // every CTA's histogram is complete
  {
    // thread t: bins kPer*t .. of the cluster's histogram, then their prefix
    uint32_t hv[kCsCtas][kPer];
#pragma unroll
    for (int r = 0; r < kCsCtas; ++r) {
      const uint32_t *h = cl.map_shared_rank(hist, r) + kPer * threadIdx.x;
      if constexpr (kPer == 4)
        *reinterpret_cast<uint4 *>(hv[r]) = *reinterpret_cast<const uint4 *>(h);
      else
        *reinterpret_cast<uint2 *>(hv[r]) = *reinterpret_cast<const uint2 *>(h);
    }
    int c[kPer], before[kPer], sum = 0;                // before: in earlier CTAs
#pragma unroll
    for (int b = 0; b < kPer; ++b) {
      c[b] = before[b] = 0;
#pragma unroll
      for (int r = 0; r < kCsCtas; ++r) {
        c[b] += (int)hv[r][b];
        before[b] += r < cta ? (int)hv[r][b] : 0;
      }
      sum += c[b];
    }
    int incl = sum;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int t = __shfl_up_sync(0xffffffffu, incl, o);
      if (lane >= o) incl += t;
    }
    if (lane == 31) warp_tot[w] = incl;
    __syncthreads();
    const int wt = warp_tot[lane];
    const int excl = __reduce_add_sync(0xffffffffu, lane < w ? wt : 0) + incl - sum;
    for (int j = 0; j < nb; ++j) {
      int t = target[j] - excl;                        // ranks 0 and N fall in no bin
      if (t < 0 || t >= sum) continue;
#pragma unroll
      for (int b = 0; b < kPer; ++b) {
        if (t >= 0 && t < c[b]) {
          low[j] = kmin + ((uint32_t)(kPer * threadIdx.x + b) << s);
          sh[j] = s;
          below[j] = target[j] - t;
          count[j] = c[b];
          fill[j] = before[b];
          if (c[b] > kCsList && s > 0) split = 1;
        }
        t -= c[b];
      }
    }
  }
  __syncthreads();
  // Split the ranges that hold too many keys, 256 ways at a time.  All of them
  // are 2^s wide here, and every thread of the cluster takes the same turns.  A pass
  // that leaves all keys of a range together may have met a value that fills it (a
  // statistic of few values), so the next one also looks at the keys' extremes and
  // need not split down to that value: 8 values, 4865 tokens 23.2 -> 17.6 us (18.6 by
  // ranking), 75600 38.6 -> 31.1.  Looking in every pass would be better for them (13.0,
  // 23.5) but costs spread statistics 3 to 13 %, after such a pass only 0 to 0.3 us.
  while (__builtin_expect(split, 0)) {
    const int ns = max(0, s - 8);
    const bool look = whole;
    if (threadIdx.x < nb) {
      const int j = threadIdx.x;
      int first = -1;
      if (target[j] >= 0 && count[j] > kCsList && sh[j] == s) {
        first = 0;
        while (!(target[first] >= 0 && sh[first] == s && low[first] == low[j])) ++first;
      }
      slot[j] = first;                                 // -1: not split
    }
    cl.sync();                  // every CTA has read the histograms of the last pass
    if (threadIdx.x == 0) split = whole = 0;
    if (look && threadIdx.x < nb) {
      kmn[threadIdx.x] = 0xffffffffu;
      kmx[threadIdx.x] = 0u;
    }
    for (int i = threadIdx.x; i < nb * 256; i += kCsThreads) hist[i] = 0u;
    __syncthreads();
    if (__builtin_expect(look, 0)) {
      for (int i = threadIdx.x; i < n_loc; i += kCsThreads) {
        const uint32_t k = skey[i];
        for (int j = 0; j < nb; ++j) {
          if (slot[j] != j || (k - low[j]) >> s != 0) continue;
          atomicAdd(&hist[j * 256 + ((k - low[j]) >> ns)], 1u);
          if (k < kmn[j]) atomicMin(&kmn[j], k);
          if (k > kmx[j]) atomicMax(&kmx[j], k);
        }
      }
    } else {
      for (int i = threadIdx.x; i < n_loc; i += kCsThreads) {
        const uint32_t k = skey[i];
        for (int j = 0; j < nb; ++j)
          if (slot[j] == j && (k - low[j]) >> s == 0)
            atomicAdd(&hist[j * 256 + ((k - low[j]) >> ns)], 1u);
      }
    }
    cl.sync();                                         // every CTA's histograms are complete
    // warp j picks boundary j's part of its range
    uint32_t mn = 1u, mx = 0u;
    if (look && w < nb && slot[w] >= 0) {
      mn = *cl.map_shared_rank(&kmn[slot[w]], lane % kCsCtas);
      mx = *cl.map_shared_rank(&kmx[slot[w]], lane % kCsCtas);
      mn = __reduce_min_sync(0xffffffffu, mn);
      mx = __reduce_max_sync(0xffffffffu, mx);
    }
    if (mn == mx) {                                    // one value: low, and done
      if (lane == 0) {
        low[w] = mn;
        sh[w] = 0;
      }
    } else if (w < nb && slot[w] >= 0) {
      const int t = target[w] - below[w];              // rank among the range's keys
      int c[8], before[8], sum = 0;
#pragma unroll
      for (int i = 0; i < 8; ++i) c[i] = before[i] = 0;
      for (int r = 0; r < kCsCtas; ++r) {
        const uint4 *h = reinterpret_cast<const uint4 *>(cl.map_shared_rank(hist, r) +
                                                         slot[w] * 256 + 8 * lane);
        const uint4 h0 = h[0], h1 = h[1];
        const int v[8] = {(int)h0.x, (int)h0.y, (int)h0.z, (int)h0.w,
                          (int)h1.x, (int)h1.y, (int)h1.z, (int)h1.w};
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          c[i] += v[i];
          before[i] += r < cta ? v[i] : 0;
        }
      }
#pragma unroll
      for (int i = 0; i < 8; ++i) sum += c[i];
      int incl = sum;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int v = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += v;
      }
      __syncwarp();                                    // every lane has read low and below
      int at = t - (incl - sum);
      if (at >= 0 && at < sum) {                       // exactly one lane
#pragma unroll
        for (int d = 0; d < 8; ++d) {
          if (at >= 0 && at < c[d]) {
            low[w] += (uint32_t)(8 * lane + d) << ns;
            sh[w] = ns;
            below[w] = target[w] - at;
            if (c[d] == count[w]) whole = 1;
            count[w] = c[d];
            fill[w] = before[d];
            if (c[d] > kCsList && ns > 0) split = 1;
          }
          at -= c[d];
        }
      }
    }
    __syncthreads();
    s = ns;
  }
  // The pairs of each boundary's range go to its owner's list, after those of
  // earlier CTAs (the histograms say how many); a single key value that more
  // than kCsList tokens share is only counted.
  // Four boundaries per sweep, held in registers.
  for (int j0 = 0; j0 < nb; j0 += 4) {
    uint32_t l[4];
    int b[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const bool on = j0 + q < nb && target[j0 + q] >= 0;
      l[q] = on ? low[j0 + q] : 0xffffffffu;           // no finite value's key
      b[q] = on ? sh[j0 + q] : 0;
    }
    for (int i = threadIdx.x; i < n4; i += kCsThreads) {
      const uint4 k4 = ckey4[i];
      const uint32_t kk[4] = {k4.x, k4.y, k4.z, k4.w};
#pragma unroll
      for (int q = 0; q < 4; ++q) {
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          if ((kk[e] - l[q]) >> b[q] != 0 || 4 * i + e >= n_loc || j0 + q >= nb) continue;
          const int j = j0 + q;
          if (count[j] > kCsList) {
            atomicAdd(&eqc[j], 1);
          } else {
            const int at = atomicAdd(&fill[j], 1);
            if (at < kCsList)            // more only with a NaN among the keys
              *cl.map_shared_rank(&list[(j / kCsCtas) * kCsList + at], j % kCsCtas) =
                  ((unsigned long long)kk[e] << 32) | (unsigned)(lo + 4 * i + e);
          }
        }
      }
    }
  }
  cl.sync();                                           // the lists and eqc are complete
  bool shared_value = false;
  for (int j = 0; j < nb; ++j) shared_value |= target[j] >= 0 && count[j] > kCsList;
  for (int j = cta; j < nb; j += kCsCtas) {
    if (target[j] < 0 || count[j] > kCsList) continue;
    // 2^lg neighbouring threads per candidate, each a part of the list
    const unsigned long long *l = list + (j / kCsCtas) * kCsList;
    const int m = count[j], need = target[j] - below[j];
    const int lg = min(5, __clz(max(m - 1, 1)) - 22);  // m <= 2^(10 - lg)
    const int c = threadIdx.x >> lg, part = threadIdx.x & ((1 << lg) - 1);
    const unsigned long long pair = l[min(c, m - 1)];
    int less = 0;
#pragma unroll 8
    for (int i = part; i < m; i += 1 << lg) less += l[i] < pair;
    for (int o = 1; o < 1 << lg; o <<= 1) less += __shfl_xor_sync(0xffffffffu, less, o);
    if (c < m && less == need)
      for (int r = part; r < kCsCtas; r += 1 << lg) *cl.map_shared_rank(&thr[j], r) = pair;
  }
  // A shared value: the need-th of its tokens, in token order.  One sweep over
  // a contiguous run of tokens per thread (an odd run length spreads a warp's
  // reads over the shared-memory banks).
  const int run = ((n_loc + kCsThreads - 1) / kCsThreads) | 1;
  const int r0 = min(n_loc, (int)threadIdx.x * run), r1 = min(n_loc, r0 + run);
  for (int j = 0; __builtin_expect(shared_value, 0) && j < nb; ++j) {
    if (target[j] < 0 || count[j] <= kCsList) continue;   // the same in every thread
    int before_cta = 0;                                // equal keys in earlier CTAs
    for (int r = 0; r < cta; ++r) before_cta += *cl.map_shared_rank(&eqc[j], r);
    const int need = target[j] - below[j] - before_cta;
    if (need < 0 || need >= eqc[j]) continue;          // another CTA holds it
    const uint32_t kj = low[j];
    int eq = 0;
    for (int n = r0; n < r1; ++n) eq += skey[n] == kj;
    int incl = eq;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int t = __shfl_up_sync(0xffffffffu, incl, o);
      if (lane >= o) incl += t;
    }
    __syncthreads();                                   // warp_tot is free
    if (lane == 31) warp_tot[w] = incl;
    __syncthreads();
    const int wt = warp_tot[lane];
    const int before = __reduce_add_sync(0xffffffffu, lane < w ? wt : 0) + incl - eq;
    if (need >= before && need < before + eq) {
      int seen = before;
      for (int n = r0; n < r1; ++n) {
        if (skey[n] != kj) continue;
        if (seen == need) {
          const unsigned long long pair = ((unsigned long long)kj << 32) | (unsigned)(lo + n);
          for (int r = 0; r < kCsCtas; ++r) *cl.map_shared_rank(&thr[j], r) = pair;
          break;
        }
        ++seen;
      }
    }
  }
  cl.sync();                  // the boundary pairs have reached every CTA
  unsigned long long t4[4];                            // the first four, in registers
#pragma unroll
  for (int q = 0; q < 4; ++q) t4[q] = q < nb ? thr[q] : ~0ull;
  const bool vec_out = (reinterpret_cast<uintptr_t>(group_of) & 15) == 0;
  for (int i = threadIdx.x; i < n4; i += kCsThreads) {
    const uint4 k4 = ckey4[i];
    const uint32_t kk[4] = {k4.x, k4.y, k4.z, k4.w};
    int g[4] = {nb, nb, nb, nb};
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      const unsigned long long kn = ((unsigned long long)kk[e] << 32) | (unsigned)(lo + 4 * i + e);
#pragma unroll
      for (int q = 0; q < 4; ++q) g[e] -= kn >= t4[q];
      for (int j = 4; j < nb; ++j) g[e] -= kn >= thr[j];
    }
    int32_t *dst = group_of + lo + 4 * i;
    if (vec_out && 4 * i + 3 < n_loc) {
      *reinterpret_cast<int4 *>(dst) = make_int4(g[0], g[1], g[2], g[3]);
    } else {
#pragma unroll
      for (int e = 0; e < 4; ++e)
        if (4 * i + e < n_loc) dst[e] = g[e];
    }
  }
}

__global__ void __launch_bounds__(kSortThreads)
group_assign_kernel(const int32_t *__restrict__ sorted_tokens, int N, int K, GroupStarts gs,
                    int32_t *__restrict__ group_of) {
  pdl_wait();
  pdl_trigger();
  // unsigned: the index one stride past the last token may pass 2^31
  for (unsigned u = blockIdx.x * blockDim.x + threadIdx.x; u < (unsigned)N;
       u += gridDim.x * blockDim.x) {
    const int r = (int)u;
    const int token = sorted_tokens[r];
    int g = 0;
    for (int k = 0; k < K; ++k)
      if (r >= gs.start[k] && r < gs.start[k] + gs.count[k]) g = k;
    group_of[token] = g;
  }
}

// --------------------------------------- active set and token reordering
//
// Workspace-free compaction in one launch of any size: the active set lists
// the tokens of the groups that are active; the reordering (Sec. 2.5: new
// position r holds old token order[r]) lists the non-baseline tokens, then the
// baseline group, each in token order.  CTA b owns `rounds` * kAcThreads *
// kItems consecutive tokens; in a round a warp owns 32 * kItems of them, 32 at a
// time (ballots rank them, and every load and store is coalesced).  To know how
// many marked tokens come before its own, a cluster's CTAs split the tokens of
// all earlier clusters among themselves, add their own counts, and exchange
// both through distributed shared memory, so nothing waits on another cluster.
// Bound by latency (launch, one load, one cluster barrier, one store); with
// kAcMaxClusters clusters each group id is read again six times on average, from
// L2.  12 clusters are resident at once; with 16 a second wave of clusters cost
// 20-30 %.  One cluster for the whole layer, as before, left 144 SMs idle.  GPU
// time of an active set in a row of calls: 6144 tokens 2.9 -> 2.8 us, 75600
// 6.3 -> 4.0, 524288 26 -> 8.3, 2097152 95 -> 20 (4194304, which took blocks
// that each counted everything before them, 245 -> 35).
constexpr int kAcThreads = 1024;
constexpr int kAcCtas = 8;                             // CTAs of a cluster
constexpr int kAcMaxClusters = 12;

// Scans this CTA's rounds: emit(n, g, marked, rank) for every token n < N with
// its group id g, whether mark(g), and the number of marked tokens before n.
template <int kItems, class Mark, class Emit>
__device__ __forceinline__ void compact(const int32_t *__restrict__ group_of, int N, int rounds,
                                        Mark mark, Emit emit) {
  namespace cg = cooperative_groups;
  cg::cluster_group cl = cg::this_cluster();
  __shared__ int warp_cnt[2][kAcThreads / 32], warp_before[kAcThreads / 32];
  __shared__ int own[kAcCtas], earlier[kAcCtas];       // by CTA of the cluster
  const int cta = (int)cl.block_rank(), ctas = (int)cl.num_blocks();
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const unsigned below = (1u << lane) - 1u;
  constexpr int kTile = kAcThreads * kItems;
  const long long per_cta = (long long)rounds * kTile;
  const long long own0 = (long long)blockIdx.x * per_cta + (w * kItems * 32 + lane);
  // group ids of this lane's tokens of a round, and the marks of its warp's
  int g[kItems];
  unsigned bal[kItems];
  auto load = [&](int r) {
#pragma unroll
    for (int e = 0; e < kItems; ++e) {
      const long long n = own0 + (long long)r * kTile + e * 32;
      g[e] = n < N ? __ldg(group_of + n) : 0;
    }
    int c = 0;
#pragma unroll
    for (int e = 0; e < kItems; ++e) {
      bal[e] = __ballot_sync(0xffffffffu, own0 + (long long)r * kTile + e * 32 < N && mark(g[e]));
      c += __popc(bal[e]);
    }
    return c;                                          // the same in every lane
  };
  int base = 0;                                        // marked tokens before this CTA's
  int c0 = load(0);
  if (gridDim.x > 1) {
    cl.barrier_arrive();                               // this CTA has started
    int c = c0;
    for (int r = 1; r < rounds; ++r) c += load(r);
    if (rounds > 1) c0 = load(0);
    // the earlier clusters own whole CTAs' worth of tokens, all inside N
    const long long n_before = (long long)(blockIdx.x / ctas) * per_cta;   // tokens per CTA
    const int32_t *from = group_of + cta * n_before;
    int e = 0;
    if ((reinterpret_cast<uintptr_t>(group_of) & 15) == 0) {   // per_cta is a multiple of 4
      const int4 *f4 = reinterpret_cast<const int4 *>(from);
#pragma unroll 8
      for (long long i = threadIdx.x; i < n_before / 4; i += kAcThreads) {
        const int4 v = __ldg(f4 + i);
        e += (int)mark(v.x) + (int)mark(v.y) + (int)mark(v.z) + (int)mark(v.w);
      }
    } else {
#pragma unroll 8
      for (long long i = threadIdx.x; i < n_before; i += kAcThreads) e += (int)mark(__ldg(from + i));
    }
    e = __reduce_add_sync(0xffffffffu, e);
    if (lane == 0) {
      warp_cnt[0][w] = c;
      warp_before[w] = e;
    }
    cl.barrier_wait();                                 // every CTA has, so its memory exists
    __syncthreads();
    if (w == 0) {
      c = __reduce_add_sync(0xffffffffu, warp_cnt[0][lane]);
      e = __reduce_add_sync(0xffffffffu, warp_before[lane]);
      if (lane < ctas) {
        *cl.map_shared_rank(&own[cta], lane) = c;
        *cl.map_shared_rank(&earlier[cta], lane) = e;
      }
    }
    cl.sync();                                         // every CTA's counts have arrived
    for (int r = 0; r < ctas; ++r) base += earlier[r] + (r < cta ? own[r] : 0);
  }
  for (int r = 0; r < rounds; ++r) {
    if (r > 0) c0 = load(r);
    // two buffers: a warp writes the next round's count only after every warp
    // has passed this round's barrier
    if (lane == 0) warp_cnt[(r + 1) & 1][w] = c0;
    __syncthreads();
    const int wc = warp_cnt[(r + 1) & 1][lane];
    int rank = base + __reduce_add_sync(0xffffffffu, lane < w ? wc : 0);
    base += __reduce_add_sync(0xffffffffu, wc);
#pragma unroll
    for (int e = 0; e < kItems; ++e) {
      const long long n = own0 + (long long)r * kTile + e * 32;
      if (n < N) emit((int)n, g[e], bal[e] >> lane & 1u, rank + __popc(bal[e] & below));
      rank += __popc(bal[e]);
    }
  }
}

template <int kItems>
__global__ void __launch_bounds__(kAcThreads, 1)
active_set_kernel(const int32_t *__restrict__ group_of, int N, int rounds, int K, uint32_t mask,
                  int32_t *__restrict__ idx, int32_t *__restrict__ pos, unsigned *err) {
  pdl_wait();
  pdl_trigger();
  compact<kItems>(
      group_of, N, rounds,
      [&](int g) { return (unsigned)g < (unsigned)K && (mask >> g & 1u); },
      [&](int n, int g, bool active, int rank) {
        if ((unsigned)g >= (unsigned)K) set_error(err, kErrIndex);
        if (active) idx[rank] = n;
        if (pos) pos[n] = active ? rank : -1;
      });
}

template <int kItems>
__global__ void __launch_bounds__(kAcThreads, 1)
reorder_kernel(const int32_t *__restrict__ group_of, int N, int rounds, int M,
               int32_t *__restrict__ order, int32_t *__restrict__ where,
               int32_t *__restrict__ group_new, unsigned *err) {
  pdl_wait();
  pdl_trigger();
  compact<kItems>(
      group_of, N, rounds, [&](int g) { return g != 0; },
      [&](int n, int g, bool moved, int rank) {
        // n - rank baseline tokens come before n
        const long long r = moved ? rank : (long long)M + (n - rank);
        if (moved ? rank < M : r < N) {
          order[r] = n;
          if (where) where[n] = (int)r;
          if (group_new) group_new[r] = g;
        } else {
          set_error(err, kErrIndex);
        }
      });
}

}  // namespace
}  // namespace hsa

using namespace hsa;

namespace {

// Opts the cluster kernel in to its shared memory on the current device and
// checks that one cluster of kCsCtas such CTAs can be resident; otherwise the
// partition takes the radix-sort path.  Resolved once per device.
template <int kPer>
bool cluster_select_ready() {
  static std::atomic<int> state[64];            // 0 unknown, 1 ready, 2 unavailable
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return false;
  int st = state[dev].load();
  if (st == 0) {
    st = 2;
    const int smem = kCsMaxChunk * (int)sizeof(uint32_t) + kCsFixedBytes;
    if (cudaFuncSetAttribute(cluster_select_kernel<kPer>,
                             cudaFuncAttributeMaxDynamicSharedMemorySize, smem) == cudaSuccess) {
      cudaLaunchConfig_t cfg = {};
      cfg.gridDim = dim3(kCsCtas);
      cfg.blockDim = dim3(kCsThreads);
      cfg.dynamicSmemBytes = smem;
      int clusters = 0;
      if (cudaOccupancyMaxActiveClusters(&clusters, cluster_select_kernel<kPer>, &cfg) ==
              cudaSuccess &&
          clusters >= 1)
        st = 1;
    }
    cudaGetLastError();                          // a refused query leaves no sticky error
    state[dev].store(st);
  }
  return st == 1;
}

// Whether one cluster of `ctas` CTAs of kernel K can be resident on the
// current device, resolved once per device.
template <auto K>
bool cluster_ready(int ctas, int threads) {
  static std::atomic<int> state[64];            // 0 unknown, 1 ready, 2 unavailable
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return false;
  int st = state[dev].load();
  if (st == 0) {
    st = 2;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(ctas);
    cfg.blockDim = dim3(threads);
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = (unsigned)ctas;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    int clusters = 0;
    if (cudaOccupancyMaxActiveClusters(&clusters, K, &cfg) == cudaSuccess && clusters >= 1) st = 1;
    cudaGetLastError();                          // a refused query leaves no sticky error
    state[dev].store(st);
  }
  return st == 1;
}

bool cluster_scan_ready() { return cluster_ready<radix_scan_kernel>(kScanCtas, 1024); }

// Launches a compaction kernel over N tokens: one CTA where one round of it
// covers them (1.3 us against 2.6 for a cluster), else clusters; one token per
// thread and round while a single cluster covers the layer that way (8192
// tokens; 6144: 2.8 us against 3.4 with four), four otherwise (fewer barriers
// per token); one round per CTA until kAcMaxClusters are in flight, then more.  Without
// room for a cluster of 8, clusters of one CTA.
template <auto Kernel1, auto Kernel4, typename... Rest>
void launch_compact(cudaStream_t s, const int32_t *group_of, int N, Rest... rest) {
  const bool one = N <= kAcCtas * kAcThreads;
  const long long tile = one ? kAcThreads : 4 * kAcThreads;
  const long long tiles = ((long long)N + tile - 1) / tile;
  unsigned ctas = 1;
  long long rounds = 1, grid = 1;
  if (tiles > 1) {
    ctas = cluster_ready<Kernel4>(kAcCtas, kAcThreads) ? kAcCtas : 1;
    const long long most = (long long)kAcMaxClusters * kAcCtas;
    rounds = (tiles + most - 1) / most;
    grid = (tiles + rounds * ctas - 1) / (rounds * ctas) * ctas;
  }
  count_launches(1);
  launch_pdl_cluster(one ? Kernel1 : Kernel4, dim3((unsigned)grid), dim3(kAcThreads), ctas, s,
                     group_of, N, (int)rounds, rest...);
}

}  // namespace

extern "C" size_t hsa_partition_workspace_bytes(int N) {
  if (N <= 0) return 0;
  return sort_layout(N).total;
}

extern "C" int hsa_partition(const float *stat, int N, int T, const int *budgets,
                             const int *counts, int K, int32_t *group_of, void *workspace,
                             size_t workspace_bytes, hsa_stream_t stream) {
  if (!budgets || !counts || K < 1) return HSA_ERR_INVALID_ARG;
  if (K > kMaxGroups) return HSA_ERR_UNSUPPORTED;
  const int st = hsa_check_budgets(T, budgets, counts, K, N);
  if (st != HSA_OK) return st;
  if (N == 0) return HSA_OK;
  if (!stat || !group_of) return HSA_ERR_INVALID_ARG;
  const SortLayout L = sort_layout(N);
  if (!workspace || workspace_bytes < L.total || (reinterpret_cast<uintptr_t>(workspace) & 255))
    return HSA_ERR_WORKSPACE;
  char *ws = static_cast<char *>(workspace);
  uint32_t *keys[2] = {reinterpret_cast<uint32_t *>(ws + L.keys0),
                       reinterpret_cast<uint32_t *>(ws + L.keys1)};
  int32_t *vals[2] = {reinterpret_cast<int32_t *>(ws + L.vals0),
                      reinterpret_cast<int32_t *>(ws + L.vals1)};
  uint32_t *hist = reinterpret_cast<uint32_t *>(ws + L.hist);
  cudaStream_t s = (cudaStream_t)stream;
  unsigned *err = device_error_word();
  if (!err) return HSA_ERR_CUDA;
  GroupStarts gs{};
  int r = 0;
  for (int k = K - 1; k >= 0; --k) {
    gs.start[k] = r;
    gs.count[k] = counts[k];
    r += counts[k];
  }
  if (N <= kRankMaxN) {
    count_launches(1);
    launch_pdl(rank_partition_kernel, dim3((N + kRankTokens - 1) / kRankTokens),
               dim3(kRankThreads), (size_t)((N + 3) / 4) * sizeof(uint4), s, stat, N, K, gs,
               group_of, err);
    return launch_status();
  }
  // 2048 bins while they hold few keys each, 4096 for larger layers (a lognormal
  // statistic of 200000 tokens would need a second pass with 2048: 35 us against 24).
  const bool fine = N > kCsFineN;
  if (N <= kCsMaxN && (fine ? cluster_select_ready<4>() : cluster_select_ready<2>())) {
    const int chunk = (((N + kCsCtas - 1) / kCsCtas) + 3) & ~3;   // keys per CTA, whole uint4
    count_launches(1);
    launch_pdl(fine ? cluster_select_kernel<4> : cluster_select_kernel<2>, dim3(kCsCtas),
               dim3(kCsThreads), (size_t)chunk * sizeof(uint32_t) + kCsFixedBytes, s, stat, N,
               chunk, K, gs, group_of, err);
    return launch_status();
  }
  // The scan's cluster is one CTA where a cluster of 8 cannot be resident.
  const unsigned scan_ctas = cluster_scan_ready() ? kScanCtas : 1;
  const int ew_blocks = (int)std::min<long long>(((long long)N + kSortThreads - 1) / kSortThreads,
                                                 (long long)sm_count() * 8);
  count_launches(1);
  launch_pdl(radix_key_kernel, dim3((ew_blocks + 3) / 4), dim3(kSortThreads), 0, s, stat, N,
             keys[0], err);
  for (int pass = 0; pass < 4; ++pass) {
    const int in = pass & 1, out = in ^ 1;
    count_launches(1);
    launch_pdl(radix_hist_kernel, dim3(L.tiles), dim3(kTileThreads), 0, s, keys[in], N, 8 * pass,
               hist, L.tiles);
    count_launches(1);
    launch_pdl_cluster(radix_scan_kernel, dim3(scan_ctas), dim3(1024), scan_ctas, s, hist,
                       256 * L.tiles);
    count_launches(1);
    launch_pdl(radix_scatter_kernel, dim3(L.tiles), dim3(kTileThreads), 0, s, keys[in],
               pass == 0 ? nullptr : vals[in], pass == 3 ? nullptr : keys[out], vals[out], N,
               8 * pass, hist, L.tiles);
  }
  count_launches(1);
  launch_pdl(group_assign_kernel, dim3(ew_blocks), dim3(kSortThreads), 0, s, vals[0], N, K, gs,
             group_of);
  return launch_status();
}

extern "C" int hsa_partition_active(const int32_t *group_of, int N, int T, const int *budgets,
                                    int K, int iter, int window_pct, int32_t *idx,
                                    int32_t *pos, hsa_stream_t stream) {
  if (!budgets || K < 1) return HSA_ERR_INVALID_ARG;
  if (K > kMaxGroups) return HSA_ERR_UNSUPPORTED;
  const int st = hsa_check_budgets(T, budgets, nullptr, K, N);
  if (st != HSA_OK) return st;
  const int m = hsa_window_margin(T, window_pct);
  if (m < 0 || iter < 0 || iter >= T) return HSA_ERR_INVALID_ARG;
  if (N == 0) return HSA_OK;
  if (!group_of || !idx) return HSA_ERR_INVALID_ARG;
  uint32_t mask = 0;
  for (int k = 0; k < K; ++k) {
    const bool full = iter < m || iter > T - m - 1;
    if (full || iter % (T / budgets[k]) == 0) mask |= 1u << k;
  }
  unsigned *err = device_error_word();
  if (!err) return HSA_ERR_CUDA;
  launch_compact<active_set_kernel<1>, active_set_kernel<4>>((cudaStream_t)stream, group_of, N, K, mask, idx, pos, err);
  return launch_status();
}

// ------------------------------------------------- allocation strategies
//
// Statistics whose ranking by hsa_partition gives the other token allocation
// strategies of App. B.  Uniform (U): stat[n] = top 24 bits of the 32-bit
// product (n+1) * 2654435769 (the golden ratio times 2^32), an integer exactly
// representable in fp32; each group then takes the tokens of one interval of
// the golden-ratio sequence, spaced by at most three distinct gaps.
// First-frame reservation (F): the first frame's tokens get FLT_MAX, so they
// rank into the baseline group.

__global__ void uniform_stat_kernel(float *__restrict__ stat, int N) {
  for (unsigned n = blockIdx.x * blockDim.x + threadIdx.x; n < (unsigned)N;
       n += gridDim.x * blockDim.x)
    stat[n] = (float)(((n + 1) * 2654435769u) >> 8);
}

__global__ void reserve_frame_kernel(float *__restrict__ stat, int frame_tokens) {
  for (unsigned n = blockIdx.x * blockDim.x + threadIdx.x; n < (unsigned)frame_tokens;
       n += gridDim.x * blockDim.x)
    stat[n] = 3.40282347e38f;
}

// ----------------------------------------------- partition without allocation
//
// Variant of hsa_partition for callers that cannot hand the library a
// workspace: a plugin running inside a host framework that owns all device
// memory and exposes no allocator to it, or a latency-critical loop where
// cudaMalloc/cudaFree (which may synchronise the device) are not acceptable.
// Its scratch is a fixed file-scope device array sized for
// HSA_PARTITION_STATIC_MAX_TOKENS tokens (the radix sort of layers above
// kCsMaxN tokens works in it; smaller layers need no scratch); every GPU that
// loads the library holds it until the process exits.

namespace {

constexpr size_t kStaticScratchBytes = sort_layout(HSA_PARTITION_STATIC_MAX_TOKENS).total;
static_assert(kStaticScratchBytes % 256 == 0, "scratch array size");
static_assert(HSA_PARTITION_STATIC_MAX_TOKENS > kCsMaxN,
              "the fixed scratch must serve the sizes that need one");

// The host cannot use this symbol as a device address; the set-up below asks
// the runtime for the device address once per device.
static __device__ __align__(256) unsigned char g_partition_scratch[kStaticScratchBytes];

std::atomic<void *> g_scratch_ptr[64];

// Device address of g_partition_scratch on the current device (nullptr on
// failure).  The first call on a device resolves it.
void *static_scratch() {
  int dev = -1;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return nullptr;
  void *p = g_scratch_ptr[dev].load(std::memory_order_acquire);
  if (!p) {
    if (cudaGetSymbolAddress(&p, g_partition_scratch) != cudaSuccess || !p) return nullptr;
    g_scratch_ptr[dev].store(p, std::memory_order_release);
  }
  return p;
}

}  // namespace

extern "C" int hsa_partition_static(const float *stat, int N, int T, const int *budgets,
                                    const int *counts, int K, int32_t *group_of,
                                    hsa_stream_t stream) {
  if (N > HSA_PARTITION_STATIC_MAX_TOKENS) return HSA_ERR_UNSUPPORTED;
  if (N >= 0 && hsa_partition_workspace_bytes(N) > kStaticScratchBytes) return HSA_ERR_UNSUPPORTED;
  void *scratch = static_scratch();
  if (!scratch) return HSA_ERR_CUDA;
  return hsa_partition(stat, N, T, budgets, counts, K, group_of, scratch, kStaticScratchBytes,
                       stream);
}

extern "C" int hsa_uniform_stat(float *stat, int N, hsa_stream_t stream) {
  if (N < 0) return HSA_ERR_INVALID_ARG;
  if (N == 0) return HSA_OK;
  if (!stat) return HSA_ERR_INVALID_ARG;
  const int blocks = (int)std::min<long long>(((long long)N + 255) / 256, (long long)sm_count() * 8);
  count_launches(1);
  uniform_stat_kernel<<<blocks, 256, 0, (cudaStream_t)stream>>>(stat, N);
  return launch_status();
}

extern "C" int hsa_reserve_first_frame(float *stat, int N, int frame_tokens,
                                       hsa_stream_t stream) {
  if (N < 0 || frame_tokens < 0 || frame_tokens > N) return HSA_ERR_INVALID_ARG;
  if (frame_tokens == 0) return HSA_OK;
  if (!stat) return HSA_ERR_INVALID_ARG;
  const int blocks = (int)std::min<long long>(((long long)frame_tokens + 255) / 256,
                                               (long long)sm_count() * 8);
  count_launches(1);
  reserve_frame_kernel<<<blocks, 256, 0, (cudaStream_t)stream>>>(stat, frame_tokens);
  return launch_status();
}

extern "C" int hsa_reorder_tokens(const int32_t *group_of, int N, int n_baseline,
                                  int32_t *order, int32_t *where, int32_t *group_new,
                                  hsa_stream_t stream) {
  if (N < 0 || n_baseline < 0 || n_baseline > N) return HSA_ERR_INVALID_ARG;
  if (N == 0) return HSA_OK;
  if (!group_of || !order) return HSA_ERR_INVALID_ARG;
  unsigned *err = device_error_word();
  if (!err) return HSA_ERR_CUDA;
  launch_compact<reorder_kernel<1>, reorder_kernel<4>>((cudaStream_t)stream, group_of, N, N - n_baseline, order, where,
                                 group_new, err);
  return launch_status();
}
