// fp32 active attention (Sec. 2.3, step 3) on the CUDA cores.
#include <cooperative_groups.h>

#include <atomic>
#include <cfloat>

#include "hsa_internal.cuh"
#include "hsa_ptx.cuh"
#include "hsa_test.h"

namespace hsa {
namespace {

// FMA-bound (fp32 has no tensor-core path of full precision): the work is laid
// out so that the FMA pipe, not shared memory, sets the pace.
//   warp     4*RT query rows x 32 keys of one head.  Lane (rg, cl) = (lane / 8,
//            lane % 8) owns rows rg + 4i (i < RT), keys cl + 8j (j < 4) of the
//            scores and dimensions 4cl + 32h of the output: per 4 dimensions
//            RT + 4 16-byte shared loads feed 16*RT FMAs, and per key RT/4 + D/32
//            loads feed RT*D/8 FMAs, all in packed pairs (fma.rn.f32x2), half
//            the issue slots of scalar FMAs.  Rows of K and P are padded by 16
//            bytes, which keeps the 8 lanes of a quarter-warp on distinct banks
//            (P rows 64 bytes longer, or not padded: 8-25 % slower; P stored as
//            the (p, p) pairs the FMAs take: 12 % slower, its wider stores and
//            loads cost more than the register moves).
//   CTA      WQ x WK warps: WQ row blocks share each key tile, WK warps take
//            different tiles of the same rows.  K and V arrive by cp.async,
//            double-buffered.
//   cluster  CTAs of a cluster split the keys of the same rows; the partial
//            (O, m, l) of all its warps are merged through distributed shared
//            memory, so small layers fill the GPU in one launch, without a
//            workspace.
// The softmax reference of a row moves only when a score passes it by more
// than 2^kLag (exact whatever the reference: the final division removes it), so
// most tiles need no reduction across lanes and no rescale of O.  The p that O is
// formed with are at most 1 all the same (times 2^-kLag, exact, given back by the
// division), so that large values of V overflow no sooner than with the row's
// maximum as the reference: 0.6 % at D = 64, 0.2 % at D = 128, the same bits.  (The
// row's sum scaled too: 1.0 %; the reference set 2^kLag above the maximum costs no
// time, but the exponents' larger arguments round more coarsely, error + 3 to 18 %; a
// second pass over the keys after an O that is not finite spills, 2 to 9 %.)
// Measured on GB300 (32 heads x 64, 3072 queries, 6144 keys): 3.05 ms, 51
// TFLOP/s (the FMA pipe allows 78), against 10.96 ms for one query row per 8
// threads with scalar shared loads and a shuffle reduction per key; 256 queries
// x 4 heads x 1024 keys: 15.4 us in a graph (64 CTAs without a split of the keys: 146
// us under ncu).
constexpr float kLag = 8.f;                        // log2 units
constexpr float kLagFactor = 256.f;                // 2^kLag

template <int D_, int RT_, int WQ_, int WK_>
struct F32Cfg {
  static constexpr int D = D_, RT = RT_, WQ = WQ_, WK = WK_;
  static constexpr int kThreads = 32 * WQ * WK;
  static constexpr int kWarpRows = 4 * RT;
  static constexpr int kRows = kWarpRows * WQ;              // query rows per CTA
  static constexpr int kKeys = 32 * WK;                     // keys per stage
  static constexpr int kQStride = D + 4, kKStride = D + 4;  // floats
  static constexpr int kPStride = 4 * RT + 4;               // floats per key of P
  static constexpr int kStage = kKeys * (kKStride + D);     // floats: K, then V
  static constexpr int kQFloats = kRows * kQStride;
  static constexpr int kPFloats = 32 * kPStride;            // per warp
  // After the key loop the same memory holds the partial results: O
  // [WK][kRows][D], then (m, l) [WK][kRows], then the merge weights and 2^kLag / l.
  static constexpr int kPartO = WK * kRows * D;
  static constexpr int kPartML = 2 * WK * kRows;
  static constexpr int kMerge = 8 * WK * kRows + kRows;
  static constexpr int kFloats = kQFloats + 2 * kStage + WQ * WK * kPFloats;
  static constexpr int kSmem = 4 * kFloats;
  static_assert(kPartO + kPartML + kMerge <= kFloats, "partials reuse the loop's memory");
  static_assert(kSmem <= 227 * 1024, "shared memory");
};

__device__ __forceinline__ void cp_async16(void *dst, const void *src, bool valid) {
  const int n = valid ? 16 : 0;       // 0: the 16 bytes are zero-filled, src is not read
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(smem_addr(dst)), "l"(src),
               "r"(n)
               : "memory");
}

// One block per SM as the stated minimum: without it the compiler holds the
// 256-thread instances (D = 128) to fewer registers, 8 % slower (16 heads x 128,
// 2000 queries, 3000 keys: 1350 against 1250 us).
template <class C>
__global__ void __launch_bounds__(C::kThreads, 1)
attn_f32_kernel(const float *__restrict__ q, const int32_t *__restrict__ q_idx,
                const float *__restrict__ kc, const float *__restrict__ vc, int rows1,
                const float *__restrict__ kb, const float *__restrict__ vb,
                float *__restrict__ out, int n_active, int N, int H, int q_rows, float scale_log2,
                int splits, unsigned *err) {
  pdl_wait();
  pdl_trigger();
  namespace cg = cooperative_groups;
  constexpr int D = C::D, RT = C::RT;
  constexpr int kDV = D / 32;                      // 16-byte output vectors per row and lane
  extern __shared__ float4 f32_smem[];
  float *smem = reinterpret_cast<float *>(f32_smem);
  float *sQ = smem;
  float *sKV = smem + C::kQFloats;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int wq = warp % C::WQ, wk = warp / C::WQ;
  const int rg = lane >> 3, cl = lane & 7;
  float *sP = sKV + 2 * C::kStage + warp * C::kPFloats;
  const int h = blockIdx.y;
  const int split = blockIdx.x % splits;           // rank in the cluster
  const int row0 = (int)(blockIdx.x / splits) * C::kRows;
  // stages [g0, g1) of kKeys keys
  const int n_stages = (N + C::kKeys - 1) / C::kKeys;
  const int g0 = (int)((long long)n_stages * split / splits);
  const int g1 = (int)((long long)n_stages * (split + 1) / splits);

  // Thread t copies 16-byte vector t % (D/4) of keys t / (D/4) + u*kStep.
  constexpr int kStep = C::kThreads / (D / 4);
  const int kk0 = threadIdx.x / (D / 4), c0 = threadIdx.x % (D / 4);
  const size_t token = (size_t)H * D;
  auto load_stage = [&](int g) {
    float *dk = sKV + (g & 1) * C::kStage + kk0 * C::kKStride + 4 * c0;
    float *dv = sKV + (g & 1) * C::kStage + C::kKeys * C::kKStride + kk0 * D + 4 * c0;
    const int base = g * C::kKeys;
    if (base + C::kKeys <= rows1) {                // whole stage in the first source
      const size_t off = (size_t)(base + kk0) * token + (size_t)h * D + 4 * c0;
      const float *pk = kc + off, *pv = vc + off;
#pragma unroll
      for (int u = 0; u < C::kKeys / kStep; ++u) {
        cp_async16(dk + u * kStep * C::kKStride, pk, true);
        cp_async16(dv + u * kStep * D, pv, true);
        pk += kStep * token;
        pv += kStep * token;
      }
      asm volatile("cp.async.commit_group;" ::: "memory");
      return;
    }
    for (int u = 0; u < C::kKeys / kStep; ++u) {
      const int key = base + kk0 + u * kStep;
      const bool ok = key < N;
      const bool first = key < rows1;
      const size_t off =
          ok ? (size_t)(first ? key : key - rows1) * token + (size_t)h * D + 4 * c0 : 0;
      const float *pk = ok && !first ? kb : (rows1 > 0 ? kc : kb);
      const float *pv = ok && !first ? vb : (rows1 > 0 ? vc : vb);
      cp_async16(dk + u * kStep * C::kKStride, pk + off, ok);
      cp_async16(dv + u * kStep * D, pv + off, ok);
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  if (g0 < g1) load_stage(g0);
  for (int e = threadIdx.x; e < C::kRows * (D / 4); e += C::kThreads) {
    const int r = e / (D / 4), c = e % (D / 4);
    const int j = row0 + r;
    float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
    if (j < n_active) {
      const int src = q_idx ? __ldg(q_idx + j) : j;
      if (src >= 0 && src < q_rows)
        v = __ldg(reinterpret_cast<const float4 *>(q + ((size_t)src * H + h) * D) + c);
      else if (c == 0)
        set_error(err, kErrIndex);
    }
    *reinterpret_cast<float4 *>(sQ + r * C::kQStride + 4 * c) = v;
  }

  uint64_t o2[RT][2 * kDV];
  // m: the row's reference in log2 units (any finite start will do: a score
  // of -inf, or 0 keys, then weighs 0 against it); l2: the sums of rows 2i, 2i+1
  float m[RT];
  uint64_t l2[RT / 2];
#pragma unroll
  for (int i = 0; i < RT; ++i) {
    m[i] = -FLT_MAX;
    l2[i / 2] = 0ull;
#pragma unroll
    for (int d = 0; d < 2 * kDV; ++d) o2[i][d] = 0ull;
  }
  constexpr float kPScale = 1.f / kLagFactor;
  const float *qrow = sQ + (wq * C::kWarpRows + rg) * C::kQStride;
  for (int g = g0; g < g1; ++g) {
    asm volatile("cp.async.wait_group 0;" ::: "memory");
    __syncthreads();              // stage g has landed, every warp is done with stage g-1
    if (g + 1 < g1) load_stage(g + 1);
    const int key0 = g * C::kKeys + 32 * wk;
    if (key0 >= N) continue;                       // this warp's tile has no key
    const float *sK = sKV + (g & 1) * C::kStage + (32 * wk + cl) * C::kKStride;
    const float *sV = sKV + (g & 1) * C::kStage + C::kKeys * C::kKStride + 32 * wk * D + 4 * cl;
    // scores: even dimensions in the low halves, odd in the high halves
    uint64_t s2[RT][4];
#pragma unroll
    for (int i = 0; i < RT; ++i)
#pragma unroll
      for (int j = 0; j < 4; ++j) s2[i][j] = 0ull;
#pragma unroll 16
    for (int d = 0; d < D; d += 4) {
      ulonglong2 kv[4];
#pragma unroll
      for (int j = 0; j < 4; ++j)
        kv[j] = *reinterpret_cast<const ulonglong2 *>(sK + 8 * j * C::kKStride + d);
#pragma unroll
      for (int i = 0; i < RT; ++i) {
        const ulonglong2 qv = *reinterpret_cast<const ulonglong2 *>(qrow + 4 * i * C::kQStride + d);
#pragma unroll
        for (int j = 0; j < 4; ++j) s2[i][j] = fma2(qv.x, kv[j].x, s2[i][j]);
#pragma unroll
        for (int j = 0; j < 4; ++j) s2[i][j] = fma2(qv.y, kv[j].y, s2[i][j]);
      }
    }
    float s[RT][4];
#pragma unroll
    for (int i = 0; i < RT; ++i)
#pragma unroll
      for (int j = 0; j < 4; ++j) s[i][j] = lo_f(s2[i][j]) + hi_f(s2[i][j]);
    if (key0 + 32 > N) {                           // keys past N count as -inf
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        if (key0 + cl + 8 * j < N) continue;
#pragma unroll
        for (int i = 0; i < RT; ++i) s[i][j] = -INFINITY;
      }
    }
    bool move = false;
#pragma unroll
    for (int i = 0; i < RT; ++i) {
      const float mx = fmaxf(max3f(s[i][0], s[i][1], s[i][2]), s[i][3]);
      move |= fmaf(mx, scale_log2, -m[i]) > kLag;
    }
    if (__any_sync(0xffffffffu, move)) {
#pragma unroll
      for (int i = 0; i < RT; ++i) {
        float mx = fmaxf(max3f(s[i][0], s[i][1], s[i][2]), s[i][3]) * scale_log2;
#pragma unroll
        for (int o = 1; o < 8; o <<= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
        const float m_new = fmaxf(m[i], mx);
        const float corr = m_new > m[i] ? exp2f(m[i] - m_new) : 1.f;
        m[i] = m_new;
        const uint64_t c2 = pack2(__float_as_uint(corr), __float_as_uint(corr));
        l2[i / 2] = mul2(l2[i / 2], (i & 1) ? pack2(0x3f800000u, __float_as_uint(corr))
                                            : pack2(__float_as_uint(corr), 0x3f800000u));
#pragma unroll
        for (int d = 0; d < 2 * kDV; ++d) o2[i][d] = mul2(o2[i][d], c2);
      }
    }
    __syncwarp();                                  // the previous tile's P has been read
#pragma unroll
    for (int i = 0; i < RT; i += 4) {
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        float p[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) p[e] = fast_exp2(fmaf(s[i + e][j], scale_log2, -m[i + e]));
        l2[i / 2] = add2(l2[i / 2], pack2(__float_as_uint(p[0]), __float_as_uint(p[1])));
        l2[i / 2 + 1] = add2(l2[i / 2 + 1], pack2(__float_as_uint(p[2]), __float_as_uint(p[3])));
        *reinterpret_cast<float4 *>(sP + (cl + 8 * j) * C::kPStride + (i + rg) * 4) =
            make_float4(p[0] * kPScale, p[1] * kPScale, p[2] * kPScale, p[3] * kPScale);
      }
    }
    __syncwarp();
#pragma unroll 16
    for (int k = 0; k < 32; ++k) {
      ulonglong2 vv[kDV];
#pragma unroll
      for (int d = 0; d < kDV; ++d)
        vv[d] = *reinterpret_cast<const ulonglong2 *>(sV + k * D + 32 * d);
#pragma unroll
      for (int i = 0; i < RT; i += 4) {
        const uint4 pp = *reinterpret_cast<const uint4 *>(sP + k * C::kPStride + (i + rg) * 4);
        const uint64_t pd[4] = {pack2(pp.x, pp.x), pack2(pp.y, pp.y), pack2(pp.z, pp.z),
                                pack2(pp.w, pp.w)};
#pragma unroll
        for (int e = 0; e < 4; ++e) {
#pragma unroll
          for (int d = 0; d < kDV; ++d) {
            o2[i + e][2 * d] = fma2(pd[e], vv[d].x, o2[i + e][2 * d]);
            o2[i + e][2 * d + 1] = fma2(pd[e], vv[d].y, o2[i + e][2 * d + 1]);
          }
        }
      }
    }
  }
  // row sums over the 8 lanes of a row
  float l[RT];
#pragma unroll
  for (int i = 0; i < RT; ++i) {
    l[i] = (i & 1) ? hi_f(l2[i / 2]) : lo_f(l2[i / 2]);
#pragma unroll
    for (int o = 1; o < 8; o <<= 1) l[i] += __shfl_xor_sync(0xffffffffu, l[i], o);
  }

  if (C::WK == 1 && splits == 1) {
#pragma unroll
    for (int i = 0; i < RT; ++i) {
      const int j = row0 + wq * C::kWarpRows + rg + 4 * i;
      if (j >= n_active) continue;
      const float inv = kLagFactor / l[i];
      float *dst = out + ((size_t)j * H + h) * D + 4 * cl;
#pragma unroll
      for (int d = 0; d < kDV; ++d)
        *reinterpret_cast<float4 *>(dst + 32 * d) =
            make_float4(lo_f(o2[i][2 * d]) * inv, hi_f(o2[i][2 * d]) * inv,
                        lo_f(o2[i][2 * d + 1]) * inv, hi_f(o2[i][2 * d + 1]) * inv);
    }
    return;
  }
  // Merge: every warp leaves (O, m, l) in its CTA's shared memory; CTA `split`
  // then merges rows [split, split+1) * kRows/splits over the whole cluster.
  __syncthreads();                                 // the loop's memory is free
  float *pO = smem, *pML = smem + C::kPartO, *pW = pML + C::kPartML;
  float *pInv = pW + 8 * C::WK * C::kRows;
#pragma unroll
  for (int i = 0; i < RT; ++i) {
    const int r = wk * C::kRows + wq * C::kWarpRows + rg + 4 * i;
#pragma unroll
    for (int d = 0; d < kDV; ++d)
      *reinterpret_cast<ulonglong2 *>(pO + r * D + 4 * cl + 32 * d) =
          make_ulonglong2(o2[i][2 * d], o2[i][2 * d + 1]);
    if (cl == 0) *reinterpret_cast<float2 *>(pML + 2 * r) = make_float2(m[i], l[i]);
  }
  cg::cluster_group cluster = cg::this_cluster();
  cluster.sync();
  const int rows = C::kRows / splits, r0 = split * rows;
  const int parts = splits * C::WK;                // partial p: warp slot p % WK of CTA p / WK
  if (threadIdx.x < rows) {
    const int r = r0 + threadIdx.x;
    float M = -FLT_MAX, L = 0.f;
    for (int p = 0; p < parts; ++p) {
      const float2 *ml = reinterpret_cast<const float2 *>(cluster.map_shared_rank(pML, p / C::WK));
      M = fmaxf(M, ml[(p % C::WK) * C::kRows + r].x);
    }
    for (int p = 0; p < parts; ++p) {
      const float2 *ml = reinterpret_cast<const float2 *>(cluster.map_shared_rank(pML, p / C::WK));
      const float2 v = ml[(p % C::WK) * C::kRows + r];
      const float w = exp2f(v.x - M);              // a part without keys: 0, or l = 0
      pW[p * C::kRows + threadIdx.x] = w;
      L = fmaf(w, v.y, L);
    }
    pInv[threadIdx.x] = kLagFactor / L;
  }
  __syncthreads();
  for (int e = threadIdx.x; e < rows * (D / 4); e += C::kThreads) {
    const int r = e / (D / 4), c = e % (D / 4);
    const int j = row0 + r0 + r;
    if (j >= n_active) break;                      // later elements are later rows
    float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
    for (int b = 0; b < splits; ++b) {
      const float4 *src = reinterpret_cast<const float4 *>(cluster.map_shared_rank(pO, b));
#pragma unroll
      for (int k = 0; k < C::WK; ++k) {
        const float4 v = src[(k * C::kRows + r0 + r) * (D / 4) + c];
        const float w = pW[(b * C::WK + k) * C::kRows + r];
        acc.x = fmaf(w, v.x, acc.x);
        acc.y = fmaf(w, v.y, acc.y);
        acc.z = fmaf(w, v.z, acc.z);
        acc.w = fmaf(w, v.w, acc.w);
      }
    }
    const float inv = pInv[r];
    *reinterpret_cast<float4 *>(out + ((size_t)j * H + h) * D + 4 * c) =
        make_float4(acc.x * inv, acc.y * inv, acc.z * inv, acc.w * inv);
  }
  cluster.sync();                 // no CTA exits while another reads its partials
}

// Launch plan of the fp32 path: the wide CTA (128 rows share each key tile) or
// the deep one (32 rows, the CTA's warps on different keys), and how many CTAs
// of a cluster split the keys.  Both run 4 or 8 warps on the same tile code, so
// the time of a plan is the CTAs per SM times the stages each runs (plus about
// half a stage for the query load and the merge); the smallest wins.  A cluster
// has no more CTAs than can be resident (`wide_most`, `deep_most`; a slice of the
// GPU may hold fewer than 8 together): a larger one would not launch.
struct F32Plan {
  bool deep;
  int splits;
};

template <class Wide, class Deep>
F32Plan f32_plan(int n_active, int N, int H, int sms, int wide_most, int deep_most) {
  F32Plan best{false, 1};
  double best_cost = 0.0;
  for (int deep = 0; deep < 2; ++deep) {
    const int rows = deep ? Deep::kRows : Wide::kRows, keys = deep ? Deep::kKeys : Wide::kKeys;
    const int threads = deep ? Deep::kThreads : Wide::kThreads;
    const int most = deep ? deep_most : wide_most;
    const long long stages = ((long long)N + keys - 1) / keys;
    const long long units = ((long long)n_active + rows - 1) / rows * H;
    for (int splits = 1; splits <= 8; splits *= 2) {
      if (splits > 1 && (stages < splits || splits > most)) break;
      const long long per_sm = (units * splits + sms - 1) / sms;
      const double cost = (double)per_sm * threads *
                          ((double)((stages + splits - 1) / splits) + (splits > 1 ? 0.6 : 0.5));
      if ((!deep && splits == 1) || cost < best_cost) {
        best_cost = cost;
        best = F32Plan{deep != 0, splits};
      }
    }
  }
  return best;
}

// D = 64: 8 rows per lane (64 accumulators of O); D = 128: 4, for the same count.
template <int D>
using F32Wide = F32Cfg<D, D == 64 ? 8 : 4, D == 64 ? 4 : 8, 1>;
template <int D>
using F32Deep = F32Cfg<D, D == 64 ? 8 : 4, D == 64 ? 1 : 2, D == 64 ? 4 : 2>;

// Opts kernel C in to its shared memory on the current device; returns the CTAs of
// the largest cluster (8, 4, 2 or 1) of which one can be resident, 0 on failure.
// Resolved once per device.
template <class C>
int f32_cluster_most() {
  static std::atomic<int> most[64];
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return 0;
  int n = most[dev].load();
  if (n) return n;
  if (cudaFuncSetAttribute(attn_f32_kernel<C>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                           C::kSmem) != cudaSuccess)
    return 0;
  for (n = 8; n > 1; n /= 2) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)n);
    cfg.blockDim = dim3(C::kThreads);
    cfg.dynamicSmemBytes = C::kSmem;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = (unsigned)n;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    int clusters = 0;
    if (cudaOccupancyMaxActiveClusters(&clusters, attn_f32_kernel<C>, &cfg) == cudaSuccess &&
        clusters >= 1)
      break;
  }
  cudaGetLastError();                          // a refused query leaves no sticky error
  most[dev].store(n);
  return n;
}

template <class C>
int launch_f32_cfg(int splits, const float *q, const int32_t *q_idx, int n_active,
                   const float *k_cache, const float *v_cache, int rows1, const float *k_base,
                   const float *v_base, int N, int H, float scale, float *out,
                   cudaStream_t stream, unsigned *err) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)((n_active + (long long)C::kRows - 1) / C::kRows * splits), H);
  cfg.blockDim = dim3(C::kThreads);
  cfg.dynamicSmemBytes = C::kSmem;
  cfg.stream = stream;
  cudaLaunchAttribute at[2];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  at[1].id = cudaLaunchAttributeClusterDimension;
  at[1].val.clusterDim.x = (unsigned)splits;
  at[1].val.clusterDim.y = 1;
  at[1].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = 2;
  count_launches(1);
  cudaLaunchKernelEx(&cfg, attn_f32_kernel<C>, q, q_idx, k_cache, v_cache, rows1, k_base, v_base,
                     out, n_active, N, H, q_idx ? N : n_active,
                     (float)((double)scale * 1.4426950408889634), splits, err);
  return launch_status();
}

template <int D>
int launch_f32(const void *q, const int32_t *q_idx, int n_active, const void *k_cache,
               const void *v_cache, int rows1, const void *k_base, const void *v_base, int rows2,
               int H, float scale, void *out, cudaStream_t stream, unsigned *err) {
  using Wide = F32Wide<D>;
  using Deep = F32Deep<D>;
  const int N = rows1 + rows2;
  const int wide_most = f32_cluster_most<Wide>(), deep_most = f32_cluster_most<Deep>();
  if (!wide_most || !deep_most) return HSA_ERR_CUDA;
  const F32Plan plan = f32_plan<Wide, Deep>(n_active, N, H, sm_count(), wide_most, deep_most);
  auto f = [](const void *p) { return static_cast<const float *>(p); };
  return plan.deep
             ? launch_f32_cfg<Deep>(plan.splits, f(q), q_idx, n_active, f(k_cache), f(v_cache),
                                    rows1, f(k_base), f(v_base), N, H, scale,
                                    static_cast<float *>(out), stream, err)
             : launch_f32_cfg<Wide>(plan.splits, f(q), q_idx, n_active, f(k_cache), f(v_cache),
                                    rows1, f(k_base), f(v_base), N, H, scale,
                                    static_cast<float *>(out), stream, err);
}

}  // namespace

int launch_attention_f32(const void *q, const int32_t *q_idx, int n_active, const void *k_cache,
                         const void *v_cache, int rows1, const void *k_base, const void *v_base,
                         int rows2, int H, int D, float scale, void *out, cudaStream_t stream,
                         unsigned *err) {
  return D == 128 ? launch_f32<128>(q, q_idx, n_active, k_cache, v_cache, rows1, k_base, v_base,
                                    rows2, H, scale, out, stream, err)
                  : launch_f32<64>(q, q_idx, n_active, k_cache, v_cache, rows1, k_base, v_base,
                                   rows2, H, scale, out, stream, err);
}

}  // namespace hsa

extern "C" int hsa_test_f32_cluster(int n_active, int N, int H, int D, int sms, int wide_most,
                                    int deep_most) {
  using namespace hsa;
  if (n_active < 1 || N < 1 || H < 1 || sms < 1 || wide_most < 1 || deep_most < 1 ||
      (D != 64 && D != 128))
    return HSA_ERR_INVALID_ARG;
  const F32Plan p =
      D == 128 ? f32_plan<F32Wide<128>, F32Deep<128>>(n_active, N, H, sms, wide_most, deep_most)
               : f32_plan<F32Wide<64>, F32Deep<64>>(n_active, N, H, sms, wide_most, deep_most);
  return p.deep ? 256 + p.splits : p.splits;
}
