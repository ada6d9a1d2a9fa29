// Memory-bound steps of the HSA iteration: gather of the active rows
// (Sec. 2.3, step 1), KV-cache synchronisation scatter (Sec. 2.3, step 2) and
// the cached Euler update (Sec. 2.4, Eq. 6).
//
// All three move whole token rows.  A row is split into 16-byte vectors and a
// group of L lanes (L a power of two <= 32) of one warp cooperates on a row, so
// a warp covers 32/L rows at once and every access is a coalesced 128-bit load
// or store.  Each lane keeps several vectors in flight before storing.
// The row index is read once per row by its lane group; indices are checked
// against the row count and a bad one skips its row and sets the error word.
#include <cuda_bf16.h>

#include <atomic>
#include <cmath>

#include "hsa_internal.cuh"

namespace hsa {
namespace {

constexpr int kThreads = 256;
// The rotation in place is best at 6, the rotating scatter, which also holds the
// table's vectors and two row pointers, at 4.
constexpr int kRopeUnroll = 6;
constexpr int kRopeScatterUnroll = 4;
// Blocks per SM of both at most: 54 to 64 registers leave 4 resident, and many short
// blocks balance better than two waves of 8: half of 75600 rows of 40 x 128, scatter
// 243 -> 232 us, in place 121.5 -> 117.7; smaller layers equal.
constexpr int kRopeBlocks = 32;
constexpr int kEulerUnroll = 2;  // float4 positions per thread per pass (long rows, large N)

__device__ __forceinline__ uint4 ld_stream(const uint4 *p) {
  uint4 v;
  asm volatile("ld.global.nc.L1::no_allocate.v4.u32 {%0,%1,%2,%3}, [%4];"
               : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(p));
  return v;
}

// One row of `vecs` 16-byte vectors by the lanes of a group, kUnroll in flight each.
template <int kUnroll>
__device__ __forceinline__ void copy_row(const uint4 *s, uint4 *d, int vecs, int sl, int L) {
  for (int v0 = sl; v0 < vecs; v0 += kUnroll * L) {
    uint4 buf[kUnroll];
#pragma unroll
    for (int u = 0; u < kUnroll; ++u) {
      const int v = v0 + u * L;
      if (v < vecs) buf[u] = ld_stream(s + v);
    }
#pragma unroll
    for (int u = 0; u < kUnroll; ++u) {
      const int v = v0 + u * L;
      if (v < vecs) d[v] = buf[u];
    }
  }
}

// The gather, the Euler step and the statistic of short rows wait for the launch
// before them (pdl_wait) and let the next one start when they end, not before: blocks
// of the next launch that take the slots they leave free lie unevenly on the SMs.  In a
// row of launches, early trigger / none: gather of half of 6144 x 4 KB 4.74 / 3.62 us,
// Euler 32760 x 128 7.39 / 6.59 and 1048576 x 16 40.9 / 40.6, statistic 6144 x 128
// 3.72 / 3.21, 24000 x 128 8.17 / 7.15 (262144 x 128, 27 passes: 105.3 / 107.0).  The
// scatter triggers early: alone 7.51 / 7.30 us at 6144 rows, but the attention after it
// has a prologue to overlap.

// Row loop shared by gather and scatter: rows are handed out to lane groups
// in a grid-stride loop; `index(j)` reads row j's token, with kAhead one row
// before its use; `map(j, r, s, d)` sets the row's source and destination, or
// returns false to skip it.  CopyPlan says which form a row length takes.
template <int kUnroll, bool kAhead, class Index, class RowMap>
__device__ __forceinline__ void copy_rows(long long n_rows, int vecs, int lpr_log2, Index index,
                                          RowMap map) {
  const int L = 1 << lpr_log2;
  const uint4 *s;
  uint4 *d;
  if constexpr (kAhead) {
    const int sl = threadIdx.x & (L - 1);            // lane within the row group
    const long long step = ((long long)gridDim.x * blockDim.x) >> lpr_log2;
    long long j = (blockIdx.x * (long long)blockDim.x + threadIdx.x) >> lpr_log2;
    int r = j < n_rows ? index(j) : 0;
    for (; j < n_rows; j += step) {
      const int r_next = j + step < n_rows ? index(j + step) : 0;
      if (map(j, r, s, d)) copy_row<kUnroll>(s, d, vecs, sl, L);
      r = r_next;
    }
  } else {
    const int lane = threadIdx.x & 31;
    const int sub = lane >> lpr_log2;                // row slot within the warp
    const int sl = lane & (L - 1);
    const int rows_per_warp = 32 >> lpr_log2;
    const long long warp = (blockIdx.x * (long long)blockDim.x + threadIdx.x) >> 5;
    const long long nwarps = ((long long)gridDim.x * blockDim.x) >> 5;
    for (long long j = warp * rows_per_warp + sub; j < n_rows; j += nwarps * rows_per_warp)
      if (map(j, index(j), s, d)) copy_row<kUnroll>(s, d, vecs, sl, L);
  }
}

template <int kUnroll, bool kAhead>
__global__ void __launch_bounds__(kThreads)
gather_rows_kernel(const uint4 *__restrict__ src, uint4 *__restrict__ dst,
                   const int32_t *__restrict__ idx, int n_active, int N, int vecs, int lpr_log2,
                   unsigned *err) {
  pdl_wait();
  copy_rows<kUnroll, kAhead>(
      n_active, vecs, lpr_log2, [&](long long j) { return __ldg(idx + j); },
      [&](long long j, int r, const uint4 *&s, uint4 *&d) {
        if (r < 0 || r >= N) {
          set_error(err, kErrIndex);
          return false;
        }
        s = src + (long long)r * vecs;
        d = dst + j * vecs;
        return true;
      });
}

// Rows 0..n_active-1 are K rows, n_active..2*n_active-1 the V rows, so a warp
// moves K and V rows of different tokens with the same code.
template <int kUnroll>
__global__ void __launch_bounds__(kThreads)
kv_scatter_kernel(uint4 *__restrict__ kc, uint4 *__restrict__ vc, const uint4 *__restrict__ kf,
                  const uint4 *__restrict__ vf, const int32_t *__restrict__ idx, int n_active,
                  int N, int vecs, int lpr_log2, unsigned *err) {
  pdl_wait();
  pdl_trigger();   // the attention's prologue runs beside the last rows
  copy_rows<kUnroll, true>(
      2LL * n_active, vecs, lpr_log2,
      [&](long long jj) { return __ldg(idx + (jj >= n_active ? jj - n_active : jj)); },
      [&](long long jj, int r, const uint4 *&s, uint4 *&d) {
        const bool is_v = jj >= n_active;
        const long long j = is_v ? jj - n_active : jj;
        if (r < 0 || r >= N) {
          if (!is_v) set_error(err, kErrIndex);
          return false;
        }
        s = (is_v ? vf : kf) + j * vecs;
        d = (is_v ? vc : kc) + (long long)r * vecs;
        return true;
      });
}

// pos[row], with a bad entry (only -1 means "no fresh row") reported and read as
// -1.
__device__ __forceinline__ int load_pos(const int32_t *__restrict__ pos, long long row,
                                        int n_fresh_rows, unsigned *err) {
  const int p = __ldg(pos + row);
  if (p >= n_fresh_rows || p < -1) {
    set_error(err, kErrIndex);
    return -1;
  }
  return p;
}

__device__ __forceinline__ float4 euler_step(const float4 &v, float dsigma, const float4 &x) {
  return make_float4(__fmaf_rn(v.x, dsigma, x.x), __fmaf_rn(v.y, dsigma, x.y),
                     __fmaf_rn(v.z, dsigma, x.z), __fmaf_rn(v.w, dsigma, x.w));
}

// x[n] = fma(vhat[n], dsigma, x[n]) with vhat[n] refreshed from
// v_fresh[pos[n]] when pos[n] >= 0.  Element-wise over the N*C/4 float4
// vectors: each thread takes kU vectors a grid-stride apart.  The pos entries
// of a pass are loaded one pass ahead (software pipelining), so a pass issues
// its x loads and its velocity loads (v_fresh rows by pos, or the cache)
// at once: 2*kU independent loads in flight per thread whatever C is.  The
// grid is the number of blocks resident at once (a single wave).  Measured on
// GB300 with an L2-flushed size sweep: kU = 2 with the pos loads one pass
// ahead reaches 0.85-1.0 of the HBM copy rate, kU = 4 (more registers, fewer
// resident threads) 0.68-0.85.  Rows below 16 vectors (C < 64) take one vector
// per thread: half the tokens fresh, 3 layers in turn, 1048576 x 16 43.7 -> 42.2
// us, 4000000 x 16 152.6 -> 147.7, 200000 x 48 26.3 -> 24.4; from 16 vectors on two
// are the better (1048576 x 64 144.6 against 148.8, 262144 x 256 140.3 against
// 146.8).
// vec_shift = log2(C/4) when C/4 is a power of two, else -1 (division).
// Small N uses one vector per thread (kU = 1) so that every SM has work.
template <int kU>
__device__ __forceinline__ void load_pos_pass(const int32_t *__restrict__ pos, long long base,
                                              long long stride, long long total, int vecs,
                                              int vec_shift, int n_fresh_rows, unsigned *err,
                                              int (&p)[kU]) {
#pragma unroll
  for (int u = 0; u < kU; ++u) {
    const long long e = base + u * stride;
    p[u] = -1;
    if (pos && e < total)
      p[u] = load_pos(pos, vec_shift >= 0 ? (e >> vec_shift) : e / vecs, n_fresh_rows, err);
  }
}

template <int kU>
__global__ void __launch_bounds__(kThreads)
cached_euler_kernel(float4 *__restrict__ x, float4 *__restrict__ vhat,
                    const float4 *__restrict__ v_fresh, const int32_t *__restrict__ pos,
                    long long total, int vecs, int vec_shift, float dsigma, int n_fresh_rows,
                    unsigned *err) {
  pdl_wait();
  const long long stride = (long long)gridDim.x * blockDim.x;
  long long base = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  int pn[kU];
  load_pos_pass<kU>(pos, base, stride, total, vecs, vec_shift, n_fresh_rows, err, pn);
  for (; base < total; base += stride * kU) {
    int p[kU];
#pragma unroll
    for (int u = 0; u < kU; ++u) p[u] = pn[u];
    load_pos_pass<kU>(pos, base + stride * kU, stride, total, vecs, vec_shift, n_fresh_rows,
                      err, pn);
    float4 vb[kU], xb[kU];
#pragma unroll
    for (int u = 0; u < kU; ++u) {
      const long long e = base + u * stride;
      if (e < total) {
        const long long row = vec_shift >= 0 ? (e >> vec_shift) : e / vecs;
        const long long c = e - row * vecs;
        xb[u] = x[e];
        vb[u] = p[u] >= 0 ? __ldg(v_fresh + (long long)p[u] * vecs + c) : vhat[e];
      }
    }
#pragma unroll
    for (int u = 0; u < kU; ++u) {
      const long long e = base + u * stride;
      if (e < total) {
        if (p[u] >= 0) vhat[e] = vb[u];
        x[e] = euler_step(vb[u], dsigma, xb[u]);
      }
    }
  }
}

// The cached Euler step fused with the velocity statistic (below) for rows of
// up to 32 vectors (C <= 128): L = 2^lpr_log2 >= C/4 neighbouring lanes take a
// token (those past its vectors idle), so its two L1 norms are reduced with
// log2(L) shuffles and its first lane updates stat.  Every lane of a warp runs
// the same passes (the shuffles span the warp).  HBM-bound, one vector per
// thread keeps the registers at 32 and the SM full (2048 threads), which holds
// more loads in flight than two vectors on half the threads.  Every token fresh,
// 3 layers in turn: 1048576 x 16 68.6 -> 56.4 us (0.92 of the measured HBM rate),
// 4000000 x 16 240 -> 208 (0.95), 1048576 x 64 244 -> 214 (0.95), 262144 x 128 125
// -> 108 (0.93); 1048576 x 48, which took two tokens per lane group and pass
// before, 270 -> 152 (1.00).
__global__ void __launch_bounds__(kThreads, 8)
euler_l1rel_elem_kernel(float4 *__restrict__ x, float4 *__restrict__ vhat,
                        const float4 *__restrict__ v_fresh, const int32_t *__restrict__ pos,
                        int N, int vecs, int lpr_log2, float dsigma, int n_fresh_rows,
                        float *__restrict__ stat, float weight, unsigned *err) {
  pdl_wait();
  const int lane = threadIdx.x & 31;
  const int L = 1 << lpr_log2;
  const int c = lane & (L - 1);
  const long long step = ((long long)gridDim.x * blockDim.x) >> lpr_log2;   // tokens per pass
  long long row = (blockIdx.x * (long long)blockDim.x + threadIdx.x) >> lpr_log2;
  int p = row < N ? load_pos(pos, row, n_fresh_rows, err) : -1;
  for (; row - (lane >> lpr_log2) < N; row += step) {
    const int p_next = row + step < N ? load_pos(pos, row + step, n_fresh_rows, err) : -1;
    const bool in = row < N && c < vecs;
    const bool first = p >= 0 && c == 0;               // p >= 0 only below N
    const long long e = row * vecs + c;
    float num = 0.f, den = 0.f, st = 0.f;
    if (in) {
      const float4 xv = x[e];
      const float4 vo = vhat[e];
      const float4 vn = p >= 0 ? __ldg(v_fresh + (long long)p * vecs + c) : vo;
      if (first) st = stat[row];                       // with the data
      if (p >= 0) {
        num = fabsf(vn.x - vo.x) + fabsf(vn.y - vo.y) + fabsf(vn.z - vo.z) + fabsf(vn.w - vo.w);
        den = fabsf(vn.x) + fabsf(vn.y) + fabsf(vn.z) + fabsf(vn.w);
        vhat[e] = vn;
      }
      x[e] = euler_step(vn, dsigma, xv);
    }
    for (int o = 1; o < L; o <<= 1) {
      num += __shfl_xor_sync(0xffffffffu, num, o);
      den += __shfl_xor_sync(0xffffffffu, den, o);
    }
    if (first) {
      const float r = den > 0.f ? num / den : (num > 0.f ? 3.402823466e38f : 0.f);
      stat[row] = fmaf(weight, r, st);
    }
    p = p_next;
  }
}

// Cached Euler step fused with the velocity statistic of the dynamic token
// selection (App. B, Eq. 7): for a refreshed token (pos[n] >= 0) the old cache
// row is v_{i-1}[n] and the fresh row v_i[n]; the kernel adds
// weight * ||v_i - v_{i-1}||_1 / ||v_i||_1 to stat[n] (a zero denominator
// counts 0 with a zero numerator, FLT_MAX otherwise), then refreshes the cache
// and advances x exactly as cached_euler_kernel does.  This layout (for more
// than 32 vectors per row): a group of L lanes owns a token; the two L1 norms
// are reduced across the group with shuffles.
constexpr int kL1relRows = 2;   // tokens per lane group per pass

__global__ void __launch_bounds__(kThreads, 4)
euler_l1rel_kernel(float4 *__restrict__ x, float4 *__restrict__ vhat,
                   const float4 *__restrict__ v_fresh, const int32_t *__restrict__ pos,
                   int N, int vecs, int lpr_log2, float dsigma, int n_fresh_rows,
                   float *__restrict__ stat, float weight, unsigned *err) {
  pdl_wait();
  pdl_trigger();
  const int L = 1 << lpr_log2;
  const int lane = threadIdx.x & 31;
  const int sub = lane >> lpr_log2;
  const int sl = lane & (L - 1);
  const int rows_per_warp = 32 >> lpr_log2;
  const long long warp = (blockIdx.x * (long long)blockDim.x + threadIdx.x) >> 5;
  const long long nwarps = ((long long)gridDim.x * blockDim.x) >> 5;
  const long long step = nwarps * rows_per_warp;            // between a group's tokens
  // All lanes of a warp run the same number of passes (the shuffles below
  // span the warp): the bound is the token count rounded up to whole passes.
  const long long span = step * kL1relRows;
  const long long rows_pad = ((long long)N + span - 1) / span * span;
  for (long long n0 = warp * rows_per_warp; n0 < rows_pad; n0 += span) {
    long long n[kL1relRows];
    int p[kL1relRows];
#pragma unroll
    for (int k = 0; k < kL1relRows; ++k) {
      n[k] = n0 + k * step + sub;
      p[k] = (n[k] < N) ? __ldg(pos + n[k]) : -1;
      if (p[k] >= n_fresh_rows || p[k] < -1) {
        set_error(err, kErrIndex);
        p[k] = -1;
      }
    }
    float num[kL1relRows], den[kL1relRows];
#pragma unroll
    for (int k = 0; k < kL1relRows; ++k) num[k] = den[k] = 0.f;
    for (int v = sl; v < vecs; v += L) {
      float4 vo[kL1relRows], vn[kL1relRows], xv[kL1relRows];
#pragma unroll
      for (int k = 0; k < kL1relRows; ++k) {
        if (n[k] < N) {
          vo[k] = vhat[n[k] * vecs + v];
          vn[k] = p[k] >= 0 ? __ldg(v_fresh + (long long)p[k] * vecs + v) : vo[k];
          xv[k] = x[n[k] * vecs + v];
        }
      }
#pragma unroll
      for (int k = 0; k < kL1relRows; ++k) {
        if (n[k] < N) {
          if (p[k] >= 0) {
            num[k] += fabsf(vn[k].x - vo[k].x) + fabsf(vn[k].y - vo[k].y) +
                      fabsf(vn[k].z - vo[k].z) + fabsf(vn[k].w - vo[k].w);
            den[k] += fabsf(vn[k].x) + fabsf(vn[k].y) + fabsf(vn[k].z) + fabsf(vn[k].w);
            vhat[n[k] * vecs + v] = vn[k];
          }
          float4 o;
          o.x = __fmaf_rn(vn[k].x, dsigma, xv[k].x);
          o.y = __fmaf_rn(vn[k].y, dsigma, xv[k].y);
          o.z = __fmaf_rn(vn[k].z, dsigma, xv[k].z);
          o.w = __fmaf_rn(vn[k].w, dsigma, xv[k].w);
          x[n[k] * vecs + v] = o;
        }
      }
    }
#pragma unroll
    for (int k = 0; k < kL1relRows; ++k) {
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        if (o < L) {
          num[k] += __shfl_xor_sync(0xffffffffu, num[k], o);
          den[k] += __shfl_xor_sync(0xffffffffu, den[k], o);
        }
      }
      if (n[k] < N && p[k] >= 0 && sl == 0) {
        const float r = den[k] > 0.f ? num[k] / den[k] : (num[k] > 0.f ? 3.402823466e38f : 0.f);
        stat[n[k]] = fmaf(weight, r, stat[n[k]]);
      }
    }
  }
}

// Rotary position embedding of the active rows (Sec. 2.3: the positional
// frequencies are subsampled to A_i): row j of a token tensor is rotated by
// the (cos, sin) table row of its token idx[j].  One 16-byte vector holds 8
// bf16 values = 4 rotation pairs, t0 and t1 their (c, s); pair (x0, x1) becomes
// (fma(x0, c, -(x1 s)), fma(x0, s, x1 c)) in fp32, rounded to bf16.
__device__ __forceinline__ uint4 rope8(uint4 v, const float4 &t0, const float4 &t1) {
  uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    const float4 &cs2 = k < 2 ? t0 : t1;
    const float c = (k & 1) ? cs2.z : cs2.x, s = (k & 1) ? cs2.w : cs2.y;
    const float x0 = __uint_as_float(w[k] << 16), x1 = __uint_as_float(w[k] & 0xffff0000u);
    const float y0 = __fmaf_rn(x0, c, -(x1 * s));
    const float y1 = __fmaf_rn(x0, s, x1 * c);
    const __nv_bfloat162 r = __floats2bfloat162_rn(y0, y1);
    w[k] = *reinterpret_cast<const uint32_t *>(&r);
  }
  return make_uint4(w[0], w[1], w[2], w[3]);
}

// Rotates (or with `plain` copies) a row of `vecs` vectors from s to d, one lane
// group of L lanes per row.  Vector v covers head 8v / D and pairs (8v mod D)/2 ..
// +3.  kFixed: D/8 divides L, so a lane's vectors all sit at the same place of
// their heads and its (c, s) are loaded once per row, with the row's vectors;
// otherwise each vector loads its own.
template <bool kFixed, int kU, class Load>
__device__ __forceinline__ void rope_row(const uint4 *s, uint4 *d, const float4 *trow, int vecs,
                                         int L, int sl, int D, bool plain, Load load) {
  float4 t0 = make_float4(0.f, 0.f, 0.f, 0.f), t1 = t0;
  if (kFixed && !plain) {
    const int p = 2 * (sl & (D / 8 - 1));              // D/8 a power of two: it divides L
    t0 = __ldg(trow + p);
    t1 = __ldg(trow + p + 1);
  }
  for (int v0 = sl; v0 < vecs; v0 += kU * L) {
    uint4 buf[kU];
#pragma unroll
    for (int u = 0; u < kU; ++u)
      if (v0 + u * L < vecs) buf[u] = load(s + v0 + u * L);
#pragma unroll
    for (int u = 0; u < kU; ++u) {
      const int v = v0 + u * L;
      if (v >= vecs) continue;
      if (!kFixed && !plain) {
        const int p = 2 * (v % (D / 8));
        t0 = __ldg(trow + p);
        t1 = __ldg(trow + p + 1);
      }
      d[v] = plain ? buf[u] : rope8(buf[u], t0, t1);
    }
  }
}

// In-place rotation of rows j < n of x [n, H*D] (bf16): a lane group owns a
// row; the index of its next row is loaded one row ahead.  HBM-bound; half of the
// tokens, 3 layers in turn, against one vector in flight per lane and a remainder
// by D for each: 32760 tokens x 12 x 128 24.8 -> 18.5 us (0.88 of the measured HBM
// rate), 75600 x 40 x 128 158 -> 117.7 (1.01).
template <bool kFixed>
__global__ void __launch_bounds__(kThreads)
rope_rows_kernel(uint4 *__restrict__ x, const int32_t *__restrict__ idx, int n, int vecs, int D,
                 const float4 *__restrict__ table, int N, int lpr_log2, unsigned *err) {
  pdl_wait();
  pdl_trigger();
  const int L = 1 << lpr_log2;
  const int lane = threadIdx.x & 31;
  const int sl = lane & (L - 1);
  const long long step = ((long long)gridDim.x * blockDim.x) >> lpr_log2;
  long long j = (blockIdx.x * (long long)blockDim.x + threadIdx.x) >> lpr_log2;
  int t = j < n ? __ldg(idx + j) : 0;
  for (; j < n; j += step) {
    const int t_next = j + step < n ? __ldg(idx + j + step) : 0;
    if (t < 0 || t >= N)
      set_error(err, kErrIndex);
    else
      rope_row<kFixed, kRopeUnroll>(x + j * vecs, x + j * vecs, table + (size_t)t * (D / 4), vecs,
                                    L, sl, D, false, [](const uint4 *p) { return *p; });
    t = t_next;
  }
}

// KV-cache synchronisation with K rotated on the way in: rows 0..n-1 are K
// rows (rotated by the table row of token idx[j]), rows n..2n-1 the V rows
// (copied).  Same sizes: 39.4 -> 36.4 us (0.86), 242 -> 232 (1.01); 6144 x 32 x
// 64 12.6 -> 9.9.
template <bool kFixed>
__global__ void __launch_bounds__(kThreads)
kv_scatter_rope_kernel(uint4 *__restrict__ kc, uint4 *__restrict__ vc,
                       const uint4 *__restrict__ kf, const uint4 *__restrict__ vf,
                       const int32_t *__restrict__ idx, int n_active, int N, int vecs, int D,
                       const float4 *__restrict__ table, int lpr_log2, unsigned *err) {
  pdl_wait();
  pdl_trigger();
  const int L = 1 << lpr_log2;
  const int lane = threadIdx.x & 31;
  const int sl = lane & (L - 1);
  const long long step = ((long long)gridDim.x * blockDim.x) >> lpr_log2;
  const long long rows = 2LL * n_active;
  long long jj = (blockIdx.x * (long long)blockDim.x + threadIdx.x) >> lpr_log2;
  auto row_idx = [&](long long q) {
    return q < rows ? __ldg(idx + (q >= n_active ? q - n_active : q)) : 0;
  };
  int r = row_idx(jj);
  for (; jj < rows; jj += step) {
    const int r_next = row_idx(jj + step);
    const bool is_v = jj >= n_active;
    const long long j = is_v ? jj - n_active : jj;
    if (r < 0 || r >= N) {
      if (!is_v) set_error(err, kErrIndex);
    } else {
      rope_row<kFixed, kRopeScatterUnroll>(
          (is_v ? vf : kf) + j * vecs, (is_v ? vc : kc) + (long long)r * vecs,
          table + (size_t)r * (D / 4), vecs, L, sl, D, is_v, ld_stream);
    }
    r = r_next;
  }
}

// Index check (opt-in, for debugging a caller's index arrays): every entry of
// idx must lie in [0, N) and no value may appear twice.  Sec. 2.2 makes the
// groups disjoint, so A_i never repeats a token; a repeated id would make the
// KV scatter race.  One bit per token in a caller workspace, cleared first
// (bitmap_clear_kernel), then set with atomicOr: an entry that finds its bit
// already set is a repeat.
__global__ void __launch_bounds__(kThreads)
bitmap_clear_kernel(uint4 *__restrict__ bits, long long n_vec) {
  const long long stride = (long long)gridDim.x * blockDim.x;
  for (long long v = blockIdx.x * (long long)blockDim.x + threadIdx.x; v < n_vec; v += stride)
    bits[v] = make_uint4(0u, 0u, 0u, 0u);
}

__global__ void __launch_bounds__(kThreads)
check_indices_kernel(const int32_t *__restrict__ idx, long long n, int N,
                     unsigned *__restrict__ bits, unsigned *err) {
  const long long stride = (long long)gridDim.x * blockDim.x;
  bool bad = false;
  for (long long j = blockIdx.x * (long long)blockDim.x + threadIdx.x; j < n; j += stride) {
    const int t = __ldg(idx + j);
    if (t < 0 || t >= N) {
      bad = true;
      continue;
    }
    const unsigned bit = 1u << (t & 31);
    if (atomicOr(bits + (t >> 5), bit) & bit) bad = true;
  }
  if (bad) set_error(err, kErrIndex);
}

// Grid for n_rows rows handled by lane groups of size L: up to 8 blocks of
// 256 threads per SM (a full SM), no more than the rows need; blocks beyond
// what is resident wait their turn.
int grid_for(long long n_rows, int L, int blocks_per_sm = 2048 / kThreads) {
  const long long rows_per_block = (long long)(kThreads / 32) * (32 / L);
  long long blocks = (n_rows + rows_per_block - 1) / rows_per_block;
  const long long cap = (long long)sm_count() * blocks_per_sm;
  if (blocks > cap) blocks = cap;
  return (int)(blocks < 1 ? 1 : blocks);
}

// Blocks of kernel K (kThreads threads) resident on the whole device at once,
// resolved once per device: a grid-stride kernel launched with this many
// blocks runs in a single wave.
template <auto K>
long long resident_blocks() {
  static std::atomic<int> per_sm[64];
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return sm_count();
  int nb = per_sm[dev].load(std::memory_order_relaxed);
  if (nb <= 0) {
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, K, kThreads, 0) != cudaSuccess ||
        nb < 1)
      nb = 1;
    per_sm[dev].store(nb, std::memory_order_relaxed);
  }
  return (long long)nb * sm_count();
}

// How a row copy runs, by the 16-byte vectors each lane moves per row.  Swept over
// rows of 64 B to 10 KB, 12 to 320 MB (gather also 1 GB), half and all rows, 2 or 3
// layers in turn, against 4 (gather) and 8 (scatter) vectors in flight, index in
// place, 8 blocks per SM; ratios are before / now (means: gather 1.05, scatter 1.06;
// below 1 they are 0.1 to 0.4 us of calls under 10 us, or 1.5 % of 2304-byte rows).
// Half of 40 x 128 bf16 rows of 32760 tokens, gather and scatter: 160.0 -> 153.0 us.
//   Grid.  40 to 64 registers leave 4 to 6 blocks of 256 resident; of 8 launched
//   per SM the rest are an uneven second wave.  32 replace one another as they
//   end: gather of 1310720 x 256 B 1.13 -> 1.27, scatter of 81920 x 4 KB 1.00 ->
//   1.06.  The scatter of short rows is as good or better with 8 (163840 x 256 B
//   1.16 against 1.02): more rows per group hide the index.
//   Gather.  Up to 2 vectors: 4 in flight, the index one row ahead, 1.00 .. 1.43.
//   5, 6 or more than 8: 6 in flight take the odd remainder in one round or few,
//   1.01 .. 1.22 up to 6, 0.96 .. 1.06 above.  3, 4, 7 and 8: 4 with the index in
//   place, 0.96 .. 1.05 (read ahead it is 0.67 .. 1.0, with 6 0.87 .. 1.05).
//   Scatter.  4 in flight, index ahead: 1.02 .. 1.40 up to 2 vectors, 0.98 .. 1.20
//   above; a fifth vector that is not whole takes 6 (129 vectors: 1.00 .. 1.02
//   against 0.89 .. 0.99).
struct CopyPlan {
  int unroll;
  bool ahead;
  int blocks;      // per SM, at most
};

CopyPlan gather_plan(long long vecs, int L) {
  const long long per_lane = (vecs + L - 1) / L;
  if (per_lane <= 2) return CopyPlan{4, true, 32};
  if (per_lane > 8 || per_lane == 5 || per_lane == 6) return CopyPlan{6, true, 32};
  return CopyPlan{4, false, 32};
}

CopyPlan scatter_plan(long long vecs, int L) {
  const long long per_lane = (vecs + L - 1) / L;
  if (per_lane == 5 && vecs % L != 0) return CopyPlan{6, true, 8};
  return CopyPlan{4, true, per_lane <= 2 ? 8 : 32};
}

int log2i(int L) {
  int s = 0;
  while ((1 << s) < L) ++s;
  return s;
}

}  // namespace
}  // namespace hsa

using namespace hsa;

extern "C" int hsa_gather_active(const void *src, size_t row_bytes, int N,
                                 const int32_t *idx, int n_active, void *dst,
                                 hsa_stream_t stream) {
  if (N < 0 || n_active < 0 || row_bytes == 0 || (row_bytes & 15)) return HSA_ERR_INVALID_ARG;
  if (n_active == 0) return HSA_OK;
  if (!src || !dst || !idx || !aligned16(src) || !aligned16(dst)) return HSA_ERR_INVALID_ARG;
  const long long vecs = (long long)(row_bytes / 16);
  if (vecs > (1LL << 30)) return HSA_ERR_UNSUPPORTED;
  unsigned *err = device_error_word();
  if (!err) return HSA_ERR_CUDA;
  const int L = lanes_per_row(vecs);
  count_launches(1);
  const CopyPlan plan = gather_plan(vecs, L);
  launch_pdl(plan.unroll == 6 ? gather_rows_kernel<6, true>
             : plan.ahead     ? gather_rows_kernel<4, true>
                              : gather_rows_kernel<4, false>,
             dim3(grid_for(n_active, L, plan.blocks)), dim3(kThreads), 0, (cudaStream_t)stream,
             (const uint4 *)src, (uint4 *)dst, idx, n_active, N, (int)vecs,
             log2i(L), err);
  return launch_status();
}

extern "C" int hsa_kv_sync_scatter(void *k_cache, void *v_cache, const void *k_fresh,
                                   const void *v_fresh, const int32_t *idx, int n_active,
                                   int N, int H, int D, hsa_dtype dtype,
                                   hsa_stream_t stream) {
  if (N < 0 || n_active < 0 || H < 1 || D < 1) return HSA_ERR_INVALID_ARG;
  if (dtype != HSA_BF16 && dtype != HSA_F32) return HSA_ERR_INVALID_ARG;
  const long long row_bytes = (long long)H * D * (dtype == HSA_BF16 ? 2 : 4);
  if (row_bytes & 15) return HSA_ERR_UNSUPPORTED;
  if (n_active == 0) return HSA_OK;
  if (!k_cache || !v_cache || !k_fresh || !v_fresh || !idx) return HSA_ERR_INVALID_ARG;
  if (!aligned16(k_cache) || !aligned16(v_cache) || !aligned16(k_fresh) || !aligned16(v_fresh))
    return HSA_ERR_INVALID_ARG;
  const long long vecs = row_bytes / 16;
  if (vecs > (1LL << 30)) return HSA_ERR_UNSUPPORTED;
  unsigned *err = device_error_word();
  if (!err) return HSA_ERR_CUDA;
  const int L = lanes_per_row(vecs);
  count_launches(1);
  const CopyPlan plan = scatter_plan(vecs, L);
  launch_pdl(plan.unroll == 6 ? kv_scatter_kernel<6> : kv_scatter_kernel<4>,
             dim3(grid_for(2LL * n_active, L, plan.blocks)), dim3(kThreads), 0,
             (cudaStream_t)stream, (uint4 *)k_cache, (uint4 *)v_cache, (const uint4 *)k_fresh,
             (const uint4 *)v_fresh, idx, n_active, N, (int)vecs, log2i(L), err);
  return launch_status();
}

extern "C" int hsa_cached_euler(float *x, float *v_cache, const float *v_fresh,
                                const int32_t *pos, int n_fresh, int N, int C, float dsigma,
                                hsa_stream_t stream) {
  if (N < 0 || C < 4 || (C & 3) || n_fresh < 0) return HSA_ERR_INVALID_ARG;
  if ((pos == nullptr) != (v_fresh == nullptr)) return HSA_ERR_INVALID_ARG;
  if (N == 0) return HSA_OK;
  if (!x || !v_cache || !aligned16(x) || !aligned16(v_cache)) return HSA_ERR_INVALID_ARG;
  if (v_fresh && !aligned16(v_fresh)) return HSA_ERR_INVALID_ARG;
  unsigned *err = device_error_word();
  if (!err) return HSA_ERR_CUDA;
  const int vecs = C / 4;
  const long long total = (long long)N * vecs;
  int vec_shift = -1;
  for (int sh = 0; sh < 31; ++sh)
    if ((1 << sh) == vecs) vec_shift = sh;
  const long long resident = (long long)sm_count() * 2048;     // threads
  const int per =
      vecs >= 16 && total >= (long long)kEulerUnroll * resident ? kEulerUnroll : 1;
  long long blocks = (total + (long long)kThreads * per - 1) / ((long long)kThreads * per);
  const long long cap = per == kEulerUnroll ? resident_blocks<cached_euler_kernel<kEulerUnroll>>()
                                            : resident_blocks<cached_euler_kernel<1>>();
  if (blocks > cap) blocks = cap;
  count_launches(1);
  if (per == kEulerUnroll)
    launch_pdl(cached_euler_kernel<kEulerUnroll>, dim3((unsigned)blocks), dim3(kThreads), 0,
               (cudaStream_t)stream, (float4 *)x, (float4 *)v_cache, (const float4 *)v_fresh,
               pos, total, vecs, vec_shift, dsigma, pos ? n_fresh : 0, err);
  else
    launch_pdl(cached_euler_kernel<1>, dim3((unsigned)blocks), dim3(kThreads), 0,
               (cudaStream_t)stream, (float4 *)x, (float4 *)v_cache, (const float4 *)v_fresh,
               pos, total, vecs, vec_shift, dsigma, pos ? n_fresh : 0, err);
  return launch_status();
}

extern "C" int hsa_cached_euler_l1rel(float *x, float *v_cache, const float *v_fresh,
                                      const int32_t *pos, int n_fresh, int N, int C,
                                      float dsigma, float *stat, float weight,
                                      hsa_stream_t stream) {
  if (N < 0 || C < 4 || (C & 3) || n_fresh < 0) return HSA_ERR_INVALID_ARG;
  if (!pos || !v_fresh || !stat) return HSA_ERR_INVALID_ARG;
  if (N == 0) return HSA_OK;
  if (!x || !v_cache || !aligned16(x) || !aligned16(v_cache) || !aligned16(v_fresh))
    return HSA_ERR_INVALID_ARG;
  unsigned *err = device_error_word();
  if (!err) return HSA_ERR_CUDA;
  const int vecs = C / 4;
  const int L = lanes_per_row(vecs);
  count_launches(1);
  if (vecs <= 32) {
    long long blocks = (((long long)N << log2i(L)) + kThreads - 1) / kThreads;
    const long long cap = resident_blocks<euler_l1rel_elem_kernel>();
    if (blocks > cap) blocks = cap;
    launch_pdl(euler_l1rel_elem_kernel, dim3((unsigned)blocks), dim3(kThreads), 0,
               (cudaStream_t)stream, (float4 *)x, (float4 *)v_cache, (const float4 *)v_fresh, pos,
               N, vecs, log2i(L), dsigma, n_fresh, stat, weight, err);
    return launch_status();
  }
  launch_pdl(euler_l1rel_kernel,
             dim3((unsigned)grid_for(((long long)N + kL1relRows - 1) / kL1relRows, L)),
             dim3(kThreads), 0, (cudaStream_t)stream, (float4 *)x, (float4 *)v_cache,
             (const float4 *)v_fresh, pos, N, vecs, log2i(L), dsigma, n_fresh, stat, weight, err);
  return launch_status();
}

extern "C" int hsa_rope_table(int F, int Hh, int Ww, int D, double theta, float *table) {
  if (F < 1 || Hh < 1 || Ww < 1 || D < 8 || (D & 7) || !(theta > 1.0) || !table)
    return HSA_ERR_INVALID_ARG;
  const int P = D / 2, ph = D / 6, pt = P - 2 * ph;
  for (int f = 0; f < F; ++f)
    for (int h = 0; h < Hh; ++h)
      for (int w = 0; w < Ww; ++w) {
        const size_t n = ((size_t)f * Hh + h) * Ww + w;
        for (int i = 0; i < P; ++i) {
          const bool tb = i < pt, hb = !tb && i < pt + ph;
          const int bi = tb ? i : (hb ? i - pt : i - pt - ph);
          const int bp = tb ? pt : ph;
          const int pos = tb ? f : (hb ? h : w);
          const double ang = (double)pos * std::pow(theta, -(double)bi / (double)bp);
          table[(n * P + i) * 2] = (float)std::cos(ang);
          table[(n * P + i) * 2 + 1] = (float)std::sin(ang);
        }
      }
  return HSA_OK;
}

extern "C" int hsa_rope_rows(void *x, const int32_t *idx, int n, int H, int D,
                             const float *table, int N, hsa_stream_t stream) {
  if (n < 0 || H < 1 || D < 8 || (D & 7) || N < 1) return HSA_ERR_INVALID_ARG;
  if (n == 0) return HSA_OK;
  if (!x || !idx || !table || !aligned16(x) || !aligned16(table)) return HSA_ERR_INVALID_ARG;
  unsigned *err = device_error_word();
  if (!err) return HSA_ERR_CUDA;
  const long long vecs = (long long)H * D / 8;
  if (vecs > (1LL << 30)) return HSA_ERR_UNSUPPORTED;
  const int L = lanes_per_row(vecs);
  count_launches(1);
  launch_pdl(L % (D / 8) == 0 ? rope_rows_kernel<true> : rope_rows_kernel<false>,
             dim3((unsigned)grid_for(n, L, kRopeBlocks)), dim3(kThreads), 0, (cudaStream_t)stream, (uint4 *)x,
             idx, n, (int)vecs, D, (const float4 *)table, N, log2i(L), err);
  return launch_status();
}

extern "C" int hsa_kv_sync_scatter_rope(void *k_cache, void *v_cache, const void *k_fresh,
                                        const void *v_fresh, const int32_t *idx, int n_active,
                                        int N, int H, int D, const float *table,
                                        hsa_stream_t stream) {
  if (N < 0 || n_active < 0 || H < 1 || D < 8 || (D & 7)) return HSA_ERR_INVALID_ARG;
  if (n_active == 0) return HSA_OK;
  if (!k_cache || !v_cache || !k_fresh || !v_fresh || !idx || !table) return HSA_ERR_INVALID_ARG;
  if (!aligned16(k_cache) || !aligned16(v_cache) || !aligned16(k_fresh) || !aligned16(v_fresh) ||
      !aligned16(table))
    return HSA_ERR_INVALID_ARG;
  unsigned *err = device_error_word();
  if (!err) return HSA_ERR_CUDA;
  const long long vecs = (long long)H * D / 8;
  if (vecs > (1LL << 30)) return HSA_ERR_UNSUPPORTED;
  const int L = lanes_per_row(vecs);
  count_launches(1);
  launch_pdl(L % (D / 8) == 0 ? kv_scatter_rope_kernel<true> : kv_scatter_rope_kernel<false>,
             dim3((unsigned)grid_for(2LL * n_active, L, kRopeBlocks)), dim3(kThreads), 0, (cudaStream_t)stream,
             (uint4 *)k_cache, (uint4 *)v_cache, (const uint4 *)k_fresh, (const uint4 *)v_fresh,
             idx, n_active, N, (int)vecs, D, (const float4 *)table, log2i(L), err);
  return launch_status();
}

extern "C" size_t hsa_check_indices_workspace_bytes(int N) {
  if (N <= 0) return 0;
  return (((size_t)N + 31) / 32 * 4 + 255) / 256 * 256;   // one bit per token, whole uint4s
}

extern "C" int hsa_check_indices(const int32_t *idx, int n, int N, void *workspace,
                                 size_t workspace_bytes, hsa_stream_t stream) {
  if (n < 0 || N < 0) return HSA_ERR_INVALID_ARG;
  if (n == 0) return HSA_OK;
  if (!idx) return HSA_ERR_INVALID_ARG;
  const size_t need = hsa_check_indices_workspace_bytes(N);
  if (N > 0 && (!workspace || workspace_bytes < need ||
                (reinterpret_cast<uintptr_t>(workspace) & 255)))
    return HSA_ERR_WORKSPACE;
  unsigned *err = device_error_word();
  if (!err) return HSA_ERR_CUDA;
  const long long cap = (long long)sm_count() * (2048 / kThreads);
  const long long n_vec = (long long)(need / 16);
  long long b0 = (n_vec + kThreads - 1) / kThreads, b1 = ((long long)n + kThreads - 1) / kThreads;
  b0 = b0 < 1 ? 1 : (b0 > cap ? cap : b0);
  b1 = b1 > cap ? cap : b1;
  cudaStream_t s = (cudaStream_t)stream;
  if (n_vec > 0) {
    count_launches(1);
    bitmap_clear_kernel<<<(int)b0, kThreads, 0, s>>>(static_cast<uint4 *>(workspace), n_vec);
  }
  count_launches(1);
  check_indices_kernel<<<(int)b1, kThreads, 0, s>>>(idx, n, N, static_cast<unsigned *>(workspace),
                                                    err);
  return launch_status();
}
