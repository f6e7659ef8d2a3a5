// knn.cu -- brute-force tiled kNN candidate selection (Gramacy & Haaland,
// Sec 2.2: the local search is restricted to the N' nearest neighbours of x).
//
// Two stages:
//  1. knn_stream: each CTA owns 32 predictive locations (4 per warp) and
//     streams the whole design through shared memory in 256-point tiles moved
//     by bulk-copy (TMA) into a double buffer.  Distances are computed in FP32
//     from centred coordinates; a point enters its location's candidate
//     buffer when d32 <= tau + 2 err, where tau is the N'-th smallest buffered
//     d32 and err a proven bound on |d32 - d64|.  A warp radix-selects tau and
//     compacts the buffer whenever the next tile might overflow it.
//  2. knn_rank: one CTA per location puts the surviving points in the order of
//     (d64, index), d64 the binary64 distance in the oracle's operation order;
//     the first N' indices are the candidate list.
// Every true member of the N'-nearest set survives stage 1: at the end at
// least N' points have d32 <= tau, so the N'-th smallest d64 is at most
// tau + err, and any member has d32 <= d64 + err <= tau + 2 err.
//
// Pilot threshold (knn_has_pilot).  Before the stream, knn_pilot estimates each
// location's N'-th distance from a sample of S = min(32768, N / 16) design points,
// one from each S-th of the rows at a place that steps through it by the golden
// ratio (at a fixed place, a gridded design whose rows are as long as the step
// gives a sample of one of its columns: 16 x 16 x 16 points, 5,000 locations, N' =
// 300 took 0.62 instead of 0.25 ms, most of them streamed again): with
// lambda = S N'/N sample points expected inside it, the m-th smallest sample
// distance, m = lambda + 4.5 sqrt(lambda) + 4, is above it except with
// probability ~1e-5.  The stream starts with tau = that value instead of
// infinity, so few points are buffered and the buffer rarely needs a
// compaction.  The estimate is checked, not trusted: at the end at least N'
// buffered points must lie at or below it (then the N'-th smallest d32 does
// too, and every point that could belong was admitted); a location that fails
// the check is streamed again with tau = infinity.
#include <cfloat>
#include <cmath>
#include <cstdint>

#include "common.cuh"
#include "knn_common.cuh"
#include "lagp_internal.h"
#include "launch_plan.h"

namespace lagp {

#define KNN_WARPS 8
#define KNN_QW 4   // locations per warp


// ---------------------------------------------------------------------------
// Preparation: bounding box (exact min/max), centred FP32 copy of the design,
// squared norms, largest squared norm.
// ---------------------------------------------------------------------------
__global__ void bbox_partial(const double* __restrict__ X, int64_t N, int p,
                             double* __restrict__ part /*[gridDim.x][2p]*/) {
  __shared__ double slo[256], shi[256];
  for (int k = 0; k < p; ++k) {
    double lo = __longlong_as_double(0x7ff0000000000000ll), hi = -lo;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < N;
         i += (int64_t)gridDim.x * blockDim.x) {
      double v = X[i * p + k];
      lo = fmin(lo, v);
      hi = fmax(hi, v);
    }
    slo[threadIdx.x] = lo;
    shi[threadIdx.x] = hi;
    __syncthreads();
    for (int s = blockDim.x / 2; s > 0; s >>= 1) {
      if (threadIdx.x < s) {
        slo[threadIdx.x] = fmin(slo[threadIdx.x], slo[threadIdx.x + s]);
        shi[threadIdx.x] = fmax(shi[threadIdx.x], shi[threadIdx.x + s]);
      }
      __syncthreads();
    }
    if (threadIdx.x == 0) {
      part[blockIdx.x * 2 * p + k] = slo[0];
      part[blockIdx.x * 2 * p + p + k] = shi[0];
    }
    __syncthreads();
  }
}

__global__ void bbox_final(const double* __restrict__ part, int nparts, int p,
                           double* __restrict__ lo, double* __restrict__ hi,
                           double* __restrict__ center) {
  int k = threadIdx.x;
  if (k >= p) return;
  double l = part[k], h = part[p + k];
  for (int b = 1; b < nparts; ++b) {
    l = fmin(l, part[b * 2 * p + k]);
    h = fmax(h, part[b * 2 * p + p + k]);
  }
  lo[k] = l;
  hi[k] = h;
  center[k] = 0.5 * (l + h);
}

// Xf[i][0..PP) = fl32(X[i] - center) (zero padded), nx[i] = |Xf[i]|^2 in FP32;
// rows N..Npad-1 are zero with nx = NaN.  maxn2 receives max_{i<N} nx[i]
// (as ordered bits).
__global__ void design_to_f32(const double* __restrict__ X, int64_t N, int64_t Npad, int p, int PP,
                              const double* __restrict__ center, float* __restrict__ Xf,
                              float* __restrict__ nx, unsigned* __restrict__ maxn2_bits) {
  float local_max = 0.f;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < Npad;
       i += (int64_t)gridDim.x * blockDim.x) {
    float acc = 0.f;
    for (int k = 0; k < PP; ++k) {
      float v = 0.f;
      if (i < N && k < p) v = (float)(X[i * p + k] - center[k]);
      Xf[i * PP + k] = v;
      acc = fmaf(v, v, acc);
    }
    // padding rows get |x|^2 = NaN, so that no distance to them passes whatever
    // the design's scale and the threshold (1e30 passed from coordinates of 1e15 on)
    nx[i] = i < N ? acc : __int_as_float(0x7fc00000);
    if (i < N) local_max = fmaxf(local_max, acc);
  }
  for (int o = 16; o > 0; o >>= 1) local_max = fmaxf(local_max, __shfl_xor_sync(0xffffffffu, local_max, o));
  if ((threadIdx.x & 31) == 0) atomicMax(maxn2_bits, __float_as_uint(local_max));
}

template <int PP>
__device__ __forceinline__ void knn_d4(const float (&qf)[KNN_QW][PP], const float (&nq)[KNN_QW],
                                       const float (&xv)[PP], float nxp, float (&d)[KNN_QW]) {
#pragma unroll
  for (int a = 0; a < KNN_QW; ++a) {
    float dot = 0.f;
#pragma unroll
    for (int k = 0; k < PP; ++k) dot = fmaf(qf[a][k], xv[k], dot);
    d[a] = fmaf(-2.f, dot, nq[a] + nxp);
  }
}

// first bin (of 256 per location, lane l owning bins 8l..8l+7) at which the
// running count reaches k; *below receives the count before that bin
__device__ __forceinline__ int warp_bin_of_kth(const uint32_t* h, int k, int* below) {
  const int lane = threadIdx.x & 31;
  uint32_t c[8], tot = 0;
#pragma unroll
  for (int b = 0; b < 8; ++b) { c[b] = h[lane * 8 + b]; tot += c[b]; }
  uint32_t incl = tot;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t t = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += t;
  }
  const uint32_t excl = incl - tot;
  const int found = ((int)excl < k && (int)incl >= k);
  const uint32_t fm = __ballot_sync(0xffffffffu, found);
  int bin = 255, run_out = 0;
  if (found) {
    uint32_t run = excl;
#pragma unroll
    for (int b = 0; b < 8; ++b) {
      if ((int)(run + c[b]) >= k) { bin = lane * 8 + b; run_out = (int)run; break; }
      run += c[b];
    }
  }
  const int src = fm ? __ffs(fm) - 1 : 0;
  *below = __shfl_sync(0xffffffffu, run_out, src);
  return fm ? __shfl_sync(0xffffffffu, bin, src) : -1;
}

// design row of sample i
__device__ __forceinline__ int64_t pilot_row(int64_t i, int64_t step) {
  return i * step + __umulhi((uint32_t)i * 2654435769u, (uint32_t)step);
}

__device__ __forceinline__ float pilot_err2(float errc, float nq, unsigned maxn2) {
  const float r = (sqrtf(__uint_as_float(maxn2)) + sqrtf(nq)) * 1.0001f;
  return 2.f * errc * r * r;
}
// Rows up to the threshold + err2 are counted by bins (2^-8 of an octave) where that
// stays in the threshold's octave b1, and else by whole octaves: those up to the one
// reached where err2 alone leads past b1 (pilot_past, 0 where it does not), else those
// up to b1.
__device__ __forceinline__ uint32_t pilot_past(uint32_t b1, float err2) {
  const uint32_t e = __float_as_uint(__uint_as_float(b1 << 23) + err2) >> 23;
  return e > b1 ? e + 1u : 0u;
}
// the first n of 256 counts, over the warp (lane l owning counts 8l..8l+7)
__device__ __forceinline__ int pilot_count(const uint32_t* h, uint32_t n) {
  const int lane = threadIdx.x & 31;
  int c = 0;
#pragma unroll
  for (int u = 0; u < 8; ++u) c += lane * 8 + u < (int)n ? (int)h[lane * 8 + u] : 0;
  return __reduce_add_sync(0xffffffffu, c);
}

// Pilot thresholds: per location the upper edge of the 2^-8-wide bin (by the
// float bit pattern: exponent, then the top 8 mantissa bits) that holds the
// m-th smallest d32 of the S sample rows; +inf where the pilot
// does not apply (m > S, or more than cap - 2 tiles expected below it).  CHECK: nor
// where the tensor-core filter, which admits up to the threshold + 2 err, err = errc
// (|a| + |b|)^2, would admit too many, more than `fit` sample rows lying below that.
// That is for strongly clustered designs, with buffers that are larger for the
// threshold's sake: 20,000 points in 20 clusters that err spans, 5,000 locations,
// N' = 30 took 1.11 ms with thresholds that admitted whole clusters, 0.51 streamed
// from infinity with the smallest buffers, and take 0.58.  The check costs the
// pilot 2 to 10% (1.50 to 1.62 ms for 40,000 locations, p = 4).
template <int PP, bool CHECK>
__global__ void __launch_bounds__(KNN_WARPS * 32)
knn_pilot(const float* __restrict__ Xf, const float* __restrict__ nx, int64_t N, int64_t S, int p,
          const double* __restrict__ xref, int64_t M, const double* __restrict__ center,
          int nc_max, const int32_t* __restrict__ nc_loc, int cap, float errc, int fit,
          const unsigned* __restrict__ maxn2_bits, float* __restrict__ thr_out) {
  // the sample rows pass through shared memory a tile at a time, shared by
  // the CTA's warps (each sample row is read from L2 once per CTA and pass);
  // a tile holds the rows' first four coordinates, then their next four, ...,
  // so that the lanes' 128-bit reads are contiguous, and the next tile is
  // loaded while this one is counted (rows side by side, loaded between barriers:
  // 5.40 ms for 100,000 locations at p = 8, S = 32768; now 5.01)
  constexpr int T = 2048 / PP, TN = (T + KNN_WARPS * 32 - 1) / (KNN_WARPS * 32);
  __shared__ uint32_t hist[KNN_WARPS][KNN_QW][256];
  __shared__ float4 sx[PP / 4][T];
  __shared__ float sn[T];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int64_t q0 = (int64_t)blockIdx.x * (KNN_WARPS * KNN_QW) + warp * KNN_QW;
  float qf[KNN_QW][PP], nq[KNN_QW];
  int m[KNN_QW];
  const int64_t step = N / S;
#pragma unroll
  for (int a = 0; a < KNN_QW; ++a) {
    const int64_t q = q0 + a;
    const bool live = q < M;
    float acc = 0.f;
#pragma unroll
    for (int k = 0; k < PP; ++k) {
      float v = 0.f;
      if (live && k < p) v = (float)(xref[q * p + k] - center[k]);
      qf[a][k] = v;
      acc = fmaf(v, v, acc);
    }
    nq[a] = acc;
    const int nc = live ? (nc_loc ? nc_loc[q] : nc_max) : 0;
    const float lam = (float)S * (float)nc / (float)N;
    m[a] = (int)ceilf(lam + 4.5f * sqrtf(lam) + 4.f);
    // expected admitted points m N / S must leave two tiles of room
    if (!live || m[a] > S || (double)m[a] * (double)N / (double)S > (double)(cap - 2 * LAGP_KNN_TILE))
      m[a] = 0;
  }
  uint32_t b1[KNN_QW];
  int below[KNN_QW];
  for (int pass = 0; pass < 2; ++pass) {
    for (int i = lane; i < KNN_QW * 256; i += 32) (&hist[warp][0][0])[i] = 0u;
    __syncwarp();
    float4 rx[2];                                  // T * PP = 8 floats per thread
    float rn[TN];
    auto fetch = [&](int64_t t0) {
#pragma unroll
      for (int u = 0; u < 2; ++u) {
        const int e = threadIdx.x + u * KNN_WARPS * 32, r = e / (PP / 4), c = e - r * (PP / 4);
        if (r < T && t0 + r < S)
          rx[u] = __ldg(reinterpret_cast<const float4*>(Xf + pilot_row(t0 + r, step) * PP) + c);
      }
#pragma unroll
      for (int u = 0; u < TN; ++u) {
        const int r = threadIdx.x + u * KNN_WARPS * 32;
        if (r < T && t0 + r < S) rn[u] = __ldg(nx + pilot_row(t0 + r, step));
      }
    };
    fetch(0);
    for (int64_t t0 = 0; t0 < S; t0 += T) {
      const int cnt = (int)(S - t0 < T ? S - t0 : T);
      __syncthreads();   // the previous tile is consumed
#pragma unroll
      for (int u = 0; u < 2; ++u) {
        const int e = threadIdx.x + u * KNN_WARPS * 32, r = e / (PP / 4), c = e - r * (PP / 4);
        if (r < T) sx[c][r] = rx[u];
      }
#pragma unroll
      for (int u = 0; u < TN; ++u) {
        const int r = threadIdx.x + u * KNN_WARPS * 32;
        if (r < T) sn[r] = rn[u];
      }
      __syncthreads();
      fetch(t0 + T);
      for (int i = lane; i < cnt; i += 32) {
        float xv[PP];
#pragma unroll
        for (int k = 0; k < PP; k += 4) {
          const float4 v4 = sx[k / 4][i];
          xv[k] = v4.x; xv[k + 1] = v4.y; xv[k + 2] = v4.z; xv[k + 3] = v4.w;
        }
        float d[KNN_QW];
        knn_d4<PP>(qf, nq, xv, sn[i], d);
#pragma unroll
        for (int a = 0; a < KNN_QW; ++a) {
          const uint32_t bits = __float_as_uint(fmaxf(d[a], 0.f));
          if (pass == 0) atomicAdd(&hist[warp][a][bits >> 23], 1u);
          else if ((bits >> 23) == b1[a]) atomicAdd(&hist[warp][a][(bits >> 15) & 255u], 1u);
        }
      }
    }
    __syncwarp();
#pragma unroll
    for (int a = 0; a < KNN_QW; ++a) {
      if (pass == 0) {
        const int b = warp_bin_of_kth(hist[warp][a], m[a] > 0 ? m[a] : 1, &below[a]);
        b1[a] = b < 0 ? 0u : (uint32_t)b;
        if (CHECK) {
          const uint32_t past = pilot_past(b1[a], pilot_err2(errc, nq[a], *maxn2_bits));
          if (past && pilot_count(hist[warp][a], past) > fit) m[a] = 0;
        }
      } else {
        int dummy = 0;
        const int b = warp_bin_of_kth(hist[warp][a], m[a] > 0 ? m[a] - below[a] : 1, &dummy);
        float thr = __uint_as_float((b1[a] << 23) | ((uint32_t)(b < 0 ? 255 : b) << 15) | 0x7fffu);
        if (CHECK) {
          const float err2 = pilot_err2(errc, nq[a], *maxn2_bits);
          if (!pilot_past(b1[a], err2)) {
            const uint32_t k = __float_as_uint(thr + err2) >> 15;
            const uint32_t n = k >> 8 == b1[a] ? (k & 255u) + 1u : 256u;
            if (below[a] + pilot_count(hist[warp][a], n) > fit) m[a] = 0;
          }
        }
        if (m[a] == 0 || b < 0 || !(thr < __int_as_float(0x7f800000))) thr = __int_as_float(0x7f800000);
        if (lane == 0 && q0 + a < M) thr_out[q0 + a] = thr;
      }
    }
    __syncwarp();
  }
}

// The same thresholds for a small batch (knn_pilot_alone): one block per location
// instead of one per 32 locations, whose two passes over the sample a lone location
// waits for (0.65 ms at S = 32768).  Every thread keeps its at most 32 distances in
// registers; the bin of the m-th smallest comes from 16 halvings of the 16-bit
// bin number by counting: 0.058 ms for one location, 0.36 ms for 1,024.
#define KNN_PILOT1_THREADS 1024
template <int PP, bool CHECK>
__global__ void __launch_bounds__(KNN_PILOT1_THREADS)
knn_pilot1(const float* __restrict__ Xf, const float* __restrict__ nx, int64_t N, int64_t S, int p,
           const double* __restrict__ xref, int64_t M, const double* __restrict__ center,
           int nc_max, const int32_t* __restrict__ nc_loc, int cap, float errc, int fit,
           const unsigned* __restrict__ maxn2_bits, float* __restrict__ thr_out) {
  constexpr int T = 32768 / KNN_PILOT1_THREADS;    // S <= 32768
  __shared__ int cnt[2][KNN_PILOT1_THREADS / 32];
  const int64_t q = blockIdx.x;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int64_t step = N / S;
  float qf[PP], nq = 0.f;
#pragma unroll
  for (int k = 0; k < PP; ++k) {
    qf[k] = k < p ? (float)(xref[q * p + k] - center[k]) : 0.f;
    nq = fmaf(qf[k], qf[k], nq);
  }
  uint32_t bin[T];
#pragma unroll
  for (int u = 0; u < T; ++u) {
    const int64_t i = (int64_t)u * KNN_PILOT1_THREADS + tid;
    bin[u] = 0xffffffffu;
    if (i < S) {
      const int64_t row = pilot_row(i, step);
      const float* x = Xf + row * PP;
      float dot = 0.f;
#pragma unroll
      for (int k = 0; k < PP; k += 4) {
        const float4 v = __ldg(reinterpret_cast<const float4*>(x + k));
        dot = fmaf(qf[k], v.x, dot);
        dot = fmaf(qf[k + 1], v.y, dot);
        dot = fmaf(qf[k + 2], v.z, dot);
        dot = fmaf(qf[k + 3], v.w, dot);
      }
      const float d = fmaf(-2.f, dot, nq + __ldg(nx + row));
      bin[u] = __float_as_uint(fmaxf(d, 0.f)) >> 15;
    }
  }
  const int nc = nc_loc ? nc_loc[q] : nc_max;
  const float lam = (float)S * (float)nc / (float)N;
  int m = (int)ceilf(lam + 4.5f * sqrtf(lam) + 4.f);
  // expected admitted points m N / S must leave two tiles of room
  if (m > S || (double)m * (double)N / (double)S > (double)(cap - 2 * LAGP_KNN_TILE)) m = 0;
  uint32_t b = 0;      // the smallest bin with at least m distances in bins <= it
  for (int bit = 15; bit >= 0; --bit) {
    const uint32_t mid = b | ((1u << bit) - 1u);
    int c = 0;
#pragma unroll
    for (int u = 0; u < T; ++u) c += bin[u] <= mid ? 1 : 0;
    c = __reduce_add_sync(0xffffffffu, c);
    if (lane == 0) cnt[bit & 1][warp] = c;
    __syncthreads();
    c = __reduce_add_sync(0xffffffffu, cnt[bit & 1][lane]);
    if (c < m) b = mid + 1u;
  }
  const float edge = __uint_as_float((b << 15) | 0x7fffu);
  if (CHECK) {
    const float err2 = pilot_err2(errc, nq, *maxn2_bits);
    const uint32_t b1 = b >> 8, past = pilot_past(b1, err2);
    const uint32_t k = __float_as_uint(edge + err2) >> 15;
    const uint32_t lim = past ? past << 8 : (k >> 8 == b1 ? k + 1u : (b1 + 1u) << 8);
    int c = 0;
#pragma unroll
    for (int u = 0; u < T; ++u) c += bin[u] < lim ? 1 : 0;
    c = __reduce_add_sync(0xffffffffu, c);
    __syncthreads();
    if (lane == 0) cnt[0][warp] = c;
    __syncthreads();
    c = __reduce_add_sync(0xffffffffu, cnt[0][lane]);
    if (c > fit) m = 0;
  }
  if (tid == 0) {
    const float inf = __int_as_float(0x7f800000);
    thr_out[q] = (m == 0 || !(edge < inf)) ? inf : edge;
  }
}

template <int PP>
__global__ void __launch_bounds__(KNN_WARPS * 32, 3)
knn_stream(const float* __restrict__ Xf, const float* __restrict__ nx, int64_t N, int64_t ntiles,
           int p, const double* __restrict__ xref, int64_t M, const double* __restrict__ center,
           const unsigned* __restrict__ maxn2_bits, int nc_max, const int32_t* __restrict__ nc_loc,
           int cap, KnnEntry* __restrict__ buf, int32_t* __restrict__ cnt_out,
           unsigned* __restrict__ status, const float* __restrict__ pilot, int redo) {
  extern __shared__ __align__(128) unsigned char smem[];
  float* tile = reinterpret_cast<float*>(smem);                    // [2][TILE][PP]
  float* tnorm = tile + 2 * LAGP_KNN_TILE * PP;                     // [2][TILE]
  uint32_t* hist = reinterpret_cast<uint32_t*>(tnorm + 2 * LAGP_KNN_TILE);  // [WARPS][256]
  uint64_t* bar = reinterpret_cast<uint64_t*>(hist + KNN_WARPS * 256);      // [2]

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int64_t q0 = (int64_t)blockIdx.x * (KNN_WARPS * KNN_QW) + warp * KNN_QW;

  float qf[KNN_QW][PP], nq[KNN_QW], err[KNN_QW], keep[KNN_QW];
  int cnt[KNN_QW], ncq[KNN_QW];
  bool live[KNN_QW];
  const float rmax = sqrtf(__uint_as_float(*maxn2_bits)) * 1.0001f;
  const float inf = __int_as_float(0x7f800000);
  bool any = false;
#pragma unroll
  for (int a = 0; a < KNN_QW; ++a) {
    int64_t q = q0 + a;
    live[a] = q < M;
    // redo pass: only the locations whose pilot threshold failed its check
    if (redo && live[a]) live[a] = cnt_out[q] < 0;
    any = any || live[a];
    float acc = 0.f;
#pragma unroll
    for (int k = 0; k < PP; ++k) {
      float v = 0.f;
      if (live[a] && k < p) v = (float)(xref[q * p + k] - center[k]);
      qf[a][k] = v;
      acc = fmaf(v, v, acc);
    }
    nq[a] = acc;
    float r = rmax + sqrtf(acc) * 1.0001f;
    err[a] = (float)(p + 12) * 0x1p-24f * 1.25f * r * r;
    const float thr = (live[a] && pilot) ? pilot[q] : inf;
    keep[a] = live[a] ? (thr < inf ? __fadd_ru(thr, 2.f * err[a]) : inf) : -1.f;
    cnt[a] = 0;
    ncq[a] = live[a] ? (nc_loc ? nc_loc[q] : nc_max) : 0;
  }
  if (!__syncthreads_or(any)) return;   // a redo pass with nothing to redo here

  const uint32_t tile_bytes = LAGP_KNN_TILE * PP * sizeof(float);
  const uint32_t norm_bytes = LAGP_KNN_TILE * sizeof(float);
  if (threadIdx.x == 0) {
    mbar_init(&bar[0], 1);
    mbar_init(&bar[1], 1);
    fence_mbar_init();
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int s = 0; s < 2 && s < ntiles; ++s) {
      mbar_expect_tx(&bar[s], tile_bytes + norm_bytes);
      bulk_g2s(tile + s * LAGP_KNN_TILE * PP, Xf + (int64_t)s * LAGP_KNN_TILE * PP, tile_bytes, &bar[s]);
      bulk_g2s(tnorm + s * LAGP_KNN_TILE, nx + (int64_t)s * LAGP_KNN_TILE, norm_bytes, &bar[s]);
    }
  }

  bool timed_out = false;
  for (int64_t t = 0; t < ntiles; ++t) {
    const int st = (int)(t & 1);
    if (!mbar_wait(&bar[st], (uint32_t)((t >> 1) & 1))) {
      timed_out = true;
    }
    if (__syncthreads_or(timed_out)) {
      if (threadIdx.x == 0) {
        atomicOr(status, LAGP_DEV_TIMEOUT);
        // drain the copies still in flight into this CTA's buffers (bounded)
        mbar_wait(&bar[st], (uint32_t)((t >> 1) & 1));
        if (t + 1 < ntiles) mbar_wait(&bar[st ^ 1], (uint32_t)(((t + 1) >> 1) & 1));
      }
      __syncthreads();
      break;
    }
    const float* T = tile + st * LAGP_KNN_TILE * PP;
    const float* TN = tnorm + st * LAGP_KNN_TILE;
    const int64_t base = t * LAGP_KNN_TILE;
#pragma unroll 1
    for (int s = 0; s < LAGP_KNN_TILE / 32; ++s) {
      const int pt = s * 32 + lane;
      const int64_t gi = base + pt;
      float xv[PP];
#pragma unroll
      for (int k = 0; k < PP; k += 4) {
        float4 v4 = *reinterpret_cast<const float4*>(T + pt * PP + k);
        xv[k] = v4.x; xv[k + 1] = v4.y; xv[k + 2] = v4.z; xv[k + 3] = v4.w;
      }
      const float nxp = TN[pt];
      float d[KNN_QW];
#pragma unroll
      for (int a = 0; a < KNN_QW; ++a) {
        float dot = 0.f;
#pragma unroll
        for (int k = 0; k < PP; ++k) dot = fmaf(qf[a][k], xv[k], dot);
        d[a] = fmaf(-2.f, dot, nq[a] + nxp);
      }
#pragma unroll
      for (int a = 0; a < KNN_QW; ++a) {
        const bool pass = d[a] <= keep[a];
        uint32_t m = __ballot_sync(0xffffffffu, pass);
        if (m) {
          int pos = cnt[a] + __popc(m & ((1u << lane) - 1u));
          if (pass && pos < cap) {
            KnnEntry e; e.d = fmaxf(d[a], 0.f); e.idx = (int32_t)gi;
            buf[(q0 + a) * (int64_t)cap + pos] = e;
          }
          cnt[a] += __popc(m);
        }
      }
    }
    // compact any buffer that the next tile could overflow
#pragma unroll
    for (int a = 0; a < KNN_QW; ++a) {
      if (live[a] && cnt[a] > cap - LAGP_KNN_TILE) {
        KnnEntry* e = buf + (q0 + a) * (int64_t)cap;
        int c = min(cnt[a], cap);
        if (cnt[a] > cap) atomicOr(status, LAGP_DEV_KNN_OVERFLOW);
        __syncwarp();
        uint32_t kb = warp_select_kth(e, c, ncq[a], hist + warp * 256);
        float kth = __uint_as_float(kb);
        keep[a] = fminf(keep[a], __fadd_ru(kth, 2.f * err[a]));
        cnt[a] = warp_compact(e, c, keep[a]);
        if (cnt[a] > cap - LAGP_KNN_TILE && lane == 0) atomicOr(status, LAGP_DEV_KNN_OVERFLOW);
      }
    }
    __syncthreads();  // every warp is done with stage st
    if (threadIdx.x == 0 && t + 2 < ntiles) {
      mbar_expect_tx(&bar[st], tile_bytes + norm_bytes);
      bulk_g2s(tile + st * LAGP_KNN_TILE * PP, Xf + (t + 2) * LAGP_KNN_TILE * PP, tile_bytes, &bar[st]);
      bulk_g2s(tnorm + st * LAGP_KNN_TILE, nx + (t + 2) * LAGP_KNN_TILE, norm_bytes, &bar[st]);
    }
  }
  // final: keep d32 <= (N'-th smallest) + 2 err
#pragma unroll
  for (int a = 0; a < KNN_QW; ++a) {
    if (!live[a]) continue;
    KnnEntry* e = buf + (q0 + a) * (int64_t)cap;
    int c = min(cnt[a], cap);
    __syncwarp();
    const float thr = pilot ? pilot[q0 + a] : inf;
    if (thr < inf) {
      // the pilot threshold holds if at least N' buffered points lie at or below it
      int below = 0;
      for (int i = lane; i < c; i += 32) below += (e[i].d <= thr) ? 1 : 0;
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) below += __shfl_xor_sync(0xffffffffu, below, o);
      if (below < ncq[a]) {
        if (lane == 0) cnt_out[q0 + a] = -1;   // stream this location again
        continue;
      }
    }
    if (c >= ncq[a] && ncq[a] > 0) {
      uint32_t kb = warp_select_kth(e, c, ncq[a], hist + warp * 256);
      c = warp_compact(e, c, __fadd_ru(__uint_as_float(kb), 2.f * err[a]));
    }
    if (lane == 0) cnt_out[q0 + a] = timed_out ? 0 : c;
  }
}

// ---------------------------------------------------------------------------
// Exact ranking: the candidates in the order of (binary64 distance in the
// oracle's order of operations, index), the first N' of them out.
//
// The binary64 distances of every survivor were most of this kernel (24 FP64
// instructions a pair at p = 8, on GB300's narrow FP64 pipe), and few of them
// decide anything: the order of two points is known from binary32 distances
// unless these lie within their error bounds.  So the pairs (binary32 distance,
// index) are sorted as one 64-bit word each, neighbours closer than their bounds
// are joined into runs, and only the members of runs (a few per cent) get
// their binary64 distance and are ranked within their run by counting.  The
// bound grows with the distance, so the cut between two runs separates
// everything below from everything above.  Runs longer than RANK_RUN (designs
// with many equal distances) then sort all the (distance, index) pairs, the members
// of runs by their binary64 distances; values that leave binary32's range sort the
// (binary64 distance, index) pairs at once; all give the one order.  100,000
// locations, p = 8, N' = 1000: 3.33 ms, 6.12 with all distances in binary64;
// 10,000 locations, p = 4, N' = 200: 0.06 against 0.42 ms (a network of 1024
// whatever the list's length).
//
// Sorts are bitonic.  Up to 2048 pairs are held in registers, E per thread
// (element E t + u on thread t): strides below E inside a thread, then between
// the lanes of a warp by shuffles, the largest through shared memory.  Distances
// are non-negative, so their IEEE bit patterns order like the values.
// ---------------------------------------------------------------------------
#define RANK_RUN 64

// Sorts the T * E words (WIDE: pairs of a word and an index) in kr (and ir); key
// and idx: shared memory for as many entries.  With one element per thread only
// the first `size` of them (a power of two) go through the network; the others
// are the largest word.
template <int T, int E, bool WIDE>
__device__ __forceinline__ void rank_sort(unsigned long long (&kr)[E], int32_t (&ir)[E],
                                          unsigned long long* key, int32_t* idx, int size) {
  const int t = threadIdx.x;
  const int last = E == 1 ? size : T * E;
  auto less = [](unsigned long long ka, int32_t ia, unsigned long long kb, int32_t ib) {
    return WIDE ? (ka < kb || (ka == kb && ia < ib)) : ka < kb;
  };
#pragma unroll 1
  for (int k = 2; k <= last; k <<= 1) {
#pragma unroll 1
    for (int jj = k >> 1; jj >= E; jj >>= 1) {
      const int x = jj / E, pt = t ^ x;    // the partner thread, same u
      if (x >= 32) {                       // another warp: through shared memory
        __syncthreads();
#pragma unroll
        for (int u = 0; u < E; ++u) {
          key[u * T + t] = kr[u];
          if (WIDE) idx[u * T + t] = ir[u];
        }
        __syncthreads();
      }
#pragma unroll
      for (int u = 0; u < E; ++u) {
        const int i = E * t + u;
        // the lower element of an ascending pair (or the upper of a descending
        // one) keeps the smaller
        const bool keep_min = ((i & jj) == 0) == ((i & k) == 0);
        unsigned long long pk;
        int32_t pi = 0;
        if (x >= 32) {
          pk = key[u * T + pt];
          if (WIDE) pi = idx[u * T + pt];
        } else {
          pk = __shfl_xor_sync(0xffffffffu, kr[u], x);
          if (WIDE) pi = __shfl_xor_sync(0xffffffffu, ir[u], x);
        }
        if (less(pk, pi, kr[u], ir[u]) == keep_min) { kr[u] = pk; ir[u] = pi; }
      }
    }
#pragma unroll
    for (int J = E / 2; J > 0; J >>= 1) {  // inside the thread, constant registers
      if (J < k) {
#pragma unroll
        for (int u = 0; u < E; ++u) {
          if (u & J) continue;
          const bool up = ((E * t + u) & k) == 0;
          if (less(kr[u | J], ir[u | J], kr[u], ir[u]) == up) {
            const unsigned long long tk = kr[u]; kr[u] = kr[u | J]; kr[u | J] = tk;
            const int32_t ti = ir[u]; ir[u] = ir[u | J]; ir[u | J] = ti;
          }
        }
      }
    }
  }
  __syncthreads();
}

// Bound on |d - D| for D the exact squared distance and d the binary32 one from
// coordinates rounded to binary32 about the centre (relative error u = 2^-24
// each, so at most u (|a| + |q|) on the difference, with |a| <= |q| + sqrt(d)):
// 2 u sqrt(d) (2|q| + sqrt(d)) from the rounded inputs, (p + 4) u d from the
// arithmetic, both with 25%, the square of the input error, and what
// underflow can lose.  The binary64 distance's own error is far below the 25%.
__device__ __forceinline__ float rank_err(float d, float qn, int p) {
  const float u = 0x1p-24f, r = sqrtf(d), s = 2.f * qn + r;
  return 1.25f * u * (2.f * r * s + (float)(p + 4) * d) + 4.f * (u * s) * (u * s) + 1e-36f;
}

template <int MAX>
struct RankRuns {
  uint32_t joined[MAX / 32];   // bit i: element i joins i - 1
  uint16_t list[MAX];          // the members of runs
  int nlist;
};

// c <= T * E survivors, at least nc of them
template <int T, int E, typename Runs>
__device__ void rank_location(const double* __restrict__ X, const float* __restrict__ Xf, int p,
                              int PP, const double* xq, const float* qf, float qn,
                              const KnnEntry* __restrict__ e, int c, int nc,
                              unsigned long long* key, int32_t* idx, Runs& runs,
                              int32_t* __restrict__ out) {
  uint32_t* joined = runs.joined;
  uint16_t* list = runs.list;
  const int t = threadIdx.x;
  unsigned long long kr[E];
  int32_t ir[E];
  bool wide = false;
#pragma unroll
  for (int u = 0; u < E; ++u) {
    const int i = E * t + u;
    kr[u] = ~0ull;
    ir[u] = 0;
    if (i < c) {
      const int32_t gi = e[i].idx;
      const float4* x = reinterpret_cast<const float4*>(Xf + (int64_t)gi * PP);
      float d = 0.f;
      for (int k = 0; k < PP / 4; ++k) {
        const float4 v = __ldg(x + k);
        const float a = v.x - qf[4 * k], b = v.y - qf[4 * k + 1];
        const float g = v.z - qf[4 * k + 2], h = v.w - qf[4 * k + 3];
        d = fmaf(a, a, d);
        d = fmaf(b, b, d);
        d = fmaf(g, g, d);
        d = fmaf(h, h, d);
      }
      wide |= !(d < 1e36f);
      kr[u] = ((unsigned long long)__float_as_uint(d) << 32) | (uint32_t)gi;
    }
  }
  int size = T;                        // (E > 1: the whole network)
  if (E == 1)
    while (size > 2 && size / 2 >= c) size >>= 1;
  if (t < T * E / 32) joined[t] = 0u;
  if (t == 0) runs.nlist = 0;
  if (!__syncthreads_or(wide || !(qn < 1e18f))) {
    rank_sort<T, E, false>(kr, ir, key, idx, size);
#pragma unroll
    for (int u = 0; u < E; ++u) {
      key[E * t + u] = kr[u];
      idx[E * t + u] = (int32_t)(uint32_t)kr[u];
    }
    __syncthreads();
    uint32_t bits = 0u;
    float before = t > 0 ? __uint_as_float((uint32_t)(key[E * t - 1] >> 32)) : 0.f;
#pragma unroll
    for (int u = 0; u < E; ++u) {
      const int i = E * t + u;
      const float d = __uint_as_float((uint32_t)(kr[u] >> 32));
      if (i > 0 && i < c && d - before <= 2.002f * rank_err(d, qn, p)) bits |= 1u << u;
      before = d;
    }
    if (bits) atomicOr(&joined[E * t >> 5], bits << (E * t & 31));
    __syncthreads();
    auto joins = [&](int i) { return i < c && (joined[i >> 5] >> (i & 31) & 1u) != 0u; };
#pragma unroll
    for (int u = 0; u < E; ++u) {
      const int i = E * t + u;
      if (i >= c) continue;
      if (joins(i) || joins(i + 1)) list[atomicAdd(&runs.nlist, 1)] = (uint16_t)i;
      else if (i < nc) out[i] = (int32_t)(uint32_t)kr[u];
    }
    __syncthreads();
    const int nl = runs.nlist;
    for (int l = t; l < nl; l += T) {
      const int i = list[l];
      key[i] = (unsigned long long)__double_as_longlong(sqdist64(X + (int64_t)idx[i] * p, xq, p));
    }
    __syncthreads();
    for (int l = t; l < nl; l += T) {
      const int i = list[l];
      int a = i, b = i + 1;
      while (b - a <= RANK_RUN && joins(a)) --a;
      while (b - a <= RANK_RUN && joins(b)) ++b;
      if (b - a > RANK_RUN) { wide = true; continue; }
      int at = a;
      for (int m = a; m < b; ++m)
        at += (key[m] < key[i] || (key[m] == key[i] && idx[m] < idx[i])) ? 1 : 0;
      if (at < nc) out[at] = idx[i];
    }
    if (!__syncthreads_or(wide)) return;
    // a run too long: all pairs, the members of runs with the distances they have
    // and the others with the binary32 one, which is on the right side of every cut
#pragma unroll
    for (int u = 0; u < E; ++u) {
      const int i = E * t + u;
      ir[u] = i < c ? (int32_t)(uint32_t)kr[u] : 0x7fffffff;
      if (joins(i) || joins(i + 1)) kr[u] = key[i];
      else if (i < c)
        kr[u] = (unsigned long long)__double_as_longlong((double)__uint_as_float((uint32_t)(kr[u] >> 32)));
    }
    __syncthreads();
  } else {
#pragma unroll
    for (int u = 0; u < E; ++u) {
      const int i = E * t + u;
      kr[u] = ~0ull;
      ir[u] = 0x7fffffff;
      if (i < c) {
        ir[u] = e[i].idx;
        kr[u] = (unsigned long long)__double_as_longlong(sqdist64(X + (int64_t)ir[u] * p, xq, p));
      }
    }
  }
  rank_sort<T, E, true>(kr, ir, key, idx, size);
#pragma unroll
  for (int u = 0; u < E; ++u)
    if (E * t + u < nc) out[E * t + u] = ir[u];
}

// T = 256 threads for lists of any length; T = 128 for short ones (rank_threads)
template <int T>
__global__ void __launch_bounds__(T, T == 128 ? 12 : 4)
knn_rank(const double* __restrict__ X, const float* __restrict__ Xf, int p, int PP,
         const double* __restrict__ xref, const double* __restrict__ center, int64_t M,
         int nc_max, const int32_t* __restrict__ nc_loc, int cap,
         const KnnEntry* __restrict__ buf, const int32_t* __restrict__ cnt,
         int32_t* __restrict__ cand /*[M][nc_max]*/, unsigned* __restrict__ status) {
  extern __shared__ __align__(128) unsigned char smem_rank[];
  const int64_t q = blockIdx.x;
  if (q >= M) return;
  const int c = cnt[q];
  const int nc = nc_loc ? nc_loc[q] : nc_max;
  unsigned long long* key = reinterpret_cast<unsigned long long*>(smem_rank);
  int32_t* idx = reinterpret_cast<int32_t*>(key + cap);
  int32_t* out = cand + q * nc_max;
  __shared__ double xq[LAGP_MAX_P];
  __shared__ float qf[LAGP_MAX_P];
  constexpr int MAX = T == 128 ? 512 : 2048;
  __shared__ RankRuns<MAX> runs;
  if (threadIdx.x < p) xq[threadIdx.x] = xref[q * p + threadIdx.x];
  if (threadIdx.x < PP)
    qf[threadIdx.x] =
        threadIdx.x < p ? (float)(xref[q * p + threadIdx.x] - center[threadIdx.x]) : 0.f;
  __syncthreads();
  const KnnEntry* e = buf + q * (int64_t)cap;
  if (c >= nc && c <= MAX) {
    float qn = 0.f;
    for (int k = 0; k < p; ++k) qn = fmaf(qf[k], qf[k], qn);
    qn = sqrtf(qn) * 1.0001f;
    if (c <= T) rank_location<T, 1>(X, Xf, p, PP, xq, qf, qn, e, c, nc, key, idx, runs, out);
    else if (c <= 2 * T) rank_location<T, 2>(X, Xf, p, PP, xq, qf, qn, e, c, nc, key, idx, runs, out);
    else if (T == 128 || c <= 4 * T)
      rank_location<T, 4>(X, Xf, p, PP, xq, qf, qn, e, c, nc, key, idx, runs, out);
    else
      rank_location<T, MAX / T>(X, Xf, p, PP, xq, qf, qn, e, c, nc, key, idx, runs, out);
    for (int r = nc + threadIdx.x; r < nc_max; r += blockDim.x) out[r] = -1;
    return;
  }
  int sz = 1;
  while (sz < c) sz <<= 1;
  for (int i = threadIdx.x; i < sz; i += blockDim.x) {
    if (i < c) {
      int32_t gi = e[i].idx;
      key[i] = (unsigned long long)__double_as_longlong(sqdist64(X + (int64_t)gi * p, xq, p));
      idx[i] = gi;
    } else {
      key[i] = ~0ull;
      idx[i] = 0x7fffffff;
    }
  }
  __syncthreads();
  for (int k = 2; k <= sz; k <<= 1) {
    for (int jj = k >> 1; jj > 0; jj >>= 1) {
      for (int t = threadIdx.x; t < (sz >> 1); t += blockDim.x) {
        // t-th compare-exchange pair of this stage
        const int i = ((t & ~(jj - 1)) << 1) | (t & (jj - 1));
        const int l = i | jj;
        const bool up = (i & k) == 0;
        const unsigned long long ki = key[i], kl = key[l];
        const int32_t ii = idx[i], il = idx[l];
        const bool gt = (ki > kl) || (ki == kl && ii > il);
        if (gt == up) {
          key[i] = kl; key[l] = ki;
          idx[i] = il; idx[l] = ii;
        }
      }
      __syncthreads();
    }
  }
  if (c < nc && threadIdx.x == 0) atomicOr(status, LAGP_DEV_KNN_OVERFLOW);
  // ranks this location lacks (a flagged overflow or timeout) repeat a valid
  // index, so that the design kernels never read outside the design
  const int32_t fill = c > 0 ? idx[0] : 0;
  for (int r = threadIdx.x; r < nc_max; r += blockDim.x)
    out[r] = (r < nc) ? (r < c ? idx[r] : fill) : -1;
}

// ---------------------------------------------------------------------------
// Host-side launchers.
// ---------------------------------------------------------------------------
size_t knn_smem_stream(int PP) {
  return (size_t)2 * LAGP_KNN_TILE * PP * 4 + 2 * LAGP_KNN_TILE * 4 + KNN_WARPS * 256 * 4 + 16;
}

// Pilot thresholds pay where the design is large against N' and the stream forms
// distances enough to be worth the 30 us of the pilot and the empty redo; the line
// lies between the sides measured.  Streams without and with them (pilot and
// redo included): 5,000 locations at p = 8, N = 2 N' (4000) 321 us against 313,
// N = 4 N' (4000) 567 against 240, N = 8 N' (1024) 128 against 104; at p = 4, 8
// locations, N = 8 N': 60 against 69 us at 1024, 80 against 83 at 2000, 142
// against 107 at 4000; one location, N = 16 N': 92 against 97 us at 8000, 169
// against 150 at 16000.
static bool knn_has_pilot(int64_t N, int64_t M, int nc_max) {
  return knn_uses_tc(N, nc_max) || (knn_mid(N, nc_max) && M * N >= 16384);
}

cudaError_t launch_prepare(const double* X, int64_t N, int p, int PP, int64_t Npad,
                           const Workspace& ws, cudaStream_t s) {
  const int parts = 64;
  prof_begin("bbox_partial", s);
  bbox_partial<<<parts, 256, 0, s>>>(X, N, p, ws.bbox_part);
  prof_end(s);
  prof_begin("bbox_final", s);
  bbox_final<<<1, 32, 0, s>>>(ws.bbox_part, parts, p, ws.lo, ws.hi, ws.center);
  prof_end(s);
  cudaMemsetAsync(ws.maxn2, 0, sizeof(unsigned), s);
  prof_begin("design_to_f32", s);
  design_to_f32<<<1216, 256, 0, s>>>(X, N, Npad, p, PP, ws.center, ws.Xf, ws.nx, ws.maxn2);
  prof_end(s);
  cudaError_t err = cudaGetLastError();
  if (err != cudaSuccess) return err;
  if ((err = launch_design_to_tc(N, p, PP, Npad, ws, s)) != cudaSuccess) return err;
  // the k-d tree of the unlimited ray scope, when the workspace has one
  return ws.kd.perm ? launch_kd_build(X, ws.Xf, N, p, PP, ws.kd, s) : cudaSuccess;
}

cudaError_t launch_knn(const double* X, int64_t N, int p, int PP, int64_t Npad,
                       const double* xref, int64_t M, int nc_max, const int32_t* nc_loc,
                       int cap, int32_t* cand, const Workspace& ws, cudaStream_t s) {
  const int64_t ntiles = Npad / LAGP_KNN_TILE;
  const int qpb = KNN_WARPS * KNN_QW;
  dim3 grid((unsigned)((M + qpb - 1) / qpb));
  size_t sm = knn_smem_stream(PP);
  const bool tc = knn_uses_tc(N, nc_max), pilot = knn_has_pilot(N, M, nc_max);
  const int64_t S = knn_sample(N);
  KnnEntry* kbuf = reinterpret_cast<KnnEntry*>(ws.knn_buf);
  // buffers that are larger for the threshold's sake: what the tensor-core filter
  // may admit to them, in sample rows
  const bool check = tc && cap > knn_cap_least(nc_max);
  const float errc = kt_err_factor(kt_ka(p));
  const int fit = (int)((cap - 2 * LAGP_KNN_TILE) * S / N);
  cudaError_t err;
  int dev = 0, sms = 0;
  if ((err = cudaGetDevice(&dev)) != cudaSuccess) return err;
  if ((err = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess)
    return err;
  const bool alone = knn_pilot_alone(M, S, PP, sms);
  switch (PP) {
#define KNN_CASE(V)                                                                          \
  case V:                                                                                    \
    err = cudaFuncSetAttribute(knn_stream<V>, cudaFuncAttributeMaxDynamicSharedMemorySize,   \
                               (int)sm);                                                     \
    if (err != cudaSuccess) return err;                                                      \
    if (pilot) {                                                                             \
      prof_begin("knn_pilot", s);                                                            \
      if (alone)                                                                             \
        (check ? knn_pilot1<V, true> : knn_pilot1<V, false>)                                 \
            <<<(unsigned)M, KNN_PILOT1_THREADS, 0, s>>>(ws.Xf, ws.nx, N, S, p, xref, M,      \
                                                        ws.center, nc_max, nc_loc, cap,      \
                                                        errc, fit, ws.maxn2, ws.knn_thr);    \
      else                                                                                   \
        (check ? knn_pilot<V, true> : knn_pilot<V, false>)                                   \
            <<<grid, KNN_WARPS * 32, 0, s>>>(ws.Xf, ws.nx, N, S, p, xref, M, ws.center,      \
                                             nc_max, nc_loc, cap, errc, fit, ws.maxn2,       \
                                             ws.knn_thr);                                    \
      prof_end(s);                                                                           \
    }                                                                                        \
    if (tc) {                                                                                \
      err = launch_knn_tc(Npad, p, xref, M, nc_max, nc_loc, cap, ws, s);                     \
      if (err != cudaSuccess) return err;                                                    \
    } else {                                                                                 \
      prof_begin("knn_stream", s);                                                           \
      knn_stream<V><<<grid, KNN_WARPS * 32, sm, s>>>(ws.Xf, ws.nx, N, ntiles, p, xref, M,    \
                                                     ws.center, ws.maxn2, nc_max, nc_loc,    \
                                                     cap, kbuf, ws.knn_cnt, ws.status,       \
                                                     pilot ? ws.knn_thr : nullptr, 0);       \
      prof_end(s);                                                                           \
    }                                                                                        \
    if (pilot) {                                                                             \
      prof_begin("knn_stream_redo", s);                                                      \
      knn_stream<V><<<grid, KNN_WARPS * 32, sm, s>>>(ws.Xf, ws.nx, N, ntiles, p, xref, M,    \
                                                     ws.center, ws.maxn2, nc_max, nc_loc,    \
                                                     cap, kbuf, ws.knn_cnt, ws.status,       \
                                                     nullptr, 1);                            \
      prof_end(s);                                                                           \
    }                                                                                        \
    break;
    KNN_CASE(4)
    KNN_CASE(8)
    KNN_CASE(12)
    KNN_CASE(16)
#undef KNN_CASE
    default:
      return cudaErrorInvalidValue;
  }
  size_t smr = (size_t)cap * (8 + 4);
  const int threads = rank_threads(nc_max);
  auto rank = threads == 128 ? knn_rank<128> : knn_rank<256>;
  err = cudaFuncSetAttribute(rank, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smr);
  if (err != cudaSuccess) return err;
  prof_begin("knn_rank", s);
  rank<<<(unsigned)M, threads, smr, s>>>(
      X, ws.Xf, p, PP, xref, ws.center, M, nc_max, nc_loc, cap,
      reinterpret_cast<const KnnEntry*>(ws.knn_buf), ws.knn_cnt, cand, ws.status);
  prof_end(s);
  return cudaGetLastError();
}

}  // namespace lagp
