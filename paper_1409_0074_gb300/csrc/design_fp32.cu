// design_fp32.cu -- exhaustive greedy local design with FP32 candidate scoring
// and an FP64 factor update, one CTA per predictive location: the exhaustive
// search of the LAGP_FP32_SCORE form for every n, and of LAGP_FP32_SCORE_TC
// for the designs larger than its tensor-core scorer (exh_tc.cu) takes.  The
// ray search of these forms is in ray32.cu.
//
// Scoring form.  With K_j = L_j L_j^T (Cholesky) the ALC integrand of Eq. alc
// (sign reading as in the FP64 path) becomes
//     w = L_j^{-1} k_j(x'),  v = (1 + g) - |w|^2,
//     ALC(x') = (w . z - K(x', x))^2 / v,   z = L_j^{-1} k_j(x),
// the same quadratic forms as k^T K^{-1} k, evaluated through the inverse
// factor.  In FP32 this keeps the error of v near eps * sqrt(cond K) instead of
// eps * cond K: on the 8-d, N = 1e6 workload (cond K_50 ~ 1e6, v ~ 1e-4) an
// explicit-inverse FP32 score has errors as large as v itself, while the
// factored score stays near 5e-6.
//
// FP64 state (the partitioned update, Sec 2.2, in factored form): appending
// x_new with l = L_j^{-1} k_j(x_new), v = (1 + g) - |l|^2 (the Schur complement
// of the paper's update), d = sqrt(v) gives
//     L_{j+1}^{-1} = [[L_j^{-1}, 0], [-(L_j^{-T} l)^T / d, 1 / d]],
// so one new row per step, O(j^2).  z and L^{-1} y grow by one entry per step
// and the predictive equations (Eq. predgp, preds2) follow as
//     mu = z . (L^{-1} y),  psi = |L^{-1} y|^2,  sigma^2 = psi (1 + g - |z|^2) / n.
//
// Incremental scores.  Because the inverse factor only gains a row, every
// candidate's w (and z) only gains an entry per step: w_cj = row_j . K(S, c).
// Each CTA keeps |w_c|^2 and w_c . z as running sums per candidate, so a step
// costs O(N' j) instead of the O(N' j^2) of re-forming every w, and a full
// design O(N' n^2) instead of O(N' n^3); the sums see the same FP32 operations
// in the same order as a from-scratch evaluation would.
// Each step is a chain (new point -> correlations -> new row -> every
// candidate's entry -> argmax) that waits on binary64 latency, barriers and
// the cache in L2, so the chain is kept short: the packed factor lies in shared
// memory (n <= 64), a row's product with the new correlations takes four lanes
// and a column sum two (one per accumulator), the new row's terms of z and
// L^{-1} y come from the threads that formed it, and a thread reads the cached
// rows of four neighbouring candidates in 128-bit loads, eight rows at a time.
// 25.7 against 35.0 ms per 20,000 locations (8-d, n = 50, N' = 1000) with the
// factor in global memory, one lane per row and column and 32-bit loads.  Four
// CTAs of 256 threads per SM keep the slots' caches near the size of L2: five
// ran 26.8 ms, five or seven of 128 threads 26.8 and 34.1 ms.  Up to N' = 512, where
// the caches are small, most calls take eight of 128 threads (d32_threads).
// Scoring coordinates are FP32 and centred on the design's bounding box.
#include <cstdint>

#include "common.cuh"
#include "lagp_internal.h"

namespace lagp {

#define D32_WARPS 8        // of the largest block (d32_threads)
// row stride of the correlation cache and of the per-candidate arrays: four
// candidates at a time
#define D32_LDC(nc) (((nc) + 3) & ~3)

struct D32Params {
  const double* X;
  const double* Y;
  int p, PP;
  const float* Xf;       // centred FP32 design [Npad][PP]
  const double* xref;
  int64_t M;
  const int32_t* cand;
  int nc_max;
  const int32_t* nc_loc;
  int n0, n_max;
  const int32_t* n_loc;
  double theta, g;
  const double* theta_loc;   // per-location lengthscale [M] or null
  const double* center;
  double* mean;
  double* s2;
  int32_t* selected;
  double* tie_gap;
  int32_t* nevals;
  double* Linv;          // [slots][n_max][n_max] FP64 inverse factor
  float* Kc;             // exhaustive: [slots][n_max][nc_max] FP32 correlation cache
  float* crow;           // [slots][nc_max][PP] the location's candidates' FP32 rows
  unsigned* status;
  unsigned* queue;       // work counter (zero at launch)
  const int32_t* order;  // item -> location, or null
  const unsigned* count; // items (device), or null (M)
  int32_t* promote;      // binary64 re-solve list, or null (promotion off)
  unsigned* promote_count;
};

struct L32 {
  float* Lf;       // [n_max] FP32 copy of the newest row of L^{-1}
  float* zf;       // [n_max]
  float* Sf;       // [n_max][PP] centred FP32 selected coordinates
  float* xf;       // [PP]
  float* vs;       // [nc_max] running |w_c|^2 of every candidate
  float* ns;       // [nc_max] running w_c . z
  float* kxc;      // [nc_max] K(c, x)
  float* red;      // [WARPS*4]
  double* S64;     // [n_max][p]
  double* xq;      // [p]
  double* kvec;    // [n_max]
  double* l;       // [n_max]
  double* ys;      // [n_max] y of the selected points
  double* tz;      // [n_max] the new row's terms of z_j
  double* ty;      // [n_max] and of (L^{-1} y)_j
  double* z;       // [n_max]
  double* zy;      // [n_max]
  double* kx;      // [n_max]
  double* dred;    // [WARPS*4]
  int* sel;        // [n_max]
  int* ired;       // [WARPS*2]
  unsigned char* used;
  int j;
  float neg_inv_theta, onepg;
};

// -1 / lengthscale of the CTA's current location (kept out of the registers,
// and divided once per location: a binary64 division by every warp of every
// step was more than a third of the kernel's binary64 work)
static __shared__ double d32_nit64;

// start of row i of the packed inverse factor
__device__ __host__ __forceinline__ int d32_tri(int i) { return i * (i + 1) / 2; }

__device__ __forceinline__ double warp_sumd(double v) {
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}
// Sums over the warp's first `active` values of a shared vector pair, each
// added up as blocks of 32 (a butterfly per block, the block totals in order):
// the sums sum_i a_i^2 (one vector) or sum_i a_i, sum_i b_i of two vectors.
// Every lane of the calling warp returns them.
__device__ __forceinline__ double sum_squares32(const double* a, int active) {
  const int lane = threadIdx.x & 31;
  double t = 0.0;
  for (int i0 = 0; i0 < active; i0 += 32) {
    const double x = i0 + lane < active ? a[i0 + lane] : 0.0;
    t += warp_sumd(__dmul_rn(x, x));     // (not contracted into the first addition)
  }
  return t;
}
__device__ __forceinline__ double sum_vector32(const double* a, int active) {
  const int lane = threadIdx.x & 31;
  double t = 0.0;
  for (int i0 = 0; i0 < active; i0 += 32)
    t += warp_sumd(i0 + lane < active ? a[i0 + lane] : 0.0);
  return t;
}

// best (value, index) over the block: larger value wins, ties to the lower index
struct VI { float v; int i; float v2; };
__device__ __forceinline__ VI vi_merge_max(VI a, VI b) {
  VI r;
  if (b.v > a.v || (b.v == a.v && b.i >= 0 && (a.i < 0 || b.i < a.i))) {
    r.v = b.v; r.i = b.i; r.v2 = fmaxf(a.v, b.v2);
  } else {
    r.v = a.v; r.i = a.i; r.v2 = fmaxf(a.v2, b.v);
  }
  return r;
}
template <int WARPS>
__device__ VI block_best(VI t, float* fs, int* is) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  for (int o = 16; o > 0; o >>= 1) {
    VI u;
    u.v = __shfl_xor_sync(0xffffffffu, t.v, o);
    u.i = __shfl_xor_sync(0xffffffffu, t.i, o);
    u.v2 = __shfl_xor_sync(0xffffffffu, t.v2, o);
    t = vi_merge_max(t, u);
  }
  if (lane == 0) { fs[2 * warp] = t.v; fs[2 * warp + 1] = t.v2; is[warp] = t.i; }
  __syncthreads();
  VI r; r.v = fs[0]; r.v2 = fs[1]; r.i = is[0];
  for (int w = 1; w < WARPS; ++w) {
    VI u; u.v = fs[2 * w]; u.v2 = fs[2 * w + 1]; u.i = is[w];
    r = vi_merge_max(r, u);
  }
  __syncthreads();
  return r;
}

// candidate rank r's FP32 row, from the slot's gathered copy
__device__ __forceinline__ const float* cand_f(const D32Params& P, const float* crow, int r) {
  return crow + (int64_t)r * P.PP;
}

// Append candidate rank r: FP64 factor row, z, L^{-1}y, FP32 copies, the
// correlation-cache row K(S_j, c) and entry j of every unselected candidate's w.
// `best` receives this thread's part of the next search: the ALC of every
// unselected candidate the thread updates, from the running sums it has just
// written (the same arithmetic and candidate order as a separate pass).
template <int THREADS>
__device__ bool add_point32(const D32Params& P, L32& L, const int32_t* cl, const float* crow,
                            int nc, int r, double* Lg, float* Kc_loc, VI* best) {
  const int tid = threadIdx.x, p = P.p, j = L.j, warp = tid >> 5;
  const double* c = P.X + (int64_t)cl[r] * p;
  if (tid < p) L.S64[j * p + tid] = c[tid];
  if (tid < P.PP) L.Sf[j * P.PP + tid] = cand_f(P, crow, r)[tid];
  if (tid == THREADS - 1) {
    L.ys[j] = P.Y[cl[r]];
    L.sel[j] = r;
    L.used[r] = 1;
  }
  __syncthreads();
  const double nit64 = d32_nit64;
  // correlations of the new point with the design, and with x (thread j)
  for (int i = tid; i <= j; i += THREADS) {
    const double kv = corr64_fast(i < j ? L.S64 + i * p : L.xq, L.S64 + j * p, p, nit64);
    if (i < j) L.kvec[i] = kv;
    else L.kx[j] = kv;
  }
  __syncthreads();
  // l = L_j^{-1} k_j(x_new): four lanes per row, each with every fourth product (the
  // first also with the remainder)
  for (int i = tid >> 2; i < ((j + 7) & ~7); i += THREADS / 4) {
    const int t = tid & 3, len = i + 1, len4 = len & ~3;
    const double* Li = Lg + d32_tri(i);
    double acc = 0.0;
    if (i < j) {
      for (int k = t; k < len4; k += 4) acc = fma(Li[k], L.kvec[k], acc);
      if (t == 0)
        for (int k = len4; k < len; ++k) acc = fma(Li[k], L.kvec[k], acc);
    }
    acc += __shfl_xor_sync(0xffffffffu, acc, 1);
    acc += __shfl_xor_sync(0xffffffffu, acc, 2);
    if (t == 0 && i < j) L.l[i] = acc;
  }
  __syncthreads();
  // the pivot v = 1 + g - |l|^2 and 1 / sqrt(v), on one warp
  double* piv = L.dred + 2 * D32_WARPS;
  if (warp == 0) {
    const double v = (1.0 + P.g) - sum_squares32(L.l, j);
    if (tid == 0) {
      piv[1] = v > 0.0 ? 1.0 / sqrt(v) : 0.0;
      L.ired[2 * D32_WARPS] = v > 0.0 ? 1 : 0;   // an integer for the other warps to test
    }
  }
  __syncthreads();
  if (!L.ired[2 * D32_WARPS]) return false;
  const double inv_d = piv[1];
  // the new row, and its terms of z_j = row_j . k(x) and (L^{-1} y)_j =
  // row_j . y_S: two lanes per column, one for its even rows and one for its
  // odd ones (the sum's two accumulators, in either order)
  double* Lj = Lg + d32_tri(j);
  for (int k = tid >> 1; k < ((j + 16) & ~15); k += THREADS / 2) {
    const int h = tid & 1;
    double acc = 0.0;
    if (k < j) {
      const double* Lk = Lg + k;
      for (int i = k + ((k ^ h) & 1); i < j; i += 2) acc = fma(L.l[i], Lk[d32_tri(i)], acc);
    }
    acc += __shfl_xor_sync(0xffffffffu, acc, 1);
    if (k <= j && h == 0) {
      const double rk = k < j ? -acc * inv_d : inv_d;
      Lj[k] = rk;
      L.Lf[k] = (float)rk;
      L.tz[k] = __dmul_rn(rk, L.kx[k]);
      L.ty[k] = __dmul_rn(rk, L.ys[k]);
    }
  }
  __syncthreads();
  // both sums side by side on two warps
  if (warp < 2) {
    const double t = sum_vector32(warp == 0 ? L.tz : L.ty, j + 1);
    if (tid == 0) {
      L.z[j] = t;
      L.zf[j] = (float)t;
    }
    if (tid == 32) L.zy[j] = t;
  }
  __syncthreads();
  // Row j of L^{-1} is final once written, so w_c = L^{-1} k_j(c) only gains
  // the entry w_cj = row_j . K(S_{0..j}, c); |w_c|^2 and w_c . z are running
  // sums in the order i = 0, 1, ..., the same FP32 operations a from-scratch
  // evaluation at every step would perform.  A thread owns four neighbouring
  // candidates, so that a row of their cached correlations is one 128-bit load
  // and eight rows' loads are in flight, and takes the newest entries from the
  // registers that computed them.  Even terms go to a0 and odd terms to a1, in
  // ascending order.
  const int64_t ldc = D32_LDC(P.nc_max);
  float* row = Kc_loc + (int64_t)j * ldc;
  const float* sj = L.Sf + j * P.PP;
  const float* Lfj = L.Lf;
  const float zj = L.zf[j];
  VI b;
  b.v = -1.f; b.v2 = -1.f; b.i = -1;
  for (int q = 4 * tid; q < nc; q += 4 * THREADS) {
    float kv[4];
#pragma unroll
    for (int u = 0; u < 4; ++u)
      kv[u] = __expf(sqdist_row32(cand_f(P, crow, min(q + u, nc - 1)), sj, P.PP) * L.neg_inv_theta);
    *reinterpret_cast<float4*>(row + q) = make_float4(kv[0], kv[1], kv[2], kv[3]);
    const float* kc = Kc_loc + q;
    float a0[4] = {0.f, 0.f, 0.f, 0.f}, a1[4] = {0.f, 0.f, 0.f, 0.f};
    int k = 0;
#pragma unroll 1
    for (; k + 8 <= j; k += 8) {
      float4 c[8];
#pragma unroll
      for (int t = 0; t < 8; ++t) c[t] = *reinterpret_cast<const float4*>(kc + (k + t) * ldc);
#pragma unroll
      for (int t = 0; t < 8; t += 2) {
        const float l0 = Lfj[k + t], l1 = Lfj[k + t + 1];
        a0[0] = fmaf(l0, c[t].x, a0[0]); a1[0] = fmaf(l1, c[t + 1].x, a1[0]);
        a0[1] = fmaf(l0, c[t].y, a0[1]); a1[1] = fmaf(l1, c[t + 1].y, a1[1]);
        a0[2] = fmaf(l0, c[t].z, a0[2]); a1[2] = fmaf(l1, c[t + 1].z, a1[2]);
        a0[3] = fmaf(l0, c[t].w, a0[3]); a1[3] = fmaf(l1, c[t + 1].w, a1[3]);
      }
    }
    if (k < j) {
      // the last rows (at most seven), loaded together; a missing one is zero
      float4 c[7];
#pragma unroll
      for (int t = 0; t < 7; ++t)
        c[t] = k + t < j ? *reinterpret_cast<const float4*>(kc + (k + t) * ldc)
                         : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
      for (int t = 0; t < 7; ++t) {
        if (k + t < j) {
          const float l = Lfj[k + t];
          float (&a)[4] = (t & 1) ? a1 : a0;
          a[0] = fmaf(l, c[t].x, a[0]); a[1] = fmaf(l, c[t].y, a[1]);
          a[2] = fmaf(l, c[t].z, a[2]); a[3] = fmaf(l, c[t].w, a[3]);
        }
      }
    }
    const float lj = Lfj[j];
    const bool odd = j & 1;
    float4 vs = *reinterpret_cast<const float4*>(L.vs + q);
    float4 ns = *reinterpret_cast<const float4*>(L.ns + q);
    const float4 kx = *reinterpret_cast<const float4*>(L.kxc + q);
    const uchar4 us = *reinterpret_cast<const uchar4*>(L.used + q);
    auto finish = [&](int u, float& v_, float& n_, float kx_, unsigned char used) {
      const float w = odd ? a0[u] + fmaf(lj, kv[u], a1[u]) : fmaf(lj, kv[u], a0[u]) + a1[u];
      v_ = fmaf(w, w, v_);
      n_ = fmaf(w, zj, n_);
      if (used || q + u >= nc) return;
      const float v = L.onepg - v_;
      const float num = n_ - kx_;
      const float alc = v > 0.f ? num * num / v : 0.f;
      if (alc > b.v) { b.v2 = b.v; b.v = alc; b.i = q + u; }
      else if (alc > b.v2) b.v2 = alc;
    };
    finish(0, vs.x, ns.x, kx.x, us.x);
    finish(1, vs.y, ns.y, kx.y, us.y);
    finish(2, vs.z, ns.z, kx.z, us.z);
    finish(3, vs.w, ns.w, kx.w, us.w);
    *reinterpret_cast<float4*>(L.vs + q) = vs;
    *reinterpret_cast<float4*>(L.ns + q) = ns;
  }
  *best = b;
  __syncthreads();
  L.j = j + 1;
  return true;
}

// ----- exhaustive search, CUDA-core FP32 scoring ---------------------------------
// ALC_c = (w_c . z - K(c, x))^2 / ((1 + g) - |w_c|^2) from the running sums;
// the largest score wins, ties to the lower candidate rank.  Each thread's part
// comes from the update loop of the last appended point (add_point32).
template <int THREADS>
__device__ int search_exh32(const L32& L, VI best, double* gap_out) {
  VI b = block_best<THREADS / 32>(best, L.red, L.ired);
  *gap_out = (b.v > 0.f && b.v2 >= 0.f) ? (double)((b.v - b.v2) / b.v) : 0.0;
  return b.i;
}

// PROMOTE: with precision promotion (a separate instantiation, so that the
// default one carries none of its code)
// SFACTOR: the packed factor in shared memory (d32_smem_factor), else in the
// slot's global scratch.  THREADS: 256 or 128 (d32_threads), 1,024 per SM.
template <bool PROMOTE, bool SFACTOR, int THREADS>
__global__ void __launch_bounds__(THREADS, 1024 / THREADS) design32(D32Params P) {
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ unsigned s_item;
  const int tid = threadIdx.x, p = P.p, PP = P.PP, ld = P.n_max;
  // scratch of this CTA slot
  const int ncp = D32_LDC(P.nc_max);
  float* Kc_loc = P.Kc + (int64_t)blockIdx.x * ld * ncp;
  float* crow = P.crow + (int64_t)blockIdx.x * P.nc_max * PP;

  L32 L;
  double* dp = reinterpret_cast<double*>(smem);
  L.S64 = dp; dp += ld * p;
  L.xq = dp; dp += p;
  L.kvec = dp; dp += ld;
  L.l = dp; dp += ld;
  L.ys = dp; dp += ld;
  L.tz = dp; dp += ld;
  L.ty = dp; dp += ld;
  L.z = dp; dp += ld;
  L.zy = dp; dp += ld;
  L.kx = dp; dp += ld;
  L.dred = dp; dp += 4 * D32_WARPS;
  double* Lg = SFACTOR ? dp : P.Linv + (int64_t)blockIdx.x * ld * ld;
  if (SFACTOR) dp += d32_tri(ld);
  // float4 arrays first, on a 16-byte boundary
  float* fp = reinterpret_cast<float*>((reinterpret_cast<uintptr_t>(dp) + 15) & ~(uintptr_t)15);
  L.vs = fp; fp += ncp;
  L.ns = fp; fp += ncp;
  L.kxc = fp; fp += ncp;
  L.used = reinterpret_cast<unsigned char*>(fp); fp += ncp / 4;
  L.Lf = fp; fp += ld;
  L.zf = fp; fp += ld;
  L.Sf = fp; fp += ld * PP;
  L.xf = fp; fp += PP;
  L.red = fp; fp += 4 * D32_WARPS;
  int* ip = reinterpret_cast<int*>(fp);
  L.sel = ip; ip += ld;
  L.ired = ip;
  L.onepg = (float)(1.0 + P.g);
  L.neg_inv_theta = (float)(-1.0 / P.theta);
  if (threadIdx.x == 0) d32_nit64 = -1.0 / P.theta;
  const unsigned items = P.count ? *P.count : (unsigned)P.M;
  for (;;) {
    if (tid == 0) s_item = atomicAdd(P.queue, 1u);
    __syncthreads();
    const unsigned it = s_item;
    __syncthreads();
    if (it >= items) break;
    const int64_t loc = P.order ? (int64_t)P.order[it] : (int64_t)it;
    const int nc = P.nc_loc ? P.nc_loc[loc] : P.nc_max;
    const int n = P.n_loc ? P.n_loc[loc] : P.n_max;
    const int32_t* cl = P.cand + loc * P.nc_max;
    L.j = 0;
    if (P.theta_loc) {
      const double th = P.theta_loc[loc];
      if (tid == 0) d32_nit64 = -1.0 / th;
      L.neg_inv_theta = (float)(-1.0 / th);
    }

    if (tid < p) L.xq[tid] = P.xref[loc * p + tid];
    if (tid < PP) L.xf[tid] = tid < p ? (float)(P.xref[loc * p + tid] - P.center[tid]) : 0.f;
    if (P.tie_gap) for (int i = tid; i < ld; i += THREADS) P.tie_gap[loc * ld + i] = 0.0;
    if (P.nevals) for (int i = tid; i < ld; i += THREADS) P.nevals[loc * ld + i] = 0;
    // the candidates' FP32 rows, gathered once into the slot in rank order
    for (int e = tid; e < nc * (PP >> 2); e += THREADS) {
      const int q = e / (PP >> 2), c4 = (e - q * (PP >> 2)) << 2;
      *reinterpret_cast<float4*>(crow + (int64_t)q * PP + c4) =
          *reinterpret_cast<const float4*>(P.Xf + (int64_t)cl[q] * PP + c4);
    }
    __syncthreads();
    for (int r = tid; r < nc; r += THREADS) {
      L.used[r] = 0;
      L.vs[r] = 0.f;
      L.ns[r] = 0.f;
      L.kxc[r] = __expf(sqdist_row32(cand_f(P, crow, r), L.xf, PP) * L.neg_inv_theta);
    }
    __syncthreads();

    bool ok = (n >= P.n0) && (n <= nc) && (n <= ld);
    VI part;
    for (int r = 0; r < P.n0 && ok; ++r) ok = add_point32<THREADS>(P, L, cl, crow, nc, r, Lg, Kc_loc, &part);
    for (int j = P.n0; j < n && ok; ++j) {
      double gap = 0.0;
      int ne = 0;
      int r = search_exh32<THREADS>(L, part, &gap);
      if (tid == 0) {
        if (P.tie_gap) P.tie_gap[loc * ld + (j - P.n0)] = gap;
        if (P.nevals) P.nevals[loc * ld + (j - P.n0)] = ne;
      }
      ok = (r >= 0) && add_point32<THREADS>(P, L, cl, crow, nc, r, Lg, Kc_loc, &part);
    }
    if (ok) {
      for (int i = tid; i < L.j; i += THREADS) L.tz[i] = __dmul_rn(L.z[i], L.zy[i]);
      __syncthreads();
      if (tid < 32) {
        const double a = sum_vector32(L.tz, L.j), b = sum_squares32(L.zy, L.j);
        const double c = sum_squares32(L.z, L.j);
        if (tid == 0) {
          P.mean[loc] = a;
          P.s2[loc] = b * ((1.0 + P.g) - c) / (double)L.j;
        }
      }
    } else if (tid == 0) {
      P.mean[loc] = __longlong_as_double(0x7ff8000000000000ll);
      P.s2[loc] = __longlong_as_double(0x7ff8000000000000ll);
      atomicOr(P.status, LAGP_DEV_BAD_UPDATE);
    }
    if (P.selected)
      for (int i = tid; i < ld; i += THREADS)
        P.selected[loc * ld + i] = (i < L.j) ? cl[L.sel[i]] : -1;
    if (PROMOTE && tid == 0) {
      // smallest binary64 pivot v of the design: the factor's diagonal holds
      // 1 / sqrt(v); a failed update promotes the location
      double vm = ok ? INFINITY : -1.0;
      for (int i = 0; i < L.j; ++i) {
        const double dg = Lg[d32_tri(i) + i];
        vm = fmin(vm, 1.0 / (dg * dg));
      }
      promote_location(P.promote, P.promote_count, loc, vm);
    }
  }
}

// The packed factor in shared memory while it leaves room for the CTAs that the
// registers allow; a larger one (up to 66 KB) would halve them.
static bool d32_smem_factor(int n_max) { return n_max <= 64; }

static size_t smem_design32(int n_max, int p, int PP, int nc_max) {
  size_t d = (size_t)n_max * p + p + 8 * n_max + 4 * D32_WARPS + (d32_smem_factor(n_max) ? d32_tri(n_max) : 0);
  const size_t ncp = D32_LDC(nc_max);
  size_t f = 2 * (size_t)n_max + (size_t)n_max * PP + PP + 3 * ncp + ncp / 4 + 4 * D32_WARPS;
  size_t i = (size_t)n_max + 2 * D32_WARPS + 2;
  return d * 8 + f * 4 + i * 4 + 16;
}

cudaError_t launch_exh32(const DesignArgs& a, cudaStream_t s) {
  D32Params P;
  P.X = a.X; P.Y = a.Y; P.p = a.p; P.PP = a.PP; P.Xf = a.ws->Xf; P.xref = a.xref; P.M = a.M;
  P.cand = a.cand; P.nc_max = a.nc_max; P.nc_loc = a.nc_loc; P.n0 = a.n0; P.n_max = a.n_max;
  P.n_loc = a.n_loc; P.theta = a.theta; P.theta_loc = a.theta_loc; P.g = a.g;
  P.center = a.ws->center; P.mean = a.mean; P.s2 = a.s2;
  P.selected = a.selected; P.tie_gap = a.tie_gap; P.nevals = a.nevals; P.Linv = a.ws->state64;
  P.Kc = a.ws->state32; P.crow = a.ws->crow; P.status = a.ws->status;
  P.queue = a.ws->queue + 2; P.order = a.order; P.count = a.count;
  P.promote = a.promote ? a.ws->promote : nullptr;
  P.promote_count = a.ws->status + 1;
  size_t sm = smem_design32(a.n_max, a.p, a.PP, a.nc_max);
  const bool sf = d32_smem_factor(a.n_max);
  int dev = 0, sms = 0;
  cudaError_t err;
  if ((err = cudaGetDevice(&dev)) != cudaSuccess ||
      (err = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess)
    return err;
  const int threads = d32_threads(a.M, a.nc_max, sms);
  auto pick = [&](auto k256, auto k128) { return threads == 256 ? k256 : k128; };
  auto k = P.promote ? (sf ? pick(design32<true, true, 256>, design32<true, true, 128>)
                           : pick(design32<true, false, 256>, design32<true, false, 128>))
                     : (sf ? pick(design32<false, true, 256>, design32<false, true, 128>)
                           : pick(design32<false, false, 256>, design32<false, false, 128>));
  err = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
  if (err != cudaSuccess) return err;
  const int64_t grid = persistent_grid(k, threads, sm, a.M, exh_slots(a.ws->chunk), 1,
                                       a.tune.exh_occ);
  if (grid < 0) return cudaErrorInvalidValue;
  if ((err = cudaMemsetAsync(P.queue, 0, sizeof(unsigned), s)) != cudaSuccess) return err;
  prof_begin("design32_exhaustive", s);
  k<<<(unsigned)grid, threads, sm, s>>>(P);
  prof_end(s);
  return cudaGetLastError();
}

}  // namespace lagp
