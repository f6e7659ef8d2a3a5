// ray32.cu -- ray search (Gramacy & Haaland, Sec 4) with FP32 scoring and an
// FP64 factor update, one warp per predictive location.
//
// Lane layout.  With R rays padded to RP (a power of two) and G = 32 / RP,
// lane = r * G + q works for ray r on every G-th row (q, q+G, ...) of each
// ALC evaluation.  All rays of a location advance together: a round evaluates
// ALC once for every ray still searching (its s = 0 point, its first golden-
// section point, or its next Brent trial point), then each ray updates its
// own Brent (1973) state.  A ray that has converged idles until the last ray
// of its location is done.  The warp never meets a CTA-wide barrier.
//
// Scoring (FP32, through the inverse Cholesky factor, as in design_fp32.cu):
//   kz_k = exp(-|S_k - z|^2 / theta),  w = L^{-1} kz,
//   ALC(z) = (w . (L^{-1} k(x)) - K(z, x))^2 / (1 + g - |w|^2).
// A ray is a straight segment z(s) = a + s d (Sec 4), so every correlation
// exponent along it is a quadratic in s:
//   -log2(e) |z(s) - S_k|^2 / theta = c_k + s (b_k + s gam),
//   c_k = nu |a - S_k|^2,  b_k = 2 nu d . (a - S_k),  gam = nu |d|^2,
// with nu = -log2(e) / theta.  c_k and b_k are formed once per greedy step;
// an evaluation then costs two FMAs and one base-2 exponential per design
// point instead of a p-coordinate distance.
// L^{-1} (FP32) sits in shared memory as lower-triangular rows padded with
// zeros to a multiple of 4, so every row is read as float4s.
// The factor itself grows in FP64 (the partitioned update in factored form,
// Sec 2.2) in global memory, packed lower-triangular.
//
// Code size.  The kernel's warps are at different places of a long loop body,
// so instruction fetches are a cost of their own: with one call site of the
// point append and of Brent's step, loops left rolled unless their trip hides
// a latency, and the k-d walk in an instantiation of its own (FULL), the
// kernel's stalls for instructions fell from 1.3 to 0.6 per issue and its time
// for 100,000 8-d locations (n = 50, N' = 1000, 8 rays) from 157 to 121.7 ms (143 ms
// before the register-held kz).
//
// Scheduling.  The kernel is persistent: each warp takes the next location
// from a device work counter until the queue is empty, optionally through a
// permutation (largest local designs first, so that uneven n does not leave a
// long tail).  The FP64 scratch belongs to the warp slot, not the location, so
// it stays within a few hundred MB (L2-resident for moderate grids) however
// many locations a launch covers.
#include <cstdint>
#include <cstring>

#include "common.cuh"
#include "kdtree.cuh"
#include "lagp_internal.h"
#include "launch_plan.h"
#include "ray32_layout.h"

namespace lagp {

#define RAY_MAX_ROUNDS 1100         // bound on evaluation rounds per step

struct RayParams {
  const double* X;
  const double* Y;
  int p, PP;
  const float* Xf;
  const double* xref;
  int64_t M;
  const int32_t* cand;
  int nc_max;
  const int32_t* nc_loc;
  int n0, n_max;
  const int32_t* n_loc;
  double theta, g;
  const double* theta_loc; // per-location lengthscale [M] or null
  int R;
  const double* lo;
  const double* hi;
  const double* center;
  double* mean;
  double* s2;
  int32_t* selected;
  double* tie_gap;
  int32_t* nevals;
  double* g64;          // per warp slot: packed L^{-1} (n(n+1)/2) then z, L^{-1} y (n each)
  int64_t g64_stride;
  unsigned* status;
  unsigned* queue;      // work counter (zero at launch)
  const int32_t* order; // item -> location, or null (identity)
  const unsigned* count;// number of items (device), or null (M)
  int full;             // snap over all of X_N through the k-d tree
  KdView<float> kd;     // the tree in centred FP32 coordinates (full scope)
  int32_t* promote;     // binary64 re-solve list, or null (promotion off)
  unsigned* promote_count;
};

// 2^x by the hardware's base-2 exponential (PTX ex2.approx); the scoring
// correlations use exp(-d / theta) = 2^(-d log2(e) / theta), with log2(e) / theta
// formed once per location
__device__ __forceinline__ float ex2_approx(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

struct Brent {
  float a, b, x, w, v, fx, fw, fv, d, e;
};

// Brent (1973) fmin on [0,1]: from the current state, either report
// convergence (false) or produce the next trial point u (true).  Same
// constants as the FP64 path: tol = 2^-13, sqrt(eps) = 2^-26.  The rays of a
// warp are at different decisions in most rounds, so both ways of each are
// computed and selected between (a branch would run both with their overhead;
// with the row sums' loads ahead, 115.1 against 117.0 ms per 100,000 locations and
// 2.19 against 2.24 for one); the quotient of a step that is not taken may be
// anything.
__device__ __forceinline__ bool brent_next(Brent& s, float* u_out) {
  const float tol3 = 0x1p-13f / 3.f, sqrt_eps = 0x1p-26f;
  const float golden = 0.381966011250105151795f;
  const float m = 0.5f * (s.a + s.b);
  const float tol1 = sqrt_eps * fabsf(s.x) + tol3;
  const float tol2 = 2.f * tol1;
  const bool go = !(fabsf(s.x - m) <= tol2 - 0.5f * (s.b - s.a));
  // the parabola through x, w, v
  const float r = (s.x - s.w) * (s.fx - s.fv);
  float q = (s.x - s.v) * (s.fx - s.fw);
  float pn = (s.x - s.v) * q - (s.x - s.w) * r;
  q = 2.f * (q - r);
  pn = q > 0.f ? -pn : pn;
  q = fabsf(q);
  const bool tried = fabsf(s.e) > tol1;
  const bool para = tried && fabsf(pn) < fabsf(0.5f * q * s.e) && pn > q * (s.a - s.x) &&
                    pn < q * (s.b - s.x);
  float dp = pn / q;
  const float u_try = s.x + dp;
  const float lim = (m - s.x >= 0.f) ? tol1 : -tol1;
  dp = (u_try - s.a < tol2 || s.b - u_try < tol2) ? lim : dp;
  // or a golden-section step into the larger part
  const float eg = (s.x < m) ? (s.b - s.x) : (s.a - s.x);
  const float en = para ? s.d : eg;
  const float dn = para ? dp : golden * eg;
  s.e = go ? en : s.e;
  s.d = go ? dn : s.d;
  *u_out = s.x + (fabsf(dn) >= tol1 ? dn : (dn >= 0.f ? tol1 : -tol1));
  return go;
}

__device__ __forceinline__ void brent_take(Brent& s, float u, float fu) {
  const bool good = fu <= s.fx, left = u < s.x;
  const bool second = !good && (fu <= s.fw || s.w == s.x);
  const bool third = !good && !second && (fu <= s.fv || s.v == s.x || s.v == s.w);
  const float end = good ? s.x : u;          // the bracket's new end
  s.b = good == left ? end : s.b;
  s.a = good == left ? s.a : end;
  const bool push = good || second;          // v <- w
  s.v = push ? s.w : (third ? u : s.v);
  s.fv = push ? s.fw : (third ? fu : s.fv);
  s.w = good ? s.x : (second ? u : s.w);
  s.fw = good ? s.fx : (second ? fu : s.fw);
  s.x = good ? u : s.x;
  s.fx = good ? fu : s.fx;
}

__device__ __forceinline__ double warp_sum64(double v) {
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// One lane's share of an ALC evaluation: rows i = q, q + G, ... of
// w = L^{-1} kz, with |w|^2 and w . z summed over them in ascending order.
// A row is two FMA chains over k (elements 0, 2 and 1, 3 of each quad, one
// paired FMA per element pair).  Shared loads return 128 bytes per cycle to
// the registers however many lanes read the same word, and that return path
// is the kernel's busiest unit, so a lane runs two rows side by side on one
// load of the ray's kz, whose first KZ_QUADS quads stay in registers for all
// rows; the row blocks that need no others are unrolled.  That leaves about
// one 128-bit load per quad of a row (two, with kz loaded per row), and two
// independent chains to cover each other's latency.  Eight quads is what fits
// in 96 registers, which 20 resident warps leave each thread: sixteen quads and
// 16 warps were slower (156.8 against 141.5 ms per 100,000 locations at 8-d,
// n = 50, N' = 1000), and so were all rows of a lane side by side, column quad
// by column quad (156.2 ms).
#define KZ_QUADS 8
__device__ __forceinline__ void fma_quad(const float4& l4, const float4& k4, float2& acc) {
  acc = __ffma2_rn(make_float2(l4.x, l4.y), make_float2(k4.x, k4.y), acc);
  acc = __ffma2_rn(make_float2(l4.z, l4.w), make_float2(k4.z, k4.w), acc);
}
template <int G>
__device__ __forceinline__ void ray_product(const float* __restrict__ Lf,
                                            const float* __restrict__ kzr,
                                            const float* __restrict__ zf, int q, int j, int n_max,
                                            float* vs_out, float* ns_out) {
  float4 kz[KZ_QUADS];
  float vs = 0.f, ns = 0.f;
  constexpr int T = 4 * KZ_QUADS / G;        // unrolled blocks of G rows, in pairs
  const int sub = q >> 2;                    // G > 4: the lane's four-row block within one of G
  auto take = [&](int i, bool in, const float2& acc) {
    if (!in) return;
    const float w = acc.x + acc.y;
    vs = fmaf(w, w, vs);
    ns = fmaf(w, zf[i], ns);
  };
#pragma unroll
  for (int t = 0; t < T; t += 2) {
    if (G * t >= j) break;
    const int k_lo = t == 0 ? 0 : ((G * t - 1) >> 2) + 1;      // first quad not yet held
    const int k_hi0 = (G * t + G - 1) >> 2, k_hi1 = (G * t + 2 * G - 1) >> 2;
#pragma unroll
    for (int k = k_lo; k <= k_hi1; ++k) kz[k] = *reinterpret_cast<const float4*>(kzr + 4 * k);
    // a row past j reads row 0's place and is not taken
    const int i0 = G * t + q, i1 = i0 + G;
    const bool in0 = i0 < j, in1 = i1 < j;
    const float* L0 = Lf + (in0 ? lf_block(i0 >> 2) + 4 * (i0 & 3) : 0);
    const float* L1 = Lf + (in1 ? lf_block(i1 >> 2) + 4 * (i1 & 3) : 0);
    float2 a0 = make_float2(0.f, 0.f), a1 = a0;
#pragma unroll
    for (int k = 0; k <= k_hi1; ++k) {
      // a block of more than four rows ends in quads that only its later rows have
      if (k <= k_hi0 && (G <= 4 || k <= ((G * t) >> 2) + sub))
        fma_quad(*reinterpret_cast<const float4*>(L0 + 16 * k), kz[k], a0);
      if (G <= 4 || k <= ((G * t + G) >> 2) + sub)
        fma_quad(*reinterpret_cast<const float4*>(L1 + 16 * k), kz[k], a1);
    }
    take(i0, in0, a0);
    take(i1, in1, a1);
  }
  for (int i0 = 4 * KZ_QUADS + q; i0 < j; i0 += 2 * G) {
    const bool in1 = i0 + G < j;
    const int i1 = in1 ? i0 + G : i0;
    const int u0 = i0 >> 2, u1 = i1 >> 2;
    const int ld0 = lf_stride(u0, n_max), ld1 = lf_stride(u1, n_max);
    const float* L0 = Lf + lf_block(u0) + 4 * (i0 & 3);
    const float* L1 = Lf + lf_block(u1) + 4 * (i1 & 3);
    float2 a0 = make_float2(0.f, 0.f), a1 = a0;
#pragma unroll
    for (int k = 0; k < KZ_QUADS; ++k, L0 += ld0, L1 += ld1) {
      fma_quad(*reinterpret_cast<const float4*>(L0), kz[k], a0);
      fma_quad(*reinterpret_cast<const float4*>(L1), kz[k], a1);
    }
    int k = KZ_QUADS;
#pragma unroll 2
    for (; k <= u0; ++k, L0 += ld0, L1 += ld1) {
      const float4 k4 = *reinterpret_cast<const float4*>(kzr + 4 * k);
      fma_quad(*reinterpret_cast<const float4*>(L0), k4, a0);
      fma_quad(*reinterpret_cast<const float4*>(L1), k4, a1);
    }
    for (; k <= u1; ++k, L1 += ld1)
      fma_quad(*reinterpret_cast<const float4*>(L1), *reinterpret_cast<const float4*>(kzr + 4 * k), a1);
    take(i0, true, a0);
    take(i1, in1, a1);
  }
  *vs_out = vs;
  *ns_out = ns;
}

// Three sums over the warp (each the value of warp_sum64, to the bit: the same
// tree of pairs) in 7 binary64 additions instead of 15: from the step where
// half the lanes hold one sum's partials, other lanes hold another's.
__device__ __forceinline__ void warp_sum64_3(double& a, double& b, double& c) {
  const int lane = threadIdx.x & 31;
  const double keep = lane < 16 ? a : b, send = lane < 16 ? b : a;
  double s = keep + __shfl_xor_sync(0xffffffffu, send, 16);   // a below lane 16, b above
  c += __shfl_xor_sync(0xffffffffu, c, 16);
  s += __shfl_xor_sync(0xffffffffu, s, 8);
  c += __shfl_xor_sync(0xffffffffu, c, 8);
  if (lane & 8) s = c;
#pragma unroll
  for (int o = 4; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  a = __shfl_sync(0xffffffffu, s, 0);
  b = __shfl_sync(0xffffffffu, s, 16);
  c = __shfl_sync(0xffffffffu, s, 8);
}

// sum_{k<len} u[k] v[k] in four sums (the first also takes the remainder), with the
// next four loads in flight during four multiply-adds
__device__ __forceinline__ double row_dot(const double* u, const double* v, int len) {
  double a0 = 0.0, a1 = 0.0, a2 = 0.0, a3 = 0.0;
  double n0 = 0.0, n1 = 0.0, n2 = 0.0, n3 = 0.0;
  if (len > 3) { n0 = u[0]; n1 = u[1]; n2 = u[2]; n3 = u[3]; }
  int k = 0;
#pragma unroll 1
  for (; k + 3 < len; k += 4) {
    const double m0 = n0, m1 = n1, m2 = n2, m3 = n3;
    if (k + 7 < len) { n0 = u[k + 4]; n1 = u[k + 5]; n2 = u[k + 6]; n3 = u[k + 7]; }
    a0 = fma(m0, v[k], a0);
    a1 = fma(m1, v[k + 1], a1);
    a2 = fma(m2, v[k + 2], a2);
    a3 = fma(m3, v[k + 3], a3);
  }
#pragma unroll 1
  for (; k < len; ++k) a0 = fma(u[k], v[k], a0);
  return (a0 + a1) + (a2 + a3);
}

enum { PH_ALC0 = 0, PH_FIRST = 1, PH_ITER = 2, PH_DONE = 3 };

// One location, by one warp, in the warp's shared-memory region and FP64 slot.
template <int RP, int PP, bool FULL>
__device__ __forceinline__ void ray32_location(const RayParams& P, const int64_t loc, float* base,
                                               double* Lg) {
  constexpr int G = 32 / RP;
  const int lane = threadIdx.x & 31;
  const int p = P.p, ldn = P.n_max, R = P.R;
  const int nc = P.nc_loc ? P.nc_loc[loc] : P.nc_max;
  const int n = P.n_loc ? P.n_loc[loc] : P.n_max;
  const int32_t* cl = P.cand + loc * P.nc_max;
  const WarpLayout lay = warp_layout(ldn, PP, RP, P.nc_max);
  float* Lf = base + lay.lf;
  float* kzb = base + lay.kz;
  float* zf = base + lay.zf;
  float* Cb = base + lay.cb;          // c_k of ray r at Cb[r * KP + k]
  float* Bb = Cb + RP * kz_ld(ldn);   // b_k of ray r at Bb[r * KP + k]
  float* taub = base + lay.tau;
  float* xf = base + lay.x;
  float* lof = xf + PP;
  float* hif = lof + PP;
  float* xs = hif + PP;
  int* gsel = reinterpret_cast<int*>(base + lay.gsel);    // design indices
  int* stk = reinterpret_cast<int*>(base + lay.stk);
  float* bnd = base + lay.bnd;
  int* starts = reinterpret_cast<int*>(base + lay.starts);
  uint32_t* mask = reinterpret_cast<uint32_t*>(base + lay.mask);     // selected candidates
  uint32_t* smask = reinterpret_cast<uint32_t*>(base + lay.smask);   // this step's ray starts
  double* vmin = reinterpret_cast<double*>(base + lay.vm);
  const int KP = kz_ld(ldn);

  double* z64 = Lg + tri(ldn);
  double* zy64 = z64 + ldn;
  const double* xq = P.xref + loc * p;

  const double theta = P.theta_loc ? P.theta_loc[loc] : P.theta;
  // -log2(e) / theta: the correlations' exponentials as one base-2 exponential
  const float nit2 = (float)(-1.4426950408889634 / theta);
  const double nit64 = -1.0 / theta;
  const float onepg = (float)(1.0 + P.g);

#pragma unroll 1
  for (int i = lane; i < lf_words(ldn); i += 32) Lf[i] = 0.f;
#pragma unroll 1
  for (int i = lane; i < RP * KP; i += 32) kzb[i] = 0.f;
#pragma unroll 1
  for (int i = lane; i < (P.nc_max + 31) / 32; i += 32) { mask[i] = 0u; smask[i] = 0u; }
  if (lane < PP) {
    const bool in = lane < p;
    xf[lane] = in ? (float)(xq[lane] - P.center[lane]) : 0.f;
    lof[lane] = in ? (float)(P.lo[lane] - P.center[lane]) : 0.f;
    hif[lane] = in ? (float)(P.hi[lane] - P.center[lane]) : 0.f;
  }
  if (P.tie_gap) {
#pragma unroll 1
    for (int i = lane; i < ldn; i += 32) P.tie_gap[loc * ldn + i] = 0.0;
  }
  if (P.nevals) {
#pragma unroll 1
    for (int i = lane; i < ldn; i += 32) P.nevals[loc * ldn + i] = 0;
  }
  __syncwarp();

  int j = 0;
  bool ok = (n >= P.n0) && (n <= nc) && (n <= ldn);
  if (lane == 0) *vmin = INFINITY;

  // ---- append design point gi (candidate rank rr, or -1) (FP64 factor row) ----
  // k_j(x_new) and l = L_j^{-1} k_j(x_new) live in shared memory, in the
  // coefficient region, which no evaluation uses while a point is appended
  double* kvs = reinterpret_cast<double*>(Cb);
  double* ls = kvs + ldn;
  auto add_point = [&](int gi, int rr) -> bool {
    const double* c64 = P.X + (int64_t)gi * p;
    double kxj = 0.0;   // K(x_new, x), on lane j mod 32
#pragma unroll 1
    for (int i = lane; i <= j; i += 32) {
      const double c = corr64_fast(i < j ? P.X + (int64_t)gsel[i] * p : xq, c64, p, nit64);
      if (i < j) kvs[i] = c;
      else kxj = c;
    }
    kxj = __shfl_sync(0xffffffffu, kxj, j & 31);
    __syncwarp();
    // l = L_j^{-1} k_j(x_new); v = 1 + g - |l|^2, d = sqrt(v), and by forward
    // substitution z_j = (K(x_new, x) - l . z) / d, (L^{-1} y)_j =
    // (y_new - l . L^{-1} y) / d, all from one pass.  A warp's FP64
    // instruction costs the same whatever its active lanes, so every lane
    // evaluates the scalar tail.
    double vv = 0.0, lz = 0.0, lzy = 0.0;
#pragma unroll 1
    for (int i = lane; i < j; i += 32) {
      const double acc = row_dot(Lg + tri(i), kvs, i + 1);
      ls[i] = acc;
      vv = fma(acc, acc, vv);
      lz = fma(acc, z64[i], lz);
      lzy = fma(acc, zy64[i], lzy);
    }
    warp_sum64_3(vv, lz, lzy);
    __syncwarp();
    const double v = (1.0 + P.g) - vv;
    if (lane == 0) *vmin = v > 0.0 ? fmin(*vmin, v) : -1.0;
    if (!(v > 0.0)) return false;
    const double inv_d = rsqrt(v);
    double* Lj = Lg + tri(j);
    float* Lfj = Lf + lf_at(j, 0, ldn);
    const int lds = lf_stride(j >> 2, ldn);
#pragma unroll 1
    for (int k = lane; k < ((j + 31) & ~31); k += 32) {
      // sum_i l_i L_ik over i >= k: the even and the odd offsets i - k apart, as
      // the even and the odd i (adding the two is commutative).  All lanes take
      // the same row i, so its elements are contiguous over them.  (The other
      // product, by rows, stays as it is: a second copy of the factor by
      // columns made it contiguous too, but doubled the scratch the slots cycle
      // through L2 and was slower, 124.0 against 117.2 ms per 100,000
      // locations.)
      const int i0 = k & ~31;
      const double* Lk = Lg + k;
      auto at = [&](int i) { return i >= k && i < j ? Lk[tri(i)] : 0.0; };
      double a0 = 0.0, a1 = 0.0;
      double n0 = at(i0), n1 = at(i0 + 1), n2 = at(i0 + 2), n3 = at(i0 + 3);
#pragma unroll 1
      for (int i = i0; i < j; i += 4) {
        // the next rows' loads are in flight during this step's FP64
        const double m0 = n0, m1 = n1, m2 = n2, m3 = n3;
        n0 = at(i + 4); n1 = at(i + 5); n2 = at(i + 6); n3 = at(i + 7);
        a0 = fma(ls[i], m0, a0);
        if (i + 1 < j) a1 = fma(ls[i + 1], m1, a1);
        if (i + 2 < j) a0 = fma(ls[i + 2], m2, a0);
        if (i + 3 < j) a1 = fma(ls[i + 3], m3, a1);
      }
      if (k >= j) break;
      const double rk = -(a0 + a1) * inv_d;
      Lj[k] = rk;
      Lfj[lds * (k >> 2) + (k & 3)] = (float)rk;
    }
    if (lane == 0) {
      Lj[j] = inv_d;
      Lfj[lds * (j >> 2) + (j & 3)] = (float)inv_d;
      gsel[j] = gi;
      if (rr >= 0) mask[rr >> 5] |= 1u << (rr & 31);
      const double zj = (kxj - lz) * inv_d;
      z64[j] = zj;
      zy64[j] = (P.Y[gi] - lzy) * inv_d;
      zf[j] = (float)zj;
    }
    __syncwarp();
    ++j;
    return true;
  };

  const int r = lane / G, q = lane % G;
#pragma unroll 1
  for (int step = 0; step < n && ok; ++step) {
    int pick = step, pick_g = -1;     // rank among the candidates (or -1) and design index
    if (step < P.n0) {
      pick_g = cl[step];
    } else {
    // ---- ray starts: unselected candidates of rank k0, k0+1, ... (mod |U|) ----
    // lane l owns mask words l, l + 32, ...; a warp scan of their unselected
    // counts locates the word holding each target rank
    {
      const int nU = nc - j;
      const int k0 = ray_offset(j, P.n0) % nU;
      const int nw = (nc + 31) >> 5;
      int seen = 0;
#pragma unroll 1
      for (int w0 = 0; w0 < nw; w0 += 32) {
        const int wd = w0 + lane;
        uint32_t un = 0u;
        if (wd < nw) {
          const int hi = min(32, nc - wd * 32);
          un = ~mask[wd] & (hi == 32 ? 0xffffffffu : ((1u << hi) - 1u));
        }
        const int c = __popc(un);
        int incl = c;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
          const int y = __shfl_up_sync(0xffffffffu, incl, o);
          if (lane >= o) incl += y;
        }
        const int first = seen + incl - c;
#pragma unroll 1
        for (int t = 0; t < R; ++t) {
          int target = k0 + t;
          if (target >= nU) target %= nU;      // (round the end: rare)
          if (target >= first && target < first + c) {
            uint32_t u = un;
#pragma unroll 1
            for (int q2 = target - first; q2 > 0; --q2) u &= u - 1u;   // drop lower bits
            const int rr = wd * 32 + __ffs(u) - 1;
            starts[t] = rr;
            smask[wd] |= 1u << (rr & 31);   // words are lane-owned: no race
          }
        }
        seen += __shfl_sync(0xffffffffu, incl, 31);
      }
    }
    __syncwarp();
    // ---- segments (FP32): end = A + tau * 10 (A - x), cut at the design's box ----
    const bool ray_live = r < R;
    float len2 = 0.f, gam = 0.f, cx = 0.f, bx = 0.f;
    if (ray_live) {
      const float* a = P.Xf + (int64_t)cl[starts[r]] * PP;
      float tau = 1.f;
#pragma unroll 1
      for (int k = 0; k < p; ++k) {
        const float dk = 10.f * (a[k] - xf[k]);
        if (dk > 0.f) tau = fminf(tau, (hif[k] - a[k]) / dk);
        else if (dk < 0.f) tau = fminf(tau, (lof[k] - a[k]) / dk);
      }
      tau = fmaxf(tau, 0.f);
      if (q == 0) taub[r] = tau;
      float av[PP], dv[PP];
      float cxs = 0.f, bxs = 0.f;
#pragma unroll
      for (int k = 0; k < PP; ++k) {
        const float ak = a[k];
        const float ek = fmaf(tau, 10.f * (ak - xf[k]), ak);
        av[k] = ak;
        dv[k] = ek - ak;
        len2 = fmaf(dv[k], dv[k], len2);
        const float tx = ak - xf[k];
        cxs = fmaf(tx, tx, cxs);
        bxs = fmaf(dv[k], tx, bxs);
      }
      // the exponents of K(z(s), x) and of K(z(s), S_k), k < j, as
      // quadratics in s; quads past j get c = -inf (a zero correlation)
      gam = nit2 * len2;
      cx = nit2 * cxs;
      bx = 2.f * nit2 * bxs;
      float* cr = Cb + r * KP;
      float* br = Bb + r * KP;
#pragma unroll 1
      for (int k4 = q; 4 * k4 < j; k4 += G) {
        float cq[4], bq[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          // a quad's rows are loaded without a branch, all in flight together
          const int k = 4 * k4 + u;
          const float* sk = P.Xf + (int64_t)gsel[min(k, j - 1)] * PP;
          float cs = 0.f, bs = 0.f;
#pragma unroll
          for (int c = 0; c < PP; c += 4) {
            const float4 s4 = *reinterpret_cast<const float4*>(sk + c);
            const float t0 = av[c] - s4.x, t1 = av[c + 1] - s4.y;
            const float t2 = av[c + 2] - s4.z, t3 = av[c + 3] - s4.w;
            cs = fmaf(t0, t0, cs); cs = fmaf(t1, t1, cs);
            cs = fmaf(t2, t2, cs); cs = fmaf(t3, t3, cs);
            bs = fmaf(dv[c], t0, bs); bs = fmaf(dv[c + 1], t1, bs);
            bs = fmaf(dv[c + 2], t2, bs); bs = fmaf(dv[c + 3], t3, bs);
          }
          cq[u] = k < j ? nit2 * cs : -__int_as_float(0x7f800000);
          bq[u] = k < j ? 2.f * nit2 * bs : 0.f;
        }
        *reinterpret_cast<float4*>(cr + 4 * k4) = make_float4(cq[0], cq[1], cq[2], cq[3]);
        *reinterpret_cast<float4*>(br + 4 * k4) = make_float4(bq[0], bq[1], bq[2], bq[3]);
      }
    }
    __syncwarp();

    // ---- lockstep Brent over the rays ----
    int phase = ray_live ? PH_ALC0 : PH_DONE;
    float s_eval = 0.f, alc0 = 0.f, s_star = 0.f, alc_star = 0.f;
    int evals = 0;
    Brent st;
    st.a = 0.f; st.b = 1.f; st.x = st.w = st.v = 0.f; st.fx = st.fw = st.fv = 0.f;
    st.d = 0.f; st.e = 0.f;
#pragma unroll 1
    for (int round = 0; round < RAY_MAX_ROUNDS; ++round) {
      const bool active = phase != PH_DONE;
      if (!__any_sync(0xffffffffu, active)) break;
      float* kzr = kzb + r * KP;
      if (active) {
        // kz over quads of design points, two exponents per paired FMA
        const float* cr = Cb + r * KP;
        const float* br = Bb + r * KP;
        const float2 s2v = make_float2(s_eval, s_eval), g2 = make_float2(gam, gam);
        auto quad = [&](const float4& c4, const float4& b4) {
          const float2 t01 = __ffma2_rn(s2v, g2, make_float2(b4.x, b4.y));
          const float2 t23 = __ffma2_rn(s2v, g2, make_float2(b4.z, b4.w));
          const float2 e01 = __ffma2_rn(s2v, t01, make_float2(c4.x, c4.y));
          const float2 e23 = __ffma2_rn(s2v, t23, make_float2(c4.z, c4.w));
          return make_float4(ex2_approx(e01.x), ex2_approx(e01.y), ex2_approx(e23.x),
                             ex2_approx(e23.y));
        };
        // two quads per trip, so that their loads and exponentials overlap
#pragma unroll 1
        for (int k4 = q; 4 * k4 < j; k4 += 2 * G) {
          const bool two = 4 * (k4 + G) < j;
          const int k5 = two ? k4 + G : k4;
          const float4 c4 = *reinterpret_cast<const float4*>(cr + 4 * k4);
          const float4 b4 = *reinterpret_cast<const float4*>(br + 4 * k4);
          const float4 c5 = *reinterpret_cast<const float4*>(cr + 4 * k5);
          const float4 b5 = *reinterpret_cast<const float4*>(br + 4 * k5);
          *reinterpret_cast<float4*>(kzr + 4 * k4) = quad(c4, b4);
          if (two) *reinterpret_cast<float4*>(kzr + 4 * k5) = quad(c5, b5);
        }
      }
      __syncwarp();
      float vs = 0.f, ns = 0.f;
      if (active) ray_product<G>(Lf, kzr, zf, q, j, ldn, &vs, &ns);
#pragma unroll
      for (int o = G / 2; o > 0; o >>= 1) {
        vs += __shfl_xor_sync(0xffffffffu, vs, o);
        ns += __shfl_xor_sync(0xffffffffu, ns, o);
      }
      float val = 0.f;
      if (active) {
        const float v = onepg - vs;
        const float num = ns - ex2_approx(fmaf(s_eval, fmaf(s_eval, gam, bx), cx));
        val = v > 0.f ? num * num / v : 0.f;
      }
      __syncwarp();
      if (active) {
        ++evals;
        bool more;
        float u = 0.381966011250105151795f;   // the first golden-section point
        if (phase == PH_ALC0) {
          alc0 = val;
          more = len2 > 0.f;
        } else {
          if (phase == PH_FIRST) {
            st.x = st.w = st.v = s_eval;
            st.fx = st.fw = st.fv = -val;
          } else {
            brent_take(st, s_eval, -val);
          }
          more = brent_next(st, &u);
        }
        if (more && evals > 1000) more = false;
        if (!more) {
          if (phase == PH_ALC0 || alc0 >= -st.fx) { s_star = 0.f; alc_star = alc0; }
          else { s_star = st.x; alc_star = -st.fx; }
          phase = PH_DONE;
        } else {
          s_eval = u;
          phase = phase == PH_ALC0 ? PH_FIRST : PH_ITER;
        }
      }
    }
    // ---- best ray, its continuous point x* ----
    float best = -1.f, second = -1.f;
    int ib = 0, ev = 0;
#pragma unroll 1
    for (int rr = 0; rr < R; ++rr) {
      const float a_r = __shfl_sync(0xffffffffu, alc_star, rr * G);
      ev += __shfl_sync(0xffffffffu, evals, rr * G);
      if (a_r > best) { second = best; best = a_r; ib = rr; }
      else if (a_r > second) second = a_r;
    }
    const float sb = __shfl_sync(0xffffffffu, s_star, ib * G);
    if (lane < PP) {
      // the best ray's segment again, in the same operations as above
      const float ak = P.Xf[(int64_t)cl[starts[ib]] * PP + lane];
      const float ek = fmaf(taub[ib], 10.f * (ak - xf[lane]), ak);
      xs[lane] = fmaf(sb, ek - ak, ak);
    }
    __syncwarp();
    // ---- snap: nearest allowed unselected candidate (ties to the lower rank) ----
    // allowed: not one of this step's ray starts unless it coincides with x*;
    // if no candidate is allowed, the nearest unselected one (second pair)
    float2 nx[PP / 2];
#pragma unroll
    for (int k = 0; k < PP; k += 2) nx[k / 2] = make_float2(-xs[k], -xs[k + 1]);
    float bd0 = __int_as_float(0x7f800000), bd1 = bd0;
    int bi0 = 0x7fffffff, bi1 = 0x7fffffff;
    if (FULL) {
      // nearest point of X_N outside the design; the step's starts are
      // forbidden unless they equal x*
      const KdView<float>& V = P.kd;
      auto excluded = [&](int32_t gi, int64_t pos, bool allow_starts) -> bool {
#pragma unroll 1
        for (int i = 0; i < j; ++i) if (gsel[i] == gi) return true;
        if (allow_starts) return false;
#pragma unroll 1
        for (int t = 0; t < R; ++t) {
          if (cl[starts[t]] != gi) continue;
#pragma unroll 1
          for (int k = 0; k < p; ++k) if (V.pts[pos * PP + k] != xs[k]) return true;
        }
        return false;
      };
      auto dist = [&](int64_t pos, int32_t) -> float {
        const float* c = V.pts + pos * PP;
        float2 d2 = make_float2(0.f, 0.f);
#pragma unroll
        for (int k = 0; k < PP; k += 4) {
          const float4 cv = *reinterpret_cast<const float4*>(c + k);
          const float2 t01 = __fadd2_rn(make_float2(cv.x, cv.y), nx[k / 2]);
          const float2 t23 = __fadd2_rn(make_float2(cv.z, cv.w), nx[k / 2 + 1]);
          d2 = __ffma2_rn(t01, t01, d2);
          d2 = __ffma2_rn(t23, t23, d2);
        }
        return d2.x + d2.y;
      };
      auto distx = [&](int64_t pos, int32_t) -> float {
        const float* c = V.pts + pos * PP;
        float d = 0.f;
#pragma unroll 1
        for (int k = 0; k < PP; ++k) { const float t = c[k] - xf[k]; d = fmaf(t, t, d); }
        return d;
      };
      const KdTop<float> b = kd_nearest<false>(V, xs, 1e-5f, stk, bnd, excluded, dist, distx);
      pick_g = b.i1;
    } else {
      // When the best ray kept s = 0, x* is its start, an allowed candidate at
      // distance 0; only a lower-ranked candidate at distance 0 (the same FP32
      // coordinates) could take it, so the scan stops at the start's rank.
      const int lim = (sb == 0.f) ? starts[ib] + 1 : nc;
      const int nw = (lim + 31) >> 5;
      const uint32_t bit = 1u << lane;
      auto consider = [&](int wd, const float4 (&cv)[PP / 4]) {
        const int rr = wd * 32 + lane;
        if (rr < lim && !(mask[wd] & bit)) {
          float2 d2 = make_float2(0.f, 0.f);
          bool same = true;                   // every coordinate equal to x*'s
#pragma unroll
          for (int k = 0; k < PP; k += 4) {
            const float4 v = cv[k / 4];
            const float2 t01 = __fadd2_rn(make_float2(v.x, v.y), nx[k / 2]);
            const float2 t23 = __fadd2_rn(make_float2(v.z, v.w), nx[k / 2 + 1]);
            same &= (t01.x == 0.f) & (t01.y == 0.f) & (t23.x == 0.f) & (t23.y == 0.f);
            d2 = __ffma2_rn(t01, t01, d2);
            d2 = __ffma2_rn(t23, t23, d2);
          }
          const float d = d2.x + d2.y;
          if (d < bd1) { bd1 = d; bi1 = rr; }
          if ((same || !(smask[wd] & bit)) && d < bd0) { bd0 = d; bi0 = rr; }
        }
      };
      // a few candidates per lane at a time, and the next ones' indices loaded
      // while their rows arrive from L2
      constexpr int NS = 2;
      int gi[NS];
#pragma unroll
      for (int t = 0; t < NS; ++t) gi[t] = cl[min(t * 32 + lane, lim - 1)];
#pragma unroll 1
      for (int wd = 0; wd < nw; wd += NS) {
        float4 v[NS][PP / 4];
#pragma unroll
        for (int t = 0; t < NS; ++t) {
          const float4* c = reinterpret_cast<const float4*>(P.Xf + (int64_t)gi[t] * PP);
#pragma unroll
          for (int k = 0; k < PP / 4; ++k) v[t][k] = c[k];
        }
#pragma unroll
        for (int t = 0; t < NS; ++t) gi[t] = cl[min((wd + NS + t) * 32 + lane, lim - 1)];
#pragma unroll
        for (int t = 0; t < NS; ++t) consider(wd + t, v[t]);
      }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      const float od0 = __shfl_xor_sync(0xffffffffu, bd0, o);
      const int oi0 = __shfl_xor_sync(0xffffffffu, bi0, o);
      const float od1 = __shfl_xor_sync(0xffffffffu, bd1, o);
      const int oi1 = __shfl_xor_sync(0xffffffffu, bi1, o);
      if (od0 < bd0 || (od0 == bd0 && oi0 < bi0)) { bd0 = od0; bi0 = oi0; }
      if (od1 < bd1 || (od1 == bd1 && oi1 < bi1)) { bd1 = od1; bi1 = oi1; }
    }
    pick = -1;
    if (!FULL) {
      pick = bi0 != 0x7fffffff ? bi0 : (bi1 != 0x7fffffff ? bi1 : -1);
      pick_g = pick >= 0 ? cl[pick] : -1;
    } else if (pick_g >= 0) {
      // its candidate rank, when it is one
      int rk = 0x7fffffff;
#pragma unroll 1
      for (int rr = lane; rr < nc; rr += 32) if (cl[rr] == pick_g) rk = min(rk, rr);
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) rk = min(rk, __shfl_xor_sync(0xffffffffu, rk, o));
      pick = rk != 0x7fffffff ? rk : -1;
    }
    __syncwarp();
    if (lane < R) smask[starts[lane] >> 5] = 0u;
    if (lane == 0) {
      if (P.tie_gap) P.tie_gap[loc * ldn + (step - P.n0)] =
          (best > 0.f && R > 1) ? (double)((best - second) / best) : 0.0;
      if (P.nevals) P.nevals[loc * ldn + (step - P.n0)] = ev;
    }
    }
    ok = (pick_g >= 0) && add_point(pick_g, pick);
  }

  if (ok) {
    double a = 0.0, b = 0.0, c = 0.0;
#pragma unroll 1
    for (int i = lane; i < j; i += 32) {
      a = fma(z64[i], zy64[i], a);
      b = fma(zy64[i], zy64[i], b);
      c = fma(z64[i], z64[i], c);
    }
    a = warp_sum64(a);
    b = warp_sum64(b);
    c = warp_sum64(c);
    if (lane == 0) {
      P.mean[loc] = a;
      P.s2[loc] = b * ((1.0 + P.g) - c) / (double)j;
    }
  } else if (lane == 0) {
    P.mean[loc] = __longlong_as_double(0x7ff8000000000000ll);
    P.s2[loc] = __longlong_as_double(0x7ff8000000000000ll);
    atomicOr(P.status, LAGP_DEV_BAD_UPDATE);
  }
  if (P.selected)
#pragma unroll 1
    for (int i = lane; i < ldn; i += 32) P.selected[loc * ldn + i] = (i < j) ? gsel[i] : -1;
  if (lane == 0) promote_location(P.promote, P.promote_count, loc, *vmin);
}

// 20 resident warps per SM (at most 96 registers per thread, 32 of them the
// ray's kz quads); the block holds 1, 2 or 4 warps
template <int RP, int PP, bool FULL>
__global__ void __launch_bounds__(128, 5) ray32_kernel(RayParams P) {
  extern __shared__ __align__(16) float sm[];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const WarpLayout lay = warp_layout(P.n_max, PP, RP, P.nc_max);
  float* base = sm + (size_t)warp * (lay.bytes / 4);
  double* Lg = P.g64 + ((int64_t)blockIdx.x * (blockDim.x >> 5) + warp) * P.g64_stride;
  const unsigned items = P.count ? *P.count : (unsigned)P.M;
  for (;;) {
    unsigned it = 0;
    if (lane == 0) it = atomicAdd(P.queue, 1u);
    it = __shfl_sync(0xffffffffu, it, 0);
    if (it >= items) break;
    ray32_location<RP, PP, FULL>(P, P.order ? (int64_t)P.order[it] : (int64_t)it, base, Lg);
    __syncwarp();
  }
}

// Warps per CTA that let the most locations reside on an SM at this shape:
// shared memory decides, under the launch bound's 20 warps per SM; ties go to
// 2, then 4, then 1, and 2 is the answer when no device can be queried.
int ray32_default_warps(int p, int n_max, int nc_max, int nrays) {
  int dev = 0, smem_sm = 0, reserved = 0;
  if (cudaGetDevice(&dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&smem_sm, cudaDevAttrMaxSharedMemoryPerMultiprocessor, dev) !=
          cudaSuccess ||
      cudaDeviceGetAttribute(&reserved, cudaDevAttrReservedSharedMemoryPerBlock, dev) !=
          cudaSuccess) {
    cudaGetLastError();
    return 2;
  }
  int RP = 2;
  while (RP < nrays) RP <<= 1;
  const size_t wb = (size_t)warp_layout(n_max, (p + 3) / 4 * 4, RP, nc_max).bytes;
  return warps_per_cta_for_residency(wb, (size_t)smem_sm, (size_t)reserved, 20);
}

size_t ray32_g64_doubles(int n_max) { return (size_t)tri(n_max) + 2 * (size_t)n_max; }

// Warp slots for a chunk: at least one CTA of the widest choice (4 warps) and a
// multiple of 4, so that every warp of every launched CTA owns a slot.
int ray32_slots(int64_t chunk) {
  const int64_t s = chunk < RAY_SLOTS ? chunk : RAY_SLOTS;
  return (int)((s + 3) / 4 * 4);
}

template <int RP, int PP>
static cudaError_t ray32_go(const RayParams& P, int RW, size_t sm, int slots, cudaStream_t s) {
  auto k = P.full ? ray32_kernel<RP, PP, true> : ray32_kernel<RP, PP, false>;
  cudaError_t err = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
  if (err != cudaSuccess) return err;
  const int64_t grid = persistent_grid(k, RW * 32, sm, P.M, slots, RW);
  if (grid < 0) return cudaErrorInvalidValue;
  if ((err = cudaMemsetAsync(P.queue, 0, sizeof(unsigned), s)) != cudaSuccess) return err;
  prof_begin("ray32", s);
  k<<<(unsigned)grid, RW * 32, sm, s>>>(P);
  prof_end(s);
  return cudaGetLastError();
}

cudaError_t launch_ray32(const DesignArgs& a, cudaStream_t s) {
  RayParams P;
  P.X = a.X; P.Y = a.Y; P.p = a.p; P.PP = a.PP; P.Xf = a.ws->Xf; P.xref = a.xref; P.M = a.M;
  P.cand = a.cand; P.nc_max = a.nc_max; P.nc_loc = a.nc_loc; P.n0 = a.n0; P.n_max = a.n_max;
  P.n_loc = a.n_loc; P.theta = a.theta; P.theta_loc = a.theta_loc; P.g = a.g; P.R = a.nrays; P.lo = a.ws->lo;
  P.hi = a.ws->hi; P.center = a.ws->center; P.mean = a.mean; P.s2 = a.s2;
  P.selected = a.selected; P.tie_gap = a.tie_gap; P.nevals = a.nevals; P.g64 = a.ws->state64;
  P.g64_stride = (int64_t)ray32_g64_doubles(a.n_max); P.status = a.ws->status;
  P.queue = a.ws->queue; P.order = a.order; P.count = a.count;
  P.full = a.full_scope;
  P.promote = a.promote ? a.ws->promote : nullptr;
  P.promote_count = a.ws->status + 1;
  if (P.full) {
    const KdTree& t = a.ws->kd;
    P.kd.box = t.box32; P.kd.stride = a.PP; P.kd.p = a.p; P.kd.D = t.D; P.kd.N = a.N;
    P.kd.perm = t.perm; P.kd.pts = t.pts32;
  } else {
    std::memset(&P.kd, 0, sizeof(P.kd));
  }
  int RP = 2;
  while (RP < a.nrays) RP <<= 1;
  const WarpLayout lay = warp_layout(a.n_max, a.PP, RP, a.nc_max);
  const int RW = a.tune.ray_warps;
  const size_t sm = (size_t)lay.bytes * RW;
  const int slots = ray32_slots(a.ws->chunk);
  switch (RP * 100 + a.PP) {
#define RAY_CASE(RPV, PPV) \
  case RPV * 100 + PPV: return ray32_go<RPV, PPV>(P, RW, sm, slots, s);
    RAY_CASE(2, 4) RAY_CASE(2, 8) RAY_CASE(2, 12) RAY_CASE(2, 16)
    RAY_CASE(4, 4) RAY_CASE(4, 8) RAY_CASE(4, 12) RAY_CASE(4, 16)
    RAY_CASE(8, 4) RAY_CASE(8, 8) RAY_CASE(8, 12) RAY_CASE(8, 16)
    RAY_CASE(16, 4) RAY_CASE(16, 8) RAY_CASE(16, 12) RAY_CASE(16, 16)
#undef RAY_CASE
    default:
      return cudaErrorInvalidValue;
  }
}

}  // namespace lagp
