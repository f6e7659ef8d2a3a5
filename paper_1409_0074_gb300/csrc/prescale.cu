// prescale.cu -- pre-scaled inputs (Sec 5.3): a crude global analysis fits a
// separable Gaussian correlation K_ab = exp(-sum_k (x_ak - x_bk)^2 / theta_k)
// (diagonal 1 + g) to a random subset of the design by maximum likelihood,
// and the inputs are divided by sqrt(theta_k) before the local approximation
// runs on them.
//
// Likelihood (the reference-prior form of Eq. gpk, as for the local
// lengthscale, with a vector theta):
//   l = lgamma(n/2) - (n/2) log(2 pi) - (1/2) log|K| - (n/2) log(psi / 2),
//   psi = y^T K^{-1} y,  alpha = K^{-1} y,
//   dl/dtheta_k = -(1/2) tr(K^{-1} K_k) + (n/2) (alpha^T K_k alpha) / psi,
//   K_k,ab = K_ab (x_ak - x_bk)^2 / theta_k^2.
// One evaluation: the gathered subset rows -> K (n x n, binary64) -> K^{-1}
// in place by Gauss-Jordan elimination without pivoting (K is symmetric
// positive definite; the pivots are the successive Schur complements, so
// their logs sum to log|K|), in panels of 32 pivots (below) -> alpha ->
// per-row partial sums of the trace and quadratic-form terms (one warp per
// row, fixed order) -> the likelihood and its gradient in eta = log theta on
// one warp, whose first lane also advances the maximiser.
//
// Panels.  Step k of the elimination is, with m_i = -A_ik / A_kk and r_j = A_kj
// as they are before the step,
//   A_ij <- m_i r_j + A_ij,  A_ik <- m_i,  A_kj <- r_j / A_kk,  A_kk <- 1 / A_kk.
// The 32 steps of a panel run first on its diagonal block (gj_diag_block: one
// CTA), then on the panel's columns and rows (gj_panels: a warp per row or
// column, every m_i^(k) and r_j^(k) kept), and then all at once, in the same
// order, on the rest (gj_rest: a rank-32 update from registers and shared
// memory).  Every element sees the operations of the one-pivot-per-launch form
// in the same order, so K^{-1} has the same bits; it is read and written once
// per panel instead of once per pivot, in 2 launches instead of 32.  The rest
// is bound by the FP64 pipe (n^3 multiply-adds, two per SM and cycle); the
// next panel's diagonal block, a chain of 32 dependent divisions, runs beside
// it on an SM of its own (block 0 of gj_rest).
//
// Maximiser: BFGS on eta from eta0 = log theta0 (inverse curvature H = I at
// the start), ascent direction d = H grad scaled so that no coordinate moves
// more than 2, trial points projected on [log tmin, log tmax]^p, steps
// t = 1, 1/2, ... (at most 41 trials) until l(eta_t) >= l(eta) + 1e-4 grad .
// (eta_t - eta); the H update is skipped unless s . y > 1e-12 |s| |y| (y the
// change of the negated gradient); the fit ends when a trial moves no
// coordinate by more than 1e-9, when no trial is accepted, or after maxit
// iterations.  The state machine runs on the device; the host only enqueues
// evaluations and reads a done flag after each.
#include <cmath>
#include <cstdint>

#include "../../include/lagp.h"
#include "common.cuh"
#include "lagp_internal.h"

namespace lagp {

#define SEP_MAX_N 1024
#define SEP_MAX_P 16
#define SEP_TOL 1e-9
#define GJ_NB 32             // pivots per panel
#define GJ_THREADS 512       // gj_rest: one 32 x 32 tile at a time, two elements per thread

enum { SEP_INIT = 0, SEP_TRIAL = 1 };

struct SepState {
  double eta[SEP_MAX_P];      // current point (log theta)
  double gr[SEP_MAX_P];       // gradient at eta
  double d[SEP_MAX_P];        // search direction
  double eta_t[SEP_MAX_P];    // point being evaluated
  double H[SEP_MAX_P * SEP_MAX_P];
  double l, t;
  int phase, it, trials, evals, done, status;
};

struct SepWork {
  double* S;       // [n][p] subset rows
  double* ys;      // [n]
  double* A;       // [n][n] K, then K^{-1}
  double* dm;      // [32][32] m_i^(k) of the panel's diagonal block (the reciprocal pivot at i = k)
  double* dr;      // [32][32] r_j^(k) of the diagonal block, row k
  double* pm;      // [n][32] m_i^(k) of the rows outside the panel
  double* pr;      // [n][32] r_j^(k) of the columns outside the panel
  double* piv;     // [n]
  double* alpha;   // [n]
  double* part;    // [n][2p] per-row partial sums
  SepState* st;
};

static size_t align256(size_t x) { return (x + 255) & ~(size_t)255; }

static size_t sep_layout(int n, int p, char* base, SepWork* w) {
  size_t off = 0;
  auto take = [&](size_t bytes) -> char* {
    char* q = base ? base + off : nullptr;
    off += align256(bytes);
    return q;
  };
  SepWork t;
  t.S = reinterpret_cast<double*>(take(sizeof(double) * n * p));
  t.ys = reinterpret_cast<double*>(take(sizeof(double) * n));
  t.A = reinterpret_cast<double*>(take(sizeof(double) * n * n));
  t.dm = reinterpret_cast<double*>(take(sizeof(double) * GJ_NB * GJ_NB));
  t.dr = reinterpret_cast<double*>(take(sizeof(double) * GJ_NB * GJ_NB));
  t.pm = reinterpret_cast<double*>(take(sizeof(double) * n * GJ_NB));
  t.pr = reinterpret_cast<double*>(take(sizeof(double) * n * GJ_NB));
  t.piv = reinterpret_cast<double*>(take(sizeof(double) * n));
  t.alpha = reinterpret_cast<double*>(take(sizeof(double) * n));
  t.part = reinterpret_cast<double*>(take(sizeof(double) * n * 2 * p));
  t.st = reinterpret_cast<SepState*>(take(sizeof(SepState)));
  if (w) *w = t;
  return off;
}

// subset rows and responses; an index outside [0, N) is reported and skipped
__global__ void sep_gather(const double* X, const double* Y, int64_t N, int p,
                           const int32_t* subset, int n, double theta0, double tmin, double tmax,
                           SepWork w) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i == 0) {
    SepState* s = w.st;
    const double e0 = log(fmin(fmax(theta0, tmin), tmax));
    for (int k = 0; k < p; ++k) { s->eta[k] = e0; s->eta_t[k] = e0; }
    s->phase = SEP_INIT;
    s->it = 0; s->trials = 0; s->evals = 0; s->done = 0; s->status = 0;
  }
  if (i >= n) return;
  const int32_t r = subset[i];
  if (r < 0 || (int64_t)r >= N) {
    atomicOr(reinterpret_cast<int*>(&w.st->status), 2);
    return;
  }
  for (int k = 0; k < p; ++k) w.S[(int64_t)i * p + k] = X[(int64_t)r * p + k];
  w.ys[i] = Y[r];
}

__device__ __forceinline__ double sep_corr(const double* a, const double* b, int p,
                                           const double* ith) {
  double s = 0.0;
  for (int k = 0; k < p; ++k) {
    const double d = a[k] - b[k];
    s += d * d * ith[k];
  }
  return exp(-s);
}

// K at theta = exp(eta_t).  The block's first p threads form 1 / theta: by every
// thread it was most of the kernel (an evaluation at n = 1000, p = 8 takes 2.89 ms,
// with it 3.11).
__global__ void sep_build(int n, int p, double g, SepWork w) {
  if (w.st->done) return;
  __shared__ double ith[SEP_MAX_P];
  const int t = threadIdx.y * blockDim.x + threadIdx.x;
  if (t < p) ith[t] = exp(-w.st->eta_t[t]);
  __syncthreads();
  const int b = blockIdx.x * blockDim.x + threadIdx.x, a = blockIdx.y * blockDim.y + threadIdx.y;
  if (a >= n || b >= n) return;
  const double v = (a == b) ? 1.0 + g : sep_corr(w.S + (int64_t)a * p, w.S + (int64_t)b * p, p, ith);
  w.A[(int64_t)a * n + b] = v;
}

__device__ __forceinline__ double shfl_d(double v, int src) {
  return __shfl_sync(0xffffffffu, v, src);
}

// The panel's steps on its diagonal block at pivot K0: warp g of 16 holds rows
// g and g + 16, lane c column c (elements past n unused).  The steps' m and r
// go to w.dm and w.dr, the pivots to w.piv, and the block to A.
__device__ void gj_diag_block(int n, int K0, double d0, double d1, SepWork w) {
  __shared__ double rowbuf[2][GJ_NB], pibuf[2];
  const int lane = threadIdx.x & 31, g = threadIdx.x >> 5;
  const int nb = min(GJ_NB, n - K0);
  for (int k = 0; k < nb; ++k) {
    const int f = k & 1;
    if ((k & 15) == g) {            // the pivot row's warp
      const double v = k < 16 ? d0 : d1;
      const double p = 1.0 / shfl_d(v, k);
      rowbuf[f][lane] = v;
      w.dr[k * GJ_NB + lane] = v;
      if (lane == k) { pibuf[f] = p; w.piv[K0 + k] = v; }
    }
    __syncthreads();
    const double r = rowbuf[f][lane], pi = pibuf[f];
    const double c0 = shfl_d(d0, k), c1 = shfl_d(d1, k);
    const double m = -((lane & 1) ? c1 : c0) * pi;
    const double m0 = g == k ? pi : shfl_d(m, 0), m1 = g + 16 == k ? pi : shfl_d(m, 1);
    // the pivot row is r pi = r pi - 0
    d0 = lane == k ? m0 : fma(m0, r, g == k ? -0.0 : d0);
    d1 = lane == k ? m1 : fma(m1, r, g + 16 == k ? -0.0 : d1);
    if (lane < 2) w.dm[(g + 16 * lane) * GJ_NB + k] = lane ? m1 : m0;
  }
  if (lane < nb && g < nb) w.A[(int64_t)(K0 + g) * n + K0 + lane] = d0;
  if (lane < nb && g + 16 < nb) w.A[(int64_t)(K0 + g + 16) * n + K0 + lane] = d1;
}

// The first panel's diagonal block (one CTA of GJ_THREADS).
__global__ void __launch_bounds__(GJ_THREADS) gj_first(int n, SepWork w) {
  if (w.st->done) return;
  const int lane = threadIdx.x & 31, g = threadIdx.x >> 5;
  const double d0 = lane < n && g < n ? w.A[(int64_t)g * n + lane] : 0.0;
  const double d1 = lane < n && g + 16 < n ? w.A[(int64_t)(g + 16) * n + lane] : 0.0;
  gj_diag_block(n, 0, d0, d1, w);
}

// The panel's steps on the rows and columns outside its block: one warp per
// row i (lane: panel column; elements A_i,K0..) or column j (lane: panel row).
__global__ void __launch_bounds__(256) gj_panels(int n, int K0, SepWork w) {
  if (w.st->done) return;
  __shared__ double dm[GJ_NB][GJ_NB + 1], dr[GJ_NB][GJ_NB + 1];
  for (int e = threadIdx.x; e < GJ_NB * GJ_NB; e += blockDim.x) {
    dm[e / GJ_NB][e % GJ_NB] = w.dm[e];
    dr[e / GJ_NB][e % GJ_NB] = w.dr[e];
  }
  __syncthreads();
  const int lane = threadIdx.x & 31, nb = min(GJ_NB, n - K0);
  const int item = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  const int out = n - nb;                            // rows, then columns, outside the block
  if (item >= 2 * out) return;
  const bool col = item >= out;
  int x = col ? item - out : item;
  if (x >= K0) x += nb;
  const bool in = lane < nb;
  double* el = col ? w.A + (int64_t)(K0 + lane) * n + x : w.A + (int64_t)x * n + K0 + lane;
  double v = in ? *el : 0.0, kept = 0.0;
  if (col) {
    for (int k = 0; k < nb; ++k) {
      const double r = shfl_d(v, k);
      if (lane == k) kept = r;
      v = fma(dm[lane][k], r, lane == k ? -0.0 : v);
    }
  } else {
    for (int k = 0; k < nb; ++k) {
      const double m = -shfl_d(v, k) * dm[k][k];
      if (lane == k) kept = m;
      v = lane == k ? m : fma(m, dr[k][lane], v);
    }
  }
  if (!in) return;
  *el = v;
  (col ? w.pr : w.pm)[(int64_t)x * GJ_NB + lane] = kept;
}

// The panel's steps on everything else, 32 x 32 tiles: block 0 takes the next
// panel's diagonal tile and then runs its steps; the other blocks stride over
// the remaining tiles, the next tile's operands loaded while one is updated.
__global__ void __launch_bounds__(GJ_THREADS) gj_rest(int n, int b, SepWork w) {
  if (w.st->done) return;
  __shared__ double M[2][GJ_NB][GJ_NB + 1], R[2][GJ_NB][GJ_NB + 1];
  const int lane = threadIdx.x & 31, g = threadIdx.x >> 5;
  const int nt = (n + GJ_NB - 1) / GJ_NB, side = nt - 1;      // tile rows outside the panel
  const int nb = min(GJ_NB, n - b * GJ_NB);
  const int next = b + 1 < nt ? b * side + b : -1;             // the next diagonal tile's index
  const int tiles = side * side;
  // block 0: only the next diagonal tile (none after the last panel)
  int t = blockIdx.x == 0 ? next : (int)blockIdx.x - 1;
  const int stride = blockIdx.x == 0 ? tiles : (int)gridDim.x - 1;
  if (blockIdx.x > 0 && t == next) t += stride;
  if (t < 0 || t >= tiles) return;
  double m0, m1, r0, r1, a0, a1;
  auto load = [&](int t) {
    int ti = t / side, tj = t - ti * side;
    ti += ti >= b; tj += tj >= b;
    const int i0 = ti * GJ_NB + g, j = tj * GJ_NB + lane, jr = tj * GJ_NB + g;
    m0 = i0 < n ? w.pm[(int64_t)i0 * GJ_NB + lane] : 0.0;
    m1 = i0 + 16 < n ? w.pm[(int64_t)(i0 + 16) * GJ_NB + lane] : 0.0;
    r0 = jr < n ? w.pr[(int64_t)jr * GJ_NB + lane] : 0.0;
    r1 = jr + 16 < n ? w.pr[(int64_t)(jr + 16) * GJ_NB + lane] : 0.0;
    a0 = i0 < n && j < n ? w.A[(int64_t)i0 * n + j] : 0.0;
    a1 = i0 + 16 < n && j < n ? w.A[(int64_t)(i0 + 16) * n + j] : 0.0;
  };
  load(t);
  for (int f = 0; t < tiles; f ^= 1) {
    M[f][g][lane] = m0; M[f][g + 16][lane] = m1;
    R[f][g][lane] = r0; R[f][g + 16][lane] = r1;
    double x0 = a0, x1 = a1;
    const int cur = t;
    t += stride;
    if (t == next && blockIdx.x > 0) t += stride;
    __syncthreads();
    if (t < tiles) load(t);
    if (nb == GJ_NB) {
#pragma unroll 8
      for (int k = 0; k < GJ_NB; ++k) {
        const double r = R[f][lane][k];
        x0 = fma(M[f][g][k], r, x0);
        x1 = fma(M[f][g + 16][k], r, x1);
      }
    } else {
      for (int k = 0; k < nb; ++k) {
        const double r = R[f][lane][k];
        x0 = fma(M[f][g][k], r, x0);
        x1 = fma(M[f][g + 16][k], r, x1);
      }
    }
    int ti = cur / side, tj = cur - ti * side;
    ti += ti >= b; tj += tj >= b;
    const int i0 = ti * GJ_NB + g, j = tj * GJ_NB + lane;
    if (blockIdx.x == 0) {
      gj_diag_block(n, (b + 1) * GJ_NB, x0, x1, w);
      return;
    }
    if (i0 < n && j < n) w.A[(int64_t)i0 * n + j] = x0;
    if (i0 + 16 < n && j < n) w.A[(int64_t)(i0 + 16) * n + j] = x1;
  }
}

__device__ __forceinline__ double warp_sum_d(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// alpha = K^{-1} y, one warp per row
__global__ void sep_alpha(int n, SepWork w) {
  if (w.st->done) return;
  const int a = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  if (a >= n) return;
  double s = 0.0;
  for (int b = lane; b < n; b += 32) s += w.A[(int64_t)a * n + b] * w.ys[b];
  s = warp_sum_d(s);
  if (lane == 0) w.alpha[a] = s;
}

// row a's sums: T_k = sum_b Kinv_ab K_ab d_abk and U_k = sum_b K_ab d_abk alpha_b
__global__ void sep_rows(int n, int p, SepWork w) {
  if (w.st->done) return;
  const int a = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  if (a >= n) return;
  double ith[SEP_MAX_P], T[SEP_MAX_P], U[SEP_MAX_P];
  for (int k = 0; k < p; ++k) { ith[k] = exp(-w.st->eta_t[k]); T[k] = 0.0; U[k] = 0.0; }
  const double* xa = w.S + (int64_t)a * p;
  for (int b = lane; b < n; b += 32) {
    if (b == a) continue;
    const double* xb = w.S + (int64_t)b * p;
    const double kab = sep_corr(xa, xb, p, ith);
    const double ki = w.A[(int64_t)a * n + b] * kab, ka = kab * w.alpha[b];
    for (int k = 0; k < p; ++k) {
      const double d = xa[k] - xb[k], dd = d * d;
      T[k] += ki * dd;
      U[k] += ka * dd;
    }
  }
  for (int k = 0; k < p; ++k) {
    const double tk = warp_sum_d(T[k]), uk = warp_sum_d(U[k]);
    if (lane == 0) {
      w.part[(int64_t)a * 2 * p + k] = tk;
      w.part[(int64_t)a * 2 * p + p + k] = uk;
    }
  }
}

__device__ void sep_propose(SepState* s, int p, double lo, double hi, int maxit, bool new_iter) {
  for (;;) {
    if (new_iter) {
      if (s->it >= maxit) { s->done = 1; return; }
      ++s->it;
      double m = 0.0;
      for (int k = 0; k < p; ++k) {
        double v = 0.0;
        for (int c = 0; c < p; ++c) v += s->H[k * SEP_MAX_P + c] * s->gr[c];
        s->d[k] = v;
        m = fmax(m, fabs(v));
      }
      if (m > 2.0)
        for (int k = 0; k < p; ++k) s->d[k] *= 2.0 / m;
      s->t = 1.0;
      s->trials = 0;
    }
    double ms = 0.0;
    for (int k = 0; k < p; ++k) {
      const double e = fmin(fmax(s->eta[k] + s->t * s->d[k], lo), hi);
      s->eta_t[k] = e;
      ms = fmax(ms, fabs(e - s->eta[k]));
    }
    ++s->trials;
    if (!(ms > SEP_TOL)) { s->done = 1; return; }     // the trial does not move: stalled
    s->phase = SEP_TRIAL;
    return;
  }
}

// Likelihood and gradient at eta_t from the partial sums; then one move of
// the BFGS state machine (one thread).
__global__ void sep_finish(int n, int p, double lo, double hi, int maxit, SepWork w) {
  SepState* s = w.st;
  if (s->done) return;
  __shared__ double red[2], sums[2 * SEP_MAX_P];
  const int lane = threadIdx.x;
  double ps = 0.0, ld = 0.0;
  for (int a = lane; a < n; a += 32) {
    ps += w.ys[a] * w.alpha[a];
    ld += log(w.piv[a]);
  }
  ps = warp_sum_d(ps);
  ld = warp_sum_d(ld);
  if (lane == 0) { red[0] = ps; red[1] = ld; }
  // the rows' partial sums in row order, one lane per sum (2p of them)
  if (lane < 2 * p) {
    double t = 0.0;
    if (lane < p) {
#pragma unroll 8
      for (int a = 0; a < n; ++a) t += w.part[(int64_t)a * 2 * p + lane];
    } else {
#pragma unroll 8
      for (int a = 0; a < n; ++a) t += w.alpha[a] * w.part[(int64_t)a * 2 * p + lane];
    }
    sums[lane] = t;
  }
  __syncwarp();
  if (lane != 0) return;
  const double psi = red[0], logdet = red[1], hn = 0.5 * n;
  double l = lgamma(hn) - hn * log(2.0 * M_PI) - 0.5 * logdet - hn * log(psi / 2.0);
  if (!(psi > 0.0)) l = NAN;
  double gt[SEP_MAX_P];
  for (int k = 0; k < p; ++k) {
    const double tr = sums[k], q = sums[p + k];
    const double th = exp(s->eta_t[k]);
    // dl/dtheta_k times theta_k (the gradient in eta)
    gt[k] = (-0.5 * tr + hn * q / psi) / th;
  }
  ++s->evals;
  if (s->phase == SEP_INIT) {
    if (!(l == l)) { s->done = 1; s->status |= 1; return; }
    s->l = l;
    for (int k = 0; k < p; ++k) s->gr[k] = gt[k];
    for (int k = 0; k < SEP_MAX_P * SEP_MAX_P; ++k) s->H[k] = 0.0;
    for (int k = 0; k < p; ++k) s->H[k * SEP_MAX_P + k] = 1.0;
    sep_propose(s, p, lo, hi, maxit, true);
    return;
  }
  double gs = 0.0;
  for (int k = 0; k < p; ++k) gs += s->gr[k] * (s->eta_t[k] - s->eta[k]);
  if (l == l && l >= s->l + 1e-4 * gs) {
    double sv[SEP_MAX_P], yv[SEP_MAX_P], sy = 0.0, ns = 0.0, ny = 0.0;
    for (int k = 0; k < p; ++k) {
      sv[k] = s->eta_t[k] - s->eta[k];
      yv[k] = s->gr[k] - gt[k];
      sy += sv[k] * yv[k];
      ns += sv[k] * sv[k];
      ny += yv[k] * yv[k];
    }
    if (sy > 1e-12 * sqrt(ns) * sqrt(ny)) {
      // H <- (I - rho s y^T) H (I - rho y s^T) + rho s s^T
      const double rho = 1.0 / sy;
      double Hy[SEP_MAX_P], yH[SEP_MAX_P], yHy = 0.0;
      for (int r = 0; r < p; ++r) {
        double a = 0.0, b = 0.0;
        for (int c = 0; c < p; ++c) {
          a += s->H[r * SEP_MAX_P + c] * yv[c];
          b += yv[c] * s->H[c * SEP_MAX_P + r];
        }
        Hy[r] = a;
        yH[r] = b;
      }
      for (int c = 0; c < p; ++c) yHy += yv[c] * Hy[c];
      for (int r = 0; r < p; ++r)
        for (int c = 0; c < p; ++c)
          s->H[r * SEP_MAX_P + c] += -rho * (sv[r] * yH[c] + Hy[r] * sv[c]) +
                                     (rho * rho * yHy + rho) * sv[r] * sv[c];
    }
    for (int k = 0; k < p; ++k) { s->eta[k] = s->eta_t[k]; s->gr[k] = gt[k]; }
    s->l = l;
    sep_propose(s, p, lo, hi, maxit, true);
  } else {
    if (s->trials >= 41) { s->done = 1; return; }   // no accepted trial
    s->t *= 0.5;
    sep_propose(s, p, lo, hi, maxit, false);
  }
}

__global__ void sep_out(int p, SepWork w, double* theta_out, int32_t* info) {
  const int k = threadIdx.x;
  if (k < p) theta_out[k] = exp(w.st->eta[k]);
  if (k == 0 && info) {
    info[0] = w.st->it;
    info[1] = w.st->evals;
    info[2] = w.st->status;
  }
}

__global__ void prescale_kernel(const double* X, int64_t rows, int p, const double* theta,
                                double* out) {
  const int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= rows * p) return;
  out[e] = X[e] / sqrt(theta[e % p]);
}

}  // namespace lagp

using namespace lagp;

extern "C" size_t laGP_sep_mle_workspace_bytes(int n_sub, int p) {
  if (n_sub < 2 || n_sub > SEP_MAX_N || p < 1 || p > SEP_MAX_P) return 0;
  return sep_layout(n_sub, p, nullptr, nullptr);
}

extern "C" int laGP_sep_mle(const double* design, const double* y, int64_t N, int p,
                            const int32_t* subset, int n_sub, double g, double theta0,
                            double tmin, double tmax, int maxit, double* theta_out,
                            int32_t* info, void* workspace, size_t workspace_bytes,
                            void* stream) {
  if (!design || !y || !subset || !theta_out || !workspace) return LAGP_ERR_INVALID;
  if (n_sub < 2 || n_sub > SEP_MAX_N || p < 1 || p > SEP_MAX_P || N < n_sub) return LAGP_ERR_INVALID;
  if (!(g >= 0.0) || !(tmin > 0.0) || !(tmax >= tmin) || !(theta0 > 0.0) || maxit < 1)
    return LAGP_ERR_INVALID;
  if (workspace_bytes < sep_layout(n_sub, p, nullptr, nullptr)) return LAGP_ERR_WORKSPACE;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  SepWork w;
  sep_layout(n_sub, p, static_cast<char*>(workspace), &w);
  const int n = n_sub;
  const double lo = log(tmin), hi = log(tmax);
  sep_gather<<<(n + 127) / 128, 128, 0, s>>>(design, y, N, p, subset, n, theta0, tmin, tmax, w);
  if (cudaGetLastError() != cudaSuccess) return LAGP_ERR_CUDA;
  const dim3 blk(32, 8), grd((n + 31) / 32, (n + 7) / 8);
  const int rows_grid = (n + 7) / 8;
  // Gauss-Jordan panels: block 0 of gj_rest is the next panel's, the others one per SM
  const int nt = (n + GJ_NB - 1) / GJ_NB, rest_tiles = (nt - 1) * (nt - 1);
  int dev = 0, sms = 0;
  if (cudaGetDevice(&dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
    return LAGP_ERR_CUDA;
  const int rest_grid = 1 + (rest_tiles < sms - 1 ? rest_tiles : (sms > 1 ? sms - 1 : 1));
  // at most maxit iterations of at most 41 trials each, plus the first evaluation
  const int64_t max_evals = (int64_t)maxit * 41 + 1;
  for (int64_t e = 0; e < max_evals; ++e) {
    sep_build<<<grd, blk, 0, s>>>(n, p, g, w);
    gj_first<<<1, GJ_THREADS, 0, s>>>(n, w);
    for (int b = 0; b < nt && rest_tiles > 0; ++b) {
      const int out = n - (n - b * GJ_NB < GJ_NB ? n - b * GJ_NB : GJ_NB);
      gj_panels<<<(2 * out + 7) / 8, 256, 0, s>>>(n, b * GJ_NB, w);
      gj_rest<<<rest_grid, GJ_THREADS, 0, s>>>(n, b, w);
    }
    sep_alpha<<<rows_grid, 256, 0, s>>>(n, w);
    sep_rows<<<rows_grid, 256, 0, s>>>(n, p, w);
    sep_finish<<<1, 32, 0, s>>>(n, p, lo, hi, maxit, w);
    if (cudaGetLastError() != cudaSuccess) return LAGP_ERR_CUDA;
    int done = 0;
    if (cudaMemcpyAsync(&done, &w.st->done, sizeof(int), cudaMemcpyDeviceToHost, s) !=
            cudaSuccess ||
        cudaStreamSynchronize(s) != cudaSuccess)
      return LAGP_ERR_CUDA;
    if (done) break;
  }
  sep_out<<<1, 32, 0, s>>>(p, w, theta_out, info);
  if (cudaGetLastError() != cudaSuccess) return LAGP_ERR_CUDA;
  int st = 0;
  if (cudaMemcpyAsync(&st, &w.st->status, sizeof(int), cudaMemcpyDeviceToHost, s) != cudaSuccess ||
      cudaStreamSynchronize(s) != cudaSuccess)
    return LAGP_ERR_CUDA;
  return st ? LAGP_ERR_DEVICE : LAGP_OK;
}

extern "C" int laGP_prescale(const double* X, int64_t rows, int p, const double* theta,
                             double* X_out, void* stream) {
  if (rows < 0 || p < 1 || p > LAGP_MAX_P) return LAGP_ERR_INVALID;
  if (rows == 0) return LAGP_OK;
  if (!X || !theta || !X_out) return LAGP_ERR_INVALID;
  const int64_t e = rows * p;
  prescale_kernel<<<(unsigned)((e + 255) / 256), 256, 0, static_cast<cudaStream_t>(stream)>>>(
      X, rows, p, theta, X_out);
  return cudaGetLastError() == cudaSuccess ? LAGP_OK : LAGP_ERR_CUDA;
}
