// kdtree.cuh -- spatial index over the design X_N for the unlimited ray scope:
// the snap of a ray step (Sec 4) searches all of X_N outside the current local
// design, which the paper allows (Sec 5 places no N' limit on ray searches).
//
// Tree.  An implicit k-d tree over tree positions 0..N-1: heap node 1 is the
// root with positions [0, N); node v of range [a, b) has children 2v over
// [a, m) and 2v+1 over [m, b), m = (a + b) / 2.  At level L the split runs
// along coordinate L mod p: the build orders every node's range by that
// coordinate (kdtree.cu), so the children are the lower and upper halves.
// Leaves are the nodes at depth D, the smallest depth whose ranges hold at
// most KD_LEAF points.  Every node keeps the exact bounding box of its points,
// in the centred FP32 coordinates (FP32 scoring form) and in binary64 (parity
// form).
//
// Query.  One warp finds, exactly, the nearest point to x* outside the design
// (and, where it is wanted for the step's decision gap, the second smallest
// distance).  A visit goes down KD_FAN = 5 levels at once: lane l takes the
// l-th of a node's 32 descendants there, whose boxes lie side by side in
// memory, so the boxes of five levels cost one round trip to L2 instead of
// five.  The walk is depth first, the nearest remaining descendant first, and
// leaves a node when its nearest is farther than the best distance so far (the
// second best where that is wanted, with a relative margin above the rounding
// of both distances).  A leaf gives one point per lane.  Ties go to the point
// nearer to x, then to the lower design index.  At N = 1e6, p = 8, n = 50 and 8
// rays the ray kernel takes 29.3 ms per 10,000 locations with this walk, 53.9 ms
// with one level per visit pruned by the second best.
#pragma once
#include <cstdint>

#include "common.cuh"

namespace lagp {

#define KD_LEAF 32
#define KD_FAN 5
// visits in progress, each with its first descendant and a row of 32 box
// distances: ceil(D / KD_FAN) of them, D <= 26 (int32 design indices).  (A word
// per box distance for the descendants too was 384 words of every warp of the ray
// kernel, also where no walk runs: with one ray, n = 64 and N' = 1000 that left 18
// instead of 20 warps per SM, 28.4 against 26.8 ms per 20,000 locations.)
#define KD_STACK 6
#define KD_BOUNDS (32 * KD_STACK)

__host__ __device__ inline int kd_depth(int64_t N) {
  int D = 0;
  while (((N + ((int64_t)1 << D) - 1) >> D) > KD_LEAF) ++D;
  return D;
}
__host__ __device__ inline int64_t kd_nodes(int D) { return (int64_t)2 << D; }

// Positions [a, b) of heap node v (at level `level`).
__device__ __forceinline__ void kd_range(int64_t N, int64_t v, int level, int64_t* a,
                                         int64_t* b) {
  int64_t lo = 0, hi = N;
  for (int l = level - 1; l >= 0; --l) {
    const int64_t m = (lo + hi) >> 1;
    if ((v >> l) & 1) lo = m; else hi = m;
  }
  *a = lo;
  *b = hi;
}

template <typename T>
struct KdTop {
  T d1, dx1, d2;
  int32_t i1;    // design index of the best, or -1
};

// Lexicographic (d, dx, index) order of the best; d2 keeps the second
// smallest distance (equal to d1 when two points tie).
template <typename T>
__device__ __forceinline__ KdTop<T> kd_merge(KdTop<T> a, KdTop<T> b) {
  const bool b_first = b.i1 >= 0 &&
      (a.i1 < 0 || b.d1 < a.d1 ||
       (b.d1 == a.d1 && (b.dx1 < a.dx1 || (b.dx1 == a.dx1 && b.i1 < a.i1))));
  KdTop<T> r;
  if (b_first) { r = b; r.d2 = a.d1 < b.d2 ? a.d1 : b.d2; }
  else { r = a; r.d2 = b.d1 < a.d2 ? b.d1 : a.d2; }
  return r;
}

template <typename T>
__device__ __forceinline__ KdTop<T> kd_warp_merge(KdTop<T> t) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    KdTop<T> u;
    u.d1 = __shfl_xor_sync(0xffffffffu, t.d1, o);
    u.dx1 = __shfl_xor_sync(0xffffffffu, t.dx1, o);
    u.d2 = __shfl_xor_sync(0xffffffffu, t.d2, o);
    u.i1 = __shfl_xor_sync(0xffffffffu, t.i1, o);
    t = kd_merge(t, u);
  }
  return t;
}

// A view of the tree for one arithmetic.  box: [kd_nodes(D)][2][stride] (lo
// row, then hi row); perm: tree position -> design index.
template <typename T>
struct KdView {
  const T* box;
  int stride, p, D;
  int64_t N;
  const int32_t* perm;
  const T* pts;        // FP32: tree-ordered rows [N][stride]; binary64: the design [N][p]
};

// Squared distance from xs to the box of node c.
__device__ __forceinline__ float kd_box_dist(const KdView<float>& V, int64_t c, const float* xs) {
  const float* lo = V.box + c * 2 * V.stride;    // rows padded to float4s, padding zero
  const float* hi = lo + V.stride;
  float d = 0.f;
  for (int k = 0; k < V.stride; k += 4) {
    const float4 l = *reinterpret_cast<const float4*>(lo + k);
    const float4 h = *reinterpret_cast<const float4*>(hi + k);
    float t = fmaxf(fmaxf(l.x - xs[k], xs[k] - h.x), 0.f);
    d = fmaf(t, t, d);
    t = fmaxf(fmaxf(l.y - xs[k + 1], xs[k + 1] - h.y), 0.f);
    d = fmaf(t, t, d);
    t = fmaxf(fmaxf(l.z - xs[k + 2], xs[k + 2] - h.z), 0.f);
    d = fmaf(t, t, d);
    t = fmaxf(fmaxf(l.w - xs[k + 3], xs[k + 3] - h.w), 0.f);
    d = fmaf(t, t, d);
  }
  return d;
}
__device__ __forceinline__ double kd_box_dist(const KdView<double>& V, int64_t c, const double* xs) {
  const double* lo = V.box + c * 2 * V.stride;
  const double* hi = lo + V.stride;
  double d = 0.0;
  for (int k = 0; k < V.p; ++k) {
    const double a = lo[k] - xs[k], b = xs[k] - hi[k];
    const double t = a > 0.0 ? a : (b > 0.0 ? b : 0.0);
    d += t * t;
  }
  return d;
}

// smallest of the lanes' non-negative values
__device__ __forceinline__ float kd_warp_min(float v) {
  return __uint_as_float(__reduce_min_sync(0xffffffffu, __float_as_uint(v)));
}
__device__ __forceinline__ double kd_warp_min(double v) {
  const unsigned hi = (unsigned)__double2hiint(v);
  const unsigned mh = __reduce_min_sync(0xffffffffu, hi);
  const unsigned ml =
      __reduce_min_sync(0xffffffffu, hi == mh ? (unsigned)__double2loint(v) : 0xffffffffu);
  return __hiloint2double((int)mh, (int)ml);
}

// Nearest point to xs outside the design (TOP2: and its second-best distance).
// Warp-collective; every lane returns the same result.  excluded(gi, pos,
// allow_starts) says whether design point gi (at tree position pos) may not be
// picked; with no allowed point at all the search repeats with the ray starts
// allowed.  dist(pos, gi) and distx(pos, gi) give a point's squared distances
// to x* and to x in the form's own arithmetic.  stk / bnd: KD_STACK and
// KD_BOUNDS entries per warp (the first descendant of each visit in progress, and
// the descendants' box distances).
template <bool TOP2, typename T, typename Excl, typename Dist, typename DistX>
__device__ KdTop<T> kd_nearest(const KdView<T>& V, const T* xs, T margin, int* stk, T* bnd,
                               Excl excluded, Dist dist, DistX distx) {
  const int lane = threadIdx.x & 31;
  const T inf = (T)INFINITY;
  // levels of the first visit, so that the others take KD_FAN each
  const int first = V.D % KD_FAN ? V.D % KD_FAN : KD_FAN;
  KdTop<T> best;
#pragma unroll 1
  for (int pass = 0; pass < 2; ++pass) {
    best.d1 = inf; best.dx1 = inf; best.d2 = inf; best.i1 = -1;
    int depth = -1;            // visit in progress (-1: none)
    int64_t v = 1;             // node to visit or, at depth V.D, to scan
    int level = 0;
    bool more = true;
    while (more) {
      if (level < V.D) {
        const int f = depth < 0 ? first : KD_FAN;
        ++depth;
        level += f;
        const int64_t c0 = v << f;
        bnd[depth * 32 + lane] = lane < (1 << f) ? kd_box_dist(V, c0 + lane, xs) : inf;
        if (lane == 0) stk[depth] = (int)c0;
        __syncwarp();
      } else {
        int64_t a, b;
        kd_range(V.N, v, V.D, &a, &b);
        const int64_t pos = a + lane;
        KdTop<T> t;
        t.d1 = inf; t.dx1 = inf; t.d2 = inf; t.i1 = -1;
        bool near = false;
        T d = inf;
        int32_t gi = -1;
        if (pos < b) {
          gi = V.perm[pos];
          d = dist(pos, gi);
          near = d <= (TOP2 ? best.d2 : best.d1);
        }
        // most leaves hold no point near enough: no merge
        if (__any_sync(0xffffffffu, near)) {
          if (near && !excluded(gi, pos, pass == 1)) {
            t.d1 = d;
            t.dx1 = distx(pos, gi);
            t.i1 = gi;
          }
          best = kd_merge(best, kd_warp_merge(t));
        }
      }
      // the nearest descendant left in the innermost visit that still has one
      // within reach
      more = false;
      const T reach = (TOP2 ? best.d2 : best.d1) * ((T)1 + margin);
      while (depth >= 0) {
        const T lb = bnd[depth * 32 + lane];
        const T m = kd_warp_min(lb);
        if (m < inf && m <= reach) {
          const int who = __ffs(__ballot_sync(0xffffffffu, lb == m)) - 1;
          if (lane == who) bnd[depth * 32 + lane] = inf;
          v = (int64_t)(unsigned)stk[depth] + who;
          level = first + KD_FAN * depth;
          more = true;
          __syncwarp();
          break;
        }
        --depth;
      }
    }
    if (best.i1 >= 0) break;
  }
  return best;
}

// Workspace pieces of the tree (design part of the workspace).
struct KdTree {
  int D;
  int32_t* perm;     // [N] tree position -> design index
  float* pts32;      // [N][PP] centred FP32 rows in tree order
  float* box32;      // [nodes][2][PP]
  double* box64;     // [nodes][2][p]
  uint64_t* keys;    // [2][N] sort scratch
  int32_t* vals;     // [N] sort scratch
  uint32_t* total;   // [256] digit totals of a sort pass
  uint32_t* hist;    // [256][blocks] tile counts, in the place of pts32 and box32
};

size_t kd_bytes(int64_t N, int p, int PP);
void kd_carve(int64_t N, int p, int PP, char* base, KdTree* t);
cudaError_t launch_kd_build(const double* X, const float* Xf, int64_t N, int p, int PP,
                            const KdTree& t, cudaStream_t s);

}  // namespace lagp
