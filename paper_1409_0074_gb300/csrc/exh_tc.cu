// exh_tc.cu -- exhaustive greedy local design (Gramacy & Haaland, Sec 2.2) with
// the candidate scores of every step computed as a dense contraction on the
// tensor cores, one CTA (4 warps) per predictive location; local designs up to
// n = 64.  This is the exhaustive search of the LAGP_FP32_SCORE_TC form; the
// default LAGP_FP32_SCORE form keeps running sums instead and only adds the
// newest column of W per step (design_fp32.cu).
//
// Scoring (the factored form of Eq. alc, as in design_fp32.cu): with the
// correlation rows Kc (N' x j, Kc[r][i] = K(c_r, S_i)) and the inverse
// Cholesky factor L_j^{-1},
//     W = Kc L_j^{-T}   (row r: w_r = L_j^{-1} k_j(c_r)),
//     v_r = 1 + g - |w_r|^2,  num_r = w_r . z - K(c_r, x),  ALC_r = num_r^2 / v_r,
// z = L_j^{-1} k_j(x).  W is a tcgen05.mma kind::tf32 product of 128-candidate
// tiles (M = 128) with rows of L_j^{-1} (N = 16, K = j rounded up to 8), 3xTF32
// (hi*hi + hi*lo + lo*hi, FP32 accumulation in TMEM).  L_j^{-1} only gains a
// row per step, so a column of W, once formed, does not change (the products
// past its diagonal are exact zeros); a step forms the newest column only and
// adds it to every candidate's running |w_r|^2 and w_r . z.  Thread t of the
// CTA owns candidate row t of every tile: it reads the column from TMEM
// (tcgen05.ld 32x32b) and scores its candidates.  The block argmax (ties to the
// lower rank) picks the next point.
//
// FP64 state (the partitioned update in factored form, Sec 2.2): L_j^{-1},
// packed by rows in shared memory, grown by one row per step, and z, L^{-1} y;
// the predictive equations (Eq. predgp, preds2) at the end.  The rows of the
// current block of 16 are also kept, split into TF32 hi + lo, as the B operand.
//
// The correlation cache is kept in global memory already in the A operand's
// form: per 128-candidate tile, TF32 hi and lo in slabs of 8 columns; each step
// writes one column (N' exponentials).  A tile's operand arrives in pieces of 16
// columns, one bulk copy (TMA) each, through a ring of four buffers: copies run
// two pieces ahead of the MMAs (warp 0 issues both), and up to XT_GROUP tiles
// run before their columns are read, each with its own TMEM columns.  (In 32
// copies of a row group each, a piece took over 3,000 cycles: the copy unit's
// time goes by copies, not bytes.)
//
// A step is a chain of latencies (copies, MMAs, the binary64 update, barriers)
// on two CTAs per SM; with W formed whole at every step, one tile at a time
// between three block barriers, and the factor in global memory, the kernel
// took 52.8 ms per 10,000 locations (8-d, n = 50, N' = 1000); it takes 41.4 ms.
#include <cstdint>

#include "common.cuh"
#include "lagp_internal.h"

namespace lagp {

#define XT_THREADS 128
#define XT_KMAX 64     // largest local design on this path
#define XT_KC 16       // columns of an A operand piece
#define XT_RING 4      // pieces in shared memory
#define XT_GROUP 8     // candidate tiles whose scores are in TMEM at a time

struct XtParams {
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
  const double* theta_loc;   // per-location lengthscale [M] or null
  const double* center;
  double* mean;
  double* s2;
  int32_t* selected;
  double* tie_gap;
  int32_t* nevals;
  float* Kc;             // [slots][ceil(nc_max / 128)] tiles of 2 x 128 x XT_KMAX floats
  float* crow;           // [slots][nc_max][PP] the location's candidates' FP32 rows
  unsigned* status;
  unsigned* queue;       // work counter (zero at launch)
  const int32_t* order;  // item -> location, or null
  const unsigned* count; // items (device), or null (M)
  int32_t* promote;      // binary64 re-solve list, or null (promotion off)
  unsigned* promote_count;
};

#define XT_TILE_FLOATS (128 * XT_KMAX)   // one of hi / lo of a 128-candidate tile

// B operand: canonical no-swizzle K-major layout with XT_KMAX columns per row
__device__ __forceinline__ uint32_t xcanon(int row, int k) {
  return (uint32_t)((row >> 3) * ((XT_KMAX >> 2) * 128) + (k >> 2) * 128 + (row & 7) * 16 +
                    (k & 3) * 4);
}
// A operand of a tile, in bytes: per 8 columns (one MMA's K) a slab of the 128
// rows' hi and then lo parts, each canonical, so that any run of columns is
// one contiguous copy
#define XT_SLAB 8192
__device__ __forceinline__ uint32_t xslab(int row, int k) {
  return (uint32_t)((k >> 3) * XT_SLAB + (row >> 3) * 256 + ((k >> 2) & 1) * 128 + (row & 7) * 16 +
                    (k & 3) * 4);
}

__device__ __forceinline__ float xtf32(float v) {
  uint32_t r;
  asm("cvt.rna.tf32.f32 %0, %1;" : "=r"(r) : "f"(v));
  return __uint_as_float(r);
}

// operand descriptor: sbo, the bytes from one 8-row group to the next
__device__ __forceinline__ uint64_t xdesc(uint32_t addr, uint32_t sbo) {
  const uint32_t lbo = 128;
  return (uint64_t)((addr >> 4) & 0x3FFF) | ((uint64_t)((lbo >> 4) & 0x3FFF) << 16) |
         ((uint64_t)((sbo >> 4) & 0x3FFF) << 32) | (1ull << 46);
}

// MMAs and their commits are issued by one elected lane in code that the whole
// warp runs, so that the descriptors stay in uniform registers (75 cycles an
// MMA; from one lane's branch, 160 and more)
__device__ __forceinline__ void xcommit(uint64_t* bar) {
  asm volatile(
      "{\n\t.reg .pred e;\n\telect.sync _|e, 0xffffffff;\n\t"
      "@e tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n\t}" ::"r"(
          smem_u32(bar))
      : "memory");
}

__device__ __forceinline__ void xmma(uint32_t d, uint64_t a, uint64_t b, uint32_t idesc,
                                     uint32_t acc) {
  asm volatile(
      "{\n\t.reg .pred p, e;\n\tsetp.ne.u32 p, %4, 0;\n\telect.sync _|e, 0xffffffff;\n\t"
      "@e tcgen05.mma.cta_group::1.kind::tf32 [%0], %1, %2, %3, p;\n\t}" ::"r"(d),
      "l"(a), "l"(b), "r"(idesc), "r"(acc)
      : "memory");
}

// one column of this thread's TMEM lane (complete after xwait_ld)
__device__ __forceinline__ float xld1(uint32_t addr) {
  uint32_t r;
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x1.b32 {%0}, [%1];" : "=r"(r) : "r"(addr));
  return __uint_as_float(r);
}

// row start of the packed factor
__device__ __host__ __forceinline__ int xtri(int i) { return i * (i + 1) / 2; }

// sum_{i=k..j-1} u[i] L_ik over the packed factor, in eight sums (as dot64_ilp8)
__device__ __forceinline__ double xcoldot(const double* u, const double* L, int k, int j) {
  double a[8] = {0.0, 0.0, 0.0, 0.0, 0.0, 0.0, 0.0, 0.0};
  int i = k;
  for (; i + 7 < j; i += 8) {
#pragma unroll
    for (int t = 0; t < 8; ++t) a[t] = fma(u[i + t], L[xtri(i + t) + k], a[t]);
  }
  for (; i < j; ++i) a[0] = fma(u[i], L[xtri(i) + k], a[0]);
  return ((a[0] + a[1]) + (a[2] + a[3])) + ((a[4] + a[5]) + (a[6] + a[7]));
}

// block sums of two values at once (one pass of shuffles and barriers)
// Sums over the block of FP64 terms held only by threads below `active`, to
// thread 0 (other threads keep partial values).  Only the warps holding terms
// shuffle and thread 0 adds the warp totals in warp order: bit-identical to a
// full block sum (the idle warps' totals are exact zeros) at a fraction of its
// FP64 instructions, which are scarce on this part.  Every thread must call.
__device__ __forceinline__ void xsum2_t0(double& a, double& b, int active, double* red) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int aw = min((active + 31) >> 5, XT_THREADS / 32);
  __syncthreads();   // earlier readers of red are done
  if (warp < aw) {
    for (int o = 16; o > 0; o >>= 1) {
      a += __shfl_xor_sync(0xffffffffu, a, o);
      b += __shfl_xor_sync(0xffffffffu, b, o);
    }
    if (lane == 0) { red[2 * warp] = a; red[2 * warp + 1] = b; }
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    double ta = 0.0, tb = 0.0;
    for (int w = 0; w < aw; ++w) { ta += red[2 * w]; tb += red[2 * w + 1]; }
    a = ta;
    b = tb;
  }
}

__device__ __forceinline__ void xsum_t0(double& v, int active, double* red) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int aw = min((active + 31) >> 5, XT_THREADS / 32);
  __syncthreads();
  if (warp < aw) {
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    if (lane == 0) red[warp] = v;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    double t = 0.0;
    for (int w = 0; w < aw; ++w) t += red[w];
    v = t;
  }
}

struct XtSmem {
  static constexpr int B_BYTES = 16 * XT_KMAX * 4;        // rows of L^{-1}, one of hi / lo
  static constexpr int A_BYTES = XT_KC / 8 * XT_SLAB;     // an A piece
  static constexpr int B_OFF = 0;
  static constexpr int A_OFF = 2 * B_BYTES;
  static constexpr int END = A_OFF + XT_RING * A_BYTES;   // 72 KB
};

__global__ void __launch_bounds__(XT_THREADS, 2) exh_tc_kernel(XtParams P) {
  extern __shared__ unsigned char smem_raw[];
  unsigned char* smem = reinterpret_cast<unsigned char*>(
      (reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
  float* Bhi = reinterpret_cast<float*>(smem + XtSmem::B_OFF);
  float* Blo = Bhi + XtSmem::B_BYTES / 4;
  // ld: rows of the packed factor (the part of a mixed launch that runs here
  // has n <= XT_KMAX); ldo: row stride of the per-step outputs
  const int p = P.p, PP = P.PP, ldo = P.n_max, nc_max = P.nc_max;
  const int ld = ldo < XT_KMAX ? ldo : XT_KMAX;
  const int ncp = (nc_max + 3) & ~3;
  // small state after the operands
  float* kap = reinterpret_cast<float*>(smem + XtSmem::END);          // [nc_max]
  float* vsum = kap + ncp;                                           // [nc_max] |w_r|^2
  float* nsum = vsum + ncp;                                          // [nc_max] w_r . z
  float* zf = nsum + ncp;                                            // [XT_KMAX]
  double* S64 = reinterpret_cast<double*>(zf + XT_KMAX);              // [XT_KMAX][p], 16B aligned
  double* kx = S64 + XT_KMAX * p;                                     // [XT_KMAX]
  double* z = kx + XT_KMAX;
  double* zy = z + XT_KMAX;
  double* kv = zy + XT_KMAX;
  double* lv = kv + XT_KMAX;
  double* ys = lv + XT_KMAX;                                          // [XT_KMAX] y of S
  double* red = ys + XT_KMAX;                                         // [8]
  double* Lg = red + 8;                                               // [ld (ld + 1) / 2]
  float* fred = reinterpret_cast<float*>(Lg + xtri(ld));              // [8]
  int* ired = reinterpret_cast<int*>(fred + 8);                       // [8]
  int* sel = ired + 8;                                                // [XT_KMAX]
  unsigned char* used = reinterpret_cast<unsigned char*>(sel + XT_KMAX);
  uint64_t* full = reinterpret_cast<uint64_t*>(
      (reinterpret_cast<uintptr_t>(used + nc_max) + 15) & ~(uintptr_t)15);   // [XT_RING] piece loaded
  uint64_t* freed = full + XT_RING;                                           // [XT_RING] piece used
  uint64_t* gdone = freed + XT_RING;                                          // group's MMAs done
  uint32_t* tbase = reinterpret_cast<uint32_t*>(gdone + 1);

  const int tid = threadIdx.x, lane = tid & 31, warp = __shfl_sync(0xffffffffu, tid >> 5, 0);
  unsigned* s_item = tbase + 1;
  if (tid == 0) {
    for (int b = 0; b < XT_RING; ++b) { mbar_init(&full[b], 1); mbar_init(&freed[b], 1); }
    mbar_init(gdone, 1);
    fence_mbar_init();
  }
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 128;" ::"r"(
        smem_u32(tbase)));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t taddr = *tbase;
  // scratch of this CTA slot; the correlation tiles start zeroed, so that the
  // columns past j and the rows past N' that the MMAs read hold finite values
  const int ntc = (nc_max + 127) / 128;
  float* Kc = P.Kc + (int64_t)blockIdx.x * ntc * 2 * XT_TILE_FLOATS;
  float* crow = P.crow + (int64_t)blockIdx.x * nc_max * PP;
  for (int64_t i = tid; i < (int64_t)ntc * 2 * XT_TILE_FLOATS / 4; i += XT_THREADS)
    reinterpret_cast<float4*>(Kc)[i] = make_float4(0.f, 0.f, 0.f, 0.f);
  asm volatile("fence.proxy.async.global;" ::: "memory");
  __syncthreads();
  // warp 0: pieces copied and pieces whose MMAs were committed, over the
  // kernel's life; piece m uses buffer m % XT_RING in its m / XT_RING-th phase
  uint32_t copied = 0, issued = 0;
  uint32_t gphase = 0;
  const float onepg = (float)(1.0 + P.g);
  const unsigned items = P.count ? *P.count : (unsigned)P.M;
  bool timed_out = false;
  while (!timed_out) {
    if (tid == 0) *s_item = atomicAdd(P.queue, 1u);
    __syncthreads();
    const unsigned it = *s_item;
    __syncthreads();
    if (it >= items) break;
    const int64_t loc = P.order ? (int64_t)P.order[it] : (int64_t)it;
    const double theta = P.theta_loc ? P.theta_loc[loc] : P.theta;
    const float nit = (float)(-1.0 / theta);
    const double nit64 = -1.0 / theta;
    const int nc = P.nc_loc ? P.nc_loc[loc] : nc_max;
    const int n = P.n_loc ? P.n_loc[loc] : P.n_max;
    const int32_t* cl = P.cand + loc * nc_max;
    const double* xq = P.xref + loc * p;

    for (int i = tid; i < 2 * XtSmem::B_BYTES / 4; i += XT_THREADS) Bhi[i] = 0.f;
    // the candidates' FP32 rows, gathered once into the slot in rank order (the
    // correlation column of every step then reads them contiguously), and K(c_r, x)
    for (int r = tid; r < nc; r += XT_THREADS) {
      used[r] = 0;
      vsum[r] = 0.f;
      nsum[r] = 0.f;
      const float* c = P.Xf + (int64_t)cl[r] * PP;
      float d = 0.f;
      for (int k = 0; k < PP; k += 4) {
        const float4 v4 = *reinterpret_cast<const float4*>(c + k);
        *reinterpret_cast<float4*>(crow + (int64_t)r * PP + k) = v4;
      }
      for (int k = 0; k < p; ++k) {
        const float t = c[k] - (float)(xq[k] - P.center[k]);
        d = fmaf(t, t, d);
      }
      kap[r] = __expf(d * nit);
    }
    if (P.tie_gap) for (int i = tid; i < ldo; i += XT_THREADS) P.tie_gap[loc * ldo + i] = 0.0;
    if (P.nevals) for (int i = tid; i < ldo; i += XT_THREADS) P.nevals[loc * ldo + i] = 0;
    __syncthreads();

    int j = 0;
    bool ok = (n >= P.n0) && (n <= nc) && (n <= ld);

    // ---- append candidate rank rr: FP64 factor row, z, L^{-1}y, B row, Kc column ----
    auto add_point = [&](int rr) -> bool {
      const double* c = P.X + (int64_t)cl[rr] * p;
      if (tid < p) S64[j * p + tid] = c[tid];
      if (tid == XT_THREADS - 1) {
        ys[j] = P.Y[cl[rr]];
        sel[j] = rr;
        used[rr] = 1;
      }
      __syncthreads();
      // correlations of the new point with the design, and with x
      if (tid <= j) {
        const double k = corr64_fast(tid < j ? S64 + tid * p : xq, S64 + j * p, p, nit64);
        if (tid < j) kv[tid] = k;
        else kx[j] = k;
      }
      __syncthreads();
      double vv = 0.0;
      if (tid < j) {
        const double acc = dot64_ilp8(Lg + xtri(tid), kv, tid + 1);
        lv[tid] = acc;
        vv = __dmul_rn(acc, acc);
      }
      // thread 0 forms the pivot v = 1 + g - |l|^2 and 1 / sqrt(v)
      xsum_t0(vv, j, red);
      if (tid == 0) {
        const double v = (1.0 + P.g) - vv;
        red[1] = v > 0.0 ? 1.0 / sqrt(v) : 0.0;
        ired[5] = v > 0.0 ? 1 : 0;
      }
      __syncthreads();
      if (!ired[5]) return false;
      const double inv_d = red[1];
      double zz = 0.0, zyy = 0.0;
      if (tid <= j) {
        const double rk = tid < j ? -xcoldot(lv, Lg, tid, j) * inv_d : inv_d;
        Lg[xtri(j) + tid] = rk;
        const float h = xtf32((float)rk);
        const uint32_t off = xcanon(j & 15, tid) >> 2;
        Bhi[off] = h;
        Blo[off] = xtf32((float)(rk - (double)h));
        zz = __dmul_rn(rk, kx[tid]);
        zyy = __dmul_rn(rk, ys[tid]);
      }
      xsum2_t0(zz, zyy, j + 1, red);
      if (tid == 0) {
        z[j] = zz;
        zy[j] = zyy;
        zf[j] = (float)zz;
      }
      // correlation cache column j: K(c_r, S_j) for every candidate, as A operand
      // (TF32 hi / lo) of its tile; then visible to the bulk copies
      const float* sj = crow + (int64_t)rr * PP;
#pragma unroll 4
      for (int q = tid; q < nc; q += XT_THREADS) {
        const float kc = __expf(sqdist_row32(crow + (int64_t)q * PP, sj, PP) * nit);
        const float h = xtf32(kc);
        float* tile = Kc + (int64_t)(q >> 7) * 2 * XT_TILE_FLOATS;
        const uint32_t off = xslab(q & 127, j) >> 2;
        tile[off] = h;
        tile[XT_SLAB / 8 + off] = xtf32(kc - h);
      }
      // this step's generic writes (the B row in shared memory, the cache column
      // in global memory) become visible to the tensor core and the bulk copies
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      asm volatile("fence.proxy.async.global;" ::: "memory");
      __syncthreads();
      ++j;
      return true;
    };

    float best = -1.f, second = -1.f;
    int bi = -1;
    // Columns lo .. j-1 of W (of one block of 16) for every candidate, added to
    // the running sums; this thread's best candidate by the new sums.  False
    // after a wait ran out.
    auto score = [&](int lo) -> bool {
      const int jk = (j + 7) & ~7;                              // K
      const int nch = (jk + XT_KC - 1) / XT_KC;                 // pieces per tile
      const int ntile = (nc + 127) >> 7;
      const uint32_t idesc = (1u << 4) | (2u << 7) | (2u << 10) | ((uint32_t)(16 >> 3) << 17) |
                             ((uint32_t)(128 >> 4) << 24);
      best = -1.f; second = -1.f; bi = -1;
      for (int g0 = 0; g0 < ntile; g0 += XT_GROUP) {
        const int gt = min(XT_GROUP, ntile - g0);
        bool got = true;
        if (warp == 0) {
          const int np = gt * nch;
          auto copy = [&](int m) {
            // piece m of the group, once the MMAs of its buffer's last piece have
            // read it
            const uint32_t b = copied % XT_RING;
            bool go = true;
            if (copied >= XT_RING) go = mbar_wait(&freed[b], ((copied - XT_RING) / XT_RING) & 1u);
            if (!__all_sync(0xffffffffu, go)) return false;
            const int t = g0 + m / nch, c = m % nch;
            const uint32_t bytes = (uint32_t)(min(XT_KC, jk - XT_KC * c) / 8) * XT_SLAB;
            if (lane == 0) {
              mbar_expect_tx(&full[b], bytes);
              bulk_g2s(smem + XtSmem::A_OFF + b * XtSmem::A_BYTES,
                       Kc + (int64_t)t * 2 * XT_TILE_FLOATS + c * (XtSmem::A_BYTES / 4), bytes,
                       &full[b]);
            }
            __syncwarp();
            ++copied;
            return true;
          };
          // copies run two pieces ahead of the MMAs
          for (int m = 0; m < 2 && m < np && got; ++m) got = copy(m);
          for (int m = 0; m < np && got; ++m) {
            if (m + 2 < np) got = copy(m + 2);
            const uint32_t b = issued % XT_RING;
            if (got) got = __all_sync(0xffffffffu, mbar_wait(&full[b], (issued / XT_RING) & 1u));
            if (!got) break;
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            const int c = m % nch;
            const uint32_t d = taddr + (uint32_t)(m / nch) * 16u;
            const uint64_t a0 = xdesc(smem_u32(smem + XtSmem::A_OFF + b * XtSmem::A_BYTES), 256);
            const uint64_t b0 = xdesc(smem_u32(Bhi) + (uint32_t)c * (XT_KC / 4) * 128u,
                                      (XT_KMAX / 4) * 128);
            const int nks = min(XT_KC, jk - XT_KC * c) / 8;
            // (addresses below 256 KB: adding to the address field does not carry)
#pragma unroll
            for (int ks = 0; ks < XT_KC / 8; ++ks) {
              if (ks >= nks) break;
              const uint64_t a_hi = a0 + ks * (XT_SLAB >> 4), a_lo = a_hi + (XT_SLAB >> 5);
              const uint64_t b_hi = b0 + ks * (256 >> 4), b_lo = b_hi + (XtSmem::B_BYTES >> 4);
              xmma(d, a_hi, b_hi, idesc, c + ks > 0 ? 1u : 0u);
              xmma(d, a_hi, b_lo, idesc, 1u);
              xmma(d, a_lo, b_hi, idesc, 1u);
            }
            xcommit(&freed[b]);
            if (m + 1 == np) xcommit(gdone);
            ++issued;
          }
        }
        __syncwarp();
        if (got) got = mbar_wait(gdone, gphase);
        if (!__syncthreads_and(got)) {
          if (tid == 0) atomicOr(P.status, LAGP_DEV_TIMEOUT);
          return false;
        }
        gphase ^= 1u;
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        const uint32_t row = taddr + ((uint32_t)(warp * 32) << 16);
        float vs[XT_GROUP], ns[XT_GROUP];
#pragma unroll
        for (int s = 0; s < XT_GROUP; ++s) {
          const int r = (g0 + s) * 128 + tid;
          vs[s] = r < nc ? vsum[r] : 0.f;
          ns[s] = r < nc ? nsum[r] : 0.f;
        }
        for (int i = lo; i < j; ++i) {
          float w[XT_GROUP];
#pragma unroll
          for (int s = 0; s < XT_GROUP; ++s) {
            w[s] = 0.f;
            if (s < gt) w[s] = xld1(row + (uint32_t)(s * 16 + (i & 15)));
          }
          asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
          const float zi = zf[i];
#pragma unroll
          for (int s = 0; s < XT_GROUP; ++s) {
            vs[s] = fmaf(w[s], w[s], vs[s]);
            ns[s] = fmaf(w[s], zi, ns[s]);
          }
        }
#pragma unroll
        for (int s = 0; s < XT_GROUP; ++s) {
          const int r = (g0 + s) * 128 + tid;
          if (r >= nc) continue;
          vsum[r] = vs[s];
          nsum[r] = ns[s];
          if (used[r]) continue;
          const float v = onepg - vs[s];
          const float num = ns[s] - kap[r];
          const float alc = v > 0.f ? num * num / v : 0.f;
          if (alc > best) { second = best; best = alc; bi = r; }
          else if (alc > second) second = alc;
        }
        asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
        __syncthreads();
      }
      return true;
    };

    // the starting points; their columns of W a block of 16 at a time (the B
    // operand holds one block)
    int scored = 0;
    for (int rr = 0; rr < P.n0 && ok; ++rr) {
      ok = add_point(rr);
      if (ok && ((j & 15) == 0 || j == P.n0) && j < n) {
        if (!score(scored)) { ok = false; timed_out = true; }
        scored = j;
      }
    }

    for (int step = P.n0; step < n && ok; ++step) {
      // block argmax, ties to the lower rank; the second best for the gap
      for (int o = 16; o > 0; o >>= 1) {
        const float ob = __shfl_xor_sync(0xffffffffu, best, o);
        const float os = __shfl_xor_sync(0xffffffffu, second, o);
        const int oi = __shfl_xor_sync(0xffffffffu, bi, o);
        if (ob > best || (ob == best && oi >= 0 && (bi < 0 || oi < bi))) {
          second = fmaxf(best, os); best = ob; bi = oi;
        } else {
          second = fmaxf(second, ob);
        }
      }
      if (lane == 0) { fred[2 * warp] = best; fred[2 * warp + 1] = second; ired[warp] = bi; }
      __syncthreads();
      if (tid == 0) {
        float b = fred[0], s = fred[1];
        int ii = ired[0];
        for (int w = 1; w < XT_THREADS / 32; ++w) {
          const float ob = fred[2 * w], os = fred[2 * w + 1];
          const int oi = ired[w];
          if (ob > b || (ob == b && oi >= 0 && (ii < 0 || oi < ii))) { s = fmaxf(b, os); b = ob; ii = oi; }
          else s = fmaxf(s, ob);
        }
        ired[4] = ii;
        if (P.tie_gap) P.tie_gap[loc * ldo + (step - P.n0)] = (b > 0.f && s >= 0.f) ? (double)((b - s) / b) : 0.0;
      }
      __syncthreads();
      const int pick = ired[4];
      ok = (pick >= 0) && add_point(pick);
      if (ok && j < n) {
        if (!score(scored)) { ok = false; timed_out = true; }
        scored = j;
      }
    }

    if (ok) {
      double a = 0.0, b = 0.0, c = 0.0;
      if (tid < j) {
        a = __dmul_rn(z[tid], zy[tid]);
        b = __dmul_rn(zy[tid], zy[tid]);
        c = __dmul_rn(z[tid], z[tid]);
      }
      xsum2_t0(a, b, j, red);
      xsum_t0(c, j, red + 4);
      if (tid == 0) {
        P.mean[loc] = a;
        P.s2[loc] = b * ((1.0 + P.g) - c) / (double)j;
      }
    } else if (tid == 0) {
      P.mean[loc] = __longlong_as_double(0x7ff8000000000000ll);
      P.s2[loc] = __longlong_as_double(0x7ff8000000000000ll);
      atomicOr(P.status, LAGP_DEV_BAD_UPDATE);
    }
    if (P.selected)
      for (int i = tid; i < ldo; i += XT_THREADS) P.selected[loc * ldo + i] = (i < j) ? cl[sel[i]] : -1;
    if (P.promote && tid == 0) {
      // smallest binary64 pivot v of the design: the factor's diagonal holds
      // 1 / sqrt(v); a failed update promotes the location
      double vm = ok ? INFINITY : -1.0;
      for (int i = 0; i < j; ++i) {
        const double dg = Lg[xtri(i) + i];
        vm = fmin(vm, 1.0 / (dg * dg));
      }
      promote_location(P.promote, P.promote_count, loc, vm);
    }
  }
  // after a timeout: wait (bounded) for the copies and MMAs still in flight
  if (timed_out && tid == 0) {
    for (uint32_t m = issued; m < copied; ++m)
      mbar_wait(&full[m % XT_RING], (m / XT_RING) & 1u);
    if (issued > 0) mbar_wait(&freed[(issued - 1) % XT_RING], ((issued - 1) / XT_RING) & 1u);
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (warp == 0) {
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 128;" ::"r"(taddr));
  }
}

int exh_tc_max_n() { return XT_KMAX; }

size_t exh_tc_cache_floats(int nc_max) { return (size_t)((nc_max + 127) / 128) * 2 * XT_TILE_FLOATS; }

cudaError_t launch_exh_tc(const DesignArgs& a, cudaStream_t s) {
  XtParams P;
  P.X = a.X; P.Y = a.Y; P.p = a.p; P.PP = a.PP; P.Xf = a.ws->Xf; P.xref = a.xref; P.M = a.M;
  P.cand = a.cand; P.nc_max = a.nc_max; P.nc_loc = a.nc_loc; P.n0 = a.n0; P.n_max = a.n_max;
  P.n_loc = a.n_loc; P.theta = a.theta; P.theta_loc = a.theta_loc; P.g = a.g; P.center = a.ws->center; P.mean = a.mean;
  P.s2 = a.s2; P.selected = a.selected; P.tie_gap = a.tie_gap; P.nevals = a.nevals;
  P.Kc = a.ws->state32; P.status = a.ws->status;
  P.queue = a.ws->queue + 1; P.order = a.order; P.count = a.count;
  P.crow = a.ws->crow;
  P.promote = a.promote ? a.ws->promote : nullptr;
  P.promote_count = a.ws->status + 1;
  const int ld = a.n_max < XT_KMAX ? a.n_max : XT_KMAX;
  const size_t small = 3 * (size_t)((a.nc_max + 3) & ~3) * 4 + XT_KMAX * 4 +
                       (size_t)XT_KMAX * a.p * 8 + 6 * XT_KMAX * 8 + 8 * 8 + (size_t)xtri(ld) * 8 +
                       8 * 4 + 8 * 4 + XT_KMAX * 4 + a.nc_max + 16 + (2 * XT_RING + 1) * 8 + 16;
  const size_t sm = 1024 + XtSmem::END + small;
  cudaError_t err =
      cudaFuncSetAttribute(exh_tc_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
  if (err != cudaSuccess) return err;
  const int64_t grid = persistent_grid(exh_tc_kernel, XT_THREADS, sm, a.M, exh_slots(a.ws->chunk), 1,
                                       a.tune.exh_occ);
  if (grid < 0) return cudaErrorInvalidValue;
  if ((err = cudaMemsetAsync(P.queue, 0, sizeof(unsigned), s)) != cudaSuccess) return err;
  prof_begin("exh_tc", s);
  exh_tc_kernel<<<(unsigned)grid, XT_THREADS, sm, s>>>(P);
  prof_end(s);
  return cudaGetLastError();
}

}  // namespace lagp
