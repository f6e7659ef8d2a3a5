// ray32_layout.h -- shared-memory layout of one warp (one location) of the
// FP32-scoring ray kernel, and the index arithmetic of its row storage.  Free
// of CUDA so that the host tests compile it; KD_STACK (the k-d tree walk's
// visits in progress, 32 box distances each) comes from kdtree.cuh, or from the
// compiler's command line.
#pragma once

#ifndef KD_STACK
#error "KD_STACK must be defined before ray32_layout.h"
#endif

#if defined(__CUDACC__)
#define LAGP_HD __device__ __host__ __forceinline__
#define LAGP_HDI __host__ __device__ inline
#else
#define LAGP_HD inline
#define LAGP_HDI inline
#endif

namespace lagp {

// start of row i if rows of i + 1 elements were only padded to quads: what the storage
// below is measured against in the tests
LAGP_HD int roff(int i) {
  const int a = i >> 2, b = i & 3;
  return 4 * (i + 2 * a * (a - 1) + a * b);
}
LAGP_HD int tri(int i) { return i * (i + 1) / 2; }
// The inverse factor's FP32 rows as the scoring product reads them: four rows
// 4u .. 4u+3 form a block of u + 1 quads per row, with the rows' k-th quads
// side by side, so that the four lanes of a ray read 64 contiguous bytes.  A
// ragged last block past row 32 holds only the rows it has (a design of 50
// points then takes what plain rows would).  lf_stride(u, n) is the words from
// one quad of a row to its next, lf_at(i, k, n) the word of element (i, k) and
// lf_words(n) the words of n rows.
LAGP_HD int lf_block(int u) { return 8 * u * (u + 1); }
LAGP_HD int lf_stride(int u, int n) { return (u >= 8 && 4 * u + 4 > n) ? 4 * (n - 4 * u) : 16; }
LAGP_HD int lf_at(int i, int k, int n) {
  return lf_block(i >> 2) + lf_stride(i >> 2, n) * (k >> 2) + 4 * (i & 3) + (k & 3);
}
LAGP_HD int lf_words(int n) {
  const int u = (n - 1) >> 2;
  return lf_block(u) + lf_stride(u, n) * (u + 1);
}
// row length of the kz buffer: a multiple of 4 whose quarter is odd, so that
// the rays' float4 reads fall on different banks
LAGP_HD int kz_ld(int n) {
  int k = (n + 3) & ~3;
  if (((k >> 2) & 1) == 0) k += 4;
  return k;
}

struct WarpLayout {
  int lf, kz, cb, zf, tau, x, gsel, stk, bnd, starts, mask, smask, vm, bytes;
};

LAGP_HDI WarpLayout warp_layout(int n, int PP, int RP, int nc) {
  WarpLayout w;
  int off = 0;   // in 4-byte words, float region first (16-byte aligned pieces)
  auto take = [&](int words) { int o = off; off += (words + 3) & ~3; return o; };
  w.lf = take(lf_words(n));
  w.kz = take(RP * kz_ld(n));
  // per-ray exponent coefficients c_k then b_k (rows of kz_ld(n)); the k-d
  // tree walk of the full-scope snap (nodes, then their box distances) and
  // the factor update's two binary64 work vectors (n each) run after the
  // step's evaluations and reuse this space
  const int cbw = 2 * RP * kz_ld(n);
  w.cb = take(cbw > 33 * KD_STACK ? cbw : 33 * KD_STACK);
  w.stk = w.cb;
  w.bnd = w.cb + KD_STACK;
  w.zf = take((n + 3) & ~3);
  w.tau = take(RP);            // each ray's segment: end = a + tau * 10 (a - x)
  w.x = take(4 * PP);          // xf, lof, hif, xs
  w.gsel = take(n);            // design indices of the selected points
  w.starts = take(RP);
  w.mask = take((nc + 31) / 32);
  w.smask = take((nc + 31) / 32);
  w.vm = take(2);              // smallest binary64 pivot of the location (lane 0)
  w.bytes = off * 4;
  return w;
}

}  // namespace lagp
