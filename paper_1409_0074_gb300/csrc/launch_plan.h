// launch_plan.h -- host-side launch arithmetic of the persistent and tiled
// kernels, kept free of CUDA so that it compiles and is tested on any host.
#pragma once
#include <cmath>
#include <cstddef>
#include <cstdint>

namespace lagp {

// The tensor-core kNN filter runs one CTA per SM (it takes all 512 TMEM
// columns) over `tiles` location tiles, each streaming `design_tiles` design
// tiles.  Tiles [0, *body) run unsplit in whole waves; the remaining
// tiles - *body run with the design split into *nseg segments (one CTA
// each).  A batch with fewer tiles than SMs splits every tile, about two CTAs
// per SM; a larger batch splits the tiles of its last, partial wave over the
// SMs that wave would leave idle.  A segment keeps at least 64 design tiles.
inline void knn_tc_plan(int64_t tiles, int64_t sms, int64_t design_tiles, int64_t* body,
                        int64_t* nseg) {
  int64_t b = tiles, s = 1;
  if (tiles > 0 && tiles < sms) {
    s = (2 * sms + tiles - 1) / tiles;
    b = 0;
  } else if (sms > 0 && tiles % sms != 0) {
    s = sms / (tiles % sms);
    b = tiles - tiles % sms;
  }
  if (s > design_tiles / 64) s = design_tiles / 64;
  if (s > 65535) s = 65535;
  if (s < 2) { s = 1; b = tiles; }
  *body = b;
  *nseg = s;
}

// Warps per CTA (2, 4 or 1) of a kernel whose warps each take `warp_bytes` of
// shared memory, so that the most warps reside on an SM with `smem_sm` bytes
// and `reserved` bytes per CTA, under a bound of `max_warps` per SM; ties go
// to 2, then 4, then 1.
inline int warps_per_cta_for_residency(size_t warp_bytes, size_t smem_sm, size_t reserved,
                                       int max_warps) {
  int best = 2, best_warps = -1;
  const int choices[3] = {2, 4, 1};
  for (int c = 0; c < 3; ++c) {
    const int rw = choices[c];
    int ctas = (int)(smem_sm / (rw * warp_bytes + reserved));
    if (ctas > max_warps / rw) ctas = max_warps / rw;
    if (ctas * rw > best_warps) {
      best_warps = ctas * rw;
      best = rw;
    }
  }
  return best;
}

// Threads of a block of the local inference for the lengthscale (the results are
// the same).  10,000 locations with 128 against 256: 13.6 and 25.2 ms at n = 2,
// 10.3 and 18.4 at n = 10, 17.6 and 27.2 at n = 24; one location 0.56 and 0.70, 1.03
// and 1.17, 0.79 and 0.82 ms.  From n = 28 on a single wave is faster with 256 (150
// locations 2.63 against 2.65 ms, at n = 33 3.19 against 3.37).
inline int mle_threads(int n) { return n <= 24 ? 128 : 256; }

// Warps of a block of the binary64 exhaustive search (the few locations of a batch
// that leaves at most one block per SM aside).  Candidates for four warps at most take
// four, and twice the blocks fit: with four and with eight warps 2,000 locations take
// 4.11 and 6.73 ms at n = N' = 30, 5.84 and 7.52 at N' = 60, n = 30, 342 and 347 at N' =
// 128, n = 100; one location at N' = 60, n = 30 1.30 and 1.34.  Where the matrix update
// is most of a step and the blocks are few, it wants the threads: 400 locations at N' =
// 60, n = 50 7.29 and 6.27 ms (900 there 9.33 and 12.53), one at N' = 90, n = 60 8.39
// and 6.67.
inline int d64_warps(int64_t M, int n, int nc_max, int64_t sms) {
  return nc_max <= 128 && (n <= 32 || M > 4 * sms) ? 4 : 8;
}

// Whether the binary64 exhaustive search forms its products on the integer units.
// That halves what a term costs where the binary64 pipe is busy; where each of an SM's
// four sub-partitions has candidates for one warp at most, a term costs its latency,
// which is longer: with the pipe's products 100 locations (p = 4, n = 30) take 1.59
// and with the integer units' 1.76 ms at N' = 60, 1.74 and 1.84 at 128, but 2.22 and
// 2.00 at 200; 304 locations 1.76 and 1.96 at N' = 60, but 2.63 and 2.17 at 100.
inline bool d64_ints(int64_t M, int nc_max, int64_t sms) {
  const int64_t per_sm = (M + sms - 1) / sms;
  return per_sm > 2 || per_sm * ((nc_max + 31) / 32) > 4;
}

// Threads of a block of the incremental exhaustive scorer, which has 1,024 per SM.
// Four candidates per thread leave most of 256 threads idle for small N', and four
// blocks per SM hide less of a step's latencies than eight: 20,000 locations (p = 4,
// n = 50) take 6.2 with 128 threads and 8.9 ms with 256 at N' = 60, 13.6 and 18.5 at
// 200, 15.6 and 20.4 at 512; 700 locations 0.69 and 0.92, 1.10 and 1.58, 1.36 and 1.86.
// Batches that fit on the SMs either way: N' = 200 0.96 and 0.97 ms at 300 locations,
// N' = 256 1.03 and 1.01, N' = 512 0.70 and 0.67 for one.
inline int d32_threads(int64_t M, int nc_max, int64_t sms) {
  return nc_max <= 200 || (nc_max <= 512 && M > 4 * sms) ? 128 : 256;
}

// Threads of a block of the exact ranking.  A short list is a chain of latencies
// that more blocks per SM hide, and its network is short: 20,000 locations at p = 4
// take 0.049 ms with 128 threads and 0.178 with 256 and a network of 256 at N' = 30,
// 0.070 and 0.186 at N' = 100; at N' = 200 0.147 and 0.184, but one location there
// 10.1 us and 8.2.
inline int rank_threads(int nc_max) { return nc_max <= 128 ? 128 : 256; }

// Sample rows of the kNN pilot.
inline int64_t knn_sample(int64_t N) { return N / 16 < 32768 ? N / 16 : 32768; }
// The tensor-core filter, and the sizes below it whose stream may take a pilot
// threshold too.
inline bool knn_uses_tc(int64_t N, int nc_max) { return N >= (int64_t)32 * nc_max; }
inline bool knn_mid(int64_t N, int nc_max) { return N >= (int64_t)4 * nc_max && N >= 1024; }

// Whether the pilot takes a block per location (knn_pilot1) instead of one per 32
// (knn_pilot), of S sample rows padded to PP coordinates: by the lines through what
// both took, in microseconds.  A block per location: 23 for up to one location per
// SM at S = 68 (p = 4), 31 at 6,250 (p = 8), 57 at 32,768, and for two per SM 41, 57
// and 109.  A block per 32: 12 at S = 68, 26 at 1,250 and 65 at 6,250 (p = 4), 35, 94
// and (at 18,750) 287 at p = 8, for any batch of up to 32 locations per SM.
inline bool knn_pilot_alone(int64_t M, int64_t S, int PP, int64_t sms) {
  const double per_sm = (double)((M + sms - 1) / sms);
  return 2.0 + per_sm * (21.0 + S / 960.0) < 9.0 + 0.75 * PP + S * (3.2 + 1.35 * PP) * 1e-3;
}

// Entries of a location's kNN candidate buffer.  It needs room for N'
// survivors, a whole tile of 256 new inserts before the next compaction, and
// N'/2 (at least 64) entries of slack for distances within the error margin of
// the N'-th; a power of two, as the bitonic sort of knn_rank wants.
inline int knn_cap_least(int nc_max) {
  const int need = (5 * nc_max) / 2 + 256;
  int cap = 512;
  while (cap < need) cap <<= 1;
  return cap;
}
// With a pilot threshold it is also to hold the points that the threshold is
// expected to admit and the two tiles that the pilot asks for beside them.
// Without that room, as for N' <= 307 at N = 1e6, the pilot gives no threshold
// and every location streams the whole design from infinity: 5.2 ms for one
// location and 9.5 ms for 10,000 at N' = 250, p = 4, where the tensor-core filter
// takes 0.035 and 4.0 ms.  The lists are the same either way, so a call whose
// workspace has no room for these buffers runs with the smallest ones.
inline int knn_cap(int nc_max, int64_t N) {
  int cap = knn_cap_least(nc_max);
  if (knn_uses_tc(N, nc_max) || knn_mid(N, nc_max)) {
    const double ratio = (double)N / (double)knn_sample(N), lam = nc_max / ratio;
    const double admits = (lam + 4.5 * std::sqrt(lam) + 6.0) * ratio;
    int more = cap;
    while (more < 16384 && admits > more - 512) more <<= 1;
    if (admits <= more - 512) cap = more;
  }
  return cap;
}

}  // namespace lagp
