// Dependent adjoint steps in one launch: what a launch is told, and which of its rows other rows of it read (host code without CUDA
// headers, and the kernel's wait).
#pragma once
#include <stdint.h>

#ifdef __CUDACC__
#define MG_HOST_DEVICE __host__ __device__ __forceinline__
#else
#define MG_HOST_DEVICE inline
#endif

struct __nv_bfloat16;

namespace mg {

typedef long long i64;

// ---- n dependent adjoint steps over the same rows (k, b) in ONE launch (bf16 operands); step 0 starts from the rows lin, every
// other one from its predecessor's results.
struct AdjSweepStep {
  float* out; i64 out_ks;          // result rows (+ k*out_ks + b*H)
  const float* g; i64 g_ks;        // optional source rows
  i64 coff;                        // coefficient rows of k = 0 (offset into the level's arrays)
  const float* ladd; i64 ladd_ks;  // optional rows that join the incoming sensitivities (stacked layers)
  int nk;                          // rows with k < nk take the step; never more than the step before
  int ahead;                       // set by plan_adj_sweep(): row r of the step replaces what row r + ahead started from; 0: nobody's
};
constexpr int kMaxAdjSweepSteps = 20;
struct AdjSweepArgs {
  int B, H, n;
  const float* lin; i64 lin_ks;
  const float* a; const __nv_bfloat16 *cr, *cz, *cn; i64 coef_ks;
  AdjSweepStep st[kMaxAdjSweepSteps];
};

// Do two sets of rows (row k: len elements from p + k*ps on) share no element?  (May answer no where the strides differ.)
inline bool rows_apart(const float* p, i64 ps, int pn, const float* q, i64 qs, int qn, i64 len) {
  if (pn < 1 || qn < 1) return true;
  const i64 d = ((i64)(intptr_t)p - (i64)(intptr_t)q) / (i64)sizeof(float);      // p in elements from q
  const i64 pl = ps * (pn - 1), ql = qs * (qn - 1);
  const i64 p0 = d + (pl < 0 ? pl : 0), p1 = d + (pl > 0 ? pl : 0) + len, q0 = ql < 0 ? ql : 0, q1 = (ql > 0 ? ql : 0) + len;
  if (p1 <= q0 || q1 <= p0) return true;
  if (ps != qs || ps < len) return false;
  const i64 r = (d % ps + ps) % ps;
  return r >= len && r <= ps - len;
}

// Rows take their steps at different times: whatever one row writes and another one reads has to be ordered.  A launch can order one
// such case: its last step may replace the rows that the NEXT interval started from (the C-step behind F-steps); `ahead` then tells
// the kernel which rows must have taken their first step before the results are stored.  false: any other overlap, not one launch.
inline bool plan_adj_sweep(AdjSweepArgs* a) {
  const i64 len = (i64)a->B * a->H;
  for (int i = 0; i < a->n; ++i) {
    AdjSweepStep& t = a->st[i];
    t.ahead = 0;
    if (!rows_apart(t.out, t.out_ks, t.nk, a->lin, a->lin_ks, a->st[0].nk, len)) {
      if (i == 0 || i + 1 < a->n || t.out_ks != a->lin_ks || a->lin_ks < len || t.out != a->lin + a->lin_ks) return false;
      t.ahead = a->B;
    }
    for (int j = 0; j < a->n; ++j) {
      const AdjSweepStep& o = a->st[j];
      if (j < i && !rows_apart(t.out, t.out_ks, t.nk, o.out, o.out_ks, o.nk, len)) return false;
      if (o.g && !rows_apart(t.out, t.out_ks, t.nk, o.g, o.g_ks, o.nk, len)) return false;
      if (o.ladd && !rows_apart(t.out, t.out_ks, t.nk, o.ladd, o.ladd_ks, o.nk, len)) return false;
    }
  }
  return true;
}

// CTAs per cluster for steps of M rows, or 0: step by step.  clusters4, clusters2: clusters of four and two that are resident at a time.
// Both ways go in jumps.  A launch walks its row tiles of 128 in rounds of as many as there are lane groups (33 clusters of four or 74
// of two over the column tiles).  A step by itself is a product of 128 x 64 tiles: one wave on 148 SMs, the reduction split by two
// where they fit twice.  us an adjoint cycle of a two-level solve (cf = 4, 8 rows a point, 11 steps; from a graph), step by step / here:
//   1 round against a split wave: H = 1024, 512 rows 250 / 250; 896 260 / 254; 768 243 / 239; 704 234 / 233; 640 225 / 227; 576 217 / 220
//   2 rounds:                     H = 896, 640 rows 306 / 314; 768, 768 rows 318 / 328; 640, 896 rows 328 / 343
//   2 rounds against one wave:    H = 1024, 640 rows 363 / 317, 1024 467 / 433; 768, 896 rows 408 / 377; 576, 1536 rows 523 / 509
//   3 rounds:                     H = 1024, 1152 rows 506 / 504; 832 496 / 508; 768, 1408 rows 548 / 563; 640, 1664 rows 577 / 596
//   3, 4 rounds against two:      H = 1024, 1280 rows 610 / 554, 2048 866 / 812; 768, 1664 rows 701 / 656; 640, 2048 rows 752 / 710
// (3072 rows at H = 1024, the larger tiles of many rows: 880 / 910.)  With half the clusters' CTAs a round takes twice as long:
//   1 round against a split wave: H = 384, 1536 rows 422 / 436; 320, 1792 rows 451 / 466
//   1 round against one wave:     H = 512, 1536 rows 454 / 440; 448, 2048 rows 598 / 593; 320, 2048 rows 543 / 532
//   2 rounds:                     H = 448, 2560 rows 461 / 494; 320, 3584 rows 521 / 563
//   2 rounds against two:         H = 512, 4096 rows 703 / 674; 384, 3328 rows 582 / 575; 320, 4096 rows 617 / 620
// Coarsening by eight, two thirds more steps a launch, has the same signs (H = 1024, 640 rows 1.29 times faster, 1024 rows 1.22, one
// round 1.04 to 1.07).  Few rows are all latency, but at H = 1024 alone eight CTAs of a cluster have two units each to reduce:
// 8 / 32 / 64 rows 83 / 77, 90 / 86, 98 / 95 (cf = 8: 147 / 122, 155 / 134, 165 / 147); H = 960 81 / 77, 79 / 86, 90 / 95.
inline int adj_sweep_split(int H, int M, int clusters4, int clusters2) {
  const int nb = H / 64, mt = (M + 127) / 128, ncol = (H + 127) / 128, tiles = mt * nb;
  auto rounds = [&](int clusters) { return clusters >= ncol ? (mt + clusters / ncol - 1) / (clusters / ncol) : 1 << 20; };
  if (nb == 16 && M <= 64) return 8;
  if (nb >= 9 && nb <= 16 && M >= 512 && M <= 2048)
    return rounds(clusters4) <= (tiles > 148 ? 4 : tiles > 74 ? 2 : nb > 10 ? 1 : 0) ? 4 : 0;
  if (nb >= 5 && nb <= 8 && M >= 1536 && M <= 4096)
    return rounds(clusters2) <= (tiles > 148 ? (nb > 5 ? 2 : 0) : tiles > 74 ? 1 : 0) ? 2 : 0;
  return 0;
}

// Tiles of `nr` rows that hold the rows which start from what rows r0 .. r0 + 3 of a step (of M rows) replace: lo .. hi, none if hi < lo.
MG_HOST_DEVICE void tiles_ahead(int r0, int M, int ahead, int nr, int* lo, int* hi) {
  const int last = r0 + 3 < M ? r0 + 3 : M - 1;
  *lo = (r0 + ahead) / nr;
  *hi = r0 < M ? (last + ahead) / nr : *lo - 1;
}

}  // namespace mg
