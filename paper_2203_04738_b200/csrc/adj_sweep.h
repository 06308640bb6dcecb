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

// Tiles of `nr` rows that hold the rows which start from what rows r0 .. r0 + 3 of a step (of M rows) replace: lo .. hi, none if hi < lo.
MG_HOST_DEVICE void tiles_ahead(int r0, int M, int ahead, int nr, int* lo, int* hi) {
  const int last = r0 + 3 < M ? r0 + 3 : M - 1;
  *lo = (r0 + ahead) / nr;
  *hi = r0 < M ? (last + ahead) / nr : *lo - 1;
}

}  // namespace mg
