// Interface of the fp32 multigrid solve as one persistent launch (f32_solve.cu).
#pragma once
#include "common.cuh"

namespace mg {

// One phase of a solve: chains of dependent steps for independent rows (k, b), k < nk.  A row loads its state from
// src + k*src_ks + b*H (optionally copying it to copy + k*copy_ks), takes n steps (ntail for k >= nfull; step j writes
// out + k*out_ks + j*out_ss and adds g + k*g_ks + j*g_ss) and, for k < nfull, a closing step of the given kind:
//   kLastNone   nothing
//   kLastStore  one more step, result to last + k*last_ks                                          (C-relaxation)
//   kLastCoarse one more step v; the C-point uc + k*uc_ks goes to ucd + k*ucd_ks (unless ucd is null: it is there already),
//               |uc - v|^2 to *acc (optional), and last + k*last_ks = v - (coarse step from src2 + k*src2_ks)
// op / op_ks / op_ss: element offset of the step's operands, into the projection (forward, rows of 3H) or into the level's
// coefficient arrays (adjoint, rows of H); op2 / op2_ks the same for the coarse step on level + 1.
// Within a phase no row may read what another row of the phase writes; the phases are separated by a grid barrier.
enum { kLastNone = 0, kLastStore = 1, kLastCoarse = 2 };
struct F32Phase {
  int nk, nfull, n, ntail, last_kind, level;
  float gamma, gamma2;
  int R;                          // rows per block: set by the launcher
  const float* src; i64 src_ks;
  float* copy; i64 copy_ks;
  float* out; i64 out_ks, out_ss;
  const float* g; i64 g_ks, g_ss;
  i64 op, op_ks, op_ss;
  float* last; i64 last_ks;
  const float* src2; i64 src2_ks;
  const float* uc; i64 uc_ks; float* ucd; i64 ucd_ks;
  i64 op2, op2_ks;
  double* acc;
};
constexpr int kF32MaxPhases = 40, kF32Levels = 16;
struct F32Args {
  int B, H, cell, nph;
  const float* W;                          // [3H, H]
  const float *gi, *b_hh;                  // forward
  const float* coef[kF32Levels][4];        // adjoint: a, c_r, c_z, c_n of every level
  unsigned* bar;                           // barrier counter, cleared by the caller
  unsigned* progress;                      // counts up while a phase lasts (any start value)
  unsigned long long limit_ns;             // longest wait without progress: set by the launcher
  F32Phase ph[kF32MaxPhases];
};
// does a solve over rows of this width fit (weights of a cluster of CTAs resident in shared memory)?
bool f32_solve_fits(int H);
// false: not available (the cooperative cluster launch was refused); nothing has been enqueued then
bool f32_solve(bool adjoint, F32Args& a, cudaStream_t s);
bool f32_linearise(const LinArgs* levels, int n, cudaStream_t s);
int f32_device_status();
int f32_clear_device_status();

}  // namespace mg
