// C ABI, argument validation, workspace layout and the host side of the multigrid cycle.
// The cycle logic is written once over an abstract "step" and instantiated for the forward
// recurrence and for its adjoint; every step, transfer and reduction is a kernel launch.
#include <limits.h>
#include <math.h>
#include <stdio.h>
#include <string.h>

#include <vector>

#include "common.cuh"
#include "f32_solve.cuh"
#include "serial_engine.cuh"
#include "umma_engine.cuh"

namespace mg {

std::atomic<unsigned long long> g_kernel_launches{0};
bool g_prof_on = false;

namespace {
struct ProfRec { int kc; double flops; cudaEvent_t e0, e1; };
std::vector<ProfRec> g_prof_recs;
std::vector<cudaEvent_t> g_prof_pool;
cudaEvent_t prof_event() {
  cudaEvent_t e = nullptr;
  if (!g_prof_pool.empty()) { e = g_prof_pool.back(); g_prof_pool.pop_back(); }
  else cudaEventCreate(&e);
  return e;
}
}  // namespace

static int g_prof_depth = 0;
void prof_begin(int kc, double flops, cudaStream_t s) {
  if (!g_prof_on) return;
  if (g_prof_depth++ > 0) return;     // inside an open record
  ProfRec r{kc, flops, prof_event(), prof_event()};
  cudaEventRecord(r.e0, s);
  g_prof_recs.push_back(r);
}
void prof_end(cudaStream_t s) {
  if (!g_prof_on || g_prof_depth == 0) return;
  if (--g_prof_depth > 0 || g_prof_recs.empty()) return;
  cudaEventRecord(g_prof_recs.back().e1, s);
}

namespace {

constexpr int kMaxLevels = 16;

struct Ws {  // bump allocator over the caller's workspace; base == nullptr only counts bytes
  char* base; size_t size; size_t off;
  template <class T> T* take(size_t n) {
    size_t bytes = (n * sizeof(T) + 255) & ~(size_t)255;
    T* p = base ? reinterpret_cast<T*>(base + off) : nullptr;
    off += bytes;
    return p;
  }
  bool fits() const { return base == nullptr || off <= size; }
};

struct Hier {
  int L; int N[kMaxLevels]; i64 stride_t[kMaxLevels]; float gamma[kMaxLevels];
  i64 rem[kMaxLevels];   // T - stride_t * N: fine steps before the first reversed (adjoint) point of the level; 0 unless T is ragged
};

// every data pointer must be 32-byte aligned (nullptr passes: optional arguments are checked for presence elsewhere)
template <class... P>
bool aligned32(P... ptrs) {
  uintptr_t m = 0;
  ((m |= (uintptr_t)(const void*)ptrs), ...);
  return (m & 31u) == 0;
}

inline bool is_tf32(const mgrit_gru_cfg* c) { return c->operands == MGRIT_OPERANDS_TF32 || c->operands == MGRIT_OPERANDS_TF32_1PASS; }

int check_cfg(const mgrit_gru_cfg* c, Hier* hr) {
  if (!c) return MGRIT_INVALID_ARG;
  if (c->T <= 0 || c->B <= 0 || c->I <= 0 || c->H <= 0 || c->levels < 1 || c->levels > kMaxLevels) return MGRIT_INVALID_ARG;
  if (c->levels > 1 && (c->cf < 2 || c->iters < 0)) return MGRIT_INVALID_ARG;
  if (c->cell != MGRIT_CELL_CLASSIC && c->cell != MGRIT_CELL_IMPLICIT) return MGRIT_INVALID_ARG;
  if (c->relax_fine < MGRIT_RELAX_F || c->relax_fine > MGRIT_RELAX_MAX) return MGRIT_INVALID_ARG;
  if (c->relax_coarse < MGRIT_RELAX_F || c->relax_coarse > MGRIT_RELAX_MAX) return MGRIT_INVALID_ARG;
  if (c->operands < MGRIT_OPERANDS_FP32 || c->operands > MGRIT_OPERANDS_TF32_1PASS) return MGRIT_INVALID_ARG;
  if (!(c->dt > 0.f)) return MGRIT_INVALID_ARG;
  if (c->H % 8 != 0 || c->I % 8 != 0) return MGRIT_UNSUPPORTED;
  // row counts (T+1)*B, widths and grid sizes are 32-bit inside the kernels; element offsets are 64-bit
  if (((i64)c->T + 1) * c->B > (i64)INT_MAX - 1024 || (i64)3 * c->H > INT_MAX / 4 || c->I > INT_MAX / 4) return MGRIT_UNSUPPORTED;
  i64 m = 1;
  hr->L = c->levels;
  const bool ragged = (c->flags & MGRIT_FLAG_RAGGED_T) != 0;
  for (int l = 0; l < c->levels; ++l) {
    // ragged: the C-points of a level are its points 0, cf, 2 cf, ...; N_{l+1} = floor(N_l / cf) = floor(T / cf^(l+1))
    if (!ragged && c->T % m != 0) return MGRIT_NOT_DIVISIBLE;
    hr->N[l] = (int)(c->T / m);
    hr->stride_t[l] = m;
    hr->gamma[l] = (float)m * c->dt;
    hr->rem[l] = c->T - m * hr->N[l];
    if (l + 1 < c->levels) {
      m *= c->cf;
      if (m > c->T) return MGRIT_NOT_DIVISIBLE;
    }
  }
  if (c->operands == MGRIT_OPERANDS_BF16) {
    int rc = umma_supported(c);
    if (rc != MGRIT_OK) return rc;
  }
  if (is_tf32(c)) {
    int rc = tf32_supported(c);
    if (rc != MGRIT_OK) return rc;
  }
  return MGRIT_OK;
}

// With MGRIT_FLAG_GI_CARRIES_COPIES the caller's gi buffer is followed by the bf16 copies that the forward call makes
// anyway and the adjoint call needs again: x as [T*B, I] and the level-0 state [h_0; h] as [(T+1)*B, H].
struct GiTail { __nv_bfloat16* xb; __nv_bfloat16* hb0; __nv_bfloat16* gib; size_t total_bytes; };
GiTail gi_tail(const mgrit_gru_cfg* c, float* gi) {
  const size_t TB = (size_t)c->T * c->B;
  size_t off = (TB * 3 * c->H * sizeof(float) + 255) & ~(size_t)255;
  GiTail t;
  t.xb = gi ? reinterpret_cast<__nv_bfloat16*>(reinterpret_cast<char*>(gi) + off) : nullptr;
  off += (TB * c->I * sizeof(__nv_bfloat16) + 255) & ~(size_t)255;
  t.hb0 = gi ? reinterpret_cast<__nv_bfloat16*>(reinterpret_cast<char*>(gi) + off) : nullptr;
  off += ((TB + c->B) * c->H * sizeof(__nv_bfloat16) + 255) & ~(size_t)255;
  t.gib = gi ? reinterpret_cast<__nv_bfloat16*>(reinterpret_cast<char*>(gi) + off) : nullptr;      // the projection itself as bf16
  off += (TB * 3 * c->H * sizeof(__nv_bfloat16) + 255) & ~(size_t)255;
  t.total_bytes = off;
  return t;
}
// The copies exist when the tensor-core engine keeps bf16 shadows of the level states in an MGRIT solve and B divides 128: for other
// batch sizes the flag's contract says that it is ignored, so that a buffer of the projection's size and one that another call
// filled (gru_input_projection, the serial sweep) serve there.
bool carries_copies(const mgrit_gru_cfg* c, bool serial) {
  return !serial && (c->flags & MGRIT_FLAG_GI_CARRIES_COPIES) && c->operands == MGRIT_OPERANDS_BF16 && 128 % c->B == 0 && c->levels > 1;
}

// MGRIT_GRU_GI_BF16=0 in the environment keeps the fused kernels on the fp32 input projection (A/B measurements).
bool gi_bf16_enabled() {
  static int v = -1;
  if (v < 0) { const char* e = getenv("MGRIT_GRU_GI_BF16"); v = (e && e[0] == '0') ? 0 : 1; }
  return v == 1;
}

struct FwdWs {
  float* U[kMaxLevels]; float* G[kMaxLevels]; double* res_acc; UmmaFwdWs um; Tf32Ws tf;
  __nv_bfloat16* chain_ub; unsigned* chain_bar; uint4* chain_xw; size_t chain_xw_bytes;   // scratch of the persistent serial-chain kernel
  unsigned chain_steps;                           // steps of its chains so far (the words are cleared once per call)
  __nv_bfloat16* Ub[kMaxLevels];                  // bf16 copies of the level states (tensor-core A operands)
  int* sweep_ctr; size_t sweep_ctr_n, sweep_ctr_used;   // progress counters of the multi-step relaxation launches (zeroed per call)
};
struct AdjWs {
  float* U[kMaxLevels]; float* G[kMaxLevels];
  float *a[kMaxLevels], *cr[kMaxLevels], *cz[kMaxLevels], *cn[kMaxLevels], *cnp;   // gate coefficients: fp32 engine
  __nv_bfloat16 *crb[kMaxLevels], *czb[kMaxLevels], *cnb[kMaxLevels], *cnpb;       // ... tensor-core engine (bf16)
  float *dA_h, *dA_i, *lam_tmp; double* res_acc; UmmaAdjWs um; Tf32Ws tf;
  float* grad_scratch;      // fp32 engine: partial weight gradients
  __nv_bfloat16* chain_dAb; unsigned* chain_bar; uint4* chain_xw; size_t chain_xw_bytes; unsigned chain_steps;
  float* chain_dA32;        // fp32 chain: [2][B][3H] operand exchange
};

void plan_fwd(const mgrit_gru_cfg* c, const Hier& hr, Ws& w, FwdWs* o) {
  size_t BH = (size_t)c->B * c->H;
  for (int l = 0; l < hr.L; ++l) {
    o->U[l] = w.take<float>((size_t)(hr.N[l] + 1) * BH);
    o->G[l] = l == 0 ? nullptr : w.take<float>((size_t)(hr.N[l] + 1) * BH);
  }
  o->res_acc = w.take<double>((size_t)(c->iters > 0 ? c->iters : 1));
  o->chain_ub = nullptr; o->chain_bar = nullptr; o->chain_xw = nullptr; o->chain_xw_bytes = 0; o->chain_steps = 0;
  o->sweep_ctr = nullptr; o->sweep_ctr_n = o->sweep_ctr_used = 0;
  for (int l = 0; l < kMaxLevels; ++l) o->Ub[l] = nullptr;
  if (c->operands == MGRIT_OPERANDS_BF16) {
    umma_plan_fwd(c, hr.N, hr.L, w.base, &w.off, &o->um);
    for (int l = 0; l < hr.L; ++l) o->Ub[l] = w.take<__nv_bfloat16>((size_t)(hr.N[l] + 1) * BH);
    o->chain_ub = w.take<__nv_bfloat16>(2 * BH);
    o->chain_bar = w.take<unsigned>(((size_t)c->B / 16 + 1) * ((size_t)c->H / 8) + 64);
    o->chain_xw_bytes = serial_xw_bytes(c->B, c->H, 1);
    o->chain_xw = reinterpret_cast<uint4*>(w.take<char>(o->chain_xw_bytes));
    o->sweep_ctr_n = 1 << 16;
    o->sweep_ctr = w.take<int>(o->sweep_ctr_n);
  } else {
    o->chain_bar = w.take<unsigned>((size_t)c->B / 16 + 64);
  }
  if (is_tf32(c)) tf32_plan_fwd(c, hr.N, hr.L, w.base, &w.off, &o->tf);
}

void plan_adj(const mgrit_gru_cfg* c, const Hier& hr, Ws& w, AdjWs* o) {
  size_t BH = (size_t)c->B * c->H;
  for (int l = 0; l < hr.L; ++l) {
    o->U[l] = w.take<float>((size_t)(hr.N[l] + 1) * BH);
    o->G[l] = w.take<float>((size_t)(hr.N[l] + 1) * BH);
    o->a[l] = w.take<float>((size_t)hr.N[l] * BH);
    if (c->operands == MGRIT_OPERANDS_BF16) {
      o->cr[l] = o->cz[l] = o->cn[l] = nullptr;
      o->crb[l] = w.take<__nv_bfloat16>((size_t)hr.N[l] * BH);
      o->czb[l] = w.take<__nv_bfloat16>((size_t)hr.N[l] * BH);
      o->cnb[l] = w.take<__nv_bfloat16>((size_t)hr.N[l] * BH);
    } else {
      o->crb[l] = o->czb[l] = o->cnb[l] = nullptr;
      o->cr[l] = w.take<float>((size_t)hr.N[l] * BH);
      o->cz[l] = w.take<float>((size_t)hr.N[l] * BH);
      o->cn[l] = w.take<float>((size_t)hr.N[l] * BH);
    }
  }
  if (c->operands == MGRIT_OPERANDS_BF16) { o->cnp = nullptr; o->cnpb = w.take<__nv_bfloat16>((size_t)hr.N[0] * BH); }
  else { o->cnpb = nullptr; o->cnp = w.take<float>((size_t)hr.N[0] * BH); }
  o->res_acc = w.take<double>((size_t)(c->iters > 0 ? c->iters : 1));
  o->chain_steps = 0;
  if (c->operands == MGRIT_OPERANDS_BF16) {
    o->dA_h = o->dA_i = o->lam_tmp = o->grad_scratch = nullptr;
    umma_plan_adj(c, hr.N, hr.L, w.base, &w.off, &o->um);
    o->chain_dA32 = nullptr;
    o->chain_dAb = w.take<__nv_bfloat16>(6 * BH);
    o->chain_bar = w.take<unsigned>(((size_t)c->B / 16 + 1) * ((size_t)c->H / 8) + 64);
    o->chain_xw_bytes = serial_xw_bytes(c->B, c->H, 3);
    o->chain_xw = reinterpret_cast<uint4*>(w.take<char>(o->chain_xw_bytes));
  } else {
    o->chain_dAb = nullptr; o->chain_xw = nullptr; o->chain_xw_bytes = 0;
    o->chain_bar = w.take<unsigned>((size_t)c->B / 16 + 64);
    o->chain_dA32 = w.take<float>(6 * BH);
    o->dA_h = o->dA_i = o->lam_tmp = o->grad_scratch = nullptr;
    if (is_tf32(c)) {
      o->dA_h = w.take<float>((size_t)c->T * BH * 3);
      o->dA_i = w.take<float>((size_t)c->T * BH * 3);
      o->lam_tmp = w.take<float>((size_t)c->T * BH);     // lambda in forward order when the caller wants no dh
    } else {
      o->grad_scratch = w.take<float>(simt_gradients_scratch(c->T * c->B, 3 * c->H, c->H, c->I));
    }
  }
  if (is_tf32(c)) tf32_plan_adj(c, hr.N, hr.L, w.base, &w.off, &o->tf);
}

// One launch of "advance nk*B rows by one step of level l".
struct StepDesc {
  int l, nk;
  int in_slot, in_stride;                 // source slots in U[l]
  float* out; int out_slot, out_stride;   // destination array (slot-major [.,B,H]) and slots
  const float* gadd; int gadd_slot, gadd_stride;
  int tgt_slot, tgt_stride;               // level-l point the step arrives at (selects input / coefficients)
  int mode;
};

// The multigrid cycle (Algorithm "MGProp" with the recursive coarse solve of the remark
// "Beyond Two-Level"), FAS form: level l solves u_j = step_l(u_{j-1}) + g_j.
struct Cycle {
  const mgrit_gru_cfg* c; Hier hr; cudaStream_t s;
  float** U; float** G; double* res_acc; int cycle_idx = 0;
  __nv_bfloat16** Ub = nullptr;   // optional bf16 copies of U (kept in step with every writer)
  size_t BH;
  int rc = MGRIT_OK;              // first failure of a launch (a step that cannot be prepared or launched)
  virtual int launch_step(const StepDesc& d) = 0;
  void step(const StepDesc& d) {
    if (rc != MGRIT_OK) return;   // after a failure nothing more is enqueued: outputs are undefined
    rc = launch_step(d);
  }
  // all N_l dependent steps of level l in one persistent launch; false = not available here
  virtual bool chain(int l) { (void)l; return false; }
  // A relaxation sweep of level l in one launch: kinds[i] = s in 1..cf-1: F-step to slot s of every interval;
  // cf: C-step; cf + 1: the step that evaluates v at the C-points into G[l+1].  false = not available here.
  // kz: the first intervals that take part (one more after every C-step while `homog`).
  virtual bool launch_sweep(int l, const int* kinds, int n, int kz) { (void)l; (void)kinds; (void)n; (void)kz; return false; }
  // F (CF)^relax (the opening F optional), optionally followed by the evaluation of v at the C-points
  bool relax_sweep(int l, bool first_f, int relax, bool with_v, int kz = INT_MAX) {
    if (rc != MGRIT_OK) return true;
    int kinds[64], n = 0;
    const int cf = c->cf;
    if ((cf - 1) * (relax + 1) + relax + 1 > 64) return false;
    if (first_f) for (int sI = 1; sI < cf; ++sI) kinds[n++] = sI;
    for (int r = 0; r < relax; ++r) { kinds[n++] = cf; for (int sI = 1; sI < cf; ++sI) kinds[n++] = sI; }
    if (with_v) kinds[n++] = cf + 1;
    if (n < 2) return false;
    return launch_sweep(l, kinds, n, kz);
  }
  virtual ~Cycle() {}

  // A recurrence without source terms that starts from a zero guess (the adjoint of a loss on the last state alone) is zero
  // behind its first points until the first coarse solve has spread the start: on the way down of the first cycle only the
  // intervals that can be non-zero are stepped (`homog`; zero_levels() clears what is then never written).  A level whose
  // unknowns and right-hand sides vanish behind point P has P / cf + 1 such intervals, one more after every C-relaxation.
  bool homog = false;
  void zero_levels(Setup* q) {
    for (int l = 1; l < hr.L; ++l) {
      if (l + 1 < hr.L) q->zero(U[l] + BH, sizeof(float) * (size_t)hr.N[l] * BH);
      q->zero(G[l] + BH, sizeof(float) * (size_t)hr.N[l] * BH);
    }
  }
  // F-relaxation: from every C-point (of the first kz intervals) the cf - 1 F-points of its interval, one dependent step per
  // launch over all intervals; a ragged level has one more, shorter interval of N % cf F-points behind its last C-point.
  void frelax(int l, int kz = INT_MAX) {
    int cf = c->cf, nki = hr.N[l] / cf, tail = hr.N[l] % cf;
    for (int sI = 1; sI < cf; ++sI) {
      const int nk = nki + (sI <= tail ? 1 : 0);
      step(StepDesc{l, nk < kz ? nk : kz, sI - 1, cf, U[l], sI, cf, G[l], sI, cf, sI, cf, 0});
    }
  }
  void crelax(int l, int kz = INT_MAX) {
    int cf = c->cf, nki = hr.N[l] / cf;
    step(StepDesc{l, nki < kz ? nki : kz, cf - 1, cf, U[l], cf, cf, G[l], cf, cf, cf, cf, 0});
  }
  // One cycle from level l down.  skip_first_f: the state of level l was F-relaxed last and no C-point has changed
  // since, so the opening F-relaxation would reproduce it bit for bit.  record: store the level-0 residual norm.
  // live: the last point with a non-zero unknown or right-hand side while `homog`.
  void cycle(int l, bool skip_first_f, bool record, int live = 0) {
    int cf = c->cf, N = hr.N[l];
    if (l == hr.L - 1) {  // coarsest level: serial propagation
      homog = false;
      if (chain(l)) return;
      for (int j = 1; j <= N; ++j) step(StepDesc{l, 1, j - 1, 1, U[l], j, 1, G[l], j, 1, j, 1, 0});
      return;
    }
    int relax = l == 0 ? c->relax_fine : c->relax_coarse;       // n: F (CF)^n
    int nc = hr.N[l + 1], kz = homog ? live / cf + 1 : INT_MAX;
    if (relax_sweep(l, !skip_first_f, relax, true, kz)) {
      if (homog) kz += relax;
    } else {
      if (!skip_first_f) frelax(l, kz);
      for (int n = 0; n < relax; ++n) { crelax(l, kz); if (homog) ++kz; frelax(l, kz); }
      // v_k = step_l(u_{cf k - 1}) + g_{cf k}  ->  G[l+1][k]
      step(StepDesc{l, nc < kz ? nc : kz, cf - 1, cf, G[l + 1], 1, 1, G[l], cf, cf, cf, cf, 0});
    }
    const int np = nc < kz ? nc : kz;
    // r_k = u_{cf k} - v_k ; U'_k = u_{cf k}
    stream_restrict_residual(U[l], cf, G[l + 1], U[l + 1], Ub ? Ub[l + 1] : nullptr, np, (i64)BH,
                             (l == 0 && record) ? res_acc + cycle_idx : nullptr, s);
    // G_k = v_k - step_{l+1}(U'_{k-1})
    step(StepDesc{l + 1, np, 0, 1, G[l + 1], 1, 1, nullptr, 0, 0, 1, 1, 1});
    cycle(l + 1, false, false, np);
    stream_correct(U[l], Ub ? Ub[l] : nullptr, cf, U[l + 1], nc, (i64)BH, s);
    if (!relax_sweep(l, true, 0, false)) frelax(l);
    // F-cycle: one more V-cycle from this level down on the corrected state (on the last two levels: a second
    // V-cycle).  Its opening F-relaxation would repeat the one just done.
    if ((c->flags & MGRIT_FLAG_F_CYCLE) && fcycle_leg) {
      const bool saved = fcycle_leg;
      fcycle_leg = false;
      cycle(l, true, false);
      fcycle_leg = saved;
    }
  }
  bool fcycle_leg = true;     // false while a trailing V-cycle of an F-cycle runs (it does not spawn further ones)
  int solve(Setup* q) {      // q: what the caller has collected
    if (hr.L == 1) { homog = false; if (!q->run()) return MGRIT_CUDA_ERROR; cycle(0, false, false); return rc; }
    if (c->iters <= 0) homog = false;
    if (homog) zero_levels(q);
    q->zero(res_acc, sizeof(double) * (size_t)(c->iters > 0 ? c->iters : 1));
    if (!q->run()) return MGRIT_CUDA_ERROR;
    for (cycle_idx = 0; cycle_idx < c->iters && rc == MGRIT_OK; ++cycle_idx) {
      // the previous cycle ended with an F-relaxation of level 0: the caller may ask not to repeat it
      const bool dup = cycle_idx > 0 && (c->flags & MGRIT_FLAG_SKIP_DUPLICATE_FRELAX);
      cycle(0, dup, true);
    }
    return rc;
  }
};

struct FwdCycle : Cycle {
  const gru_params* p; const float* gi; UmmaFwdWs* um; FwdWs* fw;
  const __nv_bfloat16* gib = nullptr;   // bf16 copy of gi: what every kernel of the solve reads when the state copies exist
  bool gi_f32 = true;                   // false: the fp32 projection was not written (MGRIT_FLAG_GI_F32_UNUSED); gib is set
  // stacked layers: the input of a layer above the first is the layer below's newest result, so its projection is kept per
  // level, one row block per point (arrays by level); null: the fine-grid projection, strided
  float* const* gi_lv = nullptr;
  i64 gi_stride(int l) const { return gi_lv ? 1 : hr.stride_t[l]; }
  const float* gi_of(int l) const { return gi_lv ? gi_lv[l] : gi; }

  bool chain(int l) override {
    if (c->operands != MGRIT_OPERANDS_BF16) {     // fp32 and tf32 modes: the chain in FFMA arithmetic
      if (!fw->chain_bar) return false;
      Serial32FwdArgs a;
      a.B = c->B; a.H = c->H; a.nsteps = hr.N[l]; a.u = U[l];
      const i64 st = gi_stride(l); const float* gi = gi_of(l);
      a.gi = gi + (st - 1) * (i64)BH * 3; a.gi_step = st * (i64)BH * 3;
      a.g = G[l]; a.W = p->W_hh; a.b_hh = p->b_hh; a.gamma = hr.gamma[l]; a.cell = c->cell;
      a.bar = fw->chain_bar + 32;       // (the words in front are the persistent solve's)
      return serial32_fwd_solve(a, s);
    }
    if (!fw->chain_ub) return false;
    SerialFwdArgs a{};
    a.B = c->B; a.H = c->H; a.nsteps = hr.N[l];
    a.u = U[l]; a.ub = fw->chain_ub;
    const i64 st = gi_stride(l); const float* gi = gi_of(l);
    a.gi = gi + (st - 1) * (i64)BH * 3; a.gi_step = st * (i64)BH * 3;
    // (the plain serial sweep has no other level to stay consistent with: it uses the fp32 projection as it is)
    a.gi_as_bf16 = (gib && hr.L > 1) ? 1 : 0;
    if (!gi_f32) { a.gi_b = gib + (st - 1) * (i64)BH * 3; a.gi = nullptr; }
    a.g = G[l]; a.W = um->W_hh; a.b_hh = p->b_hh; a.gamma = hr.gamma[l]; a.cell = c->cell; a.bar = fw->chain_bar;
    a.xw = fw->chain_xw; a.xw_bytes = fw->chain_xw_bytes; a.step0 = fw->chain_steps; fw->chain_steps += hr.N[l];
    return serial_fwd_solve(a, s) || chain_by_sweeps(l);
  }
  // The dependent steps of a level whose rows and weights do not fit the chain kernel (many batch rows at a large width): sweeps
  // over ONE interval of N_l points, up to kMaxFwdSweepSteps steps per launch (100 rows at H = 1024: 34 -> 13 us a step).
  bool chain_by_sweeps(int l) {
    const int N = hr.N[l], kMax = kMaxFwdSweepSteps;
    if (!Ub || c->B > 128 || N < 2 || !fw->sweep_ctr || fw->sweep_ctr_used + N > fw->sweep_ctr_n) return false;
    const i64 st = gi_stride(l); const float* gi = gi_of(l);
    for (int j0 = 1; j0 <= N && rc == MGRIT_OK; j0 += kMax) {
      FwdSweepArgs a{};
      a.B = c->B; a.H = c->H; a.nk = 1; a.cf = N; a.n = N - j0 + 1 < kMax ? N - j0 + 1 : kMax;
      a.U = U[l]; a.Ub = Ub[l];
      a.gi = gi + (st - 1) * (i64)BH * 3; a.gi_ss = st * (i64)BH * 3; a.gi_ks = st * N * (i64)BH * 3;
      a.gi_b = gib ? gib + (st - 1) * (i64)BH * 3 : nullptr;
      a.g = G[l] ? G[l] + BH : nullptr;
      a.b_hh = p->b_hh; a.gamma = hr.gamma[l]; a.cell = c->cell; a.ctr = fw->sweep_ctr + fw->sweep_ctr_used;
      for (int i = 0; i < a.n; ++i) {
        FwdSweepStep& q = a.st[i];
        const int j = j0 + i;
        q.in_s = q.tgt_s = j - 1; q.nk = 1; q.dep = 1;
        q.out = U[l] + (size_t)j * BH; q.out_ks = (i64)N * BH; q.out_b = Ub[l] + (size_t)j * BH;
      }
      const int r = umma_fwd_sweep(a, um, s);
      if (r == MGRIT_UNSUPPORTED && j0 == 1) return false;
      fw->sweep_ctr_used += a.n;
      if (r != MGRIT_OK) rc = r;
    }
    return true;
  }
  bool launch_sweep(int l, const int* kinds, int n, int) override {      // (a forward solve has source terms: every interval takes part)
    const int cf = c->cf;
    const int tail = hr.N[l] % cf;      // F-points behind the last C-point (ragged levels): a shorter last interval
    if (c->operands != MGRIT_OPERANDS_BF16 || !Ub || c->B > 128 || hr.N[l] < cf || n > kMaxFwdSweepSteps) return false;
    FwdSweepArgs a{};
    a.B = c->B; a.H = c->H; a.nk = hr.N[l] / cf; a.cf = cf; a.n = n;
    const int kt = 128 / c->B;
    const size_t need = (size_t)n * ((a.nk + (tail > 0 ? 1 : 0) + kt - 1) / kt);
    if (!fw->sweep_ctr || fw->sweep_ctr_used + need > fw->sweep_ctr_n) return false;
    a.U = U[l]; a.Ub = Ub[l];
    const i64 st = gi_stride(l); const float* gi = gi_of(l);
    a.gi = gi + (st - 1) * (i64)BH * 3; a.gi_ss = st * (i64)BH * 3; a.gi_ks = st * cf * (i64)BH * 3;
    a.gi_b = gib ? gib + (st - 1) * (i64)BH * 3 : nullptr;
    a.g = G[l] ? G[l] + BH : nullptr;
    a.b_hh = p->b_hh; a.gamma = hr.gamma[l]; a.cell = c->cell;
    a.ctr = fw->sweep_ctr + fw->sweep_ctr_used;
    for (int i = 0; i < n; ++i) {
      FwdSweepStep& q = a.st[i];
      const int kd = kinds[i], prev = i ? kinds[i - 1] : 0;
      q.nk = a.nk + (kd < cf && kd <= tail ? 1 : 0);
      if (kd < cf) {             // F-step to slot kd
        q.in_s = kd - 1; q.tgt_s = kd - 1;
        q.out = U[l] + (size_t)kd * BH; q.out_ks = (i64)cf * BH; q.out_b = Ub[l] + (size_t)kd * BH;
        q.dep = prev == cf ? 2 : 1;
      } else if (kd == cf) {     // C-step: slot cf of interval k = slot 0 of interval k + 1
        q.in_s = cf - 1; q.tgt_s = cf - 1;
        q.out = U[l] + (size_t)cf * BH; q.out_ks = (i64)cf * BH; q.out_b = Ub[l] + (size_t)cf * BH;
        q.dep = 3;
      } else {                   // v at the C-points, into the coarse level's G
        q.in_s = cf - 1; q.tgt_s = cf - 1;
        q.out = G[l + 1] + BH; q.out_ks = (i64)BH; q.out_b = nullptr;
        q.dep = 1;
      }
    }
    const int r = umma_fwd_sweep(a, um, s);
    if (r == MGRIT_UNSUPPORTED) return false;
    fw->sweep_ctr_used += need;
    if (r != MGRIT_OK) rc = r;
    return true;
  }
  int launch_step(const StepDesc& d) override {
    FwdStepArgs a{};
    a.M = d.nk * c->B; a.B = c->B; a.H = c->H;
    a.hin = U[d.l] + (size_t)d.in_slot * BH; a.hin_ks = (i64)d.in_stride * BH;
    a.hout = d.out + (size_t)d.out_slot * BH; a.hout_ks = (i64)d.out_stride * BH;
    a.hin_b = Ub ? Ub[d.l] + (size_t)d.in_slot * BH : nullptr;
    a.hout_b = (Ub && d.out == U[d.l]) ? Ub[d.l] + (size_t)d.out_slot * BH : nullptr;
    const i64 st = gi_stride(d.l); const float* gi = gi_of(d.l);
    a.gi = gi + ((i64)st * d.tgt_slot - 1) * (i64)BH * 3; a.gi_ks = st * d.tgt_stride * (i64)BH * 3;
    a.gi_b = gib ? gib + ((i64)st * d.tgt_slot - 1) * (i64)BH * 3 : nullptr;
    a.gadd = d.gadd ? d.gadd + (size_t)d.gadd_slot * BH : nullptr; a.gadd_ks = (i64)d.gadd_stride * BH;
    a.W_hh = p->W_hh; a.b_hh = p->b_hh; a.gamma = hr.gamma[d.l]; a.cell = c->cell; a.mode = d.mode;
    if (c->operands == MGRIT_OPERANDS_BF16) return umma_fwd_step(a, um, s);
    if (is_tf32(c)) return tf32_fwd_step(a, &fw->tf, s);
    simt_fwd_step(a, s);
    return MGRIT_OK;
  }
};

struct AdjCycle : Cycle {
  const gru_params* p; AdjWs* w;
  // stacked layers: what the layer above sends to its input joins the incoming sensitivities (rows ladd + k*ladd_ks; the sums
  // go to lsum)
  const float* ladd = nullptr; i64 ladd_ks = 0; float* lsum = nullptr;
  bool chain(int l) override { return chain_on(l, U[l], G[l]); }
  bool chain_on(int l, float* mu, const float* g) {
    if (c->operands != MGRIT_OPERANDS_BF16) {
      if (!w->chain_bar || !w->chain_dA32) return false;
      Serial32AdjArgs a;
      a.B = c->B; a.H = c->H; a.nsteps = hr.N[l]; a.mu = mu; a.dA = w->chain_dA32;
      const i64 row0 = (i64)(hr.N[l] - 1) * BH;    // step s = 1 applies forward step N_l, stored at row N_l - 1
      a.a = w->a[l] + row0; a.cr = w->cr[l] + row0; a.cz = w->cz[l] + row0; a.cn = w->cn[l] + row0;
      a.coef_step = -(i64)BH;
      a.g = g; a.W = p->W_hh; a.bar = w->chain_bar;
      return serial32_adj_solve(a, s);
    }
    if (!w->chain_dAb) return false;
    SerialAdjArgs a{};
    a.B = c->B; a.H = c->H; a.nsteps = hr.N[l];
    a.mu = mu; a.dAb = w->chain_dAb;
    i64 row0 = (i64)(hr.N[l] - 1) * BH;        // step s = 1 applies forward step N_l, stored at row N_l - 1
    a.a = w->a[l] + row0; a.cr = w->crb[l] + row0; a.cz = w->czb[l] + row0; a.cn = w->cnb[l] + row0;
    a.coef_step = -(i64)BH;
    a.g = g; a.WT = w->um.W_hhT; a.bar = w->chain_bar;
    a.xw = w->chain_xw; a.xw_bytes = w->chain_xw_bytes; a.step0 = w->chain_steps; w->chain_steps += hr.N[l];
    return serial_adj_solve(a, s);
  }
  // n dependent steps over the same rows (each starts where its predecessor ended): one launch where that is available.
  // ladds: the rows that join each step's incoming sensitivities (stacked layers), `ladds_ks` apart by k; null: none
  void run_steps(const StepDesc* d, int n, const float* const* ladds = nullptr, i64 ladds_ks = 0) {
    for (int i0 = 0; i0 < n && rc == MGRIT_OK; i0 += kMaxAdjSweepSteps) {
      const int m = n - i0 < kMaxAdjSweepSteps ? n - i0 : kMaxAdjSweepSteps;
      int r = MGRIT_UNSUPPORTED;
      if (c->operands == MGRIT_OPERANDS_BF16) {
        const StepDesc& f = d[i0];
        bool sums = true;      // (residuals are single steps)
        AdjSweepArgs a{};
        a.B = c->B; a.H = c->H; a.n = m;
        a.lin = U[f.l] + (size_t)f.in_slot * BH; a.lin_ks = (i64)f.in_stride * BH;
        a.a = w->a[f.l]; a.cr = w->crb[f.l]; a.cz = w->czb[f.l]; a.cn = w->cnb[f.l]; a.coef_ks = -(i64)f.tgt_stride * BH;
        for (int i = 0; i < m; ++i) {
          const StepDesc& e = d[i0 + i];
          AdjSweepStep& q = a.st[i];
          q.out = e.out + (size_t)e.out_slot * BH; q.out_ks = (i64)e.out_stride * BH;
          q.g = e.gadd ? e.gadd + (size_t)e.gadd_slot * BH : nullptr; q.g_ks = (i64)e.gadd_stride * BH;
          q.coff = (i64)(hr.N[e.l] - e.tgt_slot) * BH;      // (as in launch_step)
          q.ladd = ladds ? ladds[i0 + i] : nullptr; q.ladd_ks = ladds_ks;
          q.nk = e.nk;
          sums = sums && e.mode == 0;
        }
        if (sums) r = umma_adj_sweep(a, &w->um, s);
      }
      if (r == MGRIT_UNSUPPORTED) {
        for (int i = i0; i < i0 + m; ++i) {
          if (ladds) { ladd = ladds[i]; ladd_ks = ladds_ks; }
          step(d[i]);
        }
        if (ladds) ladd = nullptr;
      } else {
        rc = r;
      }
    }
  }
  bool launch_sweep(int l, const int* kinds, int n, int kz) override {
    const int cf = c->cf, nki = hr.N[l] / cf, tail = hr.N[l] % cf;
    if (c->operands != MGRIT_OPERANDS_BF16) return false;
    StepDesc d[64];      // (relax_sweep() lists at most 64 steps)
    int m = 0;
    for (int i = 0; i < n; ++i) {
      const int kd = kinds[i], nk = nki + (kd < cf && kd <= tail ? 1 : 0), live = nk < kz ? nk : kz;
      if (kd < cf) d[m++] = StepDesc{l, live, kd - 1, cf, U[l], kd, cf, G[l], kd, cf, kd, cf, 0};
      else if (kd == cf) d[m++] = StepDesc{l, live, cf - 1, cf, U[l], cf, cf, G[l], cf, cf, cf, cf, 0};
      else d[m++] = StepDesc{l, live, cf - 1, cf, G[l + 1], 1, 1, G[l], cf, cf, cf, cf, 0};
      if (kd == cf || i + 1 == n) {      // (the steps behind a C-step start from what it left in the neighbouring interval)
        run_steps(d, m);
        m = 0;
        if (homog) ++kz;
      }
    }
    return true;
  }
  int launch_step(const StepDesc& d) override {
    AdjStepArgs a{};
    a.M = d.nk * c->B; a.B = c->B; a.H = c->H;
    a.lin = U[d.l] + (size_t)d.in_slot * BH; a.lin_ks = (i64)d.in_stride * BH;
    a.ladd = ladd; a.ladd_ks = ladd_ks; a.lsum = lsum;
    a.lout = d.out + (size_t)d.out_slot * BH; a.lout_ks = (i64)d.out_stride * BH;
    a.gadd = d.gadd ? d.gadd + (size_t)d.gadd_slot * BH : nullptr; a.gadd_ks = (i64)d.gadd_stride * BH;
    // the step arriving at reversed point s applies forward step j = N_l - s + 1, stored at row N_l - s
    i64 row0 = (i64)(hr.N[d.l] - d.tgt_slot) * BH;
    a.a = w->a[d.l] + row0;
    if (c->operands == MGRIT_OPERANDS_BF16) {
      a.cr = a.cz = a.cn = nullptr;
      a.crb = w->crb[d.l] + row0; a.czb = w->czb[d.l] + row0; a.cnb = w->cnb[d.l] + row0;
    } else {
      a.crb = a.czb = a.cnb = nullptr;
      a.cr = w->cr[d.l] + row0; a.cz = w->cz[d.l] + row0; a.cn = w->cn[d.l] + row0;
    }
    a.coef_ks = -(i64)d.tgt_stride * BH;
    a.W_hh = p->W_hh; a.mode = d.mode;
    if (c->operands == MGRIT_OPERANDS_BF16) return umma_adj_step(a, &w->um, s);
    if (is_tf32(c)) return tf32_adj_step(a, &w->tf, s);
    if (ladd) {
      stream_sum_rows(lsum, a.lin, a.lin_ks, ladd, ladd_ks, d.nk, (i64)BH, s);
      a.lin = lsum; a.lin_ks = (i64)BH;
    }
    simt_adj_step(a, s);
    return MGRIT_OK;
  }
};

// fp32 forward steps that depend on one another: the chain kernel (W_hh spread over up to 148 CTAs, 16 rows each) or a phase of the
// persistent solve (a cluster per rows, weights in registers; above H = 256 a third of them in shared memory)?  us a step, chain /
// persistent: 16 rows, H = 160 2.97 / 2.82, 192 3.14 / 3.17 (one row 2.90 / 3.13), 224 3.28 / 2.73, 256 3.56 / 3.00, 288 3.59 / 4.03,
// 320 3.88 / 4.17, 352 3.94 / 4.70; where eight units a CTA do not fit one wave the chain loses (64 rows, H = 320 5.23 / 4.24)
// until the rows take the persistent clusters of eight a second wave (128 rows, H = 224 4.43 / 4.80, 288 5.12 / 6.96).  Inside a
// solve the chain is two more launches, 25 us.  Two levels, T = 2048, cf = 2, one row, a forward solve of two cycles: H = 192 6.49 ->
// 5.91 ms, 304 (no multiple of 32: no chain) 8.66, 320 7.0, 352 9.72 -> 7.23.  (Adjoint phases win everywhere: H = 288, 16 rows
// 5.17 / 3.94.)
bool chain32_wins(const mgrit_gru_cfg* c, int nsteps, bool alone) {
  const int units = serial32_fwd_units(c->B, c->H);
  int gain_ns = 0;
  if (units == 8) gain_ns = c->H > 256 ? 800 : c->H == 192 ? 150 : 0;
  else if (units > 0 && c->H > 192 && c->B > 120) gain_ns = 400;
  return gain_ns > 0 && (alone || (i64)nsteps * gain_ns >= 25000);
}

// The whole solve of an fp32-state GRU recurrence as phases of the persistent kernels in f32_solve.cu.  The same cycle as
// Cycle::cycle, phase by phase; what differs is where C-points travel: a C-relaxation of level l leaves its results in the
// coarse array U[l+1] (which the restriction would fill with them anyway) and the next one back in U[l], so that no row of
// a phase overwrites what another row of the same phase still reads; the correction is the start of the closing F-relaxation.
struct F32Cycle {
  const mgrit_gru_cfg* c; const Hier* hr; bool adjoint; cudaStream_t s;
  float** U; float** G; double* res_acc; F32Args a;
  bool ok = true, fcycle_leg = true, started = false;      // started: a launch of this solve went out
  bool homog = false;      // as Cycle::homog
  int cycle_idx = 0;
  i64 bh() const { return (i64)c->B * c->H; }
  unsigned* bars = nullptr; int bars_left = 0;      // cleared barrier counters, one per launch
  Cycle* by_steps = nullptr;                        // forward: its chain serves the coarsest level where that is faster
  void flush() {
    if (a.nph > 0 && ok) {
      unsigned* const own = a.bar;
      a.progress = own + 16;            // (behind the counters of the launches)
      if (bars_left > 0) { a.bar = bars++; --bars_left; }
      else ok = cudaMemsetAsync(own, 0, sizeof(unsigned), s) == cudaSuccess;
      ok = ok && f32_solve(adjoint, a, s);
      started = started || ok;
      a.bar = own;
    }
    a.nph = 0;
  }
  void add(const F32Phase& p) {
    if (a.nph == kF32MaxPhases) flush();
    a.ph[a.nph++] = p;
  }
  // rows start at slot s0 of their interval of level l; their first step arrives at slot s0 + 1
  F32Phase phase(int l, const float* src, i64 src_ks, int s0) {
    const i64 BH = bh(), st = hr->stride_t[l], ks = (i64)c->cf * BH;
    F32Phase p;
    memset(&p, 0, sizeof(p));
    p.level = l; p.gamma = hr->gamma[l];
    p.src = src; p.src_ks = src_ks;
    p.out = U[l] + (s0 + 1) * BH; p.out_ks = ks; p.out_ss = BH;
    p.g = G[l] ? G[l] + (s0 + 1) * BH : nullptr; p.g_ks = ks; p.g_ss = BH;
    if (adjoint) { p.op = ((i64)hr->N[l] - (s0 + 1)) * BH; p.op_ss = -BH; p.op_ks = -ks; }
    else { p.op = (st * (s0 + 1) - 1) * BH * 3; p.op_ss = st * BH * 3; p.op_ks = st * ks * 3; }
    return p;
  }
  void cycle(int l, bool skip_first_f, bool record, int live = 0) {
    const i64 BH = bh();
    const int cf = c->cf, N = hr->N[l];
    if (l == hr->L - 1) {
      homog = false;
      if (by_steps && chain32_wins(c, N, l == 0)) {
        flush();
        if (ok && by_steps->chain(l)) { started = true; return; }
      }
      F32Phase p = phase(l, U[l], 0, 0);
      p.nk = p.nfull = 1; p.n = N;
      add(p);
      return;
    }
    const int nc = hr->N[l + 1], tail = N % cf, relax = l == 0 ? c->relax_fine : c->relax_coarse;
    int kz = homog ? live / cf + 1 : INT_MAX;
    float* cp = U[l]; i64 cp_ks = (i64)cf * BH;          // where slot 0 of the intervals is: here or in the coarse array
    for (int r = 0; r <= relax; ++r) {
      const bool skip = r == 0 && skip_first_f;          // the F-points are there already: only the closing step
      const int s0 = skip ? cf - 1 : 0;
      F32Phase p = skip ? phase(l, U[l] + (cf - 1) * BH, (i64)cf * BH, s0) : phase(l, cp, cp_ks, 0);
      p.n = skip ? 0 : cf - 1; p.nfull = nc; p.ntail = skip ? 0 : tail; p.nk = nc + (p.ntail > 0 ? 1 : 0);
      if (p.nk > kz) p.nk = kz;
      if (r < relax) {
        p.last_kind = kLastStore;
        float* dst = cp == U[l] ? U[l + 1] + BH : U[l] + (i64)cf * BH;
        const i64 dst_ks = cp == U[l] ? BH : (i64)cf * BH;
        p.last = dst; p.last_ks = dst_ks;
        add(p);
        cp = dst - dst_ks; cp_ks = dst_ks;
        if (homog) ++kz;
      } else {
        p.last_kind = kLastCoarse;
        p.last = G[l + 1] + BH; p.last_ks = BH;
        p.src2 = cp; p.src2_ks = cp_ks;
        p.uc = cp + cp_ks; p.uc_ks = cp_ks;
        p.ucd = cp == U[l + 1] ? nullptr : U[l + 1] + BH; p.ucd_ks = BH;
        p.gamma2 = hr->gamma[l + 1];
        const i64 st2 = hr->stride_t[l + 1];
        if (adjoint) { p.op2 = ((i64)nc - 1) * BH; p.op2_ks = -BH; }
        else { p.op2 = (st2 - 1) * BH * 3; p.op2_ks = st2 * BH * 3; }
        p.acc = l == 0 && record ? res_acc + cycle_idx : nullptr;
        add(p);
      }
    }
    cycle(l + 1, false, false, nc < kz ? nc : kz);
    F32Phase p = phase(l, U[l + 1], BH, 0);
    p.copy = U[l]; p.copy_ks = (i64)cf * BH;
    p.nk = nc + 1; p.nfull = nc; p.n = cf - 1; p.ntail = tail;
    add(p);
    if ((c->flags & MGRIT_FLAG_F_CYCLE) && fcycle_leg) {
      fcycle_leg = false;
      cycle(l, true, false);
      fcycle_leg = true;
    }
  }
  // MGRIT_UNSUPPORTED: the first launch was refused and the arrays are as the set-up left them; the caller advances step by step
  int solve(Setup* q) {      // q: what the caller has collected
    a.nph = 0;
    bars = a.bar + 1; bars_left = 15;
    q->zero(bars - 1, 16 * sizeof(unsigned));
    if (hr->L == 1) {
      if (!q->run()) return MGRIT_CUDA_ERROR;
      cycle(0, false, false);
    } else {
      q->zero(res_acc, sizeof(double) * (size_t)(c->iters > 0 ? c->iters : 1));
      if (c->iters <= 0) homog = false;
      for (int l = 1; homog && l < hr->L; ++l) {      // what the first way down then never writes
        q->zero(U[l] + bh(), sizeof(float) * (size_t)hr->N[l] * bh());
        q->zero(G[l] + bh(), sizeof(float) * (size_t)hr->N[l] * bh());
      }
      if (!q->run()) return MGRIT_CUDA_ERROR;
      for (cycle_idx = 0; cycle_idx < c->iters; ++cycle_idx)
        cycle(0, cycle_idx > 0 && (c->flags & MGRIT_FLAG_SKIP_DUPLICATE_FRELAX), true);
    }
    flush();
    return ok ? MGRIT_OK : started ? MGRIT_CUDA_ERROR : MGRIT_UNSUPPORTED;
  }
};

// Which fp32-state solves run there: every one of the fp32 mode whose weights fit, and those of the tf32 split whose steps are
// too small for the tensor cores (rows of the largest step x H^2).  Forward and adjoint us a step there: H = 256 500 rows 11.1 and
// 8.4, 1200 rows 22 and 18, 1700 rows 32 and 26; H = 320 700 rows 25 and 25, 1100 rows 41 and 39.  The tensor-core step takes
// 27 + 6 and 24 + 4 us (product and operand split, one wave of tiles) at 512 rows and hardly more at 2000.  They meet at
// 800 to 900 (H = 320) and 1700 rows (H = 256); the line is the lower one.  Linearisation at H = 256: 2560 rows 45 against 58 us, 5120 rows 84.
constexpr double kF32TfStep = 9e7, kF32TfLin = 2.2e8;
bool use_f32_solve(const mgrit_gru_cfg* c, const Hier& hr) {
  if (!f32_solve_fits(c->H)) return false;
  if (c->operands == MGRIT_OPERANDS_FP32) return true;
  if (c->operands != MGRIT_OPERANDS_TF32) return false;
  const double rows = hr.L == 1 ? c->B : (double)(c->T / c->cf + 1) * c->B;
  return rows * c->H * c->H <= kF32TfStep;
}
bool use_f32_lin(const mgrit_gru_cfg* c, const Hier& hr) {
  if (!f32_solve_fits(c->H)) return false;
  if (c->operands == MGRIT_OPERANDS_FP32) return true;
  if (c->operands != MGRIT_OPERANDS_TF32) return false;
  double rows = 0;
  for (int l = 0; l < hr.L; ++l) rows += (double)hr.N[l] * c->B;
  return rows * c->H * c->H <= kF32TfLin;
}

// Zero initial guess of a level-0 array [T + 1 slots of `slot` elements] behind its fixed slot 0.  In a multigrid solve
// with at least one cycle only the C-points are read before they are written (the first F-relaxation fills every
// F-point from them), so only those slots are cleared: 1 / cf of the memory traffic.
template <class T>
void zero_guess(T* U0, const mgrit_gru_cfg& c, const Hier& hr, size_t slot, Setup* q) {
  if (hr.L == 1) return;      // the sweep writes every point
  if (c.iters > 0 && c.cf > 1 && c.T / c.cf > 0)
    q->zero(U0 + (size_t)c.cf * slot, slot * sizeof(T), (size_t)(c.T / c.cf), (size_t)c.cf * slot * sizeof(T));
  else
    q->zero(U0 + slot, sizeof(T) * (size_t)c.T * slot);
}

int finish(cudaStream_t s, bool sync) {
  if (sync && cudaStreamSynchronize(s) != cudaSuccess) return MGRIT_CUDA_ERROR;
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) { fprintf(stderr, "mgrit_gru: CUDA error: %s\n", cudaGetErrorString(e)); return MGRIT_CUDA_ERROR; }
  if (sync && (umma_device_status() != 0 || serial_device_status() != 0 || f32_device_status() != 0)) return MGRIT_DEVICE_TIMEOUT;
  return MGRIT_OK;
}

int fetch_resnorm(const double* acc, float* resnorm, int iters, cudaStream_t s) {
  double tmp[64];
  for (int base = 0; base < iters; base += 64) {
    int n = iters - base < 64 ? iters - base : 64;
    if (cudaMemcpyAsync(tmp, acc + base, sizeof(double) * n, cudaMemcpyDeviceToHost, s) != cudaSuccess) return MGRIT_CUDA_ERROR;
    if (cudaStreamSynchronize(s) != cudaSuccess) return MGRIT_CUDA_ERROR;
    for (int i = 0; i < n; ++i) resnorm[base + i] = (float)sqrt(tmp[i]);
  }
  return MGRIT_OK;
}

int forward_impl(const mgrit_gru_cfg* cfg_in, bool serial, const gru_params* p, const float* x, const float* h0, float* gi,
                 float* h, float* resnorm, void* ws, size_t ws_bytes, cudaStream_t s) {
  if (!cfg_in || !p || !x || !h0 || !gi || !h || !ws || !p->W_ih || !p->W_hh || !p->b_ih || !p->b_hh) return MGRIT_INVALID_ARG;
  if (!aligned32(x, h0, gi, h, ws, p->W_ih, p->W_hh, p->b_ih, p->b_hh)) return MGRIT_INVALID_ARG;
  mgrit_gru_cfg c = *cfg_in;
  if (serial) { c.levels = 1; c.iters = 1; c.cf = 2; }
  Hier hr;
  int rc = check_cfg(&c, &hr);
  if (rc) return rc;
  Ws w{(char*)ws, ws_bytes, 0};
  FwdWs fw;
  plan_fwd(&c, hr, w, &fw);
  if (!w.fits()) return MGRIT_WORKSPACE_TOO_SMALL;
  size_t BH = (size_t)c.B * c.H;
  // the caller's array has a leading slot for h_0: the level-0 unknowns live there and nothing is copied at the end
  const bool h_in_place = (c.flags & MGRIT_FLAG_H_LEADS_WITH_H0) != 0;
  if (h_in_place) fw.U[0] = h;
  if (carries_copies(&c, serial)) {      // make the copies where the adjoint call will look for them
    GiTail t = gi_tail(&c, gi);
    fw.um.xb = t.xb;
    fw.Ub[0] = t.hb0;
    fw.um.gib = t.gib;
  }
  // (the projection is staged as bf16 where B divides 128; other batch sizes keep its fp32 values, as they always have)
  if (!gi_bf16_enabled() || 128 % c.B != 0) fw.um.gib = nullptr;
  // the caller does not read the fp32 projection and every kernel of this solve reads its bf16 copy: do not write it
  const bool gi_f32 = !((c.flags & MGRIT_FLAG_GI_F32_UNUSED) && carries_copies(&c, serial) && fw.um.gib);

  if (c.operands == MGRIT_OPERANDS_BF16) {
    rc = umma_prepare_fwd(&c, p, x, gi_f32 ? gi : nullptr, &fw.um, s);
    if (rc) return rc;
  } else if (is_tf32(&c)) {
    rc = tf32_prepare_fwd(&c, p, x, gi, &fw.tf, s);
    if (rc) return rc;
  } else {
    simt_project(x, p->W_ih, p->b_ih, gi, c.T * c.B, c.I, 3 * c.H, s);
  }
  Setup setup(s);
  zero_guess(fw.U[0], c, hr, BH, &setup);
  for (int l = 0; l < hr.L; ++l) setup.copy(fw.U[l], h0, BH);
  if (fw.chain_xw) setup.zero(fw.chain_xw, fw.chain_xw_bytes);
  const bool shadows = c.operands == MGRIT_OPERANDS_BF16 && c.B <= 128;
  if (shadows && fw.sweep_ctr) setup.zero(fw.sweep_ctr, sizeof(int) * fw.sweep_ctr_n);
  if (shadows) {
    zero_guess(fw.Ub[0], c, hr, BH, &setup);
    for (int l = 0; l < hr.L; ++l) setup.to_bf16(fw.Ub[l], h0, BH);
  }

  FwdCycle cy;
  cy.c = &c; cy.hr = hr; cy.s = s; cy.U = fw.U; cy.G = fw.G; cy.res_acc = fw.res_acc; cy.BH = BH;
  cy.p = p; cy.gi = gi; cy.um = &fw.um; cy.fw = &fw;
  cy.Ub = shadows ? fw.Ub : nullptr;
  cy.gib = shadows ? fw.um.gib : nullptr;
  cy.gi_f32 = gi_f32;
  rc = MGRIT_UNSUPPORTED;
  if (use_f32_solve(&c, hr)) {
    F32Cycle fc;
    fc.c = &c; fc.hr = &hr; fc.adjoint = false; fc.s = s; fc.U = fw.U; fc.G = fw.G; fc.res_acc = fw.res_acc;
    fc.a.B = c.B; fc.a.H = c.H; fc.a.cell = c.cell; fc.a.W = p->W_hh; fc.a.gi = gi; fc.a.b_hh = p->b_hh; fc.a.bar = fw.chain_bar;
    fc.by_steps = &cy;
    rc = fc.solve(&setup);
  }
  if (rc == MGRIT_UNSUPPORTED) rc = cy.solve(&setup);
  if (rc) return rc;
  if (!h_in_place) cudaMemcpyAsync(h, fw.U[0] + BH, sizeof(float) * (size_t)c.T * BH, cudaMemcpyDeviceToDevice, s);
  if (resnorm && hr.L > 1 && c.iters > 0) {
    rc = fetch_resnorm(fw.res_acc, resnorm, c.iters, s);
    if (rc) return rc;
    return finish(s, true);
  }
  return finish(s, false);
}

int adjoint_impl(const mgrit_gru_cfg* cfg_in, bool serial, const gru_params* p, const float* x, const float* h0,
                 const float* gi, const float* h, const float* dh_seed, const float* dhT, float* dh, float* dh0, float* dx,
                 const gru_grads* g, float* resnorm, void* ws, size_t ws_bytes, cudaStream_t s) {
  if (!cfg_in || !p || !x || !h0 || !gi || !h || !dh0 || !g || !ws) return MGRIT_INVALID_ARG;
  if (!dh_seed && !dhT) return MGRIT_INVALID_ARG;
  if (!p->W_ih || !p->W_hh || !p->b_ih || !p->b_hh || !g->dW_ih || !g->dW_hh || !g->db_ih || !g->db_hh) return MGRIT_INVALID_ARG;
  if (!aligned32(x, h0, gi, h, dh_seed, dhT, dh, dh0, dx, ws, p->W_ih, p->W_hh, p->b_ih, p->b_hh, g->dW_ih, g->dW_hh, g->db_ih, g->db_hh))
    return MGRIT_INVALID_ARG;
  mgrit_gru_cfg c = *cfg_in;
  if (serial) { c.levels = 1; c.iters = 1; c.cf = 2; }
  Hier hr;
  int rc = check_cfg(&c, &hr);
  if (rc) return rc;
  Ws w{(char*)ws, ws_bytes, 0};
  AdjWs aw;
  plan_adj(&c, hr, w, &aw);
  if (!w.fits()) return MGRIT_WORKSPACE_TOO_SMALL;
  size_t BH = (size_t)c.B * c.H;
  const int T = c.T;
  const bool bf16 = c.operands == MGRIT_OPERANDS_BF16;

  const bool copies = carries_copies(&c, serial);
  if (copies) {                           // bf16 x and [h_0; h] were left behind the projection by the forward call
    GiTail t = gi_tail(&c, const_cast<float*>(gi));
    aw.um.xb = t.xb;
    aw.um.hb0 = t.hb0;
    aw.um.hb = t.hb0 + BH;
    aw.um.gib = gi_bf16_enabled() ? t.gib : nullptr;
  }
  if (bf16) {
    rc = umma_prepare_adj(&c, p, h0, h, &aw.um, copies, s);
    if (rc) return rc;
  }
  const bool tf32 = is_tf32(&c);
  if (tf32) {
    rc = tf32_prepare_adj(&c, p, &aw.tf, s);
    if (rc) return rc;
  }
  // adjoint coefficients of every level's steps at the given states (restricted by injection)
  LinArgs lins[kMaxLevels];
  for (int l = 0; l < hr.L; ++l) {
    LinArgs& a = lins[l];
    a = LinArgs{};
    a.M = hr.N[l] * c.B; a.B = c.B; a.H = c.H; a.h0 = h0; a.h = h; a.stride_t = hr.stride_t[l]; a.gi = gi;
    a.t0 = hr.rem[l];     // the level's reversed grid is anchored at T: its forward steps arrive at t0 + stride * j
    a.W_hh = p->W_hh; a.b_hh = p->b_hh; a.gamma = hr.gamma[l]; a.cell = c.cell;
    a.a = aw.a[l]; a.cr = aw.cr[l]; a.cz = aw.cz[l]; a.cn = aw.cn[l]; a.cnp = l == 0 ? aw.cnp : nullptr;
    a.crb = aw.crb[l]; a.czb = aw.czb[l]; a.cnb = aw.cnb[l]; a.cnpb = l == 0 ? aw.cnpb : nullptr;
    a.gi_b = (bf16 && copies) ? aw.um.gib : nullptr;
  }
  if (!(use_f32_lin(&c, hr) && f32_linearise(lins, hr.L, s))) {
    for (int l = 0; l < hr.L; ++l) {
      rc = MGRIT_OK;
      if (bf16) rc = umma_linearise(lins[l], &aw.um, s);
      else if (tf32) rc = tf32_linearise(lins[l], &aw.tf, s);
      else simt_linearise(lins[l], s);
      if (rc) return rc;
    }
  }
  // mu_0 = lambda_T; zero initial guess elsewhere; fine-level source = reversed dh_seed
  Setup setup(s);
  zero_guess(aw.U[0], c, hr, BH, &setup);        // (slot 0 is set below)
  const float* const last = dh_seed ? dh_seed + (size_t)(T - 1) * BH : dhT;
  for (int l = 0; l < hr.L; ++l) setup.copy(aw.U[l], last, BH, dh_seed ? dhT : nullptr);
  if (aw.chain_xw) setup.zero(aw.chain_xw, aw.chain_xw_bytes);
  if (bf16 && hr.L > 1) setup.zero(aw.um.sweep_ctr, sizeof(int) * aw.um.sweep_ctr_n);
  if (dh_seed) {
    setup.zero(aw.G[0], sizeof(float) * BH);
    setup.zero(aw.G[0] + (size_t)T * BH, sizeof(float) * BH);
    if (T > 1) stream_gather_rows(aw.G[0] + BH, (i64)BH, dh_seed + (size_t)(T - 2) * BH, -(i64)BH, T - 1, (i64)BH, s);
  }

  float* Gl[kMaxLevels];
  for (int l = 0; l < hr.L; ++l) Gl[l] = aw.G[l];
  if (!dh_seed) Gl[0] = nullptr;
  AdjCycle cy;
  cy.c = &c; cy.hr = hr; cy.s = s; cy.U = aw.U; cy.G = Gl; cy.res_acc = aw.res_acc; cy.BH = BH;
  cy.p = p; cy.w = &aw;
  cy.homog = !dh_seed;
  rc = MGRIT_UNSUPPORTED;
  if (use_f32_solve(&c, hr)) {
    F32Cycle fc;
    fc.homog = !dh_seed;
    fc.c = &c; fc.hr = &hr; fc.adjoint = true; fc.s = s; fc.U = aw.U; fc.G = Gl; fc.res_acc = aw.res_acc;
    fc.a.B = c.B; fc.a.H = c.H; fc.a.cell = c.cell; fc.a.W = p->W_hh; fc.a.bar = aw.chain_bar;
    for (int l = 0; l < hr.L; ++l) { fc.a.coef[l][0] = aw.a[l]; fc.a.coef[l][1] = aw.cr[l]; fc.a.coef[l][2] = aw.cz[l]; fc.a.coef[l][3] = aw.cn[l]; }
    rc = fc.solve(&setup);
  }
  if (rc == MGRIT_UNSUPPORTED) rc = cy.solve(&setup);
  if (rc) return rc;

  // dh[k] = lambda_{k+1} = mu_{T-1-k} (optional output);  dh0 = lambda_0 = mu_T
  if (dh) stream_gather_rows(dh, (i64)BH, aw.U[0] + (size_t)(T - 1) * BH, -(i64)BH, T, (i64)BH, s);
  cudaMemcpyAsync(dh0, aw.U[0] + (size_t)T * BH, sizeof(float) * BH, cudaMemcpyDeviceToDevice, s);

  // gradient pass g = w * dh/dTheta over all fine steps at once
  if (bf16) {
    // lambda_{t+1} for t = 0..T-1 is read in place from the reversed unknowns (row stride -B*H)
    rc = umma_gradients(&c, p, x, h0, h, aw.U[0] + (size_t)(T - 1) * BH, -(i64)BH, aw.crb[0], aw.czb[0], aw.cnb[0], aw.cnpb, dx, g,
                        &aw.um, copies, s);
    if (rc) return rc;
  } else {
    i64 M = (i64)T * c.B;
    if (!tf32) {
      simt_gradients((int)M, c.B, c.H, c.I, aw.U[0] + (size_t)(T - 1) * BH, -(i64)BH, aw.cr[0], aw.cz[0], aw.cn[0], aw.cnp, h0, h, x, p->W_ih, dx, g,
                     aw.grad_scratch, s);
    } else {
      const float* lam = dh;
      if (!lam) {   // no dh output requested: gather lambda in forward order into workspace scratch
        lam = aw.lam_tmp;
        stream_gather_rows(aw.lam_tmp, (i64)BH, aw.U[0] + (size_t)(T - 1) * BH, -(i64)BH, T, (i64)BH, s);
      }
      stream_form_dA(lam, aw.cr[0], aw.cz[0], aw.cn[0], aw.cnp, aw.dA_h, aw.dA_i, M, c.H, s);
      rc = tf32_wgrad(aw.dA_h, (int)M, 3 * c.H, h0, c.B, h, c.H, g->dW_hh, &aw.tf, s);
      if (!rc) rc = tf32_wgrad(aw.dA_i, (int)M, 3 * c.H, nullptr, 0, x, c.I, g->dW_ih, &aw.tf, s);
      if (rc) return rc;
      stream_colsum(aw.dA_h, M, 3 * c.H, g->db_hh, s);
      stream_colsum(aw.dA_i, M, 3 * c.H, g->db_ih, s);
      if (dx) { rc = tf32_dgrad(aw.dA_i, (int)M, 3 * c.H, c.I, dx, &aw.tf, s); if (rc) return rc; }
    }
  }
  if (resnorm && hr.L > 1 && c.iters > 0) {
    rc = fetch_resnorm(aw.res_acc, resnorm, c.iters, s);
    if (rc) return rc;
    return finish(s, true);
  }
  return finish(s, false);
}


// ======================================================================================================
// Stacked layers in one state: the state of a time point is the stack of all layers' hidden states, layer k's input
// at a step is layer k-1's NEW state of the same step, and ONE multigrid cycle advances the whole stack.  Level
// arrays are kept per layer ([N_l + 1][B][H] each); StackCycle below runs the same cycle operation by operation.
constexpr int kMaxStack = 8;

size_t stack_max_rows(const mgrit_gru_cfg* c, const Hier& hr) {
  size_t m = (size_t)c->B;
  for (int l = 0; l + 1 < hr.L; ++l) {
    size_t r = (size_t)((hr.N[l] + c->cf - 1) / c->cf) * c->B;
    if (r > m) m = r;
  }
  return m;
}

mgrit_gru_cfg layer_cfg(const mgrit_gru_cfg& c, int k) {
  mgrit_gru_cfg ck = c;
  if (k > 0) ck.I = c.H;
  return ck;
}

// The cycle of the stack, operation by operation.  Within one relaxation segment -- every point visited at most once -- a layer
// never waits for the layer above it (forward) or below it (adjoint), so an operation runs layer by layer on the single-layer
// kernels: a whole sweep, chain or coarse step of one layer, then ONE product that forms every point's input for the next.
// (Step by step the two-layer solve of 512 points took about 1700 launches of few rows.)
struct StackCycle {
  const mgrit_gru_cfg* c; Hier hr; cudaStream_t s; int nl;
  double* res_acc; int cycle_idx = 0; int rc = MGRIT_OK;
  bool homog = false, fcycle_leg = true;      // as in Cycle
  enum { kNone, kC, kV };
  // F-relaxation (optional) of the first kz intervals of level l, then nothing, the C-step or the evaluation of v
  virtual void segment(int l, int kz, bool f, int last) = 0;
  virtual void coarse_rhs(int l, int np) = 0;      // G_k = v_k - step_l(U'_{k-1}), k = 1..np
  virtual void coarsest(int l) = 0;
  virtual Cycle& layer(int k) = 0;
  virtual ~StackCycle() {}
  void cycle(int l, bool skip_first_f, bool record, int live = 0) {
    const int cf = c->cf;
    if (l == hr.L - 1) { homog = false; coarsest(l); return; }
    const int relax = l == 0 ? c->relax_fine : c->relax_coarse, nc = hr.N[l + 1];
    int kz = homog ? live / cf + 1 : INT_MAX;
    for (int r = 0; r < relax; ++r) { segment(l, kz, !(r == 0 && skip_first_f), kC); if (homog) ++kz; }
    segment(l, kz, !(relax == 0 && skip_first_f), kV);
    const int np = nc < kz ? nc : kz;
    for (int k = 0; k < nl; ++k) {
      Cycle& y = layer(k);
      stream_restrict_residual(y.U[l], cf, y.G[l + 1], y.U[l + 1], y.Ub ? y.Ub[l + 1] : nullptr, np, (i64)y.BH,
                               (l == 0 && record) ? res_acc + cycle_idx : nullptr, s);
    }
    coarse_rhs(l + 1, np);
    cycle(l + 1, false, false, np);
    for (int k = 0; k < nl; ++k) {
      Cycle& y = layer(k);
      stream_correct(y.U[l], y.Ub ? y.Ub[l] : nullptr, cf, y.U[l + 1], nc, (i64)y.BH, s);
    }
    segment(l, INT_MAX, true, kNone);
    if ((c->flags & MGRIT_FLAG_F_CYCLE) && fcycle_leg) {
      fcycle_leg = false;
      cycle(l, true, false);
      fcycle_leg = true;
    }
  }
  int solve(Setup* q) {      // q: what the caller has collected
    if (hr.L == 1) { homog = false; if (!q->run()) return MGRIT_CUDA_ERROR; coarsest(0); return status(); }
    q->zero(res_acc, sizeof(double) * (size_t)(c->iters > 0 ? c->iters : 1));
    if (c->iters <= 0) homog = false;
    if (homog) for (int k = 0; k < nl; ++k) layer(k).zero_levels(q);
    if (!q->run()) return MGRIT_CUDA_ERROR;
    for (cycle_idx = 0; cycle_idx < c->iters && status() == MGRIT_OK; ++cycle_idx)
      cycle(0, cycle_idx > 0 && (c->flags & MGRIT_FLAG_SKIP_DUPLICATE_FRELAX), true);
    return status();
  }
  int status() {
    for (int k = 0; k < nl && rc == MGRIT_OK; ++k) rc = layer(k).rc;
    return rc;
  }
  // the steps of a segment on layer y, one launch per step
  static void steps(Cycle& y, int l, int kz, bool f, int last) {
    const int cf = y.c->cf;
    if (f) y.frelax(l, kz);
    if (last == kC) y.crelax(l, kz);
    if (last == kV) {
      const int nc = y.hr.N[l + 1];
      y.step(StepDesc{l, nc < kz ? nc : kz, cf - 1, cf, y.G[l + 1], 1, 1, y.G[l], cf, cf, cf, cf, 0});
    }
  }
};

struct StackFwdWs {
  FwdWs L[kMaxStack];
  float* gi_l[kMaxStack][kMaxLevels];      // layers >= 1: projections by level
  float *phi, *raw;        // raw results of a coarse step; of a segment as fp32 rows (fp32 engine)
  double* res_acc;
};
// the fused kernels and the state copies they need
bool stack_fused(const mgrit_gru_cfg* c) { return c->operands == MGRIT_OPERANDS_BF16 && c->B <= 128; }

void plan_stack_fwd(const mgrit_gru_cfg* c, int nl, const Hier& hr, Ws& w, StackFwdWs* o) {
  const size_t bh = (size_t)c->B * c->H;
  for (int k = 0; k < nl; ++k) {
    mgrit_gru_cfg ck = layer_cfg(*c, k);
    plan_fwd(&ck, hr, w, &o->L[k]);
    for (int l = 0; l < hr.L; ++l) {
      o->gi_l[k][l] = k > 0 ? w.take<float>((size_t)hr.N[l] * bh * 3) : nullptr;
    }
  }
  o->phi = hr.L > 1 ? w.take<float>((size_t)hr.N[1] * bh) : nullptr;
  o->raw = c->operands == MGRIT_OPERANDS_BF16 ? nullptr : w.take<float>((size_t)c->T * bh);
  o->res_acc = w.take<double>((size_t)(c->iters > 0 ? c->iters : 1));
}

struct StackFwdCycle : StackCycle {
  FwdCycle y[kMaxStack]; const gru_params* p; StackFwdWs* fw;
  Cycle& layer(int k) override { return y[k]; }
  // projection of n points of layer k (rows raw[n, B, H], fp32 rows or already bf16 in the upper layer's xb) for layer k + 1
  void project(int k, int l, const float* raw, int n) {
    const int M = n * c->B;
    if (rc != MGRIT_OK) return;
    if (c->operands == MGRIT_OPERANDS_BF16)
      rc = umma_project_packed(fw->L[k + 1].um.xb, fw->L[k + 1].um.W_ih, p[k + 1].b_ih, fw->gi_l[k + 1][l], nullptr, M, c->H, 3 * c->H, s);
    else
      simt_project(raw, p[k + 1].W_ih, p[k + 1].b_ih, fw->gi_l[k + 1][l], M, c->H, 3 * c->H, s);
  }
  // raw results (before the FAS term) of every point of level l: its unknown, at the C-points v where the segment evaluated it
  void feed(int k, int l, bool v) {
    if (k + 1 >= nl) return;
    const bool bf = c->operands == MGRIT_OPERANDS_BF16;
    stream_raw_rows(y[k].U[l], y[k].G[l], v ? y[k].G[l + 1] : nullptr, c->cf, hr.N[l], (i64)y[k].BH, bf ? nullptr : fw->raw,
                    bf ? fw->L[k + 1].um.xb : nullptr, s);
    project(k, l, fw->raw, hr.N[l]);
  }
  // false: not available here, nothing has been enqueued
  bool run_fp32(FwdCycle& q, int k, int l, int kz, bool f, int last) {
    if (c->operands != MGRIT_OPERANDS_FP32 || !f32_solve_fits(c->H)) return false;
    F32Cycle fc;
    fc.c = c; fc.hr = &hr; fc.adjoint = false; fc.s = s; fc.U = q.U; fc.G = q.G; fc.res_acc = res_acc;
    fc.a.B = c->B; fc.a.H = c->H; fc.a.cell = c->cell; fc.a.W = p[k].W_hh; fc.a.gi = q.gi_of(l); fc.a.b_hh = p[k].b_hh; fc.a.bar = fw->L[k].chain_bar;
    fc.a.nph = 0;
    const int cf = c->cf, N = hr.N[l];
    const i64 BH = (i64)q.BH, st = q.gi_stride(l);
    const bool chain = l == hr.L - 1 && last == kNone && !f;
    const int s0 = chain || f ? 0 : cf - 1;
    F32Phase ph = fc.phase(l, q.U[l] + s0 * BH, (i64)cf * BH, s0);
    ph.op = (st * (s0 + 1) - 1) * BH * 3; ph.op_ss = st * BH * 3; ph.op_ks = st * cf * BH * 3;
    if (chain) { ph.nk = ph.nfull = 1; ph.n = N; }
    else {
      const int nc = N / cf, tail = f ? N % cf : 0;
      ph.n = f ? cf - 1 : 0; ph.nfull = nc; ph.ntail = tail; ph.nk = nc + (tail > 0 ? 1 : 0);
      if (ph.nk > kz) ph.nk = kz;
      if (last == kV) { ph.last_kind = kLastStore; ph.last = q.G[l + 1] + BH; ph.last_ks = BH; }
    }
    fc.add(ph);
    fc.flush();
    return fc.ok;
  }
  void segment(int l, int kz, bool f, int last) override {
    int kinds[32], n = 0;
    const int cf = c->cf;
    if (f) for (int i = 1; i < cf && n < 31; ++i) kinds[n++] = i;
    if (last == kC) kinds[n++] = cf;
    if (last == kV) kinds[n++] = cf + 1;
    for (int k = 0; k < nl && status() == MGRIT_OK; ++k) {
      if (!(cf <= kMaxFwdSweepSteps && y[k].launch_sweep(l, kinds, n, INT_MAX))) {
        // (fp32 phases: the C-step overwrites what other rows of a phase read, so it is a launch of its own)
        const bool part = last == kC && f;
        if (part && run_fp32(y[k], k, l, kz, true, kNone)) steps(y[k], l, kz, false, kC);
        else if (last == kC || !run_fp32(y[k], k, l, kz, f, last)) steps(y[k], l, kz, f, last);
      }
      feed(k, l, last == kV);
    }
  }
  void coarse_rhs(int l, int np) override {
    for (int k = 0; k < nl && status() == MGRIT_OK; ++k) {
      FwdCycle& q = y[k];
      if (k + 1 == nl) { q.step(StepDesc{l, np, 0, 1, q.G[l], 1, 1, nullptr, 0, 0, 1, 1, 1}); continue; }
      // the layer above reads the raw step result: keep it, then form the right-hand side
      q.step(StepDesc{l, np, 0, 1, fw->phi, 0, 1, nullptr, 0, 0, 1, 1, 0});
      const bool bf = c->operands == MGRIT_OPERANDS_BF16;
      stream_subtract_rows(q.G[l] + q.BH, fw->phi, (i64)np * (i64)q.BH, bf ? fw->L[k + 1].um.xb : nullptr, s);
      project(k, l, fw->phi, np);
    }
  }
  void coarsest(int l) override {
    for (int k = 0; k < nl && status() == MGRIT_OK; ++k) {
      FwdCycle& q = y[k];
      const bool chain_first = c->operands == MGRIT_OPERANDS_FP32 && chain32_wins(c, hr.N[l], true);
      if (!(chain_first && q.chain(l)) && !run_fp32(q, k, l, 1, false, kNone) && !q.chain(l))
        for (int j = 1; j <= hr.N[l]; ++j) q.step(StepDesc{l, 1, j - 1, 1, q.U[l], j, 1, q.G[l], j, 1, j, 1, 0});
      feed(k, l, false);
    }
  }
};

bool stack_args_ok(const mgrit_gru_cfg* c, int nl, const gru_params* p) {
  if (!c || !p || nl < 1 || nl > kMaxStack) return false;
  for (int k = 0; k < nl; ++k)
    if (!p[k].W_ih || !p[k].W_hh || !p[k].b_ih || !p[k].b_hh || !aligned32(p[k].W_ih, p[k].W_hh, p[k].b_ih, p[k].b_hh)) return false;
  return true;
}

int stack_forward_impl(const mgrit_gru_cfg* cfg, int nl, const gru_params* p, const float* x, const float* h0, float* gi0, float* h,
                       float* resnorm, void* ws, size_t ws_bytes, cudaStream_t s) {
  if (!stack_args_ok(cfg, nl, p) || !x || !h0 || !gi0 || !h || !ws) return MGRIT_INVALID_ARG;
  if (!aligned32(x, h0, gi0, h, ws)) return MGRIT_INVALID_ARG;
  mgrit_gru_cfg c = *cfg;
  Hier hr;
  int rc = check_cfg(&c, &hr);
  if (rc) return rc;
  if (is_tf32(&c)) return MGRIT_UNSUPPORTED;      // the stacked solve runs on the fp32 or the bf16 engine
  if (nl > 1) { mgrit_gru_cfg c1 = layer_cfg(c, 1); Hier h1; rc = check_cfg(&c1, &h1); if (rc) return rc; }
  Ws w{(char*)ws, ws_bytes, 0};
  StackFwdWs fw;
  plan_stack_fwd(&c, nl, hr, w, &fw);
  if (!w.fits()) return MGRIT_WORKSPACE_TOO_SMALL;
  const size_t bh = (size_t)c.B * c.H, slot = (size_t)nl * bh;
  const bool bf = c.operands == MGRIT_OPERANDS_BF16, fused = stack_fused(&c);
  if (bf) {
    for (int k = 0; k < nl; ++k) fw.L[k].um.gib = nullptr;      // stacked layers: fp32 projections throughout
    rc = umma_prepare_fwd(&c, &p[0], x, gi0, &fw.L[0].um, s);
    if (rc) return rc;
    for (int k = 1; k < nl; ++k) {
      umma_convert(p[k].W_hh, fw.L[k].um.W_hh, (i64)3 * c.H * c.H, s);
      umma_convert(p[k].W_ih, fw.L[k].um.W_ih, (i64)3 * c.H * c.H, s);
    }
  } else {
    simt_project(x, p[0].W_ih, p[0].b_ih, gi0, c.T * c.B, c.I, 3 * c.H, s);
  }
  Setup setup(s);
  StackFwdCycle cy;
  cy.c = &c; cy.hr = hr; cy.s = s; cy.nl = nl; cy.res_acc = fw.res_acc; cy.p = p; cy.fw = &fw;
  mgrit_gru_cfg ck[kMaxStack];
  for (int k = 0; k < nl; ++k) {
    FwdWs& q = fw.L[k];
    ck[k] = layer_cfg(c, k);
    zero_guess(q.U[0], c, hr, bh, &setup);
    for (int l = 0; l < hr.L; ++l) setup.copy(q.U[l], h0 + k * bh, bh);
    if (q.chain_xw) setup.zero(q.chain_xw, q.chain_xw_bytes);
    if (fused) {
      setup.zero(q.sweep_ctr, sizeof(int) * q.sweep_ctr_n);
      zero_guess(q.Ub[0], c, hr, bh, &setup);
      for (int l = 0; l < hr.L; ++l) setup.to_bf16(q.Ub[l], h0 + k * bh, bh);
    }
    FwdCycle& y = cy.y[k];
    y.c = &ck[k]; y.hr = hr; y.s = s; y.U = q.U; y.G = q.G; y.res_acc = fw.res_acc; y.BH = bh; y.p = &p[k]; y.um = &q.um; y.fw = &q;
    y.Ub = fused ? q.Ub : nullptr;
    y.gi = gi0;
    if (k > 0) y.gi_lv = fw.gi_l[k];
  }
  rc = cy.solve(&setup);
  if (rc) return rc;
  for (int k = 0; k < nl; ++k) stream_gather_rows(h + k * bh, (i64)slot, fw.L[k].U[0] + bh, (i64)bh, c.T, (i64)bh, s);
  if (resnorm && hr.L > 1 && c.iters > 0) {
    rc = fetch_resnorm(fw.res_acc, resnorm, c.iters, s);
    if (rc) return rc;
    return finish(s, true);
  }
  return finish(s, false);
}

struct StackLayerAdj {
  AdjWs w;
  float* cnp[kMaxLevels]; __nv_bfloat16* cnpb[kMaxLevels];     // c_n' of every level: what a cell sends to its input
  float* hk;                 // this layer's given states [T, B, H], contiguous
  float* gik;                // layers >= 1: input projection of the layer below's given states [T, B, 3H]
  __nv_bfloat16* Wihb;       // layers >= 1, tensor-core engine: W_ih as bf16 [3H, H]
};
struct StackAdjWs {
  double* res_acc;
  float *dx, *lsum, *nu, *gnu, *lamk, *dxk;
  StackLayerAdj L[kMaxStack];
};

void plan_stack_adj(const mgrit_gru_cfg* c, int nl, const Hier& hr, Ws& w, StackAdjWs* o) {
  const size_t bh = (size_t)c->B * c->H, TB = (size_t)c->T * c->B;
  const bool bf16 = c->operands == MGRIT_OPERANDS_BF16;
  o->res_acc = w.take<double>((size_t)(c->iters > 0 ? c->iters : 1));
  o->dx = w.take<float>(TB * c->H);                                          // rows sent to the layer below, by incoming point
  o->lsum = w.take<float>(stack_max_rows(c, hr) * c->H);
  o->nu = w.take<float>((size_t)(hr.N[hr.L - 1] + 1) * bh);
  o->gnu = w.take<float>((size_t)(hr.N[hr.L - 1] + 1) * bh);
  o->lamk = w.take<float>(TB * c->H);
  o->dxk = w.take<float>(TB * c->H);
  for (int k = 0; k < nl; ++k) {
    StackLayerAdj& L = o->L[k];
    mgrit_gru_cfg ck = layer_cfg(*c, k);
    plan_adj(&ck, hr, w, &L.w);
    for (int l = 0; l < hr.L; ++l) {
      const size_t n = (size_t)hr.N[l] * bh;
      L.cnp[l] = bf16 ? nullptr : l == 0 ? L.w.cnp : w.take<float>(n);
      L.cnpb[l] = !bf16 ? nullptr : l == 0 ? L.w.cnpb : w.take<__nv_bfloat16>(n);
    }
    L.hk = w.take<float>(TB * c->H);
    L.gik = k > 0 ? w.take<float>(TB * 3 * c->H) : nullptr;
    L.Wihb = (bf16 && k > 0) ? w.take<__nv_bfloat16>((size_t)3 * c->H * c->H) : nullptr;
  }
}

struct StackAdjCycle : StackCycle {
  AdjCycle y[kMaxStack]; const gru_params* p; StackAdjWs* w;
  Cycle& layer(int k) override { return y[k]; }
  // what layer k (>= 1) sends to its input in the n steps that leave points j0, j0 + js, ... of level l  ->  w->dx[n, B, H]
  void send(int k, int l, int j0, int js, int n) {
    if (k == 0 || status() != MGRIT_OK) return;
    const i64 bh = (i64)y[k].BH;
    StackLayerAdj& L = w->L[k];
    AdjStepArgs a{};
    a.B = c->B; a.H = c->H; a.lin_ks = js * bh; a.coef_ks = -js * bh; a.W_hh = p[k].W_hh;
    const bool bf16 = c->operands == MGRIT_OPERANDS_BF16;
    // (the operand buffer holds so many points at a time)
    const int step = bf16 ? (int)(L.w.um.apack_elems / ((size_t)3 * bh)) : n;
    for (int i0 = 0; i0 < n; i0 += step) {
      const int m = n - i0 < step ? n - i0 : step;
      const i64 row0 = ((i64)hr.N[l] - 1 - j0 - (i64)i0 * js) * bh;      // the step leaving point j is stored at row N - 1 - j
      a.M = m * c->B;
      a.lin = y[k].U[l] + ((i64)j0 + (i64)i0 * js) * bh;
      float* out = w->dx + (i64)i0 * bh;
      // (a middle layer's incoming sensitivities include what the layer above sent, which these rows still hold)
      const bool mid = k < nl - 1;
      if (bf16) {
        if (mid) { a.ladd = out; a.ladd_ks = bh; }
        a.crb = L.w.crb[l] + row0; a.czb = L.w.czb[l] + row0; a.cnb = L.cnpb[l] + row0;
        rc = umma_adj_dx(a, L.w.um.W_ihT, c->H, out, &L.w.um, s);
        if (rc) return;
      } else {
        a.cr = L.w.cr[l] + row0; a.cz = L.w.cz[l] + row0; a.cn = L.cnp[l] + row0;
        if (mid) {
          stream_sum_rows(w->lamk, a.lin, a.lin_ks, out, bh, m, bh, s);
          a.lin = w->lamk; a.lin_ks = bh;
        }
        simt_adj_dx(a, p[k].W_ih, c->H, out, s);
      }
    }
  }
  void part(int l, int kz, bool f, int last) {      // F-steps and v leave the points as they were sent; a C-step is a part of its own
    const int cf = c->cf, N = hr.N[l], nc = N / cf;
    for (int k = nl - 1; k >= 0 && status() == MGRIT_OK; --k) {
      AdjCycle& q = y[k];
      const i64 bh = (i64)q.BH;
      q.lsum = w->lsum;
      std::vector<StepDesc> d;
      std::vector<const float*> la;
      if (f) {
        const int nki = nc, tail = N % cf;
        for (int sI = 1; sI < cf; ++sI) {
          const int nk = nki + (sI <= tail ? 1 : 0);
          d.push_back(StepDesc{l, nk < kz ? nk : kz, sI - 1, cf, q.U[l], sI, cf, q.G[l], sI, cf, sI, cf, 0});
          la.push_back(w->dx + (i64)(sI - 1) * bh);
        }
      }
      if (last != kNone) {
        float* out = last == kV ? q.G[l + 1] : q.U[l];
        d.push_back(StepDesc{l, nc < kz ? nc : kz, cf - 1, cf, out, last == kV ? 1 : cf, last == kV ? 1 : cf, q.G[l], cf, cf, cf, cf, 0});
        la.push_back(f ? w->dx + (i64)(cf - 1) * bh : w->dx);
      }
      q.run_steps(d.data(), (int)d.size(), k == nl - 1 ? nullptr : la.data(), f ? (i64)cf * bh : bh);
      if (f) send(k, l, 0, 1, kz < nc ? kz * cf : N);
      else send(k, l, cf - 1, cf, nc < kz ? nc : kz);
    }
  }
  void segment(int l, int kz, bool f, int last) override {
    if (last == kC) {        // (the C-step overwrites points that F-steps left from)
      if (f) part(l, kz, true, kNone);
      part(l, kz, false, kC);
    } else {
      part(l, kz, f, last);
    }
  }
  void coarse_rhs(int l, int np) override {
    for (int k = nl - 1; k >= 0 && status() == MGRIT_OK; --k) {
      AdjCycle& q = y[k];
      q.lsum = w->lsum; q.ladd = k == nl - 1 ? nullptr : w->dx; q.ladd_ks = (i64)q.BH;
      q.step(StepDesc{l, np, 0, 1, q.G[l], 1, 1, nullptr, 0, 0, 1, 1, 1});
      q.ladd = nullptr;
      send(k, l, 0, 1, np);
    }
  }
  bool chain(int k, int l, float* mu, const float* g) {
    if (c->operands != MGRIT_OPERANDS_FP32 || !f32_solve_fits(c->H)) return y[k].chain_on(l, mu, g);
    float* Us[kMaxLevels] = {}; float* Gs[kMaxLevels] = {};
    Us[l] = mu; Gs[l] = const_cast<float*>(g);
    AdjWs& q = w->L[k].w;
    F32Cycle fc;
    fc.c = c; fc.hr = &hr; fc.adjoint = true; fc.s = s; fc.U = Us; fc.G = Gs; fc.res_acc = res_acc;
    fc.a.B = c->B; fc.a.H = c->H; fc.a.cell = c->cell; fc.a.W = p[k].W_hh; fc.a.bar = q.chain_bar;
    fc.a.coef[l][0] = q.a[l]; fc.a.coef[l][1] = q.cr[l]; fc.a.coef[l][2] = q.cz[l]; fc.a.coef[l][3] = q.cn[l];
    fc.a.nph = 0;
    fc.cycle(l, false, false);       // (the coarsest level: one phase)
    fc.flush();
    return fc.ok || y[k].chain_on(l, mu, g);
  }
  // Below the top layer mu_s = step(mu_{s-1} + d_{s-1}) + g_s: a chain in nu_s = mu_s + d_s with the source g_s + d_s.
  void coarsest(int l) override {
    const int N = hr.N[l];
    for (int k = nl - 1; k >= 0 && status() == MGRIT_OK; --k) {
      AdjCycle& q = y[k];
      const i64 bh = (i64)q.BH;
      if (k == nl - 1) {
        if (!chain(k, l, q.U[l], q.G[l]))
          for (int j = 1; j <= N; ++j) q.step(StepDesc{l, 1, j - 1, 1, q.U[l], j, 1, q.G[l], j, 1, j, 1, 0});
      } else {
        stream_nu_start(w->nu, w->gnu, q.U[l], q.G[l], w->dx, N, bh, s);
        if (chain(k, l, w->nu, w->gnu)) {
          stream_nu_finish(q.U[l], w->nu, w->dx, N, bh, s);
        } else {
          q.lsum = w->lsum; q.ladd_ks = bh;
          for (int j = 1; j <= N; ++j) { q.ladd = w->dx + (i64)(j - 1) * bh; q.step(StepDesc{l, 1, j - 1, 1, q.U[l], j, 1, q.G[l], j, 1, j, 1, 0}); }
          q.ladd = nullptr;
        }
      }
      send(k, l, 0, 1, N);
    }
  }
};

// time-parallel gradient pass of one layer given its total output sensitivities (row (t, b) at lam + t*lam_ts + b*H)
int stack_layer_gradients(const mgrit_gru_cfg& ck, const gru_params* pk, const float* xk, const float* h0k, StackLayerAdj& L,
                          const float* lam, i64 lam_ts, float* dx, const gru_grads* g, cudaStream_t s) {
  const i64 M = (i64)ck.T * ck.B;
  if (ck.operands == MGRIT_OPERANDS_BF16)
    return umma_gradients(&ck, pk, xk, h0k, L.hk, lam, lam_ts, L.w.crb[0], L.w.czb[0], L.w.cnb[0], L.cnpb[0], dx, g, &L.w.um, false, s);
  simt_gradients((int)M, ck.B, ck.H, ck.I, lam, lam_ts, L.w.cr[0], L.w.cz[0], L.w.cn[0], L.cnp[0], h0k, L.hk, xk, pk->W_ih, dx, g, L.w.grad_scratch, s);
  return MGRIT_OK;
}

int stack_adjoint_impl(const mgrit_gru_cfg* cfg, int nl, const gru_params* p, const float* x, const float* h0, const float* gi0,
                       const float* h, const float* dh_seed, const float* dhT, float* dh, float* dh0, float* dx, const gru_grads* g,
                       float* resnorm, void* ws, size_t ws_bytes, cudaStream_t s) {
  if (!stack_args_ok(cfg, nl, p) || !x || !h0 || !gi0 || !h || !dh0 || !g || !ws) return MGRIT_INVALID_ARG;
  if (!dh_seed && !dhT) return MGRIT_INVALID_ARG;
  if (!aligned32(x, h0, gi0, h, dh_seed, dhT, dh, dh0, dx, ws)) return MGRIT_INVALID_ARG;
  for (int k = 0; k < nl; ++k)
    if (!g[k].dW_ih || !g[k].dW_hh || !g[k].db_ih || !g[k].db_hh || !aligned32(g[k].dW_ih, g[k].dW_hh, g[k].db_ih, g[k].db_hh))
      return MGRIT_INVALID_ARG;
  mgrit_gru_cfg c = *cfg;
  Hier hr;
  int rc = check_cfg(&c, &hr);
  if (rc) return rc;
  if (is_tf32(&c)) return MGRIT_UNSUPPORTED;      // the stacked solve runs on the fp32 or the bf16 engine
  if (nl > 1) { mgrit_gru_cfg c1 = layer_cfg(c, 1); Hier h1; rc = check_cfg(&c1, &h1); if (rc) return rc; }
  Ws w{(char*)ws, ws_bytes, 0};
  StackAdjWs aw;
  plan_stack_adj(&c, nl, hr, w, &aw);
  if (!w.fits()) return MGRIT_WORKSPACE_TOO_SMALL;
  const size_t bh = (size_t)c.B * c.H, slot = (size_t)nl * bh;
  const int T = c.T;
  const bool bf16 = c.operands == MGRIT_OPERANDS_BF16;

  // every layer's given states as their own [T, B, H] array; input projections of the layers above the first
  for (int k = 0; k < nl; ++k) stream_gather_rows(aw.L[k].hk, (i64)bh, h + (size_t)k * bh, (i64)slot, T, (i64)bh, s);
  for (int k = 0; k < nl; ++k) {
    StackLayerAdj& L = aw.L[k];
    mgrit_gru_cfg ck = layer_cfg(c, k);
    if (bf16) {
      rc = umma_prepare_adj(&ck, &p[k], h0 + (size_t)k * bh, L.hk, &L.w.um, false, s);
      if (rc) return rc;
    }
    if (k > 0) {
      if (bf16) {
        umma_convert(p[k].W_ih, L.Wihb, (i64)3 * c.H * c.H, s);
        rc = umma_project_rows(aw.L[k - 1].hk, L.w.um.xb, L.Wihb, p[k].b_ih, L.gik, T * c.B, c.H, 3 * c.H, s);
        if (rc) return rc;
      } else {
        simt_project(aw.L[k - 1].hk, p[k].W_ih, p[k].b_ih, L.gik, T * c.B, c.H, 3 * c.H, s);
      }
    }
    for (int l = 0; l < hr.L; ++l) {
      LinArgs a{};
      a.M = hr.N[l] * c.B; a.B = c.B; a.H = c.H; a.h0 = h0 + (size_t)k * bh; a.h = L.hk; a.stride_t = hr.stride_t[l];
      a.t0 = hr.rem[l]; a.gi = k == 0 ? gi0 : L.gik;
      a.W_hh = p[k].W_hh; a.b_hh = p[k].b_hh; a.gamma = hr.gamma[l]; a.cell = c.cell;
      a.a = L.w.a[l]; a.cr = L.w.cr[l]; a.cz = L.w.cz[l]; a.cn = L.w.cn[l]; a.cnp = L.cnp[l];
      a.crb = L.w.crb[l]; a.czb = L.w.czb[l]; a.cnb = L.w.cnb[l]; a.cnpb = L.cnpb[l];
      if (bf16) { rc = umma_linearise(a, &L.w.um, s); if (rc) return rc; }
      else simt_linearise(a, s);
    }
  }
  // mu_0 = lambda_T (all layers); zero initial guess elsewhere; fine-level source = reversed dh_seed
  StackAdjCycle cy;
  cy.homog = !dh_seed;
  cy.c = &c; cy.hr = hr; cy.s = s; cy.nl = nl; cy.res_acc = aw.res_acc; cy.p = p; cy.w = &aw;
  Setup setup(s);
  mgrit_gru_cfg ck[kMaxStack];
  float* Gl[kMaxStack][kMaxLevels];
  for (int k = 0; k < nl; ++k) {
    AdjWs& q = aw.L[k].w;
    ck[k] = layer_cfg(c, k);
    zero_guess(q.U[0], c, hr, bh, &setup);
    if (q.chain_xw) setup.zero(q.chain_xw, q.chain_xw_bytes);
    if (c.operands == MGRIT_OPERANDS_BF16 && hr.L > 1) setup.zero(q.um.sweep_ctr, sizeof(int) * q.um.sweep_ctr_n);
    for (int l = 0; l < hr.L; ++l) Gl[k][l] = q.G[l];
    if (!dh_seed) Gl[k][0] = nullptr;
    const float* const seed = dh_seed ? dh_seed + (size_t)(T - 1) * slot + k * bh : nullptr;
    const float* const top = k == nl - 1 ? dhT : nullptr;      // loss on the top layer's last state
    for (int l = 0; l < hr.L; ++l) {
      if (seed || top) setup.copy(q.U[l], seed ? seed : top, bh, seed ? top : nullptr);
      else setup.zero(q.U[l], sizeof(float) * bh);
    }
    if (dh_seed) {
      setup.zero(q.G[0] + (size_t)T * bh, sizeof(float) * bh);
      if (T > 1) stream_gather_rows(q.G[0] + bh, (i64)bh, dh_seed + (size_t)(T - 2) * slot + k * bh, -(i64)slot, T - 1, (i64)bh, s);
    }
    AdjCycle& y = cy.y[k];
    y.c = &ck[k]; y.hr = hr; y.s = s; y.U = q.U; y.G = Gl[k]; y.res_acc = aw.res_acc; y.BH = bh; y.p = &p[k]; y.w = &q;
  }
  rc = cy.solve(&setup);
  if (rc) return rc;

  for (int k = 0; k < nl; ++k) {
    const float* U0 = aw.L[k].w.U[0];
    if (dh) stream_gather_rows(dh + k * bh, (i64)slot, U0 + (size_t)(T - 1) * bh, -(i64)bh, T, (i64)bh, s);
    cudaMemcpyAsync(dh0 + k * bh, U0 + (size_t)T * bh, sizeof(float) * bh, cudaMemcpyDeviceToDevice, s);
  }
  // gradient pass, top layer first: a layer's total output sensitivity is its entry of the unknown plus what the layer
  // above sends to its input (that layer's input gradient)
  for (int k = nl - 1; k >= 0; --k) {
    const float* lam = aw.L[k].w.U[0] + (size_t)(T - 1) * bh;
    i64 lam_ts = -(i64)bh;
    if (k < nl - 1) {
      stream_sum_rows(aw.lamk, lam, lam_ts, aw.dxk, (i64)bh, T, (i64)bh, s);
      lam = aw.lamk; lam_ts = (i64)bh;
    }
    rc = stack_layer_gradients(ck[k], &p[k], k == 0 ? x : aw.L[k - 1].hk, h0 + (size_t)k * bh, aw.L[k], lam, lam_ts, k > 0 ? aw.dxk : dx, &g[k], s);
    if (rc) return rc;
  }
  if (resnorm && hr.L > 1 && c.iters > 0) {
    rc = fetch_resnorm(aw.res_acc, resnorm, c.iters, s);
    if (rc) return rc;
    return finish(s, true);
  }
  return finish(s, false);
}


// ======================================================================================================
// Implicit LSTM: the state of a time point is (c, h); level arrays are [N_l + 1][2][B][H] (part 0 = c, part 1 = h) and
// the same Cycle drives them.  fp32 engine only (four-gate FFMA products).
struct LstmFwdWs {
  float* U[kMaxLevels]; float* G[kMaxLevels]; double* res_acc; float *tmpC, *tmpH; size_t maxM; Tf32Ws tf; LstmBfWs bf;
  uint4* chain_xw; size_t chain_xw_bytes; unsigned chain_steps;      // exchange words of the persistent chain kernel (bf16 operands)
};
struct LstmAdjWs {
  float* U[kMaxLevels]; float* G[kMaxLevels]; double* res_acc;
  float *a[kMaxLevels], *p[kMaxLevels], *ci[kMaxLevels], *cf[kMaxLevels], *cg[kMaxLevels], *co[kMaxLevels];
  __nv_bfloat16 *cib[kMaxLevels], *cfb[kMaxLevels], *cgb[kMaxLevels], *cob[kMaxLevels];    // bf16 operands: the gate coefficients as bf16 instead
  float *tmpC, *tmpH, *hk, *dA, *grad_scratch; size_t maxM; Tf32Ws tf; LstmBfWs bf;
  uint4* chain_xw; size_t chain_xw_bytes; unsigned chain_steps;
};

void plan_lstm_fwd(const mgrit_gru_cfg* c, const Hier& hr, Ws& w, LstmFwdWs* o) {
  const size_t slot = (size_t)2 * c->B * c->H;
  for (int l = 0; l < hr.L; ++l) {
    o->U[l] = w.take<float>((size_t)(hr.N[l] + 1) * slot);
    o->G[l] = l == 0 ? nullptr : w.take<float>((size_t)(hr.N[l] + 1) * slot);
  }
  o->res_acc = w.take<double>((size_t)(c->iters > 0 ? c->iters : 1));
  o->maxM = stack_max_rows(c, hr);
  o->tmpC = w.take<float>(o->maxM * c->H);
  o->tmpH = w.take<float>(o->maxM * c->H);
  if (is_tf32(c)) tf32_plan_fwd(c, hr.N, hr.L, w.base, &w.off, &o->tf, 4);
  if (c->operands == MGRIT_OPERANDS_BF16) lstmbf_plan_fwd(c, o->maxM, w.base, &w.off, &o->bf);
  o->chain_xw = nullptr; o->chain_xw_bytes = 0; o->chain_steps = 0;
  if (c->operands == MGRIT_OPERANDS_BF16) {
    o->chain_xw_bytes = serial_xw_bytes(c->B, c->H, 1);
    o->chain_xw = reinterpret_cast<uint4*>(w.take<char>(o->chain_xw_bytes));
  }
}

void plan_lstm_adj(const mgrit_gru_cfg* c, const Hier& hr, Ws& w, LstmAdjWs* o) {
  const size_t bh = (size_t)c->B * c->H, slot = 2 * bh, TB = (size_t)c->T * c->B;
  for (int l = 0; l < hr.L; ++l) {
    o->U[l] = w.take<float>((size_t)(hr.N[l] + 1) * slot);
    o->G[l] = w.take<float>((size_t)(hr.N[l] + 1) * slot);
    const size_t n = (size_t)hr.N[l] * bh;
    o->a[l] = w.take<float>(n); o->p[l] = w.take<float>(n);
    if (c->operands == MGRIT_OPERANDS_BF16) {
      o->ci[l] = o->cf[l] = o->cg[l] = o->co[l] = nullptr;
      o->cib[l] = w.take<__nv_bfloat16>(n); o->cfb[l] = w.take<__nv_bfloat16>(n);
      o->cgb[l] = w.take<__nv_bfloat16>(n); o->cob[l] = w.take<__nv_bfloat16>(n);
    } else {
      o->ci[l] = w.take<float>(n); o->cf[l] = w.take<float>(n); o->cg[l] = w.take<float>(n); o->co[l] = w.take<float>(n);
      o->cib[l] = o->cfb[l] = o->cgb[l] = o->cob[l] = nullptr;
    }
  }
  o->res_acc = w.take<double>((size_t)(c->iters > 0 ? c->iters : 1));
  o->maxM = stack_max_rows(c, hr);
  o->tmpC = w.take<float>(o->maxM * c->H);
  o->tmpH = w.take<float>(o->maxM * c->H);
  o->hk = w.take<float>(TB * c->H);
  o->dA = w.take<float>(TB * 4 * c->H);
  o->grad_scratch = c->operands == MGRIT_OPERANDS_FP32 ? w.take<float>(simt_gradients_scratch((int)TB, 4 * c->H, c->H, c->I)) : nullptr;
  if (is_tf32(c)) tf32_plan_adj(c, hr.N, hr.L, w.base, &w.off, &o->tf, 4);
  if (c->operands == MGRIT_OPERANDS_BF16) lstmbf_plan_adj(c, o->maxM, w.base, &w.off, &o->bf);
  o->chain_xw = nullptr; o->chain_xw_bytes = 0; o->chain_steps = 0;
  if (c->operands == MGRIT_OPERANDS_BF16) {
    o->chain_xw_bytes = serial_xw_bytes(c->B, c->H, 4);
    o->chain_xw = reinterpret_cast<uint4*>(w.take<char>(o->chain_xw_bytes));
  }
}

struct LstmFwdCycle : Cycle {
  const gru_params* p; const float* gi; LstmFwdWs* fw;
  // bf16: a step that ends at F-points leaves its hidden rows as bf16 for the next one, which reads the same slots (rows `left` in
  // the order of the step's rows).  Nothing else writes F-points between two steps of a relaxation.  Packing 16384 rows of 1024
  // units in front of a step takes 26 us; a training step at T = 2048, B = 32, H = 1024 13.88 -> 13.67 ms.
  __nv_bfloat16* left = nullptr; const float* left_of = nullptr; i64 left_ks = 0; int left_nk = 0;
  bool chain(int l) override {
    if (c->operands != MGRIT_OPERANDS_BF16 || !fw->chain_xw) return false;
    const i64 bh = (i64)c->B * c->H, st = hr.stride_t[l];
    LstmChainFwdArgs a{};
    a.B = c->B; a.H = c->H; a.nsteps = hr.N[l]; a.u = U[l];
    a.gi = gi + (st - 1) * bh * 4; a.gi_step = st * bh * 4;
    a.g = G[l]; a.W = fw->bf.W_hh; a.b_hh = p->b_hh; a.gamma = hr.gamma[l]; a.cell = c->cell;
    a.xw = fw->chain_xw; a.xw_bytes = fw->chain_xw_bytes; a.step0 = fw->chain_steps; fw->chain_steps += hr.N[l];
    return lstm_chain_fwd_solve(a, s);
  }
  int launch_step(const StepDesc& d) override {
    const size_t bh = (size_t)c->B * c->H, slot = 2 * bh;
    const i64 st = hr.stride_t[d.l];
    LstmFwdArgs a;
    a.M = d.nk * c->B; a.B = c->B; a.H = c->H;
    a.cin = U[d.l] + (size_t)d.in_slot * slot; a.hin = a.cin + bh; a.in_ks = (i64)d.in_stride * slot;
    a.cout = fw->tmpC; a.hout = fw->tmpH;
    a.gi = gi + ((i64)st * d.tgt_slot - 1) * (i64)bh * 4; a.gi_ks = st * d.tgt_stride * (i64)bh * 4;
    a.W_hh = p->W_hh; a.b_hh = p->b_hh; a.gamma = hr.gamma[d.l]; a.cell = c->cell;
    // the tensor-core engines write the level array from their epilogue; the FFMA engine leaves raw results to combine
    const bool fused = c->operands != MGRIT_OPERANDS_FP32;
    a.up = LstmUpdate{};
    if (fused)
      a.up = LstmUpdate{d.out + (size_t)d.out_slot * slot, (i64)d.out_stride * (i64)slot, d.gadd ? d.gadd + (size_t)d.gadd_slot * slot : nullptr,
                        (i64)d.gadd_stride * (i64)slot, (i64)bh, d.mode};
    if (is_tf32(c)) { int r = tf32_lstm_fwd_step(a, &fw->tf, s); if (r) return r; }
    else if (c->operands == MGRIT_OPERANDS_BF16) {
      const bool same = left && left_of == a.cin && left_ks == a.in_ks && d.nk <= left_nk;
      const bool leave = fw->bf.Apack2 && d.out == U[d.l] && d.mode == 0 && d.nk > 1 && d.out_slot % c->cf != 0 && lstmbf_leaves_rows(a.M);
      __nv_bfloat16* const to = same && left == fw->bf.Apack2 ? fw->bf.Apack : fw->bf.Apack2;      // not what this step reads
      int r = lstmbf_fwd_step(a, same ? left : nullptr, leave ? to : nullptr, &fw->bf, s);
      if (r) return r;
      left = leave ? to : nullptr; left_of = a.up.out; left_ks = a.up.out_ks; left_nk = d.nk;
    }
    else simt_lstm_fwd_step(a, s);
    for (int part = 0; part < 2 && !fused; ++part) {
      const float* g = d.gadd ? d.gadd + (size_t)d.gadd_slot * slot + part * bh : nullptr;
      stream_combine_rows(part == 0 ? fw->tmpC : fw->tmpH, g, (i64)d.gadd_stride * slot, d.out + (size_t)d.out_slot * slot + part * bh,
                          (i64)d.out_stride * slot, c->B, c->H, (i64)a.M, d.mode, s);
    }
    return MGRIT_OK;
  }
};

struct LstmAdjCycle : Cycle {
  const gru_params* p; LstmAdjWs* w;
  bool chain(int l) override {
    if (c->operands != MGRIT_OPERANDS_BF16 || !w->chain_xw) return false;
    const i64 bh = (i64)c->B * c->H;
    const i64 row0 = (i64)(hr.N[l] - 1) * bh;     // step s = 1 applies forward step N_l, stored at row N_l - 1
    LstmChainAdjArgs a{};
    a.B = c->B; a.H = c->H; a.nsteps = hr.N[l]; a.mu = U[l];
    a.a = w->a[l] + row0; a.p = w->p[l] + row0; a.ci = w->cib[l] + row0; a.cf = w->cfb[l] + row0; a.cg = w->cgb[l] + row0;
    a.co = w->cob[l] + row0; a.coef_step = -bh;
    a.g = G[l]; a.WT = w->bf.W_hhT;
    a.xw = w->chain_xw; a.xw_bytes = w->chain_xw_bytes; a.step0 = w->chain_steps; w->chain_steps += hr.N[l];
    return lstm_chain_adj_solve(a, s);
  }
  int launch_step(const StepDesc& d) override {
    const size_t bh = (size_t)c->B * c->H, slot = 2 * bh;
    const i64 row0 = (i64)(hr.N[d.l] - d.tgt_slot) * (i64)bh;
    LstmAdjArgs a;
    a.M = d.nk * c->B; a.B = c->B; a.H = c->H;
    a.lc = U[d.l] + (size_t)d.in_slot * slot; a.lh = a.lc + bh; a.in_ks = (i64)d.in_stride * slot;
    a.lc_out = w->tmpC; a.lh_out = w->tmpH;
    a.a = w->a[d.l] + row0; a.p = w->p[d.l] + row0; a.coef_ks = -(i64)d.tgt_stride * (i64)bh;
    const bool cb = w->cib[d.l] != nullptr;      // (the four gate coefficients: bf16 arrays on the bf16 engine, fp32 arrays otherwise)
    a.ci = cb ? nullptr : w->ci[d.l] + row0; a.cf = cb ? nullptr : w->cf[d.l] + row0;
    a.cg = cb ? nullptr : w->cg[d.l] + row0; a.co = cb ? nullptr : w->co[d.l] + row0;
    a.cib = cb ? w->cib[d.l] + row0 : nullptr; a.cfb = cb ? w->cfb[d.l] + row0 : nullptr;
    a.cgb = cb ? w->cgb[d.l] + row0 : nullptr; a.cob = cb ? w->cob[d.l] + row0 : nullptr;
    a.W_hh = p->W_hh;
    const bool fused = c->operands != MGRIT_OPERANDS_FP32;
    a.up = LstmUpdate{};
    if (fused)
      a.up = LstmUpdate{d.out + (size_t)d.out_slot * slot, (i64)d.out_stride * (i64)slot, d.gadd ? d.gadd + (size_t)d.gadd_slot * slot : nullptr,
                        (i64)d.gadd_stride * (i64)slot, (i64)bh, d.mode};
    if (is_tf32(c)) { int r = tf32_lstm_adj_step(a, &w->tf, s); if (r) return r; }
    else if (c->operands == MGRIT_OPERANDS_BF16) { int r = lstmbf_adj_step(a, &w->bf, s); if (r) return r; }
    else simt_lstm_adj_step(a, s);
    for (int part = 0; part < 2 && !fused; ++part) {
      const float* g = d.gadd ? d.gadd + (size_t)d.gadd_slot * slot + part * bh : nullptr;
      stream_combine_rows(part == 0 ? w->tmpC : w->tmpH, g, (i64)d.gadd_stride * slot, d.out + (size_t)d.out_slot * slot + part * bh,
                          (i64)d.out_stride * slot, c->B, c->H, (i64)a.M, d.mode, s);
    }
    return MGRIT_OK;
  }
};

int lstm_check(const mgrit_gru_cfg* cfg, Hier* hr) {
  if (!cfg) return MGRIT_INVALID_ARG;
  return check_cfg(cfg, hr);        // (bf16 and tf32 operands: check_cfg applies the tensor-core engines' shape limits)
}

int lstm_forward_impl(const mgrit_gru_cfg* cfg, const gru_params* p, const float* x, const float* u0, float* gi, float* u,
                      float* resnorm, void* ws, size_t ws_bytes, cudaStream_t s) {
  if (!cfg || !p || !x || !u0 || !gi || !u || !ws || !p->W_ih || !p->W_hh || !p->b_ih || !p->b_hh) return MGRIT_INVALID_ARG;
  if (!aligned32(x, u0, gi, u, ws, p->W_ih, p->W_hh, p->b_ih, p->b_hh)) return MGRIT_INVALID_ARG;
  mgrit_gru_cfg c = *cfg;
  Hier hr;
  int rc = lstm_check(&c, &hr);
  if (rc) return rc;
  Ws w{(char*)ws, ws_bytes, 0};
  LstmFwdWs fw;
  plan_lstm_fwd(&c, hr, w, &fw);
  if (!w.fits()) return MGRIT_WORKSPACE_TOO_SMALL;
  const size_t slot = (size_t)2 * c.B * c.H;
  if (is_tf32(&c)) { rc = tf32_prepare_fwd(&c, p, x, gi, &fw.tf, s); if (rc) return rc; }
  else if (c.operands == MGRIT_OPERANDS_BF16) { rc = lstmbf_prepare_fwd(&c, p, x, gi, &fw.bf, s); if (rc) return rc; }
  else simt_project(x, p->W_ih, p->b_ih, gi, c.T * c.B, c.I, 4 * c.H, s);
  Setup setup(s);
  zero_guess(fw.U[0], c, hr, slot, &setup);
  for (int l = 0; l < hr.L; ++l) setup.copy(fw.U[l], u0, slot);
  if (fw.chain_xw) setup.zero(fw.chain_xw, fw.chain_xw_bytes);
  LstmFwdCycle cy;
  cy.c = &c; cy.hr = hr; cy.s = s; cy.U = fw.U; cy.G = fw.G; cy.res_acc = fw.res_acc; cy.BH = slot;
  cy.p = p; cy.gi = gi; cy.fw = &fw;
  rc = cy.solve(&setup);
  if (rc) return rc;
  cudaMemcpyAsync(u, fw.U[0] + slot, sizeof(float) * (size_t)c.T * slot, cudaMemcpyDeviceToDevice, s);
  if (resnorm && hr.L > 1 && c.iters > 0) {
    rc = fetch_resnorm(fw.res_acc, resnorm, c.iters, s);
    if (rc) return rc;
    return finish(s, true);
  }
  return finish(s, false);
}

int lstm_adjoint_impl(const mgrit_gru_cfg* cfg, const gru_params* p, const float* x, const float* u0, const float* gi, const float* u,
                      const float* du_seed, const float* dhT, float* du, float* du0, float* dx, const gru_grads* g, float* resnorm,
                      void* ws, size_t ws_bytes, cudaStream_t s) {
  if (!cfg || !p || !x || !u0 || !gi || !u || !du0 || !g || !ws) return MGRIT_INVALID_ARG;
  if (!du_seed && !dhT) return MGRIT_INVALID_ARG;
  if (!p->W_ih || !p->W_hh || !p->b_ih || !p->b_hh || !g->dW_ih || !g->dW_hh || !g->db_ih || !g->db_hh) return MGRIT_INVALID_ARG;
  if (!aligned32(x, u0, gi, u, du_seed, dhT, du, du0, dx, ws, p->W_ih, p->W_hh, p->b_ih, p->b_hh, g->dW_ih, g->dW_hh, g->db_ih, g->db_hh))
    return MGRIT_INVALID_ARG;
  mgrit_gru_cfg c = *cfg;
  Hier hr;
  int rc = lstm_check(&c, &hr);
  if (rc) return rc;
  Ws w{(char*)ws, ws_bytes, 0};
  LstmAdjWs aw;
  plan_lstm_adj(&c, hr, w, &aw);
  if (!w.fits()) return MGRIT_WORKSPACE_TOO_SMALL;
  const size_t bh = (size_t)c.B * c.H, slot = 2 * bh;
  const int T = c.T;
  const bool tf32 = is_tf32(&c), bf = c.operands == MGRIT_OPERANDS_BF16;
  if (tf32) { rc = tf32_prepare_adj(&c, p, &aw.tf, s); if (rc) return rc; }
  if (bf) { rc = lstmbf_prepare_adj(&c, p, &aw.bf, s); if (rc) return rc; }
  for (int l = 0; l < hr.L; ++l) {
    LstmLinArgs a;
    a.M = hr.N[l] * c.B; a.B = c.B; a.H = c.H; a.c0 = u0; a.h0 = u0 + bh; a.c = u; a.h = u + bh; a.ts = (i64)slot;
    a.stride_t = hr.stride_t[l]; a.t0 = hr.rem[l]; a.gi = gi; a.W_hh = p->W_hh; a.b_hh = p->b_hh; a.gamma = hr.gamma[l]; a.cell = c.cell;
    a.a = aw.a[l]; a.p = aw.p[l]; a.ci = aw.ci[l]; a.cf = aw.cf[l]; a.cg = aw.cg[l]; a.co = aw.co[l];
    a.cib = aw.cib[l]; a.cfb = aw.cfb[l]; a.cgb = aw.cgb[l]; a.cob = aw.cob[l];
    if (tf32) { rc = tf32_lstm_linearise(a, &aw.tf, s); if (rc) return rc; }
    else if (bf) { rc = lstmbf_linearise(a, &aw.bf, s); if (rc) return rc; }
    else simt_lstm_linearise(a, s);
  }
  Setup setup(s);
  zero_guess(aw.U[0], c, hr, slot, &setup);
  if (aw.chain_xw) setup.zero(aw.chain_xw, aw.chain_xw_bytes);
  float* Gl[kMaxLevels];
  for (int l = 0; l < hr.L; ++l) Gl[l] = aw.G[l];
  if (!du_seed) Gl[0] = nullptr;
  const float* const last = du_seed ? du_seed + (size_t)(T - 1) * slot : nullptr;
  for (int l = 0; l < hr.L; ++l) {      // cell part, hidden part; dhT: loss on the last hidden state
    if (last) {
      setup.copy(aw.U[l], last, bh);
      setup.copy(aw.U[l] + bh, last + bh, bh, dhT);
    } else {
      setup.zero(aw.U[l], sizeof(float) * bh);
      setup.copy(aw.U[l] + bh, dhT, bh);
    }
  }
  if (du_seed) {
    setup.zero(aw.G[0] + (size_t)T * slot, sizeof(float) * slot);
    if (T > 1) stream_gather_rows(aw.G[0] + slot, (i64)slot, du_seed + (size_t)(T - 2) * slot, -(i64)slot, T - 1, (i64)slot, s);
  }
  LstmAdjCycle cy;
  cy.homog = !du_seed;
  cy.c = &c; cy.hr = hr; cy.s = s; cy.U = aw.U; cy.G = Gl; cy.res_acc = aw.res_acc; cy.BH = slot;
  cy.p = p; cy.w = &aw;
  rc = cy.solve(&setup);
  if (rc) return rc;
  if (du) stream_gather_rows(du, (i64)slot, aw.U[0] + (size_t)(T - 1) * slot, -(i64)slot, T, (i64)slot, s);
  cudaMemcpyAsync(du0, aw.U[0] + (size_t)T * slot, sizeof(float) * slot, cudaMemcpyDeviceToDevice, s);
  // gradient pass over all fine steps at once: dA_t from the step-output sensitivities (read in place, reversed in time)
  const i64 M = (i64)T * c.B;
  const float* lam_c = aw.U[0] + (size_t)(T - 1) * slot;
  if (bf) {
    // bf16 operands: dA is formed as bf16 together with the bias sums, the hidden states are packed straight from u
    rc = lstmbf_gradients(&c, lam_c, lam_c + bh, -(i64)slot, aw.p[0], aw.cib[0], aw.cfb[0], aw.cgb[0], aw.cob[0], x, g,
                          dx, &aw.bf, s);
    if (rc) return rc;
  } else {
    simt_lstm_form_dA(lam_c, lam_c + bh, -(i64)slot, c.B, aw.p[0], aw.ci[0], aw.cf[0], aw.cg[0], aw.co[0], aw.dA, M, c.H, s);
    stream_gather_rows(aw.hk, (i64)bh, u + bh, (i64)slot, T, (i64)bh, s);        // hidden states as their own [T, B, H] array
    if (tf32) {
      rc = tf32_wgrad(aw.dA, (int)M, 4 * c.H, u0 + bh, c.B, aw.hk, c.H, g->dW_hh, &aw.tf, s);
      if (!rc) rc = tf32_wgrad(aw.dA, (int)M, 4 * c.H, nullptr, 0, x, c.I, g->dW_ih, &aw.tf, s);
      if (rc) return rc;
      stream_colsum(aw.dA, M, 4 * c.H, g->db_hh, s);
      cudaMemcpyAsync(g->db_ih, g->db_hh, sizeof(float) * 4 * c.H, cudaMemcpyDeviceToDevice, s);
      if (dx) { rc = tf32_dgrad(aw.dA, (int)M, 4 * c.H, c.I, dx, &aw.tf, s); if (rc) return rc; }
    } else {
      simt_lstm_gradients((int)M, c.B, c.H, c.I, aw.dA, u0 + bh, aw.hk, x, p->W_ih, dx, g, aw.grad_scratch, s);
    }
  }
  if (resnorm && hr.L > 1 && c.iters > 0) {
    rc = fetch_resnorm(aw.res_acc, resnorm, c.iters, s);
    if (rc) return rc;
    return finish(s, true);
  }
  return finish(s, false);
}

}  // namespace
}  // namespace mg

using namespace mg;

extern "C" {

int mgrit_gru_workspace_bytes(const mgrit_gru_cfg* cfg, size_t* fwd_bytes, size_t* adj_bytes) {
  Hier hr;
  int rc = check_cfg(cfg, &hr);
  if (rc) return rc;
  // the serial entry points run the same cfg with levels = 1: take the larger of the two plans
  mgrit_gru_cfg c1 = *cfg; c1.levels = 1; c1.iters = 1; c1.cf = 2;
  Hier h1;
  rc = check_cfg(&c1, &h1);
  if (rc) return rc;
  if (fwd_bytes) {
    Ws w{nullptr, 0, 0}; FwdWs f; plan_fwd(cfg, hr, w, &f);
    Ws w1{nullptr, 0, 0}; FwdWs f1; plan_fwd(&c1, h1, w1, &f1);
    *fwd_bytes = (w.off > w1.off ? w.off : w1.off) + 256;
  }
  if (adj_bytes) {
    Ws w{nullptr, 0, 0}; AdjWs a; plan_adj(cfg, hr, w, &a);
    Ws w1{nullptr, 0, 0}; AdjWs a1; plan_adj(&c1, h1, w1, &a1);
    *adj_bytes = (w.off > w1.off ? w.off : w1.off) + 256;
  }
  return MGRIT_OK;
}

int gru_step_rows(const mgrit_gru_cfg* cfg, const gru_params* p, int32_t n, float gamma, const float* gi_rows, const float* u_prev,
                  float* out, mgrit_stream_t stream) {
  if (!cfg || !p || !p->W_hh || !p->b_hh || !gi_rows || !u_prev || !out || n < 0) return MGRIT_INVALID_ARG;
  if (cfg->B <= 0 || cfg->H <= 0 || cfg->H % 8 != 0 || !(gamma > 0.f)) return MGRIT_INVALID_ARG;
  if (cfg->cell != MGRIT_CELL_CLASSIC && cfg->cell != MGRIT_CELL_IMPLICIT) return MGRIT_INVALID_ARG;
  if (!aligned32(gi_rows, u_prev, out, p->W_hh, p->b_hh)) return MGRIT_INVALID_ARG;
  if ((i64)n * cfg->B > (i64)INT_MAX - 1024) return MGRIT_UNSUPPORTED;
  if (n == 0) return MGRIT_OK;
  cudaStream_t s = (cudaStream_t)stream;
  const i64 BH = (i64)cfg->B * cfg->H;
  FwdStepArgs a{};
  a.M = n * cfg->B; a.B = cfg->B; a.H = cfg->H;
  a.hin = u_prev; a.hin_ks = BH; a.hout = out; a.hout_ks = BH;
  a.gi = gi_rows; a.gi_ks = 3 * BH;
  a.W_hh = p->W_hh; a.b_hh = p->b_hh; a.gamma = gamma; a.cell = cfg->cell; a.mode = 0;
  simt_fwd_step(a, s);
  return finish(s, false);
}

int gru_adjoint_step_rows(const mgrit_gru_cfg* cfg, const gru_params* p, int32_t n, float gamma, const float* gi_rows,
                          const float* h_lin, const float* mu, float* out, void* ws, size_t ws_bytes, mgrit_stream_t stream) {
  if (!cfg || !p || !p->W_hh || !p->b_hh || !gi_rows || !h_lin || !mu || !out || n < 0) return MGRIT_INVALID_ARG;
  if (cfg->B <= 0 || cfg->H <= 0 || cfg->H % 8 != 0 || !(gamma > 0.f)) return MGRIT_INVALID_ARG;
  if (cfg->cell != MGRIT_CELL_CLASSIC && cfg->cell != MGRIT_CELL_IMPLICIT) return MGRIT_INVALID_ARG;
  if (!aligned32(gi_rows, h_lin, mu, out, ws, p->W_hh, p->b_hh)) return MGRIT_INVALID_ARG;
  if ((i64)n * cfg->B > (i64)INT_MAX - 1024) return MGRIT_UNSUPPORTED;
  if (n == 0) return MGRIT_OK;
  const i64 BH = (i64)cfg->B * cfg->H;
  const size_t rows = (size_t)n * BH;
  if (!ws) return MGRIT_INVALID_ARG;
  Ws w{(char*)ws, ws_bytes, 0};
  float* ca = w.take<float>(rows); float* cr = w.take<float>(rows); float* cz = w.take<float>(rows);
  float* cn = w.take<float>(rows); float* cnp = w.take<float>(rows);
  if (!w.fits()) return MGRIT_WORKSPACE_TOO_SMALL;
  cudaStream_t s = (cudaStream_t)stream;
  // coefficients of the n*B steps: row (j, b) leaves the state h_lin[j] with the input projection gi_rows[j]
  // (the level layout of the linearisation with unit stride: step j + 1 leaves fine time 1 + j)
  LinArgs l{};
  l.M = n * cfg->B; l.B = cfg->B; l.H = cfg->H; l.h0 = h_lin; l.h = h_lin; l.stride_t = 1; l.t0 = 1;
  l.gi = gi_rows - 3 * BH;      // its row t + stride - 1 = j + 1 is gi_rows[j]; row 0 is never read
  l.W_hh = p->W_hh; l.b_hh = p->b_hh; l.gamma = gamma; l.cell = cfg->cell;
  l.a = ca; l.cr = cr; l.cz = cz; l.cn = cn; l.cnp = cnp;
  simt_linearise(l, s);
  AdjStepArgs a{};
  a.M = n * cfg->B; a.B = cfg->B; a.H = cfg->H;
  a.lin = mu; a.lin_ks = BH; a.lout = out; a.lout_ks = BH;
  a.a = ca; a.cr = cr; a.cz = cz; a.cn = cn; a.coef_ks = BH;
  a.W_hh = p->W_hh; a.mode = 0;
  simt_adj_step(a, s);
  return finish(s, false);
}

size_t mgrit_gru_gi_bytes(const mgrit_gru_cfg* cfg) {
  Hier hr;
  if (check_cfg(cfg, &hr) != MGRIT_OK) return 0;
  const size_t plain = (size_t)cfg->T * cfg->B * 3 * cfg->H * sizeof(float);
  return (cfg->flags & MGRIT_FLAG_GI_CARRIES_COPIES) ? gi_tail(cfg, nullptr).total_bytes : plain;
}

int gru_input_projection(const mgrit_gru_cfg* cfg, const gru_params* p, const float* x, float* gi, void* ws, size_t ws_bytes,
                         mgrit_stream_t stream) {
  if (!cfg || !p || !x || !gi || !p->W_ih || !p->b_ih) return MGRIT_INVALID_ARG;
  if (!aligned32(x, gi, ws, p->W_ih, p->b_ih)) return MGRIT_INVALID_ARG;
  Hier hr;
  int rc = check_cfg(cfg, &hr);
  if (rc) return rc;
  cudaStream_t s = (cudaStream_t)stream;
  if (cfg->operands == MGRIT_OPERANDS_BF16) {
    if (!ws) return MGRIT_INVALID_ARG;
    Ws w{(char*)ws, ws_bytes, 0};
    FwdWs fw;
    plan_fwd(cfg, hr, w, &fw);
    if (!w.fits()) return MGRIT_WORKSPACE_TOO_SMALL;
    rc = umma_prepare_fwd(cfg, p, x, gi, &fw.um, s);
    if (rc) return rc;
  } else if (is_tf32(cfg)) {
    if (!ws) return MGRIT_INVALID_ARG;
    Ws w{(char*)ws, ws_bytes, 0};
    FwdWs fw;
    plan_fwd(cfg, hr, w, &fw);
    if (!w.fits()) return MGRIT_WORKSPACE_TOO_SMALL;
    rc = tf32_prepare_fwd(cfg, p, x, gi, &fw.tf, s);
    if (rc) return rc;
  } else {
    simt_project(x, p->W_ih, p->b_ih, gi, cfg->T * cfg->B, cfg->I, 3 * cfg->H, s);
  }
  return finish(s, false);
}

int mgrit_gru_forward(const mgrit_gru_cfg* cfg, const gru_params* p, const float* x, const float* h0, float* gi, float* h,
                      float* resnorm, void* ws, size_t ws_bytes, mgrit_stream_t stream) {
  return forward_impl(cfg, false, p, x, h0, gi, h, resnorm, ws, ws_bytes, (cudaStream_t)stream);
}

int gru_serial_forward(const mgrit_gru_cfg* cfg, const gru_params* p, const float* x, const float* h0, float* gi, float* h,
                       void* ws, size_t ws_bytes, mgrit_stream_t stream) {
  return forward_impl(cfg, true, p, x, h0, gi, h, nullptr, ws, ws_bytes, (cudaStream_t)stream);
}

int mgrit_gru_adjoint(const mgrit_gru_cfg* cfg, const gru_params* p, const float* x, const float* h0, const float* gi,
                      const float* h, const float* dh_seed, const float* dhT, float* dh, float* dh0, float* dx,
                      const gru_grads* grads, float* resnorm, void* ws, size_t ws_bytes, mgrit_stream_t stream) {
  return adjoint_impl(cfg, false, p, x, h0, gi, h, dh_seed, dhT, dh, dh0, dx, grads, resnorm, ws, ws_bytes, (cudaStream_t)stream);
}

int gru_serial_backward(const mgrit_gru_cfg* cfg, const gru_params* p, const float* x, const float* h0, const float* gi,
                        const float* h, const float* dh_seed, const float* dhT, float* dh, float* dh0, float* dx,
                        const gru_grads* grads, void* ws, size_t ws_bytes, mgrit_stream_t stream) {
  return adjoint_impl(cfg, true, p, x, h0, gi, h, dh_seed, dhT, dh, dh0, dx, grads, nullptr, ws, ws_bytes, (cudaStream_t)stream);
}

int mgrit_gru_stack_workspace_bytes(const mgrit_gru_cfg* cfg, int32_t n_layers, size_t* fwd_bytes, size_t* adj_bytes) {
  Hier hr;
  int rc = check_cfg(cfg, &hr);
  if (rc) return rc;
  if (n_layers < 1 || n_layers > kMaxStack) return MGRIT_INVALID_ARG;
  if (is_tf32(cfg)) return MGRIT_UNSUPPORTED;
  if (n_layers > 1) { mgrit_gru_cfg c1 = layer_cfg(*cfg, 1); Hier h1; rc = check_cfg(&c1, &h1); if (rc) return rc; }
  if (fwd_bytes) { Ws w{nullptr, 0, 0}; StackFwdWs f; plan_stack_fwd(cfg, n_layers, hr, w, &f); *fwd_bytes = w.off + 256; }
  if (adj_bytes) { Ws w{nullptr, 0, 0}; StackAdjWs a; plan_stack_adj(cfg, n_layers, hr, w, &a); *adj_bytes = w.off + 256; }
  return MGRIT_OK;
}

int mgrit_gru_stack_forward(const mgrit_gru_cfg* cfg, int32_t n_layers, const gru_params* layers, const float* x, const float* h0,
                            float* gi0, float* h, float* resnorm, void* ws, size_t ws_bytes, mgrit_stream_t stream) {
  return stack_forward_impl(cfg, n_layers, layers, x, h0, gi0, h, resnorm, ws, ws_bytes, (cudaStream_t)stream);
}

int mgrit_gru_stack_adjoint(const mgrit_gru_cfg* cfg, int32_t n_layers, const gru_params* layers, const float* x, const float* h0,
                            const float* gi0, const float* h, const float* dh_seed, const float* dhT, float* dh, float* dh0, float* dx,
                            const gru_grads* grads, float* resnorm, void* ws, size_t ws_bytes, mgrit_stream_t stream) {
  return stack_adjoint_impl(cfg, n_layers, layers, x, h0, gi0, h, dh_seed, dhT, dh, dh0, dx, grads, resnorm, ws, ws_bytes,
                            (cudaStream_t)stream);
}

int mgrit_lstm_workspace_bytes(const mgrit_gru_cfg* cfg, size_t* fwd_bytes, size_t* adj_bytes) {
  Hier hr;
  int rc = lstm_check(cfg, &hr);
  if (rc) return rc;
  if (fwd_bytes) { Ws w{nullptr, 0, 0}; LstmFwdWs f; plan_lstm_fwd(cfg, hr, w, &f); *fwd_bytes = w.off + 256; }
  if (adj_bytes) { Ws w{nullptr, 0, 0}; LstmAdjWs a; plan_lstm_adj(cfg, hr, w, &a); *adj_bytes = w.off + 256; }
  return MGRIT_OK;
}

int mgrit_lstm_forward(const mgrit_gru_cfg* cfg, const gru_params* p, const float* x, const float* u0, float* gi, float* u,
                       float* resnorm, void* ws, size_t ws_bytes, mgrit_stream_t stream) {
  return lstm_forward_impl(cfg, p, x, u0, gi, u, resnorm, ws, ws_bytes, (cudaStream_t)stream);
}

int mgrit_lstm_adjoint(const mgrit_gru_cfg* cfg, const gru_params* p, const float* x, const float* u0, const float* gi,
                       const float* u, const float* du_seed, const float* dhT, float* du, float* du0, float* dx,
                       const gru_grads* grads, float* resnorm, void* ws, size_t ws_bytes, mgrit_stream_t stream) {
  return lstm_adjoint_impl(cfg, p, x, u0, gi, u, du_seed, dhT, du, du0, dx, grads, resnorm, ws, ws_bytes, (cudaStream_t)stream);
}

size_t xent_head_workspace_bytes(int32_t B, int32_t C) {
  if (B <= 0 || C <= 0) return 0;
  return ((((size_t)B * C + (size_t)B) * sizeof(float)) + 255) & ~(size_t)255;     // dlogits [B, C] + per-row loss terms [B]
}

int xent_head_fwd_bwd(int32_t B, int32_t H, int32_t C, const float* hT, const float* Wc, const float* bc, const int32_t* labels,
                      float* loss, float* dhT, float* dWc, float* dbc, void* ws, size_t ws_bytes, mgrit_stream_t stream) {
  if (B <= 0 || H <= 0 || C <= 0 || !hT || !Wc || !bc || !labels || !loss || !dhT || !dWc || !dbc || !ws) return MGRIT_INVALID_ARG;
  if (C > 8192) return MGRIT_UNSUPPORTED;
  if (ws_bytes < xent_head_workspace_bytes(B, C)) return MGRIT_WORKSPACE_TOO_SMALL;
  stream_xent(B, H, C, hT, Wc, bc, labels, loss, dhT, dWc, dbc, (float*)ws, (cudaStream_t)stream);
  return finish((cudaStream_t)stream, false);
}

int sgd_update(float* p, const float* g, size_t n, float lr, mgrit_stream_t stream) {
  if (!p || !g) return MGRIT_INVALID_ARG;
  if (n == 0) return MGRIT_OK;
  if (((uintptr_t)p | (uintptr_t)g) & 15) return MGRIT_INVALID_ARG;
  stream_sgd(p, g, n, lr, (cudaStream_t)stream);
  return finish((cudaStream_t)stream, false);
}

int adam_update(float* p, const float* g, float* m, float* v, size_t n, float lr, float beta1, float beta2, float eps, int32_t step,
                mgrit_stream_t stream) {
  if (!p || !g || !m || !v || step < 1 || !(beta1 >= 0.f && beta1 < 1.f) || !(beta2 >= 0.f && beta2 < 1.f) || !(eps > 0.f))
    return MGRIT_INVALID_ARG;
  if (n == 0) return MGRIT_OK;
  stream_adam(p, g, m, v, n, lr, beta1, beta2, eps, step, (cudaStream_t)stream);
  return finish((cudaStream_t)stream, false);
}

int mgrit_gru_last_device_status(void) {
  if (cudaDeviceSynchronize() != cudaSuccess) return MGRIT_CUDA_ERROR;
  return (umma_device_status() != 0 || serial_device_status() != 0 || f32_device_status() != 0) ? MGRIT_DEVICE_TIMEOUT : MGRIT_OK;
}

int mgrit_gru_clear_device_status(void) {
  if (cudaDeviceSynchronize() != cudaSuccess) return MGRIT_CUDA_ERROR;
  return (umma_clear_device_status() == 0 && serial_clear_device_status() == 0 && f32_clear_device_status() == 0) ? MGRIT_OK : MGRIT_CUDA_ERROR;
}

int mgrit_gru_selftest_bounded_wait(int32_t limit_ms, mgrit_stream_t stream) { return umma_selftest_wait(limit_ms, (cudaStream_t)stream); }

unsigned long long mgrit_gru_kernel_launches(void) { return g_kernel_launches.load(std::memory_order_relaxed); }

int mgrit_gru_profile_enable(int on) {
  for (auto& r : g_prof_recs) { g_prof_pool.push_back(r.e0); g_prof_pool.push_back(r.e1); }
  g_prof_recs.clear();
  g_prof_depth = 0;
  g_prof_on = on != 0;
  return MGRIT_OK;
}

int mgrit_gru_profile_records(double* ms, double* flops, int32_t* kernel_class, size_t cap, size_t* n) {
  if (!n) return MGRIT_INVALID_ARG;
  if (cudaDeviceSynchronize() != cudaSuccess) return MGRIT_CUDA_ERROR;
  *n = g_prof_recs.size();
  for (size_t i = 0; i < g_prof_recs.size() && i < cap; ++i) {
    float t = 0.f;
    if (cudaEventElapsedTime(&t, g_prof_recs[i].e0, g_prof_recs[i].e1) != cudaSuccess) return MGRIT_CUDA_ERROR;
    if (ms) ms[i] = t;
    if (flops) flops[i] = g_prof_recs[i].flops;
    if (kernel_class) kernel_class[i] = g_prof_recs[i].kc;
  }
  return MGRIT_OK;
}

int mgrit_gru_profile_read(int kernel_class, double* total_ms, unsigned long long* launches, double* flops) {
  if (kernel_class < 0 || kernel_class >= KC_COUNT) return MGRIT_INVALID_ARG;
  if (cudaDeviceSynchronize() != cudaSuccess) return MGRIT_CUDA_ERROR;
  double ms = 0, fl = 0; unsigned long long n = 0;
  for (auto& r : g_prof_recs) {
    if (r.kc != kernel_class) continue;
    float t = 0.f;
    if (cudaEventElapsedTime(&t, r.e0, r.e1) != cudaSuccess) return MGRIT_CUDA_ERROR;
    ms += t; fl += r.flops; ++n;
  }
  if (total_ms) *total_ms = ms;
  if (launches) *launches = n;
  if (flops) *flops = fl;
  return MGRIT_OK;
}

const char* mgrit_gru_strerror(int code) {
  switch (code) {
    case MGRIT_OK: return "ok";
    case MGRIT_INVALID_ARG: return "invalid argument";
    case MGRIT_NOT_DIVISIBLE: return "T is not divisible by cf^(levels-1)";
    case MGRIT_WORKSPACE_TOO_SMALL: return "workspace too small";
    case MGRIT_UNSUPPORTED: return "shape not supported (operand mode limits, C > 8192 in the loss head, or sizes beyond 32-bit row counts)";
    case MGRIT_CUDA_ERROR: return "CUDA error";
    case MGRIT_DEVICE_TIMEOUT: return "a bounded device-side wait ran out";
    case MGRIT_SCRATCH_LIMIT: return "problem exceeds the built-in scratch of the no-allocation entry point (B*(C+1) <= 65536)";
    default: return "unknown error";
  }
}

}  // extern "C"
