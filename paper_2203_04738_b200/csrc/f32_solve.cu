// The fp32 multigrid solve (forward and adjoint) as ONE persistent launch for widths whose recurrent weights fit the registers
// (above H = 256: and the shared memory) of a cluster of 1 to 8 CTAs (H <= 352).
//
// Launched step by step these solves are chains of hundreds of small dependent products: bound by launch latency, by refetching
// W_hh for every step and by tiles that leave most SMs idle.  Here the weights are loaded once per solve, a row block of up to
// 64 rows keeps its state in shared memory through all steps of an interval (F-relaxation, the step that evaluates v, the coarse
// step of the FAS right-hand side), and only what other rows read -- C-points, coarse right-hand sides, corrections -- crosses
// a grid barrier: two to three of them per level and cycle.
//   forward: CTA c of the cluster owns H/NC hidden units (three gate rows each) and needs the whole state: results are
//     pushed to the peers' shared memory, one cluster barrier per step.
//   adjoint: CTA c owns the SAME gate rows, now as its slice of the reduction: it forms [c_r|c_z|c_n]*mu for its own units,
//     multiplies with its rows of W_hh and sends partial sums to the unit's owner (a third of the bytes that exchanging the
//     formed operand would take); mu itself never leaves its thread.
// The weights live in REGISTERS for the whole solve (at most 96 per thread; what does not fit, for H > 256, in shared memory).
// What a shared-memory operand costs is its delivery -- 32 words a cycle and SM, however they are shared -- so a product with both
// operands in shared memory ran at a sixth of the FFMA rate; with the weights in registers every delivered word of the state
// feeds 3 NU (forward) or 8 (adjoint) multiply-adds.  Lanes split the reduction; their sums change hands by a transposing
// reduction in which every lane ends with the sums of one (row, unit).
//   forward: 8 lanes per NU units (NU = 2 up to H = 128, else 1) and groups of 8 / NU rows: a lane finishes one row and unit.
//   adjoint: KP = 32, 16 or 8 lanes per 8 columns, groups of 4 rows.
// A step's projection, coefficients and additive terms are copied to shared memory (cp.async) during the step before: with the
// weights there is no room in registers to hold them, and requested one row group ahead they arrived late.  What is left is
// latency: a CTA has the registers for 6 to 12 warps, two or three per scheduler, which issue in half of the cycles.
// us a step, forward / adjoint, weights in shared memory -> in registers:
//   H = 32, 2 rows 1.4 / 1.9 -> 0.87 / 1.2; H = 104, 3300 rows 15 / 16 -> 12.3 / 11.5; H = 256, 16 rows 3.3 / 3.2 -> 2.9 / 2.0,
//   500 rows 14.7 / 11.8 -> 11.1 / 8.4 (18 and 24 TFLOP/s); H = 320, 16 rows 4.1 / 4.4 -> 4.4 / 3.6, 700 rows 28 / 23 -> 29 / 32.
// There every width above 256 was padded to 352 columns; padded to the next 32 (adjoint: its own operand words) H = 320 takes
// 4.0 / 3.1 and 25 / 25, H = 288, 700 rows 27 / 32 -> 22 / 25.
#include <stdlib.h>

#include "cell.cuh"
#include "f32_solve.cuh"

namespace mg {
namespace {

// threads of a CTA: twelve warps have 168 registers each (thirteen would round up to sixteen, 128), eight 255
__host__ __device__ constexpr int fwd_most(int KC) { return KC == 4 || KC == 7 || KC == 8 ? 256 : 384; }
constexpr int kMaxRows = 64;
constexpr size_t kSmemMax = 227 * 1024 - 2048;     // dynamic part: the kernels hold under 1 KiB of static shared memory

__device__ int g_f32_status = 0;
int* g_f32_status_ptrs[kMaxDevices] = {nullptr};

__device__ __forceinline__ uint32_t ctarank() { uint32_t r; asm("mov.u32 %0, %%cluster_ctarank;" : "=r"(r)); return r; }
__device__ __forceinline__ uint32_t peer_addr(const void* p, uint32_t cta) {
  uint32_t a = (uint32_t)__cvta_generic_to_shared(p), r;
  asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(cta));
  return r;
}
__device__ __forceinline__ void st_peer4(uint32_t a, float4 v) {
  asm volatile("st.shared::cluster.v4.f32 [%0], {%1,%2,%3,%4};" ::"r"(a), "f"(v.x), "f"(v.y), "f"(v.z), "f"(v.w) : "memory");
}
__device__ __forceinline__ void cluster_sync() {
  asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
template <bool MULTI> __device__ __forceinline__ void block_sync() { if (MULTI) cluster_sync(); else __syncthreads(); }
__device__ __forceinline__ uint64_t now_ns() { uint64_t t; asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t)); return t; }

// All clusters have finished the phase.  The leader CTA arrives and polls (bounded); its verdict reaches the whole cluster, so
// either every CTA of a cluster goes on or every one leaves.  A phase may be a whole serial chain of millions of steps, so what is
// bounded is the time without progress: a working cluster reports every kReport-th step (report()), and with the blocks of a phase
// dealt out evenly no wait sees more than one block's shorter chain unreported.
constexpr int kReport = 256;
__device__ __forceinline__ void report(const F32Args& a, int j, int rank) {
  if ((j & (kReport - 1)) == kReport - 1 && threadIdx.x == 0 && rank == 0)
    asm volatile("red.relaxed.gpu.global.add.u32 [%0], 1;" ::"l"(a.progress) : "memory");
}
template <bool MULTI>
__device__ bool grid_barrier(const F32Args& a, unsigned target, int nc, int* status, int* verdict) {
  block_sync<MULTI>();
  if (ctarank() == 0 && threadIdx.x == 0) {
    asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(a.bar) : "memory");
    int ok = 1;
    unsigned spins = 0, v, seen = 0;
    uint64_t t0 = 0;
    while (true) {
      asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(a.bar) : "memory");
      if (v >= target) break;
      if ((++spins & 127u) == 0) {
        int st;
        unsigned done;
        asm volatile("ld.relaxed.gpu.global.s32 %0, [%1];" : "=r"(st) : "l"(status) : "memory");
        asm volatile("ld.relaxed.gpu.global.u32 %0, [%1];" : "=r"(done) : "l"(a.progress) : "memory");
        if (st != 0) { ok = 0; break; }
        const uint64_t t = now_ns();
        if (t0 == 0 || done != seen) { t0 = t; seen = done; }
        if (t - t0 > a.limit_ns) { atomicCAS(status, 0, 41); ok = 0; break; }
      }
    }
    for (int c = 0; c < nc; ++c) asm volatile("st.shared::cluster.s32 [%0], %1;" ::"r"(peer_addr(verdict, c)), "r"(ok) : "memory");
  }
  block_sync<MULTI>();
  return *(volatile int*)verdict != 0;
}

__device__ __forceinline__ float4 lds4(const float* p) { return *reinterpret_cast<const float4*>(p); }
// two multiply-adds per issue slot: a word pair of the state against a word pair of the weights, summed apart
typedef unsigned long long u64;
struct Two { u64 lo, hi; };
__device__ __forceinline__ Two lds2(const float* p) { const ulonglong2 v = *reinterpret_cast<const ulonglong2*>(p); return Two{v.x, v.y}; }
__device__ __forceinline__ Two pack2(float4 v) {
  Two r;
  asm("mov.b64 %0, {%1,%2};" : "=l"(r.lo) : "f"(v.x), "f"(v.y));
  asm("mov.b64 %0, {%1,%2};" : "=l"(r.hi) : "f"(v.z), "f"(v.w));
  return r;
}
__device__ __forceinline__ void fma2(u64& c, u64 a, u64 b) { asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(c) : "l"(a), "l"(b)); }
__device__ __forceinline__ float2 unpack(u64 v) {
  float2 r;
  asm("mov.b64 {%0,%1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(v));
  return r;
}
// a running sum: of pairs where the registers allow, else of words
template <bool PAIR> struct Sum;
template <> struct Sum<true> {
  u64 c = 0;
  __device__ __forceinline__ void mac(u64 a, u64 b) { fma2(c, a, b); }
  __device__ __forceinline__ float value() const { const float2 v = unpack(c); return v.x + v.y; }
};
template <> struct Sum<false> {
  float c = 0.f;
  __device__ __forceinline__ void mac(u64 a, u64 b) { const float2 x = unpack(a), y = unpack(b); c = fmaf(x.y, y.y, fmaf(x.x, y.x, c)); }
  __device__ __forceinline__ float value() const { return c; }
};
// Halving of N values over the lanes that differ in bits below LANES: afterwards lane k (of LANES) holds the sums of values
// [k N / LANES, (k + 1) N / LANES) in front.
template <int N, int LANES>
__device__ __forceinline__ void fold(float* v, int k) {
  if constexpr (LANES > 1) {
    const bool up = (k & (LANES / 2)) != 0;
#pragma unroll
    for (int i = 0; i < N / 2; ++i) {
      const float keep = up ? v[i + N / 2] : v[i], send = up ? v[i] : v[i + N / 2];
      v[i] = keep + __shfl_xor_sync(0xffffffffu, send, LANES / 2);
    }
    fold<N / 2, LANES / 2>(v, k);
  }
}

__device__ __forceinline__ float4 add4(float4 a, float4 b) { return make_float4(a.x + b.x, a.y + b.y, a.z + b.z, a.w + b.w); }
__device__ __forceinline__ float4 mul4(float4 a, float4 b) { return make_float4(a.x * b.x, a.y * b.y, a.z * b.z, a.w * b.w); }
__device__ __forceinline__ void cp16(float* dst, const float* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_wait() { asm volatile("cp.async.wait_all;" ::: "memory"); }
// does row k of the phase take step j?
__device__ __forceinline__ bool takes(const F32Phase& p, int k, int j) {
  return k >= 0 && (j < (k < p.nfull ? p.n : p.ntail) || (j >= p.n && k < p.nfull));
}

// ---- forward.  KC: chunks of four state words per lane (the row is padded to 32 KC words); lane k reads chunks k, k + 8, ...
// LD, pad: rows that lanes of a warp touch together lie in different banks.  kG: gates whose weights fit the registers; the
// weights of the third one lie in shared memory then (8 rows share what is delivered).
template <int KC> struct FwdShape {
  static constexpr int NU = KC <= 4 ? 2 : 1, RT = 8 / NU, LD = 32 * KC + (NU == 2 ? 8 : 4), kPad = NU == 2 ? 8 : 4, kG = KC <= 8 ? 3 : 2;
  __host__ __device__ static constexpr int op_row(int U) { return 4 * U + kPad; }      // [gate r | z | n | additive term][U]
};
// where a lane parks its sums within a group: [row][4 NU units of the warp]
template <int KC> __device__ __forceinline__ int fwd_slot() {
  constexpr int NU = FwdShape<KC>::NU;
  const int kp = threadIdx.x & 7, n = (threadIdx.x & 31) >> 3;
  return kp / NU * 4 * NU + n * NU + kp % NU;
}
template <int KC> struct FwdWeights {
  Two w[FwdShape<KC>::kG][FwdShape<KC>::NU][KC];
  const float* wn;
};
// units u0 + [NU up, NU up + NU) of W[3H, H]; units at or beyond `lim` and columns beyond H read as zero.  Wn: [unit][32 KC]
template <int KC>
__device__ __forceinline__ void fwd_weights(FwdWeights<KC>& q, const float* W, int H, int u0, int up, int lim, int kp, float* Wn) {
  constexpr int NU = FwdShape<KC>::NU, G = FwdShape<KC>::kG;
#pragma unroll
  for (int g = 0; g < 3; ++g)
#pragma unroll
    for (int n = 0; n < NU; ++n)
#pragma unroll
      for (int i = 0; i < KC; ++i) {
        const int u = up * NU + n, k = 4 * (8 * i + kp);
        const float4 v = u < lim && k < H ? __ldg(reinterpret_cast<const float4*>(W + ((i64)g * H + u0 + u) * H + k)) : make_float4(0.f, 0.f, 0.f, 0.f);
        if (g < G) q.w[g < G ? g : 0][n][i] = pack2(v);
        else *reinterpret_cast<float4*>(Wn + (i64)up * 32 * KC + k) = v;      // (read by the lane that writes it)
      }
  q.wn = Wn + (i64)up * 32 * KC;
}
// pre[g]: this lane's row (kp / NU of the group that starts at S) and unit (kp % NU of its pair)
template <int KC>
__device__ __forceinline__ void fwd_sums(const float* S, const FwdWeights<KC>& q, int kp, float (&pre)[3]) {
  constexpr int NU = FwdShape<KC>::NU, RT = FwdShape<KC>::RT, LD = FwdShape<KC>::LD, G = FwdShape<KC>::kG;
  Sum<true> sum[8 * 3];                   // [row][unit][gate]
#pragma unroll
  for (int i = 0; i < KC; ++i) {
    Two wn;
    if constexpr (G == 2) wn = lds2(q.wn + 4 * (8 * i + kp));
#pragma unroll
    for (int r0 = 0; r0 < RT; r0 += 4) {
      Two v[4];
#pragma unroll
      for (int r = 0; r < 4; ++r) v[r] = lds2(S + (r0 + r) * LD + 4 * (8 * i + kp));
#pragma unroll
      for (int t = 0; t < 2; ++t)
#pragma unroll
        for (int r = 0; r < 4; ++r)
#pragma unroll
          for (int n = 0; n < NU; ++n)
#pragma unroll
            for (int g = 0; g < 3; ++g) {
              const Two& w = g < G ? q.w[g < G ? g : 0][n][i] : wn;
              sum[((r0 + r) * NU + n) * 3 + g].mac(t ? v[r].hi : v[r].lo, t ? w.hi : w.lo);
            }
    }
  }
  float acc[8 * 3];
#pragma unroll
  for (int i = 0; i < 24; ++i) acc[i] = sum[i].value();
  fold<24, 8>(acc, kp);
  pre[0] = acc[0]; pre[1] = acc[1]; pre[2] = acc[2];
}

__device__ __forceinline__ void block_rows(const F32Args& a, const F32Phase& p, int r0, int* rk, int* rb) {
  for (int i = threadIdx.x; i < p.R; i += blockDim.x) {      // (a block may have more rows than threads: H = 8 runs on 32)
    const int m = r0 + i;
    const bool v = m < p.nk * a.B;
    rk[i] = v ? m / a.B : -1;
    rb[i] = v ? m % a.B : 0;
  }
}
__device__ __forceinline__ void add_norm(float norm, double* acc) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) norm += __shfl_xor_sync(0xffffffffu, norm, o);
  if ((threadIdx.x & 31) == 0 && norm != 0.f) atomicAdd(acc, (double)norm);
}

// What the lanes of a warp do with the sums of a row block: with more than one group of rows they go through shared memory and come
// back as four neighbouring units of one row per lane -- the gate arithmetic is one long dependent chain, four of them side by
// side hide each other's latency -- 32 / NU rows at a time; a block of one group (a latency-bound step) keeps lane = (row, unit).
template <int KC>
__device__ __forceinline__ void fwd_park(float* P, int g, const float (&pre)[3]) {      // P: this warp's; g: group within the 32 / NU rows
#pragma unroll
  for (int i = 0; i < 3; ++i) P[i * 128 + g * 32 + fwd_slot<KC>()] = pre[i];
}
struct Pre4 { float4 r, z, n; };
__device__ __forceinline__ Pre4 fwd_parked(const float* P, float4 br, float4 bz, float4 bn) {
  const int l = (threadIdx.x & 31) * 4;
  return Pre4{add4(lds4(P + l), br), add4(lds4(P + 128 + l), bz), add4(lds4(P + 256 + l), bn)};
}
__device__ __forceinline__ float4 cell_forward4(float4 gr, float4 gz, float4 gn, const Pre4& q, float4 h, float gamma, int cell) {
  return make_float4(cell_forward<2>(gr.x, gz.x, gn.x, q.r.x, q.z.x, q.n.x, h.x, gamma, cell), cell_forward<2>(gr.y, gz.y, gn.y, q.r.y, q.z.y, q.n.y, h.y, gamma, cell),
                     cell_forward<2>(gr.z, gz.z, gn.z, q.r.z, q.z.z, q.n.z, h.z, gamma, cell), cell_forward<2>(gr.w, gz.w, gn.w, q.r.w, q.z.w, q.n.w, h.w, gamma, cell));
}

// shared: S[2][R][LD] (the whole state of the rows, this step's and the next), O[2][R][op_row] (operands of this step and the next),
// B[3][U] (biases), P[warps][384].  A warp finishes 4 NU neighbouring units of every row; it alone fetches their operands and
// passes their results on.
template <bool MULTI, int KC>
__global__ void __launch_bounds__(fwd_most(KC), 1) f32_fwd_kernel(const __grid_constant__ F32Args a, int NC, int U, int rmax, int* status) {
  constexpr int NU = FwdShape<KC>::NU, RT = FwdShape<KC>::RT, LD = FwdShape<KC>::LD, PR = 32 / NU;
  extern __shared__ __align__(16) float fsm[];
  __shared__ int rk[kMaxRows], rb[kMaxRows], verdict;
  const int H = a.H, rank = MULTI ? (int)ctarank() : 0;
  const int cid = blockIdx.x / NC, ncl = gridDim.x / NC;
  const int u0 = rank * U, Un = max(0, min(U, H - u0)), OR = FwdShape<KC>::op_row(U), sstride = rmax * LD, ostride = rmax * OR;
  float *S0 = fsm, *O0 = fsm + 2 * sstride, *Bs = O0 + 2 * ostride, *P = Bs + 3 * U + (threadIdx.x >> 5) * 384;
  for (int e = threadIdx.x; e < 2 * sstride; e += blockDim.x) S0[e] = 0.f;      // (the columns beyond H stay zero)
  for (int e = threadIdx.x; e < 3 * U; e += blockDim.x) Bs[e] = e % U < Un ? a.b_hh[e / U * H + u0 + e % U] : 0.f;
  const int kp = threadIdx.x & 7, up = threadIdx.x >> 3, u = up * NU + kp % NU, rl = kp / NU, c = u0 + u;
  FwdWeights<KC> q;
  fwd_weights<KC>(q, a.W, H, u0, up, Un, kp, Bs + 3 * U + (blockDim.x >> 5) * 384);
  // quadruple of units and row (modulo PR) of this lane when the warp works on quadruples
  const int qu = (threadIdx.x >> 5) * 4 * NU + (threadIdx.x % NU) * 4, qr = (threadIdx.x & 31) / NU;
  const bool qon = qu < Un;
  unsigned target = 0;
  for (int ip = 0; ip < a.nph; ++ip) {
    const F32Phase& p = a.ph[ip];
    const int M = p.nk * a.B, nblk = (M + p.R - 1) / p.R, R = p.R, steps = p.n + (p.last_kind != kLastNone ? 1 : 0);
    const bool coarse = p.last_kind == kLastCoarse, one = R == RT;
    float norm = 0.f;
    for (int blk = cid; blk < nblk; blk += ncl) {
      __syncthreads();
      block_rows(a, p, blk * R, rk, rb);
      __syncthreads();
      auto fetch = [&](int j, bool cs) {      // the operands of step j (cs: of the coarse step, with the C-point as the additive term)
        float* O = O0 + (j & 1) * ostride;
        if (qon)
          for (int r = qr; r < R; r += PR) {
            const int k = rk[r];
            if (!takes(p, k, cs ? p.n : j)) continue;
            const float* gp = a.gi + (cs ? p.op2 + k * p.op2_ks : p.op + k * p.op_ks + j * p.op_ss) + (i64)rb[r] * 3 * H + u0 + qu;
            float* o = O + r * OR + qu;
            cp16(o, gp); cp16(o + U, gp + H); cp16(o + 2 * U, gp + 2 * H);
            const i64 bo = (i64)rb[r] * H + u0 + qu;
            if (cs) cp16(o + 3 * U, p.uc + k * p.uc_ks + bo);
            else if (p.g) cp16(o + 3 * U, p.g + k * p.g_ks + j * p.g_ss + bo);
          }
      };
      auto load = [&](float* S, const float* src, i64 ks, float* copy, i64 cks) {
        for (int e = threadIdx.x; e < R * (H / 4); e += blockDim.x) {
          const int r = e / (H / 4), i = e % (H / 4), k = rk[r];
          float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
          if (k >= 0) {
            v = __ldcg(reinterpret_cast<const float4*>(src + k * ks + (i64)rb[r] * H) + i);
            if (copy && 4 * i >= u0 && 4 * i < u0 + Un) *(reinterpret_cast<float4*>(copy + k * cks + (i64)rb[r] * H) + i) = v;
          }
          *reinterpret_cast<float4*>(S + r * LD + 4 * i) = v;
        }
      };
      // sums of PR rows from c0 on, parked
      auto sums = [&](const float* S, int c0) {
        float pre[3];
        for (int g = 0; g < PR / RT && c0 + g * RT < R; ++g) {
          fwd_sums<KC>(S + (c0 + g * RT) * LD, q, kp, pre);
          fwd_park<KC>(P, g, pre);
        }
        __syncwarp();
      };
      if (steps > 0) fetch(0, false);
      load(S0, p.src, p.src_ks, p.copy, p.copy_ks);
      block_sync<MULTI>();       // the peers are done with the previous block before anything is pushed into S[1]
      for (int j = 0; j < steps; ++j) {
        const float *S = S0 + (j & 1) * sstride, *O = O0 + (j & 1) * ostride;
        float* N = S0 + (~j & 1) * sstride;
        // (the result of a step that only feeds the coarse right-hand side, vstep, stays in N)
        const bool closing = j + 1 == steps, vstep = j == p.n && coarse;
        if (one) {
          float pre[3];
          fwd_sums<KC>(S, q, kp, pre);
          cp_wait();
          __syncwarp();
          if (!closing || coarse) fetch(j + 1, closing);
          if (u < Un) {
            const float* o = O + rl * OR + u;
            float v = cell_forward<2>(o[0], o[U], o[2 * U], pre[0] + Bs[u], pre[1] + Bs[U + u], pre[2] + Bs[2 * U + u], S[rl * LD + c], p.gamma, a.cell);
            if (p.g) v += o[3 * U];
            float* n = N + rl * LD + c;
            *n = v;
            if (!vstep) {
              const int k = rk[rl];
              if (takes(p, k, j)) {
                const i64 bo = (i64)rb[rl] * H + c;
                *(j == p.n ? p.last + k * p.last_ks + bo : p.out + k * p.out_ks + j * p.out_ss + bo) = v;
              }
              if (MULTI && !closing)
                for (int d = 1; d < NC; ++d) {
                  const int t = rank + d;
                  asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(peer_addr(n, t < NC ? t : t - NC)), "f"(v) : "memory");
                }
            }
          }
        } else {
          for (int c0 = 0; c0 < R; c0 += PR) {
            sums(S, c0);
            if (c0 == 0) {
              cp_wait();                       // (a lane reads what it copied itself)
              if (!closing || coarse) fetch(j + 1, closing);
            }
            const int row = c0 + qr;
            if (qon && row < R) {
              const float* o = O + row * OR + qu;
              const Pre4 pre = fwd_parked(P, lds4(Bs + qu), lds4(Bs + U + qu), lds4(Bs + 2 * U + qu));
              float4 v = cell_forward4(lds4(o), lds4(o + U), lds4(o + 2 * U), pre, lds4(S + row * LD + u0 + qu), p.gamma, a.cell);
              if (p.g) v = add4(v, lds4(o + 3 * U));
              float* n = N + row * LD + u0 + qu;
              *reinterpret_cast<float4*>(n) = v;
              if (!vstep) {
                const int k = rk[row];
                if (takes(p, k, j)) {
                  const i64 bo = (i64)rb[row] * H + u0 + qu;
                  *reinterpret_cast<float4*>(j == p.n ? p.last + k * p.last_ks + bo : p.out + k * p.out_ks + j * p.out_ss + bo) = v;
                }
                if (MULTI && !closing)
                  for (int d = 1; d < NC; ++d) { const int t = rank + d; st_peer4(peer_addr(n, t < NC ? t : t - NC), v); }
              }
            }
            __syncwarp();
          }
        }
        if (!closing) block_sync<MULTI>();
        report(a, j, rank);
      }
      if (coarse) {
        float *S = S0 + ((steps - 1) & 1) * sstride, *N = S0 + (steps & 1) * sstride;
        const float* O = O0 + (steps & 1) * ostride;
        __syncthreads();
        load(S, p.src2, p.src2_ks, nullptr, 0);
        cp_wait();
        __syncthreads();
        for (int c0 = 0; c0 < R; c0 += PR) {
          sums(S, c0);
          const int row = c0 + qr, k = row < R ? rk[row] : -1;
          if (qon && takes(p, k, p.n)) {
            const float* o = O + row * OR + qu;
            const Pre4 pre = fwd_parked(P, lds4(Bs + qu), lds4(Bs + U + qu), lds4(Bs + 2 * U + qu));
            const float4 phi = cell_forward4(lds4(o), lds4(o + U), lds4(o + 2 * U), pre, lds4(S + row * LD + u0 + qu), p.gamma2, a.cell);
            const float4 v = lds4(N + row * LD + u0 + qu), uc = lds4(o + 3 * U);
            const float d0 = uc.x - v.x, d1 = uc.y - v.y, d2 = uc.z - v.z, d3 = uc.w - v.w;
            norm += d0 * d0 + d1 * d1 + d2 * d2 + d3 * d3;
            const i64 bo = (i64)rb[row] * H + u0 + qu;
            if (p.ucd) *reinterpret_cast<float4*>(p.ucd + k * p.ucd_ks + bo) = uc;
            *reinterpret_cast<float4*>(p.last + k * p.last_ks + bo) = make_float4(v.x - phi.x, v.y - phi.y, v.z - phi.z, v.w - phi.w);
          }
          __syncwarp();
        }
      }
    }
    if (p.acc) add_norm(norm, p.acc);
    if (ip + 1 < a.nph) {
      target += ncl;
      if (!grid_barrier<MULTI>(a, target, NC, status, &verdict)) return;
    }
  }
}

// ---- adjoint
// shared: Ad[R][lda] (the formed operand [gate][own units], padded with zeros to 4 KP KC words), Pb[2][NC][R][U] (partial sums for
// this CTA's units by producer) and, by row and own unit, each quadruple touched by one thread alone: mu, a second mu (the coarse
// step's start, then v), c_r, c_z, c_n, and of two steps a and the source.
// T: the most threads of the CTA.  kW: chunks whose weights fit the registers; those of the others lie in shared memory
template <int KP, int KC, int T> struct AdjShape {
  static constexpr int kRow = 4 * KP * KC, kW = KC < 3 ? KC : 3;
  static constexpr bool kPair = T == 256 || KC < 3;
};
constexpr int kAdjFields = 9;

// w[c][i]: W_hh rows of this lane's operand words (k' = 4 (KP i + kp) + 0..3, gate k' / U) at column 8 cg + c
template <int KP, int KC, int T>
__device__ __forceinline__ void adj_weights(Two (&w)[8][AdjShape<KP, KC, T>::kW], float* Wx, const float* W, int H, int U, int u0, int Un, int cg, int kp) {
  constexpr int KW = AdjShape<KP, KC, T>::kW;
#pragma unroll
  for (int i = 0; i < KC; ++i) {
    float v[4][8];
#pragma unroll
    for (int t = 0; t < 4; ++t) {
      const int k = 4 * (KP * i + kp) + t, g = k / U, j = k - g * U;
      const bool ok = g < 3 && j < Un && 8 * cg < H;
      const float4* src = reinterpret_cast<const float4*>(W + ((i64)g * H + u0 + j) * H + 8 * cg);
      const float4 lo = ok ? __ldg(src) : make_float4(0.f, 0.f, 0.f, 0.f), hi = ok ? __ldg(src + 1) : make_float4(0.f, 0.f, 0.f, 0.f);
      v[t][0] = lo.x; v[t][1] = lo.y; v[t][2] = lo.z; v[t][3] = lo.w; v[t][4] = hi.x; v[t][5] = hi.y; v[t][6] = hi.z; v[t][7] = hi.w;
    }
#pragma unroll
    for (int c = 0; c < 8; ++c) {
      const float4 x = make_float4(v[0][c], v[1][c], v[2][c], v[3][c]);
      if (i < KW) w[c][i < KW ? i : 0] = pack2(x);
      else *reinterpret_cast<float4*>(Wx + 4 * (((i - KW) * 8 + c) * blockDim.x + threadIdx.x)) = x;           // (read by the lane that writes it)
    }
  }
}
template <int KP, int KC, int T, bool MULTI>
__device__ __forceinline__ void adj_product(const Two (&w)[8][AdjShape<KP, KC, T>::kW], const float* Wx, const float* Ad, float* Pb, int lda, int R, int U,
                                            int H, int cg, int kp, int rank) {
  constexpr int NV = 32 / KP, KW = AdjShape<KP, KC, T>::kW;      // NV values a lane ends with: row and columns [kp NV, kp NV + NV) of the 4 x 8 block
  const int n = 8 * cg + kp * NV % 8, d = n / U;
  float* q = Pb + ((i64)rank * R + kp * NV / 8) * U + (n - d * U);
  const uint32_t far = MULTI && n < H ? peer_addr(q, d) : 0;
  for (int r0 = 0; r0 < R; r0 += 4) {
    Sum<AdjShape<KP, KC, T>::kPair> sum[32];
    auto chunk = [&](int i, auto weight) {
      Two v[4];
#pragma unroll
      for (int r = 0; r < 4; ++r) v[r] = lds2(Ad + (r0 + r) * lda + 4 * (KP * i + kp));
#pragma unroll
      for (int c = 0; c < 8; ++c) {
        const Two x = weight(c);
#pragma unroll
        for (int r = 0; r < 4; ++r) sum[r * 8 + c].mac(v[r].lo, x.lo);
#pragma unroll
        for (int r = 0; r < 4; ++r) sum[r * 8 + c].mac(v[r].hi, x.hi);
      }
    };
#pragma unroll
    for (int i = 0; i < KW; ++i) chunk(i, [&](int c) { return w[c][i]; });
    if constexpr (KC > KW)
      for (int i = KW; i < KC; ++i) chunk(i, [&](int c) { return lds2(Wx + 4 * (((i - KW) * 8 + c) * blockDim.x + threadIdx.x)); });
    float acc[32];
#pragma unroll
    for (int i = 0; i < 32; ++i) acc[i] = sum[i].value();
    fold<32, KP>(acc, kp);
    if (n < H) {
      if (MULTI) {
        const uint32_t t = far + r0 * U * 4;
        if constexpr (NV == 4) st_peer4(t, make_float4(acc[0], acc[1], acc[2], acc[3]));
        else if constexpr (NV == 2) asm volatile("st.shared::cluster.v2.f32 [%0], {%1,%2};" ::"r"(t), "f"(acc[0]), "f"(acc[1]) : "memory");
        else asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(t), "f"(acc[0]) : "memory");
      } else {
#pragma unroll
        for (int i = 0; i < NV; ++i) q[r0 * U + i] = acc[i];
      }
    }
  }
}

template <bool MULTI, int KP, int KC, int T>
__global__ void __launch_bounds__(T, 1) f32_adj_kernel(const __grid_constant__ F32Args a, int NC, int U, int rmax, int* status) {
  extern __shared__ __align__(16) float fsm[];
  __shared__ int rk[kMaxRows], rb[kMaxRows], verdict;
  const int H = a.H, rank = MULTI ? (int)ctarank() : 0, u0 = rank * U, Un = max(0, min(U, H - u0)), U4 = Un / 4;
  const int lda = max(3 * U, AdjShape<KP, KC, T>::kRow), cg = threadIdx.x / KP, kp = threadIdx.x % KP;
  const int cid = blockIdx.x / NC, ncl = gridDim.x / NC;
  const int pstride = NC * rmax * U, fstride = rmax * U;
  float *Ad = fsm, *Pbuf = Ad + rmax * lda, *F = Pbuf + 2 * pstride;
  float *Mu = F, *Mv = F + fstride, *Cr = F + 2 * fstride, *Cz = F + 3 * fstride, *Cn = F + 4 * fstride, *Aa = F + 5 * fstride, *Gs = F + 7 * fstride;
  float* Wx = F + kAdjFields * fstride;
  for (int e = threadIdx.x; e < rmax * lda; e += blockDim.x) Ad[e] = 0.f;
  Two w[8][AdjShape<KP, KC, T>::kW];
  adj_weights<KP, KC, T>(w, Wx, a.W, H, U, u0, Un, cg, kp);
  block_sync<MULTI>();       // (peers write to each other's shared memory from the first product on)
  // quadruples of this thread: first row and unit, and the way to the next one
  const int row0 = threadIdx.x / U4, col0 = (threadIdx.x - row0 * U4) * 4, drow = blockDim.x / U4, dcol = (blockDim.x - drow * U4) * 4;
  unsigned target = 0;
  int par = 0;
  for (int ip = 0; ip < a.nph; ++ip) {
    const F32Phase& p = a.ph[ip];
    const int M = p.nk * a.B, nblk = (M + p.R - 1) / p.R, R = p.R, steps = p.n + (p.last_kind != kLastNone ? 1 : 0);
    const bool coarse = p.last_kind == kLastCoarse;
    float norm = 0.f;
    for (int blk = cid; blk < nblk; blk += ncl) {
      __syncthreads();
      block_rows(a, p, blk * R, rk, rb);
      __syncthreads();
      auto quads = [&](auto f) {
        for (int row = row0, u = col0; row < R;) {
          f(row, u, row * U + u);
          row += drow; u += dcol;
          if (u >= Un) { u -= Un; ++row; }
        }
      };
      // coefficients and source of step j (cs: of the coarse step, with the C-point as the source and its start to Mv)
      auto fetch = [&](int j, bool cs) {
        float *A = Aa + (j & 1) * fstride, *G = Gs + (j & 1) * fstride;
        quads([&](int row, int u, int o) {
          const int k = rk[row];
          if (!takes(p, k, cs ? p.n : j)) return;
          const i64 bo = (i64)rb[row] * H + u0 + u, x = (cs ? p.op2 + k * p.op2_ks : p.op + k * p.op_ks + j * p.op_ss) + bo;
          const float* const* cf = a.coef[p.level + (cs ? 1 : 0)];
          cp16(A + o, cf[0] + x); cp16(Cr + o, cf[1] + x); cp16(Cz + o, cf[2] + x); cp16(Cn + o, cf[3] + x);
          if (cs) { cp16(G + o, p.uc + k * p.uc_ks + bo); cp16(Mv + o, p.src2 + k * p.src2_ks + bo); }
          else if (p.g) cp16(G + o, p.g + k * p.g_ks + j * p.g_ss + bo);
        });
      };
      auto form = [&](int row, int u, int o, float4 m) {
        float* d = Ad + row * lda + u;
        *reinterpret_cast<float4*>(d) = mul4(lds4(Cr + o), m);
        *reinterpret_cast<float4*>(d + U) = mul4(lds4(Cz + o), m);
        *reinterpret_cast<float4*>(d + 2 * U) = mul4(lds4(Cn + o), m);
      };
      auto product = [&]() {
        adj_product<KP, KC, T, MULTI>(w, Wx, Ad, Pbuf + par * pstride, lda, R, U, H, cg, kp, rank);
        block_sync<MULTI>();
      };
      auto result = [&](int o, int j) {                   // a*mu + sum of the partial products
        const float* Pb = Pbuf + par * pstride + o;
        float4 t = lds4(Pb);
        for (int c = 1; c < NC; ++c) t = add4(t, lds4(Pb + c * R * U));
        const float4 A = lds4(Aa + (j & 1) * fstride + o), m = lds4(Mu + o);
        return make_float4(fmaf(A.x, m.x, t.x), fmaf(A.y, m.y, t.y), fmaf(A.z, m.z, t.z), fmaf(A.w, m.w, t.w));
      };
      if (steps > 0) fetch(0, false);
      quads([&](int row, int u, int o) {
        const int k = rk[row];
        float4 m = make_float4(0.f, 0.f, 0.f, 0.f);
        if (k >= 0) {
          const i64 bo = (i64)rb[row] * H + u0 + u;
          m = __ldcg(reinterpret_cast<const float4*>(p.src + k * p.src_ks + bo));
          if (p.copy) *reinterpret_cast<float4*>(p.copy + k * p.copy_ks + bo) = m;
        }
        *reinterpret_cast<float4*>(Mu + o) = m;
      });
      cp_wait();
      if (steps > 0) quads([&](int row, int u, int o) { form(row, u, o, lds4(Mu + o)); });
      for (int j = 0; j < steps; ++j) {
        const bool closing = j + 1 == steps, vstep = j == p.n && coarse;
        __syncthreads();
        if (!closing || coarse) fetch(j + 1, closing);
        product();
        cp_wait();
        quads([&](int row, int u, int o) {
          float4 m = result(o, j);
          if (p.g) m = add4(m, lds4(Gs + (j & 1) * fstride + o));
          if (vstep) {
            const float4 t = lds4(Mv + o);
            *reinterpret_cast<float4*>(Mv + o) = m;
            m = t;
          } else {
            const int k = rk[row];
            if (takes(p, k, j)) {
              const i64 bo = (i64)rb[row] * H + u0 + u;
              *reinterpret_cast<float4*>(j == p.n ? p.last + k * p.last_ks + bo : p.out + k * p.out_ks + j * p.out_ss + bo) = m;
            }
          }
          *reinterpret_cast<float4*>(Mu + o) = m;
          if (!closing || coarse) form(row, u, o, m);
        });
        par ^= 1;
        report(a, j, rank);
      }
      if (coarse) {
        __syncthreads();
        product();
        quads([&](int row, int u, int o) {
          const int k = rk[row];
          if (!takes(p, k, p.n)) return;
          const float4 r = result(o, steps), uc = lds4(Gs + (steps & 1) * fstride + o), v = lds4(Mv + o);
          const i64 bo = (i64)rb[row] * H + u0 + u;
          const float d0 = uc.x - v.x, d1 = uc.y - v.y, d2 = uc.z - v.z, d3 = uc.w - v.w;
          norm += d0 * d0 + d1 * d1 + d2 * d2 + d3 * d3;
          if (p.ucd) *reinterpret_cast<float4*>(p.ucd + k * p.ucd_ks + bo) = uc;
          *reinterpret_cast<float4*>(p.last + k * p.last_ks + bo) = make_float4(v.x - r.x, v.y - r.y, v.z - r.z, v.w - r.w);
        });
        par ^= 1;
      }
    }
    if (p.acc) add_norm(norm, p.acc);
    if (ip + 1 < a.nph) {
      target += ncl;
      if (!grid_barrier<MULTI>(a, target, NC, status, &verdict)) return;
    }
  }
  block_sync<MULTI>();      // no CTA leaves while a peer may still write its partial sums
}

// ---- linearisation: the forward product of every level's rows with the transposed-Jacobian epilogue; no exchange
struct LinSet { LinArgs l[kF32Levels]; int n, blk0[kF32Levels + 1]; };
// The next block's rows are copied to shared memory while the current one is computed; S and O as in the forward kernel.
template <int KC>
__global__ void __launch_bounds__(fwd_most(KC), 1) f32_lin_kernel(const __grid_constant__ LinSet ls, int U, int R) {
  constexpr int NU = FwdShape<KC>::NU, RT = FwdShape<KC>::RT, LD = FwdShape<KC>::LD, PR = 32 / NU;
  extern __shared__ __align__(16) float fsm[];
  const int H = ls.l[0].H, B = ls.l[0].B, u0 = blockIdx.x * U, Un = min(U, H - u0), OR = FwdShape<KC>::op_row(U);
  const int kp = threadIdx.x & 7, up = threadIdx.x >> 3, sstride = R * LD, ostride = R * OR;
  float *S0 = fsm, *O0 = fsm + 2 * sstride, *Bs = O0 + 2 * ostride, *P = Bs + 3 * U + (threadIdx.x >> 5) * 384;
  for (int e = threadIdx.x; e < 2 * sstride; e += blockDim.x) S0[e] = 0.f;
  for (int e = threadIdx.x; e < 3 * U; e += blockDim.x) Bs[e] = e % U < Un ? ls.l[0].b_hh[e / U * H + u0 + e % U] : 0.f;
  FwdWeights<KC> q;
  fwd_weights<KC>(q, ls.l[0].W_hh, H, u0, up, Un, kp, Bs + 3 * U + (blockDim.x >> 5) * 384);
  const int qu = (threadIdx.x >> 5) * 4 * NU + (threadIdx.x % NU) * 4, qr = (threadIdx.x & 31) / NU;
  auto level = [&](int blk) { int lv = 0; while (blk >= ls.blk0[lv + 1]) ++lv; return lv; };
  auto fetch = [&](int blk, int buf) {
    const int lv = level(blk);
    const LinArgs& a = ls.l[lv];
    const int r0 = (blk - ls.blk0[lv]) * R;
    float *S = S0 + buf * sstride, *O = O0 + buf * ostride;
    for (int e = threadIdx.x; e < R * (H / 4); e += blockDim.x) {
      const int r = e / (H / 4), k = e % (H / 4), m = r0 + r;
      if (m >= a.M) break;
      const int j1 = m / B, b = m - j1 * B;
      const i64 t = a.t0 + (i64)j1 * a.stride_t;
      cp16(S + r * LD + 4 * k, (t == 0 ? a.h0 + (i64)b * H : a.h + ((t - 1) * B + b) * H) + 4 * k);
    }
    if (qu < Un)
      for (int r = qr; r < R && r0 + r < a.M; r += 32 / NU) {
        const int m = r0 + r, j1 = m / B, b = m - j1 * B;
        const i64 t = a.t0 + (i64)j1 * a.stride_t;
        const float* gp = a.gi + ((t + a.stride_t - 1) * B + b) * 3 * H + u0 + qu;
        float* o = O + r * OR + qu;
        cp16(o, gp); cp16(o + U, gp + H); cp16(o + 2 * U, gp + 2 * H);
      }
  };
  __syncthreads();
  int buf = 0;
  if (blockIdx.y < ls.blk0[ls.n]) fetch(blockIdx.y, 0);
  for (int blk = blockIdx.y; blk < ls.blk0[ls.n]; blk += gridDim.y, buf ^= 1) {
    cp_wait();
    __syncthreads();
    if (blk + gridDim.y < ls.blk0[ls.n]) fetch(blk + gridDim.y, buf ^ 1);
    const int lv = level(blk);
    const LinArgs& a = ls.l[lv];
    const int r0 = (blk - ls.blk0[lv]) * R;
    const float *S = S0 + buf * sstride, *O = O0 + buf * ostride + qu;
    for (int c0 = 0; c0 < R; c0 += PR) {
      float pre[3];
      for (int g = 0; g < PR / RT && c0 + g * RT < R; ++g) {
        fwd_sums<KC>(S + (c0 + g * RT) * LD, q, kp, pre);
        fwd_park<KC>(P, g, pre);
      }
      __syncwarp();
      const int row = c0 + qr;
      if (qu < Un && row < R && r0 + row < a.M) {
        const float* g = O + row * OR;
        const Pre4 t = fwd_parked(P, lds4(Bs + qu), lds4(Bs + U + qu), lds4(Bs + 2 * U + qu));
        const float4 gr = lds4(g), gz = lds4(g + U), gn = lds4(g + 2 * U), h = lds4(S + row * LD + u0 + qu);
        const CellLin x = cell_linearise<2>(gr.x, gz.x, gn.x, t.r.x, t.z.x, t.n.x, h.x, a.gamma, a.cell);
        const CellLin y = cell_linearise<2>(gr.y, gz.y, gn.y, t.r.y, t.z.y, t.n.y, h.y, a.gamma, a.cell);
        const CellLin z = cell_linearise<2>(gr.z, gz.z, gn.z, t.r.z, t.z.z, t.n.z, h.z, a.gamma, a.cell);
        const CellLin w = cell_linearise<2>(gr.w, gz.w, gn.w, t.r.w, t.z.w, t.n.w, h.w, a.gamma, a.cell);
        const i64 o = (i64)(r0 + row) * H + u0 + qu;
        *reinterpret_cast<float4*>(a.a + o) = make_float4(x.a, y.a, z.a, w.a);
        *reinterpret_cast<float4*>(a.cr + o) = make_float4(x.cr, y.cr, z.cr, w.cr);
        *reinterpret_cast<float4*>(a.cz + o) = make_float4(x.cz, y.cz, z.cz, w.cz);
        *reinterpret_cast<float4*>(a.cn + o) = make_float4(x.cn, y.cn, z.cn, w.cn);
        if (a.cnp) *reinterpret_cast<float4*>(a.cnp + o) = make_float4(x.cnp, y.cnp, z.cnp, w.cnp);
      }
      __syncwarp();
    }
  }
}

// How long a barrier waits without progress: 2 s, or MGRIT_GRU_TEST_F32_WAIT_US microseconds from the environment.
unsigned long long wait_limit_ns() {
  static unsigned long long v = 0;
  if (v == 0) {
    const char* e = getenv("MGRIT_GRU_TEST_F32_WAIT_US");
    const long long us = e ? atoll(e) : 0;
    v = us > 0 && us <= 2000000 ? 1000ull * (unsigned long long)us : 2000000000ull;
  }
  return v;
}

// MGRIT_GRU_F32_SOLVE=0 in the environment answers as where the cooperative cluster launch is refused: the callers then advance step
// by step, as at widths that do not fit (the linearisation, which is no cooperative launch, goes with it).
bool solve_enabled() {
  static int v = -1;
  if (v < 0) { const char* e = getenv("MGRIT_GRU_F32_SOLVE"); v = (e && e[0] == '0') ? 0 : 1; }
  return v == 1;
}

int* status_ptr() {
  const int dev = current_device_slot();
  if (dev < 0) return nullptr;
  if (!g_f32_status_ptrs[dev]) {
    int* p = nullptr;
    if (cudaGetSymbolAddress((void**)&p, g_f32_status) != cudaSuccess) { cudaGetLastError(); return nullptr; }
    g_f32_status_ptrs[dev] = p;
  }
  return g_f32_status_ptrs[dev];
}

// CTAs per cluster, units per CTA, threads, and what a row of a block takes of shared memory (besides a fixed part)
struct Shape { int NC, U, KC, fwd_threads, adj_kp, adj_kc, adj_threads; size_t fwd_row, fwd_fix, adj_row, adj_fix; };
bool pick_shape(int H, Shape* q) {
  if (H % 8 != 0 || H > 352) return false;
  q->KC = (H + 31) / 32;
  const int nc = H <= 96 ? 1 : H <= 128 ? 2 : H <= 192 ? 4 : 8;      // at most 96 (NU = 2) or 48 (NU = 1) units per CTA: 384 threads
  q->U = ((H + nc - 1) / nc + 3) / 4 * 4;
  q->NC = (H + q->U - 1) / q->U;
  const int nu = q->KC <= 4 ? 2 : 1;
  q->fwd_threads = ((q->U + nu - 1) / nu * 8 + 31) / 32 * 32;
  q->adj_kp = H <= 96 ? 32 : H <= 192 ? 16 : 8;
  q->adj_kc = (3 * q->U / 4 + q->adj_kp - 1) / q->adj_kp;
  q->adj_threads = (H / 8 * q->adj_kp + 31) / 32 * 32;
  const int lda = 3 * q->U > 4 * q->adj_kp * q->adj_kc ? 3 * q->U : 4 * q->adj_kp * q->adj_kc, pad = nu == 2 ? 8 : 4;
  q->fwd_row = (size_t)2 * (32 * q->KC + pad + 4 * q->U + pad) * 4;
  q->fwd_fix = (size_t)(3 * q->U + q->fwd_threads / 32 * 384 + (q->KC > 8 ? q->fwd_threads / 8 * 32 * q->KC : 0)) * 4;
  q->adj_row = ((size_t)lda + (2 * q->NC + kAdjFields) * q->U) * 4;
  q->adj_fix = q->adj_kc > 3 ? (size_t)(q->adj_kc - 3) * 8 * q->adj_threads * 16 : 0;
  return true;
}
// Rows per block of a phase: the fewest waves of blocks, weighed against the time of a step (instructions of its row groups plus
// about 1500 cycles of exchange, latency and epilogue).
void tune(bool adj, F32Phase& p, const Shape& q, int ncl, int M) {
  const int rt = adj || q.KC <= 4 ? 4 : 8, warps = (adj ? q.adj_threads : q.fwd_threads) / 32;
  const double group = (adj ? 128.0 * q.adj_kc + 160.0 : 96.0 * q.KC + 200.0) * ((warps + 3) / 4);
  const size_t row = adj ? q.adj_row : q.fwd_row, fix = adj ? q.adj_fix : q.fwd_fix;
  double best = 1e30;
  for (int R = rt; R <= kMaxRows && fix + row * R <= kSmemMax; R += rt) {
    const int waves = ((M + R - 1) / R + ncl - 1) / ncl;
    const double t = waves * (1500.0 + R / rt * group);
    if (t < best - 1e-9) { best = t; p.R = R; }
    if (R >= M) break;
  }
}

template <auto kern>      // (a template argument: the per-kernel caches below must not be shared by kernels of the same signature)
bool launch_solve(bool adj, F32Args& a, const Shape& q, cudaStream_t s) {
  const int most = !adj ? fwd_most(q.KC) : q.adj_threads <= 256 ? 256 : 384;
  static int cache[kMaxDevices][9] = {};       // resident clusters by cluster size
  const int dev = current_device_slot(), threads = adj ? q.adj_threads : q.fwd_threads;
  const size_t row = adj ? q.adj_row : q.fwd_row, fix = adj ? q.adj_fix : q.fwd_fix;
  int* st = status_ptr();
  if (dev < 0 || !st) return false;
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute at[2];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = q.NC; at[0].val.clusterDim.y = 1; at[0].val.clusterDim.z = 1;
  at[1].id = cudaLaunchAttributeCooperative;       // the grid barrier needs every CTA resident
  at[1].val.cooperative = 1;
  cfg.blockDim = dim3(threads); cfg.attrs = at; cfg.numAttrs = 1;
  // (widths that share a kernel share the answer: at the most threads and shared memory any of them asks for)
  int& clusters = cache[dev][q.NC];
  if (clusters == 0) {
    if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmemMax) != cudaSuccess) { cudaGetLastError(); return false; }
    cfg.gridDim = dim3(q.NC); cfg.dynamicSmemBytes = kSmemMax; cfg.blockDim = dim3(most);
    int n = 0;
    if (cudaOccupancyMaxActiveClusters(&n, kern, &cfg) != cudaSuccess) { cudaGetLastError(); n = 0; }
    clusters = n > 0 ? n : -1;
    cfg.blockDim = dim3(threads);
  }
  const int ncl = clusters;
  if (ncl <= 0) return false;
  a.limit_ns = wait_limit_ns();
  int rmax = 4, blocks = 1;
  double steps = 0;       // cell evaluations of all phases, in rows
  for (int i = 0; i < a.nph; ++i) {
    F32Phase& p = a.ph[i];
    const int full = p.nk < p.nfull ? p.nk : p.nfull;
    steps += ((double)full * (p.n + p.last_kind) + (double)(p.nk - full) * p.ntail) * a.B;      // (kLastStore one step more, kLastCoarse two)
    tune(adj, p, q, ncl, p.nk * a.B);
    if (p.R > rmax) rmax = p.R;
    const int nb = (p.nk * a.B + p.R - 1) / p.R;
    if (nb > blocks) blocks = nb;
  }
  if (blocks > ncl) blocks = ncl;
  cfg.gridDim = dim3(blocks * q.NC); cfg.dynamicSmemBytes = fix + row * rmax; cfg.stream = s; cfg.numAttrs = 2;
  ProfScope prof(adj ? KC_ADJ_STEP : KC_FWD_STEP, 6.0 * steps * a.H * a.H, s);
  if (cudaLaunchKernelEx(&cfg, kern, a, q.NC, q.U, rmax, st) != cudaSuccess) { cudaGetLastError(); return false; }
  count_launch();
  return true;
}
}  // namespace

bool f32_solve_fits(int H) {
  Shape q;
  return pick_shape(H, &q);
}

bool f32_solve(bool adjoint, F32Args& a, cudaStream_t s) {
  Shape q;
  if (!solve_enabled() || !pick_shape(a.H, &q)) return false;
  if (adjoint) {
    if (q.adj_kp == 32)
      return q.adj_kc == 1   ? launch_solve<f32_adj_kernel<false, 32, 1, 384>>(true, a, q, s)
             : q.adj_kc == 2 ? launch_solve<f32_adj_kernel<false, 32, 2, 384>>(true, a, q, s)
                             : launch_solve<f32_adj_kernel<false, 32, 3, 384>>(true, a, q, s);
    if (q.adj_kp == 16)
      return q.adj_kc == 2             ? launch_solve<f32_adj_kernel<true, 16, 2, 384>>(true, a, q, s)
             : q.adj_threads <= 256 ? launch_solve<f32_adj_kernel<true, 16, 3, 256>>(true, a, q, s)
                                    : launch_solve<f32_adj_kernel<true, 16, 3, 384>>(true, a, q, s);
    return q.adj_kc == 3   ? launch_solve<f32_adj_kernel<true, 8, 3, 256>>(true, a, q, s)
           : q.adj_kc == 4 ? launch_solve<f32_adj_kernel<true, 8, 4, 384>>(true, a, q, s)
                           : launch_solve<f32_adj_kernel<true, 8, 5, 384>>(true, a, q, s);
  }
  switch (q.KC) {
    case 1: return launch_solve<f32_fwd_kernel<false, 1>>(false, a, q, s);
    case 2: return launch_solve<f32_fwd_kernel<false, 2>>(false, a, q, s);
    case 3: return launch_solve<f32_fwd_kernel<false, 3>>(false, a, q, s);
    case 4: return launch_solve<f32_fwd_kernel<true, 4>>(false, a, q, s);
    case 5: return launch_solve<f32_fwd_kernel<true, 5>>(false, a, q, s);
    case 6: return launch_solve<f32_fwd_kernel<true, 6>>(false, a, q, s);
    case 7: return launch_solve<f32_fwd_kernel<true, 7>>(false, a, q, s);
    case 8: return launch_solve<f32_fwd_kernel<true, 8>>(false, a, q, s);
    case 9: return launch_solve<f32_fwd_kernel<true, 9>>(false, a, q, s);
    case 10: return launch_solve<f32_fwd_kernel<true, 10>>(false, a, q, s);
    default: return launch_solve<f32_fwd_kernel<true, 11>>(false, a, q, s);
  }
}

namespace {
template <int KC> bool launch_lin(const LinSet& ls, const Shape& q, int gx, int gy, int R, cudaStream_t s) {
  static bool attr[kMaxDevices] = {false};
  if (!set_smem_once(f32_lin_kernel<KC>, (int)kSmemMax, attr)) return false;
  f32_lin_kernel<KC><<<dim3(gx, gy), q.fwd_threads, q.fwd_fix + q.fwd_row * R, s>>>(ls, q.U, R);
  count_launch();
  return true;
}
}  // namespace

bool f32_linearise(const LinArgs* levels, int n, cudaStream_t s) {
  Shape q;
  const int H = levels[0].H;
  if (!solve_enabled() || !pick_shape(H, &q)) return false;
  LinSet ls;
  ls.n = n;
  i64 rows = 0;
  double flops = 0;
  for (int l = 0; l < n; ++l) { ls.l[l] = levels[l]; rows += levels[l].M; flops += 2.0 * levels[l].M * 3.0 * H * H; }
  const int gx = (H + q.U - 1) / q.U, ncl = 148 / gx;
  int R = 8;
  while (R < 32 && rows > (i64)R * ncl * 2) R += 8;      // (two blocks and more per CTA: the next one is fetched behind the current)
  ls.blk0[0] = 0;
  for (int l = 0; l < n; ++l) ls.blk0[l + 1] = ls.blk0[l] + (levels[l].M + R - 1) / R;
  const int gy = ls.blk0[n] < ncl ? ls.blk0[n] : ncl;
  ProfScope prof(KC_LINEARISE, flops, s);
  switch (q.KC) {
    case 1: return launch_lin<1>(ls, q, gx, gy, R, s);
    case 2: return launch_lin<2>(ls, q, gx, gy, R, s);
    case 3: return launch_lin<3>(ls, q, gx, gy, R, s);
    case 4: return launch_lin<4>(ls, q, gx, gy, R, s);
    case 5: return launch_lin<5>(ls, q, gx, gy, R, s);
    case 6: return launch_lin<6>(ls, q, gx, gy, R, s);
    case 7: return launch_lin<7>(ls, q, gx, gy, R, s);
    case 8: return launch_lin<8>(ls, q, gx, gy, R, s);
    case 9: return launch_lin<9>(ls, q, gx, gy, R, s);
    case 10: return launch_lin<10>(ls, q, gx, gy, R, s);
    default: return launch_lin<11>(ls, q, gx, gy, R, s);
  }
}

int f32_device_status() {
  const int dev = current_device_slot();
  if (dev < 0) return -1;
  if (!g_f32_status_ptrs[dev]) return 0;
  int v = 0;
  return cudaMemcpy(&v, g_f32_status_ptrs[dev], sizeof(int), cudaMemcpyDeviceToHost) == cudaSuccess ? v : -1;
}
int f32_clear_device_status() {
  const int dev = current_device_slot();
  if (dev < 0) return -1;
  if (!g_f32_status_ptrs[dev]) return 0;
  return cudaMemset(g_f32_status_ptrs[dev], 0, sizeof(int)) == cudaSuccess ? 0 : -1;
}

}  // namespace mg
