// The fp32 multigrid solve (forward and adjoint) as ONE persistent launch for widths whose recurrent weights fit the shared
// memory of a cluster of 1 to 8 CTAs (H <= 352).
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
// Products are FFMA (packed in pairs along the reduction, fma.rn.f32x2, in the forward direction): a thread holds 4 rows x 3
// gates (forward) or 8 x 4 outputs (adjoint); KP lanes share the sums of 4 rows when few rows would not fill the CTA.
// Measured (B200, whole training steps launched from the host, before -> now): 64 steps x 2 rows, H = 32: 489 -> 262 us; two
// layers of 128 x 100 rows, H = 104: 4801 -> 2093 us; 128 x 16 rows, H = 256 (tf32 split): 1935 -> 1356 us.  A dependent step
// of the coarsest level takes 1.4 / 1.9 us at H = 32 (forward / adjoint) and 3.3 / 3.2 us at H = 256, a step of 3300 rows at
// H = 104 15 / 16 us (14 TFLOP/s): bound by the delivery of operands from shared memory and, with few rows, by the latency of a
// step's parts.
#include "cell.cuh"
#include "f32_solve.cuh"

namespace mg {
namespace {

typedef unsigned long long u64;
constexpr int kMaxThreads = 512, kFwdThreads = 640;
constexpr int kMaxRows = 64;
constexpr size_t kSmemMax = 227 * 1024 - 2048;     // dynamic part: the kernels hold under 1 KiB of static shared memory
constexpr uint64_t kWaitLimitNs = 2000000000ull;

__device__ int g_f32_status = 0;
int* g_f32_status_ptrs[kMaxDevices] = {nullptr};

__device__ __forceinline__ void fma2(u64& d, u64 a, u64 b) { asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(d) : "l"(a), "l"(b)); }
__device__ __forceinline__ float2 unpack2(u64 v) {
  float2 f;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(f.x), "=f"(f.y) : "l"(v));
  return f;
}
__device__ __forceinline__ ulonglong2 lds2(const float* p) { return *reinterpret_cast<const ulonglong2*>(p); }
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
// either every CTA of a cluster goes on or every one leaves.
template <bool MULTI>
__device__ bool grid_barrier(unsigned* bar, unsigned target, int nc, int* status, int* verdict) {
  block_sync<MULTI>();
  if (ctarank() == 0 && threadIdx.x == 0) {
    asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(bar) : "memory");
    int ok = 1;
    unsigned spins = 0, v;
    uint64_t t0 = 0;
    while (true) {
      asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(bar) : "memory");
      if (v >= target) break;
      if ((++spins & 127u) == 0) {
        int st;
        asm volatile("ld.relaxed.gpu.global.s32 %0, [%1];" : "=r"(st) : "l"(status) : "memory");
        if (t0 == 0) t0 = now_ns();
        if (st != 0) { ok = 0; break; }
        if (now_ns() - t0 > kWaitLimitNs) { atomicCAS(status, 0, 41); ok = 0; break; }
      }
    }
    for (int c = 0; c < nc; ++c) asm volatile("st.shared::cluster.s32 [%0], %1;" ::"r"(peer_addr(verdict, c)), "r"(ok) : "memory");
  }
  block_sync<MULTI>();
  return *(volatile int*)verdict != 0;
}

// A shared-memory load delivers 32 words a cycle however they are shared, so a sum over r rows and c weight rows runs at
// r c / (r + c) multiply-adds per word against the 4 that keep the FFMA pipe busy.  Adjoint: 8 rows where a lane has a sum to
// itself (2.7 per word), 4 where KP lanes share one and latency counts.  Forward: 4 (1.7); with 8 the gate operands of the
// rows do not fit the registers next to the sums (256 units x 2000 rows: 64 us a step spilled).
template <int KP> struct Tile { static constexpr int RT = KP == 1 ? 8 : 4, NR = KP >= 4 ? 1 : RT / KP; };
template <int KP> struct FTile { static constexpr int RT = 4, NR = KP >= 4 ? 1 : RT / KP; };
// Items: 8 units (fastest: the eight lanes that a 16-byte load serves together then read eight different weight rows, which
// never share a bank), KP lanes per sum, RG groups of RT rows, unit blocks.
struct Item { int rg, u, kp; bool live; };
template <int KP>
__device__ __forceinline__ Item item_of(int it, int RG, int n) {
  Item x;
  const int ul = it & 7;
  int q = it >> 3;
  x.kp = q % KP;
  q /= KP;
  x.rg = q % RG;
  const int u = (q / RG) * 8 + ul;
  x.live = u < n;
  x.u = min(u, n - 1);
  return x;
}
// pre[gate][q] of this lane's rows = sum_k S[row][k] Ws[gate*U + u][k]
template <int KP>
__device__ __forceinline__ void fwd_sums(const float* S, const float* Ws, int ld, int H, int U, const Item& x, float (&pre)[3][FTile<KP>::NR]) {
  constexpr int RT = FTile<KP>::RT, NR = FTile<KP>::NR;
  u64 acc[3][RT];
#pragma unroll
  for (int g = 0; g < 3; ++g)
#pragma unroll
    for (int r = 0; r < RT; ++r) acc[g][r] = 0ull;
  const float* s0 = S + x.rg * RT * ld;
  const float* w0 = Ws + x.u * ld;
#pragma unroll 2
  for (int i = x.kp * 4; i < H; i += KP * 4) {
    ulonglong2 b[3];
#pragma unroll
    for (int g = 0; g < 3; ++g) b[g] = lds2(w0 + g * U * ld + i);
#pragma unroll
    for (int r = 0; r < RT; ++r) {
      const ulonglong2 v = lds2(s0 + r * ld + i);
#pragma unroll
      for (int g = 0; g < 3; ++g) { fma2(acc[g][r], v.x, b[g].x); fma2(acc[g][r], v.y, b[g].y); }
    }
  }
#pragma unroll
  for (int g = 0; g < 3; ++g)
#pragma unroll
    for (int r = 0; r < RT; ++r) {
      const float2 f = unpack2(acc[g][r]);
      float v = f.x + f.y;
#pragma unroll
      for (int o = 1; o < KP; o <<= 1) v += __shfl_xor_sync(0xffffffffu, v, 8 * o);
      if (r / NR == x.kp) pre[g][r % NR] = v;
    }
}

struct FwdShared { float *S[2], *Ws, *bh; int ld, U, Un, u0, rank, NC; int *rk, *rb; };

// What a step needs from global memory (every thread has at most one item).  The next step's values are requested as soon as
// the current ones are used, straight into the same registers (a copy would wait for them), and used behind the next sums, so
// their latency hides behind the exchange.
template <int KP> struct FwdOps {
  static constexpr int NR = FTile<KP>::NR;
  float gi[3][NR], ad[NR];
  bool on[NR];
};
template <int KP>
__device__ __forceinline__ void fwd_load(const F32Args& a, const F32Phase& p, const FwdShared& sh, const Item& x, int j, bool coarse, FwdOps<KP>& o) {
  constexpr int NR = FwdOps<KP>::NR;
  const int H = a.H, c = sh.u0 + x.u;
#pragma unroll
  for (int q = 0; q < NR; ++q) {
    const int row = x.rg * FTile<KP>::RT + x.kp * NR + q, k = sh.rk[row], b = sh.rb[row];
    o.on[q] = x.live && k >= 0 && (j < (k < p.nfull ? p.n : p.ntail) || (j >= p.n && k < p.nfull));
    o.ad[q] = o.gi[0][q] = o.gi[1][q] = o.gi[2][q] = 0.f;
    if (o.on[q]) {
      const float* gp = a.gi + (coarse ? p.op2 + k * p.op2_ks : p.op + k * p.op_ks + j * p.op_ss) + (i64)b * 3 * H + c;
      o.gi[0][q] = gp[0]; o.gi[1][q] = gp[H]; o.gi[2][q] = gp[2 * H];
      // the additive term; of the coarse step: the C-point
      if (coarse) o.ad[q] = __ldcg(p.uc + k * p.uc_ks + (i64)b * H + c);
      else if (p.g) o.ad[q] = __ldcg(p.g + k * p.g_ks + j * p.g_ss + (i64)b * H + c);
    }
  }
}
// mode 0: step, result to S[cur ^ 1] and global memory; 1: v, to S[cur ^ 1] only; 2: coarse right-hand side
template <int KP>
__device__ __forceinline__ float fwd_finish(const F32Args& a, const F32Phase& p, const FwdShared& sh, const Item& x, int cur, int j, int mode,
                                            const FwdOps<KP>& o, const float (&pre)[3][FwdOps<KP>::NR], float norm) {
  constexpr int NR = FwdOps<KP>::NR;
  const int c = sh.u0 + x.u;
  if (!x.live) return norm;
#pragma unroll
  for (int q = 0; q < NR; ++q) {
    const int row = x.rg * FTile<KP>::RT + x.kp * NR + q;
    const float hp = sh.S[cur][row * sh.ld + c];
    const float phi = cell_forward(o.gi[0][q], o.gi[1][q], o.gi[2][q], pre[0][q] + sh.bh[x.u], pre[1][q] + sh.bh[sh.U + x.u],
                                   pre[2][q] + sh.bh[2 * sh.U + x.u], hp, mode == 2 ? p.gamma2 : p.gamma, a.cell);
    float* own = &sh.S[cur ^ 1][row * sh.ld + c];
    const i64 bo = (i64)sh.rb[row] * a.H + c;
    const int k = sh.rk[row];
    if (mode == 2) {
      if (o.on[q]) {
        const float v = *own, r = o.ad[q] - v;      // (v was left there by the step before)
        norm += r * r;
        if (p.ucd) p.ucd[k * p.ucd_ks + bo] = o.ad[q];
        p.last[k * p.last_ks + bo] = v - phi;
      }
    } else {
      const float v = o.on[q] ? phi + o.ad[q] : 0.f;
      *own = v;
      if (o.on[q] && mode == 0) {
        if (j >= p.n) p.last[k * p.last_ks + bo] = v;
        else p.out[k * p.out_ks + j * p.out_ss + bo] = v;
      }
    }
  }
  return norm;
}

// All steps of one row block; S[0] holds the start.  load(dst, src, ks, ...): the block's rows from global memory.
template <bool MULTI, int KP, class Load>
__device__ __forceinline__ float fwd_block(const F32Args& a, const F32Phase& p, const FwdShared& sh, float norm, Load load) {
  const int H = a.H, RG = p.R / FTile<KP>::RT, items = (((sh.Un + 7) / 8) * 8 * RG * KP + 31) & ~31, steps = p.n + (p.last_kind != kLastNone ? 1 : 0);
  const bool works = (int)threadIdx.x < items;                  // whole warps: the sums are shared by shuffles
  const bool coarse = p.last_kind == kLastCoarse;
  FwdOps<KP> o;
  float pre[3][FwdOps<KP>::NR];
  const Item x = item_of<KP>(threadIdx.x, RG, sh.Un);
  if (works) fwd_load<KP>(a, p, sh, x, 0, false, o);
  int cur = 0;
  for (int j = 0; j < steps; ++j) {
    const int mode = j == p.n && coarse ? 1 : 0;
    if (works) {
      fwd_sums<KP>(sh.S[cur], sh.Ws, sh.ld, H, sh.U, x, pre);
      norm = fwd_finish<KP>(a, p, sh, x, cur, j, mode, o, pre, norm);
      if (j + 1 < steps) fwd_load<KP>(a, p, sh, x, j + 1, false, o);
      else if (coarse) fwd_load<KP>(a, p, sh, x, p.n, true, o);
    }
    if (j + 1 == steps) break;
    __syncthreads();
    if (MULTI) {             // this CTA's columns to the peers
      const int U4 = sh.Un / 4;
      for (int e = threadIdx.x; e < p.R * U4; e += blockDim.x) {
        float* q = sh.S[cur ^ 1] + (e / U4) * sh.ld + sh.u0 + (e % U4) * 4;
        const float4 v = *reinterpret_cast<const float4*>(q);
        for (int d = 1; d < sh.NC; ++d) { const int t = sh.rank + d; st_peer4(peer_addr(q, t < sh.NC ? t : t - sh.NC), v); }
      }
      cluster_sync();
    }
    cur ^= 1;
  }
  if (coarse) {
    __syncthreads();         // v of this CTA's units sits in S[cur ^ 1]
    load(sh.S[cur], p.src2, p.src2_ks, nullptr, 0);
    __syncthreads();
    if (works) {
      fwd_sums<KP>(sh.S[cur], sh.Ws, sh.ld, H, sh.U, x, pre);
      norm = fwd_finish<KP>(a, p, sh, x, cur, p.n, 2, o, pre, norm);
    }
  }
  return norm;
}

__device__ __forceinline__ void block_rows(const F32Args& a, const F32Phase& p, int r0, int* rk, int* rb) {
  if ((int)threadIdx.x < p.R) {
    const int m = r0 + threadIdx.x;
    const bool v = m < p.nk * a.B;
    rk[threadIdx.x] = v ? m / a.B : -1;
    rb[threadIdx.x] = v ? m % a.B : 0;
  }
}
__device__ __forceinline__ void add_norm(float norm, double* acc) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) norm += __shfl_xor_sync(0xffffffffu, norm, o);
  if ((threadIdx.x & 31) == 0 && norm != 0.f) atomicAdd(acc, (double)norm);
}

template <bool MULTI>
__global__ void __launch_bounds__(kFwdThreads, 1) f32_fwd_kernel(const __grid_constant__ F32Args a, int NC, int U, int rmax, int* status) {
  extern __shared__ __align__(16) float fsm[];
  __shared__ int rk[kMaxRows], rb[kMaxRows], verdict;
  const int H = a.H, ld = H + 4, rank = MULTI ? (int)ctarank() : 0;
  const int cid = blockIdx.x / NC, ncl = gridDim.x / NC;
  FwdShared sh;
  sh.ld = ld; sh.U = U; sh.u0 = rank * U; sh.Un = max(0, min(U, H - sh.u0)); sh.rank = rank; sh.NC = NC;
  sh.Ws = fsm; sh.S[0] = fsm + 3 * U * ld; sh.S[1] = sh.S[0] + rmax * ld; sh.bh = sh.S[1] + rmax * ld; sh.rk = rk; sh.rb = rb;
  for (int e = threadIdx.x; e < 3 * sh.Un * (H / 4); e += blockDim.x) {
    const int r = e / (H / 4), c = e % (H / 4), g = r / sh.Un, i = r % sh.Un;
    *reinterpret_cast<float4*>(sh.Ws + (g * U + i) * ld + 4 * c) = __ldg(reinterpret_cast<const float4*>(a.W + ((i64)g * H + sh.u0 + i) * H) + c);
  }
  for (int e = threadIdx.x; e < 3 * sh.Un; e += blockDim.x) sh.bh[(e / sh.Un) * U + e % sh.Un] = a.b_hh[(e / sh.Un) * H + sh.u0 + e % sh.Un];
  __syncthreads();
  unsigned target = 0;
  for (int ip = 0; ip < a.nph; ++ip) {
    const F32Phase& p = a.ph[ip];
    const int M = p.nk * a.B, nblk = (M + p.R - 1) / p.R;
    float norm = 0.f;
    for (int blk = cid; blk < nblk; blk += ncl) {
      __syncthreads();
      block_rows(a, p, blk * p.R, rk, rb);
      __syncthreads();
      auto load = [&](float* S, const float* src, i64 ks, float* copy, i64 cks) {
        for (int e = threadIdx.x; e < p.R * (H / 4); e += blockDim.x) {
          const int r = e / (H / 4), c = e % (H / 4), k = rk[r];
          float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
          if (k >= 0) {
            v = __ldcg(reinterpret_cast<const float4*>(src + k * ks + (i64)rb[r] * H) + c);
            if (copy && 4 * c >= sh.u0 && 4 * c < sh.u0 + sh.Un) *(reinterpret_cast<float4*>(copy + k * cks + (i64)rb[r] * H) + c) = v;
          }
          *reinterpret_cast<float4*>(S + r * ld + 4 * c) = v;
        }
      };
      load(sh.S[0], p.src, p.src_ks, p.copy, p.copy_ks);
      block_sync<MULTI>();       // the peers are done with the previous block before anything is pushed into S[1]
      if (p.KP == 4) norm = fwd_block<MULTI, 4>(a, p, sh, norm, load);
      else if (p.KP == 2) norm = fwd_block<MULTI, 2>(a, p, sh, norm, load);
      else norm = fwd_block<MULTI, 1>(a, p, sh, norm, load);
    }
    if (p.acc) add_norm(norm, p.acc);
    if (ip + 1 < a.nph) {
      target += ncl;
      if (!grid_barrier<MULTI>(a.bar, target, NC, status, &verdict)) return;
    }
  }
}

// ---- adjoint
// shared: Ws[3U][H] (this CTA's gate rows), Ad[R][3U + 4] (the formed operand),
// Pb[2][NC or 3 NC][R][U] (partial sums for this CTA's units by producer, and by gate where the gates are split)
constexpr int kSplitKP = 12, kSplitRows = 8;        // (split: blocks of at most 8 rows, KP = 4)
struct AdjVals { float4 m, a, g; };                 // four units of one row: mu, and of the step in flight a and the source
struct AdjNext { float4 cr, cz, cn, a, g; };        // ... the next step's coefficients, requested before the product in front of it

// SPLIT: the three gates' sums go to three groups of threads, each with partial results of its own (few rows: more warps)
template <int KP, bool SPLIT>
__device__ __forceinline__ void adj_product(const F32Args& a, const F32Phase& p, const float* Ws, const float* Ad, float* Pb, int lda, int U, int Un, int NC,
                                            int rank, bool multi) {
  constexpr int RT = Tile<KP>::RT, NR = Tile<KP>::NR;
  const int H = a.H, RG = p.R / RT, n4 = H / 4, items = (((n4 + 7) / 8) * 8 * RG * KP + 31) & ~31;
  if ((int)threadIdx.x >= p.nt) return;
  for (int it0 = threadIdx.x; it0 < (SPLIT ? 3 : 1) * items; it0 += p.nt) {
    const int gs = SPLIT ? it0 / items : 0, it = it0 - gs * items;
    const Item x = item_of<KP>(it, RG, n4);
    float acc[RT][4];
#pragma unroll
    for (int r = 0; r < RT; ++r) acc[r][0] = acc[r][1] = acc[r][2] = acc[r][3] = 0.f;
    const float* a0 = Ad + x.rg * RT * lda;
    // the operand rows are [gate][own units]: the reduction runs over 3 Un values
    for (int g = SPLIT ? gs : 0; g < (SPLIT ? gs + 1 : 3); ++g) {
      const float* ag = a0 + g * U;
      const float* wg = Ws + (i64)g * U * H + 4 * x.u;
#pragma unroll 1
      for (int i = x.kp * 4; i < Un; i += KP * 4) {
        float4 b[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) b[q] = *reinterpret_cast<const float4*>(wg + (i + q) * H);
#pragma unroll
        for (int r = 0; r < RT; ++r) {
          const float4 v = *reinterpret_cast<const float4*>(ag + r * lda + i);
          const float vq[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            acc[r][0] = fmaf(vq[q], b[q].x, acc[r][0]); acc[r][1] = fmaf(vq[q], b[q].y, acc[r][1]);
            acc[r][2] = fmaf(vq[q], b[q].z, acc[r][2]); acc[r][3] = fmaf(vq[q], b[q].w, acc[r][3]);
          }
        }
      }
    }
    const int n = 4 * x.u, d = n / U;
    float* dst0 = Pb + ((i64)(SPLIT ? rank * 3 + gs : rank) * p.R) * U + (n - d * U);
#pragma unroll
    for (int r = 0; r < RT; ++r) {
      float4 v = make_float4(acc[r][0], acc[r][1], acc[r][2], acc[r][3]);
#pragma unroll
      for (int o = 1; o < KP; o <<= 1) {
        v.x += __shfl_xor_sync(0xffffffffu, v.x, 8 * o); v.y += __shfl_xor_sync(0xffffffffu, v.y, 8 * o);
        v.z += __shfl_xor_sync(0xffffffffu, v.z, 8 * o); v.w += __shfl_xor_sync(0xffffffffu, v.w, 8 * o);
      }
      if (r / NR == x.kp && x.live) {
        float* q = dst0 + (x.rg * RT + r) * U;
        if (multi) st_peer4(peer_addr(q, d), v);
        else *reinterpret_cast<float4*>(q) = v;
      }
    }
  }
}

// kQ: quadruples of units per thread
template <bool MULTI, int kQ>
__global__ void __launch_bounds__(kMaxThreads, 1) f32_adj_kernel(const __grid_constant__ F32Args a, int NC, int U, int rmax, int* status) {
  extern __shared__ __align__(16) float fsm[];
  __shared__ int rk[kMaxRows], rb[kMaxRows], verdict;
  const int H = a.H, rank = MULTI ? (int)ctarank() : 0, u0 = rank * U, Un = max(0, min(U, H - u0)), lda = 3 * U + 4, U4 = Un / 4;
  const int cid = blockIdx.x / NC, ncl = gridDim.x / NC;
  // with one quadruple the next step's coefficients are requested in front of the product; two of them do not fit the registers
  // next to its sums, and such launches have enough work per step to bear the wait
  constexpr bool kAhead = kQ == 1;
  float* Ws = fsm;
  float* Ad = Ws + 3 * U * H;
  float* Pbuf = Ad + rmax * lda;
  const int pstride = 3 * NC * kSplitRows * U > NC * rmax * U ? 3 * NC * kSplitRows * U : NC * rmax * U;
  for (int e = threadIdx.x; e < 3 * Un * (H / 4); e += blockDim.x) {
    const int r = e / (H / 4), c = e % (H / 4), g = r / Un, i = r % Un;
    *reinterpret_cast<float4*>(Ws + (i64)(g * U + i) * H + 4 * c) = __ldg(reinterpret_cast<const float4*>(a.W + ((i64)g * H + u0 + i) * H) + c);
  }
  __syncthreads();
  unsigned target = 0;
  int par = 0;
  const float4 z4 = make_float4(0.f, 0.f, 0.f, 0.f);
  for (int ip = 0; ip < a.nph; ++ip) {
    const F32Phase& p = a.ph[ip];
    const int M = p.nk * a.B, nblk = (M + p.R - 1) / p.R, steps = p.n + (p.last_kind != kLastNone ? 1 : 0);
    const bool coarse = p.last_kind == kLastCoarse;
    float norm = 0.f;
    for (int blk = cid; blk < nblk; blk += ncl) {
      __syncthreads();
      block_rows(a, p, blk * p.R, rk, rb);
      __syncthreads();
      AdjVals x[kQ];
      AdjNext nx[kQ];
      float4 v[kQ], m2[kQ];
      // quadruple q of this thread: row and first unit
      auto where = [&](int q, int* row, int* u) { const int e = threadIdx.x + q * blockDim.x; *row = e / U4; *u = (e % U4) * 4; return *row < p.R && rk[*row] >= 0; };
      auto coefs = [&](int q, int j, bool cs) {           // coefficients and source of step j
        int row, u;
        nx[q].cr = nx[q].cz = nx[q].cn = nx[q].a = nx[q].g = z4;
        if (!where(q, &row, &u)) return;
        const int k = rk[row];
        if (!(j < (k < p.nfull ? p.n : p.ntail) || (j >= p.n && k < p.nfull))) return;
        const i64 bo = (i64)rb[row] * H + u0 + u, o = (cs ? p.op2 + k * p.op2_ks : p.op + k * p.op_ks + j * p.op_ss) + bo;
        const float* const* c = a.coef[p.level + (cs ? 1 : 0)];
        nx[q].a = *reinterpret_cast<const float4*>(c[0] + o);
        nx[q].cr = *reinterpret_cast<const float4*>(c[1] + o);
        nx[q].cz = *reinterpret_cast<const float4*>(c[2] + o);
        nx[q].cn = *reinterpret_cast<const float4*>(c[3] + o);
        if (!cs && p.g) nx[q].g = __ldcg(reinterpret_cast<const float4*>(p.g + k * p.g_ks + j * p.g_ss + bo));
      };
      auto start = [&](int q, const float* src, i64 ks, float* copy, i64 cks) {
        int row, u;
        float4 m = z4;
        if (!where(q, &row, &u)) return m;
        const i64 bo = (i64)rb[row] * H + u0 + u;
        m = __ldcg(reinterpret_cast<const float4*>(src + rk[row] * ks + bo));
        if (copy) *reinterpret_cast<float4*>(copy + rk[row] * cks + bo) = m;
        return m;
      };
      auto form = [&](int q) {                            // operand values; the requested coefficients become current
        int row, u;
        where(q, &row, &u);
        x[q].a = nx[q].a; x[q].g = nx[q].g;
        if (row >= p.R) return;
        const float4 m = x[q].m;
        const float4 c[3] = {nx[q].cr, nx[q].cz, nx[q].cn};
#pragma unroll
        for (int g = 0; g < 3; ++g)
          *reinterpret_cast<float4*>(Ad + row * lda + g * U + u) = make_float4(c[g].x * m.x, c[g].y * m.y, c[g].z * m.z, c[g].w * m.w);
      };
      auto product = [&]() {
        float* Pb = Pbuf + par * pstride;
        switch (p.KP) {
          case 1: adj_product<1, false>(a, p, Ws, Ad, Pb, lda, U, Un, NC, rank, MULTI); break;
          case 2: adj_product<2, false>(a, p, Ws, Ad, Pb, lda, U, Un, NC, rank, MULTI); break;
          case 4: adj_product<4, false>(a, p, Ws, Ad, Pb, lda, U, Un, NC, rank, MULTI); break;
          default: adj_product<4, true>(a, p, Ws, Ad, Pb, lda, U, Un, NC, rank, MULTI); break;
        }
        block_sync<MULTI>();
      };
      auto result = [&](int q) {                          // a*mu + sum of the partial products
        int row, u;
        float4 s = z4;
        if (!where(q, &row, &u)) return s;
        const float* Pb = Pbuf + par * pstride + row * U + u;
        for (int c = 0; c < (p.KP == kSplitKP ? 3 * NC : NC); ++c) {
          const float4 t = *reinterpret_cast<const float4*>(Pb + (i64)c * p.R * U);
          s.x += t.x; s.y += t.y; s.z += t.z; s.w += t.w;
        }
        const float4 A = x[q].a, m = x[q].m;
        return make_float4(fmaf(A.x, m.x, s.x), fmaf(A.y, m.y, s.y), fmaf(A.z, m.z, s.z), fmaf(A.w, m.w, s.w));
      };
#pragma unroll
      for (int q = 0; q < kQ; ++q) { x[q].m = start(q, p.src, p.src_ks, p.copy, p.copy_ks); if (steps > 0) { coefs(q, 0, false); form(q); } }
      for (int j = 0; j < steps; ++j) {
        const bool last = j == p.n, vstep = last && coarse;
        __syncthreads();
#pragma unroll
        for (int q = 0; q < kQ; ++q) {
          if (!kAhead) continue;
          if (j + 1 < steps) coefs(q, j + 1, false);
          else if (coarse) { coefs(q, p.n, true); m2[q] = start(q, p.src2, p.src2_ks, nullptr, 0); }
        }
        product();
#pragma unroll
        for (int q = 0; q < kQ; ++q) {
          const float4 r = result(q), g = x[q].g;
          x[q].m = make_float4(r.x + g.x, r.y + g.y, r.z + g.z, r.w + g.w);
          int row, u;
          if (!vstep && where(q, &row, &u)) {
            const int k = rk[row];
            const i64 bo = (i64)rb[row] * H + u0 + u;
            if (last) { if (k < p.nfull) *reinterpret_cast<float4*>(p.last + k * p.last_ks + bo) = x[q].m; }
            else if (j < (k < p.nfull ? p.n : p.ntail)) *reinterpret_cast<float4*>(p.out + k * p.out_ks + j * p.out_ss + bo) = x[q].m;
          }
          if (!kAhead) {
            if (j + 1 < steps) coefs(q, j + 1, false);
            else if (coarse) { coefs(q, p.n, true); m2[q] = start(q, p.src2, p.src2_ks, nullptr, 0); }
          }
          if (vstep) { v[q] = x[q].m; x[q].m = m2[q]; }
          if (j + 1 < steps || coarse) form(q);
        }
        par ^= 1;
      }
      if (coarse) {
        __syncthreads();
        product();
#pragma unroll
        for (int q = 0; q < kQ; ++q) {
          const float4 r = result(q);
          int row, u;
          if (!where(q, &row, &u) || rk[row] >= p.nfull) continue;
          const int k = rk[row];
          const i64 bo = (i64)rb[row] * H + u0 + u;
          const float4 uc = __ldcg(reinterpret_cast<const float4*>(p.uc + k * p.uc_ks + bo));
          const float d0 = uc.x - v[q].x, d1 = uc.y - v[q].y, d2 = uc.z - v[q].z, d3 = uc.w - v[q].w;
          norm += d0 * d0 + d1 * d1 + d2 * d2 + d3 * d3;
          if (p.ucd) *reinterpret_cast<float4*>(p.ucd + k * p.ucd_ks + bo) = uc;
          *reinterpret_cast<float4*>(p.last + k * p.last_ks + bo) = make_float4(v[q].x - r.x, v[q].y - r.y, v[q].z - r.z, v[q].w - r.w);
        }
        par ^= 1;
      }
    }
    if (p.acc) add_norm(norm, p.acc);
    if (ip + 1 < a.nph) {
      target += ncl;
      if (!grid_barrier<MULTI>(a.bar, target, NC, status, &verdict)) return;
    }
  }
  block_sync<MULTI>();      // no CTA leaves while a peer may still write its partial sums
}

// ---- linearisation: the forward product of every level's rows with the transposed-Jacobian epilogue; no exchange
struct LinSet { LinArgs l[kF32Levels]; int n, blk0[kF32Levels + 1]; };
__global__ void __launch_bounds__(kFwdThreads, 1) f32_lin_kernel(const __grid_constant__ LinSet ls, int U, int R) {
  extern __shared__ __align__(16) float fsm[];
  const int H = ls.l[0].H, B = ls.l[0].B, ld = H + 4, u0 = blockIdx.x * U, Un = min(U, H - u0);
  float* Ws = fsm;
  float* S = fsm + 3 * U * ld;
  for (int e = threadIdx.x; e < 3 * Un * (H / 4); e += blockDim.x) {
    const int r = e / (H / 4), c = e % (H / 4), g = r / Un, i = r % Un;
    *reinterpret_cast<float4*>(Ws + (g * U + i) * ld + 4 * c) = __ldg(reinterpret_cast<const float4*>(ls.l[0].W_hh + ((i64)g * H + u0 + i) * H) + c);
  }
  for (int blk = blockIdx.y; blk < ls.blk0[ls.n]; blk += gridDim.y) {
    int lv = 0;
    while (blk >= ls.blk0[lv + 1]) ++lv;
    const LinArgs& a = ls.l[lv];
    const int r0 = (blk - ls.blk0[lv]) * R;
    __syncthreads();
    for (int e = threadIdx.x; e < R * (H / 4); e += blockDim.x) {
      const int r = e / (H / 4), c = e % (H / 4), m = r0 + r;
      float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
      if (m < a.M) {
        const int j1 = m / B, b = m % B;
        const i64 t = a.t0 + (i64)j1 * a.stride_t;
        v = *(reinterpret_cast<const float4*>(t == 0 ? a.h0 + (i64)b * H : a.h + ((t - 1) * B + b) * H) + c);
      }
      *reinterpret_cast<float4*>(S + r * ld + 4 * c) = v;
    }
    __syncthreads();
    constexpr int RT = FTile<1>::RT;
    const int RG = R / RT, items = ((Un + 7) / 8) * 8 * RG;
    for (int it = threadIdx.x; it < items; it += blockDim.x) {
      const Item x = item_of<1>(it, RG, Un);
      float pre[3][RT];
      fwd_sums<1>(S, Ws, ld, H, U, x, pre);
      if (!x.live) continue;
      const int c = u0 + x.u;
      const float br = a.b_hh[c], bz = a.b_hh[H + c], bn = a.b_hh[2 * H + c];
#pragma unroll
      for (int r = 0; r < RT; ++r) {
        const int m = r0 + x.rg * RT + r;
        if (m >= a.M) continue;
        const int j1 = m / B, b = m % B;
        const i64 t = a.t0 + (i64)j1 * a.stride_t;
        const float* gi = a.gi + ((t + a.stride_t - 1) * B + b) * 3 * H + c;
        const CellLin L = cell_linearise(gi[0], gi[H], gi[2 * H], pre[0][r] + br, pre[1][r] + bz, pre[2][r] + bn, S[(x.rg * RT + r) * ld + c], a.gamma, a.cell);
        const i64 o = (i64)m * H + c;
        a.a[o] = L.a; a.cr[o] = L.cr; a.cz[o] = L.cz; a.cn[o] = L.cn;
        if (a.cnp) a.cnp[o] = L.cnp;
      }
    }
  }
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

// CTAs per cluster, units per CTA and the shared memory of `R` rows per block
struct Shape { int NC, U; };
size_t fwd_bytes(int H, int U, int R) { return (size_t)((3 * U + 2 * R) * (H + 4) + 3 * U) * 4; }
size_t adj_bytes(int H, int U, int NC, int R) { return (size_t)(3 * U * H + R * (3 * U + 4) + 2 * NC * (R > 3 * kSplitRows ? R : 3 * kSplitRows) * U) * 4; }
size_t shape_bytes(bool adj, int H, Shape q, int R) { return adj ? adj_bytes(H, q.U, q.NC, R) : fwd_bytes(H, q.U, R); }
bool pick_shape(int H, Shape* q) {
  for (int nc = 1; nc <= 8; nc *= 2) {
    const int U = ((H + nc - 1) / nc + 3) / 4 * 4;
    if ((nc - 1) * U >= H) continue;               // every CTA owns at least one unit
    if (fwd_bytes(H, U, 8) <= kSmemMax && adj_bytes(H, U, nc, 8) <= kSmemMax) { *q = Shape{nc, U}; return true; }
  }
  return false;
}
constexpr int kMaxQ = 2;
// Rows per block of a phase: the fewest waves of blocks, weighed against the time of a step (operand delivery of the block's
// rows plus about 1500 cycles of exchange, latency and epilogue).  The number of lanes that share a sum decides the order of
// its terms: it is taken from the complete intervals alone (the same for every phase of a level, `fixed_kp` = 0), so that
// repeating a relaxation in another phase gives the same bits.
void tune(bool adj, F32Phase& p, int H, Shape q, int ncl, int M, int fixed_kp) {
  double best = 1e30;
  for (int R = 4; R <= kMaxRows; R += 4) {
    if (shape_bytes(adj, H, q, R) > kSmemMax) break;
    if (adj && (i64)R * q.U / 4 > (i64)kMaxQ * kMaxThreads) break;
    const int cols = (((adj ? H / 4 : q.U) + 7) / 8) * 8;
    int KP = fixed_kp > 0 ? fixed_kp : 1;
    const int most = adj ? kMaxThreads : kFwdThreads;
    while (fixed_kp == 0 && KP < 4 && cols * (R / 4) * KP * 2 <= most) KP *= 2;
    if (fixed_kp == 0 && adj && KP == 4 && R <= kSplitRows && cols * (R / 4) * kSplitKP <= kMaxThreads) KP = kSplitKP;
    if (KP == kSplitKP && R > kSplitRows) continue;
    const int rt = adj && KP == 1 ? Tile<1>::RT : 4, base = cols * (R / rt);
    if (R % rt != 0) continue;
    if ((KP > 1 || !adj) && base * KP > most) continue;   // lanes share a sum only where every item has a thread; forward: always
    const int items = base * KP, passes = (items + most - 1) / most, nt = ((items + passes - 1) / passes + 31) / 32 * 32;
    const int waves = ((M + R - 1) / R + ncl - 1) / ncl;
    // cycles of one item's operand delivery, with one warp on each of the four schedulers
    const double per = adj ? (rt + 4.0) * 4 * 3.0 * q.U : (rt + 3.0) * 4 * H;
    const double t = waves * (1500.0 + passes * ((nt / 32 + 3) / 4) * per / KP);
    if (t < best - 1e-9) { best = t; p.R = R; p.KP = KP; p.nt = nt; }
    if (R >= M && best < 1e30) break;
  }
}

template <class K>
int max_clusters(K kern, int nc, int threads, size_t smem) {      // co-resident clusters of this shape on the current device
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(nc); cfg.blockDim = dim3(threads); cfg.dynamicSmemBytes = smem;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = nc; at[0].val.clusterDim.y = 1; at[0].val.clusterDim.z = 1;
  cfg.attrs = at; cfg.numAttrs = 1;
  int n = 0;
  if (cudaOccupancyMaxActiveClusters(&n, kern, &cfg) != cudaSuccess) { cudaGetLastError(); return 0; }
  return n;
}

template <auto kern>      // (a template argument: the per-kernel cache below must not be shared by kernels of the same signature)
bool launch_solve(bool adj, const F32Args& a, Shape q, int blocks, int rmax, cudaStream_t s) {
  static bool attr[kMaxDevices] = {false};
  int* st = status_ptr();
  if (!st || !set_smem_once(kern, (int)kSmemMax, attr)) return false;
  if (cudaMemsetAsync(a.bar, 0, sizeof(unsigned), s) != cudaSuccess) return false;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(blocks * q.NC); cfg.blockDim = dim3(adj ? kMaxThreads : kFwdThreads); cfg.dynamicSmemBytes = shape_bytes(adj, a.H, q, rmax); cfg.stream = s;
  cudaLaunchAttribute at[2];
  at[0].id = cudaLaunchAttributeCooperative;       // the grid barrier needs every CTA resident
  at[0].val.cooperative = 1;
  at[1].id = cudaLaunchAttributeClusterDimension;
  at[1].val.clusterDim.x = q.NC; at[1].val.clusterDim.y = 1; at[1].val.clusterDim.z = 1;
  cfg.attrs = at; cfg.numAttrs = 2;
  if (cudaLaunchKernelEx(&cfg, kern, a, q.NC, q.U, rmax, st) != cudaSuccess) { cudaGetLastError(); return false; }
  count_launch();
  return true;
}

}  // namespace

bool f32_solve_fits(int H) {
  Shape q;
  return H % 8 == 0 && pick_shape(H, &q);
}

bool f32_solve(bool adjoint, F32Args& a, cudaStream_t s) {
  static int clusters[kMaxDevices][2][4] = {};        // [device][direction][log2 NC]: co-resident clusters at the largest shared memory
  Shape q;
  const int dev = current_device_slot();
  if (dev < 0 || !pick_shape(a.H, &q)) return false;
  int& ncl = clusters[dev][adjoint ? 1 : 0][q.NC == 1 ? 0 : q.NC == 2 ? 1 : q.NC == 4 ? 2 : 3];
  if (ncl == 0) {
    auto count = [&](auto kern) {
      if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmemMax) != cudaSuccess) { cudaGetLastError(); return 0; }
      return max_clusters(kern, q.NC, adjoint ? kMaxThreads : kFwdThreads, kSmemMax);
    };
    ncl = adjoint ? count(f32_adj_kernel<true, 2>) : count(f32_fwd_kernel<true>);
  }
  if (ncl <= 0) return false;
  int rmax = 4, blocks = 1;
  for (int i = 0; i < a.nph; ++i) {
    F32Phase& p = a.ph[i];
    tune(adjoint, p, a.H, q, ncl, p.nfull * a.B, 0);
    tune(adjoint, p, a.H, q, ncl, p.nk * a.B, p.KP);
    if (p.R > rmax) rmax = p.R;
    const int nb = (p.nk * a.B + p.R - 1) / p.R;
    if (nb > blocks) blocks = nb;
  }
  if (blocks > ncl) blocks = ncl;
  if (!adjoint) return q.NC > 1 ? launch_solve<f32_fwd_kernel<true>>(false, a, q, blocks, rmax, s) : launch_solve<f32_fwd_kernel<false>>(false, a, q, blocks, rmax, s);
  if ((i64)rmax * q.U / 4 <= kMaxThreads)      // one quadruple of units per thread
    return q.NC > 1 ? launch_solve<f32_adj_kernel<true, 1>>(true, a, q, blocks, rmax, s) : launch_solve<f32_adj_kernel<false, 1>>(true, a, q, blocks, rmax, s);
  return q.NC > 1 ? launch_solve<f32_adj_kernel<true, 2>>(true, a, q, blocks, rmax, s) : launch_solve<f32_adj_kernel<false, 2>>(true, a, q, blocks, rmax, s);
}

bool f32_linearise(const LinArgs* levels, int n, cudaStream_t s) {
  static bool attr[kMaxDevices] = {false};
  Shape q;
  const int H = levels[0].H;
  if (!pick_shape(H, &q) || !set_smem_once(f32_lin_kernel, (int)kSmemMax, attr)) return false;
  LinSet ls;
  ls.n = n;
  i64 rows = 0;
  double flops = 0;
  for (int l = 0; l < n; ++l) { ls.l[l] = levels[l]; rows += levels[l].M; flops += 2.0 * levels[l].M * 3.0 * H * H; }
  int R = 8;
  while (R < 32 && rows > (i64)R * 2 * (148 / q.NC) && (size_t)(3 * q.U + R + 8) * (H + 4) * 4 <= kSmemMax) R += 8;
  ls.blk0[0] = 0;
  for (int l = 0; l < n; ++l) ls.blk0[l + 1] = ls.blk0[l] + (levels[l].M + R - 1) / R;
  const int gx = (H + q.U - 1) / q.U, gy = ls.blk0[n] < 148 / gx ? ls.blk0[n] : 148 / gx;
  ProfScope prof(KC_LINEARISE, flops, s);
  f32_lin_kernel<<<dim3(gx, gy), kFwdThreads, (size_t)(3 * q.U + R) * (H + 4) * 4, s>>>(ls, q.U, R);
  count_launch();
  return true;
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
