// Dependent adjoint steps over the same rows in one launch, sm_100a:
//
//   lambda_{s+1}[m, n] = a_s[m, n] * lambda_s[m, n] + sum_j dA_s[m, j] * W_hhT[n, j] (+ g_s[m, n])      dA_s = [c_r | c_z | c_n]_s * lambda_s
//
// for the steps of a relaxation between two C-points (rows m = (k, b): interval k, batch row b).  No row reads another one's, but the
// last step may replace the rows that the next interval started from (a C-step).
//
// Step by step (packing kernel, then a product) such a step costs 8.5 us at 64 rows and 12.5 at 512 (H = 1024), of which the tensor
// cores need 0.3 and 2.3: two launches, their first loads, and all of W_hhT from L2 each time.  Here
//  * the weights stay on the chip: a cluster of S CTAs owns 128 columns n, CTA j of it the reduction over its share of the units
//    (all three gates of a unit), and keeps its slice of W_hhT in TENSOR MEMORY as the A operand of tcgen05.mma.  The product is
//    formed transposed, D^T[n, m]: 128 lanes = columns, up to 128 accumulator columns = rows;
//  * partial sums change hands by st.async into the owner's shared memory (NR / S rows per CTA), added in rank order.  They are
//    finished from there, a warp four rows, a lane four neighbouring columns, so every access to global memory is a whole row of the
//    tile (512 or 256 bytes), and the operand of the next step (coefficients in, bf16 products out) is formed on the way: the packing
//    pass disappears.  (Finished in the accumulator's own layout, a lane per column with 64-byte stores of bf16: 0.27 us a row and CTA.)
//  * clusters hand a row tile's operand on through L2: a CTA's producer waits until the column tiles of its units have counted the
//    step (red.release / ld.acquire, then the TMA loads).
//  * lane groups are not ordered against one another, but for a C-step: before its results are stored, the tiles of the rows that
//    started from what they replace have counted their first step, in front of which they read it (both as that step's operand and
//    as its incoming rows).  No step in front of the C-step waits for another group, so these counts always come.
// A lane group of clusters covers all columns and takes every `lanes`-th row tile.  All CTAs are resident (cooperative launch).
// The operand of step s + 1 goes to the buffer that step s - 1 was read from: its writer holds sums of step s, which every slice
// of every column tile of step s - 1 went into.
//
// Warps: 0 = TMA producer, 1 = MMA issuer and TMEM owner, 2..9 = epilogue.  Every wait is bounded; a CTA whose wait ran out skips to
// the closing cluster barrier, behind its own loads and products in flight.
#pragma once
#include "umma_cell.cuh"
#include "umma_split.cuh"

namespace mg {
namespace umma {

struct AdjSweepK {
  AdjSweepArgs q;
  __nv_bfloat16* op[2];           // operand buffers [rows][3H]
  int* ctr;                       // [row tiles][column tiles]
  int mt, ncol, lanes;
};

template <int NR, int S> struct AdjSweepCfg {
  static constexpr int RPC = NR / S, QUADS = RPC / 4;            // rows a CTA finishes, in groups of four: a warp's share at a time
  static constexpr int EW = 8, AW = QUADS < EW ? QUADS : EW, QW = QUADS / AW;      // epilogue warps; those that finish rows; groups each
  static constexpr int RPT = NR * 4 / EW;                        // accumulator columns (rows) a warp reads
  // a stage: one unit block of the operand, three gates.  (With a stage per box the loops that issue were the bound, not the tensor
  // pipe: 490 cycles a box for four MMAs of 64.)
  static constexpr int kBoxBytes = NR * BK * 2, kStageBytes = 3 * kBoxBytes, kStages = NR == 128 ? 3 : 7;
  static constexpr int kExBytes = NR * 512;                      // partial sums [producer][row / 4][column % 4][column / 4][4 rows]
  static constexpr int kWBytes = BM * BK * 2, kWSlots = 12;      // the weights pass through the same memory, in boxes of 128 columns
  static constexpr int kData = kStages * kStageBytes + kExBytes;
  static constexpr int kSmemBytes = kData + 1024 + 512;
  static_assert(kThreads == 64 + 32 * EW && QUADS % AW == 0 && kSmemBytes + 1024 <= 232448 && kData >= kWSlots * kWBytes, "sweep shape");
};

__device__ __forceinline__ void mma_bf16_ts(uint32_t d_tmem, uint32_t a_tmem, uint64_t bdesc, uint32_t idesc, uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n\t}"
      ::"r"(d_tmem), "r"(a_tmem), "l"(bdesc), "r"(idesc), "r"(accumulate)
      : "memory");
}
__device__ __forceinline__ void tmem_st32(uint32_t taddr, const uint32_t* r) {
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x32.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31,%32};"
      ::"r"(taddr), "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]), "r"(r[8]), "r"(r[9]), "r"(r[10]),
      "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15]), "r"(r[16]), "r"(r[17]), "r"(r[18]), "r"(r[19]), "r"(r[20]), "r"(r[21]),
      "r"(r[22]), "r"(r[23]), "r"(r[24]), "r"(r[25]), "r"(r[26]), "r"(r[27]), "r"(r[28]), "r"(r[29]), "r"(r[30]), "r"(r[31])
      : "memory");
}
// 16 bytes into a peer's shared memory, counted by the peer's barrier
__device__ __forceinline__ void st_async16(uint32_t addr, uint32_t bar, const float* v) {
  asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.v4.f32 [%0], {%2,%3,%4,%5}, [%1];"
               ::"r"(addr), "r"(bar), "f"(v[0]), "f"(v[1]), "f"(v[2]), "f"(v[3]) : "memory");
}
// bounded wait on a barrier that other CTAs of the cluster signal
__device__ __forceinline__ bool mbar_wait_cluster(uint32_t bar, uint32_t parity, volatile int* abort_flag, int* status, int code) {
  uint64_t t0 = 0;
  uint32_t spins = 0;
  while (true) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.b32 %0, 1, 0, p;\n\t}"
        : "=r"(ok) : "r"(bar), "r"(parity) : "memory");
    if (ok) return true;
    if ((++spins & 63u) == 0) {
      if (*abort_flag) return false;
      const uint64_t t = global_ns();
      if (t0 == 0) t0 = t;
      if (t - t0 > kWaitLimitNs) { *abort_flag = 1; atomicCAS(status, 0, code); return false; }
    }
  }
}
// bounded wait for the CTA's own loads and products when a launch ends, whether a wait ran out before or not
__device__ __forceinline__ void mbar_drain(uint32_t bar, uint32_t parity) {
  const uint64_t t0 = global_ns();
  while (!mbar_try(bar, parity))
    if (global_ns() - t0 > kWaitLimitNs) return;
}
// element k * ks + off of rows: strides fit 32 bits (checked by the host), so an address is two multiply-adds
template <class T> __device__ __forceinline__ T* at(T* base, int k, int ks, int off) { return base + ((i64)k * ks + off); }
__device__ __forceinline__ float4 ld_f4(const float* p) {      // (rows that this launch writes too: not through the read-only path)
  float4 v;
  asm volatile("ld.global.v4.f32 {%0,%1,%2,%3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ float4 lds_f4(uint32_t a) {
  float4 v;
  asm volatile("ld.shared.v4.f32 {%0,%1,%2,%3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "r"(a) : "memory");
  return v;
}
__device__ __forceinline__ float4 add4f(float4 a, float4 b) { return make_float4(a.x + b.x, a.y + b.y, a.z + b.z, a.w + b.w); }
// four bf16 coefficients times four fp32 values, as bf16
__device__ __forceinline__ uint2 scale4(uint2 c, float4 v) {
  const __nv_bfloat162 lo = __floats2bfloat162_rn(__uint_as_float(c.x << 16) * v.x, __uint_as_float(c.x & 0xffff0000u) * v.y);
  const __nv_bfloat162 hi = __floats2bfloat162_rn(__uint_as_float(c.y << 16) * v.z, __uint_as_float(c.y & 0xffff0000u) * v.w);
  return make_uint2(*reinterpret_cast<const uint32_t*>(&lo), *reinterpret_cast<const uint32_t*>(&hi));
}

template <int NR, int S>
__global__ void __launch_bounds__(kThreads, 1)
umma_adj_sweep_kernel(const __grid_constant__ CUtensorMap tm0, const __grid_constant__ CUtensorMap tm1, const __grid_constant__ CUtensorMap tmW,
                      const __grid_constant__ AdjSweepK p, int* status) {
  using C = AdjSweepCfg<NR, S>;
  constexpr int RPC = C::RPC, RPT = C::RPT, EW = C::EW, AW = C::AW, QW = C::QW;
  extern __shared__ uint8_t smem_raw[];
  const uint32_t tiles_base = (smem_u32(smem_raw) + 1023u) & ~1023u;
  const uint32_t ex_base = tiles_base + C::kStages * C::kStageBytes, bars = tiles_base + C::kData;
  auto full_bar = [&](int s) { return bars + 8u * s; };
  auto empty_bar = [&](int s) { return bars + 8u * (C::kStages + s); };
  auto tfull_bar = [&](int a) { return bars + 8u * (2 * C::kStages + a); };
  auto tempty_bar = [&](int a) { return bars + 8u * (2 * C::kStages + 2 + a); };
  const uint32_t xfull = bars + 8u * (2 * C::kStages + 4), xempty = xfull + 8u, wfull = xfull + 16u, mma_done = xfull + 24u;
  __shared__ uint32_t tmem_base_smem;
  __shared__ int abort_flag;

  const AdjSweepArgs& q = p.q;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int rank = (int)cluster_ctarank(), cid = blockIdx.x / S, group = cid / p.ncol, ct = cid - group * p.ncol;
  const int H = q.H, B = q.B, nb = H / 64, b0 = nb * rank / S, b1 = nb * (rank + 1) / S;
  // tensor memory: one or two accumulators of NR columns, then the weights (room for the largest share of any CTA)
  const int wmax = 3 * ((nb + S - 1) / S) * 32, accs = wmax + 2 * NR <= 512 ? 2 : 1, wcol = accs * NR;

  if (threadIdx.x == 0) {
    abort_flag = 0;
    for (int s = 0; s < C::kStages; ++s) { mbar_init(full_bar(s), 1); mbar_init(empty_bar(s), 1); }
    for (int a = 0; a < 2; ++a) { mbar_init(tfull_bar(a), 1); mbar_init(tempty_bar(a), EW); }
    mbar_init(xfull, 1);
    mbar_init(xempty, AW * S);
    mbar_init(wfull, 1);
    mbar_init(mma_done, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    mbar_expect_tx(wfull, (uint32_t)(3 * (b1 - b0) * C::kWBytes));
    for (int x = 0; x < 3 * (b1 - b0); ++x) tma_load_2d(tiles_base + x * C::kWBytes, &tmW, wfull, (x % 3) * H + (b0 + x / 3) * 64, ct * 128);
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_base_smem)), "r"(512u) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = tmem_base_smem;
  volatile int* abortp = &abort_flag;

  // epilogue warps: finished are rows of four, each lane columns [c0, c0 + 4)
  const int quarter = warp & 3, ew = warp - 2, c0 = ct * 128 + lane * 4;
  const bool col = c0 < H;
  struct Rows { float4 l[4], a[4], g[4]; uint2 cr[4], cz[4], cn[4]; };
  auto ld_c = [](const __nv_bfloat16* p) { return __ldg(reinterpret_cast<const uint2*>(p)); };
  auto put_operand = [&](__nv_bfloat16* op, int r, float4 carry, uint2 cr, uint2 cz, uint2 cn) {
    __nv_bfloat16* d = op + (i64)r * (3 * H) + c0;
    *reinterpret_cast<uint2*>(d) = scale4(cr, carry);
    *reinterpret_cast<uint2*>(d + H) = scale4(cz, carry);
    *reinterpret_cast<uint2*>(d + 2 * H) = scale4(cn, carry);
  };
  auto count = [&](int m) {      // (the stores of the warp's lanes are ordered in front of this lane's release)
    __syncwarp();
    if (lane == 0) asm volatile("red.release.gpu.global.add.s32 [%0], 1;" ::"l"(p.ctr + m * p.ncol + ct) : "memory");
  };
  auto first_row = [&](int m, int j) { return m * NR + rank * RPC + (ew * QW + j) * 4; };
  // incoming rows, a, sources (step s) and the coefficients of the next step; s < 0: what the first operand is made of
  auto load = [&](int s, int r0, Rows& o) {
    const AdjSweepStep& t = q.st[s < 0 ? 0 : s];
    const AdjSweepStep& nx = q.st[s + 1 < q.n ? s + 1 : s];
    const int M = t.nk * B, Mn = s + 1 < q.n ? nx.nk * B : 0, c_ks = (int)q.coef_ks;
    const float* const in = s > 0 ? q.st[s - 1].out : q.lin;
    const int in_ks = (int)(s > 0 ? q.st[s - 1].out_ks : q.lin_ks);
    const float* const gp = t.g;
    const int g_ks = (int)t.g_ks;
    int k = r0 / B, b = r0 - k * B;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int bo = b * H + c0;
      if (col && r0 + i < M) {
        o.l[i] = ld_f4(at(in, k, in_ks, bo));
        if (s >= 0) {
          o.a[i] = ld_f4(at(q.a + t.coff, k, c_ks, bo));
          o.g[i] = gp ? ld_f4(at(gp, k, g_ks, bo)) : make_float4(0.f, 0.f, 0.f, 0.f);
        }
      }
      if (col && r0 + i < Mn) {
        o.cr[i] = ld_c(at(q.cr + nx.coff, k, c_ks, bo)); o.cz[i] = ld_c(at(q.cz + nx.coff, k, c_ks, bo)); o.cn[i] = ld_c(at(q.cn + nx.coff, k, c_ks, bo));
      }
      if (++b == B) { b = 0; ++k; }
    }
  };
  auto join = [&](const AdjSweepStep& t, int r0, float4 (&v)[4]) {      // stacked layers: rows that join the incoming ones
    int k = r0 / B, b = r0 - k * B;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      if (col && r0 + i < t.nk * B) v[i] = add4f(v[i], ld_f4(at(t.ladd, k, (int)t.ladd_ks, b * H + c0)));
      if (++b == B) { b = 0; ++k; }
    }
  };
  // The rows that started from what rows r0 .. r0 + 3 replace are `ahead` behind them, in at most two tiles: a lane polls for each.
  auto starts_read = [&](int r0, int M, int ahead) {
    int lo, hi;
    tiles_ahead(r0, M, ahead, NR, &lo, &hi);
    const int mine = lo + lane;
    bool done = true;
    if (mine <= hi && mine < p.mt) done = sweep_wait(p.ctr + mine * p.ncol + ct, 2 * AW * S, abortp, status, 68);
    done = __all_sync(0xffffffffu, done);
    __syncwarp();      // (orders what the polling lanes acquired in front of every lane's stores)
    return done;
  };
  bool ok = true;
  if (warp >= 2) {
    // the operand of the first step, while the weights arrive
    if (ew < AW) {
      for (int m = group; m < p.mt; m += p.lanes) {
#pragma unroll 1
        for (int j = 0; j < QW; ++j) {
          const int r0 = first_row(m, j);
          Rows o;
          load(-1, r0, o);
          if (q.st[0].ladd) join(q.st[0], r0, o.l);
#pragma unroll
          for (int i = 0; i < 4; ++i)
            if (col && r0 + i < q.st[0].nk * B) put_operand(p.op[0], r0 + i, o.l[i], o.cr[i], o.cz[i], o.cn[i]);
        }
        count(m);
      }
    }
    // the weights -> tensor memory
    ok = __all_sync(0xffffffffu, mbar_wait(wfull, 0u, abortp, status, 60));
    if (ok) {
      const int row = quarter * 32 + lane;
      const uint32_t w0 = tmem_base + ((uint32_t)(quarter * 32) << 16) + (uint32_t)wcol;
      for (int x = ew >> 2; x < 3 * (b1 - b0); x += EW / 4) {
        uint32_t r[32];
#pragma unroll
        for (int i = 0; i < 8; ++i)
          asm volatile("ld.shared.v4.u32 {%0,%1,%2,%3}, [%4];" : "=r"(r[4 * i]), "=r"(r[4 * i + 1]), "=r"(r[4 * i + 2]), "=r"(r[4 * i + 3])
                       : "r"(tiles_base + (uint32_t)(x * C::kWBytes + row * 128 + ((i ^ (row & 7)) << 4))) : "memory");
        tmem_st32(w0 + (uint32_t)x * 32u, r);
      }
      asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");      // (TMA writes the same memory next)
  }
  __syncthreads();
  cluster_sync_all();      // every CTA of the cluster is past its weights before anything is written into its shared memory
  tc_fence_after();

  if (warp == 0) {
    // ------------------------------------------------------------ producer: the operand rows of this CTA's units (a lane polls for
    // each column tile that they come from)
    int stage = 0, loads = 0; uint32_t phase = 0;
    const int first_ct = b0 >> 1, cts = ((b1 - 1) >> 1) - first_ct + 1;
    for (int s = 0; s < q.n && ok; ++s) {
      const CUtensorMap* tm = (s & 1) ? &tm1 : &tm0;
      for (int m = group; m < p.mt && ok; m += p.lanes) {
        if (lane < cts) ok = sweep_wait(p.ctr + m * p.ncol + first_ct + lane, AW * S * (s + 1), abortp, status, 61);
        ok = __all_sync(0xffffffffu, ok);
        __syncwarp();      // (a vote orders no memory: what the polling lanes acquired comes before lane 0's loads by this barrier)
        for (int ub = b0; ub < b1 && ok; ++ub) {
          ok = __all_sync(0xffffffffu, mbar_wait(empty_bar(stage), phase ^ 1u, abortp, status, 62));
          if (!ok) break;
          if (lane == 0) {
            asm volatile("fence.proxy.async;" ::: "memory");
            mbar_expect_tx(full_bar(stage), C::kStageBytes);
#pragma unroll
            for (int g = 0; g < 3; ++g) tma_load_2d(tiles_base + stage * C::kStageBytes + g * C::kBoxBytes, tm, full_bar(stage), g * H + ub * 64, m * NR);
          }
          __syncwarp();
          ++loads;
          if (++stage == C::kStages) { stage = 0; phase ^= 1u; }
        }
      }
    }
    if (lane == 0) {      // (after an aborted loop too, nothing leaves before its loads have landed)
      mbar_drain(wfull, 0u);
      for (int x = loads > C::kStages ? loads - C::kStages : 0; x < loads; ++x) mbar_drain(full_bar(x % C::kStages), (uint32_t)(x / C::kStages) & 1u);
    }
    __syncwarp();
  } else if (warp == 1) {
    // ------------------------------------------------------------ MMA issuer
    if (lane == 0) {
      constexpr uint32_t idesc = instr_desc_bf16(NR);
      int stage = 0, it = 0; uint32_t phase = 0;
      for (int s = 0; s < q.n && ok; ++s)
        for (int m = group; m < p.mt && ok; m += p.lanes, ++it) {
          const int as = accs == 2 ? it & 1 : 0;
          const uint32_t aphase = (uint32_t)(accs == 2 ? it >> 1 : it) & 1u;
          if (!mbar_wait(tempty_bar(as), aphase ^ 1u, abortp, status, 63)) { ok = false; break; }
          tc_fence_after();
          for (int x = 0; x < b1 - b0; ++x) {
            if (!mbar_wait(full_bar(stage), phase, abortp, status, 64)) { ok = false; break; }
            tc_fence_after();
#pragma unroll
            for (int g = 0; g < 3; ++g) {
              const uint64_t bdesc = smem_desc_sw128(tiles_base + stage * C::kStageBytes + g * C::kBoxBytes);
#pragma unroll
              for (int k = 0; k < BK / 16; ++k)
                mma_bf16_ts(tmem_base + (uint32_t)(as * NR), tmem_base + (uint32_t)(wcol + (3 * x + g) * 32 + k * 8), bdesc + (uint64_t)(k * 2), idesc,
                            (x | g | k) != 0 ? 1u : 0u);
            }
            mma_commit(empty_bar(stage));
            if (++stage == C::kStages) { stage = 0; phase ^= 1u; }
          }
          if (ok) mma_commit(tfull_bar(as));
        }
      mma_commit(mma_done);
      mbar_drain(mma_done, 0u);
    }
    __syncwarp();
  } else {
    // ------------------------------------------------------------ epilogue
    int it = 0;
    for (int s = 0; s < q.n && ok; ++s) {
      const AdjSweepStep& t = q.st[s];
      const AdjSweepStep& nx = q.st[s + 1 < q.n ? s + 1 : s];
      const int M = t.nk * B, Mn = s + 1 < q.n ? nx.nk * B : 0, out_ks = (int)t.out_ks;
      for (int m = group; m < p.mt && ok; m += p.lanes, ++it) {
        const int as = accs == 2 ? it & 1 : 0;
        const uint32_t aphase = (uint32_t)(accs == 2 ? it >> 1 : it) & 1u, xphase = (uint32_t)it & 1u;
        Rows o;
        if (ew < AW) load(s, first_row(m, 0), o);
        if (threadIdx.x == 64) mbar_expect_tx(xfull, (uint32_t)C::kExBytes);
        ok = mbar_wait(tfull_bar(as), aphase, abortp, status, 65);
        ok = ok && mbar_wait_cluster(xempty, xphase ^ 1u, abortp, status, 66);      // the owners have read the previous tile's sums
        ok = __all_sync(0xffffffffu, ok);
        if (!ok) break;
        tc_fence_after();
        {
          // this warp's rows [part, part + RPT) of the tile, up to 32 of one owner at a time
          constexpr int STEP = RPT < RPC ? (RPT < 32 ? RPT : 32) : (RPC < 32 ? RPC : 32);
          const int part = (ew >> 2) * RPT;
          const uint32_t taddr = tmem_base + ((uint32_t)(quarter * 32) << 16) + (uint32_t)(as * NR + part);
          const uint32_t slot = (uint32_t)((lane & 3) * 32 + quarter * 8 + (lane >> 2)) * 16u;
#pragma unroll
          for (int c = 0; c < RPT; c += STEP) {
            float v[STEP];
            tmem_ld_n<STEP>(taddr + (uint32_t)c, v);
            tmem_wait_n<STEP>(v);
            const int to = (part + c) / RPC, rr = (part + c) % RPC;
            const uint32_t dst = mapa_shared(ex_base + (uint32_t)(rank * RPC + rr) * 512u + slot, (uint32_t)to);
            const uint32_t bar = mapa_shared(xfull, (uint32_t)to);
#pragma unroll
            for (int i = 0; i < STEP; i += 4) st_async16(dst + (uint32_t)i * 512u, bar, v + i);
          }
        }
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(tempty_bar(as));
        if (ew >= AW) continue;
        ok = mbar_wait_cluster(xfull, xphase, abortp, status, 67);
        ok = __all_sync(0xffffffffu, ok);
        if (!ok) break;
#pragma unroll
        for (int j = 0; j < QW; ++j) {
          const int r0 = first_row(m, j);
          if (j > 0) load(s, r0, o);
          if (t.ladd) join(t, r0, o.l);
          float4 v[4];      // by row; sums in rank order
#pragma unroll
          for (int i = 0; i < 4; ++i) v[i] = make_float4(0.f, 0.f, 0.f, 0.f);
          const uint32_t src = ex_base + (uint32_t)((ew * QW + j) * 4) * 512u + (uint32_t)lane * 16u;
#pragma unroll
          for (int pr = 0; pr < S; ++pr) {
            const uint32_t sp = src + (uint32_t)(pr * RPC) * 512u;
            const float4 x = lds_f4(sp), y = lds_f4(sp + 512u), z = lds_f4(sp + 1024u), w = lds_f4(sp + 1536u);
            v[0] = add4f(v[0], make_float4(x.x, y.x, z.x, w.x)); v[1] = add4f(v[1], make_float4(x.y, y.y, z.y, w.y));
            v[2] = add4f(v[2], make_float4(x.z, y.z, z.z, w.z)); v[3] = add4f(v[3], make_float4(x.w, y.w, z.w, w.w));
          }
          if (j == QW - 1) {
            __syncwarp();
            if (lane < S) mbar_arrive_cluster(mapa_shared(xempty, (uint32_t)lane));
          }
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            const float4 u = make_float4(o.a[i].x * o.l[i].x + v[i].x, o.a[i].y * o.l[i].y + v[i].y, o.a[i].z * o.l[i].z + v[i].z, o.a[i].w * o.l[i].w + v[i].w);
            v[i] = add4f(u, o.g[i]);
          }
          if (Mn > 0) {      // the operand first: it is what the other clusters wait for
            float4 cy[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) cy[i] = v[i];
            if (nx.ladd) join(nx, r0, cy);
#pragma unroll
            for (int i = 0; i < 4; ++i)
              if (col && r0 + i < Mn) put_operand(p.op[(s + 1) & 1], r0 + i, cy[i], o.cr[i], o.cz[i], o.cn[i]);
          }
          if (j == QW - 1 && s + 1 < q.n) count(m);
          if (t.ahead > 0 && ok) ok = starts_read(r0, M, t.ahead);
          if (!ok) continue;
          int k = r0 / B, b = r0 - k * B;
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            if (col && r0 + i < M) *reinterpret_cast<float4*>(at(t.out, k, out_ks, b * H + c0)) = v[i];
            if (++b == B) { b = 0; ++k; }
          }
        }
      }
    }
    __syncwarp();
  }

  // ------------------------------------------------------------ teardown: nobody leaves while a peer may still signal it
  tc_fence_before();
  __syncthreads();
  cluster_sync_all();
  if (abort_flag != 0) {      // partial sums of peers may still be on their way to a CTA that stopped waiting for them
    const uint64_t t0 = global_ns();
    while (global_ns() - t0 < 100000) __nanosleep(1000);
  }
  tc_fence_after();
  if (warp == 1) {
    __syncwarp();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(512u) : "memory");
  }
}

}  // namespace umma
}  // namespace mg
