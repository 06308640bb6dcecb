// Few-row product with the reduction split over a thread-block cluster, sm_100a:
//
//   D[m, n] = sum_k A[m, k] * B[n, k]        A: [M, K] bf16 row-major, B: [N, K] bf16 row-major
//
// A step with few rows has too few output tiles to fill the SMs, and one CTA per tile is bound by what it can take in (about
// 130 GB/s): a 512-row adjoint step at H = 1024 (K = 3072) streamed 1.2 MB per CTA through 64 CTAs in 16.6 us.  Here the S CTAs of
// a cluster reduce K / S each for the SAME 128 x BN tile; every CTA then sends the columns it does not finish to their owner's
// shared memory (BN / S columns per CTA) and finishes its own slice, adding the S partial sums in rank order (the same bits on
// every run).  The epilogue's operands are requested before the main loop ends.  Measured: see pick_split().
//
// One tile per cluster.  Warps as in the plain product: 0 = TMA producer, 1 = MMA issuer and TMEM owner, 2..9 = epilogue (two
// threads per row, BN / (2 S) columns each).  Every wait on an mbarrier is bounded; a CTA whose wait ran out still takes part in
// the cluster barriers.
#pragma once
#include "umma_gemm_pair.cuh"

namespace mg {
namespace umma {

template <int BN, int S> struct SplitCfg {
  static constexpr int kW = BN / S, kNW = kW / 2;                    // columns a CTA finishes; per thread
  static constexpr int kStageBytes = BM * BK * 2 + BN * BK * 2;
  // exchange buffer [producer][four columns][row]: the lanes of a warp (32 rows) write 512 contiguous bytes of a peer's memory
  static constexpr int kExBytes = S * BM * kW * 4;
  static constexpr int kStages = (220 * 1024 - kExBytes) / kStageBytes > 6 ? 6 : (220 * 1024 - kExBytes) / kStageBytes;
  static constexpr int kSmemBytes = kStages * kStageBytes + kExBytes + 1024 + 256;
  static_assert(kNW >= 4 && kSmemBytes + 512 <= 232448, "split shape");
};

template <int N> __device__ __forceinline__ void tmem_ld_n(uint32_t taddr, float* v) {
  if constexpr (N == 4) {
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0,%1,%2,%3}, [%4];" : "=f"(v[0]), "=f"(v[1]), "=f"(v[2]), "=f"(v[3]) : "r"(taddr));
  } else if constexpr (N == 8) {
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
                 : "=f"(v[0]), "=f"(v[1]), "=f"(v[2]), "=f"(v[3]), "=f"(v[4]), "=f"(v[5]), "=f"(v[6]), "=f"(v[7]) : "r"(taddr));
  } else {
    tmem_ld_n<8>(taddr, v);
    tmem_ld_n<N - 8>(taddr + 8, v + 8);
  }
}
// the wait that makes loaded accumulator values usable, tied to the registers so that no use can move in front of it
template <int N> __device__ __forceinline__ void tmem_wait_n(float* v) {
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
  for (int i = 0; i < N; ++i) asm volatile("" : "+f"(v[i])::"memory");
}

// Epi: Ops ops; load(row, n, ops) requests the operands of NW columns from n on; finish(row, n, v, ops) stores
template <int BN, int S, class Epi>
__global__ void __launch_bounds__(kThreads, 1)
umma_split_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB, int N, int K, Epi epi, int* status) {
  using C = SplitCfg<BN, S>;
  constexpr int NW = C::kNW, W = C::kW;
  extern __shared__ uint8_t smem_raw[];
  const uint32_t raw = smem_u32(smem_raw);
  const uint32_t tiles_base = (raw + 1023u) & ~1023u;
  const uint32_t ex_base = tiles_base + C::kStages * C::kStageBytes;
  const uint32_t bars = ex_base + C::kExBytes;
  auto full_bar = [&](int s) { return bars + 8u * s; };
  auto empty_bar = [&](int s) { return bars + 8u * (C::kStages + s); };
  const uint32_t tfull = bars + 8u * (2 * C::kStages);
  __shared__ uint32_t tmem_base_smem;
  __shared__ int abort_flag;

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int rank = (int)cluster_ctarank(), tile = blockIdx.x / S, n_tiles = (N + BN - 1) / BN, mt = tile / n_tiles, nt = tile % n_tiles;
  const int k_blocks = (K + BK - 1) / BK, kb0 = k_blocks * rank / S, kb1 = k_blocks * (rank + 1) / S;

  if (threadIdx.x == 0) {
    abort_flag = 0;
    for (int s = 0; s < C::kStages; ++s) { mbar_init(full_bar(s), 1); mbar_init(empty_bar(s), 1); }
    mbar_init(tfull, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_base_smem)), "r"((uint32_t)BN) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  cluster_sync_all();      // every CTA of the cluster runs before anything is written into its shared memory
  tc_fence_after();
  const uint32_t tmem_base = tmem_base_smem;
  volatile int* abortp = &abort_flag;
  pdl_wait();
  pdl_trigger();

  typename Epi::Ops ops;
  float mine[NW];
  const int q = warp & 3, half = (warp - 2) >> 2, r = q * 32 + lane;        // epilogue warps: TMEM lane quarter, half of a slice, row of the tile
  const int row = mt * BM + r, n = nt * BN + rank * W + half * NW;
  if (warp == 0) {
    if (lane == 0) {
      int stage = 0; uint32_t phase = 0;
      for (int kb = kb0; kb < kb1; ++kb) {
        if (!mbar_wait(empty_bar(stage), phase ^ 1u, abortp, status, 51)) break;
        const uint32_t a_dst = tiles_base + stage * C::kStageBytes;
        mbar_expect_tx(full_bar(stage), C::kStageBytes);
        tma_load_2d(a_dst, &tmA, full_bar(stage), kb * BK, mt * BM);
        tma_load_2d(a_dst + BM * BK * 2, &tmB, full_bar(stage), kb * BK, nt * BN);
        if (++stage == C::kStages) { stage = 0; phase ^= 1u; }
      }
    }
    __syncwarp();
  } else if (warp == 1) {
    if (lane == 0) {
      constexpr uint32_t idesc = instr_desc_bf16(BN);
      int stage = 0; uint32_t phase = 0; bool ok = true;
      for (int kb = kb0; kb < kb1; ++kb) {
        if (!mbar_wait(full_bar(stage), phase, abortp, status, 52)) { ok = false; break; }
        tc_fence_after();
        const uint32_t a_src = tiles_base + stage * C::kStageBytes;
        const uint64_t adesc = smem_desc_sw128(a_src), bdesc = smem_desc_sw128(a_src + BM * BK * 2);
#pragma unroll
        for (int k = 0; k < BK / 16; ++k) mma_bf16(tmem_base, adesc + (uint64_t)(k * 2), bdesc + (uint64_t)(k * 2), idesc, ((kb - kb0) | k) != 0 ? 1u : 0u);
        mma_commit(empty_bar(stage));
        if (++stage == C::kStages) { stage = 0; phase ^= 1u; }
      }
      if (ok) mma_commit(tfull);
    }
    __syncwarp();
  } else {
    epi.load(row, n, ops);
    bool ok = mbar_wait(tfull, 0u, abortp, status, 53);
    ok = __all_sync(0xffffffffu, ok);
    tc_fence_after();
    if (ok) {
      const uint32_t taddr = tmem_base + ((uint32_t)(q * 32) << 16) + (uint32_t)(half * NW);
      const uint32_t dst = ex_base + (uint32_t)((rank * (W / 4) + half * (NW / 4)) * BM + r) * 16u;
#pragma unroll
      for (int p = 0; p < S; ++p) {
        float v[NW];
        tmem_ld_n<NW>(taddr + p * W, v);
        tmem_wait_n<NW>(v);
        if (p == rank) {
#pragma unroll
          for (int i = 0; i < NW; ++i) mine[i] = v[i];
        } else {
          const uint32_t d = mapa_shared(dst, (uint32_t)p);
#pragma unroll
          for (int i = 0; i < NW; i += 4)
            asm volatile("st.shared::cluster.v4.f32 [%0], {%1,%2,%3,%4};" ::"r"(d + (uint32_t)(i / 4) * (BM * 16u)), "f"(v[i]), "f"(v[i + 1]), "f"(v[i + 2]), "f"(v[i + 3]) : "memory");
        }
      }
    }
    __syncwarp();
  }
  tc_fence_before();
  cluster_sync_all();      // every partial sum has arrived
  if (warp >= 2 && abort_flag == 0) {
    float v[NW];
#pragma unroll
    for (int i = 0; i < NW; ++i) v[i] = 0.f;
#pragma unroll
    for (int p = 0; p < S; ++p) {
      const uint32_t src = ex_base + (uint32_t)((p * (W / 4) + half * (NW / 4)) * BM + r) * 16u;
#pragma unroll
      for (int i = 0; i < NW; i += 4) {
        float4 t;
        if (p == rank) t = make_float4(mine[i], mine[i + 1], mine[i + 2], mine[i + 3]);
        else asm volatile("ld.shared.v4.f32 {%0,%1,%2,%3}, [%4];" : "=f"(t.x), "=f"(t.y), "=f"(t.z), "=f"(t.w) : "r"(src + (uint32_t)(i / 4) * (BM * 16u)));
        v[i] += t.x; v[i + 1] += t.y; v[i + 2] += t.z; v[i + 3] += t.w;
      }
    }
    epi.finish(row, n, v, ops);
  }
  __syncthreads();
  tc_fence_after();
  if (warp == 1) {
    __syncwarp();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"((uint32_t)BN) : "memory");
  }
}

}  // namespace umma
}  // namespace mg
