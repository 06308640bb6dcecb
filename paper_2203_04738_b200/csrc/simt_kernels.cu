// fp32 FFMA engine: one tiled GEMM skeleton with operand-loader and epilogue functors.
// Used when cfg.operands == MGRIT_OPERANDS_FP32 (the precision mode whose results must agree
// with the fp64 oracle to 1e-4), and for shapes the tensor-core engine does not cover.
#include "cell.cuh"

namespace mg {

namespace {

constexpr int BM = 32, BN = 32, BK = 32, NT = 256;

// C[m, (g, n)] = sum_k A(m, k) * B(g, n, k);  epi(m, n, acc[NG]).
// AKC / BKC: the loader's fastest index is k (operand stored K-contiguous) or the row/column.
template <int NG, bool AKC, bool BKC, class AL, class BL, class Epi>
__global__ void __launch_bounds__(NT) simt_gemm_kernel(int M, int N, int K, AL al, BL bl, Epi epi) {
  __shared__ float As[BK][BM + 1];
  __shared__ float Bs[NG][BK][BN + 1];
  const int tid = threadIdx.x;
  const int m0 = blockIdx.x * BM, n0 = blockIdx.y * BN;
  const int ty = tid / 16, tx = tid % 16;
  float acc[NG][2][2];
#pragma unroll
  for (int g = 0; g < NG; ++g) { acc[g][0][0] = acc[g][0][1] = acc[g][1][0] = acc[g][1][1] = 0.f; }

  for (int k0 = 0; k0 < K; k0 += BK) {
#pragma unroll
    for (int e = tid; e < BM * BK; e += NT) {
      int r, k;
      if (AKC) { r = e / BK; k = e % BK; } else { r = e % BM; k = e / BM; }
      int gr = m0 + r, gk = k0 + k;
      As[k][r] = (gr < M && gk < K) ? al(gr, gk) : 0.f;
    }
#pragma unroll
    for (int g = 0; g < NG; ++g) {
#pragma unroll
      for (int e = tid; e < BN * BK; e += NT) {
        int c, k;
        if (BKC) { c = e / BK; k = e % BK; } else { c = e % BN; k = e / BN; }
        int gc = n0 + c, gk = k0 + k;
        Bs[g][k][c] = (gc < N && gk < K) ? bl(g, gc, gk) : 0.f;
      }
    }
    __syncthreads();
#pragma unroll 8
    for (int k = 0; k < BK; ++k) {
      float a0 = As[k][ty], a1 = As[k][ty + 16];
#pragma unroll
      for (int g = 0; g < NG; ++g) {
        float b0 = Bs[g][k][tx], b1 = Bs[g][k][tx + 16];
        acc[g][0][0] = fmaf(a0, b0, acc[g][0][0]);
        acc[g][0][1] = fmaf(a0, b1, acc[g][0][1]);
        acc[g][1][0] = fmaf(a1, b0, acc[g][1][0]);
        acc[g][1][1] = fmaf(a1, b1, acc[g][1][1]);
      }
    }
    __syncthreads();
  }
#pragma unroll
  for (int i = 0; i < 2; ++i)
#pragma unroll
    for (int j = 0; j < 2; ++j) {
      int row = m0 + ty + 16 * i, col = n0 + tx + 16 * j;
      if (row < M && col < N) {
        float v[NG];
#pragma unroll
        for (int g = 0; g < NG; ++g) v[g] = acc[g][i][j];
        epi(row, col, v);
      }
    }
}

template <int NG, bool AKC, bool BKC, class AL, class BL, class Epi>
void launch(int kc, int M, int N, int K, AL al, BL bl, Epi epi, cudaStream_t s) {
  if (M <= 0 || N <= 0) return;
  dim3 grid((M + BM - 1) / BM, (N + BN - 1) / BN);
  prof_begin(kc, 2.0 * M * N * NG * K, s);
  simt_gemm_kernel<NG, AKC, BKC><<<grid, NT, 0, s>>>(M, N, K, al, bl, epi);
  prof_end(s);
  count_launch();
}

// ---------------------------------------------------------------- loaders
struct StridedRowsA {  // rows (k_, b): p + k_*ks + b*H
  const float* p; i64 ks; int B, H;
  __device__ float operator()(int m, int k) const { return p[(i64)(m / B) * ks + (i64)(m % B) * H + k]; }
};
struct GateW {  // B(g, n, k) = W[(g*H + n)*ld + k]
  const float* W; int H; i64 ld;
  __device__ float operator()(int g, int n, int k) const { return W[((i64)g * H + n) * ld + k]; }
};
struct DenseBT {  // B(0, n, k) = W[k*ld + n]
  const float* W; i64 ld;
  __device__ float operator()(int, int n, int k) const { return W[(i64)k * ld + n]; }
};
struct LinA {  // state entering forward step j = m/B + 1 of a level: h at fine time t0 + stride*(j-1)
  const float* h0; const float* h; i64 stride_t, t0; int B, H;
  __device__ float operator()(int m, int k) const {
    int j1 = m / B, b = m % B;
    const i64 t = t0 + (i64)j1 * stride_t;
    return t == 0 ? h0[(i64)b * H + k] : h[(t - 1) * B * H + (i64)b * H + k];
  }
};
struct AdjA {  // A[m, g*H + i] = c_g[m, i] * lam[m, i]
  const float* lin; i64 lin_ks; const float *cr, *cz, *cn; i64 coef_ks; int B, H;
  __device__ float operator()(int m, int k) const {
    int kk = m / B, b = m % B, g = k / H, i = k - g * H;
    const float* c = g == 0 ? cr : (g == 1 ? cz : cn);
    return c[(i64)kk * coef_ks + (i64)b * H + i] * lin[(i64)kk * lin_ks + (i64)b * H + i];
  }
};

// ---------------------------------------------------------------- epilogues
struct StoreEpi {
  float* out; i64 ld;
  __device__ void operator()(int m, int n, const float* v) const { out[(i64)m * ld + n] = v[0]; }
};
struct FwdEpi {
  FwdStepArgs a;
  __device__ void operator()(int m, int n, const float* v) const {
    int k = m / a.B, b = m % a.B;
    const float* gi = a.gi + (i64)k * a.gi_ks + (i64)b * 3 * a.H;
    float hp = a.hin[(i64)k * a.hin_ks + (i64)b * a.H + n];
    float phi = cell_forward(gi[n], gi[a.H + n], gi[2 * a.H + n], v[0] + a.b_hh[n], v[1] + a.b_hh[a.H + n],
                             v[2] + a.b_hh[2 * a.H + n], hp, a.gamma, a.cell);
    float* o = a.hout + (i64)k * a.hout_ks + (i64)b * a.H + n;
    if (a.mode == 0) {
      if (a.gadd) phi += a.gadd[(i64)k * a.gadd_ks + (i64)b * a.H + n];
      *o = phi;
    } else {
      *o = *o - phi;
    }
  }
};
struct LinEpi {
  LinArgs a;
  __device__ void operator()(int m, int n, const float* v) const {
    int j1 = m / a.B, b = m % a.B;
    const i64 t = a.t0 + (i64)j1 * a.stride_t;        // fine time the step leaves from
    const float* gi = a.gi + ((t + a.stride_t - 1) * a.B + b) * 3 * a.H;
    float hp = t == 0 ? a.h0[(i64)b * a.H + n] : a.h[((t - 1) * a.B + b) * a.H + n];
    CellLin c = cell_linearise(gi[n], gi[a.H + n], gi[2 * a.H + n], v[0] + a.b_hh[n], v[1] + a.b_hh[a.H + n],
                               v[2] + a.b_hh[2 * a.H + n], hp, a.gamma, a.cell);
    i64 o = (i64)m * a.H + n;
    a.a[o] = c.a; a.cr[o] = c.cr; a.cz[o] = c.cz; a.cn[o] = c.cn;
    if (a.cnp) a.cnp[o] = c.cnp;
  }
};
struct AdjEpi {
  AdjStepArgs a;
  __device__ void operator()(int m, int n, const float* v) const {
    int k = m / a.B, b = m % a.B;
    float lam = a.lin[(i64)k * a.lin_ks + (i64)b * a.H + n];
    float val = a.a[(i64)k * a.coef_ks + (i64)b * a.H + n] * lam + v[0];
    float* o = a.lout + (i64)k * a.lout_ks + (i64)b * a.H + n;
    if (a.mode == 0) {
      if (a.gadd) val += a.gadd[(i64)k * a.gadd_ks + (i64)b * a.H + n];
      *o = val;
    } else {
      *o = *o - val;
    }
  }
};

// ---------------------------------------------------------------- Implicit LSTM (four gates)
struct LstmFwdEpi {
  LstmFwdArgs a;
  __device__ void operator()(int m, int n, const float* v) const {
    int k = m / a.B, b = m % a.B;
    const float* gi = a.gi + (i64)k * a.gi_ks + (i64)b * 4 * a.H;
    float cp = a.cin[(i64)k * a.in_ks + (i64)b * a.H + n];
    LstmOut o = lstm_forward(gi[n], gi[a.H + n], gi[2 * a.H + n], gi[3 * a.H + n], v[0] + a.b_hh[n], v[1] + a.b_hh[a.H + n],
                             v[2] + a.b_hh[2 * a.H + n], v[3] + a.b_hh[3 * a.H + n], cp, a.gamma, a.cell);
    a.cout[(i64)m * a.H + n] = o.c;
    a.hout[(i64)m * a.H + n] = o.h;
  }
};
struct LstmLinA {   // hidden state entering step j = m/B + 1: h at fine time t0 + stride*(j-1)
  const float* h0; const float* h; i64 ts, stride_t, t0; int B, H;
  __device__ float operator()(int m, int k) const {
    int j1 = m / B, b = m % B;
    const i64 t = t0 + (i64)j1 * stride_t;
    return t == 0 ? h0[(i64)b * H + k] : h[(t - 1) * ts + (i64)b * H + k];
  }
};
struct LstmLinEpi {
  LstmLinArgs a;
  __device__ void operator()(int m, int n, const float* v) const {
    int j1 = m / a.B, b = m % a.B;
    const i64 t = a.t0 + (i64)j1 * a.stride_t;
    const float* gi = a.gi + ((t + a.stride_t - 1) * a.B + b) * 4 * a.H;
    float cp = t == 0 ? a.c0[(i64)b * a.H + n] : a.c[(t - 1) * a.ts + (i64)b * a.H + n];
    LstmLin L = lstm_linearise(gi[n], gi[a.H + n], gi[2 * a.H + n], gi[3 * a.H + n], v[0] + a.b_hh[n], v[1] + a.b_hh[a.H + n],
                               v[2] + a.b_hh[2 * a.H + n], v[3] + a.b_hh[3 * a.H + n], cp, a.gamma, a.cell);
    i64 o = (i64)m * a.H + n;
    a.a[o] = L.a; a.p[o] = L.p; a.ci[o] = L.ci; a.cf[o] = L.cf; a.cg[o] = L.cg; a.co[o] = L.co;
  }
};
struct LstmAdjA {   // A[m, g*H + i] = coefficient_g * (g < 3 ? Lc + p*Lh : Lh)
  LstmAdjArgs a;
  __device__ float operator()(int m, int k) const {
    int kk = m / a.B, b = m % a.B, g = k / a.H, i = k - g * a.H;
    i64 ci = (i64)kk * a.coef_ks + (i64)b * a.H + i, li = (i64)kk * a.in_ks + (i64)b * a.H + i;
    float lh = a.lh[li];
    if (g == 3) return a.co[ci] * lh;
    float dc = a.lc[li] + a.p[ci] * lh;
    return (g == 0 ? a.ci[ci] : (g == 1 ? a.cf[ci] : a.cg[ci])) * dc;
  }
};
__global__ void __launch_bounds__(256) lstm_adj_c_kernel(LstmAdjArgs a) {
  i64 total = (i64)a.M * a.H;
  for (i64 e = (i64)blockIdx.x * blockDim.x + threadIdx.x; e < total; e += (i64)gridDim.x * blockDim.x) {
    i64 m = e / a.H; int i = (int)(e % a.H);
    i64 kk = m / a.B; int b = (int)(m % a.B);
    i64 ci = kk * a.coef_ks + (i64)b * a.H + i, li = kk * a.in_ks + (i64)b * a.H + i;
    a.lc_out[e] = a.a[ci] * (a.lc[li] + a.p[ci] * a.lh[li]);
  }
}
__global__ void __launch_bounds__(256) lstm_form_dA_kernel(const float* __restrict__ lc, const float* __restrict__ lh, i64 lam_ts, int B,
                                                           const float* __restrict__ p, const float* __restrict__ ci,
                                                           const float* __restrict__ cf, const float* __restrict__ cg,
                                                           const float* __restrict__ co, float* __restrict__ dA, i64 M, int H) {
  i64 total = M * H;
  for (i64 e = (i64)blockIdx.x * blockDim.x + threadIdx.x; e < total; e += (i64)gridDim.x * blockDim.x) {
    i64 m = e / H; int i = (int)(e % H);
    i64 t = m / B; int b = (int)(m % B);
    i64 li = t * lam_ts + (i64)b * H + i;
    float h = lh[li], dc = lc[li] + p[e] * h;
    float* d = dA + m * 4 * H + i;
    d[0] = ci[e] * dc; d[H] = cf[e] * dc; d[2 * H] = cg[e] * dc; d[3 * H] = co[e] * h;
  }
}

// ---------------------------------------------------------------- 64 x 64 tiles: projection and the gradient pass
// C[m, n] = sum_k A(m, k) B(n, k) for products with many rows or a long reduction (input projection, weight and input
// gradients).  256 threads hold 4 x 4 sums each, operands come as 16-byte loads (along k where the operand is stored
// K-contiguous, else along its rows) one step ahead into registers and alternate between two shared buffers.  Bound by the FFMA
// rate (two 16-byte shared reads per 16 FFMA).  The reduction may be cut into grid.z ranges whose partial results a second
// kernel adds in range order: a weight gradient has few tiles and a reduction over all T*B rows, which used to run on a
// handful of SMs (four products of 312 x (16..104) over 12800 rows: 1139 us each; a whole two-layer step of that shape went
// from 9.18 to 4.80 ms on a B200).
// Two column sets (N0 and N1 columns, each with its own B operand) may share one launch; AL / BL / Epi get the set as `side`.
struct G64 { int M, N0, N1, K, kchunk; };
constexpr int kT64 = 64, kK64 = 16, kP64 = 68;
template <bool COLSUM, class AL, class BL, class Epi>
__global__ void __launch_bounds__(256) gemm64_kernel(G64 sh, AL al, BL bl, Epi epi) {
  __shared__ __align__(16) float As[2][kK64][kP64], Bs[2][kK64][kP64];
  const int tid = threadIdx.x, ty = tid / 16, tx = tid % 16;
  const int nt0 = (sh.N0 + kT64 - 1) / kT64, side = (int)blockIdx.y >= nt0 ? 1 : 0;
  const int m0 = blockIdx.x * kT64, n0 = ((int)blockIdx.y - side * nt0) * kT64, N = side ? sh.N1 : sh.N0;
  const int kb = blockIdx.z * sh.kchunk, ke = min(sh.K, kb + sh.kchunk);
  const bool colsum = COLSUM && n0 == 0;
  // this thread's 16 bytes of each operand tile
  const int ar = AL::KC ? tid / 4 : (tid % 16) * 4, ak = AL::KC ? (tid % 4) * 4 : tid / 16;
  const int br = BL::KC ? tid / 4 : (tid % 16) * 4, bk = BL::KC ? (tid % 4) * 4 : tid / 16;
  const bool aok = m0 + ar < sh.M, bok = n0 + br < N;
  const float4 zero = make_float4(0.f, 0.f, 0.f, 0.f);
  float4 ra = aok && kb + ak < ke ? al(m0 + ar, kb + ak, side) : zero, rb = bok && kb + bk < ke ? bl(n0 + br, kb + bk, side) : zero;
  float acc[4][4], cs[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
  for (int i = 0; i < 4; ++i) acc[i][0] = acc[i][1] = acc[i][2] = acc[i][3] = 0.f;
  auto put = [](float (*S)[kP64], bool kc, int r, int k, float4 v) {
    if (kc) { S[k][r] = v.x; S[k + 1][r] = v.y; S[k + 2][r] = v.z; S[k + 3][r] = v.w; }
    else *reinterpret_cast<float4*>(&S[k][r]) = v;
  };
  int buf = 0;
  for (int k0 = kb; k0 < ke; k0 += kK64, buf ^= 1) {
    put(As[buf], AL::KC, ar, ak, ra);
    put(Bs[buf], BL::KC, br, bk, rb);
    __syncthreads();
    const int kn = k0 + kK64;
    if (kn < ke) {
      ra = aok && kn + ak < ke ? al(m0 + ar, kn + ak, side) : zero;
      rb = bok && kn + bk < ke ? bl(n0 + br, kn + bk, side) : zero;
    }
#pragma unroll
    for (int k = 0; k < kK64; ++k) {
      const float4 a = *reinterpret_cast<const float4*>(&As[buf][k][ty * 4]), b = *reinterpret_cast<const float4*>(&Bs[buf][k][tx * 4]);
      const float av[4] = {a.x, a.y, a.z, a.w}, bv[4] = {b.x, b.y, b.z, b.w};
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j] = fmaf(av[i], bv[j], acc[i][j]);
      if (COLSUM) {
#pragma unroll
        for (int i = 0; i < 4; ++i) cs[i] += av[i];
      }
    }
  }
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int m = m0 + ty * 4 + i, n = n0 + tx * 4;
    if (m >= sh.M) continue;
    if (n < N) epi(m, n, make_float4(acc[i][0], acc[i][1], acc[i][2], acc[i][3]), side, (int)blockIdx.z);
    if (colsum && tx == 0) epi.sum(m, cs[i], side, (int)blockIdx.z);
  }
}
__device__ __forceinline__ float4 f4(const float* p) { return *reinterpret_cast<const float4*>(p); }
__device__ __forceinline__ float4 mul4(float4 a, float4 b) { return make_float4(a.x * b.x, a.y * b.y, a.z * b.z, a.w * b.w); }

struct RowK {      // X(r, k) = p[r*ld + k]
  static constexpr bool KC = true;
  const float* p; i64 ld;
  __device__ float4 operator()(int r, int k, int) const { return f4(p + (i64)r * ld + k); }
};
struct ColK {      // X(r, k) = p[k*ld + r]
  static constexpr bool KC = false;
  const float* p; i64 ld;
  __device__ float4 operator()(int r, int k, int) const { return f4(p + (i64)k * ld + r); }
};
// dA(row m, column g*H + i) = c_g[m, i] * lam[m, i], formed while it is loaded (it is never stored); side 1 takes c_n' for c_n
struct FormedDA {
  const float* lam; i64 lam_ts; const float *cr, *cz, *cn, *cnp; int B, H;
  __device__ float4 at(int m, int j, int side) const {
    const int g = j / H, i = j - g * H, t = m / B, b = m - t * B;
    const float* c = g == 0 ? cr : (g == 1 ? cz : (side ? cnp : cn));
    return mul4(f4(c + (i64)m * H + i), f4(lam + (i64)t * lam_ts + (i64)b * H + i));
  }
};
struct DenseDA {
  const float* p; i64 ld;
  __device__ float4 at(int m, int j, int) const { return f4(p + (i64)m * ld + j); }
};
template <class D> struct DaCols {      // weight gradients: A(m = column of dA, k = row)
  static constexpr bool KC = false;
  D d;
  __device__ float4 operator()(int r, int k, int side) const { return d.at(k, r, side); }
};
template <class D> struct DaRows {      // input gradient: A(m = row of dA, k = column), the input-side columns
  static constexpr bool KC = true;
  D d;
  __device__ float4 operator()(int r, int k, int) const { return d.at(r, k, 1); }
};
struct WgradB {    // side 0: h_{t-1} rows (the first Bf of them from h_0), side 1: x rows
  static constexpr bool KC = false;
  const float *first, *rest, *x; int Bf, H, I;
  __device__ float4 operator()(int r, int k, int side) const {
    if (side) return f4(x + (i64)k * I + r);
    return f4((k < Bf ? first + (i64)k * H : rest + (i64)(k - Bf) * H) + r);
  }
};
struct Bias64 {
  float* out; i64 ld; const float* bias;
  __device__ void operator()(int m, int n, float4 v, int, int) const {
    const float4 b = f4(bias + n);
    *reinterpret_cast<float4*>(out + (i64)m * ld + n) = make_float4(v.x + b.x, v.y + b.y, v.z + b.z, v.w + b.w);
  }
  __device__ void sum(int, float, int, int) const {}
};
struct Store64 {
  float* out; i64 ld;
  __device__ void operator()(int m, int n, float4 v, int, int) const { *reinterpret_cast<float4*>(out + (i64)m * ld + n) = v; }
  __device__ void sum(int, float, int, int) const {}
};
struct WgradOut {  // range z of the reduction: dW_hh, dW_ih and the bias sums at their base + z * zs
  float *hh, *ih, *bhh, *bih; int H, I; i64 zs;
  __device__ void operator()(int m, int n, float4 v, int side, int z) const {
    *reinterpret_cast<float4*>((side ? ih + (i64)m * I : hh + (i64)m * H) + z * zs + n) = v;
  }
  __device__ void sum(int m, float v, int side, int z) const { (side ? bih : bhh)[m + z * zs] = v; }
};
// The partial results [z][hh | ih | bhh | bih] added in range order (the same bits on every run).
__global__ void __launch_bounds__(256) reduce_parts_kernel(const float4* __restrict__ part, i64 zs4, int nz, i64 nhh, i64 nih, i64 nb, WgradOut o) {
  const i64 n = (nhh + nih + 2 * nb) / 4;
  for (i64 e = (i64)blockIdx.x * blockDim.x + threadIdx.x; e < n; e += (i64)gridDim.x * blockDim.x) {
    float4 s = part[e];
#pragma unroll 4
    for (int z = 1; z < nz; ++z) {
      const float4 v = part[z * zs4 + e];
      s.x += v.x; s.y += v.y; s.z += v.z; s.w += v.w;
    }
    const i64 i = e * 4;
    float* dst = i < nhh ? o.hh + i : i < nhh + nih ? o.ih + (i - nhh) : i < nhh + nih + nb ? o.bhh + (i - nhh - nih) : o.bih + (i - nhh - nih - nb);
    *reinterpret_cast<float4*>(dst) = s;
  }
}
// ranges of the T*B rows: about three blocks per SM, no range shorter than 128 rows
int wgrad_ranges(int M, int GH, int H, int I) {
  const int tiles = ((GH + kT64 - 1) / kT64) * ((H + kT64 - 1) / kT64 + (I + kT64 - 1) / kT64);
  int z = (3 * 148 + tiles - 1) / tiles;
  if (z > (M + 127) / 128) z = (M + 127) / 128;
  return z < 1 ? 1 : (z > 64 ? 64 : z);
}
template <class D>
void gradients64(D d, int M, int GH, int H, int I, const float* first, int Bf, const float* rest, const float* x, const float* W_ih, float* dx,
                 const gru_grads* g, float* scratch, cudaStream_t s) {
  prof_begin(KC_WGRAD, 2.0 * M * GH * (double)(H + (dx ? 2 : 1) * I), s);
  const int z = wgrad_ranges(M, GH, H, I);
  const i64 nhh = (i64)GH * H, nih = (i64)GH * I, zs = nhh + nih + 2 * GH;
  const WgradOut out{g->dW_hh, g->dW_ih, g->db_hh, g->db_ih, H, I, 0};
  const WgradOut part{scratch, scratch + nhh, scratch + nhh + nih, scratch + nhh + nih + GH, H, I, zs};
  const int kchunk = ((M + z - 1) / z + kK64 - 1) / kK64 * kK64;
  const dim3 grid((GH + kT64 - 1) / kT64, (H + kT64 - 1) / kT64 + (I + kT64 - 1) / kT64, z);
  gemm64_kernel<true><<<grid, 256, 0, s>>>(G64{GH, H, I, M, kchunk}, DaCols<D>{d}, WgradB{first, rest, x, Bf, H, I}, z > 1 ? part : out);
  count_launch();
  if (z > 1) {
    const i64 n4 = zs / 4;
    reduce_parts_kernel<<<(int)((n4 + 255) / 256 < 1184 ? (n4 + 255) / 256 : 1184), 256, 0, s>>>(reinterpret_cast<const float4*>(scratch), zs / 4, z, nhh,
                                                                                               nih, GH, out);
    count_launch();
  }
  if (dx) {      // dx[m, c] = sum_j dA_i[m, j] W_ih[j, c]
    gemm64_kernel<false><<<dim3((M + kT64 - 1) / kT64, (I + kT64 - 1) / kT64), 256, 0, s>>>(G64{M, I, 0, GH, GH}, DaRows<D>{d}, ColK{W_ih, I},
                                                                                         Store64{dx, I});
    count_launch();
  }
  prof_end(s);
}

}  // namespace

size_t simt_gradients_scratch(int M, int GH, int H, int I) {      // floats
  const int z = wgrad_ranges(M, GH, H, I);
  return z > 1 ? (size_t)z * ((size_t)GH * (H + I) + 2 * GH) : 0;
}
void simt_gradients(int M, int B, int H, int I, const float* lam, i64 lam_ts, const float* cr, const float* cz, const float* cn, const float* cnp,
                    const float* h0, const float* h, const float* x, const float* W_ih, float* dx, const gru_grads* g, float* scratch, cudaStream_t s) {
  gradients64(FormedDA{lam, lam_ts, cr, cz, cn, cnp, B, H}, M, 3 * H, H, I, h0, B, h, x, W_ih, dx, g, scratch, s);
}
void simt_lstm_gradients(int M, int B, int H, int I, const float* dA, const float* h0, const float* h, const float* x, const float* W_ih, float* dx,
                         const gru_grads* g, float* scratch, cudaStream_t s) {
  gradients64(DenseDA{dA, (i64)4 * H}, M, 4 * H, H, I, h0, B, h, x, W_ih, dx, g, scratch, s);
}

void simt_lstm_fwd_step(const LstmFwdArgs& a, cudaStream_t s) {
  launch<4, true, true>(KC_FWD_STEP, a.M, a.H, a.H, StridedRowsA{a.hin, a.in_ks, a.B, a.H}, GateW{a.W_hh, a.H, a.H}, LstmFwdEpi{a}, s);
}
void simt_lstm_linearise(const LstmLinArgs& a, cudaStream_t s) {
  launch<4, true, true>(KC_LINEARISE, a.M, a.H, a.H, LstmLinA{a.h0, a.h, a.ts, a.stride_t, a.t0, a.B, a.H}, GateW{a.W_hh, a.H, a.H},
                        LstmLinEpi{a}, s);
}
void simt_lstm_adj_step(const LstmAdjArgs& a, cudaStream_t s) {
  i64 items = (i64)a.M * a.H;
  int grid = (int)((items + 255) / 256 < 1184 ? (items + 255) / 256 : 1184);
  lstm_adj_c_kernel<<<grid < 1 ? 1 : grid, 256, 0, s>>>(a);
  count_launch();
  launch<1, true, false>(KC_ADJ_STEP, a.M, a.H, 4 * a.H, LstmAdjA{a}, DenseBT{a.W_hh, a.H}, StoreEpi{a.lh_out, a.H}, s);
}
void simt_lstm_form_dA(const float* lc, const float* lh, i64 lam_ts, int B, const float* p, const float* ci, const float* cf,
                       const float* cg, const float* co, float* dA, i64 M, int H, cudaStream_t s) {
  i64 items = M * H;
  int grid = (int)((items + 255) / 256 < 1184 ? (items + 255) / 256 : 1184);
  lstm_form_dA_kernel<<<grid < 1 ? 1 : grid, 256, 0, s>>>(lc, lh, lam_ts, B, p, ci, cf, cg, co, dA, M, H);
  count_launch();
}

void simt_project(const float* x, const float* W_ih, const float* b_ih, float* gi, int M, int I, int H3, cudaStream_t s) {
  if (M <= 0) return;
  prof_begin(KC_PROJ, 2.0 * M * (double)H3 * I, s);
  gemm64_kernel<false><<<dim3((M + kT64 - 1) / kT64, (H3 + kT64 - 1) / kT64), 256, 0, s>>>(G64{M, H3, 0, I, I}, RowK{x, I}, RowK{W_ih, I},
                                                                                       Bias64{gi, H3, b_ih});
  prof_end(s);
  count_launch();
}

void simt_fwd_step(const FwdStepArgs& a, cudaStream_t s) {
  launch<3, true, true>(KC_FWD_STEP, a.M, a.H, a.H, StridedRowsA{a.hin, a.hin_ks, a.B, a.H}, GateW{a.W_hh, a.H, a.H}, FwdEpi{a}, s);
}

void simt_linearise(const LinArgs& a, cudaStream_t s) {
  launch<3, true, true>(KC_LINEARISE, a.M, a.H, a.H, LinA{a.h0, a.h, a.stride_t, a.t0, a.B, a.H}, GateW{a.W_hh, a.H, a.H}, LinEpi{a}, s);
}

void simt_adj_step(const AdjStepArgs& a, cudaStream_t s) {
  launch<1, true, false>(KC_ADJ_STEP, a.M, a.H, 3 * a.H, AdjA{a.lin, a.lin_ks, a.cr, a.cz, a.cn, a.coef_ks, a.B, a.H},
                         DenseBT{a.W_hh, a.H}, AdjEpi{a}, s);
}

void simt_adj_dx(const AdjStepArgs& a, const float* W_ih, int C, float* out, cudaStream_t s) {
  launch<1, true, false>(KC_ADJ_STEP, a.M, C, 3 * a.H, AdjA{a.lin, a.lin_ks, a.cr, a.cz, a.cn, a.coef_ks, a.B, a.H}, DenseBT{W_ih, C},
                         StoreEpi{out, C}, s);
}

}  // namespace mg
