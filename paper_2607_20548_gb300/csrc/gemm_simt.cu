// Batched fp32 GEMM on the CUDA cores: C_b = alpha * op(A_b) op(B_b) + beta * C_b.
//
// Exact fp32 FMAs, so it is the accuracy reference for the tensor-core path and
// the engine where the tcgen05 path does not apply: the whole step of a class with a
// side that is not a multiple of 4 (TMA copies 16-byte rows), and the basis changes
// of the first moment in soap_state_get/set.
//
// Tiling: BM x BN output tile per 256-thread CTA, K in steps of BK, operands double-buffered
// through shared memory (k-major), each thread a (BM/16) x (BN/16) micro-tile of groups of 4 rows
// by 4 columns, which it reads as float4: with 4-byte reads a 64 x 64 tile was bound by shared
// memory (8 reads to 16 FMAs). A step takes one trip to memory, so a launch with few tiles is bound
// by that latency: it takes smaller tiles, for more CTAs, and deeper steps. Every element sums its K
// products in order whatever the tile, so the tile does not change the result.
// 512 x 512 x 1001, batch 2: 141 us with 128 x 128 tiles, steps of 8 and 4-byte reads, 49 us with
// 64 x 64 tiles and steps of 32; 4097^3: 3959 -> 3352 us (41 TF/s).
#include "soap_internal.h"

namespace soap {
namespace {

constexpr int kThreads = 256;
constexpr int kSms = 152;

__device__ __forceinline__ const float* resolve(const Operand& o, int b) {
  return (o.ptrs ? o.ptrs[b] : o.base + (int64_t)b * o.stride) + o.offset;
}
__device__ __forceinline__ float* resolve(const MutOperand& o, int b) {
  return (o.ptrs ? o.ptrs[b] : o.base + (int64_t)b * o.stride) + o.offset;
}

template <int V>
__device__ __forceinline__ void read_vec(float* d, const float* s) {
  if constexpr (V == 4) *reinterpret_cast<float4*>(d) = *reinterpret_cast<const float4*>(s);
  else if constexpr (V == 2) *reinterpret_cast<float2*>(d) = *reinterpret_cast<const float2*>(s);
  else d[0] = s[0];
}

template <bool TA, bool TB, int BM, int BN, int BK>
__global__ void __launch_bounds__(kThreads) gemm_simt_kernel(int M, int N, int K, float alpha,
                                                             Operand A, Operand B, float beta,
                                                             MutOperand C) {
  constexpr int TM = BM / 16, TN = BN / 16;
  constexpr int VM = TM < 4 ? TM : 4, VN = TN < 4 ? TN : 4;
  constexpr int A_PER = BM * BK / kThreads;
  constexpr int B_PER = BN * BK / kThreads;
  __shared__ __align__(16) float As[2][BK][BM + 4];
  __shared__ __align__(16) float Bs[2][BK][BN + 4];

  const int b = blockIdx.z;
  const int m0 = blockIdx.y * BM, n0 = blockIdx.x * BN;
  const float* Ab = resolve(A, b);
  const float* Bb = resolve(B, b);
  float* Cb = resolve(C, b);
  const int tid = threadIdx.x, tx = tid % 16, ty = tid / 16;

  float ra[A_PER], rb[B_PER];
  // op(A) element (mm, kk): A stored M x K (row mm) or, transposed, K x M (row kk).
  // The fastest-varying index follows the stored row so global reads coalesce, in runs of 8 where
  // the tile is transposed on its way (whole sectors, and 4 kk + mm is a bank of its own per lane).
  auto a_coord = [](int e, int& mm, int& kk) {
    if (!TA) { mm = e / 8 % BM; kk = e % 8 + e / (8 * BM) * 8; } else { kk = e / BM; mm = e % BM; }
  };
  auto b_coord = [](int e, int& kk, int& nn) {
    if (!TB) { kk = e / BN; nn = e % BN; } else { nn = e / 8 % BN; kk = e % 8 + e / (8 * BN) * 8; }
  };
  auto load = [&](int k0) {
#pragma unroll
    for (int i = 0; i < A_PER; ++i) {
      int mm, kk;
      a_coord(tid + i * kThreads, mm, kk);
      const int gm = m0 + mm, gk = k0 + kk;
      float v = 0.f;
      if (gm < M && gk < K) v = TA ? Ab[(int64_t)gk * A.ld + gm] : Ab[(int64_t)gm * A.ld + gk];
      ra[i] = v;
    }
#pragma unroll
    for (int i = 0; i < B_PER; ++i) {
      int kk, nn;
      b_coord(tid + i * kThreads, kk, nn);
      const int gk = k0 + kk, gn = n0 + nn;
      float v = 0.f;
      if (gk < K && gn < N) v = TB ? Bb[(int64_t)gn * B.ld + gk] : Bb[(int64_t)gk * B.ld + gn];
      rb[i] = v;
    }
  };
  auto store = [&](int buf) {
#pragma unroll
    for (int i = 0; i < A_PER; ++i) {
      int mm, kk;
      a_coord(tid + i * kThreads, mm, kk);
      As[buf][kk][mm] = ra[i];
    }
#pragma unroll
    for (int i = 0; i < B_PER; ++i) {
      int kk, nn;
      b_coord(tid + i * kThreads, kk, nn);
      Bs[buf][kk][nn] = rb[i];
    }
  };

  float acc[TM][TN];
#pragma unroll
  for (int i = 0; i < TM; ++i)
#pragma unroll
    for (int j = 0; j < TN; ++j) acc[i][j] = 0.f;

  const int nk = (K + BK - 1) / BK;
  if (nk > 0) {
    load(0);
    store(0);
  }
  __syncthreads();
  for (int t = 0; t < nk; ++t) {
    const int cur = t & 1;
    if (t + 1 < nk) load((t + 1) * BK);
#pragma unroll
    for (int kk = 0; kk < BK; ++kk) {
      alignas(16) float a[TM], bv[TN];
#pragma unroll
      for (int i = 0; i < TM; i += VM) read_vec<VM>(&a[i], &As[cur][kk][VM * ty + 16 * i]);
#pragma unroll
      for (int j = 0; j < TN; j += VN) read_vec<VN>(&bv[j], &Bs[cur][kk][VN * tx + 16 * j]);
#pragma unroll
      for (int i = 0; i < TM; ++i)
#pragma unroll
        for (int j = 0; j < TN; ++j) acc[i][j] = fmaf(a[i], bv[j], acc[i][j]);
    }
    if (t + 1 < nk) store(cur ^ 1);
    __syncthreads();
  }

#pragma unroll
  for (int i = 0; i < TM; ++i) {
    const int gm = m0 + VM * ty + i % VM + 16 * (i - i % VM);
    if (gm >= M) continue;
#pragma unroll
    for (int j = 0; j < TN; ++j) {
      const int gn = n0 + VN * tx + j % VN + 16 * (j - j % VN);
      if (gn >= N) continue;
      float* c = Cb + (int64_t)gm * C.ld + gn;
      float v = alpha * acc[i][j];
      if (beta != 0.f) v = fmaf(beta, *c, v);
      *c = v;
    }
  }
}

template <int BM, int BN, int BK>
cudaError_t launch_tile(bool ta, bool tb, int M, int N, int K, float alpha, Operand A, Operand B,
                        float beta, MutOperand C, int batch, cudaStream_t s) {
  dim3 grid((N + BN - 1) / BN, (M + BM - 1) / BM, batch);
  if (!ta && !tb) gemm_simt_kernel<false, false, BM, BN, BK><<<grid, kThreads, 0, s>>>(M, N, K, alpha, A, B, beta, C);
  else if (!ta && tb) gemm_simt_kernel<false, true, BM, BN, BK><<<grid, kThreads, 0, s>>>(M, N, K, alpha, A, B, beta, C);
  else if (ta && !tb) gemm_simt_kernel<true, false, BM, BN, BK><<<grid, kThreads, 0, s>>>(M, N, K, alpha, A, B, beta, C);
  else gemm_simt_kernel<true, true, BM, BN, BK><<<grid, kThreads, 0, s>>>(M, N, K, alpha, A, B, beta, C);
  return cudaGetLastError();
}

}  // namespace

cudaError_t gemm_simt(bool ta, bool tb, int M, int N, int K, float alpha, Operand A, Operand B,
                      float beta, MutOperand C, int batch, cudaStream_t s) {
  if (M <= 0 || N <= 0 || batch <= 0) return cudaSuccess;
  // The larger tile, which reads shared memory least per FMA, as long as its CTAs fill the chip:
  // 304 of 128 x 128 (8 x 1023^3: 434 us, 64 x 64 tiles 477), of 64 x 64 at least three quarters of
  // the SMs (144: 768 x 768 x 257 takes 18.5 us, 37 with 128 x 128; with 60 CTAs 257 x 768 x 768
  // takes 34.8 us, 28.7 with 32 x 64).
  auto ctas = [&](int bm, int bn) { return (int64_t)((M + bm - 1) / bm) * ((N + bn - 1) / bn) * batch; };
  if (M > 64 && N > 64 && ctas(128, 128) >= 2 * kSms)
    return launch_tile<128, 128, 16>(ta, tb, M, N, K, alpha, A, B, beta, C, batch, s);
  if (M > 32 && ctas(64, 64) >= kSms * 3 / 4)
    return launch_tile<64, 64, 32>(ta, tb, M, N, K, alpha, A, B, beta, C, batch, s);
  return launch_tile<32, 64, 32>(ta, tb, M, N, K, alpha, A, B, beta, C, batch, s);
}

}  // namespace soap
