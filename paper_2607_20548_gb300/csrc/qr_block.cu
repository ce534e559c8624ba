// Factorisation of a 128-column block of the QR without a column loop over its positions.
//
// The block is a matrix A (m positions x kbo columns, kbo <= 128; column c of A is row k0 + c of
// At). Householder's column loop needs one reduction over all positions per column; here one
// reduction gives the Gram matrix G = A^T A, and everything sequential happens on 128 x 128
// matrices in one CTA:
//
//   G = R^T R (Cholesky), and with A1 the first kbo rows of A and D = diag(+-1)
//   D R - A1 = V1 W        V1 unit lower, W upper triangular: elimination without pivoting,
//                          D_j = the sign of the running pivot of -A1, so that |W_jj| = R_jj +
//                          |pivot| (no cancellation)
//   V2 = -A2 W^-1          the rows below the first kbo
//   T  = W (D R)^-1 V1^-T
//
// are exactly the Householder vectors and the triangular factor of H_1 ... H_kbo = I - V T V^T
// with the reflector convention of the column loop (R_jj of the reflectors is D_j R_jj; the
// reconstruction of Householder vectors from an explicit Q, Ballard et al., "Reconstructing
// Householder vectors from tall-skinny QR", applied to Q = A R^-1). In 32-bit arithmetic G carries
// an error E of about 2^-24 in units of its column norms, and Q then misses orthogonality by
// R^-T E R^-1: by E times the norm of the inverse of G^ = G scaled to a unit diagonal. The pivots do
// not bound that norm (with every squared pivot at 0.4 of its column's squared norm it can exceed
// 1e10). Its trace does: the eigenvalues of G^ add up to kbo, so that
//   ||G^^-1|| <= tr(G^^-1) - kbo + 2,   tr(G^^-1) = sum_i G_ii ||row i of R^-1||^2,
// and the kernel that forms T's rows solves for R^-1's beside them. So does its Frobenius norm, which
// is closer where many directions have lost a little each (the first steps of a run) and takes a
// product of R^-1 by its transpose. The block is taken this way only if the excess tr(G^^-1) - kbo is at
// most kQrMaxExcess, or ||G^^-1||_F at most kQrMaxInverse, and every pivot is clear of the zero-column
// threshold; a block whose columns are all below that threshold is skipped outright (no reflectors);
// any other block is left to the column loop: qr_panel_kernel decides, and writes everything that a
// block factored here leaves behind. In the steady state of a run P = F Q has nearly orthogonal columns
// (an excess of 0.1-6); a part of the first steps' blocks and those of rank-deficient factors take the
// column loop.
//
//   qr_gram_kernel  G in up to 4 partial sums: tcgen05 products of 128 x 32 chunks, cluster
//                   reduction through distributed shared memory
//   qr_core_kernel  one CTA per matrix: Cholesky and elimination in one loop over the columns,
//                   W^-1 formed in place in the finished columns (Gauss-Jordan)
//   qr_form_kernel  V2 = -A2 W^-1 in tiles of 128 positions (tcgen05), T's rows, and the squares of
//                   R^-1's
#include <cooperative_groups.h>

#include <algorithm>
#include <atomic>
#include <type_traits>

#include "profile.h"
#include "qr_block.h"
#include "tc_ptx.h"

namespace cg = cooperative_groups;

namespace soap {
namespace {

constexpr int NBO = kQrBlock;
constexpr uint64_t kWaitNs = 2000000000ull;
// Squared pivot over squared column norm below which a block leaves for the column loop at once (blocks
// of a run that the rule admits have 0.5 and more). So does one whose squared norms over squared pivots,
// squared, already add up to more than kQrMaxInverse^2: G^^-1's diagonal is at least those ratios.
// (Ending at the trace's limit in this way, QR of 64 Gaussian 768-factors, most blocks of which decline,
// went from 5.38 to 5.25 ms.)
constexpr float kRhoMin = 0.25f;

// byte offset of 16-byte unit q of row r in a tile of 128-byte rows, swizzled within 1024-byte
// groups of 8 rows (the K-major layout of tc::desc_sw128)
__device__ __forceinline__ int swz16(int r, int q) { return (r >> 3) * 1024 + (r & 7) * 128 + ((q ^ (r & 7)) << 4); }
__device__ __forceinline__ float4 lo4(float4 x) {
  return make_float4(tc::tf32_lo(x.x), tc::tf32_lo(x.y), tc::tf32_lo(x.z), tc::tf32_lo(x.w));
}
__device__ __forceinline__ void cp16(uint32_t dst, const float* src, bool ok) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(ok ? 16 : 0) : "memory");
}
// the four products of one 32-wide chunk (A hi/lo, B hi/lo tiles of 128 rows) into accumulator d,
// the small ones first: the tensor core truncates the accumulator at every addition
__device__ __forceinline__ void mma_chunk(uint32_t d, uint32_t a_hi, uint32_t a_lo, uint32_t b_hi, uint32_t b_lo) {
  constexpr uint32_t idesc = tc::idesc_tf32(NBO, NBO);
#pragma unroll
  for (int kk = 0; kk < 4; ++kk) {
    const uint32_t off = kk * 32;  // 8 tf32 = 32 bytes along K
    tc::umma_tf32(d, tc::desc_sw128(a_lo + off), tc::desc_sw128(b_lo + off), idesc, kk != 0);
    tc::umma_tf32(d, tc::desc_sw128(a_lo + off), tc::desc_sw128(b_hi + off), idesc, 1u);
    tc::umma_tf32(d, tc::desc_sw128(a_hi + off), tc::desc_sw128(b_lo + off), idesc, 1u);
  }
#pragma unroll
  for (int kk = 0; kk < 4; ++kk)
    tc::umma_tf32(d, tc::desc_sw128(a_hi + kk * 32), tc::desc_sw128(b_hi + kk * 32), idesc, 1u);
}

// M: row x is -W^-1's column x up to the diagonal and V1's column x below it. It takes the place of
// the matrix's first partial Gram matrix, which only the CTA that writes M reads.
__device__ __forceinline__ float* block_m(const QrBlockArgs& p, int b) {
  return p.Gpart + (int64_t)b * kQrGramParts * NBO * NBO;
}

// What the panel kernel decides on, and what the core kernel hands over for it, in place of the second partial Gram matrix:
// the trace of G^^-1 by rows of a CTA of the form kernel, then G's diagonal. R^-1 scaled likewise takes
// the place of the third.
__device__ __forceinline__ float* block_trace(const QrBlockArgs& p, int b) {
  return p.Gpart + ((int64_t)b * kQrGramParts + 1) * NBO * NBO;
}

constexpr int kThreads = 256;
constexpr int kTile = NBO * 32 * 4;  // one 128 x 32 fp32 tile
constexpr int kGramStages = 4;
constexpr int kGramLd = NBO + 4;
constexpr int kGramSmem = kGramStages * kTile + 2 * kTile + 1024;
static_assert(NBO * kGramLd * 4 <= kGramSmem - 1024, "the partial product fits the stages");

// Partial Gram matrices: CTA x of matrix b takes chunks [x cper, (x+1) cper) of 32 positions; a
// cluster's partial sums are added through distributed shared memory (fixed order) and written as
// Gpart[b][cluster]. Both operands are the same tile, copied once with cp.async into the swizzled
// K-major layout; every thread forms the lo part of what it copied. Each chunk is summed afresh in
// one of two accumulators and added in fp32 registers while the next chunk's products run.
__global__ void __launch_bounds__(kThreads, 1) qr_gram_kernel(QrBlockArgs p, int nch, int cper, int nclusters) {
  cg::cluster_group cluster = cg::this_cluster();
  const int rank = (int)cluster.block_rank(), cs = (int)cluster.num_blocks();
  const int b = blockIdx.y, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* sm = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  __shared__ __align__(8) uint64_t bar[2];
  __shared__ uint32_t s_tmem;
  uint8_t* st_hi = sm;
  uint8_t* st_lo = sm + kGramStages * kTile;
  const int n = p.n, k0 = p.k0, kbo = p.kbo;
  const float* S = p.At + (int64_t)b * n * n + (int64_t)k0 * n + k0;  // row c: column c of A
  const int m = n - k0;
  const int c_beg = blockIdx.x * cper, c_end = min(nch, c_beg + cper);
  const int nloc = max(0, c_end - c_beg);
  if (tid == 0) {
    tc::mbar_init(&bar[0], 1);
    tc::mbar_init(&bar[1], 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(tc::smem_u32(&s_tmem)),
                 "r"(256));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  tc::tc_fence_before();
  __syncthreads();
  tc::tc_fence_after();
  const uint32_t tmem = s_tmem;
  auto issue = [&](int ch) {
    const uint32_t dst = tc::smem_u32(st_hi + (ch % kGramStages) * kTile);
    for (int u = tid; u < NBO * 8; u += kThreads) {
      const int r = u >> 3, q = u & 7, i = (c_beg + ch) * 32 + 4 * q;
      const bool ok = r < kbo && i < m;  // m is a multiple of 4
      cp16(dst + swz16(r, q), ok ? S + (int64_t)r * n + i : p.At, ok);
    }
  };
  float y[64];
#pragma unroll
  for (int l = 0; l < 64; ++l) y[l] = 0.f;
  const uint32_t lane_base = tmem + ((uint32_t)(32 * (warp & 3)) << 16) + (uint32_t)(64 * (warp >> 2));
  auto drain = [&](int ch) {
    float v[32];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      tc::tmem_ld32(lane_base + (uint32_t)((ch & 1) * NBO + 32 * h), v);
#pragma unroll
      for (int l = 0; l < 32; ++l) y[32 * h + l] += v[l];
    }
  };
  for (int s = 0; s < kGramStages - 1; ++s) {
    if (s < nloc) issue(s);
    asm volatile("cp.async.commit_group;" ::: "memory");
  }
  int issued = 0;
  bool aborted = false, bad = false;
  for (int ch = 0; ch < nloc; ++ch) {
    asm volatile("cp.async.wait_group %0;" ::"n"(kGramStages - 2) : "memory");
    const uint8_t* hi = st_hi + (ch % kGramStages) * kTile;
    uint8_t* lo = st_lo + (ch & 1) * kTile;
    for (int u = tid; u < NBO * 8; u += kThreads) {
      const int off = swz16(u >> 3, u & 7);
      *reinterpret_cast<float4*>(lo + off) = lo4(*reinterpret_cast<const float4*>(hi + off));
    }
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    if (__syncthreads_or(bad)) {
      aborted = true;
      break;
    }
    if (tid == 0) {
      tc::tc_fence_after();
      const uint32_t h = tc::smem_u32(hi), l = tc::smem_u32(lo);
      mma_chunk(tmem + (uint32_t)((ch & 1) * NBO), h, l, h, l);
      tc::umma_commit(&bar[ch & 1]);
    }
    issued = ch + 1;
    if (ch >= 1) {  // the previous chunk's sum, and its stage refilled
      bool ok = tc::mbar_wait(&bar[(ch - 1) & 1], ((ch - 1) >> 1) & 1, kWaitNs);
      ok = __all_sync(0xffffffffu, ok);
      if (ok) {
        tc::tc_fence_after();
        drain(ch - 1);
      } else {
        bad = true;
      }
    }
    if (!bad && ch + kGramStages - 1 < nloc) issue(ch + kGramStages - 1);
    asm volatile("cp.async.commit_group;" ::: "memory");
    tc::tc_fence_before();
  }
  bool ok_last = true;
  if (issued > 0)
    ok_last = __all_sync(0xffffffffu, tc::mbar_wait(&bar[(issued - 1) & 1], ((issued - 1) >> 1) & 1, kWaitNs));
  if (!aborted && !bad && ok_last && issued > 0) {
    tc::tc_fence_after();
    drain(issued - 1);
  }
  if (aborted || bad || !ok_last) atomicOr(p.status, kStatusTimeout);
  asm volatile("cp.async.wait_all;" ::: "memory");
  tc::tc_fence_before();
  __syncthreads();
  if (warp == 0) {
    tc::tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(256));
  }
  float* P = reinterpret_cast<float*>(sm);
  {
    float* row = P + (32 * (warp & 3) + lane) * kGramLd + 64 * (warp >> 2);
#pragma unroll
    for (int l = 0; l < 16; ++l)
      *reinterpret_cast<float4*>(row + 4 * l) = make_float4(y[4 * l], y[4 * l + 1], y[4 * l + 2], y[4 * l + 3]);
  }
  cluster.sync();
  float* out = p.Gpart + ((int64_t)b * kQrGramParts + blockIdx.x / cs) * NBO * NBO;
  for (int u = tid; u < (NBO / cs) * (NBO / 4); u += kThreads) {
    const int r = rank + cs * (u >> 5), q = u & 31;
    float4 s = make_float4(0.f, 0.f, 0.f, 0.f);
    for (int z = 0; z < cs; ++z) {
      const float4 v = *reinterpret_cast<const float4*>(cluster.map_shared_rank(P, z) + r * kGramLd + 4 * q);
      s.x += v.x;
      s.y += v.y;
      s.z += v.z;
      s.w += v.w;
    }
    *reinterpret_cast<float4*>(out + r * NBO + 4 * q) = s;
  }
  cluster.sync();  // the peers have read this CTA's partial product
}

// One CTA per matrix. Two 128 x 128 matrices are held in registers, 8 x 8 elements per thread: g,
// the Schur complement of G, and s, which starts as -A1. The columns go in panels of 16:
//   1  the panel's rows of g and s and its columns of s go to shared memory
//   2  one warp factors the 16 x 16 diagonal blocks, a row of s (lanes 0-15) or of g (16-31) per
//      lane: g's Cholesky row R_j, the sign d_j, W_j = d_j R_j + (row j of s), the multipliers
//   3  one thread per row solves its 16 multipliers f (the columns of V1 below the panel; above it
//      and inside it -W^-1, Gauss-Jordan's running sums), one thread per column the panel's rows
//      of R and W
//   4  all threads apply the rank-16 updates s -= f W, g -= R^T R (packed fp32 pairs)
// Steps 2 and 3 keep a row's remaining elements in register pairs and drop a pair every second
// column, so that the loops stay rolled: the same work with a column at a time over the whole
// matrix, unrolled, took 175 us a block, bound by instruction fetch.
constexpr int kPw = 16;          // panel width
constexpr int kPairs = kPw / 2;
constexpr int kCoreLd = NBO + 1;
constexpr int kPld = NBO + 4;    // row stride of the panel's rows
constexpr int kCld = kPw + 4;    // row stride of the panel's columns
constexpr int kCoreSmem = (NBO * kCoreLd + 5 * kPw * kPld + NBO * kCld) * 4;
static_assert((NBO * kCoreLd) % 4 == 0, "16-byte aligned panel buffers");

__device__ __forceinline__ float2 ffma2(float2 a, float2 b, float2 c) {
  uint64_t d;
  asm("fma.rn.f32x2 %0, %1, %2, %3;"
      : "=l"(d)
      : "l"(reinterpret_cast<const uint64_t&>(a)), "l"(reinterpret_cast<const uint64_t&>(b)),
        "l"(reinterpret_cast<const uint64_t&>(c)));
  return reinterpret_cast<const float2&>(d);
}
__device__ __forceinline__ float2 dup(float x) { return make_float2(x, x); }
__device__ __forceinline__ void load_pairs(float2 (&v)[kPairs], const float* src) {  // 16-byte aligned
#pragma unroll
  for (int l = 0; l < kPairs / 2; ++l) {
    const float4 t = *reinterpret_cast<const float4*>(src + 4 * l);
    v[2 * l] = make_float2(t.x, t.y);
    v[2 * l + 1] = make_float2(t.z, t.w);
  }
}
__device__ __forceinline__ void store_pairs(float* dst, const float2 (&v)[kPairs]) {
#pragma unroll
  for (int l = 0; l < kPairs / 2; ++l)
    *reinterpret_cast<float4*>(dst + 4 * l) = make_float4(v[2 * l].x, v[2 * l].y, v[2 * l + 1].x, v[2 * l + 1].y);
}
// x += f v over a row's remaining pairs, whose first column is even (odd = false) or odd; after an
// odd column its pair is finished and the others move down
template <bool ODD>
__device__ __forceinline__ void eliminate(float2 (&x)[kPairs], float f, const float2 (&v)[kPairs]) {
  const float2 f2 = dup(f);
  if (!ODD) {
#pragma unroll
    for (int l = 0; l < kPairs; ++l) x[l] = ffma2(f2, v[l], x[l]);
  } else {
#pragma unroll
    for (int l = 1; l < kPairs; ++l) x[l - 1] = ffma2(f2, v[l], x[l]);
    x[kPairs - 1] = make_float2(0.f, 0.f);
  }
}

struct CoreShared {
  // the diagonal blocks, row j from column 2 floor(j / 2) on: W, R, and column j of V1 likewise
  float w[kPw][kPw], r[kPw][kPw], l[kPw][kPw];
  float pv[2][2][2][kPw];  // two pivot rows of s and of g, by pair parity: [parity][s, g][row]
  float zero[kPw];
  float iw[kPw], ir[kPw], d[kPw];  // 1 / W_jj, 1 / R_jj, sign
  float norm[NBO];                 // squared column norms
  int zero_block, fail;
};

__device__ __forceinline__ float inv_sqrt(float x) {
  const float y = rsqrtf(x);
  return fmaf(0.5f * y, fmaf(-x * y, y, 1.f), y);  // one Newton step
}
__device__ __forceinline__ float inv(float x) {
  const float y = __fdividef(1.f, x);
  return fmaf(y, fmaf(-x, y, 1.f), y);
}

// Columns j and j + 1 (j even) of the diagonal blocks (step 2), one warp; returns whether their
// pivots are good, and adds to `inverse2` what they prove of ||G^^-1||_F^2. The two pivot rows go through shared
// memory once; every lane derives both columns' reflectors from them.
__device__ __forceinline__ bool diag_pair(CoreShared& sh, float2 (&x)[kPairs], int j, float norm0, float norm1, float lim2,
                                          float& inverse2) {
  const int lane = threadIdx.x & 31, par = (j >> 1) & 1;
  const bool srow = lane < 16;
  if ((lane & 14) == j) store_pairs(sh.pv[par][lane >> 4][lane & 1], x);
  __syncwarp();
  float2 ra[kPairs], rb[kPairs], wa[kPairs], wb[kPairs];
  load_pairs(ra, sh.pv[par][1][0]);
  load_pairs(rb, sh.pv[par][1][1]);
  const float2 sa = *reinterpret_cast<const float2*>(sh.pv[par][0][0]);
  const float2 sb = *reinterpret_cast<const float2*>(sh.pv[par][0][1]);
  load_pairs(wa, srow ? sh.pv[par][0][0] : sh.zero);
  load_pairs(wb, srow ? sh.pv[par][0][1] : sh.zero);
  const float g0 = ra[0].x;
  const float ir0 = inv_sqrt(g0), r0 = g0 * ir0, r01 = ra[0].y * ir0;
  const float g1 = fmaf(-r01, r01, rb[0].y);
  const float ir1 = inv_sqrt(g1), r1 = g1 * ir1;
  const float d0 = sa.x >= 0.f ? 1.f : -1.f;
  const float w0 = fmaf(d0, r0, sa.x), w01 = fmaf(d0, r01, sa.y);
  const float iw0 = inv(w0);
  const float l10 = sb.x * iw0;
  const float s1 = fmaf(-l10, w01, sb.y);
  const float d1 = s1 >= 0.f ? 1.f : -1.f;
  const float w1 = fmaf(d1, r1, s1);
  const float iw1 = inv(w1);
  // rows j and j + 1 of R, then of W in the lanes that hold s (elsewhere R's, by d = 1, l = 0)
  const float2 cd0 = dup(srow ? d0 : 1.f), cd1 = dup(srow ? d1 : 1.f), cl = dup(srow ? -l10 : 0.f);
#pragma unroll
  for (int l = 0; l < kPairs; ++l) {
    ra[l].x *= ir0;
    ra[l].y *= ir0;
    rb[l] = ffma2(dup(-r01), ra[l], rb[l]);
    rb[l].x *= ir1;
    rb[l].y *= ir1;
    wa[l] = ffma2(cd0, ra[l], wa[l]);
    wb[l] = ffma2(cl, wa[l], ffma2(cd1, rb[l], wb[l]));
  }
  const float m0 = x[0].x * (srow ? iw0 : ir0);
  const float m1 = fmaf(-m0, srow ? w01 : r01, x[0].y) * (srow ? iw1 : ir1);
  const float2 n0 = dup(-m0), n1 = dup(-m1);
#pragma unroll
  for (int l = 1; l < kPairs; ++l) x[l - 1] = ffma2(n1, wb[l], ffma2(n0, wa[l], x[l]));
  x[kPairs - 1] = make_float2(0.f, 0.f);
  if ((lane & 15) == 0) {
    float(*out)[kPw] = srow ? sh.w : sh.r;
    store_pairs(out[j], wa);
    store_pairs(out[j + 1], wb);
    if (srow) {
      sh.iw[j] = iw0;
      sh.iw[j + 1] = iw1;
      sh.d[j] = d0;
      sh.d[j + 1] = d1;
    } else {
      sh.ir[j] = ir0;
      sh.ir[j + 1] = ir1;
    }
  }
  if (srow && lane >= j) {
    sh.l[j][lane - j] = m0;
    sh.l[j + 1][lane - j] = m1;
  }
  const float inv0 = norm0 * ir0 * ir0, inv1 = norm1 * ir1 * ir1;
  inverse2 += fmaf(inv0, inv0, inv1 * inv1);
  // (false for a non-finite value too; squares outside fp32's comfortable range go the other way)
  return g0 >= kRhoMin * norm0 && g1 >= kRhoMin * norm1 && g0 > lim2 && g1 > lim2 && g0 > 1e-30f && g1 > 1e-30f &&
         norm0 < 1e30f && norm1 < 1e30f;
}

// Column j of a row's multipliers (step 3).
template <bool ODD>
__device__ __forceinline__ void solve_row(const CoreShared& sh, float2 (&z)[kPairs], int j, float* F, float* M, int li) {
  const float f = -(ODD ? z[0].y : z[0].x) * sh.iw[j];
  F[j * kPld] = f;
  M[j * NBO] = li > j && li < kPw ? sh.l[j][li - (j - ODD)] : -f;
  float2 w[kPairs];
  load_pairs(w, sh.w[j]);
  eliminate<ODD>(z, f, w);
}

// Row j of a column's R and W (step 3).
template <bool ODD>
__device__ __forceinline__ void solve_col(const CoreShared& sh, float2 (&x)[kPairs], float2 (&t)[kPairs], int j, float* Rk,
                                          float* Wk, float* Rb, float* Wb, int lc) {
  const float R = (ODD ? x[0].y : x[0].x) * sh.ir[j], d = sh.d[j];
  const float W = fmaf(d, R, ODD ? t[0].y : t[0].x);
  Rk[j * kPld] = R;
  Wk[j * kPld] = W;
  // (entries left of the diagonal are not read)
  const int o = (lc - (j - ODD)) & (kPw - 1);
  const bool after = lc >= kPw;
  Rb[j * NBO] = d * (after ? R : sh.r[j][o]);
  Wb[j * NBO] = after ? W : sh.w[j][o];
  float2 v[kPairs];
  load_pairs(v, sh.r[j]);
  eliminate<ODD>(x, -R, v);
  load_pairs(v, sh.l[j]);
  eliminate<ODD>(t, -W, v);
}

__global__ void __launch_bounds__(kThreads, 1) qr_core_kernel(QrBlockArgs p, int nparts) {
  extern __shared__ __align__(16) float s_t[];  // [128][129]: -A1 by columns
  float* rowS = s_t + NBO * kCoreLd;   // [16][132] the panel's rows of s
  float* rowG = rowS + kPw * kPld;     // [16][132] and of g
  float* colS = rowG + kPw * kPld;     // [128][20] the panel's columns of s
  float* F = colS + NBO * kCld;        // [16][132] negated multipliers by row
  float* Wk = F + kPw * kPld;          // [16][132] rows of W, zero up to the panel's end
  float* Rk = Wk + kPw * kPld;         // [16][132] rows of R, likewise
  __shared__ __align__(16) CoreShared sh;
  const int b = blockIdx.x, tid = threadIdx.x, lane = tid & 31;
  const int tx = ((tid >> 7) << 3) + (lane & 7), ty = (((tid >> 5) & 3) << 2) + (lane >> 3);
  const int n = p.n, k0 = p.k0, kbo = p.kbo, m = n - k0;
  const float* S = p.At + (int64_t)b * n * n + (int64_t)k0 * n + k0;
  const float* Gp = p.Gpart + (int64_t)b * kQrGramParts * NBO * NBO;
  // thread (ty, tx): row a = 32 (a / 2) + 2 ty + a mod 2, column pair q = 32 q + 2 tx: groups of 32
  // rows and columns, so that the updates leave out the groups that are finished
  auto row_of = [&](int a) { return ((a >> 1) << 5) + 2 * ty + (a & 1); };
  auto col_of = [&](int q) { return (q << 5) + 2 * tx; };
  // place of row or column x in F, Wk and Rk: a thread's elements of two groups are one 16-byte
  // unit, the units of eight threads consecutive (a warp is 4 rows of 8 threads)
  auto slot = [](int x) { return ((x >> 6) << 6) + (((x & 31) >> 1) << 2) + (((x >> 5) & 1) << 1) + (x & 1); };
#pragma unroll
  for (int it = 0; it < NBO * (NBO / 4) / kThreads; ++it) {
    const int u = tid + it * kThreads, c = u >> 5, q = 4 * (u & 31);  // column c of A, positions q .. q+3
    float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
    if (c < kbo && q < m) v = *reinterpret_cast<const float4*>(S + (int64_t)c * n + q);
    s_t[c * kCoreLd + q] = -v.x;
    s_t[c * kCoreLd + q + 1] = -v.y;
    s_t[c * kCoreLd + q + 2] = -v.z;
    s_t[c * kCoreLd + q + 3] = -v.w;
  }
  float2 s[8][4], g[8][4];  // g: only groups on or above the diagonal (a / 2 <= q)
#pragma unroll
  for (int a = 0; a < 8; ++a)
#pragma unroll
    for (int q = 0; q < 4; ++q) g[a][q] = make_float2(0.f, 0.f);
  for (int z = 0; z < nparts; ++z)
#pragma unroll
    for (int a = 0; a < 8; ++a)
#pragma unroll
      for (int q = a >> 1; q < 4; ++q) {
        const float2 v =
            *reinterpret_cast<const float2*>(Gp + (int64_t)z * NBO * NBO + row_of(a) * NBO + col_of(q));
        g[a][q].x += v.x;
        g[a][q].y += v.y;
      }
  if (tid == 0) {
    sh.zero_block = 1;
    sh.fail = 0;
  }
  if (tid < kPw) sh.zero[tid] = 0.f;
  __syncthreads();
  if (nparts == 0) {
    // at most 128 positions: A1 is all of A, and its Gram matrix is formed here in fp32 FMAs (a
    // square block's T answers a bias of its Gram matrix ten times over, so the tensor core's
    // truncating sums are not good enough for it, and the sums are short)
    for (int i = 0; i < m; ++i) {
      float2 x[4];
#pragma unroll
      for (int q = 0; q < 4; ++q) x[q] = make_float2(s_t[col_of(q) * kCoreLd + i], s_t[(col_of(q) + 1) * kCoreLd + i]);
#pragma unroll
      for (int a = 0; a < 8; ++a) {
        const float z = s_t[row_of(a) * kCoreLd + i];
#pragma unroll
        for (int q = a >> 1; q < 4; ++q) g[a][q] = ffma2(dup(z), x[q], g[a][q]);
      }
    }
  }
#pragma unroll
  for (int a = 0; a < 8; ++a)
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      s[a][q] = make_float2(s_t[col_of(q) * kCoreLd + row_of(a)], s_t[(col_of(q) + 1) * kCoreLd + row_of(a)]);
      if (col_of(q) == row_of(a)) sh.norm[row_of(a)] = g[a][q].x;
      if (col_of(q) + 1 == row_of(a)) sh.norm[row_of(a)] = g[a][q].y;
    }
  __syncthreads();
  const float thresh = p.thresh[b];
  if (tid < kbo) {
    const float lim = 0.99f * thresh;
    if (!(sh.norm[tid] <= lim * lim)) sh.zero_block = 0;
  }
  const float lim2 = 4.f * thresh * thresh;
  float* Rb = p.Rf + (int64_t)b * n * NBO;
  float* Wb = p.Wf + (int64_t)b * n * NBO;
  float* M = block_m(p, b);
  __syncthreads();
  const bool zero = sh.zero_block != 0;
  bool fast = !zero;
  const int npan = (kbo + kPw - 1) / kPw;
  float inverse2 = 0.f;  // (first warp)
  for (int pp = 0; pp < npan && fast; ++pp) {
    const int j0 = kPw * pp, pw = min(kPw, kbo - j0);  // a multiple of 4
    // 1: the panel's rows and columns
    auto put = [&](auto group) {
      constexpr int h = decltype(group)::value;  // the panel is one half of this group
      if ((tx >> 3) == (pp & 1)) {
#pragma unroll
        for (int a = 0; a < 8; ++a) *reinterpret_cast<float2*>(colS + row_of(a) * kCld + 2 * (tx & 7)) = s[a][h];
      }
      if ((ty >> 3) == (pp & 1)) {
#pragma unroll
        for (int e = 0; e < 2; ++e) {
          const int a = 2 * h + e, r = 2 * (ty & 7) + e;
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            *reinterpret_cast<float2*>(rowS + r * kPld + col_of(q)) = s[a][q];
            if (q >= h) *reinterpret_cast<float2*>(rowG + r * kPld + col_of(q)) = g[a][q];
            s[a][q] = make_float2(0.f, 0.f);  // these rows restart as W_pp^-1 W
          }
        }
      }
    };
    switch (pp >> 1) {
      case 0: put(std::integral_constant<int, 0>{}); break;
      case 1: put(std::integral_constant<int, 1>{}); break;
      case 2: put(std::integral_constant<int, 2>{}); break;
      default: put(std::integral_constant<int, 3>{}); break;
    }
    __syncthreads();
    // 2: the diagonal blocks
    if (tid < 32) {
      float2 x[kPairs];
      load_pairs(x, (lane < 16 ? rowS : rowG) + (lane & 15) * kPld + j0);
      bool ok = true;
#pragma unroll 1
      for (int j = 0; j < pw; j += 2) {
        const bool good = diag_pair(sh, x, j, sh.norm[j0 + j], sh.norm[j0 + j + 1], lim2, inverse2);
        ok = ok && good;
      }
      if (lane == 0 && !(ok && inverse2 <= kQrMaxInverse * kQrMaxInverse)) sh.fail = 1;
      if (lane < pw) p.dsign[(int64_t)b * n + k0 + j0 + lane] = sh.d[lane];
    }
    __syncthreads();
    if (sh.fail) {
      fast = false;
      break;
    }
    // 3: multipliers by row, rows of R and W by column
    if (tid < NBO) {
      const int i = tid, li = i - j0;
      float2 z[kPairs];
      load_pairs(z, colS + i * kCld);
      if (li >= 0 && li < kPw) {
#pragma unroll
        for (int l = 0; l < kPairs; ++l)
          z[l] = make_float2(li == 2 * l ? -1.f : 0.f, li == 2 * l + 1 ? -1.f : 0.f);
      }
#pragma unroll 1
      for (int j = 0; j < pw; j += 2) {
        solve_row<false>(sh, z, j, F + slot(i), M + (int64_t)j0 * NBO + i, li);
        solve_row<true>(sh, z, j + 1, F + slot(i), M + (int64_t)j0 * NBO + i, li);
      }
    } else {
      const int c = tid - NBO, lc = c - j0;
      float2 x[kPairs], t[kPairs];
#pragma unroll
      for (int l = 0; l < kPairs; ++l) {
        x[l] = t[l] = make_float2(0.f, 0.f);
        if (lc >= kPw) {
          x[l] = make_float2(rowG[2 * l * kPld + c], rowG[(2 * l + 1) * kPld + c]);
          t[l] = make_float2(rowS[2 * l * kPld + c], rowS[(2 * l + 1) * kPld + c]);
        }
      }
      float* Rr = Rb + j0 * NBO + c;
      float* Wr = Wb + j0 * NBO + c;
#pragma unroll 1
      for (int j = 0; j < pw; j += 2) {
        solve_col<false>(sh, x, t, j, Rk + slot(c), Wk + slot(c), Rr, Wr, lc);
        solve_col<true>(sh, x, t, j + 1, Rk + slot(c), Wk + slot(c), Rr, Wr, lc);
      }
    }
    __syncthreads();
    if (pp + 1 == npan) break;
    // 4: rank-16 updates of the column groups after the panel
    auto update = [&](auto group) {
      constexpr int h = decltype(group)::value;  // first group still in work
#pragma unroll 2
      for (int k = 0; k < kPw; ++k) {
        float fr[8], hr[8], wc[8], rc[8];
        auto load4 = [&](float* v, const float* src) {
          const float4 t = *reinterpret_cast<const float4*>(src);
          v[0] = t.x;
          v[1] = t.y;
          v[2] = t.z;
          v[3] = t.w;
        };
#pragma unroll
        for (int f = 0; f < 2; ++f) {
          load4(fr + 4 * f, F + k * kPld + 64 * f + 4 * ty);
          if (f >= (h >> 1)) {
            load4(hr + 4 * f, Rk + k * kPld + 64 * f + 4 * ty);
            load4(wc + 4 * f, Wk + k * kPld + 64 * f + 4 * tx);
            load4(rc + 4 * f, Rk + k * kPld + 64 * f + 4 * tx);
          }
        }
#pragma unroll
        for (int a = 0; a < 8; ++a)
#pragma unroll
          for (int q = h; q < 4; ++q) {
            s[a][q].x = fmaf(fr[a], wc[2 * q], s[a][q].x);
            s[a][q].y = fmaf(fr[a], wc[2 * q + 1], s[a][q].y);
            if (a >= 2 * h && (a >> 1) <= q) {
              g[a][q].x = fmaf(-hr[a], rc[2 * q], g[a][q].x);
              g[a][q].y = fmaf(-hr[a], rc[2 * q + 1], g[a][q].y);
            }
          }
      }
    };
    switch ((pp + 1) >> 1) {
      case 0: update(std::integral_constant<int, 0>{}); break;
      case 1: update(std::integral_constant<int, 1>{}); break;
      case 2: update(std::integral_constant<int, 2>{}); break;
      default: update(std::integral_constant<int, 3>{}); break;
    }
  }
  if (tid == 0) p.state[b] = zero ? kQrBlockZero : fast ? kQrBlockFast : kQrBlockColumns;
  if (tid < NBO) block_trace(p, b)[kQrTraceParts + tid] = sh.norm[tid];
  if (tid < kbo && (zero || fast)) {
    p.skip[(int64_t)b * n + k0 + tid] = zero ? 1 : 0;
    if (zero) p.dsign[(int64_t)b * n + k0 + tid] = 1.f;
  }
}

// Blocks 0 .. kTBlocks-1 of a matrix: 16 rows of T each (two per warp), by the row solves
// u (D R) = W_i and t V1^T = u (lane l holds columns 4 l .. 4 l + 3; each finished entry is
// broadcast once), beside them x (D R) = e_i for the trace, and 16 rows of V1, to Vt and to Vpos. The
// other blocks: V2 = -A2 W^-1 on 128
// positions each, as tcgen05 products of 128 positions x 32 columns chunks; A's chunk is turned
// position-major (with its lo part) in shared memory, each chunk has its own accumulator.
constexpr int kTBlocks = kQrTraceParts;
constexpr int kFormLd = NBO + 4;
constexpr int kFormSmem = NBO * kFormLd * 4 + 2 * 4 * kTile + 1024;
constexpr int kSolveSmem = 2 * NBO * kFormLd * 4;
static_assert(kFormSmem <= 232448 - 1024 && kSolveSmem <= kFormSmem, "shared memory budget");

__device__ __forceinline__ void t_rows(const QrBlockArgs& p, int b, int rb, float* sm, bool zero) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int n = p.n, k0 = p.k0, kbo = p.kbo, m = n - k0;
  float* Rs = sm;                  // [128][132] D R, strictly upper
  float* Vs = sm + NBO * kFormLd;  // [128][132] V1^T, strictly upper
  __shared__ float s_inv[NBO];
  __shared__ float s_trace[kThreads / 32];
  const float* Rb = p.Rf + (int64_t)b * n * NBO;
  const float* Wb = p.Wf + (int64_t)b * n * NBO;
  const float* M = block_m(p, b);
  float u[2][4];
  const int i0 = rb * 16 + 2 * warp;
#pragma unroll
  for (int e = 0; e < 2; ++e)
#pragma unroll
    for (int c = 0; c < 4; ++c) u[e][c] = 0.f;
  if (!zero) {
    constexpr int kBatch = 8;  // loads in flight per thread and matrix
#pragma unroll 1
    for (int it0 = 0; it0 < NBO * 32 / kThreads; it0 += kBatch) {
      float4 r[kBatch], v[kBatch];
#pragma unroll
      for (int it = 0; it < kBatch; ++it) {
        const int e = tid + (it0 + it) * kThreads, j = min(e >> 5, kbo - 1), q = 4 * (e & 31);
        r[it] = *reinterpret_cast<const float4*>(Rb + j * NBO + q);
        v[it] = *reinterpret_cast<const float4*>(M + j * NBO + q);
      }
#pragma unroll
      for (int it = 0; it < kBatch; ++it) {
        const int e = tid + (it0 + it) * kThreads, j = e >> 5, q = 4 * (e & 31);
        float ra[4] = {r[it].x, r[it].y, r[it].z, r[it].w}, va[4] = {v[it].x, v[it].y, v[it].z, v[it].w};
#pragma unroll
        for (int c = 0; c < 4; ++c) {
          if (q + c == j) s_inv[j] = 1.f / ra[c];
          if (q + c <= j) ra[c] = va[c] = 0.f;
        }
        *reinterpret_cast<float4*>(Rs + j * kFormLd + q) = make_float4(ra[0], ra[1], ra[2], ra[3]);
        *reinterpret_cast<float4*>(Vs + j * kFormLd + q) = make_float4(va[0], va[1], va[2], va[3]);
      }
    }
#pragma unroll
    for (int e = 0; e < 2; ++e)
      if (i0 + e < kbo) {
        const float4 w = *reinterpret_cast<const float4*>(Wb + (i0 + e) * NBO + 4 * lane);
        const float wa[4] = {w.x, w.y, w.z, w.w};
#pragma unroll
        for (int c = 0; c < 4; ++c) u[e][c] = 4 * lane + c >= i0 + e ? wa[c] : 0.f;
      }
  }
  __syncthreads();
  // V1's columns 16 rb .. (rows of Vt) and its rows 16 rb .. (rows of Vpos)
  {
    float* Vt = p.Vt + (int64_t)b * n * n + (int64_t)k0 * n + k0;
    float* Vt_lo = p.Vt_lo + (int64_t)b * n * n + (int64_t)k0 * n + k0;
    float* Vpos = p.Vpos + ((int64_t)b * n + k0) * NBO;
    float* Vpos_lo = p.Vpos_lo + ((int64_t)b * n + k0) * NBO;
    for (int e = tid; e < 16 * 32; e += kThreads) {
      const int x = rb * 16 + (e >> 5), i = 4 * (e & 31);
      if (x < kbo && i < m) {
        float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
        if (!zero) {
          v = *reinterpret_cast<const float4*>(Vs + x * kFormLd + i);
          if (i == x) v.x = 1.f;
          if (i + 1 == x) v.y = 1.f;
          if (i + 2 == x) v.z = 1.f;
          if (i + 3 == x) v.w = 1.f;
        }
        *reinterpret_cast<float4*>(Vt + (int64_t)x * n + i) = v;
        *reinterpret_cast<float4*>(Vt_lo + (int64_t)x * n + i) = lo4(v);
      }
    }
    for (int e = tid; e < 16 * NBO; e += kThreads) {
      const int i = rb * 16 + (e & 15), x = e >> 4;
      if (i < m) {
        const float v = zero || x >= kbo || x > i ? 0.f : x == i ? 1.f : Vs[x * kFormLd + i];
        Vpos[(int64_t)i * NBO + x] = v;
        Vpos_lo[(int64_t)i * NBO + x] = tc::tf32_lo(v);
      }
    }
  }
  if (!zero) {
    // u_j = (u_j so far) / (D R)_jj, then t_j = u_j + (t_j so far): both solves advance together
    // (columns before a row's diagonal are zero and stay so)
    float t[2][4], w[2][4], x0[2][4], inv2[2] = {0.f, 0.f};  // w: e_i, then what is left of it; inv2: ||x||^2
#pragma unroll
    for (int e = 0; e < 2; ++e)
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        t[e][c] = x0[e][c] = 0.f;
        w[e][c] = 4 * lane + c == i0 + e ? 1.f : 0.f;
      }
#pragma unroll 1
    for (int j4 = i0 >> 2; 4 * j4 < kbo; ++j4) {
#pragma unroll
      for (int c = 0; c < 4; ++c) {  // kbo is a multiple of 4
        const int j = 4 * j4 + c;
        const float iv = s_inv[j];
        const float4 r = *reinterpret_cast<const float4*>(Rs + j * kFormLd + 4 * lane);
        const float4 v = *reinterpret_cast<const float4*>(Vs + j * kFormLd + 4 * lane);
#pragma unroll
        for (int e = 0; e < 2; ++e) {
          const float x = __shfl_sync(0xffffffffu, u[e][c], j4) * iv;
          const float y = __shfl_sync(0xffffffffu, t[e][c], j4) + x;
          u[e][0] = fmaf(-x, r.x, u[e][0]);
          u[e][1] = fmaf(-x, r.y, u[e][1]);
          u[e][2] = fmaf(-x, r.z, u[e][2]);
          u[e][3] = fmaf(-x, r.w, u[e][3]);
          t[e][0] = fmaf(-y, v.x, t[e][0]);
          t[e][1] = fmaf(-y, v.y, t[e][1]);
          t[e][2] = fmaf(-y, v.z, t[e][2]);
          t[e][3] = fmaf(-y, v.w, t[e][3]);
          if (lane == j4) t[e][c] = y;
          const float z = __shfl_sync(0xffffffffu, w[e][c], j4) * iv;
          inv2[e] = fmaf(z, z, inv2[e]);
          if (lane == j4) x0[e][c] = z;
          w[e][0] = fmaf(-z, r.x, w[e][0]);
          w[e][1] = fmaf(-z, r.y, w[e][1]);
          w[e][2] = fmaf(-z, r.z, w[e][2]);
          w[e][3] = fmaf(-z, r.w, w[e][3]);
        }
      }
    }
    {
      const float* norm = block_trace(p, b) + kQrTraceParts;
      float trace = 0.f;
#pragma unroll
      for (int e = 0; e < 2; ++e) {
        const float g = i0 + e < kbo ? norm[i0 + e] : 0.f, f = sqrtf(g);
        trace = fmaf(inv2[e], g, trace);
        *reinterpret_cast<float4*>(block_trace(p, b) + NBO * NBO + (i0 + e) * NBO + 4 * lane) =
            make_float4(f * x0[e][0], f * x0[e][1], f * x0[e][2], f * x0[e][3]);
      }
      if (lane == 0) s_trace[warp] = trace;
    }
#pragma unroll
    for (int e = 0; e < 2; ++e)
#pragma unroll
      for (int c = 0; c < 4; ++c) u[e][c] = t[e][c];
  }
  const int64_t t0 = (int64_t)b * NBO * NBO;
#pragma unroll
  for (int e = 0; e < 2; ++e) {
    const int i = i0 + e;
    const float4 t = make_float4(u[e][0], u[e][1], u[e][2], u[e][3]);
    *reinterpret_cast<float4*>(p.T + t0 + i * NBO + 4 * lane) = t;
    *reinterpret_cast<float4*>(p.T_lo + t0 + i * NBO + 4 * lane) = lo4(t);
  }
  // T^T: this CTA's 16 columns, through shared memory
  __syncthreads();
#pragma unroll
  for (int e = 0; e < 2; ++e)
#pragma unroll
    for (int c = 0; c < 4; ++c) sm[(4 * lane + c) * 17 + 2 * warp + e] = u[e][c];
  __syncthreads();
  if (tid == 0 && !zero) {
    float x = 0.f;
    for (int i = 0; i < kThreads / 32; ++i) x += s_trace[i];
    block_trace(p, b)[rb] = x;
  }
  for (int e = tid; e < NBO * 16; e += kThreads) {
    const int c = e >> 4, i = e & 15;
    const float t = sm[c * 17 + i];
    p.Tt[t0 + c * NBO + rb * 16 + i] = t;
    p.Tt_lo[t0 + c * NBO + rb * 16 + i] = tc::tf32_lo(t);
  }
}

__global__ void __launch_bounds__(kThreads, 1) qr_form_kernel(QrBlockArgs p) {
  extern __shared__ uint8_t smem_raw[];
  const int b = blockIdx.y, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int state = p.state[b];
  if (state == kQrBlockColumns) return;
  if (blockIdx.x < kTBlocks) {
    t_rows(p, b, blockIdx.x, reinterpret_cast<float*>(smem_raw), state == kQrBlockZero);
    return;
  }
  uint8_t* sm = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  __shared__ __align__(8) uint64_t bar[4];
  __shared__ uint32_t s_tmem;
  uint8_t* ops = sm;  // [2] A hi | A lo | B hi | B lo
  float* sA = reinterpret_cast<float*>(sm + 2 * 4 * kTile);  // [128 columns][132]: 128 positions
  const int n = p.n, k0 = p.k0;
  const int64_t nn = (int64_t)n * n;
  const int pos0 = k0 + NBO + (blockIdx.x - kTBlocks) * NBO;
  const int npos = min(NBO, n - pos0);  // a positive multiple of 4
  const float* S = p.At + b * nn + (int64_t)k0 * n + pos0;
  const float* M = block_m(p, b);
  if (tid == 0) {
    for (int i = 0; i < 4; ++i) tc::mbar_init(&bar[i], 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(tc::smem_u32(&s_tmem)),
                 "r"(512));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  tc::tc_fence_before();
  __syncthreads();
  tc::tc_fence_after();
  const uint32_t tmem = s_tmem;
  // chunk ch: columns 32 ch .. of A2 (into sA) and of -W^-1's rows (into the B tiles of its set)
  auto load_a = [&](int ch) {
    for (int u = tid; u < 32 * 32; u += kThreads) {
      const int c = 32 * ch + (u >> 5), q = 4 * (u & 31);
      const bool ok = q < npos;
      cp16(tc::smem_u32(sA + c * kFormLd + q), ok ? S + (int64_t)c * n + q : p.At, ok);
    }
  };
  // (-W^-1)^T: row x is M's row x up to its diagonal
  constexpr int kBu = NBO * 8 / kThreads;  // 16-byte units per thread and chunk
  float4 bx[kBu];
  auto load_b = [&](int ch) {
#pragma unroll
    for (int e = 0; e < kBu; ++e) {
      const int u = tid + e * kThreads, r = u >> 3, j = 32 * ch + 4 * (u & 7);
      bx[e] = make_float4(0.f, 0.f, 0.f, 0.f);
      if (j <= r && state == kQrBlockFast) bx[e] = *reinterpret_cast<const float4*>(M + r * NBO + j);
      if (j + 1 > r) bx[e].y = 0.f;
      if (j + 2 > r) bx[e].z = 0.f;
      if (j + 3 > r) bx[e].w = 0.f;
    }
  };
#pragma unroll
  for (int ch = 0; ch < 4; ++ch) {
    load_a(ch);
    asm volatile("cp.async.commit_group;" ::: "memory");
  }
  load_b(0);
  float y[64];
#pragma unroll
  for (int l = 0; l < 64; ++l) y[l] = 0.f;
  const uint32_t lane_base = tmem + ((uint32_t)(32 * (warp & 3)) << 16) + (uint32_t)(64 * (warp >> 2));
  auto drain = [&](int ch) {
    float v[32];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      tc::tmem_ld32(lane_base + (uint32_t)(ch * NBO + 32 * h), v);
#pragma unroll
      for (int l = 0; l < 32; ++l) y[32 * h + l] += v[l];
    }
  };
  bool bad = false;
  int issued = 0;
#pragma unroll
  for (int ch = 0; ch < 4; ++ch) {
    uint8_t* set = ops + (ch & 1) * 4 * kTile;
    if (ch >= 2) {
      // the set's previous products are done
      bad = bad || !__all_sync(0xffffffffu, tc::mbar_wait(&bar[ch - 2], 0, kWaitNs));
      if (!bad) {
        tc::tc_fence_after();
        drain(ch - 2);
        tc::tc_fence_before();
      }
    }
#pragma unroll
    for (int e = 0; e < kBu; ++e) {
      const int u = tid + e * kThreads, off = swz16(u >> 3, u & 7);
      *reinterpret_cast<float4*>(set + 2 * kTile + off) = bx[e];
      *reinterpret_cast<float4*>(set + 3 * kTile + off) = lo4(bx[e]);
    }
    if (ch < 3) load_b(ch + 1);
    if (ch == 0) asm volatile("cp.async.wait_group 3;" ::: "memory");
    if (ch == 1) asm volatile("cp.async.wait_group 2;" ::: "memory");
    if (ch == 2) asm volatile("cp.async.wait_group 1;" ::: "memory");
    if (ch == 3) asm volatile("cp.async.wait_group 0;" ::: "memory");
    if (__syncthreads_or(bad)) {  // every thread's copies of this chunk have landed
      bad = true;
      break;
    }
    for (int u = tid; u < NBO * 8; u += kThreads) {
      const int r = u & (NBO - 1), q = u >> 7;  // position r, columns 32 ch + 4 q ..
      const float* src = sA + (32 * ch + 4 * q) * kFormLd + r;
      const float4 x = make_float4(src[0], src[kFormLd], src[2 * kFormLd], src[3 * kFormLd]);
      const int off = swz16(r, q);
      *reinterpret_cast<float4*>(set + off) = x;
      *reinterpret_cast<float4*>(set + kTile + off) = lo4(x);
    }
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    __syncthreads();
    if (tid == 0) {
      tc::tc_fence_after();
      const uint32_t a = tc::smem_u32(set);
      mma_chunk(tmem + (uint32_t)(ch * NBO), a, a + kTile, a + 2 * kTile, a + 3 * kTile);
      tc::umma_commit(&bar[ch]);
    }
    issued = ch + 1;
  }
  for (int ch = max(0, issued - 2); ch < issued; ++ch) {
    const bool ok = __all_sync(0xffffffffu, tc::mbar_wait(&bar[ch], 0, kWaitNs));
    bad = bad || !ok;
    if (!bad) {
      tc::tc_fence_after();
      drain(ch);
    }
  }
  if (bad) atomicOr(p.status, kStatusTimeout);
  asm volatile("cp.async.wait_all;" ::: "memory");
  tc::tc_fence_before();
  __syncthreads();
  if (warp == 0) {
    tc::tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512));
  }
  // this thread: position r, columns c0 .. c0 + 63; the rows of Vpos through shared memory
  const int r = 32 * (warp & 3) + lane, c0 = 64 * (warp >> 2);
#pragma unroll
  for (int l = 0; l < 16; ++l)
    *reinterpret_cast<float4*>(sA + r * kFormLd + c0 + 4 * l) =
        make_float4(y[4 * l], y[4 * l + 1], y[4 * l + 2], y[4 * l + 3]);
  if (r < npos) {
    const int64_t vt = b * nn + (int64_t)(k0 + c0) * n + pos0 + r;
#pragma unroll
    for (int l = 0; l < 64; ++l) {
      p.Vt[vt + (int64_t)l * n] = y[l];
      p.Vt_lo[vt + (int64_t)l * n] = tc::tf32_lo(y[l]);
    }
  }
  __syncthreads();
  const int64_t vp = ((int64_t)b * n + pos0) * NBO;
  for (int i = warp; i < npos; i += kThreads / 32) {
    const float4 v = *reinterpret_cast<const float4*>(sA + i * kFormLd + 4 * lane);
    *reinterpret_cast<float4*>(p.Vpos + vp + i * NBO + 4 * lane) = v;
    *reinterpret_cast<float4*>(p.Vpos_lo + vp + i * NBO + 4 * lane) = lo4(v);
  }
}

// dynamic shared memory above 48 KB, once per device (one bit per device that has it)
cudaError_t prepare_kernels() {
  static std::atomic<uint64_t> done{0};
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) dev = 0;
  const uint64_t bit = (dev >= 0 && dev < 64) ? uint64_t(1) << dev : 0;
  if (bit && (done.load(std::memory_order_relaxed) & bit)) return cudaSuccess;
  cudaError_t e = cudaFuncSetAttribute(qr_gram_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kGramSmem);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(qr_core_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kCoreSmem);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(qr_form_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kFormSmem);
  if (e == cudaSuccess) done.fetch_or(bit, std::memory_order_relaxed);
  return e;
}

}  // namespace

cudaError_t qr_block_fast(const QrBlockArgs& p, int batch, cudaStream_t s) {
  cudaError_t e = prepare_kernels();
  if (e != cudaSuccess) return e;
  const int m = p.n - p.k0, nch = (m + 31) / 32;
  const double mk = (double)m * batch;
  // CTAs per matrix: at least four chunks each, about two per SM over the batch, in clusters of
  // up to 8 and at most kQrGramParts clusters (the core kernel adds their partial sums)
  const int want = std::max(1, std::min(std::max(1, nch / 4), std::max(1, 304 / batch)));
  int cs = 1;
  while (2 * cs <= std::min(8, want)) cs *= 2;
  const int ncl = std::max(1, std::min(kQrGramParts, want / cs));
  const int cper = (nch + cs * ncl - 1) / (cs * ncl);
  const bool gram = m > NBO;  // the core kernel forms the Gram matrix of a square block itself
  if (gram) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(cs * ncl, batch, 1);
    cfg.blockDim = dim3(kThreads, 1, 1);
    cfg.dynamicSmemBytes = kGramSmem;
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = cs;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    ProfScope prof(kFamQrPanel, 2.0 * p.kbo * p.kbo * mk, 4.0 * p.kbo * mk, s);
    e = cudaLaunchKernelEx(&cfg, qr_gram_kernel, p, nch, cper, ncl);
    if (e != cudaSuccess) return e;
  }
  {
    ProfScope prof(kFamQrPanel, 2.0 * NBO * NBO * NBO * batch, 4.0 * 8.0 * NBO * NBO * batch, s);
    qr_core_kernel<<<batch, kThreads, kCoreSmem, s>>>(p, gram ? ncl : 0);
    e = cudaGetLastError();
    if (e != cudaSuccess) return e;
  }
  const int tiles = m > NBO ? (m - NBO + NBO - 1) / NBO : 0;
  ProfScope prof(kFamQrPanel, 1.0 * p.kbo * p.kbo * mk, 4.0 * 5.0 * p.kbo * mk, s);
  qr_form_kernel<<<dim3(kTBlocks + tiles, batch), kThreads, kFormSmem, s>>>(p);
  return cudaGetLastError();
}

}  // namespace soap
