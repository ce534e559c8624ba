// Batched Householder QR with explicit Q for the eigenbasis refresh
// (Alg. 1, "Eigenbasis Re-computation": Q <- QR(L_t Q).Q, every step as the
// appendix on eigh vs QR settles), with diag(R) >= 0, on tensor cores.
//
// The QR works on At = P^T (row j of At is column j of P), so every product of the
// blocked algorithm is a C = A B^T of K-major operands for the tcgen05 engine. It goes in
// blocks of 128 columns:
//
//   for each block of 128 rows of At at k0 (columns k0..k0+127 of P):
//     qr_block_fast (qr_block.cu) factors the block from its Gram matrix: the Householder
//       vectors as rows of Vt (row k0+a = v_a over positions k0..n-1, zeros before its pivot)
//       and as columns of Vpos (position-major), and the block's T (H_k0 ... H_k0+127 =
//       I - V T V^T); where it leaves a matrix to the column loop, qr_panel_kernel factors
//       that matrix's block in 32-column panels in distributed shared memory, with the same
//       results;
//     VTr = V T^T                                   (tensor cores, K = 128)
//     trailing rows r >= k0+128: a_r <- a_r - (a_r V) T V^T, i.e.
//       W  = At_trail Vt^T                          (tensor cores: N = 128, K = positions)
//       At_trail -= W VTr^T                         (tensor cores: K = 128, C read in place)
//   then Q^T is accumulated backwards from diag(d) (d_j = sign of R_jj) a superblock of three or
//   four blocks, with one T, at a time, Q^T <- Q^T (I - V T^T V^T), on operands in bf16 planes:
//       W = (Qt_sub Vt^T) T^T ;  Qt_sub -= W V^T
//   and Q = (Q^T)^T. (A block at a time, in TF32, this took 2.2 of the 6.6 ms of 16 matrices of
//   2048 rows; so 1.4, and 0.5 more for the superblocks' T.)
//
// The column loop's panel of an n x n matrix spans up to n positions; it is spread over a
// thread-block cluster of ceil((n-k0)/512) CTAs (<= 16 for n <= 8192), 512 positions each, or,
// on a device that cannot run 16-CTA clusters of it, 1024 positions in clusters of <= 8 (a
// factor of at most 1024 rows takes one CTA of 1024 positions). Each Householder step needs
// one cluster-wide reduction: the squared norm of the column below the pivot and its dot
// products with the later panel columns are reduced together (the dot products with v
// follow from them once the reflector is known), and the partial sums are combined through
// distributed shared memory at one cluster barrier. No CTA waits on a flag: the only waits
// are hardware cluster barriers that every CTA of the cluster reaches unconditionally, and
// the tensor-core block product's mbarrier waits, which give up after a bounded time.
//
// Reflector convention (LAPACK larfg): for x = A[p:n, p] with alpha = x_1 and
// sigma = ||x_2:||^2, beta = -sign(alpha) ||x||, v = x / (alpha - beta) with v_1 = 1,
// tau = (beta - alpha) / beta, so H x = beta e_1 and R_pp = beta; sigma = 0 gives H = I
// and R_pp = alpha. The sign convention diag(R) >= 0 then negates column p of Q
// wherever R_pp < 0; it costs nothing because the backward accumulation starts from
// diag(d_1..d_n), d_p = sign of R_pp, instead of I. A column with
// ||x|| <= tol * ||P||_F is treated as exactly zero: H = I, R_pp = 0, d_p = +1, and the
// column is flagged in skip[]. (The convention matters beyond the sign: the columns of
// Q that complete a rank-deficient P are H_1 ... H_p-1 e_p, which depend on it.)
#include <cooperative_groups.h>

#include <algorithm>
#include <atomic>

#include "profile.h"
#include "qr_block.h"
#include "soap_internal.h"
#include "tc_ptx.h"

namespace cg = cooperative_groups;

namespace soap {

namespace {

constexpr int NB = 32;            // panel width
constexpr int NBO = 128;          // block width: the trailing matrix is updated once per block
constexpr int PT = 512;           // threads per panel CTA
constexpr int MAXC = 16;          // largest cluster (16 needs the non-portable cluster size)
constexpr int NWARP = PT / 32;
constexpr int NREST = NBO - NB;   // most block rows after a panel
constexpr int KSPLIT = 8;         // split-K workspace: 8 partial n x NBO products (shorter ones split up to 16 ways)
constexpr uint64_t kWaitNs = 2000000000ull;  // bound of every mbarrier wait in the panel kernel

// lo part of x for the tensor-core products: x - trunc_tf32(x) rounded to the nearest tf32
__device__ __forceinline__ float tf32_lo(float x) {
  uint32_t r;
  asm("cvt.rna.tf32.f32 %0, %1;" : "=r"(r) : "f"(x - __uint_as_float(__float_as_uint(x) & 0xFFFFE000u)));
  return __uint_as_float(r);
}

struct PanelArgs {
  float* At;           // [batch][n][n] working P^T
  float* Vt;           // [batch][n][n] Householder vectors as rows
  float* Vt_lo;
  float* Vpos;         // [batch][n][NBO] the block's Householder vectors, position-major
  float* Vpos_lo;
  float* T;            // [batch][NBO][NBO] the block's T (upper triangular)
  float* T_lo;
  float* Tt;           // [batch][NBO][NBO] T^T
  float* Tt_lo;
  float* Ypart;        // [batch][MAXC][NBO][NB] per-CTA partial products S V_panel (at first the
                       // Gram matrices' place, which block_left reads before any is written)
  uint8_t* skip;       // [batch][n]
  float* dsign;        // [batch][n] sign of R_pp (+1 for zero columns)
  const float* thresh; // [batch]
  const int* state;    // [batch] what qr_block_fast did with this block
  int* status;
  int n, k0, kbo;      // block start and width
};

// x = hi + lo with hi = tf32(x) rounded to nearest and lo = tf32(x - hi): both as tf32 bits
__device__ __forceinline__ void tf32_split(float x, uint32_t& hi, uint32_t& lo) {
  asm("cvt.rna.tf32.f32 %0, %1;" : "=r"(hi) : "f"(x));
  asm("cvt.rna.tf32.f32 %0, %1;" : "=r"(lo) : "f"(x - __uint_as_float(hi)));
}

// d += a b for a 16 x 8 (rows) tf32 A fragment and an 8 x 8 (columns) B fragment, fp32 d
__device__ __forceinline__ void mma_tf32_16x8x8(float (&d)[4], const uint32_t (&a)[4], const uint32_t (&b)[2]) {
  asm volatile(
      "mma.sync.aligned.m16n8k8.row.col.f32.tf32.tf32.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, "
      "{%0, %1, %2, %3};"
      : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b[0]), "r"(b[1]));
}

// One 32-column panel of a block, spread over the cluster: CTA c holds positions k + c*COLS .. of the
// panel rows in shared memory (row stride LDS, 16-byte aligned rows). A function of its own, so that
// the loop over the panels takes no registers from it (inlined, with 128 registers and spills, four
// panels of a 2048-factor took 486 us instead of 441).
template <int COLS>
__device__ __noinline__ void panel(const PanelArgs& p, int k, uint32_t tmem) {
  constexpr int LDS = COLS + 4;
  cg::cluster_group cluster = cg::this_cluster();
  const int c = (int)cluster.block_rank();
  const int C = (int)cluster.num_blocks();
  const int b = blockIdx.y;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  extern __shared__ float4 smem_dyn[];
  float* sA = reinterpret_cast<float*>(smem_dyn);  // [NB][LDS]: panel row jj, position offset i
  __shared__ float s_part[2][NB];        // this CTA's partial [sigma | x . a_c]
  __shared__ float s_pv[2][NB];          // rank 0: pivot-row values [alpha | a_c,pivot]
  __shared__ float s_scal[2];            // tau and 1 / v0 of the current reflector
  __shared__ float s_w[NB];              // v^T a_c
  __shared__ __align__(16) float s_wl[NB];  // v^T a_(j+l) by offset l from the current row j
  __shared__ float s_red[NWARP][NB];     // per-warp partial sums of the register path
  __shared__ float s_tau[NB];
  __shared__ int s_skip[NB];
  __shared__ float s_dsign[NB];
  __shared__ float s_T[NB][NB + 1];
  __shared__ float s_Y[NBO][NB + 1];     // rank 0: S V_panel summed over the cluster
  __shared__ __align__(16) float s_Z[NREST][NB];  // (S_rest V_panel) T_panel, the in-block update
  // S V_panel: with 512 positions per CTA on the tensor cores (tcgen05): SV_STG chunks of S
  // (128 rows x 32 positions, 128-byte-swizzled) in flight, and two sets of S's lo part and
  // V's hi and lo parts; with 1024 positions as warp-level MMAs over STG staged chunks of
  // 128 x 36
  constexpr int STG = 2;
  constexpr int SV_STG = 4;
  constexpr int A_BYTES = NBO * 32 * 4;
  constexpr int B_BYTES = NB * 32 * 4;
  constexpr int SV_BYTES = COLS == PT ? SV_STG * A_BYTES + 2 * (A_BYTES + 2 * B_BYTES) + 1024 : STG * NBO * 36 * 4;
  __shared__ __align__(1024) uint8_t s_sv[SV_BYTES];
  __shared__ __align__(8) uint64_t s_mma_bar[2];

  const int n = p.n, k0 = p.k0, kbo = p.kbo;
  const int kb = min(NB, n - k);
  const int jb = k - k0;                // panel offset inside its block
  const int nrest = kbo - jb - kb;      // block rows after the panel
  const int64_t nn = (int64_t)n * n;
  float* At = p.At + (int64_t)b * nn;
  const int pos0 = k + c * COLS;  // first position held by this CTA
  const int npos = max(0, min(COLS, n - pos0));  // a multiple of 4

  const int npad = (npos + 31) & ~31;  // positions read by the chunked S V product
  {
    const int q4n = npad / 4;
    for (int e = tid; e < NB * q4n; e += PT) {
      const int jj = e / q4n, i = 4 * (e % q4n);
      const bool ok = jj < kb && i < npos;
      const float* src = ok ? At + (int64_t)(k + jj) * n + pos0 + i : At;
      const uint32_t d = static_cast<uint32_t>(__cvta_generic_to_shared(&sA[jj * LDS + i]));
      asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(d), "l"(src), "r"(ok ? 16 : 0) : "memory");
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
    asm volatile("cp.async.wait_group 0;" ::: "memory");
  }
  __syncthreads();
  const float thresh = p.thresh[b];
  int nonfinite = 0;

  if constexpr (COLS == PT) {
    // One position per thread: thread tid holds the panel rows' values at position tid in
    // registers, the current row first (a[l] = row j + l; rows past the panel are zero), so
    // that the per-column dot products and the reflector's update never touch shared memory;
    // only v (row j) is written back, for the phases after the loop.
    const int i = tid;
    const bool have = i < npos;
    float a[NB];
#pragma unroll
    for (int l = 0; l < NB; ++l) a[l] = (have && l < kb) ? sA[l * LDS + i] : 0.f;
    for (int j = 0; j < kb; ++j) {
      const int par = j & 1;
      // this position's share of sigma (l = 0) and of x . a_(j+l) (l > 0), for positions
      // strictly after the pivot (pivot = local position j of rank 0)
      const float x = (have && (c != 0 || i > j)) ? a[0] : 0.f;
      float v[NB];
      // transposing butterfly over the warp: lane l ends with the warp's sum for row j + l
#define SOAP_BFLY(o, nh)                                                   \
  {                                                                        \
    const bool up = (lane & (o)) != 0;                                     \
    _Pragma("unroll") for (int q = 0; q < (nh); ++q) {                     \
      const float keep = up ? v[q + (nh)] : v[q];                          \
      const float send = up ? v[q] : v[q + (nh)];                          \
      v[q] = keep + __shfl_xor_sync(0xffffffffu, send, (o));               \
    }                                                                      \
  }
      if (kb - j > NB / 2) {
#pragma unroll
        for (int l = 0; l < NB; ++l) v[l] = x * a[l];
        SOAP_BFLY(16, 16)
        SOAP_BFLY(8, 8)
        SOAP_BFLY(4, 4)
        SOAP_BFLY(2, 2)
        SOAP_BFLY(1, 1)
      } else {
        // at most 16 rows left (the rest of a[] is zero): the butterfly over the 16 live values
        // within each half-warp (lane l ends with row j + (l mod 16)), then across the halves
#pragma unroll
        for (int l = 0; l < NB / 2; ++l) v[l] = x * a[l];
        SOAP_BFLY(8, 8)
        SOAP_BFLY(4, 4)
        SOAP_BFLY(2, 2)
        SOAP_BFLY(1, 1)
        v[0] += __shfl_xor_sync(0xffffffffu, v[0], 16);
      }
#undef SOAP_BFLY
      s_red[warp][lane] = v[0];
      // rank 0's pivot position: alpha and the later rows' values there
      if (c == 0 && i == j) {
#pragma unroll
        for (int l = 0; l < NB; ++l)
          if (j + l < kb) s_pv[par][j + l] = a[l];
      }
      __syncthreads();
      if (warp == 0) {
        float sum = 0.f;
#pragma unroll
        for (int w = 0; w < NWARP; ++w) sum += s_red[w][lane];
        if (j + lane < kb) s_part[par][j + lane] = sum;
      }
      cluster.sync();
      // threads j..kb-1 reduce sigma and their own column's sum (in the same fixed order, so
      // they all derive the same reflector) and form v^T a_tid
      if (warp == 0) {
        s_wl[lane] = 0.f;
        __syncwarp();
      }
      if (tid >= j && tid < kb) {
        float ps[MAXC], pd[MAXC];
#pragma unroll
        for (int q = 0; q < MAXC; ++q) {
          if (q < C) {
            const float* rp = cluster.map_shared_rank(&s_part[par][0], q);
            ps[q] = rp[j];
            pd[q] = rp[tid];
          }
        }
        const float* pv0 = cluster.map_shared_rank(&s_pv[par][0], 0);
        const float alpha = pv0[j], apiv = pv0[tid];
        float d = 0.f, sigma = 0.f;
#pragma unroll
        for (int q = 0; q < MAXC; ++q) {
          if (q < C) {
            sigma += ps[q];
            d += pd[q];
          }
        }
        const float xnorm = sqrtf(fmaf(alpha, alpha, sigma));
        const bool skip = !(xnorm > thresh);
        float tau = 0.f, v0 = 1.f, rsign = 1.f;
        if (!skip) {
          if (sigma == 0.f) {
            rsign = alpha < 0.f ? -1.f : 1.f;   // H = I, R_pp = alpha
          } else {
            const float beta = alpha >= 0.f ? -xnorm : xnorm;
            v0 = alpha - beta;                   // same sign as alpha: no cancellation
            tau = (beta - alpha) / beta;
            rsign = beta < 0.f ? -1.f : 1.f;
          }
        }
        if (tid == j) {
          if (!isfinite(xnorm)) nonfinite = 1;
          s_tau[j] = tau;
          s_skip[j] = skip ? 1 : 0;
          s_dsign[j] = rsign;
          s_scal[0] = tau;
          s_scal[1] = tau != 0.f ? 1.f / v0 : 0.f;
        } else {
          s_wl[tid - j] = tau != 0.f ? apiv + d / v0 : 0.f;  // v^T a_tid, with v = x / v0 after the pivot
        }
      }
      __syncthreads();
      const float tau = s_scal[0], rv0 = s_scal[1];
      // v at this position (x / v0 after the pivot, 1 at it) and H_j = I - tau v v^T on the
      // later rows, shifting them down one register; positions before the pivot only shift
      if (have && (c != 0 || i >= j)) {
        const bool at_pivot = (c == 0 && i == j);
        const float vi = at_pivot ? 1.f : a[0] * rv0;
        if (!at_pivot) sA[j * LDS + i] = vi;
        if (tau != 0.f) {
          const float tv = tau * vi;
#pragma unroll
          for (int l4 = 0; l4 < NB / 4; ++l4) {
            const float4 w4 = reinterpret_cast<const float4*>(s_wl)[l4];
            if (l4 > 0) a[4 * l4 - 1] = fmaf(-tv, w4.x, a[4 * l4]);
            a[4 * l4] = fmaf(-tv, w4.y, a[4 * l4 + 1]);
            a[4 * l4 + 1] = fmaf(-tv, w4.z, a[4 * l4 + 2]);
            a[4 * l4 + 2] = fmaf(-tv, w4.w, a[4 * l4 + 3]);
          }
          a[NB - 1] = 0.f;
        } else {
#pragma unroll
          for (int l = 0; l < NB - 1; ++l) a[l] = a[l + 1];
          a[NB - 1] = 0.f;
        }
      } else {
#pragma unroll
        for (int l = 0; l < NB - 1; ++l) a[l] = a[l + 1];
        a[NB - 1] = 0.f;
      }
      __syncthreads();  // s_wl, s_red and s_scal are rewritten by the next column
    }
  } else {
    for (int j = 0; j < kb; ++j) {
      const int par = j & 1;
      // positions strictly after the pivot (pivot = local position j of rank 0)
      const int ibeg = (c == 0) ? j + 1 : 0;
      // partial sums over this CTA: sigma (cc = j) and x . a_cc (cc > j), kept locally; after
      // the cluster barrier the threads that need them read every CTA's copy. Warp w takes
      // columns j + w and j + w + 16 in one pass over x (kb - j <= 32 columns).
      {
        const int c1 = j + warp, c2 = c1 + NWARP;
        if (c1 < kb) {
          const bool h2 = c2 < kb;
          float a0 = 0.f, a1 = 0.f, a2 = 0.f, a3 = 0.f, b0 = 0.f, b1 = 0.f, b2 = 0.f, b3 = 0.f;
          const float* xr = sA + j * LDS;
          const float* r1 = sA + c1 * LDS;
          const float* r2 = sA + (h2 ? c2 : c1) * LDS;
          int i = ibeg + lane;
          for (; i + 96 < npos; i += 128) {
            const float x0 = xr[i], x1 = xr[i + 32], x2 = xr[i + 64], x3 = xr[i + 96];
            a0 = fmaf(x0, r1[i], a0);
            a1 = fmaf(x1, r1[i + 32], a1);
            a2 = fmaf(x2, r1[i + 64], a2);
            a3 = fmaf(x3, r1[i + 96], a3);
            b0 = fmaf(x0, r2[i], b0);
            b1 = fmaf(x1, r2[i + 32], b1);
            b2 = fmaf(x2, r2[i + 64], b2);
            b3 = fmaf(x3, r2[i + 96], b3);
          }
          for (; i < npos; i += 32) {
            const float x0 = xr[i];
            a0 = fmaf(x0, r1[i], a0);
            b0 = fmaf(x0, r2[i], b0);
          }
          float da = (a0 + a1) + (a2 + a3), db = (b0 + b1) + (b2 + b3);
#pragma unroll
          for (int o = 16; o > 0; o >>= 1) {
            da += __shfl_xor_sync(0xffffffffu, da, o);
            db += __shfl_xor_sync(0xffffffffu, db, o);
          }
          if (lane == 0) {
            s_part[par][c1] = da;
            if (h2) s_part[par][c2] = db;
          }
        }
      }
      if (c == 0 && tid >= j && tid < kb) s_pv[par][tid] = sA[tid * LDS + j];  // alpha (tid == j), a_tid at the pivot
      cluster.sync();
      // threads j..kb-1 reduce sigma and their own column's sum (in the same fixed order, so
      // they all derive the same reflector) and form v^T a_tid
      if (tid >= j && tid < kb) {
        float ps[MAXC], pd[MAXC];
#pragma unroll
        for (int q = 0; q < MAXC; ++q) {
          if (q < C) {
            const float* rp = cluster.map_shared_rank(&s_part[par][0], q);
            ps[q] = rp[j];
            pd[q] = rp[tid];
          }
        }
        const float* pv0 = cluster.map_shared_rank(&s_pv[par][0], 0);
        const float alpha = pv0[j], apiv = pv0[tid];
        float d = 0.f, sigma = 0.f;
#pragma unroll
        for (int q = 0; q < MAXC; ++q) {
          if (q < C) {
            sigma += ps[q];
            d += pd[q];
          }
        }
        const float xnorm = sqrtf(fmaf(alpha, alpha, sigma));
        const bool skip = !(xnorm > thresh);
        float tau = 0.f, v0 = 1.f, rsign = 1.f;
        if (!skip) {
          if (sigma == 0.f) {
            rsign = alpha < 0.f ? -1.f : 1.f;   // H = I, R_pp = alpha
          } else {
            const float beta = alpha >= 0.f ? -xnorm : xnorm;
            v0 = alpha - beta;                   // same sign as alpha: no cancellation
            tau = (beta - alpha) / beta;
            rsign = beta < 0.f ? -1.f : 1.f;
          }
        }
        if (tid == j) {
          if (!isfinite(xnorm)) nonfinite = 1;
          s_tau[j] = tau;
          s_skip[j] = skip ? 1 : 0;
          s_dsign[j] = rsign;
          s_scal[0] = tau;
          s_scal[1] = tau != 0.f ? 1.f / v0 : 0.f;
        } else if (tau != 0.f) {
          s_w[tid] = apiv + d / v0;  // v^T a_tid, with v = x / v0 after the pivot
        }
      }
      __syncthreads();
      const float tau = s_scal[0], rv0 = s_scal[1];

      // v after the pivot (x / v0, or 0 where H = I), and H_j = I - tau v v^T on the later
      // panel rows; every thread owns its positions
      const int piv = (c == 0) ? j : 0;  // local positions >= this take part
      for (int i = piv + tid; i < npos; i += PT) {
        const bool at_pivot = (c == 0 && i == j);
        const float vi = at_pivot ? 1.f : sA[j * LDS + i] * rv0;
        if (!at_pivot) sA[j * LDS + i] = vi;
        if (tau != 0.f) {
          const float tv = tau * vi;
          for (int cc = j + 1; cc < kb; ++cc) sA[cc * LDS + i] = fmaf(-tv, s_w[cc], sA[cc * LDS + i]);
        }
      }
      __syncthreads();
    }
  }
  if (nonfinite) atomicOr(p.status, kStatusQrBreakdown);

  // V with its unit diagonal and zeros before it (rank 0 holds the first kb positions)
  if (c == 0) {
    for (int e = tid; e < kb * kb; e += PT) {
      const int jj = e / kb, i = e % kb;
      if (i < jj) sA[jj * LDS + i] = 0.f;
      else if (i == jj) sA[jj * LDS + i] = 1.f;
    }
  }
  __syncthreads();

  // V as rows of Vt (zeros at the block's positions before the panel) and as columns jb..
  // of the block's position-major Vpos
  float* Vt = p.Vt + (int64_t)b * nn;
  float* Vt_lo = p.Vt_lo + (int64_t)b * nn;
  float* Vpos = p.Vpos + (int64_t)b * n * NBO;
  float* Vpos_lo = p.Vpos_lo + (int64_t)b * n * NBO;
  {
    const int q4n = npos / 4;
    for (int e = tid; e < kb * q4n; e += PT) {
      const int jj = e / q4n, q = e - jj * q4n;
      const int64_t o = (int64_t)(k + jj) * n + pos0 + 4 * q;
      const float4 v = *reinterpret_cast<const float4*>(&sA[jj * LDS + 4 * q]);
      *reinterpret_cast<float4*>(Vt + o) = v;
      *reinterpret_cast<float4*>(Vt_lo + o) = make_float4(tf32_lo(v.x), tf32_lo(v.y), tf32_lo(v.z), tf32_lo(v.w));
    }
  }
  for (int e = tid; e < npos * (NB / 4); e += PT) {
    const int i = e >> 3, g4 = 4 * (e & 7);  // rows kb.. of sA are zero
    const float4 v = make_float4(sA[g4 * LDS + i], sA[(g4 + 1) * LDS + i], sA[(g4 + 2) * LDS + i], sA[(g4 + 3) * LDS + i]);
    const int64_t o = (int64_t)(pos0 + i) * NBO + jb + g4;
    *reinterpret_cast<float4*>(Vpos + o) = v;
    *reinterpret_cast<float4*>(Vpos_lo + o) = make_float4(tf32_lo(v.x), tf32_lo(v.y), tf32_lo(v.z), tf32_lo(v.w));
  }
  if (c == 0) {
    for (int jj = 0; jj < kb; ++jj)
      for (int i = tid; i < jb; i += PT) {
        const int64_t o = (int64_t)(k + jj) * n + k0 + i;
        Vt[o] = 0.f;
        Vt_lo[o] = 0.f;
      }
    for (int e = tid; e < jb * NB; e += PT) {
      const int64_t o = (int64_t)(k0 + e / NB) * NBO + jb + e % NB;
      Vpos[o] = 0.f;
      Vpos_lo[o] = 0.f;
    }
  }
  __syncthreads();  // this CTA's Vt rows are read back below

  // Y = S V_panel over this CTA's positions, S = the block's rows k0 .. k0+kbo-1: the block's
  // Householder vectors so far (rows before the panel's end, from Vt) and the block rows still
  // to be factored (from At), with both operands split into tf32 hi and lo parts (four
  // products: fp32 accuracy), each 32-position chunk summed afresh and added to fp32 registers,
  // so that the tensor core's own accumulation never runs longer than 32 positions.
  if constexpr (COLS == PT) {
    // On the tcgen05 tensor cores: D[128 x 32] (tensor memory) = S chunk (A: 128 rows x 32
    // positions) x V chunk^T (B: 32 rows x 32 positions), both K-major in the 128-byte-swizzled
    // layout. S's rows other than the panel's are copied with cp.async straight into that
    // layout, SV_STG - 1 chunks ahead, and each thread forms the lo part of the units it copied;
    // the panel's rows of S and the V chunk (hi and lo) come from sA. Two accumulators and two
    // lo sets alternate: while the MMAs of chunk ch run, warps 0-3 drain chunk ch-1 (warp w
    // reads lanes 32w..) and its S stage is refilled.
    uint8_t* sv = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(s_sv) + 1023) & ~uintptr_t(1023));
    uint8_t* st_a = sv;                          // [SV_STG] S chunks (fp32, read by the MMA as its hi part)
    uint8_t* st_lo = sv + SV_STG * A_BYTES;      // [2] S lo | V hi | V lo
    constexpr int LO_SET = A_BYTES + 2 * B_BYTES;
    const int nchunk = (npos + 31) / 32;
    if (tid == 0) {
      tc::mbar_init(&s_mma_bar[0], 1);
      tc::mbar_init(&s_mma_bar[1], 1);
      asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncthreads();
    // byte offset of 16-byte unit q of row r in a tile of 128-byte rows, swizzled within
    // 1024-byte groups of 8 rows
    auto swz16 = [](int r, int q) { return (r >> 3) * 1024 + (r & 7) * 128 + ((q ^ (r & 7)) << 4); };
    auto issue = [&](int ch) {
      uint8_t* dst = st_a + (ch % SV_STG) * A_BYTES;
      for (int u = tid; u < NBO * 8; u += PT) {
        const int r = u >> 3, q = u & 7;
        if (r >= jb && r < jb + NB) continue;  // the panel's own rows: V, from sA
        const int row = k0 + r, i = ch * 32 + 4 * q;
        const bool ok = r < kbo && i < npos;  // zero-filled outside the block and past the positions
        const float* src = ok ? (r < jb ? Vt : At) + (int64_t)row * n + pos0 + i : At;
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(tc::smem_u32(dst + swz16(r, q))),
                     "l"(src), "r"(ok ? 16 : 0)
                     : "memory");
      }
    };
    auto lo4 = [](float4 x) { return make_float4(tf32_lo(x.x), tf32_lo(x.y), tf32_lo(x.z), tf32_lo(x.w)); };
    float y[NB];
#pragma unroll
    for (int l = 0; l < NB; ++l) y[l] = 0.f;
    for (int st0 = 0; st0 < SV_STG - 1; ++st0) {
      if (st0 < nchunk) issue(st0);
      asm volatile("cp.async.commit_group;" ::: "memory");
    }
    int issued = 0;  // chunks whose MMAs were issued
    bool aborted = false, bad = false;
    for (int ch = 0; ch < nchunk; ++ch) {
      const int set = ch & 1;
      // this thread's copies of chunk ch have landed: their lo parts; the panel's rows of S and
      // the V chunk (hi and lo) from sA
      asm volatile("cp.async.wait_group %0;" ::"n"(SV_STG - 2) : "memory");
      {
        uint8_t* a = st_a + (ch % SV_STG) * A_BYTES;
        uint8_t* lo = st_lo + set * LO_SET;
        for (int u = tid; u < NBO * 8; u += PT) {
          const int r = u >> 3;
          if (r >= jb && r < jb + NB) continue;
          const int off = swz16(r, u & 7);
          *reinterpret_cast<float4*>(lo + off) = lo4(*reinterpret_cast<const float4*>(a + off));
        }
        uint8_t* bh = lo + A_BYTES;
        uint8_t* bl = bh + B_BYTES;
        for (int u = tid; u < NB * 8; u += PT) {
          const int jj = u >> 3, q = u & 7;
          const float4 x = *reinterpret_cast<const float4*>(&sA[jj * LDS + ch * 32 + 4 * q]);
          const float4 xl = lo4(x);
          const int off = swz16(jj, q), offa = swz16(jb + jj, q);
          *reinterpret_cast<float4*>(bh + off) = x;
          *reinterpret_cast<float4*>(bl + off) = xl;
          *reinterpret_cast<float4*>(a + offa) = x;
          *reinterpret_cast<float4*>(lo + offa) = xl;
        }
      }
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      if (__syncthreads_or(bad)) {
        aborted = true;
        break;
      }
      // the MMAs of chunk ch (its lo set and accumulator were released in the previous pass)
      if (tid == 0) {
        tc::tc_fence_after();
        constexpr uint32_t idesc = tc::idesc_tf32(NBO, NB);
        const uint32_t d = tmem + (uint32_t)(set * 32);
        const uint32_t a_hi = tc::smem_u32(st_a + (ch % SV_STG) * A_BYTES);
        const uint32_t a_lo = tc::smem_u32(st_lo + set * LO_SET);
        const uint32_t b_hi = a_lo + A_BYTES;
        const uint32_t b_lo = b_hi + B_BYTES;
#pragma unroll
        for (int kk = 0; kk < 4; ++kk) {
          const uint32_t off = kk * 32;  // 8 tf32 = 32 bytes along the positions
          tc::umma_tf32(d, tc::desc_sw128(a_lo + off), tc::desc_sw128(b_lo + off), idesc, kk != 0);
          tc::umma_tf32(d, tc::desc_sw128(a_lo + off), tc::desc_sw128(b_hi + off), idesc, 1u);
          tc::umma_tf32(d, tc::desc_sw128(a_hi + off), tc::desc_sw128(b_lo + off), idesc, 1u);
          tc::umma_tf32(d, tc::desc_sw128(a_hi + off), tc::desc_sw128(b_hi + off), idesc, 1u);
        }
        tc::umma_commit(&s_mma_bar[set]);
      }
      issued = ch + 1;
      // while they run: chunk ch-1's MMAs have completed, so its accumulator is drained and its
      // S stage refilled with chunk ch + SV_STG - 1
      if (ch >= 1) {
        bool ok = tc::mbar_wait(&s_mma_bar[(ch - 1) & 1], ((ch - 1) >> 1) & 1, kWaitNs);
        ok = __all_sync(0xffffffffu, ok);
        if (!ok) {
          bad = true;
        } else if (warp < 4) {
          float v[32];
          tc::tmem_ld32(tmem + (uint32_t)(((ch - 1) & 1) * 32) + ((uint32_t)(32 * warp) << 16), v);
#pragma unroll
          for (int l = 0; l < NB; ++l) y[l] += v[l];
        }
      }
      if (!bad && ch + SV_STG - 1 < nchunk) issue(ch + SV_STG - 1);
      asm volatile("cp.async.commit_group;" ::: "memory");
      tc::tc_fence_before();
    }
    // the last chunk's sum; after a wait that gave up, only the wait for every issued MMA (with
    // the full bound), so that the tensor memory is not freed under one
    bool ok_last = true;
    if (issued > 0)
      ok_last = __all_sync(0xffffffffu, tc::mbar_wait(&s_mma_bar[(issued - 1) & 1], ((issued - 1) >> 1) & 1, kWaitNs));
    if (!aborted && !bad && ok_last && issued > 0 && warp < 4) {
      float v[32];
      tc::tmem_ld32(tmem + (uint32_t)(((issued - 1) & 1) * 32) + ((uint32_t)(32 * warp) << 16), v);
#pragma unroll
      for (int l = 0; l < NB; ++l) y[l] += v[l];
    }
    if (aborted || bad || !ok_last) atomicOr(p.status, kStatusTimeout);
    asm volatile("cp.async.wait_all;" ::: "memory");
    tc::tc_fence_before();
    __syncthreads();
    tc::tc_fence_after();
    if (tid == 0) {  // every wait on them is over; the next panel sets them up again
      asm volatile("mbarrier.inval.shared::cta.b64 [%0];" ::"r"(tc::smem_u32(&s_mma_bar[0])) : "memory");
      asm volatile("mbarrier.inval.shared::cta.b64 [%0];" ::"r"(tc::smem_u32(&s_mma_bar[1])) : "memory");
    }
    // this CTA's partial product, kept in shared memory (the S stages are free) for the cluster
    if (warp < 4) {
      float* yp = reinterpret_cast<float*>(sv) + (32 * warp + lane) * NB;
#pragma unroll
      for (int l4 = 0; l4 < NB / 4; ++l4)
        *reinterpret_cast<float4*>(yp + 4 * l4) = make_float4(y[4 * l4], y[4 * l4 + 1], y[4 * l4 + 2], y[4 * l4 + 3]);
    }
  } else
  // With 1024 positions per CTA (factors of at most 1024 rows): S is streamed through shared
  // memory in 32-position chunks (cp.async, STG buffers, rows padded to 36 floats), and the
  // product runs as warp-level m16n8k8 TF32 MMAs. Warp w owns rows 16 (w mod 8) .. +15 and
  // columns 16 (w / 8) .. +15.
  {
    static_assert(NBO == 128 && NB == 32 && NWARP == 16, "8 x 2 warp tiles of 16 x 16");
    constexpr int CH = 32;       // positions per chunk
    constexpr int CHP = CH + 4;  // padded row stride of a staged chunk
    const int gq = lane >> 2, tg = lane & 3;
    const int m0 = 16 * (warp & 7), nb = 16 * (warp >> 3);
    float y[2][4];
#pragma unroll
    for (int e = 0; e < 4; ++e) y[0][e] = y[1][e] = 0.f;
    const int nchunk = (npos + CH - 1) / CH;
    auto issue = [&](int ch, int buf) {
      float* dst = reinterpret_cast<float*>(s_sv) + buf * NBO * CHP;
      for (int e = tid; e < NBO * (CH / 4); e += PT) {
        const int r = e / (CH / 4), q4 = e % (CH / 4);
        const int row = k0 + r, i = ch * CH + 4 * q4;
        const bool ok = r < kbo && i < npos;
        const float* src = ok ? ((row < k + kb) ? Vt : At) + (int64_t)row * n + pos0 + i : At;
        const uint32_t d = static_cast<uint32_t>(__cvta_generic_to_shared(dst + r * CHP + 4 * q4));
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(d), "l"(src), "r"(ok ? 16 : 0) : "memory");
      }
      asm volatile("cp.async.commit_group;" ::: "memory");
    };
    for (int st0 = 0; st0 < STG - 1; ++st0) {
      if (st0 < nchunk) issue(st0, st0);
      else asm volatile("cp.async.commit_group;" ::: "memory");
    }
    for (int ch = 0; ch < nchunk; ++ch) {
      if (ch + STG - 1 < nchunk) issue(ch + STG - 1, (ch + STG - 1) % STG);
      else asm volatile("cp.async.commit_group;" ::: "memory");  // keeps the group count uniform
      asm volatile("cp.async.wait_group %0;" ::"n"(STG - 1) : "memory");
      __syncthreads();
      const float* st = reinterpret_cast<const float*>(s_sv) + (ch % STG) * NBO * CHP;
      const int i0 = ch * CH;
      float d[2][4];
#pragma unroll
      for (int e = 0; e < 4; ++e) d[0][e] = d[1][e] = 0.f;
#pragma unroll
      for (int ks = 0; ks < CH / 8; ++ks) {
        // positions past npos are zero in the staged chunk and in V (zero-filled copies)
        const int kk = 8 * ks;
        const float av[4] = {st[(m0 + gq) * CHP + kk + tg], st[(m0 + gq + 8) * CHP + kk + tg],
                             st[(m0 + gq) * CHP + kk + tg + 4], st[(m0 + gq + 8) * CHP + kk + tg + 4]};
        uint32_t ah[4], al[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) tf32_split(av[e], ah[e], al[e]);
#pragma unroll
        for (int nt = 0; nt < 2; ++nt) {
          const float* vr = sA + (nb + 8 * nt + gq) * LDS + i0 + kk + tg;
          uint32_t bh[2], bl[2];
          tf32_split(vr[0], bh[0], bl[0]);
          tf32_split(vr[4], bh[1], bl[1]);
          mma_tf32_16x8x8(d[nt], al, bl);
          mma_tf32_16x8x8(d[nt], al, bh);
          mma_tf32_16x8x8(d[nt], ah, bl);
          mma_tf32_16x8x8(d[nt], ah, bh);
        }
      }
#pragma unroll
      for (int nt = 0; nt < 2; ++nt)
#pragma unroll
        for (int e = 0; e < 4; ++e) y[nt][e] += d[nt][e];
      __syncthreads();  // this buffer is refilled STG - 1 chunks later
    }
    float* yp = p.Ypart + ((int64_t)b * MAXC + c) * NBO * NB;
#pragma unroll
    for (int nt = 0; nt < 2; ++nt) {
      const int col = nb + 8 * nt + 2 * tg;
      *reinterpret_cast<float2*>(yp + (m0 + gq) * NB + col) = make_float2(y[nt][0], y[nt][1]);
      *reinterpret_cast<float2*>(yp + (m0 + gq + 8) * NB + col) = make_float2(y[nt][2], y[nt][3]);
    }
  }
  // T_panel from the Gram rows of Y, then U = X T_panel (in place) and Z (rows after the panel);
  // every thread of the CTA takes part (the barriers inside)
  auto form_tuz = [&]() {
    // T of the panel from its Gram matrix g (rows jb.. of Y): T^-1 = diag(1/tau) + striu(g)
    // (H_1 ... H_kb = I - V T V^T); a reflector with tau = 0 (v = 0) gets a zero row and column.
    // Warp w solves columns w and w + 16 by back substitution, lane i holding x_i:
    //   x_i = tau_i (delta_{i,cc} - sum_{i < l <= cc} g_il x_l)   (tau_i read as 1 where it is 0)
    // Each solved x_l is broadcast once and every lane i < l adds g_il x_l to its running sum,
    // so a step costs one shuffle instead of a warp-wide reduction.
    for (int cc = warp; cc < NB; cc += NWARP) {
      float x = 0.f, acc = 0.f;
      for (int l = cc; l >= 0; --l) {
        const float g = s_Y[jb + lane][l];
        if (lane == l) {
          const float tl = l < kb ? s_tau[l] : 0.f;
          x = ((l == cc ? 1.f : 0.f) - acc) * (tl != 0.f ? tl : 1.f);
        }
        const float xl = __shfl_sync(0xffffffffu, x, l);
        if (lane < l) acc = fmaf(g, xl, acc);
      }
      const bool live = cc < kb && s_tau[cc] != 0.f;
      s_T[lane][cc] = (live && lane <= cc && lane < kb && s_tau[lane] != 0.f) ? x : 0.f;
    }
    __syncthreads();
    // U = X T_panel with X = V_before^T V_panel (rows 0..jb-1 of Y), in place, and
    // Z = (S_rest V_panel) T_panel for the block rows after the panel: thread (r, g) forms
    // columns 8g .. 8g+7 of row r
    {
      const int r = tid >> 2, g8 = (tid & 3) * 8;
      const bool act = r < kbo && (r < jb || r >= jb + kb);
      float x[NB];
#pragma unroll
      for (int l = 0; l < NB; ++l) x[l] = act ? s_Y[r][l] : 0.f;
      __syncthreads();  // every row is read before U overwrites it
      if (act) {
#pragma unroll
        for (int u = 0; u < 8; ++u) {
          const int cc = g8 + u;
          float acc = 0.f;
#pragma unroll
          for (int l = 0; l < NB; ++l)
            if (l <= cc) acc = fmaf(x[l], s_T[l][cc], acc);
          if (r < jb) s_Y[r][cc] = acc;
          else s_Z[r - jb - kb][cc] = acc;
        }
      }
    }
    __syncthreads();
  };
  if constexpr (COLS == PT) {
    // The partial products reduced through distributed shared memory: CTA c sums rows
    // r = c mod C of every CTA's partial, in a fixed order, and every CTA then gathers the summed
    // rows and forms T_panel, U and Z itself (the same values on every CTA).
    uint8_t* sv = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(s_sv) + 1023) & ~uintptr_t(1023));
    float* P_own = reinterpret_cast<float*>(sv);
    float* Ysum = P_own + NBO * NB;
    cluster.sync();  // every CTA's partial is in place
    for (int r = c + C * warp; r < kbo; r += C * NWARP) {
      float part[MAXC];
#pragma unroll
      for (int q = 0; q < MAXC; ++q) part[q] = q < C ? cluster.map_shared_rank(P_own, q)[r * NB + lane] : 0.f;
      float sum = 0.f;
#pragma unroll
      for (int q = 0; q < MAXC; ++q) sum += part[q];
      Ysum[r * NB + lane] = sum;
    }
    cluster.sync();  // every summed row is in place
    for (int e = tid; e < kbo * NB; e += PT) s_Y[e / NB][e % NB] = cluster.map_shared_rank(Ysum, (e / NB) % C)[e];
    // (the peers may read this CTA's summed rows until the last barrier of the panel)
    __syncthreads();
    form_tuz();
    __syncthreads();
    if (c == 0 && tid < kb) {
      p.skip[(int64_t)b * n + k + tid] = (uint8_t)s_skip[tid];
      p.dsign[(int64_t)b * n + k + tid] = s_dsign[tid];
    }
  } else {
    cluster.sync();  // orders the partials in global memory before rank 0 reads them
    // rank 0 sums the partials, forms T_panel, U = X T_panel and Z, and hands Z, U and T_panel
    // to the cluster through global memory (rank 0's slots of Ypart, free once it has summed
    // them): Z at 0, U at 3072 (jb <= 96 rows), T_panel at 6144 floats
    float* xg = p.Ypart + (int64_t)b * MAXC * NBO * NB;
    float* Ug = xg + NREST * NB;
    float* Tpg = xg + 2 * NREST * NB;
    if (c == 0) {
      // sum the partials in a fixed order
      const float* yp = p.Ypart + (int64_t)b * MAXC * NBO * NB;
      for (int e = tid; e < kbo * NB; e += PT) {
        float part[MAXC];
#pragma unroll
        for (int q = 0; q < MAXC; ++q) part[q] = q < C ? yp[(int64_t)q * NBO * NB + e] : 0.f;
        float sum = 0.f;
#pragma unroll
        for (int q = 0; q < MAXC; ++q) sum += part[q];
        s_Y[e / NB][e % NB] = sum;
      }
      __syncthreads();
      form_tuz();
      __syncthreads();
      for (int e = tid; e < nrest * NB; e += PT) xg[e] = s_Z[e / NB][e % NB];
      for (int e = tid; e < jb * NB; e += PT) Ug[e] = s_Y[e / NB][e % NB];
      for (int e = tid; e < NB * NB; e += PT) Tpg[e] = s_T[e / NB][e % NB];
      if (tid < kb) {
        p.skip[(int64_t)b * n + k + tid] = (uint8_t)s_skip[tid];
        p.dsign[(int64_t)b * n + k + tid] = s_dsign[tid];
      }
    }
    cluster.sync();  // Z, U and T_panel in global memory are visible to the cluster
    if (c != 0) {
      for (int e = tid; e < nrest * NB; e += PT) s_Z[e / NB][e % NB] = xg[e];
      for (int e = tid; e < jb * NB; e += PT) s_Y[e / NB][e % NB] = Ug[e];
      for (int e = tid; e < NB * NB; e += PT) s_T[e / NB][e % NB] = Tpg[e];
    }
    __syncthreads();
  }
  // the block's T, rows spread over the cluster (row r by CTA r mod C): column block jb =
  // [-T_before U ; T_panel ; 0] and the row block jb left of it = 0
  {
    float* T = p.T + (int64_t)b * NBO * NBO;
    float* T_lo = p.T_lo + (int64_t)b * NBO * NBO;
    float* Tt = p.Tt + (int64_t)b * NBO * NBO;
    float* Tt_lo = p.Tt_lo + (int64_t)b * NBO * NBO;
    // the rows of T_before (written by the block's earlier panels) that this CTA's rows need,
    // staged in shared memory with independent loads: the S V area is free (on the cluster path
    // past its first 32 KB, the summed rows that peers may still read)
    constexpr int TBS = NBO - NB;  // jb <= 96
    float* Tb = reinterpret_cast<float*>(
        COLS == PT ? ((reinterpret_cast<uintptr_t>(s_sv) + 1023) & ~uintptr_t(1023)) + 2 * NBO * NB * sizeof(float)
                   : reinterpret_cast<uintptr_t>(s_sv));
    static_assert(TBS * TBS * sizeof(float) <= (COLS == PT ? SV_BYTES - 1024 - 2 * NBO * NB * sizeof(float) : SV_BYTES),
                  "T_before staging");
    const int nrl = jb > c ? (jb - c + C - 1) / C : 0;  // this CTA's rows r = c + C rl below jb
    for (int e = tid; e < nrl * jb; e += PT) {
      const int rl = e / jb, l = e - rl * jb, rr = c + C * rl;
      Tb[rl * TBS + l] = l >= rr ? T[rr * NBO + l] : 0.f;
    }
    __syncthreads();
    // one entry (row r = c + C rl, column jb + cc) per work unit, the 32 units of a row on
    // consecutive threads: the triangular product's long rows are spread over all threads in
    // turn. On the cluster path the column block is also staged transposed, so that Tt's rows
    // are written with consecutive stores.
    const int nr = (NBO - c + C - 1) / C;  // this CTA's rows
    float* stt = COLS == PT ? Tb + TBS * TBS : nullptr;  // [NB][NBO]: entry (cc, rl)
    static_assert(COLS != PT || (TBS * TBS + NB * NBO) * sizeof(float) <= SV_BYTES - 1024 - 2 * NBO * NB * sizeof(float),
                  "T column block staging");
    for (int u = tid; u < nr * NB; u += PT) {
      const int rl = u >> 5, cc = u & 31, r = c + C * rl;
      float t = 0.f;
      if (r < jb) {
        const float* tb_row = Tb + rl * TBS;
#pragma unroll 4
        for (int l = r; l < jb; ++l) t = fmaf(-tb_row[l], s_Y[l][cc], t);
      } else if (r < jb + NB) {
        t = s_T[r - jb][cc];
      }
      const int col = jb + cc;
      T[r * NBO + col] = t;
      T_lo[r * NBO + col] = tf32_lo(t);
      if (COLS == PT) {
        stt[cc * NBO + rl] = t;
      } else {
        Tt[col * NBO + r] = t;
        Tt_lo[col * NBO + r] = tf32_lo(t);
      }
    }
    if (COLS == PT) {
      __syncthreads();
      for (int e = tid; e < NB * nr; e += PT) {
        const int cc = e / nr, rl = e - cc * nr;
        const float t = stt[cc * NBO + rl];
        Tt[(jb + cc) * NBO + c + C * rl] = t;
        Tt_lo[(jb + cc) * NBO + c + C * rl] = tf32_lo(t);
      }
    }
    // the row block jb left of the panel is zero: T's rows jb.. and Tt's columns jb.. there
    for (int e = tid; e < NB * jb; e += PT) {
      const int rr = jb + e / jb, col = e % jb;
      if (rr % C != c) continue;
      T[rr * NBO + col] = 0.f;
      T_lo[rr * NBO + col] = 0.f;
    }
    for (int e = tid; e < NB * jb; e += PT) {
      const int col = e / NB, rr = jb + e % NB;
      if (rr % C != c) continue;
      Tt[col * NBO + rr] = 0.f;
      Tt_lo[col * NBO + rr] = 0.f;
    }
  }

  // the panel's reflectors on the block rows after it: a_r -= Z_r V^T at this CTA's
  // positions, eight rows at a time (eight independent loads in flight), then four, then one
  for (int i = tid; i < npos; i += PT) {
    float v[NB];
#pragma unroll
    for (int jj = 0; jj < NB; ++jj) v[jj] = sA[jj * LDS + i];
    float* a = At + (int64_t)(k + kb) * n + pos0 + i;
    int r = 0;
    for (; r + 8 <= nrest; r += 8) {
      float x[8];
#pragma unroll
      for (int u = 0; u < 8; ++u) x[u] = a[(int64_t)(r + u) * n];
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        float acc = 0.f;
#pragma unroll
        for (int j4 = 0; j4 < NB / 4; ++j4) {
          const float4 z = *reinterpret_cast<const float4*>(&s_Z[r + u][4 * j4]);
          acc = fmaf(z.x, v[4 * j4], fmaf(z.y, v[4 * j4 + 1], fmaf(z.z, v[4 * j4 + 2], fmaf(z.w, v[4 * j4 + 3], acc))));
        }
        a[(int64_t)(r + u) * n] = x[u] - acc;
      }
    }
    for (; r + 4 <= nrest; r += 4) {
      float x[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) x[u] = a[(int64_t)(r + u) * n];
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        float acc = 0.f;
#pragma unroll
        for (int j4 = 0; j4 < NB / 4; ++j4) {
          const float4 z = *reinterpret_cast<const float4*>(&s_Z[r + u][4 * j4]);
          acc = fmaf(z.x, v[4 * j4], fmaf(z.y, v[4 * j4 + 1], fmaf(z.z, v[4 * j4 + 2], fmaf(z.w, v[4 * j4 + 3], acc))));
        }
        a[(int64_t)(r + u) * n] = x[u] - acc;
      }
    }
    for (; r < nrest; ++r) {
      float acc = 0.f;
#pragma unroll
      for (int jj = 0; jj < NB; ++jj) acc = fmaf(s_Z[r][jj], v[jj], acc);
      a[(int64_t)r * n] -= acc;
    }
  }
  // the next panel's positions are shifted by 32: it reads rows that the other CTAs updated
  cluster.sync();
}

// Whether the column loop has to factor this matrix's block (also where a value is not finite). The
// trace decides in nearly every case; where it is not close enough, ||G^^-1||_F^2 = ||X X^T||_F^2 with X
// from qr_block_inverse takes a few us (the column loop 440 a block): warp w has the rows w + 16 r, lane l
// the columns l + 32 c on and above the diagonal, and X is zero before its diagonal. By the trace alone
// the 24-layer stack's steps 4 to 8 took 2553 ms each, 2431 with this.
constexpr int kInvLd = NBO + 4;
constexpr int kInvSmem = NBO * kInvLd * 4;
__device__ __forceinline__ bool block_left(const PanelArgs& p, int b, float* sm) {
  const int state = p.state[b];
  const float excess = qr_block_excess(p.Ypart, b, p.kbo);
  if (state != kQrBlockFast) return state == kQrBlockColumns;
  if (excess <= kQrMaxExcess) return false;
  __shared__ float s_sum[NWARP];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const float* X = qr_block_inverse(p.Ypart, b);
  for (int e = tid; e < NBO * NBO / 4; e += PT)
    *reinterpret_cast<float4*>(sm + (e >> 5) * kInvLd + 4 * (e & 31)) = reinterpret_cast<const float4*>(X)[e];
  __syncthreads();
  float sum = 0.f;
#pragma unroll
  for (int c = 0; c < 4; ++c) {
    float acc[8];
#pragma unroll
    for (int r = 0; r < 2 * c + 2; ++r) acc[r] = 0.f;
#pragma unroll 2
    for (int k = 32 * c; k < NBO; k += 4) {
      const float4 y = *reinterpret_cast<const float4*>(sm + (lane + 32 * c) * kInvLd + k);
#pragma unroll
      for (int r = 0; r < 2 * c + 2; ++r) {
        const float4 x = *reinterpret_cast<const float4*>(sm + (warp + 16 * r) * kInvLd + k);
        acc[r] = fmaf(x.x, y.x, fmaf(x.y, y.y, fmaf(x.z, y.z, fmaf(x.w, y.w, acc[r]))));
      }
    }
#pragma unroll
    for (int r = 0; r < 2 * c + 2; ++r) {
      const int i = warp + 16 * r, j = lane + 32 * c;
      sum = fmaf(j > i ? 2.f : j == i ? 1.f : 0.f, acc[r] * acc[r], sum);
    }
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
  if (lane == 0) s_sum[warp] = sum;
  __syncthreads();
  float norm2 = 0.f;
#pragma unroll
  for (int w = 0; w < NWARP; ++w) norm2 += s_sum[w];
  return !(norm2 <= kQrMaxInverse * kQrMaxInverse);
}

// The block's panels one after another, for a matrix whose block was not factored from its Gram matrix.
// One launch per block, so that a block that was costs one launch that returns at once (four, or eight
// with the column loop as a kernel of its own, cost 14-20 us).
template <int COLS>
__global__ void __launch_bounds__(PT, 1) qr_panel_kernel(const __grid_constant__ PanelArgs p) {
  const int b = blockIdx.y, warp = threadIdx.x >> 5;
  extern __shared__ float4 smem_dyn[];
  if (!block_left(p, b, reinterpret_cast<float*>(smem_dyn))) return;  // factored without the column loop
  __syncthreads();

  __shared__ uint32_t s_tmem;
  uint32_t tmem = 0;
  if constexpr (COLS == PT) {
    if (warp == 0) {
      asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(tc::smem_u32(&s_tmem)),
                   "r"(64));
      asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    tc::tc_fence_before();
    __syncthreads();
    tc::tc_fence_after();
    tmem = s_tmem;
  }
  for (int k = p.k0; k < p.k0 + p.kbo; k += NB) panel<COLS>(p, k, tmem);
  if constexpr (COLS == PT) {
    tc::tc_fence_before();
    __syncthreads();
    if (warp == 0) {
      tc::tc_fence_after();
      asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(64));
    }
  }
}

// ||P_b||_F: per-chunk partial sums in double (chunks of whole 16-byte units: nn is a
// multiple of 16), then tol * sqrt(sum)
constexpr int NORM_CHUNKS = 64;

// Partial sums of squares of P_b over NORM_CHUNKS chunks. The threshold needs ||P||_F to a few
// digits only, so each thread sums in fp32 (at most a few hundred terms) and the warps' sums are
// added in fp32 too; the chunks' partial sums are added in double by thresh_kernel.
__global__ void frob_partial_kernel(const float* P, int64_t nn, double* part) {
  const int b = blockIdx.y;
  const float4* x = reinterpret_cast<const float4*>(P + (int64_t)b * nn);
  const int64_t n4 = nn / 4;
  const int64_t per = (n4 + NORM_CHUNKS - 1) / NORM_CHUNKS;
  const int64_t beg = blockIdx.x * per, end = min(n4, beg + per);
  float s = 0.f;
  for (int64_t i = beg + threadIdx.x; i < end; i += blockDim.x) {
    const float4 v = x[i];
    s = fmaf(v.x, v.x, s);
    s = fmaf(v.y, v.y, s);
    s = fmaf(v.z, v.z, s);
    s = fmaf(v.w, v.w, s);
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  __shared__ float red[8];
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = s;
  __syncthreads();
  if (threadIdx.x == 0) {
    double t = 0.0;
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) t += red[w];
    part[(int64_t)b * NORM_CHUNKS + blockIdx.x] = t;
  }
}

// T_j of a superblock's block into its place in the superblock's T, zeros left of it.
__global__ void put_block_kernel(const float* T, const float* T_lo, float* D, float* D_lo, int64_t stride, int ld,
                                 int off, int w) {
  const int b = blockIdx.y, cols4 = (off + w) / 4;
  for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < w * cols4; e += gridDim.x * blockDim.x) {
    const int r = e / cols4, c = 4 * (e - r * cols4);
    float4 x = make_float4(0.f, 0.f, 0.f, 0.f), y = x;
    if (c >= off) {
      const int64_t o = ((int64_t)b * NBO + r) * NBO + c - off;
      x = *reinterpret_cast<const float4*>(T + o);
      y = *reinterpret_cast<const float4*>(T_lo + o);
    }
    const int64_t d = b * stride + (int64_t)(off + r) * ld + c;
    *reinterpret_cast<float4*>(D + d) = x;
    *reinterpret_cast<float4*>(D_lo + d) = y;
  }
}

// The zero-column threshold tol * ||P_b||_F; a non-finite norm (a NaN or Inf anywhere in P_b,
// wherever the Householder steps would meet it) is a breakdown of that QR.
__global__ void thresh_kernel(const double* part, float tol, int batch, float* thresh, int* status) {
  const int b = blockIdx.x * blockDim.x + threadIdx.x;
  if (b >= batch) return;
  double s = 0.0;
  for (int i = 0; i < NORM_CHUNKS; ++i) s += part[(int64_t)b * NORM_CHUNKS + i];
  if (!isfinite(s) && status) atomicOr(status, kStatusQrBreakdown);
  thresh[b] = (float)((double)tol * sqrt(s));
}

// The panel kernel variant for this device: 512 positions per CTA in clusters of up to 16
// where the device runs 16-CTA clusters of it, else 1024 positions in clusters of up to 8.
struct PanelKernel {
  void (*fn)(PanelArgs);
  int cols;
  size_t smem;
};

template <int COLS>
cudaError_t prepare_panel(PanelKernel* pk, bool wide) {
  pk->fn = qr_panel_kernel<COLS>;
  pk->cols = COLS;
  pk->smem = std::max<size_t>((size_t)NB * (COLS + 4) * sizeof(float), kInvSmem);
  cudaError_t e = cudaFuncSetAttribute(pk->fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)pk->smem);
  if (e == cudaSuccess && wide) e = cudaFuncSetAttribute(pk->fn, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
  return e;
}

// The cluster shape is chosen once per device (with that device current): 1 = clusters of
// 16 x 512 positions where the device can place them, 2 = clusters of 8 x 1024.
std::atomic<int> g_panel_choice[64];

cudaError_t panel_kernel(PanelKernel* pk, int n) {
  // a factor of at most 1024 rows fits one CTA's 1024 positions: no cluster barrier per column
  if (n <= 1024) return prepare_panel<1024>(pk, false);
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0) dev = 0;
  std::atomic<int>* slot = dev < 64 ? &g_panel_choice[dev] : nullptr;
  int choice = slot ? slot->load(std::memory_order_relaxed) : 0;
  if (choice == 0) {
    int ok = 0;
    if (prepare_panel<512>(pk, true) == cudaSuccess) {
      cudaLaunchConfig_t cfg = {};
      cfg.gridDim = dim3(16, 1, 1);
      cfg.blockDim = dim3(PT, 1, 1);
      cfg.dynamicSmemBytes = pk->smem;
      cudaLaunchAttribute attr[1];
      attr[0].id = cudaLaunchAttributeClusterDimension;
      attr[0].val.clusterDim.x = 16;
      attr[0].val.clusterDim.y = 1;
      attr[0].val.clusterDim.z = 1;
      cfg.attrs = attr;
      cfg.numAttrs = 1;
      int clusters = 0;
      if (cudaOccupancyMaxActiveClusters(&clusters, pk->fn, &cfg) == cudaSuccess && clusters > 0) ok = 1;
    }
    cudaGetLastError();
    choice = ok ? 1 : 2;
    if (slot) slot->store(choice, std::memory_order_relaxed);
  }
  if (choice != 1) return prepare_panel<1024>(pk, false);
  return prepare_panel<512>(pk, true);
}

struct Workspace {
  float* At;
  float* Vt_lo;   // after At: the two hold the planes of Q^T once the factorisation is over
  float* Vt;
  float* Tg;      // T of every superblock (see superblock()), then one operand of the Q accumulation
  float* VTr;     // [batch][n][NBO] V T^T of the current block; from here to Wsplit's end also the
  float* VTr_lo;  // operand planes of the Q accumulation
  float* Vpos;    // [batch][n][NBO]
  float* Vpos_lo;
  float* W;       // [batch][n][NBO]
  float* W_lo;
  float* Wsplit;  // [KSPLIT][batch][n][NBO] partial sums of split-K products
  float* T;       // [batch][NBO][NBO], and T^T, each with its lo part
  float* T_lo;
  float* Tt;
  float* Tt_lo;
  float* Ypart;   // [batch][MAXC][NBO][NB]
  // for the look-ahead schedule only (null otherwise): the far update's own W and split-K
  // buffers, and second V T^T, Vpos and T buffers (blocks alternate: a block's V T^T is read
  // by its far update and its Vpos and T by its V T while the next block is factored)
  float* W2;
  float* W2_lo;
  float* Wsplit2;
  float* VTr2;
  float* VTr2_lo;
  float* Vpos2;
  float* Vpos2_lo;
  float* T2;
  float* T2_lo;
  float* Tt2;
  float* Tt2_lo;
  float* thresh;
  float* dsign;
  double* part;
};

// The Q accumulation goes by superblocks of up to 4 blocks (512 columns): its last product reads and
// writes all of Q^T from the superblock on, so fewer, wider ones move less (16 of 2048 x 2048: four
// times 160 us with K = 128 and fp32 Q^T, 393 us with K = 512 and planes). 3 blocks below n = 1024, where the three operands of 4 do
// not fit the workspace that the factorisation leaves free.
struct Superblock {
  int ks, j, wk, blocks;      // first column, the block's index in it, its columns and blocks
  int64_t t_off, t_stride;    // its T (wk x wk) in a matrix's array, and between matrices (floats)
};
Superblock superblock(int n, int blk) {
  const int nblock = (n + NBO - 1) / NBO, per = n >= 1024 ? 4 : 3, sb = blk / per;
  const int64_t w = per * NBO, full = n / w, rest = n - full * w;
  Superblock o;
  o.ks = (int)(sb * w);
  o.j = blk - sb * per;
  o.wk = (int)std::min<int64_t>(w, n - o.ks);
  o.blocks = std::min(per, nblock - sb * per);
  o.t_off = sb * w * w;
  o.t_stride = full * w * w + rest * rest;
  return o;
}

size_t align256(size_t x) { return (x + 255) & ~(size_t)255; }

Workspace carve(void* base, int n, int batch, size_t* total, bool lookahead) {
  const int nblock = (n + NBO - 1) / NBO;
  size_t off = 0;
  auto take = [&](size_t bytes) {
    size_t o = off;
    off += align256(bytes);
    return o;
  };
  const size_t mat = (size_t)batch * n * n * sizeof(float);
  const size_t blocks = (size_t)batch * nblock * n * NBO * sizeof(float);
  const size_t thin = (size_t)batch * n * NBO * sizeof(float);
  const size_t tsq = (size_t)batch * NBO * NBO * sizeof(float);
  const size_t oAt = take(mat), oVtl = take(mat), oVt = take(mat);
  const size_t oTg = take(2 * blocks), oVr = take(thin), oVrl = take(thin);
  const size_t oVp = take(thin), oVpl = take(thin), oW = take(thin), oWl = take(thin);
  const size_t oWs = take((size_t)KSPLIT * thin);
  const size_t oT = take(tsq), oTl = take(tsq), oTt = take(tsq), oTtl = take(tsq);
  const size_t oY = take((size_t)batch * MAXC * NBO * NB * sizeof(float));
  const size_t oW2 = lookahead ? take(thin) : 0, oW2l = lookahead ? take(thin) : 0;
  const size_t oWs2 = lookahead ? take((size_t)KSPLIT * thin) : 0;
  const size_t oVr2 = lookahead ? take(thin) : 0, oVr2l = lookahead ? take(thin) : 0;
  const size_t oVp2 = lookahead ? take(thin) : 0, oVp2l = lookahead ? take(thin) : 0;
  const size_t oT2 = lookahead ? take(tsq) : 0, oT2l = lookahead ? take(tsq) : 0;
  const size_t oTt2 = lookahead ? take(tsq) : 0, oTt2l = lookahead ? take(tsq) : 0;
  const size_t oth = take((size_t)batch * sizeof(float));
  const size_t osg = take((size_t)batch * n * sizeof(float));
  const size_t opart = take((size_t)batch * NORM_CHUNKS * sizeof(double));
  if (total) *total = off;
  char* c = (char*)base;
  auto f = [&](size_t o) { return (float*)(c + o); };
  auto g = [&](size_t o) { return lookahead ? (float*)(c + o) : nullptr; };
  return Workspace{f(oAt), f(oVtl), f(oVt), f(oTg), f(oVr), f(oVrl), f(oVp),  f(oVpl),
                   f(oW),  f(oWl),  f(oWs), f(oT),  f(oTl),  f(oTt), f(oTtl), f(oY),  g(oW2),  g(oW2l),
                   g(oWs2), g(oVr2), g(oVr2l), g(oVp2), g(oVp2l), g(oT2),  g(oT2l),  g(oTt2), g(oTt2l),
                   f(oth), f(osg), (double*)(c + opart)};
}

TcOperand op(const float* hi, const float* lo, int64_t ld, int64_t stride, int batch) {
  return TcOperand{hi, lo, ld, stride, batch};
}

TcEpilogue out(float* C, float* C_lo, int64_t ldc, int64_t stride, float alpha, float beta, int* status) {
  return TcEpilogue{C, ldc, stride, C_lo, ldc, stride, 0, alpha, beta, status};
}

}  // namespace

size_t qr_workspace_bytes(int n, int batch, bool lookahead) {
  size_t total = 0;
  carve(nullptr, n, batch, &total, lookahead);
  return total;
}

void qr_input_buffers(void* workspace, int n, int batch, float** At) {
  Workspace w = carve(workspace, n, batch, nullptr, false);  // the input buffer comes first either way
  *At = w.At;
}

cudaError_t qr_q_t(int n, int batch, float* Q, uint8_t* skip, float tol, void* workspace, size_t workspace_bytes,
                   int* status, cudaStream_t s, const QrLookahead* lah, float** Qt_out) {
  if (n <= 0 || batch <= 0) return cudaSuccess;
  if (n > 8192 || batch > 65535 || (n & 3)) return cudaErrorInvalidValue;
  // look-ahead: a second stream and its events given, and a workspace sized for it
  const bool la = lah && lah->far && lah->vt && lah->far_done && lah->vq[0] && lah->vq[1] &&
                  workspace_bytes >= qr_workspace_bytes(n, batch, true);
  cudaStream_t far = la ? lah->far : nullptr;
  cudaEvent_t ev_vt = la ? lah->vt : nullptr, ev_far = la ? lah->far_done : nullptr;
  size_t need = 0;
  Workspace w = carve(workspace, n, batch, &need, la);
  if (workspace_bytes < need) return cudaErrorInvalidValue;
  const int nblock = (n + NBO - 1) / NBO;
  const int64_t nn = (int64_t)n * n, thin = (int64_t)n * NBO;
  cudaError_t e;

  {
    ProfScope prof(kFamOther, 2.0 * nn * batch, 4.0 * nn * batch, s);
    frob_partial_kernel<<<dim3(NORM_CHUNKS, batch), 256, 0, s>>>(w.At, nn, w.part);
  }
  {
    ProfScope prof(kFamOther, 0, 8.0 * NORM_CHUNKS * batch, s);
    thresh_kernel<<<(batch + 127) / 128, 128, 0, s>>>(w.part, tol, batch, w.thresh, status);
  }
  PanelKernel pk;
  e = panel_kernel(&pk, n);
  if (e != cudaSuccess) return e;

  if (la) {
    // the far stream starts after everything enqueued on s so far; ev_far stands for "the
    // previous far update is done" and starts out recorded
    e = cudaEventRecord(ev_far, s);
    if (e == cudaSuccess) e = cudaStreamWaitEvent(far, ev_far, 0);
    if (e != cudaSuccess) return e;
  }
  for (int blk = 0; blk < nblock; ++blk) {
    const int k0 = blk * NBO, kbo = std::min(NBO, n - k0), m = n - k0;
    const int par = blk & 1;
    const bool alt = la && par;
    float* vp = alt ? w.Vpos2 : w.Vpos;
    float* vp_lo = alt ? w.Vpos2_lo : w.Vpos_lo;
    float* Tb = alt ? w.T2 : w.T;
    float* Tb_lo = alt ? w.T2_lo : w.T_lo;
    float* Ttb = alt ? w.Tt2 : w.Tt;
    float* Ttb_lo = alt ? w.Tt2_lo : w.Tt_lo;
    // with the look-ahead, this block's Vpos and T buffers were last read by the V T of the
    // block two before, on the far stream
    if (la && blk >= 2) {
      e = cudaStreamWaitEvent(s, lah->vq[par], 0);
      if (e != cudaSuccess) return e;
    }
    // the block from its Gram matrix; matrices it leaves to the column loop are factored by the
    // panel kernels below, which return at once for the others. (The scratch it needs is free at
    // this point: W, the split-K sums, the panels' partial products and the norms' partial sums.)
    int* state = reinterpret_cast<int*>(w.part);
    {
      QrBlockArgs f{w.At, w.Vt, w.Vt_lo, vp, vp_lo, Tb, Tb_lo, Ttb, Ttb_lo, w.Ypart, w.W, w.W_lo,
                    state, skip, w.dsign, w.thresh, status, n, k0, kbo};
      e = qr_block_fast(f, batch, s);
      if (e != cudaSuccess) return e;
    }
    {
      PanelArgs a{w.At, w.Vt, w.Vt_lo, vp, vp_lo, Tb, Tb_lo, Ttb, Ttb_lo, w.Ypart, skip, w.dsign,
                  w.thresh, state, status, n, k0, kbo};
      const int C = (m + pk.cols - 1) / pk.cols;
      cudaLaunchConfig_t cfg = {};
      cfg.gridDim = dim3(C, batch, 1);
      cfg.blockDim = dim3(PT, 1, 1);
      cfg.dynamicSmemBytes = pk.smem;
      cfg.stream = s;
      cudaLaunchAttribute attr[1];
      attr[0].id = cudaLaunchAttributeClusterDimension;
      attr[0].val.clusterDim.x = C;
      attr[0].val.clusterDim.y = 1;
      attr[0].val.clusterDim.z = 1;
      cfg.attrs = attr;
      cfg.numAttrs = 1;
      // (tagged without work: what the blocks it takes cost is counted with qr_block_fast)
      ProfScope prof(kFamQrPanel, 0.0, 0.0, s);
      e = cudaLaunchKernelEx(&cfg, pk.fn, a);
      if (e != cudaSuccess) return e;
    }
    // VTr = V T^T (this block's trailing update); with the look-ahead the V T^T buffers alternate
    // between blocks, since the far update of block b still reads its V T^T while block b+1 forms
    // its own
    float* vtr = alt ? w.VTr2 : w.VTr;
    float* vtr_lo = alt ? w.VTr2_lo : w.VTr_lo;
    const TcOperand vpos = op(vp + (int64_t)k0 * NBO, vp_lo + (int64_t)k0 * NBO, NBO, thin, batch);
    // The superblock's H_ks ... H_k0+kbo-1 = I - V T V^T: block j's columns of T are
    // [-T_prev X ; T_j] with X = (V_prev^T V_j) T_j. All on one stream, in order; the block's W and
    // V T^T buffers are free by then (its trailing update has read them).
    auto grow_t = [&](cudaStream_t st) -> cudaError_t {
      const Superblock sb = superblock(n, blk);
      if (sb.blocks == 1) return cudaSuccess;  // the block's own T is all of it
      float* t = w.Tg + sb.t_off;
      float* t_lo = t + batch * sb.t_stride;
      const int kp = k0 - sb.ks;  // columns before this block
      {
        ProfScope prof(kFamOther, 0.0, 16.0 * kbo * (kp + kbo) * batch, st);
        put_block_kernel<<<dim3(8, batch), 256, 0, st>>>(Tb, Tb_lo, t, t_lo, sb.t_stride, sb.wk, kp, kbo);
      }
      cudaError_t e2 = cudaGetLastError();
      if (e2 != cudaSuccess || kp == 0) return e2;
      float* g = la ? w.W2 : w.W;
      float* g_lo = la ? w.W2_lo : w.W_lo;
      const int64_t vp0 = (int64_t)sb.ks * n + k0, vj0 = (int64_t)k0 * n + k0;
      e2 = gemm_tc_nt(kp, kbo, m, batch, op(w.Vt + vp0, w.Vt_lo + vp0, n, nn, batch),
                      op(w.Vt + vj0, w.Vt_lo + vj0, n, nn, batch), out(g, g_lo, NBO, thin, 1.f, 0.f, status), st,
                      kFamQrUpdate, la ? w.Wsplit2 : w.Wsplit, (size_t)KSPLIT * batch * n * NBO);
      if (e2 != cudaSuccess) return e2;
      TcEpilogue xt = out(vtr, vtr_lo, kp, thin, 1.f, 0.f, status);  // X^T
      xt.transpose = 1;
      e2 = gemm_tc_nt(kp, kbo, kbo, batch, op(g, g_lo, NBO, thin, batch), op(Ttb, Ttb_lo, NBO, NBO * NBO, batch), xt,
                      st, kFamQrUpdate);
      if (e2 != cudaSuccess) return e2;
      return gemm_tc_nt(kp, kbo, kp, batch, op(t, t_lo, sb.wk, sb.t_stride, batch), op(vtr, vtr_lo, kp, thin, batch),
                        out(t + kp, t_lo + kp, sb.wk, sb.t_stride, -1.f, 0.f, status), st, kFamQrUpdate);
    };
    const int nc = n - k0 - kbo;  // trailing rows of At (columns of P)
    if (nc > 0) {
      e = gemm_tc_nt(m, kbo, kbo, batch, vpos, op(Tb, Tb_lo, NBO, NBO * NBO, batch),
                     out(vtr + (int64_t)k0 * NBO, vtr_lo + (int64_t)k0 * NBO, NBO, thin, 1.f, 0.f, status), s,
                     kFamQrUpdate);
      if (e != cudaSuccess) return e;
    }
    const TcOperand vtr_trail =
        op(vtr + (int64_t)(k0 + kbo) * NBO, vtr_lo + (int64_t)(k0 + kbo) * NBO, NBO, thin, batch);
    const TcOperand vt_blk = op(w.Vt + (int64_t)k0 * n + k0, w.Vt_lo + (int64_t)k0 * n + k0, n, nn, batch);
    // rows [r0, r0 + rows) of the trailing matrix: a_r -= (a_r V) T V^T, i.e.
    //   W = At_rows Vt^T over positions k0.. ; At_rows -= W VTr^T at positions k0+kbo.. (the
    //   earlier positions of these rows are R's entries, never read again)
    auto update_rows = [&](int r0, int rows, float* Wb, float* Wb_lo, float* ws, cudaStream_t st) -> cudaError_t {
      const int64_t tr = (int64_t)r0 * n;
      cudaError_t e2 = gemm_tc_nt(rows, kbo, m, batch, op(w.At + tr + k0, nullptr, n, nn, batch), vt_blk,
                                  out(Wb, Wb_lo, NBO, thin, 1.f, 0.f, status), st, kFamQrUpdate, ws,
                                  (size_t)KSPLIT * batch * n * NBO);
      if (e2 != cudaSuccess) return e2;
      return gemm_tc_nt(rows, nc, kbo, batch, op(Wb, Wb_lo, NBO, thin, batch), vtr_trail,
                        out(w.At + tr + k0 + kbo, nullptr, n, nn, -1.f, 1.f, status), st,
                        kFamQrUpdate);
    };
    if (!la) {
      e = nc > 0 ? update_rows(k0 + kbo, nc, w.W, w.W_lo, w.Wsplit, s) : cudaSuccess;
      if (e == cudaSuccess) e = grow_t(s);
      if (e != cudaSuccess) return e;
      continue;
    }
    // look-ahead: the next block's rows now (they gate its panels), the rest on the far stream,
    // where it overlaps the next block's panels; the next block's rows wait for the previous
    // far update, which covered them. The block's part of T follows its far update there.
    const int knext = std::min(NBO, std::max(nc, 0));
    // (the far update starts once the next block's rows are done, so that those small products
    // do not wait for SMs behind it)
    e = cudaSuccess;
    if (nc > 0) e = cudaStreamWaitEvent(s, ev_far, 0);
    if (e == cudaSuccess && nc > 0) e = update_rows(k0 + kbo, knext, w.W, w.W_lo, w.Wsplit, s);
    if (e == cudaSuccess) e = cudaEventRecord(ev_vt, s);
    if (e == cudaSuccess) e = cudaStreamWaitEvent(far, ev_vt, 0);
    if (e == cudaSuccess && nc > knext) e = update_rows(k0 + kbo + knext, nc - knext, w.W2, w.W2_lo, w.Wsplit2, far);
    if (e == cudaSuccess) e = cudaEventRecord(ev_far, far);
    if (e == cudaSuccess) e = grow_t(far);
    if (e == cudaSuccess) e = cudaEventRecord(lah->vq[par], far);
    if (e != cudaSuccess) return e;
  }
  if (la) {
    // the last far update and the last of T before the Q accumulation
    e = cudaEventRecord(ev_far, far);
    if (e == cudaSuccess) e = cudaStreamWaitEvent(s, ev_far, 0);
    if (e != cudaSuccess) return e;
  }

  // Q^T = diag(d) H_n ... H_1 accumulated backwards, a superblock at a time, on planes: the sub-matrix
  // from ks on becomes Qt_sub - ((Qt_sub V) T^T) V^T, where the superblock's own rows and columns of
  // Qt_sub are still those of diag(d), and are neither multiplied nor read. With one superblock Q^T
  // ends in fp32 in place of P^T; else it is kept as planes and the last product writes it in fp32
  // over V, dead by then.
  const Superblock last = superblock(n, nblock - 1);
  const bool one = last.ks == 0;
  const Planes Qp = planes_in(w.At, n, n, batch);  // over At and Vt_lo
  float* Qt = one ? w.At : w.Vt;
  for (int blk = nblock - last.blocks; blk >= 0;) {
    const Superblock sb = superblock(n, blk);
    const int m = n - sb.ks, wk = sb.wk;
    const float* v = w.Vt + (int64_t)sb.ks * n + sb.ks;
    // operands: W, then V; W T^T; and V^T, then T
    char* room = reinterpret_cast<char*>(w.VTr);
    const size_t tall = align256(planes_bytes(m, wk, batch));
    const Planes A = planes_in(room, m, wk, batch), B = planes_in(room + tall, m, wk, batch);
    void* third = n >= 1024 ? (void*)((char*)w.Tg + align256(2 * batch * sb.t_stride * sizeof(float))) : room + 2 * tall;
    const Planes Tp = planes_in(third, wk, wk, batch);
    auto into = [&](const Planes& o) {
      B3Epilogue ep{};
      ep.P = o.p, ep.p_plane = o.plane, ep.p_ld = o.ld, ep.p_stride = o.stride;
      ep.alpha = 1.f, ep.status = status;
      return ep;
    };
    // Qt_sub V: the rows of diag(d) and, below them, the product with what is accumulated so far
    e = split_blocks(v, n, nn, true, w.dsign + sb.ks, n, NBO, A, wk, wk, batch, s);
    if (e == cudaSuccess && m > wk) {
      const Planes Vp = planes_in(third, wk, m - wk, batch);
      e = split_blocks(v + wk, n, nn, false, nullptr, 0, 0, Vp, wk, m - wk, batch, s);
      if (e == cudaSuccess)
        e = gemm_b3(m - wk, wk, m - wk, batch, b3_op(Qp.at(0, sb.ks + wk, sb.ks + wk), batch), b3_op(Vp, batch),
                    into(A.at(0, wk)), s, kFamQrUpdate);
    }
    if (e == cudaSuccess) {
      if (sb.blocks == 1) {
        const float* t = la && (blk & 1) ? w.T2 : w.T;
        e = split_blocks(t, NBO, NBO * NBO, false, nullptr, 0, 0, Tp, wk, wk, batch, s);
      } else {
        e = split_blocks(w.Tg + sb.t_off, wk, sb.t_stride, false, nullptr, 0, NBO, Tp, wk, wk, batch, s);
      }
    }
    if (e == cudaSuccess) e = gemm_b3(m, wk, wk, batch, b3_op(A, batch), b3_op(Tp, batch), into(B), s, kFamQrUpdate);
    if (e == cudaSuccess) e = split_blocks(v, n, nn, true, nullptr, 0, NBO, A, wk, m, batch, s);
    if (e != cudaSuccess) return e;
    const Planes Qs = Qp.at(0, sb.ks, sb.ks);
    B3Epilogue eq = into(Qs);
    eq.alpha = -1.f, eq.beta = 1.f;
    eq.cin = Qs.p, eq.cin_diag = w.dsign + sb.ks, eq.cin_diag_stride = n, eq.cin_from = wk;
    if (sb.ks == 0) eq.P = nullptr, eq.C = Qt, eq.ldc = n, eq.c_stride = nn;
    e = gemm_b3(m, m, wk, batch, b3_op(B, batch), b3_op(A, batch), eq, s, kFamQrUpdate);
    if (e != cudaSuccess) return e;
    blk -= n >= 1024 ? 4 : 3;
  }
  if (Qt_out) *Qt_out = Qt;
  if (Q) {
    e = planes_transpose(Qt, Planes(), Planes(), Q, n, batch, s);
    if (e != cudaSuccess) return e;
  }
  return cudaGetLastError();
}

cudaError_t qr_q(int n, int batch, const float* P, float* Q, uint8_t* skip, float tol, void* workspace,
                 size_t workspace_bytes, int* status, cudaStream_t s) {
  if (n <= 0 || batch <= 0) return cudaSuccess;
  size_t need = 0;
  Workspace w = carve(workspace, n, batch, &need, false);
  if (workspace_bytes < need || (n & 3)) return cudaErrorInvalidValue;
  // At = P^T
  cudaError_t e = planes_transpose(P, Planes(), Planes(), w.At, n, batch, s);
  if (e != cudaSuccess) return e;
  return qr_q_t(n, batch, Q, skip, tol, workspace, workspace_bytes, status, s);
}

}  // namespace soap
