// fp32-accurate batched GEMM on the 5th-generation tensor cores, operands as three bf16 planes.
//
//   C_b = alpha * A_{b mod amod} * B_{b mod bmod}^T + beta * C_b
//
// A is M x K and B is N x K, both row-major ("K-major"). An operand x is kept as three bf16
// arrays (planes) h + m + l, each the rounding to nearest of what the ones before it leave, so
// that h + m + l is x to 2^-26; the product accumulates
//   h l + l h + m m + h m + m h + h h       (kind::f16, fp32 accumulation)
// and leaves out terms of 2^-26 of |a||b| and below. Six bf16 products cost three quarters of the
// four TF32 products that a hi/lo split needs for the same accuracy (tf32 runs at half the bf16
// rate), and 6 bytes per operand element are moved instead of 8.
//
// Each 64-wide K block is accumulated afresh in one of two TMEM accumulators, its small terms
// first, and drained into fp32 registers with round-to-nearest adds while the next block's MMAs
// run: the tensor core truncates its accumulator at every MMA, and only four truncations of a
// full-size sum remain per block (measured on unit Gaussians: 1.2e-7 relative error at K = 64).
//
// The kernel is bound by the tensor pipe if the operands arrive in time. A 128 x 128 tile reads
// and refills shared memory at about 190 bytes per cycle of MMA time, above what shared memory
// sustains; a pair of CTAs (cta_group::2) on a 256 x 256 tile halves that, and halves the L2
// reads, since each CTA loads its own 128 rows of A and half of B's rows. 8192^3: 3.2 ms, 340
// fp32-equivalent TFLOP/s, against 5.7 ms, 192 with four TF32 products on 128 x 128 tiles. Products
// of at most 128 rows or columns, and those too small to fill the SM pairs, run one CTA per 128 x 128
// tile (a pair's N = 128 MMA takes as long as its N = 256).
//
// CTA: warp 0 issues the TMA loads, warp 1 allocates tensor memory and (in the pair's first CTA)
// issues the MMAs, warps 2-17 drain the accumulators and store the tile through swizzled blocks in
// shared memory. Stages are handed over with mbarriers; every wait gives up after a
// bounded time (2 s of %globaltimer time unless soap_wait_limit set another), records
// kStatusTimeout and lets the CTAs drain -- copies already issued land, issued MMAs complete -- and
// free their tensor memory. The drains themselves always keep the full 2 s bound.
#include <cuda.h>
#include <cudaTypedefs.h>

#include <algorithm>
#include <atomic>
#include <mutex>

#include "profile.h"
#include "soap_internal.h"
#include "tc_ptx.h"

namespace soap {
namespace b3 {
namespace {

using tc::smem_u32;

constexpr int BM = 128;  // rows of A per CTA
constexpr int BK = 64;   // bf16 elements per K block = one 128-byte swizzle row
constexpr int STAGES = 2;
constexpr int NACC = 2;
// Epilogue warps, each a quarter of the tile's columns: with 16 more loads of C are in flight than with
// 8 (16 of 2048 x 2048 x 512, C read and written as planes: 0.54 ms with 8, 0.44 with 16; 64 of
// 2048 x 768 x 768, written only: 0.60 and 0.57; 8192 x 8192 x 512 with C in fp32: 0.326 and 0.333)
constexpr int EPI = 16;
constexpr int THREADS = 64 + 32 * EPI;
constexpr int PLANE_A = BM * BK * 2;
constexpr uint64_t kWaitNs = 2000000000ull;

enum : int { kF32 = 1, kPlanes = 2, kTr = 4, kBeta = 8, kSym = 16, kBetaP = 32 };

// CG CTAs work on a CG * 128 x BN tile, each with its 128 rows of A and BN / CG rows of B.
template <int CG, int BN>
struct Cfg {
  static constexpr int BROWS = BN / CG;
  static constexpr int PLANE_B = BROWS * BK * 2;
  static constexpr int STAGE = 3 * (PLANE_A + PLANE_B);
  static constexpr int CPW = BN * 4 / EPI;  // accumulator columns drained by one warp
  static constexpr int NCH = CPW / 32;
  static constexpr int SMEM = STAGES * STAGE + EPI * 2048 + 1024 + 256;
  static constexpr uint32_t TMEM_COLS = NACC * BN;
  static_assert(SMEM <= 232448, "shared memory budget");
};

__device__ __forceinline__ bool flag_wait(const int* flag, uint64_t limit_ns) {
  const volatile int* f = flag;
  if (*f != 0) return true;
  const uint64_t t0 = tc::globaltimer();
  while (*f == 0)
    if (tc::globaltimer() - t0 > limit_ns) return false;
  return true;
}

// K block at c0, rows from c1, matrix c2: all three planes, into this CTA's shared memory; the
// pair's first CTA's barrier counts the bytes.
template <int CG>
__device__ __forceinline__ void tma_load(uint32_t dst, const CUtensorMap* map, uint32_t bar, int c0, int c1, int c2) {
  if (CG == 1)
    asm volatile(
        "cp.async.bulk.tensor.4d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, %5, %6}], "
        "[%2];" ::"r"(dst),
        "l"(reinterpret_cast<uint64_t>(map)), "r"(bar), "r"(c0), "r"(c1), "r"(c2), "r"(0)
        : "memory");
  else
    asm volatile(
        "cp.async.bulk.tensor.4d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, "
        "%5, %6}], [%2];" ::"r"(dst),
        "l"(reinterpret_cast<uint64_t>(map)), "r"(bar), "r"(c0), "r"(c1), "r"(c2), "r"(0)
        : "memory");
}

// Word offset of element (r, j) of a 32 x 32 block stored row-major with its 16-byte units
// XOR-swizzled by r mod 8: a warp touching one 16-byte unit per row, or one row, is
// conflict-free.
__device__ __forceinline__ int swz(int r, int j) { return r * 32 + ((((j >> 2) ^ (r & 7))) << 2) + (j & 3); }
// The same for a 32 x 16 block (two rows to a 128-byte line), element (r, 4 q).
__device__ __forceinline__ int swzh(int r, int q) { return r * 16 + ((q ^ ((r >> 1) & 3)) << 2); }

// Tile t of a launch -> (m0, n0, batch index). Within a matrix the tiles go in groups of GM row
// tiles, m fastest, so that the tiles in flight at a time share their row and column panels in L2.
template <int TM>
__device__ __forceinline__ void tile_coords(int t, int ntm, int ntn, int bn, int& m0, int& n0, int& b) {
  constexpr int GM = 1024 / TM;
  const int per = ntm * ntn;
  b = t / per;
  const int r = t - b * per;
  const int g = r / (GM * ntn);
  const int first = g * GM;
  const int gsz = min(GM, ntm - first);
  const int w = r - g * GM * ntn;
  m0 = (first + w % gsz) * TM;
  n0 = (w / gsz) * bn;
}
// Symmetric products (A = B, M = N): the tiles on or below the diagonal only, row by row.
__device__ __forceinline__ void tile_coords_sym(int t, int ntm, int tile, int& m0, int& n0, int& b) {
  const int per = ntm * (ntm + 1) / 2;
  b = t / per;
  const int r = t - b * per;
  int i = (int)((sqrtf(8.f * (float)r + 1.f) - 1.f) * 0.5f);
  while ((i + 1) * (i + 2) / 2 <= r) ++i;
  while (i * (i + 1) / 2 > r) --i;
  m0 = i * tile;
  n0 = (r - i * (i + 1) / 2) * tile;
}

__device__ __forceinline__ float4 b3_unit4(int i, float x) {
  return make_float4(i == 0 ? x : 0.f, i == 1 ? x : 0.f, i == 2 ? x : 0.f, i == 3 ? x : 0.f);
}

struct Args {
  int M, N, K, batch, a_mod, b_mod;
  B3Epilogue ep;
};

// A cluster takes several tiles in turn, so that the loads and MMAs of its next tile overlap the
// epilogue of the current one, a launch's width apart: the tiles in flight are then neighbours, whose
// row and column panels L2 holds. (Runs of consecutive tiles per cluster spread the tiles in flight
// over 8 matrices: 64 products of 2048 x 768 x 2048 took 1.64 ms, 252 TFLOP/s, and take 1.35, 305.)
template <int CG, int BN, int MODE>
__global__ void __launch_bounds__(THREADS, 1)
    gemm_b3_kernel(const __grid_constant__ CUtensorMap ta, const __grid_constant__ CUtensorMap tb,
                   const __grid_constant__ Args p) {
  using C = Cfg<CG, BN>;
  constexpr bool F32 = MODE & kF32, PL = MODE & kPlanes, TR = MODE & kTr, BETA = MODE & kBeta, SYM = MODE & kSym, BETAP = MODE & kBetaP;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  float* obuf_all = reinterpret_cast<float*>(smem + STAGES * C::STAGE);
  uint64_t* full = reinterpret_cast<uint64_t*>(smem + STAGES * C::STAGE + EPI * 2048);
  uint64_t* empty = full + STAGES;
  uint64_t* acc_full = empty + STAGES;
  uint64_t* acc_empty = acc_full + NACC;
  uint64_t* mma_done = acc_empty + NACC;
  uint32_t* tmem_holder = reinterpret_cast<uint32_t*>(mma_done + 1);
  tc::RingState* ring = reinterpret_cast<tc::RingState*>(tmem_holder + 1);  // [2]: this CTA's, the peer's
  volatile int* abort_flag = &ring->abort;
  volatile int* consumed = &ring->consumed;

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int rank = CG == 1 ? 0 : (int)(blockIdx.x & 1);
  const bool lead = rank == 0;
  const B3Epilogue& ep = p.ep;
  const uint64_t lim = ep.wait_ns ? ep.wait_ns : kWaitNs;
  constexpr int TM = CG * BM;
  const int kblocks = (p.K + BK - 1) / BK;
  const int ntn = (p.N + BN - 1) / BN, ntm = (p.M + TM - 1) / TM;
  const int ntiles = (SYM ? ntm * (ntm + 1) / 2 : ntn * ntm) * p.batch;
  const int t_begin = (int)(blockIdx.x / CG), t_step = (int)(gridDim.x / CG);
  // tile t: its first row and column, and its matrix
  auto tile = [&](int t, int& m0, int& n0, int& b) {
    if (SYM) tile_coords_sym(t, ntm, TM, m0, n0, b);
    else tile_coords<TM>(t, ntm, ntn, BN, m0, n0, b);
  };

  if (threadIdx.x == 0) {
    for (int s = 0; s < STAGES; ++s) {
      tc::mbar_init(&full[s], 1);
      tc::mbar_init(&empty[s], 1);
    }
    for (int a = 0; a < NACC; ++a) {
      tc::mbar_init(&acc_full[a], 1);
      tc::mbar_init(&acc_empty[a], EPI * CG);  // one arrival per epilogue warp
    }
    tc::mbar_init(mma_done, 1);
    *ring = tc::RingState{};
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 0 && lane == 0) {
    asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&ta)) : "memory");
    asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(&tb)) : "memory");
  }
  if (warp == 1) {
    if (CG == 1) {
      asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_holder)),
                   "r"(C::TMEM_COLS));
      asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    } else {
      asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_holder)),
                   "r"(C::TMEM_COLS));
      asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;");
    }
  }
  tc::tc_fence_before();
  __syncthreads();
  if (CG == 2) {  // the peer's barriers and tensor memory are set up
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
  }
  tc::tc_fence_after();
  const uint32_t tmem = *tmem_holder;

  if (warp == 0) {
    if (lane == 0) {
      int g = 0, issued = 0;  // K blocks over all of this cluster's tiles
      for (int t = t_begin; t < ntiles && !*abort_flag; t += t_step) {
        int m0, n0, b;
        tile(t, m0, n0, b);
        for (int kb = 0; kb < kblocks; ++kb, ++g) {
          const int s = g % STAGES;
          if (!tc::wait<CG>(&empty[s], ((g / STAGES) & 1) ^ 1, lim) || *abort_flag) {
            *abort_flag = 1;
            if (ep.status) atomicOr(ep.status, kStatusTimeout);
            break;
          }
          if (lead) tc::mbar_expect_tx(&full[s], CG * C::STAGE);
          const uint32_t st = smem_u32(smem + s * C::STAGE), bar = tc::lead_addr<CG>(smem_u32(&full[s]));
          tma_load<CG>(st, &ta, bar, kb * BK, m0 + rank * BM, b % p.a_mod);
          tma_load<CG>(st + 3 * PLANE_A, &tb, bar, kb * BK, n0 + rank * C::BROWS, b % p.b_mod);
          issued = g + 1;
        }
      }
      ring->issued = issued;
    }
  } else if (warp == 1) {
    if (lane == 0 && lead) {
      constexpr uint32_t idesc = tc::idesc_bf16(TM, BN);
      int g = 0;
      bool ok = true;
      for (int t = t_begin; t < ntiles && ok && !*abort_flag; t += t_step) {
        for (int kb = 0; kb < kblocks; ++kb, ++g) {
          const int s = g % STAGES, a = g % NACC;
          if (!tc::wait<CG>(&full[s], (g / STAGES) & 1, lim) ||
              (g >= NACC && !tc::wait<CG>(&acc_empty[a], ((g / NACC) & 1) ^ 1, lim)) || *abort_flag) {
            ok = false;
            break;
          }
          *consumed = g + 1;
          tc::tc_fence_after();
          const uint32_t d = tmem + static_cast<uint32_t>(a * BN);
          const uint32_t as = smem_u32(smem + s * C::STAGE), bs = as + 3 * PLANE_A;
          // (plane of A, plane of B) of the six products, the smallest first
#pragma unroll
          for (int kk = 0; kk < BK / 16; ++kk) {
            const uint32_t o = kk * 32;  // 16 bf16 along K inside the swizzle row
            tc::umma_f16<CG>(d, as + o, bs + 2 * C::PLANE_B + o, idesc, kk != 0);
            tc::umma_f16<CG>(d, as + 2 * PLANE_A + o, bs + o, idesc, 1u);
            tc::umma_f16<CG>(d, as + PLANE_A + o, bs + C::PLANE_B + o, idesc, 1u);
          }
#pragma unroll
          for (int kk = 0; kk < BK / 16; ++kk) {
            const uint32_t o = kk * 32;
            tc::umma_f16<CG>(d, as + o, bs + C::PLANE_B + o, idesc, 1u);
            tc::umma_f16<CG>(d, as + PLANE_A + o, bs + o, idesc, 1u);
          }
#pragma unroll
          for (int kk = 0; kk < BK / 16; ++kk) tc::umma_f16<CG>(d, as + kk * 32, bs + kk * 32, idesc, 1u);
          tc::commit<CG>(&empty[s]);     // frees the stage once these MMAs have read it
          tc::commit<CG>(&acc_full[a]);  // hands the K block's sum to the epilogue warps
        }
      }
      ring->accs = g;
      if (!ok) {
        *abort_flag = 1;
        if (ep.status) atomicOr(ep.status, kStatusTimeout);
      }
      // the tensor memory is freed below: every MMA issued must have completed first (this
      // matters only when a wait gave up; otherwise the epilogue has drained them all)
      if (g > 0) {
        tc::commit<CG>(mma_done);
        tc::wait<CG>(mma_done, 0, kWaitNs);
      }
    }
  } else {
    const int q = warp & 3;  // this warp may read accumulator lanes 32q .. 32q+31
    const int ew = warp - 2;
    const int colbase = (ew / 4) * C::CPW;
    const uint32_t lane_base = tmem + (static_cast<uint32_t>(32 * q) << 16);
    float* cb = obuf_all + ew * 512;
    int g = 0;
    bool valid = true;
    if (ep.hold && !flag_wait(ep.hold, lim)) {
      // the timeout path under test: no tile is drained, the other warps' waits run out too
      valid = false;
      *abort_flag = 1;
      if (lane == 0 && ep.status) atomicOr(ep.status, kStatusTimeout);
    }
    for (int t = t_begin; t < ntiles && valid; t += t_step) {
      int m0, n0, b;
      tile(t, m0, n0, b);
      float* Cb = F32 ? (ep.C_ptrs ? ep.C_ptrs[b] : ep.C + (int64_t)b * ep.c_stride) : nullptr;
      __nv_bfloat16* Pb = PL ? ep.P + (int64_t)b * ep.p_stride : nullptr;
      const __nv_bfloat16* Ib = BETAP ? ep.cin + (int64_t)b * ep.p_stride : nullptr;
      const float* Db = BETAP ? ep.cin_diag + (int64_t)b * ep.cin_diag_stride : nullptr;
      const int row0 = m0 + rank * BM + 32 * q;  // first of this warp's 32 rows
      const int col0 = n0 + colbase;             // first of its CPW columns
      if (BETA) {
        // C's lines into L2 while the MMAs run
        const int outer = TR ? C::CPW : 32, inner = TR ? 32 : C::CPW;  // rows of C, and floats of each
        for (int u = lane; u < outer * inner / 32; u += 32) {
          const int x = u / (inner / 32), y = 32 * (u % (inner / 32));
          const int r = TR ? row0 + y : row0 + x, col = TR ? col0 + x : col0 + y;
          if (r < p.M && col < p.N)
            asm volatile("prefetch.global.L2 [%0];" ::"l"(TR ? Cb + (int64_t)col * ep.ldc + r
                                                             : Cb + (int64_t)r * ep.ldc + col));
        }
      }
      if (BETAP) {
        static_assert(C::CPW <= 64, "one line of each plane per row");
        const int r = row0 + lane, col = col0;
        if (r < p.M && col < p.N && r >= ep.cin_from && col >= ep.cin_from) {
#pragma unroll
          for (int pl = 0; pl < 3; ++pl)
            asm volatile("prefetch.global.L2 [%0];" ::"l"(Ib + pl * ep.p_plane + (int64_t)r * ep.p_ld + col));
        }
      }
      float acc[C::NCH][32];
#pragma unroll
      for (int c = 0; c < C::NCH; ++c)
#pragma unroll
        for (int j = 0; j < 32; ++j) acc[c][j] = 0.f;
      for (int kb = 0; kb < kblocks; ++kb, ++g) {
        const int a = g % NACC;
        if (!tc::wait<CG>(&acc_full[a], (g / NACC) & 1, lim) || *abort_flag) {
          valid = false;
          break;
        }
        tc::tc_fence_after();
#pragma unroll
        for (int c = 0; c < C::NCH; ++c) {
#pragma unroll
          for (int h = 0; h < 2; ++h) {
            float v[16];
            tc::tmem_ld16(lane_base + static_cast<uint32_t>(a * BN + colbase + 32 * c + 16 * h), v);
#pragma unroll
            for (int j = 0; j < 16; ++j) acc[c][16 * h + j] += v[j];
          }
        }
        tc::tc_fence_before();
        __syncwarp();
        if (lane == 0) tc::arrive_lead<CG>(&acc_empty[a]);
      }
      if (!valid) {
        *abort_flag = 1;
        if (lane == 0 && ep.status) atomicOr(ep.status, kStatusTimeout);
        break;
      }
      if (row0 >= p.M) continue;
      // out = alpha acc + beta C through the warp's shared block, 32 rows x 16 columns at a time; C, its
      // rows and columns come in whole 16-byte units (checked on the host)
#pragma unroll
      for (int ch = 0; ch < 2 * C::NCH; ++ch) {
        const float* av = &acc[ch >> 1][16 * (ch & 1)];
        const int cc0 = col0 + 16 * ch;
        if (!TR) {
          const int col = cc0 + 4 * (lane & 3), rl = lane >> 2;  // this lane's unit, in rows rl + 8 it
          float4 cv[4];
          if (BETA || BETAP) {
#pragma unroll
            for (int it = 0; it < 4; ++it) {
              const int r2 = row0 + 8 * it + rl;
              cv[it] = make_float4(0.f, 0.f, 0.f, 0.f);
              if (r2 < p.M && col < p.N) {
                if (BETA) cv[it] = *reinterpret_cast<const float4*>(Cb + (int64_t)r2 * ep.ldc + col);
                else if (r2 >= ep.cin_from && col >= ep.cin_from)
                  cv[it] = b3_load4(Ib + (int64_t)r2 * ep.p_ld + col, ep.p_plane);
                else if ((unsigned)(r2 - col) < 4u) cv[it] = b3_unit4(r2 - col, Db[r2]);
              }
            }
          }
#pragma unroll
          for (int j4 = 0; j4 < 4; ++j4)
            *reinterpret_cast<float4*>(cb + swzh(lane, j4)) = make_float4(
                ep.alpha * av[4 * j4], ep.alpha * av[4 * j4 + 1], ep.alpha * av[4 * j4 + 2], ep.alpha * av[4 * j4 + 3]);
          __syncwarp();
#pragma unroll
          for (int it = 0; it < 4; ++it) {
            const int rr = 8 * it + rl, r2 = row0 + rr;
            float4* slot = reinterpret_cast<float4*>(cb + swzh(rr, lane & 3));
            float4 o = *slot;
            if (BETA || BETAP) {
              o.x = fmaf(ep.beta, cv[it].x, o.x);
              o.y = fmaf(ep.beta, cv[it].y, o.y);
              o.z = fmaf(ep.beta, cv[it].z, o.z);
              o.w = fmaf(ep.beta, cv[it].w, o.w);
              if (SYM) *slot = o;
            }
            if (r2 < p.M && col < p.N) {
              if (F32) *reinterpret_cast<float4*>(Cb + (int64_t)r2 * ep.ldc + col) = o;
              if (PL) b3_store4(Pb + (int64_t)r2 * ep.p_ld + col, ep.p_plane, o);
            }
          }
          if (SYM && m0 != n0) {
            // the mirror tile: element (r, j) of this block also goes to C[j][r]
            __syncwarp();
#pragma unroll 1
            for (int it = 0; it < 4; ++it) {
              const int jj = 4 * it + (lane >> 3), r4 = 4 * (lane & 7);
              const int mrow = cc0 + jj, mcol = row0 + r4;  // row and column in C
              if (mrow >= p.N || mcol >= p.M) continue;     // M = N, a multiple of 4
              auto at = [&](int r) { return cb[swzh(r, jj >> 2) + (jj & 3)]; };
              const float4 o = make_float4(at(r4), at(r4 + 1), at(r4 + 2), at(r4 + 3));
              if (F32) *reinterpret_cast<float4*>(Cb + (int64_t)mrow * ep.ldc + mcol) = o;
              if (PL) b3_store4(Pb + (int64_t)mrow * ep.p_ld + mcol, ep.p_plane, o);
            }
          }
          __syncwarp();
        } else {
          // C^T: element (row r = this lane, column j) goes to row j of the staged 16 x 32 block
          const int r2 = row0 + 4 * (lane & 7), jl = lane >> 3;  // this lane's unit, in rows jl + 4 it
          float4 cv[4];
          if (BETA) {
#pragma unroll
            for (int it = 0; it < 4; ++it) {
              const int col = cc0 + 4 * it + jl;
              cv[it] = (r2 < p.M && col < p.N) ? *reinterpret_cast<const float4*>(Cb + (int64_t)col * ep.ldc + r2)
                                               : make_float4(0.f, 0.f, 0.f, 0.f);
            }
          }
#pragma unroll
          for (int j = 0; j < 16; ++j) cb[swz(j, lane)] = ep.alpha * av[j];
          __syncwarp();
#pragma unroll
          for (int it = 0; it < 4; ++it) {
            const int jj = 4 * it + jl, col = cc0 + jj;
            float4 o = *reinterpret_cast<const float4*>(cb + swz(jj, 4 * (lane & 7)));
            if (BETA) {
              o.x = fmaf(ep.beta, cv[it].x, o.x);
              o.y = fmaf(ep.beta, cv[it].y, o.y);
              o.z = fmaf(ep.beta, cv[it].z, o.z);
              o.w = fmaf(ep.beta, cv[it].w, o.w);
            }
            if (r2 < p.M && col < p.N) {
              if (F32) *reinterpret_cast<float4*>(Cb + (int64_t)col * ep.ldc + r2) = o;
              if (PL) b3_store4(Pb + (int64_t)col * ep.p_ld + r2, ep.p_plane, o);
            }
          }
          __syncwarp();
        }
      }
    }
  }

  tc::finish<CG, STAGES, NACC>(full, empty, acc_full, mma_done, ring, lead, C::STAGE, kWaitNs);
  if (warp == 1) {
    tc::tc_fence_after();
    if (CG == 1)
      asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(C::TMEM_COLS));
    else
      asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(C::TMEM_COLS));
  }
}

// ---- host side ---------------------------------------------------------------------

PFN_cuTensorMapEncodeTiled_v12000 encode_fn() {
  static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
  static std::once_flag once;
  std::call_once(once, [] {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) ==
            cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(p);
  });
  return fn;
}

// Tensor map of the three planes of `batch` row-major rows x K matrices, boxes of 64 x box_rows
// elements of one matrix in all three planes.
bool make_map(CUtensorMap* map, const B3Operand& o, int rows, int K, int batch, int box_rows) {
  auto fn = encode_fn();
  if (!fn || !o.p || (reinterpret_cast<uintptr_t>(o.p) & 15) || (o.ld & 7) || o.ld < K) return false;
  const int64_t stride = batch > 1 ? o.stride : o.ld * (int64_t)rows;
  if ((stride & 7) || stride <= 0 || (o.plane & 7) || o.plane <= 0) return false;
  cuuint64_t dims[4] = {(cuuint64_t)K, (cuuint64_t)rows, (cuuint64_t)batch, 3};
  cuuint64_t strides[3] = {(cuuint64_t)o.ld * 2, (cuuint64_t)stride * 2, (cuuint64_t)o.plane * 2};
  cuuint32_t box[4] = {(cuuint32_t)BK, (cuuint32_t)box_rows, 1, 3};
  cuuint32_t es[4] = {1, 1, 1, 1};
  return fn(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, const_cast<__nv_bfloat16*>(o.p), dims, strides, box, es,
            CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

template <int CG, int BN, int MODE>
cudaError_t launch(int M, int N, int K, int batch, const B3Operand& A, const B3Operand& B, const B3Epilogue& ep,
                   cudaStream_t s) {
  using C = Cfg<CG, BN>;
  constexpr bool SYM = MODE & kSym;
  CUtensorMap ta, tb;
  Args p{M, N, K, batch, A.batch > 0 ? A.batch : batch, B.batch > 0 ? B.batch : batch, ep};
  if (!make_map(&ta, A, M, K, p.a_mod, BM) || !make_map(&tb, B, N, K, p.b_mod, C::BROWS)) return cudaErrorInvalidValue;
  auto* fn = gemm_b3_kernel<CG, BN, MODE>;
  // the shared-memory attribute belongs to each device's context: one bit per device that has it
  static std::atomic<uint64_t> attr_set{0};
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) dev = 0;
  const uint64_t bit = (dev >= 0 && dev < 64) ? uint64_t(1) << dev : 0;
  if (bit == 0 || !(attr_set.load(std::memory_order_relaxed) & bit)) {
    cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, C::SMEM);
    if (e != cudaSuccess) return e;
    attr_set.fetch_or(bit, std::memory_order_relaxed);
  }
  constexpr int TM = CG * BM;
  const int64_t ntm = (M + TM - 1) / TM;
  const int64_t ntiles = (SYM ? ntm * (ntm + 1) / 2 : (int64_t)((N + BN - 1) / BN) * ntm) * batch;
  if (ntiles > (int64_t)1 << 30) return cudaErrorInvalidValue;
  // short K: a cluster runs up to 8 tiles in turn, so that the next tile's loads and MMAs overlap the
  // current epilogue (for longer K the epilogue is a small part of a tile's time), the number that
  // leaves the fewest cluster slots idle in the last wave. (Not one launch-long run: clusters that
  // end give their SMs to the QR chain's small launches on the high-priority streams.)
  const int64_t slots = 152 / CG;
  int tpc = 1;
  if (K <= 2048) {
    int64_t best = ((ntiles + slots - 1) / slots);
    for (int t = 2; t <= 8; ++t) {
      const int64_t clusters = (ntiles + t - 1) / t, time = (clusters + slots - 1) / slots * t;
      if (clusters >= slots && time <= best) {
        best = time;
        tpc = t;
      }
    }
  }
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)((ntiles + tpc - 1) / tpc * CG), 1, 1);
  cfg.blockDim = dim3(THREADS, 1, 1);
  cfg.dynamicSmemBytes = C::SMEM;
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = CG;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = CG == 1 ? 0 : 1;
  return cudaLaunchKernelEx(&cfg, fn, ta, tb, p);
}

template <int MODE>
cudaError_t launch_shape(int M, int N, int K, int batch, const B3Operand& A, const B3Operand& B, const B3Epilogue& ep,
                         cudaStream_t s) {
  auto tiles = [&](int64_t t) {
    const int64_t tm = (M + t - 1) / t, tn = (N + t - 1) / t;
    return ((MODE & kSym) ? tm * (tm + 1) / 2 : tm * tn) * batch;
  };
  // waves of single CTAs and of pairs, a K block of a single CTA's tile taking about 0.6 of a pair's
  const int64_t w1 = (tiles(128) + 151) / 152, w2 = (tiles(256) + 75) / 76;
  if (M <= BM || N <= BM || 6 * w1 < 10 * w2) return launch<1, 128, MODE>(M, N, K, batch, A, B, ep, s);
  return launch<2, 256, MODE>(M, N, K, batch, A, B, ep, s);
}

bool al16(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15) == 0; }

}  // namespace
}  // namespace b3

cudaError_t gemm_b3(int M, int N, int K, int batch, const B3Operand& A, const B3Operand& B, const B3Epilogue& ep_in,
                    cudaStream_t s, int family) {
  using namespace b3;
  if (M <= 0 || N <= 0 || batch <= 0) return cudaSuccess;
  B3Epilogue ep = ep_in;
  get_wait_limit(&ep.wait_ns, &ep.hold);
  if (batch > 65535 || K <= 0) return cudaErrorInvalidValue;
  const bool f32 = ep.C || ep.C_ptrs, pl = ep.P != nullptr, tr = ep.transpose != 0, beta = ep.beta != 0.f;
  const bool betap = beta && ep.cin;
  // outputs are read and written in 16-byte units of fp32 (8-byte units of a plane)
  const int along = tr ? M : N;
  if ((along & 3) || f32 == pl || (beta && !f32 && !betap) || (betap && (tr || (pl && ep.cin != ep.P))) || (f32 && ((ep.ldc & 3) || (ep.c_stride & 3) || !al16(ep.C))) ||
      ((pl || betap) && ((ep.p_ld & 3) || (ep.p_stride & 3) || (ep.p_plane & 3) || !al16(ep.P) || !al16(ep.cin))))
    return cudaErrorInvalidValue;
  const double e = (double)M * N * batch;
  const double flops = 2.0 * e * K;  // algorithmic (six bf16 products each on the pipe)
  const double bytes = 6.0 * (double)M * K * (A.batch > 0 ? A.batch : batch) +
                       6.0 * (double)N * K * (B.batch > 0 ? B.batch : batch) + e * ((pl ? 6.0 : 4.0) + (betap ? 6.0 : beta ? 4.0 : 0.0));
  ProfScope prof(family, flops, bytes, s);
  if (tr) {
    if (pl) return launch_shape<kPlanes | kTr>(M, N, K, batch, A, B, ep, s);
    return beta ? launch_shape<kF32 | kTr | kBeta>(M, N, K, batch, A, B, ep, s)
                : launch_shape<kF32 | kTr>(M, N, K, batch, A, B, ep, s);
  }
  if (betap)
    return pl ? launch_shape<kPlanes | kBetaP>(M, N, K, batch, A, B, ep, s)
              : launch_shape<kF32 | kBetaP>(M, N, K, batch, A, B, ep, s);
  if (pl) return launch_shape<kPlanes>(M, N, K, batch, A, B, ep, s);
  return beta ? launch_shape<kF32 | kBeta>(M, N, K, batch, A, B, ep, s)
              : launch_shape<kF32>(M, N, K, batch, A, B, ep, s);
}

cudaError_t gemm_b3_syrk(int M, int K, int batch, const B3Operand& A, const B3Epilogue& ep_in, cudaStream_t s,
                         int family) {
  using namespace b3;
  if (M <= 0 || batch <= 0) return cudaSuccess;
  B3Epilogue ep = ep_in;
  get_wait_limit(&ep.wait_ns, &ep.hold);
  if (batch > 65535 || K <= 0 || !ep.C || !ep.P || ep.C_ptrs || ep.transpose || ep.beta == 0.f || (M & 3) ||
      (ep.ldc & 3) || (ep.c_stride & 3) || !al16(ep.C) || (ep.p_ld & 3) || (ep.p_stride & 3) || (ep.p_plane & 3) ||
      !al16(ep.P))
    return cudaErrorInvalidValue;
  const int tile = BM;
  const double ntm = (double)((M + tile - 1) / tile);
  const double flops = 2.0 * tile * tile * (double)K * (ntm * (ntm + 1) / 2 * batch);  // the lower tiles' products
  const double bytes = 6.0 * (double)M * K * (A.batch > 0 ? A.batch : batch) + (4.0 * 1.5 + 6.0) * (double)M * M * batch;
  ProfScope prof(family, flops, bytes, s);
  return launch_shape<kF32 | kPlanes | kBeta | kSym>(M, M, K, batch, A, A, ep, s);
}

}  // namespace soap
