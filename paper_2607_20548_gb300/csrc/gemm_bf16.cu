// Batched bf16 GEMM on the 5th-generation tensor cores (tcgen05, kind::f16), fp32 accumulation:
//
//   out_b = alpha * A_b * B_b^T + beta * Cin_b       (A_b M x K, B_b N x K, both row-major)
//
// written as bf16, row-major and optionally transposed as well. It serves the Newton-Schulz
// iterations of Muon, which run in bf16 (products of bf16 operands accumulated in fp32, results
// stored in bf16). A symmetric product (A = B, M = N) computes the tiles on or below the diagonal
// only and stores each one below it in the mirror position too: two of the three products of an
// iteration, X X^T and A A^T, at half the MMAs (the two halves' bits are the same: an element and
// its mirror sum the same products in the same order), where that saves more than the mirrored stores
// cost.
//
// A pair of CTAs (cta_group::2) works on a 256 x 256 tile: with one CTA per 128 x 128 tile, shared
// memory took 256 bytes of operand reads and refills per cycle of MMA time, twice what it sustains,
// and the products ran at 0.46 of the sustained tensor peak. In the pair each CTA loads its own 128
// rows of A and half of B's rows, and the same traffic feeds four times the MMAs. Small and ragged
// products keep one CTA per 128 x 128 tile: which one is taken is decided on the estimated times at the
// end of this file.
//
// Persistent clusters walk the output tiles in groups of row tiles. Warp 0 issues the TMA loads
// of 64-element K slices (one 128-byte swizzle row per matrix row) into a ring, warp 1 of the
// pair's first CTA issues the MMAs into one of two TMEM accumulators, used in turn by consecutive
// tiles so that a tile's epilogue overlaps the next tile's MMAs, and 8 epilogue warps drain the
// accumulator (tensor memory -> registers -> alpha/beta -> bf16 stores). Every mbarrier wait gives
// up after ~2 s of %globaltimer time, records kStatusTimeout and lets the CTAs drain and free
// their tensor memory instead of hanging.
#include <cuda.h>
#include <cuda_bf16.h>
#include <cudaTypedefs.h>

#include <algorithm>
#include <atomic>
#include <mutex>

#include "profile.h"
#include "soap_internal.h"
#include "tc_ptx.h"

namespace soap {
namespace bf16g {
namespace {

using tc::smem_u32;

constexpr int BM = 128;  // rows of A per CTA
constexpr int BK = 64;   // bf16 elements per K slice = one 128-byte swizzle row
constexpr int NACC = 2;
constexpr int EPI = 8;
constexpr int THREADS = 64 + 32 * EPI;
constexpr int STAGES = 6;
constexpr int TILE_A = BM * BK * 2;
constexpr uint64_t kWaitNs = 2000000000ull;

// CG CTAs work on a CG * 128 x CG * 128 tile, each with its 128 rows of A and 128 of B.
template <int CG>
struct Cfg {
  static constexpr int T = CG * BM;
  static constexpr int STAGE = 2 * TILE_A;
  static constexpr int SMEM = STAGES * STAGE + 1024 + 256;
  static constexpr int NCH = T / 64;  // 32-column chunks of one epilogue warp
  static constexpr uint32_t TMEM_COLS = NACC * T;
};

template <int CG>
__device__ __forceinline__ void tma_load(uint32_t dst, const CUtensorMap* map, uint32_t bar, int c0, int c1, int c2) {
  if (CG == 1)
    asm volatile(
        "cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, %5}], [%2];" ::"r"(
            dst),
        "l"(reinterpret_cast<uint64_t>(map)), "r"(bar), "r"(c0), "r"(c1), "r"(c2)
        : "memory");
  else
    asm volatile(
        "cp.async.bulk.tensor.3d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, "
        "%5}], [%2];" ::"r"(dst),
        "l"(reinterpret_cast<uint64_t>(map)), "r"(bar), "r"(c0), "r"(c1), "r"(c2)
        : "memory");
}

// Tile t -> (m0, n0, batch index): in groups of 1024 rows (m fastest inside a group), or, for a
// symmetric product, the tiles on or below the diagonal row by row.
template <int T, bool SYM>
__device__ __forceinline__ void tile_coords(int t, int ntm, int ntn, int& m0, int& n0, int& b) {
  if (SYM) {
    const int per = ntm * (ntm + 1) / 2;
    b = t / per;
    const int r = t - b * per;
    int i = (int)((sqrtf(8.f * (float)r + 1.f) - 1.f) * 0.5f);
    while ((i + 1) * (i + 2) / 2 <= r) ++i;
    while (i * (i + 1) / 2 > r) --i;
    m0 = i * T;
    n0 = (r - i * (i + 1) / 2) * T;
  } else {
    constexpr int GM = 1024 / T;
    const int per = ntm * ntn;
    b = t / per;
    const int r = t - b * per;
    const int g = r / (GM * ntn);
    const int first = g * GM;
    const int gsz = min(GM, ntm - first);
    const int w = r - g * GM * ntn;
    m0 = (first + w % gsz) * T;
    n0 = (w / gsz) * T;
  }
}

template <int CG, bool SYM>
__global__ void __launch_bounds__(THREADS, 1)
    gemm_bf16_kernel(const __grid_constant__ CUtensorMap ta, const __grid_constant__ CUtensorMap tb, int M, int N,
                     int K, int batch, const __grid_constant__ Bf16Epilogue ep) {
  using C = Cfg<CG>;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint64_t* full = reinterpret_cast<uint64_t*>(smem + STAGES * C::STAGE);
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
  const int kblocks = (K + BK - 1) / BK;
  const int ntn = (N + C::T - 1) / C::T, ntm = (M + C::T - 1) / C::T;
  const int ntiles = (SYM ? ntm * (ntm + 1) / 2 : ntn * ntm) * batch;
  const int t_first = blockIdx.x / CG, t_step = gridDim.x / CG;

  if (threadIdx.x == 0) {
    for (int s = 0; s < STAGES; ++s) {
      tc::mbar_init(&full[s], 1);
      tc::mbar_init(&empty[s], 1);
    }
    for (int a = 0; a < NACC; ++a) {
      tc::mbar_init(&acc_full[a], 1);
      tc::mbar_init(&acc_empty[a], EPI * CG);
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
      int g = 0, issued = 0;
      for (int t = t_first; t < ntiles && !*abort_flag; t += t_step) {
        int m0, n0, b;
        tile_coords<C::T, SYM>(t, ntm, ntn, m0, n0, b);
        for (int kb = 0; kb < kblocks; ++kb, ++g) {
          const int s = g % STAGES;
          if (!tc::wait<CG>(&empty[s], ((g / STAGES) & 1) ^ 1, kWaitNs) || *abort_flag) {
            *abort_flag = 1;
            break;
          }
          if (lead) tc::mbar_expect_tx(&full[s], CG * C::STAGE);
          const uint32_t st = smem_u32(smem + s * C::STAGE), bar = tc::lead_addr<CG>(smem_u32(&full[s]));
          tma_load<CG>(st, &ta, bar, kb * BK, m0 + rank * BM, b);
          tma_load<CG>(st + TILE_A, &tb, bar, kb * BK, n0 + rank * BM, b);
          issued = g + 1;
        }
      }
      ring->issued = issued;
    }
  } else if (warp == 1) {
    if (lane == 0 && lead) {
      constexpr uint32_t idesc = tc::idesc_bf16(C::T, C::T);
      int g = 0, tl = 0;
      bool ok = true;
      for (int t = t_first; t < ntiles && ok && !*abort_flag; t += t_step, ++tl) {
        const int a = tl % NACC;
        if (tl >= NACC && !tc::wait<CG>(&acc_empty[a], ((tl / NACC) & 1) ^ 1, kWaitNs)) {
          ok = false;
          break;
        }
        tc::tc_fence_after();
        const uint32_t d = tmem + static_cast<uint32_t>(a * C::T);
        for (int kb = 0; kb < kblocks; ++kb, ++g) {
          const int s = g % STAGES;
          if (!tc::wait<CG>(&full[s], (g / STAGES) & 1, kWaitNs) || *abort_flag) {
            ok = false;
            break;
          }
          *consumed = g + 1;
          tc::tc_fence_after();
          const uint32_t a_s = smem_u32(smem + s * C::STAGE), b_s = a_s + TILE_A;
#pragma unroll
          for (int kk = 0; kk < BK / 16; ++kk)  // 16 bf16 = 32 bytes along K inside the swizzle row
            tc::umma_f16<CG>(d, a_s + kk * 32, b_s + kk * 32, idesc, (kb | kk) != 0);
          tc::commit<CG>(&empty[s]);  // frees the stage once these MMAs have read it
        }
        if (ok) {
          tc::commit<CG>(&acc_full[a]);  // hands the tile's sum to the epilogue warps
          ring->accs = tl + 1;
        }
      }
      if (!ok) *abort_flag = 1;
      if (g > 0) {  // every MMA issued has completed before the tensor memory is freed
        tc::commit<CG>(mma_done);
        tc::wait<CG>(mma_done, 0, kWaitNs);
      }
    }
  } else {
    const int q = warp & 3;                              // accumulator lanes 32q .. 32q+31
    const int colbase = ((warp - 2) / 4) * (C::T / 2);   // this warp's columns: half of the tile's
    const uint32_t lane_base = tmem + (static_cast<uint32_t>(32 * q) << 16);
    int tl = 0;
    for (int t = t_first; t < ntiles; t += t_step, ++tl) {
      int m0, n0, b;
      tile_coords<C::T, SYM>(t, ntm, ntn, m0, n0, b);
      const int a = tl % NACC;
      if (!tc::wait<CG>(&acc_full[a], (tl / NACC) & 1, kWaitNs) || *abort_flag) {
        if (lane == 0 && ep.status) atomicOr(ep.status, kStatusTimeout);
        *abort_flag = 1;
        break;
      }
      tc::tc_fence_after();
      const int r = m0 + rank * BM + 32 * q + lane;  // this lane's output row
      const int64_t ob = (int64_t)b * ep.stride;
      // the transposed copy: a buffer of its own, or the mirror tile of a symmetric product
      const bool mirror = SYM && m0 != n0;
      __nv_bfloat16* out_t = SYM ? (mirror ? ep.out + ob : nullptr)
                                 : (ep.out_t ? ep.out_t + (int64_t)b * ep.stride_t : nullptr);
      const int64_t ld_t = SYM ? ep.ld : ep.ld_t;
      // a single CTA's warp takes its 64 columns out of the accumulator at once; a pair's 128 go through
      // the registers 32 at a time
      constexpr int NV = CG == 1 ? C::NCH : 1;
      float v[NV][32];
      auto drained = [&] {
        tc::tc_fence_before();
        __syncwarp();
        if (lane == 0) tc::arrive_lead<CG>(&acc_empty[a]);
      };
      if (CG == 1) {
#pragma unroll
        for (int c = 0; c < NV; ++c) tc::tmem_ld32(lane_base + static_cast<uint32_t>(a * C::T + colbase + 32 * c), v[c]);
        drained();
      }
#pragma unroll NV
      for (int c = 0; c < C::NCH; ++c) {
        float(&o)[32] = v[CG == 1 ? c : 0];
        if (CG == 2) {
          tc::tmem_ld32(lane_base + static_cast<uint32_t>(a * C::T + colbase + 32 * c), o);
          if (c == C::NCH - 1) drained();
        }
        const int c0 = n0 + colbase + 32 * c;
        if (c0 >= N) continue;
#pragma unroll
        for (int j = 0; j < 32; ++j) o[j] *= ep.alpha;
        if (r < M && ep.beta != 0.f && ep.cin) {
          const __nv_bfloat16* src = ep.cin + ob + (int64_t)r * ep.ld + c0;
#pragma unroll
          for (int u = 0; u < 4; ++u) {
            if (c0 + 8 * u >= N) break;
            const uint4 w = *reinterpret_cast<const uint4*>(src + 8 * u);
            const __nv_bfloat162* h2 = reinterpret_cast<const __nv_bfloat162*>(&w);
#pragma unroll
            for (int e = 0; e < 4; ++e) {
              const float2 f = __bfloat1622float2(h2[e]);
              o[8 * u + 2 * e] = fmaf(ep.beta, f.x, o[8 * u + 2 * e]);
              o[8 * u + 2 * e + 1] = fmaf(ep.beta, f.y, o[8 * u + 2 * e + 1]);
            }
          }
        }
        uint32_t w2[16];  // columns 2 e, 2 e + 1 of this lane's row
#pragma unroll
        for (int e = 0; e < 16; ++e) {
          const __nv_bfloat162 h = __floats2bfloat162_rn(o[2 * e], o[2 * e + 1]);
          w2[e] = reinterpret_cast<const uint32_t&>(h);
        }
        if (r < M) {
          __nv_bfloat16* dst = ep.out + ob + (int64_t)r * ep.ld + c0;
#pragma unroll
          for (int u = 0; u < 4; ++u)
            if (c0 + 8 * u < N)
              *reinterpret_cast<uint4*>(dst + 8 * u) = make_uint4(w2[4 * u], w2[4 * u + 1], w2[4 * u + 2], w2[4 * u + 3]);
        }
        if (CG == 1 && out_t) {
          // for each column the warp's 32 rows are 32 consecutive elements
          __nv_bfloat16* dst = out_t + (int64_t)c0 * ld_t + r;
          const unsigned short* h = reinterpret_cast<const unsigned short*>(w2);
#pragma unroll
          for (int j = 0; j < 32; ++j)
            if (r < M && c0 + j < N) reinterpret_cast<unsigned short*>(dst)[(int64_t)j * ld_t] = h[j];
        }
        if (CG == 2 && out_t) {
          // two neighbouring rows of a column make a 4-byte word: even lanes take the even columns,
          // odd lanes the odd ones (M is a multiple of 8, so the rows of a pair are both in or out)
          const bool odd = lane & 1;
          __nv_bfloat16* dst = out_t + (int64_t)(c0 + odd) * ld_t + (r & ~1);
#pragma unroll
          for (int e = 0; e < 16; ++e) {
            const uint32_t other = __shfl_xor_sync(0xffffffffu, w2[e], 1);
            const uint32_t v = odd ? __byte_perm(other, w2[e], 0x7632) : __byte_perm(w2[e], other, 0x5410);
            if (r < M && c0 + 2 * e < N) *reinterpret_cast<uint32_t*>(dst + (int64_t)(2 * e) * ld_t) = v;
          }
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

// Tensor map of `batch` row-major rows x K bf16 matrices, tiles of 128 x 64.
bool make_map(CUtensorMap* map, const __nv_bfloat16* base, int rows, int K, int64_t ld, int64_t stride, int batch) {
  auto fn = encode_fn();
  if (!fn || !base) return false;
  if ((reinterpret_cast<uintptr_t>(base) & 15) || (ld & 7) || ld < K) return false;
  if (batch <= 1) stride = ld * rows;
  if ((stride & 7) || stride < ld * rows) return false;
  cuuint64_t dims[3] = {(cuuint64_t)K, (cuuint64_t)rows, (cuuint64_t)(batch < 1 ? 1 : batch)};
  cuuint64_t strides[2] = {(cuuint64_t)ld * 2, (cuuint64_t)stride * 2};
  cuuint32_t box[3] = {(cuuint32_t)BK, (cuuint32_t)BM, 1};
  cuuint32_t es[3] = {1, 1, 1};
  return fn(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<__nv_bfloat16*>(base), dims, strides, box, es,
            CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

int64_t tile_count(int M, int N, int batch, int t, bool sym) {
  const int64_t tm = (M + t - 1) / t, tn = (N + t - 1) / t;
  return (sym ? tm * (tm + 1) / 2 : tm * tn) * batch;
}

// Which kernel: one CTA or a pair per tile, and for a symmetric product all tiles or the lower ones
// mirrored. The smallest estimate of  launch + waves * (K slices * slice + epilogue)  in us, the
// coefficients fitted to 2800 products (sides 64 ... 3072, K 64 ... 8192, batches of 1 ... 64, each
// timed in every form): the form taken is 0.5 % slower than the fastest on average. A pair's slice is
// as long as a single CTA's and does four times the work, but its 128 x 256 values per CTA take the
// epilogue's 8 warps two to three times as long, and partly empty tiles take whole ones' time. (Counting
// waves alone sent short and ragged products to pairs and halves: 64 of 200 x 800, 16 steps, 1.39 ms;
// 1.22 with all products whole on single CTAs.)
enum Kind { kSingles, kLowerSingles, kPairs, kLowerPairs };
Kind choose(int M, int N, int K, int batch, int sms, bool symmetric) {
  const int slices = (K + BK - 1) / BK;
  auto us = [&](int cg, bool lower, double launch, double slice, double epilogue) {
    const int64_t slots = std::max(1, sms / cg), waves = (tile_count(M, N, batch, cg * BM, lower) + slots - 1) / slots;
    return launch + waves * (slices * slice + epilogue);
  };
  if (!symmetric) return M > BM && N > BM && us(2, false, 6.4, 0.24, 9.9) < us(1, false, 4.3, 0.27, 3.5) ? kPairs : kSingles;
  const double whole = us(1, false, 4.4, 0.26, 1.6), lower = us(1, true, 4.0, 0.30, 1.9);
  if (M > BM && us(2, true, 5.9, 0.33, 4.0) < std::min(whole, lower)) return kLowerPairs;
  return lower < whole ? kLowerSingles : kSingles;
}

template <int CG, bool SYM>
cudaError_t launch(const CUtensorMap& ta, const CUtensorMap& tb, int M, int N, int K, int batch, const Bf16Epilogue& ep,
                   int dev, int sms, cudaStream_t s) {
  auto* fn = gemm_bf16_kernel<CG, SYM>;
  // the shared-memory attribute belongs to each device's context: one bit per device that has it
  static std::atomic<uint64_t> attr_set{0};
  const uint64_t bit = (dev >= 0 && dev < 64) ? uint64_t(1) << dev : 0;
  if (bit == 0 || !(attr_set.load(std::memory_order_relaxed) & bit)) {
    cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, Cfg<CG>::SMEM);
    if (e != cudaSuccess) return e;
    attr_set.fetch_or(bit, std::memory_order_relaxed);
  }
  const int64_t ntiles = tile_count(M, N, batch, CG * BM, SYM);
  if (ntiles > (int64_t)1 << 30) return cudaErrorInvalidValue;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(std::min<int64_t>(ntiles, std::max(1, sms / CG)) * CG), 1, 1);
  cfg.blockDim = dim3(THREADS, 1, 1);
  cfg.dynamicSmemBytes = Cfg<CG>::SMEM;
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = CG;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = CG == 1 ? 0 : 1;  // (a launch with a cluster of one takes up to 0.3 us longer)
  return cudaLaunchKernelEx(&cfg, fn, ta, tb, M, N, K, batch, ep);
}

}  // namespace
}  // namespace bf16g

cudaError_t gemm_bf16_nt(int M, int N, int K, int batch, const __nv_bfloat16* A, int64_t lda, int64_t a_stride,
                         const __nv_bfloat16* B, int64_t ldb, int64_t b_stride, const Bf16Epilogue& ep,
                         cudaStream_t s) {
  using namespace bf16g;
  if (M <= 0 || N <= 0 || batch <= 0) return cudaSuccess;
  if (K <= 0 || batch > 65535 || (M & 7) || (N & 7) || (K & 7) || !ep.out) return cudaErrorInvalidValue;
  if ((ep.ld & 7) || (ep.stride & 7) || (ep.out_t && ((ep.ld_t & 1) || (ep.stride_t & 1)))) return cudaErrorInvalidValue;
  int dev = 0, sms = 152;
  if (cudaGetDevice(&dev) != cudaSuccess) dev = 0;
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  const bool symmetric = A == B && M == N && lda == ldb && a_stride == b_stride && !ep.out_t && ep.symmetric;
  const Kind kind = choose(M, N, K, batch, sms, symmetric);
  const bool sym = kind == kLowerSingles || kind == kLowerPairs;
  const double mn = (double)M * N * batch;
  ProfScope prof(kFamGemmTc, 2.0 * mn * K * (sym ? 0.5 : 1.0),
                 2.0 * ((double)M * K + (symmetric ? 0.0 : (double)N * K)) * batch +
                     mn * (2 + (ep.out_t ? 2 : 0) + (ep.beta != 0.f && ep.cin ? 2 : 0)),
                 s);
  CUtensorMap ta, tb;
  if (!make_map(&ta, A, M, K, lda, a_stride, batch) || !make_map(&tb, B, N, K, ldb, b_stride, batch))
    return cudaErrorInvalidValue;
  switch (kind) {
    case kSingles: return launch<1, false>(ta, tb, M, N, K, batch, ep, dev, sms, s);
    case kLowerSingles: return launch<1, true>(ta, tb, M, N, K, batch, ep, dev, sms, s);
    case kPairs: return launch<2, false>(ta, tb, M, N, K, batch, ep, dev, sms, s);
    default: return launch<2, true>(ta, tb, M, N, K, batch, ep, dev, sms, s);
  }
}

}  // namespace soap
