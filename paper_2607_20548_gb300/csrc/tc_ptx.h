// Inline-PTX helpers shared by the tcgen05 kernels (the GEMM and the QR panel): shared-memory
// addresses, bounded mbarrier waits, the 128-byte-swizzled K-major matrix descriptor, the
// kind::tf32 instruction descriptor and MMA, tensor-memory loads, and the tf32 lo part.
#pragma once

#include <cstdint>

namespace soap {
namespace tc {

__device__ __forceinline__ uint32_t smem_u32(const void* p) {
  return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

__device__ __forceinline__ uint64_t globaltimer() {
  uint64_t t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count));
}

__device__ __forceinline__ bool mbar_try(uint64_t* bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}\n"
      : "=r"(ok)
      : "r"(smem_u32(bar)), "r"(parity)
      : "memory");
  return ok != 0;
}

// Bounded wait on an mbarrier phase: false after `limit_ns` without completion.
__device__ __forceinline__ bool mbar_wait(uint64_t* bar, uint32_t parity, uint64_t limit_ns) {
  if (mbar_try(bar, parity)) return true;
  const uint64_t t0 = globaltimer();
  for (;;) {
    for (int i = 0; i < 16; ++i)
      if (mbar_try(bar, parity)) return true;
    if (globaltimer() - t0 > limit_ns) return false;
  }
}


// Shared-memory matrix descriptor: K-major, 128-byte swizzle, 8-row atoms 1024 B apart.
__device__ __forceinline__ uint64_t desc_sw128(uint32_t addr) {
  uint64_t d = 0;
  d |= static_cast<uint64_t>((addr & 0x3FFFF) >> 4);  // start address
  d |= static_cast<uint64_t>(1) << 16;                 // leading byte offset (unused for this layout)
  d |= static_cast<uint64_t>(1024 >> 4) << 32;         // stride byte offset: next 8-row atom
  d |= static_cast<uint64_t>(1) << 46;                 // descriptor version (sm_100 family)
  d |= static_cast<uint64_t>(2) << 61;                 // 128-byte swizzle
  return d;
}

// Instruction descriptor for kind::tf32: D = f32, A = B = tf32, both K-major.
__host__ __device__ constexpr uint32_t idesc_tf32(int M, int N) {
  return (1u << 4) | (2u << 7) | (2u << 10) | (static_cast<uint32_t>(N >> 3) << 17) |
         (static_cast<uint32_t>(M >> 4) << 24);
}

__device__ __forceinline__ void umma_tf32(uint32_t tmem_d, uint64_t adesc, uint64_t bdesc, uint32_t idesc,
                                          uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::tf32 [%0], %1, %2, %3, p;\n\t}\n" ::"r"(tmem_d),
      "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate));
}

__device__ __forceinline__ void umma_commit(uint64_t* bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_u32(bar))
               : "memory");
}

__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

__device__ __forceinline__ void tmem_ld32(uint32_t taddr, float (&v)[32]) {
  uint32_t r[32];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
      "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
      "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
        "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]),
        "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]),
        "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
      : "r"(taddr));
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
  for (int i = 0; i < 32; ++i) v[i] = __uint_as_float(r[i]);
}

// 16 accumulator columns of this warp's 32 lanes (half the registers of tmem_ld32)
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, float (&v)[16]) {
  uint32_t r[16];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 "
      "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
        "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
      : "r"(taddr));
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
  for (int i = 0; i < 16; ++i) v[i] = __uint_as_float(r[i]);
}

// ---- one CTA (CG = 1) or a pair of CTAs (CG = 2, a cluster of two) on one tile ------------------

__device__ __forceinline__ void mbar_expect_tx(uint64_t* bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes)
               : "memory");
}
// Address in the pair's first CTA of this CTA's shared-memory address.
template <int CG>
__device__ __forceinline__ uint32_t lead_addr(uint32_t a) {
  if (CG == 1) return a;
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, 0;" : "=r"(r) : "r"(a));
  return r;
}
// One arrival at a barrier of the pair's first CTA, by a warp that has drained an accumulator. What it
// hands over is tensor memory, ordered by the tcgen05 fences before the arrival and after the wait, so
// across the pair it is relaxed: a release at cluster scope first waited for the warp's own stores of
// the previous tile (the largest stall of the plane products, 41 %; dense block 67.6 -> 66.7 ms,
// Muon 8.36 -> 8.16 ms).
template <int CG>
__device__ __forceinline__ void arrive_lead(uint64_t* bar) {
  if (CG == 1)
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
  else
    asm volatile("mbarrier.arrive.relaxed.cluster.shared::cluster.b64 _, [%0];" ::"r"(lead_addr<CG>(smem_u32(bar)))
                 : "memory");
}
__device__ __forceinline__ bool mbar_try_cluster(uint64_t* bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}\n"
      : "=r"(ok)
      : "r"(smem_u32(bar)), "r"(parity)
      : "memory");
  return ok != 0;
}
// Bounded wait; the barrier may have been arrived at from the other CTA.
template <int CG>
__device__ __forceinline__ bool wait(uint64_t* bar, uint32_t parity, uint64_t limit_ns) {
  if (CG == 1) return mbar_wait(bar, parity, limit_ns);
  if (mbar_try_cluster(bar, parity)) return true;
  const uint64_t t0 = globaltimer();
  for (;;) {
    for (int i = 0; i < 16; ++i)
      if (mbar_try_cluster(bar, parity)) return true;
    if (globaltimer() - t0 > limit_ns) return false;
  }
}
// Instruction descriptor for kind::f16: D = f32, A = B = bf16, both K-major.
__host__ __device__ constexpr uint32_t idesc_bf16(int M, int N) {
  return (1u << 4) | (1u << 7) | (1u << 10) | (static_cast<uint32_t>(N >> 3) << 17) |
         (static_cast<uint32_t>(M >> 4) << 24);
}
template <int CG>
__device__ __forceinline__ void umma_f16(uint32_t d, uint32_t a, uint32_t b, uint32_t idesc, uint32_t accumulate) {
  if (CG == 1)
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}\n" ::"r"(d),
        "l"(desc_sw128(a)), "l"(desc_sw128(b)), "r"(idesc), "r"(accumulate));
  else
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\n\t}\n" ::"r"(d),
        "l"(desc_sw128(a)), "l"(desc_sw128(b)), "r"(idesc), "r"(accumulate));
}
// Completion of the MMAs issued so far, to the same barrier of every CTA of the tile.
template <int CG>
__device__ __forceinline__ void commit(uint64_t* bar) {
  if (CG == 1)
    umma_commit(bar);
  else
    asm volatile(
        "tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;" ::"r"(
            smem_u32(bar)),
        "h"((uint16_t)3)
        : "memory");
}

// What the warps of a CTA that feed a pair's (or a CTA's) MMAs leave behind for finish(), in shared memory.
struct RingState {
  int abort;     // a wait gave up
  int consumed;  // K blocks whose MMAs were issued (kept by the pair's first CTA)
  int accs;      // accumulators handed to the epilogue warps (likewise)
  int issued;    // K blocks whose copies this CTA issued
};

// The last thing every thread of a tile kernel does before its tensor memory is freed and its CTA
// exits: nothing may then still arrive in the shared memory of either CTA. That is,
//  * the commits' arrivals, which go to both CTAs of a pair on their own: each waits for its own copies
//    (a single CTA's epilogue has waited for the last of them);
//  * the arrivals of the epilogue warps, performed before the cluster barrier;
//  * after a wait that gave up, copies in flight. Both CTAs' copies of a K block count on the first
//    CTA's barrier, and one producer may have gone a block further than the other: the CTAs tell each
//    other how far they got, the first one makes up the count of the halves that were never issued, or
//    not expected, and the pair leaves together.
// st[0] is this CTA's state, st[1] takes the peer's; every wait is bounded. The waits of a warp's lanes
// go side by side (in turn they cost a launch of few tiles up to a microsecond).
template <int CG, int STAGES, int NACC>
__device__ __forceinline__ void finish(uint64_t* full, uint64_t* empty, uint64_t* acc_full, uint64_t* mma_done,
                                       RingState* st_, bool lead, uint32_t stage_bytes, uint64_t limit_ns) {
  static_assert(STAGES + NACC < 32, "a lane for every barrier");
  volatile RingState* st = st_;
  tc_fence_before();
  __syncthreads();
  if (CG == 1 && !st[0].abort) return;
  if (CG == 2) {
    if (threadIdx.x < sizeof(RingState) / 4) {
      const uint32_t dst = smem_u32(st_ + 1) + 4 * threadIdx.x;
      const int v = reinterpret_cast<volatile int*>(st_)[threadIdx.x];
      asm volatile(
          "{\n\t.reg .b32 a;\n\t"
          "mapa.shared::cluster.u32 a, %0, %1;\n\t"
          "st.shared::cluster.b32 [a], %2;\n\t}\n" ::"r"(dst),
          "r"(lead ? 1 : 0), "r"(v)
          : "memory");
    }
    __syncwarp();
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
  }
  if (threadIdx.x < 32) {
    const int first = CG == 1 || lead ? 0 : 1;  // the first CTA's entry
    const int consumed = st[first].consumed, accs = st[first].accs, l = (int)threadIdx.x;
    if (l < STAGES) {
      const int g = consumed - 1 - l;
      if (g >= 0) wait<CG>(&empty[g % STAGES], (g / STAGES) & 1, limit_ns);
    } else if (l < STAGES + NACC) {
      const int g = accs - 1 - (l - STAGES);
      if (g >= 0) wait<CG>(&acc_full[g % NACC], (g / NACC) & 1, limit_ns);
    } else if (l == STAGES + NACC && consumed > 0) {
      wait<CG>(mma_done, 0, limit_ns);
    }
    if (l == 0 && lead) {
      const int mine = st[0].issued, theirs = CG == 2 ? st[1].issued : mine;
      for (int g = consumed; g < mine || g < theirs; ++g) {
        uint64_t* bar = &full[g % STAGES];
        if (g >= mine) mbar_expect_tx(bar, stage_bytes);
        if (g >= theirs)
          asm volatile("mbarrier.complete_tx.relaxed.cta.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(stage_bytes)
                       : "memory");
        wait<CG>(bar, (g / STAGES) & 1, limit_ns);
      }
    }
    __syncwarp();
  }
  if (CG == 2 && (st[0].abort | st[1].abort)) {  // the same for all threads of both CTAs
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
  }
}

// tf32 value the tensor core reads from an fp32 word (13 low mantissa bits dropped), and
// the lo part x - trunc(x) rounded to the nearest tf32 (so the tensor core reads it exactly).
__device__ __forceinline__ float tf32_trunc(float x) { return __uint_as_float(__float_as_uint(x) & 0xFFFFE000u); }
__device__ __forceinline__ float tf32_lo(float x) {
  uint32_t r;
  asm("cvt.rna.tf32.f32 %0, %1;" : "=r"(r) : "f"(x - tf32_trunc(x)));
  return __uint_as_float(r);
}

}  // namespace tc
}  // namespace soap
