// tc_ptx.cuh -- PTX wrappers shared by the tensor-core kernels: mbarriers and
// bounded waits, TMA copies, tcgen05 descriptors, MMAs, commits and TMEM
// loads, and the column sums of a 32 x 32 register chunk.
#pragma once

#include <cuda.h>
#include <cuda_bf16.h>
#include <stdint.h>

namespace tp {
namespace {

// ------------------------------------------------------------ PTX helpers
__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ uint64_t global_ns() {
  uint64_t t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint64_t* bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes) : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint64_t* bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint64_t* bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
      : "=r"(ok)
      : "r"(smem_u32(bar)), "r"(parity)
      : "memory");
  return ok != 0;
}
// Bounded wait: false if the abort flag is raised or the budget runs out
// (then the flag and the device error word are set).
// A wait that gives up records its site code in the error word (the first
// one wins): 1 producer stage empty, 3 producer dependency, 5 MMA
// accumulator free, 6 MMA stage full, 7 epilogue accumulator full, 10 final
// copy drain, 12 final MMA drain, 8 epilogue publish slot, 9 publisher,
// 13 epilogue Newton-Schulz dependency, 14 epilogue bias-partial dependency.
// 21 .. 29: the tensor-core head kernel's.
// The MMA and epilogue waits (5, 6, 7, 8) wait on another role of the same
// CTA and take twice the budget of the producer's, the publisher's (9) four
// times, so a stalled dependency is reported as its own site.
__device__ __noinline__ bool mbar_wait_slow(uint64_t* bar, uint32_t parity, volatile int* abort_flag, int* err,
                                            uint64_t budget_ns, int site) {
  if (mbar_try_wait(bar, parity)) return true;
  const uint64_t t0 = global_ns();
  while (true) {
    if (mbar_try_wait(bar, parity)) return true;
    if (*abort_flag) return false;
    if (global_ns() - t0 > budget_ns) {
      *abort_flag = 1;
      atomicCAS(err, 0, site);
      return false;
    }
  }
}

__device__ __forceinline__ bool mbar_wait(uint64_t* bar, uint32_t parity, volatile int* abort_flag, int* err,
                                          uint64_t budget_ns, int site) {
  return mbar_try_wait(bar, parity) || mbar_wait_slow(bar, parity, abort_flag, err, budget_ns, site);
}

__device__ __forceinline__ int ld_acquire(const int* p) {
  int v;
  asm volatile("ld.acquire.gpu.global.s32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ void red_release_add(int* p, int v) {
  asm volatile("red.release.gpu.global.add.s32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}
// Generic-proxy writes of other CTAs, acquired through a counter, become
// visible to this thread's subsequent TMA (async-proxy) reads.
__device__ __forceinline__ void fence_proxy_async_global() {
  asm volatile("fence.proxy.async.global;" ::: "memory");
}

// Bounded wait, by the whole warp, until counters p[0 .. n-1] each reach
// `need`.  Lane j polls counters j, j + 32, ...: a weight-gradient tile waits
// on every row block of its operand (16 counters for 2048 rows), and one
// lane reading them in turn paid 16 acquire round trips to L2 per tile even
// when all were long complete.  The warp barrier orders every lane after all
// lanes' acquires; the caller's proxy fence follows it.
__device__ __noinline__ bool dep_wait(const int* p, int n, int need, volatile int* abort_flag, int* err,
                                      uint64_t budget_ns, int site, int lane) {
  bool mine = true;
  for (int j = lane; mine && j < n; j += 32) {
    if (ld_acquire(p + j) >= need) continue;
    const uint64_t t0 = global_ns();
    while (ld_acquire(p + j) < need) {
      if (*abort_flag) {
        mine = false;
        break;
      }
      if (global_ns() - t0 > budget_ns) {
        *abort_flag = 1;
        atomicCAS(err, 0, site);
        mine = false;
        break;
      }
      __nanosleep(32);
    }
  }
  __syncwarp();
  return __all_sync(0xffffffffu, mine);
}

// Column sums of a warp's 32 x 32 chunk (lane = row, c[j] = column j):
// halving exchanges (16 + 8 + 4 + 2 + 1 shuffles), after which lane l
// holds column l's sum in c[0].  The order of the additions is fixed.
template <int W>
__device__ __forceinline__ void colsum_halve(float (&c)[32], int lane) {
  const bool up = (lane & W) != 0;
#pragma unroll
  for (int k = 0; k < W; ++k) {
    const float keep = up ? c[W + k] : c[k];
    const float send = up ? c[k] : c[W + k];
    c[k] = keep + __shfl_xor_sync(0xffffffffu, send, W);
  }
}
__device__ __forceinline__ float colsum32(float (&c)[32], int lane) {
  colsum_halve<16>(c, lane);
  colsum_halve<8>(c, lane);
  colsum_halve<4>(c, lane);
  colsum_halve<2>(c, lane);
  colsum_halve<1>(c, lane);
  return c[0];
}

// p[0] + p[ld] + ... + p[(n - 1) ld], added in that order (kept out of line:
// inlined, its loop state raised the epilogue's register spills).
__device__ __noinline__ float sum_strided(const float* p, int n, int ld) {
  float s = 0.f;
#pragma unroll 8
  for (int i = 0; i < n; ++i) s += p[(int64_t)i * ld];
  return s;
}

// Bulk prefetch of `bytes` (a multiple of 16; 16-byte aligned address) into L2.
__device__ __forceinline__ void prefetch_l2(const void* p, uint32_t bytes) {
  asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(p), "r"(bytes) : "memory");
}

__device__ __forceinline__ void tma_load_2d(uint32_t dst, const CUtensorMap* map, uint64_t* bar, int x, int y) {
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4}], [%2];" ::"r"(dst),
      "l"(map), "r"(smem_u32(bar)), "r"(x), "r"(y)
      : "memory");
}
// Copy of a box into this CTA's shared memory whose completion is counted on
// the mbarrier at shared::cluster address `bar`, which may belong to the
// peer CTA of the pair (cta_group::2).
__device__ __forceinline__ void tma_load_2d_pair(uint32_t dst, const CUtensorMap* map, uint32_t bar, int x, int y) {
  asm volatile(
      "cp.async.bulk.tensor.2d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4}], "
      "[%2];" ::"r"(dst),
      "l"(map), "r"(bar), "r"(x), "r"(y)
      : "memory");
}
// shared::cluster address of this CTA's shared variable at `addr` in CTA `rank`
__device__ __forceinline__ uint32_t mapa(uint32_t addr, uint32_t rank) {
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
  return r;
}
__device__ __forceinline__ void mbar_arrive_cluster(uint32_t bar) {
  asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(bar) : "memory");
}
// Arrivals that order no memory accesses of the arriving thread.  A release
// arrival waits until the thread's earlier global stores are performed at its
// scope; the epilogue's accumulator hand-back follows tcgen05.wait::ld, which
// has already completed every TMEM read it covers, so it needs no release.
__device__ __forceinline__ void mbar_arrive_relaxed(uint64_t* bar) {
  asm volatile("mbarrier.arrive.relaxed.cta.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}
__device__ __forceinline__ void mbar_arrive_cluster_relaxed(uint32_t bar) {
  asm volatile("mbarrier.arrive.relaxed.cluster.shared::cluster.b64 _, [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ uint32_t cluster_rank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
__device__ __forceinline__ void cluster_sync() {
  asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}

__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

// Shared-memory matrix descriptor: start, leading / stride byte offsets,
// version 1 (bits 46-48), 128-byte swizzle (layout 2, bits 61-63).
__device__ __forceinline__ uint64_t smem_desc(uint32_t addr, uint32_t lbo, uint32_t sbo) {
  uint64_t d = (uint64_t)((addr >> 4) & 0x3FFFu);
  d |= (uint64_t)((lbo >> 4) & 0x3FFFu) << 16;
  d |= (uint64_t)((sbo >> 4) & 0x3FFFu) << 32;
  d |= (uint64_t)1 << 46;
  d |= (uint64_t)2 << 61;
  return d;
}

// Instruction descriptor of kind::f16: fp32 accumulate, bf16 A and B.
__device__ __forceinline__ uint32_t instr_desc(int m, int n, int a_mn, int b_mn) {
  return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)a_mn << 15) | ((uint32_t)b_mn << 16) |
         ((uint32_t)(n >> 3) << 17) | ((uint32_t)(m >> 4) << 24);
}

template <int kCta>
__device__ __forceinline__ void umma_bf16(uint32_t d_tmem, uint64_t a, uint64_t b, uint32_t idesc, uint32_t acc) {
  if constexpr (kCta == 2)
    asm volatile(
        "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(
            d_tmem),
        "l"(a), "l"(b), "r"(idesc), "r"(acc)
        : "memory");
  else
    asm volatile(
        "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(
            d_tmem),
        "l"(a), "l"(b), "r"(idesc), "r"(acc)
        : "memory");
}
// Arrive on `bar` once this thread's MMAs so far have completed; for a CTA
// pair on the mbarrier at `bar`'s offset in both CTAs.
template <int kCta>
__device__ __forceinline__ void umma_commit(uint64_t* bar) {
  if constexpr (kCta == 2)
    asm volatile(
        "tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;" ::"r"(
            smem_u32(bar)),
        "h"((uint16_t)3)
        : "memory");
  else
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_u32(bar))
                 : "memory");
}

__device__ __forceinline__ void tmem_ld32(uint32_t taddr, uint32_t (&v)[32]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
      "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
      : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]), "=r"(v[8]),
        "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15]), "=r"(v[16]),
        "=r"(v[17]), "=r"(v[18]), "=r"(v[19]), "=r"(v[20]), "=r"(v[21]), "=r"(v[22]), "=r"(v[23]), "=r"(v[24]),
        "=r"(v[25]), "=r"(v[26]), "=r"(v[27]), "=r"(v[28]), "=r"(v[29]), "=r"(v[30]), "=r"(v[31])
      : "r"(taddr));
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
}

__device__ __forceinline__ uint32_t pack_bf16x2(float a, float b) {
  __nv_bfloat162 t = __floats2bfloat162_rn(a, b);
  return *reinterpret_cast<uint32_t*>(&t);
}


}  // namespace
}  // namespace tp
