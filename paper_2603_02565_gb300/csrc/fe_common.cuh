// Shared device helpers of the joint evaluator: split-bf16 values, mbarriers,
// TMA tile loads and tcgen05 (TMEM / UMMA) wrappers for sm_103a.
#pragma once

#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <cuda_runtime.h>
#include <stdint.h>
#include <type_traits>

#include "fe.h"
#include "fe_kernels.h"

namespace fe {

// A bounded wait gives up after this many microseconds of %globaltimer.
constexpr uint32_t kWaitLimitUs = 1000000;

// ---------------------------------------------------------------------------
// split bf16: x ~= hi + lo with hi = bf16(x), lo = bf16(x - hi)
// ---------------------------------------------------------------------------
__device__ __forceinline__ void split_bf16(float x, bf16& hi, bf16& lo) {
  hi = __float2bfloat16_rn(x);
  lo = __float2bfloat16_rn(x - __bfloat162float(hi));
}

// two floats -> packed hi pair and packed lo pair (x0 in the low half);
// the same round-to-nearest-even values as split_bf16, two lanes per cvt
// (x0 - h0, x1 - h1) in one instruction, h (-1) + x rounded once
__device__ __forceinline__ void sub2(float x0, float x1, float h0, float h1, float& r0, float& r1) {
  uint64_t r;
  asm("{\n\t.reg .b64 x, h, m;\n\tmov.b64 x, {%1, %2};\n\tmov.b64 h, {%3, %4};\n\tmov.b64 m, {%5, %5};\n\t"
      "fma.rn.f32x2 %0, h, m, x;\n\t}"
      : "=l"(r)
      : "f"(x0), "f"(x1), "f"(h0), "f"(h1), "f"(-1.f));
  asm("mov.b64 {%0, %1}, %2;" : "=f"(r0), "=f"(r1) : "l"(r));
}
__device__ __forceinline__ void split2(float x0, float x1, uint32_t& hi, uint32_t& lo) {
  __nv_bfloat162 h = __floats2bfloat162_rn(x0, x1);
  const uint32_t hu = *reinterpret_cast<uint32_t*>(&h);
  float r0, r1;
  sub2(x0, x1, __uint_as_float(hu << 16), __uint_as_float(hu & 0xFFFF0000u), r0, r1);
  __nv_bfloat162 l = __floats2bfloat162_rn(r0, r1);
  hi = hu;
  lo = *reinterpret_cast<uint32_t*>(&l);
}

// Split pair by truncation, for on-chip intermediates (softmax P, the FFN
// hidden activation): hi keeps the top 16 bits of x, r = x - hi is exact in
// fp32, lo keeps the top 16 bits of r, so |x - hi - lo| < 2^-14 |x|.  Byte
// permutes and one subtraction of a pair, no conversion instructions.
__device__ __forceinline__ void split2_trunc(float x0, float x1, uint32_t& hi, uint32_t& lo) {
  const uint32_t u0 = __float_as_uint(x0), u1 = __float_as_uint(x1);
  hi = __byte_perm(u0, u1, 0x7632);
  float r0, r1;
  sub2(x0, x1, __uint_as_float(u0 & 0xFFFF0000u), __uint_as_float(u1 & 0xFFFF0000u), r0, r1);
  lo = __byte_perm(__float_as_uint(r0), __float_as_uint(r1), 0x7632);
}

__device__ __forceinline__ float bf16lo_f(uint32_t v) { return __uint_as_float(v << 16); }
__device__ __forceinline__ float bf16hi_f(uint32_t v) { return __uint_as_float(v & 0xFFFF0000u); }

__device__ __forceinline__ uint64_t globaltimer_ns() {
  uint64_t t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

// Programmatic dependent launch.  pdl_wait: block until every earlier kernel
// of the stream has completed and its memory is visible (every batch kernel
// calls it before touching global memory, and before any early exit).
// pdl_trigger: let the next kernel of the stream start launching now.
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void pdl_trigger() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

__device__ __forceinline__ uint32_t smem_u32(const void* p) {
  return (uint32_t)__cvta_generic_to_shared(p);
}

// ---------------------------------------------------------------------------
// mbarrier
// ---------------------------------------------------------------------------
__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}

__device__ __forceinline__ void fence_mbar_init() {
  asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}

__device__ __forceinline__ void mbar_arrive_expect_tx(uint64_t* bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes)
               : "memory");
}

__device__ __forceinline__ bool mbar_try_wait(uint64_t* bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(smem_u32(bar)), "r"(parity)
      : "memory");
  return ok != 0;
}

// ---------------------------------------------------------------------------
// Whole-warp issue and bounded waits.  A role that only one thread performs
// (tcgen05.mma, its commits, TMA) is run by its whole warp in step: every lane
// keeps the loop state and polls the barriers, and the instructions themselves
// are predicated on the lane that elect.sync picks (always the same one).  The
// control flow stays uniform for the compiler; behind `if (lane == 0)` two
// satisfied waits, two MMAs of N = 64 and a commit took 475 cycles of the issuing
// thread, this form 126 to 180 (eight MMAs and one wait: 739 and 385, the tensor
// pipe's own time).  The predicate has to be elect.sync's own result: combined
// with a flag of the lane it costs as much as the branch (batch of 256 requests
// 142.6 -> 168.0 us).
//
// Every wait is bounded: it gives up when its limit has passed or another thread of
// the batch has set ST_TIMEOUT (looked up every eighth poll; a poll takes up to
// 4 us).  The results of the batch are invalid then, and nothing may fault, hang
// or outlive its block.  What could fault is a load's arrival on a barrier whose
// previous load is still on its way: one too many for it.  (Arrivals on a barrier
// without bytes cannot be too many.)  Two forms rule that out:
//  * GEMM, context, embedding and d <= 128 FFN kernels: a warp does nothing more that
//    others wait for.  A role warp leaves its loop (mbar_wait_ok).  An epilogue
//    warp, whose partners meet it at named barriers, walks on to the end of its loop;
//    a lane of it that has given up (go = 0) skips its waits, arrives no more and
//    loads no more (mbar_wait_warp).
//  * Attention, d = 256 FFN and sequence kernels: every role walks on, some 30 us a
//    wait, on addresses that stay in bounds, and in front of each load waits for the
//    previous one's bytes on that barrier, too (mbar_wait_load).  With a vote and an
//    exit in their loops the d = 256 FFN was 2 to 3 % slower, the attention up to 6 %.
// At its end each role waits for the copies and products that it has issued
// (mbar_landed, umma_drain).
// A wait ends with the warp converged: an issuing lane that ran ahead could
// advance a barrier by two phases under a lane still polling it.
// ---------------------------------------------------------------------------
__device__ __forceinline__ uint32_t elect_one() {
  uint32_t e;
  asm volatile("{\n\t.reg .pred p;\n\telect.sync _|p, 0xffffffff;\n\tselp.u32 %0, 1, 0, p;\n\t}" : "=r"(e));
  return e;
}
// State of an epilogue warp's lane: 1 for lane 0, which arrives for the warp, 2 for
// the others, 0 after a wait of this lane has given up.
__device__ __forceinline__ uint32_t lane0_go() { return (threadIdx.x & 31) == 0 ? 1u : 2u; }

__device__ __forceinline__ bool mbar_try_wait_at(uint32_t bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(bar), "r"(parity)
      : "memory");
  return ok != 0;
}

// The polling loop, out of line: false when it gives up.
static __device__ __noinline__ bool mbar_wait_slow(uint64_t* bar, uint32_t parity, int* status, uint32_t limit_us) {
  const uint64_t t0 = globaltimer_ns();
  for (uint32_t it = 1;; ++it) {
    if (mbar_try_wait(bar, parity)) return true;
    if ((it & 7u) == 0u && (*reinterpret_cast<volatile int*>(status) & ST_TIMEOUT)) return false;
    if (globaltimer_ns() - t0 > (uint64_t)limit_us * 1000u) {
      atomicOr(status, ST_TIMEOUT);
      return false;
    }
  }
}
// The wait of a warp that walks on.  Its loop is out of line: these kernels run much of their code
// once per launch, so its size shows (the loop in line at every wait made a batch
// of 256 requests 4 % slower).
__device__ __forceinline__ void mbar_wait_role(uint64_t* bar, uint32_t parity, int* status,
                                               uint32_t limit_us = kWaitLimitUs) {
  if (!mbar_try_wait(bar, parity)) mbar_wait_slow(bar, parity, status, limit_us);
  __syncwarp();
}
// The same by shared-memory address and in line, where a call would spill the
// values live across it.  The limit counts in 65.5 us (the timer's upper bits).
__device__ __forceinline__ void mbar_wait_at(uint32_t bar, uint32_t parity, int* status,
                                             uint32_t limit_us = kWaitLimitUs) {
  if (!mbar_try_wait_at(bar, parity)) {
    const uint32_t t0 = (uint32_t)(globaltimer_ns() >> 16);
    for (uint32_t it = 1; !mbar_try_wait_at(bar, parity); ++it) {
      if ((it & 7u) == 0u && (*reinterpret_cast<volatile int*>(status) & ST_TIMEOUT)) break;
      if ((uint32_t)(globaltimer_ns() >> 16) - t0 > (uint32_t)((uint64_t)limit_us * 1000u >> 16)) {
        atomicOr(status, ST_TIMEOUT);
        break;
      }
    }
  }
  __syncwarp();
}
// Whether a phase is complete, without the time that try_wait spends in an incomplete phase
__device__ __forceinline__ bool mbar_test_wait(uint64_t* bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(smem_u32(bar)), "r"(parity)
      : "memory");
  return ok != 0;
}
// The wait of a warp that leaves its loop: false, in every lane, if one has given up.
__device__ __forceinline__ bool mbar_wait_ok(uint64_t* bar, uint32_t parity, int* status,
                                             uint32_t limit_us = kWaitLimitUs) {
  if (__all_sync(0xffffffffu, mbar_try_wait(bar, parity))) return true;
  return __all_sync(0xffffffffu, mbar_wait_slow(bar, parity, status, limit_us));
}
// The wait for bytes or products on their way, which need nobody else's progress:
// whatever the status says.
static __device__ __noinline__ void mbar_landed_slow(uint64_t* bar, uint32_t parity, int* status, uint32_t limit_us) {
  const uint64_t t0 = globaltimer_ns();
  while (!mbar_try_wait(bar, parity)) {
    if (globaltimer_ns() - t0 > (uint64_t)limit_us * 1000u) {
      atomicOr(status, ST_TIMEOUT);
      break;
    }
  }
}
__device__ __forceinline__ void mbar_landed(uint64_t* bar, uint32_t parity, int* status,
                                            uint32_t limit_us = kWaitLimitUs) {
  if (!mbar_try_wait(bar, parity)) mbar_landed_slow(bar, parity, status, limit_us);
  __syncwarp();
}
// (in line, as mbar_wait_at)
__device__ __forceinline__ void mbar_landed_at(uint32_t bar, uint32_t parity, int* status,
                                               uint32_t limit_us = kWaitLimitUs) {
  if (!mbar_try_wait_at(bar, parity)) {
    const uint32_t t0 = (uint32_t)(globaltimer_ns() >> 16);
    while (!mbar_try_wait_at(bar, parity)) {
      if ((uint32_t)(globaltimer_ns() >> 16) - t0 > (uint32_t)((uint64_t)limit_us * 1000u >> 16)) {
        atomicOr(status, ST_TIMEOUT);
        break;
      }
    }
  }
  __syncwarp();
}
// The newest load on each of a ring's S barriers, the next load going to number `slot`
// with the parity `par` of its wait.
__device__ __forceinline__ void mbar_landed_ring(uint64_t* full, int slot, uint32_t par, int S, int* status) {
#pragma unroll 1
  for (int i = 0; i < S; ++i) mbar_landed(full + i, i < slot ? par ^ 1u : par, status);
}
// The wait before the next load on barrier `full`: its previous load has landed (asked
// first, off the path from the freed memory to its next load) and its memory is free.
__device__ __forceinline__ void mbar_wait_load(uint64_t* empty, uint64_t* full, uint32_t parity, int* status) {
  if (!mbar_try_wait(full, parity)) mbar_landed_slow(full, parity, status, kWaitLimitUs);
  if (!mbar_try_wait(empty, parity)) mbar_wait_slow(empty, parity, status, kWaitLimitUs);
  __syncwarp();
}
// An epilogue warp's wait (its loop in a function of its own, and `go` not asked in
// front of the first poll: either made the d = 256 FFN 2 % slower).
static __device__ __noinline__ uint32_t mbar_wait_slow_go(uint64_t* bar, uint32_t parity, int* status,
                                                          uint32_t limit_us, uint32_t go) {
  if (go == 0) return 0;
  const uint64_t t0 = globaltimer_ns();
  for (uint32_t it = 1;; ++it) {
    if (mbar_try_wait(bar, parity)) return go;
    if ((it & 7u) == 0u && (*reinterpret_cast<volatile int*>(status) & ST_TIMEOUT)) return 0;
    if (globaltimer_ns() - t0 > (uint64_t)limit_us * 1000u) {
      atomicOr(status, ST_TIMEOUT);
      return 0;
    }
  }
}
__device__ __forceinline__ void mbar_wait_warp(uint64_t* bar, uint32_t parity, int* status, uint32_t& go,
                                               uint32_t limit_us = kWaitLimitUs) {
  if (!mbar_try_wait(bar, parity)) go = mbar_wait_slow_go(bar, parity, status, limit_us, go);
  __syncwarp();
}
// The same with cluster-scope acquire (peers' stores into this CTA).
__device__ __forceinline__ bool mbar_try_wait_cluster(uint64_t* bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(smem_u32(bar)), "r"(parity)
      : "memory");
  return ok != 0;
}
static __device__ __noinline__ bool mbar_wait_cluster_slow(uint64_t* bar, uint32_t parity, int* status,
                                                           uint32_t limit_us) {
  const uint64_t t0 = globaltimer_ns();
  for (uint32_t it = 1;; ++it) {
    if (mbar_try_wait_cluster(bar, parity)) return true;
    if ((it & 7u) == 0u && (*reinterpret_cast<volatile int*>(status) & ST_TIMEOUT)) return false;
    if (globaltimer_ns() - t0 > (uint64_t)limit_us * 1000u) {
      atomicOr(status, ST_TIMEOUT);
      return false;
    }
  }
}
__device__ __forceinline__ void mbar_wait_cluster(uint64_t* bar, uint32_t parity, int* status, uint32_t& go,
                                                  uint32_t limit_us = kWaitLimitUs) {
  if (go != 0 && !mbar_wait_cluster_slow(bar, parity, status, limit_us)) go = 0;
  __syncwarp();
}

__device__ __forceinline__ void mbar_arrive_if_at(uint32_t bar, bool on) {
  asm volatile(
      "{\n\t.reg .pred q;\n\tsetp.ne.b32 q, %1, 0;\n\t"
      "@q mbarrier.arrive.shared::cta.b64 _, [%0];\n\t}" ::"r"(bar),
      "r"((uint32_t)on)
      : "memory");
}
// An epilogue warp's arrival: its lanes' earlier (fenced) writes come before it.
__device__ __forceinline__ void mbar_arrive_warp(uint64_t* bar, uint32_t go) {
  __syncwarp();
  mbar_arrive_if_at(smem_u32(bar), go == 1);
}

__device__ __forceinline__ void mbar_arrive_expect_tx_if(uint64_t* bar, uint32_t bytes, uint32_t go) {
  asm volatile(
      "{\n\t.reg .pred q;\n\tsetp.ne.b32 q, %2, 0;\n\t"
      "@q mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;\n\t}" ::"r"(smem_u32(bar)),
      "r"(bytes), "r"(go)
      : "memory");
}

// ---------------------------------------------------------------------------
// TMA: 2D tiled bulk tensor load global -> shared, completion on an mbarrier
// ---------------------------------------------------------------------------
__device__ __forceinline__ void tma_load_2d_if(void* smem_dst, const CUtensorMap* map, int x, int y, uint64_t* bar,
                                               uint32_t go) {
  asm volatile(
      "{\n\t.reg .pred q;\n\tsetp.ne.b32 q, %5, 0;\n\t"
      "@q cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes"
      " [%0], [%1, {%3, %4}], [%2];\n\t}" ::"r"(smem_u32(smem_dst)),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(smem_u32(bar)), "r"(x), "r"(y), "r"(go)
      : "memory");
}

__device__ __forceinline__ void tma_load_3d_if(void* smem_dst, const CUtensorMap* map, int x, int y, int z,
                                               uint64_t* bar, uint32_t go) {
  asm volatile(
      "{\n\t.reg .pred q;\n\tsetp.ne.b32 q, %6, 0;\n\t"
      "@q cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes"
      " [%0], [%1, {%3, %4, %5}], [%2];\n\t}" ::"r"(smem_u32(smem_dst)),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(smem_u32(bar)), "r"(x), "r"(y), "r"(z), "r"(go)
      : "memory");
}

__device__ __forceinline__ void tma_load_2d(void* smem_dst, const CUtensorMap* map, int x, int y,
                                            uint64_t* bar) {
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes"
      " [%0], [%1, {%3, %4}], [%2];" ::"r"(smem_u32(smem_dst)),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(smem_u32(bar)), "r"(x), "r"(y)
      : "memory");
}

// TMA: 3D tiled bulk tensor store shared -> global (bulk-group completion)
__device__ __forceinline__ void tma_store_3d(const CUtensorMap* map, const void* smem_src, int x, int y, int z) {
  asm volatile("cp.async.bulk.tensor.3d.global.shared::cta.bulk_group [%0, {%2, %3, %4}], [%1];" ::"l"(
                   reinterpret_cast<uint64_t>(map)),
               "r"(smem_u32(smem_src)), "r"(x), "r"(y), "r"(z)
               : "memory");
}

// TMA: 2D tiled bulk tensor store shared -> global (bulk-group completion)
__device__ __forceinline__ void tma_store_2d(const CUtensorMap* map, const void* smem_src, int x, int y) {
  asm volatile("cp.async.bulk.tensor.2d.global.shared::cta.bulk_group [%0, {%2, %3}], [%1];" ::"l"(
                   reinterpret_cast<uint64_t>(map)),
               "r"(smem_u32(smem_src)), "r"(x), "r"(y)
               : "memory");
}
__device__ __forceinline__ void bulk_commit() { asm volatile("cp.async.bulk.commit_group;" ::: "memory"); }
// wait until no bulk group of this thread still reads shared memory
__device__ __forceinline__ void bulk_wait_read0() { asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory"); }
// wait until every bulk group of this thread has completed
__device__ __forceinline__ void bulk_wait0() { asm volatile("cp.async.bulk.wait_group 0;" ::: "memory"); }
// make this thread's generic-proxy shared-memory writes visible to the async proxy (TMA)
__device__ __forceinline__ void fence_async_shared() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }

__device__ __forceinline__ void prefetch_tmap(const CUtensorMap* map) {
  asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(map)) : "memory");
}

// ---------------------------------------------------------------------------
// tcgen05
// ---------------------------------------------------------------------------
__device__ __forceinline__ void tmem_alloc(uint32_t* slot_smem, uint32_t ncols) {
  asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(slot_smem)),
               "r"(ncols)
               : "memory");
  asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}

__device__ __forceinline__ void tmem_dealloc(uint32_t taddr, uint32_t ncols) {
  asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ncols) : "memory");
}

__device__ __forceinline__ void tc_fence_before() {
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
}
__device__ __forceinline__ void tc_fence_after() {
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
}

// Shared-memory matrix descriptor of a K-major operand tile stored with the
// 128-byte swizzle: rows of 64 bf16 (128 B), 8-row groups 1024 B apart.
__device__ __forceinline__ uint64_t umma_desc_sw128(uint32_t saddr) {
  uint64_t d = 0;
  d |= (uint64_t)((saddr & 0x3FFFFu) >> 4);  // start address
  d |= (uint64_t)1 << 16;                    // leading byte offset (unused for swizzled K-major)
  d |= (uint64_t)(1024 >> 4) << 32;          // stride byte offset: 8 rows x 128 B
  d |= (uint64_t)1 << 46;                    // descriptor version for tcgen05
  d |= (uint64_t)2 << 61;                    // swizzle mode: 128 B
  return d;
}

// A descriptor advanced by `bytes` (a multiple of 16) inside the same tile:
// the start-address field counts 16-byte units and never carries here.
__device__ __forceinline__ uint64_t desc_adv(uint64_t desc, uint32_t bytes) { return desc + (uint64_t)(bytes >> 4); }

// Instruction descriptor: kind::f16, A = B = bf16, D = f32, both K-major.
__device__ __forceinline__ uint32_t umma_idesc_bf16(int M, int N) {
  return (1u << 4)                       // D format f32
         | (1u << 7)                     // A format bf16
         | (1u << 10)                    // B format bf16
         | ((uint32_t)(N >> 3) << 17)    // N / 8
         | ((uint32_t)(M >> 4) << 24);   // M / 16
}

// Instruction descriptor: kind::f16, A = B = f16, D = f32, both K-major.
__device__ __forceinline__ uint32_t umma_idesc_f16(int M, int N) {
  return (1u << 4)                       // D format f32 (A, B formats 0: f16)
         | ((uint32_t)(N >> 3) << 17)    // N / 8
         | ((uint32_t)(M >> 4) << 24);   // M / 16
}

// Two floats as an f16x2 word (x0 in the low half), round to nearest.
__device__ __forceinline__ uint32_t pack_f16x2(float x0, float x1) {
  __half2 h = __floats2half2_rn(x0, x1);
  return *reinterpret_cast<uint32_t*>(&h);
}

__device__ __forceinline__ void umma_bf16(uint32_t tmem_d, uint64_t adesc, uint64_t bdesc, uint32_t idesc,
                                          uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(tmem_d),
      "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate)
      : "memory");
}

// Arrive on an mbarrier once every tcgen05.mma issued so far by this thread completes.
__device__ __forceinline__ void umma_commit(uint64_t* bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
                   smem_u32(bar))
               : "memory");
}

// The same three for whole-warp issue: predicated on go, the elected lane's flag.
__device__ __forceinline__ void umma_bf16_if(uint32_t tmem_d, uint64_t adesc, uint64_t bdesc, uint32_t idesc,
                                             uint32_t accumulate, uint32_t go) {
  asm volatile(
      "{\n\t.reg .pred p, q;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "setp.ne.b32 q, %5, 0;\n\t"
      "@q tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(tmem_d),
      "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate), "r"(go)
      : "memory");
}

__device__ __forceinline__ void umma_bf16_tmem_a_if(uint32_t tmem_d, uint32_t tmem_a, uint64_t bdesc, uint32_t idesc,
                                                    uint32_t accumulate, uint32_t go) {
  asm volatile(
      "{\n\t.reg .pred p, q;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "setp.ne.b32 q, %5, 0;\n\t"
      "@q tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n\t}" ::"r"(tmem_d),
      "r"(tmem_a), "l"(bdesc), "r"(idesc), "r"(accumulate), "r"(go)
      : "memory");
}

__device__ __forceinline__ void umma_commit_if(uint64_t* bar, uint32_t go) {
  asm volatile(
      "{\n\t.reg .pred q;\n\tsetp.ne.b32 q, %1, 0;\n\t"
      "@q tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n\t}" ::"r"(smem_u32(bar)),
      "r"(go)
      : "memory");
}

// Every product that this warp has issued is complete before the block frees its
// TMEM.  drain: a barrier of count 1 that nothing else uses.
__device__ __forceinline__ void umma_drain(uint64_t* drain, int* status, uint32_t go) {
  umma_commit_if(drain, go);
  mbar_landed(drain, 0u, status);
}

// 32 lanes x 32 columns of 32-bit TMEM -> 32 registers per thread (row = lane).
__device__ __forceinline__ void tmem_ld32(uint32_t taddr, float* v) {
  uint32_t r[32];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
      "{%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,"
      "%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
        "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]),
        "=r"(r[15]), "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]),
        "=r"(r[22]), "=r"(r[23]), "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]),
        "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
      : "r"(taddr));
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
  for (int i = 0; i < 32; ++i) v[i] = __uint_as_float(r[i]);
}

// 32 bytes per thread, for a row per lane: each load takes a whole sector.  (16-byte
// loads take every sector in two halves, and between them a line per lane of the
// L1 that a kernel with 200 KB of shared memory leaves.)
__device__ __forceinline__ void ld_sector(const float* p, float* x) {
  asm volatile("ld.global.L1::no_allocate.v8.f32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
               : "=f"(x[0]), "=f"(x[1]), "=f"(x[2]), "=f"(x[3]), "=f"(x[4]), "=f"(x[5]), "=f"(x[6]), "=f"(x[7])
               : "l"(p)
               : "memory");
}

// the same for stores (32-byte aligned)
__device__ __forceinline__ void st_sector(float* p, const float* x) {
  asm volatile("st.global.v8.f32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8};" ::"l"(p), "f"(x[0]), "f"(x[1]), "f"(x[2]), "f"(x[3]),
               "f"(x[4]), "f"(x[5]), "f"(x[6]), "f"(x[7])
               : "memory");
}

// 32 lanes x 64 columns -> 64 registers per thread, one load and one wait
__device__ __forceinline__ void tmem_ld64(uint32_t taddr, float* v) {
  uint32_t r[64];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x64.b32 "
      "{%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,"
      "%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31,"
      "%32,%33,%34,%35,%36,%37,%38,%39,%40,%41,%42,%43,%44,%45,%46,%47,"
      "%48,%49,%50,%51,%52,%53,%54,%55,%56,%57,%58,%59,%60,%61,%62,%63}, [%64];\n\t"
      "tcgen05.wait::ld.sync.aligned;"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
        "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]),
        "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]),
        "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31]),
        "=r"(r[32]), "=r"(r[33]), "=r"(r[34]), "=r"(r[35]), "=r"(r[36]), "=r"(r[37]), "=r"(r[38]), "=r"(r[39]),
        "=r"(r[40]), "=r"(r[41]), "=r"(r[42]), "=r"(r[43]), "=r"(r[44]), "=r"(r[45]), "=r"(r[46]), "=r"(r[47]),
        "=r"(r[48]), "=r"(r[49]), "=r"(r[50]), "=r"(r[51]), "=r"(r[52]), "=r"(r[53]), "=r"(r[54]), "=r"(r[55]),
        "=r"(r[56]), "=r"(r[57]), "=r"(r[58]), "=r"(r[59]), "=r"(r[60]), "=r"(r[61]), "=r"(r[62]), "=r"(r[63])
      : "r"(taddr)
      : "memory");
#pragma unroll
  for (int i = 0; i < 64; ++i) v[i] = __uint_as_float(r[i]);
}

// 32 lanes x 8 columns -> 8 registers per thread, and back (completes at tmem_st_wait())
__device__ __forceinline__ void tmem_ld8(uint32_t taddr, uint32_t* r) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];\n\t"
      "tcgen05.wait::ld.sync.aligned;"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
      : "r"(taddr)
      : "memory");
}
__device__ __forceinline__ void tmem_st8_nowait(uint32_t taddr, const uint32_t* r) {
  asm volatile("tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8};" ::"r"(taddr), "r"(r[0]),
               "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7])
               : "memory");
}

// 32 lanes x 16 columns -> 16 registers per thread
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, float* v) {
  uint32_t r[16];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 "
      "{%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];\n\t"
      "tcgen05.wait::ld.sync.aligned;"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
        "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
      : "r"(taddr)
      : "memory");
#pragma unroll
  for (int i = 0; i < 16; ++i) v[i] = __uint_as_float(r[i]);
}

// Two fp32 values in one 64-bit register: one instruction for both, each rounded as its scalar form.
__device__ __forceinline__ uint64_t f32x2_pack(float a, float b) {
  uint64_t r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
  return r;
}
__device__ __forceinline__ void f32x2_unpack(uint64_t v, float& a, float& b) {
  asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(v));
}
__device__ __forceinline__ uint64_t f32x2_fma(uint64_t a, uint64_t b, uint64_t c) {
  uint64_t r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
  return r;
}
__device__ __forceinline__ uint64_t f32x2_add(uint64_t a, uint64_t b) {
  uint64_t r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ uint64_t f32x2_mul(uint64_t a, uint64_t b) {
  uint64_t r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}

// LayerNorm passes over N values of a row, two values per instruction: sums in four
// interleaved chains (chain j % 4, two to a register pair), with the results of the
// scalar forms.  The epilogues that use them, and the split pairs' sub2, are bound by the
// instructions they issue and fetch: with them 256 requests took 1.8 % less in all, the
// largest batch 0.4 %.
struct RowSum {
  uint64_t s01 = 0, s23 = 0;  // (0.f, 0.f)
  __device__ __forceinline__ float total() const {
    float a, b, c, d;
    f32x2_unpack(s01, a, b);
    f32x2_unpack(s23, c, d);
    return (a + b) + (c + d);
  }
};
template <int N>
__device__ __forceinline__ void row_add(RowSum& s, const float* v) {  // s += v
#pragma unroll
  for (int j = 0; j < N; j += 4) {
    s.s01 = f32x2_add(s.s01, f32x2_pack(v[j], v[j + 1]));
    s.s23 = f32x2_add(s.s23, f32x2_pack(v[j + 2], v[j + 3]));
  }
}
template <int N>
__device__ __forceinline__ void row_add_sq(RowSum& s, const float* v, float mean) {  // s += (v - mean)^2
  const uint64_t nm = f32x2_pack(-mean, -mean);
#pragma unroll
  for (int j = 0; j < N; j += 4) {
    const uint64_t d0 = f32x2_add(f32x2_pack(v[j], v[j + 1]), nm), d1 = f32x2_add(f32x2_pack(v[j + 2], v[j + 3]), nm);
    s.s01 = f32x2_fma(d0, d0, s.s01);
    s.s23 = f32x2_fma(d1, d1, s.s23);
  }
}
template <int N>
__device__ __forceinline__ void row_norm(float* v, float mean, float rstd) {  // v = (v - mean) rstd
  const uint64_t nm = f32x2_pack(-mean, -mean), rr = f32x2_pack(rstd, rstd);
#pragma unroll
  for (int j = 0; j < N; j += 2)
    f32x2_unpack(f32x2_mul(f32x2_add(f32x2_pack(v[j], v[j + 1]), nm), rr), v[j], v[j + 1]);
}
template <int N>
__device__ __forceinline__ void row_plus(float* v, const float* w) {  // v += w
#pragma unroll
  for (int j = 0; j < N; j += 2)
    f32x2_unpack(f32x2_add(f32x2_pack(v[j], v[j + 1]), f32x2_pack(w[j], w[j + 1])), v[j], v[j + 1]);
}

// 2^x with the hardware approximation (ex2.approx.ftz.f32)
__device__ __forceinline__ float ex2_approx(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

__device__ __forceinline__ void tmem_st32(uint32_t taddr, const float* v) {
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x32.b32 [%0], "
      "{%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16,"
      "%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31,%32};" ::"r"(taddr),
      "r"(__float_as_uint(v[0])), "r"(__float_as_uint(v[1])), "r"(__float_as_uint(v[2])),
      "r"(__float_as_uint(v[3])), "r"(__float_as_uint(v[4])), "r"(__float_as_uint(v[5])),
      "r"(__float_as_uint(v[6])), "r"(__float_as_uint(v[7])), "r"(__float_as_uint(v[8])),
      "r"(__float_as_uint(v[9])), "r"(__float_as_uint(v[10])), "r"(__float_as_uint(v[11])),
      "r"(__float_as_uint(v[12])), "r"(__float_as_uint(v[13])), "r"(__float_as_uint(v[14])),
      "r"(__float_as_uint(v[15])), "r"(__float_as_uint(v[16])), "r"(__float_as_uint(v[17])),
      "r"(__float_as_uint(v[18])), "r"(__float_as_uint(v[19])), "r"(__float_as_uint(v[20])),
      "r"(__float_as_uint(v[21])), "r"(__float_as_uint(v[22])), "r"(__float_as_uint(v[23])),
      "r"(__float_as_uint(v[24])), "r"(__float_as_uint(v[25])), "r"(__float_as_uint(v[26])),
      "r"(__float_as_uint(v[27])), "r"(__float_as_uint(v[28])), "r"(__float_as_uint(v[29])),
      "r"(__float_as_uint(v[30])), "r"(__float_as_uint(v[31]))
      : "memory");
  asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
}

// 32 lanes x 16 columns from 16 registers per thread; completes at tmem_st_wait()
__device__ __forceinline__ void tmem_st16_nowait(uint32_t taddr, const uint32_t* r) {
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], "
      "{%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16};" ::"r"(taddr),
      "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]), "r"(r[8]),
      "r"(r[9]), "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15])
      : "memory");
}

__device__ __forceinline__ void tmem_st16_nowait(uint32_t taddr, const float* v) {
  uint32_t r[16];
#pragma unroll
  for (int i = 0; i < 16; ++i) r[i] = __float_as_uint(v[i]);
  tmem_st16_nowait(taddr, r);
}

__device__ __forceinline__ void tmem_st_wait() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }

}  // namespace fe
