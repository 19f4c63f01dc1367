// tma.cuh -- thin inline-PTX wrappers for the Tensor Memory Accelerator (cp.async.bulk*)
// and shared-memory mbarriers, as used by the tiled FFT passes.
//
// Every wait is bounded: mbar_wait gives up after `limit` polls and returns false; the
// caller then records an error code in device memory that the host checks after each block
// of iterations, instead of spinning forever.
#pragma once
#include <cuda.h>
#include <cuda_runtime.h>
#include <cstdint>

namespace cbs {

constexpr unsigned kWaitLimit = 1u << 24;   // polls of try_wait (each may suspend briefly)
constexpr int kErrTmaTimeout = 1;
constexpr int kErrMisaligned = 2;

__device__ __forceinline__ uint32_t smem_u32(const void* p) {
  return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}

// Make barrier initialisation visible to the async proxy before the first TMA uses it.
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
      "selp.u32 %0, 1, 0, p;\n\t}\n"
      : "=r"(ok)
      : "r"(smem_u32(bar)), "r"(parity)
      : "memory");
  return ok != 0;
}

// Bounded wait for phase `parity` of an mbarrier; false on timeout.
__device__ __forceinline__ bool mbar_wait(uint64_t* bar, uint32_t parity, unsigned limit = kWaitLimit) {
  for (unsigned i = 0; i < limit; ++i)
    if (mbar_try_wait(bar, parity)) return true;
  return false;
}

// The same for a warp that works as one (all 32 lanes call it): the lanes' verdicts are joined, so
// that none goes on where another gives up.  A wait that is not over at once gives up where another
// warp has set *failed (STRICT: also one that is), and sets it (and *err) when it gives up.
template <bool STRICT = false>
__device__ __forceinline__ bool warp_wait(uint64_t* bar, uint32_t parity, volatile int* failed, int* err,
                                          unsigned limit) {
  bool ok = limit > 0 && mbar_try_wait(bar, parity);
  for (unsigned i = 1; i < limit && !ok && !*failed; ++i) ok = mbar_try_wait(bar, parity);
  ok = __all_sync(0xffffffffu, STRICT ? ok && !*failed : ok);
  if (!ok && (threadIdx.x & 31) == 0) {
    *failed = 1;
    atomicExch(err, kErrTmaTimeout);
  }
  return ok;
}

// The copies of tiles first, first + step, ... last of a ring of n sets (tile i in set i mod n) have
// landed, or the waits' limit is over: what a thread that issued them does before it may leave.
__device__ __forceinline__ void settle(uint64_t* full, int n, int first, int last, int step = 1) {
  for (int i = first; i <= last; i += step) mbar_wait(full + i % n, (uint32_t)((i / n) & 1));
}

// 5D tiled tensor load global -> shared (completion counted on `bar` in bytes) and store shared ->
// global (bulk async group; out-of-range elements skipped), for the y-blocked workspace: x, y in
// block, z, y block, component.
__device__ __forceinline__ void tma_load_5d(void* dst, const CUtensorMap* tm, int c0, int c1, int c2, int c3, int c4,
                                            uint64_t* bar) {
  asm volatile(
      "cp.async.bulk.tensor.5d.shared::cluster.global.tile.mbarrier::complete_tx::bytes"
      " [%0], [%1, {%2, %3, %4, %5, %6}], [%7];" ::"r"(smem_u32(dst)),
      "l"(reinterpret_cast<uint64_t>(tm)), "r"(c0), "r"(c1), "r"(c2), "r"(c3), "r"(c4), "r"(smem_u32(bar))
      : "memory");
}
__device__ __forceinline__ void tma_store_5d(const CUtensorMap* tm, int c0, int c1, int c2, int c3, int c4,
                                             const void* src) {
  asm volatile(
      "cp.async.bulk.tensor.5d.global.shared::cta.tile.bulk_group [%0, {%1, %2, %3, %4, %5}], [%6];" ::"l"(
          reinterpret_cast<uint64_t>(tm)),
      "r"(c0), "r"(c1), "r"(c2), "r"(c3), "r"(c4), "r"(smem_u32(src))
      : "memory");
}

// Contiguous bulk copy global -> shared (16-byte aligned addresses, size a multiple of 16).
__device__ __forceinline__ void bulk_load(void* dst, const void* src, uint32_t bytes, uint64_t* bar) {
  asm volatile(
      "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
          smem_u32(dst)),
      "l"(src), "r"(bytes), "r"(smem_u32(bar))
      : "memory");
}

// Contiguous bulk copy shared -> global (bulk async group).
__device__ __forceinline__ void bulk_store(void* dst, const void* src, uint32_t bytes) {
  asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], %2;" ::"l"(dst), "r"(smem_u32(src)),
               "r"(bytes)
               : "memory");
}

__device__ __forceinline__ void bulk_commit() { asm volatile("cp.async.bulk.commit_group;" ::: "memory"); }
__device__ __forceinline__ void bulk_wait_all() { asm volatile("cp.async.bulk.wait_group 0;" ::: "memory"); }
__device__ __forceinline__ void bulk_wait_read_all() {
  asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");
}
// All committed bulk groups but the newest one have finished reading their sources.
__device__ __forceinline__ void bulk_wait_read_1() {
  asm volatile("cp.async.bulk.wait_group.read 1;" ::: "memory");
}

// Order this thread's generic-proxy shared-memory writes before later async-proxy reads.
__device__ __forceinline__ void fence_async_smem() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }

// Programmatic dependent launch: let the next kernel of the stream take up processors as this
// one's blocks leave them, and wait for the kernel before (its writes are then visible).
__device__ __forceinline__ void launch_dependents() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void wait_for_previous() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// Block set-up of a pipelined tile kernel: thread 0 checks that the tile base is 128-byte
// aligned (as tensor copies require; the tile kernels declare no static shared memory, so the
// dynamic base is) and initialises the `nbar` mbarriers; a misaligned tile aborts the block
// uniformly.
__device__ __forceinline__ bool block_setup_n(const void* tile, uint64_t* bars, int nbar, int* fail, int* err) {
  if (threadIdx.x == 0) {
    *fail = (smem_u32(tile) & 127u) ? 1 : 0;
    if (*fail) atomicExch(err, kErrMisaligned);
    for (int i = 0; i < nbar; ++i) mbar_init(bars + i, 1);
    fence_mbar_init();
  }
  __syncthreads();
  return *fail == 0;
}

// Bounded wait for phase `parity` of a tile's copies, shared by the block: every thread
// polls; a timeout anywhere aborts the whole block (uniformly) and records an error.
__device__ __forceinline__ bool block_wait(uint64_t* bar, int* fail, int* err, uint32_t parity, unsigned limit) {
  if (!mbar_wait(bar, parity, limit)) *fail = 1;
  __syncthreads();
  if (*fail) {
    if (threadIdx.x == 0) atomicExch(err, kErrTmaTimeout);
    return false;
  }
  return true;
}

}  // namespace cbs
