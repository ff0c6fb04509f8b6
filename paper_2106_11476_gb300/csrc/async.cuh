// Asynchronous bulk copies (TMA, cp.async.bulk) into shared memory, their
// mbarriers, and the bounded wait every kernel uses on them (sm_90 and
// later PTX; built for sm_103a).
//
// A wait never spins forever: it gives up after a time limit measured on the
// global nanosecond timer (and after a fixed number of polls, should that
// timer not advance), so a copy that never lands turns into an error status
// the host can read instead of a hung kernel.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

namespace fw2 {

// limit of one bounded wait on a copy of a few hundred KB
constexpr unsigned long long kWaitLimitNs = 2000000000ull;  // 2 s
constexpr int kStatusWaitTimeout = 1;

__device__ __forceinline__ unsigned smem_u32(const void *p) {
  return static_cast<unsigned>(__cvta_generic_to_shared(p));
}

__device__ __forceinline__ void mbar_init(uint64_t *bar, unsigned count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;\n" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}

// make initialised mbarriers visible to the async proxy (the copies)
__device__ __forceinline__ void fence_mbarrier_init() {
  asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
}

// one arrival that also announces `bytes` of transactions for the phase
__device__ __forceinline__ void mbar_arrive_expect_tx(uint64_t *bar, unsigned bytes) {
  asm volatile(
      "{\n"
      " .reg .b64 st;\n"
      " mbarrier.arrive.expect_tx.shared::cta.b64 st, [%0], %1;\n"
      "}\n" ::"r"(smem_u32(bar)),
      "r"(bytes)
      : "memory");
}

// one arrival (release)
__device__ __forceinline__ void mbar_arrive(uint64_t *bar) {
  asm volatile(
      "{\n"
      " .reg .b64 st;\n"
      " mbarrier.arrive.shared::cta.b64 st, [%0];\n"
      "}\n" ::"r"(smem_u32(bar))
      : "memory");
}

__device__ __forceinline__ bool mbar_try_wait(uint64_t *bar, unsigned parity) {
  unsigned ok;
  asm volatile(
      "{\n"
      " .reg .pred p;\n"
      " mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n"
      " selp.u32 %0, 1, 0, p;\n"
      "}\n"
      : "=r"(ok)
      : "r"(smem_u32(bar)), "r"(parity)
      : "memory");
  return ok != 0;
}

__device__ __forceinline__ unsigned long long global_ns() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;\n" : "=l"(t));
  return t;
}

// true when the phase of the given parity completed within limit_ns
__device__ __forceinline__ bool mbar_wait_bounded(uint64_t *bar, unsigned parity,
                                                  unsigned long long limit_ns = kWaitLimitNs) {
  if (mbar_try_wait(bar, parity)) return true;
  const unsigned long long t0 = global_ns();
  for (long long polls = 0; polls < (1ll << 34); polls += 64) {
    for (int i = 0; i < 64; ++i)
      if (mbar_try_wait(bar, parity)) return true;
    if (global_ns() - t0 > limit_ns) return false;
  }
  return false;
}

// order this thread's earlier shared-memory accesses (made visible to it by
// a barrier) before its later async-proxy copies into the same memory
__device__ __forceinline__ void fence_proxy_async_smem() {
  asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
}

// a tensor map in global memory (written by a host copy before the launch,
// possibly at an address an earlier table used): order that write before
// this thread's tensor copies through the map
__device__ __forceinline__ void fence_tensormap_acquire(const void *map) {
  asm volatile("fence.proxy.tensormap::generic.acquire.gpu [%0], 128;\n" ::"l"(map) : "memory");
}

// Tiled tensor copies global -> shared through a tensor map (a kernel
// parameter declared __grid_constant__): the box at element coordinates
// (x, y[, z]) lands densely in shared memory (128-byte aligned destination),
// x innermost; x * element size must be a multiple of 16 bytes.
__device__ __forceinline__ void tma_load_2d(void *dst, const void *tmap, int x, int y, uint64_t *bar) {
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];\n" ::"r"(
          smem_u32(dst)),
      "l"(tmap), "r"(x), "r"(y), "r"(smem_u32(bar))
      : "memory");
}
__device__ __forceinline__ void tma_load_3d(void *dst, const void *tmap, int x, int y, int z, uint64_t *bar) {
  asm volatile(
      "cp.async.bulk.tensor.3d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4}], [%5];\n" ::"r"(
          smem_u32(dst)),
      "l"(tmap), "r"(x), "r"(y), "r"(z), "r"(smem_u32(bar))
      : "memory");
}

__device__ __forceinline__ void tma_load_4d(void *dst, const void *tmap, int x, int y, int z, int w,
                                            uint64_t *bar) {
  asm volatile(
      "cp.async.bulk.tensor.4d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4, %5}], [%6];\n" ::"r"(
          smem_u32(dst)),
      "l"(tmap), "r"(x), "r"(y), "r"(z), "r"(w), "r"(smem_u32(bar))
      : "memory");
}

// Tiled tensor copies shared -> global (bulk async-group); the box lands at
// (x, y[, z[, w]]); cells outside the tensor are not written.
__device__ __forceinline__ void tma_store_2d(const void *tmap, int x, int y, const void *src) {
  asm volatile("cp.async.bulk.tensor.2d.global.shared::cta.bulk_group [%0, {%1, %2}], [%3];\n" ::"l"(tmap), "r"(x),
               "r"(y), "r"(smem_u32(src))
               : "memory");
}
__device__ __forceinline__ void tma_store_3d(const void *tmap, int x, int y, int z, const void *src) {
  asm volatile("cp.async.bulk.tensor.3d.global.shared::cta.bulk_group [%0, {%1, %2, %3}], [%4];\n" ::"l"(tmap),
               "r"(x), "r"(y), "r"(z), "r"(smem_u32(src))
               : "memory");
}
__device__ __forceinline__ void tma_store_4d(const void *tmap, int x, int y, int z, int w, const void *src) {
  asm volatile("cp.async.bulk.tensor.4d.global.shared::cta.bulk_group [%0, {%1, %2, %3, %4}], [%5];\n" ::"l"(tmap),
               "r"(x), "r"(y), "r"(z), "r"(w), "r"(smem_u32(src))
               : "memory");
}
__device__ __forceinline__ void bulk_commit() { asm volatile("cp.async.bulk.commit_group;\n" ::: "memory"); }
// wait until at most K committed store groups still read shared memory
template <int K>
__device__ __forceinline__ void bulk_wait_read() {
  asm volatile("cp.async.bulk.wait_group.read %0;\n" ::"n"(K) : "memory");
}
// wait until every committed store group has completed
__device__ __forceinline__ void bulk_wait_all() { asm volatile("cp.async.bulk.wait_group 0;\n" ::: "memory"); }

// prefetch a tensor box into L2 (no shared memory, no completion to wait for)
__device__ __forceinline__ void tma_prefetch_2d(const void *tmap, int x, int y) {
  asm volatile("cp.async.bulk.prefetch.tensor.2d.L2.global.tile [%0, {%1, %2}];\n" ::"l"(tmap), "r"(x), "r"(y)
               : "memory");
}
__device__ __forceinline__ void tma_prefetch_3d(const void *tmap, int x, int y, int z) {
  asm volatile("cp.async.bulk.prefetch.tensor.3d.L2.global.tile [%0, {%1, %2, %3}];\n" ::"l"(tmap), "r"(x), "r"(y),
               "r"(z)
               : "memory");
}

// per-thread 4-byte asynchronous copy (for rows only 4-byte aligned) and
// its group bookkeeping
__device__ __forceinline__ void cp_async4(void *dst, const void *src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4;\n" ::"r"(smem_u32(dst)), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
template <int K>
__device__ __forceinline__ void cp_async_wait() {
  asm volatile("cp.async.wait_group %0;\n" ::"n"(K) : "memory");
}

// order this thread's generic accesses against async-proxy copies of the same
// memory (global and shared), both ways: around a grid barrier, so that the
// copies after it see what other SMs' bulk stores wrote before it
__device__ __forceinline__ void fence_proxy_async_all() { asm volatile("fence.proxy.async;\n" ::: "memory"); }

// Status word of a context: not 0 after a bounded wait gave up.
__device__ __forceinline__ unsigned status_of(const unsigned int *status) {
  unsigned v = 0;
  if (status) asm volatile("ld.relaxed.gpu.global.u32 %0, [%1];\n" : "=r"(v) : "l"(status) : "memory");
  return v;
}

// Barrier over all blocks of a cooperative launch (thread 0 of each): a
// counter in global memory that every block adds 1 to per barrier.  It only
// grows, by the grid size per barrier, so a launch finds its start from the
// counter itself (this block has not arrived yet, so the counter cannot have
// passed the next multiple) and a captured launch can be replayed.  The wait
// is bounded like the copy waits, and ends early once another block has
// reported a wait that gave up.
struct GridBarrier {
  unsigned long long *count;
  unsigned long long target;
  __device__ __forceinline__ void init(unsigned long long *c) {
    count = c;
    target = 0;
    if (!c) return;
    unsigned long long v;
    asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];\n" : "=l"(v) : "l"(c) : "memory");
    target = v / gridDim.x * gridDim.x;
  }
  __device__ __forceinline__ void arrive() {
    target += gridDim.x;
    asm volatile("red.release.gpu.global.add.u64 [%0], %1;\n" ::"l"(count), "l"(1ull) : "memory");
  }
  __device__ __forceinline__ bool reached() const {
    unsigned long long v;
    asm volatile("ld.acquire.gpu.global.u64 %0, [%1];\n" : "=l"(v) : "l"(count) : "memory");
    return v >= target;
  }
  __device__ __forceinline__ bool wait(const unsigned int *status, unsigned long long limit_ns = kWaitLimitNs) {
    if (reached()) return true;
    const unsigned long long t0 = global_ns();
    for (long long polls = 0; polls < (1ll << 34); polls += 64) {
      for (int i = 0; i < 64; ++i)
        if (reached()) return true;
      if (status_of(status) != 0 || global_ns() - t0 > limit_ns) return false;
    }
    return false;
  }
};

__device__ __forceinline__ void report_status(unsigned int *status, unsigned bits) {
  if (status) atomicOr(status, bits);
}

}  // namespace fw2
