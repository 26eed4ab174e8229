// Device and launch helpers shared by the kernel translation units: bulk
// (TMA) copies completed on mbarriers with bounded waits, programmatic
// dependent launch, and kernel shared memory limits.
#pragma once

#include <cuda_runtime.h>

#include <cstdint>
#include <map>
#include <mutex>
#include <utility>

#include "tx_internal.h"

namespace {

using namespace tx;

__device__ __forceinline__ uint32_t smem_addr(const void* p) {
  return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

__device__ __forceinline__ void cp_async16(void* smem, const void* gmem) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_addr(smem)), "l"(gmem));
}
__device__ __forceinline__ void cp_async4(void* smem, const void* gmem) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(smem_addr(smem)), "l"(gmem));
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;"); }

// Bulk (TMA) copies into shared memory, completed on an mbarrier: the
// issuing side announces the byte count (expect_tx, one arrival) and each
// copy completes its bytes on the barrier; waiting threads poll the phase.
__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count) {
  asm volatile("mbarrier.init.shared.b64 [%0], %1;" ::"r"(smem_addr(bar)), "r"(count) : "memory");
}
__device__ __forceinline__ void fence_mbar_init() { asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory"); }
// orders this CTA's earlier generic-proxy accesses of shared memory before later bulk copies into it
__device__ __forceinline__ void fence_proxy_async() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }
__device__ __forceinline__ void mbar_expect_tx(uint64_t* bar, uint32_t bytes) {
  asm volatile("{\n\t.reg .b64 st;\n\tmbarrier.arrive.expect_tx.shared.b64 st, [%0], %1;\n\t}"
               ::"r"(smem_addr(bar)), "r"(bytes) : "memory");
}
// announces `bytes` without arriving
__device__ __forceinline__ void mbar_expect_only(uint64_t* bar, uint32_t bytes) {
  asm volatile("mbarrier.expect_tx.relaxed.cta.shared::cta.b64 [%0], %1;" ::"r"(smem_addr(bar)), "r"(bytes) : "memory");
}
// global -> shared, `bytes` a multiple of 16, both addresses 16-byte aligned
__device__ __forceinline__ void bulk_g2s(void* dst, const void* src, uint32_t bytes, uint64_t* bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
               ::"r"(smem_addr(dst)), "l"(src), "r"(bytes), "r"(smem_addr(bar)) : "memory");
}
// waits for phase `parity` of bar to complete, giving up after max_iter polls
__device__ __forceinline__ bool mbar_wait(uint64_t* bar, uint32_t parity, uint32_t max_iter) {
  for (uint32_t i = 0; i < max_iter; ++i) {
    uint32_t done;
    asm volatile(
        "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(done)
        : "r"(smem_addr(bar)), "r"(parity)
        : "memory");
    if (done) return true;
  }
  return false;
}
constexpr uint32_t kMbarPolls = kWaitPolls;   // the full limit

// Waits that gave up (a copy that never completed) in this translation
// unit's kernels; a kernel that saw one returns early and its results are not
// valid. Read by tx_wait_timeouts.
__device__ int g_tx_wait_timeouts = 0;
// Records a wait that gave up: in the counter above and in the beam's own
// count, which marks the beam's state (tail, running statistics) and every
// later result as not valid until the beam is reset or imported.
template <typename A>
__device__ __forceinline__ void record_give_up(const A& a) {
  atomicAdd(&g_tx_wait_timeouts, 1);
  if (a.run) atomicAdd(reinterpret_cast<int32_t*>(a.run + 2 * (size_t)a.ndm), 1);
}
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_group 0;" ::: "memory"); }

// Programmatic dependent launch: a kernel launched with programmatic stream
// serialization may start while the kernel before it in the stream is still
// finishing. Each kernel of the path waits (pdl_wait) before it touches
// memory, so it runs on the completed results of everything before it; and
// lets the next kernel start launching at once (pdl_trigger), so that the
// next kernel's launch and block set-up overlap this one's tail. Both are
// no-ops for a kernel launched without the attribute.
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void pdl_trigger() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

__device__ __forceinline__ bool mbar_try(uint64_t* bar, uint32_t parity) {
  uint32_t done;
  asm volatile("{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n\t}"
               : "=r"(done)
               : "r"(smem_addr(bar)), "r"(parity)
               : "memory");
  return done != 0u;
}
__device__ __forceinline__ void mbar_arrive(uint64_t* bar) {
  asm volatile("{\n\t.reg .b64 st;\n\tmbarrier.arrive.shared.b64 st, [%0];\n\t}" ::"r"(smem_addr(bar)) : "memory");
}
// Bounded wait that also gives up as soon as another thread of the block has
// raised the abort flag.
__device__ __forceinline__ bool mbar_wait_or_abort(uint64_t* bar, uint32_t parity, uint32_t polls,
                                                   const volatile int* abort) {
  for (uint32_t i = 0; i < polls; ++i) {
    if (mbar_try(bar, parity)) return true;
    if (*abort) return false;
  }
  return false;
}
// The same for a whole warp, which goes on or gives up together: lanes poll for
// themselves, and one that saw the phase complete may stand beside one that ran out of
// polls or saw the flag. A warp that issues copies and parted there would copy what its
// lane 0 never announced, from places shuffled from lanes that have left. (The vote in
// the consumers of k_stage1_wide costs 0.2% of a MeerKAT-L block.)
__device__ __forceinline__ bool mbar_wait_warp(uint64_t* bar, uint32_t parity, uint32_t polls,
                                               const volatile int* abort) {
  return __all_sync(0xffffffffu, mbar_wait_or_abort(bar, parity, polls, abort));
}

// ---------------------------------------------------------------------------
// host side
// ---------------------------------------------------------------------------
// Launches kernel k with programmatic stream serialization (see pdl_wait):
// the launch and block set-up overlap the tail of the kernel before it.
template <typename... KArgs, typename... Args>
cudaError_t launch_pdl(void (*k)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, Args&&... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, k, std::forward<Args>(args)...);
}

// Raises kernel k's dynamic shared memory limit on the current device to at
// least `bytes`, never lowering it: plans of different shapes share kernels,
// and the limit one plan needs must survive another plan's set-up.
inline cudaError_t raise_smem_limit(const void* k, int bytes) {
  static std::mutex mu;
  static std::map<std::pair<int, const void*>, int> lim;
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  std::lock_guard<std::mutex> g(mu);
  const auto key = std::make_pair(dev, k);
  const auto it = lim.find(key);
  const int cur = it == lim.end() ? 48 * 1024 : it->second;  // the default limit
  if (bytes <= cur) return cudaSuccess;
  e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
  if (e == cudaSuccess) lim[key] = bytes;
  return e;
}

}  // namespace
