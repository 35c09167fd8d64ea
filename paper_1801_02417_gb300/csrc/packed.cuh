// Device helpers shared by the CUDA kernels (sm_100 family and later).
// Packed FP32x2 arithmetic: two FP32 lanes in one 64-bit register pair, one
// fma.rn.f32x2 for both; each lane is rounded exactly like a separate fmaf.
// Bulk copies (cp.async.bulk, global to shared) completing on mbarriers, with
// bounded waits.
#pragma once

#include <cstdint>

#include <cuda.h>
#include <cuda_runtime.h>

namespace ps {

typedef unsigned long long u64;
__device__ __forceinline__ u64 f2pack(float a, float b) {
  u64 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
  return r;
}
__device__ __forceinline__ void f2unpack(u64 v, float& a, float& b) {
  asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(v));
}
__device__ __forceinline__ u64 ffma2(u64 a, u64 b, u64 c) {
  u64 d;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
  return d;
}
__device__ __forceinline__ u64 fdup(float a) { return f2pack(a, a); }
// Ordering of generic-proxy shared-memory accesses before later bulk (async-proxy) copies.
__device__ __forceinline__ void fence_proxy_async() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }

// ---- bulk-copy (TMA) and mbarrier helpers (inline PTX, sm_90+).
__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
  asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint64_t* bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes) : "memory");
}
__device__ __forceinline__ void bulk_g2s(void* dst, const void* src, uint32_t bytes, uint64_t* bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                   smem_u32(dst)),
               "l"(src), "r"(bytes), "r"(smem_u32(bar))
               : "memory");
}
// Bulk reduction: global[0 .. bytes) += shared[0 .. bytes) in FP32 (16-byte aligned, a multiple of 16
// bytes), in this thread's bulk groups: commit closes a group; wait_read<N> waits until at most N
// groups have still to read their shared memory, wait_all until every group is done.
__device__ __forceinline__ void bulk_reduce_add(float* dst, const float* src, uint32_t bytes) {
  asm volatile("cp.reduce.async.bulk.global.shared::cta.bulk_group.add.f32 [%0], [%1], %2;" ::"l"(dst),
               "r"(smem_u32(src)), "r"(bytes)
               : "memory");
}
__device__ __forceinline__ void bulk_commit() { asm volatile("cp.async.bulk.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void bulk_wait_read() {
  asm volatile("cp.async.bulk.wait_group.read %0;" ::"n"(N) : "memory");
}
__device__ __forceinline__ void bulk_wait_all() { asm volatile("cp.async.bulk.wait_group 0;" ::: "memory"); }
// 2D tensor-map copy (TMA) of one box into shared memory (128-byte aligned destination), completing
// on `bar`. The map lives in kernel-parameter space (a __grid_constant__ argument). x is the
// innermost coordinate in elements (x * 4 bytes a multiple of 16 for float data); parts of the
// box outside the tensor are filled with zeros and still count toward the transaction bytes.
__device__ __forceinline__ void tma_load_2d(void* dst, const CUtensorMap* map, int x, int y, uint64_t* bar) {
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];" ::"r"(
          smem_u32(dst)),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(x), "r"(y), "r"(smem_u32(bar))
      : "memory");
}

// The same tile brought to the L2 alone.
__device__ __forceinline__ void tma_prefetch_2d(const CUtensorMap* map, int x, int y) {
  asm volatile("cp.async.bulk.prefetch.tensor.2d.L2.global [%0, {%1, %2}];" ::"l"(reinterpret_cast<uint64_t>(map)),
               "r"(x), "r"(y)
               : "memory");
}

// ---- programmatic dependent launch. A kernel launched by launch_after (below) may start while the
// kernel before it in the stream still runs; pdl_wait returns when that kernel has completed and
// its writes are visible (at once if it already has, or the launch was an ordinary one). Every
// kernel launched so calls it first, before any access to global memory, so a kernel's completion
// implies that of every kernel before it. The kernel before lets it in when its own CTAs have ended:
// letting it in sooner (griddepcontrol.launch_dependents at the start) was slower, 491 against 455 us
// per iteration at 1024^2, its waiting CTAs taking room from the other branch of the iteration.
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// ---- thread-block clusters: the barrier of all threads of a cluster (release / acquire, so
// shared memory written before it is seen after it), and loads from the shared memory of
// the CTA of rank `r` at the address that `p` has in this CTA.
__device__ __forceinline__ void cluster_barrier() {
  asm volatile("barrier.cluster.arrive.release.aligned;\n barrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ uint32_t cluster_addr(const void* p, int r) {
  uint32_t a;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"(smem_u32(p)), "r"(r));
  return a;
}
__device__ __forceinline__ int ld_cluster(const int* p, int r) {
  int v;
  asm volatile("ld.shared::cluster.s32 %0, [%1];" : "=r"(v) : "r"(cluster_addr(p, r)) : "memory");
  return v;
}
__device__ __forceinline__ float4 ld_cluster4(const float* p, int r) {
  float4 v;
  asm volatile("ld.shared::cluster.v4.f32 {%0, %1, %2, %3}, [%4];"
               : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w)
               : "r"(cluster_addr(p, r))
               : "memory");
  return v;
}

// Poll budget of the bounded waits. c_wait_polls (one copy per translation unit,
// set by set_wait_polls_here) bounds the first wait on a barrier phase; a CTA
// whose wait gave up drains its copies still in flight with the full budget
// (mbar_drain) before it returns, so no copy lands after it has exited.
constexpr uint32_t kWaitPolls = 1u << 22;
static __constant__ uint32_t c_wait_polls = kWaitPolls;

__device__ __forceinline__ bool mbar_poll(uint64_t* bar, uint32_t parity, uint32_t polls) {
  const uint32_t a = smem_u32(bar);
  for (uint32_t i = 0; i < polls; ++i) {
    uint32_t ok;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(ok)
        : "r"(a), "r"(parity)
        : "memory");
    if (ok) return true;
  }
  return false;
}
// Bounded wait on phase `parity`: false (and the caller raises the error flag) if it never completes.
__device__ __forceinline__ bool mbar_wait(uint64_t* bar, uint32_t parity) { return mbar_poll(bar, parity, c_wait_polls); }
// Second wait of a CTA that gave up: the copies it issued get the full budget to land.
__device__ __forceinline__ bool mbar_drain(uint64_t* bar, uint32_t parity) { return mbar_poll(bar, parity, kWaitPolls); }

// Host side: launches a kernel that begins with pdl_wait so that it may start before the kernel
// before it in the stream has ended (in a captured stream: a programmatic graph edge); with
// early = false, an ordinary launch.
template <typename... P, typename... A>
static inline cudaError_t launch_after(bool early, void (*kern)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t stream,
                                       A&&... args) {
  cudaLaunchAttribute attr{};
  attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr.val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = stream;
  cfg.attrs = &attr;
  cfg.numAttrs = early ? 1 : 0;
  return cudaLaunchKernelEx(&cfg, kern, static_cast<P>(args)...);
}

// Host side: sets this translation unit's c_wait_polls (polls < 0: the default).
static inline cudaError_t set_wait_polls_here(int polls) {
  const uint32_t v = polls < 0 ? kWaitPolls : (uint32_t)polls;
  return cudaMemcpyToSymbol(c_wait_polls, &v, sizeof(v));
}
}  // namespace ps
