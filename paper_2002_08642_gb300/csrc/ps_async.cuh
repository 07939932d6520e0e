// ps_async.cuh -- bulk asynchronous copies global -> shared through the
// tensor memory accelerator (cp.async.bulk, completion counted on an
// mbarrier), with bounded waits: a wait that does not complete within its
// iteration cap returns false so that the kernel can record an error and
// finish instead of spinning forever.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

namespace ps {

// Programmatic dependent launch: a kernel launched with launch() may start
// while the previous kernel of the stream ends (its blocks are scheduled when
// the last of that kernel's blocks has exited, before its writes are flushed)
// and does its set-up (barriers, twiddle tables: written once, when the
// context is made) there; pdl_wait() then holds every block, before its first
// access to anything an earlier kernel touched, until all earlier kernels are
// complete and their writes visible. Every kernel launched with launch()
// calls pdl_wait() in every block, so completion carries over from kernel to
// kernel. A no-op in a plain launch.
// GB300: decaying box 32^3 FP64 (100 small kernels) 1090 -> 851 us, wing 48^3
// 794 -> 665, plate 128^3 945 -> 805, wing 256^3 2247 -> 2164, 512^3 unchanged.
// Not kept: an explicit early trigger (griddepcontrol.launch_dependents) at
// the kernels' start; the next kernel's blocks then gather on the SMs that are
// free first (32^3 FP64 1175 us, wing 256^3 2295, adjoint 512^3 5 % slower).
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

template <class... P, class... A>
inline cudaError_t launch(void (*kernel)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t s, A&&... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute at = {};
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kernel, static_cast<A&&>(args)...);
}

__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}

// make mbarrier initialisation visible to the async proxy
__device__ __forceinline__ void fence_mbar_init() {
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}

// order this thread's earlier generic-proxy shared-memory accesses before
// later async-proxy (bulk copy) accesses
__device__ __forceinline__ void fence_proxy_async() {
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}

__device__ __forceinline__ void mbar_arrive_expect_tx(uint64_t* bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes)
                 : "memory");
}

// bytes and both addresses must be multiples of 16
__device__ __forceinline__ void bulk_g2s(void* dst, const void* src, uint32_t bytes, uint64_t* bar) {
    asm volatile(
        "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
            smem_u32(dst)),
        "l"(src), "r"(bytes), "r"(smem_u32(bar))
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

// Bounded wait for the phase with the given parity: false after `cap`
// polls (each poll may itself suspend the thread for a short while).
__device__ __forceinline__ bool mbar_wait_cap(uint64_t* bar, uint32_t parity, uint32_t cap) {
    for (uint32_t i = 0; i < cap; ++i)
        if (mbar_try_wait(bar, parity)) return true;
    return false;
}

// The kernels' wait: 2^22 polls, far longer than any copy takes.
__device__ __forceinline__ bool mbar_wait(uint64_t* bar, uint32_t parity) {
    return mbar_wait_cap(bar, parity, 1u << 22);
}

}  // namespace ps

#include <cuda.h>

namespace ps {

// Tiled TMA loads of a box at element coordinates (c0 innermost).
__device__ __forceinline__ void tma_load_2d(void* dst, const CUtensorMap* tm, int c0, int c1, uint64_t* bar) {
    asm volatile(
        "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];" ::"r"(
            smem_u32(dst)),
        "l"(tm), "r"(c0), "r"(c1), "r"(smem_u32(bar))
        : "memory");
}

__device__ __forceinline__ void tma_load_3d(void* dst, const CUtensorMap* tm, int c0, int c1, int c2,
                                            uint64_t* bar) {
    asm volatile(
        "cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4}], [%5];" ::"r"(
            smem_u32(dst)),
        "l"(tm), "r"(c0), "r"(c1), "r"(c2), "r"(smem_u32(bar))
        : "memory");
}

// Pull a box into L2 ahead of use (no shared memory, no completion).
__device__ __forceinline__ void tma_prefetch_2d(const CUtensorMap* tm, int c0, int c1) {
    asm volatile("cp.async.bulk.prefetch.tensor.2d.L2.global [%0, {%1, %2}];" ::"l"(tm), "r"(c0), "r"(c1) : "memory");
}

}  // namespace ps
