// Device helpers shared by the library's kernels: mbarrier + bulk-copy PTX,
// bounded waits, the device status word.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

namespace ndf {

// Programmatic dependent launch.  A kernel that begins with pdl_wait() may be launched by
// launch_after() while its predecessor on the stream still runs: its CTAs take the places that
// the predecessor's leave, and pdl_wait() holds them until that grid has completed and its writes
// are visible.  pdl_launch() in the predecessor allows it as soon as all its CTAs have started
// (without it, when they have ended).  Hides the launch and the ramp of short dependent kernels.
// Such a kernel takes what its predecessor writes through plain pointers: a load through a const
// __restrict__ one (or __ldg) counts as invariant, and the compiler may move it above the wait.
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void pdl_launch() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

template <class... P, class... A>
inline cudaError_t launch_after(void (*kern)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t s, A... args) {
    cudaLaunchAttribute at;
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kern, static_cast<P>(args)...);
}

// Lifts a kernel's dynamic shared memory limit to the most a CTA can have, whatever the launch at
// hand needs: the limit belongs to the function and the device, so a smaller one set for one
// thread's launch would refuse another thread's larger launch that is about to follow.
constexpr size_t kMaxDynamicSmem = 227 * 1024;
template <class Kern>
inline cudaError_t allow_dynamic_smem(Kern kern) {
    return cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kMaxDynamicSmem);
}

// Bit flags of the device status word (ctx->flag, word 1).
enum : unsigned { kDevTimeout = 1u, kDevBadInput = 2u };

// Bounds of an mbarrier wait: at most kWaitPolls polls (each a hardware try_wait
// with its own short suspend window) and at most kWaitNs nanoseconds of
// %globaltimer, checked every 1024 polls; both far above any real completion
// time, far below a hang.
constexpr uint32_t kWaitPolls = 1u << 24;
constexpr uint64_t kWaitNs = 1000000000ull;

__device__ __forceinline__ uint64_t global_ns() {
    uint64_t t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

__device__ __forceinline__ uint32_t smem_u32(const void* p) {
    return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count)
                 : "memory");
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}

__device__ __forceinline__ void mbar_expect_tx(uint64_t* bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)),
                 "r"(bytes)
                 : "memory");
}

// Returns true when the phase with parity `phase` has completed, false when
// the poll budget ran out.
__device__ __forceinline__ bool mbar_wait(uint64_t* bar, uint32_t phase) {
    uint32_t addr = smem_u32(bar);
    uint64_t t0 = 0;
    for (uint32_t i = 0; i < kWaitPolls; ++i) {
        uint32_t done;
        asm volatile(
            "{\n\t.reg .pred p;\n\t"
            "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
            "selp.u32 %0, 1, 0, p;\n\t}"
            : "=r"(done)
            : "r"(addr), "r"(phase)
            : "memory");
        if (done) return true;
        if ((i & 1023u) == 1023u) {
            const uint64_t t = global_ns();
            if (t0 == 0) t0 = t;
            else if (t - t0 > kWaitNs) return false;
        }
    }
    return false;
}

// 1-D bulk copy global -> shared, completion counted on `bar` (bytes and both
// addresses must be multiples of 16).
__device__ __forceinline__ void bulk_g2s(void* dst, const void* src, uint32_t bytes,
                                         uint64_t* bar) {
    asm volatile(
        "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::
            "r"(smem_u32(dst)),
        "l"(src), "r"(bytes), "r"(smem_u32(bar))
        : "memory");
}

__device__ __forceinline__ void report(unsigned* status, unsigned bit) {
    if (status) atomicOr(status, bit);
}

}  // namespace ndf
