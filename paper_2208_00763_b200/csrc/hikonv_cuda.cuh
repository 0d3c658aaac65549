// Small device/host helpers shared by the CUDA translation units.
#pragma once

#include <cuda_runtime.h>

#include <cstdint>

#include "hikonv_internal.h"

namespace hikonv {

// Evaluates a CUDA runtime call; on failure returns HIKONV_ERR_CUDA from the enclosing function.
#define HIKONV_CUDA_TRY(expr)                                 \
    do {                                                      \
        cudaError_t _e = (expr);                              \
        if (_e != cudaSuccess) return HIKONV_ERR_CUDA;        \
    } while (0)

// Plain launch that is judged by its own result: the status is what cudaLaunchKernelEx returns for THIS launch,
// so an error that an earlier, unrelated call left unread in the thread's error state is neither reported here
// nor cleared.
template <typename... Params, typename... Args>
inline int launch_plain(void (*kernel)(Params...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, Args... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cfg.attrs = nullptr;
    cfg.numAttrs = 0;
    return cudaLaunchKernelEx(&cfg, kernel, args...) == cudaSuccess ? HIKONV_OK : HIKONV_ERR_CUDA;
}

// Programmatic dependent launch.  A kernel launched with launch_dependent() may be scheduled while the
// kernel before it on the stream is still running; it must call grid_dependency_wait() before its first
// access to global memory (the wait returns once the earlier kernel has finished and its writes are
// visible).  grid_dependency_release() lets the NEXT kernel of the stream be scheduled early; it takes
// effect once every CTA of this grid has called it or exited.  Every CTA of every such kernel waits, so
// completion of a kernel still implies completion of all kernels before it.
// What a kernel reads that is launched this way may be written by the kernel before while it already runs, so it is not constant
// over the kernel's lifetime: ordinary loads, which stay behind the wait, and not the read-only path (__ldg, const __restrict__).
template <typename T>
__device__ __forceinline__ T load_ordered(const T *p) {
    return *p;
}
__device__ __forceinline__ void grid_dependency_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void grid_dependency_release() { asm volatile("griddepcontrol.launch_dependents;"); }

template <typename... Params, typename... Args>
inline int launch_dependent(void (*kernel)(Params...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, Args... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kernel, args...) == cudaSuccess ? HIKONV_OK : HIKONV_ERR_CUDA;
}

// Runs `launch` (which returns a hikonv status) for a kernel that needs `bytes` of dynamic shared memory.  Beyond 48 KB the
// kernel's limit has to be raised, once per device; every thread remembers for which kernels it has seen that done.  A launch
// that fails all the same (the device may have been reset in between) is tried once more with the limit raised again.
template <typename Launch>
inline int with_dynamic_smem(const void *kernel, size_t bytes, Launch launch) {
    constexpr size_t kPlain = 48 * 1024;
    constexpr int kMost = 227 * 1024, kSlots = 256;
    struct Raised {
        const void *kernel;
        int dev;
    };
    static thread_local Raised raised[kSlots];
    if (bytes <= kPlain) return launch();
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return HIKONV_ERR_CUDA;
    Raised &r = raised[(((uintptr_t)kernel >> 4) ^ (uintptr_t)dev) % kSlots];
    const bool known = r.kernel == kernel && r.dev == dev;
    if (!known && cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kMost) != cudaSuccess) return HIKONV_ERR_CUDA;
    r.kernel = kernel;
    r.dev = dev;
    const int rc = launch();
    if (rc == HIKONV_OK || !known) return rc;
    if (cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kMost) != cudaSuccess) return HIKONV_ERR_CUDA;
    return launch();
}

// The 32x32->64 product of two packed words (Eq. 9).  The multiply is given as inline PTX (mul.wide) and the
// 64-bit add is left to the compiler, which fuses the pair into one wide multiply-add.  Two other spellings were
// tried and dropped after counting instructions per opcode in the profiler: mad.wide as inline PTX came out as a
// multiply plus separate 64-bit additions, and the plain C++ expression (int64)a * (int64)b + c becomes a full
// 64-bit multiply (three multiplies and adds) whenever the optimiser has hoisted or combined one of the sign
// extensions.
template <bool SIGNED>
__device__ __forceinline__ uint64_t mul_wide(uint32_t a, uint32_t b) {
    uint64_t r;
    if (SIGNED)
        asm("mul.wide.s32 %0, %1, %2;" : "=l"(r) : "r"(a), "r"(b));
    else
        asm("mul.wide.u32 %0, %1, %2;" : "=l"(r) : "r"(a), "r"(b));
    return r;
}

// acc += a * b.
template <bool SIGNED>
__device__ __forceinline__ void mad_wide(uint64_t &acc, uint32_t a, uint32_t b) {
    acc += mul_wide<SIGNED>(a, b);
}

// a * b + c with the addend as an operand of its own.
template <bool SIGNED>
__device__ __forceinline__ uint64_t mul_wide_add(uint32_t a, uint32_t b, uint64_t c) {
    return c + mul_wide<SIGNED>(a, b);
}

// Low 32 bits of (v >> sh) for 0 <= sh < 64.
__device__ __forceinline__ uint32_t shr64_lo(uint64_t v, int sh) { return (uint32_t)(v >> sh); }

// A code byte as a 32-bit value (sign- or zero-extended).
template <bool SIGNED>
__device__ __forceinline__ int32_t code_value(int8_t b) {
    return SIGNED ? (int32_t)b : (int32_t)(uint8_t)b;
}

template <bool SIGNED>
__device__ __forceinline__ int32_t load_code(const int8_t *p) {
    return code_value<SIGNED>(load_ordered(p));
}

// prmt with a selector known at run time (__byte_perm ignores the bit that replicates a byte's sign).
__device__ __forceinline__ uint32_t byte_permute(uint32_t a, uint32_t b, uint32_t sel) {
    uint32_t r;
    asm("prmt.b32 %0, %1, %2, %3;" : "=r"(r) : "r"(a), "r"(b), "r"(sel));
    return r;
}

// Byte `b` (0..3) of w as a 32-bit value, sign- or zero-extended: one prmt.
template <bool SIGNED>
__device__ __forceinline__ uint32_t extract_code(uint32_t w, int b) {
    uint32_t r;
    // selector nibbles: low nibble picks byte b; in the upper three, bit 3 replicates that byte's sign,
    // or index 4 picks byte 0 of the zero second operand
    const uint32_t sel = SIGNED ? (uint32_t)(b | ((8 | b) << 4) | ((8 | b) << 8) | ((8 | b) << 12)) : (uint32_t)(b | 0x4440);
    asm("prmt.b32 %0, %1, %2, %3;" : "=r"(r) : "r"(w), "r"(0u), "r"(sel));
    return r;
}

// Asynchronous global -> shared copies (cp.async); src_bytes < 4 zero-fills the rest of the 4-byte word.
__device__ __forceinline__ void cp_async_4(void *smem_dst, const void *gmem_src, int src_bytes) {
    const unsigned dst = (unsigned)__cvta_generic_to_shared(smem_dst);
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(dst), "l"(gmem_src), "r"(src_bytes) : "memory");
}
__device__ __forceinline__ void cp_async_16_at(uint32_t smem_dst, const void *gmem_src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_dst), "l"(gmem_src) : "memory");
}
__device__ __forceinline__ void cp_async_16(void *smem_dst, const void *gmem_src) {
    cp_async_16_at((uint32_t)__cvta_generic_to_shared(smem_dst), gmem_src);
}

// Bulk copies (one thread moves up to a whole tile through the TMA unit) that report their bytes to an mbarrier in shared
// memory.  Both addresses are 16-byte aligned and the size is a multiple of 16.
__device__ __forceinline__ uint32_t smem_address(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ void mbarrier_init(uint32_t bar, uint32_t arrivals) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(arrivals) : "memory");
}
__device__ __forceinline__ void mbarrier_init_fence() { asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory"); }
__device__ __forceinline__ void mbarrier_arrive_expect(uint32_t bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ void bulk_copy(uint32_t smem_dst, const void *gmem_src, uint32_t bytes, uint32_t bar) {
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(smem_dst), "l"(gmem_src),
                 "r"(bytes), "r"(bar)
                 : "memory");
}
__device__ __forceinline__ bool mbarrier_try_wait(uint32_t bar, uint32_t parity) {
    uint32_t done;
    asm volatile("{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n\t}"
                 : "=r"(done)
                 : "r"(bar), "r"(parity)
                 : "memory");
    return done != 0;
}
// Waits for the phase of this parity to complete, for so many cycles at most (the default, one second, is far above any copy's
// time).  Returns false when they ran out.
constexpr long long kWaitCycles = 2000000000ll;
__device__ __forceinline__ bool mbarrier_wait(uint32_t bar, uint32_t parity, long long cycles = kWaitCycles) {
    if (mbarrier_try_wait(bar, parity)) return true;
    const long long start = clock64();
    do {
        if (mbarrier_try_wait(bar, parity)) return true;
    } while (clock64() - start < cycles);
    return false;
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_group 0;" ::: "memory"); }

}  // namespace hikonv
