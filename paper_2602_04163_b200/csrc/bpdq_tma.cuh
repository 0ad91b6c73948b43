// mbarrier and TMA wrappers shared by the kernels that stage packed weights through shared memory, and the host-side
// tensor-map encoder (fetched from the driver at run time: the library does not link libcuda).
#pragma once
#include <cstdint>
#include <cuda.h>

#include "bpdq.h"

namespace bpdq {

typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
EncodeTiledFn encode_tiled_fn();      // null when the driver does not offer cuTensorMapEncodeTiled

#if defined(__CUDACC__)
namespace tma {

__device__ __forceinline__ unsigned smem_u32(const void* p) { return (unsigned)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void mbar_init(unsigned bar, unsigned count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_arrive(unsigned bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void mbar_expect_tx(unsigned bar, unsigned bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(unsigned bar, unsigned parity) {
    unsigned ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok) : "r"(bar), "r"(parity) : "memory");
    return ok != 0;
}
// Bounded wait: gives up after max_ns nanoseconds (mbarrier.try_wait itself blocks for a hardware-defined slice per
// poll, so the bound is taken on the clock, read every 64 polls, not on the poll count).  Returns false if the CTA has
// been aborted or the limit ran out (and aborts it, recording BPDQ_ERR_TIMEOUT in the status word).
__device__ __forceinline__ unsigned long long global_ns() {
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}
__device__ __forceinline__ bool mbar_wait_ns(unsigned bar, unsigned parity, volatile int* abort_flag, int* status, unsigned long long max_ns) {
    if (mbar_try_wait(bar, parity)) return true;
    const unsigned long long t0 = global_ns();
    for (unsigned n = 1;; ++n) {
        if (mbar_try_wait(bar, parity)) return true;
        if ((n & 63u) == 63u) {
            if (*abort_flag) return false;
            if (global_ns() - t0 > max_ns) break;
        }
    }
    *abort_flag = 1;
    atomicExch(status, BPDQ_ERR_TIMEOUT);
    return false;
}
constexpr unsigned long long kWaitNanos = 2000000000ull;       // two seconds: far beyond any wait of a healthy launch
__device__ __forceinline__ bool mbar_wait(unsigned bar, unsigned parity, volatile int* abort_flag, int* status) {
    return mbar_wait_ns(bar, parity, abort_flag, status, kWaitNanos);
}
// One lane of a converged warp.  Code behind it (unlike behind "lane == 0") is known to run in a single thread of a
// warp that is otherwise together, so the operands of a tcgen05.mma stay in uniform registers: the issue loops of the
// tensor-core kernels then keep up with the pipe (four 72B-shaped launches with 48 tokens, K = 2: 367 -> 329 us, a
// 7B-shaped layer with 777 tokens 785 -> 724 us, a 72B-shaped layer with 4096 tokens 6.92 -> 6.71 ms).
__device__ __forceinline__ bool elect_one() {
    unsigned is;
    asm volatile("{\n\t.reg .pred p;\n\telect.sync _|p, 0xffffffff;\n\tselp.u32 %0, 1, 0, p;\n\t}" : "=r"(is));
    return is != 0;
}
// The bounded wait by a whole warp: the same answer in every lane, also when the wait of some lanes ran out.
__device__ __forceinline__ bool mbar_wait_warp(unsigned bar, unsigned parity, volatile int* abort_flag, int* status) {
    return __all_sync(0xffffffffu, mbar_wait(bar, parity, abort_flag, status)) != 0;
}
// A CTA that gave up may have copies under way, and its shared memory must outlive them: it stays for a millisecond, a thousand times
// what a copy takes.  (Waiting on the rings' barriers instead cost every launch up to 1 % in registers or polls.)
constexpr unsigned long long kLingerNanos = 1000000ull;
__device__ __forceinline__ void linger() {
    const unsigned long long t0 = global_ns();
    while (global_ns() - t0 < kLingerNanos) {}
}
__device__ __forceinline__ void fence_proxy_async() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }
__device__ __forceinline__ void fence_barrier_init() { asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory"); }

__device__ __forceinline__ void tma_load_2d(unsigned dst, const CUtensorMap* map, int c0, int c1, unsigned bar) {
    asm volatile(
        "cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];"
        ::"r"(dst), "l"(map), "r"(c0), "r"(c1), "r"(bar) : "memory");
}
__device__ __forceinline__ void tma_load_3d(unsigned dst, const CUtensorMap* map, int c0, int c1, int c2, unsigned bar) {
    asm volatile(
        "cp.async.bulk.tensor.3d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4}], [%5];"
        ::"r"(dst), "l"(map), "r"(c0), "r"(c1), "r"(c2), "r"(bar) : "memory");
}
}  // namespace tma
#endif

}  // namespace bpdq
