// Thin inline-PTX wrappers shared by the kernels: mbarrier, bounded waits, proxy fences.
#pragma once

#include <stdint.h>

namespace fq {

constexpr uint64_t kWaitLimitNs = 2000000000ull;   // every device-side wait gives up after 2 s

__device__ __forceinline__ uint32_t smem_u32(const void* p) {
    return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}
// One lane of a fully converged warp.  Issue work placed under `if (elect_one())` was measured
// much cheaper than under `if (lane == 0)`: the compiler then knows that a single thread runs it.
__device__ __forceinline__ bool elect_one() {
    uint32_t pred;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "elect.sync _|p, 0xffffffff;\n\t"
        "selp.b32 %0, 1, 0, p;\n\t}"
        : "=r"(pred));
    return pred != 0;
}
__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void mbar_arrive_expect_tx(uint32_t bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint32_t bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.b32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(bar), "r"(parity)
        : "memory");
    return ok != 0;
}
// Same, but the thread may stay suspended for up to `hint_ns` before the instruction returns:
// long waits then cost far fewer issue slots (and less power) than a tight polling loop.
__device__ __forceinline__ bool mbar_try_wait_hint(uint32_t bar, uint32_t parity, uint32_t hint_ns) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %3;\n\t"
        "selp.b32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(bar), "r"(parity), "r"(hint_ns)
        : "memory");
    return ok != 0;
}
__device__ __forceinline__ uint64_t global_timer_ns() {
    uint64_t t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

// Non-blocking test of a phase (never suspends the thread): used to look one stage ahead, so that
// the ~100-cycle latency of a barrier test overlaps with the work issued in between.
__device__ __forceinline__ bool mbar_test_wait(uint32_t bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.b32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(bar), "r"(parity)
        : "memory");
    return ok != 0;
}

// Bounded wait.  Returns false if the CTA is aborting or the limit expired
// (in which case the abort flag and the watchdog word are set).  The clock is read only after a
// few thousand failed tries (each try may itself suspend the thread for a while), so that the
// common short wait pays for nothing but the tries.
static __device__ __noinline__ bool mbar_wait_slow(uint32_t bar, uint32_t parity, volatile int* abort_flag,
                                            uint32_t* watchdog, uint32_t code, uint64_t limit_ns = kWaitLimitNs) {
    uint64_t t0 = 0;
    for (uint32_t spin = 1;; ++spin) {
        if (mbar_try_wait(bar, parity)) return true;
        if ((spin & 0xfff) == 0) {
            if (*abort_flag) return false;
            const uint64_t now = global_timer_ns();
            if (t0 == 0) t0 = now;
            if (now - t0 > limit_ns) {
                *abort_flag = 1;
                atomicOr(watchdog, code);
                return false;
            }
        }
    }
}
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity, volatile int* abort_flag,
                                          uint32_t* watchdog, uint32_t code, uint64_t limit_ns = kWaitLimitNs) {
    if (mbar_try_wait(bar, parity)) return true;
    if (mbar_try_wait(bar, parity)) return true;
    return mbar_wait_slow(bar, parity, abort_flag, watchdog, code, limit_ns);
}
// Warp-converged wait: every lane polls the same barrier, the result is made warp-uniform.
// Roles that hand work over through barriers run their loops with the whole warp converged and
// elect a lane only for the issue itself: a lone lane looping while its warp-mates are parked at a
// CTA barrier was measured 2-3x slower per dependent wait/arrive pair.
// `peeked` is the result of an earlier mbar_test_wait on the same phase: when it was already true
// the wait costs nothing.
__device__ __forceinline__ bool mbar_wait_all(uint32_t bar, uint32_t parity, volatile int* abort_flag,
                                              uint32_t* watchdog, uint32_t code, bool peeked = false,
                                              uint64_t limit_ns = kWaitLimitNs) {
    if (__all_sync(0xffffffffu, peeked)) return true;
    const bool ok = mbar_wait(bar, parity, abort_flag, watchdog, code, limit_ns);
    return __all_sync(0xffffffffu, ok);
}
// Converged wait for roles that run far ahead of their consumer (TMA producers behind a full ring): between
// tries the warp sleeps, so that it does not take issue slots from the warps on the critical path.
__device__ __forceinline__ bool mbar_wait_all_lazy(uint32_t bar, uint32_t parity, volatile int* abort_flag,
                                                   uint32_t* watchdog, uint32_t code, bool peeked = false) {
    if (__all_sync(0xffffffffu, peeked)) return true;
    bool ok = true;
    if (!mbar_try_wait(bar, parity)) {
        const uint64_t t0 = global_timer_ns();
        for (uint32_t spin = 1; !mbar_try_wait(bar, parity); ++spin) {
            __nanosleep(100);
            if ((spin & 0x3ff) == 0) {
                if (*abort_flag) { ok = false; break; }
                if (global_timer_ns() - t0 > kWaitLimitNs) {
                    *abort_flag = 1;
                    atomicOr(watchdog, code);
                    ok = false;
                    break;
                }
            }
        }
    }
    return __all_sync(0xffffffffu, ok);
}
// Wait for latency-tolerant roles (epilogue): lane 0 polls with a short sleep between tries so that
// an idle warp does not compete for issue slots with the warps feeding the tensor core.
__device__ __forceinline__ bool mbar_wait_warp_relaxed(uint32_t bar, uint32_t parity, volatile int* abort_flag,
                                                       uint32_t* watchdog, uint32_t code) {
    int ok = 1;
    if ((threadIdx.x & 31) == 0) {
        const uint64_t t0 = global_timer_ns();
        for (uint32_t spin = 1; !mbar_try_wait(bar, parity); ++spin) {
            __nanosleep(200);
            if ((spin & 0x3f) == 0) {
                if (*abort_flag) { ok = 0; break; }
                if (global_timer_ns() - t0 > kWaitLimitNs) {
                    *abort_flag = 1;
                    atomicOr(watchdog, code);
                    ok = 0;
                    break;
                }
            }
        }
    }
    return __shfl_sync(0xffffffffu, ok, 0) != 0;
}
// Warp-collective wait: lane 0 waits, the result is broadcast (one poller per warp instead of 32).
__device__ __forceinline__ bool mbar_wait_warp(uint32_t bar, uint32_t parity, volatile int* abort_flag,
                                               uint32_t* watchdog, uint32_t code) {
    int ok = 1;
    if ((threadIdx.x & 31) == 0) ok = mbar_wait(bar, parity, abort_flag, watchdog, code) ? 1 : 0;
    return __shfl_sync(0xffffffffu, ok, 0) != 0;
}

// Programmatic dependent launch.  A kernel launched with the programmatic-serialization attribute
// may start while the kernel before it in the stream is still running; griddep_wait() returns once
// that kernel has completed and its writes are visible, so everything that touches global memory
// comes after it and only on-chip setup (barriers, TMEM, descriptor prefetch) runs ahead.
// griddep_launch_dependents() lets the NEXT kernel in the stream begin its own setup early; issued ahead of griddep_wait(),
// even before the kernel in front of this one has ended (what comes before a wait must not depend on either of them).
__device__ __forceinline__ void griddep_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void griddep_launch_dependents() {
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

// Loads, behind griddep_wait(), of memory that a kernel ahead may have written while this one was already resident: what
// the caller passes in (tokens, steps, codes, a multiplier of its own) and what an earlier kernel of the call left in the
// workspace.  Not __ldg and not through `const T* __restrict__`, which become loads of the non-coherent kind: those are for
// memory that nobody writes as long as the kernel lives, and the compiler may move them across the wait.  Three calls in a
// row share an SM (the third one is resident before the first has ended), so a line read by the first may have been
// rewritten when the third one reads it.  (What a complete handle holds is written by nobody: __ldg, ahead of the wait or behind.)
__device__ __forceinline__ uint4 ld_global_v4(const void* p, bool ok = true) {      // zeros where !ok
    uint4 v;
    asm volatile(
        "{\n\t.reg .pred q;\n\t"
        "setp.ne.b32 q, %5, 0;\n\t"
        "mov.b32 %0, 0;\n\tmov.b32 %1, 0;\n\tmov.b32 %2, 0;\n\tmov.b32 %3, 0;\n\t"
        "@q ld.global.v4.b32 {%0, %1, %2, %3}, [%4];\n\t}"
        : "=&r"(v.x), "=&r"(v.y), "=&r"(v.z), "=&r"(v.w)
        : "l"(p), "r"((uint32_t)ok));
    return v;
}
__device__ __forceinline__ float4 ld_global_f4(const void* p, bool ok = true) {
    const uint4 v = ld_global_v4(p, ok);
    return make_float4(__uint_as_float(v.x), __uint_as_float(v.y), __uint_as_float(v.z), __uint_as_float(v.w));
}
__device__ __forceinline__ uint32_t ld_global_u32(const void* p) {
    uint32_t v;
    asm volatile("ld.global.b32 %0, [%1];" : "=r"(v) : "l"(p));
    return v;
}
__device__ __forceinline__ float ld_global_f32(const float* p) { return __uint_as_float(ld_global_u32(p)); }
__device__ __forceinline__ uint32_t ld_global_u16(const void* p) {
    uint16_t v;
    asm volatile("ld.global.b16 %0, [%1];" : "=h"(v) : "l"(p));
    return v;
}

// Ask for the 128-byte line at p to be brought into L2.  No value is read: allowed ahead of griddep_wait() even for memory
// that the kernel in front is writing.
__device__ __forceinline__ void prefetch_l2(const void* p) { asm volatile("prefetch.global.L2 [%0];" ::"l"(p)); }

__device__ __forceinline__ void sts32(uint32_t addr, uint32_t v) { asm volatile("st.shared.b32 [%0], %1;" ::"r"(addr), "r"(v) : "memory"); }
__device__ __forceinline__ void fence_proxy_async_smem() {
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}
__device__ __forceinline__ void fence_mbarrier_init() {
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}
// Bulk stores: groups per issuing thread.
__device__ __forceinline__ void bulk_commit() { asm volatile("cp.async.bulk.commit_group;" ::: "memory"); }
// At most N of this thread's bulk groups still read their shared-memory source.
template <int N>
__device__ __forceinline__ void bulk_wait_read() { asm volatile("cp.async.bulk.wait_group.read %0;" ::"n"(N) : "memory"); }
// 1-D bulk copy global -> shared (16-byte aligned addresses, size a multiple of 16 bytes).
__device__ __forceinline__ void bulk_load_1d(uint32_t dst, const void* src, uint32_t bytes, uint32_t bar) {
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                 ::"r"(dst), "l"(src), "r"(bytes), "r"(bar)
                 : "memory");
}

}  // namespace fq
