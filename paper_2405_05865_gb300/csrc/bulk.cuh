// Shared-memory staging primitives for sm_103a kernels: mbarrier waits with a
// wall-clock limit, bulk (TMA engine) global->shared copies, Ampere-style
// 16-byte async copies, and a named barrier for the worker warps of a
// warp-specialised block.
#pragma once

#include "msp_internal.cuh"

namespace msp {

__device__ inline uint32_t smem_u32(const void* p) {
    return (uint32_t)__cvta_generic_to_shared(p);
}

__device__ inline void mbar_init(uint64_t* bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count)
                 : "memory");
}

__device__ inline void mbar_arrive_expect_tx(uint64_t* bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.release.cta.shared::cta.b64 _, [%0], %1;" ::"r"(
                     smem_u32(bar)),
                 "r"(bytes)
                 : "memory");
}

__device__ inline void mbar_arrive(uint64_t* bar) {
    asm volatile("mbarrier.arrive.release.cta.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar))
                 : "memory");
}

// Cluster: the phase completes by what other CTAs of the cluster send here, which a
// wait orders at the cluster's scope only.
template <bool Cluster = false>
__device__ inline bool mbar_try_wait(uint64_t* bar, uint32_t parity) {
    uint32_t ok;
    if constexpr (Cluster)
        asm volatile(
            "{\n .reg .pred p;\n mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n"
            " selp.u32 %0, 1, 0, p;\n}\n"
            : "=r"(ok)
            : "r"(smem_u32(bar)), "r"(parity)
            : "memory");
    else
        asm volatile(
            "{\n .reg .pred p;\n mbarrier.try_wait.parity.acquire.cta.shared::cta.b64 p, [%1], %2;\n"
            " selp.u32 %0, 1, 0, p;\n}\n"
            : "=r"(ok)
            : "r"(smem_u32(bar)), "r"(parity)
            : "memory");
    return ok != 0;
}

// Bounded wait on the phase of the given parity: false (and *err =
// MSP_ETIMEOUT) after kWaitLimitNs. The phase is polled before the clock, so
// warps waiting on the same phase all see a completion that happened before
// any of them gave up; callers that meet at named barriers afterwards rely on
// every warp taking the same branch.
template <bool Cluster = false>
__device__ inline bool mbar_wait_timed(uint64_t* bar, uint32_t parity, int* err) {
    if (mbar_try_wait<Cluster>(bar, parity)) return true;
    const uint64_t t0 = globaltimer_ns();
    for (int spins = 0;; ++spins) {
        if (mbar_try_wait<Cluster>(bar, parity)) return true;
        if ((spins & 63) == 63 && globaltimer_ns() - t0 > kWaitLimitNs) {
            atomicExch(err, (int)MSP_ETIMEOUT);
            return false;
        }
    }
}

// try_wait with a suspend-time hint: the thread may sleep until the phase
// completes (or about `ns` nanoseconds pass) instead of polling.
__device__ inline bool mbar_try_wait_sleep(uint64_t* bar, uint32_t parity, uint32_t ns) {
    uint32_t ok;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.acquire.cta.shared::cta.b64 p, [%1], %2, %3;\n"
        " selp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(ok)
        : "r"(smem_u32(bar)), "r"(parity), "r"(ns)
        : "memory");
    return ok != 0;
}

// mbar_wait_timed with sleeping polls (long waits of warp-specialised roles)
__device__ inline bool mbar_wait_sleep(uint64_t* bar, uint32_t parity, int* err) {
    if (mbar_try_wait(bar, parity)) return true;
    const uint64_t t0 = globaltimer_ns();
    for (;;) {
        if (mbar_try_wait_sleep(bar, parity, 20000u)) return true;
        if (globaltimer_ns() - t0 > kWaitLimitNs) {
            atomicExch(err, (int)MSP_ETIMEOUT);
            return false;
        }
    }
}

__device__ inline void bulk_g2s(void* dst, const void* src, uint32_t bytes, uint64_t* bar) {
    asm volatile(
        "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
            smem_u32(dst)),
        "l"(src), "r"(bytes), "r"(smem_u32(bar))
        : "memory");
}

__device__ inline void bulk_g2s_hint(void* dst, const void* src, uint32_t bytes, uint64_t* bar,
                                     uint64_t policy) {
    asm volatile(
        "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint [%0], [%1], "
        "%2, [%3], %4;" ::"r"(smem_u32(dst)),
        "l"(src), "r"(bytes), "r"(smem_u32(bar)), "l"(policy)
        : "memory");
}

__device__ inline uint64_t policy_evict_first() {
    uint64_t pol;
    asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(pol));
    return pol;
}

// Explicit shared-memory accesses by 32-bit shared address (no generic
// address resolution).
__device__ inline float4 lds128(uint32_t a) {
    float4 v;
    asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "r"(a));
    return v;
}
__device__ inline void sts64(uint32_t a, uint32_t x, uint32_t y) {
    asm volatile("st.shared.v2.b32 [%0], {%1, %2};" ::"r"(a), "r"(x), "r"(y) : "memory");
}

// 16-byte async copy global -> shared; with valid == false the 16 bytes are
// zero-filled and nothing is read (src must still be a mapped address).
__device__ inline void cp_async16(void* dst, const void* src, bool valid) {
    const uint32_t sz = valid ? 16u : 0u;
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(smem_u32(dst)), "l"(src),
                 "r"(sz)
                 : "memory");
}

__device__ inline void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }

template <int N>
__device__ inline void cp_async_wait() {
    asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

// Barrier 1 over the first `count` threads of the block (the worker warps).
template <int Count>
__device__ inline void bar_workers() {
    asm volatile("bar.sync 1, %0;" ::"n"(Count) : "memory");
}

}  // namespace msp
