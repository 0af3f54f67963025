// PTX wrappers shared by the kernels: asynchronous copies, shared-memory accesses, packed fp32 pairs, mbarriers with bounded waits,
// fences, tensor-memory loads, operand descriptors.
#pragma once
#include <stdint.h>

namespace rptq {
namespace tc {

constexpr long long WAIT_BUDGET_CYCLES = 4000000000ll;   // about two seconds at the SM clock

__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

// 16 bytes global -> shared without passing through registers; `valid` false writes zeros and reads nothing
__device__ __forceinline__ void cp_async16(uint32_t dst, const void* src, bool valid)
{
    const uint32_t n = valid ? 16u : 0u;
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(n) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

__device__ __forceinline__ void sts128(uint32_t addr, uint32_t a, uint32_t b, uint32_t c, uint32_t d)
{
    asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(addr), "r"(a), "r"(b), "r"(c), "r"(d) : "memory");
}
__device__ __forceinline__ void sts32(uint32_t addr, uint32_t a) { asm volatile("st.shared.b32 [%0], %1;" ::"r"(addr), "r"(a) : "memory"); }
__device__ __forceinline__ uint4 lds128(uint32_t addr)
{
    uint4 v;
    asm volatile("ld.shared.v4.b32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(addr) : "memory");
    return v;
}
__device__ __forceinline__ uint32_t lds32(uint32_t addr)
{
    uint32_t v;
    asm volatile("ld.shared.b32 %0, [%1];" : "=r"(v) : "r"(addr) : "memory");
    return v;
}
__device__ __forceinline__ uint16_t lds16(uint32_t addr)
{
    uint16_t v;
    asm volatile("ld.shared.b16 %0, [%1];" : "=h"(v) : "r"(addr) : "memory");
    return v;
}

// packed fp32 pairs: one instruction, two independent IEEE results
__device__ __forceinline__ float2 add2(float2 a, float2 b)
{
    float2 d;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(reinterpret_cast<uint64_t&>(d))
        : "l"(reinterpret_cast<uint64_t&>(a)), "l"(reinterpret_cast<uint64_t&>(b)));
    return d;
}
__device__ __forceinline__ float2 mul2(float2 a, float2 b)
{
    float2 d;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(reinterpret_cast<uint64_t&>(d))
        : "l"(reinterpret_cast<uint64_t&>(a)), "l"(reinterpret_cast<uint64_t&>(b)));
    return d;
}
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c)
{
    float2 d;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(reinterpret_cast<uint64_t&>(d))
        : "l"(reinterpret_cast<uint64_t&>(a)), "l"(reinterpret_cast<uint64_t&>(b)), "l"(reinterpret_cast<uint64_t&>(c)));
    return d;
}

__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint32_t bar)
{
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
// Arrive on the barrier at the same shared-memory offset in CTA `rank` of the cluster.
__device__ __forceinline__ void mbar_arrive_remote(uint32_t bar, uint32_t rank)
{
    asm volatile(
        "{\n\t.reg .b32 ra;\n\t"
        "mapa.shared::cluster.u32 ra, %0, %1;\n\t"
        "mbarrier.arrive.shared::cluster.b64 _, [ra];\n\t}"
        ::"r"(bar), "r"(rank) : "memory");
}
__device__ __forceinline__ void mbar_arrive_expect_tx(uint32_t bar, uint32_t bytes)
{
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint32_t bar, uint32_t parity)
{
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok) : "r"(bar), "r"(parity) : "memory");
    return ok != 0;
}
// Bounded wait of a whole warp, for kernels with many waiting warps: sleeps in the barrier instruction instead of polling it. The
// limit is a number of wake-ups (each at most about a microsecond: two seconds in all). Every lane leaves with the same answer, or
// the lanes for which the barrier completed would wait for ever, at the next instruction that the whole warp takes part in, for
// those that gave up. One block of PTX, because a call site then takes half a dozen instructions: kernels with many roles
// are short of instruction cache.
__device__ __forceinline__ bool mbar_sleep_warp(uint32_t bar, uint32_t parity, volatile int* abort_flag)
{
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p, q;\n\t.reg .b32 n, f;\n\t"
        "mov.b32 n, 0;\n\t"
        "again:\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, 1000;\n\t"
        "@p bra done;\n\t"
        "ld.volatile.shared.b32 f, [%3];\n\t"
        "setp.ne.b32 q, f, 0;\n\t"
        "@q bra done;\n\t"
        "add.u32 n, n, 1;\n\t"
        "setp.lt.u32 q, n, 2097152;\n\t"
        "@q bra again;\n\t"
        "st.volatile.shared.b32 [%3], 1;\n\t"
        "done:\n\t"
        "vote.sync.all.pred p, p, 0xffffffff;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok) : "r"(bar), "r"(parity), "r"(smem_u32(const_cast<const int*>(abort_flag))) : "memory");
    return ok != 0;
}
// The same wait for a loop of a fixed trip count, which goes on whatever came of it and asks for the flag when it has ended: the
// lanes cannot part, and there is no vote (16 x 9216 x 36864: a vote per K block costs 0.8 of 45.8 us).
__device__ __forceinline__ void mbar_sleep_or_abort(uint32_t bar, uint32_t parity, volatile int* abort_flag)
{
    asm volatile(
        "{\n\t.reg .pred p;\n\t.reg .b32 n, f;\n\t"
        "mov.b32 n, 0;\n\t"
        "again:\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%0], %1, 1000;\n\t"
        "@p bra done;\n\t"
        "ld.volatile.shared.b32 f, [%2];\n\t"
        "setp.ne.b32 p, f, 0;\n\t"
        "@p bra done;\n\t"
        "add.u32 n, n, 1;\n\t"
        "setp.lt.u32 p, n, 2097152;\n\t"
        "@p bra again;\n\t"
        "st.volatile.shared.b32 [%2], 1;\n\t"
        "done:\n\t}"
        ::"r"(bar), "r"(parity), "r"(smem_u32(const_cast<const int*>(abort_flag))) : "memory");
}
// Bounded wait. Returns false when the budget ran out or another role already gave up. The common
// case (the phase has already completed, or completes within a few polls) touches no timer; the
// budget is counted on the SM's cycle counter, read once per batch of polls. Each lane has its own answer: for blocks that one
// lane executes, and for loops of a fixed trip count that go on whatever came of it.
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity, volatile int* abort_flag, bool heed_abort = true)
{
    auto poll = [&]() { return mbar_try_wait(bar, parity); };
    if (poll()) return true;
    if (poll()) return true;
    const long long t0 = clock64();
#pragma unroll 1
    while (true) {
#pragma unroll 1
        for (int i = 0; i < 16; ++i)
            if (poll()) return true;
        if (heed_abort && *abort_flag) return false;
        if (clock64() - t0 > WAIT_BUDGET_CYCLES) { *abort_flag = 1; return false; }
    }
}
// The same wait for a whole warp that must stay converged (the MMA-issuing warp): the lanes vote on
// every poll, so all of them leave the loop in the same iteration whatever each one saw.
__device__ __forceinline__ bool mbar_wait_warp(uint32_t bar, uint32_t parity, volatile int* abort_flag)
{
    if (__any_sync(0xffffffffu, mbar_try_wait(bar, parity))) return true;
    const long long t0 = clock64();
#pragma unroll 1
    while (true) {
#pragma unroll 1
        for (int i = 0; i < 1024; ++i)
            if (__any_sync(0xffffffffu, mbar_try_wait(bar, parity))) return true;
        const bool give_up = *abort_flag != 0 || clock64() - t0 > WAIT_BUDGET_CYCLES;
        if (__any_sync(0xffffffffu, give_up)) { *abort_flag = 1; return false; }
    }
}
__device__ __forceinline__ void fence_proxy_async() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_ld16(uint32_t taddr, uint32_t (&v)[16])
{
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
        : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]),
          "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15])
        : "r"(taddr) : "memory");
}
__device__ __forceinline__ void tc_wait_ld() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }

// K-major operand tile with 128-byte rows and the 128-byte swizzle: 8-row groups are 1024 bytes
// apart (stride byte offset), the leading byte offset is unused for swizzled K-major layouts.
__device__ __forceinline__ uint64_t smem_desc_sw128(uint32_t addr)
{
    uint64_t d = 0;
    d |= (uint64_t)((addr & 0x3FFFFu) >> 4);        // start address, 16-byte units
    d |= (uint64_t)1 << 16;                         // leading byte offset (ignored)
    d |= (uint64_t)(1024 >> 4) << 32;               // stride byte offset
    d |= (uint64_t)1 << 46;                         // descriptor version of this architecture
    d |= (uint64_t)2 << 61;                         // 128-byte swizzle
    return d;
}

}  // namespace tc
}  // namespace rptq
