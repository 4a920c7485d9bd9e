// Helpers of several kernels: shared-memory addresses, the global timer for
// bounded waits, mbarrier set-up / arrive / try-wait, and conversions between
// FP32 and FP64.
#pragma once

#include <stdint.h>

namespace lbm {

// Bound on any wait for an mbarrier phase: 2 s of wall time.
constexpr uint64_t WAIT_NS = 2000000000ull;

static __device__ __forceinline__ uint32_t smem_u32(const void* p) {
    return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

static __device__ __forceinline__ uint64_t globaltimer_ns() {
    uint64_t t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

// The timer once x is there: the read is predicated on x, so that it waits for
// the loads x was formed from. (t where x is -1e30, which no density is.)
static __device__ __forceinline__ uint64_t globaltimer_ns_after(float x, uint64_t t) {
    asm volatile("{\n\t.reg .pred p;\n\tsetp.neu.f32 p, %1, 0fF149F2CA;\n\t@p mov.u64 %0, %%globaltimer;\n\t}" : "+l"(t) : "f"(x));
    return t;
}
static __device__ __forceinline__ uint64_t globaltimer_ns_after(double x, uint64_t t) {
    return globaltimer_ns_after(__int_as_float(__double2hiint(x)), t);
}

static __device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}

static __device__ __forceinline__ void fence_mbar_init() {
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}

static __device__ __forceinline__ void fence_proxy_async() {
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}

static __device__ __forceinline__ void mbar_arrive_expect_tx(uint64_t* bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes)
                 : "memory");
}

static __device__ __forceinline__ bool mbar_try_wait(uint64_t* bar, uint32_t parity) {
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

// float <-> double by integer arithmetic, the same bits as the conversions: the
// conversion unit takes a warp every 16 cycles, as FP64 arithmetic does, the
// integer units eight operations in that time on each of the four schedulers.
// (Values out of the normal FP32 range are left to the unit.)
// (The unit's conversions are calls: as predicated instructions they would take
// their cycles on the path that skips them too.)
static __device__ __noinline__ double widen_unit(float v) { return (double)v; }
static __device__ __noinline__ float narrow_unit(double v) { return (float)v; }
static __device__ __forceinline__ double widen(float v) {
    const uint32_t u = __float_as_uint(v), a = u << 1;
    if (a - 0x01000000u >= 0xfe000000u) return widen_unit(v);  // zero, subnormal, infinite or NaN
    return __hiloint2double((int)((u & 0x80000000u) | ((a >> 4) + 0x38000000u)), (int)(u << 29));
}
static __device__ __forceinline__ float narrow(double v) {  // to nearest, ties to even
    const uint32_t h = (uint32_t)__double2hiint(v), l = (uint32_t)__double2loint(v);
    const uint32_t a = h & 0x7fffffffu;
    if (a - 0x38100000u >= 0x0fd00000u) return narrow_unit(v);  // below 2^-126, or 2^127 and more
    // the exponent and the upper 23 bits of the fraction; the 29 below round
    const uint32_t m = ((a - 0x38000000u) << 3) | (l >> 29), rest = l << 3;
    const uint32_t up = (rest > 0x80000000u || (rest == 0x80000000u && (m & 1u))) ? 1u : 0u;
    return __uint_as_float((h & 0x80000000u) | (m + up));
}

}  // namespace lbm
