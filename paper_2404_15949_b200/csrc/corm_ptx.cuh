// Instructions without a CUDA C++ spelling (barriers in shared memory, asynchronous copies, fences) and fp64 exponentials,
// shared by the kernels.
#pragma once

#include "corm_common.cuh"

namespace corm {

constexpr long long kWaitLimitCycles = 4000000000ll;   // bounded mbarrier waits (about 2 s)

__device__ __forceinline__ uint32_t smem_addr(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint32_t bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint32_t bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(ok) : "r"(bar), "r"(parity) : "memory");
    return ok != 0;
}
// Waits for the phase with the given parity; gives up after kWaitLimitCycles and reports false.
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity) {
    if (mbar_try_wait(bar, parity)) return true;
    const long long start = clock64();
    while (!mbar_try_wait(bar, parity))
        if (clock64() - start > kWaitLimitCycles) return false;
    return true;
}
// Waits until the unit's stamp says that at least `steps_done` decode steps of it are complete and returns the stamp.
// Gives up (all ones) after kWaitLimitCycles, reporting a timeout, or as soon as another block has reported a
// failure that leaves the cache unusable anyway.
__device__ __forceinline__ unsigned long long wait_unit_stamp(const unsigned long long* stamp, uint32_t steps_done, int32_t* status) {
    const long long start = clock64();
    for (;;) {
        unsigned long long v;
        asm volatile("ld.acquire.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(stamp) : "memory");
        if ((uint32_t)(v >> 32) >= steps_done) return v;
        const int32_t s = *reinterpret_cast<volatile int32_t*>(status);
        if (s == CORM_ERR_TIMEOUT || s == CORM_ERR_INTERNAL) return ~0ull;
        if (clock64() - start > kWaitLimitCycles) { report_status(status, CORM_ERR_TIMEOUT); return ~0ull; }
        __nanosleep(64);
    }
}
__device__ __forceinline__ void bulk_load(uint32_t dst_smem, const void* src_gmem, uint32_t bytes, uint32_t bar) {
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                 ::"r"(dst_smem), "l"(src_gmem), "r"(bytes), "r"(bar) : "memory");
}
// 16-byte asynchronous copy global -> shared by the calling thread, and the wait for all of the thread's own
__device__ __forceinline__ void cp_async16(uint32_t dst_smem, const void* src_gmem) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst_smem), "l"(src_gmem) : "memory");
}
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_all;" ::: "memory"); }
__device__ __forceinline__ void fence_async_smem() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }
__device__ __forceinline__ void fence_mbar_init() { asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory"); }

// exp(x) for x <= ~0 (small positive arguments are fine), 0 below the normal range. Argument reduction by ln 2 in
// two pieces, degree-11 Taylor polynomial on |r| <= ln2/2 (truncation ~6e-15 relative), scaling through the exponent.
// Branch-free, so that several independent calls interleave.
__device__ __forceinline__ double exp_reduced(double x) {
    const double t = fma(x, 1.4426950408889634074, 6755399441055744.0);   // round(x / ln 2) in the low word
    const int n = __double2loint(t);
    const double nf = t - 6755399441055744.0;
    double r = fma(nf, -6.93147180369123816490e-01, x);
    r = fma(nf, -1.90821492927058770002e-10, r);
    double p = 2.505210838544172e-08;            // 1/11!
    p = fma(p, r, 2.755731922398589e-07);        // 1/10!
    p = fma(p, r, 2.755731922398589e-06);        // 1/9!
    p = fma(p, r, 2.48015873015873e-05);         // 1/8!
    p = fma(p, r, 1.984126984126984e-04);        // 1/7!
    p = fma(p, r, 1.388888888888889e-03);        // 1/6!
    p = fma(p, r, 8.333333333333333e-03);        // 1/5!
    p = fma(p, r, 4.166666666666666e-02);        // 1/4!
    p = fma(p, r, 1.666666666666667e-01);        // 1/3!
    p = fma(p, r, 0.5);
    p = fma(p, r, 1.0);
    p = fma(p, r, 1.0);
    return p * __hiloint2double((1023 + n) << 20, 0);
}
__device__ __forceinline__ double exp_nonpos(double x0) {
    const double y = exp_reduced(fmax(x0, -708.0));
    return x0 > -708.0 ? y : 0.0;
}
// the caller has seen to the range: exp(x) where `on` holds (which implies x > -708), else 0
__device__ __forceinline__ double exp_nonpos_where(bool on, double x) {
    const double y = exp_reduced(x);
    return on ? y : 0.0;
}

__device__ __forceinline__ void unpack8_to_double(const uint4& raw, double (&kd)[8]) {
    kd[0] = (double)__uint_as_float(raw.x << 16); kd[1] = (double)__uint_as_float(raw.x & 0xffff0000u);
    kd[2] = (double)__uint_as_float(raw.y << 16); kd[3] = (double)__uint_as_float(raw.y & 0xffff0000u);
    kd[4] = (double)__uint_as_float(raw.z << 16); kd[5] = (double)__uint_as_float(raw.z & 0xffff0000u);
    kd[6] = (double)__uint_as_float(raw.w << 16); kd[7] = (double)__uint_as_float(raw.w & 0xffff0000u);
}

}  // namespace corm
