// L2 residency hints.  Per iteration the FP32 path streams the matrix of
// K~ (about 170 MB at n = 373k, read once per product, evict-first loads)
// and re-reads a much smaller set: E^-1 (k^2 floats), the box blocks of
// Z~ and W~ and their row maps.  Loads of that set carry an evict-last L2
// cache policy (PTX createpolicy + ld.global.L2::cache_hint), so it tends to
// survive the matrix stream in the 129 MB L2 from one iteration to the next.
#pragma once

#include <cstdint>

namespace xdcg {

__device__ __forceinline__ uint64_t l2_keep_policy() {
    uint64_t p;
    asm("createpolicy.fractional.L2::evict_last.b64 %0, 1.0;" : "=l"(p));
    return p;
}

__device__ __forceinline__ float ld_keep(const float *a, uint64_t pol) {
    float v;
    asm("ld.global.nc.L2::cache_hint.f32 %0, [%1], %2;" : "=f"(v) : "l"(a), "l"(pol));
    return v;
}

__device__ __forceinline__ int ld_keep(const int *a, uint64_t pol) {
    int v;
    asm("ld.global.nc.L2::cache_hint.s32 %0, [%1], %2;" : "=r"(v) : "l"(a), "l"(pol));
    return v;
}

__device__ __forceinline__ float4 ld_keep(const float4 *a, uint64_t pol) {
    float4 v;
    asm("ld.global.nc.L2::cache_hint.v4.f32 {%0, %1, %2, %3}, [%4], %5;"
        : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w)
        : "l"(a), "l"(pol));
    return v;
}

// What a kernel reads before its wait for the kernel before it (pdl.cuh) and is
// not set-up data: from L2, where everything that a finished kernel wrote is.
// A plain load might find an older line in the SM's L1, since the wait, which
// makes earlier writes visible, has yet to come.  Not moved across the wait.
__device__ __forceinline__ float ld_early(const float *a) {
    float v;
    asm volatile("ld.global.cg.f32 %0, [%1];" : "=f"(v) : "l"(a) : "memory");
    return v;
}

__device__ __forceinline__ double ld_early(const double *a) {
    double v;
    asm volatile("ld.global.cg.f64 %0, [%1];" : "=d"(v) : "l"(a) : "memory");
    return v;
}

// What an earlier kernel of the run wrote, read after the wait: the ordinary
// path through L1.  The read-only path (__ldg, or what the compiler makes of a
// const __restrict__ pointer) is for data that nothing writes while the kernel
// is resident, and a kernel launched early is resident while the one before it
// still writes; nor is such a load held behind the wait.  (No memory clobber: a
// kernel does not write what it reads so.)
__device__ __forceinline__ float ld_dep(const float *a) {
    float v;
    asm volatile("ld.global.f32 %0, [%1];" : "=f"(v) : "l"(a));
    return v;
}
__device__ __forceinline__ double ld_dep(const double *a) {
    double v;
    asm volatile("ld.global.f64 %0, [%1];" : "=d"(v) : "l"(a));
    return v;
}
__device__ __forceinline__ float4 ld_dep(const float4 *a) {
    float4 v;
    asm volatile("ld.global.v4.f32 {%0, %1, %2, %3}, [%4];"
                 : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w)
                 : "l"(a));
    return v;
}
__device__ __forceinline__ double2 ld_dep(const double2 *a) {
    double2 v;
    asm volatile("ld.global.v2.f64 {%0, %1}, [%2];" : "=d"(v.x), "=d"(v.y) : "l"(a));
    return v;
}

// asynchronous 4-byte copy into shared memory with the same policy; a thread
// that reads back only what it copied itself needs no barrier, just the wait
__device__ __forceinline__ void cp_keep(float *smem, const float *a, uint64_t pol) {
    asm volatile("cp.async.ca.shared.global.L2::cache_hint [%0], [%1], 4, %2;" ::"r"(
                     (uint32_t)__cvta_generic_to_shared(smem)),
                 "l"(a), "l"(pol)
                 : "memory");
}
__device__ __forceinline__ void cp_wait_all() {
    asm volatile("cp.async.wait_all;" ::: "memory");
}

}  // namespace xdcg
