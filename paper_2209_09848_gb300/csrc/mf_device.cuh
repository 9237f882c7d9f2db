// Device helpers shared by the numerator kernels: mbarriers, TMA and bulk
// copies (inline PTX for sm_103a), and the packed (SNR, k) key.
#pragma once

#include <cuda.h>
#include <cuda_runtime.h>

#include <cstdint>

namespace mf {
namespace dev {

constexpr long long kWaitCycles = 1ll << 31;  // about one second at 2 GHz

__device__ __forceinline__ uint32_t smem_u32(const void *p) {
    return (uint32_t)__cvta_generic_to_shared(p);
}

__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}

__device__ __forceinline__ void mbar_expect_tx(uint32_t bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}

__device__ __forceinline__ bool mbar_try_wait(uint32_t bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(bar), "r"(parity)
        : "memory");
    return ok != 0;
}

// Non-blocking check of a phase (acquire on success).
__device__ __forceinline__ bool mbar_test_wait(uint32_t bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(bar), "r"(parity)
        : "memory");
    return ok != 0;
}

__device__ __forceinline__ int status_now(const int *status) { return *(const volatile int *)status; }

// Wait for a phase of an mbarrier, giving up after kWaitCycles or as soon as
// another CTA has recorded a failure in the device status word; on giving up
// the status word records `code` (if nothing was recorded before).
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity, int code, int *status) {
    if (mbar_try_wait(bar, parity)) return true;
    const long long t0 = clock64();
    for (unsigned it = 1;; it++) {
        if (mbar_try_wait(bar, parity)) return true;
        if ((it & 255u) == 0 && status_now(status) != 0) return false;
        if (clock64() - t0 > kWaitCycles) {
            atomicCAS(status, 0, code);
            return false;
        }
    }
}

__device__ __forceinline__ void mbar_inval(uint32_t bar) {
    asm volatile("mbarrier.inval.shared::cta.b64 [%0];" ::"r"(bar) : "memory");
}

__device__ __forceinline__ void fence_barrier_init() {
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}

__device__ __forceinline__ void fence_proxy_async() {
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}

__device__ __forceinline__ void tma_load_3d(uint32_t dst, const CUtensorMap *map, int x, int y, int z,
                                            uint32_t bar) {
    asm volatile(
        "cp.async.bulk.tensor.3d.shared::cluster.global.tile.mbarrier::complete_tx::bytes"
        " [%0], [%1, {%2, %3, %4}], [%5];" ::"r"(dst),
        "l"(map), "r"(x), "r"(y), "r"(z), "r"(bar)
        : "memory");
}

__device__ __forceinline__ void bulk_load(uint32_t dst, const void *src, uint32_t bytes, uint32_t bar) {
    asm volatile(
        "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst),
        "l"(src), "r"(bytes), "r"(bar)
        : "memory");
}

// Programmatic dependent launches: a kernel lets the next one in its stream
// start once all its CTAs have (or have ended), and a kernel waits for the one
// before it to have completed, with everything it wrote.  Without that launch
// attribute both do nothing.  Two reads of a search come without a wait of
// their own: lambda in k_den_box and the weighted stack in a factored
// numerator's later segments (see enqueue_den and start_early).
__device__ __forceinline__ void launch_dependents() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void wait_previous() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// Loads of what the awaited kernel wrote: from L2 (a line that an earlier CTA
// of this SM cached may be older), and in program order with the wait, which
// loads through const __restrict__ pointers need not be.
__device__ __forceinline__ void load_awaited(float &v, const float *p) {
    asm volatile("ld.global.cg.f32 %0, [%1];" : "=f"(v) : "l"(p));
}
__device__ __forceinline__ void load_awaited(float4 &v, const float4 *p) {
    asm volatile("ld.global.cg.v4.f32 {%0, %1, %2, %3}, [%4];"
                 : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w)
                 : "l"(p));
}

// Order-preserving 64-bit key: larger SNR first, then smaller k.  Any valid
// key is nonzero, so 0 means "no filter with D > 0".
__device__ __forceinline__ unsigned long long pack_key(float snr, int k) {
    uint32_t b = __float_as_uint(snr);
    b = (b & 0x80000000u) ? ~b : (b | 0x80000000u);
    return ((unsigned long long)b << 32) | (unsigned long long)(0xFFFFFFFFu - (uint32_t)k);
}

// Selection key: larger score first, then smaller index; unique per index.
__device__ __forceinline__ unsigned long long sel_key(float score, uint32_t i) {
    uint32_t b = __float_as_uint(score);
    b = (b & 0x80000000u) ? ~b : (b | 0x80000000u);
    return ((unsigned long long)b << 32) | (unsigned long long)(0xFFFFFFFFu - i);
}

// An FP32 value as FP64, by its bits: a conversion instruction costs an FP64
// operation (1/64 of the FP32 rate on this GPU).  Exact for every value:
// subnormals are scaled by 2^64 first, infinities and NaN keep their exponent.
__device__ __forceinline__ double widen(float v) {
    const uint32_t b = __float_as_uint(v), m = b & 0x7FFFFFFFu;
    const bool small = m < 0x00800000u;
    const uint32_t n = small ? __float_as_uint(__uint_as_float(m) * 18446744073709551616.f) : m;
    const uint32_t off = small ? 0x38000000u - (64u << 20) : (m >= 0x7F800000u ? 0x70000000u : 0x38000000u);
    const uint32_t hi = n ? (n >> 3) + off : 0u;
    return __hiloint2double((int)(hi | (b & 0x80000000u)), (int)(n << 29));
}

}  // namespace dev
}  // namespace mf
