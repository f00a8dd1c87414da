// What the stage kernels share in moving tiles: line bases, the walk over a
// tile's values, 8- and 16-byte copies into shared memory, and, for tiles that
// arrive by tensor or bulk copies, the barrier that counts their bytes and the
// bounded wait for it.
#pragma once

#include "p3_internal.h"

namespace p3 {

__device__ __forceinline__ unsigned smem_u32(const void* p) { return (unsigned)__cvta_generic_to_shared(p); }

// Offset (elements) of line L.
__device__ __forceinline__ long long line_base(const LineMap& m, long long L)
{
    if (m.pm) {  // L < 2^31: quotient by multiply-high (line_magic)
        const unsigned u = (unsigned)L;
        const unsigned q = (unsigned)(((unsigned long long)u * m.pm) >> m.ps);
        const unsigned r = u - q * (unsigned)m.per;
        return (long long)q * m.gstride + (long long)r * m.lstride;
    }
    return (L / m.per) * m.gstride + (L % m.per) * m.lstride;
}

// Calls f(l, e) for every value of a tile of `rows` lines of `len` values,
// threads walking the values together; the loop unrolled UNROLL times.
template <int UNROLL, class F> __device__ __forceinline__ void walk(int rows, int len, F f)
{
    const int NT = blockDim.x, tid = threadIdx.x;
    int l = tid / len, e = tid - l * len;
    const int dq = NT / len, dr = NT - dq * len;
#pragma unroll UNROLL
    while (l < rows) {
        f(l, e);
        e += dr;
        l += dq;
        if (e >= len) {
            e -= len;
            ++l;
        }
    }
}

__device__ __forceinline__ void cp_async16(unsigned d, const void* g)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(d), "l"(g) : "memory");
}
__device__ __forceinline__ void cp_async8(unsigned d, const void* g)
{
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;\n" ::"r"(d), "l"(g) : "memory");
}
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_all;\n" ::: "memory"); }

__device__ __forceinline__ bool mbar_try_wait(unsigned bar, unsigned parity)
{
    unsigned done;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(done)
        : "r"(bar), "r"(parity)
        : "memory");
    return done != 0;
}

// Copy barrier of a tile: arrival count 1, or 2 in the test mode of
// StageArgs::wait_extra (one arrival never comes, so the wait runs out).
__device__ __forceinline__ void copy_bar_init(unsigned bar, int extra)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;\n" ::"r"(bar), "r"(extra ? 2 : 1) : "memory");
    asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
}

// Every thread waits (at most a.spin polls) for the tile's copies; true when
// all threads saw them land.  Otherwise bit 2 of *a.err is set, the missing
// test-mode arrival is supplied, and the CTA waits (again bounded) for the
// copies still in flight into its shared memory before the caller leaves.
__device__ __forceinline__ bool copy_bar_wait(const StageArgs& a, unsigned bar)
{
    int ok = 0;
    for (unsigned it = 0; it < a.spin; ++it)
        if (mbar_try_wait(bar, 0)) {
            ok = 1;
            break;
        }
    if (__syncthreads_and(ok)) return true;
    if (threadIdx.x == 0) {
        atomicOr(a.err, 2u);
        if (a.wait_extra) asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];\n" ::"r"(bar) : "memory");
    }
    __syncthreads();
    for (unsigned it = 0; it < a.spin && !mbar_try_wait(bar, 0); ++it) {
    }
    return false;
}

// One thread: the barrier expects `bytes` of copies.
__device__ __forceinline__ void copy_bar_expect(unsigned bar, unsigned bytes)
{
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;\n" ::"r"(bar), "r"(bytes) : "memory");
}
// One thread: `bytes` (a multiple of 16) from global g to shared address d, both 16-byte aligned.
__device__ __forceinline__ void copy_bulk(unsigned d, const void* g, unsigned bytes, unsigned bar)
{
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];\n" ::"r"(d), "l"(g),
                 "r"(bytes), "r"(bar)
                 : "memory");
}

}  // namespace p3
