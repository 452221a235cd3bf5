// Device helpers shared by the tensor-core X-engines (xeng_tc.cu, xeng_pair.cu):
// mbarriers with bounded waits, TMA, tcgen05 and the decoding of packed samples.
#pragma once

#include <cuda.h>

#include "internal.cuh"

namespace corr {
namespace {

// ------------------------------------------------------------ PTX helpers --
__device__ __forceinline__ uint32_t smem_u32(const void *p)
{
    return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count));
}

__device__ __forceinline__ void mbar_arrive(uint32_t bar)
{
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}

__device__ __forceinline__ void mbar_expect_tx(uint32_t bar, uint32_t bytes)
{
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes)
                 : "memory");
}

__device__ __forceinline__ bool mbar_try(uint32_t bar, uint32_t parity)
{
    uint32_t done;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n"
        " selp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(done)
        : "r"(bar), "r"(parity)
        : "memory");
    return done != 0;
}

// As mbar_try, but a thread whose phase is not complete may be suspended for
// up to 1 ms (it resumes as soon as the phase completes), so bounded waits
// poll rarely instead of spinning.
__device__ __forceinline__ bool mbar_try_sleep(uint32_t bar, uint32_t parity)
{
    uint32_t done;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %3;\n"
        " selp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(done)
        : "r"(bar), "r"(parity), "n"(1000000)
        : "memory");
    return done != 0;
}

// Bounded wait.  Returns false on timeout or if another role aborted.
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity, volatile int *abort,
                                          DeviceStatus *status, int where, long long limit)
{
    if (mbar_try(bar, parity)) return true;
    const long long t0 = clock64();
    while (true) {
        // the checks cost issue slots that the working warps want: a few tries between them
#pragma unroll
        for (int k = 0; k < 4; ++k)
            if (mbar_try_sleep(bar, parity)) return true;
        if (*abort) return false;
        if (clock64() - t0 > limit) {
            *abort = 1;
            if (atomicCAS(&status->code, 0, CORR_E_TIMEOUT) == 0) {
                status->where = where;
                status->detail0 = int(blockIdx.x);
            }
            return false;
        }
    }
}

// Warp-wide bounded wait: lane 0 polls (with an optional back-off), then every
// lane confirms once, so each lane gets the barrier's acquire ordering while
// only one lane keeps hitting shared memory.
__device__ __forceinline__ bool warp_wait(uint32_t bar, uint32_t parity, volatile int *abort,
                                          DeviceStatus *status, int where, int lane, long long limit,
                                          unsigned sleep_ns = 0)
{
    int ok = 1;
    if (lane == 0) {
        if (!mbar_try(bar, parity)) {
            const long long t0 = clock64();
            while (true) {
                if (mbar_try(bar, parity)) break;
                if (*abort) {
                    ok = 0;
                    break;
                }
                if (clock64() - t0 > limit) {
                    *abort = 1;
                    if (atomicCAS(&status->code, 0, CORR_E_TIMEOUT) == 0) {
                        status->where = where;
                        status->detail0 = int(blockIdx.x);
                    }
                    ok = 0;
                    break;
                }
                if (sleep_ns) __nanosleep(sleep_ns);
            }
        }
    }
    ok = __shfl_sync(0xFFFFFFFFu, ok, 0);
    if (!ok) return false;
    return mbar_try(bar, parity);        // completed: returns at once, with acquire
}

// index of input n (0..127) in a row of per-input sums: [n % 16][n / 16], so
// that the eight lanes adding sums of the same offset within their 16-input
// chunk hit eight consecutive words (no bank conflicts)
__device__ __forceinline__ int sum_slot(int n) { return (n & 15) * 8 + (n >> 4); }

__device__ __forceinline__ void tma_load_3d(uint32_t dst, const CUtensorMap *map, uint32_t bar,
                                            int x, int y, int z)
{
    asm volatile(
        "cp.async.bulk.tensor.3d.shared::cluster.global.tile.mbarrier::complete_tx::bytes"
        " [%0], [%1, {%2, %3, %4}], [%5];" ::"r"(dst),
        "l"(reinterpret_cast<uint64_t>(map)), "r"(x), "r"(y), "r"(z), "r"(bar)
        : "memory");
}

__device__ __forceinline__ void tma_prefetch_3d(const CUtensorMap *map, int x, int y, int z)
{
    asm volatile("cp.async.bulk.prefetch.tensor.3d.L2.global.tile [%0, {%1, %2, %3}];" ::"l"(
                     reinterpret_cast<uint64_t>(map)),
                 "r"(x), "r"(y), "r"(z)
                 : "memory");
}

__device__ __forceinline__ uint64_t smem_desc(uint32_t saddr, uint32_t lbo, uint32_t sbo)
{
    uint64_t d = 0;
    d |= uint64_t((saddr >> 4) & 0x3FFFu);
    d |= uint64_t((lbo >> 4) & 0x3FFFu) << 16;
    d |= uint64_t((sbo >> 4) & 0x3FFFu) << 32;
    d |= uint64_t(1) << 46;                     // descriptor version
    d |= uint64_t(2) << 61;                     // 128-byte swizzle
    return d;
}

template <uint32_t kIdesc>
__device__ __forceinline__ void mma_f8(uint32_t tmem, uint64_t a, uint64_t b, uint32_t accum)
{
    asm volatile(
        "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
        " tcgen05.mma.cta_group::1.kind::f8f6f4 [%0], %1, %2, %3, p;\n}\n" ::"r"(tmem),
        "l"(a), "l"(b), "r"(kIdesc), "r"(accum));
}

__device__ __forceinline__ void mma_commit(uint32_t bar)
{
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar)
                 : "memory");
}

__device__ __forceinline__ void fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

__device__ __forceinline__ void tmem_ld8(uint32_t taddr, uint32_t (&r)[8])
{
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];\n"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
                   "=r"(r[7])
                 : "r"(taddr));
}

__device__ __forceinline__ void tmem_wait_ld() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }

__device__ __forceinline__ void named_sync(int id, int threads)
{
    asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(threads) : "memory");
}

// 256 (r^2 + m^2) summed over the 4 packed samples of w, plus acc: the high
// nibble with the low one cleared is the signed byte 16 r, the low nibble
// moved up the signed byte 16 m (Appendix A: two's complement, real high).
// With zero_invalid, samples with a nibble of 8 count as zero.
__device__ __forceinline__ int power256(uint32_t w, bool zero_invalid, int acc)
{
    uint32_t hr = w & 0xF0F0F0F0u, hm = (w << 4) & 0xF0F0F0F0u;
    if (zero_invalid) {
        const uint32_t bad = __vcmpeq4(hr, 0x80808080u) | __vcmpeq4(hm, 0x80808080u);
        hr &= ~bad;
        hm &= ~bad;
    }
    return __dp4a(int(hm), int(hm), __dp4a(int(hr), int(hr), acc));
}

// 4 packed bytes (r << 4 | m) -> E4M3 codes u = nibble ^ 8 (value u * 2^-9).
__device__ __forceinline__ void codes(uint32_t w, bool zero_invalid, uint32_t &R, uint32_t &M)
{
    R = ((w >> 4) & 0x0F0F0F0Fu) ^ 0x08080808u;
    M = (w & 0x0F0F0F0Fu) ^ 0x08080808u;
    if (zero_invalid) {
        // a nibble code of 8 (value -8) has u == 0: such samples become 0 + 0i (u = 8, 8)
        const uint32_t nzR = (R + 0x7F7F7F7Fu) & 0x80808080u;   // bit 7 set where u != 0
        const uint32_t nzM = (M + 0x7F7F7F7Fu) & 0x80808080u;
        const uint32_t bad = (~(nzR & nzM)) & 0x80808080u;      // bit 7 set where invalid
        const uint32_t mask = (bad >> 7) * 0xFFu;
        R = (R & ~mask) | (0x08080808u & mask);
        M = (M & ~mask) | (0x08080808u & mask);
    }
}

}  // namespace

// One launch of the CTA-pair X-engine (xeng_pair.cu) over every channel of up
// to kTcMaxArrays arrays of 129 to 256 inputs.
cudaError_t launch_xeng_pair(const TcArray *arrays, int count, bool zero_invalid, int dev, DeviceStatus *status,
                             const TcOptions &opt, cudaStream_t s);

}  // namespace corr
