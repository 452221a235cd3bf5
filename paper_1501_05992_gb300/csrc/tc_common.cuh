// Device helpers shared by the tensor-core X-engines (xeng_diag.cuh, xeng_off.cuh):
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

// Limit of the waits for copies and MMAs in flight before their memory is given up (a
// parameter of the launches, Params::drain_limit).  They end whatever the roles' waits came
// to, so these waits don't take the caller's limit, which may be shorter than they need.
constexpr long long kDefaultWaitLimit = 1LL << 31;

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

__device__ __forceinline__ void mma_f8(uint32_t tmem, uint64_t a, uint64_t b, uint32_t idesc, uint32_t accum)
{
    asm volatile(
        "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
        " tcgen05.mma.cta_group::1.kind::f8f6f4 [%0], %1, %2, %3, p;\n}\n" ::"r"(tmem),
        "l"(a), "l"(b), "r"(idesc), "r"(accum));
}

__device__ __forceinline__ void mma_commit(uint32_t bar)
{
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar)
                 : "memory");
}

__device__ __forceinline__ void fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

__device__ __forceinline__ void tmem_wait_ld() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }

__device__ __forceinline__ void named_sync(int id, int threads)
{
    asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(threads) : "memory");
}

__device__ __forceinline__ void tmem_ld16(uint32_t taddr, uint32_t (&r)[16])
{
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];\n"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
          "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(taddr));
}

// Rows ic .. ic + 15 of a channel's packed triangle at out_f, column j (this
// lane's; a warp's 32 columns are consecutive): v[k] = (Re, Im) of row ic + k,
// stored (kFresh) or added, where ic + k < n and j <= ic + k; `full`: everywhere,
// for the whole warp.
template <bool kFresh>
__device__ __forceinline__ void put_rows16(uint8_t *out_f, int ic, int j, int n, int lane, bool full,
                                           const int2 (&v)[16])
{
    // byte offset of element (ic, j), < 2^32
    uint32_t off = (unsigned(ic) * unsigned(ic + 1) / 2u + unsigned(j)) * 8u;
    if (!kFresh && full) {
        // the integer adds are done in L2 (red).  The warp's halves trade Im and Re of 16
        // columns each, so that an instruction adds to 128 contiguous bytes (4 whole
        // sectors; lanes 0-15 Re, 16-31 Im) instead of every other word of 256: 0.46 ->
        // 0.42 ms per 500 samples added to the full band's triangle (256 inputs)
        const bool low = lane < 16;
        off += low ? 0u : 4u - 128u;
#pragma unroll
        for (int k = 0; k < 16; ++k) {
            const int other = __shfl_xor_sync(0xFFFFFFFFu, low ? v[k].y : v[k].x, 16);
            asm volatile("red.global.add.s32 [%0], %1;" ::"l"(out_f + off), "r"(low ? v[k].x : other) : "memory");
            asm volatile("red.global.add.s32 [%0+128], %1;" ::"l"(out_f + off), "r"(low ? other : v[k].y) : "memory");
            off += unsigned(ic + k + 1) * 8u;
        }
    } else if (!kFresh) {
#pragma unroll
        for (int k = 0; k < 16; ++k) {
            if (ic + k < n && j <= ic + k) {
                asm volatile("red.global.add.s32 [%0], %1;" ::"l"(out_f + off), "r"(v[k].x) : "memory");
                asm volatile("red.global.add.s32 [%0+4], %1;" ::"l"(out_f + off), "r"(v[k].y) : "memory");
            }
            off += unsigned(ic + k + 1) * 8u;
        }
    } else if (full) {
#pragma unroll
        for (int k = 0; k < 16; ++k) {
            *reinterpret_cast<int2 *>(out_f + off) = v[k];
            off += unsigned(ic + k + 1) * 8u;
        }
    } else {
#pragma unroll
        for (int k = 0; k < 16; ++k) {
            if (ic + k < n && j <= ic + k) *reinterpret_cast<int2 *>(out_f + off) = v[k];
            off += unsigned(ic + k + 1) * 8u;
        }
    }
}

// ------------------------------------------------- CTA pairs (cta_group::2) --
// instruction descriptor: kind::f8f6f4, E4M3 x E4M3 -> F32, both MN-major, M=256, N=256
constexpr uint32_t kIdescPair = (1u << 4) | (1u << 15) | (1u << 16) | ((256u >> 3) << 17) | ((256u >> 4) << 24);

__device__ __forceinline__ uint32_t cluster_rank()
{
    uint32_t r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}

__device__ __forceinline__ void cluster_sync()
{
    asm volatile("barrier.cluster.arrive.release;\n barrier.cluster.wait.acquire;" ::: "memory");
}

// address of `addr` (an address in this CTA's shared memory) in CTA `rank`
__device__ __forceinline__ uint32_t map_rank(uint32_t addr, uint32_t rank)
{
    uint32_t r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
    return r;
}

// Arrival on a barrier of either CTA.  The hand-overs are ordered by the proxy
// and tcgen05 fences before them (or follow reads only), so they use the default
// (CTA) scope: a release at cluster scope waits for every earlier write of the
// thread, about 1000 cycles per stage (2.30 against 1.57 ms on the full band).
__device__ __forceinline__ void remote_arrive(uint32_t bar)
{
    asm volatile("mbarrier.arrive.shared::cluster.b64 _, [%0];" ::"r"(bar) : "memory");
}

// Stores to the other CTA's shared memory that count their bytes on its barrier.
__device__ __forceinline__ void store_async(uint32_t addr, uint32_t v, uint32_t bar)
{
    asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.b32 [%0], %1, [%2];" ::"r"(addr), "r"(v),
                 "r"(bar)
                 : "memory");
}

__device__ __forceinline__ void store_async4(uint32_t addr, const uint32_t *v, uint32_t bar)
{
    asm volatile("st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.v4.b32 [%0], {%1, %2, %3, %4}, [%5];" ::"r"(
                     addr),
                 "r"(v[0]), "r"(v[1]), "r"(v[2]), "r"(v[3]), "r"(bar)
                 : "memory");
}

__device__ __forceinline__ void store_peer(uint32_t addr, int v)
{
    asm volatile("st.shared::cluster.u32 [%0], %1;" ::"r"(addr), "r"(v) : "memory");
}

__device__ __forceinline__ bool mbar_try_cluster(uint32_t bar, uint32_t parity)
{
    uint32_t done;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2, %3;\n"
        " selp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(done)
        : "r"(bar), "r"(parity), "n"(1000000)
        : "memory");
    return done != 0;
}

// Bounded wait (of a whole warp) on a barrier that the other CTA completes.
__device__ __forceinline__ bool cluster_wait(uint32_t bar, uint32_t parity, volatile int *abort, DeviceStatus *status,
                                             int where, long long limit)
{
    const long long t0 = clock64();
    while (true) {
#pragma unroll
        for (int k = 0; k < 4; ++k)
            if (mbar_try_cluster(bar, parity)) return true;
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

__device__ __forceinline__ void mma_f8_pair(uint32_t tmem, uint64_t a, uint64_t b, uint32_t accum)
{
    asm volatile(
        "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
        " tcgen05.mma.cta_group::2.kind::f8f6f4 [%0], %1, %2, %3, p;\n}\n" ::"r"(tmem),
        "l"(a), "l"(b), "r"(kIdescPair), "r"(accum));
}

// arrives on the barrier at this offset in both CTAs once the MMAs issued so far are done
__device__ __forceinline__ void commit_both(uint32_t bar)
{
    asm volatile(
        "tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;" ::"r"(bar),
        "h"((uint16_t)3)
        : "memory");
}

__device__ __forceinline__ void commit_own(uint32_t bar)
{
    asm volatile("tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}

// a * b + c as one multiply-add (the FMA pipe).  b is a kernel parameter, so that
// the compiler cannot turn it back into an add or a shift: the ALU pipe takes one
// warp instruction per two cycles, the FMA pipe beside it another, and this
// spreads the converters over both (1.35 -> 1.31 ms with the decoding's other
// instructions cut from 17 to 14 per word).
__device__ __forceinline__ uint32_t imad(uint32_t a, uint32_t b, uint32_t c)
{
    uint32_t d;
    asm("mad.lo.u32 %0, %1, %2, %3;" : "=r"(d) : "r"(a), "r"(b), "r"(c));
    return d;
}

// TMEM allocation by one warp (kPair: of both CTAs of a pair); the address goes to `slot`.
template <bool kPair>
__device__ __forceinline__ void tmem_alloc(uint32_t slot, uint32_t cols)
{
    if (kPair) {
        asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(slot), "r"(cols));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;");
    } else {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(slot), "r"(cols));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
}

template <bool kPair>
__device__ __forceinline__ void tmem_dealloc(uint32_t tmem, uint32_t cols)
{
    if (kPair)
        asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(cols));
    else
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(cols));
}

}  // namespace

// One launch over every channel of up to kTcMaxArrays arrays, storing (fresh) or
// adding: the 256-input blocks on the diagonal (arrays of 129 or more inputs), and
// the last tile of an odd number of 128-input tiles.  `overlap`: the launch may start
// while the one before it on the stream, also one of these, still runs.
cudaError_t launch_xeng_pair(const TcArray *arrays, int count, bool fresh, bool zero_invalid, int dev,
                             DeviceStatus *status, const TcOptions &opt, bool overlap, cudaStream_t s);
cudaError_t launch_xeng_tile(const TcArray *arrays, int count, bool fresh, bool zero_invalid, int dev,
                             DeviceStatus *status, const TcOptions &opt, bool overlap, cudaStream_t s);
// The rest of their triangles (xeng_off.cuh), for arrays of 257 or more inputs;
// maps[k] is array k's tensor map (boxes of 128 inputs x 1 channel x 64 samples).
cudaError_t launch_xeng_off(const TcArray *arrays, const CUtensorMap *maps, int count, bool fresh, bool zero_invalid,
                            int dev, DeviceStatus *status, const TcOptions &opt, bool overlap, cudaStream_t s);
// Both for one array, on pairs of CTAs of their own each.
cudaError_t launch_xeng_both(const TcArray &A, const CUtensorMap &map, int block_pairs, int off_pairs, bool fresh,
                             bool zero_invalid, int dev, DeviceStatus *status, const TcOptions &opt, bool overlap,
                             cudaStream_t s);

}  // namespace corr
