// Packet ingest: one 50 ms bank of PFB packets (Appendix A, "Data Format")
// into the assembled voltage block the X-engine reads (Appendix B: each
// packet's input order kept, the four PFBs concatenated; Appendix C "GPU
// Input": time, channel, input).
//
// Packet: 264 bytes = header word 0x0800, word two (sec_tick bit 0, pfb_id
// bits 4-5, mgt_id bits 6-8, mgt_bank bits 9-13), word three (mgt_frame bits
// 0-8, mgt_group bits 9-10, mgt_channel bits 11-15), 256 sample bytes (byte
// 64 f2 + k: fine channel 128 mgt_channel + 16 mgt_id + 4 mgt_group + f2,
// input 64 pfb_id + k), and the XOR of the 128 data words; 16-bit words most
// significant byte first.
//
// A warp takes two groups of four packets, eight lanes to a packet.  Both groups are on
// their way into shared memory at once (cp.async in the widest pieces that the stream's
// alignment allows), and a warp waits for nothing but its own copies.  Lane j owns
// the packet's sample bytes 16 j .. 16 j + 15 and those 128 further: it realigns them (the data
// start at byte 6), XOR-reduces over the packet's lanes against the checksum, decodes the
// header, and stores two 16-byte pieces; the lanes of one store fill the 64-byte runs of
// two channels.  A slot is marked filled with a plain one-byte store (no value comes
// back, so no lane waits on it).  A last pass, a lane per (frame, group of four
// channels) reading the four PFBs' marks as one word, writes the slots no good packet
// filled with 0x88, the appendix's invalid code (CORR_ZERO_INVALID turns it into zeros),
// and counts them, the whole warp storing a group's bytes; the repeats are the good
// packets minus the distinct filled slots, added up in the same pass.  The three launches
// overlap: the packets are on their way while the marks are still being cleared.
//
// What bounds it: HBM, whose writes come in runs of 64 bytes spread over the block.  A whole
// bank (799 MB read and written, 117 us at the measured copy rate) takes 125 us in the
// receiver's order and 146 us shuffled; with nine-word loads into registers, one group
// ahead, and 16-byte stores of every other 16 bytes, 158 and 164 us.  Blocks take
// neighbouring stretches of the stream, so that the four PFBs' parts of a row meet in
// L2: 130 us with each warp's groups a grid apart, 127 us with three groups and 133
// with eight per warp, 131 us with blocks of four warps.
#include "internal.cuh"

namespace corr {
namespace {

constexpr int kFrames = CORR_PKT_FRAMES, kChannels = CORR_PKT_CHANNELS, kInputs = CORR_PKT_INPUTS;
constexpr int kGroups = kChannels / 4;
constexpr int kIngestThreads = 256, kIngestWarps = kIngestThreads / 32;
constexpr int kIngestBlocks = 6;                         // per SM
constexpr int kPackets = 4;                              // packets of a warp's group
constexpr int kGroupBytes = kPackets * CORR_PKT_BYTES;   // 1056
constexpr int kRounds = 2;                               // groups a warp takes (the waits below know it)
constexpr int kBlockPackets = kRounds * kIngestWarps * kPackets;
static_assert(kRounds == 2 && kGroupBytes % 16 == 0, "a group starts where the stream's alignment holds");

__device__ __forceinline__ unsigned be16(uint32_t w, int byte)   // big-endian 16-bit word at byte 0 or 2
{
    return ((w >> (8 * byte)) & 0xFFu) << 8 | ((w >> (8 * byte + 8)) & 0xFFu);
}

// kBytes (16, 8 or 4) of global memory, of which the first n are there, to shared memory
template <int kBytes>
__device__ __forceinline__ void copy_async(uint32_t dst, const uint8_t *src, int n)
{
    if (kBytes == 16)
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(n) : "memory");
    else
        asm volatile("cp.async.ca.shared.global [%0], [%1], %2, %3;" ::"r"(dst), "l"(src), "n"(kBytes), "r"(n)
                     : "memory");
}

// kBytes: alignment of the stream (16, 8 or 4), the size of its pieces.
template <int kBytes>
__global__ void __launch_bounds__(kIngestThreads, kIngestBlocks)
ingest_kernel(const uint8_t *__restrict__ packets, long long n_packets, int bank, uint8_t *__restrict__ volt,
              uint8_t *__restrict__ seen, int *__restrict__ counters)
{
    __shared__ __align__(16) uint8_t groups[kIngestWarps][kRounds][kGroupBytes];
    __shared__ int block_counts[CORR_PKT_COUNTERS];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, sub = lane >> 3, j = lane & 7;
    let_next_launch_start();
    if (threadIdx.x < CORR_PKT_COUNTERS) block_counts[threadIdx.x] = 0;
    __syncthreads();
    // this warp's groups lie a block's warps apart, all on their way at once
    const long long total = n_packets * CORR_PKT_BYTES;
    const long long first = (blockIdx.x * (long long)(kRounds * kIngestWarps) + warp) * kGroupBytes;
#pragma unroll
    for (int k = 0; k < kRounds; ++k) {
        const long long at = first + k * (kIngestWarps * kGroupBytes);
        const uint32_t dst = uint32_t(__cvta_generic_to_shared(groups[warp][k]));
#pragma unroll
        for (int c = lane * kBytes; c < kGroupBytes; c += 32 * kBytes) {
            const long long left = total - at - c;
            if (left > 0) copy_async<kBytes>(dst + c, packets + at + c, left < kBytes ? int(left) : kBytes);
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
    }
    wait_for_launch_before();                            // the marks and counters are clear
    int good = 0;
#pragma unroll
    for (int k = 0; k < kRounds; ++k) {
        const long long at = first + k * (kIngestWarps * kGroupBytes);
        if (at >= total) break;                          // the whole warp (the shuffles below take all lanes)
        if (k + 1 < kRounds) asm volatile("cp.async.wait_group 1;" ::: "memory");
        else asm volatile("cp.async.wait_group 0;" ::: "memory");
        __syncwarp();
        const uint8_t *const pk = groups[warp][k] + sub * CORR_PKT_BYTES;
        // data word l (bytes 6 + 4 l ..) from packet words l + 1 and l + 2; this lane's
        // are 4 j .. 4 j + 3 and 32 more
        uint4 d[2];
        uint32_t x = 0;
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const uint2 *const w = reinterpret_cast<const uint2 *>(pk + 16 * j + 128 * h);
            const uint2 a = w[0], b = w[1], c = w[2];
            d[h] = make_uint4(__byte_perm(a.y, b.x, 0x5432), __byte_perm(b.x, b.y, 0x5432),
                              __byte_perm(b.y, c.x, 0x5432), __byte_perm(c.x, c.y, 0x5432));
            x ^= d[h].x ^ d[h].y ^ d[h].z ^ d[h].w;
        }
        const uint2 w01 = *reinterpret_cast<const uint2 *>(pk);
        const uint32_t w65 = *reinterpret_cast<const uint32_t *>(pk + CORR_PKT_BYTES - 4);
#pragma unroll
        for (int o = 4; o > 0; o >>= 1) x ^= __shfl_xor_sync(0xFFFFFFFFu, x, o);
        if (at + sub * CORR_PKT_BYTES < total) {
            // even packet bytes are the words' high bytes: data bytes 0 and 2 of each group of four
            const unsigned xhi = (x ^ (x >> 16)) & 0xFFu, xlo = ((x >> 8) ^ (x >> 24)) & 0xFFu;
            const unsigned header = be16(w01.x, 0), word2 = be16(w01.x, 2), word3 = be16(w01.y, 0);
            const unsigned ck_hi = (w65 >> 16) & 0xFFu, ck_lo = (w65 >> 24) & 0xFFu;
            const int tick = int(word2 & 1u), pfb = int((word2 >> 4) & 3u), mgt = int((word2 >> 6) & 7u);
            const int bnk = int((word2 >> 9) & 31u);
            const int frame = int(word3 & 511u), grp = int((word3 >> 9) & 3u), chan = int((word3 >> 11) & 31u);
            int code = CORR_PKT_GOOD;
            if (header != 0x0800u) code = CORR_PKT_BAD_HEADER;
            else if (xhi != ck_hi || xlo != ck_lo) code = CORR_PKT_BAD_CHECKSUM;
            else if (bnk != bank || chan >= 24 || frame >= kFrames ||
                     (tick && (bnk | chan | grp | frame) != 0))
                code = CORR_PKT_BAD_FIELD;
            if (code == CORR_PKT_GOOD) {
                const int cgroup = 32 * chan + 4 * mgt + grp;
                if (j == 0) {
                    seen[(frame * kGroups + cgroup) * 4 + pfb] = 1;
                    ++good;
                }
                // sample bytes 16 j ..: channel j / 4, inputs 64 pfb + 16 (j % 4) ..; 128 more: two channels on
                uint8_t *const o =
                    volt + ((long long)frame * kChannels + 4 * cgroup + (j >> 2)) * kInputs + 64 * pfb + 16 * (j & 3);
                *reinterpret_cast<uint4 *>(o) = d[0];
                *reinterpret_cast<uint4 *>(o + 2 * kInputs) = d[1];
            } else if (j == 0) {
                atomicAdd(block_counts + code, 1);
            }
        }
    }
    if (good) atomicAdd(block_counts + CORR_PKT_GOOD, good);
    __syncthreads();
    if (threadIdx.x < CORR_PKT_COUNTERS && block_counts[threadIdx.x])
        atomicAdd(counters + threadIdx.x, block_counts[threadIdx.x]);
}

// One lane per (frame, group of four channels): its four slots (one per PFB) are
// the four mark bytes of one word.  A group with a slot that nobody filled is taken by
// the whole warp: lane l holds bytes 16 (l % 16) .. of channels l / 16 and l / 16 + 2, and
// writes 0x88 where its PFB's mark is missing (a bank nothing of which arrived: 235 us
// with a lane writing a group's runs by itself, 64 us so).
__global__ void __launch_bounds__(kIngestThreads)
ingest_missing_kernel(uint8_t *__restrict__ volt, const uint32_t *__restrict__ seen4, int *__restrict__ counters)
{
    wait_for_launch_before();
    int missing = 0;
    const int lane = threadIdx.x & 31;
    for (int base = (blockIdx.x * kIngestThreads + threadIdx.x) & ~31; base < CORR_PKT_SLOTS / 4;
         base += gridDim.x * kIngestThreads) {
        const uint32_t marks = base + lane < CORR_PKT_SLOTS / 4 ? seen4[base + lane] : 0x01010101u;
        unsigned todo = __ballot_sync(0xFFFFFFFFu, !(marks & 0x000000FFu) || !(marks & 0x0000FF00u) ||
                                                       !(marks & 0x00FF0000u) || !(marks & 0xFF000000u));
        while (todo) {
            const int l = __ffs(todo) - 1;
            todo &= todo - 1;
            const uint32_t m = __shfl_sync(0xFFFFFFFFu, marks, l);
            const int fg = base + l;                     // frame * kGroups + channel group
            if (!((m >> (8 * ((lane & 15) >> 2))) & 0xFFu)) {
                const uint4 inv = make_uint4(0x88888888u, 0x88888888u, 0x88888888u, 0x88888888u);
                uint8_t *const o = volt + ((long long)fg * 4 + (lane >> 4)) * kInputs + 16 * (lane & 15);
                *reinterpret_cast<uint4 *>(o) = inv;
                *reinterpret_cast<uint4 *>(o + 2 * kInputs) = inv;
                missing += (lane & 19) == 0;             // one lane per slot
            }
        }
    }
    __shared__ int block_missing;
    if (threadIdx.x == 0) block_missing = 0;
    __syncthreads();
    if (missing) atomicAdd(&block_missing, missing);
    __syncthreads();
    // repeats = good packets - distinct filled slots = GOOD - (SLOTS - MISSING):
    // every block adds its missing slots to both counters, and block 0 adds
    // GOOD - SLOTS (final: the ingest kernel ran before this one)
    if (threadIdx.x == 0) {
        int dup = block_missing;
        if (blockIdx.x == 0) dup += counters[CORR_PKT_GOOD] - CORR_PKT_SLOTS;
        if (block_missing) atomicAdd(counters + CORR_PKT_MISSING, block_missing);
        if (dup) atomicAdd(counters + CORR_PKT_DUPLICATE, dup);
    }
}

// The slot marks (one byte each, cleared four at a time) and the counters, in
// one launch.
__global__ void __launch_bounds__(kIngestThreads)
ingest_clear_kernel(uint32_t *__restrict__ seen4, int *__restrict__ counters)
{
    let_next_launch_start();
    for (int e = blockIdx.x * kIngestThreads + threadIdx.x; e < CORR_PKT_SLOTS / 4; e += gridDim.x * kIngestThreads)
        seen4[e] = 0u;
    if (blockIdx.x == 0 && threadIdx.x < CORR_PKT_COUNTERS) counters[threadIdx.x] = 0;
}

}  // namespace

cudaError_t launch_ingest(const uint8_t *packets, long long n_packets, int bank, uint8_t *volt, void *seen,
                          int32_t *counters, cudaStream_t s)
{
    static_assert(CORR_PKT_SLOTS % 4 == 0, "four slots per mark word");
    constexpr int clear_blocks = (CORR_PKT_SLOTS / 4 + kIngestThreads - 1) / kIngestThreads;
    ingest_clear_kernel<<<clear_blocks, kIngestThreads, 0, s>>>(static_cast<uint32_t *>(seen), counters);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    if (n_packets > 0) {
        const int grid = int((n_packets + kBlockPackets - 1) / kBlockPackets);
        const uintptr_t at = reinterpret_cast<uintptr_t>(packets);
        e = launch_overlapping(at % 16 == 0  ? ingest_kernel<16>
                               : at % 8 == 0 ? ingest_kernel<8>
                                             : ingest_kernel<4>,
                               grid, kIngestThreads, 0, true, s, packets, n_packets, bank, volt,
                               static_cast<uint8_t *>(seen), static_cast<int *>(counters));
        if (e != cudaSuccess) return e;
    }
    return launch_overlapping(ingest_missing_kernel, clear_blocks, kIngestThreads, 0, true, s, volt,
                              static_cast<const uint32_t *>(seen), static_cast<int *>(counters));
}

}  // namespace corr
