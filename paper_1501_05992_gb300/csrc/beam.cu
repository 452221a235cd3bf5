// Incoherent beam: total power of all inputs per channel and sample.
//
// Section 3.4 lists incoherent beam forming among the XMAC's modes beside the
// correlation: the power sum over every input of a channel, at the voltage
// time resolution (or integrated over n_avg samples):
//
//     beam[k][f] = sum over the n_avg samples t of block k, over inputs n, of |x_n(t,f)|^2
//
// The kernel is bound by HBM reads (N bytes per sample and channel, 4 bytes
// written per output).  Where N is a multiple of 16 a group of L lanes (L the
// largest power of two up to 32 dividing N / 16) reads one channel's row of a
// sample, each lane 16-byte chunks L chunks apart, so a warp's load covers
// 32 / L neighbouring rows, i.e. 512 contiguous bytes; the group adds its
// lanes' sums with shuffles once per output.  A block takes 32
// neighbouring channels (8 KB per sample at N = 256).  Per 32-bit word (four samples) the
// high nibbles with the low ones cleared are the signed bytes 16 r, the low
// nibbles moved up 16 m, and two dp4a add 256 (r^2 + m^2); each row's sum is
// divided by 256 before it is added, which keeps every partial sum within
// int32 wherever the result is.  Other input counts take one thread per
// channel and output, walking the row byte by byte.
#include "internal.cuh"

namespace corr {
namespace {

constexpr int kBeamThreads = 128;

// |x|^2 of the four samples in w, summed (4-bit two's complement nibbles, real
// in the high nibble).  With zero_invalid a sample with either nibble 8
// contributes nothing.
template <bool kZeroInvalid>
__device__ __forceinline__ int power4(uint32_t w, int acc)
{
    const uint32_t uh = ((w >> 4) & 0x0F0F0F0Fu) ^ 0x08080808u;   // code + 8, 0..15
    const uint32_t ul = (w & 0x0F0F0F0Fu) ^ 0x08080808u;
    uint32_t vh = __vsub4(uh, 0x08080808u);                       // signed bytes -8..7
    uint32_t vl = __vsub4(ul, 0x08080808u);
    if (kZeroInvalid) {
        // a nibble code 8 has u == 0; zero both parts of such samples
        const uint32_t bad = __vcmpeq4(uh, 0u) | __vcmpeq4(ul, 0u);
        vh &= ~bad;
        vl &= ~bad;
    }
    acc = __dp4a(int(vh), int(vh), acc);
    return __dp4a(int(vl), int(vl), acc);
}

// One thread per channel and output; one sample per word (the three zero bytes
// are valid samples of value 0).
template <bool kZeroInvalid>
__global__ void __launch_bounds__(kBeamThreads)
beam_bytes_kernel(const uint8_t *__restrict__ volt, int n, int n_chan, int n_avg, int n_out,
                  int32_t *__restrict__ out)
{
    const int f = blockIdx.x * kBeamThreads + threadIdx.x;
    if (f >= n_chan) return;
    for (int k = blockIdx.y; k < n_out; k += gridDim.y) {
        int acc = 0;
        for (int t = k * n_avg; t < (k + 1) * n_avg; ++t) {
            const uint8_t *row = volt + ((size_t)t * n_chan + f) * n;
            for (int c = 0; c < n; ++c) acc = power4<kZeroInvalid>(uint32_t(row[c]), acc);
        }
        out[(size_t)k * n_chan + f] = acc;
    }
}

// 256 (r^2 + m^2) summed over the four samples of w, plus acc (the high nibble
// with the low one cleared is the signed byte 16 r; the low nibble moved up,
// 16 m).
__device__ __forceinline__ int power4x256(uint32_t w, int acc)
{
    const uint32_t hr = w & 0xF0F0F0F0u, hm = (w << 4) & 0xF0F0F0F0u;
    return __dp4a(int(hm), int(hm), __dp4a(int(hr), int(hr), acc));
}

// Nonzero where any nibble of w is the code 8.
__device__ __forceinline__ uint32_t has_invalid(uint32_t w)
{
    const uint32_t x = w ^ 0x88888888u;
    return (x - 0x11111111u) & ~x & 0x88888888u;
}

// w with the samples that have a nibble of 8 set to zero.
__device__ __forceinline__ uint32_t drop_invalid(uint32_t w)
{
    const uint32_t x = w ^ 0x88888888u;
    uint32_t t = x | (x >> 1);
    t |= t >> 2;                                  // bit 0 of each nibble: the code was not 8
    return w & ((t & (t >> 4) & 0x01010101u) * 0xFFu);
}

// kL lanes per channel row (N a multiple of 16 kL; 16-byte aligned rows).  A
// block of kThreads takes kIter channels per group of lanes, a thread kU of them
// at a time, so that kU loads (per chunk) are in flight before the first is used.
// kEven: the blocks of a sample take `per` channels each instead of as many as they can.
template <bool kZeroInvalid, int kL, int kThreads, int kIter, bool kEven>
__global__ void __launch_bounds__(kThreads)
beam_rows_kernel(const uint8_t *__restrict__ volt, int n, int n_chan, int n_avg, int n_out,
                 int32_t *__restrict__ out, int per)
{
    constexpr int kGroups = kThreads / kL, kChans = kGroups * kIter;
    constexpr int kU = kIter < 4 ? kIter : 4;
    const int sub = threadIdx.x % kL, group = threadIdx.x / kL;
    const int per_lane = n / (16 * kL);
    const int f0 = blockIdx.x * (kEven ? per : kChans), f1 = kEven ? min(n_chan, f0 + per) : n_chan;
    for (int k = blockIdx.y; k < n_out; k += gridDim.y) {
        // the trip counts are the same for every group, so whole warps shuffle
        for (int fb = group; fb < kChans; fb += kU * kGroups) {
            int acc[kU];
#pragma unroll
            for (int u = 0; u < kU; ++u) acc[u] = 0;
            for (int t = k * n_avg; t < (k + 1) * n_avg; ++t) {
                const uint4 *row[kU];
#pragma unroll
                for (int u = 0; u < kU; ++u) {
                    // a channel past the end reads another's row and is not stored
                    const int f = f0 + fb + u * kGroups;
                    row[u] = reinterpret_cast<const uint4 *>(volt + ((size_t)t * n_chan + (f < f1 ? f : kEven ? f0 : 0)) * n) +
                             sub;
                }
                int p[kU];
#pragma unroll
                for (int u = 0; u < kU; ++u) p[u] = 0;
                for (int j = 0; j < per_lane; ++j) {
                    uint4 w[kU];
#pragma unroll
                    for (int u = 0; u < kU; ++u) w[u] = row[u][j * kL];
#pragma unroll
                    for (int u = 0; u < kU; ++u) {
                        // invalid samples are rare: one test per 16 samples
                        if (kZeroInvalid && (has_invalid(w[u].x) | has_invalid(w[u].y) | has_invalid(w[u].z) |
                                             has_invalid(w[u].w)))
                            w[u] = make_uint4(drop_invalid(w[u].x), drop_invalid(w[u].y), drop_invalid(w[u].z),
                                              drop_invalid(w[u].w));
                        p[u] = power4x256(w[u].x, p[u]);
                        p[u] = power4x256(w[u].y, p[u]);
                        p[u] = power4x256(w[u].z, p[u]);
                        p[u] = power4x256(w[u].w, p[u]);
                    }
                }
#pragma unroll
                for (int u = 0; u < kU; ++u) acc[u] += p[u] >> 8;
            }
#pragma unroll
            for (int u = 0; u < kU; ++u) {
#pragma unroll
                for (int o = kL / 2; o >= 1; o /= 2) acc[u] += __shfl_xor_sync(0xFFFFFFFFu, acc[u], o);
                const int f = f0 + fb + u * kGroups;
                if (sub == 0 && f < f1) out[(size_t)k * n_chan + f] = acc[u];
            }
        }
    }
}

template <bool kZeroInvalid, int kL, int kThreads, int kIter, bool kEven = false>
void launch_blocks(const uint8_t *volt, int n, int n_chan, int n_avg, int n_out, int32_t *out, cudaStream_t s)
{
    // a few outputs per block: 1024 rows of blocks at most
    const int blocks = div_up(n_chan, kThreads / kL * kIter), rows = n_out < 1024 ? n_out : 1024;
    const dim3 grid{unsigned(blocks), unsigned(rows)};
    beam_rows_kernel<kZeroInvalid, kL, kThreads, kIter, kEven>
        <<<grid, kThreads, 0, s>>>(volt, n, n_chan, n_avg, n_out, out, div_up(n_chan, blocks));
}

// Threads of a block and channels it takes, for kL lanes per row.  Small blocks leave
// a shorter tail and need no more loads in flight than four per thread: 256 inputs x
// 3072 channels x 500 samples 69.5 us with 256 threads and 128 channels, 66.3 with 128
// and 64, 64.1 with 64 and 32 (59 us at the measured copy rate).  Testing 16 samples at a
// time for invalid ones: 111 -> 92 us with one sample in eight invalid, 99 with smaller
// blocks and no such test.
//  - 16 or 32 lanes: a thread's turns of four channels follow each other, so that few blocks
//    are bound by latency.  One turn (8 channels of 32 lanes; 16 of 16 lanes up to six blocks
//    of 32 per SM): 1024 inputs x 40 channels x 400 samples, ten added, 25.5 -> 9.1 us, 256 x 40 x
//    400 / 10 11.1 -> 7.0; with more blocks 16 channels are slower (768 x 1500 x 300 / 10 60 us, 68).
//  - 1 or 2 lanes: where a sample takes two blocks and the second is partly empty, the full
//    ones land on every other SM; two of equal shares don't mind (1008 x 130 x 800 31.3 -> 19.3 us).
//    Rows of up to 64 bytes by themselves are a load or two a thread and want bigger blocks
//    (32 x 3072 x 800 23.4 -> 20.0 us).
template <bool kZeroInvalid, int kL>
void launch_rows(const uint8_t *volt, int n, int n_chan, int n_avg, int n_out, int32_t *out, cudaStream_t s)
{
    constexpr long long kFewBlocks = 6 * 152;
    if constexpr (kL <= 2) {
        constexpr int kChans = 128 / kL;
        if (n <= 64 && n_avg == 1)
            launch_blocks<kZeroInvalid, kL, 256, 1>(volt, n, n_chan, n_avg, n_out, out, s);
        else if (n_chan > kChans && n_chan < 2 * kChans)
            launch_blocks<kZeroInvalid, kL, 128, 1, true>(volt, n, n_chan, n_avg, n_out, out, s);
        else
            launch_blocks<kZeroInvalid, kL, 128, 1>(volt, n, n_chan, n_avg, n_out, out, s);
    } else if constexpr (kL == 4) {
        launch_blocks<kZeroInvalid, kL, 128, 2>(volt, n, n_chan, n_avg, n_out, out, s);
    } else if constexpr (kL == 16) {
        if ((long long)div_up(n_chan, 32) * n_out <= kFewBlocks)
            launch_blocks<kZeroInvalid, kL, 64, 4>(volt, n, n_chan, n_avg, n_out, out, s);
        else
            launch_blocks<kZeroInvalid, kL, 64, 8>(volt, n, n_chan, n_avg, n_out, out, s);
    } else {
        launch_blocks<kZeroInvalid, kL, 64, 4>(volt, n, n_chan, n_avg, n_out, out, s);
    }
}

template <bool kZeroInvalid>
cudaError_t launch_rows(int lanes, const uint8_t *volt, int n, int n_chan, int n_avg, int n_out, int32_t *out,
                        cudaStream_t s)
{
    switch (lanes) {
    case 1: launch_rows<kZeroInvalid, 1>(volt, n, n_chan, n_avg, n_out, out, s); break;
    case 2: launch_rows<kZeroInvalid, 2>(volt, n, n_chan, n_avg, n_out, out, s); break;
    case 4: launch_rows<kZeroInvalid, 4>(volt, n, n_chan, n_avg, n_out, out, s); break;
    case 8: launch_rows<kZeroInvalid, 8>(volt, n, n_chan, n_avg, n_out, out, s); break;
    case 16: launch_rows<kZeroInvalid, 16>(volt, n, n_chan, n_avg, n_out, out, s); break;
    default: launch_rows<kZeroInvalid, 32>(volt, n, n_chan, n_avg, n_out, out, s); break;
    }
    return cudaGetLastError();
}

}  // namespace

cudaError_t launch_beam(const uint8_t *volt, int n_time, int n_chan, int n, int n_avg, bool zero_invalid,
                        int32_t *out, cudaStream_t s)
{
    const int n_out = n_time / n_avg;
    if (n_out == 0) return cudaSuccess;
    if (n % 16 == 0 && (reinterpret_cast<uintptr_t>(volt) & 15) == 0) {
        // lanes per row: the largest power of two up to 32 dividing the row's chunks
        const int chunks = n / 16;
        int lanes = 1;
        while (lanes < 32 && chunks % (2 * lanes) == 0) lanes *= 2;
        return zero_invalid ? launch_rows<true>(lanes, volt, n, n_chan, n_avg, n_out, out, s)
                            : launch_rows<false>(lanes, volt, n, n_chan, n_avg, n_out, out, s);
    }
    const dim3 grid(unsigned(div_up(n_chan, kBeamThreads)), unsigned(n_out < 65535 ? n_out : 65535));
    if (zero_invalid) beam_bytes_kernel<true><<<grid, kBeamThreads, 0, s>>>(volt, n, n_chan, n_avg, n_out, out);
    else beam_bytes_kernel<false><<<grid, kBeamThreads, 0, s>>>(volt, n, n_chan, n_avg, n_out, out);
    return cudaGetLastError();
}

}  // namespace corr
