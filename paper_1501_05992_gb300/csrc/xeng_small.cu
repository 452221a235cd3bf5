// X-engine for small arrays (up to 64 inputs) on the CUDA cores, straight from the
// packed voltages.
//
// The same dp4a form as xeng_dp4a.cu (two samples of a complex product per
// instruction and component), but one launch and no operands in device memory:
// a block takes one channel over a slice of time, decodes the packed bytes into
// the A words and their twisted copies in shared memory (4 KB of samples at a
// time, the next 4 KB already loading), and its threads are (4 x 4 tile of the
// triangle, group): group g takes words g, g + G, ... of each piece.  The groups'
// sums meet in shared memory, and the slices of a channel, which are the CTAs of
// one cluster, through distributed shared memory, so that a launch that stores
// needs no zeroed output and one that adds touches the output once.
//
// Why: a small array is bound by latency, not by arithmetic.  The staged path
// walks a whole integration in one 32-thread block per channel and writes and
// reads eight bytes of operands per sample.  Four-by-four tiles waste less of the
// diagonal than 32 x 32 ones (16 inputs: 10 tiles of 16 products for 136 pairs).
// Slices: as many (1, 2, 4 or 8) as bring the grid to two blocks per SM, while
// each keeps 64 samples.
//
// Measured against the staged path's better tile: 16 inputs x 32 channels x 1000
// samples 47 -> 9 us, 16 x 1 x 100000 3.85 -> 0.06 ms, 16 x 2048 x 5000 1.17 -> 0.21
// ms, 32 x 1024 x 5000 0.70 -> 0.30 ms, 48 x 512 x 5000 0.82 -> 0.34 ms, 63 x 512 x
// 5000 1.02 -> 0.68 ms, 64 x 512 x 5000 0.82 -> 0.64 ms.  Large ones are bound by the
// dp4a rate (two cycles a warp) and the three 16-byte shared loads per 32 of them.
#include "decode.cuh"
#include "internal.cuh"

namespace corr {
namespace {

constexpr int kThreads = 288;             // 9 warps: 28 groups at 16 inputs, 8 at 32, 2 at 64
constexpr int kPieceWords = 1024;         // 32-bit words of packed samples per piece (4 KB)
constexpr int kPieceUnits = kPieceWords / 2;   // (word, four inputs) units of a piece
constexpr int kUnitsPerThread = (kPieceUnits + kThreads - 1) / kThreads;
constexpr int kMaxSlices = 8;
constexpr int kMinSliceSamples = 64;

struct SmallArgs {
    const uint8_t *volt;
    int32_t *out;
    int n, n_chan, nt, slice;             // slice: samples per slice (even)
    int vec;                              // rows start on word boundaries, n a multiple of 4
};

__device__ __forceinline__ uint32_t cluster_ctarank()
{
    uint32_t r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}

__device__ __forceinline__ void cluster_barrier()
{
    asm volatile("barrier.cluster.arrive.release.aligned;\n barrier.cluster.wait.acquire.aligned;" ::: "memory");
}

__device__ __forceinline__ int2 load_peer(uint32_t addr, uint32_t rank)
{
    uint32_t a;
    int2 v;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"(addr), "r"(rank));
    asm volatile("ld.shared::cluster.v2.s32 {%0, %1}, [%2];" : "=r"(v.x), "=r"(v.y) : "r"(a) : "memory");
    return v;
}

// row i >= j of the lower triangle from its packed index
__device__ __forceinline__ void triangle_of(int b, int &i, int &j)
{
    i = int((sqrtf(8.0f * float(b) + 1.0f) - 1.0f) * 0.5f);
    while ((i + 1) * (i + 2) / 2 <= b) ++i;
    while (i * (i + 1) / 2 > b) --i;
    j = b - i * (i + 1) / 2;
}

template <bool kZeroInvalid, bool kFresh>
__global__ void __launch_bounds__(kThreads)
xeng_small_kernel(SmallArgs a)
{
    extern __shared__ __align__(16) int32_t smem[];
    const int cols = (a.n + 3) / 4;               // groups of four inputs
    const int pitch = cols * 4;                   // words of a row of A (or W)
    const int words = kPieceUnits / cols;         // words (two samples each) per piece
    int32_t *const A = smem, *const W = smem + words * pitch;

    const int f = blockIdx.y;
    const int slices = gridDim.x, rank = slices > 1 ? int(cluster_ctarank()) : 0;
    const int t_begin = rank * a.slice, t_end = min(a.nt, t_begin + a.slice);
    const size_t row_t = size_t(a.n_chan) * a.n;
    const uint8_t *const base = a.volt + size_t(f) * a.n;

    const int tiles = cols * (cols + 1) / 2, groups = kThreads / tiles;
    const int tile = threadIdx.x % tiles, group = threadIdx.x / tiles;
    const bool works = group < groups;
    int ta, tb;
    triangle_of(tile, ta, tb);

    // the packed samples of this thread's units of a piece: four inputs at two times
    uint32_t p0[kUnitsPerThread], p1[kUnitsPerThread];
    auto fetch = [&](int t0) {
#pragma unroll
        for (int k = 0; k < kUnitsPerThread; ++k) {
            const int e = threadIdx.x + k * kThreads, tw = e / cols, g = e - tw * cols;
            const int t = t0 + 2 * tw, n0 = 4 * g;
            p0[k] = p1[k] = 0;
            if (tw >= words || t >= t_end) continue;
            const uint8_t *s = base + size_t(t) * row_t + n0;
            if (a.vec) {
                p0[k] = __ldg(reinterpret_cast<const uint32_t *>(s));
                if (t + 1 < t_end) p1[k] = __ldg(reinterpret_cast<const uint32_t *>(s + row_t));
            } else {
                for (int b = 0; b < 4 && n0 + b < a.n; ++b) {
                    p0[k] |= uint32_t(__ldg(s + b)) << (8 * b);
                    if (t + 1 < t_end) p1[k] |= uint32_t(__ldg(s + row_t + b)) << (8 * b);
                }
            }
        }
    };
    int re[4][4], im[4][4];
#pragma unroll
    for (int r = 0; r < 4; ++r)
#pragma unroll
        for (int c = 0; c < 4; ++c) re[r][c] = im[r][c] = 0;

    fetch(t_begin);
    for (int t0 = t_begin; t0 < t_end; t0 += 2 * words) {
#pragma unroll
        for (int k = 0; k < kUnitsPerThread; ++k) {
            const int e = threadIdx.x + k * kThreads, tw = e / cols, g = e - tw * cols;
            if (tw >= words) continue;
            uint32_t wa[4], ww[4];
            words4(p0[k], p1[k], kZeroInvalid, wa, ww);
            *reinterpret_cast<uint4 *>(A + tw * pitch + 4 * g) = make_uint4(wa[0], wa[1], wa[2], wa[3]);
            *reinterpret_cast<uint4 *>(W + tw * pitch + 4 * g) = make_uint4(ww[0], ww[1], ww[2], ww[3]);
        }
        __syncthreads();
        if (t0 + 2 * words < t_end) fetch(t0 + 2 * words);
        const int here = min(words, (t_end - t0 + 1) / 2);
        if (works) {
            for (int k = group; k < here; k += groups) {
                const int4 x = *reinterpret_cast<const int4 *>(A + k * pitch + 4 * ta);
                const int4 y = *reinterpret_cast<const int4 *>(A + k * pitch + 4 * tb);
                const int4 z = *reinterpret_cast<const int4 *>(W + k * pitch + 4 * tb);
                const int xs[4] = {x.x, x.y, x.z, x.w}, ys[4] = {y.x, y.y, y.z, y.w}, zs[4] = {z.x, z.y, z.z, z.w};
#pragma unroll
                for (int r = 0; r < 4; ++r)
#pragma unroll
                    for (int c = 0; c < 4; ++c) {
                        re[r][c] = __dp4a(xs[r], ys[c], re[r][c]);
                        im[r][c] = __dp4a(xs[r], zs[c], im[r][c]);
                    }
            }
        }
        __syncthreads();
    }

    // the groups' sums: [group][tile][16] pairs, then added into group 0's
    int2 *const part = reinterpret_cast<int2 *>(smem);
    if (works) {
#pragma unroll
        for (int r = 0; r < 4; ++r)
#pragma unroll
            for (int c = 0; c < 4; ++c) part[(group * tiles + tile) * 16 + r * 4 + c] = make_int2(re[r][c], im[r][c]);
    }
    __syncthreads();
    for (int e = threadIdx.x; e < tiles * 16; e += kThreads) {
        int2 v = part[e];
        for (int g = 1; g < groups; ++g) {
            const int2 u = part[g * tiles * 16 + e];
            v.x += u.x;
            v.y += u.y;
        }
        part[e] = v;
    }
    // the slices: each CTA adds up and writes its share of the pairs
    if (slices > 1) cluster_barrier();
    else __syncthreads();
    const int P = a.n * (a.n + 1) / 2;
    const uint32_t part_addr = static_cast<uint32_t>(__cvta_generic_to_shared(part));
    int2 *const out = reinterpret_cast<int2 *>(a.out) + size_t(f) * size_t(P);
    for (int e = rank * kThreads + threadIdx.x; e < P; e += slices * kThreads) {
        int i, j;
        triangle_of(e, i, j);
        const int ti = i >> 2, tj = j >> 2;
        const int at = (ti * (ti + 1) / 2 + tj) * 16 + (i & 3) * 4 + (j & 3);
        int2 v = make_int2(0, 0);
        if (slices > 1) {
            for (int s = 0; s < slices; ++s) {
                const int2 u = load_peer(part_addr + uint32_t(at) * 8u, uint32_t(s));
                v.x += u.x;
                v.y += u.y;
            }
        } else {
            v = part[at];
        }
        if (!kFresh) {
            const int2 old = out[e];
            v.x += old.x;
            v.y += old.y;
        }
        out[e] = v;
    }
    if (slices > 1) cluster_barrier();            // the peers' sums have been read
}

}  // namespace

cudaError_t launch_xeng_small(const uint8_t *volt, int n_chan, int n, int nt, bool zero_invalid, int32_t *out,
                              bool fresh, int sm_count, cudaStream_t s)
{
    if (n < 1 || n > kSmallMaxInputs || nt < 1 || n_chan < 1 || n_chan > 65535) return cudaErrorInvalidValue;
    int slices = 1;
    while (slices < kMaxSlices && (long long)n_chan * slices < 2LL * sm_count && nt >= 2 * slices * kMinSliceSamples)
        slices *= 2;
    SmallArgs a;
    a.volt = volt;
    a.out = out;
    a.n = n;
    a.n_chan = n_chan;
    a.nt = nt;
    a.slice = 2 * div_up(div_up(nt, 2), slices);
    a.vec = n % 4 == 0 && (reinterpret_cast<uintptr_t>(volt) & 3) == 0;
    // a piece's A and W words, then every group's sums
    const int cols = div_up(n, 4), tiles = cols * (cols + 1) / 2;
    const size_t operands = size_t(2) * (kPieceUnits / cols) * cols * 4 * sizeof(int32_t);
    const size_t sums = size_t(kThreads / tiles) * tiles * 16 * sizeof(int2);
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(unsigned(slices), unsigned(n_chan));
    cfg.blockDim = dim3(kThreads);
    cfg.dynamicSmemBytes = operands > sums ? operands : sums;
    cfg.stream = s;
    cudaLaunchAttribute attr{};
    attr.id = cudaLaunchAttributeClusterDimension;
    attr.val.clusterDim.x = unsigned(slices);
    attr.val.clusterDim.y = 1;
    attr.val.clusterDim.z = 1;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    const auto fn = zero_invalid ? (fresh ? xeng_small_kernel<true, true> : xeng_small_kernel<true, false>)
                                 : (fresh ? xeng_small_kernel<false, true> : xeng_small_kernel<false, false>);
    return cudaLaunchKernelEx(&cfg, fn, a);
}

}  // namespace corr
