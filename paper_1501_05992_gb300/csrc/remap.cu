// Output remap (Appendix C, "GPU Output"), with optional further integration
// over adjacent channels and consecutive dumps (Section 3.4.3).
//
// The X-engine correlates the inputs in the order the PFBs deliver them
// (Appendix A: within each PFB's 64 inputs, position k carries input
// (k mod 4) * 16 + k div 4; Appendix B: the four PFBs' blocks follow each
// other) and writes the lower triangle over those positions.  The archived
// order is per station pair, natural input order, polarisation products
// innermost:
//
//     out[g][s1(s1+1)/2 + s2][p1][p2] = sum over dumps d and channels f of group g of
//                                       V_{2 s1 + p1, 2 s2 + p2}(f)
//
// with natural input a = 2 * station + pol.  V_AB with pos(A) >= pos(B) is a
// stored triangle element; otherwise it is the conjugate of the element
// (pos(B), pos(A)).  One thread owns one station pair: it finds the pair's
// four triangle elements once and then gathers them from every (dump,
// channel) of each channel group its block visits, four (group, dump,
// channel) triples at a time (16 loads in flight), writing the four
// polarisation products of a group (32 contiguous bytes) after its last
// triple.  The inverse permutation is arithmetic for Appendix A's order; for another it
// lives in shared memory, built once per block.  What bounds it is HBM (reads of the
// triangles, which the gather touches inside one channel's triangle at a time, and the
// coalesced writes): 256 inputs x 1536 channels, two by two channels and dumps, 148 us
// (1.01 GB, 149 us at the measured copy rate).  It took 171 us, 128 inputs x 3072
// channels / 4 57 us (now 46) and 64 x 3072 / 2 27 us (now 19.5), with divisions by
// f_avg and the dumps for every triple and a table in every block.
#include "internal.cuh"

namespace corr {
namespace {

constexpr int kRemapThreads = 256;
constexpr int kRemapMaxDumps = 8;
// Blocks of a launch, about: many, so that the last of them leave no gap (1600, 3200, 6400
// and 12800 blocks: 166, 156, 150 and 148 us for the shape above), fewer where each of
// them builds the table (512 inputs x 600 channels 198 us with 6400, 210 with 12800).  A thread
// finds its station pair's elements once and loads four triples at a time, so no block has a
// single group of one triple (256 inputs x 200, 300 and 400 channels 26.6 -> 20.5, 37.0 -> 29.1
// and 47.2 -> 37.0 us, with two groups at least), nor of two unless blocks are few (256 x 600 / 2
// 44.4 -> 39.2 us, but 128 x 600 / 2, 2700 blocks, 13.2 -> 14.3).
constexpr int kRemapBlocks = 12800, kRemapTableBlocks = 6400, kRemapFewBlocks = 3200;

struct RemapArgs {
    const int32_t *tri[kRemapMaxDumps];
    int n_dumps;
};

// Appendix A's position of natural input a (of a multiple of 64 inputs; within the array
// whatever n is)
__device__ __forceinline__ int pfb_position(int a, int n)
{
    const int i = (a & ~63) + 4 * (a & 15) + ((a >> 4) & 3);
    return i < n ? i : 0;
}

// kTable: the inputs' order comes in nat_of_pfb, otherwise it is Appendix A's.
template <bool kTable>
__global__ void __launch_bounds__(kRemapThreads)
remap_kernel(const __grid_constant__ RemapArgs args, int n, int n_chan, int f_avg,
             const int32_t *__restrict__ nat_of_pfb, int32_t *__restrict__ out)
{
    extern __shared__ int pos[];                    // pos[a]: PFB position of natural input a
    if (kTable) {
        // every entry starts as a valid position, so a table that is not a
        // permutation gives wrong products but never an access out of bounds
        for (int a = threadIdx.x; a < n; a += blockDim.x) pos[a] = 0;
        __syncthreads();
        for (int i = threadIdx.x; i < n; i += blockDim.x) {
            const int a = nat_of_pfb[i];
            if (a >= 0 && a < n) pos[a] = i;
        }
        __syncthreads();
    }
    const long long P = n_pairs(n);
    const int S = n / 2;
    const long long Q = n_pairs(S);
    const int n_groups = n_chan / f_avg, n_comb = args.n_dumps * f_avg;
    for (long long q = blockIdx.x * (long long)blockDim.x + threadIdx.x; q < Q;
         q += (long long)gridDim.x * blockDim.x) {
        int s1 = int((sqrtf(8.0f * float(q) + 1.0f) - 1.0f) * 0.5f);
        while (n_pairs(s1 + 1) <= q) ++s1;
        while (n_pairs(s1) > q) --s1;
        const int s2 = int(q - n_pairs(s1));
        long long k[4];
        bool conj[4];
#pragma unroll
        for (int pp = 0; pp < 4; ++pp) {
            const int a = 2 * s1 + (pp >> 1), b = 2 * s2 + (pp & 1);
            const int i = kTable ? pos[a] : pfb_position(a, n), j = kTable ? pos[b] : pfb_position(b, n);
            conj[pp] = i < j;
            k[pp] = conj[pp] ? n_pairs(j) + i : n_pairs(i) + j;
        }
        // the (channel group, dump, channel) triples of this thread's station pair,
        // groups blockIdx.y + j gridDim.y, taken four at a time (16 loads in flight);
        // the triple to load next is (g, d, f), the group being summed is g_out
        const int n_j = (n_groups - int(blockIdx.y) + int(gridDim.y) - 1) / int(gridDim.y);
        const int n_e = n_j * n_comb;
        int g = blockIdx.y, d = 0, f = 0, g_out = blockIdx.y, left = n_comb;
        int re[4] = {0, 0, 0, 0}, im[4] = {0, 0, 0, 0};
        for (int e0 = 0; e0 < n_e; e0 += 4) {
            int2 v[4][4];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                if (e0 + u >= n_e) break;
                const int2 *tri = reinterpret_cast<const int2 *>(args.tri[d]) + (long long)(g * f_avg + f) * P;
#pragma unroll
                for (int pp = 0; pp < 4; ++pp) v[u][pp] = __ldg(tri + k[pp]);
                if (++f == f_avg) {
                    f = 0;
                    if (++d == args.n_dumps) {
                        d = 0;
                        g += gridDim.y;
                    }
                }
            }
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                if (e0 + u >= n_e) break;
#pragma unroll
                for (int pp = 0; pp < 4; ++pp) {
                    re[pp] += v[u][pp].x;
                    im[pp] += v[u][pp].y;
                }
                if (--left == 0) {
                    // the group's last triple: write its four products and start the next
                    int4 *o = reinterpret_cast<int4 *>(out) + ((long long)g_out * Q + q) * 2;
                    o[0] = make_int4(re[0], conj[0] ? -im[0] : im[0], re[1], conj[1] ? -im[1] : im[1]);
                    o[1] = make_int4(re[2], conj[2] ? -im[2] : im[2], re[3], conj[3] ? -im[3] : im[3]);
#pragma unroll
                    for (int pp = 0; pp < 4; ++pp) re[pp] = im[pp] = 0;
                    left = n_comb;
                    g_out += gridDim.y;
                }
            }
        }
    }
}

}  // namespace

cudaError_t launch_remap(const int32_t *const *tri, int n_dumps, int n, int n_chan, int f_avg,
                         const int32_t *nat_of_pfb, int32_t *out, cudaStream_t s)
{
    if (n_dumps < 1 || n_dumps > kRemapMaxDumps) return cudaErrorInvalidValue;
    RemapArgs args{};
    for (int d = 0; d < n_dumps; ++d) args.tri[d] = tri[d];
    args.n_dumps = n_dumps;
    const long long Q = n_pairs(n / 2);
    const long long want = (Q + kRemapThreads - 1) / kRemapThreads;
    const int bx = int(want < 4096 ? want : 4096);
    const int groups = n_chan / f_avg;
    int by = ((nat_of_pfb ? kRemapTableBlocks : kRemapBlocks) + bx - 1) / bx;
    const int comb = n_dumps * f_avg;
    const bool two = comb == 1 || (comb == 2 && (long long)groups * bx >= kRemapFewBlocks);
    const int most = two ? (groups + 1) / 2 : groups;
    if (by > most) by = most;
    const dim3 grid{unsigned(bx), unsigned(by)};
    if (nat_of_pfb)
        remap_kernel<true><<<grid, kRemapThreads, size_t(n) * sizeof(int), s>>>(args, n, n_chan, f_avg, nat_of_pfb, out);
    else
        remap_kernel<false><<<grid, kRemapThreads, 0, s>>>(args, n, n_chan, f_avg, nullptr, out);
    return cudaGetLastError();
}

}  // namespace corr
