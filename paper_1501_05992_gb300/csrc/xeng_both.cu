// The 256-input blocks of an array of more than 256 inputs and the tiles off them in one
// launch: some pairs of CTAs take the blocks (xeng_diag.cuh), the others the tiles
// (xeng_off.cuh).  For calls of few rounds of items (launch_large in xeng_tc.cu): a second
// launch's CTAs start where the first one's have left, 9 us for items of short integrations
// that a CTA already there does in 6 us more.
#include "xeng_diag.cuh"
#include "xeng_off.cuh"

namespace corr {
namespace {

constexpr int kBothSmem = kSmemBytes > off::kSmemBytes ? kSmemBytes : off::kSmemBytes;
static_assert(off::kThreads >= kThreads, "warps for either kind of items");

// The first block_pairs pairs of CTAs take the blocks.
template <bool kFresh, bool kZeroInvalid, bool kBeam>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(off::kThreads, 1)
xeng_both_kernel(const __grid_constant__ off::Tmaps tmaps, const __grid_constant__ off::Params po,
                 const __grid_constant__ Params pb, int block_pairs)
{
    extern __shared__ __align__(1024) uint8_t smem[];
    const int pair = blockIdx.x >> 1, pairs = gridDim.x >> 1;
    if (pair < block_pairs)
        block_body<true, true, kFresh, kZeroInvalid, kBeam, true>(pb, smem, pair, block_pairs);
    else
        off::off_body<kFresh, kZeroInvalid>(tmaps, po, smem, pair - block_pairs, pairs - block_pairs);
}

// [fresh][zero_invalid][beam]
void (*const g_kernels[8])(off::Tmaps, off::Params, Params, int) = {
    xeng_both_kernel<false, false, false>, xeng_both_kernel<false, false, true>, xeng_both_kernel<false, true, false>,
    xeng_both_kernel<false, true, true>,   xeng_both_kernel<true, false, false>, xeng_both_kernel<true, false, true>,
    xeng_both_kernel<true, true, false>,   xeng_both_kernel<true, true, true>};

std::mutex g_mu;
bool g_ready[64] = {};

}  // namespace

cudaError_t launch_xeng_both(const TcArray &A, const CUtensorMap &map, int block_pairs, int off_pairs, bool fresh,
                             bool zero_invalid, int dev, DeviceStatus *status, const TcOptions &opt, bool overlap,
                             cudaStream_t s)
{
    if (dev < 0 || dev >= 64 || block_pairs < 1 || off_pairs < 1) return cudaErrorInvalidValue;
    Params pb{};
    off::Params po{};
    off::Tmaps tm;
    cudaError_t e = make_params(&A, 1, true, status, opt, pb);
    if (e == cudaSuccess) e = off::make_params(&A, &map, 1, status, opt, po, tm);
    if (e != cudaSuccess) return e;
    {
        std::lock_guard<std::mutex> lock(g_mu);
        for (int k = 0; k < 8 && !g_ready[dev]; ++k) {
            e = cudaFuncSetAttribute(g_kernels[k], cudaFuncAttributeMaxDynamicSharedMemorySize, kBothSmem);
            if (e != cudaSuccess) return e;
        }
        g_ready[dev] = true;
    }
    const int k = (fresh ? 4 : 0) + (zero_invalid ? 2 : 0) + (A.beam ? 1 : 0);
    return launch_overlapping(g_kernels[k], 2 * (block_pairs + off_pairs), off::kThreads, kBothSmem, overlap, s, tm, po,
                              pb, block_pairs);
}

}  // namespace corr
