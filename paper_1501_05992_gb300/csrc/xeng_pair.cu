// The 256-input blocks on the diagonal of a channel's triangle, one per pair of
// CTAs: xeng_diag.cuh.
#include "xeng_diag.cuh"

namespace corr {
namespace {

template <bool kAligned, bool kFresh, bool kZeroInvalid, bool kBeam>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(kThreads, 1) xeng_pair_kernel(const __grid_constant__ Params p)
{
    extern __shared__ __align__(1024) uint8_t smem[];
    block_body<true, kAligned, kFresh, kZeroInvalid, kBeam>(p, smem, blockIdx.x >> 1, gridDim.x >> 1);
}

// [aligned][fresh][zero_invalid][beam]
void (*const g_kernels[16])(Params) = {
    xeng_pair_kernel<false, false, false, false>, xeng_pair_kernel<false, false, false, true>,
    xeng_pair_kernel<false, false, true, false>, xeng_pair_kernel<false, false, true, true>,
    xeng_pair_kernel<false, true, false, false>, xeng_pair_kernel<false, true, false, true>,
    xeng_pair_kernel<false, true, true, false>, xeng_pair_kernel<false, true, true, true>,
    xeng_pair_kernel<true, false, false, false>, xeng_pair_kernel<true, false, false, true>,
    xeng_pair_kernel<true, false, true, false>, xeng_pair_kernel<true, false, true, true>,
    xeng_pair_kernel<true, true, false, false>, xeng_pair_kernel<true, true, false, true>,
    xeng_pair_kernel<true, true, true, false>, xeng_pair_kernel<true, true, true, true>};

std::mutex g_mu;
int g_sms[64] = {0};

}  // namespace

cudaError_t launch_xeng_pair(const TcArray *arrays, int count, bool fresh, bool zero_invalid, int dev,
                             DeviceStatus *status, const TcOptions &opt, bool overlap, cudaStream_t s)
{
    Params prm{};
    cudaError_t e = make_params(arrays, count, true, status, opt, prm);
    if (e == cudaSuccess) e = prepare_device(g_kernels, dev, g_mu, g_sms);
    if (e != cudaSuccess) return e;
    const int cap = g_sms[dev] / 2;
    const int grid = 2 * (prm.n_items < cap ? prm.n_items : cap);
    return launch_overlapping(g_kernels[kernel_index(prm, fresh, zero_invalid)], grid, kThreads, kSmemBytes, overlap, s,
                              prm);
}

}  // namespace corr
