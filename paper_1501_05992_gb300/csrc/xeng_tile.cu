// The last 128-input tile of an odd number of tiles (the only one of an array of up
// to 128 inputs), one per CTA: xeng_diag.cuh.
#include "xeng_diag.cuh"

namespace corr {
namespace {

template <bool kAligned, bool kFresh, bool kZeroInvalid, bool kBeam>
__global__ void __launch_bounds__(kThreads, 1) xeng_tile_kernel(const __grid_constant__ Params p)
{
    extern __shared__ __align__(1024) uint8_t smem[];
    block_body<false, kAligned, kFresh, kZeroInvalid, kBeam>(p, smem, blockIdx.x, gridDim.x);
}

// [aligned][fresh][zero_invalid][beam]
void (*const g_kernels[16])(Params) = {
    xeng_tile_kernel<false, false, false, false>, xeng_tile_kernel<false, false, false, true>,
    xeng_tile_kernel<false, false, true, false>, xeng_tile_kernel<false, false, true, true>,
    xeng_tile_kernel<false, true, false, false>, xeng_tile_kernel<false, true, false, true>,
    xeng_tile_kernel<false, true, true, false>, xeng_tile_kernel<false, true, true, true>,
    xeng_tile_kernel<true, false, false, false>, xeng_tile_kernel<true, false, false, true>,
    xeng_tile_kernel<true, false, true, false>, xeng_tile_kernel<true, false, true, true>,
    xeng_tile_kernel<true, true, false, false>, xeng_tile_kernel<true, true, false, true>,
    xeng_tile_kernel<true, true, true, false>, xeng_tile_kernel<true, true, true, true>};

std::mutex g_mu;
int g_sms[64] = {0};

}  // namespace

cudaError_t launch_xeng_tile(const TcArray *arrays, int count, bool fresh, bool zero_invalid, int dev,
                             DeviceStatus *status, const TcOptions &opt, bool overlap, cudaStream_t s)
{
    Params prm{};
    cudaError_t e = make_params(arrays, count, false, status, opt, prm);
    if (e == cudaSuccess) e = prepare_device(g_kernels, dev, g_mu, g_sms);
    if (e != cudaSuccess) return e;
    const int cap = g_sms[dev];
    const int grid = (prm.n_items < cap ? prm.n_items : cap);
    return launch_overlapping(g_kernels[kernel_index(prm, fresh, zero_invalid)], grid, kThreads, kSmemBytes, overlap, s,
                              prm);
}

}  // namespace corr
