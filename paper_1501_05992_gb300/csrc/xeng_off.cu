// The tiles off the 256-input diagonal blocks of arrays of more than 256 inputs, by pairs
// of CTAs: xeng_off.cuh.
#include <mutex>

#include "xeng_off.cuh"

namespace corr {
namespace {

template <bool kFresh, bool kZeroInvalid>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(off::kThreads, 1)
xeng_off_kernel(const __grid_constant__ off::Tmaps tmaps, const __grid_constant__ off::Params p)
{
    extern __shared__ __align__(1024) uint8_t smem[];
    off::off_body<kFresh, kZeroInvalid>(tmaps, p, smem, blockIdx.x >> 1, gridDim.x >> 1);
}

std::mutex g_mu;
int g_clusters[64] = {0};

}  // namespace

cudaError_t launch_xeng_off(const TcArray *arrays, const CUtensorMap *maps, int count, bool fresh, bool zero_invalid,
                            int dev, DeviceStatus *status, const TcOptions &opt, bool overlap, cudaStream_t s)
{
    if (dev < 0 || dev >= 64) return cudaErrorInvalidValue;
    {
        std::lock_guard<std::mutex> lock(g_mu);
        if (!g_clusters[dev]) {
            cudaError_t e;
            for (auto fn : {xeng_off_kernel<false, false>, xeng_off_kernel<false, true>, xeng_off_kernel<true, false>,
                            xeng_off_kernel<true, true>}) {
                e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, off::kSmemBytes);
                if (e != cudaSuccess) return e;
            }
            int sms = 0;
            e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
            if (e != cudaSuccess) return e;
            g_clusters[dev] = sms / 2;
        }
    }
    off::Params prm{};
    off::Tmaps tm;
    const cudaError_t ep = off::make_params(arrays, maps, count, status, opt, prm, tm);
    if (ep != cudaSuccess) return ep;
    const int grid = 2 * (prm.n_items < g_clusters[dev] ? prm.n_items : g_clusters[dev]);
    const auto fn = fresh ? (zero_invalid ? xeng_off_kernel<true, true> : xeng_off_kernel<true, false>)
                          : (zero_invalid ? xeng_off_kernel<false, true> : xeng_off_kernel<false, false>);
    return launch_overlapping(fn, grid, off::kThreads, off::kSmemBytes, overlap, s, tm, prm);
}

}  // namespace corr
