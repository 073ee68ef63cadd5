// Instantiates the fused 2:4 kernel for 64- and 128-wide tiles.
#include "sparq_gemm_sparse24_kernel.cuh"

namespace sparq {

template <int BN, int XN, bool RND, int OUT>
static cudaError_t launch_x24_out(const CUtensorMap &ma, const CUtensorMap &mb, const GemmArgs &g, int grid, cudaStream_t st)
{
    auto kfn = sparq_gemm_sparse24_kernel<BN, XN, RND, OUT>;
    static bool attr_set[64] = {};   // per device ordinal
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= 64 || !attr_set[dev]) {
        e = cudaFuncSetAttribute(kfn, cudaFuncAttributeMaxDynamicSharedMemorySize, X24Cfg<BN>::kSmemBytes);
        if (e != cudaSuccess) return e;
        if (dev >= 0 && dev < 64) attr_set[dev] = true;
    }
    return launch_overlapped(kfn, grid, kX24Threads, X24Cfg<BN>::kSmemBytes, st, ma, mb, g);
}

template <int BN, int XN, bool RND>
static cudaError_t launch_x24_kernel(const CUtensorMap &ma, const CUtensorMap &mb, const GemmArgs &g, int grid, cudaStream_t st)
{
    return make_epi_view(g).out == kOutBytes ? launch_x24_out<BN, XN, RND, kOutBytes>(ma, mb, g, grid, st)
                                             : launch_x24_out<BN, XN, RND, kOutGeneral>(ma, mb, g, grid, st);
}

template <int BN>
static cudaError_t launch_x24_bn(const CUtensorMap &ma, const CUtensorMap &mb, const GemmArgs &g, int n, int rnd, int grid, cudaStream_t st)
{
    if (n == 8) return launch_x24_kernel<BN, 8, true>(ma, mb, g, grid, st);
    if (n == 5) return rnd ? launch_x24_kernel<BN, 5, true>(ma, mb, g, grid, st) : launch_x24_kernel<BN, 5, false>(ma, mb, g, grid, st);
    if (n == 4) return rnd ? launch_x24_kernel<BN, 4, true>(ma, mb, g, grid, st) : launch_x24_kernel<BN, 4, false>(ma, mb, g, grid, st);
    return rnd ? launch_x24_kernel<BN, 0, true>(ma, mb, g, grid, st) : launch_x24_kernel<BN, 0, false>(ma, mb, g, grid, st);
}

cudaError_t launch_x24(int bn, const CUtensorMap &ma, const CUtensorMap &mb, const GemmArgs &g, int n, int rnd, int grid, cudaStream_t st)
{
    return bn == 64 ? launch_x24_bn<64>(ma, mb, g, n, rnd, grid, st) : launch_x24_bn<128>(ma, mb, g, n, rnd, grid, st);
}

}  // namespace sparq
