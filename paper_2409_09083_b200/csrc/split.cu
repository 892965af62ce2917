// Host-side launchers of the split kernels (the fp32 path on the tensor cores).
#include <cuda_runtime.h>

#include <algorithm>

#include "split.cuh"

namespace ftp {

namespace {

typedef void (*conv_fn)(SplitConvArgs);
conv_fn conv_kernel(int k, int nb)
{
    if (k == 3) return nb == 1 ? sp::conv_split_kernel<3, 1> : nb == 2 ? sp::conv_split_kernel<3, 2> : sp::conv_split_kernel<3, 4>;
    return nb == 1 ? sp::conv_split_kernel<1, 1> : nb == 2 ? sp::conv_split_kernel<1, 2> : sp::conv_split_kernel<1, 4>;
}

int helper_blocks(long long total) { return (int)std::min<long long>((total + 255) / 256, (long long)kSmCount * 16); }

}  // namespace

bool split_prepare_device()
{
    for (int k : {1, 3})
        for (int nb : {1, 2, 4})
            if (cudaFuncSetAttribute(conv_kernel(k, nb), cudaFuncAttributeMaxDynamicSharedMemorySize, kSplitSmemBudget) != cudaSuccess) return false;
    return cudaFuncSetAttribute(sp::fgrad_split_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kSplitSmemBudget) == cudaSuccess;
}

void split_launch_conv(const SplitConvArgs& a, int nb, int blocks, int smem, LaunchStream ls)
{
    launch(conv_kernel(a.K, nb), blocks, sp::kConvThreads, one_block_smem(smem), ls, a);
}

void split_launch_fgrad(const SplitFgArgs& a, int blocks, int smem, LaunchStream ls)
{
    launch(sp::fgrad_split_kernel, blocks, sp::kFgThreads, one_block_smem(smem), ls, a);
}

void split_launch_planes(const float* src, uint4* dst, const SplitGeom& g, int C, LaunchStream ls)
{
    launch(sp::split_planes_kernel, helper_blocks((long long)g.planes * g.tp), 256, 0, ls, src, dst, g, C);
}

void split_launch_delta(const SplitDeltaArgs& a, LaunchStream ls)
{
    launch(sp::split_delta_kernel, helper_blocks((long long)a.low.planes * a.low.tp), 256, 0, ls, a);
}

void split_launch_pack(const PackTilesArgs& a, const float* params, LaunchStream ls)
{
    launch(sp::pack_split_kernel, a.tiles, 256, 0, ls, a, params);
}

}  // namespace ftp
