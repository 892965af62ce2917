// Launches that follow one another on a stream overlap at their edges (programmatic dependent launch).  A step is a chain of 10
// to 60 launches of 5 to 200 us, and between two of them every SM used to idle from the end of its last block to the end of the
// slowest one, then through the launch, the set-up of the block (barriers, tensor memory, up to 200 KB of zeros) and the
// first copies.
//
// The rules.  Every kernel that launch() below starts calls previous_launches() before its first access to global memory: it
// returns when all launches before it on the stream have completed and their writes are visible.  Since each of them waits, a
// kernel's completion implies that of all before it, so only the previous launch has to be waited for, and a buffer is
// never written before its readers are through.  A launch behind an event or a copy, with `overlap` off (per-launch
// timing), or without launch() (sgd_kernel, fma_peak_kernel, wait_probe_kernel, noalloc.cu) starts as any launch does, when all before it have
// ended.
//
// A kernel that takes tensor memory calls next_launch() only when its whole block is behind the allocation.  The next launch
// may take all columns of an SM before it waits for this one, and tcgen05.alloc waits without a limit: a block of this
// launch that had let it in without having its own columns would wait for columns that are given back only after it
// has ended.  With the rule, whoever waits in an allocation waits for earlier launches alone, and these have what they need
// (a launch starts only when all blocks of the one before have triggered or ended, so this holds along the stream,
// helpers in between included; launches of other streams that share the SM depend on their own stream only).
//
// next_launch() lets the blocks of the next launch onto SMs that have room before this launch has ended.  Kernels whose blocks
// fill the GPU once and end together gain from it when they are short; long ones lose, because the next kernel's blocks then
// land on the SMs in the order in which these fall free and its neighbours in the grid, which read the same rows or
// filters, are scattered over the two dies.  So the banded kernels call it, at their end, when the tensor core works less than
// kHurryCycles per block, the fused stacks always, and never the split kernels (whose launches are six times as long), the fp32
// row kernels and the helpers of many blocks an SM.  Measured, us a step (launches as before | without next_launch in the banded
// kernels | below 20000 cycles | always): 8 layers, batch 4, bf16: 403 | 351 | 344 | 347; 16 layers, 2 x 336 x 464: 729 | 627 |
// 597 | 597; 23 layers, batch 8: 1753 | 1633 | 1602 | 1584; 16 layers, batch 16: 2916 | 2811 | 2801 | 2922 (called at the start of
// every kernel: 2963); fp32, 3 x 200 x 312: 501 | 455 (with it in the split kernels: 480); fp32, 37 x 48 x
// 56 (row kernels): 493 | 471 (with it: 656).
#pragma once

#include <cuda_runtime.h>

#include <utility>

#include "launch_stream.hpp"

namespace ftp {

constexpr double kHurryCycles = 20000.0;

__device__ __forceinline__ void next_launch() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void previous_launches() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

template <class... P, class... A>
inline void launch(void (*kernel)(P...), dim3 grid, dim3 block, size_t smem, LaunchStream ls, A&&... args)
{
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = grid; cfg.blockDim = block; cfg.dynamicSmemBytes = smem; cfg.stream = ls.st;
    cfg.attrs = &at; cfg.numAttrs = ls.overlap ? 1 : 0;
    cudaLaunchKernelEx(&cfg, kernel, std::forward<A>(args)...);       // (an error stays for the caller's cudaGetLastError)
}

// Dynamic shared memory of a kernel that takes all 512 tensor-memory columns of an SM: more than half of the 227 KB, so that
// never two of its blocks share an SM (the second would wait for the first one's columns).
constexpr size_t kOneBlockPerSm = 116 * 1024;
inline size_t one_block_smem(size_t need) { return need > kOneBlockPerSm ? need : kOneBlockPerSm; }

}  // namespace ftp
