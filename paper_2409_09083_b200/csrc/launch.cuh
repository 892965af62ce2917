// Launches that follow one another on a stream overlap at their edges (programmatic dependent launch).  A step is a chain of 10
// to 60 launches of 5 to 200 us, and between two of them every SM used to idle from the end of its last block to the end of the
// slowest one, then through the launch, the set-up of the block (barriers, tensor memory, up to 200 KB of zeros) and the
// first copies.
//
// The rules.  EVERY kernel calls previous_launches() before its first access to global memory: it returns when all launches
// before it on the stream have completed and their writes are visible.  Since every kernel waits, a kernel's completion implies
// that of all before it, so only the previous launch has to be waited for, and a buffer is never written before its
// readers are through.  A launch behind an event or a copy, or with `overlap` off (per-launch timing), starts as any
// launch does.
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
