// Programmatic dependent launch of the step's kernels.
//
// The kernels of consecutive steps run one after the other on one stream. A
// kernel launched with launch_step may begin while its predecessor's last
// blocks still run (on SMs that have room); it sets up and waits in
// step_wait() until the predecessor has finished and its writes are
// visible, before it touches what a step writes or reads. That hides the
// launch latency and the set-up, a microsecond or so per kernel. A kernel lets its
// successor start as soon as all its own blocks have (step_trigger()).
// Launched any other way, or with `overlap` false, step_wait() does not wait.
//
// So the kernel is resident while what it will read is still written: that
// data is not read-only for the kernel's lifetime, and its loads are plain
// ones, through pointers that are neither __ldg's nor const __restrict__ (the
// compiler may take those through the non-coherent path, or above the
// wait). Masks, wall bits, tensor maps and work items, which no step writes,
// may be read either way and before the wait.
//
// Blocks that wait also take up room: a successor that fits beside its
// predecessor is handed out while SMs are unevenly busy and stays that way.
// Measured (us a step, with and without): D2Q9 FP32 64^2 2.60 / 2.82, 128^2
// 2.70 / 2.84, 256^2 3.79 / 3.34, 384^2 5.13 / 4.13, 512^2 6.16 / 6.44; FP64 64^2
// 7.4 / 8.2, 96^2 11.7 / 8.1, 301x202 38.5 / 20.0; D3Q27 FP32 TMA-staged (one
// block per SM) 32^3 9.0 / 9.5, 64^3 18.9 / 19.5, 128^3 101.2 / 101.6; the shifted
// D3Q27 kernels, which lost by it (32^3 23.3 / 21.3), do not overlap. So
// it is used where two steps' blocks have an SM each or nearly (side_by_side), where
// a step's blocks leave no room for the next ones' (leaves_no_room), and not in between.
#pragma once

#include <cuda_runtime.h>

namespace lbmpdl {

__device__ __forceinline__ void step_trigger() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void step_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// Whether the blocks of two consecutive steps find an SM each, or nearly.
inline bool side_by_side(long long blocks, int sms) { return 4 * blocks <= 3ll * sms; }

template <typename... P, typename... A>
void launch_step(bool overlap, void (*kernel)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t s,
                 const A &...args)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute attr = {};
    attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr.val.programmaticStreamSerializationAllowed = overlap;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    cudaLaunchKernelEx(&cfg, kernel, static_cast<P>(args)...);   // an error is the caller's cudaGetLastError's
}

}  // namespace lbmpdl
