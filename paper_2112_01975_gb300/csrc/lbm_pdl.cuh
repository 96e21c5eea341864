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
// Measured (us a step, with and without): D2Q9 FP32 64^2 2.82 / 2.92, 128^2
// 2.84 / 3.26, 256^2 3.82 / 3.60, 384^2 4.85 / 4.63, 512^2 6.76 / 7.09; FP64 64^2
// 7.9 / 8.3, 96^2 14.9 / 8.5; D3Q27 FP32 TMA-staged (one block per SM) 32^3 9.6 /
// 10.1, 64^3 19.7 / 20.4, 128^3 105.1 / 105.2; FP16-shifted 32^3 23.3 / 21.3. So
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
