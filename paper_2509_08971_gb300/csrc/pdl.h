// Programmatic dependent launch (sm_90 and later).  A kernel launched with
// programmatic stream serialization may begin while the kernel before it in
// the stream is still running, so its launch latency and set-up overlap that
// kernel.  Such a kernel calls griddep_wait() before its first access to memory
// that an earlier kernel reads or writes (a hardware wait for that grid to complete
// and its writes to be visible, not a spin), and griddep_launch_dependents() when
// the next such kernel may take free slots of the chip and wait there in its turn;
// that one does nothing else before this grid is complete, so the trigger's place
// changes no order, only where the next blocks land.  Without the call each block
// releases at its exit, which is best for grids of up to about a wave, whose free
// slots are unevenly spread (FP64 WENO sweeps of 47 x 25 x 35: 1.67 ms a step, 2.40
// with the call at the head; 256^2 shear layer 0.53 against 0.55).  At the head is
// best where blocks fill their SMs (the 3D stage, by shared memory: 1.03 against
// 1.04 ms at 150 x 117 x 93), for a grid of one block, and for memory-bound grids of
// two waves and more.
// Such a kernel loads what others write with plain loads: not __ldg and not
// through __restrict__ pointers, which a compiler may move above the wait and the
// read-only path need not keep coherent while the grids overlap.
// Chains of short dependent kernels (the time loop, the adjoint's passes, the multigrid
// levels) lose most of their launch gaps this way.
#pragma once
#include <cuda_runtime.h>

#include <utility>

namespace hh {

__device__ __forceinline__ void griddep_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void griddep_launch_dependents() {
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

__device__ __forceinline__ bool griddep_many_blocks() {
    return gridDim.x * gridDim.y * gridDim.z >= 2u * 6u * 152u;
}

template <typename... KArgs, typename... Args>
inline cudaError_t launch_pdl(void (*kern)(KArgs...), dim3 grid, dim3 block, size_t smem,
                              cudaStream_t s, Args&&... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    const cudaError_t e = cudaLaunchKernelEx(&cfg, kern, std::forward<Args>(args)...);
    if (e != cudaSuccess) cudaGetLastError();          // returned to the caller, not left behind
    return e;
}

}  // namespace hh
