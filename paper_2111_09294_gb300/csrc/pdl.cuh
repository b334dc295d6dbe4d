// Programmatic dependent launch.  The kernels of the iteration loop are
// launched with programmatic stream serialisation: a kernel's blocks may be
// launched while its predecessor still runs, once every block of the
// predecessor has triggered (pdl_trigger) or exited, and they wait (pdl_wait,
// griddepcontrol.wait) for the predecessor's completion and memory before
// touching anything it wrote.  A kernel triggers only after its own wait: so
// when its successor's blocks run, everything up to the kernel before the
// predecessor is complete, and the successor may read, before its own wait,
// set-up data and, from L2 (ld_early: it is the wait that makes earlier writes
// visible to ordinary loads), whatever the predecessor does not write.  That
// is what the early launch is for: the blocks that fill an SM as it drains
// load the next kernel's factors, bases and matrix stages meanwhile.  The wait
// is a no-op for a kernel launched without the attribute.
//
// The dense inverse (set-up) departs from this: its pivot and panel kernels
// trigger as their first step, so that a launch independent of them starts
// beside them, and that one waits only at its end, in one block, so that what
// follows both follows.  That is sound because the kernels that trigger so are
// themselves launched without the attribute (all before them is complete when
// they start), and so is whatever follows the one beside them.  A kernel
// launched with the attribute must not trigger before its wait.
//
// Triggers pay where measured: in the FP32 product, the coarse solve and (up
// to kTriggerBlocks blocks) the prolongation, 31.8 against 35.3 us per FP32
// iteration at 12^3 and 50.4 against 52.7 at 32^3.  In the FP32 restriction
// (the coarse solve's loads of E^-1 then compete with it: 90 against 85 us at
// 48^3), in a large prolongation (79.4 against 78.0 us at 48^3) and in the
// FP64 kernels (up to 258 against 231 us at 48^3) they cost time.
#pragma once

#include <cuda_runtime.h>

namespace xdcg {

__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void pdl_trigger() {
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

template <typename... KArgs, typename... Args>
cudaError_t launch_pdl(void (*kernel)(KArgs...), dim3 grid, int block, size_t smem,
                       cudaStream_t st, Args... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = dim3((unsigned)block);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kernel, static_cast<KArgs>(args)...);
}

}  // namespace xdcg
