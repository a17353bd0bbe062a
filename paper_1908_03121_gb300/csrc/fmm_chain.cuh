// Launching the kernels of a dependent chain (the levels of the upward and
// downward passes, the leaf pass, the sums).
//
// Such a kernel is launched with programmatic stream serialization: its CTAs
// may become resident, and read the tree's tables (which no kernel writes),
// while the kernel before it on the stream drains.  Every one of them calls
// chain_begin() before it touches anything that an earlier kernel wrote or
// still reads: it waits until the kernel before has completed with all its
// stores visible, then lets the next one start its own prologue.  A kernel that
// calls it before its predecessor's completion has waited for that one too, so
// the order holds along the whole chain.
// What earlier kernels write changes while such a kernel is resident, so its
// parameters carry no __restrict__ but for the tables: the compiler could move
// accesses through it before the wait, and with const use the non-coherent load
// path (tests/test_chained_kernels.py).  Functions called after chain_begin()
// may promise it again for what they store.
// Upward pass of a level-6 binary 107 -> 93 us, downward pass and forces 257 ->
// 236 us, step of 73 sub-grids 157 -> 148 us (of which the queue reset in P2M
// instead of a memset, and the leaf pass on the main stream instead of behind two
// event waits, are part).
#pragma once

#include <cuda_runtime.h>

namespace fmm {

#ifdef __CUDACC__
__device__ __forceinline__ void chain_begin()
{
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

// a load past L1 that stays behind barriers and fences: of what other CTAs wrote
__device__ __forceinline__ double load_cg(const double *p)
{
    double v;
    asm volatile("ld.global.cg.f64 %0, [%1];" : "=d"(v) : "l"(p) : "memory");
    return v;
}

template <class... Params, class... Args>
cudaError_t launch_chained(void (*kern)(Params...), dim3 grid, dim3 block, cudaStream_t s, Args... args)
{
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.stream = s;
    cfg.attrs = &at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kern, static_cast<Params>(args)...);
}
#endif

}  // namespace fmm
