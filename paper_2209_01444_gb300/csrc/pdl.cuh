// Programmatic dependent launch: a kernel is launched before its predecessor
// on the stream has drained, so that its launch and the start of its CTAs overlap
// the predecessor's last wave.
#pragma once

#include <cuda_runtime.h>

#include <utility>

namespace lbm {

// Lets the stream's next kernel, if launched as a dependent, start.
__device__ __forceinline__ void pdl_release() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

// Waits until every kernel before this one has completed and its writes are visible.
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// Both, at a kernel's start: no buffer is touched before it.  The wait comes first,
// so that one kernel at most is resident ahead of its turn.  Released before the
// wait, every kernel queued behind would take what slots are free, and the CTAs of
// each would come to lie on few SMs: 30,000 pixels of 256 channels projected to 8
// fields, call after call, 50 us against 18 (22 without programmatic launches); two
// flow steps of 4 x 8000 nodes with four walls 49 against 23 (31).  The same happens
// on a smaller scale to a kernel released by one that leaves many slots free for long:
// such a one waits here and releases near its end (k_proj_fwd_vec; k_flow_multi
// before a wall pass).  k_conv_roll, which fills every SM, releases first.
__device__ __forceinline__ void pdl_begin()
{
    pdl_wait();
    pdl_release();
}

// Launches `kernel` on s as a programmatic dependent of the kernel before it.
template <class... Par, class... Arg>
cudaError_t launch_pdl(void (*kernel)(Par...), dim3 grid, dim3 block, size_t smem, cudaStream_t s, Arg&&... arg)
{
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = s;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kernel, std::forward<Arg>(arg)...);
}

}  // namespace lbm
