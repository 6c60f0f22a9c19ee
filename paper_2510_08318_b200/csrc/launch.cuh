// Kernels launched one behind the other on a stream without the gap between them: programmatic dependent launch.
//
// A kernel of a chain starts with pdl_trigger() (the next kernel's CTAs may take their places as soon as SMs become free) and
// pdl_wait() (returns when every kernel before it has completed and its writes are visible).  Everything before pdl_wait() is
// set-up that touches no global memory; everything after it is ordered as in an ordinary launch, so what a kernel may read
// and overwrite does not change.  Every CTA waits, so a kernel cannot complete before those in front of it and the order
// holds along the whole chain.
// Measured: ten launches, B=2 H=3 n=777 d=64 fp32 forward + backward 121.2 -> 110.7 us; three, B=1 H=2 n=1024 d=64 fp32 forward 25.0 ->
// 23.4 us; six, B=1 H=12 n=32760 d=128 bf16 backward 255.1 -> 251.6 us.
#pragma once
#include <cuda_runtime.h>

#include <utility>

namespace linattn {

__device__ __forceinline__ void pdl_trigger() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

struct ChainedLaunch {
    cudaLaunchAttribute attr[1];
    cudaLaunchConfig_t cfg{};
    ChainedLaunch(dim3 grid, dim3 block, size_t smem, cudaStream_t stream)
    {
        attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        attr[0].val.programmaticStreamSerializationAllowed = 1;
        cfg.gridDim = grid;
        cfg.blockDim = block;
        cfg.dynamicSmemBytes = smem;
        cfg.stream = stream;
        cfg.attrs = attr;
        cfg.numAttrs = 1;
    }
};
template <class... P, class... A>
inline cudaError_t launch_chained(void (*kernel)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t stream, A&&... args)
{
    ChainedLaunch l(grid, block, smem, stream);
    return cudaLaunchKernelEx(&l.cfg, kernel, std::forward<A>(args)...);
}
inline cudaError_t launch_chained_ptr(const void* kernel, dim3 grid, dim3 block, void** args, size_t smem, cudaStream_t stream)
{
    ChainedLaunch l(grid, block, smem, stream);
    return cudaLaunchKernelExC(&l.cfg, kernel, args);
}

}  // namespace linattn
