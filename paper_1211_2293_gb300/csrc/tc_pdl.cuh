// tc_pdl.cuh -- programmatic dependent launch: a kernel launched by pdl_launch
// may be resident before the kernel before it in the stream has ended; it
// starts by pdl_begin, which lets the next one come and waits until the one
// before has ended and its writes are visible.  Every kernel of a chain begins
// so, before any access to memory: the wait for the one before is then a wait
// for all before it.  Their pointers are not __restrict__: a load through a
// const __restrict__ pointer counts as one of constant memory, which the
// compiler may move up past the wait.
#pragma once
#include <cuda_runtime.h>

#include "tc_internal.cuh"

namespace tc {

namespace {

__device__ __forceinline__ void pdl_begin()
{
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    asm volatile("griddepcontrol.wait;" ::: "memory");
}

template <typename... P, typename... A>
void pdl_launch(void (*kernel)(P...), int64_t grid, int block, size_t smem, ChainStream s, A... a)
{
    cudaLaunchConfig_t c{};
    c.gridDim = dim3((unsigned)grid);
    c.blockDim = dim3((unsigned)block);
    c.dynamicSmemBytes = smem;
    c.stream = s.s;
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    c.attrs = &at;
    c.numAttrs = s.chain ? 1 : 0;
    cudaLaunchKernelEx(&c, kernel, static_cast<P>(a)...);
}

}  // namespace

}  // namespace tc
