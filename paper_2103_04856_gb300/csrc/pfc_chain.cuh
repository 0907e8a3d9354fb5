// pfc_chain.cuh -- launches that follow one another on a stream without a gap:
// the next kernel's blocks start while the one before drains (programmatic
// dependent launch) and wait for it before they touch memory.
//
// Every kernel launched with `chained` calls chain_wait() first, in every
// thread: its end then implies the end of all before it.  For the two kernels of
// a small FP64 step, about 10 us each, between which the launch shows (a 32^3
// run of 100 steps 2265 -> 2050 us).  The FP32 sweep, whose blocks fill their SM,
// and the kernels of Alg. 1 (100^3: 2667 and 2698 us) gain nothing from it.
#pragma once

#include <cuda_runtime.h>

namespace pfc {

// The kernels before on the stream have ended and their writes are visible;
// from here on the next one's blocks may take the room that this one leaves.
__device__ __forceinline__ void chain_wait()
{
    asm volatile("griddepcontrol.wait;\n\tgriddepcontrol.launch_dependents;" ::: "memory");
}

// A pointer as one that is known only from here on: loads through it, read-only
// ones too, stay after chain_wait().
template <typename P>
__device__ __forceinline__ P* after_wait(P* p)
{
    asm volatile("" : "+l"(p)::"memory");
    return p;
}

// chained: what is before on the stream is a kernel of this library, enqueued by the same call.
template <typename... P, typename... A>
cudaError_t launch_chained(bool chained, void (*kernel)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t s, const A&... args)
{
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t c{};
    c.gridDim = grid;
    c.blockDim = block;
    c.dynamicSmemBytes = smem;
    c.stream = s;
    c.attrs = &at;
    c.numAttrs = chained ? 1 : 0;
    return cudaLaunchKernelEx(&c, kernel, args...);
}

}  // namespace pfc
