// Launches whose start overlaps the end of the launch before them on the stream
// (programmatic stream serialization), shared by the window and surrogate
// kernels.
#pragma once

#include <cuda_runtime.h>

#include "internal.h"

namespace tvbx {

// At the head of a kernel that launch_next starts: until this returns, the launch
// before it may still run, and a block reads only its arguments and tables that
// the host wrote. No launch_dependents: with it, the next launch's blocks take
// slots early and unevenly, and the windows of a 1,500 x 68 sweep went from 1.31
// to 1.50 ms instead of to 1.28.
__device__ __forceinline__ void after_last_launch() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// A launch start takes about 2 us, which short kernels would otherwise wait for
// after each other.
template <class... P, class... A>
static inline cudaError_t launch_next(void (*kern)(P...), dim3 grid, unsigned threads, size_t smem, cudaStream_t s,
                                      A... args)
{
    cudaLaunchConfig_t c = {};
    c.gridDim = grid;
    c.blockDim = dim3(threads);
    c.dynamicSmemBytes = smem;
    c.stream = s;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    c.attrs = at;
    c.numAttrs = 1;
    note_launch();
    return cudaLaunchKernelEx(&c, kern, P(args)...);
}

}  // namespace tvbx
