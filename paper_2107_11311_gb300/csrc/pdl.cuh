// Programmatic dependent launch: a kernel launched with launch_after may have its
// CTAs placed, and run up to its pdl_wait, while the last CTAs of the kernel
// before it finish; pdl_wait returns when that kernel is complete and its writes
// are visible. A step is a chain of short kernels, and this hides about 1 us of
// launch latency between two of them (192 atoms from host arrays, 6 kernels: 69 ->
// 57 us a call; MD of 1,536 atoms: 50.2 -> 47.6 us a step).
//
// Every kernel launched this way calls pdl_wait before it touches global memory
// that another kernel of the chain reads or writes (launched without the
// attribute the call does nothing), and lets its own successor start after that:
// whatever came before its predecessor is then complete for the successor too.
//
// The kernel runs while its predecessor still writes, so what it reads of it is not
// read-only memory. Loads through a __restrict__ parameter are not bound by the wait's
// memory clobber (nothing else may alias them), and those through a `const
// __restrict__` one may become non-coherent loads besides: either could be moved above
// the wait. Pointers to memory that an earlier kernel of the chain writes are therefore
// declared without __restrict__; plain loads through them, and the volatile load
// intrinsics, stay below the wait. Never __ldg: it reads through the non-coherent path.
// What no kernel of an evaluation writes (network parameters, batch layouts, species)
// needs none of this.
#pragma once

#include <cuda_runtime.h>

#include <utility>

namespace aenet {

__device__ __forceinline__ void pdl_wait() {
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

// on: false gives an ordinary launch (inside conditional bodies and between event
// records of a captured step, whose nodes are no kernels).
template <class... P, class... A>
inline cudaError_t launch_after(bool on, void (*kern)(P...), int grid, int block, size_t smem, cudaStream_t stream,
                                A &&...args) {
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((unsigned)grid);
    cfg.blockDim = dim3((unsigned)block);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = on ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, kern, std::forward<A>(args)...);
}

}  // namespace aenet
