// Launches that overlap the end of the kernel before them on the stream
// (programmatic dependent launch).  A step is a chain of short kernels, each
// reading what the one before wrote; on small meshes the launch gap and the
// row tables a block builds first are a large part of each.  A chained kernel
// allows its successor to start as soon as its own blocks have started
// (chain_begin), builds what depends on the mesh and the projector tables
// alone, and waits for its predecessor to be complete and visible (chain_wait)
// before it touches a state, a coefficient or a counter.  Every thread of a
// chained kernel calls chain_wait before it leaves, so it never completes
// before its predecessor; a kernel launched without the attribute waits for
// all of it.  32^3 x 4 complex128: 16.4 to 12.5 us per application; 48^3 x 16
// with projectors 36.9 to 33.3 us.  Where it does not pay: the projector scatter
// (its early blocks hold registers the stencil's last blocks need: 192^3 + 3%)
// and the coefficients in front of the plain kernels (+15%) launch as usual.
#pragma once

#include <cuda_runtime.h>

#include <utility>

namespace rsg {

__device__ __forceinline__ void chain_begin() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void chain_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

template <typename... P, typename... A>
cudaError_t launch_chained(void (*kernel)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, bool chained,
                           A &&...args) {
    cudaLaunchConfig_t c = {};
    c.gridDim = grid;
    c.blockDim = block;
    c.dynamicSmemBytes = smem;
    c.stream = st;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    c.attrs = at;
    c.numAttrs = chained ? 1 : 0;
    return cudaLaunchKernelEx(&c, kernel, P(args)...);
}

}  // namespace rsg
