// Programmatic dependent launch: a kernel launched with launch_pdl may be placed on the SMs
// while the kernel before it in the stream still runs.  It calls pdl_wait() before it touches
// global memory, which returns when the kernel before it has completed and its writes are
// visible (so buffers may be read and rewritten as after an ordinary launch), then
// pdl_trigger(), which allows the kernel after it to be placed as soon as every block of this
// one has started.  The trigger comes after the wait, so that at most two grids overlap.  What
// the grids before it write is not read-only data for such a kernel, although it reads it only
// after the wait: its loads are plain ones (__ldca), not ld.global.nc (__ldg).
// Both are no-ops without the launch attribute.  What overlaps is the launch itself, 1 to
// 2 us; us per window without and with it: 384 x 4 D2Q9 50 steps 323 and 204, 331 x 203 x 2 737
// and 633, 64^2 FP64 20 steps of four stage kernels 888 and 692, 256^2 x 16 50 steps 2447 and
// 2360, 75 x 50 x 61 D3Q27 20 steps 1613 and 1582.
#pragma once

#include <cuda_runtime.h>

namespace evlbm {

// SMs of the device (152 where there is none to ask).
inline int sm_count()
{
    static const int sms = [] {
        int dev = 0, n = 0;
        const bool ok = cudaGetDevice(&dev) == cudaSuccess &&
                        cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) == cudaSuccess;
        return ok && n > 0 ? n : 152;
    }();
    return sms;
}

__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void pdl_trigger() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

template <class... P, class... Q>
cudaError_t launch_overlap(bool overlap, void (*kernel)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t st,
                           Q... args)
{
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = overlap ? 1 : 0;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    const cudaError_t e = cudaLaunchKernelEx(&cfg, kernel, static_cast<P>(args)...);
    if (e != cudaSuccess) cudaGetLastError();      // reported here: not left for a later call to find
    return e;
}
template <class... P, class... Q>
cudaError_t launch_pdl(void (*kernel)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, Q... args)
{
    return launch_overlap(true, kernel, grid, block, smem, st, args...);
}

}  // namespace evlbm
