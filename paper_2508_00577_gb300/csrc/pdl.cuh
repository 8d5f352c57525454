// Programmatic dependent launch: a kernel launched with launch_pdl may be placed on the SMs
// while the kernel before it in the stream still runs.  It calls pdl_wait() before it touches
// global memory, which returns when the kernel before it has completed and its writes are
// visible (so buffers may be read and rewritten as after an ordinary launch), then
// pdl_trigger(), which allows the kernel after it to be placed as soon as every block of this
// one has started.  (The trigger comes after the wait, so that at most two grids overlap and
// the L1 lines a grid cached of a buffer are dropped before a later grid reads it rewritten.)
// Both are no-ops without the launch attribute.  What overlaps is the launch itself, 1 to
// 2 us; us per window: 384 x 4 D2Q9 50 steps 320 -> 204, 64^2 FP64 20 steps of four stage
// kernels 885 -> 694, 256^2 x 16 50 steps 2504 -> 2407, 75 x 50 x 61 D3Q27 20 steps 2041 -> 1950.
#pragma once

#include <cuda_runtime.h>

namespace evlbm {

__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void pdl_trigger() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

// Dynamic shared memory of a kernel whose grid leaves slots of the SMs free: as much as keeps
// one more CTA than the grid's share from fitting on an SM.  Otherwise the next grid's CTAs
// would be placed while this one still runs, several on the SMs that happen to have free slots,
// and stay there (136 CTAs of the 331 x 203 x 2 lattice on 152 SMs: 818 us per 50 steps, 660
// with one CTA per SM handing over to the next, 736 without overlap).  The D3Q27 kernel loses
// more by the smaller L1 than it gains (75 x 50 x 61: 1950 us, 2021 with this), and the FP64
// stage kernels gain nothing (694, 690), so neither uses it.
constexpr size_t kSmemPerSM = 233472, kSmemPerCta = 1024;
inline size_t handoff_smem(size_t smem, long long ctas, int sms)
{
    const long long r = (ctas + sms - 1) / sms;
    if (r > 3) return smem;
    const size_t least = kSmemPerSM / (size_t)(r + 1) - kSmemPerCta + 128;
    return smem > least ? smem : least / 128 * 128;
}
constexpr size_t kHandoffMax = kSmemPerSM / 2;

template <class... P, class... Q>
cudaError_t launch_pdl(void (*kernel)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, Q... args)
{
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
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

}  // namespace evlbm
