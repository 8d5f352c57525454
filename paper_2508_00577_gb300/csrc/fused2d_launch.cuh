// Kernels and launch of the fused single-pass D2Q9 step, templated on the storage type
// ST (float, or __half / __nv_bfloat16 deviations): one launch per time step, one CTA per
// tile (strip x chunk x layer) or the balanced persistent grid.  Included by fused2d.cu
// (FP32 storage) and fused2d16.cu (16-bit storage), which instantiate it.
#pragma once

#include "fused2d_tile.cuh"
#include "pdl.cuh"

namespace evlbm {
namespace fused2d_impl {

using namespace fused;

template <int kW, bool THERMAL, bool WALLS, typename ST>
__global__ void __launch_bounds__(threads_of<kW>(), Shape<kW>::MINB) k_fused2d(FusedArgs A)
{
    extern __shared__ v2 smem[];
    pdl_wait();
    pdl_trigger();
    const int y0 = blockIdx.y * A.H;                       // H is even
    fused_tile<kW, THERMAL, WALLS, ST>(A, blockIdx.x, y0, min(A.H, A.ny - y0), A.z0 + (int)blockIdx.z, smem);
}

// Balanced persistent variant: a grid of S x parts CTAs (S strips, parts = the
// resident CTAs of the GPU / S), CTA b taking strip b % S and the equal share b / S of
// that strip's row pairs over all layers (layer after layer).  Neighbouring strips
// then march over the same rows at the same time, as in the chunked grid, so the
// halo columns they share are re-read from L2 and each row is fetched from DRAM in
// one stretch.  A share that crosses the end of a layer becomes two tiles.
template <int kW, bool THERMAL, bool WALLS, typename ST>
__global__ void __launch_bounds__(threads_of<kW>(), Shape<kW>::MINB) k_fused2d_bal(FusedArgs A)
{
    extern __shared__ v2 smem[];
    pdl_wait();
    pdl_trigger();
    const int S = (A.nx + kW - 1) / kW, P = (A.ny + 1) / 2;
    const int parts = gridDim.x / S, strip = blockIdx.x % S, part = blockIdx.x / S;
    const long long T = (long long)A.nz * P;                 // row pairs of one strip, all layers
    const long long g1 = T * (part + 1) / parts;
    for (long long g = T * part / parts; g < g1;) {
        const int layer = (int)(g / P);
        const int p0 = (int)(g - (long long)layer * P);
        const int p1 = (int)min((long long)P, p0 + (g1 - g));
        const int y0 = 2 * p0;
        fused_tile<kW, THERMAL, WALLS, ST>(A, strip, y0, min(2 * p1, A.ny) - y0, layer, smem);
        __syncthreads();
        g += p1 - p0;
    }
}

// A grid of chunks by layers takes at most kGridYZ of either: taller chunks where there would
// be more of them, and larger stacks in parts.
constexpr int kGridYZ = 65535;
template <class ARGS, class F> cudaError_t in_layers(ARGS A, int nz, F launch_part)
{
    while ((A.ny + A.H - 1) / A.H > kGridYZ) A.H *= 2;
    for (; A.z0 < nz; A.z0 += kGridYZ) {
        const cudaError_t e = launch_part(A, min(nz - A.z0, kGridYZ));
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

// Macroscopic fields of the current state: stages A to C of the step in one pass, reading the
// populations once and writing the fields (72 + 16 bytes per node with FP32 storage).  The
// four stage kernels it replaces passed through ~20 scratch fields per node: 555 us on nine
// thermal 1024^2 layers (moments 141, stress 88, macro 153, export 173).
template <int kW, bool THERMAL, bool WALLS, typename ST>
__global__ void __launch_bounds__(threads_of<kW>(), (kW == 64 ? 6 : 4) - (WALLS || Store<ST>::dev ? (kW == 64 ? 2 : 1) : 0))
    k_moments2d(MomentArgs A)
{
    extern __shared__ v2 smem[];
    pdl_wait();
    const int y0 = blockIdx.y * A.H;                       // H is even
    fused_tile<kW, THERMAL, WALLS, ST>(A, blockIdx.x, y0, min(A.H, A.ny - y0), A.z0 + (int)blockIdx.z, smem);
}

// Chunks of 32 rows at most (16 row pairs after 3 that fill the pipeline), shorter while the
// grid would leave SMs without a CTA; narrow strips on narrow lattices.
template <bool THERMAL, bool WALLS, typename ST>
cudaError_t launch_moments(MomentArgs A, int nz, cudaStream_t st)
{
    const int W = A.nx > 64 ? 128 : 64, S = (A.nx + W - 1) / W;
    A.H = 32;
    while (A.H > 4 && (long long)S * ((A.ny + A.H - 1) / A.H) * nz < 3 * sm_count()) A.H >>= 1;
    return in_layers(A, nz, [&](const MomentArgs &B, int layers) {
        const dim3 grid(S, (B.ny + B.H - 1) / B.H, layers);
        return W == 64 ? launch_pdl(k_moments2d<64, THERMAL, WALLS, ST>, grid, threads_of<64>(), moments_smem_of<64>(), st, B)
                       : launch_pdl(k_moments2d<128, THERMAL, WALLS, ST>, grid, threads_of<128>(), moments_smem_of<128>(), st,
                                    B);
    });
}

// One step.  A step that follows a step of its context overlaps that one's end (pdl.cuh); the
// first after other work does not.  Overlapping grids keep the places of the grid before: the
// CTAs of a grid that leaves slots of the SMs free would else be placed around those of, say,
// the kernel that set the populations, several on the SMs that have slots at that moment, and
// all steps after it would keep to these SMs.  331 x 203 x 2 (136 CTAs), reset, 50 steps and
// fields: 758 us with every step overlapping, 638 so, 737 with none.  (Claiming the rest of an
// SM's shared memory, so that no second CTA fits beside the first, gave 647, but kept the grids
// of other streams out too: eight such lattices at once 104 us a step, now 59.)
template <int W, bool THERMAL, bool WALLS, typename ST>
cudaError_t launch_w(const FusedArgs &A, int nz, bool balanced, bool follows, cudaStream_t st)
{
    static bool attr = false;
    static int resident = 0;
    constexpr size_t smem = smem_of<W>();
    if (!attr) {
        cudaError_t e = cudaFuncSetAttribute(k_fused2d<W, THERMAL, WALLS, ST>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             (int)smem);
        if (e == cudaSuccess)
            e = cudaFuncSetAttribute(k_fused2d_bal<W, THERMAL, WALLS, ST>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                     (int)smem);
        int per_sm = 0;
        if (e == cudaSuccess)
            e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_fused2d_bal<W, THERMAL, WALLS, ST>,
                                                              threads_of<W>(), smem);
        if (e != cudaSuccess) return e;
        if (per_sm < 1) return cudaErrorLaunchOutOfResources;
        resident = per_sm * sm_count();
        attr = true;
    }
    // Wall columns make the CTAs of a strip's two ends longer than the others (they solve for the
    // wall's density).  Where about all slots are taken, the next grid's CTAs would fill them in the
    // order in which this one's end, the long ones last and together: 512^2 x 4 layers 75.0 us a
    // step overlapping and 72.9 apart, 1024^2 x 4 in strips of 128 and chunks of 128 rows 269 and
    // 259; but 130 x 130 7.9 and 10.2, and 2048 CTAs (64 x 32) 232 and 235.
    auto overlaps = [&](long long ctas) {
        return follows && !(WALLS && 2 * ctas > resident && ctas < 2LL * resident);
    };
    if (balanced) {
        const int S = (A.nx + W - 1) / W;
        const long long parts = min((long long)max(resident / S, 1), (long long)nz * ((A.ny + 1) / 2));
        return launch_overlap(overlaps(S * parts), k_fused2d_bal<W, THERMAL, WALLS, ST>, dim3((unsigned)(S * parts)),
                              threads_of<W>(), smem, st, A);
    }
    return in_layers(A, nz, [&](const FusedArgs &B, int layers) {
        const dim3 grid((B.nx + W - 1) / W, (B.ny + B.H - 1) / B.H, layers);
        return launch_overlap(overlaps((long long)grid.x * grid.y * grid.z), k_fused2d<W, THERMAL, WALLS, ST>, grid,
                              threads_of<W>(), smem, st, B);
    });
}

template <bool THERMAL, bool WALLS, typename ST>
cudaError_t launch(int W, const FusedArgs &A, int nz, bool balanced, bool follows, cudaStream_t st)
{
    switch (W) {
    case 64: return launch_w<64, THERMAL, WALLS, ST>(A, nz, balanced, follows, st);
    case 96: return launch_w<96, THERMAL, WALLS, ST>(A, nz, balanced, follows, st);
    case 192: return launch_w<192, THERMAL, WALLS, ST>(A, nz, balanced, follows, st);
    default: return launch_w<128, THERMAL, WALLS, ST>(A, nz, balanced, follows, st);
    }
}

// Kernel arguments of a lattice (populations, records and the T field as passed by the caller).
inline FusedArgs make_args(const KParams &p, const void *f, const void *g, void *fo, void *go, const void *RT_iso,
                           const void *Rin, void *Rout)
{
    FusedArgs A;
    A.f = static_cast<const float *>(f);
    A.g = static_cast<const float *>(g);
    A.fo = static_cast<float *>(fo);
    A.go = static_cast<float *>(go);
    A.Rin = static_cast<const float *>(Rin);
    A.Rout = static_cast<float *>(Rout);
    A.RT_iso = static_cast<const float *>(RT_iso);
    A.nx = p.nx;
    A.ny = p.ny;
    A.nz = p.nz;
    A.N = (unsigned)p.N;
    A.eos = p.eos;
    A.a = float(p.a);
    A.b = float(p.b);
    A.kappa = float(p.kappa);
    A.lambda = float(p.lambda);
    A.c_eq = float(p.c_eq);
    A.c_star = float(p.c_star);
    A.walls = p.walls;
    A.wall_uy[0] = float(p.wall_u[0][1]);
    A.wall_uy[1] = float(p.wall_u[1][1]);
    A.wall_RT = float(p.wall_RT);
    A.z0 = 0;
    return A;
}

// Arguments of the moments kernel: a state, outputs (any may be NULL) and the gas constant T is
// divided by (1: R T itself).
inline MomentArgs moment_args(const KParams &p, const void *f, const void *g, const void *RT_iso, const void *Rin,
                              const MomentOut &o)
{
    MomentArgs A;
    static_cast<FusedArgs &>(A) = make_args(p, f, g, nullptr, nullptr, RT_iso, Rin, nullptr);
    A.m_rho = o.rho;
    A.m_u = o.u;
    A.m_T = o.T;
    A.m_F = o.F;
    A.R = GasConstant(o.R);
    return A;
}

// Launch shape of a step: strip width W and chunk height (A.H); balanced persistent grid.
inline void launch_shape(const KParams &p, FusedArgs &A, int &W, bool &balanced)
{
    int H = p.tile_h;
    W = p.tile_w;
    if (W <= 0 || (H <= 0 && H != kTileBalanced)) fused2d_default_tile(p, &W, &H);
    balanced = H == kTileBalanced;
    A.H = balanced ? 0 : H + (H & 1);  // row pairs: chunks of an even number of rows
}

}  // namespace fused2d_impl
}  // namespace evlbm
