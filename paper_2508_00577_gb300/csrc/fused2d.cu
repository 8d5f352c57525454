// Fused single-pass D2Q9 step with FP32 storage: one launch per time step (kernels in
// fused2d_launch.cuh, tile body in fused2d_tile.cuh); 16-bit storage is instantiated in
// fused2d16.cu.
#include "fused2d_launch.cuh"

namespace evlbm {

using namespace fused2d_impl;

EVLBM_DEFINE_OOB_READER(fused2d_oob)

const int kFusedWidths[kFusedWidthCount] = {64, 96, 128, 192};

bool fused2d_supported(int prec, int Q, const KParams &p)
{
    return prec >= 1 && prec <= 3 && Q == 9 && p.force_form == 0 && (prec == 1 || !p.walls) &&
           (long long)9 * p.N < (1LL << 31);
}

// Default launch shape: the candidate with the least estimated time.  A CTA that marches p
// row pairs runs p + 5 iterations per tile (the pipeline of four stages fills first); those of
// the fill, without some of the stages, take about the time of 4 (with 5 in its place the shapes
// picked for 70 lattices take 1.107 times the best one's time on average, with 4 1.093).  The
// time of one iteration depends on the strip width and on how many CTAs share an SM.  Measured
// (us, thermal FP32, before the launches overlapped; the ratios hold for the isothermal kernel
// and 16-bit storage):
//   CTAs per SM       1     2     3     4
//   W =  64         1.28  1.60  2.20  2.90
//   W =  96         1.20  2.25
//   W = 128         1.50  2.35
// so few row pairs per CTA win as long as the GPU is not full, and beyond that the wide
// strips of the balanced grid.  Against strips of 128 columns and 128 rows a CTA, us per step
// (the launches overlapping, too): 331 x 203 x 2 104.6 -> 12.5, 512^2 102.4 -> 16.7, 256^2 x 16
// 123.0 -> 46.6, 1024^2 122.7 -> 42.8, 256^2 x 64 161.6 -> 149.8, 64^2 45.1 -> 5.4, 384 x 4
// isothermal 8.2 -> 4.0.
void fused2d_default_tile(const KParams &p, int *W, int *H)
{
    static const int widths[3] = {128, 96, 64}, per_sm[3] = {2, 2, 4};
    static const float iter_us[3][4] = {{1.50f, 2.35f, 0.f, 0.f}, {1.20f, 2.25f, 0.f, 0.f}, {1.28f, 1.60f, 2.20f, 2.90f}};
    static const int heights[] = {2, 4, 6, 8, 12, 16, 24, 32, 48, 64, 96, 128, 256};
    constexpr int kFill = 4;
    const int sms = sm_count();
    const long long P = (p.ny + 1) / 2;                      // row pairs of a layer
    double best = 1e300;
    for (int k = 0; k < 3; ++k) {
        const long long S = (p.nx + widths[k] - 1) / widths[k], slots = (long long)sms * per_sm[k];
        auto iter = [&](long long ctas) {
            const long long r = (ctas + sms - 1) / sms;
            return (double)iter_us[k][r < 1 ? 0 : (r > per_sm[k] ? per_sm[k] : r) - 1];
        };
        auto offer = [&](double t, int h) {
            if (t < best) {
                best = t;
                *W = widths[k];
                *H = h;
            }
        };
        for (int h : heights) {
            const long long pairs = h / 2 < P ? h / 2 : P, ctas = S * ((P + pairs - 1) / pairs) * p.nz;
            const long long waves = (ctas + slots - 1) / slots;
            if ((P + pairs - 1) / pairs <= 65535) offer((double)(waves * (pairs + kFill)) * iter(ctas), h);
            if (pairs == P) break;
        }
        // Balanced grid: equal shares of the strip's row pairs; a share that crosses the end
        // of a layer fills the pipeline once more.
        const long long T = P * p.nz;
        long long parts = slots / S;
        parts = parts < 1 ? 1 : (parts > T ? T : parts);
        const long long share = (T + parts - 1) / parts, tiles = 1 + (share + P - 2) / P;
        const long long waves = (S * parts + slots - 1) / slots;
        offer((double)(waves * (share + kFill * (p.nz > 1 ? tiles : 1))) * iter(S * parts), kTileBalanced);
    }
}

cudaError_t fused2d_step(int prec, const KParams &p, const void *f, const void *g, void *fo, void *go,
                         const void *RT_iso, const void *Rin, void *Rout, cudaStream_t st)
{
    if (!fused2d_supported(prec, 9, p)) return cudaErrorNotSupported;
    if (prec != 1) return fused2d_step16(prec, p, f, g, fo, go, RT_iso, Rin, Rout, st);
    FusedArgs A = make_args(p, f, g, fo, go, RT_iso, Rin, Rout);
    int W;
    bool balanced;
    launch_shape(p, A, W, balanced);
    if (p.walls)
        return p.thermal ? launch<true, true, float>(W, A, p.nz, balanced, p.follows != 0, st)
                         : launch<false, true, float>(W, A, p.nz, balanced, p.follows != 0, st);
    return p.thermal ? launch<true, false, float>(W, A, p.nz, balanced, p.follows != 0, st)
                     : launch<false, false, float>(W, A, p.nz, balanced, p.follows != 0, st);
}

cudaError_t fused2d_moments(int prec, const KParams &p, const void *f, const void *g, const void *RT_iso,
                            const void *Rin, const MomentOut &o, cudaStream_t st)
{
    if (!fused2d_supported(prec, 9, p)) return cudaErrorNotSupported;
    if (prec != 1) return fused2d_moments16(prec, p, f, g, RT_iso, Rin, o, st);
    const MomentArgs A = moment_args(p, f, g, RT_iso, Rin, o);
    if (p.walls)
        return p.thermal ? launch_moments<true, true, float>(A, p.nz, st) : launch_moments<false, true, float>(A, p.nz, st);
    return p.thermal ? launch_moments<true, false, float>(A, p.nz, st) : launch_moments<false, false, float>(A, p.nz, st);
}

}  // namespace evlbm
