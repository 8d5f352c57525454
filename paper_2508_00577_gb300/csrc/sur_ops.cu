// Elementwise and reduction kernels of the learned surrogate on halo-padded
// NHWC tensors (see surrogate.cuh): SiLU backward (with the pooling's adjoint), bias
// gradients, 2x2 average pooling, input packing, the 1x1 head with the loss and its
// gradients or the state update, the loss terms and first-layer input gradient of
// unrolled training, Adam, the BF16 operand copies of the weights, and the per-domain
// fallback indicators.  The kernels over activations are bound by HBM: 16-byte accesses,
// consecutive threads on consecutive bytes, pixel indices by shifts.  The kernels of a pass are
// dependent launches (pdl.cuh): a training step has 80 of them, 2612 -> 2503 us at 16 x 256^2,
// and a window of 32 x 256^2 1319 -> 1303 us.
#include <stdint.h>

#include "pdl.cuh"
#include "surrogate.cuh"

namespace evsur {

using evlbm::launch_pdl;

namespace {

inline int grid_1d(long long n)
{
    long long g = (n + 255) / 256;
    return (int)(g > 8192 ? 8192 : (g < 1 ? 1 : g));
}

// Grid of the activation kernels: what is resident at once (per_sm blocks of 256 threads, by
// registers, on each SM), each block striding over the tensor.  Those that end in
// per-channel atomics (block_colsum8) so add at most that many values to each accumulator.
inline int grid_res(long long n, int per_sm)
{
    const int g = grid_1d(n), most = evlbm::sm_count() * per_sm;
    return g > most ? most : g;
}

inline int log2i(int v)
{
    int l = 0;
    while ((1 << l) < v) ++l;
    return l;
}

#define GRID_STRIDE(e, total)                                                                    \
    for (long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x; e < (long long)(total); \
         e += (long long)gridDim.x * blockDim.x)

// Sum over the block of each thread's 8-channel partial sums into out[c] (atomic).  Every
// thread of a block keeps one channel group, threadIdx.x % C8: the grid stride and the
// block size (256) are multiples of C8 = C / 8 <= 32, a power of two.  The sums are added by
// consecutive threads to consecutive channels: with a thread adding its 8 channels in turn
// (32-byte strides in a warp) the additions to one sector, 8 times as many, took most of the
// time of the narrow levels (SiLU backward of 2^14 pixels x 256 channels: 63 us).
__device__ __forceinline__ void block_colsum8(const float acc[8], int C8, float *out)
{
    __shared__ float red[256][9];
    const int t = threadIdx.x, C = C8 * 8, parts = 256 / C;
#pragma unroll
    for (int j = 0; j < 8; ++j) red[t][j] = acc[j];
    __syncthreads();
    // Thread = (channel t % C, part t / C of the threads that hold its group).
    const int c = t % C;
    float s = 0.f;
    for (int k = (c >> 3) + C8 * (t / C); k < 256; k += C8 * parts) s += red[k][c & 7];
    __syncthreads();
    red[t][8] = s;
    __syncthreads();
    if (t < C) {
        for (int q = 1; q < parts; ++q) s += red[t + q * C][8];
        atomicAdd(out + t, s);
    }
}

// dZ = dY * silu'(Z), silu'(z) = s (1 + z (1 - s)) with s = 1 / (1 + e^-z);
// 8 channels per thread; dZ gets its halo copies (it is gathered by the adjoint
// convolution).  dbias += the column sums of the stored (BF16) dZ over the interior
// pixels: the bias gradient, without a second pass over dZ.  POOL: the layer's output also
// went into the 2x2 average pooling, whose gradient dP (coarse grid, halo-padded, ld C)
// adds a quarter to each child; the sum is rounded to BF16 as a stored gradient would be.
// C8 = C / 8 = 1 << c8s.
// Bound by HBM: 6 bytes per element (4 + 2), and the divide of s, whose slow-path branch
// serialised the eight channels, was most of the rest: 71 us at 2^20 pixels x 32 channels
// with it, 512 blocks, 64-bit divisions and a halo list in local memory.
template <bool POOL>
__global__ void __launch_bounds__(256, 4) k_silu_bwd(const bf16 *dY, int ldd, const bf16 *dP, const bf16 *Z, long long M,
                                                  int lh, int lw, int c8s, bf16 *dZ, float *dbias)
{
    evlbm::pdl_wait();
    evlbm::pdl_trigger();
    const int C8 = 1 << c8s, C = C8 << 3;
    float acc[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
    GRID_STRIDE(e, M << c8s)
    {
        const long long m = e >> c8s;
        const int c = (int)(e & (C8 - 1)) << 3;
        const long long p = pad_pix(m, lh, lw);
        const uint4 dv = *reinterpret_cast<const uint4 *>(dY + p * ldd + c);
        const uint4 zv = *reinterpret_cast<const uint4 *>(Z + p * C + c);
        const bf16 *dh = reinterpret_cast<const bf16 *>(&dv), *zh = reinterpret_cast<const bf16 *>(&zv);
        float d[8], o[8];
#pragma unroll
        for (int j = 0; j < 8; ++j) d[j] = __bfloat162float(dh[j]);
        if constexpr (POOL) {
            const int H = 1 << lh, W = 1 << lw;
            const long long b = m >> (lh + lw);
            const int y = (int)((m >> lw) & (H - 1)), x = (int)(m & (W - 1));
            const long long pc = (b * (H / 2 + 2) + y / 2 + 1) * (W / 2 + 2) + x / 2 + 1;
            const uint4 pv = *reinterpret_cast<const uint4 *>(dP + pc * C + c);
            const bf16 *ph = reinterpret_cast<const bf16 *>(&pv);
#pragma unroll
            for (int j = 0; j < 8; ++j)
                d[j] = __bfloat162float(__float2bfloat16_rn(d[j] + 0.25f * __bfloat162float(ph[j])));
        }
        float z[8];
#pragma unroll
        for (int j = 0; j < 8; ++j) z[j] = __bfloat162float(zh[j]);
        silu_grad_n<8>(z, d, o);
        const uint4 ov = pack8(o);
        const bf16 *oh = reinterpret_cast<const bf16 *>(&ov);
#pragma unroll
        for (int j = 0; j < 8; ++j) acc[j] += __bfloat162float(oh[j]);
        for_halo(m, lh, lw, [&](long long t) { *reinterpret_cast<uint4 *>(dZ + t * C + c) = ov; });
    }
    if (dbias) block_colsum8(acc, C8, dbias);
}

// out[c] += sum over interior pixels of X[pix*ldx + c], c < C (bias gradients), 8
// channels (16 bytes) per load.
__global__ void __launch_bounds__(256) k_colsum(const bf16 *X, int ldx, long long M, int lh, int lw, int c8s,
                                                float *out)
{
    evlbm::pdl_wait();
    evlbm::pdl_trigger();
    const int C8 = 1 << c8s;
    float acc[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
#pragma unroll 4
    GRID_STRIDE(e, M << c8s)
    {
        const long long m = e >> c8s;
        const int c = (int)(e & (C8 - 1)) << 3;
        const uint4 v = *reinterpret_cast<const uint4 *>(X + pad_pix(m, lh, lw) * ldx + c);
        const bf16 *h = reinterpret_cast<const bf16 *>(&v);
#pragma unroll
        for (int j = 0; j < 8; ++j) acc[j] += __bfloat162float(h[j]);
    }
    block_colsum8(acc, C8, out);
}

// 2x2 average pooling: X (fine grid, ld ldx, first C channels) -> Y (coarse grid
// 2^lh x 2^lw, ld C) with halo copies; 8 channels per thread (one channel per thread, with
// 2-byte accesses, took 46 us at 2^18 coarse pixels x 32 channels).
__global__ void __launch_bounds__(256) k_pool2(const bf16 *X, int ldx, long long Mc, int lh, int lw, int c8s, bf16 *Y)
{
    evlbm::pdl_wait();
    evlbm::pdl_trigger();
    const int Wf2 = 2 * (1 << lw) + 2, C8 = 1 << c8s, C = C8 << 3;
    GRID_STRIDE(e, Mc << c8s)
    {
        const long long q = e >> c8s;
        const int c = (int)(e & (C8 - 1)) << 3;
        const bf16 *f = X + child0(q, lh, lw) * ldx + c;
        const uint4 v[4] = {*reinterpret_cast<const uint4 *>(f), *reinterpret_cast<const uint4 *>(f + ldx),
                            *reinterpret_cast<const uint4 *>(f + (long long)Wf2 * ldx),
                            *reinterpret_cast<const uint4 *>(f + (long long)(Wf2 + 1) * ldx)};
        float o[8];
#pragma unroll
        for (int j = 0; j < 8; ++j) {
            float s = 0.f;
#pragma unroll
            for (int k = 0; k < 4; ++k) {
                const float t = __bfloat162float(reinterpret_cast<const bf16 *>(&v[k])[j]);
                s = k ? s + t : t;
            }
            o[j] = 0.25f * s;
        }
        const uint4 ov = pack8(o);
        for_halo(q, lh, lw, [&](long long t) { *reinterpret_cast<uint4 *>(Y + t * C + c) = ov; });
    }
}

// Input packing: x fields [4][M] FP32 -> X (8 channels, halo-padded) BF16,
// channels 4..7 zero.
__global__ void k_pack_in(const float *x, long long M, int lh, int lw, const float *norm, bf16 *X)
{
    evlbm::pdl_wait();
    evlbm::pdl_trigger();
    GRID_STRIDE(m, M)
    {
        float v[8];
#pragma unroll
        for (int c = 0; c < 4; ++c) v[c] = (x[c * M + m] - norm[c]) / norm[4 + c];
#pragma unroll
        for (int c = 4; c < 8; ++c) v[c] = 0.f;
        const uint4 pv = pack8(v);
        for_halo(m, lh, lw, [&](long long t) { *reinterpret_cast<uint4 *>(X + t * 8) = pv; });
    }
}

// 1x1 head (32 -> 4 channels) and its use:
//   o[m][k] = bh[k] + sum_c Y[m][c] Wh[k][c]
//   kHeadNext: xn[k][m] = x[k][m] + out_scale[k] o[m][k]
//   kHeadLoss: r = o - (yt - x)/out_scale; loss += r^2 / (4M); dO = 2 r / (4M); then the
//              head's backward pass on dO
//   kHeadBwd:  the backward pass on a given dO [M][4]:
//              dY[m][c] = sum_k dO[m][k] Wh[k][c]; dWh[k][c] += sum_m dO[m][k] Y[m][c];
//              dbh[k] += sum_m dO[m][k]
// A block stages the 64-byte rows of 256 pixels in shared memory (80-byte pitch: 16-byte
// reads of consecutive rows hit distinct banks), so that global accesses are whole lines;
// thread = pixel for o, lane = channel (a warp on its own 32 pixels) for the backward pass,
// which overwrites the staged Y with dY.  Bound by HBM: Y read once, dY written once.  As
// separate kernels, with each thread reading its pixel's 64 bytes itself, loss + backward
// took 110 + 129 us at 2^20 pixels and the state update 166 us at 2^21.
enum { kHeadNext, kHeadLoss, kHeadBwd };
template <int MODE>
__global__ void __launch_bounds__(256) k_head(const bf16 *Y, long long M, int lh, int lw, const float *Wh,
                                              const float *bh, const float *norm, const float *x, const float *yt,
                                              const float *dO, float *loss, float *xn, bf16 *dY, float *dWh,
                                              float *dbh)
{
    evlbm::pdl_wait();
    evlbm::pdl_trigger();
    __shared__ uint4 sy[256 * 5];
    __shared__ float w[4 * 32];
    __shared__ float4 sd[MODE == kHeadNext ? 1 : 256];
    const int t = threadIdx.x, lane = t & 31, wi = t >> 5;
    if (t < 128) w[t] = Wh[t];
    float o0[4] = {0.f, 0.f, 0.f, 0.f}, wl[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        if (MODE != kHeadBwd) o0[k] = bh[k];
        wl[k] = Wh[k * 32 + lane];
    }
    const float inv = 1.f / (4.f * (float)M);
    float acc = 0.f, gw[4] = {0.f, 0.f, 0.f, 0.f}, gb = 0.f;
    for (long long base = (long long)blockIdx.x * 256; base < M; base += (long long)gridDim.x * 256) {
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const int px = (t >> 2) + 64 * j, ch = t & 3;
            if (base + px < M)
                sy[px * 5 + ch] = *reinterpret_cast<const uint4 *>(Y + pad_pix(base + px, lh, lw) * 32 + ch * 8);
        }
        const long long m = base + t;
        float xv[4], yv[4];
        float4 d = make_float4(0.f, 0.f, 0.f, 0.f);
        if (m < M) {
            if (MODE == kHeadBwd) {
                d = *reinterpret_cast<const float4 *>(dO + m * 4);
            } else {
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    xv[k] = x[k * M + m];
                    if (MODE == kHeadLoss) yv[k] = yt[k * M + m];
                }
            }
        }
        __syncthreads();
        if (MODE != kHeadBwd && m < M) {
            float o[4] = {o0[0], o0[1], o0[2], o0[3]};
#pragma unroll
            for (int c8 = 0; c8 < 4; ++c8) {
                const uint4 v = sy[t * 5 + c8];
                const bf16 *h = reinterpret_cast<const bf16 *>(&v);
#pragma unroll
                for (int j = 0; j < 8; ++j) {
                    const float f = __bfloat162float(h[j]);
#pragma unroll
                    for (int k = 0; k < 4; ++k) o[k] += f * w[k * 32 + c8 * 8 + j];
                }
            }
            if (MODE == kHeadLoss) {
                float r[4];
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    r[k] = o[k] - (yv[k] - xv[k]) / norm[8 + k];
                    acc += r[k] * r[k];
                }
                d = make_float4(2.f * r[0] * inv, 2.f * r[1] * inv, 2.f * r[2] * inv, 2.f * r[3] * inv);
            } else {
#pragma unroll
                for (int k = 0; k < 4; ++k) xn[k * M + m] = xv[k] + norm[8 + k] * o[k];
            }
        }
        if (MODE != kHeadNext) {
            sd[t] = d;
            __syncwarp();
            // Eight pixels at a time: their reads go before the writes to the same array.
#pragma unroll 1
            for (int k8 = 0; k8 < 32; k8 += 8) {
                float f[8];
                float4 dk[8];
#pragma unroll
                for (int k = 0; k < 8; ++k) {
                    const int px = wi * 32 + k8 + k;
                    dk[k] = sd[px];
                    f[k] = base + px < M ? __bfloat162float(reinterpret_cast<const bf16 *>(sy + px * 5)[lane]) : 0.f;
                }
#pragma unroll
                for (int k = 0; k < 8; ++k) {
                    reinterpret_cast<bf16 *>(sy + (wi * 32 + k8 + k) * 5)[lane] =
                        __float2bfloat16_rn(dk[k].x * wl[0] + dk[k].y * wl[1] + dk[k].z * wl[2] + dk[k].w * wl[3]);
                    gw[0] += dk[k].x * f[k];
                    gw[1] += dk[k].y * f[k];
                    gw[2] += dk[k].z * f[k];
                    gw[3] += dk[k].w * f[k];
                    if (lane < 4) gb += lane == 0 ? dk[k].x : (lane == 1 ? dk[k].y : (lane == 2 ? dk[k].z : dk[k].w));
                }
            }
            __syncthreads();
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const int px = (t >> 2) + 64 * j, ch = t & 3;
                if (base + px < M)
                    *reinterpret_cast<uint4 *>(dY + pad_pix(base + px, lh, lw) * 32 + ch * 8) = sy[px * 5 + ch];
            }
        }
        __syncthreads();
    }
    if (MODE == kHeadNext) return;
    // Block sums of the loss and of the gradients: red[warp][channel-major gw, gb], loss in sd.
    float *red = reinterpret_cast<float *>(sy);
    float *rl = reinterpret_cast<float *>(sd);
#pragma unroll
    for (int k = 0; k < 4; ++k) red[wi * 132 + k * 32 + lane] = gw[k];
    if (lane < 4) red[wi * 132 + 128 + lane] = gb;
    rl[t] = acc;
    __syncthreads();
    if (t < 132) {
        float s = 0.f;
        for (int j = 0; j < 8; ++j) s += red[j * 132 + t];
        if (t < 128) atomicAdd(dWh + t, s);
        else atomicAdd(dbh + t - 128, s);
    }
    if (MODE == kHeadLoss) {
        for (int s = 128; s > 0; s >>= 1) {
            if (t < s) rl[t] += rl[t + s];
            __syncthreads();
        }
        if (t == 0) atomicAdd(loss, rl[0] * inv);
    }
}

// Unrolled training (k windows, each applied to the previous prediction): the loss
// term of a prediction x'_j against its target y_j, r = (x'_j - y_j) / out_scale, added
// to the planar field gradient G = dL/dx'_j as 2 r / out_scale * inv (inv = 1 / (4 M k)),
// and the output gradient of the window that produced x'_j, dO = out_scale * G
// (x'_j = x'_{j-1} + out_scale o).  loss += sum r^2 * inv.
__global__ void k_unroll_term(const float *xp, const float *yt, long long M, const float *norm, float inv, float *G,
                              float *dO, float *loss)
{
    evlbm::pdl_wait();
    evlbm::pdl_trigger();
    __shared__ float red[256];
    float acc = 0.f;
    GRID_STRIDE(m, M)
    {
        float d[4];
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            const float s = norm[8 + c];
            const float r = (xp[c * M + m] - yt[c * M + m]) / s;
            acc += r * r;
            const float g = G[c * M + m] + 2.f * r / s * inv;
            G[c * M + m] = g;
            d[c] = s * g;
        }
        *reinterpret_cast<float4 *>(dO + m * 4) = make_float4(d[0], d[1], d[2], d[3]);
    }
    red[threadIdx.x] = acc;
    __syncthreads();
    for (int k = blockDim.x / 2; k > 0; k >>= 1) {
        if ((int)threadIdx.x < k) red[threadIdx.x] += red[threadIdx.x + k];
        __syncthreads();
    }
    if (threadIdx.x == 0) atomicAdd(loss, red[0] * inv);
}

// Input gradient of the first convolution (8 -> 32 channels) in its 4 field channels,
// dxin[p][c] = sum_tap sum_co W[tap * 8 + c][co] dZ[p - s_tap][co] (s_tap = (dy, dx); the
// periodic neighbours come from the halo of dZ), added to the planar field gradient:
// G[c][m] += dxin[m][c] / in_scale[c].  Wb is the forward BF16 copy [32][Kp].
__global__ void k_conv0_dx(const bf16 *dZ, const bf16 *Wb, int Kp, long long M, int lh, int lw, const float *norm,
                           float *G)
{
    evlbm::pdl_wait();
    evlbm::pdl_trigger();
    __shared__ float w[9][32][4];
    for (int e = threadIdx.x; e < 9 * 32 * 4; e += blockDim.x) {
        const int tap = e / 128, co = (e / 4) % 32, c = e % 4;
        w[tap][co][c] = __bfloat162float(Wb[co * Kp + tap * 8 + c]);
    }
    __syncthreads();
    const long long Wp = (1 << lw) + 2;
    GRID_STRIDE(m, M)
    {
        const long long p = pad_pix(m, lh, lw);
        float acc[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
        for (int tap = 0; tap < 9; ++tap) {
            const int dy = tap / 3 - 1, dx = tap % 3 - 1;
            const bf16 *z = dZ + (p - dy * Wp - dx) * 32;
#pragma unroll
            for (int c8 = 0; c8 < 32; c8 += 8) {
                const uint4 v = *reinterpret_cast<const uint4 *>(z + c8);
                const bf16 *h = reinterpret_cast<const bf16 *>(&v);
#pragma unroll
                for (int j = 0; j < 8; ++j) {
                    const float zv = __bfloat162float(h[j]);
#pragma unroll
                    for (int c = 0; c < 4; ++c) acc[c] += w[tap][c8 + j][c] * zv;
                }
            }
        }
#pragma unroll
        for (int c = 0; c < 4; ++c) G[c * M + m] += acc[c] / norm[4 + c];
    }
}

// Adam with bias correction on FP32 masters (c1 = 1 - b1^t, c2 = 1 - b2^t).
__global__ void k_adam(float *w, const float *gr, float *m, float *v, long long n, float lr, float b1, float b2,
                       float eps, float c1, float c2)
{
    evlbm::pdl_wait();
    evlbm::pdl_trigger();
    GRID_STRIDE(i, n)
    {
        const float g = gr[i];
        const float mi = b1 * m[i] + (1.f - b1) * g;
        const float vi = b2 * v[i] + (1.f - b2) * g * g;
        m[i] = mi;
        v[i] = vi;
        w[i] -= lr * (mi / c1) / (sqrtf(vi / c2) + eps);
    }
}

// BF16 operand copies of every layer's weights in one launch (one launch per layer took
// 17 x ~4.5 us); block b works on a stretch of kWeightChunk elements of one layer.
//   3x3 convolution, master W [Kp][Cout]:
//     fwd [Cout][Kp]   (forward B operand, K = tap*Cin + ci)
//     adj [Cin][Kpo]   (adjoint B operand, K = tap*Cout + co, taken at the mirrored tap 8 - tap)
//   transposed convolution, master W [4 Cout][Cin]:
//     fwd [4 Cout][Cin] (forward B operand), adj [Cin][4 Cout] (adjoint B operand).
constexpr int kWeightChunk = 1024;
struct WeightTab {
    WeightCopy L[kMaxWeightCopies];
    int first[2 * kMaxWeightCopies + 1];      // first block of each layer's fwd and adj copies
    int n;
};
__global__ void __launch_bounds__(256) k_weights(const __grid_constant__ WeightTab tab)
{
    evlbm::pdl_wait();
    evlbm::pdl_trigger();
    int j = 0;
    while (j + 1 < 2 * tab.n && (int)blockIdx.x >= tab.first[j + 1]) ++j;
    const WeightCopy &w = tab.L[j >> 1];
    const bool adj = j & 1;
    const int total = w.up ? 4 * w.cout * w.cin : (adj ? w.cin * w.kpo : w.cout * w.kp);
    const int e0 = ((int)blockIdx.x - tab.first[j]) * kWeightChunk;
    for (int e = e0 + threadIdx.x; e < total && e < e0 + kWeightChunk; e += 256) {
        float v = 0.f;
        if (w.up) {
            v = adj ? w.w[(e % (4 * w.cout)) * w.cin + e / (4 * w.cout)] : w.w[e];
        } else if (!adj) {
            const int co = e / w.kp, k = e - co * w.kp;
            v = w.w[k * w.cout + co];
        } else {
            const int ci = e / w.kpo, k = e - ci * w.kpo;
            if (k < 9 * w.cout) {
                const int tap = k / w.cout, co = k - tap * w.cout;
                v = w.w[((8 - tap) * w.cin + ci) * w.cout + co];
            }
        }
        (adj ? w.adj : w.fwd)[e] = __float2bfloat16_rn(v);
    }
}

// Per-domain FP64 sums of rho and of the liquid count (rho > rho_mid): out[2b],
// out[2b+1]; invalid[0] |= 1 if any field is not finite or rho or T is not > 0.
// Interface-position indicator: per domain, the number of nodes whose phase (rho above or
// below rho_mid) differs between the density fields A and B (out[b] += count).
__global__ void k_phase_flips(const float *A, const float *B, long long Mb, float rho_mid, double *out)
{
    __shared__ double s1[256];
    const long long b = blockIdx.y;
    double a = 0.0;
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < Mb; i += (long long)gridDim.x * blockDim.x) {
        const long long n = b * Mb + i;
        a += ((A[n] > rho_mid) != (B[n] > rho_mid)) ? 1.0 : 0.0;
    }
    s1[threadIdx.x] = a;
    __syncthreads();
    for (int s = blockDim.x / 2; s > 0; s >>= 1) {
        if ((int)threadIdx.x < s) s1[threadIdx.x] += s1[threadIdx.x + s];
        __syncthreads();
    }
    if (threadIdx.x == 0) atomicAdd(out + b, s1[0]);
}

__global__ void k_indicators(const float *F, long long M, long long Mb, float rho_mid, double *out, int *invalid)
{
    __shared__ double s1[256], s2[256];
    const long long b = blockIdx.y;
    double a1 = 0.0, a2 = 0.0;
    bool bad = false;
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < Mb; i += (long long)gridDim.x * blockDim.x) {
        const long long n = b * Mb + i;
        const float r = F[n];
        a1 += r;
        a2 += r > rho_mid ? 1.0 : 0.0;
        if (invalid) {
            for (int c = 0; c < 4; ++c) bad |= !isfinite(F[c * M + n]);
            bad |= !(r > 0.f) || !(F[3 * M + n] > 0.f);
        }
    }
    if (bad) atomicOr(invalid, 1);
    s1[threadIdx.x] = a1;
    s2[threadIdx.x] = a2;
    __syncthreads();
    for (int s = blockDim.x / 2; s > 0; s >>= 1) {
        if ((int)threadIdx.x < s) {
            s1[threadIdx.x] += s1[threadIdx.x + s];
            s2[threadIdx.x] += s2[threadIdx.x + s];
        }
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        atomicAdd(out + 2 * b, s1[0]);
        atomicAdd(out + 2 * b + 1, s2[0]);
    }
}

// rho[b*Mb + i] -= delta[b]: restores each domain's mass (the lattice Boltzmann
// step conserves it exactly).
__global__ void k_shift_rho(float *rho, long long Mb, const float *delta)
{
    const long long b = blockIdx.y;
    const float d = delta[b];
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < Mb; i += (long long)gridDim.x * blockDim.x)
        rho[b * Mb + i] -= d;
}

}  // namespace

cudaError_t shift_rho(float *rho, int batch, long long Mb, const float *delta, cudaStream_t st)
{
    long long gx = (Mb + 255) / 256;
    if (gx > 64) gx = 64;
    k_shift_rho<<<dim3((unsigned)gx, (unsigned)batch), 256, 0, st>>>(rho, Mb, delta);
    return cudaGetLastError();
}

cudaError_t silu_bwd(const bf16 *dY, int ldd, const bf16 *dP, const bf16 *Z, long long M, int lh, int lw, int C,
                     bf16 *dZ, float *dbias, cudaStream_t st)
{
    const int s = log2i(C >> 3);
    if (C != 8 << s || C > 256) return cudaErrorInvalidValue;
    const int g = grid_res(M << s, 4);
    if (dP) return launch_pdl(k_silu_bwd<true>, g, 256, 0, st, dY, ldd, dP, Z, M, lh, lw, s, dZ, dbias);
    return launch_pdl(k_silu_bwd<false>, g, 256, 0, st, dY, ldd, dP, Z, M, lh, lw, s, dZ, dbias);
}

cudaError_t colsum(const bf16 *X, int ldx, long long M, int lh, int lw, int C, float *out, cudaStream_t st)
{
    const int s = log2i(C >> 3);
    if (C != 8 << s || C > 256 || ldx % 8 || (reinterpret_cast<uintptr_t>(X) & 15)) return cudaErrorInvalidValue;
    return launch_pdl(k_colsum, grid_res(M << s, 6), 256, 0, st, X, ldx, M, lh, lw, s, out);
}

cudaError_t pool2(const bf16 *X, int ldx, long long Mc, int lh, int lw, int C, bf16 *Y, cudaStream_t st)
{
    const int s = log2i(C >> 3);
    if (C != 8 << s || ldx % 8 || (reinterpret_cast<uintptr_t>(X) & 15)) return cudaErrorInvalidValue;
    return launch_pdl(k_pool2, grid_1d(Mc << s), 256, 0, st, X, ldx, Mc, lh, lw, s, Y);
}

cudaError_t pack_in(const float *x, long long M, int lh, int lw, const float *norm, bf16 *X, cudaStream_t st)
{
    return launch_pdl(k_pack_in, grid_1d(M), 256, 0, st, x, M, lh, lw, norm, X);
}

cudaError_t head_next(const bf16 *Y, long long M, int lh, int lw, const float *Wh, const float *bh, const float *norm,
                      const float *x, float *xn, cudaStream_t st)
{
    return launch_pdl(k_head<kHeadNext>, grid_res(M, 5), 256, 0, st, Y, M, lh, lw, Wh, bh, norm, x, nullptr, nullptr,
                      nullptr, xn, nullptr, nullptr, nullptr);
}

cudaError_t head_loss_bwd(const bf16 *Y, long long M, int lh, int lw, const float *Wh, const float *bh,
                          const float *norm, const float *x, const float *yt, float *loss, bf16 *dY, float *dWh,
                          float *dbh, cudaStream_t st)
{
    return launch_pdl(k_head<kHeadLoss>, grid_res(M, 3), 256, 0, st, Y, M, lh, lw, Wh, bh, norm, x, yt, nullptr, loss,
                      nullptr, dY, dWh, dbh);
}

cudaError_t head_bwd(const bf16 *Y, long long M, int lh, int lw, const float *Wh, const float *dO, bf16 *dY,
                     float *dWh, float *dbh, cudaStream_t st)
{
    return launch_pdl(k_head<kHeadBwd>, grid_res(M, 6), 256, 0, st, Y, M, lh, lw, Wh, nullptr, nullptr, nullptr, nullptr,
                      dO, nullptr, nullptr, dY, dWh, dbh);
}

cudaError_t unroll_term(const float *xp, const float *yt, long long M, const float *norm, float inv, float *G, float *dO,
                        float *loss, cudaStream_t st)
{
    return launch_pdl(k_unroll_term, grid_1d(M), 256, 0, st, xp, yt, M, norm, inv, G, dO, loss);
}

cudaError_t conv0_dx(const bf16 *dZ, const bf16 *Wb, int Kp, long long M, int lh, int lw, const float *norm, float *G,
                     cudaStream_t st)
{
    if (Kp < 72 || (reinterpret_cast<uintptr_t>(dZ) & 15)) return cudaErrorInvalidValue;
    return launch_pdl(k_conv0_dx, grid_1d(M), 256, 0, st, dZ, Wb, Kp, M, lh, lw, norm, G);
}

cudaError_t adam(float *w, const float *g, float *m, float *v, long long n, float lr, float b1, float b2, float eps,
                 float c1, float c2, cudaStream_t st)
{
    return launch_pdl(k_adam, grid_1d(n), 256, 0, st, w, g, m, v, n, lr, b1, b2, eps, c1, c2);
}

cudaError_t copy_weights(const WeightCopy *layers, int n, cudaStream_t st)
{
    if (n < 1 || n > kMaxWeightCopies) return cudaErrorInvalidValue;
    WeightTab tab;
    tab.n = n;
    int blocks = 0;
    for (int k = 0; k < n; ++k) {
        const WeightCopy &w = tab.L[k] = layers[k];
        const int fwd = w.up ? 4 * w.cout * w.cin : w.cout * w.kp, adj = w.up ? fwd : w.cin * w.kpo;
        tab.first[2 * k] = blocks;
        blocks += (fwd + kWeightChunk - 1) / kWeightChunk;
        tab.first[2 * k + 1] = blocks;
        blocks += (adj + kWeightChunk - 1) / kWeightChunk;
    }
    tab.first[2 * n] = blocks;
    return launch_pdl(k_weights, blocks, 256, 0, st, tab);
}

cudaError_t indicators(const float *F, int batch, long long Mb, float rho_mid, double *out, int *invalid,
                       cudaStream_t st)
{
    cudaError_t e = cudaMemsetAsync(out, 0, sizeof(double) * 2 * batch, st);
    if (e != cudaSuccess) return e;
    long long gx = (Mb + 255) / 256;
    if (gx > 64) gx = 64;
    const dim3 grid((unsigned)gx, (unsigned)batch);
    k_indicators<<<grid, 256, 0, st>>>(F, (long long)batch * Mb, Mb, rho_mid, out, invalid);
    return cudaGetLastError();
}

cudaError_t phase_flips(const float *A, const float *B, int batch, long long Mb, float rho_mid, double *out,
                        cudaStream_t st)
{
    cudaError_t e = cudaMemsetAsync(out, 0, sizeof(double) * batch, st);
    if (e != cudaSuccess) return e;
    long long gx = (Mb + 255) / 256;
    if (gx > 64) gx = 64;
    const dim3 grid((unsigned)gx, (unsigned)batch);
    k_phase_flips<<<grid, 256, 0, st>>>(A, B, Mb, rho_mid, out);
    return cudaGetLastError();
}

}  // namespace evsur

extern "C" int sur_indicators(const float *d_fields, int batch, int H, int W, float rho_mid, double *d_out,
                              void *stream)
{
    if (!d_fields || !d_out || batch < 1 || H < 1 || W < 1) return SUR_EINVAL;
    const cudaError_t e = evsur::indicators(d_fields, batch, (long long)H * W, rho_mid, d_out, nullptr,
                                            static_cast<cudaStream_t>(stream));
    return e == cudaSuccess ? SUR_OK : SUR_ECUDA;
}
