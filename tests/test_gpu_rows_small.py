"""Small batches of wide images on the row-marching kernels: every SM works, so that they take no
longer than the TMA mainloop on narrower images of as many pixels; the sums stay those of the
oracle at one row a CTA."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle.unet as U
from paper_2508_00577_gb300 import surrogate as S

pytestmark = pytest.mark.gpu

if torch.cuda.is_available():
    from test_gpu_surrogate import bf, bf16_round, close, interior, op, padded

dev = "cuda"


def us(launch, n=20):
    """Device time of one of n launches of a replayed graph."""
    stream = torch.cuda.Stream()
    with torch.cuda.stream(stream):
        launch(stream)
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=stream):
        for _ in range(n):
            launch(stream)
    best = 1e30
    for _ in range(7):
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        with torch.cuda.stream(stream):
            e0.record()
            g.replay()
            e1.record()
        torch.cuda.synchronize()
        best = min(best, e0.elapsed_time(e1) * 1e3 / n)
    return best


def layer(Bn, H, W, C, N, weight_gradient):
    """(launch(stream), status, output, reference, absolute reference) of one layer."""
    r = np.random.default_rng(H + W + C)
    x = bf16_round(r.normal(size=(Bn, H, W, C)))
    X, _ = bf(padded(x))
    kp = U.kp_of(C)
    M = Bn * H * W
    g = S.sur_gemm_args()
    if weight_gradient:
        Z, Zd = bf(r.normal(size=(Bn, H + 2, W + 2, N)))
        out = torch.zeros(kp, N, device=dev)
        g.a, g.b = op(X, S.SUR_OP_TCONV3, C, 0, C, 9 * C, H, W), op(Z, S.SUR_OP_TPIX, N, 0, 0, N, H, W)
        g.M, g.N, g.K, g.splits, g.epi = kp, N, M, 4, S.SUR_EPI_F32_ATOMIC
        ref = [U.conv3_bwd_weight(f(x), f(interior(Zd)))[0].reshape(9 * C, N) for f in (lambda v: v, np.abs)]
        operands = X, Z
        got = lambda: out[:9 * C].cpu().numpy()
    else:
        Wt, Wd = bf(r.normal(size=(9, C, N)) / np.sqrt(9 * C))
        Wb = torch.zeros(N, kp, dtype=torch.bfloat16, device=dev)
        Wb[:, :9 * C] = Wt.reshape(9 * C, N).t()
        out = torch.zeros(Bn, H + 2, W + 2, N, device=dev)
        g.a, g.b = op(X, S.SUR_OP_CONV3, C, 0, C, M, H, W), op(Wb, S.SUR_OP_DENSE, kp, rows=N)
        g.M, g.N, g.K, g.splits, g.epi = M, N, kp, 1, S.SUR_EPI_F32
        ref = [U.conv3(f(x), f(Wd), np.zeros(N)) for f in (lambda v: v, np.abs)]
        operands = X, Wb
        got = lambda: interior(out.cpu().numpy())
    g.out, g.ldo = out.data_ptr(), N
    status = torch.zeros(2, dtype=torch.int32, device=dev)

    def launch(stream, alive=(operands, out)):       # the addresses in g stay those of live tensors
        S.sur_gemm(g, status.data_ptr(), stream.cuda_stream)

    return launch, status, got, ref


@pytest.mark.parametrize("C,N", [(32, 32), (64, 32), (64, 64)])
@pytest.mark.parametrize("weight_gradient", [False, True], ids=["conv", "wgrad"])
@pytest.mark.parametrize("Bn,H,W,narrow", [(1, 16, 256, 64), (1, 32, 256, 64), (3, 16, 128, 64)])
def test_small_batches_use_the_gpu(Bn, H, W, narrow, C, N, weight_gradient):
    launch, status, got, ref = layer(Bn, H, W, C, N, weight_gradient)
    launch(torch.cuda.current_stream())
    torch.cuda.synchronize()
    close(got(), *ref)                            # FP32 accumulation of BF16 products
    other = layer(Bn, H * W // narrow, narrow, C, N, weight_gradient)
    a, b = us(launch), us(other[0])
    print(f"{'wgrad' if weight_gradient else 'conv'} {C} -> {N}, {Bn} x {H} x {W}: {a:.1f} us, "
          f"{Bn} x {H * W // narrow} x {narrow}: {b:.1f}")
    assert int(status[0]) == 0
    assert a <= 1.3 * b
