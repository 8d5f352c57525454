"""The row-marching 3x3 convolution (images at least 128 pixels wide) against the oracle's
layer routines: every channel pair it is instantiated for, one CTA and several, stretches of
rows that end inside a column and cross columns and images, and its epilogues."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle.unet as U
from paper_2508_00577_gb300 import surrogate as S

pytestmark = pytest.mark.gpu

if torch.cuda.is_available():
    from test_gpu_surrogate import bf, bf16_round, close, gemm, interior, op, padded

dev = "cuda"


def weights(r, Cin, Cout):
    Wt, Wd = bf(r.normal(size=(9, Cin, Cout)) / np.sqrt(9 * Cin))
    kp = U.kp_of(Cin)
    Wb = torch.zeros(Cout, kp, dtype=torch.bfloat16, device=dev)
    Wb[:, :9 * Cin] = Wt.reshape(9 * Cin, Cout).t()
    return Wb, Wd, kp


@pytest.mark.parametrize("Cin,Cout", [(32, 32), (32, 64), (64, 32), (64, 64)])
@pytest.mark.parametrize("Bn,H,W", [(1, 2, 128), (2, 16, 128), (3, 32, 256), (1, 8, 512), (5, 256, 128)])
def test_matches_oracle(Cin, Cout, Bn, H, W):
    r = np.random.default_rng(Cin + 2 * Cout + Bn + H + W)
    ld, c0 = Cin + 32, 32                       # channels of a wider tensor
    x = bf16_round(r.normal(size=(Bn, H, W, ld)))
    X, _ = bf(padded(x))
    Wb, Wd, kp = weights(r, Cin, Cout)
    M = Bn * H * W
    out = torch.full((Bn, H + 2, W + 2, Cout), float("nan"), device=dev)
    gemm(op(X, S.SUR_OP_CONV3, ld, c0, Cin, M, H, W), op(Wb, S.SUR_OP_DENSE, kp, rows=Cout), M, Cout, kp,
         out=out, ldo=Cout)
    xs = x[..., c0:]
    # FP32 accumulation of BF16 products, as the tests of the other mainloops.
    close(interior(out.cpu().numpy()), U.conv3(xs, Wd, np.zeros(Cout)),
          U.conv3(np.abs(xs), np.abs(Wd), np.zeros(Cout)))
    assert torch.isnan(out[:, 0]).all() and torch.isnan(out[:, :, -1]).all()      # BF16/FP32 epilogues write no halo


@pytest.mark.parametrize("Cout", [32, 64])
def test_epilogue_bias_silu_halo(Cout):
    Bn, H, W, Cin = 2, 16, 128, 32
    r = np.random.default_rng(Cout)
    x = bf16_round(3 * r.normal(size=(Bn, H, W, Cin)))
    X, _ = bf(padded(x))
    Wb, Wd, kp = weights(r, Cin, Cout)
    bias = torch.tensor(r.normal(size=Cout + 1), dtype=torch.float32, device=dev)[1:]      # not 16-byte aligned
    M = Bn * H * W
    Z = torch.zeros(Bn, H + 2, W + 2, Cout, dtype=torch.bfloat16, device=dev)
    Y = torch.full((Bn, H + 2, W + 2, 2 * Cout), 7.0, dtype=torch.bfloat16, device=dev)
    gemm(op(X, S.SUR_OP_CONV3, Cin, 0, Cin, M, H, W), op(Wb, S.SUR_OP_DENSE, kp, rows=Cout), M, Cout, kp,
         epi=S.SUR_EPI_CONV, out=Z, ldo=Cout, bias=bias, y=Y, ldy=2 * Cout, cy0=Cout)
    z = U.conv3(x, Wd, bias.cpu().numpy().astype(np.float64))
    zg = interior(Z.float().cpu().numpy())
    # one BF16 rounding of z; silu within its slope (at most 1.1) of that and one more rounding
    assert np.all(np.abs(zg - z) <= 2 ** -8 * np.abs(z) + 1e-5)
    yg = Y.float().cpu().numpy()
    yi = interior(yg)[..., Cout:]
    assert np.all(np.abs(yi - U.silu(z)) <= 2 ** -7 * np.abs(U.silu(z)) + 1e-4)
    np.testing.assert_array_equal(yg[..., Cout:], padded(yi))
    assert np.all(yg[..., :Cout] == 7.0)
