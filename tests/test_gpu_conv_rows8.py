"""The row-marching convolution of eight channels (the first layer, images at least 128 pixels
wide) against the oracle's layer routine, and its padding: a tap paired with zeros must not
spread an infinity beyond the 3x3 neighbourhood of its pixel."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle.unet as U
from paper_2508_00577_gb300 import surrogate as S

pytestmark = pytest.mark.gpu

if torch.cuda.is_available():
    from test_gpu_conv_rows import dev, weights
    from test_gpu_surrogate import bf, bf16_round, close, gemm, interior, op, padded


@pytest.mark.parametrize("Bn,H,W,ld,c0", [(1, 2, 128, 8, 0), (2, 16, 128, 24, 16), (3, 32, 256, 8, 0), (1, 8, 512, 8, 0),
                                          (9, 256, 128, 8, 0)])
def test_matches_oracle(Bn, H, W, ld, c0):
    r = np.random.default_rng(Bn + H + W + ld)
    x = bf16_round(r.normal(size=(Bn, H, W, ld)))
    X, _ = bf(padded(x))
    Wb, Wd, kp = weights(r, 8, 32)
    M = Bn * H * W
    out = torch.full((Bn, H + 2, W + 2, 32), float("nan"), device=dev)
    gemm(op(X, S.SUR_OP_CONV3, ld, c0, 8, M, H, W), op(Wb, S.SUR_OP_DENSE, kp, rows=32), M, 32, kp, out=out, ldo=32)
    xs = x[..., c0:c0 + 8]
    # FP32 accumulation of BF16 products, as the tests of the other mainloops.
    close(interior(out.cpu().numpy()), U.conv3(xs, Wd, np.zeros(32)), U.conv3(np.abs(xs), np.abs(Wd), np.zeros(32)))


def test_infinity_stays_in_its_neighbourhood():
    r = np.random.default_rng(5)
    Bn, H, W = 1, 8, 256
    x = bf16_round(r.normal(size=(Bn, H, W, 8)))
    x[0, 3, 100, 2] = np.inf
    X, _ = bf(padded(x))
    Wb, _, kp = weights(r, 8, 32)
    out = torch.zeros((Bn, H + 2, W + 2, 32), device=dev)
    M = Bn * H * W
    gemm(op(X, S.SUR_OP_CONV3, 8, 0, 8, M, H, W), op(Wb, S.SUR_OP_DENSE, kp, rows=32), M, 32, kp, out=out, ldo=32)
    bad = ~np.isfinite(interior(out.cpu().numpy())).all(-1)[0]
    want = np.zeros((H, W), bool)
    want[2:5, 99:102] = True
    np.testing.assert_array_equal(bad, want)


def test_silu_over_the_whole_range():
    """Zero input, so that z is the bias: ordinary values, values beyond the packed form's range
    beside them, and the ends of the range, against FP64 (one BF16 rounding of z and one of
    silu; where e^-z overflows silu is -0, at -inf NaN)."""
    Bn, H, W = 1, 2, 128
    M = Bn * H * W
    X = torch.zeros((Bn, H + 2, W + 2, 8), dtype=torch.bfloat16, device=dev)
    Wb = torch.zeros((32, 128), dtype=torch.bfloat16, device=dev)
    for big in ([], [79.5, 80.5, -80.5, 1e30], [-87.5, -88.5, -90.0, -1e30], [float("inf"), float("-inf"), float("nan")]):
        z = np.array((big + list(np.linspace(-30.0, 30.0, 32)))[:32], dtype=np.float32)
        z[31], z[30] = 0.0, 17.5
        bias = torch.tensor(z, device=dev)
        Y = torch.full((Bn, H + 2, W + 2, 32), 3.0, dtype=torch.bfloat16, device=dev)
        gemm(op(X, S.SUR_OP_CONV3, 8, 0, 8, M, H, W), op(Wb, S.SUR_OP_DENSE, 128, rows=32), M, 32, 128,
             epi=S.SUR_EPI_CONV, bias=bias, y=Y, ldy=32)
        got = interior(Y.float().cpu().numpy())
        with np.errstate(over="ignore", invalid="ignore"):
            want = z.astype(np.float64) / (1.0 + np.exp(-z.astype(np.float64)))
        want[z < -88.8] = 0.0
        want[np.isneginf(z)] = np.nan
        np.testing.assert_array_equal(np.isnan(got), np.broadcast_to(np.isnan(want), got.shape))
        np.testing.assert_array_equal(np.isinf(got), np.broadcast_to(np.isinf(want), got.shape))
        ok = np.isfinite(want)
        assert np.all(np.abs(got[..., ok] - want[ok]) <= 2 ** -8 * np.abs(want[ok]) + 1e-35)
