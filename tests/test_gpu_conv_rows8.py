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
