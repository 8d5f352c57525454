"""The row-marching weight gradient of a 3x3 convolution (images at least 128 pixels wide)
against the oracle: every operand width it is instantiated for, channel blocks of a wider
input, one CTA and several, stretches of rows that cross columns and images, and an output
that already holds values."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle.unet as U
from paper_2508_00577_gb300 import surrogate as S

pytestmark = pytest.mark.gpu

if torch.cuda.is_available():
    from test_gpu_surrogate import bf, bf16_round, close, gemm, interior, op, padded

dev = "cuda"


@pytest.mark.parametrize("Cin,Cout", [(8, 32), (32, 32), (64, 32), (8, 64), (32, 64), (64, 64), (128, 64), (128, 32)])
@pytest.mark.parametrize("Bn,H,W", [(1, 2, 128), (2, 16, 128), (3, 32, 256), (1, 8, 512)])
def test_matches_oracle(Cin, Cout, Bn, H, W):
    r = np.random.default_rng(Cin + 2 * Cout + Bn + H + W)
    x = bf16_round(r.normal(size=(Bn, H, W, Cin)))
    X, _ = bf(padded(x))
    ldz, c0 = Cout + 32, 32                     # columns of a wider gradient tensor
    dZ, dZd = bf(r.normal(size=(Bn, H + 2, W + 2, ldz)))
    kp = U.kp_of(Cin)
    out = torch.ones(kp, Cout, device=dev)
    gemm(op(X, S.SUR_OP_TCONV3, Cin, 0, Cin, 9 * Cin, H, W), op(dZ, S.SUR_OP_TPIX, ldz, c0, 0, Cout, H, W),
         kp, Cout, Bn * H * W, epi=S.SUR_EPI_F32_ATOMIC, out=out, ldo=Cout, splits=3)
    dz = interior(dZd)[..., c0:]
    ref = U.conv3_bwd_weight(x, dz)[0].reshape(9 * Cin, Cout) + 1
    absref = U.conv3_bwd_weight(np.abs(x), np.abs(dz))[0].reshape(9 * Cin, Cout) + 1
    g = out.cpu().numpy()
    close(g[:9 * Cin], ref, absref)             # FP32 accumulation of BF16 products
    assert np.all(g[9 * Cin:] == 1)
