"""The gathers of the transposed convolution's gradients (children of the coarse pixels, UPADJ and
TUP) against the oracle's layer routines, on the TMA mainloop and on the cp.async one: every box
width, several boxes a child, coarse grids from 2 x 4 (which TMA leaves to cp.async where it
cannot take them) to 32 x 128, three images, and rows of a weight gradient beyond the children's."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle.unet as U
from paper_2508_00577_gb300 import surrogate as S

pytestmark = pytest.mark.gpu

if torch.cuda.is_available():
    from test_gpu_surrogate import bf, close, gemm, interior, op, tma  # noqa: F401 (fixture)
else:
    @pytest.fixture
    def tma():
        return True

dev = "cuda"
SIZES = [(3, 2, 4), (3, 4, 8), (2, 8, 16), (3, 16, 32), (1, 32, 128)]


def tensors(Bn, h, w, Cin, Cout):
    """The gradient of the concatenated fine tensor, whose last Cout channels are the children's."""
    r = np.random.default_rng(Bn + h + w + Cin + Cout)
    dcat, d = bf(r.normal(size=(Bn, 2 * h + 2, 2 * w + 2, 2 * Cout)))
    return r, dcat, interior(d)[..., Cout:]


@pytest.mark.parametrize("Cout", [32, 64, 128])
@pytest.mark.parametrize("Bn,h,w", SIZES)
def test_input_gradient(Bn, h, w, Cout, tma):
    Cin, Mc = 64, Bn * h * w
    r, dcat, dy = tensors(Bn, h, w, Cin, Cout)
    Wu, Wud = bf(r.normal(size=(4, Cout, Cin)))
    WuT = Wu.reshape(4 * Cout, Cin).t().contiguous()
    out = torch.full((Bn, h + 2, w + 2, Cin), float("nan"), device=dev)
    gemm(op(dcat, S.SUR_OP_UPADJ, 2 * Cout, Cout, Cout, Mc, h, w), op(WuT, S.SUR_OP_DENSE, 4 * Cout, rows=Cin),
         Mc, Cin, 4 * Cout, out=out, ldo=Cin)
    x0 = np.zeros((Bn, h, w, Cin))
    # FP32 accumulation of BF16 products, as the other mainloops' tests.
    close(interior(out.cpu().numpy()), U.tconv2_bwd(x0, dy, Wud)[0], U.tconv2_bwd(x0, np.abs(dy), np.abs(Wud))[0])


@pytest.mark.parametrize("Cout", [32, 64, 128])
@pytest.mark.parametrize("extra", [0, 64])
@pytest.mark.parametrize("Bn,h,w", SIZES)
def test_weight_gradient(Bn, h, w, Cout, extra, tma):
    Cin, Mc = 64, Bn * h * w
    r, dcat, dy = tensors(Bn, h, w, Cin, Cout)
    X, Xd = bf(r.normal(size=(Bn, h + 2, w + 2, Cin)))
    M = 4 * Cout + extra                                    # rows beyond the children's: zero
    out = torch.ones(M, Cin, device=dev)
    gemm(op(dcat, S.SUR_OP_TUP, 2 * Cout, Cout, Cout, 4 * Cout, h, w), op(X, S.SUR_OP_TPIX, Cin, 0, 0, Cin, h, w),
         M, Cin, Mc, epi=S.SUR_EPI_F32_ATOMIC, out=out, ldo=Cin, splits=2 if Mc > 64 else 1)
    xi = interior(Xd)
    w0 = np.zeros((4, Cout, Cin))
    ref = U.tconv2_bwd(xi, dy, w0)[1].reshape(4 * Cout, Cin) + 1
    absref = U.tconv2_bwd(np.abs(xi), np.abs(dy), w0)[1].reshape(4 * Cout, Cin) + 1
    o = out.cpu().numpy()
    close(o[:4 * Cout], ref, absref)
    assert np.all(o[4 * Cout:] == 1)
