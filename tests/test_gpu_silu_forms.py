"""SiLU and its derivative have a packed form and, for a thread that holds a value beyond |z| = 80,
a scalar one: what the one gives for a value, the other gives beside large neighbours."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2508_00577_gb300 import surrogate as S

pytestmark = pytest.mark.gpu

if torch.cuda.is_available():
    from test_gpu_surrogate import NORM, gemm, op, rel_l2, smooth_fields

dev = "cuda"


def silu_of(z):
    """bf16(silu(z)) as bits, of the convolution epilogue: a zero product plus the bias z."""
    H = W = 8
    N = len(z)
    X = torch.zeros((1, H + 2, W + 2, 64), dtype=torch.bfloat16, device=dev)
    Wb = torch.zeros((N, 64), dtype=torch.bfloat16, device=dev)
    Y = torch.zeros((1, H + 2, W + 2, N), dtype=torch.bfloat16, device=dev)
    gemm(op(X, S.SUR_OP_PIX, 64, 0, 64, H * W, H, W), op(Wb, S.SUR_OP_DENSE, 64, rows=N), H * W, N, 64,
         epi=S.SUR_EPI_CONV, bias=torch.tensor(z, device=dev), y=Y, ldy=N)
    return Y[0, 3, 5].view(torch.int16).cpu().numpy()


@pytest.mark.parametrize("big", [80.5, -81.0, 1e30, float("inf"), float("-inf")])
def test_forward_does_not_depend_on_neighbours(big):
    n, every = 1 << 15, 16                          # a thread works on 16 or 32 consecutive columns
    r = np.random.default_rng(3)
    for k in range(4):
        if k < 2:                                   # all magnitudes up to the packed form's end
            z = r.uniform(-80, 80, n).astype(np.float32)
        else:
            z = (10.0 ** r.uniform(-38, 1.9, n) * r.choice([-1, 1], n)).astype(np.float32)
        mixed = z.copy()
        mixed[5::every] = big
        rest = np.ones(n, bool)
        rest[5::every] = False
        np.testing.assert_array_equal(silu_of(z)[rest], silu_of(mixed)[rest])


@pytest.mark.parametrize("layer", [0, 1])           # the plain derivative, and the one with the pooling's adjoint
def test_gradient_does_not_depend_on_neighbours(layer):
    """One channel holds z = 70 or z = 100 everywhere and goes nowhere: the gradients of the others
    (eight to a thread) are the same but for the order of their FP32 atomic sums."""
    Bn, H, W, ch = 2, 16, 32, 3
    x, y = smooth_fields(Bn, H, W, 3)
    dx, dy = (torch.tensor(v, dtype=torch.float32, device=dev).contiguous() for v in (x, y))
    off = {name: (o, shape) for name, o, shape in S.param_layout()[0]}

    def view(theta, name):
        o, shape = off[name]
        return theta[o:o + int(np.prod(shape))].reshape(shape)

    got = []
    for z in (70.0, 100.0):
        with S.Surrogate(H, W, seed=5) as m:
            m.set_norm(*NORM)
            theta = m.params()
            view(theta, "head.w")[:] *= 10.0
            view(theta, f"conv{layer}.w")[:, ch] = 0.0
            view(theta, f"conv{layer}.b")[ch] = z
            view(theta, f"conv{layer + 1}.w")[ch:9 * 32:32] = 0.0
            if layer == 1:
                view(theta, "conv12.w")[ch:9 * 64:64] = 0.0
            m.set_params(theta)
            torch.cuda.synchronize()
            m.forward_backward(dx.data_ptr(), dy.data_ptr(), Bn)
            g = m.grads()
            got.append([view(g, f"conv{k}.{s}").astype(np.float64) for k in range(layer + 1) for s in "wb"])
    for a, b in zip(*got):
        assert np.isfinite(a).all() and np.linalg.norm(a) > 0
        assert rel_l2(b, a) <= 1e-4
