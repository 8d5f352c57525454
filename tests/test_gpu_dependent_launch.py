"""Steps whose launches overlap (programmatic dependent launch) hold, bit for bit, the
populations of steps that each wait for the one before on the host, and of a captured graph:
lattices of one CTA, of fewer CTAs than SMs (one CTA per SM handing over to the next grid), of
more than one and of more than the GPU holds, and the FP64 stage kernels."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import paper_2508_00577_gb300 as ev
from test_gpu_launch_shapes import A, B, fields

pytestmark = pytest.mark.gpu

CASES = [(ev.LBM_D2Q9, 40, 6, 1, ev.LBM_FP32), (ev.LBM_D2Q9, 331, 203, 2, ev.LBM_FP32),
         (ev.LBM_D2Q9, 256, 256, 6, ev.LBM_FP32), (ev.LBM_D2Q9, 700, 380, 9, ev.LBM_FP32),
         (ev.LBM_D2Q9, 331, 203, 1, ev.LBM_FP16_DEV), (ev.LBM_D2Q9, 64, 64, 1, ev.LBM_FP64),
         (ev.LBM_D3Q27, 33, 20, 17, ev.LBM_FP32), (ev.LBM_D3Q27, 75, 50, 61, ev.LBM_FP32),
         (ev.LBM_D3Q27, 40, 40, 20, ev.LBM_BF16_DEV), (ev.LBM_D3Q27, 12, 10, 8, ev.LBM_FP64)]


def params(lattice, nx, ny, nz, precision):
    return ev.lbm_params.make(lattice=lattice, nx=nx, ny=ny, nz=nz, eos=ev.LBM_EOS_CS, a=A, b=B, kappa=0.05,
                              precision=precision)


@pytest.mark.parametrize("case", CASES)
def test_overlapping_launches_change_nothing(case):
    p, f = params(*case), fields(*case[:4])
    stream = torch.cuda.Stream()
    with ev.Lattice(p, *f) as apart, ev.Lattice(p, *f) as own, ev.Lattice(p, *f, stream=stream.cuda_stream) as cap:
        for _ in range(14):
            apart.step(1)
            torch.cuda.synchronize()
        want = apart.populations()
        for a, b in zip(want, own.step(14).populations()):
            assert np.array_equal(a, b)
        cap.step(2)
        torch.cuda.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=stream):
            cap.step(4)                              # an even count: the buffers' roles are back
        for _ in range(3):
            graph.replay()
        torch.cuda.synchronize()
        for a, b in zip(want, cap.populations()):
            assert np.array_equal(a, b)
