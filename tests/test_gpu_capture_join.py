"""Overlapping steps after a join of streams: captured into a graph where a step's launch depends on
a copy and a kernel of another stream, and uncaptured behind an event, the steps see what the other
stream wrote and hold the populations of steps apart."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import paper_2508_00577_gb300 as ev
from test_gpu_dependent_launch import params
from test_gpu_launch_shapes import fields

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("case", [(ev.LBM_D2Q9, 331, 203, 2, ev.LBM_FP32), (ev.LBM_D2Q9, 64, 64, 1, ev.LBM_FP64),
                                  (ev.LBM_D3Q27, 33, 20, 17, ev.LBM_FP32)])
@pytest.mark.parametrize("captured", [True, False])
def test_steps_after_a_join(case, captured):
    p, f = params(*case), fields(*case[:4])
    N = p.N
    main, side = torch.cuda.Stream(), torch.cuda.Stream()
    # The restart's fields are written on the side stream right before the join (not for FP64,
    # which has no restart).
    restart = case[-1] != ev.LBM_FP64
    src = torch.tensor(np.concatenate([np.asarray(a).reshape(-1) for a in f]), dtype=torch.float32, device="cuda")
    dst = torch.zeros_like(src)
    q = dst.data_ptr()
    D = p.D
    torch.cuda.synchronize()
    with ev.Lattice(p, *f, stream=main.cuda_stream) as g, ev.Lattice(p, *f) as apart:
        g.step(2)
        apart.step(2)
        if restart:
            ev.lbm_reset_device(apart.ctx, src.data_ptr(), src.data_ptr() + 4 * N, src.data_ptr() + 4 * N * (D + 1))
        for _ in range(6):
            apart.step(1)
            torch.cuda.synchronize()

        def work():
            side.wait_stream(main)
            with torch.cuda.stream(side):
                torch.mul(src, 0.5, out=dst)
                dst.copy_(src)
            main.wait_stream(side)
            if restart:
                ev.lbm_reset_device(g.ctx, q, q + 4 * N, q + 4 * N * (D + 1))
            g.step(4)
            side.wait_stream(main)
            with torch.cuda.stream(side):
                dst.zero_()                                        # a join right before a step
            main.wait_stream(side)
            g.step(2)

        torch.cuda.synchronize()
        if captured:
            graph = torch.cuda.CUDAGraph()
            with torch.cuda.graph(graph, stream=main):
                work()
            graph.replay()
        else:
            with torch.cuda.stream(main):
                work()
        torch.cuda.synchronize()
        for a, b in zip(apart.populations(), g.populations()):
            assert np.array_equal(a, b)
