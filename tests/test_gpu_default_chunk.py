"""The D3Q27 z-chunk that the library picks is not worse than chunks of 64 planes, on lattices
whose grids end on one long chunk if the estimate counts only the work."""
import pytest

torch = pytest.importorskip("torch")

import paper_2508_00577_gb300 as ev
from test_gpu_dependent_launch import params
from test_gpu_launch_shapes import fields

pytestmark = pytest.mark.gpu


def us_per_step(g, stream, steps=10):
    best = 1e30
    for _ in range(5):
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        with torch.cuda.stream(stream):
            e0.record()
            g.step(steps)
            e1.record()
        torch.cuda.synchronize()
        best = min(best, e0.elapsed_time(e1) * 1e3 / steps)
    return best


@pytest.mark.parametrize("n", [(170, 96, 161), (153, 125, 195), (160, 160, 160), (75, 50, 61)])
@pytest.mark.parametrize("precision", [ev.LBM_FP32, ev.LBM_BF16_DEV])
def test_not_slower_than_64_planes(n, precision):
    case = (ev.LBM_D3Q27, *n, precision)
    stream = torch.cuda.Stream()
    with ev.Lattice(params(*case), *fields(*case[:4]), stream=stream.cuda_stream) as g:
        own = us_per_step(g, stream)
        ev.lbm_set_tile(g.ctx, 0, 64)
        planes64 = us_per_step(g, stream)
    print(f"{case}: own {own:.1f} us a step, 64 planes {planes64:.1f}")
    # Up to 3 % measured where 64 planes happen to fit; 1.2 to 1.5 times where the end was not seen.
    assert own <= 1.08 * planes64
