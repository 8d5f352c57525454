"""Short items of the persistent ensemble: work items of 8 and 16 rows (and fewer than a
pipeline's fill), and whatever the autotuner picks for a small ensemble, leave the same values
as items of 64 rows, bit for bit."""
import numpy as np
import pytest

import paper_2508_00577_gb300 as ev
from test_gpu_batch import ensemble

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("sizes", [[(64, 64), (160, 96), (80, 144)], [(100, 75), (33, 7)]])
def test_short_items_are_bit_identical(sizes):
    p, fields, _ = ensemble([(64, 64)] * len(sizes))
    r = np.random.default_rng(7)
    fields = [(f[0][0] * (1 + 0.02 * r.random(nx * ny)), 0.001 * r.normal(size=(2, nx * ny)), np.full(nx * ny, f[2][0]))
              for f, (nx, ny) in zip(fields, sizes)]
    rho, u, T = ([f[k] for f in fields] for k in range(3))
    out = []
    for tile in ((128, 64), (128, 16), (96, 8), (64, 2), None):
        with ev.Batch(p, sizes, rho, u, T) as bt:
            if tile:
                bt.set_tile(*tile)
            else:
                bt.autotune(2)
            bt.step(7)
            out.append(np.concatenate([np.concatenate([x.ravel() for x in bt.moments(d)]) for d in range(len(sizes))]))
    assert np.isfinite(out[0]).all()
    for o in out[1:]:
        assert np.array_equal(out[0], o)
