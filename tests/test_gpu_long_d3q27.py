"""D3Q27 lattices of more tiles in y, or more z-chunks, than a grid holds in that direction
(65535).  They repeat a short lattice, so they must hold its fields, repeated, bit for bit."""
import numpy as np
import pytest

import oracle.eos as E
import paper_2508_00577_gb300 as ev
from paper_2508_00577_gb300 import inputs

pytestmark = pytest.mark.gpu

A, B, SHORT, TIMES = 0.1, 4.0, 50, 12000


def lattice(ny, nz, f, precision):
    return ev.Lattice(ev.lbm_params.make(lattice=ev.LBM_D3Q27, nx=2, ny=ny, nz=nz, eos=ev.LBM_EOS_CS, a=A, b=B,
                                         kappa=0.05, precision=precision), *f)


@pytest.mark.parametrize("axis,precision,steps,tile", [
    ("y", ev.LBM_FP32, 0, None),                        # 75000 tiles of the fields (the step has no such grid)
    ("y", ev.LBM_FP16_DEV, 2, None),                    # 75000 tiles of the fields, 37500 of the step
    ("z", ev.LBM_FP32, 2, 1), ("z", ev.LBM_BF16_DEV, 2, 4), ("z", ev.LBM_FP32, 2, None), ("z", ev.LBM_FP32, 2, "tuned")])
def test_long_lattice_repeats_the_short_one(axis, precision, steps, tile):
    RT = 0.85 * E.critical_point(E.CS, A, B)[1]
    short = inputs.spinodal_noise(2, *((SHORT, 1) if axis == "y" else (1, SHORT)), 0.5 * sum(E.spinodal(E.CS, A, B, RT)),
                                  RT, D=3)
    long_ = [np.tile(np.asarray(a).reshape(-1, 2 * SHORT), (1, TIMES)).reshape(np.asarray(a).shape[:-1] + (-1,))
             for a in short]
    n = (SHORT, 1), (SHORT * TIMES, 1)
    if axis == "z":
        n = (1, SHORT), (1, SHORT * TIMES)
    with lattice(*n[0], short, precision) as a, lattice(*n[1], long_, precision) as b:
        if tile == "tuned":
            ev.lbm_autotune(b.ctx, 1)
        elif tile:
            ev.lbm_set_tile(b.ctx, 0, tile)
        for x, y in zip(a.step(steps).moments(), b.step(steps).moments()):
            x, y = np.atleast_2d(x), np.atleast_2d(y)
            assert np.array_equal(np.tile(x, (1, TIMES)), y)
