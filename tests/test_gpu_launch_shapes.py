"""The launch shapes the library picks by itself change no result.

A fused step's arithmetic does not depend on the strip width, the chunk height or the
z-chunk, so a context that picks its own shape holds, bit for bit, the populations of one
with a fixed shape: lattices of one strip and several, flat and tall ones, stacks of layers,
and D3Q27 sizes on both sides of the resident number of CTAs.
"""
import numpy as np
import pytest

import oracle.eos as E
import paper_2508_00577_gb300 as ev
from paper_2508_00577_gb300 import inputs

pytestmark = pytest.mark.gpu

A, B = 0.1, 4.0


def fields(lattice, nx, ny, nz):
    _, Tc = E.critical_point(E.CS, A, B)
    RT = 0.85 * Tc
    s1, s2 = E.spinodal(E.CS, A, B, RT)
    return inputs.spinodal_noise(nx, ny, nz, 0.5 * (s1 + s2), RT, D=2 if lattice == ev.LBM_D2Q9 else 3)


@pytest.mark.parametrize("lattice,nx,ny,nz,tile", [
    (ev.LBM_D2Q9, 1, 1, 1, (64, 2)), (ev.LBM_D2Q9, 65, 3, 1, (128, 128)), (ev.LBM_D2Q9, 64, 64, 1, (64, 64)),
    (ev.LBM_D2Q9, 129, 1, 5, (128, 128)), (ev.LBM_D2Q9, 331, 203, 2, (128, 128)), (ev.LBM_D2Q9, 30, 2501, 1, (96, 64)),
    (ev.LBM_D2Q9, 700, 380, 9, (192, 32)),
    (ev.LBM_D3Q27, 5, 3, 2, (0, 64)), (ev.LBM_D3Q27, 75, 50, 61, (0, 64)), (ev.LBM_D3Q27, 33, 9, 140, (0, 32)),
    (ev.LBM_D3Q27, 130, 90, 40, (0, 8))])
@pytest.mark.parametrize("precision", [ev.LBM_FP32, ev.LBM_FP16_DEV])
def test_default_shape_is_bit_identical(lattice, nx, ny, nz, tile, precision):
    p = ev.lbm_params.make(lattice=lattice, nx=nx, ny=ny, nz=nz, eos=ev.LBM_EOS_CS, a=A, b=B, kappa=0.05,
                           precision=precision)
    f = fields(lattice, nx, ny, nz)
    with ev.Lattice(p, *f) as own, ev.Lattice(p, *f) as fixed:
        ev.lbm_set_tile(fixed.ctx, *tile)
        for a, b in zip(own.step(3).populations(), fixed.step(3).populations()):
            assert np.array_equal(a, b)
