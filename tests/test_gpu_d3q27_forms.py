"""The two forms of the FP32 D3Q27 step (one CTA per SM with its loads issued together, and
two) round alike: z-chunks that make few CTAs and z-chunks that make many leave, bit for bit,
the same populations."""
import numpy as np
import pytest

import paper_2508_00577_gb300 as ev
from test_gpu_launch_shapes import A, B, fields

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,ny,nz,few,many", [(64, 64, 40, 40, 2), (75, 50, 61, 61, 4), (33, 9, 200, 200, 2),
                                                (200, 130, 7, 7, 3)])
@pytest.mark.parametrize("thermal", [1, 0])
@pytest.mark.parametrize("eos", [ev.LBM_EOS_CS, ev.LBM_EOS_VDW])
def test_forms_round_alike(nx, ny, nz, few, many, thermal, eos):
    f = fields(ev.LBM_D3Q27, nx, ny, nz)
    # The van der Waals gas at a pressure near the Carnahan-Starling fluid's: b small enough that
    # 1 - b rho stays positive.
    b = B if eos == ev.LBM_EOS_CS else 0.5
    p = ev.lbm_params.make(lattice=ev.LBM_D3Q27, nx=nx, ny=ny, nz=nz, eos=eos, a=A, b=b, kappa=0.05, thermal=thermal,
                           precision=ev.LBM_FP32)
    with ev.Lattice(p, *f) as one, ev.Lattice(p, *f) as two:
        ev.lbm_set_tile(one.ctx, 0, few)
        ev.lbm_set_tile(two.ctx, 0, many)
        for x, y in zip(one.step(4).populations(), two.step(4).populations()):
            if x is not None:
                assert np.isfinite(x).all()
                assert np.array_equal(x, y)
