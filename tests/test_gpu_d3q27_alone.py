"""The D3Q27 FP32 form that takes whole SMs: only where the library picks the shape, the same
populations as with a shape of the caller's, and no index out of range."""
import json
import os
import subprocess
import sys

import numpy as np
import pytest

torch = pytest.importorskip("torch")

import paper_2508_00577_gb300 as ev
from test_gpu_contexts_at_once import check
from test_gpu_launch_shapes import A, B, fields

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("tile_h", [10, 61])
def test_set_shapes_share_the_sms(tile_h):
    # Two grids of at most one CTA per SM fit on the GPU at once; taking whole SMs they would take
    # twice the time of one (1.8 times, measured, when they did).
    check((ev.LBM_D3Q27, 75, 50, 61, ev.LBM_FP32), 2, 1.6, (0, tile_h))


@pytest.mark.parametrize("nx,ny,nz,fixed", [(64, 64, 40, 2), (75, 50, 61, 61), (33, 9, 200, 200), (200, 130, 7, 7),
                                            (5, 3, 2, 1)])
@pytest.mark.parametrize("thermal", [1, 0])
@pytest.mark.parametrize("eos", [ev.LBM_EOS_CS, ev.LBM_EOS_VDW])
def test_own_shape_rounds_as_a_set_one(nx, ny, nz, fixed, thermal, eos):
    f = fields(ev.LBM_D3Q27, nx, ny, nz)
    b = B if eos == ev.LBM_EOS_CS else 0.5               # van der Waals: 1 - b rho stays positive
    p = ev.lbm_params.make(lattice=ev.LBM_D3Q27, nx=nx, ny=ny, nz=nz, eos=eos, a=A, b=b, kappa=0.05, thermal=thermal,
                           precision=ev.LBM_FP32)
    with ev.Lattice(p, *f) as own, ev.Lattice(p, *f) as tuned, ev.Lattice(p, *f) as other:
        ev.lbm_autotune(tuned.ctx, 1)
        ev.lbm_set_tile(other.ctx, 0, fixed)
        want = other.step(4).populations()
        for g in (own, tuned):
            for x, y in zip(want, g.step(4).populations()):
                if x is not None:
                    assert np.isfinite(x).all()
                    assert np.array_equal(x, y)


CHILD = r'''
import json, sys
import numpy as np
sys.path[:0] = [ROOT, ROOT + "/tests"]
import paper_2508_00577_gb300 as ev
from test_gpu_launch_shapes import A, B, fields
out = [ev.lbm_bounds_violations()]
for nx, ny, nz in [(20, 18, 11), (33, 16, 7), (5, 3, 4), (75, 50, 61), (64, 8, 50), (1, 1, 1)]:
    for thermal in (1, 0):
        p = ev.lbm_params.make(lattice=ev.LBM_D3Q27, nx=nx, ny=ny, nz=nz, eos=ev.LBM_EOS_CS, a=A, b=B, kappa=0.05,
                               thermal=thermal, precision=ev.LBM_FP32)
        with ev.Lattice(p, *fields(ev.LBM_D3Q27, nx, ny, nz)) as g:
            assert np.isfinite(g.step(4).moments()[0]).all()
        out.append(ev.lbm_bounds_violations())
print(json.dumps(out))
'''


def test_own_shape_stays_in_bounds():
    from paper_2508_00577_gb300 import _build
    lib = _build.build(bounds_check=True)
    r = subprocess.run([sys.executable, "-c", f"ROOT = {ROOT!r}\n" + CHILD], capture_output=True, text=True,
                       env=dict(os.environ, EVLBM_LIBRARY=lib), timeout=600)
    assert r.returncode == 0, r.stderr[-2000:]
    counts = json.loads(r.stdout.strip().splitlines()[-1])
    assert counts == [0] * len(counts)
