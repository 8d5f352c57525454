"""D2Q9 stacks of more layers, and layers of more chunks, than one launch grid holds (65535):
the step and the fields with the shape the library picks, a tuned one and chunks of two rows."""
import numpy as np
import pytest

import oracle.eos as E
import paper_2508_00577_gb300 as ev
from paper_2508_00577_gb300 import inputs

pytestmark = pytest.mark.gpu

A, B = 0.1, 4.0


def lattice(nx, ny, nz, f, precision):
    return ev.Lattice(ev.lbm_params.make(nx=nx, ny=ny, nz=nz, eos=ev.LBM_EOS_CS, a=A, b=B, kappa=0.05,
                                         precision=precision), *f)


def noise(nx, ny, nz):
    RT = 0.85 * E.critical_point(E.CS, A, B)[1]
    return inputs.spinodal_noise(nx, ny, nz, 0.5 * sum(E.spinodal(E.CS, A, B, RT)), RT, D=2)


@pytest.mark.parametrize("precision", [ev.LBM_FP32, ev.LBM_FP16_DEV])
@pytest.mark.parametrize("shape", ["own", "tuned", (64, 2), (128, ev.LBM_TILE_BALANCED)])
def test_layers_beyond_one_grid(shape, precision):
    nx, ny, nz = 4, 4, 66000
    pick = [0, 1, 65534, 65535, 65536, nz - 1]
    f = [np.asarray(a).reshape(-1, nz, ny * nx) for a in noise(nx, ny, nz)]
    few = [np.ascontiguousarray(a[:, pick]).reshape(-1) for a in f]
    with lattice(nx, ny, nz, [a.reshape(-1) for a in f], precision) as deep, \
            lattice(nx, ny, len(pick), few, precision) as ref:
        if shape == "tuned":
            ev.lbm_autotune(deep.ctx, 1)
        elif shape != "own":
            ev.lbm_set_tile(deep.ctx, *shape)
        for a, b in zip(deep.step(3).moments(), ref.step(3).moments()):
            assert np.array_equal(np.asarray(a).reshape(-1, nz, ny * nx)[:, pick].reshape(-1), np.asarray(b).reshape(-1))
        for a, b in zip(deep.populations(), ref.populations()):
            assert np.array_equal(np.asarray(a).reshape(-1, nz, ny * nx)[:, pick].reshape(-1), np.asarray(b).reshape(-1))


@pytest.mark.parametrize("shape", ["own", "tuned", (64, 2)])
def test_chunks_beyond_one_grid(shape):
    nx, ny = 2, 1200001
    f = noise(nx, ny, 1)
    with lattice(nx, ny, 1, f, ev.LBM_FP32) as g, lattice(nx, ny, 1, f, ev.LBM_FP32) as ref:
        ev.lbm_set_tile(ref.ctx, 64, 128)
        if shape == "tuned":
            ev.lbm_autotune(g.ctx, 1)
        elif shape != "own":
            ev.lbm_set_tile(g.ctx, *shape)
        for a, b in zip(g.step(2).populations() + g.moments(), ref.step(2).populations() + ref.moments()):
            assert np.array_equal(a, b)
