"""T = R T / R of the fused fields at the ends of the FP32 range: gas constants beyond it, an
infinite R T, and subnormal values.  A frozen temperature field gives back R T as it was stored."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import paper_2508_00577_gb300 as ev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("lattice,nx,ny,nz", [(ev.LBM_D2Q9, 70, 9, 1), (ev.LBM_D3Q27, 33, 5, 3)])
@pytest.mark.parametrize("R", [1.0, 2.5, 3e-42, 1e-35, 2.0 ** -100, 1e29, 1e31, 1e39, 1e150])
@pytest.mark.parametrize("precision", [ev.LBM_FP32, ev.LBM_FP16_DEV])
def test_temperature_over_the_range(lattice, nx, ny, nz, R, precision):
    N, D = nx * ny * nz, 2 if lattice == ev.LBM_D2Q9 else 3
    # R T over the FP32 range and past its ends (0 after rounding, infinite).
    RT = 10.0 ** np.random.default_rng(0).uniform(-46, 40, N)
    T = RT / R
    T = np.where((T > 0) & np.isfinite(T), T, 1.0)
    with np.errstate(over="ignore", under="ignore"):
        held = (R * T).astype(np.float32).astype(np.float64)
        want = (held / R).astype(np.float32).astype(np.float64)
    p = ev.lbm_params.make(lattice=lattice, nx=nx, ny=ny, nz=nz, eos=ev.LBM_EOS_VDW, a=0.1, b=0.0, R=R, thermal=0,
                           precision=precision)
    with ev.Lattice(p, np.full(N, 0.1), np.zeros((D, N)), T) as g:
        d = torch.full((N,), -1.0, device="cuda")
        ev.lbm_moments_device(g.ctx, 0, 0, d.data_ptr())
        ev.lbm_sync(g.ctx)
        got = d.cpu().numpy().astype(np.float64)
        host = g.moments()[2]
    np.testing.assert_array_equal(np.isinf(got), np.isinf(want))
    fin = np.isfinite(want)
    # one FP32 rounding; below the normal range one unit of the smallest number
    assert np.all(np.abs(got[fin] - want[fin]) <= 2.0 ** -23 * np.abs(want[fin]) + 2.0 ** -149)
    np.testing.assert_array_equal(host, held / R)
