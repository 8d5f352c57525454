"""Macroscopic fields of the fused kernels against the oracle with wall columns, and with FP16
storage (the forms that the other tests of the fields leave out)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle
import oracle.eos as E
import paper_2508_00577_gb300 as ev
from paper_2508_00577_gb300 import inputs

pytestmark = pytest.mark.gpu

A, B = 0.1, 4.0


def compare(o, g, tol):
    ro, uo, To, Fo = o.macro()
    rg, ug, Tg, Fg = g.moments()
    assert np.abs(rg / ro - 1).max() <= tol and np.abs(Tg / To - 1).max() <= tol
    assert np.abs(ug - uo.reshape(ug.shape)).max() <= 0.1 * tol
    assert np.abs(Fg - Fo.reshape(Fg.shape)).max() <= 0.1 * tol
    N = ro.size
    d = torch.full((ug.shape[0] + 2, N), float("nan"), device="cuda")
    q = d.data_ptr()
    ev.lbm_moments_device(g.ctx, q, q + 4 * N, q + 4 * N * (ug.shape[0] + 1))
    ev.lbm_sync(g.ctx)
    d = d.cpu().numpy()
    np.testing.assert_array_equal(d[0], rg.astype(np.float32))
    np.testing.assert_array_equal(d[1:-1], ug.astype(np.float32))
    np.testing.assert_array_equal(d[-1], Tg.astype(np.float32))           # R = 1


@pytest.mark.parametrize("nx,ny,nz", [(3, 1, 1), (64, 7, 2), (65, 33, 1), (131, 5, 3)])
@pytest.mark.parametrize("thermal", [1, 0])
def test_walls(nx, ny, nz, thermal):
    N = nx * ny * nz
    r = np.random.default_rng(nx)
    rho, T = 1.0 + 0.02 * r.random(N), 0.2 + 0.002 * r.random(N)
    u = 0.01 * r.standard_normal((2, N))
    walls = ((0, 0, 0), (0, 0.1, 0), 0.2)
    p = ev.lbm_params.make(nx=nx, ny=ny, nz=nz, eos=ev.LBM_EOS_VDW, a=0.05, b=0.1, kappa=0.0, tau=0.5, thermal=thermal,
                           precision=ev.LBM_FP32)
    o = oracle.State(oracle.Params(Q=9, nx=nx, ny=ny, nz=nz, eos=E.VDW, a=0.05, b=0.1, kappa=0.0, tau=0.5,
                                   thermal=thermal, walls=walls), rho, u, T)
    with ev.Lattice(p, rho, u, T) as g:
        ev.lbm_set_walls(g.ctx, 1, *walls)
        o.step(3)
        g.step(3)
        compare(o, g, 1e-5)                     # FP32 arithmetic, as the parity tests


@pytest.mark.parametrize("Q,nx,ny,nz", [(9, 65, 33, 2), (9, 300, 5, 1), (27, 33, 9, 35)])
@pytest.mark.parametrize("thermal", [1, 0])
def test_fp16(Q, nx, ny, nz, thermal):
    RT = 0.85 * E.critical_point(E.CS, A, B)[1]
    rho, u, T = inputs.spinodal_noise(nx, ny, nz, 0.5 * sum(E.spinodal(E.CS, A, B, RT)), RT, D=2 if Q == 9 else 3)
    o = oracle.State(oracle.Params(Q=Q, nx=nx, ny=ny, nz=nz, eos=E.CS, a=A, b=B, kappa=0.05, tau=0.3, thermal=thermal),
                     rho, u, T)
    p = ev.lbm_params.make(lattice=ev.LBM_D2Q9 if Q == 9 else ev.LBM_D3Q27, nx=nx, ny=ny, nz=nz, eos=ev.LBM_EOS_CS,
                           a=A, b=B, kappa=0.05, thermal=thermal, precision=ev.LBM_FP16_DEV)
    with ev.Lattice(p, rho, u, T) as g:
        o.step(2)
        g.step(2)
        compare(o, g, 1e-3)                     # deviations rounded to FP16, as the tests with BF16
