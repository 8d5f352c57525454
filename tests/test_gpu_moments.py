"""Macroscopic fields of the fused moments kernels against the oracle, at lattices around the
strip, chunk and tile edges, with a gas constant other than 1 and with outputs left out."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle
import oracle.eos as E
import paper_2508_00577_gb300 as ev
from paper_2508_00577_gb300 import inputs

pytestmark = pytest.mark.gpu

A, B, R = 0.1, 4.0, 2.5


@pytest.mark.parametrize("Q,nx,ny,nz", [
    (9, 1, 1, 1), (9, 63, 5, 2), (9, 65, 33, 1), (9, 129, 31, 3), (9, 300, 67, 1), (9, 33, 200, 5),
    (27, 1, 1, 1), (27, 31, 7, 3), (27, 32, 8, 33), (27, 33, 9, 35), (27, 70, 20, 5)])
@pytest.mark.parametrize("thermal", [1, 0])
@pytest.mark.parametrize("precision", [ev.LBM_FP32, ev.LBM_BF16_DEV])
def test_fields_match_oracle(Q, nx, ny, nz, thermal, precision):
    _, Tc = E.critical_point(E.CS, A, B)
    RT = 0.85 * Tc
    s1, s2 = E.spinodal(E.CS, A, B, RT)
    D = 2 if Q == 9 else 3
    rho, u, T = inputs.spinodal_noise(nx, ny, nz, 0.5 * (s1 + s2), RT / R, D=D)
    u = 0.01 * np.random.default_rng(1).standard_normal(u.shape)
    o = oracle.State(oracle.Params(Q=Q, nx=nx, ny=ny, nz=nz, eos=E.CS, a=A, b=B, R=R, kappa=0.05, tau=0.3,
                                   thermal=thermal), rho, u, T)
    p = ev.lbm_params.make(lattice=ev.LBM_D2Q9 if Q == 9 else ev.LBM_D3Q27, nx=nx, ny=ny, nz=nz, eos=ev.LBM_EOS_CS,
                           a=A, b=B, R=R, kappa=0.05, thermal=thermal, precision=precision)
    N = p.N
    with ev.Lattice(p, rho, u, T) as g:
        o.step(2)
        g.step(2)
        ro, uo, To, Fo = o.macro()
        rg, ug, Tg, Fg = g.moments()
        # Two steps of FP32 arithmetic, as the parity tests (1e-5 on rho and T, 1e-6 on u);
        # 16-bit storage rounds deviations of relative size ~u, 1e-3 there.
        tol = 1e-5 if precision == ev.LBM_FP32 else 1e-3
        assert np.abs(rg / ro - 1).max() <= tol and np.abs(Tg / To - 1).max() <= tol
        assert np.abs(ug - uo.reshape(ug.shape)).max() <= 0.1 * tol
        assert np.abs(Fg - Fo.reshape(Fg.shape)).max() <= 0.1 * tol
        d = torch.full((D + 3, N), float("nan"), device="cuda")
        q = d.data_ptr()
        ev.lbm_moments_device(g.ctx, q, q + 4 * N, q + 4 * N * (D + 1))
        ev.lbm_moments_device(g.ctx, 0, 0, q + 4 * N * (D + 2))               # T alone
        ev.lbm_sync(g.ctx)
        d = d.cpu().numpy()
        np.testing.assert_array_equal(d[0], rg.astype(np.float32))
        np.testing.assert_array_equal(d[1:D + 1], ug.astype(np.float32).reshape(D, N))
        np.testing.assert_array_equal(d[D + 1], d[D + 2])
        assert np.abs(d[D + 1] / Tg - 1).max() <= 2 ** -23                  # one FP32 rounding
