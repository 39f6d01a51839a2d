"""H1 of a mixed-precision trajectory takes Re <X, r> of the last FP64 residual r = phi - O X:
2 Re <phi, X> - <X, O X> = phi^dagger O^{-1} phi - r^dagger O^{-1} r, second order in r.

Steps of 1e-13 leave the field where it was, so that dH = -r^dagger O^{-1} r with r of the
solve from zero (with the chronological guess X becomes c X, c the Galerkin coefficient,
which moves the value by <X, r>^2 / <X, O X>, below 1e-12 here).  Tolerance: 1 % and 3e-7, the
rounding of r to float, 6e-8 |r| |X|.  Without the term dH is off by Re <X, r>: 6e-5 for the
mixed solver at 12^2 x 48, and 2e-4 and 8e-4 with the guess, which is not orthogonal to r.
"""
import numpy as np
import pytest
import torch

from paper_2508_16298_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def hq():
    from paper_2508_16298_gb300 import build
    build.build()
    from paper_2508_16298_gb300 import hqmc
    return hqmc


@pytest.mark.parametrize("L,N", [(12, 48), (18, 60)])
@pytest.mark.parametrize("solver", ["mixed", "pmixed"])
@pytest.mark.parametrize("guess", [0, 4])
def test_h1_is_second_order_in_the_residual(hq, L, N, solver, guess):
    th = torch.from_numpy(inputs.theta_ordered(L, N, 301, tau_walk=0.0)).cuda()
    R = torch.from_numpy(inputs.complex_gaussian(L, N, 302)).cuda()
    with hq.Config(L, N, reliable_interval=10) as cfg:
        phi = hq.apply_M(cfg, th, R, dagger=True)
        X, _ = hq.cg_solve(cfg, th, phi, tol=1e-5, solver=solver)
        r = phi - hq.apply_MdagM(cfg, th, X)
        w, _ = hq.cg_solve(cfg, th, r, tol=1e-8, solver="pcg64")
        want = -torch.vdot(r.flatten(), w.flatten()).real.item()
        hq.set_guess_history(cfg, guess)
        info = hq.trajectory(cfg, th.clone(), seed=7, traj_counter=1, R_in=R, u_in=0.5, nsteps=3, dt=1e-13, tol=1e-5,
                             solver=solver)
    assert abs(info["dH"] - want) <= 0.01 * abs(want) + 3e-7, (info["dH"], want)
