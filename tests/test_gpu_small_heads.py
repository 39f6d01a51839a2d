"""CG scalars of the strip kernels whose blocks have fewer than 32 threads (L <= 10: 9, 16 and
25): their heads sum up to a few hundred partials with the lanes there are.  A wrong sum
makes a wrong beta, which the FP64 residual checks turn into iterations, so the counts are
compared with the oracle's recurrences.

Tolerances: FP64 preconditioned CG follows the oracle's to rounding: 5 % and 3 iterations
(those of test_gpu_precond.py are within 2 of 170).  The mixed solvers lose some of their
directions to FP32 and to the residual updates: 1.3 times the oracle's count and 50.  The
updates come every 10 iterations here: a preconditioned mixed solve that meets its
tolerance in FP32 before the first update goes on with a direction that is too long for
the true residual (the generic kernels, whose blocks have full warps, do the same).
"""
import numpy as np
import pytest
import torch

import oracle
from oracle import precond as opc
from paper_2508_16298_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def hq():
    from paper_2508_16298_gb300 import build
    build.build()
    from paper_2508_16298_gb300 import hqmc
    return hqmc


def cuda(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


@pytest.mark.parametrize("L,N", [(6, 64), (8, 40), (10, 100), (8, 192)])
@pytest.mark.parametrize("variant,autotune", [(0, False), (2, False), (3, False), (0, True)])
def test_iterations_of_small_lattices(hq, L, N, variant, autotune):
    lat, theta, phi = oracle.Lattice(L, N), inputs.theta_ordered(L, N, 61, tau_walk=0.0), inputs.complex_gaussian(L, N, 62)
    th, b = cuda(theta), cuda(phi)
    it_p = opc.pcg(lat, theta, phi, opc.coefficients(lat), tol=1e-8)[1]
    it_c = oracle.cg(lat, theta, phi, tol=1e-8)[1]
    bound = {"pcg64": 1.05 * it_p + 3, "cg64": 1.05 * it_c + 3, "pmixed": 1.3 * it_p + 50, "mixed": 1.3 * it_c + 50}
    with hq.Config(L, N, variant=variant, autotune=autotune, reliable_interval=10) as cfg:
        for solver, most in bound.items():
            hq.set_timing(cfg, solver == "cg64")  # timed: the two-kernel loop instead of one cluster
            x, i = hq.cg_solve(cfg, th, b, tol=1e-8, maxit=20 * it_c, solver=solver, raise_on_fail=False)
            assert i["status"] == 0 and i["iterations"] <= most, (solver, i["iterations"], most)
        hq.set_timing(cfg, False)
        if variant == 2:  # no tau-walking kernel, which systems solved together need
            return
        hq.set_multi_rhs(cfg, 3)
        X, infos = hq.cg_solve_multi(cfg, th, torch.stack([b, 2 * b, b.conj().resolve_conj()]), tol=1e-8, maxit=20 * it_c,
                                     solver="pmixed", raise_on_fail=False)
        for i in infos:
            assert i["status"] == 0 and i["iterations"] <= bound["pmixed"]
