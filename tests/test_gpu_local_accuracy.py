"""Accuracy element by element of the operators a program can call, on vectors that are not of
one size: point sources, sparse vectors and vectors that fall off over a slice.  The
fixed-point kernels hold a slice to a fraction of its largest component, so slices
like these take FP64 arithmetic.

Bound: |y - y_oracle|_i <= c 2^-53 (A |x|)_i with A = |M|^T |M| or |M| of non-negative entries
(theta = 0, all signs positive), the form of any FP64 evaluation's error.  A sweep is
seven factors of four roundings each (two products, two additions, the link's own error
among them), so M has 30 and M^dagger M 66 on either side: c = 150 covers both sides of
both operators.
"""
import numpy as np
import pytest
import torch

import oracle
from paper_2508_16298_gb300 import inputs

pytestmark = pytest.mark.gpu
C = 150 * 2.0 ** -53


@pytest.fixture(scope="module")
def hq():
    from paper_2508_16298_gb300 import build
    build.build()
    from paper_2508_16298_gb300 import hqmc
    return hqmc


def cuda(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def vectors(L, N):
    """Sources by name: ones a slice, a few sites, a fall-off within every slice (below, at and far
    beyond 2^-6 of its largest value, where the arithmetic changes), and one in tau."""
    base = inputs.complex_gaussian(L, N, seed=202 + L)
    g = inputs.rng(203 + L)
    y, x = np.indices((L, L))
    d = np.minimum(x, L - x) + np.minimum(y, L - y)
    point = np.zeros_like(base)
    point[N // 2, 3, L - 1] = 1.0
    sparse = np.where(g.random(base.shape) < 0.01, base, 0)
    out = {"point": point, "sparse": sparse, "two sizes": np.where(g.random(base.shape) < 0.5, base, base * 1e-12)}
    for total in (3, 5, 6, 7, 9, 30, 300):  # binary orders over the slice
        out["fall-off %d" % total] = base / np.abs(base) * 2.0 ** (-total * d / L)[None]
    tau = out["fall-off 30"].copy()
    for k in range(N):
        tau[k] *= 10.0 ** (-7 * k)
    out["fall-off in tau too"] = tau
    return out


def positive_M(lat, x, dagger):
    """|M| |x|: apply_M at theta = 0 is x minus or plus B of the neighbour, B of positive entries."""
    a = np.abs(x).astype(complex)
    return a + np.abs(oracle.apply_M(lat, np.zeros((lat.Ntau, lat.L, lat.L, 2)), a, dagger=dagger) - a)


@pytest.mark.parametrize("L,N", [(18, 6), (50, 3), (54, 4), (66, 3)])
@pytest.mark.parametrize("start", ["zero", "hot"])
def test_operators(hq, L, N, start):
    lat = oracle.Lattice(L, N)
    th = np.zeros((N, L, L, 2)) if start == "zero" else inputs.theta_hot(L, N, seed=201 + L)
    with hq.Config(L, N) as cfg:
        assert cfg.launch_shape(hq.FP64)["variant"] >= 200
        for name, x in vectors(L, N).items():
            for dagger in (False, True):
                y = hq.apply_M(cfg, cuda(th), cuda(x), dagger=dagger).cpu().numpy()
                bound = positive_M(lat, x, dagger).real
                assert np.all(np.abs(y - oracle.apply_M(lat, th, x, dagger=dagger)) <= C * bound), (name, dagger)
            y = hq.apply_MdagM(cfg, cuda(th), cuda(x)).cpu().numpy()
            bound = positive_M(lat, positive_M(lat, x, False), True).real
            assert np.all(np.abs(y - oracle.apply_MdagM(lat, th, x)) <= C * bound), name


@pytest.mark.parametrize("L,N", [(18, 6), (50, 3), (54, 4), (66, 3)])
def test_force(hq, L, N):
    """dS_f of bond (i, j) is a product of u = P^-1 ... P X_tau and w = P ... Y_{tau+1}: the bound takes
    each through non-negative B (theta = 0), and their errors together, 60 roundings of u, 40
    of w and 5 of the product on either side: 210 2^-53."""
    lat = oracle.Lattice(L, N)
    th = inputs.theta_hot(L, N, seed=211 + L)
    zero = np.zeros((L, L, 2))
    t1 = np.tanh(lat.dtau * lat.t)
    cB = np.cosh(lat.dtau * lat.t) * np.cosh(lat.dtau * lat.t / 2) ** 6
    with hq.Config(L, N) as cfg:
        for name, X in vectors(L, N).items():
            d = torch.empty((N, L, L, 2), dtype=torch.float64, device="cuda")
            hq.force(cfg, cuda(th), cuda(X), dSf=d)
            a = np.abs(X).astype(complex)
            b = np.stack([oracle.apply_B(lat, zero, v) for v in a])
            u = np.stack([oracle.apply_B(lat, zero, v) for v in b]).real
            w = np.stack([oracle.apply_B(lat, zero, v) for v in np.roll(a, -1, 0) + b]).real
            bound = np.stack([w * np.roll(u, -1, ax) + np.roll(w, -1, ax) * u for ax in (2, 1)], axis=-1)
            err = np.abs(d.cpu().numpy() - oracle.fermion_dS(lat, th, X))
            assert np.all(err <= 210 * 2.0 ** -53 * 4 * t1 * cB * bound), name


@pytest.mark.parametrize("L,N,dtau", [(18, 240, 0.1), (24, 131, 0.05), (10, 300, 0.2), (18, 20, 0.1)])
def test_line_preconditioner(hq, L, N, dtau):
    """Each pass is a sum over a site's line by a recursion acc <- v + rho acc: a rounding of one step
    decays with rho, so the errors of x are those of |x| under the untruncated recursion G, and
    z's those of both passes, scale G^T G^T G G |u|.  Three roundings a step here, W + 1 terms
    summed one by one in the oracle: c = 2 (W + 1) + 16."""
    from oracle import precond as opc
    c = opc.coefficients(oracle.Lattice(L, N, dtau=dtau))

    def recursion(v, back):
        v = v[::-1] if back else v
        acc, out = np.zeros_like(v[0]), np.empty_like(v)
        for k in range(4 * N):  # until the start is forgotten: rho^(3 N) < 1e-9
            acc = v[k % N] + c.rho * acc
            out[k % N] = acc
        return out[::-1] if back else out

    along = inputs.complex_gaussian(L, N, seed=221)
    k = np.arange(N)
    lines = {"fall-off along tau %d" % s: along * 2.0 ** (-s * np.minimum(k, N - k) / N)[:, None, None] for s in (4, 40, 400)}
    with hq.Config(L, N, dtau=dtau) as cfg:
        for name, u in {**vectors(L, N), **lines, "real": along.real + 0j}.items():
            z = hq.apply_precond(cfg, cuda(u)).cpu().numpy()
            bound = np.abs(u)
            for back in (False, False, True, True):
                bound = recursion(bound, back)
            tol = (2 * (c.W + 1) + 16) * 2.0 ** -53 * c.scale
            assert np.all(np.abs(z - opc.apply(c, u)) <= tol * bound), name
